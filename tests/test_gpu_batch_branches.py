"""The groups of a batch run as branches of one CUDA graph: every chain must follow the
single-context chain of the same key, whatever else is in the batch."""
import numpy as np
import pytest

from paper_1306_1821_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[32], [64, 8], [96, 16, 32, 64, 32], [32] * 9 + [16] * 5],
                         ids=["one group", "two", "four", "many chains"])
def test_chains_of_every_branch_equal_single_contexts(sizes):
    import torch

    from paper_1306_1821_gb300 import bps
    kw = dict(n_leapfrog=3, eps_max=0.25, jump=1, jump_leapfrog=2, jump_eps_max=0.2, fixed_bias_index=0)
    nsub = [1 + j % 2 for j in range(len(sizes))]
    ps = []
    for j, (N, ns) in enumerate(zip(sizes, nsub)):
        wl = inputs.small_workload(N, n_bins=3, n_sub=ns, f_sky=0.6, seed=70 + j)
        delta, counts, R = inputs.make_survey(wl)
        ps.append((wl, torch.from_numpy(counts).cuda(), torch.from_numpy(R).cuda(),
                   torch.from_numpy((0.8 * delta).astype(np.float32)).cuda()))
    batch = bps.bps_create_batch(sizes, [p[0].box for p in ps], nsub, bps.make_config(3, seed=21, **kw))
    try:
        for j, (wl, counts, R, d) in enumerate(ps):
            bps.bps_batch_set_chain(batch, j, counts, R, d, *inputs.initial_state(wl), 0)
        # the first call captures the graph, the second replays it twice
        rec = np.concatenate([bps.bps_batch_gibbs_iterate(batch, n, len(ps)) for n in (1, 2)])
        slots = [bps.bps_batch_record_slot(batch, j) for j in range(len(ps))]
        assert sorted(slots) == list(range(len(ps)))
        for j, (wl, counts, R, d) in enumerate(ps):
            s = bps.Sampler(wl.N, wl.box, wl.n_sub, 3, seed=21 + j, **kw)
            bps.bps_set_data(s.ctx, counts, R)
            bps.bps_set_state(s.ctx, d, *inputs.initial_state(wl), 0)
            single = bps.bps_gibbs_iterate(s.ctx, 3, s.rec_len)
            # the two may sum the energies over tiles of different sizes: FP32 rounding apart
            assert np.allclose(rec[:, slots[j], :s.rec_len], single, rtol=1e-5, atol=1e-6), j
            s.close()
    finally:
        bps.bps_destroy(batch)
