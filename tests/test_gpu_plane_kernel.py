"""The fused plane kernel at both of its block widths (one wide block per SM when the planes are
fewer than the SMs, several narrow ones otherwise) on every grid that has it: moves of the chains of
a batch against the FP64 oracle.  Surveys with one observed octant leave planes, warps' lines and
parts of lines without support; chain 0 sees the whole sky."""
import numpy as np
import pytest

from oracle import gibbs, grid
from paper_1306_1821_gb300 import inputs
from tests.helpers import compare_chain

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,chains", [(32, 1), (32, 6), (64, 1), (64, 4), (96, 1), (96, 3), (128, 1), (128, 2)])
def test_moves_match_the_oracle(N, chains):
    import torch

    from paper_1306_1821_gb300 import bps
    cfg = bps.make_config(4, n_leapfrog=3, eps_max=0.1, jump=0, fixed_bias_index=0, seed=900)
    box = 500.0 * N / 32
    batch = bps.bps_create_batch([N] * chains, [box] * chains, [1] * chains, cfg)
    try:
        starts = []
        for j in range(chains):
            wl = inputs.small_workload(N, n_bins=4, n_sub=1, f_sky=1.0, seed=60 + j)
            delta, counts, R = inputs.make_survey(wl)
            if j > 0:
                R[:, : N // 2] = 0
                R[:, :, : N // 2 + 3] = 0
                R[..., : N // 2 - 5] = 0
                counts[R == 0] = 0
            d32 = (0.8 * delta).astype(np.float32)
            P, b, nbar = inputs.initial_state(wl)
            bps.bps_batch_set_chain(batch, j, torch.from_numpy(counts).cuda(), torch.from_numpy(R).cuda(),
                                    torch.from_numpy(d32).cuda(), P, b, nbar, 0)
            starts.append((counts, R, d32, P, b, nbar))
        rec = bps.bps_batch_gibbs_iterate(batch, 1, chains)
        for j in sorted({0, chains - 1}):
            counts, R, d32, P, b, nbar = starts[j]
            dh = grid.forward(d32.astype(np.float64))
            dh[0, 0, 0] = 0
            ch = gibbs.Chain(grid.Geometry(N, box, 4), counts, R, P, b, nbar, delta_hat=dh, n_leapfrog=3, eps_max=0.1,
                             jump=False, fixed_bias=0, seed=900 + j)
            compare_chain(rec[:, bps.bps_batch_record_slot(batch, j), : 4 + 2 + 2], ch, 1)
            out = torch.zeros((N,) * 3, dtype=torch.float32, device="cuda")
            bps.bps_batch_get_chain(batch, j, out, 4, 1)
            ref = grid.inverse(ch.delta_hat, N)
            err = np.linalg.norm(out.cpu().numpy() - ref) / np.linalg.norm(ref)
            assert err < 2e-4, (j, err)      # the bound of test_hmc_moves_match_oracle
    finally:
        bps.bps_destroy(batch)
