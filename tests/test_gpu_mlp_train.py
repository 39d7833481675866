"""bps_mlp_train against its definition, step by step through bps_mlp_loss_grad and
bps_mlp_adam_step on the rows that Philox draws (block r of stream (seed, step, 100, 0), word 0
modulo the number of examples): the same parameters, bit for bit, and the last step's loss.  Sizes
on both sides of the rule that runs small steps in one cluster, with ragged tiles, single layers,
single rows, more steps than one launch takes, and inputs off an 8-byte boundary."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,batch,steps,offset", [
    ([32, 128, 128, 64], 64, 20, 0), ([8, 33, 33, 9], 17, 20, 0), ([5, 7], 1, 8, 0), ([32, 64], 64, 300, 0),
    ([2, 16, 8, 24, 40], 48, 12, 1), ([6, 100, 1], 1024, 4, 1), ([40, 160, 160, 64], 96, 8, 0),
    ([128, 512, 512, 64], 64, 3, 0), ([16, 16], 1025, 3, 0)])
def test_training_is_its_steps(sizes, batch, steps, offset):
    import torch

    from paper_1306_1821_gb300 import bps
    rng = np.random.default_rng(11)
    n, lr, seed = 700, 1e-3, 21
    params = (rng.standard_normal(sum(a * b + b for a, b in zip(sizes[:-1], sizes[1:]))) * 0.2).astype(np.float32)

    def data(d):
        buf = torch.from_numpy(rng.standard_normal(n * d + offset).astype(np.float32)).cuda()
        return buf[offset:].view(n, d)

    x, t = data(sizes[0]), data(sizes[-1])
    one, ref = bps.MLP(sizes), bps.MLP(sizes)
    try:
        one.set_params(params)
        ref.set_params(params)
        loss = one.train(x, t, batch, steps, lr, seed)
        words = torch.zeros(4 * batch, dtype=torch.int64, device="cuda")
        for s in range(steps):
            bps.bps_philox_words(seed, s, 100, 0, 0, words)
            rows = words[::4].cpu().numpy().view(np.uint64) % np.uint64(n)
            rows = torch.from_numpy(rows.astype(np.int64)).cuda()
            last, _ = ref.loss_grad(x[rows].contiguous(), t[rows].contiguous())
            ref.adam_step(lr)
        assert np.array_equal(one.get_params().view(np.uint32), ref.get_params().view(np.uint32))
        assert loss == pytest.approx(last, rel=1e-12)
        # the gradients of the last step are kept for bps_mlp_adam_step
        one.adam_step(lr)
        ref.adam_step(lr)
        assert np.array_equal(one.get_params().view(np.uint32), ref.get_params().view(np.uint32))
    finally:
        one.close()
        ref.close()
