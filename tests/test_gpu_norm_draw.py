"""The generalised-inverse-Gaussian draw of the normalisations over its range of shapes, from one
observed voxel (|p| = 1/2) and two (p = 0) to a full grid, peaked and flat: against the oracle's draw
for the same sums.  Responses of 1/2 and 1 and small counts make the data constants exact, so the two
sides differ by FP64 rounding: the bounds of the rectangle agree to about 1e-12 (the oracle's
y - m loses m / (y - m) ulps), far inside the 1e-9 asked for."""
import numpy as np
import pytest

from oracle import draws, philox

pytestmark = pytest.mark.gpu

N, N_SUB = 16, 6
OBSERVED = [1, 2, 3, 7, 200, N ** 3]


@pytest.mark.parametrize("scale,count", [(1.0, 3), (0.01, 1), (1.0, 4000)])
def test_draws_over_shapes(scale, count):
    import torch

    from paper_1306_1821_gb300 import bps
    rng = np.random.default_rng(2)
    R = np.zeros((N_SUB, N ** 3), dtype=np.float32)
    counts = np.zeros((N_SUB, N ** 3), dtype=np.int32)
    for l, n in enumerate(OBSERVED):
        at = rng.choice(N ** 3, n, replace=False)
        R[l, at] = rng.choice([0.5, 1.0], n)
        counts[l, at] = rng.integers(1, count + 1, n)
    delta = (scale * rng.standard_normal((N, N, N))).astype(np.float32)
    b0, nbar0 = np.linspace(0.8, 1.5, N_SUB), np.linspace(0.5, 6.0, N_SUB)
    s = bps.Sampler(N, 250.0, N_SUB, 4, fixed_bias_index=2, seed=31)
    try:
        bps.bps_set_data(s.ctx, torch.from_numpy(counts).cuda(), torch.from_numpy(R).cuda())
        for it in range(12):
            bps.bps_set_state(s.ctx, torch.from_numpy(delta).cuda(), np.ones(4), b0, nbar0, it)
            b, nbar, sums = bps.bps_sample_bias_norm(s.ctx, N_SUB)
            for l in range(N_SUB):
                S1, S2, S3 = sums[l]
                if l != 2:
                    C = nbar0[l] * S3
                    z = draws.normal_draw(31, it, philox.STAGE_BIAS, l)
                    assert b[l] == pytest.approx((S1 - nbar0[l] * S2) / C + z / np.sqrt(C), rel=1e-9, abs=1e-9)
                R64 = R[l].astype(np.float64)
                obs = R64 > 0
                B = np.sum(counts[l][obs].astype(np.float64) ** 2 / R64[obs])
                A = R64.sum() + 2.0 * b[l] * S2 + b[l] ** 2 * S3
                ref, _ = draws.gig_draw(1.0 - 0.5 * OBSERVED[l], A, B, 31, it, philox.STAGE_NBAR, l)
                assert nbar[l] == pytest.approx(ref, rel=1e-9), (it, l)
    finally:
        s.close()
