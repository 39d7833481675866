"""Half spectra that the library writes into callers' arrays: straight from the kernels, and by a
copy where the array starts off an 8-byte boundary.  Both give the same bits on every grid, and
nothing is written outside the array."""
import numpy as np
import pytest

from tests.helpers import Problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [8, 16, 32, 96, 256])
def test_aligned_and_unaligned_arrays(N):
    import torch

    from paper_1306_1821_gb300 import bps
    pb = Problem(N, n_sub=1, n_bins=3)
    s = pb.gpu(seed=5)
    n = N * N * (N // 2 + 1) * 2
    real = torch.from_numpy(pb.delta_true.astype(np.float32)).cuda()
    try:
        calls = {"spectrum": lambda out: bps.bps_get_spectrum(s.ctx, out),
                 "gradient": lambda out: bps.bps_gradient(s.ctx, out),
                 "r2c": lambda out: bps.bps_fft_r2c(s.ctx, real, out)}
        for name, call in calls.items():
            got = []
            for off in (2, 1):
                buf = torch.full((n + 6,), 7.5, dtype=torch.float32, device="cuda")
                call(buf[off:off + n])
                h = buf.cpu().numpy()
                assert (h[:off] == 7.5).all() and (h[off + n:] == 7.5).all(), name
                got.append(h[off:off + n])
            assert np.array_equal(got[0], got[1]), name
            if name == "spectrum":
                assert np.array_equal(got[0], pb.dh32.view(np.float32).ravel())
    finally:
        s.close()
