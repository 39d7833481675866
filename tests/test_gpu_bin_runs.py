"""The k-bin sums where half a warp takes a column (grids up to 128^3): a lane adds up to five
neighbouring |nx| before anything is combined.  A spectrum whose every L-th |nx| is large and the
others just below half an ulp of it loses L - 1 terms per lane in plain FP32 (1.0e-7 to 2.2e-7 of a
bin's sum); a lane's sum rounded once keeps them to one rounding, 2^-24."""
import numpy as np
import pytest

from tests.helpers import Problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,L,s", [(64, 3, 31 / 32), (96, 4, 26 / 32), (128, 5, 31 / 32)])
def test_small_terms_of_a_lane_are_kept(N, L, s):
    import torch

    from paper_1306_1821_gb300 import bps
    nb = 4
    nx = np.minimum(np.arange(N), N - np.arange(N))
    line = np.where(nx % L == 0, 1.0, s * 2.0 ** -12).astype(np.complex64)
    line[0] = 1 + 1j                    # kx = 0 stands alone where the others come in pairs
    spec = np.ascontiguousarray(np.broadcast_to(line[:, None, None], (N, N, N // 2 + 1)))
    spec[0, 0, 0] = 0
    pb = Problem(N, n_sub=1, n_bins=nb)
    sp = pb.gpu()
    try:
        bps.bps_set_spectrum(sp.ctx, torch.from_numpy(spec).cuda())
        _, sigma = bps.bps_sample_power(sp.ctx, nb)
    finally:
        sp.close()
    g = pb.geom
    e = g.w * (spec.real.astype(np.float64) ** 2 + spec.imag.astype(np.float64) ** 2)
    live = g.bin >= 0
    ref = g.Vc / g.Nv * np.bincount(g.bin[live], e[live], nb)
    assert np.max(np.abs(sigma / ref - 1)) < 2.0 ** -24
