"""The FP32 screens of the mock kernels against the FP64 definitions (oracle/mock.py), where they
can go wrong: counts of every mean up to the limit and beyond, voxels without response, special
values, and arrays that start off a 16-byte boundary; responses of caps whose edge and radius pass
through voxel centres.  Counts and responses are bit-exact."""
import numpy as np
import pytest

from oracle import mock

pytestmark = pytest.mark.gpu


def place(a, offset):
    """`a` on the GPU, `offset` elements after an aligned start."""
    import torch
    t = torch.empty(a.size + offset, dtype=torch.from_numpy(a).dtype, device="cuda")
    t[offset:] = torch.from_numpy(a.ravel()).cuda()
    return t[offset:]


@pytest.mark.parametrize("offset", [0, 1])
def test_counts_of_every_mean(offset):
    import torch

    from paper_1306_1821_gb300 import bps
    N, n_sub = 32, 3
    rng = np.random.default_rng(5)
    nv = N ** 3
    d = rng.uniform(-1.5, 1.5, nv).astype(np.float32)
    R = np.exp(rng.uniform(np.log(1e-7), np.log(3000.0), (n_sub, nv))).astype(np.float32)
    R[1] = rng.uniform(0.0, 4.0, nv)
    R[2, ::3] = 0.0
    d[:8] = [np.inf, -np.inf, np.nan, 0.0, -1.0, 1e30, -1e30, 1e-30]
    R[:, :4] = [0.0, 1e-45, 1.0, 32.0]
    b, nbar = [1.0, 1.3, 0.7], [1.0, 7.9, 2.0]
    s = bps.Sampler(N, 500.0, n_sub, 4)
    try:
        c = place(np.zeros(n_sub * nv, dtype=np.int32), offset)
        bps.bps_mock_counts(s.ctx, 99, place(d, offset), place(R, offset), b, nbar, 0, c)
        got = c.cpu().numpy().reshape(n_sub, nv)
    finally:
        s.close()
    for l in range(n_sub):
        with np.errstate(invalid="ignore", over="ignore"):
            t = 1.0 + b[l] * d.astype(np.float64)
            lam = (R[l].astype(np.float64) * nbar[l]) * np.where(t > 0.0, t, 0.0)
        ok = lam <= 4096.0
        ref = np.full(nv, 65536, dtype=np.int64)
        ref[ok] = mock.poisson_counts(lam[ok], 99, l, index=np.nonzero(ok)[0])
        assert np.array_equal(got[l], ref), np.nonzero(got[l] != ref)[0][:10]
    assert (got == 65536).any() and (got > 1000).any()


@pytest.mark.parametrize("N,axis,f_sky,offset", [(32, (0.0, 0.0, 1.0), 0.5, 0), (64, (1.0, 1.0, 0.0), 0.5, 0),
                                                 (32, (0.3, -0.4, 0.87), 1.0, 1), (96, (0.0, -2.0, 0.0), 0.1, 0)])
def test_response_at_the_edges_of_the_cap(N, axis, f_sky, offset):
    from paper_1306_1821_gb300 import bps
    box, n_sub = 750.0, 2
    table = np.random.default_rng(1).uniform(0.0, 1.0, (n_sub, 33))
    s = bps.Sampler(N, box, n_sub, 4)
    try:
        R = place(np.zeros(n_sub * N ** 3, dtype=np.float32), offset)
        bps.bps_mock_response(s.ctx, f_sky, axis, table, R)
        got = R.cpu().numpy().reshape(n_sub, N, N, N)
    finally:
        s.close()
    ref = mock.response(N, box, f_sky, axis, table, box / 2)
    assert np.array_equal(got.view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("N,n_r", [(64, 363), (128, 179), (256, 282), (64, 1 << 20), (128, 16385), (256, 4501), (256, 7000), (256, 65537)])
def test_response_of_rough_tables(N, n_r):
    """Random tables of many radii: whatever rounding leaves of a voxel's place in the table, the
    value comes from the segment of the FP64 definition (a neighbouring one gives another slope)."""
    from paper_1306_1821_gb300 import bps
    box, axis = 750.0, (0.0, 0.0, 1.0)
    table = np.random.default_rng(2).uniform(0.0, 1.0, (1, n_r))
    s = bps.Sampler(N, box, 1, 4)
    try:
        R = place(np.zeros(N ** 3, dtype=np.float32), 0)
        bps.bps_mock_response(s.ctx, 1.0, axis, table, R)
        got = R.cpu().numpy().reshape(1, N, N, N)
    finally:
        s.close()
    ref = mock.response(N, box, 1.0, axis, table, box / 2)
    assert np.array_equal(got.view(np.uint32), ref.view(np.uint32)), int((got != ref).sum())


@pytest.mark.parametrize("box", [1e160, 1e150, 1e-150, 1e-158, 1e-170])
def test_response_of_boxes_whose_squares_leave_fp64(box):
    """Squared distances that overflow, lose bits or vanish in FP64 decide the radius cut of the
    definition; the kernel follows it there too."""
    from paper_1306_1821_gb300 import bps
    N, axis = 32, (0.3, -0.4, 0.87)
    table = np.random.default_rng(3).uniform(0.5, 1.0, (1, 17))
    s = bps.Sampler(N, box, 1, 4)
    try:
        R = place(np.zeros(N ** 3, dtype=np.float32), 0)
        bps.bps_mock_response(s.ctx, 0.5, axis, table, R)
        got = R.cpu().numpy().reshape(1, N, N, N)
    finally:
        s.close()
    with np.errstate(over="ignore", invalid="ignore"):
        ref = mock.response(N, box, 0.5, axis, table, box / 2)
    assert np.array_equal(got.view(np.uint32), ref.view(np.uint32)), int((got != ref).sum())


def test_counts_of_factors_far_from_one():
    """lambda of ordinary size from factors that FP32 cannot hold, and voxels without response whose
    field overflows: the counts are those of the FP64 definition."""
    from paper_1306_1821_gb300 import bps
    N, n_sub = 32, 2
    nv = N ** 3
    rng = np.random.default_rng(8)
    d = rng.uniform(0.0, 1e7, nv).astype(np.float32)
    d[:2] = [1e20, -1e20]
    R = np.zeros((n_sub, nv), dtype=np.float32)
    R[0] = rng.uniform(1e37, 3e38, nv)
    b, nbar = [1.0, 1e300], [1e-44, 1.0]
    s = bps.Sampler(N, 500.0, n_sub, 4)
    try:
        c = place(np.zeros(n_sub * nv, dtype=np.int32), 0)
        bps.bps_mock_counts(s.ctx, 7, place(d, 0), place(R, 0), b, nbar, 0, c)
        got = c.cpu().numpy().reshape(n_sub, nv)
    finally:
        s.close()
    for l in range(n_sub):
        with np.errstate(invalid="ignore", over="ignore"):
            lam = mock.mean_counts(d, R[l], b[l], nbar[l])
        ok = lam <= 4096.0
        ref = np.full(nv, 65536, dtype=np.int64)
        ref[ok] = mock.poisson_counts(lam[ok], 7, l, index=np.nonzero(ok)[0])
        assert np.array_equal(got[l], ref), (l, int((got[l] != ref).sum()))
