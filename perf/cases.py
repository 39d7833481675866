"""The work that users of the sampler have it do, as cases that can be timed and compared.

Every case goes through the library's Python binding (paper_1306_1821_gb300.bps), as the
benchmark, the tests and the preconditioner's training do.  Surveys follow the recipe of
paper_1306_1821_gb300.inputs, made here with torch from a seed: a field of the spectrum
P(k) ~ k (1 + (k/0.02)^2)^-2, a spherical cap about the box centre with a radial selection,
Poisson counts.  Kinds of case:

  gibbs   bps_gibbs_iterate: whole iterations of the scan, and the field sample they end on
  stream  the same with every iteration's survey uploaded from pinned host memory
  batch   bps_batch_gibbs_iterate: one iteration of many chains on small grids
  hmc     bps_hmc_step: one density move
  force   bps_gradient: one force evaluation and its energies
  power   bps_sample_power: k-bin power and the spectrum draw
  bias    bps_sample_bias_norm: the survey sums and the bias and normalisation draws
  mock    bps_mock_field / _response / _counts: an artificial survey
  train   bps_mlp_train: Adam steps of the mass-preconditioner network

A chain's record (P, b, Nbar, dH, accepted) is kept as float32 rows beside the float32
field that its numbers are computed from.
"""
import functools
import math

import numpy as np
import torch

from paper_1306_1821_gb300 import bps

GRIDS = (32, 64, 96, 128, 256)
# step sizes of the repository's workloads (acceptance of about 0.8 to 0.9 on each grid)
EPS_MAX = {32: 0.15, 64: 0.1, 96: 0.08, 128: 0.06, 256: 0.05}
BOX = {32: 500.0, 64: 1000.0, 96: 1500.0, 128: 750.0, 256: 1000.0}


def listed():
    return [
        # the headline workload: 256^3, six luminosity subsamples, 20 leapfrog steps, the jump on
        dict(name="gibbs256", kind="gibbs", N=256, n_sub=6, n_bins=32, leap=20, jump=10, f_sky=0.25, iters=1),
        # the paper's own setup (Sec. 5): 128^3 with fifteen subsamples, the jump on
        dict(name="gibbs128", kind="gibbs", N=128, n_sub=15, n_bins=16, leap=10, jump=10, f_sky=0.25, iters=2),
        # the smallest survey, run as a chain of several iterations: launches and latency
        dict(name="gibbs32", kind="gibbs", N=32, n_sub=1, n_bins=16, leap=10, jump=0, f_sky=0.4, iters=8),
        # end to end: each iteration's survey comes from pinned host memory, staged one ahead
        dict(name="stream128", kind="stream", N=128, n_sub=6, n_bins=16, leap=10, jump=10, f_sky=0.25, iters=1),
        # 96 small independent surveys (32 each of 32^3, 64^3 and 96^3) in one replay
        dict(name="batch96", kind="batch", n32=32, n64=32, n96=32, n_bins=16, leap=10, jump=5),
        # one density move on a mixed-radix grid, its outcome read back, as in burn-in
        dict(name="hmc96", kind="hmc", N=96, n_sub=3, n_bins=21, leap=10, f_sky=0.5),
        # one force evaluation of a full-sky survey at the largest grid
        dict(name="force256", kind="force", N=256, n_sub=1, n_bins=32, f_sky=1.0),
        # the same at the smallest survey's grid: launches and the wait for the result
        dict(name="force32", kind="force", N=32, n_sub=1, n_bins=16, f_sky=0.4),
        # the spectrum draw alone, with a bin count that is no power of two
        dict(name="power256", kind="power", N=256, n_sub=1, n_bins=41, f_sky=0.25),
        # the bias and normalisation draws alone: six subsamples' sums and the rebuild
        dict(name="bias256", kind="bias", N=256, n_sub=6, n_bins=32, f_sky=0.25),
        # an artificial survey of the headline workload, made on the device
        dict(name="mock256", kind="mock", N=256, n_sub=6, f_sky=0.25),
        # training of the preconditioner network at its default shape and minibatch
        dict(name="train64", kind="train", n_in=32, hidden=128, n_out=64, examples=5000, batch=64, steps=100),
    ]


def draw(rng):
    kind = rng.choice(("gibbs", "gibbs", "stream", "batch", "hmc", "force", "power", "bias", "mock", "train"))
    N = rng.choice(GRIDS)
    c = dict(kind=kind)
    if kind == "train":
        return dict(c, n_in=2 * rng.randint(4, 40), hidden=rng.randint(33, 160), n_out=rng.randint(8, 64),
                    examples=rng.randint(200, 5000), batch=rng.randint(16, 96), steps=rng.randint(20, 120))
    if kind == "batch":
        return dict(c, n32=rng.randint(1, 32), n64=rng.randint(0, 32), n96=rng.randint(0, 32),
                    n_bins=rng.randint(5, 16), leap=rng.randint(4, 10), jump=rng.choice((0, 3, 5)))
    c.update(N=N, n_sub=rng.randint(1, 15 if N <= 128 else 6), f_sky=round(rng.uniform(0.15, 1.0), 3))
    if kind == "mock":
        return c
    c.update(n_bins=rng.randint(4, min(64, N // 2)))
    if kind in ("gibbs", "stream", "hmc"):
        c.update(leap=rng.randint(3, 20 if kind != "stream" else 10))
    if kind in ("gibbs", "stream"):
        c.update(jump=rng.choice((0, 4, 10)), iters=1)
    if kind == "stream":
        c.update(N=min(N, 128))
        c.update(n_bins=min(c["n_bins"], c["N"] // 2))
    return c


# ---------------------------------------------------------------- surveys
def biases(n_sub):
    return [1.0 + 0.65 * l / max(n_sub - 1, 1) for l in range(n_sub)]


def numbers(n_sub):
    return [8.0 * 16.0 ** (-l / max(n_sub - 1, 1)) for l in range(n_sub)]


def response(N, box, n_sub, f_sky, device):
    """R [n_sub][N]^3: a cap about +z times exp(-(r/r_l)^2), brighter subsamples reaching further."""
    x = (torch.arange(N, device=device, dtype=torch.float64) + 0.5) * (box / N) - box / 2
    r = torch.sqrt(x[:, None, None] ** 2 + x[None, :, None] ** 2 + x[None, None, :] ** 2)
    seen = (x[None, None, :] >= (1.0 - 2.0 * f_sky) * r) & (r <= box / 2)
    out = torch.empty((n_sub, N, N, N), device=device)
    for l in range(n_sub):
        r_l = box * (0.35 + 0.15 * l / max(n_sub - 1, 1))
        out[l] = torch.where(seen, torch.exp(-(r / r_l) ** 2), 0.0)
    return out


def shape(k):
    return k * (1.0 + (k / 0.02) ** 2) ** -2


@functools.lru_cache(None)
def amplitude(N, box):
    """A of P(k) = A shape(k) for a voxel variance of 0.5."""
    return 0.5 * box ** 3 / float((multiplicity(N) * shape(2 * np.pi / box * np.sqrt(mode_n2(N)))).sum())


def survey(N, box, n_sub, f_sky, seed):
    """(delta, counts int32, R) of one artificial survey, on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    i = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64) ** 2
    z = torch.arange(N // 2 + 1, device="cuda", dtype=torch.float64) ** 2
    P = amplitude(N, box) * shape(2 * np.pi / box * torch.sqrt(i[:, None, None] + i[None, :, None] + z[None, None, :]))
    xi = torch.randn((N, N, N), generator=g, device="cuda")
    delta = torch.fft.irfftn(torch.fft.rfftn(xi) * torch.sqrt(P * (N / box) ** 3).float(), s=(N, N, N)).contiguous()
    R = response(N, box, n_sub, f_sky, "cuda")
    counts = torch.empty((n_sub, N, N, N), device="cuda", dtype=torch.int32)
    for l, (b, nb) in enumerate(zip(biases(n_sub), numbers(n_sub))):
        counts[l] = torch.poisson(R[l] * nb * (1.0 + b * delta).clamp_min(0.0), generator=g).int()
    return delta, counts, R


def start_spectrum(N, box, n_bins, seed):
    """The true spectrum at the bin centres with a few per cent of scatter, as a chain meets it."""
    rng = np.random.Generator(np.random.PCG64(seed))
    k = 2 * np.pi / box * (np.arange(n_bins) + 0.5) * math.sqrt(3.0) * N / 2 / n_bins
    return amplitude(N, box) * shape(k) * np.exp(0.03 * rng.standard_normal(n_bins))


# ---------------------------------------------------------------- prepare
class Chain:
    """A context with its survey and state, and the buffer that the field sample is read into."""

    def __init__(self, case, seed):
        N, ns, nb = case["N"], case["n_sub"], case["n_bins"]
        box = BOX[N]
        self.case, self.seed, self.it = case, seed, 3
        self.s = bps.Sampler(N, box, ns, nb, n_leapfrog=case.get("leap", 10), eps_max=EPS_MAX[N],
                             jump=1 if case.get("jump") else 0, jump_leapfrog=case.get("jump") or 10,
                             jump_eps_max=0.15, fixed_bias_index=ns // 2, seed=seed)
        delta, counts, R = survey(N, box, ns, case["f_sky"], seed)
        delta = 0.9 * delta
        self.P, self.b, self.nbar = start_spectrum(N, box, nb, seed), biases(ns), numbers(ns)
        bps.bps_set_data(self.s.ctx, counts, R)
        bps.bps_set_state(self.s.ctx, delta, self.P, self.b, self.nbar, self.it)
        self.spec = torch.zeros((N, N, N // 2 + 1), dtype=torch.complex64, device="cuda")
        self.field = delta
        if case["kind"] == "stream":
            # pinned host arrays of the survey in the upload's own types; the first one is staged
            self.host = (counts.to(torch.int16).cpu().pin_memory().numpy().view(np.uint16), R.cpu().pin_memory().numpy())
            bps.bps_stage_data_host_u16(self.s.ctx, *self.host)


class Batch:
    """Many chains on small grids in one batch context."""

    def __init__(self, case, seed):
        rng = np.random.Generator(np.random.PCG64(seed))
        self.grid = [32] * case["n32"] + [64] * case["n64"] + [96] * case["n96"]
        self.n_sub = [1 + j % 4 for j in range(len(self.grid))]
        self.n_bins = case["n_bins"]
        box = [BOX[N] for N in self.grid]
        cfg = bps.make_config(self.n_bins, n_leapfrog=case["leap"], eps_max=0.1, jump=1 if case["jump"] else 0,
                              jump_leapfrog=case["jump"] or 5, jump_eps_max=0.05, fixed_bias_index=0, seed=seed)
        self.ctx = bps.bps_create_batch(self.grid, box, self.n_sub, cfg)
        for j, (N, ns) in enumerate(zip(self.grid, self.n_sub)):
            delta, counts, R = survey(N, box[j], ns, float(rng.uniform(0.2, 0.6)), seed + 1 + j)
            bps.bps_batch_set_chain(self.ctx, j, counts, R, 0.9 * delta, start_spectrum(N, box[j], self.n_bins, seed + j),
                                    biases(ns), numbers(ns), 3)
        self.slot = [bps.bps_batch_record_slot(self.ctx, j) for j in range(len(self.grid))]
        # the field samples that are read back: the last chain of every grid size
        self.last = {N: j for j, N in enumerate(self.grid)}
        self.field = {N: torch.zeros((N, N, N), device="cuda") for N in self.last}

    def __del__(self):
        bps.bps_destroy(self.ctx)


class Mock:
    """A context of the survey's grid, the spectrum at every |n|^2 and the output buffers."""

    def __init__(self, case, seed):
        N, ns = case["N"], case["n_sub"]
        self.case, self.seed, self.box = case, seed, BOX[N]
        self.s = bps.Sampler(N, self.box, ns, 4, seed=seed)
        self.P = mock_spectrum(N, self.box)
        self.table = mock_table(self.box, ns)
        self.b, self.nbar = biases(ns), numbers(ns)
        self.delta = torch.zeros((N, N, N), device="cuda")
        self.R = torch.zeros((ns, N, N, N), device="cuda")
        self.counts = torch.zeros((ns, N, N, N), device="cuda", dtype=torch.int32)


class Train:
    """The network at its He initialisation and a training set of features and targets."""

    def __init__(self, case, seed):
        rng = np.random.Generator(np.random.PCG64(seed))
        sizes = [case["n_in"], case["hidden"], case["hidden"], case["n_out"]]
        self.case, self.seed, self.net = case, seed, bps.MLP(sizes)
        flat = []
        for a, b in zip(sizes[:-1], sizes[1:]):
            flat += [rng.uniform(-1.0, 1.0, a * b) * math.sqrt(6.0 / a), np.zeros(b)]
        self.net.set_params(np.concatenate(flat))
        x = rng.standard_normal((case["examples"], case["n_in"])).clip(-4, 4)
        mix = rng.standard_normal((case["n_in"], case["n_out"])) / math.sqrt(case["n_in"])
        t = (0.5 * x @ mix + 0.1 * rng.standard_normal((case["examples"], case["n_out"]))).clip(-math.log(16), math.log(16))
        self.x, self.t = torch.from_numpy(x).float().cuda(), torch.from_numpy(t).float().cuda()


def prepare(case, seed):
    return {"batch": Batch, "mock": Mock, "train": Train}.get(case["kind"], Chain)(case, seed)


# ---------------------------------------------------------------- run
def float_rows(a):
    return torch.from_numpy(np.ascontiguousarray(a)).float()


def run(state):
    if isinstance(state, Batch):
        rec = bps.bps_batch_gibbs_iterate(state.ctx, 1, len(state.grid))[0]
        rows = [rec[k, : state.n_bins + 2 * ns + 2] for k, ns in zip(state.slot, state.n_sub)]
        for N, j in state.last.items():
            bps.bps_batch_get_chain(state.ctx, j, state.field[N])
        return {"chains": float_rows(np.concatenate(rows)), "fields": list(state.field.values())}
    if isinstance(state, Mock):
        ctx = state.s.ctx
        bps.bps_mock_field(ctx, state.seed, state.P, state.delta)
        bps.bps_mock_response(ctx, state.case["f_sky"], (0.0, 0.0, 1.0), state.table, state.R)
        bps.bps_mock_counts(ctx, state.seed, state.delta, state.R, state.b, state.nbar, 0, state.counts)
        return {"delta": state.delta, "R": state.R, "counts": state.counts}
    if isinstance(state, Train):
        c = state.case
        loss = state.net.train(state.x, state.t, c["batch"], c["steps"], 2e-3, state.seed)
        return {"loss": loss, "params": state.net.get_params()}
    kind, s = state.case["kind"], state.s
    if kind in ("gibbs", "stream"):
        if kind == "stream":
            bps.bps_stage_data_host_u16(s.ctx, *state.host)
        rec = bps.bps_gibbs_iterate(s.ctx, state.case["iters"], s.rec_len)
        bps.bps_get_spectrum(s.ctx, state.spec)
        return {"chain": float_rows(rec), "spectrum": state.spec}
    if kind == "hmc":
        info = bps.bps_hmc_step(s.ctx)
        bps.bps_get_spectrum(s.ctx, state.spec)
        return {"move": torch.tensor([float(v) for v in info]), "spectrum": state.spec}
    if kind == "force":
        e = bps.bps_gradient(s.ctx, state.spec)
        return {"gradient": state.spec, "prior": float(e[0]), "likelihood": float(e[1])}
    if kind == "power":
        P, sigma = bps.bps_sample_power(s.ctx, s.n_bins)
        return {"P": float_rows(P), "sigma": float_rows(sigma)}
    b, nbar, sums = bps.bps_sample_bias_norm(s.ctx, s.n_sub)
    return {"b": float_rows(b), "nbar": float_rows(nbar), "sums": float_rows(sums)}


# ---------------------------------------------------------------- work
def work(case):
    """Bytes and operations of one pass.  A force evaluation needs the field's half spectrum, a and c on
    the survey's voxels and two real transforms; a leapfrog step also updates the field and the momentum
    (4 half spectra).  What a transform holds between its axes is not counted."""
    kind = case["kind"]
    if kind == "train":
        n = case["n_in"] * case["hidden"] + case["hidden"] ** 2 + case["hidden"] * case["n_out"]
        p = n + 2 * case["hidden"] + case["n_out"]
        row = case["n_in"] + case["n_out"]
        return {"bytes": 4.0 * case["steps"] * case["batch"] * row + 24.0 * p, "flops": 6.0 * case["steps"] * case["batch"] * n}
    if kind == "batch":
        parts = [(32, case["n32"]), (64, case["n64"]), (96, case["n96"])]
        w = [scan_work(N, 2.5, case["leap"], case["jump"], 0.4) for N, n in parts for _ in range(n)]
        return {"bytes": sum(b for b, _ in w), "flops": sum(f for _, f in w)}
    N, ns, f_sky = case["N"], case["n_sub"], case["f_sky"]
    seen = math.pi / 6 * f_sky
    sc, sr = 8.0 * N * N * (N // 2 + 1), 4.0 * N ** 3
    fft = 2.5 * N ** 3 * math.log2(N ** 3)
    if kind in ("gibbs", "stream"):
        b, f = scan_work(N, ns, case["leap"], case["jump"], f_sky)
        b = b * case["iters"] + (6.0 * ns * N ** 3 if kind == "stream" else 0.0)
        return {"bytes": b + sc, "flops": f * case["iters"]}
    if kind == "hmc":
        return {"bytes": case["leap"] * (4 * sc + 2 * sr * seen) + 2 * sc, "flops": (2 * case["leap"] + 3) * fft}
    if kind == "force":
        return {"bytes": 2 * sc + 2 * sr * seen, "flops": 2 * fft}
    if kind == "power":
        return {"bytes": sc, "flops": 4.0 * N ** 3}
    if kind == "bias":
        return {"bytes": sc + 6.0 * ns * N ** 3 * seen + 2 * sr * seen, "flops": fft + 12.0 * ns * seen * N ** 3}
    return {"bytes": sr + 2 * ns * sr, "flops": 2 * fft + 100.0 * ns * seen * N ** 3}


def scan_work(N, ns, leap, jump, f_sky):
    """(bytes, operations) of one Gibbs iteration."""
    seen = math.pi / 6 * f_sky
    sc, sr = 8.0 * N * N * (N // 2 + 1), 4.0 * N ** 3
    fft = 2.5 * N ** 3 * math.log2(N ** 3)
    ac, data = 2 * sr * seen, 6.0 * ns * N ** 3 * seen
    grads = jump + 1 if jump else 0
    b = leap * (4 * sc + ac) + sc + grads * (sc + ac) + sc + data + ac
    return b, (2 * leap + 3 + 2 * grads + 1) * fft + 12.0 * ns * seen * N ** 3


# ---------------------------------------------------------------- exact values, in 64 bits
def mode_n2(N):
    i = np.fft.fftfreq(N, 1.0 / N) ** 2
    z = np.arange(N // 2 + 1, dtype=np.float64) ** 2
    return i[:, None, None] + i[None, :, None] + z[None, None, :]


def mode_bins(N, n_bins):
    """Bin of every half-spectrum mode (linear in |n| over (0, sqrt(3) N/2]); -1 for k = 0."""
    n2 = mode_n2(N)
    m = np.minimum(np.floor(n_bins * np.sqrt(n2) / (math.sqrt(3.0) * N / 2.0)).astype(np.int64), n_bins - 1)
    m[0, 0, 0] = -1
    return m


def multiplicity(N):
    w = np.full(N // 2 + 1, 2.0)
    w[0] = w[-1] = 1.0
    return w


def mulhilo(a, b):
    """High and low halves of 64 x 64-bit products, from 32-bit halves."""
    s, low = np.uint64(32), np.uint64(0xFFFFFFFF)
    b0, b1 = np.uint64(b & 0xFFFFFFFF), np.uint64(b >> 32)
    a0, a1 = a & low, a >> s
    p00, p01, p10 = a0 * b0, a0 * b1, a1 * b0
    mid = (p00 >> s) + (p01 & low) + (p10 & low)
    return a1 * b1 + (p01 >> s) + (p10 >> s) + (mid >> s), a * np.uint64(b)


def philox(c0, c1, c2, c3, key):
    """Philox4x64-10 (Salmon et al., SC'11) of counters (c0[], c1, c2, c3) and key (key, 0)."""
    x0 = np.asarray(c0, dtype=np.uint64)
    x1, x2, x3 = (np.full_like(x0, c) for c in (c1, c2, c3))
    k0, k1, top = key, 0, (1 << 64) - 1
    with np.errstate(over="ignore"):
        for _ in range(10):
            h0, l0 = mulhilo(x0, 0xD2E7470EE14C6C93)
            h1, l1 = mulhilo(x2, 0xCA5A826395121157)
            x0, x1, x2, x3 = h1 ^ x1 ^ np.uint64(k0), l1, h0 ^ x3 ^ np.uint64(k1), l0
            k0, k1 = (k0 + 0x9E3779B97F4A7C15) & top, (k1 + 0xBB67AE8584CAA73B) & top
    return x0, x1, x2, x3


def uniform(w):
    return ((np.asarray(w, dtype=np.uint64) >> np.uint64(12)).astype(np.float64) + 0.5) * 2.0 ** -52


def normal(wa, wb):
    return np.sqrt(-2.0 * np.log(uniform(wa))) * np.cos(2.0 * np.pi * uniform(wb))


def voxel_normals(seed, iteration, stage, n):
    """Element i from block i // 8: Box-Muller of the two float32 uniforms in word (i % 8) // 2."""
    out = np.empty((n // 8, 8))
    one, half = np.float32(2.0 ** -32), np.float32(2.0 ** -33)
    for j, w in enumerate(philox(np.arange(n // 8), iteration, stage, 0, seed)):
        u1 = ((w & np.uint64(0xFFFFFFFF)).astype(np.uint32).astype(np.float32) * one + half).astype(np.float64)
        u2 = ((w >> np.uint64(32)).astype(np.uint32).astype(np.float32) * one + half).astype(np.float64)
        r = np.sqrt(-2.0 * np.log(u1))
        out[:, 2 * j], out[:, 2 * j + 1] = r * np.cos(2 * np.pi * u2), r * np.sin(2 * np.pi * u2)
    return out.reshape(-1)


def rfft(x):
    return torch.fft.rfftn(x)


def irfft(x, N):
    return torch.fft.irfftn(x, s=(N, N, N))


class Model:
    """One survey's posterior in 64 bits: the local fields, the mode tables and the force."""

    def __init__(self, case, seed):
        N, ns = case["N"], case["n_sub"]
        self.N, self.box = N, BOX[N]
        delta, counts, R = survey(N, self.box, ns, case["f_sky"], seed)
        self.R, self.counts, self.b, self.nbar = R, counts, biases(ns), numbers(ns)
        self.d = rfft((0.9 * delta).double())
        self.d[0, 0, 0] = 0
        self.P = start_spectrum(N, self.box, case["n_bins"], seed)
        self.vc = (self.box / N) ** 3
        self.bins = mode_bins(N, case["n_bins"])
        self.a, self.c = torch.zeros((N, N, N), device="cuda", dtype=torch.float64), 0.0
        for l in range(ns):
            self.a += self.b[l] ** 2 * self.nbar[l] * R[l].double()
            self.c = self.c + self.b[l] * (counts[l].double() - self.nbar[l] * R[l].double())
        il = np.where(self.bins >= 0, self.vc / self.P[self.bins], 0.0)
        self.il = torch.from_numpy(il).cuda()
        self.w = torch.from_numpy(multiplicity(N)).cuda()
        self.live = torch.from_numpy(self.bins >= 0).cuda()

    def force(self, d):
        delta = irfft(d, self.N)
        return (d * self.il + rfft(self.a * delta - self.c)) * self.live, delta

    def norm(self, x, by):
        return float((self.w * (x.real ** 2 + x.imag ** 2) * by).sum()) / self.N ** 3

    def binned(self, x):
        """sigma_m = V_cell / N^3 sum over the bin of |x|^2."""
        e = (self.w * (x.real ** 2 + x.imag ** 2)).cpu().numpy()[self.bins >= 0]
        return self.vc / self.N ** 3 * np.bincount(self.bins[self.bins >= 0], e, len(self.P))


def exact_move(m, case, seed, it):
    w = philox([0], it, 2, 0, seed)
    eps, u = EPS_MAX[m.N] * float(uniform(w[0])[0]), float(uniform(w[1])[0])
    M = m.il + m.a.mean()
    xi = torch.from_numpy(voxel_normals(seed, it, 1, m.N ** 3).reshape(m.N, m.N, m.N)).cuda()
    p, d = torch.sqrt(M) * rfft(xi) * m.live, m.d.clone()

    def energy(d, p, delta):
        return 0.5 * m.norm(p, 1.0 / M) + 0.5 * m.norm(d, m.il) + 0.5 * float((m.a * delta ** 2 - 2.0 * m.c * delta).sum())

    g, delta = m.force(d)
    h0 = energy(d, p, delta)
    p = p - 0.5 * eps * g
    for i in range(case["leap"]):
        d = d + eps * p / M * m.live
        g, delta = m.force(d)
        p = p - (0.5 * eps if i == case["leap"] - 1 else eps) * g
    dH = energy(d, p, delta) - h0
    ok = math.log(u) < -dH
    # the energy difference is what remains of two sums of the size of N^3: its last digits are one
    # sample of their rounding, so only the field is given in 64 bits
    return {"move": None, "spectrum": d if ok else m.d}


def exact_spectrum_draw(m, case, seed, it):
    """P_m = sigma_m / (2 Gamma(beta_m / 2)), the Gamma variate by Marsaglia and Tsang (2000)."""
    sigma = m.binned(m.d)
    w = np.broadcast_to(multiplicity(m.N), m.bins.shape)
    modes = np.bincount(m.bins[m.bins >= 0], w[m.bins >= 0], len(sigma))
    P = np.zeros(len(sigma))
    for k, n in enumerate(modes):
        half = 0.5 * n                       # beta = n + 2 alpha - 2 with alpha = 1
        a = half + 1.0 if half < 1.0 else half
        d = a - 1.0 / 3.0
        for j in range(64):
            q = philox([k], it, 3, j, seed)
            z = float(normal(q[0], q[1])[0])
            t = 1.0 + z / math.sqrt(9.0 * d)
            if t > 0 and math.log(float(uniform(q[2])[0])) < 0.5 * z * z + d - d * t ** 3 + d * math.log(t ** 3):
                break
        x = d * t ** 3
        if half < 1.0:
            x *= float(uniform(philox([k], it, 3, 0, seed)[3])[0]) ** (1.0 / half)
        P[k] = sigma[k] / (2.0 * x)
    return {"P": P, "sigma": sigma}


def exact_bias(m, case, seed, it):
    delta = irfft(m.d, m.N)
    sums, b = np.zeros((case["n_sub"], 3)), np.array(m.b)
    for l in range(case["n_sub"]):
        R, n = m.R[l].double(), m.counts[l].double()
        sums[l] = [float((n * delta).sum()), float((R * delta).sum()), float((R * delta ** 2).sum())]
        if l != case["n_sub"] // 2:
            c = m.nbar[l] * sums[l, 2]
            q = philox([l], it, 4, 0, seed)
            b[l] = (sums[l, 0] - m.nbar[l] * sums[l, 1]) / c + float(normal(q[0], q[1])[0]) / math.sqrt(c)
    return {"b": b, "nbar": None, "sums": sums}


def mock_spectrum(N, box):
    k = 2 * np.pi / box * np.sqrt(np.arange(3 * (N // 2) ** 2 + 1, dtype=np.float64))
    return amplitude(N, box) * shape(k)


def mock_table(box, n_sub, n_r=2049):
    r = np.arange(n_r) * (box / 2 / (n_r - 1))
    return np.stack([np.exp(-(r / (box * (0.35 + 0.15 * l / max(n_sub - 1, 1)))) ** 2) for l in range(n_sub)])


def exact_mock(case, seed):
    N, ns = case["N"], case["n_sub"]
    box = BOX[N]
    amp = np.sqrt(mock_spectrum(N, box) * (N / box) ** 3)
    xi = torch.from_numpy(voxel_normals(seed, 0, 8, N ** 3).reshape(N, N, N)).cuda()
    delta = irfft(rfft(xi) * torch.from_numpy(amp[mode_n2(N).astype(np.int64)]).cuda(), N)
    x = (torch.arange(N, device="cuda", dtype=torch.float64) + 0.5) * (box / N) - box / 2
    r = torch.sqrt(x[:, None, None] ** 2 + x[None, :, None] ** 2 + x[None, None, :] ** 2)
    seen = (x[None, None, :] / r >= 1.0 - 2.0 * case["f_sky"]) & (r <= box / 2)
    table = torch.from_numpy(mock_table(box, ns)).cuda()
    t = (r / (box / 2) * (table.shape[1] - 1)).clamp_max(table.shape[1] - 1.0)
    j = t.floor().clamp_max(table.shape[1] - 2.0).long()
    R = torch.stack([torch.where(seen, table[l][j] * (1.0 - (t - j)) + table[l][j + 1] * (t - j), 0.0) for l in range(ns)])
    return {"delta": delta, "R": R, "counts": None}


def exact(case, seed):
    """None for whole scans (their random variates come from rejection samplers on top of every earlier
    stage) and for training (operands rounded to 16 bits: its path has no 64-bit value)."""
    kind = case["kind"]
    if kind == "mock":
        return exact_mock(case, seed)
    if kind in ("hmc", "force", "power", "bias"):
        m = Model(case, seed)
        if kind == "hmc":
            return exact_move(m, case, seed, 3)
        if kind == "power":
            return exact_spectrum_draw(m, case, seed, 3)
        if kind == "bias":
            return exact_bias(m, case, seed, 3)
        g, delta = m.force(m.d)
        return {"gradient": g, "prior": 0.5 * m.norm(m.d, m.il), "likelihood": 0.5 * float((m.a * delta ** 2 - 2.0 * m.c * delta).sum())}
    return None
