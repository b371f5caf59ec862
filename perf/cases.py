"""The work that is measured: operator calls and solves over the sizes this framework is used at.

A case is a dict of plain values.  Its "kind" says what it stands for:

* "slice"  - a 2D Cartesian slice with a dense Maxwell basis (forward, adjoint, the
             forward+adjoint pair of a SENSE normal operator, or the Jacobian pair that one
             IRGN CG iteration applies);
* "radial" - the same operators on a golden-angle radial trajectory (Kaiser-Bessel gridding);
* "volume" - the same operators on a 3D volume with a Tucker-factored basis;
* "exam"   - a batch of mixed 2D slices, recorded once and replayed per exam;
* "admm"   - TV-regularised image reconstruction (MPI-L) of one slice, or of several frames of it.

Sensitivity estimation (MPI-BL) is measured by the Jacobian pairs, which are all of its work but a few
vector updates: the whole call's maps and image share a free scale and are too loosely determined by the
data for two roundings of the same arithmetic to agree closely.

Every state owns its context, plan and basis, as a program that reconstructs one scan does.
All inputs are synthetic and made from the seed.
"""

import math

import numpy as np
import torch

import paper_2008_09042_gb300 as mp

DEV = "cuda"
FFT_LENGTHS = (48, 64, 96, 128, 192, 256, 320)
RADIAL_N = (32, 48, 64, 96, 128, 160, 256)  # grids of twice these lengths are supported
EXAM_SIZES = (128, 192, 256, 320)
EXAM_COILS = (8, 16, 32)
EXAM_Q = {128: 64, 192: 96, 256: 128, 320: 160}


def listed():
    return [
        # the smallest call: a 64 x 64 calibration-size slice, where latency is all that counts
        dict(name="slice64_forward", kind="slice", op="forward", ny=64, nx=64, C=4, q=32, mask="lines", R=3, acs=16,
             prec="fp32"),
        # the ordinary 2D slice of an iterative SENSE reconstruction: one normal-operator application
        dict(name="slice256_pair", kind="slice", op="pair", ny=256, nx=256, C=16, q=128, mask="points", R=6, acs=24,
             prec="fp32"),
        # the same on the 320 x 320 brain-slice shape with every second line, BF16 basis
        dict(name="slice320_pair_bf16", kind="slice", op="pair", ny=320, nx=320, C=16, q=100, mask="lines", R=2,
             acs=16, prec="bf16"),
        # one CG iteration's operators of the sensitivity estimation on the ordinary slice
        dict(name="slice256_jacobian", kind="slice", op="jacobian", ny=256, nx=256, C=16, q=128, mask="points", R=6,
             acs=24, prec="fp32"),
        # a rectangular slice with an odd coil count and an odd basis size, BF16 basis
        dict(name="slice128x192_jacobian_bf16", kind="slice", op="jacobian", ny=128, nx=192, C=9, q=51,
             mask="points", R=4, acs=16, prec="bf16"),
        # the radial slice: one normal-operator application
        dict(name="radial256_pair", kind="radial", op="pair", n=256, C=12, q=96, spokes=64, readout=512, W=6,
             prec="fp32"),
        # a small radial slice (real-time imaging sizes: few spokes, odd coil count): one CG iteration's operators
        dict(name="radial96_jacobian", kind="radial", op="jacobian", n=96, C=5, q=24, spokes=21, readout=192, W=4,
             prec="fp32"),
        # the 3D volume with a Tucker basis: one normal-operator application
        dict(name="volume_pair", kind="volume", op="pair", nz=96, ny=128, nx=128, C=32, q=256, r1=32, r2=40, r3=40,
             R=8, acs=24, prec="fp32"),
        # the same volume: one CG iteration's operators of the sensitivity estimation
        dict(name="volume_jacobian", kind="volume", op="jacobian", nz=96, ny=128, nx=128, C=32, q=256, r1=32, r2=40,
             r3=40, R=8, acs=24, prec="fp32"),
        # an exam of 64 slices of four sizes and three coil arrays, replayed as one graph
        dict(name="exam64_pair", kind="exam", slices=64, prec="fp32"),
        # image reconstruction of the ordinary slice, whole call
        dict(name="admm256", kind="admm", frames=1, n=256, C=16, q=128, mask="points", R=6, acs=24, n_outer=50,
             n_cg=5, n_tv=10, prec="fp32"),
        # dynamic reconstruction of four frames of a small slice, each with its own sampling, whole call
        dict(name="dynamic128", kind="admm", frames=4, n=128, C=8, q=64, mask="lines", R=2, acs=16, n_outer=20,
             n_cg=5, n_tv=10, prec="fp32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["slice"] * 5 + ["radial"] * 3 + ["volume"] * 2 + ["exam", "admm", "admm"])
    prec = rng.choice(["fp32", "fp32", "bf16"])
    op = rng.choice(["forward", "adjoint", "pair", "jacobian"])
    if kind == "slice":
        ny, nx = rng.choice(FFT_LENGTHS), rng.choice(FFT_LENGTHS)
        mask = rng.choice(["lines", "points"])
        return dict(kind=kind, op=op, ny=ny, nx=nx, C=_log_int(rng, 1, 32), q=_log_int(rng, 6, 160), mask=mask,
                    R=rng.randint(2, 3) if mask == "lines" else rng.randint(2, 8), acs=rng.choice([8, 12, 16]),
                    prec=prec)
    if kind == "radial":
        n = rng.choice(RADIAL_N)
        return dict(kind=kind, op=op, n=n, C=_log_int(rng, 1, 20), q=_log_int(rng, 4, 128),
                    spokes=_log_int(rng, 8, 96), readout=2 * n, W=rng.randint(3, 8), prec=prec)
    if kind == "volume":
        nz, ny, nx = rng.choice([32, 64, 96]), rng.choice([64, 96, 128]), rng.choice([64, 96, 128])
        return dict(kind=kind, op=op, nz=nz, ny=ny, nx=nx, C=_log_int(rng, 2, 32), q=_log_int(rng, 12, 256),
                    r1=rng.randint(3, 16) * 2, r2=rng.randint(3, 20) * 2, r3=rng.randint(6, 40), R=rng.randint(3, 8),
                    acs=rng.choice([8, 12, 16]), prec=prec)
    if kind == "exam":
        return dict(kind=kind, slices=_log_int(rng, 4, 40), prec=prec)
    mask, frames = rng.choice(["lines", "points"]), rng.choice([1, 1, rng.randint(2, 6)])
    return dict(kind=kind, frames=frames, n=rng.choice([64, 96, 128, 192]), C=rng.randint(4, 12), q=rng.randint(12, 64),
                mask=mask, R=2 if mask == "lines" else rng.randint(2, 4), acs=16, n_outer=rng.randint(10, 40 // frames + 8),
                n_cg=rng.randint(3, 6), n_tv=rng.randint(5, 10), prec="fp32")


# ------------------------------------------------------------------ inputs


def _gen(seed, what):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + what) % (1 << 62))
    return g


def _noise(g, *shape):
    """Complex Gaussian values of unit variance (complex64)."""
    return torch.randn(*shape, dtype=torch.complex64, device=DEV, generator=g)


def _coefficients(g, C, q):
    """Coil coefficients whose variance falls with the basis index, as those of an SVD-ordered basis do."""
    return _noise(g, C, q) / torch.sqrt(1.0 + torch.arange(q, device=DEV, dtype=torch.float32))


def _coil_ring(g, dims, C):
    """Sensitivity maps of C coils around the slice, each falling off from its place with a phase of its own (C, N)."""
    pos = torch.meshgrid(*[(torch.arange(n, device=DEV) - n / 2) / (n / 2) for n in dims], indexing="ij")
    turn, phase = torch.rand(1, device=DEV, generator=g), 2 * math.pi * torch.rand(C, device=DEV, generator=g)
    ang = 2 * math.pi * (torch.arange(C, device=DEV) + turn) / C
    dy, dx = (p[None] - 1.2 * f(ang)[:, None, None] for p, f in zip(pos, (torch.sin, torch.cos)))
    mag = 1.0 / (1.0 + (dy ** 2 + dx ** 2) / 0.5)
    return torch.polar(mag, phase[:, None, None] + torch.atan2(dy, dx) * 0.25).reshape(C, -1)


def _phantom(g, dims):
    """A piecewise-constant density: a background ellipse and eight random ones."""
    axes = [(torch.arange(n, device=DEV) - n / 2) / (n / 2) for n in dims]
    pos = torch.meshgrid(*axes, indexing="ij")
    img = torch.where(sum((x / 0.85) ** 2 for x in pos) <= 1.0, 0.2, 0.0)
    for _ in range(8):
        u = torch.rand(2 * len(dims) + 1, device=DEV, generator=g)
        d2 = sum(((x - (u[i] - 0.5)) / (0.1 + 0.4 * u[len(dims) + i])) ** 2 for i, x in enumerate(pos))
        img = torch.where(d2 <= 1.0, 0.1 + 0.9 * u[-1], img)
    return img.reshape(-1).to(torch.complex64)


def _low_modes(n, count):
    k = np.arange(n) - n // 2
    return k[np.argsort(np.abs(k) + 0.25 * (k < 0), kind="stable")[:count]]


def _dense_basis(g, ny, nx, q):
    """(q, N) orthonormal smooth fields: the q slowest Fourier modes times one smooth random phase."""
    ky, kx = np.meshgrid(np.arange(ny) - ny // 2, np.arange(nx) - nx // 2, indexing="ij")
    order = np.lexsort((kx.ravel(), ky.ravel(), (ky ** 2 + kx ** 2).ravel()))[:q]
    ky = torch.from_numpy(ky.ravel()[order].astype(np.float32)).to(DEV)
    kx = torch.from_numpy(kx.ravel()[order].astype(np.float32)).to(DEV)
    y = torch.arange(ny, device=DEV, dtype=torch.float32) / ny
    x = torch.arange(nx, device=DEV, dtype=torch.float32) / nx
    c = torch.randn(4, device=DEV, generator=g)
    env = c[0] * torch.cos(2 * math.pi * y + c[1])[:, None] + c[2] * torch.cos(2 * math.pi * x + c[3])[None, :]
    ph = 2 * math.pi * ((ky[:, None] * y)[:, :, None] + (kx[:, None] * x)[:, None, :]) + env
    return torch.polar(torch.full_like(ph, 1.0 / math.sqrt(ny * nx)), ph).reshape(q, ny * nx)


def _tucker_basis(g, dims, ranks, q):
    """Core (r1, r2, r3, q) and factors (n_k, r_k) with orthonormal columns, as numpy arrays."""
    factors = []
    for n, r in zip(dims, ranks):
        t = np.arange(n)
        env = float(torch.randn(1, device=DEV, generator=g)) * np.cos(2 * np.pi * t / n)
        f = np.exp(1j * (2 * np.pi * np.outer(t, _low_modes(n, r)) / n + env[:, None])) / math.sqrt(n)
        factors.append(f.astype(np.complex64))
    core = _noise(g, *ranks, q) / math.sqrt(ranks[0] * ranks[1] * ranks[2])
    return core.cpu().numpy(), factors


def _point_mask(seed, n0, n1, R, acs):
    """round(n0 n1 / R) positions: the central acs x acs box, the rest denser towards the centre."""
    rng = np.random.default_rng(seed)
    k0 = (np.arange(n0) - n0 // 2) / (n0 / 2.0)
    k1 = (np.arange(n1) - n1 // 2) / (n1 / 2.0)
    w = 1.0 / (1.0 + 1.5 * np.sqrt(k0[:, None] ** 2 + k1[None, :] ** 2)) ** 2
    score = np.log(w) + rng.gumbel(size=(n0, n1))
    b0, b1 = min(acs, n0), min(acs, n1)
    score[n0 // 2 - b0 // 2:n0 // 2 - b0 // 2 + b0, n1 // 2 - b1 // 2:n1 // 2 - b1 // 2 + b1] = np.inf
    count = max(int(round(n0 * n1 / R)), b0 * b1)
    mask = np.zeros(n0 * n1, dtype=bool)
    mask[np.argpartition(-score.ravel(), count - 1)[:count]] = True
    return mask.reshape(n0, n1)


def _line_mask(seed, ny, nx, R, acs):
    """round(ny / R) whole lines: the acs central ones, the rest denser towards the centre."""
    rng = np.random.default_rng(seed)
    k = np.arange(ny) - ny // 2
    score = 2.0 * np.log(1.0 - np.abs(k) / (ny / 2.0 + 1.0)) + rng.gumbel(size=ny)
    score[ny // 2 - acs // 2:ny // 2 - acs // 2 + acs] = np.inf
    mask = np.zeros((ny, nx), dtype=bool)
    mask[np.argsort(-score)[:max(int(round(ny / R)), acs)]] = True
    return mask


def _slice_mask(case, seed, ny, nx):
    make = _line_mask if case["mask"] == "lines" else _point_mask
    return np.flatnonzero(make(seed, ny, nx, case["R"], case["acs"])).astype(np.int32)


def _slice_samples(case, ny, nx):
    if case["mask"] == "lines":
        return max(int(round(ny / case["R"])), case["acs"]) * nx
    return max(int(round(ny * nx / case["R"])), min(case["acs"], ny) * min(case["acs"], nx))


def _trajectory(seed, spokes, readout):
    """Golden-angle spokes through the k-space centre, rad/pixel, with a random first angle."""
    theta = np.random.default_rng(seed).uniform(0, math.pi) + np.arange(spokes) * math.pi * (math.sqrt(5.0) - 1) / 2
    r = math.pi * (np.arange(readout) - readout // 2) / (readout / 2.0)
    return np.stack([np.outer(np.cos(theta), r).ravel(), np.outer(np.sin(theta), r).ravel()], 1).astype(np.float32)


def _exam_layout(case):
    """(n, C, R) of each slice; the smallest exams still mix sizes and coil arrays."""
    return [(EXAM_SIZES[i % 4], EXAM_COILS[(i // 4 + i) % 3], 4 + (7 * i) % 5) for i in range(case["slices"])]


def _dims(case):
    if case["kind"] == "slice":
        return (case["ny"], case["nx"])
    if case["kind"] == "volume":
        return (case["nz"], case["ny"], case["nx"])
    return (case["n"], case["n"])


def _inputs(case, seed):
    """Everything that is given: sampling, basis and the operator's or solver's arguments."""
    kind = case["kind"]
    if kind == "exam":
        bases = {n: _dense_basis(_gen(seed, n), n, n, EXAM_Q[n]) for n in EXAM_SIZES[:case["slices"]]}
        slices = []
        for i, (n, C, R) in enumerate(_exam_layout(case)):
            g = _gen(seed, 1000 + i)
            idx = np.flatnonzero(_point_mask(seed * 64 + i, n, n, R, 24)).astype(np.int32)
            slices.append(dict(n=n, idx=idx, alpha=_coefficients(g, C, EXAM_Q[n]), p=_phantom(g, (n, n))))
        return dict(bases=bases, slices=slices)
    dims, C, q = _dims(case), case["C"], case["q"]
    N = int(np.prod(dims))
    g = _gen(seed, 1)
    d = dict(dims=dims)
    if kind == "radial":
        d["traj"] = _trajectory(seed, case["spokes"], case["readout"])
        M = len(d["traj"])
    elif kind == "volume":
        plane = _point_mask(seed, dims[0], dims[1], case["R"], case["acs"])
        d["idx"] = np.flatnonzero(np.repeat(plane[:, :, None], dims[2], axis=2)).astype(np.int32)
        M = len(d["idx"])
    else:
        d["idx"] = _slice_mask(case, seed, *dims)
        M = len(d["idx"])
    if kind == "volume":
        d["core"], d["factors"] = _tucker_basis(g, dims, (case["r1"], case["r2"], case["r3"]), q)
    else:
        d["U"] = _dense_basis(g, dims[0], dims[1], q)
    d["alpha"], d["p"] = _coefficients(g, C, q), _phantom(g, dims)
    if kind == "admm":
        # a ring of coils, data with 30 dB of noise, the noise ball that MPI-L is constrained to
        d["alpha"] = _coil_ring(g, dims, C) @ d["U"].conj().T
        maps = _maps(d, d["alpha"], torch.complex64)
        d["frames"], ys = [d["idx"]], []
        for t in range(1, case["frames"]):
            d["frames"].append(_slice_mask(case, seed + 7919 * t, *dims))
        for t, idx in enumerate(d["frames"]):  # the image fades from frame to frame
            ys.append(_forward(_Cartesian(dims, idx), maps, d["p"] * (1.0 - 0.1 * t)))
        clean = torch.stack(ys)
        sigma = float(clean.abs().square().mean().sqrt()) / 10.0 ** 1.5
        d["y"] = clean + sigma * _noise(g, case["frames"], C, M)
        d["eps"] = np.full((case["frames"], C), sigma * math.sqrt(M))
    elif case["op"] == "adjoint":
        d["y"] = _noise(g, C, M)
    elif case["op"] == "jacobian":
        d["dp"], d["dalpha"] = _noise(g, N), _coefficients(g, C, q)
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    ctx = mp.Context(0)
    if case["kind"] == "exam":
        bases = {n: mp.Basis(ctx, U) for n, U in d["bases"].items()}
        count = [(s["alpha"].shape[0] * len(s["idx"]), s["n"] ** 2) for s in d["slices"]]
        # one buffer for the exam's k-space data and one for its images; every slice has its part
        offs = np.cumsum([0] + [m + m % 2 for m, _ in count]), np.cumsum([0] + [n for _, n in count])
        y = torch.zeros(int(offs[0][-1]), dtype=torch.complex64, device=DEV)
        x = torch.zeros(int(offs[1][-1]), dtype=torch.complex64, device=DEV)
        parts = []
        for i, s in enumerate(d["slices"]):
            C, M = s["alpha"].shape[0], len(s["idx"])
            parts.append(dict(plan=mp.Plan(ctx, (s["n"], s["n"]), sample_idx=s["idx"]), basis=bases[s["n"]],
                              alpha=s["alpha"], p=s["p"], y=y[int(offs[0][i]):int(offs[0][i]) + C * M].view(C, M),
                              x=x[int(offs[1][i]):int(offs[1][i + 1])]))
        return dict(case=case, ctx=ctx, batch=mp.Batch(ctx, parts, kind="pair", prec=case["prec"]), y=y, x=x)
    if "traj" in d:
        plan = mp.Plan(ctx, d["dims"], traj=d["traj"], kb_width=case["W"], oversamp=2.0)
    else:
        plan = mp.Plan(ctx, d["dims"], sample_idx=d["idx"])
    basis = mp.TuckerBasis(ctx, d["core"], d["factors"]) if "core" in d else mp.Basis(ctx, d["U"])
    ctx.reserve(plan, basis, case["C"])
    frames = [plan] + [mp.Plan(ctx, d["dims"], sample_idx=idx) for idx in d.get("frames", [])[1:]]
    keep = {k: d[k] for k in ("alpha", "p", "dp", "dalpha", "y", "eps") if k in d}
    return dict(case=case, ctx=ctx, plan=plan, frames=frames, basis=basis, **keep)


def run(s):
    case, ctx = s["case"], s["ctx"]
    if case["kind"] == "exam":
        s["batch"].run()
        return [s["y"], s["x"]]
    plan, basis, prec = s["plan"], s["basis"], case["prec"]
    if case["kind"] == "admm":
        opts = dict(n_outer=case["n_outer"], n_cg=case["n_cg"], n_tv=case["n_tv"], prec=prec)
        if case["frames"] == 1:
            p, _ = mp.image_solve(ctx, plan, basis, s["alpha"], s["y"][0], s["eps"][0], **opts)
        else:
            p, _ = mp.image_solve_dynamic(ctx, s["frames"], basis, s["alpha"], s["y"], s["eps"], **opts)
        return [p]
    if case["op"] == "forward":
        return [mp.forward(ctx, plan, basis, s["alpha"], s["p"], prec=prec)]
    if case["op"] == "adjoint":
        return [mp.adjoint(ctx, plan, basis, s["alpha"], s["y"], prec=prec)]
    if case["op"] == "pair":
        y = mp.forward(ctx, plan, basis, s["alpha"], s["p"], prec=prec)
        return [y, mp.adjoint(ctx, plan, basis, s["alpha"], y, prec=prec)]
    dy = mp.jacobian(ctx, plan, basis, s["alpha"], s["p"], s["dp"], s["dalpha"], prec=prec)
    gp, ga = mp.jacobian_adjoint(ctx, plan, basis, s["alpha"], s["p"], dy, prec=prec)
    return [dy, gp, ga]


# -------------------------------------------------------------------- work


def _samples(case):
    if case["kind"] == "radial":
        return case["spokes"] * case["readout"]
    if case["kind"] == "volume":
        acs = min(case["acs"], case["nz"]) * min(case["acs"], case["ny"])
        return case["nx"] * max(int(round(case["nz"] * case["ny"] / case["R"])), acs)
    return _slice_samples(case, *_dims(case))


def _op_work(case):
    """(expansions, projections onto the basis, transforms) of one pass, in units of all coils."""
    return {"forward": (1, 0, 1), "adjoint": (1, 0, 1), "pair": (2, 0, 2), "jacobian": (3, 1, 2)}[case["op"]]


def _transform_flops(case, N, C):
    if case["kind"] == "radial":
        return C * (5.0 * 4 * N * math.log2(4 * N) + 4.0 * case["W"] ** 2 * _samples(case))
    return 5.0 * C * N * math.log2(N)


def work(case):
    """Each input read once and each output written once; the basis in the type it is read in."""
    ub = 4 if case["prec"] == "bf16" else 8
    if case["kind"] == "exam":
        layout = _exam_layout(case)
        nbytes = sum(ub * n * n * EXAM_Q[n] for n in {n for n, _, _ in layout})
        flops = 0.0
        for n, C, R in layout:
            N, q, M = n * n, EXAM_Q[n], int(round(n * n / R))
            nbytes += 8 * (2 * N + C * q + 2 * C * M)
            flops += 2 * (8.0 * N * q * C + 5.0 * C * N * math.log2(N))
        return dict(bytes=nbytes, flops=flops)
    dims, C, q, M = _dims(case), case["C"], case["q"], _samples(case)
    N = int(np.prod(dims))
    if case["kind"] == "volume":
        nz, ny, nx = dims
        r1, r2, r3 = case["r1"], case["r2"], case["r3"]
        basis = ub * r1 * r2 * r3 * q
        expand = 8.0 * C * (r1 * r2 * r3 * q + r1 * r2 * r3 * nx + r1 * r2 * nx * ny + r1 * nx * ny * nz)
    else:
        basis, expand = ub * N * q, 8.0 * N * q * C
    if case["kind"] == "admm":
        # the maps once, then for each frame of an outer step n_cg + 2 normal operators and the TV iterations
        T = case["frames"]
        flops = expand + T * case["n_outer"] * ((case["n_cg"] + 2) * (2 * _transform_flops(case, N, C) + 16.0 * C * N)
                                                + 40.0 * case["n_tv"] * N)
        return dict(bytes=basis + 8 * (T * C * M + C * q + T * N), flops=flops)
    e, u, t = _op_work(case)
    flops = (e + u) * expand + t * _transform_flops(case, N, C)
    given = {"forward": C * q + N, "adjoint": C * q + C * M, "pair": C * q + N, "jacobian": 2 * (C * q + N)}[case["op"]]
    made = {"forward": C * M, "adjoint": N, "pair": C * M + N, "jacobian": C * M + N + C * q}[case["op"]]
    return dict(bytes=basis + 8 * (given + made), flops=flops)


# ------------------------------------------------- the same in 64 bits, plainly


class _Cartesian:
    """Centred unitary DFT of each coil, then the sampled points."""

    def __init__(self, dims, idx):
        self.dims, self.idx = dims, torch.from_numpy(idx.astype(np.int64)).to(DEV)
        self.axes = tuple(range(-len(dims), 0))

    def fwd(self, v):
        k = torch.fft.ifftshift(v.reshape(-1, *self.dims), dim=self.axes)
        k = torch.fft.fftshift(torch.fft.fftn(k, dim=self.axes, norm="ortho"), dim=self.axes)
        return k.reshape(v.shape[0], -1)[:, self.idx]

    def adj(self, y):
        k = torch.zeros(y.shape[0], int(np.prod(self.dims)), dtype=y.dtype, device=DEV)
        k[:, self.idx] = y
        k = torch.fft.ifftshift(k.reshape(-1, *self.dims), dim=self.axes)
        return torch.fft.fftshift(torch.fft.ifftn(k, dim=self.axes, norm="ortho"), dim=self.axes).reshape(
            y.shape[0], -1)


class _Gridding:
    """Kaiser-Bessel gridding on the twice oversampled grid (W taps per axis, deapodised)."""

    def __init__(self, n, traj, W, dtype):
        self.n, self.G, self.W = n, 2 * n, W
        beta = math.pi * math.sqrt((W / 2.0) ** 2 * 2.25 - 0.8)
        kappa = torch.from_numpy(traj).to(DEV).double() * (self.G / (2.0 * math.pi))
        taps = torch.floor(kappa)[:, :, None] + (torch.arange(W, device=DEV) - W // 2 + 1)
        arg = 1.0 - (2.0 * (kappa[:, :, None] - taps) / W) ** 2
        i0b = torch.special.i0(torch.tensor(beta, dtype=torch.float64, device=DEV))
        w = torch.where(arg >= 0, torch.special.i0(beta * torch.sqrt(arg.clamp(min=0))) / i0b, 0.0)
        g = torch.remainder(taps.long() + self.G // 2, self.G)
        self.cell = (g[:, 1, :, None] * self.G + g[:, 0, None, :]).reshape(-1)  # (M W W) cells, y taps slowest
        self.w = (w[:, 1, :, None] * w[:, 0, None, :]).to(dtype)
        t = torch.arange(n, device=DEV).double() - n // 2
        z2 = beta ** 2 - (math.pi * W * t / self.G) ** 2
        z = torch.sqrt(z2.abs())
        phi = W / i0b * torch.where(z2 > 0, torch.sinh(z) / z, torch.sin(z) / z)
        self.deap = (phi[:, None] * phi[None, :]).to(dtype)

    def fwd(self, v):
        n, G, o = self.n, self.G, self.G // 2 - self.n // 2
        out = []
        for c in range(v.shape[0]):
            grid = torch.zeros(G, G, dtype=v.dtype, device=DEV)
            grid[o:o + n, o:o + n] = v[c].reshape(n, n) / self.deap
            k = torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(grid)))
            out.append((k.reshape(-1)[self.cell].reshape(self.w.shape) * self.w).sum((1, 2)) / n)
        return torch.stack(out)

    def adj(self, y):
        n, G, o = self.n, self.G, self.G // 2 - self.n // 2
        out = []
        for c in range(y.shape[0]):
            part = torch.view_as_real(self.w * y[c][:, None, None]).reshape(-1, 2)
            grid = torch.zeros(G * G, 2, dtype=part.dtype, device=DEV).index_add_(0, self.cell, part)
            grid = torch.view_as_complex(grid).reshape(G, G)
            img = torch.fft.fftshift(torch.fft.ifft2(torch.fft.ifftshift(grid), norm="forward"))
            out.append((img[o:o + n, o:o + n] / self.deap).reshape(-1) / n)
        return torch.stack(out)


def _sampling(case, d):
    if "traj" in d:
        return _Gridding(case["n"], d["traj"], case["W"], torch.complex128)
    return _Cartesian(d["dims"], d["idx"])


def _maps(d, alpha, dtype=torch.complex128):
    """U alpha for every coil (C, N)."""
    a = alpha.to(dtype)
    if "core" not in d:
        return a @ d["U"].to(dtype)
    core = torch.from_numpy(d["core"]).to(DEV).to(dtype)
    f1, f2, f3 = (torch.from_numpy(f).to(DEV).to(dtype) for f in d["factors"])
    t = torch.einsum("abdq,cq->cabd", core, a)
    t = torch.einsum("cabd,xd->cabx", t, f3)
    t = torch.einsum("cabx,yb->cayx", t, f2)
    return torch.einsum("cayx,za->czyx", t, f1).reshape(a.shape[0], -1)


def _project(d, v):
    """U^H v for every coil (C, q)."""
    if "core" not in d:
        return v @ d["U"].to(v.dtype).conj().T
    core = torch.from_numpy(d["core"]).to(DEV).to(v.dtype)
    f1, f2, f3 = (torch.from_numpy(f).to(DEV).to(v.dtype) for f in d["factors"])
    t = torch.einsum("czyx,za->cayx", v.reshape(-1, *d["dims"]), f1.conj())
    t = torch.einsum("cayx,yb->cabx", t, f2.conj())
    t = torch.einsum("cabx,xd->cabd", t, f3.conj())
    return torch.einsum("cabd,abdq->cq", t, core.conj())


def _forward(fs, s, p):
    return fs.fwd(s * p[None, :])


def _adjoint(fs, s, y):
    return (s.conj() * fs.adj(y)).sum(0)


def _dot(a, b):
    return sum(float((x.conj() * y).sum().real) for x, y in zip(a, b))


def _cg(apply, x, b, count):
    r = [u - v for u, v in zip(b, apply(x))]
    d, rr = r, _dot(r, r)
    for _ in range(count):
        ad = apply(d)
        dad = _dot(d, ad)
        a = rr / dad if dad > 0 else 0.0
        x = [u + a * v for u, v in zip(x, d)]
        r = [u - a * v for u, v in zip(r, ad)]
        new = _dot(r, r)
        beta = new / rr if rr > 0 else 0.0
        d, rr = [u + beta * v for u, v in zip(r, d)], new
    return x


def _tv_prox(b, lam, count):
    """argmin 1/2 |x - b|^2 + lam TV(x) by fast gradient projection on the dual (isotropic TV over all axes of b)."""
    nd = b.dim()

    def grad(x):
        g = torch.zeros(nd, *x.shape, dtype=x.dtype, device=DEV)
        for a in range(nd):
            g[a].narrow(a, 0, x.shape[a] - 1).copy_(torch.diff(x, dim=a))
        return g

    def grad_adj(P):
        x = torch.zeros_like(b)
        for a in range(nd):
            n = b.shape[a] - 1
            x.narrow(a, 1, n).add_(P[a].narrow(a, 0, n))
            x.narrow(a, 0, n).sub_(P[a].narrow(a, 0, n))
        return x

    P = torch.zeros(nd, *b.shape, dtype=b.dtype, device=DEV)
    R, t = P, 1.0
    for _ in range(count):
        Pn = R + grad(b - lam * grad_adj(R)) / (4.0 * nd * lam)
        Pn = Pn / Pn.abs().square().sum(0).sqrt().clamp(min=1.0)
        tn = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * t * t))
        R, P, t = Pn + ((t - 1.0) / tn) * (Pn - P), Pn, tn
    return b - lam * grad_adj(P)


def _admm(samplings, s, y, eps, case):
    """Scaled ADMM: TV prox, projection onto the noise balls, CG for the frames, dual update, balanced rho."""
    T, shape = case["frames"], (case["n"], case["n"])
    shape = shape if T == 1 else (T, *shape)

    def fwd(v):
        return torch.stack([_forward(fs, s, v[t]) for t, fs in enumerate(samplings)])

    def adj(w):
        return torch.stack([_adjoint(fs, s, w[t]) for t, fs in enumerate(samplings)])

    p = torch.zeros(T, s.shape[1], dtype=y.dtype, device=DEV)
    u0, uk, ap, rho = torch.zeros_like(p), torch.zeros_like(y), torch.zeros_like(y), 1.0
    eps = torch.from_numpy(eps).to(DEV)
    for _ in range(case["n_outer"]):
        z0 = _tv_prox((p + u0).reshape(shape), 1.0 / rho, case["n_tv"]).reshape(T, -1)
        diff = ap + uk - y
        zk = y + (eps / torch.maximum(torch.linalg.vector_norm(diff, dim=2), eps))[:, :, None] * diff
        rhs = z0 - u0 + adj(zk - uk)
        last, ap_last = p, ap
        (p,) = _cg(lambda v: [v[0] + adj(fwd(v[0]))], [p], [rhs], case["n_cg"])
        ap = fwd(p)
        u0, uk = u0 + p - z0, uk + ap - zk
        primal = math.sqrt(_dot([p - z0, ap - zk], [p - z0, ap - zk]))
        dual = rho * math.sqrt(_dot([p - last, ap - ap_last], [p - last, ap - ap_last]))
        f = 2.0 if primal > 10.0 * dual else 0.5 if dual > 10.0 * primal else 1.0
        rho, u0, uk = rho * f, u0 / f, uk / f
    return p[0] if T == 1 else p


def exact(case, seed):
    d = _inputs(case, seed)
    wide = torch.complex128
    if case["kind"] == "exam":
        ys, xs = [], []
        for i in d["slices"]:
            s = i["alpha"].to(wide) @ d["bases"][i["n"]].to(wide)
            fs = _Cartesian((i["n"], i["n"]), i["idx"])
            y = _forward(fs, s, i["p"].to(wide))
            ys.append(torch.nn.functional.pad(torch.view_as_real(y.reshape(-1)), (0, 0, 0, y.numel() % 2)))
            xs.append(_adjoint(fs, s, y))
        return [torch.view_as_complex(torch.cat(ys)), torch.cat(xs)]
    fs = _sampling(case, d)
    s = _maps(d, d["alpha"])
    if case["kind"] == "admm":
        return [_admm([_Cartesian(d["dims"], idx) for idx in d["frames"]], s, d["y"].to(wide), d["eps"], case)]
    p = d["p"].to(wide)
    if case["op"] == "forward":
        return [_forward(fs, s, p)]
    if case["op"] == "adjoint":
        return [_adjoint(fs, s, d["y"].to(wide))]
    if case["op"] == "pair":
        y = _forward(fs, s, p)
        return [y, _adjoint(fs, s, y)]
    dy = fs.fwd(s * d["dp"].to(wide) + p * _maps(d, d["dalpha"]))
    w = fs.adj(dy)
    return [dy, (s.conj() * w).sum(0), _project(d, p.conj() * w)]
