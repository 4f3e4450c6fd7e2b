"""Workloads of the solver, as a user's program runs them: what its speed is measured on.

A case is a dict of plain values.  prepare() builds what such a program holds before the call (the grid
handle with its phases, the batch handle, the output tensors), run() is one call through the public
binding `paper_2009_03762_gb300.gfp`, work() the bytes and operations the call cannot do without, and
exact() the same results from plain torch in 64 bits (its own operators and iteration, torch.fft).

Sizes and options are those of the repository's experiments, tests and benchmark: 16-48 voxels per axis for
the allocation-free solve and small effective-stiffness calls, 64-128 for gradients, batches and the
scheme comparison, 256 and 512 for the mixed-precision benchmark, 81 and 162 = 2 81 and non-cubic
2^a 3^b grids for the paper's convergence experiment and ragged shapes.  Grids run with the library's default
tiles, as a program that does not call the autotuner has them.

A mixed-precision solve forms its strain by FP32 corrections, so its digits beyond FP32 are rounding: the
program keeps that strain (and what is averaged from it) in float32.
"""
import math

import numpy as np
import torch

from paper_2009_03762_gb300 import gfp

PAIRS = ((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))  # tensor components (11, 22, 33, 23, 13, 12)


def _case(name, kind, n, **kw):
    n1, n2, n3 = (n, n, n) if isinstance(n, int) else n
    c = dict(name=name, kind=kind, n1=n1, n2=n2, n3=n3, op="AFB_R", disc="PCD", prec="FP64", field="spheres",
             contrast=10.0, tol=1e-8, maxit=5000)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: allocation-free solve of a small cell inside a host framework (launch latency)
        _case("noalloc_16", "noalloc", 16, field="noise"),
        # effective stiffness of a small cell in the default precision: six solves of about 40 iterations
        _case("ceff_fp64_32", "ceff", 32),
        # the plain Fourier scheme on an odd 3^4 grid (one of the lengths without a register plan)
        _case("fourier_fp64_81", "solve", 81, op="F", disc="TD", field="cube", contrast=5.0, tol=1e-6),
        # the scheme comparison's smooth-interface cube, FP64 to 1e-10
        _case("smooth_fp64_128", "solve", 128, field="smooth", tol=1e-10),
        # a ragged cell with an eigenstrain, and its displacement field
        _case("eigen_disp_fp64_162x108x54", "solve", (162, 108, 54), op="ACD", eigenstrain=True, displacement=True,
              tol=1e-6),
        # a large cell in the default precision
        _case("spheres_fp64_256", "solve", 256, tol=1e-4),
        # sensitivities of a shear entry of C_eff on the perturbed smooth cube: two solves and the contraction
        _case("grad_fp64_64", "grad", 64, disc="TD", field="lognormal", row=5, col=3, tol=1e-10),
        # the discrete Green operator (alias half-range 4), its table kept by the grid
        _case("dgo_fp64_64", "solve", 64, op="DGO", dgo_m=4),
        # the convergence experiment's n = 162 cube in mixed precision
        _case("cube_mixed_162", "solve", 162, op="ACD", prec="MIXED", field="cube"),
        # the benchmark's random-sphere cell in mixed precision
        _case("spheres_mixed_256", "solve", 256, prec="MIXED", contrast=100.0, tol=1e-6),
        # the largest mixed-precision cell
        _case("spheres_mixed_512", "solve", 512, prec="MIXED", tol=1e-6),
        # batched homogenization: cells of the batch experiment's sizes x six loads, one graph launch
        _case("batch_mixed_64_96_128", "batch", 0, prec="MIXED", cells="64,96,128", tol=1e-8),
    ]


_REGISTER = (32, 64, 96, 128, 192, 256)
_OTHER = (18, 24, 27, 36, 48, 54, 72, 81, 108, 144, 162)


def _length(rng, lo, hi):
    """A grid length 2^a 3^b in [lo, hi], spread over its logarithm, register-plan lengths as often as others."""
    pool = [n for n in (_REGISTER if rng.random() < 0.5 else _OTHER) if lo <= n <= hi] or [lo]
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(pool, key=lambda n: abs(math.log(n / x)))


def _shape(rng, lo, hi):
    """A cubic cell as often as a ragged one."""
    n = _length(rng, lo, hi)
    return n if rng.random() < 0.5 else (n, _length(rng, lo, hi), _length(rng, lo, hi))


def draw(rng):
    kind = rng.choice(("noalloc", "ceff", "solve", "solve", "solve", "mixed", "mixed", "mixed", "grad", "dgo", "batch"))
    contrast = round(math.exp(rng.uniform(math.log(2.0), math.log(30.0))), 3)
    op = rng.choice(("AFB_R", "AFB_R", "ACD", "CD"))
    disc = rng.choice(("TD", "PCD"))
    tol = rng.choice((1e-6, 1e-8))
    if kind == "noalloc":
        c = _case("", "noalloc", _shape(rng, 18, 36), op=op, disc=disc, field="noise", tol=tol)
    elif kind == "ceff":
        c = _case("", "ceff", _shape(rng, 18, 64), op=op, disc=disc, contrast=contrast, tol=tol,
                  prec=rng.choice(("FP64", "MIXED")))
    elif kind == "solve":
        c = _case("", "solve", _shape(rng, 24, 192), op=op, disc=disc, contrast=contrast, tol=tol,
                  field=rng.choice(("spheres", "smooth", "noise")), eigenstrain=rng.random() < 0.3,
                  displacement=rng.random() < 0.3)
    elif kind == "mixed":
        c = _case("", "solve", _shape(rng, 48, 256), op=op, disc=disc, contrast=contrast, tol=tol, prec="MIXED",
                  field=rng.choice(("spheres", "smooth", "noise")))
    elif kind == "grad":
        c = _case("", "grad", _shape(rng, 32, 96), op=op, disc=disc, field="lognormal", row=rng.randrange(6),
                  col=rng.randrange(6), tol=tol)
    elif kind == "dgo":
        c = _case("", "solve", _shape(rng, 18, 64), op="DGO", dgo_m=rng.choice((2, 4)), tol=tol, contrast=contrast)
    else:
        cells = ",".join(str(rng.choice((48, 64, 96, 128))) for _ in range(rng.choice((2, 3))))
        c = _case("", "batch", 0, prec="MIXED", cells=cells, op=op, contrast=contrast, tol=tol)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------ inputs
def _lame(E, nu=0.3):
    return E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu)), E / (2.0 * (1.0 + nu))


def _spheres(rng, n1, n2, n3, vf=0.25):
    """Indicator [n3, n2, n1] (GPU, bool) of random non-overlapping periodic spheres, radii U[6, 16] / 128 of the
    shortest axis, added until they fill the volume fraction."""
    dims = np.array([n1, n2, n3], dtype=float)
    scale = dims.min() / 128.0
    centres, radii, filled = np.zeros((0, 3)), np.zeros(0), 0.0
    for _ in range(20000):
        r, x = rng.uniform(6.0, 16.0) * scale, rng.uniform(0.0, 1.0, 3) * dims
        d = np.abs(centres - x)
        d = np.minimum(d, dims - d)
        if radii.size and np.any((d * d).sum(1) < (radii + r) ** 2):
            continue
        centres, radii = np.vstack([centres, x]), np.append(radii, r)
        filled += 4.0 / 3.0 * math.pi * r ** 3
        if filled >= vf * dims.prod():
            break
    ind = torch.zeros(n3, n2, n1, dtype=torch.bool, device="cuda")
    for x, r in zip(centres, radii):
        at, dist = [], []
        for q in range(3):
            i = torch.arange(math.floor(x[q] - r), math.ceil(x[q] + r) + 1, device="cuda")
            at.append(i % int(dims[q]))
            dist.append((i + 0.5 - x[q]).double() ** 2)
        inside = dist[2][:, None, None] + dist[1][None, :, None] + dist[0][None, None, :] <= r * r
        block = (at[2][:, None, None], at[1][None, :, None], at[0][None, None, :])
        ind[block] = ind[block] | inside
    return ind


def _phases(case, n1, n2, n3, seed, contrast):
    """Lame fields (lambda, mu) [n3, n2, n1] on the GPU."""
    rng = np.random.default_rng([seed, n1, n2, n3])
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
    shape, field = (n3, n2, n1), case["field"]
    off = 0.0 if case["disc"] == "TD" else 0.5
    if field == "noise":  # voxelwise random moduli, E log-uniform over the contrast, nu uniform
        u = torch.rand(2, *shape, dtype=torch.float64, device="cuda", generator=gen)
        return tuple(t.contiguous() for t in _lame(torch.exp(u[0] * math.log(contrast)), 0.1 + 0.3 * u[1]))
    if field == "spheres":
        E = torch.where(_spheres(rng, n1, n2, n3), contrast, 1.0).double()
        return tuple(t.contiguous() for t in _lame(E))
    # a cube of about half the edge, moved and sized by the seed; smooth: tanh interface of half-width 2 voxels
    f = torch.ones(1, 1, 1, dtype=torch.float64, device="cuda")
    for q, n in enumerate((n3, n2, n1)):
        x = torch.arange(n, dtype=torch.float64, device="cuda") + off
        edge = max(1, int(round(n * rng.uniform(0.4, 0.6))))
        a = (n - edge) // 2
        if field == "cube":
            g = ((x >= a) & (x < a + edge)).double()
        else:
            g = 0.5 * (torch.tanh((x - a) / 2.0) - torch.tanh((x - a - edge) / 2.0))
        f = f * g.reshape([-1 if i == q else 1 for i in range(3)])
    lam, mu = _lame(torch.exp(f * math.log(contrast)))
    if field == "lognormal":
        z = torch.randn(2, *shape, dtype=torch.float64, device="cuda", generator=gen)
        lam, mu = lam * torch.exp(0.1 * z[0]), mu * torch.exp(0.1 * z[1])
    return lam.contiguous(), mu.contiguous()


def _load(seed):
    """Mean strain of a general load case, about one percent."""
    return [float(v) for v in 0.01 * np.random.default_rng([seed, 6]).standard_normal(6)]


def _inputs(case, seed):
    n1, n2, n3 = case["n1"], case["n2"], case["n3"]
    lam, mu = _phases(case, n1, n2, n3, seed, case["contrast"])
    estar = None
    if case.get("eigenstrain"):  # thermal-like mismatch: isotropic and proportional to the inclusion's excess stiffness
        f = (mu - mu.min()) / (mu.max() - mu.min())
        estar = torch.stack([0.005 * f * (1.0 if c < 3 else 0.2) for c in range(6)])
    return lam, mu, estar, _load(seed)


def _cells(case, seed):
    """The batch's cells: their sizes, and contrasts from a tenth to the case's, log-uniform."""
    rng = np.random.default_rng([seed, 77])
    out = []
    for k, n in enumerate(int(v) for v in case["cells"].split(",")):
        contrast = float(np.exp(rng.uniform(np.log(case["contrast"] / 10.0), np.log(case["contrast"]))))
        out.append(_phases(case, n, n, n, seed + 1000 * (k + 1), contrast))
    return out


# ------------------------------------------------------------------------------------------------ the calls
def _scheme(case):
    return gfp.scheme(case["op"], case["disc"], case["prec"], dgo_m=case.get("dgo_m", 0))


def prepare(case, seed):
    s = {"case": case, "sch": _scheme(case)}
    if case["kind"] == "batch":
        s["grids"] = []
        for lam, mu in _cells(case, seed):
            n3, n2, n1 = lam.shape
            g = gfp.Grid(n1, n2, n3)
            g.set_phases(lam, mu)
            s["grids"].append(g)
        s["batch"] = gfp.Batch(s["grids"], s["sch"])
        return s
    lam, mu, estar, s["E"] = _inputs(case, seed)
    shape = tuple(lam.shape)
    if case["kind"] == "noalloc":
        s["lam"], s["mu"], s["eps"] = lam, mu, torch.empty((6,) + shape, dtype=torch.float64, device="cuda")
        return s
    g = s["grid"] = gfp.Grid(case["n1"], case["n2"], case["n3"])
    g.set_phases(lam, mu)
    if estar is not None:
        g.set_eigenstrain(estar)
    if case["kind"] == "solve":
        s["eps"] = torch.empty((6,) + shape, dtype=torch.float64, device="cuda")
    if case.get("displacement"):
        s["u"] = torch.empty((3,) + shape, dtype=torch.float64, device="cuda")
    if case["kind"] == "grad":
        s["dlam"], s["dmu"] = (torch.empty(shape, dtype=torch.float64, device="cuda") for _ in range(2))
    return s


def run(s):
    case, sch, tol, maxit = s["case"], s["sch"], s["case"]["tol"], s["case"]["maxit"]
    if case["kind"] == "batch":
        C, _, rc = s["batch"].solve(tol, maxit)
        return {"C": C.astype(np.float32), "status": rc}
    if case["kind"] == "noalloc":
        rc, r = gfp.solve_noalloc(s["lam"], s["mu"], s["eps"], sch, s["E"], tol, maxit)
        return {"eps": s["eps"], "sigma": r.sigma_mean, "iters": r.iters, "status": rc}
    g = s["grid"]
    if case["kind"] == "ceff":
        C, iters, rc = g.effective_stiffness(sch, tol, maxit)
        if case["prec"] == "MIXED":
            return {"C": C.astype(np.float32), "status": rc}
        return {"C": C, "iters": np.array(iters), "status": rc}
    if case["kind"] == "grad":
        g.grad(sch, case["row"], case["col"], tol, maxit, s["dlam"], s["dmu"])
        return {"dlam": s["dlam"], "dmu": s["dmu"]}
    r = g.solve(sch, s["E"], tol, maxit)
    eps = g.strain(s["eps"])
    if case["prec"] == "MIXED":
        return {"eps": eps.float(), "sigma": r.sigma_mean.astype(np.float32), "status": r.status}
    out = {"eps": eps, "sigma": r.sigma_mean, "iters": r.iters, "status": r.status}
    if case.get("displacement"):
        out["u"] = g.displacement(sch, s["u"])
    return out


def _iterations(case, contrast):
    """Iterations of the basic scheme with the reference medium (min + max) / 2: its contraction is at most
    (c - 1) / (c + 1), reached on few modes, so about half that bound's count."""
    c = max(contrast, 1.5)
    return max(3.0, 0.5 * math.log(case["tol"]) / math.log((c - 1.0) / (c + 1.0)))


def work(case):
    """Bytes: the moduli (and eigenstrain) read once, the results written once.  Operations: per iteration 12 real
    transforms of the six components per voxel at 2.5 log2 n flops (the half spectrum's count) and about 65 flops of
    stress, Green operator and update."""
    def one(n1, n2, n3, solves, contrast):
        N = n1 * n2 * n3
        per = 12 * 2.5 * math.log2(max(2, N)) + 65
        return N, solves * _iterations(case, contrast) * N * per
    if case["kind"] == "batch":
        got = [one(n, n, n, 6, case["contrast"] / math.sqrt(10.0)) for n in map(int, case["cells"].split(","))]
        return {"bytes": sum(16.0 * N + 288 for N, _ in got), "flops": sum(f for _, f in got)}
    solves = {"ceff": 6, "grad": 2}.get(case["kind"], 1)
    N, flops = one(case["n1"], case["n2"], case["n3"], solves, 3.0 if case["field"] == "lognormal" else case["contrast"])
    words = 2 + {"ceff": 0, "grad": 2}.get(case["kind"], 3 if case["prec"] == "MIXED" else 6)
    words += (6 if case.get("eigenstrain") else 0) + (3 if case.get("displacement") else 0)
    return {"bytes": 8.0 * words * N, "flops": flops}


# ------------------------------------------------------------------------------------------------ in 64 bits
def _angles(n):
    k = torch.arange(n, device="cuda")
    k = torch.where(k < (n + 1) // 2, k, k - n)  # the Nyquist index of an even axis is -n/2
    return 2.0 * math.pi * k.double() / n


def _real_vectors(case, ns):
    """The real vector kt(k) of the scheme on the full grid of modes, three broadcastable tensors [n3, n2, n1]."""
    A, B = [], []
    for r, n in enumerate(ns):
        th = _angles(n)
        if case["op"] == "F":
            a, b = th, torch.ones_like(th)
        elif case["op"] in ("CD", "ACD"):
            a, b = torch.sin(th), torch.cos(th) if case["op"] == "ACD" else torch.ones_like(th)
        else:  # AFB_R
            a, b = 2.0 * torch.sin(0.5 * th), torch.cos(0.5 * th)
        a, b = (torch.where(t.abs() < 1e-12, 0.0, t) for t in (a, b))
        view = [1, 1, 1]
        view[2 - r] = n
        A.append(a.reshape(view))
        B.append(b.reshape(view))
    return [A[0] * B[1] * B[2], A[1] * B[2] * B[0], A[2] * B[0] * B[1]]


def _times_k(T, k):
    return [T[0] * k[0] + T[5] * k[1] + T[4] * k[2], T[5] * k[0] + T[1] * k[1] + T[3] * k[2],
            T[4] * k[0] + T[3] * k[1] + T[2] * k[2]]


def _gamma(T, k, lam, mu):
    """The isotropic Green operator on a transformed symmetric tensor, 0 where k = 0."""
    v = _times_k(T, k)
    s = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    inv = torch.where(s == 0, 0.0, 1.0 / torch.where(s == 0, 1.0, s))
    kv = (k[0] * v[0] + k[1] * v[1] + k[2] * v[2]) * inv
    out = []
    for i, j in PAIRS:
        out.append(inv * ((k[i] * v[j] + k[j] * v[i]) / (2.0 * mu) - (lam + mu) / (mu * (lam + 2.0 * mu)) * k[i] * k[j] * kv))
    return torch.stack(out)


def _stress(lam, mu, e):
    s = 2.0 * mu * e
    s[:3] += lam * (e[0] + e[1] + e[2])
    return s


def _dgo_sums(case, ns, lam, mu):
    """Moments of the alias sum with the weights sinc^2: S2 [3][3] and S4 as functions of sorted indices."""
    m = case["dgo_m"]
    axes, weights = [], []
    for r, n in enumerate(ns):
        o = torch.arange(n, device="cuda").double()
        kr, wr = [], []
        for nu in range(-m, m):
            j = nu * n + o
            x = math.pi * j / n
            sinc = torch.where(j == 0, 1.0, torch.where(j % n == 0, 0.0, torch.sin(x) / torch.where(j == 0, 1.0, x)))
            view = [1, 1, 1]
            view[2 - r] = n
            kr.append((2.0 * math.pi * j / n).reshape(view))
            wr.append((sinc * sinc).reshape(view))
        axes.append(kr)
        weights.append(wr)
    S2, S4 = {}, {}
    for c in range(2 * m):
        for b in range(2 * m):
            for a in range(2 * m):
                k = (axes[0][a], axes[1][b], axes[2][c])
                w = weights[0][a] * weights[1][b] * weights[2][c]
                s = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
                inv = torch.where(s == 0, 0.0, 1.0 / torch.where(s == 0, 1.0, s))
                for i, j in PAIRS:
                    t = w * inv * k[i] * k[j]
                    S2[min(i, j), max(i, j)] = S2.get((min(i, j), max(i, j)), 0.0) + t
                    t = t * inv
                    for p, q in PAIRS:
                        key = tuple(sorted((i, j, p, q)))
                        if (tuple(sorted((i, j))), tuple(sorted((p, q)))) == (key[:2], key[2:]):
                            S4[key] = S4.get(key, 0.0) + t * k[p] * k[q]
    return S2, S4


def _dgo_apply(T, S2, S4, lam, mu):
    s2 = lambda a, b: S2[min(a, b), max(a, b)]  # noqa: E731
    cc = (lam + mu) / (lam + 2.0 * mu)
    out = []
    for i, j in PAIRS:
        acc = 0.0
        for q, (a, b) in enumerate(PAIRS):
            g = cc / mu * S4[tuple(sorted((i, j, a, b)))]
            for d, x, y in ((i == a, b, j), (i == b, a, j), (j == a, b, i), (j == b, a, i)):
                if d:
                    g = g - s2(x, y) / (4.0 * mu)
            acc = acc + g * T[q] * (1.0 if a == b else 2.0)
        acc = acc.clone()
        acc[0, 0, 0] = 0.0
        out.append(acc)
    return torch.stack(out)


def _solve64(case, lam, mu, estar, E, ops):
    """The basic scheme in 64 bits: (strain, mean stress, increment spectrum of the last iterate)."""
    ns = (lam.shape[2], lam.shape[1], lam.shape[0])
    N = lam.numel()
    lh, mh = (float(0.5 * (t.min() + t.max())) for t in (lam, mu))
    Eb = torch.tensor(E, dtype=torch.float64, device="cuda").reshape(6, 1, 1, 1)
    w = torch.tensor([1, 1, 1, 2, 2, 2], dtype=torch.float64, device="cuda")
    eps = Eb.expand(6, *lam.shape).clone()
    dims = (1, 2, 3)
    k = _real_vectors(case, ns) if case["op"] != "DGO" else None
    for _ in range(case["maxit"]):
        if case["op"] == "DGO":
            if "dgo" not in ops:
                ops["dgo"] = _dgo_sums(case, ns, lh, mh)
            T = torch.fft.fftn(_stress(lam - lh, mu - mh, eps), dim=dims)
            new = Eb + torch.fft.ifftn(_dgo_apply(T, *ops["dgo"], lh, mh), dim=dims).real
            eta = math.sqrt(float(((new - eps) ** 2).sum(dims) @ w)) / math.sqrt(N * float(Eb.flatten() ** 2 @ w))
            eps = new
            if eta < case["tol"]:
                break
            continue
        T = torch.fft.fftn(_stress(lam, mu, eps if estar is None else eps - estar), dim=dims)
        T0 = math.sqrt(float(T[:, 0, 0, 0].real ** 2 @ w))
        eta = math.sqrt(sum(float((v.real ** 2 + v.imag ** 2).sum()) for v in _times_k(T, k))) / T0
        if eta < case["tol"]:
            break
        eps -= torch.fft.ifftn(_gamma(T, k, lh, mh), dim=dims).real
        del T
    sig = _stress(lam, mu, eps if estar is None else eps - estar)
    return eps, sig.mean(dims)


def _displacement64(case, eps, E):
    """u^ of eps - E = sym(u (x) q): q = i kt for ACD and CD, e^{i sum(theta)/2} i kt for AFB_R."""
    ns = (eps.shape[3], eps.shape[2], eps.shape[1])
    k = _real_vectors(case, ns)
    T = torch.fft.fftn(eps - torch.tensor(E, dtype=torch.float64, device="cuda").reshape(6, 1, 1, 1), dim=(1, 2, 3))
    v = _times_k(T, k)
    s = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    inv = torch.where(s == 0, 0.0, 1.0 / torch.where(s == 0, 1.0, s))
    kv = (k[0] * v[0] + k[1] * v[1] + k[2] * v[2]) * inv
    c = torch.ones(1, dtype=torch.complex128, device="cuda")
    if case["op"] == "AFB_R":
        th = [_angles(n) for n in ns]
        c = torch.exp(0.5j * (th[2][:, None, None] + th[1][None, :, None] + th[0][None, None, :]))
    u = torch.stack([(2.0 * v[i] - k[i] * kv) * inv / (1j * c) for i in range(3)])
    return torch.fft.ifftn(u, dim=(1, 2, 3)).real


def _unit(J):
    return [(1.0 if J < 3 else 0.5) if c == J else 0.0 for c in range(6)]


def _ceff64(case, lam, mu):
    return np.stack([_solve64(case, lam, mu, None, _unit(J), {})[1].cpu().numpy() for J in range(6)], axis=1)


def exact(case, seed):
    if case["kind"] == "batch":
        return {"C": np.stack([_ceff64(case, lam, mu) for lam, mu in _cells(case, seed)]), "status": None}
    if case["n1"] * case["n2"] * case["n3"] > 300 ** 3:
        return None  # minutes of 64-bit transforms
    lam, mu, estar, E = _inputs(case, seed)
    if case["kind"] == "ceff":
        return {"C": _ceff64(case, lam, mu), "iters": None, "status": None}
    if case["kind"] == "grad":
        a, b = (_solve64(case, lam, mu, None, _unit(J), {})[0] for J in (case["row"], case["col"]))
        n = lam.numel()
        dmu = 2.0 / n * ((a[:3] * b[:3]).sum(0) + 2.0 * (a[3:] * b[3:]).sum(0))
        return {"dlam": a[:3].sum(0) * b[:3].sum(0) / n, "dmu": dmu}
    eps, sigma = _solve64(case, lam, mu, estar, E, {})
    out = {"eps": eps, "sigma": sigma, "iters": None, "status": None}
    if case.get("displacement"):
        out["u"] = _displacement64(case, eps, E)
    return out
