"""Performance cases: the work a user of the library has it do, through its public entry points.

Every case is one call (or one short sequence of calls) of the Python binding on inputs made from a seed:
lognormal conductivities a = exp(g), g a periodic Gaussian random field of squared-exponential covariance (the
material of the benchmark), and smooth random fields as operands.  Low-rank results are compared as the grid
values they stand for, since a tensor train's carriages are unique only up to a change of basis at each bond.
``exact`` evaluates the same definitions in FP64 with plain torch (FFTs of the whole grid, QR and SVD on the
carriages), independent of the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1902_07455_gb300 as lrfg

# grid sizes: odd, prime factors 3, 5, 7 (the sizes of the serving workload), and for Ga those whose double grid
# 2N - 1 the transforms accept too
SIZES = [27, 35, 45, 49, 63, 75, 81, 105, 125, 135, 147, 175, 189, 225, 243, 245, 315, 343, 375, 405, 441, 525, 567,
         625, 675, 729]
GA_SIZES = [25, 33, 35, 39, 63, 77, 81]

# the constant anisotropic parts of the paper's anisotropic materials (eigenvalues (1, 10) in 2D, (1, 5, 10) in 3D
# in an oblique basis)
_Q2 = np.array([[0.8, -0.6], [0.6, 0.8]])
_Q3 = np.array([[2.0, -2.0, 1.0], [1.0, 2.0, 2.0], [2.0, 1.0, -2.0]]) / 3.0
ANISO = {2: _Q2 @ np.diag([1.0, 10.0]) @ _Q2.T, 3: _Q3 @ np.diag([1.0, 5.0, 10.0]) @ _Q3.T}

DEV = "cuda"
F64 = torch.float64


def _grid(case):
    return tuple(int(case[k]) for k in ("n0", "n1", "n2") if case.get(k))


def _case(kind, n, **kw):
    c = {"kind": kind, "n0": n[0], "n1": n[1]}
    if len(n) == 3:
        c["n2"] = n[2]
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one 2D full-format solve of a small microstructure (about fifty CG steps of a few
        # microseconds of work each: launches and latency)
        dict(_case("full_solve", (63, 63), prec="fp64", tol=1e-8), name="full-2d-63-solve"),
        # the benchmark's grid: one preconditioned application of the full-format FP64 operator (a CG step's work)
        dict(_case("full_apply", (243, 243, 243), disc="gani", aniso=False), name="full-3d-243-apply"),
        # unequal, non-power-of-three axes with an anisotropic part
        dict(_case("full_apply", (105, 147, 75), disc="gani", aniso=True), name="full-3d-ragged-aniso-apply"),
        # the fastest full-format route to the effective property at the benchmark's grid
        dict(_case("full_solve", (243, 243, 243), prec="mixed", tol=1e-5), name="full-3d-243-mixed-solve"),
        # exact integration of a voxel image on the double grid
        dict(_case("full_apply", (63, 63, 63), disc="ga", aniso=False), name="ga-3d-63-apply"),
        # the benchmark's low-rank solve is 80-100 of these: rank 20, randomised rounding of the products
        dict(_case("tt_apply", (243, 243, 243), rank=20, coeff_rank=10, over=10), name="tt-243-r20-apply"),
        # the same at a batch request's size and low rank, on unequal axes
        dict(_case("tt_apply", (63, 105, 45), rank=8, coeff_rank=6, over=8), name="tt-ragged-r8-apply"),
        # the truncation of an iterate plus its step, T(u + omega r), on a large uneven grid
        dict(_case("tt_round", (729, 525, 405), rank=20), name="tt-729-r20-round"),
        # a coefficient given as grid values, compressed before a low-rank solve (inside every grid request)
        dict(_case("tt_compress", (135, 135, 135), rank=10), name="tt-135-compress"),
        # the homogenised tensor: six right-hand sides in lockstep, a few iterations with the deterministic rounding
        # the library uses by default
        dict(_case("tt_tensor", (81, 81, 81), rank=10, coeff_rank=5, over=0, maxit=2), name="tt-81-tensor"),
        # the Tucker truncation of an iterate plus its step
        dict(_case("tucker_round", (135, 135, 135), rank=12), name="tucker-135-r12-round"),
        # the serving executor: a burst of requests of mixed dimension, size and format from host memory
        dict(_case("serve", (81, 81, 45), count=8, workers=4, rank=8, maxit=2), name="serve-8"),
    ]


def _near(rng, lo, hi, sizes=SIZES):
    """A size of the list between lo and hi, even over the logarithm."""
    s = [n for n in sizes if lo <= n <= hi]
    x = math.exp(rng.uniform(math.log(s[0]), math.log(s[-1])))
    return min(s, key=lambda n: abs(math.log(n / x)))


def draw(rng):
    kind = rng.choice(["full_solve", "full_apply", "full_apply", "tt_apply", "tt_apply", "tt_round", "tt_compress",
                       "tt_tensor", "tucker_round", "serve"])
    if kind == "full_solve":
        if rng.random() < 0.5:
            n = (_near(rng, 27, 405), _near(rng, 27, 405))
            return _case(kind, n, prec="fp64", tol=1e-8)
        return _case(kind, tuple(_near(rng, 45, 243) for _ in range(3)), prec="mixed", tol=1e-5)
    if kind == "full_apply":
        if rng.random() < 0.3:
            d = rng.choice([2, 3])
            return _case(kind, tuple(_near(rng, 25, 81, GA_SIZES) for _ in range(d)), disc="ga", aniso=rng.random() < 0.5)
        d = rng.choice([2, 3, 3])
        n = tuple(_near(rng, 27, 729 if d == 2 else 243) for _ in range(d))
        return _case(kind, n, disc="gani", aniso=rng.random() < 0.5)
    if kind == "tt_apply":
        d = rng.choice([2, 3, 3])
        return _case(kind, tuple(_near(rng, 45, 243) for _ in range(d)), rank=rng.randint(6, 20),
                     coeff_rank=rng.randint(3, 10), over=rng.randint(5, 10))
    if kind == "tt_round":
        return _case(kind, tuple(_near(rng, 45, 567) for _ in range(3)), rank=rng.randint(5, 20))
    if kind == "tt_compress":
        return _case(kind, tuple(_near(rng, 45, 135) for _ in range(3)), rank=rng.randint(4, 10))
    if kind == "tt_tensor":
        d = rng.choice([2, 3])
        return _case(kind, tuple(_near(rng, 45, 105) for _ in range(d)), rank=rng.randint(6, 10),
                     coeff_rank=rng.randint(2, 5), over=rng.choice([0, 0, 6]), maxit=2)
    if kind == "tucker_round":
        return _case(kind, tuple(_near(rng, 45, 243) for _ in range(3)), rank=rng.randint(5, 12))
    return _case(kind, (_near(rng, 45, 105), _near(rng, 45, 105), _near(rng, 27, 45)), count=rng.randint(4, 8),
                 workers=rng.randint(2, 4), rank=rng.randint(4, 8), maxit=2)


# ---------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------
_ctx = []


def context():
    """The process's library context on the current stream, as a program keeps one."""
    if not _ctx:
        _ctx.append(lrfg.Context(0))
    return _ctx[0]


def _k(n):
    return torch.fft.fftfreq(n, d=1.0 / n, dtype=F64, device=DEV)


def _axis(v, j, d):
    return v.reshape([-1 if a == j else 1 for a in range(d)])


def _grf(shape, seed, ell):
    """Periodic Gaussian random field of unit variance and squared-exponential covariance of length ell."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    white = torch.randn(shape, generator=gen, dtype=F64, device=DEV)
    d = len(shape)
    lam1 = [torch.exp(-2.0 * math.pi ** 2 * ell ** 2 * _k(n) ** 2) for n in shape]
    total = 1.0
    for l1 in lam1:
        total *= float(l1.sum())
    spec = torch.fft.fftn(white)
    for j, l1 in enumerate(lam1):
        spec *= _axis(torch.sqrt(l1 * shape[j]), j, d)
    return torch.fft.ifftn(spec).real / math.sqrt(total)


def _lognormal(shape, seed, var=1.0):
    return torch.exp(math.sqrt(var) * _grf(shape, seed, 0.2))


def _operand(rank):
    """Zero-mean random fields whose singular values at the bonds fall to about a fifth of the largest at `rank`: what
    a residual truncated to that rank looks like (the residuals of the low-rank iteration fill their rank)."""

    def make(shape, seed):
        g = _grf(shape, seed, 0.8 / rank)
        return g - g.mean()

    return make


def _tt_svd(x, r):
    """TT-SVD of a grid to ranks r."""
    shape, cores, a = x.shape, [], 1
    for n in shape[:-1]:
        m = x.reshape(a * n, -1)
        u, s, vh = torch.linalg.svd(m, full_matrices=False)
        k = min(r, s.numel())
        cores.append(u[:, :k].reshape(a, n, k).contiguous())
        x = s[:k, None] * vh[:k]
        a = k
    cores.append(x.reshape(a, shape[-1], 1).contiguous())
    return cores


def _refine(core, n):
    """A carriage or factor (a, m, b) on the grid of n >= m points by band-limited interpolation along its mode."""
    m = core.shape[1]
    if m == n:
        return core.contiguous()
    f = torch.fft.fft(core, dim=1)
    h = (m - 1) // 2
    big = torch.zeros((core.shape[0], n, core.shape[2]), dtype=f.dtype, device=DEV)
    big[:, : h + 1] = f[:, : h + 1]
    big[:, n - h:] = f[:, m - h:]
    return (torch.fft.ifft(big, dim=1).real * (n / m)).contiguous()


def _tt_of(make, shape, seed, r):
    """Rank-r tensor train on `shape` of a random field resolved on a coarser grid (the fields are smooth)."""
    coarse = tuple(min(n, 63) for n in shape)
    return [_refine(c, n) for c, n in zip(_tt_svd(make(coarse, seed), r), shape)]


def _unfold(x, j):
    return x.movedim(j, 0).reshape(x.shape[j], -1)


def _tucker_of(make, shape, seed, r):
    coarse = tuple(min(n, 63) for n in shape)
    x = make(coarse, seed)
    facs = [torch.linalg.svd(_unfold(x, j), full_matrices=False)[0][:, :r] for j in range(len(shape))]
    core = x
    for j, f in enumerate(facs):
        core = torch.tensordot(core, f, dims=([0], [0]))  # the contracted mode goes to the back: order restored
    return core.contiguous(), [_refine(f[None].contiguous(), n)[0].contiguous() for f, n in zip(facs, shape)]


def _step_pair(case, seed, of):
    """An iterate u, a residual r a tenth of its size, and a step length."""
    n, rank = _grid(case), int(case["rank"])
    return of(_operand(rank), n, seed, rank), of(_operand(rank), n, seed + 7919, rank), 0.1


def _tt_sum(x, y, w):
    """x + w y in block form."""
    out, d = [], len(x)
    for j, (a, b) in enumerate(zip(x, y)):
        if j == 0:
            out.append(torch.cat([a, w * b], dim=2))
        elif j == d - 1:
            out.append(torch.cat([a, b], dim=0))
        else:
            c = torch.zeros((a.shape[0] + b.shape[0], a.shape[1], a.shape[2] + b.shape[2]), dtype=F64, device=DEV)
            c[: a.shape[0], :, : a.shape[2]] = a
            c[a.shape[0]:, :, a.shape[2]:] = b
            out.append(c)
    return [c.contiguous() for c in out]


def _tucker_sum(x, y, w):
    (cx, fx), (cy, fy) = x, y
    core = torch.zeros([a + b for a, b in zip(cx.shape, cy.shape)], dtype=F64, device=DEV)
    core[tuple(slice(0, a) for a in cx.shape)] = cx
    core[tuple(slice(a, None) for a in cx.shape)] = w * cy
    return core, [torch.cat([a, b], dim=1).contiguous() for a, b in zip(fx, fy)]


def _requests(case, seed):
    """A burst: every second request a 2D full-format solve, the others low-rank solves with their coefficient as
    grid values (2D) or tensor-train carriages (3D), all in host memory."""
    n0, n1, n2 = _grid(case)
    reqs = []
    for i in range(int(case["count"])):
        s = seed + 101 * i
        if i % 2 == 0:
            reqs.append((_lognormal((n0, n1), s).cpu().numpy(), [1.0, 0.0], dict(fmt=lrfg.FULL, tol=1e-8)))
        else:
            lr = dict(fmt=lrfg.TT, rank=int(case["rank"]), tol=1e-12, maxit=int(case["maxit"]), stop_on_increase=False)
            if i % 4 == 1:
                reqs.append((_lognormal((n1, n0), s).cpu().numpy(), [0.0, 1.0], dict(lr, coeff_rank=6)))
            else:
                cores = [c.cpu().numpy() for c in _tt_of(_lognormal, (n2, n2, n2), s, 3)]
                reqs.append((cores, [0.0, 0.0, 1.0], lr))
    return reqs


def prepare(case, seed):
    kind, n, ctx, seed = case["kind"], _grid(case), context(), int(seed)
    st = {"kind": kind, "ctx": ctx}
    if kind == "full_solve":
        st["P"] = ctx.problem(_lognormal(n, seed), lrfg.FULL, tol=float(case["tol"]),
                              prec=lrfg.MIXED if case["prec"] == "mixed" else lrfg.FP64)
        st["E"] = [1.0] + [0.0] * (len(n) - 1)
        st["want"] = case["prec"] == "fp64"
    elif kind == "full_apply":
        st["P"] = ctx.problem(_lognormal(n, seed), lrfg.FULL, B=ANISO[len(n)] if case["aniso"] else None,
                              disc=lrfg.GA if case["disc"] == "ga" else lrfg.GANI)
        st["v"] = ctx.field_from_full(_operand(15)(n, seed + 7919))
    elif kind == "tt_apply":
        a = lrfg.TTensor(_tt_of(_lognormal, n, seed, int(case["coeff_rank"])))
        st["P"] = ctx.problem(a, lrfg.TT, rank=int(case["rank"]), sketch_over=int(case["over"]))
        st["v"] = ctx.field_from_tt(lrfg.TTensor(_tt_of(_operand(int(case["rank"])), n, seed + 7919, int(case["rank"]))))
    elif kind == "tt_tensor":
        a = lrfg.TTensor(_tt_of(_lognormal, n, seed, int(case["coeff_rank"])))
        st["P"] = ctx.problem(a, lrfg.TT, rank=int(case["rank"]), sketch_over=int(case["over"]), tol=1e-12,
                              maxit=int(case["maxit"]), stop_on_increase=False)
    elif kind == "tt_round":
        u, r, st["w"] = _step_pair(case, seed, _tt_of)
        st["u"], st["r"], st["rank"] = lrfg.TTensor(u), lrfg.TTensor(r), int(case["rank"])
    elif kind == "tucker_round":
        u, r, w = _step_pair(case, seed, _tucker_of)
        st["x"], st["rank"] = lrfg.TuckerTensor(*_tucker_sum(u, r, w)), int(case["rank"])
    elif kind == "tt_compress":
        st["values"], st["rank"] = _lognormal(n, seed), int(case["rank"])
    else:
        st["B"] = lrfg.Batch(0, workers=int(case["workers"]))
        st["reqs"] = _requests(case, seed)
    return st


def run(st):
    kind, ctx = st["kind"], st["ctx"]
    if kind == "full_solve":
        res, u = st["P"].solve(st["E"], want_field=st["want"])
        return {"Aeff": res.Aeff, "iters": res.iters, "u": u.full(device=True)} if st["want"] else {"Aeff": res.Aeff}
    if kind in ("full_apply", "tt_apply"):
        return st["P"].apply(st["v"]).full(device=True)
    if kind == "tt_tensor":
        return st["P"].aeff_tensor()
    if kind == "tt_round":
        y = ctx.tt_round(ctx.tt_add(1.0, st["u"], st["w"], st["r"]), st["rank"])
        return _small_grid(ctx, y)
    if kind == "tucker_round":
        y = ctx.tucker_round(st["x"], st["rank"])
        return ctx.field_from_tucker(y).full(device=True)
    if kind == "tt_compress":
        return ctx.tt_expand(ctx.tt_compress(st["values"], st["rank"]))
    B = st["B"]
    tickets = [B.submit(c, E, **kw) for c, E, kw in st["reqs"]]
    res = [B.wait(t).result for t in tickets]
    return {"Aeff": np.array([r.Aeff for r in res]), "iters": np.array([r.iters for r in res])}


def _ninth(core):
    q = (core.shape[1] + 8) // 9
    return core[:, : 9 * (q - (q + 1) % 2): 9].contiguous()  # an odd number of points, as every grid


def _small_grid(ctx, y):
    """The train's values on every ninth point of each axis (the whole grid of a large train is never formed by a
    low-rank program)."""
    return ctx.tt_expand(lrfg.TTensor([_ninth(c) for c in y.cores]))


def work(case):
    """Inputs read once, outputs written once; the floating-point work of the method at these sizes."""
    kind, n = case["kind"], _grid(case)
    d, pts = len(n), math.prod(n)
    half = pts // n[-1] * ((n[-1] + 1) // 2)
    fft = 2.5 * pts * math.log2(pts)  # one real transform
    if kind in ("full_apply", "full_solve"):
        w = 4 if case.get("prec") == "mixed" else 8
        if case.get("disc") == "ga":
            m = math.prod(2 * q - 1 for q in n)
            return {"bytes": 2 * 16 * half + 8 * m + 8 * pts, "flops": d * 2 * 2.5 * m * math.log2(m)}
        one = {"bytes": 2 * 2 * w * half + w * pts, "flops": 2 * d * fft}
        steps = (25 if w == 4 else 50) if kind == "full_solve" else 1
        return {"bytes": one["bytes"] + (16 * half if w == 8 else 0), "flops": one["flops"] * steps}
    if kind == "serve":
        q = n[0] * n[1]
        return {"bytes": 8.0 * q * case["count"], "flops": case["count"] / 2 * 50 * 4 * 2.5 * q * math.log2(q)}
    r = int(case["rank"])
    if kind == "tt_compress":
        return {"bytes": 16.0 * pts, "flops": 2.0 * pts * n[0]}
    if kind == "tucker_round":
        return {"bytes": 8.0 * (sum(n) * 3 * r + 9 * r ** 3 + pts), "flops": sum(12.0 * q * r * r for q in n) + 2.0 * pts * r}
    one = sum(q for q in (n[1:-1] if d == 3 else [])) * r * r + (n[0] + n[-1]) * r
    if kind == "tt_round":
        return {"bytes": 8.0 * 3 * one, "flops": 2.0 * one * (2 * r) * 8}
    ra, l = int(case["coeff_rank"]), r + int(case["over"])
    mid = n[1] if d == 3 else 0
    per = d * 4.0 * (mid * l * ra * r * (ra + r) + (mid * l + n[0]) * l * l) + 4.0 * 10 * mid * r * r * l
    if kind == "tt_tensor":
        k = d * (d + 1) // 2
        return {"bytes": 8.0 * (mid * ra * ra + (n[0] + n[-1]) * ra), "flops": k * per * 2 * int(case["maxit"])}
    return {"bytes": 8.0 * (2 * one + mid * ra * ra + (n[0] + n[-1]) * ra + pts), "flops": per + 2.0 * pts * r}


# ---------------------------------------------------------------------------------------------------------------
# the same results in FP64 with plain torch
# ---------------------------------------------------------------------------------------------------------------
def _freqs(n):
    """Frequencies along each axis of the half spectrum of a real grid, shaped to broadcast."""
    d = len(n)
    ks = [_k(q) for q in n]
    ks[-1] = torch.arange((n[-1] + 1) // 2, dtype=F64, device=DEV)
    return [_axis(k, j, d) for j, k in enumerate(ks)]


def _inv_kk(n):
    kk = sum(k ** 2 for k in _freqs(n))
    return torch.where(kk > 0, 1.0 / torch.clamp(kk, min=1.0), torch.zeros_like(kk))


def _full_operator(a, n, B=None):
    """v^ -> grad^* F (a I + B) F^-1 grad^ v^ on half spectra."""
    ks = _freqs(n)

    def op(v):
        out = torch.zeros_like(v)
        for k in ks:
            out -= 2j * math.pi * k * torch.fft.rfftn(a * torch.fft.irfftn(2j * math.pi * k * v, s=n))
        if B is not None:
            q = sum(float(B[i][j]) * ks[i] * ks[j] for i in range(len(n)) for j in range(len(n)))
            out += 4.0 * math.pi ** 2 * q * v
        return out

    return op


def _ga_operator(a, n, B=None):
    """The same with the exact integration of the voxel-wise constant a: the product on the double grid M."""
    d, M = len(n), tuple(2 * q - 1 for q in n)
    N_tot, M_tot = math.prod(n), math.prod(M)
    spec = torch.fft.fftn(a)
    for j, (q, m) in enumerate(zip(n, M)):
        f = _k(m)
        spec = spec.index_select(j, torch.remainder(f.round().long(), q))
        x = math.pi * f
        s = torch.where(f == 0, torch.full_like(f, 1.0 / q), torch.sin(x / q) / torch.where(f == 0, torch.ones_like(f), x))
        spec = spec * _axis(s, j, d)
    a_ga = torch.fft.ifftn(spec).real * (N_tot / M_tot)
    at = [torch.remainder(_k(q).round().long(), m) for q, m in zip(n, M)]
    at[-1] = torch.arange((n[-1] + 1) // 2, device=DEV)
    half_m = M[:-1] + ((M[-1] + 1) // 2,)
    where = torch.meshgrid(*at, indexing="ij")
    ks = _freqs(n)

    def op(v):
        out = torch.zeros_like(v)
        for k in ks:
            up = torch.zeros(half_m, dtype=v.dtype, device=DEV)
            up[where] = 2j * math.pi * k * v / N_tot
            e = torch.fft.irfftn(up, s=M) * M_tot
            out -= 2j * math.pi * k * torch.fft.rfftn(a_ga * e)[where]
        if B is not None:
            q = sum(float(B[i][j]) / M_tot * ks[i] * ks[j] for i in range(d) for j in range(d))
            out += 4.0 * math.pi ** 2 * q * v
        return out

    return op


def _dot(x, y):
    """Real inner product over the full spectrum from half spectra."""
    w = torch.full((x.shape[-1],), 2.0, dtype=F64, device=DEV)
    w[0] = 1.0
    return float(((x.real * y.real + x.imag * y.imag) * w).sum())


def _full_solution(a, n):
    """u^ of the cell problem for E = e_1 by conjugate gradients to the rounding level, and A_eff."""
    op, p_inv, ks = _full_operator(a, n), _inv_kk(n), _freqs(n)
    r = 2j * math.pi * ks[0] * torch.fft.rfftn(a)
    u = torch.zeros_like(r)
    z = p_inv * r
    p, rz = z, _dot(r, z)
    stop = rz * 1e-26
    for _ in range(400):
        q = op(p)
        al = rz / _dot(p, q)
        u = u + al * p
        r = r - al * q
        z = p_inv * r
        new = _dot(r, z)
        if new <= stop:
            break
        p, rz = z + (new / rz) * p, new
    val = 0.0
    for j, k in enumerate(ks):
        e = torch.fft.irfftn(2j * math.pi * k * u, s=n) + (1.0 if j == 0 else 0.0)
        val += float((a * e * e).mean())
    return u, val


def _dmode(core):
    """The derivative of a carriage along its mode."""
    k = _k(core.shape[1])[None, :, None]
    return torch.fft.ifft(2j * math.pi * k * torch.fft.fft(core, dim=1), dim=1).real


def _expsum(n, eps=0.1):
    """Nodes and weights of the exponential sum of 1/x on [1, sum ((n-1)/2)^2] (trapezoidal rule)."""
    xmax = float(sum(((q - 1) // 2) ** 2 for q in n))
    h = math.pi ** 2 / math.log(32.0 / eps)
    lo, hi = math.log(eps / (2.0 * xmax)), math.log(math.log(2.0 / eps))
    taus = [lo + h * m for m in range(math.ceil((hi - lo) / h) + 1)]
    return [math.exp(t) for t in taus], [h * math.exp(t) for t in taus]


def _gauss(core, t):
    k = _k(core.shape[1])[None, :, None]
    return torch.fft.ifft(torch.exp(-t * k * k) * torch.fft.fft(core, dim=1), dim=1).real


def _kr(x, y):
    return torch.einsum("inj,knl->iknjl", x, y).reshape(x.shape[0] * y.shape[0], x.shape[1], x.shape[2] * y.shape[2])


def _round(cores, r):
    """TT rounding: orthogonalise from the right, truncated SVDs from the left."""
    c = list(cores)
    for j in range(len(c) - 1, 0, -1):
        a, n, b = c[j].shape
        q, t = torch.linalg.qr(c[j].reshape(a, n * b).T)
        c[j] = q.T.reshape(-1, n, b)
        c[j - 1] = torch.einsum("anb,cb->anc", c[j - 1], t)
    for j in range(len(c) - 1):
        a, n, b = c[j].shape
        u, s, vh = torch.linalg.svd(c[j].reshape(a * n, b), full_matrices=False)
        k = min(r, s.numel())
        c[j] = u[:, :k].reshape(a, n, k)
        c[j + 1] = torch.einsum("ab,bnc->anc", s[:k, None] * vh[:k], c[j + 1])
    return c


def _signs(n, ell, seed=0):
    """The Rademacher sketch: carriage j's entry t is the top bit of output (j + 1) 2^40 + t of SplitMix64."""
    d, out = len(n), []
    r = [1] + [ell] * (d - 1) + [1]
    for j, q in enumerate(n):
        with np.errstate(over="ignore"):
            i = (np.uint64(j + 1) << np.uint64(40)) + np.arange(r[j] * q * r[j + 1], dtype=np.uint64)
            z = np.uint64(seed) + (i + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z = z ^ (z >> np.uint64(31))
        s = np.where(z >> np.uint64(63), -1.0, 1.0).reshape(r[j], q, r[j + 1])
        out.append(torch.as_tensor(s, device=DEV))
    return out


def _round_sketch(z, om, r):
    """Randomised rounding: sketch from the right, orthogonalise from the left, truncated SVDs from the right."""
    d = len(z)
    W = [None] * (d + 1)
    W[d] = torch.ones((1, 1), dtype=F64, device=DEV)
    for j in range(d - 1, 0, -1):
        W[j] = torch.einsum("anb,lnb->al", torch.einsum("anb,bc->anc", z[j], W[j + 1]), om[j])
    c, x = [], z[0]
    for j in range(d - 1):
        a, n, _ = x.shape
        q, _ = torch.linalg.qr(x.reshape(a * n, -1) @ W[j + 1])
        m = q.T @ x.reshape(a * n, -1)
        c.append(q.reshape(a, n, -1))
        x = torch.einsum("ab,bnc->anc", m, z[j + 1])
    c.append(x)
    wgt = torch.ones(1, dtype=F64, device=DEV)
    for j in range(d - 1, 0, -1):
        a, n, b = c[j].shape
        u, s, _ = torch.linalg.svd((c[j] * wgt).reshape(a, n * b), full_matrices=False)
        k = min(r, s.numel())
        u, wgt = u[:, :k], s[:k]
        c[j] = torch.einsum("ak,anb->knb", u, c[j])
        c[j - 1] = torch.einsum("anb,bk->ank", c[j - 1], u)
    return c


def _expand(c):
    x = c[0].reshape(c[0].shape[1], -1)
    for core in c[1:]:
        x = (x @ core.reshape(core.shape[0], -1)).reshape(-1, core.shape[2])
    return x.reshape([core.shape[1] for core in c])


def _blocks(terms):
    """Block-diagonal sum of tensor trains."""
    out = terms[0]
    for t in terms[1:]:
        out = _tt_sum(out, t, 1.0)
    return out


def _tt_operator(a, v, r, over):
    """T P~^-1 T sum_j -D_j T(a (.) D_j v) with the truncations the options ask for."""
    d, n = len(v), [c.shape[1] for c in v]
    om = _signs(n, r + over) if over else None
    cut = (lambda x: _round_sketch(x, om, r)) if over else (lambda x: _round(x, r))
    terms = []
    for j in range(d):
        w = cut([_kr(x, _dmode(y) if i == j else y) for i, (x, y) in enumerate(zip(a, v))])
        w[j] = -_dmode(w[j])
        terms.append(w)
    s = _round(_blocks(terms), r)
    ts, ws = _expsum(n)
    return cut(_blocks([[(w if i == 0 else 1.0) * _gauss(c, t) for i, c in enumerate(s)] for t, w in zip(ts, ws)]))


def _tucker_round(core, facs, r):
    d, qs = len(facs), []
    for j, f in enumerate(facs):
        q, t = torch.linalg.qr(f)
        qs.append(q)
        core = torch.tensordot(core, t, dims=([0], [1]))
    us = [torch.linalg.svd(_unfold(core, j), full_matrices=False)[0][:, :r] for j in range(d)]
    for u in us:
        core = torch.tensordot(core, u, dims=([0], [0]))
    return core, [q @ u for q, u in zip(qs, us)]


def exact(case, seed):
    kind, n, seed = case["kind"], _grid(case), int(seed)
    if kind == "full_solve":
        u, val = _full_solution(_lognormal(n, seed), n)
        full = {"Aeff": val, "iters": None, "u": torch.fft.irfftn(u, s=n)}
        return full if case["prec"] == "fp64" else {"Aeff": val}
    if kind == "full_apply":
        a, v = _lognormal(n, seed), torch.fft.rfftn(_operand(15)(n, seed + 7919))
        B = ANISO[len(n)] if case["aniso"] else None
        op = (_ga_operator if case["disc"] == "ga" else _full_operator)(a, n, B)
        return torch.fft.irfftn(_inv_kk(n) * op(v), s=n)
    if kind == "tt_apply":
        a = _tt_of(_lognormal, n, seed, int(case["coeff_rank"]))
        v = _tt_of(_operand(int(case["rank"])), n, seed + 7919, int(case["rank"]))
        return _expand(_tt_operator(a, v, int(case["rank"]), int(case["over"])))
    if kind == "tt_round":
        u, r, w = _step_pair(case, seed, _tt_of)
        return _expand([_ninth(c) for c in _round(_tt_sum(u, r, w), int(case["rank"]))])
    if kind == "tucker_round":
        u, r, w = _step_pair(case, seed, _tucker_of)
        core, facs = _tucker_round(*_tucker_sum(u, r, w), int(case["rank"]))
        for f in facs:
            core = torch.tensordot(core, f, dims=([0], [1]))
        return core
    if kind == "tt_compress":
        return _expand(_tt_svd(_lognormal(n, seed), int(case["rank"])))
    return None  # iterations of several solves: compared with the start's alone
