"""The calls that a user of this library makes, over the range of lattices that it is used on.

    listed()            the cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) what the caller holds before the call: links in device or host memory, the context
    run(state)          one pass through the public entry points
    work(case)          the bytes and operations that the pass cannot do without
    exact(case, seed)   the same outputs in plain torch float64

Links are complex128 (4, Nt, Nz, Ny, Nx, 3, 3); extents are given as (nx, ny, nz, nt).
"""
import math

import torch

import paper_1210_8018_gb300 as lgf

ALPHA = 0.08   # the paper's step
EPS = 1e-15    # the paper's stopping criterion
MAX_ITER = 400
DEVICE = "cuda"

# Sites of the largest drawn case of each kind, and of the smallest.
SITES = {"fix": (2048, 64 ** 4), "fix_fp64": (2048, 2 ** 20), "fix_host": (2 ** 15, 2 ** 20), "ensemble": (4096, 2 ** 17),
         "functional": (4096, 2 ** 20), "measure": (4096, 2 ** 23), "delta": (4096, 2 ** 22), "transform": (4096, 2 ** 21)}
EXTENTS = [6, 8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 54, 60, 64, 72, 80, 96]


def _case(name, kind, dims, precision="fp64", rough=0.6, host=False, count=1):
    c = {"kind": kind, "nx": dims[0], "ny": dims[1], "nz": dims[2], "nt": dims[3], "precision": precision,
         "rough": rough, "host": host, "count": count}
    return dict(c, name=name) if name else c


def listed():
    return [
        # Whole gauge fixings to theta < 1e-15. The benchmark's own: one 64^4 configuration, mixed schedule.
        _case("fix_mixed_64x4", "fix", (64, 64, 64, 64), "mixed"),
        # The paper's lattice.
        _case("fix_mixed_32x4", "fix", (32, 32, 32, 32), "mixed"),
        # The smallest lattice of the tests: launches and host round trips count.
        _case("fix_mixed_8x4", "fix", (8, 8, 8, 8), "mixed", 0.3),
        # Unequal extents with factors 3 and 5: the passes for general lengths, blocks that do not divide.
        _case("fix_mixed_30x20x24x36", "fix", (30, 20, 24, 36), "mixed", 0.5),
        # The default precision on a shape of the benchmark's ensemble, and on a small ragged lattice.
        _case("fix_fp64_24x24x24x48", "fix", (24, 24, 24, 48), "fp64"),
        _case("fix_fp64_18x12x10x15", "fix", (18, 12, 10, 15), "fp64", 0.5),
        # Configurations read from disk: page-locked host memory in and out.
        _case("fix_host_16x16x16x32", "fix", (16, 16, 16, 32), "mixed", 0.6, True),
        # An ensemble of equal lattices fixed together.
        _case("ensemble_6_of_16x4", "ensemble", (16, 16, 16, 16), "fp64", 0.5, False, 6),
        # One step of gradient-based fixing: F_U[exp(i omega)], its su(3) gradient, and the gradient
        # preconditioned by the Fourier filter (what adam_fix does in a step); the benchmark's 24^4.
        _case("functional_24x4", "functional", (24, 24, 24, 24), "fp64", 0.5),
        # theta, F and the plaquette of a configuration (the checks before and after a fixing).
        _case("measure_48x48x48x40", "measure", (48, 48, 48, 40)),
        # Delta(x) itself, for observables built on it; extents with a factor 5.
        _case("delta_40x40x40x20", "delta", (40, 40, 40, 20)),
        # A gauge transformation g(x) U g^+(x + mu) in double precision (gauge copies, re-basing).
        _case("transform_32x4", "transform", (32, 32, 32, 32)),
    ]


def _extents(rng, lo, hi):
    """Four extents with a volume in [lo, hi], spread over its logarithm; every other one is L^3 x T."""
    while True:
        target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = target ** 0.25
        near = [n for n in EXTENTS if side / 2.1 <= n <= side * 2.1]
        if not near:
            continue
        if rng.random() < 0.5:
            n = rng.choice(near)
            d = (n, n, n, rng.choice(near))
        else:
            d = tuple(rng.choice(near) for _ in range(4))
        v = d[0] * d[1] * d[2] * d[3]
        if lo <= v <= hi and target / 3 <= v <= target * 3:
            return d


def draw(rng):
    kind = rng.choice(["fix", "fix", "fix", "fix_fp64", "fix_host", "ensemble", "functional", "measure", "delta", "transform"])
    dims = _extents(rng, *SITES[kind])
    rough = round(rng.uniform(0.3, 0.65), 3)
    if kind == "fix":
        return _case(None, "fix", dims, "mixed", rough)
    if kind == "fix_fp64":
        return _case(None, "fix", dims, "fp64", rough)
    if kind == "fix_host":
        return _case(None, "fix", dims, rng.choice(["mixed", "fp64"]), rough, True)
    if kind == "ensemble":
        return _case(None, "ensemble", dims, "fp64", rough, False, rng.randint(2, 8))
    return _case(None, kind, dims, "fp64", rough)


def _dims(case):
    return (case["nx"], case["ny"], case["nz"], case["nt"])


def _sites(case):
    return case["nx"] * case["ny"] * case["nz"] * case["nt"]


# ---------------------------------------------------------------------------------------------------
# Inputs: U_mu(x) = h(x) V_mu(x) h^+(x + mu), h Haar-random on SU(3) and V near exp(i rough A), A Gaussian
# over the generators: a rough configuration in a random gauge, as a Monte-Carlo code leaves it. Each site
# draws its h and V from 2^16 matrices of the seed, so that a large lattice is made quickly.
# ---------------------------------------------------------------------------------------------------
def _su3(m):
    """Gram-Schmidt of rows 0 and 1, row 2 = conj(row0 x row1)."""
    r0 = m[..., 0, :]
    r0 = r0 / torch.linalg.vector_norm(r0, dim=-1, keepdim=True)
    r1 = m[..., 1, :]
    r1 = r1 - (r0.conj() * r1).sum(-1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    return torch.stack((r0, r1, torch.linalg.cross(r0, r1, dim=-1).conj()), dim=-2)


def _haar(n, gen):
    return _su3(torch.randn(n, 3, 3, dtype=torch.complex128, device=DEVICE, generator=gen))


def _near_one(n, scale, gen):
    """Near exp(i scale A) with A = sum_a A^a lambda^a / (2 sqrt 2), A^a ~ N(0, 1)."""
    z = torch.randn(n, 3, 3, dtype=torch.complex128, device=DEVICE, generator=gen)
    one = torch.eye(3, dtype=z.dtype, device=z.device)
    x = (z - z.mH) * (scale / math.sqrt(8.0))
    x = x - torch.diagonal(x, dim1=-2, dim2=-1).mean(-1)[..., None, None] * one
    return _su3(one + x + x @ x / 2)


def _forward(f, mu):
    """f(x + mu) of a site field (Nt, Nz, Ny, Nx, ...)."""
    return torch.roll(f, -1, dims=3 - mu)


def _site_matrices(dims, pool, gen):
    return pool[torch.randint(pool.shape[0], dims[::-1], device=DEVICE, generator=gen)]


def _links(dims, rough, gen):
    nx, ny, nz, nt = dims
    U = torch.empty(4, nt, nz, ny, nx, 3, 3, dtype=torch.complex128, device=DEVICE)
    h = _site_matrices(dims, _haar(1 << 16, gen), gen)
    near = _near_one(1 << 16, rough, gen)
    for mu in range(4):
        U[mu] = h @ _site_matrices(dims, near, gen) @ _forward(h, mu).mH
    return U


def _gen(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed))


def _inputs(case, seed):
    gen, dims = _gen(seed), _dims(case)
    links = [_links(dims, case["rough"], gen) for _ in range(case["count"])]
    more = None
    if case["kind"] == "functional":
        more = torch.randn(_sites(case), 8, dtype=torch.float64, device=DEVICE, generator=gen) * 0.05
    elif case["kind"] == "transform":
        more = _site_matrices(dims, _haar(1 << 16, gen), gen)
    return links, more


def prepare(case, seed):
    links, more = _inputs(case, seed)
    dims, kind = _dims(case), case["kind"]
    s = {"case": dict(case), "links": links, "more": more}
    if kind == "ensemble":
        s["batch"] = lgf.Batch([dims] * case["count"])
        s["out"] = [torch.empty_like(U) for U in links]
        return s
    s["lattice"] = lgf.Lattice(dims)
    if kind == "fix":
        if case["host"]:
            s["links"] = [torch.empty(U.shape, dtype=U.dtype, pin_memory=True).copy_(U) for U in links]
            s["out"] = torch.empty(links[0].shape, dtype=links[0].dtype, pin_memory=True)
        else:
            s["out"] = torch.empty_like(links[0])
    elif kind == "functional":
        s["more"] = more.requires_grad_(True)
        s["out"] = torch.empty_like(more)
    elif kind == "delta":
        s["out"] = torch.empty_like(links[0][0])
    elif kind == "transform":
        s["out"] = torch.empty_like(links[0])
    return s


def run(s):
    case, kind, U = s["case"], s["case"]["kind"], s["links"][0]
    if kind == "ensemble":
        for out, U in zip(s["out"], s["links"]):
            out.copy_(U)
        r = s["batch"].fix(s["out"], ALPHA, EPS, case["precision"], max_iter=MAX_ITER)
        return {"links": s["out"], "F": [c["F"] for c in r], "theta": [c["theta"] for c in r], "iters": [c["iters"] for c in r]}
    lat = s["lattice"]
    if kind == "fix":
        lat.load(U, case["precision"])
        r = lat.iterate(MAX_ITER, ALPHA, EPS)
        lat.store(s["out"])
        return {"links": s["out"], "F": r["F"], "theta": r["theta"], "iters": r["iters"]}
    if kind == "functional":
        F = lgf.LandauF().apply(s["more"], U, lat)
        grad, = torch.autograd.grad(-24.0 * _sites(case) * F, s["more"])
        lat.filter_coeffs(grad, s["out"])
        return {"F": F, "grad": grad, "filtered": s["out"]}
    if kind == "measure":
        return lat.measure(U)
    if kind == "delta":
        theta, F = lat.delta(U, s["out"])
        return {"delta": s["out"], "theta": theta, "F": F}
    s["out"].copy_(U)
    lat.update(s["out"], s["more"])
    return {"links": s["out"]}


def work(case):
    """Each input read once and each output written once. A fixing also reads and writes the links, and does
    the operations of Delta, the transforms, g and the update, in every one of about 45 iterations: with two
    rows of a link in the precision of the schedule that iterates them."""
    V, kind = _sites(case), case["kind"]
    links = 576.0 * V
    if kind in ("fix", "ensemble"):
        it = 45.0
        real = 4 if case["precision"] == "mixed" else 8
        fft = 4 * 2 * 5 * math.log2(V)          # four complex fields, there and back
        site = 4 * 24 * 8 + 8 * 30 + 150 + fft  # update, Delta, g
        n = case["count"]
        return {"bytes": n * (2 * links + it * V * 2 * 4 * 12 * real), "flops": n * it * V * site}
    if kind == "functional":
        return {"bytes": links + 4 * 64.0 * V, "flops": V * (4 * 216 + 8 * 216 + 6 * 216 + 500 + 4 * 10 * math.log2(V))}
    if kind == "measure":
        return {"bytes": links, "flops": V * (8 * 18 + 6 * 2 * 216 + 6 * 36)}
    if kind == "delta":
        return {"bytes": links + 144.0 * V, "flops": V * 8 * 18}
    return {"bytes": 2 * links + 144.0 * V, "flops": V * 4 * 2 * 216}


# ---------------------------------------------------------------------------------------------------
# The same in plain torch.
# ---------------------------------------------------------------------------------------------------
def _delta(U):
    B = torch.zeros_like(U[0])
    for mu in range(4):
        B += torch.roll(U[mu], 1, dims=3 - mu) - U[mu]
    D = B - B.mH
    tr = torch.diagonal(D, dim1=-2, dim2=-1).mean(-1)
    return D - tr[..., None, None] * torch.eye(3, dtype=D.dtype, device=D.device)


def _theta(D):
    return float((D.abs() ** 2).sum() / (3 * D[..., 0, 0].numel()))


def _trace(U):
    return float(torch.diagonal(U, dim1=-2, dim2=-1).real.sum() / (3 * U[..., 0, 0].numel()))


def _weights(shape):
    """p^2_max / p^2 on the momenta of a field (Nt, Nz, Ny, Nx), 0 at zero momentum."""
    p2, top = torch.zeros(shape, dtype=torch.float64, device=DEVICE), 0.0
    for ax, n in enumerate(shape):
        k = torch.arange(n, dtype=torch.float64, device=DEVICE)
        p2 += (4 * torch.sin(math.pi * k / n) ** 2).reshape([-1 if a == ax else 1 for a in range(4)])
        top += 4 * math.sin(math.pi * (n // 2) / n) ** 2
    w = top / p2
    w[0, 0, 0, 0] = 0
    return w


def _filter(f, w):
    """Filters a field (Nt, Nz, Ny, Nx, ...), its components one at a time."""
    flat = f.reshape(*f.shape[:4], -1)
    out = torch.empty_like(flat)
    for j in range(flat.shape[-1]):
        k = torch.fft.fft(torch.fft.fftn(flat[..., j], dim=(1, 2, 3)), dim=0) * w
        k = torch.fft.ifftn(torch.fft.ifft(k, dim=0), dim=(1, 2, 3))
        out[..., j] = k if f.is_complex() else k.real
    return out.reshape(f.shape)


def _transform(U, g):
    return torch.stack([g @ U[mu] @ _forward(g, mu).mH for mu in range(4)])


def _fix(U):
    w = _weights(U.shape[1:5])
    one = torch.eye(3, dtype=U.dtype, device=U.device)
    for _ in range(MAX_ITER):
        D = _delta(U)
        if _theta(D) < EPS:
            break
        U = _transform(U, _su3(one + (ALPHA / 2) * _filter(D, w)))
    return U


def exact(case, seed):
    kind = case["kind"]
    if kind in ("fix", "ensemble"):
        if _sites(case) * case["count"] > 1 << 20:
            return None
        fixed = [_fix(U) for U in _inputs(case, seed)[0]]
        # theta at the end is what rounding and the last step leave, and the mixed schedule's links are as
        # far from the double path's as both are from the maximum: neither has a value in 64 bits.
        links = [None if case["precision"] == "mixed" else (U.cpu() if case["host"] else U) for U in fixed]
        F = [_trace(U) for U in fixed]
        if kind == "ensemble":
            return {"links": links, "F": F, "theta": None, "iters": None}
        return {"links": links[0], "F": F[0], "theta": None, "iters": None}
    (U,), more = _inputs(case, seed)
    if kind == "functional":
        V, s3 = _sites(case), 1 / math.sqrt(3.0)
        w = more.requires_grad_(True)
        o = w.reshape(*U.shape[1:5], 8)
        d0, d1, d2 = 0.5 * (o[..., 2] + s3 * o[..., 7]), 0.5 * (-o[..., 2] + s3 * o[..., 7]), -s3 * o[..., 7]
        c = [torch.complex(0.5 * o[..., a], -0.5 * o[..., a + 1]) for a in (0, 3, 5)]
        zero = torch.zeros_like(d0)
        H = torch.stack((torch.complex(d0, zero), c[0], c[1], c[0].conj(), torch.complex(d1, zero), c[2],
                         c[1].conj(), c[2].conj(), torch.complex(d2, zero)), dim=-1).reshape(*U.shape[1:5], 3, 3)
        g = torch.linalg.matrix_exp(1j * H)
        F = torch.diagonal(_transform(U, g), dim1=-2, dim2=-1).real.sum() / (12.0 * V)
        grad, = torch.autograd.grad(-24.0 * V * F, w)
        return {"F": F.detach(), "grad": grad, "filtered": _filter(grad.reshape(*U.shape[1:5], 8), _weights(U.shape[1:5])).reshape(V, 8)}
    if kind == "measure":
        D = _delta(U)
        theta = _theta(D)
        del D
        plaq = 0.0
        for mu in range(4):
            for nu in range(mu + 1, 4):
                p = U[mu] @ _forward(U[nu], mu)
                q = U[nu] @ _forward(U[mu], nu)
                plaq += float((p * q.conj()).real.sum())
                del p, q
        return {"theta": theta, "F": _trace(U), "plaquette": plaq / (18.0 * _sites(case))}
    if kind == "delta":
        D = _delta(U)
        return {"delta": D, "theta": _theta(D), "F": _trace(U)}
    return {"links": _transform(U, more)}
