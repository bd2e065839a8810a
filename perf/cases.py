"""The measured cases: what a program that uses this library has it do.

Whole solves (Algorithm 1) in both precisions, a batch of them, a differentiable solve
with its backward pass, and the single steps that custom drivers call (CG on one grid,
residual, gradient, EXP_finite, EXP_true).  Every input is made on the GPU from a seed:
a manufactured solution u (an exponential, a corner singularity r^{5/3} or a sum of sines,
with seeded coefficients) and its right-hand side f = u_xx + u_yy + u_zz.
"""
import math

import numpy as np
import torch

from paper_1507_05063_gb300 import excmg as X
from paper_1507_05063_gb300.autograd import excmg_solve


def _case(kind, N, L=(1.0, 1.0, 1.0), N0=(0, 0, 0), **more):
    c = {"kind": kind, "nx": N[0], "ny": N[1], "nz": N[2], "lx": L[0], "ly": L[1], "lz": L[2],
         "nx0": N0[0], "ny0": N0[1], "nz0": N0[2]}
    c.update(more)
    return c


def listed():
    return [
        # the smallest solve a user makes (and the smoke test's): latency and launches
        dict(_case("solve", (32, 32, 32), N0=(4, 4, 4), precision="fp64", eps=1e-8, ut=False,
                   data="sines"), name="solve_32_fp64"),
        # a production box with unequal meshsizes, with the sixth-order result
        dict(_case("solve", (512, 256, 128), N0=(8, 4, 2), precision="fp64", eps=1e-9, ut=True,
                   data="exp"), name="solve_512x256x128_fp64_ut"),
        # the largest: the mixed-precision solve of the benchmark
        dict(_case("solve", (1024, 512, 512), N0=(8, 4, 4), precision="mixed", eps=1e-9, ut=False,
                   data="corner"), name="solve_1024x512x512_mixed"),
        # a box whose cell counts are no powers of two and whose meshsizes have no simple
        # ratio; its second coarsest grid is too large for the direct solve
        dict(_case("solve", (192, 320, 224), L=(1.0, 1.5, 1.25), N0=(12, 20, 14), precision="fp64",
                   eps=1e-10, ut=False, data="exp"), name="solve_192x320x224_fp64"),
        # a tight tolerance, where the mixed mode's float32 steps do the work
        dict(_case("solve", (512, 256, 128), N0=(8, 4, 2), precision="mixed", eps=1e-12, ut=False,
                   data="exp"), name="solve_512x256x128_mixed_tight"),
        # many small problems of different shapes in one call
        dict(_case("batch", (0, 0, 0), count=16, most=128, eps=1e-8, data="sines"), name="batch_16"),
        # one gradient step of a source recovery: forward solve and adjoint
        dict(_case("adjoint", (128, 128, 128), N0=(4, 4, 4), precision="fp64", eps=1e-10,
                   data="sines"), name="adjoint_128"),
        # a custom driver's smoothing steps on one grid with odd cell counts
        dict(_case("cg", (385, 201, 121), L=(2.0, 1.0, 0.6), steps=20, data="exp"),
             name="cg_385x201x121"),
        # a driver's residual check of an iterate
        dict(_case("residual", (320, 255, 257), data="exp"), name="residual_320x255x257"),
        # the gradient of a solution
        dict(_case("grad", (512, 256, 256), L=(2.0, 1.0, 1.0), data="exp"), name="grad_512x256x256"),
        # the prolongation of two coarser solutions
        dict(_case("exp_finite", (512, 256, 128), data="exp"), name="exp_finite_512x256x128"),
        # the sixth-order extrapolation of two solutions
        dict(_case("exp_true", (384, 256, 192), data="exp"), name="exp_true_384x256x192"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "mixed", "batch", "adjoint", "cg", "residual", "grad",
                       "exp_finite", "exp_true"])
    data = rng.choice(["exp", "corner", "sines"])
    L = (1.0, rng.choice([1.0, 0.5, 1.5, 0.8]), rng.choice([1.0, 2.0, 1.25]))
    if data == "sines":
        L = (1.0, float(rng.choice([1, 2])), float(rng.choice([1, 2])))
    if kind in ("solve", "mixed"):
        k = rng.choice([3, 4]) if kind == "solve" else 5
        N0 = tuple(rng.choice([4, 6, 8, 10]) for _ in range(3))
        return _case("solve", tuple(n << k for n in N0), L, N0,
                     precision="fp64" if kind == "solve" else "mixed",
                     eps=rng.choice([1e-8, 1e-9, 1e-10]), ut=rng.random() < 0.5, data=data)
    if kind == "batch":
        return _case("batch", (0, 0, 0), count=rng.randint(3, 20), most=rng.choice([32, 64, 128]),
                     eps=1e-8, data="sines")
    if kind == "adjoint":
        N0 = tuple(rng.choice([4, 6, 8]) for _ in range(3))
        k = rng.choice([2, 3, 4])
        return _case("adjoint", tuple(n << k for n in N0), L, N0, precision="fp64", eps=1e-10, data=data)
    if kind == "cg":
        return _case("cg", tuple(_log_int(rng, 9, 400) for _ in range(3)), L, steps=rng.randint(5, 30),
                     data=data)
    if kind in ("residual", "grad"):
        return _case(kind, tuple(_log_int(rng, 9, 500) for _ in range(3)), L, data=data)
    m = 8 if kind == "exp_finite" else 2
    return _case(kind, tuple(m * max(1, _log_int(rng, 16, 512) // m) for _ in range(3)), L, data=data)


def _dims(case):
    return ((case["nx"], case["ny"], case["nz"]), (case["lx"], case["ly"], case["lz"]),
            (case["nx0"], case["ny0"], case["nz0"]))


def _axes(N, L, dev):
    """Node coordinates along x, y, z, shaped to broadcast to (Nz+1, Ny+1, Nx+1)."""
    out = []
    for d, shape in ((0, (1, 1, -1)), (1, (1, -1, 1)), (2, (-1, 1, 1))):
        c = torch.arange(N[d] + 1, dtype=torch.float64, device=dev) * (L[d] / N[d])
        out.append(c.reshape(shape))
    return out


def _manufactured(data, N, L, seed, dev):
    """(f, u) on all nodes."""
    rng = np.random.default_rng(seed)
    x, y, z = _axes(N, L, dev)
    if data == "exp":
        a = rng.uniform(0.5, 1.2, 3)
        c = float(rng.uniform(0.5, 1.5))
        u = (c * torch.exp(a[0] * x)) * torch.exp(a[1] * y) * torch.exp(a[2] * z)
        return float(a @ a) * u, u
    if data == "corner":
        # c r^{5/3}, r the distance from the corner; f = c (40/9) r^{-1/3}, 0 at the corner
        c = float(rng.uniform(0.5, 1.5))
        r2 = (x * x + y * y) + z * z
        u = c * r2 ** (5.0 / 6.0)
        r2.reshape(-1)[0] = 1.0
        f = (c * 40.0 / 9.0) * r2 ** (-1.0 / 6.0)
        f.reshape(-1)[0] = 0.0
        return f, u
    # sum of products of sines that vanish on the boundary of a box with integer sides
    f = u = 0.0
    for _ in range(8):
        a = float(rng.standard_normal())
        m = rng.integers(1, 9, 3)
        t = torch.sin(m[0] * math.pi * x) * torch.sin(m[1] * math.pi * y) * torch.sin(m[2] * math.pi * z)
        f = f + a * t
        u = u - (a / (math.pi ** 2 * float(m @ m))) * t
    u[0], u[-1] = 0.0, 0.0
    u[:, 0], u[:, -1] = 0.0, 0.0
    u[:, :, 0], u[:, :, -1] = 0.0, 0.0
    return f.contiguous(), u.contiguous()


def _batch_grids(case, seed):
    """Grids of a batch: each side a power of two, each box side 1 or 2, the coarsest grid's
    smallest side 4.  They are the same for every seed: a user's batch has its shapes."""
    rng = np.random.default_rng(case["count"] * 1000 + case["most"])
    sizes = [s for s in (32, 64, 128) if s <= case["most"]]
    out = []
    for _ in range(case["count"]):
        N = tuple(int(v) for v in rng.choice(sizes, size=3))
        L = tuple(float(v) for v in rng.integers(1, 3, size=3))
        k = int(math.log2(min(N))) - 2
        out.append((L, N, tuple(n >> k for n in N)))
    return out


def _solve_opts(case):
    return {"precision": case["precision"], "eps": case["eps"]}


def _noise(shape, seed, dev):
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) + 77)
    return torch.randn(shape, dtype=torch.float64, device=dev, generator=gen)


def _coarser(data, N, L, seed, dev):
    """Two FD-like solutions: u + A h^4 on the grids of N and N / 2 cells."""
    out = []
    for s, amp in ((1, 1e-4), (2, 16e-4)):
        n = tuple(v // s for v in N)
        _, u = _manufactured(data, n, L, seed, dev)
        x, y, z = _axes(n, L, dev)
        out.append(u + amp * (1.0 + 0.3 * x) * (1.0 - 0.2 * y) * (1.0 + 0.1 * z))
    return out


def _inputs(case, seed, dev):
    """The input tensors of a case (the same for run and exact)."""
    N, L, _ = _dims(case)
    kind, data = case["kind"], case["data"]
    if kind == "batch":
        got = []
        for i, (Li, Ni, _N0) in enumerate(_batch_grids(case, seed)):
            f, _u = _manufactured("sines", Ni, Li, 100 * seed + i, dev)
            got.append((f, torch.zeros_like(f)))
        return {"problems": got}
    if kind in ("solve", "adjoint"):
        f, g = _manufactured(data, N, L, seed, dev)
        s = {"f": f, "g": g}
        if kind == "adjoint":
            # dL/du of L = |u - target|^2 / 2 for a target off by a smooth field and noise
            s["dLdu"] = 0.1 * g + 1e-2 * _noise(g.shape, seed, dev)
        return s
    if kind in ("cg", "residual"):
        f, u = _manufactured(data, N, L, seed, dev)
        e = 1e-3 * _noise(u.shape, seed, dev)
        w = u.clone()  # an iterate: right on the boundary, off inside
        w[1:-1, 1:-1, 1:-1] += e[1:-1, 1:-1, 1:-1]
        return {"f": f, "u": w}
    if kind == "grad":
        return {"u": _manufactured(data, N, L, seed, dev)[1]}
    if kind == "exp_finite":
        u2, u4 = _coarser(data, tuple(n // 2 for n in N), L, seed, dev)
        return {"u2h": u2, "u4h": u4, "g": _manufactured(data, N, L, seed, dev)[1]}
    u1, u2 = _coarser(data, N, L, seed, dev)
    return {"u1": u1, "u2": u2}


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    s = _inputs(case, seed, dev)
    N, L, N0 = _dims(case)
    s.update(case=case, N=N, L=L, N0=N0)
    if case["kind"] == "solve":
        s["ws"] = X.workspace(X.solve_workspace_bytes(L, N, N0, **_solve_opts(case)), dev)
        s["out"] = torch.empty_like(s["f"])
    elif case["kind"] == "batch":
        grids = _batch_grids(case, seed)
        s["list"] = [X.BatchedProblem(Li, Ni, N0i, f, g)
                     for (Li, Ni, N0i), (f, g) in zip(grids, s["problems"])]
    elif case["kind"] == "adjoint":
        s["f"].requires_grad_(True)
        s["g"].requires_grad_(True)
    return s


def run(state):
    s = state
    case, kind, L = s["case"], s["case"]["kind"], s["L"]
    if kind == "solve":
        r = X.solve(s["f"], s["g"], L, s["N0"], want_utilde=case["ut"], ws=s["ws"], out=s["out"],
                    **_solve_opts(case))
        return [r["u"], r["ut"]] if case["ut"] else [r["u"]]
    if kind == "batch":
        return X.solve_batched(s["list"], eps=case["eps"])["u"]
    if kind == "adjoint":
        u = excmg_solve(s["f"], s["g"], L, s["N0"], **_solve_opts(case))
        gf, gg = torch.autograd.grad(u, (s["f"], s["g"]), grad_outputs=s["dLdu"])
        return [u.detach(), gf, gg]
    if kind == "cg":
        u = s["u"].clone()
        X.cg(s["f"], u, L, fixed_iters=[case["steps"]])
        return [u]
    if kind == "residual":
        return list(X.residual(s["f"], s["u"], L))
    if kind == "grad":
        return list(X.grad(s["u"], L))
    if kind == "exp_finite":
        return [X.exp_finite(s["u2h"], s["u4h"], L, g=s["g"])]
    return [X.exp_true(s["u1"], s["u2"], L)]


def _nodes(N):
    return float((N[0] + 1) * (N[1] + 1) * (N[2] + 1))


def work(case):
    N, _, _ = _dims(case)
    n, kind = _nodes(N), case["kind"]
    faces = 2.0 * ((N[0] + 1) * (N[1] + 1) + (N[0] + 1) * (N[2] + 1) + (N[1] + 1) * (N[2] + 1))
    if kind == "solve":
        # f and the boundary in, u (and u~) out; the prolongation and one residual on the
        # finest grid, and the same on the coarser ones (1/8 + 1/64 + ...)
        return {"bytes": (16.0 + 8.0 * case["ut"]) * n + 8.0 * faces, "flops": (8 / 7) * 46.0 * n}
    if kind == "batch":
        n = sum(_nodes(Ni) for _L, Ni, _N0 in _batch_grids(case, 0))
        return {"bytes": 16.0 * n, "flops": (8 / 7) * 46.0 * n}
    if kind == "adjoint":
        return {"bytes": 40.0 * n + 8.0 * faces, "flops": (8 / 7) * 46.0 * n + 60.0 * n}
    if kind == "cg":
        # f in, u in and out, once; every step a 19-point product, two dot products and
        # three vector updates
        return {"bytes": 24.0 * n, "flops": (32.0 + 10.0) * case["steps"] * n}
    if kind == "residual":
        return {"bytes": 24.0 * n, "flops": 46.0 * n}
    if kind == "grad":
        return {"bytes": 32.0 * n, "flops": 18.0 * n}
    if kind == "exp_finite":
        return {"bytes": 8.0 * n * (1 + 1 / 8 + 1 / 64) + 8.0 * faces, "flops": 11.0 * n}
    return {"bytes": 8.0 * n * (2 + 1 / 8), "flops": 6.0 * n}


# ---- the same results from plain torch in 64 bits ----

def _shift(v, di, dj, dk):
    """Interior-sized view of v displaced by (di, dj, dk) in (x, y, z)."""
    nz, ny, nx = v.shape
    return v[1 + dk:nz - 1 + dk, 1 + dj:ny - 1 + dj, 1 + di:nx - 1 + di]


def _lhs(u, h):
    """The 19-point left-hand side at the interior nodes, from second differences:
    a D_x + b D_y + c D_z + (1/12) sum over pairs of (a + b) D_x D_y."""
    a, b, c = (1.0 / (v * v) for v in h)
    S = lambda i, j, k: _shift(u, i, j, k)  # noqa: E731
    c0 = S(0, 0, 0)
    sx, sy, sz = S(-1, 0, 0) + S(1, 0, 0), S(0, -1, 0) + S(0, 1, 0), S(0, 0, -1) + S(0, 0, 1)
    out = (sx - 2 * c0) * (6 * a) + (sy - 2 * c0) * (6 * b) + (sz - 2 * c0) * (6 * c)
    e = (S(-1, -1, 0) + S(1, -1, 0)) + (S(-1, 1, 0) + S(1, 1, 0))
    out += (0.5 * (a + b)) * (e - 2 * sx - 2 * sy + 4 * c0)
    e = (S(-1, 0, -1) + S(1, 0, -1)) + (S(-1, 0, 1) + S(1, 0, 1))
    out += (0.5 * (a + c)) * (e - 2 * sx - 2 * sz + 4 * c0)
    e = (S(0, -1, -1) + S(0, 1, -1)) + (S(0, -1, 1) + S(0, 1, 1))
    out += (0.5 * (b + c)) * (e - 2 * sy - 2 * sz + 4 * c0)
    return out


def _rhs(f):
    S = lambda i, j, k: _shift(f, i, j, k)  # noqa: E731
    return 3.0 * S(0, 0, 0) + 0.5 * ((S(-1, 0, 0) + S(1, 0, 0)) + (S(0, -1, 0) + S(0, 1, 0)) +
                                     (S(0, 0, -1) + S(0, 0, 1)))


def _boundary_only(g):
    u = g.clone()
    u[1:-1, 1:-1, 1:-1] = 0.0
    return u


def _dst(v, dim):
    """sum_j v_j sin(pi j k / n) along dim (n - 1 interior nodes)."""
    n = v.shape[dim] + 1
    shape = list(v.shape)
    shape[dim] = 1
    zero = v.new_zeros(shape)
    w = torch.fft.rfft(torch.cat([zero, v, zero, -v.flip(dim)], dim), dim=dim)
    return -0.5 * w.imag.narrow(dim, 1, n - 1)


def _solve_interior(b, N, h):
    """A^{-1} b, A = -(19-point left-hand side), by the sine transform."""
    a = [1.0 / (v * v) for v in h]
    mu = []
    for d, shape in ((0, (1, 1, -1)), (1, (1, -1, 1)), (2, (-1, 1, 1))):
        k = torch.arange(1, N[d], dtype=torch.float64, device=b.device)
        mu.append((-4.0 * torch.sin(0.5 * math.pi * k / N[d]) ** 2).reshape(shape))  # of D_d
    for d in (2, 1, 0):
        b = _dst(b, d)
    lam = 6.0 * (a[0] * mu[0] + a[1] * mu[1] + a[2] * mu[2])
    for i, j in ((0, 1), (0, 2), (1, 2)):
        lam = lam + (0.5 * (a[i] + a[j])) * mu[i] * mu[j]
    b = b * (-8.0 / (N[0] * N[1] * N[2]) / lam)
    for d in (2, 1, 0):
        b = _dst(b, d)
    return b


def _discrete(f, g, N, L):
    """The FD solution u_h of (f, g)."""
    h = [L[d] / N[d] for d in range(3)]
    u = _boundary_only(g)
    u[1:-1, 1:-1, 1:-1] = _solve_interior(_lhs(u, h) - _rhs(f), N, h)
    return u


def _weights(points, data):
    """Rows of the Lagrange interpolation on nodes 0 .. len - 1."""
    t = np.arange(points)
    W = np.zeros((len(data), points))
    for r, x in enumerate(data):
        for m in range(points):
            W[r, m] = np.prod([(x - k) / (m - k) for k in t if k != m])
    return W


def _spread_linear(v, dim):
    """Trilinear midpoints along dim: n + 1 nodes to 2 n + 1."""
    n = v.shape[dim] - 1
    shape = list(v.shape)
    shape[dim] = 2 * n + 1
    out = v.new_empty(shape)
    idx = [slice(None)] * 3
    idx[dim] = slice(0, None, 2)
    out[tuple(idx)] = v
    idx[dim] = slice(1, None, 2)
    out[tuple(idx)] = 0.5 * (v.narrow(dim, 0, n) + v.narrow(dim, 1, n))
    return out


def _corner_mean(d):
    for dim in range(3):
        d = _spread_linear(d, dim)
    return d


def _exp_true(u1, u2):
    return u1 + _corner_mean(u1[::2, ::2, ::2] - u2) / 15.0


def _exp_finite(u2, u4, g):
    w = u2 + _corner_mean(u2[::2, ::2, ::2] - u4) / 16.0
    W = torch.from_numpy(_weights(5, np.arange(9) / 2.0)).to(w)  # 5 nodes -> 9 fine nodes
    for dim in range(3):
        v = w.movedim(dim, -1)
        cells = v.unfold(-1, 5, 4) @ W.T                          # (..., cells, 9)
        fine = torch.cat([cells[..., :8].reshape(*v.shape[:-1], -1), cells[..., -1, 8:]], -1)
        w = fine.movedim(-1, dim).contiguous()
    out = g.clone()
    out[1:-1, 1:-1, 1:-1] = w[1:-1, 1:-1, 1:-1]
    return out


def _grad_axis(u, dim, h):
    u = u.movedim(dim, 0).contiguous()
    n = u.shape[0] - 1
    d = torch.empty_like(u)
    k = (-25.0 / 12.0, 4.0, -3.0, 4.0 / 3.0, -0.25)
    d[0] = sum(c * u[i] for i, c in enumerate(k)) / h
    d[n] = -sum(c * u[n - i] for i, c in enumerate(k)) / h
    # (1/6, 4/6, 1/6) by elimination
    cp, prev = [], d[0]
    for i in range(1, n):
        m = 4.0 / 6.0 - (cp[-1] / 6.0 if cp else 0.0)
        rhs = (u[i + 1] - u[i - 1]) / (2.0 * h)
        if i == n - 1:
            rhs = rhs - d[n] / 6.0
        d[i] = (rhs - prev / 6.0) / m
        cp.append(1.0 / 6.0 / m)
        prev = d[i]
    for i in range(n - 2, 0, -1):
        d[i] -= cp[i - 1] * d[i + 1]
    return d.movedim(0, dim).contiguous()


def _cg(f, u, h, steps):
    u = u.clone()
    inner = (slice(1, -1),) * 3
    r = _lhs(u, h) - _rhs(f)
    p = torch.zeros_like(u)
    p[inner] = r
    rr = (r * r).sum()
    for _ in range(steps):
        q = -_lhs(p, h)
        alpha = rr / (p[inner] * q).sum()
        u[inner] += alpha * p[inner]
        r = r - alpha * q
        new = (r * r).sum()
        p[inner] = r + (new / rr) * p[inner]
        rr = new
    return u


def exact(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device()) if torch.cuda.is_available() else torch.device("cpu")
    N, L, _ = _dims(case)
    s, kind = _inputs(case, seed, dev), case["kind"]
    if kind == "batch":
        return [_discrete(f, g, Ni, Li) for (Li, Ni, _N0), (f, g) in zip(_batch_grids(case, seed), s["problems"])]
    h = [L[d] / N[d] for d in range(3)]
    if kind == "solve":
        u = _discrete(s["f"], s["g"], N, L)
        if not case["ut"]:
            return [u]
        half = tuple(n // 2 for n in N)
        return [u, _exp_true(u, _discrete(s["f"][::2, ::2, ::2], s["g"][::2, ::2, ::2], half, L))]
    if kind == "adjoint":
        u, w = _discrete(s["f"], s["g"], N, L), s["dLdu"]
        lam = torch.zeros([n + 2 for n in w.shape], dtype=w.dtype, device=w.device)
        lam[2:-2, 2:-2, 2:-2] = _solve_interior(w[1:-1, 1:-1, 1:-1], N, h)
        gg = _lhs(lam, h) + w
        gg[1:-1, 1:-1, 1:-1] = 0.0
        return [u, -_rhs(lam), gg]
    if kind == "cg":
        return [_cg(s["f"], s["u"], h, case["steps"])]
    if kind == "residual":
        r = torch.zeros_like(s["u"])
        r[1:-1, 1:-1, 1:-1] = _lhs(s["u"], h) - _rhs(s["f"])
        b = _lhs(_boundary_only(s["u"]), h) - _rhs(s["f"])
        return [r, float(r.norm()), float(b.norm())]
    if kind == "grad":
        return [_grad_axis(s["u"], d, v) for d, v in ((2, h[0]), (1, h[1]), (0, h[2]))]
    if kind == "exp_finite":
        return [_exp_finite(s["u2h"], s["u4h"], s["g"])]
    return [_exp_true(s["u1"], s["u2"])]
