"""What block fixed point has to keep of float64 arithmetic: the symmetry in sign (every
rounding of a sum of -x is that of x with the sign changed), zeros of either sign, and the
accuracy of small values beside large ones.
"""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def X():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05063_gb300 import excmg
    return excmg


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def fields(N, seed, kind):
    """Two node arrays: normal deviates, or small multiples of 1/4 (whose sums tie when they
    are rounded)."""
    rng = np.random.default_rng(seed)
    shape = (N[2] + 1, N[1] + 1, N[0] + 1)
    if kind == "ties":
        return rng.integers(-9, 10, shape) / 4.0, rng.integers(-9, 10, shape) / 4.0
    return rng.standard_normal(shape), rng.standard_normal(shape)


@pytest.mark.parametrize("kind", ["normal", "ties"])
@pytest.mark.parametrize("N,L", [((33, 9, 5), (1.0, 1.0, 1.0)), ((70, 40, 31), (1.0, 0.7, 0.3)),
                                 ((100, 41, 63), (3.0, 0.2, 1.7))])
def test_residual_changes_sign(X, N, L, kind):
    f, u = (dev(a) for a in fields(N, 1, kind))
    r, rn, bn = X.residual(f, u, L)
    m, mn, mb = X.residual(-f, -u, L)
    assert torch.equal(m, -r) and mn == rn and mb == bn


@pytest.mark.parametrize("kind", ["normal", "ties"])
def test_exp_finite_changes_sign(X, kind):
    N = (72, 16, 40)
    u2, u4 = (dev(fields(tuple(n // s for n in N), s, kind)[0]) for s in (2, 4))
    assert torch.equal(X.exp_finite(-u2, -u4, (1.0, 1.0, 1.0)), -X.exp_finite(u2, u4, (1.0, 1.0, 1.0)))


@pytest.mark.parametrize("N,engine", [((31, 33, 35), "cg_resident_f64"), ((70, 260, 70), "cg_f64")])
def test_cg_changes_sign(X, N, engine):
    """CG's scalars are products of two vectors: the same for the negated system."""
    L = (1.0, 0.9, 1.1)
    f, start = (dev(a) for a in fields(N, 2, "normal"))
    u, v = start.clone(), -start
    st = X.cg(f, u, L, eps=0.0, fixed_iters=[5], profile=1)
    assert engine in st["profile"]
    X.cg(-f, v, L, eps=0.0, fixed_iters=[5])
    assert torch.equal(v, -u)


@pytest.mark.parametrize("opts", [{}, {"precision": "mixed", "mixed_min_nodes": 1}])
def test_solve_changes_sign(X, opts):
    N, N0, L = (64, 32, 48), (8, 4, 6), (1.0, 0.5, 0.7)
    f, g = (dev(a) for a in fields(N, 3, "normal"))
    a = X.solve(f, g, L, N0, eps=1e-9, want_utilde=True, **opts)
    b = X.solve(-f, -g, L, N0, eps=1e-9, want_utilde=True, **opts)
    assert a["stats"]["iters"] == b["stats"]["iters"]
    assert torch.equal(b["u"], -a["u"]) and torch.equal(b["ut"], -a["ut"])


def test_negative_zeros_are_zeros(X):
    """-0.0 in u and f: alone, and beside values of size one."""
    N, L = (40, 19, 22), (1.0, 0.5, 0.7)
    f, u = fields(N, 4, "normal")
    zero = np.zeros_like(f)
    for a, b in ((-zero, zero), (zero, -zero), (-zero, -zero)):
        r, rn, bn = X.residual(dev(a), dev(b), L)
        assert not torch.any(r) and rn == 0.0 and bn == 0.0
    mask = np.random.default_rng(5).random(f.shape) < 0.5
    plus = [np.where(mask, 0.0, a) for a in (f, u)]
    minus = [np.where(mask, -0.0, a) for a in (f, u)]
    r = X.residual(dev(plus[0]), dev(plus[1]), L)
    s = X.residual(dev(minus[0]), dev(minus[1]), L)
    assert torch.equal(r[0], s[0]) and r[1:] == s[1:]


# A grid whose slabs (18 planes and their halo) hold four groups of six planes, and enough
# nodes for the streaming CG.
GROUPS_N, GROUPS_L = (70, 260, 70), (1.0, 0.9, 1.1)


def near(a, planes):
    """The largest |a| within one column, one row and `planes` planes of a node."""
    m = np.abs(a)
    for axis, reach in ((2, 1), (1, 1), (0, planes)):
        out = m.copy()
        for d in range(1, reach + 1):
            lo, hi = [slice(None)] * 3, [slice(None)] * 3
            lo[axis], hi[axis] = slice(None, -d), slice(d, None)
            out[tuple(lo)] = np.maximum(out[tuple(lo)], m[tuple(hi)])
            out[tuple(hi)] = np.maximum(out[tuple(hi)], m[tuple(lo)])
        m = out
    return m


def ranged(kind, N, seed):
    """Node arrays with a large range of values: exponential layers, a narrow Gaussian, steps
    of many powers of ten along z (aligned with the groups of planes or not), compact support."""
    rng = np.random.default_rng(seed)
    i, j, k = np.meshgrid(*[np.arange(n + 1) for n in N], indexing="ij")
    i, j, k = (a.transpose(2, 1, 0) for a in (i, j, k))
    base = rng.standard_normal(i.shape)
    if kind.startswith("layer"):
        return base * np.exp(-{"x": i, "y": j, "z": k}[kind[5]] * 0.9)
    if kind == "gauss":
        return np.exp(-0.02 * ((i - N[0] / 2) ** 2 + (j - N[1] / 3) ** 2 + (k - N[2] / 2) ** 2))
    if kind == "compact":  # ends within rows, columns and planes
        return np.where((i - 20) ** 2 + (j - 30) ** 2 + (k - 30) ** 2 < 14 ** 2, base, 0.0)
    step = {"steps6": 6, "steps4": 4, "steps11": 11}[kind]
    w = 10.0 ** rng.integers(-25, 26, size=N[2] // step + 1)
    w[rng.integers(0, len(w))] = 0.0
    return base * np.repeat(w, step)[:N[2] + 1][:, None, None]


KINDS = ["layerx", "layery", "layerz", "gauss", "compact", "steps6", "steps4", "steps11"]


@pytest.mark.parametrize("which", ["u", "f"])
@pytest.mark.parametrize("kind", KINDS)
def test_residual_is_accurate_where_values_are_small(X, kind, which):
    """Every node's r within 2^-50 of its neighbourhood's values times the weights -- eight
    roundings in a row of a float64 sum; the absolute weights add up to less than 3 c0 for u
    and are 6 for f -- not of the largest value of the grid.  Twice that: the oracle rounds as
    well."""
    N, L = GROUPS_N, GROUPS_L
    rng = np.random.default_rng(7)
    zero = np.zeros([n + 1 for n in N[::-1]])
    f, u = zero, zero
    if which == "u":
        u = ranged(kind, N, 8)
    else:
        f = ranged(kind, N, 9)
    h = O.meshsizes(L, N)
    got = X.residual(dev(f), dev(u), L)[0].cpu().numpy()[1:-1, 1:-1, 1:-1]
    want = O.residual(u, f, h)
    if want.shape != got.shape:
        want = want[1:-1, 1:-1, 1:-1]
    c0 = 8 * sum(1.0 / v ** 2 for v in h)
    tol = 2 * 2.0 ** -50 * (3 * c0 * near(u, 4) + 6 * near(f, 4))[1:-1, 1:-1, 1:-1]
    assert np.all(np.abs(got - want) <= tol)


@pytest.mark.parametrize("N,engine", [(GROUPS_N, "cg_f64"), ((60, 90, 50), "cg_resident_f64"),
                                      ((20, 24, 40), "cg_resident_f64")])
@pytest.mark.parametrize("kind", KINDS)
def test_cg_is_accurate_where_values_are_small(X, kind, N, engine):
    """Two steps of CG on A u = 0 from an iterate with a large range: x_2 = x_0 + a_0 r_0 + a_1 (r_0 - a_0 A r_0 + b_1 r_0), node by node.  Sixteen
    roundings in a row and the scalars' (some 1e-13 of themselves) on each term."""
    L = GROUPS_L
    u0 = ranged(kind, N, 10)
    for a in (u0[0], u0[-1], u0[:, 0], u0[:, -1], u0[:, :, 0], u0[:, :, -1]):
        a[...] = 0.0
    f = np.zeros_like(u0)
    h = O.meshsizes(L, N)
    inner = (slice(1, -1),) * 3

    def full(v):
        if v.shape == u0.shape:
            return v
        w = np.zeros_like(u0)
        w[inner] = v
        return w

    r0 = full(O.residual(u0, f, h))
    q0 = -full(O.residual(r0, f, h))  # A r_0
    a0 = np.sum(r0 * r0) / np.sum(r0 * q0)
    r1 = r0 - a0 * q0
    b1 = np.sum(r1 * r1) / np.sum(r0 * r0)
    p1 = r1 + b1 * r0
    a1 = np.sum(r1 * r1) / -np.sum(p1 * full(O.residual(p1, f, h)))
    want = u0 + a0 * r0 + a1 * p1
    u = dev(u0)
    st = X.cg(dev(f), u, L, eps=0.0, fixed_iters=[2], profile=1)
    assert engine in st["profile"]
    c0 = 8 * sum(1.0 / v ** 2 for v in h)
    # r_0 is itself off by its neighbourhood's rounding; A r_0 likewise, one node further
    dr = 3 * c0 * near(u0, 4)
    size = np.abs(u0) + (a0 + a1 * (1 + b1)) * dr + a0 * a1 * 3 * c0 * near(dr, 4)
    assert np.all(np.abs(u.cpu().numpy() - want) <= (16 * 2.0 ** -50 + 1e-13) * size)


@pytest.mark.parametrize("value", [np.inf, np.nan, 1e290])
def test_residual_slab_taken_again(X, value):
    """A value that is not for fixed point in a slab's third group, after two groups were
    written: the slab is taken again in float64, and no other node sees it."""
    N, L = GROUPS_N, GROUPS_L
    f, u = fields(N, 11, "normal")
    r0 = X.residual(dev(f), dev(u), L)[0].cpu().numpy()
    u[32, 40, 20] = value
    r1, rn, bn = X.residual(dev(f), dev(u), L)
    r1 = r1.cpu().numpy()
    bad = np.zeros(u.shape, bool)
    bad[31:34, 39:42, 19:22] = True
    c0 = 8 * sum(1.0 / v ** 2 for v in O.meshsizes(L, N))
    assert np.all(np.abs(r1 - r0)[~bad] <= 2 * 2.0 ** -50 * 3 * c0 * np.max(np.abs(np.where(bad, 0.0, u))))
    assert not np.isfinite(rn)  # 1e290: the square overflows


def stencil(v, h):
    """A v on the interior of a node array, in the array's own precision."""
    a, b, c = (np.longdouble(1) / np.longdouble(t) ** 2 for t in h)
    nz, ny, nx = v.shape

    def s(i, j, k):
        return v[1 + k:nz - 1 + k, 1 + j:ny - 1 + j, 1 + i:nx - 1 + i]

    sx, sy, sz = s(-1, 0, 0) + s(1, 0, 0), s(0, -1, 0) + s(0, 1, 0), s(0, 0, -1) + s(0, 0, 1)
    exy = s(-1, -1, 0) + s(1, -1, 0) + s(-1, 1, 0) + s(1, 1, 0)
    exz = s(-1, 0, -1) + s(1, 0, -1) + s(-1, 0, 1) + s(1, 0, 1)
    eyz = s(0, -1, -1) + s(0, 1, -1) + s(0, -1, 1) + s(0, 1, 1)
    return (8 * (a + b + c) * s(0, 0, 0) - (4 * a - b - c) * sx - (4 * b - a - c) * sy - (4 * c - a - b) * sz
            - ((a + b) * exy + (a + c) * exz + (b + c) * eyz) / 2)


def stencil_rhs(f):
    """RHS(f) on the interior of a node array, in the array's own precision."""
    c = f[1:-1, 1:-1, 1:-1]
    return 3 * c + ((f[1:-1, 1:-1, :-2] + f[1:-1, 1:-1, 2:]) + (f[1:-1, :-2, 1:-1] + f[1:-1, 2:, 1:-1])
                    + (f[:-2, 1:-1, 1:-1] + f[2:, 1:-1, 1:-1])) / 2


@pytest.mark.parametrize("N", [(48, 100, 37), (20, 70, 23), (100, 24, 50)])
def test_residual_of_a_smooth_field_rounds_to_nearest(X, N):
    """Values within 2^3 of a slab's largest are exact as integers, so r is off by half a unit of
    the weighted sum (2^-57 of the powers of two above the largest value and weight) and the
    float64 roundings of the two sums and their difference."""
    L = (1.0, 1.0, 1.0)
    i, j, k = np.meshgrid(*[np.arange(n + 1) / n for n in N], indexing="ij")
    u = np.exp(i + j + k).transpose(2, 1, 0)
    f = 3.0 * u
    r = X.residual(dev(f), dev(u), L)[0].cpu().numpy()[1:-1, 1:-1, 1:-1]
    h = O.meshsizes(L, N)
    # the weights 1/h^2 as float64 has them: stencil() squares and divides in long double
    w = [1.0 / (t * t) for t in h]
    lhs = -stencil(u.astype(np.longdouble), [1 / np.sqrt(np.longdouble(t)) for t in w])
    rhs = -stencil_rhs(f.astype(np.longdouble))
    unit = 2.0 ** (np.frexp(max(w))[1] + np.frexp(np.max(u))[1] - 57)
    tol = 0.5 * unit * (1 + 2.0 ** -8) + 2.0 ** -52 * (np.abs(lhs) + np.abs(rhs))
    tol += 32 * np.finfo(np.longdouble).eps * 8 * sum(w) * np.abs(u[1:-1, 1:-1, 1:-1])  # the reference's own
    assert np.all(np.abs(r - (lhs + rhs)) <= tol)


@pytest.mark.parametrize("n", [16, 32, 64])
@pytest.mark.parametrize("kind", ["normal", "sine", "peak", "corner"])
def test_resident_cg_scalars(X, kind, n):
    """r.r and w.r of the shared-memory CG, through the first step from zero: x_1 = a r_0 gives
    a = r_0.r_0 / r_0.A r_0, and the history r_1.r_1 of r_1 = r_0 - a A r_0.  The sums: 2^-50 of
    themselves (eight roundings in a row).  The terms: A r_0 is off by 2^-50 of its
    neighbourhood's values times the weights at most, r_1 by as much times a."""
    N, L = (n, n, n), (1.0, 1.0, 1.0)
    i, j, k = np.meshgrid(*[np.arange(n + 1)] * 3, indexing="ij")
    f = {"normal": lambda: np.random.default_rng(12).standard_normal(i.shape),
         "sine": lambda: np.sin(np.pi * i / n) * np.sin(np.pi * j / n) * np.sin(np.pi * k / n),
         "peak": lambda: 1.0 * ((i == n // 2) & (j == n // 3) & (k == n // 2 + 1)),
         "corner": lambda: np.exp(-0.4 * (i + j + k))}[kind]()
    zero = torch.zeros((n + 1,) * 3, dtype=torch.float64, device="cuda")
    r0 = X.residual(dev(f), zero, L)[0].cpu().numpy()
    u = zero.clone()
    st = X.cg(dev(f), u, L, eps=0.0, fixed_iters=[1], history=2, profile=1)
    assert "cg_resident_f64" in st["profile"]
    u = u.cpu().numpy()
    at = np.unravel_index(np.argmax(np.abs(r0)), r0.shape)
    alpha = np.longdouble(u[at]) / np.longdouble(r0[at])
    inner = (slice(1, -1),) * 3
    r = r0.astype(np.longdouble)
    w = stencil(r, [1.0 / n] * 3)
    c0 = 24.0 * n * n
    dw = 2.0 ** -50 * 3 * c0 * near(r0, 4)[inner]
    want = np.sum(r * r) / np.sum(r[inner] * w)
    tol = 3 * 2.0 ** -50 + np.sum(np.abs(r0[inner]) * dw) / np.sum(r[inner] * w)
    assert abs(alpha / want - 1) <= tol
    # the history's entries are sqrt(r_k.r_k / b.b), and r_0 = b here
    r1 = r[inner] - alpha * w
    g1 = np.sum(r1 * r1)
    dr = alpha * dw + 2.0 ** -52 * (np.abs(r0[inner]) + np.abs(r1))
    got = np.longdouble(st["history"][1]) ** 2 * np.sum(r * r)
    assert abs(got - g1) <= 8 * 2.0 ** -50 * g1 + 2 * np.sum(np.abs(r1) * dr) + np.sum(dr * dr)


@pytest.mark.parametrize("kind", KINDS)
def test_exp_finite_is_accurate_where_values_are_small(X, kind):
    """Every interpolated value within its cell's rounding (the tolerance of a brick of values
    of one size, on the largest value of the cell and those that share a node with it)."""
    N = (96, 48, 64)
    u2 = ranged(kind, tuple(n // 2 for n in N), 13)
    u4 = np.ascontiguousarray(u2[::2, ::2, ::2]) * (1 + 1e-3)
    want = O.exp_finite(u2, u4)
    got = X.exp_finite(dev(u2), dev(u4), (1.0, 1.0, 1.0)).cpu().numpy()
    m = np.abs(u2)
    for axis in range(3):  # the largest value of each cell (5 nodes, 4 apart), on its 9 fine nodes
        m = np.moveaxis(m, axis, -1)
        cells = np.max([m[..., s:s + m.shape[-1] - 4:4] for s in range(5)], axis=0)
        fine = np.repeat(cells, 8, axis=-1)
        last = fine[..., -1:]
        low = np.concatenate([fine[..., :1], fine], axis=-1)   # a node between two cells: the larger
        high = np.concatenate([fine, last], axis=-1)
        m = np.moveaxis(np.maximum(low, high), -1, axis)
    assert np.all(np.abs(got - want) <= 15 * 11.6 * m * 2.0 ** -53 * 2)


def relres_of(X, f, u, L):
    """||r|| / ||b|| of the iterate u with the sums of a tolerance below 1e-13 (float64)."""
    return X.cg(f, u.clone(), L, eps=1e-15, max_iter=0, allow_not_converged=True)["relres"][0]


def test_tight_mixed_residual_is_float64(X):
    """MIXED at 1e-14: the outer residual that decides on convergence has the sums of an FP64
    solve at that tolerance, to the last bit."""
    N, L = (48, 40, 36), (1.0, 0.9, 1.1)
    f, u = (dev(a) for a in fields(N, 14, "normal"))
    st = X.cg(f, u, L, precision="mixed", mixed_min_nodes=1, eps=1e-14, max_refine=4, allow_not_converged=True)
    assert st["refinements"][0] >= 2
    assert st["relres"][0] == relres_of(X, f, u, L)


def test_one_arithmetic_per_solve(X):
    """A tolerance below 1e-13 on one level is the whole solve's: here level 2's (eps_ratio), the
    finest level's start meets its own and is not changed."""
    N, N0, L = (64, 48, 32), (8, 6, 4), (1.0, 0.9, 1.1)
    i, j, k = np.meshgrid(*[np.arange(n + 1) / n for n in N], indexing="ij")
    g = np.exp(i + j + k).transpose(2, 1, 0)
    f, g = dev(3.1 * g), dev(g)
    res = X.solve(f, g, L, N0, eps=0.5, eps_ratio=1e-14, max_iter=200, allow_not_converged=True)
    assert res["stats"]["iters"][3] == 0
    assert res["stats"]["relres"][3] == relres_of(X, f, res["u"], L)


def test_slab_depth_reaches_the_float64_kernels(X):
    """options.tile_z moves the slabs of the residual and of the streaming float64 CG (their
    sums add in another order: other last bits, the same solution), and autotune = 1 times
    them."""
    N, L = GROUPS_N, GROUPS_L
    f, start = (dev(a) for a in fields(N, 15, "normal"))
    runs = []
    for tz in (2, 3, 5, 8, 11, 23):
        u = start.clone()
        st = X.cg(f, u, L, eps=0.0, fixed_iters=[4], history=1, tile_z=tz, profile=1)
        assert "cg_f64" in st["profile"]
        runs.append((u, st["history"][0]))
    a, ra = runs[0]
    for b, rb in runs[1:]:
        assert not torch.equal(a, b)
        assert torch.max(torch.abs(a - b)) <= 1e-12 * torch.max(torch.abs(a)) and ra == pytest.approx(rb, rel=1e-13)
    assert len({r for _, r in runs}) > 1
    N, N0 = (128, 128, 128), (8, 8, 8)
    i, j, k = np.meshgrid(*[np.arange(n + 1) / n for n in N], indexing="ij")
    g = dev(np.exp(i + j + k))
    X.excmg_tuning_clear()
    X.solve(3.0 * g, g, (1.0, 1.0, 1.0), N0, eps=1e-9, autotune=1)
    e = {tuple(t["N"]): t for t in X.tuning_entries()}
    X.excmg_tuning_clear()
    t = e[N]
    assert t["cg_tz"] >= 1 and 0 < t["cg_ms"] <= t["cg_ms_model"] * 1.0001
    assert any(v["res_tz"] != v["res_tz_model"] or v["res_ms"] == v["res_ms_model"] for v in e.values())
    assert all(0 < v["res_ms"] <= v["res_ms_model"] * 1.0001 for v in e.values())


def test_tuning_times_no_layers_of_its_own(X):
    """The tuning pass times the slabs on values of one size, whatever g: from a large g on the
    boundary and zeros inside, slabs next to the boundary took the float64 form, more than twice
    the time."""
    N, N0, L = (256, 256, 128), (8, 8, 4), (1.0, 1.0, 1.0)
    f = dev(np.random.default_rng(16).standard_normal([n + 1 for n in N[::-1]]))
    times = []
    for value in (0.0, 1e3):
        X.excmg_tuning_clear()
        X.solve(f, torch.full_like(f, value), L, N0, eps=1e-2, autotune=1)
        times.append({tuple(t["N"]): t for t in X.tuning_entries()}[N])
        X.excmg_tuning_clear()
    for key in ("res_ms_model", "cg_ms_model"):
        a, b = (t[key] for t in times)
        assert 0 < max(a, b) <= 1.4 * min(a, b)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_profiled_batch_runs_as_it_does(X, precision):
    """options.profile changes nothing about a batch: the same launches and the same bits, its
    problems of 2^18 nodes in teams; a shared launch's time and node-steps count to the
    group's first problem."""
    N, N0, L = (64, 64, 64), (8, 8, 8), (1.0, 1.0, 1.0)
    i, j, k = np.meshgrid(*[np.arange(n + 1) / n for n in N], indexing="ij")
    batch = []
    for a in (1.0, 1.3, 0.7):
        g = np.exp(a * i + j + k)
        batch.append(X.BatchedProblem(L, N, N0, dev((a * a + 2) * g), dev(g)))
    kw = dict(eps=1e-9, precision=precision, mixed_min_nodes=1 << 15)
    plain = X.solve_batched(batch, **kw)
    prof = X.solve_batched(batch, profile=1, **kw)
    for a, b in zip(plain["u"], prof["u"]):
        assert torch.equal(a, b)
    for a, b in zip(plain["stats"], prof["stats"]):
        assert a["iters"] == b["iters"] and a["launches"] == b["launches"]
    p = prof["stats"][0]["profile"]
    assert not any(s["profile"] for s in prof["stats"][1:]) and not plain["stats"][0]["profile"]
    steps = sum(st["iters"][l] * ((n := 8 << l) + 1) ** 3 for st in prof["stats"] for l in range(2, 4))
    assert sum(v["nodes"] for name, v in p.items() if name.startswith("cg_")) == steps
    assert ("cg_f64" if precision == "fp64" else "cg_f32") in p and "cg_resident_f64" not in p
