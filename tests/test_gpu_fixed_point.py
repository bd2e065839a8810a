"""The block fixed-point kernels: the residual and CG's 19-point sums, and EXP_finite.

These kernels bring a block's float64 values to one power of two and sum 64-bit integers.
The tests take them where that can go wrong: slab and group edges (32 x 8 columns, groups
of six planes), partial slabs, the smallest grids, scales from 1e-300 to 1e300, steps of
many orders of magnitude between neighbouring groups, zeros, infinities and NaN.  The
reference is the float64 oracle; tolerances come from float64's own rounding of a 19-point
sum: c0 = 8 (1/hx^2 + 1/hy^2 + 1/hz^2) is its largest weight and the absolute weights add up
to less than 3 c0, so a sum of ~20 rounded terms of |u| <= U is within 20 * 3 c0 U 2^-53.
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


def sum_tol(h, U):
    return 60 * 8 * sum(1.0 / v ** 2 for v in h) * U * 2.0 ** -53


def fields(N, seed=0):
    rng = np.random.default_rng(seed)
    shape = (N[2] + 1, N[1] + 1, N[0] + 1)
    return rng.standard_normal(shape), rng.standard_normal(shape)


def check(X, f, u, L, N):
    """r, ||r|| and ||b|| against the oracle, by the bound above (f: 9 terms of weight <= 3)."""
    h = O.meshsizes(L, N)
    r, rn, bn = X.residual(dev(f), dev(u), L)
    r = r.cpu().numpy()
    want = O.residual(u, f, h)
    if want.shape != r.shape:
        full = np.zeros_like(r)
        full[1:-1, 1:-1, 1:-1] = want
        want = full
    tol = sum_tol(h, np.max(np.abs(u))) + 60 * np.max(np.abs(f)) * 2.0 ** -53
    assert np.max(np.abs(r - want)) <= tol
    for a in (r[0], r[-1], r[:, 0], r[:, -1], r[:, :, 0], r[:, :, -1]):
        assert not np.any(a)
    n = np.prod([v - 1 for v in N])
    b = O.rhs_vector(f, u, h)
    with np.errstate(over="ignore"):
        assert rn == pytest.approx(np.sqrt(np.sum(want * want)), rel=1e-12, abs=tol * np.sqrt(n))
        assert bn == pytest.approx(np.sqrt(np.sum(b * b)), rel=1e-12, abs=tol * np.sqrt(n))


SIZES = [(2, 2, 2), (3, 2, 5), (33, 9, 5), (34, 10, 6), (32, 8, 4), (65, 17, 9), (31, 7, 130), (100, 41, 63)]


@pytest.mark.parametrize("N", SIZES)
@pytest.mark.parametrize("L", [(1.0, 1.0, 1.0), (3.0, 0.2, 1.7)])
def test_residual_sizes(X, N, L):
    f, u = fields(N)
    check(X, f, u, L, N)


@pytest.mark.parametrize("scale", [1e-290, 1e-200, 1e-60, 1e60, 1e140])
def test_residual_scales(X, scale):
    """Far below and above 1: inside fixed point's range of exponents, and outside it (the
    float64 form)."""
    N, L = (40, 19, 22), (1.0, 0.5, 0.7)
    f, u = fields(N, 1)
    check(X, f * scale * 1e3, u * scale, L, N)


@pytest.mark.parametrize("which", ["u", "f", "both"])
def test_residual_steps_between_groups(X, which):
    """Values that change by ten orders of magnitude from one group of planes to the next (up
    and down), and planes of zeros: the sums carried from group to group are rescaled."""
    N, L = (40, 19, 45), (1.0, 0.5, 0.7)
    f, u = fields(N, 2)
    w = 10.0 ** np.random.default_rng(3).integers(-10, 11, size=N[2] + 1)
    w[20:30] = 0.0
    w = np.repeat(w[::4], 4)[:N[2] + 1][:, None, None]
    check(X, f * w if which != "u" else f, u * w if which != "f" else u, L, N)


def test_residual_zero_fields(X):
    N, L = (36, 12, 11), (1.0, 1.0, 1.0)
    f, u = fields(N, 4)
    zero = np.zeros_like(f)
    check(X, zero, u, L, N)
    check(X, f, zero, L, N)
    r, rn, bn = X.residual(dev(zero), dev(zero), L)
    assert not torch.any(r) and rn == 0.0 and bn == 0.0


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_residual_nonfinite_stays_local(X, value):
    """An infinity or a NaN in u or f reaches exactly the nodes whose sums read it."""
    N, L = (40, 19, 30), (1.0, 0.5, 0.7)
    for name in ("u", "f"):
        f, u = fields(N, 5)
        (u if name == "u" else f)[13, 7, 33] = value
        r = X.residual(dev(f), dev(u), L)[0].cpu().numpy()
        bad = np.zeros(r.shape, bool)
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    n = abs(dx) + abs(dy) + abs(dz)
                    if n <= (2 if name == "u" else 1):
                        bad[13 + dz, 7 + dy, 33 + dx] = True
        assert np.array_equal(~np.isfinite(r), bad)


@pytest.mark.parametrize("N,steps,scale", [((208, 104, 52), 6, 1e-150), ((105, 106, 104), 6, 1e100),
                                           ((70, 260, 70), 6, 1.0)])
def test_streaming_cg_sums(X, N, steps, scale):
    """The streaming float64 CG (grids of more than 2^20 nodes) after fixed steps, relative to
    the oracle's: 1e-12 of the solution's size, a few hundred roundings of its sums."""
    L = (1.0, 0.9, 1.1)
    f, start = fields(N, 6)
    f, start = f * scale, start * scale
    want, _, _ = O.cg(start, f, O.meshsizes(L, N), 0.0, fixed_iters=steps)
    u = dev(start)
    st = X.cg(dev(f), u, L, eps=0.0, fixed_iters=[steps], profile=1)
    assert "cg_f64" in st["profile"]
    assert np.max(np.abs(u.cpu().numpy() - want)) <= 1e-12 * np.max(np.abs(want))


@pytest.mark.parametrize("N,scale,steps", [((16, 17, 18), 1.0, 6), ((31, 33, 35), 1e-60, 6), ((40, 9, 70), 1e60, 6),
                                           ((100, 80, 60), 1.0, 6), ((120, 65, 80), 1.0, 3)])
def test_resident_cg_sums(X, N, scale, steps):
    """The shared-memory CG (up to 2^20 nodes) after fixed steps: boxes cut by the grid's far
    faces, one node per thread and several; tolerance as above."""
    L = (1.0, 0.9, 1.1)
    f, start = fields(N, 8)
    f, start = f * scale, start * scale
    want, _, _ = O.cg(start, f, O.meshsizes(L, N), 0.0, fixed_iters=steps)
    u = dev(start)
    st = X.cg(dev(f), u, L, eps=0.0, fixed_iters=[steps], profile=1)
    assert "cg_resident_f64" in st["profile"]
    assert np.max(np.abs(u.cpu().numpy() - want)) <= 1e-12 * np.max(np.abs(want))


@pytest.mark.parametrize("N", [(8, 8, 8), (24, 8, 16), (32, 16, 8), (40, 24, 16), (72, 16, 40)])
@pytest.mark.parametrize("scale", [1.0, 1e-250, 1e250])
def test_exp_finite_bricks(X, N, scale):
    """Whole and partial bricks (32 x 8 x 8 fine cells), inside and outside fixed point's
    exponents, with and without Dirichlet data.  Three passes of five products whose absolute
    weights add up to 278/128 each, on values of at most 1.13 U: 15 roundings of 11.6 U."""
    rng = np.random.default_rng(7)
    u2 = rng.standard_normal([n // 2 + 1 for n in N[::-1]]) * scale
    u4 = u2[::2, ::2, ::2] + 0.1 * scale * rng.standard_normal([n // 4 + 1 for n in N[::-1]])
    g = rng.standard_normal([n + 1 for n in N[::-1]]) * scale
    want = O.exp_finite(u2, u4)
    tol = 15 * 11.6 * np.max(np.abs(u2)) * 2.0 ** -53
    L = (1.0, 1.0, 1.0)
    got = X.exp_finite(dev(u2), dev(u4), L).cpu().numpy()
    assert np.max(np.abs(got - want)) <= tol
    got = X.exp_finite(dev(u2), dev(u4), L, g=dev(g)).cpu().numpy()
    inner = (slice(1, -1),) * 3
    assert np.max(np.abs(got[inner] - want[inner])) <= tol
    edge = np.ones(got.shape, bool)
    edge[inner] = False
    assert np.array_equal(got[edge], g[edge])


def test_exp_finite_nonfinite(X):
    """A NaN reaches the bricks that hold it and no others."""
    N = (64, 16, 16)
    rng = np.random.default_rng(8)
    u2 = rng.standard_normal([n // 2 + 1 for n in N[::-1]])
    u4 = rng.standard_normal([n // 4 + 1 for n in N[::-1]])
    clean = X.exp_finite(dev(u2), dev(u4), (1.0, 1.0, 1.0)).cpu().numpy()
    u2[1, 1, 1] = np.nan
    got = X.exp_finite(dev(u2), dev(u4), (1.0, 1.0, 1.0)).cpu().numpy()
    assert np.isnan(got[2, 2, 2])
    assert np.array_equal(got[9:], clean[9:]) and np.array_equal(got[:, :, 33:], clean[:, :, 33:])


@pytest.mark.parametrize("N", [(2, 2, 2), (4, 2, 6), (62, 6, 14), (64, 8, 16), (66, 10, 18), (126, 30, 34),
                               (128, 10, 20)])
def test_exp_true_tiles(X, N):
    """EXP_true across its 64 x 8 columns and chunks of eight coarse planes: a sum of eight
    differences of at most 2 U, and the addition: ten roundings of 3 U."""
    rng = np.random.default_rng(9)
    uh = rng.standard_normal([n + 1 for n in N[::-1]])
    u2 = rng.standard_normal([n // 2 + 1 for n in N[::-1]])
    got = X.exp_true(dev(uh), dev(u2), (1.0, 1.0, 1.0)).cpu().numpy()
    want = O.extrapolate_true(uh, u2)
    assert np.max(np.abs(got - want)) <= 30 * max(np.max(np.abs(uh)), np.max(np.abs(u2))) * 2.0 ** -53


@pytest.mark.parametrize("N", [(4, 4, 4), (4, 5, 67), (33, 4, 6), (6, 131, 5), (31, 32, 33), (65, 34, 66)])
def test_gradient_line_edges(X, N):
    """All three directions from one launch: lengths about the groups of line steps (4), the
    staged chunks of x-lines (32) and the factors' table (64), and unequal numbers of lines.
    The compact system's inverse is below 3 and its right-hand sides below 3 U / h, so some
    tens of rounded operations stay within 200 U / h 2^-53."""
    L = (1.0, 0.7, 1.9)
    u, _ = fields(N, 7)
    h = O.meshsizes(L, N)
    for got, want, hd in zip(X.grad(dev(u), L), O.gradient(u, h), h):
        assert np.max(np.abs(got.cpu().numpy() - want)) <= 200 * np.max(np.abs(u)) / hd * 2.0 ** -53
