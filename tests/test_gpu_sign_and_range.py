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
