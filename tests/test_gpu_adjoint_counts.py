"""The adjoint's per-shell sums over the shapes and count ranges at which the
kernel changes its form: tiles of 16 shells, batches of 16 and 32 rows, 512-
and 256-pixel tiles, a map that ends inside a tile, and counts of one, two,
three and four bytes (the last one signed).

Reference: the sums in extended precision on the host.  e and e^2 enter the
sums rounded to 43 bits of the tiles' maxima or finer, so a sum's error is at
most sum_b |n_bp| max|e| 2^-43 and the double-float e itself is within 2^-44 of
max(|E|, |C|): 2^-41 of the scale holds both with a margin of 2.  The number of
counts is a whole number and exact."""
import numpy as np
import pytest

from tests.gpu_common import api_ctx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [  # nside, shells, with g, largest |count|, negative counts too
    (1, 1, False, 3, False),
    (8, 15, True, 200, False),
    (8, 16, False, 255, False),
    (16, 17, True, 256, False),
    (32, 32, False, 65535, False),
    (8, 33, True, 65536, False),
    (32, 60, False, 40, False),
    (16, 64, False, (1 << 23) - 1, False),
    (16, 65, True, 1 << 23, False),
    (16, 96, True, 1 << 24, False),
    (16, 97, True, (1 << 31) - 1, False),
    (32, 108, False, 255, False),
    (32, 128, False, 256, False),
    (32, 129, False, 5, True),
    (16, 140, False, 100000, True),
    (64, 256, True, (1 << 31) - 1, True),
]


def to_dev(x):
    return torch.from_numpy(x).cuda()


def _counts(rng, S, npix, top, neg):
    n = rng.integers(0, min(top, 3) + 1, size=(S, npix))
    big = rng.random((S, npix)) < 0.02
    n[big] = rng.integers(0, top + 1, size=int(big.sum()))
    n[rng.integers(S), rng.integers(npix)] = top
    if neg:
        n = np.where(rng.random((S, npix)) < 0.3, -n, n)
        n[0, 0] = -top - 1 if top == (1 << 31) - 1 else -top
    return n.astype(np.int32)


@pytest.mark.parametrize("nside,S,use_g,top,neg", CASES)
def test_adjoint_sums_against_exact(nside, S, use_g, top, neg):
    _, ctx = api_ctx()
    npix = 12 * nside * nside
    rng = np.random.default_rng(1000 * nside + S)
    cn = _counts(rng, S, npix, top, neg)
    E = rng.normal(size=npix) * 10.0 ** rng.uniform(-4, 2, size=npix)
    C = 0.8125
    g = rng.normal(size=npix).astype(np.float32) if use_g else None
    sums, _, _, _ = ctx.kappa_adjoint_sums(to_dev(cn), to_dev(E), C,
                                           to_dev(g) if use_g else None)
    rows = sums[:4 * S].reshape(S, 4)
    n = cn.astype(np.longdouble)
    e = (E - C).astype(np.longdouble)
    an = np.abs(n).sum(1)
    scale = max(float(np.abs(e).max()), np.abs(E).max())
    for k, (q, s) in enumerate([(e, scale), (e * e, scale * scale),
                                (g.astype(np.longdouble) if use_g else 0 * e,
                                 float(np.abs(g).max()) if use_g else 0.0)]):
        err = np.abs(rows[:, k] - (n * q).sum(1))
        assert (err <= an * s * 2.0 ** -41).all(), (k, float((err / (an * s + 1e-300)).max()))
    assert np.array_equal(rows[:, 3], cn.astype(np.int64).sum(1).astype(np.float64))


@pytest.mark.parametrize("nside,S,use_g,top,neg", CASES)
def test_gradient_weights_against_exact(nside, S, use_g, top, neg):
    """The same shapes with the map from the counts themselves: G_b of
    w_var var + sum_p g_p kappa_p.  The weights A_b are FP32 numbers that keep
    the map below 16 (and exact in 64 bits for counts of at most 24 bits and a
    few shells; the host sums in extended precision)."""
    _, ctx = api_ctx()
    npix = 12 * nside * nside
    rng = np.random.default_rng(2000 * nside + S)
    cn = _counts(rng, S, npix, top, neg)
    n = cn.astype(np.longdouble)
    A = (rng.uniform(0.5, 1.5, size=S) * 8.0 / np.abs(n).sum(0).max().astype(np.float64)
         ).astype(np.float32).astype(np.float64)
    C = 0.015625
    g = rng.normal(size=npix).astype(np.float32) if use_g else None
    dA, dC = np.ones((5, S)), np.ones(5)
    grad, G, H = ctx.kappa_backward(to_dev(cn), A, C, dA, dC, 0.75, 0.0,
                                    to_dev(g) if use_g else None)
    # (the map takes a count as an FP32 number, rounded from 2^24 on, as the forward pass does)
    n32 = cn.astype(np.float32).astype(np.longdouble)
    e = (A.astype(np.longdouble)[:, None] * n32).sum(0) - C
    gl = g.astype(np.longdouble) if use_g else 0 * e
    ref = 0.75 * 2.0 * (n * (e - e.mean())).sum(1) / npix + (n * gl).sum(1)
    an = np.abs(n).sum(1)
    # the sums' error as above, the mean's as large again, and the products and
    # differences of 64-bit sums (2^-50)
    tol = an * (4.0 * 0.75 / npix * 12.0 + (np.abs(gl).max() if use_g else 0.0)) * 2.0 ** -41
    err = np.abs(G - ref)
    assert (err <= tol).all(), float((err / (tol + 1e-300)).max())
    assert abs(H - gl.sum()) <= 2.0 ** -41 * (float(np.abs(gl).sum()) + 1e-300)


@pytest.mark.parametrize("rising", [True, False])
def test_sums_of_an_ordered_map(rising):
    """A map in order of |e|: with rising values every tile has a new maximum, some
    of them in a new power of two, and what was summed before moves to the wider
    scale; the tolerance is that of the sums above."""
    _, ctx = api_ctx()
    nside, S = 128, 20
    npix = 12 * nside * nside
    rng = np.random.default_rng(5)
    cn = _counts(rng, S, npix, 300, False)
    E = 10.0 ** np.linspace(-3, 3, npix) * rng.choice([-1.0, 1.0], size=npix)
    if not rising:
        E = E[::-1].copy()
    sums, _, _, _ = ctx.kappa_adjoint_sums(to_dev(cn), to_dev(E), 0.0)
    rows = sums[:4 * S].reshape(S, 4)
    n, e = cn.astype(np.longdouble), E.astype(np.longdouble)
    for k, q in enumerate([e, e * e]):
        err = np.abs(rows[:, k] - (n * q).sum(1))
        # every term at the scale of its running maximum, which is at most the last one
        assert (err <= n.sum(1) * float(np.abs(q).max()) * 2.0 ** -41).all(), k
    assert np.array_equal(rows[:, 3], cn.astype(np.int64).sum(1).astype(np.float64))
