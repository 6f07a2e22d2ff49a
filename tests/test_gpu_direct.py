"""The direct binning path, the batched call's stages and the Welford update at
the sizes where their splits have edges: particle counts around a warp, a task
and the chip, periodic images whose list is cut by the particles' bounds, and
vectors around the update's tile and run."""
import numpy as np
import pytest

from paper_1801_05745_gb300 import synth
from tests.gpu_common import api_ctx, both_boxes, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2", [(0, 1), (31, 32), (33, 95), (97, 0), (1023, 40_001),
                                   (350_209, 2_000_003)])
def test_direct_counts_match_oracle(orc, n1, n2):
    api, ctx = api_ctx()
    nside, nshell = 32, 11
    chi = orc.chi_edges(0.3, 0.7, 1, np.linspace(0.1, 1.5, nshell + 1))
    x = [synth.particles_numpy(n1, 2000.0, 5.0, 91), synth.particles_numpy(n2, 6400.0, 20.0, 92)]
    for k in range(2):                         # invalid ones among them
        x[k][5::97, 1] = np.nan
        x[k][7::101, 2] = np.inf
    b1 = both_boxes(api, orc, 2000.0, [1000.0] * 3, max(n1, 1), 0, 4)
    b2 = both_boxes(api, orc, 6400.0, [3200.0] * 3, max(n2, 1), 4, nshell)
    ref = np.zeros((nshell, 12 * nside * nside), np.int32)
    ninv = 0
    for xk, b in zip(x, (b1, b2)):
        orc.bin_counts(xk, b[1], chi, nside, ref)
        ninv += int((~np.isfinite(xk).all(axis=1)).sum())
    # views at a 4-byte offset: the path takes any float alignment
    dev = [to_dev(np.concatenate([[0.0], xk.ravel()]))[1:].view(-1, 3) for xk in x]
    got = ctx.bin(dev, [b1[0], b2[0]], chi, nside, path="direct")
    assert np.array_equal(got.cpu().numpy(), ref)
    info = ctx.bin_info()
    assert info["invalid"] == ninv and info["keyed"] == int(ref.sum())
    got = ctx.bin(dev, [b1[0], b2[0]], chi, nside, counts=got, accumulate=True, path="direct")
    assert np.array_equal(got.cpu().numpy(), 2 * ref)


@pytest.mark.parametrize("n,layers,spread", [(1, 1, 1.0), (33, 2, 1.0), (5000, 4, 1.0),
                                             (4001, 3, 3.0), (3000, 2, 0.05)])
def test_images_cut_by_bounds_match_oracle(orc, n, layers, spread):
    """Positions over `spread` boxes (also outside [0, L)), the observer off
    centre, shells that do not reach the observer: the image list drops images
    on both sides, and the counts equal the oracle's over all images."""
    api, ctx = api_ctx()
    nside, L = 16, 500.0
    rng = np.random.default_rng(n + layers)
    x = ((rng.random((n, 3)) - 0.5) * spread + 0.5).astype(np.float32) * np.float32(L)
    if n > 100:
        x[11] = [np.nan, 1.0, 2.0]
        x[12] = [1e30, 1.0, 2.0]               # r^2 overflows FP32
    obs = [100.0, 250.0, 490.0]
    chi = np.linspace(300.0, 900.0, 8)
    ba, bo = both_boxes(api, orc, L, obs, n, 1, 6, layers)
    ref = np.zeros((7, 12 * nside * nside), np.int32)
    orc.bin_counts(x, bo, chi, nside, ref)
    got = ctx.bin([to_dev(x)], [ba], chi, nside)
    assert np.array_equal(got.cpu().numpy(), ref)


def test_images_around_the_observer(orc):
    """The first shell starts next to the observer and a particle sits on it:
    images that hold the observer stay in the list."""
    api, ctx = api_ctx()
    rng = np.random.default_rng(3)
    x = (rng.random((2000, 3)) * 400.0).astype(np.float32)
    x[5] = [200.0, 200.0, 200.0]
    chi = np.array([0.5, 10.0, 50.0, 350.0])
    ba, bo = both_boxes(api, orc, 400.0, [200.0] * 3, 2000, 0, 3, 1)
    ref = np.zeros((3, 12 * 8 * 8), np.int32)
    orc.bin_counts(x, bo, chi, 8, ref)
    assert np.array_equal(ctx.bin([to_dev(x)], [ba], chi, 8).cpu().numpy(), ref)
    assert ctx.bin_info()["invalid"] == 1


@pytest.mark.parametrize("sizes", [[(1, 0)], [(0, 0), (40, 33), (0, 5000)],
                                   [(3000 + 7 * r, 2500 - 11 * r) for r in range(9)]])
def test_batched_odd_sizes_equal_serial(orc, sizes):
    api, ctx = api_ctx()
    nside, nshell, nbins, lo, hi = 16, 6, 21, -0.3, 0.9
    z = np.linspace(0.1, 1.5, nshell + 1)
    chi = orc.chi_edges(0.3, 0.7, 1, z)
    xs, bxs, A, C = [], [], [], []
    for r, (n1, n2) in enumerate(sizes):
        xs.append([to_dev(synth.particles_numpy(n1, 2000.0, 5.0, 2 * r)),
                   to_dev(synth.particles_numpy(n2, 6400.0, 20.0, 2 * r + 1))])
        bxs.append([api.make_box(2000.0, [1000.0] * 3, max(n1, 1), 0, 2),
                    api.make_box(6400.0, [3200.0] * 3, max(n2, 1), 2, nshell)])
        a, _, c = api.kappa_coeffs(api.make_cosmo(), bxs[-1], z, nside, api.make_source(kind=1))
        A.append(a)
        C.append(c)
    st = api.welford_state(6 + nbins)
    for _ in range(2):                         # the second call reuses the staging buffer
        st.zero_()
        mom, pdf, vec = ctx.batched_stats(xs, bxs, chi, nside, np.array(A), np.array(C), lo, hi,
                                          nbins, st)
    st_s = api.welford_state(6 + nbins)
    for r in range(len(sizes)):
        counts = ctx.bin(xs[r], bxs[r], chi, nside)
        _, m, p = ctx.kappa_stats(counts, A[r], C[r], lo, hi, nbins)
        v = ctx.stats_vector(m, p)
        ctx.welford_update(v.view(1, -1), st_s)
        for got, ref in ((mom[r], m), (vec[r], v)):
            assert torch.equal(got.view(torch.int64), ref.view(torch.int64)), r   # (NaN included)
        assert torch.equal(pdf[r], p), r
    assert torch.equal(st.view(torch.int64), st_s.view(torch.int64))


@pytest.mark.parametrize("d", [1, 15, 16, 17, 33, 206])
@pytest.mark.parametrize("nvec", [1, 15, 16, 17, 40])
def test_welford_tiles_and_runs(orc, d, nvec):
    """Tiles of 16 x 16 elements and runs of 16 vectors, against numpy; two
    updates in a row equal one, bit for bit."""
    api, ctx = api_ctx()
    rng = np.random.default_rng(100 * d + nvec)
    v = rng.normal(size=(nvec, d)) * 10.0 ** rng.integers(-3, 4, size=d) + 5.0
    dev = torch.from_numpy(v).cuda()
    st, two = api.welford_state(d), api.welford_state(d)
    ctx.welford_update(dev, st)
    ctx.welford_update(dev[:nvec // 2 + 1], two)
    if nvec > 1:
        ctx.welford_update(dev[nvec // 2 + 1:], two)
    assert torch.equal(st, two)
    h = st.cpu().numpy()
    mean = v.mean(axis=0)
    m2 = (v - mean).T @ (v - mean)
    assert h[0] == nvec
    assert np.allclose(h[1:1 + d], mean, rtol=1e-13)
    s = np.sqrt(np.outer(np.diag(m2), np.diag(m2)))
    # 1e-12 of the product of the components' spreads, plus the rounding of the
    # deltas against the means
    eps = 1e-12 * s + 1e-14 * nvec * np.outer(np.abs(v).max(0), np.abs(v).max(0))
    assert np.all(np.abs(h[1 + d:].reshape(d, d) - m2) <= eps + 1e-300)
