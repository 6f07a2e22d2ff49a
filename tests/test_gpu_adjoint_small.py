"""The adjoint's per-shell sums of small maps: the fixed-point rows keep e^2 to
2^-56, so what a block adds to them has to be rounded once and without bias."""
import numpy as np
import pytest

from tests.gpu_common import api_ctx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,nshell,use_g", [(32, 10, False), (64, 40, True), (128, 140, False),
                                                (64, 130, True)])
def test_second_sums_of_a_small_map(nside, nshell, use_g):
    """S2_b = sum_p e_p^2 n_bp of a map of values near 1e-6 against quad
    precision.  Rounded to nearest at 2^-56, the blocks' shares (at most one per
    256 pixels, and for each at most one flush per scale it meets, fewer than 8)
    err by 2^-57 each at most and like the root of their number together: 6
    standard deviations of sqrt(8 blocks) 2^-56 / sqrt(12), and the quantised e^2
    by 2^-42 of its maximum per count, as randomly.  (Dropped bits give a bias of
    up to 6 2^-57 per share, many times that.)"""
    api, ctx = api_ctx()
    npix = 12 * nside * nside
    rng = np.random.default_rng(nside + nshell)
    cn = torch.from_numpy(rng.poisson(1.3, (nshell, npix)).astype(np.int32)).cuda()
    e = (rng.normal(0.0, 1e-6, npix)).astype(np.float32).astype(np.float64)
    g = torch.from_numpy(rng.normal(0.0, 1.0, npix).astype(np.float32)).cuda() if use_g else None
    sm, _, _, _ = ctx.kappa_adjoint_sums(cn, torch.from_numpy(e).cuda(), 0.0, g_kappa=g)
    got = sm[:4 * nshell].reshape(nshell, 4)[:, 1]
    c = cn.cpu().numpy().astype(np.longdouble)
    e2 = e.astype(np.longdouble) ** 2
    ref = c @ e2
    blocks = npix // 256 + 1
    tol = 6 * np.sqrt(8.0 * blocks / 12) * 2.0 ** -56
    tol += 6 * 2.0 ** -42 * float(e2.max()) * np.sqrt(float((c ** 2).sum(1).max()))
    assert np.abs((got - ref).astype(float)).max() <= tol
