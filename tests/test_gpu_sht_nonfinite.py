"""alm2map with a coefficient that is not finite: every pixel of the map is a
NaN, on the rings too whose share of that order is too small to be formed."""
import numpy as np
import pytest

from tests.gpu_common import api_ctx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside", [1, 16, 64, 256])
@pytest.mark.parametrize("value", [complex(np.nan, 0.0), complex(0.0, np.inf), complex(-1e300, 0.0)])
def test_not_finite_coefficient_reaches_every_pixel(nside, value):
    api, ctx = api_ctx()
    lmax = 3 * nside
    nalm = (lmax + 1) * (lmax + 2) // 2
    rng = np.random.default_rng(nside)
    base = rng.normal(size=nalm) + 1j * rng.normal(size=nalm)
    base[:lmax + 1] = base[:lmax + 1].real
    alm = torch.from_numpy(base).cuda()
    assert torch.isfinite(ctx.alm2map(alm, nside, lmax)).all()
    for l, m in ((lmax, lmax), (lmax, lmax // 2), (lmax // 2 + 1, lmax // 2), (lmax, 0)):
        if m == 0 and value.real == 0.0:
            continue                       # (the imaginary part of order 0 does not enter)
        i = m * (2 * lmax + 1 - m) // 2 + l
        bad = alm.clone()
        bad[i] = value
        out = ctx.alm2map(bad, nside, lmax)
        assert torch.isnan(out).all(), (l, m)
