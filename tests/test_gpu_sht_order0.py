"""alm2map takes the real field: the imaginary parts of the coefficients of
order 0 do not enter it, on rings of every kind of transform."""
import numpy as np
import pytest

from tests.gpu_common import api_ctx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,lmax", [(1, 4), (4, 9), (16, 47), (64, 130), (256, 300)])
def test_imaginary_part_of_order_0_does_not_enter(nside, lmax):
    api, ctx = api_ctx()
    nalm = (lmax + 1) * (lmax + 2) // 2
    rng = np.random.default_rng(nside)
    a = rng.normal(size=nalm) + 1j * rng.normal(size=nalm)
    b = a.copy()
    b[:lmax + 1] = b[:lmax + 1].real
    got, ref = (ctx.alm2map(torch.from_numpy(x).cuda(), nside, lmax) for x in (a, b))
    assert torch.equal(got, ref)
