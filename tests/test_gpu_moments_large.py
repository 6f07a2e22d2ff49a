"""Moments of the largest maps a thread adds hundreds of pixels of: a map of two
values, where the rounding errors of a thread's sums are the same in every thread
and do not average out."""
from fractions import Fraction

import numpy as np
import pytest

from tests.gpu_common import api_ctx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1])
def test_two_valued_map(offset):
    """mu2 = c^2 and mu4 = c^4 of a map of +-c.  At Nside 4096 a thread adds 650
    pairs of pixels (of two threads' halves side by side) to its sums.  The low part
    of a sum that is renormalised every four additions stays below 5 2^-24 of the
    high part; an addition rounds it twice, so errs by less than 2^-46 of the sum
    so far: 325 2^-46 in all, and 2^-42 for the products, lanes and blocks.  offset
    1: a map that is not 16-byte aligned (through the counts: scalar loads)."""
    api, ctx = api_ctx()
    nside = 4096
    npix = 12 * nside * nside
    tol = 325 * 2.0 ** -46 + 2.0 ** -42
    if offset == 0:
        m = torch.empty(npix, dtype=torch.float32, device="cuda").view(-1, 2)
    else:
        counts = (torch.arange(npix, device="cuda", dtype=torch.int32) & 1).view(1, npix) * 2
        buf = torch.empty(npix + 4, dtype=torch.float32, device="cuda")
    for c in (0.00713, 0.0091, 0.0117, 0.01321, 0.0158, 0.0177):
        c = np.float32(c)
        if offset == 0:
            m[:, 0], m[:, 1] = float(c), -float(c)
            mom, _ = ctx.map_stats(m.view(-1), nside, -0.05, 0.05, 50)
        else:
            _, mom, _ = ctx.kappa_stats(counts, np.array([float(c)]), float(c), -0.05, 0.05, 50,
                                        kappa=buf[1:1 + npix])
        got = mom.cpu().numpy()
        c2 = Fraction(float(c)) ** 2
        assert got[0] == 0.0
        assert abs(float((Fraction(float(got[1])) - c2) / c2)) <= tol
        assert abs(float((Fraction(float(got[3])) - c2 * c2) / (c2 * c2))) <= tol
