"""Batched calls of more realisations than one launch takes (rows of a grid,
numbers of the binning's items): the same statistics as one map at a time."""
import numpy as np
import pytest

from paper_1801_05745_gb300 import synth
from tests.gpu_common import api_ctx, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nreal,nbox", [(65_540, 1), (65_540, 2), (7_720, 17)])
def test_many_realisations_equal_serial(orc, nreal, nbox):
    """65 535 realisations or 2^17 (realisation, box) items end a launch; more
    boxes than a binning call takes are accepted, as ever."""
    api, ctx = api_ctx()
    nside, nshell, nbins, lo, hi = 1, 2, 8, -0.5, 3.0
    chi = np.array([100.0, 500.0, 900.0])
    x = to_dev(synth.particles_numpy(4096, 2000.0, 5.0, 3))
    rng = np.random.default_rng(nreal + nbox)
    n = rng.integers(0, 40, (nreal, nbox))                 # empty ones among them
    at = rng.integers(0, 4096 - 40, (nreal, nbox))
    xs = [[x[a:a + m] for a, m in zip(ar, nr)] for ar, nr in zip(at, n)]
    box = api.make_box(2000.0, [1000.0] * 3, 40, 0, nshell)
    A = rng.uniform(0.1, 0.2, (nreal, nshell))
    C = rng.uniform(0.0, 0.1, nreal)
    d = 6 + nbins
    state = api.welford_state(d)
    mom, pdf, stats = ctx.batched_stats(xs, [[box] * nbox] * nreal, chi, nside, A, C, lo, hi, nbins,
                                        state)
    torch.cuda.synchronize()
    assert state[0].item() == nreal
    for r in (0, 1, 7_709, 7_710, 7_711, nreal // 2, 65_534, 65_535, 65_536, nreal - 1):
        if r >= nreal:
            continue
        counts = None
        for k in range(0, nbox, 16):                       # (a binning call takes 16 boxes)
            part = xs[r][k:k + 16]
            counts = ctx.bin(part, [box] * len(part), chi, nside, counts=counts, accumulate=k > 0)
        _, m, p = ctx.kappa_stats(counts, A[r], C[r], lo, hi, nbins)
        v = ctx.stats_vector(m, p)
        torch.cuda.synchronize()
        assert torch.equal(mom[r].view(torch.int64), m.view(torch.int64)), r   # (NaN included)
        assert torch.equal(pdf[r], p), r
        assert torch.equal(stats[r].view(torch.int64), v.view(torch.int64)), r
    assert int(pdf.sum().item()) == nreal * 12
