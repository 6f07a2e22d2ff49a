"""The cached graph of ufc_batched_stats on the path that captures one (a launch
sequence per realisation on the lanes): relaunched by an identical call, updated
for other arguments, dropped when a lane's workspace grows."""
import numpy as np
import pytest

from paper_1801_05745_gb300 import synth
from tests.gpu_common import api_ctx, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NBINS, LO, HI = 30, -0.05, 0.2


def _set(orc, api, nreal, nside, nshell, n, seed=0):
    z = np.linspace(0.1, 1.5, nshell + 1)
    chi = orc.chi_edges(0.3, 0.7, 1, z)
    split = int(np.argmin(np.abs(chi - 1000.0)))
    xs, bxs, A, C = [], [], [], []
    src = api.make_source(kind=1, alpha=2.0, beta=1.5, z0=0.5, z_max=1.5)
    for r in range(nreal):
        xs.append([to_dev(synth.particles_numpy(n, 2000.0, 5.0, 1000 + seed + 2 * r)),
                   to_dev(synth.particles_numpy(n, 6400.0, 20.0, 1001 + seed + 2 * r))])
        bxs.append([api.make_box(2000.0, [1000.0] * 3, n, 0, split),
                    api.make_box(6400.0, [3200.0] * 3, n, split, nshell)])
        a, _, c = api.kappa_coeffs(api.make_cosmo(), bxs[-1], z, nside, src)
        A.append(a)
        C.append(c)
    return chi, xs, bxs, np.array(A), np.array(C)


class _Call:
    """One batched call with fixed output buffers, so that its arguments can be
    identical from call to call, and the one-at-a-time results to compare."""

    def __init__(self, api, ctx, data, nside):
        self.api, self.ctx, self.nside = api, ctx, nside
        self.chi, self.xs, self.bxs, self.A, self.C = data
        nreal, S = self.A.shape
        npix = 12 * nside * nside
        self.counts = torch.empty((S, npix), dtype=torch.int32, device="cuda")
        self.kappa = torch.empty(npix, dtype=torch.float32, device="cuda")
        self.state = api.welford_state(6 + NBINS)

    def run(self, lo=LO, hi=HI):
        """The outputs' storage is torch's: freed blocks of the same sizes come back
        at the same addresses, which makes a repeated call identical."""
        self.state.zero_()
        out = self.ctx.batched_stats(self.xs, self.bxs, self.chi, self.nside, self.A, self.C, lo, hi,
                                     NBINS, self.state, graph=True, launches=True,
                                     counts=self.counts, kappa=self.kappa)
        got = [t.clone() for t in out] + [self.state.clone()]
        ptrs = tuple(t.data_ptr() for t in out)
        return got, ptrs

    def check(self, got, lo=LO, hi=HI):
        mom, pdf, stats, state = got
        ref = self.api.welford_state(6 + NBINS)
        for r in range(len(self.xs)):
            counts = self.ctx.bin(self.xs[r], self.bxs[r], self.chi, self.nside)
            _, m, p = self.ctx.kappa_stats(counts, self.A[r], self.C[r], lo, hi, NBINS)
            v = self.ctx.stats_vector(m, p)
            self.ctx.welford_update(v.view(1, -1), ref)
            torch.cuda.synchronize()
            assert torch.equal(mom[r], m) and torch.equal(pdf[r], p) and torch.equal(stats[r], v), r
        assert torch.equal(state, ref)


@pytest.mark.parametrize("nreal", [3, 11])
def test_identical_call_relaunches_with_new_data(orc, nreal):
    api, ctx = api_ctx()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        call = _Call(api, ctx, _set(orc, api, nreal, 64, 10, 40_000), 64)
        ctx.profile(False)
        seen = []
        for k in range(3):
            if k:
                for row in call.xs:                      # new positions in the same buffers
                    for x in row:
                        x.copy_(torch.roll(x.flip(0), 1, dims=1))
            got, ptrs = call.run()
            stream.synchronize()
            call.check(got)
            seen.append(ptrs)
        assert seen[1] == seen[0] or seen[2] == seen[1]  # identical arguments: a relaunch


def test_other_arguments_update_the_graph(orc):
    """The PDF range, the coefficients and fewer realisations, each against the maps
    one at a time; then the first arguments again."""
    api, ctx = api_ctx()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        call = _Call(api, ctx, _set(orc, api, 10, 64, 12, 30_000), 64)
        for lo, hi in ((LO, HI), (-0.1, 0.3), (LO, HI)):
            got, _ = call.run(lo, hi)
            stream.synchronize()
            call.check(got, lo, hi)
        call.A, call.C = call.A * 0.5, call.C * 0.5
        got, _ = call.run()
        stream.synchronize()
        call.check(got)
        call.xs, call.bxs, call.A, call.C = call.xs[:4], call.bxs[:4], call.A[:4], call.C[:4]
        got, _ = call.run()
        stream.synchronize()
        call.check(got)


def test_workspace_growth_drops_the_graph(orc):
    """A call of few particles, one of fifty times as many, which grows the lanes'
    workspace (a context of its own, so that it does), and the first one again; maps
    of 39 MB, which take the dense binning path."""
    api, _ = api_ctx()
    ctx = api.Context(0)
    try:
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            small = _Call(api, ctx, _set(orc, api, 9, 128, 50, 20_000), 128)
            got, _ = small.run()
            stream.synchronize()
            held = ctx.workspace_bytes()
            small.check(got)
            large = _Call(api, ctx, _set(orc, api, 9, 128, 50, 1_000_000, seed=100), 128)
            got, _ = large.run()
            stream.synchronize()
            assert ctx.workspace_bytes() > held
            large.check(got)
            got, _ = small.run()
            stream.synchronize()
            small.check(got)
    finally:
        ctx.close()
