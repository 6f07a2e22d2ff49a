"""Calls of one context that overlap on different streams, and under stream
capture: a Welford update keeps nothing outside the caller's state, so it may
run beside any other call, allocates nothing and can be captured before the
context has made a first call; a moment pass counts its blocks in the scratch
that holds its sums; a batched call has its own tables and counters."""
import ctypes

import numpy as np
import pytest

from paper_1801_05745_gb300 import synth
from tests.gpu_common import api_ctx, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _vectors(nvec, d, seed):
    return torch.from_numpy(np.random.default_rng(seed).normal(1.0, 0.1, size=(nvec, d))).cuda()


@pytest.mark.parametrize("d", [1, 206, 2049])
def test_welford_update_keeps_nothing_in_the_context(d):
    """No workspace, and the state of 17 + 2 vectors equals the host's chain."""
    api, _ = api_ctx()
    ctx = api.Context(0)
    try:
        held = ctx.workspace_bytes()
        v = _vectors(19, d, d)
        st = api.welford_state(d)
        ctx.welford_update(v[:17], st)
        ctx.welford_update(v[17:], st)
        torch.cuda.synchronize()
        assert ctx.workspace_bytes() == held
        one = api.welford_state(d)
        ctx.welford_update(v, one)
        torch.cuda.synchronize()
        assert torch.equal(st, one) and st[0].item() == 19.0
        # a mean of 19 values near 1 by 19 rounded steps, M2 by 19 fused ones: each
        # step errs by at most 2^-53 of values below 2 (a few steps for M2's sums)
        host = np.zeros(1 + d + d * d)
        api.welford_update_host(v.cpu().numpy(), host)
        assert np.abs(st.cpu().numpy() - host).max() <= 19 * 4 * 2.0 ** -52
    finally:
        ctx.close()


@pytest.mark.parametrize("d", [1, 15, 206, 256, 257])
def test_one_vector_at_a_time_equals_all_at_once(d):
    """One vector takes a launch of its own up to 256 components: the same bits."""
    api, ctx = api_ctx()
    v = _vectors(7, d, d + 1)
    st, one = api.welford_state(d), api.welford_state(d)
    ctx.welford_update(v, one)
    for r in range(7):
        ctx.welford_update(v[r:r + 1], st)
    torch.cuda.synchronize()
    assert torch.equal(st, one)


@pytest.mark.parametrize("nvec", [1, 5])
def test_first_welford_update_can_be_captured(nvec):
    api, _ = api_ctx()
    ctx = api.Context(0)
    try:
        v = _vectors(nvec, 206, 1)
        st = api.welford_state(206)
        ref = api.welford_state(206)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            ctx.welford_update(v, st)
        assert st.abs().max().item() == 0.0              # captured, not run
        for _ in range(2):
            graph.replay()
            ctx.welford_update(v, ref)
        torch.cuda.synchronize()
        assert torch.equal(st, ref)
    finally:
        ctx.close()


def test_welford_updates_overlap_with_each_other_and_with_moments():
    """Updates of two states and moment passes of a map, enqueued in turn on
    three streams without waiting: the same results as one after the other."""
    api, ctx = api_ctx()
    nside, rounds = 64, 24
    kap = torch.from_numpy(np.random.default_rng(3).normal(0.0, 0.01, 12 * nside * nside)
                           .astype(np.float32)).cuda()
    va, vb = _vectors(40, 1030, 4), _vectors(33, 46, 5)
    vc = _vectors(1, 206, 6)
    sa, sb, ra, rb, sc, rc = (api.welford_state(d) for d in (1030, 46, 1030, 46, 206, 206))
    m0, p0 = (t.clone() for t in ctx.map_stats(kap, nside, -0.05, 0.05, 64))
    for _ in range(rounds):
        ctx.welford_update(va, ra)
        ctx.welford_update(vb, rb)
        ctx.welford_update(vc, rc)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(3)]
    out = []
    for _ in range(rounds):
        with torch.cuda.stream(streams[0]):
            ctx.welford_update(va, sa)
        with torch.cuda.stream(streams[1]):
            ctx.welford_update(vb, sb)
            ctx.welford_update(vc, sc)
        with torch.cuda.stream(streams[2]):
            out.append(ctx.map_stats(kap, nside, -0.05, 0.05, 64))
    torch.cuda.synchronize()
    assert torch.equal(sa, ra) and torch.equal(sb, rb) and torch.equal(sc, rc)
    for m, p in out:
        assert torch.equal(m, m0) and torch.equal(p, p0)
    m, p = ctx.map_stats(kap, nside, -0.05, 0.05, 64)    # and the context still works
    torch.cuda.synchronize()
    assert torch.equal(m, m0) and torch.equal(p, p0)


def _noalloc(api, ctx, counts, A, C, lo, hi, nbins):
    S, npix = counts.shape
    kap = torch.empty(npix, dtype=torch.float32, device="cuda")
    mom = torch.empty(10, dtype=torch.float64, device="cuda")
    pdf = torch.empty(nbins + 3, dtype=torch.int64, device="cuda")
    ctx._stream()
    st = api._lib.ufc_kappa_stats_noalloc(
        ctx.h, ctypes.c_void_p(counts.data_ptr()), S, int(round((npix / 12) ** 0.5)),
        A.ctypes.data_as(ctypes.c_void_p), C, lo, hi, nbins, ctypes.c_void_p(kap.data_ptr()),
        ctypes.c_void_p(mom.data_ptr()), ctypes.c_void_p(pdf.data_ptr()))
    assert st == 0
    return kap, mom, pdf


def test_noalloc_call_overlaps_with_moment_passes_of_the_workspace():
    """ufc_kappa_stats_noalloc (scratch of its own) on one stream, ufc_kappa_stats
    (scratch in the workspace) on another: the results of both alone."""
    api, ctx = api_ctx()
    nside, S, nbins, lo, hi = 64, 5, 33, -0.5, 0.5
    rng = np.random.default_rng(9)
    counts = [torch.from_numpy(rng.poisson(3.0, (S, 12 * nside * nside)).astype(np.int32)).cuda()
              for _ in range(2)]
    A, C = np.linspace(0.01, 0.05, S), 0.4
    ref = [_noalloc(api, ctx, counts[0], A, C, lo, hi, nbins),
           ctx.kappa_stats(counts[1], A, C, lo, hi, nbins)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    out = []
    for _ in range(40):
        with torch.cuda.stream(streams[0]):
            out.append((0, _noalloc(api, ctx, counts[0], A, C, lo, hi, nbins)))
        with torch.cuda.stream(streams[1]):
            out.append((1, ctx.kappa_stats(counts[1], A, C, lo, hi, nbins)))
    torch.cuda.synchronize()
    for which, got in out:
        for a, b in zip(got, ref[which]):
            assert torch.equal(a, b)


def test_moment_passes_of_changing_sizes_clear_their_own_count():
    """The count's place depends on the map's size, so a pass finds the sums of
    passes of other sizes there: the results equal those of a new context."""
    api, _ = api_ctx()
    ctx = api.Context(0)
    try:
        for nside in (64, 16, 128, 1, 256, 32, 64, 2, 16):
            kap = torch.from_numpy(np.random.default_rng(nside).normal(0.0, 0.01, 12 * nside ** 2)
                                   .astype(np.float32)).cuda()
            m, p = ctx.map_stats(kap, nside, -0.05, 0.05, 64)
            new = api.Context(0)
            m0, p0 = new.map_stats(kap, nside, -0.05, 0.05, 64)
            torch.cuda.synchronize()
            new.close()
            assert torch.equal(m, m0) and torch.equal(p, p0)
    finally:
        ctx.close()


def _batch(api, orc, nreal, n, nside, nshell):
    z = np.linspace(0.1, 1.5, nshell + 1)
    chi = orc.chi_edges(0.3, 0.7, 1, z)
    split = int(np.argmin(np.abs(chi - 1000.0)))
    xs, boxes = [], []
    for r in range(nreal):
        xs.append([to_dev(synth.particles_numpy(n, 2000.0, 5.0, 700 + 2 * r)),
                   to_dev(synth.particles_numpy(n, 6400.0, 20.0, 701 + 2 * r))])
        boxes.append([api.make_box(2000.0, [1000.0] * 3, n, 0, split),
                      api.make_box(6400.0, [3200.0] * 3, n, split, nshell)])
    A = np.tile(np.linspace(0.01, 0.05, nshell), (nreal, 1))
    return chi, xs, boxes, A, np.full(nreal, 0.1)


def test_batched_call_leaves_the_last_binning_calls_diagnostics(orc):
    """ufc_bin_info tells of the last ufc_bin or ufc_keys call."""
    api, ctx = api_ctx()
    chi, xs, boxes, A, C = _batch(api, orc, 3, 20_000, 16, 6)
    ctx.bin([xs[0][0][:1234]], boxes[0][:1], chi, 16)
    info = ctx.bin_info()
    assert info["keyed"] > 0
    ctx.batched_stats(xs, boxes, chi, 16, A, C, -0.5, 0.5, 20, api.welford_state(26))
    assert ctx.bin_info() == info


def test_batched_call_overlaps_with_binning_and_kappa(orc):
    """Batched calls on one stream, binning (dense and direct, with other shell
    edges) and map statistics on two others: the results of each alone."""
    api, ctx = api_ctx()
    nside, nshell, nbins = 32, 8, 20
    chi, xs, boxes, A, C = _batch(api, orc, 12, 60_000, nside, nshell)
    chi2 = np.linspace(150.0, 900.0, 31)
    x2 = to_dev(synth.particles_numpy(700_001, 2000.0, 5.0, 77))
    b2 = [api.make_box(2000.0, [1000.0] * 3, 700_001, 0, 30)]
    kap = torch.from_numpy(np.random.default_rng(1).normal(0.0, 0.1, 12 * 64 * 64)
                           .astype(np.float32)).cuda()

    def batched():
        st = api.welford_state(6 + nbins)
        return [*ctx.batched_stats(xs, boxes, chi, nside, A, C, -0.5, 0.5, nbins, st), st]

    def others(path):
        return [ctx.bin([x2], b2, chi2, 128, path=path)]

    ref = [t.clone() for t in batched()]
    torch.cuda.synchronize()
    counts = {p: others(p)[0].clone() for p in ("dense", "direct")}
    stats = [t.clone() for t in ctx.map_stats(kap, 64, -0.5, 0.5, 50)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(3)]
    got = []
    for k in range(12):
        with torch.cuda.stream(streams[0]):
            got.append((batched(), ref))
        with torch.cuda.stream(streams[1]):
            p = ("dense", "direct")[k % 2]
            got.append((others(p), [counts[p]]))
        with torch.cuda.stream(streams[2]):
            got.append((ctx.map_stats(kap, 64, -0.5, 0.5, 50), stats))
    torch.cuda.synchronize()
    for a, b in got:
        for u, v in zip(a, b):
            assert torch.equal(u, v)


def test_adjoint_range_report_beside_binning(orc):
    """A cotangent outside the adjoint's fixed-point range is reported while binning
    calls, which clear their counters, run on another stream."""
    api, ctx = api_ctx()
    nside, S = 64, 3
    chi, xs, boxes, _, _ = _batch(api, orc, 1, 2_000, 16, 6)
    counts = torch.ones((S, 12 * nside * nside), dtype=torch.int32, device="cuda")
    counts[1, ::3] = 2
    g = torch.zeros(12 * nside * nside, dtype=torch.float32, device="cuda")
    g[7] = 3.0e4
    A, dA, dC = np.linspace(0.01, 0.02, S), np.zeros((5, S)), np.zeros(5)
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(20):
        with torch.cuda.stream(streams[0]):
            for _ in range(30):
                ctx.bin(xs[0], boxes[0], chi, 16)
        with torch.cuda.stream(streams[1]):
            with pytest.raises(api.UfcError, match="fixed-point range"):
                ctx.kappa_backward(counts, A, 0.04, dA, dC, 1.0, 0.0, g)
    torch.cuda.synchronize()
    g[7] = 1.0
    ctx.kappa_backward(counts, A, 0.04, dA, dC, 1.0, 0.0, g)       # and it was cleared
