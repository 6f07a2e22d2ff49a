"""The forward pass over the counts at the edges of its form: rows held four at a
time (a remainder of 1 to 4 shells), maps that leave some threads without pixels
or with several, and counts whose FP32 conversion takes the other route (2^23
and more, or negative).

Reference: the same double-float operations, shell by shell, in FP32 on the
host (the fused multiply-adds formed exactly in extended precision and rounded
once), bit for bit."""
import numpy as np
import pytest

from tests.gpu_common import api_ctx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
f32, ld = np.float32, np.longdouble


def _two_sum(a, b):
    s = a + b
    bb = s - a
    return s, (a - (s - bb)) + (b - bb)


def _norm(h, l):
    s = h + l
    return s, l - (s - h)


def _sums(cn, A):
    """The unnormalised double-float sums sum_b A_b n_bp, the shells in order."""
    h = np.zeros(cn.shape[1], f32)
    l = np.zeros(cn.shape[1], f32)
    for b in range(cn.shape[0]):
        n = cn[b].astype(f32)
        ah = f32(A[b])
        al = f32(A[b] - np.float64(ah))
        ph = ah * n
        pe = (ld(ah) * n.astype(ld) - ph.astype(ld)).astype(f32)
        h, e = _two_sum(h, ph)
        l = l + (e + (ld(al) * n.astype(ld) + pe.astype(ld)).astype(f32))
    return h, l


@pytest.mark.parametrize("nside,S,top,neg", [
    (1, 1, 3, False), (1, 5, 1 << 23, False), (2, 4, 255, False), (16, 3, (1 << 23) - 1, False),
    (16, 7, 1 << 23, True), (64, 8, 300, False), (256, 9, (1 << 31) - 1, True),
    (512, 2, 40, False), (32, 256, 1 << 24, False)])
def test_map_and_partial_bit_for_bit(nside, S, top, neg):
    _, ctx = api_ctx()
    npix = 12 * nside * nside
    rng = np.random.default_rng(77 * nside + S)
    n = rng.integers(0, min(top, 5) + 1, size=(S, npix))
    big = rng.random((S, npix)) < 0.01
    n[big] = rng.integers(0, top + 1, size=int(big.sum()))
    n[S - 1, npix - 1] = top
    if neg:
        n[rng.random((S, npix)) < 0.2] *= -1
    cn = n.astype(np.int32)
    A = rng.uniform(-1.0, 1.0, size=S) / max(top, 1)
    C = 0.3
    eh, el = _norm(*_sums(cn, A))
    dev = torch.from_numpy(cn).cuda()
    part = ctx.kappa_partial(dev, A).cpu().numpy()
    assert np.array_equal(part, eh.astype(np.float64) + el.astype(np.float64))
    ch = f32(C)
    cl = f32(C - np.float64(ch))
    sh, se = _two_sum(eh, -ch)
    kh, kl = _norm(sh, se + (el - cl))
    kap, _, _ = ctx.kappa_stats(dev, A, C, -1.0, 1.0, 16)
    assert np.array_equal(kap.cpu().numpy(), kh + kl)


@pytest.mark.parametrize("nside", [1, 4, 64, 256])
def test_moments_of_an_unaligned_map(nside):
    """A map that is not 16-byte aligned takes the scalar loads of both passes: the
    map and the PDF are the same bit for bit; the sums run in another order, each
    in double-float (2^-44 per addition, the additions' errors spread over 2^5 and
    more partial sums): 1e-12 of the spread's powers."""
    _, ctx = api_ctx()
    npix, S = 12 * nside * nside, 5
    rng = np.random.default_rng(nside)
    dev = torch.from_numpy(rng.poisson(2.0, size=(S, npix)).astype(np.int32)).cuda()
    A = rng.uniform(0.5, 1.5, size=S) * 1e-3
    k0, m0, p0 = ctx.kappa_stats(dev, A, 0.01, -0.01, 0.02, 30)
    odd = torch.empty(npix + 1, dtype=torch.float32, device="cuda")[1:]
    k1, m1, p1 = ctx.kappa_stats(dev, A, 0.01, -0.01, 0.02, 30, kappa=odd)
    assert torch.equal(k0, k1) and torch.equal(p0, p1)
    m0, m1 = m0.cpu().numpy(), m1.cpu().numpy()
    sd = m0[1] ** 0.5
    for i, s in enumerate([sd, sd ** 2, sd ** 3, sd ** 4, 1.0, 1.0]):
        assert abs(m0[i] - m1[i]) <= 1e-12 * s, i
