"""a_lm and maps at sizes that take each of the Legendre kernels' block shapes
(ring pairs per block: 128, 256, 512, several blocks per order), with lmax
that no round of degrees divides, against an FP64 numpy recurrence for
selected orders."""
import numpy as np
import pytest

from tests.gpu_common import api_ctx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rings(N):
    """(first pixel, pixels, z, sin theta, first azimuth) of every ring."""
    out = []
    for i in range(1, 4 * N):
        k = min(i, 4 * N - i)
        if k < N:
            t = k * k / (3.0 * N * N)
            start = 2 * k * (k - 1) if i < 2 * N else 12 * N * N - 2 * k * (k + 1)
            out.append((start, 4 * k, (1 - t) if i < 2 * N else t - 1, np.sqrt(t * (2 - t)),
                        np.pi / (4 * k)))
        else:
            z = 4 / 3 - 2 * i / (3 * N)
            out.append((2 * N * (N - 1) + 4 * N * (i - N), 4 * N, z, np.sqrt(1 - z * z),
                        ((i - N + 1) % 2) * np.pi / (4 * N)))
    return out


def _lambda(m, lmax, z, s):
    """lambda_lm [lmax + 1 - m, rings] by the recurrence in l; values kept as
    v 2^e with an exponent per ring."""
    k = np.arange(1, m + 1)
    e = np.full(len(z), 0.5 * np.sum(np.log2((2 * k + 1) / (2 * k))) - 0.5 * np.log2(4 * np.pi))
    e = e + m * np.log2(s)
    n = np.floor(e)
    v1, v2 = (-1.0) ** m * 2.0 ** (e - n), np.zeros(len(z))
    out = np.empty((lmax + 1 - m, len(z)))
    for l in range(m, lmax + 1):
        if l > m:
            a = np.sqrt((4.0 * l * l - 1) / (l * l - m * m))
            b = np.sqrt(max((l - 1.0) ** 2 - m * m, 0.0) / (4 * (l - 1.0) ** 2 - 1))
            v1, v2 = a * (z * v1 - b * v2), v1
            big = np.abs(v1) > 2.0 ** 60
            f = np.where(big, 2.0 ** -60, 1.0)
            v1, v2, n = v1 * f, v2 * f, n + 60 * big
        out[l - m] = np.ldexp(v1, np.clip(n, -1000, 900).astype(int)) * (n > -1000)
    return out


SIZES = [(1, 4), (2, 3), (64, 151), (128, 300), (256, 513), (512, 700), (1024, 1025)]


def _orders(lmax):
    return sorted({0, 1, 2, lmax // 3, (2 * lmax) // 3, lmax - 1, lmax})


@pytest.mark.parametrize("nside,lmax", SIZES)
def test_map2alm_of_selected_orders(nside, lmax):
    api, ctx = api_ctx()
    rng = np.random.default_rng(nside + lmax)
    mp = (rng.normal(size=12 * nside ** 2) + (rng.random(12 * nside ** 2) < 0.01)).astype(np.float32)
    got = ctx.map2alm(torch.from_numpy(mp).cuda(), nside, lmax).cpu().numpy()
    rings = _rings(nside)
    z, s = np.array([r[2] for r in rings]), np.array([r[3] for r in rings])
    scale = np.abs(got).max()
    fft = [np.fft.fft(mp[st:st + n].astype(np.float64)) for st, n, *_ in rings]
    for m in _orders(lmax):
        F = np.array([f[m % r[1]] * np.exp(-1j * m * r[4]) for f, r in zip(fft, rings)])
        ref = 4 * np.pi / (12 * nside ** 2) * (_lambda(m, lmax, z, s) @ F)
        at = m * (2 * lmax + 1 - m) // 2
        # the tolerance of the oracle comparison (tests/test_gpu_sht.py)
        assert np.abs(got[at + m:at + lmax + 1] - ref).max() <= 1e-12 * scale * lmax, m


@pytest.mark.parametrize("nside,lmax", SIZES)
def test_alm2map_of_selected_orders(nside, lmax):
    api, ctx = api_ctx()
    rng = np.random.default_rng(nside + 7 * lmax)
    rings = _rings(nside)
    z, s = np.array([r[2] for r in rings]), np.array([r[3] for r in rings])
    alm = np.zeros((lmax + 1) * (lmax + 2) // 2, dtype=np.complex128)
    ref = np.zeros(12 * nside ** 2)
    for m in _orders(lmax):
        a = rng.normal(size=lmax + 1 - m) + 1j * rng.normal(size=lmax + 1 - m) * (m > 0)
        at = m * (2 * lmax + 1 - m) // 2
        alm[at + m:at + lmax + 1] = a
        g = a @ _lambda(m, lmax, z, s)
        for (st, n, _, _, p0), gm in zip(rings, g):
            ph = p0 + 2 * np.pi * np.arange(n) / n
            ref[st:st + n] += (2 - (m == 0)) * (gm * np.exp(1j * m * ph)).real
    got = ctx.alm2map(torch.from_numpy(alm).cuda(), nside, lmax).cpu().numpy()
    assert np.abs(got - ref).max() <= 2e-6 * np.abs(ref).max()
