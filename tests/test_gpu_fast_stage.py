"""The FP32 stages of the dense and the direct path at the edges of their form: pieces of 128 particles
with every kind of remainder (none, less than a piece, not a multiple of 4),
fewer pieces than warps, several shell edges in one bin of the lookup table,
particles at and around the observer, outside every shell, and non-finite or
overflowing coordinates.  Keys and counts are whole numbers: equal to the FP64
procedure's."""
import numpy as np
import pytest

from tests.gpu_common import api_ctx, both_boxes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nside,nshell", [(1, 16, 3), (127, 16, 3), (128, 32, 200), (129, 1, 1),
                                            (128 * 3648 + 5, 64, 7), (300_001, 256, 200),
                                            (1_000_000, 128, 40)])
def test_keys_and_counts_at_the_edges(orc, n, nside, nshell):
    api, ctx = api_ctx()
    L = 2000.0
    rng = np.random.default_rng(n + nside)
    x = rng.uniform(0.0, L, size=(n, 3)).astype(np.float32)
    k = n // 8
    x[:k] = 1000.0 + rng.normal(0.0, 1e-4, size=(k, 3))            # around the observer
    if n > 100:
        x[k] = 1000.0                                              # at it
        x[k + 1] = [np.nan, 1.0, 2.0]
        x[k + 2] = [np.inf, 0.0, 0.0]
        x[k + 3] = [3e38, -3e38, 3e38]                             # r^2 overflows
        x[k + 4] = [1e19, 0.0, 0.0]                                # r^2 = 1e38
        x[k + 5] = [1000.0, 1000.0, 1300.0]                        # on the polar axis
        x[k + 6] = [1300.0, 1000.0, 1000.0]
    # edges closer than a bin of the table at the low end, then wide shells
    m = nshell // 2
    chi = np.concatenate([0.5 * (1.0 + 1e-4 * np.arange(m)), np.linspace(5.0, 950.0, nshell + 1 - m)])
    if n > 100:                                                    # radii on and next to edges
        e = rng.choice(chi, size=16) * (1.0 + rng.choice([-1, 0, 1], size=16) * 1e-7)
        x[-16:, 0], x[-16:, 1], x[-16:, 2] = 1000.0 + e, 1000.0, 1000.0
    ba, bo = both_boxes(api, orc, L, [1000.0] * 3, n, 0, nshell)
    dev = torch.from_numpy(x).cuda()
    ref, inv = orc.bin_counts(x, bo, chi, nside)
    for path in ["direct"] + (["dense"] if nside >= 64 else []):   # (the dense path's least)
        counts = ctx.bin([dev], [ba], chi, nside, path=path).cpu().numpy()
        info = ctx.bin_info()
        assert np.array_equal(counts, ref), path
        assert info["invalid"] == inv and info["keyed"] == int(ref.sum())
    keys = ctx.keys(dev, ba, chi, nside).cpu().numpy()
    assert np.array_equal(keys, orc.keys(x, bo, chi, nside))
