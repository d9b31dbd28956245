"""The least-cost cyclic shift of the hue specification (csrc/huepipe.cu) against the cost of every shift in FP64: images
at the edge between the exhaustive search and the convex one (2048 pixels), lengths that are not whole tiles or sort
runs, hues that sit at the wrap, coincide or lie outside [0, 1)."""
import numpy as np
import pytest

from oracle import huepipe as hp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_04840_gb300 import _build
    _build.build()
    from paper_1501_04840_gb300 import huepipe
    huepipe.lib()
    return huepipe


def _hues(kind, n, rng):
    if kind == "wrap":
        return ((0.02 * rng.standard_normal(n)) % 1.0).astype(np.float32) % np.float32(1)
    if kind == "constant":
        return np.full(n, 0.37, np.float32)
    if kind == "two":
        return np.where(rng.random(n) < 0.4, 0.999, 0.25).astype(np.float32)
    return rng.random(n).astype(np.float32) * np.float32(1.5 if kind == "outside" else 0.999)


@pytest.mark.parametrize("kind", ["uniform", "wrap", "constant", "two", "outside"])
@pytest.mark.parametrize("n", [3, 2048, 2049, 4097, 10007])
def test_shift_is_least(H, n, kind):
    import torch
    rng = np.random.default_rng(n)
    bins = 180
    h = _hues(kind, n, rng)
    target = rng.random(bins).astype(np.float32) ** 4
    out = H.specify(torch.from_numpy(h).cuda(), bins, torch.from_numpy(target).cuda()).cpu().numpy()
    cnt = hp.exact_counts(target, n)
    start = np.cumsum(cnt) - cnt
    b = np.repeat(np.arange(bins), cnt)
    y = (b + (np.arange(n) - start[b] + 0.5) / cnt[b]) / bins
    order = np.lexsort((np.arange(n), np.minimum(np.floor(h.astype(np.float64) * 2.0 ** 32), 2.0 ** 32 - 1)))
    x = h[order].astype(np.float64)
    # the shift of the output, from the pixel of rank 0, then every pixel
    s = -int(np.flatnonzero(y.astype(np.float32) == out[order[0]])[0]) % n
    assert np.array_equal(out[order], y[(np.arange(n) - s) % n].astype(np.float32))
    cost = np.empty(n)
    for s0 in range(0, n, 512):
        q = (np.arange(n)[None, :] - np.arange(s0, min(n, s0 + 512))[:, None]) % n
        e = np.abs(x[None, :] - y[q])
        cost[s0:s0 + 512] = (np.minimum(e, 1 - e) ** 2).sum(1)
    # the float sums of 256 terms: 1e-5 of the cost
    assert cost[s] <= cost.min() * (1 + 1e-5) + 1e-12
