"""Images of one hue, where every cyclic shift of the specification costs the same: the shift is the first minimiser of the
float costs over all shifts, as for every other image, repeated here in numpy term by term."""
import numpy as np
import pytest

from oracle import huepipe as hp

pytestmark = pytest.mark.gpu

TILE = 256


def _fma_square(d, part):
    """float32(d * d + part) with one rounding: the product is exact in double, the sum is rounded to odd first."""
    p, c = d.astype(np.float64) ** 2, part.astype(np.float64)
    s = p + c
    v = s - p
    err = (p - (s - v)) + (c - v)
    bits = s.view(np.int64)
    odd = (err != 0) & ((bits & 1) == 0)
    bits = np.where(odd, np.where(err > 0, bits + 1, bits - 1), bits)   # s >= 0
    return bits.view(np.float64).astype(np.float32)


def _first_minimum(x, y):
    n = len(x)
    hi = y.astype(np.float32)
    lo = (y - hi.astype(np.float64)).astype(np.float32)
    s = np.arange(n)
    cost = np.zeros(n)
    for r0 in range(0, n, TILE):
        part = np.zeros(n, np.float32)
        for r in range(r0, min(n, r0 + TILE)):
            q = (r - s) % n
            e = np.abs((x[r] - hi[q]) - lo[q])
            part = _fma_square(np.minimum(e, np.float32(1) - e), part)
        cost += part.astype(np.float64)
    return int(np.argmin(cost))


@pytest.mark.parametrize("n,hue", [(1500, 0.0), (2049, 0.0), (2500, 0.37), (3001, 1.0), (4099, 0.0), (4801, 0.37)])
def test_constant_image(n, hue):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_04840_gb300 import _build
    _build.build()
    from paper_1501_04840_gb300 import huepipe
    bins = 180
    h = np.full(n, hue, np.float32)
    target = np.random.default_rng(n).random(bins).astype(np.float32) ** 4
    out = huepipe.specify(torch.from_numpy(h).cuda(), bins, torch.from_numpy(target).cuda()).cpu().numpy()
    y = hp.target_hues(hp.exact_counts(target, n), bins)
    s = _first_minimum(h, y)
    assert np.array_equal(out, y[(np.arange(n) - s) % n].astype(np.float32))
