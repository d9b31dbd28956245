"""The packed path at scale 1 holds the values of the state as they are: infinities, NaN, the largest and the smallest FP32
numbers among them (state_set then state_get and path, no iteration between)."""
import numpy as np
import pytest

from _helpers import f32, oracle_grid, random_pair

pytestmark = pytest.mark.gpu

N, R = "neumann", "periodic"


@pytest.mark.parametrize("precision", [0, 2], ids=["f32", "f64"])
@pytest.mark.parametrize("n,bc,P", [((20, 12, 3), (N, N, R), 6), ((37,), (R,), 5)])
def test_values_pass_unchanged(n, bc, P, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_04840_gb300 import _build
    _build.build()
    import paper_1501_04840_gb300 as ot
    plan = ot.Plan(ot.grid(n, bc, P, precision=precision))
    f0, f1 = random_pair(oracle_grid(n, bc, P), 5)
    rng = np.random.default_rng(11)
    x = rng.standard_normal(plan.path_size).astype(np.float32)
    big, small = np.finfo(np.float32).max, np.float32(1e-45)
    odd = np.array([np.inf, -np.inf, np.nan, big, -big, small, -small, 3e-39, -0.0], np.float32)
    x[rng.permutation(len(x))[:9 * 4]] = np.tile(odd, 4)
    plan.state_set(f32(f0), f32(f1), x, np.zeros(plan.dual_size, np.float32))
    got = plan.state_get()[0]
    p = plan.path()
    path = np.concatenate([m.ravel() for m in p["m"]] + [p["f"].ravel()])
    nan = np.isnan(x)
    for v in (got, path):
        assert np.array_equal(np.isnan(v), nan)
        assert np.array_equal(v[~nan], x[~nan])
