"""Residual checks of FP32 plans on states whose squares leave the FP32 range: the sums of the hue checks are those of FP64
for every finite state, and the sums across the lanes of the tiled checks do not overflow where a lane's own do not."""
import numpy as np
import pytest

import oracle as o
from _helpers import f32, oracle_grid

pytestmark = pytest.mark.gpu

SIG = 0.3
N, R = "neumann", "periodic"


def _plan(n, bc, P):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_04840_gb300 import _build
    _build.build()
    import paper_1501_04840_gb300 as ot
    return ot.Plan(ot.grid(n, bc, P, sigma=SIG, tau=0.99 / SIG)), tuple(n)


@pytest.mark.parametrize("n,bc,P,size", [((64,), (R,), 5, 4e19), ((101,), (R,), 16, 1e25), ((64, 16, 3), (N, N, R), 3, 4e18),
                                         ((33, 9, 2), (N, N, N), 3, 4e18)])
def test_large_state(n, bc, P, size):
    """x is a path constant in time, feasible as it is, b_f so low that the prox is zero: K x + (0, f_b^+) = (0, F) and the
    next b is b + (0, F).  The dual weights are those of the oracle's projection of zero."""
    plan, n = _plan(n, bc, P)
    rng = np.random.default_rng(2)
    F = f32(size * (0.25 + 0.75 * rng.random(n[::-1])))
    bf = np.float32(-1.5 * size)
    f = np.broadcast_to(F, (P - 1,) + F.shape).ravel()
    x = np.concatenate([np.zeros(plan.path_size - f.size, np.float32), f])
    b = np.concatenate([np.zeros(plan.dual_size - plan.N, np.float32), np.full(plan.N, bf)])
    plan.state_set(F, F, x, b, np.zeros_like(b))
    st = plan.iterate(1)
    F = F.astype(np.float64)
    g = oracle_grid(n, bc, P)
    _, f0, _ = o.project(g, [np.zeros(g.m_shape(k)) for k in range(g.d)], np.zeros(g.f_shape), F, F)
    w = o.S_F(g, f0) + o.f_b_plus(g, F, F)
    # the projection's rounding: 1e-5 of phi, which is zero but for rounding here
    assert st.residual == pytest.approx(1.0, rel=1e-4)
    assert st.energy == 0.0
    assert st.dual_value == pytest.approx(SIG * float(np.mean((float(bf) + F) * w)), rel=1e-4)
    assert st.mass_drift == pytest.approx(abs(F.sum() - F.size) / F.size, rel=1e-4)


def test_small_momenta():
    """f = 1 everywhere and b_m = 1e-25: the prox keeps v = 1 and u = z / (1 + z) b_m at z = sigma, and the energy is the
    mean of u^2 / 2, although u^2 is no FP32 number."""
    plan, n = _plan((96,), (R,), 7)
    one = np.ones(96, np.float32)
    x = np.concatenate([np.zeros(plan.path_size - 6 * 96, np.float32), np.ones(6 * 96, np.float32)])
    b = np.concatenate([np.full(plan.N, 1e-25, np.float32), np.zeros(plan.N, np.float32)])
    plan.state_set(one, one, x, b, np.zeros_like(b))
    st = plan.iterate(1)
    assert st.energy == pytest.approx(0.5 * (SIG / (1 + SIG) * 1e-25) ** 2, rel=1e-4, abs=0.0)
