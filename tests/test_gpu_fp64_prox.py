"""The FP64 plan's prox (FP32 start, FP64 Newton) against the oracle over the scales that its branch accepts and beyond:
one iteration from a zero path and duals of mixed magnitude, cell by cell to the float32 output."""
import numpy as np
import pytest

import oracle as o
from _helpers import f32, oracle_grid, pack_dual, random_pair

pytestmark = pytest.mark.gpu

SIG, TAU = 0.3, 0.99 / 0.3


@pytest.mark.parametrize("lo,hi", [(-9, -3), (-2, 2), (3, 7), (9, 11)])
def test_dual_step(lo, hi):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_04840_gb300 import _build
    _build.build()
    import paper_1501_04840_gb300 as ot
    n, bc, P = (20, 12, 3), ("neumann", "neumann", "periodic"), 6
    plan = ot.Plan(ot.grid(n, bc, P, sigma=SIG, tau=TAU, precision=ot.PREC_FP64))
    g = oracle_grid(n, bc, P)
    rng = np.random.default_rng(7)
    shape = g.cell_shape
    scale = 10.0 ** rng.uniform(lo, hi, shape)
    bm = [(scale * rng.standard_normal(shape)).astype(np.float32).astype(np.float64) for _ in range(3)]
    # half of the cells just inside or outside the zero case b_f = -sigma |b_m|^2 / 2
    edge = -0.5 * SIG * sum(v * v for v in bm) * (1 + 1e-3 * rng.standard_normal(shape))
    bf = np.where(rng.random(shape) < 0.5, edge, scale * rng.standard_normal(shape)).astype(np.float32).astype(np.float64)
    f0, f1 = random_pair(g, 2)
    zero = np.zeros(plan.path_size, np.float32)
    dual = f32(pack_dual(g, bm, bf))
    plan.state_set(f32(f0), f32(f1), zero, dual, np.zeros_like(dual))
    plan.iterate(1)
    _, b, _ = plan.state_get()
    # K x + (0, f_b^+) of the projected zero path, then b + K x - prox
    m, f, _ = o.project(g, [np.zeros(g.m_shape(k)) for k in range(3)], np.zeros(g.f_shape), f0, f1)
    u = [o.S_M(g, m)[k] + bm[k] for k in range(3)]
    v = o.S_F(g, f) + o.f_b_plus(g, f0, f1) + bf
    pu, pv = o.prox_J(u, v, SIG)
    want = pack_dual(g, [a - c for a, c in zip(u, pu)], v - pv)
    size = pack_dual(g, [np.maximum(np.abs(a), np.abs(c)) for a, c in zip(u, pu)], np.abs(v) + np.abs(pv))
    # float32 output plus the rounding of the differences from numbers of this size
    assert np.all(np.abs(b - want) <= 2.0 ** -23 * np.abs(want) + 1e-12 * size + 1e-12)
