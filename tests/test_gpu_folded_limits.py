"""Grids on either side of the rules that choose between the folded products and the dense sums (csrc/plan.cuh choose_mm):
the last FP32 lengths whose planes and strips fit shared memory and the first that do not, FP64 grids where either loads the
FP64 pipe less; one projection each against the FP64 oracle with the tolerances of test_gpu_parity."""
import numpy as np
import pytest

import oracle as o
from _helpers import correction_tolerance, f32, oracle_grid, pack_path, random_pair, rel, smooth_field

pytestmark = pytest.mark.gpu

N, R = "neumann", "periodic"
RGB = (N, N, R)
# at 227 KB of shared memory per block
F32 = [((359, 6, 3), RGB, 64), ((360, 6, 3), RGB, 64), ((401, 6, 3), (R, N, R), 64), ((624, 5, 1), (N, N, N), 32),
       ((641, 5, 1), (N, N, N), 32), ((4, 1023, 3), RGB, 6), ((4, 1031, 3), (N, R, R), 6)]
F64 = [((64, 150, 1), (N, N, N), 16), ((96, 130, 1), (N, N, N), 20), ((63,), (N,), 9), ((150, 24, 3), RGB, 12),
       ((36, 160, 3), RGB, 25), ((58, 59, 3), RGB, 48), ((33, 24, 3), (R, R, R), 9), ((128, 40, 3), RGB, 16), ((75, 64, 2), RGB, 16),
       ((100, 75, 4), RGB, 18)]


def _check(n, bc, P, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_04840_gb300 import _build
    _build.build()
    import paper_1501_04840_gb300 as ot
    plan = ot.Plan(ot.grid(n, bc, P, sigma=0.3, tau=0.99 / 0.3, precision=precision))
    g = oracle_grid(n, bc, P)
    rng = np.random.default_rng(3)
    f0, f1 = random_pair(g, 4)
    am = [smooth_field(g.m_shape(k), rng).astype(np.float32).astype(np.float64) for k in range(g.d)]
    af = smooth_field(g.f_shape, rng).astype(np.float32).astype(np.float64)
    m, f, phi = o.project(g, am, af, f0, f1)
    x, got = plan.project(f32(f0), f32(f1), f32(pack_path(g, am, af)), with_phi=True)
    tol = 1e-6 if precision == 2 else 1e-5
    assert rel(got, phi.ravel()) <= tol
    want = pack_path(g, m, f)
    assert rel(x, want) <= (tol if precision == 2 else correction_tolerance(g, phi, want))


@pytest.mark.parametrize("n,bc,P", F32, ids=["x".join(map(str, q[0])) + "_P%d" % q[2] for q in F32])
def test_shared_memory(n, bc, P):
    _check(n, bc, P, 0)


@pytest.mark.parametrize("n,bc,P", F64, ids=["x".join(map(str, q[0])) + "_P%d" % q[2] for q in F64])
def test_fp64_load(n, bc, P):
    _check(n, bc, P, 2)
