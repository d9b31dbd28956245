"""Grids on either side of the rules that choose between the folded products and the dense sums (csrc/plan.cuh choose_mm,
choose_hue_mm): the last FP32 lengths whose planes, strips and rows fit shared memory and the first that do not, FP64 grids
where either loads the FP64 pipe less, and hue batches that take each form of the products; one projection each against the
FP64 oracle with the tolerances of test_gpu_parity."""
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
# bins, P, pairs, precision: few rows in slices, 8 and 16 rows per block, one and several chunks of items, chunks of 8 and
# 16 steps, per-row kernels
HUES = [(2339, 9, 1, 0), (2341, 9, 1, 0), (2905, 8, 1, 0), (720, 32, 8, 0), (720, 32, 16, 0), (1000, 64, 8, 0), (1000, 64, 16, 0),
        (850, 40, 32, 0), (500, 64, 64, 0), (360, 64, 24, 0), (101, 20, 60, 0), (37, 5, 160, 0), (1500, 17, 1, 0), (4096, 64, 1, 0), (3500, 20, 2, 0),
        (720, 32, 1, 2), (720, 32, 32, 2), (180, 36, 32, 2), (64, 16, 32, 2), (333, 27, 4, 2), (1024, 9, 1, 2)]


def _check(n, bc, P, precision, batch=1):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_04840_gb300 import _build
    _build.build()
    import paper_1501_04840_gb300 as ot
    plan = ot.Plan(ot.grid(n, bc, P, sigma=0.3, tau=0.99 / 0.3, precision=precision), batch=batch)
    g = oracle_grid(n, bc, P)
    rng = np.random.default_rng(3)
    ins, refs = [], {}
    for s in range(batch):
        f0, f1 = random_pair(g, 4 + s)
        am = [smooth_field(g.m_shape(k), rng).astype(np.float32).astype(np.float64) for k in range(g.d)]
        af = smooth_field(g.f_shape, rng).astype(np.float32).astype(np.float64)
        if s in (0, batch - 1):
            refs[s] = o.project(g, am, af, f0, f1)
        ins.append((f0, f1, pack_path(g, am, af)))
    x, got = plan.project(*(f32(np.stack([q[k] for q in ins])) for k in range(3)), with_phi=True)
    x, got = x.reshape(batch, -1), got.reshape(batch, -1)
    tol = 1e-6 if precision == 2 else 1e-5
    for s, (m, f, phi) in refs.items():
        assert rel(got[s], phi.ravel()) <= tol
        want = pack_path(g, m, f)
        assert rel(x[s], want) <= (tol if precision == 2 else correction_tolerance(g, phi, want))


@pytest.mark.parametrize("n,bc,P", F32, ids=["x".join(map(str, q[0])) + "_P%d" % q[2] for q in F32])
def test_shared_memory(n, bc, P):
    _check(n, bc, P, 0)


@pytest.mark.parametrize("n,bc,P", F64, ids=["x".join(map(str, q[0])) + "_P%d" % q[2] for q in F64])
def test_fp64_load(n, bc, P):
    _check(n, bc, P, 2)


@pytest.mark.parametrize("bins,P,batch,precision", HUES)
def test_hue(bins, P, batch, precision):
    _check((bins,), (R,), P, precision, batch)
