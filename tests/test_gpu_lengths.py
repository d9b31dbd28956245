"""GPU parity of the transforms over axis lengths (folded products, csrc/mm_kernels.cuh; fused FFT passes,
csrc/fft_kernels.cuh) against the FP64 oracle: one projection and one iteration per grid, with the tolerances of test_gpu_parity.  The grids sit at the
kernels' edges: lengths around whole groups of four outputs and eight time planes, one to four channels, odd and short
axes, P beside each register width, periodic axes with and without a Nyquist slot, and both precisions."""
import numpy as np
import pytest

import oracle as o
from _helpers import correction_tolerance, f32, oracle_grid, pack_path, random_pair, rel, smooth_field

pytestmark = pytest.mark.gpu

SIG, TAU = 0.3, 0.99 / 0.3
N, R = "neumann", "periodic"
RGB = (N, N, R)
GRIDS = [
    ((5, 3, 3), RGB, 3),
    ((37, 61, 4), (N, N, R), 33),
    ((180, 135, 3), RGB, 24),
    ((45, 200, 2), (N, N, N), 50),
    ((321, 33), (N, N), 64),
    ((63,), (N,), 9),
    ((31, 17, 3), (R, R, R), 5),
    ((30, 18, 3), (R, N, R), 25),
    ((100, 128, 3), RGB, 17),
    ((128, 100, 1), (N, N, N), 16),
    ((130, 7, 3), RGB, 49),
    ((2, 515, 3), RGB, 6),
    # FFT lengths (csrc/fft_kernels.cuh): every length on either axis, channels, and time lengths that fill, leave or
    # exceed a register transform
    ((512, 64, 3), RGB, 64),
    ((64, 512, 2), (N, N, N), 20),
    ((96, 96, 4), (R, N, R), 40),
    ((192, 128, 1), (N, R, N), 63),
    ((256, 192), (R, R), 16),
    ((512, 30), (R, N), 15),
    ((33, 256, 3), RGB, 3),
]
IDS = ["x".join(map(str, n)) + "_" + "".join(b[0] for b in bc) + "_P%d" % P for n, bc, P in GRIDS]


@pytest.fixture(scope="module")
def ot():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_04840_gb300 import _build
    _build.build()
    import paper_1501_04840_gb300 as p
    p.load_library()
    return p


@pytest.mark.parametrize("precision", [0, 2], ids=["f32", "f64"])
@pytest.mark.parametrize("n,bc,P", GRIDS, ids=IDS)
def test_projection(ot, n, bc, P, precision):
    _check_projection(ot, n, bc, P, precision, 2)


HUES = [(2, 2, 1), (9, 3, 2), (101, 20, 3), (360, 64, 1), (722, 33, 2), (37, 13, 90), (250, 64, 40), (1001, 17, 70),
        (3001, 8, 1)]


@pytest.mark.parametrize("precision", [0, 2], ids=["f32", "f64"])
@pytest.mark.parametrize("bins,P,batch", HUES)
def test_hue_projection(ot, bins, P, batch, precision):
    """Hue rows: sums in slices (few rows) and whole (many), chunks of slots, odd and even bins and P."""
    _check_projection(ot, (bins,), (R,), P, precision, batch)


def _check_projection(ot, n, bc, P, precision, batch):
    """Problems 0 and batch - 1 of one plan: phi to 1e-5 (1e-6 in FP64, the float32 output) and x to the FP32 bound of
    A^T phi."""
    plan = ot.Plan(ot.grid(n, bc, P, sigma=SIG, tau=TAU, precision=precision), batch=batch)
    g = oracle_grid(n, bc, P)
    rng = np.random.default_rng(3)
    ins, refs, phis = [], [], []
    for s in range(4, 4 + batch):
        f0, f1 = random_pair(g, s)
        am = [smooth_field(g.m_shape(k), rng).astype(np.float32).astype(np.float64) for k in range(g.d)]
        af = smooth_field(g.f_shape, rng).astype(np.float32).astype(np.float64)
        ins.append((f0, f1, pack_path(g, am, af)))
        m, f, phi = o.project(g, am, af, f0, f1) if s in (4, 3 + batch) else (None, None, None)
        refs.append(pack_path(g, m, f) if m is not None else None)
        phis.append(phi)
    x, phi = plan.project(*(f32(np.stack([p[k] for p in ins])) for k in range(3)), with_phi=True)
    x, phi = x.reshape(batch, -1), phi.reshape(batch, -1)
    for i in sorted({0, batch - 1}):
        tol = 1e-6 if precision == 2 else 1e-5
        assert rel(phi[i], phis[i].ravel()) <= tol
        assert rel(x[i], refs[i]) <= (tol if precision == 2 else correction_tolerance(g, phis[i], refs[i]))
