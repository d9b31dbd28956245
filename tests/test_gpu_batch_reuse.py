"""A batch solved a second time: problems that the first solve retired take part in everything again, the dual weights of
the residual checks included, so the second solve's statistics are those of a fresh batch."""
import pytest

from _helpers import f32

pytestmark = pytest.mark.gpu


def test_statistics_of_a_second_solve():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_04840_gb300 import _build
    _build.build()
    import paper_1501_04840_gb300 as ot
    from paper_1501_04840_gb300 import synth
    grids = [ot.rgb_grid(24, 20, 8), ot.rgb_grid(24, 20, 8), ot.hue_grid(64, 16), ot.hue_grid(64, 16)]

    def pairs(seed):
        pr = [synth.rgb_pair(24, 20, 8, seed + k) for k in range(2)] + [synth.hue_pair(64, seed + k) for k in range(2)]
        return [f32(p[0]) for p in pr], [f32(p[1]) for p in pr]

    used, fresh = ot.Batch(grids), ot.Batch(grids)
    first = used.solve(*pairs(0), 4000, tol=1e-3, check_every=10)
    assert all(s.converged for s in first)          # every problem retires
    again, new = (b.solve(*pairs(10), 30, check_every=10) for b in (used, fresh))
    for a, n in zip(again, new):
        # the sums of a hue check meet in no fixed order: FP64 rounding of sums of up to 1e4 terms
        assert a.residual == pytest.approx(n.residual, rel=1e-9)
        assert a.energy == pytest.approx(n.energy, rel=1e-9)
        assert a.dual_value == pytest.approx(n.dual_value, rel=1e-9)
        assert a.gap == pytest.approx(n.gap, rel=1e-9, abs=1e-12)
