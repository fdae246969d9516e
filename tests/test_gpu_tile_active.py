"""The default handle of levels of up to 80,000 rows (FP32) and 60,000 rows (FP64) does run tiled sweeps: with
the colour launches chosen by hand on its finest level, a cycle has as many launches more as these take."""
import pytest

import meshgen
import paper_1505_03615_gb300 as L

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")


# parts: launches per sweep; two (from 12,000 rows on) have a launch of their own for the residual; 0: not tiled
@pytest.mark.parametrize("build,prec,rows,parts", [
    (lambda: L.lbmg_build_hierarchy(*meshgen.torus_knot_tube(2, 3, 1.0, 0.12, 48, 8, 1e-6, 3), 5), L.LBMG_FP64,
     (1000, 12_000), 1),
    (lambda: L.lbmg_build_hierarchy(*meshgen.double_sheet(60, 0.05, 6), 6), L.LBMG_FP64, (12_000, 60_000), 2),
    (lambda: L.lbmg_build_hierarchy(*meshgen.torus_knot_tube(2, 3, 1.0, 0.04, 600, 60, 1e-6, 2), 8), L.LBMG_MIXED,
     (60_000, 80_000), 2),
    (lambda: L.lbmg_build_hierarchy(*meshgen.torus_knot_tube(2, 3, 1.0, 0.04, 600, 60, 1e-6, 2), 8), L.LBMG_FP64,
     (60_000, 80_000), 0),
])
def test_the_finest_level_is_tiled(build, prec, rows, parts):
    h = build()
    try:
        L.lbmg_assemble(h, 1e-3)
        D = L.lbmg_levels(h)[1]
        assert rows[0] <= L.lbmg_level_info(h, D)[0] < rows[1]
        before = L.lbmg_launch_counts(h, prec)[2]
        L.lbmg_set_launch_shape(h, D, prec, 0, 4, 256)
        after = L.lbmg_launch_counts(h, prec)[2]
        # four sweeps, residual, restriction, prolongation against four sweeps with these, and the restriction
        assert after - before == ((4 * 8 + 3) - (4 * parts + (parts > 1) + 1) if parts else 0)
    finally:
        L.lbmg_destroy(h)
