"""Tuning files from before the tiled sweep name the fastest colour launches; tiled levels stay tiled when
they are loaded, and the loaded entries stay what they are when saved again."""
import pytest

import meshgen
import paper_1505_03615_gb300 as L

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("form", ["nine", "eight", "now"])
def test_files_from_before_the_tiled_sweep_leave_levels_tiled(tmp_path, form):
    V, F = meshgen.torus(1.0, 0.3, 84, 30)
    hs = [L.lbmg_build_hierarchy(V, F, 6) for _ in range(3)]
    try:
        for h in hs:
            L.lbmg_assemble(h, 1e-2)
        d0, D = L.lbmg_levels(hs[0])
        default = L.lbmg_launch_counts(hs[0], L.LBMG_FP64)[2]
        for d in range(d0 + 1, D + 1):
            L.lbmg_set_launch_shape(hs[2], d, L.LBMG_FP64, 0, 4, 256)
        colours = L.lbmg_launch_counts(hs[2], L.LBMG_FP64)[2]
        assert default < colours
        L.lbmg_autotune(hs[0], 3, L.LBMG_FP64, reps=1)
        L.lbmg_tune_cache_save(str(tmp_path / "now.txt"))
        cols = [ln.split() for ln in (tmp_path / "now.txt").read_text().splitlines() if not ln.startswith("#")]
        head = {"nine": "# device fp64 kind lanes rows nnz threads_per_row threads_per_block [sweep_grid]\n", "eight": "",
                "now": "# device fp64 kind lanes rows nnz threads_per_row threads_per_block [sweep_grid, -1: tiled sweep]\n"}
        old = tmp_path / "old.txt"
        old.write_text(head[form] + "".join(" ".join(c[:8] + ([] if form == "eight" else ["0"])) + "\n" for c in cols))
        for again in range(2):
            L.lbmg_tune_cache_load(str(old))
            h = hs[1] if again == 0 else L.lbmg_build_hierarchy(V, F, 6)
            if again:
                L.lbmg_assemble(h, 1e-2)
                hs.append(h)
            assert L.lbmg_autotune(h, 3, L.LBMG_FP64, reps=1) == 0   # all from the file
            assert L.lbmg_launch_counts(h, L.LBMG_FP64)[2] == (colours if form == "now" else default)
            old = tmp_path / "again.txt"
            L.lbmg_tune_cache_save(str(old))
    finally:
        for h in hs:
            L.lbmg_destroy(h)
