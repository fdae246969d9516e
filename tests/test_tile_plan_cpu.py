"""Host checks of the tiled sweep's plans, by a small program linked against the library."""
import os
import subprocess

import numpy as np
import pytest

import meshgen
import paper_1505_03615_gb300 as L
from paper_1505_03615_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))

MESHES = {
    "sphere": (5, [lambda: meshgen.icosphere(3, 1.0, 1e-3, 1)]),
    "sheet": (5, [lambda: meshgen.double_sheet(24, 0.05, 5)]),   # long rows
    "batch": (5, [lambda: meshgen.torus(1.0, 0.3, 40, 16), lambda: meshgen.icosphere(2, 1.0, 1e-3, 1)]),
}


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    L.load_library()
    exe = str(tmp_path_factory.mktemp("tile") / "check")
    lib = os.path.dirname(build.LIB)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fopenmp", "-ffp-contract=off", "-I", build.CSRC,
                           os.path.join(HERE, "tile_plan_check.cpp"), "-o", exe, build.LIB, f"-Wl,-rpath,{lib}"])
    return exe


def _run(program, mode, name, tmp_path):
    depth, makes = MESHES[name]
    files = []
    for k, make in enumerate(makes):
        V, F = make()
        path = tmp_path / f"{k}.bin"
        with open(path, "wb") as f:
            np.array([V.shape[0], F.shape[0]], dtype=np.int32).tofile(f)
            np.ascontiguousarray(V, dtype=np.float64).tofile(f)
            np.ascontiguousarray(F, dtype=np.int32).tofile(f)
        files.append(str(path))
    env = dict(os.environ, OMP_NUM_THREADS="4")
    done = subprocess.run([program, mode, str(depth), *files], env=env, capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stdout + done.stderr


def test_a_failed_host_allocation_comes_back_as_an_exception(program, tmp_path):
    """Also one that a thread of a parallel region meets: an exception that leaves the region, or a task,
    ends the process."""
    _run(program, "alloc", "sphere", tmp_path)


@pytest.mark.parametrize("name", ["sphere", "sheet", "batch"])
def test_every_tile_gives_the_whole_sweep_bit_for_bit(program, tmp_path, name):
    _run(program, "plan", name, tmp_path)
