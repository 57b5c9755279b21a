"""Host set-up of the dense inverse of small meshes (no GPU): the band order is a permutation, the inverse is symmetric and
meets the residual bound of a Cholesky solve, matrices that are indefinite or whose inverse a precision cannot hold are
rejected, and the set-up stays within a small multiple of the multigrid set-up that it replaces (506 vertices: 6.0 times
before its sums ran in registers, 3.0 since; the limit lies between)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import shellgen as sg
from oracle import system as osys

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path_factory.mktemp("band") / "band_host_check")
    subprocess.run([gxx, "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "band_host_check.cpp"), "-lpthread"], check=True)
    return exe


@pytest.mark.parametrize("sc,limit", [(sg.plate_clamped_x0(16, model="EP"), None), (sg.cylinder_panel(24, "SS", ny=17), None),
                                      (sg.jittered_plate(22, steps=1), None), (sg.cylinder_panel(12, "ES", ny=3), None),
                                      (sg.cylinder_panel(22, "FS", ny=21), 4.5)], ids=lambda v: getattr(v, "name", None))
def test_band_inverse(checker, tmp_path, sc, limit):
    A = osys.system_matrix(osys.from_scenario(sc, factor=False)).tocsr()
    A.sort_indices()
    path = str(tmp_path / "A.bin")
    with open(path, "wb") as f:
        np.array([A.shape[0], A.nnz], dtype=np.int32).tofile(f)
        for a, t in ((A.indptr, np.int32), (A.indices, np.int32), (A.data, np.float64)):
            a.astype(t).tofile(f)
    out = subprocess.run([checker, path], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.startswith("OK"), out.stdout + out.stderr
    assert limit is None or float(out.stdout.split()[1]) <= limit
