"""The library built with tiles of 64 cells in the FP32C Euler reconstruction (WENO_K1_TILE), the largest it takes."""
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest

import synthetic as S
from oracle import OracleMesh, OracleSolver, Params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TOL = 2e-3  # the bound of the FP32C parity tests

RUN = """
import sys
import numpy as np
from paper_1712_08317_gb300 import _build
_build.build(force=True)
import synthetic as S
from paper_1712_08317_gb300.api import Mesh, Solver
assert _build.__file__.startswith(sys.argv[1])
out = {}
for kind in ("quad", "tri", "mixed"):
    mi = S.mesh_for_config(2, n=15, seed=3, kind=kind)
    W = S.cell_average(mi, S.density_wave)
    for characteristic in (False, True):
        sol = Solver(Mesh.from_input(mi), eqn="euler", precision="fp32c", characteristic=characteristic)
        U, Ul = sol.to_device(W)
        out[f"{kind}{int(characteristic)}"] = sol.to_host(sol.residual(U, Ul))
        sol.check()
np.savez(sys.argv[1] + "/out.npz", **out)
"""


def test_tiles_of_64_cells(tmp_path):
    for part in ("paper_1712_08317_gb300", "include"):
        shutil.copytree(os.path.join(ROOT, part), tmp_path / part, ignore=shutil.ignore_patterns("_obj", "*.so", "__pycache__"))
    env = dict(os.environ, WENO_NVCC_FLAGS="-DWENO_K1_TILE=64", PYTHONPATH=os.pathsep.join([str(tmp_path), ROOT]))
    r = subprocess.run([sys.executable, "-c", RUN, str(tmp_path)], cwd=tmp_path, env=env, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    with np.load(tmp_path / "out.npz") as out:
        for kind in ("quad", "tri", "mixed"):
            mi = S.mesh_for_config(2, n=15, seed=3, kind=kind)
            om, W = OracleMesh.from_input(mi), S.cell_average(mi, S.density_wave)
            for characteristic in (False, True):
                ref = OracleSolver(om, Params(characteristic=characteristic)).residual(W)
                scale = np.abs(ref).max(axis=1, keepdims=True)
                R = out[f"{kind}{int(characteristic)}"]
                assert float((np.abs(R - ref) / np.where(scale > 0, scale, 1.0)).max()) < TOL
