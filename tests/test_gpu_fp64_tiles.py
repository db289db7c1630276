"""FP64 reconstruction kernels at the edges of their tiles and of their arithmetic, against the oracle."""
import numpy as np
import pytest

import synthetic as S
from oracle import OracleMesh, OracleSolver, Params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1712_08317_gb300.api import Mesh, Solver  # noqa: E402

TOL = 1e-11  # the bound of the FP64 parity tests: max over cells of |dR|, relative to the largest |R| of the variable


def _compare(mi, W, **prm):
    osol = OracleSolver(OracleMesh.from_input(mi), Params(**prm))
    ref = osol.residual(W)
    sol = Solver(Mesh.from_input(mi), precision="fp64", **prm)
    U, _ = sol.to_device(W)
    R = sol.to_host(sol.residual(U))
    sol.check()
    scale = np.abs(ref).max(axis=1, keepdims=True)
    assert float((np.abs(R - ref) / np.where(scale > 0, scale, 1.0)).max()) < TOL


# tiles of 8, 16 and 32 columns (cells x variables), none of them filled by the last cells
@pytest.mark.parametrize("eqn,kind,n,characteristic,linear", [
    ("euler", "quad", 5, False, False), ("euler", "tri", 5, False, False), ("euler", "mixed", 7, True, False),
    ("euler", "quad", 51, False, False), ("euler", "tri", 37, True, False), ("euler", "quad", 73, False, False),
    ("euler", "tri", 51, False, True), ("euler", "quad", 9, True, True), ("scalar", "mixed", 11, False, False),
    ("scalar", "quad", 101, False, False)])
def test_ragged_tiles_match_oracle(eqn, kind, n, characteristic, linear):
    mi = S.mesh_for_config(2, n=n, seed=3, kind=kind)
    W = S.cell_average(mi, S.scalar_wave if eqn == "scalar" else S.density_wave)
    _compare(mi, W, eqn=eqn, characteristic=characteristic, linear=linear)


# eps^2 = 2.6e-308 at the cells whose indicators are zero: below the range in which the kernels take
# reciprocals by iteration, so those Gauss points are redone with IEEE division
@pytest.mark.parametrize("kind", ["quad", "tri"])
def test_weights_outside_the_iteration_range_match_oracle(kind):
    mi = S.mesh_for_config(2, n=9, seed=3, kind=kind)
    W = np.ones((1, mi.n_cells))
    W[0, mi.n_cells // 2] = 1.25
    _compare(mi, W, eqn="scalar", eps=1.6e-154)


@pytest.mark.parametrize("precision", ["fp64", "fp32c"])
def test_autotune_works_on_the_given_state(precision):
    """The passes are timed on the state's own Gauss values: a physical state raises no flag."""
    mi = S.mesh_for_config(2, n=21, seed=3, kind="mixed")
    sol = Solver(Mesh.from_input(mi), eqn="euler", precision=precision)
    U, Ul = sol.to_device(S.cell_average(mi, S.density_wave))
    sol.autotune(U, Ul)
    sol.check()
