"""FP32C Euler: cells redone with FP64 weights within the pass, in each instance of the reconstruction."""
import numpy as np
import pytest

import synthetic as S
from oracle import OracleMesh, OracleSolver, Params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1712_08317_gb300.api import Mesh, Solver  # noqa: E402

TOL = 2e-3  # the bound of the FP32C parity tests: max over cells of |dR|, relative to the largest |R| of the variable


def _steep(x, y):
    """Isothermal density ramp, moving: the indicators of every cell, 1e9 and more at these sizes (1e7^2 |Omega|),
    are outside the FP32 range component-wise and in the entropy field, and no Gauss point leaves the physical set."""
    rho = 1e7 * (0.5 + x + 0.3 * y)
    one = np.ones_like(rho)
    return S.euler_prim_to_cons(rho, one, 0.5 * one, rho, 1.4)


def _residual(mesh, W, characteristic):
    sol = Solver(mesh, eqn="euler", precision="fp32c", characteristic=characteristic)
    U, Ul = sol.to_device(W)
    R = sol.to_host(sol.residual(U, Ul))
    sol.check()
    assert np.isfinite(R).all()
    return R


# Below and above three 16-cell tiles an SM, where a thread of the characteristic kernel has one face of its cell
# and all of them: there its warp redoes what its lanes have stored
@pytest.mark.parametrize("characteristic", [False, True])
@pytest.mark.parametrize("kind", ["quad", "tri", "mixed"])
@pytest.mark.parametrize("large", [False, True])
def test_redone_cells_match_the_oracle(kind, characteristic, large):
    tiles = 3.2 * torch.cuda.get_device_properties(0).multi_processor_count if large else 6.3
    n = int(np.sqrt(16 * tiles / {"quad": 1.0, "tri": 2.0, "mixed": 1.3}[kind])) | 1
    mi = S.mesh_for_config(3, n=n, seed=2, kind=kind)
    mi.walls = (0, 3)
    W = S.cell_average(mi, _steep)
    ref = OracleSolver(OracleMesh.from_input(mi), Params(characteristic=characteristic)).residual(W)
    R = _residual(Mesh.from_input(mi), W, characteristic)
    scale = np.abs(ref).max(axis=1, keepdims=True)
    assert float((np.abs(R - ref) / scale).max()) < TOL


@pytest.mark.parametrize("characteristic", [False, True])
@pytest.mark.parametrize("kind", ["quad", "tri", "mixed"])
def test_redone_cells_have_the_same_bits_alone_and_in_a_large_batch(kind, characteristic):
    mi = S.mesh_for_config(3, n=13, seed=7, kind=kind)
    mi.walls = (0, 3)
    W = S.cell_average(mi, _steep)
    mesh = Mesh.from_input(mi)
    copies = 16 * 8 * torch.cuda.get_device_properties(0).multi_processor_count // mi.n_cells + 1
    R = _residual(mesh, W, characteristic)
    Rb = _residual(Mesh.concat([mesh] * copies), np.tile(W, (1, copies)), characteristic)
    for k in (0, copies - 1):
        assert np.array_equal(Rb[:, k * mi.n_cells:(k + 1) * mi.n_cells], R)
