"""The passes that run alone are those of the residual, kernel by kernel."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from captured import kernels  # noqa: E402
from paper_1712_08317_gb300 import _capi  # noqa: E402
from paper_1712_08317_gb300.api import Mesh, Solver  # noqa: E402

# small meshes, whose fluxes and gather may be one kernel, and one above that size (4 lanes a cell, 1,024 an SM)
SMALL, LARGE = 13, int(np.sqrt(1.1 * 256 * torch.cuda.get_device_properties(0).multi_processor_count / 1.3))


def _solver(n, kind, **prm):
    mi = S.mesh_for_config(2, n=n, seed=3, kind=kind)
    sol = Solver(Mesh.from_input(mi), **prm)
    W = S.cell_average(mi, S.density_wave if prm.get("eqn", "euler") == "euler" else S.scalar_wave)
    return sol, sol.to_device(W), W


@pytest.mark.parametrize("n,kind,prm", [
    (SMALL, "mixed", dict(precision="fp32c")), (SMALL, "quad", dict(precision="fp32c")),
    (SMALL, "tri", dict(precision="fp32c", characteristic=True)), (LARGE, "mixed", dict(precision="fp32c")),
    (SMALL, "mixed", dict(precision="fp64")), (SMALL, "tri", dict(precision="fp64", characteristic=True)),
    (SMALL, "mixed", dict(eqn="scalar", precision="fp32c")), (SMALL, "quad", dict(eqn="scalar", precision="fp64"))])
def test_passes_launch_the_kernels_of_the_residual(n, kind, prm):
    sol, (U, Ul), _ = _solver(n, kind, **prm)
    R = torch.empty_like(U)
    sol.residual(U, Ul, R)  # what the first call sets up
    whole = kernels(lambda st: sol.residual(U, Ul, R, stream=st))
    parts = [kernels(lambda st: sol.run_pass(p, U, Ul, stream=st)) for p in (1, 2, 3)]
    assert whole and parts[0] + parts[1] + parts[2] == whole


def test_passes_of_a_small_mesh_report_its_states():
    sol, _, W = _solver(SMALL, "mixed", precision="fp32c")
    W = W.copy()
    W[0, 5] = -0.1
    U, Ul = sol.to_device(W)
    for p in (1, 2, 3):
        sol.run_pass(p, U, Ul)
    with pytest.raises(_capi.WenoError) as e:
        sol.check()
    assert e.value.code == _capi.WENO_ENONPHYS
