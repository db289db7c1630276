"""The benchmark's count of kernel launches a step, against the launches themselves."""
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from bench import step_launches  # noqa: E402
from captured import kernels  # noqa: E402
from paper_1712_08317_gb300.api import Mesh, Solver  # noqa: E402

SMS = torch.cuda.get_device_properties(0).multi_processor_count


# the sizes on both sides of the fused update (256 cells an SM) and of one launch for both cell types (2,048)
@pytest.mark.parametrize("kind,cells_per_sm", [("mixed", 200), ("mixed", 300), ("mixed", 1900), ("mixed", 2200),
                                               ("tri", 2200)])
def test_launches_of_a_step(kind, cells_per_sm):
    mi = S.mesh_for_config(2, n=23, seed=3, kind=kind)
    mesh = Mesh.from_input(mi)
    sol = Solver(Mesh.concat([mesh] * round(cells_per_sm * SMS / mi.n_cells)), precision="fp32c")
    U = torch.ones(sol.n_cells, 4, device="cuda")
    Ul, R = torch.zeros_like(U), torch.empty_like(U)
    stage = kernels(lambda st: sol.residual(U, Ul, R, stream=st))
    info = sol.mesh.info
    # a step: three stages between the time steps' kernel and the times'
    assert step_launches(int(info.n_quads), int(info.n_tris), SMS) == 2 + 3 * len(stage)
