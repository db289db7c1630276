"""States and time steps that start at any element of a buffer."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1712_08317_gb300.api import Mesh, Solver  # noqa: E402


def _at(t, first):
    """t's values in a buffer of their own, from its element `first` on."""
    if t is None:
        return None
    out = torch.zeros(t.numel() + first, dtype=t.dtype, device=t.device)[first:].view(t.shape)
    out.copy_(t)
    assert out.data_ptr() % 16 == first * t.element_size() % 16
    return out


# Time step and integrals read one element at a time where a cell's values don't start on a 16-byte boundary
@pytest.mark.parametrize("eqn,precision,first", [("euler", "fp32c", (1, 0)), ("euler", "fp32c", (0, 2)),
                                                 ("euler", "fp32c", (3, 3)), ("euler", "fp64", (1, 0)),
                                                 ("scalar", "fp32c", (1, 3)), ("scalar", "fp64", (1, 0))])
def test_reductions_of_a_state_inside_a_buffer(eqn, precision, first):
    mi = S.mesh_for_config(2, n=13, seed=3, kind="mixed")
    W = S.cell_average(mi, S.density_wave if eqn == "euler" else S.scalar_wave)
    sol = Solver(Mesh.from_input(mi), eqn=eqn, precision=precision)
    U, Ul = sol.to_device(W)
    V, Vl = _at(U, first[0]), _at(Ul, first[1])
    assert np.array_equal(sol.max_dt(V, Vl, 0.4), sol.max_dt(U, Ul, 0.4))
    assert np.array_equal(sol.conservation(V, Vl), sol.conservation(U, Ul))
