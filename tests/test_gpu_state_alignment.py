"""States and time steps that start at any element of a buffer."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

import ctypes  # noqa: E402

from paper_1712_08317_gb300 import _capi  # noqa: E402
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


# The steps of the instances are copied, not read in place, where they are no doubles of this device's memory
@pytest.mark.parametrize("precision", ["fp64", "fp32c"])
def test_time_steps_that_start_at_any_byte(precision):
    mi = S.mesh_for_config(2, n=9, seed=3, kind="mixed")
    mesh = Mesh.from_input(mi)
    sol = Solver(Mesh.concat([mesh] * 3), eqn="euler", precision=precision)
    W = np.tile(S.cell_average(mi, S.density_wave), (1, 3))
    dts = np.array([1.0, 0.5, 0.25]) * sol.max_dt(*sol.to_device(W), 0.4)[0]
    out = []
    for first in (0, 4, 1):
        raw = torch.zeros(32, dtype=torch.uint8, device="cuda")
        raw[first:first + 24] = torch.from_numpy(dts.view(np.uint8).copy()).cuda()
        U, Ul = sol.to_device(W)
        p = [None if t is None else ctypes.c_void_p(t.data_ptr()) for t in (U, Ul)]
        _capi.check(_capi.load().weno_step_instances(sol._h, *p, ctypes.c_void_p(raw.data_ptr() + first),
                                                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
        out.append(sol.to_host(U, Ul))
    assert np.array_equal(out[1], out[0]) and np.array_equal(out[2], out[0])
    assert not np.array_equal(out[0], W)
