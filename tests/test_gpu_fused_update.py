"""FP32C Euler kernels of small meshes against those of large ones: the fused update, faces split over threads."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1712_08317_gb300.api import Mesh, Solver  # noqa: E402


# walls, inflow and outflow faces; cell counts that leave the last warp of four-lane cells partly filled
@pytest.mark.parametrize("kind,n", [("quad", 7), ("tri", 5), ("mixed", 13)])
def test_mesh_alone_and_in_a_large_batch_give_the_same_bits(kind, n):
    """Alone the mesh takes the fused kernel; with copies to more than 1,024 lanes for every SM the
    separate ones.  Both compute a flux by the same rounded operations, so results are equal."""
    sh = S.moving_shock(2.5, 0.3, 0.0, 60.0)
    mi = S.tube_mesh(3 * n, n, (3.0, 1.0), kind, delta=0.1, seed=9, walls=(2,), wall_from=(0, 0, 0.5, 0),
                     inflow=(0, 2, 3))
    prm = dict(eqn="euler", precision="fp32c", inflow_a=sh["post"], inflow_b=sh["pre"], inflow_line=sh["line"])
    W = S.cell_average(mi, sh["f"])
    mesh = Mesh.from_input(mi)
    one = Solver(mesh, **prm)
    U, Ul = one.to_device(W)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    copies = 1024 * sms // (4 * mi.n_cells) + 1
    big = Solver(Mesh.concat([mesh] * copies), **prm)
    V, Vl = big.to_device(np.tile(W, (1, copies)))
    R, Rb = one.to_host(one.residual(U, Ul)), big.to_host(big.residual(V, Vl))
    dt = float(one.max_dt(U, Ul, 0.4)[0])
    for _ in range(3):
        one.step(U, Ul, dt)
        big.step(V, Vl, dt)
    torch.cuda.synchronize()
    a, b = one.to_host(U, Ul), big.to_host(V, Vl)
    for k in (0, copies - 1):
        cells = slice(k * mi.n_cells, (k + 1) * mi.n_cells)
        assert np.array_equal(Rb[:, cells], R)
        assert np.array_equal(b[:, cells], a)


# characteristic variables on a mesh whose blocks have a set of threads for every face (few tiles for every
# SM), with indicators inside and outside the FP32 range; the last tile of a type is partly filled
@pytest.mark.parametrize("flow", ["wave", "ramp"])
@pytest.mark.parametrize("kind,n", [("quad", 9), ("tri", 5), ("mixed", 13)])
def test_faces_split_over_threads_give_the_same_bits(kind, n, flow):
    """In a large batch a thread walks all faces of its cell; the arithmetic of a Gauss point is the same."""
    def ramp(x, y):
        rho = 1.0 + 1e7 * (x + 0.3 * y)
        one = np.ones_like(rho)
        return S.euler_prim_to_cons(rho, one, 0.5 * one, rho, 1.4)

    mi = S.mesh_for_config(3, n=n, seed=7, kind=kind)
    mi.walls = (0, 3)
    mesh = Mesh.from_input(mi)
    W = S.cell_average(mi, S.density_wave if flow == "wave" else ramp)
    prm = dict(eqn="euler", precision="fp32c", characteristic=True)
    one = Solver(mesh, **prm)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    copies = 16 * 8 * sms // mi.n_cells + 1  # more than eight tiles of 16 cells for every SM
    big = Solver(Mesh.concat([mesh] * copies), **prm)
    U, Ul = one.to_device(W)
    V, Vl = big.to_device(np.tile(W, (1, copies)))
    R, Rb = one.to_host(one.residual(U, Ul)), big.to_host(big.residual(V, Vl))
    for k in (0, copies - 1):
        assert np.array_equal(Rb[:, k * mi.n_cells:(k + 1) * mi.n_cells], R, equal_nan=True)
