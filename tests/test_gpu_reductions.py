"""Time step and integrals: chunks, instances, widening of FP32 states, cells without a step."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle import OracleMesh, OracleSolver, Params  # noqa: E402
from paper_1712_08317_gb300.api import Mesh, Solver  # noqa: E402


# one partly filled chunk; several of each type; more than 256 cells a chunk (in the batch)
@pytest.mark.parametrize("precision", ["fp64", "fp32c"])
@pytest.mark.parametrize("kind,n", [("quad", 5), ("tri", 12), ("mixed", 31)])
def test_instances_equal_the_mesh_alone_and_the_oracle(precision, kind, n):
    mi = S.mesh_for_config(2, n=n, seed=3, kind=kind)
    W = S.cell_average(mi, S.density_wave)
    mesh = Mesh.from_input(mi)
    one = Solver(mesh, eqn="euler", precision=precision)
    copies = 256 * 8 * torch.cuda.get_device_properties(0).multi_processor_count // mi.n_cells + 2
    big = Solver(Mesh.concat([mesh] * copies), eqn="euler", precision=precision)
    U, Ul = one.to_device(W)
    V, Vl = big.to_device(np.tile(W, (1, copies)))
    dt, sums = one.max_dt(U, Ul, 0.5)[0], one.conservation(U, Ul)[0]
    orc = OracleSolver(OracleMesh.from_input(mi), Params())
    assert dt == pytest.approx(orc.max_dt(W, 0.5), rel=1e-12)
    # n_cells roundings of 2^-53 at most in a sum of n_cells terms
    tol = 2 * mi.n_cells * 2.0 ** -53 * orc.conservation(np.abs(W)).max() + 1e-14
    assert np.abs(sums - orc.conservation(W)).max() <= tol
    assert np.array_equal(big.max_dt(V, Vl, 0.5), np.full(copies, dt))  # a minimum has no order
    assert np.abs(big.conservation(V, Vl) - sums).max() <= tol


def test_fp32_states_are_widened_exactly():
    """Signs, zeros, subnormals and the ends of the range; one cell at a time carries the value."""
    mi = S.mesh_for_config(1, n=6, seed=1)
    sol = Solver(Mesh.from_input(mi), eqn="scalar", precision="fp32c")
    ones = torch.zeros(mi.n_cells, 1, dtype=torch.float32, device="cuda")
    ones[7] = 1.0
    zero = torch.zeros_like(ones)
    area = sol.conservation(ones, zero)[0, 0]
    for x in (1.0, -1.5, 0.1, 2.0 ** -126, -2.0 ** -127, 2.0 ** -149, 3.4028234663852886e38, -0.0):
        x = float(np.float32(x))
        assert sol.conservation(ones * x, zero)[0, 0] == area * x
        assert sol.conservation(zero, ones * x)[0, 0] == area * x
    for x in (float("inf"), float("nan")):
        assert np.array_equal(sol.conservation(torch.where(ones > 0, x, 0.0), zero)[0, 0], x, equal_nan=True)


@pytest.mark.parametrize("precision", ["fp64", "fp32c"])
def test_cells_without_a_step_are_left_out(precision):
    mi = S.mesh_for_config(2, n=9, seed=4, kind="mixed")
    W = S.cell_average(mi, S.density_wave)
    sol = Solver(Mesh.from_input(mi), eqn="euler", precision=precision)
    dt = sol.max_dt(*sol.to_device(W), 0.5)[0]
    got = []
    for v, c, x in ((3, 2, -1.0), (3, 70, -1.0), (0, 40, float("nan"))):  # sound speed of a negative pressure; NaN
        B = W.copy()
        B[v, c] = x
        got.append(sol.max_dt(*sol.to_device(B), 0.5)[0])
    assert min(got) == dt and np.all(np.isfinite(got))  # at most one of the three cells set the step
