"""Autotune and the launch shapes it reports, over the forms a residual takes."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from captured import kernels  # noqa: E402
from paper_1712_08317_gb300.api import Mesh, Solver  # noqa: E402

SMS = torch.cuda.get_device_properties(0).multi_processor_count
# below and above the size at which fluxes and gather are kernels of their own (four lanes a cell, 1,024 an SM)
SMALL, LARGE = 13, int(np.sqrt(1.1 * 256 * SMS / 1.3))


# One launch for both cell types with and without the fused update; faces split over threads; types alone; FP64
@pytest.mark.parametrize("n,kind,prm", [
    (SMALL, "mixed", dict(precision="fp32c")), (LARGE, "mixed", dict(precision="fp32c")),
    (LARGE, "tri", dict(precision="fp32c")), (SMALL, "quad", dict(precision="fp32c", characteristic=True)),
    (SMALL, "tri", dict(precision="fp32c", characteristic=True)),
    (LARGE, "mixed", dict(precision="fp32c", characteristic=True)), (SMALL, "tri", dict(precision="fp64")),
    (SMALL, "mixed", dict(precision="fp64", characteristic=True)), (SMALL, "mixed", dict(eqn="scalar", precision="fp32c"))])
def test_shapes_are_those_of_the_launches(n, kind, prm):
    mi = S.mesh_for_config(2, n=n, seed=3, kind=kind)
    sol = Solver(Mesh.from_input(mi), **prm)
    U, Ul = sol.to_device(S.cell_average(mi, S.scalar_wave if prm.get("eqn") == "scalar" else S.density_wave))
    dt = float(sol.max_dt(U, Ul, 0.4)[0])

    def shapes():
        run = kernels(lambda st: sol.residual(U, Ul, R, stream=st))
        cfg = sol.launch_config().tolist()
        # first the quads' reconstruction (or the only one); last the gather, before it the fluxes, or one kernel for both
        for (_, grid, block), (b, g) in ((run[0], cfg[0:2]), (run[-1], cfg[4:6])):
            assert block == b and (g == 0 or grid <= g)
        if any("k_update" in name for name, _, _ in run):
            assert cfg[2:4] == cfg[4:6]
        else:
            assert run[-2][2] == cfg[2] and (cfg[3] == 0 or run[-2][1] <= cfg[3])

    R = sol.residual(U, Ul).clone()
    states = [[t.clone() if t is not None else None for t in (U, Ul)] for _ in range(2)]
    sol.step(*states[0], dt)
    R0 = R.clone()
    shapes()
    sol.autotune(U, Ul)
    shapes()
    sol.step(*states[1], dt)
    assert torch.equal(sol.residual(U, Ul), R0)
    for a, b in zip(*states):
        assert a is None or torch.equal(a, b)
    sol.check()
