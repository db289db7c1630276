"""Results of a mesh have the same bits in whichever instance of a kernel its cells are computed: alone, and in
batches that cross the sizes at which the instance changes."""
import numpy as np
import pytest

import synthetic as S
from oracle import OracleMesh, OracleSolver, Params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1712_08317_gb300.api import Mesh, Solver  # noqa: E402

SMS = torch.cuda.get_device_properties(0).multi_processor_count


def _flow(x, y):
    rho = 1.0 + 0.2 * np.sin(2 * np.pi * x) * np.cos(np.pi * y)
    one = np.ones_like(rho)
    return S.euler_prim_to_cons(rho, 0.5 * one, -0.4 * one, 1.0 + 0.1 * np.cos(2 * np.pi * y), 1.4)


def _meshes(n):
    """A mesh of quads, one of triangles and a mixed one, with reflective walls."""
    out = []
    for kind, m in (("quad", n), ("tri", n - 2), ("mixed", n - 1)):
        mi = S.mesh_for_config(3, n=m, seed=11, kind=kind)
        mi.walls = (0, 3)
        out.append((mi, Mesh.from_input(mi), S.cell_average(mi, _flow)))
    return out


def _residual(mesh, W, prm):
    sol = Solver(mesh, eqn="euler", **prm)
    U, Ul = sol.to_device(W)
    R = sol.to_host(sol.residual(U, Ul))
    sol.check()
    return R


def _compare(parts, copies, prm):
    alone = [_residual(mesh, W, prm) for _, mesh, W in parts]
    big = _residual(Mesh.concat([m for _, m, _ in parts] * copies), np.concatenate([W for _, _, W in parts] * copies, axis=1),
                    prm)
    sizes = [mi.n_cells for mi, _, _ in parts]
    for k in (0, copies - 1):
        at = k * sum(sizes)
        for R, n in zip(alone, sizes):
            assert np.array_equal(big[:, at:at + n], R)
            at += n


# both types in one launch (up to 16 rounds of eight 16-cell tiles an SM), and each in its own (above)
@pytest.mark.parametrize("characteristic", [False, True])
@pytest.mark.parametrize("rounds", [2, 16.5])
def test_fp32c_types_alone_in_one_launch_and_in_two(rounds, characteristic):
    parts = _meshes(47)
    copies = int(rounds * 8 * 16 * SMS / sum(mi.n_cells for mi, _, _ in parts)) + 1
    _compare(parts, copies, dict(precision="fp32c", characteristic=characteristic))


# 8 and 32 (cell, variable) columns a block; in characteristic variables one and two points of a face a thread
@pytest.mark.parametrize("linear", [False, True])
@pytest.mark.parametrize("characteristic", [False, True])
def test_fp64_tiles_of_a_small_and_of_a_large_mesh(characteristic, linear):
    parts = _meshes(15)
    quads, tris = (sum(int((np.diff(mi.cell_ptr) == k).sum()) for mi, _, _ in parts) for k in (4, 3))
    copies = int(max(512 * SMS / 16 / quads, 512 * SMS / 12 / tris)) + 2
    _compare(parts, copies, dict(precision="fp64", characteristic=characteristic, linear=linear))


# The FP64 characteristic kernel with both points of a face in a thread (from 32 cell faces an SM and quarter on:
# 4,864 quads, 6,486 triangles), last tile partly filled; the oracle's bound is that of the FP64 parity tests
@pytest.mark.parametrize("kind", ["quad", "tri"])
@pytest.mark.parametrize("walls", [(), (0, 3)])
def test_fp64_characteristic_on_a_large_mesh_matches_the_oracle(kind, walls):
    cells = 512 * SMS / (16 if kind == "quad" else 12)
    n = int(np.sqrt(1.05 * cells / (1 if kind == "quad" else 2))) | 1
    mi = S.mesh_for_config(3, n=n, seed=5, kind=kind)
    mi.walls = walls
    W = S.cell_average(mi, _flow)
    assert mi.n_cells > cells and mi.n_cells % 8
    ref = OracleSolver(OracleMesh.from_input(mi), Params(characteristic=True)).residual(W)
    R = _residual(Mesh.from_input(mi), W, dict(precision="fp64", characteristic=True))
    scale = np.abs(ref).max(axis=1, keepdims=True)
    assert float((np.abs(R - ref) / scale).max()) < 1e-11
