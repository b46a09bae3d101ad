"""Mixed solves of small meshes (up to 256 vertices, one row per thread in the
FP32 CG) around a vertex of many neighbours: a local table of 21 entries or more
per row passes 48 KB of shared memory together with the kernel's static arrays.
Positions within 1e-4 of the rest diagonal of the FP64 oracle's (the bound of
the other mixed parity tests).
"""
import numpy as np
import pytest

from emu_inputs import MeshSpec
from oracle import EmuOracle, OracleParams

pytestmark = pytest.mark.gpu


def _hub(spokes):
    """Tets fanned around one inner vertex with ``spokes`` neighbours, three of them pinned."""
    from scipy.spatial import ConvexHull

    k = np.arange(spokes) + 0.5
    z, phi = 1 - 2 * k / spokes, np.pi * (1 + 5 ** 0.5) * k
    rim = np.stack([np.sqrt(1 - z * z) * np.cos(phi), np.sqrt(1 - z * z) * np.sin(phi), z], axis=1)
    tri = ConvexHull(rim).simplices.astype(np.int32)
    rest = np.concatenate([rim, [[0.05, -0.03, 0.02]]]) * 0.01
    tets = np.concatenate([tri, np.full((len(tri), 1), spokes, dtype=np.int32)], axis=1)
    D = (rest[tets[:, :3]] - rest[tets[:, 3:]]).transpose(0, 2, 1)
    flip = np.linalg.det(D) < 0
    tets[flip] = tets[flip][:, [1, 0, 2, 3]]
    m = len(tets)
    fib = np.zeros((m, 3))
    fib[:, 2] = 1.0
    return MeshSpec("hub", rest, tets, np.array([6e5]), np.array([0.45]), np.zeros(m, np.uint8), fib,
                    tri[0].astype(np.int32), np.zeros((1, m)))


@pytest.mark.parametrize("spokes", [16, 23, 24, 40])
def test_mixed_solve_around_a_vertex_of_many_neighbours(spokes):
    import paper_2006_08821_gb300 as emu

    mesh = _hub(spokes)
    r = EmuOracle(mesh, OracleParams(alpha_rel=1.0, weight_mode=0)).solve(0.4, tol=1e-10)
    s = emu.Solver(mesh, emu.Params(precision=emu.PRECISION_MIXED, tol_rel_residual=1e-6))
    s.set_activation(0.4)
    st = s.solve()
    diag = float(np.linalg.norm(mesh.rest_pos.max(0) - mesh.rest_pos.min(0)))
    assert st.status == 0 and np.abs(s.positions() - r.q).max() <= 1e-4 * diag
    s.close()
