"""The FP64 CG with its rows on chip (csrc/emu_pcg64.cu) at the edges of its
launch shapes: fewer than 32 rows, exactly one block, a ragged last block,
several rows groups per block, and matrix rows longer than the 16 entries it
holds in shared memory.

Each case solves Eq. 4 for given deformation gradients through
emu_acap_solve_noalloc and checks the residual of the result in an
independently assembled system. The solve stops at |r| <= 1e-12 |b| of the
recursive residual, b the right-hand side of the solver's system (pinned rows
are identity rows, their b the pinned positions); FP64 rounding of K q adds
about 1e-14 |K| |q|, below 1e-12 |b| on these meshes, so the true residual is
held to 1e-11 |b|.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from emu_inputs import MeshSpec, box_beam
from emu_inputs.meshes import mtu_for_tet_count, single_tet

pytestmark = pytest.mark.gpu


def _hub(spokes=40):
    """Tets fanned around one inner vertex: its matrix row has spokes + 1 entries."""
    from scipy.spatial import ConvexHull

    k = np.arange(spokes) + 0.5
    z, phi = 1 - 2 * k / spokes, np.pi * (1 + 5 ** 0.5) * k
    rim = np.stack([np.sqrt(1 - z * z) * np.cos(phi), np.sqrt(1 - z * z) * np.sin(phi), z], axis=1)
    tri = ConvexHull(rim).simplices.astype(np.int32)
    rest = np.concatenate([rim, [[0.05, -0.03, 0.02]]]) * 0.01
    tets = np.concatenate([tri, np.full((len(tri), 1), spokes, dtype=np.int32)], axis=1)
    m = len(tets)
    fib = np.zeros((m, 3))
    fib[:, 2] = 1.0
    return MeshSpec("hub", rest, tets, np.array([6e5]), np.array([0.45]), np.zeros(m, np.uint8), fib,
                    tri[0].astype(np.int32), np.zeros((1, m)))


MESHES = {
    "tet_4": single_tet,
    "cube_8": lambda: box_beam(1, 1, 1),
    "one_block_32": lambda: box_beam(1, 1, 7),
    "ragged_36": lambda: box_beam(1, 1, 8),
    "hub_41": _hub,
    "beam_425": lambda: box_beam(4, 4, 16),
    "two_groups_6k": lambda: mtu_for_tet_count(30000),
    "five_groups_20k": lambda: mtu_for_tet_count(98400),
    "nine_groups_37k": lambda: mtu_for_tet_count(189600),
}


@pytest.mark.parametrize("name", list(MESHES))
def test_coupling_solve_residual(name):
    import torch

    import paper_2006_08821_gb300 as emu

    mesh = MESHES[name]()
    rng = np.random.default_rng(5)
    F = np.eye(3) + 0.1 * rng.standard_normal((mesh.n_tets, 3, 3))
    s = emu.Solver(mesh, emu.Params(pcg_tol=1e-12))
    Fd = torch.from_numpy(F).cuda()
    q = torch.zeros((mesh.n_verts, 3), dtype=torch.float64, device="cuda")
    assert s.acap_solve_noalloc(Fd.data_ptr(), q.data_ptr()) == 0
    q = q.cpu().numpy()
    s.close()

    Q, T, n, m = mesh.rest_pos, mesh.tets.astype(np.int64), mesh.n_verts, mesh.n_tets
    Dm = (Q[T[:, :3]] - Q[T[:, 3:]]).transpose(0, 2, 1)
    V, Di = np.abs(np.linalg.det(Dm)) / 6.0, np.linalg.inv(Dm)
    N = np.concatenate([Di, -Di.sum(axis=1, keepdims=True)], axis=1)  # (m, 4, 3) shape gradients
    L = V[:, None, None] * np.einsum("mac,mbc->mab", N, N)
    K = sp.csr_matrix((L.ravel(), (np.repeat(T, 4, axis=1).ravel(), np.tile(T, (1, 4)).ravel())), shape=(n, n))
    b = np.zeros((n, 3))
    np.add.at(b, T.ravel(), (V[:, None, None] * np.einsum("mrc,mac->mar", F, N)).reshape(4 * m, 3))
    free = np.ones(n, bool)
    free[mesh.fixed_verts] = False
    np.testing.assert_array_equal(q[~free], Q[~free])
    scale = np.linalg.norm(np.where(free[:, None], b - K @ (Q * ~free[:, None]), Q))
    assert np.linalg.norm((b - K @ q)[free]) <= 1e-11 * scale


# Set-up of the low-rank basis with one, two and four columns per block and on
# the generic kernel (csrc/emu_pcg64.cu, pcg16_columns), with a full and a
# ragged last block of 128 rows, and the FP32 CG of its solves as one block, as
# clusters of two and of the largest eight blocks, and as the first cooperative
# grid above: a handle's first solve reaches its tolerance.
SETUPS = {
    "rows_128": lambda: box_beam(3, 3, 7),
    "rows_132": lambda: box_beam(2, 3, 10),
    "two_blocks_817": lambda: mtu_for_tet_count(3000),
    "eight_blocks_3993": lambda: box_beam(10, 10, 32),
    "nine_blocks_4114": lambda: box_beam(10, 10, 33),
    "two_columns_3k": lambda: mtu_for_tet_count(12000),
    "four_columns_9k": lambda: mtu_for_tet_count(40000),
    "generic_13k": lambda: mtu_for_tet_count(60000),
}


@pytest.mark.parametrize("name", list(SETUPS))
def test_first_solve_after_setup(name):
    import paper_2006_08821_gb300 as emu

    mesh = SETUPS[name]()
    s = emu.Solver(mesh, emu.Params(precision=emu.PRECISION_MIXED))
    s.set_activation(0.4)
    st = s.solve()
    assert st.status == 0 and st.rel_residual <= 1e-6
    s.close()
