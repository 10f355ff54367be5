"""The FP64 re-score's ranking on both sides of its 32-pose path, and its
cell arithmetic on box faces and on axes longer than its integer floor takes,
against FP64 values of the returned poses."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 31, 32, 33, 70])
def test_ranks_and_scores(small32, oracle_lib, K):
    import paper_2303_06150_gb300 as lg
    w, lib, grid = small32
    lib = lib.subset(range(0, 32, 6))
    v32 = grid.values.astype(np.float32)
    og = oracle_lib.OGrid(v32.astype(np.float64), grid.origin, grid.spacing)
    L = lg.Ligands.from_arrays(lib, "cuda")
    G = lg.PocketGrid.from_array(v32, grid.origin, grid.spacing, "cuda")
    r = lg.dock_batch(L, G, restarts=70, torsion_step_deg=24, passes=1, top_k=K, seed=3, rescore_fp64=True,
                      top_restart=True)
    s64, top, poses = r.scores_f64.cpu().numpy(), r.top_restart.cpu().numpy(), r.poses.cpu().numpy().astype(np.float64)
    np.testing.assert_array_equal(r.scores.cpu().numpy(), s64.astype(np.float32))
    off = lg.pose_offsets(lib.rot_off, K)
    for l in range(lib.n_ligands):
        assert len(set(top[l])) == K
        assert all(a > b or (a == b and i < j) for a, b, i, j in zip(s64[l], s64[l][1:], top[l], top[l][1:]))
        xyz = lib.ligand(l)["xyz"].astype(np.float32).astype(np.float64)
        g = lib.ligand(l)
        lig = oracle_lib.OLigand(xyz, g["type"], g["bonds"], g["rot_edge"])
        for k in range(K):
            S, D, _ = oracle_lib.score_pose(lig, og, poses[off[l]:off[l + 1]].reshape(K, -1)[k], 5.0)
            assert abs(s64[l, k] - S) <= 1e-9 * D


# values of all sizes: zeros, subnormals and large ones take the other branches of the widening
@pytest.mark.parametrize("shape", [(2, 2, 2), (5, 3, 2 ** 20), (3, 2, 2 ** 20 + 1)])
def test_cells_and_node_values(shape):
    import torch

    import paper_2303_06150_gb300 as lg
    nx, ny, nz = shape
    rng = np.random.default_rng(nz % 1000)
    v = rng.normal(size=(nz, ny, nx, 1)).astype(np.float32)
    v[rng.random(v.shape) < 0.2] = 0.0
    v[rng.random(v.shape) < 0.2] *= np.float32(1e-41)
    v[rng.random(v.shape) < 0.1] *= np.float32(1e30)
    z = torch.zeros(2, dtype=torch.int32)
    L = lg.Ligands(torch.tensor([0, 1], dtype=torch.int32).cuda(), torch.zeros((1, 3)).cuda(),
                   torch.zeros(1, dtype=torch.uint8).cuda(), torch.zeros((0, 2), dtype=torch.int32).cuda(), z.cuda(),
                   z[:0].cuda())
    G = lg.PocketGrid.from_array(v, (0.0, 0.0, 0.0), 1.0, "cuda")
    R = 200
    r = lg.dock_batch(L, G, restarts=R, torsion_step_deg=30, passes=0, top_k=R, seed=5, n_rigid=1,
                      jitter=0.75 * max(nx, ny), rescore_fp64=True)
    u = r.poses.cpu().numpy().reshape(R, 7)[:, :3].astype(np.float64)   # origin 0, spacing 1: exact
    got = r.scores_f64.cpu().numpy()[0]
    top = np.array([nx, ny, nz]) - 1
    inside = ((u >= 0) & (u <= top)).all(1)
    assert inside.any() and not inside.all()
    i = np.minimum(np.floor(np.where(inside[:, None], u, 0)).astype(int), top - 1)
    f = np.where(inside[:, None], u, 0) - i
    e = big = 0.0
    for k in range(8):
        d = np.array([k & 1, k >> 1 & 1, k >> 2])
        node = v[i[:, 2] + d[2], i[:, 1] + d[1], i[:, 0] + d[0], 0].astype(np.float64)
        e = e + np.where(d, f, 1 - f).prod(1) * node
        big = np.maximum(big, np.abs(node))
    want = np.where(inside, -e, -5.0)
    assert (np.abs(got - want) <= 32 * 2.0 ** -53 * (big + 5.0)).all()
