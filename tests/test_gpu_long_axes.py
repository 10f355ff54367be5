"""Scoring, gradients and refinement on a grid whose axis has more than 2^23
cells, where the pose-per-lane samplers' floor by addition ends: one-atom
ligands on nodes on both sides of cell 2^23, every entry point and pose count
against the node values themselves."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

EDGE = 1 << 23


def _case(axis, P):
    import paper_2303_06150_gb300 as lg
    n = EDGE + 3001
    node = ((np.arange(n, dtype=np.int64) * 37) % 11).astype(np.float32)
    shape = [1, 1, 1, 1]
    shape[2 - axis] = n   # values are [z][y][x][c]
    dims = [2, 2, 2, 1]
    dims[2 - axis] = n
    values = np.ascontiguousarray(np.broadcast_to(node.reshape(shape), dims))
    lib = type("Lib", (), dict(atom_off=np.arange(4), xyz=np.zeros((3, 3)), type=np.zeros(3), bonds=np.zeros((0, 2)),
                               rot_off=np.zeros(4), rot_edge=np.zeros(0)))()
    cell = np.random.default_rng(axis).integers(EDGE - 1500, EDGE + 2990, size=3 * P)
    cell[:4] = [EDGE - 1, EDGE, EDGE + 1, EDGE + 2999]
    poses = np.zeros((3 * P, 7), dtype=np.float32)
    poses[:, :3] = 0.25
    poses[:, axis] = cell
    poses[:, 3] = 1
    poses = torch.from_numpy(poses.ravel()).cuda()
    return (lg, lg.Ligands.from_arrays(lib, "cuda"), lg.PocketGrid.from_array(values, (0, 0, 0), 1.0, "cuda"), poses,
            node, cell)


@pytest.mark.parametrize("axis,P", [(0, 16), (0, 3), (1, 17), (2, 33), (2, 16)])
def test_values_and_gradients_past_the_edge(axis, P):
    lg, L, G, poses, node, cell = _case(axis, P)
    want = -node[cell]   # positions on nodes: every weight is 0 or 1, 0.25 of equal values exact
    one_shot = lg.score_poses(L, G, poses, P).cpu().numpy().ravel()
    prepared = lg.prepare_scoring(L, G).score(poses, P).cpu().numpy().ravel()
    s, g = lg.pose_grad(L, G, poses, P)
    assert np.array_equal(one_shot, want)
    assert np.array_equal(prepared, want)
    assert np.array_equal(s.cpu().numpy().ravel(), want)
    slope = g.cpu().numpy().reshape(-1, 7)[:, axis]
    assert np.array_equal(slope, node[cell] - node[cell + 1])


def test_refinement_keeps_the_best_past_the_edge():
    P = 16
    lg, L, G, poses, node, cell = _case(2, P)
    start = lg.score_poses(L, G, poses, P)
    out, s, _ = lg.refine_poses(L, G, poses, P, steps=3, step_t=1.0)
    again = lg.score_poses(L, G, out, P)
    assert bool((s >= start).all())
    assert torch.allclose(s, again, rtol=0, atol=2e-5)   # values to 10, at most 16 roundings of 6e-8 each
