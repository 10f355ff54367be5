"""The packer at the edges of its 32-atom words and on deep and flat trees:
masks, axes, touch masks and status against the oracle's fragments, and the
forward-kinematics table through the pose-per-lane scores and gradients."""
import numpy as np
import pytest

import gen
import oracle
from gen.library import from_ligands

pytestmark = pytest.mark.gpu


def _tree(rng, N, kind, n_rot):
    """A ligand of N atoms: a chain, a star or a random tree, its bond rows shuffled."""
    i = np.arange(1, N)
    par = {"chain": i - 1, "star": np.zeros(N - 1, int), "random": (rng.random(N - 1) * i).astype(int)}[kind]
    label = rng.permutation(N)
    rows = np.stack([label[par], label[i]], 1).reshape(-1, 2)
    flip = rng.random(len(rows)) < 0.5
    rows[flip] = rows[flip][:, ::-1]
    rows = rows[rng.permutation(len(rows))]
    rot = rng.permutation(N - 1)[:n_rot]
    return dict(xyz=rng.normal(size=(N, 3)) * 3, type=rng.integers(0, 4, N), bonds=rows, rot_edge=rot)


def _library(kind, sizes, seed):
    rng = np.random.default_rng(seed)
    return from_ligands([_tree(rng, N, kind, min(N - 1, n)) for N, n in sizes])


SIZES = {1: [(1, 0), (2, 1), (31, 5), (32, 31)],
         2: [(33, 32), (5, 2), (63, 7), (64, 32)],
         4: [(65, 3), (100, 24), (127, 32), (128, 12)],
         8: [(129, 32), (3, 2), (255, 16), (256, 32), (256, 0)]}


@pytest.mark.parametrize("words", SIZES)
@pytest.mark.parametrize("kind", ["chain", "star", "random"])
def test_packer_and_table_at_word_edges(kind, words):
    import torch

    import paper_2303_06150_gb300 as lg
    lib = _library(kind, SIZES[words], 100 * words + len(kind))
    L = lg.Ligands.from_arrays(lib, "cuda")
    bits, axis, _, status = (t.cpu().numpy() for t in lg.pack_ligands(L, 4))
    touch = lg.pack_touch(L, 4).cpu().numpy()
    assert not status.any()
    grid = gen.make_grid(gen.WORKLOADS["small32"]["grid"])
    G = lg.PocketGrid.from_array(grid.values, grid.origin, grid.spacing, "cuda")
    og = oracle.OGrid.from_grid(grid)
    rng = np.random.default_rng(5)
    P = 16
    poses = []
    for l in range(lib.n_ligands):
        N, n, r0 = lib.n_atoms[l], lib.n_rot[l], lib.rot_off[l]
        _, frag, ax = oracle.fragments(oracle.OLigand.from_library(lib, l))
        got = (bits[r0:r0 + n].view(np.uint32)[:, :, None] >> np.arange(32) & 1).reshape(n, 256).astype(bool)
        frag = np.asarray(frag, bool).reshape(n, N)
        np.testing.assert_array_equal(got[:, :N], frag)
        assert not got[:, N:].any()
        np.testing.assert_array_equal(axis[r0:r0 + n], np.asarray(ax).reshape(n, 2))
        for b2 in range(n):
            moved = frag[b2].copy()
            moved[ax[b2][1]] = False
            want = sum(1 << b for b in range(n) if b == b2 or (moved & (frag[b] | (np.arange(N) == ax[b][0]))).any())
            assert touch[r0 + b2] == want
        q = rng.normal(size=(P, 4))
        poses.append(np.concatenate([grid.center + rng.uniform(-1, 1, (P, 3)),
                                     q / np.linalg.norm(q, axis=1, keepdims=True),
                                     rng.uniform(-3, 3, (P, n))], 1).astype(np.float32))
    flat = torch.from_numpy(np.concatenate([p.ravel() for p in poses])).cuda()
    sc = lg.score_poses(L, G, flat, P).cpu().numpy()
    gsc = lg.pose_grad(L, G, flat, P)[0].cpu().numpy()
    eps = 2.0 ** -24
    for l in range(lib.n_ligands):
        lig = oracle.OLigand.from_library(lib, l)
        # FP32 rounding of a position grows along the chain of transforms: 24 units
        # (measured on libraries of at most 8 depths) per 8 depths, 32 bonds at most
        ulps = 24 * (1 + lib.n_rot[l] / 8)
        for p in range(P):
            S, D, _, Gs = oracle.score_pose(lig, og, poses[l][p].astype(np.float64), 5.0, sensitivity=True)
            tol = 1e-5 * D + ulps * eps * Gs
            assert abs(sc[l, p] - S) <= tol and abs(gsc[l, p] - S) <= tol, (l, p, sc[l, p], gsc[l, p], S, tol)


def test_packer_rejects_graphs_that_are_not_trees():
    import paper_2303_06150_gb300 as lg
    rng = np.random.default_rng(9)
    good = _tree(rng, 40, "random", 4)
    cycle = dict(good, bonds=good["bonds"].copy())
    cycle["bonds"][7] = cycle["bonds"][3][::-1]          # an edge twice: some atom is not reached
    loop = dict(good, bonds=good["bonds"].copy())
    loop["bonds"][0] = [5, 5]
    lib = from_ligands([good, cycle, loop, good])
    bits, axis, _, status = (t.cpu().numpy() for t in lg.pack_ligands(lg.Ligands.from_arrays(lib, "cuda"), 4))
    assert list(status) == [0, -6, -6, 0]
    assert not bits[4:12].any() and (axis[4:12] == -1).all()
