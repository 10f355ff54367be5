"""The pose-group gradient kernel at the ends of its fetch batches: ligands
of 1 to 14 atoms (a batch is 3 or 4 records per lane), every group width,
poses with atoms outside the box and on its faces, against the oracle."""
import numpy as np
import pytest
import torch

import gen
import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [4, 9, 17])   # 4, 2 and 1 lanes per pose
def test_gradient_batches_and_box_faces(oracle_lib, P):
    import paper_2303_06150_gb300 as lg
    from gen.library import from_ligands
    parts = [gen.make_library(dict(kind="uniform", n_ligands=1, n_atoms=(N, N), n_rot=(3, 3), n_types=4, seed=N))
             for N in range(1, 15)]
    lib = from_ligands([p.ligand(0) for p in parts])
    grid = gen.make_grid(gen.WORKLOADS["small32"]["grid"])
    box = grid.spacing * (grid.dims[0] - 1)
    rng = np.random.default_rng(P)
    blocks = []
    for l in range(lib.n_ligands):
        q = rng.normal(size=(P, 4))
        t = grid.center + rng.uniform(-2, 2, (P, 3))
        t[0] = [box, 9.0, 9.0]   # half of the ligand outside; the one-atom ligand exactly on the upper face
        t[1] = [-50.0, 0.0, 0.0]
        t[2] = [0.0, 9.0, -0.0]
        blocks.append(np.concatenate([t, q / np.linalg.norm(q, axis=1, keepdims=True),
                                      rng.uniform(-3, 3, (P, lib.n_rot[l]))], 1).astype(np.float32))
    L = lg.Ligands.from_arrays(lib, "cuda")
    G = lg.PocketGrid.from_array(grid.values, grid.origin, grid.spacing, "cuda")
    flat = torch.from_numpy(np.concatenate([b.ravel() for b in blocks])).cuda()
    s, g = (x.cpu().numpy() for x in lg.pose_grad(L, G, flat, P))
    off = lg.pose_offsets(lib.rot_off, P)
    og = oracle_lib.OGrid.from_grid(grid)
    for l in range(lib.n_ligands):
        lig = oracle_lib.OLigand.from_library(lib, l)
        got = g[off[l]:off[l + 1]].reshape(P, -1)
        for p in range(P):
            pose = blocks[l][p].astype(np.float64)
            S, D, _, Gs = oracle_lib.score_pose(lig, og, pose, 5.0, sensitivity=True)
            if p > 2 or p == 1 or lib.n_atoms[l] == 1:   # poses 0, 2: an atom may round across the face
                assert abs(s[l, p] - S) <= parity.score_tol(D, Gs), (l, p, s[l, p], S)
            if p == 1:
                assert not got[p].any()   # everything outside: no gradient
            elif p > 2:
                u = oracle_lib.pose_coords(lig, pose) / grid.spacing   # origin 0
                if np.abs(u - np.round(u)).min() < 1e-4:
                    continue   # an atom at a cell face: FP32 may take the other cell's slope
                ref = oracle_lib.pose_grad(lig, og, pose)[-1]
                # the measured 8.2e-5 of the gradient's norm against the oracle, with a margin of 3
                assert np.abs(got[p] - ref).max() <= 2.5e-4 * max(np.abs(ref).max(), 1e-3), (l, p)
