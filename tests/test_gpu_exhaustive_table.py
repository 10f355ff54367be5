"""The exhaustive search's energy table at its limits, against the oracle's
brute force: nested bonds whose table does not fit (rebuilt per combination),
four bonds, no bonds, one increment, few rotations, empty moving lists."""
import numpy as np
import pytest

import gen
import parity
from gen.library import from_ligands

pytestmark = pytest.mark.gpu


def _ligand(rng, N, kind, bonds):
    i = np.arange(1, N)
    par = {"chain": i - 1, "star": np.zeros(N - 1, int), "random": (rng.random(N - 1) * i).astype(int)}[kind]
    xyz = np.zeros((N, 3))
    for k in i:
        d = rng.normal(size=3)
        xyz[k] = xyz[par[k - 1]] + 1.5 * d / np.linalg.norm(d)
    return dict(xyz=xyz, type=rng.integers(0, 4, N), bonds=np.stack([par, i], 1).reshape(-1, 2), rot_edge=bonds)


CASES = {
    # 20 degree steps: 18^3 = 5,832 entries per atom behind three bonds, two such atoms
    "table_overflow": ("chain", 12, [2, 3, 4], 20, 24, "f32"),
    "table_overflow_f16": ("chain", 12, [2, 3, 4], 20, 3, "f16"),
    "two_bonds_10_degrees": ("chain", 14, [3, 8], 10, 24, "bf16"),
    "four_bonds": ("random", 13, [1, 4, 6, 9], 45, 24, "f32"),
    "four_nested": ("chain", 11, [1, 2, 3, 4], 60, 7, "f32"),
    "empty_lists": ("star", 6, [0, 2, 3], 30, 24, "f32"),
    "no_bonds": ("random", 40, [], 30, 24, "f16"),
    "one_atom": ("chain", 1, [], 30, 1, "f32"),
    "one_increment": ("random", 33, [3, 7], 360, 24, "f32"),
    "two_increments": ("random", 65, [3, 7, 9], 180, 2, "f32"),
}


@pytest.mark.parametrize("case", CASES)
def test_exhaustive_table_against_brute_force(case, oracle_lib):
    import paper_2303_06150_gb300 as lg
    kind, N, bonds, step, n_rigid, fmt = CASES[case]
    rng = np.random.default_rng(len(case))
    lib = from_ligands([_ligand(rng, N, kind, bonds), _ligand(rng, max(2, N - 1), kind, bonds)])
    grid = gen.make_grid(gen.WORKLOADS["small32"]["grid"])
    s = dict(restarts=3, torsion_step_deg=step, passes=1, top_k=3, seed=11, n_rigid=n_rigid, jitter=1.0,
             out_penalty=5.0)
    L = lg.Ligands.from_arrays(lib, "cuda")
    G = lg.PocketGrid.from_array(grid.values, grid.origin, grid.spacing, "cuda")
    ex = lg.dock_batch(L, G, mode="exhaustive", grid_format=fmt, top_restart=True, **s)
    sc, top, poses = ex.scores.cpu().numpy(), ex.top_restart.cpu().numpy(), ex.poses.cpu().numpy()
    og = parity.oracle_grid(oracle_lib, grid, fmt)
    off = lg.pose_offsets(lib.rot_off, 3)
    for l in range(lib.n_ligands):
        lig = oracle_lib.OLigand.from_library(lib, l)
        ref = oracle_lib.dock_exhaustive(lig, og, s, l, range(3))
        for k in range(3):
            r = int(top[l, k])
            S_ref = ref["score"][r]
            _, D, _, Gs = oracle_lib.score_pose(lig, og, ref["pose"][r], 5.0, sensitivity=True)
            assert abs(sc[l, k] - S_ref) <= parity.score_tol(D, Gs) + parity.gap_tol(D, Gs), (l, r, sc[l, k], S_ref)
            pose = poses[off[l]:off[l + 1]].reshape(3, -1)[k].astype(np.float64)
            S_gpu, Dg, _, Gg = oracle_lib.score_pose(lig, og, pose, 5.0, sensitivity=True)
            assert S_gpu >= S_ref - parity.gap_tol(D, Gs), (l, r, S_gpu, S_ref)
            assert abs(sc[l, k] - S_gpu) <= parity.score_tol(Dg, Gg), (l, r, sc[l, k], S_gpu)
