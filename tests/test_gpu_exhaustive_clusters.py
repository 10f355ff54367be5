"""Exhaustive search over the range of its launch rule: one to eight CTAs per
(ligand, restart), the build for little work, few rotations, many restarts. A
restart's result does not depend on how many others the call has, so calls of
few restarts (the widest clusters) give the same bits as calls of many (one
CTA). Little work costs about what the greedy search of it costs."""
import numpy as np
import pytest

import gen
from gen.library import from_ligands

pytestmark = pytest.mark.gpu


def _ligand(rng, N, n):
    i = np.arange(1, N)
    par = (rng.random(N - 1) * i).astype(int)
    xyz = np.zeros((N, 3))
    for k in i:
        d = rng.normal(size=3)
        xyz[k] = xyz[par[k - 1]] + 1.5 * d / np.linalg.norm(d)
    return dict(xyz=xyz, type=rng.integers(0, 4, N), bonds=np.stack([par, i], 1).reshape(-1, 2),
                rot_edge=np.sort(rng.choice(N - 1, n, replace=False)) if n else np.zeros(0, int))


def _setup(sizes, seed=3):
    import paper_2303_06150_gb300 as lg
    rng = np.random.default_rng(seed)
    grid = gen.make_grid(gen.WORKLOADS["small32"]["grid"])
    return (lg, lg.Ligands.from_arrays(from_ligands([_ligand(rng, N, n) for N, n in sizes]), "cuda"),
            lg.PocketGrid.from_array(grid.values, grid.origin, grid.spacing, "cuda"))


# (ligands, step, rotations, restarts of the small call): rigid and one-bond ligands on the small build, two and
# three bonds on wide and narrow clusters, a table of one rotation at a time, one atom, rotations fewer than CTAs
CASES = {
    "rigid": ([(1, 0), (17, 0), (33, 0), (42, 0)], 30, 24, 1),
    "one_bond_one_rotation": ([(8, 1), (20, 1), (85, 1)], 30, 1, 2),
    "one_bond": ([(8, 1), (20, 0), (200, 1)], 30, 24, 2),
    "two_bonds": ([(14, 2), (20, 2), (9, 1)], 30, 24, 1),
    "two_bonds_three_rotations": ([(14, 2), (20, 2)], 24, 3, 1),
    "two_bonds_five_rotations": ([(14, 2), (20, 2)], 20, 5, 1),
    "three_bonds": ([(14, 3), (20, 3), (11, 0)], 30, 7, 1),
    "mixed": ([(20, 3), (8, 0), (12, 1), (16, 2)], 45, 24, 2),
}


@pytest.mark.parametrize("fmt", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("case", CASES)
def test_restarts_do_not_depend_on_the_launch(case, fmt):
    sizes, step, n_rigid, few = CASES[case]
    lg, L, G = _setup(sizes)
    kw = dict(torsion_step_deg=step, passes=1, seed=5, n_rigid=n_rigid, mode="exhaustive", grid_format=fmt,
              top_restart=True)
    a = lg.dock_batch(L, G, restarts=few, top_k=few, **kw)
    many = 1500
    b = lg.dock_batch(L, G, restarts=many, top_k=many, **kw)
    for l in range(len(sizes)):
        at = b.top_restart[l].argsort()                      # rank of each restart
        pa, pb = a.ligand_poses(L.h_rot_off, l), b.ligand_poses(L.h_rot_off, l)
        for k in range(few):
            r = int(a.top_restart[l, k])
            assert a.scores[l, k] == b.scores[l, at[r]]
            assert (pa[k] == pb[at[r]]).all()


@pytest.mark.parametrize("n_rigid", [1, 24])
def test_rigid_ligands_cost_what_the_greedy_search_costs(n_rigid):
    import torch
    lg, L, G = _setup([(8 + i % 13, 0) for i in range(3000)])
    kw = dict(restarts=16, torsion_step_deg=30, passes=1, top_k=1, seed=5, n_rigid=n_rigid)

    def us(mode):
        t = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        best = float("inf")
        for _ in range(6):
            t[0].record()
            lg.dock_batch(L, G, mode=mode, **kw)
            t[1].record()
            t[1].synchronize()
            best = min(best, t[0].elapsed_time(t[1]) * 1000)
        return best

    # the same poses are scored (3.2 and 4 times the greedy call at 24 and 1 rotations); eight CTAs per restart took
    # ten times as long as one
    assert us("exhaustive") <= 8 * us("greedy")
