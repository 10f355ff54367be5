"""Overlapping sites equal the sites docked one by one: odd and even counts,
grids of different sizes, FP64 re-score, two streams at once, and a workspace
limit that only one set of buffers fits."""
import numpy as np
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu


def _sites(lg, small32, n):
    w, _, _ = small32
    out = []
    for g, spec in enumerate(gen.site_grids(w["grid"], n)):
        spec = dict(spec, points=40 - 3 * (g % 3))
        v = gen.make_grid(spec)
        out.append(lg.PocketGrid.from_array(v.values, v.origin, v.spacing, "cuda"))
    return out


def _equal(a, b, g):
    return (torch.equal(a.scores[g], b.scores) and torch.equal(a.poses[g], b.poses) and
            torch.equal(a.trace[g], b.trace) and torch.equal(a.top_restart[g], b.top_restart))


@pytest.mark.parametrize("rescore", [False, True])
@pytest.mark.parametrize("n", [2, 3, 6])
def test_sites_overlap(small32, n, rescore):
    import paper_2303_06150_gb300 as lg
    _, lib, _ = small32
    lib = gen.from_ligands([lib.ligand(l % 32) for l in range(200)])
    L = lg.Ligands.from_arrays(lib, "cuda")
    grids = _sites(lg, small32, n)
    kw = dict(restarts=40, torsion_step_deg=30, passes=2, top_k=5, seed=7, rescore_fp64=rescore, trace=True,
              top_restart=True)
    one = [lg.dock_batch(L, g, **kw) for g in grids]
    a = lg.dock_sites(L, grids, **kw)
    b = lg.dock_sites(L, grids, **kw)        # the same streams and buffers again
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        c = lg.dock_sites(L, grids, **kw)
    d = lg.dock_sites(L, grids, **kw)        # beside c
    torch.cuda.synchronize()
    for g in range(n):
        assert all(_equal(x, one[g], g) for x in (a, b, c, d))
        if rescore:
            assert torch.equal(a.scores_f64[g], one[g].scores_f64)


def test_one_set_under_a_workspace_limit(small32):
    import paper_2303_06150_gb300 as lg
    _, lib, _ = small32
    L = lg.Ligands.from_arrays(lib, "cuda")
    grids = _sites(lg, small32, 3)
    kw = dict(restarts=8, torsion_step_deg=30, passes=1, top_k=2, seed=7, trace=True, top_restart=True)
    one = [lg.dock_batch(L, g, **kw) for g in grids]
    lg.release_workspaces()
    records = 39 ** 3 * 4 * 32
    try:
        lg.set_workspace_limit(records + records // 2)   # one grid's records, not two
        a = lg.dock_sites(L, grids, **kw)
        torch.cuda.synchronize()
    finally:
        lg.set_workspace_limit(0)
        lg.release_workspaces()
    assert all(_equal(a, one[g], g) for g in range(3))
    assert np.isfinite(a.scores.cpu().numpy()).all()
