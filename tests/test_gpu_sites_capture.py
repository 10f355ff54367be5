"""Sites docked under stream capture: overlapped where the workspace already
holds two sets of buffers, one after another where the second would have to be
allocated. Replays equal the sites docked one by one."""
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu


def _inputs(small32, ligands):
    import paper_2303_06150_gb300 as lg
    w, lib, _ = small32
    L = lg.Ligands.from_arrays(gen.from_ligands([lib.ligand(l % 32) for l in range(ligands)]), "cuda")
    grids = []
    for spec in gen.site_grids(w["grid"], 3):
        v = gen.make_grid(spec)
        grids.append(lg.PocketGrid.from_array(v.values, v.origin, v.spacing, "cuda"))
    return lg, L, grids


@pytest.mark.parametrize("warm", ["sites", "one site", "larger call"])
def test_captured_sites(small32, warm):
    lg, L, grids = _inputs(small32, 100)
    kw = dict(restarts=16, torsion_step_deg=30, passes=2, top_k=4, seed=9)
    one = [lg.dock_batch(L, g, **kw) for g in grids]
    lg.release_workspaces()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        out = lg.dock_sites(L, grids, **kw)
        torch.cuda.synchronize()
        lg.release_workspaces()
        if warm == "sites":
            lg.dock_sites(L, grids, **kw)
        elif warm == "one site":             # room for one set of records, not for two
            lg.dock_batch(L, grids[0], **kw)
        else:                                # room for two, by a call that needs no second set
            _, many, _ = _inputs(small32, 20000)
            lg.dock_batch(many, grids[0], **dict(kw, restarts=64, top_k=1))
        out.scores.zero_()
        out.poses.zero_()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            lg.dock_sites(L, grids, out=out, **kw)
        for _ in range(2):
            out.scores.zero_()
            graph.replay()
            torch.cuda.synchronize()
            for g in range(3):
                assert torch.equal(out.scores[g], one[g].scores) and torch.equal(out.poses[g], one[g].poses)
    del graph
    lg.release_workspaces()


def test_uncaptured_sites_after_a_capture(small32):
    lg, L, grids = _inputs(small32, 50)
    kw = dict(restarts=16, torsion_step_deg=30, passes=2, top_k=4, seed=9)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        want = lg.dock_sites(L, grids, **kw)
        out = lg.dock_sites(L, grids, **kw)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            lg.dock_sites(L, grids, out=out, **kw)
        again = lg.dock_sites(L, grids, **kw)    # the same side streams and events, outside the capture
        graph.replay()
        torch.cuda.synchronize()
    assert torch.equal(want.scores, again.scores) and torch.equal(want.scores, out.scores)
    assert torch.equal(want.poses, again.poses) and torch.equal(want.poses, out.poses)
