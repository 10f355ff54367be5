"""Every kernel shape gives the same bits: 8, 16 and 32 lanes per restart,
each record format, increments below, at and above a shape's slots; and the
plain launch, whatever lanes and ligand order it picks, equals them."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lg():
    import paper_2303_06150_gb300 as lg
    yield lg
    lg.tune_set([(8, 16)] * 44)


def _same(a, b):
    return (torch.equal(a.scores, b.scores) and torch.equal(a.poses, b.poses) and torch.equal(a.trace, b.trace) and
            torch.equal(a.top_restart, b.top_restart))


@pytest.mark.parametrize("fmt", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("step,restarts,n_rigid", [(10, 9, 24), (30, 5, 24), (24, 4, 7), (12, 3, 24), (3, 2, 1),
                                                   (360, 4, 24), (180, 33, 23)])
def test_shapes_agree_bit_for_bit(lg, screen_sample, fmt, step, restarts, n_rigid):
    _, lib, grid = screen_sample
    lib = lib.subset(range(0, 64, 5))
    L = lg.Ligands.from_arrays(lib, "cuda")
    G = lg.PocketGrid.from_array(grid.values, grid.origin, grid.spacing, "cuda")
    kw = dict(restarts=restarts, torsion_step_deg=step, passes=2, top_k=min(3, restarts), seed=4, n_rigid=n_rigid,
              grid_format=fmt, trace=True, top_restart=True)
    out = []
    for shape in ((8, 16), (16, 8), (16, 2), (32, 4), (32, 1)):
        lg.tune_set([shape] * 44)
        out.append(lg.dock_batch(L, G, batching="buckets_static", **kw))
    out.append(lg.dock_batch(L, G, **kw))
    assert all(_same(out[0], o) for o in out[1:])


# plain launches of one ligand up to a full chip; the static call shares the
# lanes but not the ligand order
@pytest.mark.parametrize("n,restarts", [(1, 1), (1, 256), (2, 40), (7, 100), (40, 64), (400, 8), (700, 96)])
def test_plain_launch_lanes_and_order(lg, small32, n, restarts):
    import gen
    w, _, grid = small32
    lib = gen.make_library(dict(w["library"], n_ligands=n, n_atoms=(1, 60), n_rot=(0, 9), seed=n))
    L = lg.Ligands.from_arrays(lib, "cuda")
    G = lg.PocketGrid.from_array(grid.values, grid.origin, grid.spacing, "cuda")
    kw = dict(restarts=restarts, torsion_step_deg=30, passes=2, top_k=1, seed=2, trace=True, top_restart=True)
    lg.tune_set([(8, 16)] * 44)
    ref = lg.dock_batch(L, G, batching="queue", **kw)   # 8 lanes
    assert _same(ref, lg.dock_batch(L, G, **kw))
    assert _same(ref, lg.dock_batch_static(L, G, **kw))
