"""Grid records of grids whose planes have fewer (x, y, channel) columns than
a block of the preparation has threads: node values, and no more time than the
same number of records in wide planes takes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _one_atom_ligands(lg, nc):
    import torch
    off = torch.arange(nc + 1, dtype=torch.int32)
    z = torch.zeros(nc + 1, dtype=torch.int32)
    return lg.Ligands(off.cuda(), torch.zeros((nc, 3)).cuda(), torch.arange(nc, dtype=torch.uint8).cuda(),
                      torch.zeros((0, 2), dtype=torch.int32).cuda(), z.cuda(), z[:0].cuda())


# columns 1, 3, 64, 63 and 127 of FP32 records; ends of marches and blocks along z
@pytest.mark.parametrize("nx,ny,nz,nc", [(2, 2, 2, 1), (2, 2, 257, 1), (2, 2, 70001, 1), (4, 2, 5000, 1),
                                         (9, 9, 333, 1), (2, 22, 900, 3), (128, 2, 40, 1)])
@pytest.mark.parametrize("fmt", ["f32", "f16"])
def test_node_values(nx, ny, nz, nc, fmt):
    import torch

    import paper_2303_06150_gb300 as lg
    rng = np.random.default_rng(nz)
    v = rng.integers(-64, 65, size=(nz, ny, nx, nc)).astype(np.float32)   # exact in every format, and their differences
    G = lg.PocketGrid.from_array(v, (0.0, 0.0, 0.0), 1.0, "cuda")
    P = 2000
    node = np.stack([rng.integers(0, n, (nc, P)) for n in (nx, ny, nz)], -1)
    node[:, 0], node[:, 1] = 0, [nx - 1, ny - 1, nz - 1]
    L = _one_atom_ligands(lg, nc)
    want = -v[node[..., 2], node[..., 1], node[..., 0], np.arange(nc)[:, None]]
    if fmt == "f32":
        pose = np.zeros((nc, P, 7), np.float32)
        pose[..., :3], pose[..., 3] = node, 1
        s = lg.score_poses(L, G, torch.from_numpy(pose).cuda().reshape(-1), P).cpu().numpy()
        assert (s == want).all()
    else:   # the docking kernel's samples, at the box's midpoint (jitter 0): the mean of the nodes around it
        r = lg.dock_batch(L, G, restarts=1, torsion_step_deg=30, passes=1, top_k=1, jitter=0.0, seed=1,
                          grid_format=fmt)
        i = [(n - 1) // 2 for n in (nx, ny, nz)]
        j = [n // 2 for n in (nx, ny, nz)]   # equal to i where the midpoint lies on a node
        mean = np.mean([v[z, y, x] for z in (i[2], j[2]) for y in (i[1], j[1]) for x in (i[0], j[0])], axis=0)
        assert (r.scores.cpu().numpy()[:, 0] == -mean).all()


def test_thin_planes_cost_no_more_than_wide_ones():
    import torch

    import paper_2303_06150_gb300 as lg
    lig = _one_atom_ligands(lg, 1)
    pose = torch.tensor([0.5, 0.5, 0.5, 1.0, 0, 0, 0]).cuda()

    def us(nx, ny, nz):
        g = lg.PocketGrid(torch.rand((nz, ny, nx, 1), device="cuda"), (0.0, 0.0, 0.0), 1.0)
        t = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        best = float("inf")
        for _ in range(20):
            t[0].record()
            for _ in range(4):
                lg.score_poses(lig, g, pose, 1)
            t[1].record()
            t[1].synchronize()
            best = min(best, t[0].elapsed_time(t[1]) * 250)
        return best

    # 4.0 M records; the rest of the call (packer, scoring, launches) is in both. With a march to a block: 242
    # against 44 us
    assert us(2, 2, 4000001) <= 2 * us(2001, 2001, 2)
