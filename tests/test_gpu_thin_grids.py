"""Grid records of grids with few points along x: the values of the same field
with its axes exchanged, and no more time than the preparation of the same
number of records with long rows takes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _one_atom(lg):
    import torch
    return lg.Ligands(torch.tensor([0, 1], dtype=torch.int32).cuda(), torch.zeros((1, 3)).cuda(),
                      torch.zeros(1, dtype=torch.uint8).cuda(), torch.zeros((0, 2), dtype=torch.int32).cuda(),
                      torch.zeros(2, dtype=torch.int32).cuda(), torch.zeros(0, dtype=torch.int32).cuda())


@pytest.mark.parametrize("nx,ny,nz,nc", [(2, 300, 11, 1), (2, 129, 7, 3), (3, 65, 65, 1), (5, 2, 300, 2), (33, 257, 2, 1)])
def test_axes_exchanged(nx, ny, nz, nc):
    import torch

    import paper_2303_06150_gb300 as lg
    rng = np.random.default_rng(nx + ny)
    v = rng.normal(size=(nz, ny, nx, nc)).astype(np.float32)
    a = lg.PocketGrid.from_array(v, (0.0, 0.0, 0.0), 1.0, "cuda")
    b = lg.PocketGrid.from_array(v.transpose(1, 2, 0, 3), (0.0, 0.0, 0.0), 1.0, "cuda")   # x <- z, y <- x, z <- y
    P = 256
    # node positions: the trilinear value is the node's own, through any cell around it, exactly at f = 0 and
    # within the three roundings of each coefficient and seven of the polynomial at f = 1
    node = np.stack([rng.integers(0, n, P) for n in (nx, ny, nz)], 1)
    pose = np.zeros((P, 7), np.float32)
    pose[:, :3], pose[:, 3] = node, 1
    turned = pose.copy()
    turned[:, :3] = node[:, [2, 0, 1]]
    want = -v[node[:, 2], node[:, 1], node[:, 0], 0]
    tol = 10 * 8 * 2.0 ** -24 * 8 * np.abs(v).max()
    for grid, p in ((a, pose), (b, turned)):
        s = lg.score_poses(_one_atom(lg), grid, torch.from_numpy(p).cuda().reshape(-1), P).cpu().numpy()[0]
        assert (np.abs(s - want) <= tol).all()


def test_short_rows_cost_no_more_than_long_ones():
    import torch

    import paper_2303_06150_gb300 as lg
    lig = _one_atom(lg)
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

    # 4.0 M records; the rest of the call (packer, scoring, launches) is in both. With a row of cells to a block:
    # 369 against 44 us
    assert us(2, 2000, 2000) <= 2 * us(2000, 2000, 2)
