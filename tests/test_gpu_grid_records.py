"""Grid records of odd shapes (two-node axes, many channels, uneven axes)
sampled through one-atom ligands, on the box's upper faces too, against the
trilinear value of the node values in FP64."""
import numpy as np
import pytest

import parity

pytestmark = pytest.mark.gpu

SHAPES = [(2, 2, 2, 1), (3, 5, 7, 1), (41, 2, 3, 64), (2, 50, 33, 5), (17, 40, 14, 3), (130, 4, 2, 1)]   # nx, ny, nz, nc


def _trilinear(v, u, c):
    n = np.array([v.shape[2], v.shape[1], v.shape[0]])
    i = np.minimum(np.floor(u).astype(int), n - 2)
    f = u - i
    e = g = 0.0
    for k in range(8):
        d = np.array([k & 1, k >> 1 & 1, k >> 2])
        w = np.where(d, f, 1 - f)
        node = v[i[:, 2] + d[2], i[:, 1] + d[1], i[:, 0] + d[0], c]
        e = e + w.prod(1) * node
        g = g + np.abs(node)
    return e, g


def _one_atom_ligands(lg, nc):
    import torch
    off = torch.arange(nc + 1, dtype=torch.int32)
    z = torch.zeros(nc + 1, dtype=torch.int32)
    return lg.Ligands(off.cuda(), torch.zeros((nc, 3)).cuda(), torch.arange(nc, dtype=torch.uint8).cuda(),
                      torch.zeros((0, 2), dtype=torch.int32).cuda(), z.cuda(), z[:0].cuda())


@pytest.mark.parametrize("shape", SHAPES)
def test_fp32_records(shape):
    import torch

    import paper_2303_06150_gb300 as lg
    nx, ny, nz, nc = shape
    rng = np.random.default_rng(nx)
    v = rng.normal(size=(nz, ny, nx, nc)).astype(np.float32)
    G = lg.PocketGrid.from_array(v, (0.0, 0.0, 0.0), 1.0, "cuda")
    P = 64
    top = np.array([nx - 1, ny - 1, nz - 1])
    u = (rng.random((nc, P, 3)) * top).astype(np.float32)
    for k in range(8):   # points on the upper faces, edges and the corner
        u[:, k] = np.where([k & 1, k >> 1 & 1, k >> 2], top, u[:, k])
    poses = np.concatenate([u, np.tile(np.float32([1, 0, 0, 0]), (nc, P, 1))], 2)
    s = lg.score_poses(_one_atom_ligands(lg, nc), G, torch.from_numpy(poses).cuda().reshape(-1), P).cpu().numpy()
    for c in range(nc):
        e, g = _trilinear(v.astype(np.float64), u[c].astype(np.float64), c)
        # 3 roundings per coefficient and 7 of the polynomial, each of at most 8 node values' magnitude;
        # a position is rounded once, to 2^-24 of itself, in a field of slope <= g
        tol = (10 * 8 + top.max()) * 2.0 ** -24 * g
        assert (np.abs(s[c] + e) <= tol).all(), (c, np.abs(s[c] + e).max())


@pytest.mark.parametrize("fmt", ["f16", "bf16"])
@pytest.mark.parametrize("shape", SHAPES)
def test_16_bit_records(shape, fmt):
    import paper_2303_06150_gb300 as lg
    nx, ny, nz, nc = shape
    rng = np.random.default_rng(ny)
    v = rng.normal(size=(nz, ny, nx, nc)).astype(np.float32)
    G = lg.PocketGrid.from_array(v, (0.0, 0.0, 0.0), 1.0, "cuda")
    R = 64
    r = lg.dock_batch(_one_atom_ligands(lg, nc), G, restarts=R, torsion_step_deg=30, passes=0, top_k=R, seed=1,
                      n_rigid=1, jitter=0.5, grid_format=fmt)
    u = r.poses.cpu().numpy().reshape(nc, R, 7)[:, :, :3].astype(np.float64)
    s = r.scores.cpu().numpy()
    w = parity.record_values(v, fmt)
    top = np.array([nx - 1, ny - 1, nz - 1])
    for c in range(nc):
        e, g = _trilinear(w, u[c], c)
        tol = (10 * 8 + top.max()) * 2.0 ** -24 * g
        assert (np.abs(s[c] + e) <= tol).all(), (c, np.abs(s[c] + e).max())


@pytest.mark.parametrize("fmt", ["f32", "f16", "bf16"])
def test_docking_on_an_axis_of_2_to_the_23_cells(fmt):
    import torch

    import paper_2303_06150_gb300 as lg
    nz, R = 2 ** 23 + 1, 64
    v = torch.rand((nz, 2, 2, 1), generator=torch.Generator("cuda").manual_seed(1), device="cuda") - 0.5
    G = lg.PocketGrid(v, (0.0, 0.0, 0.0), 1.0)
    r = lg.dock_batch(_one_atom_ligands(lg, 1), G, restarts=R, torsion_step_deg=30, passes=0, top_k=R, seed=1,
                      n_rigid=1, jitter=0.5, grid_format=fmt)
    u = r.poses.cpu().numpy().reshape(R, 7)[:, :3].astype(np.float64)   # z: near 2^22, on multiples of 1/2
    z0 = int(u[:, 2].min()) - 1
    part = v[z0:z0 + 4].cpu().numpy()
    u[:, 2] -= z0
    e, g = _trilinear(parity.record_values(part, fmt), u, 0)
    # positions are exact here (origin 0, spacing 1): only the record's and the polynomial's roundings
    assert (np.abs(r.scores.cpu().numpy()[0] + e) <= 10 * 8 * 2.0 ** -24 * g).all()
