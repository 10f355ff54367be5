"""ligen_pose_grad_weighted is ligen_pose_grad times the weights, bit for bit
(every kernel and group width, device and host memory, a malformed ligand),
and autograd's backward equals it for dense, expanded and double-backward
upstream gradients."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _case(small32, P, device):
    import paper_2303_06150_gb300 as lg
    _, lib, grid = small32
    lib = lib.subset(range(9))
    lib.bonds[int(lib.atom_off[4]) - 4] = [1, 1]   # ligand 4: not a tree
    rng = np.random.default_rng(P)
    parts = [np.concatenate([grid.center + rng.uniform(-1, 1, (P, 3)), rng.normal(size=(P, 4)),
                             rng.uniform(-3, 3, (P, n))], 1).ravel() for n in lib.n_rot]
    poses = torch.from_numpy(np.concatenate(parts).astype(np.float32))
    w = torch.from_numpy(rng.normal(size=(9, P)).astype(np.float32))
    return (lg, lg.Ligands.from_arrays(lib, device), lg.PocketGrid.from_array(grid.values, grid.origin, grid.spacing, device),
            poses.to(device), w.to(device))


@pytest.mark.parametrize("device", ["cuda", "cpu"])
@pytest.mark.parametrize("P", [1, 3, 4, 9, 16, 20])
def test_weighted_gradient(small32, P, device):
    lg, L, G, poses, w = _case(small32, P, device)
    s, g = lg.pose_grad(L, G, poses, P)
    n = torch.from_numpy(L.n_rot.astype(np.int64)) + 7
    per_value = w.cpu().reshape(-1).repeat_interleave(n.repeat_interleave(P)).to(device)
    x = poses.clone().requires_grad_(True)
    lg.pose_score(x, L, G, P).backward(w)
    assert torch.equal(x.grad, g * per_value)
    valid = torch.arange(9) != 4
    assert not torch.isfinite(s.cpu()[4]).any() and torch.isfinite(s.cpu()[valid]).all()


def test_backward_of_expanded_and_differentiable_gradients(small32):
    lg, L, G, poses, w = _case(small32, 16, "cuda")
    _, g = lg.pose_grad(L, G, poses, 16)
    x = poses.clone().requires_grad_(True)
    scores = lg.pose_score(x, L, G, 16)
    (gx,) = torch.autograd.grad(scores, x, torch.ones((), device="cuda").expand_as(scores), retain_graph=True)
    assert torch.equal(gx, g)
    u = w.clone().requires_grad_(True)   # d(w . dS/dx)/dw through the backward
    (gu,) = torch.autograd.grad(scores, x, u, create_graph=True)
    (du,) = torch.autograd.grad(gu.sum(), u)
    n = torch.from_numpy(L.n_rot.astype(np.int64)) + 7
    rows = torch.split(g, n.repeat_interleave(16).tolist())
    assert torch.allclose(du.reshape(-1), torch.stack([r.sum() for r in rows]), rtol=1e-5, atol=1e-4)
