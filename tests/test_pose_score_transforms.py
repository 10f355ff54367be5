"""pose_score's backward under torch's transforms: batched gradients, vmap,
forward mode over the upstream gradient and create_graph go through torch's
product; a plain upstream gradient goes to the kernel. The library calls are
replaced by a linear score on the CPU, so every value is exact."""
import numpy as np
import pytest
import torch
from torch.autograd import forward_ad

import paper_2303_06150_gb300.api as api


@pytest.fixture
def score(monkeypatch):
    routes = []

    def weighted(l, g, poses, P, pen, w):
        w.data_ptr()   # what the kernel is given
        routes.append("kernel")
        return 2 * poses * w.reshape(-1).repeat_interleave(7)

    def plain(l, g, poses, P, pen):
        routes.append("torch")
        return None, 2 * poses

    monkeypatch.setattr(api, "_weighted_pose_grad", weighted)
    monkeypatch.setattr(api, "pose_grad", plain)
    monkeypatch.setattr(api, "score_poses", lambda l, g, p, P, pen: (p * p).reshape(2, 7).sum(1).reshape(1, 2))
    lig = type("L", (), {"h_rot_off": np.array([0, 0], dtype=np.int32)})()
    poses = torch.arange(1.0, 15.0).requires_grad_()
    return poses, api.pose_score(poses, lig, None, 2), routes


def _rows(poses):
    want = torch.zeros(2, 14)
    want[0, :7], want[1, 7:] = 2 * poses.detach()[:7], 2 * poses.detach()[7:]
    return want


def test_plain_backward_takes_the_kernel(score):
    poses, s, routes = score
    g, = torch.autograd.grad(s, poses, torch.tensor([[1.0, 3.0]]))
    assert routes == ["kernel"]
    assert torch.equal(g, _rows(poses)[0] + 3 * _rows(poses)[1])


@pytest.mark.parametrize("how", ["is_grads_batched", "vmap"])
def test_batched_upstream_gradients(score, how):
    poses, s, routes = score
    ups = torch.eye(2).reshape(2, 1, 2)
    if how == "vmap":
        g = torch.vmap(lambda u: torch.autograd.grad(s, poses, u, retain_graph=True)[0])(ups)
    else:
        g, = torch.autograd.grad(s, poses, ups, is_grads_batched=True)
    assert routes == ["torch"]
    assert torch.equal(g, _rows(poses))


def test_tangent_of_the_upstream_gradient(score):
    poses, s, routes = score
    with forward_ad.dual_level():
        up = forward_ad.make_dual(torch.ones(1, 2), torch.tensor([[3.0, 5.0]]))
        g, = torch.autograd.grad(s, poses, up)
        tangent = forward_ad.unpack_dual(g).tangent
        assert torch.equal(tangent, 3 * _rows(poses)[0] + 5 * _rows(poses)[1])
    assert routes == ["torch"]


def test_create_graph_stays_differentiable(score):
    poses, s, routes = score
    up = torch.ones(1, 2, requires_grad=True)
    g, = torch.autograd.grad(s, poses, up, create_graph=True)
    d, = torch.autograd.grad(g.sum(), up)
    assert routes == ["torch"]
    assert torch.equal(d, _rows(poses).sum(1).reshape(1, 2))
