"""pose_score's backward asks torch about the upstream gradient by private
names; where a torch version lacks one, torch multiplies, with the same
gradient."""
import numpy as np
import pytest
import torch
from torch.autograd import forward_ad

import paper_2303_06150_gb300.api as api


@pytest.mark.parametrize("owner, name", [(torch._C, "_has_storage"), (torch._C, "_len_torch_dispatch_stack"),
                                         (torch._C, "_functorch"), (forward_ad, "_current_level")])
def test_backward_without_a_private_name(monkeypatch, owner, name):
    def weighted(*a):
        raise AssertionError("the kernel was given a gradient that could not be looked over")

    lig = type("L", (), {"h_rot_off": np.array([0, 0], dtype=np.int32)})()
    monkeypatch.setattr(api, "score_poses", lambda l, g, p, P, pen: (p * p).sum().reshape(1, 1))
    monkeypatch.setattr(api, "pose_grad", lambda l, g, poses, P, pen: (None, 2 * poses))
    monkeypatch.setattr(api, "_weighted_pose_grad", weighted)
    if owner is torch._C:   # torch itself goes on using its own names: hide them from this module only
        class Without:
            def __getattr__(self, n):
                if n == name:
                    raise AttributeError(n)
                return getattr(torch._C, n)

        class Torch:
            _C = Without()

            def __getattr__(self, n):
                return getattr(torch, n)

        monkeypatch.setattr(api, "torch", Torch())
    else:
        monkeypatch.setattr(api, "forward_ad", object())
    poses = torch.arange(1.0, 8.0).requires_grad_()
    g, = torch.autograd.grad(api.PoseScore.apply(poses, lig, None, 1, 5.0), poses, torch.tensor([[3.0]]))
    assert torch.equal(g, 6 * poses.detach())
