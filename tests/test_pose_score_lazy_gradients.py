"""pose_score's backward with an upstream gradient whose memory is not its
value: torch's negative bit (set on real gradients that come out of conjugated
complex expressions) and zero tensors without storage. The library calls are
replaced at the C entry by a quadratic score that reads the memory behind the
pointers, as the kernels do, so every value is exact."""
import ctypes as C

import numpy as np
import pytest
import torch

import paper_2303_06150_gb300.api as api


class _Memory:
    """The C entries on host memory: score = sum of squares of a pose's 7 floats."""

    def __init__(self, P):
        self.P = P

    def _array(self, ptr, n):
        return np.ctypeslib.as_array(C.cast(ptr, C.POINTER(C.c_float)), (n,))

    def ligen_score_poses(self, lig, grid, P, poses, pen, scores, stream):
        self._array(scores, P)[:] = (self._array(poses, 7 * P).reshape(P, 7) ** 2).sum(1)
        return 0

    def ligen_pose_grad(self, lig, grid, P, poses, pen, scores, grads, stream):
        self._array(grads, 7 * P)[:] = 2 * self._array(poses, 7 * P)
        return 0

    def ligen_pose_grad_weighted(self, lig, grid, P, poses, pen, weights, scores, grads, stream):
        w = self._array(weights, P)   # an address of 0 raises here
        self._array(grads, 7 * P)[:] = 2 * self._array(poses, 7 * P) * w.repeat(7)
        return 0


def _scored(monkeypatch, P):
    monkeypatch.setattr(api._abi, "load", lambda: _Memory(P))
    monkeypatch.setattr(api, "_stream_handle", lambda device: None)
    lig = type("L", (), {"h_rot_off": np.array([0, 0], dtype=np.int32), "n_ligands": 1, "_s": C.c_int(0)})()
    grid = type("G", (), {"_s": C.c_int(0)})()
    poses = torch.arange(1.0, 7.0 * P + 1).requires_grad_()
    return poses, api.pose_score(poses, lig, grid, P)


def test_conjugated_complex_expression(monkeypatch):
    poses, s = _scored(monkeypatch, 1)
    # d/ds Re(conj(i s) (1 + 2i)) = 2; torch hands it down as the negative of a -2
    (torch.complex(torch.zeros_like(s), s).conj() * (1 + 2j)).real.sum().backward()
    assert torch.equal(poses.grad, 4 * poses.detach())


@pytest.mark.parametrize("P", [1, 2, 5])
def test_negative_view(monkeypatch, P):
    poses, s = _scored(monkeypatch, P)
    up = torch._neg_view(torch.arange(1.0, P + 1).reshape(1, P))
    assert up.is_neg() and up.is_contiguous()
    g, = torch.autograd.grad(s, poses, up)
    assert torch.equal(g, -2 * poses.detach() * torch.arange(1.0, P + 1).repeat_interleave(7))


@pytest.mark.parametrize("P", [1, 2])
def test_zero_tensor(monkeypatch, P):
    poses, s = _scored(monkeypatch, P)
    g, = torch.autograd.grad(s, poses, torch._efficientzerotensor((1, P)))
    assert torch.equal(g, torch.zeros(7 * P))


def test_plain_gradient(monkeypatch):
    poses, s = _scored(monkeypatch, 2)
    g, = torch.autograd.grad(s, poses, torch.tensor([[1.0, 3.0]]))
    assert torch.equal(g, 2 * poses.detach() * torch.tensor([1.0, 3.0]).repeat_interleave(7))
