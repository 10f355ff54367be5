"""Packer outputs at device addresses that are no multiple of four: the
library copies to them, its kernel does not store there."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [1, 2, 3, 4, 8, 16])
def test_outputs_at_any_address(small32, shift):
    import torch

    import paper_2303_06150_gb300 as lg
    _, lib, _ = small32
    L = lg.Ligands.from_arrays(lib, "cuda")
    bits, axis, bucket, status = lg.pack_ligands(L, 4)
    touch = lg.pack_touch(L, 4).to(torch.int32)
    want = [t.contiguous().view(torch.uint8).reshape(-1) for t in (bits, axis, bucket, status, touch)]
    got = [torch.full((len(w) + 32,), 7, dtype=torch.uint8, device="cuda") for w in want]
    at = [C.c_void_p(g.data_ptr() + shift) for g in got]
    abi = lg._abi
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    abi.check(abi.load().ligen_pack_ligands(C.byref(L._s), 4, *at[:4], stream))
    abi.check(abi.load().ligen_pack_touch(C.byref(L._s), 4, at[4], stream))
    torch.cuda.synchronize()
    for g, w in zip(got, want):
        assert torch.equal(g[shift:shift + len(w)], w)
        assert (g[:shift] == 7).all() and (g[shift + len(w):] == 7).all()
