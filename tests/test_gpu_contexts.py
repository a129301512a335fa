"""The library in a second CUDA context of a device: what it asks of the runtime for a kernel holds for the context that
is current, not for the device."""
import ctypes as C

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


class Driver:
    """The few driver calls that a program with a context of its own makes."""

    def __init__(self):
        self.lib = C.CDLL("libcuda.so.1")

    def __call__(self, name, *args):
        rc = getattr(self.lib, name)(*args)
        assert rc == 0, (name, rc)

    def upload(self, a):
        p = C.c_uint64()
        self("cuMemAlloc_v2", C.byref(p), C.c_size_t(a.nbytes))
        self("cuMemcpyHtoD_v2", p, a.ctypes.data_as(C.c_void_p), C.c_size_t(a.nbytes))
        return p.value


def test_attention_in_a_second_context():
    from paper_2605_14513_b200 import heart

    H, N = 2, 700
    g = torch.Generator("cuda").manual_seed(0)
    Q, K, V = (torch.randn((1, H, N, 128), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    cfg = heart.make_config(1, H, N, 64, flags=heart.FORCE_DENSE)
    O = torch.empty_like(Q)
    heart.heart_block_sparse_attn(cfg, Q, K, V, None, None, O, heart.new_workspace(cfg))
    want = O.cpu().view(torch.int16).numpy()
    host = [x.cpu().view(torch.int16).numpy() for x in (Q, K, V)]
    cu, ctx, dev, code = Driver(), C.c_void_p(), C.c_int(), C.c_int32(-1)
    got = np.zeros_like(want)
    cu("cuDeviceGet", C.byref(dev), torch.cuda.current_device())
    cu("cuCtxCreate_v2", C.byref(ctx), C.c_uint(0), dev)
    try:
        q, k, v, o = (cu.upload(x) for x in (*host, got))
        ws = cu.upload(np.zeros(heart.workspace_bytes(cfg), np.uint8))
        lib = heart.lib()
        assert lib.heart_block_sparse_attn(C.byref(cfg), q, k, v, None, None, o, None, ws, None) == heart.OK
        assert lib.heart_get_status(ws, None, C.byref(code)) == heart.OK and code.value == 0
        cu("cuMemcpyDtoH_v2", got.ctypes.data_as(C.c_void_p), C.c_uint64(o), C.c_size_t(got.nbytes))
    finally:
        cu("cuCtxDestroy_v2", ctx)
    assert np.array_equal(got, want)
    # and the first context is as it was
    heart.heart_block_sparse_attn(cfg, Q, K, V, None, None, O, heart.new_workspace(cfg))
    assert np.array_equal(O.cpu().view(torch.int16).numpy(), want)
