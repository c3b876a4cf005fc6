"""One process, one GPU, two CUDA contexts: what the library sets up once belongs to the context it was set up in."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import ctypes as C
import numpy as np
import torch
from paper_2503_00245_b200 import binding as B
from synth import workloads as W
from tests import gpu_util as U

cases = [(W.TINY, 16), (W.TINY, 40), (W.LayerShape("t", 9, 256, 512, wd_rank=64), 5), (W.LayerShape("t", 9, 256, 512, wd_rank=64), 1)]
want = []
for sh, T in cases:                                   # the primary context, through PyTorch
    lay, t, host = U.build(sh, T)
    want.append((lay, t, lay.forward(t["x"]).cpu()))
torch.cuda.synchronize()

cu = C.CDLL("libcuda.so.1")
def ok(name, *args):
    rc = getattr(cu, name)(*args)
    assert rc == 0, (name, rc)
ctx2 = C.c_void_p()
ok("cuCtxCreate_v2", C.byref(ctx2), 0, 0)             # made and made current
def put(tensor):
    h = tensor.detach().cpu().contiguous()
    p = C.c_uint64()
    ok("cuMemAlloc_v2", C.byref(p), C.c_size_t(max(h.nbytes, 16)))
    ok("cuMemcpyHtoD_v2", p, C.c_void_p(h.data_ptr()), C.c_size_t(h.nbytes))
    return p.value
for lay, t, y in want:
    kept = lay.weights._keep                          # w_router, b_router, gud, wd_a ... wd_d, expert_slot
    w = B.moe_weights(*[None if k is None else put(k) for k in kept])
    h = B.moe_create(lay.cfg)
    nbytes = B.moe_workspace_bytes(lay.cfg, y.shape[0])
    ws, out = put(torch.empty(nbytes, dtype=torch.uint8)), put(torch.zeros_like(y))
    rc = B._lib().moe_layer_forward(h, put(t["x"]), y.shape[0], C.addressof(w), out, None, None, ws, nbytes, None)
    assert rc == 0, (rc, B._lib().moe_last_cuda_error(), lay.cfg.wd_rank, y.shape)
    assert B.moe_check(h, 0) == 0
    got = torch.empty_like(y)
    ok("cuMemcpyDtoH_v2", C.c_void_p(got.data_ptr()), C.c_uint64(out), C.c_size_t(got.nbytes))
    assert torch.equal(got, y), "outputs differ between the contexts"
    B.moe_destroy(h)
ok("cuCtxDestroy_v2", ctx2)
print("two contexts: same outputs")
"""


def test_a_second_cuda_context_on_the_same_gpu():
    run = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=240)
    assert run.returncode == 0 and "same outputs" in run.stdout, run.stdout[-500:] + run.stderr[-2000:]
