"""The Python side of the C boundary: what imports, and what its calls accept (no GPU needed)."""
import ctypes
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_package_imports_with_a_pytorch_built_without_cuda():
    """Such a build has none of the CUDA entry points of torch._C."""
    code = ("import torch\n"
            "for n in [n for n in dir(torch._C) if n.startswith('_cuda_get')]:\n"
            "    delattr(torch._C, n)\n"
            "import paper_2503_00245_b200 as P\n"
            "assert P.binding.moe_workspace_bytes(P.binding.make_config(256, 512, 8, 2), 1) > 0\n")
    run = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert run.returncode == 0, run.stderr


def test_layer_forward_takes_weights_only_where_weights_are_due():
    from paper_2503_00245_b200 import binding as B

    class Scratch(int):  # stands in for a tensor: an address with a size
        nbytes = 0

    cfg = B.make_config(256, 512, 8, 2)
    for wrong in (cfg, ctypes.c_int(0), None):
        with pytest.raises((ctypes.ArgumentError, TypeError)):
            B.moe_layer_forward(None, 16, 1, wrong, 16, ws=Scratch(16), stream=0)
    with pytest.raises(B.MoeError) as e:  # the right type reaches the library (which has no context here)
        B.moe_layer_forward(None, 16, 1, B.moe_weights(), 16, ws=Scratch(16), stream=0)
    assert e.value.status == 1
