"""The Python side of the C boundary: what imports, and what its calls accept (no GPU needed)."""
import ctypes
import os
import subprocess
import sys

import pytest
import torch

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


def test_y_is_a_plain_tensor_on_the_layers_device(monkeypatch):
    """Wherever x lies and whatever subclass it is."""
    from paper_2503_00245_b200 import layer as L

    class Tagged(torch.Tensor):
        is_cuda = True  # (as far as the layer can tell)

        def get_device(self):
            return 1

    lay = object.__new__(L.MoELayer)
    lay.d, lay.x_dtype, lay.max_tokens, lay.device, lay._cuda_index = 8, torch.float32, 4, torch.device("cpu"), 0
    lay.ctx = lay.weights = lay.ws = None
    monkeypatch.setattr(L.B, "moe_layer_forward", lambda *a: None)
    for index in (0, 1):
        lay._cuda_index = index
        y = lay.forward(torch.zeros(2, 8).as_subclass(Tagged))
        assert type(y) is torch.Tensor and y.device == lay.device and y.shape == (2, 8) and y.is_contiguous()
