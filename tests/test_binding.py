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


# (d, f, E, k, rank), token counts, and whether the router places the rows at these sizes
SCRATCH = [
    ((2048, 5632, 8, 2, 0), (17, 333, 2048), True),
    ((2048, 5632, 8, 2, 128), (512, 2048), True),
    ((2048, 5632, 8, 2, 128), (17, 511), False),        # decomposed experts: from 1024 pairs on
    ((2048, 5632, 32, 2, 0), (17, 1024, 2048), False),  # w_router is too large for the router that places rows
    ((2048, 5632, 64, 8, 512), (300, 4000), False),
    ((512, 512, 64, 2, 0), (4000,), False),
    ((512, 512, 32, 2, 0), (17, 4000), True),
    ((16384, 64, 1, 1, 0), (40, 9000), True),           # 9000 tokens would take 295 MB: as much as fits into 256
    ((256, 512, 8, 2, 0), (1, 16), False),              # decode only
]


@pytest.mark.parametrize("cfg,tokens,placed", SCRATCH)
def test_scratch_has_room_for_placed_rows_only_where_rows_are_placed(cfg, tokens, placed):
    from paper_2503_00245_b200 import binding as B
    d, f, E, k, r = cfg
    c = B.make_config(d, f, E, k, r)
    rp = (r + 63) // 64 * 64
    for T in tokens:
        def rest(n):  # everything but the rows: routing, hidden activations, intermediates, outputs, and what decode keeps
            planes = 4 if n * k <= 2048 else 1
            return n * k * (6 * 4 + 2 * f + 12 * rp + 4 * d * planes) + 16 * d * 6 + 16 * k * (2 * f + 4 * r + 64 * 12) * 6 * 2 + 65536
        most = max(rest(n) for n in (T, min(T, 16), min(T, 2048 // k)))
        rows = min(2 * d * E * T, 256 << 20) if placed else 2 * d * T * k
        got = B.moe_workspace_bytes(c, T)
        assert got <= most + max(rows, 2 * d * T * k), (T, got, most, rows)
        if placed:
            assert got >= 0.98 * rows, (T, got, rows)


@pytest.mark.parametrize("cfg", sorted({c for c, _, _ in SCRATCH}))
def test_scratch_for_many_tokens_is_enough_for_fewer(cfg):
    from paper_2503_00245_b200 import binding as B
    d, f, E, k, r = cfg
    c = B.make_config(d, f, E, k, r)
    sizes = [B.moe_workspace_bytes(c, T) for T in [*range(1, 70), *range(70, 9000, 37)]]
    assert sizes == sorted(sizes)


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
