"""The Python side of the C boundary: what imports, and what its calls accept (no GPU needed)."""
import os
import subprocess
import sys

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
