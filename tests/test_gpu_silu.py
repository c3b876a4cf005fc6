"""silu of the prefill's epilogues against 64 bits, over the whole range of its argument.

Weights that are zero but for single ones make y[t, c] the hidden activation silu(g), rounded to bf16, with g = x[t] * w[c] exact in
fp32.  A bf16 is coarse, but with a hundred thousand values some lie next to every boundary between two of them: the test asks for
the bf16 nearest to a value within the bound of the exact one, which a larger error misses.
"""
import numpy as np
import pytest
import torch

from synth import workloads as W
from tests import gpu_util as U

pytestmark = pytest.mark.gpu
N = 128  # all mantissas of a bf16


def arguments():
    """x: every bf16 of [2^-4, 256), larger and smaller powers of two and zero, both signs; w: every bf16 of [1, 2)."""
    m = 1 + np.arange(N) / N
    x = np.concatenate([m * 2.0 ** e for e in range(-4, 8)] + [2.0 ** np.array([8, 20, 60, 126, -8, -20, -60, -120]), [0.0]])
    return np.concatenate([x, -x]), m


def bound(g):
    """2^-22 for the power of two, 2^-23 for the reciprocal, one rounding of the exponent (and of its factor, a quarter of that) and
    three more roundings at 2^-24; below, what is lost where the reciprocal would not be a normal number."""
    with np.errstate(over="ignore"):
        p = 1 / (1 + np.exp(g))                          # e^-g / (1 + e^-g)
    rel = p * (np.abs(g) * 1.25 * 2.0 ** -24 + 2.0 ** -22) + 5 * 2.0 ** -24
    return rel, np.where(g < -86, np.abs(g) * 2.0 ** -125, 0.0)


def to_bf16(v):
    return torch.from_numpy(v).to(torch.float32).to(torch.bfloat16).to(torch.float64).numpy()


@pytest.mark.parametrize("r", [0, N])
def test_silu_within_the_bound_of_its_instructions(r):
    xs, ws = arguments()
    T = len(xs)
    sh = W.LayerShape("t", 9, N, N, n_experts=1, top_k=1, wd_rank=r, x_dtype="f32")
    t = {k: v if v is None else torch.zeros_like(v) for k, v in W.make_layer(sh, T, device="cuda").items()}
    eye, w = torch.eye(N, device="cuda").to(torch.bfloat16), torch.from_numpy(ws).to(torch.bfloat16).cuda()
    t["x"][:, 0], t["x"][:, 1] = torch.from_numpy(xs).float().cuda(), 1.0
    gate, up, down = ("gR", "uR", "dR") if r else ("w_gate", "w_up", "w_down")
    t[gate][0, 0], t[up][0, 1], t[down][0] = w, 1.0, eye
    if r:
        t["gL"][0], t["uL"][0], t["dL"][0] = eye, eye, eye
    lay, t, _ = U.build(sh, T, tensors=t)
    y = lay.forward(t["x"]).double().cpu().numpy()
    assert lay.check() == 0
    g = xs[:, None] * ws[None, :]
    with np.errstate(over="ignore"):
        s = g / (1 + np.exp(-g))
    rel, lost = bound(g)
    lo, hi = s - np.abs(s) * rel - lost, s + np.abs(s) * rel + lost
    bad = (y < to_bf16(lo)) | (y > to_bf16(hi)) | ~np.isfinite(y)
    assert not bad.any(), (g[bad][:5], s[bad][:5], y[bad][:5], int(bad.sum()))
