"""What the RMS bound on decomposed experts in a decode step (tests/test_gpu_edges.py) can tell, on the CPU: the oracle's chain with
ONE of its vectors kept in two bf16 terms instead of three is outside of it, fp32 vectors are inside."""
import numpy as np
import pytest

from oracle import moe_oracle as O
from synth import workloads as W

RMS_BOUND = 2.0 ** -22


def bf16_terms(v, n):
    """The sum of the first n bf16 terms of a value (round to nearest even, every remainder exact)."""
    rest, total = v.astype(np.float64), np.zeros(v.shape)
    for _ in range(n):
        bits = rest.astype(np.float32).view(np.uint32).astype(np.uint64)
        bits = ((bits + 0x7fff + ((bits >> 16) & 1)) >> 16) << 16
        term = bits.astype(np.uint32).view(np.float32).astype(np.float64)
        total, rest = total + term, rest - term
    return total


def chain(x, e, keep):
    """One expert's x -> t -> h -> v -> y; `keep(name, vector)` is what the next product gets to see."""
    x = keep("x", x)
    tg, tu = keep("t", x @ e["gL"]), keep("t", x @ e["uL"])
    g = tg @ e["gR"]
    h = keep("h", g / (1.0 + np.exp(-g)) * (tu @ e["uR"]))
    return keep("v", h @ e["dL"]) @ e["dR"]


@pytest.mark.parametrize("d,f,r", [(448, 456, 448), (264, 1000, 232), (256, 512, 40), (136, 64, 16), (904, 896, 8)])
def test_a_vector_in_two_terms_is_seen(d, f, r):
    sh = W.LayerShape("t", 9, d, f, n_experts=1, top_k=1, wd_rank=r, x_dtype="f32")
    t = {k: O.widen(W.to_host_bits(v)) for k, v in W.make_layer(sh, 8).items() if v is not None}
    e = {k: t[k][0] for k in ("gL", "gR", "uL", "uR", "dL", "dR")}
    want = chain(t["x"], e, lambda name, v: v)

    def rms(keep):
        return np.sqrt(((chain(t["x"], e, keep) - want) ** 2).sum() / (want ** 2).sum())

    assert rms(lambda name, v: v.astype(np.float32).astype(np.float64)) < RMS_BOUND / 2
    assert rms(lambda name, v: bf16_terms(v, 3)) < RMS_BOUND / 2
    for cut in ("x", "t", "h", "v"):
        assert rms(lambda name, v: bf16_terms(v, 2 if name == cut else 3)) > 4 * RMS_BOUND, cut
