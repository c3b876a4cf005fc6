"""GPU parity at the sizes where the kernels' splits change: slices and tiles with remainders, more pairs than a warp has
lanes, expert counts that are no multiple of eight, contractions that are cut into planes."""
import pytest
import torch

from oracle import moe_oracle as O
from synth import workloads as W
from tests import gpu_util as U

pytestmark = pytest.mark.gpu

# Decomposed experts in a decode step carry their intermediates as fp32 (one token) or as three bf16 terms of an fp32 value
# (several): every product is a sum of at most K = 5632 terms, rounded at 2^-24 each, and its rounding errors add up like a
# random walk, sqrt(K) * 2^-24 = 4.5e-6 per product at most; four products in a row, of the output's RMS.
F32_TOL = 4 * 5632 ** 0.5 * 2.0 ** -24


def check_prefill(lay, t, host, k):
    """Element by element: half a unit in the last place of y's type, and six standard deviations of what rounding the
    hidden activations to bf16 leaves in y.  Rounding changes a value by 2^-9 / sqrt(3) of itself (RMS), y is a sum of
    f >= 512 such terms of random sign, so an element's standard deviation is that share of its own TOKEN's RMS; fp32 token
    rows are rounded to bf16 as well, which both products pass on: about twice that in all."""
    _, ora, y = U.check_layer(lay, t, host, k, tol=1.0)
    sigma = 2.0 ** -9 / 3 ** 0.5 * (2.0 if t["x"].dtype == torch.float32 else 1.0)
    widest = max(U.rms(row) for row in ora["y"]) / U.rms(ora["y"])
    U.assert_close_in_output_type(U.to64(y), ora["y"], rms_tol=6 * sigma * widest, mant_bits=8 if y.dtype == torch.bfloat16 else 24)


def shape(d, f, E=8, k=2, r=0, xd="bf16", bias="none"):
    return W.LayerShape("t", 9, d, f, n_experts=E, top_k=k, wd_rank=r, x_dtype=xd, bias=bias)


@pytest.mark.parametrize("sh,T", [
    (shape(448, 456, r=448, xd="f32"), 2),              # a whole slice of the contraction, and one of eight values beside it
    (shape(904, 896, r=8, xd="f32"), 3),                # a rank below one unit, a slice of eight values
    (shape(264, 1000, E=6, k=3, r=232, xd="f32"), 5),   # router as a launch of its own
    (shape(256, 520, E=1, k=1, r=72, xd="f32"), 16),    # one expert with two groups of eight tokens
    (shape(256, 512, E=16, k=4, r=40, xd="f32"), 16),   # 64 pairs: grouped in rounds
    (shape(136, 64, E=64, k=8, r=16, xd="f32"), 9),     # more active experts than CTAs share evenly
    (shape(2312, 512, r=64, xd="f32"), 4),              # more features than one round of the router holds
    (shape(2048, 5632, r=1024), 8),
])
def test_decomposed_decode_of_several_tokens(sh, T):
    lay, t, host = U.build(sh, T)
    U.check_layer(lay, t, host, sh.top_k, tol=F32_TOL if sh.x_dtype == "f32" else U.Y_TOL)
    # the per-slot form of the same kernel
    ora = U.oracle_layer(host, sh.top_k)
    out = lay.expert_ffn(t["x"], torch.from_numpy(ora["offsets"]).cuda(), torch.from_numpy(ora["perm"]).cuda())
    torch.cuda.synchronize()
    assert lay.check() == 0
    U.assert_close_rms(out.cpu().numpy().astype("float64"), ora["out_slots"], tol=F32_TOL, what="out_slots")


@pytest.mark.parametrize("sh", [
    shape(2048, 5632, r=128, xd="f32"),                 # every later weight of a warp in registers
    shape(2048, 5632, r=136, xd="f32"),                 # product 2's rows longer than a chunk per lane
    shape(256, 5632, E=4, k=4, r=128, xd="f32"),        # more units per warp than registers hold
    shape(72, 40, E=5, k=1, r=8, xd="f32"),
])
def test_decomposed_decode_of_one_token(sh):
    lay, t, host = U.build(sh, 1)
    U.check_layer(lay, t, host, sh.top_k, tol=F32_TOL)


@pytest.mark.parametrize("sh,T", [
    (shape(72, 512, E=2, k=2), 17),                     # one CTA and a remainder of one token; features no multiple of 32
    (shape(264, 512, E=6, k=3, xd="f32"), 33),
    (shape(128, 512, E=16, k=1, bias="normal"), 1000),
    (shape(64, 512, E=64, k=8), 700),                   # two logits per lane
    (shape(64, 512, E=8, k=4), 2100),                   # more pairs per warp than it keeps in registers
    (shape(2048, 512, E=32, k=2), 40),                  # W_r too large for shared memory: the plain router
])
def test_many_tokens_routed_and_grouped(sh, T):
    lay, t, host = U.build(sh, T)
    idx, w, probs = lay.route(t["x"], want_probs=True)
    torch.cuda.synchronize()
    R, Wt, S, wo = O.route(host["x"], host["w_router"], host["b_router"], sh.top_k, True)
    U.check_routing(idx.cpu().numpy(), w.cpu().numpy(), {"logits": R, "topk_idx": S, "topk_w": wo}, sh.top_k)
    assert abs(probs.cpu().numpy() - Wt).max() <= U.W_TOL
    for _ in range(2):                                  # (the CTAs' counter is back at zero after a call)
        check_prefill(lay, t, host, sh.top_k)


@pytest.mark.parametrize("xd", ["bf16", "f32"])
@pytest.mark.parametrize("d", [8, 16, 24, 40])
@pytest.mark.parametrize("T", [17, 32])
def test_rows_shorter_than_a_unit_of_the_router(d, T, xd):
    """Fewer features than the 32 a group of lanes takes at once (and one more than that): nothing past a row counts, wherever x
    lies in memory."""
    sh = shape(d, 64, xd=xd)
    t = W.make_layer(sh, T, device="cuda")
    room = torch.full((T * d + 64,), float("nan"), dtype=t["x"].dtype, device="cuda")
    room[:T * d] = t["x"].reshape(-1)
    t["x"] = room[:T * d].view(T, d)
    lay, t, host = U.build(sh, T, tensors=t)
    idx, w, probs = lay.route(t["x"], want_probs=True)
    torch.cuda.synchronize()
    R, Wt, S, wo = O.route(host["x"], host["w_router"], host["b_router"], sh.top_k, True)
    U.check_routing(idx.cpu().numpy(), w.cpu().numpy(), {"logits": R, "topk_idx": S, "topk_w": wo}, sh.top_k)
    assert abs(probs.cpu().numpy() - Wt).max() <= U.W_TOL
    offsets, perm, inv = lay.permute(idx)
    assert torch.equal(lay.forward(t["x"]), lay.combine(lay.expert_ffn(t["x"], offsets, perm), w, inv))
    assert lay.check() == 0


@pytest.mark.parametrize("sh,T", [
    (shape(1440, 1280), 100),                           # three or four planes, columns no multiple of a tile
    (shape(200, 2000, E=2, k=1), 40),                   # a row of d shorter than one round of the combine's loads
    (shape(1024, 1024, xd="f32"), 300),
    (shape(512, 2048, r=64), 600),                      # third GEMM cut into planes
    (shape(512, 2048, r=72, E=4), 129),
])
def test_prefill_with_a_cut_contraction(sh, T):
    lay, t, host = U.build(sh, T)
    check_prefill(lay, t, host, sh.top_k)
    idx, w, _ = lay.route(t["x"])
    offsets, perm, inv = lay.permute(idx)
    y = lay.combine(lay.expert_ffn(t["x"], offsets, perm), w, inv)
    assert torch.equal(y, lay.forward(t["x"]))          # the layer and its four calls add the planes in the same order
    assert lay.check() == 0


@pytest.mark.parametrize("sh,T", [
    (shape(72, 512, E=2, k=2), 17),                     # few tiles: some pairs of CTAs start with the second product
    (shape(264, 520, E=33, k=8, xd="f32"), 31),         # a second expert per lane; experts with fewer tokens than a tile's 32
    (shape(136, 5632, E=1, k=1), 257),                  # two token tiles, uneven
    (shape(1024, 520, E=4, k=4), 129),                  # more than 128 columns: one accumulator buffer, then two again
    (shape(2056, 512, bias="normal"), 200),             # features beyond a tile of 256, uneven load
    (shape(512, 512, E=64, k=2), 4100),                 # room for every token at every expert would be too much: grouped by slot
    (shape(512, 512, E=64, k=2, r=64), 4100),
    (shape(264, 520, E=33, k=8, r=40, xd="f32"), 31),
    (shape(512, 1024, E=4, k=4, r=128, bias="normal"), 300),
])
def test_prefill_tiles_and_the_rows_places(sh, T):
    lay, t, host = U.build(sh, T)
    check_prefill(lay, t, host, sh.top_k)
    idx, w, _ = lay.route(t["x"])
    offsets, perm, inv = lay.permute(idx)
    y = lay.combine(lay.expert_ffn(t["x"], offsets, perm), w, inv)
    for _ in range(3):                                  # the rows' places differ from call to call, an element's value does not
        assert torch.equal(y, lay.forward(t["x"]))
    fewer = t["x"][:max(17, T // 3)].contiguous()
    assert torch.equal(lay.forward(fewer), lay.forward(fewer))
    assert lay.check() == 0


@pytest.mark.parametrize("sh,T,bias,spread", [
    (shape(264, 520, E=16, k=2), 600, 30.0, 1),         # every token at the same two experts: tiles far wider than an even share
    (shape(264, 520, E=16, k=2), 600, 30.0, 8),         # ... and the others' few tokens beside them
    (shape(1024, 1032, E=8, k=2, xd="f32"), 257, 30.0, 1),  # two tiles of 160 columns
    (shape(136, 512, E=64, k=1), 1100, 30.0, 8),
    (shape(304, 904, E=2, k=1), 1900, 0.0, 1),          # short contractions: tiles of at most 128 columns
])
def test_prefill_of_unevenly_routed_tokens(sh, T, bias, spread):
    """The first experts' logits are `bias` higher, all logits `spread` times as wide as usual (in w_router, a power of two, so that
    the rows keep the one scale that check_prefill's bound is derived for)."""
    t = W.make_layer(sh, T, device="cuda")
    t["b_router"] = torch.zeros(sh.n_experts, device="cuda")
    t["b_router"][:sh.top_k] = bias
    t["w_router"] *= spread
    lay, t, host = U.build(sh, T, tensors=t)
    check_prefill(lay, t, host, sh.top_k)
    idx, w, _ = lay.route(t["x"])
    offsets, perm, inv = lay.permute(idx)
    assert torch.equal(lay.combine(lay.expert_ffn(t["x"], offsets, perm), w, inv), lay.forward(t["x"]))
    assert lay.check() == 0


@pytest.mark.parametrize("sh,T,bias", [
    (shape(264, 520, E=33, k=8, r=40, xd="f32"), 200, 0.0),  # a second expert per lane, rows placed by the router
    (shape(136, 512, E=64, k=8, r=64), 300, 0.0),
    (shape(136, 512, E=64, k=8, r=64), 300, 30.0),           # ... most experts without a token
    (shape(264, 520, E=33, k=8), 200, 30.0),
])
def test_prefill_of_many_experts_and_then_of_fewer_tokens(sh, T, bias):
    t = W.make_layer(sh, T, device="cuda")
    t["b_router"] = torch.zeros(sh.n_experts, device="cuda")
    t["b_router"][-sh.top_k:] = bias
    lay, t, host = U.build(sh, T, tensors=t)
    check_prefill(lay, t, host, sh.top_k)
    for n in (T, 150, 129, 17):                         # (decomposed experts: placed from 1024 pairs, 128 tokens, on)
        x = t["x"][:n].contiguous()
        idx, w, _ = lay.route(x)
        offsets, perm, inv = lay.permute(idx)
        y = lay.combine(lay.expert_ffn(x, offsets, perm), w, inv)
        assert torch.equal(y, lay.forward(x)), n
    assert lay.check() == 0


@pytest.mark.parametrize("r", [0, 64])
def test_captured_prefill_follows_its_inputs(r):
    """One graph of two calls, replayed on other rows in the same buffer: routing, places, tile counts and sums are those of the new
    rows, and the counters are where the next call wants them."""
    sh = shape(512, 1024, r=r, bias="normal")
    lay, t, host = U.build(sh, 600)
    x, others = t["x"].clone(), [t["x"], t["x"].flip(0).contiguous(), (t["x"] * 0.5).roll(3, 1).contiguous(), t["x"]]
    others[1][::3] = others[1][0]                       # a third of the tokens share their experts
    want = [lay.forward(v) for v in others]
    y = torch.empty_like(x)
    torch.cuda.synchronize()                            # (a context serves one stream at a time)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        lay.forward(x, y=y)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            lay.forward(x, y=y)
            z = lay.forward(x)
        for v, ref in zip(others, want):
            x.copy_(v), y.zero_(), z.zero_()
            graph.replay()
            stream.synchronize()
            assert torch.equal(y, ref) and torch.equal(z, ref)
    assert lay.check() == 0
    assert torch.equal(lay.forward(others[2]), want[2])


@pytest.mark.parametrize("T", [8, 16])
def test_dense_decode_of_several_tokens_with_many_pairs(T):
    sh = shape(512, 1024, E=16, k=8)                    # 64 and 128 pairs: beyond one per lane; every expert active
    lay, t, host = U.build(sh, T, path=1)
    U.check_layer(lay, t, host, sh.top_k)


def error_against_64_bits(got, want):
    """Of an output as a whole: its RMS error, and how far it is pulled along the result (both relative)."""
    err = got - want
    return (err ** 2).sum() ** 0.5 / (want ** 2).sum() ** 0.5, float((err * want).sum() / (want ** 2).sum())


@pytest.mark.parametrize("sh,T", [(shape(1600, 4352, r=800, xd="f32"), 5), (shape(512, 1024, E=16, k=4, r=256, xd="f32"), 7),
                                  (shape(256, 512, r=32, xd="f32"), 16)])
def test_decomposed_decode_of_several_tokens_sums_like_fp32(sh, T):
    """Four products in a row, each a sum in fp32: about ten roundings in pairs or runs, 0.42 * 2^-24 of the value each (RMS), are
    1.4 * 2^-24 per product; h takes t's error twice, y all of them: 3.5 * 2^-24, so below 2^-22.  Sums that are rounded pull the
    result nowhere; 2^-23 of it is allowed (sums that a tensor core cuts over 32 products pull by 3 * 2^-24, four of them)."""
    lay, t, host = U.build(sh, T)
    rel, ora, y = U.check_layer(lay, t, host, sh.top_k, tol=F32_TOL)
    rms, pull = error_against_64_bits(U.to64(y), ora["y"])
    assert rms <= 2.0 ** -22 and abs(pull) <= 2.0 ** -23, (rms, pull)


@pytest.mark.parametrize("d,E,k,T", [(1024, 8, 2, 512), (2048, 16, 4, 600), (512, 8, 2, 1000)])
def test_router_of_many_tokens_sums_like_fp32(d, E, k, T):
    """bf16 rows: products are exact in fp32, and fp32 multiply-adds with the same number of additions in a row leave
    1.3 * 2^-24 to 1.6 * 2^-24 of the probabilities (measured: 512 to 2048 features); sums cut over 64 products 1.7 to 2.1."""
    sh = shape(d, 64, E=E, k=k)
    lay, t, host = U.build(sh, T)
    _, _, probs = lay.route(t["x"], want_probs=True)
    rms, _ = error_against_64_bits(probs.cpu().numpy().astype("float64"), O.route(host["x"], host["w_router"], None, k)[1])
    assert rms <= (1.5 if E == 8 else 1.8) * 2.0 ** -24, rms / 2.0 ** -24


@pytest.mark.parametrize("r,T,k", [(0, 40, 2), (0, 100, 2), (64, 5, 2), (64, 16, 4), (64, 40, 2)])
def test_router_weights_written_by_the_call_before(r, T, k):
    """The kernel in front of a layer in the stream may be what writes its w_router, and may let its successor start early (as this
    library's do): here another layer's output is that matrix.  Nothing of it may be read before it is complete."""
    writer, tw, _ = U.build(W.WEARABLE, 8)
    lay, t, _ = U.build(shape(1024, 1024, k=k, r=r), T)
    matrix = t["w_router"].view(8, 1024)             # [d][E] = [1024][8], as the writer's [T][d]
    out, want = [], []
    for step in range(12):
        xw = W.make_x(W.WEARABLE, 8, device="cuda", step=step)
        writer.forward(xw, y=matrix)
        out.append(lay.forward(t["x"]))
        torch.cuda.synchronize()
        want.append(lay.forward(t["x"]))
        torch.cuda.synchronize()
    assert lay.check() == 0 and writer.check() == 0
    assert all(torch.equal(a, b) for a, b in zip(out, want))
    assert not torch.equal(want[0], want[1])         # (the matrix does change)
