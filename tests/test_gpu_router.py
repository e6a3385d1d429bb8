"""The router for many tokens: the bits of the router for few, whatever the tokens of a cluster, the ranges and the chains."""
import numpy as np
import pytest

from tests import helpers as H

pytestmark = pytest.mark.gpu


# One and several rounds of clusters, a last cluster with few tokens, chains of unequal length (2880 rows, 64 experts), one row to a chain (512 x 16),
# more than 128 experts (a shorter block of tokens where shared memory is full); equal logits and a NaN among the tokens.
@pytest.mark.parametrize("hidden,E,k,M", [(2048, 128, 8, 96), (2048, 128, 8, 513), (2880, 64, 4, 130), (512, 16, 2, 700), (1024, 32, 4, 2000), (1024, 256, 8, 250),
                                          (3072, 256, 6, 97), (4096, 64, 4, 1100), (2048, 128, 8, 56), (2880, 64, 4, 121), (2048, 128, 8, 250)])
def test_router_of_many_tokens_has_the_bits_of_the_router_of_few(hidden, E, k, M):
    import torch
    from paper_2607_10183_b200 import binding as B
    rng = np.random.default_rng(hidden + E + M)
    wr = (rng.standard_normal((hidden, E)) * 0.02).astype(np.float16)
    wr[:, 5] = wr[:, 3]  # equal logits: the lower index first
    ctx = B.Context(4 * hidden * E + (8 << 20), workspace_bytes=1 << 20)
    rid = ctx.register_f16(wr)
    ctx.set_placement([])
    h = H.to_dev(rng.standard_normal((M, hidden)).astype(np.float16))
    h[M - 2, 7] = float("nan")

    def route(lo, hi):
        ids = torch.full((hi - lo, k), -1, dtype=torch.int32, device="cuda")
        gates = torch.zeros((hi - lo, k), dtype=torch.float32, device="cuda")
        ctx.route_topk(rid, h[lo:hi].contiguous(), hi - lo, k, ids, gates)
        ctx.sync()
        return ids, gates.view(torch.int32)

    ids, gates = route(0, M)
    parts = [route(lo, min(M, lo + 48)) for lo in range(0, M, 48)]
    assert torch.equal(ids, torch.cat([p[0] for p in parts]))
    assert torch.equal(gates, torch.cat([p[1] for p in parts]))
    ctx.close()


# The streamed form: matrices whose eighth does not fit beside the tokens (256 experts of 4096 and 5120, 512, 1024) or leaves room for too few (128 of
# 4096), the fewest tokens it takes and one less, a last CTA of one to three tokens, two waves.
@pytest.mark.parametrize("hidden,E,k,M", [(2048, 512, 8, 128), (2048, 512, 8, 127), (1024, 1024, 32, 131), (4096, 256, 8, 186), (4096, 256, 8, 183), (5120, 256, 8, 613),
                                          (4096, 128, 8, 511)])
def test_streamed_router_has_the_bits_of_the_router_of_few(hidden, E, k, M):
    test_router_of_many_tokens_has_the_bits_of_the_router_of_few(hidden, E, k, M)


# A wave of the streamed form takes as long for 512 tokens as for 200 (25 % are left for noise), a cluster per token more than twice as long.
@pytest.mark.parametrize("hidden,E", [(2048, 512), (1024, 1024), (4096, 256), (5120, 256)])
def test_a_wave_of_the_streamed_router_takes_as_long_whatever_the_tokens(hidden, E):
    import torch
    from paper_2607_10183_b200 import binding as B
    rng = np.random.default_rng(5)
    ctx = B.Context(4 * hidden * E + (8 << 20), workspace_bytes=1 << 20)
    rid = ctx.register_f16((rng.standard_normal((hidden, E)) * 0.02).astype(np.float16))
    ctx.set_placement([])
    times = []
    for M in (200, 512):
        h = H.to_dev(rng.standard_normal((M, hidden)).astype(np.float16))
        ids = torch.empty((M, 8), dtype=torch.int32, device="cuda")
        gates = torch.empty((M, 8), dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        passes = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(ctx.compute)
            for _ in range(10):
                ctx.route_topk(rid, h, M, 8, ids, gates)
            b.record(ctx.compute)
            b.synchronize()
            passes.append(a.elapsed_time(b) * 100)
        times.append(sorted(passes[2:])[5])
    ctx.close()
    print(f"{hidden} x {E}: {times[0]:.1f} us for 200 tokens, {times[1]:.1f} for 512")
    assert times[1] <= 1.25 * times[0]


# Numbers of experts that are no power of two (chains of unequal length, lanes without an expert in the selection), several tokens more than clusters
# take evenly; the streamed form.
@pytest.mark.parametrize("hidden,E,k,M", [(512, 56, 4, 97), (1024, 72, 8, 131), (512, 168, 8, 250), (2048, 240, 32, 99), (512, 248, 1, 77)])
def test_router_of_many_tokens_and_any_number_of_experts(hidden, E, k, M):
    test_router_of_many_tokens_has_the_bits_of_the_router_of_few(hidden, E, k, M)


# Gates of the softmax over all experts: a layer's outputs have the bits of the layer over 48 tokens at a time (a cluster per token), and what the
# experts add is the renormalised layer's times the selected experts' share of the softmax.
@pytest.mark.parametrize("E,k,M", [(56, 4, 97), (72, 8, 131), (128, 8, 200), (240, 8, 99), (512, 8, 130)])
def test_gates_that_are_not_renormalised(E, k, M):
    import torch
    from paper_2607_10183_b200 import binding as B
    Hd, F = 512, 96
    rng = np.random.default_rng(E)
    router = (rng.standard_normal((Hd, E)) * 0.05).astype(np.float16)
    x = rng.standard_normal((M, Hd)).astype(np.float16)
    mats = [(rng.integers(0, 256, (E, n, kk // 2), dtype=np.uint8), np.abs(rng.standard_normal((E, n, kk // 32)) * 0.02).astype(np.float16))
            for n, kk in ((F, Hd), (F, Hd), (Hd, F))]
    ws = B.workspace_bytes(B.layer_desc(hidden=Hd, ffn=F, n_experts=E, top_k=k, w_gate=0, w_up=0, w_down=0), M)
    ctx = B.Context(ws + 3 * E * F * Hd + (8 << 20), workspace_bytes=ws)
    ids = dict(ffn_norm=ctx.register_f16(np.ones(Hd, np.float16)), router=ctx.register_f16(router))
    ids.update(zip(("w_gate", "w_up", "w_down"), (ctx.register_q4(*m) for m in mats)))
    ctx.set_placement([(ids[n], e, B.ATS_GPU) for n in ("w_gate", "w_up", "w_down") for e in range(E)])

    def layer(flags, lo, hi):
        desc = B.layer_desc(hidden=Hd, ffn=F, n_experts=E, top_k=k, flags=flags, **ids)
        y = torch.empty((hi - lo, Hd), dtype=torch.float16, device="cuda")
        ctx.layer_prefill(desc, H.to_dev(x[lo:hi]), y, None, None, 0, hi - lo)
        ctx.sync()
        return y.cpu().numpy()

    plain, whole = layer(0, 0, M), layer(B.ATS_LAYER_NO_TOPK_RENORM, 0, M)
    parts = np.concatenate([layer(B.ATS_LAYER_NO_TOPK_RENORM, lo, min(M, lo + 48)) for lo in range(0, M, 48)])
    ctx.close()
    assert np.array_equal(whole.view(np.uint16), parts.view(np.uint16))
    x64 = x.astype(np.float64)
    h = (x64 / np.sqrt((x64 ** 2).mean(1, keepdims=True) + 1e-5)).astype(np.float16).astype(np.float64)
    p = np.exp(h @ router.astype(np.float64))
    share = -np.sort(-p, axis=1)[:, :k].sum(1, keepdims=True) / p.sum(1, keepdims=True)
    want = x64 + share * (plain.astype(np.float64) - x64)
    # half a unit of fp16 (2^-11) for each of the two layers' outputs, the share of the softmax to 1e-3 (h's rounding)
    assert np.all(np.abs(whole - want) <= 2.0 ** -11 * (np.abs(plain) + np.abs(whole)) + 1e-3 * np.abs(want - x64) + 1e-6)
