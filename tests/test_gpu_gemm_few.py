"""The GEMM of few tokens at the edges of its tiles, clusters and chains, against 64-bit sums of the oracle's weights."""
import numpy as np
import pytest

from oracle import ats_oracle as O
from paper_2607_10183_b200 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu
MB = 1 << 20


# Tiles of 16 to 128 tokens, several of them, the last one lower; one block of 128 features and its neighbours, two, whole waves of them; rows of
# y that are not 16-byte aligned.  Tiles shared by two to six CTAs, with one, two and four accumulators to a half (4096 x 4096, 704 x 4096,
# 2048 x 5632, 1536 x 8192, 5120 x 5120, 512 x 512: more CTAs than some have tokens for); sums that are handed over (6144 x 4096, 4096 x 14336).
@pytest.mark.parametrize("fmt", ["q4", "mxfp4"])
@pytest.mark.parametrize("N,K,T", [(1, 256, 9), (127, 256, 16), (129, 512, 17), (255, 768, 48), (257, 1280, 64), (300, 1024, 65), (513, 256, 129), (1000, 1280, 33),
                                   (9600, 512, 12), (28672, 512, 77), (19200, 768, 128), (512, 512, 15), (4096, 4096, 16), (4095, 4096, 77), (704, 4096, 40),
                                   (2048, 5632, 31), (2048, 5632, 112), (1536, 8192, 100), (5120, 5120, 77), (6144, 4096, 77), (6141, 4096, 300), (6144, 4096, 512),
                                   (4096, 14336, 77), (4096, 14336, 300),
                                   # k that end within a unit, a chunk of 64 or half of one; rows of scales at 2, 4 and 8-byte boundaries
                                   (1, 32, 9), (129, 96, 33), (300, 288, 65), (513, 2080, 100), (200, 4128, 70), (2048, 2880, 77), (2047, 2912, 16), (19200, 416, 60),
                                   (5120, 2880, 300), (2880, 5664, 40), (2880, 1408, 500)])
def test_gemm_of_few_tokens_matches_oracle(fmt, N, K, T):
    import torch
    from paper_2607_10183_b200 import binding as B
    packed, scales = (W.q4_packed if fmt == "q4" else W.mxfp4_packed)(101, 0, W.ROLE_UP, N, K)
    ws = 8 * T * N * 4 + 2 * MB
    ctx = B.Context(ws + W.q4_bytes(N, K) + 2 * MB, workspace_bytes=ws)
    tid = ctx.register_q4(packed, scales)
    ctx.set_placement([(tid, -1, B.ATS_GPU)])
    x = H.to_dev(W.activations(101, 0, (T, K)))
    outs = []
    for _ in range(3):
        y = torch.full((T + 1, N), 7.0, dtype=torch.float16, device="cuda")
        ctx.linear(tid, x, y, T)
        ctx.sync()
        outs.append(y)
    assert ctx.stats().kernel_launches == 3
    ctx.close()
    w = torch.from_numpy(O.dequantize(packed, scales, O.WEIGHT_F16).astype(np.float32)).cuda().double()
    H.assert_close(outs[0][:T].cpu().numpy(), (x.double() @ w.t()).cpu().numpy(), what=f"{fmt} {N}x{K} T={T}")
    assert torch.all(outs[0][T] == 7.0)
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])


# Gate and up side by side with SwiGLU, and a down projection with the residual, in every way the sums go: whole tiles, clusters, several
# accumulators.  act = rn16(silu(g) u) and y = rn16(x + d), bit for bit, with the g, u and d that are stored beside them.
@pytest.mark.parametrize("fmt,Hd,F,T", [("q4", 4096, 4096, 16), ("mxfp4", 2048, 5632, 77), ("q4", 512, 256, 9), ("mxfp4", 1024, 2816, 100), ("q4", 5120, 1000, 40), ("q4", 2048, 12032, 130), ("mxfp4", 2880, 1440, 60), ("q4", 1536, 4128, 20)])
def test_swiglu_and_residual_of_few_tokens(fmt, Hd, F, T):
    import torch
    from paper_2607_10183_b200 import binding as B
    F = F // 32 * 32
    pack = W.q4_packed if fmt == "q4" else W.mxfp4_packed
    mats = [pack(102, 0, role, n, k) for role, n, k in ((W.ROLE_GATE, F, Hd), (W.ROLE_UP, F, Hd), (W.ROLE_DOWN, Hd, F))]
    x = W.activations(102, 0, (T, Hd))
    ws = B.workspace_bytes(B.layer_desc(hidden=Hd, ffn=F, w_gate=0, w_up=0, w_down=0), T)
    ctx = B.Context(ws + 3 * Hd * F + 4 * MB, workspace_bytes=ws)
    ids = dict(ffn_norm=ctx.register_f16(W.norm_gain(102, 0, W.ROLE_FFN_NORM, Hd)))
    ids.update(zip(("w_gate", "w_up", "w_down"), (ctx.register_q4(*m) for m in mats)))
    ctx.set_placement([(ids[n], -1, B.ATS_GPU) for n in ("w_gate", "w_up", "w_down")])
    desc = B.layer_desc(hidden=Hd, ffn=F, **ids)
    y = torch.empty((T, Hd), dtype=torch.float16, device="cuda")
    outs = []
    for _ in range(2):
        ctx.layer_prefill(desc, H.to_dev(x), y, None, None, 0, T)
        ctx.sync()
        outs.append(y.cpu().numpy())
    h2, gu, act, d = (ctx.debug_prefill_buffer(desc, T, i) for i in (6, 7, 8, 9))
    ctx.close()
    dev = lambda a: torch.from_numpy(np.array(a)).cuda()  # noqa: E731
    w = [dev(O.dequantize(*m, O.WEIGHT_F16).astype(np.float32)).double() for m in mats]
    for i in range(2):
        H.assert_close(gu[:, i * F:(i + 1) * F], (dev(h2).double() @ w[i].t()).cpu().numpy(), what=f"{fmt} {'up' if i else 'gate'} T={T}")
    g, u = gu[:, :F].astype(np.float64), gu[:, F:].astype(np.float64)
    H.assert_close(act, g / (1 + np.exp(-g)) * u, what=f"{fmt} act T={T}")
    H.assert_close(d, (dev(act).double() @ w[2].t()).cpu().numpy(), what=f"{fmt} down T={T}")
    assert np.array_equal(outs[0].view(np.uint16), (x.astype(np.float32) + d.astype(np.float32)).astype(np.float16).view(np.uint16))
    assert np.array_equal(outs[0].view(np.uint16), outs[1].view(np.uint16))


# Routed experts, blocks of rows of every height, experts without rows, one expert with most of them: the bits of the kernel that the host
# sorts for (one chain per sum in both).
@pytest.mark.parametrize("fmt", ["q4", "mxfp4"])
@pytest.mark.parametrize("E,k,T,F,skew", [(16, 4, 1, 256, 0.0), (24, 2, 333, 256, 0.0), (40, 3, 129, 512, 8.0), (64, 8, 500, 256, 0.0), (8, 2, 200, 768, 4.0), (16, 4, 90, 1440, 0.0), (32, 2, 257, 96, 2.0)])
def test_experts_of_few_rows_have_the_bits_of_the_host_sort(fmt, E, k, T, F, skew):
    import torch
    from paper_2607_10183_b200 import binding as B
    Hd = 512
    rng = np.random.default_rng(11)
    router = (rng.standard_normal((Hd, E)) * 0.02).astype(np.float16)
    x = (rng.standard_normal((T, Hd)) + 0.5).astype(np.float16)
    router[:, 3] += np.float16(skew * 0.01)

    def weight(n, kk):
        codes = rng.integers(0, 256, (E, n, kk // 2), dtype=np.uint8)
        if fmt == "mxfp4":
            return codes, rng.integers(119, 124, (E, n, kk // 32), dtype=np.uint8)
        return codes, np.abs(rng.standard_normal((E, n, kk // 32)) * 0.02).astype(np.float16)

    mats = [weight(n, kk) for n, kk in ((F, Hd), (F, Hd), (Hd, F))]
    outs = []
    for flags in (0, B.ATS_FLAG_NO_GEMM_PAIR):
        ws = B.workspace_bytes(B.layer_desc(hidden=Hd, ffn=F, n_experts=E, top_k=k, w_gate=0, w_up=0, w_down=0), T)
        ctx = B.Context(ws + 3 * E * F * Hd + 4 * MB, workspace_bytes=ws, flags=flags)
        ids = dict(ffn_norm=ctx.register_f16(np.ones(Hd, np.float16)), router=ctx.register_f16(router))
        ids.update(zip(("w_gate", "w_up", "w_down"), (ctx.register_q4(*m) for m in mats)))
        ctx.set_placement([(ids[n], e, B.ATS_GPU) for n in ("w_gate", "w_up", "w_down") for e in range(E)])
        y = torch.empty((T, Hd), dtype=torch.float16, device="cuda")
        ctx.layer_prefill(B.layer_desc(hidden=Hd, ffn=F, n_experts=E, top_k=k, **ids), H.to_dev(x), y, None, None, 0, T)
        ctx.sync()
        outs.append(y.cpu().numpy())
        ctx.close()
    assert np.all(np.isfinite(outs[0].astype(np.float64)))
    assert np.array_equal(outs[0].view(np.uint16), outs[1].view(np.uint16))
