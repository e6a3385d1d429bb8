"""The sort of a prompt's (token, slot) pairs by expert, with the copy of their rows, for routings far from even."""
import numpy as np
import pytest

from tests import helpers as H
from tests.test_gpu_prefill import test_moe_prefill_sorted_on_the_device_has_the_bits_of_the_host_sort as same_bits

pytestmark = pytest.mark.gpu
MB = 1 << 20


# Runs of rows per expert: one expert with hundreds of them, all rows in one expert, more experts than four to an SM, most of them without
# rows, the most experts; a last run of one row and full ones; ids beyond the sixteen that a thread keeps.
@pytest.mark.parametrize("E,k,T,skew", [(128, 8, 513, 6.0), (264, 8, 1100, 4.0), (600, 4, 301, 6.0), (1024, 8, 70, 0.0), (8, 1, 3000, 30.0), (4, 1, 129, 0.0), (128, 8, 1024, 0.0), (128, 8, 160, 6.0), (128, 8, 161, 6.0), (32, 4, 320, 30.0)])
def test_rows_of_any_routing_have_the_bits_of_the_host_sort(E, k, T, skew):
    import torch
    from paper_2607_10183_b200 import binding as B
    same_bits(B, torch, E, k, T, skew)


# As many rows are sorted, copied and multiplied whoever gets them, and fewer weights are read where all tokens want the same experts: that may
# not take longer (15 % are left for noise).
@pytest.mark.parametrize("E,hot,T", [(128, 8, 4096), (128, 1, 8192), (512, 8, 2048)])
def test_tokens_that_want_the_same_experts_take_no_longer(E, hot, T):
    import torch
    from paper_2607_10183_b200 import binding as B
    Hd, F, k = 2048, 256, 8
    rng = np.random.default_rng(17)
    mats = [(rng.integers(0, 256, (E, n, kk // 2), dtype=np.uint8), np.abs(rng.standard_normal((E, n, kk // 32)) * 0.02).astype(np.float16))
            for n, kk in ((F, Hd), (F, Hd), (Hd, F))]
    x = H.to_dev((rng.standard_normal((T, Hd)) + 0.3).astype(np.float16))
    y = torch.empty_like(x)
    times = []
    for lift in (0.0, 0.1):
        router = (rng.standard_normal((Hd, E)) * 0.02).astype(np.float16)
        router[:, :hot] += np.float16(lift)
        ws = B.workspace_bytes(B.layer_desc(hidden=Hd, ffn=F, n_experts=E, top_k=k, w_gate=0, w_up=0, w_down=0), T)
        ctx = B.Context(ws + 3 * E * F * Hd + 8 * MB, workspace_bytes=ws)
        ids = dict(ffn_norm=ctx.register_f16(np.ones(Hd, np.float16)), router=ctx.register_f16(router))
        ids.update(zip(("w_gate", "w_up", "w_down"), (ctx.register_q4(*m) for m in mats)))
        ctx.set_placement([(ids[n], e, B.ATS_GPU) for n in ("w_gate", "w_up", "w_down") for e in range(E)])
        desc = B.layer_desc(hidden=Hd, ffn=F, n_experts=E, top_k=k, **ids)
        passes = []
        for _ in range(15):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(ctx.compute)
            ctx.layer_prefill(desc, x, y, None, None, 0, T)
            b.record(ctx.compute)
            b.synchronize()
            passes.append(a.elapsed_time(b) * 1e3)
        ctx.close()
        times.append(sorted(passes[3:])[6])
    print(f"{E} experts, {T} tokens: {times[0]:.0f} us evenly, {times[1]:.0f} us where all want the same {hot}")
    assert times[1] <= 1.15 * times[0]
