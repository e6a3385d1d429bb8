"""The fp16 GEMV of two to eight rows in both of its forms."""
import numpy as np
import pytest

from paper_2607_10183_b200 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu


# CTAs for less than a wave, for two waves of one form and one of the other, for several; an odd number of rows, K that ends within a part.
@pytest.mark.parametrize("N,K", [(96, 2048), (777, 2440), (1024, 8192), (2500, 1000)])
@pytest.mark.parametrize("M", [2, 3, 4, 5, 6, 7, 8])
def test_rows_match_64_bit_sums(N, K, M):
    import torch
    from paper_2607_10183_b200 import binding as B
    w = W.w16_matrix(111, 0, W.ROLE_UP, N, K)
    ctx = B.Context(2 * N * K + (2 << 20), workspace_bytes=65536)
    tid = ctx.register_w16(w)
    ctx.set_placement([(tid, -1, B.ATS_GPU)])
    x = H.to_dev(W.activations(111, 0, (M, K)))
    y = torch.full((M + 1, N), 7.0, dtype=torch.float16, device="cuda")
    ctx.linear(tid, x, y, M)
    ctx.sync()
    ctx.close()
    want = x.double() @ torch.from_numpy(w).cuda().double().t()
    H.assert_close(y[:M].cpu().numpy(), want.cpu().numpy(), what=f"{N}x{K} M={M}")
    assert torch.all(y[M] == 7.0)


# Few output rows of a long K: five rows take no longer than eight, over four matrices together.
def test_five_rows_take_no_longer_than_eight():
    import torch
    from paper_2607_10183_b200 import binding as B
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    total = {5: 0.0, 8: 0.0}
    for N, K in ((512, 16384), (500, 12000), (1024, 16384), (600, 4096)):
        ctx = B.Context(2 * N * K + (2 << 20), workspace_bytes=65536)
        tid = ctx.register_w16((np.random.default_rng(3).standard_normal((N, K)) * 0.09).astype(np.float16))
        ctx.set_placement([(tid, -1, B.ATS_GPU)])
        for M in (5, 8):
            x = H.to_dev(W.activations(112, 0, (M, K)))
            y = torch.empty((M, N), dtype=torch.float16, device="cuda")
            torch.cuda.synchronize()
            events = []
            with torch.cuda.stream(ctx.compute):
                for _ in range(60):  # every pass finds the weights in memory, not in the L2 cache
                    flush.fill_(1)
                    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    a.record()
                    ctx.linear(tid, x, y, M)
                    b.record()
                    events.append((a, b))
            torch.cuda.synchronize()
            total[M] += sum(sorted(a.elapsed_time(b) * 1e3 for a, b in events[10:])[5:35]) / 30
        ctx.close()
    print(f"five rows {total[5]:.2f} us, eight {total[8]:.2f}")
    assert total[5] <= total[8]
