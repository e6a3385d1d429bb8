"""The prompt attention kernels against the oracle on the queries and caches they consumed, at the edges of their tiles."""
import numpy as np
import pytest

from oracle import ats_oracle as O
from paper_2607_10183_b200 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu
MB = 1 << 20


# One or two key blocks of 128 and their edges, one to three query blocks, chunks that start inside a block; groups of one,
# two, three (odd: two token blocks of one head share a CTA) and eight heads; a cache that ends with the context, and one
# that goes on with Inf and NaN (which no output may see).
@pytest.mark.parametrize("T,pos0,nq,nkv,d", [(130, 0, 2, 1, 64), (129, 1, 2, 2, 128), (256, 0, 4, 2, 128), (129, 127, 3, 1, 128),
                                             (256, 128, 8, 1, 64), (257, 3, 6, 2, 64), (300, 200, 8, 1, 128), (385, 640, 1, 1, 128)])
@pytest.mark.parametrize("spare", [0, 70])
def test_prompt_attention_matches_oracle(T, pos0, nq, nkv, d, spare):
    import torch
    from paper_2607_10183_b200 import binding as B
    shape = W.DenseShape(hidden=64, n_q_heads=nq, n_kv_heads=nkv, head_dim=d, ffn=64)
    cap = pos0 + T + spare
    L = W.dense_layer(77, 0, shape)
    probe = B.layer_desc(hidden=shape.hidden, ffn=shape.ffn, wq=0, n_q_heads=nq, n_kv_heads=nkv, head_dim=d, kv_capacity=cap)
    ws = B.workspace_bytes(probe, T) + MB
    ctx = B.Context(ws + H.dense_layer_bytes(shape) + MB, workspace_bytes=ws)
    desc, ids = H.register_dense_layer(ctx, L, 0, cap)
    ctx.set_placement([(ids[n], -1, B.ATS_GPU) for n in H.ROLE_NAME.values()])
    kc, vc = W.kv_cache(77, 0, nkv, cap, d, pos0)
    kc[:, pos0 + T:], vc[:, pos0 + T:] = np.nan, np.inf
    kd, vd = H.to_dev(kc), H.to_dev(vc)
    x = W.activations(77, 0, (T, shape.hidden))
    y = torch.empty((T, shape.hidden), dtype=torch.float16, device="cuda")
    ctx.layer_prefill(desc, H.to_dev(x), y, kd, vd, pos0, T)
    ctx.sync()
    q, a = (ctx.debug_prefill_buffer(desc, T, i).astype(np.float64) for i in (2, 3))
    kg, vg = kd.cpu().numpy(), vd.cpu().numpy()
    ctx.close()
    want = np.stack([O.attention_one(q[i].reshape(nq, d), kg, vg, pos0 + i + 1).reshape(-1) for i in range(T)])
    H.assert_close(a, O.rn16(want), what="attention")


# Contexts of six blocks and more, whose tiles take the even and the odd blocks: six, seven, eight and eleven of them, last blocks that the first
# rows do not see, a second token block with one block more than the first.
@pytest.mark.parametrize("T,pos0,nq,nkv,d", [(129, 639, 2, 1, 64), (130, 700, 3, 1, 128), (200, 701, 6, 2, 64), (130, 1151, 4, 2, 128), (260, 1020, 8, 1, 128)])
@pytest.mark.parametrize("spare", [0, 70])
def test_prompt_attention_over_even_and_odd_blocks(T, pos0, nq, nkv, d, spare):
    test_prompt_attention_matches_oracle(T, pos0, nq, nkv, d, spare)
