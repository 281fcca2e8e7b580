"""TQ4 batches under the span plan: pieces that begin or end inside a request,
cover several, or only a request's first places; empty and one-position
requests; decode and the fused step.  Against the fp64 oracle."""
import math

import pytest
import torch

import paper_2609_17475_gb300 as jf
from oracle import attention as OT
from tests.cases import assert_attention_close, bits, make_case
from tests.test_gpu_tq4 import DEV, gpu_decode, oracle_pool, pool_from_numpy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,D,P,ctx,splits", [
    (6, 1, 256, 64, [0, 1, 33, 700, 5000, 0], 40),     # many pieces of 16 places
    (6, 1, 256, 256, [3000, 3000], 2),                 # few workspace rows: 3 pieces
    (8, 2, 128, 128, [31, 32, 33, 64, 2047, 2048], 6),
    (12, 4, 128, 64, [512 * i + 7 for i in range(9)], 3),
    (4, 4, 256, 64, [9000, 5], 30),
])
def test_tq4_batch_spans_match_oracle(Hq, Hkv, D, P, ctx, splits):
    case = make_case(sum(ctx) + D, Hq, Hkv, D, P, ctx)
    lay, ref_pool = oracle_pool(case)
    pool = pool_from_numpy(case, ref_pool)
    out = gpu_decode(case, pool, splits)
    ref = OT.paged_decode(ref_pool, lay, case.page_table.numpy(), ctx, bits(case.q),
                          1 / math.sqrt(D))
    assert_attention_close(out, ref)
    for b, c in enumerate(ctx):
        if c == 0:
            assert not out[b].any()


@pytest.mark.parametrize("D,P,ctx,splits", [(256, 64, [1, 32, 33, 2500, 0, 777], 30),
                                            (128, 128, [4096, 1, 63], 50)])
def test_tq4_batch_span_step_equals_append_then_decode(D, P, ctx, splits):
    case = make_case(D + len(ctx), 8, 2, D, P, ctx)
    B = len(ctx)
    _, ref_pool = oracle_pool(case)
    g = torch.Generator().manual_seed(D)
    k, v = (torch.randn(B, 2, D, generator=g).to(torch.bfloat16).to(DEV) for _ in range(2))
    pt = case.page_table.to(DEV)
    lens = torch.tensor(ctx, dtype=torch.int32, device=DEV)
    a, b = pool_from_numpy(case, ref_pool), pool_from_numpy(case, ref_pool)
    live = [i for i, c in enumerate(ctx) if c > 0]
    jf.jf_kv_quantize_append(a, pt, torch.tensor(live, dtype=torch.int32, device=DEV),
                             lens[live] - 1, k[live].contiguous(), v[live].contiguous())
    outs = []
    for pool in (a, b):
        out = torch.full((B, 8, D), float("nan"), dtype=torch.bfloat16, device=DEV)
        ws = jf.decode_workspace(B, 8, 2, D, splits, device=DEV)
        args = (case.q.to(DEV), 1 / math.sqrt(D), out, ws, splits)
        if pool is a:
            jf.jf_paged_decode_attn(pool, pt, lens, *args)
        else:
            jf.jf_paged_decode_append_attn(pool, pt, lens, k, v, *args)
        torch.cuda.synchronize()
        assert jf.workspace_status(ws) == 0
        outs.append(out)
    assert torch.equal(a.data, b.data)
    assert torch.equal(outs[0], outs[1])
