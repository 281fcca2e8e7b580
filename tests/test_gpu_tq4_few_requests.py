"""TQ4 batches on both sides of the line between whole-request pieces and spans
(19 SMs for each request and KV head): empty, one-position and unequal requests,
few workspace rows, and the fused step.  Against the fp64 oracle and the append
followed by the decode."""
import math

import pytest
import torch

import paper_2609_17475_gb300 as jf
from oracle import attention as OT
from tests.cases import assert_attention_close, bits, make_case
from tests.test_gpu_tq4 import DEV, gpu_decode, oracle_pool, pool_from_numpy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,D,P,ctx,splits", [
    (6, 1, 256, 64, [3000, 1], 78),                                      # 2 to 8 requests: pieces
    (6, 1, 256, 128, [0, 1, 33, 700, 2500, 0, 64, 31], 21),
    (6, 1, 256, 64, [0, 1, 33, 700, 2500, 0, 64, 31, 5], 19),            # 9: spans
    (8, 2, 128, 256, [2047, 0, 2048, 1], 21),
    (8, 2, 128, 64, [2047, 0, 2048, 1, 90], 18),
    (8, 2, 128, 64, [4000, 33, 900, 1], 2),                              # few workspace rows
    (24, 4, 256, 64, [0, 900], 21),
    (32, 8, 128, 64, [1500, 40], 12),
])
def test_tq4_few_requests_match_oracle(Hq, Hkv, D, P, ctx, splits):
    case = make_case(sum(ctx) + D, Hq, Hkv, D, P, ctx)
    lay, ref_pool = oracle_pool(case)
    pool = pool_from_numpy(case, ref_pool)
    out = gpu_decode(case, pool, splits)
    ref = OT.paged_decode(ref_pool, lay, case.page_table.numpy(), ctx, bits(case.q),
                          1 / math.sqrt(D))
    live = [b for b, c in enumerate(ctx) if c > 0]
    if live:
        assert_attention_close(out[live], ref[live])
    for b, c in enumerate(ctx):
        if c == 0:
            assert not out[b].any()


@pytest.mark.parametrize("Hkv,D,ctx,splits", [(1, 256, [1, 32, 33, 2500, 0, 777, 64, 65], 21),
                                              (2, 128, [1500, 1, 63], 28), (4, 256, [2, 900], 2)])
def test_tq4_few_requests_step_equals_append_then_decode(Hkv, D, ctx, splits):
    case = make_case(D + len(ctx), 4 * Hkv, Hkv, D, 64, ctx)
    B = len(ctx)
    _, ref_pool = oracle_pool(case)
    g = torch.Generator().manual_seed(D)
    k, v = (torch.randn(B, Hkv, D, generator=g).to(torch.bfloat16).to(DEV) for _ in range(2))
    pt = case.page_table.to(DEV)
    lens = torch.tensor(ctx, dtype=torch.int32, device=DEV)
    a, b = pool_from_numpy(case, ref_pool), pool_from_numpy(case, ref_pool)
    live = [i for i, c in enumerate(ctx) if c > 0]
    jf.jf_kv_quantize_append(a, pt, torch.tensor(live, dtype=torch.int32, device=DEV),
                             lens[live] - 1, k[live].contiguous(), v[live].contiguous())
    outs = []
    for pool in (a, b):
        out = torch.full((B, 4 * Hkv, D), float("nan"), dtype=torch.bfloat16, device=DEV)
        ws = jf.decode_workspace(B, 4 * Hkv, Hkv, D, splits, device=DEV)
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
