"""The split merge at the sizes where its kernels change over: the splits that
fill 5, 10 or 16 rows a thread and one more, and row counts on both sides of
one CTA per SM, two, and the per-row kernel.  Against the fp64 oracle."""
import math

import pytest
import torch

import paper_2609_17475_gb300 as jf
from oracle import attention as OT
from tests.cases import assert_attention_close, bits, make_case

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _run(case, splits):
    pool = jf.KVPool.allocate(case.num_pages, case.P, case.Hkv, case.D, device=DEV, fill=None)
    ref_pool = case.oracle_pool()
    pool.data.copy_(torch.from_numpy(ref_pool))
    B = len(case.ctx)
    out = torch.full((B, case.Hq, case.D), float("nan"), dtype=torch.bfloat16, device=DEV)
    ws = jf.decode_workspace(B, case.Hq, case.Hkv, case.D, splits, device=DEV)
    ws[256:] = 0xFF    # NaN partials: rows past the split plan must never be used
    jf.jf_paged_decode_attn(pool, case.page_table.to(DEV),
                            torch.tensor(case.ctx, dtype=torch.int32, device=DEV), case.q.to(DEV),
                            1 / math.sqrt(case.D), out, ws, splits)
    torch.cuda.synchronize()
    assert jf.workspace_status(ws) == 0
    ref = OT.paged_decode(ref_pool, case.layout, case.page_table.numpy(), case.ctx,
                          bits(case.q), 1 / math.sqrt(case.D))
    assert_attention_close(out, ref)


@pytest.mark.parametrize("splits", [39, 40, 41, 80, 81, 128, 129])
def test_decode_merge_split_counts(splits):
    """One KV head: up to 152 splits of 512 positions or more each."""
    _run(make_case(splits, 2, 1, 128, 256, [splits * 512 - 3]), splits)


@pytest.mark.parametrize("D,B", [(128, 1), (256, 4), (256, 5), (256, 9), (256, 10), (128, 19),
                                 (128, 20)])
def test_decode_merge_row_counts(D, B):
    """8 query heads: up to 152 CTAs of 64 columns one per SM, up to 304 two, more
    rows one CTA each (152 SMs)."""
    _run(make_case(D + B, 8, 2, D, 64, [600 + 37 * b for b in range(B)]), 4)


@pytest.mark.parametrize("D,B", [(256, 18), (256, 19), (256, 20), (256, 38), (256, 39), (128, 21),
                                 (128, 38), (128, 39)])
def test_decode_merge_row_counts_past_two_per_sm(D, B):
    """8 query heads: slices with four and eight CTAs on an SM up to 304 rows, then
    a CTA per row (152 SMs); some requests empty."""
    _run(make_case(D + B, 8, 2, D, 64, [0 if b % 7 == 3 else 150 + 41 * b for b in range(B)]), 4)


def test_verify_merge_over_several_ctas_per_sm():
    """Three tokens of 5 requests: 360 rows of a verifier's batch, past the slices'
    rows, and 4 requests' 288 within."""
    for B in (4, 5):
        case = make_case(B, 24, 4, 256, 64, [400 + 111 * b for b in range(B)])
        pool = jf.KVPool.allocate(case.num_pages, case.P, case.Hkv, case.D, device=DEV, fill=None)
        ref_pool = case.oracle_pool()
        pool.data.copy_(torch.from_numpy(ref_pool))
        L = 3
        q = torch.randn(B, L, 24, 256, generator=torch.Generator().manual_seed(B)).to(torch.bfloat16)
        out = torch.full(q.shape, float("nan"), dtype=torch.bfloat16, device=DEV)
        ws = jf.verify_workspace(B, L, 24, 4, 256, 6, device=DEV)
        ws[256:] = 0xFF
        jf.jf_paged_verify_attn(pool, case.page_table.to(DEV),
                                torch.tensor(case.ctx, dtype=torch.int32, device=DEV), q.to(DEV),
                                1 / 16, out, ws, 6)
        torch.cuda.synchronize()
        assert jf.workspace_status(ws) == 0
        for b, c in enumerate(case.ctx):
            ref = OT.prefill_chunk(ref_pool, case.layout, case.page_table[b].numpy(), bits(q[b]),
                                   c - L, 1 / 16)
            assert_attention_close(out[b], ref)
