"""Prefill's query rows: chunks that fill part of a CTA's 128 rows, rows whose fp16
form needs a power of two of its own beside rows that do not, against the fp64
oracle (small keys that fp16 holds exactly, so that the large rows' logits are
ordinary); and the time that a warp's rows add to a chunk."""
import math

import numpy as np
import pytest
import torch

import paper_2609_17475_gb300 as jf
from oracle import attention as OT
from paper_2609_17475_gb300 import synth
from tests.cases import assert_attention_close, bits, make_case
from tests.helpers import exact_groups, f64_to_bf16_tensor
from tests.launches import device_us

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("big", ["none", "one", "third", "all"])
@pytest.mark.parametrize("Hq,Hkv,D,q_start,C", [
    (8, 2, 128, 90, 33),      # 132 rows: a full CTA and 4 rows
    (24, 4, 256, 400, 45),
    (24, 4, 256, 0, 6),       # 36: a warp and 4 rows
    (4, 4, 256, 7, 1),        # one row
    (8, 1, 128, 64, 4),       # 32: one warp
])
def test_affine_prefill_large_query_rows(Hq, Hkv, D, q_start, C, big):
    case = make_case(D + C, Hq, Hkv, D, 64, [q_start + C])
    case.k = f64_to_bf16_tensor(exact_groups(np.random.default_rng(C), case.k.shape) * 2.0 ** -17)
    ref_pool = case.oracle_pool()
    pool = jf.KVPool.allocate(case.num_pages, case.P, Hkv, D, device=DEV)
    pool.data.copy_(torch.from_numpy(ref_pool))
    q = synth.normal_bf16(synth.generator(C), (C, Hq, D))
    rows = {"none": [], "one": [C - 1], "third": list(range(0, C, 3)), "all": list(range(C))}[big]
    q[rows] = (q[rows].float() * 2.0 ** 17).to(torch.bfloat16)
    out = torch.full(q.shape, float("nan"), dtype=torch.bfloat16, device=DEV)
    ws = jf.prefill_batch_workspace(C, Hq, D, 1, device=DEV)
    jf.jf_prefill_batch_attn(pool, case.page_table.to(DEV), [q_start], [C], q.to(DEV),
                             1 / math.sqrt(D), True, out, ws)
    torch.cuda.synchronize()
    assert jf.workspace_status(ws) == 0
    ref = OT.prefill_chunk(ref_pool, case.layout, case.page_table[0].numpy(), bits(q), q_start,
                           1 / math.sqrt(D))
    assert_attention_close(out, ref)


def _device_us(fmt, Hq, Hkv, D, C):
    codec = jf.Tq4Codec(D, [1] * D, [1] * D) if fmt == jf.JF_FMT_TQ4 else None
    pool = jf.KVPool.allocate(2, 64, Hkv, D, device=DEV, format=fmt, codec=codec)
    row = torch.zeros(2, dtype=torch.int32, device=DEV)
    q = torch.randn(C, Hq, D, device=DEV).to(torch.bfloat16)
    out = torch.empty_like(q)
    ws = jf.prefill_chunk_workspace(pool, 0, C, Hq)

    def call():
        jf.jf_prefill_chunk_attn(pool, row, q, 0, 0.1, True, out, ws)

    return device_us(call)


@pytest.mark.parametrize("fmt,C,bound", [(jf.JF_FMT_AFFINE4_G64, 8, 1.22), (jf.JF_FMT_TQ4, 20, 1.45)])
def test_short_chunks_cost_little_more_than_one_query(fmt, C, bound):
    """24/4/256 at position 0: 48 rows cost 1.36 times one query's where each row is
    read twice (1.09 now), 120 TQ4 rows 1.62 times where each waits for its own
    load (1.31 now)."""
    assert _device_us(fmt, 24, 4, 256, C) <= bound * _device_us(fmt, 24, 4, 256, 1)
