"""TQ4 prefill: query rows whose fp16 form needs a power of two of its own, beside
rows that do not, with one history range and with several.  Keys are scaled down so
that the large rows' logits are ordinary.  Against the fp64 oracle."""
import math

import pytest
import torch

import paper_2609_17475_gb300 as jf
from oracle import attention as OT
from paper_2609_17475_gb300 import synth
from tests.cases import assert_attention_close, bits, make_case
from tests.test_gpu_tq4 import DEV, oracle_pool, pool_from_numpy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("big", ["none", "one", "third", "all"])
@pytest.mark.parametrize("Hq,Hkv,D,q_start,C,splits", [
    (8, 2, 128, 90, 33, 1),
    (24, 4, 256, 400, 45, 3),
    (4, 4, 256, 7, 1, 1),
])
def test_tq4_prefill_large_query_rows(Hq, Hkv, D, q_start, C, splits, big):
    case = make_case(D + C, Hq, Hkv, D, 64, [q_start + C])
    case.k = (case.k.float() * 2.0 ** -16).to(torch.bfloat16)
    lay, ref_pool = oracle_pool(case)
    pool = pool_from_numpy(case, ref_pool)
    q = synth.normal_bf16(synth.generator(C), (C, Hq, D))
    rows = {"none": [], "one": [C - 1], "third": list(range(0, C, 3)), "all": list(range(C))}[big]
    q[rows] = (q[rows].float() * 2.0 ** 17).to(torch.bfloat16)
    out = torch.full(q.shape, float("nan"), dtype=torch.bfloat16, device=DEV)
    ws = jf.prefill_batch_workspace(C, Hq, D, splits, device=DEV, format=jf.JF_FMT_TQ4)
    jf.jf_prefill_batch_attn(pool, case.page_table.to(DEV), [q_start], [C], q.to(DEV),
                             1 / math.sqrt(D), True, out, ws, num_splits=splits)
    torch.cuda.synchronize()
    assert jf.workspace_status(ws) == 0
    ref = OT.prefill_chunk(ref_pool, lay, case.page_table[0].numpy(), bits(q), q_start,
                           1 / math.sqrt(D))
    assert_attention_close(out, ref)
