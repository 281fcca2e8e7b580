"""The sliced merge holds a plan's partial rows in one batch: 40, 80 or 152 of
them, and loops past that.  Counts around 152 against the fp64 oracle, and the
time that a plan of more than 128 rows takes."""
import math

import pytest
import torch

import paper_2609_17475_gb300 as jf
from oracle import attention as OT
from tests.cases import assert_attention_close, bits, make_case
from tests.launches import device_us

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("splits", [151, 152, 153, 304])
def test_verify_merge_around_one_batch(splits):
    """One KV head, two tokens of 2 rows each: one split per 4 chunks."""
    case = make_case(splits, 2, 1, 128, 256, [splits * 128 - 5])
    ref_pool = case.oracle_pool()
    pool = jf.KVPool.allocate(case.num_pages, case.P, 1, 128, device=DEV, fill=None)
    pool.data.copy_(torch.from_numpy(ref_pool))
    q = torch.randn(1, 2, 2, 128, generator=torch.Generator().manual_seed(splits))
    q = q.to(torch.bfloat16)
    out = torch.full(q.shape, float("nan"), dtype=torch.bfloat16, device=DEV)
    ws = jf.verify_workspace(1, 2, 2, 1, 128, splits, device=DEV)
    ws[256:] = 0xFF    # NaN partials: rows past the plan must never be used
    jf.jf_paged_verify_attn(pool, case.page_table.to(DEV),
                            torch.tensor(case.ctx, dtype=torch.int32, device=DEV), q.to(DEV),
                            1 / math.sqrt(128), out, ws, splits)
    torch.cuda.synchronize()
    assert jf.workspace_status(ws) == 0
    ref = OT.prefill_chunk(ref_pool, case.layout, case.page_table[0].numpy(), bits(q[0]),
                           case.ctx[0] - 2, 1 / math.sqrt(128))
    assert_attention_close(out[0], ref)


def test_a_plan_of_133_splits_takes_one_batch():
    """4/1/256: 17,000 positions in 133 splits take 1.21 times the time of 12,000 in
    94 where they are merged in two batches, 1.04 now."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms < 133:
        pytest.skip("133 splits need as many SMs")
    times = []
    for ctx in (12000, 17000):
        pages = -(-ctx // 64)
        pool = jf.KVPool.allocate(pages, 64, 1, 256, device=DEV)
        table = torch.arange(pages, dtype=torch.int32, device=DEV).view(1, -1)
        lens = torch.tensor([ctx], dtype=torch.int32, device=DEV)
        q = torch.randn(1, 4, 256, device=DEV).to(torch.bfloat16)
        out = torch.empty_like(q)
        ws = jf.decode_workspace(1, 4, 1, 256, sms, device=DEV)
        times.append(device_us(lambda: jf.jf_paged_decode_attn(pool, table, lens, q, 0.1, out, ws,
                                                               sms)))
    assert times[1] <= 1.12 * times[0], times
