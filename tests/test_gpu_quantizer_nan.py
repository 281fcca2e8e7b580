"""NaN elements among finite ones of a group: they exceed no threshold, so
their code is 0, and the group's scale, bias and other codes are those of its
finite elements.  The append and the fused step store the same bytes."""
import math

import numpy as np
import pytest
import torch

import paper_2609_17475_gb300 as jf
from tests.cases import make_case

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _with_nan(x, seed):
    """(x with NaN elements, the same with each group's finite minimum there)."""
    n, H, D = x.shape
    g = x.float().reshape(n, H, D // 64, 64)
    rng = np.random.default_rng(seed)
    bad = torch.from_numpy(rng.random(g.shape) < 0.2)
    bad[..., 5] = False                                # a finite element in every group
    bad[::3] = False                                   # and groups without any NaN
    low = g.masked_fill(bad, math.inf).amin(-1, keepdim=True)
    nan = g.masked_fill(bad, math.nan).reshape(x.shape).to(torch.bfloat16)
    return nan, torch.where(bad, low, g).reshape(x.shape).to(torch.bfloat16)


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -104, 2.0 ** 104])   # the last two divide
@pytest.mark.parametrize("Hkv,D,P", [(1, 128, 64), (3, 256, 128)])
def test_nan_elements_take_code_zero(Hkv, D, P, scale):
    B = 40
    case = make_case(D, 2 * Hkv, Hkv, D, P, [1] * B)
    k, case.k = _with_nan(case.k * scale, 1)
    v, case.v = _with_nan(case.v * scale, 2)
    assert k.isnan().any() and v.isnan().any() and not case.k.isnan().any()
    ref = case.oracle_pool(fill=0x44)
    pools = [jf.KVPool.allocate(case.num_pages, P, Hkv, D, device=DEV, fill=0x44)
             for _ in range(2)]
    err = torch.zeros(1, dtype=torch.int32, device=DEV)
    pt, k, v, q = (t.to(DEV) for t in (case.page_table, k, v, case.q))
    jf.jf_kv_quantize_append(pools[0], pt, case.req.to(DEV), case.pos.to(DEV), k, v, err)
    ws = jf.decode_workspace(B, 2 * Hkv, Hkv, D, 2, device=DEV)
    jf.jf_paged_decode_append_attn(pools[1], pt, torch.ones(B, dtype=torch.int32, device=DEV),
                                   k, v, q, 0.1, torch.empty_like(q), ws, 2)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert np.array_equal(pools[0].data.cpu().numpy(), ref)
    assert np.array_equal(pools[1].data.cpu().numpy(), ref)
