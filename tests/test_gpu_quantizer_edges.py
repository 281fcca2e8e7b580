"""The division-free quantizer where it could differ from the IEEE rule: values
on and beside the midpoints, midpoints approached from a far smaller bias, and
scales on both sides of its range (the division takes the others).  Bytes
equal the oracle's."""
import numpy as np
import pytest
import torch

import paper_2609_17475_gb300 as jf
from tests.cases import make_case

pytestmark = pytest.mark.gpu


def _midpoints(rng, n, H, D):
    """Groups {0, 15 s, s (k + 1/2) and its bf16 neighbours}, s with few bits."""
    s = np.exp2(rng.integers(-6, 6, (n, H, D // 64, 1))) * rng.integers(1, 16, (n, H, D // 64, 1))
    k = rng.integers(0, 15, (n, H, D // 64, 64)) + 0.5
    x = torch.from_numpy((s * k).astype(np.float32)).to(torch.bfloat16)
    nudge = torch.from_numpy(rng.integers(-1, 2, x.shape).astype(np.int16))
    x = (x.view(torch.int16) + nudge).view(torch.bfloat16)
    x[..., 0] = 0.0
    x[..., 1] = torch.from_numpy((15 * s[..., 0]).astype(np.float32)).to(torch.bfloat16)
    return x.reshape(n, H, D)


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -104, 2.0 ** -97, 2.0 ** 97, 2.0 ** 104])
@pytest.mark.parametrize("kind", ["midpoints", "tiny bias", "normal"])
@pytest.mark.parametrize("Hkv,D,P,rows", [(1, 128, 64, 3), (3, 256, 128, 70)])
def test_append_quantizer_edges(Hkv, D, P, rows, kind, scale):
    rng = np.random.default_rng(rows + D)
    case = make_case(rows, Hkv, Hkv, D, P, [rows], num_pages=-(-rows // P) + 1)
    if kind != "normal":
        case.k = _midpoints(rng, rows, Hkv, D)
        case.v = _midpoints(rng, rows, Hkv, D)
    if kind == "tiny bias":   # x - bias rounds: the quotient falls beside a midpoint
        case.k[..., ::64] = -(2.0 ** -20)
        case.v[..., ::64] = 2.0 ** -24
    case.k, case.v = case.k * scale, case.v * scale
    ref = case.oracle_pool(fill=0x44)
    pool = jf.KVPool.allocate(case.num_pages, P, Hkv, D, device="cuda", fill=0x44)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    jf.jf_kv_quantize_append(pool, case.page_table.cuda(), case.req.cuda(), case.pos.cuda(),
                             case.k.cuda(), case.v.cuda(), err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert np.array_equal(pool.data.cpu().numpy(), ref)
