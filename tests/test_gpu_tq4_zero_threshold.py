"""TQ4 codebooks with a threshold at zero or beside it, at every index: the
append's threshold table and the fused step's encoder store the oracle's bytes,
and the same ones."""
import numpy as np
import pytest
import torch

import paper_2609_17475_gb300 as jf
from oracle import tq4 as OQ
from paper_2609_17475_gb300 import synth
from tests.cases import bits, make_case

pytestmark = pytest.mark.gpu
DEV = "cuda"
Hkv, P, B = 2, 64, 48


@pytest.mark.parametrize("beside", [0, 1, -1])
@pytest.mark.parametrize("index", range(15))
@pytest.mark.parametrize("D", [128, 256])
def test_zero_threshold_at_any_index(D, index, beside):
    # thresholds 0.2 rho apart, number `index` at zero (or next to it): within
    # the table's reach of 3.9 rho on either side, more than 0.13 rho apart
    c = (0.2 * (np.arange(16) - index - 0.5) / np.sqrt(D)).astype(np.float32)
    if beside:
        c[index + 1] = np.nextafter(c[index + 1], np.float32(beside))
    t = np.float32(c[index] + c[index + 1]) * np.float32(0.5)
    assert np.sign(t) == beside and abs(t) < 2.0 ** -30
    case = make_case(D + index, 2 * Hkv, Hkv, D, P, [1] * B)
    signs = OQ.sign_vector(OQ.SEED_K, D), OQ.sign_vector(OQ.SEED_V, D)
    lay = OQ.Tq4Layout(Hkv, P, D, OQ.Codec(D, c, *signs))
    ref = OQ.new_pool(lay, case.num_pages, fill=0x33)
    OQ.append(ref, lay, case.page_table.numpy(), case.req.numpy(), case.pos.numpy(),
              bits(case.k), bits(case.v))
    codec = jf.Tq4Codec(D, synth.tq4_signs(synth.TQ4_SEED_K, D),
                        synth.tq4_signs(synth.TQ4_SEED_V, D), centroids=c)
    pools = [jf.KVPool.allocate(case.num_pages, P, Hkv, D, device=DEV, fill=0x33,
                                format=jf.JF_FMT_TQ4, codec=codec) for _ in range(2)]
    err = torch.zeros(1, dtype=torch.int32, device=DEV)
    pt, k, v = case.page_table.to(DEV), case.k.to(DEV), case.v.to(DEV)
    jf.jf_kv_quantize_append(pools[0], pt, case.req.to(DEV), case.pos.to(DEV), k, v, err)
    q = case.q.to(DEV)
    ws = jf.decode_workspace(B, 2 * Hkv, Hkv, D, 2, device=DEV)
    jf.jf_paged_decode_append_attn(pools[1], pt, torch.ones(B, dtype=torch.int32, device=DEV),
                                   k, v, q, 0.1, torch.empty_like(q), ws, 2)
    torch.cuda.synchronize()
    assert int(err.item()) == 0 and jf.workspace_status(ws) == 0
    assert np.array_equal(pools[0].data.cpu().numpy(), ref)
    assert np.array_equal(pools[1].data.cpu().numpy(), ref)
