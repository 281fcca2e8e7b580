"""TQ4 append where its two kernels and their tails meet: vector counts that
leave part of a warp empty, zero vectors and out-of-range norms among others,
and codebooks on both sides of the lookup table's limits.  Bytes equal the
oracle's."""
import numpy as np
import pytest
import torch

import paper_2609_17475_gb300 as jf
from oracle import tq4 as OQ
from paper_2609_17475_gb300 import synth
from tests.cases import bits, make_case

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _codebook(name, D):
    if name == "lloyd-max":
        return OQ.codebook(D)
    # thresholds `gap` rho apart, the middle one at `mid` rho
    gap, mid = {"gap 0.13": (0.13, 0.0), "gap 0.127": (0.127, 0.0), "gap 0.12": (0.12, 0.0),
                "gap 0.02": (0.02, 0.0), "wide": (0.5, 0.0), "past the table": (0.3, 2.5)}[name]
    return ((mid + gap * (np.arange(16) - 7.5)) / np.sqrt(D)).astype(np.float32)


@pytest.mark.parametrize("book", ["lloyd-max", "gap 0.13", "gap 0.127", "gap 0.12", "gap 0.02",
                                  "wide", "past the table"])
@pytest.mark.parametrize("Hkv,D,P,rows", [(1, 128, 64, 1), (1, 256, 64, 3), (3, 256, 128, 65),
                                          (5, 128, 256, 33)])
def test_tq4_append_tails_and_codebooks(Hkv, D, P, rows, book):
    case = make_case(rows + D, Hkv, Hkv, D, P, [rows], num_pages=-(-rows // P) + 1)
    for i in range(0, rows, 2):   # beside ordinary vectors of the same warp
        case.k[i, 0] = 0.0
        case.v[i, Hkv - 1] *= 2.0 ** (-110 if i % 4 else 118)
    c = _codebook(book, D)
    lay = OQ.Tq4Layout(Hkv, P, D, OQ.make_codec(D, OQ.sign_vector(OQ.SEED_K, D),
                                                OQ.sign_vector(OQ.SEED_V, D)))
    lay = OQ.Tq4Layout(Hkv, P, D, OQ.Codec(D, c, lay.codec.signs_k, lay.codec.signs_v))
    ref = OQ.new_pool(lay, case.num_pages, fill=0x33)
    OQ.append(ref, lay, case.page_table.numpy(), case.req.numpy(), case.pos.numpy(),
              bits(case.k), bits(case.v))
    codec = jf.Tq4Codec(D, synth.tq4_signs(synth.TQ4_SEED_K, D),
                        synth.tq4_signs(synth.TQ4_SEED_V, D), centroids=c)
    pool = jf.KVPool.allocate(case.num_pages, P, Hkv, D, device=DEV, fill=0x33,
                              format=jf.JF_FMT_TQ4, codec=codec)
    err = torch.zeros(1, dtype=torch.int32, device=DEV)
    jf.jf_kv_quantize_append(pool, case.page_table.to(DEV), case.req.to(DEV), case.pos.to(DEV),
                             case.k.to(DEV), case.v.to(DEV), err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert np.array_equal(pool.data.cpu().numpy(), ref)
