"""TQ4 append of vectors whose indices and norm are far from any rounding boundary:
none of them needs fp64, so many rows take little longer than one; bytes against
the oracle."""
import numpy as np
import pytest
import torch

import paper_2609_17475_gb300 as jf
from oracle import tq4 as OQ
from paper_2609_17475_gb300 import synth
from tests.cases import bits
from tests.launches import device_us

pytestmark = pytest.mark.gpu
DEV = "cuda"
Hkv, P, ROWS = 4, 64, 64


def _easy_vectors(D, n, sign, seed):
    """n bf16 vectors of N(0, 1) values, [n, D]: every |u / rho - threshold| above
    2^-14, the norm over 2^-6 half-ulps from a rounding boundary."""
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(2 * n, D, generator=g).to(torch.bfloat16)
    h = np.ones((1, 1))
    while h.shape[0] < D:
        h = np.block([[h, h], [h, -h]])
    xd = x.double().numpy()
    s = np.sqrt((xd * xd).sum(1))
    rho = s.astype(np.float32)
    c = np.asarray(jf.jf_tq4_codebook(D), dtype=np.float64)
    t = (c[1:] + c[:-1]) / 2 * np.sqrt(D)
    near = np.abs((xd * sign) @ h / rho[:, None].astype(np.float64) - t[:, None, None]).min((0, 2))
    half = (np.nextafter(rho, np.float32(np.inf)).astype(np.float64) - rho) / 2
    edge = np.abs(np.abs(s - rho) - half) / half
    good = np.flatnonzero((near > 2.0 ** -14) & (edge > 2.0 ** -6))
    assert len(good) >= n
    return x[good[:n]]


@pytest.mark.parametrize("D", [128, 256])
def test_rows_without_a_doubt_take_no_fp64(D):
    signs = [synth.tq4_signs(s, D) for s in (synth.TQ4_SEED_K, synth.TQ4_SEED_V)]
    k, v = (_easy_vectors(D, ROWS * Hkv, np.asarray(signs[i], dtype=np.float64), D + i)
            .reshape(ROWS, Hkv, D) for i in range(2))
    table = torch.tensor([[2, 0, 1]], dtype=torch.int32)
    req = torch.zeros(ROWS, dtype=torch.int32)
    pos = torch.arange(5, 5 + ROWS, dtype=torch.int32)
    lay = OQ.Tq4Layout(Hkv, P, D, OQ.Codec(D, jf.jf_tq4_codebook(D), *signs))
    ref = OQ.new_pool(lay, 3, fill=0x33)
    OQ.append(ref, lay, table.numpy(), req.numpy(), pos.numpy(), bits(k), bits(v))
    pool = jf.KVPool.allocate(3, P, Hkv, D, device=DEV, fill=0x33, format=jf.JF_FMT_TQ4,
                              codec=jf.Tq4Codec(D, *signs))
    table, req, pos, k, v = (t.to(DEV) for t in (table, req, pos, k, v))

    def append(n):
        jf.jf_kv_quantize_append(pool, table, req[:n], pos[:n], k[:n], v[:n])

    append(ROWS)
    torch.cuda.synchronize()
    assert np.array_equal(pool.data.cpu().numpy(), ref)
    one, many = device_us(lambda: append(1)), device_us(lambda: append(ROWS))
    assert many <= 1.35 * one, (one, many)
