"""Launch shapes over the batch sizes and head counts a server uses, from a
stream capture: no kernel runs."""
import pytest
import torch

import paper_2609_17475_gb300 as jf
from tests.launches import launches

pytestmark = pytest.mark.gpu
DEV = "cuda"
PAGE = 64


def _batch(fmt, Hq, Hkv, D, B, q_len=1):
    """The launches of one decode (or verifier) call."""
    codec = jf.Tq4Codec(D, [1] * D, [1] * D) if fmt == jf.JF_FMT_TQ4 else None
    pool = jf.KVPool.allocate(4, PAGE, Hkv, D, device=DEV, format=fmt, codec=codec)
    table = torch.zeros(B, 4, dtype=torch.int32, device=DEV)
    lens = torch.full((B,), 4 * PAGE, dtype=torch.int32, device=DEV)
    if q_len == 1:
        S = jf.default_num_splits(B, Hkv, format=fmt)
        ws = jf.decode_workspace(B, Hq, Hkv, D, S, device=DEV)
        q = torch.zeros(B, Hq, D, dtype=torch.bfloat16, device=DEV)
        call = jf.jf_paged_decode_attn
    else:
        S = jf.default_verify_splits(B, q_len, Hq, Hkv, format=fmt)
        ws = jf.verify_workspace(B, q_len, Hq, Hkv, D, S, device=DEV)
        q = torch.zeros(B, q_len, Hq, D, dtype=torch.bfloat16, device=DEV)
        call = jf.jf_paged_verify_attn
    out = torch.empty_like(q)
    return launches(lambda stream: call(pool, table, lens, q, 0.1, out, ws, S, stream=stream))


@pytest.mark.parametrize("q_len", [1, 3])
@pytest.mark.parametrize("Hq,Hkv,D", [(8, 1, 128), (6, 1, 256), (12, 2, 256), (24, 4, 256),
                                      (32, 8, 128)])
@pytest.mark.parametrize("fmt", [jf.JF_FMT_AFFINE4_G64, jf.JF_FMT_TQ4])
def test_sliced_merge_fits_on_the_chip_at_once(fmt, Hq, Hkv, D, q_len):
    """A merge in column slices whose CTAs do not all fit at once takes longer
    than a CTA per row, whatever its plan's length: 24.9 against 18.0 us."""
    kinds = set()
    for B in (2, 3, 5, 9, 13, 19, 25, 38, 49, 60):
        if B * Hq * q_len > 1000:
            break
        (merge,) = [x for x in _batch(fmt, Hq, Hkv, D, B, q_len) if "merge" in x.name]
        sliced = "merge_sg" in merge.name
        kinds.add(sliced)
        if sliced:
            assert merge.ctas <= merge.resident, (B, merge)
    assert kinds == {True, False}


@pytest.mark.parametrize("Hq,Hkv,D", [(64, 16, 128), (24, 6, 256), (12, 3, 256), (10, 5, 128),
                                      (24, 12, 128), (28, 7, 128), (24, 4, 256), (200, 200, 128)])
def test_tq4_batch_pieces_fit_on_the_chip_at_once(Hq, Hkv, D):
    """A TQ4 batch's pieces are equal, so one more than fit at once makes two
    rounds of them: 172.6 against 104.9 us (16 KV heads, 160 pieces)."""
    for B in (2, 8, 24):
        (split,) = [x for x in _batch(jf.JF_FMT_TQ4, Hq, Hkv, D, B) if "tq4_split" in x.name]
        assert split.ctas <= max(split.resident, Hkv), (B, split)


@pytest.mark.parametrize("Hq,Hkv,D", [(6, 1, 256), (8, 2, 128), (12, 3, 256), (24, 4, 256),
                                      (32, 8, 128)])
def test_tq4_few_requests_take_whole_request_pieces(Hq, Hkv, D):
    """With 19 SMs or more for each request and KV head; spans from there on."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for B in range(2, 12):
        (split,) = [x for x in _batch(jf.JF_FMT_TQ4, Hq, Hkv, D, B) if "tq4_split" in x.name]
        spans = f"ILi{D}ELb0ELb0ELb1E" in split.name
        assert spans or f"ILi{D}ELb0ELb0ELb0E" in split.name, split
        assert spans == (19 * B * Hkv > sms), (B, split)
        assert split.ctas <= split.resident, (B, split)


@pytest.mark.parametrize("Hq,Hkv,D", [(64, 16, 128), (24, 6, 256), (12, 3, 256), (10, 5, 128),
                                      (24, 12, 128), (28, 7, 128), (24, 4, 256), (200, 200, 128)])
@pytest.mark.parametrize("fmt", [jf.JF_FMT_AFFINE4_G64, jf.JF_FMT_TQ4])
def test_decode_splits_fit_on_the_chip_at_once(fmt, Hq, Hkv, D):
    """One request and (affine) batches, at the default split counts."""
    for B in (1, 2, 12):
        (split,) = [x for x in _batch(fmt, Hq, Hkv, D, B) if "merge" not in x.name]
        assert split.ctas <= max(split.resident, Hkv), (B, split)
