"""A TQ4 codec, and a pool that holds one, can be copied and pickled (a server
hands them to its workers), and the copy's calls read the copy's own codec."""
import copy
import ctypes
import pickle

import numpy as np
import pytest
import torch

import paper_2609_17475_gb300 as jf
from paper_2609_17475_gb300 import synth

D = 128


def _codec():
    return jf.Tq4Codec(D, synth.tq4_signs(synth.TQ4_SEED_K, D), synth.tq4_signs(synth.TQ4_SEED_V, D))


def _bytes(codec):
    return ctypes.string_at(ctypes.addressof(codec._c), ctypes.sizeof(codec._c))


@pytest.mark.parametrize("again", [copy.copy, copy.deepcopy,
                                   lambda x: pickle.loads(pickle.dumps(x))])
def test_codec_and_pool_copies(again):
    codec = _codec()
    other = again(codec)
    assert np.array_equal(other.centroids, codec.centroids) and _bytes(other) == _bytes(codec)
    pool = jf.KVPool(torch.zeros(2, jf.jf_kv_page_bytes_fmt(jf.JF_FMT_TQ4, 2, 64, D),
                                 dtype=torch.uint8), 64, 2, D, format=jf.JF_FMT_TQ4, codec=codec)
    twin = again(pool)
    c = twin.c_struct()
    assert ctypes.addressof(c.tq4.contents) == ctypes.addressof(twin.codec._c)
    assert _bytes(twin.codec) == _bytes(codec) and torch.equal(twin.data, pool.data)
