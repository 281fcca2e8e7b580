"""The TQ4 fused step encodes a request's new K and V vectors on two warps, and
the warp that copies their chunk waits for the other: one after the other on one
warp, a step at 600 to 18,000 positions took 1.8 us (a seventh) longer.  Both
vectors' stores are fenced before that barrier, and the copying warp fences
after it (its copies go through the async proxy).  A missing fence is a race
that no run is sure to show, so this reads the source."""
import os
import re

TQ4 = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2609_17475_gb300", "csrc", "tq4.cu")
SOURCE = re.sub(r"//[^\n]*", "", open(TQ4).read())


def test_two_warps_encode():
    roles = {k: re.search(rf"encodes_{k} = APP && owns_last && warp == (.*?);", SOURCE).group(1)
             for k in "kv"}
    assert roles == {"k": "(n_cta - 1) % TQ_WARPS", "v": "n_cta % TQ_WARPS"}
    calls = re.findall(r"if \(encodes_(\w)[^)]*\)\s*append_new_vector<D>\(a, prm, b, kvh, (\d),",
                       SOURCE)
    assert sorted(calls) == [("k", "0"), ("k", "0"), ("v", "1")]


def test_stores_are_fenced_on_both_sides_of_the_barrier():
    body = SOURCE[SOURCE.index("void append_new_vector("):]
    body = body[:body.index("\n}\n")]
    assert re.search(r"tq4_store<D>\(.*?fence_proxy_async_global\(\);\s*__syncwarp\(\);"
                     r"\s*if \(kind\) \{\s*asm volatile\(\"bar\.arrive.*?"
                     r"\} else \{\s*asm volatile\(\"bar\.sync.*?fence_proxy_async_global\(\);",
                     body, re.S), body
