"""Decode of 46 to 76 items on 152 SMs (39 to 152 at head_dim 64, two CTAs per SM; decode_tc.cu):
several waves with one split more than a wave holds, which stands down where the batch's lengths
are even.

Sizes: the ends of the ranges and one item past each, even lengths (within 10%), mixed ones, one
long among short, an empty history, a sequence out of range; both head dims.  The second of two
calls on the same context checks that the first left the claim counters clean.
"""
import numpy as np
import pytest

from oracle import oracle as O
from synthetic import workloads as w
from synthetic.workloads import Shape
from tests.gpu_util import assert_cache, assert_out_close, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    assert t.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build()
    return t


def lengths(kind, batch):
    if kind == "even":
        return [1400 - 20 * (b % 3) for b in range(batch)]
    if kind == "short":
        return [b % 100 for b in range(batch)]
    return [1490] + [(50 * b) % 1500 for b in range(batch - 1)] if kind == "mixed" else [1490] + [7] * (batch - 1)


GROUP = 2  # query heads per kv head
CASES = [(b, hkv, d, kind) for b, hkv in ((45, 1), (46, 1), (8, 8), (19, 4), (11, 7)) for d in (128, 64)
         for kind in (("even", "mixed") if b != 8 else ("even", "mixed", "long", "short"))]
CASES += [(b, hkv, 64, kind) for b, hkv in ((38, 1), (39, 1), (38, 4), (51, 3)) for kind in ("even", "mixed")]


@pytest.mark.parametrize("batch,hkv,d,kind", CASES)
def test_mid_items_match_oracle(torch, batch, hkv, d, kind, group=GROUP):
    from paper_2607_15865_gb300.attention import Attention
    shape = Shape("mid", batch, group * hkv, hkv, d, 3000, 1.0e5)
    hist = np.asarray(lengths(kind, batch), np.int32)
    q, k, v = w.tokens(shape, "mid", 1)
    kc, vc = w.cache(shape, "mid", int(hist.max()), fill="random")
    rk, rv = kc.copy(), vc.copy()
    ref = O.decode(shape, q, k, v, hist, rk, rv)
    attn = Attention.for_shape(shape)
    for _ in range(2):
        gk, gv = to_dev(kc), to_dev(vc)
        out = attn.decode(to_dev(q), to_dev(k), to_dev(v), torch.from_numpy(hist).cuda(), gk, gv)
        torch.cuda.synchronize()
        assert attn.device_error() == 0
        assert_out_close(to_host(out), ref, "out")
        assert_cache(to_host(gk), to_host(gv), rk, rv, kc, vc, [(int(h), int(h) + 1) for h in hist], "cache")
    attn.close()


@pytest.mark.parametrize("batch,hkv", [(1, 2), (10, 4), (80, 2)])
def test_d64_sixteen_heads_per_kv_head(torch, batch, hkv):
    test_mid_items_match_oracle(torch, batch, hkv, 64, "mixed", group=16)


def test_mid_items_even_with_a_sequence_out_of_range(torch):
    from paper_2607_15865_gb300 import _lib
    from paper_2607_15865_gb300.attention import Attention
    shape = Shape("mido", 8, 16, 8, 128, 1500, 1.0e5)
    hist = np.asarray([1400] * 7 + [1500], np.int32)  # the last one is full: flagged and skipped
    q, k, v = w.tokens(shape, "mido", 1)
    kc, vc = w.cache(shape, "mido", 1500, fill="random")
    rk, rv = kc.copy(), vc.copy()
    ok = hist.copy()
    ok[7] = 0
    ref = O.decode(shape, q, k, v, ok, rk, rv)
    attn = Attention.for_shape(shape)
    gk, gv = to_dev(kc), to_dev(vc)
    out = attn.decode(to_dev(q), to_dev(k), to_dev(v), torch.from_numpy(hist).cuda(), gk, gv)
    torch.cuda.synchronize()
    assert attn.device_error() & _lib.DEVERR_HIST_RANGE
    assert_out_close(to_host(out)[:7], ref[:7], "sequences in range")
    assert (to_host(gk)[7] == kc[7]).all() and (to_host(gv)[7] == vc[7]).all()
    attn.close()
