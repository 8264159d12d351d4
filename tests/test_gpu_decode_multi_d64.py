"""Decode at head_dim 64 on the tensor cores (decode_tc.cu), several new tokens per sequence:
the (token, query head) columns run 16 to a CTA and 16 tokens to a launch, P in three parts.

Sizes where that can go wrong: two columns, 8 and 9 columns, many column groups, 17 tokens (two
launches), new tokens that straddle a key tile, an empty history; then
tokens outside [0, max_len) (flagged and skipped one by one, the others of the sequence
computed) and a later token's NaN v, which an earlier token must not see.  The reference is
the oracle's decode, one token after the other (that order is the definition; the parity bar
is that of gpu_util).
"""
import dataclasses

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


def run_gpu(torch, shape, q, k, v, kc, vc, hist):
    from paper_2607_15865_gb300.attention import Attention
    attn = Attention.for_shape(shape)
    gk, gv = to_dev(kc), to_dev(vc)
    out0 = np.full(q.shape, 0x1234, np.uint16)
    out = attn.decode_multi(to_dev(q), to_dev(k), to_dev(v), torch.from_numpy(np.asarray(hist, np.int32)).cuda(), gk, gv,
                            out=to_dev(out0))
    torch.cuda.synchronize()
    flags = attn.device_error()
    attn.close()
    return to_host(out), to_host(gk), to_host(gv), flags


def reference(shape, q, k, v, kc, vc, hist):
    """Token after token and sequence by sequence; returns out, caches and the tokens computed."""
    one = dataclasses.replace(shape, batch=1)
    out = np.full(q.shape, 0x1234, np.uint16)
    rk, rv = kc.copy(), vc.copy()
    done = np.zeros(q.shape[:2], bool)
    for b, h in enumerate(hist):
        for i in range(q.shape[1]):
            if not 0 <= h + i < shape.max_len:
                continue
            ck, cv = rk[b:b + 1].copy(), rv[b:b + 1].copy()
            out[b:b + 1, i:i + 1] = O.decode(one, q[b:b + 1, i:i + 1].copy(), k[b:b + 1, i:i + 1].copy(),
                                             v[b:b + 1, i:i + 1].copy(), np.array([h + i], np.int32), ck, cv)
            rk[b:b + 1], rv[b:b + 1] = ck, cv
            done[b, i] = True
    return out, rk, rv, done


CASES = [
    ("g8_one_token_few_items_32_splits", Shape("m64j", 1, 16, 2, 64, 9000, 1.0e4), [8500], 1),
    ("g4_one_token_several_waves", Shape("m64k", 24, 16, 4, 64, 700, 1.0e4), [29 * i for i in range(24)], 1),
    ("g1_two_tokens_empty_history", Shape("m64a", 2, 2, 2, 64, 128, 1.0e4), [0, 3], 2),
    ("g4_two_tokens_8_columns", Shape("m64b", 1, 4, 1, 64, 256, 1.0e4), [63], 2),
    ("g3_three_tokens_9_columns", Shape("m64c", 2, 6, 2, 64, 512, 1.0e4), [62, 300], 3),
    ("g7_five_tokens", Shape("m64d", 2, 14, 2, 64, 2048, 1.0e6), [126, 1900], 5),
    ("g16_sixteen_tokens", Shape("m64e", 1, 16, 1, 64, 700, 1.0e4), [600], 16),
    ("g2_seventeen_tokens_two_launches", Shape("m64f", 2, 4, 2, 64, 300, 1.0e4), [0, 250], 17),
    ("g4_four_tokens_several_waves", Shape("m64l", 12, 32, 8, 64, 1000, 1.0e4), [80 * i for i in range(12)], 4),
    ("g4_four_tokens_many_splits", Shape("m64g", 1, 32, 8, 64, 8192, 5.0e5), [8000], 4),
]


@pytest.mark.parametrize("name,shape,hist,n", CASES, ids=[c[0] for c in CASES])
def test_d64_multi_token_decode_matches_oracle(torch, name, shape, hist, n):
    q, k, v = w.tokens(shape, "mt64", n)
    kc, vc = w.cache(shape, "mt64", int(max(hist)), fill="random")
    out, gk, gv, flags = run_gpu(torch, shape, q, k, v, kc, vc, hist)
    assert flags == 0
    ref, rk, rv, _ = reference(shape, q, k, v, kc, vc, hist)
    assert_out_close(out, ref, f"{name} out")
    assert_cache(gk, gv, rk, rv, kc, vc, [(h, h + n) for h in hist], f"{name} cache")


def test_d64_multi_token_decode_skips_tokens_out_of_range(torch):
    from paper_2607_15865_gb300 import _lib
    shape, n = Shape("m64h", 4, 8, 2, 64, 128, 1.0e4), 4
    hist = [126, -2, 128, 40]  # two tokens past the end, two before the start, all past the end, none
    q, k, v = w.tokens(shape, "mt64e", n)
    kc, vc = w.cache(shape, "mt64e", 128, fill="random")
    out, gk, gv, flags = run_gpu(torch, shape, q, k, v, kc, vc, hist)
    assert flags & _lib.DEVERR_HIST_RANGE
    ref, rk, rv, done = reference(shape, q, k, v, kc, vc, hist)
    assert (out[~done] == ref[~done]).all(), "a skipped token's output was written"
    assert_out_close(out[done], ref[done], "tokens in range")
    ranges = [(max(h, 0), min(h + n, shape.max_len)) if h < shape.max_len else (0, 0) for h in hist]
    assert_cache(gk, gv, rk, rv, kc, vc, ranges, "range cache")


def test_d64_decode_weights_keep_float_precision(torch):
    """Against the oracle's attention (float64) before its rounding the kernel is off by the bf16
    rounding of out alone: as many outputs differ from the oracle's bits as float sums of that
    length leave on the other side of a rounding boundary (2^-24 per sum against 2^-9 per step;
    weights rounded to bf16 would leave most of them different)."""
    shape, hist = Shape("m64p", 2, 32, 8, 64, 4096, 1.0e4), [3000, 4000]
    q, k, v = w.tokens(shape, "mt64p", 1)
    kc, vc = w.cache(shape, "mt64p", 4000, fill="random")
    out, _, _, flags = run_gpu(torch, shape, q, k, v, kc, vc, hist)
    assert flags == 0
    ref, _, _, _ = reference(shape, q, k, v, kc, vc, hist)
    share = float((out != ref).mean())
    print(f"share of outputs that differ by a bf16 step: {share:.4f}")
    assert share <= 0.02


def test_d64_multi_token_decode_later_nan_v_not_seen(torch):
    shape, n, hist = Shape("m64i", 1, 8, 2, 64, 256, 1.0e4), 4, [62]
    q, k, v = w.tokens(shape, "mt64n", n)
    v[:, 2:] = 0x7FC0  # tokens 2 and 3 carry NaN
    kc, vc = w.cache(shape, "mt64n", 62, fill="random")
    out, _, gv, flags = run_gpu(torch, shape, q, k, v, kc, vc, hist)
    assert flags == 0
    ref, _, rv, _ = reference(shape, q[:, :2], k[:, :2], v[:, :2], kc, vc, hist)
    assert_out_close(out[:, :2], ref, "tokens before the NaN")
    assert ((out[:, 2:] & 0x7FFF) > 0x7F80).all(), "the tokens that see it are NaN"
    assert (gv[:, :, 64:66] == 0x7FC0).all()
