"""Prefill chunks of up to one query tile, whose tiles pack the query heads of a kv head into
their rows (flash_fwd.cu).

Sizes: one token, one token around the tokens that fill a tile with all heads (32 of 4 heads, 18
of 7 with two rows left over), the longest packed chunk and the first unpacked one; 1 to 16 heads
per kv head; one tile, and two or more (whole items of many sequences, a long history); both head
dims; pieces merged in a two-piece cluster (up to 16 sequences; one with two rows left over) and by
the merge kernel, whole items; against the oracle's prefill_kv at the parity bar of gpu_util.  Each
case asserts the heads packed and how its items are cut.  The slots past the chunk hold NaN.
"""
import pytest

from oracle import oracle as O
from synthetic import workloads as w
from synthetic.workloads import Shape
from tests import plan_util
from tests.gpu_util import assert_cache, assert_out_close, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    assert t.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build()
    return t


WHOLE, PIECES, PAIR = "whole", "pieces", "pair"  # pieces: for the merge kernel; pair: a two-piece cluster
# batch, query heads, kv heads, head_dim, history, chunk; heads packed into a tile's rows, cut
CASES = [
    (1, 32, 8, 128, 0, 1, 1, WHOLE), (1, 32, 8, 128, 100, 31, 1, WHOLE), (1, 32, 8, 128, 127, 32, 1, WHOLE),
    (1, 32, 8, 128, 0, 33, 1, WHOLE), (1, 32, 8, 128, 4900, 128, 4, PIECES), (1, 32, 8, 128, 4900, 129, 1, PIECES),
    (1, 8, 8, 128, 400, 100, 1, PIECES), (2, 28, 4, 128, 700, 18, 7, PIECES), (2, 28, 4, 128, 700, 19, 1, PAIR),
    (1, 12, 2, 128, 1500, 21, 6, PIECES), (1, 7, 1, 128, 1500, 9, 7, PIECES), (1, 64, 8, 128, 5, 16, 1, WHOLE),
    (2, 64, 8, 128, 1200, 16, 8, PIECES), (1, 64, 4, 128, 60, 8, 1, WHOLE), (16, 40, 8, 128, 300, 5, 5, WHOLE),
    (1, 120, 40, 128, 130, 42, 1, WHOLE), (1, 16, 1, 64, 20, 8, 1, WHOLE), (1, 14, 2, 64, 640, 18, 7, PIECES),
    (3, 32, 8, 64, 1000, 32, 4, PIECES), (1, 32, 4, 64, 2000, 1, 8, PIECES), (6, 56, 8, 64, 500, 70, 7, WHOLE),
    (40, 8, 2, 128, 200, 70, 4, WHOLE), (1, 512, 64, 64, 300, 20, 8, WHOLE), (22, 14, 2, 128, 0, 128, 7, WHOLE),
    (8, 64, 8, 128, 1000, 16, 8, PAIR), (8, 32, 8, 128, 1500, 16, 4, PAIR), (8, 32, 8, 128, 1000, 1, 4, PAIR),
    (16, 28, 4, 64, 1500, 8, 7, PAIR), (8, 32, 8, 64, 1500, 40, 4, PAIR),
]


@pytest.mark.parametrize("case", CASES, ids=["b%d_h%d_kv%d_d%d_hist%d_n%d" % c[:6] for c in CASES])
def test_packed_heads_match_oracle(torch, case):
    from paper_2607_15865_gb300.attention import Attention
    batch, hq, hkv, d, hist, n, heads, cut = case
    shape = Shape("pk%d_%d" % (hq, n), batch, hq, hkv, d, hist + n + 20, 1.0e5)
    attn = Attention.for_shape(shape)
    packed, pieces, pair, _ = plan_util.prefill(attn, hist, n)
    assert (packed, PAIR if pair else PIECES if pieces > 1 else WHOLE) == (heads, cut)
    q, k, v = w.tokens(shape, "pk", n)
    kc, vc = w.cache(shape, "pk", hist, fill="nan")
    rk, rv = kc.copy(), vc.copy()
    ref = O.prefill_kv(shape, q, k, v, hist, rk, rv)
    gk, gv = to_dev(kc), to_dev(vc)
    out = attn.prefill_kv(to_dev(q), to_dev(k), to_dev(v), hist, gk, gv)
    torch.cuda.synchronize()
    assert attn.device_error() == 0
    assert_out_close(to_host(out), ref, "out")
    assert_cache(to_host(gk), to_host(gv), rk, rv, kc, vc, [(hist, hist + n)] * batch, "cache")
    attn.close()
