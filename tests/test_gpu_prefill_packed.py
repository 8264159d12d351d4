"""Prefill chunks of up to one query tile, whose tiles pack the query heads of a kv head into
their rows (flash_fwd.cu).

Sizes: one token, one token around the tokens that fill a tile with all heads (32 of 4 heads, 18
of 7 with two rows left over), the longest packed chunk and the first unpacked one; 1 to 16 heads
per kv head; one tile, and two or more (whole items of many sequences, a long history); both head
dims; pieces merged in a cluster and by the merge kernel; against the oracle's prefill_kv at the
parity bar of gpu_util.  The slots past the chunk hold NaN.
"""
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


# batch, query heads, kv heads, head_dim, history, chunk
CASES = [
    (1, 32, 8, 128, 0, 1), (1, 32, 8, 128, 100, 31), (1, 32, 8, 128, 127, 32), (1, 32, 8, 128, 0, 33),
    (1, 32, 8, 128, 4900, 128), (1, 32, 8, 128, 4900, 129), (1, 8, 8, 128, 400, 100), (2, 28, 4, 128, 700, 18),
    (2, 28, 4, 128, 700, 19), (1, 12, 2, 128, 1500, 21), (1, 7, 1, 128, 1500, 9), (1, 64, 8, 128, 5, 16),
    (2, 64, 8, 128, 1200, 16), (1, 64, 4, 128, 60, 8), (16, 40, 8, 128, 300, 5), (1, 120, 40, 128, 130, 42),
    (1, 16, 1, 64, 20, 8), (1, 14, 2, 64, 640, 18), (3, 32, 8, 64, 1000, 32), (1, 32, 4, 64, 2000, 1),
    (6, 56, 8, 64, 500, 70), (40, 8, 2, 128, 200, 70), (1, 512, 64, 64, 300, 20), (22, 14, 2, 128, 0, 128),
]


@pytest.mark.parametrize("case", CASES, ids=["b%d_h%d_kv%d_d%d_hist%d_n%d" % c for c in CASES])
def test_packed_heads_match_oracle(torch, case):
    from paper_2607_15865_gb300.attention import Attention
    batch, hq, hkv, d, hist, n = case
    shape = Shape("pk%d_%d" % (hq, n), batch, hq, hkv, d, hist + n + 20, 1.0e5)
    attn = Attention.for_shape(shape)
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
