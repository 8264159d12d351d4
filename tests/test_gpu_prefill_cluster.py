"""Prefill chunks small enough that every work item is cut into KV pieces.  Two pieces of an item
are one thread-block cluster and merge in the kernel (flash_fwd.cu), each CTA half of the
columns; more go through the merge kernel.

Sizes: 2 to 16 pieces (by the number of heads), both head dims, one row (one query head per kv
head, and packed heads), one and two query tiles with ragged rows, a piece whose keys the first
tile does not see, two sequences; and chunks whose items stay whole; against the oracle's
prefill_kv at the parity bar of gpu_util.  Each case asserts its number of pieces.  The slots past
the chunk hold NaN.
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


# name, shape, history, chunk, pieces per item
CASES = [
    ("h64_two_pieces", Shape("pc1", 1, 64, 8, 128, 900, 1.0e4), 600, 250, 2),
    ("h32_two_pairs_of_tiles_ragged", Shape("pc0", 1, 32, 8, 128, 1400, 1.0e4), 1000, 300, 2),
    ("h70_two_pieces_one_row", Shape("pc12", 1, 70, 70, 128, 1400, 1.0e4), 1300, 1, 2),
    ("h64_d64_two_pieces_one_row", Shape("pc14", 1, 64, 64, 64, 1600, 1.0e4), 1500, 1, 2),
    ("h70_packed_eleven_pieces_one_row", Shape("pc15", 1, 70, 7, 128, 1400, 1.0e4), 1300, 1, 11),
    ("h36_two_sequences_two_pieces", Shape("pc13", 2, 36, 4, 128, 1400, 1.0e4), 1100, 140, 2),
    ("h32_two_sequences", Shape("pc2", 2, 32, 8, 128, 1400, 1.0e6), 1100, 200, 2),
    ("h56_two_pieces", Shape("pc11", 1, 56, 8, 128, 860, 1.0e4), 600, 256, 2),
    ("h8_last_of_six_pieces_past_first_tile", Shape("pc18", 1, 8, 8, 128, 760, 1.0e4), 500, 256, 6),
    ("h40_three_pieces", Shape("pc3", 1, 40, 8, 128, 1300, 1.0e6), 1000, 256, 3),
    ("h32_four_pieces_one_row", Shape("pc4", 1, 32, 32, 128, 2100, 5.0e5), 2000, 1, 4),
    ("h32_packed_sixteen_pieces_one_row", Shape("pc16", 1, 32, 8, 128, 2100, 5.0e5), 2000, 1, 16),
    ("h28_five_pieces_ragged", Shape("pc5", 1, 28, 4, 128, 1800, 1.0e6), 1500, 131, 5),
    ("h24_five_pieces", Shape("pc6", 1, 24, 8, 128, 1900, 1.0e4), 1600, 250, 5),
    ("h16_eight_pieces", Shape("pc7", 1, 16, 2, 128, 3000, 1.0e4), 2600, 140, 8),
    ("h64_d64_two_pieces", Shape("pc8", 1, 64, 8, 64, 900, 1.0e4), 600, 256, 2),
    ("h32_d64_four_pieces", Shape("pc9", 1, 32, 8, 64, 2000, 1.0e4), 1700, 77, 4),
    ("h32_no_history_whole", Shape("pc10", 1, 32, 8, 128, 256, 1.0e4), 0, 256, 1),
    ("h56_short_history_whole", Shape("pc17", 1, 56, 8, 128, 512, 1.0e4), 256, 256, 1),
]


@pytest.mark.parametrize("name,shape,hist,n,pieces", CASES, ids=[c[0] for c in CASES])
def test_cluster_pieces_match_oracle(torch, name, shape, hist, n, pieces):
    from paper_2607_15865_gb300.attention import Attention
    attn = Attention.for_shape(shape)
    _, cut, cluster, whole = plan_util.prefill(attn, hist, n)
    assert cut == pieces and cluster == (pieces == 2) and (pieces == 1 or whole == 0)
    q, k, v = w.tokens(shape, "pc", n)
    kc, vc = w.cache(shape, "pc", hist, fill="nan")
    rk, rv = kc.copy(), vc.copy()
    ref = O.prefill_kv(shape, q, k, v, hist, rk, rv)
    gk, gv = to_dev(kc), to_dev(vc)
    out = attn.prefill_kv(to_dev(q), to_dev(k), to_dev(v), hist, gk, gv)
    again = attn.prefill_kv(to_dev(q), to_dev(k), to_dev(v), hist, gk, gv)
    torch.cuda.synchronize()
    assert attn.device_error() == 0
    assert (to_host(out) == to_host(again)).all()
    assert_out_close(to_host(out), ref, f"{name} out")
    assert_cache(to_host(gk), to_host(gv), rk, rv, kc, vc, [(hist, hist + n)] * shape.batch, f"{name} cache")
    attn.close()
