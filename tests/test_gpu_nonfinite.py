"""NaN keys inside the valid history, and infinite values, in every merge of split work.

A NaN key makes the softmax of each query that sees it NaN, whatever the number of pieces that
the history is cut into: a piece whose row sum is NaN must not be left out as if it held no
keys.  The other kv heads and sequences stay at the parity bar of gpu_util against the oracle.

Paths: prefill_kv in two-piece clusters (plain tiles, packed heads), through the merge kernel and
whole; decode merged in a cluster, through global memory and in several waves, with one new token
and several; both head dims.  Each case asserts its path.
"""
import numpy as np
import pytest

from oracle import oracle as O
from synthetic import workloads as w
from synthetic.workloads import Shape
from tests import plan_util
from tests.gpu_util import assert_out_close, to_dev, to_host
from tests.plan_util import CLUSTER, GLOBAL, WAVES

pytestmark = pytest.mark.gpu

NAN = 0x7FC0


@pytest.fixture(scope="module")
def torch():
    import torch as t
    assert t.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build()
    return t


def is_nan(bits):
    return (bits & 0x7FFF) > 0x7F80


# name, shape, history, chunk, (packed heads, two-piece cluster, pieces or None)
PREFILL = [
    ("cluster_d128", Shape("nfc", 1, 64, 8, 128, 900, 1.0e4), 600, 250, (1, True, 2)),
    ("cluster_d64", Shape("nfc64", 1, 64, 8, 64, 900, 1.0e4), 600, 256, (1, True, 2)),
    ("cluster_packed_d128", Shape("nfp", 8, 32, 8, 128, 1100, 1.0e4), 1000, 16, (4, True, 2)),
    ("cluster_packed_d64", Shape("nfp64", 16, 28, 4, 64, 1600, 1.0e4), 1500, 8, (7, True, 2)),
    ("merge_kernel_d128", Shape("nfm", 1, 24, 8, 128, 1900, 1.0e4), 1600, 250, (1, False, None)),
    ("merge_kernel_d64", Shape("nfm64", 1, 24, 8, 64, 1900, 1.0e4), 1600, 250, (1, False, None)),
    ("whole_d128", Shape("nfw", 4, 64, 8, 128, 400, 1.0e4), 100, 140, (1, False, 1)),
]


@pytest.mark.parametrize("slot_from_end", [False, True], ids=["first_piece", "last_piece"])
@pytest.mark.parametrize("name,shape,hist,n,path", PREFILL, ids=[c[0] for c in PREFILL])
def test_prefill_nan_key_in_the_history(torch, name, shape, hist, n, path, slot_from_end):
    from paper_2607_15865_gb300.attention import Attention
    attn = Attention.for_shape(shape)
    heads, pieces, cluster, whole = plan_util.prefill(attn, hist, n)
    assert (heads, cluster) == path[:2] and (pieces == path[2] if path[2] else pieces > 2 and whole == 0)
    q, k, v = w.tokens(shape, "nf", n)
    kc, vc = w.cache(shape, "nf", hist, fill="zero")
    ref = O.prefill_kv(shape, q, k, v, hist, kc.copy(), vc.copy())
    g = shape.n_kv_heads - 1
    kc[0, g, hist - 2 if slot_from_end else 3, 5] = NAN
    out = to_host(attn.prefill_kv(to_dev(q), to_dev(k), to_dev(v), hist, to_dev(kc), to_dev(vc)))
    assert attn.device_error() == 0
    attn.close()
    sees = np.zeros(out.shape[:3], bool)
    sees[0, :, g * shape.group:] = True
    assert is_nan(out[sees]).all(), f"{name}: {is_nan(out[sees]).mean():.3f} of the outputs that see the NaN are NaN"
    assert_out_close(out[~sees], ref[~sees], f"{name} rest")


LOW = 63  # the slowest pair's first dimension at head_dim 128 (31 at 64): barely rotated over these positions


def one_key_takes_all(shape, q, kc, slot):
    """q and the key at `slot` such that this key's softmax weight is 1 and every other's 0."""
    d = LOW if shape.head_dim == 128 else 31
    q[...] = 0
    q[..., d] = 0x3F80  # 1.0
    kc[:, :, slot] = 0
    kc[:, :, slot, d] = 0x4580  # 4096


@pytest.mark.parametrize("name,shape,hist,n,path", [c for c in PREFILL if "cluster" in c[0] or "merge" in c[0]],
                         ids=[c[0] for c in PREFILL if "cluster" in c[0] or "merge" in c[0]])
def test_prefill_infinite_value_in_a_piece_of_weight_zero(torch, name, shape, hist, n, path):
    from paper_2607_15865_gb300.attention import Attention
    q, k, v = w.tokens(shape, "nfz", n)
    kc, vc = w.cache(shape, "nfz", hist, fill="zero")
    one_key_takes_all(shape, q, kc, hist - 2)
    vc[:, :, 3, 1] = 0x7F80
    attn = Attention.for_shape(shape)
    out = to_host(attn.prefill_kv(to_dev(q), to_dev(k), to_dev(v), hist, to_dev(kc), to_dev(vc)))
    attn.close()
    want = np.repeat(vc[:, :, hist - 2], shape.group, axis=1)[:, None]  # [B, 1, Hq, D]
    assert (out == want).all()


# name, shape, lengths, new tokens, merge mode
DECODE = [
    ("cluster_d128", Shape("nfd1", 1, 32, 8, 128, 2048, 1.0e4), [2000], 1, CLUSTER),
    ("cluster_d64", Shape("nfd2", 1, 32, 8, 64, 2048, 1.0e4), [2000], 1, CLUSTER),
    ("global_d128", Shape("nfd3", 8, 8, 1, 128, 8320, 1.0e4), [8200] + [500] * 7, 1, GLOBAL),
    ("global_d64", Shape("nfd4", 1, 16, 2, 64, 9000, 1.0e4), [8500], 1, GLOBAL),
    ("waves_d128", Shape("nfd5", 20, 16, 8, 128, 4096, 1.0e4), [4000] + [60 * b for b in range(19)], 1, WAVES),
    ("waves_d64", Shape("nfd6", 24, 16, 8, 64, 4096, 1.0e4), [4000] + [60 * b for b in range(23)], 1, WAVES),
    ("cluster_d128_three_tokens", Shape("nfd7", 1, 32, 8, 128, 2048, 1.0e4), [2000], 3, CLUSTER),
    ("cluster_d64_three_tokens", Shape("nfd8", 1, 32, 8, 64, 2048, 1.0e4), [2000], 3, CLUSTER),
    ("waves_d64_four_tokens", Shape("nfd9", 12, 32, 8, 64, 2100, 1.0e4), [2000] + [80 * b for b in range(11)], 4, WAVES),
]


def run_decode(torch, shape, hist, n, mode, edit=None):
    """The decode of n tokens after edit(kc, vc, v); and the oracle's without the edit."""
    from paper_2607_15865_gb300.attention import Attention
    hist = np.asarray(hist, np.int32)
    q, k, v = w.tokens(shape, "nfd", n)
    kc, vc = w.cache(shape, "nfd", int(hist.max()), fill="zero")
    ref = np.zeros(q.shape, np.uint16)
    rk, rv = kc.copy(), vc.copy()
    for i in range(n):
        ref[:, i:i + 1] = O.decode(shape, q[:, i:i + 1].copy(), k[:, i:i + 1].copy(), v[:, i:i + 1].copy(), hist + i, rk, rv)
    edit(kc, vc, v)
    attn = Attention.for_shape(shape)
    assert plan_util.decode(attn, n)[1] == mode
    hl = torch.from_numpy(hist).cuda()
    out = to_host(attn.decode_multi(to_dev(q), to_dev(k), to_dev(v), hl, to_dev(kc), to_dev(vc)))
    assert attn.device_error() == 0
    attn.close()
    return out, ref


@pytest.mark.parametrize("slot_from_end", [False, True], ids=["first_split", "last_split"])
@pytest.mark.parametrize("name,shape,hist,n,mode", DECODE, ids=[c[0] for c in DECODE])
def test_decode_nan_key_in_the_history(torch, name, shape, hist, n, mode, slot_from_end):
    g = shape.n_kv_heads - 1

    def edit(kc, vc, v):
        kc[0, g, hist[0] - 2 if slot_from_end else 3, 5] = NAN
    out, ref = run_decode(torch, shape, hist, n, mode, edit)
    sees = np.zeros(out.shape[:3], bool)
    sees[0, :, g * shape.group:] = True
    assert is_nan(out[sees]).all(), f"{name}: {is_nan(out[sees]).mean():.3f} of the outputs that see the NaN are NaN"
    assert_out_close(out[~sees], ref[~sees], f"{name} rest")


@pytest.mark.parametrize("name,shape,hist,n,mode", DECODE, ids=[c[0] for c in DECODE])
def test_decode_infinite_values(torch, name, shape, hist, n, mode):
    """Infinite values of a cached token, and at head_dim 64 of the first new token: that sign in their
    dimensions, NaN where both signs meet, the other dimensions unchanged."""
    g, h, d64 = shape.n_kv_heads - 1, hist[0], shape.head_dim == 64

    def edit(kc, vc, v):
        vc[0, g, h // 2, 1] = vc[0, g, h - 1, 3] = vc[0, g, 5, 7] = 0x7F80  # +inf
        vc[0, g, h - 1, 7] = 0xFF80  # -inf
        if d64:
            v[0, 0, g, 9] = 0xFF80
            v[0, 0, g, 3] = 0x7F80
    out, ref = run_decode(torch, shape, hist, n, mode, edit)
    hot = out[0, :, g * shape.group:]
    assert (hot[..., [1, 3]] == 0x7F80).all(), hot[0, 0, :10]
    assert is_nan(hot[..., 7]).all()
    if d64:
        assert (hot[..., 9] == 0xFF80).all()
    plain = np.ones(out.shape, bool)
    plain[0, :, g * shape.group:, [1, 3, 7, 9]] = False
    assert_out_close(out[plain], ref[plain], f"{name} other dimensions")
