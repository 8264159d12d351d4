"""GPU parity of the W4BF16 GEMV where the K groups are split over a thread-block cluster (x
too large to stage whole: several rows, or long ones).  Bound and oracle as in
tests/test_gpu_w4.py: the partial sums meet in float, which that bound covers.

Sizes: clusters of 2, 4 and 8, groups that divide unevenly over the CTAs and over the warps of
one, a single unit, row-tiles past N, several rounds of units, two launches (11 rows), the split
output with a residual-free part and the residual, and a product that chains on its own output;
and shapes just short of a cluster, which run the plain kernel.  Each case asserts the CTAs per
cluster of its first launch and whether there are several rounds.
"""
import numpy as np
import pytest

from oracle import w4_oracle as W
from synthetic import gen
from tests import plan_util
from tests.test_gpu_w4 import check, make, partial_sum_bound, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    assert t.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build()
    return t


# name, rows, N, K, CTAs per cluster (1: the plain kernel), several rounds
CASES = [
    ("plain_m4_k4096", 4, 200, 4096, 1, False),
    ("plain_m1_k18944_single_unit", 1, 7, 18944, 1, False),
    ("plain_m8_k4096_plus_uneven", 8, 130, 4096 + 640, 1, False),
    ("plain_m11_two_launches", 11, 40, 6144, 1, False),
    ("plain_m4_many_rounds", 4, 30000, 4096, 1, False),
    ("c2_m2_k18944", 2, 200, 18944, 2, False),
    ("c2_m2_k18944_several_rounds", 2, 16384, 18944, 2, True),
    ("c4_m3_k11008", 3, 49, 11008, 4, False),
    ("c4_m4_k10368_uneven_single_unit", 4, 7, 10368, 4, False),
    ("c4_m4_k13824_several_rounds", 4, 5120, 13824, 4, True),
    ("c4_m11_two_launches", 11, 40, 11008, 4, False),
    ("c8_m8_k18944", 8, 33, 18944, 8, False),
    ("c8_m5_k16512", 5, 16, 16512, 8, False),
    ("c8_m8_k18944_several_rounds", 8, 3000, 18944, 8, True),
]


@pytest.mark.parametrize("tag,M,N,K,C,several", CASES, ids=[c[0] for c in CASES])
def test_w4_gemv_cluster_matches_oracle(torch, tag, M, N, K, C, several):
    from paper_2607_15865_gb300.w4 import pack_codes
    rows, ctas, rounds, _ = plan_util.gemv(M, N, K)
    assert ctas == C and (rounds > 1) == several and rows == min(M, 8)
    codes, zeros, scales, x = make(tag, M, N, K)
    y = run(torch, pack_codes(codes), zeros, scales, x)
    rows = None if N < 1000 else np.unique(np.concatenate([np.arange(20), np.arange(N - 20, N),
                                                           np.random.default_rng(5).integers(0, N, 200)]))
    check(codes, zeros, scales, x, y, rows)


def test_w4_gemv_cluster_residual_and_split(torch):
    from paper_2607_15865_gb300.w4 import pack_codes, pack_tiles, w4bf16_gemv, w4bf16_gemv_fused
    M, N, K = 6, 400, 11008
    assert plan_util.gemv(M, N, K)[:2] == (M, 4)
    codes, zeros, scales, x = make("cl_fused", M, N, K)
    res = gen.normal_bf16("w4gpu", "cl_fused_res", (M, N), 1.0)
    tiles = torch.from_numpy(pack_tiles(pack_codes(codes), scales, zeros)).cuda()
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).cuda().view(torch.bfloat16)
    xd, rd = dev(x), dev(res)
    y = w4bf16_gemv(tiles, xd, N)
    parts = w4bf16_gemv_fused(tiles, xd, N, split=(128, 272))
    assert torch.equal(torch.cat(parts, dim=1), y)
    h = w4bf16_gemv_fused(tiles, xd, N, residual=rd, out=rd)  # in place over the residual
    torch.cuda.synchronize()
    ref = W.gemv(codes, scales, zeros, x) + W.bf16_to_f64(res)
    got = W.bf16_to_f64(h.view(torch.int16).cpu().numpy().view(np.uint16))
    bound = 2.0 ** -8 * np.abs(ref) + 2.0 ** -18 * partial_sum_bound(codes, scales, zeros, x)
    assert (np.abs(got - ref) <= bound).all()


def test_w4_gemv_cluster_chain(torch):
    """Each call's x is the previous call's y (dependent launches, weights streamed early): the
    result of the chain is that of the same calls with a synchronisation between them."""
    from paper_2607_15865_gb300.w4 import pack_codes, pack_tiles, w4bf16_gemv
    M, N, K = 8, 11008, 11008
    rows, ctas, rounds, _ = plan_util.gemv(M, N, K)
    assert (rows, ctas) == (M, 4) and rounds > 1
    codes, zeros, scales, x = make("cl_chain", M, N, K)
    scales = (scales & np.uint16(0x007F)) | np.uint16(0x3A80)  # about 1e-3: the chain keeps its size
    tiles = torch.from_numpy(pack_tiles(pack_codes(codes), scales, zeros)).cuda()
    xd = torch.from_numpy(x.view(np.int16)).cuda().view(torch.bfloat16)

    def chain(sync):
        v = xd
        for _ in range(5):
            v = w4bf16_gemv(tiles, v, N, weights_static=True)
            if sync:
                torch.cuda.synchronize()
        return v
    a, b = chain(False), chain(True)
    torch.cuda.synchronize()
    assert torch.equal(a, b) and torch.isfinite(a.float()).all()
