"""How the library cuts a call on this device (attn_plan_*: exported for tests, not in attn.h)."""
from __future__ import annotations

import ctypes

from paper_2607_15865_gb300 import _lib

GLOBAL, CLUSTER, WAVES = 0, 1, 2  # merges of the decode's splits


def _call(name, *args):
    out = (ctypes.c_int * 4)()
    rc = getattr(_lib.load(), name)(*args, out)
    assert rc == _lib.ATTN_OK, f"{name}: {rc}"
    return list(out)


def prefill(attn, hist, chunk):
    """(query heads packed into a tile's rows, pieces per split item, two-piece clusters?, whole items)"""
    heads, pieces, cluster, whole = _call("attn_plan_prefill", attn._ctx, hist, chunk)
    return heads, pieces, bool(cluster), whole


def decode(attn, n_new=1):
    """(splits per item, merge mode)"""
    return tuple(_call("attn_plan_decode", attn._ctx, n_new)[:2])


def gemv(M, N, K, rms=False):
    """(rows of the first launch, CTAs per cluster or 1 for the plain kernel, rounds, warps per unit)"""
    return tuple(_call("attn_plan_w4bf16", 0, M, N, K, int(rms)))


def gemm(T, N, K):
    """(tokens per tile, pairs that share a tile's K, tiles, clusters of the grid)"""
    return tuple(_call("attn_plan_w4bf16", 1, T, N, K, 0))
