"""The RoPE table rows that flash_fwd's threads load (csrc/flash_rows.h, compiled here for the
host): every one lies in [0, max_len), also where a pair's second query tile is past the chunk
and the chunk ends at max_len, with and without packed heads.
"""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_15865_gb300", "csrc")
SRC = '#include "flash_rows.h"\nextern "C" int pos(int r, int n, int k, int p) { return attn::rope_table_pos(r, n, k, p); }\n'


@pytest.fixture(scope="module")
def pos(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("rows") / "rows.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-x", "c++", "-", "-o", so], input=SRC, text=True,
                   check=True)
    return ctypes.CDLL(so).pos


@pytest.mark.parametrize("heads", [1, 2, 5, 7, 16])
@pytest.mark.parametrize("hist,chunk", [(0, 1), (0, 16), (16, 8), (500, 100), (0, 128), (7, 129), (100, 300), (0, 640)])
def test_rope_rows_stay_in_the_tables(pos, heads, hist, chunk):
    if heads > 1 and chunk > 128:
        pytest.skip("longer chunks are never packed")
    max_len, tok = hist + chunk, 128 // heads
    for q0 in range(0, -(-chunk // tok) * tok + tok, tok):  # one tile past the last: the pair's absent one
        rows = max(0, min(tok, chunk - q0)) * heads
        for row in range(128):
            p = pos(row, rows, row // heads, hist + q0)
            assert 0 <= p < max_len, (q0, row)
            assert row >= rows or p == hist + q0 + row // heads
