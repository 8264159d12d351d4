// flash_rows.h -- where a row of a query tile lies, as plain C++ (host tests include it too).
#pragma once

#ifdef __CUDACC__
#define ATTN_HD __host__ __device__ __forceinline__
#else
#define ATTN_HD inline
#endif

namespace attn {

// Position whose row of the RoPE tables the thread of tile row `row` loads.  pos0: position of the
// tile's first token, row_tok: the row's token from there.  A row past the tile's `rows` rotates
// nothing and loads position 0: its own position, and for a tile wholly past the chunk also pos0,
// may lie past the tables' last row (a chunk that ends at max_len).
ATTN_HD int rope_table_pos(int row, int rows, int row_tok, int pos0) { return row < rows ? pos0 + row_tok : 0; }

}  // namespace attn
