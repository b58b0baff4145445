// Where a CTA of the one-launch training step (k_tr_chain) stages the
// transposed tile of a product for its bulk stores, as a plain function that
// the launch lays out and a host check goes through (tests/test_chain_tiles.py).
#pragma once

#if defined(__CUDACC__)
#define LS_CHAIN_FN __host__ __device__ __forceinline__ constexpr
#else
#define LS_CHAIN_FN inline constexpr
#endif

namespace ls {
namespace chain {

// K-blocks (of 64 columns) of the operand that a product of NT columns a CTA
// leaves for the next one: CTA `rank` writes blocks [first, first + NT / 64) of
// both ranks' copies.
LS_CHAIN_FN int first_block(int rank, int NT) { return rank * (NT / 64); }

// First K-block, in the operand copy that a product of NT columns a CTA has
// just read, of its transposed tile (NT / 64 blocks); the next product has
// NT_next columns a CTA (NT again after the last one).  The other CTA of a
// cluster may be an epilogue ahead: once it has this CTA's columns it stores
// those of the next product into the same copy, while the bulk stores still
// read the tile.  So the tile keeps out of the other's blocks of the next
// product; with layers of one width those are simply not this CTA's own.  The
// widths of a cluster of two are 128 and 256, the copy as wide as the widest
// layer, so what does not fit in front of the other's blocks fits behind them.
LS_CHAIN_FN int stage_block(int CL, int rank, int NT, int NT_next) {
  if (CL == 1) return 0;
  if (rank == 1) return first_block(1, NT_next);  // rank 0 writes the blocks before
  return NT <= NT_next ? 0 : 2 * (NT_next / 64);  // rank 1 writes [NT_next / 64, 2 NT_next / 64)
}

}  // namespace chain
}  // namespace ls
