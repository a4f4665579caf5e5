// Shared memory of chain_quad.cu: what the launch asks for and the kernel's addresses, apart from both so that the one is checked against the
// other without a GPU (tests/test_chain_quad_layout.py).
#pragma once
#include "fp_internal.h"

namespace fp {

constexpr int kQuadStages = 8, kQuadMaxTiles = 8;
constexpr unsigned kQuadSmemMax = 232448u - 2048u;       // (the layer table is static)

struct QuadCtrl {
    uint64_t w_full[2], w_empty[2], sum_full[kQuadStages], sum_empty[kQuadStages], tile_done[2][kQuadMaxTiles], group_sync;
    uint32_t tmem_base;
    int abort_flag;
    uint32_t next_tile;                                  // whose MMAs are issued next
    int pad_[3];
};
static_assert(sizeof(QuadCtrl) % 16 == 0, "buffers behind the control block must stay 16-byte aligned");

// Vectors of a row of blocks, and of a plane of G images: blocks with their borders, and the zeros behind the last.
constexpr int quad_pitch(int W) { return W / 2 + 1; }
constexpr int quad_plane_rows(int G, int H, int W) { return (G * (H / 2 + 1) * quad_pitch(W) + W / 2 + 2 + 7) / 8 * 8; }
constexpr int quad_tiles(int plane_rows) { return (plane_rows + 127) / 128; }
// Where window pixel w = 4 iy + ix of a block is: the plane of its parity, `rows` vectors a plane, from the block row and column it lies in.
// (The kernel has these two written out.)
constexpr uint32_t quad_window_plane(int w, uint32_t rows) { return (uint32_t)(((((w >> 2) + 1) & 1) * 2 + (((w & 3) + 1) & 1)) * 2) * rows; }
constexpr uint32_t quad_window_row(int w, uint32_t pitch) {
    return ((w >> 2) == 0 ? 0u - pitch : (w >> 2) == 3 ? pitch : 0u) + ((w & 3) == 0 ? 0u - 1u : (w & 3) == 3 ? 1u : 0u);
}
// Two buffers of eight planes, and behind them what the last tile's operands read past the last plane: its rows up to a multiple of 128, and
// a row and a block below them.  (The rows before the first plane lie in the filters.)
constexpr unsigned quad_smem(int G, int H, int W) {
    const unsigned rows = (unsigned)quad_plane_rows(G, H, W), read = (unsigned)quad_tiles((int)rows) * 128u + (unsigned)quad_pitch(W) + 1;
    return (unsigned)sizeof(QuadCtrl) + 128u + 2u * (unsigned)kQuadBlobBytes + (15u * rows + read) * 16u;
}

}  // namespace fp
