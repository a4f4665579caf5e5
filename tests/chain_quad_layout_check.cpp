// Every operand of chain_quad.cu's MMAs, for a group of G images: inside the shared memory the launch asks for and, where its row is a block
// of pixels, inside the plane it is meant to read.
#include "../paper_2010_16165_b200/csrc/chain_quad_layout.h"

#include <cstdio>

using namespace fp;

// 0: all in order, and *tiles_out, *smem_out as the planner has them; 1: the planner does not take it; -1: message
extern "C" int check_chain_quad(int G, int H, int W, int* tiles_out, unsigned* smem_out, char* msg) {
    const int rows = quad_plane_rows(G, H, W), tiles = quad_tiles(rows), pitch = quad_pitch(W), image = (H / 2 + 1) * pitch;
    const unsigned smem = quad_smem(G, H, W);
    *tiles_out = tiles; *smem_out = smem;
    if (smem > kQuadSmemMax || tiles > kQuadMaxTiles) return 1;
    for (unsigned start = 0; start < 128; start += 16) {                // where dynamic shared memory begins, behind a multiple of 128 bytes
        const long long w0 = (long long)(start + sizeof(QuadCtrl) + 127) / 128 * 128, act0 = w0 + 2ll * kQuadBlobBytes, end = (long long)start + smem;
        for (int buf = 0; buf < 2; ++buf)
            for (int t = 0; t < tiles; ++t)
                for (int w = 0; w < 16; ++w)
                    for (int chunk = 0; chunk < 2; ++chunk) {
                        const long long plane = (int32_t)quad_window_plane(w, (uint32_t)rows), shift = (int32_t)quad_window_row(w, (uint32_t)pitch);
                        const long long first = act0 + 16ll * (8ll * buf * rows + plane + (long long)chunk * rows + 128ll * t + shift), last = first + 128 * 16;
                        if (first < w0 || last > end) { snprintf(msg, 200, "buffer %d tile %d window pixel %d: bytes %lld to %lld of %lld to %lld", buf, t, w, first, last, w0, end); return -1; }
                        for (int r = 0; r < 128 && start == 0; ++r) {
                            const int f = 128 * t + r, img = f / image, i = f % image / pitch, j = f % image % pitch;
                            if (img >= G || i == 0 || j == 0) continue;              // no block of pixels: nobody stores its row
                            if (f + shift < 0 || f + shift >= rows) { snprintf(msg, 200, "block (%d, %d) of image %d, window pixel %d: row %lld of %d", i, j, img, w, f + shift, rows); return -1; }
                        }
                    }
    }
    return 0;
}
