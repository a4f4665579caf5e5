// A run of stride-1 3x3 convolutions of at most 16 channels on images 32 pixels wide - the first stage of a CIFAR-shaped network - as
// one kernel, activations in shared memory from the run's input to its output, like chain_tc.cu, with another view of the convolution.
//
//   What bounds chain_tc.cu here.  With 16 filters it stacks the three horizontal taps along N and adds them up in the epilogue: 48
//   accumulator columns and 32 shuffles for 16 values, a chain of some 2400 cycles per 128 pixels, four of which are in flight: 520
//   cycles a tile of 128 pixels, against 130 of its MMAs.  Here the tensor pipe does the adding and the epilogue is the shorter half.
//   GEMM view     A row is a block of 2 x 2 pixels, N = 4 pixels x 16 filters, K = the 4 x 4 pixels the block's windows cover x 16 channels:
//                 16 MMAs of M 128, N 64, K 16 for 512 pixels.  28 of the 16 x 4 (pixel, output) places are outside the output's window
//                 (7 of its 16 pixels each) and hold zero filters; an MMA of N = 64 costs the pipe little more than one of N = 16 (48 cycles against 39, the fetch of
//                 the 128 x 16 operand), so that is 192 cycles per 128 pixels where nine MMAs of N = 16 take 350.
//   Layout        planar-8 per parity: plane (row parity, column parity, chunk) holds the blocks' pixels of that parity at
//                 img * (H/2 + 1)(W/2 + 1) + (i + 1)(W/2 + 1) + (j + 1), zeros above and to the left of an image and behind the last.
//                 Window row iy = 0 .. 3 is row parity 1, 0, 1, 0 at -1, 0, 0, +1 block rows, columns alike: an operand is a plane from a
//                 start row, its two 8-channel halves a plane apart.
//   Epilogue      a thread has a block: 64 columns, of 16 each shift, shortcut, ReLU, two 16-byte vectors.  No neighbours, no masks but
//                 the border's, and additions two at a time.
//   Filters       32 KB a layer, [window pixel][2 chunks][4 outputs x 16 filters][8], a double buffer; the 16 shifts behind them.
//   Roles         sixteen warps load, finish and store, every fourth tile each four; four issue the MMAs, every fourth tile each, and
//                 bring the filters.  Tiles are numbered through the layers, so all have the same to do.
//   Order         16 MMAs, a commit and four barriers are 1900 cycles of a warp's own, 770 of the pipe's; two issuing warps left the
//                 pipe waiting (5700 cycles for a layer of five tiles), four at will share it, so that all tiles of a layer end together and
//                 the next layer's begin when the last epilogue is through (5600).  So four wait and commit side by side, but issue
//                 in the tiles' order (5000).
//   Pipelining    as chain_tc.cu: eight accumulator stages, a barrier pair per tile says when its outputs are there, layers overlap.
//   Measured      ResNet-110's 37 layers of 1024 images 695 -> 400 us, of 148 images 105 -> 88 us (a layer of one image's three tiles is
//                 4500 cycles, of two images' five 5100: the chain of MMAs, commit and epilogue behind a tile's neighbours).
//   Not finite    An infinity or a NaN reaches every output of the blocks whose 4 x 4 pixels hold it, also those it is multiplied by a zero
//                 filter for.  It stays within its image: above, below and between images' columns lie zeros.
//   Waits         bounded as in conv_tc.cu.
#include "chain_quad_layout.h"
#include "fp_internal.h"
#include "tc_common.cuh"

#include <cstdio>
#include <cstring>

namespace fp {

namespace {

using namespace tc;

constexpr int kN = 64, kStages = kQuadStages, kIssuers = 4, kGroups = 4, kWindow = 16;
constexpr int kFilterBytes = kQuadFilterBytes, kBlobBytes = kQuadBlobBytes;
constexpr int kIssuer0 = 4 * kGroups, kThreads = 32 * (kIssuer0 + kIssuers);
constexpr int kHandOver = 6;                             // the MMA behind which the next warp may begin: it needs some 400 cycles to get there
constexpr int kMaxTiles = kQuadMaxTiles;

struct QuadParams {
    ChainArgs a;
    FastDiv div_image, div_pitch;
    int G, tiles, n_groups, pitch, image, rows;          // blocks of a row and of an image, borders included; vectors of a plane in shared memory
    int Wp, P2;
    long long plane_in, plane_out;
    int* status;
};

// two fp32 additions in one instruction
__device__ __forceinline__ unsigned long long pair_of(uint32_t lo, uint32_t hi) { return (unsigned long long)hi << 32 | lo; }
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__global__ void __launch_bounds__(kThreads, 1) chain_quad_kernel(const __grid_constant__ QuadParams p) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    QuadCtrl* ctrl = reinterpret_cast<QuadCtrl*>(smem_raw);
    const uint32_t base = smem_u32(smem_raw);
    const uint32_t w0 = (base + (uint32_t)sizeof(QuadCtrl) + 127u) & ~127u;
    const uint32_t act0 = w0 + 2u * kBlobBytes, plane_bytes = (uint32_t)p.rows * 16u, buf_bytes = 8u * plane_bytes;
    uint8_t* const act = smem_raw + (act0 - base);
    const uint32_t w_full0 = base + (uint32_t)offsetof(QuadCtrl, w_full), w_empty0 = base + (uint32_t)offsetof(QuadCtrl, w_empty);
    const uint32_t sum_full0 = base + (uint32_t)offsetof(QuadCtrl, sum_full), sum_empty0 = base + (uint32_t)offsetof(QuadCtrl, sum_empty);
    const uint32_t done0 = base + (uint32_t)offsetof(QuadCtrl, tile_done), group_sync = base + (uint32_t)offsetof(QuadCtrl, group_sync);
    volatile int* abort_flag = &ctrl->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, L = p.a.n_layers, tiles = p.tiles;

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(w_full0 + 8 * s, 1);
            mbar_init(w_empty0 + 8 * s, kIssuers + 4 * kGroups);
        }
        for (int s = 0; s < kStages; ++s) {
            mbar_init(sum_full0 + 8 * s, 1);
            mbar_init(sum_empty0 + 8 * s, 128);
        }
        for (int t = 0; t < 2 * kMaxTiles; ++t) mbar_init(done0 + 8 * t, 128);
        mbar_init(group_sync, 128 * kGroups);
        ctrl->abort_flag = 0;
        ctrl->next_tile = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __shared__ ChainLayer layers[kChainMaxLayers];       // (see chain_tc.cu)
    for (int i = threadIdx.x; i < L * (int)(sizeof(ChainLayer) / 4); i += kThreads)
        reinterpret_cast<int*>(layers)[i] = reinterpret_cast<const int*>(p.a.layers)[i];
    // The second buffer's border stays zero: epilogues write pixels alone.  (The first one is written whole by every load.)
    for (int i = threadIdx.x; i < 8 * p.rows; i += kThreads) *reinterpret_cast<uint4*>(act + buf_bytes + (uint32_t)i * 16u) = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (warp == kIssuer0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(base + (uint32_t)offsetof(QuadCtrl, tmem_base)), "r"((uint32_t)(kStages * kN)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&ctrl->tmem_base);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (warp < kIssuer0) asm volatile("griddepcontrol.wait;" ::: "memory");            // (the other warps touch filters and shared memory only)

    auto wait_all = [&](uint32_t bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag)) != 0; };
    // `it` numbers the layers of all groups.  Tile t's input of layer `it` is there when barrier (it & 1, t) has completed its
    // (it / 2)th phase: by the load before a group's first layer, by the layer before for the others.
    auto done = [&](uint32_t it, int t) { return done0 + 8u * ((it & 1u) * kMaxTiles + (uint32_t)t); };
    bool ok = true;
    uint32_t it = 0;
    if (warp >= kIssuer0) {
        // ------------------------------ MMAs and filters ------------------------------
        const uint32_t leader = elect_one(), turn = (uint32_t)(warp - kIssuer0);
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kN >> 3) << 17) | ((128u >> 4) << 24);
        const uint32_t rows = (uint32_t)p.rows, pitch = (uint32_t)p.pitch;
        volatile uint32_t* next_tile = &ctrl->next_tile;
        auto bring_filters = [&](uint32_t n, int l) {        // of layer n, the group's l-th
            const uint32_t wb = n & 1, bar = w_full0 + 8 * wb;
            if (!wait_all(w_empty0 + 8 * wb, ((n >> 1) & 1) ^ 1)) return false;
            if (lane == 0) mbar_expect_tx(bar, kBlobBytes);
            __syncwarp();
            const uint8_t* src = reinterpret_cast<const uint8_t*>(p.a.w) + layers[l].blob_off;
            if (lane * 8192 < kBlobBytes)
                bulk_copy(w0 + wb * kBlobBytes + (uint32_t)lane * 8192u, src + lane * 8192, (uint32_t)min(8192, kBlobBytes - lane * 8192), bar);
            __syncwarp();
            return true;
        };
        if (turn == 0) ok = bring_filters(0, 0);
        uint32_t q = 0;
        for (int g = blockIdx.x; g < p.n_groups && ok; g += gridDim.x)
            for (int l = 0; l < L && ok; ++l, ++it) {
                const uint32_t wb = it & 1, ph = (it >> 1) & 1;
                if (!(ok = wait_all(w_full0 + 8 * wb, ph))) break;
                const uint32_t b0 = ((w0 + wb * kBlobBytes) >> 4) | ((uint32_t)kN << 16);
                const uint32_t a0 = ((act0 + (uint32_t)(l & 1) * buf_bytes) >> 4) | (rows << 16);
                // The next layer's filters go where the layer before had its own, by the warp whose tile here comes last: that layer's
                // MMAs are over before it is due.  (No warp has skipped more than one use of a buffer without a wait for its filters.)
                if ((q + kIssuers - 1) % kIssuers == turn && (l + 1 < L || g + (int)gridDim.x < p.n_groups) &&
                    !(ok = bring_filters(it + 1, l + 1 < L ? l + 1 : 0))) break;
                for (int t = 0; t < tiles; ++t, ++q) {
                    if (q % kIssuers != turn) continue;
                    const uint32_t stage = q % kStages;
                    ok = wait_all(sum_empty0 + 8 * stage, ((q / kStages) & 1) ^ 1) && (t == 0 || wait_all(done(it, t - 1), ph)) &&
                         wait_all(done(it, t), ph) && (t + 1 == tiles || wait_all(done(it, t + 1), ph));
                    if (!ok) break;
                    for (uint32_t spins = 0; *next_tile != q; ++spins)
                        if ((spins & 255) == 255 && (*abort_flag || spins > kWaitLimit)) { ok = false; break; }
                    ok = __all_sync(0xffffffffu, ok) != 0;
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d = tmem + stage * (uint32_t)kN, at = a0 + (uint32_t)(t * 128);
#pragma unroll
                    for (int w = 0; w < kWindow; ++w) {
                        // The plane of the window pixel's parity, from the block row and column it lies in: quad_window_plane and quad_window_row,
                        // written out.  (As calls they compile to a slower order of the same work: the 37 layers below 400.5 -> 416.3 us.)
                        const int iy = w >> 2, ix = w & 3;
                        const uint32_t plane = (uint32_t)((((iy + 1) & 1) * 2 + ((ix + 1) & 1)) * 2) * rows;
                        const uint32_t row = (iy == 0 ? 0u - pitch : iy == 3 ? pitch : 0u) + (ix == 0 ? 0u - 1u : ix == 3 ? 1u : 0u);
                        umma_bf16_lo_if(leader, d, at + plane + row, b0 + (uint32_t)(w * 2 * kN), idesc, w ? 1u : 0u);
                        if (w == kHandOver && leader) *next_tile = q + 1;
                    }
                    if (leader) umma_commit(sum_full0 + 8 * stage);
                    __syncwarp();
                }
                if (ok && leader) umma_commit(w_empty0 + 8 * wb);
                __syncwarp();
            }
        if (!ok && leader) { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 21); }
    } else {
        // ------------------------------ load, finish, store ------------------------------
        const uint32_t mine = (uint32_t)warp >> 2;
        const int quarter = warp & 3, row0 = quarter * 32 + lane, W = p.a.W, H = p.a.H;
        const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16);
        const uint4* xv = reinterpret_cast<const uint4*>(p.a.x);
        uint4* yv = reinterpret_cast<uint4*>(p.a.y);
        struct Block { bool pixels; int n, h, w; };          // of image n, with the pixel (h, w) at its upper left
        auto block_at = [&](int g, int t) {
            Block b;
            const int f = t * 128 + row0, img = (int)fdiv((uint32_t)f, p.div_image), rem = f - img * p.image;
            const int i = (int)fdiv((uint32_t)rem, p.div_pitch), j = rem - i * p.pitch;
            b.n = g * p.G + img;
            b.pixels = img < p.G && b.n < p.a.N && i >= 1 && j >= 1;
            b.h = 2 * (i - 1); b.w = 2 * (j - 1);
            return b;
        };
        uint32_t q = 0, groups_done = 0;
        for (int g = blockIdx.x; g < p.n_groups && ok; g += gridDim.x) {
            if (groups_done) {
                // every MMA and every epilogue of the group before has finished before its buffers are overwritten
                mbar_arrive(group_sync);
                if (!(ok = wait_all(group_sync, (groups_done - 1) & 1))) break;
            }
            ++groups_done;
            // ---- the group's images: every thread its blocks, zeros on the border and behind the last image ----
            uint32_t pixels = 0;                              // bit t: this thread's block of tile t is one of an image
            for (int t = 0; t < tiles; ++t) {
                const Block b = block_at(g, t);
                pixels |= (b.pixels ? 1u : 0u) << t;
                if ((uint32_t)t % kGroups != mine) continue;
                uint4 v[4][2];
#pragma unroll
                for (int o = 0; o < 4; ++o) v[o][0] = v[o][1] = make_uint4(0, 0, 0, 0);
                if (b.pixels && p.a.in_mode == 0) {
#pragma unroll
                    for (int o = 0; o < 4; ++o) {
                        const long long at = (long long)b.n * p.P2 + (long long)(b.h + (o >> 1) + 1) * p.Wp + (b.w + (o & 1) + 1);
                        v[o][0] = xv[at];
                        v[o][1] = xv[at + p.plane_in];
                    }
                } else if (b.pixels) {
                    // two rows of two pixels of every channel, rounded to bf16; four channels' loads in flight
#pragma unroll
                    for (int c0 = 0; c0 < 16; c0 += 4) {
                        if (c0 >= p.a.in_C) break;
                        float x[4][4];
#pragma unroll
                        for (int c = 0; c < 4; ++c)
#pragma unroll
                            for (int o = 0; o < 4; ++o) {
                                const long long e = (((long long)b.n * p.a.in_C + min(c0 + c, p.a.in_C - 1)) * H + b.h + (o >> 1)) * W + b.w + (o & 1);
                                x[c][o] = p.a.in_mode == 1 ? __ldg(reinterpret_cast<const float*>(p.a.x) + e) : __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p.a.x)[e]);
                            }
#pragma unroll
                        for (int o = 0; o < 4; ++o) {
                            const uint32_t lo = pack_bf16x2(x[0][o], c0 + 1 < p.a.in_C ? x[1][o] : 0.0f);
                            const uint32_t hi = pack_bf16x2(c0 + 2 < p.a.in_C ? x[2][o] : 0.0f, c0 + 3 < p.a.in_C ? x[3][o] : 0.0f);
                            uint4& to = v[o][c0 >> 3];
                            if (c0 & 4) { to.z = lo; to.w = hi; } else { to.x = lo; to.y = hi; }
                        }
                    }
                }
                if (t * 128 + row0 < p.rows)
#pragma unroll
                    for (int o = 0; o < 4; ++o)
#pragma unroll
                        for (int c = 0; c < 2; ++c) *reinterpret_cast<uint4*>(act + (uint32_t)(o * 2 + c) * plane_bytes + (uint32_t)(t * 128 + row0) * 16u) = v[o][c];
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            for (int t = (int)mine; t < tiles; t += kGroups) mbar_arrive(done(it, t));
            // ---- the border of the group's images in memory: the row above, the left column, W + 2 zeros behind the last image ----
            const int border = 2 * p.Wp + 1 + H;
            for (int i = (int)threadIdx.x; i < p.G * border * 2; i += 128 * kGroups) {
                const int c = i / (p.G * border), r = i - c * (p.G * border), img = r / border, b = r - img * border, n = g * p.G + img;
                if (n >= p.a.N || (b >= p.Wp + H && n != p.a.N - 1)) continue;
                const int at = b < p.Wp ? b : b < p.Wp + H ? (1 + b - p.Wp) * p.Wp : p.P2 + b - p.Wp - H;
                yv[(long long)c * p.plane_out + (long long)n * p.P2 + at] = make_uint4(0, 0, 0, 0);
            }
            // the next group's images are on their way to L2 by the time it is loaded
            if (p.a.in_mode) {
                const long long image = (long long)p.a.in_C * H * W * (p.a.in_mode == 1 ? 4 : 2), first = ((long long)g + gridDim.x) * p.G;
                const long long bytes = (min((long long)p.a.N, first + p.G) - first) * image;
                for (long long i = 128LL * threadIdx.x; i < bytes; i += 128LL * 128 * kGroups)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const uint8_t*>(p.a.x) + first * image + i));
            }
            // ---- layers ----
            for (int l = 0; l < L && ok; ++l, ++it) {
                const uint32_t wb = it & 1;
                const bool last = l == L - 1, res = layers[l].res != 0, relu = layers[l].relu != 0;
                if (!(ok = wait_all(w_full0 + 8 * wb, (it >> 1) & 1))) break;        // the shifts come with the filters
                const ulonglong2* shift2 = reinterpret_cast<const ulonglong2*>(smem_raw + (w0 - base) + wb * kBlobBytes + kFilterBytes);
                unsigned long long shift[8];                                 // of filters 2 i and 2 i + 1
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const ulonglong2 b = shift2[i];
                    shift[2 * i] = b.x; shift[2 * i + 1] = b.y;
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(w_empty0 + 8 * wb);
                for (int t = 0; t < tiles; ++t, ++q) {
                    if (q % kGroups != mine) continue;
                    const uint32_t stage = q % kStages;
                    const bool inside = (pixels >> t) & 1u;
                    uint8_t* at = act + (uint32_t)((l + 1) & 1) * buf_bytes + (uint32_t)(t * 128 + row0) * 16u;
                    if (!(ok = wait_all(sum_full0 + 8 * stage, (q / kStages) & 1))) break;
                    tc_fence_after();
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        uint32_t v[32];
                        tmem_ld32(taddr + stage * (uint32_t)kN + (uint32_t)(32 * half), v);
                        uint4 r[2][2];
#pragma unroll
                        for (int o = 0; o < 2; ++o)
#pragma unroll
                            for (int c = 0; c < 2; ++c)
                                r[o][c] = res && inside ? *reinterpret_cast<const uint4*>(at + (uint32_t)((2 * half + o) * 2 + c) * plane_bytes) : make_uint4(0, 0, 0, 0);
                        tmem_ld_wait();
                        if (half == 1) {
                            tc_fence_before();
                            mbar_arrive(sum_empty0 + 8 * stage);
                        }
#pragma unroll
                        for (int o = 0; o < 2; ++o)
#pragma unroll
                            for (int c = 0; c < 2; ++c) {
                                const uint32_t rw[4] = {r[o][c].x, r[o][c].y, r[o][c].z, r[o][c].w};
                                uint32_t out[4];
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    const int col = 8 * c + 2 * i;
                                    unsigned long long s = add2(pair_of(v[16 * o + col], v[16 * o + col + 1]), shift[col / 2]);
                                    if (res) s = add2(s, pair_of(rw[i] << 16, rw[i] & 0xffff0000u));
                                    const float lo = __uint_as_float((uint32_t)s), hi = __uint_as_float((uint32_t)(s >> 32));
                                    out[i] = relu ? pack_bf16x2_relu(lo, hi) : pack_bf16x2(lo, hi);
                                }
                                const uint4 y = make_uint4(out[0], out[1], out[2], out[3]);
                                if (!last) {
                                    if (inside) *reinterpret_cast<uint4*>(at + (uint32_t)((2 * half + o) * 2 + c) * plane_bytes) = y;
                                } else if (inside) {
                                    const Block b = block_at(g, t);
                                    yv[(long long)c * p.plane_out + (long long)b.n * p.P2 + (long long)(b.h + half + 1) * p.Wp + (b.w + o + 1)] = y;
                                }
                            }
                    }
                    if (!last) {
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        mbar_arrive(done(it + 1, t));
                    }
                }
            }
        }
        if (!ok && lane == 0) { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 22); }
    }

    // ---- teardown: everyone arrives here, also after a wait that ran out ----
    if (*abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);         // copies in flight land before the memory is given back
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == kIssuer0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)(kStages * kN)) : "memory");
    }
}

}  // namespace

// Runs whose layers have 16 filters and channels (padded), on images 32 pixels wide and of even height.  (The first layer may not add a
// tensor: the run's second buffer is not loaded.)  There it was the shorter form at every batch: 37 layers, us of chain_tc.cu -> of
// this one, 32 images 103 -> 86, 149 174 -> 103, 444 234 -> 201, 592 343 -> 201, 1024 695 -> 400.
bool chain_quad_supported(const ChainArgs& a) {
    if (a.W != 32 || a.H % 2 || a.H < 2 || a.res_mode) return false;
    for (int l = 0; l < a.n_layers; ++l)
        if (a.layers[l].K_pad != 16 || a.layers[l].cchunks != 2) return false;
    return quad_smem(1, a.H, a.W) <= kQuadSmemMax;
}

// A layer of one image's 3 tiles takes 2.38 us, of two images' 5 2.75 us: two images a CTA wherever that saves a round.
double chain_quad_layer_us(int tiles) { return 1.84 + 0.183 * tiles; }

int plan_chain_quad(const ChainArgs& a, ChainPlan* plan, char* err, size_t err_len) {
    memset(plan, 0, sizeof(*plan));
    int best = 0;
    double best_cost = 0;
    for (int G = 1; G <= a.N; ++G) {
        const int tiles = quad_tiles(quad_plane_rows(G, a.H, a.W));
        if (quad_smem(G, a.H, a.W) > kQuadSmemMax || tiles > kMaxTiles) break;
        const int groups = (a.N + G - 1) / G;
        const double cost = ((groups + sm_count() - 1) / sm_count()) * chain_quad_layer_us(tiles);
        if (!best || cost <= best_cost) { best = G; best_cost = cost; }
    }
    if (!best || cudaFuncSetAttribute(chain_quad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQuadSmemMax) != cudaSuccess) {
        cudaGetLastError();
        snprintf(err, err_len, "one image does not fit shared memory");
        return 1;
    }
    plan->quad = 1; plan->G = best; plan->plane_rows = quad_plane_rows(best, a.H, a.W);
    plan->tiles = quad_tiles(plan->plane_rows);
    plan->smem_bytes = quad_smem(best, a.H, a.W);
    if (plan->smem_bytes < 120u * 1024u) plan->smem_bytes = 120u * 1024u;      // one CTA per SM: tensor memory is never contended
    plan->valid = 1;
    return 0;
}

void launch_chain_quad(const ChainPlan& plan, const ChainArgs& a, int* d_status, cudaStream_t st) {
    QuadParams p;
    memset(&p, 0, sizeof(p));
    p.a = a;
    p.G = plan.G; p.tiles = plan.tiles; p.rows = plan.plane_rows;
    p.n_groups = (a.N + plan.G - 1) / plan.G;
    p.pitch = quad_pitch(a.W); p.image = (a.H / 2 + 1) * p.pitch;
    p.div_image = make_fastdiv((uint32_t)p.image); p.div_pitch = make_fastdiv((uint32_t)p.pitch);
    p.Wp = row_vecs(a.W); p.P2 = image_vecs(a.H, a.W);
    p.plane_in = p.plane_out = plane_vecs(a.N, a.H, a.W);
    p.status = d_status;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(p.n_groups < sm_count() ? p.n_groups : sm_count()));
    cfg.blockDim = dim3((unsigned)kThreads);
    cfg.dynamicSmemBytes = plan.smem_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    void* args[1] = {(void*)&p};
    cudaLaunchKernelExC(&cfg, (const void*)chain_quad_kernel, args);
}

}  // namespace fp
