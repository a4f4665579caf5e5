// A whole CIFAR-shaped residual network - every 3x3 convolution, shortcut, the average pooling and the FC layer - as ONE
// kernel: a CTA (or, for few images, a cluster of two or four CTAs that share an image by rows) carries its images from
// the NCHW input to the logits with the activations in shared memory.  Only the input, the filters and the logits touch
// global memory, and there is one launch.
//
//   Why mma.sync and not tcgen05 here.  These layers are 8 to 64 channels wide.  A tcgen05.mma of 128 positions x 16
//   channels needs 39-59 cycles for its operand fetch whatever N <= 48 is, which at N = 16 is 560-840 FMA per cycle and SM,
//   and its results come back through tensor memory about a thousand cycles after the issue; a run of such layers is bound
//   by that round trip (chain_tc.cu: 2400 cycles per tile and layer, four tiles in flight).  mma.sync m16n8k16 runs at
//   1018 FMA per cycle and SM with 20 cycles of latency (measured, 8 warps), takes filters in steps of 8 instead of 16,
//   and leaves its results in the registers of the warp that finishes them.
//
//   Activations   planar-8: [chunk of 8 channels][row][pixel], one 16-byte vector per pixel and chunk, row pitch W + 1 (a
//                 zero vector before every row is also the one behind the row above), a zero or halo row above and below:
//                 ldmatrix takes eight pixels' vectors as they lie, at any row and column offset, without conflicts.
//   GEMM view     M = 16 pixels (half an image row of 32, a row of 16, two rows of 8), N = 8 filters, K = 16 channels of one
//                 tap.  Filters arrive as [tap][chunk][filter][8] by bulk copies, one or two layers ahead of their use.
//   Two forms     width >= 16: a warp takes four rows of a column strip and 16 filters, keeps the filters of 16 input
//                 channels (all nine taps) in registers and reads an input row's fragments once for the three output rows
//                 they touch.  Width 8: a warp owns 1-2 pairs of rows and 8-32 filters and streams the filters'
//                 fragments from shared memory, activations still read once for three taps.  A result's order of
//                 summation depends on the layer alone, so it does not depend on the batch it was computed in.
//   Clusters      an image's rows are split over the CTAs; a CTA also sends the first and last row of its result into its
//                 neighbours' halo rows (st.async to distributed shared memory, counted on a barrier there).
#include "fp_internal.h"
#include "tc_common.cuh"

#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>
#include <type_traits>
#include <vector>

namespace fp {

namespace {

using namespace tc;

constexpr int kWarps = 8;                       // computing warps per image
constexpr int kThreads = 32 * kWarps;           // threads per image
constexpr int kMaxG = kNetMaxG;                 // images a CTA carries at a time, each by eight warps of its own
constexpr int kLayerCode = 21, kHaloCode = 22;  // status words: a layer's filters / the neighbours' rows did not come
constexpr int kRing = 4;                        // layers whose descriptor (and filters) can be on the way or in use

struct NetCtrl {
    uint64_t full[kRing];
    uint64_t halo[2];                           // clusters: the neighbours' rows of an even / odd layer's result are here
    NetLayer layer[kRing];
    int done[kRing];                            // images that are through with a layer
    int abort_flag;
    int pad_[3];
};
static_assert(((sizeof(NetCtrl) + 127) & ~(size_t)127) + 128 == (size_t)kNetCtrlBytes, "the planner leaves this much for it, alignment included");
static_assert(sizeof(NetLayer) % 16 == 0 && sizeof(NetCtrl) % 16 == 0, "bulk copies need 16-byte alignment");

struct NetParams {
    NetArgs a;
    const NetLayer* table;
    int G, cs, L, img_bytes, n_clusters;
    int in_off, in_rows;                        // slab of the network input: rows per CTA
    int head_off, last_off, last_PV, first_requests;
    int* status;
};

__device__ __forceinline__ void ldm4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldm2(uint32_t (&r)[2], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}
__device__ __forceinline__ void ldm_filters(uint32_t (&r)[4], uint32_t addr) { ldm4(r, addr); }     // 16 filters
__device__ __forceinline__ void ldm_filters(uint32_t (&r)[2], uint32_t addr) { ldm2(r, addr); }     // 8 filters
__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v) { asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ void sts128_zero(uint32_t addr) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "r"(0) : "memory");
}
__device__ __forceinline__ uint32_t remote(uint32_t addr, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// the same, counted in bytes on a barrier of the CTA it goes to
__device__ __forceinline__ void st_async32(uint32_t addr, uint32_t v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_remote32(uint32_t addr, uint32_t v) { asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
// acc + the lower / upper bf16 of a pair: one instruction, one rounding
__device__ __forceinline__ void add_pair(float& lo, float& hi, uint32_t v) {
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\tadd.rn.f32.bf16 %0, l, %0;\n\tadd.rn.f32.bf16 %1, h, %1;\n\t}" : "+f"(lo), "+f"(hi) : "r"(v));
}
__device__ __forceinline__ float bf_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

// ends a layer: all warps of an image in this CTA
template <int WARPS>
__device__ __forceinline__ void layer_sync(int slot) { asm volatile("bar.sync %0, %1;" ::"r"(slot + 1), "n"(32 * WARPS) : "memory"); }
// all CTAs that share the image
template <bool CLUSTER, int WARPS>
__device__ __forceinline__ void image_sync(int slot) {
    if (CLUSTER) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else layer_sync<WARPS>(slot);
}

// What a warp needs to know of a layer to finish a tile.
struct Out {
    uint32_t plane, pitch;  // bytes per output chunk plane and row
    uint32_t slab;          // bytes of this CTA's rows of a plane: R * pitch
    int relu;
    uint32_t bias;          // address of the fp32 shifts
    int R, rank, cs, res_mode;
    uint32_t halo;          // clusters: barrier that this layer's rows for the neighbours are counted on
    int turn;               // > 0: two images take turns on the tensor pipe; this image's barrier (the other's is 7 - turn)
    uint32_t res;           // option A: address of the shortcut operand, its plane and row strides, first channel, channels
    uint32_t res_plane, res_pitch;
    int res_pad_lo, res_C;
};

// Finishes M tiles of NT x 8 filters: of tile m, accumulator rows 0-7 are this lane's word `dst` + m * step of the first
// chunk, rows 8-15 lie `half` bytes further on.  The bias is already in the accumulator.  res_mode 1: the tensor two layers back
// lies where the result goes - all of its words are read before the first result is written; 2: every second pixel of
// it, channel k from k - pad_lo.  row: first output row, W8: a tile is two rows (else one), x: column of rows 0-7.
template <bool CLUSTER, int M, int NT, bool W8>
__device__ __forceinline__ void finish(const Out& o, float (&acc)[M][NT][4], int n8, uint32_t dst, uint32_t step, uint32_t half, int row, int x, int t) {
    uint32_t v[M][NT][2];
    if (o.res_mode) {
        if (o.res_mode == 1) {
#pragma unroll
            for (int m = 0; m < M; ++m)
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) v[m][j][hh] = lds32(dst + (uint32_t)m * step + (uint32_t)j * o.plane + hh * half);
        } else {
#pragma unroll
            for (int m = 0; m < M; ++m)
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const int c0 = (n8 + j) * 8 + 2 * t - o.res_pad_lo, c1 = c0 + 1;
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        const int rr = W8 ? row + 2 * m + hh : row + m, xx = W8 ? x : x + 8 * hh;
                        const uint32_t p = o.res + (uint32_t)(2 * rr + 1) * o.res_pitch + (uint32_t)(2 * xx + 1) * 16u;
                        uint32_t lo = 0u, hi = 0u;
                        if (c0 >= 0 && c0 < o.res_C) lo = lds32(p + (uint32_t)(c0 >> 3) * o.res_plane + (uint32_t)((c0 & 6) * 2)) >> (16 * (c0 & 1));
                        if (c1 >= 0 && c1 < o.res_C) hi = lds32(p + (uint32_t)(c1 >> 3) * o.res_plane + (uint32_t)((c1 & 6) * 2)) >> (16 * (c1 & 1));
                        v[m][j][hh] = (lo & 0xffffu) | (hi << 16);
                    }
                }
        }
#pragma unroll
        for (int m = 0; m < M; ++m)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) add_pair(acc[m][j][2 * hh], acc[m][j][2 * hh + 1], v[m][j][hh]);
    }
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) v[m][j][hh] = pack_bf16x2_relu(acc[m][j][2 * hh], acc[m][j][2 * hh + 1]);
    if (!o.relu) {
#pragma unroll
        for (int m = 0; m < M; ++m)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) v[m][j][hh] = pack_bf16x2(acc[m][j][2 * hh], acc[m][j][2 * hh + 1]);
    }
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) sts32(dst + (uint32_t)m * step + (uint32_t)j * o.plane + hh * half, v[m][j][hh]);
    if (CLUSTER) {
        // the neighbours' halo rows: our first row is row R of the CTA above, our last row is row -1 of the CTA below
        const bool first = o.halo && row == 0 && o.rank > 0, last = o.halo && row + (W8 ? 2 * M : M) == o.R && o.rank + 1 < o.cs;
        if (first) {
            const uint32_t d = remote(dst + o.slab, o.rank - 1), bar = remote(o.halo, o.rank - 1);
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                st_async32(d + (uint32_t)j * o.plane, v[0][j][0], bar);
                if (!W8) st_async32(d + (uint32_t)j * o.plane + half, v[0][j][1], bar);
            }
        }
        if (last) {
            const uint32_t d = remote(dst + (uint32_t)(M - 1) * step - o.slab, o.rank + 1), bar = remote(o.halo, o.rank + 1);
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                if (!W8) st_async32(d + (uint32_t)j * o.plane, v[M - 1][j][0], bar);
                st_async32(d + (uint32_t)j * o.plane + half, v[M - 1][j][1], bar);
            }
        }
    }
}

// Two images of a CTA, eight warps each, take strict turns: while one issues its MMAs, the other finishes its tile, ends its
// layer and gets ready for the next.  (Left to themselves both went through the same phases at the same time, and the tensor
// pipe stood still in the phases without MMAs: ResNet-56's first stage 8000 cycles a layer and pair of images.)  A turn is
// given away a row of MMAs before its end, so that the other image's loads are on the way when the pipe falls free.
template <bool CLUSTER>
__device__ __forceinline__ void take_turn(const Out& o) {
    if (!CLUSTER && o.turn) asm volatile("bar.sync %0, %1;" ::"r"(o.turn), "n"(2 * kThreads) : "memory");
}
template <bool CLUSTER>
__device__ __forceinline__ void give_turn(const Out& o) {
    if (!CLUSTER && o.turn) asm volatile("bar.arrive %0, %1;" ::"r"(7 - o.turn), "n"(2 * kThreads) : "memory");
}

__device__ __forceinline__ float2 lds_bias(uint32_t bias, int n8, int t) {
    float2 b;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(b.x), "=f"(b.y) : "r"(bias + (uint32_t)(n8 * 8 + 2 * t) * 4u));
    return b;
}

// RUN rows of a strip of 16 columns and NT x 8 filters (NT 1 or 2): per 16 input channels the nine taps' filters are read
// into registers once, and every input row's fragments feed the up to three output rows they touch.  `a0`: this lane's
// ldmatrix address of (input row `row` - 1, strip's first column), `b0`: of the filters, `dst`: its word of the first output row.
template <bool CLUSTER, int RUN, int NT>
__device__ __forceinline__ void conv_strip(const Out& o, uint32_t a0, uint32_t row_step, uint32_t k_step, int kc_n, uint32_t b0, uint32_t b_tap,
                                           uint32_t b_k, int row, int x, int n8, uint32_t dst, int lane) {
    const int t = lane & 3;
    float acc[RUN][NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const float2 b = lds_bias(o.bias, n8 + j, t);
#pragma unroll
        for (int q = 0; q < RUN; ++q) { acc[q][j][0] = acc[q][j][2] = b.x; acc[q][j][1] = acc[q][j][3] = b.y; }
    }
#pragma unroll 1
    for (int kc = 0; kc < kc_n; ++kc) {
        uint32_t w[9][2 * NT];
#pragma unroll
        for (int i = 0; i < RUN + 2; ++i) {                    // input row `row` - 1 + i
            uint32_t f[3][4];
            if (i < 3) {
#pragma unroll
                for (int s = 0; s < 3; ++s) ldm_filters(w[3 * i + s], b0 + (uint32_t)(3 * i + s) * b_tap);
            }
#pragma unroll
            for (int s = 0; s < 3; ++s) ldm4(f[s], a0 + (uint32_t)i * row_step + (uint32_t)s * 16u);
            if (i == 0 && kc == 0) take_turn<CLUSTER>(o);
            if (i == RUN + 1 && kc == kc_n - 1) give_turn<CLUSTER>(o);
#pragma unroll
            for (int s = 0; s < 3; ++s)
#pragma unroll
                for (int r = 0; r < 3; ++r)
                    if (i - r >= 0 && i - r < RUN) {
#pragma unroll
                        for (int j = 0; j < NT; ++j)
                            mma16816(acc[i - r][j], f[s][0], f[s][1], f[s][2], f[s][3], w[3 * r + s][2 * j], w[3 * r + s][2 * j + 1]);
                    }
        }
        a0 += k_step;
        b0 += b_k;
    }
    finish<CLUSTER, RUN, NT, false>(o, acc, n8, dst, o.pitch, 128u, row, x, t);
}

// Images 8 pixels wide: a tile of MT pairs of rows and NT x 8 filters, filters' fragments streamed.  `a0`: this lane's address of the tile's first input row (output row - 1), `b0`: of its filters.
template <bool CLUSTER, int MT, int NT>
__device__ __forceinline__ void conv_tile(const Out& o, uint32_t a0, uint32_t row_step, uint32_t k_step, int kc_n, uint32_t b0, uint32_t b_tap,
                                          uint32_t b_k, int row, int n8, uint32_t dst, int lane) {
    const int t = lane & 3;
    float acc[MT][NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const float2 b = lds_bias(o.bias, n8 + j, t);
#pragma unroll
        for (int m = 0; m < MT; ++m) { acc[m][j][0] = acc[m][j][2] = b.x; acc[m][j][1] = acc[m][j][3] = b.y; }
    }
    constexpr int NF = MT + 1;                        // fragments that cover the tile's input rows
    constexpr int NB = (NT + 1) / 2;
    // nine (s, r) steps per 16 channels; a step's filters are fetched during the step before, a column's activations
    // during the last row of the column before
    uint32_t f[2][NF][4], b[2][NB][4];
    auto load_f = [&](uint32_t (&d)[NF][4], uint32_t at) {
#pragma unroll
        for (int q = 0; q < NF; ++q) ldm4(d[q], at + (uint32_t)(2 * q) * row_step);
    };
    auto load_b = [&](uint32_t (&d)[NB][4], uint32_t at) {
#pragma unroll
        for (int q = 0; q < NB; ++q) ldm4(d[q], at + (uint32_t)q * 256u);
    };
    load_f(f[0], a0);
    load_b(b[0], b0);
    take_turn<CLUSTER>(o);
    auto turn = [&](auto P, bool more) {              // one group of 16 channels; P: the buffer its first step reads (nine steps: it alternates)
        constexpr int p = decltype(P)::value;
#pragma unroll
        for (int s = 0; s < 3; ++s)
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const int k = 3 * s + r;
                uint32_t (&bc)[NB][4] = b[(k + p) & 1];
                uint32_t (&fc)[NF][4] = f[(s + p) & 1];
                if (k < 8) {
                    const int ns = (k + 1) / 3, nr = (k + 1) % 3;
                    load_b(b[(k + 1 + p) & 1], b0 + (uint32_t)(3 * nr + ns) * b_tap);
                    if (r == 1 && s < 2) load_f(f[(s + 1 + p) & 1], a0 + (uint32_t)(s + 1) * 16u);
                } else if (more) {
                    load_b(b[(k + 1 + p) & 1], b0 + b_k);
                }
                if (k == 7 && more) load_f(f[(3 + p) & 1], a0 + k_step);
                if (k == 7 && !more) give_turn<CLUSTER>(o);
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    uint32_t x[4];
                    if (r == 1) {              // rows 2m+1 and 2m+2: the lower half of one fragment, the upper of the next
                        x[0] = fc[m][1]; x[1] = fc[m + 1][0]; x[2] = fc[m][3]; x[3] = fc[m + 1][2];
                    } else {
#pragma unroll
                        for (int e = 0; e < 4; ++e) x[e] = fc[m + r / 2][e];
                    }
#pragma unroll
                    for (int j = 0; j < NT; ++j) mma16816(acc[m][j], x[0], x[1], x[2], x[3], bc[j / 2][2 * (j & 1)], bc[j / 2][2 * (j & 1) + 1]);
                }
            }
        a0 += k_step;
        b0 += b_k;
    };
#pragma unroll 1
    for (int kc = 0; kc < kc_n; kc += 2) {
        turn(std::integral_constant<int, 0>(), kc + 1 < kc_n);
        if (kc + 1 < kc_n) turn(std::integral_constant<int, 1>(), kc + 2 < kc_n);
    }
    finish<CLUSTER, MT, NT, true>(o, acc, n8, dst, 2u * o.pitch, o.pitch, row, lane >> 2, t);
}

// 16 output pixels of a stride-2 layer and NT x 8 filters.
template <bool CLUSTER, int NT, bool W8>
__device__ __forceinline__ void conv_strided(const Out& o, uint32_t a0, uint32_t row_step, uint32_t k_step, int kc_n, uint32_t b0,
                                             uint32_t b_tap, uint32_t b_k, int row, int x, int n8, uint32_t dst, int lane) {
    const int t = lane & 3;
    float acc[1][NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const float2 b = lds_bias(o.bias, n8 + j, t);
        acc[0][j][0] = acc[0][j][2] = b.x; acc[0][j][1] = acc[0][j][3] = b.y;
    }
    take_turn<CLUSTER>(o);
#pragma unroll 1
    for (int kc = 0; kc < kc_n; ++kc) {
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                uint32_t f[4], b[(NT + 1) / 2][4];
                ldm4(f, a0 + (uint32_t)r * row_step + (uint32_t)s * 16u);
#pragma unroll
                for (int q = 0; q < (NT + 1) / 2; ++q) ldm4(b[q], b0 + (uint32_t)(3 * r + s) * b_tap + (uint32_t)q * 256u);
#pragma unroll
                for (int j = 0; j < NT; ++j) mma16816(acc[0][j], f[0], f[1], f[2], f[3], b[j / 2][2 * (j & 1)], b[j / 2][2 * (j & 1) + 1]);
            }
        a0 += k_step;
        b0 += b_k;
    }
    give_turn<CLUSTER>(o);
    finish<CLUSTER, 1, NT, W8>(o, acc, n8, dst, 0u, W8 ? o.pitch : 128u, row, x, t);
}

// What is left for a warp whose wait ran out in layer l (`inside`: behind the layer's start) of the round that begins with image n0: it
// raises the status and computes nothing any more - a descriptor that never came must not be followed - but keeps to the barriers and
// turns that others count on, which it knows from the table in global memory, and then ends the thread, so that nothing in the layers'
// way has to ask.  (As a state that every layer asked about, ResNet-20 batch 1 took 36.0 us instead of 33.8, ResNet-56 batch 256 222
// instead of 216; so they take 34.1 and 214.5.)
template <bool CLUSTER, int WARPS>
__device__ __noinline__ void keep_to_barriers(const NetParams& p, int code, int n0, int l, bool inside) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    NetCtrl* ctrl = reinterpret_cast<NetCtrl*>(smem_raw);
    if ((threadIdx.x & 31) == 0) { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, code); }
    __syncwarp();
    const int slot = CLUSTER || WARPS > kWarps ? 0 : (int)threadIdx.x / (32 * WARPS);
    for (;;) {
        int active = 1;
        for (int s = 1; s < p.G; ++s) active += n0 + s * p.n_clusters < p.a.N;
        if (slot < active) {
            for (; l < p.L; ++l, inside = false) {
                const int4 q = __ldg(reinterpret_cast<const int4*>(&p.table[l].form));
                if (!inside) {
                    if (q.w) {
                        if (!CLUSTER && (q.w & 1) && active > 1) asm volatile("bar.sync 5, %0;" ::"n"(2 * kThreads) : "memory");
                        image_sync<CLUSTER, WARPS>(slot);
                    }
                    for (int k = CLUSTER || active == 1 ? 0 : (q.y + WARPS - 1) / WARPS; k > 0; --k) {
                        asm volatile("bar.sync %0, %1;" ::"r"(3 + slot), "n"(2 * kThreads) : "memory");
                        asm volatile("bar.arrive %0, %1;" ::"r"(4 - slot), "n"(2 * kThreads) : "memory");
                    }
                }
                if (CLUSTER && l + 1 == p.L) image_sync<CLUSTER, WARPS>(slot);
                else layer_sync<WARPS>(slot);
                if (l == p.a.dump_layer) layer_sync<WARPS>(slot);
            }
            image_sync<CLUSTER, WARPS>(slot);              // the head's two
            image_sync<CLUSTER, WARPS>(slot);
        }
        n0 += p.n_clusters * p.G;
        if (n0 >= p.a.N) break;
        __syncthreads();
        if (n0 + slot * p.n_clusters < p.a.N) {            // the next round's images: cleared, then read
            image_sync<CLUSTER, WARPS>(slot);
            image_sync<CLUSTER, WARPS>(slot);
        }
        l = 0;
    }
    for (int i = 0; i < 200; ++i) __nanosleep(1000);       // let copies in flight land before shared memory is released
    asm volatile("exit;");
}

// A warp's wait, all lanes with one answer; it ends the warp's work where it runs out.  Where clusters share an image the polling stays
// out of line as well: their layers are the shortest (inlined: ResNet-20 batch 1 34.9 us instead of 34.1).
template <int WARPS>
__device__ __noinline__ void cluster_wait_or_leave(const NetParams& p, uint32_t bar, uint32_t parity, int code, int n0, int l) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    if (!__all_sync(0xffffffffu, mbar_wait(bar, parity, &reinterpret_cast<NetCtrl*>(smem_raw)->abort_flag, p.a.wait_cycles > 0 ? p.a.wait_cycles : kWaitCycles)))
        keep_to_barriers<true, WARPS>(p, code, n0, l, code == kHaloCode);
}
template <bool CLUSTER, int WARPS>
__device__ __forceinline__ void wait_or_leave(const NetParams& p, uint32_t bar, uint32_t parity, int code, int n0, int l, volatile int* abort_flag) {
    if (__all_sync(0xffffffffu, mbar_test_wait(bar, parity))) return;
    if (CLUSTER) {
        cluster_wait_or_leave<WARPS>(p, bar, parity, code, n0, l);
    } else if (!__all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag))) {
        keep_to_barriers<CLUSTER, WARPS>(p, code, n0, l, false);
        __builtin_unreachable();
    }
}

// One layer: the warp's units of work, one after the other.  Everything that does not depend on the lane was worked out by
// the planner: a layer of one image is five thousand cycles, and a division or a chain of address arithmetic in front of
// every unit was a tenth of that.
template <bool CLUSTER, int WARPS>
__device__ __forceinline__ void run_layer(const NetParams& p, const NetLayer& ly, int n0, int l, int res_mode, int turn, uint32_t send, uint32_t wait, uint32_t wait_phase, volatile int* abort_flag,
                                          int form, int units, uint32_t act0, uint32_t img0, int rank, int warp,
                                          int lane) {
    const int4 c0 = *reinterpret_cast<const int4*>(&ly.in_off), c1 = *reinterpret_cast<const int4*>(&ly.row_step);
    const int4 c2 = *reinterpret_cast<const int4*>(&ly.out_plane), c3 = *reinterpret_cast<const int4*>(&ly.a_chunk);
    Out o;
    o.plane = (uint32_t)c2.x; o.pitch = (uint32_t)c2.y; o.slab = (uint32_t)c2.z; o.relu = c2.w;
    o.bias = act0 + (uint32_t)c0.w;
    o.R = c3.w; o.rank = rank; o.cs = p.cs; o.res_mode = res_mode; o.turn = turn; o.halo = send;
    if (res_mode == 2) {
        const int4 c4 = *reinterpret_cast<const int4*>(&ly.res_plane);
        o.res = img0 + (uint32_t)ly.res_off;
        o.res_plane = (uint32_t)c4.x; o.res_pitch = (uint32_t)c4.y; o.res_pad_lo = c4.z; o.res_C = c4.w;
    }
    const uint32_t row_step = (uint32_t)c1.x, k_step = (uint32_t)c1.y, b_k = (uint32_t)c1.z, b_tap = (uint32_t)c1.w;
    const int kc = form >> 8 & 255, run_rows = form >> 16 & 255, w8 = form >> 24;
    // ldmatrix addresses relative to a tile: activations - matrices (pixels 0-7 | 8-15) x (first | second chunk); filters -
    // matrices (first | second chunk) x (filters 0-7 | 8-15)
    const int mi = lane >> 3, mr = lane & 7;
    const uint32_t a_lane = img0 + (uint32_t)c0.x + (uint32_t)((mi >> 1) * c3.x + (mi & 1) * c3.y + mr * c3.z);
    const uint32_t b_lane = act0 + (uint32_t)c0.z + (mi & 1) * (b_k >> 1) + (uint32_t)((mi >> 1) * 128 + mr * 16);
    const uint32_t d_lane = img0 + (uint32_t)c0.y + (uint32_t)((lane >> 2) * 16 + (lane & 3) * 4);
    const int turns = (units + WARPS - 1) / WARPS;
    for (int k = 0, u = warp; k < turns; ++k, u += WARPS) {
        if (u >= units) {                        // nothing for this warp, but the turns go on
            take_turn<CLUSTER>(o);
            give_turn<CLUSTER>(o);
            continue;
        }
        const uint2 un = *reinterpret_cast<const uint2*>(&ly.unit[u]);
        const uint32_t a0 = a_lane + (un.x & 0xffffu) * 16u, dst = d_lane + (un.x >> 16) * 16u;
        const int n8 = (int)(un.y & 255u), nt = (int)(un.y >> 8 & 255u), row = (int)(un.y >> 16 & 255u), x = (int)(un.y >> 24) + (lane >> 2);
        const uint32_t b0 = b_lane + (uint32_t)n8 * 128u;
        if (CLUSTER && wait && (row == 0 || row + run_rows == o.R))
            wait_or_leave<CLUSTER, WARPS>(p, wait, wait_phase, kHaloCode, n0, l, abort_flag);
        switch (form & 255) {
            case NET_STRIP:
#define FP_STRIP(RUN, NT) conv_strip<CLUSTER, RUN, NT>(o, a0, row_step, k_step, kc, b0, b_tap, b_k, row, x, n8, dst, lane)
                if (run_rows == 4) { if (nt == 2) FP_STRIP(4, 2); else FP_STRIP(4, 1); }
                else { if (nt == 2) FP_STRIP(2, 2); else FP_STRIP(2, 1); }
#undef FP_STRIP
                break;
            case NET_TILE:
#define FP_TILE(MT, NT) conv_tile<CLUSTER, MT, NT>(o, a0, row_step, k_step, kc, b0, b_tap, b_k, row, n8, dst, lane)
                if (run_rows == 4) {
                    switch (nt) { case 4: FP_TILE(2, 4); break; case 3: FP_TILE(2, 3); break; case 2: FP_TILE(2, 2); break; default: FP_TILE(2, 1); }
                } else {
                    switch (nt) { case 4: FP_TILE(1, 4); break; case 3: FP_TILE(1, 3); break; case 2: FP_TILE(1, 2); break; default: FP_TILE(1, 1); }
                }
#undef FP_TILE
                break;
            default:
#define FP_STRIDED(NT, W8) conv_strided<CLUSTER, NT, W8>(o, a0, row_step, k_step, kc, b0, b_tap, b_k, row, x, n8, dst, lane)
                    if (w8) { switch (nt) { case 4: FP_STRIDED(4, true); break; case 3: FP_STRIDED(3, true); break; case 2: FP_STRIDED(2, true); break; default: FP_STRIDED(1, true); } }
                    else { switch (nt) { case 4: FP_STRIDED(4, false); break; case 3: FP_STRIDED(3, false); break; case 2: FP_STRIDED(2, false); break; default: FP_STRIDED(1, false); } }
#undef FP_STRIDED
        }
    }
}

__device__ __forceinline__ void zero_bytes(uint32_t addr, int bytes, int tid, int threads) {
    for (int i = tid; i < bytes / 16; i += threads) sts128_zero(addr + (uint32_t)i * 16u);
}

// WARPS: 8, or 16 where an image has a CTA to itself (G = 1).
template <bool CLUSTER, int WARPS>
__global__ void __launch_bounds__(CLUSTER ? kThreads : kMaxG * kThreads, 1) resident_net_kernel(const __grid_constant__ NetParams p) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    NetCtrl* ctrl = reinterpret_cast<NetCtrl*>(smem_raw);
    const uint32_t ctrl_addr = smem_u32(smem_raw);
    const uint32_t act0 = (ctrl_addr + (uint32_t)sizeof(NetCtrl) + 127u) & ~127u;
    uint8_t* const act = smem_raw + (act0 - ctrl_addr);
    volatile int* abort_flag = &ctrl->abort_flag;
    // every image has eight warps and a memory of its own; the images of a CTA share the filters as they come in
    const int lane = threadIdx.x & 31;
    const uint32_t full0 = ctrl_addr + (uint32_t)offsetof(NetCtrl, full);
    const int rank = CLUSTER ? (int)(blockIdx.x % (unsigned)p.cs) : 0;
    const int cluster_id = CLUSTER ? (int)(blockIdx.x / (unsigned)p.cs) : (int)blockIdx.x;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kRing; ++s) { mbar_init(full0 + 8 * s, 1); ctrl->done[s] = 0; }
        for (int s = 0; s < 2; ++s) mbar_init(ctrl_addr + (uint32_t)offsetof(NetCtrl, halo) + 8 * s, 1);
        ctrl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int L = p.L, H = p.a.H, W = p.a.W, dump_layer = p.a.dump_layer;
    uint32_t it = 0;                   // layers run so far, over all rounds
    const uint32_t halo0 = ctrl_addr + (uint32_t)offsetof(NetCtrl, halo);
    uint32_t sent = rank == 1 ? p.a.other_barrier : 0;       // layers whose border rows went to the neighbours (all but a round's last)
    const int neighbours = CLUSTER ? (rank > 0) + (rank + 1 < p.cs) : 0;
    for (int n0 = cluster_id; n0 < p.a.N; n0 += p.n_clusters * p.G) {
        int active = 1;                                    // the last round may have fewer
        for (int s = 1; s < p.G; ++s) active += n0 + s * p.n_clusters < p.a.N;
        constexpr int threads = 32 * WARPS;
        const int slot = CLUSTER || WARPS > kWarps ? 0 : (int)threadIdx.x / threads, tid = (int)threadIdx.x - slot * threads, warp = tid >> 5;
        const int n = n0 + slot * p.n_clusters;            // this image
        const uint32_t img0 = act0 + (uint32_t)(slot * p.img_bytes);
        uint8_t* const img = act + slot * p.img_bytes;
        const uint32_t it0 = it;
        const int turn = active > 1 ? 3 + slot : 0;
        // Requests the descriptor and filters of layer `next` (one warp).  What other threads read or wrote in the place they
        // go to lies behind the barrier just passed.
        auto request = [&](int next, int off, int src, int bytes) {
            const uint32_t ring = (it0 + (uint32_t)next) & (kRing - 1), bar = full0 + 8 * ring;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (lane == 0) {
                mbar_expect_tx(bar, (uint32_t)bytes + (uint32_t)sizeof(NetLayer));
                bulk_copy(ctrl_addr + (uint32_t)offsetof(NetCtrl, layer) + ring * (uint32_t)sizeof(NetLayer), p.table + next, (uint32_t)sizeof(NetLayer), bar);
            }
            __syncwarp();
            for (int o = lane * 16384; o < bytes; o += 32 * 16384)
                bulk_copy(act0 + (uint32_t)(off + o), reinterpret_cast<const uint8_t*>(p.a.w) + src + o, (uint32_t)min(16384, bytes - o), bar);
        };
        __syncthreads();               // the previous round is over
        if (threadIdx.x < 32)
            for (int k = 0; k < p.first_requests; ++k) {
                const int4 q = __ldg(reinterpret_cast<const int4*>(p.table + k));
                request(k, q.x, q.y, q.z);
            }
        if (n >= p.a.N) continue;
        if (turn == 4 && it == 0) asm volatile("bar.arrive 3, %0;" ::"n"(2 * kThreads) : "memory");      // the first image begins
        zero_bytes(img0, p.img_bytes, tid, threads);
        if (it == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
        image_sync<CLUSTER, WARPS>(slot);
        // ---- the network input: NCHW to the first chunk of the input buffer, halo rows included ----
        {
            const int rows = p.in_rows + 2, C = p.a.in_C;
            for (int i = tid; i < rows * W; i += threads) {
                const int w = i % W, rr = i / W, h = rank * p.in_rows + rr - 1;
                if (h < 0 || h >= H) continue;
                const size_t e0 = ((size_t)n * C * H + h) * W + w;
                float v[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    v[c] = 0.0f;
                    if (c < C) v[c] = p.a.in_mode == 1 ? __ldg(reinterpret_cast<const float*>(p.a.x) + e0 + (size_t)c * H * W)
                                                      : __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p.a.x)[e0 + (size_t)c * H * W]);
                }
                uint4 q;
                q.x = pack_bf16x2(v[0], v[1]); q.y = pack_bf16x2(v[2], v[3]); q.z = pack_bf16x2(v[4], v[5]); q.w = pack_bf16x2(v[6], v[7]);
                *reinterpret_cast<uint4*>(img + p.in_off + ((size_t)rr * (W + 1) + w + 1) * 16) = q;
            }
        }
        image_sync<CLUSTER, WARPS>(slot);
        // ---- layers ----
        for (int l = 0; l < L; ++l, ++it) {
            const uint32_t ring = it & (kRing - 1), bar = full0 + 8 * ring, parity = (it / kRing) & 1;
            wait_or_leave<CLUSTER, WARPS>(p, bar, parity, kLayerCode, n0, l, abort_flag);
            const NetLayer& ly = ctrl->layer[ring];
            const int4 q = *reinterpret_cast<const int4*>(&ly.form);         // form, units, res_mode, zero_bytes
            if (q.w) {                                 // another geometry moves in: its borders have to be zero
                // bit 0: the other image may still read filters from that place (plan_net)
                if (!CLUSTER && (q.w & 1) && active > 1) asm volatile("bar.sync 5, %0;" ::"n"(2 * kThreads) : "memory");
                zero_bytes(img0 + (uint32_t)ly.out_off, q.w, tid, threads);
                image_sync<CLUSTER, WARPS>(slot);
            }
            uint32_t send = 0, wait = 0, wait_phase = 0;
            if (CLUSTER) {
                // A layer's border rows are sent as they are finished and counted in bytes on one of two barriers in turn; the
                // pieces of the next layer that touch the border wait for them.  (A neighbour that is a layer ahead writes
                // into a buffer that nobody reads: its rows needed ours of the layer before.)
                if (l > 0) { wait = halo0 + 8 * ((sent - 1) & 1); wait_phase = ((sent - 1) >> 1) & 1; }
                if (l + 1 < L) {
                    send = halo0 + 8 * (sent & 1);
                    // (warp 0 has a piece that touches the border in every layer, so it has waited for this barrier's last use)
                    if (tid == 0) mbar_expect_tx(send, (uint32_t)(neighbours * ly.W * ly.n8 * 16));
                    ++sent;
                }
            }
            run_layer<CLUSTER, WARPS>(p, ly, n0, l, q.z, turn, send, wait, wait_phase, abort_flag, q.x, q.y, act0, img0, rank, warp, lane);
            if (CLUSTER && l + 1 == L) image_sync<CLUSTER, WARPS>(slot);          // (the head's sums may go where other CTAs still read)
            else layer_sync<WARPS>(slot);
            if (l == dump_layer) {                 // diagnostic: this layer's output as a planar-8 tensor with border
                const int H = ly.R * p.cs, out_PV = ly.out_plane / 16;
                uint4* y = reinterpret_cast<uint4*>(p.a.dump);
                for (int i = tid; i < ly.n8 * ly.R * ly.W; i += threads) {
                    const int w = i % ly.W, r = i / ly.W % ly.R, c = i / (ly.W * ly.R);
                    y[(size_t)c * plane_vecs(p.a.N, H, ly.W) + (size_t)n * image_vecs(H, ly.W) + (size_t)(rank * ly.R + r + 1) * row_vecs(ly.W) + w + 1] =
                        *reinterpret_cast<const uint4*>(img + ly.out_off + ((size_t)c * out_PV + (size_t)(r + 1) * (ly.W + 1) + w + 1) * 16);
                }
                layer_sync<WARPS>(slot);
            }
            if (warp == (l & (kWarps - 1))) {          // the image that is through with the layer last makes the request
                const int4 r = *reinterpret_cast<const int4*>(&ly.requests);         // layers to request; the first one's place, source and size
                if (active > 1) {
                    int last = 0;
                    if (lane == 0) {
                        __threadfence_block();
                        last = atomicAdd(&ctrl->done[ring], 1) == active - 1;
                        if (last) { ctrl->done[ring] = 0; __threadfence_block(); }
                    }
                    if (!__shfl_sync(0xffffffffu, last, 0)) continue;
                }
                const int next = ly.next;
                for (int k = 0; k < r.x; ++k) {
                    int4 e = make_int4(r.y, r.z, r.w, 0);
                    if (k) e = __ldg(reinterpret_cast<const int4*>(p.table + next + k));
                    request(next + k, e.x, e.y, e.z);
                }
            }
        }
        // ---- average pooling and FC: sums along the rows into the first CTA, then over rows, then the matrix ----
        {
            const int Wl = p.a.last_W, Rl = p.a.last_H / p.cs, C = p.a.last_chunks * 8;
            const int head = p.head_off + slot * (p.a.last_H + 1) * C * 4;
            float* rows = reinterpret_cast<float*>(act + head);
            for (int i = tid; i < Rl * p.a.last_chunks; i += threads) {
                const int c = i % p.a.last_chunks, r = i / p.a.last_chunks;
                const uint4* v = reinterpret_cast<const uint4*>(img + p.last_off + ((size_t)c * p.last_PV + (size_t)(r + 1) * (Wl + 1) + 1) * 16);
                float s[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) s[e] = 0.0f;
                for (int w = 0; w < Wl; ++w) {
                    const uint4 q = v[w];
                    s[0] += bf_lo(q.x); s[1] += bf_hi(q.x); s[2] += bf_lo(q.y); s[3] += bf_hi(q.y);
                    s[4] += bf_lo(q.z); s[5] += bf_hi(q.z); s[6] += bf_lo(q.w); s[7] += bf_hi(q.w);
                }
                uint32_t dst = act0 + (uint32_t)(head + ((rank * Rl + r) * C + c * 8) * 4);
                if (CLUSTER) dst = remote(dst, 0);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    if (CLUSTER) st_remote32(dst + 4 * e, __float_as_uint(s[e]));
                    else sts32(dst + 4 * e, __float_as_uint(s[e]));
                }
            }
            image_sync<CLUSTER, WARPS>(slot);
            float* pooled = rows + p.a.last_H * C;
            if (rank == 0)
                for (int c = tid; c < C; c += threads) {
                    float s = 0.0f;
                    for (int r = 0; r < p.a.last_H; ++r) s += rows[r * C + c];
                    pooled[c] = s;
                }
            image_sync<CLUSTER, WARPS>(slot);                 // (and no CTA of a cluster leaves while others write to it)
            if (rank == 0)
                for (int k = warp; k < p.a.n_classes; k += WARPS) {
                    float s = 0.0f;
                    for (int c = lane; c < C; c += 32) s = fmaf(pooled[c], __ldg(p.a.fcw + (size_t)k * p.a.fc_pitch + c), s);
#pragma unroll
                    for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
                    if (lane == 0) p.a.logits[(size_t)n * p.a.n_classes + k] = s + (p.a.fcb ? p.a.fcb[k] : 0.0f);
                }
        }
    }
    if (*abort_flag) {
        for (int i = 0; i < 200; ++i) __nanosleep(1000);     // let copies in flight land before shared memory is released
    }
}

}  // namespace

bool prepare_net() {
    for (const void* fn : {(const void*)resident_net_kernel<true, kWarps>, (const void*)resident_net_kernel<false, kWarps>, (const void*)resident_net_kernel<false, 2 * kWarps>}) {
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kNetSmemMax) != cudaSuccess) { cudaGetLastError(); return false; }
    }
    return true;
}

// CTAs or clusters that run at once.  A cluster lies within a group of SMs, so that not every SM finds a place in one: 33 clusters
// of four on a B200, not 37 (ResNet-56, 36 images: 165 us as two waves of clusters of four, 104 us in clusters of two).
int net_at_once(int cs) {
    if (cs == 1) return sm_count();
    static std::atomic<int> known[64][9];              // (threads may all be the first: each finds the same)
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || cs > 8) { cudaGetLastError(); return std::max(1, sm_count() / cs); }
    if (!known[dev][cs]) {
        cudaFuncSetAttribute(resident_net_kernel<true, kWarps>, cudaFuncAttributeMaxDynamicSharedMemorySize, kNetSmemMax);
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3((unsigned)(cs * 512));
        cfg.blockDim = dim3((unsigned)kThreads);
        cfg.dynamicSmemBytes = kNetSmemMax / 2 + 1024;         // one CTA on an SM
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = (unsigned)cs; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, resident_net_kernel<true, kWarps>, &cfg) != cudaSuccess || n < 1) { cudaGetLastError(); n = sm_count() / cs; }
        known[dev][cs] = std::max(1, std::min(n, sm_count() / cs));
    }
    return known[dev][cs];
}

void launch_net(const NetPlan& plan, const NetArgs& a, const NetLayer* d_table, int* d_status, cudaStream_t st) {
    NetParams p;
    memset(&p, 0, sizeof(p));
    p.a = a;
    p.table = d_table;
    p.G = plan.G; p.cs = plan.cs; p.L = (int)plan.table.size();
    p.img_bytes = plan.img_bytes;
    p.in_off = plan.table[0].in_off; p.in_rows = a.H / plan.cs;
    p.head_off = plan.head_off; p.last_off = plan.last_off; p.last_PV = plan.last_PV; p.first_requests = plan.first_requests;
    p.status = d_status;
    int clusters = net_at_once(plan.cs);
    if (clusters > a.N) clusters = a.N;
    p.n_clusters = clusters;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(clusters * plan.cs));
    cfg.blockDim = dim3((unsigned)(32 * plan.warps * plan.G));
    cfg.dynamicSmemBytes = plan.smem_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)plan.cs; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = plan.cs > 1 ? 2 : 1;
    void* args[1] = {(void*)&p};
    cudaLaunchKernelExC(&cfg, plan.cs > 1 ? (const void*)resident_net_kernel<true, kWarps> : plan.warps > kWarps ? (const void*)resident_net_kernel<false, 2 * kWarps> : (const void*)resident_net_kernel<false, kWarps>, args);
}

}  // namespace fp
