// First convolution + max pooling of an ImageNet-shaped network in one kernel for sm_100a:
//     NCHW bf16 or fp32 input  ->  7x7 / stride 2 / pad 3 convolution (folded-BN bias, ReLU)  ->  3x3 / stride 2 / pad 1
//     max pooling  ->  planar-8 bf16 tensor with a zero border (fp_internal.h).
// The convolution's output, four times the size of the pooled tensor, never leaves the tensor memory and registers.
//
//   GEMM           The 7x7 / stride-2 window over C channels is a 4x4 / stride-1 window over the 4 C channels of the
//                  input's four pixel parities at half resolution (input row 2i + a, column 2j + b -> channel
//                  (2a + b) C + c of half-resolution pixel (i, j); filter tap r = 2 ta + a - 1, s = 2 tb + b - 1, the taps
//                  with r or s = -1 being zero): sixteen taps of one K = 16 step each.  M = 128 positions = ONE row of half
//                  resolution, read as it lies in shared memory from column tb - 2 on; as tap row ta it belongs to convolution
//                  row i + 2 - ta, so the filters of all four tap rows stand side by side along N: one MMA of N = 4 K_pad adds
//                  a column tap to four convolution rows' accumulators, which are a ring of four in tensor memory (the filter
//                  blocks are kept in the order 3 2 1 0 3 2 1, so that the ring may begin anywhere).  Per row 4 MMAs of 128
//                  cycles instead of 16 of 48, and 480 instead of 770 cycles of shared-memory bandwidth, which the
//                  pooling needs as well.
//                  The filters' shifts come out of the MMAs too: three spare channels of the sixteen are ones.
//   Work           A CTA takes a run of consecutive pooled rows and goes down it: half-resolution rows pass through a ring of
//                  shared memory, each made once; convolution rows through a ring of accumulators, each computed once (the
//                  row that two pooled rows share is carried over in registers); a run starts with one extra row, an
//                  image with none.  Two CTAs share an SM.
//   Parts          Where a row has more than 128 convolution columns, or there are more than 64 filters, a CTA takes a strip of the
//                  pooled columns (its tile begins one convolution column to the left of them) and a part of the filters; strips and
//                  parts are the grid's other dimensions.  Every part makes the half-resolution rows it reads itself.
//   Roles          five warps turn input rows into half-resolution rows (a thread per pixel: one load per channel and row
//                  parity gives both column parities; the next row's are asked for before this one's place is waited
//                  for), one warp issues the MMAs, eight warps pool.
//   Pooling        A thread holds a column and half of the filters: the maximum over three rows (one is carried over), ReLU, bf16
//                  pairs, through shared memory to a thread per output position for the three columns.  Rows and columns
//                  outside the image never win: behind the ReLU a zero is below every window's maximum.
//   What bounds it the tensor pipe and shared memory, some 1100 cycles per pooled row for the MMAs (N = 256), and the pooling
//                  warps' latency.  (Units of two pooled rows with the convolution rows in shared memory, the first form:
//                  72 us at ResNet-18 batch 64, 224 x 224; one tile and one accumulator per convolution row: 45 us.)
//   Waits          bounded, as in the other tensor-core kernels: a wait that runs out raises the status word, every role
//                  leaves its loops, tensor memory is released.
#include "fp_internal.h"
#include "tc_common.cuh"

#include <algorithm>
#include <cstdio>
#include <cstring>

namespace fp {

using namespace tc;

namespace {

constexpr int kRowWarps = 5, kPoolWarps = 8;
constexpr int kThreads = 32 * (kRowWarps + 1 + kPoolWarps);
constexpr int kRing = 4;                   // half-resolution rows in shared memory
constexpr int kAcc = 4;                    // convolution rows in tensor memory: those that a half-resolution row adds to
constexpr int kBlocks = 7;                 // filter blocks of a column tap: ta = 3, 2, 1, 0, 3, 2, 1

struct SpParams {
    StemPoolArgs a;
    int Hc, Wc, Hp, Wp;            // convolution and pooled sizes
    int strip, k_tile;             // pooled columns of a strip and filters of a part (the last ones may have fewer); Wp and K_pad where there is one
    int pitch;                     // half-resolution pixels per row of a strip: its convolution columns and 3 more (-2 .. +1)
    int plane;                     // 16-byte rows per chunk of the ring (kRing * pitch, plus what the last row's taps reach)
    int b_bytes;                   // filters: 4 column taps * 2 chunks * 7 blocks * k_tile * 16
    int tmem_cols;
    int rows;                      // pooled rows of all images
    int* status;
};

struct __align__(16) SpCtrl {
    uint64_t b_full;
    uint64_t x_full[kRing], x_empty[kRing];
    uint64_t acc_full[kAcc], acc_empty[kAcc];
    uint32_t tmem_base;
    int abort_flag;
    int pad_[2];
};

// A CTA's run, image by image: pooled rows q0 .. q1 - 1 of image n; convolution rows first_row .. last_row.
struct Segment { int n, q0, q1, first_row, last_row; };
__device__ __forceinline__ Segment segment_at(const SpParams& p, int b, int end) {
    Segment s;
    s.n = b / p.Hp;
    s.q0 = b - s.n * p.Hp;
    s.q1 = min(p.Hp, s.q0 + (end - b));
    s.first_row = s.q0 > 0 ? 2 * s.q0 - 1 : 0;
    s.last_row = min(2 * s.q1 - 1, p.Hc - 1);
    s.n += p.a.n0;
    return s;
}

// Maxima of bf16 pairs none of which is below zero: they are ordered as 16-bit integers are.
__device__ __forceinline__ uint32_t max2(uint32_t a, uint32_t b) { return __vmaxs2(a, b); }
__device__ __forceinline__ uint32_t max3(uint32_t a, uint32_t b, uint32_t c) { return __vimax3_s16x2(a, b, c); }

// The 2 x C input words of a half-resolution pixel: rows 2i and 2i + 1, columns 2j and 2j + 1 as a pair of bf16 each, `at` being
// the first channel's pixel (2i, 2j).  Outside the image zero: a column for every row (`in` false), a row by its number.  (The
// pointer steps from row to row: an address worked out for every load was a tenth of the kernel's instructions, of which it
// issues in 54 % of the cycles - ResNet-18 batch 64 43.1 -> 41.0 us, ResNet-50 batch 128 71.8 -> 68.2 us.)
template <bool F32, int C>
__device__ __forceinline__ void load_pixel(const uint8_t* at, int row_bytes, size_t plane_bytes, int row, int H, bool in, bool second, bool paired, uint32_t (&v)[2 * C]) {
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        const bool there = in && (unsigned)(row + a) < (unsigned)H;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const uint8_t* x = at + c * plane_bytes + a * row_bytes;
            uint32_t w = 0u;
            if (there) {
                if (F32) {
                    float2 f;
                    if (paired) f = *reinterpret_cast<const float2*>(x);
                    else { f.x = *reinterpret_cast<const float*>(x); f.y = second ? reinterpret_cast<const float*>(x)[1] : 0.0f; }
                    w = pack_bf16x2(f.x, f.y);
                } else {
                    if (paired) w = *reinterpret_cast<const uint32_t*>(x);
                    else w = (uint32_t)*reinterpret_cast<const unsigned short*>(x) | (second ? (uint32_t)reinterpret_cast<const unsigned short*>(x)[1] << 16 : 0u);
                }
            }
            v[a * C + c] = w;
        }
    }
}

// PARTS: there are several strips or parts of the filters (W > 256 or K_pad > 64).
template <bool F32, int C, bool PARTS>
__global__ void __launch_bounds__(kThreads, 2) stem_pool_kernel(const SpParams p, const int paired) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    SpCtrl* ctrl = reinterpret_cast<SpCtrl*>(smem_raw);
    const uint32_t base = smem_u32(smem_raw);
    const int k_base = PARTS ? (int)blockIdx.z * p.k_tile : 0, K_pad = PARTS ? min(p.k_tile, p.a.K_pad - k_base) : p.a.K_pad;
    const int x0 = PARTS ? (int)blockIdx.y * p.strip : 0, Wp = PARTS ? min(p.strip, p.Wp - x0) : p.Wp;       // this CTA's pooled columns
    const int left = x0 > 0, c0 = 2 * x0 - left, Wc = PARTS ? min(p.Wc - c0, 2 * Wp + left) : p.Wc;         // and convolution columns
    const uint32_t b_addr = (base + (uint32_t)sizeof(SpCtrl) + 127u) & ~127u;
    const uint32_t x_addr = b_addr + (uint32_t)p.b_bytes;
    uint4* ring = reinterpret_cast<uint4*>(smem_raw + (x_addr - base));
    volatile int* abort_flag = &ctrl->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t b_full = base + (uint32_t)offsetof(SpCtrl, b_full);
    const uint32_t x_full0 = base + (uint32_t)offsetof(SpCtrl, x_full), x_empty0 = base + (uint32_t)offsetof(SpCtrl, x_empty);
    const uint32_t acc_full0 = base + (uint32_t)offsetof(SpCtrl, acc_full), acc_empty0 = base + (uint32_t)offsetof(SpCtrl, acc_empty);

    if (threadIdx.x == 0) {
        mbar_init(b_full, 1);
        for (int s = 0; s < kRing; ++s) { mbar_init(x_full0 + 8 * s, 32 * kRowWarps); mbar_init(x_empty0 + 8 * s, 1); }
        for (int s = 0; s < kAcc; ++s) { mbar_init(acc_full0 + 8 * s, 1); mbar_init(acc_empty0 + 8 * s, kPoolWarps); }
        ctrl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    // the places of the columns left and right of the row: zero, and never written
    for (int i = threadIdx.x; i < 4 * (K_pad >> 3); i += kThreads)
        (ring + 2 * p.plane)[(size_t)(i >> 1) * (2 * Wp + 1) + Wp + (i & 1) * Wp] = make_uint4(0, 0, 0, 0);
    if (warp == kRowWarps) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(base + (uint32_t)offsetof(SpCtrl, tmem_base)), "r"((uint32_t)p.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&ctrl->tmem_base);
    // filters: resident for the whole kernel (they are not written by the previous kernel in the stream).  All warps ask for them: a warp's
    // copies go out one after the other, and 56 from one warp were two microseconds of a forward that begins with this kernel (ResNet-18, one
    // image 87.0 -> 85.4 us, ResNet-50 186.4 -> 184.2).
    {
        const uint32_t block = (uint32_t)K_pad * 16u;
        if (threadIdx.x == 0) mbar_expect_tx(b_full, 8u * kBlocks * block);
        __syncwarp();
        for (int i = warp + (kThreads / 32) * lane; i < 8 * kBlocks; i += kThreads) {
            const int plane = i / kBlocks, blk = i - plane * kBlocks, tb = plane >> 1, ta = 3 - (blk & 3);
            bulk_copy(b_addr + (uint32_t)i * block, reinterpret_cast<const uint8_t*>(p.a.w) + (size_t)((ta * 4 + tb) * 2 + (plane & 1)) * (size_t)(p.a.K_pad * 16) + k_base * 16, block, b_full);
        }
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    const int begin = (int)((long long)p.rows * blockIdx.x / gridDim.x), end = (int)((long long)p.rows * (blockIdx.x + 1) / gridDim.x);
    bool ok = true;
    if (warp < kRowWarps) {
        // ------------------------------ half-resolution rows ------------------------------
        const int jx = threadIdx.x;                      // pixel of the row: half-resolution column c0 + jx - 2
        const bool mine = jx < p.pitch;
        constexpr int elem = F32 ? 4 : 2;
        const int col = 2 * (c0 + jx - 2), row_bytes = p.a.W * elem;
        const size_t plane_bytes = (size_t)p.a.H * row_bytes;
        const bool in = (unsigned)col < (unsigned)p.a.W, second = col + 1 < p.a.W;
        uint32_t slot = 0, phase = 0;
        for (int b = begin; b < end && ok;) {
            const Segment s = segment_at(p, b, end);
            const int last = s.last_row + 1;
            uint32_t next[2 * C];
            const uint8_t* at_row = reinterpret_cast<const uint8_t*>(p.a.x) + ((long long)s.n * C * p.a.H + 2 * (s.first_row - 2)) * row_bytes + col * elem;
            if (mine) load_pixel<F32, C>(at_row, row_bytes, plane_bytes, 2 * (s.first_row - 2), p.a.H, in, second, paired != 0, next);
            for (int i = s.first_row - 2; i <= last; ++i) {
                uint32_t v[2 * C];
#pragma unroll
                for (int e = 0; e < 2 * C; ++e) v[e] = next[e];
                at_row += 2 * row_bytes;
                if (mine && i < last) load_pixel<F32, C>(at_row, row_bytes, plane_bytes, 2 * (i + 1), p.a.H, in, second, paired != 0, next);
                ok = __all_sync(0xffffffffu, mbar_wait(x_empty0 + 8 * slot, phase ^ 1, abort_flag));
                if (!ok) break;
                if (mine) {
                    // channel (2a + b) C + c = column parity b of row parity a: the lower or upper half of v[a C + c]
                    uint32_t h[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int e0 = 2 * k, e1 = 2 * k + 1;
                        const uint32_t lo = e0 < 4 * C ? v[e0 / (2 * C) * C + e0 % C] : 0u, hi = e1 < 4 * C ? v[e1 / (2 * C) * C + e1 % C] : 0u;
                        h[k] = e0 < 4 * C ? __byte_perm(lo, hi, (e0 / C % 2 ? 0x0032 : 0x0010) | (e1 / C % 2 ? 0x7600 : 0x5400))
                             : e0 == 4 * C ? 0x3f803f80u : e0 == 4 * C + 2 ? 0x3f80u : 0u;       // ones for the shifts
                    }
                    uint4* at = ring + (size_t)slot * p.pitch + jx;
                    at[0] = make_uint4(h[0], h[1], h[2], h[3]);
                    at[p.plane] = make_uint4(h[4], h[5], h[6], h[7]);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // generic-proxy stores -> MMA reads
                mbar_arrive(x_full0 + 8 * slot);
                if (++slot == kRing) { slot = 0; phase ^= 1; }
            }
            b += s.q1 - s.q0;
        }
    } else if (warp == kRowWarps) {
        // ------------------------------ MMAs ------------------------------
        // the whole warp goes through the loops, one elected lane issues: see umma_bf16_lo_if
        const uint32_t leader = elect_one();
        const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24), n_unit = (uint32_t)(K_pad >> 3) << 17;
        const uint32_t b_pitch = (uint32_t)(kBlocks * K_pad);                // rows between a column tap's two chunks
        const uint32_t b_lo0 = (b_addr >> 4) | (b_pitch << 16), x_lo0 = (x_addr >> 4) | ((uint32_t)p.plane << 16);
        auto wait_for = [&](uint32_t bar, uint32_t ph) { return __all_sync(0xffffffffu, mbar_wait(bar, ph, abort_flag)); };
        ok = wait_for(b_full, 0);
        uint32_t slot = 0, phase = 0;                    // half-resolution row
        uint32_t used = 0;                               // convolution rows begun so far: row number `used` has place used % 4
        for (int b = begin; b < end && ok;) {
            const Segment s = segment_at(p, b, end);
            const int place0 = (int)(used & 3) - s.first_row;                // row r of the segment: place (r + place0) & 3
            for (int i = s.first_row - 2; i <= s.last_row + 1; ++i) {
                // row i of half resolution is tap row ta of convolution rows i + 2 - ta: rows lo .. hi, block 3 - ta = r - (i - 1)
                const int lo = max(i - 1, s.first_row), hi = min(i + 2, s.last_row), grown = min(i + 1, s.last_row);
                ok = wait_for(x_full0 + 8 * slot, phase);
                if (!ok) break;
                tc_fence_after();
                const uint32_t a_row = x_lo0 + slot * (uint32_t)p.pitch;
                // rows r0 .. r1 at once: accumulators that follow one another in tensor memory, blocks that do in shared memory
                auto rows_at_once = [&](int r0, int r1, uint32_t tb, uint32_t accumulate) {
                    while (r0 <= r1) {
                        const int at = (r0 + place0) & 3, n = min(r1 - r0 + 1, kAcc - at);
                        umma_bf16_lo_if(leader, tmem_base + (uint32_t)(at * K_pad), a_row + tb, b_lo0 + tb * 2u * b_pitch + (uint32_t)((r0 - i + 1) * K_pad),
                                        idesc0 + (uint32_t)n * n_unit, accumulate);
                        r0 += n;
                    }
                };
                // column tap 0: rows that have sums already, which no pooling warp is waited for (41.0 -> 39.9 us, ResNet-50 68.2 -> 65.6),
                rows_at_once(lo, grown, 0, 1u);
                if (hi == i + 2) {                                           // and the one that begins, in the place of row i - 2
                    ok = wait_for(acc_empty0 + 8 * (used & 3), ((used >> 2) & 1) ^ 1);
                    ++used;
                    if (!ok) break;
                    tc_fence_after();
                    rows_at_once(hi, hi, 0, 0u);
                }
                if (hi - lo == 3) {                      // all four places: the blocks from the first place's row on, round the seven
                    const uint32_t turn = (uint32_t)(-(lo + place0) & 3);
#pragma unroll
                    for (uint32_t tb = 1; tb < 4; ++tb)
                        umma_bf16_lo_if(leader, tmem_base, a_row + tb, b_lo0 + tb * 2u * b_pitch + turn * (uint32_t)K_pad, idesc0 + 4u * n_unit, 1u);
                } else {
#pragma unroll 1
                    for (uint32_t tb = 1; tb < 4; ++tb) rows_at_once(lo, hi, tb, 1u);
                }
                if (leader) {
                    umma_commit(x_empty0 + 8 * slot);
                    if (i - 1 >= s.first_row) umma_commit(acc_full0 + 8 * (uint32_t)((i - 1 + place0) & 3));      // row i - 1 is complete
                }
                __syncwarp();
                if (++slot == kRing) { slot = 0; phase ^= 1; }
            }
            b += s.q1 - s.q0;
        }
    } else {
        // ------------------------------ pooling ------------------------------
        const int pw = warp - (kRowWarps + 1), quarter = warp & 3, half = pw >> 2;
        const int col = quarter * 32 + lane;             // convolution column; the lower or the upper half of the filter groups
        const int first_group = half ? ((K_pad >> 4) + 1) >> 1 : 0, groups = half ? (K_pad >> 4) - first_group : ((K_pad >> 4) + 1) >> 1;
        const bool live = col < Wc;
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + 16u * (uint32_t)min(first_group, (K_pad >> 4) - 1);
        const int Wq = row_vecs(p.Wp), P2o = image_vecs(p.Hp, p.Wp), pitch = 2 * Wp + 1;
        const long long plane_out = plane_vecs(p.a.N, p.Hp, p.Wp);
        uint4* yout = reinterpret_cast<uint4*>(p.a.y);
        uint4* cols_s = reinterpret_cast<uint4*>(smem_raw + (x_addr - base)) + 2 * p.plane;      // [row parity][chunk]: even columns, then odd ones from -1 on
        const int off = col - left, place = off & 1 ? Wp + ((off + 1) >> 1) : off >> 1;      // off: from the strip's first even column
        uint32_t acc = 0, acc_phase = 0;
        uint32_t m[2][8];                                // the convolution row above the pooled row's two, then the maxima with them: bf16 pairs
        // The next convolution row, ReLU and bf16 (the filters' shifts are in the sums): use(group, row, carried row or maxima so far).
        // (A warp whose wait ran out goes on without its rows: the others of its half count on it at their barrier.)
        auto take_row = [&](auto use) {
            if (ok && !(ok = __all_sync(0xffffffffu, mbar_wait(acc_full0 + 8 * acc, acc_phase, abort_flag))) && lane == 0) atomicExch(&ctrl->abort_flag, 1);
            tc_fence_after();
            uint32_t v[2][16];
#pragma unroll
            for (int g = 0; g < 2; ++g) tmem_ld16(taddr + acc * (uint32_t)K_pad + 16u * (uint32_t)max(0, min(g, groups - 1)), v[g]);
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty0 + 8 * acc);
            if (++acc == kAcc) { acc = 0; acc_phase ^= 1; }
#pragma unroll
            for (int g = 0; g < 2; ++g)
                if (g < groups) {
                    uint32_t row[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) row[e] = pack_bf16x2_relu(__uint_as_float(v[g][2 * e]), __uint_as_float(v[g][2 * e + 1]));
                    use(g, row, m[g]);
                }
        };
        int parity = 0;
        for (int b = begin; b < end;) {
            const Segment s = segment_at(p, b, end);
#pragma unroll
            for (int g = 0; g < 2; ++g)
#pragma unroll
                for (int e = 0; e < 8; ++e) m[g][e] = 0u;
            if (s.q0 > 0) take_row([&](int, const uint32_t (&row)[8], uint32_t (&m)[8]) {
#pragma unroll
                for (int e = 0; e < 8; ++e) m[e] = row[e];
            });
            for (int q = s.q0; q < s.q1; ++q) {
                // down the rows: maxima, the column's vectors into shared memory.  A row is given back before the next is waited for:
                // the MMAs that complete it begin the row four further on, in this one's place.
                const bool two = 2 * q + 1 < p.Hc;
                uint4* const at = cols_s + (size_t)(parity * (K_pad >> 3) + 2 * first_group) * pitch + place;
                auto put = [&](int g, const uint32_t (&o)[8]) {
                    if (live) {
                        at[(2 * g) * pitch] = make_uint4(o[0], o[1], o[2], o[3]);
                        at[(2 * g + 1) * pitch] = make_uint4(o[4], o[5], o[6], o[7]);
                    }
                };
                take_row([&](int g, const uint32_t (&row)[8], uint32_t (&m)[8]) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) m[e] = max2(m[e], row[e]);
                    if (!two) put(g, m);
                });
                if (two) take_row([&](int g, const uint32_t (&row)[8], uint32_t (&m)[8]) {
                    uint32_t o[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) { o[e] = max2(m[e], row[e]); m[e] = row[e]; }
                    put(g, o);
                });
                asm volatile("bar.sync %0, 128;" ::"r"(1 + half) : "memory");
                // across the columns: a warp takes every fourth chunk, a lane a position of the output row, border included
                for (int ch = quarter; ch < 2 * groups; ch += 4) {
                    const int chunk = 2 * first_group + ch;
                    const uint4* from = cols_s + (size_t)(parity * (K_pad >> 3) + chunk) * pitch;
                    uint4* to = yout + (long long)((k_base >> 3) + chunk) * plane_out + (long long)s.n * P2o + (long long)(q + 1) * Wq + x0;
                    for (int k0 = lane; k0 < Wp + 1; k0 += 64) {
                        uint4 l[2], c[2], r[2];          // two positions' loads in flight
#pragma unroll
                        for (int i = 0; i < 2; ++i) {    // columns 2k - 3 .. 2k - 1
                            const int k = max(1, min(k0 + 32 * i, Wp));
                            l[i] = from[Wp + k - 1]; c[i] = from[k - 1]; r[i] = from[Wp + k];
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const int k = k0 + 32 * i;
                            if (k >= Wp + 1) break;
                            if (PARTS && k == 0 && x0 > 0) continue;                      // another strip's column
                            uint4 o = make_uint4(0, 0, 0, 0);
                            if (k >= 1)
                                o = make_uint4(max3(l[i].x, c[i].x, r[i].x), max3(l[i].y, c[i].y, r[i].y), max3(l[i].z, c[i].z, r[i].z), max3(l[i].w, c[i].w, r[i].w));
                            to[k] = o;
                            if (q == 0) to[k - Wq] = make_uint4(0, 0, 0, 0);
                            if (q == p.Hp - 1 && s.n == p.a.N - 1) {                      // the zeros behind the last image
                                to[k + Wq] = make_uint4(0, 0, 0, 0);
                                if (k == 0) to[2 * Wq] = make_uint4(0, 0, 0, 0);
                            }
                        }
                    }
                }
                parity ^= 1;                             // (the next row's vectors go to the other half: nobody waits for this one's readers)
            }
            b += s.q1 - s.q0;
        }
    }
    if (!ok && lane == 0) { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 6); }

    // ---- teardown ----
    if (*abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);         // copies in flight land before the memory is given back
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == kRowWarps) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)p.tmem_cols) : "memory");
    }
}

constexpr unsigned kSmemMax = 233472u / 2 - 1024u;       // two CTAs on an SM

struct Shape { int Hc, Wc, Hp, Wp, strips, strip, parts, k_tile, pitch, plane, b_bytes; unsigned smem; };
Shape shape_of(int H, int W, int K_pad) {
    Shape s;
    s.Hc = (H - 1) / 2 + 1; s.Wc = (W - 1) / 2 + 1; s.Hp = (s.Hc - 1) / 2 + 1; s.Wp = (s.Wc - 1) / 2 + 1;
    // a strip's convolution columns - two for a pooled one, and one to the left - are a tile of 128
    s.strips = s.Wc <= 128 ? 1 : (s.Wp + 62) / 63;
    s.strip = (s.Wp + s.strips - 1) / s.strips;
    s.parts = (kAcc * K_pad + 255) / 256;
    s.k_tile = (K_pad / 16 + s.parts - 1) / s.parts * 16;
    s.pitch = std::min(s.Wc, s.strips == 1 ? s.Wc : 2 * s.strip + 1) + 3;
    s.plane = (kRing * s.pitch + 128 + 7) & ~7;
    s.b_bytes = 8 * kBlocks * s.k_tile * 16;
    s.smem = (unsigned)sizeof(SpCtrl) + 128u + (unsigned)s.b_bytes + 2u * (unsigned)s.plane * 16u +
             2u * (unsigned)(s.k_tile / 8) * (unsigned)(2 * s.strip + 1) * 16u;
    return s;
}

typedef void (*StemKernel)(const SpParams, const int);
template <bool F32, bool PARTS>
StemKernel kernel_of(int C) { return C == 3 ? stem_pool_kernel<F32, 3, PARTS> : C == 2 ? stem_pool_kernel<F32, 2, PARTS> : stem_pool_kernel<F32, 1, PARTS>; }
StemKernel kernel_of(const StemPoolArgs& a) {
    const Shape s = shape_of(a.H, a.W, a.K_pad);
    if (s.strips * s.parts > 1) return a.in_f32 ? kernel_of<true, true>(a.C) : kernel_of<false, true>(a.C);
    return a.in_f32 ? kernel_of<true, false>(a.C) : kernel_of<false, false>(a.C);
}

}  // namespace

bool stem_pool_supported(int C, int H, int W, int K_pad) {
    if (C < 1 || C > 3 || H < 8 || W < 8 || W > kMaxWidth || K_pad % 16 || K_pad < 16 || K_pad > 128) return false;
    return shape_of(H, W, K_pad).smem <= kSmemMax;
}

int plan_stem_pool(const StemPoolArgs& a, StemPoolPlan* plan, char* err, size_t err_len) {
    memset(plan, 0, sizeof(*plan));
    if (!stem_pool_supported(a.C, a.H, a.W, a.K_pad)) { snprintf(err, err_len, "first convolution + pooling: shape not supported"); return 1; }
    plan->smem_bytes = shape_of(a.H, a.W, a.K_pad).smem;
    plan->tmem_cols = 64;
    while (plan->tmem_cols < kAcc * shape_of(a.H, a.W, a.K_pad).k_tile) plan->tmem_cols *= 2;           // at most half of an SM's, for two CTAs
    if (cudaFuncSetAttribute(kernel_of(a), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax) != cudaSuccess) {
        snprintf(err, err_len, "cannot raise the dynamic shared memory limit");
        cudaGetLastError();
        return 1;
    }
    plan->valid = 1;
    return 0;
}

void launch_stem_pool(const StemPoolPlan& plan, const StemPoolArgs& a, int* d_status, cudaStream_t st) {
    SpParams p;
    memset(&p, 0, sizeof(p));
    const Shape s = shape_of(a.H, a.W, a.K_pad);
    p.a = a;
    p.Hc = s.Hc; p.Wc = s.Wc; p.Hp = s.Hp; p.Wp = s.Wp; p.strip = s.strip; p.k_tile = s.k_tile; p.pitch = s.pitch; p.plane = s.plane; p.b_bytes = s.b_bytes;
    p.tmem_cols = plan.tmem_cols;
    p.rows = a.n_count * s.Hp;
    p.status = d_status;
    // two columns with one load where a row's pairs are aligned
    const int paired = a.W % 2 == 0 && (uintptr_t)a.x % (a.in_f32 ? 8 : 4) == 0;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)std::max(1, std::min(2 * sm_count() / (s.strips * s.parts), p.rows)), (unsigned)s.strips, (unsigned)s.parts);
    cfg.blockDim = dim3((unsigned)kThreads);
    cfg.dynamicSmemBytes = plan.smem_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void* args[2] = {(void*)&p, (void*)&paired};
    cudaLaunchKernelExC(&cfg, (const void*)kernel_of(a), args);
}

}  // namespace fp
