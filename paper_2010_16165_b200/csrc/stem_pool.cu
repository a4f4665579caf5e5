// First convolution + max pooling of an ImageNet-shaped network in one kernel for sm_100a:
//     NCHW bf16 or fp32 input  ->  7x7 / stride 2 / pad 3 convolution (folded-BN bias, ReLU)  ->  3x3 / stride 2 / pad 1
//     max pooling  ->  planar-8 bf16 tensor with a zero border (fp_internal.h).
// The convolution's output, four times the size of the pooled tensor, never leaves the tensor memory and registers.
//
//   GEMM           The 7x7 / stride-2 window over C channels is a 4x4 / stride-1 window over the 4 C channels of the
//                  input's four pixel parities at half resolution (input row 2i + a, column 2j + b -> channel
//                  (2a + b) C + c of half-resolution pixel (i, j); filter tap r = 2 ta + a - 1, s = 2 tb + b - 1, the taps
//                  with r or s = -1 being zero): sixteen taps of one K = 16 step each.  M = 128 positions = ONE convolution
//                  row, N = K_pad filters; the operand of tap (ta, tb) for row r is half-resolution row r - 2 + ta from
//                  column tb - 2 on, read as it lies in shared memory.
//   Work           A CTA takes a run of consecutive pooled rows and goes down it: half-resolution rows pass through a ring of
//                  shared memory, each made once; convolution rows through a ring of accumulators, each computed once (the
//                  row that two pooled rows share is carried over in registers); a run starts with one extra row, an
//                  image with none.  Two CTAs share an SM.
//   Roles          five warps turn input rows into half-resolution rows (a thread per pixel: one load per channel and row
//                  parity gives both column parities; the next row's are asked for before this one's place is waited
//                  for), one warp issues the MMAs, eight warps pool.
//   Pooling        A thread holds a column and half of the filters: bias and ReLU into bf16 pairs, the maximum with the rows
//                  above, then with the neighbouring columns by shuffles - the column left of a warp's first comes from the
//                  next warp through shared memory - and the even columns are stored.  Rows and columns outside the image
//                  count as zeros: behind the ReLU a zero never wins a window it should not.
//   What bounds it 32 MMAs per pooled row at 40-60 cycles apiece (N = 64).  The form before this one - units of two pooled
//                  rows, fifteen staged input rows rewritten per unit, the five convolution rows written to shared memory
//                  and read back - spent 9.6 k cycles per unit on rewriting, read-out and pooling one after the other:
//                  72 us at ResNet-18 batch 64 (224 x 224).
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
constexpr int kTaps = 16;                  // 4 x 4 taps over the parity channels, one K = 16 step each
constexpr int kRing = 8;                   // half-resolution rows in shared memory
constexpr int kMaxAcc = 8;                 // convolution rows in tensor memory, at most
constexpr int kMaxGroups = 3;              // 16-filter groups a pooling warp has (K_pad <= 96)

struct SpParams {
    StemPoolArgs a;
    int Hc, Wc, Hp, Wp;            // convolution and pooled sizes
    int pitch;                     // half-resolution pixels per row: Wc + 3 (columns -2 .. Wc)
    int plane;                     // 16-byte rows per chunk of the ring (kRing * pitch, plus what the last row's taps reach)
    int b_bytes;                   // filters: 16 taps * 2 chunks * K_pad * 16
    int acc_rows, tmem_cols;
    int rows;                      // pooled rows of all images
    int* status;
};

struct SpCtrl {
    uint64_t b_full;
    uint64_t x_full[kRing], x_empty[kRing];
    uint64_t acc_full[kMaxAcc], acc_empty[kMaxAcc];
    uint32_t tmem_base;
    int abort_flag;
    uint4 edge[2][2][4][kMaxGroups][2];        // [pooled row parity][half][quarter][group]: a warp's last column
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

// The 2 x C input words of half-resolution pixel (i, j): rows 2i and 2i + 1, columns 2j and 2j + 1 (zero outside the image) as a
// pair of bf16 each.
template <bool F32, int C>
__device__ __forceinline__ void load_pixel(const SpParams& p, int n, int i, int j, bool paired, uint32_t (&v)[2 * C]) {
    const int col = 2 * j;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        const int row = 2 * i + a;
        const bool in = row >= 0 && row < p.a.H && col >= 0 && col < p.a.W;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const size_t at = (((size_t)n * C + c) * p.a.H + row) * p.a.W + col;
            uint32_t w = 0u;
            if (in) {
                if (F32) {
                    const float* x = reinterpret_cast<const float*>(p.a.x) + at;
                    float2 f;
                    if (paired) f = *reinterpret_cast<const float2*>(x);
                    else { f.x = x[0]; f.y = col + 1 < p.a.W ? x[1] : 0.0f; }
                    w = pack_bf16x2(f.x, f.y);
                } else {
                    const unsigned short* x = reinterpret_cast<const unsigned short*>(p.a.x) + at;
                    if (paired) w = *reinterpret_cast<const uint32_t*>(x);
                    else w = (uint32_t)x[0] | (col + 1 < p.a.W ? (uint32_t)x[1] << 16 : 0u);
                }
            }
            v[a * C + c] = w;
        }
    }
}

// NG: groups of 16 filters a pooling warp has, at most.
template <bool F32, int C, int NG>
__global__ void __launch_bounds__(kThreads, NG <= 2 ? 2 : 1) stem_pool_kernel(const SpParams p, const int paired) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    SpCtrl* ctrl = reinterpret_cast<SpCtrl*>(smem_raw);
    const uint32_t base = smem_u32(smem_raw);
    const int K_pad = p.a.K_pad;
    float* bias_s = reinterpret_cast<float*>(smem_raw + sizeof(SpCtrl));                     // K_pad floats
    const uint32_t b_addr = (base + (uint32_t)sizeof(SpCtrl) + (uint32_t)K_pad * 4u + 127u) & ~127u;
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
        for (int s = 0; s < kMaxAcc; ++s) { mbar_init(acc_full0 + 8 * s, 1); mbar_init(acc_empty0 + 8 * s, kPoolWarps); }
        ctrl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    for (int i = threadIdx.x; i < K_pad; i += kThreads) bias_s[i] = p.a.bias[i];
    if (warp == kRowWarps) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(base + (uint32_t)offsetof(SpCtrl, tmem_base)), "r"((uint32_t)p.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&ctrl->tmem_base);
    // filters: resident for the whole kernel (they are not written by the previous kernel in the stream)
    if (threadIdx.x == 0) {
        mbar_expect_tx(b_full, (uint32_t)p.b_bytes);
        for (int off = 0; off < p.b_bytes; off += 16384)
            bulk_copy(b_addr + off, reinterpret_cast<const uint8_t*>(p.a.w) + off, (uint32_t)min(16384, p.b_bytes - off), b_full);
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    const int begin = (int)((long long)p.rows * blockIdx.x / gridDim.x), end = (int)((long long)p.rows * (blockIdx.x + 1) / gridDim.x);
    bool ok = true;
    if (warp < kRowWarps) {
        // ------------------------------ half-resolution rows ------------------------------
        const int jx = threadIdx.x;                      // pixel of the row: half-resolution column jx - 2
        const bool mine = jx < p.pitch;
        uint32_t slot = 0, phase = 0;
        for (int b = begin; b < end && ok;) {
            const Segment s = segment_at(p, b, end);
            const int last = s.last_row + 1;
            uint32_t next[2 * C];
            if (mine) load_pixel<F32, C>(p, s.n, s.first_row - 2, jx - 2, paired != 0, next);
            for (int i = s.first_row - 2; i <= last; ++i) {
                uint32_t v[2 * C];
#pragma unroll
                for (int e = 0; e < 2 * C; ++e) v[e] = next[e];
                if (mine && i < last) load_pixel<F32, C>(p, s.n, i + 1, jx - 2, paired != 0, next);
                ok = __all_sync(0xffffffffu, mbar_wait(x_empty0 + 8 * slot, phase ^ 1, abort_flag));
                if (!ok) break;
                if (mine) {
                    // channel (2a + b) C + c: the b = 0 values of a row's channels, then the b = 1 values
                    uint32_t h[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) h[e] = 0u;
#pragma unroll
                    for (int a = 0; a < 2; ++a)
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            h[2 * a * C + c] = v[a * C + c] & 0xffffu;
                            h[(2 * a + 1) * C + c] = v[a * C + c] >> 16;
                        }
                    uint4* at = ring + (size_t)slot * p.pitch + jx;
                    at[0] = make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
                    at[p.plane] = make_uint4(h[8] | (h[9] << 16), h[10] | (h[11] << 16), h[12] | (h[13] << 16), h[14] | (h[15] << 16));
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
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(K_pad >> 3) << 17) | ((128u >> 4) << 24);
        const uint32_t b_lo0 = (b_addr >> 4) | ((uint32_t)K_pad << 16), b_step = 2u * (uint32_t)K_pad;
        const uint32_t x_lo0 = (x_addr >> 4) | ((uint32_t)p.plane << 16);
        auto wait_for = [&](uint32_t bar, uint32_t ph) { return __all_sync(0xffffffffu, mbar_wait(bar, ph, abort_flag)); };
        ok = wait_for(b_full, 0);
        uint32_t slot = 0, phase = 0;                    // of the newest row waited for
        uint32_t acc = 0, acc_phase = 0;
        for (int b = begin; b < end && ok;) {
            const Segment s = segment_at(p, b, end);
            uint32_t first = slot;                       // ring place of the row's tap 0
            for (int r = s.first_row; r <= s.last_row && ok; ++r) {
                for (int w = r == s.first_row ? 4 : 1; w > 0 && ok; --w) {
                    ok = wait_for(x_full0 + 8 * slot, phase);
                    if (++slot == kRing) { slot = 0; phase ^= 1; }
                }
                if (!ok || !(ok = wait_for(acc_empty0 + 8 * acc, acc_phase ^ 1))) break;
                tc_fence_after();
                const uint32_t d = tmem_base + acc * (uint32_t)K_pad;
                uint32_t b_lo = b_lo0;
#pragma unroll 1
                for (int ta = 0; ta < 4; ++ta) {
                    const uint32_t a_row = x_lo0 + ((first + (uint32_t)ta) & (kRing - 1)) * (uint32_t)p.pitch;
#pragma unroll
                    for (int tb = 0; tb < 4; ++tb) umma_bf16_lo_if(leader, d, a_row + (uint32_t)tb, b_lo + (uint32_t)tb * b_step, idesc, (ta | tb) ? 1u : 0u);
                    b_lo += 4u * b_step;
                }
                if (leader) {
                    umma_commit(acc_full0 + 8 * acc);
                    umma_commit(x_empty0 + 8 * first);
                    if (r == s.last_row)                 // nobody reads the segment's last rows again
                        for (uint32_t t = 1; t < 4; ++t) umma_commit(x_empty0 + 8 * ((first + t) & (kRing - 1)));
                }
                __syncwarp();
                first = (first + 1) & (kRing - 1);
                if (++acc == (uint32_t)p.acc_rows) { acc = 0; acc_phase ^= 1; }
            }
            b += s.q1 - s.q0;
        }
    } else {
        // ------------------------------ pooling ------------------------------
        const int pw = warp - (kRowWarps + 1), quarter = warp & 3, half = pw >> 2;
        const int col = quarter * 32 + lane;             // convolution column; filter groups half, half + 2, ...
        const int groups = ((K_pad >> 4) - half + 1) >> 1;
        const bool live = col < p.Wc;
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + 16u * (uint32_t)half;
        const int Wq = p.Wp + 2, P2o = (p.Hp + 2) * Wq;
        const long long plane_out = (long long)p.a.N * P2o;
        uint4* yout = reinterpret_cast<uint4*>(p.a.y);
        uint32_t acc = 0, acc_phase = 0;
        uint32_t m[NG][8];                       // the row carried over, then the maxima so far: bf16 pairs
        auto hmax = [](uint32_t a, uint32_t b) {
            const __nv_bfloat162 r = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
            return *reinterpret_cast<const uint32_t*>(&r);
        };
        // the next convolution row: its values become the row carried over in `keep`, the maxima in m take them in
        // (a warp whose wait ran out goes on without its rows: the others of its half count on it at their barrier)
        auto take_row = [&](uint32_t (&keep)[NG][8], bool into_max) {
            if (!ok || !(ok = __all_sync(0xffffffffu, mbar_wait(acc_full0 + 8 * acc, acc_phase, abort_flag)))) {
                if (lane == 0) atomicExch(&ctrl->abort_flag, 1);
                return;
            }
            tc_fence_after();
#pragma unroll
            for (int g = 0; g < NG; ++g)
                if (g < groups) {
                    const float4* b4 = reinterpret_cast<const float4*>(bias_s + 16 * half + 32 * g);
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        uint32_t v[8];
                        tmem_ld8(taddr + acc * (uint32_t)K_pad + 32u * (uint32_t)g + 8u * (uint32_t)k, v);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float4 bb = b4[2 * k + e];
                            const uint32_t lo = pack_bf16x2_relu(__uint_as_float(v[4 * e]) + bb.x, __uint_as_float(v[4 * e + 1]) + bb.y);
                            const uint32_t hi = pack_bf16x2_relu(__uint_as_float(v[4 * e + 2]) + bb.z, __uint_as_float(v[4 * e + 3]) + bb.w);
                            const int at = 4 * k + 2 * e;
                            keep[g][at] = live ? lo : 0u;
                            keep[g][at + 1] = live ? hi : 0u;
                            if (into_max) { m[g][at] = hmax(m[g][at], keep[g][at]); m[g][at + 1] = hmax(m[g][at + 1], keep[g][at + 1]); }
                        }
                    }
                }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty0 + 8 * acc);
            if (++acc == (uint32_t)p.acc_rows) { acc = 0; acc_phase ^= 1; }
        };
        int parity = 0;
        for (int b = begin; b < end;) {
            const Segment s = segment_at(p, b, end);
#pragma unroll
            for (int g = 0; g < NG; ++g)
#pragma unroll
                for (int e = 0; e < 8; ++e) m[g][e] = 0u;
            if (s.q0 > 0) take_row(m, false);
            for (int q = s.q0; q < s.q1; ++q) {
                uint32_t last[NG][8];
#pragma unroll
                for (int g = 0; g < NG; ++g)
#pragma unroll
                    for (int e = 0; e < 8; ++e) last[g][e] = 0u;
                take_row(last, true);
                if (2 * q + 1 < p.Hc) {
                    take_row(last, true);
                } else {
#pragma unroll
                    for (int g = 0; g < NG; ++g)
#pragma unroll
                        for (int e = 0; e < 8; ++e) last[g][e] = 0u;
                }
                // across the columns: the neighbours' maxima; lane 0's left neighbour is the previous warp's last lane
                if (lane == 31) {
#pragma unroll
                    for (int g = 0; g < NG; ++g)
                        if (g < groups) {
                            ctrl->edge[parity][half][quarter][g][0] = make_uint4(m[g][0], m[g][1], m[g][2], m[g][3]);
                            ctrl->edge[parity][half][quarter][g][1] = make_uint4(m[g][4], m[g][5], m[g][6], m[g][7]);
                        }
                }
                asm volatile("bar.sync %0, 128;" ::"r"(1 + half) : "memory");
                uint4* y_row = yout + (long long)s.n * P2o + (long long)(q + 1) * Wq;
#pragma unroll
                for (int g = 0; g < NG; ++g)
                    if (g < groups) {
                        uint4 e0 = make_uint4(0, 0, 0, 0), e1 = e0;
                        if (lane == 0 && quarter > 0) { e0 = ctrl->edge[parity][half][quarter - 1][g][0]; e1 = ctrl->edge[parity][half][quarter - 1][g][1]; }
                        const uint32_t edge[8] = {e0.x, e0.y, e0.z, e0.w, e1.x, e1.y, e1.z, e1.w};
                        uint32_t o[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            uint32_t l = __shfl_up_sync(0xffffffffu, m[g][e], 1);
                            const uint32_t r = __shfl_down_sync(0xffffffffu, m[g][e], 1);
                            if (lane == 0) l = edge[e];
                            o[e] = hmax(hmax(l, r), m[g][e]);
                            m[g][e] = last[g][e];
                        }
                        const int chunk = 2 * half + 4 * g;
                        uint4* y0 = y_row + (long long)chunk * plane_out;
                        if (live && (lane & 1) == 0) {
                            y0[(col >> 1) + 1] = make_uint4(o[0], o[1], o[2], o[3]);
                            y0[plane_out + (col >> 1) + 1] = make_uint4(o[4], o[5], o[6], o[7]);
                        }
                        // the zero border: two columns of this row, and the rows above and below the image
                        if (quarter == 0 && (lane & 1) && lane < 8) {
                            uint4* z = y0 + (lane & 2 ? plane_out : 0) + (lane & 4 ? Wq - 1 : 0);
                            *z = make_uint4(0, 0, 0, 0);
                        }
                        if (q == 0 || q == p.Hp - 1)
                            for (int k = col; k < Wq; k += 128) {
                                if (q == 0) { y0[k - Wq] = make_uint4(0, 0, 0, 0); y0[plane_out + k - Wq] = make_uint4(0, 0, 0, 0); }
                                if (q == p.Hp - 1) { y0[k + Wq] = make_uint4(0, 0, 0, 0); y0[plane_out + k + Wq] = make_uint4(0, 0, 0, 0); }
                            }
                    }
                parity ^= 1;
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

struct Shape { int Hc, Wc, Hp, Wp, pitch, plane, b_bytes; unsigned smem; };
Shape shape_of(int H, int W, int K_pad) {
    Shape s;
    s.Hc = (H - 1) / 2 + 1; s.Wc = (W - 1) / 2 + 1; s.Hp = (s.Hc - 1) / 2 + 1; s.Wp = (s.Wc - 1) / 2 + 1;
    s.pitch = s.Wc + 3;
    s.plane = (kRing * s.pitch + 128 + 7) & ~7;
    s.b_bytes = kTaps * 2 * K_pad * 16;
    s.smem = (unsigned)sizeof(SpCtrl) + (unsigned)K_pad * 4u + 128u + (unsigned)s.b_bytes + 2u * (unsigned)s.plane * 16u;
    return s;
}

typedef void (*StemKernel)(const SpParams, const int);
template <bool F32>
StemKernel kernel_of(int C, int K_pad) {
    if (K_pad <= 64) return C == 3 ? stem_pool_kernel<F32, 3, 2> : C == 2 ? stem_pool_kernel<F32, 2, 2> : stem_pool_kernel<F32, 1, 2>;
    return C == 3 ? stem_pool_kernel<F32, 3, 3> : C == 2 ? stem_pool_kernel<F32, 2, 3> : stem_pool_kernel<F32, 1, 3>;
}
StemKernel kernel_of(const StemPoolArgs& a) { return a.in_f32 ? kernel_of<true>(a.C, a.K_pad) : kernel_of<false>(a.C, a.K_pad); }

}  // namespace

// A convolution row is one tile of 128 positions, so images up to 256 wide.
bool stem_pool_supported(int C, int H, int W, int K_pad) {
    if (C < 1 || C > 3 || H < 8 || W < 8 || W > 256 || K_pad % 16 || K_pad < 16 || K_pad > 32 * kMaxGroups) return false;
    return shape_of(H, W, K_pad).smem <= kSmemMax;
}

int plan_stem_pool(const StemPoolArgs& a, StemPoolPlan* plan, char* err, size_t err_len) {
    memset(plan, 0, sizeof(*plan));
    if (!stem_pool_supported(a.C, a.H, a.W, a.K_pad)) { snprintf(err, err_len, "first convolution + pooling: shape not supported"); return 1; }
    plan->smem_bytes = shape_of(a.H, a.W, a.K_pad).smem;
    plan->tmem_cols = 256;                               // half of an SM's, for two CTAs
    plan->acc_rows = std::min(kMaxAcc, plan->tmem_cols / a.K_pad);
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
    p.Hc = s.Hc; p.Wc = s.Wc; p.Hp = s.Hp; p.Wp = s.Wp; p.pitch = s.pitch; p.plane = s.plane; p.b_bytes = s.b_bytes;
    p.acc_rows = plan.acc_rows; p.tmem_cols = plan.tmem_cols;
    p.rows = a.n_count * s.Hp;
    p.status = d_status;
    // two columns with one load where a row's pairs are aligned
    const int paired = a.W % 2 == 0 && (uintptr_t)a.x % (a.in_f32 ? 8 : 4) == 0;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)std::max(1, std::min((a.K_pad <= 64 ? 2 : 1) * sm_count(), p.rows)));
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
