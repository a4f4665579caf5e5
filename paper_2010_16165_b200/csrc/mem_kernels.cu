// Memory-bound operators of the fused graph in the planar-8 layout with a zero border (see
// fp_internal.h): boundary layout conversion, max pooling, the global-average-pool + FC head,
// and a debug dump.  One thread handles one vector (8 channels of one pixel), so a warp touches
// 32 consecutive vectors of a chunk plane: 512 contiguous bytes of bf16.
#include "fp_internal.h"

#include <algorithm>
#include <atomic>
#include <cstring>

namespace fp {

namespace {

struct __align__(16) Vec8h { __nv_bfloat162 v[4]; };
struct __align__(32) Vec8f { float v[8]; };

template <bool BF16>
__device__ __forceinline__ void load_vec8(const void* base, size_t vec, float (&f)[8]) {
    if constexpr (BF16) {
        const Vec8h r = reinterpret_cast<const Vec8h*>(base)[vec];
#pragma unroll
        for (int i = 0; i < 4; ++i) { const float2 g = __bfloat1622float2(r.v[i]); f[2 * i] = g.x; f[2 * i + 1] = g.y; }
    } else {
        const Vec8f r = reinterpret_cast<const Vec8f*>(base)[vec];
#pragma unroll
        for (int i = 0; i < 8; ++i) f[i] = r.v[i];
    }
}

template <bool BF16>
__device__ __forceinline__ void store_vec8(void* base, size_t vec, const float (&f)[8]) {
    if constexpr (BF16) {
        Vec8h r;
#pragma unroll
        for (int i = 0; i < 4; ++i) r.v[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
        reinterpret_cast<Vec8h*>(base)[vec] = r;
    } else {
        Vec8f r;
#pragma unroll
        for (int i = 0; i < 8; ++i) r.v[i] = f[i];
        reinterpret_cast<Vec8f*>(base)[vec] = r;
    }
}

// NCHW (fp32 or bf16) -> planar-8 with border.  Thread = (chunk, flat position); reads of one
// channel plane are coalesced along w, writes are contiguous vectors.
// Images n0 .. n0 + n_count - 1 of a batch of N (the others are left alone: a caller that receives its input in
// pieces converts each piece as it arrives).
template <bool OUT_BF16>
__global__ void input_to_planar_kernel(const void* __restrict__ in, int in_is_bf16, void* __restrict__ out, int N, int C,
                                       int H, int W, int chunks, int n0, int n_count) {
    const int Wp = row_vecs(W), P2 = image_vecs(H, W);
    const size_t plane = (size_t)plane_vecs(N, H, W);
    const size_t part = (size_t)n_count * P2 + (n0 + n_count == N ? W + 2 : 0);      // the last images' part: with the zeros behind them
    const size_t total = part * chunks;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int j = (int)(i / part);
        const size_t f = i - (size_t)j * part;
        const size_t n = n0 + f / P2;
        const int rem = (int)(f % P2);
        const int h = rem / Wp - 1, w = rem % Wp - 1;
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = 0.0f;
        if (h >= 0 && h < H && w >= 0 && w < W) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int c = j * 8 + e;
                if (c < C) {
                    const size_t src = ((n * C + c) * H + h) * W + w;
                    v[e] = in_is_bf16 ? __bfloat162float(((const __nv_bfloat16*)in)[src]) : ((const float*)in)[src];
                }
            }
        }
        store_vec8<OUT_BF16>(out, (size_t)j * plane + n * P2 + rem, v);
    }
}

// Network input for a 7x7 / stride-2 / pad-3 first convolution with at most 3 input channels, packed so
// that the convolution becomes a stride-1 3x1 convolution at the output resolution (P = H/2, Q = W/2):
// the 7 horizontal taps and the input channels become 24 packed channels j = s*C + c, and the input
// rows are split by parity into three 24-channel groups
//     E (chunks 0-2):  E [p][q][j] = x[c][2p    ][2q + s - 3]
//     O'(chunks 3-5):  O'[p][q][j] = x[c][2p - 1][2q + s - 3]      (odd rows, shifted down by one)
//     O (chunks 6-8):  O [p][q][j] = x[c][2p + 1][2q + s - 3]
// (chunk 9 is zero padding to an even chunk count).  Output row p needs input rows 2p-3 .. 2p+3, which
// are O'(p-1), E(p-1), O'(p), E(p), O(p), E(p+1), O(p+1): vertical offsets -1, 0, +1 only.
// One block per (image, output row incl. the border row): the three input rows the output row needs are
// staged in shared memory (coalesced reads, each input element read once per block), then every thread builds
// packed vectors from them.  32-bit index arithmetic only.
__global__ void input_to_stem_planar_kernel(const void* __restrict__ in, int in_is_bf16, __nv_bfloat16* __restrict__ out,
                                            int N, int C, int H, int W, int n0) {
    extern __shared__ float rows[];                  // [3 rows: 2p-1, 2p, 2p+1][C][W + 6], zero where outside the image
    __shared__ int tap_off[24];                      // packed channel j = s*C + c -> c*(W+6) + s, or -1 (padding)
    const int P = H / 2, Q = W / 2, Qp = row_vecs(Q), P2 = image_vecs(P, Q);
    const int n = n0 + blockIdx.x / (P + 1), pp = blockIdx.x % (P + 1);
    const int p = pp - 1;
    const size_t plane = (size_t)plane_vecs(N, P, Q);
    uint4* outv = reinterpret_cast<uint4*>(out) + (size_t)n * P2 + (size_t)pp * Qp;
    if (n == N - 1 && p == P - 1)                    // the zeros behind the last image
        for (int i = threadIdx.x; i < 10 * (Q + 2); i += blockDim.x) outv[(size_t)(i / (Q + 2)) * plane + Qp + i % (Q + 2)] = make_uint4(0, 0, 0, 0);
    if (p < 0) {                                     // border row: zeros in every chunk
        for (int i = threadIdx.x; i < 10 * Qp; i += blockDim.x) {
            const int j8 = i / Qp, qq = i - j8 * Qp;
            outv[(size_t)j8 * plane + qq] = make_uint4(0, 0, 0, 0);
        }
        return;
    }
    const int Ws = W + 6;
    if (threadIdx.x < 24) {
        const int sx = threadIdx.x / C, c = threadIdx.x - sx * C;
        tap_off[threadIdx.x] = sx < 7 ? c * Ws + sx : -1;
    }
    for (int i = threadIdx.x; i < 3 * C * Ws; i += blockDim.x) {
        const int rc = i / Ws, col = i - rc * Ws;
        const int r = rc / C, c = rc - r * C;
        const int ih = 2 * p - 1 + r, iw = col - 3;
        float v = 0.0f;
        if (ih >= 0 && ih < H && iw >= 0 && iw < W) {
            const size_t src = (((size_t)n * C + c) * H + ih) * W + iw;
            v = in_is_bf16 ? __bfloat162float(((const __nv_bfloat16*)in)[src]) : ((const float*)in)[src];
        }
        rows[i] = v;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 10 * Qp; i += blockDim.x) {
        const int j8 = i / Qp, qq = i - j8 * Qp;
        const int q = qq - 1;
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = 0.0f;
        if (j8 < 9 && q >= 0 && q < Q) {
            const int group = j8 / 3;                // 0 = E (row 2p), 1 = O' (row 2p-1), 2 = O (row 2p+1)
            const int r = group == 0 ? 1 : group == 1 ? 0 : 2;
            const float* base = rows + r * C * Ws + 2 * q;          // input column 2q + s - 3 sits at 2q + s
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int off = tap_off[(j8 - group * 3) * 8 + e];
                if (off >= 0) v[e] = base[off];
            }
        }
        Vec8h o;
#pragma unroll
        for (int e = 0; e < 4; ++e) o.v[e] = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
        reinterpret_cast<Vec8h*>(outv)[(size_t)j8 * plane + qq] = o;
    }
}

// The same packing for exactly three input channels (RGB): with C fixed, tap s and channel c of packed channel j
// are compile-time constants, so a vector is eight shared-memory loads at immediate offsets (no table, no
// divisions), and the rows are staged row by row.  One thread per output column.
__global__ void input_to_stem_planar_rgb_kernel(const void* __restrict__ in, int in_is_bf16, __nv_bfloat16* __restrict__ out,
                                                int N, int H, int W, int n0) {
    constexpr int C = 3;
    extern __shared__ float rows[];                  // [3 rows: 2p-1, 2p, 2p+1][C][W + 6], zero where outside the image
    const int P = H / 2, Q = W / 2, Qp = row_vecs(Q), P2 = image_vecs(P, Q);
    const int n = n0 + blockIdx.x / (P + 1), pp = blockIdx.x % (P + 1);
    const int p = pp - 1;
    const size_t plane = (size_t)plane_vecs(N, P, Q);
    Vec8h* outv = reinterpret_cast<Vec8h*>(out) + (size_t)n * P2 + (size_t)pp * Qp;
    Vec8h zero;
#pragma unroll
    for (int e = 0; e < 4; ++e) zero.v[e] = __floats2bfloat162_rn(0.0f, 0.0f);
    if (n == N - 1 && p == P - 1)                    // the zeros behind the last image
        for (int i = threadIdx.x; i < 10 * (Q + 2); i += blockDim.x) outv[(size_t)(i / (Q + 2)) * plane + Qp + i % (Q + 2)] = zero;
    if (p < 0) {                                     // border row: zeros in every chunk
        for (int j8 = 0; j8 < 10; ++j8)
            for (int qq = threadIdx.x; qq < Qp; qq += blockDim.x) outv[(size_t)j8 * plane + qq] = zero;
        return;
    }
    const int Ws = W + 6;
    for (int rc = 0; rc < 3 * C; ++rc) {
        const int r = rc / C, c = rc - r * C;
        const int ih = 2 * p - 1 + r;
        const bool row_in = ih >= 0 && ih < H;
        const size_t src = (((size_t)n * C + c) * H + (row_in ? ih : 0)) * W;
        for (int col = threadIdx.x; col < Ws; col += blockDim.x) {
            const int iw = col - 3;
            float v = 0.0f;
            if (row_in && iw >= 0 && iw < W)
                v = in_is_bf16 ? __bfloat162float(((const __nv_bfloat16*)in)[src + iw]) : ((const float*)in)[src + iw];
            rows[rc * Ws + col] = v;
        }
    }
    __syncthreads();
    for (int qq = threadIdx.x; qq < Qp; qq += blockDim.x) {
        const int q = qq - 1;
        const bool inside = q >= 0 && q < Q;
#pragma unroll
        for (int group = 0; group < 3; ++group) {    // 0 = E (row 2p), 1 = O' (row 2p-1), 2 = O (row 2p+1)
            const int r = group == 0 ? 1 : group == 1 ? 0 : 2;
            const float* base = rows + r * C * Ws + (inside ? 2 * q : 0);    // input column 2q + s - 3 sits at 2q + s
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                float v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int j = k * 8 + e, sx = j / C, c = j - sx * C;     // constants after unrolling
                    v[e] = (sx < 7 && inside) ? base[c * Ws + sx] : 0.0f;
                }
                Vec8h o;
#pragma unroll
                for (int e = 0; e < 4; ++e) o.v[e] = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
                outv[(size_t)(group * 3 + k) * plane + qq] = o;
            }
        }
        outv[(size_t)9 * plane + qq] = zero;
    }
}

// Max pooling; padded positions never win.  Output border positions are written as zeros.
// blockIdx.x = (chunk, image, output row incl. borders), threads run along the row: no divisions per element,
// 32-bit arithmetic, and a warp reads runs of neighbouring vectors.
template <bool BF16>
__global__ void maxpool_kernel(const void* __restrict__ x, void* __restrict__ y, int N, int H, int W, int chunks, int P,
                               int Q, int R, int stride, int pad) {
    const int Wp = row_vecs(W), Qp = row_vecs(Q);
    const int rows_per_image = P + 1;
    const int row = blockIdx.x * blockDim.y + threadIdx.y;
    if (row >= chunks * N * rows_per_image) return;
    const int jn = row / rows_per_image, pp = row - jn * rows_per_image;     // jn = chunk * N + image
    const int p = pp - 1, j = jn / N, n = jn - j * N;
    const size_t in_base = (size_t)j * plane_vecs(N, H, W) + (size_t)n * image_vecs(H, W);
    const size_t out_base = (size_t)j * plane_vecs(N, P, Q) + (size_t)n * image_vecs(P, Q) + (size_t)pp * Qp;
    for (int qq = threadIdx.x; qq < Qp; qq += blockDim.x) {
        const int q = qq - 1;
        float m[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) m[e] = 0.0f;
        if (p >= 0 && p < P && q >= 0 && q < Q) {
#pragma unroll
            for (int e = 0; e < 8; ++e) m[e] = -INFINITY;
            for (int r = 0; r < R; ++r) {
                const int ih = p * stride + r - pad;
                if (ih < 0 || ih >= H) continue;
                for (int sx = 0; sx < R; ++sx) {
                    const int iw = q * stride + sx - pad;
                    if (iw < 0 || iw >= W) continue;
                    float v[8];
                    load_vec8<BF16>(x, in_base + (size_t)((ih + 1) * Wp + (iw + 1)), v);
#pragma unroll
                    for (int e = 0; e < 8; ++e) m[e] = fmaxf(m[e], v[e]);
                }
            }
        }
        store_vec8<BF16>(y, out_base + qq, m);
    }
    if (n == N - 1 && p == P - 1) {                  // the zeros behind the last image
        const float zeros[8] = {};
        for (int i = threadIdx.x; i < Q + 2; i += blockDim.x) store_vec8<BF16>(y, out_base + Qp + i, zeros);
    }
}

// 3x3 / stride-2 / pad-1 max pooling of bf16 activations, the ImageNet stem's pooling.  The generic kernel above
// issues nine 16-byte loads per output whose addresses are 32 bytes apart between neighbouring threads (eight
// cache lines per warp-wide load), and the L1 pipeline, not DRAM, bounds it.  Here a warp that owns 32 neighbouring
// outputs reads the 64 input columns under them with two fully coalesced loads per input row (lane l holds
// columns 2*q0 + l and 2*q0 + 32 + l; lane 0 also fetches column 2*q0 - 1), takes the maximum down the three rows
// first, then across each window of three columns with warp shuffles.  The maximum of bf16 values is one of them,
// so packed bf16 compares give the same result as fp32 ones.  Same block shape as the generic kernel.
__device__ __forceinline__ Vec8h vmax(const Vec8h& a, const Vec8h& b) {
    Vec8h r;
#pragma unroll
    for (int i = 0; i < 4; ++i) r.v[i] = __hmax2(a.v[i], b.v[i]);
    return r;
}
__device__ __forceinline__ Vec8h vshfl(const Vec8h& a, int src_lane) {
    Vec8h r;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t w = __shfl_sync(0xffffffffu, *reinterpret_cast<const uint32_t*>(&a.v[i]), src_lane);
        r.v[i] = *reinterpret_cast<const __nv_bfloat162*>(&w);
    }
    return r;
}
__global__ void maxpool3s2_bf16_kernel(const Vec8h* __restrict__ x, Vec8h* __restrict__ y, int N, int H, int W, int chunks,
                                       int P, int Q) {
    const int Wp = row_vecs(W), Qp = row_vecs(Q);
    const int rows_per_image = P + 1;
    const int row = blockIdx.x * blockDim.y + threadIdx.y;
    if (row >= chunks * N * rows_per_image) return;                           // the same for a whole warp
    const int jn = row / rows_per_image, pp = row - jn * rows_per_image;     // jn = chunk * N + image
    const int p = pp - 1, j = jn / N, n = jn - j * N;
    const size_t in_base = (size_t)j * plane_vecs(N, H, W) + (size_t)n * image_vecs(H, W);
    const size_t out_base = (size_t)j * plane_vecs(N, P, Q) + (size_t)n * image_vecs(P, Q) + (size_t)pp * Qp;
    const int lane = threadIdx.x & 31;
    Vec8h ninf, zero;
#pragma unroll
    for (int i = 0; i < 4; ++i) { ninf.v[i] = __floats2bfloat162_rn(-INFINITY, -INFINITY); zero.v[i] = __floats2bfloat162_rn(0.0f, 0.0f); }
    for (int qq0 = threadIdx.x - lane; qq0 < Qp; qq0 += blockDim.x) {         // warp-uniform: all 32 lanes take part
        const int qq = qq0 + lane, q = qq - 1;
        if (p < 0) {                                                          // border row: zeros
            if (qq < Qp) y[out_base + qq] = zero;
            continue;
        }
        const int c0 = 2 * (qq0 - 1);                  // input column under the warp's first output
        const int ca = c0 + lane, cb = c0 + 32 + lane, ce = c0 - 1;
        Vec8h A = ninf, B = ninf, E = ninf;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int ih = 2 * p - 1 + r;
            if (ih < 0 || ih >= H) continue;
            const Vec8h* src = x + in_base + (size_t)(ih + 1) * Wp + 1;
            if (ca >= 0 && ca < W) A = vmax(A, src[ca]);
            if (cb >= 0 && cb < W) B = vmax(B, src[cb]);
            if (lane == 0 && ce >= 0 && ce < W) E = vmax(E, src[ce]);
        }
        // windows centred on the even lanes: W_A[l] = max(A[l-1], A[l], A[l+1]) with A[-1] = E; W_B alike with B[-1] = A[31]
        Vec8h upA = vshfl(A, (lane + 31) & 31), dnA = vshfl(A, (lane + 1) & 31);
        Vec8h upB = vshfl(B, (lane + 31) & 31), dnB = vshfl(B, (lane + 1) & 31);
        const Vec8h a31 = upA;                          // on lane 0 the rotation delivered A[31]
        if (lane == 0) { upA = E; upB = a31; }
        const Vec8h WA = vmax(vmax(upA, A), dnA), WB = vmax(vmax(upB, B), dnB);
        // output j of the warp sits over columns 2j-1 .. 2j+1: window 2j of A (j < 16) or 2j-32 of B
        const Vec8h fa = vshfl(WA, (2 * lane) & 31), fb = vshfl(WB, (2 * lane) & 31);
        if (qq < Qp) y[out_base + qq] = (q >= 0 && q < Q) ? (lane < 16 ? fa : fb) : zero;
    }
    if (n == N - 1 && p == P - 1)                                             // the zeros behind the last image
        for (int i = threadIdx.x; i < Q + 2; i += blockDim.x) y[out_base + Qp + i] = zero;
}

// Head, step 1: spatial sum per channel in fp32.  One warp per (image, chunk of 8 channels): lanes stride over the interior
// positions with 16-byte loads, then the lanes' eight sums are added with nine shuffles - every exchange halves the channels
// a lane still carries - instead of five per channel (ResNet-50 at batch 128, 32768 warps: the shuffles were half of 17 us).
// (x here and sums below are the previous kernel's: not __restrict__, so that no load of them moves in front of the wait for it.)
template <bool BF16>
__global__ void pool_sum_kernel(const void* x, int N, int H, int W, int chunks, float* __restrict__ sums) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int Wp = row_vecs(W), P2 = image_vecs(H, W), HW = H * W;
    const size_t plane = (size_t)plane_vecs(N, H, W);
    const int lane = threadIdx.x & 31;
    const unsigned warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (warp >= (unsigned)N * (unsigned)chunks) return;
    const unsigned n = warp / (unsigned)chunks, j = warp - n * (unsigned)chunks;
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.0f;
    for (int i = lane; i < HW; i += 64) {  // two positions' loads in flight
        float v[2][8];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int at = min(i + 32 * k, HW - 1), h = at / W, w = at - h * W;
            load_vec8<BF16>(x, (size_t)j * plane + (size_t)n * P2 + (size_t)(h + 1) * Wp + (w + 1), v[k]);
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] += v[0][e];
        if (i + 32 < HW)
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] += v[1][e];
    }
    int first = 0;                         // of the channels this lane still carries
#pragma unroll
    for (int d = 16, keep = 4; d >= 4; d >>= 1, keep >>= 1) {
        const bool up = (lane & d) != 0;   // keeps the upper half, hands the lower one over
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (e < keep) {
                const float give = up ? acc[e] : acc[e + keep];
                const float got = __shfl_xor_sync(0xffffffffu, give, d);
                acc[e] = (up ? acc[e + keep] : acc[e]) + got;
            }
        if (up) first += keep;
    }
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 2);
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
    if ((lane & 3) == 0) sums[(size_t)n * chunks * 8 + j * 8 + first] = acc[0];
}

// Head, step 2: logits[n][k] = sum_c sums[n][c] * Wfc[k][c] + b[k]; the 1/(H*W) of the average is already folded into Wfc.
// A block handles IMAGES images (one, four or eight: the sums of images that do not exist would be computed as well), whose channel sums it holds in shared memory, and 8 * CPW classes: a warp walks the FC
// rows of its CPW classes with 16-byte loads, all images a time.  The first rows are asked for before the channel sums
// exist (programmatic dependent launch).  Each (image, class) sum has a fixed order: lanes stride over the channels, then a
// butterfly (the kernels for handles made for many images, below, have another).  CPW: every sum read from shared memory serves CPW classes, which bounds large batches (128 images x 1000 classes
// x 2048 channels: 7 us of FMAs at full rate, four classes a warp bring the shared-memory reads down to that); one class a warp
// spreads the FC matrix of a single image over 125 SMs instead of 32.
constexpr int kFcWarps = 8, kFcSlab4 = 512, kFcPitch4 = kFcSlab4 + 1;       // channels / 4 held at a time, and a zero behind them
// AHEAD: places of the rows a lane has on the way at a time; a place is asked for again as soon as it has been used.
template <int IMAGES, int CPW, int AHEAD>
__global__ void __launch_bounds__(32 * kFcWarps, 2) fc_kernel(const float* sums, int N, int C_pad, const float* __restrict__ fcw,
                                                           const float* __restrict__ fcb, int n_classes, float* __restrict__ logits) {
    extern __shared__ float4 sh4[];        // IMAGES x kFcPitch4
    const int n0 = blockIdx.x * IMAGES;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k0 = ((int)(blockIdx.z * gridDim.y + blockIdx.y) * kFcWarps + warp) * CPW, c4 = C_pad >> 2;
    const float4* wr[CPW];
    float4 w[CPW][AHEAD];
    auto rows = [&](int c, int i) {        // 128 channels of the warp's rows, zeros behind the last
#pragma unroll
        for (int t = 0; t < CPW; ++t) w[t][i] = c < c4 ? __ldg(wr[t] + c) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    };
#pragma unroll
    for (int t = 0; t < CPW; ++t) wr[t] = reinterpret_cast<const float4*>(fcw + (size_t)min(k0 + t, n_classes - 1) * C_pad);
#pragma unroll
    for (int i = 0; i < AHEAD; ++i) rows(lane + 32 * i, i);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int images = min(IMAGES, N - n0);
    float acc[CPW][IMAGES];
#pragma unroll
    for (int t = 0; t < CPW; ++t)
#pragma unroll
        for (int i = 0; i < IMAGES; ++i) acc[t][i] = 0.0f;
    for (int slab = 0; slab < c4; slab += kFcSlab4) {
        const int n4 = min(kFcSlab4, c4 - slab);
        if (slab) __syncthreads();         // the previous slab has been consumed
        for (int img = warp; img < IMAGES; img += kFcWarps) {
            const float4* from = reinterpret_cast<const float4*>(sums + (size_t)(n0 + min(img, images - 1)) * C_pad) + slab;
            for (int i = lane; i < n4; i += 32) sh4[img * kFcPitch4 + i] = from[i];
            if (lane == 0) sh4[img * kFcPitch4 + n4] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        __syncthreads();
        for (int c = lane; c < n4; c += 32 * AHEAD) {                // (a slab that is not the last is a multiple of that)
#pragma unroll
            for (int i = 0; i < AHEAD; ++i) {
                const int cc = min(c + 32 * i, n4);      // behind the last channel a zero, as the rows' are: a sum that is infinite would make them NaN
#pragma unroll
                for (int img = 0; img < IMAGES; ++img) {
                    const float4 s = sh4[img * kFcPitch4 + cc];
#pragma unroll
                    for (int t = 0; t < CPW; ++t)
                        acc[t][img] = fmaf(s.w, w[t][i].w, fmaf(s.z, w[t][i].z, fmaf(s.y, w[t][i].y, fmaf(s.x, w[t][i].x, acc[t][img]))));
                }
                rows(slab + c + 32 * (AHEAD + i), i);
            }
        }
    }
#pragma unroll
    for (int t = 0; t < CPW; ++t) {
        float mine = 0.0f;                 // lane i ends up with image i's sum
#pragma unroll
        for (int img = 0; img < IMAGES; ++img) {
            float v = acc[t][img];
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
            if (lane == img) mine = v;
        }
        if (lane < images && k0 + t < n_classes) logits[(size_t)(n0 + lane) * n_classes + k0 + t] = mine + (fcb ? fcb[k0 + t] : 0.0f);
    }
}

// Head, step 2, of a handle made for many images: a block takes 8 * IPL images times 4 * CPL classes.  Slabs of 128 channels of the sums and of the FC rows go through
// shared memory (two on the way behind the one in use), a warp takes 16 channels of each, a lane IPL images times CPL classes of the tile: a
// vector of 4 channels of an image serves CPL classes and one of a class IPL images, so that (IPL 4, CPL 8) 12 shared-memory reads feed 64
// pairs of FMAs.  (In the kernel above every lane reads its own channels of every image, four wavefronts for 4 classes: both that and the L2
// reads of the FC matrix, once for every 8 images, took longer than the FMAs.)  Channels are added in pairs (one instruction
// for two), each warp's in order, then the pair, then the warps' sums in order: another order than the kernel's above, the same for every
// IPL and CPL.  Which of the two kernels a handle uses goes by the batch it is made for, so that an image's logits do not depend on the
// call it came in.
constexpr int kTileSlab4 = 32, kTilePitch4 = kTileSlab4 + 1;      // (rows 16 bytes off a multiple of 128: no bank twice)
constexpr int kTileStages = 3;
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
constexpr int fc_tile_smem(int ipl, int cpl) { return kTileStages * (4 * cpl + 8 * ipl) * kTilePitch4 * (int)sizeof(float4); }
template <int IPL, int CPL>
__global__ void __launch_bounds__(256, 2) fc_tile_kernel(const float* sums, int N, int C_pad, const float* __restrict__ fcw,
                                                         const float* __restrict__ fcb, int n_classes, float* __restrict__ logits) {
    extern __shared__ float4 sh4[];        // stages: FC rows, then the images' sums
    constexpr int kRows = 256 / kTileSlab4, kImages = 8 * IPL, kTileClasses = 4 * CPL, kStage4 = (kTileClasses + kImages) * kTilePitch4;
    const int n0 = blockIdx.x * kImages, k0 = (int)(blockIdx.z * gridDim.y + blockIdx.y) * kTileClasses, c4 = C_pad >> 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int slabs = (c4 + kTileSlab4 - 1) / kTileSlab4;
    // A thread brings the same channel vector of every eighth row.  Rows of the tile that do not exist repeat the last one (nobody reads
    // what they give); channels behind the last are zeros.
    const int col = threadIdx.x & (kTileSlab4 - 1), row = threadIdx.x / kTileSlab4;
    const uint32_t mine = (uint32_t)__cvta_generic_to_shared(sh4) + (uint32_t)(row * kTilePitch4 + col) * 16u;
    auto fetch_rows = [&](int slab, uint32_t stage, bool images) {
        const int at = slab * kTileSlab4 + col;
        const float* from = (images ? sums : fcw) + 4 * (size_t)min(at, c4 - 1);
        const int first = (images ? n0 : k0) + row, last = (images ? N : n_classes) - 1;
        const uint32_t to = mine + (stage * kStage4 + (images ? kTileClasses * kTilePitch4 : 0)) * 16u;
#pragma unroll
        for (int j = 0; j < (images ? kImages : kTileClasses) / kRows; ++j)
            cp_async16(to + (uint32_t)(kRows * j * kTilePitch4) * 16u, from + (size_t)min(first + kRows * j, last) * C_pad, at < c4);
    };
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
    fetch_rows(0, 0, false);               // the FC matrix does not wait for the kernel before
    if (slabs > 1) fetch_rows(1, 1, false);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    fetch_rows(0, 0, true);
    commit();
    if (slabs > 1) fetch_rows(1, 1, true);
    commit();
    unsigned long long acc[IPL][CPL];
#pragma unroll
    for (int i = 0; i < IPL; ++i)
#pragma unroll
        for (int t = 0; t < CPL; ++t) acc[i][t] = 0ull;
    const int li = lane & 7, lc = lane >> 3;      // image li + 8 i, class lc + 4 t
    uint32_t stage = 0;
    for (int slab = 0; slab < slabs; ++slab) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();                   // this slab is there, and the one before has been used
        if (slab + 2 < slabs) {
            const uint32_t to = stage == 0 ? 2 : stage - 1;
            fetch_rows(slab + 2, to, false);
            fetch_rows(slab + 2, to, true);
        }
        commit();
        const ulonglong2* w = reinterpret_cast<const ulonglong2*>(sh4 + stage * kStage4 + lc * kTilePitch4 + warp * (kTileSlab4 / 8));
        const ulonglong2* s = reinterpret_cast<const ulonglong2*>(sh4 + stage * kStage4 + (kTileClasses + li) * kTilePitch4 + warp * (kTileSlab4 / 8));
#pragma unroll
        for (int c = 0; c < kTileSlab4 / 8; ++c) {
            ulonglong2 sv[IPL];
#pragma unroll
            for (int i = 0; i < IPL; ++i) sv[i] = s[8 * i * kTilePitch4 + c];
#pragma unroll
            for (int t = 0; t < CPL; ++t) {
                const ulonglong2 wv = w[4 * t * kTilePitch4 + c];
#pragma unroll
                for (int i = 0; i < IPL; ++i) {
                    fma2(acc[i][t], sv[i].x, wv.x);
                    fma2(acc[i][t], sv[i].y, wv.y);
                }
            }
        }
        if (++stage == kTileStages) stage = 0;
    }
    __syncthreads();
    float* part = reinterpret_cast<float*>(sh4);                 // [warp][image][class], a float behind every row
#pragma unroll
    for (int i = 0; i < IPL; ++i)
#pragma unroll
        for (int t = 0; t < CPL; ++t) {
            const float2 v = *reinterpret_cast<const float2*>(&acc[i][t]);
            part[(warp * kImages + li + 8 * i) * (kTileClasses + 1) + lc + 4 * t] = v.x + v.y;
        }
    __syncthreads();
    for (int o = threadIdx.x; o < kImages * kTileClasses; o += 256) {
        const int i = o / kTileClasses, t = o - i * kTileClasses;
        float v = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k) v += part[(k * kImages + i) * (kTileClasses + 1) + t];
        if (n0 + i < N && k0 + t < n_classes) logits[(size_t)(n0 + i) * n_classes + k0 + t] = v + (fcb ? fcb[k0 + t] : 0.0f);
    }
}

// Head, step 2, of a call of up to four images on a handle made for many: the tiles' sums in the tiles' order, for one image a block and without the
// tiles' passes through shared memory.  Eight lanes share a class; a lane does what a warp does there, 16 channels of every 128, and the eight
// sums are added in order.  Half of 2048 channels of the FC rows are on the way before the channel sums exist.  What bounds it is that
// latency: a forward of one image (ResNet-18 at 32x32 on a handle made for 24, 512 channels; ResNet-50 at 32x32 made for 64, 2048 channels) takes
// 78.1 and 186.3 us, with tiles of 8 images times 8 classes 82.5 and 191.5, with the first of these kernels, whose order is another, 78.3 and
// 182.9; four images 81.2 and 189.6, 84.0 and 191.1, 80.3 and 187.0.  At eight images the tiles are as fast (82.0, 190.5).
constexpr int kFewImages = 4, kFewWarps = 2, kFewAhead = 8, kFewSlabs = 16;           // slabs of FC rows on the way, of sums held at a time
__global__ void __launch_bounds__(32 * kFewWarps) fc_few_kernel(const float* sums, int N, int C_pad, const float* __restrict__ fcw,
                                                               const float* __restrict__ fcb, int n_classes, float* __restrict__ logits) {
    constexpr int kPitch4 = kTileSlab4 + kTileSlab4 / 4;   // of a slab: behind a lane's four vectors 16 bytes, so that eight lanes meet no bank twice
    __shared__ float4 sh[kFewSlabs * kPitch4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, part = lane & 7, c4 = C_pad >> 2, slabs = (c4 + kTileSlab4 - 1) / kTileSlab4;
    const int n = blockIdx.x, k = ((int)(blockIdx.z * gridDim.y + blockIdx.y) * kFewWarps + warp) * 4 + (lane >> 3);
    const float4* row = reinterpret_cast<const float4*>(fcw + (size_t)min(k, n_classes - 1) * C_pad) + 4 * part;
    float4 w[kFewAhead][4];
    auto fetch = [&](int slab, int i) {    // zeros behind the last channel
#pragma unroll
        for (int c = 0; c < 4; ++c) w[i][c] = kTileSlab4 * slab + 4 * part + c < c4 ? __ldg(row + kTileSlab4 * slab + c) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    };
#pragma unroll
    for (int i = 0; i < kFewAhead; ++i) fetch(i, i);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    unsigned long long acc = 0ull;
    for (int first = 0; first < slabs; first += kFewSlabs) {
        const int n_slabs = min(kFewSlabs, slabs - first);
        const float4* from = reinterpret_cast<const float4*>(sums + (size_t)n * C_pad) + first * kTileSlab4;
        if (first) __syncthreads();        // the slabs before have been used
#pragma unroll 8
        for (int v = threadIdx.x; v < n_slabs * kTileSlab4; v += 32 * kFewWarps)
            sh[v + (v >> 2)] = first * kTileSlab4 + v < c4 ? from[v] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        __syncthreads();
        for (int slab = 0; slab < n_slabs; slab += kFewAhead) {      // (which divides kFewSlabs)
#pragma unroll
            for (int i = 0; i < kFewAhead; ++i) {
                if (slab + i >= n_slabs) break;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const ulonglong2 wv = *reinterpret_cast<const ulonglong2*>(&w[i][c]);
                    const ulonglong2 sv = *reinterpret_cast<const ulonglong2*>(&sh[(slab + i) * kPitch4 + 5 * part + c]);
                    fma2(acc, sv.x, wv.x);
                    fma2(acc, sv.y, wv.y);
                }
                fetch(first + slab + i + kFewAhead, i);
            }
        }
    }
    const float mine = __uint_as_float((uint32_t)acc) + __uint_as_float((uint32_t)(acc >> 32));
    float v = 0.0f;
#pragma unroll
    for (int p = 0; p < 8; ++p) v += __shfl_sync(0xffffffffu, mine, (lane & 24) + p);
    if (part == 0 && k < n_classes) logits[(size_t)n * n_classes + k] = v + (fcb ? fcb[k] : 0.0f);
}

template <bool BF16>
__global__ void planar_to_nchw_f32_kernel(const void* __restrict__ x, float* __restrict__ out, int N, int H, int W,
                                          int chunks, int C_out, int split) {
    // a parity-split tensor (see ConvArgs) is 4 N images of half the size
    const int Hs = split ? (H + 1) / 2 : H, Ws = split ? (W + 1) / 2 : W, Wp = row_vecs(Ws), P2 = image_vecs(Hs, Ws);
    const size_t plane = (size_t)plane_vecs(split ? 4 * N : N, Hs, Ws);
    const size_t total = (size_t)N * chunks * H * W;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int w = (int)(i % W);
        size_t t = i / W;
        const int h = (int)(t % H); t /= H;
        const int j = (int)(t % chunks);
        const size_t n = t / chunks;
        float v[8];
        size_t pos = n * P2 + (size_t)(h + 1) * Wp + (w + 1);
        if (split) {
            const int pp = (h & 1) ? ((w & 1) ? 2 : 1) : ((w & 1) ? 3 : 0);
            pos = ((size_t)pp * N + n) * P2 + (size_t)((h >> 1) + 1) * Wp + ((w >> 1) + 1);
        }
        load_vec8<BF16>(x, (size_t)j * plane + pos, v);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int c = j * 8 + e;
            if (c < C_out) out[((n * C_out + c) * H + h) * W + w] = v[e];
        }
    }
}

inline int grid_for(size_t n, int threads) {
    size_t b = (n + threads - 1) / threads;
    const size_t cap = (size_t)sm_count() * 16;
    if (b < 1) b = 1;
    return (int)(b > cap ? cap : b);
}

}  // namespace

void launch_input_to_planar(const void* in, int in_is_bf16, void* out, int out_is_bf16, int N, int C, int H, int W,
                            int C_pad, int n0, int n_count, cudaStream_t st) {
    const size_t n = (size_t)used_vecs(n_count, H, W) * (C_pad / 8);
    if (out_is_bf16) input_to_planar_kernel<true><<<grid_for(n, 256), 256, 0, st>>>(in, in_is_bf16, out, N, C, H, W, C_pad / 8, n0, n_count);
    else input_to_planar_kernel<false><<<grid_for(n, 256), 256, 0, st>>>(in, in_is_bf16, out, N, C, H, W, C_pad / 8, n0, n_count);
}

void launch_input_to_stem_planar(const void* in, int in_is_bf16, void* out, int N, int C, int H, int W, int n0, int n_count,
                                 cudaStream_t st) {
    const size_t smem = (size_t)3 * C * (W + 6) * sizeof(float);      // <= 36 KB for the supported widths
    if (C == 3) input_to_stem_planar_rgb_kernel<<<n_count * (H / 2 + 1), 128, smem, st>>>(in, in_is_bf16, (__nv_bfloat16*)out, N, H, W, n0);
    else input_to_stem_planar_kernel<<<n_count * (H / 2 + 1), 256, smem, st>>>(in, in_is_bf16, (__nv_bfloat16*)out, N, C, H, W, n0);
}

void launch_maxpool(const void* x, void* y, int is_bf16, int N, int H, int W, int C_pad, int P, int Q, int R,
                    int stride, int pad, cudaStream_t st) {
    // the chunk planes are contiguous over the batch: (chunk, image) pairs are numbered jn = chunk * N + image
    const int tx = Q + 1 <= 32 ? 32 : Q + 1 <= 64 ? 64 : 128, ty = 256 / tx;
    const int rows = (C_pad / 8) * N * (P + 1);
    const dim3 block(tx, ty), grid((rows + ty - 1) / ty);
    if (is_bf16 && R == 3 && stride == 2 && pad == 1)
        maxpool3s2_bf16_kernel<<<grid, block, 0, st>>>((const Vec8h*)x, (Vec8h*)y, N, H, W, C_pad / 8, P, Q);
    else if (is_bf16) maxpool_kernel<true><<<grid, block, 0, st>>>(x, y, N, H, W, C_pad / 8, P, Q, R, stride, pad);
    else maxpool_kernel<false><<<grid, block, 0, st>>>(x, y, N, H, W, C_pad / 8, P, Q, R, stride, pad);
}

void launch_head(const void* x, int is_bf16, int N, int H, int W, int C_pad, const float* fcw, const float* fcb,
                 int n_classes, float* logits, float* pool_scratch, int max_batch, cudaStream_t st) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.stream = st;
    cfg.blockDim = dim3(256);
    cfg.gridDim = dim3((unsigned)(((size_t)N * (C_pad / 8) * 32 + 255) / 256));
    const int chunks = C_pad / 8;
    cudaLaunchKernelEx(&cfg, is_bf16 ? pool_sum_kernel<true> : pool_sum_kernel<false>, x, N, H, W, chunks, pool_scratch);
    // classes per warp: one while that is what fills the GPU, four once there are blocks enough
    typedef void (*Fc)(const float*, int, int, const float*, const float*, int, float*);
    // A handle made for many images: tiles, and a kernel of the same order of sums for a few images.  By the handle's batch, not the call's: an
    // image's logits are the same bits in every call.
    const bool tiled = max_batch >= 16 && n_classes >= 32;
    // The widest tile of which there are enough: a wide one reads least, but its block works longest, and the last blocks' time is the
    // kernel's.  (Forward of ResNet-50 at 32x32 with 1000 classes, us, tiles of 8 x 8, 8 x 16, 16 x 16, 16 x 32, 32 x 32 images x classes, in brackets
    // the kernel above: 16 images 187.1, 190.3, 188.7, 192.4, 201.3 (187.7); 32 207.0, 204.2, 208.4, 215.2, 230.1 (202.2); 48 221.8, 218.5, 217.8, 224.4,
    // 240.2 (219.1); 64 241.1, 238.3, 233.2, 231.2, 254.5 (235.5); 100 275.7, 270.5, 264.2, 263.5, 280.8 (265.4); 128 316.5, 306.9, 299.6, 293.7, 308.0
    // (296.8); 200 379.1, 361.8, 348.2, 340.7, 346.1 (345.3); 256 425.9, 405.0, 384.7, 378.5, 373.3 (385.2).)
    static const struct { int ipl, cpl; float blocks_per_sm; } kTiles[] = {{4, 8, 1.7f}, {2, 8, 0.85f}, {2, 4, 1.2f}, {1, 4, 1.2f}, {1, 2, 0.0f}};
    int ipl = 0, cpl = 0;
    for (const auto& t : kTiles) {
        ipl = t.ipl; cpl = t.cpl;
        if ((N + 8 * ipl - 1) / (8 * ipl) * (float)((n_classes + 4 * cpl - 1) / (4 * cpl)) >= t.blocks_per_sm * sm_count()) break;
    }
    const bool few = tiled && N <= kFewImages;
    const int images = few ? 1 : tiled ? 8 * ipl : N == 1 ? 1 : N <= 4 ? 4 : 8, groups = (N + images - 1) / images;
    const int cpw = images < 8 ? 1 : groups * ((n_classes + 31) / 32) >= 2 * sm_count() ? 4 : groups * ((n_classes + 15) / 16) >= sm_count() ? 2 : 1;
    const Fc fn = few ? (Fc)fc_few_kernel
                : tiled ? (ipl == 4 ? (Fc)fc_tile_kernel<4, 8> : ipl == 2 ? (cpl == 8 ? (Fc)fc_tile_kernel<2, 8> : (Fc)fc_tile_kernel<2, 4>)
                                  : cpl == 4 ? (Fc)fc_tile_kernel<1, 4> : (Fc)fc_tile_kernel<1, 2>)
                : cpw == 4 ? (Fc)fc_kernel<8, 4, 2> : cpw == 2 ? (Fc)fc_kernel<8, 2, 4> : images == 8 ? (Fc)fc_kernel<8, 1, 8>
                : images == 4 ? (Fc)fc_kernel<4, 1, 8> : (Fc)fc_kernel<1, 1, 16>;
    // (65535 blocks are the most along y; a matrix of more classes goes on along z)
    const int classes = few ? 4 * kFewWarps : tiled ? 4 * cpl : kFcWarps * cpw;      // of a block
    const unsigned class_blocks = (unsigned)((n_classes + classes - 1) / classes), along_y = std::min(class_blocks, 65535u);
    cfg.gridDim = dim3((unsigned)groups, along_y, (class_blocks + along_y - 1) / along_y);
    if (few) cfg.blockDim = dim3(32 * kFewWarps);
    cfg.dynamicSmemBytes = few ? 0 : tiled ? (size_t)fc_tile_smem(ipl, cpl) : (size_t)images * kFcPitch4 * sizeof(float4);
    static std::atomic<bool> raised[64];   // per device, once (threads may all be the first)
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || !raised[dev]) {
        for (Fc f : {(Fc)fc_kernel<8, 1, 8>, (Fc)fc_kernel<8, 2, 4>, (Fc)fc_kernel<8, 4, 2>})
            cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(8 * kFcPitch4 * sizeof(float4)));
        cudaFuncSetAttribute(fc_tile_kernel<4, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, fc_tile_smem(4, 8));
        cudaFuncSetAttribute(fc_tile_kernel<2, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, fc_tile_smem(2, 8));
        cudaFuncSetAttribute(fc_tile_kernel<2, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, fc_tile_smem(2, 4));
        if (dev >= 0 && dev < 64) raised[dev] = true;
    }
    cudaLaunchKernelEx(&cfg, fn, (const float*)pool_scratch, N, C_pad, fcw, fcb, n_classes, logits);
}

void launch_planar_to_nchw_f32(const void* x, int is_bf16, float* out, int N, int H, int W, int C_pad, int C_out,
                               int split, cudaStream_t st) {
    const size_t n = (size_t)N * (C_pad / 8) * H * W;
    if (is_bf16) planar_to_nchw_f32_kernel<true><<<grid_for(n, 256), 256, 0, st>>>(x, out, N, H, W, C_pad / 8, C_out, split);
    else planar_to_nchw_f32_kernel<false><<<grid_for(n, 256), 256, 0, st>>>(x, out, N, H, W, C_pad / 8, C_out, split);
}

}  // namespace fp
