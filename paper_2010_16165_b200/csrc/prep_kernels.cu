// Filter preparation kernels: BN folding (Eq. 3-5 merged into the convolution), identity
// filters of the auxiliary convolutions (Sec. IV-B.1), filter scoring (Eq. 6), ranking and
// masking (Algorithm 1), and repacking of the surviving filters into K,R,S,C order.
#include "fp_internal.h"

namespace fp {

constexpr int kSmallRank = 512;        // filters that one cluster scores and ranks in a single launch,
constexpr int kSmallBank = 1 << 17;    // if the bank has no more weights than this: eight SMs read half a megabyte in about a microsecond
constexpr int kRankCtas = 8;

// omega_k with one rounded fp32 operation per step: t = var + eps; r = sqrt(t); omega = gamma / r.
__device__ __forceinline__ float bn_omega(const float* bn, int K, int k, float eps) {
    const float t = __fadd_rn(bn[3 * K + k], eps);
    const float r = __fsqrt_rn(t);
    return __fdiv_rn(bn[k], r);
}

__global__ void fold_weights_kernel(const float* __restrict__ w, const float* __restrict__ bn, int K, int C, int R,
                                    int S, float eps, float* __restrict__ dst, int C_dst, int R_dst, int S_dst,
                                    int k0, int c0, int r0, int s0) {
    const int per = C * R * S;
    const size_t total = (size_t)K * per;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(i / per);
        int rem = (int)(i - (size_t)k * per);
        const int c = rem / (R * S);
        rem -= c * R * S;
        const int r = rem / S, s = rem - r * S;
        const float omega = bn_omega(bn, K, k, eps);
        dst[(((size_t)(k0 + k) * C_dst + (c0 + c)) * R_dst + (r + r0)) * S_dst + (s + s0)] = __fmul_rn(omega, w[i]);
    }
}

// lambda = beta - omega * mean, the product and the difference rounded separately.
__global__ void fold_bias_kernel(const float* __restrict__ bn, int K, float eps, float* __restrict__ dst, int k0,
                                 int accumulate) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    const float omega = bn_omega(bn, K, k, eps);
    const float m = __fmul_rn(omega, bn[2 * K + k]);
    const float lam = __fsub_rn(bn[K + k], m);
    dst[k0 + k] = accumulate ? __fadd_rn(dst[k0 + k], lam) : lam;
}

__global__ void identity_filters_kernel(float* dst, int C_dst, int R, int S, int k0, int c0, int K_id, int C_id,
                                        int shift) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K_id) return;
    const int c = k - shift;
    if (c < 0 || c >= C_id) return;
    dst[(((size_t)(k0 + k) * C_dst + (c0 + c)) * R + R / 2) * S + S / 2] = 1.0f;
}

__global__ void count_nonfinite_kernel(const float* __restrict__ p, size_t n, int* count) {
    int bad = 0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        bad += !isfinite(p[i]);
    if (bad) atomicAdd(count, bad);
}

// A filter's score by one warp.  Lane l accumulates elements l, l+32, ... in increasing order in fp64 (each |w| or
// w*w is exact in fp64), then the 32 partial sums are combined pairwise with partners at distance 16, 8, 4, 2, 1.  The
// order is part of the definition of the score, so that the resulting double - and therefore the ranking - does not
// depend on the launch shape.  A lane's additions are one chain, but its loads are not: a batch of them is in flight at
// once (with one load per addition a filter of 4608 weights waited for 144 memory latencies one after the other).
constexpr int kScoreBatch = 8;
template <bool UPDATE>
__device__ __forceinline__ double score_filter(float* __restrict__ f, const float* __restrict__ d, int per, int norm, int lane) {
    double s = 0.0;
    float v[kScoreBatch], u[kScoreBatch];
    auto load = [&](int t0) {
#pragma unroll
        for (int i = 0; i < kScoreBatch; ++i) v[i] = t0 + 32 * i < per ? f[t0 + 32 * i] : 0.0f;
        if (UPDATE) {
#pragma unroll
            for (int i = 0; i < kScoreBatch; ++i) u[i] = t0 + 32 * i < per ? __ldg(d + t0 + 32 * i) : 0.0f;
        }
    };
    load(lane);
    for (int t0 = lane; t0 - lane < per; t0 += 32 * kScoreBatch) {
        float x[kScoreBatch];
#pragma unroll
        for (int i = 0; i < kScoreBatch; ++i) x[i] = UPDATE ? __fadd_rn(v[i], u[i]) : v[i];
        load(t0 + 32 * kScoreBatch);                 // on their way while these are added up
        if (UPDATE) {
#pragma unroll
            for (int i = 0; i < kScoreBatch; ++i)
                if (t0 + 32 * i < per) f[t0 + 32 * i] = x[i];
        }
#pragma unroll
        for (int i = 0; i < kScoreBatch; ++i) {      // behind the filter's end: + 0.0, which changes no bit of a sum of non-negative terms
            const double y = (double)x[i];
            s = __dadd_rn(s, norm ? __dmul_rn(y, y) : fabs(y));
        }
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) s = __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
    return s;
}

__global__ void score_filters_kernel(const float* __restrict__ w, int K, int per, int norm, double* __restrict__ scores) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= K) return;
    const double s = score_filter<false>(const_cast<float*>(w) + (size_t)warp * per, nullptr, per, norm, lane);
    if (lane == 0) scores[warp] = s;
}

// How many of a bank's K scores come before filter k's in ascending (score, index) order, counted by a whole warp.  (One
// block per bank, every thread counting for its own filters, took 60-130 us for a bank of 2048 filters: K * K / 256
// comparisons one after the other on one SM.)
__device__ __forceinline__ int rank_of(const double* __restrict__ scores, int K, int k, int lane) {
    const double sk = scores[k];
    int before = 0;
#pragma unroll 4
    for (int j = lane; j < K; j += 32) {
        const double sj = scores[j];
        before += (sj < sk) || (sj == sk && j < k);
    }
    return __reduce_add_sync(0xffffffffu, before);
}

// rank[k] = number of filters ordered before k in ascending (score, index) order; the first q are masked.
__global__ void rank_mask_kernel(const double* scores, int K, int q, int32_t* __restrict__ rank, uint8_t* __restrict__ mask) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (k >= K) return;
    const int before = rank_of(scores, K, k, lane);
    if (lane == 0) { rank[k] = before; mask[k] = before >= q ? 1 : 0; }
}

// Score, rank and mask of a small bank in one launch: a cluster of eight CTAs, every warp scores filters and puts each
// score into all eight CTAs' shared memory; behind the cluster's barrier every CTA ranks an eighth of the filters, several
// threads per filter.  No second launch and no scratch in global memory.
__global__ void __cluster_dims__(kRankCtas, 1, 1) __launch_bounds__(256)
score_rank_cluster_kernel(const float* __restrict__ w, int K, int per, int norm, int q, int32_t* __restrict__ rank,
                          uint8_t* __restrict__ mask) {
    __shared__ double sh[kSmallRank];
    const int warp = (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
    // nobody writes into another CTA's shared memory before that CTA runs
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    for (int k = (int)blockIdx.x * 8 + warp; k < K; k += 8 * kRankCtas) {
        const double s = score_filter<false>(const_cast<float*>(w) + (size_t)k * per, nullptr, per, norm, lane);
        if (lane < kRankCtas) {
            uint32_t dst;
            const uint32_t own = (uint32_t)__cvta_generic_to_shared(sh + k);
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(own), "r"(lane));
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(dst), "d"(s) : "memory");
        }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    const int mine = (K + kRankCtas - 1) / kRankCtas;          // <= 64 filters of this CTA
    int share = 1;                                             // threads of one warp per filter, a power of two
    while (share < 32 && 2 * share * mine <= 256) share *= 2;
    const int i = threadIdx.x / share, k = (int)blockIdx.x * mine + i, part = threadIdx.x & (share - 1);
    const bool live = i < mine && k < K;
    int before = 0;
    if (live) {
        const double sk = sh[k];
        for (int j = part; j < K; j += share) before += (sh[j] < sk) || (sh[j] == sk && j < k);
    }
    for (int o = share >> 1; o >= 1; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    if (live && part == 0) { rank[k] = before; mask[k] = before >= q ? 1 : 0; }
}

// The same for all filter banks of a model at once, one warp per filter: (update and) score ...
template <bool UPDATE>
__global__ void bank_score_kernel(const SoftBank* __restrict__ banks, const int32_t* __restrict__ filter_bank, int total_filters,
                                  const float* __restrict__ dw, int norm, double* __restrict__ scores) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (g >= total_filters) return;
    const SoftBank& b = banks[filter_bank[g]];
    const size_t first = (size_t)(g - b.k_off) * b.per;
    const double s = score_filter<UPDATE>(b.w + first, UPDATE ? dw + b.dw_off + first : nullptr, b.per, norm, lane);
    if (lane == 0) scores[g] = s;
}

// ... then rank, mask and, where asked, zeroize the masked filter in place.  A warp ranks kRankGroup filters of a bank with one
// pass over the bank's scores: with one filter per warp the 26,560 warps of ResNet-50 read 200 MB of scores through L1
// (18 us; now 12).
constexpr int kRankGroup = 4;
__global__ void bank_rank_kernel(const SoftBank* __restrict__ banks, const int32_t* __restrict__ filter_bank, int total_filters,
                                 const double* scores, int zeroize, int32_t* __restrict__ rank, uint8_t* __restrict__ mask) {
    const int g0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kRankGroup;
    const int lane = threadIdx.x & 31;
    if (g0 >= total_filters) return;
    const int n = min(kRankGroup, total_filters - g0);
    for (int at = 0; at < n;) {                      // a bank's end may lie inside the group
        const SoftBank& b = banks[filter_bank[g0 + at]];
        const int K = b.K, k = g0 + at - b.k_off, m = min(n - at, K - k);
        const double* sc = scores + b.k_off;
        if (at == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
        double sk[kRankGroup];
        int before[kRankGroup];
#pragma unroll
        for (int i = 0; i < kRankGroup; ++i) { sk[i] = sc[min(k + i, K - 1)]; before[i] = 0; }
        // blocks of 32 scores before the group (an equal score comes first), around it, and behind it (an equal one comes later)
        const int low = k & ~31, high = min(K, (k + kRankGroup + 31) & ~31);
#pragma unroll 8
        for (int j = lane; j < low; j += 32) {
            const double sj = sc[j];
#pragma unroll
            for (int i = 0; i < kRankGroup; ++i) before[i] += sj <= sk[i];
        }
        for (int j = low + lane; j < high; j += 32) {
            const double sj = sc[j];
#pragma unroll
            for (int i = 0; i < kRankGroup; ++i) before[i] += (sj < sk[i]) || (sj == sk[i] && j < k + i);
        }
#pragma unroll 8
        for (int j = high + lane; j < K; j += 32) {
            const double sj = sc[j];
#pragma unroll
            for (int i = 0; i < kRankGroup; ++i) before[i] += sj < sk[i];
        }
#pragma unroll
        for (int i = 0; i < kRankGroup; ++i) {
            if (i >= m) break;
            const int r = __reduce_add_sync(0xffffffffu, before[i]);
            if (lane == 0) { rank[g0 + at + i] = r; mask[g0 + at + i] = r >= b.q ? 1 : 0; }
            if (zeroize && r < b.q) {
                float* f = b.w + (size_t)(k + i) * b.per;
                if (b.per % 4 == 0)
                    for (int t = lane; t < b.per / 4; t += 32) reinterpret_cast<float4*>(f)[t] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                else
                    for (int t = lane; t < b.per; t += 32) f[t] = 0.0f;
            }
        }
        at += m;
    }
}

// ---- everything a (re)planned graph reads besides activations, packed by ONE launch: a table of jobs, and for every block
// the job it works for.  (One launch, one allocation and one upload per array made fp_prune of ResNet-50 take 25-45 ms.)
__device__ __forceinline__ uint4 pack8(const float (&v)[8]) {
    uint4 o;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    return o;
}

__device__ __forceinline__ void store8(const PackJob& j, size_t vec, const float (&v)[8]) {
    if (j.f32) {
        float4* o = reinterpret_cast<float4*>(j.out) + 2 * vec;
        o[0] = make_float4(v[0], v[1], v[2], v[3]);
        o[1] = make_float4(v[4], v[5], v[6], v[7]);
    } else {
        reinterpret_cast<uint4*>(j.out)[vec] = pack8(v);
    }
}

// The filters of a convolution: a block = 32 filter rows x a run of units, a unit being a few chunks of 8 input channels with at
// most nine taps together; the next unit's weights are on their way while this one is written.  Where the
// vector of (row k, chunk c, tap) goes is the kernels' affair:
//   PACK_CONV   [filter tile][K group][tap][chunk in group][row in tile]: with one tile and one group the plain layout
//               [tap][chunk][row], otherwise a block per pipeline stage / a contiguous part per filter tile (conv_tc.cu).
//               Chunks >= chunks1 are the second bank's (a projection shortcut stacked along the channels).
//   PACK_QUAD   a fused run's layer of 16 filters, 2 x 2 outputs a row: [window pixel][chunk][output][filter], zeros where the pixel is
//               outside the output's window
//   PACK_CHAIN  a fused run's layer: per tap row and chunk a stack of 3 * K_pad rows, row 48 * (k / 16) + 16 * s + k % 16
//               for horizontal tap s (chain_tc.cu)
// The weights are laid [filter][channel][tap], the banks have the filters innermost: a transposition, through shared memory.
// A warp reads one filter's (kept) channels side by side, then neighbouring threads write neighbouring filters' vectors; the
// row pitch of 73 words keeps both free of bank conflicts.  (A thread per vector, reading its weights from global memory
// itself, had every lane of a load in another line: ResNet-50 pruned at 0.4 inside its blocks, 77 MB read: 74 us, now 48.)
constexpr int kPackPitch = kPackElems + 1;
template <int kRS>                                   // taps, 0: j.RS of them
__device__ __forceinline__ void pack_filters(const PackJob& j, const int32_t* __restrict__ idx, int blk, float* sh) {
    const int lane = threadIdx.x & 31, warp = (int)threadIdx.x >> 5;
    const int RS = kRS ? kRS : j.RS, span = pack_span(RS), pieces = kRS ? 1 : (RS + kPackTaps - 1) / kPackTaps;
    const int units = (j.chunks + span - 1) / span * pieces, run = pack_run(units), runs = (units + run - 1) / run;
    const int kb = blk / runs, k0 = kb * 32, u0 = (blk - kb * runs) * run, u1 = min(units, u0 + run);
    const int chunks1 = j.chunks1, chunks = j.chunks;
    const size_t pitch = (size_t)j.C * RS;
    // the rows this warp reads
    const float* __restrict__ wk[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int k = k0 + warp + 8 * i, ks = k < j.K_pad ? idx[j.row + k] : -1;
        wk[i] = ks >= 0 ? j.w + ks * pitch : nullptr;
    }
    // the row this lane writes
    const int k = k0 + lane;
    const bool chain = j.kind == PACK_CHAIN;
    const int tile = chain ? 0 : k / j.n_tile, tile_rows = chain ? 3 * j.K_pad : j.n_tile, cg = j.cg;
    const size_t row = chain ? 48 * (k >> 4) + (k & 15) : (size_t)tile * RS * chunks * j.n_tile + (k - tile * j.n_tile);

    struct Unit { int c0, n_chunks, r0, T; };
    auto unit = [&](int u) {
        Unit x;
        const int g = u / pieces;
        x.c0 = g * span; x.n_chunks = min(span, chunks - x.c0);
        x.r0 = (u - g * pieces) * kPackTaps; x.T = kRS ? min(kRS, kPackTaps) : min(kPackTaps, RS - x.r0);
        return x;
    };
    // this lane's places in a row it reads: the weight's place in its filter, -1 where no channel is packed
    int off[3], v_second;
    float v[4][3];
    auto places = [&](const Unit& x) {
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const int e = lane + 32 * s, ch = e / x.T;
            off[s] = -1;
            if (e < x.n_chunks * 8 * x.T) {
                const int cs = idx[(x.c0 + ch / 8 >= chunks1 ? j.chan2 - 8 * chunks1 : j.chan) + x.c0 * 8 + ch];
                if (cs >= 0) off[s] = cs * RS + x.r0 + (e - ch * x.T);
            }
        }
    };
    auto load = [&](const Unit& x) {
        v_second = 0;
        if (x.c0 + x.n_chunks > chunks1) {            // a second bank's channels among them
#pragma unroll
            for (int s = 0; s < 3; ++s) v_second |= (x.c0 + (lane + 32 * s) / x.T / 8 >= chunks1) << s;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int s = 0; s < 3; ++s) v[i][s] = wk[i] && off[s] >= 0 && !(v_second >> s & 1) ? __ldg(wk[i] + off[s]) : 0.0f;
        if (x.c0 + x.n_chunks > chunks1) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int kk = k0 + warp + 8 * i, ks = kk < j.K_pad ? idx[j.row2 + kk] : -1;
#pragma unroll
                for (int s = 0; s < 3; ++s)
                    if ((v_second >> s & 1) && ks >= 0 && off[s] >= 0) v[i][s] = __ldg(j.w2 + (size_t)ks * j.C2 * RS + off[s]);
            }
        }
    };
    Unit x = unit(u0);
    places(x);
    load(x);
    for (int u = u0; u < u1; ++u) {
        const Unit next = unit(u + 1 < u1 ? u + 1 : u);
        places(next);
        if (u > u0) __syncthreads();
        const int elems = x.n_chunks * 8 * x.T;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int s = 0; s < 3; ++s)
                if (lane + 32 * s < elems) sh[(warp + 8 * i) * kPackPitch + lane + 32 * s] = v[i][s];
        __syncthreads();
        if (u + 1 < u1) load(next);                   // in flight while this unit is written
        for (int y = warp; k < j.rows && y < x.n_chunks * x.T; y += kPackThreads / 32) {
            const int cc = y / x.T, t = y - cc * x.T, c = x.c0 + cc, rs = x.r0 + t;
            float o[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) o[e] = sh[lane * kPackPitch + (cc * 8 + e) * x.T + t];
            int place;                                // of the row's vector, in tiles' rows
            if (chain) {
                place = (rs / 3) * chunks * tile_rows + c * tile_rows + 16 * (rs % 3);
            } else {
                const int g = c / cg, cgg = min(cg, chunks - g * cg);
                place = (g * RS * cg + rs * cgg + (c - g * cg)) * tile_rows;
            }
            store8(j, row + place, o);
        }
        x = next;
    }
}

// A 7x7 first convolution in the order the packed network input wants it (see input_to_stem_planar_kernel): a 3x1
// convolution over 80 packed channels.  Tap dr (0..2 = offsets -1,0,+1), chunk 0-2 (group E) take filter row
// r = 2*dr + 1, chunks 3-5 (O') take r = 2*dr at dr = 0, 1, chunks 6-8 (O) take r = 2*dr + 2 at dr = 1, 2; packed channel
// j = s*C + c within a group; everything else zero.  (Input row 2p+1 is held twice, as O of packed row p and as O' of row
// p+1; it is taken from row p, because below the last image row there is only the zero border.)
__device__ __forceinline__ void pack_stem_vec(const PackJob& j, const int32_t* __restrict__ idx, int u) {
    // [filter tile][K group][tap row][chunk in group][row in tile], as a convolution's bank
    const int tile = u / (30 * j.n_tile), at = u / j.n_tile - 30 * tile, k = tile * j.n_tile + u % j.n_tile;
    const int g = at / (3 * j.cg), in_group = at - 3 * j.cg * g, cgg = min(j.cg, 10 - g * j.cg), dr = in_group / cgg, chunk = g * j.cg + in_group % cgg;
    const int ks = k < j.K_pad ? idx[j.row + k] : -1;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        v[e] = 0.0f;
        if (ks < 0 || chunk >= 9) continue;
        const int group = chunk / 3, q = (chunk % 3) * 8 + e;
        const int sx = q / j.C, c = q - sx * j.C;
        int r = -1;
        if (group == 0) r = 2 * dr + 1;
        else if (group == 1) { if (dr < 2) r = 2 * dr; }
        else if (dr >= 1) r = 2 * dr + 2;
        if (r >= 0 && sx < 7) v[e] = j.w[(((size_t)ks * j.C + c) * 7 + r) * 7 + sx];
    }
    store8(j, u, v);
}

// A 7x7 first convolution for the kernel that fuses it with the pooling: the 7x7 / stride-2 window over C channels as a
// 4x4 window over the 4 C parity channels of the half-resolution input - tap (ta, tb), channel (2a + b) C + c takes
// w[k][c][2 ta + a - 1][2 tb + b - 1] (zero where an index is -1) - as [tap][chunk of 8][filter][8].  Channels 4 C .. 4 C + 2,
// which the kernel feeds with ones, hold the filter's shift at tap 0, as three bf16 that add up to the fp32 value.
__device__ __forceinline__ void pack_stem_direct_vec(const PackJob& j, const int32_t* __restrict__ idx, int u) {
    const int k = u % j.K_pad, chunk = u / j.K_pad % 2, tap = u / (2 * j.K_pad);
    const int ta = tap >> 2, tb = tap & 3;
    const int ks = idx[j.row + k];
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const int ch = chunk * 8 + e;
        v[e] = 0.0f;
        if (ks >= 0 && tap == 0 && ch >= 4 * j.C && ch < 4 * j.C + 3) {
            float b = j.w2[ks];
            for (int i = 4 * j.C; i < ch; ++i) b -= __bfloat162float(__float2bfloat16(b));
            v[e] = b;
        }
        if (ks < 0 || ch >= 4 * j.C) continue;
        const int par = ch / j.C, c = ch - par * j.C;
        const int r = 2 * ta + (par >> 1) - 1, s = 2 * tb + (par & 1) - 1;
        if (r >= 0 && s >= 0) v[e] = j.w[(((size_t)ks * j.C + c) * 7 + r) * 7 + s];
    }
    store8(j, u, v);
}

__global__ void __launch_bounds__(kPackThreads) pack_kernel(const PackJob* __restrict__ jobs, const int32_t* __restrict__ block_job,
                                                            const int32_t* __restrict__ idx) {
    __shared__ float sh[32 * kPackPitch];
    const PackJob& j = jobs[block_job[blockIdx.x]];
    const int blk = (int)blockIdx.x - j.first_block;
    if (j.kind == PACK_CONV || j.kind == PACK_CHAIN) {
        if (j.RS == 9) pack_filters<9>(j, idx, blk, sh);
        else if (j.RS == 1) pack_filters<1>(j, idx, blk, sh);
        else pack_filters<0>(j, idx, blk, sh);
        return;
    }
    const int u = blk * kPackThreads + threadIdx.x;
    if (u >= j.units) return;
    switch (j.kind) {
        case PACK_STEM: pack_stem_vec(j, idx, u); break;
        case PACK_STEM_DIRECT: pack_stem_direct_vec(j, idx, u); break;
        case PACK_QUAD: {
            const int k = u & 15, o = u >> 4 & 3, c8 = u >> 6 & 1, w = u >> 7, r = (w >> 2) - (o >> 1), s = (w & 3) - (o & 1), f = idx[j.row + k];
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int c = idx[j.chan + c8 * 8 + e];
                v[e] = f >= 0 && c >= 0 && r >= 0 && r < 3 && s >= 0 && s < 3 ? j.w[((size_t)f * j.C + c) * 9 + r * 3 + s] : 0.0f;
            }
            store8(j, u, v);
            break;
        }
        case PACK_FC: {              // out[k][cp] = w[k][chan[cp]] * scale, fp32
            const int chunks = j.chunks, k = u / chunks, c = u - k * chunks;
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int cs = idx[j.chan + c * 8 + e];
                v[e] = cs >= 0 ? j.w[(size_t)k * j.C + cs] * j.scale : 0.0f;
            }
            store8(j, u, v);
            break;
        }
        default: {                   // PACK_BIAS: the kept filters' shifts, a taken-in projection's added
            const int r1 = idx[j.row + u];
            float b = r1 >= 0 ? j.w[r1] : 0.0f;
            if (j.w2) { const int r2 = idx[j.row2 + u]; b += r2 >= 0 ? j.w2[r2] : 0.0f; }
            reinterpret_cast<float*>(j.out)[u] = b;
        }
    }
}

static inline int blocks_for(size_t n, int threads) {
    const int cap = fp::sm_count() * 8;
    size_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    return (int)(b > (size_t)cap ? cap : b);
}

void launch_fold_weights(const float* w, const float* bn, int K, int C, int R, int S, float eps, float* dst,
                         int C_dst, int R_dst, int S_dst, int k0, int c0, int r0, int s0, cudaStream_t st) {
    const size_t n = (size_t)K * C * R * S;
    fold_weights_kernel<<<blocks_for(n, 256), 256, 0, st>>>(w, bn, K, C, R, S, eps, dst, C_dst, R_dst, S_dst, k0, c0, r0, s0);
}

void launch_fold_bias(const float* bn, int K, float eps, float* dst_b, int k0, int accumulate, cudaStream_t st) {
    fold_bias_kernel<<<(K + 127) / 128, 128, 0, st>>>(bn, K, eps, dst_b, k0, accumulate);
}

void launch_identity_filters(float* dst, int C_dst, int R, int S, int k0, int c0, int K_id, int C_id, int shift,
                             cudaStream_t st) {
    identity_filters_kernel<<<(K_id + 127) / 128, 128, 0, st>>>(dst, C_dst, R, S, k0, c0, K_id, C_id, shift);
}

void launch_count_nonfinite(const float* p, size_t n, int* d_count, cudaStream_t st) {
    if (n == 0) return;
    count_nonfinite_kernel<<<blocks_for(n, 256), 256, 0, st>>>(p, n, d_count);
}

void launch_score_filters(const float* w, int K, int per_filter, int norm, double* scores, cudaStream_t st) {
    score_filters_kernel<<<(K + 7) / 8, 256, 0, st>>>(w, K, per_filter, norm, scores);
}

// `blocks` blocks of 256 threads that may start while the launch before them still runs (they wait for it themselves).
template <typename... Params, typename... Args>
static void launch_behind(void (*kernel)(Params...), int blocks, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
}

void launch_score_rank(const float* w, int K, int per_filter, int norm, int q, double* scores, int32_t* rank, uint8_t* mask,
                       cudaStream_t st) {
    if (K <= kSmallRank && (long long)K * per_filter <= kSmallBank) {
        score_rank_cluster_kernel<<<kRankCtas, 256, 0, st>>>(w, K, per_filter, norm, q, rank, mask);
        return;
    }
    launch_score_filters(w, K, per_filter, norm, scores, st);
    launch_behind(rank_mask_kernel, (K + 7) / 8, st, (const double*)scores, K, q, rank, mask);
}

void launch_bank_score(const SoftBank* banks, const int32_t* filter_bank, int total_filters, const float* dw, int norm,
                       double* scores, cudaStream_t st) {
    const int blocks = (total_filters + 7) / 8;
    if (dw) bank_score_kernel<true><<<blocks, 256, 0, st>>>(banks, filter_bank, total_filters, dw, norm, scores);
    else bank_score_kernel<false><<<blocks, 256, 0, st>>>(banks, filter_bank, total_filters, nullptr, norm, scores);
}
void launch_bank_rank(const SoftBank* banks, const int32_t* filter_bank, int total_filters, const double* scores, int zeroize,
                      int32_t* rank, uint8_t* mask, cudaStream_t st) {
    launch_behind(bank_rank_kernel, (total_filters + 8 * kRankGroup - 1) / (8 * kRankGroup), st, banks, filter_bank, total_filters, scores,
                  zeroize, rank, mask);
}

void launch_pack(const PackJob* jobs, const int32_t* block_job, int n_blocks, const int32_t* idx, cudaStream_t st) {
    if (n_blocks > 0) pack_kernel<<<n_blocks, kPackThreads, 0, st>>>(jobs, block_job, idx);
}

}  // namespace fp
