// Convolution layers with few output positions (small batches, small images): one wave of CTAs, the reduction of a tile
// split over the CTAs of a cluster.
//
//   What bounds such a layer.  A layer of ResNet-50 at batch 1 has 1 to 27 tiles of 128 positions: in the persistent form
//   (conv_tc.cu) that many CTAs read the whole filter bank through one shared-memory pipe each and issue all K steps one
//   after the other while the other SMs stand still (2048 -> 308 at 7x7: 6 CTAs, 128 K steps, 17 us; 308 -> 308 3x3: 22 us).
//   Here the chain is cut: `splits` CTAs of a cluster take K groups of the same output tile each, filter tiles
//   are as narrow as it takes to give every SM a part, and the partial sums meet in distributed shared memory.
//   Layout     operands, descriptors and bank order are those of conv_tc.cu's unified stages: a stage holds a K group's
//              activation rows (one bulk copy per channel chunk, or per chunk and parity image) and its filters (one copy).
//   Roles      warp 0 copies, warp 1 allocates tensor memory and issues the MMAs, eight warps finish.  The filters of the
//              first round of stages are asked for before the previous kernel has ended (programmatic dependent launch):
//              mostly those are all the filters a CTA needs.
//   Reduction  chunk q of 8 filters is finished by the cluster's CTA q % splits: every CTA writes its partial sums of the chunk
//              into that CTA's memory ([source][chunk][half][row] float4, lanes 16 bytes apart), one cluster barrier, then
//              the owner adds them in the order of the ranks: the result does not depend on who was first.
//   Waits      bounded as in conv_tc.cu; every thread goes through both cluster barriers whatever happened, so no CTA leaves while
//              another may still write into it.
#include "fp_internal.h"
#include "tc_common.cuh"

#include <algorithm>
#include <cstring>
#include <mutex>

namespace fp {

namespace {

using namespace tc;

constexpr int kStages = 8;
constexpr int kEpi = 8;                                  // finishing warps
constexpr int kThreads = 32 * (2 + kEpi);
constexpr int kMaxNTile = 128;
constexpr int kMaxSplits = 8;

struct SplitCtrl {
    uint64_t full[kStages];
    uint64_t empty[kStages];
    uint64_t done;
    uint32_t tmem_base;
    int abort_flag;
    float bias[kMaxNTile];
};
static_assert(sizeof(SplitCtrl) % 16 == 0, "the reduction buffer behind it holds 16-byte vectors");

struct SplitParams {
    ConvArgs a;
    FastDiv div_ntiles, div_splits, div_p2out, div_qp;
    int Wp_in, Qp, P2_out;
    int plane_in, plane_in2, plane_out, plane_y, par_stride;      // vectors
    int m_total, taps, cchunks, cchunks2, cg, groups, groups2, halo, rows_a, a_par, stages, splits;
    int n_tile, n_tiles, tmem_cols, a_stage_bytes, stage_bytes, red_bytes, slots;   // slots: chunks a CTA finishes at most
    int bank_tile_vecs;
    int tap_off[9];
    int y_P2h, y_Wh2;
    int skip_round;
    long long wait_cycles;
    int* status;
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t remote_addr(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_remote16(uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}

// The taps of one K group: every tap's operand starts at its own row of the stage, its filters follow the previous
// tap's.  Unrolled: an index into the parameters that is not a constant costs the issuing thread some 300 cycles.
template <int TAPS>
__device__ __forceinline__ void issue_taps(int ksteps, uint32_t d, uint32_t a_lo, const int (&tap_off)[9], uint32_t b_lo, uint32_t b_tap,
                                           uint32_t a_ks, uint32_t b_ks, uint32_t idesc, uint32_t accumulate) {
    if (ksteps == 1) {
#pragma unroll
        for (int t = 0; t < TAPS; ++t)
            umma_bf16_lo(d, a_lo + (uint32_t)tap_off[t], b_lo + (uint32_t)t * b_tap, idesc, t ? 1u : accumulate);
        return;
    }
#pragma unroll
    for (int t = 0; t < TAPS; ++t) {
        uint32_t al = a_lo + (uint32_t)tap_off[t], bl = b_lo + (uint32_t)t * b_tap;
#pragma unroll 1
        for (int ks = 0; ks < ksteps; ++ks) {
            umma_bf16_lo(d, al, bl, idesc, (t | ks) ? 1u : accumulate);
            al += a_ks;
            bl += b_ks;
        }
    }
}

__global__ void __launch_bounds__(kThreads) conv_split_kernel(const SplitParams p) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    SplitCtrl* ctrl = reinterpret_cast<SplitCtrl*>(smem_raw);
    const uint32_t base = smem_u32(smem_raw);
    const uint32_t red_base = base + (uint32_t)sizeof(SplitCtrl);
    const uint32_t stage0 = (red_base + (uint32_t)p.red_bytes + 127u) & ~127u;
    const uint32_t full0 = base + (uint32_t)offsetof(SplitCtrl, full), empty0 = base + (uint32_t)offsetof(SplitCtrl, empty);
    const uint32_t done = base + (uint32_t)offsetof(SplitCtrl, done);
    volatile int* abort_flag = &ctrl->abort_flag;
    const long long limit = p.wait_cycles > 0 ? p.wait_cycles : kWaitCycles;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    const int unit = (int)fdiv(blockIdx.x, p.div_splits), rank = (int)blockIdx.x - unit * p.splits;
    const int mt = (int)fdiv((uint32_t)unit, p.div_ntiles), nt = unit - mt * p.n_tiles;
    const int k_base = nt * p.n_tile;
    const int cols = min(p.n_tile, p.a.K_pad - k_base);
    const int f0 = mt * 128;
    // this CTA's K groups: equal shares of the MMAs (a group of the second input has one tap)
    const int work = p.groups * p.taps + p.groups2;
    auto group_at = [&](int w) { const int m = p.groups * p.taps; return w <= m ? (w + p.taps - 1) / p.taps : p.groups + (w - m); };
    const int g_begin = group_at(work * rank / p.splits), g_end = group_at(work * (rank + 1) / p.splits);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
        mbar_init(done, 1);
        ctrl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (threadIdx.x >= 64 && (int)threadIdx.x - 64 < cols) ctrl->bias[threadIdx.x - 64] = p.a.bias[k_base + threadIdx.x - 64];
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(base + (uint32_t)offsetof(SplitCtrl, tmem_base)), "r"((uint32_t)p.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&ctrl->tmem_base);
    if (p.splits > 1) cluster_arrive();                  // this CTA runs: its memory may be written to
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == 0) {
        // ------------------------------ copies ------------------------------
        const uint4* xv = reinterpret_cast<const uint4*>(p.a.x);
        const uint4* x2v = reinterpret_cast<const uint4*>(p.a.x2);
        const uint4* wv = reinterpret_cast<const uint4*>(p.a.w);
        const uint4* w2v = reinterpret_cast<const uint4*>(p.a.w2);
        auto chunks_of = [&](int g) { return g < p.groups ? min(p.cg, p.cchunks - g * p.cg) : min(p.cg, p.cchunks2 - (g - p.groups) * p.cg); };
        auto arm_and_filters = [&](int g, uint32_t stage) {
            const int cgg = chunks_of(g);
            const uint32_t fb = full0 + 8 * stage, dst = stage0 + stage * (uint32_t)p.stage_bytes + (uint32_t)p.a_stage_bytes;
            if (g < p.groups) {
                const uint32_t b_bytes = (uint32_t)(p.taps * cgg * p.n_tile * 16);
                if (lane == 0) {
                    mbar_expect_tx(fb, b_bytes + (uint32_t)(p.a_par * cgg * p.rows_a * 16));
                    bulk_copy(dst, wv + (long long)nt * p.bank_tile_vecs + (long long)p.taps * (g * p.cg) * p.n_tile, b_bytes, fb);
                }
            } else {                                     // centre tap of the second input: its own bank, [chunk][K_pad][8]
                if (lane == 0) mbar_expect_tx(fb, (uint32_t)(cgg * (cols + p.rows_a) * 16));
                __syncwarp();
                if (lane < cgg)
                    bulk_copy(dst + (uint32_t)(lane * p.n_tile * 16), w2v + (long long)((g - p.groups) * p.cg + lane) * p.a.K_pad + k_base,
                              (uint32_t)(cols * 16), fb);
            }
            __syncwarp();
        };
        auto activations = [&](int g, uint32_t stage) {
            const int na = p.a_par * chunks_of(g);
            const uint32_t fb = full0 + 8 * stage, dst = stage0 + stage * (uint32_t)p.stage_bytes;
            if (lane < na) {
                const int c = p.a_par == 1 ? lane : lane >> 2, pp = p.a_par == 1 ? 0 : lane & 3;
                const uint4* src;
                if (g < p.groups) {
                    const int chunk = g * p.cg + c;
                    src = p.a.x2_chunk0 > 0 && chunk >= p.a.x2_chunk0 ? x2v + (long long)(chunk - p.a.x2_chunk0) * p.plane_in2
                                                                      : xv + (long long)chunk * p.plane_in + (long long)pp * p.par_stride;
                } else {
                    src = x2v + (long long)((g - p.groups) * p.cg + c) * p.plane_in2;
                }
                bulk_copy(dst + (uint32_t)(lane * p.rows_a * 16), src + f0 - p.halo, (uint32_t)(p.rows_a * 16), fb);
            }
        };
        const int first = min(p.stages, g_end - g_begin);
        for (int i = 0; i < first; ++i) arm_and_filters(g_begin + i, (uint32_t)i);
        asm volatile("griddepcontrol.wait;" ::: "memory");
        for (int i = 0; i < first; ++i)
            if (i != p.skip_round) activations(g_begin + i, (uint32_t)i);
        uint32_t stage = 0, phase = 0;
        bool ok = true;
        for (int g = g_begin + first; g < g_end; ++g) {
            ok = __all_sync(0xffffffffu, mbar_wait(empty0 + 8 * stage, phase, abort_flag, limit));
            if (!ok) break;
            arm_and_filters(g, stage);
            activations(g, stage);
            if (++stage == (uint32_t)p.stages) { stage = 0; phase ^= 1; }
        }
        if (!ok && lane == 0) { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 1); }
    } else if (warp == 1) {
        // ------------------------------ MMAs ------------------------------
        if (lane == 0) {
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.n_tile >> 3) << 17) | ((128u >> 4) << 24);
            uint32_t stage = 0, phase = 0, accumulate = 0;
            bool ok = true;
            for (int g = g_begin; g < g_end; ++g) {
                if (!mbar_wait(full0 + 8 * stage, phase, abort_flag, limit)) { ok = false; break; }
                tc_fence_after();
                const uint32_t sa = stage0 + stage * (uint32_t)p.stage_bytes;
                const uint32_t pitch = (uint32_t)(p.a_par * p.rows_a);          // rows between chunks
                // (14 address bits: in a cluster a shared address carries the CTA's rank from bit 24 on, which would end up in
                // the descriptor's plane pitch)
                uint32_t a_lo = ((sa >> 4) & 0x3fffu) | (pitch << 16);
                const uint32_t b_lo = (((sa + (uint32_t)p.a_stage_bytes) >> 4) & 0x3fffu) | ((uint32_t)p.n_tile << 16);
                const bool second = g >= p.groups;
                const int cgg = second ? min(p.cg, p.cchunks2 - (g - p.groups) * p.cg) : min(p.cg, p.cchunks - g * p.cg);
                if (p.taps == 9 && !second) {
                    issue_taps<9>(cgg >> 1, tmem, a_lo, p.tap_off, b_lo, (uint32_t)(cgg * p.n_tile), 2u * pitch, 2u * (uint32_t)p.n_tile, idesc, accumulate);
                } else {
                    uint32_t bl = b_lo;
                    if (second) a_lo += (uint32_t)p.halo;
#pragma unroll 1
                    for (int ks = 0; ks < cgg >> 1; ++ks) {
                        umma_bf16_lo(tmem, a_lo, bl, idesc, ks ? 1u : accumulate);
                        a_lo += 2u * pitch;
                        bl += 2u * (uint32_t)p.n_tile;
                    }
                }
                accumulate = 1;
                umma_commit(empty0 + 8 * stage);
                if (++stage == (uint32_t)p.stages) { stage = 0; phase ^= 1; }
            }
            if (ok) umma_commit(done);
            else { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 2); }
        }
        __syncwarp();
    }

    // ------------------------------ finish ------------------------------
    const bool finisher = warp >= 2;
    const int quarter = warp & 3, half = finisher ? (warp - 2) >> 2 : 0, row = quarter * 32 + lane;
    const int f = f0 + row;
    const bool exists = finisher && f < p.m_total;
    const int n = (int)fdiv((uint32_t)f, p.div_p2out);
    const int rem = f - n * p.P2_out;
    const int hp = (int)fdiv((uint32_t)rem, p.div_qp), wq = rem - hp * p.Qp;
    const bool interior = exists && hp >= 1 && hp <= p.a.P && wq >= 1 && wq <= p.a.Q;
    int fy = f;
    if (p.a.y_split) {                                   // see conv_tc.cu: the pixel's place in its parity image
        const int h = hp - 1, w = wq - 1;
        const int pp = (h & 1) ? ((w & 1) ? 2 : 1) : ((w & 1) ? 3 : 0);
        fy = (pp * p.a.N + n) * p.y_P2h + ((h >> 1) + 1) * p.y_Wh2 + ((w >> 1) + 1);
    }
    const uint4* res = reinterpret_cast<const uint4*>(p.a.res) + (long long)(k_base >> 3) * p.plane_out + f;
    uint4* y = reinterpret_cast<uint4*>(p.a.y) + (long long)(k_base >> 3) * p.plane_y + fy;
    const int nch = cols >> 3;
    auto finish = [&](int q, const float (&v)[8], const uint4& r) {
        const float4 ba = *reinterpret_cast<const float4*>(&ctrl->bias[8 * q]), bb = *reinterpret_cast<const float4*>(&ctrl->bias[8 * q + 4]);
        float s[8] = {v[0] + ba.x, v[1] + ba.y, v[2] + ba.z, v[3] + ba.w, v[4] + bb.x, v[5] + bb.y, v[6] + bb.z, v[7] + bb.w};
        if (p.a.res_mode == 1) {
            s[0] += __uint_as_float(r.x << 16); s[1] += __uint_as_float(r.x & 0xffff0000u);
            s[2] += __uint_as_float(r.y << 16); s[3] += __uint_as_float(r.y & 0xffff0000u);
            s[4] += __uint_as_float(r.z << 16); s[5] += __uint_as_float(r.z & 0xffff0000u);
            s[6] += __uint_as_float(r.w << 16); s[7] += __uint_as_float(r.w & 0xffff0000u);
        }
        uint4 o;
        if (p.a.relu) {
            o.x = pack_bf16x2_relu(s[0], s[1]); o.y = pack_bf16x2_relu(s[2], s[3]);
            o.z = pack_bf16x2_relu(s[4], s[5]); o.w = pack_bf16x2_relu(s[6], s[7]);
        } else {
            o.x = pack_bf16x2(s[0], s[1]); o.y = pack_bf16x2(s[2], s[3]);
            o.z = pack_bf16x2(s[4], s[5]); o.w = pack_bf16x2(s[6], s[7]);
        }
        if (!interior) o = make_uint4(0, 0, 0, 0);
        if (exists) y[(long long)q * p.plane_y] = o;
    };
    const bool res1 = interior && p.a.res_mode == 1;
    const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16);
    bool ok = true;
    if (p.splits == 1) {
        if (finisher) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            uint4 rq[8];                                 // the shortcut's vectors, asked for before the sums are there
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int q = 4 * (i >> 1) + 2 * half + (i & 1);
                rq[i] = make_uint4(0, 0, 0, 0);
                if (res1 && q < nch) rq[i] = __ldg(res + (long long)q * p.plane_out);
            }
            ok = __all_sync(0xffffffffu, mbar_wait(done, 0, abort_flag, limit));
            if (ok) {
                tc_fence_after();
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int q = 4 * i + 2 * half;
                    if (q < nch) {
                        uint32_t v[16];
                        tmem_ld16(taddr + 8u * (uint32_t)q, v);
                        tmem_ld_wait();
                        float lo[8], hi[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) { lo[e] = __uint_as_float(v[e]); hi[e] = __uint_as_float(v[8 + e]); }
                        finish(q, lo, rq[2 * i]);
                        finish(q + 1, hi, rq[2 * i + 1]);
                    }
                }
            }
        }
    } else {
        // chunk q goes to CTA q % splits, place q / splits of its buffer
        uint4 rq[4];
        if (finisher) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int q = rank + (2 * i + half) * p.splits;
                rq[i] = make_uint4(0, 0, 0, 0);
                if (res1 && q < nch) rq[i] = __ldg(res + (long long)q * p.plane_out);
            }
            ok = __all_sync(0xffffffffu, mbar_wait(done, 0, abort_flag, limit));
        }
        __syncwarp();
        cluster_wait();                                  // all CTAs of the cluster run
        if (finisher && ok) {
            tc_fence_after();
            int dst = (2 * half) % p.splits, place = (2 * half) / p.splits;
#pragma unroll 1
            for (int q = 2 * half; q < nch; q += 4) {
                uint32_t v[16];
                tmem_ld16(taddr + 8u * (uint32_t)q, v);
                tmem_ld_wait();
                const uint32_t mine = red_base + (uint32_t)(rank * p.slots) * 4096u + (uint32_t)row * 16u;
                uint32_t at = remote_addr(mine + (uint32_t)place * 4096u, (uint32_t)dst);
                st_remote16(at, v[0], v[1], v[2], v[3]);
                st_remote16(at + 2048u, v[4], v[5], v[6], v[7]);
                if (++dst == p.splits) { dst = 0; ++place; }
                at = remote_addr(mine + (uint32_t)place * 4096u, (uint32_t)dst);
                st_remote16(at, v[8], v[9], v[10], v[11]);
                st_remote16(at + 2048u, v[12], v[13], v[14], v[15]);
#pragma unroll
                for (int k = 0; k < 3; ++k)              // to chunk q + 4
                    if (++dst == p.splits) { dst = 0; ++place; }
            }
        }
        __syncwarp();
        cluster_arrive();
        cluster_wait();                                  // all partial sums are here
        if (finisher && ok) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int l = 2 * i + half, q = rank + l * p.splits;
                if (q < nch) {
                    float s[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) s[e] = 0.0f;
                    const uint8_t* from = smem_raw + sizeof(SplitCtrl) + (size_t)l * 4096 + (size_t)row * 16;
#pragma unroll 4
                    for (int c = 0; c < p.splits; ++c) {
                        const float4 u = *reinterpret_cast<const float4*>(from + (size_t)c * p.slots * 4096);
                        const float4 w = *reinterpret_cast<const float4*>(from + (size_t)c * p.slots * 4096 + 2048);
                        s[0] += u.x; s[1] += u.y; s[2] += u.z; s[3] += u.w;
                        s[4] += w.x; s[5] += w.y; s[6] += w.z; s[7] += w.w;
                    }
                    finish(q, s, rq[i]);
                }
            }
        }
    }
    if (!ok && lane == 0) { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 3); }

    if (*abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);         // copies in flight land before the memory is given back
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)p.tmem_cols) : "memory");
    }
}

int round_up_i(int v, int m) { return (v + m - 1) / m * m; }

constexpr unsigned kSmemOne = 232448u - 1024u;
constexpr unsigned kSmemTwo = 233472u / 2 - 1024u;       // two CTAs on an SM

// CTAs that run at once in clusters of a size, with one ([0]) or two ([1]) of them on an SM: a cluster lies within a group of
// SMs, so that not every SM finds a place in one (B200: 148 CTAs alone or in pairs, 132 in fours, 120 in eights).
struct Room { int ctas[2][kMaxSplits + 1]; };
const Room& cluster_room() {
    static Room known[64];
    static bool asked[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); dev = 0; }
    static std::mutex m;
    std::lock_guard<std::mutex> lock(m);
    if (!asked[dev]) {
        for (int two = 0; two < 2; ++two)
            for (int c = 1; c <= kMaxSplits; ++c) {
                cudaLaunchConfig_t cfg;
                memset(&cfg, 0, sizeof(cfg));
                cfg.gridDim = dim3((unsigned)(c * 512));
                cfg.blockDim = dim3((unsigned)kThreads);
                cfg.dynamicSmemBytes = two ? kSmemTwo : kSmemOne;
                cudaLaunchAttribute attr;
                attr.id = cudaLaunchAttributeClusterDimension;
                attr.val.clusterDim.x = (unsigned)c;
                attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
                cfg.attrs = &attr;
                cfg.numAttrs = 1;
                int n = 0;
                if (cudaOccupancyMaxActiveClusters(&n, conv_split_kernel, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
                known[dev].ctas[two][c] = std::min(n * c, (two + 1) * sm_count());
            }
        asked[dev] = true;
    }
    return known[dev];
}

}  // namespace

bool plan_conv_split(const ConvArgs& a, ConvPlanTC* plan) {
    const int sms = sm_count();
    const int taps = a.R * a.S;
    const bool flat = a.stride == 1 && a.P == a.H && a.Q == a.W && ((taps == 1 && a.pad == 0) || (a.R == 3 && a.S == 3 && a.pad == 1));
    if (!flat || a.scatter || a.n_tile_forced > 0 || a.res_mode == 2) return false;
    const long long m_total = (long long)a.N * (a.P + 2) * (a.Q + 2);
    const int m_tiles = (int)std::min<long long>((m_total + 127) / 128, 1 << 20);
    if (m_tiles > sms) return false;
    const int cchunks = a.C_pad / 8, a_par = a.x_s2d ? 4 : 1;
    const int halo = taps == 1 ? 0 : a.W + 3;
    const int rows_a = round_up_i(128 + (a_par > 1 ? 1 : 2) * halo, 8);
    if (cudaFuncSetAttribute(conv_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemOne) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    const Room& room = cluster_room();
    double best = 0;
    bool found = false;
    for (int n_tile = 16; n_tile <= kMaxNTile; n_tile += 16) {
        const int n_tiles = (a.K_pad + n_tile - 1) / n_tile;
        if (n_tile > 16 && (a.K_pad + n_tile - 17) / (n_tile - 16) == n_tiles) continue;       // a narrower tile does the same
        for (int splits = 1; splits <= kMaxSplits; ++splits) {
            const long long units = (long long)m_tiles * n_tiles * splits;
            if (units > 2 * sms) break;
            if (units > room.ctas[1][splits]) continue;
            const int per_sm = units > room.ctas[0][splits] ? 2 : 1;
            const int slots = (n_tile / 8 + splits - 1) / splits;
            const unsigned red = splits > 1 ? (unsigned)(splits * slots) * 4096u : 0u;
            const unsigned fixed = (unsigned)sizeof(SplitCtrl) + red + 128u;
            for (int cg = std::min(cchunks, taps == 9 ? 4 : 16); cg >= 2; cg = cg > 8 ? 8 : cg - 2) {
                const int groups = (cchunks + cg - 1) / cg;
                if (groups < splits) continue;
                const int mine = (groups + splits - 1) / splits;
                const unsigned a_bytes = (unsigned)(a_par * cg * rows_a * 16), b_bytes = (unsigned)(taps * cg * n_tile * 16);
                const unsigned avail = (per_sm == 2 ? kSmemTwo : kSmemOne);
                if (fixed + a_bytes + b_bytes > avail) continue;
                // two CTAs' worth of shared memory is left free where three stages fit the half: the next layer's CTAs then
                // start early and fetch their filters
                int stages = fixed < kSmemTwo ? (int)((kSmemTwo - fixed) / (a_bytes + b_bytes)) : 0;
                if (stages < std::min(mine, 3)) stages = std::min((int)((avail - fixed) / (a_bytes + b_bytes)), std::min(mine, 4));
                stages = std::min(std::min(stages, mine), kStages);
                if (stages < std::min(mine, 2)) continue;
                // cycles (measured: see above): first bytes, bytes at 64 per cycle, MMAs, reduction, finishing
                const double bytes = (double)mine * (a_bytes + 0.7 * b_bytes) * per_sm;
                const double load = 900.0 + bytes / 64.0 + (stages < mine ? 400.0 : 0.0);
                const double mma = 500.0 + (double)mine * (taps * (cg / 2) * std::max(59.0, n_tile / 2.0) + 100.0) * (per_sm == 2 ? 1.5 : 1.0);
                const double red_c = splits > 1 ? 700.0 + n_tile * 512.0 / 48.0 * per_sm : 0.0;
                const double cost = std::max(load, mma) + red_c + 60.0 * slots * per_sm;
                if (!found || cost < best) {
                    found = true;
                    best = cost;
                    plan->split = splits; plan->n_tile = n_tile; plan->n_tiles = n_tiles; plan->cg = cg; plan->groups = groups;
                    plan->a_stages = stages;
                    plan->smem_bytes = fixed + (unsigned)stages * (a_bytes + b_bytes);
                }
            }
        }
    }
    if (!found) return false;
    plan->flat = 1; plan->blocked_bank = 1; plan->halo = halo; plan->rows_a = rows_a; plan->tps = 1;
    plan->tmem_cols = 32;
    while (plan->tmem_cols < plan->n_tile) plan->tmem_cols *= 2;
    plan->ctas_per_sm = 1;
    plan->epi_warps = kEpi;
    plan->valid = 1;
    return true;
}

void launch_conv_split(const ConvPlanTC& plan, const ConvArgs& a, int* d_status, cudaStream_t st, int skip_round, long long wait_cycles) {
    SplitParams p;
    memset(&p, 0, sizeof(p));
    p.a = a;
    const int P2_in = (a.H + 2) * (a.W + 2);
    p.Wp_in = a.W + 2; p.Qp = a.Q + 2; p.P2_out = (a.P + 2) * (a.Q + 2);
    p.plane_in = a.N * P2_in * (a.x_plane_mult > 1 || a.x_s2d ? 4 : 1);
    p.plane_in2 = a.N * P2_in * (a.x2_plane_mult > 1 ? 4 : 1);
    p.par_stride = a.N * P2_in;
    p.m_total = p.plane_out = p.plane_y = a.N * p.P2_out;
    if (a.y_split) {
        p.y_Wh2 = (a.Q + 1) / 2 + 2; p.y_P2h = ((a.P + 1) / 2 + 2) * p.y_Wh2;
        p.plane_y = 4 * a.N * p.y_P2h;
    }
    p.taps = a.R * a.S; p.cchunks = a.C_pad / 8; p.cg = plan.cg; p.groups = plan.groups;
    p.cchunks2 = a.x2_C_pad / 8; p.groups2 = (p.cchunks2 + plan.cg - 1) / plan.cg;
    p.halo = plan.halo; p.rows_a = plan.rows_a; p.a_par = a.x_s2d ? 4 : 1; p.stages = plan.a_stages; p.splits = plan.split;
    p.n_tile = plan.n_tile; p.n_tiles = plan.n_tiles; p.tmem_cols = plan.tmem_cols;
    p.slots = (plan.n_tile / 8 + plan.split - 1) / plan.split;
    p.red_bytes = plan.split > 1 ? plan.split * p.slots * 4096 : 0;
    p.a_stage_bytes = p.a_par * plan.cg * plan.rows_a * 16;
    p.stage_bytes = p.a_stage_bytes + p.taps * plan.cg * plan.n_tile * 16;
    p.bank_tile_vecs = p.taps * p.cchunks * plan.n_tile;
    for (int t = 0; t < 9; ++t) {
        const int r = t / 3, s = t % 3;
        if (a.x_s2d) {                                   // see conv_tc.cu
            const int pa = r == 1 ? 0 : 1, pb = s == 1 ? 0 : 1;
            p.tap_off[t] = (pa ? (pb ? 2 : 1) : (pb ? 3 : 0)) * plan.rows_a + plan.halo + (r == 0 ? -p.Wp_in : 0) + (s == 0 ? -1 : 0);
        } else {
            p.tap_off[t] = r * p.Wp_in + s;
        }
    }
    p.skip_round = skip_round; p.wait_cycles = wait_cycles; p.status = d_status;
    p.div_ntiles = make_fastdiv((uint32_t)plan.n_tiles);
    p.div_splits = make_fastdiv((uint32_t)plan.split);
    p.div_p2out = make_fastdiv((uint32_t)p.P2_out);
    p.div_qp = make_fastdiv((uint32_t)p.Qp);
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(((p.m_total + 127) / 128) * plan.n_tiles * plan.split));
    cfg.blockDim = dim3((unsigned)kThreads);
    cfg.dynamicSmemBytes = plan.smem_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)plan.split;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    void* args[1] = {(void*)&p};
    cudaLaunchKernelExC(&cfg, (const void*)conv_split_kernel, args);
}

}  // namespace fp
