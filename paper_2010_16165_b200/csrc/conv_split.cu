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
//   Roles      warp 0 copies, warp 1 allocates tensor memory and issues the MMAs, eight warps ask for the first activations and finish.  The filters of the
//              first round of stages are asked for before the previous kernel has ended (programmatic dependent launch):
//              mostly those are all the filters a CTA needs.
//   Reduction  chunk q of 8 filters is finished by the cluster's CTA q % splits: every CTA sends its partial sums of the chunk
//              into that CTA's memory ([source][chunk][half][row] float4, lanes 16 bytes apart) with st.async, counted in
//              bytes on a barrier there, and the owner adds them in the order of the ranks: the result does not depend on
//              who was first.  (A layer of one image is 5000 cycles; plain remote stores behind a releasing cluster barrier
//              took 1500-2400 of them, staging in shared memory and one bulk copy per destination 1000-2500.)
//   Latency    Everything that does not depend on the sums - places, addresses in other CTAs, shortcut vectors - is worked out
//              while the activations are on the way.  A K group costs the issuing warp some 400 cycles whatever its MMAs (a
//              barrier test 125, a commit 190), so groups are long, and a stage is committed only where it is
//              filled again.
//   Waits      bounded as in conv_tc.cu; every thread goes through both cluster barriers whatever happened, so no CTA leaves while
//              another may still send to it.
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
    uint64_t sums;                                       // the cluster's partial sums of this CTA's chunks are here
    uint32_t tmem_base;
    int abort_flag;
    int pad_[2];
    float bias[kMaxNTile];
};
static_assert(sizeof(SplitCtrl) % 16 == 0, "the reduction buffer behind it holds 16-byte vectors");

struct SplitParams {
    ConvArgs a;
    FastDiv div_ntiles, div_splits, div_p2out, div_qp;
    int Wp_in, Qp, P2_out;
    int plane_in, plane_in2, plane_out, plane_y, par_stride;      // vectors
    int m_total, taps, cchunks, cchunks2, cg, groups, groups2, halo, rows_a, a_par, stages, splits, tps;
    int n_tile, n_tiles, tmem_cols, a_stage_bytes, stage_bytes, red_bytes, slots;   // slots: chunks a CTA finishes at most
    int bank_tile_vecs;
    int tap_off[9];
    int y_P2h, y_Wh2;
    int skip_round;
    long long wait_cycles;
    int* status;
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t remote_addr(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// counted in bytes on a barrier of the CTA it goes to
__device__ __forceinline__ void st_async16(uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(addr), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar) : "memory");
}
__device__ __forceinline__ void sts16(uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
__device__ __forceinline__ void lds16(uint32_t addr, float (&v)[4]) {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(addr) : "memory");
}
// A load that stays behind griddepcontrol.wait (__ldg may be moved in front of it: the previous kernel's tensor is not
// read-only data until that kernel has ended).
__device__ __forceinline__ uint4 ld_global16(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint2 ld_global8(const uint2* p) {
    uint2 v;
    asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}

// (At least two CTAs on an SM: the next layer's start while this layer's work.  The code is kept short - an instance per kind
// of layer (EDGES: a parity-split output of an odd height or width), loops instead of unrolled bodies - because a launch meets it cold: the same kernel with everything unrolled,
// 106 instead of 64 registers, took 3.9 us instead of 3.0 for a 48 -> 256 layer of one image.)
template <int TAPS, bool SPLIT, bool EDGES>
__global__ void __launch_bounds__(kThreads, 3) conv_split_kernel(const SplitParams p) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    SplitCtrl* ctrl = reinterpret_cast<SplitCtrl*>(smem_raw);
    const uint32_t base = smem_u32(smem_raw);
    const uint32_t red_base = base + (uint32_t)sizeof(SplitCtrl);
    const uint32_t stage0 = (red_base + (uint32_t)p.red_bytes + 127u) & ~127u;
    const uint32_t full0 = base + (uint32_t)offsetof(SplitCtrl, full), empty0 = base + (uint32_t)offsetof(SplitCtrl, empty);
    const uint32_t done = base + (uint32_t)offsetof(SplitCtrl, done), sums = base + (uint32_t)offsetof(SplitCtrl, sums);
    volatile int* abort_flag = &ctrl->abort_flag;
    const long long limit = p.wait_cycles > 0 ? p.wait_cycles : kWaitCycles;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    const int unit = (int)fdiv(blockIdx.x, p.div_splits), rank = (int)blockIdx.x - unit * p.splits;
    const int mt = (int)fdiv((uint32_t)unit, p.div_ntiles), nt = unit - mt * p.n_tiles;
    const int k_base = nt * p.n_tile;
    const int cols = min(p.n_tile, p.a.K_pad - k_base);
    const int f0 = mt * p.tps * 128;
    const int nch = cols >> 3;
    // this CTA's K groups: equal shares of the MMAs (a group of the second input has one tap)
    const int work = p.groups * TAPS + p.groups2;
    auto group_at = [&](int w) { const int m = p.groups * TAPS; return w <= m ? (w + TAPS - 1) / TAPS : p.groups + (w - m); };
    const int g_begin = group_at(work * rank / p.splits), g_end = group_at(work * (rank + 1) / p.splits);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
        mbar_init(done, 1);
        mbar_init(sums, 1);
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
    if (SPLIT) {
        if (threadIdx.x == 64 && rank < nch)
            mbar_expect_tx(sums, (uint32_t)(p.tps * ((nch - rank + p.splits - 1) / p.splits) * (p.splits - 1)) * 4096u);
        __syncwarp();
        cluster_arrive();                                // this CTA runs: its memory may be written to
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const uint4* xv = reinterpret_cast<const uint4*>(p.a.x);
    const uint4* x2v = reinterpret_cast<const uint4*>(p.a.x2);
    auto chunks_of = [&](int g) { return g < p.groups ? min(p.cg, p.cchunks - g * p.cg) : min(p.cg, p.cchunks2 - (g - p.groups) * p.cg); };
    auto run_of = [&](int g, int i) -> const uint4* {    // activation run i of K group g: a channel chunk, or a parity image of one
        const int c = p.a_par == 1 ? i : i >> 2, pp = p.a_par == 1 ? 0 : i & 3;
        if (g >= p.groups) return x2v + (long long)((g - p.groups) * p.cg + c) * p.plane_in2 + f0 - p.halo;
        const int chunk = g * p.cg + c;
        if (p.a.x2_chunk0 > 0 && chunk >= p.a.x2_chunk0) return x2v + (long long)(chunk - p.a.x2_chunk0) * p.plane_in2 + f0 - p.halo;
        return xv + (long long)chunk * p.plane_in + (long long)pp * p.par_stride + f0 - p.halo;
    };
    const int first = min(p.stages, g_end - g_begin);
    if (warp == 0) {
        // ------------------------------ copies: filters, and activations behind the first round of stages ------------------------------
        const uint4* wv = reinterpret_cast<const uint4*>(p.a.w);
        const uint4* w2v = reinterpret_cast<const uint4*>(p.a.w2);
        auto arm_and_filters = [&](int g, uint32_t stage) {
            const int cgg = chunks_of(g);
            const uint32_t fb = full0 + 8 * stage, dst = stage0 + stage * (uint32_t)p.stage_bytes + (uint32_t)p.a_stage_bytes;
            if (g < p.groups) {
                const uint32_t b_bytes = (uint32_t)(TAPS * cgg * p.n_tile * 16);
                if (lane == 0) {
                    mbar_expect_tx(fb, b_bytes + (uint32_t)(p.a_par * cgg * p.rows_a * 16));
                    bulk_copy(dst, wv + (long long)nt * p.bank_tile_vecs + (long long)TAPS * (g * p.cg) * p.n_tile, b_bytes, fb);
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
        for (int i = 0; i < first; ++i) arm_and_filters(g_begin + i, (uint32_t)i);
        asm volatile("griddepcontrol.wait;" ::: "memory");
        uint32_t stage = 0, phase = 0;
        bool ok = true;
        for (int g = g_begin + first; g < g_end; ++g) {
            ok = __all_sync(0xffffffffu, mbar_wait(empty0 + 8 * stage, phase, abort_flag, limit));
            if (!ok) break;
            arm_and_filters(g, stage);
            if (lane < p.a_par * chunks_of(g))
                bulk_copy(stage0 + stage * (uint32_t)p.stage_bytes + (uint32_t)(lane * p.rows_a * 16), run_of(g, lane), (uint32_t)(p.rows_a * 16), full0 + 8 * stage);
            __syncwarp();
            if (++stage == (uint32_t)p.stages) { stage = 0; phase ^= 1; }
        }
        if (!ok && lane == 0) { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 1); }
    } else if (warp == 1) {
        // ------------------------------ MMAs ------------------------------
        const uint32_t leader = elect_one();
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.n_tile >> 3) << 17) | ((128u >> 4) << 24);
        uint32_t stage = 0, phase = 0, accumulate = 0;
        bool ok = true;
        uint32_t off[TAPS];                              // rows from a stage's start to each tap's operand
#pragma unroll
        for (int tap = 0; tap < TAPS; ++tap) off[tap] = TAPS == 1 ? 0u : (uint32_t)p.tap_off[tap];
        const uint32_t pitch = (uint32_t)(p.a_par * p.rows_a);              // rows between chunks
        const uint32_t a_ks = 2u * pitch, b_ks = 2u * (uint32_t)p.n_tile;
        // (14 address bits: in a cluster a shared address carries the CTA's rank from bit 24 on, which would end up in the
        // descriptor's plane pitch)
        const uint32_t stage_rows = (uint32_t)p.stage_bytes >> 4, a_first = ((stage0 >> 4) & 0x3fffu) | (pitch << 16);
        const uint32_t b_first = (((stage0 + (uint32_t)p.a_stage_bytes) >> 4) & 0x3fffu) | ((uint32_t)p.n_tile << 16);
        uint32_t row0 = 0;                               // of the stage
        for (int g = g_begin; g < g_end; ++g) {
            if (!__all_sync(0xffffffffu, mbar_wait(full0 + 8 * stage, phase, abort_flag, limit))) { ok = false; break; }
            const uint32_t empty = empty0 + 8 * stage;
            const bool second = g >= p.groups;
            const int cgg = chunks_of(g);
            const uint32_t b_tap = (uint32_t)(cgg * p.n_tile);
            uint32_t a_lo = a_first + row0 + (second ? (uint32_t)p.halo : 0u);
            const uint32_t b_lo = b_first + row0;
            row0 += stage_rows;
            if (++stage == (uint32_t)p.stages) { stage = 0; phase ^= 1; row0 = 0; }
            for (int t = 0; t < p.tps; ++t) {
                const uint32_t d = tmem + (uint32_t)(t * p.n_tile);
                uint32_t al = a_lo, bl = b_lo;
#pragma unroll 1
                for (int ks = 0; ks < cgg >> 1; ++ks) {
                    if (TAPS == 9 && !second) {
                        // every tap's operand starts at its own row of the stage, its filters follow the previous tap's
#pragma unroll
                        for (int tap = 0; tap < TAPS; ++tap)
                            umma_bf16_lo_if(leader, d, al + off[tap], bl + (uint32_t)tap * b_tap, idesc, (tap | ks) ? 1u : accumulate);
                    } else {
                        umma_bf16_lo_if(leader, d, al, bl, idesc, ks ? 1u : accumulate);
                    }
                    al += a_ks;
                    bl += b_ks;
                }
                a_lo += 128u;
            }
            accumulate = 1;
            if (leader && g + p.stages < g_end) umma_commit(empty);          // (190 cycles: only where the stage is filled again)
            __syncwarp();
        }
        if (leader) {
            if (ok) umma_commit(done);
            else { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 2); }
        }
        __syncwarp();
    }

    // ------------------------------ finish ------------------------------
    const bool finisher = warp >= 2;
    const int quarter = warp & 3, half = finisher ? (warp - 2) >> 2 : 0, row = quarter * 32 + lane;
    struct Place { bool exists, interior; const uint4* res; uint4* y; };
    auto place_of = [&](int t) {                         // this thread's position in position tile t of the CTA
        Place o;
        const int f = f0 + t * 128 + row;
        const int n = (int)fdiv((uint32_t)f, p.div_p2out);
        const int rem = f - n * p.P2_out;
        const int hp = (int)fdiv((uint32_t)rem, p.div_qp), wq = rem - hp * p.Qp;
        o.exists = f < p.m_total;
        o.interior = o.exists && hp >= 1 && hp <= p.a.P && wq >= 1 && wq <= p.a.Q;
        int fy = f;
        if (p.a.y_split) {                               // see conv_tc.cu: the pixel's place in its parity image
            const int h = hp - 1, w = wq - 1;
            const int pp = (h & 1) ? ((w & 1) ? 2 : 1) : ((w & 1) ? 3 : 0);
            fy = (pp * p.a.N + n) * p.y_P2h + ((h >> 1) + 1) * p.y_Wh2 + ((w >> 1) + 1);
        }
        o.res = reinterpret_cast<const uint4*>(p.a.res) + (long long)(k_base >> 3) * p.plane_out + f;
        o.y = reinterpret_cast<uint4*>(p.a.y) + (long long)(k_base >> 3) * p.plane_y + fy;
        return o;
    };
    auto shortcut = [&](const Place& o, int q) {
        return p.a.res_mode == 1 && o.interior && q < nch ? ld_global16(o.res + (long long)q * p.plane_out) : make_uint4(0, 0, 0, 0);
    };
    auto finish = [&](const Place& o, int q, const float (&v)[8], const uint4& r) {
        const float4 ba = *reinterpret_cast<const float4*>(&ctrl->bias[8 * q]), bb = *reinterpret_cast<const float4*>(&ctrl->bias[8 * q + 4]);
        float s[8] = {v[0] + ba.x, v[1] + ba.y, v[2] + ba.z, v[3] + ba.w, v[4] + bb.x, v[5] + bb.y, v[6] + bb.z, v[7] + bb.w};
        if (p.a.res_mode == 1) {
            s[0] += __uint_as_float(r.x << 16); s[1] += __uint_as_float(r.x & 0xffff0000u);
            s[2] += __uint_as_float(r.y << 16); s[3] += __uint_as_float(r.y & 0xffff0000u);
            s[4] += __uint_as_float(r.z << 16); s[5] += __uint_as_float(r.z & 0xffff0000u);
            s[6] += __uint_as_float(r.w << 16); s[7] += __uint_as_float(r.w & 0xffff0000u);
        }
        uint4 out;
        if (p.a.relu) {
            out.x = pack_bf16x2_relu(s[0], s[1]); out.y = pack_bf16x2_relu(s[2], s[3]);
            out.z = pack_bf16x2_relu(s[4], s[5]); out.w = pack_bf16x2_relu(s[6], s[7]);
        } else {
            out.x = pack_bf16x2(s[0], s[1]); out.y = pack_bf16x2(s[2], s[3]);
            out.z = pack_bf16x2(s[4], s[5]); out.w = pack_bf16x2(s[6], s[7]);
        }
        if (!o.interior) out = make_uint4(0, 0, 0, 0);
        if (o.exists) o.y[(long long)q * p.plane_y] = out;
    };
    const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16);
    bool ok = true;
    Place o = place_of(0);
    if (finisher) {
        // The activations of the first round of stages are asked for by the finishing warps, which have nothing else to do yet: a
        // warp's copies are issued one after the other, some 60 cycles each (one warp needed 2700 cycles for 32 of them).
        const int runs = p.a_par * p.cg, ci = warp - 2 + kEpi * lane, i = ci / runs, sub = ci - i * runs, g = g_begin + i;
        const bool mine = i < first && sub < p.a_par * chunks_of(g) && i != p.skip_round;
        const uint4* src = mine ? run_of(g, sub) : nullptr;
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (mine) bulk_copy(stage0 + (uint32_t)(i * p.stage_bytes + sub * p.rows_a * 16), src, (uint32_t)(p.rows_a * 16), full0 + 8 * (uint32_t)i);
        __syncwarp();
    }
    if (!SPLIT) {
        // chunks half, half + 2, ... are this warp's, two at a time
        if (finisher) {
            uint4 r0 = shortcut(o, half), r1 = shortcut(o, half + 2);          // the shortcut's vectors, asked for before the sums are there
            ok = __all_sync(0xffffffffu, mbar_wait(done, 0, abort_flag, limit));
            if (ok) {
                tc_fence_after();
                int t = 0, q = half;
#pragma unroll 1
                while (t < p.tps) {
                    uint32_t v[2][8];
                    tmem_ld8(taddr + (uint32_t)(t * p.n_tile + 8 * q), v[0]);
                    tmem_ld8(taddr + (uint32_t)(t * p.n_tile + 8 * min(q + 2, nch - 1)), v[1]);
                    const Place now = o;
                    const int q0 = q;
                    const uint4 c0 = r0, c1 = r1;
                    q += 4;
                    if (q >= nch) {
                        q = half;
                        if (++t < p.tps) o = place_of(t);
                    }
                    if (t < p.tps) { r0 = shortcut(o, q); r1 = shortcut(o, q + 2); }
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        float s[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) s[e] = __uint_as_float(v[j][e]);
                        if (q0 + 2 * j < nch) finish(now, q0 + 2 * j, s, j ? c1 : c0);
                    }
                }
            }
        }
    } else {
        // Chunk q of position tile t goes to CTA q % splits, place t * slots + q / splits of its buffer; of the chunks it owns a
        // thread finishes channels 4 * half .. + 3, so that all eight warps have the same to do.
        const uint32_t per_source = (uint32_t)(p.tps * p.slots) * 4096u;
        auto shortcut4 = [&](const Place& o, int q) {
            return p.a.res_mode == 1 && o.interior && q < nch ? ld_global8(reinterpret_cast<const uint2*>(o.res + (long long)q * p.plane_out) + half) : make_uint2(0, 0);
        };
        uint2 r = make_uint2(0, 0);
        if (finisher) r = shortcut4(o, rank);
        const uint32_t mine = red_base + (uint32_t)rank * per_source + (uint32_t)row * 16u;
        __syncwarp();
        cluster_wait();                                  // all CTAs of the cluster run
        if (finisher) {
            ok = __all_sync(0xffffffffu, mbar_wait(done, 0, abort_flag, limit));
            if (ok) {
                tc_fence_after();
#pragma unroll 1
                for (int t = 0; t < p.tps; ++t) {
                    int dst = half, place = t * p.slots;                        // splits >= 2: chunk `half` is CTA `half`'s
#pragma unroll 1
                    for (int q = half; q < nch; q += 2) {
                        uint32_t v[8];
                        tmem_ld8(taddr + (uint32_t)(t * p.n_tile + 8 * q), v);
                        uint32_t to = mine + (uint32_t)place * 4096u;
                        if (dst == rank) {               // this CTA's own
                            tmem_ld_wait();
                            sts16(to, v[0], v[1], v[2], v[3]);
                            sts16(to + 2048u, v[4], v[5], v[6], v[7]);
                        } else {
                            const uint32_t bar = remote_addr(sums, (uint32_t)dst);
                            to = remote_addr(to, (uint32_t)dst);
                            tmem_ld_wait();
                            st_async16(to, v[0], v[1], v[2], v[3], bar);
                            st_async16(to + 2048u, v[4], v[5], v[6], v[7], bar);
                        }
                        dst += 2;
                        if (dst >= p.splits) { dst -= p.splits; ++place; }
                    }
                }
            }
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kEpi) : "memory");
            if (ok && rank < nch) ok = __all_sync(0xffffffffu, mbar_wait(sums, 0, abort_flag, limit));
        }
        __syncwarp();
        cluster_arrive();                                // what was sent here has arrived (waited for at the end)
        if (finisher && ok && rank < nch) {
            int t = 0, l = 0, q = rank;
#pragma unroll 1
            while (t < p.tps) {
                uint32_t from = red_base + (uint32_t)(t * p.slots + l) * 4096u + (uint32_t)(half * 2048 + row * 16);
                const float4 b = *reinterpret_cast<const float4*>(&ctrl->bias[8 * q + 4 * half]);
                const Place now = o;
                const int q0 = q;
                const uint2 rc = r;
                ++l;
                q += p.splits;
                if (q >= nch) {
                    q = rank; l = 0;
                    if (++t < p.tps) o = place_of(t);
                }
                if (t < p.tps) r = shortcut4(o, q);
                float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
                for (int c = 0; c < p.splits; c += 4) {  // four loads in flight
                    float u[4][4];
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (c + i < p.splits) lds16(from + (uint32_t)i * per_source, u[i]);
                    from += 4u * per_source;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (c + i < p.splits)
#pragma unroll
                            for (int e = 0; e < 4; ++e) s[e] += u[i][e];
                }
                s[0] += b.x; s[1] += b.y; s[2] += b.z; s[3] += b.w;
                if (p.a.res_mode == 1) {
                    s[0] += __uint_as_float(rc.x << 16); s[1] += __uint_as_float(rc.x & 0xffff0000u);
                    s[2] += __uint_as_float(rc.y << 16); s[3] += __uint_as_float(rc.y & 0xffff0000u);
                }
                uint2 out = p.a.relu ? make_uint2(pack_bf16x2_relu(s[0], s[1]), pack_bf16x2_relu(s[2], s[3]))
                                     : make_uint2(pack_bf16x2(s[0], s[1]), pack_bf16x2(s[2], s[3]));
                if (!now.interior) out = make_uint2(0, 0);
                if (now.exists) reinterpret_cast<uint2*>(now.y + (long long)q0 * p.plane_y)[half] = out;
            }
        }
    }
    if (EDGES && finisher && half == 0 && rank == 0)
        for (int t = 0; t < p.tps; ++t) {                // see conv_tc.cu: the row and column behind an odd image's last
            const int f = f0 + t * 128 + row, n = (int)fdiv((uint32_t)f, p.div_p2out), rem = f - n * p.P2_out;
            const int hp = (int)fdiv((uint32_t)rem, p.div_qp), wq = rem - hp * p.Qp;
            auto zeros = [&](int h, int w) {
                const int pp = (h & 1) ? ((w & 1) ? 2 : 1) : ((w & 1) ? 3 : 0);
                uint4* y = reinterpret_cast<uint4*>(p.a.y) + (long long)(k_base >> 3) * p.plane_y + (pp * p.a.N + n) * p.y_P2h + ((h >> 1) + 1) * p.y_Wh2 + ((w >> 1) + 1);
                for (int q = 0; q < nch; ++q) y[(long long)q * p.plane_y] = make_uint4(0, 0, 0, 0);
            };
            const bool below = f < p.m_total && (p.a.P & 1) && hp == p.a.P, right = f < p.m_total && (p.a.Q & 1) && wq == p.a.Q;
            if (below) zeros(hp, wq - 1);
            if (right) zeros(hp - 1, wq);
            if (below && right) zeros(hp, wq);
        }
    if (!ok && lane == 0) { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 3); }

    if (*abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);         // copies in flight land before the memory is given back
    __syncwarp();
    if (SPLIT) cluster_wait();                           // no CTA leaves while another may still send to it
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

typedef void (*SplitKernel)(const SplitParams);
SplitKernel kernel_of(int taps, int splits, bool edges) {
    if (edges)
        return taps == 9 ? (splits > 1 ? conv_split_kernel<9, true, true> : conv_split_kernel<9, false, true>)
                         : (splits > 1 ? conv_split_kernel<1, true, true> : conv_split_kernel<1, false, true>);
    return taps == 9 ? (splits > 1 ? conv_split_kernel<9, true, false> : conv_split_kernel<9, false, false>)
                     : (splits > 1 ? conv_split_kernel<1, true, false> : conv_split_kernel<1, false, false>);
}

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
                if (cudaOccupancyMaxActiveClusters(&n, conv_split_kernel<9, true, false>, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
                known[dev].ctas[two][c] = std::min(n * c, (two + 1) * sm_count());
            }
        asked[dev] = true;
    }
    return known[dev];
}

}  // namespace

namespace {

// One way of giving the layer to the CTAs: position tiles per CTA, filters per tile, CTAs that share a tile's reduction, channel chunks
// per K group.  False where it does not fit; else the launch figures and the time expected.
bool candidate(const ConvArgs& a, const Room& room, int tps, int n_tile, int splits, int cg, ConvPlanTC* c, double* cost) {
    const int taps = a.R * a.S, cchunks = a.C_pad / 8, a_par = a.x_s2d ? 4 : 1;
    const int halo = taps == 1 ? 0 : round_up_i(row_vecs(a.W) + 1, 2);      // (copies begin at a 32-byte sector)
    const int rows_a = round_up_i(128 * tps + (a_par > 1 ? 1 : 2) * halo, 8);
    if (rows_a + 8 > kGuardVectors || tps * n_tile > 256) return false;
    const int m_tiles = (int)((used_vecs(a.N, a.P, a.Q) + 127) / 128), steps = (m_tiles + tps - 1) / tps;
    const int n_tiles = (a.K_pad + n_tile - 1) / n_tile, groups = (cchunks + cg - 1) / cg;
    const int units = steps * n_tiles * splits;
    if (groups < splits || units > room.ctas[1][splits]) return false;
    const int per_sm = units > room.ctas[0][splits] ? 2 : 1;
    const int slots = (n_tile / 8 + splits - 1) / splits;
    const unsigned red = splits > 1 ? (unsigned)(tps * splits * slots) * 4096u : 0u, fixed = (unsigned)sizeof(SplitCtrl) + red + 128u;
    const int mine = (groups + splits - 1) / splits;
    const unsigned a_bytes = (unsigned)(a_par * cg * rows_a * 16), b_bytes = (unsigned)(taps * cg * n_tile * 16);
    const unsigned avail = per_sm == 2 ? kSmemTwo : kSmemOne;
    if (fixed + a_bytes + b_bytes > avail) return false;
    // two CTAs' worth of shared memory is left free where three stages fit the half: the next layer's CTAs then
    // start early and fetch their filters
    int stages = fixed < kSmemTwo ? (int)((kSmemTwo - fixed) / (a_bytes + b_bytes)) : 0;
    if (stages < std::min(mine, 3)) stages = std::min((int)((avail - fixed) / (a_bytes + b_bytes)), std::min(mine, 4));
    stages = std::min(std::min(stages, mine), kStages);
    if (stages < std::min(mine, 2)) return false;
    c->split = splits; c->tps = tps; c->n_tile = n_tile; c->n_tiles = n_tiles; c->cg = cg; c->groups = groups;
    c->halo = halo; c->rows_a = rows_a; c->a_stages = stages;
    c->smem_bytes = fixed + (unsigned)stages * (a_bytes + b_bytes);
    // Microseconds, fitted to some 600 ways of running 17 layers (ResNet-34 and -50 at batches 1 to 17; 8 % rms, the layers' chosen ways
    // 3 % slower than their best): a launch in a chain and its fixed latencies; every K group; every group that waits
    // for a stage to fall free; the MMAs, max(n / 2, 32 + n / 4) cycles each; the bytes of all CTAs; the exchange; finishing,
    // a chunk of 8 filters of 128 positions after the other.
    const double mmas = (double)std::min(mine * cg, cchunks) / 2 * taps * tps, pipe = std::max(n_tile / 2.0, 32.0 + n_tile / 4.0);
    *cost = 2.30 + 0.114 * mine + 0.25 * std::max(0, mine - stages) + 0.00052 * mmas * pipe * per_sm +
            0.025e-6 * (double)units * mine * (a_bytes + b_bytes) + (splits > 1 ? 0.66 + 0.0205 * tps * n_tile * (splits - 1) / splits : 0.0) +
            0.117 * tps * slots * per_sm;
    return true;
}

}  // namespace

bool plan_conv_split(const ConvArgs& a, ConvPlanTC* plan) {
    const int taps = a.R * a.S;
    const bool flat = a.stride == 1 && a.P == a.H && a.Q == a.W && ((taps == 1 && a.pad == 0) || (a.R == 3 && a.S == 3 && a.pad == 1));
    if (!flat || a.scatter || a.n_tile_forced > 0 || a.res_mode == 2) return false;
    if ((used_vecs(a.N, a.P, a.Q) + 127) / 128 > 2 * sm_count()) return false;
    for (int k = 0; k < 8; ++k)
        if (cudaFuncSetAttribute(kernel_of(k & 1 ? 9 : 1, 1 + (k >> 1 & 1), k >> 2), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemOne) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
    const Room& room = cluster_room();
    double best = 0;
    bool found = false;
    ConvPlanTC c = *plan, chosen = *plan;
    for (int tps = 1; tps <= 2; ++tps)
        for (int n_tile = 16; n_tile <= kMaxNTile; n_tile += 16) {
            if (n_tile > 16 && (a.K_pad + n_tile - 17) / (n_tile - 16) == (a.K_pad + n_tile - 1) / n_tile) continue;    // a narrower tile does the same
            for (int splits = 1; splits <= kMaxSplits; ++splits)
                for (int cg = std::min(a.C_pad / 8, taps == 1 ? 16 : a.x_s2d ? 4 : 8); cg >= 2; cg = cg > 8 ? 8 : cg - 2) {
                    double cost = 0;
                    if (candidate(a, room, tps, n_tile, splits, cg, &c, &cost) && (!found || cost < best)) { found = true; best = cost; chosen = c; }
                }
        }
    if (!found) return false;
    // Two position tiles per CTA: there the persistent form does better where it keeps its filters in shared memory and the
    // layer is bound by its MMAs or its output (48 -> 48 3x3 at 56x56, batch 10: 5.5 us against 6.8; 48 -> 256 at batch 5: 5.2
    // against 5.7), not by its input (512 -> 80 at 28x28, batch 22: 11.8 against 7.5), and on strided layers (256 -> 192,
    // batch 64: 17.2 against 18.5).
    const long long per_filter = (long long)taps * a.C_pad * 2;
    const bool resident = per_filter * a.K_pad <= 100 * 1024 || per_filter * std::min(a.K_pad, 128) <= 48 * 1024;
    if (chosen.tps > 1 && (a.x_s2d || (resident && !(taps == 1 && a.K_pad <= 96)))) return false;
    *plan = chosen;
    plan->flat = 1; plan->blocked_bank = 1;
    plan->tmem_cols = 32;
    while (plan->tmem_cols < plan->tps * plan->n_tile) plan->tmem_cols *= 2;
    plan->ctas_per_sm = 1;
    plan->epi_warps = kEpi;
    plan->valid = 1;
    return true;
}

void launch_conv_split(const ConvPlanTC& plan, const ConvArgs& a, int* d_status, cudaStream_t st, int skip_round, long long wait_cycles) {
    SplitParams p;
    memset(&p, 0, sizeof(p));
    p.a = a;
    p.Wp_in = row_vecs(a.W); p.Qp = row_vecs(a.Q); p.P2_out = image_vecs(a.P, a.Q);
    p.plane_in = (int)plane_vecs(a.x_plane_mult > 1 || a.x_s2d ? 4 * a.N : a.N, a.H, a.W);
    p.plane_in2 = (int)plane_vecs(a.x2_plane_mult > 1 ? 4 * a.N : a.N, a.H, a.W);
    p.par_stride = a.N * image_vecs(a.H, a.W);
    p.plane_out = p.plane_y = (int)plane_vecs(a.N, a.P, a.Q);
    p.m_total = (int)used_vecs(a.N, a.P, a.Q);
    if (a.y_split) {
        p.y_Wh2 = row_vecs((a.Q + 1) / 2); p.y_P2h = image_vecs((a.P + 1) / 2, (a.Q + 1) / 2);
        p.plane_y = (int)plane_vecs(4 * a.N, (a.P + 1) / 2, (a.Q + 1) / 2);
        p.m_total = a.N * p.P2_out;                      // (nobody reads behind the last image of a split tensor)
    }
    p.taps = a.R * a.S; p.cchunks = a.C_pad / 8; p.cg = plan.cg; p.groups = plan.groups;
    p.cchunks2 = a.x2_C_pad / 8; p.groups2 = (p.cchunks2 + plan.cg - 1) / plan.cg;
    p.halo = plan.halo; p.rows_a = plan.rows_a; p.a_par = a.x_s2d ? 4 : 1; p.stages = plan.a_stages; p.splits = plan.split; p.tps = plan.tps;
    p.n_tile = plan.n_tile; p.n_tiles = plan.n_tiles; p.tmem_cols = plan.tmem_cols;
    p.slots = (plan.n_tile / 8 + plan.split - 1) / plan.split;
    p.red_bytes = plan.split > 1 ? plan.tps * plan.split * p.slots * 4096 : 0;
    p.a_stage_bytes = p.a_par * plan.cg * plan.rows_a * 16;
    p.stage_bytes = p.a_stage_bytes + p.taps * plan.cg * plan.n_tile * 16;
    p.bank_tile_vecs = p.taps * p.cchunks * plan.n_tile;
    for (int t = 0; t < 9; ++t) {
        const int r = t / 3, s = t % 3;
        if (a.x_s2d) {                                   // see conv_tc.cu
            const int pa = r == 1 ? 0 : 1, pb = s == 1 ? 0 : 1;
            p.tap_off[t] = (pa ? (pb ? 2 : 1) : (pb ? 3 : 0)) * plan.rows_a + plan.halo + (r == 0 ? -p.Wp_in : 0) + (s == 0 ? -1 : 0);
        } else {
            p.tap_off[t] = plan.halo - (p.Wp_in + 1) + r * p.Wp_in + s;
        }
    }
    p.skip_round = skip_round; p.wait_cycles = wait_cycles; p.status = d_status;
    p.div_ntiles = make_fastdiv((uint32_t)plan.n_tiles);
    p.div_splits = make_fastdiv((uint32_t)plan.split);
    p.div_p2out = make_fastdiv((uint32_t)p.P2_out);
    p.div_qp = make_fastdiv((uint32_t)p.Qp);
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)((p.m_total + 128 * plan.tps - 1) / (128 * plan.tps) * plan.n_tiles * plan.split));
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
    cudaLaunchKernelExC(&cfg, (const void*)kernel_of(p.taps, plan.split, a.y_split && (a.P % 2 || a.Q % 2)), args);
}

}  // namespace fp
