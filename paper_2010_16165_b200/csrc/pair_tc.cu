// Two 1x1 convolutions of a bottleneck network in one kernel: the layer that widens a block's tensor, adds the shortcut and writes
// the residual stream, and the narrow layer of the next block that reads the stream.
//
//   y = relu(W1 . x + b1 + shortcut),   z = relu(W2 . y + b2)            (position by position)
//
//   What bounds the two.  The stream is the widest tensor of the network - 220 MB at 56x56 and batch 128 - and the two layers do
//   little arithmetic on it (48 -> 256 -> 48 channels): as kernels of their own they write it and read it again at the copy rate.
//   Here a tile of y stays in shared memory, where it is the second convolution's operand as it lies.
//   CTA tile      128 consecutive flat positions, all channels; one persistent CTA per SM.
//   Groups        y is made 64 channels at a time.  A slot of a ring in shared memory holds a group's shortcut (bulk copies, one run
//                 of 2 KB per 8 channels) and then, in its place, y: the thread that adds a vector of 8 channels writes the sum where it
//                 read it.  From there the second convolution's MMAs and the bulk copies to memory both take it; the slot is free
//                 when both have read it.
//   Filters       a group's rows of W1 and its columns of W2 have rings of their own, since either is in use for a short part of a slot's
//                 time; where both banks fit they are brought once and stay.  Coming with every tile again they come from L2.
//   Tensor memory the second convolution's sums (K2 columns, over all groups of a tile; two tiles' where they fit) and four stages of
//                 64 columns of the first's.
//   Latency       A group's way - slot filled, MMAs, commit, accumulator read, sum written, MMAs, copies out - is some 3000 cycles
//                 of barriers and round trips for a few hundred of work.  So no role waits for another's group before it starts
//                 its next: each convolution has its issuing warp, and two teams of eight finishing warps take the groups in turn.
//                 A warp's bulk copies go out one after the other, some 110 cycles each, so several warps share them (one warp for
//                 a group's dozen took 1100-1500 cycles a group, and that was the kernel's time).
//                 z of a tile is finished behind the first groups of the next, so that nobody waits for its last MMAs.
//   Turns         the numbers of slots and stages are multiples of the number of teams, so a slot, a stage and the barriers of both always
//                 meet the same team: a warp that skips the others' uses of a barrier could take the parity of an older phase for its own.
//   Warp roles    warps 0 and 1 bring x and shortcuts, 2 and 3 the filters of the two convolutions, sixteen warps finish both, one
//                 warp each issues the MMAs of the first and of the second, two copy y out.
//   Sums          in the order of the two kernels this stands for (conv_tc.cu), so the results are theirs bit by bit.
//   Waits         bounded as in conv_tc.cu.
#include "fp_internal.h"
#include "tc_common.cuh"

#include <cstring>

namespace fp {

namespace {

using namespace tc;

constexpr int G = kPairGroup, GC = G / 8;      // channels and chunks of a group
constexpr int kMaxSlots = 8, kSums = 4, kMaxFilters = 8;
constexpr int kRunWarps = 2, kInWarps = kRunWarps + 2, kTeams = 2, kTeamWarps = 8, kOutWarps = 2;
constexpr int kEpi0 = kInWarps, kFirst = kEpi0 + kTeams * kTeamWarps, kSecond = kFirst + 1, kOut0 = kSecond + 1;      // warps
constexpr int kThreads = 32 * (kOut0 + kOutWarps);
constexpr unsigned kSmemMax = 232448u - 1024u;

struct PairCtrl {
    uint64_t slot_full[kMaxSlots], slot_empty[kMaxSlots], y_ready[kMaxSlots];
    uint64_t sum1_full[kSums], sum1_empty[kSums];
    uint64_t w_full[2][kMaxFilters], w_empty[2][kMaxFilters];
    uint64_t x_full[2], x_empty[2];
    uint64_t sum2_full[2], sum2_empty[2];      // by the parity of the tile's number, which is its team and, with two stages, its stage
    uint32_t tmem_base;
    int abort_flag;
    int pad_[2];
};
static_assert(sizeof(PairCtrl) % 16 == 0, "the tables of shifts behind it are read as 16-byte vectors");

struct PairParams {
    PairArgs a;
    FastDiv div_p2out, div_qp;
    int Qp, P2, m_total, m_tiles, m_first, m_sign;
    long long plane_x, plane_x2, plane_res, plane_y;      // vectors per chunk plane
    int chunks1, chunks, groups;               // channel chunks of x, of y; groups of y
    int x_stages, sum2_stages, slots, w_stages, w_stays, tmem_cols;      // w_stays: all groups' filters have a stage of their own
    int y_P2h, y_Wh2;                          // parity-split output: half-resolution grid
    long long wait_cycles;
    int* status;
};

__device__ __forceinline__ void bulk_store(void* dst, uint32_t src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_store_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// A place in a ring of barriers: its index and the parity of its current use.
struct Ring {
    uint32_t at = 0, phase = 0;
    __device__ __forceinline__ void next(int n) { if (++at == (uint32_t)n) { at = 0; phase ^= 1; } }
};

__global__ void __launch_bounds__(kThreads, 1) conv_pair_kernel(const PairParams p) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    PairCtrl* ctrl = reinterpret_cast<PairCtrl*>(smem_raw);
    const uint32_t base = smem_u32(smem_raw);
    float* bias1 = reinterpret_cast<float*>(smem_raw + sizeof(PairCtrl));
    float* bias2 = bias1 + p.a.K;
    const uint32_t x0 = (base + (uint32_t)sizeof(PairCtrl) + (uint32_t)(p.a.K + p.a.K2) * 4u + 127u) & ~127u;
    const uint32_t x_bytes = (uint32_t)p.chunks1 * 2048u;
    const uint32_t slot0 = x0 + (uint32_t)p.x_stages * x_bytes;
    constexpr uint32_t slot_bytes = GC * 2048u;
    const uint32_t w1_bytes = (uint32_t)(p.chunks1 * G) * 16u, w2_bytes = (uint32_t)(GC * p.a.K2) * 16u;
    const uint32_t w1_at = slot0 + (uint32_t)p.slots * slot_bytes, w2_at = w1_at + (uint32_t)p.w_stages * w1_bytes;
    const uint32_t slot_full0 = base + (uint32_t)offsetof(PairCtrl, slot_full), slot_empty0 = base + (uint32_t)offsetof(PairCtrl, slot_empty);
    const uint32_t y_ready0 = base + (uint32_t)offsetof(PairCtrl, y_ready);
    const uint32_t x_full0 = base + (uint32_t)offsetof(PairCtrl, x_full), x_empty0 = base + (uint32_t)offsetof(PairCtrl, x_empty);
    const uint32_t sum1_full0 = base + (uint32_t)offsetof(PairCtrl, sum1_full), sum1_empty0 = base + (uint32_t)offsetof(PairCtrl, sum1_empty);
    const uint32_t w_full0 = base + (uint32_t)offsetof(PairCtrl, w_full), w_empty0 = base + (uint32_t)offsetof(PairCtrl, w_empty);
    const uint32_t sum2_full0 = base + (uint32_t)offsetof(PairCtrl, sum2_full), sum2_empty0 = base + (uint32_t)offsetof(PairCtrl, sum2_empty);
    volatile int* abort_flag = &ctrl->abort_flag;
    const long long limit = p.wait_cycles > 0 ? p.wait_cycles : kWaitCycles;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxSlots; ++s) {
            mbar_init(slot_full0 + 8 * s, kRunWarps);
            mbar_init(slot_empty0 + 8 * s, 1 + kOutWarps);          // the second convolution's MMAs, the copies to memory
            mbar_init(y_ready0 + 8 * s, 32 * kTeamWarps);
        }
        for (int s = 0; s < kSums; ++s) {
            mbar_init(sum1_full0 + 8 * s, 1);
            mbar_init(sum1_empty0 + 8 * s, 32 * kTeamWarps);
        }
        for (int s = 0; s < 2 * kMaxFilters; ++s) {
            mbar_init(w_full0 + 8 * s, 1);
            mbar_init(w_empty0 + 8 * s, 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(x_full0 + 8 * s, kRunWarps);
            mbar_init(x_empty0 + 8 * s, 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(sum2_full0 + 8 * s, 1);
            mbar_init(sum2_empty0 + 8 * s, 32 * kTeamWarps);
        }
        ctrl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    for (int i = threadIdx.x; i < p.a.K; i += kThreads) bias1[i] = p.a.bias1[i];
    for (int i = threadIdx.x; i < p.a.K2; i += kThreads) bias2[i] = p.a.bias2[i];
    if (warp == kFirst) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(base + (uint32_t)offsetof(PairCtrl, tmem_base)), "r"((uint32_t)p.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&ctrl->tmem_base);
    const uint32_t tmem_sum1 = tmem + (uint32_t)(p.sum2_stages * p.a.K2);             // the first convolution's stages behind the second's sums
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (warp < kRunWarps || warp >= kInWarps) asm volatile("griddepcontrol.wait;" ::: "memory");      // (filters: not the previous kernel's)

    auto wait_all = [&](uint32_t bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, limit)) != 0; };
    auto chunks_of = [&](int g) { return min(GC, p.chunks - g * GC); };
    const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);      // see conv_tc.cu
    bool ok = true;
    Ring slot, sum, xs, filters;
    // the next group's filters: their stage is another, or - where all stay - the group's own, filled once
    auto next_filters = [&](int g) {
        if (!p.w_stays) filters.next(p.w_stages);
        else filters.at = g + 1 < p.groups ? (uint32_t)g + 1u : 0u;
    };
    if (warp < kRunWarps) {
        // ------------------------------ x and the shortcut: each warp half of the runs ------------------------------
        const uint4* xv = reinterpret_cast<const uint4*>(p.a.x);
        const uint4* x2v = reinterpret_cast<const uint4*>(p.a.x2);
        const uint4* rv = reinterpret_cast<const uint4*>(p.a.res);
        const int chunk2 = p.a.x2_chunk0 > 0 ? p.a.x2_chunk0 : p.chunks1;
        auto share = [&](int n) { return (uint32_t)((n + kRunWarps - 1 - warp) / kRunWarps) * 2048u; };
        for (int tile = blockIdx.x; tile < p.m_tiles && ok; tile += gridDim.x) {
            const long long f0 = (long long)(p.m_first + p.m_sign * tile) * 128;
            if (!(ok = wait_all(x_empty0 + 8 * xs.at, xs.phase ^ 1))) break;
            if (lane == 0) mbar_expect_tx(x_full0 + 8 * xs.at, share(p.chunks1));
            __syncwarp();
            for (int c = warp + kRunWarps * lane; c < p.chunks1; c += 32 * kRunWarps)
                bulk_copy(x0 + xs.at * x_bytes + (uint32_t)c * 2048u,
                          (c < chunk2 ? xv + (long long)c * p.plane_x : x2v + (long long)(c - chunk2) * p.plane_x2) + f0, 2048u, x_full0 + 8 * xs.at);
            xs.next(p.x_stages);
            for (int g = 0; g < p.groups; ++g) {
                if (!(ok = wait_all(slot_empty0 + 8 * slot.at, slot.phase ^ 1))) break;
                const int cg = rv ? chunks_of(g) : 0, c = warp + kRunWarps * lane;
                if (lane == 0) mbar_expect_tx(slot_full0 + 8 * slot.at, share(cg));
                __syncwarp();
                if (c < cg)
                    bulk_copy(slot0 + slot.at * slot_bytes + (uint32_t)c * 2048u, rv + (long long)(g * GC + c) * p.plane_res + f0, 2048u, slot_full0 + 8 * slot.at);
                __syncwarp();
                slot.next(p.slots);
            }
        }
        if (!ok && lane == 0) { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 1); }
    } else if (warp < kInWarps) {
        // ------------------------------ filters of one convolution ------------------------------
        const int which = warp - kRunWarps;
        const uint8_t* src = reinterpret_cast<const uint8_t*>(which ? p.a.w2 : p.a.w1);
        const uint32_t stage_bytes = which ? w2_bytes : w1_bytes, at = which ? w2_at : w1_at;
        const uint32_t full = w_full0 + (uint32_t)which * 8u * kMaxFilters, empty = w_empty0 + (uint32_t)which * 8u * kMaxFilters;
        for (int tile = blockIdx.x; tile < p.m_tiles && ok; tile += gridDim.x) {
            for (int g = 0; g < p.groups; ++g) {
                if (!p.w_stays && !(ok = wait_all(empty + 8 * filters.at, filters.phase ^ 1))) break;
                const uint32_t bytes = which ? (uint32_t)(chunks_of(g) * p.a.K2) * 16u : w1_bytes, half = bytes / 32u * 16u;
                if (lane == 0) mbar_expect_tx(full + 8 * filters.at, bytes);
                __syncwarp();
                if (lane < 2) {
                    const uint32_t off = lane ? half : 0u;
                    bulk_copy(at + filters.at * stage_bytes + off, src + (long long)g * stage_bytes + off, lane ? bytes - half : half, full + 8 * filters.at);
                }
                __syncwarp();
                next_filters(g);
            }
            if (p.w_stays) break;
        }
        if (!ok && lane == 0) { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 1); }
    } else if (warp == kFirst) {
        // ------------------------------ first convolution's MMAs ------------------------------
        const uint32_t leader = elect_one();
        for (int tile = blockIdx.x; tile < p.m_tiles && ok; tile += gridDim.x) {
            if (!(ok = wait_all(x_full0 + 8 * xs.at, xs.phase))) break;
            for (int g = 0; g < p.groups; ++g) {
                if (!(ok = wait_all(w_full0 + 8 * filters.at, filters.phase) && wait_all(sum1_empty0 + 8 * sum.at, sum.phase ^ 1))) break;
                tc_fence_after();
                const uint32_t idesc = idesc0 | ((uint32_t)chunks_of(g) << 17);
                uint32_t a_lo = ((x0 + xs.at * x_bytes) >> 4) | (128u << 16);
                uint32_t b_lo = ((w1_at + filters.at * w1_bytes) >> 4) | ((uint32_t)G << 16);
                const uint32_t d = tmem_sum1 + sum.at * (uint32_t)G;
#pragma unroll 1
                for (int i = 0; i < p.chunks1 >> 1; ++i) {
                    umma_bf16_lo_if(leader, d, a_lo, b_lo, idesc, i ? 1u : 0u);
                    a_lo += 256u;
                    b_lo += 2u * (uint32_t)G;
                }
                if (leader) umma_commit(sum1_full0 + 8 * sum.at);
                if (leader && !p.w_stays) umma_commit(w_empty0 + 8 * filters.at);
                if (leader && g == p.groups - 1) umma_commit(x_empty0 + 8 * xs.at);
                __syncwarp();
                next_filters(g);
                sum.next(kSums);
            }
            xs.next(p.x_stages);
        }
        if (!ok && leader) { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 2); }
    } else if (warp < kFirst) {
        // ------------------------------ finish ------------------------------
        constexpr int HC = G / 16;                                  // chunks of a group that a warp finishes: half of them
        const int team = (warp - kEpi0) / kTeamWarps, quarter = warp & 3, half = ((warp - kEpi0) >> 2) & 1, row = quarter * 32 + lane;
        const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
        struct Place { bool exists, interior, y_kept; long long f; };
        auto place_of = [&](int tile) {                             // this thread's position; f: its vector in y's and z's planes
            Place o;
            const int f = (p.m_first + p.m_sign * tile) * 128 + row;
            const int n = (int)fdiv((uint32_t)f, p.div_p2out), rem = f - n * p.P2;
            const int hp = (int)fdiv((uint32_t)rem, p.div_qp), wq = rem - hp * p.Qp;
            o.exists = f < p.m_total;
            o.interior = o.exists && hp >= 1 && hp <= p.a.P && wq >= 1 && wq <= p.a.Q;
            o.f = f;
            o.y_kept = o.exists;
            if (p.a.y_split) {                                      // see conv_tc.cu: the pixel's place in its parity image
                const int h = hp - 1, w = wq - 1;
                const int pp = (h & 1) ? ((w & 1) ? 2 : 1) : ((w & 1) ? 3 : 0);
                if (p.a.y_quarter && pp) o.y_kept = false;
                o.f = ((long long)pp * p.a.N + n) * p.y_P2h + ((h >> 1) + 1) * p.y_Wh2 + ((w >> 1) + 1);
            }
            return o;
        };
        auto pack = [&](const float (&s)[8], int relu) {
            return relu ? make_uint4(pack_bf16x2_relu(s[0], s[1]), pack_bf16x2_relu(s[2], s[3]), pack_bf16x2_relu(s[4], s[5]), pack_bf16x2_relu(s[6], s[7]))
                        : make_uint4(pack_bf16x2(s[0], s[1]), pack_bf16x2(s[2], s[3]), pack_bf16x2(s[4], s[5]), pack_bf16x2(s[6], s[7]));
        };
        uint4* yv = reinterpret_cast<uint4*>(p.a.y);
        uint4* zv = reinterpret_cast<uint4*>(p.a.z);
        const int cols2 = p.a.K2 / 16, first2 = (cols2 + 1) / 2;    // units of 16 columns of z, those of the first half
        // z of this CTA's tile number `local`: the teams take turns
        auto finish_z = [&](const Place& o, int local) -> bool {
            if (!wait_all(sum2_full0 + 8 * team, (uint32_t)(local / kTeams) & 1u)) return false;
            tc_fence_after();
            const uint32_t sums = tmem + lanes + (uint32_t)((local & (p.sum2_stages - 1)) * p.a.K2);
#pragma unroll 1
            for (int u = half ? first2 : 0; u < (half ? cols2 : first2); ++u) {
                uint32_t v[16];
                tmem_ld16(sums + (uint32_t)(16 * u), v);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float4 ba = *reinterpret_cast<const float4*>(bias2 + 16 * u + 8 * j), bb = *reinterpret_cast<const float4*>(bias2 + 16 * u + 8 * j + 4);
                    const float s[8] = {__uint_as_float(v[8 * j]) + ba.x, __uint_as_float(v[8 * j + 1]) + ba.y, __uint_as_float(v[8 * j + 2]) + ba.z,
                                        __uint_as_float(v[8 * j + 3]) + ba.w, __uint_as_float(v[8 * j + 4]) + bb.x, __uint_as_float(v[8 * j + 5]) + bb.y,
                                        __uint_as_float(v[8 * j + 6]) + bb.z, __uint_as_float(v[8 * j + 7]) + bb.w};
                    uint4 out = pack(s, p.a.relu2);
                    if (!o.interior) out = make_uint4(0, 0, 0, 0);
                    if (o.exists) zv[(long long)(2 * u + j) * p.plane_y + o.f] = out;
                }
            }
            tc_fence_before();
            mbar_arrive(sum2_empty0 + 8 * team);
            return true;
        };
        Place before;
        int local = 0, q = 0;
        for (int tile = blockIdx.x; tile < p.m_tiles && ok; tile += gridDim.x, ++local) {
            const Place o = place_of(tile);
            bool z_due = local > 0 && ((local - 1) & 1) == team;
            for (int g = 0; g < p.groups; ++g, ++q) {
                if (q % kTeams == team) {
                    if (!(ok = wait_all(sum1_full0 + 8 * sum.at, sum.phase) && wait_all(slot_full0 + 8 * slot.at, slot.phase))) break;
                    tc_fence_after();
                    uint32_t v[8 * HC];
                    tmem_ld32(tmem_sum1 + lanes + sum.at * (uint32_t)G + (uint32_t)(half * (G / 2)), v);
                    const int c0 = g * GC + half * HC;
                    uint8_t* at = smem_raw + (slot0 - base) + slot.at * slot_bytes + (uint32_t)(half * HC) * 2048u + (uint32_t)row * 16u;
                    uint4 r[HC];
#pragma unroll
                    for (int c = 0; c < HC; ++c) r[c] = p.a.res ? *reinterpret_cast<const uint4*>(at + c * 2048) : make_uint4(0, 0, 0, 0);
                    tmem_ld_wait();
                    tc_fence_before();
                    mbar_arrive(sum1_empty0 + 8 * sum.at);
#pragma unroll
                    for (int c = 0; c < HC; ++c) {
                        if (c0 + c >= p.chunks) break;
                        const float4 ba = *reinterpret_cast<const float4*>(bias1 + 8 * (c0 + c)), bb = *reinterpret_cast<const float4*>(bias1 + 8 * (c0 + c) + 4);
                        float s[8] = {__uint_as_float(v[8 * c]) + ba.x, __uint_as_float(v[8 * c + 1]) + ba.y, __uint_as_float(v[8 * c + 2]) + ba.z,
                                      __uint_as_float(v[8 * c + 3]) + ba.w, __uint_as_float(v[8 * c + 4]) + bb.x, __uint_as_float(v[8 * c + 5]) + bb.y,
                                      __uint_as_float(v[8 * c + 6]) + bb.z, __uint_as_float(v[8 * c + 7]) + bb.w};
                        if (p.a.res) {
                            s[0] += __uint_as_float(r[c].x << 16); s[1] += __uint_as_float(r[c].x & 0xffff0000u);
                            s[2] += __uint_as_float(r[c].y << 16); s[3] += __uint_as_float(r[c].y & 0xffff0000u);
                            s[4] += __uint_as_float(r[c].z << 16); s[5] += __uint_as_float(r[c].z & 0xffff0000u);
                            s[6] += __uint_as_float(r[c].w << 16); s[7] += __uint_as_float(r[c].w & 0xffff0000u);
                        }
                        uint4 out = pack(s, p.a.relu1);
                        if (!o.interior) out = make_uint4(0, 0, 0, 0);
                        *reinterpret_cast<uint4*>(at + c * 2048) = out;
                        if (p.a.y_split && o.y_kept) yv[(long long)(c0 + c) * p.plane_y + o.f] = out;
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // for the MMAs and the copies out
                    mbar_arrive(y_ready0 + 8 * slot.at);
                    if (z_due) {
                        z_due = false;
                        if (!(ok = finish_z(before, local - 1))) break;
                    }
                }
                slot.next(p.slots);
                sum.next(kSums);
            }
            if (ok && z_due) ok = finish_z(before, local - 1);      // (a tile of one group: the other team's)
            before = o;
        }
        if (ok && local > 0 && ((local - 1) & 1) == team) ok = finish_z(before, local - 1);
        if (!ok && lane == 0) { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 3); }
    } else if (warp == kSecond) {
        // ------------------------------ second convolution's MMAs ------------------------------
        const uint32_t leader = elect_one();
        const uint32_t idesc = idesc0 | ((uint32_t)(p.a.K2 >> 3) << 17);
        int local = 0;
        for (int tile = blockIdx.x; tile < p.m_tiles && ok; tile += gridDim.x, ++local) {
            const uint32_t d = tmem + (uint32_t)((local & (p.sum2_stages - 1)) * p.a.K2);
            for (int g = 0; g < p.groups; ++g) {
                if (!(ok = wait_all(w_full0 + 8 * (kMaxFilters + filters.at), filters.phase) && wait_all(y_ready0 + 8 * slot.at, slot.phase))) break;
                // the stage's columns were last used sum2_stages tiles ago: z of that tile has been read
                const int read = local - p.sum2_stages;
                if (g == 0 && read >= 0 && !(ok = wait_all(sum2_empty0 + 8 * (read & 1), (uint32_t)(read >> 1) & 1u))) break;
                tc_fence_after();
                uint32_t a_lo = ((slot0 + slot.at * slot_bytes) >> 4) | (128u << 16), b_lo = ((w2_at + filters.at * w2_bytes) >> 4) | ((uint32_t)p.a.K2 << 16);
                const int ks = chunks_of(g) >> 1;
#pragma unroll 1
                for (int i = 0; i < ks; ++i) {
                    umma_bf16_lo_if(leader, d, a_lo, b_lo, idesc, (g | i) ? 1u : 0u);
                    a_lo += 256u;
                    b_lo += 2u * (uint32_t)p.a.K2;
                }
                if (leader) umma_commit(slot_empty0 + 8 * slot.at);
                if (leader && !p.w_stays) umma_commit(w_empty0 + 8 * (kMaxFilters + filters.at));
                if (leader && g == p.groups - 1) umma_commit(sum2_full0 + 8 * (local & 1));
                __syncwarp();
                slot.next(p.slots);
                next_filters(g);
            }
        }
        if (!ok && leader) { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 4); }
    } else {
        // ------------------------------ copies out: half of the chunks each ------------------------------
        const int turn = warp - kOut0;
        uint4* yv = reinterpret_cast<uint4*>(p.a.y);
        for (int tile = blockIdx.x; tile < p.m_tiles && ok; tile += gridDim.x) {
            const long long f0 = (long long)(p.m_first + p.m_sign * tile) * 128;
            const uint32_t bytes = (uint32_t)min(128LL, p.m_total - f0) * 16u;
            for (int g = 0; g < p.groups; ++g) {
                if (!(ok = wait_all(y_ready0 + 8 * slot.at, slot.phase))) break;
                const int c = turn + kOutWarps * lane;
                if (!p.a.y_split && c < chunks_of(g)) {
                    bulk_store(yv + (long long)(g * GC + c) * p.plane_y + f0, slot0 + slot.at * slot_bytes + (uint32_t)c * 2048u, bytes);
                    bulk_store_commit();
                    bulk_store_wait_read();
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(slot_empty0 + 8 * slot.at);
                slot.next(p.slots);
            }
        }
        bulk_store_wait();
        if (!ok && lane == 0) { atomicExch(&ctrl->abort_flag, 1); atomicExch(p.status, 5); }
    }

    // ---- teardown: everyone arrives here, also after a wait that ran out ----
    if (*abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);            // copies in flight land before the memory is given back
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == kFirst) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)p.tmem_cols) : "memory");
    }
}

}  // namespace

// One CTA per SM takes a tile of 128 positions at a time: below that many tiles the layers of their own spread over more SMs.  And the ring
// needs four slots: a layer with a projection's channels behind its own (336 -> 512 -> 80 at 28x28, batch 128) leaves room for one; with
// groups of 32 channels, which would fit, it took 121 us against 87 of the two kernels.  Where it fits it was the shorter
// way at every size measured, ResNet-50, us of the two kernels -> of this one: batch 128, 56x56 48 -> 256 -> 48 136 -> 84, 28x28
// 80 -> 512 -> 80 83 -> 50, 14x14 160 -> 1024 -> 160 46 -> 34; batch 32, 56x56 34 -> 23; batch 8, 56x56 13.5 -> 10.2.
bool plan_pair(const PairArgs& a, PairPlan* plan) {
    plan->valid = 0;
    const int m_tiles = (int)((used_vecs(a.N, a.P, a.Q) + 127) / 128);
    if (m_tiles < sm_count() || a.K2 > 256 || (a.y_split && (a.P % 2 || a.Q % 2))) return false;
    const int sum2_stages = 2 * a.K2 + kSums * G <= 512 ? 2 : 1, groups = (a.K + G - 1) / G;
    int cols = 32;
    while (cols < sum2_stages * a.K2 + kSums * G) cols *= 2;
    const unsigned x_bytes = (unsigned)(a.C_pad / 8) * 2048u, slot = (unsigned)GC * 2048u;
    const unsigned filters = (unsigned)(a.C_pad / 8 * G) * 16u + (unsigned)(GC * a.K2) * 16u;
    const unsigned fixed = (unsigned)sizeof(PairCtrl) + (unsigned)(a.K + a.K2) * 4u + 128u;
    auto slots_with = [&](int xs, int ws) {
        const unsigned used = fixed + (unsigned)xs * x_bytes + (unsigned)ws * filters;
        return used < kSmemMax ? (int)((kSmemMax - used) / slot) / kTeams * kTeams : 0;
    };
    const bool stays = groups <= kMaxFilters && slots_with(2, groups) >= 4;
    const int ws = stays ? groups : 2;
    int xs = 2, slots = slots_with(xs, ws);
    if (slots < 4) slots = slots_with(--xs, ws);
    if (slots < 4) return false;
    if (cudaFuncSetAttribute(conv_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    plan->x_stages = xs; plan->sum2_stages = sum2_stages; plan->slots = slots < kMaxSlots ? slots : kMaxSlots;
    plan->w_stages = ws; plan->w_stays = stays; plan->tmem_cols = cols;
    plan->smem_bytes = fixed + (unsigned)xs * x_bytes + (unsigned)ws * filters + (unsigned)plan->slots * slot;
    plan->valid = 1;
    return true;
}

void launch_pair(const PairPlan& plan, const PairArgs& a, int* d_status, cudaStream_t st) {
    PairParams p;
    memset(&p, 0, sizeof(p));
    p.a = a;
    p.Qp = row_vecs(a.Q); p.P2 = image_vecs(a.P, a.Q);
    const long long plane = plane_vecs(a.N, a.P, a.Q);
    p.m_total = a.y_split ? a.N * p.P2 : (int)used_vecs(a.N, a.P, a.Q); p.m_tiles = (p.m_total + 127) / 128;
    p.m_first = a.reverse ? p.m_tiles - 1 : 0; p.m_sign = a.reverse ? -1 : 1;
    p.plane_x = p.plane_res = p.plane_y = plane;
    p.plane_x2 = a.x2_plane_mult > 1 ? plane_vecs(4 * a.N, a.P, a.Q) : plane;
    if (a.y_split) {
        p.y_Wh2 = row_vecs((a.Q + 1) / 2); p.y_P2h = image_vecs((a.P + 1) / 2, (a.Q + 1) / 2);
        p.plane_y = plane_vecs(4 * a.N, (a.P + 1) / 2, (a.Q + 1) / 2);
    }
    p.chunks1 = a.C_pad / 8; p.chunks = a.K / 8; p.groups = (a.K + G - 1) / G;
    p.x_stages = plan.x_stages; p.sum2_stages = plan.sum2_stages; p.slots = plan.slots; p.w_stages = plan.w_stages; p.w_stays = plan.w_stays; p.tmem_cols = plan.tmem_cols;
    p.status = d_status;
    p.div_p2out = make_fastdiv((uint32_t)p.P2);
    p.div_qp = make_fastdiv((uint32_t)p.Qp);
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(p.m_tiles < sm_count() ? p.m_tiles : sm_count()));
    cfg.blockDim = dim3((unsigned)kThreads);
    cfg.dynamicSmemBytes = plan.smem_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    void* args[1] = {(void*)&p};
    cudaLaunchKernelExC(&cfg, (const void*)conv_pair_kernel, args);
}

}  // namespace fp
