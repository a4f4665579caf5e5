// Internal declarations shared by the host graph builder and the kernel launchers.
//
// Activation layout ("planar-8 with border"): channels are grouped in chunks of 8 (one 16-byte
// vector of bf16, or 32 bytes of fp32); every image has a row of zeros above it and a column of
// zeros to its left.  The row below an image is the next image's upper one, the column to the
// right of a row the next row's left one; behind the last image of a plane come W + 2 zeros.
// For a batch of N images of H x W pixels and C_pad channels the vector of chunk j, image n,
// pixel (h, w) sits at vector index
//       j * plane  +  n * P2  +  (h + 1) * (W + 1)  +  (w + 1),      P2 = (H + 1) * (W + 1),
// plane = N * P2 + W + 2 rounded up to whole cache lines.
// So each chunk is one contiguous plane over the whole batch; a run of consecutive "flat
// positions" f = n*P2 + (h+1)*(W+1) + (w+1) is contiguous in memory for every chunk, and the
// 3x3 neighbourhood of position f is f + dr*(W+1) + ds.  Every kernel that writes a whole tensor
// writes all of its positions, zeros on the border, so the border never has to be cleared.  What rounds a
// plane up to whole lines, and the guard vectors, are defined nowhere.
// Of a parity-split tensor (ConvArgs::y_split) less is written: not the border row of the images of even rows,
// nor the border column of those of even columns, nor anything behind the last image - and with
// PairArgs::y_quarter the parity-00 images alone.  Buffers are reused, so those places hold other tensors' values,
// which need not be finite.  A reader may fetch them, as rows of an operand, but has to leave the results they give
// where they are (by position; a product with zero would not do): the strided convolutions read no such place for a
// position of theirs that exists, 1x1 layers give each position's to that position.
// (With a border on all four sides, which was the layout before, 7x7 pixels took 81 positions instead
// of 64, 14x14 256 instead of 225, 28x28 900 instead of 841: work of every convolution and bytes of every tensor.)
// Buffers carry `kGuardVectors` vectors of slack before and after the data, because tiles of
// flat positions read a halo that may start before the first plane or end after the last.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stddef.h>

#include <atomic>
#include <vector>

namespace fp {

// Streaming multiprocessors of the current device (asked once per device; 148 on a B200).  Grids are sized from it.
inline int sm_count() {
    static std::atomic<int> cached[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return 148; }
    if (cached[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) { cudaGetLastError(); n = 148; }
        cached[dev] = n;
    }
    return cached[dev];
}

constexpr int kGuardVectors = 1024;   // >= 128 + (W + 3) + 8 for every supported width (W <= 512)
constexpr int kMaxWidth = 512;
// Vectors of a row, of an image, of N images with the zeros behind them, and from a chunk's plane to the next one's: whole lines of
// 128 bytes (without, a warp's 512 bytes lay across 17 sectors: ResNet-50 batch 1 190 -> 195 us).
__host__ __device__ constexpr int row_vecs(int W) { return W + 1; }
__host__ __device__ constexpr int image_vecs(int H, int W) { return (H + 1) * (W + 1); }
__host__ __device__ constexpr long long used_vecs(int N, int H, int W) { return (long long)N * image_vecs(H, W) + W + 2; }
__host__ __device__ constexpr long long plane_vecs(int N, int H, int W) { return (used_vecs(N, H, W) + 7) / 8 * 8; }

// ---------------------------------------------------------------------------------------
// Convolution launch description (one fused operator: conv + bias + residual + ReLU)
// ---------------------------------------------------------------------------------------
struct ConvArgs {
    const void* x;        // input activations, planar-8 with border (vector 0 of plane 0)
    void* y;              // output activations, same layout, P x Q pixels, K_pad channels
    const void* res;      // residual operand or nullptr
    const void* w;        // packed filters [R*S][C_pad/8][K_pad][8]
    const float* bias;    // [K_pad]
    int N, H, W, C_pad, P, Q, K_pad, R, S, stride, pad;   // pad: rows; columns are padded by pad when S == R, by (S-1)/2 otherwise
    int relu;
    int res_mode;         // 0 none, 1 same shape as y, 2 subsample + zero-channel pad
    int res_H, res_W, res_C_pad, res_C, res_pad_lo, res_stride;
    // Scattered output (tensor-core path): the K_pad packed filter rows hold only the kept filters of a convolution
    // whose output tensor keeps its full width out_C_pad (a residual stream that other layers write too); output
    // channel c takes accumulator column out_map[c], or only the shortcut when out_map[c] < 0.  Filter tile t
    // (rows t*n_tile ..) owns the output chunks tile_chunk0[t] .. tile_chunk0[t+1]-1 and holds exactly their filters.
    int scatter, out_C_pad;
    const int32_t* out_map;        // [out_C_pad], device
    const int32_t* tile_chunk0;    // [n_tiles + 1], device
    int n_tile_forced;             // > 0: filters per CTA tile fixed by the caller (scatter), else chosen by the plan
    // Parity-split tensors (tensor-core path).  A tensor that only stride-2 convolutions read is stored as four
    // half-resolution tensors, one per (row parity, column parity) of its pixels, in the order 00, 10, 11, 01, laid out
    // as 4 N images of (H/2) x (W/2) pixels: image pp * N + n holds the pixels (2i + a, 2j + b) of image n.
    int y_split;                   // write the output that way (the kernel's own grid stays P x Q)
    int x_plane_mult;              // 0/1: x is a plain tensor; 4: x is a split tensor and this 1x1 layer reads its images
                                   //      0 .. N-1 only (parity 00 = the pixels a 1x1 / stride-2 convolution reads)
    // A second input tensor along the reduction (tensor-core path, 1x1 / stride-1 layers): channel chunks >= x2_chunk0 of
    // the C_pad channels come from x2 (chunk - x2_chunk0 of it), a tensor on the same position grid - the input of a
    // projection shortcut, whose filters are then stacked behind this layer's along the channels (Sec. IV-B: one
    // convolution [W2' || S_w] instead of two and an add).  x2_plane_mult 4: x2 is parity-split and its images 0..N-1
    // (parity 00) are the ones read, as for a 1x1 / stride-2 convolution.
    const void* x2;
    int x2_chunk0;                 // 0: no second input stacked along the channels
    int x2_plane_mult;
    // The same for a 3x3 / stride-1 layer with streamed filters: the projection enters as extra K groups that have a
    // centre tap only - x2_C_pad channels of x2, filters w2 = [chunk][K_pad][8] (the projection's own packed bank).
    const void* w2;
    int x2_C_pad;                  // 0: none
    int x_s2d;                     // x is a split tensor and this is the 3x3 / stride 2 / pad 1 convolution over the tensor
                                   // it was split from: H, W, P, Q are the half resolution, stride is given as 1; the nine
                                   // taps read the parity images at offsets -1 / 0 rows and columns
    int reverse;                   // walk the output positions from the last to the first (tensor-core path)
};

// Filter preparation --------------------------------------------------------------------
// W'[k0+k][c0+c][r+r0][s+s0] = omega_k * W[k][c][r][s] inside a (K_dst, C_dst, R_dst, S_dst) bank.
void launch_fold_weights(const float* w, const float* bn, int K, int C, int R, int S, float eps,
                         float* dst, int C_dst, int R_dst, int S_dst, int k0, int c0, int r0, int s0,
                         cudaStream_t st);
// b[k0+k] = lambda_k (accumulate = 0) or b[k0+k] + lambda_k (accumulate = 1)
void launch_fold_bias(const float* bn, int K, float eps, float* dst_b, int k0, int accumulate, cudaStream_t st);
// unit centre taps: dst[k0+k][c0 + k - shift][R/2][S/2] = 1 for 0 <= k-shift < C_id
void launch_identity_filters(float* dst, int C_dst, int R, int S, int k0, int c0, int K_id, int C_id, int shift,
                             cudaStream_t st);
void launch_count_nonfinite(const float* p, size_t n, int* d_count, cudaStream_t st);
void launch_score_filters(const float* w, int K, int per_filter, int norm, double* scores, cudaStream_t st);
// score, rank and mask one bank; `scores` has room for K
void launch_score_rank(const float* w, int K, int per_filter, int norm, int q, double* scores, int32_t* rank, uint8_t* mask,
                       cudaStream_t st);
// Selection over ALL filter banks of a model (fp_prune, and the loop body of Algorithm 1).  One SoftBank per convolution;
// filter_bank[g] names the bank of global filter g (filters of all banks numbered consecutively, bank by bank).
struct SoftBank {
    float* w;             // K x per fp32
    long long dw_off;     // element offset of the bank's addends in the update array
    int K, per, q;        // filters, weights per filter, filters to mask
    int k_off;            // global number of the bank's first filter
};
// w += dw (one fp32 addition per weight; dw may be nullptr: the weights stay) and the scores of the weights that result, in
// the fixed summation order of launch_score_filters
void launch_bank_score(const SoftBank* banks, const int32_t* filter_bank, int total_filters, const float* dw, int norm,
                       double* scores, cudaStream_t st);
// per bank: rank by (score, index) ascending, mask the first q - and, with zeroize, set their weights to zero
void launch_bank_rank(const SoftBank* banks, const int32_t* filter_bank, int total_filters, const double* scores, int zeroize,
                      int32_t* rank, uint8_t* mask, cudaStream_t st);

// Packing of a planned graph's filters, biases and FC matrix: all jobs in one launch.  Index arrays (packed row -> fused
// filter, packed channel -> fused channel, -1 = zeros) are parts of one array, named by their offsets.
enum { PACK_CONV = 0, PACK_CHAIN = 1, PACK_STEM = 2, PACK_STEM_DIRECT = 3, PACK_FC = 4, PACK_BIAS = 5, PACK_QUAD = 6 };
constexpr int kPackThreads = 256;
// A block of a convolution's filters: 32 filter rows times a run of units, a unit being as many chunks of 8 channels as have at
// most nine taps together (eight chunks of a 1x1 filter; of a filter with more taps, nine at a time).  Runs of four where a bank
// has many units - the start of a block, four dependent loads, is then paid once -, of one where it is small.
constexpr int kPackTaps = 9, kPackElems = 8 * kPackTaps;
__host__ __device__ constexpr int pack_span(int RS) { return RS == 1 ? 8 : RS >= kPackTaps ? 1 : kPackTaps / RS; }
__host__ __device__ constexpr int pack_run(int units) { return units >= 16 ? 4 : units >= 8 ? 2 : 1; }
struct PackJob {
    const float* w;       // fused fp32 filters K x C x RS (PACK_FC: the FC matrix; PACK_BIAS: the shifts)
    const float* w2;      // a second bank stacked behind the first along the channels / a second shift to add, or nullptr
    void* out;
    int kind, f32;        // f32: fp32 vectors instead of bf16
    int units, first_block;   // units: one thread's work each (not of filters, see pack_blocks)
    int C, C2, RS;        // channels of the fused banks (row pitches), taps
    int rows, K_pad;      // packed rows with and without the last filter tile's padding
    int chunks, chunks1;  // packed channel chunks, those of the first bank
    int n_tile, cg;       // PACK_CONV: rows per filter tile, chunks per K group
    int row, chan, row2, chan2;
    float scale;          // PACK_FC
};
inline int pack_blocks(const PackJob& j) {
    if (j.kind == PACK_CONV || j.kind == PACK_CHAIN) {
        const int span = pack_span(j.RS), units = (j.chunks + span - 1) / span * ((j.RS + kPackTaps - 1) / kPackTaps), run = pack_run(units);
        return (j.rows + 31) / 32 * ((units + run - 1) / run);
    }
    return (j.units + kPackThreads - 1) / kPackThreads;
}
void launch_pack(const PackJob* jobs, const int32_t* block_job, int n_blocks, const int32_t* idx, cudaStream_t st);

// Memory-bound operators ------------------------------------------------------------------
// Both convert images n0 .. n0 + n_count - 1 of a batch of N images (`in` and `out` are the whole batch's buffers).
void launch_input_to_planar(const void* in, int in_is_bf16, void* out, int out_is_bf16, int N, int C, int H, int W,
                            int C_pad, int n0, int n_count, cudaStream_t st);
void launch_input_to_stem_planar(const void* in, int in_is_bf16, void* out, int N, int C, int H, int W, int n0, int n_count,
                                 cudaStream_t st);
void launch_maxpool(const void* x, void* y, int is_bf16, int N, int H, int W, int C_pad, int P, int Q, int R,
                    int stride, int pad, cudaStream_t st);
void launch_head(const void* x, int is_bf16, int N, int H, int W, int C_pad, const float* fcw, const float* fcb,
                 int n_classes, float* logits, float* pool_scratch, int max_batch, cudaStream_t st);      // max_batch: of the handle
void launch_planar_to_nchw_f32(const void* x, int is_bf16, float* out, int N, int H, int W, int C_pad, int C_out,
                               int split, cudaStream_t st);

// Convolutions ------------------------------------------------------------------------------
// CUDA-core validation kernels: fp32 activations/filters, or bf16 activations/filters with
// fp32 accumulation (same storage as the tensor-core path, used to localise differences).
void launch_conv_simt(const ConvArgs& a, int is_bf16, cudaStream_t st);

// Tensor-core path: per-layer plan built once per fp_prune.
struct ConvPlanTC {
    int valid;
    int split;            // > 0: few positions - conv_split_kernel, the reduction over that many CTAs (conv_split.cu)
    int flat;             // 1: stride-1 "same" convolution, activation tiles fetched as contiguous runs
                          //    of flat positions (bulk copies); 0: gathered by loader threads
    int b_resident;       // flat only: the whole filter bank stays in shared memory
    int blocked_bank;     // 1: 1x1 layer with unified stages, bank stored block by block; 2: gathered or resident layer with
                          // several filter tiles, bank stored tile by tile; 3: streamed filters, stored as for 1, a row of
                          // taps of a K group being one copy (PackJob in each case)
    int cg;               // channel chunks (of 8) per K block
    int groups;           // K blocks per filter tap = ceil((C_pad/8) / cg)
    int halo;             // flat: vectors fetched before and after the 128 positions of a tile
    int rows_a;           // flat: vectors per chunk per tile (128 + 2*halo, rounded up to 8)
    int a_stages, b_stages;
    int tpk;              // gather: filter taps per K block (several when the channel count is small)
    int n_tile, n_tiles;  // filters per CTA tile (multiple of 16, <= 256)
    int epi_warps;        // 4, 8 for wide filter tiles, 16 where several tiles are complete together
    int alternate;        // eight epilogue warps as two teams that take every other tile, in launches of more tiles than CTAs
    int tps;              // streamed filters: 128-position tiles per pipeline step
    int b_kept;           // streamed filters: a stage for every block of the bank, copied once
    int tmem_cols;
    unsigned smem_bytes;
    int ctas_per_sm;
};
// Filters per CTA tile the plan would choose for K_pad filter rows of this geometry (used to lay out scattered banks).
void conv_tc_filter_tile(const ConvArgs& a, int K_pad, int* n_tile, int* n_tiles);
// The plan for few output positions, where it applies: false, and nothing changed, where it does not.
bool plan_conv_split(const ConvArgs& a, ConvPlanTC* plan);
void launch_conv_split(const ConvPlanTC& plan, const ConvArgs& a, int* d_status, cudaStream_t st, int skip_round, long long wait_cycles);
// Returns 0 on success, otherwise writes a message.
int plan_conv_tc(const ConvArgs& a, ConvPlanTC* plan, char* err, size_t err_len);
// ConvPlanTC::tps and ::alternate, in a launch with these arguments
int conv_tc_step_tiles(const ConvPlanTC& plan, const ConvArgs& a);
bool conv_tc_alternates(const ConvPlanTC& plan, const ConvArgs& a);
// skip_round / wait_cycles: diagnostic launch (see fp_debug_expire_wait): the activation producer of a stride-1 layer leaves
// out one round of copies and every wait gives up after wait_cycles SM clock cycles; -1 / 0 for a normal launch
void launch_conv_tc(const ConvPlanTC& plan, const ConvArgs& a, int* d_status, cudaStream_t st, int skip_round = -1,
                    long long wait_cycles = 0);

// Two 1x1 / stride-1 convolutions as one kernel, the second reading the first's output (pair_tc.cu): the layer that writes a bottleneck
// network's residual stream, and the narrow layer that reads it.
struct PairArgs {
    const void *x, *x2;   // input of the first layer; chunks >= x2_chunk0 (0: none) come from x2, as in ConvArgs
    const void* res;      // its shortcut operand, on its output's grid, or nullptr
    const void *w1, *w2;  // filters: [group of kPairGroup][C_pad / 8][kPairGroup rows][8] and [K / 8][K2][8]
    const float *bias1, *bias2;
    void *y, *z;          // the two outputs, y_split: both parity-split
    int N, P, Q, C_pad, K, K2;          // K, K2: padded filters of the two
    int x2_chunk0, x2_plane_mult, y_split, relu1, relu2, reverse;
    int y_quarter;                      // y_split: only the parity-00 images of y are written - nobody but 1x1 / stride-2 convolutions reads the rest
};
constexpr int kPairGroup = 64;          // channels of y made at a time
struct PairPlan { int valid, x_stages, sum2_stages, slots, w_stages, w_stays, tmem_cols; unsigned smem_bytes; };
bool plan_pair(const PairArgs& a, PairPlan* plan);       // false where the two do better, or only run, as kernels of their own
void launch_pair(const PairPlan& plan, const PairArgs& a, int* d_status, cudaStream_t st);

// First convolution (7x7 / stride 2 / pad 3, at most 3 input channels, ReLU) and the 3x3 / stride 2 / pad 1 max pooling
// behind it as one kernel that reads the NCHW network input  and writes the pooled tensor.
struct StemPoolArgs {
    const void* x;        // network input, N x C x H x W, NCHW, bf16 or fp32 (rounded to bf16 on load)
    void* y;              // pooled tensor, planar-8 with border, K_pad channels, N images
    const void* w;        // filters [16 taps (ta, tb)][2 chunks of 8][K_pad rows][8] bf16 over the parity channels, shifts included
                          // (PACK_STEM_DIRECT)
    int N, C, H, W, K_pad, in_f32;
    int n0, n_count;      // the images this launch handles (the tensor's plane pitch is that of all N)
};
struct StemPoolPlan { int valid, tmem_cols; unsigned smem_bytes; };
bool stem_pool_supported(int C, int H, int W, int K_pad);
int plan_stem_pool(const StemPoolArgs& a, StemPoolPlan* plan, char* err, size_t err_len);
void launch_stem_pool(const StemPoolPlan& plan, const StemPoolArgs& a, int* d_status, cudaStream_t st);

// A whole network of 3x3 convolutions on square images of 32, 16 or 8 pixels, from the NCHW input to the logits, as one
// kernel (resident_net.cu).  How its layers are placed and split depends on how many images a CTA carries (G) or how many
// CTAs share an image (cs): one plan per choice, the launch takes the cheapest for its batch.
enum { NET_STRIP = 0, NET_TILE = 1, NET_STRIDED = 2 };
constexpr int kNetUnits = 32;
constexpr int kNetMaxG = 2;                      // images a CTA carries at a time
constexpr int kNetSmemMax = 232448;              // opt-in dynamic shared memory per CTA,
constexpr int kNetCtrlBytes = 1920;              // of which the kernel's barriers and descriptors take this much, alignment included
struct NetUnit { uint16_t a_vec, dst_vec; uint8_t n8, nt, row, x; };   // a warp's piece of a layer: where its input and output start (vectors),
                                                 // first filter / 8, filters / 8, first output row and column
struct NetLayer {             // one layer as the kernel reads it (offsets and strides in bytes; buffers relative to an image's memory)
    int w_off, w_src, w_bytes, next;             // filters: place in shared memory, place in `w`, size; next: first layer to request behind this one
    int requests, req_off, req_src, req_bytes;   // how many to request, the first one's w_off, w_src, w_bytes
    int form, units, res_mode, zero_bytes;       // form | input channels / 16 << 8 | rows of a piece << 16 | width 8 << 24; clear that much of the output first (bit 0: begin together)
    int in_off, out_off, w_addr, bias_addr;
    int row_step, k_step, b_k, b_tap;            // input row, 16 input channels, filters of 16 channels, of a tap
    int out_plane, out_pitch, out_slab, relu;
    int a_chunk, a_px8, a_px, R;                 // a chunk, pixels 8-15 of a tile, a pixel of the input; output rows per CTA
    int res_plane, res_pitch, res_pad_lo, res_C;
    int res_off, W, n8, pad_;
    NetUnit unit[kNetUnits];
};
struct NetSpecLayer { int chunks, n8, stride, relu, res_mode, res_pad_lo, res_C, Hin, Win, blob_off, blob_bytes; };
struct NetSpec { std::vector<NetSpecLayer> layers; };
struct NetPlan {
    int G = 0, cs = 0, warps = 8, img_bytes = 0, act_bytes = 0, head_off = 0, last_off = 0, last_PV = 0, first_requests = 0;
    unsigned smem_bytes = 0;
    double cycles = 0;        // what the layers of one image take by the planner's estimate of each
    std::vector<NetLayer> table;
};
struct NetArgs {
    const void* x;            // network input, N x in_C x H x W, NCHW; in_mode 1: fp32, 2: bf16
    float* logits;
    const void* w;            // blobs of all layers
    const float *fcw, *fcb;   // FC matrix [class][fc_pitch] scaled by 1 / (H * W) of the last tensor; fcb may be nullptr
    void* dump;               // diagnostic: planar-8 tensor with border that layer dump_layer's output is written to
    int N, H, W, in_C, in_mode, n_classes, fc_pitch, last_H, last_W, last_chunks, dump_layer;
    int other_barrier;        // diagnostic (fp_debug_expire_wait): 1: CTA 1 of a cluster counts border rows on the wrong one of the two barriers, and
    long long wait_cycles;    // every wait gives up after this many SM clock cycles; 0: a normal launch
};
int net_blob_bytes(int chunks, int n8);
bool net_layer_supported(int H, int W, int P, int Q, int C_pad, int K, int stride);
bool plan_net(const NetSpec& spec, int G, int cs, int warps, NetPlan* plan);
bool prepare_net();              // lets the kernel have that much shared memory; false where the device refuses
int net_at_once(int cs);
void launch_net(const NetPlan& plan, const NetArgs& a, const NetLayer* d_table, int* d_status, cudaStream_t st);

// A run of stride-1 3x3 convolutions executed by one kernel with the activations in shared memory.
constexpr int kChainMaxLayers = 40;
struct ChainLayer {
    int cchunks;          // input channels / 8
    int K_pad;            // output channels, multiple of 16, <= 80
    int relu;
    int res;              // 1: add the tensor two layers back (the one this layer overwrites in place)
    int blob_off;         // byte offset of the layer's filter blob (filters, then K_pad fp32 biases) in `w`
    int blob_bytes;
};
struct ChainArgs {
    const void* x;        // input of the first layer (global): planar-8 with border, or, with in_mode 1 / 2, the
                          // network input itself: N x in_C x H x W, NCHW, fp32 / bf16 (rounded to bf16 on load)
    void* y;              // output of the last layer, same layout
    const void* res;      // shortcut operand of the FIRST layer (global) or nullptr
    const void* w;        // filter blobs of all layers
    int N, H, W, n_layers;
    int in_mode, in_C;
    int res_mode;         // first layer: 0 none, 1 same shape as its output, 2 subsample + zero-channel pad
    int res_H, res_W, res_C_pad, res_C, res_pad_lo, res_stride;
    ChainLayer layers[kChainMaxLayers];
};
struct ChainPlan {
    int valid;
    int quad;             // 1: 2 x 2 pixels a row of the GEMM (chain_quad.cu); of the rest then G, tiles, plane_rows and smem_bytes
    int G;                // images per group (per CTA at a time)
    int tiles;            // 128-position tiles per group
    int plane_rows;       // vectors per channel chunk of an activation buffer
    int buf_bytes, wbuf_bytes, acc_cols, tmem_cols;
    int stages;           // accumulator stages in tensor memory (ring)
    int issuers;          // MMA-issuing warps (each owns stages/issuers accumulator stages)
    int split;            // epilogue groups per tile (1, 2, 4): each takes every split-th channel chunk
    unsigned smem_bytes;
};
int chain_layer_blob_bytes(int cchunks, int K_pad);
bool chain_layer_supported(int H, int W, int K_pad, int C_pad);
int plan_chain_tc(const ChainArgs& a, ChainPlan* plan, char* err, size_t err_len);
void launch_chain_tc(const ChainPlan& plan, const ChainArgs& a, int* d_status, cudaStream_t st);
// The same for layers of 16 filters on images 32 pixels wide (chain_quad.cu): filters of a layer [4 x 4 window pixels][2 chunks][4 outputs x
// 16 filters][8] bf16, then the 16 fp32 biases.
constexpr int kQuadFilterBytes = 16 * 2 * 64 * 16, kQuadBlobBytes = kQuadFilterBytes + 64;
bool chain_quad_supported(const ChainArgs& a);
int plan_chain_quad(const ChainArgs& a, ChainPlan* plan, char* err, size_t err_len);
double chain_quad_layer_us(int tiles);         // a layer of a group of that many tiles
void launch_chain_quad(const ChainPlan& plan, const ChainArgs& a, int* d_status, cudaStream_t st);

}  // namespace fp
