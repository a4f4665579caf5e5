// Planning of the whole-network kernel (resident_net.cu): how every layer is split over the warps, and where the activations and
// filters of all layers lie in shared memory.  Host code without a CUDA call, so that it can be checked without a GPU.
#include "fp_internal.h"

#include <algorithm>
#include <vector>

namespace fp {

namespace {

struct NetGeom { int kc, n8, W, Win, R, stride, out_PV; };        // what a layer's split depends on

int up(int v, int m) { return (v + m - 1) / m * m; }

struct Span { int off, bytes, birth, death; };      // a piece of shared memory in use from layer `birth` to layer `death`

// Form and split of one layer over the warps of an image (eight; sixteen where an image has a CTA of that many to itself) (R: output rows of this CTA).
bool split_layer(NetLayer* e, const NetGeom& q, int warps, double* cycles) {
    const int kc = q.kc, n8 = q.n8, R = q.R, strips = q.W >= 16 ? q.W / 16 : 1;
    double best = 0;
    int form_ = 0, nt_ = 1, run_ = 1;
    auto offer = [&](int form, int nt, int run) {
        const int runs = (R + run - 1) / run, groups = (n8 + nt - 1) / nt, units = strips * runs * groups;
        if (units > kNetUnits) return;
        double tensor, shared;                              // cycles of a unit: one warp's MMAs, shared-memory reads
        if (form == NET_STRIP) {
            tensor = 9.0 * kc * nt * run * 8 + 150;
            shared = kc * (18.0 * nt + 12.0 * (run + 2)) + 16;
        } else if (form == NET_TILE) {
            const int mt = run / 2;
            tensor = 9.0 * kc * mt * nt * 8 + 150;
            shared = 3.0 * kc * (4 * (mt + 1) + 3 * (nt == 1 ? 2 : 4 * ((nt + 1) / 2)));
        } else {
            tensor = 9.0 * kc * nt * 8 + 150;
            shared = 9.0 * kc * (4 + 4 * ((nt + 1) / 2));
        }
        const int turns = (units + warps - 1) / warps;
        // units of one scheduler; a warp alone on it leaves the tensor pipe waiting for its loads
        const double busy = units >= warps ? warps / 4 * turns : units > 4 ? (units + 3) / 4 : 1.4;
        const double cost = std::max(busy * tensor * (n8 / (double)(groups * nt)), units * shared);
        if (best == 0 || cost < best * 0.999) { best = cost; form_ = form; nt_ = nt; run_ = run; }
    };
    if (q.stride == 2) {
        for (int nt = std::min(4, n8); nt >= 1; --nt) offer(NET_STRIDED, nt, q.W == 8 ? 2 : 1);
    } else if (q.W >= 16) {
        for (int run : {4, 2})
            for (int nt = std::min(2, n8); nt >= 1; --nt) if (R % run == 0) offer(NET_STRIP, nt, run);
    } else {
        for (int run : {4, 2})
            for (int nt = std::min(4, n8); nt >= 1; --nt) if (R % run == 0) offer(NET_TILE, nt, run);
    }
    *cycles += best;
    if (best == 0) return false;                            // more pieces than a layer's table holds
    const int runs = (R + run_ - 1) / run_, groups = (n8 + nt_ - 1) / nt_;
    e->form = form_ | kc << 8 | run_ << 16 | (q.W == 8 ? 1 : 0) << 24;
    e->units = strips * runs * groups;
    // filter groups outermost: a narrower last group then falls to the schedulers evenly
    int u = 0;
    for (int g = 0; g < groups; ++g)
        for (int s = 0; s < strips; ++s)
            for (int r = 0; r < runs; ++r, ++u) {
                const int row = r * run_, x = 16 * s;
                NetUnit& v = e->unit[u];
                v.a_vec = (uint16_t)(row * q.stride * (q.Win + 1) + x * q.stride);
                v.dst_vec = (uint16_t)(g * nt_ * q.out_PV + (row + 1) * (q.W + 1) + x + 1);
                v.n8 = (uint8_t)(g * nt_); v.nt = (uint8_t)std::min(nt_, n8 - g * nt_);
                v.row = (uint8_t)row; v.x = (uint8_t)x;
            }
    return true;
}

}  // namespace

// A layer's filters and shifts as they travel: [tap][chunk][filter][8] bf16, then fp32 shifts.
int net_blob_bytes(int chunks, int n8) { return 9 * chunks * n8 * 128 + n8 * 32; }

bool net_layer_supported(int H, int W, int P, int Q, int C_pad, int K, int stride) {
    if (H != W || P != Q || !(W == 8 || W == 16 || W == 32) || !(stride == 1 || stride == 2)) return false;
    if (Q != W / stride || Q < 8) return false;
    return C_pad % 16 == 0 && C_pad <= 64 && K >= 1 && K <= 64;
}

// Places the activations and every layer's filters in shared memory for groups of G images over cs CTAs.  Activations:
// tensors live from the layer that writes them to the last that reads them, a result with an identity shortcut takes the
// place of that operand; filters go where nothing is alive from the moment they are requested.  Returns false if it does
// not fit.
//
// Two images in a CTA (G = 2) are not at the same point.  Taking turns at the tensor pipe orders an image's results behind the
// other's reads of the layer before (a turn is given away behind the last of them), and filters are requested when both are through
// with a layer; but an image that has finished layer l goes on to clear the place of its next result, or to write the head's sums,
// while the other may not have begun to read layer l's filters.  So a layer that may write where the filters of the layer before
// lie begins when both images have ended that layer (bit 0 of zero_bytes), and the head's sums go over nothing that the last layer reads.
bool plan_net(const NetSpec& spec, int G, int cs, int warps, NetPlan* plan) {
    const int L = (int)spec.layers.size();
    plan->G = G; plan->cs = cs; plan->warps = warps;
    plan->table.assign(L, NetLayer());
    plan->first_requests = 0;
    plan->cycles = 0;
    struct Buf { int W, R, PV, chunks, birth, death, off; };
    std::vector<Buf> bufs;
    std::vector<int> buf_of(L + 1);                        // tensor (0 = network input, l + 1 = layer l's output) -> buffer
    auto make = [&](int W, int H, int chunks, int birth) -> int {
        if (H % cs) return -1;
        Buf b;
        b.W = W; b.R = H / cs; b.PV = (b.R + 2) * (W + 1) + 1; b.chunks = chunks; b.birth = birth; b.death = birth; b.off = -1;
        bufs.push_back(b);
        return (int)bufs.size() - 1;
    };
    if ((buf_of[0] = make(spec.layers[0].Win, spec.layers[0].Hin, spec.layers[0].chunks, -1)) < 0) return false;
    for (int l = 0; l < L; ++l) {
        const NetSpecLayer& s = spec.layers[l];
        const int W = s.Win / s.stride, H = s.Hin / s.stride;
        if (W == 8 && (H / cs) % 2) return false;          // an MMA's 16 pixels are two rows
        if (s.res_mode == 1) buf_of[l + 1] = buf_of[l - 1];
        else if ((buf_of[l + 1] = make(W, H, up(s.n8, 2), l)) < 0) return false;
        Buf& in = bufs[buf_of[l]];
        in.death = std::max(in.death, l);
        if (s.res_mode) bufs[buf_of[l - 1]].death = std::max(bufs[buf_of[l - 1]].death, l);
        bufs[buf_of[l + 1]].death = std::max(bufs[buf_of[l + 1]].death, l);
    }
    bufs[buf_of[L]].death = L;
    // one chunk count per geometry, so that buffers of a stage can follow one another without clearing borders
    for (Buf& b : bufs)
        for (const Buf& o : bufs) if (o.W == b.W) b.chunks = std::max(b.chunks, o.chunks);
    auto bytes_of = [](const Buf& b) { return b.chunks * b.PV * 16; };
    // first fit, but for the stream of the first stage, which is kept clear of the room that the second stage's two tensors
    // need: they are written while it is still read
    int second = 0;
    for (const Buf& b : bufs) if (b.W == bufs[0].W / 2) second = std::max(second, 2 * bytes_of(b));
    int img_bytes = 0;
    for (size_t i = 0; i < bufs.size(); ++i) {
        int at = i == 1 ? std::max(bytes_of(bufs[0]), second) : 0;
        for (bool moved = true; moved;) {
            moved = false;
            for (size_t j = 0; j < i; ++j)
                if (bufs[j].birth <= bufs[i].death && bufs[j].death >= bufs[i].birth && at < bufs[j].off + bytes_of(bufs[j]) &&
                    at + bytes_of(bufs[i]) > bufs[j].off) { at = bufs[j].off + bytes_of(bufs[j]); moved = true; }
        }
        bufs[i].off = at;
        img_bytes = std::max(img_bytes, at + bytes_of(bufs[i]));
    }
    plan->img_bytes = img_bytes;
    plan->act_bytes = G * img_bytes;
    const int room = kNetSmemMax - kNetCtrlBytes;
    if (plan->act_bytes > room || G > kNetMaxG) return false;
    std::vector<Span> spans;
    for (const Buf& b : bufs)
        for (int i = 0; i < G; ++i) spans.push_back({i * img_bytes + b.off, bytes_of(b), b.birth, b.death});
    // the activations' memory is cleared while the first layers' filters already come in
    spans.push_back({0, plan->act_bytes, -1, 0});
    // Where a piece can go so that it can be requested earliest (behind layer `after`, not before `floor`).  Few places are
    // different ones and few spans still alive; going through all of both for every layer took 5 ms for a network of 109.
    std::vector<int> ends;                                  // distinct places behind a span, in the spans' order
    auto add_end = [&](const Span& s) {
        const int c = up(s.off + s.bytes, 128);
        if (std::find(ends.begin(), ends.end(), c) == ends.end()) ends.push_back(c);
    };
    for (const Span& s : spans) add_end(s);
    std::vector<int> cand;
    std::vector<Span> alive;
    auto place = [&](int bytes, int birth_floor, int death, int* off, int* after) {
        int best_after = 1 << 30, best_off = 0;
        cand.assign(1, 0);
        cand.insert(cand.end(), ends.begin(), ends.end());
        cand.push_back(up(plan->act_bytes, 128));
        alive.clear();
        for (const Span& s : spans)
            if (s.death > birth_floor && s.birth <= death) alive.push_back(s);
        for (int c : cand) {
            if (c + bytes > room) continue;
            int a = birth_floor;
            bool ok = true;
            for (const Span& s : alive) {
                if (c >= s.off + s.bytes || c + bytes <= s.off || s.birth > death) continue;
                if (s.death >= death) { ok = false; break; }
                a = std::max(a, s.death);
            }
            if (!ok) continue;
            // nothing may move in between the request and the use
            for (const Span& s : alive)
                if (c < s.off + s.bytes && c + bytes > s.off && s.death > a) ok = false;
            if (ok && a < best_after) { best_after = a; best_off = c; }
        }
        if (best_after >= death) return false;
        *off = best_off; *after = best_after;
        return true;
    };
    struct Format { int off, bytes, PV; };
    std::vector<Format> formats;                            // what the borders in memory are zero for
    int prev_after = -1;
    for (int l = 0; l < L; ++l) {
        const NetSpecLayer& s = spec.layers[l];
        NetLayer& e = plan->table[l];
        const Buf &in = bufs[buf_of[l]], &out = bufs[buf_of[l + 1]];
        NetGeom q;
        q.kc = s.chunks / 2; q.n8 = s.n8; q.stride = s.stride; q.W = out.W; q.Win = in.W; q.R = out.R; q.out_PV = out.PV;
        if (!split_layer(&e, q, warps, &plan->cycles)) return false;
        e.in_off = in.off; e.out_off = out.off; e.R = out.R; e.W = out.W; e.n8 = s.n8; e.res_mode = s.res_mode;
        e.row_step = (in.W + 1) * 16; e.k_step = 2 * in.PV * 16;
        e.b_k = 2 * s.n8 * 128; e.b_tap = q.kc * e.b_k;
        e.out_plane = out.PV * 16; e.out_pitch = (out.W + 1) * 16; e.out_slab = out.R * e.out_pitch; e.relu = s.relu;
        e.a_chunk = in.PV * 16; e.a_px8 = out.W == 8 ? s.stride * e.row_step : 8 * s.stride * 16; e.a_px = s.stride * 16;
        e.res_pad_lo = s.res_pad_lo; e.res_C = s.res_C;
        if (s.res_mode) { const Buf& r = bufs[buf_of[l - 1]]; e.res_off = r.off; e.res_plane = r.PV * 16; e.res_pitch = (r.W + 1) * 16; }
        if (bytes_of(out) / 16 > 65535 || bytes_of(in) / 16 > 65535) return false;
        e.w_src = s.blob_off; e.w_bytes = s.blob_bytes;
        int after;
        // (a fragment load of an odd last group reaches 128 bytes behind the filters)
        if (!place(s.blob_bytes + 128, std::max(-1, l - 3), l, &e.w_off, &after)) return false;
        after = std::max(after, prev_after);                // requests are in order
        if (after >= l) return false;
        prev_after = after;
        e.w_addr = e.w_off; e.bias_addr = e.w_off + s.blob_bytes - s.n8 * 32;
        if (after < 0) ++plan->first_requests;
        else {
            NetLayer& f = plan->table[after];
            if (f.requests++ == 0) { f.req_off = e.w_off; f.req_src = e.w_src; f.req_bytes = e.w_bytes; f.next = l; }
        }
        spans.push_back({e.w_off, s.blob_bytes + 128, after + 1, l});
        add_end(spans.back());
        // Borders: everything is cleared before the first layer; a buffer of another geometry than what its place held (or
        // whose place held filters in between) is cleared by the layer that writes it first.
        if (s.res_mode != 1) {
            bool clean = l < 1;
            for (const Format& f : formats) clean |= f.off == out.off && f.PV == out.PV && f.bytes == bytes_of(out);
            if (!clean) e.zero_bytes = bytes_of(out);
            std::vector<Format> left;
            for (const Format& f : formats)
                if (f.off + f.bytes <= out.off || out.off + bytes_of(out) <= f.off) left.push_back(f);
            left.push_back({out.off, bytes_of(out), out.PV});
            if (l == 0) left.push_back({in.off, bytes_of(in), in.PV});
            formats = left;
        }
        if (G > 1 && l > 0) {
            const NetLayer& before = plan->table[l - 1];
            const int bytes = std::max(e.zero_bytes, s.n8 * e.out_plane);
            for (int i = 0; i < G; ++i) {
                const int at = i * img_bytes + out.off;
                if (at < before.w_off + before.w_bytes + 128 && at + bytes > before.w_off) e.zero_bytes |= 1;
            }
        }
        // filters that went over an activation buffer's place unformat it
        std::vector<Format> left;
        for (const Format& f : formats) {
            bool hit = false;
            for (int i = 0; i < G; ++i)
                hit |= e.w_off < i * img_bytes + f.off + f.bytes && e.w_off + s.blob_bytes + 128 > i * img_bytes + f.off;
            if (!hit) left.push_back(f);
        }
        formats = left;
    }
    {   // the head's sums: rows, then pooled channels
        const Buf& last = bufs[buf_of[L]];
        const int H = last.R * cs, C = spec.layers[L - 1].n8 * 8;
        int after;
        if (!place(G * (H + 1) * C * 4, L - 2, L, &plan->head_off, &after) || (G > 1 && after > L - 2)) return false;
        plan->last_off = last.off; plan->last_PV = last.PV;
    }
    int top = plan->act_bytes;
    for (const Span& s : spans) top = std::max(top, s.off + s.bytes);
    top = std::max(top, plan->head_off + G * (bufs[buf_of[L]].R * cs + 1) * spec.layers[L - 1].n8 * 32);
    plan->smem_bytes = (unsigned)(kNetCtrlBytes + top);
    return true;
}

}  // namespace fp
