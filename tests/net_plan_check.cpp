// Goes through a plan of the whole-network kernel (net_plan.cpp) layer by layer with a tag for every 16 bytes of a CTA's memory: what
// lies there when it is read has to be what was put there for that read.  Written from what the kernel does, not from the planner.
//
// What the order of events leaves open is taken the worse way, in turn: filters land as soon as they may be requested or at the last
// moment; of two images in a CTA either one is ahead.  How far ahead: an image clears the place of its next result (or writes the
// head's sums) as soon as it has finished its own layer, while the other one may not have begun to read that layer's filters - unless
// the next layer begins with both images (bit 0 of its zero_bytes).  Results are written behind the turn, which the other image gives
// away only behind its last read.
#include "../paper_2010_16165_b200/csrc/fp_internal.h"

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <vector>

using namespace fp;

namespace {

int up(int v, int m) { return (v + m - 1) / m * m; }

struct Sim {
    const NetSpec& spec;
    const NetPlan& plan;
    int L, late, ahead;                  // ahead: the image that leads
    std::vector<int> tag;                // 0 zero, t + 1 tensor t, -(l + 1) filters of layer l, 1 << 20 head's sums of an image
    std::vector<int> landed;
    char* msg;
    bool bad = false;

    void fail(int l, int s, const char* what) {
        if (!bad) snprintf(msg, 200, "layer %d image %d (late %d, ahead %d): %s", l, s, late, ahead, what);
        bad = true;
    }
    void fill(int off, int bytes, int t) {
        for (int i = off / 16; i < (off + bytes + 15) / 16; ++i) tag[i] = t;
    }
    void land(int l) {
        if (landed[l]) return;
        landed[l] = 1;
        fill(plan.table[l].w_off, plan.table[l].w_bytes, -(l + 1));
    }
    // the filters requested behind layer `after` (-1: at the start)
    void request(int after) {
        const int first = after < 0 ? 0 : plan.table[after].next, n = after < 0 ? plan.first_requests : plan.table[after].requests;
        for (int k = 0; k < n; ++k) if (!late) land(first + k);
    }
    void clear(int s, int l) {
        const NetLayer& e = plan.table[l];
        if (e.zero_bytes >> 4) fill(s * plan.img_bytes + e.out_off, e.zero_bytes & ~15, 0);
    }
    // a tensor of C8 chunks, R rows of W pixels: interior tagged `t` (chunks from `n8` on: anything but filters), border zero
    void expect(int l, int s, int off, int plane, int R, int W, int chunks, int n8, int t, int step) {
        for (int c = 0; c < chunks; ++c)
            for (int r = -1; r <= R; ++r)
                for (int w = -1; w <= W; ++w) {
                    const int v = tag[(off + c * plane) / 16 + (r + 1) * (W + 1) + w + 1];
                    const bool halo = r < 0 || r == R, border = w < 0 || w == W;
                    if (border || (halo && plan.cs == 1)) { if (v != 0) return fail(l, s, "border of an input not zero"); }
                    else if (halo) { if (v < 0) return fail(l, s, "filters in a halo row"); }
                    else if (r % step == 0 && w % step == 0 && (c < n8 ? v != t : v < 0)) return fail(l, s, "input overwritten");
                }
    }
    void layer(int s, int l) {
        const NetLayer& e = plan.table[l];
        const NetSpecLayer& q = spec.layers[l];
        const int img = s * plan.img_bytes, R_in = q.Hin / plan.cs;
        if (late) land(l);
        for (int i = e.w_off / 16; i < (e.w_off + e.w_bytes) / 16; ++i)
            if (tag[i] != -(l + 1)) { fail(l, s, "filters overwritten"); break; }
        expect(l, s, img + e.in_off, e.a_chunk, R_in, q.Win, q.chunks, l ? spec.layers[l - 1].n8 : 1, l + 1, 1);
        if (q.res_mode == 1) expect(l, s, img + e.out_off, e.out_plane, e.R, e.W, q.n8, q.n8, l, 1);
        if (q.res_mode == 2) expect(l, s, img + e.res_off, e.res_plane, e.R * 2, e.W * 2, (q.res_C + 7) / 8, (q.res_C + 7) / 8, l, 2);
        for (int c = 0; c < e.n8; ++c)
            for (int r = 0; r < e.R; ++r)
                for (int w = 0; w < e.W; ++w) tag[(img + e.out_off + c * e.out_plane) / 16 + (r + 1) * (e.W + 1) + w + 1] = l + 2;
        if (l + 1 < L && plan.cs > 1) {
            // a neighbour one layer ahead sends border rows of the next layer's result while this one's filters are still read
            const NetLayer& f = plan.table[l + 1];
            for (int c = 0; c < f.n8 && l + 2 < L && !f.zero_bytes; ++c)
                for (int r : {0, f.R + 1}) {
                    const int at = img + f.out_off + c * f.out_plane + r * (f.W + 1) * 16;
                    if (at < e.w_off + e.w_bytes && at + (f.W + 1) * 16 > e.w_off) fail(l, s, "a halo row of the next result in the filters' place");
                }
        }
    }
    int head_bytes() const { return (spec.layers[L - 1].Hin / spec.layers[L - 1].stride + 1) * spec.layers[L - 1].n8 * 32; }
    void head(int s) {
        const NetLayer& e = plan.table[L - 1];
        fill(plan.head_off + s * head_bytes(), head_bytes(), (1 << 20) + s);
        if (plan.head_off < s * plan.img_bytes + plan.last_off + e.n8 * e.out_plane && plan.head_off + plan.G * head_bytes() > s * plan.img_bytes + plan.last_off)
            fail(L, s, "the head's sums over the last tensor");
    }
    bool run() {
        L = (int)spec.layers.size();
        tag.assign((kNetSmemMax - kNetCtrlBytes) / 16 + 16, 7777);
        landed.assign(L, 0);
        if ((int)plan.smem_bytes > kNetSmemMax) fail(-1, 0, "more shared memory than there is");
        fill(0, plan.act_bytes, 0);
        request(-1);
        for (int s = 0; s < plan.G; ++s) {
            const NetLayer& e = plan.table[0];
            for (int r = 0; r < spec.layers[0].Hin / plan.cs; ++r)
                for (int w = 0; w < spec.layers[0].Win; ++w) tag[(s * plan.img_bytes + e.in_off) / 16 + (r + 1) * (spec.layers[0].Win + 1) + w + 1] = 1;
        }
        const int first = plan.G > 1 ? ahead : 0, second = 1 - first;
        for (int l = 0; l < L && !bad; ++l) {
            const bool together = plan.table[l].zero_bytes & 1;
            if (plan.G == 1) {
                clear(0, l);
                layer(0, l);
            } else {
                if (l == 0 || together) clear(first, l);      // (else it was cleared while the other image was a layer behind)
                layer(first, l);
                const bool next_together = l + 1 < L && (plan.table[l + 1].zero_bytes & 1);
                if (l + 1 < L && !next_together) clear(first, l + 1);
                if (l + 1 == L) head(first);
                clear(second, l);
                layer(second, l);
            }
            request(l);
        }
        if (!bad) head(plan.G > 1 ? second : 0);
        for (int s = 0; s < plan.G && !bad; ++s)
            for (int i = 0; i < head_bytes() / 16; ++i)
                if (tag[(plan.head_off + s * head_bytes()) / 16 + i] != (1 << 20) + s) { fail(L, s, "the head's sums overwritten"); break; }
        return !bad;
    }
};

}  // namespace

// A CIFAR-shaped network of basic blocks (`per_stage` blocks in every stage, stages of widths[] filters, the first on hw x hw pixels),
// keep[i] filters of convolution i kept where it is the first of a block.  0: fine, 1: no plan, -1: a fault, described in `msg`.
extern "C" int check_net_plan(int hw, int stages, const int* widths, int per_stage, const int* keep, int G, int cs, int warps, int meet_off, char* msg) {
    NetSpec spec;
    int off = 0, conv = 1, C = widths[0], H = hw;
    auto layer = [&](int C_in, int K, int stride, int H_in, int res_mode, int res_C) {
        NetSpecLayer l;
        memset(&l, 0, sizeof(l));
        l.chunks = up(C_in, 16) / 8; l.n8 = (K + 7) / 8; l.stride = stride; l.relu = 1; l.res_mode = res_mode; l.res_C = res_C;
        l.Hin = l.Win = H_in;
        l.blob_off = off; l.blob_bytes = net_blob_bytes(l.chunks, l.n8);
        off += up(l.blob_bytes, 128);
        spec.layers.push_back(l);
    };
    layer(3, C, 1, H, 0, 0);
    for (int s = 0; s < stages; ++s)
        for (int b = 0; b < per_stage; ++b, conv += 2) {
            const int stride = b == 0 && s > 0 ? 2 : 1;
            layer(C, keep[conv], stride, H, 0, 0);
            H /= stride;
            layer(keep[conv], widths[s], 1, H, stride == 2 ? 2 : 1, C);
            C = widths[s];
        }
    NetPlan plan;
    if (!plan_net(spec, G, cs, warps, &plan)) return 1;
    if (meet_off) for (NetLayer& e : plan.table) e.zero_bytes &= ~1;
    for (int late = 0; late < 2; ++late)
        for (int ahead = 0; ahead < G; ++ahead) {
            Sim sim{spec, plan, 0, late, ahead, {}, {}, msg};
            if (!sim.run()) return -1;
        }
    return 0;
}
