// The stage object and the C ABI: layer range -> execution units, arenas (parameters,
// activation slots, gradient workspace), and the per-call launch sequences.
#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/asteroid.h"
#include "kernels.h"
#include "pw_mma.h"
#include "replay.h"

namespace ast {

static thread_local std::string g_err;

static int fail(int code, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

int report_error(int code, const char* msg) { return fail(code, "%s", msg); }

#define CU(call)                                                                                     \
    do {                                                                                             \
        cudaError_t e_ = (call);                                                                     \
        if (e_ != cudaSuccess) return fail(AST_ERR_CUDA, "%s: %s", #call, cudaGetErrorString(e_));   \
    } while (0)

enum { U_CONV = 0, U_DW = 1, U_ADD = 2, U_GAP = 3, U_SILU = 4, U_SE = 5 };
enum { G_NONE = 0, G_ALIAS = 1, G_OWNED = 2 };

static size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

struct Val {
    int h = 0, w = 0, c = 0;
    size_t elems = 0;       // per micro-batch
    int unit = -1;          // producing unit, -1: the stage input
    size_t buf_off = 0;     // bytes into a slot: raw tensor (conv output / add or pool output / copy of x)
    bool affine = false;    // BatchNorm applied while loading
    int act = ACT_NONE;     // activation applied while loading
    size_t stat_off = 0;    // floats into a slot's statistics area: mean, rstd, scale, shift (c each)
    size_t grad_off = 0;    // bytes into the gradient workspace
    int consumers = 0;
    int first_cons = -1;    // lowest-index consuming unit: the last one to run in the backward pass, so the
                            // kernel that writes its input gradient writes the value's complete gradient
};

struct Unit {
    int kind = U_CONV;
    int l_main = -1, l_bn = -1, l_act = -1;
    int act = ACT_NONE;
    int in = -1, in2 = -1, out = -1;
    ConvGeom g{};
    long w_off = -1, b_off = -1, gamma_off = -1, beta_off = -1;   // floats into the parameter arena
    size_t k_off = 0;       // floats into the backward-coefficient arena (k1,k2,k3)
    size_t run_off = 0;     // floats into the running-statistics arena
    size_t acc_off = 0;     // 3x3 and 5x5 depthwise units: the weight gradient's accumulators, [taps][c], in the backward sums
    size_t sum_off = 0;     // BatchNorm units: channels before this unit's (its sums: 2c at 2*sum_off, its pivots at sum_off)
    // dense conv with a short reduction, bfloat16 mode: forward and weight gradient run as pointwise tensor-core GEMMs
    // over an explicit im2col tensor kept in the slot (col_kp = padded reduction length, 0 = not such a unit)
    int col_kp = 0;
    size_t col_off = 0;     // bytes into a slot
    long sub_off = -1;      // bytes into a slot: the input of a stride-2 1x1 conv sampled at the positions the conv reads
    size_t wpad_off = 0;    // elements into the padded bf16 weight arena
    // stride-2 3x3 conv on the stride-1 tensor-core kernels: bytes into the arena of zero-inserted output gradients (one
    // buffer per such unit: the weight-gradient kernel reads it on the second stream while the pass goes on), -1 = none
    long up_off = -1;
    // squeeze-excite: hidden width, floats into a slot's statistics area of the saved vectors (s [B][c], p1 [B][k], gate [B][c]),
    // floats into the backward-coefficient arena of its work vectors (B*(3c+k))
    int se_k = 0;
    size_t se_off = 0, se_work_off = 0;
};

// Arenas of a stage carry a guard band of GUARD bytes of a fixed pattern on both sides.  With the environment variable
// ASTEROID_CHECK_GUARDS=1 export_state reads the bands back and reports an arena whose band was overwritten (an
// out-of-bounds write of some kernel) as AST_ERR_CUDA.  The check runs on the host, between rounds.
constexpr size_t GUARD = 256;
constexpr unsigned char GUARD_BYTE = 0xA5;
struct Arena {
    char* base;
    size_t bytes;      // payload bytes (the guards lie at base and base + GUARD + bytes)
    const char* name;
};

struct Timing {
    bool on = false;
    std::vector<cudaEvent_t> ev;    // per unit: f0 f1 f2 b0 b1 b2
};

}  // namespace ast

using namespace ast;

struct asteroid_stage {
    std::vector<ast_layer> net;
    int first = 0, last = 0, in_h = 0, in_w = 0, B = 0, M = 0, dtype = 0, slots = 0, need_dx = 1;
    float eps = 1e-5f, bn_mom = 0.1f;
    size_t esz = 4;
    std::vector<Val> vals;          // vals[0] = stage input
    std::vector<Unit> units;
    std::vector<int> val_of_layer;  // layer index - (first-1) -> value id or -1
    // n_params: values of the caller's flat state (layers back to back); n_pad: floats of the internal parameter arenas, where
    // every layer starts on a multiple of 8 floats (16-byte aligned in the bfloat16 copies, whatever precedes it)
    size_t n_params = 0, n_pad = 0, n_run = 0, n_coef = 0, n_bn_ch = 0, n_bsum = 0, n_dw_weights = 0;
    struct Seg { size_t pub, in, n; };
    std::vector<Seg> segs;
    // device arenas
    float *w = nullptr, *v = nullptr, *G = nullptr, *g = nullptr, *derived = nullptr, *run = nullptr, *coef = nullptr, *scratch = nullptr;
    RefreshSeg* dense = nullptr;                   // how the derived weights come about (plan_refresh)
    int32_t* rest = nullptr;
    int n_dense = 0, tiles = 0, n_rest = 0;
    __nv_bfloat16 *wb = nullptr, *wtb = nullptr;   // bf16 copies of the weights and of the derived (transposed) weights
    __nv_bfloat16* wpad = nullptr;                 // [co][Kp] bf16 weights of the im2col units
    float* gpad = nullptr;                         // [co][Kp] padded weight gradient of the im2col unit at hand
    size_t n_wpad = 0, n_gpad = 0;
    // per-channel sums of the BatchNorms' forward (fin.cuh) and the pivots they were taken with.  The backward's lie in the slot, together with the
    // accumulators of the depthwise weight gradients.  A forward's first kernel zeroes both, so that a backward starts from zero
    // whatever ran on the stage before its forward: calls that an import dropped, a replay of a captured round.  Accumulate zeroes the
    // backward's again, for graphs of a caller's own that hold a backward and its accumulate without the forward.
    char* fsum = nullptr;
    float* pivots = nullptr;
    DwSettle* dw_tab = nullptr;                    // the depthwise units' accumulators and weight gradients
    int n_dw = 0;
    int* err = nullptr;                            // device error word (bounded waits)
    // Weight-gradient kernels depend only on the BatchNorm-backward coefficients of their unit and nothing in the rest of
    // the backward pass depends on them: they run on a second stream (forked from and joined back into the caller's
    // stream inside each backward call), with their own split-sum scratch, and fill the gaps of the dependent chain.
    std::vector<Replay> replays;
    uint64_t rounds = 0;                           // updates so far
    cudaStream_t cap = nullptr;                    // calls are captured on it
    cudaStream_t side = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    float* scratch_side = nullptr;
    char* up_mem = nullptr;                        // zero-inserted gradients of the stride-2 3x3 units
    size_t up_bytes = 0;
    char *slot_mem = nullptr, *grad_mem = nullptr;
    size_t slot_bytes = 0, slot_stat_off = 0, slot_bsum_off = 0, grad_bytes = 0, scratch_floats = 0;
    size_t bytes_mod = 0, bytes_opt = 0, bytes_work = 0;
    // round state
    std::vector<int> slot_of_mb, mb_of_slot;
    int pending_g = -1, n_acc = 0;
    int pending_slot = -1;                         // where that backward's sums lie
    std::vector<char> sums_left;                   // per slot: its backward failed on the way and may have left sums behind
    Timing tm;
    std::vector<ast::Arena> arenas;                // every device allocation of the stage, with its guard bands
    bool check_guards = false;
    std::vector<asteroid_stage*> prof_cache;
    std::vector<std::vector<double>> prof_ms;   // per cached stage: 4 per unit (f_main, f_bn, b_bn, b_main)
    // what the last forward / backward did, per unit: statistics partials written by the producing kernel (their count, 0 =
    // standalone pass); unit whose backward-data kernel took this unit's BatchNorm-backward sums (-1 = standalone pass)
    std::vector<int> fwd_stats_blocks, bwd_sums_by;
    std::vector<char> add_deferred;                // ... residual sums that the pointwise layer behind formed
};

namespace ast {

static float* g_loss_scratch[64] = {};
static int loss_scratch(float** out) {
    int dev = 0;
    CU(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(AST_ERR_ARG, "device index %d out of range", dev);
    if (!g_loss_scratch[dev]) {
        CU(cudaMalloc(&g_loss_scratch[dev], (65536 + 64) * sizeof(float)));
        CU(cudaMemset(g_loss_scratch[dev], 0, (65536 + 64) * sizeof(float)));
    }
    *out = g_loss_scratch[dev];
    return AST_OK;
}

static int n_layer_params(const ast_layer& L) {
    switch (L.op) {
        case AST_CONV: return L.c_out * L.k * L.k * L.c_in;
        case AST_DWCONV: return L.c_out * L.k * L.k;
        case AST_BN: return 2 * L.c_out;
        case AST_LINEAR: return L.c_out * L.c_in + L.c_out;
        case AST_SE: return 2 * L.k * L.c_out + L.k + L.c_out;
        default: return 0;
    }
}

static bool is_act(int op) { return op == AST_RELU6 || op == AST_RELU; }

// Parse layers [first,last] into fused units; fill values, geometry and parameter offsets.
static int build_plan(asteroid_stage* s) {
    const auto& net = s->net;
    const int first = s->first, last = s->last;
    const int vecw = s->dtype == AST_F32 ? 4 : 8;
    std::vector<long> poff(net.size(), -1);
    long off = 0, pub = 0;
    for (int i = first; i <= last; ++i) {
        const long n = n_layer_params(net[i]);
        poff[i] = off;
        if (n) s->segs.push_back({(size_t)pub, (size_t)off, (size_t)n});
        pub += n;
        off = (off + n + 7) / 8 * 8;
    }
    s->n_params = (size_t)pub;
    s->n_pad = (size_t)off;
    s->val_of_layer.assign(last - first + 2, -1);
    auto vol = [&](int layer) -> int& { return s->val_of_layer[layer - (first - 1)]; };

    Val in;
    in.h = s->in_h; in.w = s->in_w; in.c = net[first].c_in;
    in.elems = (size_t)s->B * in.h * in.w * in.c;
    s->vals.push_back(in);
    vol(first - 1) = 0;

    auto resolve = [&](int layer, int at, int* out) -> int {
        if (layer < first - 1 || layer >= at) return fail(AST_ERR_ARG, "layer %d reads layer %d, outside the stage [%d,%d]", at, layer, first, last);
        int v = vol(layer);
        if (v < 0) return fail(AST_ERR_UNSUPPORTED, "layer %d reads layer %d, an intermediate of a fused conv-BN-activation chain", at, layer);
        *out = v;
        return AST_OK;
    };

    int i = first;
    while (i <= last) {
        const ast_layer& L = net[i];
        Unit u;
        u.l_main = i;
        int rc;
        if (L.op == AST_CONV || L.op == AST_DWCONV || L.op == AST_LINEAR) {
            if ((rc = resolve(L.src, i, &u.in))) return rc;
            const Val& x = s->vals[u.in];
            if (x.c != L.c_in) return fail(AST_ERR_ARG, "layer %d: c_in %d but its input has %d channels", i, L.c_in, x.c);
            u.kind = L.op == AST_DWCONV ? U_DW : U_CONV;
            ConvGeom& g = u.g;
            g.n = s->B; g.hi = x.h; g.wi = x.w; g.ci = L.c_in; g.co = L.c_out;
            if (L.op == AST_LINEAR) {
                if (x.h != 1 || x.w != 1) return fail(AST_ERR_UNSUPPORTED, "layer %d: linear needs a 1x1 spatial input (put a gap before it)", i);
                g.k = 1; g.stride = 1; g.pad = 0;
                u.b_off = poff[i] + (long)L.c_out * L.c_in;
            } else {
                g.k = L.k; g.stride = L.stride; g.pad = L.pad;
                if (g.k < 1 || g.stride < 1 || g.pad < 0) return fail(AST_ERR_ARG, "layer %d: bad k/stride/pad", i);
            }
            if (L.op == AST_DWCONV) {
                if ((L.k != 3 && L.k != 5 && L.k != 7) || L.pad != (L.k - 1) / 2 || L.c_in != L.c_out || (L.stride != 1 && L.stride != 2))
                    return fail(AST_ERR_UNSUPPORTED, "layer %d: depthwise conv must be 3x3, 5x5 or 7x7 with pad (k-1)/2 and stride 1 or 2", i);
                if (L.c_in % vecw) return fail(AST_ERR_UNSUPPORTED, "layer %d: depthwise channels must be a multiple of %d", i, vecw);
            }
            g.ho = (g.hi + 2 * g.pad - g.k) / g.stride + 1;
            g.wo = (g.wi + 2 * g.pad - g.k) / g.stride + 1;
            if (g.ho < 1 || g.wo < 1) return fail(AST_ERR_ARG, "layer %d: empty output", i);
            u.w_off = poff[i];
            int j = i + 1;
            if (j <= last && net[j].op == AST_BN && net[j].src == i) {
                if (net[j].c_out != L.c_out) return fail(AST_ERR_ARG, "layer %d: BN channel count mismatch", j);
                u.l_bn = j;
                u.gamma_off = poff[j];
                u.beta_off = poff[j] + L.c_out;
                ++j;
            }
            if (j <= last && is_act(net[j].op) && net[j].src == j - 1) {
                u.l_act = j;
                u.act = net[j].op == AST_RELU6 ? ACT_RELU6 : ACT_RELU;
                ++j;
            }
            Val o;
            o.h = g.ho; o.w = g.wo; o.c = g.co;
            o.affine = u.l_bn >= 0;
            o.act = u.act;
            o.unit = (int)s->units.size();
            o.elems = (size_t)s->B * o.h * o.w * o.c;
            u.out = (int)s->vals.size();
            s->vals.push_back(o);
            vol(j - 1) = u.out;
            i = j;
        } else if (L.op == AST_ADD) {
            if ((rc = resolve(L.src, i, &u.in))) return rc;
            if ((rc = resolve(L.add_from, i, &u.in2))) return rc;
            const Val &a = s->vals[u.in], &b = s->vals[u.in2];
            if (a.h != b.h || a.w != b.w || a.c != b.c) return fail(AST_ERR_ARG, "layer %d: add operands differ in shape", i);
            u.kind = U_ADD;
            int j = i + 1;
            if (j <= last && is_act(net[j].op) && net[j].src == i) {
                if (net[j].op != AST_RELU) return fail(AST_ERR_UNSUPPORTED, "layer %d: only ReLU may follow an add", j);
                u.l_act = j;
                u.act = ACT_RELU;
                ++j;
            }
            Val o;
            o.h = a.h; o.w = a.w; o.c = a.c;
            o.unit = (int)s->units.size();
            o.elems = a.elems;
            u.out = (int)s->vals.size();
            s->vals.push_back(o);
            vol(j - 1) = u.out;
            i = j;
        } else if (L.op == AST_SILU || L.op == AST_SE) {
            // materialising units: the value they read keeps its on-load BatchNorm; their own output is a plain stored tensor
            if ((rc = resolve(L.src, i, &u.in))) return rc;
            const Val& a = s->vals[u.in];
            if (a.c != L.c_in || L.c_in != L.c_out) return fail(AST_ERR_ARG, "layer %d: channel count %d does not match its input's %d", i, L.c_in, a.c);
            if (L.op == AST_SE) {
                if (L.k < 1 || L.k > 1024) return fail(AST_ERR_ARG, "layer %d: squeeze width must be in [1,1024]", i);
                if (a.c > 8192) return fail(AST_ERR_UNSUPPORTED, "layer %d: squeeze-excite takes at most 8192 channels", i);
                u.kind = U_SE;
                u.se_k = L.k;
                u.w_off = poff[i];
                u.g.n = s->B; u.g.hi = u.g.ho = a.h; u.g.wi = u.g.wo = a.w; u.g.ci = u.g.co = a.c;
            } else {
                u.kind = U_SILU;
            }
            Val o;
            o.h = a.h; o.w = a.w; o.c = a.c;
            o.unit = (int)s->units.size();
            o.elems = a.elems;
            u.out = (int)s->vals.size();
            s->vals.push_back(o);
            vol(i) = u.out;
            i = i + 1;
        } else if (L.op == AST_GAP) {
            if ((rc = resolve(L.src, i, &u.in))) return rc;
            const Val& a = s->vals[u.in];
            u.kind = U_GAP;
            Val o;
            o.h = 1; o.w = 1; o.c = a.c;
            o.unit = (int)s->units.size();
            o.elems = (size_t)s->B * o.c;
            u.out = (int)s->vals.size();
            s->vals.push_back(o);
            vol(i) = u.out;
            i = i + 1;
        } else {
            return fail(AST_ERR_UNSUPPORTED, "layer %d: a BN or activation must directly follow the conv (or add) it belongs to", i);
        }
        for (int vin : {u.in, u.in2}) {
            if (vin < 0) continue;
            Val& iv = s->vals[vin];
            iv.consumers++;
            if (iv.first_cons < 0) iv.first_cons = (int)s->units.size();
        }
        s->units.push_back(u);
    }
    for (size_t v = 0; v + 1 < s->vals.size(); ++v)
        if (v > 0 && s->vals[v].consumers == 0) return fail(AST_ERR_UNSUPPORTED, "an intermediate value of the stage is never used");
    if (vol(last) != (int)s->vals.size() - 1) return fail(AST_ERR_UNSUPPORTED, "the stage output must be the output of its last layer");

    // slot layout, gradient workspace, coefficient and running-statistics arenas
    size_t sb = 0, gb = 0, nstat = 0, ncoef = 0, nrun = 0;
    for (auto& v : s->vals) {
        v.buf_off = sb;
        sb += align_up(v.elems * s->esz, 256);
        v.grad_off = gb;
        gb += align_up(v.elems * s->esz, 256);
    }
    for (auto& u : s->units) {
        const int K = u.g.k * u.g.k * u.g.ci;
        if (u.kind == U_CONV && s->dtype == AST_BF16 && u.g.k > 1 && K <= 64 && u.g.co % 8 == 0 && u.g.co <= 256 && u.b_off < 0) {
            u.col_kp = (K + 15) / 16 * 16;
            u.col_off = sb;
            sb += align_up((size_t)u.g.n * u.g.ho * u.g.wo * u.col_kp * 2, 256);
            u.wpad_off = s->n_wpad;
            s->n_wpad += (size_t)u.g.co * u.col_kp;
            s->n_gpad = std::max(s->n_gpad, (size_t)u.g.co * u.col_kp);
        }
    }
    // A 1x1 conv with stride 2 reads one input position in four: the forward copies those positions into a dense tensor kept
    // in the slot, and the forward and the weight gradient then run the stride-1 pointwise pipelines on it.
    for (auto& u : s->units) {
        if (u.kind == U_CONV && s->dtype == AST_BF16 && u.g.k == 1 && u.g.stride == 2 && u.g.pad == 0 && u.g.ci % 8 == 0 && u.g.co % 8 == 0 &&
            u.b_off < 0 && !u.col_kp) {
            u.sub_off = (long)sb;
            sb += align_up((size_t)u.g.n * u.g.ho * u.g.wo * u.g.ci * 2, 256);
        }
    }
    s->slot_stat_off = sb;
    for (auto& u : s->units) {
        if (u.l_bn >= 0) {
            Val& o = s->vals[u.out];
            o.stat_off = nstat;
            nstat += 4 * (size_t)o.c;
            u.k_off = ncoef;
            ncoef += 3 * (size_t)o.c;
            u.run_off = nrun;
            nrun += 2 * (size_t)o.c;
            u.sum_off = s->n_bn_ch;
            s->n_bn_ch += align_up((size_t)o.c, 4);   // kernels read and write pivots in vectors
        }
    }
    s->n_bsum = 2 * s->n_bn_ch;
    for (auto& u : s->units)
        if (u.kind == U_DW && u.g.k <= 5) {
            const size_t weights = (size_t)u.g.k * u.g.k * u.g.ci;
            u.acc_off = s->n_bsum;
            s->n_bsum += weights;
            s->n_dw_weights += weights;
            ++s->n_dw;
        }
    for (auto& u : s->units)
        if (u.kind == U_SE) {
            u.se_off = nstat;
            nstat += (size_t)s->B * (2 * (size_t)u.g.ci + u.se_k);
            u.se_work_off = ncoef;
            ncoef += (size_t)s->B * (3 * (size_t)u.g.ci + u.se_k);
        }
    s->slot_bsum_off = align_up(sb + nstat * sizeof(float), 256);
    s->slot_bytes = align_up(s->slot_bsum_off + chan_sums_bytes(s->n_bsum), 256);
    s->grad_bytes = gb;
    s->n_coef = ncoef;
    s->n_run = nrun;
    return AST_OK;
}

// How the derived weights come from the weights: dense layers turned tile by tile, everything else by (destination, source) lists.
static void plan_refresh(const asteroid_stage* s, std::vector<RefreshSeg>& segs, int* tiles, std::vector<int32_t>& rest) {
    std::vector<int32_t> src(s->n_pad);
    for (size_t i = 0; i < src.size(); ++i) src[i] = (int32_t)i;
    *tiles = 0;
    for (const auto& u : s->units) {
        const ConvGeom& g = u.g;
        const int taps = g.k * g.k;
        if (u.kind == U_CONV) {          // derived: wt[c][r][s][ko] <- w[ko][r][s][c]
            segs.push_back(RefreshSeg{(size_t)u.w_off, g.co, g.ci, taps, *tiles});
            *tiles += ((g.ci + 31) / 32) * ((g.co + 31) / 32) * taps;
            std::fill(src.begin() + u.w_off, src.begin() + u.w_off + (size_t)g.co * taps * g.ci, -1);
        } else if (u.kind == U_DW) {     // derived: tap-major wkc[t][c] <- w[c][t]
            for (int c = 0; c < g.ci; ++c)
                for (int t = 0; t < taps; ++t) src[u.w_off + (size_t)t * g.ci + c] = (int32_t)(u.w_off + (size_t)c * taps + t);
        }
    }
    for (size_t i = 0; i < src.size(); ++i)
        if (src[i] >= 0) rest.push_back((int32_t)i);
    const size_t n = rest.size();
    for (size_t i = 0; i < n; ++i) rest.push_back(src[rest[i]]);
}

static void free_stage(asteroid_stage* s) {
    if (!s) return;
    for (auto* p : s->prof_cache) free_stage(p);
    for (auto e : s->tm.ev) cudaEventDestroy(e);
    for (const Arena& a : s->arenas) cudaFree(a.base);
    if (s->ev_fork) cudaEventDestroy(s->ev_fork);
    if (s->ev_join) cudaEventDestroy(s->ev_join);
    for (Replay& r : s->replays)
        if (r.exec) cudaGraphExecDestroy(r.exec);
    if (s->cap) cudaStreamDestroy(s->cap);
    if (s->side) cudaStreamDestroy(s->side);
    delete s;
}


template <typename P> static int arena_alloc(asteroid_stage* s, const char* name, P** p, size_t bytes, size_t* tally);

template <typename P> static int dev_alloc(P** p, size_t bytes, size_t* tally) {
    if (bytes == 0) bytes = 256;
    cudaError_t e = cudaMalloc((void**)p, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(AST_ERR_ALLOC, "cudaMalloc of %zu bytes failed: %s", bytes, cudaGetErrorString(e));
    }
    e = cudaMemset(*p, 0, bytes);
    if (e != cudaSuccess) return fail(AST_ERR_CUDA, "cudaMemset: %s", cudaGetErrorString(e));
    *tally += bytes;
    return AST_OK;
}

template <typename P> static int arena_alloc(asteroid_stage* s, const char* name, P** p, size_t bytes, size_t* tally) {
    if (bytes == 0) bytes = 256;
    bytes = align_up(bytes, 256);
    char* base = nullptr;
    cudaError_t e = cudaMalloc((void**)&base, bytes + 2 * GUARD);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(AST_ERR_ALLOC, "cudaMalloc of %zu bytes (%s) failed: %s", bytes, name, cudaGetErrorString(e));
    }
    s->arenas.push_back(Arena{base, bytes, name});
    e = cudaMemset(base, GUARD_BYTE, GUARD);
    if (e == cudaSuccess) e = cudaMemset(base + GUARD, 0, bytes);
    if (e == cudaSuccess) e = cudaMemset(base + GUARD + bytes, GUARD_BYTE, GUARD);
    if (e != cudaSuccess) return fail(AST_ERR_CUDA, "cudaMemset: %s", cudaGetErrorString(e));
    *p = reinterpret_cast<P*>(base + GUARD);
    *tally += bytes + 2 * GUARD;
    return AST_OK;
}

static int check_guards(asteroid_stage* s) {
    unsigned char h[2 * GUARD];
    for (const Arena& a : s->arenas) {
        CU(cudaMemcpy(h, a.base, GUARD, cudaMemcpyDeviceToHost));
        CU(cudaMemcpy(h + GUARD, a.base + GUARD + a.bytes, GUARD, cudaMemcpyDeviceToHost));
        for (size_t i = 0; i < 2 * GUARD; ++i)
            if (h[i] != GUARD_BYTE)
                return fail(AST_ERR_CUDA, "guard band of arena '%s' overwritten %s the arena (byte %zu)", a.name, i < GUARD ? "before" : "after", i % GUARD);
    }
    return AST_OK;
}

static int reset_bn_running(asteroid_stage* s) {
    if (!s->n_run) return AST_OK;
    std::vector<float> h(s->n_run, 0.f);
    for (const auto& u : s->units)
        if (u.l_bn >= 0)
            for (int c = 0; c < u.g.co; ++c) h[u.run_off + u.g.co + c] = 1.f;
    CU(cudaMemcpy(s->run, h.data(), h.size() * sizeof(float), cudaMemcpyHostToDevice));
    return AST_OK;
}

// derived weight copies of every kind, after the master weights changed
static void refresh_weights(asteroid_stage* s, cudaStream_t st) {
    refresh_derived(s->w, s->dense, s->n_dense, s->tiles, s->rest, s->n_rest, s->derived, s->wb, s->wtb, s->n_pad, st);
    for (const auto& u : s->units)
        if (u.col_kp) conv_pad_weights(s->w + u.w_off, u.g.co, u.g.k * u.g.k * u.g.ci, u.col_kp, s->wpad + u.wpad_off, st);
}

// A stride-2 3x3 conv (pad 1, bfloat16, channel counts the stride-1 tensor-core kernels take) runs on those kernels:
// forward as the stride-1 conv on the input grid followed by a 2x subsampling, backward-data as the stride-1 input
// gradient of the zero-inserted output gradient.  Four times the multiply-adds of the direct form, on tensor cores
// instead of FFMA.  Both need one full-resolution tensor in the scratch arena.
static ConvGeom s1_geom(const Unit& u) {
    ConvGeom g = u.g;
    g.ho = u.g.hi; g.wo = u.g.wi; g.stride = 1;
    return g;
}
static bool conv3_s2_tc_supported(const asteroid_stage* s, const Unit& u) {
    if (s->dtype != AST_BF16 || u.kind != U_CONV || u.g.k != 3 || u.g.stride != 2 || u.g.pad != 1) return false;
    if (!conv3_tc_supported(s->dtype, s1_geom(u))) return false;
    const size_t full = (size_t)u.g.n * u.g.hi * u.g.wi * std::max(u.g.ci, u.g.co) * 2;
    return full <= s->scratch_floats * sizeof(float);
}

static double conv_flops(const ConvGeom& g) { return 2.0 * g.n * g.ho * g.wo * (double)g.co * g.k * g.k * g.ci; }

// geometry of the pointwise GEMM that stands for an im2col unit
// stride-2 1x1 conv on its subsampled input: a stride-1 conv over the output grid
static ConvGeom sub_geom(const Unit& u) {
    ConvGeom g = u.g;
    g.hi = u.g.ho; g.wi = u.g.wo; g.stride = 1;
    return g;
}
static ConvGeom col_geom(const Unit& u) {
    ConvGeom g = u.g;
    g.hi = u.g.ho; g.wi = u.g.wo; g.ci = u.col_kp; g.k = 1; g.stride = 1; g.pad = 0;
    return g;
}

// ---------------------------------------------------------------------------------------------
struct SlotView {
    char* base;
    float* stats;
    char* bsum;
};

static SlotView slot_view(asteroid_stage* s, int slot) {
    char* b = s->slot_mem + (size_t)slot * s->slot_bytes;
    return SlotView{b, reinterpret_cast<float*>(b + s->slot_stat_off), b + s->slot_bsum_off};
}

static ValSrc val_src(asteroid_stage* s, const SlotView& sv, int v) {
    const Val& a = s->vals[v];
    ValSrc r;
    r.p = sv.base + a.buf_off;
    r.scale = a.affine ? sv.stats + a.stat_off + 2 * (size_t)a.c : nullptr;
    r.shift = a.affine ? sv.stats + a.stat_off + 3 * (size_t)a.c : nullptr;
    r.act = a.act;
    return r;
}

static void tick(asteroid_stage* s, size_t unit, int which, cudaStream_t st) {
    if (s->tm.on) cudaEventRecord(s->tm.ev[unit * 6 + which], st);
}

// ---- BatchNorm coefficients that are still sums (fin.cuh)
static ChanSums fsums(const asteroid_stage* s) { return chan_sums(s->fsum, 2 * s->n_bn_ch, false); }
static ChanSums bsums(const asteroid_stage* s, const SlotView& sv) { return chan_sums(sv.bsum, s->n_bsum, true); }
static BnFwdOut fwd_out(asteroid_stage* s, const SlotView& sv, const Unit& u) {
    const Val& o = s->vals[u.out];
    float* stt = sv.stats + o.stat_off;
    return BnFwdOut{stt, stt + o.c, stt + 2 * (size_t)o.c, stt + 3 * (size_t)o.c, s->run + u.run_off, s->run + u.run_off + o.c};
}
static BnBwdOut bwd_out(asteroid_stage* s, const Unit& u) {
    float* kc = s->coef + u.k_off;
    const size_t c = (size_t)s->vals[u.out].c;
    return BnBwdOut{s->g + u.gamma_off, s->g + u.beta_off, kc, kc + c, kc + 2 * c};
}
static BnPendFwd pend_fwd(asteroid_stage* s, const SlotView& sv, const Unit& u) {
    const Val& o = s->vals[u.out];
    const double n = (double)(o.elems / o.c);
    return BnPendFwd{fsums(s) + 2 * u.sum_off, s->pivots + u.sum_off, s->w + u.gamma_off, s->w + u.beta_off, 1.0 / n, n > 1.0 ? n / (n - 1.0) : 1.0,
                     s->eps, s->bn_mom, o.c, fwd_out(s, sv, u)};
}
static BnPendBwd pend_bwd(asteroid_stage* s, const SlotView& sv, const Unit& u) {
    const Val& o = s->vals[u.out];
    const float* stt = sv.stats + o.stat_off;
    return BnPendBwd{bsums(s, sv) + 2 * u.sum_off, s->w + u.gamma_off, stt, stt + o.c, 1.0 / (double)(o.elems / o.c), o.c, bwd_out(s, u)};
}
static BnSumsOut sums_fwd(asteroid_stage* s, const Unit& u) { return BnSumsOut{fsums(s) + 2 * u.sum_off, s->run + u.run_off, s->pivots + u.sum_off}; }

// which BatchNorm units' coefficients are pending in the pass at hand
struct Pending {
    asteroid_stage* s;
    SlotView sv;
    cudaStream_t st;
    std::vector<char> unit;
    Pending(asteroid_stage* s_, const SlotView& v, cudaStream_t st_) : s(s_), sv(v), st(st_), unit(s_->units.size(), 0) {}
    bool has(int u) const { return u >= 0 && unit[u] != 0; }
    // the unit's pending coefficients for a kernel that forms them itself (nothing is pending afterwards); empty if none are
    BnPendFwd take_fwd(int u) {
        if (!has(u)) return BnPendFwd{};
        unit[u] = 0;
        return pend_fwd(s, sv, s->units[u]);
    }
    void settle_fwd(int u) {
        if (has(u)) bn_settle_fwd(take_fwd(u), st);
    }
    void settle_bwd(int u) {
        if (has(u)) bn_settle_bwd(pend_bwd(s, sv, s->units[u]), st);
        if (u >= 0) unit[u] = 0;
    }
};

// Pointwise problem of a unit on the register-operand kernels; false: it does not run there.
static bool mma_unit(const asteroid_stage* s, const ConvGeom& g, bool bwd, MmaTiling* t) {
    if (s->dtype != AST_BF16 || g.k != 1 || g.stride != 1 || g.pad != 0) return false;
    return bwd ? mma_choose(true, g.n * g.ho * g.wo, g.co, g.ci, t) : mma_choose(false, g.n * g.ho * g.wo, g.ci, g.co, t);
}

// ... and on the float32 ones
static bool f32_unit(const asteroid_stage* s, const Unit& u, bool bwd, F32Tiling* t) {
    const ConvGeom& g = u.g;
    if (s->dtype != AST_F32 || u.kind != U_CONV || g.k != 1 || g.stride != 1 || g.pad != 0) return false;
    return bwd ? f32_choose(true, g.n * g.ho * g.wo, g.co, g.ci, t) : f32_choose(false, g.n * g.ho * g.wo, g.ci, g.co, t);
}

// A residual sum of two tensors without activations of their own, read next by a pointwise layer on the register-operand or float32
// kernels: that layer forms it as it loads, and writes it out for the others.  Up to 4 M elements, where the sum is mostly a launch in the chain (a
// round of a sixth of MobileNetV2 at batch 4 1681 -> 1647 us, of small images 1469 -> 1440); beyond, where every CTA of that layer takes all of its columns and has a reduction
// long enough to request several steps ahead (pw_mma.cu): each operand is then read once, and the sum not again.  In front of 256 -> 64, pass and layer 40.9 -> 28.5 us at 57 000 pixels,
// 61.6 -> 39.3 at 100 352.  ResNet stage at batch 32, with such requests in all persistent layers: no large sum left to the layer behind 19 871 us a round, all of them 19 651, those of
// 12.8 M elements in front of 512 -> 128 alone, whose columns take three CTAs, 20 055.
// The value is the elementwise pass's: beyond 4 M elements to the bit, up to there but for the shifts, which are added first.
static bool small_sum(const Val& sum) { return sum.elems <= (size_t)4 << 20; }
static bool defers_add(const asteroid_stage* s, size_t ui) {
    const Unit& u = s->units[ui];
    if (ui + 1 >= s->units.size()) return false;
    const Unit& v = s->units[ui + 1];
    MmaTiling t{};
    F32Tiling t32;
    if (v.kind != U_CONV || v.in != u.out || v.col_kp || v.sub_off >= 0) return false;
    if (u.in == u.in2 || s->vals[u.in].act != ACT_NONE || s->vals[u.in2].act != ACT_NONE) return false;
    const bool mma = mma_unit(s, v.g, false, &t);
    return small_sum(s->vals[u.out]) ? mma || f32_unit(s, v, false, &t32) : mma && 8 * t.nj >= v.g.co && mma_deep_sum(v.g.n * v.g.ho * v.g.wo, v.g.ci, t);
}

static int forward_impl(asteroid_stage* s, int slot, const void* x, void* y, cudaStream_t st) {
    SlotView sv = slot_view(s, slot);
    const int dt = s->dtype;
    {
        // the slot's copy of x (backward reads it); a kernel rather than a memcpy node where the alignment allows vector
        // accesses, so that the chain of programmatic dependent launches is not interrupted.  It also zeroes the channel sums of
        // this forward and of its backward.
        const Val& v0 = s->vals[0];
        if (!slot_copy(x, sv.base + v0.buf_off, v0.elems * s->esz, fsums(s), 2 * s->n_bn_ch, bsums(s, sv), s->n_bsum, st)) {
            CU(cudaMemcpyAsync(sv.base + v0.buf_off, x, v0.elems * s->esz, cudaMemcpyDeviceToDevice, st));
            if (s->n_bn_ch) CU(cudaMemsetAsync(s->fsum, 0, chan_sums_bytes(2 * s->n_bn_ch), st));
            if (s->n_bsum) CU(cudaMemsetAsync(sv.bsum, 0, chan_sums_bytes(s->n_bsum), st));
        }
    }
    Pending pend(s, sv, st);
    int deferred = -1;             // a residual sum left to the pointwise layer behind it
    int squeeze_splits = 0;        // > 0: the unit before left the squeeze of this one as that many partials in the scratch arena
    const auto producer = [&](int v) { return s->vals[v].affine ? s->vals[v].unit : -1; };
    for (size_t ui = 0; ui < s->units.size(); ++ui) {
        const Unit& u = s->units[ui];
        const Val& o = s->vals[u.out];
        const bool is_last = ui + 1 == s->units.size();
        void* obuf = sv.base + o.buf_off;
        tick(s, ui, 0, st);
        int fused_stats = 0;       // > 0: the producing kernel wrote that many statistics partials into the scratch arena; -1: it took the sums
        const bool bn = u.l_bn >= 0;
        MmaTiling til;
        F32Tiling til32;
        // the pointwise layer on the register-operand kernels: forms its input's pending coefficients, takes its output's sums
        auto on_mma = [&](const ConvGeom& g, const ValSrc& xs, int in_unit, const void* w) {
            MmaProblem p{};
            p.P = g.n * g.ho * g.wo; p.K = g.ci; p.N = g.co;
            p.x = xs; p.w = w; p.out = obuf;
            p.bias = u.b_off >= 0 ? s->w + u.b_off : nullptr;
            p.pf = pend.take_fwd(in_unit);
            if (deferred >= 0) {
                const Unit& au = s->units[deferred];
                p.x2 = val_src(s, sv, au.in2);
                p.pf2 = pend.take_fwd(producer(au.in2));
                p.sum_out = sv.base + s->vals[au.out].buf_off;
                p.sum_act = au.act;
                p.sum_large = !small_sum(s->vals[au.out]);
                deferred = -1;
            }
            if (bn) p.so = sums_fwd(s, u);
            const double elems = (double)p.P * p.K + (double)p.P * p.N + (double)p.N * p.K;
            if (dt == AST_F32) f32_launch(false, p, til32, K_CONV_FWD, 4.0 * elems, st);
            else mma_launch(false, p, til, K_PW_FWD_TC, 2.0 * elems, st);
            fused_stats = bn ? -1 : 0;
        };
        if (u.kind == U_CONV && !u.col_kp && u.sub_off < 0 && mma_unit(s, u.g, false, &til)) {
            const int from = deferred >= 0 ? s->units[deferred].in : u.in;
            on_mma(u.g, val_src(s, sv, from), producer(from), s->wb + u.w_off);
        } else if (f32_unit(s, u, false, &til32)) {
            const int from = deferred >= 0 ? s->units[deferred].in : u.in;
            on_mma(u.g, val_src(s, sv, from), producer(from), s->w + u.w_off);
        } else if (u.kind == U_CONV) {
            pend.settle_fwd(producer(u.in));
            const float* bias = u.b_off >= 0 ? s->w + u.b_off : nullptr;
            if (u.col_kp) {
                void* col = sv.base + u.col_off;
                conv_im2col(u.g, val_src(s, sv, u.in), u.col_kp, col, st);
                const ValSrc cs{col, nullptr, nullptr, ACT_NONE};
                if (mma_unit(s, col_geom(u), false, &til)) on_mma(col_geom(u), cs, -1, s->wpad + u.wpad_off);
                else
                fused_stats = pw_fwd_tc(col_geom(u), cs, s->wpad + u.wpad_off, nullptr, obuf,
                                        bn ? s->run + u.run_off : nullptr, bn ? s->scratch : nullptr, s->scratch_floats, s->err, st);
            } else if (u.sub_off >= 0) {
                ValSrc xs = val_src(s, sv, u.in);
                void* sub = sv.base + u.sub_off;
                ew_subsample2(xs.p, u.g.n, u.g.hi, u.g.wi, u.g.ho, u.g.wo, u.g.ci, sub, st);
                xs.p = sub;                                  // the producer's BatchNorm / activation is per channel: applied on load as before
                if (mma_unit(s, sub_geom(u), false, &til)) on_mma(sub_geom(u), xs, -1, s->wb + u.w_off);
                else
                fused_stats = pw_fwd_tc(sub_geom(u), xs, s->wb + u.w_off, bias, obuf, bn ? s->run + u.run_off : nullptr,
                                        bn ? s->scratch : nullptr, s->scratch_floats, s->err, st);
            } else if (pw_tc_supported(dt, u.g))
                fused_stats = pw_fwd_tc(u.g, val_src(s, sv, u.in), s->wb + u.w_off, bias, obuf, bn ? s->run + u.run_off : nullptr,
                                        bn ? s->scratch : nullptr, s->scratch_floats, s->err, st);
            else if (conv3_tc_supported(dt, u.g)) conv3_fwd_tc(u.g, val_src(s, sv, u.in), s->wb + u.w_off, obuf, s->err, st);
            else if (conv3_s2_tc_supported(s, u)) {
                conv3_fwd_tc(s1_geom(u), val_src(s, sv, u.in), s->wb + u.w_off, s->scratch, s->err, st, conv_flops(u.g));
                ew_subsample2(s->scratch, u.g.n, u.g.hi, u.g.wi, u.g.ho, u.g.wo, u.g.co, obuf, st);
            }
            else conv_fwd(dt, u.g, val_src(s, sv, u.in), s->w + u.w_off, bias, obuf, st);
        } else if (u.kind == U_DW) {
            if (u.g.k > 5) {
                pend.settle_fwd(producer(u.in));
                dwk_fwd(dt, u.g, val_src(s, sv, u.in), s->derived + u.w_off, obuf, st);
            } else {
                const BnPendFwd pf = pend.take_fwd(producer(u.in));
                const BnSumsOut so = bn ? sums_fwd(s, u) : BnSumsOut{};
                if (u.g.k == 5) dw5_fwd(dt, u.g, val_src(s, sv, u.in), pf, s->derived + u.w_off, obuf, so, dw5_choose(dt, false, u.g), st);
                else dw3_fwd(dt, u.g, val_src(s, sv, u.in), pf, s->derived + u.w_off, obuf, so, dw3_choose(dt, false, u.g), st);
                fused_stats = bn ? -1 : 0;
            }
        } else if (u.kind == U_SILU) {
            // a squeeze-excite layer right behind: its squeeze comes with this pass
            const bool squeeze = o.consumers == 1 && ui + 1 < s->units.size() && s->units[ui + 1].kind == U_SE && s->units[ui + 1].in == u.out;
            const BnPendFwd pf = pend.take_fwd(producer(u.in));
            squeeze_splits = silu_fwd(dt, val_src(s, sv, u.in), pf, s->B, o.h * o.w, o.c, obuf, is_last ? y : nullptr, squeeze ? s->scratch : nullptr,
                                      s->scratch_floats, st);
        } else if (u.kind == U_SE) {
            pend.settle_fwd(producer(u.in));
            const int c = o.c, k = u.se_k;
            const float* wp = s->w + u.w_off;        // w1 [k][c], b1 [k], w2 [c][k], b2 [c]
            float* sev = sv.stats + u.se_off;        // s [B][c], p1 [B][k], gate [B][c]
            se_forward(dt, val_src(s, sv, u.in), s->B, o.h * o.w, c, k, wp, wp + (size_t)k * c, wp + (size_t)k * c + k, wp + 2 * (size_t)k * c + k, sev,
                       sev + (size_t)s->B * c, sev + (size_t)s->B * (c + k), s->scratch, s->scratch_floats, squeeze_splits, obuf, is_last ? y : nullptr, st);
            squeeze_splits = 0;
        } else if (u.kind == U_ADD && defers_add(s, ui)) {
            deferred = (int)ui;
            s->add_deferred[ui] = 1;
        } else if (u.kind == U_ADD) {
            if (!ew_takes_pending(dt, o.c)) {
                pend.settle_fwd(producer(u.in));
                pend.settle_fwd(producer(u.in2));
            }
            const BnPendFwd pa = pend.take_fwd(producer(u.in)), pb = pend.take_fwd(producer(u.in2));
            ew_add(dt, val_src(s, sv, u.in), val_src(s, sv, u.in2), pa, pb, u.act, o.elems / o.c, o.c, obuf, is_last ? y : nullptr, st);
        } else {
            const Val& a = s->vals[u.in];
            if (!gap_takes_pending(dt, a.c)) pend.settle_fwd(producer(u.in));
            const BnPendFwd pf = pend.take_fwd(producer(u.in));
            gap_fwd(dt, val_src(s, sv, u.in), pf, s->B, a.h * a.w, a.c, obuf, st);
        }
        tick(s, ui, 1, st);
        s->fwd_stats_blocks[ui] = fused_stats < 0 ? 1 : fused_stats;
        if (bn) {
            if (fused_stats > 0)
                bn_stats_finish_partials(s->scratch, fused_stats, o.elems / o.c, o.c, s->w + u.gamma_off, s->w + u.beta_off, s->eps, s->bn_mom,
                                         fwd_out(s, sv, u), st);
            else {
                if (fused_stats == 0) bn_stats(dt, obuf, o.elems / o.c, o.c, sums_fwd(s, u), s->scratch_floats, st);
                pend.unit[ui] = 1;
            }
        }
        tick(s, ui, 2, st);
        if (is_last) {
            if (!ew_takes_pending(dt, o.c)) pend.settle_fwd(producer(u.out));
            if (u.kind == U_CONV || u.kind == U_DW) ew_apply(dt, val_src(s, sv, u.out), pend.take_fwd(producer(u.out)), o.elems / o.c, o.c, y, st);
            else if (u.kind == U_GAP) CU(cudaMemcpyAsync(y, obuf, o.elems * s->esz, cudaMemcpyDeviceToDevice, st));
        }
    }
    CU(cudaGetLastError());
    return AST_OK;
}

struct GradState {
    int state = G_NONE;
    const void* ptr = nullptr;
};

// A squeeze-excite layer's backward left to the SiLU unit in front: its output gradient counts as dy*gate + ds there.
struct GatedGrad {
    const float *gate = nullptr, *ds = nullptr;
};

// The conv->BN unit whose BatchNorm-backward sums can be taken by the kernel that writes the complete gradient of
// value `v`: the unit that produced v, or, when v is a plain residual sum, the one operand branch that is used
// nowhere else (its gradient is the sum's gradient, by alias).  -1: none, or more than one.
static int bn_reduce_target(const asteroid_stage* s, int v) {
    const int p = s->vals[v].unit;
    if (p < 0) return -1;
    const Unit& pu = s->units[p];
    if (pu.kind == U_CONV || pu.kind == U_DW) return pu.l_bn >= 0 ? p : -1;
    if (pu.kind != U_ADD || pu.act != ACT_NONE) return -1;
    int target = -1, n = 0;
    for (int o : {pu.in, pu.in2}) {
        const Val& ov = s->vals[o];
        if (ov.consumers != 1 || ov.unit < 0) continue;
        const Unit& q = s->units[ov.unit];
        if ((q.kind == U_CONV || q.kind == U_DW) && q.l_bn >= 0) {
            target = ov.unit;
            ++n;
        }
    }
    return n == 1 ? target : -1;
}

static int backward_impl(asteroid_stage* s, int slot, const void* dy, void* dx, cudaStream_t st) {
    SlotView sv = slot_view(s, slot);
    const int dt = s->dtype;
    std::vector<GradState> gs(s->vals.size());
    auto own = [&](int v) -> void* { return v == 0 ? dx : (void*)(s->grad_mem + s->vals[v].grad_off); };
    auto pass = [&](int v, const void* src) {
        GradState& t = gs[v];
        if (t.state == G_NONE) {
            t.state = G_ALIAS;
            t.ptr = src;
        } else {
            ew_sum(dt, t.ptr, src, s->vals[v].elems, own(v), st);
            t.state = G_OWNED;
            t.ptr = own(v);
        }
    };
    gs.back().state = G_ALIAS;
    gs.back().ptr = dy;
    GatedGrad gated;
    std::vector<char> reduced(s->units.size(), 0);   // BatchNorm-backward sums already taken by the kernel that wrote dy
    Pending pend(s, sv, st);                         // ... and not yet turned into coefficients
    // The kernel that takes a unit's sums forms its activation's mask for them anyway.  Where it can it stores the gradient masked, and the two or three kernels
    // that read it are spared the mask, a third of their transform.
    std::vector<char> masked(s->units.size(), 0);
    std::fill(s->bwd_sums_by.begin(), s->bwd_sums_by.end(), -1);
    // weight gradients go to the second stream (not while a profile run times the units one by one, nor while a
    // per-launch trace brackets every kernel with events: a kernel's duration is then that of the kernel running alone)
    const bool use_side = s->side != nullptr && !s->tm.on && !tracing();
    bool side_used = false;
    cudaStream_t wst = use_side ? s->side : st;
    float* wscratch = use_side ? s->scratch_side : s->scratch;
    // What follows `on_side` on the second stream comes after everything that was on the caller's at the last `mark`.
    auto mark = [&]() -> int {
        if (use_side) CU(cudaEventRecord(s->ev_fork, st));
        return AST_OK;
    };
    auto on_side = [&]() -> int {
        if (!use_side) return AST_OK;
        CU(cudaStreamWaitEvent(s->side, s->ev_fork, 0));
        side_used = true;
        return AST_OK;
    };

    for (int ui = (int)s->units.size() - 1; ui >= 0; --ui) {
        const Unit& u = s->units[ui];
        const Val& o = s->vals[u.out];
        GradState& go = gs[u.out];
        const bool want_in = u.in != 0 || s->need_dx;
        tick(s, ui, 3, st);
        if (u.kind == U_CONV || u.kind == U_DW) {
            float* stt = sv.stats + o.stat_off;
            float* kc = s->coef + u.k_off;
            GradSrc d{};
            d.dy = go.ptr;
            d.z = sv.base + o.buf_off;
            d.act = masked[ui] ? ACT_NONE : u.act;
            if (u.l_bn >= 0) {
                if (!masked[ui]) {
                    d.scale = stt + 2 * (size_t)o.c;
                    d.shift = stt + 3 * (size_t)o.c;
                }
                if (!reduced[ui]) {
                    bn_bwd_reduce(dt, d.dy, d.z, o.elems / o.c, o.c, d.scale, d.shift, u.act, stt, stt + o.c, bsums(s, sv) + 2 * u.sum_off, s->scratch_floats, st);
                    pend.unit[ui] = 1;
                }
                d.k1 = kc; d.k2 = kc + o.c; d.k3 = kc + 2 * (size_t)o.c;
            }
            // pending coefficients stay pending where both kernels of the unit can form them
            MmaTiling til_d{};
            WgradTiling til_w{};
            ConvGeom wg = u.g;
            if (u.col_kp) wg = col_geom(u);
            else if (u.sub_off >= 0) wg = sub_geom(u);
            const bool pw = u.kind == U_CONV && dt == AST_BF16 && wg.k == 1 && wg.stride == 1 && wg.pad == 0;
            const bool mma_w = pw && wgrad_mma_choose(wg.n * wg.ho * wg.wo, wg.co, wg.ci, pw_wgrad_pipeline_fits(wg, grad_needs_z(d), s->scratch_floats),
                                                      s->scratch_floats, &til_w);
            const bool mma_d = want_in && u.kind == U_CONV && !u.col_kp && mma_unit(s, u.g, true, &til_d);
            F32Tiling til_d32{};
            F32WgradTiling til_w32{};
            const bool f32_d = want_in && f32_unit(s, u, true, &til_d32);
            const bool f32_w = u.kind == U_CONV && dt == AST_F32 && wg.k == 1 && wg.stride == 1 && wg.pad == 0 &&
                               f32_wgrad_choose(wg.n * wg.ho * wg.wo, wg.co, wg.ci, s->scratch_floats, &til_w32);
            const bool dw = u.kind == U_DW && u.g.k <= 5;
            if (!dw && ((!mma_w && !f32_w) || (want_in && !mma_d && !f32_d))) pend.settle_bwd(ui);
            const BnPendBwd pb = pend.has(ui) ? pend_bwd(s, sv, u) : BnPendBwd{};
            pend.unit[ui] = 0;
            tick(s, ui, 4, st);
            ValSrc xin = val_src(s, sv, u.in);
            if (dw) {
                // input gradient, weight gradient and, where x is the raw output of a conv -> BatchNorm unit read by nobody after this one, that
                // BatchNorm's sums
                GradState& gi = gs[u.in];
                const void* addend = gi.state == G_NONE ? nullptr : gi.ptr;
                const int tgt = want_in && s->vals[u.in].first_cons == ui && bn_reduce_target(s, u.in) == s->vals[u.in].unit ? s->vals[u.in].unit : -1;
                ChanSums sums{};
                const float* ts = nullptr;
                if (tgt >= 0) {
                    const Unit& tu = s->units[tgt];
                    sums = bsums(s, sv) + 2 * tu.sum_off;
                    ts = sv.stats + s->vals[tu.out].stat_off;
                    pend.unit[tgt] = 1;
                    reduced[tgt] = 1;
                    s->bwd_sums_by[tgt] = ui;
                }
                void* to = want_in ? own(u.in) : nullptr;
                const float* trs = ts ? ts + u.g.ci : nullptr;
                if (u.g.k == 5) dw5_bwd(dt, u.g, d, pb, xin, s->derived + u.w_off, addend, to, bsums(s, sv) + u.acc_off, sums, ts, trs, dw5_choose(dt, true, u.g), st);
                else {
                    if (tgt >= 0) masked[tgt] = s->units[tgt].act != ACT_NONE;
                    dw3_bwd(dt, u.g, d, pb, xin, s->derived + u.w_off, addend, to, bsums(s, sv) + u.acc_off, sums, ts, trs, tgt >= 0 && masked[tgt], dw3_choose(dt, true, u.g), st);
                }
                if (want_in) {
                    gi.state = G_OWNED;
                    gi.ptr = own(u.in);
                }
                tick(s, ui, 5, st);
                continue;
            }
            const bool s2_tc = u.kind == U_CONV && u.up_off >= 0;
            void* up = s2_tc ? s->up_mem + u.up_off : nullptr;
            // stride 2 on the stride-1 kernels: the zero-inserted output gradient (BatchNorm / activation backward applied
            // on the way) serves both the weight gradient and the input gradient
            if (s2_tc) ew_upsample2_grad(d, u.g.n, u.g.hi, u.g.wi, u.g.ho, u.g.wo, u.g.co, up, st);
            const GradSrc dup{up, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, ACT_NONE};
            if (int rc = mark()) return rc;
            const auto weights = [&]() -> int {
                if (int rc = on_side()) return rc;
                // a BatchNorm behind takes the bias out again with the mean: the gradient behind its backward sums to zero over the micro-batch
                if (u.b_off >= 0 && u.l_bn >= 0) CU(cudaMemsetAsync(s->g + u.b_off, 0, (size_t)o.c * sizeof(float), wst));
                else if (u.b_off >= 0) bias_grad(dt, d.dy, d.z, o.elems / o.c, o.c, u.act, wscratch, s->scratch_floats, s->g + u.b_off, wst);
                if (s2_tc && conv3_wgrad_tc_supported(dt, s1_geom(u)))
                    conv3_bwd_weight_tc(s1_geom(u), dup, xin, wscratch, s->scratch_floats, s->g + u.w_off, s->err, wst, conv_flops(u.g));
                else if (mma_w || f32_w) {
                    WgradProblem p{};
                    p.P = wg.n * wg.ho * wg.wo; p.CO = wg.co; p.CI = wg.ci;
                    p.dz = d; p.x = xin; p.pb = pb; p.pend_write = want_in ? 0 : 1;
                    if (u.col_kp) p.x = ValSrc{sv.base + u.col_off, nullptr, nullptr, ACT_NONE};
                    else if (u.sub_off >= 0) p.x.p = sv.base + u.sub_off;                  // written by the forward of this micro-batch
                    if (f32_w) f32_wgrad_launch(p, til_w32, wscratch, s->g + u.w_off, wst);
                    else wgrad_mma_launch(p, til_w, wscratch, u.col_kp ? s->gpad : s->g + u.w_off, wst);
                    if (u.col_kp) conv_unpad_grad(s->gpad, u.g.co, u.g.k * u.g.k * u.g.ci, u.col_kp, s->g + u.w_off, wst);
                } else if (u.kind == U_CONV && u.col_kp) {
                    pw_bwd_weight_tc(col_geom(u), d, ValSrc{sv.base + u.col_off, nullptr, nullptr, ACT_NONE}, wscratch, s->scratch_floats, s->gpad, s->err, wst);
                    conv_unpad_grad(s->gpad, u.g.co, u.g.k * u.g.k * u.g.ci, u.col_kp, s->g + u.w_off, wst);
                } else if (u.kind == U_CONV && u.sub_off >= 0) {
                    ValSrc xs = xin;
                    xs.p = sv.base + u.sub_off;                  // written by the forward of this micro-batch
                    pw_bwd_weight_tc(sub_geom(u), d, xs, wscratch, s->scratch_floats, s->g + u.w_off, s->err, wst);
                } else if (u.kind == U_CONV && pw_tc_supported(dt, u.g))
                    pw_bwd_weight_tc(u.g, d, xin, wscratch, s->scratch_floats, s->g + u.w_off, s->err, wst);
                else if (u.kind == U_CONV && conv3_wgrad_tc_supported(dt, u.g))
                    conv3_bwd_weight_tc(u.g, d, xin, wscratch, s->scratch_floats, s->g + u.w_off, s->err, wst);
                else if (u.kind == U_CONV) conv_bwd_weight(dt, u.g, d, xin, wscratch, s->scratch_floats, s->g + u.w_off, wst);
                else dwk_bwd_weight(dt, u.g, d, xin, wscratch, s->scratch_floats, s->g + u.w_off, wst);
                return AST_OK;
            };
            // The order of the two branches of a fork is the order a replayed graph places them in.  At the first fork the dependent chain goes first and so stays in
            // line with the kernel in front; second, its next kernel starts 3.4 us after that one has ended (a round of the smallest block in float32 270 ->
            // 264 us, of the ragged stage 640 -> 622, of a sixth of MobileNetV2 at batch 4 1497 -> 1475, EfficientNet 7135 -> 7070).  At the others, and at a first
            // one that begins the call, the weight gradients do: placed second they are scattered over streams of the graph's own and
            // lose their programmatic launches (half of MobileNetV2 with the head 4170 -> 4640 us).
            // On one stream (a trace, a profile) there is no fork: each layer's weight gradient in front of its input gradient.
            const bool chain_first = use_side && !side_used && (ui + 1 < (int)s->units.size() || u.l_bn >= 0);
            if (!chain_first)
                if (int rc = weights()) return rc;
            if (want_in) {
                GradState& gi = gs[u.in];
                const void* addend = gi.state == G_NONE ? nullptr : gi.ptr;
                // this kernel writes the complete gradient of its input value: let it also take the BatchNorm-backward
                // sums of the unit that gradient belongs to
                const int tgt = s->vals[u.in].first_cons == ui ? bn_reduce_target(s, u.in) : -1;
                if (mma_d || f32_d) {
                    MmaProblem p{};
                    BnRed red{};
                    p.P = u.g.n * u.g.ho * u.g.wo; p.K = u.g.co; p.N = u.g.ci;
                    p.dz = d; p.pb = pb; p.w = f32_d ? (const void*)(s->derived + u.w_off) : s->wtb + u.w_off; p.addend = addend; p.out = own(u.in);
                    if (tgt >= 0) {
                        const Unit& tu = s->units[tgt];
                        const Val& tv = s->vals[tu.out];
                        float* ts = sv.stats + tv.stat_off;
                        masked[tgt] = tgt == s->vals[u.in].unit && tu.act != ACT_NONE;      // through an alias the gradient is another value's too
                        red = BnRed{sv.base + tv.buf_off, ts + 2 * (size_t)tv.c, ts + 3 * (size_t)tv.c, ts, ts + tv.c, tu.act, nullptr, 0, masked[tgt] != 0};
                        p.red = &red;
                        p.so = BnSumsOut{bsums(s, sv) + 2 * tu.sum_off, nullptr, nullptr};
                        pend.unit[tgt] = 1;
                        reduced[tgt] = 1;
                        s->bwd_sums_by[tgt] = ui;
                    }
                    const double elems = (double)p.P * p.K * (grad_needs_z(d) ? 2.0 : 1.0) + (double)p.P * p.N * (addend ? 2.0 : 1.0) + (double)p.N * p.K;
                    if (f32_d) f32_launch(true, p, til_d32, K_CONV_BWD_DATA, 4.0 * elems, st);
                    else mma_launch(true, p, til_d, K_PW_BWD_DATA_TC, 2.0 * elems, st);
                } else if (u.kind == U_CONV && pw_tc_supported(dt, u.g)) {
                    BnRed red{};
                    if (tgt >= 0) {
                        const Unit& tu = s->units[tgt];
                        const Val& tv = s->vals[tu.out];
                        float* ts = sv.stats + tv.stat_off;
                        red = BnRed{sv.base + tv.buf_off, ts + 2 * (size_t)tv.c, ts + 3 * (size_t)tv.c, ts, ts + tv.c, tu.act, s->scratch, s->scratch_floats, false};
                    }
                    const int blocks = pw_bwd_data_tc(u.g, d, s->wtb + u.w_off, addend, own(u.in), tgt >= 0 ? &red : nullptr, s->err, st);
                    if (blocks > 0) {
                        const Unit& tu = s->units[tgt];
                        const Val& tv = s->vals[tu.out];
                        float* ts = sv.stats + tv.stat_off;
                        float* tk = s->coef + tu.k_off;
                        BnBwdOut tbo{s->g + tu.gamma_off, s->g + tu.beta_off, tk, tk + tv.c, tk + 2 * (size_t)tv.c};
                        bn_bwd_finish_partials(s->scratch, blocks, tv.elems / tv.c, tv.c, ts, ts + tv.c, s->w + tu.gamma_off, tbo, st);
                        reduced[tgt] = 1;
                        s->bwd_sums_by[tgt] = ui;
                    }
                } else if (u.kind == U_CONV && conv3_tc_supported(dt, u.g)) conv3_bwd_data_tc(u.g, d, s->wtb + u.w_off, addend, own(u.in), s->err, st);
                else if (s2_tc) conv3_bwd_data_tc(s1_geom(u), dup, s->wtb + u.w_off, addend, own(u.in), s->err, st, conv_flops(u.g));
                else if (u.kind == U_CONV) conv_bwd_data(dt, u.g, d, s->derived + u.w_off, addend, own(u.in), st);
                else dwk_bwd_data(dt, u.g, d, s->derived + u.w_off, addend, own(u.in), st);
                gi.state = G_OWNED;
                gi.ptr = own(u.in);
            }
            if (chain_first)
                if (int rc = weights()) return rc;
        } else if (u.kind == U_ADD) {
            tick(s, ui, 4, st);
            if (u.act == ACT_RELU) {
                // The masked gradient is the complete gradient of every operand used nowhere else.  If such an operand is
                // the output of a conv -> BatchNorm unit without activation, the mask kernel also takes that BatchNorm's
                // backward sums (one such operand: a second one keeps its own pass).
                int tgt = -1;
                for (int v : {u.in, u.in2}) {
                    const Val& ov = s->vals[v];
                    if (tgt >= 0 || ov.consumers != 1 || ov.unit < 0) continue;
                    const Unit& q = s->units[ov.unit];
                    if ((q.kind == U_CONV || q.kind == U_DW) && q.l_bn >= 0 && q.act == ACT_NONE && !reduced[ov.unit]) tgt = ov.unit;
                }
                bool fused = false;
                if (tgt >= 0) {
                    const Unit& tu = s->units[tgt];
                    const Val& tv = s->vals[tu.out];
                    float* ts = sv.stats + tv.stat_off;
                    fused = ew_relu_mask_bn_sums(dt, go.ptr, sv.base + o.buf_off, sv.base + tv.buf_off, o.elems / o.c, o.c, ts, ts + tv.c, own(u.out),
                                                 bsums(s, sv) + 2 * tu.sum_off, s->scratch_floats, st);
                    if (fused) {
                        pend.unit[tgt] = 1;
                        reduced[tgt] = 1;
                        s->bwd_sums_by[tgt] = ui;
                    }
                }
                if (!fused) ew_relu_mask(dt, go.ptr, sv.base + o.buf_off, o.elems, own(u.out), st);
                go.state = G_OWNED;
                go.ptr = own(u.out);
            }
            if (u.in != 0 || s->need_dx) pass(u.in, go.ptr);
            if (u.in2 != 0 || s->need_dx) pass(u.in2, go.ptr);
        } else if (u.kind == U_SILU || u.kind == U_SE) {
            tick(s, ui, 4, st);
            GradState& gi = gs[u.in];
            const void* addend = gi.state == G_NONE ? nullptr : gi.ptr;
            if (u.kind == U_SE) {
                // the parameter gradients are wanted even when the input gradient is not
                const int c = o.c, k = u.se_k;
                const float* wp = s->w + u.w_off;
                float* gp = s->g + u.w_off;
                const float *sev = sv.stats + u.se_off, *p1 = sev + (size_t)s->B * c, *gate = sev + (size_t)s->B * (c + k);
                float* work = s->coef + u.se_work_off;
                const SeWork wk{work, work + (size_t)s->B * c, work + 2 * (size_t)s->B * c};
                se_backward_gate(dt, go.ptr, val_src(s, sv, u.in), s->B, o.h * o.w, c, k, wp, wp + (size_t)k * c + k, p1, gate, wk, s->scratch, s->scratch_floats, st);
                if (int rc = mark()) return rc;
                if (int rc = on_side()) return rc;
                se_param_grads(sev, p1, wk, s->B, c, k, gp, gp + (size_t)k * c, gp + (size_t)k * c + k, gp + 2 * (size_t)k * c + k, wst);
                const int si = s->vals[u.in].unit;
                if (want_in && si == ui - 1 && s->units[si].kind == U_SILU && s->vals[u.in].consumers == 1) {
                    // the SiLU in front applies gate and squeeze gradient as it reads this unit's output gradient
                    gated = GatedGrad{gate, wk.ds};
                    gi.state = G_ALIAS;
                    gi.ptr = go.ptr;
                    tick(s, ui, 5, st);
                    continue;
                }
                if (want_in) se_backward_scale(dt, go.ptr, s->B, o.h * o.w, c, gate, wk.ds, addend, own(u.in), st);
            } else if (want_in) {
                ChanSums sums{};
                const float* ts = nullptr;
                const int tgt = s->vals[u.in].first_cons == ui && bn_reduce_target(s, u.in) == s->vals[u.in].unit ? s->vals[u.in].unit : -1;
                if (tgt >= 0 && s->units[tgt].act == ACT_NONE && s->B <= MAX_SUM_BLOCKS) {      // the pass has at least one block a sample
                    const Unit& tu = s->units[tgt];
                    sums = bsums(s, sv) + 2 * tu.sum_off;
                    ts = sv.stats + s->vals[tu.out].stat_off;
                    pend.unit[tgt] = 1;
                    reduced[tgt] = 1;
                    s->bwd_sums_by[tgt] = ui;
                }
                silu_bwd(dt, go.ptr, gated.gate, gated.ds, val_src(s, sv, u.in), addend, s->B, o.h * o.w, o.c, own(u.in), sums, ts, ts ? ts + o.c : nullptr, st);
            }
            gated = GatedGrad{};
            if (want_in) {
                gi.state = G_OWNED;
                gi.ptr = own(u.in);
            }
        } else {  // U_GAP
            tick(s, ui, 4, st);
            if (want_in) {
                const Val& a = s->vals[u.in];
                GradState& gi = gs[u.in];
                const void* addend = gi.state == G_NONE ? nullptr : gi.ptr;
                gap_bwd(dt, go.ptr, s->B, a.h * a.w, a.c, addend, own(u.in), st);
                gi.state = G_OWNED;
                gi.ptr = own(u.in);
            }
        }
        tick(s, ui, 5, st);
    }
    if (s->need_dx && gs[0].state == G_ALIAS)
        CU(cudaMemcpyAsync(dx, gs[0].ptr, s->vals[0].elems * s->esz, cudaMemcpyDeviceToDevice, st));
    if (s->n_dw_weights) dw_settle(bsums(s, sv), s->dw_tab, s->n_dw, s->n_dw_weights, s->g, st);
    if (side_used) {            // join: the call's work is complete, in the caller's stream order, when the second stream's is
        CU(cudaEventRecord(s->ev_join, s->side));
        CU(cudaStreamWaitEvent(st, s->ev_join, 0));
    }
    CU(cudaGetLastError());
    return AST_OK;
}

// While it lives the calling thread may create streams and graphs although a capture is open elsewhere: one that the caller has begun in the
// global mode, on another stream of this thread or in another thread, would be invalidated by such a call.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// Runs a forward or backward call; from the third call with the same slot and buffers on as a graph.  A call is 20 to 190 kernels of a few
// microseconds, and launching them one by one costs the host 2.5 us each: on small maps or micro-batches more than the device needs (a sixth of
// MobileNetV2 at batch 4: 52 launches, 240 us a micro-batch against 130 us from a graph).  Not while the caller captures (the
// kernels then belong to the caller's graph), or a trace or a profile brackets single launches.  replay.h says which calls are kept; their graphs go with the
// stage.
template <typename F> static int run_call(asteroid_stage* s, bool bwd, int slot, const void* a, const void* b, cudaStream_t st, F call) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (tracing() || s->tm.on) return call(st);
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
        cudaGetLastError();
        return call(st);
    }
    if (cs != cudaStreamCaptureStatusNone) return call(st);
    RelaxedCapture relaxed;
    cudaGraphExec_t dropped;
    Replay* r = replay_entry(s->replays, bwd, slot, a, b, s->rounds, &dropped);
    if (dropped) cudaGraphExecDestroy(dropped);
    if (!r) return call(st);
    if (!r->exec && r->seen >= 0 && r->seen < 2) ++r->seen;
    else if (!r->exec && r->seen == 2) {
        r->seen = -1;
        if (!s->cap && cudaStreamCreateWithFlags(&s->cap, cudaStreamNonBlocking) != cudaSuccess) s->cap = nullptr;
        if (s->cap && cudaStreamBeginCapture(s->cap, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
            const uint64_t n0 = thread_launches();
            const int rc = call(s->cap);
            const uint64_t n = thread_launches() - n0;
            cudaGraph_t g = nullptr;
            const bool ended = cudaStreamEndCapture(s->cap, &g) == cudaSuccess;
            if (rc == AST_OK && ended && g && cudaGraphInstantiate(&r->exec, g, 0) != cudaSuccess) r->exec = nullptr;
            if (g) cudaGraphDestroy(g);
            if (r->exec) r->launches = n;
            count_launches((uint64_t)0 - n);       // captured, not launched
        }
        cudaGetLastError();
    }
    if (!r->exec) return call(st);
    CU(cudaGraphLaunch(r->exec, st));
    count_launches(r->launches);
    return AST_OK;
}

static int create_impl(const ast_layer* net, int n_layers, int first, int last, int in_h, int in_w, int B, int M, const ast_opts* opts,
                       asteroid_stage* s) {
    s->net.assign(net, net + n_layers);
    s->first = first; s->last = last; s->in_h = in_h; s->in_w = in_w; s->B = B; s->M = M;
    s->dtype = opts ? opts->dtype : AST_F32;
    if (s->dtype != AST_F32 && s->dtype != AST_BF16) return fail(AST_ERR_ARG, "dtype must be AST_F32 or AST_BF16");
    s->esz = s->dtype == AST_F32 ? 4 : 2;
    s->slots = (opts && opts->slots > 0) ? opts->slots : M;
    if (s->slots > M) s->slots = M;
    s->need_dx = opts ? (opts->need_input_grad != 0) : 1;
    s->eps = (opts && opts->bn_eps > 0.f) ? opts->bn_eps : 1e-5f;
    s->bn_mom = (opts && opts->bn_momentum > 0.f) ? opts->bn_momentum : 0.1f;
    {
        const char* e = getenv("ASTEROID_CHECK_GUARDS");
        s->check_guards = e && e[0] == '1';
    }
    int rc = build_plan(s);
    if (rc) return rc;

    const size_t np = s->n_pad;
    size_t mod = 0, opt = 0, act = 0, work = 0;
    if ((rc = arena_alloc(s, "parameters", &s->w, np * 4, &mod))) return rc;
    if ((rc = arena_alloc(s, "accumulated gradients", &s->G, np * 4, &mod))) return rc;
    if ((rc = arena_alloc(s, "micro-batch gradients", &s->g, np * 4, &mod))) return rc;
    if ((rc = arena_alloc(s, "derived weights", &s->derived, np * 4, &mod))) return rc;
    std::vector<RefreshSeg> segs;
    std::vector<int32_t> rest;
    plan_refresh(s, segs, &s->tiles, rest);
    s->n_dense = (int)segs.size();
    s->n_rest = (int)(rest.size() / 2);
    if ((rc = arena_alloc(s, "weight layers", &s->dense, segs.size() * sizeof(RefreshSeg), &mod))) return rc;
    if ((rc = arena_alloc(s, "other parameters", &s->rest, rest.size() * 4, &mod))) return rc;
    if ((rc = arena_alloc(s, "running statistics", &s->run, s->n_run * 4, &mod))) return rc;
    if (s->dtype == AST_BF16) {
        if ((rc = arena_alloc(s, "bf16 weights", &s->wb, np * 2, &mod))) return rc;
        if ((rc = arena_alloc(s, "bf16 derived weights", &s->wtb, np * 2, &mod))) return rc;
    }
    if (s->n_wpad) {
        if ((rc = arena_alloc(s, "padded weights", &s->wpad, s->n_wpad * 2, &mod))) return rc;
        if ((rc = arena_alloc(s, "padded weight gradient", &s->gpad, s->n_gpad * 4, &work))) return rc;
    }
    if ((rc = arena_alloc(s, "forward channel sums", &s->fsum, chan_sums_bytes(2 * s->n_bn_ch), &work))) return rc;
    if (s->n_dw) {
        std::vector<DwSettle> tab;
        for (const auto& u : s->units)
            if (u.kind == U_DW && u.g.k <= 5) tab.push_back(DwSettle{u.acc_off, (size_t)u.w_off, u.g.ci, u.g.k * u.g.k});
        if ((rc = arena_alloc(s, "depthwise layer table", &s->dw_tab, tab.size() * sizeof(DwSettle), &work))) return rc;
        CU(cudaMemcpy(s->dw_tab, tab.data(), tab.size() * sizeof(DwSettle), cudaMemcpyHostToDevice));
    }
    if ((rc = arena_alloc(s, "statistics pivots", &s->pivots, s->n_bn_ch * 4, &work))) return rc;
    if ((rc = arena_alloc(s, "error word", &s->err, 256, &work))) return rc;
    if ((rc = arena_alloc(s, "momentum", &s->v, np * 4, &opt))) return rc;
    if ((rc = arena_alloc(s, "activation slots", &s->slot_mem, s->slot_bytes * s->slots, &act))) return rc;
    if ((rc = arena_alloc(s, "gradient workspace", &s->grad_mem, s->grad_bytes, &work))) return rc;
    if ((rc = arena_alloc(s, "BatchNorm-backward coefficients", &s->coef, s->n_coef * 4, &work))) return rc;
    s->scratch_floats = (size_t)8 << 20;
    for (const auto& u : s->units)
        if (u.kind == U_CONV) s->scratch_floats = std::max(s->scratch_floats, (size_t)4 * u.g.co * u.g.k * u.g.k * u.g.ci);
    if ((rc = arena_alloc(s, "scratch", &s->scratch, s->scratch_floats * 4, &work))) return rc;
    if ((rc = arena_alloc(s, "scratch of the second stream", &s->scratch_side, s->scratch_floats * 4, &work))) return rc;
    for (auto& u : s->units)
        if (conv3_s2_tc_supported(s, u)) {
            u.up_off = (long)s->up_bytes;
            s->up_bytes += align_up((size_t)u.g.n * u.g.hi * u.g.wi * u.g.co * 2, 256);
        }
    if (s->up_bytes && (rc = arena_alloc(s, "zero-inserted gradients", &s->up_mem, s->up_bytes, &work))) return rc;
    CU(cudaStreamCreateWithFlags(&s->side, cudaStreamNonBlocking));
    CU(cudaEventCreateWithFlags(&s->ev_fork, cudaEventDisableTiming));
    CU(cudaEventCreateWithFlags(&s->ev_join, cudaEventDisableTiming));
    s->bytes_mod = mod; s->bytes_opt = opt; s->bytes_work = work;
    if (!segs.empty()) CU(cudaMemcpy(s->dense, segs.data(), segs.size() * sizeof(RefreshSeg), cudaMemcpyHostToDevice));
    if (!rest.empty()) CU(cudaMemcpy(s->rest, rest.data(), rest.size() * 4, cudaMemcpyHostToDevice));
    if ((rc = reset_bn_running(s))) return rc;
    s->slot_of_mb.assign(M, -1);
    s->mb_of_slot.assign(s->slots, -1);
    s->sums_left.assign(s->slots, 0);
    s->fwd_stats_blocks.assign(s->units.size(), 0);
    s->bwd_sums_by.assign(s->units.size(), -1);
    s->add_deferred.assign(s->units.size(), 0);
    return AST_OK;
}

}  // namespace ast

// ================================================================================ C ABI
extern "C" {

int asteroid_stage_create(const ast_layer* net, int n_layers, int first, int last, int in_h, int in_w, int micro_batch, int M,
                          const ast_opts* opts, asteroid_stage** out) {
    if (!net || !out) return fail(AST_ERR_ARG, "null argument");
    *out = nullptr;
    if (n_layers < 1 || first < 0 || last < first || last >= n_layers) return fail(AST_ERR_ARG, "bad layer range [%d,%d] of %d layers", first, last, n_layers);
    if (in_h < 1 || in_w < 1 || micro_batch < 1 || M < 1) return fail(AST_ERR_ARG, "sizes must be positive");
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev < 1) {
        cudaGetLastError();
        return fail(AST_ERR_CUDA, "no CUDA device: this library has no CPU path");
    }
    asteroid_stage* s = new asteroid_stage();
    int rc = create_impl(net, n_layers, first, last, in_h, in_w, micro_batch, M, opts, s);
    if (rc) {
        free_stage(s);
        return rc;
    }
    *out = s;
    return AST_OK;
}

void asteroid_stage_destroy(asteroid_stage* s) {
    if (!s) return;
    cudaDeviceSynchronize();
    free_stage(s);
}

size_t asteroid_stage_param_count(const asteroid_stage* s) { return s ? s->n_params : 0; }

size_t asteroid_stage_output_elems(const asteroid_stage* s, int* h, int* w, int* c) {
    if (!s) return 0;
    const Val& o = s->vals.back();
    if (h) *h = o.h;
    if (w) *w = o.w;
    if (c) *c = o.c;
    return o.elems;
}

int asteroid_stage_grad_buffer(asteroid_stage* s, float** G, size_t* n) {
    if (!s || !G || !n) return fail(AST_ERR_ARG, "null argument");
    *G = s->G;
    *n = s->n_pad;
    return AST_OK;
}

int asteroid_stage_import_state(asteroid_stage* s, const float* params, const float* momentum, size_t n) {
    if (!s || !params) return fail(AST_ERR_ARG, "null argument");
    if (n != s->n_params) return fail(AST_ERR_ARG, "state has %zu values, the stage has %zu parameters", n, s->n_params);
    CU(cudaDeviceSynchronize());
    if (n) {
        std::vector<float> h(s->n_pad, 0.f);
        for (const auto& g : s->segs) memcpy(h.data() + g.in, params + g.pub, g.n * 4);
        CU(cudaMemcpy(s->w, h.data(), s->n_pad * 4, cudaMemcpyHostToDevice));
        if (momentum) {
            for (const auto& g : s->segs) memcpy(h.data() + g.in, momentum + g.pub, g.n * 4);
            CU(cudaMemcpy(s->v, h.data(), s->n_pad * 4, cudaMemcpyHostToDevice));
        } else CU(cudaMemset(s->v, 0, s->n_pad * 4));
        CU(cudaMemset(s->G, 0, s->n_pad * 4));
        refresh_weights(s, 0);
    }
    int rc = reset_bn_running(s);
    if (rc) return rc;
    s->n_acc = 0;
    s->pending_g = -1;
    CU(cudaDeviceSynchronize());
    return AST_OK;
}

int asteroid_stage_export_state(asteroid_stage* s, float* params, float* momentum, float* grad_accum, float* micro_grad, size_t n) {
    if (!s) return fail(AST_ERR_ARG, "null argument");
    if (n != s->n_params) return fail(AST_ERR_ARG, "state has %zu values, the stage has %zu parameters", n, s->n_params);
    CU(cudaDeviceSynchronize());
    int errw = 0;
    CU(cudaMemcpy(&errw, s->err, sizeof errw, cudaMemcpyDeviceToHost));
    if (errw) {
        CU(cudaMemset(s->err, 0, sizeof errw));
        return fail(AST_ERR_TIMEOUT, "a bounded device-side wait expired in a tensor-core kernel; results of this round are invalid");
    }
    if (s->check_guards) {
        int grc = check_guards(s);
        if (grc) return grc;
    }
    if (n) {
        std::vector<float> h(s->n_pad);
        const std::pair<float*, const float*> outs[4] = {{params, s->w}, {momentum, s->v}, {grad_accum, s->G}, {micro_grad, s->g}};
        for (const auto& o : outs) {
            if (!o.first) continue;
            CU(cudaMemcpy(h.data(), o.second, s->n_pad * 4, cudaMemcpyDeviceToHost));
            for (const auto& g : s->segs) memcpy(o.first + g.pub, h.data() + g.in, g.n * 4);
        }
    }
    return AST_OK;
}

int asteroid_stage_export_bn_running(asteroid_stage* s, float* mean, float* var, size_t n) {
    if (!s || !mean || !var) return fail(AST_ERR_ARG, "null argument");
    if (n * 2 != s->n_run) return fail(AST_ERR_ARG, "expected %zu channels", s->n_run / 2);
    CU(cudaDeviceSynchronize());
    std::vector<float> h(s->n_run);
    if (s->n_run) CU(cudaMemcpy(h.data(), s->run, s->n_run * 4, cudaMemcpyDeviceToHost));
    size_t o = 0;
    for (const auto& u : s->units)
        if (u.l_bn >= 0) {
            memcpy(mean + o, h.data() + u.run_off, u.g.co * sizeof(float));
            memcpy(var + o, h.data() + u.run_off + u.g.co, u.g.co * sizeof(float));
            o += u.g.co;
        }
    return AST_OK;
}

int asteroid_stage_forward(asteroid_stage* s, int mb, const void* x, void* y, void* stream) {
    if (!s || !x || !y) return fail(AST_ERR_ARG, "null argument");
    if (mb < 0 || mb >= s->M) return fail(AST_ERR_ARG, "micro-batch %d outside [0,%d)", mb, s->M);
    if (s->slot_of_mb[mb] >= 0) return fail(AST_ERR_ORDER, "micro-batch %d is already resident (forward twice without backward)", mb);
    int slot = -1;
    for (int i = 0; i < s->slots; ++i)
        if (s->mb_of_slot[i] < 0) {
            slot = i;
            break;
        }
    if (slot < 0) return fail(AST_ERR_ORDER, "all %d activation slots hold micro-batches awaiting backward", s->slots);
    int rc = run_call(s, false, slot, x, y, (cudaStream_t)stream, [&](cudaStream_t st) { return forward_impl(s, slot, x, y, st); });
    if (rc) return rc;
    s->slot_of_mb[mb] = slot;
    s->mb_of_slot[slot] = mb;
    return AST_OK;
}

int asteroid_stage_backward(asteroid_stage* s, int mb, const void* dy, void* dx, void* stream) {
    if (!s || !dy) return fail(AST_ERR_ARG, "null argument");
    if (mb < 0 || mb >= s->M) return fail(AST_ERR_ARG, "micro-batch %d outside [0,%d)", mb, s->M);
    if (s->need_dx && !dx) return fail(AST_ERR_ARG, "dx is required unless need_input_grad is 0");
    int slot = s->slot_of_mb[mb];
    if (slot < 0) return fail(AST_ERR_ORDER, "backward of micro-batch %d without a resident forward", mb);
    if (s->pending_g >= 0) return fail(AST_ERR_ORDER, "gradients of micro-batch %d have not been accumulated yet", s->pending_g);
    if (s->sums_left[slot] && s->n_bsum) CU(cudaMemsetAsync(slot_view(s, slot).bsum, 0, chan_sums_bytes(s->n_bsum), (cudaStream_t)stream));
    int rc = run_call(s, true, slot, dy, dx, (cudaStream_t)stream, [&](cudaStream_t st) { return backward_impl(s, slot, dy, dx, st); });
    s->sums_left[slot] = rc != AST_OK;
    if (rc) return rc;
    s->pending_slot = slot;
    s->slot_of_mb[mb] = -1;
    s->mb_of_slot[slot] = -1;
    s->pending_g = mb;
    return AST_OK;
}

int asteroid_stage_accumulate(asteroid_stage* s, int mb, void* stream) {
    if (!s) return fail(AST_ERR_ARG, "null argument");
    if (s->pending_g < 0 || s->pending_g != mb) return fail(AST_ERR_ORDER, "accumulate(%d): the last backward was of micro-batch %d", mb, s->pending_g);
    if (s->n_acc >= s->M) return fail(AST_ERR_ORDER, "already accumulated %d micro-batches this round", s->M);
    accumulate(s->G, s->g, s->n_pad, bsums(s, slot_view(s, s->pending_slot)), s->n_bsum, (cudaStream_t)stream);
    CU(cudaGetLastError());
    s->pending_g = -1;
    s->n_acc++;
    return AST_OK;
}

int asteroid_stage_step(asteroid_stage* s, float lr, float momentum, void* stream) {
    if (!s) return fail(AST_ERR_ARG, "null argument");
    if (s->n_acc != s->M) return fail(AST_ERR_ORDER, "step after %d of %d micro-batches accumulated", s->n_acc, s->M);
    cudaStream_t st = (cudaStream_t)stream;
    sgd_step(s->w, s->v, s->G, s->n_pad, 1.f / (float)s->M, lr, momentum, st);
    refresh_weights(s, st);
    CU(cudaGetLastError());
    s->n_acc = 0;
    ++s->rounds;
    return AST_OK;
}

int asteroid_loss_mse(const void* y, const void* target, size_t n, int dtype, void* dy, float* loss, void* stream) {
    if (!y || !target || !dy || !loss || n == 0) return fail(AST_ERR_ARG, "null or empty argument");
    if (dtype != AST_F32 && dtype != AST_BF16) return fail(AST_ERR_ARG, "bad dtype");
    float* sc;
    int rc = loss_scratch(&sc);
    if (rc) return rc;
    loss_mse(dtype, y, target, n, dy, loss, sc, (cudaStream_t)stream);
    CU(cudaGetLastError());
    return AST_OK;
}

int asteroid_loss_softmax_xent(const void* logits, const int32_t* labels, int rows, int classes, int dtype, void* dlogits, float* loss,
                               void* stream) {
    if (!logits || !labels || !dlogits || !loss) return fail(AST_ERR_ARG, "null argument");
    if (rows < 1 || rows > 65536 || classes < 1) return fail(AST_ERR_ARG, "rows must be in [1,65536], classes positive");
    if (dtype != AST_F32 && dtype != AST_BF16) return fail(AST_ERR_ARG, "bad dtype");
    float* sc;
    int rc = loss_scratch(&sc);
    if (rc) return rc;
    loss_xent(dtype, logits, labels, rows, classes, dlogits, loss, sc, (cudaStream_t)stream);
    CU(cudaGetLastError());
    return AST_OK;
}

int asteroid_stage_profile(asteroid_stage* s, int layer, int batch, ast_layer_profile* out) {
    if (!s || !out) return fail(AST_ERR_ARG, "null argument");
    if (layer < s->first || layer > s->last) return fail(AST_ERR_ARG, "layer %d outside the stage [%d,%d]", layer, s->first, s->last);
    if (batch < 1) return fail(AST_ERR_ARG, "batch must be positive");
    CU(cudaDeviceSynchronize());
    asteroid_stage* t = nullptr;
    size_t ti = 0;
    for (; ti < s->prof_cache.size(); ++ti)
        if (s->prof_cache[ti]->B == batch) {
            t = s->prof_cache[ti];
            break;
        }
    if (!t) {
        t = new asteroid_stage();
        ast_opts o{s->dtype, 1, s->need_dx, s->eps, s->bn_mom};
        int rc = create_impl(s->net.data(), (int)s->net.size(), s->first, s->last, s->in_h, s->in_w, batch, 1, &o, t);
        if (rc) {
            free_stage(t);
            return rc;
        }
        const size_t nu = t->units.size();
        t->tm.ev.resize(nu * 6);
        for (auto& e : t->tm.ev) CU(cudaEventCreate(&e));
        if (s->n_pad) {
            CU(cudaMemcpy(t->w, s->w, s->n_pad * 4, cudaMemcpyDeviceToDevice));
            CU(cudaMemcpy(t->derived, s->derived, s->n_pad * 4, cudaMemcpyDeviceToDevice));
            if (s->wb) {
                CU(cudaMemcpy(t->wb, s->wb, s->n_pad * 2, cudaMemcpyDeviceToDevice));
                CU(cudaMemcpy(t->wtb, s->wtb, s->n_pad * 2, cudaMemcpyDeviceToDevice));
            }
            if (s->wpad && t->wpad && s->n_wpad == t->n_wpad) CU(cudaMemcpy(t->wpad, s->wpad, s->n_wpad * 2, cudaMemcpyDeviceToDevice));
        }
        const Val &vi = t->vals[0], &vo = t->vals.back();
        char *x = nullptr, *y = nullptr, *dy = nullptr, *dx = nullptr;
        size_t tally = 0;
        int rc2 = dev_alloc(&x, vi.elems * t->esz, &tally);
        if (!rc2) rc2 = dev_alloc(&dx, vi.elems * t->esz, &tally);
        if (!rc2) rc2 = dev_alloc(&y, vo.elems * t->esz, &tally);
        if (!rc2) rc2 = dev_alloc(&dy, vo.elems * t->esz, &tally);
        std::vector<std::vector<float>> samples(nu * 4);
        const int warm = 3, timed = 7;
        for (int it = 0; !rc2 && it < warm + timed; ++it) {
            t->tm.on = it >= warm;
            rc2 = forward_impl(t, 0, x, y, 0);
            if (!rc2) rc2 = backward_impl(t, 0, dy, dx, 0);
            if (!rc2 && cudaDeviceSynchronize() != cudaSuccess) rc2 = fail(AST_ERR_CUDA, "profile run failed: %s", cudaGetErrorString(cudaGetLastError()));
            if (!rc2 && t->tm.on)
                for (size_t u = 0; u < nu; ++u) {
                    const int pairs[4][2] = {{0, 1}, {1, 2}, {3, 4}, {4, 5}};
                    for (int q = 0; q < 4; ++q) {
                        float ms = 0.f;
                        cudaEventElapsedTime(&ms, t->tm.ev[u * 6 + pairs[q][0]], t->tm.ev[u * 6 + pairs[q][1]]);
                        samples[u * 4 + q].push_back(ms);
                    }
                }
        }
        t->tm.on = false;
        cudaFree(x); cudaFree(y); cudaFree(dy); cudaFree(dx);
        if (rc2) {
            free_stage(t);
            return rc2;
        }
        std::vector<double> med(nu * 4);
        for (size_t q = 0; q < med.size(); ++q) {
            std::sort(samples[q].begin(), samples[q].end());
            med[q] = samples[q][samples[q].size() / 2];
        }
        s->prof_cache.push_back(t);
        s->prof_ms.push_back(med);
        ti = s->prof_cache.size() - 1;
    }
    memset(out, 0, sizeof *out);
    out->fused_into = -1;
    out->mem_mod = t->bytes_mod;
    out->mem_opt = t->bytes_opt;
    out->mem_act = t->slot_bytes;
    out->mem_work = t->bytes_work;
    const ast_layer& L = s->net[layer];
    out->w_l_bytes = 4ull * (uint64_t)n_layer_params(L);
    const std::vector<double>& ms = s->prof_ms[ti];
    for (size_t ui = 0; ui < t->units.size(); ++ui) {
        const Unit& u = t->units[ui];
        int lo = u.l_main, hi = std::max(u.l_main, std::max(u.l_bn, u.l_act));
        if (layer < lo || layer > hi) continue;
        const Val &vin = t->vals[u.in], &vout = t->vals[u.out];
        const uint64_t e = t->esz, xin = vin.elems * e, zo = vout.elems * e;
        out->a_l_bytes = zo;
        if (layer == u.l_main) {
            out->t_f_ms = ms[ui * 4 + 0];
            out->t_b_ms = ms[ui * 4 + 3];
            if (u.kind == U_CONV || u.kind == U_DW) {
                uint64_t macs = (uint64_t)vout.elems * (u.kind == U_DW ? (uint64_t)u.g.k * u.g.k : (uint64_t)u.g.k * u.g.k * u.g.ci);
                out->flops = 2 * macs;
                out->alg_bytes_f = xin + zo + out->w_l_bytes;
                // bwd-weight reads dy, z, x; bwd-data reads dy, z and writes dx
                out->alg_bytes_b = 2 * (zo + zo) + xin + ((u.in != 0 || t->need_dx) ? xin : 0) + 2 * out->w_l_bytes;
                if (ui > 0 && t->add_deferred[ui - 1]) out->alg_bytes_f += 2 * xin;    // the second operand of the sum in front, and the sum written
            } else if (u.kind == U_ADD) {
                out->alg_bytes_f = 3 * zo;
                out->alg_bytes_b = u.act == ACT_RELU ? 3 * zo : 0;
                if (t->add_deferred[ui]) {             // formed by the pointwise layer behind
                    out->t_f_ms = 0;
                    out->alg_bytes_f = 0;
                    out->fused_into = t->units[ui + 1].l_main;
                }
            } else if (u.kind == U_SILU) {
                out->alg_bytes_f = xin + zo;
                out->alg_bytes_b = 3 * zo;              // dy, x -> dx
            } else if (u.kind == U_SE) {
                out->alg_bytes_f = 2 * xin + zo;        // x for the squeeze, x again for the scaling
                out->alg_bytes_b = 5 * zo;              // x and dout for the gate gradient, both again for dx
            } else {
                out->alg_bytes_f = xin + zo;
                out->alg_bytes_b = xin + zo;
            }
        } else if (layer == u.l_bn) {
            out->t_f_ms = ms[ui * 4 + 1];
            out->t_b_ms = ms[ui * 4 + 2];
            // Statistics: a standalone pass over z, or - taken inside the producing kernel - only the finishing of that
            // kernel's per-CTA partials.  Backward sums: a standalone pass over dy and z, or nothing here when the
            // backward-data kernel of the consuming unit took them (its record carries the time; fused_into names it).
            const int fb = t->fwd_stats_blocks[ui];
            out->alg_bytes_f = fb > 0 ? 8ull * vout.c * (uint64_t)(fb + 4) : zo;
            if (fb > 0) out->fused_into = u.l_main;
            const int by = t->bwd_sums_by[ui];
            out->alg_bytes_b = by >= 0 ? 0 : 2 * zo;
            if (by >= 0) out->fused_into = t->units[by].l_main;
        } else {                            // activation: applied inside the neighbouring kernels
            out->fused_into = u.l_bn >= 0 ? u.l_bn : u.l_main;
        }
        return AST_OK;
    }
    return fail(AST_ERR_ARG, "layer %d not found in the plan", layer);
}

int asteroid_selftest_bounded_wait(void) {
    int* err = nullptr;
    CU(cudaMalloc((void**)&err, sizeof(int)));
    cudaError_t e = cudaMemset(err, 0, sizeof(int));
    int h = 0;
    if (e == cudaSuccess) {
        launch_bounded_wait_probe(err, 1024u, 0);
        e = cudaDeviceSynchronize();
    }
    if (e == cudaSuccess) e = cudaMemcpy(&h, err, sizeof h, cudaMemcpyDeviceToHost);
    cudaFree(err);
    if (e != cudaSuccess) return fail(AST_ERR_CUDA, "bounded-wait self-test: %s", cudaGetErrorString(e));
    if (h) return fail(AST_ERR_TIMEOUT, "a bounded device-side wait expired (self-test: expected)");
    return AST_OK;
}

uint64_t asteroid_launch_count(void) { return launches(); }
const char* asteroid_last_error(void) { return g_err.c_str(); }

}  // extern "C"
