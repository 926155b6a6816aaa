// Launch side of the register-operand pointwise kernels (pw_mma.cuh): instantiations, shared-memory layout and the choice of a
// tiling for a layer.
#include <string.h>

#include "pw_mma.cuh"
#include "pw_mma.h"

namespace ast {
namespace {

using namespace mma;

typedef void (*KernelFn)(const Args);

constexpr size_t SMEM_MOST = 200 * 1024;
// Whether a persistent layer's operands are requested several steps ahead (pw_mma.cuh): input gradients of 128 channels and more in blocks of 64 columns and the large residual sums of
// defers_add (stage.cu), where a CTA has more than one tile.  Both read two operands, and a step took 0.75 to 1 us, a trip to memory, whatever its work was: ResNet stage at batch 32
// 20 592 -> 19 523 us a round.  A forward of one operand has its steps in time, and slots only add a store and a load of shared memory a vector: 128 -> 512 at 25 088 pixels 27.3 -> 29.9 us,
// 256 -> 512 39.3 -> 43.7, 256 -> 64 at 57 000 19.0 -> 21.0 (that stage with such forwards 19 735 instead of 19 622).  Only operands beyond L2 gain there: 512 -> 64 from 94 000 pixels on,
// 49 -> 43.  In narrower blocks one step ahead is as good or better too: slots in all persistent kernels took half of MobileNetV2 with the head 4140 -> 4210 us, EfficientNet 6941 -> 7029,
// the ragged stage 613 -> 637; input gradients in narrower blocks EfficientNet 6955 -> 6994 from 128 channels on, 6936 -> 6955 from 256; single tiles the ragged ResNet share 1681 -> 1689.
// The form is built for what is launched: gradients with a transform (the others have one operand), whose blocks of 64 columns bwd_choose offers one pixel tile a warp, and large sums, for which
// fwd_choose takes two.  Where the slots do not fit beside the weights and coefficients, one step ahead stays: gradients of 512 channels behind an unapplied activation, two CTAs.
constexpr bool deep_form(bool bwd, int mi, int nj, int xf) { return nj == 8 && (bwd ? mi == 1 && xf != XF_NONE : mi == 2 && xf == XF_SUM); }
// The slots lie behind the coefficients that the transform has, not the most it could have: the 8 KB of two CTAs decide whether gradients of 512 channels in blocks of 64 columns fit two to a
// multiprocessor (ResNet stage at batch 32 19 830 -> 19 636 us a round).  Five steps ahead instead of three: 19 855.
size_t deep_smem(bool bwd, int K, const MmaTiling& c, int xf) {
    const size_t Kp = (size_t)(K + 31) / 32 * 32;
    return mma_smem(bwd, K, c) - (bwd && xf != XF_ACT ? 8 * Kp : 0) + (xf == XF_SUM ? 4 * Kp : 0) + (size_t)(c.mi == 1 ? Slots<1>::BYTES : Slots<2>::BYTES) * 32 * c.wm;
}
// Rows that are no whole 32-byte sectors gain only where the two operands, 32 MB and more, come from beyond L2 in good part: the copies pass L1 by, where a load in registers finds the sector it
// shares with the row before.  A unit's forward and backward, one step ahead against several (reduction -> columns of the gradient): 136 -> 256 at 10 000 pixels 49.8 us against 50.2, with a ReLU
// 52.0 against 53.0, but 264 -> 512 at 57 000 410 against 377.  All others gain from 5 000 pixels on (512 -> 512 104.2 against 101.8) or stay (128 -> 64 at 25 088 44.5 against 44.6).  Behind an
// activation that is not in them yet, small maps lose up to 1.4 us of 50 to 170 alone, but gain beside weight gradients: rounds of the ResNet stage, four micro-batches, without them below 20 000
// pixels 5 494 us instead of 5 489 (10 192 pixels), 7 015 instead of 6 989 (15 680); of 32 samples without them below 8 M elements 19 686 instead of 19 521 (eight micro-batches).
bool deep_layer(bool bwd, int P, int K, const MmaTiling& c, int xf) {
    const size_t smem = deep_smem(bwd, K, c, xf);
    return c.wk == 1 && deep_form(bwd, c.mi, c.nj, xf) && K >= 128 && (!bwd || K % 16 == 0 || (size_t)P * K >= (size_t)8 << 20) && smem <= SMEM_MOST &&
           (smem + 1024) * c.ctas <= 227 * 1024;
}

template <bool BWD, int NJ, int G, int XF> KernelFn pick(int mi, int wk, bool deep) {
    if constexpr (deep_form(BWD, 1, NJ, XF))
        if (deep && mi == 1 && wk == 1) return pw_mma_kernel<BWD, 1, NJ, G, XF, true>;
    if (wk == 1) return mi == 1 ? pw_mma_kernel<BWD, 1, NJ, G, XF, false> : pw_mma_kernel<BWD, 2, NJ, G, XF, false>;
    return wk == 2 ? pw_mma_split_kernel<BWD, NJ, G, 2, XF> : wk == 4 ? pw_mma_split_kernel<BWD, NJ, G, 4, XF> : pw_mma_split_kernel<BWD, NJ, G, 8, XF>;
}
template <bool BWD, int XF> KernelFn by_columns(const MmaTiling& c, bool deep) {
    switch (c.nj) {
        case 2: return pick<BWD, 2, 2, XF>(c.mi, c.wk, deep);
        case 3: return pick<BWD, 3, 1, XF>(c.mi, c.wk, deep);
        case 4: return pick<BWD, 4, 4, XF>(c.mi, c.wk, deep);
        case 6: return pick<BWD, 6, 2, XF>(c.mi, c.wk, deep);
        default: return pick<BWD, 8, 4, XF>(c.mi, c.wk, deep);
    }
}
template <bool BWD> KernelFn kernel_for(const MmaTiling& c, int xf, bool deep) {
    if (!BWD && xf == XF_SUM) return pw_mma_kernel<false, 2, 8, 4, XF_SUM, true>;
    if (!BWD && xf == XF_ADD) return by_columns<false, XF_ADD>(c, deep);
    return xf == XF_NONE ? by_columns<BWD, XF_NONE>(c, deep) : xf == XF_AFFINE ? by_columns<BWD, XF_AFFINE>(c, deep) : by_columns<BWD, XF_ACT>(c, deep);
}
// the shared-memory limit of every instantiation, raised once per device
template <bool BWD> void raise_limits() {
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load(std::memory_order_acquire) & bit) return;
    for (int nj : {2, 3, 4, 6, 8})
        for (int v = 0; v < 5; ++v)
            for (int xf = XF_NONE; xf <= (BWD ? XF_ACT : XF_SUM); ++xf) {
                MmaTiling c{};
                c.nj = nj;
                c.mi = v == 1 ? 2 : 1;
                c.wk = v < 2 ? 1 : 1 << (v - 1);
                for (bool deep : {false, true}) cudaFuncSetAttribute(kernel_for<BWD>(c, xf, deep), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MOST);
            }
    done.fetch_or(bit, std::memory_order_release);
}

uint32_t w_pitch(int K) {
    uint32_t b = (uint32_t)((K + 31) / 32) * 64u;      // whole 32-channel chunks
    return b % 128 == 0 ? b + 64 : b;                  // an odd multiple of 64 bytes: a fragment read meets every bank once
}


// Backward tilings by a cost model (us), fitted to 1 500 timings over 49 layers (512 to 200 704 pixels, 16 to 1280 channels, with and without an
// addend): within 2.2 % of the best tiling on average, at worst 27 %.  Persistent form: a CTA's tile takes the longer of its own latency
// and the issue time of all warps on the multiprocessor, per 32-channel chunk and column tile, plus the epilogue, which an addend makes longer;
// weights are staged once per CTA.  Split form: one tile per CTA, waves over the chip.  Offered are the tilings that won somewhere: with two
// pixel tiles per warp one CTA of eight warps or two of four; eight column tiles per warp only with one pixel tile (the epilogue holds four
// vectors per column tile).  The timings are of kernels that request one step ahead; gradients that request several (deep_layer) take the tiling that the model names and were not fitted
// again.  Before the model (one rule as in the forward): 128 -> 512 at 25 088 pixels 57.6 -> 52.2 us, 64 -> 64 at 100 352
// 27.5 -> 21.4, 160 -> 960 at 784 8.1 -> 6.0, 384 -> 64 at 3136 10.5 -> 6.7.
bool bwd_choose(int P, int K, int N, MmaTiling* out) {
    const int KCH = (K + 31) / 32, sms = sm_count();
    double best = 0;
    auto offer = [&](int mi, int nj, int wm, int wk, int ctas) {
        const MmaTiling c{mi, nj, wm, wk, ctas};
        if (mma_smem(true, K, c) * (wk == 1 ? ctas : 1) > 200 * 1024) return;
        const int cols = (N + 8 * nj - 1) / (8 * nj);
        double t;
        if (wk == 1) {
            const int tiles = (P + 16 * mi * wm - 1) / (16 * mi * wm), cap = sms * ctas / cols > 0 ? sms * ctas / cols : 1, gx = tiles < cap ? tiles : cap;
            const int turns = (tiles + gx - 1) / gx;
            int r = (gx * cols + sms - 1) / sms;
            if (r > ctas) r = ctas;
            const double issue = (double)r * wm * mi * (KCH * (0.0502 + 0.00418 * nj) + nj * 0.0315);
            const double lat = 1.01 + 0.476 * KCH * (1.0 + 0.269 * (mi - 1)) + 0.0202 * mi * nj;
            t = 1.53 + 0.0154 * r * nj * KCH + turns * (lat > issue ? lat : issue);
        } else {
            const int bm = 128 / wk, waves = ((P + bm - 1) / bm * cols + sms - 1) / sms, kc = (KCH + wk - 1) / wk;
            t = 0.714 + waves * (1.85 + kc * (0.651 + 0.00019 * nj) + nj * 0.0301 * (1.0 + 0.0529 * wk) + 0.0224 * nj * KCH);
        }
        if (best == 0 || t < best) {
            best = t;
            *out = c;
        }
    };
    for (int nj : {8, 6, 4, 3, 2}) {
        const bool narrow = (nj == 2 && N > 16) || (nj == 3 && N > 24);       // only where the weights of more columns do not fit
        if (narrow ? best != 0 : (N + 8 * nj - 1) / (8 * nj) * nj * 8 > N * 1.35 + 8) continue;
        if (nj == 8) {
            offer(1, 8, 4, 1, 2);
            if (P < 20000) offer(1, 8, 8, 1, 1);           // on larger maps 5 to 30 % slower than two CTAs of four warps, which the model does not see
        } else {
            offer(2, nj, 8, 1, 1);
            offer(2, nj, 4, 1, 2);
            offer(1, nj, 8, 1, 2);
        }
        if (P <= 30000)
            for (int wk : {2, 4, 8}) offer(1, nj, 8 / wk, wk, 1);
    }
    return best != 0;
}

// Forward tilings by a model of the same form, fitted to 1 300 timings over the same layers: within 3.3 % of the best tiling on average, at worst 36 %.
// The forward kernels need fewer registers, so two CTAs of eight warps or four of four share a multiprocessor where the warp's tile is small.
// Before the model (a rule of thumb on the map and the channels, 11 % above the best on average): 24 -> 144 at 100 352 pixels 20.1 -> 15.7 us, 16 -> 96 at
// 200 704 26.1 -> 18.6, 32 -> 192 at 12 544 7.4 -> 4.2, 64 -> 384 at 3 136 7.5 -> 4.1, 96 -> 576 8.8 -> 5.4, 512 -> 128 at 4 704 10.0 -> 7.5.
bool fwd_choose(int P, int K, int N, MmaTiling* out) {
    const int KCH = (K + 31) / 32, sms = sm_count();
    double best = 0;
    auto offer = [&](int mi, int nj, int wm, int wk, int ctas) {
        const MmaTiling c{mi, nj, wm, wk, ctas};
        if (mma_smem(false, K, c) * (wk == 1 ? ctas : 1) > 200 * 1024) return;
        const int cols = (N + 8 * nj - 1) / (8 * nj);
        double t;
        if (wk == 1) {
            const int tiles = (P + 16 * mi * wm - 1) / (16 * mi * wm), cap = sms * ctas / cols > 0 ? sms * ctas / cols : 1, gx = tiles < cap ? tiles : cap;
            const int turns = (tiles + gx - 1) / gx;
            int r = (gx * cols + sms - 1) / sms;
            if (r > ctas) r = ctas;
            const double issue = (double)r * wm * mi * (KCH * (0.0108 + 0.00169 * nj) + nj * 0.01086);
            const double lat = 0.0046 + 0.312 * KCH * (1.0 + 0.0966 * (mi - 1)) + 0.0912 * mi * nj;
            t = 1.085 + 0.0253 * r * nj * KCH + turns * (lat > issue ? lat : issue);
        } else {
            const int bm = 128 / wk, per = ((P + bm - 1) / bm * cols + sms - 1) / sms, r = per < 2 ? per : 2, waves = (per + r - 1) / r, kc = (KCH + wk - 1) / wk;
            t = 4.177 + waves * (kc * (0.447 + 0.00146 * nj * r) + r * (0.00019 * nj + 0.00831 * nj * KCH));
        }
        if (best == 0 || t < best) {
            best = t;
            *out = c;
        }
    };
    for (int nj : {8, 6, 4, 3, 2}) {
        const bool narrow = (nj == 2 && N > 32) || (nj == 3 && N > 24);       // only where the weights of more columns do not fit
        if (narrow ? best != 0 : (N + 8 * nj - 1) / (8 * nj) * nj * 8 > N * 1.35 + 8) continue;
        for (int mi = 2; mi >= 1; --mi) {
            offer(mi, nj, 8, 1, 1);
            if (mi == 1 || nj <= 3) offer(mi, nj, 8, 1, 2);
            offer(mi, nj, 4, 1, 2);
            if (nj == 4 || (mi == 1 && nj >= 3)) offer(mi, nj, 4, 1, 4);
        }
        if (P <= 30000)
            for (int wk : {2, 4, 8}) offer(1, nj, 8 / wk, wk, 1);
    }
    return best != 0;
}

}  // namespace

// Which layers run here: all whose channel counts are whole vectors, but for more than 256 x 64 products per pixel on more than 50 000 pixels with at most
// 256 channels a side.  There the arithmetic of mma.sync (and the shared-memory reads of its weights) is the bound and the tensor-memory
// pipeline of pw_tc.cu is as fast or faster: 64 -> 256 at 100 352 pixels 26.3 us against 29.3, backward to 256 channels 71 against 77.  To at
// most 64 channels it is not: 256 -> 64 30.6 against 24.0, backward 45 against 42.  (One layer with its BatchNorm sums in a captured chain.)  Requests several steps ahead do not move the
// line: with them and 256 -> 128 forward here the ResNet stage at batch 32 takes 19 660 us a round, with its backward 19 671, without 19 611.
// With 192 to 256 channels on both sides the pipeline does not fit and pw_stream.cu and the one-tile kernel take the layer: 256 -> 256 on 50 176
// pixels forward 33 us with its pass for the sums (37 here), backward with a transform 49 (72), without 23 (49).
bool mma_choose(bool bwd, int P, int K, int N, MmaTiling* out) {
    if (K % 8 || N % 8 || (double)P * (K > N ? K : N) * 2.0 >= 4.0e9) return false;
    if (P >= 50000 && K <= 256 && N <= 256 && K * N >= 256 * 64 && N > 64) return false;
    return bwd ? bwd_choose(P, K, N, out) : fwd_choose(P, K, N, out);
}

bool mma_deep_sum(int P, int K, const MmaTiling& c) { return deep_layer(false, P, K, c, XF_SUM) && (P + 16 * c.mi * c.wm - 1) / (16 * c.mi * c.wm) > sm_count() * c.ctas; }

size_t mma_smem(bool bwd, int K, const MmaTiling& c) {
    const int Kp = (K + 31) / 32 * 32, BN = c.nj * 8;
    size_t b = (size_t)BN * w_pitch(K) + (size_t)(bwd ? 5 : 3) * Kp * 4 + (size_t)(bwd ? 4 : 1) * BN * 4;
    if (c.wk == 1) b += (size_t)c.wm * 2 * BN * 4;
    else {
        const size_t acc = (size_t)128 * (BN + 4) * 4;
        b += acc > 16384 ? acc : 16384;
    }
    return b < 8192 ? 8192 : b;
}

void mma_launch(bool bwd, const MmaProblem& p, const MmaTiling& c, int kind, double bytes, cudaStream_t st) {
    Args a;
    memset(&a, 0, sizeof a);
    a.P = p.P; a.K = p.K; a.N = p.N;
    a.KCH = (p.K + 31) / 32;
    int xf;
    if (bwd) {
        a.a = p.dz.dy; a.az = p.dz.z; a.act = p.dz.act;
        a.c0 = p.dz.k1; a.c1 = p.dz.k2; a.c2 = p.dz.k3; a.c3 = p.dz.scale; a.c4 = p.dz.shift;
        a.pb = p.pb;
        xf = p.dz.act != ACT_NONE ? XF_ACT : (p.dz.k1 || p.pb.sums) ? XF_AFFINE : XF_NONE;
    } else {
        a.a = p.x.p; a.act = p.x.act;
        a.c0 = p.x.scale; a.c1 = p.x.shift;
        a.pf = p.pf;
        xf = p.x.act != ACT_NONE ? XF_ACT : (p.x.scale || p.pf.sums) ? XF_AFFINE : XF_NONE;
        if (p.sum_out) {
            xf = p.sum_large ? XF_SUM : XF_ADD;
            a.az = p.x2.p; a.d0 = p.x2.scale; a.d1 = p.x2.shift;
            a.pf2 = p.pf2;
            a.sum_out = (__nv_bfloat16*)p.sum_out;
            a.act = p.sum_act;
        }
    }
    a.w = (const __nv_bfloat16*)p.w; a.bias = p.bias; a.addend = p.addend; a.out = (__nv_bfloat16*)p.out;
    a.WM = c.wm;
    a.wpitch = w_pitch(p.K);
    const int BN = c.nj * 8, BM = c.wk == 1 ? 16 * c.mi * c.wm : 16 * (8 / c.wk);
    a.m_tiles = (p.P + BM - 1) / BM;
    const int ny = (p.N + BN - 1) / BN;
    int gx = a.m_tiles;
    if (c.wk == 1) {
        int cap = sm_count() * c.ctas / ny;
        if (cap < 1) cap = 1;
        if (gx > cap) gx = cap;
    }
    a.so = p.so;
    if (p.red) {
        a.rz = (const __nv_bfloat16*)p.red->z;
        a.r_scale = p.red->scale; a.r_shift = p.red->shift; a.r_mean = p.red->mean; a.r_rstd = p.red->rstd;
        a.r_act = p.red->act;
        a.r_mask = p.red->mask;
    }
    if (bwd) raise_limits<true>();
    else raise_limits<false>();
    a.late = !bwd && c.wk == 1 && gx * ny > sm_count();
    const bool deep = xf == XF_SUM || (deep_layer(bwd, p.P, p.K, c, xf) && a.m_tiles > gx);
    const size_t smem = deep ? deep_smem(bwd, p.K, c, xf) : mma_smem(bwd, p.K, c);
    LaunchScope ls(kind, bytes + (bwd && p.so.sums ? 2.0 * p.P * p.N : 0.0) + (p.sum_out ? 4.0 * p.P * p.K : 0.0), 2.0 * p.P * p.N * p.K, st);
    launch_pdl(bwd ? kernel_for<true>(c, xf, deep) : kernel_for<false>(c, xf, deep), dim3(gx, ny), c.wk == 1 ? 32 * c.wm : 256, smem, st, a);
}

}  // namespace ast
