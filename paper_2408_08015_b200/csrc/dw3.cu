// Depthwise 3x3 convolution (pad 1, stride 1 or 2), NHWC, float32 and bfloat16: forward and the fused backward.
//
// Forward: out = conv(act(x*scale + shift)), with the statistics of its output.  Backward: one pass over the output gradient and its raw
// output, and over the raw input x of the layer, gives the input gradient, the weight gradient and the two BatchNorm-backward sums of the
// unit in front: an input position (h, w) meets the same 3x3 window of dz for dx (times the weights) and for the weight gradient
// (times x), and x's raw value is also what that unit's sums need.
//
// These layers move 2 (forward) or 4 (backward) tensors and are bound by latency on small maps and by instruction issue on large ones (backward
// of 56x56x144x32: 26 M warp instructions, 55 % of the issue slots with another fifth lost to the packed FMAs' second dispatch cycle, DRAM at a
// quarter): the nine multiply-adds per element and direction are a third of the instructions, the rest converts, masks and addresses.  Hence what keeps
// those few: weights, coefficients and weight-gradient sums in registers (two channels per thread), one kernel per direction so that the
// gradient is transformed once, strips of four pixels (1.5 decoded columns per column), no checks inside strips that fit.
// Measured, one layer in a captured chain with its BatchNorm sums, before -> now (us; before: 4 channels per thread, weights re-read
// from memory or staged for all channels by every block, two or three backward kernels, sums in kernels of their own):
//   bf16 56x56x144 x32   forward 35.1 -> 24.8  backward 101 -> 44      28x28x192 x32  17.7 -> 9.3, 63.6 -> 19.1
//   bf16 stride 2, same  forward 24.4 -> 19.0  backward  79 -> 26.6    112x112x32 x16 17.9 -> 12.2, 62.7 -> 23.0
//   bf16 14x14x384 x4    forward 12.6 ->  3.8  backward  27 ->  5.7    7x7x960 x16    21.5 -> 4.8, 40.6 -> 8.3
//   f32  28x28x144 x16   forward 10.7 ->  5.9  backward  35 -> 13.0    f32 56x56x96 x16  16.8 -> 13.5, 45.5 -> 28.9
#include "dw.cuh"

namespace ast {
namespace {

using namespace dw;
// In all three kernels EX says that the strips cover the columns exactly, so that only the first and the last column a strip reads can lie
// outside the image; the row loop is unrolled by three so that the rotating rows (or accumulators) need no moves.

// ------------------------------------------------------------------------------------------ forward
template <typename T, int S, int TW, bool EX>
__global__ void __launch_bounds__(BT) dw3_fwd_kernel(const DwFwdArgs a) {
    constexpr int NIN = (TW - 1) * S + 3;
    extern __shared__ __align__(16) float sm[];            // scale and shift [2][width]; reused for the sums
    const DwGeom& g = a.g;
    const int jl = threadIdx.x % g.lanes, row = threadIdx.x / g.lanes, width = 2 * g.lanes, cb = blockIdx.y * width, c0 = cb + 2 * jl;
    const bool live = row < g.rows && c0 < g.c;
    const uint32_t cby = g.c * sizeof(T);
    float2 w[9];
    load_weights<9>(a.wkc, g.c, c0, live, w);
    pdl_wait();
    if (!a.late) pdl_launch();
    int item = blockIdx.x * g.rows + row, wo0 = 0, oh0 = 0, oh1 = 0, n = 0;
    uint32_t col[NIN];
    P2<T> nx[NIN];
    auto place = [&] {
        wo0 = (item % g.sw) * TW;
        const int t2 = item / g.sw;
        oh0 = (t2 % g.nrc) * g.th;
        n = t2 / g.nrc;
        oh1 = min(g.ho, oh0 + g.th);
#pragma unroll
        for (int q = 0; q < NIN; ++q) col[q] = (uint32_t)min(max(wo0 * S - 1 + q, 0), g.wi - 1) * cby + c0 * (uint32_t)sizeof(T);
    };
    auto fetch = [&](int ih) {
        const uint32_t rb = (uint32_t)((n * g.hi + min(max(ih, 0), g.hi - 1)) * g.wi) * cby;
#pragma unroll
        for (int q = 0; q < NIN; ++q) nx[q].load(a.x.p, rb + col[q]);
    };
    const bool work = live && item < g.items;
    if (work) {
        place();
        fetch(oh0 * S - 1);
    }
    const bool stats = (bool)a.so.sums;
    float2 piv = stats && live ? ld2(a.so.pivot + c0) : zero2();
    stage_val(a.x, a.pf, cb, width, g.c, a.first && blockIdx.x == 0, sm);
    __syncthreads();
    const float2 sc = ld2(sm + 2 * jl), sh = ld2(sm + width + 2 * jl);
    if (stats && live) {
        if (blockIdx.x == 0 && row == 0) *reinterpret_cast<float2*>(a.so.pivot_copy + c0) = piv;
        piv = make_float2(-piv.x, -piv.y);
    }
    const float blo = a.x.act == ACT_NONE ? -INFINITY : 0.f, bhi = a.x.act == ACT_RELU6 ? 6.f : INFINITY;
    float2 s[2] = {zero2(), zero2()};
    if (work)
        for (;;) {
            // columns outside the image: a clamp to 0..0 in place of the activation's bounds
            float lo[NIN], hi[NIN];
#pragma unroll
            for (int q = 0; q < NIN; ++q) {
                const int wi = wo0 * S - 1 + q;
                const bool ok = (EX && q > 0 && q < NIN - 1) || (wi >= 0 && wi < g.wi);
                lo[q] = ok ? blo : 0.f;
                hi[q] = ok ? bhi : 0.f;
            }
            const int i1 = (oh1 - 1) * S + 1;
            float2 xin[NIN];
            // the row just fetched -> xin, the next one on its way
            auto take = [&](int ih) {
#pragma unroll
                for (int q = 0; q < NIN; ++q) xin[q] = clamp2(__ffma2_rn(nx[q].get(), sc, sh), lo[q], hi[q]);
                if (ih < i1) fetch(ih + 1);
                if (ih < 0 || ih >= g.hi)
#pragma unroll
                    for (int q = 0; q < NIN; ++q) xin[q] = zero2();
            };
            auto taps = [&](int r, float2* ac) {
#pragma unroll
                for (int sx = 0; sx < 3; ++sx)
#pragma unroll
                    for (int t = 0; t < TW; ++t) ac[t] = __ffma2_rn(xin[t * S + sx], w[r * 3 + sx], r == 0 && sx == 0 ? zero2() : ac[t]);
            };
            auto emit = [&](int oh, const float2* ac) {
                const uint32_t ob = (uint32_t)((n * g.ho + oh) * g.wo + wo0) * cby + c0 * (uint32_t)sizeof(T);
#pragma unroll
                for (int t = 0; t < TW; ++t)
                    if (EX || wo0 + t < g.wo) {
                        const float2 v = P2<T>::put(a.out, ob + t * cby, ac[t]);
                        const float2 d = __fadd2_rn(v, piv);
                        s[0] = __fadd2_rn(s[0], d);
                        s[1] = __ffma2_rn(d, d, s[1]);
                    }
            };
            if (S == 1) {
                float2 acc[3][TW];
                // row ih: the first of output ih + 1 (c), the middle one of ih (b) and the last of ih - 1 (a)
                auto step = [&](int ih, float2* pa, float2* pb, float2* pc) {
                    take(ih);
                    taps(2, pa);
                    taps(1, pb);
                    taps(0, pc);
                    if (ih > oh0) emit(ih - 1, pa);
                };
#pragma unroll
                for (int t = 0; t < TW; ++t) acc[0][t] = acc[1][t] = zero2();
                for (int ih = oh0 - 1;;) {
                    step(ih, acc[0], acc[1], acc[2]);
                    if (++ih > i1) break;
                    step(ih, acc[1], acc[2], acc[0]);
                    if (++ih > i1) break;
                    step(ih, acc[2], acc[0], acc[1]);
                    if (++ih > i1) break;
                }
            } else {
                float2 acc[2][TW];
                auto pair = [&](int oh, float2* pa, float2* pb) {  // rows 2*oh and 2*oh + 1; the latter also is the first of oh + 1
                    take(2 * oh);
                    taps(1, pa);
                    take(2 * oh + 1);
                    taps(2, pa);
                    taps(0, pb);
                    emit(oh, pa);
                };
                take(2 * oh0 - 1);
                taps(0, acc[0]);
                for (int oh = oh0;;) {
                    pair(oh, acc[0], acc[1]);
                    if (++oh >= oh1) break;
                    pair(oh, acc[1], acc[0]);
                    if (++oh >= oh1) break;
                }
            }
            item += gridDim.x * g.rows;
            if (item >= g.items) break;
            place();
            fetch(oh0 * S - 1);
        }
    if (a.late) pdl_launch();
    if (stats) block_sums<2>(s, g.lanes, g.rows, cb, g.c, a.so.sums, sm);
}

// ------------------------------------------------------------------------------------------ backward
// Coefficients of a thread's two channels, in registers for the kernel's life: the gradient's transform, the input's, and what the sums
// of the unit in front need.  Two pixels of two channels at a time go through packed arithmetic.
enum { Z_PLAIN = 0, Z_AFFINE = 1, Z_ACT = 2 };          // the gradient's transform: none, BatchNorm's, BatchNorm's behind an activation
template <typename T, int XF> struct BwdCoef {
    float2 k1, k2, k3, zs, zh, sc, sh, rs, rm;
    float zlo, zhi, xlo, xhi;
    // dz = k1*dy*[lo < pre < hi] + k2 + k3*z
    __device__ __forceinline__ float2 grad(const P2<T>& rd, const P2<T>& rz) const {
        float2 o = rd.get();
        if (XF != Z_PLAIN) {
            const float2 z = rz.get();
            if (XF == Z_ACT) {
                const float2 pre = __ffma2_rn(z, zs, zh);
                o.x = pre.x > zlo && pre.x < zhi ? o.x : 0.f;
                o.y = pre.y > zlo && pre.y < zhi ? o.y : 0.f;
            }
            o = __ffma2_rn(k1, o, __ffma2_rn(k3, z, k2));
        }
        return o;
    }
    // dx of a position whose raw input is given: stored, and as stored into the sums
    __device__ __forceinline__ void put(void* p, uint32_t e, float2 dx, const float2& raw, bool mask, float2* s) const {
        const float2 pre = __ffma2_rn(raw, sc, sh), xh = __ffma2_rn(raw, rs, rm);
        const bool mx = pre.x > xlo && pre.x < xhi, my = pre.y > xlo && pre.y < xhi;
        if (mask) dx = make_float2(mx ? dx.x : 0.f, my ? dx.y : 0.f);
        const float2 v = P2<T>::put(p, e, dx);
        float2 d;
        d.x = mx ? v.x : 0.f;
        d.y = my ? v.y : 0.f;
        s[0] = __fadd2_rn(s[0], d);
        s[1] = __ffma2_rn(d, xh, s[1]);
    }
};
// shared memory of a backward block until its sums: gradient coefficients [5][width], input coefficients [4][width]
template <typename T, int XF>
__device__ __forceinline__ BwdCoef<T, XF> bwd_coefs(const DwBwdArgs& a, int cb, int width, int jl, float* sm) {
    stage_bwd(a.dz, a.pb, a.x, a.sums ? a.mean : nullptr, a.sums ? a.rstd : nullptr, cb, width, a.g.c, a.first && blockIdx.x == 0, sm);
    __syncthreads();
    const float* p = sm + 2 * jl;
    BwdCoef<T, XF> k;
    k.k1 = ld2(p);
    k.k2 = ld2(p + width);
    k.k3 = ld2(p + 2 * width);
    k.zs = ld2(p + 3 * width);
    k.zh = ld2(p + 4 * width);
    k.sc = ld2(p + 5 * width);
    k.sh = ld2(p + 6 * width);
    k.rs = ld2(p + 7 * width);
    k.rm = ld2(p + 8 * width);
    k.zlo = a.dz.act == ACT_NONE ? -INFINITY : 0.f;
    k.zhi = a.dz.act == ACT_RELU6 ? 6.f : INFINITY;
    k.xlo = a.x.act == ACT_NONE ? -INFINITY : 0.f;
    k.xhi = a.x.act == ACT_RELU6 ? 6.f : INFINITY;
    return k;
}

template <typename T, int TW, int XF, bool EX>
__global__ void __launch_bounds__(BT, 3) dw3_bwd_s1_kernel(const DwBwdArgs a) {
    constexpr int NZ = TW + 2;
    extern __shared__ __align__(16) float sm[];
    const DwGeom& g = a.g;
    const int jl = threadIdx.x % g.lanes, row = threadIdx.x / g.lanes, width = 2 * g.lanes, cb = blockIdx.y * width, c0 = cb + 2 * jl;
    const bool live = row < g.rows && c0 < g.c;
    const uint32_t cby = g.c * sizeof(T), rby = g.wi * cby;
    float2 w[9], gw[9];
    load_weights<9>(a.wkc, g.c, c0, live, w);
    pdl_wait();
    P2<T> nd[NZ], nz[NZ], nx[TW];
    uint32_t col[NZ];
    int item = blockIdx.x * g.rows + row, wo0 = 0, r0 = 0, r1 = 0, n = 0;
    auto place = [&] {
        wo0 = (item % g.sw) * TW;
        const int t2 = item / g.sw;
        r0 = (t2 % g.nrc) * g.th;
        n = t2 / g.nrc;
        r1 = min(g.hi, r0 + g.th);
#pragma unroll
        for (int q = 0; q < NZ; ++q) col[q] = (uint32_t)min(max(wo0 - 1 + q, 0), g.wi - 1) * cby + c0 * (uint32_t)sizeof(T);
    };
    auto fetch_z = [&](int r) {
        const uint32_t rb = (uint32_t)(n * g.hi + min(max(r, 0), g.hi - 1)) * rby;
#pragma unroll
        for (int q = 0; q < NZ; ++q) {
            nd[q].load(a.dz.dy, rb + col[q]);
            if (XF != Z_PLAIN) nz[q].load(a.dz.z, rb + col[q]);
        }
    };
    auto fetch_x = [&](int r) {
        const uint32_t rb = (uint32_t)(n * g.hi + r) * rby;
#pragma unroll
        for (int t = 0; t < TW; ++t) nx[t].load(a.x.p, rb + col[t + 1]);
    };
    const bool work = live && item < g.items;
    if (work) {
        place();
        fetch_z(r0 - 1);
    }
    const BwdCoef<T, XF> k = bwd_coefs<T, XF>(a, cb, width, jl, sm);
    float2 fs[2] = {zero2(), zero2()};
#pragma unroll
    for (int t = 0; t < 9; ++t) gw[t] = zero2();
    if (work)
        for (;;) {
            float2 dz[3][NZ];
            auto decode = [&](int r, float2* d) {
#pragma unroll
                for (int q = 0; q < NZ; ++q) {
                    d[q] = k.grad(nd[q], nz[q]);
                    if (!(EX && q > 0 && q < NZ - 1) && !(wo0 - 1 + q >= 0 && wo0 - 1 + q < g.wi)) d[q] = zero2();
                }
                if (r < 0 || r >= g.hi)
#pragma unroll
                    for (int q = 0; q < NZ; ++q) d[q] = zero2();
            };
            decode(r0 - 1, dz[0]);
            fetch_z(r0);
            fetch_x(r0);
            decode(r0, dz[1]);
            fetch_z(r0 + 1);
            // input row ih between the gradient rows da (ih - 1), db (ih) and dc (ih + 1, decoded here)
            auto step = [&](int ih, const float2* da, const float2* db, float2* dc) {
                decode(ih + 1, dc);
                float2 raw[TW], xv[TW], o[TW];
#pragma unroll
                for (int t = 0; t < TW; ++t) {
                    const bool ok = EX || wo0 + t < g.wi;
                    raw[t] = nx[t].get();
                    xv[t] = clamp2(__ffma2_rn(raw[t], k.sc, k.sh), ok ? k.xlo : 0.f, ok ? k.xhi : 0.f);
                }
                const uint32_t rb = (uint32_t)(n * g.hi + ih) * rby;
                if (ih + 1 < r1) {
                    fetch_z(ih + 2);
                    fetch_x(ih + 1);
                }
#pragma unroll
                for (int r = 0; r < 3; ++r)
#pragma unroll
                    for (int s = 0; s < 3; ++s)
#pragma unroll
                        for (int t = 0; t < TW; ++t) {
                            const float2 d = (r == 0 ? dc : r == 1 ? db : da)[t + 2 - s];
                            o[t] = __ffma2_rn(d, w[r * 3 + s], r == 0 && s == 0 ? zero2() : o[t]);
                            gw[r * 3 + s] = __ffma2_rn(d, xv[t], gw[r * 3 + s]);
                        }
                if (!a.dx) return;
                if (a.addend) {
                    P2<T> ad[TW];
#pragma unroll
                    for (int t = 0; t < TW; ++t) ad[t].load(a.addend, rb + col[t + 1]);
#pragma unroll
                    for (int t = 0; t < TW; ++t) o[t] = __fadd2_rn(o[t], ad[t].get());
                }
#pragma unroll
                for (int t = 0; t < TW; ++t)
                    if (EX || wo0 + t < g.wi) {
                        k.put(a.dx, rb + col[t + 1], o[t], raw[t], a.mask, fs);
                    }
            };
            for (int ih = r0;;) {
                step(ih, dz[0], dz[1], dz[2]);
                if (++ih >= r1) break;
                step(ih, dz[1], dz[2], dz[0]);
                if (++ih >= r1) break;
                step(ih, dz[2], dz[0], dz[1]);
                if (++ih >= r1) break;
            }
            item += gridDim.x * g.rows;
            if (item >= g.items) break;
            place();
            fetch_z(r0 - 1);
        }
    pdl_launch();
    block_sums<9>(gw, g.lanes, g.rows, cb, g.c, a.gw, sm);  // the staged coefficients are not needed any more
    if (a.sums) block_sums<2>(fs, g.lanes, g.rows, cb, g.c, a.sums, sm);
}

// Stride 2: dz(i, j) meets input rows 2i-1..2i+1 and columns 2j-1..2j+1, so the 2x2 input positions (2i + a, 2j + b) need dz(i, j), and where
// a or b is 1 also dz(i+1, .) and dz(., j+1).  A thread owns TZ columns of dz = 2*TZ input columns and walks down the rows of dz.
template <typename T, int TZ, int XF, bool EX>
__global__ void __launch_bounds__(BT, 3) dw3_bwd_s2_kernel(const DwBwdArgs a) {
    extern __shared__ __align__(16) float sm[];
    const DwGeom& g = a.g;
    const int jl = threadIdx.x % g.lanes, row = threadIdx.x / g.lanes, width = 2 * g.lanes, cb = blockIdx.y * width, c0 = cb + 2 * jl;
    const bool live = row < g.rows && c0 < g.c;
    const uint32_t cby = g.c * sizeof(T);
    float2 w[9], gw[9];
    load_weights<9>(a.wkc, g.c, c0, live, w);
    pdl_wait();
    P2<T> nd[TZ + 1], nz[TZ + 1], nx[2][2 * TZ];
    uint32_t zcol[TZ + 1], xcol[2 * TZ];
    int item = blockIdx.x * g.rows + row, j0 = 0, r0 = 0, r1 = 0, n = 0;
    auto place = [&] {
        j0 = (item % g.sw) * TZ;
        const int t2 = item / g.sw;
        r0 = (t2 % g.nrc) * g.th;
        n = t2 / g.nrc;
        r1 = min(g.ho, r0 + g.th);
#pragma unroll
        for (int q = 0; q <= TZ; ++q) zcol[q] = (uint32_t)min(j0 + q, g.wo - 1) * cby + c0 * (uint32_t)sizeof(T);
#pragma unroll
        for (int q = 0; q < 2 * TZ; ++q) xcol[q] = (uint32_t)min(2 * j0 + q, g.wi - 1) * cby + c0 * (uint32_t)sizeof(T);
    };
    auto x_base = [&](int r) { return (uint32_t)((n * g.hi + min(r, g.hi - 1)) * g.wi) * cby; };
    auto fetch_z = [&](int r) {
        const uint32_t rb = (uint32_t)((n * g.ho + min(r, g.ho - 1)) * g.wo) * cby;
#pragma unroll
        for (int q = 0; q <= TZ; ++q) {
            nd[q].load(a.dz.dy, rb + zcol[q]);
            if (XF != Z_PLAIN) nz[q].load(a.dz.z, rb + zcol[q]);
        }
    };
    auto fetch_x = [&](int i) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t rb = x_base(2 * i + h);
#pragma unroll
            for (int q = 0; q < 2 * TZ; ++q) nx[h][q].load(a.x.p, rb + xcol[q]);
        }
    };
    const bool work = live && item < g.items;
    if (work) {
        place();
        fetch_z(r0);
    }
    const BwdCoef<T, XF> k = bwd_coefs<T, XF>(a, cb, width, jl, sm);
    float2 fs[2] = {zero2(), zero2()};
#pragma unroll
    for (int t = 0; t < 9; ++t) gw[t] = zero2();
    if (work)
        for (;;) {
            float2 dz[2][TZ + 1];
            auto decode = [&](int r, float2* d) {
#pragma unroll
                for (int q = 0; q <= TZ; ++q) {
                    d[q] = k.grad(nd[q], nz[q]);
                    if (!(EX && q < TZ) && j0 + q >= g.wo) d[q] = zero2();
                }
                if (r >= g.ho)
#pragma unroll
                    for (int q = 0; q <= TZ; ++q) d[q] = zero2();
            };
            fetch_x(r0);
            decode(r0, dz[0]);
            fetch_z(r0 + 1);
            // input rows 2*i, 2*i + 1 from the gradient rows i (cur) and i + 1 (nxt, decoded here)
            auto step = [&](int i, const float2* cur, float2* nxt) {
                decode(i + 1, nxt);
                float2 raw[2][2 * TZ];
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int q = 0; q < 2 * TZ; ++q) raw[h][q] = nx[h][q].get();
                if (i + 1 < r1) {
                    fetch_z(i + 2);
                    fetch_x(i + 1);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const bool rok = h == 0 || 2 * i + 1 < g.hi;
                    float2 o[2 * TZ];
                    bool ok[2 * TZ];
#pragma unroll
                    for (int q = 0; q < 2 * TZ; ++q) {
                        const int j = q >> 1;
                        ok[q] = rok && ((EX && q < 2 * TZ - 1) || 2 * j0 + q < g.wi);
                        const float2 xv = clamp2(__ffma2_rn(raw[h][q], k.sc, k.sh), ok[q] ? k.xlo : 0.f, ok[q] ? k.xhi : 0.f);
                        auto tap = [&](int t, const float2& d, bool first = false) {
                            o[q] = __ffma2_rn(d, w[t], first ? zero2() : o[q]);
                            gw[t] = __ffma2_rn(d, xv, gw[t]);
                        };
                        if (h == 0 && (q & 1) == 0) {
                            tap(4, cur[j], true);
                        } else if (h == 0) {
                            tap(5, cur[j], true);
                            tap(3, cur[j + 1]);
                        } else if ((q & 1) == 0) {
                            tap(7, cur[j], true);
                            tap(1, nxt[j]);
                        } else {
                            tap(8, cur[j], true);
                            tap(6, cur[j + 1]);
                            tap(2, nxt[j]);
                            tap(0, nxt[j + 1]);
                        }
                    }
                    if (!a.dx) continue;
                    const uint32_t rb = x_base(2 * i + h);
                    if (a.addend) {
                        P2<T> ad[2 * TZ];
#pragma unroll
                        for (int q = 0; q < 2 * TZ; ++q) ad[q].load(a.addend, rb + xcol[q]);
#pragma unroll
                        for (int q = 0; q < 2 * TZ; ++q) o[q] = __fadd2_rn(o[q], ad[q].get());
                    }
#pragma unroll
                    for (int q = 0; q < 2 * TZ; ++q)
                        if (ok[q]) {
                            k.put(a.dx, rb + xcol[q], o[q], raw[h][q], a.mask, fs);
                        }
                }
            };
            for (int i = r0;;) {
                step(i, dz[0], dz[1]);
                if (++i >= r1) break;
                step(i, dz[1], dz[0]);
                if (++i >= r1) break;
            }
            item += gridDim.x * g.rows;
            if (item >= g.items) break;
            place();
            fetch_z(r0);
        }
    pdl_launch();
    block_sums<9>(gw, g.lanes, g.rows, cb, g.c, a.gw, sm);
    if (a.sums) block_sums<2>(fs, g.lanes, g.rows, cb, g.c, a.sums, sm);
}

// (also of dw5.cu) gw[c][t] = acc[t][c] for the weight gradients of several layers at once
__global__ void __launch_bounds__(256) dw_settle_kernel(const ChanSums acc, const DwSettle* __restrict__ tab, int layers, float* __restrict__ g) {
    pdl_wait();
    pdl_launch();
    int i = blockIdx.x * 256 + threadIdx.x;
    for (int l = 0; l < layers; ++l) {
        const DwSettle e = tab[l];
        const int n = e.taps * e.c;
        if (i < n) {
            const int c = i / e.taps, t = i - e.taps * c;
            const int at = (int)(e.acc_off + (size_t)t * e.c + c);
            const longlong2 n = acc.near[at];
            g[e.g_off + i] = (float)(n.x & 1 ? full_totals(acc.near, acc.far, acc.shift, at, at).x : near_total(n, acc.shift));
            return;
        }
        i -= n;
    }
}

}  // namespace

void dw3_fwd(int dtype, const ConvGeom& g, const ValSrc& x, const BnPendFwd& pf, const float* wkc, void* z, const BnSumsOut& so, const DwTiling& t, cudaStream_t st) {
    typedef void (*Fn)(const DwFwdArgs);
    using B = __nv_bfloat16;
    Fn f;
    const bool ex = g.wo % t.tw == 0;
#define DW3_FWD(T, S, TW) (ex ? (Fn)dw3_fwd_kernel<T, S, TW, true> : (Fn)dw3_fwd_kernel<T, S, TW, false>)
    if (dtype == 0) f = g.stride == 2 ? DW3_FWD(float, 2, 2) : DW3_FWD(float, 1, 4);
    else f = g.stride == 2 ? DW3_FWD(B, 2, 2) : DW3_FWD(B, 1, 4);
#undef DW3_FWD
    const double in_e = (double)g.hi * g.wi * g.ci, out_e = (double)g.ho * g.wo * g.ci;
    const int chunk = image_chunk(dtype, g), launches = (g.n + chunk - 1) / chunk;
    for (int n0 = 0; n0 < g.n; n0 += chunk) {
        const int n = g.n - n0 < chunk ? g.n - n0 : chunk;
        DwFwdArgs a{};
        a.x = x; a.pf = pf; a.wkc = wkc; a.so = so; a.first = n0 == 0;
        a.x.p = at(x.p, (size_t)n0 * g.hi * g.wi * g.ci, dtype);
        a.out = (void*)at(z, (size_t)n0 * g.ho * g.wo * g.ci, dtype);
        DwGeom& d = a.g;
        d = DwGeom{n, g.hi, g.wi, g.ho, g.wo, g.ci, 0, 0, t.th, (g.ho + t.th - 1) / t.th, (g.wo + t.tw - 1) / t.tw, 0};
        d.items = n * d.nrc * d.sw;
        cut_channels(d);
        LaunchScope ls(K_DW_FWD, n * (in_e + out_e) * esz(dtype) + 36.0 * g.ci, 18.0 * n * out_e, st);
        const dim3 grid = cut_grid(d, t.ctas, launches);
        a.late = (int)(grid.x * grid.y) <= 3 * sm_count();
        launch_pdl(f, grid, BT, (size_t)BT * 2 * 2 * 4, st, a);
    }
}

void dw3_bwd(int dtype, const ConvGeom& g, const GradSrc& dz, const BnPendBwd& pb, const ValSrc& x, const float* wkc, const void* addend, void* dx, const ChanSums& gw,
             const ChanSums& sums, const float* mean, const float* rstd, bool mask, const DwTiling& t, cudaStream_t st) {
    typedef void (*Fn)(const DwBwdArgs);
    using B = __nv_bfloat16;
    const int xf = dz.act != ACT_NONE ? Z_ACT : dz.k1 || pb.sums ? Z_AFFINE : Z_PLAIN;
    Fn f;
    const bool ex = (g.stride == 1 ? g.wi : g.wo) % t.tw == 0;
#define DW3_X(K, T, TW, XF) (ex ? (Fn)K<T, TW, XF, true> : (Fn)K<T, TW, XF, false>)
#define DW3_BWD(K, T, TW) (xf == Z_ACT ? DW3_X(K, T, TW, Z_ACT) : xf == Z_AFFINE ? DW3_X(K, T, TW, Z_AFFINE) : DW3_X(K, T, TW, Z_PLAIN))
    if (g.stride == 1) f = dtype == 0 ? DW3_BWD(dw3_bwd_s1_kernel, float, 2) : t.tw == 4 ? DW3_BWD(dw3_bwd_s1_kernel, B, 4) : DW3_BWD(dw3_bwd_s1_kernel, B, 2);
    else f = dtype == 0 ? DW3_BWD(dw3_bwd_s2_kernel, float, 2) : DW3_BWD(dw3_bwd_s2_kernel, B, 2);
#undef DW3_BWD
#undef DW3_X
    const int rows_out = g.stride == 1 ? g.hi : g.ho, cols_out = g.stride == 1 ? g.wi : g.wo;
    const double in_e = (double)g.hi * g.wi * g.ci, out_e = (double)g.ho * g.wo * g.ci;
    const int chunk = image_chunk(dtype, g), launches = (g.n + chunk - 1) / chunk;
    for (int n0 = 0; n0 < g.n; n0 += chunk) {
        const int n = g.n - n0 < chunk ? g.n - n0 : chunk;
        const size_t ie = (size_t)n0 * g.hi * g.wi * g.ci, oe = (size_t)n0 * g.ho * g.wo * g.ci;
        DwBwdArgs a{};
        a.dz = dz; a.pb = pb; a.x = x; a.wkc = wkc; a.gw = gw; a.sums = dx ? sums : ChanSums{}; a.mean = mean; a.rstd = rstd; a.mask = mask; a.first = n0 == 0;
        a.dz.dy = at(dz.dy, oe, dtype);
        a.dz.z = at(dz.z, oe, dtype);
        a.x.p = at(x.p, ie, dtype);
        a.addend = at(addend, ie, dtype);
        a.dx = (void*)at(dx, ie, dtype);
        DwGeom& d = a.g;
        d = DwGeom{n, g.hi, g.wi, g.ho, g.wo, g.ci, 0, 0, t.th, (rows_out + t.th - 1) / t.th, (cols_out + t.tw - 1) / t.tw, 0};
        d.items = n * d.nrc * d.sw;
        cut_channels(d);
        LaunchScope ls(K_DW_BWD_FUSED, n * (out_e * (xf ? 2.0 : 1.0) + in_e * (dx ? (addend ? 3.0 : 2.0) : 1.0)) * esz(dtype) + 36.0 * g.ci, 36.0 * n * out_e, st);
        launch_pdl(f, cut_grid(d, t.ctas, launches), BT, (size_t)BT * 2 * 9 * 4, st, a);
    }
}

void dw_settle(const ChanSums& acc, const DwSettle* tab, int layers, size_t total, float* g, cudaStream_t st) {
    LaunchScope ls(K_DW_BWD_WEIGHT_FINISH, 20.0 * total, 0.0, st);
    launch_pdl(dw_settle_kernel, (unsigned)((total + 255) / 256), 256, 0, st, acc, tab, layers, g);
}

// Strips of 4 pixels (2 where registers or the halo do not allow 4) and the height that makes the longest chain of row steps cheapest.
// In units of a block's issue time for one row: a forward row takes max(3.7, r) with r blocks on the multiprocessor (3.7: the latency of a
// row, hidden from the fourth block on), a backward row of 2-pixel strips max(1.2, r) and one of 4-pixel strips 5 (three blocks saturate
// it).  A strip pays for its halo rows (2 forward, 0.8 and 0.5 backward), so tall strips win until a multiprocessor would run dry.
// Fitted to 1 700 timings (maps of 7 to 112, 24 to 960 channels, 4 to 32 images): within 3 % of the best tiling on average.
DwTiling dw3_choose(int dtype, bool bwd, const ConvGeom& g) {
    DwGeom d{};
    d.c = g.ci;
    cut_channels(d);
    const int gy = (g.ci / 2 + d.lanes - 1) / d.lanes, sms = sm_count();
    const int rows = g.stride == 1 ? g.hi : g.ho, cols = g.stride == 1 ? g.wi : g.wo, occ = bwd ? 3 : dtype == 0 && g.stride == 1 ? 4 : 5;
    DwTiling best{};
    double best_t = 0;
    for (int tw = g.stride == 2 || (bwd && dtype == 0) ? 2 : 4; tw >= (bwd ? 2 : g.stride == 2 ? 2 : 4); tw -= 2)
        for (int th = !bwd && g.stride == 1 && rows > 1 ? 2 : 1; th <= rows && th <= 64; ++th) {
            const long long items = (long long)g.n * ((rows + th - 1) / th) * ((cols + tw - 1) / tw), gx = (items + d.rows - 1) / d.rows;
            double t;
            if (!bwd) {
                const long long per = (gx * gy + sms - 1) / sms, full = per / occ, rem = per % occ;
                t = (th + 2) * ((double)full * (occ > 3.7 ? occ : 3.7) + (rem ? (rem > 3.7 ? (double)rem : 3.7) : 0.0));
            } else {
                const long long cap = sms * occ / gy > 0 ? sms * occ / gy : 1, used = gx < cap ? gx : cap, turns = (gx + used - 1) / used;
                const double r = (double)((used * gy + sms - 1) / sms);
                t = g.stride == 1 ? turns * (th + 0.8) * (tw == 4 ? 5.0 : r > 1.2 ? r : 1.2) : turns * (th + 0.5);
            }
            if (best.tw == 0 || t < best_t) {
                best = DwTiling{tw, th, bwd ? occ : 1 << 16};
                best_t = t;
            }
        }
    return best;
}

}  // namespace ast
