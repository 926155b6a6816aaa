// Depthwise 5x5 convolution (pad 2, stride 1 or 2), NHWC, float32 and bfloat16: forward and the fused backward.
//
// 25 multiply-adds per element and direction: these layers are bound by arithmetic issue (28x28x240 at 32 images: 4 us of FMAs forward, 8
// backward, against 4 to 7 us of memory), once nothing else gets in their way.  Before, the weights were read from memory for every row and
// strip, every output row re-read its five input rows, and backward ran as data, weight and finishing kernels.  As in dw3.cu a thread owns its
// channels' weights in registers and walks down a strip, rows rotate through registers by unrolling, pending coefficients are formed in the prologue
// and channel sums taken from the results.  The forward has two channels per thread; the backward, which holds the 25 weights, the 25 sums and
// a five-row window, has one.
// Measured, one layer with its BatchNorm sums in a captured chain, bf16, before -> now (us): 28x28x240 x32 forward 68.8 -> 20.4, backward
// 217 -> 47.6; 56x56x144 x32 stride 2 74.0 -> 22.5, 249 -> 49.9; 28x28x240 x4 17 -> 6.3, 60 -> 11; 14x14x480 x16 24.5 -> 9.1, 71.5 -> 14.2.
#include "dw.cuh"

namespace ast {
namespace {

using namespace dw;

// one channel of either storage type
template <typename T> struct P1;
template <> struct P1<float> {
    float r;
    __device__ __forceinline__ void load(const void* p, uint32_t e) { r = *reinterpret_cast<const float*>(reinterpret_cast<const char*>(p) + e); }
    __device__ __forceinline__ float get() const { return r; }
    static __device__ __forceinline__ float put(void* p, uint32_t e, float f) {
        *reinterpret_cast<float*>(reinterpret_cast<char*>(p) + e) = f;
        return f;
    }
};
template <> struct P1<__nv_bfloat16> {
    unsigned short r;
    __device__ __forceinline__ void load(const void* p, uint32_t e) { r = *reinterpret_cast<const unsigned short*>(reinterpret_cast<const char*>(p) + e); }
    __device__ __forceinline__ float get() const { return __uint_as_float((uint32_t)r << 16); }
    static __device__ __forceinline__ float put(void* p, uint32_t e, float f) {
        const __nv_bfloat16 v = __float2bfloat16_rn(f);
        *reinterpret_cast<__nv_bfloat16*>(reinterpret_cast<char*>(p) + e) = v;
        return __bfloat162float(v);
    }
};

// EX: the strips cover the columns exactly, only the two first and two last columns a strip reads can lie outside the image.
// ------------------------------------------------------------------------------------------ forward
template <typename T, int S, int TW, bool EX>
__global__ void __launch_bounds__(BT) dw5_fwd_kernel(const DwFwdArgs a) {
    constexpr int NIN = (TW - 1) * S + 5;
    extern __shared__ __align__(16) float sm[];            // scale and shift [2][width]; reused for the sums
    const DwGeom& g = a.g;
    const int jl = threadIdx.x % g.lanes, row = threadIdx.x / g.lanes, width = 2 * g.lanes, cb = blockIdx.y * width, c0 = cb + 2 * jl;
    const bool live = row < g.rows && c0 < g.c;
    const uint32_t cby = g.c * sizeof(T);
    float2 w[25];
    load_weights<25>(a.wkc, g.c, c0, live, w);
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
        for (int q = 0; q < NIN; ++q) col[q] = (uint32_t)min(max(wo0 * S - 2 + q, 0), g.wi - 1) * cby + c0 * (uint32_t)sizeof(T);
    };
    auto fetch = [&](int ih) {
        const uint32_t rb = (uint32_t)((n * g.hi + min(max(ih, 0), g.hi - 1)) * g.wi) * cby;
#pragma unroll
        for (int q = 0; q < NIN; ++q) nx[q].load(a.x.p, rb + col[q]);
    };
    const bool work = live && item < g.items;
    if (work) {
        place();
        fetch(oh0 * S - 2);
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
            const int i1 = (oh1 - 1) * S + 2;
            float2 xin[NIN];
            auto take = [&](int ih) {                      // the row just fetched -> xin, the next one on its way
#pragma unroll
                for (int q = 0; q < NIN; ++q) {
                    const int wi = wo0 * S - 2 + q;
                    const bool ok = (EX && q > 1 && q < NIN - 2) || (wi >= 0 && wi < g.wi);
                    xin[q] = clamp2(__ffma2_rn(nx[q].get(), sc, sh), ok ? blo : 0.f, ok ? bhi : 0.f);
                }
                if (ih < i1) fetch(ih + 1);
                if (ih < 0 || ih >= g.hi)
#pragma unroll
                    for (int q = 0; q < NIN; ++q) xin[q] = zero2();
            };
            auto taps = [&](int r, float2* ac) {
#pragma unroll
                for (int sx = 0; sx < 5; ++sx)
#pragma unroll
                    for (int t = 0; t < TW; ++t) ac[t] = __ffma2_rn(xin[t * S + sx], w[r * 5 + sx], r == 0 && sx == 0 ? zero2() : ac[t]);
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
                // input row ih is the last tap row of output ih - 2 and the first of ih + 2; accumulators rotate
                float2 acc[5][TW];
#pragma unroll
                for (int k = 0; k < 4; ++k)
#pragma unroll
                    for (int t = 0; t < TW; ++t) acc[k][t] = zero2();
                auto step = [&](int ih, float2* p0, float2* p1, float2* p2, float2* p3, float2* p4) {
                    take(ih);
                    taps(4, p0);
                    taps(3, p1);
                    taps(2, p2);
                    taps(1, p3);
                    taps(0, p4);
                    if (ih - 2 >= oh0) emit(ih - 2, p0);
                };
                for (int ih = oh0 - 2;;) {
                    step(ih, acc[0], acc[1], acc[2], acc[3], acc[4]);
                    if (++ih > i1) break;
                    step(ih, acc[1], acc[2], acc[3], acc[4], acc[0]);
                    if (++ih > i1) break;
                    step(ih, acc[2], acc[3], acc[4], acc[0], acc[1]);
                    if (++ih > i1) break;
                    step(ih, acc[3], acc[4], acc[0], acc[1], acc[2]);
                    if (++ih > i1) break;
                    step(ih, acc[4], acc[0], acc[1], acc[2], acc[3]);
                    if (++ih > i1) break;
                }
            } else {
                // rows 2q and 2q + 1: tap rows 4 | 2, 3 | 0, 1 of outputs q - 1 | q | q + 1
                float2 acc[3][TW];
                auto pair = [&](int q, float2* pa, float2* pb, float2* pc) {
                    take(2 * q);
                    taps(4, pa);
                    taps(2, pb);
                    taps(0, pc);
                    if (q - 1 >= oh0) emit(q - 1, pa);
                    if (q >= oh1) return;
                    take(2 * q + 1);
                    taps(3, pb);
                    taps(1, pc);
                };
#pragma unroll
                for (int t = 0; t < TW; ++t) acc[0][t] = acc[1][t] = zero2();
                for (int q = oh0 - 1;;) {
                    pair(q, acc[0], acc[1], acc[2]);
                    if (++q > oh1) break;
                    pair(q, acc[1], acc[2], acc[0]);
                    if (++q > oh1) break;
                    pair(q, acc[2], acc[0], acc[1]);
                    if (++q > oh1) break;
                }
            }
            item += gridDim.x * g.rows;
            if (item >= g.items) break;
            place();
            fetch(oh0 * S - 2);
        }
    if (a.late) pdl_launch();
    if (stats) block_sums<2>(s, g.lanes, g.rows, cb, g.c, a.so.sums, sm);
}

// ------------------------------------------------------------------------------------------ backward
enum { Z_PLAIN = 0, Z_AFFINE = 1, Z_ACT = 2 };
// coefficients of a thread's channel: the gradient's transform, the input's, and what the sums of the unit in front need
template <typename T, int XF> struct Coef1 {
    float k1, k2, k3, zs, zh, sc, sh, rs, rm, zlo, zhi, xlo, xhi;
    __device__ __forceinline__ float grad(const P1<T>& rd, const P1<T>& rz) const {
        const float d = rd.get();
        if (XF == Z_PLAIN) return d;
        const float z = rz.get(), o = fmaf(k3, z, k2);
        if (XF == Z_AFFINE) return fmaf(k1, d, o);
        const float pre = fmaf(z, zs, zh);
        return pre > zlo && pre < zhi ? fmaf(k1, d, o) : o;
    }
    __device__ __forceinline__ float value(float raw, bool ok) const { return fminf(fmaxf(fmaf(raw, sc, sh), ok ? xlo : 0.f), ok ? xhi : 0.f); }
    __device__ __forceinline__ void add(float dx, float raw, float* s) const {
        const float pre = fmaf(raw, sc, sh), d = pre > xlo && pre < xhi ? dx : 0.f;
        s[0] += d;
        s[1] = fmaf(d, fmaf(raw, rs, rm), s[1]);
    }
};
template <typename T, int XF> __device__ __forceinline__ Coef1<T, XF> coefs1(const DwBwdArgs& a, int cb, int width, int jl, float* sm) {
    stage_bwd(a.dz, a.pb, a.x, a.sums ? a.mean : nullptr, a.sums ? a.rstd : nullptr, cb, width, a.g.c, a.first && blockIdx.x == 0, sm);
    __syncthreads();
    const float* p = sm + jl;
    Coef1<T, XF> k;
    k.k1 = p[0];
    k.k2 = p[width];
    k.k3 = p[2 * width];
    k.zs = p[3 * width];
    k.zh = p[4 * width];
    k.sc = p[5 * width];
    k.sh = p[6 * width];
    k.rs = p[7 * width];
    k.rm = p[8 * width];
    k.zlo = a.dz.act == ACT_NONE ? -INFINITY : 0.f;
    k.zhi = a.dz.act == ACT_RELU6 ? 6.f : INFINITY;
    k.xlo = a.x.act == ACT_NONE ? -INFINITY : 0.f;
    k.xhi = a.x.act == ACT_RELU6 ? 6.f : INFINITY;
    return k;
}

template <typename T, int TW, int XF, bool EX>
__global__ void __launch_bounds__(BT, 3) dw5_bwd_s1_kernel(const DwBwdArgs a) {
    constexpr int NZ = TW + 4;
    extern __shared__ __align__(16) float sm[];
    const DwGeom& g = a.g;
    const int width = g.lanes, jl = threadIdx.x % width, row = threadIdx.x / width, cb = blockIdx.y * width, c0 = cb + jl;
    const bool live = row < g.rows && c0 < g.c;
    const uint32_t cby = g.c * sizeof(T), rby = g.wi * cby;
    float w[25], gw[25];
#pragma unroll
    for (int t = 0; t < 25; ++t) w[t] = live ? __ldg(a.wkc + (size_t)t * g.c + c0) : 0.f;
    pdl_wait();
    P1<T> nd[NZ], nz[NZ], nx[TW];
    uint32_t col[NZ];
    int item = blockIdx.x * g.rows + row, wo0 = 0, r0 = 0, r1 = 0, n = 0;
    auto place = [&] {
        wo0 = (item % g.sw) * TW;
        const int t2 = item / g.sw;
        r0 = (t2 % g.nrc) * g.th;
        n = t2 / g.nrc;
        r1 = min(g.hi, r0 + g.th);
#pragma unroll
        for (int q = 0; q < NZ; ++q) col[q] = (uint32_t)min(max(wo0 - 2 + q, 0), g.wi - 1) * cby + c0 * (uint32_t)sizeof(T);
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
        for (int t = 0; t < TW; ++t) nx[t].load(a.x.p, rb + col[t + 2]);
    };
    const bool work = live && item < g.items;
    if (work) {
        place();
        fetch_z(r0 - 2);
    }
    const Coef1<T, XF> k = coefs1<T, XF>(a, cb, width, jl, sm);
    float fs[2] = {0.f, 0.f};
#pragma unroll
    for (int t = 0; t < 25; ++t) gw[t] = 0.f;
    if (work)
        for (;;) {
            float dz[5][NZ];
            auto decode = [&](int r, float* d) {
#pragma unroll
                for (int q = 0; q < NZ; ++q) {
                    d[q] = k.grad(nd[q], nz[q]);
                    if (!(EX && q > 1 && q < NZ - 2) && !(wo0 - 2 + q >= 0 && wo0 - 2 + q < g.wi)) d[q] = 0.f;
                }
                if (r < 0 || r >= g.hi)
#pragma unroll
                    for (int q = 0; q < NZ; ++q) d[q] = 0.f;
            };
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                decode(r0 - 2 + q, dz[q]);
                fetch_z(r0 - 1 + q);
                if (q == 2) fetch_x(r0);
            }
            // input row ih between the gradient rows ih - 2 .. ih + 2 (d0 .. d4, the last decoded here)
            auto step = [&](int ih, const float* d0, const float* d1, const float* d2, const float* d3, float* d4) {
                decode(ih + 2, d4);
                float raw[TW], xv[TW], o[TW];
#pragma unroll
                for (int t = 0; t < TW; ++t) {
                    raw[t] = nx[t].get();
                    xv[t] = k.value(raw[t], EX || wo0 + t < g.wi);
                }
                const uint32_t rb = (uint32_t)(n * g.hi + ih) * rby;
                if (ih + 1 < r1) {
                    fetch_z(ih + 3);
                    fetch_x(ih + 1);
                }
#pragma unroll
                for (int r = 0; r < 5; ++r)
#pragma unroll
                    for (int s = 0; s < 5; ++s)
#pragma unroll
                        for (int t = 0; t < TW; ++t) {
                            const float d = (r == 0 ? d4 : r == 1 ? d3 : r == 2 ? d2 : r == 3 ? d1 : d0)[t + 4 - s];
                            o[t] = fmaf(d, w[r * 5 + s], r == 0 && s == 0 ? 0.f : o[t]);
                            gw[r * 5 + s] = fmaf(d, xv[t], gw[r * 5 + s]);
                        }
                if (!a.dx) return;
#pragma unroll
                for (int t = 0; t < TW; ++t)
                    if (EX || wo0 + t < g.wi) {
                        if (a.addend) {
                            P1<T> ad;
                            ad.load(a.addend, rb + col[t + 2]);
                            o[t] += ad.get();
                        }
                        const float v = P1<T>::put(a.dx, rb + col[t + 2], o[t]);
                        if (a.sums) k.add(v, raw[t], fs);
                    }
            };
            for (int ih = r0;;) {
                step(ih, dz[0], dz[1], dz[2], dz[3], dz[4]);
                if (++ih >= r1) break;
                step(ih, dz[1], dz[2], dz[3], dz[4], dz[0]);
                if (++ih >= r1) break;
                step(ih, dz[2], dz[3], dz[4], dz[0], dz[1]);
                if (++ih >= r1) break;
                step(ih, dz[3], dz[4], dz[0], dz[1], dz[2]);
                if (++ih >= r1) break;
                step(ih, dz[4], dz[0], dz[1], dz[2], dz[3]);
                if (++ih >= r1) break;
            }
            item += gridDim.x * g.rows;
            if (item >= g.items) break;
            place();
            fetch_z(r0 - 2);
        }
    pdl_launch();
    block_sums<25>(gw, g.lanes, g.rows, cb, g.c, a.gw, sm);
    if (a.sums) block_sums<2>(fs, g.lanes, g.rows, cb, g.c, a.sums, sm);
}

// Stride 2: dz(i, j) meets input rows 2i-2..2i+2 and columns 2j-2..2j+2, so the input positions (2i + a, 2j + b) need the rows i+1, i and, where a
// is 0, i-1 (tap rows a, a + 2, 4), and columns likewise.  A thread owns TZ columns of dz = 2*TZ input columns and walks down the rows of dz.
template <typename T, int TZ, int XF, bool EX>
__global__ void __launch_bounds__(BT, 3) dw5_bwd_s2_kernel(const DwBwdArgs a) {
    constexpr int NZ = TZ + 2, NX = 2 * TZ;
    extern __shared__ __align__(16) float sm[];
    const DwGeom& g = a.g;
    const int width = g.lanes, jl = threadIdx.x % width, row = threadIdx.x / width, cb = blockIdx.y * width, c0 = cb + jl;
    const bool live = row < g.rows && c0 < g.c;
    const uint32_t cby = g.c * sizeof(T);
    float w[25], gw[25];
#pragma unroll
    for (int t = 0; t < 25; ++t) w[t] = live ? __ldg(a.wkc + (size_t)t * g.c + c0) : 0.f;
    pdl_wait();
    P1<T> nd[NZ], nz[NZ], nx[2][NX];
    uint32_t zcol[NZ], xcol[NX];
    int item = blockIdx.x * g.rows + row, j0 = 0, r0 = 0, r1 = 0, n = 0;
    auto place = [&] {
        j0 = (item % g.sw) * TZ;
        const int t2 = item / g.sw;
        r0 = (t2 % g.nrc) * g.th;
        n = t2 / g.nrc;
        r1 = min(g.ho, r0 + g.th);
#pragma unroll
        for (int q = 0; q < NZ; ++q) zcol[q] = (uint32_t)min(max(j0 - 1 + q, 0), g.wo - 1) * cby + c0 * (uint32_t)sizeof(T);
#pragma unroll
        for (int q = 0; q < NX; ++q) xcol[q] = (uint32_t)min(2 * j0 + q, g.wi - 1) * cby + c0 * (uint32_t)sizeof(T);
    };
    auto x_base = [&](int r) { return (uint32_t)((n * g.hi + min(r, g.hi - 1)) * g.wi) * cby; };
    auto fetch_z = [&](int r) {
        const uint32_t rb = (uint32_t)((n * g.ho + min(max(r, 0), g.ho - 1)) * g.wo) * cby;
#pragma unroll
        for (int q = 0; q < NZ; ++q) {
            nd[q].load(a.dz.dy, rb + zcol[q]);
            if (XF != Z_PLAIN) nz[q].load(a.dz.z, rb + zcol[q]);
        }
    };
    auto fetch_x = [&](int i) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t rb = x_base(2 * i + h);
#pragma unroll
            for (int q = 0; q < NX; ++q) nx[h][q].load(a.x.p, rb + xcol[q]);
        }
    };
    const bool work = live && item < g.items;
    if (work) {
        place();
        fetch_z(r0 - 1);
    }
    const Coef1<T, XF> k = coefs1<T, XF>(a, cb, width, jl, sm);
    float fs[2] = {0.f, 0.f};
#pragma unroll
    for (int t = 0; t < 25; ++t) gw[t] = 0.f;
    if (work)
        for (;;) {
            float dz[3][NZ];
            auto decode = [&](int r, float* d) {
#pragma unroll
                for (int q = 0; q < NZ; ++q) {
                    d[q] = k.grad(nd[q], nz[q]);
                    if (!(EX && q > 0 && q < NZ - 1) && !(j0 - 1 + q >= 0 && j0 - 1 + q < g.wo)) d[q] = 0.f;
                }
                if (r < 0 || r >= g.ho)
#pragma unroll
                    for (int q = 0; q < NZ; ++q) d[q] = 0.f;
            };
            decode(r0 - 1, dz[0]);
            fetch_z(r0);
            fetch_x(r0);
            decode(r0, dz[1]);
            fetch_z(r0 + 1);
            // input rows 2i, 2i + 1 from the gradient rows i - 1 (dp), i (dc) and i + 1 (dn, decoded here)
            auto step = [&](int i, const float* dp, const float* dc, float* dn) {
                decode(i + 1, dn);
                float raw[2][NX];
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int q = 0; q < NX; ++q) raw[h][q] = nx[h][q].get();
                if (i + 1 < r1) {
                    fetch_z(i + 2);
                    fetch_x(i + 1);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const bool rok = h == 0 || 2 * i + 1 < g.hi;
                    const uint32_t rb = x_base(2 * i + h);
#pragma unroll
                    for (int q = 0; q < NX; ++q) {
                        const int j = q >> 1, b = q & 1;
                        const bool ok = rok && ((EX && q < NX - 1) || 2 * j0 + q < g.wi);
                        const float xv = k.value(raw[h][q], ok);
                        float o = 0.f;
#pragma unroll
                        for (int r = h; r < 5; r += 2)
#pragma unroll
                            for (int s = b; s < 5; s += 2) {
                                const float d = (r < 2 ? dn : r < 4 ? dc : dp)[j + 2 - (s >> 1)];
                                o = fmaf(d, w[r * 5 + s], o);
                                gw[r * 5 + s] = fmaf(d, xv, gw[r * 5 + s]);
                            }
                        if (a.dx && ok) {
                            if (a.addend) {
                                P1<T> ad;
                                ad.load(a.addend, rb + xcol[q]);
                                o += ad.get();
                            }
                            const float v = P1<T>::put(a.dx, rb + xcol[q], o);
                            if (a.sums) k.add(v, raw[h][q], fs);
                        }
                    }
                }
            };
            for (int i = r0;;) {
                step(i, dz[0], dz[1], dz[2]);
                if (++i >= r1) break;
                step(i, dz[1], dz[2], dz[0]);
                if (++i >= r1) break;
                step(i, dz[2], dz[0], dz[1]);
                if (++i >= r1) break;
            }
            item += gridDim.x * g.rows;
            if (item >= g.items) break;
            place();
            fetch_z(r0 - 1);
        }
    pdl_launch();
    block_sums<25>(gw, g.lanes, g.rows, cb, g.c, a.gw, sm);
    if (a.sums) block_sums<2>(fs, g.lanes, g.rows, cb, g.c, a.sums, sm);
}

}  // namespace

void dw5_fwd(int dtype, const ConvGeom& g, const ValSrc& x, const BnPendFwd& pf, const float* wkc, void* z, const BnSumsOut& so, const DwTiling& t, cudaStream_t st) {
    typedef void (*Fn)(const DwFwdArgs);
    using B = __nv_bfloat16;
    const bool ex = g.wo % t.tw == 0;
    Fn f;
#define DW5_FWD(T, S, TW) (ex ? (Fn)dw5_fwd_kernel<T, S, TW, true> : (Fn)dw5_fwd_kernel<T, S, TW, false>)
    if (dtype == 0) f = g.stride == 2 ? DW5_FWD(float, 2, 2) : DW5_FWD(float, 1, 2);
    else f = g.stride == 2 ? DW5_FWD(B, 2, 2) : t.tw == 4 ? DW5_FWD(B, 1, 4) : DW5_FWD(B, 1, 2);
#undef DW5_FWD
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
        LaunchScope ls(K_DW_FWD, n * (in_e + out_e) * esz(dtype) + 100.0 * g.ci, 50.0 * n * out_e, st);
        const dim3 grid = cut_grid(d, t.ctas, launches);
        a.late = (int)(grid.x * grid.y) <= 3 * sm_count();
        launch_pdl(f, grid, BT, (size_t)BT * 2 * 2 * 4, st, a);
    }
}

void dw5_bwd(int dtype, const ConvGeom& g, const GradSrc& dz, const BnPendBwd& pb, const ValSrc& x, const float* wkc, const void* addend, void* dx, const ChanSums& gw,
             const ChanSums& sums, const float* mean, const float* rstd, const DwTiling& t, cudaStream_t st) {
    typedef void (*Fn)(const DwBwdArgs);
    using B = __nv_bfloat16;
    const int xf = dz.act != ACT_NONE ? Z_ACT : (grad_needs_z(dz) || pb.sums) ? Z_AFFINE : Z_PLAIN;
    const bool ex = (g.stride == 1 ? g.wi : g.wo) % t.tw == 0;
    Fn f;
#define DW5_X(K, T, TW, XF) (ex ? (Fn)K<T, TW, XF, true> : (Fn)K<T, TW, XF, false>)
#define DW5_BWD(K, T, TW) (xf == Z_ACT ? DW5_X(K, T, TW, Z_ACT) : xf == Z_AFFINE ? DW5_X(K, T, TW, Z_AFFINE) : DW5_X(K, T, TW, Z_PLAIN))
    if (g.stride == 1) f = dtype == 0 ? (t.tw == 4 ? DW5_BWD(dw5_bwd_s1_kernel, float, 4) : DW5_BWD(dw5_bwd_s1_kernel, float, 2))
                                      : (t.tw == 4 ? DW5_BWD(dw5_bwd_s1_kernel, B, 4) : DW5_BWD(dw5_bwd_s1_kernel, B, 2));
    else f = dtype == 0 ? DW5_BWD(dw5_bwd_s2_kernel, float, 2) : DW5_BWD(dw5_bwd_s2_kernel, B, 2);
#undef DW5_BWD
#undef DW5_X
    const int rows_out = g.stride == 1 ? g.hi : g.ho, cols_out = g.stride == 1 ? g.wi : g.wo;
    const double in_e = (double)g.hi * g.wi * g.ci, out_e = (double)g.ho * g.wo * g.ci;
    const int chunk = image_chunk(dtype, g), launches = (g.n + chunk - 1) / chunk;
    for (int n0 = 0; n0 < g.n; n0 += chunk) {
        const int n = g.n - n0 < chunk ? g.n - n0 : chunk;
        const size_t ie = (size_t)n0 * g.hi * g.wi * g.ci, oe = (size_t)n0 * g.ho * g.wo * g.ci;
        DwBwdArgs a{};
        a.dz = dz; a.pb = pb; a.x = x; a.wkc = wkc; a.gw = gw; a.sums = dx ? sums : ChanSums{}; a.mean = mean; a.rstd = rstd; a.first = n0 == 0;
        a.dz.dy = at(dz.dy, oe, dtype);
        a.dz.z = at(dz.z, oe, dtype);
        a.x.p = at(x.p, ie, dtype);
        a.addend = at(addend, ie, dtype);
        a.dx = (void*)at(dx, ie, dtype);
        DwGeom& d = a.g;
        d = DwGeom{n, g.hi, g.wi, g.ho, g.wo, g.ci, 0, 0, t.th, (rows_out + t.th - 1) / t.th, (cols_out + t.tw - 1) / t.tw, 0};
        d.items = n * d.nrc * d.sw;
        cut_channels(d, 1);
        LaunchScope ls(K_DW_BWD_FUSED, n * (out_e * (xf ? 2.0 : 1.0) + in_e * (dx ? (addend ? 3.0 : 2.0) : 1.0)) * esz(dtype) + 100.0 * g.ci, 100.0 * n * out_e, st);
        launch_pdl(f, cut_grid(d, t.ctas, launches, 1), BT, (size_t)BT * 25 * 4, st, a);
    }
}

// As dw3_choose: the strip whose longest chain of row steps is cheapest, in units of a block's issue time for one row of 2-pixel strips.  Three blocks
// of the register-heavy kernels share a multiprocessor (four of the stride-2 forward); a row takes at least 1.3 (forward) or 2.5 units of latency, a
// row of 4-pixel strips 1.7 times one of 2-pixel strips.  Fitted to 700 timings (maps of 14 to 56, 40 to 480 channels, 1 to 32 images): 4 %
// above the best on average.
DwTiling dw5_choose(int dtype, bool bwd, const ConvGeom& g) {
    const int per = bwd ? 1 : 2;
    DwGeom d{};
    d.c = g.ci;
    cut_channels(d, per);
    const int gy = (g.ci / per + d.lanes - 1) / d.lanes, sms = sm_count();
    const int rows = g.stride == 1 ? g.hi : g.ho, cols = g.stride == 1 ? g.wi : g.wo, occ = !bwd && g.stride == 2 ? 4 : 3;
    const double halo = bwd && g.stride == 2 ? 1.0 : 1.5, lat = !bwd && g.stride == 1 ? 1.3 : 2.5;
    // 4 pixels: stride 1, in registers only where strips need no column checks (backward) or the storage type is small (forward)
    const bool four = g.stride == 1 && (bwd ? cols % 4 == 0 : dtype != 0);
    DwTiling best{};
    double best_t = 0;
    for (int tw = four ? 4 : 2; tw >= 2; tw -= 2)
        for (int th = 1; th <= rows && th <= 64; ++th) {
            const long long items = (long long)g.n * ((rows + th - 1) / th) * ((cols + tw - 1) / tw), gx = (items + d.rows - 1) / d.rows;
            double t = (th + halo) * (tw == 4 ? 1.7 : 1.0);
            if (!bwd) {
                const long long p = (gx * gy + sms - 1) / sms, full = p / occ, rem = p % occ;
                t *= (double)full * (occ > lat ? occ : lat) + (rem ? (rem > lat ? (double)rem : lat) : 0.0);
            } else {
                const long long cap = sms * occ / gy > 0 ? sms * occ / gy : 1, used = gx < cap ? gx : cap, turns = (gx + used - 1) / used;
                const double r = (double)((used * gy + sms - 1) / sms);
                t *= turns * (r > lat ? r : lat);
            }
            if (best.tw == 0 || t < best_t) {
                best = DwTiling{tw, th, bwd ? occ : 1 << 14};
                best_t = t;
            }
        }
    return best;
}

}  // namespace ast
