// Depthwise convolution, NHWC: pieces shared by the 3x3 (dw3.cu) and 5x5 (dw5.cu) kernels.
//
// A thread owns two channels and a strip of TW pixels and walks down its rows.  Two channels, not four or eight: the nine weights, the
// coefficients of every transform and the nine weight-gradient sums of two channels fit in registers (72 of them), where four channels'
// had to be re-read from shared memory for every row, 72 of the 116 shared-memory/L1 wavefronts a row of the backward took.  A warp's vector
// is then 128 (bf16) or 256 (float) consecutive bytes, still whole sectors.
#pragma once
#include <algorithm>

#include "fin.cuh"

namespace ast {
namespace dw {

// two channels of either storage type; offsets in bytes, 32-bit (a launch covers at most 2 GB of a tensor)
template <typename T> struct P2;
template <> struct P2<float> {
    float2 r;
    __device__ __forceinline__ void load(const void* p, uint32_t e) { r = *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(p) + e); }
    __device__ __forceinline__ float2 get() const { return r; }
    // rounds, stores and returns the values as stored
    static __device__ __forceinline__ float2 put(void* p, uint32_t e, float2 f) {
        *reinterpret_cast<float2*>(reinterpret_cast<char*>(p) + e) = f;
        return f;
    }
};
template <> struct P2<__nv_bfloat16> {
    uint32_t r;
    __device__ __forceinline__ void load(const void* p, uint32_t e) { r = *reinterpret_cast<const uint32_t*>(reinterpret_cast<const char*>(p) + e); }
    static __device__ __forceinline__ float2 up(uint32_t w) { return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); }
    __device__ __forceinline__ float2 get() const { return up(r); }
    static __device__ __forceinline__ float2 put(void* p, uint32_t e, float2 f) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(f.x, f.y);
        const uint32_t v = *reinterpret_cast<const uint32_t*>(&a);
        *reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(p) + e) = v;
        return up(v);
    }
};

__device__ __forceinline__ float2 clamp2(float2 v, float lo, float hi) {
    return make_float2(fminf(fmaxf(v.x, lo), hi), fminf(fmaxf(v.y, lo), hi));
}
__device__ __forceinline__ float2 zero2() { return make_float2(0.f, 0.f); }
__device__ __forceinline__ float2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }

// scale and shift of the block's channels -> shared memory [2][width], pending ones formed here
__device__ __forceinline__ void stage_val(const ValSrc& v, const BnPendFwd& p, int c0, int width, int c, bool write, float* s) {
    for (int i = threadIdx.x; i < width; i += blockDim.x) {
        const int ch = c0 + i;
        float2 k = make_float2(1.f, 0.f);
        if (ch < c) {
            if (p.sums) k = bn_fwd_coef(p, ch, write);
            else if (v.scale) k = make_float2(v.scale[ch], v.shift[ch]);
        }
        s[i] = k.x;
        s[width + i] = k.y;
    }
}
// Backward: k1, k2, k3, scale, shift of the gradient's transform, scale and shift of x, rstd and -mean*rstd of the unit that produced x -> [9][width].  All of a
// channel's values are requested before any is used: one after the other they were four trips to memory, 2 us of a kernel of 5.
__device__ __forceinline__ void stage_bwd(const GradSrc& g, const BnPendBwd& p, const ValSrc& x, const float* mean, const float* rstd, int c0, int width, int c, bool write,
                                          float* s) {
    for (int i = threadIdx.x; i < width; i += blockDim.x) {
        const int ch = c0 + i;
        float3 k = make_float3(1.f, 0.f, 0.f);
        float sc = 1.f, sh = 0.f, xs = 1.f, xh = 0.f, r = 0.f, m = 0.f;
        BnBwdIn in;
        if (ch < c) {
            if (p.sums) in.load(p, ch);
            else if (g.k1) k = make_float3(g.k1[ch], g.k2[ch], g.k3[ch]);
            if (g.scale) {
                sc = g.scale[ch];
                sh = g.shift[ch];
            }
            if (x.scale) {
                xs = x.scale[ch];
                xh = x.shift[ch];
            }
            if (rstd) {
                r = rstd[ch];
                m = mean[ch];
            }
            if (p.sums) k = in.coef(p, ch, write);
        }
        s[i] = k.x;
        s[width + i] = k.y;
        s[2 * width + i] = k.z;
        s[3 * width + i] = sc;
        s[4 * width + i] = sh;
        s[5 * width + i] = xs;
        s[6 * width + i] = xh;
        s[7 * width + i] = r;
        s[8 * width + i] = -m * r;
    }
}

// Sum over the block's threads that own the same channels (tid % lanes), in thread order, of N values of V (float: one channel a lane, float2:
// two) per thread; channel c's sum k goes to acc[k * c_total + c0 + c].  red: N * blockDim.x V.
template <int N, typename V> __device__ __forceinline__ void block_sums(const V* v, int lanes, int rows, int c0, int c, const ChanSums& acc, float* red) {
    constexpr int CH = sizeof(V) / 4;
    const int width = CH * lanes, pitch = CH * lanes * rows;
    __syncthreads();
    if ((int)threadIdx.x < lanes * rows)
#pragma unroll
        for (int k = 0; k < N; ++k) *reinterpret_cast<V*>(red + k * pitch + threadIdx.x * CH) = v[k];
    __syncthreads();
    for (int i = threadIdx.x; i < N * width; i += blockDim.x) {
        const int k = i / width, j = i - k * width;
        if (c0 + j < c) {
            float s = 0.f;
            for (int r = 0; r < rows; ++r) s += red[k * pitch + r * width + j];
            add_sum(acc, (size_t)k * c + c0 + j, s);
        }
    }
}

// the thread's N weights of its two channels
template <int N> __device__ __forceinline__ void load_weights(const float* wkc, int c, int c0, bool live, float2* w) {
#pragma unroll
    for (int t = 0; t < N; ++t) w[t] = live ? __ldg(reinterpret_cast<const float2*>(wkc + (size_t)t * c + c0)) : zero2();
}

constexpr int BT = 128;

struct DwGeom {
    int n, hi, wi, ho, wo, c;
    int lanes, rows;             // channel groups per block; strips a block works on side by side
    int th, nrc, sw, items;      // rows per strip, row chunks, strips across, work items
};

struct DwFwdArgs {
    DwGeom g;
    ValSrc x;
    BnPendFwd pf;
    const float* wkc;           // tap-major weights
    void* out;
    BnSumsOut so;
    bool first;                  // writes the pending coefficients out
    bool late;                   // dependents are released when the rows are done (common.cuh)
};

struct DwBwdArgs {
    DwGeom g;
    GradSrc dz;
    BnPendBwd pb;
    ValSrc x;                    // raw input with its (final) coefficients
    const float* wkc;           // tap-major weights
    const void* addend;
    void* dx;                    // may be null: weight gradient only
    ChanSums gw;                 // [taps][c] accumulators of the weight gradient
    ChanSums sums;               // [2][c] of the unit that produced x, or none
    const float *mean, *rstd;    // of that unit
    bool mask;                   // dx is stored as that unit's activation lets it through
    bool first;
};

inline double esz(int dtype) { return dtype == 0 ? 4.0 : 2.0; }

// lanes of a block over the groups of `per` channels: an even split in at most 32
inline void cut_channels(DwGeom& d, int per = 2) {
    const int cv = d.c / per, parts = (cv + 31) / 32;
    d.lanes = (cv + parts - 1) / parts;
    d.rows = BT / d.lanes;
}
// launches: how many of them share the layer's images, and with them the room its sums have
inline dim3 cut_grid(const DwGeom& d, int ctas, int launches, int per = 2) {
    const int gy = (d.c / per + d.lanes - 1) / d.lanes, gx = (d.items + d.rows - 1) / d.rows;
    const int cap = (int)std::min((long long)sm_count() * ctas / gy, (long long)MAX_SUM_BLOCKS / launches);
    return dim3(gx < cap ? gx : cap > 0 ? cap : 1, gy);
}
// images per launch: byte offsets within a launch are 32-bit
inline int image_chunk(int dtype, const ConvGeom& g) {
    const size_t img = (size_t)g.hi * g.wi * g.ci * (dtype == 0 ? 4 : 2), m = 0x7fffffffu / img;
    return m < 1 ? 1 : m < (size_t)g.n ? (int)m : g.n;
}
inline const void* at(const void* p, size_t e, int dtype) { return p ? (const char*)p + e * (dtype == 0 ? 4 : 2) : nullptr; }

}  // namespace dw
}  // namespace ast
