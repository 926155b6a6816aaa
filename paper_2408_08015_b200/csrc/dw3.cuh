// Depthwise 3x3 convolution, NHWC: pieces shared by the forward and the fused backward kernels (dw3.cu).
//
// A thread owns two channels and a strip of TW pixels and walks down its rows.  Two channels, not four or eight: the nine weights, the
// coefficients of every transform and the nine weight-gradient sums of two channels fit in registers (72 of them), where four channels'
// had to be re-read from shared memory for every row, 72 of the 116 shared-memory/L1 wavefronts a row of the backward took.  A warp's vector
// is then 128 (bf16) or 256 (float) consecutive bytes, still whole sectors.
#pragma once
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
// k1, k2, k3, scale, shift of the gradient's transform -> [5][width]
__device__ __forceinline__ void stage_grad(const GradSrc& g, const BnPendBwd& p, int c0, int width, int c, bool write, float* s) {
    for (int i = threadIdx.x; i < width; i += blockDim.x) {
        const int ch = c0 + i;
        float3 k = make_float3(1.f, 0.f, 0.f);
        float sc = 1.f, sh = 0.f;
        if (ch < c) {
            if (p.sums) k = bn_bwd_coef(p, ch, write);
            else if (g.k1) k = make_float3(g.k1[ch], g.k2[ch], g.k3[ch]);
            if (g.scale) {
                sc = g.scale[ch];
                sh = g.shift[ch];
            }
        }
        s[i] = k.x;
        s[width + i] = k.y;
        s[2 * width + i] = k.z;
        s[3 * width + i] = sc;
        s[4 * width + i] = sh;
    }
}

// Sum over the block's threads that own the same channels (tid % lanes), in thread order, of N pairs per thread; channel c's sum k goes to
// acc[k * c_total + c0 + c].  red: N * blockDim.x pairs.
template <int N> __device__ __forceinline__ void block_sums(const float2* v, int lanes, int rows, int c0, int c, double* acc, float* red) {
    const int width = 2 * lanes, pitch = 2 * lanes * rows;
    __syncthreads();
    if ((int)threadIdx.x < lanes * rows)
#pragma unroll
        for (int k = 0; k < N; ++k) *reinterpret_cast<float2*>(red + k * pitch + threadIdx.x * 2) = v[k];
    __syncthreads();
    for (int i = threadIdx.x; i < N * width; i += blockDim.x) {
        const int k = i / width, j = i - k * width;
        if (c0 + j < c) {
            float s = 0.f;
            for (int r = 0; r < rows; ++r) s += red[k * pitch + r * width + j];
            add_sum(acc + (size_t)k * c + c0 + j, s);
        }
    }
}

}  // namespace dw
}  // namespace ast
