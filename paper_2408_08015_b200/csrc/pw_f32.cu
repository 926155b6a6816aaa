// Pointwise (1x1, stride 1) convolution in float32: forward, backward-data and weight gradient on packed FFMA tiles.
//
//   out[p][n] = sum_k A[p][k] * W[n][k]     forward: A = act(x*scale + shift);  backward: A = BatchNorm/activation backward of (dy, z)
//   gw[k][c]  = sum_p dz[p][k] * x[p][c]
//
// The layers of the float32 path are thin (16 to 192 channels a side), so a layer is 1 to 3 us of arithmetic and of memory each; the general
// implicit-GEMM tile of conv_simt.cu took 15 to 42 us for one: 64-column tiles half empty at 24 channels, an index decomposition with divisions
// and four scalar loads per element, one 16-deep stage in flight, 40 CTAs on 148 multiprocessors, and BatchNorm sums as passes of their own.
// With this file alone a training round of the four-block 56x56 stage at batch 8, 4 micro-batches, went from 3.68 to 2.05 ms, of one block at
// 32x32, batch 8, 4 micro-batches, from 512 to 311 us (with all that came after 1.69 ms and 291 us).
#include <string.h>

#include "pw_mma.cuh"
#include "pw_mma.h"

namespace ast {
namespace {

using mma::cp_async16;
using mma::cp_commit;
using mma::cp_wait;

constexpr int NT = 128;

struct F32Args {
    const float *a, *az;       // [P][K]: x, or dy and z
    const float *c0, *c1, *c2, *c3, *c4;   // forward scale, shift; backward k1, k2, k3, scale, shift (null: identity)
    float lo, hi;              // bounds of the operand's activation
    const float* w;            // [N][K]
    const float* bias;
    const float* addend;
    float* out;
    int P, K, N;
    int bp;                    // floats between the rows of the staged weights
    int m_tiles;
    BnPendFwd pf;
    BnPendFwd pf2;             // a deferred residual sum: the second operand's coefficients (the tensor is az), and where the sum goes
    const float *d0, *d1;
    float* sum_out;
    BnPendBwd pb;
    BnSumsOut so;
    const float* rz;           // backward sums: raw output of the unit whose gradient this is
    const float *r_scale, *r_shift, *r_mean, *r_rstd;
    float r_lo, r_hi;
    bool r_mask;               // the output is stored as that unit's activation lets it through
};

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float clampf(float v, float lo, float hi) { return fminf(fmaxf(v, lo), hi); }
__device__ __forceinline__ float grad1(float d, float z, float k1, float k2, float k3, float s, float h, float lo, float hi) {
    const float pre = fmaf(z, s, h), o = fmaf(k3, z, k2);
    return pre > lo && pre < hi ? fmaf(k1, d, o) : o;
}

// A warp owns 32 pixels x 4*TN columns; lane (r, t) holds pixels r + 8i (i < 4) and TN columns.  The accumulators are pairs over even and odd k, so
// that the float4 fragments of both operands (four k of one row) feed packed FMAs as they are: 4 + TN shared-memory reads for 8*TN of them.
// WK warps share a tile's reduction where the map is small.  The operand goes global -> registers (one chunk ahead) -> transform -> shared memory;
// the weights of the CTA's columns stay in shared memory, row order permuted so that a lane's columns come in groups of G consecutive ones.
// Operand transform: XF_VALUE BatchNorm and activation, XF_ADD (forward) a residual sum, XF_AFFINE (backward) BatchNorm of a gradient stored masked
enum { XF_NONE = 0, XF_VALUE = 1, XF_ADD = 2, XF_AFFINE = 2 };
template <bool BWD, int TN, int WK, int XF>
__global__ void __launch_bounds__(NT) pw_f32_kernel(const F32Args a) {
    if (!BWD) pdl_launch();
    constexpr int WM = 4 / WK, BM = 32 * WM, BK = 16 * WK, AP = BK + 4, QC = BK / 4, BN = 4 * TN, G = TN % 4 == 0 ? 4 : 2, NG = TN / G;
    extern __shared__ __align__(16) float sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, r = lane >> 2, t = lane & 3, wm = warp % WM, wk = warp / WM;
    const int n0 = blockIdx.y * BN, Kp = (a.K + 15) & ~15;
    float* sB = sm;                                        // [BN][bp]
    float* sK = sB + BN * a.bp;                            // operand coefficients [5 | 3][Kp]
    float* sN = sK + (BWD ? 5 : 3) * Kp;                   // column coefficients [4][BN]
    float* sA = sN + 4 * BN;                               // [2][BM][AP]
    float* sR = sA + 2 * BM * AP;                          // partial tiles of the other WK - 1 warps; the column sums [WM][2][BN]
    {
        const int kv = a.K >> 2;
        const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(sB);
        for (int i = tid; i < BN * kv; i += NT) {
            const int sr = i / kv, v = i - sr * kv, j = sr >> 2;
            const int n = n0 + (j / G) * 4 * G + (sr & 3) * G + j % G;
            cp_async16(s0 + (uint32_t)(sr * a.bp + v * 4) * 4u, a.w + (n < a.N ? (size_t)n * a.K + v * 4 : 0), n < a.N);
        }
        cp_commit();
    }
    pdl_wait();

    const int kq = tid % QC, prow = tid / QC;
    const int chunks = (a.K + BK - 1) / BK;
    float4 nx[4], nz[4];
    auto fetch = [&](int tile, int ch) {
        const int k = ch * BK + kq * 4;
        if (k >= a.K) return;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const size_t e = (size_t)min(tile * BM + prow + j * (NT / QC), a.P - 1) * a.K + k;
            nx[j] = ld4(a.a + e);
            if ((BWD && XF) || XF == XF_ADD) nz[j] = ld4(a.az + e);
        }
    };
    int tile = blockIdx.x;
    fetch(tile, 0);
    const bool first = blockIdx.x == 0 && blockIdx.y == 0;
    // everything a thread reads from memory is requested before it uses anything; BN <= NT: a column a thread
    const bool sums = (bool)a.so.sums, col = sums && tid < BN && n0 + tid < a.N;
    float nr = 0.f, ns = 0.f, nh = 0.f, nm = 0.f;
    if (col) {
        if (BWD) {
            nr = a.r_rstd[n0 + tid];
            ns = a.r_scale[n0 + tid];
            nh = a.r_shift[n0 + tid];
            nm = a.r_mean[n0 + tid];
        } else nm = a.so.pivot[n0 + tid];
    }
    if (XF)
        for (int c = tid; c < a.K; c += NT) {
            if (BWD) {
                float3 k = make_float3(1.f, 0.f, 0.f);
                float s = 1.f, h = 0.f;
                BnBwdIn in;
                if (a.pb.sums) in.load(a.pb, c);
                else if (a.c0) k = make_float3(a.c0[c], a.c1[c], a.c2[c]);
                if (a.c3) {
                    s = a.c3[c];
                    h = a.c4[c];
                }
                if (a.pb.sums) k = in.coef(a.pb, c, first);
                sK[c] = k.x;
                sK[Kp + c] = k.y;
                sK[2 * Kp + c] = k.z;
                if (XF == XF_VALUE) {
                    sK[3 * Kp + c] = s;
                    sK[4 * Kp + c] = h;
                }
            } else {
                float2 k = make_float2(1.f, 0.f), k2 = k;
                BnFwdIn in, in2;
                if (a.pf.sums) in.load(a.pf, c, first);
                else if (a.c0) k = make_float2(a.c0[c], a.c1[c]);
                if (XF == XF_ADD) {
                    if (a.pf2.sums) in2.load(a.pf2, c, first);
                    else if (a.d0) k2 = make_float2(a.d0[c], a.d1[c]);
                }
                if (a.pf.sums) k = in.coef(a.pf, c, first);
                sK[c] = k.x;
                if (XF == XF_ADD) {
                    if (a.pf2.sums) k2 = in2.coef(a.pf2, c, first);
                    sK[2 * Kp + c] = k2.x;
                    k.y += k2.y;
                }
                sK[Kp + c] = k.y;
            }
        }
    if (sums && tid < BN) {
        if (BWD) {
            sN[tid] = ns;
            sN[BN + tid] = nh;
            sN[2 * BN + tid] = nr;
            sN[3 * BN + tid] = -nm * nr;
        } else {
            sN[tid] = nm;
            if (col && blockIdx.x == 0) a.so.pivot_copy[n0 + tid] = nm;
        }
    }
    cp_wait<0>();
    __syncthreads();

    float s1[TN], s2[TN];
#pragma unroll
    for (int j = 0; j < TN; ++j) s1[j] = s2[j] = 0.f;
    int buf = 0;
    for (; tile < a.m_tiles; tile += gridDim.x) {
        float2 acc[4][TN];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int ch = 0; ch < chunks; ++ch) {
            float* d = sA + buf * BM * AP;
            const int k = ch * BK + kq * 4;
            if (k < a.K) {
                if (BWD) {
                    float4 k1, k2, k3, s, h;
                    if (XF) {
                        k1 = ld4(sK + k); k2 = ld4(sK + Kp + k); k3 = ld4(sK + 2 * Kp + k);
                    }
                    if (XF == XF_VALUE) {
                        s = ld4(sK + 3 * Kp + k); h = ld4(sK + 4 * Kp + k);
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float4 v = nx[j];
                        if (XF == XF_AFFINE) {
                            v.x = fmaf(k1.x, v.x, fmaf(k3.x, nz[j].x, k2.x));
                            v.y = fmaf(k1.y, v.y, fmaf(k3.y, nz[j].y, k2.y));
                            v.z = fmaf(k1.z, v.z, fmaf(k3.z, nz[j].z, k2.z));
                            v.w = fmaf(k1.w, v.w, fmaf(k3.w, nz[j].w, k2.w));
                        } else if (XF) {
                            v.x = grad1(v.x, nz[j].x, k1.x, k2.x, k3.x, s.x, h.x, a.lo, a.hi);
                            v.y = grad1(v.y, nz[j].y, k1.y, k2.y, k3.y, s.y, h.y, a.lo, a.hi);
                            v.z = grad1(v.z, nz[j].z, k1.z, k2.z, k3.z, s.z, h.z, a.lo, a.hi);
                            v.w = grad1(v.w, nz[j].w, k1.w, k2.w, k3.w, s.w, h.w, a.lo, a.hi);
                        }
                        *reinterpret_cast<float4*>(d + (prow + j * (NT / QC)) * AP + kq * 4) = v;
                    }
                } else {
                    float4 s, h, s2;
                    if (XF) {
                        s = ld4(sK + k); h = ld4(sK + Kp + k);
                        if (XF == XF_ADD) s2 = ld4(sK + 2 * Kp + k);
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float4 v = nx[j];
                        if (XF == XF_ADD) {
                            v.x = clampf(fmaf(v.x, s.x, fmaf(nz[j].x, s2.x, h.x)), a.lo, a.hi);
                            v.y = clampf(fmaf(v.y, s.y, fmaf(nz[j].y, s2.y, h.y)), a.lo, a.hi);
                            v.z = clampf(fmaf(v.z, s.z, fmaf(nz[j].z, s2.z, h.z)), a.lo, a.hi);
                            v.w = clampf(fmaf(v.w, s.w, fmaf(nz[j].w, s2.w, h.w)), a.lo, a.hi);
                            const int p = tile * BM + prow + j * (NT / QC);
                            if (blockIdx.y == 0 && p < a.P) *reinterpret_cast<float4*>(a.sum_out + (size_t)p * a.K + k) = v;
                        } else if (XF) {
                            v.x = clampf(fmaf(v.x, s.x, h.x), a.lo, a.hi);
                            v.y = clampf(fmaf(v.y, s.y, h.y), a.lo, a.hi);
                            v.z = clampf(fmaf(v.z, s.z, h.z), a.lo, a.hi);
                            v.w = clampf(fmaf(v.w, s.w, h.w), a.lo, a.hi);
                        }
                        *reinterpret_cast<float4*>(d + (prow + j * (NT / QC)) * AP + kq * 4) = v;
                    }
                }
            }
            if (ch + 1 < chunks) fetch(tile, ch + 1);
            else if (tile + (int)gridDim.x < a.m_tiles) fetch(tile + gridDim.x, 0);
            __syncthreads();
            const float* ap = d + (wm * 32 + r) * AP + wk * 16;
            const float* bq = sB + t * a.bp + ch * BK + wk * 16;
            const int left = (a.K - ch * BK - wk * 16) >> 2;       // quads of four k this warp still has
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (u >= left) break;
                float4 av[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) av[i] = ld4(ap + 8 * i * AP + 4 * u);
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    const float4 b = ld4(bq + 4 * j * a.bp + 4 * u);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        acc[i][j] = __ffma2_rn(make_float2(av[i].x, av[i].y), make_float2(b.x, b.y), acc[i][j]);
                        acc[i][j] = __ffma2_rn(make_float2(av[i].z, av[i].w), make_float2(b.z, b.w), acc[i][j]);
                    }
                }
            }
            buf ^= 1;
        }
        float v[4][TN];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) v[i][j] = acc[i][j].x + acc[i][j].y;
        if (WK > 1) {
            float* q = sR + (size_t)wm * 32 * 4 * TN + lane;
            if (wk > 0) {
                q += (size_t)(wk - 1) * WM * 32 * 4 * TN;
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < TN; ++j) q[(i * TN + j) * 32] = v[i][j];
            }
            __syncthreads();
            if (wk > 0) continue;
#pragma unroll
            for (int w = 0; w < WK - 1; ++w)
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < TN; ++j) v[i][j] += q[(size_t)w * WM * 32 * 4 * TN + (i * TN + j) * 32];
        }
        // ---- epilogue: groups of G consecutive columns
        const int p0 = tile * BM + wm * 32 + r;
#pragma unroll
        for (int gr = 0; gr < NG; ++gr) {
            const int cl = gr * 4 * G + t * G, n = n0 + cl;
            if (n >= a.N) continue;
            float ad[4][G], rz[4][G];
            auto ldg = [&](const float* p, float (*o)[G]) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float* q = p + (size_t)min(p0 + 8 * i, a.P - 1) * a.N + n;
                    if constexpr (G == 4) {
                        const float4 f = ld4(q);
                        o[i][0] = f.x; o[i][1] = f.y; o[i][2] = f.z; o[i][3] = f.w;
                    } else {
                        const float2 f = *reinterpret_cast<const float2*>(q);
                        o[i][0] = f.x; o[i][1] = f.y;
                    }
                }
            };
            if (BWD && a.addend) ldg(a.addend, ad);
            if (BWD && sums) ldg(a.rz, rz);
#pragma unroll
            for (int q = 0; q < G; ++q) {
                const int j = gr * G + q;
                const float bs = !BWD && a.bias ? __ldg(a.bias + n + q) : 0.f;
                float c0 = 0.f, c1 = 0.f, c2 = 0.f, c3 = 0.f;
                if (sums) {
                    c0 = sN[cl + q];
                    if (BWD) {
                        c1 = sN[BN + cl + q]; c2 = sN[2 * BN + cl + q]; c3 = sN[3 * BN + cl + q];
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (!BWD) v[i][j] += bs;
                    if (BWD && a.addend) v[i][j] += ad[i][q];
                    if (sums && p0 + 8 * i < a.P) {
                        if (BWD) {
                            const float pre = fmaf(rz[i][q], c0, c1), xh = fmaf(rz[i][q], c2, c3), g = pre > a.r_lo && pre < a.r_hi ? v[i][j] : 0.f;
                            s1[j] += g;
                            s2[j] = fmaf(g, xh, s2[j]);
                            if (a.r_mask) v[i][j] = g;
                        } else {
                            const float dd = v[i][j] - c0;
                            s1[j] += dd;
                            s2[j] = fmaf(dd, dd, s2[j]);
                        }
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (p0 + 8 * i >= a.P) continue;
                float* o = a.out + (size_t)(p0 + 8 * i) * a.N + n;
                if constexpr (G == 4) *reinterpret_cast<float4*>(o) = make_float4(v[i][gr * 4], v[i][gr * 4 + 1], v[i][gr * 4 + 2], v[i][gr * 4 + 3]);
                else *reinterpret_cast<float2*>(o) = make_float2(v[i][gr * 2], v[i][gr * 2 + 1]);
            }
        }
    }
    if (BWD) pdl_launch();
    if (!sums) return;
    __syncthreads();                                       // sR: the last tile's partials have been read
    if (wk == 0) {
#pragma unroll
        for (int j = 0; j < TN; ++j) {
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) {
                s1[j] += __shfl_xor_sync(0xffffffffu, s1[j], o);
                s2[j] += __shfl_xor_sync(0xffffffffu, s2[j], o);
            }
        }
        if (r == 0) {
#pragma unroll
            for (int j = 0; j < TN; ++j) {
                const int cl = (j / G) * 4 * G + t * G + j % G;
                sR[(wm * 2) * BN + cl] = s1[j];
                sR[(wm * 2 + 1) * BN + cl] = s2[j];
            }
        }
    }
    __syncthreads();
    for (int i = tid; i < 2 * BN; i += NT) {
        const int s = i >= BN ? 1 : 0, cl = i - s * BN;
        if (n0 + cl >= a.N) continue;
        float x = 0.f;
        for (int m = 0; m < WM; ++m) x += sR[(m * 2 + s) * BN + cl];
        add_sum(a.so.sums, (size_t)s * a.N + n0 + cl, x);
    }
}

// ------------------------------------------------------------------------------------------ weight gradient
// A warp owns a 48 x 4*TN block of the gradient (48 of the wider side) and its own pixels: eight at a time go global -> registers (one stage
// ahead) -> transform -> its part of shared memory, and 6 x TN products per lane and pixel are packed over the narrow side.  Warps, then the
// CTAs of a cluster, add their blocks in order; with one cluster per block that is the gradient, more leave a partial each.
constexpr int WTM = 6, WBM = 8 * WTM, WPX = 8, WWARPS = NT / 32;

struct F32WArgs {
    const float *dy, *z, *x;
    GradSrc dz;
    ValSrc xs;
    BnPendBwd pb;
    int pend_write;
    float* out;
    int P, CO, CI, mb, pix_per_cta, xf_d;
};

// One side: W channels from c0; `co`: coefficients in shared memory, [5 | 2][W]
template <int W, bool GRAD> struct Side32 {
    static constexpr int Q = W / 4, SL = (WPX * Q + 31) / 32;
    const float *p, *pz, *co;
    int c0, total, lane;
    bool xf;
    float lo, hi;
    float4 rv[SL], rz[SL];
    __device__ __forceinline__ void init(const F32WArgs& a, int c, const float* coef, int ln) {
        c0 = c; co = coef; lane = ln;
        total = GRAD ? a.CO : a.CI;
        p = GRAD ? a.dy : a.x;
        pz = a.z;
        const int act = GRAD ? a.dz.act : a.xs.act;
        lo = act == ACT_NONE ? -INFINITY : 0.f;
        hi = act == ACT_RELU6 ? 6.f : INFINITY;
        xf = GRAD ? a.xf_d != 0 : (a.xs.scale != nullptr || act != ACT_NONE);
    }
    __device__ __forceinline__ void fetch(int p0, int last) {
#pragma unroll
        for (int j = 0; j < SL; ++j) {
            const int i = lane + 32 * j, px = i / Q, c = c0 + (i - px * Q) * 4;
            if (px >= WPX) continue;
            const size_t e = (size_t)min(p0 + px, last) * total + min(c, total - 4);
            rv[j] = ld4(p + e);
            if (GRAD && xf) rz[j] = ld4(pz + e);
        }
    }
    __device__ __forceinline__ void stage(int p0, int pend, float* d) const {
#pragma unroll
        for (int j = 0; j < SL; ++j) {
            const int i = lane + 32 * j, px = i / Q, c = (i - px * Q) * 4;
            if (px >= WPX) continue;
            float4 v = rv[j];
            if (xf) {
                if (GRAD) {
                    const float4 k1 = ld4(co + c), k2 = ld4(co + W + c), k3 = ld4(co + 2 * W + c), s = ld4(co + 3 * W + c), h = ld4(co + 4 * W + c);
                    v.x = grad1(v.x, rz[j].x, k1.x, k2.x, k3.x, s.x, h.x, lo, hi);
                    v.y = grad1(v.y, rz[j].y, k1.y, k2.y, k3.y, s.y, h.y, lo, hi);
                    v.z = grad1(v.z, rz[j].z, k1.z, k2.z, k3.z, s.z, h.z, lo, hi);
                    v.w = grad1(v.w, rz[j].w, k1.w, k2.w, k3.w, s.w, h.w, lo, hi);
                } else {
                    const float4 s = ld4(co + c), h = ld4(co + W + c);
                    v.x = clampf(fmaf(v.x, s.x, h.x), lo, hi);
                    v.y = clampf(fmaf(v.y, s.y, h.y), lo, hi);
                    v.z = clampf(fmaf(v.z, s.z, h.z), lo, hi);
                    v.w = clampf(fmaf(v.w, s.w, h.w), lo, hi);
                }
            }
            if (p0 + px >= pend) v = make_float4(0.f, 0.f, 0.f, 0.f);
            *reinterpret_cast<float4*>(d + px * W + c) = v;
        }
    }
};

__device__ __forceinline__ float ld_cluster(uint32_t addr, uint32_t rank) {
    uint32_t a;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// MDZ: the gradient is the wide side (CO >= CI)
template <int TN, bool MDZ> __global__ void __launch_bounds__(NT) pw_f32_wgrad_kernel(const F32WArgs a) {
    constexpr int BN = 4 * TN, G = TN % 4 == 0 ? 4 : 2, SP = BN + 1, BLK = WBM * SP, NM = MDZ ? 5 : 2, NN = MDZ ? 2 : 5;
    constexpr int STG = WPX * (WBM + BN);
    __shared__ __align__(16) float coef[NM * WBM + NN * BN];
    __shared__ __align__(16) float st[WWARPS * (BLK > STG ? BLK : STG)];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, r = lane >> 2, t = lane & 3;
    const int m0 = ((int)blockIdx.y % a.mb) * WBM, n0 = ((int)blockIdx.y / a.mb) * BN;
    pdl_wait();
    const int pbeg = blockIdx.x * a.pix_per_cta, pend = min(a.P, pbeg + a.pix_per_cta);
    Side32<WBM, MDZ> sw;
    Side32<BN, !MDZ> sn;
    sw.init(a, m0, coef, lane);
    sn.init(a, n0, coef + NM * WBM, lane);
    int p0 = pbeg + warp * WPX;
    if (p0 < pend) {
        sw.fetch(p0, a.P - 1);
        sn.fetch(p0, a.P - 1);
    }
    {
        const int dw = MDZ ? WBM : BN, d0 = MDZ ? m0 : n0, xw = MDZ ? BN : WBM, x0 = MDZ ? n0 : m0;
        float *sk = MDZ ? coef : coef + NM * WBM, *sx = MDZ ? coef + NM * WBM : coef;
        const bool wr = a.pend_write && blockIdx.x == 0 && (MDZ ? n0 == 0 : m0 == 0);
        for (int c = tid; c < dw; c += NT) {
            const bool ok = d0 + c < a.CO;
            float3 k = make_float3(1.f, 0.f, 0.f);
            if (ok && a.pb.sums) k = bn_bwd_coef(a.pb, d0 + c, wr);
            else if (ok && a.dz.k1) k = make_float3(a.dz.k1[d0 + c], a.dz.k2[d0 + c], a.dz.k3[d0 + c]);
            sk[c] = k.x;
            sk[dw + c] = k.y;
            sk[2 * dw + c] = k.z;
            sk[3 * dw + c] = ok && a.dz.scale ? a.dz.scale[d0 + c] : 1.f;
            sk[4 * dw + c] = ok && a.dz.scale ? a.dz.shift[d0 + c] : 0.f;
        }
        for (int c = tid; c < xw; c += NT) {
            const bool ok = x0 + c < a.CI && a.xs.scale;
            sx[c] = ok ? a.xs.scale[x0 + c] : 1.f;
            sx[xw + c] = ok ? a.xs.shift[x0 + c] : 0.f;
        }
    }
    __syncthreads();
    float2 acc[WTM][TN / 2];
#pragma unroll
    for (int i = 0; i < WTM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = make_float2(0.f, 0.f);
    float *dw_ = st + warp * STG, *dn = dw_ + WPX * WBM;
    for (; p0 < pend; p0 += WWARPS * WPX) {
        sw.stage(p0, pend, dw_);
        sn.stage(p0, pend, dn);
        if (p0 + WWARPS * WPX < pend) {
            sw.fetch(p0 + WWARPS * WPX, a.P - 1);
            sn.fetch(p0 + WWARPS * WPX, a.P - 1);
        }
        __syncwarp();
#pragma unroll
        for (int px = 0; px < WPX; ++px) {
            float2 av[WTM / 2], bv[TN / 2];
#pragma unroll
            for (int i = 0; i < WTM / 2; ++i) av[i] = *reinterpret_cast<const float2*>(dw_ + px * WBM + 16 * i + 2 * r);
#pragma unroll
            for (int j = 0; j < TN / G; ++j) {
                if constexpr (G == 4) {
                    const float4 f = ld4(dn + px * BN + 16 * j + 4 * t);
                    bv[2 * j] = make_float2(f.x, f.y);
                    bv[2 * j + 1] = make_float2(f.z, f.w);
                } else {
                    bv[j] = *reinterpret_cast<const float2*>(dn + px * BN + 8 * j + 2 * t);
                }
            }
#pragma unroll
            for (int i = 0; i < WTM; ++i) {
                const float s = i & 1 ? av[i >> 1].y : av[i >> 1].x;
#pragma unroll
                for (int j = 0; j < TN / 2; ++j) acc[i][j] = __ffma2_rn(make_float2(s, s), bv[j], acc[i][j]);
            }
        }
        __syncwarp();
    }
    pdl_launch();
    __syncthreads();                                       // the blocks below reuse the stages of all warps
#pragma unroll
    for (int i = 0; i < WTM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) {
            const int m = 16 * (i >> 1) + 2 * r + (i & 1), n = G == 4 ? 16 * (j >> 1) + 4 * t + 2 * (j & 1) : 8 * j + 2 * t;
            st[warp * BLK + m * SP + n] = acc[i][j].x;
            st[warp * BLK + m * SP + n + 1] = acc[i][j].y;
        }
    __syncthreads();
    for (int e = tid; e < WBM * BN; e += NT) {
        float* d = st + (e / BN) * SP + e % BN;
        float s = d[0];
#pragma unroll
        for (int w = 1; w < WWARPS; ++w) s += d[w * BLK];
        d[0] = s;
    }
    uint32_t cs, rank;
    asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(cs));
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    if (cs > 1) cluster_sync();
    else __syncthreads();
    float* out = a.out + (size_t)(blockIdx.x / cs) * a.CO * a.CI;
    const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(st);
    const int per = (WBM * BN + (int)cs - 1) / (int)cs, e0 = (int)rank * per, e1 = min(WBM * BN, e0 + per);
    for (int e = e0 + tid; e < e1; e += NT) {
        const int m = MDZ ? e / BN : e % WBM, n = MDZ ? e % BN : e / WBM;      // consecutive threads write consecutive input channels
        float s = 0.f;
        if (cs == 1) s = st[m * SP + n];
        else {
            const uint32_t ad = s0 + (uint32_t)(m * SP + n) * 4u;
            float q[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) q[k] = k < (int)cs ? ld_cluster(ad, k) : 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) s += q[k];
        }
        const int k = MDZ ? m0 + m : n0 + n, c = MDZ ? n0 + n : m0 + m;
        if (k < a.CO && c < a.CI) out[(size_t)k * a.CI + c] = s;
    }
    if (cs > 1) cluster_sync();                            // no CTA leaves while another still reads its block
}

typedef void (*Fn)(const F32Args);
template <bool BWD, int TN, int XF> Fn by_wk(int wk) { return wk == 1 ? pw_f32_kernel<BWD, TN, 1, XF> : wk == 2 ? pw_f32_kernel<BWD, TN, 2, XF> : pw_f32_kernel<BWD, TN, 4, XF>; }
template <bool BWD, int XF> Fn by_tn(const F32Tiling& c) { return c.tn == 4 ? by_wk<BWD, 4, XF>(c.wk) : c.tn == 6 ? by_wk<BWD, 6, XF>(c.wk) : by_wk<BWD, 8, XF>(c.wk); }
Fn kernel_for(bool bwd, int xf, const F32Tiling& c) {
    if (bwd) return xf == XF_AFFINE ? by_tn<true, XF_AFFINE>(c) : xf ? by_tn<true, XF_VALUE>(c) : by_tn<true, XF_NONE>(c);
    return xf == XF_ADD ? by_tn<false, XF_ADD>(c) : xf ? by_tn<false, XF_VALUE>(c) : by_tn<false, XF_NONE>(c);
}

int w_pitch(int K) { return ((K + 15) & ~15) + 4; }        // 4 or 20 modulo 32 banks: the rows of four lanes in distinct banks

}  // namespace

size_t f32_smem(bool bwd, int K, const F32Tiling& c) {
    const int BN = 4 * c.tn, WM = 4 / c.wk, Kp = (K + 15) & ~15;
    const size_t part = (size_t)(c.wk - 1) * WM * 32 * 4 * c.tn, sums = (size_t)WM * 2 * BN;
    return 4 * ((size_t)BN * w_pitch(K) + (size_t)(bwd ? 5 : 3) * Kp + 4 * BN + (size_t)2 * 32 * WM * (16 * c.wk + 4) + (part > sums ? part : sums));
}

// Column tile: 16, 24 or 32, the one with the least padding; 16 where even the widest split of the reduction leaves less than one and a half CTAs per
// multiprocessor (192 -> 32 on 1 568 pixels 6.4 -> 5.5 us forward, 7.6 -> 6.5 backward; 16 -> 96 on 1 000 pixels 3.9 -> 3.0 and 5.2 -> 4.0), in the
// backward only up to 256 channels, since every column tile transforms the gradient anew (384 -> 64 on 1 568 pixels 11.7 -> 12.4 with 16).  The
// backward with several tiles of 24 columns takes 16 and three CTAs per multiprocessor (24 -> 144 on 25 088 pixels 20.4 -> 16.8, on 100 352 82.8 ->
// 63.1), the forward with 24 columns three (13.9 -> 12.3, 40.8 -> 37.6).  The reduction is split over two or four warps (32- and 64-deep chunks)
// where tiles of 128 pixels would leave multiprocessors without one and a half CTAs - three quarters of one in the backward with wide tiles, where
// unsplit tiles read the gradient in longer rows (144 -> 24 on 25 088 pixels 21.5 -> 16.6) - and every warp still gets a 16-deep share.
bool f32_choose(bool bwd, int P, int K, int N, F32Tiling* out) {
    if (K % 4 || N % 4) return false;
    const int sms = sm_count();
    F32Tiling c{};
    int best = 0;
    for (int tn : {8, 6, 4}) {
        const int cols = (N + 4 * tn - 1) / (4 * tn), cost = cols * 4 * tn * 8 + cols * 16;
        if (!c.tn || cost < best) {
            c.tn = tn;
            best = cost;
        }
    }
    const int most = K >= 64 ? 4 : K >= 32 ? 2 : 1;
    if ((!bwd || K <= 256) && (P + 128 / most - 1) / (128 / most) * ((N + 4 * c.tn - 1) / (4 * c.tn)) < sms * 3 / 2) c.tn = 4;
    const bool thin = bwd && c.tn == 6 && N > 24;
    if (thin) c.tn = 4;
    const int cols = (N + 4 * c.tn - 1) / (4 * c.tn);
    c.wk = 1;
    while (c.wk < 4 && K >= 32 * c.wk && (P + 128 / c.wk - 1) / (128 / c.wk) * cols < (bwd && c.tn > 4 ? sms * 3 / 4 : sms * 3 / 2)) c.wk *= 2;
    c.ctas = thin || (!bwd && c.tn == 6 && c.wk == 1) ? 3 : 4;
    while (f32_smem(bwd, K, c) > 200 * 1024) {
        if (c.tn == 4) return false;
        c.tn -= 2;
    }
    *out = c;
    return true;
}

void f32_launch(bool bwd, const MmaProblem& p, const F32Tiling& c, int kind, double bytes, cudaStream_t st) {
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(done.load(std::memory_order_acquire) & bit)) {
        for (int tn : {4, 6, 8})
            for (int wk : {1, 2, 4})
                for (int v = 0; v < 6; ++v)
                    cudaFuncSetAttribute(kernel_for(v < 3, v % 3, F32Tiling{tn, wk, 0}), cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        done.fetch_or(bit, std::memory_order_release);
    }
    F32Args a;
    memset(&a, 0, sizeof a);
    a.P = p.P; a.K = p.K; a.N = p.N;
    int xf;
    const int act = bwd ? p.dz.act : p.sum_out ? p.sum_act : p.x.act;
    if (bwd) {
        a.a = (const float*)p.dz.dy; a.az = (const float*)p.dz.z;
        a.c0 = p.dz.k1; a.c1 = p.dz.k2; a.c2 = p.dz.k3; a.c3 = p.dz.scale; a.c4 = p.dz.shift;
        a.pb = p.pb;
        xf = act != ACT_NONE ? XF_VALUE : p.dz.k1 || p.pb.sums ? XF_AFFINE : XF_NONE;
    } else {
        a.a = (const float*)p.x.p;
        a.c0 = p.x.scale; a.c1 = p.x.shift;
        a.pf = p.pf;
        xf = act != ACT_NONE || p.x.scale || p.pf.sums ? XF_VALUE : XF_NONE;
        if (p.sum_out) {
            xf = XF_ADD;
            a.az = (const float*)p.x2.p; a.d0 = p.x2.scale; a.d1 = p.x2.shift;
            a.pf2 = p.pf2;
            a.sum_out = (float*)p.sum_out;
        }
    }
    a.lo = act == ACT_NONE ? -INFINITY : 0.f;
    a.hi = act == ACT_RELU6 ? 6.f : INFINITY;
    a.w = (const float*)p.w; a.bias = p.bias; a.addend = (const float*)p.addend; a.out = (float*)p.out;
    a.bp = w_pitch(p.K);
    a.so = p.so;
    if (p.red) {
        a.rz = (const float*)p.red->z;
        a.r_scale = p.red->scale; a.r_shift = p.red->shift; a.r_mean = p.red->mean; a.r_rstd = p.red->rstd;
        a.r_mask = p.red->mask;
        a.r_lo = p.red->act == ACT_NONE ? -INFINITY : 0.f;
        a.r_hi = p.red->act == ACT_RELU6 ? 6.f : INFINITY;
    }
    const int BM = 128 / c.wk, ny = (p.N + 4 * c.tn - 1) / (4 * c.tn);
    a.m_tiles = (p.P + BM - 1) / BM;
    int gx = sm_count() * c.ctas / ny;
    if (gx < 1) gx = 1;
    if (gx > a.m_tiles) gx = a.m_tiles;
    LaunchScope ls(kind, bytes + (bwd && p.so.sums ? 4.0 * p.P * p.N : 0.0) + (p.sum_out ? 8.0 * p.P * p.K : 0.0), 2.0 * p.P * p.N * p.K, st);
    launch_pdl(kernel_for(bwd, xf, c), dim3(gx, ny), NT, f32_smem(bwd, p.K, c), st, a);
}

// Three CTAs per multiprocessor, four with 24 columns (24 x 144 on 100 352 pixels 41.8 -> 34.3 us), no pixel range below 64.  Up to 11 ranges one cluster adds its blocks and writes the result (160 x 960 on 784
// pixels: 20.0 us, against 23.0 with a split sum).  From 12 ranges up the split sum runs in any case, and single CTAs that start and end on their own beat
// clusters of eight: 24 x 144 on 25 088 pixels 22.3 -> 14.3 us, 32 x 192 on 6 272 19.1 -> 9.3, 16 x 96 on 8 192 9.9 -> 6.4.
bool f32_wgrad_choose(int P, int CO, int CI, size_t scratch_floats, F32WgradTiling* out) {
    if (CO % 4 || CI % 4) return false;
    const int CM = CO > CI ? CO : CI, CN = CO > CI ? CI : CO;
    F32WgradTiling c{8, 1, 1};
    int best = 0;
    for (int tn : {8, 6, 4}) {
        const int cols = (CN + 4 * tn - 1) / (4 * tn), cost = cols * (4 * tn + 12);
        if (!best || cost < best) {
            c.tn = tn;
            best = cost;
        }
    }
    const int blocks = ((CM + WBM - 1) / WBM) * ((CN + 4 * c.tn - 1) / (4 * c.tn));
    int sp = sm_count() * (c.tn == 6 ? 4 : 3) / blocks;
    const int most = P / 64 > 0 ? P / 64 : 1;
    if (sp > most) sp = most;
    c.cluster = sp >= 12 ? 1 : sp >= 6 ? 8 : sp >= 3 ? 4 : sp >= 2 ? 2 : 1;
    c.splits = sp >= 12 ? sp : c.cluster;
    while ((size_t)(c.splits / c.cluster) * CO * CI > scratch_floats && c.splits > c.cluster) c.splits -= c.cluster;
    *out = c;
    return true;
}

void f32_wgrad_launch(const WgradProblem& p, const F32WgradTiling& c, float* scratch, float* gw, cudaStream_t st) {
    F32WArgs a;
    memset(&a, 0, sizeof a);
    a.dy = (const float*)p.dz.dy; a.z = (const float*)p.dz.z; a.x = (const float*)p.x.p;
    a.dz = p.dz; a.xs = p.x; a.pb = p.pb; a.pend_write = p.pend_write;
    a.xf_d = p.dz.act != ACT_NONE || p.dz.k1 || p.pb.sums;
    a.P = p.P; a.CO = p.CO; a.CI = p.CI;
    const bool mdz = p.CO >= p.CI;
    const int CM = mdz ? p.CO : p.CI, CN = mdz ? p.CI : p.CO, BN = 4 * c.tn, parts = c.splits / c.cluster;
    a.mb = (CM + WBM - 1) / WBM;
    a.pix_per_cta = ((p.P + c.splits - 1) / c.splits + WPX - 1) / WPX * WPX;
    const size_t out_elems = (size_t)p.CO * p.CI;
    a.out = parts > 1 ? scratch : gw;
    {
        LaunchScope ls(K_CONV_BWD_WEIGHT, 4.0 * p.P * p.CO * (a.xf_d ? 2.0 : 1.0) + 4.0 * (double)p.P * p.CI + 4.0 * out_elems, 2.0 * p.P * (double)out_elems, st);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c.splits, a.mb * ((CN + BN - 1) / BN));
        cfg.blockDim = dim3(NT);
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = c.cluster;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = c.cluster > 1 ? 2 : 1;
        typedef void (*WFn)(const F32WArgs);
        WFn f;
        if (mdz) f = c.tn == 4 ? (WFn)pw_f32_wgrad_kernel<4, true> : c.tn == 6 ? (WFn)pw_f32_wgrad_kernel<6, true> : (WFn)pw_f32_wgrad_kernel<8, true>;
        else f = c.tn == 4 ? (WFn)pw_f32_wgrad_kernel<4, false> : c.tn == 6 ? (WFn)pw_f32_wgrad_kernel<6, false> : (WFn)pw_f32_wgrad_kernel<8, false>;
        cudaLaunchKernelEx(&cfg, f, a);
    }
    if (parts > 1) {
        LaunchScope ls(K_REDUCE_SPLITS, 4.0 * out_elems * (parts + 1), (double)out_elems * parts, st);
        reduce_splits_f4(scratch, parts, out_elems, gw, st);
    }
}

}  // namespace ast
