// Pointwise (1x1) convolution with register-resident operands: forward and backward-data of the thin layers.
//
//   out[p][n] = sum_k A[p][k] * W[n][k]
//   forward    A = act(x*scale + shift) of the producing unit's raw output, W = weights [c_out][c_in]
//   backward   A = BatchNorm/activation backward of (dy, z), W = transposed weights [c_in][c_out]
//
// These layers move 2 (K + N) bytes and do 2 K N operations per pixel: at the channel counts of the compact networks they are
// bound by memory, and on small maps by latency.  What the tensor-memory pipeline of pw_tc.cu pays for them is not the
// arithmetic but the way of the operand: bulk copy -> shared memory -> transform -> shared memory -> MMA -> tensor memory ->
// shared memory -> bulk copy, with an mbarrier hand-off at every arrow.  Here a thread loads 16 bytes (8 channels) of a pixel
// row straight into registers, transforms them there and feeds them to mma.sync.m16n8k16 as they are: the reduction index may be
// permuted freely as long as both operands agree, so channels 8t..8t+7 of a 32-channel chunk are simply DECLARED to be the k
// slots that lane quad position t holds in two consecutive k-steps.  The same trick on the columns makes the 2G
// accumulator columns a thread ends up with consecutive channels (G column tiles interleaved), so results leave as one vector
// store.  Shared memory holds only the weights (read by every warp as 16-byte fragments) and per-channel coefficients.
// mma.sync reaches 553 TFLOP/s here (tcgen05: 1 600), which is beyond what any of these layers asks for.
//
// The column sums the BatchNorms need are taken from the registers the output is stored from; the coefficients of a
// BatchNorm in front are formed in the prologue (fin.cuh).
#pragma once
#include <type_traits>

#include "fin.cuh"

namespace ast {
namespace mma {

struct Args {
    const void* a;             // [P][K]: x, or dy
    const void* az;            // backward: z [P][K]; forward of a deferred sum: its second operand
    const float *c0, *c1, *c2, *c3, *c4;   // operand transform: forward scale, shift; backward k1, k2, k3, scale, shift (null: identity)
    int act;
    const __nv_bfloat16* w;    // [N][K]
    const float* bias;         // forward, may be null
    const void* addend;        // backward, may be null: [P][N]
    __nv_bfloat16* out;        // [P][N]
    int P, K, N;
    int KCH;                   // 32-channel chunks of the reduction
    int WM;                    // warps, each with pixels of its own
    int m_tiles;
    uint32_t wpitch;           // bytes between rows of the staged weights
    BnPendFwd pf;              // pending coefficients of the operand (sums null: c0.. are final)
    BnPendFwd pf2;             // deferred sum: pending coefficients of the second operand
    const float *d0, *d1;      // ... its scale and shift (null: identity)
    __nv_bfloat16* sum_out;    // ... where the sum goes, [P][K]
    BnPendBwd pb;
    BnSumsOut so;              // column sums of the output (sums null: none)
    const __nv_bfloat16* rz;   // backward sums: raw output [P][N] of the unit whose gradient this is, its coefficients and activation
    const float *r_scale, *r_shift, *r_mean, *r_rstd;
    int r_act;
    bool r_mask;               // the output is stored as that unit's activation lets it through
    bool late;                 // persistent form: dependents are released when the products are done (common.cuh)
};

__device__ __forceinline__ void mma16816(float* c, const uint32_t a0, const uint32_t a1, const uint32_t a2, const uint32_t a3, const uint32_t b0, const uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool ok) {
    const int n = ok ? 16 : 0;            // 0: the sixteen bytes are filled with zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void lds8(const float* p, float* o) {
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w; o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
}
__device__ __forceinline__ float2 unpack2(uint32_t w) { return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); }
__device__ __forceinline__ uint32_t pack2(float2 f) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(f.x, f.y);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// Operand transforms of 8 channels.  Forward: the activation is applied after rounding on packed pairs, as one integer
// min-then-max-with-0 (the bit patterns of non-negative bfloat16 numbers order like integers and negative ones are negative
// integers; rounding is monotonic and 0 and 6 are bfloat16 numbers, so clamping before or after it is the same).
// XF_ADD, XF_SUM (forward): the operand is a residual sum that has not been formed yet, act(x*s + z*s2 + h) of two tensors with their shifts added first, or
// act((x*s + h) + (z*s2 + h2)), the roundings of the elementwise pass (bn_ew.cu).  Only a ReLU may follow a sum.  Either applies it as a maximum of packed pairs, by which what is not a number
// leaves as it does there by fmaxf, as the activation's lower end.
enum { XF_NONE = 0, XF_AFFINE = 1, XF_ACT = 2, XF_ADD = 3, XF_SUM = 4 };
__host__ __device__ constexpr bool xf_sum(int xf) { return xf == XF_ADD || xf == XF_SUM; }
template <int XF> struct XfFwd {
    float s[8], h[8], s2[8], h2[8];
    __nv_bfloat162 lo;         // of a sum
    uint32_t top;              // of a value
    __device__ __forceinline__ void load(const float* sm, int Kp, int c) {
        if (XF == XF_NONE) return;
        lds8(sm + c, s);
        lds8(sm + Kp + c, h);
        if (xf_sum(XF)) lds8(sm + 2 * Kp + c, s2);
        if (XF == XF_SUM) lds8(sm + 3 * Kp + c, h2);
    }
    __device__ __forceinline__ uint32_t sum(uint32_t w, uint32_t z, int q) const {
        const float2 x = unpack2(w), y = unpack2(z), sx = make_float2(s[q], s[q + 1]), hx = make_float2(h[q], h[q + 1]), sy = make_float2(s2[q], s2[q + 1]);
        const float2 r = XF == XF_SUM ? __fadd2_rn(__ffma2_rn(x, sx, hx), __ffma2_rn(y, sy, make_float2(h2[q], h2[q + 1]))) : __ffma2_rn(x, sx, __ffma2_rn(y, sy, hx));
        const __nv_bfloat162 o = __hmax2(__floats2bfloat162_rn(r.x, r.y), lo);
        return *reinterpret_cast<const uint32_t*>(&o);
    }
    __device__ __forceinline__ uint32_t two(uint32_t w, int q) const {
        const uint32_t r = pack2(__ffma2_rn(unpack2(w), make_float2(s[q], s[q + 1]), make_float2(h[q], h[q + 1])));
        return XF == XF_ACT ? __vimin_s16x2_relu(r, top) : r;
    }
    __device__ __forceinline__ uint4 apply(const uint4& v, const uint4& z) const {
        if (XF == XF_NONE) return v;
        if (xf_sum(XF)) return make_uint4(sum(v.x, z.x, 0), sum(v.y, z.y, 2), sum(v.z, z.z, 4), sum(v.w, z.w, 6));
        return make_uint4(two(v.x, 0), two(v.y, 2), two(v.z, 4), two(v.w, 6));
    }
};
// Backward: dz = k1*dy*[0 < pre < hi] + k2 + k3*z; the mask guards one fused multiply-add.
template <int XF> struct XfBwd {
    float k1[8], k2[8], k3[8], s[8], h[8], hi;
    __device__ __forceinline__ void load(const float* sm, int Kp, int c) {
        if (XF == XF_NONE) return;
        lds8(sm + c, k1);
        lds8(sm + Kp + c, k2);
        lds8(sm + 2 * Kp + c, k3);
        if (XF == XF_ACT) {
            lds8(sm + 3 * Kp + c, s);
            lds8(sm + 4 * Kp + c, h);
        }
    }
    __device__ __forceinline__ uint32_t two(uint32_t wd, uint32_t wz, int q) const {
        const float2 d = unpack2(wd), z = unpack2(wz);
        float2 o = __ffma2_rn(make_float2(k3[q], k3[q + 1]), z, make_float2(k2[q], k2[q + 1]));
        if (XF == XF_ACT) {
            const float2 pre = __ffma2_rn(z, make_float2(s[q], s[q + 1]), make_float2(h[q], h[q + 1]));
            if (pre.x > 0.f && pre.x < hi) o.x = fmaf(k1[q], d.x, o.x);
            if (pre.y > 0.f && pre.y < hi) o.y = fmaf(k1[q + 1], d.y, o.y);
        } else {
            o = __ffma2_rn(make_float2(k1[q], k1[q + 1]), d, o);
        }
        return pack2(o);
    }
    __device__ __forceinline__ uint4 apply(const uint4& d, const uint4& z) const {
        if (XF == XF_NONE) return d;
        return make_uint4(two(d.x, z.x, 0), two(d.y, z.y, 2), two(d.z, z.z, 4), two(d.w, z.w, 6));
    }
};
template <bool BWD, int XF> struct Xf;
template <int XF> struct Xf<false, XF> : XfFwd<XF> {
    __device__ __forceinline__ void set_act(int act) {
        this->top = act == ACT_RELU6 ? 0x40C040C0u : 0x7F807F80u;
        this->lo = __float2bfloat162_rn(act == ACT_NONE ? -INFINITY : 0.f);
    }
};
template <int XF> struct Xf<true, XF> : XfBwd<XF> {
    __device__ __forceinline__ void set_act(int act) { this->hi = act == ACT_RELU6 ? 6.f : INFINITY; }
};

// Weights of this CTA's BN columns -> shared memory.  Row jt*8 + g holds the channel that column g of column tile jt stands for
// (G tiles interleaved: a thread's columns 2t, 2t+1 of G tiles are 2G consecutive channels); channels beyond N and k beyond K are zeros.
template <int G> __device__ __forceinline__ void stage_weights(const Args& a, uint8_t* sW, int n0, int BN) {
    const int vpr = a.KCH * 4, kv = a.K >> 3;
    const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(sW);
    for (int i = threadIdx.x; i < BN * vpr; i += blockDim.x) {
        const int sr = i / vpr, v = i - sr * vpr, jt = sr >> 3, g = sr & 7;
        const int n = n0 + (jt / G) * 8 * G + 2 * G * (g >> 1) + 2 * (jt % G) + (g & 1);
        const bool ok = n < a.N && v < kv;
        cp_async16(s0 + (uint32_t)sr * a.wpitch + (uint32_t)v * 16u, a.w + (ok ? (size_t)n * a.K + v * 8 : 0), ok);
    }
    cp_commit();
}

// Coefficients of the operand transform and of the column sums -> shared memory (after the dependency wait).  Everything a thread reads from memory is
// requested before it uses anything: sums, pivots, the other operand's and the columns' coefficients were up to four trips one after the other, of
// 0.6 us each.
template <bool BWD, int XF> __device__ __forceinline__ void stage_coefs(const Args& a, float* sK, float* sN, int n0, int BN) {
    const int Kp = a.KCH * 32, nt = blockDim.x;
    const bool first = blockIdx.x == 0 && blockIdx.y == 0;
    const int cn = threadIdx.x;                            // BN <= 64: a column a thread
    const bool col = a.so.sums && cn < BN && n0 + cn < a.N;
    float nr = 0.f, ns = 0.f, nh = 0.f, nm = 0.f;
    if (col) {
        if (BWD) {
            nr = a.r_rstd[n0 + cn];
            ns = a.r_scale[n0 + cn];
            nh = a.r_shift[n0 + cn];
            nm = a.r_mean[n0 + cn];
        } else nm = a.so.pivot[n0 + cn];
    }
    if (XF != XF_NONE) {
        struct In {
            typename std::conditional<BWD, BnBwdIn, BnFwdIn>::type in;
            BnFwdIn in2;
            float k1, k2, k3, s, h;
        } in, next;                                        // those of the thread's next channel are under way
        const auto request = [&](int ch, In& to) {
            if (ch >= a.K) return;
            if constexpr (BWD) {
                if (a.pb.sums) to.in.load(a.pb, ch);
                else if (a.c0) {
                    to.k1 = a.c0[ch];
                    to.k2 = a.c1[ch];
                    to.k3 = a.c2[ch];
                }
                if (XF == XF_ACT && a.c3) {
                    to.s = a.c3[ch];
                    to.h = a.c4[ch];
                }
            } else {
                if (a.pf.sums) to.in.load(a.pf, ch, first);
                else if (a.c0) {
                    to.k1 = a.c0[ch];
                    to.k2 = a.c1[ch];
                }
                if (xf_sum(XF)) {
                    if (a.pf2.sums) to.in2.load(a.pf2, ch, first);
                    else if (a.d0) {
                        to.s = a.d0[ch];
                        to.h = a.d1[ch];
                    }
                }
            }
        };
        int c = threadIdx.x;
        request(c, in);
#pragma unroll 1
        for (; c < Kp; c += nt) {
            const bool ok = c < a.K;
            request(c + nt, next);
            if constexpr (BWD) {
                float3 k = make_float3(1.f, 0.f, 0.f);
                if (ok && a.pb.sums) k = in.in.coef(a.pb, c, first);
                else if (ok && a.c0) k = make_float3(in.k1, in.k2, in.k3);
                sK[c] = k.x;
                sK[Kp + c] = k.y;
                sK[2 * Kp + c] = k.z;
                if (XF == XF_ACT) {
                    sK[3 * Kp + c] = ok && a.c3 ? in.s : 1.f;
                    sK[4 * Kp + c] = ok && a.c3 ? in.h : 0.f;
                }
            } else {
                float2 k = make_float2(1.f, 0.f);
                if (ok && a.pf.sums) k = in.in.coef(a.pf, c, first);
                else if (ok && a.c0) k = make_float2(in.k1, in.k2);
                sK[c] = k.x;
                if (xf_sum(XF)) {
                    float2 k2 = make_float2(1.f, 0.f);
                    if (ok && a.pf2.sums) k2 = in.in2.coef(a.pf2, c, first);
                    else if (ok && a.d0) k2 = make_float2(in.s, in.h);
                    sK[2 * Kp + c] = k2.x;
                    if (XF == XF_SUM) sK[3 * Kp + c] = k2.y;
                    else k.y += k2.y;
                }
                sK[Kp + c] = k.y;
            }
            in = next;
        }
    }
    if (a.so.sums && cn < BN) {
        if (BWD) {
            sN[cn] = ns;
            sN[BN + cn] = nh;
            sN[2 * BN + cn] = nr;
            sN[3 * BN + cn] = -nm * nr;
        } else {
            sN[cn] = nm;
            if (col && blockIdx.x == 0) a.so.pivot_copy[n0 + cn] = nm;
        }
    }
}

// C consecutive channels of one pixel
template <int C> struct CVec {
    uint32_t w[C / 2];
    __device__ __forceinline__ void load(const void* p, uint32_t byte) {
        const uint8_t* q = reinterpret_cast<const uint8_t*>(p) + (size_t)byte;
        if constexpr (C == 8) *reinterpret_cast<uint4*>(w) = *reinterpret_cast<const uint4*>(q);
        else if constexpr (C == 4) *reinterpret_cast<uint2*>(w) = *reinterpret_cast<const uint2*>(q);
        else w[0] = *reinterpret_cast<const uint32_t*>(q);
    }
    __device__ __forceinline__ void store(void* p, uint32_t byte) const {
        uint8_t* q = reinterpret_cast<uint8_t*>(p) + (size_t)byte;
        if constexpr (C == 8) *reinterpret_cast<uint4*>(q) = *reinterpret_cast<const uint4*>(w);
        else if constexpr (C == 4) *reinterpret_cast<uint2*>(q) = *reinterpret_cast<const uint2*>(w);
        else *reinterpret_cast<uint32_t*>(q) = w[0];
    }
};
// the pair's contribution to the two sums of its channels; returns the pair as it is to be stored
template <bool BWD> struct SumCoef;
template <> struct SumCoef<false> {
    float2 pv;
    __device__ __forceinline__ void load(const float* sN, int, int c) { pv = make_float2(-sN[c], -sN[c + 1]); }
    __device__ __forceinline__ uint32_t add(uint32_t d, uint32_t, float, float, bool, float2& s1, float2& s2) const {
        const float2 q = __fadd2_rn(unpack2(d), pv);
        s1 = __fadd2_rn(s1, q);
        s2 = __ffma2_rn(q, q, s2);
        return d;
    }
};
template <> struct SumCoef<true> {
    float2 sc, sh, rs, rm;
    __device__ __forceinline__ void load(const float* sN, int BN, int c) {
        sc = *reinterpret_cast<const float2*>(sN + c);
        sh = *reinterpret_cast<const float2*>(sN + BN + c);
        rs = *reinterpret_cast<const float2*>(sN + 2 * BN + c);
        rm = *reinterpret_cast<const float2*>(sN + 3 * BN + c);
    }
    __device__ __forceinline__ uint32_t add(uint32_t d, uint32_t z, float lo, float hi, bool mask, float2& s1, float2& s2) const {
        const float2 zz = unpack2(z), pre = __ffma2_rn(zz, sc, sh), xh = __ffma2_rn(zz, rs, rm);
        float2 q = unpack2(d);
        if (!(pre.x > lo && pre.x < hi)) q.x = 0.f;
        if (!(pre.y > lo && pre.y < hi)) q.y = 0.f;
        s1 = __fadd2_rn(s1, q);
        s2 = __ffma2_rn(q, xh, s2);
        return mask ? __byte_perm(__float_as_uint(q.x), __float_as_uint(q.y), 0x7632) : d;
    }
};

// ---------------------------------------------------------------------------------------------------------------------
// Large maps: CTAs walk down the pixel tiles, every warp has 16*MI pixels x 8*NJ columns and the whole reduction.
//
// A chunk of 32 channels is a step, whose operands are requested one step ahead, in registers.  DEEP (two operands): two or three steps ahead, by asynchronous copies into shared-memory slots that
// no other thread reads, so that no barrier is needed.
template <int MI> struct Slots {
    static constexpr int VECS = MI * 4, STEPS = VECS >= 8 ? 3 : 4;      // 16-byte vectors a thread and step, steps there is room for
    static constexpr int BYTES = VECS * STEPS * 16;                     // of a thread
};
template <bool BWD, int MI, int NJ, int G, int XF, bool DEEP>
__global__ void __launch_bounds__(256) pw_mma_kernel(const Args a) {
    using S = Slots<MI>;
    constexpr bool USE_Z = BWD ? XF != XF_NONE : xf_sum(XF);
    static_assert(USE_Z || !DEEP, "slots are laid out for two operands");
    constexpr int D = S::STEPS;
    extern __shared__ __align__(16) uint8_t sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int wm = warp;
    const int BN = NJ * 8, n0 = blockIdx.y * BN, Kp = a.KCH * 32;
    uint8_t* sW = sm;
    float* sK = reinterpret_cast<float*>(sW + (size_t)BN * a.wpitch);
    float* sN = sK + (BWD && XF == XF_ACT ? 5 : XF == XF_SUM ? 4 : 3) * Kp;
    float* red = sN + (BWD ? 4 : 1) * BN;                  // [WM][2][BN]
    stage_weights<G>(a, sW, n0, BN);
    pdl_wait();
    if (!a.late) pdl_launch();

    const uint8_t* pa = reinterpret_cast<const uint8_t*>(a.a);
    const uint8_t* pz = reinterpret_cast<const uint8_t*>(a.az);
    const int warp_row = wm * (16 * MI) + g, BM = a.WM * 16 * MI;
    const uint32_t row_bytes = (uint32_t)a.K * 2u;
    const uint32_t last_off = (uint32_t)min((a.KCH - 1) * 64 + t * 16, a.K * 2 - 16);     // beyond K: any finite value, its weights are zero
    uint32_t roff[MI][2];
    auto set_rows = [&](int tile) {
#pragma unroll
        for (int mi = 0; mi < MI; ++mi)
#pragma unroll
            for (int h = 0; h < 2; ++h) roff[mi][h] = (uint32_t)min(tile * BM + warp_row + mi * 16 + h * 8, a.P - 1) * row_bytes;
    };
    uint4 nx[MI][2], nz[MI][2];
    const uint32_t pitch = blockDim.x * 16u;               // DEEP: from one vector of a thread to its next, [slot][vector][thread]
    const uint8_t* slots = reinterpret_cast<const uint8_t*>(red + a.WM * 2 * BN) + tid * 16;
    const uint32_t slots_s = (uint32_t)__cvta_generic_to_shared(slots);
    int ftile = blockIdx.x, fkc = 0, fslot = 0, slot = 0;  // DEEP: the step requested next, its slot; the slot of the step at hand
    auto fetch = [&](int kc) {
        const uint32_t o = kc == a.KCH - 1 ? last_off : (uint32_t)(kc * 64 + t * 16);
        uint32_t d = slots_s + (uint32_t)(fslot * S::VECS) * pitch;
#pragma unroll
        for (int mi = 0; mi < MI; ++mi)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if constexpr (DEEP) {
                    cp_async16(d, pa + (size_t)(roff[mi][h] + o), true);
                    cp_async16(d + pitch, pz + (size_t)(roff[mi][h] + o), true);
                    d += 2 * pitch;
                } else {
                    nx[mi][h] = *reinterpret_cast<const uint4*>(pa + (size_t)(roff[mi][h] + o));
                    if (USE_Z) nz[mi][h] = *reinterpret_cast<const uint4*>(pz + (size_t)(roff[mi][h] + o));
                }
            }
    };
    auto fetch_next = [&] {                                // DEEP
        if (ftile < a.m_tiles) {
            fetch(fkc);
            if (++fkc == a.KCH) {
                fkc = 0;
                ftile += gridDim.x;
                set_rows(ftile);
            }
        }
        cp_commit();
        if (++fslot == D) fslot = 0;
    };
    int tile = blockIdx.x;
    set_rows(tile);
    if constexpr (DEEP) {
#pragma unroll
        for (int i = 0; i < D - 1; ++i) fetch_next();
    } else {
        fetch(0);
    }
    stage_coefs<BWD, XF>(a, sK, sN, n0, BN);
    cp_wait<DEEP ? D - 1 : 0>();
    __syncthreads();

    const float rlo = a.r_act == ACT_NONE ? -INFINITY : 0.f, rhi = a.r_act == ACT_RELU6 ? 6.f : INFINITY;
    const uint8_t* wb = sW + (uint32_t)g * a.wpitch + t * 16;
    const bool sums = (bool)a.so.sums;
    float2 s1[NJ], s2[NJ];
#pragma unroll
    for (int i = 0; i < NJ; ++i) s1[i] = s2[i] = make_float2(0.f, 0.f);
    Xf<BWD, XF> xf;
    xf.set_act(a.act);
    xf.load(sK, Kp, t * 8);
    // 2G consecutive channels of rows g and g+8 per column group: the raw outputs the backward sums need are requested one tile ahead
    constexpr int C = 2 * G, NG = NJ / G;
    CVec<C> zv[NG][MI][2];
    auto fetch_z = [&](int tl) {
#pragma unroll
        for (int gr = 0; gr < NG; ++gr) {
            const uint32_t n = (uint32_t)min(n0 + gr * 8 * G + C * t, a.N - C);
#pragma unroll
            for (int mi = 0; mi < MI; ++mi)
#pragma unroll
                for (int h = 0; h < 2; ++h) zv[gr][mi][h].load(a.rz, ((uint32_t)min(tl * BM + warp_row + mi * 16 + h * 8, a.P - 1) * (uint32_t)a.N + n) * 2u);
        }
    };
    if (BWD && sums) fetch_z(tile);
    // the addend one column group ahead (the first one before the products), where registers allow
    constexpr bool AHEAD = MI * NJ < 16;
    CVec<C> av[2][MI][2];
    auto fetch_add = [&](int gr, int row0, CVec<C> (*v)[2]) {
        const uint32_t n = (uint32_t)min(n0 + gr * 8 * G + C * t, a.N - C);
#pragma unroll
        for (int mi = 0; mi < MI; ++mi)
#pragma unroll
            for (int h = 0; h < 2; ++h) v[mi][h].load(a.addend, ((uint32_t)min(row0 + mi * 16 + h * 8, a.P - 1) * (uint32_t)a.N + n) * 2u);
    };
    for (; tile < a.m_tiles; tile += gridDim.x) {
        const int row0 = tile * BM + warp_row;
        if (BWD && AHEAD && a.addend) fetch_add(0, row0, av[0]);
        float acc[MI][NJ][4];
#pragma unroll
        for (int mi = 0; mi < MI; ++mi)
#pragma unroll
            for (int j = 0; j < NJ; ++j)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[mi][j][q] = 0.f;
#pragma unroll 1
        for (int kc = 0; kc < a.KCH; ++kc) {
            uint4 cu[MI][2];
            if (a.KCH > 1) xf.load(sK, Kp, kc * 32 + t * 8);
            if constexpr (DEEP) {
                cp_wait<D - 2>();
                const uint8_t* q = slots + (uint32_t)(slot * S::VECS) * pitch;
#pragma unroll
                for (int mi = 0; mi < MI; ++mi)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        nx[mi][h] = *reinterpret_cast<const uint4*>(q);
                        nz[mi][h] = *reinterpret_cast<const uint4*>(q + pitch);
                        q += 2 * pitch;
                    }
                if (++slot == D) slot = 0;
            }
#pragma unroll
            for (int mi = 0; mi < MI; ++mi)
#pragma unroll
                for (int h = 0; h < 2; ++h) cu[mi][h] = xf.apply(nx[mi][h], nz[mi][h]);
            if constexpr (DEEP) fetch_next();
            if (!BWD && xf_sum(XF) && blockIdx.y == 0 && kc * 64 + t * 16 < a.K * 2)
#pragma unroll
                for (int mi = 0; mi < MI; ++mi)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int p = row0 + mi * 16 + h * 8;
                        if (p < a.P) *reinterpret_cast<uint4*>(reinterpret_cast<uint8_t*>(a.sum_out) + (size_t)p * row_bytes + (uint32_t)(kc * 64 + t * 16)) = cu[mi][h];
                    }
            if constexpr (!DEEP) {
                if (kc + 1 < a.KCH) fetch(kc + 1);
                else if (tile + (int)gridDim.x < a.m_tiles) {
                    set_rows(tile + gridDim.x);
                    fetch(0);
                }
            }
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const uint4 b = *reinterpret_cast<const uint4*>(wb + (uint32_t)(j * 8) * a.wpitch + (uint32_t)kc * 64u);
#pragma unroll
                for (int mi = 0; mi < MI; ++mi) {
                    mma16816(acc[mi][j], cu[mi][0].x, cu[mi][1].x, cu[mi][0].y, cu[mi][1].y, b.x, b.y);
                    mma16816(acc[mi][j], cu[mi][0].z, cu[mi][1].z, cu[mi][0].w, cu[mi][1].w, b.z, b.w);
                }
            }
        }
#pragma unroll
        for (int gr = 0; gr < NG; ++gr) {
            const int cl = gr * 8 * G + C * t, n = n0 + cl;
            if (BWD && AHEAD && a.addend && gr + 1 < NG) fetch_add(gr + 1, row0, av[(gr + 1) & 1]);
            if (BWD && !AHEAD && a.addend) fetch_add(gr, row0, av[gr & 1]);
            if (n >= a.N) continue;
            SumCoef<BWD> sc[G];
            if (sums) {
#pragma unroll
                for (int q = 0; q < G; ++q) sc[q].load(sN, BN, cl + 2 * q);
            }
#pragma unroll
            for (int mi = 0; mi < MI; ++mi)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int p = row0 + mi * 16 + h * 8;
                    if (p >= a.P) continue;
                    const uint32_t e = ((uint32_t)p * (uint32_t)a.N + (uint32_t)n) * 2u;
                    CVec<C> ov;
#pragma unroll
                    for (int q = 0; q < G; ++q) {
                        float2 v = make_float2(acc[mi][gr * G + q][2 * h], acc[mi][gr * G + q][2 * h + 1]);
                        if (BWD && a.addend) v = __fadd2_rn(v, unpack2(av[gr & 1][mi][h].w[q]));
                        if (!BWD && a.bias) v = __fadd2_rn(v, make_float2(__ldg(a.bias + n + 2 * q), __ldg(a.bias + n + 2 * q + 1)));
                        ov.w[q] = pack2(v);
                        if (sums) ov.w[q] = sc[q].add(ov.w[q], BWD ? zv[gr][mi][h].w[q] : 0u, rlo, rhi, BWD && a.r_mask, s1[gr * G + q], s2[gr * G + q]);
                    }
                    ov.store(a.out, e);
                }
        }
        if (BWD && sums && tile + (int)gridDim.x < a.m_tiles) fetch_z(tile + gridDim.x);
    }
    if (a.late) pdl_launch();
    if (!sums) return;
#pragma unroll
    for (int i = 0; i < NJ; ++i) {
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            s1[i].x += __shfl_xor_sync(0xffffffffu, s1[i].x, o);
            s1[i].y += __shfl_xor_sync(0xffffffffu, s1[i].y, o);
            s2[i].x += __shfl_xor_sync(0xffffffffu, s2[i].x, o);
            s2[i].y += __shfl_xor_sync(0xffffffffu, s2[i].y, o);
        }
    }
    if (g == 0) {
#pragma unroll
        for (int i = 0; i < NJ; ++i) {
            const int cl = (i / G) * 8 * G + 2 * G * t + 2 * (i % G);
            *reinterpret_cast<float2*>(red + (wm * 2 + 0) * BN + cl) = s1[i];
            *reinterpret_cast<float2*>(red + (wm * 2 + 1) * BN + cl) = s2[i];
        }
    }
    __syncthreads();
    for (int i = tid; i < 2 * BN; i += blockDim.x) {
        const int s = i >= BN ? 1 : 0, cl = i - s * BN;
        if (n0 + cl >= a.N) continue;
        float v = 0.f;
        for (int m = 0; m < a.WM; ++m) v += red[(m * 2 + s) * BN + cl];
        add_sum(a.so.sums, (size_t)s * a.N + n0 + cl, v);
    }
}

// ---------------------------------------------------------------------------------------------------------------------
// Small maps: one tile of 16*WM pixels x 8*NJ columns per CTA, the reduction split over WK warps (256 threads = WM * WK warps) so that
// a layer of a few hundred pixels still spreads over the chip and a long reduction costs one memory latency instead of K/32.
template <bool BWD, int NJ, int G, int WK, int XF>
__global__ void __launch_bounds__(256) pw_mma_split_kernel(const Args a) {
    if (BWD) pdl_launch();
    extern __shared__ __align__(16) uint8_t sm[];
    constexpr int WM = 8 / WK, BM = 16 * WM, BN = 8 * NJ, RP = BN + 4, D = BWD ? 3 : 4;
    constexpr bool USE_Z = BWD ? XF != XF_NONE : XF == XF_ADD;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int wm = warp % WM, wk = warp / WM;
    const int n0 = blockIdx.y * BN, Kp = a.KCH * 32, p0 = blockIdx.x * BM;
    uint8_t* sW = sm;
    float* sK = reinterpret_cast<float*>(sW + (size_t)BN * a.wpitch);
    float* sN = sK + (BWD ? 5 : 3) * Kp;
    float* racc = sN + (BWD ? 4 : 1) * BN;                 // [WK][BM][RP]
    stage_weights<G>(a, sW, n0, BN);
    pdl_wait();
    if (!BWD) pdl_launch();

    const size_t r0 = (size_t)min(p0 + wm * 16 + g, a.P - 1) * a.K * 2, r1 = (size_t)min(p0 + wm * 16 + g + 8, a.P - 1) * a.K * 2;
    const uint8_t *ra0 = reinterpret_cast<const uint8_t*>(a.a) + r0, *ra1 = reinterpret_cast<const uint8_t*>(a.a) + r1;
    const uint8_t *rz0 = reinterpret_cast<const uint8_t*>(a.az) + r0, *rz1 = reinterpret_cast<const uint8_t*>(a.az) + r1;
    uint4 rx[D][2], rzv[D][2];
    auto fetch = [&](int kc, uint4* x, uint4* z) {
        const int o = min(kc * 64 + t * 16, a.K * 2 - 16);
        x[0] = *reinterpret_cast<const uint4*>(ra0 + o);
        x[1] = *reinterpret_cast<const uint4*>(ra1 + o);
        if (USE_Z) {
            z[0] = *reinterpret_cast<const uint4*>(rz0 + o);
            z[1] = *reinterpret_cast<const uint4*>(rz1 + o);
        }
    };
#pragma unroll
    for (int d = 0; d < D; ++d)
        if (wk + d * WK < a.KCH) fetch(wk + d * WK, rx[d], rzv[d]);
    // epilogue operands of this thread's first output vector (8 channels of one pixel): requested before the reduction
    constexpr int EPT = 256 / NJ;                          // pixel rows per epilogue pass
    const int er = tid / NJ, ej = tid - er * NJ, en = n0 + ej * 8;
    const bool eact = er < EPT && en < a.N, sums = (bool)a.so.sums;
    uint4 ead = make_uint4(0, 0, 0, 0), erz = ead;
    if (BWD && eact && er < BM && p0 + er < a.P) {
        const size_t e = ((size_t)(p0 + er) * a.N + en) >> 3;
        if (a.addend) ead = reinterpret_cast<const uint4*>(a.addend)[e];
        if (sums) erz = reinterpret_cast<const uint4*>(a.rz)[e];
    }
    stage_coefs<BWD, XF>(a, sK, sN, n0, BN);
    cp_wait<0>();
    __syncthreads();

    const uint8_t* wb = sW + (uint32_t)g * a.wpitch + t * 16;
    float acc[NJ][4];
#pragma unroll
    for (int j = 0; j < NJ; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[j][q] = 0.f;
    Xf<BWD, XF> xf;
    xf.set_act(a.act);
    for (int kb = wk; kb < a.KCH; kb += D * WK) {
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const int kc = kb + d * WK;
            if (kc < a.KCH) {
                xf.load(sK, Kp, kc * 32 + t * 8);
                const uint4 c0 = xf.apply(rx[d][0], rzv[d][0]), c1 = xf.apply(rx[d][1], rzv[d][1]);
                if (!BWD && XF == XF_ADD && blockIdx.y == 0 && kc * 64 + t * 16 < a.K * 2) {
                    const int p = p0 + wm * 16 + g;
                    uint8_t* so = reinterpret_cast<uint8_t*>(a.sum_out) + (size_t)p * a.K * 2 + (uint32_t)(kc * 64 + t * 16);
                    if (p < a.P) *reinterpret_cast<uint4*>(so) = c0;
                    if (p + 8 < a.P) *reinterpret_cast<uint4*>(so + (size_t)16 * a.K) = c1;
                }
                if (kc + D * WK < a.KCH) fetch(kc + D * WK, rx[d], rzv[d]);
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    const uint4 b = *reinterpret_cast<const uint4*>(wb + (uint32_t)(j * 8) * a.wpitch + (uint32_t)kc * 64u);
                    mma16816(acc[j], c0.x, c1.x, c0.y, c1.y, b.x, b.y);
                    mma16816(acc[j], c0.z, c1.z, c0.w, c1.w, b.z, b.w);
                }
            }
        }
    }
    constexpr int C = 2 * G;
#pragma unroll
    for (int gr = 0; gr < NJ / G; ++gr)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float* d = racc + ((size_t)wk * BM + wm * 16 + g + h * 8) * RP + gr * 8 * G + C * t;
#pragma unroll
            for (int i = 0; i < C; i += 2) *reinterpret_cast<float2*>(d + i) = make_float2(acc[gr * G + (i >> 1)][2 * h], acc[gr * G + (i >> 1)][2 * h + 1]);
        }
    __syncthreads();
    const float rlo = a.r_act == ACT_NONE ? -INFINITY : 0.f, rhi = a.r_act == ACT_RELU6 ? 6.f : INFINITY;
    float2 s1[4], s2[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) s1[i] = s2[i] = make_float2(0.f, 0.f);
    if (eact) {
        for (int r = er; r < BM && p0 + r < a.P; r += EPT) {
            float v[8];
            lds8(racc + (size_t)r * RP + ej * 8, v);
#pragma unroll
            for (int k = 1; k < WK; ++k) {
                float u[8];
                lds8(racc + ((size_t)k * BM + r) * RP + ej * 8, u);
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] += u[i];
            }
            const size_t e = ((size_t)(p0 + r) * a.N + en) >> 3;
            if (BWD && r != er) {
                if (a.addend) ead = reinterpret_cast<const uint4*>(a.addend)[e];
                if (sums) erz = reinterpret_cast<const uint4*>(a.rz)[e];
            }
            const uint32_t wa[4] = {ead.x, ead.y, ead.z, ead.w}, wz[4] = {erz.x, erz.y, erz.z, erz.w};
            uint32_t wo[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float2 f = make_float2(v[2 * q], v[2 * q + 1]);
                if (BWD && a.addend) f = __fadd2_rn(f, unpack2(wa[q]));
                if (!BWD && a.bias) f = __fadd2_rn(f, make_float2(__ldg(a.bias + en + 2 * q), __ldg(a.bias + en + 2 * q + 1)));
                wo[q] = pack2(f);
                if (sums) {
                    SumCoef<BWD> sc;
                    sc.load(sN, BN, ej * 8 + 2 * q);
                    wo[q] = sc.add(wo[q], wz[q], rlo, rhi, BWD && a.r_mask, s1[q], s2[q]);
                }
            }
            reinterpret_cast<uint4*>(a.out)[e] = make_uint4(wo[0], wo[1], wo[2], wo[3]);
        }
    }
    if (!sums) return;
    __syncthreads();
    float* red = racc;                                     // [EPT][2][BN]
    constexpr int used = BM < EPT ? BM : EPT;
    if (er < used) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            *reinterpret_cast<float2*>(red + (er * 2 + 0) * BN + ej * 8 + 2 * q) = s1[q];
            *reinterpret_cast<float2*>(red + (er * 2 + 1) * BN + ej * 8 + 2 * q) = s2[q];
        }
    }
    __syncthreads();
    // four threads per (sum, channel), their shares combined in order
    for (int i0 = 0; i0 < 2 * BN * 4; i0 += 256) {
        const int i = i0 + tid, u = i >> 2, part = i & 3;
        float v = 0.f;
        if (u < 2 * BN)
            for (int m = part; m < used; m += 4) v += red[(m * 2 + (u >= BN ? 1 : 0)) * BN + (u >= BN ? u - BN : u)];
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        const int s = u >= BN ? 1 : 0, cl = u - s * BN;
        if (part == 0 && u < 2 * BN && n0 + cl < a.N) add_sum(a.so.sums, (size_t)s * a.N + n0 + cl, v);
    }
}

}  // namespace mma
}  // namespace ast
