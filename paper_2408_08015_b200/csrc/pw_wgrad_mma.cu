// Weight gradient of a pointwise convolution,  gw[k][c] = sum_p dz[p][k] * x[p][c],  on mma.sync with register operands.
//
// The reduction runs over the pixels, so a fragment register holds two PIXELS of one channel while memory has the channels of a
// pixel side by side.  A lane therefore loads the same VM (VN) consecutive channels of four pixels, transforms them (BatchNorm +
// activation of x, BatchNorm backward of dy with z), rounds, and pairs the pixels up with byte permutes: what it then holds are the
// registers of VM / 2 row tiles (VN column tiles) at once, with row g of the tiles standing for channels VM*g + i.  No operand passes
// through shared memory and no barrier separates the warps: every warp owns an 8*VM x 8*VN block of the gradient and walks its
// own pixels.
//
// At the end the warps of a CTA add their blocks in order through shared memory, and the CTAs of a cluster (up to eight pixel ranges
// of one block) through each other's shared memory, a slice each.  With one cluster per block that is the gradient; more
// leave a partial each for the split-sum kernel.
#include <string.h>

#include "pw_mma.cuh"
#include "pw_mma.h"

namespace ast {
namespace {

using namespace mma;
constexpr int WARPS = 8;

struct WmArgs {
    const void *dy, *z, *x;
    GradSrc dz;                           // coefficients of the gradient's transform
    ValSrc xs;                            // coefficients of x's
    BnPendBwd pb;
    int pend_write;                       // this kernel also writes the pending coefficients and parameter gradients out
    float* out;                           // gw, or the clusters' partials [gridDim.x / cluster][CO][CI]
    int P, CO, CI;
    int mb;                               // blocks along the M side (blockIdx.y % mb), rest along the N side
    int pix_per_cta;                      // multiple of 16
    int xf_d;                             // the gradient needs z
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

// Warps and pixel ranges are added in pairs: four ranges, whose warps chain two products, instead of eight leave 64 x 384 at 784 pixels 7.8e-8 (2-norm, against
// 7.6e-8) from its sum in 64 bits when added one after the other, in pairs 7.0e-8.  The same number of additions; the other cuts gain as well: 576 x 96
// 7.8 -> 7.0e-8, 160 x 960 10.9 -> 10.4e-8.
__device__ __forceinline__ float sum8(const float* q) { return ((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7])); }

// V consecutive channels (V * 2 bytes)
template <int V> struct Raw {
    uint32_t w[V / 2];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < V / 2; ++i) w[i] = 0;
    }
    __device__ __forceinline__ void load(const uint8_t* p) {
        if constexpr (V == 8) *reinterpret_cast<uint4*>(w) = *reinterpret_cast<const uint4*>(p);
        else if constexpr (V == 4) *reinterpret_cast<uint2*>(w) = *reinterpret_cast<const uint2*>(p);
        else w[0] = *reinterpret_cast<const uint32_t*>(p);
    }
};

// One side of the product: 8*V channels from c0 of one operand.  GRAD: the gradient (dy with z), else x.
template <int V, bool GRAD> struct Side {
    const uint8_t *p, *pz;
    size_t pitch;
    const float* co;                      // shared: gradient k1, k2, k3, scale, shift; x scale, shift; [.][8*V]
    int g;
    bool ok, act, xf;
    float hi;
    uint32_t top;
    Raw<V> r[4], z[4];
    __device__ __forceinline__ void init(const WmArgs& a, int c0, int lane_g, const float* coef) {
        g = lane_g;
        co = coef + V * lane_g;
        const int c = c0 + V * lane_g, total = GRAD ? a.CO : a.CI;
        ok = c < total;
        pitch = (size_t)total * 2;
        p = reinterpret_cast<const uint8_t*>(GRAD ? a.dy : a.x) + (size_t)(ok ? c : 0) * 2;
        pz = reinterpret_cast<const uint8_t*>(a.z) + (size_t)(ok ? c : 0) * 2;
        const int ac = GRAD ? a.dz.act : a.xs.act;
        act = ac != ACT_NONE;
        xf = GRAD ? a.xf_d != 0 : (a.xs.scale != nullptr || act);
        hi = ac == ACT_RELU6 ? 6.f : INFINITY;
        top = ac == ACT_RELU6 ? 0x40C040C0u : 0x7F807F80u;
    }
    // pixels p0 + 2t, +1, +8, +9 (those at or past pend re-read the last one: a finite value, zeroed after the transform)
    __device__ __forceinline__ void fetch(int p0, int t, int last) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const size_t px = (size_t)min(p0 + 2 * t + (i & 1) + (i >> 1) * 8, last);
            r[i].load(p + px * pitch);
            if (GRAD && xf) z[i].load(pz + px * pitch);
        }
    }
    // transformed, rounded, pixels paired: f[j][0..1] channel 2j, f[j][2..3] channel 2j+1 (pixel pairs 2t and 2t+8)
    __device__ __forceinline__ void fragments(int p0, int t, int pend, uint32_t (*f)[4]) {
        constexpr int CW = 8 * V;
#pragma unroll
        for (int j = 0; j < V / 2; ++j) {
            uint32_t w[4];
            if (xf) {
                if (GRAD) {
                    const float2 k1 = *reinterpret_cast<const float2*>(co + 2 * j), k2 = *reinterpret_cast<const float2*>(co + CW + 2 * j),
                                 k3 = *reinterpret_cast<const float2*>(co + 2 * CW + 2 * j);
                    if (act) {
                        const float2 s = *reinterpret_cast<const float2*>(co + 3 * CW + 2 * j), h = *reinterpret_cast<const float2*>(co + 4 * CW + 2 * j);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float2 d = unpack2(r[i].w[j]), zz = unpack2(z[i].w[j]), pre = __ffma2_rn(zz, s, h);
                            float2 o = __ffma2_rn(k3, zz, k2);
                            if (pre.x > 0.f && pre.x < hi) o.x = fmaf(k1.x, d.x, o.x);
                            if (pre.y > 0.f && pre.y < hi) o.y = fmaf(k1.y, d.y, o.y);
                            w[i] = pack2(o);
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i) w[i] = pack2(__ffma2_rn(k1, unpack2(r[i].w[j]), __ffma2_rn(k3, unpack2(z[i].w[j]), k2)));
                    }
                } else {
                    const float2 s = *reinterpret_cast<const float2*>(co + 2 * j), h = *reinterpret_cast<const float2*>(co + CW + 2 * j);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        w[i] = pack2(__ffma2_rn(unpack2(r[i].w[j]), s, h));
                        if (act) w[i] = __vimin_s16x2_relu(w[i], top);
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) w[i] = r[i].w[j];
            }
            if (p0 + 16 > pend) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (p0 + 2 * t + (i & 1) + (i >> 1) * 8 >= pend) w[i] = 0;
            }
            f[j][0] = __byte_perm(w[0], w[1], 0x5410);
            f[j][1] = __byte_perm(w[2], w[3], 0x5410);
            f[j][2] = __byte_perm(w[0], w[1], 0x7632);
            f[j][3] = __byte_perm(w[2], w[3], 0x7632);
        }
    }
};

// MDZ: the gradient is the M side (CO >= CI)
template <int VM, int VN, bool MDZ>
__global__ void __launch_bounds__(WARPS * 32) pw_wgrad_mma_kernel(const WmArgs a) {
    extern __shared__ __align__(16) float st[];
    // the block in shared memory with the input channels contiguous: what is summed over the cluster and written out is then read and written in rows
    constexpr int BM = 8 * VM, BN = 8 * VN, BC = MDZ ? BN : BM, SP = BC + 1, BLK = (BM * BN / BC) * SP, NM = MDZ ? 5 : 2, NN = MDZ ? 2 : 5;
    __shared__ __align__(16) float coef[NM * BM + NN * BN];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int m0 = ((int)blockIdx.y % a.mb) * BM, n0 = ((int)blockIdx.y / a.mb) * BN;
    pdl_wait();
    pdl_launch();

    const int pbeg = blockIdx.x * a.pix_per_cta, pend = min(a.P, pbeg + a.pix_per_cta);
    Side<VM, MDZ> sm_;
    Side<VN, !MDZ> sn_;
    sm_.init(a, m0, g, coef);
    sn_.init(a, n0, g, coef + NM * BM);
    int p0 = pbeg + warp * 16;
    if (p0 < pend) {
        sm_.fetch(p0, t, a.P - 1);
        sn_.fetch(p0, t, a.P - 1);
    }
    {
        const int dw = MDZ ? BM : BN, d0 = MDZ ? m0 : n0, xw = MDZ ? BN : BM, x0 = MDZ ? n0 : m0;
        float *sk = MDZ ? coef : coef + NM * BM, *sx = MDZ ? coef + NM * BM : coef;
        const bool wr = a.pend_write && blockIdx.x == 0 && (MDZ ? n0 == 0 : m0 == 0);
        for (int c = tid; c < dw; c += WARPS * 32) {
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
        for (int c = tid; c < xw; c += WARPS * 32) {
            const bool ok = x0 + c < a.CI && a.xs.scale;
            sx[c] = ok ? a.xs.scale[x0 + c] : 1.f;
            sx[xw + c] = ok ? a.xs.shift[x0 + c] : 0.f;
        }
    }
    __syncthreads();
    float acc[VM / 2][VN][4];
#pragma unroll
    for (int i = 0; i < VM / 2; ++i)
#pragma unroll
        for (int j = 0; j < VN; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;
    for (; p0 < pend; p0 += WARPS * 16) {
        uint32_t fm[VM / 2][4], fn[VN / 2][4];
        sm_.fragments(p0, t, pend, fm);
        sn_.fragments(p0, t, pend, fn);
        if (p0 + WARPS * 16 < pend) {
            sm_.fetch(p0 + WARPS * 16, t, a.P - 1);
            sn_.fetch(p0 + WARPS * 16, t, a.P - 1);
        }
#pragma unroll
        for (int i = 0; i < VM / 2; ++i)
#pragma unroll
            for (int j = 0; j < VN; ++j)
                mma16816(acc[i][j], fm[i][0], fm[i][2], fm[i][1], fm[i][3], fn[j >> 1][(j & 1) * 2], fn[j >> 1][(j & 1) * 2 + 1]);
    }
    // ---- this warp's block -> shared memory, the CTA's sum into the first block
    {
        float* d = st + warp * BLK;
#pragma unroll
        for (int i = 0; i < VM / 2; ++i)
#pragma unroll
            for (int j = 0; j < VN; ++j) {
                const int m = VM * g + 2 * i, n = VN * 2 * t + j;
                auto at = [&](int mm, int nn) -> float& { return d[MDZ ? mm * SP + nn : nn * SP + mm]; };
                at(m, n) = acc[i][j][0];
                at(m, n + VN) = acc[i][j][1];
                at(m + 1, n) = acc[i][j][2];
                at(m + 1, n + VN) = acc[i][j][3];
            }
    }
    __syncthreads();
    for (int e = tid; e < BM * BN; e += WARPS * 32) {
        float* d = st + (e / BC) * SP + e % BC;
        float q[8];
#pragma unroll
        for (int w = 0; w < WARPS; ++w) q[w] = d[w * BLK];
        d[0] = sum8(q);
    }
    uint32_t cs, rank;
    asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(cs));
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    if (cs > 1) cluster_sync();
    else __syncthreads();
    float* out = a.out + (size_t)(blockIdx.x / cs) * a.CO * a.CI;
    const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(st);
    const int per = (BM * BN + (int)cs - 1) / (int)cs, e0 = (int)rank * per, e1 = min(BM * BN, e0 + per);
    for (int e = e0 + tid; e < e1; e += WARPS * 32) {
        const int kr = e / BC, cc = e - kr * BC;
        float s = 0.f;
        if (cs == 1) s = st[kr * SP + cc];
        else {
            const uint32_t ad = s0 + (uint32_t)(kr * SP + cc) * 4u;
            float q[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) q[k] = k < (int)cs ? ld_cluster(ad, k) : 0.f;
            s = sum8(q);
        }
        const int k = (MDZ ? m0 : n0) + kr, c = (MDZ ? n0 : m0) + cc;
        if (k < a.CO && c < a.CI) out[(size_t)k * a.CI + c] = s;
    }
    if (cs > 1) cluster_sync();               // no CTA leaves while another still reads its block
}

typedef void (*WKernel)(const WmArgs);
template <bool MDZ> WKernel wkernel(int vm, int vn) {
    if (vm == 8) return vn == 8 ? pw_wgrad_mma_kernel<8, 8, MDZ> : vn == 4 ? pw_wgrad_mma_kernel<8, 4, MDZ> : pw_wgrad_mma_kernel<8, 2, MDZ>;
    return vn == 4 ? pw_wgrad_mma_kernel<4, 4, MDZ> : pw_wgrad_mma_kernel<4, 2, MDZ>;
}

}  // namespace

// Which layers run here and how they are cut.  Times: the weight gradient of one layer with its split sum, in a captured chain; "before"
// is the tensor-memory pipeline of pw_tc.cu, or its one-tile kernel where the pipeline does not fit the layer.
//   - Up to 4 096 pixels, everything: 160 x 960 at 784 pixels 56.4 -> 10.6 us, 576 x 96 at 3 136 34.5 -> 13.1, 384 x 64 at 784 10.4 -> 5.3,
//     192 x 32 at 3 136 8.5 -> 6.7.  On larger maps the pipeline's bulk copies and larger tiles win (144 x 24 at 50 176 pixels:
//     15.9 us against 23.5), except over layers it does not fit (480 x 80 at 6 272 pixels: 34.5 -> 18.5) and gradients so small that one
//     warp block holds them (16 x 32 at 200 704 pixels: 20.4 -> 14.0).
//   - 32 x 32 blocks (64 x 64 from 960 x 320 up, where the re-reads of 32 x 32 blocks cost more than the idle multiprocessors); about one
//     and a half CTAs per multiprocessor, of which two fit one (one of the 64 x 64 blocks': a second wave for the last two of 150 CTAs made
//     320 x 960 at 784 pixels 25.9 us instead of 14.9); up to eight pixel ranges are one cluster, which writes the gradient itself.  In clusters of four and eight a range
//     is at least a group of 16 pixels for every warp (512, 1 024 pixels): shorter ones are as fast alone, but the sums over a CTA's warps and its coefficients are paid
//     for by the dependent chain beside it (four ranges instead of eight at 784 pixels: sixth of MobileNetV2 at batch 4 1427 -> 1380 us a round).  Clusters of
//     two and ranges with a partial each go down to 64 pixels; there the longer range has not been measured.
bool wgrad_mma_choose(int P, int CO, int CI, bool pipeline_fits, size_t scratch_floats, WgradTiling* out) {
    if (CO % 8 || CI % 8) return false;
    if (P > 4096 && !(P <= 16384 && !pipeline_fits) && CO * CI > 512) return false;
    const int CM = CO > CI ? CO : CI, CN = CO > CI ? CI : CO;
    WgradTiling c{4, CN <= 16 ? 2 : 4, 1, 1};
    if ((size_t)CM * CN >= 300000) c = WgradTiling{8, 8, 1, 1};
    const int blocks = ((CM + 8 * c.vm - 1) / (8 * c.vm)) * ((CN + 8 * c.vn - 1) / (8 * c.vn));
    int sp = sm_count() * (c.vm == 8 ? 2 : 3) / 2 / blocks;
    const int most = P / 64 > 0 ? P / 64 : 1;
    if (sp > most) sp = most;
    if (P > 50000) sp = 2 * sm_count() / 8 * 8;
    if (sp <= 11) {
        c.cluster = sp >= 6 && P >= 8 * 16 * WARPS ? 8 : sp >= 3 && P >= 4 * 16 * WARPS ? 4 : sp >= 2 ? 2 : 1;
        if (c.cluster > most) c.cluster = 1;
        c.splits = c.cluster;
    } else {
        c.cluster = P > 50000 ? 8 : 1;
        c.splits = sp > 32 && P <= 50000 ? 32 : sp;
        if ((size_t)(c.splits / c.cluster) * CO * CI > scratch_floats) return false;
    }
    *out = c;
    return true;
}

size_t wgrad_mma_smem(const WgradTiling& c) {                // the larger of the two layouts
    const size_t a = (size_t)8 * c.vm * (8 * c.vn + 1), b = (size_t)8 * c.vn * (8 * c.vm + 1);
    return (size_t)WARPS * (a > b ? a : b) * 4;
}

void wgrad_mma_launch(const WgradProblem& p, const WgradTiling& c, float* scratch, float* gw, cudaStream_t st) {
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(done.load(std::memory_order_acquire) & bit)) {
        for (int vm : {8, 4})
            for (int vn : {8, 4, 2}) {
                if (vn > vm) continue;
                cudaFuncSetAttribute(wkernel<true>(vm, vn), cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
                cudaFuncSetAttribute(wkernel<false>(vm, vn), cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
            }
        done.fetch_or(bit, std::memory_order_release);
    }
    WmArgs a;
    memset(&a, 0, sizeof a);
    a.dy = p.dz.dy; a.z = p.dz.z; a.x = p.x.p;
    a.dz = p.dz; a.xs = p.x; a.pb = p.pb; a.pend_write = p.pend_write;
    a.xf_d = p.dz.act != ACT_NONE || p.dz.k1 || p.pb.sums;
    a.P = p.P; a.CO = p.CO; a.CI = p.CI;
    const bool mdz = p.CO >= p.CI;
    const int BM = 8 * c.vm, BN = 8 * c.vn, CM = mdz ? p.CO : p.CI, CN = mdz ? p.CI : p.CO;
    a.mb = (CM + BM - 1) / BM;
    const int nb = (CN + BN - 1) / BN, parts = c.splits / c.cluster;
    a.pix_per_cta = ((p.P + c.splits - 1) / c.splits + 15) / 16 * 16;
    const size_t out_elems = (size_t)p.CO * p.CI;
    a.out = parts > 1 ? scratch : gw;
    const double bytes = 2.0 * p.P * p.CO * (a.xf_d ? 2.0 : 1.0) + 2.0 * (double)p.P * p.CI + 4.0 * out_elems;
    {
        LaunchScope ls(K_PW_BWD_WEIGHT_TC, bytes, 2.0 * p.P * (double)out_elems, st);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c.splits, a.mb * nb);
        cfg.blockDim = dim3(32 * WARPS);
        cfg.dynamicSmemBytes = wgrad_mma_smem(c);
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
        cudaLaunchKernelEx(&cfg, mdz ? wkernel<true>(c.vm, c.vn) : wkernel<false>(c.vm, c.vn), a);
    }
    if (parts > 1) {
        LaunchScope ls(K_REDUCE_SPLITS, 4.0 * out_elems * (parts + 1), (double)out_elems * parts, st);
        reduce_splits_f4(scratch, parts, out_elems, gw, st);
    }
}

}  // namespace ast
