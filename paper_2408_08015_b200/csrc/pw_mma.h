// Host interface of the register-operand pointwise kernels (pw_mma.cu).
#pragma once
#include "kernels.h"

namespace ast {

// A tiling of the layer.  wk == 1: persistent CTAs of wm warps, a warp owns 16*mi pixels x 8*nj columns and the whole reduction;
// wk > 1: one tile of 16*(8/wk) pixels x 8*nj columns per CTA, the reduction split over wk warps.
struct MmaTiling {
    int mi, nj, wm, wk;
    int ctas;                  // wk == 1: CTAs per multiprocessor the grid is sized for
};

struct MmaProblem {
    int P, K, N;
    ValSrc x;                  // forward operand
    GradSrc dz;                // backward operand
    BnPendFwd pf;              // pending coefficients of x
    // a deferred residual sum (sum_out not null): the forward operand is sum_act(x + x2), both without an activation of their own, and the
    // kernel also writes it out
    ValSrc x2;
    BnPendFwd pf2;
    void* sum_out;
    int sum_act;
    bool sum_large;            // mma_deep_sum said so: the roundings of the elementwise pass, operands requested several steps ahead
    BnPendBwd pb;              // pending coefficients of dz
    const void* w;             // [N][K]
    const float* bias;
    const void* addend;
    void* out;
    BnSumsOut so;              // column sums of the output (sums null: none)
    const BnRed* red;          // backward: the unit the sums belong to
};

// Chooses a tiling; false: the layer does not run here (pw_tc.cu has the kernels for it).
bool mma_choose(bool bwd, int P, int K, int N, MmaTiling* out);
// whether a forward of this tiling, one CTA to all of the layer's columns, can request the operands of a deferred sum several steps ahead
bool mma_deep_sum(int P, int K, const MmaTiling& c);
size_t mma_smem(bool bwd, int K, const MmaTiling& c);
void mma_launch(bool bwd, const MmaProblem& p, const MmaTiling& c, int kind, double bytes, cudaStream_t st);

// ---- weight gradient (pw_wgrad_mma.cu)
struct WgradProblem {
    int P, CO, CI;
    ValSrc x;
    GradSrc dz;
    BnPendBwd pb;              // pending coefficients of dz; pend_write: this kernel also writes them out
    int pend_write;
};
// a CTA: 8*vm channels of the wider side x 8*vn of the narrower; `splits` pixel ranges, `cluster` of them summed in the kernel
struct WgradTiling {
    int vm, vn, splits, cluster;
};
// pipeline_fits: the pipelined kernel of pw_tc.cu takes the layer
bool wgrad_mma_choose(int P, int CO, int CI, bool pipeline_fits, size_t scratch_floats, WgradTiling* out);
size_t wgrad_mma_smem(const WgradTiling& c);
void wgrad_mma_launch(const WgradProblem& p, const WgradTiling& c, float* scratch, float* gw, cudaStream_t st);

// ---- float32 (pw_f32.cu): columns per lane, warps on the reduction, CTAs per multiprocessor; false: not whole vectors of four channels
struct F32Tiling {
    int tn, wk, ctas;
};
bool f32_choose(bool bwd, int P, int K, int N, F32Tiling* out);
size_t f32_smem(bool bwd, int K, const F32Tiling& c);
void f32_launch(bool bwd, const MmaProblem& p, const F32Tiling& c, int kind, double bytes, cudaStream_t st);
// narrow-side channels per lane; pixel ranges, `cluster` of them summed in the kernel
struct F32WgradTiling {
    int tn, splits, cluster;
};
bool f32_wgrad_choose(int P, int CO, int CI, size_t scratch_floats, F32WgradTiling* out);
void f32_wgrad_launch(const WgradProblem& p, const F32WgradTiling& c, float* scratch, float* gw, cudaStream_t st);

}  // namespace ast
