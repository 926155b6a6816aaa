// BatchNorm coefficients formed where they are used.
//
// A kernel that writes a tensor also takes two sums per channel of it (the statistics of the BatchNorm behind it, or the
// two sums of a BatchNorm's backward) and adds its CTAs' partial sums to a double per channel and sum in global memory.  The
// first kernel that READS the tensor turns the sums into the layer's coefficients in its prologue (a few channels per
// thread, ~0.5 us, overlapped with its first operand loads) and one of its CTAs also writes them out for the kernels that
// come later.  No finishing kernel sits on the dependent chain: one cost 4-6 us per BatchNorm and direction, and finishing in the
// producer's last CTA (ticket, fence, one round of L2 reads) still 4 us on a kernel of 2.3 us.
//
// Order of the additions: the partial sums are floats (24 bits) and the accumulators doubles (53 bits), so the additions of a
// channel are exact, and therefore independent of their order, as long as its partial sums lie within 2^-29 / n of each other
// in magnitude; below that the part that could be rounded is 2^-53 of a sum that is itself rounded to 24 bits in the end.
#pragma once
#include "kernels.h"

namespace ast {

// Sums of (z - pivot) and (z - pivot)^2 of one channel -> scale and shift; `write`: also everything the slot and the running
// estimates keep.  Arithmetic in double, as the standalone finishing kernels of bn_ew.cu.
__device__ __forceinline__ float2 bn_fwd_coef(const BnPendFwd& b, int ch, bool write) {
    const double s1 = b.sums[ch], s2 = b.sums[b.c + ch];
    const float pivot = b.pivot[ch], gamma = b.gamma[ch], beta = b.beta[ch];
    const double m1 = s1 * b.inv_count, mean = (double)pivot + m1;
    double var = fma(-m1, m1, s2 * b.inv_count);
    if (var < 0.0) var = 0.0;
    const double rstd = rsqrt(var + (double)b.eps), sc = (double)gamma * rstd;
    const float2 r = make_float2((float)sc, (float)((double)beta - mean * sc));
    if (write) {
        b.o.mean[ch] = (float)mean;
        b.o.rstd[ch] = (float)rstd;
        b.o.scale[ch] = r.x;
        b.o.shift[ch] = r.y;
        b.o.run_mean[ch] = (float)((1.0 - b.momentum) * b.o.run_mean[ch] + b.momentum * mean);
        b.o.run_var[ch] = (float)((1.0 - b.momentum) * b.o.run_var[ch] + b.momentum * (var * b.unbias));
    }
    return r;
}

// Sums of dpre and dpre * xhat of one channel -> the coefficients of dz = k1*dpre + k2 + k3*z; `write`: also the parameter
// gradients and the coefficients themselves.
__device__ __forceinline__ float3 bn_bwd_coef(const BnPendBwd& b, int ch, bool write) {
    const double s1 = b.sums[ch], s2 = b.sums[b.c + ch], r = b.rstd[ch], m = b.mean[ch], k1 = (double)b.gamma[ch] * r;
    const float3 k = make_float3((float)k1, (float)(k1 * (s2 * m * r - s1) * b.inv_count), (float)(-k1 * s2 * r * b.inv_count));
    if (write) {
        b.o.dbeta[ch] = (float)s1;
        b.o.dgamma[ch] = (float)s2;
        b.o.k1[ch] = k.x;
        b.o.k2[ch] = k.y;
        b.o.k3[ch] = k.z;
    }
    return k;
}

// One CTA's partial sum of a channel -> the channel's accumulator.
__device__ __forceinline__ void add_sum(double* acc, float v) { atomicAdd(acc, (double)v); }

}  // namespace ast
