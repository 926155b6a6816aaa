// BatchNorm coefficients formed where they are used.
//
// A kernel that writes a tensor also takes two sums per channel of it (the statistics of the BatchNorm behind it, or the
// two sums of a BatchNorm's backward) and adds its CTAs' partial sums to an accumulator per channel and sum in global memory.  The
// first kernel that READS the tensor turns the sums into the layer's coefficients in its prologue (a few channels per
// thread, ~0.5 us, overlapped with its first operand loads) and one of its CTAs also writes them out for the kernels that
// come later.  No finishing kernel sits on the dependent chain: one cost 4-6 us per BatchNorm and direction, and finishing in the
// producer's last CTA (ticket, fence, one round of L2 reads) still 4 us on a kernel of 2.3 us.
//
// Order of the additions: CTAs add in any order, and the results must not depend on it.  An accumulator is therefore an integer: a partial sum (a
// float) is its 24-bit mantissa shifted by its exponent's place among the 26 that share a 64-bit word, and one integer addition, exact
// in any order.  Two such words cover what partial sums are in earnest.  The lowest bit of the first stays free of sums and says that the
// accumulator has something in the words for the rest, from subnormal numbers to the largest float, and what is not finite.  There is
// room for MAX_SUM_BLOCKS partial sums a channel: a launch has at most some 2 000 blocks a channel, the SiLU backward at least one a sample.
// Before, an accumulator was a double, whose additions are exact only as long as the partial sums lie within 2^-30 of the sum of their
// magnitudes.  A round of a sixth of MobileNetV2 at batch 4 takes 1639 us, with doubles 1581.  Also exact and slower: two-sums, each addition's rounding
// taken from the value the atomic addition returns (1743: the kernels wait for it); a second atomic addition for every partial sum, as a
// checksum beside a double (1753) or as the upper half of a word (1768); four words (1684) or a conversion for each of two (1649).
#pragma once
#include "kernels.h"

namespace ast {

constexpr int SUM_STEP = 26;       // exponents that share a word
constexpr int NEAR_WORD = 4;       // words 4 and 5 are ChanSums::near, the others FarSum::word (6 to 10 at 4 to 8; 9: what is not finite)

// One CTA's partial sum of a channel -> the channel's accumulator.
__device__ __forceinline__ void add_sum(const ChanSums& a, size_t i, float v) {
    const unsigned u = __float_as_uint(v), e = (u >> 23) & 255u;
    const int d = (int)e - 1 + a.shift - NEAR_WORD * SUM_STEP;
    unsigned long long* near = reinterpret_cast<unsigned long long*>(a.near + i);
    if ((unsigned)d < 2u * SUM_STEP) {
        const int w = d >= SUM_STEP;
        const unsigned long long m = (unsigned long long)((u & 0x7fffffu) | 0x800000u) << (d - SUM_STEP * w + 1);
        atomicAdd(near + w, (int)u < 0 ? 0ull - m : m);
    } else if (u << 1) {
        const int p = (e ? (int)e - 1 : 0) + a.shift, w = p / SUM_STEP;
        unsigned long long m = (unsigned long long)((u & 0x7fffffu) | (e ? 0x800000u : 0u)) << (p - SUM_STEP * w);
        if ((int)u < 0) m = 0ull - m;
        if (e == 255u) m = u & 0x7fffffu ? 1ull << 40 : (int)u < 0 ? 1ull << 20 : 1ull;       // counts of NaN, -inf, +inf
        atomicAdd(reinterpret_cast<unsigned long long*>(a.far[i].word + (e == 255u ? 9 : w < NEAR_WORD ? w : w - 2)), m);
        atomicOr(near, 1ull);
    }
}
__device__ __forceinline__ void zero_sum(const ChanSums& a, size_t i) {
    if (a.near[i].x & 1) a.far[i] = FarSum{};
    a.near[i] = make_longlong2(0, 0);
}
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }
// The two words as one number, less as many of its last bits as it has beyond 61, rounded to double.  One conversion: each costs 2 % of a round of
// small maps.
__device__ __forceinline__ double near_total(const longlong2& n, int shift) {
    const int top = (int)(n.y >> 32), drop = min(max(29 - __clz(top ^ (top >> 31)), 0), SUM_STEP);       // |n.y| < 2^(35 + drop)
    return (double)((n.x >> drop) + (n.y << (SUM_STEP - drop))) * pow2(NEAR_WORD * SUM_STEP - 150 - shift + drop);
}
// Sums i and j with all their words.
static __device__ __noinline__ double2 full_totals(longlong2* near, const FarSum* far, int shift, int i, int j) {
    double t[2];
    for (int k = 0; k < 2; ++k) {
        longlong2 n = near[k ? j : i];
        const bool more = n.x & 1;
        n.x &= ~1ll;
        t[k] = near_total(n, shift);
        if (!more) continue;
        const FarSum& f = far[k ? j : i];
        double up = 0.0, down = 0.0;
        for (int w = 8; w >= NEAR_WORD; --w) up = fma((double)f.word[w], pow2(SUM_STEP * (w + 2) - 149 - shift), up);
        for (int w = NEAR_WORD - 1; w >= 0; --w) down = fma((double)f.word[w], pow2(SUM_STEP * w - 149 - shift), down);
        t[k] = up + t[k] + down;
        const long long s = f.word[9], neg = (s >> 20) & 0xfffff, pos = s & 0xfffff;
        if (s) t[k] = s >> 40 || (pos && neg) ? (double)NAN : pos ? (double)INFINITY : -(double)INFINITY;
    }
    return make_double2(t[0], t[1]);
}
// Two sums of a channel.  `load` requests them; a thread with several channels requests all of them before it uses any.
struct TwoSums {
    longlong2 n1, n2;
    __device__ __forceinline__ void load(const ChanSums& a, int i, int j) {
        n1 = a.near[i];
        n2 = a.near[j];
    }
    __device__ __forceinline__ void get(const ChanSums& a, int i, int j, double* s1, double* s2) const {
        *s1 = near_total(n1, a.shift);
        *s2 = near_total(n2, a.shift);
        if (__builtin_expect((n1.x | n2.x) & 1, 0)) {
            const double2 f = full_totals(a.near, a.far, a.shift, i, j);
            *s1 = f.x;
            *s2 = f.y;
        }
    }
};

// Sums of (z - pivot) and (z - pivot)^2 of one channel -> scale and shift; `write`: also everything the slot and the running
// estimates keep.  Arithmetic in double, as the standalone finishing kernels of bn_ew.cu.
struct BnFwdIn {
    TwoSums s;
    float pivot, gamma, beta, run_mean, run_var;
    // everything `coef` needs, the running estimates too: read there they are another trip to memory, and the CTA that writes is the one the
    // kernel behind waits for
    __device__ __forceinline__ void load(const BnPendFwd& b, int ch, bool write) {
        s.load(b.sums, ch, b.c + ch);
        pivot = b.pivot[ch];
        gamma = b.gamma[ch];
        beta = b.beta[ch];
        if (write) {
            run_mean = b.o.run_mean[ch];
            run_var = b.o.run_var[ch];
        }
    }
    __device__ __forceinline__ float2 coef(const BnPendFwd& b, int ch, bool write) const {
        double s1, s2;
        s.get(b.sums, ch, b.c + ch, &s1, &s2);
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
            b.o.run_mean[ch] = (float)((1.0 - b.momentum) * run_mean + b.momentum * mean);
            b.o.run_var[ch] = (float)((1.0 - b.momentum) * run_var + b.momentum * (var * b.unbias));
        }
        return r;
    }
};
__device__ __forceinline__ float2 bn_fwd_coef(const BnPendFwd& b, int ch, bool write) {
    BnFwdIn in;
    in.load(b, ch, write);
    return in.coef(b, ch, write);
}

// Sums of dpre and dpre * xhat of one channel -> the coefficients of dz = k1*dpre + k2 + k3*z; `write`: also the parameter
// gradients and the coefficients themselves.
struct BnBwdIn {
    TwoSums s;
    float rstd, mean, gamma;
    __device__ __forceinline__ void load(const BnPendBwd& b, int ch) {
        s.load(b.sums, ch, b.c + ch);
        rstd = b.rstd[ch];
        mean = b.mean[ch];
        gamma = b.gamma[ch];
    }
    __device__ __forceinline__ float3 coef(const BnPendBwd& b, int ch, bool write) const {
        double s1, s2;
        s.get(b.sums, ch, b.c + ch, &s1, &s2);
        const double r = rstd, m = mean, k1 = (double)gamma * r;
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
};
__device__ __forceinline__ float3 bn_bwd_coef(const BnPendBwd& b, int ch, bool write) {
    BnBwdIn in;
    in.load(b, ch);
    return in.coef(b, ch, write);
}

}  // namespace ast
