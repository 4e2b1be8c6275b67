// Acceptance weights of the multi-draft greedy block verifier (Eq. 2 and Eq. 3, float64) and the scan of
// Algorithm 1, shared by the finishing kernels of the one-device path and of the vocabulary-sharded path.
#pragma once

#include "sgbv_common.cuh"

namespace sgbv {

// 1 - (1-u)^K as the geometric sum u (1 + (1-u) + ... + (1-u)^(K-1)): all terms are positive, so
// a tiny u keeps its full relative accuracy, and no transcendental function is needed.  gsum: the sum, that is (1 - (1-u)^K) / u.
__device__ __forceinline__ double gsum(double u, int K) {
    const double v = 1.0 - fmin(fmax(u, 0.0), 1.0);
    double sum = 1.0;
#pragma unroll 1
    for (int j = 1; j < K; ++j) sum = fma(sum, v, 1.0);
    return sum;
}
__device__ __forceinline__ double gfun(double u, int K) { return fmin(fmax(u, 0.0), 1.0) * gsum(u, K); }

__device__ __forceinline__ double clamp01(double x) {
    if (!(x > 0.0)) return 0.0;
    return x > 1.0 ? 1.0 : x;
}

// Eq. 2 from the three cached sums of the row that follows the sub-block (all divided by Zq):
//   R = sum_x q (1 - min{c p/q,1})^K,  Dp = sum_x max(c p - q, 0),  M = sum_x q (c-t)^2 Q(t).
// numerator/a   = R                                  (c >= 1)
//               = M + K (1-c)^(K-1) Dp               (c <  1, `exact`; equals R - (1-c)^K term by term)
//               = R - (1-c)^K                        (c <  1, not `exact`: only where plain_form_is_safe says so)
// denominator/a = numerator/a + g(b)/a - g(min(c,1))
// with g(b)/a = c (g(b)/b).  a = exp(la).  Hardly a branch: the kernels run this once per CTA, on code that no cache holds yet and
// with lanes that take every way (5,500 cycles with branches, three divisions and serial exponentials).
static __device__ double weight_sub(double a, double la, double lb, double R, double Dp, double M, int K, bool below_one, bool exact) {
    const double b = exp_flat(lb), c = exp_flat(lb - la);
    const double gba = c * gsum(b, K);
    // (1-c)^(K-1) and g(c)/c side by side; below_one was decided on the float32 c that the reduction pass used
    const double v = 1.0 - c, v01 = 1.0 - fmin(c, 1.0);
    double pw = 1.0, sum = 1.0;
#pragma unroll 1
    for (int j = 1; j < K; ++j) {
        pw *= v;
        sum = fma(sum, v01, 1.0);
    }
    const double num = !below_one ? R : exact ? fma((double)K * pw, Dp, M) : fmax(fma(-pw, v, R), 0.0);
    const double extra = !below_one ? gba - 1.0 : K == 1 ? 0.0 : gba - fmin(c, 1.0) * sum;
    const double den = num + fmax(extra, 0.0);
    if (!(a > 0.0)) return b > 0.0 ? 0.0 : 1.0;
    if (!(gba < (double)INFINITY)) return 0.0;  // c beyond the largest double, a beyond the smallest normal one: num / den without a number
    if (!(den > 1e-12 * (gba + 1.0))) return 1.0;  // 0/0: accept, as single-draft GBV does
    return clamp01(num / den);
}

// For c < 1 the numerator of Eq. 2 over a is R - (1-c)^K, a difference of two numbers of which R carries the rounding
// of a float32 vocabulary sum (a few 1e-7 relative).  As long as (1-c)^K is at most half of R the difference loses at
// most one bit of that; beyond (p close to q on the part of the vocabulary that matters) the sums Dp and M, whose
// terms are all non-negative, are needed.
static __device__ bool plain_form_is_safe(double R, double c, int K) {
    double pw = 1.0;
    for (int j = 0; j < K; ++j) pw *= (1.0 - c);
    return pw <= 0.5 * R;
}

// Eq. 3.
static __device__ double weight_full(double la, double lb, int K) {
    const double a = exp_flat(la), b = exp_flat(lb);
    double c = exp_flat(lb - la);
    if (!(a > 0.0) || c > 1.0) c = 1.0;
    const double den = gfun(b, K);
    if (!(den > 0.0)) return 0.0;
    return clamp01(a * gfun(c, K) / den);
}

// Sets one bit of a 64-bit set in shared memory: an atomic on its 32-bit half, which the hardware does in one go (on 64
// bits it is a loop of compare-and-swaps).
__device__ __forceinline__ void set_bit(unsigned long long *set, int bit) {
    atomicOr(reinterpret_cast<unsigned *>(set) + (bit >> 5), 1u << (bit & 31));
}

// Algorithm 1's scan over drafts and lengths by one warp (all 32 lanes call).  pass_s[k]: bit i-1 is set when the
// trial of length i of draft k succeeds (eta < h); lcp_s[k*K+k']: longest common prefix of drafts k and k'.
// Every lane returns the accepted length tau and the draft f (-1 if none).
static __device__ void scan_block(const unsigned long long *pass_s, const unsigned char *lcp_s, int K, int g, int &tau, int &f) {
    const int lane = threadIdx.x & 31;
    // The state is bit sets over the lengths 1..gamma (bit i-1 = length i).  Lane l owns drafts l and l + 32: pass = the
    // lengths whose Bernoulli trial succeeds (eta < h), inH = the lengths at which an earlier draft with the same prefix
    // of that length entered H (tested and not accepted).  A draft's walk over i = tau+1..gamma does not depend on its own
    // progress (the start is fixed when the draft is entered, H only holds earlier drafts), so it is evaluated for all
    // lengths at once: the accepted length is the largest one in the range whose trial passes and whose sub-block is not
    // in H.  Per draft: its owner's two sets to all lanes (four shuffles), and every lane marks its own drafts' common
    // prefixes with it.  No branch in the loop, so that the lanes stay together (8 drafts: 4.7 -> 0.8 us).
    auto low = [](int l) { return l >= 64 ? ~0ull : (1ull << l) - 1ull; };  // lengths 1..l
    const unsigned long long pass0 = lane < K ? pass_s[lane] : 0ull, pass1 = lane + 32 < K ? pass_s[lane + 32] : 0ull;
    unsigned long long inH0 = 0, inH1 = 0;
    const unsigned char *row0 = lcp_s + (lane < K ? lane : 0) * K, *row1 = lcp_s + (lane + 32 < K ? lane + 32 : 0) * K;
    tau = 0;
    f = -1;
#pragma unroll 1
    for (int k = 0; k < K; ++k) {
        const int l0 = row0[k], l1 = row1[k];
        const unsigned long long passk = __shfl_sync(0xffffffffu, k < 32 ? pass0 : pass1, k & 31);
        const unsigned long long inHk = __shfl_sync(0xffffffffu, k < 32 ? inH0 : inH1, k & 31);
        const unsigned long long range = low(g) & ~low(tau);  // lengths tau+1..gamma (none behind a whole block)
        const unsigned long long acc = passk & ~inHk & range, rej = range & ~acc;
        f = acc != 0ull ? k : f;
        tau = acc != 0ull ? 64 - __clzll((long long)acc) : tau;
        inH0 |= rej & low(l0);  // (a draft before k never looks again)
        inH1 |= rej & low(l1);
    }
}

}  // namespace sgbv
