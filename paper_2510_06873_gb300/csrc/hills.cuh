// The FP64 hill sum of one system (Methods, Eqs. 2-3, a per-dimension sigma)
// and the well-tempered deposit, shared by the hill kernels and the fused
// small-system step.  Include only from files compiled with -fmad=false, so
// every instantiation rounds every operation alike.
#pragma once

#include "exp2.cuh"
#include "metad_impl.cuh"

namespace metad {

// The difference s - c along CV d wrapped to the nearest image: hill_diff for
// a difference of at most 1.5 periods either way (any hill centre within one
// period of the CV's own range), with the image chosen by integer compares of
// the bit patterns instead of FP64 multiplies and a rounding; further away
// hill_diff itself.
static __device__ __forceinline__ double hill_wrap(const Sys &s, int d, double x)
{
    const double P = s.period[d];
    if (!(__double2hiint(P) > 0)) return x;
    const long long ax = __double_as_longlong(x) & 0x7fffffffffffffffll;  // |x|, ordered as an integer
    if (ax >= __double_as_longlong(s.three_half[d])) return hill_diff(s, d, x);
    const double k = ax > __double_as_longlong(s.half[d]) ? (__double2hiint(x) < 0 ? P : -P) : 0.0;
    return x + k;
}

// V and dV/ds at xin into out (V, then dV/ds_d, kMaxCv of them); with
// deposit, also appends the well-tempered hill there as hill s.K.  s.D
// dimensions (at most kMaxCv).  Every block sums its chunk of the hills; the
// last block to finish adds the block partials in a fixed order and its
// thread 0 writes out.  Returns true in every thread of that last block.
// kD: the most dimensions this instance takes (fewer registers with two).
//
// Bound by the FP64 pipe (two lanes per clock and SM).  A hill of a two-CV
// bias takes 11 FP64 instructions (two differences, the exponent in units of
// log 2, the height, four sums) where exp and the scaled gradient terms made
// it 43, and the block sums go through shared memory, every lane adding eight
// values, instead of a shuffle tree per warp and value (about 40 warp
// instructions a block for 120).
template <int kD>
static __device__ __forceinline__ bool hill_sum(const Sys &s, Blk blk, const double *xin, double *out, int deposit)
{
    const int K = s.K, D = s.D, hs = s.hstride;
    double x[kD], k2v[kD], v[kD + 1];
#pragma unroll
    for (int d = 0; d < kD; ++d) {
        x[d] = d < D ? xin[d] : 0.0;
        k2v[d] = d < D ? s.k2v[d] : 0.0;  // log2(e) / (2 sigma_d^2), formed on the host
        v[1 + d] = 0.0;
    }
    v[0] = 0.0;
    // block b takes the contiguous chunk [b chunk, (b + 1) chunk) of the hills
    const int chunk = (K + blk.nb - 1) / blk.nb;
    const int k1 = min(K, (blk.b + 1) * chunk);
    for (int k = blk.b * chunk + threadIdx.x; k < k1; k += blockDim.x) {
        const double *c = s.hc + (size_t)hs * k;
        double dd[kD];
        double y = 0.0;
#pragma unroll
        for (int d = 0; d < kD; ++d) {
            if (d >= D) break;
            dd[d] = hill_wrap(s, d, x[d] - c[d]);
            y = d == 0 ? dd[d] * dd[d] * k2v[d] : y + dd[d] * dd[d] * k2v[d];
        }
        const double gk = s.hw[k] * exp2_neg(y);
        v[0] += gk;
#pragma unroll
        for (int d = 0; d < kD; ++d) {
            if (d >= D) break;
            v[1 + d] = fma(gk, dd[d], v[1 + d]);
        }
    }
    // block sums in a fixed order: warp q sums value q, lane l the threads
    // l, l + 32, ..., then a tree
    constexpr int kW = kBlockBias / 32;
    static_assert(kW == 8 && kW > kD, "a warp per value, eight terms per lane");
    __shared__ double sh[kD + 1][kBlockBias];
    __shared__ double tot[kD + 1];
    __shared__ bool am_last;
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    __syncthreads();  // a caller's earlier use of the arrays is over
#pragma unroll
    for (int d = 0; d <= kD; ++d)
        if (d <= D) sh[d][threadIdx.x] = v[d];
    __syncthreads();
    double *part = s.part + 2 * (size_t)s.part_stride;
    double a = 0.0;
    if (q <= D) {
        const double *t = sh[q] + lane;
        a = ((t[0] + t[32]) + (t[64] + t[96])) + ((t[128] + t[160]) + (t[192] + t[224]));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    }
    if (blk.nb > 1) {
        if (q <= D && lane == 0) {
            part[(D + 1) * blk.b + q] = a;
            __threadfence();
        }
        __syncthreads();
        if (threadIdx.x == 0) am_last = atomicAdd(&s.ticket[2], 1u) == (unsigned)blk.nb - 1u;
        __syncthreads();
        if (!am_last) return false;
        __threadfence();
        // the last block adds the partials: lane l of warp q takes blocks
        // l, l + 32, ... of value q in order, then the same tree
        if (q <= D) {
            a = 0.0;
            for (int b = lane; b < blk.nb; b += 32) a += ld_l2(part + (D + 1) * b + q);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
        }
    }
    if (q <= kD && lane == 0)  // a gradient's factor -1 / sigma^2 comes once, at the end
        tot[q] = q > D ? 0.0 : (q == 0 ? a : a * (-2.0 * s.inv2v[q - 1]));
    __syncthreads();
    if (threadIdx.x != 0) return true;
    double out_v[kD + 1];
    for (int i = 0; i <= kD; ++i) out_v[i] = tot[i];
    if (s.ncv == 2 && D == 2) {
        double gv, gg0, gg1;
        grid_value(s, x[0], x[1], gv, gg0, gg1);
        out_v[0] += gv;
        out_v[1] += gg0;
        out_v[2] += gg1;
    }
    for (int i = 0; i <= kMaxCv; ++i) out[i] = i <= kD ? out_v[i] : 0.0;
    if (out == s.scal + kV) s.scal[kCnFac] = out_v[1] * 2.0 / s.n;
    if (blk.nb > 1) s.ticket[2] = 0u;
    if (deposit) {
        const double w = s.w0 * exp(-out_v[0] / s.kbdt);
        for (int d = 0; d < hs; ++d) s.hc[(size_t)hs * K + d] = x[d];
        s.hw[K] = w;
        s.scal[kDepW] = w;
    }
    return true;
}

}  // namespace metad
