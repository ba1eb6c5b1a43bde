// Steps a4-a5 (CV forward) and a7-a8 (adjoint and bias forces).
//
// Per-atom definitions (sorted order i; N(i) the full neighbour list):
//   w_ij = s(r_ij)                 rational switch, stretched to vanish at rc
//   CN_i = sum_j w_ij [unlike]     s1 = (1/N) sum_i CN_i
//   W_i  = sum_j w_ij              q_m(i) = sum_j w_ij Y_m(rhat_ij) / W_i
//   qb_m(i) = (q_m(i) + sum_j w_ij q_m(j)) / (1 + W_i)
//   qb6(i)  = sqrt(4 pi / 13 sum_m qb_m(i)^2)     s2 = (1/N) sum_i qb6(i)
// (computed with unnormalised harmonics and weights K_m, see below)
// Adjoint (reverse mode, the paper's autograd written by hand):
//   b_m(i) = K_m qb_m(i) / (N qb6(i) (1 + W_i))                ds2/dA_m(i)
//   g_m(k) = b_m(k) + sum_i w_ik b_m(i)                        ds2/dq_m(k)
//   h_m(k) = g_m(k) / W_k                                      ds2/dQ_m(k)
//   gam_k  = h(k).q(k) + b(k).qb(k)                            -ds2/dW_k
//   per pair (i, j), d = r_j - r_i:
//     ds2/dw = (h_i + h_j).Y - gam_i - gam_j + b(i).q(j) + b(j).q(i)
//     ds2/dd = ds2/dw w'(r) d/r + w sum_m (h_m(i)+h_m(j)) dY_m/dd
//     ds1/dd = (2/N) w'(r) d/r [unlike]
//   F_i = sum_{j in N(i)} (V1 ds1/dd + V2 ds2/dd)
// Every pass walks full rows, each atom gathering its own sums: no atomics,
// bit-reproducible.  (FP64 with two CVs instead evaluates each unordered pair
// once and adds the pair forces up per atom in a fixed order.)
#include "metad_impl.cuh"

namespace metad {

// Real Y_6^m on the unit sphere, unnormalised: the pole-free associated-
// Legendre parts P_m(z) = d^m P_6 / dz^m (dyadic coefficients from the
// recurrence, exact in float32) times C_m, S_m, the real and imaginary parts
// of (x + i y)^m.  The normalisation enters only through the weights
//   K_0 = 1,  K_m = 2 (6-m)!/(6+m)!   (m > 0),
// with qbar6^2 = sum_m K_m (unnormalised qbar_m)^2 (the 4 pi / 13 of the
// Steinhardt definition cancels against the Y_6^m norms).  K_m is carried as
// a float pair so no rounded constant biases the CV.
// Layout: Y[0] m = 0; Y[2m-1] = P_m C_m; Y[2m] = P_m S_m, m = 1..6.
struct YlmConst {
    float pf[7][4];  // P_m(z) coefficients over z^2 powers (highest first)
    double pd[7][4];
};
__constant__ YlmConst c_ylm;

template <typename real>
__device__ __forceinline__ real ylm_c(int m, int k);
template <>
__device__ __forceinline__ float ylm_c<float>(int m, int k) { return c_ylm.pf[m][k]; }
template <>
__device__ __forceinline__ double ylm_c<double>(int m, int k) { return c_ylm.pd[m][k]; }

// P_m(z): degree 6 - m with the parity of 6 - m.
template <typename real>
__device__ __forceinline__ void legendre_parts(real z, real P[7])
{
#define C_(m, k) ylm_c<real>(m, k)
    real z2 = z * z;
    P[0] = ((C_(0, 0) * z2 + C_(0, 1)) * z2 + C_(0, 2)) * z2 + C_(0, 3);
    P[1] = z * ((C_(1, 0) * z2 + C_(1, 1)) * z2 + C_(1, 2));
    P[2] = (C_(2, 0) * z2 + C_(2, 1)) * z2 + C_(2, 2);
    P[3] = z * (C_(3, 0) * z2 + C_(3, 1));
    P[4] = C_(4, 0) * z2 + C_(4, 1);
    P[5] = z * C_(5, 0);
    P[6] = C_(6, 0);
#undef C_
}

template <typename real>
__device__ __forceinline__ void cs_powers(real x, real y, real C[7], real S[7])
{
    // (x + iy)^m; the first power written out (x 1 - y 0 is not folded to x
    // under IEEE rules: y 0 is not 0 for every y)
    C[0] = real(1);
    S[0] = real(0);
    C[1] = x;
    S[1] = y;
#pragma unroll
    for (int m = 2; m <= 6; ++m) {
        C[m] = x * C[m - 1] - y * S[m - 1];
        S[m] = x * S[m - 1] + y * C[m - 1];
    }
}

// v_k += w Y_k(u) for the 13 harmonics, w applied to the seven Legendre
// parts (seven products before the thirteen accumulations, where forming
// the harmonics first takes twelve).
template <typename real>
__device__ __forceinline__ void ylm13_acc(real x, real y, real z, real w, real v[kNY])
{
    real P[7], C[7], S[7];
    legendre_parts<real>(z, P);
    cs_powers<real>(x, y, C, S);
    v[0] += w * P[0];
#pragma unroll
    for (int m = 1; m <= 6; ++m) {
        const real wp = w * P[m];
        v[2 * m - 1] += wp * C[m];
        v[2 * m] += wp * S[m];
    }
}

// sum_k h_k Y_k(u) and g = (I - u u^T) grad(sum_k h_k Y_k) / r in one loop,
// without materialising the harmonics (fewer live registers in the pair pass).
// dP_m/dz = P_{m+1}, so the parts serve the gradient too, and with
// e_m = hc_m C_m + hs_m S_m a power adds P_m e_m to the sum and P_{m+1} e_m to
// its z derivative: 11 operations a power, and none for the parts'
// derivatives (14 and 12 when each was formed on its own).
template <typename real>
__device__ __forceinline__ real ylm13_dot_grad(real x, real y, real z, real inv_r, const real h[kNY], real g[3])
{
    real P[7], C[7], S[7];
    legendre_parts<real>(z, P);
    cs_powers<real>(x, y, C, S);
    real t = h[0] * P[0];
    real gx = real(0), gy = real(0), gz = h[0] * P[1];
#pragma unroll
    for (int m = 1; m <= 6; ++m) {
        const real hc = h[2 * m - 1], hs = h[2 * m];
        const real e = hc * C[m] + hs * S[m];
        t += P[m] * e;
        if (m < 6) gz += P[m + 1] * e;
        if (m == 1) {  // C_0 = 1, S_0 = 0 (not folded by the compiler: y 0 is not 0 for every y)
            gx += P[1] * hc;
            gy += P[1] * hs;
        } else {
            const real pm = P[m] * real(m);
            gx += pm * (hc * C[m - 1] + hs * S[m - 1]);
            gy += pm * (hs * C[m - 1] - hc * S[m - 1]);
        }
    }
    const real ug = x * gx + y * gy + z * gz;
    g[0] = (gx - ug * x) * inv_r;
    g[1] = (gy - ug * y) * inv_r;
    g[2] = (gz - ug * z) * inv_r;
    return t;
}

// The weights K per Y slot (0 past the 13), as float pairs and in FP64.  Read
// by slots that depend on the lane, so they sit in global memory: a constant
// bank serves one address of a warp at a time.
constexpr double k_weight(int slot)
{
    const int m = (slot + 1) / 2;
    if (slot >= kNY) return 0.0;
    double f = m > 0 ? 2.0 : 1.0;
    for (int k = 6 - m + 1; k <= 6 + m; ++k) f /= k;
    return f;
}
#define METAD_K16(f) f(0), f(1), f(2), f(3), f(4), f(5), f(6), f(7), f(8), f(9), f(10), f(11), f(12), f(13), f(14), f(15)
#define METAD_KHI(m) (float)k_weight(m)
#define METAD_KLO(m) (float)(k_weight(m) - (double)(float)k_weight(m))
static __device__ __align__(16) const float kKhi[16] = {METAD_K16(METAD_KHI)};
static __device__ __align__(16) const float kKlo[16] = {METAD_K16(METAD_KLO)};
static __device__ __align__(16) const double kKd[16] = {METAD_K16(k_weight)};
#undef METAD_K16
#undef METAD_KHI
#undef METAD_KLO

// K of slots 4l .. 4l + 3, and the terms K_m a_m^2 of them.
template <typename real>
struct KWeights;
template <>
struct KWeights<float> {
    float4 hi, lo;
    __device__ __forceinline__ explicit KWeights(int l)
        : hi(__ldg(reinterpret_cast<const float4 *>(kKhi) + l)), lo(__ldg(reinterpret_cast<const float4 *>(kKlo) + l))
    {
    }
    __device__ __forceinline__ void get(float k[4]) const
    {
        k[0] = hi.x;
        k[1] = hi.y;
        k[2] = hi.z;
        k[3] = hi.w;
    }
    __device__ __forceinline__ float sum_sq(const float a[4]) const
    {
        const float x = a[0] * a[0], y = a[1] * a[1], z = a[2] * a[2], w = a[3] * a[3];
        const float h = fmaf(hi.w, w, fmaf(hi.z, z, fmaf(hi.y, y, hi.x * x)));
        const float e = fmaf(lo.w, w, fmaf(lo.z, z, fmaf(lo.y, y, lo.x * x)));
        return h + e;
    }
};
template <>
struct KWeights<double> {
    double k_[4];
    __device__ __forceinline__ explicit KWeights(int l)
    {
#pragma unroll
        for (int c = 0; c < 4; ++c) k_[c] = __ldg(kKd + 4 * l + c);
    }
    __device__ __forceinline__ void get(double k[4]) const
    {
#pragma unroll
        for (int c = 0; c < 4; ++c) k[c] = k_[c];
    }
    __device__ __forceinline__ double sum_sq(const double a[4]) const
    {
        double s = 0.0;
#pragma unroll
        for (int c = 0; c < 4; ++c) s += k_[c] * a[c] * a[c];
        return s;
    }
};

// 16-wide per-atom records (13 used): one 64 B (FP32) or 128 B (FP64) row
// per atom, so a neighbour's record is two sectors, not thirteen.
constexpr int kRec = 16;

template <typename real>
__device__ __forceinline__ void load_rec(const real *base, int i, real v[kRec]);
template <>
__device__ __forceinline__ void load_rec<float>(const float *base, int i, float v[kRec])
{
    const float4 *p = reinterpret_cast<const float4 *>(base + (size_t)i * kRec);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float4 t = p[k];
        v[4 * k] = t.x;
        v[4 * k + 1] = t.y;
        v[4 * k + 2] = t.z;
        v[4 * k + 3] = t.w;
    }
}
template <>
__device__ __forceinline__ void load_rec<double>(const double *base, int i, double v[kRec])
{
    const double2 *p = reinterpret_cast<const double2 *>(base + (size_t)i * kRec);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        double2 t = p[k];
        v[2 * k] = t.x;
        v[2 * k + 1] = t.y;
    }
}
namespace {

template <typename real>
__device__ __forceinline__ real *R(void *p) { return reinterpret_cast<real *>(p); }

// Fixed-order FP64 block sum (result valid in thread 0).
__device__ __forceinline__ double block_sum(double v, double *sh)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
    __syncthreads();
    return t;
}

// Displacement (cached by the exact filter), 1/r, switch weight and its
// derivative of one exact entry, with its neighbour and CN mask.
template <typename real, bool kLast = false>
__device__ __forceinline__ void cached_geometry(const Sys &s, size_t slot, Vec3<real> &d, real &inv_r, real &w,
                                                real &dw, bool &cn, int &j)
{
    load_geo<real, kLast>(s, slot, d, cn, j);
    real r2 = d.x * d.x + d.y * d.y + d.z * d.z;
    inv_r = rsqrt_r<real>(r2);
    switch_eval<real>(s, r2 * inv_r, w, dw);
}

// Butterfly reduce-scatter of 16 values over the G lanes of a group:
// afterwards lane l holds the group sums of values l 16/G .. in v[0] ...
template <typename real, int G>
__device__ __forceinline__ void reduce_scatter16(real v[kRec], int l)
{
    int len = kRec;
#pragma unroll
    for (int o = G / 2; o >= 1; o >>= 1) {
        len >>= 1;
        const bool upper = (l & o) != 0;
#pragma unroll
        for (int t = 0; t < kRec / 2; ++t) {
            if (t < len) {
                real a = v[t], b = v[t + len];
                real send = upper ? a : b;
                real keep = upper ? b : a;
                v[t] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
    }
}

// Sum over the kG lanes of a group, result in every lane.
template <typename real>
__device__ __forceinline__ real group_sum(real v)
{
#pragma unroll
    for (int o = kG / 2; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Components c l .. c l + c - 1 of record i of kLen (c = 2 or 4).
template <typename real, int kLen, int c>
__device__ __forceinline__ void store_part(real *base, int i, int l, const real v[])
{
    struct alignas(c * sizeof(real) < 16 ? c * sizeof(real) : 16) Part {
        real v[c];
    };
    Part p;
#pragma unroll
    for (int k = 0; k < c; ++k) p.v[k] = v[k];
    reinterpret_cast<Part *>(base + (size_t)i * kLen)[l] = p;
}

__device__ __forceinline__ const int *nbr_row(const Sys &s, int i) { return s.nbr + (size_t)i * s.max_nb; }

// Per-thread running sum of a per-atom CV or of pairs' virials.  With FP32
// records it is a compensated pair (Knuth's TwoSum: s + c holds the sum with
// only c's own rounding), so no FP64 instruction runs per atom (their pipe is
// narrow on this part); it enters the FP64 block and grid sums once per thread.
template <typename real>
struct RunSum;
template <>
struct RunSum<float> {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float x)
    {
        const float t = s + x;
        const float bp = t - s;
        c += (s - (t - bp)) + (x - bp);
        s = t;
    }
    // f (hi + lo), the product's rounding error kept
    __device__ __forceinline__ void add_scaled(float f, float hi, float lo)
    {
        const float p = f * hi;
        add(p);
        c += fmaf(f, lo, fmaf(f, hi, -p));
    }
    __device__ __forceinline__ void halve()
    {
        s *= 0.5f;
        c *= 0.5f;
    }
    __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};
template <>
struct RunSum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double x) { s += x; }
    __device__ __forceinline__ void add_scaled(double f, double hi, double) { s += f * hi; }
    __device__ __forceinline__ double value() const { return s; }
};

// Warp tree over RunSum values (lane 0 ends with the warp's sum): FP32
// pairs combine by TwoSum on s and a plain sum of the c terms.
__device__ __forceinline__ void warp_sum(RunSum<float> &v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float os = __shfl_down_sync(0xffffffffu, v.s, o);
        const float oc = __shfl_down_sync(0xffffffffu, v.c, o);
        const float t = v.s + os;
        const float bp = t - v.s;
        v.c += oc + ((v.s - (t - bp)) + (os - bp));
        v.s = t;
    }
}
__device__ __forceinline__ void warp_sum(RunSum<double> &v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v.s += __shfl_down_sync(0xffffffffu, v.s, o);
}
// The sums of four consecutive lanes, the same bits in each.
__device__ __forceinline__ void group4_sum(RunSum<float> &v)
{
#pragma unroll
    for (int o = 2; o >= 1; o >>= 1) {
        const float os = __shfl_xor_sync(0xffffffffu, v.s, o);
        const float oc = __shfl_xor_sync(0xffffffffu, v.c, o);
        const float t = v.s + os;
        const float bp = t - v.s;
        v.c = (v.c + oc) + ((v.s - (t - bp)) + (os - bp));
        v.s = t;
    }
}

// a4: CN_i, W_i and q_m(i) = sum_j w_ij Y_m(rhat_ij) / W_i.  With one CV, CN_i
// and what its force and virial need: sum_j w' d / r and sum_j w' d_a^2 / r
// over the counted pairs (the force on an atom is 2 V1 / N times the first,
// so no later pass walks the rows).
// With kFilter the exact row is first compacted from the Verlet row.
constexpr int kCnRec = 8;  // fx fy fz, vx vy vz; FP32: the error terms of vx vy (that of vz lies in W)

template <typename real, bool kFilter, int G>
__device__ __forceinline__ void cv_fwd_group(const Sys &s, const AtomLane a)
{
    const bool two = sizeof(real) == 4 || s.ncv == 2;  // FP32 with one CV: cv_cn
    int nn_f = 0;
    if (kFilter) nn_f = filter_row<real, G>(s, a);
    real v[kRec];  // 0..12: sum w Y_m (one CV: 0..5 as above) ; 13: W ; 14: CN
#pragma unroll
    for (int m = 0; m < kRec; ++m) v[m] = real(0);
    if (a.ok) {
        const int nn = kFilter ? nn_f : s.nn[a.i];
        JW<real> *jwrow = reinterpret_cast<JW<real> *>(s.wl) + (size_t)a.i * s.max_nb;
        const size_t e0 = entry_base(s, a.i);
        for (int k = a.l; k < nn; k += G) {
            Vec3<real> d;
            real inv_r, w, dw;
            bool cn;
            int j;
            cached_geometry<real>(s, e0 + entry_off(k), d, inv_r, w, dw, cn, j);
            if (cn) v[14] += w;
            v[13] += w;
            if (two) {
                jwrow[k] = JW<real>{j, w};
                ylm13_acc<real>(d.x * inv_r, d.y * inv_r, d.z * inv_r, w, v);
            } else if (cn) {
                const real gx = dw * inv_r * d.x, gy = dw * inv_r * d.y, gz = dw * inv_r * d.z;
                v[0] += gx;
                v[1] += gy;
                v[2] += gz;
                if (s.virial) {
                    v[3] += gx * d.x;
                    v[4] += gy * d.y;
                    v[5] += gz * d.z;
                }
            }
        }
    }
    reduce_scatter16<real, G>(v, a.l);
    // lane l holds values c l .. c l + c - 1; 13: W, 14: CN
    constexpr int c = kRec / G;
    const real W = __shfl_sync(0xffffffffu, v[13 % c], ((threadIdx.x & 31) & ~(G - 1)) + 13 / c);
    if (a.ok) {
        if (a.l == 14 / c) R<real>(s.cn)[a.i] = v[14 % c];
        if (two) {
            if (a.l == 13 / c) R<real>(s.W)[a.i] = W;
            const real inv_W = W > real(0) ? real(1) / W : real(0);
            real q[c];
#pragma unroll
            for (int k = 0; k < c; ++k) q[k] = c * a.l + k < kNY ? v[k] * inv_W : real(0);
            store_part<real, kRec, c>(R<real>(s.q), a.i, a.l, q);
        } else if (a.l < kCnRec / c) {
            store_part<real, kCnRec, c>(R<real>(s.q), a.i, a.l, v);
        }
    }
}

// a4 for FP32 and one CV: CN_i and the force and virial sums straight from the
// candidates, a pair evaluated where it is found.  No row is written (16 B an
// entry, most of the pass's DRAM traffic) or read back; a round evaluates for
// the pairs counted alone, where compacted rows held all.  Each pair's virial
// enters a compensated sum (kVir).
template <bool kVir>
__device__ __forceinline__ void cv_cn_group(const Sys &s, const AtomLane a)
{
    const int i = a.ok ? a.i : 0, vn = a.ok ? s.vnn[i] : 0;
    const float4 pi = s.pos_s[i];
    const int vmax = __reduce_max_sync(0xffffffffu, vn);
    float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};  // force, CN
    RunSum<float> vir[3];
    int cnt = 0;
    sweep_candidates<4>(s, i, a.l, vn, vmax, [&](bool valid, int, float4 pj) {
        Vec3<float> d;
        const bool in = pair_in_warp(s, valid, pi, pj, d);
        cnt += in ? 1 : 0;
        if (in && (!s.cn_unlike || pj.w != pi.w)) {
            const float r2 = d.x * d.x + d.y * d.y + d.z * d.z;
            const float inv_r = rsqrt_r<float>(r2);
            float w, dw;
            switch_eval<float>(s, r2 * inv_r, w, dw);
            // products of their own rounding in both instances: the same forces
            // with the virial and without
            const float g = dw * inv_r;
            const float gx = __fmul_rn(g, d.x), gy = __fmul_rn(g, d.y), gz = __fmul_rn(g, d.z);
            v[0] += gx;
            v[1] += gy;
            v[2] += gz;
            if (kVir) {
                vir[0].add(gx * d.x);
                vir[1].add(gy * d.y);
                vir[2].add(gz * d.z);
            }
            v[3] += w;
        }
    });
#pragma unroll
    for (int o = 2; o >= 1; o >>= 1) {
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    }
    if (kVir) {
#pragma unroll
        for (int k = 0; k < 3; ++k) group4_sum(vir[k]);
    }
    if (!a.ok) return;
    float4 *q = reinterpret_cast<float4 *>(R<float>(s.q) + (size_t)i * kCnRec);
    if (a.l == 0) q[0] = make_float4(v[0], v[1], v[2], vir[0].s);
    if (kVir && a.l == 1) {
        q[1] = make_float4(vir[1].s, vir[2].s, vir[0].c, vir[1].c);
        R<float>(s.W)[i] = vir[2].c;
    }
    if (a.l == 2) R<float>(s.cn)[i] = v[3];
    if (a.l == 3 && cnt > s.max_nb) set_err(s, kErrCapacity);
}

template <bool kVir>
__device__ __forceinline__ void cv_cn(const Sys &s, Blk k)
{
    const int groups = (s.n + kRowAtoms - 1) / kRowAtoms;
    for (int it = 0, g; (g = work_item(k, it)) < groups; ++it) cv_cn_group<kVir>(s, atom_lane_at<4>(s, g));
}

// Resident blocks per SM: 12 without the virial; with its compensated sums 8:
// 30,000 / 900,000 atoms a step 42.5 / 218.8 us, 12: 45.1 / 219.3, 9: 43.0 /
// 226.7.  (The row's virial as a plain float32 sum: 43.6 / 199.8, and three
// times the error of rows of 450.)
template <bool kVir>
constexpr int kCnBlocks = kVir ? 8 : 12;

template <bool kVir>
__global__ void __launch_bounds__(kBlockAtoms, kCnBlocks<kVir>) k_cv_cn(Sys s)
{
    chain_enter();
    cv_cn<kVir>(s, own_blk());
}

template <bool kVir>
__global__ void __launch_bounds__(kBlockAtoms, kCnBlocks<kVir>) kb_cv_cn(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    cv_cn<kVir>(s, k);
}

// Lanes per atom: four in the FP32 pass.  Bound by instruction issue (64 to
// 69%); with eight lanes the last round of a row leaves more lanes idle and
// the reduction over the lanes costs twice as much an atom.  1M atoms 264 ->
// 220 us, 262,144 76 -> 66, 27,648 14.3 -> 14.7 (its warps halve, too few to
// hide the loads' latency).  FP64 keeps eight: its arithmetic is the bound.
template <typename real>
constexpr int kFwdLanes = sizeof(real) == 4 ? 4 : kG;

template <typename real, bool kFilter>
__device__ __forceinline__ void cv_fwd(const Sys &s, Blk k)
{
    constexpr int G = kFwdLanes<real>, atoms = kBlockAtoms / G;
    const int groups = (s.n + atoms - 1) / atoms;
    for (int it = 0, g; (g = work_item(k, it)) < groups; ++it)
        cv_fwd_group<real, kFilter, G>(s, atom_lane_at<G>(s, g));
}

// Resident blocks per SM: 12 in FP32 (40 registers; 10 / 14 / 16: 228 / 230 /
// 230 us at 1M atoms), none asked for in FP64 (40 registers spill there).
template <typename real>
constexpr int kFwdBlocks = sizeof(real) == 4 ? 12 : 0;

template <typename real, bool kFilter>
__global__ void __launch_bounds__(kBlockAtoms, kFwdBlocks<real>) k_cv_fwd(Sys s)
{
    chain_enter();
    cv_fwd<real, kFilter>(s, own_blk());
}

template <typename real>
__global__ void __launch_bounds__(kBlockAtoms, kFwdBlocks<real>) kb_cv_fwd(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    cv_fwd<real, true>(s, k);
}

// Row entries k and k + 1 (k even, so k + 1 lies inside the row's capacity,
// a multiple of four entries; the caller uses the second only below the row
// length).  FP32 entries share one 16 B word (rows start on 32 B): one load,
// and for a lane group reading the same entries one L1 wavefront where two
// 8 B loads take two.  (Four entries in one 32 B load measured slower in
// the Q6 pass: 242 against 158 us at 1M atoms, its registers 32 -> 42.)
template <typename real>
__device__ __forceinline__ void load_jw2(const JW<real> *row, int k, JW<real> &e0, JW<real> &e1)
{
    e0 = row[k];
    e1 = row[k + 1];
}
template <>
__device__ __forceinline__ void load_jw2<float>(const JW<float> *row, int k, JW<float> &e0, JW<float> &e1)
{
    const int4 v = *reinterpret_cast<const int4 *>(row + k);
    e0 = JW<float>{v.x, __int_as_float(v.y)};
    e1 = JW<float>{v.z, __int_as_float(v.w)};
}

// The CV sums: each block's C and Q -> part[b], part[part_stride + b]; the
// last block to finish adds them (lane l of warp 0 resp. 1 takes blocks l,
// l + 32, ... in order, then a fixed tree): s1 = C / N, s2 = Q / N.  A fixed
// association for a given grid.
__device__ void finish_cv_sums(const Sys &s, Blk k, double sum, int which)
{
    // thread 0 holds the block's C, thread 32 its Q
    __shared__ bool am_last;
    const int lane = threadIdx.x & 31;
    if (k.nb > s.part_stride) {  // never with the grids used; refuse rather than overrun
        if (k.b == 0 && threadIdx.x == 0) set_err(s, kErrInternal);
        return;
    }
    if (k.nb > 1) {
        double *part = s.part + (size_t)which * s.part_stride;
        if (which < 2 && lane == 0) {
            part[k.b] = sum;
            __threadfence();
        }
        __syncthreads();
        if (threadIdx.x == 0) am_last = atomicAdd(&s.ticket[0], 1u) == (unsigned)k.nb - 1u;
        __syncthreads();
        if (!am_last) return;
        __threadfence();
        if (which < 2) {
            sum = 0.0;
            for (int b = lane; b < k.nb; b += 32) sum += ld_l2(part + b);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
        }
        if (threadIdx.x == 0) s.ticket[0] = 0u;
    }
    if (which == 0 && lane == 0) s.scal[kS0] = sum / s.n;
    if (which == 1 && lane == 0) {
        if (s.ncv == 2) s.scal[kS1] = sum / s.n;
        else if (!s.lattice) s.scal[kS1] = 0.0;
        if (s.lattice)  // the triaxial lattice parameters follow the per-atom CVs
            for (int a = 0; a < 3; ++a) s.scal[kS0 + s.ncv + a] = s.L[a];
    }
}

// s1, s2: thread t of block b sums CN and qbar6 of atoms b kSumThreads + t,
// + blocks kSumThreads, ... in order (compensated FP32 pairs with FP32
// records), four loads in flight; the warps' trees stay compensated FP32 and
// only one value per warp enters the FP64 sums (a warp-wide FP64 add holds
// the pipe for 64 cycles).  Its own pass, beside the adjoint in a step: the
// Q6 pass then carries no sums, and its blocks no FP64 epilogue (27,648
// atoms: Q6 pass 25.6 -> 10.2 us).
template <typename real>
__device__ __forceinline__ void cv_sum(const Sys &s, Blk k)
{
    RunSum<real> c, q;
    const real *cn = R<real>(s.cn), *q6 = R<real>(s.qb6);
    const int step = k.nb * blockDim.x;
    for (int i = k.b * blockDim.x + threadIdx.x; i < s.n; i += 4 * step) {
        real x[4], y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool in = i + u * step < s.n;
            x[u] = in ? cn[i + u * step] : real(0);
            y[u] = in && s.ncv == 2 ? q6[i + u * step] : real(0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            c.add(x[u]);
            q.add(y[u]);
        }
    }
    constexpr int kW = kSumThreads / 32;
    __shared__ double sh[2][kW];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    warp_sum(c);
    warp_sum(q);
    if (lane == 0) {
        sh[0][wid] = c.value();
        sh[1][wid] = q.value();
    }
    __syncthreads();
    double t = 0.0;
    if (wid < 2 && lane == 0)
        for (int w = 0; w < kW; ++w) t += sh[wid][w];
    finish_cv_sums(s, k, t, wid);
}

template <typename real>
__global__ void __launch_bounds__(kSumThreads) k_cv_sum(Sys s)
{
    chain_enter();
    cv_sum<real>(s, own_blk());
}

template <typename real>
__global__ void __launch_bounds__(kSumThreads) kb_cv_sum(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    cv_sum<real>(s, k);
}

// The row passes a5, a7 and a8 give an atom four lanes; lane l owns record
// components 4l .. 4l + 3 (one 16 B load of each neighbour record per lane),
// so a warp has eight atoms' gathers in flight.
constexpr int kG4 = 4;
static_assert(kRowAtoms * kG4 == kRowThreads && kRowThreads == kBlockAtoms, "four lanes per atom");
constexpr int kRecQB = 32;  // FP32: q and b side by side, in chunks of four

template <typename real>
__device__ __forceinline__ void load4(const real *base, int i, int l, real v[4]);
template <>
__device__ __forceinline__ void load4<float>(const float *base, int i, int l, float v[4])
{
    const float4 t = reinterpret_cast<const float4 *>(base + (size_t)i * kRec)[l];
    v[0] = t.x;
    v[1] = t.y;
    v[2] = t.z;
    v[3] = t.w;
}
template <>
__device__ __forceinline__ void load4<double>(const double *base, int i, int l, double v[4])
{
    const double2 *p = reinterpret_cast<const double2 *>(base + (size_t)i * kRec) + 2 * l;
    const double2 a = p[0], b = p[1];
    v[0] = a.x;
    v[1] = a.y;
    v[2] = b.x;
    v[3] = b.y;
}
template <typename real>
__device__ __forceinline__ void store4(real *base, int i, int l, const real v[4]);
template <>
__device__ __forceinline__ void store4<float>(float *base, int i, int l, const float v[4])
{
    reinterpret_cast<float4 *>(base + (size_t)i * kRec)[l] = make_float4(v[0], v[1], v[2], v[3]);
}
template <>
__device__ __forceinline__ void store4<double>(double *base, int i, int l, const double v[4])
{
    double2 *p = reinterpret_cast<double2 *>(base + (size_t)i * kRec) + 2 * l;
    p[0] = make_double2(v[0], v[1]);
    p[1] = make_double2(v[2], v[3]);
}

// Chunk l of record i of the FP32 q-and-b records: q then b, one 32 B load.
__device__ __forceinline__ void load_qb(const float *base, int i, int l, float q[4], float b[4])
{
    ld_8(base + (size_t)i * kRecQB + 8 * l, q, b);
}

__device__ __forceinline__ void store_b(const Sys &s, int i, int l, const float q[4], const float b[4])
{
    float4 *p = reinterpret_cast<float4 *>(R<float>(s.b) + (size_t)i * kRecQB) + 2 * l;
    p[0] = make_float4(q[0], q[1], q[2], q[3]);
    p[1] = make_float4(b[0], b[1], b[2], b[3]);
}
__device__ __forceinline__ void store_b(const Sys &s, int i, int l, const double *, const double b[4])
{
    store4<double>(R<double>(s.b), i, l, b);
}

template <typename real>
__device__ __forceinline__ real group4_sum(real v)
{
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v;
}

// a5: qbar_m(i), qbar6(i).  Record b: b_m(i) = K_m qbar_m(i) / (N qbar6
// (1 + W_i)) (slots 0..12) and beta_i = b(i).qbar(i) (slot 13); FP32 records
// carry q beside b, for the adjoint to gather both with one load.
template <typename real>
__device__ __forceinline__ void cv_avg_group(const Sys &s, int g)
{
    const int i = g * kRowAtoms + (threadIdx.x / kG4), l = threadIdx.x & (kG4 - 1);
    const bool ok = i < s.n;
    const real *q = R<real>(s.q);
    real a[4] = {real(0), real(0), real(0), real(0)}, o[4] = {real(0), real(0), real(0), real(0)};
    real inv_D = real(0);
    const KWeights<real> K(l);
    if (ok) {
        const int nn = s.nn[i];
        inv_D = real(1) / (real(1) + R<real>(s.W)[i]);
        load4<real>(q, i, l, o);
        const JW<real> *jwrow = reinterpret_cast<const JW<real> *>(s.wl) + (size_t)i * s.max_nb;
        JW<real> n0, n1;  // the entries one round ahead
        load_jw2<real>(jwrow, 0, n0, n1);
#pragma unroll 2
        for (int k = 0; k < nn; k += 2) {
            const JW<real> e0 = n0, e1 = n1;
            if (k + 2 < nn) load_jw2<real>(jwrow, k + 2, n0, n1);
            const bool two = k + 1 < nn;
            real x[4], y[4] = {real(0), real(0), real(0), real(0)};
            load4<real>(q, e0.j, l, x);
            if (two) load4<real>(q, e1.j, l, y);
#pragma unroll
            for (int c = 0; c < 4; ++c) a[c] += e0.w * x[c];
            if (two) {
#pragma unroll
                for (int c = 0; c < 4; ++c) a[c] += e1.w * y[c];
            }
        }
    }
    // slots 13 .. 15 hold 0 in q, so qb is 0 there too
    real qb[4], kw[4], b[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) qb[c] = (o[c] + a[c]) * inv_D;
    const real sq = group4_sum<real>(K.sum_sq(qb));
    const real qb6 = sqrt(sq);
    const real ci = qb6 > real(0) ? inv_D / (n_real<real>(s) * qb6) : real(0);
    K.get(kw);
    real bq = real(0);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        b[c] = ci * kw[c] * qb[c];
        bq += b[c] * qb[c];
    }
    const real beta = group4_sum<real>(bq);
    if (ok) {
        if (l == 3) b[1] = beta;  // slot 13
        store_b(s, i, l, o, b);
        if (l == 0) R<real>(s.qb6)[i] = qb6;
    }
}

template <typename real>
__device__ __forceinline__ void cv_avg(const Sys &s, Blk k)
{
    const int groups = (s.n + kRowAtoms - 1) / kRowAtoms;
    for (int it = 0, g; (g = work_item(k, it)) < groups; ++it) cv_avg_group<real>(s, g);
}

// Blocks per SM: 10 (48 registers); at 1M atoms 8 / 9 / 10 / 12: 145 / 137 / 129
// / 135 us, and 145 without the entries one round ahead.
template <typename real>
constexpr int kAvgBlocks = sizeof(real) == 4 ? 10 : 0;

template <typename real>
__global__ void __launch_bounds__(kRowThreads, kAvgBlocks<real>) k_cv_avg(Sys s)
{
    chain_enter();
    cv_avg<real>(s, own_blk());
}

template <typename real>
__global__ void __launch_bounds__(kRowThreads, kAvgBlocks<real>) kb_cv_avg(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    cv_avg<real>(s, k);
}

// a7: g_m(k) = b_m(k) + sum_i w_ik b_m(i) ; h = g / W ; record h holds h_m
// (0..12) and gamma_k = h(k).q(k) + beta_k (slot 13).
//
// Reduce-scatter of four values over the four lanes of this thread's group:
// lane l returns the group sum of v[l].  The shuffle masks name the group
// alone, so groups of one warp may run different trip counts.
template <typename real>
__device__ __forceinline__ real group4_reduce_scatter(const real v[4], int l)
{
    const unsigned mask = 0xfu << (threadIdx.x & 28);
    const bool hi2 = (l & 2) != 0, hi1 = (l & 1) != 0;
    // lanes 2, 3 keep values 2, 3 and send 0, 1; lanes 0, 1 the reverse
    const real a0 = (hi2 ? v[2] : v[0]) + __shfl_xor_sync(mask, hi2 ? v[0] : v[2], 2);
    const real a1 = (hi2 ? v[3] : v[1]) + __shfl_xor_sync(mask, hi2 ? v[1] : v[3], 2);
    // odd lanes keep the second of their pair, even lanes the first
    return (hi1 ? a1 : a0) + __shfl_xor_sync(mask, hi1 ? a0 : a1, 1);
}

// h and gamma from the gathered sum (acc), the atom's own b (o) and q.
template <typename real>
__device__ __forceinline__ void store_h(const Sys &s, int i, int l, bool ok, const real acc[4], const real o[4],
                                        const real q[4])
{
    real h[4] = {real(0), real(0), real(0), real(0)};
    real alpha = real(0), beta = real(0);
    if (ok) {
        const real W = R<real>(s.W)[i];
        const real inv_W = W > real(0) ? real(1) / W : real(0);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int m = 4 * l + c;
            if (m < kNY) {
                h[c] = (o[c] + acc[c]) * inv_W;
                alpha += h[c] * q[c];
            }
            if (m == 13) beta = o[c];
        }
    }
    alpha = group4_sum<real>(alpha);
    beta = group4_sum<real>(beta);
    if (ok) {
        if (l == 3) h[1] = alpha + beta;  // slot 13: gamma = h.q + b.qbar
        store4<real>(R<real>(s.h), i, l, h);
    }
}

// With each gathered record also the pair's cross term b_i.q_j + b_j.q_i of
// ds2/dw (a8), stored per entry: the neighbour's q lies beside its b, so it
// costs half a line and eight multiply-adds, and the force pass needs nothing
// from the mirror entry.  Two chains, added last: both ends of a pair get the
// same bits.  Entries go four at a time; a reduce-scatter over the group
// leaves entry k0 + l's sum in lane l, so the group stores 16 contiguous
// bytes.
//
// Bound by the latency of the gathered lines: a round's four loads a lane all
// have to be in flight, which takes 64 registers, and the round's entries are
// loaded one round ahead.  1M atoms: 197 us with 40 registers, 229 with 40 and
// the entries after the records, 182 so.  (Eight lanes an atom with 16 B
// loads, half the L1 wavefronts: 233 to 257 us.)
__device__ __forceinline__ void adjoint_group(const Sys &s, int g, float)
{
    const int i = g * kRowAtoms + (threadIdx.x / kG4), l = threadIdx.x & (kG4 - 1);
    const bool ok = i < s.n;
    const float *qb = R<float>(s.b);
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f}, o[4] = {0.0f, 0.0f, 0.0f, 0.0f}, q[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (ok) {
        load_qb(qb, i, l, q, o);
        const int nn = s.nn[i];
        const JW<float> *jwrow = reinterpret_cast<const JW<float> *>(s.wl) + (size_t)i * s.max_nb;
        float *crow = R<float>(s.cross) + entry_base(s, i);
        JW<float> n4[4];  // the entries one round ahead (a row holds at least four)
        load_jw2<float>(jwrow, 0, n4[0], n4[1]);
        load_jw2<float>(jwrow, 2, n4[2], n4[3]);
        for (int k0 = 0; k0 < nn; k0 += 4) {
            JW<float> e4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) e4[u] = n4[u];
            if (k0 + 4 < nn) {
                load_jw2<float>(jwrow, k0 + 4, n4[0], n4[1]);
                load_jw2<float>(jwrow, k0 + 6, n4[2], n4[3]);
            }
            float p[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                p[u] = 0.0f;
                if (k0 + u < nn) {
                    float xq[4], xb[4];
                    load_qb(qb, e4[u].j, l, xq, xb);
                    // slot 13: 0 in q beside beta in b; 14, 15: 0 in both
                    float p1 = xq[0] * o[0], p2 = xb[0] * q[0];
                    acc[0] += e4[u].w * xb[0];
#pragma unroll
                    for (int c = 1; c < 4; ++c) {
                        acc[c] += e4[u].w * xb[c];
                        p1 = fmaf(xq[c], o[c], p1);
                        p2 = fmaf(xb[c], q[c], p2);
                    }
                    p[u] = p1 + p2;
                }
            }
            const float t = group4_reduce_scatter<float>(p, l);
            if (k0 + l < nn) crow[entry_off(k0) + l] = t;
        }
    }
    store_h<float>(s, i, l, ok, acc, o, q);
}

// FP64: the half b_j.q_i of the cross term per entry; the pair pass adds the
// halves of entry ij and its mirror ji.
__device__ __forceinline__ void adjoint_group(const Sys &s, int g, double)
{
    const int i = g * kRowAtoms + (threadIdx.x / kG4), l = threadIdx.x & (kG4 - 1);
    const bool ok = i < s.n;
    const double *bb = R<double>(s.b);
    double acc[4] = {0.0, 0.0, 0.0, 0.0}, o[4] = {0.0, 0.0, 0.0, 0.0}, q[4] = {0.0, 0.0, 0.0, 0.0};
    if (ok) {
        load4<double>(bb, i, l, o);
        load4<double>(R<double>(s.q), i, l, q);
        const int nn = s.nn[i];
        const JW<double> *jwrow = reinterpret_cast<const JW<double> *>(s.wl) + (size_t)i * s.max_nb;
        double *crow = R<double>(s.cross) + entry_base(s, i);
        for (int k0 = 0; k0 < nn; k0 += 4) {
            JW<double> e4[4];
            load_jw2<double>(jwrow, k0, e4[0], e4[1]);
            load_jw2<double>(jwrow, k0 + 2, e4[2], e4[3]);
            double p[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                p[u] = 0.0;
                if (k0 + u < nn) {
                    double x[4];
                    load4<double>(bb, e4[u].j, l, x);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        acc[c] += e4[u].w * x[c];
                        if (4 * l + c < kNY) p[u] += x[c] * q[c];
                    }
                }
            }
            const double t = group4_reduce_scatter<double>(p, l);
            if (k0 + l < nn) crow[entry_off(k0) + l] = t;
        }
    }
    store_h<double>(s, i, l, ok, acc, o, q);
}

template <typename real>
__device__ __forceinline__ void adjoint(const Sys &s, Blk k)
{
    const int groups = (s.n + kRowAtoms - 1) / kRowAtoms;
    for (int it = 0, g; (g = work_item(k, it)) < groups; ++it) adjoint_group(s, g, real(0));
}

// Resident blocks per SM the adjoint is compiled for (none in FP64): 1M atoms
// at 7 / 8 / 9 / 10 / 12: 198 / 182 / 199 / 197 / 324 us (the last two spill).
// Blocks of 256 / 512 / 1024 threads measured no faster: the neighbours'
// records are found in L2 either way, and small blocks balance better.
template <typename real>
constexpr int kAdjointBlocks = sizeof(real) == 4 ? 8 : 0;

template <typename real>
__global__ void __launch_bounds__(kRowThreads, kAdjointBlocks<real>) k_adjoint(Sys s)
{
    chain_enter();
    adjoint<real>(s, own_blk());
}

template <typename real>
__global__ void __launch_bounds__(kRowThreads, kAdjointBlocks<real>) kb_adjoint(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    adjoint<real>(s, k);
}

// a8: G_ij = V1 ds1/dd + V2 ds2/dd at d = r_j - r_i:
//   ds2/dw = (h_i + h_j).Y - gamma_i - gamma_j + b_i.q_j + b_j.q_i
//   ds2/dd = ds2/dw w' d/r + w sum_m (h_i + h_j)_m dY_m/dd
//   ds1/dd = (2/N) w' d/r [unlike]
// and F_i = sum_j G_ij over the whole row (G_ji = -G_ij).
//
// One pair's G (without a CN part, radial is V2 ds2/dw w' alone).
template <typename real>
__device__ __forceinline__ Vec3<real> pair_gradient(const Vec3<real> &d, real inv_r, real w, real dw, real cn_radial,
                                                    real V2, real cross, const real hi[kRec], const real hj[kRec])
{
    const real ux = d.x * inv_r, uy = d.y * inv_r, uz = d.z * inv_r;
    real t = cross - (hi[13] + hj[13]);
    real hs[kNY];
#pragma unroll
    for (int m = 0; m < kNY; ++m) hs[m] = hi[m] + hj[m];
    // (h_i + h_j).Y and its transverse gradient; the w Y term's gradient
    // is w times it
    real gY[3];
    t += ylm13_dot_grad<real>(ux, uy, uz, inv_r, hs, gY);
    const real radial = cn_radial + V2 * t * dw, vw = V2 * w;
    return Vec3<real>{vw * gY[0] + radial * ux, vw * gY[1] + radial * uy, vw * gY[2] + radial * uz};
}

// The chain-rule factors of the two CVs, 2 V1 scale / N and V2 scale.  The
// division is the hill kernel's (an FP64 chain is long and its pipe narrow on
// this part); plain forces take no FP64 arithmetic here.
template <typename real>
__device__ __forceinline__ void chain_factors(const Sys &s, real fac[2])
{
    double f0 = s.scal[kCnFac], f1 = s.ncv == 2 ? s.scal[kDV1] : 0.0;
    if (s.fscale_dev || s.fscale != 1.0) {
        const double scale = force_scale(s);
        f0 *= scale;
        f1 *= scale;
    }
    fac[0] = (real)f0;
    fac[1] = (real)f1;
}

template <typename real>
__device__ __forceinline__ void put_force(const Sys &s, int i, int comp, real f)
{
    float *o = s.F_out + (size_t)s.F_stride * s.perm[i] + comp;
    *o = s.accumulate ? *o + (float)f : (float)f;
}

// The bias virial W_a = sum_pairs (dV/dd)_a d_a, which a barostat needs: it
// gives dV/dL_a at fixed fractional coordinates as W_a / L_a, plus dV/ds of
// a lattice CV.  Per-thread compensated sums, a warp tree, FP64 block
// partials in slot 1 of `part` (free once the CV sums are taken), and the
// last block to finish adds them in block order.
template <typename real>
__device__ void virial_finish(const Sys &s, Blk k, RunSum<real> &vx, RunSum<real> &vy, RunSum<real> &vz)
{
    constexpr int kMaxW = (kRowThreads > kBlockAtoms ? kRowThreads : kBlockAtoms) / 32;
    const int kW = blockDim.x >> 5;
    __shared__ double sh[3][kMaxW];
    __shared__ bool am_last;
    if (3 * k.nb > s.part_stride) {  // never with the grids used; refuse rather than overrun
        if (k.b == 0 && threadIdx.x == 0) set_err(s, kErrInternal);
        return;
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    warp_sum(vx);
    warp_sum(vy);
    warp_sum(vz);
    if (lane == 0) {
        sh[0][wid] = vx.value();
        sh[1][wid] = vy.value();
        sh[2][wid] = vz.value();
    }
    __syncthreads();
    double *part = s.part + s.part_stride;
    if (threadIdx.x == 0) {
        for (int a = 0; a < 3; ++a) {
            double t = 0.0;
            for (int w = 0; w < kW; ++w) t += sh[a][w];
            part[3 * k.b + a] = t;
        }
        __threadfence();
        am_last = atomicAdd(&s.ticket[3], 1u) == (unsigned)k.nb - 1u;
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    // thread t adds partials t, t + blockDim, ... in order into four
    // interleaved accumulators (a short FP64 chain), combined in order
    double acc[3][4] = {};
    for (int b0 = threadIdx.x; b0 < k.nb; b0 += 4 * blockDim.x) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int b = b0 + r * blockDim.x;
            if (b < k.nb) {
#pragma unroll
                for (int a = 0; a < 3; ++a) acc[a][r] += ld_l2(part + 3 * b + a);
            }
        }
    }
    double v[3];
    for (int a = 0; a < 3; ++a) {
        v[a] = (acc[a][0] + acc[a][1]) + (acc[a][2] + acc[a][3]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[a] += __shfl_down_sync(0xffffffffu, v[a], o);
    }
    __syncthreads();
    if (lane == 0)
        for (int a = 0; a < 3; ++a) sh[a][wid] = v[a];
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int a = 0; a < 3; ++a) {
            double t = 0.0;
            for (int w = 0; w < kW; ++w) t += sh[a][w];
            s.scal[kVir0 + a] = t;
            s.scal[kBoxG0 + a] = (s.lattice ? force_scale(s) * s.scal[kDV0 + s.ncv + a] : 0.0) + t / s.L[a];
        }
        s.ticket[3] = 0u;
    }
}

// FP32, two CVs: every atom walks its own row, four lanes an atom, one entry
// per lane, so each pair is evaluated at both ends.  That repeats the pair's
// arithmetic but needs no slots for the pair forces, no search for i in j's
// row and no pass to add the slots up: what bound the half-row form was its
// scattered line accesses (per pair four for h_j, one each for the mirror
// entry's place, its cross half and its force slot), and its 32 B of slots
// per entry were most of the step's DRAM traffic.  Bound by instruction issue
// (about 55%) and the latency of the gathered records.  1M atoms: half rows
// and slot sums 300 us and more, 268 us in a row per atom; 251 with the parts'
// derivatives shared (ylm13_dot_grad), 235 with the rows of eight atoms
// interleaved (entry_slot), 214 with the streamed entries one round ahead, 198
// without a division, a barrier and shared memory in every block
// (chain_factors).
template <bool kVir>
__device__ __forceinline__ void force_rows(const Sys &s, Blk k)
{
    float fac[2];
    chain_factors<float>(s, fac);
    const float cn_fac = fac[0], V2 = fac[1];
    const int l = threadIdx.x & (kG4 - 1);
    const int groups = (s.n + kRowAtoms - 1) / kRowAtoms;
    const float *hh = R<float>(s.h);
    RunSum<float> vx, vy, vz;
    for (int it = 0, g; (g = work_item(k, it)) < groups; ++it) {
        const int i = g * kRowAtoms + (threadIdx.x / kG4);
        float fx = 0.0f, fy = 0.0f, fz = 0.0f;
        if (i < s.n) {
            const int nn = s.nn[i];
            const size_t row = entry_base(s, i) + l;
            const float4 *grow = reinterpret_cast<const float4 *>(s.geo) + row;
            const float *crow = R<float>(s.cross) + row;
            float hi[kRec];
            load_rec<float>(hh, i, hi);
            // the streamed entries one round ahead: their latency is DRAM's
            float4 geo_next = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            float cross_next = 0.0f;
            if (l < nn) {
                geo_next = ld_stream(grow);
                cross_next = ld_stream(crow);
            }
            for (int e = l; e < nn; e += kG4) {
                const float4 geo = geo_next;
                const float cross = cross_next;
                int j;
                bool cn;
                untag(__float_as_uint(geo.w), j, cn);
                float hj[kRec];
                load_rec<float>(hh, j, hj);
                if (e + kG4 < nn) {
                    geo_next = ld_stream(grow + entry_off(e - l + kG4));
                    cross_next = ld_stream(crow + entry_off(e - l + kG4));
                }
                const Vec3<float> d{geo.x, geo.y, geo.z};
                const float r2 = d.x * d.x + d.y * d.y + d.z * d.z;
                const float inv_r = rsqrt_r<float>(r2);
                float w, dw;
                switch_eval<float>(s, r2 * inv_r, w, dw);
                const Vec3<float> G = pair_gradient<float>(d, inv_r, w, dw, cn ? cn_fac * dw : 0.0f, V2, cross, hi, hj);
                fx += G.x;
                fy += G.y;
                fz += G.z;
                if (kVir) {
                    vx.add(G.x * d.x);
                    vy.add(G.y * d.y);
                    vz.add(G.z * d.z);
                }
            }
        }
        fx = group4_sum<float>(fx);
        fy = group4_sum<float>(fy);
        fz = group4_sum<float>(fz);
        if (i < s.n && l < s.F_stride)
            put_force<float>(s, i, l, l == 0 ? fx : (l == 1 ? fy : (l == 2 ? fz : 0.0f)));
    }
    if (kVir) {  // each pair is met at both ends
        vx.halve();
        vy.halve();
        vz.halve();
        virial_finish<float>(s, k, vx, vy, vz);
    }
}

// Resident blocks per SM: 8 (64 registers) in the plain pass, 198 us at 1M
// atoms and 28.6 at 100,000; 9 (56) 196 and 29.3, 7 (72) 210 and 28.7, 10 259
// and 36.7 (spilling); with the virial 7 (72): 250,001 atoms 69.2 us.  (With a
// lane's share of a row's virial summed plainly 67.2, where 8 blocks (64,
// spilling) took 69.7, 6 71.2, and 100 when 86 registers left five of the
// grid's eight blocks per SM resident.)
template <bool kVir>
constexpr int kForceBlocks = kVir ? 7 : 8;

template <bool kVir>
__global__ void __launch_bounds__(kRowThreads, kForceBlocks<kVir>) k_force_rows(Sys s)
{
    chain_enter();
    force_rows<kVir>(s, own_blk());
}

template <bool kVir>
__global__ void __launch_bounds__(kRowThreads, kForceBlocks<kVir>) kb_force_rows(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    force_rows<kVir>(s, k);
}

// One CV: the CV pass left each atom's sum_j w' d / r, so the force is a
// factor away.  One thread per atom.
template <typename real, bool kVir>
__device__ __forceinline__ void force_cn(const Sys &s, Blk k)
{
    real fac[2];
    chain_factors<real>(s, fac);
    const real f = fac[0];
    RunSum<real> vx, vy, vz;
    for (int i = k.b * blockDim.x + threadIdx.x; i < s.n; i += k.nb * blockDim.x) {
        const real *r = R<real>(s.q) + (size_t)i * kCnRec;
        put_force<real>(s, i, 0, f * r[0]);
        put_force<real>(s, i, 1, f * r[1]);
        put_force<real>(s, i, 2, f * r[2]);
        if (s.F_stride == 4) put_force<real>(s, i, 3, real(0));
        if (kVir) {  // each pair is met at both ends
            const real hf = real(0.5) * f;
            vx.add_scaled(hf, r[3], r[6]);
            vy.add_scaled(hf, r[4], r[7]);
            vz.add_scaled(hf, r[5], sizeof(real) == 4 ? R<real>(s.W)[i] : real(0));
        }
    }
    if (kVir) virial_finish<real>(s, k, vx, vy, vz);
}

template <typename real, bool kVir>
__global__ void __launch_bounds__(kBlockAtoms) k_force_cn(Sys s)
{
    chain_enter();
    force_cn<real, kVir>(s, own_blk());
}

template <typename real, bool kVir>
__global__ void __launch_bounds__(kBlockAtoms) kb_force_cn(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    force_cn<real, kVir>(s, k);
}

// FP64, two CVs, pass 1: each unordered pair once (its ~200 FP64 operations
// bound this form, so they are not repeated), from the row of its lower index
// i (entries k < nh_i, j > i): G_ij into the slot of entry k in i's row and
// -G_ij into the slot of i in the j < i part of j's row (rows are symmetric:
// the neighbour predicate is), found by a search of that part.  Pass 2 sums
// each atom's own slots in row order.  The slots are a stream (written once,
// read once): stored and loaded evict-first.
//
// Pair-parallel: the half-row entries of a chunk of atoms are numbered in
// atom order and the lanes of a warp take them in turn: every lane has a pair
// while the chunk lasts, whatever the spread of the half-row lengths.
template <bool kVir>
__device__ __forceinline__ void pair_force(const Sys &s, int i, int k, double cn_fac, double V2, RunSum<double> &vx,
                                           RunSum<double> &vy, RunSum<double> &vz)
{
    Vec3<double> d;
    double inv_r, w, dw;
    bool cn;
    int j;
    cached_geometry<double, true>(s, entry_slot(s, i, k), d, inv_r, w, dw, cn, j);
    int kk = -1;
    const int nhj = s.nh[j], nnj = s.nn[j];
    const int *rj = nbr_row(s, j);
    for (int b = nhj & ~3; b < nnj && kk < 0; b += 4) {  // four entries per load
        const int4 v = *reinterpret_cast<const int4 *>(rj + b);
        if (v.x == i && b >= nhj) kk = b;
        else if (v.y == i && b + 1 >= nhj && b + 1 < nnj) kk = b + 1;
        else if (v.z == i && b + 2 >= nhj && b + 2 < nnj) kk = b + 2;
        else if (v.w == i && b + 3 >= nhj && b + 3 < nnj) kk = b + 3;
    }
    if (kk < 0 || kk >= s.max_nb) {
        set_err(s, kErrInternal);  // rows not symmetric: never expected
        return;
    }
    const double *hh = R<double>(s.h), *cc = R<double>(s.cross);
    double hi[kRec], hj[kRec];
    load_rec<double>(hh, i, hi);
    load_rec<double>(hh, j, hj);
    // cross term b_i.q_j + b_j.q_i: the halves the adjoint pass stored
    // in entry ij (b_j.q_i) and in its mirror ji (b_i.q_j)
    const double cross = cc[entry_slot(s, i, k)] + cc[entry_slot(s, j, kk)];
    const Vec3<double> G = pair_gradient<double>(d, inv_r, w, dw, cn ? cn_fac * dw : 0.0, V2, cross, hi, hj);
    if (kVir) {  // (dV/dd)_a d_a of this pair
        vx.add(G.x * d.x);
        vy.add(G.y * d.y);
        vz.add(G.z * d.z);
    }
    double2 *pi = reinterpret_cast<double2 *>(s.pairF) + 2 * ((size_t)i * s.max_nb + k);
    double2 *pj = reinterpret_cast<double2 *>(s.pairF) + 2 * ((size_t)j * s.max_nb + kk);
    __stcs(pi, make_double2(G.x, G.y));
    __stcs(pi + 1, make_double2(G.z, 0.0));
    __stcs(pj, make_double2(-G.x, -G.y));
    __stcs(pj + 1, make_double2(-G.z, 0.0));
}

template <bool kVir>
__device__ __forceinline__ void force_pairs(const Sys &s, Blk k)
{
    double fac[2];
    chain_factors<double>(s, fac);
    const double cn_fac = fac[0], V2 = fac[1];
    // each warp takes its own chunk of atoms (a block is one work item): no barrier
    constexpr int kWarps = kBlockAtoms / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int chunk = pair_chunk(s.n);
    const int items = (s.n + chunk * kWarps - 1) / (chunk * kWarps);
    RunSum<double> vx, vy, vz;
    for (int it = 0, g; (g = work_item(k, it)) < items; ++it) {
        const int i0 = (g * kWarps + warp) * chunk;
        if (i0 >= s.n) continue;  // warp-uniform
        // inclusive prefix of the half-row lengths, one lane per atom
        int off = lane < chunk && i0 + lane < s.n ? s.nh[i0 + lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, off, o);
            if (lane >= o) off += y;
        }
        const int T = __shfl_sync(0xffffffffu, off, 31);
        for (int p0 = 0; p0 < T; p0 += 32) {
            const int p = p0 + lane;
            // the atom of entry p: the first a whose inclusive prefix exceeds p
            int lo = 0, hi = 31;
#pragma unroll
            for (int step = 0; step < 5; ++step) {
                const int mid = (lo + hi) >> 1;
                if (__shfl_sync(0xffffffffu, off, mid) > p) hi = mid;
                else lo = mid + 1;
            }
            const int prev = __shfl_sync(0xffffffffu, off, lo > 0 ? lo - 1 : 0);  // every lane shuffles
            const int start = lo > 0 ? prev : 0;
            if (p < T) pair_force<kVir>(s, i0 + lo, p - start, cn_fac, V2, vx, vy, vz);
        }
    }
    if (kVir) virial_finish<double>(s, k, vx, vy, vz);
}

template <bool kVir>
__global__ void __launch_bounds__(kBlockAtoms) k_force_pairs(Sys s)
{
    chain_enter();
    force_pairs<kVir>(s, own_blk());
}

template <bool kVir>
__global__ void __launch_bounds__(kBlockAtoms) kb_force_pairs(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    force_pairs<kVir>(s, k);
}

// Pass 2: the slots of i's row summed in row order per lane and by a fixed
// shuffle tree across lanes.
__device__ __forceinline__ void force_gather(const Sys &s, Blk k)
{
    const int groups = group_grid(s.n);
    for (int it = 0, g; (g = work_item(k, it)) < groups; ++it) {
        const AtomLane a = atom_lane_at(s, g);
        double fx = 0.0, fy = 0.0, fz = 0.0;
        if (a.ok) {
            const int nn = s.nn[a.i];
            const double2 *pf = reinterpret_cast<const double2 *>(s.pairF) + 2 * (size_t)a.i * s.max_nb;
            for (int e = a.l; e < nn; e += kG) {
                const double2 u = ld_stream(pf + 2 * e), v = ld_stream(pf + 2 * e + 1);
                fx += u.x;
                fy += u.y;
                fz += v.x;
            }
        }
        fx = group_sum<double>(fx);
        fy = group_sum<double>(fy);
        fz = group_sum<double>(fz);
        if (a.ok && a.l < s.F_stride)
            put_force<double>(s, a.i, a.l, a.l == 0 ? fx : (a.l == 1 ? fy : (a.l == 2 ? fz : 0.0)));
    }
}

__global__ void __launch_bounds__(kBlockAtoms) k_force_gather(Sys s)
{
    chain_enter();
    force_gather(s, own_blk());
}

__global__ void __launch_bounds__(kBlockAtoms) kb_force_gather(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    force_gather(s, k);
}

template <typename real>
__global__ void k_per_atom_out(Sys s, double *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= s.n) return;
    const int u = s.perm[i];
    out[u] = (double)R<real>(s.cn)[i];
    if (s.ncv == 2) out[(size_t)s.n + u] = (double)R<real>(s.qb6)[i];
}


}  // namespace

void launch_cv_fwd(const Sys &s, int fp64, int fused_filter, cudaStream_t st)
{
    const int nb = grid_blocks(s, fp64 ? GK_GROUPS : GK_ROWS, 0);  // by kFwdLanes
    if (!stores_rows(s, fp64)) {
        chained_live(s.virial ? k_cv_cn<true> : k_cv_cn<false>, nb, kBlockAtoms, st, s);
        return;
    }
    if (fp64) {
        if (fused_filter)
            chained_live(k_cv_fwd<double, true>, nb, kBlockAtoms, st, s);
        else
            chained_live(k_cv_fwd<double, false>, nb, kBlockAtoms, st, s);
    } else {
        if (fused_filter)
            chained_live(k_cv_fwd<float, true>, nb, kBlockAtoms, st, s);
        else
            chained_live(k_cv_fwd<float, false>, nb, kBlockAtoms, st, s);
    }
}

void launch_cv_avg(const Sys &s, int fp64, cudaStream_t st)
{
    const int nb = grid_blocks(s, GK_ROWS, 0);
    if (fp64)
        chained_live(k_cv_avg<double>, nb, kRowThreads, st, s);
    else
        chained_live(k_cv_avg<float>, nb, kRowThreads, st, s);
}

void launch_cv_sum(const Sys &s, int fp64, cudaStream_t st)
{
    const int nb = grid_blocks(s, GK_SUM, 0);
    if (fp64)
        chained_live(k_cv_sum<double>, nb, kSumThreads, st, s);
    else
        chained_live(k_cv_sum<float>, nb, kSumThreads, st, s);
}

void launch_adjoint(const Sys &s, int fp64, cudaStream_t st)
{
    const int nb = grid_blocks(s, GK_ROWS, 0);
    if (fp64)
        chained_live(k_adjoint<double>, nb, kRowThreads, st, s);
    else
        chained_live(k_adjoint<float>, nb, kRowThreads, st, s);
}

namespace {

// The force pass of one system (Arg = Sys) or a batch (BatchView).
template <typename Arg>
using Kern = void (*)(Arg);

Kern<Sys> force_kernel(int fp64, int ncv, int virial)
{
    if (ncv == 1) {
        if (fp64) return virial ? k_force_cn<double, true> : k_force_cn<double, false>;
        return virial ? k_force_cn<float, true> : k_force_cn<float, false>;
    }
    if (fp64) return virial ? k_force_pairs<true> : k_force_pairs<false>;
    return virial ? k_force_rows<true> : k_force_rows<false>;
}

int force_threads(int fp64, int ncv) { return ncv == 2 && !fp64 ? kRowThreads : kBlockAtoms; }

Kern<BatchView> batch_force_kernel(int fp64, int ncv, int virial)
{
    if (ncv == 1) {
        if (fp64) return virial ? kb_force_cn<double, true> : kb_force_cn<double, false>;
        return virial ? kb_force_cn<float, true> : kb_force_cn<float, false>;
    }
    if (fp64) return virial ? kb_force_pairs<true> : kb_force_pairs<false>;
    return virial ? kb_force_rows<true> : kb_force_rows<false>;
}

}  // namespace

void launch_forces(const Sys &s, int fp64, const ForceOut &out, cudaStream_t st)
{
    Sys t = s;
    out.set(t);
    chained_live(force_kernel(fp64, s.ncv, s.virial), grid_blocks(t, GK_FORCE, 0), force_threads(fp64, s.ncv), st, t);
}

void launch_force_gather(const Sys &s, int fp64, const ForceOut &out, cudaStream_t st)
{
    if (!pair_slots(s, fp64)) return;
    Sys t = s;
    out.set(t);
    chained_live(k_force_gather, group_grid(s.n), kBlockAtoms, st, t);
}

void launch_batch_cv(const BatchView &groups, int group_total, const BatchView &rows, int row_total, int fp64, int ncv,
                     int virial, cudaStream_t st)
{
    if (group_total <= 0) return;
    if (fp64) {
        chained_live(kb_cv_fwd<double>, group_total, kBlockAtoms, st, groups);
        if (ncv == 2) chained_live(kb_cv_avg<double>, row_total, kRowThreads, st, rows);
    } else if (ncv == 1) {
        chained_live(virial ? kb_cv_cn<true> : kb_cv_cn<false>, row_total, kBlockAtoms, st, rows);
    } else {
        chained_live(kb_cv_fwd<float>, row_total, kBlockAtoms, st, rows);
        chained_live(kb_cv_avg<float>, row_total, kRowThreads, st, rows);
    }
}

void launch_batch_sum(const BatchView &sums, int sum_total, int fp64, cudaStream_t st)
{
    if (sum_total <= 0) return;
    if (fp64)
        chained_live(kb_cv_sum<double>, sum_total, kSumThreads, st, sums);
    else
        chained_live(kb_cv_sum<float>, sum_total, kSumThreads, st, sums);
}

void launch_batch_adjoint(const BatchView &rows, int total, int fp64, cudaStream_t st)
{
    if (total <= 0) return;
    if (fp64)
        chained_live(kb_adjoint<double>, total, kRowThreads, st, rows);
    else
        chained_live(kb_adjoint<float>, total, kRowThreads, st, rows);
}

int launch_batch_forces(const BatchView &force, int force_total, const BatchView &groups, int group_total, int fp64,
                        int ncv, int virial, cudaStream_t st)
{
    if (force_total <= 0) return 0;
    chained_live(batch_force_kernel(fp64, ncv, virial), force_total, force_threads(fp64, ncv), st, force);
    if (!(fp64 && ncv == 2)) return 1;
    chained_live(kb_force_gather, group_total, kBlockAtoms, st, groups);
    return 2;
}

// The gather kernels without shared memory prefer the SM's unified storage
// as L1.  (It makes no difference to the force pass.)
void configure_kernels()
{
    const int l1 = cudaSharedmemCarveoutMaxL1;
    cudaFuncSetAttribute(k_cv_avg<float>, cudaFuncAttributePreferredSharedMemoryCarveout, l1);
    cudaFuncSetAttribute(kb_cv_avg<float>, cudaFuncAttributePreferredSharedMemoryCarveout, l1);
    cudaFuncSetAttribute(k_adjoint<float>, cudaFuncAttributePreferredSharedMemoryCarveout, l1);
    cudaFuncSetAttribute(kb_adjoint<float>, cudaFuncAttributePreferredSharedMemoryCarveout, l1);
    cudaGetLastError();
}

void launch_per_atom_out(const Sys &s, int fp64, double *out, cudaStream_t st)
{
    if (fp64)
        k_per_atom_out<double><<<(s.n + 255) / 256, 256, 0, st>>>(s, out);
    else
        k_per_atom_out<float><<<(s.n + 255) / 256, 256, 0, st>>>(s, out);
}

// Polynomial parts from the associated-Legendre recurrence on coefficient
// arrays (pole-free, unnormalised):
//   P_m^m = (2m-1)!!,  P_{m+1}^m = (2m+1) z P_m^m,
//   P_l^m = ((2l-1) z P_{l-1}^m - (l+m-1) P_{l-2}^m) / (l-m);
// every coefficient is a dyadic rational, exact in float32.
void set_ylm_constants(cudaStream_t st)
{
    YlmConst h{};
    const int l = 6;
    for (int m = 0; m <= l; ++m) {
        double prev2[8] = {0}, prev1[8] = {0}, cur[8] = {0};
        double dfact = 1.0;
        for (int k = 1; k <= 2 * m - 1; k += 2) dfact *= k;
        prev1[0] = dfact;
        if (m == l) {
            for (int p = 0; p < 8; ++p) cur[p] = prev1[p];
        } else {
            for (int p = 0; p < 7; ++p) cur[p + 1] = (2 * m + 1) * prev1[p];
            for (int ll = m + 2; ll <= l; ++ll) {
                for (int p = 0; p < 8; ++p) { prev2[p] = prev1[p]; prev1[p] = cur[p]; cur[p] = 0.0; }
                for (int p = 0; p < 7; ++p) cur[p + 1] += (2 * ll - 1) * prev1[p];
                for (int p = 0; p < 8; ++p) cur[p] -= (ll + m - 1) * prev2[p];
                for (int p = 0; p < 8; ++p) cur[p] /= (ll - m);
            }
        }
        const int deg = l - m;
        int t = 0;
        for (int p = deg; p >= 0; p -= 2, ++t) {
            h.pd[m][t] = cur[p];
            h.pf[m][t] = (float)cur[p];
        }
    }
    cudaMemcpyToSymbolAsync(c_ylm, &h, sizeof(h), 0, cudaMemcpyHostToDevice, st);
}


// The kernels of this file whose only argument is the system descriptor
// (a captured step's nodes of these can take new I/O buffers in place).
SysKernel sys_kernel_cv(const void *func)
{
    static const void *const io[] = {
        (const void *)k_force_rows<false>,
        (const void *)k_force_rows<true>,
        (const void *)k_force_cn<float, false>,
        (const void *)k_force_cn<float, true>,
        (const void *)k_force_cn<double, false>,
        (const void *)k_force_cn<double, true>,
        (const void *)k_force_gather,
    };
    static const void *const rest[] = {
        (const void *)k_cv_cn<false>,
        (const void *)k_cv_cn<true>,
        (const void *)k_cv_fwd<float, true>,
        (const void *)k_cv_fwd<float, false>,
        (const void *)k_cv_fwd<double, true>,
        (const void *)k_cv_fwd<double, false>,
        (const void *)k_cv_avg<float>,
        (const void *)k_cv_avg<double>,
        (const void *)k_cv_sum<float>,
        (const void *)k_cv_sum<double>,
        (const void *)k_adjoint<float>,
        (const void *)k_adjoint<double>,
        (const void *)k_force_pairs<false>,
        (const void *)k_force_pairs<true>,
    };
    for (const void *k : io)
        if (k == func) return kSysIo;
    for (const void *k : rest)
        if (k == func) return kSysOnly;
    return kNotSys;
}

}  // namespace metad
