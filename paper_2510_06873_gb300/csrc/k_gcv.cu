// Steps a4-a8 for the small-system CV families, which need no neighbour list:
//
//   torsion angles (the backbone Phi / Psi of the alanine-dipeptide runs,
//   Section "Alanine dipeptide torsion"), and
//   the distance from a reference atom to the nearest atom of a group (the
//   surface-oxygen to nearest-hydrogen CV of the rutile runs, Section "Water
//   dissociation on rutile (110) surface"), exact or as a soft minimum.
//
// Each system's CVs take one block (k_gcv_forward): its threads split the
// candidate group and reduce in a fixed tree, so the result does not depend
// on scheduling, and it leaves the gradient terms of every CV in s.gcv.
// The force pass (k_gcv_forces) gives one thread to each atom in the
// caller's order; it writes every atom (0 for atoms on no CV), adding the
// terms of each CV it belongs to in CV order: deterministic, no atomics.
// Positions are float32; bond and distance vectors are exact FP64
// differences.  The nearest-distance CV stays FP64 throughout (its nearest
// candidate is decided on the FP64 squared distance, as the definition);
// a torsion's angle and gradient run in FP32 (precision 0) or FP64
// (precision 1).  The file is compiled without multiply-add contraction, so
// squared distances round exactly as their plain definition.
#include <float.h>
#include <limits.h>

#include "hills.cuh"

namespace metad {

namespace {

constexpr int kGcvThreads = 256;

__device__ __forceinline__ double min_image(double d, double L)
{
    if (d > 0.5 * L)
        d -= L;
    else if (d < -0.5 * L)
        d += L;
    return d;
}

// Caller atom i, wrapped into the box; flags a non-finite input.
__device__ __forceinline__ void atom_posf(const Sys &s, int i, float p[3], bool &bad)
{
    const float4 q = s.pos_in[i];
    bad |= !(isfinite(q.x) && isfinite(q.y) && isfinite(q.z));
    p[0] = wrap_coord(isfinite(q.x) ? q.x : 0.0f, s.Lin[0], s.L[0]);
    p[1] = wrap_coord(isfinite(q.y) ? q.y : 0.0f, s.Lin[1], s.L[1]);
    p[2] = wrap_coord(isfinite(q.z) ? q.z : 0.0f, s.Lin[2], s.L[2]);
}

// The same in FP64.
__device__ __forceinline__ void atom_pos(const Sys &s, int i, double p[3], bool &bad)
{
    float f[3];
    atom_posf(s, i, f, bad);
#pragma unroll
    for (int k = 0; k < 3; ++k) p[k] = (double)f[k];
}

// One component of the minimum-image bond from pi to pj: the exact FP64
// difference rounded to `real`.  In FP32 a difference clear of half the box
// needs no image and is the float32 difference itself, so the usual bond
// takes no FP64 instruction (each holds a warp for 64 cycles here).
template <typename real>
__device__ __forceinline__ real bond_comp(const Sys &s, float pi, float pj, int k);
template <>
__device__ __forceinline__ double bond_comp<double>(const Sys &s, float pi, float pj, int k)
{
    return min_image((double)pj - (double)pi, s.L[k]);
}
template <>
__device__ __forceinline__ float bond_comp<float>(const Sys &s, float pi, float pj, int k)
{
    const float d = pj - pi;
    if (fabsf(d) < 0.999f * s.halfL[k]) return d;
    return (float)bond_comp<double>(s, pi, pj, k);
}

// Minimum-image displacement r_j - r_i.
__device__ __forceinline__ void disp(const Sys &s, const double pi[3], const double pj[3], double d[3])
{
#pragma unroll
    for (int k = 0; k < 3; ++k) d[k] = min_image(pj[k] - pi[k], s.L[k]);
}

template <typename real>
__device__ __forceinline__ real dot3(const real a[3], const real b[3])
{
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}

template <typename real>
__device__ __forceinline__ void cross3(const real a[3], const real b[3], real c[3])
{
    c[0] = a[1] * b[2] - a[2] * b[1];
    c[1] = a[2] * b[0] - a[0] * b[2];
    c[2] = a[0] * b[1] - a[1] * b[0];
}

__device__ __forceinline__ double sq_dist(const double d[3])
{
    const double xy = d[0] * d[0] + d[1] * d[1];
    return xy + d[2] * d[2];
}

__device__ __forceinline__ float real_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double real_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float real_atan2(float y, float x) { return atan2f(y, x); }
__device__ __forceinline__ double real_atan2(double y, double x) { return atan2(y, x); }

// Torsion d of the system: with bonds b1 = r_b - r_a, b2 = r_c - r_b,
// b3 = r_d - r_c, the angle is atan2(y, x) where
//   x = (b1 x b2) . (b2 x b3) = (b1.b2)(b2.b3) - (b1.b3)(b2.b2)
//   y = |b2| b1 . (b2 x b3),
// and its gradient follows from d(atan2) = (x dy - y dx) / (x^2 + y^2) with
//   dx/db1 = (b2.b3) b2 - (b2.b2) b3
//   dx/db2 = (b2.b3) b1 + (b1.b2) b3 - 2 (b1.b3) b2
//   dx/db3 = (b1.b2) b2 - (b2.b2) b1
//   dy/db1 = |b2| (b2 x b3),  dy/db3 = |b2| (b1 x b2),
//   dy/db2 = |b2| (b3 x b1) + (b1 . (b2 x b3)) b2 / |b2|.
// Collinear atoms (x = y = 0): angle 0, no gradient.  The bonds are exact
// FP64 differences of the float32 positions (minimum image); the rest runs
// in `real` (float: a dependent FP64 chain is long on this part, and the
// angle of float32 positions needs no more).
template <typename real>
__device__ void torsion(const Sys &s, int d, bool &bad, double *xo, double *go)
{
    const int *q = s.cv_atoms + 4 * d;
    float ra[3], rb[3], rc[3], rd[3];
    atom_posf(s, q[0], ra, bad);
    atom_posf(s, q[1], rb, bad);
    atom_posf(s, q[2], rc, bad);
    atom_posf(s, q[3], rd, bad);
    real b1[3], b2[3], b3[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        b1[k] = bond_comp<real>(s, ra[k], rb[k], k);
        b2[k] = bond_comp<real>(s, rb[k], rc[k], k);
        b3[k] = bond_comp<real>(s, rc[k], rd[k], k);
    }
    real n1[3], n2[3], n3[3];
    cross3(b1, b2, n1);
    cross3(b2, b3, n2);
    cross3(b3, b1, n3);
    const real m2 = dot3(b2, b2), m = real_sqrt(m2);
    const real x = dot3(n1, n2);
    const real T = dot3(b1, n2);
    const real y = m * T;
    const real D = x * x + y * y;
    double *g = go + 16 * d;
    if (D == (real)0 || m == (real)0) {
        xo[d] = 0.0;
        for (int k = 0; k < 12; ++k) g[k] = 0.0;
        return;
    }
    xo[d] = (double)real_atan2(y, x);
    const real b12 = dot3(b1, b2), b23 = dot3(b2, b3), b13 = dot3(b1, b3);
    const real invD = (real)1 / D, inv_m = (real)1 / m;
    const real cx = x * invD, cy = y * invD;  // dphi = cx dy - cy dx
    const real tm = T * inv_m;
    for (int k = 0; k < 3; ++k) {
        const real dx1 = b23 * b2[k] - m2 * b3[k];
        const real dx2 = b23 * b1[k] + b12 * b3[k] - (real)2 * b13 * b2[k];
        const real dx3 = b12 * b2[k] - m2 * b1[k];
        const real dy1 = m * n2[k];
        const real dy2 = m * n3[k] + tm * b2[k];
        const real dy3 = m * n1[k];
        const real p1 = cx * dy1 - cy * dx1;  // dphi/db1
        const real p2 = cx * dy2 - cy * dx2;
        const real p3 = cx * dy3 - cy * dx3;
        g[k] = (double)(-p1);           // r_a
        g[3 + k] = (double)(p1 - p2);   // r_b
        g[6 + k] = (double)(p2 - p3);   // r_c
        g[9 + k] = (double)p3;          // r_d
    }
}

// The smallest (v, arg) over the block's threads, ties to the lower arg, in
// every thread; v >= 0 or infinite, compared as integers (no FP64
// instruction).  Threads with nothing pass an infinite v.
__device__ __forceinline__ void block_argmin(double &v, int &arg)
{
    __shared__ long long shv[kGcvThreads / 32];
    __shared__ int sha[kGcvThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const long long none = 0x7ff0000000000000ll;  // infinity
    long long b = __double_as_longlong(v);
    if (__any_sync(0xffffffffu, b != none)) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const long long ob = __shfl_down_sync(0xffffffffu, b, o);
            const int oa = __shfl_down_sync(0xffffffffu, arg, o);
            if (ob < b || (ob == b && oa < arg)) { b = ob; arg = oa; }
        }
    }
    __syncthreads();  // an earlier call's results are read
    if (lane == 0) { shv[wid] = b; sha[wid] = arg; }
    __syncthreads();
    b = shv[0];
    arg = sha[0];
#pragma unroll
    for (int w = 1; w < kGcvThreads / 32; ++w)
        if (shv[w] < b || (shv[w] == b && sha[w] < arg)) { b = shv[w]; arg = sha[w]; }
    v = __longlong_as_double(b);
}

// The smallest v over the block's threads, v >= 0 (or infinite).
__device__ __forceinline__ float block_min(float v)
{
    __shared__ unsigned sh[kGcvThreads / 32];
    const unsigned m = __reduce_min_sync(0xffffffffu, __float_as_uint(v));
    __syncthreads();  // an earlier call's results are read
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
    __syncthreads();
    unsigned r = sh[0];
#pragma unroll
    for (int w = 1; w < kGcvThreads / 32; ++w) r = min(r, sh[w]);
    return __uint_as_float(r);
}

// Four sums at once; the totals land in thread 0 only.
__device__ __forceinline__ void block_sum4(double v[4], double (*sh)[kGcvThreads / 32])
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < 4; ++k) sh[k][wid] = v[k];
    __syncthreads();
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            double t = 0.0;
            for (int w = 0; w < kGcvThreads / 32; ++w) t += sh[k][w];
            v[k] = t;
        }
    __syncthreads();
}

// Soft-minimum weight numerator exp(-beta (r - r_min)) of one candidate;
// the forward and force passes share it, so they round alike.
__device__ __forceinline__ double soft_weight(const Sys &s, double r, double rmin)
{
    return exp(-s.sm_beta * (r - rmin));
}

// Squared distance of a candidate in FP32, within 2e-5 of the FP64 one
// relative and 1e-10 absolute: each component is one correctly rounded
// difference (across the box faces of exact ones, mi_axis).
__device__ __forceinline__ float sq_dist_f(const Sys &s, const float a[3], const float b[3])
{
    float r2 = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float d = mi_axis(b[k], a[k], s.halfL[k], s.Lhi[k], s.Llo[k]);
        r2 = fmaf(d, d, r2);
    }
    return r2;
}

// Nearest-distance CV d (all threads of the block): go[16 d] holds the
// nearest slot, r_min, the soft-minimum normaliser Z and d s/d r_ref.
//
// The nearest candidate is decided on FP64 squared distances, but only those
// whose FP32 estimate lies within the estimates' error of the smallest one
// are formed: FP64 takes 16 cycles a warp instruction on this part, about 30
// of them a candidate.
__device__ void nearest(const Sys &s, int d, bool &bad, double *xo, double *go)
{
    __shared__ double dsh[3];
    const int o = s.cv_atoms[d];
    const int *cand = s.cv_atoms + s.ncv;
    float pof[3];
    atom_posf(s, o, pof, bad);
    const double po[3] = {(double)pof[0], (double)pof[1], (double)pof[2]};
    float est = INFINITY;
    for (int m = threadIdx.x; m < s.n_cand; m += kGcvThreads) {
        float pj[3];
        atom_posf(s, cand[m], pj, bad);
        est = fminf(est, sq_dist_f(s, pof, pj));
    }
    const float lim = block_min(est) * (1.0f + 5e-5f) + 1e-9f;
    double best = INFINITY, dv[3] = {0.0, 0.0, 0.0};
    int arg = INT_MAX;
    if (est <= lim) {
        for (int m = threadIdx.x; m < s.n_cand; m += kGcvThreads) {
            float pf[3];
            atom_posf(s, cand[m], pf, bad);
            if (sq_dist_f(s, pof, pf) > lim) continue;
            const double pj[3] = {(double)pf[0], (double)pf[1], (double)pf[2]};
            double t[3];
            disp(s, po, pj, t);
            const double r2 = sq_dist(t);
            if (r2 < best) {
                best = r2;
                arg = m;
                for (int k = 0; k < 3; ++k) dv[k] = t[k];
            }
        }
    }
    const int mine = arg;
    block_argmin(best, arg);
    const double rmin = sqrt(best);
    double *g = go + 16 * d;
    if (s.sm_beta <= 0.0) {
        if (mine == arg)  // one thread: a candidate belongs to one
            for (int k = 0; k < 3; ++k) dsh[k] = dv[k];
        __syncthreads();
        if (threadIdx.x < 3) g[3 + threadIdx.x] = rmin > 0.0 ? -dsh[threadIdx.x] / rmin : 0.0;
        if (threadIdx.x == 0) {
            xo[d] = rmin;
            g[0] = (double)arg;
            g[1] = rmin;
            g[2] = 1.0;
        }
        __syncthreads();  // dsh is read before the next CV's
        return;
    }
    __shared__ double sh4[4][kGcvThreads / 32];
    double acc[4] = {0.0, 0.0, 0.0, 0.0};  // Z and sum_j e_j u_j
    for (int m = threadIdx.x; m < s.n_cand; m += kGcvThreads) {
        double pj[3], dv[3];
        atom_pos(s, cand[m], pj, bad);
        disp(s, po, pj, dv);
        const double r = sqrt(sq_dist(dv));
        const double e = soft_weight(s, r, rmin);
        acc[0] += e;
        if (r > 0.0) {
            acc[1] += e * (dv[0] / r);
            acc[2] += e * (dv[1] / r);
            acc[3] += e * (dv[2] / r);
        }
    }
    block_sum4(acc, sh4);
    if (threadIdx.x == 0) {
        const double Z = acc[0];
        xo[d] = rmin - log(Z) / s.sm_beta;
        g[0] = (double)arg;
        g[1] = rmin;
        g[2] = Z;
        g[3] = -acc[1] / Z;
        g[4] = -acc[2] / Z;
        g[5] = -acc[3] / Z;
    }
}

// The CVs into xo[d] and their gradient terms into go[16 d ...] (shared or
// global memory).
template <typename real>
__device__ void gcv_eval(const Sys &s, double *xo, double *go)
{
    bool bad = false;
    if (s.kind == kKindTorsion) {
        if (threadIdx.x < s.ncv) torsion<real>(s, threadIdx.x, bad, xo, go);
    } else {
        for (int d = 0; d < s.ncv; ++d) nearest(s, d, bad, xo, go);
    }
    if (bad) atomicOr(s.err, kErrNonFinite);
}

template <typename real>
__device__ void gcv_forward(const Sys &s)
{
    gcv_eval<real>(s, s.scal + kS0, s.gcv);
    if (threadIdx.x == 0 && s.ncv == 1) s.scal[kS1] = 0.0;
}

// F_i = (accumulate ? F_i : 0) - scale sum_d dV/ds_d ds_d/dr_i, with the
// gradient terms gterms of the CV pass.
__device__ __forceinline__ void gcv_force(const Sys &s, int i, const double *gterms)
{
        const int *cand = s.cv_atoms + s.ncv;
        double f[3] = {0.0, 0.0, 0.0};
        for (int d = 0; d < s.ncv; ++d) {
            const double dv = s.scal[kDV0 + d];
            const double *g = gterms + 16 * d;
            if (s.kind == kKindTorsion) {
                // an atom sits in a quadruplet at most once: find its place,
                // then one set of FP64 terms for the whole warp
                int at = -1;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (s.cv_atoms[4 * d + q] == i) at = q;
                if (at >= 0)
                    for (int k = 0; k < 3; ++k) f[k] -= dv * g[3 * at + k];
                continue;
            }
            if (s.cv_atoms[d] == i)
                for (int k = 0; k < 3; ++k) f[k] -= dv * g[3 + k];
            const int m = s.cand_slot[i];
            if (m < 0) continue;
            const bool exact = s.sm_beta <= 0.0;
            if (exact && m != (int)g[0]) continue;
            bool bad = false;
            double po[3], pj[3], dd[3];
            atom_pos(s, s.cv_atoms[d], po, bad);
            atom_pos(s, cand[m], pj, bad);
            disp(s, po, pj, dd);
            const double r = sqrt(sq_dist(dd));
            if (!(r > 0.0)) continue;
            const double w = exact ? 1.0 : soft_weight(s, r, g[1]) / g[2];
            for (int k = 0; k < 3; ++k) f[k] -= dv * (w * (dd[k] / r));
        }
        float *out = s.F_out + (size_t)s.F_stride * i;
        if (s.F_stride == 4) out[3] = 0.0f;
        const double scale = force_scale(s);
        for (int k = 0; k < 3; ++k) {
            const float v = (float)(scale * f[k]);
            out[k] = s.accumulate ? out[k] + v : v;
        }
}

__device__ void gcv_forces(const Sys &s, Blk blk, const double *gterms)
{
    for (int i = blk.b * kGcvThreads + threadIdx.x; i < s.n; i += blk.nb * kGcvThreads) gcv_force(s, i, gterms);
}

// Whether atom i can have a force with these gradient terms (an atom of a
// torsion; a reference; the nearest candidate, or any with the soft minimum).
__device__ __forceinline__ bool gcv_moves(const Sys &s, int i, const double *gterms)
{
    bool in = false;
    if (s.kind == kKindTorsion) {
        for (int q = 0; q < 4 * s.ncv; ++q) in |= s.cv_atoms[q] == i;
        return in;
    }
    const int m = s.cand_slot[i];
    for (int d = 0; d < s.ncv; ++d)
        in |= s.cv_atoms[d] == i || (m >= 0 && (s.sm_beta > 0.0 || m == (int)gterms[16 * d]));
    return in;
}

template <typename real>
__global__ void __launch_bounds__(kGcvThreads) k_gcv_forward(Sys s) { gcv_forward<real>(s); }

__global__ void __launch_bounds__(kGcvThreads) k_gcv_forces(Sys s) { gcv_forces(s, own_blk(), s.gcv); }

// The whole step in one launch (systems of up to kFuseAtoms atoms): every
// block evaluates the CVs (a few atoms, or one pass over the candidates)
// into shared memory and sums its share of the hills there; block 0
// publishes the CVs; the last block to finish the hill sum (which also
// deposits, if asked) writes the forces from its own copy of the CV gradient
// terms.  Atoms that no gradient term reaches get their zero (or, when
// accumulating, nothing) before the hill sum, from all blocks, off the chain
// that a lone step waits for.  The same arithmetic as the three-kernel path,
// so the same bits.
template <typename real>
__device__ void gcv_step(const Sys &s, Blk blk)
{
    __shared__ double xs[kMaxCv];
    __shared__ double gs[16 * 2];
    if (threadIdx.x < kMaxCv) xs[threadIdx.x] = 0.0;
    if (threadIdx.x < 16 * 2) gs[threadIdx.x] = 0.0;
    __syncthreads();
    gcv_eval<real>(s, xs, gs);
    __syncthreads();
    if (blk.b == 0) {
        if (threadIdx.x < kMaxCv) s.scal[kS0 + threadIdx.x] = xs[threadIdx.x];
        if (threadIdx.x < 16 * s.ncv) s.gcv[threadIdx.x] = gs[threadIdx.x];
    }
    if (!s.accumulate)
        for (int i = blk.b * kGcvThreads + threadIdx.x; i < s.n; i += blk.nb * kGcvThreads)
            if (!gcv_moves(s, i, gs))
                for (int k = 0; k < 3; ++k) s.F_out[3 * (size_t)i + k] = 0.0f;
    if (!hill_sum<2>(s, blk, xs, s.scal + kV, s.deposit)) return;
    __syncthreads();  // thread 0 of this block wrote dV/ds
    // the atoms that move: each of the few, or the soft minimum's candidates
    const int *list = s.cv_atoms;
    const bool exact = s.kind == kKindNearest && s.sm_beta <= 0.0;
    const int refs = s.kind == kKindTorsion ? 4 * s.ncv : s.ncv;
    const int count = refs + (s.kind == kKindTorsion ? 0 : (exact ? s.ncv : s.n_cand));
    for (int q = threadIdx.x; q < count; q += kGcvThreads) {
        const int at = q >= refs && exact ? s.ncv + (int)gs[16 * (q - refs)] : q;
        const int i = list[at];
        bool first = true;  // an atom may serve both CVs
        for (int p = 0; p < min(q, 8); ++p) {
            const int pt = p >= refs && exact ? s.ncv + (int)gs[16 * (p - refs)] : p;
            first = first && (p >= refs && !exact ? true : list[pt] != i);
        }
        if (first) gcv_force(s, i, gs);
    }
}

template <typename real>
__global__ void __launch_bounds__(kGcvThreads) k_gcv_step(Sys s)
{
    chain_enter();
    gcv_step<real>(s, own_blk());
}

template <typename real>
__global__ void __launch_bounds__(kGcvThreads, 4) kb_gcv_step(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    gcv_step<real>(s, k);
}

template <typename real>
__global__ void __launch_bounds__(kGcvThreads) kb_gcv_forward(BatchView v)
{
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    gcv_forward<real>(s);
}

__global__ void __launch_bounds__(kGcvThreads) kb_gcv_forces(BatchView v)
{
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    gcv_forces(s, k, s.gcv);
}

}  // namespace

void launch_gcv_forward(const Sys &s, int fp64, cudaStream_t st)
{
    if (fp64)
        k_gcv_forward<double><<<1, kGcvThreads, 0, st>>>(s);
    else
        k_gcv_forward<float><<<1, kGcvThreads, 0, st>>>(s);
}

void launch_gcv_forces(const Sys &s, const ForceOut &out, cudaStream_t st)
{
    Sys t = s;
    out.set(t);
    k_gcv_forces<<<grid_blocks(t, GK_ATOM256, 0), kGcvThreads, 0, st>>>(t);
}

void launch_batch_gcv(const BatchView &one, int one_total, int fp64, cudaStream_t st)
{
    if (one_total <= 0) return;
    if (fp64)
        kb_gcv_forward<double><<<one_total, kGcvThreads, 0, st>>>(one);
    else
        kb_gcv_forward<float><<<one_total, kGcvThreads, 0, st>>>(one);
}

void launch_batch_gcv_forces(const BatchView &atoms, int atom_total, cudaStream_t st)
{
    if (atom_total > 0) kb_gcv_forces<<<atom_total, kGcvThreads, 0, st>>>(atoms);
}

void launch_gcv_step(const Sys &s, int K, float *F, int accumulate, int deposit, int fp64, cudaStream_t st)
{
    Sys t = s;
    t.K = K;
    t.F_out = F;
    t.accumulate = accumulate;
    t.fscale = 1.0;
    t.deposit = deposit;
    const int nb = bias_blocks(K);
    if (fp64)
        chained_live(k_gcv_step<double>, nb, kGcvThreads, st, t);
    else
        chained_live(k_gcv_step<float>, nb, kGcvThreads, st, t);
}

void launch_batch_gcv_step(const BatchView &hills, int hill_total, int fp64, cudaStream_t st)
{
    if (hill_total <= 0) return;
    if (fp64)
        chained_live(kb_gcv_step<double>, hill_total, kGcvThreads, st, hills);
    else
        chained_live(kb_gcv_step<float>, hill_total, kGcvThreads, st, hills);
}


// The kernels of this file whose only argument is the system descriptor
// (a captured step's nodes of these can take new I/O buffers in place).
SysKernel sys_kernel_gcv(const void *func)
{
    static const void *const io[] = {
        (const void *)k_gcv_forward<float>,
        (const void *)k_gcv_forward<double>,
        (const void *)k_gcv_forces,
        (const void *)k_gcv_step<float>,
        (const void *)k_gcv_step<double>,
    };
    for (const void *k : io)
        if (k == func) return kSysIo;
    return kNotSys;
}

}  // namespace metad
