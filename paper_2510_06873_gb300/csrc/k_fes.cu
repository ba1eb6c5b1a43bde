// Free-energy surface from a context's bias (an analysis pass, not per step).
//
// The methods section recovers the FES by reweighting the biased ensemble,
// P_unbias(s) = <delta(s - s(R)) exp(beta V)> / <exp(beta V)> and
// F = -(1/beta) log P (Eqs. 4-5); for a well-tempered bias the deposited
// bias itself estimates it, F = -(gamma / (gamma - 1)) V + const.  Both are
// computed here in FP64 with fixed summation orders.
#include "exp2.cuh"
#include "metad_impl.cuh"

namespace metad {

namespace {

constexpr int kFesThreads = 256;

__device__ __forceinline__ double fes_block_sum(double v, double *sh)
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

struct FesGrid {
    double lo[2], hi[2];
    int n[2];
};

// Sums of two-CV hills over a regular grid as a contraction.  A Gaussian hill
// is a product of one factor per axis, so
//   V[a][b] = sum_k (w_k X_k(x_a)) Y_k(y_b),  X_k(x) = exp(-(x - c_k0)^2 / 2 s0^2)
// needs K (n0 + n1) exponentials and one FP64 multiply-add per point and
// hill, where evaluating each hill at each point takes an exponential (about
// 30 FP64 instructions) there; the grid's node derivatives are the same sums
// with the factors' own derivatives.  Bound by the FP64 pipe (two lanes per
// clock and SM).  Two passes: the axis factors of a chunk of hills into a
// table (points x hills), then one thread per point and a 16 x 16 tile per
// block, staged 32 hills at a time in shared memory.  The hills are split
// over enough blocks (slices) to fill the GPU, each slice's sums to its own
// partial array, added in slice order afterwards: a fixed order.
// Measured: sum-of-hills surface of 101 x 96 bins and 5,000 hills
// 3,508 -> 155 us; fold of 20,000 hills into 200 x 200 nodes 145.6 -> 7.0 ms.
struct Axis {
    double lo, step, off;  // point i: lo + (i + off) step
    int n;
};

constexpr int kSepTile = 16;
constexpr int kSepK = 32;

// Tables of the hills [k0, k0 + kn): row i < n0 holds w_k X_k of axis-0 point
// i, row n0 + j the Y_k of axis-1 point j.  kDeriv: a second table, rows
// offset by n0 + n1, of the factors' derivatives.
template <bool kDeriv>
__global__ void __launch_bounds__(kFesThreads) k_axis_factors(Sys s, int k0, int kn, int ld, Axis ax0, Axis ax1, double *tab)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= kn) return;
    for (int row = blockIdx.y; row < ax0.n + ax1.n; row += gridDim.y) {
        const int d = row < ax0.n ? 0 : 1, i = d == 0 ? row : row - ax0.n;
        const double x = d == 0 ? ax0.lo + (i + ax0.off) * ax0.step : ax1.lo + (i + ax1.off) * ax1.step;
        const double dx = hill_diff(s, d, x - s.hc[(size_t)s.hstride * (k0 + k) + d]);
        double g = exp2_neg(dx * dx * s.k2v[d]);
        if (d == 0) g *= s.hw[k0 + k];
        tab[(size_t)row * ld + k] = g;
        if (kDeriv) tab[(size_t)(ax0.n + ax1.n + row) * ld + k] = -g * dx * (2.0 * s.inv2v[d]);
    }
}

// t + v with the rounding error gathered in c (Knuth's TwoSum).
__device__ __forceinline__ void add_exact(double &t, double &c, double v)
{
    const double n = t + v, b = n - t;
    c += (t - (n - b)) + (v - b);
    t = n;
}

// Slice z of the chunk's hills: part[z][point][kOut] (+)= the tile's sums.
// A stage's 32 products are summed on their own, then added to the slice's
// sum: a slice's hundreds of products in one chain gather several roundings of
// the whole sum (up to 8e-16 of the surface, where one sum per thread and a
// tree over the threads left 3e-16).
// kOut 1: V; 4: V, dV/dx0, dV/dx1, d2V/dx0dx1.
template <int kOut>
__global__ void __launch_bounds__(kSepTile * kSepTile)
    k_axis_contract(const double *tab, int kn, int ld, int per, int n0, int n1, int first, double *part)
{
    constexpr int kT = kOut == 4 ? 2 : 1;
    __shared__ double A[kT][kSepTile][kSepK + 1], B[kT][kSepTile][kSepK + 1];
    const int tx = threadIdx.x % kSepTile, ty = threadIdx.x / kSepTile;
    const int tiles1 = (n1 + kSepTile - 1) / kSepTile;
    const int a0 = (blockIdx.x / tiles1) * kSepTile, b0 = (blockIdx.x % tiles1) * kSepTile;
    const int k_lo = blockIdx.y * per, k_hi = min(kn, k_lo + per);
    double acc[kOut] = {};
    for (int kb = k_lo; kb < k_hi; kb += kSepK) {
#pragma unroll
        for (int t = 0; t < kT; ++t) {
            const double *tt = tab + (size_t)t * (n0 + n1) * ld;
            for (int e = threadIdx.x; e < kSepTile * kSepK; e += kSepTile * kSepTile) {
                const int r = e / kSepK, c = e % kSepK;
                const bool in = kb + c < k_hi;
                A[t][r][c] = in && a0 + r < n0 ? tt[(size_t)(a0 + r) * ld + kb + c] : 0.0;
                B[t][r][c] = in && b0 + r < n1 ? tt[(size_t)(n0 + b0 + r) * ld + kb + c] : 0.0;
            }
        }
        __syncthreads();
        double sub[kOut] = {};
#pragma unroll 8
        for (int c = 0; c < kSepK; ++c) {
            sub[0] = fma(A[0][ty][c], B[0][tx][c], sub[0]);
            if (kOut == 4) {
                sub[kOut - 3] = fma(A[kT - 1][ty][c], B[0][tx][c], sub[kOut - 3]);
                sub[kOut - 2] = fma(A[0][ty][c], B[kT - 1][tx][c], sub[kOut - 2]);
                sub[kOut - 1] = fma(A[kT - 1][ty][c], B[kT - 1][tx][c], sub[kOut - 1]);
            }
        }
#pragma unroll
        for (int o = 0; o < kOut; ++o) acc[o] += sub[o];
        __syncthreads();
    }
    if (a0 + ty >= n0 || b0 + tx >= n1) return;
    double *p = part + ((size_t)blockIdx.y * n0 * n1 + (size_t)(a0 + ty) * n1 + (b0 + tx)) * kOut;
#pragma unroll
    for (int o = 0; o < kOut; ++o) p[o] = (first ? 0.0 : p[o]) + acc[o];
}

// Fold: grid node values += the slices' sums, in slice order.
__global__ void k_fold_add(double *grid, const double *part, int values, int slices)
{
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= values) return;
    double t = 0.0, c = 0.0;
    for (int z = 0; z < slices; ++z) add_exact(t, c, part[(size_t)z * values + v]);
    grid[v] += t + c;
}

// Block-wide minimum and sum in a fixed order, in every thread.
__device__ __forceinline__ double fes_block_min(double v, double *sh)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    v = sh[lane & (kFesThreads / 32 - 1)];
#pragma unroll
    for (int o = kFesThreads / 64; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    return v;
}

// Grids of the passes over the bins: at most kFesBlocks blocks, so that
// every block can reduce all the blocks' partials again by itself.
constexpr int kFesBlocks = 304;

// V = the slices' sums (+ the grid patch) with slices > 0, else V as given;
// F = -fac V, and each block's minimum of it.
__global__ void __launch_bounds__(kFesThreads)
    k_fes_value(Sys s, FesGrid g, const double *part, int slices, int M, double fac, const double *V, double *F, double *bmin)
{
    __shared__ double sh[kFesThreads / 32];
    double lo = INFINITY;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < M; b += gridDim.x * blockDim.x) {
        double v = 0.0;
        if (slices > 0) {
            double c = 0.0;
            for (int z = 0; z < slices; ++z) add_exact(v, c, part[(size_t)z * M + b]);
            v += c;
            const int i0 = b / g.n[1], i1 = b % g.n[1];
            double gv, g0, g1;
            grid_value(s, g.lo[0] + (i0 + 0.5) * ((g.hi[0] - g.lo[0]) / g.n[0]),
                       g.lo[1] + (i1 + 0.5) * ((g.hi[1] - g.lo[1]) / g.n[1]), gv, g0, g1);
            v += gv;
        } else {
            v = V[b];
        }
        const double f = -fac * v;
        F[b] = f;
        lo = fmin(lo, f);
    }
    lo = fes_block_min(lo, sh);
    if (threadIdx.x == 0) bmin[blockIdx.x] = lo;
}

// F -= min F (finite entries only when keep_inf: empty bins stay +inf).
__global__ void __launch_bounds__(kFesThreads) k_fes_shift(double *F, int M, const double *bmin, int blocks, int keep_inf)
{
    __shared__ double sh[kFesThreads / 32];
    double m = INFINITY;
    for (int b = threadIdx.x; b < blocks; b += blockDim.x) m = fmin(m, bmin[b]);
    m = fes_block_min(m, sh);
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < M; b += gridDim.x * blockDim.x)
        if (!keep_inf || F[b] < INFINITY) F[b] -= m;
}

// One CV, or an axis too short for the contraction: V at grid point b, the
// centre of bin b (one block per point): thread t
// sums hills t, t + blockDim, ... in order, then a fixed tree, then the grid
// patch (as the hill kernel).
__global__ void __launch_bounds__(kFesThreads) k_fes_points(Sys s, int K, FesGrid g, int M, double *V)
{
    __shared__ double sh[kFesThreads / 32];
    const int b = blockIdx.x;
    if (b >= M) return;
    const int i0 = s.ncv == 2 ? b / g.n[1] : b, i1 = s.ncv == 2 ? b % g.n[1] : 0;
    const double x0 = g.lo[0] + (i0 + 0.5) * ((g.hi[0] - g.lo[0]) / g.n[0]);
    const double x1 = s.ncv == 2 ? g.lo[1] + (i1 + 0.5) * ((g.hi[1] - g.lo[1]) / g.n[1]) : 0.0;
    double acc = 0.0;
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        const double d0 = hill_diff(s, 0, x0 - s.hc[(size_t)s.hstride * k]);
        double y = d0 * d0 * s.k2v[0];
        if (s.ncv == 2) {
            const double d1 = hill_diff(s, 1, x1 - s.hc[(size_t)s.hstride * k + 1]);
            y += d1 * d1 * s.k2v[1];
        }
        acc += s.hw[k] * exp2_neg(y);
    }
    acc = fes_block_sum(acc, sh);
    if (threadIdx.x == 0) {
        if (s.ncv == 2) {
            double gv, g0, g1;
            grid_value(s, x0, x1, gv, g0, g1);
            acc += gv;
        }
        V[b] = acc;
    }
}

// Bin of a CV point on the regular grid [lo, hi), the first CV slowest; -1
// when outside.  h: the bin widths.
__device__ __forceinline__ int fes_bin(const double *x, int ncv, const FesGrid &g, const double *h)
{
    int idx = 0;
    for (int d = 0; d < ncv; ++d) {
        if (!(x[d] >= g.lo[d] && x[d] < g.hi[d])) return -1;
        const int b = (int)floor((x[d] - g.lo[d]) / h[d]);
        if (b >= g.n[d]) return -1;
        idx = idx * g.n[d] + b;
    }
    return idx;
}

// Each block's maximum of V_t (kFesThreads threads).
__global__ void __launch_bounds__(kFesThreads) k_fes_vmax(const double *V, long long T, double *bmax)
{
    __shared__ double sh[kFesThreads / 32];
    double m = INFINITY;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < T; t += (long long)gridDim.x * blockDim.x)
        m = fmin(m, -V[t]);
    m = fes_block_min(m, sh);
    if (threadIdx.x == 0) bmax[blockIdx.x] = -m;
}

// Weight sums per bin, exp(beta (V_t - max V)), every sum in a fixed order.
// Walking all samples for every bin costs bins x samples bin computations
// (FP64 divides); here each sample is binned once.  The samples are cut into
// chunks of `per` in time order, one warp and one row of bins per chunk, and
// the rows are added by k_fes_bin_sum, in an order that follows from their
// number.  A warp takes 32 samples at a time: the lanes of one bin are found by
// a match vote, their lowest lane adds their weights in lane order and adds the
// sum to the chunk's row.  A lone read-modify-write chain per 32 samples is
// what bounds it; chunks are short (64 samples) as long as the rows fit 64 MB
// (rw_per).  Measured (9,696 bins, 20,001 samples): 33,600 -> 14 us.  Fine
// grids leave few chunks, one warp each, and the pass turns serial: a million
// samples 0.15 ms at 9,696 bins, 14 at 1M (eight chunks), 95 at 2^24 (one).
__global__ void __launch_bounds__(kFesThreads)
    k_fes_accum(const double *S, const double *V, long long T, int ncv, FesGrid g, double beta, const double *bmax,
                int vblocks, long long per, int chunks, int nbins, double *rows)
{
    __shared__ double sh[kFesThreads / 32];
    __shared__ double w_sh[kFesThreads];
    double m = INFINITY;
    for (int b = threadIdx.x; b < vblocks; b += blockDim.x) m = fmin(m, -bmax[b]);
    m = -fes_block_min(m, sh);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * (kFesThreads / 32) + warp;
    if (c >= chunks) return;  // warp-uniform, no block barrier below
    double h[2] = {(g.hi[0] - g.lo[0]) / g.n[0], ncv == 2 ? (g.hi[1] - g.lo[1]) / g.n[1] : 1.0};
    double *row = rows + (size_t)c * nbins, *wv = w_sh + 32 * warp;
    const long long t1 = min(T, (c + 1) * per);
    for (long long t0 = c * per; t0 < t1; t0 += 32) {
        const long long t = t0 + lane;
        int bin = -1;
        double w = 0.0;
        if (t < t1) {
            const double x[2] = {S[(size_t)ncv * t], ncv == 2 ? S[(size_t)ncv * t + 1] : 0.0};
            bin = fes_bin(x, ncv, g, h);
            if (bin >= 0) w = exp(beta * (V[t] - m));
        }
        wv[lane] = w;
        __syncwarp();
        const unsigned same = __match_any_sync(0xffffffffu, bin);
        if (bin >= 0 && lane == __ffs(same) - 1) {
            double a = row[bin];
            for (unsigned r = same; r; r &= r - 1) a += wv[__ffs(r) - 1];
            row[bin] = a;
        }
        __syncwarp();
    }
}

// Bin sums over the chunks' rows, and each block's total of them.  A block
// takes 32 bins at a time: its warp g adds rows g, g + 8, ... in order (32
// neighbouring bins a load, four loads in flight), then warp 0 adds the eight
// sums in order.  (One thread walking all the rows of a bin: 139 us for 313 rows of
// 9,696 bins.)
__global__ void __launch_bounds__(kFesThreads) k_fes_bin_sum(const double *rows, int chunks, int nbins, double *acc, double *btot)
{
    constexpr int kGroups = kFesThreads / 32;
    __shared__ double part[kGroups][32];
    const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
    double t = 0.0;
    for (int b0 = blockIdx.x * 32; b0 < nbins; b0 += gridDim.x * 32) {
        const int b = b0 + lane;
        double a = 0.0;
        if (b < nbins) {
#pragma unroll 4
            for (int c = grp; c < chunks; c += kGroups) a += rows[(size_t)c * nbins + b];
        }
        part[grp][lane] = a;
        __syncthreads();
        if (grp == 0 && b < nbins) {
            double v = part[0][lane];
            for (int g = 1; g < kGroups; ++g) v += part[g][lane];
            acc[b] = v;
            t += v;
        }
        __syncthreads();
    }
    if (grp == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if (lane == 0) btot[blockIdx.x] = t;
    }
}

// P_b = acc_b / sum acc, F_b = -(1/beta) log P_b (empty bins +inf), and each
// block's minimum; the shift to minimum 0 follows (k_fes_shift).
__global__ void __launch_bounds__(kFesThreads)
    k_fes_log(const double *acc, int nbins, double beta, const double *btot, int blocks, double *F, double *bmin)
{
    __shared__ double sh[kFesThreads / 32];
    __shared__ double tot_s;
    double t = 0.0;
    for (int b = threadIdx.x; b < blocks; b += blockDim.x) t += btot[b];
    t = fes_block_sum(t, sh);
    if (threadIdx.x == 0) tot_s = t;
    __syncthreads();
    const double tot = tot_s;
    double m = INFINITY;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nbins; b += gridDim.x * blockDim.x) {
        const double f = acc[b] > 0.0 ? -log(acc[b] / tot) / beta : INFINITY;
        F[b] = f;
        m = fmin(m, f);
    }
    m = fes_block_min(m, sh);
    if (threadIdx.x == 0) bmin[blockIdx.x] = m;
}

int fes_blocks(long long items)
{
    const long long b = (items + kFesThreads - 1) / kFesThreads;
    return b < 1 ? 1 : (b > kFesBlocks ? kFesBlocks : (int)b);
}

// Shape of the contraction for K hills on n0 x n1 points: the table's hills
// per pass and the slices.
struct SepPlan {
    int chunk, slices, per, ld;
    size_t tab, part;  // doubles
    size_t most;       // of both together, for any number of hills up to K
};

SepPlan sep_plan(int K, int n0, int n1, int out)
{
    SepPlan p;
    const long long rows = (long long)(n0 + n1) * (out == 4 ? 2 : 1);
    // the table stays near 32 MB (it then lives in L2); a fold's near 8 MB, as
    // every context with a grid holds one (20,000 hills into 200 x 200 nodes
    // 7.00 ms, with 32 MB 6.89)
    long long chunk = (out == 4 ? 1LL << 20 : 4LL << 20) / rows / kSepK * kSepK;
    if (chunk < kSepK) chunk = kSepK;
    if (chunk > K) chunk = K;
    p.chunk = (int)chunk;
    p.ld = (p.chunk + kSepK - 1) / kSepK * kSepK;
    const long long tiles = (long long)((n0 + kSepTile - 1) / kSepTile) * ((n1 + kSepTile - 1) / kSepTile);
    // two resident sets of blocks over the SMs, at least 64 hills a slice
    long long sl = (4 * 152 + tiles - 1) / tiles;
    const long long most = (p.chunk + 63) / 64;
    if (sl > most) sl = most;
    if (sl < 1) sl = 1;
    p.per = (int)(((p.chunk + sl - 1) / sl + kSepK - 1) / kSepK * kSepK);
    p.slices = (p.chunk + p.per - 1) / p.per;
    p.tab = (size_t)rows * p.ld;
    p.part = (size_t)p.slices * n0 * n1 * out;
    p.most = p.tab + (size_t)sl * n0 * n1 * out;  // table and sl grow with the chunk, and slices <= sl
    return p;
}

// The contraction of K hills into p.slices partial arrays.
template <int kOut>
void contract(const Sys &s, int K, const SepPlan &p, const Axis &a0, const Axis &a1, double *tab, double *part,
              cudaStream_t st)
{
    const int rows = a0.n + a1.n;
    const int tiles = ((a0.n + kSepTile - 1) / kSepTile) * ((a1.n + kSepTile - 1) / kSepTile);
    for (int k0 = 0; k0 < K; k0 += p.chunk) {
        const int kn = K - k0 < p.chunk ? K - k0 : p.chunk;
        const dim3 g((kn + kFesThreads - 1) / kFesThreads, rows < 65535 ? rows : 65535);
        k_axis_factors<kOut == 4><<<g, kFesThreads, 0, st>>>(s, k0, kn, p.ld, a0, a1, tab);
        k_axis_contract<kOut><<<dim3(tiles, p.slices), kSepTile * kSepTile, 0, st>>>(tab, kn, p.ld, p.per, a0.n, a1.n,
                                                                                   k0 == 0 ? 1 : 0, part);
    }
}

}  // namespace

// Two CVs, and the axes short beside the grid (a table entry costs about as
// much as 25 multiply-adds): 8 points along each axis or more.
bool fes_separable(const Sys &s, int K, const int *n) { return s.ncv == 2 && K > 0 && n[0] >= 8 && n[1] >= 8; }

size_t fes_points_doubles(const Sys &s, int K, const int *n, bool separable)
{
    const size_t M = (size_t)n[0] * (s.ncv == 2 ? n[1] : 1);
    const size_t base = M + kFesBlocks;  // F and the blocks' minima
    if (!separable) return base + M;     // V
    const SepPlan p = sep_plan(K, n[0], n[1], 1);
    return base + p.tab + p.part;
}

int launch_fes_points(const Sys &s, int K, const double *lo, const double *hi, const int *n, double *scratch,
                      bool separable, double fac, cudaStream_t st)
{
    FesGrid g{};
    int M = 1;
    for (int d = 0; d < s.ncv; ++d) {
        g.lo[d] = lo[d];
        g.hi[d] = hi[d];
        g.n[d] = n[d];
        M *= n[d];
    }
    double *F = scratch, *bmin = F + M, *work = bmin + kFesBlocks;
    const int nb = fes_blocks(M);
    int launched = 2;
    if (separable) {
        const SepPlan p = sep_plan(K, n[0], n[1], 1);
        const Axis a0{lo[0], (hi[0] - lo[0]) / n[0], 0.5, n[0]}, a1{lo[1], (hi[1] - lo[1]) / n[1], 0.5, n[1]};
        contract<1>(s, K, p, a0, a1, work, work + p.tab, st);
        k_fes_value<<<nb, kFesThreads, 0, st>>>(s, g, work + p.tab, p.slices, M, fac, nullptr, F, bmin);
        launched += 2 * ((K + p.chunk - 1) / p.chunk);
    } else {
        k_fes_points<<<M, kFesThreads, 0, st>>>(s, K, g, M, work);
        k_fes_value<<<nb, kFesThreads, 0, st>>>(s, g, nullptr, 0, M, fac, work, F, bmin);
        launched += 1;
    }
    k_fes_shift<<<nb, kFesThreads, 0, st>>>(F, M, bmin, nb, 0);
    return launched;
}

// A grid whose workspace would pass 256 MB (from about 8M nodes, or 500,000
// along both axes together) is folded node by node instead (k_grid_fold).  By
// the grid and the capacity alone, so that a context always sums alike.
size_t fold_doubles(const Sys &s)
{
    if (!s.grid_on) return 0;
    const size_t most = sep_plan(s.hill_cap, s.gn[0], s.gn[1], 4).most;
    return most * sizeof(double) <= (256u << 20) ? most : 0;
}

int launch_fold_separable(const Sys &s, int K, double *work, cudaStream_t st)
{
    const SepPlan p = sep_plan(K, s.gn[0], s.gn[1], 4);
    const Axis a0{s.glo[0], s.gh[0], 0.0, s.gn[0]}, a1{s.glo[1], s.gh[1], 0.0, s.gn[1]};
    contract<4>(s, K, p, a0, a1, work, work + p.tab, st);
    const int values = s.gn[0] * s.gn[1] * 4;
    k_fold_add<<<(values + 255) / 256, 256, 0, st>>>(s.grid, work + p.tab, values, p.slices);
    return 1 + 2 * ((K + p.chunk - 1) / p.chunk);
}

// Samples per chunk: 64, or as many as keep the chunks' rows within 64 MB (at
// least one row).  By T and the bins alone: the chunks decide the order of the
// sums, which must not depend on the memory that happens to be free.
static long long rw_per(long long T, int nbins)
{
    constexpr long long kRows = 8 << 20;  // doubles
    long long chunks = (T + 63) / 64;
    if (chunks > 2048) chunks = 2048;  // the rows' sum walks them one after another
    const long long most = kRows / nbins;
    if (chunks > most) chunks = most;
    if (chunks < 1) chunks = 1;
    return ((T + chunks - 1) / chunks + 31) / 32 * 32;
}

size_t reweight_doubles(long long T, int ncv, int nbins)
{
    const long long per = rw_per(T, nbins), chunks = (T + per - 1) / per;
    return (size_t)T * (ncv + 1) + 2 * (size_t)nbins + 2 * kFesBlocks + (chunks > 1 ? (size_t)chunks * nbins : 0);
}

int launch_fes_reweight(const double *S, const double *V, long long T, int ncv, const double *lo, const double *hi,
                        const int *n, double beta, double *work, double *F, cudaStream_t st)
{
    FesGrid g{};
    int nbins = 1;
    for (int d = 0; d < ncv; ++d) {
        g.lo[d] = lo[d];
        g.hi[d] = hi[d];
        g.n[d] = n[d];
        nbins *= n[d];
    }
    const long long per = rw_per(T, nbins);
    const int chunks = (int)((T + per - 1) / per);
    double *acc = work, *b0 = acc + nbins, *b1 = b0 + kFesBlocks;
    double *rows = chunks > 1 ? b1 + kFesBlocks : acc;  // a lone row is the bins' sums itself
    const int vb = fes_blocks(T), nb = fes_blocks(nbins);
    constexpr int kWarps = kFesThreads / 32;
    cudaMemsetAsync(rows, 0, sizeof(double) * (size_t)chunks * nbins, st);
    k_fes_vmax<<<vb, kFesThreads, 0, st>>>(V, T, b0);
    k_fes_accum<<<(chunks + kWarps - 1) / kWarps, kFesThreads, 0, st>>>(S, V, T, ncv, g, beta, b0, vb, per, chunks,
                                                                       nbins, rows);
    const int sb = fes_blocks((long long)nbins * (kFesThreads / 32));  // 32 bins a block
    k_fes_bin_sum<<<sb, kFesThreads, 0, st>>>(rows, chunks, nbins, acc, b0);
    k_fes_log<<<nb, kFesThreads, 0, st>>>(acc, nbins, beta, b0, sb, F, b1);
    k_fes_shift<<<nb, kFesThreads, 0, st>>>(F, nbins, b1, nb, 1);
    return 5;
}

}  // namespace metad
