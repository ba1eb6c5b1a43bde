// Internal declarations of the sm_103a metadynamics bias path.
//
// One `Sys` value describes one system: geometry, switch constants and the
// device pointers of all its per-atom state.  Kernels take it by value; the
// batched kernels take a device array of them.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace metad {

constexpr int kNY = 13;          // real Y_6^m, m = -6..6
constexpr int kBlockAtoms = 128; // threads per block of the per-atom kernels
constexpr int kBlockBias = 256;  // threads per block of the hill kernels
constexpr int kMaxBiasBlocks = 304;  // two per SM
constexpr int kHillsPerBlock = 512;  // hill kernel: blocks of kBlockBias threads take this many hills each
constexpr int kMaxCv = 5;        // CN, Q6 and the three lattice parameters

enum ErrBits : int {
    kErrCapacity = 1,   // an atom had more neighbours than max_nb
    kErrNonFinite = 2,  // a position was NaN or infinite
    kErrHills = 4,      // live hill list overflow
    kErrInternal = 8,   // a launch shape the buffers were not sized for
};

// Slots of the per-system FP64 scalar block `scal` (D = ncv + 3 lattice CVs
// at most kMaxCv; each vector slot holds kMaxCv entries).
enum Scal : int {
    kS0 = 0, kS1 = 1,            // CVs s1, s2 (then the lattice CVs, if any)
    kV = 5, kDV0 = 6, kDV1 = 7,  // bias and its gradient at the CVs
    kDepV = 11, kDepDV0 = 12,    // bias and gradient at the last deposit centre
    kDepW = 17,                  // height of the last deposited hill
    kDepC0 = 18,                 // the last deposit centre (or a caller's CV point)
    kVir0 = 23,                  // bias virial sum_pairs (dV/dd)_a d_a, a = x, y, z
    kBoxG0 = 26,                 // dV/dL_a at fixed fractional coordinates
    kCnFac = 29,                 // 2 dV/ds1 / N, left by the hill kernel for the force pass
    kErrWord = 31,               // the device error word (an int)
    kNumScal = 32
};

// CV families (the metad_params.cv_kind values).
enum CvKind : int { kKindCoord = 0, kKindTorsion = 1, kKindNearest = 2 };

struct Sys {
    int n;          // atoms
    int ncv;        // 1 or 2
    int kind;       // CvKind
    int cn_unlike;  // CN mask
    int max_nb;     // ELL capacity per atom
    // box
    double L[3];
    float Lhi[3], Llo[3], halfL[3];
    float Lin[3];          // the largest float below L: x < L  <=>  x <= Lin
    // cells (edge >= rc, Morton-ranked)
    int nc[3];
    int ncell;
    float inv_h[3];
    // neighbour predicate: r^2 < rc^2 decided in FP64 inside the guard band
    double rc2;
    float rc2_lo, rc2_hi;
    float wrap2;           // below (half the shortest box length)^2, with margin
    // switch
    int sw_n, sw_m, stretch;
    float sw_nf;                 // sw_n and N as floating point: an int
    double sw_nd;                // conversion in a per-pair loop runs on
    float n_f;                   // the slow FP64 pipe of this part
    double n_d;
    double r0, rc;
    float inv_r0_hi, inv_r0_lo;  // 1/r0 as a float pair
    float a_hi, a_lo;            // 1/(1 - s_raw(rc)) (1 when not stretched)
    float k_hi, k_lo;            // s_raw(rc)/(1 - s_raw(rc)) (0 when not stretched)
    double a_d, k_d, inv_r0_d;
    // per-atom state, sorted (Morton) order unless noted
    const float4 *pos_in;  // caller order
    float4 *pos_s;
    int *perm;             // sorted -> caller
    unsigned *raw;         // rebuild: each cell's atoms before they are ordered
    int *ucell, *uslot;    // caller order: cell and slot within it
    int *cell_count;       // [ncell]
    int *cell_start;       // [ncell + 1]
    int *scan_part;        // block partial sums of the cell scan
    const int *rank_of_xyz;  // cell (x, y, z) -> Morton rank
    const int *xyz_of_rank;  // Morton rank -> packed x | y << 10 | z << 20
    int *nbr;              // [n][max_nb] FP64, two CVs: sorted indices of the exact row,
                           // entries j > i first (nh of them), then j < i; its pair pass
                           // searches them
    int *nn;               // [n]
    int *nh;               // [n] entries with j > i
    void *wl;              // JW<real> [n][max_nb]: neighbour and switch weight of each entry
    void *pairF;           // FP64, two CVs: [n][max_nb][4], G_ij in i's entry of j, -G_ji in the others
    void *cross;           // two CVs, real of each entry (entry_slot): b_i.q_j + b_j.q_i
                           // (FP64: its half b_j.q_i)
    void *geo;             // real[4] of each entry (entry_slot): r_j - r_i (minimum image) and
                           // the CN mask, written by the exact filter
    // Verlet list (cutoff rc + skin, built at the reference positions)
    float4 *pos_ref;       // sorted positions at the last rebuild
    int *vnbr;             // [n][max_vnb]
    int *vnn;              // [n]
    int max_vnb;
    int *flag;             // 1: rebuild the cell order and Verlet list this step
    float disp_thr2;       // (skin / 2)^2 with margin: rebuild above it
    float skin_eff;        // skin with margin
    float *Lref;           // [3] the box at the last rebuild (float)
    float rv2;             // (rc + skin)^2 with margin: Verlet cutoff
    int always_rebuild;    // skin == 0
    unsigned long long *rebuilds;  // number of rebuilds done
    void *cn, *W, *qb6;    // real-typed per-atom scalars (one CV, FP32, virial: W holds an error term, see k_cv.cu)
    void *q, *b, *h;       // real-typed per-atom records [n][16]: q_m; b_m, beta; h_m, gamma.
                           // FP32: b is [n][32], q and b side by side in chunks of four
                           // (q0..3 b0..3 q4..7 ...).  One CV: q is [n][8], the sums of
                           // the coordination number's force and virial
    double *part;          // per-block FP64 partial sums, slots of part_stride
    int part_stride;
    unsigned *ticket;      // completion counters of the last-block reductions
    double *scal;          // kNumScal doubles
    int *err;
    // hills and grid
    double *hc;            // [cap][hstride]
    double *hw;            // [cap]
    int hill_cap;
    double sigma[kMaxCv];  // per CV (the lattice CVs last)
    double inv2v[kMaxCv];  // 0.5 / sigma^2 per CV
    double k2v[kMaxCv];    // log2(e) / (2 sigma^2) per CV
    int D;                 // CVs the hills see: ncv (+ 3 lattice parameters)
    int hstride;           // doubles per hill centre: max(D, 2)
    int lattice;           // 1: the box lengths are CVs ncv .. ncv + 2
    int virial;            // 1: the force pass also sums the bias virial
    int pairs;             // 1: the force pass is the FP64 two-CV pair pass
    double w0, kbdt;
    int grid_on;
    int gn[2];
    double glo[2], ghi[2], gh[2];
    double *grid;          // [gn0][gn1][4]
    // per-step arguments, set on the copy of the descriptor a launch takes
    int K;                 // live hills
    const double *bias_x;  // CV point of the hill kernel
    double *bias_out;      // V, dV/ds1, dV/ds2 of the hill kernel
    int deposit;           // hill kernel: 1 = append a hill at bias_x
    float *F_out;          // caller's forces [n][F_stride]
    int F_stride;          // 3, or 4 with the fourth component written as 0
    int accumulate;        // 1: F_out += force, 0: F_out = force
    double fscale;         // forces are scaled by this, and by *fscale_dev unless NULL
    const double *fscale_dev;
    // torsion and nearest-distance families (no neighbour list)
    double period[kMaxCv];      // 0, or the period of a periodic CV (2 pi for a torsion)
    double inv_period[kMaxCv];  // 1 / period (0 when not periodic)
    double half[kMaxCv], three_half[kMaxCv];  // 1/2 and 3/2 periods
    const int *cv_atoms;   // torsion: [ncv][4]; nearest: [ncv] references, then n_cand candidates
    const int *cand_slot;  // nearest: [n] position of each atom in the candidate group, or -1
    int n_cand;
    double sm_beta;        // nearest: 0 = exact, > 0 = soft minimum
    double *gcv;           // [ncv][16] per-CV gradient terms of the last CV pass
};

// Programmatic dependent launch along the kernels of a step.  A kernel of the
// chain lets the next one be scheduled once all its own blocks have started
// (so the next launch overlaps its run instead of following it), and waits
// for the previous kernel to complete, its memory visible, before it reads or
// writes anything.  Every kernel that may be launched so waits in every
// thread that goes on, so completion carries along the chain.  (Without a
// programmatic launch the wait returns at once: the previous kernel has
// completed.)  Loads of data that an earlier kernel of the step writes are
// plain ones or the ld_* below: a read-only load (__ldg) may be moved before
// the wait, and so may assembly that is neither volatile nor marked as
// touching memory (to the compiler a function of its address alone), which
// the toolkit's cache-hint loads (__ldcs, __ldcg) need not be.
__device__ __forceinline__ void chain_enter()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Loads with a cache hint or of 32 B, kept in program order with the wait
// above, fences and stores by "volatile" and the memory clobber.  ld_stream:
// evict-first, for data read for the last time; ld_l2: past the L1, for what
// other blocks of the same kernel wrote.
__device__ __forceinline__ float ld_stream(const float *p)
{
    float v;
    asm volatile("ld.global.cs.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float4 ld_stream(const float4 *p)
{
    float4 v;
    asm volatile("ld.global.cs.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ double2 ld_stream(const double2 *p)
{
    double2 v;
    asm volatile("ld.global.cs.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ double ld_l2(const double *p)
{
    double v;
    asm volatile("ld.global.cg.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_l2(const int *p)
{
    int v;
    asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void ld_8(const float *p, float a[4], float b[4])
{
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(a[0]), "=f"(a[1]), "=f"(a[2]), "=f"(a[3]), "=f"(b[0]), "=f"(b[1]), "=f"(b[2]), "=f"(b[3])
                 : "l"(p)
                 : "memory");
}

// The difference s - c a hill sees along CV d: wrapped into [-P/2, P/2]
// (nearest image) for a periodic CV, x - P rint(x / P), with x / P taken as
// x * (1 / P) (no division per hill; the two can pick different images only
// within an ulp of a half period, where both images are equally near).
__device__ __forceinline__ double hill_diff(const Sys &s, int d, double x)
{
    const double P = s.period[d];
    if (P > 0.0) x -= P * rint(x * s.inv_period[d]);
    return x;
}

// A coordinate wrapped into [0, L): x - L floor(x / L) in FP64, rounded to
// float32; a result that rounds up to L becomes 0.  The in-box test is the
// FP32 comparison with Lin (exact: x < L iff x <= Lin for a float x), so a
// wrapped input costs no FP64 instruction (their pipe is narrow here).
__device__ __forceinline__ float wrap_coord(float x, float Lin, double L)
{
    if (x >= 0.0f && x <= Lin) return x;
    double xd = (double)x;
    double w = xd - L * floor(xd / L);
    float f = (float)w;
    if ((double)f >= L) f = 0.0f;
    return f;
}

// What the forces are scaled by.
__device__ __forceinline__ double force_scale(const Sys &s)
{
    return s.fscale_dev ? s.fscale * *s.fscale_dev : s.fscale;
}

// Where a block works: block b of a grid of nb blocks of its system.  A
// single-system launch is that grid; a batched launch concatenates the grids
// of all its systems.
struct Blk {
    int b, nb;
};

__device__ __forceinline__ Blk own_blk() { return Blk{(int)blockIdx.x, (int)gridDim.x}; }

// A batched launch: block x belongs to system k with pre[k] <= x < pre[k + 1]
// (systems with no block in this launch have pre[k] == pre[k + 1]).
struct BatchView {
    const Sys *sys;  // device [nsys]
    const int *pre;  // device [nsys + 1], this launch's row
    int nsys;
};

// The warp's lanes probe the table together, 32 entries a round (two dependent
// loads up to 1,024 systems where a search by halves chains ten).  The whole
// warp calls it.
__device__ __forceinline__ int batch_system(const BatchView &v, Blk &k)
{
    const int x = (int)blockIdx.x, lane = threadIdx.x & 31;
    int lo = 0, n = v.nsys;  // the system is one of lo .. lo + n - 1
    while (n > 1) {
        const int step = (n + 31) >> 5, at = lo + lane * step;
        const bool in = at < lo + n && __ldg(v.pre + at) <= x;  // true for a prefix of the lanes, lane 0 among them
        const int last = __popc(__ballot_sync(0xffffffffu, in)) - 1;
        n = min(step, lo + n - (lo + last * step));
        lo += last * step;
    }
    const int p0 = __ldg(v.pre + lo);
    k.b = x - p0;
    k.nb = __ldg(v.pre + lo + 1) - p0;
    return lo;
}

// Grids of a step, one row of block counts per launch kind.
enum GridKind : int {
    GK_ATOM256 = 0,    // one thread per atom, 256 per block
    GK_ATOM256_CAP,    // rebuild: binning, scatter and cell sort
    GK_SCAN_TILES,     // rebuild: cell scan
    GK_GROUPS_CAP,     // rebuild: Verlet rows
    GK_ONE,            // one block per system
    GK_GROUPS,         // one block per 16 atoms (lane-group kernels); a batch tile caps it
    GK_ROWS,           // one block per kRowAtoms atoms (four-lane kernels); a batch tile caps it
    GK_FORCE,          // the force pass
    GK_SUM,            // the CV sums: blocks by N only
    GK_HILLS,          // hill kernel, evaluation
    GK_DEPOSIT,        // hill kernel, deposit (systems that deposit)
    kGridKinds
};

// Block count of one system for a grid kind (host side; shared by the
// single-system launches and the batch tables).  persist_cap > 0 caps the
// lane-group grids (a batch tile setting), 0 keeps the default.
int grid_blocks(const Sys &s, int kind, int persist_cap);

// A kernel of a step, launched so it may be scheduled while the previous
// kernel of the stream still runs (it waits for it on the device).
template <typename... Args>
void chained(void (*kern)(Args...), int grid, int block, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
    if (e == cudaErrorNotSupported || e == cudaErrorInvalidValue) {
        // a stream that refuses the attribute gets a plain launch (the
        // device-side wait is then already satisfied); the refusal is this
        // launch's own error, cleared before the retry.  Any other launch
        // error stays pending for the caller's check.
        cudaGetLastError();
        cfg.numAttrs = 0;
        cudaLaunchKernelEx(&cfg, kern, args...);
    }
}

// The same for the kernels outside the rebuild chain, but plain in a stream
// that is being captured: us a step of 1,000 / 27,648 / 100,000 atoms, all
// launches plain, then chained: launched 46.7 / 62.0 / 120.4, 39.1 / 55.6 /
// 108.9; replayed from a graph 37.4 / 51.0 / 107.9, 35.6 / 54.1 / 106.4 (at
// 10,000 41.3, 43.7), so a graph keeps the plain ones.
template <typename... Args>
void chained_live(void (*kern)(Args...), int grid, int block, cudaStream_t st, Args... args)
{
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone)
        chained(kern, grid, block, st, args...);
    else
        kern<<<grid, block, 0, st>>>(args...);
}

// Batched stage launches (one launch each over every system of the view).
void launch_batch_gather(const BatchView &v, int total, cudaStream_t st);
void launch_batch_rebuild(const BatchView *rows, const int *totals, cudaStream_t st);
void launch_batch_cv(const BatchView &groups, int group_total, const BatchView &rows, int row_total, int fp64, int ncv,
                     int virial, cudaStream_t st);
void launch_batch_sum(const BatchView &sums, int sum_total, int fp64, cudaStream_t st);
void launch_cv_sum(const Sys &s, int fp64, cudaStream_t st);
void launch_batch_bias(const BatchView &v, int total, int deposit, cudaStream_t st);
void launch_batch_adjoint(const BatchView &rows, int total, int fp64, cudaStream_t st);
// The kernels after dV/ds is known; returns how many.
int launch_batch_forces(const BatchView &force, int force_total, const BatchView &groups, int group_total, int fp64,
                        int ncv, int virial, cudaStream_t st);
void launch_batch_collect(const BatchView &v, double *out, cudaStream_t st);

// Launch entry points (stream-ordered, no host synchronisation).
void launch_gather_check(const Sys &s, cudaStream_t st);
void launch_rebuild(const Sys &s, cudaStream_t st);  // kernels early-exit unless *flag
int rebuild_kernels(const Sys &s);                   // how many they are
void launch_filter(const Sys &s, int fp64, cudaStream_t st);
void launch_cv_fwd(const Sys &s, int fp64, int fused_filter, cudaStream_t st);
void launch_cv_avg(const Sys &s, int fp64, cudaStream_t st);
void launch_bias(const Sys &s, int K, const double *s_dev, double *out_dev, int deposit, cudaStream_t st);
void launch_adjoint(const Sys &s, int fp64, cudaStream_t st);
// Where forces go, and by what they are scaled.
struct ForceOut {
    float *F;
    int stride, accumulate;
    double scale;
    const double *scale_dev;
    void set(Sys &s) const
    {
        s.F_out = F;
        s.F_stride = stride;
        s.accumulate = accumulate;
        s.fscale = scale;
        s.fscale_dev = scale_dev;
    }
};
// The force pass (+ virial if s.virial): one kernel, except that the FP64
// two-CV one leaves its pair forces for launch_force_gather.
void launch_forces(const Sys &s, int fp64, const ForceOut &out, cudaStream_t st);
inline bool pair_slots(const Sys &s, int fp64) { return fp64 && s.ncv == 2; }
// Whether the CV pass leaves the exact rows behind it (the FP32 pass of one CV
// goes over the candidates without them; whoever wants them runs the filter).
inline bool stores_rows(const Sys &s, int fp64) { return fp64 || s.ncv == 2; }
void launch_force_gather(const Sys &s, int fp64, const ForceOut &out, cudaStream_t st);
void configure_kernels();
void launch_grid_fold(const Sys &s, int K, cudaStream_t st);
void launch_nn_stats(const Sys &s, unsigned long long *sum, int *mx, cudaStream_t st);
// Kernels whose only argument is the descriptor, per file, and which of them
// read the positions or write the forces (step graphs patch those in place).
enum SysKernel : int { kNotSys = 0, kSysOnly = 1, kSysIo = 2 };
SysKernel sys_kernel_neighbors(const void *func);
SysKernel sys_kernel_cv(const void *func);
SysKernel sys_kernel_bias(const void *func);
SysKernel sys_kernel_gcv(const void *func);
void launch_export_pairs(const Sys &s, int fp64, long long *pairs, int *count, cudaStream_t st);
void launch_per_atom_out(const Sys &s, int fp64, double *out, cudaStream_t st);
void set_ylm_constants(cudaStream_t st);
// Torsion and nearest-distance families: the CV pass (one block per system)
// and the force pass (one thread per atom).
void launch_gcv_forward(const Sys &s, int fp64, cudaStream_t st);
void launch_gcv_forces(const Sys &s, const ForceOut &out, cudaStream_t st);
void launch_batch_gcv(const BatchView &one, int one_total, int fp64, cudaStream_t st);
void launch_batch_gcv_forces(const BatchView &atoms, int atom_total, cudaStream_t st);
// The whole small-system step in one launch (CVs, hills, deposit, forces),
// for systems of at most kFuseAtoms atoms.
constexpr int kFuseAtoms = 32768;
void launch_gcv_step(const Sys &s, int K, float *F, int accumulate, int deposit, int fp64, cudaStream_t st);
void launch_batch_gcv_step(const BatchView &hills, int hill_total, int fp64, cudaStream_t st);

int bias_blocks(int K);

// Free-energy passes (k_fes.cu): F at the bin centres of a regular grid from
// the hills (and grid), and F reweighted from biased samples; F: device
// [prod n].  Each takes a workspace of *_doubles() doubles (launch_fes_points
// leaves F at its start) and returns the kernels launched.  fes_separable:
// whether the contraction form serves this grid.
bool fes_separable(const Sys &s, int K, const int *n);
size_t fes_points_doubles(const Sys &s, int K, const int *n, bool separable);
int launch_fes_points(const Sys &s, int K, const double *lo, const double *hi, const int *n, double *scratch,
                      bool separable, double fac, cudaStream_t st);
size_t reweight_doubles(long long T, int ncv, int nbins);
int launch_fes_reweight(const double *S, const double *V, long long T, int ncv, const double *lo, const double *hi,
                        const int *n, double beta, double *work, double *F, cudaStream_t st);
// Fold of the live hills into the grid through the contraction; the doubles
// its workspace takes for any number of hills the context holds, 0: the fold
// runs node by node, without one (launch_grid_fold).
size_t fold_doubles(const Sys &s);
int launch_fold_separable(const Sys &s, int K, double *work, cudaStream_t st);

// ----------------------------------------------------------------- device math
__device__ __forceinline__ float mi_f(float d, float halfL, float Lhi, float Llo)
{
    // one periodic shift, L carried as a float pair so the shift adds no
    // systematic error
    if (d > halfL) d = (d - Lhi) - Llo;
    else if (d < -halfL) d = (d + Lhi) + Llo;
    return d;
}

__device__ __forceinline__ double mi_d(double d, double L)
{
    if (d > 0.5 * L) d -= L;
    else if (d < -0.5 * L) d += L;
    return d;
}

template <typename real>
struct Vec3 {
    real x, y, z;
};

// Displacement r_j - r_i, minimum image, in the pair precision.
template <typename real>
__device__ __forceinline__ Vec3<real> displacement(const Sys &s, float4 pi, float4 pj);

// One axis of the minimum-image displacement xj - xi in float32.  Across the
// periodic boundary xj - xi is about +-L and would round at ulp(L) (7.6e-6 A
// for a 230 A box, a 1e-5 relative error in the switch of that pair); instead
// the coordinate near L is shifted first (x - L_hi is exact by Sterbenz), so
// only the small remainder is rounded.  The two directions of a pair give
// exactly opposite results.
__device__ __forceinline__ float mi_axis(float xj, float xi, float halfL, float Lhi, float Llo)
{
    const float d = xj - xi;
    if (d > halfL) return ((xj - Lhi) - xi) - Llo;   // xj near L
    if (d < -halfL) return (xj - (xi - Lhi)) + Llo;  // xi near L
    return d;
}

template <>
__device__ __forceinline__ Vec3<float> displacement<float>(const Sys &s, float4 pi, float4 pj)
{
    Vec3<float> d;
    d.x = mi_axis(pj.x, pi.x, s.halfL[0], s.Lhi[0], s.Llo[0]);
    d.y = mi_axis(pj.y, pi.y, s.halfL[1], s.Lhi[1], s.Llo[1]);
    d.z = mi_axis(pj.z, pi.z, s.halfL[2], s.Lhi[2], s.Llo[2]);
    return d;
}

template <>
__device__ __forceinline__ Vec3<double> displacement<double>(const Sys &s, float4 pi, float4 pj)
{
    Vec3<double> d;
    d.x = mi_d((double)pj.x - (double)pi.x, s.L[0]);
    d.y = mi_d((double)pj.y - (double)pi.y, s.L[1]);
    d.z = mi_d((double)pj.z - (double)pi.z, s.L[2]);
    return d;
}

// 1/sqrt(v) and 1/v in FP32, branch-free: the SFU estimate y refined by one
// Newton-Raphson step whose residual is formed without losing the product's
// rounding error (Markstein's scheme; the exact error of v*y recovered by an
// FMA, as in Dekker's two-product).  The step's result is y (1 + r/2) (resp.
// y (1 + r)) rounded once, within a few units of 2^-44 of the exact value:
// correctly rounded except next to a rounding tie, and with no rounding
// bias.  (An estimate refined with a rounded residual rounds with a bias:
// over many pairs it shifted the averaged Q6 by about -2e-7 relative, which
// the bias gradient amplifies past the 1e-5 tolerance.)  Positive normal
// arguments only (squared pair distances, switch denominators >= 1).
__device__ __forceinline__ float rsqrt_newton(float v)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(v));
    const float p = v * y;
    const float pe = fmaf(v, y, -p);                  // v y = p + pe exactly
    const float r = fmaf(-pe, y, fmaf(-p, y, 1.0f));  // 1 - v y^2
    return fmaf(0.5f * y, r, y);
}
__device__ __forceinline__ float recip_newton(float v)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(v));
    const float r = fmaf(-v, y, 1.0f);  // 1 - v y, one rounding of a quantity of order 2^-22
    return fmaf(y, r, y);
}

template <typename real>
__device__ __forceinline__ real rsqrt_r(real v);
template <>
__device__ __forceinline__ float rsqrt_r<float>(float v) { return rsqrt_newton(v); }
template <>
__device__ __forceinline__ double rsqrt_r<double>(double v) { return 1.0 / sqrt(v); }

template <typename real>
__device__ __forceinline__ real recip_r(real v);
template <>
__device__ __forceinline__ float recip_r<float>(float v) { return recip_newton(v); }
template <>
__device__ __forceinline__ double recip_r<double>(double v) { return 1.0 / v; }

// Rational switch s_raw = (1 - x^n)/(1 - x^m), x = r/r0.  For integer n, m
// it equals S_n(x)/S_m(x) with S_k = 1 + x + ... + x^(k-1): sums of positive
// terms, so no cancellation near x = 1 (where float32 would lose 1e-4 of its
// precision) and no removable singularity.  m == 2n reduces to 1/(1 + x^n).
// Returns w and dw/dr (stretched: shifted and scaled to vanish at rc).
template <typename real>
__device__ __forceinline__ void switch_eval(const Sys &s, real r, real &w, real &dw);

template <typename real>
__device__ __forceinline__ real ipow(real x, int n)
{
    real v = real(1);
    real b = x;
    while (n > 0) {
        if (n & 1) v *= b;
        b *= b;
        n >>= 1;
    }
    return v;
}

// S_k(x) and S_k'(x) by Horner.
template <typename real>
__device__ __forceinline__ void geom_sum(real x, int k, real &S, real &dS)
{
    S = real(0);
    dS = real(0);
    for (int t = k - 1; t >= 0; --t) {
        dS = dS * x + S;
        S = S * x + real(1);
    }
}

template <typename real>
__device__ __forceinline__ real sw_n_real(const Sys &s);
template <>
__device__ __forceinline__ float sw_n_real<float>(const Sys &s) { return s.sw_nf; }
template <>
__device__ __forceinline__ double sw_n_real<double>(const Sys &s) { return s.sw_nd; }

template <typename real>
__device__ __forceinline__ real n_real(const Sys &s);
template <>
__device__ __forceinline__ float n_real<float>(const Sys &s) { return s.n_f; }
template <>
__device__ __forceinline__ double n_real<double>(const Sys &s) { return s.n_d; }

template <typename real>
__device__ __forceinline__ void switch_raw(const Sys &s, real x, real &f, real &dfdx)
{
    const int n = s.sw_n, m = s.sw_m;
    if (m == 2 * n) {
        real xn1;
        if (n == 6) {  // the common 6-12 switch: x^5 without the power loop
            const real x2 = x * x;
            xn1 = x2 * x2 * x;
        } else {
            xn1 = ipow<real>(x, n - 1);
        }
        real xn = xn1 * x;
        real inv = recip_r<real>(real(1) + xn);
        f = inv;
        dfdx = -sw_n_real<real>(s) * xn1 * inv * inv;
        return;
    }
    real Sn, dSn, Sm, dSm;
    geom_sum<real>(x, n, Sn, dSn);
    geom_sum<real>(x, m, Sm, dSm);
    const real inv = recip_r<real>(Sm);
    f = Sn * inv;
    dfdx = (dSn * Sm - Sn * dSm) * inv * inv;
}

template <>
__device__ __forceinline__ void switch_eval<float>(const Sys &s, float r, float &w, float &dw)
{
    float x = fmaf(r, s.inv_r0_hi, r * s.inv_r0_lo);
    float f, dfdx;
    switch_raw<float>(s, x, f, dfdx);
    // (f - s_c) / (1 - s_c) = f*a - k with a, k carried as float pairs
    w = (fmaf(f, s.a_hi, f * s.a_lo) - s.k_hi) - s.k_lo;
    dw = dfdx * s.a_hi * s.inv_r0_hi;
}

template <>
__device__ __forceinline__ void switch_eval<double>(const Sys &s, double r, double &w, double &dw)
{
    double x = r * s.inv_r0_d;
    double f, dfdx;
    switch_raw<double>(s, x, f, dfdx);
    w = f * s.a_d - s.k_d;
    dw = dfdx * s.a_d * s.inv_r0_d;
}



__device__ __forceinline__ void set_err(const Sys &s, int bits) { atomicOr(s.err, bits); }

// ------------------------------------------------------------------ bias grid
__device__ __forceinline__ void hermite(double t, double A[2], double B[2], double dA[2], double dB[2])
{
    const double t2 = t * t, t3 = t2 * t;
    A[0] = 2.0 * t3 - 3.0 * t2 + 1.0;
    A[1] = 3.0 * t2 - 2.0 * t3;
    B[0] = t3 - 2.0 * t2 + t;
    B[1] = t3 - t2;
    dA[0] = 6.0 * (t2 - t);
    dA[1] = 6.0 * (t - t2);
    dB[0] = 3.0 * t2 - 4.0 * t + 1.0;
    dB[1] = 3.0 * t2 - 2.0 * t;
}

// Bicubic Hermite patch of the node grid; zero outside [lo, hi].
__device__ __forceinline__ void grid_value(const Sys &s, double x0, double x1, double &V, double &g0, double &g1)
{
    V = g0 = g1 = 0.0;
    if (!s.grid_on) return;
    const double x[2] = {x0, x1};
    int c[2];
    double t[2];
    for (int a = 0; a < 2; ++a) {
        if (!(x[a] >= s.glo[a] && x[a] <= s.ghi[a])) return;
        int k = (int)floor((x[a] - s.glo[a]) / s.gh[a]);
        k = k < 0 ? 0 : (k > s.gn[a] - 2 ? s.gn[a] - 2 : k);
        c[a] = k;
        t[a] = (x[a] - (s.glo[a] + k * s.gh[a])) / s.gh[a];
    }
    double A0[2], B0[2], dA0[2], dB0[2], A1[2], B1[2], dA1[2], dB1[2];
    hermite(t[0], A0, B0, dA0, dB0);
    hermite(t[1], A1, B1, dA1, dB1);
    const double h0 = s.gh[0], h1 = s.gh[1];
    for (int a = 0; a < 2; ++a)
        for (int b = 0; b < 2; ++b) {
            const double *nd = s.grid + ((size_t)(c[0] + a) * s.gn[1] + (c[1] + b)) * 4;
            const double f = nd[0], fx = h0 * nd[1], fy = h1 * nd[2], fxy = h0 * h1 * nd[3];
            V += A0[a] * A1[b] * f + B0[a] * A1[b] * fx + A0[a] * B1[b] * fy + B0[a] * B1[b] * fxy;
            g0 += dA0[a] * A1[b] * f + dB0[a] * A1[b] * fx + dA0[a] * B1[b] * fy + dB0[a] * B1[b] * fxy;
            g1 += A0[a] * dA1[b] * f + B0[a] * dA1[b] * fx + A0[a] * dB1[b] * fy + B0[a] * dB1[b] * fxy;
        }
    g0 /= h0;
    g1 /= h1;
}


// ------------------------------------------------------------ lane groups
// Per-atom kernels give one atom a group of kG lanes; lane l handles the
// atom's neighbours l, l + kG, ... so all its neighbour loads are in flight
// together.
constexpr int kG = 8;
constexpr int kAtomsPerBlock = kBlockAtoms / kG;

// Grid of the eight-lane kernels.
__host__ __device__ inline int group_grid(int n) { return (n + kAtomsPerBlock - 1) / kAtomsPerBlock; }

// The CV sums run in their own kernel: kSumThreads threads per block, one
// block per kSumAtoms atoms (at most kMaxBiasBlocks blocks).
constexpr int kSumThreads = 256;
constexpr int kSumAtoms = 1024;
__host__ __device__ inline int sum_blocks(int n)
{
    const int b = (n + kSumAtoms - 1) / kSumAtoms;
    return b < 1 ? 1 : (b > kMaxBiasBlocks ? kMaxBiasBlocks : b);
}

// Atoms per warp of the FP64 pair pass: 32 keep its lanes full, but leave a
// small system on few SMs.  A step in us with 8 / 32 atoms (and with the
// virial): 2,000 atoms 103 / 172, 20,000 298 / 341 (298 / 349), 60,000 717 / 741
// (745 / 757), 80,000 935 / 950 (983 / 968), 150,000 1,692 / 1,661 (1,784 / 1,673).
__host__ __device__ inline int pair_chunk(int n) { return n < 70000 ? 8 : 32; }

// The row passes (Q6 average, adjoint, FP32 force) give an atom four lanes and
// a block kRowAtoms consecutive atoms.
constexpr int kRowThreads = 128;
constexpr int kRowAtoms = kRowThreads / 4;

// Blocks of the force pass: a thread per atom with one CV, four lanes per
// atom in FP32, a warp per chunk of atoms in the FP64 pair pass.
__host__ __device__ inline int force_grid(int n, int ncv, int pairs)
{
    const int atoms = ncv == 1 ? kBlockAtoms : (pairs ? pair_chunk(n) * (kBlockAtoms / 32) : kRowAtoms);
    return (n + atoms - 1) / atoms;
}

// Persistent grids (the capped rebuild kernels) have at
// most kPersistBlocks blocks, walking their work grid-stride.
constexpr int kPersistBlocks = 152 * 16;

// Blocks of the force pass with the virial, at most: the seven per SM that its
// registers leave resident, walking their work, so that no part of a second
// wave is left over and the last block has few partials to add.
constexpr int kVirialBlocks = 152 * 7;

// The it-th work item (atom group or chunk) of block b of nb: items b,
// b + nb, b + 2 nb, ...  The items of one sweep form one compact window of
// the Morton order, so the records they gather stay in L2.  (Mapping the
// blocks that share an SM to consecutive items, for L1 reuse, measured
// slower: the gather kernels lost more to L2 misses than they won in L1.)
__device__ __forceinline__ int work_item(Blk k, int it) { return k.b + it * k.nb; }

struct AtomLane {
    int i;    // atom (sorted index), may be >= n for idle groups
    int l;    // lane within the group
    bool ok;  // i < n
};

template <int G = kG>
__device__ __forceinline__ AtomLane atom_lane_at(const Sys &s, int blk)
{
    AtomLane a;
    a.i = blk * (kBlockAtoms / G) + (threadIdx.x / G);
    a.l = threadIdx.x & (G - 1);
    a.ok = a.i < s.n;
    return a;
}


template <int G>
__device__ __forceinline__ unsigned group_mask_bits(unsigned ballot)
{
    const int base = (threadIdx.x & 31) & ~(G - 1);
    return (ballot >> base) & ((1u << G) - 1u);
}

// Exact FP64 pair test: r^2 = (dx*dx + dy*dy) + dz*dz < rc^2 on the
// minimum-image displacement, no contraction.  Kept out of line and given
// plain values (no reference to the kernel's descriptor): it runs only for
// candidates inside the guard band, and inlined the compiler may evaluate
// it for every candidate under a predicate, on the slow FP64 pipe.
static __device__ __noinline__ bool pair_exact_fp64(float4 pi, float4 pj, double L0, double L1, double L2, double rc2)
{
    double dx = mi_d(__dadd_rn((double)pj.x, -(double)pi.x), L0);
    double dy = mi_d(__dadd_rn((double)pj.y, -(double)pi.y), L1);
    double dz = mi_d(__dadd_rn((double)pj.z, -(double)pi.z), L2);
    double r2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
    r2 = __dadd_rn(r2, __dmul_rn(dz, dz));
    return r2 < rc2;
}

__device__ __forceinline__ bool pair_exact(const Sys &s, float4 pi, float4 pj)
{
    return pair_exact_fp64(pi, pj, s.L[0], s.L[1], s.L[2], s.rc2);
}

// The float32 estimate decides every candidate outside a relative guard band
// of 3e-5 around rc^2; inside it the FP64 definition decides.  d is the
// float32 displacement of the pair.
__device__ __forceinline__ bool pair_in(const Sys &s, float4 pi, float4 pj, const Vec3<float> &d)
{
    float r2 = fmaf(d.x, d.x, fmaf(d.y, d.y, d.z * d.z));
    if (r2 < s.rc2_lo) return true;
    if (r2 > s.rc2_hi) return false;
    return pair_exact(s, pi, pj);
}

// displacement<float> and pair_in for code where the whole warp is converged:
// the plain difference decides unless its square lies in the guard band or
// above wrap2, which it does whenever some axis needs the minimum image; then
// the full forms run, behind one warp vote.  The same bits and decisions: the
// full displacement is the plain difference on an axis within half the box,
// and one beyond it has a square above the band (half the box is at least rc).
__device__ __forceinline__ bool pair_in_warp(const Sys &s, bool valid, float4 pi, float4 pj, Vec3<float> &d)
{
    d = Vec3<float>{pj.x - pi.x, pj.y - pi.y, pj.z - pi.z};
    const float r2 = fmaf(d.x, d.x, fmaf(d.y, d.y, d.z * d.z));
    bool in = valid && r2 < s.rc2_lo;
    const bool full = valid && r2 >= s.rc2_lo && (r2 <= s.rc2_hi || r2 > s.wrap2);
    if (__any_sync(0xffffffffu, full)) {
        if (full) {
            d = displacement<float>(s, pi, pj);
            in = pair_in(s, pi, pj, d);
        }
    }
    return in;
}

// The geometry of an exact entry, cached by the filter so the CV and force
// passes read one contiguous record per entry instead of gathering the
// neighbour's position again: r_j - r_i, and in the fourth slot a tag
// (carried through float registers unchanged): j, with the CN mask in bit 31.
// The force pass reads it for the last time (kLast: an evict-first load, so
// the stream does not push the gathered per-atom records out of L2).
constexpr unsigned kCnBit = 0x80000000u;

__device__ __forceinline__ unsigned make_tag(const Sys &s, int j, float4 pi, float4 pj)
{
    return (unsigned)j | ((!s.cn_unlike || pj.w != pi.w) ? kCnBit : 0u);
}

// An accepted candidate of the filter: FP32 writes the record whole, FP64 its
// tag alone (the displacement follows from it, fill_geo).
__device__ __forceinline__ void store_entry(const Sys &s, float, size_t slot, const Vec3<float> &df, unsigned tag)
{
    reinterpret_cast<float4 *>(s.geo)[slot] = make_float4(df.x, df.y, df.z, __uint_as_float(tag));
}
__device__ __forceinline__ void store_entry(const Sys &s, double, size_t slot, const Vec3<float> &, unsigned tag)
{
    reinterpret_cast<double *>(s.geo)[4 * slot + 3] = __longlong_as_double((long long)tag);
}

__device__ __forceinline__ void untag(unsigned tag, int &j, bool &cn)
{
    j = (int)(tag & ~kCnBit);
    cn = (tag & kCnBit) != 0u;
}

template <typename real, bool kLast = false>
__device__ __forceinline__ void load_geo(const Sys &s, size_t slot, Vec3<real> &d, bool &cn, int &j);
template <>
__device__ __forceinline__ void load_geo<float, false>(const Sys &s, size_t slot, Vec3<float> &d, bool &cn, int &j)
{
    const float4 g = reinterpret_cast<const float4 *>(s.geo)[slot];
    d = Vec3<float>{g.x, g.y, g.z};
    untag(__float_as_uint(g.w), j, cn);
}
template <>
__device__ __forceinline__ void load_geo<double, true>(const Sys &s, size_t slot, Vec3<double> &d, bool &cn, int &j)
{
    const double2 *g = reinterpret_cast<const double2 *>(s.geo) + 2 * slot;
    const double2 a = ld_stream(g), b = ld_stream(g + 1);
    d = Vec3<double>{a.x, a.y, b.x};
    untag((unsigned)__double_as_longlong(b.y), j, cn);
}
template <>
__device__ __forceinline__ void load_geo<double, false>(const Sys &s, size_t slot, Vec3<double> &d, bool &cn, int &j)
{
    const double2 *g = reinterpret_cast<const double2 *>(s.geo) + 2 * slot;
    const double2 a = g[0], b = g[1];
    d = Vec3<double>{a.x, a.y, b.x};
    untag((unsigned)__double_as_longlong(b.y), j, cn);
}

// Where the exact rows keep entry k of atom i (geometry, cross terms): the rows
// of eight consecutive atoms are interleaved by chunks of four entries, so that
// what the lane groups of a warp read or write at the same k lies together.
// The L1 serves a warp's access a 128 B line at a time, and with a row per atom
// each of the eight groups touches a line of its own, for 16 or 64 B of it
// (force pass, 1M atoms: 254 -> 235 us).  Row capacities are multiples of four, and the arrays
// hold whole slices of eight atoms.  (The entries of the gather passes, JW,
// stay a row per atom: a line of a row is then fetched once for sixteen
// entries, where interleaved pairs fetched one every round: Q6 pass 145 ->
// 188 us, adjoint 197 -> 313.)
constexpr int kSlice = 8;
__host__ __device__ inline size_t slice_rows(int n) { return ((size_t)n + kSlice - 1) / kSlice * kSlice; }
__device__ __forceinline__ size_t entry_base(const Sys &s, int i)
{
    return (size_t)(i & ~(kSlice - 1)) * s.max_nb + 4 * (i & (kSlice - 1));
}
__device__ __forceinline__ int entry_off(int k) { return (k >> 2) * (4 * kSlice) + (k & 3); }
__device__ __forceinline__ size_t entry_slot(const Sys &s, int i, int k) { return entry_base(s, i) + entry_off(k); }

// One exact entry for the gather passes: the neighbour and the switch
// weight side by side, read with one load.
template <typename real>
struct alignas(2 * sizeof(real)) JW {
    int j;
    real w;
};

// The candidates of atom i's Verlet row (vn of them; vmax the warp's most), G
// a round: each(valid, j, pj) in every lane of the warp, lane l of G taking
// candidates l, l + G, ...  Positions are loaded a round ahead of their use
// and indices two.
template <int G, typename F>
__device__ __forceinline__ void sweep_candidates(const Sys &s, int i, int l, int vn, int vmax, F &&each)
{
    const int *vrow = s.vnbr + (size_t)i * s.max_vnb;
    int j1 = l < vn ? vrow[l] : i;
    float4 p1 = s.pos_s[j1];
    int j2 = l + G < vn ? vrow[l + G] : i;
    for (int base = 0; base < vmax; base += G) {
        const int k = base + l, j = j1;
        const float4 pj = p1;
        j1 = j2;
        p1 = s.pos_s[j1];
        j2 = k + 2 * G < vn ? vrow[k + 2 * G] : i;
        each(k < vn, j, pj);
    }
}

// The accepted candidates of atom a.i's Verlet row compacted by ballot from
// entry cnt on.  kPart: 0 every exact entry, 1 those with j > i, 2 those with
// j < i.
template <typename real, int kPart, int G>
__device__ __forceinline__ int filter_sweep(const Sys &s, const AtomLane &a, int vn, int vmax, float4 pi, int cnt)
{
    const int i = a.ok ? a.i : 0;
    const size_t e0 = entry_base(s, i), row0 = (size_t)i * s.max_nb;
    const unsigned lt = (1u << a.l) - 1u;
    sweep_candidates<G>(s, i, a.l, vn, vmax, [&](bool valid, int j, float4 pj) {
        const bool part = kPart == 0 || (kPart == 1 ? j > a.i : j < a.i);
        Vec3<float> d;
        const bool in = pair_in_warp(s, valid && part, pi, pj, d);  // every lane: a warp vote inside
        const unsigned gm = group_mask_bits<G>(__ballot_sync(0xffffffffu, in));
        const int at = cnt + __popc(gm & lt);
        if (in && at < s.max_nb) {
            if (kPart != 0) s.nbr[row0 + at] = j;
            store_entry(s, real(0), e0 + entry_off(at), d, make_tag(s, j, pi, pj));
        }
        cnt += __popc(gm);
    });
    return cnt;
}

// FP64: the displacements of atom i's first nn entries from their tags, every
// lane with an entry.  Formed in the sweeps, few lanes of a round have one, and
// the warp pays for all (250,001 atoms, a step: one CV 906 -> 813 us, two 2,984 ->
// 2,665; build and filter 385 -> 322, 584 -> 324).
__device__ __forceinline__ void fill_geo(const Sys &s, int i, int l, int G, int nn, float4 pi)
{
    const size_t e0 = entry_base(s, i);
    for (int k = l; k < nn; k += G) {
        double *g = reinterpret_cast<double *>(s.geo) + 4 * (e0 + entry_off(k));
        int j;
        bool cn;
        untag((unsigned)__double_as_longlong(g[3]), j, cn);
        const Vec3<double> d = displacement<double>(s, pi, s.pos_s[j]);
        reinterpret_cast<double2 *>(g)[0] = make_double2(d.x, d.y);
        g[2] = d.z;
    }
}

// The exact row of atom a.i from its Verlet row.  For the FP64 two-CV pair
// pass the j > i entries come first, in a sweep of their own, and the row's
// indices are kept (it searches them); everyone else reads j from the tags.
template <typename real, int G>
__device__ __forceinline__ int filter_row(const Sys &s, const AtomLane &a)
{
    const int vn = a.ok ? s.vnn[a.i] : 0;
    const float4 pi = a.ok ? s.pos_s[a.i] : make_float4(0.f, 0.f, 0.f, 0.f);
    const int vmax = __reduce_max_sync(0xffffffffu, vn);
    int cnt;
    if (sizeof(real) == 8 && s.ncv == 2) {
        const int nh = filter_sweep<real, 1, G>(s, a, vn, vmax, pi, 0);
        cnt = filter_sweep<real, 2, G>(s, a, vn, vmax, pi, nh);
        if (a.ok && a.l == 0) s.nh[a.i] = min(nh, s.max_nb);
    } else {
        cnt = filter_sweep<real, 0, G>(s, a, vn, vmax, pi, 0);
    }
    if (a.ok && a.l == 0) {
        if (cnt > s.max_nb) set_err(s, kErrCapacity);
        s.nn[a.i] = min(cnt, s.max_nb);
    }
    __syncwarp();  // the group's lanes wrote the row
    cnt = min(cnt, s.max_nb);
    if (sizeof(real) == 8) {
        fill_geo(s, a.i, a.l, G, a.ok ? cnt : 0, pi);
        __syncwarp();
    }
    return cnt;
}

}  // namespace metad
