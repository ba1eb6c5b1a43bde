// Steps a1-a3: ingest, Morton-ranked cell order, Verlet list and the exact
// neighbour list.
//
// Each step:
//   k_gather_check  positions in cell order (wrapped), and a flag when any
//                   atom moved more than skin/2 since the last rebuild
//   rebuild chain   (early exit unless flagged) counting sort of the atoms
//                   into Morton-ranked cells of edge >= rc + skin (by octant,
//                   then caller index within a cell), and the Verlet list
//                   r < rc + skin
//   filter          exact rows {j : r_ij^2 < rc^2} from the Verlet rows
//                   (fused into the CV kernel, or k_filter on its own)
// The exact rows are the FP64 definition bit for bit: while no atom has moved
// more than skin/2, every pair now inside rc was inside rc + skin at the
// rebuild, and the float32 estimate only decides outside a guard band.
#include "metad_impl.cuh"

namespace metad {

namespace {

__device__ __forceinline__ float4 load_wrapped(const Sys &s, int u, bool &bad)
{
    float4 p = s.pos_in[u];
    bad = !(isfinite(p.x) && isfinite(p.y) && isfinite(p.z));
    if (bad) {
        p.x = p.y = p.z = 0.0f;
        return p;
    }
    p.x = wrap_coord(p.x, s.Lin[0], s.L[0]);
    p.y = wrap_coord(p.y, s.Lin[1], s.L[1]);
    p.z = wrap_coord(p.z, s.Lin[2], s.L[2]);
    return p;
}

__device__ __forceinline__ int cell_axis(float x, float inv_h, int nc)
{
    int c = (int)floorf(x * inv_h);
    return c < 0 ? 0 : (c >= nc ? nc - 1 : c);
}

// Current positions in the cell order of the last rebuild, and the rebuild
// test.  Before the first rebuild the flag is already set.  The Verlet rows
// hold every pair within rc + skin at the last rebuild; a pair's
// displacement has since changed by at most |dr_i| + |dr_j| + |L - L_ref|
// (the last term for pairs across the box faces when the box changed), so
// the rows stay valid while every |dr| <= (skin - |L - L_ref|) / 2.
__device__ __forceinline__ void gather_check(const Sys &s, Blk k)
{
    const int t = k.b * blockDim.x + threadIdx.x;
    bool move = false;
    float thr2 = s.disp_thr2;
    {
        const float ex = s.Lhi[0] - s.Lref[0], ey = s.Lhi[1] - s.Lref[1], ez = s.Lhi[2] - s.Lref[2];
        const float dL2 = ex * ex + ey * ey + ez * ez;
        if (dL2 > 0.0f) {
            const float half = 0.5f * (s.skin_eff - sqrtf(dL2));
            thr2 = half > 0.0f ? half * half : -1.0f;
        }
    }
    if (t < s.n) {
        bool bad;
        float4 p = load_wrapped(s, s.perm[t], bad);
        if (bad) set_err(s, kErrNonFinite);
        s.pos_s[t] = p;
        const float4 r = s.pos_ref[t];
        float dx = mi_f(p.x - r.x, s.halfL[0], s.Lhi[0], s.Llo[0]);
        float dy = mi_f(p.y - r.y, s.halfL[1], s.Lhi[1], s.Llo[1]);
        float dz = mi_f(p.z - r.z, s.halfL[2], s.Lhi[2], s.Llo[2]);
        move = !(dx * dx + dy * dy + dz * dz <= thr2) || p.w != r.w;
    }
    if (__any_sync(0xffffffffu, move) && (threadIdx.x & 31) == 0) atomicOr(s.flag, 1);
}

__global__ void k_gather_check(Sys s)
{
    chain_enter();
    gather_check(s, own_blk());
}

// Cell of an atom, its slot there, and the octant of the cell it lies in (in
// the top bits of the slot, and of the caller index where the cells are
// sorted; systems of 2^28 atoms and more need those bits and have no octants).
__device__ __forceinline__ int oct_shift(const Sys &s) { return s.n <= 1 << 28 ? 28 : 31; }
__device__ __forceinline__ unsigned low_bits(unsigned v, int shift) { return v & ((1u << shift) - 1u); }

__device__ __forceinline__ void bin_one(const Sys &s, int u)
{
    bool bad;
    float4 p = load_wrapped(s, u, bad);
    int cx = cell_axis(p.x, s.inv_h[0], s.nc[0]);
    int cy = cell_axis(p.y, s.inv_h[1], s.nc[1]);
    int cz = cell_axis(p.z, s.inv_h[2], s.nc[2]);
    int c = s.rank_of_xyz[(cz * s.nc[1] + cy) * s.nc[0] + cx];
    const int shift = oct_shift(s);
    unsigned oct = 0;
    if (shift == 28)  // explicit multiply-adds: single and batched kernels decide alike
        oct = (fmaf(p.x, s.inv_h[0], -(float)cx) >= 0.5f ? 1u : 0u) | (fmaf(p.y, s.inv_h[1], -(float)cy) >= 0.5f ? 2u : 0u) |
              (fmaf(p.z, s.inv_h[2], -(float)cz) >= 0.5f ? 4u : 0u);
    s.ucell[u] = c;
    s.uslot[u] = (int)((unsigned)atomicAdd(&s.cell_count[c], 1) | (oct << shift));
}

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ int block_exclusive_scan(int v, int *warp_sums, int &total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int w = warp_sums[lane];
        int t = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        warp_sums[lane] = t - w;
        if (lane == 31) warp_sums[32] = t;
    }
    __syncthreads();
    total = warp_sums[32];
    int r = warp_sums[wid] + x - v;
    __syncthreads();
    return r;
}

// The cell starts of a grid of at most kScanOne cells, by the 256 threads of
// one block, each 16 consecutive cells.
constexpr int kBinThreads = 256;
constexpr int kScanOne = kBinThreads * 16;
__device__ __forceinline__ void scan_one(const Sys &s, int *ws)
{
    const int base = threadIdx.x * 16;
    int c[16], v = 0;
#pragma unroll
    for (int t = 0; t < 16; ++t) {
        c[t] = base + t < s.ncell ? ld_l2(s.cell_count + base + t) : 0;
        v += c[t];
    }
    if (threadIdx.x < 32) ws[threadIdx.x] = 0;  // the scan sums 32 warps; a block has eight
    __syncthreads();
    int total;
    int ex = block_exclusive_scan(v, ws, total);
#pragma unroll
    for (int t = 0; t < 16; ++t) {
        if (base + t < s.ncell) s.cell_start[base + t] = ex;
        ex += c[t];
    }
    if (threadIdx.x == 0) s.cell_start[s.ncell] = s.n;
}

// kScan: the grid has at most kScanOne cells, and the last block to finish
// scans them (two kernels fewer in the chain, which a step without a rebuild
// pays for too).
template <bool kScan>
__device__ __forceinline__ void bin_count(const Sys &s, Blk k)
{
    if (!*s.flag) return;
    for (int u = k.b * blockDim.x + threadIdx.x; u < s.n; u += k.nb * blockDim.x) bin_one(s, u);
    if (!kScan) return;
    __shared__ int ws[33];
    __shared__ bool am_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) am_last = atomicAdd(&s.ticket[5], 1u) == (unsigned)k.nb - 1u;
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    scan_one(s, ws);
    if (threadIdx.x == 0) s.ticket[5] = 0u;
}

__device__ __forceinline__ void scan_reduce(const Sys &s, Blk k)
{
    if (!*s.flag) return;
    __shared__ int ws[33];
    int base = k.b * kScanTile + threadIdx.x * kScanItems;
    int v = 0;
#pragma unroll
    for (int t = 0; t < kScanItems; ++t)
        if (base + t < s.ncell) v += s.cell_count[base + t];
    int total;
    block_exclusive_scan(v, ws, total);
    if (threadIdx.x == 0) s.scan_part[k.b] = total;
}

// kDirect: a block adds the counts before its tile itself (a grid of few
// tiles), else the tiles' sums of scan_reduce.
constexpr int kDirectTiles = 48;
template <bool kDirect>
__device__ __forceinline__ void scan_down(const Sys &s, Blk k)
{
    if (!*s.flag) return;
    __shared__ int ws[33];
    __shared__ int prefix;
    if (kDirect) {
        const int4 *c4 = reinterpret_cast<const int4 *>(s.cell_count);
        int acc = 0;
#pragma unroll 4
        for (int q = threadIdx.x; q < k.b * (kScanTile / 4); q += kScanThreads) {
            const int4 v = c4[q];
            acc += (v.x + v.y) + (v.z + v.w);
        }
        int total;
        block_exclusive_scan(acc, ws, total);
        if (threadIdx.x == 0) prefix = total;
    } else if (threadIdx.x < 32) {
        int acc = 0;
        for (int b = threadIdx.x; b < k.b; b += 32) acc += s.scan_part[b];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (threadIdx.x == 0) prefix = acc;
    }
    __syncthreads();
    int base = k.b * kScanTile + threadIdx.x * kScanItems;
    int c[kScanItems];
    int v = 0;
#pragma unroll
    for (int t = 0; t < kScanItems; ++t) {
        c[t] = base + t < s.ncell ? s.cell_count[base + t] : 0;
        v += c[t];
    }
    int total;
    int ex = block_exclusive_scan(v, ws, total) + prefix;
#pragma unroll
    for (int t = 0; t < kScanItems; ++t) {
        if (base + t < s.ncell) s.cell_start[base + t] = ex;
        ex += c[t];
    }
    if (base <= s.ncell - 1 && s.ncell - 1 < base + kScanItems) s.cell_start[s.ncell] = s.n;
}

// Each cell's atoms, in the order of their atomic slots: octant and caller
// index, one word each.  The scanned counters are left zero for the next
// rebuild (zero from creation on, so no pass of their own clears them).
__device__ __forceinline__ void bin_scatter(const Sys &s, Blk k)
{
    if (!*s.flag) return;
    const int shift = oct_shift(s);
    for (int u = k.b * blockDim.x + threadIdx.x; u < s.n; u += k.nb * blockDim.x) {
        const unsigned v = (unsigned)s.uslot[u], slot = low_bits(v, shift);
        s.raw[s.cell_start[s.ucell[u]] + slot] = (unsigned)u | (v - slot);
    }
    for (int c = k.b * blockDim.x + threadIdx.x; c < s.ncell; c += k.nb * blockDim.x) s.cell_count[c] = 0;
}

// The sorted order: within a cell by octant, then caller index (the atomic
// slots are not deterministic).  Octants put atoms half a cell apart next to
// each other in memory, so a line of per-atom records holds more atoms that
// are neighbours of the same atom.  One thread per atom: its place is the
// number of smaller words in its cell (about eight, read from cache), where
// one thread sorting a cell by insertion chains its loads (48 us at 1M
// atoms).  Its wrapped position becomes the reference of the new Verlet list.
__device__ __forceinline__ void cell_sort_gather(const Sys &s, Blk k)
{
    if (!*s.flag) return;
    const int shift = oct_shift(s);
    for (int t = k.b * blockDim.x + threadIdx.x; t < s.n; t += k.nb * blockDim.x) {
        const unsigned v = s.raw[t];
        const int u = (int)low_bits(v, shift);
        const int c = s.ucell[u];
        const int a = s.cell_start[c], e = s.cell_start[c + 1];
        int at = a;
        for (int q = a; q < e; ++q) at += s.raw[q] < v ? 1 : 0;
        bool bad;
        const float4 p = load_wrapped(s, u, bad);
        s.perm[at] = u;
        s.pos_s[at] = p;
        s.pos_ref[at] = p;
    }
}

__device__ __forceinline__ int wrap_cell(int c, int nc)
{
    c += (c < 0) ? nc : 0;
    c -= (c >= nc) ? nc : 0;
    return c;
}

// Stencil offsets along one axis: -1, 0, 1 with three or more cells (each
// distinct cell once with fewer).
__device__ __forceinline__ int axis_span(int nc) { return nc >= 3 ? 3 : nc; }
__device__ __forceinline__ int axis_off(int nc, int idx) { return nc >= 3 ? idx - 1 : idx; }

// Verlet rows {j : r_ij^2 < (rc + skin)^2 (1 + 1e-4)} over the 27 cells
// around each atom's own (each distinct cell once), in stencil-cell order (x
// fastest), atoms in cell order.
//
// One warp per cell at a time.  The candidates of the cell's atoms are the
// same list; the warp stages it in shared memory (position, index, stencil
// cell), then gives each of the cell's na atoms 32 / na lanes, which take the
// list's entries in turn and compact the accepted ones with a ballot: the row
// comes out in list order whatever na is.  Bound by instruction issue: about
// 22 a round, and rounds x lanes is the cell's na x candidates (208 at skin 1)
// whatever their split, where a warp sweeping the list for one atom at a time
// spent its per-atom and partial-round overheads seven or eight times a cell.
// A list longer than the buffer is staged and swept in chunks.
//
// Displacements: with three or more cells along every axis each stencil cell
// is a distinct cell at one periodic image, and d = (r_j - r_i) + shift with
// the cell's image shift (0 or +-L per axis): no minimum-image test per
// candidate.  With fewer cells along an axis, the minimum image per
// candidate.  The 1e-4 margin on the cutoff covers the rounding of either
// form.
constexpr int kStencil = 27;
constexpr int kVerletWarps = kBlockAtoms / 32;
constexpr int kCandBuf = 320;  // staged candidates per warp

struct VerletWarpSmem {
    float4 pos[kCandBuf];      // candidate position, index bits in w
    unsigned char q[kCandBuf]; // candidate's stencil cell
    float4 shift[kStencil];    // image shift of each stencil cell
};

// Copy the candidates [k0, k0 + len) of the list into the buffer: lane q
// copies its stencil cell's n atoms from st on (list positions from o on), so
// the warp's loads are all independent of one another.
__device__ __forceinline__ void verlet_stage(const Sys &s, VerletWarpSmem &w, int st, int n, int o, int k0, int len,
                                             int lane)
{
    const int lo = max(o, k0), hi = min(o + n, k0 + len);
#pragma unroll 4
    for (int t = lo; t < hi; ++t) {
        const int j = st + (t - o);
        float4 pj = s.pos_s[j];
        pj.w = __int_as_float(j);
        w.pos[t - k0] = pj;
        w.q[t - k0] = (unsigned char)lane;
    }
    __syncwarp();
}

// Sweep the staged candidates [0, len): lane l of G takes candidates l, l + G,
// ... for atom i (its position pi; lanes past the atoms have on = false).
// gsh: the group's first lane.  kShift: some stencil cell of this one is a
// periodic image (a cell on the box faces); interior cells need no shift.
template <bool kImages, bool kShift>
__device__ __forceinline__ int verlet_sweep(const Sys &s, const VerletWarpSmem &w, int i, float4 pi, bool on, int l,
                                            int G, int gsh, int len, int *vrow, int cnt)
{
    const unsigned gmask = G == 32 ? 0xffffffffu : (1u << G) - 1u, lt = (1u << l) - 1u;
#pragma unroll 2
    for (int r = 0; r < len; r += G) {
        const int t = r + l;
        const int tc = min(t, kCandBuf - 1);  // in bounds; masked by t < len
        const float4 cp = w.pos[tc];
        const int j = __float_as_int(cp.w);
        Vec3<float> d;
        if (!kImages) {
            d = displacement<float>(s, pi, cp);
        } else {
            d.x = cp.x - pi.x;
            d.y = cp.y - pi.y;
            d.z = cp.z - pi.z;
            if (kShift) {
                // past the staged length w.q is stale: keep the index in the table
                const float4 h = w.shift[min((int)w.q[tc], kStencil - 1)];
                d.x += h.x;
                d.y += h.y;
                d.z += h.z;
            }
        }
        const bool in = on && t < len && j != i && fmaf(d.x, d.x, fmaf(d.y, d.y, d.z * d.z)) < s.rv2;
        const unsigned m = (__ballot_sync(0xffffffffu, in) >> gsh) & gmask;
        const int at = cnt + __popc(m & lt);
        if (in && at < s.max_vnb) vrow[at] = j;
        cnt += __popc(m);
    }
    return cnt;
}

template <bool kImages>
__device__ __forceinline__ void verlet_cell(const Sys &s, VerletWarpSmem &w, int c, int lane)
{
    const int a0 = s.cell_start[c], na = s.cell_start[c + 1] - a0;
    if (na == 0) return;
    const int xyz = s.xyz_of_rank[c];
    const int cx = xyz & 1023, cy = (xyz >> 10) & 1023, cz = xyz >> 20;
    // with images every axis spans three cells: constant divisions below
    const int sx = kImages ? 3 : axis_span(s.nc[0]), sy = kImages ? 3 : axis_span(s.nc[1]),
              sz = kImages ? 3 : axis_span(s.nc[2]);
    const int nq = sx * sy * sz;
    // a cell on the box faces has stencil cells at a periodic image
    const bool shifted = cx == 0 || cy == 0 || cz == 0 || cx == s.nc[0] - 1 || cy == s.nc[1] - 1 || cz == s.nc[2] - 1;
    // the stencil: lane q < nq looks up cell q (x fastest)
    int st = 0, n = 0;
    if (lane < nq) {
        const int ex = lane % sx, ey = (lane / sx) % sy, ez = lane / (sx * sy);
        const int x = cx + axis_off(s.nc[0], ex), y = cy + axis_off(s.nc[1], ey), z = cz + axis_off(s.nc[2], ez);
        const int cq = s.rank_of_xyz[(wrap_cell(z, s.nc[2]) * s.nc[1] + wrap_cell(y, s.nc[1])) * s.nc[0] +
                                     wrap_cell(x, s.nc[0])];
        st = s.cell_start[cq];
        n = s.cell_start[cq + 1] - st;
        if (kImages && shifted)  // only a cell on the box faces reads the shifts
            w.shift[lane] = make_float4(x < 0 ? -s.Lhi[0] : (x >= s.nc[0] ? s.Lhi[0] : 0.0f),
                                        y < 0 ? -s.Lhi[1] : (y >= s.nc[1] ? s.Lhi[1] : 0.0f),
                                        z < 0 ? -s.Lhi[2] : (z >= s.nc[2] ? s.Lhi[2] : 0.0f), 0.0f);
    }
    int o = n;  // inclusive, then exclusive scan of the cells' sizes
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, o, k);
        if (lane >= k) o += y;
    }
    const int T = __shfl_sync(0xffffffffu, o, 31);
    o -= n;
    // lanes per atom; more than 32 atoms go in batches of 32
    const int G = na <= 32 ? 32 / na : 1, per = 32 / G;
    const int g = lane / G, l = lane - g * G, gsh = g * G < 32 ? g * G : 0;
    for (int k0 = 0; k0 < T; k0 += kCandBuf) {
        const int len = min(kCandBuf, T - k0);
        const bool last = k0 + len == T;
        verlet_stage(s, w, st, n, o, k0, len, lane);
        for (int ab = 0; ab < na; ab += per) {
            const bool on = g < per && ab + g < na;
            const int i = a0 + (on ? ab + g : 0);
            const float4 pi = s.pos_s[i];
            int *vrow = s.vnbr + (size_t)i * s.max_vnb;
            int cnt = k0 > 0 ? s.vnn[i] : 0;  // lane 0 of the group left it there
            __syncwarp();
            if (shifted) cnt = verlet_sweep<kImages, true>(s, w, i, pi, on, l, G, gsh, len, vrow, cnt);
            else cnt = verlet_sweep<kImages, false>(s, w, i, pi, on, l, G, gsh, len, vrow, cnt);
            if (on && l == 0) {
                if (last && cnt > s.max_vnb) set_err(s, kErrCapacity);
                s.vnn[i] = last ? min(cnt, s.max_vnb) : cnt;
            }
        }
        __syncwarp();  // the chunk is read (and the counts written) before the next is staged
    }
}

// End of a rebuild, run once by the last Verlet block to finish: the rows'
// box becomes the reference, and the flag is
// cleared for the next step (kept set when the skin is zero, so every step
// rebuilds).
__device__ __forceinline__ void finish_rebuild(const Sys &s, Blk k)
{
    __shared__ bool am_last;
    __syncthreads();
    if (threadIdx.x == 0) am_last = atomicAdd(&s.ticket[4], 1u) == (unsigned)k.nb - 1u;
    __syncthreads();
    if (!am_last || threadIdx.x != 0) return;
    s.ticket[4] = 0u;
    *s.rebuilds += 1ull;
    for (int a = 0; a < 3; ++a) s.Lref[a] = s.Lhi[a];
    *s.flag = s.always_rebuild ? 1 : 0;
}

// Grid-stride over cells, one warp per cell, so an idle launch (no rebuild)
// retires at once.
__device__ __forceinline__ void verlet(const Sys &s, Blk k)
{
    if (!*s.flag) return;
    __shared__ VerletWarpSmem sh[kVerletWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const bool images = s.nc[0] >= 3 && s.nc[1] >= 3 && s.nc[2] >= 3;
    const int warps = k.nb * kVerletWarps;
    for (int c = k.b * kVerletWarps + wid; c < s.ncell; c += warps) {
        if (images) verlet_cell<true>(s, sh[wid], c, lane);
        else verlet_cell<false>(s, sh[wid], c, lane);
    }
    finish_rebuild(s, k);
}

// Exact rows from the Verlet rows, when the CV kernel does not fuse it.
template <typename real>
__global__ void __launch_bounds__(kBlockAtoms) k_filter(Sys s)
{
    const int groups = group_grid(s.n);
    for (int blk = blockIdx.x; blk < groups; blk += gridDim.x) filter_row<real, kG>(s, atom_lane_at(s, blk));
}


// Single-system kernels of the rebuild chain.
template <bool kScan>
__global__ void __launch_bounds__(kBinThreads) k_bin_count(Sys s)
{
    chain_enter();
    bin_count<kScan>(s, own_blk());
}
__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(Sys s)
{
    chain_enter();
    scan_reduce(s, own_blk());
}
template <bool kDirect>
__global__ void __launch_bounds__(kScanThreads) k_scan_down(Sys s)
{
    chain_enter();
    scan_down<kDirect>(s, own_blk());
}
__global__ void k_bin_scatter(Sys s)
{
    chain_enter();
    bin_scatter(s, own_blk());
}
__global__ void k_cell_sort_gather(Sys s)
{
    chain_enter();
    cell_sort_gather(s, own_blk());
}
__global__ void __launch_bounds__(kBlockAtoms) k_verlet(Sys s)
{
    chain_enter();
    verlet(s, own_blk());
}

// The same kernels over every system of a batch.
__global__ void kb_gather_check(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    gather_check(s, k);
}
__global__ void kb_bin_count(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    bin_count<false>(s, k);
}
__global__ void __launch_bounds__(kScanThreads) kb_scan_reduce(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    scan_reduce(s, k);
}
__global__ void __launch_bounds__(kScanThreads) kb_scan_down(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    scan_down<false>(s, k);
}
__global__ void kb_bin_scatter(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    bin_scatter(s, k);
}
__global__ void kb_cell_sort_gather(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    cell_sort_gather(s, k);
}
__global__ void __launch_bounds__(kBlockAtoms) kb_verlet(BatchView v)
{
    chain_enter();
    Blk k;
    const Sys &s = v.sys[batch_system(v, k)];
    verlet(s, k);
}

// Pairs (i < j) in caller indices, for export: one thread per sorted atom,
// entries with caller(i) < caller(j) appended through one counter.  Each
// exact entry's j is read from its geometry tag.
template <typename real>
__global__ void k_export_pairs(Sys s, long long *pairs, int *count)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= s.n) return;
    int ui = s.perm[i];
    for (int k = 0; k < s.nn[i]; ++k) {
        Vec3<real> d;
        bool cn;
        int j;
        load_geo<real>(s, entry_slot(s, i, k), d, cn, j);
        int uj = s.perm[j];
        if (ui < uj) {
            int slot = atomicAdd(count, 1);
            pairs[2 * (size_t)slot] = ui;
            pairs[2 * (size_t)slot + 1] = uj;
        }
    }
}

// Sum and maximum of the per-atom neighbour counts.
__global__ void k_nn_stats(Sys s, unsigned long long *sum, int *mx)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int v = i < s.n ? s.nn[i] : 0;
    int m = v;
    unsigned long long t = (unsigned long long)v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        t += __shfl_xor_sync(0xffffffffu, t, o);
        m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(sum, t);
        atomicMax(mx, m);
    }
}

}  // namespace

// Grids of the rebuild chain are capped (grid-stride loops inside) so that
// the common no-rebuild step pays a few microseconds of launches.
constexpr int kRebuildGrid = 152 * 8;

inline int capped(int blocks) { return blocks < kRebuildGrid ? (blocks < 1 ? 1 : blocks) : kRebuildGrid; }

int grid_blocks(const Sys &s, int kind, int persist_cap)
{
    if (s.kind != kKindCoord) {  // no neighbour list: a CV block, an atom grid, hills
        switch (kind) {
        case GK_ONE: return 1;
        case GK_ATOM256: return (s.n + 255) / 256;
        case GK_HILLS: return bias_blocks(s.K);
        case GK_DEPOSIT: return s.deposit ? bias_blocks(s.K) : 0;
        }
        return 0;
    }
    switch (kind) {
    case GK_ATOM256: return (s.n + 255) / 256;
    case GK_ATOM256_CAP: return capped((s.n + 255) / 256);
    case GK_SCAN_TILES: return (s.ncell + kScanTile - 1) / kScanTile;
    case GK_GROUPS_CAP: {  // Verlet rows: a warp per cell, up to 16 blocks per SM
        const int g = (s.ncell + kVerletWarps - 1) / kVerletWarps;
        return g < kPersistBlocks ? g : kPersistBlocks;
    }
    case GK_ONE: return 1;
    case GK_GROUPS: {
        const int g = group_grid(s.n);
        return persist_cap > 0 && persist_cap < g ? persist_cap : g;
    }
    case GK_ROWS: {
        const int g = (s.n + kRowAtoms - 1) / kRowAtoms;
        return persist_cap > 0 && persist_cap < g ? persist_cap : g;
    }
    case GK_FORCE: {
        // with the virial its grid fixes the order of the virial's partials:
        // by N only, few enough for the last block to add
        const int g = force_grid(s.n, s.ncv, s.pairs);
        if (s.virial) return g < kVirialBlocks ? g : kVirialBlocks;
        return persist_cap > 0 && persist_cap < g ? persist_cap : g;
    }
    case GK_SUM: return sum_blocks(s.n);
    case GK_HILLS: return bias_blocks(s.K);
    case GK_DEPOSIT: return s.deposit ? bias_blocks(s.K) : 0;
    }
    return 0;
}

void launch_gather_check(const Sys &s, cudaStream_t st)
{
    chained_live(k_gather_check, grid_blocks(s, GK_ATOM256, 0), 256, st, s);
}

// The cell scan's kernels, fewer for small grids: none up to kScanOne cells
// (about 36,000 atoms), one up to kDirectTiles tiles (about 1.8 million).
// Adding up the tiles before its own, a block reads more the larger the grid: a
// step that rebuilds, one / two scan kernels, 100,000 atoms 108.4 / 109.5 us,
// 800,000 559 / 557, 1.6 million 1,084 / 1,081, 3 million 2,028 / 2,023; one that
// does not (nine in ten) is a launch shorter: 42.9 / 44.0, 158.5 / 159.9, 287.5 /
// 289.0, 522.0 / 523.5.  That passes the loss at all of these; the line bounds
// what the last tile reads (0.8 MB).
inline int scan_kernels(const Sys &s)
{
    return s.ncell <= kScanOne ? 0 : (grid_blocks(s, GK_SCAN_TILES, 0) <= kDirectTiles ? 1 : 2);
}

int rebuild_kernels(const Sys &s) { return 4 + scan_kernels(s); }

void launch_rebuild(const Sys &s, cudaStream_t st)
{
    const int scans = scan_kernels(s), tiles = grid_blocks(s, GK_SCAN_TILES, 0);
    chained(scans == 0 ? k_bin_count<true> : k_bin_count<false>, grid_blocks(s, GK_ATOM256_CAP, 0), kBinThreads, st, s);
    if (scans == 2) chained(k_scan_reduce, tiles, kScanThreads, st, s);
    if (scans > 0) chained(scans == 1 ? k_scan_down<true> : k_scan_down<false>, tiles, kScanThreads, st, s);
    chained(k_bin_scatter, grid_blocks(s, GK_ATOM256_CAP, 0), 256, st, s);
    chained(k_cell_sort_gather, grid_blocks(s, GK_ATOM256_CAP, 0), 256, st, s);
    chained(k_verlet, grid_blocks(s, GK_GROUPS_CAP, 0), kBlockAtoms, st, s);
}

void launch_batch_gather(const BatchView &v, int total, cudaStream_t st)
{
    if (total > 0) chained_live(kb_gather_check, total, 256, st, v);
}

void launch_batch_rebuild(const BatchView *rows, const int *totals, cudaStream_t st)
{
    chained(kb_bin_count, totals[GK_ATOM256_CAP], 256, st, rows[GK_ATOM256_CAP]);
    chained(kb_scan_reduce, totals[GK_SCAN_TILES], kScanThreads, st, rows[GK_SCAN_TILES]);
    chained(kb_scan_down, totals[GK_SCAN_TILES], kScanThreads, st, rows[GK_SCAN_TILES]);
    chained(kb_bin_scatter, totals[GK_ATOM256_CAP], 256, st, rows[GK_ATOM256_CAP]);
    chained(kb_cell_sort_gather, totals[GK_ATOM256_CAP], 256, st, rows[GK_ATOM256_CAP]);
    chained(kb_verlet, totals[GK_GROUPS_CAP], kBlockAtoms, st, rows[GK_GROUPS_CAP]);
}

void launch_filter(const Sys &s, int fp64, cudaStream_t st)
{
    if (fp64)
        k_filter<double><<<group_grid(s.n), kBlockAtoms, 0, st>>>(s);
    else
        k_filter<float><<<group_grid(s.n), kBlockAtoms, 0, st>>>(s);
}

void launch_nn_stats(const Sys &s, unsigned long long *sum, int *mx, cudaStream_t st)
{
    cudaMemsetAsync(sum, 0, sizeof(unsigned long long), st);
    cudaMemsetAsync(mx, 0, sizeof(int), st);
    k_nn_stats<<<(s.n + 255) / 256, 256, 0, st>>>(s, sum, mx);
}

void launch_export_pairs(const Sys &s, int fp64, long long *pairs, int *count, cudaStream_t st)
{
    cudaMemsetAsync(count, 0, sizeof(int), st);
    if (fp64)
        k_export_pairs<double><<<(s.n + 255) / 256, 256, 0, st>>>(s, pairs, count);
    else
        k_export_pairs<float><<<(s.n + 255) / 256, 256, 0, st>>>(s, pairs, count);
}


// The kernels of this file whose only argument is the system descriptor
// (a captured step's nodes of these can take new I/O buffers in place).
SysKernel sys_kernel_neighbors(const void *func)
{
    static const void *const io[] = {
        (const void *)k_gather_check,
        (const void *)k_bin_count<true>,
        (const void *)k_bin_count<false>,
        (const void *)k_cell_sort_gather,
    };
    static const void *const rest[] = {
        (const void *)k_scan_reduce,
        (const void *)k_scan_down<true>,
        (const void *)k_scan_down<false>,
        (const void *)k_bin_scatter,
        (const void *)k_verlet,
        (const void *)k_filter<float>,
        (const void *)k_filter<double>,
    };
    for (const void *k : io)
        if (k == func) return kSysIo;
    for (const void *k : rest)
        if (k == func) return kSysOnly;
    return kNotSys;
}

}  // namespace metad
