// Cell-list neighbor builder producing destination-sorted CSR edges.
//
// Atoms are folded into the cell, binned into cells at least r_list wide, sorted by cell
// (stable radix sort, so the internal numbering is deterministic) and renumbered in that
// order.  A warp takes a few centres of one cell and walks the surrounding cells twice -- a
// count pass and a fill pass with an in-warp prefix count that keeps candidates in traversal
// order -- so the edge list comes out grouped by destination with no atomics and a
// reproducible order.  A last pass finds, for every edge (i <- j, n), the slot of its reverse
// (j <- i, -n).
//
// The distance predicate is the paper's neighbor-set definition evaluated in double
// precision with explicit round-to-nearest adds and multiplies (no contraction into fused
// multiply-adds), which makes the edge set reproducible bit for bit.  The scans decide in
// single precision every candidate whose distance is further from the list radius than single
// precision can be wrong (Near), and evaluate that predicate for the others.
#include <cub/cub.cuh>
#include <thrust/iterator/transform_iterator.h>

#include <cmath>
#include <cstring>

#include "alloc.h"
#include "kernels.h"

namespace umd {

namespace {

struct Grid {
    double L[3];        // cell edge lengths (orthorhombic cells)
    double H[9];        // cell vectors as rows; H[3 k + k] = L[k] for an orthorhombic cell
    double Hinv[9];     // inverse of H (general cells): fractional coordinates f = r Hinv
    int tri;            // general cell: fold and bin in fractional coordinates
    double lo[3];       // binning origin (Cartesian; fractional when tri)
    double inv_cw[3];   // 1 / bin width (per unit of the binning coordinate)
    int nc[3];          // bins per direction
    int m[3];           // bin reach per direction
    int pbc[3];
    int ncell;          // bins in all
    int halves;         // 2 when ghost atoms are binned apart from owned ones (keys ncell .. 2 ncell - 1), else 1
    int n_owned;        // caller indices >= n_owned are ghosts
    int sorted;         // every periodic direction has at least 2 m + 1 bins: bins are visited in
                        // increasing bin index, so each row comes out sorted by neighbour index
};

// first offset of the walk over the 2 m + 1 bins around bin c of a direction: the one whose wrapped
// bin index is smallest, so that the walk (continuing cyclically) visits bins in increasing index
__device__ __forceinline__ int walk_start(int c, int m, int nc, int pbc, int sorted) {
    if (!sorted || !pbc) return -m;
    if (c - m < 0) return -c;
    if (c + m >= nc) return nc - c;
    return -m;
}

__device__ __forceinline__ int floor_div(int a, int b) {
    int q = a / b;
    if ((a % b != 0) && ((a < 0) != (b < 0))) --q;
    return q;
}

__device__ __forceinline__ int pack_shift(int nx, int ny, int nz) {
    return (nx & 0xff) | ((ny & 0xff) << 8) | ((nz & 0xff) << 16);
}

// order-preserving map of a double onto an unsigned integer, for atomicMin / atomicMax
__device__ __forceinline__ unsigned long long ordered_key(double x) {
    const long long b = __double_as_longlong(x);
    return b < 0 ? ~(unsigned long long)b : (unsigned long long)b | 0x8000000000000000ull;
}
inline double ordered_value(unsigned long long k) {
    const unsigned long long b = (k & 0x8000000000000000ull) ? (k & 0x7fffffffffffffffull) : ~k;
    double x;
    std::memcpy(&x, &b, sizeof(x));
    return x;
}
// smallest and largest binning coordinate of the atoms along each direction (Cartesian for an
// orthorhombic cell, fractional for a general one): keys[k] = min, keys[3 + k] = max
__global__ void k_bounds(int N, const double* __restrict__ pos, Grid g, unsigned long long* __restrict__ keys) {
    __shared__ unsigned long long smin[3][8], smax[3][8];
    unsigned long long mn[3] = {~0ull, ~0ull, ~0ull}, mx[3] = {0ull, 0ull, 0ull};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        const double x = pos[3 * (size_t)i], y = pos[3 * (size_t)i + 1], z = pos[3 * (size_t)i + 2];
        for (int k = 0; k < 3; ++k) {
            const double v = g.tri ? x * g.Hinv[k] + y * g.Hinv[3 + k] + z * g.Hinv[6 + k] : (k == 0 ? x : (k == 1 ? y : z));
            const unsigned long long key = ordered_key(v);
            if (key < mn[k]) mn[k] = key;
            if (key > mx[k]) mx[k] = key;
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = 0; k < 3; ++k) {
        for (int off = 16; off > 0; off >>= 1) {
            const unsigned long long a = __shfl_xor_sync(0xffffffffu, mn[k], off), b = __shfl_xor_sync(0xffffffffu, mx[k], off);
            if (a < mn[k]) mn[k] = a;
            if (b > mx[k]) mx[k] = b;
        }
        if (lane == 0) { smin[k][warp] = mn[k]; smax[k][warp] = mx[k]; }
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        const int k = threadIdx.x;
        unsigned long long a = smin[k][0], b = smax[k][0];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) { if (smin[k][w] < a) a = smin[k][w]; if (smax[k][w] > b) b = smax[k][w]; }
        atomicMin(keys + k, a);
        atomicMax(keys + 3 + k, b);
    }
}

// fold the position of atom i into the cell; its bin
__device__ __forceinline__ int fold_atom(int i, const double* __restrict__ pos, const Grid& g, double* wpos, int* img_o, int* __restrict__ err) {
    int c[3];
    bool bad = false;
    if (g.tri) {
        // general cell: f = r Hinv, fold by whole cell vectors along periodic directions (the same
        // arithmetic k_gather_positions applies later), bin by the folded fractional coordinate
        const double x = pos[3 * (size_t)i], y = pos[3 * (size_t)i + 1], z = pos[3 * (size_t)i + 2];
        if (!isfinite(x) || !isfinite(y) || !isfinite(z)) bad = true;
        double f[3], fl[3];
        for (int k = 0; k < 3; ++k) {
            f[k] = x * g.Hinv[k] + y * g.Hinv[3 + k] + z * g.Hinv[6 + k];
            fl[k] = g.pbc[k] ? floor(f[k]) : 0.0;
            if (fabs(fl[k]) > 1.0e6) bad = true;
            img_o[3 * (size_t)i + k] = bad ? 0 : (int)fl[k];
        }
        for (int k = 0; k < 3; ++k) {
            const double r = k == 0 ? x : (k == 1 ? y : z);
            wpos[3 * (size_t)i + k] = r - ((fl[0] * g.H[k] + fl[1] * g.H[3 + k]) + fl[2] * g.H[6 + k]);
            int ck = (int)floor(((f[k] - fl[k]) - g.lo[k]) * g.inv_cw[k]);
            ck = ck < 0 ? 0 : (ck >= g.nc[k] ? g.nc[k] - 1 : ck);
            c[k] = ck;
        }
    }
    for (int k = 0; k < 3 && !g.tri; ++k) {
        const double x = pos[3 * (size_t)i + k];
        if (!isfinite(x)) bad = true;
        double w = x;
        int fl = 0;
        if (g.pbc[k]) {
            const double frac = x / g.L[k];
            const double f = floor(frac);
            w = __dmul_rn(__dsub_rn(frac, f), g.L[k]);
            fl = (int)f;
            if (fabs(f) > 1.0e6) bad = true;
        }
        wpos[3 * (size_t)i + k] = w;
        img_o[3 * (size_t)i + k] = fl;
        int ck = (int)floor((w - g.lo[k]) * g.inv_cw[k]);
        ck = ck < 0 ? 0 : (ck >= g.nc[k] ? g.nc[k] - 1 : ck);
        c[k] = ck;
    }
    if (bad) {
        atomicOr(err, kErrNonFinite);
        c[0] = c[1] = c[2] = 0;
    }
    return (c[2] * g.nc[1] + c[1]) * g.nc[0] + c[0] + (i >= g.n_owned ? g.ncell : 0);
}
__global__ void k_fold_bin(int N, const double* __restrict__ pos, Grid g, double* __restrict__ wpos,
                           int* __restrict__ img_o, int* __restrict__ key, int* __restrict__ idx,
                           int* __restrict__ err) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    key[i] = fold_atom(i, pos, g, wpos, img_o, err);
    idx[i] = i;
}

// atom o as the i-th of the internal order
__device__ __forceinline__ void sorted_atom(int i, int o, const double* wpos, const int* img_o, const int* __restrict__ type,
                                            int* __restrict__ perm, double* __restrict__ xs0, double* __restrict__ xs, float4* __restrict__ rec,
                                            int* __restrict__ img, int* __restrict__ type_s) {
    perm[i] = o;
    type_s[i] = type[o];
    float hi[3];
    for (int k = 0; k < 3; ++k) {
        const double w = wpos[3 * (size_t)o + k];
        xs0[3 * (size_t)i + k] = w;
        xs[3 * (size_t)i + k] = w;
        img[3 * (size_t)i + k] = img_o[3 * (size_t)o + k];
        hi[k] = (float)w;
    }
    rec[i] = make_float4(hi[0], hi[1], hi[2], 0.f);   // what the scans read
}

// gather the per-atom arrays into sorted order; where the sorted key rises from one atom to the next,
// the cells in between start at the latter (a gap of more than four cells is filled by the whole warp)
__global__ void k_gather_sorted(int N, int nkeys, const int* __restrict__ skey, const int* __restrict__ sidx,
                                const double* __restrict__ wpos, const int* __restrict__ img_o, const int* __restrict__ type,
                                int* __restrict__ perm, double* __restrict__ xs0, double* __restrict__ xs,
                                float4* __restrict__ rec, int* __restrict__ img, int* __restrict__ type_s,
                                int* __restrict__ cell_start) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    int lo = 0, n = 0;                           // this atom's gap: cells lo .. lo + n - 1 start at atom i
    if (i <= N) {
        lo = i > 0 ? skey[i - 1] + 1 : 0;
        n = (i < N ? skey[i] : nkeys) - lo + 1;
    }
    if (n <= 4) for (int c = 0; c < n; ++c) cell_start[lo + c] = i;
    unsigned wide = __ballot_sync(0xffffffffu, n > 4);
    while (wide) {
        const int l = __ffs(wide) - 1;
        wide &= wide - 1;
        const int lo_l = __shfl_sync(0xffffffffu, lo, l), n_l = __shfl_sync(0xffffffffu, n, l), i_l = i - lane + l;
        for (int c = lane; c < n_l; c += 32) cell_start[lo_l + c] = i_l;
    }
    if (i >= N) return;
    sorted_atom(i, sidx[i], wpos, img_o, type, perm, xs0, xs, rec, img, type_s);
}

// Up to kBinTogether atoms: bins, their order and the sorted arrays by one block in one launch (fold, sort and gather as three
// took 3.5 + 6.1 + 4.9 us at 597 atoms, and the gaps between them).  Builds in us, together and apart: 108 atoms 94 and 100, 512 72 and
// 77, 1024 81 and 82; from two atoms per thread on the block's sort and its passes take longer than several blocks': 1500 atoms 100
// and 91, 4096 128 and 88, and 119 and 63 where most bins are empty.
constexpr int kBinTogether = 1024;
__global__ void __launch_bounds__(kBinTogether) k_bin_together(int N, int nkeys, int end_bit, const double* __restrict__ pos, Grid g,
                                                               const int* __restrict__ type, double* wpos, int* img_o,
                                                               int* __restrict__ skey, int* __restrict__ perm, double* __restrict__ xs0,
                                                               double* __restrict__ xs, float4* __restrict__ rec, int* __restrict__ img,
                                                               int* __restrict__ type_s, int* __restrict__ cell_start, int* __restrict__ err) {
    using Sort = cub::BlockRadixSort<int, kBinTogether, 1, int>;
    __shared__ union { typename Sort::TempStorage sort; int keys[kBinTogether]; } sh;
    const int i = threadIdx.x;
    int key[1] = {i < N ? fold_atom(i, pos, g, wpos, img_o, err) : nkeys}, idx[1] = {i};     // (what is no atom comes last: nkeys < 2^end_bit)
    Sort(sh.sort).Sort(key, idx, 0, end_bit);
    __syncthreads();                                  // (the folded positions of the block are there, the sort is done with its area)
    sh.keys[i] = key[0];
    if (i < N) {
        skey[i] = key[0];
        sorted_atom(i, idx[0], wpos, img_o, type, perm, xs0, xs, rec, img, type_s);
    }
    __syncthreads();
    for (int c = i; c <= nkeys; c += kBinTogether) {                            // first atom of every bin, and N
        int lo = 0, hi = N;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (sh.keys[mid] < c) lo = mid + 1;
            else hi = mid;
        }
        cell_start[c] = lo;
    }
}

// Up to kOffsetsTogether rows: row offsets from row lengths and all that the host waits for, by one block, which writes the results
// to the host's pinned memory itself (otherwise the scan's two launches, the flags' kernel, three clears and four copies).
// h_flags null: the totals alone.  Builds of 8192 and 8193 atoms, us: 142 and 165, 144 and 168 in an open box, 99 and 128 where most
// bins are empty.
constexpr int kOffsetsTogether = 8192;
__global__ void __launch_bounds__(1024) k_row_offsets(int N, int n_owned, const int* __restrict__ deg, eidx_t* __restrict__ row_ptr,
                                                      const int* __restrict__ type, int T, eidx_t* __restrict__ h_totals,
                                                      int* __restrict__ h_flags, int* __restrict__ h_err, int* __restrict__ err) {
    __shared__ eidx_t warp_sum[32];
    __shared__ int present[1024];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (N + 1023) / 1024, first = tid * per, last = min(first + per, N);
    present[tid] = 0;
    __syncthreads();
    eidx_t sum = 0;
    bool bad = false;
    for (int i = first; i < last; ++i) {
        sum += deg[i];
        if (h_flags) {
            const int t = type[i];
            if (t < 0 || t >= T) bad = true;
            else present[t] = 1;
        }
    }
    eidx_t upto = sum;                                // inclusive over the warp
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const eidx_t v = __shfl_up_sync(0xffffffffu, upto, off);
        if (lane >= off) upto += v;
    }
    if (lane == 31) warp_sum[warp] = upto;
    if (bad) atomicOr(err, kErrSpecies);
    __syncthreads();
    eidx_t at = upto - sum;
    for (int w = 0; w < warp; ++w) at += warp_sum[w];
    for (int i = first; i < last; ++i) {
        row_ptr[i] = at;
        if (i == n_owned) h_totals[1] = at;
        at += deg[i];
    }
    if (tid == 1023) { row_ptr[N] = at; h_totals[0] = at; }     // (the last thread's end is everyone's)
    if (h_flags) {
        for (int t = tid; t < T; t += 1024) h_flags[t] = present[t];
        if (tid == 0) *h_err = atomicExch(err, 0);
    }
}

// Squared list radius, its single-precision value, and a band around that outside of which a squared
// distance computed in single precision from rounded coordinates falls on the right side of it.
struct Near { double rl2; float mid, tol; };

// X bounds the magnitude of the coordinates.  With u = 2^-24 a rounded candidate is off by u X, its
// rounded image shift by u (2 X + r), their sum by u (X + r), the rounded centre by u X and the
// difference, near the list radius r, by u r: err = u (5 X + 3 r) in all.  The square sum is then off
// by 2 sqrt(3) r err + 3 err^2 and the rounding of products and sums, 8 u r^2; the band is twice that.
__host__ __device__ inline Near near_band(double r, double X) {
    const double u = 5.9604644775390625e-8, err = u * (5.0 * X + 3.0 * r);
    Near nr;
    nr.rl2 = r * r;
    nr.mid = (float)nr.rl2;
    const double tol = 2.0 * (3.4641016151377546 * r * err + 3.0 * err * err + 8.0 * u * r * r);
    nr.tol = tol < 1.0e30 ? (float)tol : 1.0e30f;
    return nr;
}

__device__ __forceinline__ bool exact_inside(const double* __restrict__ xj, double sx, double sy, double sz, double xi, double yi,
                                             double zi, double rl2) {
    const double ddx = __dsub_rn(__dadd_rn(xj[0], sx), xi), ddy = __dsub_rn(__dadd_rn(xj[1], sy), yi),
                 ddz = __dsub_rn(__dadd_rn(xj[2], sz), zi);
    return __dadd_rn(__dadd_rn(__dmul_rn(ddx, ddx), __dmul_rn(ddy, ddy)), __dmul_rn(ddz, ddz)) < rl2;
}
// component c of the shift vector n . H, built up one cell vector after another without fused
// multiply-add; for an orthorhombic cell all but one term of each component are exact zeros
__device__ __forceinline__ double image_shift(const Grid& g, int nx, int ny, int nz, int c) {
    return __dadd_rn(__dadd_rn(__dmul_rn((double)nz, g.H[6 + c]), __dmul_rn((double)ny, g.H[3 + c])), __dmul_rn((double)nx, g.H[c]));
}

// A warp takes G centres of one cell; its lanes are 32 candidates at a time, tested against all G
// centres (held in registers of every lane), so that the walk over the cells, the candidate loads
// and the loop around them are paid once per G centres.  The walk is cut into runs: bins that follow
// one another along x under the same image hold consecutive atoms.  The warp lays out 32 runs at a
// time, a lane each, and then goes through their candidates end to end, so that short runs leave no
// lane idle.  FILL = false: count the neighbours.  FILL = true: write them, in the order of the walk.
// Bound by instruction issue: nine instructions per centre and 32 candidates in the count pass,
// about twenty in the fill pass.
// SPREAD = false: the warps of a few blocks share a cell, and with it the candidates in L1.  SPREAD = true: a cell's atoms
// are cut into groups of G from its first atom on, and a warp takes the groups that start among `span` consecutive
// atoms of the internal order, so that there are N / span warps however the atoms are spread over the cells.
template <bool FILL, int G, bool SPREAD>
__global__ void __launch_bounds__(128) k_scan_cells(int N, int span, Grid g, Near nr, const int* __restrict__ skey,
                                                    const int* __restrict__ cell_start, const float4* __restrict__ rec,
                                                    const double* __restrict__ xs0, int* __restrict__ deg,
                                                    const eidx_t* __restrict__ row_ptr, int2* __restrict__ nbr, int* __restrict__ err) {
    struct Run { int end, first, code; float sx, sy, sz; };   // candidates before its end; atom of candidate 0; image
    __shared__ Run runs_s[4][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    Run* const runs = runs_s[warp];
    const unsigned lt_mask = (1u << lane) - 1u;
    const int wz = 2 * g.m[2] + 1, wy = 2 * g.m[1] + 1, wx = 2 * g.m[0] + 1;
    const int n_keys = g.halves * g.ncell;
    const int64_t span0 = SPREAD ? ((int64_t)blockIdx.x * n_warps + warp) * span : 0;
    int key_l = 0;
    unsigned todo = 0;                           // SPREAD: lanes whose atom starts a group
    if (SPREAD) {
        bool lead = false;
        if (lane < span && span0 + lane < N) {
            key_l = skey[span0 + lane];
            lead = ((int)span0 + lane - cell_start[key_l]) % G == 0;
        }
        todo = __ballot_sync(0xffffffffu, lead);
    }
    for (int key0 = blockIdx.x; SPREAD ? todo != 0 : key0 < n_keys; key0 += gridDim.x) {
    int first_i = 0;
    if (SPREAD) {
        const int l = __ffs(todo) - 1;
        todo &= todo - 1;
        first_i = (int)span0 + l;
        key0 = __shfl_sync(0xffffffffu, key_l, l);
    }
    const int c_end = cell_start[key0 + 1];
    if (!SPREAD) {
        first_i = cell_start[key0] + G * (warp + n_warps * blockIdx.y);
        if (first_i >= c_end) continue;
    }
    const int key = key0 < g.ncell ? key0 : key0 - g.ncell;         // a ghost's own bin
    const int cx = key % g.nc[0], cy = (key / g.nc[0]) % g.nc[1], cz = key / (g.nc[0] * g.nc[1]);
    const int sz0 = walk_start(cz, g.m[2], g.nc[2], g.pbc[2], g.sorted);
    const int sy0 = walk_start(cy, g.m[1], g.nc[1], g.pbc[1], g.sorted);
    const int sx0 = walk_start(cx, g.m[0], g.nc[0], g.pbc[0], g.sorted);
    // the walk along x, the same on every line of bins: the run at offset tx of the walk, and how far
    // it goes (a run that is off the grid of an open direction is empty)
    auto x_run = [&](int tx, int* xc, int* nx) {
        int dx = sx0 + tx;
        if (dx > g.m[0]) dx -= wx;
        *xc = cx + dx; *nx = 0;
        if (g.pbc[0]) {
            *nx = floor_div(*xc, g.nc[0]);
            *xc -= *nx * g.nc[0];
            return min(min(g.nc[0] - *xc, g.m[0] - dx + 1), wx - tx);
        }
        return *xc < 0 ? -*xc : min(max(g.nc[0] - *xc, 1), wx - tx);
    };
    int per_line = 0;
    for (int tx = 0, xc, nx; tx < wx; ++per_line) tx += x_run(tx, &xc, &nx);
    const int n_runs = wz * wy * per_line;
    for (int i0 = first_i; SPREAD ? i0 == first_i : i0 < c_end; i0 += G * n_warps * gridDim.y) {
    const int gn = min(G, c_end - i0);
    // lane k < G keeps centre k in double precision; every lane has all of them in single precision
    double xi = 0, yi = 0, zi = 0;
    if (lane < gn) { const double* x = xs0 + 3 * (size_t)(i0 + lane); xi = x[0]; yi = x[1]; zi = x[2]; }
    float fx[G], fy[G], fz[G];
    int cnt[G];                                  // FILL: next slot, counted from the first centre's row
#pragma unroll
    for (int k = 0; k < G; ++k) {
        fx[k] = __shfl_sync(0xffffffffu, lane < gn ? (float)xi : -3.0e18f, k);
        fy[k] = __shfl_sync(0xffffffffu, (float)yi, k); fz[k] = __shfl_sync(0xffffffffu, (float)zi, k);
        cnt[k] = FILL && k < gn ? (int)(row_ptr[i0 + k] - row_ptr[i0]) : 0;
    }
    int2* const out = FILL ? nbr + row_ptr[i0] : nullptr;
    // with ghosts the bins are walked twice, owned atoms first: ghosts follow every owned atom in
    // the internal order, so the row still ascends in the neighbour index
    for (int half = 0; half < g.halves; ++half)
    for (int r0 = 0; r0 < n_runs; r0 += 32) {
        int n = 0;
        Run my = {0, 0, 0, 0.f, 0.f, 0.f};
        if (r0 + lane < n_runs) {
            const int line = (r0 + lane) / per_line, seg = (r0 + lane) - line * per_line;
            int dz = sz0 + line / wy, dy = sy0 + line % wy;
            if (dz > g.m[2]) dz -= wz;
            if (dy > g.m[1]) dy -= wy;
            int zc = cz + dz, yc = cy + dy, xc = 0, nx = 0, ny = 0, nz = 0, run = 0;
            bool in = true;
            if (g.pbc[2]) { nz = floor_div(zc, g.nc[2]); zc -= nz * g.nc[2]; }
            else if (zc < 0 || zc >= g.nc[2]) in = false;
            if (g.pbc[1]) { ny = floor_div(yc, g.nc[1]); yc -= ny * g.nc[1]; }
            else if (yc < 0 || yc >= g.nc[1]) in = false;
            for (int q = 0, tx = 0; q <= seg; ++q) { tx += run; run = x_run(tx, &xc, &nx); }
            if (xc < 0 || xc >= g.nc[0]) in = false;
            if (in) {
                const int cell = (zc * g.nc[1] + yc) * g.nc[0] + xc + half * g.ncell;
                my.first = cell_start[cell];
                n = cell_start[cell + run] - my.first;
                my.code = pack_shift(nx, ny, nz);
                my.sx = (float)image_shift(g, nx, ny, nz, 0); my.sy = (float)image_shift(g, nx, ny, nz, 1);
                my.sz = (float)image_shift(g, nx, ny, nz, 2);
                if (nx < -127 || nx > 127 || ny < -127 || ny > 127 || nz < -127 || nz > 127) atomicOr(err, kErrShiftRange);
            }
        }
        my.end = n;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, my.end, off);
            if (lane >= off) my.end += v;
        }
        my.first -= my.end - n;
        const int total = __shfl_sync(0xffffffffu, my.end, 31);
        __syncwarp();
        runs[lane] = my;
        __syncwarp();
        int r = 0, j_next = 0, code_next = 0;
        float4 p_next = make_float4(3.0e18f, 0.f, 0.f, 0.f);
        auto fetch = [&](int f) {                // candidate f of these runs, its image applied
            p_next = make_float4(3.0e18f, 0.f, 0.f, 0.f);
            j_next = -1; code_next = 0;
            if (f < total) {
                while (f >= runs[r].end) ++r;
                j_next = runs[r].first + f;
                code_next = runs[r].code;
                p_next = __ldg(rec + j_next);
            }
        };
        fetch(lane);
        for (int f0 = 0; f0 < total; f0 += 32) {
            float4 p = p_next;
            const int j = j_next, code = code_next;
            if (code != 0) { p.x += runs[r].sx; p.y += runs[r].sy; p.z += runs[r].sz; }
            fetch(f0 + 32 + lane);
            auto distance = [&](int k) {         // squared, minus the squared list radius
                const float ddx = p.x - fx[k], ddy = p.y - fy[k], ddz = p.z - fz[k];
                return fmaf(ddx, ddx, fmaf(ddy, ddy, fmaf(ddz, ddz, -nr.mid)));
            };
            float closest = 1.0e30f;
            unsigned hit[G];
#pragma unroll
            for (int k = 0; k < G; ++k) {
                const float off = distance(k);
                closest = fminf(closest, fabsf(off));
                if (FILL) hit[k] = __ballot_sync(0xffffffffu, off < 0.f);
                else cnt[k] += off < 0.f;
            }
            if (__any_sync(0xffffffffu, closest <= nr.tol)) {
                const int nx = (int)(signed char)(code & 0xff), ny = (int)(signed char)((code >> 8) & 0xff), nz = (int)(signed char)((code >> 16) & 0xff);
                const double sx = image_shift(g, nx, ny, nz, 0), sy = image_shift(g, nx, ny, nz, 1), sz = image_shift(g, nx, ny, nz, 2);
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    const double xk = __shfl_sync(0xffffffffu, xi, k), yk = __shfl_sync(0xffffffffu, yi, k), zk = __shfl_sync(0xffffffffu, zi, k);
                    const bool in = j >= 0 && k < gn && exact_inside(xs0 + 3 * (size_t)j, sx, sy, sz, xk, yk, zk, nr.rl2);
                    if (FILL) hit[k] = __ballot_sync(0xffffffffu, in);
                    else cnt[k] += (int)in - (int)(distance(k) < 0.f);
                }
            }
            if (FILL) {
                const bool self = code == 0 && (unsigned)(j - i0) < (unsigned)G;    // no atom is its own neighbour
                if (__any_sync(0xffffffffu, self)) {
#pragma unroll
                    for (int k = 0; k < G; ++k) hit[k] &= ~__ballot_sync(0xffffffffu, self && j - i0 == k);
                }
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    if (!hit[k]) continue;
                    if ((hit[k] >> lane) & 1u) out[cnt[k] + __popc(hit[k] & lt_mask)] = make_int2(j, code);
                    cnt[k] += __popc(hit[k]);
                }
            }
        }
    }
    if (!FILL) {
#pragma unroll
        for (int k = 0; k < G; ++k) {
            const int v = __reduce_add_sync(0xffffffffu, cnt[k]);
            if (k < gn && lane == k) deg[i0 + k] = max(v - 1, 0);    // the walk meets the centre itself once (unless it is not a number)
        }
    }
    }
    }
}

// How the rows of a list are ordered, i.e. how the reverse of an edge is searched for.
//   kByIndex   ascending in the neighbour index, each neighbour at most once
//   kByBin     by the neighbour's bin counted across images (z, then y, then x), then by index:
//              boxes so small that a walk visits a bin under several images
//   kByImage   by image (z, then y, then x), then by index: batched frames
enum RowOrder { kByIndex = 0, kByBin = 1, kByImage = 2 };

// position of neighbour (s, n) in the order of a row
template <int ORDER>
__device__ __forceinline__ unsigned long long order_key(const Grid& g, const int* __restrict__ skey, int s, int n) {
    const int nx = (int)(signed char)(n & 0xff), ny = (int)(signed char)((n >> 8) & 0xff), nz = (int)(signed char)((n >> 16) & 0xff);
    unsigned long long k = 0;
    if (ORDER == kByBin) {
        int c = skey[s], half = 0;
        if (c >= g.ncell) { c -= g.ncell; half = 1; }
        // bins are counted from -m, fewer than 2^18 of them (127 images of at most 1024 bins)
        const int uz = c / (g.nc[0] * g.nc[1]) + nz * g.nc[2] + (1 << 17), uy = (c / g.nc[0]) % g.nc[1] + ny * g.nc[1] + (1 << 17),
                  ux = c % g.nc[0] + nx * g.nc[0] + (1 << 17);
        k = ((((unsigned long long)half << 18 | (unsigned)uz) << 18 | (unsigned)uy) << 18) | (unsigned)ux;
    } else {
        k = (((unsigned)(nz + 128) << 8 | (unsigned)(ny + 128)) << 8) | (unsigned)(nx + 128);
    }
    return k;
}

// rev[e] = slot of (j <- i, -n) for e = (i <- j, n); stays at the -1 it comes with when absent (can only
// happen for pairs whose two orientations round to opposite sides of the list radius).  Rows that
// ascend in the neighbour index are searched for the neighbours above the row's own index only: an
// edge and its reverse are each other's reverse, so one search fills both slots.
// Bound by the tag lookups of its uncoalesced probes (eight per search, one lane each): 1.11 ms when every
// edge was searched for, 0.65 now (59 M edges, rows of 273).
template <int ORDER>
__global__ void k_reverse_map(int N, Grid g, const int* __restrict__ skey, const eidx_t* __restrict__ row_ptr,
                              const int2* __restrict__ nbr, eidx_t* __restrict__ rev) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= N) return;
    const int i = warp;
    const eidx_t e0 = row_ptr[i];
    const int len = (int)(row_ptr[i + 1] - e0);
    for (int k = lane; k < len; k += 32) {
        const eidx_t e = e0 + k;
        const int2 js = nbr[e];
        const int j = js.x, s = js.y;
        if (ORDER == kByIndex && j <= i) continue;
        const int want = pack_shift(-(int)(signed char)(s & 0xff), -(int)(signed char)((s >> 8) & 0xff), -(int)(signed char)((s >> 16) & 0xff));
        const eidx_t f0 = row_ptr[j];
        const int flen = (int)(row_ptr[j + 1] - f0);
        const int2* row = nbr + f0;
        int lo = 0, hi = flen;                                 // offsets inside one row: no overflow
        unsigned long long target = 0;
        if constexpr (ORDER != kByIndex) target = order_key<ORDER>(g, skey, i, want);
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            const int2 at = row[mid];
            bool below = at.x < i;
            if constexpr (ORDER != kByIndex) {
                const unsigned long long km = order_key<ORDER>(g, skey, at.x, at.y);
                below = km < target || (km == target && below);
            }
            if (below) lo = mid + 1; else hi = mid;
        }
        if (lo < flen && row[lo].x == i && row[lo].y == want) {
            rev[e] = f0 + lo;
            if (ORDER == kByIndex) rev[f0 + lo] = e;
        }
    }
}

// ---- batched frames -------------------------------------------------------------------------
// fold the atoms of frame blockIdx.x into its cell, write positions, records, species, frame index; with an open
// direction the magnitude of the coordinates, and with it the band of the scans, is known only here (without a band
// every candidate was decided twice)
__global__ void k_batch_fold(FrameCell* __restrict__ frames, const double* __restrict__ pos,
                             const int* __restrict__ type, int T, double rc, double inv_q, double* __restrict__ xs, float4* __restrict__ rec,
                             int4* __restrict__ fix, int* __restrict__ type_s, int* __restrict__ frame_of, int* __restrict__ perm,
                             int* __restrict__ err) {
    __shared__ double far_s[32];
    FrameCell& fc = frames[blockIdx.x];
    double X = 0;                                // largest magnitude of a coordinate
    for (int i = fc.a0 + threadIdx.x; i < fc.a1; i += blockDim.x) {
        const double x = pos[3 * (size_t)i], y = pos[3 * (size_t)i + 1], z = pos[3 * (size_t)i + 2];
        bool bad = !isfinite(x) || !isfinite(y) || !isfinite(z);
        double fl[3];
        for (int k = 0; k < 3; ++k) {
            const double f = x * fc.Hinv[k] + y * fc.Hinv[3 + k] + z * fc.Hinv[6 + k];
            fl[k] = fc.pbc[k] ? floor(f) : 0.0;
            if (!(fabs(fl[k]) <= 1.0e6)) { bad = true; fl[k] = 0.0; }
        }
        float hi[3];
        int fx[3];
        for (int k = 0; k < 3; ++k) {
            const double r = k == 0 ? x : (k == 1 ? y : z);
            const double w = bad ? 0.0 : r - ((fl[0] * fc.H[k] + fl[1] * fc.H[3 + k]) + fl[2] * fc.H[6 + k]);
            xs[3 * (size_t)i + k] = w;
            X = fmax(X, fabs(w));
            hi[k] = (float)w;
            fx[k] = to_quanta(w, inv_q);
        }
        int t = type[i];
        if (t < 0 || t >= T) { atomicOr(err, kErrSpecies); t = 0; }
        if (bad) atomicOr(err, kErrNonFinite);
        rec[i] = make_float4(hi[0], hi[1], hi[2], 0.f);
        fix[i] = make_int4(fx[0], fx[1], fx[2], t);
        type_s[i] = t;
        frame_of[i] = blockIdx.x;
        perm[i] = i;
    }
    if (fc.pbc[0] && fc.pbc[1] && fc.pbc[2]) return;      // (bounded by the cell: the host has set the band)
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) X = fmax(X, __shfl_xor_sync(0xffffffffu, X, off));
    if ((threadIdx.x & 31) == 0) far_s[threadIdx.x >> 5] = X;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) X = fmax(X, far_s[w]);
        fc.near_tol = near_band(rc, X).tol;
    }
}

// One warp per centre: every atom of the centre's frame under every image within reach, in the
// order image (z slowest), then atom; the same predicate as the cell-list scan.  An image is left out
// when the planes that bound it along some cell vector are further than the cutoff from the centre.
template <bool FILL>
__global__ void k_batch_scan(int N, const FrameCell* __restrict__ frames, const int* __restrict__ frame_of, double rc,
                             const double* __restrict__ xs, const float4* __restrict__ rec, int* __restrict__ deg,
                             const eidx_t* __restrict__ row_ptr, int2* __restrict__ nbr) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= N) return;
    const int i = warp;
    const FrameCell& fc = frames[frame_of[i]];
    const double xi = xs[3 * (size_t)i], yi = xs[3 * (size_t)i + 1], zi = xs[3 * (size_t)i + 2];
    const double rl2 = rc * rc;
    const float mid = (float)rl2, tol = fc.near_tol;
    const unsigned lt_mask = (1u << lane) - 1u;
    const eidx_t base_out = FILL ? row_ptr[i] : 0;
    int count = 0;
    // image n along cell vector k can reach the centre for n in [lo, hi]: its atoms lie at fractional
    // coordinates [n, n + 1) (within rounding), the cutoff spans `reach` of them
    int lo[3], hi[3];
    for (int k = 0; k < 3; ++k) {
        const double f = xi * fc.Hinv[k] + yi * fc.Hinv[3 + k] + zi * fc.Hinv[6 + k];
        lo[k] = hi[k] = 0;
        if (fc.pbc[k]) {
            lo[k] = max(-fc.m[k], (int)floor(f - fc.reach[k]));
            hi[k] = min(fc.m[k], (int)floor(f + fc.reach[k]));
        }
    }
    for (int nz = lo[2]; nz <= hi[2]; ++nz) {
        const double szx = __dmul_rn((double)nz, fc.H[6]), szy = __dmul_rn((double)nz, fc.H[7]), szz = __dmul_rn((double)nz, fc.H[8]);
        for (int ny = lo[1]; ny <= hi[1]; ++ny) {
            const double syx = __dadd_rn(szx, __dmul_rn((double)ny, fc.H[3])), syy = __dadd_rn(szy, __dmul_rn((double)ny, fc.H[4])),
                         syz = __dadd_rn(szz, __dmul_rn((double)ny, fc.H[5]));
            for (int nx = lo[0]; nx <= hi[0]; ++nx) {
                const double sx = __dadd_rn(syx, __dmul_rn((double)nx, fc.H[0])), sy = __dadd_rn(syy, __dmul_rn((double)nx, fc.H[1])),
                             sz = __dadd_rn(syz, __dmul_rn((double)nx, fc.H[2]));
                const bool self_img = nx == 0 && ny == 0 && nz == 0;
                const float fx = (float)(xi - sx), fy = (float)(yi - sy), fz = (float)(zi - sz);
                // two candidates per lane and turn, both loaded before either is tested (one by one the tests in single
                // precision were no faster than in double: energies of four open frames of 16,000 atoms 5.6 ms, so 3.5)
                for (int b = fc.a0; b < fc.a1; b += 64) {
                    float4 p[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int j = b + 32 * h + lane;
                        p[h] = j < fc.a1 ? __ldg(rec + j) : make_float4(1.0e18f, 0.f, 0.f, 0.f);
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (b + 32 * h >= fc.a1) break;
                        const int j = b + 32 * h + lane;
                        const float ddx = p[h].x - fx, ddy = p[h].y - fy, ddz = p[h].z - fz;
                        const float off = fmaf(ddx, ddx, fmaf(ddy, ddy, ddz * ddz)) - mid;
                        bool ok = off < 0.f;
                        if (fabsf(off) <= tol) ok = j < fc.a1 && exact_inside(xs + 3 * (size_t)j, sx, sy, sz, xi, yi, zi, rl2);
                        const unsigned mask = __ballot_sync(0xffffffffu, ok && !(self_img && j == i));
                        if (FILL && ((mask >> lane) & 1u))
                            nbr[base_out + count + __popc(mask & lt_mask)] = make_int2(j, pack_shift(nx, ny, nz));
                        count += __popc(mask);
                    }
                }
            }
        }
    }
    if (!FILL && lane == 0) deg[i] = count;
}

// ---- export in caller numbering ------------------------------------------------------
__global__ void k_export_deg(int N, const int* __restrict__ perm, const eidx_t* __restrict__ row_ptr,
                             int* __restrict__ deg_o) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    deg_o[perm[i]] = (int)(row_ptr[i + 1] - row_ptr[i]);
    if (i == 0) deg_o[N] = 0;
}

__global__ void k_export_rows(int N, const int* __restrict__ perm, const eidx_t* __restrict__ row_ptr,
                              const int2* __restrict__ nbr, const int* __restrict__ row_ptr_o, int* __restrict__ src_o,
                              signed char* __restrict__ shift_o) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= N) return;
    const int i = warp, o = perm[i];
    const eidx_t e0 = row_ptr[i];
    const int n = (int)(row_ptr[i + 1] - e0), q0 = row_ptr_o[o];
    for (int k = lane; k < n; k += 32) {
        const int s = nbr[e0 + k].y;
        src_o[q0 + k] = perm[nbr[e0 + k].x];
        shift_o[3 * (size_t)(q0 + k)] = (signed char)(s & 0xff);
        shift_o[3 * (size_t)(q0 + k) + 1] = (signed char)((s >> 8) & 0xff);
        shift_o[3 * (size_t)(q0 + k) + 2] = (signed char)((s >> 16) & 0xff);
    }
}

// the same export restricted to the centres first .. first + n - 1 of the caller's numbering, with
// 64-bit row offsets (a list may hold more than 2^31 edges; a range of rows rarely does)
__global__ void k_export_deg_range(int N, int first, int n, const int* __restrict__ perm,
                                   const eidx_t* __restrict__ row_ptr, int* __restrict__ deg_o) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) deg_o[n] = 0;
    if (i >= N) return;
    const int o = perm[i] - first;
    if (o >= 0 && o < n) deg_o[o] = (int)(row_ptr[i + 1] - row_ptr[i]);
}

__global__ void k_export_rows_range(int N, int first, int n, const int* __restrict__ perm,
                                    const eidx_t* __restrict__ row_ptr, const int2* __restrict__ nbr,
                                    const long long* __restrict__ row_ptr_o,
                                    long long cap, int* __restrict__ src_o, signed char* __restrict__ shift_o) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= N) return;
    const int o = perm[warp] - first;
    if (o < 0 || o >= n) return;
    const eidx_t e0 = row_ptr[warp];
    const int len = (int)(row_ptr[warp + 1] - e0);
    const long long q0 = row_ptr_o[o];
    for (int k = lane; k < len; k += 32) {
        if (q0 + k >= cap) break;
        const int s = nbr[e0 + k].y;
        src_o[q0 + k] = perm[nbr[e0 + k].x];
        shift_o[3 * (size_t)(q0 + k)] = (signed char)(s & 0xff);
        shift_o[3 * (size_t)(q0 + k) + 1] = (signed char)((s >> 8) & 0xff);
        shift_o[3 * (size_t)(q0 + k) + 2] = (signed char)((s >> 16) & 0xff);
    }
}

struct WidenDeg {
    __host__ __device__ eidx_t operator()(int v) const { return (eidx_t)v; }
};

#define NB_CHECK(call)                                                              \
    do {                                                                            \
        cudaError_t e__ = (call);                                                   \
        if (e__ != cudaSuccess) {                                                   \
            *err = std::string(#call) + ": " + cudaGetErrorString(e__);             \
            return UMLMD_E_CUDA;                                                    \
        }                                                                           \
    } while (0)

}  // namespace

void neighbor_free(NeighborDev* nb) {
    void* ptrs[] = {nb->frames, nb->rec, nb->fix, nb->edge_fix, nb->edge_nbr, nb->wpos, nb->img, nb->perm, nb->type_s, nb->xs0, nb->xs, nb->row_ptr, nb->nbr, nb->rev, nb->key, nb->key2, nb->idx, nb->idx2, nb->cell_start, nb->deg,
                    nb->cub_tmp, nb->bounds};
    for (void* p : ptrs)
        dev_free(p);
    *nb = NeighborDev();
}

// The one synchronisation of a build: the edge counts come back, with whatever else the caller wants to
// know by then, and the edge arrays grow to hold the list.
static int read_totals(NeighborDev* nb, int N, int n_owned, const int* d_type, int* d_err, const BuildFetch* fetch, cudaStream_t st,
                       std::string* err) {
    if (N <= kOffsetsTogether) {
        k_row_offsets<<<1, 1024, 0, st>>>(N, n_owned, nb->deg, nb->row_ptr, d_type, fetch ? fetch->T : 0, nb->h_totals,
                                          fetch ? fetch->h_flags : nullptr, fetch ? fetch->h_err : nullptr, d_err);
        NB_CHECK(cudaGetLastError());
    } else {
        NB_CHECK(cudaMemsetAsync(nb->deg + N, 0, sizeof(int), st));
        size_t tmp_bytes = nb->cub_bytes;
        auto deg_wide = thrust::make_transform_iterator(static_cast<const int*>(nb->deg), WidenDeg());
        NB_CHECK(cub::DeviceScan::ExclusiveScan(nb->cub_tmp, tmp_bytes, deg_wide, nb->row_ptr, cub::Sum(), (eidx_t)0, N + 1, st));
        NB_CHECK(cudaMemcpyAsync(nb->h_totals, nb->row_ptr + N, sizeof(eidx_t), cudaMemcpyDeviceToHost, st));
        if (n_owned < N) NB_CHECK(cudaMemcpyAsync(nb->h_totals + 1, nb->row_ptr + n_owned, sizeof(eidx_t), cudaMemcpyDeviceToHost, st));
        if (fetch) {
            NB_CHECK(launch_species_present(N, d_type, fetch->T, fetch->d_flags, d_err, st));
            NB_CHECK(cudaMemcpyAsync(fetch->h_flags, fetch->d_flags, sizeof(int) * (size_t)fetch->T, cudaMemcpyDeviceToHost, st));
            NB_CHECK(cudaMemcpyAsync(fetch->h_err, d_err, sizeof(int), cudaMemcpyDeviceToHost, st));
            NB_CHECK(cudaMemsetAsync(d_err, 0, sizeof(int), st));
        }
    }
    NB_CHECK(cudaStreamSynchronize(st));
    const int64_t total = nb->h_totals[0];
    nb->E = total;
    nb->E_owned = n_owned < N ? nb->h_totals[1] : total;
    if (total > nb->E_cap) {
        int64_t c;
        nb->E_cap = 0;                           // (until all of them are there)
        c = 0; NB_CHECK(dev_ensure(&nb->nbr, &c, total, 1.1));
        c = 0; NB_CHECK(dev_ensure(&nb->rev, &c, total, 1.1));
        nb->E_cap = c;
    }
    if (nb->per_edge && N + total > 0x7fffffffLL) nb->per_edge = false;         // (more than the list can name: the coarse ones)
    if (nb->per_edge) {
        if (N + total > nb->edge_fix_cap) NB_CHECK(dev_ensure(&nb->edge_fix, &nb->edge_fix_cap, N + total, 1.1));
        if (total > nb->edge_nbr_cap) NB_CHECK(dev_ensure(&nb->edge_nbr, &nb->edge_nbr_cap, total, 1.1));
    }
    return UMLMD_OK;
}

int neighbor_launches(int64_t N, bool fetch) { return N <= kBinTogether ? 5 : (N <= kOffsetsTogether ? 6 : 5 + fetch); }

int neighbor_build(NeighborDev* nb, int64_t N64, int64_t n_owned64, const double* d_pos, const int32_t* d_type,
                   const double cell[9], const int pbc[3], double skin, double rc, int* d_err,
                   const BuildFetch* fetch, cudaStream_t st, std::string* err) {
    if (N64 > 0x7fff0000LL) { *err = "too many atoms for 32-bit indices"; return UMLMD_E_INVALID_ARG; }
    const int N = (int)N64;
    const int n_owned = n_owned64 < 0 || n_owned64 > N64 ? N : (int)n_owned64;
    const double r_list = rc + skin;
    nb->batch = false; nb->n_frames = 0; nb->frame_of = nullptr;
    Grid g;
    const double L[3] = {cell[0], cell[4], cell[8]};
    g.tri = 0;
    for (int k = 0; k < 9; ++k) { g.H[k] = cell[k]; g.Hinv[k] = 0; if (k % 4 != 0 && cell[k] != 0.0) g.tri = 1; }
    // perpendicular height of the cell along each cell vector (the edge length when orthorhombic)
    double height[3] = {L[0], L[1], L[2]};
    if (g.tri) {
        const double* h = cell;
        const double c00 = h[4] * h[8] - h[5] * h[7], c01 = h[5] * h[6] - h[3] * h[8], c02 = h[3] * h[7] - h[4] * h[6];
        const double det = h[0] * c00 + h[1] * c01 + h[2] * c02;
        const double scale = std::fabs(h[0]) + std::fabs(h[1]) + std::fabs(h[2]) + std::fabs(h[3]) + std::fabs(h[4]) +
                             std::fabs(h[5]) + std::fabs(h[6]) + std::fabs(h[7]) + std::fabs(h[8]);
        if (!(std::fabs(det) > 1e-12 * scale * scale * scale)) { *err = "singular cell"; return UMLMD_E_UNSUPPORTED_CELL; }
        const double id = 1.0 / det;
        g.Hinv[0] = c00 * id; g.Hinv[3] = c01 * id; g.Hinv[6] = c02 * id;
        g.Hinv[1] = (h[2] * h[7] - h[1] * h[8]) * id; g.Hinv[4] = (h[0] * h[8] - h[2] * h[6]) * id; g.Hinv[7] = (h[1] * h[6] - h[0] * h[7]) * id;
        g.Hinv[2] = (h[1] * h[5] - h[2] * h[4]) * id; g.Hinv[5] = (h[2] * h[3] - h[0] * h[5]) * id; g.Hinv[8] = (h[0] * h[4] - h[1] * h[3]) * id;
        for (int k = 0; k < 3; ++k)     // f_k = r . column k of Hinv: planes of constant f_k are 1 / |column| apart
            height[k] = 1.0 / std::sqrt(g.Hinv[k] * g.Hinv[k] + g.Hinv[3 + k] * g.Hinv[3 + k] + g.Hinv[6 + k] * g.Hinv[6 + k]);
    }
    // per-direction bounding interval for non-periodic directions (host reduction of a
    // device min/max would cost a sync as well; the list build synchronises anyway)
    // binning coordinate: Cartesian for an orthorhombic cell, fractional for a general one; `ext` is
    // the extent along it, `unit` the perpendicular length of one unit of it
    double lo[3] = {0, 0, 0}, ext[3] = {L[0], L[1], L[2]}, unit[3] = {1, 1, 1};
    if (g.tri) for (int k = 0; k < 3; ++k) { ext[k] = 1.0; unit[k] = height[k]; }
    if (!(pbc[0] && pbc[1] && pbc[2]) && N > 0) {
        // the extent of the atoms along the open directions, reduced on the device (six keys come back)
        if (!nb->bounds) { int64_t c = 0; NB_CHECK(dev_ensure(&nb->bounds, &c, 6)); }
        const unsigned long long init[6] = {~0ull, ~0ull, ~0ull, 0ull, 0ull, 0ull};
        unsigned long long keys[6];
        NB_CHECK(cudaMemcpyAsync(nb->bounds, init, sizeof(init), cudaMemcpyHostToDevice, st));
        int blocks = (N + 255) / 256;
        if (blocks > 1184) blocks = 1184;
        k_bounds<<<blocks, 256, 0, st>>>(N, d_pos, g, nb->bounds);
        NB_CHECK(cudaMemcpyAsync(keys, nb->bounds, sizeof(keys), cudaMemcpyDeviceToHost, st));
        NB_CHECK(cudaStreamSynchronize(st));
        for (int k = 0; k < 3; ++k) {
            if (pbc[k]) continue;
            const double mn = ordered_value(keys[k]), mx = ordered_value(keys[3 + k]);
            if (!std::isfinite(mn) || !std::isfinite(mx)) { *err = "non-finite position"; return UMLMD_E_NONFINITE; }
            lo[k] = mn; ext[k] = (mx - mn) + 1e-6 / unit[k];
        }
    }
    int64_t ncell = 1;
    bool coarse = false;                        // fewer bins than the list radius allows: two list radii wide or more
    const double rl_pad = r_list * (1.0 + 1e-9) + 1e-12;
    for (int k = 0; k < 3; ++k) {
        g.L[k] = L[k]; g.lo[k] = lo[k]; g.pbc[k] = pbc[k] ? 1 : 0;
        const double whole = std::floor(ext[k] * unit[k] / rl_pad);
        if (whole > 1024) coarse = true;
        int nc = whole > 1024 ? 1024 : (int)whole;
        // a periodic box of less than three list radii: bins of a half, third or quarter of the list
        // radius still give 2 m + 1 distinct bins (from 2.5, 2.33 and 2.25 list radii on), and with them
        // rows sorted by neighbour index
        if (pbc[k] && nc == 2)
            for (int q = 2; q <= 4; ++q) {
                const int fine = (int)std::floor(q * ext[k] * unit[k] / rl_pad);
                if (fine >= 2 * q + 1) { nc = fine; break; }
            }
        if (nc < 1) nc = 1;
        g.nc[k] = nc;
    }
    // keep the cell table modest relative to the atom count
    while ((int64_t)g.nc[0] * g.nc[1] * g.nc[2] > 8 * (int64_t)N + 64) {
        int kmax = 0;
        for (int k = 1; k < 3; ++k) if (g.nc[k] > g.nc[kmax]) kmax = k;
        if (g.nc[kmax] == 1) break;
        g.nc[kmax] = (g.nc[kmax] + 1) / 2;
        coarse = true;
    }
    for (int k = 0; k < 3; ++k) {
        const double cw = ext[k] / g.nc[k];
        g.inv_cw[k] = 1.0 / cw;
        g.m[k] = pbc[k] || g.nc[k] > 1 ? (int)std::ceil(r_list / (cw * unit[k])) : 0;
        if (!pbc[k] && g.m[k] > g.nc[k] - 1) g.m[k] = g.nc[k] - 1;
        if (g.m[k] > 127) { *err = "cell much smaller than the list radius (more than 127 images)"; return UMLMD_E_UNSUPPORTED_CELL; }
        ncell *= g.nc[k];
    }
    g.sorted = 1;
    for (int k = 0; k < 3; ++k)
        if (g.pbc[k] && g.nc[k] < 2 * g.m[k] + 1) g.sorted = 0;
    double X = 0;                               // bound of the coordinates' magnitude
    for (int c = 0; c < 3; ++c) {
        double v = 0;
        if (g.tri) for (int k = 0; k < 3; ++k) v += std::fmax(std::fabs(lo[k]), std::fabs(lo[k] + ext[k])) * std::fabs(cell[3 * k + c]);
        else v = std::fmax(std::fabs(lo[c]), std::fabs(lo[c] + ext[c]));
        X = std::fmax(X, v);
    }
    const Near nr = near_band(r_list, X);
    g.ncell = (int)ncell; g.n_owned = n_owned; g.halves = n_owned < N ? 2 : 1;
    const int64_t nkeys = (int64_t)g.halves * ncell;

    int images = 0;                             // the farthest along a cell vector
    for (int k = 0; k < 3; ++k) if (pbc[k]) images = std::max(images, (int)std::floor(r_list / height[k]) + 1);
    nb->N = N; nb->skin = skin; nb->r_list = r_list; nb->quantum = position_quantum(r_list); nb->n_owned = n_owned; nb->E_owned = 0;
    nb->per_edge = edge_records_needed(r_list, images);
    for (int k = 0; k < 3; ++k) { nb->L[k] = L[k]; nb->pbc[k] = pbc[k] ? 1 : 0; }
    for (int k = 0; k < 9; ++k) nb->H[k] = cell[k];
    nb->tri = g.tri;
    if (N == 0) { nb->E = 0; return UMLMD_OK; }

    // per-atom arrays (all sized from one capacity)
    if (N > nb->N_cap) {
        const int64_t need = N + 1;
        int64_t c;
        nb->N_cap = 0;
        c = 0; NB_CHECK(dev_ensure(&nb->wpos, &c, need * 3));
        c = 0; NB_CHECK(dev_ensure(&nb->xs0, &c, need * 3));
        c = 0; NB_CHECK(dev_ensure(&nb->xs, &c, need * 3));
        c = 0; NB_CHECK(dev_ensure(&nb->rec, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->fix, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->img, &c, need * 6));   // sorted-order and caller-order halves
        c = 0; NB_CHECK(dev_ensure(&nb->perm, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->type_s, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->row_ptr, &c, need + 1));
        c = 0; NB_CHECK(dev_ensure(&nb->key, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->key2, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->idx, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->idx2, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->deg, &c, need + 1));
        nb->N_cap = N;
    }
    NB_CHECK(dev_ensure(&nb->cell_start, &nb->ncell_cap, nkeys + 2));
    int* img_o = nb->img + 3 * (size_t)(N + 1);

    const int TB = 256;
    int end_bit = 1;
    while ((1LL << end_bit) < nkeys) ++end_bit;
    size_t need_tmp = 0, need_scan = 0;
    cub::DeviceRadixSort::SortPairs(nullptr, need_tmp, nb->key, nb->key2, nb->idx, nb->idx2, N, 0, end_bit, st);
    // row offsets are accumulated in 64 bits from the 32-bit row lengths
    auto deg_wide = thrust::make_transform_iterator(static_cast<const int*>(nb->deg), WidenDeg());
    cub::DeviceScan::ExclusiveScan(nullptr, need_scan, deg_wide, nb->row_ptr, cub::Sum(), (eidx_t)0, N + 1, st);
    size_t need_scan32 = 0;                     // the export scans into the caller's 32-bit row pointers
    cub::DeviceScan::ExclusiveSum(nullptr, need_scan32, nb->deg, (int*)nullptr, N + 1, st);
    if (need_scan32 > need_scan) need_scan = need_scan32;
    if (need_scan > need_tmp) need_tmp = need_scan;
    if (need_tmp > nb->cub_bytes) {
        if (nb->cub_tmp) dev_free(nb->cub_tmp);
        nb->cub_tmp = nullptr; nb->cub_bytes = 0;
        NB_CHECK(dev_malloc(&nb->cub_tmp, need_tmp + 256));
        nb->cub_bytes = need_tmp + 256;
    }
    if (N <= kBinTogether) {
        int bits = 1;
        while ((1LL << bits) <= nkeys) ++bits;           // (one key more: no atom)
        k_bin_together<<<1, kBinTogether, 0, st>>>(N, (int)nkeys, bits, d_pos, g, d_type, nb->wpos, img_o, nb->key2, nb->perm, nb->xs0, nb->xs, nb->rec,
                                       nb->img, nb->type_s, nb->cell_start, d_err);
    } else {
        k_fold_bin<<<(N + TB - 1) / TB, TB, 0, st>>>(N, d_pos, g, nb->wpos, img_o, nb->key, nb->idx, d_err);
        size_t tmp_bytes = nb->cub_bytes;
        NB_CHECK(cub::DeviceRadixSort::SortPairs(nb->cub_tmp, tmp_bytes, nb->key, nb->key2, nb->idx, nb->idx2, N,
                                                 0, end_bit, st));
        k_gather_sorted<<<N / TB + 1, TB, 0, st>>>(N, (int)nkeys, nb->key2, nb->idx2, nb->wpos, img_o, d_type, nb->perm, nb->xs0,
                                                  nb->xs, nb->rec, nb->img, nb->type_s, nb->cell_start);
    }
    // Eight centres per warp and a block of four warps per cell; below 16384 atoms, where the cells are
    // too few to fill the machine that way, two centres per warp and four blocks per cell (4000 atoms,
    // 125 cells: count and fill 19 + 24 us; with one block per cell they took 34 + 45).
    // Both are bound by instruction issue.  With one warp per centre and every test in double precision
    // 216,000 atoms with 273 neighbours took 1.21 + 1.49 ms, so 0.32 + 0.52.
    // Where cells hold more than their own warps take at a time, the groups of centres are spread over warps atom by
    // atom instead: in cells two list radii wide and more (coarse: a box mostly empty, in which a cluster of atoms
    // falls into a few cells; 200,000 atoms in a box of 5000 Angstrom build in 20 ms, by the cells' own warps in 604; 2000
    // in 400 Angstrom in 149 us, so 425), and in small systems of more than 32 atoms per cell (108 atoms in one cell 146 us,
    // so 265; 4000 of dense carbon 154, so 212, and 194, so 393, without periodicity).  Elsewhere the shared candidates win
    // (9000 atoms of water 194 us, spread 200), also in larger dense systems, whose cells are many (30,000 atoms of
    // carbon 287 us, spread 330).  Spans of eight atoms for eight centres, of one for two (no warp then has two groups).
    const bool few = N < 16384, apart = coarse || (few && N > 32 * nkeys);
    const int span = few ? 1 : 8;
    const dim3 scan_blocks(apart ? (unsigned)((N64 + span - 1) / span) : (unsigned)(nkeys < 148 * 64 ? nkeys : 148 * 64), !apart && few ? 4 : 1);
    const int scan_threads = apart ? 32 : 128;
    auto scan = apart ? (few ? k_scan_cells<false, 2, true> : k_scan_cells<false, 8, true>)
                       : (few ? k_scan_cells<false, 2, false> : k_scan_cells<false, 8, false>);
    scan<<<scan_blocks, scan_threads, 0, st>>>(N, span, g, nr, nb->key2, nb->cell_start, nb->rec, nb->xs0, nb->deg, nullptr, nullptr, d_err);
    int code = read_totals(nb, N, n_owned, d_type, d_err, fetch, st, err);
    if (code != UMLMD_OK) return code;
    if (nb->E > 0) {
        auto fill = apart ? (few ? k_scan_cells<true, 2, true> : k_scan_cells<true, 8, true>)
                           : (few ? k_scan_cells<true, 2, false> : k_scan_cells<true, 8, false>);
        fill<<<scan_blocks, scan_threads, 0, st>>>(N, span, g, nr, nb->key2, nb->cell_start, nb->rec, nb->xs0, nullptr, nb->row_ptr, nb->nbr, d_err);
        NB_CHECK(cudaMemsetAsync(nb->rev, 0xff, sizeof(eidx_t) * (size_t)nb->E, st));
        auto reverse = g.sorted ? k_reverse_map<kByIndex> : k_reverse_map<kByBin>;
        reverse<<<(N + TB / 32 - 1) / (TB / 32), TB, 0, st>>>(N, g, nb->key2, nb->row_ptr, nb->nbr, nb->rev);
    }
    NB_CHECK(cudaGetLastError());
    return UMLMD_OK;
}

int neighbor_export(NeighborDev* nb, int32_t* d_row_ptr, int32_t* d_src, int8_t* d_shift,
                    cudaStream_t st, std::string* err) {
    const int N = (int)nb->N;
    if (N == 0) {
        NB_CHECK(cudaMemsetAsync(d_row_ptr, 0, sizeof(int), st));
        return UMLMD_OK;
    }
    const int TB = 256;
    k_export_deg<<<(N + TB - 1) / TB, TB, 0, st>>>(N, nb->perm, nb->row_ptr, nb->deg);
    size_t tmp_bytes = nb->cub_bytes;
    NB_CHECK(cub::DeviceScan::ExclusiveSum(nb->cub_tmp, tmp_bytes, nb->deg, d_row_ptr, N + 1, st));
    const int wb = (N + TB / 32 - 1) / (TB / 32);
    if (nb->E > 0)
        k_export_rows<<<wb, TB, 0, st>>>(N, nb->perm, nb->row_ptr, nb->nbr, d_row_ptr, d_src,
                                         (signed char*)d_shift);
    NB_CHECK(cudaGetLastError());
    return UMLMD_OK;
}

int neighbor_build_batch(NeighborDev* nb, int n_frames, const int64_t* offsets, const double* cells, const int pbc[3],
                         const double* d_pos, const int32_t* d_type, int T, double rc, int* d_err, const BuildFetch* fetch,
                         cudaStream_t st, std::string* err) {
    const int64_t N = offsets[n_frames];
    std::vector<FrameCell> fr((size_t)n_frames);
    int images = 0;                             // the farthest along a cell vector
    for (int f = 0; f < n_frames; ++f) {
        FrameCell& c = fr[f];
        const double* H = cells + 9 * (size_t)f;
        for (int k = 0; k < 9; ++k) {
            if (!std::isfinite(H[k])) { *err = "non-finite cell in a frame"; return UMLMD_E_UNSUPPORTED_CELL; }
            c.H[k] = H[k];
            c.Hq[k] = to_quanta(H[k], 1.0 / position_quantum(rc));
        }
        const double cx[3] = {H[4] * H[8] - H[5] * H[7], H[5] * H[6] - H[3] * H[8], H[3] * H[7] - H[4] * H[6]};   // b x c
        const double cy[3] = {H[7] * H[2] - H[8] * H[1], H[8] * H[0] - H[6] * H[2], H[6] * H[1] - H[7] * H[0]};   // c x a
        const double cz[3] = {H[1] * H[5] - H[2] * H[4], H[2] * H[3] - H[0] * H[5], H[0] * H[4] - H[1] * H[3]};   // a x b
        const double det = H[0] * cx[0] + H[1] * cx[1] + H[2] * cx[2];
        double scale = 0;
        for (int k = 0; k < 9; ++k) scale = std::fmax(scale, std::fabs(H[k]));
        if (!(std::fabs(det) > 1e-12 * scale * scale * scale)) { *err = "singular cell in a frame"; return UMLMD_E_UNSUPPORTED_CELL; }
        const double* cr[3] = {cx, cy, cz};
        for (int k = 0; k < 3; ++k) {           // column k of the inverse = (cross product k) / det
            for (int r = 0; r < 3; ++r) c.Hinv[3 * r + k] = cr[k][r] / det;
            const double nrm = std::sqrt(cr[k][0] * cr[k][0] + cr[k][1] * cr[k][1] + cr[k][2] * cr[k][2]);
            const double height = std::fabs(det) / nrm;
            c.pbc[k] = pbc[k] ? 1 : 0;
            c.reach[k] = rc / height + 1e-6;
            c.m[k] = pbc[k] ? (int)std::ceil(rc / height) : 0;
            images = std::max(images, c.m[k]);
            if (c.m[k] > 127) { *err = "frame cell much smaller than the cutoff (more than 127 images)"; return UMLMD_E_UNSUPPORTED_CELL; }
        }
        // coordinates of a folded atom are bounded by the cell along periodic directions only (else see k_batch_fold)
        double X = 0;
        for (int k = 0; k < 9; ++k) X = std::fmax(X, std::fabs(H[k]));
        c.near_tol = pbc[0] && pbc[1] && pbc[2] ? near_band(rc, 3.0 * X).tol : 1.0e30f;
        c.a0 = (int)offsets[f]; c.a1 = (int)offsets[f + 1];
    }
    nb->N = N; nb->skin = 0; nb->r_list = rc; nb->quantum = position_quantum(rc); nb->tri = 1; nb->batch = true; nb->n_frames = n_frames;
    nb->per_edge = edge_records_needed(rc, images);
    for (int k = 0; k < 3; ++k) { nb->pbc[k] = pbc[k] ? 1 : 0; nb->L[k] = 0; }
    for (int k = 0; k < 9; ++k) nb->H[k] = 0;
    nb->E = 0;
    if (N == 0) return UMLMD_OK;
    if (N > nb->N_cap) {
        const int64_t need = N + 1;
        int64_t c;
        nb->N_cap = 0;
        // the same per-atom arrays as the cell-list build sizes (the two builds may alternate on one handle)
        c = 0; NB_CHECK(dev_ensure(&nb->wpos, &c, need * 3));
        c = 0; NB_CHECK(dev_ensure(&nb->xs0, &c, need * 3));
        c = 0; NB_CHECK(dev_ensure(&nb->xs, &c, need * 3));
        c = 0; NB_CHECK(dev_ensure(&nb->rec, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->fix, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->img, &c, need * 6));
        c = 0; NB_CHECK(dev_ensure(&nb->perm, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->type_s, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->row_ptr, &c, need + 1));
        c = 0; NB_CHECK(dev_ensure(&nb->key, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->key2, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->idx, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->idx2, &c, need));
        c = 0; NB_CHECK(dev_ensure(&nb->deg, &c, need + 1));
        nb->N_cap = N;
    }
    nb->frame_of = nb->key;                    // scratch of the cell-list build, free here
    NB_CHECK(dev_ensure(&nb->frames, &nb->frames_cap, (int64_t)n_frames));
    // (pageable memory: the call returns once the frames have been staged)
    NB_CHECK(cudaMemcpyAsync(nb->frames, fr.data(), sizeof(FrameCell) * (size_t)n_frames, cudaMemcpyHostToDevice, st));
    auto deg_wide = thrust::make_transform_iterator(static_cast<const int*>(nb->deg), WidenDeg());
    size_t need_scan = 0;
    cub::DeviceScan::ExclusiveScan(nullptr, need_scan, deg_wide, nb->row_ptr, cub::Sum(), (eidx_t)0, (int)N + 1, st);
    if (need_scan > nb->cub_bytes) {
        if (nb->cub_tmp) dev_free(nb->cub_tmp);
        nb->cub_tmp = nullptr; nb->cub_bytes = 0;
        NB_CHECK(dev_malloc(&nb->cub_tmp, need_scan + 256));
        nb->cub_bytes = need_scan + 256;
    }
    const int TB = 256;
    k_batch_fold<<<n_frames, TB, 0, st>>>(nb->frames, d_pos, d_type, T, rc, 1.0 / nb->quantum, nb->xs, nb->rec, nb->fix, nb->type_s, nb->frame_of, nb->perm, d_err);
    const int wb = (int)((N + TB / 32 - 1) / (TB / 32));
    k_batch_scan<false><<<wb, TB, 0, st>>>((int)N, nb->frames, nb->frame_of, rc, nb->xs, nb->rec, nb->deg, nullptr, nullptr);
    nb->n_owned = N;
    int code = read_totals(nb, (int)N, (int)N, nb->type_s, d_err, fetch, st, err);
    if (code != UMLMD_OK) return code;
    if (nb->E > 0) {
        k_batch_scan<true><<<wb, TB, 0, st>>>((int)N, nb->frames, nb->frame_of, rc, nb->xs, nb->rec, nullptr, nb->row_ptr, nb->nbr);
        NB_CHECK(cudaMemsetAsync(nb->rev, 0xff, sizeof(eidx_t) * (size_t)nb->E, st));
        k_reverse_map<kByImage><<<wb, TB, 0, st>>>((int)N, Grid(), nullptr, nb->row_ptr, nb->nbr, nb->rev);
    }
    NB_CHECK(cudaGetLastError());
    return UMLMD_OK;
}

int neighbor_export_rows(NeighborDev* nb, int64_t first, int64_t n, int64_t* d_row_ptr, int32_t* d_src,
                         int8_t* d_shift, int64_t cap, cudaStream_t st, std::string* err) {
    const int N = (int)nb->N;
    if (n == 0 || N == 0) {
        NB_CHECK(cudaMemsetAsync(d_row_ptr, 0, sizeof(int64_t), st));
        return UMLMD_OK;
    }
    const int TB = 256;
    k_export_deg_range<<<(N + TB - 1) / TB, TB, 0, st>>>(N, (int)first, (int)n, nb->perm, nb->row_ptr, nb->deg);
    auto deg_wide = thrust::make_transform_iterator(static_cast<const int*>(nb->deg), WidenDeg());
    size_t tmp_bytes = nb->cub_bytes;
    NB_CHECK(cub::DeviceScan::ExclusiveScan(nb->cub_tmp, tmp_bytes, deg_wide, reinterpret_cast<eidx_t*>(d_row_ptr), cub::Sum(),
                                            (eidx_t)0, (int)n + 1, st));
    if (cap > 0 && d_src && d_shift) {
        const int wb = (N + TB / 32 - 1) / (TB / 32);
        k_export_rows_range<<<wb, TB, 0, st>>>(N, (int)first, (int)n, nb->perm, nb->row_ptr, nb->nbr,
                                               reinterpret_cast<const long long*>(d_row_ptr), (long long)cap, d_src,
                                               (signed char*)d_shift);
    }
    NB_CHECK(cudaGetLastError());
    return UMLMD_OK;
}

}  // namespace umd
