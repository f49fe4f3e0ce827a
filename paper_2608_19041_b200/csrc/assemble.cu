// Force / virial / energy assembly and the velocity-Verlet update.
//
// Forces: each atom is written by exactly one warp, which sums, over the atom's own CSR
// row, the gradient of each edge minus the gradient of its reverse edge (the reverse-edge
// map turns the source-sorted view into a gather).  No floating-point atomics anywhere,
// sums in double, fixed order, so results are bitwise reproducible.
#include <atomic>
#include "kernels.h"

namespace umd {

namespace {

constexpr int kRedBlock = 256;
constexpr int kRedMaxBlocks = 1024;
constexpr int kReduceBlocks = 296;        // two per SM
static_assert(kReduceBlocks * 10 >= kRedMaxBlocks, "one scratch area serves both kinds of reduction");

// kicks = 0: none; 1: v += (dt/2) a; 2: the closing half kick of one step and the opening half kick of the next, one
// after the other exactly as two launches would
__device__ __forceinline__ double vv_kicks(double v, double c, double f, int kicks) {
    if (kicks >= 1) v = v + c * f;
    if (kicks == 2) v = v + c * f;
    return v;
}

// Current position of sorted atom i, given that of its caller's atom: minus the image offset found at the build, in double
// (a.xs) and as the edge kernels' record (a.fix); false for a position that is not finite.
__device__ __forceinline__ bool gather_position(const GatherArgs& a, int i, double x0, double x1, double x2) {
    const double pos[3] = {x0, x1, x2};
    const double n0 = (double)a.img[3 * (size_t)i], n1 = (double)a.img[3 * (size_t)i + 1], n2 = (double)a.img[3 * (size_t)i + 2];
    const double n[3] = {n0, n1, n2};
    bool finite = true;
    int fx[3];
    for (int k = 0; k < 3; ++k) {
        const double x = a.tri ? pos[k] - ((n0 * a.h[k] + n1 * a.h[3 + k]) + n2 * a.h[6 + k]) : pos[k] - n[k] * a.h[4 * k];
        if (!isfinite(x)) finite = false;
        a.xs[3 * (size_t)i + k] = x;
        fx[k] = to_quanta(x, a.inv_q);
    }
    const int t = a.type_s[i];
    a.fix[i] = make_int4(fx[0], fx[1], fx[2], a.species_slot ? a.species_slot[t] : t);
    return finite;
}
// whether sorted atom i has moved more than half the skin since the build
__device__ __forceinline__ bool moved_too_far(const GatherArgs& a, int i) {
    double d2 = 0;
    for (int k = 0; k < 3; ++k) {
        const double d = a.xs[3 * (size_t)i + k] - a.xs0[3 * (size_t)i + k];
        d2 += d * d;
    }
    return d2 > a.max_disp2;
}

// Force on the atom of one row, by a whole warp: every lane ends with all three components.
__device__ __forceinline__ void force_of_row(int row, const eidx_t* __restrict__ row_ptr, const eidx_t* __restrict__ rev,
                                             const float* __restrict__ g, double* f) {
    const int lane = threadIdx.x & 31;
    const eidx_t e0 = row_ptr[row];
    const int len = (int)(row_ptr[row + 1] - e0);
    double fx = 0, fy = 0, fz = 0;
    for (int k = lane; k < len; k += 32) {
        const eidx_t e = e0 + k;
        const float* a = g + 3 * (size_t)e;
        float bx = 0.f, by = 0.f, bz = 0.f;
        const eidx_t r = rev[e];
        if (r >= 0) { const float* b = g + 3 * (size_t)r; bx = b[0]; by = b[1]; bz = b[2]; }
        fx += (double)a[0] - (double)bx;
        fy += (double)a[1] - (double)by;
        fz += (double)a[2] - (double)bz;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        fx += __shfl_xor_sync(0xffffffffu, fx, off);
        fy += __shfl_xor_sync(0xffffffffu, fy, off);
        fz += __shfl_xor_sync(0xffffffffu, fz, off);
    }
    f[0] = fx; f[1] = fy; f[2] = fz;
}

// Per-atom share of the virial, one warp per atom over its own row: every directed edge gives half
// of -g_e (x) r_e to its centre and half to its neighbour, so atom i collects
// -1/2 sum_{e in row(i)} (g_e - g_rev(e)) (x) r_e (the reverse edge has the opposite vector).
// Edge vectors are recomputed in double from the positions of the last evaluation.
struct CellRowsA { double h[9]; };
__global__ void k_atom_virial(int N, const eidx_t* __restrict__ row_ptr, const int2* __restrict__ nbr,
                              const eidx_t* __restrict__ rev,
                              const float* __restrict__ g, const double* __restrict__ xs, CellRowsA H,
                              const int* __restrict__ perm, double* __restrict__ out) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= N) return;
    const eidx_t e0 = row_ptr[warp];
    const int len = (int)(row_ptr[warp + 1] - e0);
    const double xi = xs[3 * (size_t)warp], yi = xs[3 * (size_t)warp + 1], zi = xs[3 * (size_t)warp + 2];
    double w[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) w[k] = 0.0;
    for (int k = lane; k < len; k += 32) {
        const eidx_t e = e0 + k;
        const float* a = g + 3 * (size_t)e;
        double d[3] = {(double)a[0], (double)a[1], (double)a[2]};
        const eidx_t r = rev[e];
        if (r >= 0) { const float* b = g + 3 * (size_t)r; d[0] -= (double)b[0]; d[1] -= (double)b[1]; d[2] -= (double)b[2]; }
        const int j = nbr[e].x, s = nbr[e].y;
        const double nx = (double)(signed char)(s & 0xff), ny = (double)(signed char)((s >> 8) & 0xff),
                     nz = (double)(signed char)((s >> 16) & 0xff);
        const double* xj = xs + 3 * (size_t)j;
        const double rx = (xj[0] + ((nx * H.h[0] + ny * H.h[3]) + nz * H.h[6])) - xi;
        const double ry = (xj[1] + ((nx * H.h[1] + ny * H.h[4]) + nz * H.h[7])) - yi;
        const double rz = (xj[2] + ((nx * H.h[2] + ny * H.h[5]) + nz * H.h[8])) - zi;
#pragma unroll
        for (int p = 0; p < 3; ++p) { w[3 * p] += d[p] * rx; w[3 * p + 1] += d[p] * ry; w[3 * p + 2] += d[p] * rz; }
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) w[k] += __shfl_xor_sync(0xffffffffu, w[k], off);
    }
    if (lane < 9) {
        double v = 0.0;
#pragma unroll
        for (int k = 0; k < 9; ++k) if (lane == k) v = w[k];
        out[9 * (size_t)perm[warp] + lane] = -0.5 * v;
    }
}

// Records of the edges of a row, a warp per row: edge vectors in double, rounded to quanta.  An edge beyond the cutoff, whose vector
// may be longer than the quanta reach, is put just outside it.  frames: of a batched list, whose cells differ (null: the cell H).
struct CellRows { double h[9]; };
__global__ void k_edge_records(int n_rows, int N, const eidx_t* __restrict__ row_ptr, const int2* __restrict__ nbr, const double* __restrict__ xs,
                               const int4* __restrict__ fix, CellRows cell, const FrameCell* __restrict__ frames, const int* __restrict__ frame_of,
                               double inv_q, double far, int4* __restrict__ out, int2* __restrict__ out_nbr) {
    chain_begin();
    const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (row >= n_rows) return;
    double H[9];
    for (int k = 0; k < 9; ++k) H[k] = frames ? frames[frame_of[row]].H[k] : cell.h[k];
    if (lane == 0) out[row] = make_int4(0, 0, 0, fix[row].w);
    const eidx_t e1 = row_ptr[row + 1];
    for (eidx_t e = row_ptr[row] + lane; e < e1; e += 32) {
        const int2 js = nbr[e];
        const int s = js.y;
        const int nx = (int)(signed char)(s & 0xff), ny = (int)(signed char)((s >> 8) & 0xff), nz = (int)(signed char)((s >> 16) & 0xff);
        double r[3];
        for (int k = 0; k < 3; ++k)
            r[k] = (xs[3 * (size_t)js.x + k] + ((nx * H[k] + ny * H[3 + k]) + nz * H[6 + k])) - xs[3 * (size_t)row + k];
        const bool near = r[0] * r[0] + r[1] * r[1] + r[2] * r[2] < far * far;
        out[N + e] = make_int4(to_quanta(near ? r[0] : far, inv_q), near ? to_quanta(r[1], inv_q) : 0, near ? to_quanta(r[2], inv_q) : 0, fix[js.x].w);
        out_nbr[e] = make_int2((int)(N + e), 0);
    }
}

__global__ void k_unsort_rows(int N, const int* __restrict__ perm, const float* __restrict__ in, int stride,
                              int width, float* __restrict__ out) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= N) return;
    const float* r = in + (size_t)warp * stride;
    float* w = out + (size_t)perm[warp] * width;
    for (int k = lane; k < width; k += 32) w[k] = r[k];
}

// flags[t] = 1 for every species that occurs (flags cleared by the caller); an index outside
// [0, T) is reported in the error word
__global__ void k_species_present(int64_t N, const int* __restrict__ type, int T, int* __restrict__ flags,
                                  int* __restrict__ err) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int t = type[i];
    if (t < 0 || t >= T) atomicOr(err, kErrSpecies);
    else if (flags[t] == 0) flags[t] = 1;
}

__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    double s = 0;
    if (threadIdx.x == 0) for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sh[w];
    return s;   // valid in thread 0
}

// Sums of K values over the threads of a block, in thread 0 .. K - 1's return value (sum of value
// threadIdx.x); sh holds K doubles per warp.  Lanes by butterfly, then warps in order.
template <int K>
__device__ __forceinline__ double block_sums(double* v, double* sh) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], off);
        if (lane == 0) sh[wid * K + k] = v[k];
    }
    __syncthreads();
    double s = 0;
    if (threadIdx.x < K) for (int w = 0; w < nw; ++w) s += sh[w * K + threadIdx.x];
    return s;
}

// Rows of a batched evaluation, a warp each: the force on the row's atom (caller order is internal order) and, when asked
// (row_virial), the nine sums of g (x) r over its edges, edge vectors recomputed in double from the positions and the
// frame's cell.  With the virial in the reduction by frame, a block each, 64 frames of 54 to 108 atoms took 6.7 + 15 us.
__global__ void k_frame_rows(int N, const eidx_t* __restrict__ row_ptr, const eidx_t* __restrict__ rev, const int2* __restrict__ nbr,
                             const float* __restrict__ g, const double* __restrict__ xs, const FrameCell* __restrict__ frames,
                             const int* __restrict__ frame_of, double* __restrict__ out, double* __restrict__ row_virial, int* __restrict__ err) {
    chain_begin();
    const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (row >= N) return;
    if (out) {
        double f[3];
        force_of_row(row, row_ptr, rev, g, f);
        if (lane < 3) {
            const double mine = lane == 0 ? f[0] : (lane == 1 ? f[1] : f[2]);
            out[3 * (size_t)row + lane] = mine;
            if (!isfinite(mine)) atomicOr(err, kErrNonFinite);
        }
    }
    if (!row_virial) return;
    const double* const H = frames[frame_of[row]].H;
    const double xi = xs[3 * (size_t)row], yi = xs[3 * (size_t)row + 1], zi = xs[3 * (size_t)row + 2];
    double v[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    const eidx_t e1 = row_ptr[row + 1];
    for (eidx_t k = row_ptr[row] + lane; k < e1; k += 32) {
        const int2 js = nbr[k];
        const int j = js.x, s = js.y;
        const int nx = (int)(signed char)(s & 0xff), ny = (int)(signed char)((s >> 8) & 0xff), nz = (int)(signed char)((s >> 16) & 0xff);
        const double r[3] = {(xs[3 * (size_t)j] + ((nx * H[0] + ny * H[3]) + nz * H[6])) - xi,
                             (xs[3 * (size_t)j + 1] + ((nx * H[1] + ny * H[4]) + nz * H[7])) - yi,
                             (xs[3 * (size_t)j + 2] + ((nx * H[2] + ny * H[5]) + nz * H[8])) - zi};
        const double gg[3] = {(double)g[3 * (size_t)k], (double)g[3 * (size_t)k + 1], (double)g[3 * (size_t)k + 2]};
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) v[3 * a + b] += gg[a] * r[b];
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], off);
        if (lane == k) row_virial[9 * (size_t)row + k] = v[k];
    }
}

// Segmented reduction of a batched evaluation: block f sums the atomic energies of frame f, which go to e_out (may be null) on
// the way, and, when asked, its rows' virials, in a fixed order.
constexpr int kFrameBlock = 256;
__global__ void __launch_bounds__(kFrameBlock) k_frame_reduce(const FrameCell* __restrict__ frames, const double* __restrict__ e_atom,
                                                              double* __restrict__ e_out, const double* __restrict__ row_virial,
                                                              double* __restrict__ out, int* __restrict__ err) {
    __shared__ double sh[kFrameBlock / 32 * 10];
    chain_begin();
    const FrameCell& fc = frames[blockIdx.x];
    double v[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int i = fc.a0 + threadIdx.x; i < fc.a1; i += kFrameBlock) {
        const double e = e_atom[i];
        v[0] += e;
        if (e_out) e_out[i] = e;
        if (row_virial) {
#pragma unroll
            for (int k = 0; k < 9; ++k) v[1 + k] += row_virial[9 * (size_t)i + k];
        }
    }
    const double s = block_sums<10>(v, sh);
    if (threadIdx.x < 10) {
        if (!isfinite(s)) atomicOr(err, kErrNonFinite);
        out[10 * (size_t)blockIdx.x + threadIdx.x] = threadIdx.x ? -s : s;
    }
}

// Energy and virial of an evaluation: out[0] = sum of the atomic energies, out[1 + k] = -sum of the k-th
// component of the virial partials; e_out (may be null) receives the atomic energies in the caller's
// numbering on the way.  Each of n_blocks blocks sums a strided share of both arrays; the last block of the grid
// to finish adds up their sums in order, so the result does not depend on which one it is.  h_out / h_err
// (pinned host memory, may be null) get the results and the error word, which is then cleared: a caller
// that waits for this call needs no copies.
struct ReduceArgs {
    const double* e_atom; int N; const int* perm; double* e_out;
    const double* vpart; int n_vpart;
    double* part; unsigned* done; double* out; int* err; double* h_out; int* h_err;
    int n_blocks;
};
__device__ __forceinline__ void reduce_share(const ReduceArgs& a, int block, double* sh) {
    double v[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    const int first = block * kRedBlock + threadIdx.x, step = a.n_blocks * kRedBlock;
    for (int i = first; i < a.N; i += step) {
        const double e = a.e_atom[i];
        v[0] += e;
        if (a.e_out) a.e_out[a.perm[i]] = e;
    }
    for (int i = first; i < a.n_vpart; i += step) {
#pragma unroll
        for (int k = 0; k < 9; ++k) v[1 + k] += a.vpart[(size_t)i * 9 + k];
    }
    const double s = block_sums<10>(v, sh);
    if (threadIdx.x < 10) a.part[(size_t)block * 10 + threadIdx.x] = s;
}
__device__ __forceinline__ void reduce_finish(const ReduceArgs& a, double* sh, bool* last) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) *last = atomicAdd(a.done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!*last) return;
    __threadfence();
    double v[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int i = threadIdx.x; i < a.n_blocks; i += kRedBlock) {
#pragma unroll
        for (int k = 0; k < 10; ++k) v[k] += __ldcg(a.part + (size_t)i * 10 + k);
    }
    const double t = block_sums<10>(v, sh);
    if (threadIdx.x == 0 && !isfinite(t)) atomicOr(a.err, kErrNonFinite);
    if (threadIdx.x < 10) {
        const double r = threadIdx.x ? -t : t;
        a.out[threadIdx.x] = r;
        if (a.h_out) a.h_out[threadIdx.x] = r;
    }
    if (threadIdx.x == 0) {
        *a.done = 0;
        if (a.h_err) *a.h_err = atomicExch(a.err, 0);
    }
}

// Energies alone, and larger systems.  Bound by latency (128,000 atoms, 32,000 partials of 72 bytes: 9.6 us; 108 atoms: 8.3 us.  One block per
// component behind a pass over the energies took 28 and 11 us, and a copy of the energies 2.5 more).
__global__ void __launch_bounds__(kRedBlock) k_reduce(const ReduceArgs a) {
    __shared__ double sh[kRedBlock / 32 * 10];
    __shared__ bool last;
    chain_begin();
    reduce_share(a, blockIdx.x, sh);
    reduce_finish(a, sh, &last);
}

// The forces of eight rows per block; REDUCE: the first n_blocks blocks of the grid reduce energy and virial instead.  In an
// MD run (t.pos given) the row's warp goes on with what is local to its atom: the kicks and the drift of velocity Verlet, with
// the arithmetic of k_vv, and after a drift the records of the next evaluation, with that of the gather.  As launches of
// their own the reduction took 8 us, kick and drift 4.4 and the gather 3.6 of the 135 us that a step of 4000 atoms took.
// REDUCE up to kReduceTogether atoms: it costs every block a fence and an atomic, which from there on is more than a launch
// (40,009 atoms 45.5 us together, 31 + 14 apart; 64,000 of dense carbon 145, 116 + 14).
constexpr int kReduceTogether = 32768;
template <bool REDUCE>
__global__ void __launch_bounds__(kRedBlock) k_assemble(int N, const eidx_t* __restrict__ row_ptr, const eidx_t* __restrict__ rev,
                                                        const float* __restrict__ g, const int* __restrict__ perm,
                                                        double* __restrict__ out, int* __restrict__ err, const ReduceArgs a, const StepTail t) {
    __shared__ double sh[kRedBlock / 32 * 10];
    __shared__ bool last;
    chain_begin();
    if (REDUCE && (int)blockIdx.x < a.n_blocks) {
        reduce_share(a, blockIdx.x, sh);
    } else {
        const int row = (int)(blockIdx.x - (REDUCE ? a.n_blocks : 0)) * (kRedBlock / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
        if (row < N) {
            double v[3];
            force_of_row(row, row_ptr, rev, g, v);
            const int o = perm[row];
            const double mine = lane == 0 ? v[0] : (lane == 1 ? v[1] : v[2]);
            if (lane < 3) {
                out[3 * (size_t)o + lane] = mine;
                if (!isfinite(mine)) atomicOr(err, kErrNonFinite);
            }
            if (t.pos) {
                // (of the positions that this step has evaluated: the next ones may be binned anew first)
                if (lane == 0 && moved_too_far(t.gather, row)) atomicOr(err, kErrStale);
                const int type = t.gather.type_s[row];
                double x = 0;
                if (lane < 3) {
                    const size_t at = 3 * (size_t)o + lane;
                    x = t.pos[at];
                    double u = t.vel[at];
                    u = vv_kicks(u, 0.5 * t.dt * kAccelUnit * t.inv_mass[type], mine, t.kicks);
                    t.vel[at] = u;
                    if (t.drift) { x += t.dt * u; t.pos[at] = x; }
                }
                if (t.drift) {
                    const double x0 = __shfl_sync(0xffffffffu, x, 0), x1 = __shfl_sync(0xffffffffu, x, 1), x2 = __shfl_sync(0xffffffffu, x, 2);
                    if (lane == 0 && !gather_position(t.gather, row, x0, x1, x2)) atomicOr(err, kErrNonFinite);
                }
            }
        }
    }
    if (REDUCE) reduce_finish(a, sh, &last);
}

__global__ void k_gather_positions(int N, const int* __restrict__ perm, const double* __restrict__ pos, const GatherArgs a, int* __restrict__ err) {
    chain_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const size_t o = 3 * (size_t)perm[i];
    if (!gather_position(a, i, pos[o], pos[o + 1], pos[o + 2])) atomicOr(err, kErrNonFinite);
    else if (moved_too_far(a, i)) atomicOr(err, kErrStale);
}

// kicks: see vv_kicks; drift: x += dt v after them; scale (may be null): the thermostat's velocity factor, applied first
__global__ void k_vv(int64_t N, double* __restrict__ pos, double* __restrict__ vel, const double* __restrict__ force,
                     const int* __restrict__ type, const double* __restrict__ inv_mass, double dt, int kicks, bool drift,
                     const double* __restrict__ scale) {
    chain_begin();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double c = 0.5 * dt * kAccelUnit * inv_mass[type[i]];
    const double sc = scale ? *scale : 1.0;
    for (int k = 0; k < 3; ++k) {
        const double f = force[3 * i + k];
        double v = vel[3 * i + k];
        if (scale) v *= sc;
        v = vv_kicks(v, c, f, kicks);
        vel[3 * i + k] = v;
        if (drift) pos[3 * i + k] += dt * v;
    }
}

// Nose-Hoover chain of kNhcChain thermostats (Martyna-Tuckerman-Klein form): `halves` successive
// half-step propagations of the chain given the current kinetic energy; leaves the product of the
// velocity scale factors and the kinetic energy after scaling.  One thread: the chain is a handful
// of scalars.  st = [eta[M], v_eta[M], scale, kinetic energy]
__device__ void propagate_chain(double* __restrict__ st, double ke, int halves, const NhcParams& p) {
    constexpr int M = kNhcChain;
    double* eta = st;
    double* v = st + M;
    double ke2 = 2.0 * ke;
    double scale = 1.0;
    const double d2 = p.dt_half, d4 = 0.5 * d2, d8 = 0.25 * d2;
    for (int h = 0; h < halves; ++h) {
        double G = (p.Q[M - 2] * v[M - 2] * v[M - 2] - p.kT) / p.Q[M - 1];
        v[M - 1] += G * d4;
        for (int k = M - 2; k >= 0; --k) {
            const double e = exp(-v[k + 1] * d8);
            G = (k == 0 ? (ke2 - p.dof * p.kT) : (p.Q[k - 1] * v[k - 1] * v[k - 1] - p.kT)) / p.Q[k];
            v[k] = (v[k] * e + G * d4) * e;
        }
        const double sfac = exp(-v[0] * d2);
        scale *= sfac;
        ke2 *= sfac * sfac;
        for (int k = 0; k < M; ++k) eta[k] += v[k] * d2;
        for (int k = 0; k < M - 1; ++k) {
            const double e = exp(-v[k + 1] * d8);
            G = (k == 0 ? (ke2 - p.dof * p.kT) : (p.Q[k - 1] * v[k - 1] * v[k - 1] - p.kT)) / p.Q[k];
            v[k] = (v[k] * e + G * d4) * e;
        }
        G = (p.Q[M - 2] * v[M - 2] * v[M - 2] - p.kT) / p.Q[M - 1];
        v[M - 1] += G * d4;
    }
    st[2 * M] = scale;
    st[2 * M + 1] = 0.5 * ke2;
}

// The closing half kick of a thermostatted step (kick), the kinetic energy after it and the chain's
// propagation, in one launch: blocks sum a strided share, the last one to finish adds up the blocks'
// sums in their order and propagates the chain.  Latency-bound: 9.0 us at 128,000 atoms (kick, sum in two
// passes and chain as four launches took 6.8 + 14.3 + 2.6 + 3.6 us at 216,000).
__global__ void __launch_bounds__(kRedBlock) k_kick_thermostat(int64_t N, double* __restrict__ vel, const double* __restrict__ force,
                                                               const int* __restrict__ type, const double* __restrict__ mass,
                                                               const double* __restrict__ inv_mass, double dt, bool kick,
                                                               double* __restrict__ part, unsigned* __restrict__ done,
                                                               double* __restrict__ st, int halves, NhcParams p) {
    __shared__ double sh[kRedBlock / 32];
    __shared__ bool last;
    chain_begin();
    double v[1] = {0};
    for (int64_t i = (int64_t)blockIdx.x * kRedBlock + threadIdx.x; i < N; i += (int64_t)gridDim.x * kRedBlock) {
        const int t = type[i];
        double u[3];
        const double c = 0.5 * dt * kAccelUnit * inv_mass[t];
        for (int k = 0; k < 3; ++k) {
            u[k] = vel[3 * i + k];
            if (kick) { u[k] = u[k] + c * force[3 * i + k]; vel[3 * i + k] = u[k]; }
        }
        v[0] += 0.5 * mass[t] * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]) / kAccelUnit;
    }
    const double s = block_sums<1>(v, sh);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = s;
        __threadfence();
        last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    v[0] = 0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += kRedBlock) v[0] += __ldcg(part + i);
    const double ke = block_sums<1>(v, sh);
    if (threadIdx.x == 0) {
        *done = 0;
        propagate_chain(st, ke, halves, p);
    }
}

__global__ void __launch_bounds__(kRedBlock) k_ke_slices(const double* __restrict__ vel, const int* __restrict__ type,
                                                         const double* __restrict__ mass, int64_t N, int64_t chunk,
                                                         double* __restrict__ part) {
    __shared__ double sh[kRedBlock / 32];
    const int64_t lo = (int64_t)blockIdx.x * chunk;
    const int64_t hi = lo + chunk < N ? lo + chunk : N;
    double v = 0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += kRedBlock) {
        const double vx = vel[3 * i], vy = vel[3 * i + 1], vz = vel[3 * i + 2];
        v += 0.5 * mass[type[i]] * (vx * vx + vy * vy + vz * vz) / kAccelUnit;
    }
    const double s = block_sum(v, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

__global__ void __launch_bounds__(kRedBlock) k_sum_small(const double* __restrict__ part, int n, double* out) {
    __shared__ double sh[kRedBlock / 32];
    double v = 0;
    for (int i = threadIdx.x; i < n; i += kRedBlock) v += part[i];
    const double s = block_sum(v, sh);
    if (threadIdx.x == 0) *out = s;
}

inline void slices(int64_t N, int* blocks, int64_t* chunk) {
    int64_t b = (N + 1023) / 1024;       // four atoms per thread, up to the 1024 partials there is room for
    if (b < 1) b = 1;
    if (b > kRedMaxBlocks) b = kRedMaxBlocks;
    *blocks = (int)b;
    *chunk = (N + b - 1) / b;
}

}  // namespace

int reduce_scratch_doubles(int64_t) { return kReduceBlocks * 10; }      // (more than kRedMaxBlocks)

cudaError_t launch_atom_virial(const NeighborDev& nb, const float* g, double* d_out, cudaStream_t st) {
    const int N = (int)nb.N;
    if (N == 0) return cudaSuccess;
    CellRowsA H;
    for (int k = 0; k < 9; ++k) H.h[k] = nb.H[k];
    k_atom_virial<<<(N + 7) / 8, 256, 0, st>>>(N, nb.row_ptr, nb.nbr, nb.rev, g, nb.xs, H, nb.perm, d_out);
    return cudaGetLastError();
}

cudaError_t launch_frame_rows(const NeighborDev& nb, const float* g, double* d_force, double* row_virial, int* d_err, cudaStream_t st) {
    const int N = (int)nb.N;
    if (N == 0 || (!d_force && !row_virial)) return cudaSuccess;
    return launch_chained(k_frame_rows, (N + 7) / 8, 256, 0, st, N, nb.row_ptr, nb.rev, nb.nbr, g, nb.xs, nb.frames, nb.frame_of, d_force,
                          row_virial, d_err);
}

cudaError_t launch_frame_reduce(const NeighborDev& nb, const double* e_atom, double* d_atom_energy, const double* row_virial, double* d_out,
                                int* d_err, cudaStream_t st) {
    if (nb.n_frames <= 0) return cudaSuccess;
    return launch_chained(k_frame_reduce, nb.n_frames, kFrameBlock, 0, st, nb.frames, e_atom, d_atom_energy, row_virial, d_out, d_err);
}

static ReduceArgs reduce_args(const NeighborDev& nb, const double* e_atom, double* d_atom_energy, const double* virial_part, int n_part,
                              double* scratch, unsigned* counter, double* out, int* d_err, double* h_out, int* h_err) {
    const int N = (int)nb.N, blocks = (N + 4 * kRedBlock - 1) / (4 * kRedBlock);
    return {e_atom, N, nb.perm, d_atom_energy, virial_part, n_part, scratch, counter, out, d_err, h_out, h_err,
            blocks < 1 ? 1 : (blocks < kReduceBlocks ? blocks : kReduceBlocks)};
}

cudaError_t launch_reduce_energy_virial(const NeighborDev& nb, const double* e_atom, double* d_atom_energy, const double* virial_part,
                                        int n_part, double* scratch, unsigned* counter, double* out, int* d_err, double* h_out,
                                        int* h_err, cudaStream_t st) {
    const ReduceArgs a = reduce_args(nb, e_atom, d_atom_energy, virial_part, n_part, scratch, counter, out, d_err, h_out, h_err);
    return launch_chained(k_reduce, a.n_blocks, kRedBlock, 0, st, a);
}

int assemble_launches(int64_t N) { return N <= kReduceTogether ? 1 : 2; }
cudaError_t launch_assemble(const NeighborDev& nb, const float* g, double* d_force, const StepTail& tail,
                            const double* e_atom, double* d_atom_energy, const double* virial_part, int n_part, double* scratch,
                            unsigned* counter, double* out, int* d_err, double* h_out, int* h_err, cudaStream_t st) {
    const int N = (int)nb.N;
    const ReduceArgs a = reduce_args(nb, e_atom, d_atom_energy, virial_part, n_part, scratch, counter, out, d_err, h_out, h_err);
    const int rows = (N + kRedBlock / 32 - 1) / (kRedBlock / 32);
    if (N <= kReduceTogether)
        return launch_chained(k_assemble<true>, a.n_blocks + rows, kRedBlock, 0, st, N, nb.row_ptr, nb.rev, g, nb.perm, d_force, d_err, a, tail);
    const cudaError_t e = launch_chained(k_assemble<false>, rows, kRedBlock, 0, st, N, nb.row_ptr, nb.rev, g, nb.perm, d_force, d_err, a, tail);
    return e != cudaSuccess ? e : launch_chained(k_reduce, a.n_blocks, kRedBlock, 0, st, a);
}

GatherArgs gather_args(const NeighborDev& nb, const int* species_slot) {
    const double half = 0.5 * nb.skin;
    GatherArgs a;
    a.img = nb.img; a.xs0 = nb.xs0; a.type_s = nb.type_s; a.species_slot = species_slot; a.xs = nb.xs; a.fix = nb.fix;
    for (int k = 0; k < 9; ++k) a.h[k] = nb.H[k];
    a.tri = nb.tri; a.inv_q = 1.0 / nb.quantum;
    // a tiny slack keeps a fresh build with zero skin from tripping on its own rounding
    a.max_disp2 = half * half + 1e-20;
    return a;
}

cudaError_t launch_gather_positions(const NeighborDev& nb, const double* d_pos, const int* species_slot, int* d_err, cudaStream_t st) {
    const int N = (int)nb.N;
    if (N == 0) return cudaSuccess;
    return launch_chained(k_gather_positions, (N + 255) / 256, 256, 0, st, N, nb.perm, d_pos, gather_args(nb, species_slot), d_err);
}

cudaError_t launch_edge_records(const NeighborDev& nb, double rc, cudaStream_t st) {
    const int N = (int)nb.n_owned;
    if (N == 0) return cudaSuccess;
    CellRows cell;
    for (int k = 0; k < 9; ++k) cell.h[k] = nb.H[k];
    return launch_chained(k_edge_records, (N + 7) / 8, 256, 0, st, N, (int)nb.N, nb.row_ptr, nb.nbr, nb.xs, nb.fix, cell,
                          nb.batch ? nb.frames : nullptr, nb.frame_of, 1.0 / position_quantum(kEdgeRecordReach * rc), kEdgeRecordReach * rc,
                          nb.edge_fix, nb.edge_nbr);
}

cudaError_t launch_unsort_state(const NeighborDev& nb, const float* in, int stride, int width, float* out,
                                cudaStream_t st) {
    const int N = (int)nb.N;
    if (N == 0) return cudaSuccess;
    k_unsort_rows<<<(N + 7) / 8, 256, 0, st>>>(N, nb.perm, in, stride, width, out);
    return cudaGetLastError();
}

cudaError_t launch_species_present(int64_t N, const int* type, int T, int* d_flags, int* d_err, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(d_flags, 0, sizeof(int) * T, st);
    if (e != cudaSuccess || N == 0) return e;
    k_species_present<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(N, type, T, d_flags, d_err);
    return cudaGetLastError();
}

cudaError_t launch_vv_kick_drift(int64_t N, double* pos, double* vel, const double* force, const int* type,
                                 const double* inv_mass, double dt, int kicks, bool drift, const double* d_scale,
                                 cudaStream_t st) {
    if (N == 0) return cudaSuccess;
    return launch_chained(k_vv, (unsigned)((N + 255) / 256), 256, 0, st, N, pos, vel, force, type, inv_mass, dt, kicks, drift, d_scale);
}

cudaError_t launch_kick_thermostat(int64_t N, double* vel, const double* force, const int* type, const double* mass,
                                   const double* inv_mass, double dt, bool kick, double* scratch, unsigned* counter, double* d_state,
                                   int halves, const NhcParams& p, cudaStream_t st) {
    const int64_t blocks = (N + 2 * kRedBlock - 1) / (2 * kRedBlock);
    return launch_chained(k_kick_thermostat, (unsigned)(blocks < 1 ? 1 : (blocks < kReduceBlocks ? blocks : kReduceBlocks)), kRedBlock, 0, st,
                          N, vel, force, type, mass, inv_mass, dt, kick, scratch, counter, d_state, halves, p);
}

cudaError_t launch_kinetic_energy(int64_t N, const double* vel, const int* type, const double* mass,
                                  double* scratch, double* out, cudaStream_t st) {
    int blocks; int64_t chunk;
    slices(N, &blocks, &chunk);
    k_ke_slices<<<blocks, kRedBlock, 0, st>>>(vel, type, mass, N, chunk, scratch);
    k_sum_small<<<1, kRedBlock, 0, st>>>(scratch, blocks, out);
    return cudaGetLastError();
}

}  // namespace umd

// ---------------------------------------------------------------------------------------
// Kinetic energy without any allocation (see umlmd_kinetic_energy_static in umlmd.h).
//
// Same two kernels as launch_kinetic_energy; the only difference is where the per-block
// partial sums live: in a fixed array inside this library's device image instead of
// workspace obtained from cudaMalloc.
// ---------------------------------------------------------------------------------------
namespace umd {
namespace {

constexpr int64_t kStaticMaxAtoms = (int64_t)kRedMaxBlocks * 4096;      // 4,194,304
constexpr int kMaxDevices = 64;

// Partial sums of one reduction (8 KB).  Every GPU that loads the library holds a copy
// until the process exits.
static __device__ __align__(256) double g_static_partials[kRedMaxBlocks];

// g_static_partials is only a host-side handle in host code; the device address has to be
// asked for, once per device, with that device current.  The cached addresses are atomics: two
// host threads may make the first call on a device at the same time (both resolve the same
// address).  They belong to the device's primary context: after cudaDeviceReset they are stale,
// which the header states.
std::atomic<double*> g_static_partials_dev[kMaxDevices];
thread_local char g_static_err[256] = "";

int static_fail(int code, const char* msg) {
    snprintf(g_static_err, sizeof(g_static_err), "%s", msg);
    return code;
}

}  // namespace
}  // namespace umd

extern "C" int umlmd_kinetic_energy_static(int64_t N, const double* d_vel, const int32_t* d_type,
                                           const double* d_mass_per_type, double* d_e_kin, void* stream) {
    using namespace umd;
    if (N < 0 || !d_e_kin || (N > 0 && (!d_vel || !d_type || !d_mass_per_type)))
        return static_fail(UMLMD_E_INVALID_ARG, "umlmd_kinetic_energy_static: null pointer or negative atom count");
    if (N > kStaticMaxAtoms) {
        char msg[200];
        snprintf(msg, sizeof(msg), "umlmd_kinetic_energy_static: %lld atoms exceed the fixed scratch limit of %lld",
                 (long long)N, (long long)kStaticMaxAtoms);
        return static_fail(UMLMD_E_CAPACITY, msg);
    }
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
        return static_fail(UMLMD_E_CUDA, "umlmd_kinetic_energy_static: no current CUDA device");
    double* partials = g_static_partials_dev[dev].load(std::memory_order_acquire);
    if (!partials) {
        double* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress((void**)&p, g_static_partials);
        if (e != cudaSuccess || !p) {
            char msg[200];
            snprintf(msg, sizeof(msg), "umlmd_kinetic_energy_static: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
            return static_fail(UMLMD_E_CUDA, msg);
        }
        g_static_partials_dev[dev].store(p, std::memory_order_release);
        partials = p;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // every partial that the final pass reads is written by the first pass of the same call,
    // so nothing left over from an earlier call needs clearing
    cudaError_t e = launch_kinetic_energy(N, d_vel, d_type, d_mass_per_type, partials, d_e_kin, st);
    if (e != cudaSuccess) {
        char msg[200];
        snprintf(msg, sizeof(msg), "umlmd_kinetic_energy_static: launch failed: %s", cudaGetErrorString(e));
        return static_fail(UMLMD_E_CUDA, msg);
    }
    return UMLMD_OK;
}

extern "C" const char* umlmd_static_last_error(void) { return umd::g_static_err; }
