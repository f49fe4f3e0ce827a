// Fused per-edge kernels: edge featurisation + per-destination aggregation (forward) and
// the recomputing edge backward pass that returns dE/dr_ij for every edge.
//
// One warp owns one destination atom and walks its contiguous CSR interval, 32 listed edges
// at a time: each lane computes the geometry of one edge (displacement from fixed-point
// positions, regularised length, direction, cutoff envelope, table row) and the edges inside
// the cutoff are queued in shared memory.  Full batches of queued edges are then processed
// with lanes split over channels -- a group of lanes handles one edge, each lane holding one
// or two runs of four consecutive channels, so table and pair-cache reads are 16-byte vector
// loads that a group issues as contiguous segments -- followed by a lane-per-edge phase for
// the degree >= 1 blocks.  The S+2 sums live in registers and are written once per
// destination; nothing per-edge is stored in the forward pass.  The backward pass recomputes
// the per-edge quantities, contracts them with dE/d(sums) and writes one 3-vector per edge; the
// virial is accumulated in the same pass.  The two passes read different tables of one cubic
// interpolant (the forward pass quadratic pieces of its values, the backward pass its own pieces with
// derivatives or, from C0 = 32 on, quadratic pieces of the derivative of envelope times
// amplitude): energy and force agree to the tables' rounding (common.cuh, value_piece), not exactly.
//
// Harmonics are evaluated with |u|^2 set to one; the regularised direction differs from a
// unit vector by eps^2/rho^2, far below single precision.
#include "kernels.h"

namespace umd {

namespace {

// A block is done when its slowest row is: with fewer rows per block fewer finished warps sit on
// registers and shared memory waiting for it (measured at eight / four / two warps per block, 131072
// atoms of the 64-species workload: backward 1.535 / 1.487 / 1.479 ms, forward 1.318 / 1.301 / 1.294 ms;
// four keeps the per-block virial partials at a quarter of the atom count).
constexpr int kWarpsPerBlock = kEdgeRowsPerBlock;
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float4 ldg4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }

// the part of a row of *len edges from *e0 on that warp w takes, where the warps of a block share a row
__device__ __forceinline__ void quarter_of_row(int w, eidx_t* e0, int* len) {
    const int first = (int)((int64_t)*len * w / kWarpsPerBlock), last = (int)((int64_t)*len * (w + 1) / kWarpsPerBlock);
    *e0 += first;
    *len = last - first;
}

struct Geom {
    float dx, dy, dz, rho, inv_rho, ux, uy, uz, chi, dchi, t;
    int row, pair;
    bool valid;
};

// phase 1: one lane, one edge
// c: record of the destination; Hf: cell of its frame in a batched evaluation (rows, in quanta), null for a single system.
// The edge vector is a difference of integers (common.cuh, position_quantum).  With float pairs, two 16-byte loads and an
// addition in double per component, this phase was half of what the narrow kernels sent through the L1 data pipe (32 scattered
// 16-byte loads are 32 of its wavefronts) and a quarter of their instructions.
// VALUE: row and offset in the value table, else in the table with derivatives
template <bool VALUE>
__device__ __forceinline__ Geom edge_geometry(const EdgeArgs& a, eidx_t e, bool in_range, const int4& c, int ti,
                                              const int* __restrict__ Hf) {
    Geom g;
    g.valid = false;
    g.dx = g.dy = g.dz = 0.f; g.rho = 1.f; g.inv_rho = 1.f; g.ux = g.uy = g.uz = 0.f;
    g.chi = 0.f; g.dchi = 0.f; g.t = 0.f; g.row = 0; g.pair = 0;
    if (!in_range) return g;
    const int2 js = a.nbr[e];      // (through the read-only path the forward kernel's loads were scheduled 6 % slower at C0 = 128)
    const int j = js.x, s = js.y;
    const int nx = (int)(signed char)(s & 0xff), ny = (int)(signed char)((s >> 8) & 0xff),
              nz = (int)(signed char)((s >> 16) & 0xff);
    const int4 r = __ldg(a.fix + j);
    const int tj = r.w;
    unsigned ix = (unsigned)r.x - (unsigned)c.x, iy = (unsigned)r.y - (unsigned)c.y, iz = (unsigned)r.z - (unsigned)c.z;   // (wraps)
    if (Hf) {
        ix += nx * (unsigned)__ldg(Hf + 0) + ny * (unsigned)__ldg(Hf + 3) + nz * (unsigned)__ldg(Hf + 6);
        iy += nx * (unsigned)__ldg(Hf + 1) + ny * (unsigned)__ldg(Hf + 4) + nz * (unsigned)__ldg(Hf + 7);
        iz += nx * (unsigned)__ldg(Hf + 2) + ny * (unsigned)__ldg(Hf + 5) + nz * (unsigned)__ldg(Hf + 8);
    } else if (a.tri) {        // general cell: the image offset is n . H
        ix += nx * (unsigned)a.Hq[0] + ny * (unsigned)a.Hq[3] + nz * (unsigned)a.Hq[6];
        iy += nx * (unsigned)a.Hq[1] + ny * (unsigned)a.Hq[4] + nz * (unsigned)a.Hq[7];
        iz += nx * (unsigned)a.Hq[2] + ny * (unsigned)a.Hq[5] + nz * (unsigned)a.Hq[8];
    } else {
        ix += nx * (unsigned)a.Hq[0]; iy += ny * (unsigned)a.Hq[4]; iz += nz * (unsigned)a.Hq[8];
    }
    g.dx = a.quantum * (float)(int)ix; g.dy = a.quantum * (float)(int)iy; g.dz = a.quantum * (float)(int)iz;
    const float r2 = g.dx * g.dx + g.dy * g.dy + g.dz * g.dz + kEpsReg * kEpsReg;
    g.rho = sqrtf(r2);
    if (!(g.rho < a.d.rc)) return g;       // skin-shell edge: zero weight
    g.valid = true;
    g.inv_rho = 1.0f / g.rho;
    g.ux = g.dx * g.inv_rho; g.uy = g.dy * g.inv_rho; g.uz = g.dz * g.inv_rho;
    const float inv_rc = 1.0f / a.d.rc;
    const float x = g.rho * inv_rc, t = 1.0f - x;
    const float t2 = t * t, x2 = x * x;
    const float poly = 1.0f + x * (4.0f + x * (10.0f + x * (20.0f + 35.0f * x)));
    g.chi = t2 * t2 * poly;
    g.dchi = -280.0f * x2 * x2 * t2 * t * inv_rc;
    const int n_rows = VALUE ? a.d.n_vrows : a.d.n_rows;
    int row = (int)(g.rho * (VALUE ? a.d.inv_vdx : a.d.inv_dx));
    row = row < n_rows - 1 ? row : n_rows - 1;
    g.row = row;
    g.t = VALUE ? fmaf(-((float)row + 0.5f), a.d.vdx, g.rho) : fmaf(-(float)row, a.d.dx, g.rho);
    if (a.uni) {
        // per-pair amplitude tables, one after another: the pair selects the table (ti is
        // already the compact index of the centre's species)
        if (a.n_present > 1) {           // with one species there is one table and no lookup
            g.pair = ti * a.n_present + (a.species_slot ? a.species_slot[tj] : tj);
            g.row += g.pair * n_rows;
        }
    } else {
        g.pair = ti * a.d.T + tj;
    }
    return g;
}

template <int L>
__device__ __forceinline__ void harmonics_s1(float x, float y, float z, float* B1, float* B2, float* B3, float* B4) {
    const float r3 = 1.7320508075688772f;
    B1[0] = x; B1[1] = y; B1[2] = z;
    B2[0] = r3 * x * y; B2[1] = r3 * y * z; B2[2] = 0.5f * (3.0f * z * z - 1.0f); B2[3] = r3 * x * z;
    B2[4] = 0.5f * r3 * (x * x - y * y);
    if (L >= 3) {
        const float a = 0.7905694150420949f, b = 3.872983346207417f, c = 0.6123724356957945f;
        B3[0] = a * y * (3.0f * x * x - y * y);
        B3[1] = b * x * y * z;
        B3[2] = c * y * (5.0f * z * z - 1.0f);
        B3[3] = 0.5f * z * (5.0f * z * z - 3.0f);
        B3[4] = c * x * (5.0f * z * z - 1.0f);
        B3[5] = 0.5f * b * z * (x * x - y * y);
        B3[6] = a * x * (x * x - 3.0f * y * y);
    }
    if (L >= 4) {   // degree four of the supplementary note, |u|^2 = 1
        const float xx = x * x, yy = y * y, zz = z * z;
        const float a0 = 2.958039891549808f, a1 = 2.0916500663351889f, a2 = 1.118033988749895f, a3 = 0.7905694150420949f,
                    a6 = 0.5590169943749475f, a8 = 0.739509972887452f;
        B4[0] = a0 * x * y * (xx - yy);
        B4[1] = a1 * y * z * (3.0f * xx - yy);
        B4[2] = a2 * x * y * (7.0f * zz - 1.0f);
        B4[3] = a3 * y * z * (7.0f * zz - 3.0f);
        B4[4] = 0.125f * (35.0f * zz * zz - 30.0f * zz + 3.0f);
        B4[5] = a3 * x * z * (7.0f * zz - 3.0f);
        B4[6] = a6 * (xx - yy) * (7.0f * zz - 1.0f);
        B4[7] = a1 * x * z * (xx - 3.0f * yy);
        B4[8] = a8 * (xx * xx - 6.0f * xx * yy + yy * yy);
    }
}

// sum over l >= 1 of t_lm * grad_u B_lm (|u|^2 = 1 convention)
template <int L>
__device__ __forceinline__ void harmonics_grad_contract(float x, float y, float z, const float* t1,
                                                        const float* t2, const float* t3, const float* t4, float* gx,
                                                        float* gy, float* gz) {
    const float r3 = 1.7320508075688772f;
    float ax = t1[0], ay = t1[1], az = t1[2];
    ax += r3 * (t2[0] * y + t2[3] * z + t2[4] * x);
    ay += r3 * (t2[0] * x + t2[1] * z - t2[4] * y);
    az += r3 * (t2[1] * y + t2[3] * x) + 3.0f * t2[2] * z;
    if (L >= 3) {
        const float a = 0.7905694150420949f, b = 3.872983346207417f, c = 0.6123724356957945f;
        const float xx = x * x, yy = y * y, zz = z * z;
        ax += t3[0] * (6.0f * a * x * y) + t3[1] * (b * y * z) + t3[4] * (c * (5.0f * zz - 1.0f)) +
              t3[5] * (b * x * z) + t3[6] * (3.0f * a * (xx - yy));
        ay += t3[0] * (3.0f * a * (xx - yy)) + t3[1] * (b * x * z) + t3[2] * (c * (5.0f * zz - 1.0f)) -
              t3[5] * (b * y * z) - t3[6] * (6.0f * a * x * y);
        az += t3[1] * (b * x * y) + t3[2] * (10.0f * c * y * z) + t3[3] * (0.5f * (15.0f * zz - 3.0f)) +
              t3[4] * (10.0f * c * x * z) + t3[5] * (0.5f * b * (xx - yy));
    }
    if (L >= 4) {
        const float xx = x * x, yy = y * y, zz = z * z;
        const float a0 = 2.958039891549808f, a1 = 2.0916500663351889f, a2 = 1.118033988749895f, a3 = 0.7905694150420949f,
                    a6 = 0.5590169943749475f, a8 = 0.739509972887452f;
        const float s7 = 7.0f * zz - 1.0f, s73 = 7.0f * zz - 3.0f, s21 = 21.0f * zz - 3.0f;
        ax += t4[0] * (a0 * y * (3.0f * xx - yy)) + t4[1] * (6.0f * a1 * x * y * z) + t4[2] * (a2 * y * s7) + t4[5] * (a3 * z * s73) +
              t4[6] * (2.0f * a6 * x * s7) + t4[7] * (3.0f * a1 * z * (xx - yy)) + t4[8] * (4.0f * a8 * x * (xx - 3.0f * yy));
        ay += t4[0] * (a0 * x * (xx - 3.0f * yy)) + t4[1] * (3.0f * a1 * z * (xx - yy)) + t4[2] * (a2 * x * s7) + t4[3] * (a3 * z * s73) -
              t4[6] * (2.0f * a6 * y * s7) - t4[7] * (6.0f * a1 * x * y * z) + t4[8] * (4.0f * a8 * y * (yy - 3.0f * xx));
        az += t4[1] * (a1 * y * (3.0f * xx - yy)) + t4[2] * (14.0f * a2 * x * y * z) + t4[3] * (a3 * y * s21) +
              t4[4] * (z * (17.5f * zz - 7.5f)) + t4[5] * (a3 * x * s21) + t4[6] * (14.0f * a6 * z * (xx - yy)) +
              t4[7] * (a1 * x * (xx - 3.0f * yy));
    }
    *gx = ax; *gy = ay; *gz = az;
}

// a b + c of two channels: in one instruction (PAIR), which saves issue slots, or in two, which leaves the registers where they
// are: the forward kernel at C0 = 128 with the pair cache takes 378 us with single multiply-adds and 443 with pairs (40,009 atoms of
// 64 species, 80 registers), the backward kernel 449 with pairs and 466 without; C0 = 64, 32,400 atoms, forward 160 and 164.
template <bool PAIR>
__device__ __forceinline__ float2 axpy2(float2 a, float2 b, float2 c) {
    return PAIR ? ffma2(a, b, c) : make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
}
__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 lo2(const float4& v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4& v) { return make_float2(v.z, v.w); }
// the two numbers of a packed word of two channels (common.cuh, tab_pack)
__device__ __forceinline__ float2 word_hi2(int a, int b) { return make_float2(tab_hi(a), tab_hi(b)); }
__device__ __forceinline__ float2 word_lo2(int a, int b) { return make_float2(tab_lo(a), tab_lo(b)); }

// value and derivative of four consecutive table channels at offset t in row `row`: three
// 16-byte loads, c0, c1 and the packed (c2, c3) words with steps k2, k3
__device__ __forceinline__ void table_eval4(const float* __restrict__ table, int CP, int row, int c, float t,
                                            float k2, float k3, float* v, float* dv) {
    const float* p = table + (size_t)row * 3 * CP + c;
    const float4 c0 = ldg4(p), c1 = ldg4(p + CP);
    const int4 w = __ldg(reinterpret_cast<const int4*>(p + 2 * CP));
    const float s2 = k2 * kTabHi * t, s3 = k3 * kTabLo * t * t;
    const float2 tt = both(t), u2 = both(s2 * t), u3 = both(s3 * t), v2 = both(2.0f * s2), v3 = both(3.0f * s3);
    const float2 ha = word_hi2(w.x, w.y), hb = word_hi2(w.z, w.w), la = word_lo2(w.x, w.y), lb = word_lo2(w.z, w.w);
    const float2 a = ffma2(la, u3, ffma2(ha, u2, ffma2(lo2(c1), tt, lo2(c0)))), b = ffma2(lb, u3, ffma2(hb, u2, ffma2(hi2(c1), tt, hi2(c0))));
    const float2 da = ffma2(la, v3, ffma2(ha, v2, lo2(c1))), db = ffma2(lb, v3, ffma2(hb, v2, hi2(c1)));
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    dv[0] = da.x; dv[1] = da.y; dv[2] = db.x; dv[3] = db.y;
}
// values alone, from the value table (common.cuh, value_piece): two 16-byte loads, t from the middle of the
// piece, k2 and k3 the steps of its linear and quadratic coefficients.  The forward kernel is bound by what it
// pulls from L2 and through the L1 data pipe, and a row is 8 bytes per channel instead of the 12 of the table
// with derivatives: 1,000,000 atoms of 64 species at C0 = 128 11.9 -> 10.3 ms, 128,000 of five species 0.84 ->
// 0.69, 64,000 of one 1.02 -> 0.84, 216,000 at C0 = 8 0.867 -> 0.807.
template <bool PAIR = true>
__device__ __forceinline__ void value_eval4(const float* __restrict__ table, int CP, int row, int c, float t,
                                            float k2, float k3, float* v) {
    const float* p = table + (size_t)row * 2 * CP + c;
    const float4 a0 = ldg4(p);
    const int4 w = __ldg(reinterpret_cast<const int4*>(p + CP));
    const float2 u1 = both(k2 * kTabHi * t), u2 = both(k3 * kTabLo * t * t);
    const float2 a = axpy2<PAIR>(word_lo2(w.x, w.y), u2, axpy2<PAIR>(word_hi2(w.x, w.y), u1, lo2(a0)));
    const float2 b = axpy2<PAIR>(word_lo2(w.z, w.w), u2, axpy2<PAIR>(word_hi2(w.z, w.w), u1, hi2(a0)));
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
// v += s u, four channels
template <bool PAIR = true>
__device__ __forceinline__ void axpy4(float s, const float4& u, float* v) {
    const float2 a = axpy2<PAIR>(both(s), lo2(u), make_float2(v[0], v[1])), b = axpy2<PAIR>(both(s), hi2(u), make_float2(v[2], v[3]));
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
template <bool PAIR = true>
__device__ __forceinline__ void axpy4(float s, const float* u, float* v) { axpy4<PAIR>(s, make_float4(u[0], u[1], u[2], u[3]), v); }
// v = u v + w, four channels
template <bool PAIR = true>
__device__ __forceinline__ void affine4(const float4& u, const float4& w, float* v) {
    const float2 a = axpy2<PAIR>(lo2(u), make_float2(v[0], v[1]), lo2(w)), b = axpy2<PAIR>(hi2(u), make_float2(v[2], v[3]), hi2(w));
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ float4 scaled(float s, const float4& u) { return make_float4(s * u.x, s * u.y, s * u.z, s * u.w); }

// Shared radial modes q_mu(rho) of the first nb queued edges, an edge per lane, parked as qm[edge * PQ + mu]: evaluated once
// per edge here instead of once per lane in the channel-parallel phase.  (Rows are padded to whole fours of columns.)
// DQ: what comes with them in dqm: nothing, their derivatives, or the products (chi q)' (product table).
enum : int { kValuesOnly = 0, kDerivatives = 1, kProducts = 2 };
template <int DQ, int PQ>
__device__ __forceinline__ void eval_modes(const EdgeArgs& a, const int4* qes, int nb, int lane, float* qm, float* dqm) {
    if (lane >= nb) return;
    const int4 es = qes[lane];
    const float t = __int_as_float(es.z);
    for (int q = 0; q < a.d.R; q += 4) {
        float v[4], dv[4];
        if (DQ == kDerivatives) table_eval4(a.table, a.d.CP, es.x, a.d.C0 + q, t, a.d.tab_k2, a.d.tab_k3, v, dv);
        else value_eval4(a.vtable, a.d.CP, es.x, a.d.C0 + q, t, a.d.tab_v1, a.d.tab_v2, v);
        if (DQ == kProducts) value_eval4(a.dtable, a.d.CP, es.x, a.d.C0 + q, t, a.d.tab_d1, a.d.tab_d2, dv);
        *reinterpret_cast<float4*>(qm + lane * PQ + q) = make_float4(v[0], v[1], v[2], v[3]);
        if (DQ) *reinterpret_cast<float4*>(dqm + lane * PQ + q) = make_float4(dv[0], dv[1], dv[2], dv[3]);
    }
}

// What a kernel does about shared radial modes (without per-pair tables): there are none; every edge reads its pair's mixing
// rows; or the scalar channels get them, and beta, from the row's moments (moments.cu).  kSplines: one species, whose scalar
// channels are B-splines and enter through the row's spline weights (moments.cu)
enum : int { kNoModes = 0, kModesPerEdge = 1, kMoments = 2, kSplines = 3 };

// interval of a distance and place in it
__device__ __forceinline__ int spline_interval(const EdgeArgs& a, float rho, float* t) {
    const int k = min((int)(rho * a.spline_inv_h), a.spline_n - 1);
    *t = fmaf(rho, a.spline_inv_h_lo, fmaf(rho, a.spline_inv_h, -(float)k));
    return k;
}
// basis functions of degree six (times 6!) and seven (times 7!) that are not zero on the interval, by their recursion.  The
// coefficients (moments.cu) are divided by 7!, in double: a factor of 1 / 5040 in single precision is 1.4e-8 off, the same way for
// every edge of every atom.
__device__ __forceinline__ void spline_basis(float t, float* u6, float* u7) {
    float u[7];
    u[0] = 1.0f;
#pragma unroll
    for (int d = 1; d <= 6; ++d) {
#pragma unroll
        for (int j = d; j >= 0; --j)
            u[j] = j == d ? t * u[j - 1] : (j == 0 ? (1.0f - t) * u[0] : fmaf(t + (float)(d - j), u[j - 1], ((float)(j + 1) - t) * u[j]));
    }
#pragma unroll
    for (int j = 0; j < 7; ++j) u6[j] = u[j];
#pragma unroll
    for (int j = 0; j < 8; ++j)
        u7[j] = j == 7 ? t * u[6] : (j == 0 ? (1.0f - t) * u[0] : fmaf(t + (float)(7 - j), u[j - 1], ((float)(j + 1) - t) * u[j]));
}

// adds sum_mu U_c,mu q_mu of four channels; pm: the pair's rows at the channel
template <int C0, bool PAIR = true>
__device__ __forceinline__ void add_modes4(const EdgeArgs& a, const float* pm, const float* qm, float* v) {
    const int R = a.d.R;
    float q[kMaxR];
    const float4 v0 = *reinterpret_cast<const float4*>(qm);
    q[0] = v0.x; q[1] = v0.y; q[2] = v0.z; q[3] = v0.w;
    if (R > 4) { const float4 v1 = *reinterpret_cast<const float4*>(qm + 4); q[4] = v1.x; q[5] = v1.y; q[6] = v1.z; q[7] = v1.w; }
#pragma unroll
    for (int m = 0; m < kMaxR; ++m) {
        if (m >= R) break;
        axpy4<PAIR>(q[m], ldg4(pm + (size_t)(2 + m) * C0), v);
    }
}

// amplitude psi (and d psi / d rho) of this lane's four channels for one edge; qm / dqm: the
// edge's parked radial modes (only read when HASR).  UNI: psi_c(rho) of every ordered pair of
// species present is tabulated by itself (a.table_uni, row pitch C0; `row` already points into
// the edge's pair), so neither pair rows nor modes are read.  k2, k3: steps of the packed
// coefficients of the table that is read
template <int C0, bool HASR, bool DERIV, bool UNI, bool PAIR = true>
__device__ __forceinline__ void amplitude4(const EdgeArgs& a, int row, float t, int pair, int c, float* psi,
                                           float* dpsi, const float* qm, const float* dqm, float k2, float k3) {
    if (UNI) {
        if (DERIV) table_eval4(a.table_uni, C0, row, c, t, k2, k3, psi, dpsi);
        else value_eval4<PAIR>(a.vtable_uni, C0, row, c, t, k2, k3, psi);
        return;
    }
    if (DERIV) table_eval4(a.table, a.d.CP, row, c, t, k2, k3, psi, dpsi);
    else value_eval4<PAIR>(a.vtable, a.d.CP, row, c, t, k2, k3, psi);
    const float* pm = a.pairmod + (size_t)pair * (2 + (HASR ? a.d.R : 0)) * C0 + c;
    const float4 ga = ldg4(pm), be = ldg4(pm + C0);
    affine4<PAIR>(ga, be, psi);
    if (DERIV) { dpsi[0] *= ga.x; dpsi[1] *= ga.y; dpsi[2] *= ga.z; dpsi[3] *= ga.w; }
    if (HASR) {
        add_modes4<C0, PAIR>(a, pm, qm, psi);
        if (DERIV) add_modes4<C0>(a, pm, dqm, dpsi);
    }
}

// (chi psi_c)' of this lane's four channels for one edge, from the product table; row and t of the value grid, dchi
// the envelope's derivative (only without per-pair tables), dqm the edge's parked (chi q)' (MODES).  With moments
// the beta and mode parts are left out.
template <int C0, int MODES, bool UNI>
__device__ __forceinline__ void product4(const EdgeArgs& a, int row, float t, int pair, int c, float dchi, const float* dqm, float d1, float d2,
                                         float* d) {
    if (UNI) {
        value_eval4(a.dtable_uni, C0, row, c, t, d1, d2, d);
        return;
    }
    value_eval4(a.dtable, a.d.CP, row, c, t, d1, d2, d);
    const float* pm = a.pairmod + (size_t)pair * (MODES ? 2 + a.d.R : 2) * C0 + c;
    const float4 ga = ldg4(pm);
    if (MODES == kMoments) {
        d[0] *= ga.x; d[1] *= ga.y; d[2] *= ga.z; d[3] *= ga.w;
        return;
    }
    affine4(ga, scaled(dchi, ldg4(pm + C0)), d);
    if (MODES) add_modes4<C0>(a, pm, dqm, d);
}
// G = groups of four channels a lane holds in the channel-parallel phase (group g starts at
// channel 4 * lane_in_group + g * C0 / G, so every 16-byte load instruction of a group of lanes
// still covers one contiguous segment)
// ROWS: amplitudes and weights of an edge in one row at C0 = 128 too (see VECW)
template <int C0, int L, int G = 1, bool ROWS = false> struct Widths {
    static constexpr int C1 = C0 <= 16 ? 4 : (C0 <= 64 ? 8 : 16);
    static constexpr int C2 = C1 / 2 > 4 ? C1 / 2 : 4;
    static constexpr int LPE = C0 / (4 * G);    // lanes per edge in the channel-parallel phase
    static constexpr int GOFF = C0 / G;         // channel offset between a lane's groups
    static constexpr int LH = LPE / 2;          // parked partial dot products per edge (lanes paired)
    static constexpr int EPI = 32 / LPE;        // edges per replay step
    static constexpr int NL1 = C1 / 4;          // lanes of a group that hold degree-1 channels
    static constexpr int NHI = 3 * C1 + 5 * C2 + (L >= 3 ? 7 : 0) + (L >= 4 ? 9 : 0);   // sums of degree >= 1
    static constexpr int PB = ((2 * C1 / 4 + 1) & 1) ? 2 * C1 + 4 : 2 * C1 + 8;   // backward: psi, dpsi
    // Forward, sums of degree >= 1: a job is four consecutive channels (vector) of two components of degrees 1 and 2, in their
    // order (scalars; PAIRS): two reads of the parked row for eight multiply-adds.  (The L1 data pipe takes a cycle for every word
    // that a lane reads, broadcast or not: a job of one component reads five words for four multiply-adds.  C0 = 64, 32,400 atoms,
    // 170 -> 160 us; at C0 = 8, whose eight jobs of one component fill a group, 234 -> 244 for 64,000 atoms with 158 neighbours.)
    // The channels that only degree 1 has get two pairs for its three components.  Degrees 3 and 4 have one channel: four
    // components of them (vector) times that (scalar).  EG groups of JW lanes take every EG-th edge each.
    static constexpr bool PAIRS = C0 >= 32;
    static constexpr int JFULL = C2 / 4 * (PAIRS ? 4 : 8), JLOW = (C1 - C2) / 4 * (PAIRS ? 2 : 3), J3 = L >= 3 ? 2 : 0, J4 = L >= 4 ? 3 : 0;
    static constexpr int NJ = JFULL + JLOW + J3 + J4;
    static constexpr int JW = NJ <= 4 ? 4 : (NJ <= 8 ? 8 : (NJ <= 16 ? 16 : 32)), EG = 32 / JW;
    // the parked row of an edge: leading C1 amplitudes, harmonic weights (degree 3 from 8 on, degree 4 from 16).  VECW: one
    // row, pitch / 4 odd, so that 16-byte accesses of eight consecutive lanes fall on distinct banks.  C0 = 128 with per-pair
    // tables: amplitude rows need no padding, and the weights sit behind them (40,009 atoms of five species 197 us, 214 in one
    // row; with the pair cache the other way, 410 and 378 for 64 species).
    static constexpr bool VECW = C0 <= 64 || ROWS;
    static constexpr int NM = L >= 4 ? 28 : (L >= 3 ? 16 : 8);
    static constexpr int PP = VECW ? (((C1 + NM) / 4) & 1 ? C1 + NM : C1 + NM + 4) : C1;      // pitch of the amplitudes
    static constexpr int PW = VECW ? PP : ((NM / 4) & 1 ? NM : NM + 4);                       // pitch of the weights
    static constexpr int OW = VECW ? C1 : 32 * C1;                                            // offset of the weights
    static constexpr int PQ = VECW ? PP : kMaxR;     // the radial modes sit where the weights come later
    static constexpr int SCRATCH = VECW ? 32 * PP : 32 * C1 + (32 * PW > 32 * kMaxR ? 32 * PW : 32 * kMaxR);
};

// The channel-parallel phase of the backward pass waits on load latency, and what hides it best
// depends on the width and on what is read (all measured on the edge backward kernel).  C0 = 128 with shared
// table and pair cache, or degree three: four channel groups per lane, that many times the loads in flight,
// at 16 resident warps per SM (128 registers): 64,007 atoms of one species by tables (as its rows go below 8192, or
// where they are short) 1.10 ms against 1.19 with two groups at 24 warps (85 registers, spilled words), a million atoms of
// the 64-species mixture, when its kernel took 12.6 ms, 14.6.  By splines the same.  With shared modes,
// and with per-pair tables at degree two (fewer registers spilled): the latter, 1.62 -> 1.49 ms for 40,009 atoms
// with four modes, 1.00 -> 0.94 for 128,000 atoms of five species.  C0 = 32 and 64: two groups at 24 warps;
// C0 <= 16: one group, 24 warps.  FEW: rows for more than 24 but not more than 32 warps per SM (3553 to 4736): 64
// registers and one wave beat 85 and two (4000 atoms at C0 = 64: 41 -> 35 us; 597 atoms 25 against 21, 32,400
// atoms 254 against 234).
template <int C0, int L, int MODES, bool UNI, bool FEW> struct BwdShape {
    static constexpr bool two = C0 >= 128 && (MODES == kModesPerEdge || (MODES == kNoModes && UNI && L == 2));
    static constexpr int G = C0 >= 128 ? (two ? 2 : 4) : (C0 >= 32 ? 2 : 1);
    static constexpr int warps = C0 >= 128 ? (two ? 24 : 16) : (MODES == kMoments ? 16 : (FEW ? 32 : 24));
    static constexpr bool tight = two || FEW;
};

template <int C0, int L, int MODES, bool UNI> struct BwdSmem {          // dynamic shared memory of the backward kernel
    using W = Widths<C0, L, BwdShape<C0, L, MODES, UNI, false>::G>;
    static constexpr int queue_floats = 32 * 4 + 5 * 32;    // queue of in-range edges: int4 and five scalars per slot
    static constexpr int mode_floats = MODES == kModesPerEdge || MODES == kMoments ? 2 * 32 * kMaxR : 0;   // parked radial modes and their derivatives or products
    static constexpr bool products = wide_channels(C0);             // reads the product table (product_piece)
    static constexpr int n_red = MODES == kSplines ? 0 : (products ? 1 : 2);                  // partial dot products per edge and lane pair
    static constexpr int per_warp = (32 * W::PB + n_red * 32 * (W::LH + 1) + W::NHI + 3) / 4 * 4 + mode_floats + queue_floats;   // floats
    static constexpr size_t bytes = kWarpsPerBlock * 9 * sizeof(double) + sizeof(float) * kWarpsPerBlock * per_warp;
};

// ------------------------------------------------------------------------------- forward
//
// The row is scanned 32 listed edges at a time (lane = edge: geometry); the edges that fall
// inside the cutoff are appended to a 32-slot per-warp queue in shared memory (edges that do
// not fit wait in their lane's registers), and whenever 32 are there (and once more at the end
// of the row) a full batch is processed, so the later phases never run on skin-shell edges:
//   2. lanes = channels (a group of C0/4 lanes per edge): amplitude psi of all C0 channels,
//      degree-0 sums accumulated in registers; the leading C1 amplitudes of each edge are
//      parked in shared memory.
//   3. lane = edge again: harmonics of the lane's own edge, parked as weights chi^2 B_lm; then
//      lane = job: a lane owns four consecutive channels of two harmonic components (of one below C0 = 32,
//      or up to four components of a one-channel degree) for the whole row, and for every edge of its group
//      of edges adds vector x scalar from the parked row: two shared-memory reads per edge and group of
//      lanes, where summing per-edge products by transposition took six.
// One species by splines: phase 2 adds eight spline weights per edge to the row's, and forms the leading amplitudes alone.
// What hides the load latency of the channel-parallel phase best depends on the width and on what is read.  Up to C0 = 64, 32
// warps per SM (64 registers, a few spilled words; 24 were 6 to 10 % slower).  C0 = 128: with per-pair tables an edge per half
// warp, two channel groups per lane, at 24 warps (40,009 atoms of five species 196 us; two at 16 warps 242, four at 20 warps
// 194); with shared table and pair cache four groups at 16 warps (131,072 atoms of 64 species 1184 us, 8000 93; two groups 1232
// and 95, one at 24 warps 1212 and 100); the same by moments two groups at 20 warps (688 us, one at 24 700, four at 16 723,
// 40,009 atoms with four modes).
template <int C0, int MODES, bool UNI> struct FwdShape {
    static constexpr bool cache = !UNI && MODES == kNoModes;
    static constexpr int G = C0 < 128 || MODES == kModesPerEdge ? 1 : (cache ? 4 : 2);
    static constexpr int warps = C0 < 128 ? (MODES < kMoments ? 32 : 24) : (cache ? 16 : (MODES == kMoments ? 20 : 24));
};
// SPLIT: the warps of a block take a quarter each of one row (edge_rows_split) and add up their sums at the end.
// MODES == kMoments: the scalar channels' sums get gamma g alone from the edges; the row's moments, for every species t of the
// neighbours sum chi and sum chi q_mu, are left for moments.cu, which adds beta and U times them.  40,009 atoms of 64 species
// with four modes: 1168 us with the 2.5 KB of these rows read per edge.
template <int C0, int L, int MODES, bool UNI, bool SPLIT>
__global__ void __launch_bounds__(kWarpsPerBlock * 32, FwdShape<C0, MODES, UNI>::warps / kWarpsPerBlock)
k_edge_forward(const EdgeArgs a) {
    constexpr int G = FwdShape<C0, MODES, UNI>::G;          // channel groups of a lane
    constexpr bool PAIR = C0 < 128 || UNI;                  // see axpy2
    using W = Widths<C0, L, G, !UNI>;
    constexpr bool HASR = MODES == kModesPerEdge || MODES == kMoments, SPL = MODES == kSplines;
    static_assert(C0 + W::NHI <= W::SCRATCH, "a split row's partial sums take the place of the batch");
    // scratch per warp: the parked amplitudes of the batch, first the radial modes and then (once the
    // amplitudes are done) the harmonic weights chi^2 B_lm
    __shared__ __align__(16) float scratch[kWarpsPerBlock][W::SCRATCH];
    // queue of edges inside the cutoff: row, pair, t, chi (fetched with one 16-byte broadcast
    // load in the channel-parallel phase; shuffles would go through the same L1 data pipe as
    // the table reads) and the edge vector
    __shared__ int4 q_es[kWarpsPerBlock][32];
    __shared__ float q_d[kWarpsPerBlock][3 * 32];
    __shared__ double s_part[SPLIT ? kWarpsPerBlock : 1][2];
    extern __shared__ __align__(16) float moments_s[];         // [warp][a.n_moments]
    chain_begin();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int i = a.a0 + (SPLIT ? blockIdx.x : blockIdx.x * kWarpsPerBlock + wid);
    if (i >= a.a1) return;
    float* const psi_s = scratch[wid];             // [32][PP]
    float* const qm = scratch[wid] + W::OW;        // [32][PQ] radial modes
    float* const wbs = scratch[wid] + W::OW;       // [32][PW] harmonic weights, in the same place later
    int4* const qes = q_es[wid];
    float* const qd = q_d[wid];
    const int sub = lane / W::LPE, cl = lane % W::LPE, c = 4 * cl;
    const int4 ci = __ldg(a.fix + i);
    const int ti = UNI && a.species_slot ? a.species_slot[ci.w] : ci.w;
    const float k2 = UNI ? tab_step2(__ldg(a.uni_scale + 2)) : a.d.tab_v1, k3 = UNI ? tab_step3(__ldg(a.uni_scale + 3)) : a.d.tab_v2;
    eidx_t e0 = a.row_ptr[i];
    int len = (int)(a.row_ptr[i + 1] - e0);      // edge offsets are 64-bit, offsets inside a row are not
    if (SPLIT) quarter_of_row(wid, &e0, &len);
    const int* Hf = a.frames ? a.frames[a.frame_of[i]].Hq : nullptr;
    const unsigned lt_mask = (1u << lane) - 1u;
    float acc0[4 * G];
#pragma unroll
    for (int k = 0; k < 4 * G; ++k) acc0[k] = 0.f;
    // this lane's job of the degree >= 1 sums: where its vector and its scalars are in the rows of edge 0, offset of the
    // results in the output block and their number, for each of its components
    float2 accJ[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) accJ[k] = make_float2(0.f, 0.f);
    int j_v = 0, j_s = W::OW, j_out[2] = {0, 0}, j_n[2] = {0, 0};
    const int eg = lane / W::JW, job = lane % W::JW;
    if (job < W::JFULL + W::JLOW) {
        constexpr int NF = W::PAIRS ? 4 : 8, NL = W::PAIRS ? 2 : 3, NC = W::PAIRS ? 2 : 1;      // jobs of a run of channels, components of a job
        const int cb = job < W::JFULL ? job / NF : W::C2 / 4 + (job - W::JFULL) / NL, part = job < W::JFULL ? job % NF : (job - W::JFULL) % NL;
        j_v = 4 * cb; j_s += NC * part;
#pragma unroll
        for (int h = 0; h < NC; ++h) {
            const int m = NC * part + h;
            if (m < 3) { j_out[h] = m * W::C1 + 4 * cb; j_n[h] = 4; }
            else if (4 * cb < W::C2) { j_out[h] = 3 * W::C1 + (m - 3) * W::C2 + 4 * cb; j_n[h] = 4; }
        }
    } else if (job < W::NJ) {
        const int jj = job - W::JFULL - W::JLOW;
        const bool deg3 = jj < W::J3;
        const int first = deg3 ? 4 * jj : 4 * (jj - W::J3);      // component
        j_v = W::OW + (deg3 ? 8 : 16) + first; j_s = 0;
        j_out[0] = 3 * W::C1 + 5 * W::C2 + (deg3 ? 0 : 7) + first;
        j_n[0] = min(4, (deg3 ? 7 : 9) - first);
    }
    const bool swapped = job >= W::JFULL + W::JLOW && job < W::NJ;      // (weights and amplitudes change places in the jobs of one channel)
    const int pitch_v = swapped ? W::PW : W::PP, pitch_s = swapped ? W::PP : W::PW;
    // (splines: four partial rows, one for each group of eight lanes)
    float* const mom = moments_s + (MODES == kMoments ? 1 : (SPL ? 4 : 0)) * wid * a.n_moments;
    if (MODES == kMoments || SPL) {
        for (int v = lane; v < (SPL ? 4 : 1) * a.n_moments; v += 32) mom[v] = 0.f;
        __syncwarp();
    }
    double s0 = 0.0, s1 = 0.0;   // normaliser sums in double: the calibration subtracts their mean

    auto run_batch = [&](const int nb) {     // the first nb queue slots
        if (HASR) {
            eval_modes<kValuesOnly, W::PQ>(a, qes, nb, lane, qm, nullptr);
            __syncwarp();
        }
        if constexpr (MODES == kMoments) {
            // moments: the edges of a species are added up by the first of them
            const int tj = lane < nb ? qes[lane].y - ti * a.d.T : -1;
            const unsigned same = __match_any_sync(kFull, tj);
            if (tj >= 0 && (same & lt_mask) == 0) {
                float v[1 + kMaxR];
#pragma unroll
                for (int q = 0; q <= kMaxR; ++q) v[q] = 0.f;
                for (unsigned m = same; m; m &= m - 1) {
                    const int b = __ffs(m) - 1;
                    const float chi = __int_as_float(qes[b].w);
                    v[0] += chi;
#pragma unroll
                    for (int q = 0; q < kMaxR; ++q) if (q < a.d.R) v[1 + q] += chi * qm[b * W::PQ + q];
                }
                float* const p = mom + tj * (1 + a.d.R);
#pragma unroll
                for (int q = 0; q <= kMaxR; ++q) if (q <= a.d.R) p[q] += v[q];
            }
            // the leading channels' whole amplitudes, four channels of an edge per lane
            constexpr int LE = 32 / W::NL1;
            for (int b0 = 0; b0 < nb; b0 += LE) {
                const int b = b0 + lane / W::NL1, cc = 4 * (lane % W::NL1);
                if (b < nb) {
                    const int4 es = qes[b];
                    float psi[4];
                    amplitude4<C0, true, false, false, PAIR>(a, es.x, __int_as_float(es.z), es.y, cc, psi, nullptr, qm + b * W::PQ, nullptr, k2, k3);
                    *reinterpret_cast<float4*>(psi_s + b * W::PP + cc) = make_float4(psi[0], psi[1], psi[2], psi[3]);
                }
            }
        }
        if constexpr (SPL) {
            // lane = edge: eight spline weights times the envelope, parked in rows of twelve with their first place; then
            // eight lanes per edge add them to their group's row
            constexpr int TP = 12;
            static_assert(32 * TP <= W::SCRATCH, "spline weights of a batch");
            if (lane < nb) {
                const int4 es = qes[lane];
                float t, u6[7], u7[8];
                const int k = spline_interval(a, __int_as_float(es.y), &t);
                spline_basis(t, u6, u7);
                const float w = __int_as_float(es.w);            // (the coefficients hold 1 / 7!)
                float4* const o = reinterpret_cast<float4*>(psi_s + lane * TP);
                o[0] = make_float4(w * u7[0], w * u7[1], w * u7[2], w * u7[3]);
                o[1] = make_float4(w * u7[4], w * u7[5], w * u7[6], w * u7[7]);
                psi_s[lane * TP + 8] = __int_as_float(k);
            }
            __syncwarp();
            // (the places of successive edges overlap: a lane adds to what another lane of its group left there)
            float* const part = mom + (lane >> 3) * a.n_moments + (lane & 7);
            for (int e0 = 0; e0 < nb; e0 += 4) {
                const int e = e0 + (lane >> 3);
                if (e < nb) part[__float_as_int(psi_s[e * TP + 8])] += psi_s[e * TP + (lane & 7)];
                __syncwarp();
            }
            // amplitudes of the leading channels, four channels of an edge per lane
            constexpr int LE = 32 / W::NL1;
            for (int b0 = 0; b0 < nb; b0 += LE) {
                const int b = b0 + lane / W::NL1, cc = 4 * (lane % W::NL1);
                if (b < nb) {
                    float psi[4];
                    value_eval4(a.vtable_uni, C0, qes[b].x, cc, __int_as_float(qes[b].z), k2, k3, psi);
                    *reinterpret_cast<float4*>(psi_s + b * W::PP + cc) = make_float4(psi[0], psi[1], psi[2], psi[3]);
                }
            }
        }
        // lanes = channels, a group of lanes per edge
        constexpr int UNR = C0 >= 32 ? 1 : 2;     // (unrolled as the compiler would: C0 = 64, 32,400 atoms 185 us, so 160)
#pragma unroll UNR
        for (int it = 0; !SPL && it * W::EPI < nb; ++it) {
            const int b = it * W::EPI + sub;
            if (b >= nb) continue;
            const int4 es = qes[b];
            const float t = __int_as_float(es.z), chi = __int_as_float(es.w);
            float psi[4 * G];
#pragma unroll
            for (int gq = 0; gq < G; ++gq) {
                const int cc = c + gq * W::GOFF;
                if (MODES == kMoments) {
                    value_eval4<PAIR>(a.vtable, a.d.CP, es.x, cc, t, k2, k3, psi + 4 * gq);
                    const float4 ga = scaled(chi, ldg4(a.pairmod + (size_t)es.y * (2 + a.d.R) * C0 + cc));
                    acc0[4 * gq] += ga.x * psi[4 * gq]; acc0[4 * gq + 1] += ga.y * psi[4 * gq + 1];
                    acc0[4 * gq + 2] += ga.z * psi[4 * gq + 2]; acc0[4 * gq + 3] += ga.w * psi[4 * gq + 3];
                } else {
                    amplitude4<C0, HASR, false, UNI, PAIR>(a, es.x, t, es.y, cc, psi + 4 * gq, nullptr, qm + b * W::PQ, nullptr, k2, k3);
                    axpy4<PAIR>(chi, psi + 4 * gq, acc0 + 4 * gq);
                }
            }
            // (the leading C1 channels all sit in group 0)
            if (MODES != kMoments && cl < W::NL1) *reinterpret_cast<float4*>(psi_s + b * W::PP + c) = make_float4(psi[0], psi[1], psi[2], psi[3]);
        }
        __syncwarp();
        // lane = edge: the harmonic weights chi^2 B_lm of the lane's edge, parked next to the amplitudes
        if (lane < nb) {
            float B1[3], B2[5], B3[7], B4[9];
            const float dx = qd[lane], dy = qd[32 + lane], dz = qd[64 + lane];
            const float inv_rho = 1.0f / sqrtf(dx * dx + dy * dy + dz * dz + kEpsReg * kEpsReg);
            harmonics_s1<L>(dx * inv_rho, dy * inv_rho, dz * inv_rho, B1, B2, B3, B4);
            const float chi = __int_as_float(qes[lane].w);
            const float w = chi * chi;
            float* wr = wbs + lane * W::PW;
            float4* w4 = reinterpret_cast<float4*>(wr);
            w4[0] = make_float4(w * B1[0], w * B1[1], w * B1[2], w * B2[0]);
            w4[1] = make_float4(w * B2[1], w * B2[2], w * B2[3], w * B2[4]);
            if (L >= 3) {
                w4[2] = make_float4(w * B3[0], w * B3[1], w * B3[2], w * B3[3]);
                w4[3] = make_float4(w * B3[4], w * B3[5], w * B3[6], 0.f);
            }
            if (L >= 4) {
                w4[4] = make_float4(w * B4[0], w * B4[1], w * B4[2], w * B4[3]);
                w4[5] = make_float4(w * B4[4], w * B4[5], w * B4[6], w * B4[7]);
                w4[6] = make_float4(w * B4[8], 0.f, 0.f, 0.f);
            }
        }
        __syncwarp();
        // lane = job: the sums over the batch stay in the lane's registers for the whole row; per edge of
        // its group a lane reads its vector and its scalars (every lane of a group inside the same two rows)
#pragma unroll 2
        for (int e = eg; e < nb; e += W::EG) {
            const float4 p4 = *reinterpret_cast<const float4*>(psi_s + e * pitch_v + j_v);
            if constexpr (W::PAIRS) {
                const float2 w2 = *reinterpret_cast<const float2*>(psi_s + e * pitch_s + j_s);
                accJ[0] = axpy2<PAIR>(both(w2.x), lo2(p4), accJ[0]); accJ[1] = axpy2<PAIR>(both(w2.x), hi2(p4), accJ[1]);
                accJ[2] = axpy2<PAIR>(both(w2.y), lo2(p4), accJ[2]); accJ[3] = axpy2<PAIR>(both(w2.y), hi2(p4), accJ[3]);
            } else {
                const float wv = psi_s[e * pitch_s + j_s];
                accJ[0] = axpy2<PAIR>(both(wv), lo2(p4), accJ[0]); accJ[1] = axpy2<PAIR>(both(wv), hi2(p4), accJ[1]);
            }
        }
        __syncwarp();                           // the next batch overwrites both
    };

    int qn = 0;
    for (int base = 0; base < len; base += 32) {
        const Geom g = edge_geometry<true>(a, e0 + base + lane, base + lane < len, ci, ti, Hf);
        const unsigned vmask = __ballot_sync(kFull, g.valid);
        const int p = qn + __popc(vmask & lt_mask);       // queue slot of this lane's edge, if it has one
        if (g.valid) { const double c2 = (double)g.chi * (double)g.chi; s0 += c2; s1 += c2 * c2; }
        if (g.valid && p < 32) {
            qes[p] = make_int4(g.row, SPL ? __float_as_int(g.rho) : g.pair, __float_as_int(g.t), __float_as_int(g.chi));
            qd[p] = g.dx; qd[32 + p] = g.dy; qd[64 + p] = g.dz;
        }
        qn += __popc(vmask);
        __syncwarp();
        if (qn >= 32) {                                   // a full batch; the overflow waits in registers
            run_batch(32);
            if (g.valid && p >= 32) {
                qes[p - 32] = make_int4(g.row, SPL ? __float_as_int(g.rho) : g.pair, __float_as_int(g.t), __float_as_int(g.chi));
                qd[p - 32] = g.dx; qd[p] = g.dy; qd[32 + p] = g.dz;
            }
            qn -= 32;
            __syncwarp();
        }
    }
    if (qn > 0) run_batch(qn);
    // combine the edge slots of the warp (lanes with equal channel offset)
#pragma unroll
    for (int off = W::LPE; off < 32; off <<= 1) {
#pragma unroll
        for (int k = 0; k < 4 * G; ++k) acc0[k] += __shfl_xor_sync(kFull, acc0[k], off);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        s0 += __shfl_xor_sync(kFull, s0, off);
        s1 += __shfl_xor_sync(kFull, s1, off);
    }
    float* const row_glob = a.state + (size_t)(i - a.a0) * a.d.SP;
    float* const row_out = SPLIT ? psi_s : row_glob;        // (the batches are done with the scratch)
    if (!SPL && sub == 0) {
#pragma unroll
        for (int gq = 0; gq < G; ++gq)
            *reinterpret_cast<float4*>(row_out + c + gq * W::GOFF) = make_float4(acc0[4 * gq], acc0[4 * gq + 1], acc0[4 * gq + 2], acc0[4 * gq + 3]);
    }
#pragma unroll
    for (int off = W::JW; off < 32; off <<= 1) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            accJ[k].x += __shfl_xor_sync(kFull, accJ[k].x, off);
            accJ[k].y += __shfl_xor_sync(kFull, accJ[k].y, off);
        }
    }
    if (eg == 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float* o = row_out + a.d.offA[1] + j_out[h];
            const float v[4] = {accJ[2 * h].x, accJ[2 * h].y, accJ[2 * h + 1].x, accJ[2 * h + 1].y};
            if (j_n[h] == 4 && !swapped) *reinterpret_cast<float4*>(o) = make_float4(v[0], v[1], v[2], v[3]);
            else {
#pragma unroll
                for (int k = 0; k < 4; ++k) if (k < j_n[h]) o[k] = v[k];
            }
        }
    }
    if (MODES == kMoments) {
        float* const out = a.moments + (size_t)(i - a.a0) * a.n_moments;
        for (int v = lane; v < a.n_moments; v += 32) out[v] = mom[v];
    }
    if (SPL) {
        float* const out = a.moments + (size_t)(i - a.a0) * a.n_moments;
        const float *p1 = mom + a.n_moments, *p2 = p1 + a.n_moments, *p3 = p2 + a.n_moments;
        for (int v = lane; v < a.n_moments; v += 32) out[v] = (mom[v] + p1[v]) + (p2[v] + p3[v]);
    }
    if (SPLIT) {
        if (lane == 0) { s_part[wid][0] = s0; s_part[wid][1] = s1; }
        __syncthreads();
        for (int v = threadIdx.x; v < C0 + W::NHI; v += kWarpsPerBlock * 32) {      // (S = C0 + NHI)
            float t = scratch[0][v];
#pragma unroll
            for (int w = 1; w < kWarpsPerBlock; ++w) t += scratch[w][v];
            row_glob[v] = t;
        }
        if (threadIdx.x == 0) {
#pragma unroll
            for (int w = 1; w < kWarpsPerBlock; ++w) { s0 += s_part[w][0]; s1 += s_part[w][1]; }
        }
    }
    if (SPLIT ? threadIdx.x == 0 : lane == 0) {
        const float h0 = (float)s0, h1 = (float)s1;
        row_glob[a.d.S] = h0; row_glob[a.d.S + 1] = h1;
        row_glob[a.d.S + 2] = (float)(s0 - (double)h0); row_glob[a.d.S + 3] = (float)(s1 - (double)h1);
    }
}

// ------------------------------------------------------------------------------ backward
//
// Same scan, queue and phases.  The channel-parallel phase produces, per edge, the two
// degree-0 dot products sum_c G0_c psi_c and sum_c G0_c dpsi_c (partial sums parked in shared
// memory and finished by the edge's own lane) and parks psi, dpsi of the leading C1 channels;
// the edge's lane then does the whole degree >= 1 contraction by itself against the
// destination's gradient block held in shared memory, and assembles dE/dr_ij.  Edges in the
// skin shell get a zero gradient as soon as their geometry is known.
// MODES == kMoments: beta and the modes enter the scalar channels through the row's H = (beta | U) G_0 (moments.cu).
template <int C0, int L, int MODES, bool UNI, bool FEW, bool SPLIT>
__global__ void __launch_bounds__(kWarpsPerBlock * 32, BwdShape<C0, L, MODES, UNI, FEW>::warps / kWarpsPerBlock)
k_edge_backward(const EdgeArgs a) {
    using SM = BwdSmem<C0, L, MODES, UNI>;
    constexpr int G = BwdShape<C0, L, MODES, UNI, FEW>::G;
    constexpr bool PR = SM::products, HASR = MODES == kModesPerEdge || MODES == kMoments, SPL = MODES == kSplines;
    using W = Widths<C0, L, G>;
    extern __shared__ __align__(16) unsigned char dsm[];
    double (*vsum)[9] = reinterpret_cast<double (*)[9]>(dsm);
    chain_begin();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float* const wbase = reinterpret_cast<float*>(dsm + kWarpsPerBlock * 9 * sizeof(double)) + wid * SM::per_warp;
    float* const psi_s = wbase;                                  // [32][PB]: psi, dpsi of the leading channels
    float* const red = psi_s + 32 * W::PB;                       // [n_red][32][LH+1] partial dot products
    float* const hi_s = red + SM::n_red * 32 * (W::LH + 1);   // [NHI] gradient of the degree >= 1 sums
    // queue of edges inside the cutoff: (row, pair, t, chi), then dx, dy, dz, dchi, edge index
    int4* const qes = reinterpret_cast<int4*>(wbase + SM::per_warp - SM::queue_floats);
    float* const qm = reinterpret_cast<float*>(qes) - SM::mode_floats;   // [2][32][kMaxR]
    float* const qd = reinterpret_cast<float*>(qes + 32);        // [5][32]
    float* const mom = reinterpret_cast<float*>(dsm + SM::bytes) + (MODES == kMoments || SPL ? wid * a.n_moments : 0);   // [n_moments]
    const int i = a.a0 + (SPLIT ? blockIdx.x : blockIdx.x * kWarpsPerBlock + wid);
    const bool active = i < a.a1;
    const int sub = lane / W::LPE, cl = lane % W::LPE, c = 4 * cl;
    const unsigned lt_mask = (1u << lane) - 1u;
    float vir[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) vir[k] = 0.f;

    if (active) {
        const int4 ci = __ldg(a.fix + i);
        const int ti = UNI && a.species_slot ? a.species_slot[ci.w] : ci.w;
        // steps of the packed words: of the table with derivatives, or of the value and the product table
        const float k2 = UNI ? tab_step2(__ldg(a.uni_scale + (PR ? 2 : 0))) : (PR ? a.d.tab_v1 : a.d.tab_k2),
                    k3 = UNI ? tab_step3(__ldg(a.uni_scale + (PR ? 3 : 1))) : (PR ? a.d.tab_v2 : a.d.tab_k3);
        const float d1 = UNI ? tab_step2(__ldg(a.uni_scale + 4)) : a.d.tab_d1, d2 = UNI ? tab_step3(__ldg(a.uni_scale + 5)) : a.d.tab_d2;
        eidx_t e0 = a.row_ptr[i];
        int len = (int)(a.row_ptr[i + 1] - e0);
        if (SPLIT) quarter_of_row(wid, &e0, &len);
        const int* Hf = a.frames ? a.frames[a.frame_of[i]].Hq : nullptr;
        const float* grow = a.state + (size_t)(i - a.a0) * a.d.SP;
        float h0[4 * G];
#pragma unroll
        for (int gq = 0; gq < (SPL ? 0 : G); ++gq) {
            const float4 v = *reinterpret_cast<const float4*>(grow + c + gq * W::GOFF);
            h0[4 * gq] = v.x; h0[4 * gq + 1] = v.y; h0[4 * gq + 2] = v.z; h0[4 * gq + 3] = v.w;
        }
        for (int v = lane; v < W::NHI; v += 32) hi_s[v] = grow[a.d.offA[1] + v];
        if (MODES == kMoments || SPL)
            for (int v = lane; v < a.n_moments; v += 32) mom[v] = a.moments[(size_t)(i - a.a0) * a.n_moments + v];
        const float ds0 = grow[a.d.S], ds1 = grow[a.d.S + 1];
        __syncwarp();
        const float* H1 = hi_s;
        const float* H2 = H1 + 3 * W::C1;
        const float* H3 = H2 + 5 * W::C2;
        const float* H4 = H3 + (L >= 3 ? 7 : 0);

        auto run_batch = [&](const int nb) {     // the first nb queue slots
            if (HASR) {
                eval_modes<PR ? kProducts : kDerivatives, kMaxR>(a, qes, nb, lane, qm, qm + 32 * kMaxR);
                __syncwarp();
            }
            if constexpr (PR) {
                // the leading channels' amplitudes, four channels of an edge per lane
                constexpr int LE = 32 / W::NL1;             // edges per step
                for (int b0 = 0; b0 < nb; b0 += LE) {
                    const int b = b0 + lane / W::NL1, cc = 4 * (lane % W::NL1);
                    if (b < nb) {
                        const int4 es = qes[b];
                        const float t = __int_as_float(es.z);
                        float psi[4];
                        if constexpr (SPL) {                       // and their products
                            float d[4];
                            value_eval4(a.vtable_uni, C0, es.x, cc, t, k2, k3, psi);
                            value_eval4(a.dtable_uni, C0, es.x, cc, t, d1, d2, d);
                            *reinterpret_cast<float4*>(psi_s + b * W::PB + W::C1 + cc) = make_float4(d[0], d[1], d[2], d[3]);
                        } else if constexpr (MODES == kMoments) {  // the same, from the same pair rows
                            float d[4];
                            const float* pm = a.pairmod + (size_t)es.y * (2 + a.d.R) * C0 + cc;
                            const float dchi = qd[96 + b];
                            value_eval4(a.vtable, a.d.CP, es.x, cc, t, k2, k3, psi);
                            value_eval4(a.dtable, a.d.CP, es.x, cc, t, d1, d2, d);
                            const float4 ga = ldg4(pm), be = ldg4(pm + C0);
                            affine4(ga, be, psi);
                            affine4(ga, scaled(dchi, be), d);
                            const float *qv = qm + b * kMaxR, *dq = qm + (32 + b) * kMaxR;
#pragma unroll
                            for (int m = 0; m < kMaxR; ++m) {
                                if (m >= a.d.R) break;
                                const float4 U = ldg4(pm + (size_t)(2 + m) * C0);
                                axpy4(qv[m], U, psi);
                                axpy4(dq[m], U, d);
                            }
                            *reinterpret_cast<float4*>(psi_s + b * W::PB + W::C1 + cc) = make_float4(d[0], d[1], d[2], d[3]);
                        } else {
                            amplitude4<C0, HASR, false, UNI>(a, es.x, t, es.y, cc, psi, nullptr, qm + b * kMaxR, nullptr, k2, k3);
                        }
                        *reinterpret_cast<float4*>(psi_s + b * W::PB + cc) = make_float4(psi[0], psi[1], psi[2], psi[3]);
                    }
                }
                // all channels: sum_c G_c (chi psi_c)'
                for (int it = 0; !SPL && it * W::EPI < nb; ++it) {
                    const int b = it * W::EPI + sub;
                    const bool act = b < nb;
                    float2 p2 = make_float2(0.f, 0.f);
                    if (act) {
                        const int4 es = qes[b];
                        const float t = __int_as_float(es.z), dchi = UNI ? 0.f : qd[96 + b];
#pragma unroll
                        for (int gq = 0; gq < G; ++gq) {
                            float d[4];
                            product4<C0, MODES, UNI>(a, es.x, t, es.y, c + gq * W::GOFF, dchi, qm + (32 + b) * kMaxR, d1, d2, d);
                            p2 = ffma2(make_float2(h0[4 * gq], h0[4 * gq + 1]), make_float2(d[0], d[1]), p2);
                            p2 = ffma2(make_float2(h0[4 * gq + 2], h0[4 * gq + 3]), make_float2(d[2], d[3]), p2);
                            // the leading C1 channels all sit in group 0
                            if (MODES != kMoments && gq == 0 && cl < W::NL1)
                                *reinterpret_cast<float4*>(psi_s + b * W::PB + W::C1 + c) = make_float4(d[0], d[1], d[2], d[3]);
                        }
                    }
                    // neighbouring lanes are paired before the partial sums are parked, which halves
                    // the parking area (it decides how many blocks fit on an SM)
                    float pa = p2.x + p2.y;
                    pa += __shfl_xor_sync(kFull, pa, 1);
                    if (act && !(cl & 1)) red[b * (W::LH + 1) + (cl >> 1)] = pa;
                }
            } else {
                for (int it = 0; it * W::EPI < nb; ++it) {
                    const int b = it * W::EPI + sub;
                    const bool act = b < nb;
                    float pa = 0.f, pb = 0.f;
                    if (act) {
                        const int4 es = qes[b];
                        const int row = es.x, pair = es.y;
                        const float t = __int_as_float(es.z);
                        float psi[4 * G], dpsi[4 * G];
    #pragma unroll
                        for (int gq = 0; gq < G; ++gq)
                            amplitude4<C0, HASR, true, UNI>(a, row, t, pair, c + gq * W::GOFF, psi + 4 * gq, dpsi + 4 * gq,
                                                            qm + b * kMaxR, qm + (32 + b) * kMaxR, k2, k3);
    #pragma unroll
                        for (int k = 0; k < 4 * G; ++k) { pa += h0[k] * dpsi[k]; pb += h0[k] * psi[k]; }
                        if (cl < W::NL1) {       // the leading C1 channels all sit in group 0
                            *reinterpret_cast<float4*>(psi_s + b * W::PB + c) = make_float4(psi[0], psi[1], psi[2], psi[3]);
                            *reinterpret_cast<float4*>(psi_s + b * W::PB + W::C1 + c) = make_float4(dpsi[0], dpsi[1], dpsi[2], dpsi[3]);
                        }
                    }
                    // neighbouring lanes are paired before the partial sums are parked, which halves
                    // the parking area (it decides how many blocks fit on an SM)
                    pa += __shfl_xor_sync(kFull, pa, 1);
                    pb += __shfl_xor_sync(kFull, pb, 1);
                    if (act && !(cl & 1)) {
                        red[b * (W::LH + 1) + (cl >> 1)] = pa;
                        red[(32 + b) * (W::LH + 1) + (cl >> 1)] = pb;
                    }
                }
            }
            __syncwarp();
            if (lane < nb) {
                const float gdx = qd[lane], gdy = qd[32 + lane], gdz = qd[64 + lane], dchi = qd[96 + lane];
                const int e = __float_as_int(qd[128 + lane]);       // offset inside the warp's part of the row
                const float chi = __int_as_float(qes[lane].w);
                const float inv_rho = 1.0f / sqrtf(gdx * gdx + gdy * gdy + gdz * gdz + kEpsReg * kEpsReg);
                const float gux = gdx * inv_rho, guy = gdy * inv_rho, guz = gdz * inv_rho;
                float sa = 0.f, sb = 0.f;
#pragma unroll
                for (int j = 0; !SPL && j < W::LH; ++j) {
                    sa += red[lane * (W::LH + 1) + j];
                    if (!PR) sb += red[(32 + lane) * (W::LH + 1) + j];
                }
                // degrees >= 1: t_lm = sum_c psi_c G_lmc (for the harmonics' gradient), bt = sum_lm B_lm t_lm and
                // pr1 = sum_lm B_lm sum_c dps_c G_lmc.  By component, all channels in registers; where the registers are
                // few (BwdShape), by four channels, which keeps the components' sums instead: 0.94 against 1.02 ms for
                // the 128,000 atoms of five species, but 1.12 against 1.10 at 128 registers.
                if (SPL) {           // (chi S)' of the spline of the row's coefficients
                    float t, u6[7], u7[8], v = 0.f, dv = 0.f;
                    const float* const h = mom + spline_interval(a, __int_as_float(qes[lane].y), &t);
                    spline_basis(t, u6, u7);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float hj = h[j];
                        v = fmaf(hj, u7[j], v);
                        dv = fmaf(hj, j == 0 ? -u6[0] : (j == 7 ? u6[6] : u6[j - 1] - u6[j]), dv);
                    }
                    sa = dchi * v + chi * (7.0f * a.spline_inv_h) * dv;
                }
                if (MODES == kMoments) {
                    const float* hr = mom + (qes[lane].y - ti * a.d.T) * (1 + a.d.R);
                    sa += dchi * hr[0];
#pragma unroll
                    for (int q = 0; q < kMaxR; ++q) if (q < a.d.R) sa += qm[(32 + lane) * kMaxR + q] * hr[1 + q];
                }
                float B1[3], B2[5], B3[7], B4[9], t1[3], t2[5], t3[7], t4[9];
                harmonics_s1<L>(gux, guy, guz, B1, B2, B3, B4);
                float bt = 0.f, pr1 = 0.f;
                if constexpr (BwdShape<C0, L, MODES, UNI, FEW>::tight) {
                    const float* pr = psi_s + lane * W::PB;
#pragma unroll
                    for (int m = 0; m < 3; ++m) t1[m] = 0.f;
#pragma unroll
                    for (int m = 0; m < 5; ++m) t2[m] = 0.f;
#pragma unroll
                    for (int m = 0; m < 7; ++m) t3[m] = 0.f;
#pragma unroll
                    for (int m = 0; m < 9; ++m) t4[m] = 0.f;
#pragma unroll
                    for (int q = 0; q < W::C1 / 4; ++q) {
                        const float4 p = *reinterpret_cast<const float4*>(pr + 4 * q), d = *reinterpret_cast<const float4*>(pr + W::C1 + 4 * q);
#pragma unroll
                        for (int m = 0; m < 3; ++m) {
                            const float4 hv = *reinterpret_cast<const float4*>(H1 + m * W::C1 + 4 * q);
                            t1[m] += p.x * hv.x + p.y * hv.y + p.z * hv.z + p.w * hv.w;
                            pr1 += B1[m] * (d.x * hv.x + d.y * hv.y + d.z * hv.z + d.w * hv.w);
                        }
                        if (4 * q < W::C2) {
#pragma unroll
                            for (int m = 0; m < 5; ++m) {
                                const float4 hv = *reinterpret_cast<const float4*>(H2 + m * W::C2 + 4 * q);
                                t2[m] += p.x * hv.x + p.y * hv.y + p.z * hv.z + p.w * hv.w;
                                pr1 += B2[m] * (d.x * hv.x + d.y * hv.y + d.z * hv.z + d.w * hv.w);
                            }
                        }
                        if (q == 0 && L >= 3) {
#pragma unroll
                            for (int m = 0; m < 7; ++m) { const float hv = H3[m]; t3[m] = p.x * hv; pr1 += B3[m] * (d.x * hv); }
                        }
                        if (q == 0 && L >= 4) {
#pragma unroll
                            for (int m = 0; m < 9; ++m) { const float hv = H4[m]; t4[m] = p.x * hv; pr1 += B4[m] * (d.x * hv); }
                        }
                    }
#pragma unroll
                    for (int m = 0; m < 3; ++m) bt += B1[m] * t1[m];
#pragma unroll
                    for (int m = 0; m < 5; ++m) bt += B2[m] * t2[m];
                    if (L >= 3) {
#pragma unroll
                        for (int m = 0; m < 7; ++m) bt += B3[m] * t3[m];
                    }
                    if (L >= 4) {
#pragma unroll
                        for (int m = 0; m < 9; ++m) bt += B4[m] * t4[m];
                    }
                } else if constexpr (C0 >= 128) {      // pairs of channels (narrower ones were 1 % slower that way)
                    float2 ps[W::C1 / 2], dps[W::C1 / 2], ec[W::C1 / 2], pr2 = make_float2(0.f, 0.f);
#pragma unroll
                    for (int q = 0; q < W::C1 / 4; ++q) {
                        const float4 p4 = *reinterpret_cast<const float4*>(psi_s + lane * W::PB + 4 * q);
                        const float4 d4 = *reinterpret_cast<const float4*>(psi_s + lane * W::PB + W::C1 + 4 * q);
                        ps[2 * q] = lo2(p4); ps[2 * q + 1] = hi2(p4);
                        dps[2 * q] = lo2(d4); dps[2 * q + 1] = hi2(d4);
                    }
#pragma unroll
                    for (int k = 0; k < W::C1 / 2; ++k) ec[k] = make_float2(0.f, 0.f);
#pragma unroll
                    for (int m = 0; m < 3; ++m) {
                        float2 tm = make_float2(0.f, 0.f);
#pragma unroll
                        for (int k = 0; k < W::C1 / 2; ++k) {
                            const float2 hv = *reinterpret_cast<const float2*>(H1 + m * W::C1 + 2 * k);
                            tm = ffma2(ps[k], hv, tm); ec[k] = ffma2(both(B1[m]), hv, ec[k]);
                        }
                        t1[m] = tm.x + tm.y; bt += B1[m] * t1[m];
                    }
#pragma unroll
                    for (int m = 0; m < 5; ++m) {
                        float2 tm = make_float2(0.f, 0.f);
#pragma unroll
                        for (int k = 0; k < W::C2 / 2; ++k) {
                            const float2 hv = *reinterpret_cast<const float2*>(H2 + m * W::C2 + 2 * k);
                            tm = ffma2(ps[k], hv, tm); ec[k] = ffma2(both(B2[m]), hv, ec[k]);
                        }
                        t2[m] = tm.x + tm.y; bt += B2[m] * t2[m];
                    }
#pragma unroll
                    for (int m = 0; m < 7; ++m) {
                        float tm = 0.f;
                        if (L >= 3) { const float hv = H3[m]; tm = ps[0].x * hv; ec[0].x += B3[m] * hv; bt += B3[m] * tm; }
                        t3[m] = tm;
                    }
#pragma unroll
                    for (int m = 0; m < 9; ++m) {
                        float tm = 0.f;
                        if (L >= 4) { const float hv = H4[m]; tm = ps[0].x * hv; ec[0].x += B4[m] * hv; bt += B4[m] * tm; }
                        t4[m] = tm;
                    }
#pragma unroll
                    for (int k = 0; k < W::C1 / 2; ++k) pr2 = ffma2(ec[k], dps[k], pr2);
                    pr1 = pr2.x + pr2.y;
                } else {
                    float ps[W::C1], dps[W::C1], ec[W::C1];
#pragma unroll
                    for (int q = 0; q < W::C1 / 4; ++q) {
                        const float4 p4 = *reinterpret_cast<const float4*>(psi_s + lane * W::PB + 4 * q);
                        const float4 d4 = *reinterpret_cast<const float4*>(psi_s + lane * W::PB + W::C1 + 4 * q);
                        ps[4 * q] = p4.x; ps[4 * q + 1] = p4.y; ps[4 * q + 2] = p4.z; ps[4 * q + 3] = p4.w;
                        dps[4 * q] = d4.x; dps[4 * q + 1] = d4.y; dps[4 * q + 2] = d4.z; dps[4 * q + 3] = d4.w;
                    }
#pragma unroll
                    for (int k = 0; k < W::C1; ++k) ec[k] = 0.f;
#pragma unroll
                    for (int m = 0; m < 3; ++m) {
                        float tm = 0.f;
#pragma unroll
                        for (int k = 0; k < W::C1; ++k) { const float hv = H1[m * W::C1 + k]; tm += ps[k] * hv; ec[k] += B1[m] * hv; }
                        t1[m] = tm; bt += B1[m] * tm;
                    }
#pragma unroll
                    for (int m = 0; m < 5; ++m) {
                        float tm = 0.f;
#pragma unroll
                        for (int k = 0; k < W::C2; ++k) { const float hv = H2[m * W::C2 + k]; tm += ps[k] * hv; ec[k] += B2[m] * hv; }
                        t2[m] = tm; bt += B2[m] * tm;
                    }
#pragma unroll
                    for (int m = 0; m < 7; ++m) {
                        float tm = 0.f;
                        if (L >= 3) { const float hv = H3[m]; tm = ps[0] * hv; ec[0] += B3[m] * hv; bt += B3[m] * tm; }
                        t3[m] = tm;
                    }
#pragma unroll
                    for (int m = 0; m < 9; ++m) {
                        float tm = 0.f;
                        if (L >= 4) { const float hv = H4[m]; tm = ps[0] * hv; ec[0] += B4[m] * hv; bt += B4[m] * tm; }
                        t4[m] = tm;
                    }
#pragma unroll
                    for (int k = 0; k < W::C1; ++k) pr1 += ec[k] * dps[k];
                }
                const float w = chi * chi;
                float ux, uy, uz;
                harmonics_grad_contract<L>(gux, guy, guz, t1, t2, t3, t4, &ux, &uy, &uz);
                const float pux = w * ux, puy = w * uy, puz = w * uz;
                float dEdrho;
                if (PR) {        // sa = sum_c G_c (chi psi_c)', dps = (chi psi)'
                    dEdrho = sa + chi * (pr1 + dchi * bt) + (2.0f * chi * ds0 + 4.0f * w * chi * ds1) * dchi;
                } else {         // sa = sum_c G_c psi_c', sb = sum_c G_c psi_c, dps = psi'
                    const float p_rho = chi * sa + w * pr1;
                    const float p_chi = sb + 2.0f * chi * bt;
                    dEdrho = p_rho + (p_chi + 2.0f * chi * ds0 + 4.0f * w * chi * ds1) * dchi;
                }
                const float dot = pux * gux + puy * guy + puz * guz;
                const float gx = dEdrho * gux + (pux - dot * gux) * inv_rho;
                const float gy = dEdrho * guy + (puy - dot * guy) * inv_rho;
                const float gz = dEdrho * guz + (puz - dot * guz) * inv_rho;
                vir[0] += gx * gdx; vir[1] += gx * gdy; vir[2] += gx * gdz;
                vir[3] += gy * gdx; vir[4] += gy * gdy; vir[5] += gy * gdz;
                vir[6] += gz * gdx; vir[7] += gz * gdy; vir[8] += gz * gdz;
                float* go = a.g + 3 * (size_t)(e0 + e);
                go[0] = gx; go[1] = gy; go[2] = gz;
            }
            __syncwarp();
        };

        int qn = 0;
        for (int base = 0; base < len; base += 32) {
            const int e = base + lane;
            const Geom g = edge_geometry<PR>(a, e0 + e, e < len, ci, ti, Hf);
            const unsigned vmask = __ballot_sync(kFull, g.valid);
            const int p = qn + __popc(vmask & lt_mask);   // queue slot of this lane's edge, if it has one
            if (g.valid && p < 32) {
                qes[p] = make_int4(g.row, SPL ? __float_as_int(g.rho) : g.pair, __float_as_int(g.t), __float_as_int(g.chi));
                qd[p] = g.dx; qd[32 + p] = g.dy; qd[64 + p] = g.dz; qd[96 + p] = g.dchi;
                qd[128 + p] = __int_as_float(e);
            } else if (!g.valid && e < len) {
                float* go = a.g + 3 * (size_t)(e0 + e);
                go[0] = 0.f; go[1] = 0.f; go[2] = 0.f;
            }
            qn += __popc(vmask);
            __syncwarp();
            if (qn >= 32) {                               // a full batch; the overflow waits in registers
                run_batch(32);
                if (g.valid && p >= 32) {
                    const int r = p - 32;
                    qes[r] = make_int4(g.row, SPL ? __float_as_int(g.rho) : g.pair, __float_as_int(g.t), __float_as_int(g.chi));
                    qd[r] = g.dx; qd[32 + r] = g.dy; qd[64 + r] = g.dz; qd[96 + r] = g.dchi;
                    qd[128 + r] = __int_as_float(e);
                }
                qn -= 32;
                __syncwarp();
            }
        }
        if (qn > 0) run_batch(qn);
    }
    // block partial of sum_e g (x) r, in double, fixed order: eight components change lanes in halves, so that
    // lane 4 k ends with the sum of component k; the ninth goes through every step
    double v9 = (double)vir[8], v8[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v8[k] = (double)vir[k];
#pragma unroll
    for (int n = 4, off = 16; n >= 1; n >>= 1, off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int k = 0; k < n; ++k) {
            const double send = up ? v8[k] : v8[k + n], mine = up ? v8[k + n] : v8[k];
            v8[k] = mine + __shfl_xor_sync(kFull, send, off);
        }
    }
    v8[0] += __shfl_xor_sync(kFull, v8[0], 2);
    v8[0] += __shfl_xor_sync(kFull, v8[0], 1);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v9 += __shfl_xor_sync(kFull, v9, off);
    if ((lane & 3) == 0) vsum[wid][lane >> 2] = v8[0];
    if (lane == 0) vsum[wid][8] = v9;
    __syncthreads();
    if (threadIdx.x < 9) {
        double v = 0.0;
        for (int w = 0; w < kWarpsPerBlock; ++w) v += vsum[w][threadIdx.x];
        a.virial_part[(size_t)blockIdx.x * 9 + threadIdx.x] = v;
    }
}


// per-pair amplitude tables already hold the modes, so the kernels without them are used
// (The limit of dynamic shared memory belongs to the kernel, whichever thread and model launches it: always the largest that
// any model takes, so that one thread's cannot come between another's limit and launch.)
template <int C0, int L, bool SPLIT>
cudaError_t launch_fwd_r(const EdgeArgs& a, int blocks, cudaStream_t st) {
    auto kern = a.uni ? k_edge_forward<C0, L, kNoModes, true, SPLIT>
                      : (a.d.R > 0 ? k_edge_forward<C0, L, kModesPerEdge, false, SPLIT> : k_edge_forward<C0, L, kNoModes, false, SPLIT>);
    if constexpr (C0 >= 64 && !SPLIT) {
        if (a.spline_n) {
            kern = k_edge_forward<C0, L, kSplines, true, false>;
            const size_t bytes = sizeof(float) * kWarpsPerBlock * 4 * a.n_moments;
            const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(float) * kWarpsPerBlock * 4 * kMaxSplinePitch));
            if (e != cudaSuccess) return e;
            kern<<<blocks, kWarpsPerBlock * 32, bytes, st>>>(a);
            return cudaGetLastError();
        }
    }
    if constexpr (wide_channels(C0) && !SPLIT) {
        if (a.moments) {
            kern = k_edge_forward<C0, L, kMoments, false, false>;
            const size_t bytes = sizeof(float) * kWarpsPerBlock * a.n_moments;
            const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(float) * kWarpsPerBlock * kMaxMoments));
            if (e != cudaSuccess) return e;
            kern<<<blocks, kWarpsPerBlock * 32, bytes, st>>>(a);
            return cudaGetLastError();
        }
    }
    kern<<<blocks, kWarpsPerBlock * 32, 0, st>>>(a);
    return cudaGetLastError();
}
template <int C0, int L, int MODES, bool UNI>
cudaError_t launch_bwd_r(const EdgeArgs& a, int blocks, bool split, cudaStream_t st) {
    const bool few = a.a1 - a.a0 > 148 * 24 && a.a1 - a.a0 <= 148 * 32;
    constexpr bool FEW = C0 <= 64 && MODES < kMoments;           // (the others have no such variant)
    size_t bytes = BwdSmem<C0, L, MODES, UNI>::bytes;
    auto kern = few ? k_edge_backward<C0, L, MODES, UNI, FEW, false> : k_edge_backward<C0, L, MODES, UNI, false, false>;
    size_t most = bytes;
    if constexpr (MODES >= kMoments) {
        most += sizeof(float) * kWarpsPerBlock * (MODES == kSplines ? kMaxSplinePitch : kMaxMoments);
        bytes += sizeof(float) * kWarpsPerBlock * a.n_moments;
    } else if (split) kern = k_edge_backward<C0, L, MODES, UNI, false, true>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (e != cudaSuccess) return e;
    kern<<<blocks, kWarpsPerBlock * 32, bytes, st>>>(a);
    return cudaGetLastError();
}
template <bool FWD, int C0, int L>
cudaError_t launch(const EdgeArgs& a, int blocks, bool split, cudaStream_t st) {
    if (FWD) return split ? launch_fwd_r<C0, L, true>(a, blocks, st) : launch_fwd_r<C0, L, false>(a, blocks, st);
    if constexpr (C0 >= 64) {
        if (a.spline_n) return launch_bwd_r<C0, L, kSplines, true>(a, blocks, false, st);
    }
    if (a.uni) return launch_bwd_r<C0, L, kNoModes, true>(a, blocks, split, st);
    if constexpr (wide_channels(C0)) {
        if (a.moments) return launch_bwd_r<C0, L, kMoments, false>(a, blocks, false, st);
    }
    if (a.d.R > 0) return launch_bwd_r<C0, L, kModesPerEdge, false>(a, blocks, split, st);
    return launch_bwd_r<C0, L, kNoModes, false>(a, blocks, split, st);
}

template <bool FWD>
cudaError_t dispatch(const EdgeArgs& a, cudaStream_t st) {
    const int rows = a.a1 - a.a0, blocks = edge_blocks(rows);
    const bool split = edge_rows_split(rows);
#define UMLMD_CASE(C0v, Lv) \
    if (a.d.C0 == C0v && a.d.L == Lv) return launch<FWD, C0v, Lv>(a, blocks, split, st);
    UMLMD_CASE(8, 2) UMLMD_CASE(8, 3) UMLMD_CASE(16, 2) UMLMD_CASE(16, 3) UMLMD_CASE(32, 2)
    UMLMD_CASE(32, 3) UMLMD_CASE(64, 2) UMLMD_CASE(64, 3) UMLMD_CASE(128, 2) UMLMD_CASE(128, 3)
    UMLMD_CASE(8, 4) UMLMD_CASE(16, 4) UMLMD_CASE(32, 4) UMLMD_CASE(64, 4) UMLMD_CASE(128, 4)
#undef UMLMD_CASE
    return cudaErrorInvalidValue;
}

// Tables of psi_c(rho) = gamma_c g_c(rho) + beta_c + sum_mu U_c,mu q_mu(rho) for the ordered
// pairs (present[a], present[b]), stored as [a * n_present + b][row][3][C0] (below C0 = 32) in the format of the
// radial table: the cubic coefficients are linear in the tabulated functions, so the same
// combination of the coefficient rows of [g, q] gives them; and as [..][n_vrows][2][C0] in those of the
// value and product tables.  Two passes: the first finds the largest magnitudes of the coefficients that are packed (the scale
// of the words), the second writes the rows.  A thread takes one channel of one row for kPairsPerThread pairs: the six
// maxima then meet in memory once per warp and that many pairs (with a thread per pair 25 pairs at C0 = 128 took 1.46 ms,
// most of it in atomics on six addresses, so 0.32).
constexpr int kPairsPerThread = 32;
template <bool WRITE>
__global__ void k_fuse_pair_tables(Dims d, const float* __restrict__ table, const float* __restrict__ pairmod,
                                   const int* __restrict__ present, int n_present, float* __restrict__ scale,
                                   float* __restrict__ out, float* __restrict__ vout, float* __restrict__ dout) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;                // over [row][c]
    const int first = blockIdx.y * kPairsPerThread, last = min(first + kPairsPerThread, n_present * n_present);
    float mx[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};       // |c2|, |c3|, |a1|, |a2| of the values, |a1|, |a2| of the products
    if (idx < d.n_rows * d.C0) {
        const int row = idx / d.C0, c = idx - row * d.C0;
        const float* tr = table + (size_t)row * 3 * d.CP;
        const double w = (double)d.dx / d.v_sub;
        for (int pr = first; pr < last; ++pr) {
            const int si = present[pr / n_present], sj = present[pr % n_present];
            double v[4];
            pair_cubic(d, tr, pairmod + (size_t)(si * d.T + sj) * (2 + d.R) * d.C0 + c, c, v);
            const float c2 = (float)v[2], c3 = (float)v[3];
            mx[0] = fmaxf(mx[0], fabsf(c2)); mx[1] = fmaxf(mx[1], fabsf(c3));
            for (int sub = 0; sub < d.v_sub; ++sub) {          // values alone (common.cuh, value_piece)
                double p[3];
                value_piece(v[0], v[1], v[2], v[3], (sub + 0.5) * w, 0.5 * w, p);
                mx[2] = fmaxf(mx[2], fabsf((float)p[1])); mx[3] = fmaxf(mx[3], fabsf((float)p[2]));
                if (WRITE) {
                    float* vrow = vout + ((size_t)pr * d.n_vrows + (size_t)row * d.v_sub + sub) * 2 * d.C0;
                    vrow[c] = (float)p[0];
                    vrow[d.C0 + c] = __uint_as_float(tab_pack((float)p[1], (float)p[2], tab_step2(scale[2]), tab_step3(scale[3])));
                }
                if (!wide_channels(d.C0)) continue;
                double q[4];                                   // envelope products (product_piece)
                double e[5];
                envelope_derivatives((double)row * d.dx + (sub + 0.5) * w, (double)d.rc, e);
                product_piece(v[0], v[1], v[2], v[3], (sub + 0.5) * w, 0.5 * w, e, q);
                mx[4] = fmaxf(mx[4], fabsf((float)q[1])); mx[5] = fmaxf(mx[5], fabsf((float)q[2]));
                if (WRITE) {
                    float* drow = dout + ((size_t)pr * d.n_vrows + (size_t)row * d.v_sub + sub) * 2 * d.C0;
                    drow[c] = (float)q[0];
                    drow[d.C0 + c] = __uint_as_float(tab_pack((float)q[1], (float)q[2], tab_step2(scale[4]), tab_step3(scale[5])));
                }
            }
            if (WRITE && !wide_channels(d.C0)) {
                float* orow = out + ((size_t)pr * d.n_rows + row) * 3 * d.C0;
                orow[c] = (float)v[0];
                orow[d.C0 + c] = (float)v[1];
                orow[2 * d.C0 + c] = __uint_as_float(tab_pack(c2, c3, tab_step2(scale[0]), tab_step3(scale[1])));
            }
        }
    }
    if (!WRITE) {        // non-negative floats order like their bit patterns
#pragma unroll
        for (int k = 0; k < 6; ++k) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) mx[k] = fmaxf(mx[k], __shfl_xor_sync(0xffffffffu, mx[k], off));
            if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<unsigned*>(scale) + k, __float_as_uint(mx[k]));
        }
    }
}

}  // namespace

cudaError_t launch_fuse_pair_tables(const Dims& d, const float* table, const float* pairmod, const int* present,
                                    int n_present, float* scale, float* out, float* vout, float* dout, cudaStream_t st) {
    const int n = d.n_rows * d.C0, pairs = n_present * n_present;
    if (n == 0 || pairs == 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(scale, 0, 6 * sizeof(float), st);
    if (e != cudaSuccess) return e;
    const dim3 blocks((unsigned)((n + 255) / 256), (unsigned)((pairs + kPairsPerThread - 1) / kPairsPerThread));
    k_fuse_pair_tables<false><<<blocks, 256, 0, st>>>(d, table, pairmod, present, n_present, scale, out, vout, dout);
    k_fuse_pair_tables<true><<<blocks, 256, 0, st>>>(d, table, pairmod, present, n_present, scale, out, vout, dout);
    return cudaGetLastError();
}

cudaError_t launch_edge_forward(const EdgeArgs& a, cudaStream_t st) {
    return a.a1 > a.a0 ? dispatch<true>(a, st) : cudaSuccess;
}

cudaError_t launch_edge_backward(const EdgeArgs& a, int* n_blocks, cudaStream_t st) {
    *n_blocks = edge_blocks(a.a1 - a.a0);
    return a.a1 > a.a0 ? dispatch<false>(a, st) : cudaSuccess;
}

}  // namespace umd
