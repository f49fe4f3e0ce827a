// Shared declarations of the library's translation units: structural widths, the
// device-resident model constants, the per-handle workspace and the kernel launchers.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstdio>
#include <string>
#include <vector>

#include "../../include/umlmd.h"

namespace umd {

constexpr float kEpsReg = 1.0e-7f;     // direction regulariser, Angstrom (edge geometry)
constexpr int kMaxDeg = 4;             // highest angular degree compiled in
constexpr int kMaxR = 8;               // most shared radial modes
constexpr int kMaxGaunt = 96;          // non-zeros kept per coupling tensor of the degree <= 3 triples
constexpr int kMaxGauntBig = 256;      // the same for the triples that involve degree 4 (up to 9 x 9 x 9 entries)
constexpr double kAccelUnit = 9648.53321;   // (eV/Angstrom/amu) in Angstrom/ps^2
constexpr double kBoltzmann = 8.617333262e-5;

// error word bits set by kernels (read back at synchronisation points)
enum : int { kErrStale = 1, kErrNonFinite = 2, kErrShiftRange = 8, kErrPipelineTimeout = 16, kErrSpecies = 32 };

// Widths derived from (C0, L, R): degree-wise channels, probe ranks, feature-state width
// S, feature-vector width D_out, gated hidden widths, and the flat offsets used by the
// kernels.  Host and device both read this struct (it is passed by value).
struct Dims {
    int C0, L, R, N_rbf, n_hidden, F, T;
    int C[kMaxDeg + 1];      // channels per degree
    int K[kMaxDeg + 1];      // probe ranks (index 0 unused)
    int S, SP;               // state width S; row stride SP >= S+4 (s0, s1 as float pairs), multiple of 4
    int offA[kMaxDeg + 1];   // offset of degree block in the state row
    int D_out, DP;           // feature-vector width; row stride (multiple of 32)
    int oG[kMaxDeg + 1];     // offsets of vech(G_l) in D
    int oJ112, oJ123, oJ222, oJ233, oPi;
    int oJ134, oJ224, oJ244, oJ334, oJ444;   // blocks of the triples that exist only for L = 4
    int H, Hp;
    int CP;                  // table channels C0+R rounded up to 4
    int n_rows;              // table intervals
    float tab_k2, tab_k3;    // steps of the packed quadratic and cubic coefficients of the radial table
    int v_sub, unused, n_vrows;    // value table (below): intervals per table interval (a power of two), and in all.  (The word
                             // between them holds the offsets behind it: with four bytes less the forward kernel at C0 = 8 came
                             // out 1.8 % slower, 216,000 atoms 9.74 -> 9.92 ms in a run of ten steps.)
    float vdx, inv_vdx;      // its spacing
    float tab_v1, tab_v2;    // steps of its packed linear and quadratic coefficients
    float tab_d1, tab_d2;    // the same for the product table
    float rc, dx, inv_dx;
};

struct GauntSparse {         // non-zeros of one unit-norm coupling tensor
    int n;
    unsigned char m1[kMaxGaunt], m2[kMaxGaunt], m3[kMaxGaunt];
    float v[kMaxGaunt];
};
struct GauntSparseBig {      // the same with room for the degree-4 triples
    int n;
    unsigned char m1[kMaxGauntBig], m2[kMaxGauntBig], m3[kMaxGauntBig];
    float v[kMaxGauntBig];
};

// Device-resident constants of one model.
struct ModelDev {
    float* table;     // [n_rows][3][CP] cubic Hermite pieces of [g, q]: c0, c1 (fp32), packed (c2, c3)
    float* vtable;    // [n_vrows][2][CP] quadratic pieces of [g, q] for their values alone: a0 (fp32), packed (a1, a2)
    float* dtable;    // [n_vrows][2][CP] the same format: derivative of envelope times g (C0 >= 32)
    float* pairmod;   // [T*T][2+R][C0]: scale gamma, shift beta, mode mixing U[:, mu]
    float* X0;        // [T][C0]
    float* W1p;       // [C1][C1]  I + W_1
    float* W2p;       // [C2][C2]  I + W_2
    float* A1;        // [C1][K1]
    float* A2;        // [C2][K2]
    float* mu;        // [D_out]
    float* inv_sigma; // [D_out]
    float* theta[8];  // Theta_t, row-major [K_in (padded)][F]; theta[0] has DP rows
    float* thetaT[8]; // transposes, [F][K_in (padded)]
    // half-precision split (x = hi + lo) of w_scale[t] * theta and of its transpose; w_scale[t] is
    // the power of two that brings the largest |weight| of the layer to [2^9, 2^10), so that the
    // low parts are normal half-precision numbers; w_scale_inv[t] undoes it on the accumulator
    __half* theta_hi[8];  __half* theta_lo[8];
    __half* thetaT_hi[8]; __half* thetaT_lo[8];
    float w_scale_inv[8];
    float grad_scale; // power of two the tensor-core backward chain multiplies its gradients by (from max |w_head|)
    float* bias[8];   // b_t [F]
    float* type_bias; // [T][F] first-layer bias with the centre's initial features folded in
    float* w_head;    // [F]
    float* e_ref;     // [T]
    float b_head;
    GauntSparse* g123;   // device copies (NULL when L < 3)
    GauntSparse* g233;
    GauntSparseBig* g4;  // [5] device copies of (1,3,4), (2,2,4), (2,4,4), (3,3,4), (4,4,4) (NULL when L < 4)
};

struct Handle;  // defined in api.cu

// ---- launchers (each enqueues on `st`; none synchronises) ---------------------------

typedef long long eidx_t;      // edge offsets are 64-bit: a list may hold more than 2^31 edges

// Packed high-order coefficients of a cubic table piece.  c2 and c3 only enter through c2 t^2 and
// c3 t^3 with t below the table spacing, so a 20-bit and a 12-bit fixed-point number on the table's
// own scale (c2 = k2 I2, c3 = k3 I3; k = largest magnitude in the table / largest integer) cost
// nothing in the value and leave the derivative within a few 1e-7 of its largest entry at the
// default spacing (the error grows with the spacing like the interpolation error itself).
// One 32-bit word: 4096 I2 + I3, two's complement.  The word as a whole, as a number, is 4096 times I2 + I3 / 4096, and I2 is
// rounded so that this is what represents c2: one conversion gives it (scale k2 / 4096), a shift and another one I3 (the
// lower 12 bits at the top of a word, scale k3 / 2^20), where the two parts as bit fields took two shifts more per channel.
// (A word whose parts decode without conversions, the low bits through the mantissa of 2^23, took an addition more and
// was 3 to 8 % slower in the forward kernel.)
constexpr int kTabI2Max = (1 << 19) - 2, kTabI3Max = (1 << 11) - 1;
constexpr float kTabHi = 1.0f / 4096.0f, kTabLo = 1.0f / 1048576.0f;     // scales of the two converted numbers, in units of k2 and k3
__host__ __device__ inline float tab_step2(float max_abs_c2) { return max_abs_c2 * (1.0f / (float)kTabI2Max); }
__host__ __device__ inline float tab_step3(float max_abs_c3) { return max_abs_c3 * (1.0f / (float)kTabI3Max); }
__host__ __device__ inline unsigned tab_pack(float c2, float c3, float k2, float k3) {
    // (no branch in it: the host packs rows of channels, several at a time)
    float q2 = c2 / (k2 > 0.f ? k2 : 1.f), q3 = c3 / (k3 > 0.f ? k3 : 1.f);      // (a step of zero has zeros to pack)
    q3 = q3 < (float)kTabI3Max ? q3 : (float)kTabI3Max; q3 = q3 > -(float)kTabI3Max ? q3 : -(float)kTabI3Max;
    const int i3 = (int)(q3 + copysignf(0.5f, q3));
    q2 -= (float)i3 * kTabHi;
    q2 = q2 < (float)kTabI2Max ? q2 : (float)kTabI2Max; q2 = q2 > -(float)kTabI2Max ? q2 : -(float)kTabI2Max;
    const int i2 = (int)(q2 + copysignf(0.5f, q2));
    return ((unsigned)i2 << 12) + (unsigned)i3;
}
__host__ __device__ inline float tab_hi(unsigned w) { return (float)(int)w; }
__host__ __device__ inline float tab_lo(unsigned w) { return (float)(int)(w << 20); }
__host__ __device__ inline void tab_unpack(unsigned w, float k2, float k3, float* c2, float* c3) {
    *c2 = (k2 * kTabHi) * tab_hi(w);
    *c3 = (k3 * kTabLo) * tab_lo(w);
}

// Value table.  A pass that needs no derivative reads two words per channel instead of three: the piece is
// expanded about the middle of the interval, p(s) = a0 + a1 s + a2 s^2 with |s| <= h = spacing / 2, a0 in
// single precision and (a1, a2) packed like (c2, c3) above.  The cubic term is folded into a1 (s^3 is within
// h^3 / 4 of (3/4) h^2 s); what is left of it, and the rounding of a1 and a2 to 20 and 12 bits, add up to less
// than half of the rounding of a0 at the default spacing (0.07 to 0.4 of 2^-24 of the largest value for the
// workloads' radial maps).  An interval is cut into v_sub pieces of at most 0.0025 Angstrom, and into more until
// they add up to no more than that rounding for g and q, and for their products (below, from C0 = 32 on, whichever
// table holds them) to no more than 2^-23 of the largest; once there are more than 100,000 pieces the table is cut no further.
__host__ __device__ inline void value_piece(double c0, double c1, double c2, double c3, double mid, double h, double* a) {
    a[0] = ((c3 * mid + c2) * mid + c1) * mid + c0;
    a[1] = (3 * c3 * mid + 2 * c2) * mid + c1 + 0.75 * h * h * c3;
    a[2] = 3 * c3 * mid + c2;
}

// Product table.  Of the scalar channels the backward pass needs one number per edge, sum_c G_c (chi psi_c)':
// the derivative of the product of envelope and amplitude is tabulated by itself, in the format and on the
// grid of the value table (expanded from the cubic piece and the envelope's derivatives, cubic term folded),
// two words per channel and one dot product instead of three words and two.  The leading C1 channels, which
// also carry the degrees >= 1, add their amplitude from the value table: (chi^2 psi)' = chi ((chi psi)' + chi' psi).
// chi = 1 - I_x(5, 4); e: its value and derivatives of order 1 .. 4 at rho.
__host__ __device__ inline void envelope_derivatives(double rho, double rc, double* e) {
    const double x = rho / rc, u = 1 - x, r = 1 / rc;
    e[0] = u * u * u * u * (1 + x * (4 + x * (10 + x * (20 + 35 * x))));
    e[1] = -280 * r * x * x * x * x * u * u * u;
    e[2] = -280 * r * r * x * x * x * u * u * (4 * u - 3 * x);
    e[3] = -280 * r * r * r * x * x * u * (12 * u * u - 24 * x * u + 6 * x * x);
    e[4] = -280 * r * r * r * r * x * (24 * u * u * u - 108 * x * u * u + 72 * x * x * u - 6 * x * x * x);
}
// e: at the middle of the piece
__host__ __device__ inline void product_piece(double c0, double c1, double c2, double c3, double mid, double h, const double* e, double* a) {
    const double p0 = ((c3 * mid + c2) * mid + c1) * mid + c0, p1 = (3 * c3 * mid + 2 * c2) * mid + c1, p2 = 6 * c3 * mid + 2 * c2, p3 = 6 * c3;
    const double d3 = (e[4] * p0 + 4 * e[3] * p1 + 6 * e[2] * p2 + 4 * e[1] * p3) / 6;
    a[0] = e[1] * p0 + e[0] * p1;
    a[1] = e[2] * p0 + 2 * e[1] * p1 + e[0] * p2 + 0.75 * h * h * d3;
    a[2] = 0.5 * (e[3] * p0 + 3 * e[2] * p1 + 3 * e[1] * p2 + e[0] * p3);
    a[3] = d3;
}
// The cubic piece of the amplitude psi_c = gamma_c g_c + beta_c + sum_mu U_c,mu q_mu of one species pair in one row of
// the radial table (linear in the tabulated functions): `row` that row, `pm` channel c of the pair's row in the cache.
__host__ __device__ inline void pair_cubic(const Dims& d, const float* row, const float* pm, int c, double* v) {
    for (int q = -1; q < d.R; ++q) {
        const int col = q < 0 ? c : d.C0 + q;
        unsigned w;
        memcpy(&w, row + 2 * d.CP + col, sizeof(w));
        float c2, c3;
        tab_unpack(w, d.tab_k2, d.tab_k3, &c2, &c3);
        const double o[4] = {(double)row[col], (double)row[d.CP + col], (double)c2, (double)c3};
        const double u = (double)pm[(size_t)(q < 0 ? 0 : 2 + q) * d.C0];
        for (int k = 0; k < 4; ++k) v[k] = q < 0 ? u * o[k] : v[k] + u * o[k];
        if (q < 0) v[0] += (double)pm[d.C0];
    }
}
// One spline coefficient of the amplitude psi_c of a pair from those of the radial map and modes: `coef` their row, `pm` channel c of
// the pair's row.  The basis functions add up to one; the kernels' are 7! times them.  *left: what the coefficient before has lost by
// rounding, which this one makes up for (a row's mean error over its channels 3e-9 of the sums, so 3e-10; by the tables it is 7e-10
// to 1e-9).
__host__ __device__ inline float spline_coefficient(const Dims& d, const double* coef, const float* pm, int c, double* left) {
    double v = (double)pm[0] * coef[c] + (double)pm[d.C0];
    for (int q = 0; q < d.R; ++q) v += (double)pm[(size_t)(2 + q) * d.C0] * coef[d.C0 + q];
    v = v / 5040 - *left;
    const float r = (float)v;
    *left = (double)r - v;
    return r;
}
// Models of at least 32 channels use the product table and none with derivatives.  At C0 = 8 and 16 a quarter or more of the
// channels are leading ones, which need both: there the table with derivatives is less to read.
__host__ __device__ constexpr bool wide_channels(int C0) { return C0 >= 32; }

// Positions for the edge kernels are whole multiples of a power of two q, kept modulo 2^32: an edge vector is an exact
// difference of integers (image offsets are whole multiples too), rounded once when it becomes single precision.  With R = 2^31 q
// beyond the list radius rc + skin a component up to that wraps to itself; the longest edge of a list that is not stale is rc + 2 skin,
// and what lies beyond R comes out as at least 2 R - (rc + 2 skin) > rc, outside the cutoff as it is.  Half a quantum is 1.9e-9 at
// a list radius of 6 or 7 Angstrom, where the rounding of a component between 1 and 8 to single precision is 6e-8 to 2.4e-7.
// The quantum grows with the list radius, and an image offset's rounding with the number of the image.  From a list radius of 16
// Angstrom on, and in cells so small that offsets could be 3e-8 off, every edge gets a record of its own instead, formed in double
// and in quanta for the cutoff (edge_records_needed, k_edge_records).
inline double position_quantum(double r_list) {
    int e;
    std::frexp(r_list, &e);
    return std::ldexp(1.0, e - 31);
}
constexpr double kEdgeRecordReach = 1.001;      // times the cutoff: where the records of edges beyond it are
inline bool edge_records_needed(double r_list, int images) {
    const double q = position_quantum(r_list);
    return q > 0x1p-27 || 0.5 * q * images > 0x1p-25;
}
__host__ __device__ inline int to_quanta(double x, double inv_q) {
#ifdef __CUDA_ARCH__
    return (int)__double2ll_rn(x * inv_q);
#else
    return (int)std::llrint(x * inv_q);
#endif
}

#ifdef __CUDACC__
// two multiply-adds in one instruction (the pipe takes as long as for two; the issue slot is one)
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
    float2 r;
    asm("{.reg .b64 x, y, z, w; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; mov.b64 z, {%6, %7}; fma.rn.f32x2 w, x, y, z; mov.b64 {%0, %1}, w;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
#endif

// One frame of a batched evaluation (umlmd_compute_batch): its own cell and its slice of the
// concatenated atom arrays.
struct FrameCell {
    double H[9];      // cell vectors as rows
    double Hinv[9];   // inverse (fractional coordinates f = r Hinv)
    double reach[3];  // cutoff in fractional coordinates along each cell vector, rounded up
    int Hq[9];        // cell vectors in position quanta (position_quantum), as rows
    float near_tol;   // band around the squared cutoff inside which the scan decides in double precision
    int m[3];         // periodic images to visit along each cell vector (0 for an open direction)
    int pbc[3];
    int a0, a1;       // atoms [a0, a1) of the concatenated arrays
};

struct NeighborDev {
    int64_t N = 0, E = 0, E_cap = 0, N_cap = 0;
    unsigned long long* bounds = nullptr;   // [6] scratch of the extent reduction (open directions)
    int64_t n_owned = 0, E_owned = 0;   // rows [0, n_owned) and edges [0, E_owned) belong to owned atoms (all of them without ghosts)
    double L[3] = {0, 0, 0};     // cell edge lengths (the diagonal of H)
    double H[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};   // cell vectors as rows
    int tri = 0;                 // the cell has off-diagonal components
    int pbc[3] = {1, 1, 1};
    double skin = 0, r_list = 0;
    double* wpos = nullptr;      // [N][3] folded positions, caller order (build time)
    int* img = nullptr;          // [N][3] floor(frac) per atom, sorted order
    int* perm = nullptr;         // [N] sorted index -> caller index
    int* type_s = nullptr;       // [N] species, sorted order
    double* xs0 = nullptr;       // [N][3] folded positions at build time, sorted order
    double* xs = nullptr;        // [N][3] current positions minus img*L, sorted order
    float4* rec = nullptr;       // [N] positions in single precision, what the list search reads
    // [N] current positions in quanta and the species, one 16-byte load per neighbour of the edge kernels.  x = q llrint(x / q)
    // modulo 2^32: differences of two coordinates wrap to the true one, whatever the size of the box (position_quantum)
    int4* fix = nullptr;
    double quantum = 1;
    // where `fix` is too coarse (edge_records_needed): a record for every row, at the origin, and for every edge, at its edge vector,
    // and a list that names them
    bool per_edge = false;
    int4* edge_fix = nullptr; int64_t edge_fix_cap = 0;
    int2* edge_nbr = nullptr; int64_t edge_nbr_cap = 0;
    eidx_t* row_ptr = nullptr;   // [N+1]
    int2* nbr = nullptr;         // [E] x: sorted index of the neighbour, y: its image n, packed int8 x3
    eidx_t* rev = nullptr;       // [E] index of the reverse edge, -1 if absent
    // batched evaluation: per-frame cells and the frame of every atom (null for a single system)
    FrameCell* frames = nullptr; int64_t frames_cap = 0; int n_frames = 0;
    int* frame_of = nullptr;
    bool batch = false;          // the list in here is the union of per-frame lists
    // scratch
    int* key = nullptr; int* key2 = nullptr; int* idx = nullptr; int* idx2 = nullptr;
    int* cell_start = nullptr; int64_t ncell_cap = 0;
    int* deg = nullptr;
    eidx_t* h_totals = nullptr;  // pinned [2], the caller's: edges in all, edges of owned atoms
    void* cub_tmp = nullptr; size_t cub_bytes = 0;
};

}  // namespace umd
