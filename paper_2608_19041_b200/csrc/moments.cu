// Shared radial modes by moments of the rows.
//
// Without per-pair tables the amplitude of an edge i -> j is psi_c = gamma_c g_c(rho) + beta_c + sum_mu U_c,mu q_mu(rho) with gamma,
// beta and U of the ordered species pair (t_i, t_j): an edge that reads these rows pulls 2 + R of them.  All but gamma g is a
// channel vector of the pair times a scalar of the edge, so over a row
//   sum_j chi_j (beta_c + sum_mu U_c,mu q_mu) = sum_t (beta^t_c m_t,0 + sum_mu U^t_c,mu m_t,mu),
//   m_t,0 = sum_{j of species t} chi_j,  m_t,mu = sum_{j of species t} chi_j q_mu(rho_j).
// The edge kernel leaves the T (1 + R) moments m of each row; here they meet the rows of the centre's species, once per row and
// not per edge, as a matrix product whose rows are grouped by species.  The backward pass forms H = (beta | U) G_0 the same way,
// and its edge kernel adds sum_c G_0,c (chi (beta_c + U q))' = chi' H_t,0 + sum_mu (chi q_mu)' H_t,mu for each edge.
//
// Scalar channels by splines.
//
// Where all atoms are of one species, psi_c(rho) of the one pair is written as a B-spline of degree seven on a few hundred intervals,
// psi_c = sum_a B_a(t) S_{k + a, c}, and the sum over a row becomes sum_j chi_j psi_c = sum_k S_k,c p_k with
// p_{k + a} = sum_j chi_j B_a(t_j): an edge adds eight numbers whatever C0 is, where it read 8 bytes per channel and multiplied them out.
// The rows of p meet S in the same matrix product, and the backward pass reads H = S G_0 of its row: sum_c G_0,c (chi psi_c)' is
// the derivative of chi times the spline of coefficients H.
#include "kernels.h"

namespace umd {

namespace {

constexpr int kRows = 64;            // rows of a block, all of one species
constexpr int KC = 16;               // depth of a step

// ---- rows of a tile grouped by the species of their atom --------------------------------------------------------------
// order: rows of the first species, then of the second ..., each padded with -1 to whole blocks; which place a row gets inside its
// group changes nothing that is computed from it.
__global__ void k_group_count(int n, const int* __restrict__ type, int* __restrict__ count) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int t = i < n ? type[i] : -1 - (int)(threadIdx.x & 31);
    const unsigned same = __match_any_sync(0xffffffffu, t);
    if (i < n && __ffs(same) - 1 == (int)(threadIdx.x & 31)) atomicAdd(count + t, __popc(same));
}
__global__ void k_group_fill(int n, int T, const int* __restrict__ type, const int* __restrict__ count, int* __restrict__ cursor,
                             int* __restrict__ order) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const int t = i < n ? type[i] : -1 - lane;
    const unsigned same = __match_any_sync(0xffffffffu, t);
    if (i >= n) return;
    const int leader = __ffs(same) - 1;
    int at = 0;
    if (lane == leader) {
        for (int u = 0; u < t; ++u) at += (count[u] + kRows - 1) / kRows * kRows;
        at += atomicAdd(cursor + t, __popc(same));
    }
    at = __shfl_sync(same, at, leader) + __popc(same & ((1u << lane) - 1u));
    order[at] = i;
}

// ---- C[64 x NT] = A[64 x K] B[K x NT] in single precision -----------------------------------------------------------------
// FORWARD: A = moments of the rows, B = beta and U of the centre's species (or the spline coefficients), added to (or put into) the
// scalar channels' sums.  Backward: A = gradient of those sums, B the transpose, into the moments' place.
// NT threads of eight rows and eight columns each: sixteen words from shared memory for 64 multiply-adds, pairs of them in one
// instruction.  The L1 data pipe takes a cycle for every word that the lanes of a warp read, the FMA pipe one for every
// multiply-add, so that both are busy alike.
// A step's products are added up by themselves first: in one chain of 168 the rounding of a row of splines is 2.7e-7 of the sums'
// rms, in two levels 1.1e-7 to 1.5e-7, as the sums over the edges have it (1.1e-7 to 1.6e-7).  Operands come by asynchronous
// copies, two steps ahead; those whose depth is contiguous in memory lie in rows of KC + 4.
template <bool FORWARD, int NT>
__global__ void __launch_bounds__(NT, 256 / NT) k_moments(int a0, int K, int N, Dims d, const float* __restrict__ pairmod, const int* __restrict__ type_s,
                                                          const int* __restrict__ order, float* __restrict__ state, float* __restrict__ moments, int km,
                                                          const float* __restrict__ spline, int n) {
    constexpr int STAGES = 3, AP = KC + 4, BP = FORWARD ? NT : KC + 4, BROWS = FORWARD ? KC : NT;
    __shared__ __align__(16) float As[STAGES][kRows * AP];
    __shared__ __align__(16) float Bs[STAGES][BROWS * BP];
    __shared__ int row_s[kRows];
    const int tid = threadIdx.x, tx = tid % (NT / 8), ty = tid / (NT / 8);
    for (int r = tid; r < kRows; r += NT) {
        const int at = blockIdx.x * kRows + r;
        row_s[r] = spline ? (at < n ? at : -1) : order[at];
    }
    __syncthreads();
    if (row_s[0] < 0) return;                                    // past the last group
    const int R1 = 1 + d.R, C0 = d.C0, ti = spline ? 0 : type_s[a0 + row_s[0]], kb = spline ? km : d.T * R1;
    const int n0 = FORWARD ? 0 : blockIdx.y * NT;                 // first column
    // row k of (beta | U) of the centre's species: moment k = t (1 + R) + mu
    auto mixing = [&](int k) {
        if (spline) return spline + (size_t)k * C0;
        const int t = k / R1;
        return pairmod + ((size_t)(ti * d.T + t) * (2 + d.R) + 1 + (k - t * R1)) * C0;
    };
    const int lda = FORWARD ? km : d.SP;
    const float* const A = FORWARD ? moments : state;
    auto copy16 = [](float* dst, const float* src, bool on) {     // 16 bytes, zeros where there is nothing
        const unsigned at = (unsigned)__cvta_generic_to_shared(dst);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(at), "l"(src), "r"(on ? 16 : 0) : "memory");
    };
    auto fetch = [&](int step) {
        const int k0 = step * KC, st = step % STAGES;
        if (k0 < K) {
#pragma unroll
            for (int p = 0; p < kRows * KC / 4 / NT; ++p) {
                const int at = tid + p * NT, r = at / (KC / 4), k = 4 * (at % (KC / 4)), row = row_s[r];
                const bool on = row >= 0 && k0 + k < K;
                copy16(&As[st][r * AP + k], on ? A + (size_t)row * lda + k0 + k : A, on);
            }
#pragma unroll
            for (int p = 0; p < KC / 4; ++p) {
                const int at = tid + p * NT;
                const int k = FORWARD ? k0 + at / (NT / 4) : n0 + at / (KC / 4), c = FORWARD ? 4 * (at % (NT / 4)) : k0 + 4 * (at % (KC / 4));
                const bool on = k < kb && (FORWARD || c < C0);
                copy16(&Bs[st][FORWARD ? (at / (NT / 4)) * BP + c : (at / (KC / 4)) * BP + 4 * (at % (KC / 4))], on ? mixing(k) + c : pairmod, on);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float2 acc[8][4], part[8][4];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = make_float2(0.f, 0.f);
    // rows of a thread: four at 4 ty, four at 32 + 4 ty; columns: forward four at 4 tx and four at NT / 2 + 4 tx, backward every NT / 8-th
    auto row_of = [&](int r) { return 4 * ty + (r & 3) + 32 * (r >> 2); };
    auto column = [&](int c) { return tx + NT / 8 * c; };
    const int steps = (K + KC - 1) / KC;
    fetch(0);
    fetch(1);
    for (int s = 0; s < steps; ++s) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();                                         // (this step is there, and nobody reads the stage that is filled next)
        fetch(s + 2);
        const float *as = As[s % STAGES], *bs = Bs[s % STAGES];
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) part[r][c] = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < KC; k += 4) {
            float4 a[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) a[r] = *reinterpret_cast<const float4*>(as + row_of(r) * AP + k);
            float4 bt[8];                                        // backward: four depths of eight columns
            if (!FORWARD) {
#pragma unroll
                for (int c = 0; c < 8; ++c) bt[c] = *reinterpret_cast<const float4*>(bs + column(c) * BP + k);
            }
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                auto at = [&](const float4& v) { return kk == 0 ? v.x : (kk == 1 ? v.y : (kk == 2 ? v.z : v.w)); };
                float2 b[4];
                if (FORWARD) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float4 v = *reinterpret_cast<const float4*>(bs + (k + kk) * BP + 4 * tx + NT / 2 * h);
                        b[2 * h] = make_float2(v.x, v.y); b[2 * h + 1] = make_float2(v.z, v.w);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < 4; ++c) b[c] = make_float2(at(bt[2 * c]), at(bt[2 * c + 1]));
                }
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const float2 ar = make_float2(at(a[r]), at(a[r]));
#pragma unroll
                    for (int c = 0; c < 4; ++c) part[r][c] = ffma2(ar, b[c], part[r][c]);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) { acc[r][c].x += part[r][c].x; acc[r][c].y += part[r][c].y; }
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int row = row_s[row_of(r)];
        if (row < 0) continue;
        if (FORWARD) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float4* const o = reinterpret_cast<float4*>(state + (size_t)row * d.SP + 4 * tx + NT / 2 * h);
                const float4 v = spline ? make_float4(0.f, 0.f, 0.f, 0.f) : *o;
                const float2 x = acc[r][2 * h], y = acc[r][2 * h + 1];
                *o = make_float4(v.x + x.x, v.y + x.y, v.z + y.x, v.w + y.y);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int m = n0 + column(c);
                if (m < N) moments[(size_t)row * km + m] = c & 1 ? acc[r][c >> 1].y : acc[r][c >> 1].x;
            }
        }
    }
}

// A thread per channel, the rows one after the other (spline_coefficient); once per species that a handle meets.
__global__ void k_spline_pair(Dims d, const double* __restrict__ coef, const float* __restrict__ pairmod, int t, int n, int pitch,
                              float* __restrict__ spline) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.C0) return;
    const float* const pm = pairmod + (size_t)(t * d.T + t) * (2 + d.R) * d.C0 + c;
    double left = 0;
    for (int k = 0; k < pitch; ++k)
        spline[(size_t)k * d.C0 + c] = k < n + 7 ? spline_coefficient(d, coef + (size_t)k * (d.C0 + d.R), pm, c, &left) : 0.0f;
}

}  // namespace

int moment_pitch(const Dims& d) { return (d.T * (1 + d.R) + 3) / 4 * 4; }
bool moments_pick(const Dims& d, int64_t rows) {
    return wide_channels(d.C0) && d.R > 0 && moment_pitch(d) <= kMaxMoments && rows >= kMomentRows;
}
int64_t moment_order_ints(const Dims& d, int64_t rows) { return rows + (int64_t)kRows * d.T; }

cudaError_t launch_moment_groups(const Dims& d, const int* type_s, int n, int* scratch, int* order, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(scratch, 0, sizeof(int) * 2 * (size_t)d.T, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(order, 0xff, sizeof(int) * (size_t)moment_order_ints(d, n), st);
    if (e != cudaSuccess || n == 0) return e;
    k_group_count<<<(n + 255) / 256, 256, 0, st>>>(n, type_s, scratch);
    k_group_fill<<<(n + 255) / 256, 256, 0, st>>>(n, d.T, type_s, scratch, scratch + d.T, order);
    return cudaGetLastError();
}

template <bool FORWARD>
static cudaError_t launch(const MomentArgs& a, cudaStream_t st) {
    const Dims& d = a.d;
    const int km = a.pitch, K = FORWARD ? km : d.C0, N = FORWARD ? d.C0 : km;
    const unsigned groups = a.spline ? (unsigned)((a.n + kRows - 1) / kRows) : (unsigned)(moment_order_ints(d, a.n) / kRows);
    auto go = [&](auto kern, int NT) {
        kern<<<dim3(groups, (unsigned)((N + NT - 1) / NT)), NT, 0, st>>>(a.a0, K, N, d, a.pairmod, a.type_s, a.order, a.state, a.moments, km, a.spline, a.n);
        return cudaGetLastError();
    };
    // (backward: the width that pads fewer columns)
    const int width = FORWARD ? d.C0 : ((N + 63) / 64 * 64 < (N + 127) / 128 * 128 ? 64 : 128);
    if (width == 128) return go(k_moments<FORWARD, 128>, 128);
    return width == 64 ? go(k_moments<FORWARD, 64>, 64) : go(k_moments<true, 32>, 32);
}
cudaError_t launch_spline_pair(const Dims& d, const double* coef, const float* pairmod, int t, int n, int pitch, float* spline, cudaStream_t st) {
    k_spline_pair<<<(d.C0 + 31) / 32, 32, 0, st>>>(d, coef, pairmod, t, n, pitch, spline);
    return cudaGetLastError();
}
cudaError_t launch_moments_forward(const MomentArgs& a, cudaStream_t st) { return launch<true>(a, st); }
cudaError_t launch_moments_backward(const MomentArgs& a, cudaStream_t st) { return launch<false>(a, st); }

}  // namespace umd
