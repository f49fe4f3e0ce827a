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
#include "kernels.h"

namespace umd {

namespace {

constexpr int kRows = 64;            // rows of a block, all of one species
constexpr int KC = 32;               // depth of a step
constexpr int AP = kRows + 4;        // pitch of the transposed operands (16-byte reads of four rows)
constexpr int kThreads = 256;

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
// FORWARD: A = moments of the rows, B = beta and U of the centre's species, added to the scalar channels' sums.
// Backward: A = gradient of those sums, B the transpose, into the moments' place.
// A thread holds four rows and NT / 16 columns; a step's operands are fetched while the one before is multiplied, pairs of
// multiply-adds in one instruction.  40,009 rows of 320 moments and 128 channels (3.3 GFLOP) take 142 us forward, 134 backward, a
// third of the FMA rate: 689 blocks are 2.3 rounds of the machine, and the L1 data pipe, which a thread's twelve words per 32
// multiply-adds occupy, is 65 to 80 % busy.  The edge kernels, which read these rows for every edge, took 543 us and 820 us more.
template <bool FORWARD, int NT>
__global__ void __launch_bounds__(kThreads) k_moments(int a0, int K, int N, Dims d, const float* __restrict__ pairmod, const int* __restrict__ type_s,
                                                      const int* __restrict__ order, float* __restrict__ state, float* __restrict__ moments, int km) {
    constexpr int TC = NT / 16;                                   // columns of a thread: TC / 4 runs of four (or one of two)
    constexpr int BP = FORWARD ? NT : NT + 4;
    __shared__ __align__(16) float As[KC][AP];
    __shared__ __align__(16) float Bs[KC][BP];
    __shared__ int row_s[kRows];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    if (tid < kRows) row_s[tid] = order[(size_t)blockIdx.x * kRows + tid];
    __syncthreads();
    if (row_s[0] < 0) return;                                    // past the last group
    const int ti = type_s[a0 + row_s[0]], R1 = 1 + d.R, C0 = d.C0;
    const int n0 = FORWARD ? 0 : blockIdx.y * NT;                 // first column
    // row k of (beta | U) of the centre's species: moment k = t (1 + R) + mu
    auto mixing = [&](int k) { const int t = k / R1; return pairmod + ((size_t)(ti * d.T + t) * (2 + d.R) + 1 + (k - t * R1)) * C0; };
    const int lda = FORWARD ? km : d.SP;
    const float* const A = FORWARD ? moments : state;
    float4 ra[2];
    constexpr int NB = KC * NT / 4 / kThreads;                    // 16-byte pieces of B per thread
    float4 rb[NB];
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    auto fetch = [&](int k0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = row_s[(tid >> 3) + 32 * h], k = k0 + 4 * (tid & 7);
            ra[h] = row >= 0 && k < K ? *reinterpret_cast<const float4*>(A + (size_t)row * lda + k) : zero;
        }
#pragma unroll
        for (int p = 0; p < NB; ++p) {
            const int at = tid + p * kThreads;
            if (FORWARD) {
                const int k = k0 + at / (NT / 4), c = 4 * (at % (NT / 4));
                rb[p] = k < K && k < d.T * R1 ? *reinterpret_cast<const float4*>(mixing(k) + c) : zero;
            } else {
                const int m = n0 + (at >> 3), k = k0 + 4 * (at & 7);
                rb[p] = m < d.T * R1 ? *reinterpret_cast<const float4*>(mixing(m) + k) : zero;
            }
        }
    };
    auto park = [&]() {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = (tid >> 3) + 32 * h, k = 4 * (tid & 7);
            As[k][r] = ra[h].x; As[k + 1][r] = ra[h].y; As[k + 2][r] = ra[h].z; As[k + 3][r] = ra[h].w;
        }
#pragma unroll
        for (int p = 0; p < NB; ++p) {
            const int at = tid + p * kThreads;
            if (FORWARD) {
                *reinterpret_cast<float4*>(&Bs[at / (NT / 4)][4 * (at % (NT / 4))]) = rb[p];
            } else {
                const int m = at >> 3, k = 4 * (at & 7);
                Bs[k][m] = rb[p].x; Bs[k + 1][m] = rb[p].y; Bs[k + 2][m] = rb[p].z; Bs[k + 3][m] = rb[p].w;
            }
        }
    };
    float2 acc[4][TC / 2];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < TC / 2; ++c) acc[r][c] = make_float2(0.f, 0.f);
    // columns of a thread: runs of four at 4 tx + 64 run, or two at 2 tx
    auto column = [&](int c) { return TC == 2 ? 2 * tx : 4 * tx + 64 * (c >> 1) + 2 * (c & 1); };
    fetch(0);
    for (int k0 = 0; k0 < K; k0 += KC) {
        park();
        __syncthreads();
        if (k0 + KC < K) fetch(k0 + KC);
#pragma unroll 8
        for (int k = 0; k < KC; ++k) {
            const float4 a = *reinterpret_cast<const float4*>(&As[k][4 * ty]);
            float2 b[TC / 2];
            if (TC == 2) b[0] = *reinterpret_cast<const float2*>(&Bs[k][2 * tx]);
            else {
#pragma unroll
                for (int c = 0; c < TC / 2; c += 2) {
                    const float4 v = *reinterpret_cast<const float4*>(&Bs[k][column(c)]);
                    b[c] = make_float2(v.x, v.y);
                    b[c + 1 < TC / 2 ? c + 1 : c] = make_float2(v.z, v.w);
                }
            }
#pragma unroll
            for (int c = 0; c < TC / 2; ++c) {
                acc[0][c] = ffma2(make_float2(a.x, a.x), b[c], acc[0][c]);
                acc[1][c] = ffma2(make_float2(a.y, a.y), b[c], acc[1][c]);
                acc[2][c] = ffma2(make_float2(a.z, a.z), b[c], acc[2][c]);
                acc[3][c] = ffma2(make_float2(a.w, a.w), b[c], acc[3][c]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int row = row_s[4 * ty + r];
        if (row < 0) continue;
#pragma unroll
        for (int c = 0; c < TC / 2; ++c) {
            const int n = n0 + column(c);
            if (n >= N) continue;                                // (N is even)
            if (FORWARD) {
                float2* const o = reinterpret_cast<float2*>(state + (size_t)row * d.SP + n);
                const float2 v = *o;
                *o = make_float2(v.x + acc[r][c].x, v.y + acc[r][c].y);
            } else {
                *reinterpret_cast<float2*>(moments + (size_t)row * km + n) = acc[r][c];
            }
        }
    }
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
    const int km = moment_pitch(d), K = FORWARD ? km : d.C0, N = FORWARD ? d.C0 : km;
    const unsigned groups = (unsigned)(moment_order_ints(d, a.n) / kRows);
    auto go = [&](auto kern, int NT) {
        kern<<<dim3(groups, (unsigned)((N + NT - 1) / NT)), kThreads, 0, st>>>(a.a0, K, N, d, a.pairmod, a.type_s, a.order, a.state, a.moments, km);
        return cudaGetLastError();
    };
    if (!FORWARD || d.C0 == 128) return go(k_moments<FORWARD, 128>, 128);
    return d.C0 == 64 ? go(k_moments<FORWARD, 64>, 64) : go(k_moments<FORWARD, 32>, 32);
}
cudaError_t launch_moments_forward(const MomentArgs& a, cudaStream_t st) { return launch<true>(a, st); }
cudaError_t launch_moments_backward(const MomentArgs& a, cudaStream_t st) { return launch<false>(a, st); }

}  // namespace umd
