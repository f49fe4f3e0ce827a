// The whole atomic-energy MLP of a block of atoms in one kernel: all forward layers, the scalar head, and
// the input vector-Jacobian product.
//
// A chain of one GEMM per layer spends its time around the tensor pipe: every layer's activations leave
// the chip as half-precision splits and pre-activations and come back once per column tile, and each
// layer pays a launch, a tensor-memory allocation and a cold pipeline.  Here a CTA takes NA atoms (16 ..
// 128) and keeps their activations in shared memory from layer to layer, as the half-precision split that
// the next layer's MMAs read; only the weights stream.  The weights are the M operand (128 features per
// tile) and the atoms the N operand, so that a block may be as small as 16 atoms: a system of a few
// thousand atoms still gives every SM a block, and all four lane quarters of tensor memory have work in
// the epilogue.
//
// Roles: warp 0 copies (TMA), warp 1 issues the MMAs, sixteen warps run the epilogues: a thread owns a
// feature (lane quarter and lane) and eight atoms at a time.  Neighbouring lanes are neighbouring features,
// so every global access of the epilogue is a contiguous 128 bytes and every operand access 64.
// All feature tiles of a layer sit side by side in tensor memory, two accumulators each: hi * hi, and the
// two cross terms (the accumulator truncates once per instruction; the cross terms are 2^-11 of the result
// and lose nothing that shows).  The hi and lo parts of the atoms follow each other in shared memory, so
// one MMA of N = 2 NA takes W_hi times both, into both accumulators; a second one adds W_lo A_hi (an MMA
// of M = 128 costs about 50 cycles however small N is, so fewer and wider ones).
// An epilogue hands its output over a feature tile (128 of the next layer's K) at a time, and the next
// layer's MMAs are issued in the order in which operand blocks and accumulators come free: step l takes
// every (K group, tile) with max(group, tile) = l.
// What the backward pass needs of the forward pass (the SiLU derivative, and the hidden gradient where a
// residual joins) is kept per CTA, in shared memory when it fits, else in a scratch area that stays in L2.
//
// Every wait is bounded, as in the one-layer kernels: on expiry the CTA raises its abort flag, stops issuing,
// lets copies in flight land and issued MMAs retire, frees its tensor memory and returns with an error bit.
#include "common.cuh"
#include "kernels.h"
#include "mlp_gemm.h"
#include "tcgen05.cuh"

namespace umd {

namespace {

constexpr int kMaxLayers = 8;
constexpr int EPW = 16;                                  // epilogue warps
constexpr int THREADS = (2 + EPW) * 32;
constexpr uint32_t W_HALF = 128 * 64;                    // 128 features x 32 halves
constexpr uint32_t W_BYTES = 2 * W_HALF;                 // hi and lo: one stage of the weight ring
constexpr int MAX_KB = 20, MAX_STAGES = 8, MAX_TILES = 4;
constexpr int MAX_F = 384, MAX_NA = 128;
constexpr uint32_t SMEM_MAX = 232448, BAR_AREA = 512;

struct FusedMaps {
    CUtensorMap a[2];                                    // split of the feature vector: hi, lo
    CUtensorMap w[2 * kMaxLayers][2];                    // weights of GEMM q: hi, lo
};
struct FusedArgs {
    int M, NA;                  // atoms; atoms of a block
    int F, K0, N0, NH;
    int grad;
    int a_blocks, stages, bufs; // operand blocks of 32 features; ring stages; accumulator sets in tensor memory
    int keep_in_smem;
    const float* bias[kMaxLayers];       // layers 1 ..
    const float* bias_rows; const int* row_type;         // layer 0: bias by species
    const float* head_w; float b_head; const float* e_ref;
    double* e_atom;             // [M]
    float* out; int ldout;      // gradient of the feature columns [M][N0]
    float acc_scale[2 * kMaxLayers];     // per GEMM: the inverse of the weights' scale
    float gs;                   // factor the back-propagated gradients carry
    float* scratch; size_t scratch_stride;               // floats per CTA
    int* err; int spin_limit; int test_skip;
};

__device__ __forceinline__ void tmem_ld8x2(uint32_t t0, uint32_t t1, float* v, float* w) {
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(t0));
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(t1));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) { v[i] = __uint_as_float(r[i]); w[i] = __uint_as_float(r[8 + i]); }
}
__device__ __forceinline__ uint32_t lds16(uint32_t a) {
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts16(uint32_t a, uint32_t v) {
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((uint16_t)v) : "memory");
}
__device__ __forceinline__ float2 half2_of(uint32_t lo, uint32_t hi) {
    const uint32_t v = lo | (hi << 16);
    return __half22float2(*reinterpret_cast<const __half2*>(&v));
}
__device__ __forceinline__ void arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__global__ void __launch_bounds__(THREADS, 1) k_mlp_fused(const __grid_constant__ FusedMaps maps, const __grid_constant__ FusedArgs g) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t abase = (raw + 1023u) & ~1023u;
    const uint32_t a_half = (uint32_t)g.NA * 64, a_bytes = 2 * a_half;       // one operand block: hi, then lo
    const uint32_t wbase = abase + (uint32_t)g.a_blocks * a_bytes;
    const uint32_t bars = wbase + (uint32_t)g.stages * W_BYTES;
    const uint32_t w_full = bars, w_empty = w_full + 8 * MAX_STAGES, a0_full = w_empty + 8 * MAX_STAGES, acc_full = a0_full + 8 * MAX_KB,
                   acc_free = acc_full + 16, a_ready = acc_free + 16, item_done = a_ready + 8 * MAX_TILES, drain_bar = item_done + 8;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_raw + (drain_bar + 8 - raw));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_raw + (drain_bar + 12 - raw));
    float* const head_part = reinterpret_cast<float*>(smem_raw + (bars + BAR_AREA - raw));      // [tiles * 4][NA]
    const int limit = g.spin_limit > 0 ? g.spin_limit : kSpinLimit;
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int items = (g.M + g.NA - 1) / g.NA;
    const int F32 = (g.F + 31) & ~31, N32 = (g.N0 + 31) & ~31;
    const int KBF = F32 >> 5, KB0 = (g.K0 + 31) >> 5;
    const int tiles_f = (g.F + 127) >> 7, tiles_0 = (g.N0 + 127) >> 7;
    const int n_gemm = g.grad ? 2 * g.NH : g.NH;
    // GEMM q: 0 .. NH - 1 the forward layers; then the backward ones, from the last layer to the first.  A
    // pass covers up to tiles_f feature tiles (only the last GEMM can take more than one pass).
    auto n_tiles = [&](int q) { return q == 2 * g.NH - 1 ? tiles_0 : tiles_f; };
    auto n_blocks = [&](int q) { return q == 0 ? KB0 : KBF; };
    const uint32_t buf_cols = 512u / (uint32_t)g.bufs;

    if (threadIdx.x == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) { mbar_init(w_full + 8 * s, 1); mbar_init(w_empty + 8 * s, 1); }
        for (int s = 0; s < MAX_KB; ++s) mbar_init(a0_full + 8 * s, 1);
        for (int s = 0; s < 2; ++s) { mbar_init(acc_full + 8 * s, 1); mbar_init(acc_free + 8 * s, EPW); }
        for (int s = 0; s < MAX_TILES; ++s) mbar_init(a_ready + 8 * s, EPW);
        mbar_init(item_done, EPW);
        mbar_init(drain_bar, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32((const void*)tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    chain_begin();

    // The copy and the issue warp run their loops as whole warps, one elected lane issuing: the loop state
    // and the descriptors are then warp-uniform and live in uniform registers, where the copy and MMA
    // instructions take their operands from (issued from a lane's own registers a stage of six MMAs took
    // three times as long as the MMAs themselves).
    // A wait of a whole warp: the lanes poll by themselves and can disagree where it gives up, so they vote;
    // everything after it is decided by all lanes alike (an election among lanes that went different ways
    // would never end).
    auto wait_all = [&](uint32_t bar, uint32_t parity) {
        return __all_sync(0xffffffffu, mbar_wait_a(bar, parity, g.err, abort_flag, limit)) != 0;
    };
    if (warp == 0) {                                       // copies
        uint32_t s = 0, lap = 0;                           // stage, and how often the ring has gone round
        int loaded = 0, block = 0;
        bool go = true;
        for (int it = blockIdx.x; it < items; it += gridDim.x, ++block) {
            for (int q = 0; q < n_gemm; ++q) {
                const CUtensorMap *hi = &maps.w[q][0], *lo = &maps.w[q][1];
                const int nt = n_tiles(q), nk = n_blocks(q);
                for (int t0 = 0; t0 < nt; t0 += tiles_f) {
                    const int nl = min(tiles_f, nt - t0), ng = (nk + 3) >> 2;
                    for (int l = 0; l < max(ng, nl); ++l)
                    for (int gr = 0; gr <= min(l, ng - 1); ++gr)
                    for (int j = gr < l ? l : 0; j <= min(l, nl - 1); ++j)
                    for (int kb = 4 * gr; kb < min(4 * gr + 4, nk); ++kb) {
                        if (q == 0 && j == 0) {            // the first layer's operand comes from memory
                            if (kb == 0 && block > 0) {
                                // its area is free when the MMAs of the block before have read it (the last of them
                                // release the stage loaded last), and without a backward pass when its last epilogue
                                // has taken the residual from there
                                const uint32_t sl = s == 0 ? (uint32_t)g.stages - 1 : s - 1, ll = s == 0 ? lap - 1 : lap;
                                go = go && wait_all(w_empty + 8 * sl, ll & 1);
                                if (!g.grad) go = go && wait_all(item_done, (block - 1) & 1);
                            }
                            const uint32_t dst = abase + (uint32_t)kb * a_bytes, full = a0_full + 8 * kb;
                            if (go) if (elect_one()) {
                                mbar_expect_tx(full, a_bytes);
                                tma_load_2d(dst, &maps.a[0], kb * 32, it * g.NA, full);
                                tma_load_2d(dst + a_half, &maps.a[1], kb * 32, it * g.NA, full);
                            }
                        }
                        if (lap > 0) go = go && wait_all(w_empty + 8 * s, (lap - 1) & 1);
                        const uint32_t dst = wbase + s * W_BYTES, full = w_full + 8 * s;
                        loaded += go;
                        if (go && (g.test_skip == 0 || loaded != g.test_skip)) if (elect_one()) {    // (diagnostic: that stage never arrives)
                            mbar_expect_tx(full, W_BYTES);
                            tma_load_2d(dst, hi, kb * 32, (t0 + j) * 128, full);
                            tma_load_2d(dst + W_HALF, lo, kb * 32, (t0 + j) * 128, full);
                        }
                        if (++s == (uint32_t)g.stages) { s = 0; ++lap; }
                    }
                }
            }
        }
        // giving up: let the copies still in flight land first
        if (__any_sync(0xffffffffu, *abort_flag)) {
            for (int k = 0; k < g.stages && k < loaded; ++k)
                mbar_wait_quiet(w_full + 8 * k, ((loaded - 1 - k) / g.stages) & 1, limit);
            for (int k = 0; k < KB0; ++k)
                for (int par = 0; par < 2; ++par) mbar_wait_quiet(a0_full + 8 * k, par, limit / 16 + 1);
        }
    } else if (warp == 1) {                                // MMAs
        uint32_t s = 0, phase = 0;                         // stage of the weight ring
        int pass = 0, uses = 0, block = 0;
        bool go = true;
        // descriptors: the address field is the low word's, everything else is constant
        const uint64_t a_desc = umma_desc(abase), w_desc = umma_desc(wbase);
        const uint32_t AB = a_bytes >> 4;
        constexpr uint32_t K16 = 32 >> 4, WH = W_HALF >> 4, WB = W_BYTES >> 4;
        // instruction descriptors: D = F32, A = B = F16, both K-major, N = NA or 2 NA, M = 128
        const uint32_t idesc1 = (1u << 4) | ((uint32_t)(g.NA >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        const uint32_t idesc2 = (1u << 4) | ((uint32_t)(g.NA >> 2) << 17) | ((uint32_t)(128 >> 4) << 24);
        for (int it = blockIdx.x; it < items; it += gridDim.x, ++block)
            for (int q = 0; q < n_gemm; ++q) {
                const int nt = n_tiles(q), nk = n_blocks(q);
                for (int t0 = 0; t0 < nt; t0 += tiles_f, ++pass) {
                    const int buf = pass & (g.bufs - 1), use = g.bufs == 2 ? pass >> 1 : pass;
                    // one accumulator set and the operand from the epilogue before: a tile's accumulators are
                    // free as soon as that epilogue has handed over the tile (a_ready below)
                    const bool by_tile = g.bufs == 1 && q > 0 && t0 == 0;
                    if (use > 0 && !by_tile) go = go && wait_all(acc_free + 8 * buf, (use - 1) & 1);
                    tc_fence_after();
                    const int nl = min(tiles_f, nt - t0), ng = (nk + 3) >> 2;
                    for (int l = 0; l < max(ng, nl); ++l) {
                        if (q > 0 && t0 == 0 && l < tiles_f) {
                            go = go && wait_all(a_ready + 8 * l, uses & 1);
                            tc_fence_after();
                        }
                        for (int gr = 0; gr <= min(l, ng - 1); ++gr)
                        for (int j = gr < l ? l : 0; j <= min(l, nl - 1); ++j) {
                            const uint32_t d = tmem + (uint32_t)buf * buf_cols + (uint32_t)j * 2 * (uint32_t)g.NA, dc = d + (uint32_t)g.NA;
                            for (int kb = 4 * gr; kb < min(4 * gr + 4, nk); ++kb) {
                                if (q == 0 && j == 0) go = go && wait_all(a0_full + 8 * kb, block & 1);
                                const uint64_t ad = a_desc + (uint64_t)((uint32_t)kb * AB);
                                const uint64_t wd = w_desc + (uint64_t)(s * WB);
                                go = go && wait_all(w_full + 8 * s, phase);
                                tc_fence_after();
                                if (go) if (elect_one()) {
                                    umma_f16(d, wd, ad, idesc2, kb > 0 ? 1u : 0u);
                                    umma_f16(dc, wd + WH, ad, idesc1, 1u);
                                    umma_f16(d, wd + K16, ad + K16, idesc2, 1u);
                                    umma_f16(dc, wd + WH + K16, ad + K16, idesc1, 1u);
                                    umma_commit(w_empty + 8 * s);          // frees the stage when these MMAs retire
                                }
                                if (++s == (uint32_t)g.stages) { s = 0; phase ^= 1; }
                            }
                        }
                    }
                    // by_tile: the phase of the epilogue before is complete or about to be.  It is waited for ahead of the
                    // commit: once that is out, the next epilogue may complete a phase of the same parity as the one before
                    if (by_tile) go = go && wait_all(acc_free, (use - 1) & 1);
                    if (go) if (elect_one()) umma_commit(acc_full + 8 * buf);
                }
                if (q > 0) ++uses;
            }
        if (__any_sync(0xffffffffu, *abort_flag)) {        // every instruction issued so far has to retire before the
            if (elect_one()) umma_commit(drain_bar);       // tensor memory goes back
            __syncwarp();
            mbar_wait_quiet(drain_bar, 0, limit);
        }
    } else {                                               // epilogues
        const int quarter = warp & 3, cg = (warp - 2) >> 2;
        const int chunks = g.NA >> 3, per_tile = (chunks - cg + 3) >> 2;     // this warp's groups of eight atoms in a tile
        float* const keep = g.keep_in_smem ? head_part + MAX_F / 32 * g.NA : g.scratch + (size_t)blockIdx.x * g.scratch_stride;
        const size_t layer_floats = (size_t)g.NA * F32;
        float* const dh_keep = keep + (size_t)(g.NH - 1) * layer_floats;
        const uint32_t seg = (uint32_t)lane >> 3;
        int pass = 0;
        for (int it = blockIdx.x; it < items; it += gridDim.x) {
            const int m0 = it * g.NA;
            for (int q = 0; q < n_gemm; ++q) {
                const bool fwd = q < g.NH, last_fwd = q == g.NH - 1, final_gemm = q == 2 * g.NH - 1;
                const int t = fwd ? q : 2 * g.NH - 1 - q;          // layer
                const int nt = n_tiles(q), width = final_gemm ? g.N0 : g.F, width32 = final_gemm ? N32 : F32;
                const bool feeds = q + 1 < n_gemm;                 // leaves the operand of another GEMM
                const bool first_bwd = t == g.NH - 1;
                const float sc = final_gemm ? g.acc_scale[q] / g.gs : g.acc_scale[q];
                for (int t0 = 0; t0 < nt; t0 += tiles_f, ++pass) {
                    const int buf = pass & (g.bufs - 1), use = g.bufs == 2 ? pass >> 1 : pass;
                    const int n_here = min(tiles_f, nt - t0) * per_tile;
                    float nx[8], ny[8];
                    // what a group of eight atoms takes from memory, requested one group ahead: the bias by species,
                    // or the derivative and the joining gradient
                    auto request = [&](int j, int c) {
                        const int n = (t0 + j) * 128 + quarter * 32 + lane, a0 = (cg + 4 * c) * 8;
                        if (final_gemm || n - lane >= width32) return;
                        if (fwd) {
                            if (q > 0) return;
                            const int ml = m0 + a0 + (lane & 7), type = ml < g.M ? __ldg(g.row_type + ml) : 0;
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                const int ti = __shfl_sync(0xffffffffu, type, i);      // (by all lanes, also those past a ragged width)
                                nx[i] = n < width ? __ldg(g.bias_rows + (size_t)ti * g.F + n) : 0.f;
                            }
                        } else {
                            const float *kd = keep + (size_t)(t - 1) * layer_floats + (size_t)a0 * F32 + n, *kh = dh_keep + (size_t)a0 * F32 + n;
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                ny[i] = kd[(size_t)i * F32];
                                if (!first_bwd) nx[i] = kh[(size_t)i * F32];
                            }
                        }
                    };
                    if (n_here > 0) request(0, 0);
                    mbar_wait_a(acc_full + 8 * buf, use & 1, g.err, abort_flag, limit);
                    tc_fence_after();
                    for (int j = 0; j < min(tiles_f, nt - t0); ++j) {
                        const int n0 = (t0 + j) * 128 + quarter * 32, n = n0 + lane;
                        const bool on = n < width;
                        const float hw = on && !final_gemm && (last_fwd || (!fwd && first_bwd)) ? __ldg(g.head_w + n) : 0.f;
                        const float bias = on && fwd && q > 0 ? __ldg(g.bias[q] + n) : 0.f;
                        const uint32_t a_col = abase + (uint32_t)(n >> 5) * a_bytes + (uint32_t)(lane & 7) * 2;
                        const uint32_t tcol = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)buf * buf_cols + (uint32_t)(j * 2 * g.NA);
#pragma unroll 1
                        for (int c = 0; c < per_tile; ++c) {
                            const int a0 = (cg + 4 * c) * 8;
                            float x[8], y[8];
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                x[i] = fwd ? (q == 0 ? nx[i] : bias) : (final_gemm ? 0.f : (first_bwd ? g.gs * hw : nx[i]));
                                y[i] = ny[i];
                            }
                            if (c + 1 < per_tile) request(j, c + 1);
                            else if ((j + 1) * per_tile < n_here) request(j + 1, 0);
                            if (n0 >= width32) continue;
                            float v[8], w[8];
                            tmem_ld8x2(tcol + (uint32_t)a0, tcol + (uint32_t)(g.NA + a0), v, w);
#pragma unroll
                            for (int i = 0; i < 8; ++i) v[i] = fmaf(sc, v[i] + w[i], x[i]);
                            if (final_gemm) {
#pragma unroll
                                for (int i = 0; i < 8; ++i)
                                    if (on && m0 + a0 + i < g.M) g.out[(size_t)(m0 + a0 + i) * g.ldout + n] = v[i];
                                continue;
                            }
                            float* const kd = keep + (size_t)(fwd ? q : t - 1) * layer_floats + (size_t)a0 * F32 + n;
                            float* const kh = dh_keep + (size_t)a0 * F32 + n;
                            float o[8];
                            if (fwd) {
#pragma unroll
                                for (int i = 0; i < 8; i += 2) {
                                    float2 r = make_float2(0.f, 0.f);
                                    if (q > 0) {                   // the residual is the operand that is replaced
                                        const uint32_t at = a_col + (uint32_t)(a0 + i) * 64 + ((seg ^ (uint32_t)(i >> 1)) << 4);
                                        const float2 rh = half2_of(lds16(at), lds16(at + 64)), rl = half2_of(lds16(at + a_half), lds16(at + a_half + 64));
                                        r.x = rh.x + rl.x; r.y = rh.y + rl.y;
                                    }
#pragma unroll
                                    for (int k = 0; k < 2; ++k) {
                                        const float z = v[i + k], s = sigmoidf_(z);
                                        w[i + k] = s * (1.0f + z * (1.0f - s));          // SiLU'
                                        o[i + k] = fmaf(z, s, k ? r.y : r.x);
                                    }
                                }
                                if (last_fwd) {                    // head, and the seed of the backward pass
                                    float p[8];
#pragma unroll
                                    for (int i = 0; i < 8; ++i) { p[i] = o[i] * hw; o[i] = g.gs * hw * w[i]; }
                                    // sums over the 32 features of eight atoms: halves of the atoms change lanes
#pragma unroll
                                    for (int k = 4, off = 16; k >= 1; k >>= 1, off >>= 1) {
                                        const bool up = lane & off;
#pragma unroll
                                        for (int i = 0; i < k; ++i) {
                                            const float send = up ? p[i] : p[i + k], mine = up ? p[i + k] : p[i];
                                            p[i] = mine + __shfl_xor_sync(0xffffffffu, send, off);
                                        }
                                    }
                                    p[0] += __shfl_xor_sync(0xffffffffu, p[0], 2);
                                    p[0] += __shfl_xor_sync(0xffffffffu, p[0], 1);
                                    if ((lane & 3) == 0) head_part[((t0 + j) * 4 + quarter) * g.NA + a0 + (lane >> 2)] = p[0];
                                } else if (g.grad) {
#pragma unroll
                                    for (int i = 0; i < 8; ++i) kd[(size_t)i * F32] = w[i];
                                }
                            } else {
#pragma unroll
                                for (int i = 0; i < 8; ++i) o[i] = v[i] * y[i];
                                if (t > 1) {
#pragma unroll
                                    for (int i = 0; i < 8; ++i) kh[(size_t)i * F32] = v[i];
                                }
                            }
                            if (feeds) {
#pragma unroll
                                for (int i = 0; i < 8; i += 2) {
                                    const uint32_t at = a_col + (uint32_t)(a0 + i) * 64 + ((seg ^ (uint32_t)(i >> 1)) << 4);
                                    const __half2 h = __floats2half2_rn(o[i], o[i + 1]);
                                    const float2 f = __half22float2(h);
                                    const __half2 l = __floats2half2_rn(o[i] - f.x, o[i + 1] - f.y);
                                    const uint32_t hb = *reinterpret_cast<const uint32_t*>(&h), lb = *reinterpret_cast<const uint32_t*>(&l);
                                    sts16(at, hb); sts16(at + 64, hb >> 16);
                                    sts16(at + a_half, lb); sts16(at + a_half + 64, lb >> 16);
                                }
                            }
                        }
                        if (feeds) {                               // this tile of the next operand is written, its accumulators read
                            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) arrive(a_ready + 8 * j);
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (last_fwd) {                                // energies: partial sums of all warps, in a fixed order
                        asm volatile("bar.sync 1, 512;" ::: "memory");
                        const int a = threadIdx.x - 64;
                        if (a < g.NA && m0 + a < g.M) {
                            double e = 0.0;
                            for (int k = 0; k < F32 / 32; ++k) e += (double)head_part[k * g.NA + a];
                            g.e_atom[m0 + a] = e + (double)g.b_head + (double)__ldg(g.e_ref + __ldg(g.row_type + m0 + a));
                        }
                        asm volatile("bar.sync 1, 512;" ::: "memory");     // the next block of atoms rewrites them
                    }
                    if (lane == 0) arrive(acc_free + 8 * buf);     // the accumulators have been read out
                }
            }
            if (lane == 0) arrive(item_done);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

int f32_of(const Dims& d) { return (d.F + 31) & ~31; }
int a_blocks_of(const Dims& d) {
    const int kb0 = (d.DP - d.C0 + 31) / 32, kbf = f32_of(d) / 32;
    return kb0 > kbf ? kb0 : kbf;
}
uint32_t fixed_bytes(const Dims& d, int NA) {           // operand, barriers and partial energies
    return 1024 + (uint32_t)a_blocks_of(d) * (uint32_t)NA * 128 + BAR_AREA + (uint32_t)(MAX_F / 32 * NA) * 4;
}
// most atoms of a block: two accumulators per feature tile in 512 columns, four stages of weights in shared memory
int max_atoms(const Dims& d) {
    const int tiles = (d.F + 127) / 128;
    int na = 512 / (2 * tiles) / 16 * 16;
    if (na > MAX_NA) na = MAX_NA;
    while (na > 16 && fixed_bytes(d, na) + 4 * W_BYTES > SMEM_MAX) na -= 16;
    return na;
}
// atoms per block for n atoms: as many as keep the number of turns of the whole machine at what the largest
// block would need
int pick_atoms(const Dims& d, int n) {
    const int na = max_atoms(d), turns = (n + 148 * na - 1) / (148 * na);
    return ((n + 148 * turns - 1) / (148 * turns) + 15) / 16 * 16;
}

}  // namespace

// One turn of the machine (148 blocks of max_atoms) costs about the same whether the blocks are full or not,
// because the weights stream once per block; a chain of GEMMs costs a launch and a cold pipeline per layer,
// and then passes its rows at a higher rate.  Measured, forward and backward / forward alone, this kernel
// against the chain, us:
//   atoms      F = 96, 3 layers       F = 192, 3 layers      F = 256, 3 layers      F = 256, 2 layers     F = 384, 3 layers
//     500    21 / 15  106 /  66     31 / 21  112 /  70     37 / 24  116 /  70     27 / 19   78 / 48     66 /  40   128 /  77
//   11800    37 / 25  114 /  68     60 / 38  114 /  60     68 / 41  121 /  64     48 / 31   82 / 44    116 /  66   152 /  77
//   23600    62 / 42  108 /  56    109 / 68  171 /  92    126 / 72  188 /  96     87 / 52  118 / 66    220 / 122   246 / 111
//   47000   111 / 70  157 /  86    199 /121  254 / 123    226 /129  280 / 131    152 / 93  166 / 86    427 / 235   414 / 189
//  150000   299 /183  340 / 161    551 /334  637 / 306    625 /358  681 / 321    416 /255  387 /199   1345 / 729  1142 / 505
// (F = 96, forward alone: the line lies below 47,000 atoms, where this kernel is still the faster one; drawn by turns, not by width.)
bool mlp_fused_pick(const Dims& d, int path, int64_t n, bool grad) {
    const bool applies = path == 2 && d.D_out != d.F && (d.F & 7) == 0 && d.F <= MAX_F && d.n_hidden <= kMaxLayers && a_blocks_of(d) <= MAX_KB &&
                         gemm_tc_available();
    if (!applies) return false;
    const int64_t turn = 148 * (int64_t)max_atoms(d);
    if (grad) return d.F <= 192 || (d.F <= 256 && d.n_hidden >= 3) || n <= (d.F <= 256 ? 4 : 2) * turn;
    return n <= (d.F <= 256 ? 2 : 1) * turn;
}

// an upper bound over all n <= n_max
int64_t mlp_fused_scratch_floats(const Dims& d, int64_t n_max) {
    const int64_t na_max = max_atoms(d), blocks = n_max < 148 * 16 ? (n_max + 15) / 16 : 148;
    const int64_t na = n_max >= 148 * na_max ? na_max : ((n_max + 147) / 148 + 15) / 16 * 16;
    return blocks * d.n_hidden * f32_of(d) * na;
}

cudaError_t launch_mlp_fused(const MlpArgs& a, cudaStream_t st) {
    const Dims& d = a.d;
    if (a.n <= 0) return cudaSuccess;
    FusedMaps maps;
    FusedArgs g = {};
    g.M = a.n; g.F = d.F; g.K0 = d.DP - d.C0; g.N0 = d.DP - d.C0; g.NH = d.n_hidden; g.grad = a.want_grad;
    g.NA = pick_atoms(d, a.n);
    g.a_blocks = a_blocks_of(d);
    const int tiles = (d.F + 127) / 128;
    g.bufs = 2 * tiles * 2 * g.NA <= 512 ? 2 : 1;
    const uint32_t fixed = fixed_bytes(d, g.NA);
    const uint32_t keep_floats = (uint32_t)(d.n_hidden * f32_of(d) * g.NA);
    g.keep_in_smem = a.want_grad && fixed + 4 * W_BYTES + 4 * keep_floats <= SMEM_MAX;
    const uint32_t used = fixed + (g.keep_in_smem ? 4 * keep_floats : 0);
    g.stages = (int)((SMEM_MAX - used) / W_BYTES);
    if (g.stages > MAX_STAGES) g.stages = MAX_STAGES;
    g.bias_rows = a.m.type_bias; g.row_type = a.type_s + a.a0;
    g.head_w = a.m.w_head; g.b_head = a.m.b_head; g.e_ref = a.m.e_ref; g.e_atom = a.e_atom + a.a0;
    g.out = a.desc + d.C0; g.ldout = d.DP; g.gs = a.m.grad_scale;
    g.scratch = a.fused_scratch; g.scratch_stride = (size_t)keep_floats;
    g.err = a.err; g.spin_limit = a.spin_limit; g.test_skip = a.test_skip_kblock;
    bool ok = make_map(&maps.a[0], a.tc_hi + d.C0, a.n, g.K0, d.DP, g.NA) && make_map(&maps.a[1], a.tc_lo + d.C0, a.n, g.K0, d.DP, g.NA);
    for (int t = 0; t < d.n_hidden && ok; ++t) {
        const int b = 2 * d.n_hidden - 1 - t;
        g.bias[t] = a.m.bias[t];
        g.acc_scale[t] = g.acc_scale[b] = a.m.w_scale_inv[t];
        if (t == 0) {          // the first C0 feature columns are in the species bias; no gradient is needed for them
            ok = make_map(&maps.w[0][0], a.m.thetaT_hi[0] + d.C0, d.F, g.K0, d.DP) && make_map(&maps.w[0][1], a.m.thetaT_lo[0] + d.C0, d.F, g.K0, d.DP) &&
                 make_map(&maps.w[b][0], a.m.theta_hi[0] + (size_t)d.C0 * d.F, g.N0, d.F, d.F) &&
                 make_map(&maps.w[b][1], a.m.theta_lo[0] + (size_t)d.C0 * d.F, g.N0, d.F, d.F);
        } else {
            ok = make_map(&maps.w[t][0], a.m.thetaT_hi[t], d.F, d.F, d.F) && make_map(&maps.w[t][1], a.m.thetaT_lo[t], d.F, d.F, d.F) &&
                 make_map(&maps.w[b][0], a.m.theta_hi[t], d.F, d.F, d.F) && make_map(&maps.w[b][1], a.m.theta_lo[t], d.F, d.F, d.F);
        }
    }
    if (!ok) return cudaErrorInvalidValue;
    // (per launch, as a kernel's attributes belong to one device and a process may have handles on several)
    const cudaError_t attr = cudaFuncSetAttribute(k_mlp_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX);
    if (attr != cudaSuccess) return attr;
    const int items = (a.n + g.NA - 1) / g.NA;
    return launch_chained(k_mlp_fused, items < 148 ? items : 148, THREADS, used + (uint32_t)g.stages * W_BYTES, st, maps, g);
}

}  // namespace umd
