// Launchers implemented across the .cu files.  Every launcher enqueues work on the given
// stream and returns the CUDA status of the launch; none of them synchronises unless
// stated.
#pragma once

#include <utility>
#include "common.cuh"

namespace umd {

// ---- neighbor.cu ---------------------------------------------------------------------
// What a build brings back to the host with the edge count, in its one synchronisation: which of the
// T species occur, and the device error word, which is cleared (an image index out of range, a
// non-finite position or a bad species are all found before that point).
struct BuildFetch { int T; int* d_flags; int* h_flags; int* h_err; };
// Full build: fold + bin + sort + count + scan + fill + reverse map.  Synchronises once
// (to learn the edge count and grow the edge arrays).  Returns a UMLMD_* code.
// n_owned < N: the atoms with caller index >= n_owned are ghosts; they come after all owned atoms
// in the internal order (owned atoms in cell order, then ghosts in cell order), so that rows
// [0, n_owned) are the owned atoms' and nb->E_owned edges belong to them.
int neighbor_build(NeighborDev* nb, int64_t N, int64_t n_owned, const double* d_pos, const int32_t* d_type,
                   const double cell[9], const int pbc[3], double skin, double rc, int* d_err,
                   const BuildFetch* fetch, cudaStream_t st, std::string* err);   // cell: the three cell vectors as rows
int neighbor_launches(int64_t N, bool fetch);     // kernels of this library that a build launches
void neighbor_free(NeighborDev* nb);
// Export the list in caller numbering (device buffers of the caller).
int neighbor_export(NeighborDev* nb, int32_t* d_row_ptr, int32_t* d_src, int8_t* d_shift,
                    cudaStream_t st, std::string* err);
// Union of the neighbor lists of n_frames independent frames (atoms concatenated, frame f = atoms
// offsets[f] .. offsets[f+1]-1 with cell cells[9 f ..]), list radius rc, by exhaustive search inside
// each frame (meant for many small frames); atoms keep the caller's order.  Returns a UMLMD_* code.
int neighbor_build_batch(NeighborDev* nb, int n_frames, const int64_t* offsets, const double* cells, const int pbc[3],
                         const double* d_pos, const int32_t* d_type, int T, double rc, int* d_err, const BuildFetch* fetch,
                         cudaStream_t st, std::string* err);
// batched evaluation: forces (caller order is internal order; may be null) and per-row sums of g (x) r (may be null)
cudaError_t launch_frame_rows(const NeighborDev& nb, const float* g, double* d_force, double* row_virial, int* d_err, cudaStream_t st);
// per-frame energy and virial: out[10 f] = sum of e_atom over the frame, out[10 f + 1 ..] = -sum over the frame's rows of
// row_virial (may be null), each by one block in a fixed order; the atomic energies go to d_atom_energy (may be null) as well
cudaError_t launch_frame_reduce(const NeighborDev& nb, const double* e_atom, double* d_atom_energy, const double* row_virial, double* d_out,
                                int* d_err, cudaStream_t st);
// Rows first .. first + n - 1 of the caller's numbering with 64-bit offsets: d_row_ptr [n + 1] is
// always filled; edges are copied while they fit `cap` (cap = 0 or null buffers: offsets only).
int neighbor_export_rows(NeighborDev* nb, int64_t first, int64_t n, int64_t* d_row_ptr, int32_t* d_src,
                         int8_t* d_shift, int64_t cap, cudaStream_t st, std::string* err);
// ---- edge.cu ---------------------------------------------------------------------------
struct EdgeArgs {
    Dims d;
    const float* table;
    const float* pairmod;
    const int4* fix;        // [N] positions in quanta and species (or its slot, see species_slot), one record per atom
    const eidx_t* row_ptr;
    const int2* nbr;        // [E] neighbour (sorted index) and its image
    int Hq[9];              // cell vectors as rows, in quanta; only the diagonal is read unless tri
    int tri;
    float quantum;
    int a0, a1;             // destination range [a0, a1) of this tile
    float* state;           // [a1-a0][SP]: forward writes sums; backward reads dE/d(sums)
    float* g;               // [E][3] per-edge gradient (backward)
    double* virial_part;    // [blocks][9] partial virial sums (backward)
    bool uni;               // the species present are few enough for per-pair amplitude tables:
    // [n_present^2][n_rows][3][C0] cubic pieces of psi_c(rho) of each ordered pair, in the format
    // of the radial table (launch_fuse_pair_tables), read instead of table, pairmod and the radial
    // modes; uni_scale[0..1] = largest |c2|, |c3| of these tables (scale of their packed words)
    // batched evaluation: the image offsets of a row come from the cell of the destination's frame
    const FrameCell* frames;    // null for a single system
    const int* frame_of;
    const float* table_uni;
    const float* uni_scale;
    // the same two tables for values alone (value_piece), read by the forward pass; uni_scale[2..3] = largest
    // |a1|, |a2| of vtable_uni
    const float* vtable;
    const float* vtable_uni;
    // product tables (product_piece), read by the backward pass (wide_channels); uni_scale[4..5] = largest |a1|,
    // |a2| of dtable_uni.  There is no table_uni then.
    const float* dtable;
    const float* dtable_uni;
    const int* species_slot;    // [T] species -> index among the species present; null: the records hold that index
    int n_present;
    // shared radial modes without per-pair tables, from enough rows on: [a1 - a0][n_moments] moments of the rows (forward)
    // or gradients of them (backward), see moments.cu; null: every edge reads its pair's mode mixing
    float* moments;
    int n_moments;
    // one species, from enough rows on: n_moments spline weights per row (moments.cu); spline_n intervals of 1 / spline_inv_h,
    // 0: not by splines
    int spline_n;
    float spline_inv_h, spline_inv_h_lo;      // (as two numbers)
};
constexpr int kEdgeRowsPerBlock = 4, kEdgeSplitRows = 1184;
// present: device array of the n_present species indices, ascending
cudaError_t launch_fuse_pair_tables(const Dims& d, const float* table, const float* pairmod, const int* present,
                                    int n_present, float* scale, float* out, float* vout, float* dout, cudaStream_t st);
cudaError_t launch_edge_forward(const EdgeArgs& a, cudaStream_t st);
cudaError_t launch_edge_backward(const EdgeArgs& a, int* n_blocks, cudaStream_t st);
// Few rows: the four warps of a block share a row, a quarter of its edges each.  A warp works through a row as a
// serial chain of table reads, which a chip with few warps per scheduler does not hide.  One line for both kernels and all
// widths, drawn where the two together were measured: 1184 rows are the 32 warps per SM of the forward kernel up to C0 = 64
// (at C0 = 128 it holds 24, the backward kernel 16 to 24, so that rows then come in more than one wave).  The two kernels
// together took, a warp per row against shared, at
// 108 / 592 / 1184 rows: C0 = 32 28 / 29 / 29 against 21 / 21 / 27 us, C0 = 64 with degree three 44 / 44 / 46 against
// 26 / 27 / 37, C0 = 128 with 64 species 49 / 52 / 58 against 24 / 32 / 52, with four modes 173 / 191 / 208 against
// 62 / 78 / 137; at 1776 rows sharing loses or gains nothing (C0 = 32: 31 against 35, C0 = 128: 63 against 63; with modes not
// measured there).
inline bool edge_rows_split(int64_t rows) { return rows <= kEdgeSplitRows; }
inline int edge_blocks(int rows) { return edge_rows_split(rows) ? rows : (rows + kEdgeRowsPerBlock - 1) / kEdgeRowsPerBlock; }
// most blocks (partial virials) that the tiles of up to N rows, B at a time, have
inline int64_t edge_blocks_max(int64_t N, int64_t B) {
    if (B <= 0) return 0;
    const int64_t last = edge_blocks((int)B), split = B < kEdgeSplitRows ? B : kEdgeSplitRows;
    return N / B * last + (last > split ? last : split);
}

// Plain launches follow one another closely: the kernels around the edge kernels are launched with launch_chained and
// call chain_begin() before they touch global memory that another kernel writes, so that their blocks are set up
// while the kernel before still runs.  The trigger comes after the wait: no more than two kernels of the
// chain are on the chip at a time, and whatever the one before the last wrote is complete.  Build and evaluation of
// 597 atoms 215 -> 206 us, a batch of 64 frames 265 -> 253 us.  Not so launched: the edge kernels themselves (their blocks
// would come up under the shared-memory split of the kernel before, with less L1: 20 steps of 32,400 atoms 14.5 ->
// 16 ms), and any kernel in a captured sequence (50 steps of 4000 atoms 6.85 -> 7.05 ms with such edges in the graph).
#ifdef __CUDACC__
__device__ __forceinline__ void chain_begin() {
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
}
#endif
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kern)(P...), unsigned blocks, unsigned threads, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(blocks); c.blockDim = dim3(threads); c.dynamicSmemBytes = smem; c.stream = st;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(st, &capturing);
    if (e != cudaSuccess) return e;
    c.attrs = &at; c.numAttrs = capturing == cudaStreamCaptureStatusNone ? 1 : 0;
    return cudaLaunchKernelEx(&c, kern, std::forward<A>(args)...);
}

// ---- moments.cu ----------------------------------------------------------------------
struct MomentArgs {
    Dims d;
    const float* pairmod;
    const int* type_s;
    const int* order;       // rows of the tile by species (launch_moment_groups); null with splines
    int a0, n;              // tile start (sorted index) and row count
    float* state;           // [n][SP]
    float* moments;         // [n][pitch]
    int pitch;
    const float* spline;    // [pitch][C0] spline coefficients of the pair's amplitude, null: the pair rows of the modes
};
// From 2048 rows on (the two edge kernels and the products, C0 = 128 with 64 species and four modes, by moments against every
// edge reading its pair's rows: 2100 rows 150 against 211 us, 4000 235 against 406, 40,009 1510 against 2638); below, whole
// blocks of 64 rows of a species are mostly padding.  640 moments (2.5 KB a row) keep the blocks that fit on an SM.
constexpr int kMaxMoments = 640, kMomentRows = 2048;
constexpr int kMaxSplinePitch = 264;            // rows of spline coefficients of the largest fit, 256 intervals
int moment_pitch(const Dims& d);
// whether a tile of so many rows, without per-pair tables, takes the way over moments (true for n implies true for more)
bool moments_pick(const Dims& d, int64_t rows);
int64_t moment_order_ints(const Dims& d, int64_t rows);
// type_s: of the tile; scratch: 2 T ints
cudaError_t launch_moment_groups(const Dims& d, const int* type_s, int n, int* scratch, int* order, cudaStream_t st);
// spline coefficients [pitch][C0] of psi of the pair (t, t) from those of the radial map, coef [n + 7][C0 + R]
cudaError_t launch_spline_pair(const Dims& d, const double* coef, const float* pairmod, int t, int n, int pitch, float* spline, cudaStream_t st);
cudaError_t launch_moments_forward(const MomentArgs& a, cudaStream_t st);    // state += (beta | U)^T moments; = spline^T moments
cudaError_t launch_moments_backward(const MomentArgs& a, cudaStream_t st);   // moments = (beta | U) state; spline state
// Whether the scalar channels of a tile of so many rows, all of one species, go by splines (true for n implies true for more), given
// that the list's rows, with so many listed neighbours on average, are long enough for it to pay.  The products with the coefficients
// cost the same for every row, the edges save with their number and the width.  Edge kernels and products, tables against splines,
// us: C0 = 64 with 274 listed neighbours 30,000 rows 609 and 484, 9000 197 and 178, with 122 neighbours 10,000 rows 118 and 132;
// C0 = 128 with 274 30,000 rows 966 and 675, 9000 304 and 223.
constexpr int kSplineRows = 8192;
inline bool splines_pick(const Dims& d, int64_t rows) { return d.C0 >= 64 && rows >= kSplineRows; }
inline bool splines_pay(const Dims& d, double row_length) { return row_length * d.C0 >= 64 * 180; }

// ---- invariants.cu -------------------------------------------------------------------
struct InvArgs {
    Dims d;
    ModelDev m;
    const int* type_s;
    int a0, n;              // tile start (sorted index) and atom count
    float* state;           // [n][SP]
    float* desc;            // [n][DP]
    // forward only: when non-null the feature rows are also written as their half-precision split
    // (row pitch DP), the form the tensor-core MLP reads; write_desc = false then skips the fp32 copy
    __half* desc_hi;
    __half* desc_lo;
    bool write_desc;
    bool skip_x0_split;     // the split omits the first C0 columns (the MLP folds them into a per-species bias)
};
cudaError_t launch_invariants_forward(const InvArgs& a, cudaStream_t st);
cudaError_t launch_invariants_backward(const InvArgs& a, cudaStream_t st);

// ---- mlp.cu ----------------------------------------------------------------------------
struct MlpArgs {
    Dims d;
    ModelDev m;
    const int* type_s;
    int a0, n;
    float* desc;            // [n][DP]  in: D, out (backward): dE/dD
    float* pre;             // [n_hidden][n][F] pre-activations, overwritten by dE/dY
    float* hbuf;            // [2][n][F] ping-pong activations / hidden gradients
    double* e_atom;         // [N] sorted order, eV (written at a0..a0+n)
    int path;               // 1 = CUDA-core fp32, 2 = tcgen05
    bool want_grad;
    __half* tc_hi;          // two slots of [n][max(DP, F)]: half-precision splits of the activations (tensor-core path)
    __half* tc_lo;
    bool desc_presplit;     // slot 0 already holds the split of desc (written by the invariants kernel)
    bool fold_x0;           // tensor-core path: the first C0 feature columns enter through m.type_bias instead of the GEMM
    size_t tc_slot;         // elements per slot
    int* err;               // device error word
    int spin_limit;         // tensor-core path: polls before a pipeline wait gives up (0 = default)
    int test_skip_kblock;   // diagnostic, first layer of the forward pass only: see GemmArgs
    float* fused_scratch;   // mlp_fused_scratch_floats(); null: one GEMM per layer
};
// mlp_fused.cu: forward layers, head and (grad) input gradient in one kernel.  Path 2, when the first layer has
// no identity residual, a block's activations fit in shared memory (F <= 384) and n atoms are few enough for it
// to be the faster way (true for n implies true for fewer).
bool mlp_fused_pick(const Dims& d, int path, int64_t n, bool grad);
int64_t mlp_fused_scratch_floats(const Dims& d, int64_t n_max);
cudaError_t launch_mlp_fused(const MlpArgs& a, cudaStream_t st);
cudaError_t launch_mlp_forward(const MlpArgs& a, cudaStream_t st);   // layers + head (+ backward seed)
cudaError_t launch_mlp_backward(const MlpArgs& a, cudaStream_t st);  // needs a forward with want_grad

// ---- assemble.cu ---------------------------------------------------------------------
// Current positions of the sorted atoms, from the caller's: see gather_position
struct GatherArgs {
    const int* img; const double* xs0; const int* type_s;
    const int* species_slot;    // what the records hold in place of the species (null: the species itself)
    double* xs; int4* fix;
    double h[9]; int tri;
    double inv_q, max_disp2;
};
GatherArgs gather_args(const NeighborDev& nb, const int* species_slot);
// xs[i] = pos[perm[i]] - img[i]*L and the records of the edge kernels; flags stale / non-finite atoms in *d_err
cudaError_t launch_gather_positions(const NeighborDev& nb, const double* d_pos, const int* species_slot, int* d_err, cudaStream_t st);
// the records of every edge, from the current positions (nb.xs) and the records' species (nb.fix): nb.edge_fix and nb.edge_nbr
cudaError_t launch_edge_records(const NeighborDev& nb, double rc, cudaStream_t st);
// What an MD step does with the forces of an atom once they are there (pos null: nothing): kicks and, if drift, the drift and
// the records of the next evaluation
struct StepTail {
    double* pos; double* vel; const double* inv_mass;
    double dt; int kicks; int drift;
    GatherArgs gather;
};
// d_flags[t] = 1 for every species t in [0, T) that occurs among the N atoms, 0 otherwise;
// kErrSpecies is or-ed into *d_err when an index lies outside [0, T)
cudaError_t launch_species_present(int64_t N, const int* type, int T, int* d_flags, int* d_err, cudaStream_t st);
// per-atom virial shares [N][9] in the caller's numbering from the edge gradients of the last
// backward pass: W_i = -1/2 sum over the edges that touch atom i of g_e (x) r_e
cudaError_t launch_atom_virial(const NeighborDev& nb, const float* g, double* d_out, cudaStream_t st);
// out[0] = sum e_atom, out[1..9] = -sum virial partials (fixed order, double), in one launch; the atomic
// energies go to d_atom_energy (caller's numbering, may be null) on the way.  counter: a zero that comes
// back as zero.  h_out, h_err (pinned, may be null): results and error word for the host; clears the word.
cudaError_t launch_reduce_energy_virial(const NeighborDev& nb, const double* e_atom, double* d_atom_energy, const double* virial_part,
                                        int n_part, double* scratch, unsigned* counter, double* out, int* d_err, double* h_out,
                                        int* h_err, cudaStream_t st);
int reduce_scratch_doubles(int64_t N);
// the same and the force assembly (in one launch, where few atoms make that the better one), with the rest of an MD step (tail)
int assemble_launches(int64_t N);
cudaError_t launch_assemble(const NeighborDev& nb, const float* g, double* d_force, const StepTail& tail,
                            const double* e_atom, double* d_atom_energy, const double* virial_part, int n_part, double* scratch,
                            unsigned* counter, double* out, int* d_err, double* h_out, int* h_err, cudaStream_t st);
cudaError_t launch_unsort_state(const NeighborDev& nb, const float* in, int stride, int width,
                                float* out, cudaStream_t st);
// velocity Verlet pieces (caller order, double)
cudaError_t launch_vv_kick_drift(int64_t N, double* pos, double* vel, const double* force, const int* type,
                                 const double* inv_mass, double dt, int kicks, bool drift, const double* d_scale,
                                 cudaStream_t st);
// Nose-Hoover chain thermostat: chain length, parameters (energies in eV, times in ps) and the
// propagation of `halves` half steps on the device; d_state = [eta[M], v_eta[M], scale, kinetic energy]
constexpr int kNhcChain = 3;
struct NhcParams { double dof, kT, Q[kNhcChain], dt_half; };
// closing half kick (if kick), kinetic energy and `halves` half-step propagations of the chain, one launch
cudaError_t launch_kick_thermostat(int64_t N, double* vel, const double* force, const int* type, const double* mass,
                                   const double* inv_mass, double dt, bool kick, double* scratch, unsigned* counter, double* d_state,
                                   int halves, const NhcParams& p, cudaStream_t st);
cudaError_t launch_kinetic_energy(int64_t N, const double* vel, const int* type, const double* mass,
                                  double* scratch, double* out, cudaStream_t st);

}  // namespace umd
