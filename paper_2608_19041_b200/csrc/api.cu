// extern "C" entry points of libumlmd (see include/umlmd.h for the contract).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>

#include "alloc.h"
#include "kernels.h"
#include "mlp_gemm.h"
#include "model.h"

using namespace umd;

struct umlmd {
    HostModel hm;
    ModelDev md{};
    Dims d{};
    cudaStream_t st = nullptr;
    std::string err;
    NeighborDev nb;
    int node_tile = 524288;
    int mlp_path = 2;   // tensor-core GEMM wherever it applies, CUDA-core GEMM otherwise
    int gemm_spin_limit = 0;      // polls before a tensor-core pipeline wait gives up (0 = default)
    int fault_skip_stage = 0;     // diagnostic, consumed by the first evaluation: see umlmd_options
    bool have_list = false;
    bool on_device = false;
    std::vector<void*> model_allocs;
    // workspace
    float* state = nullptr; float* desc = nullptr; float* pre = nullptr; float* hbuf = nullptr;
    __half* tc_hi = nullptr; __half* tc_lo = nullptr;   // half-precision split of the current GEMM's activations
    float* fused_scratch = nullptr; int64_t fused_cap = 0;      // per-CTA areas of the one-kernel MLP
    int64_t tile_cap = 0;
    // shared radial modes without per-pair tables (moments.cu): moments of a tile's rows, rows of every tile by species
    float* moments = nullptr; int64_t moments_cap = 0;
    int* moment_order = nullptr; int64_t order_cap = 0;
    int* moment_scratch = nullptr;
    // scalar channels by splines (moments.cu): coefficients of the radial map and modes, and of the pair of spline_species
    double* spline_coef = nullptr;
    float* spline = nullptr;
    int spline_species = -1;
    bool splines = false;                            // the list that the caller has built goes that way, and so do the driver's rebuilds of it
    bool have_groups = false;                        // moment_order belongs to the current list
    float* g = nullptr; int64_t g_cap = 0;
    double* e_atom = nullptr; int* type_o = nullptr; int64_t n_cap = 0;
    double* virial_part = nullptr; int64_t vpart_cap = 0;
    double* frame_out = nullptr; int64_t frame_out_cap = 0;     // batched evaluation: [n_frames][10] energy, virial
    double* h_frame = nullptr; int64_t h_frame_cap = 0;         // pinned copy of it: part of `pinned`, or frame_pinned for many frames
    void* frame_pinned = nullptr;
    double* scratch = nullptr; double* d_out = nullptr; int* d_err = nullptr;
    void* pinned = nullptr;                             // one allocation for h_out, h_frame, h_err, h_species and the list's h_totals
    double* h_out = nullptr; int* h_err = nullptr;
    // per-pair amplitude tables of the species present (set up by umlmd_build_neighbors)
    int64_t pair_table_budget = 0;                      // bytes; 0 = the default rule, negative = never build them
    bool pair_tables = false;                           // in use for the current system
    std::vector<int> present;                           // species the tables were built for, ascending
    float* uni = nullptr; int64_t uni_cap = 0;              // one allocation for the four below
    float* uni_scale = nullptr;                         // [6] largest |c2|, |c3|, |a1|, |a2| and |a1|, |a2| of those tables
    float* table_uni = nullptr;                         // [present^2][n_rows][3][C0] (C0 < 32)
    float* vtable_uni = nullptr;                        // [present^2][n_vrows][2][C0], the same for values alone
    float* dtable_uni = nullptr;                        // [present^2][n_vrows][2][C0], envelope products (from C0 = 32 on, instead of table_uni)
    int* d_species = nullptr;                           // [3T]: occurrence flags, species -> slot, present list
    int* h_species = nullptr;                           // [T]
    // MD
    double* md_pos = nullptr; double* md_vel = nullptr; double* md_force = nullptr; int64_t md_cap = 0;    // (capacity in doubles)
    double* d_mass = nullptr; double* d_inv_mass = nullptr;
    bool have_md = false, have_force = false;
    bool have_edge_grad = false;     // h->g holds the edge gradients of the positions in nb.xs
    int steps_since_build = 0;
    double* d_nhc = nullptr;      // thermostat chain on the device: eta[M], v_eta[M], scale, kinetic energy
    bool nhc_reset = true;
    // launch accounting and optional per-class timing
    bool prof_on = false;
    struct Span { int cls; cudaEvent_t a, b; };
    std::vector<Span> spans;
    std::vector<cudaEvent_t> free_events;
    double prof_ms[16] = {0};
    int64_t prof_launches[16] = {0};
    int64_t launches_total = 0;
    // replay of repeated launch sequences as CUDA graphs (see run_replayed)
    struct Replay {
        cudaGraphExec_t exec = nullptr;
        const void* key[4] = {nullptr, nullptr, nullptr, nullptr}; double key_dt = 0, key_x0 = 0, key_x1 = 0; int64_t key_serial = -1; int key_flags = 0;
        bool seen = false;                           // the key's sequence has run once as plain launches
        bool edge_grad = false;                      // it leaves edge gradients (have_edge_grad after it)
        int64_t launches[16] = {0}; int64_t total = 0;   // what one replay launches, per class
    };
    Replay rp_compute, rp_step, rp_nvt;
    int launch_graphs = 0;                           // option: 0 = automatic, 1 = always, -1 = never
    bool graphs_broken = false;                      // a capture failed on this handle: plain launches from then on
    cudaStream_t cap_st = nullptr;                   // stream the sequences are captured on
    int64_t n_owned = -1;                            // atoms [n_owned, N) are ghosts (neighbours only); negative = none
    int64_t graph_replays = 0;
    int64_t list_serial = 0;                         // bumped by everything that changes what a sequence launches
};

enum KernelClass { kGather = 0, kEdgeFwd, kInvFwd, kMlpFwd, kMlpBwd, kInvBwd, kEdgeBwd, kForce, kReduce, kIntegrate,
                   kNeighbor, kClassCount };
static const char* const kClassNames[kClassCount] = {
    "gather_positions", "edge_forward", "invariants_forward", "mlp_forward", "mlp_backward", "invariants_backward",
    "edge_backward", "force_assembly", "energy_virial_reduce", "integrate", "neighbor_build"};

namespace {

// counts the kernels a call site launches and, when profiling is on, brackets them with events
struct Scope {
    umlmd_t* h; int cls; cudaEvent_t a = nullptr;
    static cudaEvent_t get(umlmd_t* h) {
        cudaEvent_t e = nullptr;
        if (!h->free_events.empty()) { e = h->free_events.back(); h->free_events.pop_back(); }
        else cudaEventCreate(&e);
        return e;
    }
    Scope(umlmd_t* h_, int cls_, int n) : h(h_), cls(cls_) {
        h->launches_total += n; h->prof_launches[cls] += n;
        if (h->prof_on) { a = get(h); cudaEventRecord(a, h->st); }
    }
    ~Scope() {
        if (a) { cudaEvent_t b = get(h); cudaEventRecord(b, h->st); h->spans.push_back({cls, a, b}); }
    }
};

int fail(umlmd_t* h, int code, const std::string& msg) {
    if (h) h->err = msg;
    return code;
}

#define API_CUDA(h, call)                                                                     \
    do {                                                                                      \
        cudaError_t e__ = (call);                                                             \
        if (e__ != cudaSuccess)                                                               \
            return fail(h, UMLMD_E_CUDA, std::string(#call) + ": " + cudaGetErrorString(e__)); \
    } while (0)

template <typename T>
cudaError_t upload(umlmd_t* h, const std::vector<T>& v, T** out) {
    *out = nullptr;
    void* p = nullptr;
    cudaError_t e = dev_malloc(&p, v.size() * sizeof(T) + 16);
    if (e != cudaSuccess) return e;
    h->model_allocs.push_back(p);
    if (!v.empty()) e = cudaMemcpyAsync(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, h->st);
    if (e == cudaSuccess) *out = static_cast<T*>(p);
    return e;
}

void fill_info(const Dims& d, umlmd_info* o) {
    o->C0 = d.C0; o->L = d.L; o->R = d.R; o->N_rbf = d.N_rbf; o->n_hidden = d.n_hidden; o->F = d.F; o->T = d.T;
    o->C1 = d.C[1]; o->C2 = d.C[2]; o->K1 = d.K[1]; o->K2 = d.K[2]; o->S = d.S; o->D_out = d.D_out;
    o->H = d.H; o->H_pair = d.Hp; o->table_rows = d.n_rows;
}

// the state of a small single-tile system stays readable after an evaluation (umlmd_get_intermediates)
constexpr int64_t kIntermediatesMaxAtoms = 65536;
bool keeps_intermediates(const umlmd_t* h) { return h->nb.N < kIntermediatesMaxAtoms && h->nb.N <= h->node_tile; }

// whether some evaluation of up to B rows runs its MLP as a chain of GEMMs
bool mlp_needs_chain(const umlmd_t* h, int64_t B) {
    return !(mlp_fused_pick(h->d, h->mlp_path, B, true) && mlp_fused_pick(h->d, h->mlp_path, B, false));
}

// floats that the one-kernel MLP needs for the tiles of `rows` rows, B at a time (none where the rule takes the chain
// for all of them; it takes it for an energy alone wherever it does with a gradient)
int64_t fused_floats(const umlmd_t* h, int64_t rows, int64_t B) {
    int64_t need = 0;
    for (const int64_t n : {rows < B ? rows : B, B > 0 ? rows % B : 0})
        if (n > 0 && mlp_fused_pick(h->d, h->mlp_path, n, true)) need = std::max(need, mlp_fused_scratch_floats(h->d, n));
    return need;
}

int ensure_workspace(umlmd_t* h) {
    const Dims& d = h->d;
    const int64_t N = h->nb.N, E = h->nb.E;
    const int64_t B = N < h->node_tile ? N : h->node_tile;
    // (a capacity of several buffers is zero until all of them are there, so that a failed allocation is made up for later)
    if (B > h->tile_cap) {
        int64_t c;
        h->tile_cap = 0;
        c = 0; API_CUDA(h, dev_ensure(&h->state, &c, B * d.SP));
        c = 0; API_CUDA(h, dev_ensure(&h->desc, &c, B * d.DP));
        const int64_t wmax = d.DP > d.F ? d.DP : d.F;
        const bool chain = mlp_needs_chain(h, B);
        if (chain) {
            c = 0; API_CUDA(h, dev_ensure(&h->pre, &c, B * d.F * d.n_hidden));
            c = 0; API_CUDA(h, dev_ensure(&h->hbuf, &c, B * d.F * 2));
        }
        const int64_t split = chain ? 2 * B * wmax : B * d.DP;      // the one-kernel MLP only reads the feature split
        c = 0; API_CUDA(h, dev_ensure(&h->tc_hi, &c, split));
        c = 0; API_CUDA(h, dev_ensure(&h->tc_lo, &c, split));
        h->tile_cap = B;
    }
    if (const int64_t need = fused_floats(h, h->nb.n_owned, B)) API_CUDA(h, dev_ensure(&h->fused_scratch, &h->fused_cap, need));
    if (E > h->g_cap || !h->g) { API_CUDA(h, dev_ensure(&h->g, &h->g_cap, E * 3, 1.1)); h->g_cap /= 3; }
    if (N > h->n_cap) {
        int64_t c;
        h->n_cap = 0;
        c = 0; API_CUDA(h, dev_ensure(&h->e_atom, &c, N));
        c = 0; API_CUDA(h, dev_ensure(&h->type_o, &c, N));
        h->n_cap = N;
    }
    const int64_t vneed = std::max(edge_blocks_max(N, B) + 2, h->nb.batch ? N : 0) * 9;       // (a batch keeps them by row)
    if (vneed > h->vpart_cap || !h->virial_part) API_CUDA(h, dev_ensure(&h->virial_part, &h->vpart_cap, vneed));
    return UMLMD_OK;
}

int decode_device_errors(umlmd_t* h, int word) {
    if (word & kErrSpecies) return fail(h, UMLMD_E_INVALID_ARG, "species index outside [0, T)");
    if (word & kErrNonFinite) return fail(h, UMLMD_E_NONFINITE, "non-finite value in positions, energy or forces");
    if (word & kErrPipelineTimeout) return fail(h, UMLMD_E_CUDA, "tensor-core GEMM pipeline wait expired");
    if (word & kErrShiftRange) return fail(h, UMLMD_E_UNSUPPORTED_CELL, "periodic image index outside [-127, 127]");
    if (word & kErrStale)
        return fail(h, UMLMD_E_STALE_NEIGHBORS, "an atom moved more than skin/2 since the neighbor list was built");
    return UMLMD_OK;
}

double mean_row(const umlmd_t* h) { return h->nb.N > 0 ? (double)h->nb.E / (double)h->nb.N : 0.0; }      // listed neighbours
// rows of spline coefficients, padded to whole 16-byte pieces
int spline_pitch(const umlmd_t* h) { return (h->hm.spline_n + 7 + 3) / 4 * 4; }
bool use_splines(const umlmd_t* h, int64_t rows) { return h->splines && splines_pick(h->d, rows); }

// what the records of the edge kernels hold in place of the species, null for the species itself
const int* record_slots(const umlmd_t* h) { return h->pair_tables ? h->d_species + h->d.T : nullptr; }

// enqueue one full evaluation; results stay on the device (d_out[0] energy, d_out[1..9] virial)
// (to_host: results and error word also go to h_out and h_err, and the word is cleared; tail: an MD step, whose rest comes
// in the launch that assembles the forces, and whose positions have been gathered)
int enqueue_compute(umlmd_t* h, const double* d_pos, bool want_grad, double* d_force, double* d_atom_energy, bool to_host = false,
                    const StepTail* tail = nullptr) {
    const Dims& d = h->d;
    NeighborDev& nb = h->nb;
    const int N = (int)nb.N;
    const int NR = (int)nb.n_owned;      // rows that are evaluated: the owned atoms, first in the internal order
    // (a batched list was built from these very positions: nothing to gather)
    if (!nb.batch && !tail) { Scope sc(h, kGather, 1); API_CUDA(h, launch_gather_positions(nb, d_pos, record_slots(h), h->d_err, h->st)); }
    if (nb.per_edge) { Scope sc(h, kGather, 1); API_CUDA(h, launch_edge_records(nb, h->hm.rc, h->st)); }
    const int B = N < h->node_tile ? N : h->node_tile;
    int vpart_used = 0;
    for (int a0 = 0; a0 < NR; a0 += B) {
        const int n = NR - a0 < B ? NR - a0 : B;
        EdgeArgs ea;
        ea.d = d; ea.table = h->md.table; ea.pairmod = h->md.pairmod; ea.fix = nb.per_edge ? nb.edge_fix : nb.fix; ea.quantum = (float)(nb.per_edge ? position_quantum(kEdgeRecordReach * h->hm.rc) : nb.quantum);
        ea.uni = h->pair_tables; ea.table_uni = h->table_uni;
        ea.vtable = h->md.vtable; ea.vtable_uni = h->vtable_uni;
        ea.dtable = h->md.dtable; ea.dtable_uni = h->dtable_uni;
        ea.uni_scale = h->uni_scale;
        ea.species_slot = nb.batch ? h->d_species + d.T : nullptr; ea.n_present = (int)h->present.size();
        ea.frames = nb.batch ? nb.frames : nullptr; ea.frame_of = nb.frame_of;
        ea.row_ptr = nb.row_ptr; ea.nbr = nb.per_edge ? nb.edge_nbr : nb.nbr;
        for (int k = 0; k < 9; ++k) ea.Hq[k] = to_quanta(nb.H[k], 1.0 / nb.quantum);
        ea.tri = nb.tri;
        ea.a0 = a0; ea.a1 = a0 + n; ea.state = h->state; ea.g = h->g;
        const bool by_splines = use_splines(h, n), by_moments = by_splines || (h->have_groups && !h->pair_tables && moments_pick(d, n));
        ea.moments = by_moments ? h->moments : nullptr; ea.n_moments = by_splines ? spline_pitch(h) : moment_pitch(d);
        ea.spline_n = by_splines ? h->hm.spline_n : 0; ea.spline_inv_h = (float)(h->hm.spline_n / h->hm.rc);
        ea.spline_inv_h_lo = (float)(h->hm.spline_n / h->hm.rc - (double)ea.spline_inv_h);
        const int* order = by_splines || !by_moments ? nullptr : h->moment_order + (a0 / B) * moment_order_ints(d, B);
        const MomentArgs mo = {d, h->md.pairmod, nb.type_s, order, a0, n, h->state, h->moments, ea.n_moments, by_splines ? h->spline : nullptr};
        ea.virial_part = h->virial_part + (size_t)vpart_used * 9;
        {
            Scope sc(h, kEdgeFwd, 1 + by_moments);
            API_CUDA(h, launch_edge_forward(ea, h->st));
            if (by_moments) API_CUDA(h, launch_moments_forward(mo, h->st));
        }
        InvArgs ia;
        ia.d = d; ia.m = h->md; ia.type_s = nb.type_s; ia.a0 = a0; ia.n = n; ia.state = h->state; ia.desc = h->desc;
        // tensor-core MLP: the invariants kernel writes the first GEMM's operand split itself, and the fp32
        // feature rows only where something still reads them (the identity residual of a first layer as wide
        // as the feature vector; umlmd_get_intermediates makes its own from the state)
        const bool presplit = mlp_uses_tc(d.F, h->mlp_path);
        ia.desc_hi = presplit ? h->tc_hi : nullptr; ia.desc_lo = presplit ? h->tc_lo : nullptr;
        ia.write_desc = !presplit || d.D_out == d.F;
        const bool fold_x0 = presplit && d.D_out != d.F;      // first GEMM skips the per-species constant columns
        ia.skip_x0_split = fold_x0;
        { Scope sc(h, kInvFwd, 1); API_CUDA(h, launch_invariants_forward(ia, h->st)); }
        MlpArgs ma;
        ma.d = d; ma.m = h->md; ma.type_s = nb.type_s; ma.a0 = a0; ma.n = n; ma.desc = h->desc; ma.pre = h->pre;
        ma.hbuf = h->hbuf; ma.e_atom = h->e_atom; ma.path = h->mlp_path; ma.want_grad = want_grad;
        ma.tc_hi = h->tc_hi; ma.tc_lo = h->tc_lo; ma.err = h->d_err; ma.desc_presplit = presplit; ma.fold_x0 = fold_x0;
        ma.tc_slot = (size_t)h->tile_cap * (size_t)(d.DP > d.F ? d.DP : d.F);
        ma.spin_limit = h->gemm_spin_limit; ma.test_skip_kblock = h->fault_skip_stage;
        h->fault_skip_stage = 0;                      // one shot
        ma.fused_scratch = mlp_fused_pick(d, h->mlp_path, n, want_grad) ? h->fused_scratch : nullptr;
        { Scope sc(h, kMlpFwd, ma.fused_scratch ? 1 : d.n_hidden + 1); API_CUDA(h, launch_mlp_forward(ma, h->st)); }
        if (want_grad) {
            if (!ma.fused_scratch) { Scope sc(h, kMlpBwd, d.n_hidden); API_CUDA(h, launch_mlp_backward(ma, h->st)); }
            { Scope sc(h, kInvBwd, 1); API_CUDA(h, launch_invariants_backward(ia, h->st)); }
            int blocks = 0;
            {
                Scope sc(h, kEdgeBwd, 1 + by_moments);
                if (by_moments) API_CUDA(h, launch_moments_backward(mo, h->st));
                API_CUDA(h, launch_edge_backward(ea, &blocks, h->st));
            }
            vpart_used += blocks;
        }
    }
    h->have_edge_grad = want_grad;
    if (nb.batch) return UMLMD_OK;    // (frames are reduced one by one: umlmd_compute_batch)
    double* const ho = to_host ? h->h_out : nullptr;
    int* const he = to_host ? h->h_err : nullptr;
    unsigned* const counter = (unsigned*)h->d_err + 1;
    if (d_force) {
        Scope sc(h, kForce, assemble_launches(N));
        API_CUDA(h, launch_assemble(nb, h->g, d_force, tail ? *tail : StepTail{}, h->e_atom, d_atom_energy,
                                    h->virial_part, vpart_used, h->scratch, counter, h->d_out, h->d_err, ho, he, h->st));
    } else {
        Scope sc(h, kReduce, 1);
        API_CUDA(h, launch_reduce_energy_virial(nb, h->e_atom, d_atom_energy, h->virial_part, vpart_used, h->scratch, counter, h->d_out,
                                                h->d_err, ho, he, h->st));
    }
    return UMLMD_OK;
}

// copy results and the error word to the host and clear the error word (enqueue_fetch), then
// synchronise and decode (finish_fetch)
int enqueue_fetch(umlmd_t* h, int n_out) {
    if (n_out > 0) API_CUDA(h, cudaMemcpyAsync(h->h_out, h->d_out, sizeof(double) * n_out, cudaMemcpyDeviceToHost, h->st));
    API_CUDA(h, cudaMemcpyAsync(h->h_err, h->d_err, sizeof(int), cudaMemcpyDeviceToHost, h->st));
    API_CUDA(h, cudaMemsetAsync(h->d_err, 0, sizeof(int), h->st));
    return UMLMD_OK;
}
int finish_fetch(umlmd_t* h) {
    API_CUDA(h, cudaStreamSynchronize(h->st));
    return decode_device_errors(h, *h->h_err);
}
int fetch_results(umlmd_t* h, int n_out) {
    int rc = enqueue_fetch(h, n_out);
    return rc != UMLMD_OK ? rc : finish_fetch(h);
}

// Replay of a repeated launch sequence.  A system of a few thousand atoms spends more time between
// its two dozen kernels than inside them, so a sequence that recurs with the same arguments (an
// evaluation of the same buffers, a middle step of an MD run between two list builds) is recorded
// once as a CUDA graph and replayed with one launch.  `body` enqueues the sequence on h->st; `key`
// names everything its launches depend on besides the handle's own state, which list_serial covers.
// The first occurrence of a key runs as plain launches (it also performs every lazy one-time
// initialisation of the launch helpers), the second is captured on a stream of the handle's own
// (the caller's may be the legacy default stream, which cannot capture) and every later one
// replayed.  A capture that fails for any reason leaves the handle on plain launches for good.
bool replay_allowed(const umlmd_t* h) {
    if (h->graphs_broken || h->prof_on || h->fault_skip_stage || h->launch_graphs < 0) return false;
    if (h->launch_graphs > 0) return true;
    return h->nb.N <= 65536 && h->nb.N <= h->node_tile;       // automatic: systems where launch latency shows
}
void replay_drop(umlmd_t::Replay& r) {
    if (r.exec) cudaGraphExecDestroy(r.exec);
    r.exec = nullptr;
}
template <class Body>
int run_replayed(umlmd_t* h, umlmd_t::Replay& r, const void* k0, const void* k1, const void* k2, const void* k3,
                 double dt, int flags, Body body, double x0 = 0.0, double x1 = 0.0) {
    if (!replay_allowed(h)) return body();
    const bool same = r.key[0] == k0 && r.key[1] == k1 && r.key[2] == k2 && r.key[3] == k3 && r.key_dt == dt && r.key_x0 == x0 && r.key_x1 == x1 &&
                      r.key_flags == flags && r.key_serial == h->list_serial;
    if (!same) {
        replay_drop(r);
        r.key[0] = k0; r.key[1] = k1; r.key[2] = k2; r.key[3] = k3; r.key_dt = dt; r.key_x0 = x0; r.key_x1 = x1; r.key_flags = flags;
        r.key_serial = h->list_serial; r.seen = true;
        return body();
    }
    if (!r.exec) {
        if (!h->cap_st && cudaStreamCreateWithFlags(&h->cap_st, cudaStreamNonBlocking) != cudaSuccess) {
            cudaGetLastError(); h->graphs_broken = true;
            return body();
        }
        int64_t before[16], total = h->launches_total;
        for (int c = 0; c < 16; ++c) before[c] = h->prof_launches[c];
        cudaStream_t real = h->st;
        h->st = h->cap_st;
        int rc = UMLMD_OK;
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamBeginCapture(h->cap_st, cudaStreamCaptureModeRelaxed);
        if (e == cudaSuccess) {
            rc = body();
            r.edge_grad = h->have_edge_grad;
            e = cudaStreamEndCapture(h->cap_st, &graph);
            if (rc == UMLMD_OK && e == cudaSuccess) e = cudaGraphInstantiate(&r.exec, graph, 0);
            if (graph) cudaGraphDestroy(graph);
        }
        h->st = real;
        for (int c = 0; c < 16; ++c) { r.launches[c] = h->prof_launches[c] - before[c]; h->prof_launches[c] = before[c]; }
        r.total = h->launches_total - total; h->launches_total = total;      // nothing has run yet
        if (rc != UMLMD_OK || e != cudaSuccess || !r.exec) {
            cudaGetLastError();
            replay_drop(r);
            h->graphs_broken = true;
            h->err.clear();
            return body();
        }
    }
    for (int c = 0; c < 16; ++c) h->prof_launches[c] += r.launches[c];
    h->launches_total += r.total;
    ++h->graph_replays;
    API_CUDA(h, cudaGraphLaunch(r.exec, h->st));
    h->have_edge_grad = r.edge_grad;                 // (body, which sets it, has not run)
    return UMLMD_OK;
}

constexpr int64_t kFrameDoubles = 256 * 10;      // results of 256 frames have a place from the start

// first use on a device: upload the model constants and allocate the small result buffers
int ensure_device_model(umlmd_t* h) {
    if (h->on_device) return UMLMD_OK;
    const HostModel& m = h->hm;
    ModelDev& md = h->md;
    cudaError_t e = cudaSuccess;
    auto up = [&](const std::vector<float>& v, float** p) { if (e == cudaSuccess) e = upload(h, v, p); };
    auto uph = [&](const std::vector<__half>& v, __half** p) { if (e == cudaSuccess) e = upload(h, v, p); };
    up(m.pairmod, &md.pairmod); up(m.X0, &md.X0); up(m.W1p, &md.W1p); up(m.W2p, &md.W2p);
    up(m.A1, &md.A1); up(m.A2, &md.A2); up(m.mu, &md.mu); up(m.inv_sigma, &md.inv_sigma);
    up(m.type_bias, &md.type_bias);
    for (int t = 0; t < h->d.n_hidden; ++t) { up(m.theta[t], &md.theta[t]); up(m.thetaT[t], &md.thetaT[t]); up(m.bias[t], &md.bias[t]);
        uph(m.theta_hi[t], &md.theta_hi[t]); uph(m.theta_lo[t], &md.theta_lo[t]);
        uph(m.thetaT_hi[t], &md.thetaT_hi[t]); uph(m.thetaT_lo[t], &md.thetaT_lo[t]);
        md.w_scale_inv[t] = 1.0f / m.w_scale[t]; }
    md.grad_scale = m.grad_scale;
    up(m.w_head, &md.w_head); up(m.e_ref, &md.e_ref);
    md.b_head = m.b_head;
    if (e == cudaSuccess && h->d.L >= 3) {
        std::vector<GauntSparse> g1(1, m.g123), g2(1, m.g233);
        e = upload(h, g1, &md.g123);
        if (e == cudaSuccess) e = upload(h, g2, &md.g233);
    }
    if (e == cudaSuccess && h->d.L >= 4) e = upload(h, m.g4, &md.g4);
    void* p = nullptr;
    if (e == cudaSuccess) { e = dev_malloc(&p, sizeof(double) * (reduce_scratch_doubles(0) + 16)); h->scratch = (double*)p; }
    if (e == cudaSuccess) { e = dev_malloc(&p, sizeof(double) * 16); h->d_out = (double*)p; }
    if (e == cudaSuccess) { e = dev_malloc(&p, sizeof(int) * 4); h->d_err = (int*)p; }
    if (e == cudaSuccess) e = cudaMemsetAsync(h->d_err, 0, sizeof(int) * 4, h->st);
    if (e == cudaSuccess) { e = dev_malloc(&p, sizeof(int) * 3 * (size_t)h->d.T); h->d_species = (int*)p; }
    if (e == cudaSuccess) e = cudaMallocHost(&h->pinned, sizeof(double) * (16 + kFrameDoubles) + sizeof(eidx_t) * 2 + sizeof(int) * (4 + (size_t)h->d.T));
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->st);
    if (e != cudaSuccess) {                    // nothing stays half done: the next call starts over
        cudaStreamSynchronize(h->st);
        for (void* q : h->model_allocs) dev_free(q);
        h->model_allocs.clear();
        dev_free(h->scratch); dev_free(h->d_out); dev_free(h->d_err); dev_free(h->d_species);
        h->scratch = h->d_out = nullptr; h->d_err = h->d_species = nullptr;
        if (h->pinned) cudaFreeHost(h->pinned);
        h->pinned = nullptr;
        return fail(h, UMLMD_E_CUDA, std::string("model upload: ") + cudaGetErrorString(e));
    }
    h->h_out = (double*)h->pinned;
    h->h_frame = h->h_out + 16;
    h->h_frame_cap = kFrameDoubles;
    h->nb.h_totals = (eidx_t*)(h->h_frame + kFrameDoubles);
    h->h_err = (int*)(h->nb.h_totals + 2);
    h->h_species = h->h_err + 4;
    h->on_device = true;
    return UMLMD_OK;
}

// The radial tables that the kernels of the current system read (a list of species with per-pair tables needs the cubic
// pieces to make them, others the value table and, for the backward pass, products or cubic pieces).  The first build
// of a handle waits for these copies: all three took 1 to 1.8 ms more than the one that is needed.
int ensure_radial_tables(umlmd_t* h, bool pair_tables) {
    const bool products = !h->hm.dtable.empty();
    if ((pair_tables || !products) && !h->md.table) API_CUDA(h, upload(h, h->hm.table, &h->md.table));
    if (!pair_tables && !h->md.vtable) API_CUDA(h, upload(h, h->hm.vtable, &h->md.vtable));
    if (!pair_tables && products && !h->md.dtable) API_CUDA(h, upload(h, h->hm.dtable, &h->md.dtable));
    return UMLMD_OK;
}

int build_list(umlmd_t* h, int64_t N, const double* d_pos, const int32_t* d_type, const double cell[9],
               const int pbc[3], double skin, const BuildFetch* fetch) {
    int rc = ensure_device_model(h);
    if (rc != UMLMD_OK) return rc;
    h->have_list = false;            // (until it and the workspace for it are complete)
    { Scope sc(h, kNeighbor, neighbor_launches(N, fetch != nullptr)); rc = neighbor_build(&h->nb, N, h->n_owned, d_pos, d_type, cell, pbc, skin, h->hm.rc, h->d_err, fetch, h->st, &h->err); }
    if (rc != UMLMD_OK) return rc;
    h->have_edge_grad = false;       // edges were renumbered
    h->have_groups = false;          // rows as well
    h->steps_since_build = 0;
    ++h->list_serial;                // recorded launch sequences name the old list
    rc = ensure_workspace(h);
    if (rc != UMLMD_OK) return rc;
    if (h->nb.n_owned < h->nb.N) {
        // ghost atoms come last in the internal order and no stage visits their rows: their atomic
        // energies and the gradients of their edges are zero from here until the next build
        API_CUDA(h, cudaMemsetAsync(h->e_atom + h->nb.n_owned, 0, sizeof(double) * (size_t)(h->nb.N - h->nb.n_owned), h->st));
        if (h->nb.E > h->nb.E_owned)
            API_CUDA(h, cudaMemsetAsync(h->g + 3 * (size_t)h->nb.E_owned, 0, sizeof(float) * 3 * (size_t)(h->nb.E - h->nb.E_owned), h->st));
    }
    h->have_list = true;
    return UMLMD_OK;
}

// Spline coefficients of the one pair of a system of one species.
int setup_splines(umlmd_t* h) {
    const int t = h->present[0];
    if (h->spline_species == t) return UMLMD_OK;
    if (!h->spline_coef) API_CUDA(h, upload(h, h->hm.spline, &h->spline_coef));
    int64_t c = 0;
    if (!h->spline) API_CUDA(h, dev_ensure(&h->spline, &c, (int64_t)spline_pitch(h) * h->d.C0));
    Scope sc(h, kNeighbor, 1);
    API_CUDA(h, launch_spline_pair(h->d, h->spline_coef, h->md.pairmod, t, h->hm.spline_n, spline_pitch(h), h->spline, h->st));
    h->spline_species = t;
    return UMLMD_OK;
}

// Makes room for the moments of a tile's rows, and groups the rows of the current list by species, where its kernels take that way.
// rebuild: of the same atoms by an MD driver, which keeps what the caller's list has decided, so that the way, and with it the
// energy in its last digits, does not change in the middle of a run.
int setup_moments(umlmd_t* h, bool rebuild = false) {
    const Dims& d = h->d;
    const int64_t NR = h->nb.n_owned, B = h->nb.N < h->node_tile ? h->nb.N : h->node_tile, rows = NR < B ? NR : B;
    h->have_groups = false;
    if (!rebuild) h->splines = h->pair_tables && h->present.size() == 1 && h->hm.spline_n > 0 && splines_pick(d, rows) && splines_pay(d, mean_row(h));
    if (h->splines) {
        if (rows * spline_pitch(h) > h->moments_cap) API_CUDA(h, dev_ensure(&h->moments, &h->moments_cap, rows * spline_pitch(h)));
        return setup_splines(h);
    }
    if (h->pair_tables || !moments_pick(d, rows)) return UMLMD_OK;
    const int64_t per_tile = moment_order_ints(d, B);
    int64_t c = 0;
    if (!h->moment_scratch) API_CUDA(h, dev_ensure(&h->moment_scratch, &c, 2 * d.T));
    if (rows * moment_pitch(d) > h->moments_cap) API_CUDA(h, dev_ensure(&h->moments, &h->moments_cap, rows * moment_pitch(d)));
    if ((NR + B - 1) / B * per_tile > h->order_cap) API_CUDA(h, dev_ensure(&h->moment_order, &h->order_cap, (NR + B - 1) / B * per_tile));
    for (int64_t a0 = 0; a0 < NR; a0 += B) {
        const int n = (int)(NR - a0 < B ? NR - a0 : B);
        Scope sc(h, kNeighbor, 2);
        API_CUDA(h, launch_moment_groups(d, h->nb.type_s + a0, n, h->moment_scratch, h->moment_order + a0 / B * per_tile, h->st));
    }
    h->have_groups = true;
    return UMLMD_OK;
}

constexpr int64_t kPairTablesFull = 192ll << 20, kPairTablesMost = 320ll << 20;

// With few species present, psi_c(rho) of every ordered pair among them is tabulated by itself,
// so that the edge kernels read one table row per edge and neither pair rows nor shared modes.
// The tables depend on the model and the set of species only, so they are kept across builds.
int setup_pair_tables(umlmd_t* h) {
    const Dims& d = h->d;
    std::vector<int> present;
    for (int t = 0; t < d.T; ++t) if (h->h_species[t]) present.push_back(t);
    const size_t np = present.size();
    // By default the rule counts tables of three words per channel, of which 4/3 (values and products, from C0 = 32 on) or 5/3
    // (cubic pieces and values) is kept at the usual spacings; a limit that the caller has set bounds what is kept.
    const bool wide = wide_channels(d.C0);
    const int64_t full = (int64_t)(np * np) * d.n_rows * 3 * d.C0 * (int64_t)sizeof(float);
    const size_t vfloats = np * np * (size_t)d.n_vrows * 2 * d.C0, dfloats = wide ? vfloats : 0;
    const size_t floats = wide ? 0 : np * np * (size_t)d.n_rows * 3 * d.C0;
    constexpr size_t head = 32;                       // floats for the scales; the tables behind start on 128 bytes
    const int64_t kept = (int64_t)((head + floats + vfloats + dfloats + 16) * sizeof(float));       // (as dev_ensure pads it)
    const bool fits = h->pair_table_budget > 0 ? kept <= h->pair_table_budget : full <= kPairTablesFull && kept <= kPairTablesMost;
    const bool use = np > 0 && h->pair_table_budget >= 0 && fits;
    h->pair_tables = use && present == h->present;
    if (h->pair_tables) return UMLMD_OK;
    const int rc = ensure_radial_tables(h, use);
    if (rc != UMLMD_OK || !use) return rc;
    h->present.clear();                               // no tables until all of them are made
    API_CUDA(h, dev_ensure(&h->uni, &h->uni_cap, (int64_t)(head + floats + vfloats + dfloats)));
    h->uni_scale = h->uni;
    h->table_uni = h->uni + head;
    h->vtable_uni = h->table_uni + floats;
    h->dtable_uni = h->vtable_uni + vfloats;
    std::vector<int> up(2 * (size_t)d.T, 0);          // species -> slot, then the present list
    for (size_t k = 0; k < np; ++k) { up[present[k]] = (int)k; up[d.T + k] = present[k]; }
    API_CUDA(h, cudaMemcpyAsync(h->d_species + d.T, up.data(), sizeof(int) * up.size(), cudaMemcpyHostToDevice, h->st));
    API_CUDA(h, launch_fuse_pair_tables(d, h->md.table, h->md.pairmod, h->d_species + 2 * d.T, (int)np, h->uni_scale, h->table_uni, h->vtable_uni, h->dtable_uni, h->st));
    API_CUDA(h, cudaStreamSynchronize(h->st));       // `up` is pageable host memory
    h->launches_total += 2;
    h->present = present;
    h->pair_tables = true;
    return UMLMD_OK;
}

}  // namespace

extern "C" {

int umlmd_profile_widths(int32_t C0, int32_t L, int32_t R, umlmd_info* out) {
    if (!out) return UMLMD_E_INVALID_ARG;
    Dims d;
    if (!derive_dims(C0, L, R, &d)) return UMLMD_E_UNSUPPORTED_PROFILE;
    std::memset(out, 0, sizeof(*out));
    fill_info(d, out);
    return UMLMD_OK;
}

int umlmd_create(const void* blob, size_t blob_bytes, const umlmd_options* opt, void* stream, umlmd_t** out) {
    if (!blob || !out) return UMLMD_E_INVALID_ARG;
    *out = nullptr;
    umlmd_t* h = new (std::nothrow) umlmd();
    if (!h) return UMLMD_E_INVALID_ARG;
    h->st = static_cast<cudaStream_t>(stream);
    double dx_override = 0;
    if (opt) {
        if (opt->struct_bytes != sizeof(umlmd_options)) { delete h; return UMLMD_E_INVALID_ARG; }
        if (opt->table_dx < 0 || opt->node_tile < 0 || opt->mlp_path < 0 || opt->mlp_path > 4) { delete h; return UMLMD_E_INVALID_ARG; }
        dx_override = opt->table_dx;
        if (opt->node_tile > 0) h->node_tile = opt->node_tile;
        if (opt->mlp_path > 0) h->mlp_path = opt->mlp_path;
        if (opt->pair_table_mb != 0) h->pair_table_budget = opt->pair_table_mb < 0 ? -1 : (int64_t)opt->pair_table_mb << 20;
        if (opt->gemm_spin_limit < 0 || opt->fault_skip_gemm_stage < 0) { delete h; return UMLMD_E_INVALID_ARG; }
        h->gemm_spin_limit = opt->gemm_spin_limit;
        h->fault_skip_stage = opt->fault_skip_gemm_stage;
        if (opt->launch_graphs < -1 || opt->launch_graphs > 1) { delete h; return UMLMD_E_INVALID_ARG; }
        h->launch_graphs = opt->launch_graphs;
    }
    int rc = build_host_model(blob, blob_bytes, dx_override, &h->hm, &h->err);
    if (rc != UMLMD_OK) { delete h; return rc; }
    h->d = h->hm.d;
    *out = h;
    return UMLMD_OK;
}

int umlmd_destroy(umlmd_t* h) {
    if (!h) return UMLMD_OK;
    if (h->on_device) cudaStreamSynchronize(h->st);
    for (void* p : h->model_allocs) dev_free(p);
    neighbor_free(&h->nb);
    void* ptrs[] = {h->frame_out, h->state, h->desc, h->pre, h->hbuf, h->tc_hi, h->tc_lo, h->fused_scratch, h->moments, h->moment_order, h->moment_scratch, h->spline, h->g, h->e_atom, h->type_o, h->virial_part,
                    h->scratch, h->d_out, h->d_err, h->md_force, h->d_mass, h->d_inv_mass, h->d_nhc, h->uni, h->d_species};
    for (void* p : ptrs) dev_free(p);
    for (auto& sp : h->spans) { cudaEventDestroy(sp.a); cudaEventDestroy(sp.b); }
    for (cudaEvent_t e : h->free_events) cudaEventDestroy(e);
    if (h->rp_compute.exec) cudaGraphExecDestroy(h->rp_compute.exec);
    if (h->rp_step.exec) cudaGraphExecDestroy(h->rp_step.exec);
    if (h->rp_nvt.exec) cudaGraphExecDestroy(h->rp_nvt.exec);
    if (h->cap_st) cudaStreamDestroy(h->cap_st);
    if (h->pinned) cudaFreeHost(h->pinned);
    if (h->frame_pinned) cudaFreeHost(h->frame_pinned);
    delete h;
    return UMLMD_OK;
}

int umlmd_query(const umlmd_t* h, umlmd_info* out) {
    if (!h || !out) return UMLMD_E_INVALID_ARG;
    std::memset(out, 0, sizeof(*out));
    fill_info(h->d, out);
    out->rc = h->hm.rc; out->table_dx = h->hm.dx;
    out->n_atoms = h->have_list ? h->nb.N : 0;
    out->n_edges = h->have_list ? h->nb.E : 0;
    out->device_bytes = dev_bytes_held();
    out->kernel_launches = h->launches_total;
    out->graph_replays = h->graph_replays;
    return UMLMD_OK;
}

const char* umlmd_last_error(const umlmd_t* h) { return h ? h->err.c_str() : "null handle"; }

int umlmd_build_neighbors(umlmd_t* h, int64_t N, const double* d_pos, const int32_t* d_type, const double cell[9],
                          const int pbc[3], double skin) {
    if (!h) return UMLMD_E_INVALID_ARG;
    if (N < 0 || !cell || !pbc || !(skin >= 0) || !std::isfinite(skin) || (N > 0 && (!d_pos || !d_type)))
        return fail(h, UMLMD_E_INVALID_ARG, "bad argument to umlmd_build_neighbors");
    bool diagonal = true;
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) {
            const double v = cell[3 * i + j];
            if (!std::isfinite(v)) return fail(h, UMLMD_E_UNSUPPORTED_CELL, "non-finite cell");
            if (i != j && v != 0.0) diagonal = false;
        }
    if (diagonal)
        for (int i = 0; i < 3; ++i)
            if (!(cell[4 * i] > 0.0)) return fail(h, UMLMD_E_UNSUPPORTED_CELL, "cell edges must be positive");
    h->have_md = false;
    // which species occur: few enough of them get per-pair amplitude tables (see below); comes back with
    // the edge count, and with what the device found wrong (non-finite positions, image range, species)
    int rc = ensure_device_model(h);
    if (rc != UMLMD_OK) return rc;
    *h->h_err = 0;
    for (int t = 0; t < h->d.T; ++t) h->h_species[t] = 0;
    const BuildFetch fetch = {h->d.T, h->d_species, h->h_species, h->h_err};
    rc = build_list(h, N, d_pos, d_type, cell, pbc, skin, &fetch);
    if (rc != UMLMD_OK) return rc;
    h->have_list = false;                        // (until the rest has worked as well)
    rc = decode_device_errors(h, *h->h_err);
    if (rc != UMLMD_OK) return rc;
    if (N > 0) API_CUDA(h, cudaMemcpyAsync(h->type_o, d_type, sizeof(int) * N, cudaMemcpyDeviceToDevice, h->st));
    rc = setup_pair_tables(h);
    if (rc == UMLMD_OK) rc = setup_moments(h);
    h->have_list = rc == UMLMD_OK;
    return rc;
}

int umlmd_get_neighbors(umlmd_t* h, int32_t* d_row_ptr, int32_t* d_src, int8_t* d_shift, int64_t cap,
                        int64_t* n_edges) {
    if (!h || !n_edges) return UMLMD_E_INVALID_ARG;
    if (!h->have_list) return fail(h, UMLMD_E_NO_NEIGHBORS, "no neighbor list built");
    *n_edges = h->nb.E;
    if (cap == 0) return UMLMD_OK;
    if (cap < h->nb.E) return fail(h, UMLMD_E_CAPACITY, "edge buffers smaller than the list");
    if (h->nb.E > 0x7fffffffll) return fail(h, UMLMD_E_CAPACITY, "the export has 32-bit row pointers; this list has more than 2^31 - 1 edges");
    if (!d_row_ptr || (h->nb.E > 0 && (!d_src || !d_shift))) return fail(h, UMLMD_E_INVALID_ARG, "null output buffer");
    int rc = neighbor_export(&h->nb, d_row_ptr, d_src, d_shift, h->st, &h->err);
    if (rc != UMLMD_OK) return rc;
    API_CUDA(h, cudaStreamSynchronize(h->st));
    return UMLMD_OK;
}

int umlmd_get_neighbor_rows(umlmd_t* h, int64_t first_row, int64_t n_rows, int64_t* d_row_ptr, int32_t* d_src,
                            int8_t* d_shift, int64_t cap, int64_t* n_edges) {
    if (!h || !n_edges) return UMLMD_E_INVALID_ARG;
    if (!h->have_list) return fail(h, UMLMD_E_NO_NEIGHBORS, "no neighbor list built");
    if (first_row < 0 || n_rows < 0 || first_row + n_rows > h->nb.N) return fail(h, UMLMD_E_INVALID_ARG, "row range outside [0, N)");
    if (!d_row_ptr) return fail(h, UMLMD_E_INVALID_ARG, "null row offsets");
    if (cap < 0 || (cap > 0 && (!d_src || !d_shift))) return fail(h, UMLMD_E_INVALID_ARG, "null edge buffers");
    int rc = neighbor_export_rows(&h->nb, first_row, n_rows, d_row_ptr, d_src, d_shift, cap, h->st, &h->err);
    if (rc != UMLMD_OK) return rc;
    int64_t total = 0;
    API_CUDA(h, cudaMemcpyAsync(&total, d_row_ptr + n_rows, sizeof(total), cudaMemcpyDeviceToHost, h->st));
    API_CUDA(h, cudaStreamSynchronize(h->st));
    *n_edges = total;
    if (cap > 0 && cap < total) return fail(h, UMLMD_E_CAPACITY, "edge buffers smaller than the rows asked for");
    return UMLMD_OK;
}

int umlmd_workspace_bytes(const umlmd_t* h, int64_t N, int64_t n_edges, int64_t* bytes) {
    if (!h || !bytes || N < 0 || n_edges < 0) return UMLMD_E_INVALID_ARG;
    const Dims& d = h->d;
    const HostModel& m = h->hm;
    auto buf = [](int64_t n, int64_t elem) { return (n + 16) * elem; };          // dev_ensure pads by 16 elements
    auto grown = [](int64_t n, int64_t elem) { return ((int64_t)(n * 1.1) + 16) * elem; };
    int64_t t = 0;
    // model constants (uploaded by the first build)
    auto vec = [&](size_t n, size_t elem) { t += (int64_t)(n * elem + 16); };
    vec(m.table.size(), 4); vec(m.vtable.size(), 4); vec(m.dtable.size(), 4); vec(m.pairmod.size(), 4); vec(m.X0.size(), 4); vec(m.W1p.size(), 4); vec(m.W2p.size(), 4);
    vec(m.A1.size(), 4); vec(m.A2.size(), 4); vec(m.mu.size(), 4); vec(m.inv_sigma.size(), 4); vec(m.type_bias.size(), 4);
    for (int k = 0; k < d.n_hidden; ++k) {
        vec(m.theta[k].size(), 4); vec(m.thetaT[k].size(), 4); vec(m.bias[k].size(), 4);
        vec(m.theta_hi[k].size(), 2); vec(m.theta_lo[k].size(), 2); vec(m.thetaT_hi[k].size(), 2); vec(m.thetaT_lo[k].size(), 2);
    }
    vec(m.w_head.size(), 4); vec(m.e_ref.size(), 4);
    if (d.L >= 3) t += 2 * (int64_t)(sizeof(GauntSparse) + 16);
    if (d.L >= 4) t += (int64_t)(5 * sizeof(GauntSparseBig) + 16);
    t += 8 * (reduce_scratch_doubles(0) + 16) + 8 * 16 + 4 * 4 + 4 * 3 * d.T + 16;
    // neighbor list: per-atom arrays, cell table (at most 8 N + 64 cells), edges, sort / scan scratch
    const int64_t A = N + 1;
    t += buf(3 * A, 8) * 3 + buf(6 * A, 4) + buf(A, 4) * 2 + buf(A + 1, 8) + buf(A, 4) * 4 + buf(A + 1, 4);
    t += buf(8 * N + 64 + 2, 4);
    t += grown(n_edges, 8) * 2;
    t += 16 * A + (2 << 20);
    // evaluation workspace of one node tile, per-edge gradients, per-atom results, MD forces
    const int64_t Bt = N < h->node_tile ? N : h->node_tile;
    const int64_t wmax = d.DP > d.F ? d.DP : d.F;
    t += buf(Bt * d.SP, 4) + buf(Bt * d.DP, 4);
    if (const int64_t need = fused_floats(h, N, Bt)) t += buf(need, 4);
    // rows of spline weights or of moments, never both; which, the species decide: those of this handle's list where that is the
    // system asked for, else the larger
    const bool known = h->have_list && h->nb.N == N && h->nb.E == n_edges;
    const bool splines = known ? h->splines : m.spline_n > 0 && N > 0 && splines_pick(d, Bt) && splines_pay(d, (double)n_edges / (double)N);
    const bool moments = known ? h->have_groups : moments_pick(d, Bt);
    t += std::max(splines ? buf(Bt * spline_pitch(h), 4) + buf((int64_t)spline_pitch(h) * d.C0, 4) + buf((int64_t)m.spline.size(), 8) : 0,
                  moments ? buf(Bt * moment_pitch(d), 4) + buf((N + Bt - 1) / Bt * moment_order_ints(d, Bt), 4) + buf(2 * d.T, 4) : 0);
    if (!mlp_needs_chain(h, Bt)) t += 2 * buf(Bt * d.DP, 2);
    else t += buf(Bt * d.F * d.n_hidden, 4) + buf(Bt * d.F * 2, 4) + 2 * buf(2 * Bt * wmax, 2);
    t += grown(3 * n_edges, 4);
    t += buf(N, 8) + buf(N, 4);
    t += buf(std::max(edge_blocks_max(N, Bt) + 2, N) * 9, 8);
    t += buf(3 * N, 8) + 2 * buf(d.T, 8) + buf(2 * kNhcChain + 2, 8);
    *bytes = t;
    return UMLMD_OK;
}

int umlmd_get_nvt_state(umlmd_t* h, double state[UMLMD_NVT_STATE_DOUBLES]) {
    if (!h || !state) return UMLMD_E_INVALID_ARG;
    static_assert(UMLMD_NVT_STATE_DOUBLES == 2 * kNhcChain, "thermostat state size");
    for (int k = 0; k < UMLMD_NVT_STATE_DOUBLES; ++k) state[k] = 0.0;
    if (!h->d_nhc || h->nhc_reset) return UMLMD_OK;            // chain at rest
    API_CUDA(h, cudaMemcpyAsync(state, h->d_nhc, sizeof(double) * UMLMD_NVT_STATE_DOUBLES, cudaMemcpyDeviceToHost, h->st));
    API_CUDA(h, cudaStreamSynchronize(h->st));
    return UMLMD_OK;
}

int umlmd_set_nvt_state(umlmd_t* h, const double state[UMLMD_NVT_STATE_DOUBLES]) {
    if (!h || !state) return UMLMD_E_INVALID_ARG;
    if (!h->have_md) return fail(h, UMLMD_E_NO_MD_STATE, "umlmd_set_md_state must be called first");
    for (int k = 0; k < UMLMD_NVT_STATE_DOUBLES; ++k)
        if (!std::isfinite(state[k])) return fail(h, UMLMD_E_INVALID_ARG, "non-finite thermostat state");
    if (!h->d_nhc) { int64_t c = 0; API_CUDA(h, dev_ensure(&h->d_nhc, &c, 2 * kNhcChain + 2)); }
    double full[2 * kNhcChain + 2] = {0};
    for (int k = 0; k < UMLMD_NVT_STATE_DOUBLES; ++k) full[k] = state[k];
    full[2 * kNhcChain] = 1.0;
    API_CUDA(h, cudaMemcpyAsync(h->d_nhc, full, sizeof(full), cudaMemcpyHostToDevice, h->st));
    API_CUDA(h, cudaStreamSynchronize(h->st));
    h->nhc_reset = false;
    return UMLMD_OK;
}

int umlmd_compute(umlmd_t* h, const double* d_pos, double* energy, double* d_force, double virial[9],
                  double* d_atom_energy) {
    if (!h) return UMLMD_E_INVALID_ARG;
    if (!h->have_list) return fail(h, UMLMD_E_NO_NEIGHBORS, "umlmd_build_neighbors must be called first");
    if (h->nb.N > 0 && !d_pos) return fail(h, UMLMD_E_INVALID_ARG, "null positions");
    const bool want_grad = d_force != nullptr || virial != nullptr;
    if (h->nb.N == 0) {
        if (energy) *energy = 0;
        if (virial) for (int k = 0; k < 9; ++k) virial[k] = 0;
        return UMLMD_OK;
    }
    int rc = run_replayed(h, h->rp_compute, d_pos, d_force, d_atom_energy, nullptr, 0.0, want_grad ? 1 : 0, [&]() {
        return enqueue_compute(h, d_pos, want_grad, d_force, d_atom_energy, true);
    });
    if (rc != UMLMD_OK) return rc;
    rc = finish_fetch(h);
    if (rc != UMLMD_OK) return rc;
    if (energy) *energy = h->h_out[0];
    if (virial) for (int k = 0; k < 9; ++k) virial[k] = h->h_out[1 + k];
    return UMLMD_OK;
}

int umlmd_compute_batch(umlmd_t* h, int32_t n_frames, const int64_t* frame_offsets, const double* d_pos,
                        const int32_t* d_type, const double* cells, const int pbc[3], double* energies, double* d_force,
                        double* virials, double* d_atom_energy) {
    if (!h) return UMLMD_E_INVALID_ARG;
    if (n_frames < 0 || (n_frames > 0 && (!frame_offsets || !cells)) || !pbc)
        return fail(h, UMLMD_E_INVALID_ARG, "bad argument to umlmd_compute_batch");
    if (n_frames == 0) return UMLMD_OK;
    if (frame_offsets[0] != 0) return fail(h, UMLMD_E_INVALID_ARG, "frame_offsets must start at 0");
    for (int f = 0; f < n_frames; ++f) {
        const int64_t n = frame_offsets[f + 1] - frame_offsets[f];
        if (n < 0) return fail(h, UMLMD_E_INVALID_ARG, "frame_offsets must not decrease");
        if (n > UMLMD_BATCH_MAX_FRAME_ATOMS)
            return fail(h, UMLMD_E_CAPACITY, "a frame of a batch holds more atoms than the exhaustive per-frame search is meant for; use umlmd_build_neighbors");
    }
    const int64_t N = frame_offsets[n_frames];
    if (N > 0x7fff0000LL) return fail(h, UMLMD_E_INVALID_ARG, "too many atoms for 32-bit indices");
    if (N > 0 && (!d_pos || !d_type)) return fail(h, UMLMD_E_INVALID_ARG, "null positions or species");
    int rc = ensure_device_model(h);
    if (rc != UMLMD_OK) return rc;
    h->have_list = false; h->have_md = false; h->have_edge_grad = false;     // the handle's list is replaced
    ++h->list_serial;
    const BuildFetch fetch = {h->d.T, h->d_species, h->h_species, h->h_err};
    { Scope sc(h, kNeighbor, 5); rc = neighbor_build_batch(&h->nb, n_frames, frame_offsets, cells, pbc, d_pos, d_type, h->d.T, h->hm.rc, h->d_err, &fetch, h->st, &h->err); }
    if (rc != UMLMD_OK) return rc;
    const bool want_grad = d_force != nullptr || virials != nullptr;
    if (N > 0) {
        if ((rc = decode_device_errors(h, *h->h_err)) != UMLMD_OK) return rc;
        if ((rc = ensure_workspace(h)) != UMLMD_OK) return rc;
        if ((rc = setup_pair_tables(h)) != UMLMD_OK || (rc = setup_moments(h)) != UMLMD_OK) return rc;
        if ((rc = enqueue_compute(h, d_pos, want_grad, d_force, d_atom_energy)) != UMLMD_OK) return rc;
    }
    const int64_t n_out = (int64_t)n_frames * 10;
    API_CUDA(h, dev_ensure(&h->frame_out, &h->frame_out_cap, n_out));
    if (n_out > h->h_frame_cap) {
        if (h->frame_pinned) cudaFreeHost(h->frame_pinned);
        h->frame_pinned = nullptr; h->h_frame_cap = 0;
        API_CUDA(h, cudaMallocHost(&h->frame_pinned, sizeof(double) * (size_t)n_out));
        h->h_frame = (double*)h->frame_pinned;
        h->h_frame_cap = n_out;
    }
    if (N > 0) {
        double* const row_virial = virials ? h->virial_part : nullptr;         // (the edge kernels' partial sums are not needed)
        if (want_grad) { Scope sc(h, kForce, 1); API_CUDA(h, launch_frame_rows(h->nb, h->g, d_force, row_virial, h->d_err, h->st)); }
        Scope sc(h, kReduce, 1);
        API_CUDA(h, launch_frame_reduce(h->nb, h->e_atom, d_atom_energy, row_virial, h->frame_out, h->d_err, h->st));
    } else {
        API_CUDA(h, cudaMemsetAsync(h->frame_out, 0, sizeof(double) * (size_t)n_out, h->st));
    }
    API_CUDA(h, cudaMemcpyAsync(h->h_frame, h->frame_out, sizeof(double) * (size_t)n_out, cudaMemcpyDeviceToHost, h->st));
    if (N > 0) { if ((rc = fetch_results(h, 0)) != UMLMD_OK) return rc; }
    else API_CUDA(h, cudaStreamSynchronize(h->st));
    for (int f = 0; f < n_frames; ++f) {
        if (energies) energies[f] = h->h_frame[10 * (size_t)f];
        if (virials) for (int k = 0; k < 9; ++k) virials[9 * (size_t)f + k] = h->h_frame[10 * (size_t)f + 1 + k];
    }
    return UMLMD_OK;
}

int umlmd_set_md_state(umlmd_t* h, double* d_pos, double* d_vel, const double* mass_per_type) {
    if (!h) return UMLMD_E_INVALID_ARG;
    if (!h->have_list) return fail(h, UMLMD_E_NO_NEIGHBORS, "umlmd_build_neighbors must be called first");
    if (!d_pos || !d_vel || !mass_per_type) return fail(h, UMLMD_E_INVALID_ARG, "null MD state");
    const int T = h->d.T;
    std::vector<double> m(T), im(T);
    for (int t = 0; t < T; ++t) {
        if (!(mass_per_type[t] > 0) || !std::isfinite(mass_per_type[t])) return fail(h, UMLMD_E_INVALID_ARG, "masses must be positive");
        m[t] = mass_per_type[t]; im[t] = 1.0 / mass_per_type[t];
    }
    h->have_md = false;                          // (until the buffers are there)
    int64_t c = 0;
    if (!h->d_mass) API_CUDA(h, dev_ensure(&h->d_mass, &c, T));
    c = 0;
    if (!h->d_inv_mass) API_CUDA(h, dev_ensure(&h->d_inv_mass, &c, T));
    API_CUDA(h, cudaMemcpyAsync(h->d_mass, m.data(), sizeof(double) * T, cudaMemcpyHostToDevice, h->st));
    API_CUDA(h, cudaMemcpyAsync(h->d_inv_mass, im.data(), sizeof(double) * T, cudaMemcpyHostToDevice, h->st));
    API_CUDA(h, cudaStreamSynchronize(h->st));
    API_CUDA(h, dev_ensure(&h->md_force, &h->md_cap, h->nb.N * 3));
    h->md_pos = d_pos; h->md_vel = d_vel;
    h->have_md = true; h->have_force = false; h->nhc_reset = true;
    ++h->list_serial;                // masses and buffers of the recorded step sequence may have changed
    return UMLMD_OK;
}

// after a drift: rebuild the list if the schedule (rebuild_every > 0) or the displacement
// criterion (rebuild_every < 0) asks for it
static int maybe_rebuild(umlmd_t* h, int rebuild_every) {
    const int64_t N = h->nb.N;
    bool rebuild = rebuild_every > 0 && h->steps_since_build >= rebuild_every;
    if (rebuild_every < 0) {
        // displacement-triggered: the gather pass flags any atom that has moved more than half
        // the skin since the build; read the flag (one host synchronisation per step)
        API_CUDA(h, launch_gather_positions(h->nb, h->md_pos, record_slots(h), h->d_err, h->st));
        API_CUDA(h, cudaMemcpyAsync(h->h_err, h->d_err, sizeof(int), cudaMemcpyDeviceToHost, h->st));
        API_CUDA(h, cudaStreamSynchronize(h->st));
        const int word = *h->h_err;
        if (word & ~kErrStale) {
            API_CUDA(h, cudaMemsetAsync(h->d_err, 0, sizeof(int), h->st));
            return decode_device_errors(h, word & ~kErrStale);
        }
        if (word & kErrStale) {
            API_CUDA(h, cudaMemsetAsync(h->d_err, 0, sizeof(int), h->st));
            rebuild = true;
        }
    }
    if (rebuild) {
        const double skin = h->nb.skin;
        double cell[9];
        for (int k = 0; k < 9; ++k) cell[k] = h->nb.H[k];
        const int pbc[3] = {h->nb.pbc[0], h->nb.pbc[1], h->nb.pbc[2]};
        // The build synchronises the stream anyway (it reads the edge count), so this is the place
        // to look at what the steps since the previous build reported: a list that went stale, or a
        // non-finite value, ends the run here instead of after the last step.
        API_CUDA(h, cudaMemcpyAsync(h->h_err, h->d_err, sizeof(int), cudaMemcpyDeviceToHost, h->st));
        int rc = build_list(h, N, h->md_pos, h->type_o, cell, pbc, skin, nullptr);
        if (rc != UMLMD_OK) return rc;
        const int word = *h->h_err;                  // the build has synchronised the stream since the copy
        if (word) {
            API_CUDA(h, cudaMemsetAsync(h->d_err, 0, sizeof(int), h->st));
            return decode_device_errors(h, word);
        }
        if ((rc = setup_moments(h, true)) != UMLMD_OK) return rc;
    }
    return UMLMD_OK;
}

// error exit of a stepping loop: the error word must not leak into the next call, and the forces
// kept for the next step's opening kick no longer match the positions
static int stop_run(umlmd_t* h, int rc) {
    h->have_force = false;
    if (h->d_err) cudaMemsetAsync(h->d_err, 0, sizeof(int), h->st);
    return rc;
}

int umlmd_step(umlmd_t* h, int nsteps, double dt_ps, int rebuild_every, double* e_pot, double* e_kin) {
    if (!h) return UMLMD_E_INVALID_ARG;
    if (!h->have_list) return fail(h, UMLMD_E_NO_NEIGHBORS, "umlmd_build_neighbors must be called first");
    if (!h->have_md) return fail(h, UMLMD_E_NO_MD_STATE, "umlmd_set_md_state must be called first");
    if (nsteps < 0 || !(dt_ps > 0) || !std::isfinite(dt_ps)) return fail(h, UMLMD_E_INVALID_ARG, "bad step count or time step");
    if (h->nb.n_owned < h->nb.N)
        return fail(h, UMLMD_E_INVALID_ARG, "this driver integrates every atom of the handle; with ghost atoms use umlmd_compute and umlmd_vv_update");
    const int64_t N = h->nb.N;
    int rc;
    if (!h->have_force) {
        if ((rc = enqueue_compute(h, h->md_pos, true, h->md_force, nullptr)) != UMLMD_OK) return rc;
        h->have_force = true;
    }
    bool gathered = false;           // the records of the positions to evaluate are there
    for (int s = 0; s < nsteps; ++s) {
        // opening half kick and drift; from the second step on they come with the forces of the step before
        if (s == 0) { Scope sc(h, kIntegrate, 1); API_CUDA(h, launch_vv_kick_drift(N, h->md_pos, h->md_vel, h->md_force, h->type_o, h->d_inv_mass, dt_ps, 1, true, nullptr, h->st)); }
        ++h->steps_since_build;
        const int64_t serial = h->list_serial;
        if ((rc = maybe_rebuild(h, rebuild_every)) != UMLMD_OK) return stop_run(h, rc);
        if (h->list_serial != serial) gathered = false;
        else if (rebuild_every < 0) gathered = true;         // (by the test for displacements)
        if (!gathered) { Scope sc(h, kGather, 1); API_CUDA(h, launch_gather_positions(h->nb, h->md_pos, record_slots(h), h->d_err, h->st)); }
        const bool last = s + 1 == nsteps;
        auto body = [&]() {
            StepTail t = {h->md_pos, h->md_vel, h->d_inv_mass, dt_ps, last ? 1 : 2, !last, gather_args(h->nb, record_slots(h))};
            return enqueue_compute(h, h->md_pos, true, h->md_force, nullptr, false, &t);
        };
        // a middle step between two list builds launches the same sequence as the one before it
        rc = last ? body() : run_replayed(h, h->rp_step, h->md_pos, h->md_vel, h->md_force, nullptr, dt_ps, 0, body);
        if (rc != UMLMD_OK) return stop_run(h, rc);
        gathered = !last;
    }
    { Scope sc(h, kIntegrate, 2); API_CUDA(h, launch_kinetic_energy(N, h->md_vel, h->type_o, h->d_mass, h->scratch, h->d_out + 10, h->st)); }
    rc = fetch_results(h, 11);
    if (rc != UMLMD_OK) return stop_run(h, rc);
    if (e_pot) *e_pot = h->h_out[0];
    if (e_kin) *e_kin = h->h_out[10];
    return UMLMD_OK;
}

int umlmd_step_nvt(umlmd_t* h, int nsteps, double dt_ps, int rebuild_every, double temperature_K, double t_damp_ps,
                   double* e_pot, double* e_kin, double* e_conserved) {
    if (!h) return UMLMD_E_INVALID_ARG;
    if (!h->have_list) return fail(h, UMLMD_E_NO_NEIGHBORS, "umlmd_build_neighbors must be called first");
    if (!h->have_md) return fail(h, UMLMD_E_NO_MD_STATE, "umlmd_set_md_state must be called first");
    if (nsteps < 0 || !(dt_ps > 0) || !std::isfinite(dt_ps) || !(temperature_K > 0) || !std::isfinite(temperature_K) ||
        !(t_damp_ps > 0) || !std::isfinite(t_damp_ps))
        return fail(h, UMLMD_E_INVALID_ARG, "bad step count, time step, temperature or damping time");
    const int64_t N = h->nb.N;
    if (h->nb.n_owned < N)
        return fail(h, UMLMD_E_INVALID_ARG, "this driver integrates every atom of the handle; with ghost atoms use umlmd_compute and umlmd_vv_update");
    if (N < 2) return fail(h, UMLMD_E_INVALID_ARG, "the thermostat needs at least two atoms");
    constexpr int M = kNhcChain;
    int rc;
    if (!h->d_nhc) { int64_t c = 0; API_CUDA(h, dev_ensure(&h->d_nhc, &c, 2 * M + 2)); h->nhc_reset = true; }
    if (h->nhc_reset) { API_CUDA(h, cudaMemsetAsync(h->d_nhc, 0, sizeof(double) * (2 * M + 2), h->st)); h->nhc_reset = false; }
    NhcParams p;
    p.dof = 3.0 * (double)N - 3.0;
    p.kT = kBoltzmann * temperature_K;
    p.Q[0] = p.dof * p.kT * t_damp_ps * t_damp_ps;
    for (int k = 1; k < M; ++k) p.Q[k] = p.kT * t_damp_ps * t_damp_ps;
    p.dt_half = 0.5 * dt_ps;
    if (!h->have_force) {
        if ((rc = enqueue_compute(h, h->md_pos, true, h->md_force, nullptr)) != UMLMD_OK) return rc;
        h->have_force = true;
    }
    double* d_ke = h->d_out + 10;      // (only of a call without steps)
    double* d_scale = h->d_nhc + 2 * M;
    if (nsteps > 0) {      // opening half step of the chain for the first step
        Scope sc(h, kIntegrate, 1);
        API_CUDA(h, launch_kick_thermostat(N, h->md_vel, h->md_force, h->type_o, h->d_mass, h->d_inv_mass, dt_ps, false, h->scratch,
                                           (unsigned*)h->d_err + 2, h->d_nhc, 1, p, h->st));
    }
    for (int s = 0; s < nsteps; ++s) {
        { Scope sc(h, kIntegrate, 1); API_CUDA(h, launch_vv_kick_drift(N, h->md_pos, h->md_vel, h->md_force, h->type_o, h->d_inv_mass, dt_ps, 1, true, d_scale, h->st)); }
        ++h->steps_since_build;
        if ((rc = maybe_rebuild(h, rebuild_every)) != UMLMD_OK) return stop_run(h, rc);
        const bool last = s + 1 == nsteps;
        auto body = [&]() {
            int r = enqueue_compute(h, h->md_pos, true, h->md_force, nullptr);
            if (r != UMLMD_OK) return r;
            Scope sc(h, kIntegrate, 1);
            // closing half kick and half step of the chain, and the next step's opening one in the same launch
            API_CUDA(h, launch_kick_thermostat(N, h->md_vel, h->md_force, h->type_o, h->d_mass, h->d_inv_mass, dt_ps, true, h->scratch,
                                               (unsigned*)h->d_err + 2, h->d_nhc, last ? 1 : 2, p, h->st));
            return (int)UMLMD_OK;
        };
        // a middle step between two list builds launches the same sequence as the one before it (the
        // opening kick and drift above differ between the first step of a call and the others: plain)
        rc = last ? body() : run_replayed(h, h->rp_nvt, h->md_pos, h->md_vel, h->md_force, h->d_nhc, dt_ps, 0, body,
                                          temperature_K, t_damp_ps);
        if (rc != UMLMD_OK) return stop_run(h, rc);
    }
    if (nsteps > 0) {      // the last scale factor has not been applied to the velocities yet
        Scope sc(h, kIntegrate, 1);
        API_CUDA(h, launch_vv_kick_drift(N, h->md_pos, h->md_vel, h->md_force, h->type_o, h->d_inv_mass, dt_ps, 0, false, d_scale, h->st));
    } else {
        Scope sc(h, kIntegrate, 2);
        API_CUDA(h, launch_kinetic_energy(N, h->md_vel, h->type_o, h->d_mass, h->scratch, d_ke, h->st));
        API_CUDA(h, cudaMemcpyAsync(h->d_nhc + 2 * M + 1, d_ke, sizeof(double), cudaMemcpyDeviceToDevice, h->st));
    }
    double chain[2 * M + 2];
    API_CUDA(h, cudaMemcpyAsync(chain, h->d_nhc, sizeof(chain), cudaMemcpyDeviceToHost, h->st));
    rc = fetch_results(h, 10);
    if (rc != UMLMD_OK) return stop_run(h, rc);
    const double ke = chain[2 * M + 1];
    if (e_pot) *e_pot = h->h_out[0];
    if (e_kin) *e_kin = ke;
    if (e_conserved) {
        double e = h->h_out[0] + ke + p.dof * p.kT * chain[0];
        for (int k = 0; k < M; ++k) e += 0.5 * p.Q[k] * chain[M + k] * chain[M + k];
        for (int k = 1; k < M; ++k) e += p.kT * chain[k];
        *e_conserved = e;
    }
    return UMLMD_OK;
}

int umlmd_atom_virial(umlmd_t* h, double* d_atom_virial) {
    if (!h) return UMLMD_E_INVALID_ARG;
    if (!h->have_list) return fail(h, UMLMD_E_NO_NEIGHBORS, "umlmd_build_neighbors must be called first");
    if (!h->have_edge_grad) return fail(h, UMLMD_E_INVALID_ARG, "no evaluation with forces or virial since the last build");
    if (h->nb.N > 0 && !d_atom_virial) return fail(h, UMLMD_E_INVALID_ARG, "null output buffer");
    { Scope sc(h, kForce, 1); API_CUDA(h, launch_atom_virial(h->nb, h->g, d_atom_virial, h->st)); }
    API_CUDA(h, cudaStreamSynchronize(h->st));
    return UMLMD_OK;
}

int umlmd_set_owned_atoms(umlmd_t* h, int64_t n_owned) {
    if (!h) return UMLMD_E_INVALID_ARG;
    h->n_owned = n_owned < 0 ? -1 : n_owned;
    // the internal order of the atoms depends on it: the next evaluation needs a new list
    h->have_list = false; h->have_md = false; h->have_force = false; h->have_edge_grad = false;
    ++h->list_serial;
    return UMLMD_OK;
}

int umlmd_vv_update(int64_t N, double* d_pos, double* d_vel, const double* d_force, const int32_t* d_type,
                    const double* d_inv_mass_per_type, double dt_ps, int32_t half_kicks, int32_t drift, void* stream) {
    if (N < 0 || half_kicks < 0 || half_kicks > 2 || !(dt_ps > 0) || !std::isfinite(dt_ps)) return UMLMD_E_INVALID_ARG;
    if (N > 0 && (!d_vel || !d_type || !d_inv_mass_per_type || (half_kicks > 0 && !d_force) || (drift && !d_pos)))
        return UMLMD_E_INVALID_ARG;
    if (N == 0 || (half_kicks == 0 && !drift)) return UMLMD_OK;
    cudaError_t e = launch_vv_kick_drift(N, d_pos, d_vel, d_force, d_type, d_inv_mass_per_type, dt_ps, half_kicks, drift != 0,
                                         nullptr, static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? UMLMD_OK : UMLMD_E_CUDA;
}

int umlmd_get_intermediates(umlmd_t* h, float* d_state, float* d_desc) {
    if (!h) return UMLMD_E_INVALID_ARG;
    if (!h->have_list) return fail(h, UMLMD_E_NO_NEIGHBORS, "no neighbor list built");
    if (!keeps_intermediates(h)) return fail(h, UMLMD_E_CAPACITY, "intermediates are only kept for systems of one tile and fewer than 65536 atoms");
    if (d_state) API_CUDA(h, launch_unsort_state(h->nb, h->state, h->d.SP, h->d.S + 2, d_state, h->st));
    if (d_desc && !h->have_edge_grad && h->nb.n_owned > 0) {      // (after a backward pass both buffers hold gradients)
        InvArgs ia = {};
        ia.d = h->d; ia.m = h->md; ia.type_s = h->nb.type_s; ia.a0 = 0; ia.n = (int)h->nb.n_owned; ia.state = h->state; ia.desc = h->desc;
        ia.write_desc = true;
        API_CUDA(h, launch_invariants_forward(ia, h->st));
    }
    if (d_desc) API_CUDA(h, launch_unsort_state(h->nb, h->desc, h->d.DP, h->d.D_out, d_desc, h->st));
    API_CUDA(h, cudaStreamSynchronize(h->st));
    return UMLMD_OK;
}

int umlmd_eval_radial_table(const umlmd_t* h, int64_t n, const double* rho, double* out_g, double* out_dg) {
    if (!h || n < 0 || (n > 0 && (!rho || !out_g))) return UMLMD_E_INVALID_ARG;
    const Dims& d = h->d;
    const int NC = d.C0 + d.R;
    for (int64_t i = 0; i < n; ++i) {
        int row = (int)std::floor(rho[i] / h->hm.dx);
        if (row < 0) row = 0;
        if (row > d.n_rows - 1) row = d.n_rows - 1;
        const double t = rho[i] - row * h->hm.dx;
        const float* p = &h->hm.table[(size_t)row * 3 * d.CP];
        for (int c = 0; c < NC; ++c) {
            unsigned w;
            std::memcpy(&w, &p[2 * d.CP + c], sizeof(w));
            float h2, h3;
            tab_unpack(w, d.tab_k2, d.tab_k3, &h2, &h3);
            const double c0 = p[c], c1 = p[d.CP + c], c2 = h2, c3 = h3;
            out_g[i * NC + c] = ((c3 * t + c2) * t + c1) * t + c0;
            if (out_dg) out_dg[i * NC + c] = (3 * c3 * t + 2 * c2) * t + c1;
        }
    }
    return UMLMD_OK;
}

int umlmd_eval_edge_splines(umlmd_t* h, int32_t type, int64_t n, const double* rho, double* out_psi, double* out_dpsi) {
    if (!h || n < 0 || (n > 0 && (!rho || !out_psi)) || type < 0 || type >= h->d.T) return UMLMD_E_INVALID_ARG;
    const Dims& d = h->d;
    const HostModel& m = h->hm;
    if (m.spline_n == 0) return fail(h, UMLMD_E_UNSUPPORTED_PROFILE, "this model has no splines");
    const int rows = m.spline_n + 7;
    std::vector<float> S((size_t)rows * d.C0);
    const float* pm = &m.pairmod[(size_t)(type * d.T + type) * (2 + d.R) * d.C0];
    for (int c = 0; c < d.C0; ++c) {
        double left = 0;
        for (int k = 0; k < rows; ++k) S[(size_t)k * d.C0 + c] = spline_coefficient(d, &m.spline[(size_t)k * (d.C0 + d.R)], pm + c, c, &left);
    }
    for (int64_t i = 0; i < n; ++i) {
        const double x = std::min(std::max(rho[i], 0.0), m.rc) * (m.spline_n / m.rc);
        const int k = std::max(0, std::min((int)x, m.spline_n - 1));          // (a distance that is no number gives no number)
        double w[8], dw[8];
        spline_weights(x - k, w, dw);
        for (int c = 0; c < d.C0; ++c) {
            double v = 0, dv = 0;
            for (int a = 0; a < 8; ++a) { const double q = 5040.0 * S[(size_t)(k + a) * d.C0 + c]; v += w[a] * q; dv += dw[a] * q; }
            out_psi[i * d.C0 + c] = v;
            if (out_dpsi) out_dpsi[i * d.C0 + c] = dv * (m.spline_n / m.rc);
        }
    }
    return UMLMD_OK;
}

int umlmd_eval_edge_tables(const umlmd_t* h, int32_t type_i, int32_t type_j, int32_t per_pair, int64_t n, const double* rho,
                           double* out_psi, double* out_dchipsi) {
    if (!h || n < 0 || (n > 0 && (!rho || !out_psi))) return UMLMD_E_INVALID_ARG;
    const Dims& d = h->d;
    if (type_i < 0 || type_j < 0 || type_i >= d.T || type_j >= d.T) return UMLMD_E_INVALID_ARG;
    const HostModel& m = h->hm;
    const int C0 = d.C0, R = d.R;
    const double dx = h->hm.dx, w = dx / d.v_sub;
    const bool products = wide_channels(C0);             // what the backward pass reads: else rows with derivatives
    auto pair_row = [&](int a, int b) { return &m.pairmod[(size_t)(a * d.T + b) * (2 + R) * C0]; };
    auto word = [](const float* p) { unsigned u; std::memcpy(&u, p, sizeof(u)); return u; };
    // steps of the packed words of tables made for a system of these two species
    double big[6] = {0, 0, 0, 0, 0, 0};
    const int two[2] = {type_i, type_j};
    for (int s = 0; per_pair && s < d.n_rows; ++s)
        for (int ab = 0; ab < 4; ++ab)
            for (int c = 0; c < C0; ++c) {
                double v[4], q[4];
                pair_cubic(d, &m.table[(size_t)s * 3 * d.CP], pair_row(two[ab >> 1], two[ab & 1]) + c, c, v);
                auto grow = [&](int k, double x) { big[k] = std::fmax(big[k], std::fabs((double)(float)x)); };
                grow(0, v[2]); grow(1, v[3]);
                for (int sub = 0; sub < d.v_sub; ++sub) {
                    value_piece(v[0], v[1], v[2], v[3], (sub + 0.5) * w, 0.5 * w, q);
                    grow(2, q[1]); grow(3, q[2]);
                    if (!products) continue;
                    double e[5];
                    envelope_derivatives(s * dx + (sub + 0.5) * w, (double)d.rc, e);
                    product_piece(v[0], v[1], v[2], v[3], (sub + 0.5) * w, 0.5 * w, e, q);
                    grow(4, q[1]); grow(5, q[2]);
                }
            }
    const float step[6] = {per_pair ? tab_step2((float)big[0]) : d.tab_k2, per_pair ? tab_step3((float)big[1]) : d.tab_k3,
                           per_pair ? tab_step2((float)big[2]) : d.tab_v1, per_pair ? tab_step3((float)big[3]) : d.tab_v2,
                           per_pair ? tab_step2((float)big[4]) : d.tab_d1, per_pair ? tab_step3((float)big[5]) : d.tab_d2};
    const float* pm = pair_row(type_i, type_j);
    for (int64_t i = 0; i < n; ++i) {
        const double r = rho[i], x = r / (double)d.rc, u = 1 - x;
        const double chi = u * u * u * u * (1 + x * (4 + x * (10 + x * (20 + 35 * x)))), dchi = -280 * x * x * x * x * u * u * u / (double)d.rc;
        auto at = [&](double spacing, int rows) {
            const int row = (int)std::floor(r / spacing);
            return row < 0 ? 0 : (row > rows - 1 ? rows - 1 : row);
        };
        const int vrow = at(w, d.n_vrows), row = at(dx, d.n_rows), crow = vrow / d.v_sub;
        const double t = r - (vrow + 0.5) * w, tc = r - row * dx, mid = (vrow % d.v_sub + 0.5) * w, rho_mid = (vrow + 0.5) * w;
        // one piece: from the stored word, or rounded and packed as the tables of a pair are
        auto stored = [&](const std::vector<float>& tab, int c, const float* st) {
            const float* p = &tab[(size_t)vrow * 2 * d.CP + c];
            float a1, a2;
            tab_unpack(word(p + d.CP), st[0], st[1], &a1, &a2);
            return ((double)a2 * t + (double)a1) * t + (double)p[0];
        };
        auto packed = [&](const double* a, const float* st) {
            float a1, a2;
            tab_unpack(tab_pack((float)a[1], (float)a[2], st[0], st[1]), st[0], st[1], &a1, &a2);
            return ((double)a2 * t + (double)a1) * t + (double)(float)a[0];
        };
        for (int c = 0; c < C0; ++c) {
            double v[4], q[4], psi, out;
            if (per_pair) {
                pair_cubic(d, &m.table[(size_t)crow * 3 * d.CP], pm + c, c, v);
                value_piece(v[0], v[1], v[2], v[3], mid, 0.5 * w, q);
                psi = packed(q, step + 2);
            } else {
                psi = (double)pm[c] * stored(m.vtable, c, step + 2) + (double)pm[C0 + c];
                for (int k = 0; k < R; ++k) psi += (double)pm[(size_t)(2 + k) * C0 + c] * stored(m.vtable, C0 + k, step + 2);
            }
            if (products && per_pair) {
                double e[5];
                envelope_derivatives(rho_mid, (double)d.rc, e);
                product_piece(v[0], v[1], v[2], v[3], mid, 0.5 * w, e, q);
                out = packed(q, step + 4);
            } else if (products) {
                out = (double)pm[c] * stored(m.dtable, c, step + 4) + (double)pm[C0 + c] * dchi;
                for (int k = 0; k < R; ++k) out += (double)pm[(size_t)(2 + k) * C0 + c] * stored(m.dtable, C0 + k, step + 4);
            } else {
                pair_cubic(d, &m.table[(size_t)row * 3 * d.CP], pm + c, c, v);
                float c2 = (float)v[2], c3 = (float)v[3];
                if (per_pair) {
                    tab_unpack(tab_pack(c2, c3, step[0], step[1]), step[0], step[1], &c2, &c3);
                    v[0] = (float)v[0]; v[1] = (float)v[1]; v[2] = c2; v[3] = c3;
                }
                out = chi * ((3 * v[3] * tc + 2 * v[2]) * tc + v[1]) + dchi * (((v[3] * tc + v[2]) * tc + v[1]) * tc + v[0]);
            }
            out_psi[i * C0 + c] = psi;
            if (out_dchipsi) out_dchipsi[i * C0 + c] = out;
        }
    }
    return UMLMD_OK;
}

int umlmd_set_profiling(umlmd_t* h, int enabled) {
    if (!h) return UMLMD_E_INVALID_ARG;
    h->prof_on = enabled != 0;
    return UMLMD_OK;
}

int umlmd_get_profile(umlmd_t* h, int32_t max_classes, double* ms, int64_t* launches, int32_t* n_classes) {
    if (!h || !n_classes || max_classes < 0) return UMLMD_E_INVALID_ARG;
    if (h->on_device) API_CUDA(h, cudaStreamSynchronize(h->st));
    for (auto& sp : h->spans) {
        float t = 0.f;
        if (cudaEventElapsedTime(&t, sp.a, sp.b) == cudaSuccess) h->prof_ms[sp.cls] += t;
        h->free_events.push_back(sp.a);
        h->free_events.push_back(sp.b);
    }
    h->spans.clear();
    *n_classes = kClassCount;
    for (int k = 0; k < kClassCount && k < max_classes; ++k) {
        if (ms) ms[k] = h->prof_ms[k];
        if (launches) launches[k] = h->prof_launches[k];
    }
    for (int k = 0; k < kClassCount; ++k) { h->prof_ms[k] = 0; h->prof_launches[k] = 0; }
    return UMLMD_OK;
}

const char* umlmd_profile_class_name(int32_t cls) {
    return (cls >= 0 && cls < kClassCount) ? kClassNames[cls] : "";
}

int umlmd_eval_pair_cache(const umlmd_t* h, int32_t type_i, int32_t type_j, double* out) {
    if (!h || !out) return UMLMD_E_INVALID_ARG;
    const Dims& d = h->d;
    if (type_i < 0 || type_j < 0 || type_i >= d.T || type_j >= d.T) return UMLMD_E_INVALID_ARG;
    const size_t n = (size_t)(2 + d.R) * d.C0;
    const float* p = &h->hm.pairmod[(size_t)(type_i * d.T + type_j) * n];
    for (size_t k = 0; k < n; ++k) out[k] = p[k];
    return UMLMD_OK;
}

}  // extern "C"
