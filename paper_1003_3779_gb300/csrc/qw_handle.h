// qw_handle.h -- the walk handle behind the opaque qw_walk of the C ABI, and the
// host helpers every ABI source file shares.
#pragma once
#include <string>

#include "qw_internal.cuh"

struct qw_walk {
    // lattice (Sec. 2.2): 1D cycle of nx sites or 2D torus nx * ny, coin dim d
    int ndim = 1, d = 2;
    int64_t nx = 1, ny = 1, ns = 1;
    int bc = QW_BC_PERIODIC, shift = QW_SHIFT_MOVING, prec = QW_F32;
    cudaStream_t stream = nullptr;
    int device = 0;

    // state: two buffers (current / next) of nslots padded planes
    int64_t pitch = 0;
    int nslots = 0, slot_bytes = 0;
    size_t state_bytes = 0;
    void *buf[2] = {nullptr, nullptr};
    int cur = 0;

    // coin
    int kind = qw::CK_REAL;
    int base_kind = qw::CK_REAL;           // CK_PHASE on the torus: the class of the base coin
    double coin_host[32] = {0};            // global / base coin, row-major complex
    double coin_alpha = 1.0;               // sqrt(tr(C_f^dagger C_f) / d) of the rounded coin
    // Hadamard-class coin lambda * diag(a, c) H diag(1, s) (1D moving shift)
    double sign_lambda = 1.0;
    int sign_a = 1, sign_c = 1, sign_s = 1, sign_sigma = 1;
    // error feedback of the rounded per-launch gains: product of applied / ideal
    double gain_fb = 1.0;
    // norm-drift factor of the rounded coin not yet applied to the state
    double drift_pending = 1.0;
    alignas(16) unsigned char coinp[512];  // CoinP<real> in compute precision
    void *coins_dev = nullptr;             // per-site matrices (compute precision)
    size_t coins_bytes = 0;
    float *phi_dev = nullptr;              // per-site phases, nsites * d
    uint8_t *links_dev = nullptr;          // closed-link flags, ndim * nsites
    bool has_links = false;
    // links broken at random at every step (qw_set_link_noise): Philox threshold
    // (0: off), key, and the index of the next forward step
    uint32_t link_thr = 0;
    uint64_t link_seed = 0;
    int64_t link_step = 0;

    // reductions
    double *partials = nullptr;
    double *norm_dev = nullptr;
    double *host_scalar = nullptr;  // pinned
    void *p_dev = nullptr;          // device probabilities for host readout
    size_t p_bytes = 0;

    // staging for host conversions
    void *staging = nullptr;
    size_t staging_bytes = 0;
    // pipelined host runs (qw_run_host_batch): a third state buffer, two
    // probability / norm slots and the copy streams
    void *buf3 = nullptr;
    void *pipe_p[2] = {nullptr, nullptr};
    size_t pipe_p_bytes = 0;
    double *pipe_norm = nullptr;   // one norm per run of qw_run_host_batch
    int64_t pipe_norm_cap = 0;
    cudaStream_t s_in = nullptr, s_out = nullptr;

    // Light-cone clipping (the growing computation window of a localised walk,
    // Sec. 3): the bounding box of the state's support, columns [bx0, bx0 + bw)
    // and rows [by0, by0 + bh) modulo the lattice.  sup_mode 0: the whole
    // lattice is stepped; 1: qw_set_state has queued the box search, whose
    // result arrives in sup_host (event sup_ev); 2: the box is known and the
    // steps run on it, widening it by one site per step and side.  next_clear:
    // the other state buffer is zero outside the box.
    bool clip_on = true;
    int sup_mode = 0;
    int64_t bx0 = 0, bw = 0, by0 = 0, bh = 0;
    bool next_clear = false;
    // dirty_known: no step has run since the state was set, and the other buffer
    // is zero outside the box dirty (the box of the clipped steps before that)
    bool dirty_known = false;
    qw::SupportBox dirty = {0, 0, 0, 0, 1, 1};
    // a call on this handle was captured into a CUDA graph: its replays change
    // the buffers and tables at times the host does not see
    bool captured = false;
    unsigned long long *sup_dev = nullptr;    // 4 values (device)
    unsigned long long *sup_host = nullptr;   // 4 values (pinned)
    cudaEvent_t sup_ev = nullptr;

    // execution plan
    int plan_k = 0, plan_tile = 0;
    int plan_variant = -1;   // 1D kernel: -1 automatic, 0 independent warp tiles, 1 time-skewed sweep
    bool plan_user = false;

    // momentum-space steps of the cycle (k_spectral1d.cuh): calls of at least
    // spec_min steps on an unclipped state run them in launches of up to spec_k
    // steps on blocks of 32 * spec_tile sites (spec_tile 0: off).  Each tile has
    // a table of its own, which stays as long as the handle: captured calls go on
    // reading its twiddles when the other tile is in use.  The matrices of
    // spec_key are in its tile's table; a captured call writes them on every
    // replay, so no matrices are reused after one.
    int spec_tile = 0, spec_k = 0;
    int64_t spec_min = 0;
    bool spec_user = false;   // chosen by qw_set_plan_ex
    void *spec_tables[2] = {nullptr, nullptr};   // by spectral1d_groups(tile) - 1
    // ... of the torus (k_spectral2d.cuh): calls of at least spec_min steps, in
    // the workspace spec_table
    bool spec2 = false;
    void *spec_table = nullptr;
    struct SpecKey {
        double coin[8];
        double scale;
        int K, tile, adjoint;
    } spec_key = {};

    // adjoint / gradient scratch
    void *grad_scratch = nullptr;
    size_t grad_scratch_bytes = 0;

    std::string err;
};

// NVTX ranges around the public calls that launch work, for timelines in a
// profiler; header-only, and nothing happens when no tool is attached
#if __has_include(<nvtx3/nvToolsExt.h>)
#include <nvtx3/nvToolsExt.h>
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
};
#else
struct NvtxRange {
    explicit NvtxRange(const char *) {}
};
#endif

namespace qw {

qw_status set_error(qw_walk *w, qw_status st, const std::string &msg);
qw_status cuda_error(qw_walk *w, cudaError_t e, const char *where);
bool fault_injected(const char *what);
cudaError_t dev_alloc(void **p, size_t bytes);

inline View view_of(const qw_walk *w, int which) {
    return View{w->buf[which], w->pitch, w->d};
}
inline View cur_view(const qw_walk *w) { return view_of(w, w->cur); }
// any closed links, fixed or broken at random: the generic kernel then runs
inline bool links_on(const qw_walk *w) { return w->has_links || w->link_thr != 0; }
inline View next_view(const qw_walk *w) { return view_of(w, w->cur ^ 1); }

// Runs T steps of U (adj = 0) or U^dagger (adj = 1) from buffer `src` into
// the other buffer and flips w->cur; used by qw_step and the adjoint.
qw_status run_steps(qw_walk *w, int64_t T, int adj);

// The support box of the current state (w = 0: the whole lattice, or not known):
// the one the clipped steps track, or, with clipping off, one searched now.
qw_status start_support(qw_walk *w, SupportBox &box);

// Launch helpers implemented in the per-precision translation units.
cudaError_t launch_step1d_f32(const Step1DArgs &, const void *, int, cudaStream_t);
cudaError_t launch_step1d_f64(const Step1DArgs &, const void *, int, cudaStream_t);
cudaError_t launch_step1d_bf16(const Step1DArgs &, const void *, int, cudaStream_t);
cudaError_t launch_step1d_comp(const Step1DArgs &, const void *, int, cudaStream_t);
cudaError_t launch_step2d_f32(const Step2DArgs &, const void *, int, cudaStream_t);
cudaError_t launch_step2d_f64(const Step2DArgs &, const void *, int, cudaStream_t);
cudaError_t launch_step2d_bf16(const Step2DArgs &, const void *, int, cudaStream_t);
cudaError_t launch_step2d_comp(const Step2DArgs &, const void *, int, cudaStream_t);
cudaError_t launch_generic_f32(const StepGenericArgs &, const void *, cudaStream_t);
cudaError_t launch_generic_f64(const StepGenericArgs &, const void *, cudaStream_t);
cudaError_t launch_generic_bf16(const StepGenericArgs &, const void *, cudaStream_t);
cudaError_t launch_generic_comp(const StepGenericArgs &, const void *, cudaStream_t);
cudaError_t launch_window1d_f32(const StepGenericArgs &, const void *, const double *, int, int64_t, int64_t, cudaStream_t);
cudaError_t launch_window1d_f64(const StepGenericArgs &, const void *, const double *, int, int64_t, int64_t, cudaStream_t);
cudaError_t launch_window1d_bf16(const StepGenericArgs &, const void *, const double *, int, int64_t, int64_t, cudaStream_t);
cudaError_t launch_window1d_comp(const StepGenericArgs &, const void *, const double *, int, int64_t, int64_t, cudaStream_t);
bool sweep_ok_f32(int64_t, int, int, int);
bool sweep_ok_f64(int64_t, int, int, int);
bool sweep_ok_bf16(int64_t, int, int, int);
int sweep_tile_f32(int64_t, int);
int sweep_tile_f64(int64_t, int);
int sweep_tile_bf16(int64_t, int);
int tile1d_f32(int, int, int);
int tile1d_f64(int, int, int);
int tile1d_bf16(int, int, int);
int tile1d_comp(int, int, int);

// streaming temporal blocking on the torus (step2d_tb.cu)
bool step2d_tb_ok(int prec, int kind, int K, int shift);
cudaError_t launch_step2d_tb(const Step2DArgs &a, const void *coinp, cudaStream_t s);

// momentum-space steps of the cycle (spectral1d.cu)
int spectral1d_groups(int tile);
bool spectral1d_ok(int prec, int64_t n, int K, int tile);
size_t spectral1d_table_bytes(int prec, int tile);
cudaError_t launch_spectral1d_twiddles(int prec, int tile, void *table, cudaStream_t s);
cudaError_t launch_spectral1d_matrices(int prec, const Spec1DArgs &a, const double *coin, double scale, cudaStream_t s);
cudaError_t launch_spectral1d(int prec, const Spec1DArgs &a, cudaStream_t s);

// momentum-space steps of the torus (spectral2d.cu, FP32): the Grover coin, in
// even numbers of steps, and H (x) H on the diagonal lattice
struct Spec2Plan {
    int K = 0;        // steps per launch (0: none fits)
    double ms = 0;    // estimated time of all launches
};
bool spectral2d_ok(int prec, int kind, int shift);
size_t spectral2d_workspace(int64_t nx, int64_t ny);
Spec2Plan spectral2d_plan(int64_t nx, int64_t ny, int64_t T, bool even);
cudaError_t launch_spectral2d_tables(void *work, cudaStream_t s);
cudaError_t launch_spectral2d(const Step2DArgs &a, int cut_K, int adjoint, void *work, cudaStream_t s);

// a batch of localised walks in momentum space (spectral_batch.cu, FP32)
struct SpecWalk {
    int64_t n, x0, base, pitch, poff;   // as WalkDesc
    int T, id;
    float ah[2], al[2];                 // alpha (re, im), high and low parts
    float b[2], b2h, b2l;               // beta; |beta|^2 in two parts
    float c[4];                         // coin state times e^{i delta T}
};
constexpr int SPEC_BATCH_CLASSES = 6;   // transform lengths 2^8 .. 2^13
int batch_spectral_length(int64_t T);   // log2 of the transform length, 0: T too long
size_t batch_spectral_table_bytes();
cudaError_t launch_batch_spectral_tables(void *table, cudaStream_t s);
cudaError_t launch_batch_spectral(const SpecWalk *walks, const int *count, void *state, float *P, double *norms, int *final_buf,
                                  const void *table, cudaStream_t s);

// K steps in shared-memory tiles (tile2d.cu, FP32); kind: the global coin, or
// with a.phi the base coin of the phases; links: broken links or an edge
cudaError_t launch_tile2d(int shift, int kind, bool links, const Tile2DArgs &a, const void *coinp, cudaStream_t s);

// per-site coin conversion kernels (qw_coins.cu)
cudaError_t launch_convert_coins(int prec, const double *src, void *dst, int64_t count, cudaStream_t s);
cudaError_t launch_phase_coins(int prec, const double *base, const float *phi, void *dst, int64_t ns,
                               int d, cudaStream_t s);

}  // namespace qw
