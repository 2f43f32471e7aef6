// launch.h -- internal (C++) launchers of the libsphtv kernels.  Each takes
// the precision (32 or 64) and dimension (2 or 3) at run time and picks the
// template instantiation.  Not part of the C ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace sphtv {

// Launch with programmatic stream serialization: the kernel is placed as the
// blocks of the one before it exit, without the full drain and flush of a
// plain launch in between, and waits for that kernel's end in pdl_wait(),
// which every kernel launched this way calls before anything else.  Measured
// against plain launches of the same kernels: dual-criteria advection step of
// the 200^2 cavity 192 -> 144 us, rollout 256^2 3.71 -> 3.51 ms, steps
// replayed from a graph 1-3 % (cavity 256^2 43.2 -> 42.2 us).
template <typename... P, typename... A>
inline cudaError_t launch(void (*kern)(P...), int grid, int block, size_t smem, cudaStream_t st, A&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// Forward values of one step kept for the adjoint (device pointers).
struct TapeView {
    const int32_t* id;
    const int8_t* kind;
    const double* x;
    const double* h;
    const double* m;
    const double* s0;
    const void* vr;
    const void* R;
    const int32_t* start;
    const float4* pos4;
    const int32_t* cell;
    const double* dt;
    const uint32_t* nbl;   // the step's force-neighbour list (transposed, nbl_capacity rows)
    const int32_t* nbc;    // and its counts
};

// Adjoint buffers: cotangents in the caller's order ([3][n] FP64) and
// per-step scratch in the sorted order.
struct AdjView {
    double *xc, *vc, *ac, *drc;
    void *AR, *xbp, *vbp, *sigb;   // AR: per particle {Abar, Rbar} (k_adjoint.cu's record layout)
    double* partials;
    double* eta;
};

// k_cells.cu.  Buffers of the sort: each particle's bin (key), the bins'
// counts (zero between sorts) and list heads, the lists' links, the scan's
// within-tile prefixes and tile offsets, and what the sort leaves: the starts
// of the cells and of their sub-cells along x (null without sub-cells).
struct SortBufs {
    int32_t *key, *next;
    int32_t *count, *head, *prefix;
    int32_t* tile_off;
    int32_t *cell_start, *sub_start;
    unsigned* done;        // zero between launches
};
cudaError_t launch_kick_drift_key(int prec, int dim, int n, void* S, const double* dt, int drift, const Grid& G,
                                  int32_t* key, int32_t* count, int32_t* head, int32_t* next, uint32_t* err,
                                  cudaStream_t st);
size_t scan_temp_elems(int n);
cudaError_t launch_bin_scan(int32_t* count, int32_t* prefix, int n, int32_t* tile_off, unsigned* done,
                            cudaStream_t st);
// old_of null: one kernel; else scratch of n for two (see k_order_permute).
cudaError_t launch_order_permute(int prec, int dim, int n, int nbin, const SortBufs& B, void* src, void* dst,
                                 const Grid& G, float4* pos4, int32_t* cell, float* mf, int uniform_h, int carry_ad,
                                 cudaStream_t st, const uint32_t* varies, float4* pos4c, int32_t* old_of);
cudaError_t launch_offsets(int dim, int n, const double* x, const double* h, const double* m, const int32_t* cell,
                           const Grid& G, int uniform_h, float4* pos4, cudaStream_t st);

// What the last block of a pass needs to fold the grid's partials and set the
// next step size: the partials' buffers, the counters (zero between
// launches), the diagnostics and the step size, and whether the pass ends a
// step.
struct FinishArgs {
    double* partials;
    double* rows;          // [grid_groups()][kNPart]
    unsigned* counters;    // [1 + grid_groups()]
    const sph_params* P;
    double* diag;
    double* dt;
    int count_step;
};
struct GridSum;
struct DtConsts;
GridSum grid_sum(const FinishArgs& F, int nblocks);
// After a pass that writes partials (forces, diag_only): the fold of a large
// grid's rows and the end of the step; nothing for a grid that did both.
cudaError_t launch_finish_step(int prec, int n, int sms, const FinishArgs& F, cudaStream_t st, int64_t* launches);
int grid_groups();
DtConsts dt_consts(const sph_params& P);

// k_pair.cu (FP64 form; FP32 calls are forwarded to k_pair32.cu)
int pair_threads(int prec, int n, int sms);
int pair_blocks(int prec, int n, int sms);
// FP64 form: nbl / nbc may be null (no list); with them the density pass
// writes the neighbour list the dual-criteria integrator uses.
cudaError_t launch_density(int prec, int dim, int n, void* S, const int32_t* start, const Grid& G, const void* K,
                           void* vr, const float4* pos4, const int32_t* cell_of, uint32_t* nbl, int32_t* nbc,
                           cudaStream_t st, double* vol = nullptr, const float4* pos4c = nullptr, int tiles = 0);
cudaError_t launch_forces(int prec, int dim, int n, void* S, const int32_t* start, const Grid& G, const void* K,
                          const float* mf, const void* vr, const float4* pos4, const int32_t* cell_of,
                          const uint32_t* nbl, const int32_t* nbc, int kick_on, int write_ad,
                          void* Rout, void* chi, const FinishArgs& F, cudaStream_t st, const double* vol = nullptr);

// k_pair32.cu
int nbl_capacity(int dim);
// tiles: at uniform resolution, the pass on cell-blocked shared-memory tiles
// (same results bit for bit as the row walk over global memory, tiles = 0)
cudaError_t launch_density32(int dim, int n, void* S, const int32_t* start, const Grid& G, const void* K, void* vr,
                             const float4* pos4, const int32_t* cell_of, uint32_t* nbl, int32_t* nbc,
                             cudaStream_t st, const float4* pos4c, int tiles = 0);
cudaError_t launch_forces32(int dim, int n, void* S, const int32_t* start, const Grid& G, const void* K,
                            const float* mf, const void* vr, const float4* pos4, const int32_t* cell_of,
                            const uint32_t* nbl, const int32_t* nbc, int kick_on, int write_ad, void* Rout,
                            void* chi, const FinishArgs& F, cudaStream_t st);
cudaError_t launch_diag_only(int prec, int dim, int n, void* S, const FinishArgs& F, int sms, cudaStream_t st);

// k_io.cu
cudaError_t launch_vec_in(int prec, int dim, int n, const double* src3, void* dst, cudaStream_t st);
// Sources of a state load, in the caller's order, readable by this device's
// kernels.  Null x, v or a, dr: already in the state set, or (zero_v, zero_ad)
// zero; null kind: all fluid; null vw: walls at rest; null sigma0: computed,
// through s0_first.  orig_*: the adjoint's copies, or null.
struct LoadArgs {
    const double *x, *v, *a, *dr, *h, *m, *vw, *sigma0;
    const int8_t* kind;
    int zero_v, zero_ad;
    double* s0_first;
    double *orig_h, *orig_m, *orig_s0, *orig_vw;
    int8_t* orig_kind;
};
cudaError_t launch_load_state(int prec, int dim, int n, const LoadArgs& A, void* S0, void* S1, double rho0,
                              double h_min, double h_max, uint32_t* err, cudaStream_t st, int64_t* launches);
cudaError_t launch_store_state(int prec, int dim, int n, const void* S, const void* vr, double rho0, double* x,
                               double* v, double* a, double* dr, double* rho, cudaStream_t st);
template <typename T>
struct Four {
    T* p[4];
};
cudaError_t launch_cotangents_in(int n, int dim, const Four<const double>& src, const Four<double>& dst,
                                 cudaStream_t st);
cudaError_t launch_cotangents_out(int n, const Four<const double>& src, const Four<double>& dst, cudaStream_t st);
// Output by gathering (coalesced writes in the caller's order): pos from
// launch_inverse_perm of the sorted ids.
cudaError_t launch_inverse_perm(int n, const int32_t* id, int32_t* pos, cudaStream_t st);
cudaError_t launch_vec_out_gather(int prec, int dim, int n, const void* src, const int32_t* pos, double* dst3,
                                  cudaStream_t st);
cudaError_t launch_rho_out_gather(int prec, int n, const void* vr, const int8_t* kind, const int32_t* pos,
                                  double rho0, double* dst, cudaStream_t st);
cudaError_t launch_rho_out(int prec, int n, const void* vr, const int8_t* kind, const int32_t* id, double rho0,
                           double* dst, cudaStream_t st);
cudaError_t launch_scalar_out(int prec, int n, const void* src, const int32_t* id, double* dst, cudaStream_t st);
cudaError_t launch_scalar_in(int prec, int n, const double* src, const int8_t* kind, void* dst, cudaStream_t st);

// k_dual.cu (dual-criteria time stepping).  Device pointers of one context;
// S points at the StateSet<Real> of the current (sorted) copy.
struct DualArgs {
    int n, cap, sms;
    const void* S;
    void* vr;
    float4* pos4;
    void* vr_b;            // FP32 form: second pair of buffers (see k_dual.cu)
    float4* pos4_b;
    const int32_t* cell_of;
    const float* mf;
    const uint32_t* nbl;
    const int32_t* nbc;
    void* anu;
    void* R;
    void* chi;
    double* du;
    FinishArgs F;
    uint32_t* err;
};
cudaError_t launch_dual_begin(const sph_params& P, const double* diag, double* du, cudaStream_t st);
cudaError_t launch_dual_advect(int prec, int dim, const DualArgs& a, const Grid& G, const void* K, cudaStream_t st);
cudaError_t launch_dual_substep(int prec, int dim, const DualArgs& a, const Grid& G, const void* K,
                                cudaStream_t st, int64_t* launches);
cudaError_t launch_dual_complete(int prec, const DualArgs& a, cudaStream_t st);

// k_adjoint.cu
size_t adj_partials(int n);
cudaError_t launch_save_tape(int prec, int dim, int n, int nstart, const void* S, const void* vr, const void* R,
                             const int32_t* start, const float4* pos4, const int32_t* cell, const TapeView& V,
                             cudaStream_t st);
cudaError_t launch_adjoint_step(int prec, int dim, int n, const TapeView& V, const Grid& G, const void* K,
                                const AdjView& A, int step_mode, cudaStream_t st);

}  // namespace sphtv
