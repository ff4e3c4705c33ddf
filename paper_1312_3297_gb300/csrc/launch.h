// Internal launch interface between the C-ABI layer (lbmrv_api.cu) and the kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "d2q9.cuh"
#include "d3q19.cuh"

namespace lbmrv {

enum { kStoreF32 = 0, kStoreF16 = 1, kStoreBF16 = 2 };

constexpr int kReduceThreads = 256;
// Most partial sums of a reduction (8 blocks per SM of a 152-SM GB300; any GPU works with
// it). A compile-time constant because it sizes the fixed scratch of
// lbmrv_conserved_noalloc.
constexpr int kReduceMaxBlocks = 152 * 8;
// Blocks of the reduction kernels resident on one SM, at least (their launch bounds).
constexpr int kReduceMinBlocks = 4;

// Blocks of a grid-stride kernel over n items with `threads` per block: enough for every
// item, at most 16 per SM of the current device (found once per device).
int grid_stride_blocks(int64_t n, int threads);

// Widest vector pack (nodes per thread) the fused step can use for this row length.
int step_vector_width(int storage, int nx);

// One fused step src -> dst. um: UM_* of d2q9.cuh; nv: 1 (scalar kernel) or a vector
// width returned by step_vector_width (or any smaller power of two dividing nx); basis 0:
// the orthogonal moments of the paper's D2Q9 example, 1: Geier's (cascaded) basis.
cudaError_t launch_step(int storage, int um, int nv, const void* src, void* dst,
                        const StepArgs& a, cudaStream_t st, int basis = 0);

// SMs of the current device (152 if the runtime does not say).
int sm_count();

// Modelled times of one step in microseconds, for the choice between the forms of the D2Q9
// step: one launch per step at pack width nv; one of launch_march's three (kNoForm where it does
// not suit the lattice: row length, alignment; ut0 the stored field, or null).
constexpr double kNoForm = 1e30;
double single_step_us(int storage, int um, int basis, int nv, int nx, int ny);
double beyond_l2(int storage, int um, int nx, int ny, double lo, double hi);
double march_step_us(int storage, int um, int basis, int nx, int ny, const void* a,
                     const void* b, const float* ut0);

// kMarchSteps steps src -> dst in one pass over memory (d2q9_march.cu), the bits of that many
// launch_step calls. a: the arguments of the first of them; amps: amp_t of each.
constexpr int kMarchSteps = 3;
constexpr int kMarchMany = 8;  // passes of a call from which on the first of them starts alone
enum class MarchStart { kShare, kAlone, kFollow };  // see launch_w in d2q9_march.cu
struct MarchAmps {
    float v[kMarchSteps];
};
cudaError_t launch_march(int storage, int um, const void* src, void* dst, const StepArgs& a,
                         const MarchAmps& amps, cudaStream_t st, int basis,
                         MarchStart start);

// p.steps steps src -> dst in one launch on shared-memory tiles (d2q9_tile.cuh): arrays of p.rx
// x p.ry nodes, blocks of p.warps warps. The bits of that many launch_step calls at pack width nv.
constexpr int kTileMaxSteps = 12;
constexpr int kTileMaxSmem = 224 * 1024;
constexpr int kTileWarps = 24;  // most per block and per SM
struct TileAmps {
    float v[kTileMaxSteps];  // amp_t of each step
};
struct TilePlan {
    int steps = 1;  // 1: single-step launches are faster
    int rx = 0, ry = 0, warps = 0;
    int per_sm = 0;  // blocks per SM if that makes one wave (else 0: as many as fit)
    int64_t launches = 0;  // for the n steps planned: `launches` passes of at most `steps`
    double us = 0.0;       // modelled time of the n steps
};
// The fastest array for a launch of s steps, found when it is first asked for. It depends on the
// lattice only, so a handle searches once per s, whatever step counts it is called with. us: the
// modelled time of that launch or, with steps = 1, a time that no array undercuts.
struct TileTable {
    TilePlan best[kTileMaxSteps + 1];
};
inline int64_t tile_bytes(int rx, int ry, int elem, int um) {
    return 9LL * rx * (ry + 3) * elem +
           (um == UM_FIELD ? 8LL * rx * (ry + 1) : um == UM_ANALYTIC ? 4LL * (ry + 1) : 0);
}
// Plan of n steps; steps = 1 unless it takes less than `least` microseconds.
TilePlan tile_plan(TileTable& table, int storage, int um, int basis, int nv, int nx, int ny,
                   int64_t n, double least);
cudaError_t launch_tile(int storage, int um, int basis, int nv, const void* src, void* dst,
                        const StepArgs& a, const TileAmps& amps, const TilePlan& p,
                        cudaStream_t st);
cudaError_t launch_tile16(int storage, int um, int basis, int nv, const void* src, void* dst,
                          const StepArgs& a, const TileAmps& amps, const TilePlan& p,
                          cudaStream_t st);

// The same step (nv >= 2) with the FP64 conserved sums of dst fused in, written to out[4]
// as launch_conserved does; partials: step_sum_scratch(nx, ny, nv) doubles of scratch; ticket: a
// device word that is 0 between calls. step_fuses_sums: whether that beats the step followed by
// launch_conserved.
bool step_fuses_sums(int nx, int ny, int nv);
int64_t step_sum_scratch(int nx, int ny, int nv);
cudaError_t launch_step_conserved(int storage, int um, int nv, const void* src, void* dst,
                                  const StepArgs& a, cudaStream_t st, int basis, double rho_ref,
                                  double jx_ref, double jy_ref, double lambda,
                                  double* partials, unsigned* ticket, double* out);

// Initial fields: density (or null: 1) and velocity components, n floats each.
struct Fields {
    const float* rho = nullptr;
    const float* u[3] = {nullptr, nullptr, nullptr};
};

cudaError_t launch_init_eq(int storage, void* dst, const Fields& f, int64_t n,
                           const StoreRef& ref, float inv_lambda, cudaStream_t st,
                           int basis = 0);

cudaError_t launch_moments(int storage, const void* src, float* rho, float* u, int64_t n,
                           const StoreRef& ref, float lambda, cudaStream_t st);

int conserved_blocks(int64_t n);

// Sums over nodes 0 .. n-1 of src, whose planes are `plane` >= n elements apart.
// partials: 4 * nblk doubles of scratch; out: 4 doubles (device). rho_ref, jx_ref, jy_ref:
// the stored reference state (jx_ref = rho_ref U_x / lambda).
cudaError_t launch_conserved(int storage, const void* src, int64_t n, int64_t plane,
                             double rho_ref, double jx_ref, double jy_ref, double lambda,
                             double* partials, int nblk, double* out, cudaStream_t st);

// Sums {rho, rho u_x, rho u_y, rho u_z} over nodes 0 .. n-1 of initial fields into out[4]
// (device); partials: 4 * nblk doubles; ticket: a device word that is 0 between calls. FP32
// arithmetic with the rounding errors carried along, for densities and momenta well inside the
// range of FP32; _fp64 for any.
cudaError_t launch_mean_flow(const Fields& f, int64_t n, int dim, double* partials, int nblk,
                             unsigned* ticket, double* out, cudaStream_t st);
cudaError_t launch_mean_flow_fp64(const Fields& f, int64_t n, int dim, double* partials,
                                  int nblk, double* out, cudaStream_t st);

// ---------------------------------------------------------------- D3Q19
int step3_vector_width(int storage, int nx);
cudaError_t launch_step3(int storage, int um, int nv, const void* src, void* dst,
                         const StepArgs3& a, cudaStream_t st);
cudaError_t launch_init_eq3(int storage, void* dst, const Fields& f, int64_t n,
                            const StoreRef3& ref, float inv_lambda, cudaStream_t st);
cudaError_t launch_moments3(int storage, const void* src, float* rho, float* u, int64_t n,
                            const StoreRef3& ref, float lambda, cudaStream_t st);
// The step with the FP64 conserved sums of dst fused in (FP32 with 4-node packs, 16-bit with
// 8-node packs), written to out[5] as launch_conserved3 does; partials: scratch of
// step3_sum_scratch(...) doubles (-1 on a CUDA error).
bool step3_fuses_sums(int storage, int nv, int ny, int nz);
int64_t step3_sum_scratch(int storage, int nv, const StepArgs3& a);
cudaError_t launch_step3_conserved(int storage, int um, int nv, const void* src, void* dst,
                                   const StepArgs3& a, cudaStream_t st, double lambda,
                                   double* partials, int64_t scratch, double* out);
// partials: 8 * nblk doubles; out: 5 doubles (sum rho, sum q (3), non-finite nodes) over
// nodes 0 .. n-1 of src, whose planes are `plane` >= n elements apart.
cudaError_t launch_conserved3(int storage, const void* src, int64_t n, int64_t plane,
                              const StoreRef3& ref, double lambda, double* partials, int nblk,
                              double* out, cudaStream_t st);

// ---------------------------------------------------------------- adjoint (FP32 adjoint
// vectors; forward states in the handle's storage type)
struct AdjointArgs {
    StepArgs step;     // step arguments of the relaxation being reversed (time k)
    float da_factor;   // d(u~/lambda)/dA = cos(2 pi k / P) / lambda for dL/dA
    float* dut0;       // optional [2][n]: accumulates amp_t * dL/d(u~/lambda) per node
    double* acc;       // per-block FP64 accumulators, 8 per block (6 rates, dL/dA, unused)
    int y0 = 0, y1 = 0;  // rows reversed: [y0, y1) (a slab's own rows; else 0 .. ny)
};

dim3 adjoint_grid(int nx, int ny, int nv);
int64_t adjoint_blocks(int nx, int ny, int nv);

// mu_out = J_C(P s_prev)^T a, a = (gather ? P^T a_in : a_in); accumulates into aa.acc;
// nv nodes per thread (1, 2 or 4, dividing nx unless 1); s_prev in the storage type.
cudaError_t launch_adjoint_step(int storage, int um, int nv, const void* s_prev,
                                const float* a_in, bool gather, float* mu_out,
                                const AdjointArgs& aa, cudaStream_t st);
// The same for FP16 / BF16 forward states (d2q9_adjoint16.cu).
cudaError_t launch_adjoint_step16(int storage, int um, int nv, const void* s_prev,
                                  const float* a_in, bool gather, float* mu_out,
                                  const AdjointArgs& aa, cudaStream_t st);
cudaError_t launch_gather(const float* src, float* dst, int nx, int ny, cudaStream_t st);
cudaError_t launch_acc_final(const double* acc, int64_t nblk, double* out, cudaStream_t st);
cudaError_t launch_equilibrium_vjp(const float* rho, const float* u, const float* a, float* drho,
                                   float* du, int64_t n, float inv_lambda, cudaStream_t st);
cudaError_t launch_moments_vjp(int storage, const void* g, const float* drho, const float* du,
                               float* out, int64_t n, const StoreRef& ref, float lambda,
                               cudaStream_t st);
// partials: 4 * nblk doubles of scratch (slot 0 of each used); out: 1 double (device).
// Over nodes 0 .. n-1 of g (and grad), planes `plane` elements apart.
cudaError_t launch_kinetic_energy(int storage, const void* g, float* grad, int64_t n,
                                  int64_t plane, const StoreRef& ref, float lambda,
                                  double* partials, int nblk, double* out, cudaStream_t st);

}  // namespace lbmrv
