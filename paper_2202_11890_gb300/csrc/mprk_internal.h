// mprk_internal.h — structures shared by the CUDA kernels and the host runtime.
//
// Device layout of one instance (all planes row-major with a padded pitch):
//   qA   [4][nz][pitch] double   the state q_n (S, B rows) and the fast state
//                                at even fast substeps (F rows)
//   qB   [4][nz][pitch] double   the fast state at odd fast substeps (F rows)
//   Ra   [4][nz][pitch] double   (FP64) or float (FP32FLUX): the right-hand
//                                side of the first stage of the current fast
//                                substep (and of stage 1 on S rows)
//   accB [4][nB][pitch] double   running sum of the buffer right-hand sides,
//                                then q_{n+1} on B rows
//   accS [4][nS][pitch] double   q_{n+1} on S rows until the step ends
// FP32-flux mode only:
//   dA, dB [4][nz][pitch] float  deviations q - q_ref of qA, qB (float shadows)
//   rowc [NROWC][nz] float       per-row reference constants (stage_tile_mixed.cuh)
#pragma once

#include <cuda.h>  // CUtensorMap (types only; the encoder is looked up at run time)
#include <cuda_runtime.h>
#include <cstdint>
#include <string>

#include "mprk.h"

namespace mprk {

// Tile of the stage kernels: TX columns by TZ rows.
constexpr int TX = 32;
constexpr int TZ = 8;
constexpr int NTHREADS = TX * TZ;
// Threads of the FP64 tile of TZ rows: nine warps, two face jobs each
// (stage_tile.cuh).
constexpr int FP64_THREADS = NTHREADS + TX;
// The FP32-flux kernel's tile is TX x 2*TZ cells; each thread of its fast
// path carries two cells of one column, rows k and k + TZ.
constexpr int MTZ = 2 * TZ;
// Floats of per-row constants in the FP32-flux mode (layout in stage_tile_mixed.cuh).
constexpr int NROWC = 48;
// Threads of the FP32-flux tile: nine warps. Warps 0-7 own the TX x TZ cell
// pairs, warp 8 computes the faces on the tile's top edge (one pass) and
// right edge (one pass), so every warp makes two face passes.
constexpr int MIXED_THREADS = NTHREADS + 32;

// Status bits written by device code.
constexpr unsigned ST_NONFINITE = 1u;
constexpr unsigned ST_CFL = 2u;
constexpr unsigned ST_TIMEOUT = 4u;

// A factor of a fixed-point product, hi 2^32 + lo with lo signed (fixed_point.cuh).
struct FxW {
  int lo, hi;
};
// A factor in (0, 1) scaled to [1/2, 1): f 2^-62 2^-s.
struct FxN {
  FxW f;
  int s;
};
// Coefficients of the viscous face flux over half the divergence factor.
enum {
  FXC_A,  // (8/3) mu / d_n: sigma_nn from the normal difference of u_n
  FXC_B,  // -mu / (3 d_t): sigma_nn from the two cells' tangential differences of u_t
  FXC_C,  // 2 mu / d_n: sigma_nt from the normal difference of u_t
  FXC_D,  // mu / (2 d_t): sigma_nt from the two cells' tangential differences of u_n
  FXC_K,  // 2 kappa gamma (gamma - 1) / d_n: heat flux from the difference of e
  FXC_N
};

// Interface: the wall velocity u_w = u_1 + LID_1 (u_2 - u_1) = u_2 - LID_2
// (u_2 - u_1), so that the ghost 2 u_w - u of either fluid is u + 2 LID_f
// (other fluid's u - u).
enum {
  LID_S,  // 2 b_u: twice the shear stress from u_2 - u_1
  LID_1,  // b_u dz1 / (2 mu1)
  LID_2,  // b_u dz2 / (2 mu2) = 1 - LID_1
  LID_T,  // 2 b_T gamma (gamma - 1): twice -Pi_z from e_2 - e_1
  LID_N
};

// Fixed-point constants of the FP64 tile's face fluxes (fixed_point.cuh).
struct FxConst {
  int on;              // every factor below fits its scale: the fluxes run in fixed point
  int square;          // dx = dz1 = dz2: x and z differences add before the scaling
  double scale;        // their factor: 2^-57 of half of 1/dx
  double scale_z[2];   // 2^-57 of half of 1/dz per fluid
  FxW gm1;             // (gamma - 1).61
  FxW gg;              // gamma (gamma - 1).62
  FxW lid[LID_N];      // interface, .62
  FxW fc[2][2][FXC_N]; // viscous coefficients per direction (x, z) and fluid, .62
  double fd[2][2][FXC_N];  // the same in double, of the double pass
  FxN tc[2][2][2];     // of them C and D for the tangential stress
  FxN ts;              // LID_S likewise
  double tlid[LID_N];  // the interface's factors in double, LID_1 and LID_2 doubled
};

// The same of the 3-D tiles: directions x (tangents y, z), y (x, z) and z
// (x, y), the coefficients in fixed point and in double.
enum {
  F3_A,   // (8/3) mu / d_n: sigma_nn from the normal difference of u_n
  F3_B1,  // -mu / (3 d_t1): sigma_nn from the differences of u_t1 along t1
  F3_B2,  // -mu / (3 d_t2): of u_t2 along t2
  F3_C,   // 2 mu / d_n: sigma_nt from the normal difference of u_t
  F3_D1,  // mu / (2 d_t1): sigma_nt1 from the differences of u_n along t1
  F3_D2,  // mu / (2 d_t2)
  F3_K,   // 2 kappa gamma (gamma - 1) / d_n: heat flux from the difference of e
  F3_N
};
struct Fx3Const {
  FxConst k;  // its fc, fd and tc unused; square: dx = dy = dz1 = dz2
  FxW fc[3][2][F3_N];
  double fd[3][2][F3_N];
  FxN tc[3][2][3];  // C, D1, D2 for the tangential stresses
  double scale_y;  // 2^-57 of half of 1/dy
};

// Physics and grid of one instance, constant over its life.
struct Geom {
  int nx, pitch, nz;
  int n1;          // rows of fluid 1 (S and B): the interface lies below row n1
  int nS_r, n1_r;  // region bounds used by the stage combination: rows < nS_r are
                   // S, rows < n1_r are B, the rest F (single rate: 0 and 0)
  int nS_g;        // rows of the slow band of the grid (Courant numbers per band)
  int m;           // fast substeps per slow step
  int wall;        // 0 no-slip, 1 slip
  int xwall;       // 0 periodic x, 1 walls (of kind `wall`) at both x ends
  double dt;
  double inv_dx, inv_dz1, inv_dz2;
  double gamma, gm1;
  double mu1, mu2, kap1, kap2;
  double G;
  double bu, bT;       // interface bulk coefficients (App. B)
  double cu1, cT1;     // dz1/(2 mu1), dz1/(2 kappa1): wall states from fluid 1
  double cu2, cT2;     // dz2/(2 mu2), dz2/(2 kappa2): wall states from fluid 2
  int ny;              // columns in y: 1 in 2-D
  int nc;              // conserved components: 4 (2-D) or 5 (3-D)
  double inv_dy;       // 3-D only
  // base method of the MPRK framework (Sec. 3 remark): s stages, A, b.
  // gen = 0 for Heun (Table 1), which runs the dedicated RK2 low-storage
  // path; otherwise the general s-stage path with s R_a slots.
  int s, gen;
  double bA[4][4], bb[4];
  double hF;           // dt / m
  double h2;           // dt / (2 m)
  double hdt;          // dt / 2
  // the same constants rounded to float once on the host, so that float
  // kernels never convert (conversions run at the FP64 rate on this GPU)
  float gammaf, gm1f, mu1f, mu2f, kap1f, kap2f, Gf;
  float inv_dxf, inv_dz1f, inv_dz2f;
  float dtf, hFf, h2f;
};


// Buffers of one instance.
struct Bufs {
  double* qA;
  double* qB;
  void* Ra;
  double* accB;
  double* accS;
  float* dA;    // FP32-flux mode only (else null)
  float* dB;
  float* rowc;
};

// One launch of the stage kernel over rows [row0, nz) of one instance.
struct StageArgs {
  Geom g;
  Bufs b;
  const double* qF;   // base state of F rows this substep (qA or qB)
  double* qF_next;    // F rows of the next substep (the other one)
  const float* dF;    // FP32-flux mode: shadows matching qF and qF_next
  float* dF_next;
  int stage;          // 0-based stage index i in [0, 2m)
  int row0;           // first row of the launch (0 at stages 0, 1; nS_r later)
  int tiles_x;        // tiles across x
  int tz;             // tile rows: TZ (FP64) or MTZ (FP32-flux)
  int rhs_only;       // test hook: write R to rhs_out instead of combining
  double* rhs_out;    // [4][nz][pitch] when rhs_only
  int rhs_hi;         // last row (exclusive) when rhs_only
  const double* rhs_in;  // full stage state when rhs_only
  double* gy;         // 3-D: y-face fluxes [5][nz][ny][pitch] (face j+1/2 at j)
  int bulk;           // FP32-flux: interior tiles stage their float planes by
                      // tensor copies (set by launch_stage when maps exist)
  unsigned* status;   // status word for device-side errors, or null
  FxConst fx;         // FP64, 2-D
};

// The viscous coefficient j of direction dir (0 x, 1 z) in fluid fl (0, 1),
// over half the divergence factor 1/d_n of the direction.
__host__ __device__ inline double visc_coef(const Geom& g, int dir, int fl, int j) {
  const double iz = fl ? g.inv_dz2 : g.inv_dz1, mu = fl ? g.mu2 : g.mu1;
  const double in = dir ? iz : g.inv_dx, it = dir ? g.inv_dx : iz;
  switch (j) {
    case FXC_A: return 8.0 / 3.0 * mu * in;
    case FXC_B: return -mu * it / 3.0;
    case FXC_C: return 2.0 * mu * in;
    case FXC_D: return 0.5 * mu * it;
    default: return 2.0 * (fl ? g.kap2 : g.kap1) * g.gamma * g.gm1 * in;
  }
}
__host__ __device__ inline double lid_coef(const Geom& g, int j) {
  switch (j) {
    case LID_S: return 2.0 * g.bu;
    case LID_1: return g.bu * g.cu1;
    case LID_2: return g.bu * g.cu2;
    default: return 2.0 * g.bT * g.gamma * g.gm1;
  }
}
// Fills the fixed-point constants of a geometry (mprk_runtime.cu).
void fixed_point_const(const Geom& g, FxConst* out);
void fixed_point_const3(const Geom& g, Fx3Const* out);

// Arguments of stage st of one slow step: F rows ping-pong between the A and
// B buffers at every fast substep.
inline StageArgs stage_args(const Geom& g, const Bufs& b, int st) {
  StageArgs a{};
  a.g = g;
  a.b = b;
  const bool even_sub = ((st / g.s) % 2) == 0;
  a.qF = even_sub ? b.qA : b.qB;
  a.qF_next = even_sub ? b.qB : b.qA;
  a.dF = even_sub ? b.dA : b.dB;
  a.dF_next = even_sub ? b.dB : b.dA;
  a.stage = st;
  a.row0 = st < g.s ? 0 : g.nS_r;  // S rows only during the first substep
  a.tiles_x = (g.nx + TX - 1) / TX;
  a.tz = b.dA ? MTZ : TZ;  // float shadows exist only in the FP32-flux mode
  if (!b.dA && g.ny == 1) fixed_point_const(g, &a.fx);
  return a;
}
__host__ __device__ inline int stage_tiles(const StageArgs& a) {
  const int hi = a.rhs_only ? a.rhs_hi : a.g.nz;
  return a.tiles_x * ((hi - a.row0 + a.tz - 1) / a.tz);
}

// FP32-flux tiles: the TX x MTZ tile from row k0, column i0 takes the pair path
// (stage_tile_mixed.cuh). An interior tile needs none of the ghost rules: rows k0-2 .. k0+MTZ+1 lie
// inside the grid and inside one fluid, and with x walls its halo columns
// i0-2 .. i0+TX+1 lie between them. For a stage (not the right-hand-side
// hook) they also lie on one side of the F-row bound.
__host__ __device__ inline bool pair_interior(const StageArgs& a, int k0, int i0) {
  const Geom& g = a.g;
  const int hi = a.rhs_only ? a.rhs_hi : g.nz;
  const int lo_h = k0 - 2, hi_h = k0 + MTZ + 2;  // halo rows [lo_h, hi_h)
  if (lo_h < 0 || hi_h > g.nz || k0 + MTZ > hi || !(g.n1 <= lo_h || g.n1 >= hi_h)) return false;
  if (g.xwall && (i0 < 2 || i0 + TX + 2 > g.nx)) return false;  // halo columns inside the walls
  if (a.rhs_only) return true;
  // S and B rows may share a tile (the combination picks per cell, and both
  // take their stage values from q_n with dt); the F rows' state and step
  // differ, so no F row lies within the halo of a tile with S or B rows
  return g.n1_r <= lo_h || g.n1_r >= hi_h;
}

// Tensor maps of the FP32-flux float planes ([4][nz][pitch] float each) for
// the bulk tensor copies of the stage kernel (mprk_kernels.cu).
struct StageMaps {
  CUtensorMap dA, dB, Ra;
  bool valid;
};
// Encodes the maps of b's float planes. Sets valid = false (and returns
// cudaSuccess) where the planes cannot be tensor-copied (pitch not a
// multiple of 4 floats, or no encoder in the driver); tiles then load
// directly.
cudaError_t make_stage_maps(const Geom& g, const Bufs& b, StageMaps* out);

// Shape of the FP64 stage tile: rows per tile (TZ, TZ/2 or TZ/4, with TX
// columns) and tpc: 1 for two face jobs per warp (rows + 1 warps), 2 for one (2
// rows + 3; the tables' "threads per cell"). Every shape computes the same
// arithmetic in the same order, so results do not depend on it.
struct TileShape {
  int rows, tpc;
};
inline bool tile_shape_valid(const TileShape& t) {
  return (t.rows == TZ || t.rows == TZ / 2 || t.rows == TZ / 4) && (t.tpc == 1 || t.tpc == 2);
}
// The tuned shape of single-instance FP64 stage launches of `cells` cells,
// when the tuning table has one for their size bucket (mprk_batch.cu).
bool tuned_tile_shape(long long cells, TileShape* out);
// The shape launch_stage takes without a tuned one: the shortest tile whose
// launch fits in one wave (n tiles <= SMs), with a warp per face job; a
// launch that does not fit even with TZ rows keeps them, two jobs per warp.
TileShape default_tile_shape(const StageArgs& a);

// Launchers (mprk_kernels.cu). All enqueue on `stream` and return the launch error.
// chained: the launch before it on the stream is one of the same slow step
// (or of the step before), so the two may overlap at their ends: the kernel
// is launched as soon as every CTA of the one before allows it (chain_next), and
// its CTAs wait for that one's completion before they touch memory (chain_wait).
// FP32-flux launches are chained only within one wave (launch_stage): longer
// ones ran 3 to 7 % slower (4096 x 2048: 5.04 -> 5.24 ms for two steps).
// maps (FP32-flux only, may be null) enables the staged tiles. shape (FP64
// only, may be null) overrides the tuned and the default tile shape.
cudaError_t launch_stage(const StageArgs& a, int precision, int n_tiles, cudaStream_t stream,
                         const StageMaps* maps = nullptr, const TileShape* shape = nullptr, bool chained = false);
cudaError_t launch_finalize(const Geom& g, const Bufs& b, int m_odd, cudaStream_t stream, bool chained = false);
// 3-D (g.ny > 1): the y-face launch and the stage launch of one stage; a.gy
// must point at a state-sized buffer.
cudaError_t launch_stage3(const StageArgs& a, cudaStream_t stream, bool chained = false);
// FP32-flux mode: per-row reference of q (row means, refd [4][nz] scratch)
// and the float shadow dA = q - q_ref of qA.
cudaError_t launch_reference(const Geom& g, const double* q, double* refd, float* rowc,
                             cudaStream_t stream);
// `rows` rows of `width` doubles from src (row stride spitch) to dst (row
// stride dpitch; null: not copied), and where rowc is given the float shadow
// of row r = c nz + k into `shadow` (row stride dpitch).
cudaError_t launch_copy_state(double* dst, size_t dpitch, const double* src, size_t spitch, int width, long long rows,
                              int nz, const float* rowc, float* shadow, cudaStream_t stream);
cudaError_t launch_shadow(const Geom& g, const double* q, const float* rowc, float* d,
                          cudaStream_t stream);
cudaError_t launch_diag(const Geom& g, const double* q, double* partials, int nblocks,
                        double* out, unsigned* status, double cfl_limit, cudaStream_t stream);
int diag_blocks(const Geom& g);
cudaError_t launch_convert_check(const double* in, int n, float* nar, float* nar_hw, double* wid,
                                 double* wid_hw, cudaStream_t stream);
cudaError_t prepare_kernels();  // one-time attribute setup (dynamic shared memory)
size_t stage_smem_bytes(int precision);

#ifdef __CUDACC__
// Overlap of consecutive launches (programmatic dependent launch).
// chain_wait waits until the launch before this one has completed and its
// writes are visible; every thread calls it before its first access to the
// step's buffers, so a launch's completion implies that of all before it.
// chain_next lets the next launch's CTAs start, once every CTA of this one has
// called it. Without a chained launch both are no-ops. A slow step of 64 x 64
// cells, launched on a stream, 105.6 -> 94.3 us (nine launches); as a graph
// 85.7 -> 84.6 us. chain_next stands behind the faces: called as the kernel
// starts, the next launch's CTAs fill the SMs that have room first, two or
// three on some while others stay empty (321 x 273 cells, m = 4, 166 against
// 131 us per step; 128 x 128 61.5 against 57.2). The 3-D ones, whose launches
// are many waves long, call it first (the same within 0.5 %).
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// One launch, chained to the one before it on the stream or not.
template <typename... P, typename... A>
cudaError_t launch_kernel(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool chained,
                          const A&... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&c, k, args...);
}
#endif

// Fills g from a configuration; pitch is the row pitch of the buffers
// (mprk_runtime.cu).
void geom_from_config(const mprk_config& c, int pitch, Geom* g);

// Sets the calling thread's message for mprk_last_error (mprk_runtime.cu).
void set_last_error(const std::string& msg);

}  // namespace mprk

struct mprk_instance;

namespace mprk {
// Instance internals the batch path uses (mprk_runtime.cu).
int instance_view(const mprk_instance* inst, Geom* g, Bufs* b, int* precision, cudaStream_t* stream,
                  unsigned** status);
cudaStream_t instance_stream(const mprk_instance* inst);
void instance_count_steps(mprk_instance* inst, int n);
// One slow step of an instance by its own stage launches on stream s (the
// kernels mprk_step's graph replays), counted in its steps; cell_stages gets
// the step's cell-stages (mprk_runtime.cu).
int instance_step_alone(mprk_instance* inst, cudaStream_t s, long long* cell_stages);
// Cells of an instance (nx ny nz).
long long instance_cells(const mprk_instance* inst);
// Drops cached batch plans that mention inst (mprk_batch.cu).
void batch_forget(const void* inst);
// One batched launch per slow step on an explicit stream (mprk_batch.cu).
int batch_step_on(mprk_instance* const* insts, int count, int n, cudaStream_t stream, long long* cell_stages);
// A persistent batch launcher for a resident set that changes between slow
// steps (mprk_batch.cu); one launch per call, no graph.
struct BatchRunner;
BatchRunner* runner_create(int precision, cudaStream_t stream);
void runner_destroy(BatchRunner* r);
int runner_step(BatchRunner* r, mprk_instance* const* insts, int count, long long* cell_stages);
// Forget the cached work list (the resident set changed; an address may be reused).
void runner_invalidate(BatchRunner* r);
// Device bytes mprk_create allocates for a configuration (mprk_runtime.cu).
long long instance_bytes(const mprk_config& c);
// Configuration check of mprk_create (sets the error message).
int validate_config(const mprk_config* c);
// mprk_create with an option: stream_ordered instances allocate with
// cudaMallocAsync on cuda_stream, free with cudaFreeAsync, capture no graph
// and advance only through batches (the server's instances).
int create_instance(const mprk_config* cfg, const double* q0, int q0_location, void* cuda_stream,
                    bool stream_ordered, mprk_instance** out);
long long instance_steps(const mprk_instance* inst);
long long instance_device_bytes(const mprk_instance* inst);
void destroy_instance(mprk_instance* inst);

}  // namespace mprk
