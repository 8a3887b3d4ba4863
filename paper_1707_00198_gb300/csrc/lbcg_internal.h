// Internal interface between the host runtime (lbcg_host.cu) and the kernel launchers
// (lbcg_kernels.cu, lbcg_obs.cu).  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lbcg_device.cuh"
#include "lbcg_plan.h"

namespace lbcg {

// Everything one launch of the step kernels needs (device pointers).
struct LaunchStep {
  const LatDev* lats;
  const WallGroup* groups;   // wall kernel work units
  int ngroups;
  const int* wband;          // band nodes of the groups (population offset in their lattice)
  const WallSten* wvirt;     // virtual (outermost solid) nodes of the groups
  const WallSten* wsten;     // per outermost fluid node: its 8 neighbours' local indices
  const OfbEntry* ofb;       // outermost fluid list
  const int4* tiles;      // tile list (lattice, x0, y0, -)
  int ntiles;
  int ty;                 // tile height (tiles are 32 wide)
  const void* src;
  void* dst;
  const uint8_t* flags;
  const uint8_t* nbmask;  // per node: bit a-1 set if the neighbour in direction a is solid
  void* wall;
  long long node_total;
  const int4* strips;     // sweep schedule: (lattice, x0, y_begin, y_end)
  int nstrips;
  int sweep;              // 1: k_sweep over strips, 0: k_step over tiles
  int scheme_b;           // 1: some lattice of the batch uses wetting scheme (b)
  double* macro;          // non-null: write macroscopic fields instead of stepping (tiles)
  cudaEvent_t* ev;        // non-null: 4 events recorded around k_wall and the step kernel
  int* err;               // device error word: a sweep block's bounded wait ran out
  int poll_limit;         // polls before a sweep block's wait for a staged row gives up
  const uint32_t* sr_epoch;   // 16-bit storage: stochastic-rounding replay counter (device)
  uint32_t sr_step;           // and the step within the replay / the absolute step
};

cudaError_t launch_step(int prec, const LaunchStep& p, cudaStream_t st);
// the number of kernels launch_step launches for p (the wall kernel, the bulk kernel)
inline int step_kernels(const LaunchStep& p) {
  return (p.ngroups > 0 ? 1 : 0) + ((p.sweep && p.macro == nullptr) ? (p.nstrips > 0 ? 1 : 0) : (p.ntiles > 0 ? 1 : 0));
}
// Advances the stochastic-rounding replay counter (one single-thread launch).
cudaError_t launch_sr_tick(uint32_t* epoch, cudaStream_t st);
// One-time kernel attributes for a precision (the sweep's dynamic shared memory); called
// before any launch or graph capture of that precision.
cudaError_t prepare_kernels(int prec);

// Lets a kernel's launches take all the dynamic shared memory a block can have on the device.
template <typename K>
inline cudaError_t allow_max_smem(K* k) {
  int dev = 0, most = 0;
  cudaFuncAttributes a{};
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, most - int(a.sharedSizeBytes));
  return e;
}

// ---- the resident step kernel (lbcg_run.cu)
constexpr int kRunFlagStride = 32;   // unsigned ints between the tiles' progress words (128 bytes)
constexpr int kReplaySteps = 32;     // steps of one graph replay of the launch-per-step schedule
// Steps 0 .. nsteps - 1 of one launch: step s reads state(s) and writes state(s + 1).
struct RunArgs {
  const LatDev* lats;
  const RunTile* tiles;
  const int *nb, *extra, *w_ofb;
  const uint16_t* band;
  const WallSten *w_sten, *v_sten;
  const uint32_t* copies;
  const RunVirtN* vn;
  const OfbEntry* ofb;
  const uint8_t* flags;
  const uint8_t* nbmask;
  char *pool0, *pool1;    // the states: pool0 and pool1 in turn (stride 0),
  long long stride;       // or one after another from pool0, `stride` bytes apart
  int nsteps;
  unsigned* progress;     // per tile: base + the steps it has finished
  unsigned base;
  int* err;
  int poll_limit;
  // Stochastic rounding draws the keys of the launch-per-step schedule: `pre` direct steps,
  // nrep graph replays of kReplaySteps steps, then direct steps (absolute step numbers from
  // step0).  The launcher advances the replay counter by nrep afterwards.
  const uint32_t* sr_epoch;
  uint32_t step0;
  int pre, nrep;
  __device__ __forceinline__ char* state(int s) const {
    if (stride) return pool0 + s * stride;
    return (s & 1) ? pool1 : pool0;
  }
  __device__ __forceinline__ uint32_t key(uint32_t epoch, int s, long long pop_off) const {
    const int q = s - pre;
    if (q >= 0 && q < nrep * kReplaySteps)
      return sr_key(epoch + 1u + uint32_t(q / kReplaySteps), uint32_t(q % kReplaySteps), pop_off);
    return sr_key(q < 0 ? epoch : epoch + uint32_t(nrep), step0 + uint32_t(s), pop_off);
  }
};
cudaError_t launch_run(int prec, const RunArgs& a, int ntiles, int threads, size_t smem, cudaStream_t st);
// sets the kernel's shared memory and asks how many of its blocks an SM holds
cudaError_t prepare_run(int prec, int threads, size_t smem, int* per_sm);
cudaError_t launch_sr_add(uint32_t* epoch, uint32_t n, cudaStream_t st);

cudaError_t launch_to_storage(int prec, const LatDev* lats, int lat, long long nn, const double* in,
                              const uint8_t* flags, void* pool, cudaStream_t st);
cudaError_t launch_from_storage(int prec, const LatDev* lats, int lat, long long nn, const void* pool,
                                const uint8_t* flags, double* out, cudaStream_t st);

// Observable reductions over one lattice's macroscopic fields (lbcg_obs.cu).
// `partials` must hold obs_partials_doubles(nx*ny) doubles; `out` receives kObsOut doubles.
constexpr int kObsQ = 17;     // reduced quantities
constexpr int kObsRows = 3;   // row-crossing results
constexpr int kObsOut = kObsQ + kObsRows;
constexpr int kObsBlocks = 304;  // 2 x 152 SMs
size_t obs_partials_doubles();
// Steady-state diagnostics (lbcg_obs.cu): 6 doubles into `out` -- max |du_x|, max |du_y|
// against usnap ([2][node_total], overwritten with the current velocity), rho_R inside / outside
// the circle, rho_B inside / outside.  `partials` holds kObsBlocks * 6 doubles.
cudaError_t launch_diagnostics(const LatDev* lats, int lat, const double* macro, long long node_total,
                               const uint8_t* flags, double* usnap, bool have_snap, double cx, double cy, double r,
                               double* partials, double* out, cudaStream_t st);
cudaError_t launch_observables(const LatDev* lats, int lat, int nx, int ny, const double* macro,
                               long long node_total, const uint8_t* flags, int tip0, int tip1, int cl0, int cl1,
                               double* partials, double* out, cudaStream_t st);

// Device pointers of one reverse step of the adjoint (lbcg_adjoint.cu); node arrays are
// compact [ny][nx], FP64.
template <typename R>
struct AdjDevT {
  LatDev L;
  LatConst<R> C;
  int N;
  int M;   // elements per plane of the arrays only a node's own threads use (fr, fb, rr, rb, gr*,
           // gc*, dn, pick, lf_*, ln_*, lg_*, lrn): N, or a block's nodes in its shared memory
  const void* src;       // stored state (population pool of the lattice), FP64 or FP32
  int src_fp32;          // 1: the state is stored in FP32 (an FP32 forward)
  // |grad rho^N| at or below which the reverse sweep takes n = g/|g| as constant.  FP64
  // states: the forward's own guard.  FP32 states: 1e-5 -- their pure phases carry rounding
  // noise |grad rho^N| ~ 1e-7 whose normals the forward only ever multiplies by ~0, but whose
  // 1/|g| ~ 1e8 would give the linearised map a spurious growing mode.
  double n_eps;
  const uint8_t* flags;  // node flags (pitch layout)
  const uint8_t* sol;    // compact [ny][nx]: 1 on solid nodes
  const uint8_t* nbm;    // compact [ny][nx], every node: bit a-1 set if its neighbour in
                         // direction a (periodic wrap, else clamp) is solid
  const R* nsx;     // solid normal at outermost fluid nodes (compact, 0 elsewhere)
  const R* nsy;
  const R* cos_t;   // cos and sin of the contact angle per node (compact)
  const R* sin_t;
  // forward intermediates (compact)
  R *fr, *fb;       // [9][N] post-streaming populations after the Zou-He columns
  R *rr, *rb, *rn;  // colour densities, rho^N (fluid nodes; 0 on solid nodes)
  R *grx, *gry;     // raw gradient (Eq. 28)
  R *gcx, *gcy;     // corrected gradient (Eq. 31; = raw off Omega_Fb)
  R *nxv, *nyv;     // n on fluid nodes (0 on solid nodes)
  R *dn;            // [4][N] d_x n_x, d_y n_x, d_x n_y, d_y n_y
  int *pick;             // 1 or 2: the candidate Eq. 36 chose (0 off Omega_Fb / below guard)
  // adjoints
  const R* lam_next;  // [18][N] adjoint of the stored state after the step: (fr, fb) pairs
  R* lam;             // [18][N] adjoint of the stored state before the step
  R *lf_r, *lf_b;     // [9][N] adjoint of the post-Zou-He populations
  R *ln_x, *ln_y;     // adjoint of n (local part)
  R *lnt_x, *lnt_y;   // adjoint of n through the neighbours' grad n (scatter target)
  R *lg_x, *lg_y;     // adjoint of the corrected gradient (force path)
  R *lrn, *lrnt;      // adjoint of rho^N: local part, and through the neighbours' gradient
  double *p_sigma, *p_hR, *p_hB, *p_theta;  // per-node parameter adjoints (accumulated)
};

// R: the arithmetic of the reverse kernels (double, or float for the FP32 reverse sweep);
// the per-node parameter adjoints accumulate in double either way.
// adjoint_forward: the forward intermediates of state A.src into A's intermediate arrays.
// adjoint_step: the reverse of the step from A.src (lam <- J^T lam_next), using A's
// intermediates; with B non-null it also computes B's (the state before A's), which must use
// other intermediate and scatter-target arrays than A (the reverse arrays may be shared).
template <typename R>
cudaError_t adjoint_forward(const AdjDevT<R>& A, cudaStream_t st);
template <typename R>
cudaError_t adjoint_step(const AdjDevT<R>& A, const AdjDevT<R>* B, cudaStream_t st);
// A segment's reverse sweep as one cooperative launch (k_reverse): the states at `states`,
// `stride` bytes apart, reversed from state ns - 1 to state 0; lam_next and lam take turns, so
// that the result is in lam_next's array if ns is even, in lam's if it is odd.  Tiles and
// neighbours of the resident step kernel's plan; progress words of its own, 3 ns + 1 phases from
// base on.  `threads`: twice the nodes of the largest tile, rounded up to whole warps each.
constexpr int kRevMaxThreads = 256;
constexpr int kRevMaxSlots = 512;   // nodes of a tile plus two all round, at most
template <typename R>
struct RevRunT {
  AdjDevT<R> V[2];
  const RunTile* tiles;
  const int* nb;
  unsigned* progress;
  unsigned base;
  int* err;
  int poll_limit;
  const char* states;
  long long stride;
  int ns;
  const R* lam_next;
  R* lam;
};
template <typename R>
cudaError_t launch_reverse(const RevRunT<R>& P, int ntiles, int threads, cudaStream_t st);
template <typename R>
cudaError_t reverse_blocks(int threads, int* per_sm);
// seed lam = dJ/d(state): J = sum weight * rho^N (red_mass false) or the red mass (true)
template <typename R>
cudaError_t adjoint_seed(const AdjDevT<R>& A, const R* weight, bool red_mass, cudaStream_t st);

// Sets the calling thread's message returned by lbcg_last_error() (lbcg_host.cu).
void set_last_error(const char* msg);

}  // namespace lbcg
