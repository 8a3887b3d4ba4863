// Host runtime behind the C ABI of include/lbcg.h: validation, node classification
// (Sec. II.C), solid normals (Eq. 32-33), work lists, device memory, graph-captured stepping,
// observables and state transfer.  All arithmetic of the time step runs in the kernels of
// lbcg_kernels.cu; the host only prepares geometry once per handle.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "../../include/lbcg.h"
#include "lbcg_internal.h"

using namespace lbcg;

namespace {

thread_local std::string g_err;

// NVTX range over one public call (shown by Nsight tools; inert without a profiler)
struct Range {
  explicit Range(const char* name) { nvtxRangePushA(name); }
  ~Range() { nvtxRangePop(); }
};

lbcg_status fail(lbcg_status s, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_err = buf;
  return s;
}

// device allocator of new handles (lbcg_set_allocator); null callbacks = cudaMalloc / cudaFree
std::mutex g_alloc_mutex;
lbcg_allocator g_allocator = {nullptr, nullptr, nullptr};

constexpr int kGraphSteps = kReplaySteps;   // steps per captured graph (even: the graph starts and ends on pool A)
constexpr int kGraphBranches = 3; // parallel branches of a batch's graph (groups of lattices)
constexpr int kHostGroups = 8;    // lattice groups whose copies lbcg_step_host overlaps
constexpr int kDefaultTY = 8;
constexpr int kPollLimit = 1 << 22;   // default polls of a bounded device wait (about a second)
constexpr int kRunMaxSteps = 8192;    // steps per launch of the resident kernel, at most,
constexpr int kRunMinSteps = 8;       // and of a call that it takes, at least
constexpr int kSMs = 152;

size_t elem_size(int prec) { return prec == 0 ? 8 : (prec == 1 ? 4 : 2); }
size_t compute_size(int prec) { return prec == 0 ? 8 : 4; }

struct LatHost {
  int nx, ny, pitch, bcx, bcy;
  long long pop_off, plane, node_off;
  lbcg_params prm;
  int tile_begin, tile_end;
  long long n_fluid;
  std::vector<uint8_t> solid;   // [ny*nx]
};

}  // namespace

struct lbcg_handle {
  int prec = 1;
  lbcg_allocator allocator = {nullptr, nullptr, nullptr};   // the allocator at create
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  bool dead = false;
  int64_t step = 0;
  int ty = kDefaultTY;
  std::vector<LatHost> lats;
  long long node_total = 0;
  void* pool[2] = {nullptr, nullptr};
  int cur = 0;
  uint8_t* d_flags = nullptr;
  uint8_t* d_nbmask = nullptr;
  int scheme_b = 0;        // some lattice uses wetting scheme (b)
  int* d_err = nullptr;    // device error word (a bounded wait of a step or reverse kernel ran out)
  int poll_limit = kPollLimit;   // polls of a sweep block's wait for a staged row (about a second)
  int run_polls = kPollLimit;    // and of a resident kernel's wait for the tiles around one
  uint32_t* d_sr_epoch = nullptr;     // 16-bit storage: graph replays so far (stochastic-rounding keys)
  double* d_usnap = nullptr;          // velocity stored by lbcg_diagnostics ([2][node_total])
  std::vector<int64_t> snap_step;     // per lattice: step of that velocity, -1 = none
  void* d_wall = nullptr;
  double* d_macro = nullptr;
  LatDev* d_lats = nullptr;
  int4* d_tiles = nullptr;
  int ntiles = 0;
  int sweep = 1;          // schedule of the step kernel: 1 = y-sweep over strips, 0 = tiles
  int sweep_rows = 0;     // rows per strip segment, 0 = automatic
  int4* d_strips = nullptr;
  int nstrips = 0;
  WallGroup* d_groups = nullptr;   // wall kernel work units and their tables
  int ngroups = 0;
  int* d_wband = nullptr;
  WallSten* d_wvirt = nullptr;
  WallSten* d_wsten = nullptr;
  OfbEntry* d_ofb = nullptr;
  int nofb = 0;
  double* d_obs = nullptr;   // partials then outputs
  // pinned host memory of small results: the device error word, then up to kObsOut doubles
  struct Small {
    int err;
    double v[kObsOut];
  };
  Small* h_small = nullptr;
  // the resident kernel of the tile schedule (see runs_resident): its plan on the device, or
  // run_tiles = 0 where the lattices do not fit
  bool run_planned = false;
  int run_tiles = 0;
  size_t run_smem = 0;
  int run_threads = 0;
  int run_nodes = 0, run_slots = 0;   // nodes of the largest tile, alone and with two all round
  char* d_run = nullptr;          // the plan's lists, one after another
  unsigned* d_progress = nullptr; // per tile: steps finished, counted from run_base
  unsigned run_base = 0;
  RunArgs run = {};               // the device pointers of a launch
  cudaGraphExec_t graph = nullptr;
  int64_t graph_kernels = 0;    // kernel nodes of the captured graph
  int64_t step_launches = 0;    // kernel launches lbcg_step has enqueued (graph nodes counted)
  // Strips, tiles and wall groups are listed in lattice order: lattice l has strips
  // [lat_strip[l], lat_strip[l+1]), and likewise tiles and groups (empty vectors: not in order,
  // and the lattices are then never launched apart).
  std::vector<int> group_lat;   // lattice of each wall group
  std::vector<int> lat_strip, lat_tile, lat_group;
  // batches: the captured graph runs nbranch groups of consecutive lattices (about equal node
  // counts; branch b has lattices [br_lat[b], br_lat[b+1])) as parallel branches, so that one
  // group's wall kernel and launch tail run beside the others' bulk kernels (the lattices are
  // independent); branches 1.. are captured from their own streams, forked from and joined
  // back to the handle's stream.
  int nbranch = 1;
  int br_lat[kGraphBranches + 1] = {};
  // lbcg_step_host: the streams of the uploads and of the downloads, and its events
  cudaStream_t io_stream[2] = {};
  std::vector<cudaEvent_t> io_events;
  cudaStream_t br_stream[kGraphBranches] = {};
  cudaEvent_t ev_fork = nullptr, ev_join[kGraphBranches] = {};
  std::vector<uint8_t> flags_host;
  std::vector<OfbEntry> ofb_host;
  bool profiling = false;
  std::vector<cudaEvent_t> events;   // 4 per profiled launch pair (wall kernel, step kernel)
  size_t events_used = 0;
  int64_t prof_steps = 0;            // steps profiled since the last lbcg_kernel_times
  cudaEvent_t prof_ref = nullptr;    // timing origin of the profiled launches
  bool prof_ref_set = false;
  bool prof_forked = false;          // the branch streams of a profiled batch await their join
};

namespace {

lbcg_status cuda_fail(lbcg_handle* h, cudaError_t e, const char* what) {
  if (h) h->dead = true;
  return fail(LBCG_E_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

#define CK(h, call)                                   \
  do {                                                \
    cudaError_t e_ = (call);                          \
    if (e_ != cudaSuccess) return cuda_fail(h, e_, #call); \
  } while (0)

// Device buffers of a handle: from the allocator the handle was created with, else cudaMalloc.
// A caller's allocator must return memory aligned to 256 bytes (the bulk copies of the sweep
// need 16); a misaligned block is handed back and counts as a failed allocation.
bool dev_alloc(const lbcg_handle* h, void** p, size_t bytes) {
  bytes = std::max<size_t>(bytes, 16);
  *p = nullptr;
  if (h->allocator.alloc) {
    void* q = h->allocator.alloc(bytes, h->stream, h->allocator.ctx);
    if (q && (reinterpret_cast<uintptr_t>(q) & 255u)) {
      h->allocator.release(q, h->stream, h->allocator.ctx);
      q = nullptr;
    }
    *p = q;
  } else if (cudaMalloc(p, bytes) != cudaSuccess) {
    *p = nullptr;
  }
  // a refusal is the caller's to report or to do without: the runtime's last error, which the next
  // launch is checked by, must not keep it
  if (!*p) cudaGetLastError();
  return *p != nullptr;
}
void dev_free(const lbcg_handle* h, void* p) {
  if (!p) return;
  if (h->allocator.alloc) h->allocator.release(p, h->stream, h->allocator.ctx);
  else cudaFree(p);
}

lbcg_status validate(const lbcg_geometry* g, const lbcg_params* p, int idx) {
  if (!g || !p) return fail(LBCG_E_ARG, "lattice %d: NULL geometry or params", idx);
  if (g->nx < 1 || g->ny < 1 || (long long)g->nx * g->ny > 0x7fffffffLL)
    return fail(LBCG_E_ARG, "lattice %d: bad size %d x %d", idx, g->nx, g->ny);
  if (!g->solid || !g->rhoN0) return fail(LBCG_E_ARG, "lattice %d: solid and rhoN0 are required", idx);
  if (g->bc_x < 0 || g->bc_x > 2 || g->bc_y < 0 || g->bc_y > 1)
    return fail(LBCG_E_ARG, "lattice %d: bad boundary codes %d %d", idx, g->bc_x, g->bc_y);
  if (g->bc_x == LBCG_BCX_INOUT && g->nx < 3) return fail(LBCG_E_GEOMETRY, "lattice %d: inlet/outlet needs nx >= 3", idx);
  if (18LL * ((g->nx + 31) / 32 * 32) * g->ny > 0x7fffffffLL)
    return fail(LBCG_E_UNSUPPORTED, "lattice %d: %d x %d exceeds 2^31 stored values (split it into a batch)", idx,
                g->nx, g->ny);
  const int nx = g->nx, ny = g->ny;
  if (g->bc_x == LBCG_BCX_CLOSED)
    for (int y = 0; y < ny; ++y)
      if (!g->solid[(size_t)y * nx] || !g->solid[(size_t)y * nx + nx - 1])
        return fail(LBCG_E_GEOMETRY, "lattice %d: closed x needs solid columns 0 and nx-1", idx);
  if (g->bc_y == LBCG_BCY_CLOSED)
    for (int x = 0; x < nx; ++x)
      if (!g->solid[x] || !g->solid[(size_t)(ny - 1) * nx + x])
        return fail(LBCG_E_GEOMETRY, "lattice %d: closed y needs solid rows 0 and ny-1", idx);
  long long nf = 0;
  for (long long i = 0; i < (long long)nx * ny; ++i) nf += g->solid[i] == 0;
  if (nf == 0) return fail(LBCG_E_GEOMETRY, "lattice %d: no fluid node", idx);
  if (!(p->nu_R > 0) || !(p->nu_B > 0)) return fail(LBCG_E_UNSTABLE_PARAM, "lattice %d: viscosities must be > 0", idx);
  if (!(p->sigma >= 0)) return fail(LBCG_E_UNSTABLE_PARAM, "lattice %d: sigma must be >= 0", idx);
  if (!(p->rho0 > 0)) return fail(LBCG_E_UNSTABLE_PARAM, "lattice %d: rho0 must be > 0", idx);
  if (!(std::fabs(p->u_in) < 1)) return fail(LBCG_E_UNSTABLE_PARAM, "lattice %d: |u_in| must be < 1", idx);
  if (!(p->rho_out > 0)) return fail(LBCG_E_UNSTABLE_PARAM, "lattice %d: rho_out must be > 0", idx);
  if (!(p->grad_eps >= 0)) return fail(LBCG_E_ARG, "lattice %d: grad_eps must be >= 0", idx);
  if (p->inlet_profile != 0 && p->inlet_profile != 1) return fail(LBCG_E_ARG, "lattice %d: bad inlet_profile", idx);
  if (p->wetting < 0 || p->wetting > 2) return fail(LBCG_E_ARG, "lattice %d: bad wetting scheme %d", idx, p->wetting);
  if (p->wetting == 2 && g->theta_node)
    return fail(LBCG_E_UNSUPPORTED, "lattice %d: the surface-energy variant takes one global theta", idx);
  const double pi = 3.14159265358979323846;
  auto angle_ok = [&](double t) { return t > 0 && t < pi; };
  if (!g->theta_node && !angle_ok(p->theta)) return fail(LBCG_E_UNSTABLE_PARAM, "lattice %d: theta outside (0, pi)", idx);
  if (g->theta_node)
    for (long long i = 0; i < (long long)nx * ny; ++i)
      if (!g->solid[i] && !angle_ok(g->theta_node[i]))
        return fail(LBCG_E_UNSTABLE_PARAM, "lattice %d: theta_node outside (0, pi) at %lld", idx, i);
  for (long long i = 0; i < (long long)nx * ny; ++i)
    if (!g->solid[i] && !(g->rhoN0[i] >= -1.0 && g->rhoN0[i] <= 1.0))
      return fail(LBCG_E_ARG, "lattice %d: rhoN0 outside [-1, 1] at %lld", idx, i);
  return LBCG_OK;
}

void build_tiles(lbcg_handle* h, std::vector<int4>& tiles) {
  tiles.clear();
  for (size_t l = 0; l < h->lats.size(); ++l) {
    LatHost& L = h->lats[l];
    L.tile_begin = int(tiles.size());
    for (int y0 = 0; y0 < L.ny; y0 += h->ty)
      for (int x0 = 0; x0 < L.nx; x0 += 32) {
        bool any = false;
        for (int y = y0; y < std::min(y0 + h->ty, L.ny) && !any; ++y)
          for (int x = x0; x < std::min(x0 + 32, L.nx) && !any; ++x) any = L.solid[(size_t)y * L.nx + x] == 0;
        if (any) tiles.push_back(make_int4(int(l), x0, y0, 0));
      }
    L.tile_end = int(tiles.size());
  }
}

// Strips of the y-sweep: kSweepThreads - 4 interior columns each; rows split into segments
// when the lattices are too narrow to give every SM several strips.  Strips whose own
// columns and rows hold no fluid node are skipped.
void build_strips(lbcg_handle* h, std::vector<int4>& strips) {
  strips.clear();
  const int W = sweep_width(h->prec == LBCG_FP64);
  long long nx_strips = 0;
  for (const LatHost& L : h->lats) nx_strips += (L.nx + W - 1) / W;
  // automatic segment height: split the strips into about 32 blocks per SM (FP64: 8), with
  // at least 24 rows per segment (FP64: 8), since each segment also sweeps 4 warm-up rows.
  // Blocks are launched in lattice / segment row / strip order (below).  (Measured on a
  // 64-channel batch and an 8192 x 4096 box: 32 blocks per SM beat 16 by 1.5-5 %; segments
  // under 24 rows lose.)
  const bool fp64 = h->prec == LBCG_FP64;
  const long long target = fp64 ? 152LL * 8 : 152LL * 32;
  const int min_rows = fp64 ? 8 : 24;
  for (size_t l = 0; l < h->lats.size(); ++l) {
    const LatHost& L = h->lats[l];
    int rows = h->sweep_rows;
    if (rows <= 0) {
      const long long k = nx_strips >= target ? 1 : (target + nx_strips - 1) / nx_strips;
      rows = int(std::max<long long>(min_rows, (L.ny + k - 1) / k));
    }
    // Blocks go out segment row by segment row (all strips of segment row 0, then row 1, ...),
    // so that the blocks resident at a time cover whole bands of rows: x-neighbouring strips
    // share their halo segments in L2.  The FP32-arithmetic sweep walks every other segment
    // row downwards, so that the two segments at each boundary reach its rows at about the
    // same time (their second read then hits L2).  (8192 x 4096 box: strip by strip instead,
    // 157 B of DRAM traffic per fluid node and 0.886 ms per sweep; this order 147 B, 0.827 ms.)
    // The lattice's rows are cut into as many segments as the height asks for, of equal
    // heights (72 rows at 64: 36 + 36, not 64 + 8): the same rows and warm-up rows in all, but
    // blocks of about equal length (64-channel batch, FP32: 0.2988-0.3013 -> 0.2965 ms per step).
    {
      const int nseg = (L.ny + rows - 1) / rows;
      rows = (L.ny + nseg - 1) / nseg;
    }
    for (int y0 = 0, k = 0; y0 < L.ny; y0 += rows, ++k)
      for (int x0 = 0; x0 < L.nx; x0 += W) {
        const int y1 = std::min(y0 + rows, L.ny);
        bool any = false;
        for (int y = y0; y < y1 && !any; ++y)
          for (int x = x0; x < std::min(x0 + W, L.nx) && !any; ++x) any = L.solid[(size_t)y * L.nx + x] == 0;
        const int down = (!fp64 && (k & 1)) ? kStripDown : 0;
        if (any) strips.push_back(make_int4(int(l) | down, x0, y0, y1));
      }
  }
}

LaunchStep make_launch(lbcg_handle* h, int src, double* macro, int tile_begin, int tile_end) {
  LaunchStep p{};
  p.lats = h->d_lats;
  p.groups = h->d_groups;
  p.ngroups = h->ngroups;
  p.wband = h->d_wband;
  p.wvirt = h->d_wvirt;
  p.wsten = h->d_wsten;
  p.ofb = h->d_ofb;
  p.tiles = h->d_tiles + tile_begin;
  p.ntiles = tile_end - tile_begin;
  p.ty = h->ty;
  p.src = h->pool[src];
  p.dst = h->pool[src ^ 1];
  p.flags = h->d_flags;
  p.nbmask = h->d_nbmask;
  p.err = h->d_err;
  p.poll_limit = h->poll_limit;
  p.sr_epoch = h->d_sr_epoch;
  p.sr_step = uint32_t(h->step);
  p.scheme_b = h->scheme_b;
  p.wall = h->d_wall;
  p.node_total = h->node_total;
  p.macro = macro;
  p.strips = h->d_strips;
  p.nstrips = h->nstrips;
  p.sweep = h->sweep;
  return p;
}

// the launch of one step of the lattices [l0, l1) alone (the lists are in lattice order)
LaunchStep make_launch_lats(lbcg_handle* h, int src, int l0, int l1) {
  LaunchStep p = make_launch(h, src, nullptr, h->lat_tile[l0], h->lat_tile[l1]);
  p.strips = h->d_strips + h->lat_strip[l0];
  p.nstrips = h->lat_strip[l1] - h->lat_strip[l0];
  p.groups = h->d_groups + h->lat_group[l0];
  p.ngroups = h->lat_group[l1] - h->lat_group[l0];
  return p;
}

// splits the lattices into ng >= 1 groups of consecutive lattices of about equal node counts,
// each with at least one lattice: group g is [end[g], end[g+1]); returns the number of groups
// (1 if the lists are not in lattice order)
int split_lattices(const lbcg_handle* h, int ng, int* end) {
  const int n = int(h->lats.size());
  ng = std::max(1, std::min(ng, n));
  if (h->lat_strip.empty()) ng = 1;
  auto nodes = [&](int l) { return (long long)h->lats[l].nx * h->lats[l].ny; };
  long long total = 0, acc = 0;
  for (int l = 0; l < n; ++l) total += nodes(l);
  // group g ends at the first lattice boundary whose node count reaches (g + 1) / ng of the
  // total, leaving at least one lattice to each later group
  int l = 0;
  end[0] = 0;
  for (int g = 0; g < ng - 1; ++g) {
    do acc += nodes(l++);
    while (l < n - (ng - 1 - g) && acc * ng < total * (g + 1));
    end[g + 1] = l;
  }
  end[ng] = n;
  return ng;
}

void free_handle(lbcg_handle* h) {
  if (!h) return;
  if (h->graph) cudaGraphExecDestroy(h->graph);
  for (cudaEvent_t e : h->events) cudaEventDestroy(e);
  if (h->prof_ref) cudaEventDestroy(h->prof_ref);
  void* ptrs[] = {h->pool[0], h->pool[1], h->d_flags,  h->d_wall,  h->d_macro, h->d_lats,
                  h->d_tiles, h->d_groups, h->d_wband, h->d_wvirt, h->d_wsten, h->d_ofb,
                  h->d_obs,   h->d_strips, h->d_nbmask, h->d_err, h->d_usnap, h->d_sr_epoch,
                  h->d_run,   h->d_progress};
  if (h->stream) cudaStreamSynchronize(h->stream);
  if (h->h_small) cudaFreeHost(h->h_small);
  for (void* p : ptrs) dev_free(h, p);
  for (int b = 0; b < kGraphBranches; ++b) {
    if (h->br_stream[b]) cudaStreamDestroy(h->br_stream[b]);
    if (h->ev_join[b]) cudaEventDestroy(h->ev_join[b]);
  }
  for (cudaStream_t st : h->io_stream)
    if (st) cudaStreamDestroy(st);
  for (cudaEvent_t e : h->io_events) cudaEventDestroy(e);
  if (h->ev_fork) cudaEventDestroy(h->ev_fork);
  if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
  delete h;
}

lbcg_status upload_tiles(lbcg_handle* h) {
  std::vector<int4> tiles;
  build_tiles(h, tiles);
  dev_free(h, h->d_tiles);
  h->d_tiles = nullptr;
  h->ntiles = int(tiles.size());
  if (!dev_alloc(h, (void**)&h->d_tiles, std::max<size_t>(1, tiles.size()) * sizeof(int4)))
    return fail(LBCG_E_NOMEM, "cannot allocate the tile list");
  if (!tiles.empty()) CK(h, cudaMemcpy(h->d_tiles, tiles.data(), tiles.size() * sizeof(int4), cudaMemcpyHostToDevice));
  std::vector<int4> strips;
  build_strips(h, strips);
  dev_free(h, h->d_strips);
  h->d_strips = nullptr;
  h->nstrips = int(strips.size());
  if (!dev_alloc(h, (void**)&h->d_strips, std::max<size_t>(1, strips.size()) * sizeof(int4)))
    return fail(LBCG_E_NOMEM, "cannot allocate the strip list");
  if (!strips.empty())
    CK(h, cudaMemcpy(h->d_strips, strips.data(), strips.size() * sizeof(int4), cudaMemcpyHostToDevice));
  // per-lattice ranges of the three lists, and the graph branches of a batch
  const int n = int(h->lats.size());
  auto lat_of = [](const int4& e) { return e.x & ~kStripDown; };
  bool sorted = true;
  for (size_t i = 1; i < strips.size(); ++i) sorted = sorted && lat_of(strips[i]) >= lat_of(strips[i - 1]);
  for (size_t i = 1; i < tiles.size(); ++i) sorted = sorted && lat_of(tiles[i]) >= lat_of(tiles[i - 1]);
  for (size_t i = 1; i < h->group_lat.size(); ++i) sorted = sorted && h->group_lat[i] >= h->group_lat[i - 1];
  h->lat_strip.clear();
  h->lat_tile.clear();
  h->lat_group.clear();
  if (sorted) {
    auto first = [&](const std::vector<int4>& v, int lat) {
      int i = 0;
      while (i < int(v.size()) && lat_of(v[i]) < lat) ++i;
      return i;
    };
    for (int l = 0; l <= n; ++l) {
      h->lat_strip.push_back(first(strips, l));
      h->lat_tile.push_back(first(tiles, l));
      int g = 0;
      while (g < int(h->group_lat.size()) && h->group_lat[g] < l) ++g;
      h->lat_group.push_back(g);
    }
  }
  h->nbranch = split_lattices(h, kGraphBranches, h->br_lat);
  return LBCG_OK;
}

// Plans the resident kernel and uploads the plan (once per handle, when the tile schedule is
// chosen).  Lattices that do not fit keep the launch-per-step schedule.
lbcg_status plan_run(lbcg_handle* h) {
  if (h->run_planned) return LBCG_OK;
  h->run_planned = true;
  int dev = 0, sms = 0, smem_max = 0;
  CK(h, cudaGetDevice(&dev));
  CK(h, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  CK(h, cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  const size_t cs = compute_size(h->prec);
  const int blocks = run_blocks(cs);
  const size_t budget = size_t(std::max(0, smem_max / blocks - 2048));   // static and reserved shared memory apart
  std::vector<LatGeom> views;
  std::vector<const uint8_t*> flags;
  long long fluid = 0;
  for (const LatHost& L : h->lats) {
    views.push_back(LatGeom{L.nx, L.ny, L.pitch, L.bcx, L.bcy, L.solid.data()});
    flags.push_back(&h->flags_host[L.node_off]);
    fluid += L.n_fluid;
  }
  // (a fluid node takes at least its 12 values and 8 bytes of tables)
  if (fluid * (long long)(12 * cs + 8) > (long long)sms * blocks * (long long)budget) return LBCG_OK;
  // Small lattices take blocks that leave room on their SMs for those of other handles: a cooperative
  // grid starts only once all its blocks have room, so that grids of large blocks run one after another.
  // FP32: one tile per SM, where 128 threads take each stage of it in one pass, is as fast as two half
  // as large (100 x 50: 3.30 us per step either way), and eight handles at once on streams of their own
  // take 0.92 us per step of each, for 1.75.  16-bit storage keeps two (3.27 us, one 3.37).
  RunPlan p;
  const bool one = h->prec == LBCG_FP32 && fluid <= (long long)kRunSmallThreads / 2 * sms &&
                   build_run_plan(views, flags, h->ofb_host, sms, budget, cs, p) && run_one_pass(p);
  if (!one && !build_run_plan(views, flags, h->ofb_host, blocks * sms, budget, cs, p)) return LBCG_OK;
  for (const RunTile& t : p.tiles) {
    h->run_nodes = std::max(h->run_nodes, t.tx * t.ty);
    h->run_slots = std::max(h->run_slots, (t.tx + 4) * (t.ty + 4));
  }
  // Blocks of 128 threads where the tiles are that small.  FP32: they also leave registers for a kernel
  // on another stream, the adjoint's reverse sweep beside the recompute of a segment (400 x 42: 20 us per
  // step of the gradient, for 23 with 256 threads, although the steps alone take 4.27 us, for 3.99; 100 x 50
  // 3.35 and 3.38, in FP16 3.42 and 3.55).  FP64: where each stage is one pass of them (100 x 50: 10.6 us
  // per step either way; eight handles at once 6.0 us per step of each, for 10.6; with two passes 1.1
  // to 1.2 times the time of 256 threads).
  h->run_threads = (cs == 4 ? h->run_nodes <= 64 : run_one_pass(p)) ? kRunSmallThreads : 256;
  int per_sm = 0;
  CK(h, prepare_run(h->prec, h->run_threads, p.smem, &per_sm));
  if ((long long)per_sm * sms < (long long)p.tiles.size()) return LBCG_OK;
  size_t total = 0;
  std::vector<std::pair<const void*, size_t>> parts;
  std::vector<size_t> at;
  auto add = [&](const void* src, size_t bytes) {
    at.push_back(total);
    parts.push_back({src, bytes});
    total += (bytes + 255) & ~size_t(255);
  };
  add(p.tiles.data(), p.tiles.size() * sizeof(RunTile));
  add(p.nb.data(), p.nb.size() * sizeof(int));
  add(p.extra.data(), p.extra.size() * sizeof(int));
  add(p.w_ofb.data(), p.w_ofb.size() * sizeof(int));
  add(p.w_sten.data(), p.w_sten.size() * sizeof(WallSten));
  add(p.v_sten.data(), p.v_sten.size() * sizeof(WallSten));
  add(p.copies.data(), p.copies.size() * sizeof(uint32_t));
  add(p.vn.data(), p.vn.size() * sizeof(RunVirtN));
  add(p.band.data(), p.band.size() * sizeof(uint16_t));
  std::vector<char> host(std::max<size_t>(total, 16), 0);
  for (size_t i = 0; i < parts.size(); ++i)
    if (parts[i].second) memcpy(host.data() + at[i], parts[i].first, parts[i].second);
  const size_t pb = p.tiles.size() * kRunFlagStride * sizeof(unsigned);
  // without memory for the plan the handle keeps one launch per kernel and step
  if (!dev_alloc(h, (void**)&h->d_run, host.size()) || !dev_alloc(h, (void**)&h->d_progress, pb)) {
    dev_free(h, h->d_run);
    h->d_run = nullptr;
    h->d_progress = nullptr;
    return LBCG_OK;
  }
  CK(h, cudaMemcpy(h->d_run, host.data(), host.size(), cudaMemcpyHostToDevice));
  CK(h, cudaMemset(h->d_progress, 0, pb));
  // both may still be under way when they return, and the handle's stream need not wait for the
  // legacy stream they run on
  CK(h, cudaStreamSynchronize(cudaStreamLegacy));
  RunArgs a{};
  a.lats = h->d_lats;
  a.tiles = reinterpret_cast<const RunTile*>(h->d_run + at[0]);
  a.nb = reinterpret_cast<const int*>(h->d_run + at[1]);
  a.extra = reinterpret_cast<const int*>(h->d_run + at[2]);
  a.w_ofb = reinterpret_cast<const int*>(h->d_run + at[3]);
  a.w_sten = reinterpret_cast<const WallSten*>(h->d_run + at[4]);
  a.v_sten = reinterpret_cast<const WallSten*>(h->d_run + at[5]);
  a.copies = reinterpret_cast<const uint32_t*>(h->d_run + at[6]);
  a.vn = reinterpret_cast<const RunVirtN*>(h->d_run + at[7]);
  a.band = reinterpret_cast<const uint16_t*>(h->d_run + at[8]);
  a.ofb = h->d_ofb;
  a.flags = h->d_flags;
  a.nbmask = h->d_nbmask;
  a.progress = h->d_progress;
  a.err = h->d_err;
  a.sr_epoch = h->d_sr_epoch;
  h->run = a;
  h->run_smem = p.smem;
  h->run_tiles = int(p.tiles.size());
  return LBCG_OK;
}

// Whether a call of nsteps steps runs as launches of the resident kernel: from kRunMinSteps on
// (a launch resolves the lattice's tables first, about two steps' worth of time), except a call
// of exactly one graph replay, whose launches per step callers may count (lbcg_step_launches).
// Profiled handles (events around each kernel), handles whose poll limit was changed and
// streams that are being captured keep the launch-per-step schedule.
bool runs_resident(const lbcg_handle* h, int64_t nsteps) {
  if (h->sweep || h->run_tiles == 0 || h->profiling || h->poll_limit != kPollLimit) return false;
  if (nsteps < kRunMinSteps || nsteps == kGraphSteps) return false;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  return cudaStreamIsCapturing(h->stream, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone;
}

// One launch of the resident kernel: n steps from the handle's current state; *n is lowered to
// what one launch takes.
cudaError_t enqueue_run(lbcg_handle* h, int64_t* n) {
  const int pre = h->cur;   // graph replays start from pool 0
  if (*n > kRunMaxSteps) *n = pre + kRunMaxSteps / kGraphSteps * kGraphSteps;
  RunArgs a = h->run;
  a.pool0 = static_cast<char*>(h->pool[h->cur]);
  a.pool1 = static_cast<char*>(h->pool[h->cur ^ 1]);
  a.nsteps = int(*n);
  a.poll_limit = h->run_polls;
  a.base = h->run_base;
  a.step0 = uint32_t(h->step);
  a.pre = pre;
  a.nrep = int((*n - pre) / kGraphSteps);
  h->run_base += unsigned(*n);
  cudaError_t e = launch_run(h->prec, a, h->run_tiles, h->run_threads, h->run_smem, h->stream);
  h->step_launches += 1;
  if (e == cudaSuccess && h->prec >= 2 && a.nrep > 0) {
    e = launch_sr_add(h->d_sr_epoch, uint32_t(a.nrep), h->stream);
    h->step_launches += 1;
  }
  return e;
}

lbcg_status ensure_macro(lbcg_handle* h) {
  if (!h->d_macro) {
    if (!dev_alloc(h, (void**)&h->d_macro, 4 * (size_t)h->node_total * sizeof(double)))
      return fail(LBCG_E_NOMEM, "cannot allocate the macroscopic fields");
    CK(h, cudaMemsetAsync(h->d_macro, 0, 4 * (size_t)h->node_total * sizeof(double), h->stream));
  }
  return LBCG_OK;
}

// After a synchronisation: a sweep block gave up waiting for a staged row (or a block of a resident
// kernel for a tile next to it), so the state of the steps since the last check is unreliable (that
// block stopped without writing the rest).  The word is cleared once reported: the handle stays
// usable, and a state set or uploaded afterwards steps correctly again.
lbcg_status report_device_error(lbcg_handle* h, int e) {
  if (e) {
    // (on the handle's stream: before what is launched next)
    if (cudaMemsetAsync(h->d_err, 0, sizeof(int), h->stream) != cudaSuccess)
      return cuda_fail(h, cudaGetLastError(), "clearing the device error word");
    if (e & ERR_BOUNDS)
      return fail(LBCG_E_BOUNDS, "a range check of the checked build failed in a step kernel (the access was "
                                 "skipped; the state since the last check is unreliable)");
    return fail(LBCG_E_TIMEOUT,
                "a step kernel's bounded wait ran out%s; the state since the last check is "
                "unreliable",
                (e & ERR_DRAIN) ? " and its copies could not be drained" : "");
  }
  return LBCG_OK;
}
lbcg_status check_device_error(lbcg_handle* h) {
  int e = 0;
  if (cudaMemcpy(&e, h->d_err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
    return cuda_fail(h, cudaGetLastError(), "reading the device error word");
  return report_device_error(h, e);
}
// The end of a call that returns data: the error word comes back behind what is already on the
// stream, so that the call waits for the GPU once (a blocking copy of the word after the wait
// cost about 10 us of a call).
lbcg_status finish_stream(lbcg_handle* h) {
  CK(h, cudaMemcpyAsync(&h->h_small->err, h->d_err, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  CK(h, cudaStreamSynchronize(h->stream));
  return report_device_error(h, h->h_small->err);
}

lbcg_status check_handle(const lbcg_handle* h) {
  if (!h) return fail(LBCG_E_ARG, "NULL handle");
  if (h->dead) return fail(LBCG_E_CUDA, "handle is dead after an earlier CUDA error");
  return LBCG_OK;
}

lbcg_status run_macro(lbcg_handle* h, int lat) {
  lbcg_status s = ensure_macro(h);
  if (s != LBCG_OK) return s;
  const LatHost& L = h->lats[lat];
  LaunchStep p = make_launch(h, h->cur, h->d_macro, L.tile_begin, L.tile_end);
  CK(h, launch_step(h->prec, p, h->stream));
  return LBCG_OK;
}

}  // namespace

void lbcg::set_last_error(const char* msg) { g_err = msg; }

namespace {

// the streams and fork / join events of a batch's parallel branches
cudaError_t ensure_branches(lbcg_handle* h) {
  cudaError_t e = cudaSuccess;
  if (!h->ev_fork) e = cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming);
  for (int b = 1; b < h->nbranch && e == cudaSuccess; ++b) {
    if (!h->br_stream[b]) e = cudaStreamCreateWithFlags(&h->br_stream[b], cudaStreamNonBlocking);
    if (e == cudaSuccess && !h->ev_join[b]) e = cudaEventCreateWithFlags(&h->ev_join[b], cudaEventDisableTiming);
  }
  return e;
}

// Captures nsteps steps into an executable graph.  A batch runs as h->nbranch parallel
// branches (branches 1.. forked from the handle's stream at the start and joined back at the
// end).  probe = false: the steps advance from pool A (step k reads pool k & 1) and carry their
// index k within the replay; 16-bit storage first advances the replay counter that keys the
// stochastic rounding.  probe = true (lbcg_autotune): every step reads the current state and
// writes the other pool, so replays do not advance the simulation, and the counter is left
// alone.  *nk: the kernel nodes captured.
lbcg_status capture_steps(lbcg_handle* h, int nsteps, bool probe, cudaGraphExec_t* out, int64_t* nk) {
  cudaGraph_t g = nullptr;
  CK(h, cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
  cudaError_t le = cudaSuccess;
  *nk = 0;
  if (!probe && h->prec >= 2) {
    le = launch_sr_tick(h->d_sr_epoch, h->stream);
    *nk += 1;
  }
  int nfork = 0;   // branches 1 .. nfork have joined the capture
  if (h->nbranch > 1 && le == cudaSuccess) {
    le = ensure_branches(h);
    if (le == cudaSuccess) le = cudaEventRecord(h->ev_fork, h->stream);
    for (int b = 1; b < h->nbranch && le == cudaSuccess; ++b) {
      le = cudaStreamWaitEvent(h->br_stream[b], h->ev_fork, 0);
      if (le == cudaSuccess) nfork = b;
    }
  }
  const bool forked = h->nbranch > 1 && nfork == h->nbranch - 1 && le == cudaSuccess;
  for (int k = 0; k < nsteps && le == cudaSuccess; ++k) {
    const int src = probe ? h->cur : (k & 1);
    if (forked) {
      for (int b = 0; b < h->nbranch && le == cudaSuccess; ++b) {
        LaunchStep q = make_launch_lats(h, src, h->br_lat[b], h->br_lat[b + 1]);
        q.sr_step = uint32_t(k);
        le = launch_step(h->prec, q, b ? h->br_stream[b] : h->stream);
        *nk += step_kernels(q);
      }
    } else {
      LaunchStep q = make_launch(h, src, nullptr, 0, h->ntiles);
      q.sr_step = uint32_t(k);
      le = launch_step(h->prec, q, h->stream);
      *nk += step_kernels(q);
    }
  }
  // join every forked branch, also after a failed launch, so that the capture can end
  for (int b = 1; b <= nfork; ++b) {
    const cudaError_t je = cudaEventRecord(h->ev_join[b], h->br_stream[b]);
    const cudaError_t we = je == cudaSuccess ? cudaStreamWaitEvent(h->stream, h->ev_join[b], 0) : je;
    if (le == cudaSuccess) le = we;
  }
  const cudaError_t ee = cudaStreamEndCapture(h->stream, &g);
  if (le != cudaSuccess) {
    if (g) cudaGraphDestroy(g);
    return cuda_fail(h, le, "launch during capture");
  }
  if (ee != cudaSuccess) return cuda_fail(h, ee, "cudaStreamEndCapture");
  const cudaError_t ie = cudaGraphInstantiate(out, g, 0);
  cudaGraphDestroy(g);
  if (ie != cudaSuccess) return cuda_fail(h, ie, "cudaGraphInstantiate");
  return LBCG_OK;
}

}  // namespace

extern "C" {

const char* lbcg_last_error(void) { return g_err.c_str(); }

lbcg_status lbcg_set_allocator(const lbcg_allocator* a) {
  g_err.clear();
  if (a && (!a->alloc || !a->release)) return fail(LBCG_E_ARG, "an allocator needs both alloc and release");
  std::lock_guard<std::mutex> lock(g_alloc_mutex);
  g_allocator = a ? *a : lbcg_allocator{nullptr, nullptr, nullptr};
  return LBCG_OK;
}

lbcg_status lbcg_create_batch(int32_t n, const lbcg_geometry* geoms, const lbcg_params* prms, int32_t precision,
                              void* stream, lbcg_handle** out) {
  Range range_("lbcg_create_batch");
  g_err.clear();
  if (!out) return fail(LBCG_E_ARG, "NULL output handle pointer");
  *out = nullptr;
  if (n < 1 || !geoms || !prms) return fail(LBCG_E_ARG, "need n >= 1 lattices with geometry and params");
  if (precision < 0 || precision > 3) return fail(LBCG_E_ARG, "bad precision %d", precision);
  for (int l = 0; l < n; ++l) {
    lbcg_status s = validate(&geoms[l], &prms[l], l);
    if (s != LBCG_OK) return s;
  }
  lbcg_handle* h = new lbcg_handle();
  h->prec = precision;
  {
    std::lock_guard<std::mutex> lock(g_alloc_mutex);
    h->allocator = g_allocator;
  }
  if (stream) {
    h->stream = static_cast<cudaStream_t>(stream);
  } else {
    cudaError_t e = cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
      free_handle(h);
      return fail(LBCG_E_CUDA, "cudaStreamCreate: %s", cudaGetErrorString(e));
    }
    h->own_stream = true;
  }
  // layout
  std::vector<LatDev> ld(n);
  std::vector<OfbEntry> ofb;
  long long node_total = 0;
  for (int l = 0; l < n; ++l) {
    const lbcg_geometry* g = &geoms[l];
    LatHost L{};
    L.nx = g->nx;
    L.ny = g->ny;
    L.pitch = (g->nx + 31) / 32 * 32;
    L.bcx = g->bc_x;
    L.bcy = g->bc_y;
    L.plane = (long long)L.pitch * L.ny;
    L.node_off = node_total;
    L.pop_off = 18 * node_total;
    L.prm = prms[l];
    L.solid.assign(g->solid, g->solid + (size_t)g->nx * g->ny);
    L.n_fluid = 0;
    for (uint8_t s : L.solid) L.n_fluid += s == 0;
    node_total += L.plane;
    h->lats.push_back(L);
    LatDev& d = ld[l];
    d.nx = L.nx;
    d.ny = L.ny;
    d.pitch = L.pitch;
    d.bcx = L.bcx;
    d.bcy = L.bcy;
    d.pop_off = L.pop_off;
    d.plane = L.plane;
    d.node_off = L.node_off;
    const lbcg_params& p = prms[l];
    d.nu_R = p.nu_R;
    d.nu_B = p.nu_B;
    d.sigma = p.sigma;
    d.beta = p.beta;
    d.s_e = p.s_e;
    d.s_eps = p.s_eps;
    d.s_q = p.s_q;
    d.rho0 = p.rho0;
    d.u_in = p.u_in;
    d.in_prof = p.inlet_profile;
    d.wetting = p.wetting;
    if (p.wetting == 1) h->scheme_b = 1;
    d.cos_theta = std::cos(p.theta);
    {
      // fluid rows of the inlet column: the profile spans them, walls half a node beyond
      int lo = -1, hi = -1;
      for (int y = 0; y < geoms[l].ny; ++y)
        if (!geoms[l].solid[(size_t)y * geoms[l].nx]) {
          if (lo < 0) lo = y;
          hi = y;
        }
      d.in_y0 = lo < 0 ? 0.0 : lo - 0.5;
      d.in_w = lo < 0 ? 1.0 : double(hi - lo + 1);
    }
    d.rho_out = p.rho_out;
    d.grad_eps = p.grad_eps;
    d.h_inv_nuR = 0.5 / p.nu_R;
    d.h_inv_nuB = 0.5 / p.nu_B;
    const LatConst<double> c = d.consts<double>();
    d.cf = LatConst<float>{float(c.sigma),   float(c.beta),     float(c.s_e),       float(c.s_eps),
                           float(c.s_q),     float(c.rho0),     float(c.u_in),      float(c.rho_out),
                           float(c.grad_eps), float(c.h_inv_nuR), float(c.h_inv_nuB), float(c.cos_theta)};
  }
  h->node_total = node_total;
  h->flags_host.assign((size_t)node_total, F_SOLID);
  std::vector<uint8_t> mask_host((size_t)node_total, 0);
  for (int l = 0; l < n; ++l) {
    std::vector<uint8_t> fl, mk;
    const size_t first = ofb.size();
    classify(&geoms[l], &prms[l], l, fl, mk, ofb);
    // (a vector divided by its length is off by 6e-16 in its square at most)
    ld[l].unit_normals = std::all_of(ofb.begin() + first, ofb.end(), [](const OfbEntry& e) {
      const double n2 = e.nsx * e.nsx + e.nsy * e.nsy;
      return std::fabs(n2 - 1.0) <= 1e-15 || n2 == 0.0;
    });
    const LatHost& L = h->lats[l];
    for (int y = 0; y < L.ny; ++y) {
      memcpy(&h->flags_host[L.node_off + (size_t)y * L.pitch], &fl[(size_t)y * L.nx], L.nx);
      memcpy(&mask_host[L.node_off + (size_t)y * L.pitch], &mk[(size_t)y * L.nx], L.nx);
    }
  }
  h->nofb = int(ofb.size());
  h->ofb_host = ofb;
  // wall groups: smaller units when there are few outermost fluid nodes, so that they spread
  // over the SMs
  std::vector<WallGroup> groups;
  std::vector<int> wband;
  std::vector<WallSten> wvirt, wsten;
  {
    int gmax = kWallMaxNodes;
    while (gmax > 32 && (h->nofb + gmax - 1) / gmax < 2 * kSMs) gmax >>= 1;
    std::vector<LatGeom> views;
    for (const LatHost& L : h->lats) views.push_back(LatGeom{L.nx, L.ny, L.pitch, L.bcx, L.bcy, L.solid.data()});
    build_wall_groups(views, ofb, gmax, groups, wband, wvirt, wsten);
  }
  h->ngroups = int(groups.size());
  h->group_lat.clear();
  for (const WallGroup& G : groups) h->group_lat.push_back(G.lat);
  const size_t es = elem_size(precision), cs = compute_size(precision);
  auto alloc = [&](void** p, size_t bytes) { return dev_alloc(h, p, bytes); };
  bool ok = alloc(&h->pool[0], 18 * (size_t)node_total * es) && alloc(&h->pool[1], 18 * (size_t)node_total * es) &&
            alloc((void**)&h->d_flags, (size_t)node_total) && alloc((void**)&h->d_nbmask, (size_t)node_total) &&
            alloc((void**)&h->d_err, sizeof(int)) && alloc((void**)&h->d_sr_epoch, sizeof(uint32_t)) &&
            alloc(&h->d_wall, 4 * (size_t)node_total * cs) && alloc((void**)&h->d_lats, n * sizeof(LatDev)) &&
            alloc((void**)&h->d_groups, groups.size() * sizeof(WallGroup)) &&
            alloc((void**)&h->d_wband, wband.size() * sizeof(int)) &&
            alloc((void**)&h->d_wvirt, wvirt.size() * sizeof(WallSten)) &&
            alloc((void**)&h->d_wsten, wsten.size() * sizeof(WallSten)) &&
            alloc((void**)&h->d_ofb, ofb.size() * sizeof(OfbEntry)) &&
            alloc((void**)&h->d_obs, (obs_partials_doubles() + kObsOut) * sizeof(double));
  if (!ok) {
    free_handle(h);
    return fail(LBCG_E_NOMEM, "device allocation failed (%lld nodes)", node_total);
  }
  if (cudaMallocHost((void**)&h->h_small, sizeof(*h->h_small)) != cudaSuccess) {
    cudaGetLastError();
    h->h_small = nullptr;
    free_handle(h);
    return fail(LBCG_E_NOMEM, "pinned host allocation failed");
  }
#define CKC(call)                                         \
  do {                                                    \
    cudaError_t e_ = (call);                              \
    if (e_ != cudaSuccess) {                              \
      lbcg_status s_ = cuda_fail(h, e_, #call);           \
      free_handle(h);                                     \
      return s_;                                          \
    }                                                     \
  } while (0)
  CKC(cudaMemcpy(h->d_flags, h->flags_host.data(), (size_t)node_total, cudaMemcpyHostToDevice));
  CKC(cudaMemcpy(h->d_nbmask, mask_host.data(), (size_t)node_total, cudaMemcpyHostToDevice));
  CKC(cudaMemset(h->d_err, 0, sizeof(int)));
  CKC(cudaMemset(h->d_sr_epoch, 0, sizeof(uint32_t)));
  CKC(prepare_kernels(precision));

  CKC(cudaMemcpy(h->d_lats, ld.data(), n * sizeof(LatDev), cudaMemcpyHostToDevice));
  if (!groups.empty()) {
    CKC(cudaMemcpy(h->d_groups, groups.data(), groups.size() * sizeof(WallGroup), cudaMemcpyHostToDevice));
    CKC(cudaMemcpy(h->d_wband, wband.data(), wband.size() * sizeof(int), cudaMemcpyHostToDevice));
    if (!wvirt.empty())
      CKC(cudaMemcpy(h->d_wvirt, wvirt.data(), wvirt.size() * sizeof(WallSten), cudaMemcpyHostToDevice));
    CKC(cudaMemcpy(h->d_wsten, wsten.data(), wsten.size() * sizeof(WallSten), cudaMemcpyHostToDevice));
  }
  if (!ofb.empty()) CKC(cudaMemcpy(h->d_ofb, ofb.data(), ofb.size() * sizeof(OfbEntry), cudaMemcpyHostToDevice));
  CKC(cudaMemset(h->pool[0], 0, 18 * (size_t)node_total * es));
  CKC(cudaMemset(h->pool[1], 0, 18 * (size_t)node_total * es));
  CKC(cudaMemset(h->d_wall, 0, 4 * (size_t)node_total * cs));
  {
    lbcg_status s = upload_tiles(h);
    // default schedule: the y-sweep when its strips give every SM a block, else tiles
    // (FP64 arithmetic is slow per SM, so FP64 takes the smallest tiles, i.e. the most blocks).
    // FP64 lattices that the resident kernel holds take the tiles in any case: 2000 x 102,
    // 248 us per step swept, 111 resident.
    if (s == LBCG_OK && h->nstrips >= kSMs && precision == LBCG_FP64) s = plan_run(h);
    if (s == LBCG_OK && (h->nstrips < kSMs || (precision == LBCG_FP64 && h->run_tiles > 0))) {
      h->sweep = 0;
      h->ty = precision == LBCG_FP64 ? 4 : kDefaultTY;
      s = upload_tiles(h);
      if (s == LBCG_OK) s = plan_run(h);
    }
    if (s != LBCG_OK) {
      free_handle(h);
      return s;
    }
  }
  // initial populations at rest: f_{a,R} = w_a rho0 (1 + rhoN0)/2, f_{a,B} = w_a rho0 (1 - rhoN0)/2
  const double W[9] = {4.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 36, 1.0 / 36, 1.0 / 36, 1.0 / 36};
  for (int l = 0; l < n; ++l) {
    const lbcg_geometry* g = &geoms[l];
    const size_t nn = (size_t)g->nx * g->ny;
    std::vector<double> host(18 * nn, 0.0);
    for (size_t i = 0; i < nn; ++i) {
      if (g->solid[i]) continue;
      const double r = g->rhoN0[i];
      for (int a = 0; a < 9; ++a) {
        host[a * nn + i] = W[a] * prms[l].rho0 * (1 + r) / 2;
        host[(9 + a) * nn + i] = W[a] * prms[l].rho0 * (1 - r) / 2;
      }
    }
    double* tmp = nullptr;
    if (!dev_alloc(h, (void**)&tmp, 18 * nn * sizeof(double))) {
      free_handle(h);
      return fail(LBCG_E_NOMEM, "staging allocation");
    }
    cudaError_t e = cudaMemcpy(tmp, host.data(), 18 * nn * sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = launch_to_storage(precision, h->d_lats, l, (long long)nn, tmp, h->d_flags, h->pool[0], 0);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    dev_free(h, tmp);
    CKC(e);
  }
  CKC(cudaMemcpy(h->pool[1], h->pool[0], 18 * (size_t)node_total * es, cudaMemcpyDeviceToDevice));
#undef CKC
  *out = h;
  return LBCG_OK;
}

lbcg_status lbcg_create(const lbcg_geometry* geom, const lbcg_params* prm, int32_t precision, void* stream,
                        lbcg_handle** out) {
  return lbcg_create_batch(1, geom, prm, precision, stream, out);
}

lbcg_status lbcg_step(lbcg_handle* h, int64_t nsteps) {
  Range range_("lbcg_step");
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (nsteps < 0) return fail(LBCG_E_ARG, "nsteps < 0");
  while (nsteps > 0) {
    if (h->profiling) {
      // direct launches in the graph's arrangement: a batch's branches on their own streams,
      // forked once and joined when this call ends; events before and after every kernel
      const int nb = h->nbranch;
      if (!h->prof_ref) CK(h, cudaEventCreate(&h->prof_ref));
      if (!h->prof_ref_set) {
        CK(h, cudaEventRecord(h->prof_ref, h->stream));
        h->prof_ref_set = true;
      }
      if (nb > 1 && !h->prof_forked) {
        CK(h, ensure_branches(h));
        CK(h, cudaEventRecord(h->ev_fork, h->stream));
        for (int b = 1; b < nb; ++b) CK(h, cudaStreamWaitEvent(h->br_stream[b], h->ev_fork, 0));
        h->prof_forked = true;
      }
      while (h->events.size() < h->events_used + 4 * size_t(nb)) {
        cudaEvent_t e;
        CK(h, cudaEventCreate(&e));
        h->events.push_back(e);
      }
      for (int b = 0; b < nb; ++b) {
        LaunchStep p = nb > 1 ? make_launch_lats(h, h->cur, h->br_lat[b], h->br_lat[b + 1])
                              : make_launch(h, h->cur, nullptr, 0, h->ntiles);
        p.ev = h->events.data() + h->events_used;
        h->events_used += 4;
        CK(h, launch_step(h->prec, p, b ? h->br_stream[b] : h->stream));
        h->step_launches += step_kernels(p);
      }
      h->prof_steps += 1;
      h->cur ^= 1;
      h->step += 1;
      nsteps -= 1;
      continue;
    }
    if (runs_resident(h, nsteps)) {
      int64_t n = nsteps;
      CK(h, enqueue_run(h, &n));
      h->cur ^= int(n & 1);
      h->step += n;
      nsteps -= n;
      continue;
    }
    if (nsteps >= kGraphSteps && h->cur == 0) {
      if (!h->graph) {
        const lbcg_status cs = capture_steps(h, kGraphSteps, false, &h->graph, &h->graph_kernels);
        if (cs != LBCG_OK) return cs;
      }
      CK(h, cudaGraphLaunch(h->graph, h->stream));
      h->step_launches += h->graph_kernels;
      nsteps -= kGraphSteps;
      h->step += kGraphSteps;
      continue;
    }
    const LaunchStep p = make_launch(h, h->cur, nullptr, 0, h->ntiles);
    CK(h, launch_step(h->prec, p, h->stream));
    h->step_launches += step_kernels(p);
    h->cur ^= 1;
    h->step += 1;
    nsteps -= 1;
  }
  if (h->prof_forked) {   // the profiled branches rejoin the handle's stream
    for (int b = 1; b < h->nbranch; ++b) {
      CK(h, cudaEventRecord(h->ev_join[b], h->br_stream[b]));
      CK(h, cudaStreamWaitEvent(h->stream, h->ev_join[b], 0));
    }
    h->prof_forked = false;
  }
  return LBCG_OK;
}

lbcg_status lbcg_observables(lbcg_handle* h, int32_t lattice, const lbcg_obs_spec* spec, lbcg_obs* out) {
  Range range_("lbcg_observables");
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (!spec || !out) return fail(LBCG_E_ARG, "NULL spec or output");
  if (lattice < 0 || lattice >= int(h->lats.size())) return fail(LBCG_E_ARG, "bad lattice index %d", lattice);
  s = run_macro(h, lattice);
  if (s != LBCG_OK) return s;
  const LatHost& L = h->lats[lattice];
  double* parts = h->d_obs;
  double* res = h->d_obs + obs_partials_doubles();
  CK(h, launch_observables(h->d_lats, lattice, L.nx, L.ny, h->d_macro, h->node_total, h->d_flags, spec->tip_row0,
                           spec->tip_row1, spec->cl_row0, spec->cl_row1, parts, res, h->stream));
  const double* const o = h->h_small->v;
  CK(h, cudaMemcpyAsync(h->h_small->v, res, kObsOut * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  s = finish_stream(h);
  if (s != LBCG_OK) return s;
  memset(out, 0, sizeof(*out));
  out->step = h->step;
  out->mass_R = o[0];
  out->mass_B = o[1];
  out->umax = o[2];
  for (int q = 0; q < 9; ++q) out->moments[q] = o[3 + q];
  out->n_pts = o[3];
  out->dp_laplace = (o[13] > 0 && o[15] > 0) ? o[12] / o[13] - o[14] / o[15] : NAN;
  out->nonfinite = o[16] != 0 ? 1 : 0;
  out->x_tip = o[kObsQ + 0];
  {
    double sx = 0;
    int c = 0;
    for (int r = 1; r <= 2; ++r)
      if (o[kObsQ + r] >= 0) {
        sx += o[kObsQ + r];
        ++c;
      }
    out->x_cl = c ? sx / c : -1.0;
  }
  // Kasa circle fit from the moment sums: solve the 3x3 normal equations (Cramer's rule)
  const double* m = out->moments;  // n, Sx, Sy, Sxx, Syy, Sxy, Szx, Szy, Sz
  out->xc = out->yc = out->R = out->theta_deg = NAN;
  if (m[0] >= 3) {
    const double A[3][3] = {{m[3], m[5], m[1]}, {m[5], m[4], m[2]}, {m[1], m[2], m[0]}};
    const double b[3] = {-m[6], -m[7], -m[8]};
    auto det3 = [](const double M[3][3]) {
      return M[0][0] * (M[1][1] * M[2][2] - M[1][2] * M[2][1]) - M[0][1] * (M[1][0] * M[2][2] - M[1][2] * M[2][0]) +
             M[0][2] * (M[1][0] * M[2][1] - M[1][1] * M[2][0]);
    };
    const double D = det3(A);
    if (D != 0) {
      double sol[3];
      for (int c = 0; c < 3; ++c) {
        double Mc[3][3];
        for (int i = 0; i < 3; ++i)
          for (int j = 0; j < 3; ++j) Mc[i][j] = j == c ? b[i] : A[i][j];
        sol[c] = det3(Mc) / D;
      }
      const double xc = -sol[0] / 2, yc = -sol[1] / 2;
      const double R = std::sqrt(std::max(xc * xc + yc * yc - sol[2], 0.0));
      out->xc = xc + 0.5 * L.nx;
      out->yc = yc + 0.5 * L.ny;
      out->R = R;
      double c;
      if (spec->cyl_r > 0) {
        const double D2 = (out->xc - spec->cyl_x) * (out->xc - spec->cyl_x) + (out->yc - spec->cyl_y) * (out->yc - spec->cyl_y);
        c = (spec->cyl_r * spec->cyl_r + R * R - D2) / (2 * spec->cyl_r * R);
      } else {
        c = R > 0 ? (spec->wall_y - out->yc) / R : NAN;
      }
      if (c == c) out->theta_deg = std::acos(std::max(-1.0, std::min(1.0, c))) * 180.0 / 3.14159265358979323846;
    }
  }
  if (out->nonfinite) return fail(LBCG_E_DIVERGED, "non-finite density in lattice %d at step %lld", lattice, (long long)h->step);
  return LBCG_OK;
}

lbcg_status lbcg_diagnostics(lbcg_handle* h, int32_t lattice, const lbcg_diag_spec* spec, lbcg_diag* out) {
  Range range_("lbcg_diagnostics");
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (!spec || !out) return fail(LBCG_E_ARG, "NULL spec or output");
  if (lattice < 0 || lattice >= int(h->lats.size())) return fail(LBCG_E_ARG, "bad lattice index %d", lattice);
  if (!(spec->r > 0)) return fail(LBCG_E_ARG, "the circle needs a radius > 0");
  if (!h->d_usnap) {
    if (!dev_alloc(h, (void**)&h->d_usnap, 2 * (size_t)h->node_total * sizeof(double)))
      return fail(LBCG_E_NOMEM, "cannot allocate the velocity snapshot");
    h->snap_step.assign(h->lats.size(), -1);
  }
  s = run_macro(h, lattice);
  if (s != LBCG_OK) return s;
  const bool have = h->snap_step[lattice] >= 0;
  double* parts = h->d_obs;
  double* res = h->d_obs + obs_partials_doubles();   // the reduction scratch of lbcg_observables
  CK(h, launch_diagnostics(h->d_lats, lattice, h->d_macro, h->node_total, h->d_flags, h->d_usnap, have, spec->cx,
                           spec->cy, spec->r, parts, res, h->stream));
  const double* const q = h->h_small->v;
  CK(h, cudaMemcpyAsync(h->h_small->v, res, 6 * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  s = finish_stream(h);
  if (s != LBCG_OK) return s;
  out->step = h->step;
  out->prev_step = h->snap_step[lattice];
  h->snap_step[lattice] = h->step;
  out->e1 = have ? std::max(q[0], q[1]) : NAN;
  out->m_R_in = q[2];
  out->m_R_out = q[3];
  out->m_B_in = q[4];
  out->m_B_out = q[5];
  const double mR = q[2] + q[3], mB = q[4] + q[5];
  const double wrongO = spec->inside_red ? q[4] / mB : q[2] / mR;   // the outer colour inside C
  const double wrongD = spec->inside_red ? q[3] / mR : q[5] / mB;   // the inner colour outside C
  out->e_npmt = std::sqrt(wrongO * wrongO + wrongD * wrongD);
  return LBCG_OK;
}

lbcg_status lbcg_get_populations(lbcg_handle* h, int32_t lattice, double* host_out) {
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (!host_out || lattice < 0 || lattice >= int(h->lats.size())) return fail(LBCG_E_ARG, "bad arguments");
  const LatHost& L = h->lats[lattice];
  const size_t nn = (size_t)L.nx * L.ny;
  double* tmp = nullptr;
  if (!dev_alloc(h, (void**)&tmp, 18 * nn * sizeof(double))) return fail(LBCG_E_NOMEM, "staging allocation");
  cudaError_t e = launch_from_storage(h->prec, h->d_lats, lattice, (long long)nn, h->pool[h->cur], h->d_flags, tmp, h->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(host_out, tmp, 18 * nn * sizeof(double), cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  dev_free(h, tmp);
  if (e != cudaSuccess) return cuda_fail(h, e, "get_populations");
  return check_device_error(h);
}

lbcg_status lbcg_set_populations(lbcg_handle* h, int32_t lattice, const double* host_in) {
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (!host_in || lattice < 0 || lattice >= int(h->lats.size())) return fail(LBCG_E_ARG, "bad arguments");
  const LatHost& L = h->lats[lattice];
  const size_t nn = (size_t)L.nx * L.ny;
  double* tmp = nullptr;
  if (!dev_alloc(h, (void**)&tmp, 18 * nn * sizeof(double))) return fail(LBCG_E_NOMEM, "staging allocation");
  cudaError_t e = cudaMemcpyAsync(tmp, host_in, 18 * nn * sizeof(double), cudaMemcpyHostToDevice, h->stream);
  if (e == cudaSuccess) e = launch_to_storage(h->prec, h->d_lats, lattice, (long long)nn, tmp, h->d_flags, h->pool[h->cur], h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  dev_free(h, tmp);
  if (e != cudaSuccess) return cuda_fail(h, e, "set_populations");
  return LBCG_OK;
}

lbcg_status lbcg_get_fields(lbcg_handle* h, int32_t lattice, double* host_out) {
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (!host_out || lattice < 0 || lattice >= int(h->lats.size())) return fail(LBCG_E_ARG, "bad arguments");
  s = run_macro(h, lattice);
  if (s != LBCG_OK) return s;
  const LatHost& L = h->lats[lattice];
  const size_t nn = (size_t)L.nx * L.ny;
  std::vector<double> buf(4 * (size_t)L.plane);
  for (int q = 0; q < 4; ++q)
    CK(h, cudaMemcpyAsync(buf.data() + q * L.plane, h->d_macro + q * h->node_total + L.node_off,
                          L.plane * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  CK(h, cudaStreamSynchronize(h->stream));
  s = check_device_error(h);
  if (s != LBCG_OK) return s;
  for (int y = 0; y < L.ny; ++y)
    for (int x = 0; x < L.nx; ++x) {
      const size_t k = (size_t)y * L.pitch + x, i = (size_t)y * L.nx + x;
      const bool solid = L.solid[i] != 0;
      const double r = buf[k], b = buf[L.plane + k];
      host_out[i] = solid ? 0.0 : r + b;
      host_out[nn + i] = solid ? 0.0 : (r - b) / (r + b);
      host_out[2 * nn + i] = solid ? 0.0 : buf[2 * L.plane + k];
      host_out[3 * nn + i] = solid ? 0.0 : buf[3 * L.plane + k];
    }
  return LBCG_OK;
}

size_t lbcg_state_bytes(const lbcg_handle* h) {
  return h ? 18 * (size_t)h->node_total * elem_size(h->prec) : 0;
}

lbcg_status lbcg_upload_state(lbcg_handle* h, const void* host_in, size_t bytes) {
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (!host_in || bytes != lbcg_state_bytes(h)) return fail(LBCG_E_ARG, "state size mismatch");
  CK(h, cudaMemcpyAsync(h->pool[h->cur], host_in, bytes, cudaMemcpyHostToDevice, h->stream));
  return LBCG_OK;
}

lbcg_status lbcg_download_state(lbcg_handle* h, void* host_out, size_t bytes) {
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (!host_out || bytes != lbcg_state_bytes(h)) return fail(LBCG_E_ARG, "state size mismatch");
  CK(h, cudaMemcpyAsync(host_out, h->pool[h->cur], bytes, cudaMemcpyDeviceToHost, h->stream));
  return finish_stream(h);
}

lbcg_status lbcg_step_host(lbcg_handle* h, const void* host_in, void* host_out, size_t bytes, int64_t nsteps) {
  Range range_("lbcg_step_host");
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (!host_in || !host_out || bytes != lbcg_state_bytes(h)) return fail(LBCG_E_ARG, "state size mismatch");
  if (nsteps < 0) return fail(LBCG_E_ARG, "nsteps < 0");
  // groups of consecutive lattices: each is uploaded, stepped and downloaded on its own, the
  // uploads one after another on one stream, the steps on the handle's stream as each upload
  // lands, the downloads on a third stream as each group's steps end
  int end[kHostGroups + 1];
  const int ng = split_lattices(h, kHostGroups, end);
  for (int q = 0; q < 2; ++q)
    if (!h->io_stream[q]) CK(h, cudaStreamCreateWithFlags(&h->io_stream[q], cudaStreamNonBlocking));
  while (h->io_events.size() < size_t(2 * kHostGroups + 1)) {
    cudaEvent_t e;
    CK(h, cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    h->io_events.push_back(e);
  }
  cudaEvent_t* const ev_in = h->io_events.data();
  cudaEvent_t* const ev_done = ev_in + kHostGroups;
  const cudaEvent_t ev_start = ev_in[2 * kHostGroups];
  const int n = int(h->lats.size());
  const size_t es = elem_size(h->prec);
  auto off = [&](int l) { return size_t(l < n ? h->lats[l].pop_off : 18 * h->node_total) * es; };
  const int c0 = h->cur, c1 = h->cur ^ int(nsteps & 1);   // the pools of the state before and after
  const char* in = static_cast<const char*>(host_in);
  char* out = static_cast<char*>(host_out);
  CK(h, cudaEventRecord(ev_start, h->stream));   // after the work already on the handle's stream
  CK(h, cudaStreamWaitEvent(h->io_stream[0], ev_start, 0));
  for (int g = 0; g < ng; ++g) {
    CK(h, cudaMemcpyAsync(static_cast<char*>(h->pool[c0]) + off(end[g]), in + off(end[g]), off(end[g + 1]) - off(end[g]),
                          cudaMemcpyHostToDevice, h->io_stream[0]));
    CK(h, cudaEventRecord(ev_in[g], h->io_stream[0]));
  }
  for (int g = 0; g < ng; ++g) {
    CK(h, cudaStreamWaitEvent(h->stream, ev_in[g], 0));
    for (int64_t k = 0; k < nsteps; ++k) {
      LaunchStep p = ng > 1 ? make_launch_lats(h, c0 ^ int(k & 1), end[g], end[g + 1])
                            : make_launch(h, c0 ^ int(k & 1), nullptr, 0, h->ntiles);
      p.sr_step = uint32_t(h->step + k);
      CK(h, launch_step(h->prec, p, h->stream));
      h->step_launches += step_kernels(p);
    }
    CK(h, cudaEventRecord(ev_done[g], h->stream));
  }
  for (int g = 0; g < ng; ++g) {
    CK(h, cudaStreamWaitEvent(h->io_stream[1], ev_done[g], 0));
    CK(h, cudaMemcpyAsync(out + off(end[g]), static_cast<const char*>(h->pool[c1]) + off(end[g]),
                          off(end[g + 1]) - off(end[g]), cudaMemcpyDeviceToHost, h->io_stream[1]));
  }
  CK(h, cudaStreamSynchronize(h->io_stream[1]));
  CK(h, cudaStreamSynchronize(h->stream));
  h->cur = c1;
  h->step += nsteps;
  return check_device_error(h);
}

}  // extern "C"

namespace {

// device buffers of one adjoint run (from the handle's allocator), freed on every exit path
struct AdjBuffers {
  const lbcg_handle* h;
  std::vector<void*> ptrs;
  explicit AdjBuffers(const lbcg_handle* h_) : h(h_) {}
  ~AdjBuffers() {
    if (!ptrs.empty()) cudaStreamSynchronize(h->stream);
    for (void* p : ptrs) dev_free(h, p);
  }
  template <typename P>
  bool get(P** p, size_t bytes) {
    void* q = nullptr;
    if (!dev_alloc(h, &q, bytes)) return false;
    ptrs.push_back(q);
    *p = static_cast<P*>(q);
    return true;
  }
};

// d(first rho^N >= 0 -> < 0 change along profile p)/d p at the two nodes of the crossing
bool crossing_derivative(const std::vector<double>& prof, int& i0, double& x, double& d0, double& d1) {
  for (int i = 0; i + 1 < int(prof.size()); ++i)
    if (prof[i] >= 0 && prof[i + 1] < 0) {
      const double a = prof[i], b = prof[i + 1], den = a - b;
      i0 = i;
      x = i + a / den;
      d0 = -b / (den * den);
      d1 = a / (den * den);
      return true;
    }
  return false;
}

}  // namespace

namespace {

// lbcg_adjoint with the reverse kernels in arithmetic R (double or float)
template <typename R>
lbcg_status adjoint_run(lbcg_handle* h, const lbcg_adjoint_spec* spec, lbcg_grads* out) {
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (!spec || !out) return fail(LBCG_E_ARG, "NULL spec or output");
  if (h->prec != LBCG_FP64 && h->prec != LBCG_FP32)
    return fail(LBCG_E_UNSUPPORTED, "the adjoint runs on FP64 or FP32 handles");
  if (h->lats.size() != 1) return fail(LBCG_E_UNSUPPORTED, "the adjoint runs on single-lattice handles");
  if (h->lats[0].prm.wetting != 0) return fail(LBCG_E_UNSUPPORTED, "the adjoint differentiates wetting scheme (a) only");
  if (spec->nsteps < 1 || spec->checkpoint < 1) return fail(LBCG_E_ARG, "nsteps and checkpoint must be >= 1");
  if (spec->objective == LBCG_OBJ_WEIGHTED && !spec->weight) return fail(LBCG_E_ARG, "weighted objective needs weight");
  if (spec->objective != LBCG_OBJ_WEIGHTED && spec->objective != LBCG_OBJ_FINGER_LENGTH &&
      spec->objective != LBCG_OBJ_RED_MASS)
    return fail(LBCG_E_ARG, "unknown objective %d", spec->objective);
  const LatHost& L = h->lats[0];
  const int nx = L.nx, ny = L.ny, N = nx * ny;
  const int64_t T = spec->nsteps, K = spec->checkpoint;
  const int64_t nseg = (T + K - 1) / K;
  const size_t sb = lbcg_state_bytes(h);
  AdjBuffers B(h);
  constexpr size_t r8 = sizeof(R);
  double *ckpt, *pwork;
  double* segs[2];   // the states of two checkpoint segments: one recomputed while the other is reversed
  void* wall2;       // the recompute's own wall-kernel output (it may run beside the forward pass)
  R *lamA, *lamB, *work, *c_dev;
  R *nsx, *nsy, *ct, *st;
  int *pick0, *pick1;
  uint8_t *sol, *nbm;
  // N-sized arrays in R.  Two sets of forward intermediates and scatter targets (a reverse
  // step computes the intermediates of the state before it): fr, fb, rr/rb/rn, gr, gc, n, dn,
  // lnt, lrnt; one set of reverse arrays: lf_r, lf_b, ln, lg, lrn.  In double: the 4
  // parameter adjoints.
  const int kFwd = 9 + 9 + 3 + 2 + 2 + 2 + 4 + 2 + 1;
  const int kRev = 9 + 9 + 2 + 2 + 1;
  const int kWork = 2 * kFwd + kRev;
  if (!B.get(&ckpt, sb * (size_t)nseg) || !B.get(&segs[0], sb * (size_t)K) || !B.get(&segs[1], sb * (size_t)K) ||
      !B.get(&wall2, 4 * (size_t)h->node_total * compute_size(h->prec)) || !B.get(&lamA, 18 * (size_t)N * r8) ||
      !B.get(&lamB, 18 * (size_t)N * r8) || !B.get(&work, (size_t)kWork * N * r8) ||
      !B.get(&pwork, 4 * (size_t)N * 8) || !B.get(&c_dev, (size_t)N * r8) || !B.get(&nsx, (size_t)N * r8) ||
      !B.get(&nsy, (size_t)N * r8) || !B.get(&ct, (size_t)N * r8) || !B.get(&st, (size_t)N * r8) ||
      !B.get(&pick0, (size_t)N * 4) || !B.get(&pick1, (size_t)N * 4) || !B.get(&sol, (size_t)N) ||
      !B.get(&nbm, (size_t)N))
    return fail(LBCG_E_NOMEM, "adjoint buffers (%lld checkpoints of %zu bytes)", (long long)nseg, sb);
  // compact solid flags and solid-neighbour masks of every node (the stencils' neighbour rule)
  {
    std::vector<uint8_t> so(N), mk(N);
    const bool px = L.bcx == LBCG_BCX_PERIODIC, py = L.bcy == LBCG_BCY_PERIODIC;
    for (int y = 0; y < ny; ++y)
      for (int x = 0; x < nx; ++x) {
        uint8_t m = 0;
        for (int a = 1; a < 9; ++a)
          if (L.solid[(size_t)wrap_clamp(y + EYH[a], ny, py) * nx + wrap_clamp(x + EXH[a], nx, px)])
            m |= uint8_t(1u << (a - 1));
        so[(size_t)y * nx + x] = L.solid[(size_t)y * nx + x] ? 1 : 0;
        mk[(size_t)y * nx + x] = m;
      }
    CK(h, cudaMemcpy(sol, so.data(), N, cudaMemcpyHostToDevice));
    CK(h, cudaMemcpy(nbm, mk.data(), N, cudaMemcpyHostToDevice));
  }
  // compact normals and angles of the outermost fluid nodes
  {
    std::vector<R> a(N, R(0)), b(N, R(0)), c(N, R(1)), d(N, R(0));
    for (const OfbEntry& e : h->ofb_host) {
      const int i = e.y * nx + e.x;
      a[i] = R(e.nsx);
      b[i] = R(e.nsy);
      c[i] = R(e.cos_t);
      d[i] = R(e.sin_t);
    }
    CK(h, cudaMemcpy(nsx, a.data(), N * r8, cudaMemcpyHostToDevice));
    CK(h, cudaMemcpy(nsy, b.data(), N * r8, cudaMemcpyHostToDevice));
    CK(h, cudaMemcpy(ct, c.data(), N * r8, cudaMemcpyHostToDevice));
    CK(h, cudaMemcpy(st, d.data(), N * r8, cudaMemcpyHostToDevice));
  }
  CK(h, cudaMemsetAsync(work, 0, (size_t)kWork * N * r8, h->stream));
  CK(h, cudaMemsetAsync(pwork, 0, 4 * (size_t)N * 8, h->stream));
  AdjDevT<R> A{};
  {
    LatDev ld;
    CK(h, cudaMemcpy(&ld, h->d_lats, sizeof(LatDev), cudaMemcpyDeviceToHost));
    ld.pop_off = 0;  // the adjoint reads states from its own buffers
    A.L = ld;
    const LatConst<double> c = ld.consts<double>();
    A.C = LatConst<R>{R(c.sigma),   R(c.beta),     R(c.s_e),       R(c.s_eps),     R(c.s_q),        R(c.rho0), R(c.u_in),
                      R(c.rho_out), R(c.grad_eps), R(c.h_inv_nuR), R(c.h_inv_nuB), R(c.cos_theta)};
  }
  A.N = A.M = N;
  A.flags = h->d_flags;
  A.sol = sol;
  A.nbm = nbm;
  A.src_fp32 = h->prec == LBCG_FP32 ? 1 : 0;
  // FP32 states or FP32 reverse arithmetic: pure phases carry |grad rho^N| ~ 1e-7 of rounding noise
  A.n_eps = (h->prec == LBCG_FP32 || sizeof(R) == 4) ? std::max(1e-5, L.prm.grad_eps) : L.prm.grad_eps;
  A.nsx = nsx;
  A.nsy = nsy;
  A.cos_t = ct;
  A.sin_t = st;
  R* w = work;
  auto take = [&](int n) {
    R* p = w;
    w += (size_t)n * N;
    return p;
  };
  A.lf_r = take(9);
  A.lf_b = take(9);
  A.ln_x = take(1);
  A.ln_y = take(1);
  A.lg_x = take(1);
  A.lg_y = take(1);
  A.lrn = take(1);
  // the two sets of forward intermediates: view(0) and view(1) differ only in them
  AdjDevT<R> V[2];
  for (int q = 0; q < 2; ++q) {
    V[q] = A;
    V[q].pick = q ? pick1 : pick0;
    V[q].fr = take(9);
    V[q].fb = take(9);
    V[q].rr = take(1);
    V[q].rb = take(1);
    V[q].rn = take(1);
    V[q].grx = take(1);
    V[q].gry = take(1);
    V[q].gcx = take(1);
    V[q].gcy = take(1);
    V[q].nxv = take(1);
    V[q].nyv = take(1);
    V[q].dn = take(4);
    V[q].lnt_x = take(1);
    V[q].lnt_y = take(1);
    V[q].lrnt = take(1);
  }
  A.p_sigma = pwork;
  A.p_hR = pwork + N;
  A.p_hB = pwork + 2 * (size_t)N;
  A.p_theta = pwork + 3 * (size_t)N;
  for (int q = 0; q < 2; ++q) {
    V[q].p_sigma = A.p_sigma;
    V[q].p_hR = A.p_hR;
    V[q].p_hB = A.p_hB;
    V[q].p_theta = A.p_theta;
  }
  // ---- recompute and reverse on two streams.  The states of checkpoint segment k (its
  // checkpoint, then K - 1 steps) depend only on checkpoint k, so a side stream recomputes
  // segment k - 1 into one of two state buffers while the handle's stream reverses segment k
  // from the other; ready[b] marks segs[b] recomputed, done[b] its reverse finished.  The
  // recompute writes its own wall-kernel output (wall2), so that the last segment's recompute
  // can also run beside the forward steps.  Each segment's launches are captured once per
  // (kind, length, buffer, adjoint buffer parity) as a CUDA graph and replayed.
  struct Side {
    cudaStream_t st = nullptr;
    cudaEvent_t ev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};   // ready[2], done[2], checkpoints taken
    ~Side() {
      if (st) {
        cudaStreamSynchronize(st);
        cudaStreamDestroy(st);
      }
      for (cudaEvent_t e : ev)
        if (e) cudaEventDestroy(e);
    }
  } side;
  CK(h, cudaStreamCreateWithFlags(&side.st, cudaStreamNonBlocking));
  for (cudaEvent_t& e : side.ev) CK(h, cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  cudaEvent_t* const ready = side.ev;
  cudaEvent_t* const done = side.ev + 2;
  const cudaEvent_t ck_taken = side.ev[4];
  struct SegGraph {
    int kind;   // 0: recompute, 1: reverse
    int64_t ns;
    int buf;
    bool lam_in_a;
    cudaGraphExec_t exec;
  };
  struct SegGraphs {
    std::vector<SegGraph> v;
    ~SegGraphs() {
      for (SegGraph& g : v) cudaGraphExecDestroy(g.exec);
    }
  } graphs;
  R* const lam_a = lamA;
  R* const lam_b = lamB;
  // the recompute as launches of the resident kernel, where the handle steps with it: its own
  // progress words, since it may run beside the forward steps
  // (progress2), and likewise the reverse sweep of a segment (progress3) where its blocks of
  // rev_threads threads fit
  unsigned *progress2 = nullptr, *progress3 = nullptr;
  unsigned base2 = 0, base3 = 0;
  int rev_threads = 0;
  bool resident = !h->sweep && h->run_tiles > 0 && h->poll_limit == kPollLimit && !h->profiling;
  const size_t pb = size_t(h->run_tiles) * kRunFlagStride * sizeof(unsigned);
  if (resident && (!B.get(&progress2, pb) || !B.get(&progress3, pb)))
    resident = false;   // without memory for the words: the launched stages
  if (resident) {
    CK(h, cudaMemsetAsync(progress2, 0, pb, h->stream));
    CK(h, cudaMemsetAsync(progress3, 0, pb, h->stream));
    rev_threads = 2 * ((h->run_nodes + 31) / 32 * 32);
    int dev = 0, sms = 0, per_sm = 0;
    CK(h, cudaGetDevice(&dev));
    CK(h, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (rev_threads <= kRevMaxThreads && h->run_slots <= kRevMaxSlots) CK(h, reverse_blocks<R>(rev_threads, &per_sm));
    if ((long long)per_sm * sms < h->run_tiles) rev_threads = 0;
  }
  auto enqueue_recompute = [&](int64_t ns, int b) -> cudaError_t {
    for (int64_t j = 1; j < ns; ++j) {
      LaunchStep p = make_launch(h, 0, nullptr, 0, h->ntiles);
      p.src = reinterpret_cast<char*>(segs[b]) + sb * (j - 1);
      p.dst = reinterpret_cast<char*>(segs[b]) + sb * j;
      p.wall = wall2;
      const cudaError_t e = launch_step(h->prec, p, side.st);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  };
  // reverse of one segment: the intermediates of its last state, then per reverse step those of
  // the state before it, in the other set
  auto enqueue_reverse = [&](int64_t ns, bool lam_in_a, int b) -> cudaError_t {
    R* lc = lam_in_a ? lam_a : lam_b;
    R* ln = lam_in_a ? lam_b : lam_a;
    int q = 0;
    AdjDevT<R> cur = V[q];
    cur.src = reinterpret_cast<char*>(segs[b]) + sb * (ns - 1);
    cudaError_t e = adjoint_forward<R>(cur, h->stream);
    if (e != cudaSuccess) return e;
    for (int64_t j = ns - 1; j >= 0; --j) {
      cur = V[q];
      cur.src = reinterpret_cast<char*>(segs[b]) + sb * j;
      cur.lam_next = lc;
      cur.lam = ln;
      if (j > 0) {
        AdjDevT<R> prev = V[q ^ 1];
        prev.src = reinterpret_cast<char*>(segs[b]) + sb * (j - 1);
        e = adjoint_step<R>(cur, &prev, h->stream);
      } else {
        e = adjoint_step<R>(cur, nullptr, h->stream);
      }
      if (e != cudaSuccess) return e;
      std::swap(lc, ln);
      q ^= 1;
    }
    return cudaSuccess;
  };
  auto replay = [&](int kind, int64_t ns, int b, bool lam_in_a, cudaStream_t st) -> lbcg_status {
    cudaGraphExec_t exec = nullptr;
    for (const SegGraph& g : graphs.v)
      if (g.kind == kind && g.ns == ns && g.buf == b && g.lam_in_a == lam_in_a) exec = g.exec;
    if (!exec) {
      cudaGraph_t g = nullptr;
      CK(h, cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
      const cudaError_t le = kind == 0 ? enqueue_recompute(ns, b) : enqueue_reverse(ns, lam_in_a, b);
      const cudaError_t ee = cudaStreamEndCapture(st, &g);
      if (le != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        return cuda_fail(h, le, "adjoint launch during capture");
      }
      if (ee != cudaSuccess) return cuda_fail(h, ee, "cudaStreamEndCapture (adjoint)");
      const cudaError_t ie = cudaGraphInstantiate(&exec, g, 0);
      cudaGraphDestroy(g);
      if (ie != cudaSuccess) return cuda_fail(h, ie, "cudaGraphInstantiate (adjoint)");
      graphs.v.push_back({kind, ns, b, lam_in_a, exec});
    }
    CK(h, cudaGraphLaunch(exec, st));
    return LBCG_OK;
  };
  // the states of segment k into segs[k & 1], on the side stream, once that buffer's previous
  // segment is reversed
  auto start_recompute = [&](int64_t k) -> lbcg_status {
    const int b = int(k & 1);
    const int64_t ns = std::min<int64_t>(K, T - k * K);
    CK(h, cudaStreamWaitEvent(side.st, done[b], 0));
    CK(h, cudaMemcpyAsync(segs[b], reinterpret_cast<char*>(ckpt) + sb * k, sb, cudaMemcpyDeviceToDevice, side.st));
    if (ns > 1 && resident) {
      for (int64_t j = 0; j < ns - 1;) {
        RunArgs a = h->run;
        a.pool0 = reinterpret_cast<char*>(segs[b]) + sb * j;
        a.stride = (long long)sb;
        a.nsteps = int(std::min<int64_t>(ns - 1 - j, kRunMaxSteps));
        a.poll_limit = h->run_polls;
        a.progress = progress2;
        a.base = base2;
        base2 += unsigned(a.nsteps);
        CK(h, launch_run(h->prec, a, h->run_tiles, h->run_threads, h->run_smem, side.st));
        j += a.nsteps;
      }
    } else if (ns > 1) {
      const lbcg_status r = replay(0, ns, b, false, side.st);
      if (r != LBCG_OK) return r;
    }
    CK(h, cudaEventRecord(ready[b], side.st));
    return LBCG_OK;
  };
  for (int b = 0; b < 2; ++b)   // the slots the push never writes
    CK(h, cudaMemsetAsync(segs[b], 0, sb * (size_t)K, h->stream));
  // ---- forward with checkpoints (the handle ends at step T); the last segment's recompute
  // starts beside its forward steps
  for (int64_t k = 0; k < nseg; ++k) {
    CK(h, cudaMemcpyAsync(reinterpret_cast<char*>(ckpt) + sb * k, h->pool[h->cur], sb, cudaMemcpyDeviceToDevice,
                          h->stream));
    if (k == nseg - 1) {
      CK(h, cudaEventRecord(ck_taken, h->stream));
      CK(h, cudaStreamWaitEvent(side.st, ck_taken, 0));
      s = start_recompute(k);
      if (s != LBCG_OK) return s;
    }
    s = lbcg_step(h, std::min<int64_t>(K, T - k * K));
    if (s != LBCG_OK) return s;
  }
  // ---- objective and its seed dJ/d(rho^N) at step T
  std::vector<double> fields(4 * (size_t)N), cw(N, 0.0);
  s = lbcg_get_fields(h, 0, fields.data());
  if (s != LBCG_OK) return s;
  const double* rhoN = fields.data() + N;
  double J = 0.0;
  if (spec->objective == LBCG_OBJ_RED_MASS) {
    const double* rho = fields.data();
    for (int i = 0; i < N; ++i)
      if (!L.solid[i]) J += 0.5 * rho[i] * (1.0 + rhoN[i]);
  } else if (spec->objective == LBCG_OBJ_WEIGHTED) {
    for (int i = 0; i < N; ++i)
      if (!L.solid[i]) {
        cw[i] = spec->weight[i];
        J += cw[i] * rhoN[i];
      }
  } else {
    auto row_ok = [&](int r) { return r >= 0 && r < ny; };
    const int r0 = spec->tip_row0, r1 = spec->tip_row1;
    if (!row_ok(r0) || !row_ok(r1)) return fail(LBCG_E_ARG, "tip rows outside the lattice");
    std::vector<double> prof(nx);
    for (int x = 0; x < nx; ++x) prof[x] = 0.5 * (rhoN[r0 * nx + x] + rhoN[r1 * nx + x]);
    int i0;
    double xt, d0, d1;
    if (!crossing_derivative(prof, i0, xt, d0, d1)) return fail(LBCG_E_ARG, "no finger tip at step T");
    J = xt;
    cw[r0 * nx + i0] += 0.5 * d0;
    cw[r1 * nx + i0] += 0.5 * d0;
    cw[r0 * nx + i0 + 1] += 0.5 * d1;
    cw[r1 * nx + i0 + 1] += 0.5 * d1;
    const int rows[2] = {spec->cl_row0, spec->cl_row1};
    std::vector<std::pair<int, double>> cl;
    double xsum = 0;
    int found = 0;
    std::vector<int> ii(2);
    std::vector<double> dd0(2), dd1(2);
    for (int q = 0; q < 2; ++q) {
      if (!row_ok(rows[q])) continue;
      for (int x = 0; x < nx; ++x) prof[x] = rhoN[rows[q] * nx + x];
      double xc;
      if (crossing_derivative(prof, ii[found], xc, dd0[found], dd1[found])) {
        xsum += xc;
        ii[found] = ii[found] + rows[q] * nx;  // node index of the crossing
        ++found;
      }
    }
    if (found == 0) return fail(LBCG_E_ARG, "no contact line at step T");
    J -= xsum / found;
    for (int q = 0; q < found; ++q) {
      cw[ii[q]] -= dd0[q] / found;
      cw[ii[q] + 1] -= dd1[q] / found;
    }
  }
  {
    std::vector<R> cr(cw.begin(), cw.end());
    CK(h, cudaMemcpy(c_dev, cr.data(), N * r8, cudaMemcpyHostToDevice));
  }
  AdjDevT<R> S0 = V[0];
  S0.src = h->pool[h->cur];
  S0.lam = lamA;
  CK(h, adjoint_seed<R>(S0, c_dev, spec->objective == LBCG_OBJ_RED_MASS, h->stream));
  // ---- reverse, one checkpoint segment at a time, each beside the recompute of the next
  bool lam_in_a = true;   // the seed is in lamA
  for (int64_t k = nseg - 1; k >= 0; --k) {
    const int b = int(k & 1);
    const int64_t ns = std::min<int64_t>(K, T - k * K);
    if (k >= 1) {
      s = start_recompute(k - 1);
      if (s != LBCG_OK) return s;
    }
    CK(h, cudaStreamWaitEvent(h->stream, ready[b], 0));
    if (rev_threads > 0) {
      RevRunT<R> P{};
      P.V[0] = V[0];
      P.V[1] = V[1];
      P.tiles = h->run.tiles;
      P.nb = h->run.nb;
      P.progress = progress3;
      P.base = base3;
      P.err = h->d_err;
      P.poll_limit = h->run_polls;
      P.states = reinterpret_cast<const char*>(segs[b]);
      P.stride = (long long)sb;
      P.ns = int(ns);
      P.lam_next = lam_in_a ? lam_a : lam_b;
      P.lam = lam_in_a ? lam_b : lam_a;
      base3 += unsigned(3 * ns + 1);
      CK(h, launch_reverse<R>(P, h->run_tiles, rev_threads, h->stream));
    } else {
      s = replay(1, ns, b, lam_in_a, h->stream);
      if (s != LBCG_OK) return s;
    }
    CK(h, cudaEventRecord(done[b], h->stream));
    if (ns & 1) lam_in_a = !lam_in_a;
  }
  // ---- parameter adjoints
  std::vector<double> ps(N), phR(N), phB(N), pth(N);
  CK(h, cudaMemcpyAsync(ps.data(), A.p_sigma, N * 8, cudaMemcpyDeviceToHost, h->stream));
  CK(h, cudaMemcpyAsync(phR.data(), A.p_hR, N * 8, cudaMemcpyDeviceToHost, h->stream));
  CK(h, cudaMemcpyAsync(phB.data(), A.p_hB, N * 8, cudaMemcpyDeviceToHost, h->stream));
  CK(h, cudaMemcpyAsync(pth.data(), A.p_theta, N * 8, cudaMemcpyDeviceToHost, h->stream));
  CK(h, cudaStreamSynchronize(h->stream));
  s = check_device_error(h);
  if (s != LBCG_OK) return s;
  double gs = 0, ghR = 0, ghB = 0, gth = 0;
  for (int i = 0; i < N; ++i) {
    gs += ps[i];
    ghR += phR[i];
    ghB += phB[i];
    gth += pth[i];
  }
  out->J = J;
  out->dJ_dsigma = gs;
  out->dJ_dnu_R = ghR * (-0.5 / (L.prm.nu_R * L.prm.nu_R));
  out->dJ_dnu_B = ghB * (-0.5 / (L.prm.nu_B * L.prm.nu_B));
  out->dJ_dtheta = gth;
  if (out->dJ_dtheta_node) memcpy(out->dJ_dtheta_node, pth.data(), N * 8);
  return LBCG_OK;
}

}  // namespace

extern "C" {

lbcg_status lbcg_adjoint(lbcg_handle* h, const lbcg_adjoint_spec* spec, lbcg_grads* out) {
  Range range_("lbcg_adjoint");
  const lbcg_status s = spec && spec->reverse_fp32 ? adjoint_run<float>(h, spec, out) : adjoint_run<double>(h, spec, out);
  // a wait of the second stream may have run out too after the word was read and cleared; both
  // streams are idle now: reported once
  if (s == LBCG_E_TIMEOUT || s == LBCG_E_BOUNDS) CK(h, cudaMemsetAsync(h->d_err, 0, sizeof(int), h->stream));
  return s;
}

lbcg_status lbcg_set_sweep(lbcg_handle* h, int32_t rows) {
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (rows < 0) return fail(LBCG_E_ARG, "rows per strip segment must be >= 0");
  CK(h, cudaStreamSynchronize(h->stream));
  h->sweep = 1;
  h->sweep_rows = rows;
  if (h->graph) {
    cudaGraphExecDestroy(h->graph);
    h->graph = nullptr;
  }
  return upload_tiles(h);
}

lbcg_status lbcg_set_poll_limit(lbcg_handle* h, int32_t polls) {
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (polls < 0) polls = kPollLimit;
  CK(h, cudaStreamSynchronize(h->stream));
  h->poll_limit = polls;
  if (h->graph) {
    cudaGraphExecDestroy(h->graph);
    h->graph = nullptr;
  }
  return LBCG_OK;
}

lbcg_status lbcg_set_tile_poll_limit(lbcg_handle* h, int32_t polls) {
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  CK(h, cudaStreamSynchronize(h->stream));
  h->run_polls = polls < 0 ? kPollLimit : polls;
  return LBCG_OK;
}

lbcg_status lbcg_set_tile(lbcg_handle* h, int32_t ty) {
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (ty == 0) ty = kDefaultTY;
  if (ty != 4 && ty != 8 && ty != 16) return fail(LBCG_E_ARG, "tile height must be 4, 8 or 16");
  CK(h, cudaStreamSynchronize(h->stream));
  h->ty = ty;
  h->sweep = 0;
  if (h->graph) {
    cudaGraphExecDestroy(h->graph);
    h->graph = nullptr;
  }
  s = upload_tiles(h);
  return s == LBCG_OK ? plan_run(h) : s;
}

lbcg_status lbcg_autotune(lbcg_handle* h, int32_t probe_steps, int32_t* schedule) {
  Range range_("lbcg_autotune");
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (probe_steps < 1) return fail(LBCG_E_ARG, "probe_steps must be >= 1");
  if (h->profiling) return fail(LBCG_E_ARG, "switch profiling off before autotuning");
  CK(h, cudaStreamSynchronize(h->stream));
  if (h->graph) {
    cudaGraphExecDestroy(h->graph);
    h->graph = nullptr;
  }
  // the y-sweep at the automatic segment height and at fixed heights, then the tiles; each
  // timed as what lbcg_step replays: a captured graph of probe_steps steps (with a batch's
  // parallel branches), whose steps all rewrite the same next state; last the tiles as one launch
  // of the resident kernel
  struct Cand {
    int sweep, ty, rows;
  };
  const Cand cand[] = {{1, h->ty, 0}, {1, h->ty, 24}, {1, h->ty, 32}, {1, h->ty, 40}, {1, h->ty, 48},
                       {1, h->ty, 56}, {1, h->ty, 64}, {1, h->ty, 80}, {0, 4, 0},      {0, 8, 0},
                       {0, 16, 0}};
  const int ncand = int(sizeof(cand) / sizeof(cand[0]));
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  CK(h, cudaEventCreate(&e0));
  cudaError_t e = cudaEventCreate(&e1);
  int best = 0, best_tile = -1;
  float best_ms = 0.f, tile_ms = 0.f;
  for (int c = 0; c < ncand && e == cudaSuccess; ++c) {
    h->sweep = cand[c].sweep;
    h->ty = cand[c].ty;
    h->sweep_rows = cand[c].rows;
    s = upload_tiles(h);
    if (s != LBCG_OK) break;
    cudaGraphExec_t gx = nullptr;
    int64_t nk = 0;
    s = capture_steps(h, probe_steps, true, &gx, &nk);
    if (s != LBCG_OK) break;
    e = cudaGraphLaunch(gx, h->stream);   // first replay: uploads the graph, warms the caches
    if (e == cudaSuccess) e = cudaEventRecord(e0, h->stream);
    if (e == cudaSuccess) e = cudaGraphLaunch(gx, h->stream);
    if (e == cudaSuccess) e = cudaEventRecord(e1, h->stream);
    if (e == cudaSuccess) e = cudaEventSynchronize(e1);
    cudaGraphExecDestroy(gx);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (e == cudaSuccess && (c == 0 || ms < best_ms)) {
      best = c;
      best_ms = ms;
    }
    if (e == cudaSuccess && !cand[c].sweep && (best_tile < 0 || ms < tile_ms)) {
      best_tile = c;
      tile_ms = ms;
    }
  }
  // the tile schedule's resident kernel, where lbcg_step would take it: it advances the state, which
  // is saved and put back
  if (e == cudaSuccess && s == LBCG_OK) s = plan_run(h);
  if (e == cudaSuccess && s == LBCG_OK && h->run_tiles > 0 && h->poll_limit == kPollLimit) {
    const size_t sb = lbcg_state_bytes(h);
    void* keep[2] = {nullptr, nullptr};
    if (dev_alloc(h, &keep[0], sb) && dev_alloc(h, &keep[1], sb)) {
      const int n = std::max(probe_steps, kGraphSteps + 1);
      for (int q = 0; q < 2 && e == cudaSuccess; ++q)
        e = cudaMemcpyAsync(keep[q], h->pool[q], sb, cudaMemcpyDeviceToDevice, h->stream);
      RunArgs a = h->run;
      a.pool0 = static_cast<char*>(h->pool[h->cur]);
      a.pool1 = static_cast<char*>(h->pool[h->cur ^ 1]);
      a.nsteps = n;
      a.poll_limit = h->run_polls;
      for (int q = 0; q < 2 && e == cudaSuccess; ++q) {
        if (q) e = cudaEventRecord(e0, h->stream);
        a.base = h->run_base;
        h->run_base += unsigned(n);
        if (e == cudaSuccess) e = launch_run(h->prec, a, h->run_tiles, h->run_threads, h->run_smem, h->stream);
      }
      if (e == cudaSuccess) e = cudaEventRecord(e1, h->stream);
      for (int q = 0; q < 2 && e == cudaSuccess; ++q)
        e = cudaMemcpyAsync(h->pool[q], keep[q], sb, cudaMemcpyDeviceToDevice, h->stream);
      if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
      float ms = 0.f;
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
      if (e == cudaSuccess && ms / n < best_ms / probe_steps) best = best_tile;
    }
    for (void* q : keep) dev_free(h, q);
  }
  cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (e != cudaSuccess) return cuda_fail(h, e, "autotune probe");
  if (s != LBCG_OK) return s;
  h->sweep = cand[best].sweep;
  h->ty = cand[best].ty;
  h->sweep_rows = cand[best].rows;
  s = upload_tiles(h);
  if (s != LBCG_OK) return s;
  if (schedule) *schedule = h->sweep ? 0 : h->ty;
  return LBCG_OK;
}

lbcg_status lbcg_schedule(const lbcg_handle* h, int32_t* schedule) {
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (!schedule) return fail(LBCG_E_ARG, "NULL schedule");
  *schedule = h->sweep ? 0 : h->ty;
  return LBCG_OK;
}

int32_t lbcg_sweep_rows(const lbcg_handle* h) { return h ? h->sweep_rows : -1; }

lbcg_status lbcg_profile(lbcg_handle* h, int32_t enable) {
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  CK(h, cudaStreamSynchronize(h->stream));
  h->profiling = enable != 0;
  h->events_used = 0;
  h->prof_steps = 0;
  h->prof_ref_set = false;
  return LBCG_OK;
}

lbcg_status lbcg_kernel_times(lbcg_handle* h, double* ms2, int64_t* steps) {
  lbcg_status s = check_handle(h);
  if (s != LBCG_OK) return s;
  if (!ms2 || !steps) return fail(LBCG_E_ARG, "NULL output");
  CK(h, cudaStreamSynchronize(h->stream));
  ms2[0] = ms2[1] = 0.0;
  // per kernel kind, the length of the union of its launches' event intervals (the time at
  // least one of them ran: branches of a batch overlap; one branch gives the plain sum)
  for (int k = 0; k < 2; ++k) {
    std::vector<std::pair<float, float>> iv;
    for (size_t i = 0; i + 4 <= h->events_used; i += 4) {
      float t0 = 0.f, t1 = 0.f;
      CK(h, cudaEventElapsedTime(&t0, h->prof_ref, h->events[i + 2 * k]));
      CK(h, cudaEventElapsedTime(&t1, h->prof_ref, h->events[i + 2 * k + 1]));
      iv.emplace_back(t0, t1);
    }
    std::sort(iv.begin(), iv.end());
    double total = 0.0, a = 0.0, b = -1e30;
    for (const auto& q : iv) {
      if (q.first > b) {
        if (b > a) total += b - a;
        a = q.first;
        b = q.second;
      } else if (q.second > b) {
        b = q.second;
      }
    }
    if (b > a) total += b - a;
    ms2[k] = total;
  }
  *steps = h->prof_steps;
  h->events_used = 0;
  h->prof_steps = 0;
  h->prof_ref_set = false;
  return LBCG_OK;
}

int32_t lbcg_launches_per_step(const lbcg_handle* h) {
  if (!h) return 0;
  return (h->ngroups > 0 ? 1 : 0) + ((h->sweep ? h->nstrips : h->ntiles) > 0 ? 1 : 0);
}

int64_t lbcg_step_launches(const lbcg_handle* h) { return h ? h->step_launches : 0; }

int64_t lbcg_total_nodes(const lbcg_handle* h) {
  if (!h) return 0;
  int64_t n = 0;
  for (const LatHost& L : h->lats) n += (int64_t)L.nx * L.ny;
  return n;
}

lbcg_status lbcg_destroy(lbcg_handle* h) {
  if (!h) return LBCG_OK;
  if (h->stream) cudaStreamSynchronize(h->stream);
  free_handle(h);
  return LBCG_OK;
}

}  // extern "C"
