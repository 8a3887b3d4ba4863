// The resident step kernel: many time steps of the colour-gradient LBM (arXiv 1707.00198,
// Sec. II) in one cooperative launch.
//
// A lattice of the paper's sizes (5 k to 0.3 M nodes) is far too small to keep the GPU busy:
// with one launch per kernel and step, a step lasts as long as two grids' launches, their
// chains of dependent loads and the flushes between them, whatever its arithmetic.  Here the
// lattices are cut into one tile per block, at most as many as the GPU holds at a time, and a
// block stays on its SM for all the steps of the call.  Per step it waits until the tiles
// around it have finished the step before (one flag per tile, no grid-wide barrier), evaluates
// its own wall nodes (the chain of Eq. 28-36 that the launch-per-step schedule gives to a kernel
// of its own) beside its bulk nodes, and pushes.  What does not change between steps is
// resolved once per launch into tables in shared memory: the population offset of every slot,
// the row and column offsets of every push, the wall stencils.
//
// The arithmetic of a node is that of k_wall and k_step (lbcg_node.cuh), so that a call may mix
// the two without a change of bits.
//
// What bounds it: on the smallest lattices the chain of one step (a flag's round trip through
// L2, about 3300 cycles with the release of the stores before it, then the loads, the wall chain and
// the collision of one pass); on the larger ones instruction issue; in FP64 the FP64 pipe.  Per step,
// launch per kernel -> resident: 100 x 50 FP64 26.5 -> 12.6 us, 1200 x 80 FP64 72 -> 35.5, FP32 10.5 ->
// 5.3, 2000 x 102 FP32 17.3 -> 9.4, FP16 18.6 -> 9.3, 8 x 630 x 60 FP32 with Poiseuille inlets 36 -> 12.8
// (18.4 with the inlet profile evaluated, in FP64, at every read of an edge node).  FP32 arithmetic:
// two blocks of 256 threads per SM, whose waits overlap each other's work, against one of 512:
// 2000 x 102 FP32 9.4 -> 9.1, FP16 9.3 -> 8.7, 8 x 630 x 60 12.8 -> 11.8; with the push offsets of
// bulk nodes apart from those of wall nodes 8.7, 8.5 and 11.3.  FP64 with one reciprocal square root
// per node in the wall chain (lbcg_node.cuh): 100 x 50 12.6 -> 10.6 us, 1200 x 80 35.5 -> 35.4,
// 2000 x 102 123 -> 111 (9.9, 34.6 and 111 with the divisions of rho^N and of Eq. 29 also reciprocals,
// which decides near ties of Eq. 36 otherwise than the equations' own operations).
#include "lbcg_internal.h"
#include "lbcg_node.cuh"
#include "lbcg_wait.cuh"

namespace lbcg {

namespace {

// Populations are read past L1 (.cg): the tile's halo was written by other SMs one step ago.
template <typename S>
__device__ __forceinline__ void load_pair_cg(const S* p, typename Store<S>::T& lo, typename Store<S>::T& hi) {
  if constexpr (sizeof(S) == 8) {
    asm volatile("ld.global.cg.v2.f64 {%0, %1}, [%2];" : "=d"(lo), "=d"(hi) : "l"(p));
  } else if constexpr (sizeof(S) == 4) {
    asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(lo), "=f"(hi) : "l"(p));
  } else {
    uint32_t w;
    asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(w) : "l"(p));
    Store<S>::unpack(w, lo, hi);
  }
}

__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// slot table entry: own index in the low half (0xFFFF: not of the tile), and
constexpr uint32_t kSlotEdge = 1u << 17;     // in an open column: Zou-He on every read
constexpr uint32_t kSlotOutlet = 1u << 18;   // and that column is the outlet
constexpr int kSlotRow = 20;                 // its row in the table of inlet velocities, from this bit
// own-node table entry: neighbour-solid mask, column and row in the tile (from bits 16 and 24), and
constexpr uint32_t kOwnSolid = 1u << 8, kOwnEdge = 1u << 9, kOwnOfb = 1u << 10;
constexpr uint16_t kNone = 0xFFFF;   // no entry (of a position in the bulk, of a slot in the band)


template <typename T>
__device__ __forceinline__ T* carve(unsigned char*& p, size_t n) {
  T* q = reinterpret_cast<T*>(p);
  p += (n * sizeof(T) + 15) & ~size_t(15);
  return q;
}

template <typename S, int NT>
__global__ void __launch_bounds__(NT, run_blocks(sizeof(typename Store<S>::T))) k_run(RunArgs A) {
  using T = typename Store<S>::T;
  constexpr int kWallTeam = NT / 2;   // threads that evaluate a tile's wall nodes beside its bulk nodes
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ LatDev sL;
  const RunTile tl = A.tiles[blockIdx.x];
  const int t = threadIdx.x;
  if (t == 0) sL = A.lats[tl.lat];
  const int CW = tl.tx + 4, PW = tl.tx + 2;
  const int ND = CW * (tl.ty + 4), NR = ND + tl.ne, NP = PW * (tl.ty + 2), NO = tl.tx * tl.ty;
  unsigned char* sp = smem;
  T* const srn = carve<T>(sp, NR);             // rho^N of the slots
  T* const swv = carve<T>(sp, tl.nband + tl.nv);   // the wall chain's rho^N: band slots, then virtual nodes
  T* const snx = carve<T>(sp, NP);             // n and gradient on tile + 1
  T* const sny = carve<T>(sp, NP);
  T* const sgx = carve<T>(sp, NP);
  T* const sgy = carve<T>(sp, NP);
  // own nodes: the totals f_a (FP64: replaced by their moments and s_v), rho_R, rho_B, 1 / rho
  T* const sf = carve<T>(sp, size_t(12) * NO);
  T* const sw = carve<T>(sp, size_t(8) * tl.nw);       // wall nodes: the candidates of Eq. 34; gradient, n
  T* const sden = carve<T>(sp, tl.nv + tl.nvn);        // virtual nodes: the weight (of rho^N), mean_factor (of n)
  int* const r_off = carve<int>(sp, NR);
  uint32_t* const r_tab = carve<uint32_t>(sp, NR);
  uint16_t* const r_band = carve<uint16_t>(sp, NR);
  T* const s_u = carve<T>(sp, tl.ty + 8);
  uint16_t* const p_src = carve<uint16_t>(sp, NP);
  uint32_t* const o_tab = carve<uint32_t>(sp, NO);
  int* const colk = carve<int>(sp, PW);
  int* const rowk = carve<int>(sp, tl.ty + 2);
  WallSten* const w_sten = carve<WallSten>(sp, tl.nw);
  WallSten* const v_sten = carve<WallSten>(sp, tl.nv);
  RunVirtN* const vn = carve<RunVirtN>(sp, tl.nvn);
  uint32_t* const copies = carve<uint32_t>(sp, tl.ncopy);
  __syncthreads();
  const int nx = sL.nx, ny = sL.ny, pitch = sL.pitch;
  const bool px = sL.bcx == BC_PERIODIC, py = sL.bcy == BC_PERIODIC, inout = sL.bcx == BC_INOUT;
  const LatConst<T> C = sL.consts<T>();
  const Collide<T> K(C);
  const T eps2 = rmul(C.grad_eps, C.grad_eps);
  // (in registers: read from shared memory in every step, 2000 x 102 FP16 8.36 us per step, for 8.33)
  const int wetting = sL.wetting;
  const bool unit = sL.unit_normals;
  const uint8_t* __restrict__ fl = A.flags + sL.node_off;
  const uint8_t* __restrict__ nbm = A.nbmask + sL.node_off;
  const long long pop_off = sL.pop_off, pop_n = 18 * sL.plane;

  // ---- tables
  for (int i = t; i < NR; i += NT) {
    int x, y;
    uint32_t own = 0xFFFFu;
    if (i < ND) {
      const int cx = i % CW, cy = i / CW;
      x = wrap_or_clamp(tl.x0 + cx - 2, nx, px);
      y = wrap_or_clamp(tl.y0 + cy - 2, ny, py);
      if (cx >= 2 && cx < tl.tx + 2 && cy >= 2 && cy < tl.ty + 2)
        own = uint32_t((cy - 2) * tl.tx + cx - 2);
    } else {
      const int node = A.extra[tl.extra0 + i - ND];
      x = node % nx;
      y = node / nx;
    }
    const bool solid = fl[(long long)y * pitch + x] & F_SOLID;
    uint32_t tab = own;
    if (inout && (x == 0 || x == nx - 1)) {
      int row = y - (tl.y0 - 4);   // the slots' rows are y0 - 4 .. y0 + ty + 3
      if (row < 0) row += ny;
      if (row >= tl.ty + 8) row -= ny;
      tab |= kSlotEdge | (x == 0 ? 0u : kSlotOutlet) | uint32_t(row) << kSlotRow;
    }
    r_off[i] = solid ? -1 : pop_node(x, y, pitch);
    r_tab[i] = tab;
    r_band[i] = kNone;
    srn[i] = T(0);
  }
  for (int i = t; i < tl.ty + 8; i += NT) s_u[i] = inlet_u<T>(sL, wrap_or_clamp(tl.y0 - 4 + i, ny, py));
  for (int i = t; i < NP; i += NT) {
    const int cx = i % PW, cy = i / PW;
    // a position beyond a non-periodic edge is a ghost copy of the edge node (zero normal
    // gradient): it is evaluated at the slot of the node it copies
    const int xr = tl.x0 + cx - 1, yr = tl.y0 + cy - 1;
    const int x = wrap_or_clamp(xr, nx, px), y = wrap_or_clamp(yr, ny, py);
    const int sx = px ? cx : cx + x - xr, sy = py ? cy : cy + y - yr;
    const uint8_t f = fl[(long long)y * pitch + x];
    p_src[i] = (f & (F_SOLID | F_OFB)) ? kNone : uint16_t((sy + 1) * CW + sx + 1);
    snx[i] = sny[i] = sgx[i] = sgy[i] = T(0);
  }
  for (int i = t; i < NO; i += NT) {
    const int lx = i % tl.tx, ly = i / tl.tx;
    const long long k = (long long)(tl.y0 + ly) * pitch + tl.x0 + lx;
    const uint8_t f = fl[k];
    o_tab[i] = uint32_t(nbm[k]) | (f & F_SOLID ? kOwnSolid : 0u) | (f & F_EDGE ? kOwnEdge : 0u) |
               (f & F_OFB ? kOwnOfb : 0u) | uint32_t(lx) << 16 | uint32_t(ly) << 24;
  }
  for (int i = t; i < PW; i += NT) {
    const int x = wrap_or_clamp(tl.x0 + i - 1, nx, px);
    colk[i] = (x >> 5) * kSeg + (x & 31) * 2;
  }
  for (int i = t; i < tl.ty + 2; i += NT) rowk[i] = wrap_or_clamp(tl.y0 + i - 1, ny, py) * ((pitch >> 5) * kSeg);
  for (int i = t; i < tl.nw; i += NT) {
    const OfbEntry e = A.ofb[A.w_ofb[tl.w0 + i]];
    wall_candidates<T>(T(e.nsx), T(e.nsy), T(e.cos_t), T(e.sin_t), sw[i], sw[tl.nw + i], sw[2 * tl.nw + i],
                       sw[3 * tl.nw + i]);
    w_sten[i] = A.w_sten[tl.w0 + i];
  }
  for (int i = t; i < tl.nv; i += NT) {
    v_sten[i] = A.v_sten[tl.v0 + i];
    sden[i] = virtual_weight<T>(v_sten[i].i);
  }
  for (int i = t; i < tl.nvn; i += NT) {
    vn[i] = A.vn[tl.vn0 + i];
    sden[tl.nv + i] = mean_factor(virtual_weight<T>(vn[i].w));
  }
  for (int i = t; i < tl.ncopy; i += NT) copies[i] = A.copies[tl.copy0 + i];
  __syncthreads();
  for (int i = t; i < tl.nband; i += NT) r_band[A.band[tl.band0 + i]] = uint16_t(i);
  // the tile's wall nodes have threads of their own beside the bulk nodes' (when it has any)
  const bool walls = tl.nw > 0;
  const int team = walls ? NT - kWallTeam : NT;
  uint32_t epoch0 = 0;
  if constexpr (Store<S>::kDeviation) epoch0 = *A.sr_epoch;
  __syncthreads();

  for (int s = 0; s < A.nsteps; ++s) {
    // ---- the tiles around this one have finished the step before: what this step reads is
    // written, and what it will overwrite has been read
    bool lost = false;
    if (s > 0) {
      const unsigned want = A.base + unsigned(s);
      for (int j = t; j < tl.nnb && !lost; j += NT)
        lost = !wait_reached(A.progress + A.nb[tl.nb0 + j] * kRunFlagStride, want, A.poll_limit, A.err);
    }
    if (__syncthreads_or(lost)) {
      if (t == 0) atomicOr(A.err, ERR_TIMEOUT);
      return;
    }
    const S* const src = reinterpret_cast<const S*>(A.state(s)) + pop_off;
    S* const dst = reinterpret_cast<S*>(A.state(s + 1)) + pop_off;
    uint32_t srk = 0;
    if constexpr (Store<S>::kDeviation) srk = A.key(epoch0, s, pop_off);

    // ---- rho^N on the tile + 2 and on the band of its wall nodes; the own nodes' totals
    for (int i = t; i < NR; i += NT) {
      const int off = r_off[i];
      if (off < 0 || !checked(in_extent(off, 8 * kDir + 2, pop_n), A.err)) continue;
      const uint32_t tab = r_tab[i];
      T fr[9], fb[9];
#pragma unroll
      for (int a = 0; a < 9; ++a) load_pair_cg<S>(src + off + a * kDir, fr[a], fb[a]);
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        const T lo = fr[a], hi = fb[a];
        decode<S, T>(lo, hi, wgt<T>(a) * C.rho0, fr[a], fb[a]);
      }
      if (tab & kSlotEdge) zou_he<T>(tab & kSlotOutlet ? nx - 1 : 0, nx, s_u[tab >> kSlotRow], C.rho_out, fr, fb);
      T rhoR, rhoB, irho;
      srn[i] = indicator(fr, fb, rhoR, rhoB, irho);
      const uint32_t own = tab & 0xFFFFu;
      if (own != 0xFFFFu) {
#pragma unroll
        for (int a = 0; a < 9; ++a) sf[a * NO + own] = radd(fr[a], fb[a]);
        sf[9 * NO + own] = rhoR;
        sf[10 * NO + own] = rhoB;
        sf[11 * NO + own] = irho;
      }
      const uint32_t band = r_band[i];
      if (band != kNone) swv[band] = rdiv(rsub(rhoR, rhoB), radd(rhoR, rhoB));   // as k_wall rounds it
    }
    __syncthreads();
    // ---- gradient and n of the bulk nodes of tile + 1, beside the wall chain (Eq. 28-36)
    if (t < team) {
      for (int i = t; i < NP; i += team) {
        const uint32_t c = p_src[i];
        if (c == kNone) continue;
        T ax, ay, nxv, nyv;
        grad_normal<T>(srn + c, CW, eps2, ax, ay, nxv, nyv);
        sgx[i] = ax;
        sgy[i] = ay;
        snx[i] = nxv;
        sny[i] = nyv;
      }
      if constexpr (sizeof(T) == 8) {
        // what the collision needs of the totals alone, while the wall chain runs
        for (int i = t; i < NO; i += team) {
          const uint32_t e = o_tab[i];
          if (e & kOwnSolid) continue;
          T f[9];
#pragma unroll
          for (int a = 0; a < 9; ++a) f[a] = sf[a * NO + i];
          const int c = ((e >> 24) + 2) * CW + ((e >> 16) & 0xFFu) + 2;
          Moments<T> m;
          m.of(f);
          relax_rest(m, radd(sf[9 * NO + i], sf[10 * NO + i]), K);
          sf[i] = m.e;
          sf[NO + i] = m.eps;
          sf[2 * NO + i] = m.jx;
          sf[3 * NO + i] = m.jy;
          sf[4 * NO + i] = m.qx;
          sf[5 * NO + i] = m.qy;
          sf[6 * NO + i] = m.pxx;
          sf[7 * NO + i] = m.pxy;
          sf[8 * NO + i] = viscous_rate<T>(srn[c], K);
        }
      }
    } else {
      const int w = t - team;
      for (int j = w; j < tl.nv; j += kWallTeam)
        swv[tl.nband + j] = wetting == 2 ? C.cos_theta : virtual_value<T>(v_sten[j], swv, sden[j]);
      bar_sync(1, kWallTeam);
      for (int j0 = w & ~31; j0 < 2 * tl.nw; j0 += kWallTeam) {   // two lanes per node, whole warps
        const int j = min((j0 + (w & 31)) >> 1, tl.nw - 1), r = w & 1;
        T g, n;
        wall_normal_pair<T>(C.grad_eps, wetting, unit, sw[r * tl.nw + j], sw[(2 + r) * tl.nw + j],
                            sw[2 * r * tl.nw + j], sw[(2 * r + 1) * tl.nw + j], w_sten[j], swv, r, g, n);
        sw[(4 + r) * tl.nw + j] = g;   // (lanes past the end repeat the last node)
        sw[(6 + r) * tl.nw + j] = n;
      }
      bar_sync(1, kWallTeam);
      for (int j = w; j < tl.ncopy; j += kWallTeam) {
        const uint32_t c = copies[j], i = c & 0xFFFFu, k = c >> 16;
        sgx[i] = sw[4 * tl.nw + k];
        sgy[i] = sw[5 * tl.nw + k];
        snx[i] = sw[6 * tl.nw + k];
        sny[i] = sw[7 * tl.nw + k];
      }
      // virtual n on the outermost solid nodes (Eq. 29), a lane per component
      for (int j = w; j < 2 * tl.nvn; j += kWallTeam) {
        const RunVirtN& q = vn[j >> 1];
        const T* const wn = sw + (6 + (j & 1)) * tl.nw;
        T v = T(0);
#pragma unroll
        for (int b = 1; b < 9; ++b)
          if (q.w[b - 1] != kWallNone) v = fma_(wgt<T>(b), wn[q.w[b - 1]], v);
        (j & 1 ? sny : snx)[q.pos] = mean_of(v, sden[tl.nv + (j >> 1)]);
      }
    }
    __syncthreads();
    // ---- curvature, force, collision, recolouring, push
    for (int i = t; i < NO; i += NT) {
      const uint32_t e = o_tab[i];
      if (e & kOwnSolid) continue;
      const int lx = (e >> 16) & 0xFFu, ly = e >> 24, o1 = (ly + 1) * PW + lx + 1;
      const T rhoR = sf[9 * NO + i], rhoB = sf[10 * NO + i], irho = sf[11 * NO + i];
      T f[9], sv;
      Moments<T> m;
      if constexpr (sizeof(T) == 8) {
        m.e = sf[i];
        m.eps = sf[NO + i];
        m.jx = sf[2 * NO + i];
        m.jy = sf[3 * NO + i];
        m.qx = sf[4 * NO + i];
        m.qy = sf[5 * NO + i];
        m.pxx = sf[6 * NO + i];
        m.pxy = sf[7 * NO + i];
        sv = sf[8 * NO + i];
      } else {
#pragma unroll
        for (int a = 0; a < 9; ++a) f[a] = sf[a * NO + i];
        m.of(f);
        sv = viscous_rate<T>(srn[(ly + 2) * CW + lx + 2], K);
      }
      T dxx, dxy, dyx, dyy;
      grad_n<T>(snx + o1, sny + o1, PW, dxx, dyx, dxy, dyy);
      const unsigned mask = e & 0xFFu;
      if (wetting == 1 && (e & kOwnOfb)) {
        T nxs[9], nys[9];
#pragma unroll
        for (int a = 0; a < 9; ++a) {
          nxs[a] = snx[o1 + ey(a) * PW + ex(a)];
          nys[a] = sny[o1 + ey(a) * PW + ex(a)];
        }
        grad_n_scheme_b<T>(nxs, nys, mask, kStencilScale<T>, dxx, dyx, dxy, dyy);
      }
      const T nxo = snx[o1], nyo = sny[o1];
      T Fx, Fy;
      csf_force<T>(sgx[o1], sgy[o1], nxo, nyo, dxx, dyx, dxy, dyy, K, Fx, Fy);
      T fp[9];
      collide_node<T>(f, m, radd(rhoR, rhoB), irho, sv, Fx, Fy, K, fp);
      const Recolour<T> rc(rhoR, rhoB, irho, nxo, nyo, K);
      const int kn = rowk[ly + 1] + colk[lx + 1];
      uint32_t srh = 0;
      if constexpr (Store<S>::kDeviation) srh = sr_node(srk, kn);
      // streaming (Eq. 15): to x + e_a if that node is fluid; half-way bounce-back into the
      // opposite slot of this node if it is solid; dropped if it lies beyond an open edge
      int k[9];
#pragma unroll
      for (int a = 0; a < 9; ++a) k[a] = rowk[ly + 1 + ey(a)] + colk[lx + 1 + ex(a)] + a * kDir;
      if (e & (0xFFu | kOwnEdge)) {
#pragma unroll
        for (int a = 1; a < 9; ++a) {
          if (mask & (1u << (a - 1))) k[a] = kn + opp(a) * kDir;
          const int xr = tl.x0 + lx + ex(a);
          if ((e & kOwnEdge) && (xr < 0 || xr >= nx)) k[a] = -1;
        }
      }
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        if (a != 0 && k[a] < 0) continue;
        T oR, oB;
        rc.out(a, fp, oR, oB);
        if (checked(in_extent(k[a], 2, pop_n), A.err))
          store_pair_sr<S>(dst + k[a], oR, oB, wgt<T>(a) * C.rho0, sr_bits(srh, a));
      }
    }
    __syncthreads();
    if (t == 0) {
      // the release at GPU scope orders the whole block's stores, which the barrier puts before it;
      // a __threadfence ahead of it was a second trip to L2: 100 x 50 FP32 3.61 -> 3.28 us per step,
      // 1200 x 80 FP32 5.66 -> 5.38, 2000 x 102 FP32 9.0 -> 8.6, FP16 8.6 -> 8.3
      store_release(A.progress + blockIdx.x * kRunFlagStride, A.base + unsigned(s) + 1u);
    }
  }
}

__global__ void k_sr_add(uint32_t* epoch, uint32_t n) { *epoch += n; }

template <typename S>
cudaError_t launch(const RunArgs& a, int ntiles, int threads, size_t smem, cudaStream_t st) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;   // every block resident: they wait for one another
  at[0].val.cooperative = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(ntiles));
  cfg.blockDim = dim3(unsigned(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return threads == 128 ? cudaLaunchKernelEx(&cfg, k_run<S, 128>, a) : cudaLaunchKernelEx(&cfg, k_run<S, 256>, a);
}

template <typename K>
cudaError_t prepare_k(K* k, int threads, size_t smem, int* per_sm) {
  // the attribute belongs to the kernel, not to a handle: always the most a block can have, so
  // that a later handle with smaller tiles takes nothing from an earlier one
  cudaError_t e = allow_max_smem(k);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k, threads, smem);
  return e;
}
template <typename S>
cudaError_t prepare(int threads, size_t smem, int* per_sm) {
  return threads == 128 ? prepare_k(k_run<S, 128>, threads, smem, per_sm)
                        : prepare_k(k_run<S, 256>, threads, smem, per_sm);
}

}  // namespace

cudaError_t launch_run(int prec, const RunArgs& a, int ntiles, int threads, size_t smem, cudaStream_t st) {
  cudaError_t e = cudaErrorInvalidValue;
  switch (prec) {
    case 0: e = launch<double>(a, ntiles, threads, smem, st); break;
    case 1: e = launch<float>(a, ntiles, threads, smem, st); break;
    case 2: e = launch<__half>(a, ntiles, threads, smem, st); break;
    case 3: e = launch<__nv_bfloat16>(a, ntiles, threads, smem, st); break;
  }
  return e;
}

cudaError_t prepare_run(int prec, int threads, size_t smem, int* per_sm) {
  switch (prec) {
    case 0: return prepare<double>(threads, smem, per_sm);
    case 1: return prepare<float>(threads, smem, per_sm);
    case 2: return prepare<__half>(threads, smem, per_sm);
    case 3: return prepare<__nv_bfloat16>(threads, smem, per_sm);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_sr_add(uint32_t* epoch, uint32_t n, cudaStream_t st) {
  k_sr_add<<<1, 1, 0, st>>>(epoch, n);
  return cudaGetLastError();
}

}  // namespace lbcg
