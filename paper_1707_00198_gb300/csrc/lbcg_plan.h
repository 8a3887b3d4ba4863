// Plan of the resident step kernel (lbcg_run.cu): the cut of a handle's lattices into one tile
// per block, and the tables of the tiles' wall nodes.  Plain C++ (no CUDA types): the runtime and
// the kernel share these layouts, and the host tests build them without a GPU.
#pragma once

#include <stdint.h>

#include <vector>

#include "lbcg_geom.h"

namespace lbcg {

// A tile: nodes [x0, x0 + tx) x [y0, y0 + ty) of lattice `lat`, owned by one block.  The block
// evaluates rho^N on the tile plus 2 nodes all round (its dense slots, row-major, (tx + 4) per
// row) and on `ne` further nodes (extra slots, numbered after the dense ones) that the wall
// chain reads.  Ranges into the plan's lists:
//   nb     tiles that read what this one writes or write what it reads: those within
//          kRunReach nodes
//   extra  the extra slots' nodes (y * nx + x)
//   band   slots whose rho^N the wall chain reads
//   w      outermost fluid nodes whose corrected gradient the tile needs: index into the
//          outermost-fluid list, and where the wall chain has their 8 neighbours (index in band,
//          or, after those, the virtual nodes)
//   v      virtual (outermost solid) nodes of rho^N: the indices in band of their fluid neighbours
//   copy   positions of the n array (tile plus 1 node all round, row-major, (tx + 2) per row)
//          that hold an outermost fluid node: position, and its index in w
//   vn     positions that hold an outermost solid node: position, and the indices in w of its
//          fluid neighbours
struct RunTile {
  int lat, x0, y0, tx, ty;
  int nb0, nnb, extra0, ne, band0, nband, w0, nw, v0, nv, copy0, ncopy, vn0, nvn;
  int pad_;
};
struct RunVirtN {
  uint16_t w[8];   // index in w of the fluid neighbour in direction a (element a - 1), or kWallNone
  uint32_t pos;
  uint32_t pad_[3];
};
// A block reads at most 4 nodes beyond its tile (two stencils, and along walls the neighbours
// of the outermost fluid nodes next to a solid node of its halo), and a block writes at most 1
// node beyond its own.
constexpr int kRunReach = 5;
constexpr int kRunMaxSide = 250;   // nodes per tile side, at most

struct RunPlan {
  std::vector<RunTile> tiles;
  std::vector<int> nb, extra, w_ofb;
  std::vector<WallSten> w_sten, v_sten;
  std::vector<uint16_t> band;
  std::vector<uint32_t> copies;   // position | index in w << 16
  std::vector<RunVirtN> vn;
  size_t smem = 0;                // dynamic shared memory of the largest tile
};

// Blocks, i.e. tiles, per SM, at most, for `cs` bytes per value of the compute type.  FP32 arithmetic: two, so
// that one works while the other waits for its neighbours.  FP64: one, since the FP64 pipe is
// the bound and a tile half as large recomputes more of its halo.
LBCG_HD constexpr int run_blocks(size_t cs) { return cs == 4 ? 2 : 1; }
// A block of kRunSmallThreads threads, half of them beside the tile's wall nodes where it has any.
constexpr int kRunSmallThreads = 128;
// Whether such blocks take every stage of every tile in one pass, so that more threads would only idle.
bool run_one_pass(const RunPlan& plan);
// Dynamic shared memory of a tile: `cs` bytes per value of the compute type.
size_t run_smem_bytes(const RunTile& t, size_t cs);

// Cuts the lattices into at most max_tiles tiles (tiles without fluid nodes are dropped) whose
// shared memory fits in max_smem, with the largest tile's work as small as the search finds, and
// builds the wall tables.  flags: per lattice [ny][pitch] node flags; ofb: the outermost-fluid
// list of the whole handle, row-major within a lattice.  False if they do not fit.
bool build_run_plan(const std::vector<LatGeom>& lats, const std::vector<const uint8_t*>& flags,
                    const std::vector<OfbEntry>& ofb, int max_tiles, size_t max_smem, size_t cs, RunPlan& plan);

}  // namespace lbcg
