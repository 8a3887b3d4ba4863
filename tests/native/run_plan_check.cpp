// Checks the plan of the resident step kernel (lbcg_plan.h) on the host: every fluid node has one
// owner; every node a tile reads is written by the tile itself or by tiles it waits for; waiting is
// mutual; every table entry names the node it stands for and lies inside the tile's arrays.
#include <cstdio>
#include <cstdlib>
#include <random>
#include <set>

#include "lbcg_plan.h"

using namespace lbcg;

static void require(bool ok, const char* what) {
  if (!ok) {
    std::printf("FAILED: %s\n", what);
    std::exit(1);
  }
}

struct Box {
  int nx, ny, bcx, bcy;
  std::vector<uint8_t> solid;
};

static Box make(int nx, int ny, int bcx, int bcy, unsigned seed, double porous) {
  Box b{nx, ny, bcx, bcy, std::vector<uint8_t>(size_t(nx) * ny, 0)};
  std::mt19937 rng(seed);
  std::uniform_real_distribution<double> u(0, 1);
  for (auto& s : b.solid) s = u(rng) < porous;
  for (int y = 0; y < ny; ++y)
    if (bcx == 1) b.solid[size_t(y) * nx] = b.solid[size_t(y) * nx + nx - 1] = 1;
  for (int x = 0; x < nx; ++x)
    if (bcy == 1) b.solid[x] = b.solid[size_t(ny - 1) * nx + x] = 1;
  return b;
}

static void check(const std::vector<Box>& boxes, int max_tiles, size_t cs) {
  std::vector<OfbEntry> ofb;
  std::vector<std::vector<uint8_t>> flags;
  std::vector<LatGeom> lats;
  std::vector<const uint8_t*> fp;
  int l = 0;
  for (const Box& b : boxes) {
    const std::vector<double> r(b.solid.size(), 0.0);
    lbcg_geometry g{b.nx, b.ny, b.bcx, b.bcy, b.solid.data(), r.data(), nullptr, nullptr};
    lbcg_params p{};
    p.theta = 1.0;
    std::vector<uint8_t> f, m;
    classify(&g, &p, l++, f, m, ofb);
    const int pitch = (b.nx + 31) / 32 * 32;
    std::vector<uint8_t> padded(size_t(pitch) * b.ny, F_SOLID);
    for (int y = 0; y < b.ny; ++y)
      for (int x = 0; x < b.nx; ++x) padded[size_t(y) * pitch + x] = f[size_t(y) * b.nx + x];
    flags.push_back(padded);
    lats.push_back(LatGeom{b.nx, b.ny, pitch, b.bcx, b.bcy, b.solid.data()});
  }
  for (auto& f : flags) fp.push_back(f.data());
  RunPlan plan;
  const size_t budget = 230000;
  require(build_run_plan(lats, fp, ofb, max_tiles, budget, cs, plan), "the lattices fit");
  require(int(plan.tiles.size()) <= max_tiles && plan.smem <= budget, "tiles and shared memory within the limits");
  // owners
  std::vector<std::vector<int>> owner;
  for (const Box& b : boxes) owner.emplace_back(b.solid.size(), -1);
  for (size_t k = 0; k < plan.tiles.size(); ++k) {
    const RunTile& t = plan.tiles[k];
    require(t.tx >= 1 && t.ty >= 1 && t.tx <= kRunMaxSide && t.ty <= kRunMaxSide, "tile sides");
    require(run_smem_bytes(t, cs) <= plan.smem, "the plan's shared memory covers the tile");
    for (int y = t.y0; y < t.y0 + t.ty; ++y)
      for (int x = t.x0; x < t.x0 + t.tx; ++x) {
        int& o = owner[t.lat][size_t(y) * boxes[t.lat].nx + x];
        require(o == -1, "one owner per node");
        o = int(k);
      }
  }
  for (size_t b = 0; b < boxes.size(); ++b)
    for (size_t i = 0; i < boxes[b].solid.size(); ++i)
      require(boxes[b].solid[i] || owner[b][i] >= 0, "every fluid node is owned");
  for (size_t k = 0; k < plan.tiles.size(); ++k) {
    const RunTile& t = plan.tiles[k];
    const Box& b = boxes[t.lat];
    const bool px = b.bcx == 0, py = b.bcy == 0;
    std::set<int> nb(plan.nb.begin() + t.nb0, plan.nb.begin() + t.nb0 + t.nnb);
    for (int q : nb) {
      require(q >= 0 && q < int(plan.tiles.size()) && q != int(k) && plan.tiles[q].lat == t.lat, "neighbour index");
      const RunTile& o = plan.tiles[q];
      bool mutual = false;
      for (int j = 0; j < o.nnb; ++j) mutual = mutual || plan.nb[o.nb0 + j] == int(k);
      require(mutual, "waiting is mutual");
    }
    auto node = [&](int x, int y) { return wrap_clamp(y, b.ny, py) * b.nx + wrap_clamp(x, b.nx, px); };
    const int cw = t.tx + 4, nd = cw * (t.ty + 4), nr = nd + t.ne;
    std::vector<int> at;   // node of each slot
    for (int cy = 0; cy < t.ty + 4; ++cy)
      for (int cx = 0; cx < cw; ++cx) at.push_back(node(t.x0 + cx - 2, t.y0 + cy - 2));
    for (int i = 0; i < t.ne; ++i) {
      const int n = plan.extra[t.extra0 + i];
      require(n >= 0 && n < b.nx * b.ny && !b.solid[n], "extra slots are fluid nodes");
      at.push_back(n);
    }
    auto known = [&](int q) { return q == int(k) || nb.count(q); };
    for (int n : at) {
      if (b.solid[n]) continue;
      // the node's populations are written by itself and its fluid neighbours
      for (int a = 0; a < 9; ++a) {
        const int x = n % b.nx - EXH[a], y = n / b.nx - EYH[a];
        if ((!px && (x < 0 || x >= b.nx)) || (!py && (y < 0 || y >= b.ny))) continue;
        const int w = node(x, y);
        require(b.solid[w] || known(owner[t.lat][w]), "a tile waits for every writer of what it reads");
      }
    }
    // what it writes (its own nodes and their neighbours) is read only by itself and by tiles it waits for:
    // mutual waiting turns the check above into this one
    auto of_w = [&](int w) {
      require(w >= 0 && w < t.nw, "index in w");
      const OfbEntry& e = ofb[plan.w_ofb[t.w0 + w]];
      require(e.lat == t.lat, "outermost fluid node of the same lattice");
      return e.y * b.nx + e.x;
    };
    std::set<int> band(plan.band.begin() + t.band0, plan.band.begin() + t.band0 + t.nband);
    require(int(band.size()) == t.nband && (band.empty() || *band.rbegin() < nr), "band slots");
    std::vector<int> virt(t.nv, -1);
    for (int w = 0; w < t.nw; ++w) {
      const int n = of_w(w);
      for (int a = 1; a < 9; ++a) {
        const int m = node(n % b.nx + EXH[a], n / b.nx + EYH[a]);
        const int i = plan.w_sten[t.w0 + w].i[a - 1];
        require(i < t.nband + t.nv, "stencil index");
        if (b.solid[m]) {
          const int j = i - t.nband;
          require(j >= 0, "a solid neighbour is a virtual node");
          require(virt[j] == -1 || virt[j] == m, "one virtual node per index");
          virt[j] = m;
        } else {
          require(i < t.nband && at[plan.band[t.band0 + i]] == m, "a fluid neighbour's slot");
        }
      }
    }
    for (int v = 0; v < t.nv; ++v) {
      require(virt[v] >= 0, "every virtual node is read");
      for (int a = 1; a < 9; ++a) {
        const int m = node(virt[v] % b.nx + EXH[a], virt[v] / b.nx + EYH[a]);
        const int i = plan.v_sten[t.v0 + v].i[a - 1];
        require(b.solid[m] ? i == kWallNone : (i < t.nband && at[plan.band[t.band0 + i]] == m),
                "a virtual node's neighbours");
      }
    }
    const int pw = t.tx + 2, np = pw * (t.ty + 2);
    std::set<int> placed;
    for (int i = 0; i < t.ncopy; ++i) {
      const uint32_t c = plan.copies[t.copy0 + i];
      const int pos = c & 0xFFFF;
      require(pos < np && placed.insert(pos).second, "position of an outermost fluid node");
      require(of_w(c >> 16) == node(t.x0 + pos % pw - 1, t.y0 + pos / pw - 1), "the position's node");
    }
    for (int i = 0; i < t.nvn; ++i) {
      const RunVirtN& v = plan.vn[t.vn0 + i];
      require(int(v.pos) < np && placed.insert(int(v.pos)).second, "position of an outermost solid node");
      const int n = node(t.x0 + int(v.pos) % pw - 1, t.y0 + int(v.pos) / pw - 1);
      for (int a = 1; a < 9; ++a) {
        const int m = node(n % b.nx + EXH[a], n / b.nx + EYH[a]);
        require(b.solid[m] ? v.w[a - 1] == kWallNone : of_w(v.w[a - 1]) == m, "a virtual normal's neighbours");
      }
    }
    for (int pos = 0; pos < np; ++pos) {
      const int xr = t.x0 + pos % pw - 1, yr = t.y0 + pos / pw - 1;
      const int n = node(xr, yr);
      const uint8_t f = flags[t.lat][size_t(n / b.nx) * lats[t.lat].pitch + n % b.nx];
      require(placed.count(pos) == ((f & (F_OFB | F_OSOLID)) != 0), "every wall position is placed");
      if (!(f & (F_SOLID | F_OFB))) {
        // a bulk position is evaluated at the slot of the node it stands for, inside the dense slots
        const int sx = px ? pos % pw : pos % pw + n % b.nx - xr, sy = py ? pos / pw : pos / pw + n / b.nx - yr;
        const int c = (sy + 1) * cw + sx + 1;
        require(sx >= 0 && sx < pw && sy >= 0 && sy < t.ty + 2, "a ghost position's source");
        for (int a = 0; a < 9; ++a) {
          const int i = c + EYH[a] * cw + EXH[a];
          require(i >= 0 && i < nd && at[i] == node(n % b.nx + EXH[a], n / b.nx + EYH[a]), "a bulk stencil");
        }
      }
    }
  }
  std::printf("%zu lattices, first %d x %d: %zu tiles, %zu bytes\n", boxes.size(), boxes[0].nx, boxes[0].ny,
              plan.tiles.size(), plan.smem);
}

int main() {
  unsigned seed = 1;
  const int sizes[][2] = {{5, 5}, {7, 6}, {48, 20}, {100, 50}, {33, 40}, {200, 31}, {631, 60}, {61, 200}};
  for (auto& s : sizes)
    for (int bcx = 0; bcx < 3; ++bcx)
      for (int bcy = 0; bcy < 2; ++bcy)
        for (double porous : {0.0, 0.05, 0.4})
          for (int tiles : {1, 7, 152}) {
            if (tiles == 1 && s[0] * s[1] > 1000) continue;
            if (tiles == 7 && s[0] * s[1] > 6000) continue;
            check({make(s[0], s[1], bcx, bcy, seed++, porous)}, tiles, tiles == 7 ? 8 : 4);
          }
  check({make(2000, 102, 2, 1, 1, 0.0)}, 152, 4);
  check({make(1200, 80, 0, 0, 1, 0.0)}, 152, 8);
  check({make(40, 22, 2, 1, 3, 0.0), make(33, 40, 0, 0, 4, 0.1), make(5, 5, 1, 1, 5, 0.0)}, 152, 8);
  std::vector<Box> study;
  for (int i = 0; i < 8; ++i) study.push_back(make(630, 60, 2, 1, 1, 0.0));
  check(study, 152, 4);
  std::printf("ALL OK\n");
  return 0;
}
