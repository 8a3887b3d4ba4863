// Plan of the resident step kernel (declarations in lbcg_plan.h).
#include "lbcg_plan.h"

#include <algorithm>
#include <cmath>

namespace lbcg {

size_t run_smem_bytes(const RunTile& t, size_t cs) {
  auto up = [](size_t b) { return (b + 15) & ~size_t(15); };
  const size_t nr = size_t(t.tx + 4) * (t.ty + 4) + t.ne, np = size_t(t.tx + 2) * (t.ty + 2);
  const size_t no = size_t(t.tx) * t.ty;
  return up(nr * cs) + up((size_t(t.nband) + t.nv) * cs) + 4 * up(np * cs) + up(12 * no * cs) +
         up(8 * size_t(t.nw) * cs) + up((size_t(t.nv) + t.nvn) * cs) + up(nr * 4) * 2 + up(nr * 2) +
         up((size_t(t.ty) + 8) * cs) + up(np * 2) + up(no * 4) + up((size_t(t.tx) + 2) * 4) +
         up((size_t(t.ty) + 2) * 4) + up(t.nw * sizeof(WallSten)) + up(t.nv * sizeof(WallSten)) +
         up(t.nvn * sizeof(RunVirtN)) + up(size_t(t.ncopy) * 4);
}

bool run_one_pass(const RunPlan& plan) {
  for (const RunTile& t : plan.tiles) {
    const int half = kRunSmallThreads / 2, team = t.nw > 0 ? half : kRunSmallThreads;
    if ((t.tx + 4) * (t.ty + 4) + t.ne > kRunSmallThreads || (t.tx + 2) * (t.ty + 2) > team) return false;
    if (t.nv > half || 2 * t.nw > half || 2 * t.nvn > half || t.ncopy > half) return false;
  }
  return true;
}

namespace {

// fluid nodes of a lattice in any rectangle, from a summed-area table
struct Area {
  int nx, ny;
  std::vector<int> s;   // [(ny + 1)][(nx + 1)]
  explicit Area(const LatGeom& L) : nx(L.nx), ny(L.ny), s(size_t(L.nx + 1) * (L.ny + 1), 0) {
    for (int y = 0; y < ny; ++y) {
      int row = 0;
      for (int x = 0; x < nx; ++x) {
        row += L.solid[size_t(y) * nx + x] == 0;
        s[size_t(y + 1) * (nx + 1) + x + 1] = s[size_t(y) * (nx + 1) + x + 1] + row;
      }
    }
  }
  int fluid(int x0, int y0, int x1, int y1) const {
    auto at = [&](int x, int y) { return s[size_t(y) * (nx + 1) + x]; };
    return at(x1, y1) - at(x0, y1) - at(x1, y0) + at(x0, y0);
  }
};

int cut(int n, int parts, int i) { return int((long long)n * i / parts); }

}  // namespace

bool build_run_plan(const std::vector<LatGeom>& lats, const std::vector<const uint8_t*>& flags,
                    const std::vector<OfbEntry>& ofb, int max_tiles, size_t max_smem, size_t cs, RunPlan& plan) {
  plan = RunPlan{};
  const int nl = int(lats.size());
  if (nl > max_tiles) return false;
  std::vector<Area> area;
  for (const LatGeom& L : lats) area.emplace_back(L);
  // ---- the cut.  For each tile width, the smallest height whose tiles are few enough; then
  // the pair whose largest tile costs least: a collision per own node, rho^N per halo slot
  // (whole 32-byte sectors of the population rows) and n per slot of the ring around it weigh
  // about 6 : 1.2 : 1 in both arithmetics' instructions
  auto columns = [](int n, int side) { return (n + side - 1) / side; };
  long long fluid = 0;
  int nxmax = 1, nymax = 1;
  for (int l = 0; l < nl; ++l) {
    nxmax = std::max(nxmax, lats[l].nx);
    nymax = std::max(nymax, lats[l].ny);
    fluid += area[l].fluid(0, 0, lats[l].nx, lats[l].ny);
  }
  // f(lattice, x0, y0, x1, y1, fluid nodes) on every tile that has any; false once f is
  auto each = [&](int tx, int ty, auto f) {
    for (int l = 0; l < nl; ++l) {
      const int gx = columns(lats[l].nx, tx), gy = columns(lats[l].ny, ty);
      for (int j = 0; j < gy; ++j) {
        const int y0 = cut(lats[l].ny, gy, j), y1 = cut(lats[l].ny, gy, j + 1);
        for (int i = 0, x0 = 0; i < gx; ++i) {
          const int x1 = cut(lats[l].nx, gx, i + 1);
          const int own = area[l].fluid(x0, y0, x1, y1);
          if (own && !f(l, x0, y0, x1, y1, own)) return false;
          x0 = x1;
        }
      }
    }
    return true;
  };
  auto few = [&](int tx, int ty) {
    int n = 0;
    return each(tx, ty, [&](int, int, int, int, int, int) { return ++n <= max_tiles; });
  };
  auto cost = [&](int tx, int ty, double limit) {   // of the largest tile; `limit` or more: not measured to the end
    double c = 0.0;
    each(tx, ty, [&](int l, int x0, int y0, int x1, int y1, int own) {
      const int hx0 = std::max(x0 - 2, 0), hy0 = std::max(y0 - 2, 0);
      const int hx1 = std::min(x1 + 2, lats[l].nx), hy1 = std::min(y1 + 2, lats[l].ny);
      const double halo = area[l].fluid(hx0, hy0, hx1, hy1) + 3.0 * (hy1 - hy0);
      c = std::max(c, 6.0 * own + 1.2 * halo + double(x1 - x0 + 2) * (y1 - y0 + 2));
      return c < limit;
    });
    return c;
  };
  int btx = 0, bty = 0;
  double best = 1e300;
  for (int tx = 4; tx <= std::min(kRunMaxSide, std::max(4, nxmax)); tx += tx < 16 ? 1 : (tx < 48 ? 2 : (tx < 96 ? 4 : 16))) {
    // a tile holds at most tx * ty fluid nodes: no height below lo can do
    const int top = std::min(kRunMaxSide, nymax);
    int lo = int(std::min<long long>(top, std::max<long long>(1, fluid / ((long long)max_tiles * tx))));
    int hi = std::min(top, lo + lo / 4 + 2);
    while (!few(tx, hi) && hi < top) {
      lo = hi + 1;
      hi = std::min(top, 2 * hi);
    }
    if (hi == top && !few(tx, hi)) continue;
    while (lo < hi) {
      const int mid = (lo + hi) / 2;
      if (few(tx, mid)) hi = mid;
      else lo = mid + 1;
    }
    const double c = cost(tx, lo, best);
    if (c < best) {
      best = c;
      btx = tx;
      bty = lo;
    }
  }
  if (btx == 0) return false;
  // ---- tiles, their neighbours and wall tables
  size_t first_ofb = 0;
  for (int l = 0; l < nl; ++l) {
    const LatGeom& L = lats[l];
    const int nx = L.nx, ny = L.ny;
    const bool px = L.bcx == 0, py = L.bcy == 0;
    const int gx = columns(nx, btx), gy = columns(ny, bty);
    auto solid = [&](int x, int y) { return L.solid[size_t(y) * nx + x] != 0; };
    // per node: its index in the outermost-fluid list; and for the tile in hand, its index in w
    // or among the virtual nodes (valid where the stamp is the tile's)
    std::vector<int> ofb_at(size_t(nx) * ny), local(size_t(nx) * ny), stamp(size_t(nx) * ny, -1);
    for (; first_ofb < ofb.size() && ofb[first_ofb].lat == l; ++first_ofb)
      ofb_at[ofb[first_ofb].y * nx + ofb[first_ofb].x] = int(first_ofb);
    std::vector<int> col(nx), row(ny), id(size_t(gx) * gy, -1);
    for (int i = 0; i < gx; ++i)
      for (int x = cut(nx, gx, i); x < cut(nx, gx, i + 1); ++x) col[x] = i;
    for (int j = 0; j < gy; ++j)
      for (int y = cut(ny, gy, j); y < cut(ny, gy, j + 1); ++y) row[y] = j;
    const size_t base = plan.tiles.size();
    for (int j = 0; j < gy; ++j)
      for (int i = 0; i < gx; ++i) {
        RunTile t{};
        t.lat = l;
        t.x0 = cut(nx, gx, i);
        t.y0 = cut(ny, gy, j);
        t.tx = cut(nx, gx, i + 1) - t.x0;
        t.ty = cut(ny, gy, j + 1) - t.y0;
        if (area[l].fluid(t.x0, t.y0, t.x0 + t.tx, t.y0 + t.ty) == 0) continue;
        id[size_t(j) * gx + i] = int(plan.tiles.size());
        plan.tiles.push_back(t);
      }
    std::vector<int> near, cols, rows;
    // the columns (rows) of tiles that hold a node within kRunReach of [a, b)
    auto reach = [&](int a, int b, int n, bool periodic, const std::vector<int>& of, std::vector<int>& out) {
      out.clear();
      for (int v = a - kRunReach; v < b + kRunReach; ++v) {
        if (!periodic && (v < 0 || v >= n)) continue;
        const int q = of[wrap_clamp(v, n, periodic)];
        if (out.empty() || out.back() != q) out.push_back(q);
        if (v == a) v = b - 1;   // inside [a, b) there is one
      }
      std::sort(out.begin(), out.end());
      out.erase(std::unique(out.begin(), out.end()), out.end());
    };
    for (size_t k = base; k < plan.tiles.size(); ++k) {
      RunTile& t = plan.tiles[k];
      near.clear();
      reach(t.x0, t.x0 + t.tx, nx, px, col, cols);
      reach(t.y0, t.y0 + t.ty, ny, py, row, rows);
      for (int j : rows)
        for (int i : cols) {
          const int q = id[size_t(j) * gx + i];
          if (q >= 0 && q != int(k)) near.push_back(q);
        }
      t.nb0 = int(plan.nb.size());
      t.nnb = int(near.size());
      plan.nb.insert(plan.nb.end(), near.begin(), near.end());
      // slots: the dense ones by position, the extra ones as they are asked for
      const int cw = t.tx + 4, ch = t.ty + 4, nd = cw * ch;
      std::vector<int> extra;                          // nodes of the extra slots
      std::vector<uint16_t> band_of(size_t(nd), kWallNone), band_of_extra;
      int nw = 0, nband = 0;
      t.extra0 = int(plan.extra.size());
      t.band0 = int(plan.band.size());
      t.w0 = int(plan.w_ofb.size());
      t.v0 = int(plan.v_sten.size());
      t.copy0 = int(plan.copies.size());
      t.vn0 = int(plan.vn.size());
      auto inside = [](int d, int n, bool periodic, int m) {
        if (d >= 0 && d < m) return d;
        if (periodic && d + n >= 0 && d + n < m) return d + n;
        if (periodic && d - n >= 0 && d - n < m) return d - n;
        return -1;
      };
      auto slot = [&](int x, int y) {   // of a fluid node of the lattice
        const int cx = inside(x - t.x0 + 2, nx, px, cw), cy = inside(y - t.y0 + 2, ny, py, ch);
        if (cx >= 0 && cy >= 0) return cy * cw + cx;
        const int node = y * nx + x;
        for (size_t i = 0; i < extra.size(); ++i)
          if (extra[i] == node) return nd + int(i);
        extra.push_back(node);
        band_of_extra.push_back(kWallNone);
        plan.extra.push_back(node);
        return nd + int(extra.size()) - 1;
      };
      auto in_band = [&](int x, int y) {
        const int i = slot(x, y);
        uint16_t& b = i < nd ? band_of[i] : band_of_extra[i - nd];
        if (b == kWallNone) {
          b = uint16_t(nband++);
          plan.band.push_back(uint16_t(i));
        }
        return b;
      };
      auto want_w = [&](int x, int y) {   // of an outermost fluid node of the lattice
        const size_t n = size_t(y) * nx + x;
        if (stamp[n] != int(k)) {
          stamp[n] = int(k);
          local[n] = nw++;
          plan.w_ofb.push_back(ofb_at[n]);
        }
        return local[n];
      };
      const uint8_t* fl = flags[l];
      for (int cy = 0; cy < t.ty + 2; ++cy) {
        const int y = wrap_clamp(t.y0 + cy - 1, ny, py);
        for (int cx = 0; cx < t.tx + 2; ++cx) {
          const int xr = t.x0 + cx - 1, x = xr >= 0 && xr < nx ? xr : wrap_clamp(xr, nx, px);
          const uint8_t f = fl[size_t(y) * L.pitch + x];
          if (!(f & (F_OFB | F_OSOLID))) continue;
          const uint32_t pos = uint32_t(cy * (t.tx + 2) + cx);
          if (f & F_OFB) {
            plan.copies.push_back(pos | uint32_t(want_w(x, y)) << 16);
          } else {
            RunVirtN v{};
            v.pos = pos;
            for (int b = 1; b < 9; ++b) {
              const int x2 = wrap_clamp(x + EXH[b], nx, px), y2 = wrap_clamp(y + EYH[b], ny, py);
              v.w[b - 1] = solid(x2, y2) ? kWallNone : uint16_t(want_w(x2, y2));
            }
            plan.vn.push_back(v);
          }
        }
      }
      // stencils of the outermost fluid nodes; virtual nodes are numbered after the band, so
      // their indices are fixed up once the band is known
      std::vector<int> vnodes;
      const size_t s0 = plan.w_sten.size();
      std::vector<uint8_t> is_virt;
      for (size_t w = size_t(t.w0); w < plan.w_ofb.size(); ++w) {
        const OfbEntry& e = ofb[plan.w_ofb[w]];
        WallSten q{};
        for (int a = 1; a < 9; ++a) {
          const int x = wrap_clamp(e.x + EXH[a], nx, px), y = wrap_clamp(e.y + EYH[a], ny, py);
          const bool s = solid(x, y);
          is_virt.push_back(s);
          if (s) {
            const size_t n = size_t(y) * nx + x;
            if (stamp[n] != int(k)) {
              stamp[n] = int(k);
              local[n] = int(vnodes.size());
              vnodes.push_back(int(n));
            }
            q.i[a - 1] = uint16_t(local[n]);
          } else {
            q.i[a - 1] = uint16_t(in_band(x, y));
          }
        }
        plan.w_sten.push_back(q);
      }
      for (int node : vnodes) {
        WallSten q{};
        for (int b = 1; b < 9; ++b) {
          const int x = wrap_clamp(node % nx + EXH[b], nx, px), y = wrap_clamp(node / nx + EYH[b], ny, py);
          q.i[b - 1] = solid(x, y) ? kWallNone : uint16_t(in_band(x, y));
        }
        plan.v_sten.push_back(q);
      }
      t.ne = int(extra.size());
      t.nband = nband;
      for (size_t w = s0; w < plan.w_sten.size(); ++w)
        for (int a = 0; a < 8; ++a)
          if (is_virt[(w - s0) * 8 + a]) plan.w_sten[w].i[a] = uint16_t(plan.w_sten[w].i[a] + t.nband);
      t.nw = nw;
      t.nv = int(vnodes.size());
      t.ncopy = int(plan.copies.size()) - t.copy0;
      t.nvn = int(plan.vn.size()) - t.vn0;
      if (nd + t.ne >= int(kWallNone) || t.nband + t.nv >= int(kWallNone) || t.nw >= int(kWallNone)) return false;
      plan.smem = std::max(plan.smem, run_smem_bytes(t, cs));
      if (plan.smem > max_smem) return false;
    }
  }
  return true;
}

}  // namespace lbcg
