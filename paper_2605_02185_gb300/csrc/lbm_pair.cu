// lbm_pair.cu -- the split of one or many lattices into the cells of the
// two-step kernel.
#include "lbm_pair_host.h"

#include <algorithm>
#include <cmath>

#include "lbm_device.cuh"
#include "lbm_host.h"

namespace gblbm {

namespace {

struct Window {
  int lat, w;      // lattice, window
  double row;      // cost of a plain row
  int y0, y1;      // rows [y0, y1) that meet the body
  double total;
};

// Cost of a row of the inlet's or outlet's window, and of a row that meets the
// body, against a plain row.  A pass ends with its slowest cell: 3200 x 1600 with
// body rows counted as 1, 1.3, 1.6 and 2 plain ones ran at 61, 53, 47 and 45 us a
// step, edge windows at 1.4 instead of 1.2 made no difference.
constexpr double kEdgeCost = 1.2, kBodyCost = 2.0;
// Cost of a cell beyond its rows, in plain rows: two rows computed twice, the
// filling of its ring.
constexpr double kCellCost = 3.0;

// Nodes from which a launch runs one pass only.  Within a launch the cells drift
// apart, and on a large lattice the columns and DRAM pages that neighbouring
// windows share are then fetched twice; the launch between passes lines them up
// again.  us a step with 32 passes a launch and with one: 3200 x 1600 41 and 45,
// 4400 x 2200 (9.7M nodes) 75.3 and 77.1, 4800 x 2400 92.9 and 91.3, 5600 x 2800 (15.7M)
// 126 and 121, 6400 x 3200 172 and 155, 8000 x 4000 259 and 235: the two meet near 10M
// nodes, and between there and this line up to 4 % is left.
constexpr long long kPairManyNodes = 16ll << 20;

// Windows of a row: the last one yields column nx - 2 (and column nx - 1, its
// copy, even where that lies one past the columns a window yields).
int pair_windows(int nx) { return (nx + 1 + kPairOut - 1) / kPairOut; }

size_t part(size_t n, size_t bytes) { return align_up(n * bytes, kAlign); }

}  // namespace

size_t pair_region_bytes(int cells, int slots, int cases) {
  return part(cells, sizeof(int4)) + part((size_t)cells * 32, sizeof(int)) + part(cells, sizeof(unsigned)) +
         part((size_t)2 * kPairMax * slots, sizeof(double2)) + part(cases, sizeof(int2));
}

int pair_plan(const std::vector<PairLattice> &lattices, int sms, void *region, int cells_cap, int slots_cap,
              cudaStream_t st, PairParams *q, int *grid) {
  *grid = 0;
  int warps = sms * kPairWarps;
  std::vector<Window> win;
  for (size_t l = 0; l < lattices.size(); ++l) {
    const PairLattice &t = lattices[l];
    const Geometry &g = *t.geo;
    const int windows = pair_windows(t.nx);
    if (windows > 0xffff || l > 0x7fff) return LBM_OK;
    for (int w = 0; w < windows; ++w) {
      const int x0 = w * kPairOut - kPairMargin;
      const bool body = g.fx1 >= g.fx0 && x0 <= g.fx1 && x0 + kPairCols > g.fx0;
      Window v = {(int)l, w, w == 0 || w == windows - 1 ? kEdgeCost : 1.0, body ? g.fy0 : 0, body ? g.fy1 + 1 : 0, 0.0};
      v.total = v.row * (t.ny + (kBodyCost - 1.0) * (v.y1 - v.y0));
      win.push_back(v);
    }
  }
  // A lattice of about as many rows as half the warps leaves the other half: it gains 1 %
  // from the rest (400 x 200, 1,400 rows: 4.78 us a step, with 1,216 warps 4.83), and the
  // launches of two such lattices on two streams then run at the same time (9.16 and 5.49
  // us a step of both; four of them 18.5 and 10.6).  With 3,300 rows, 600 x 300, half the
  // warps would cost it 10 %.
  if (lattices.size() == 1 && (long long)win.size() * lattices[0].ny * 5 <= 3ll * warps) warps /= 2;
  // One cell per warp where that can be: every window is cut into bands of rows
  // of equal cost, as cheap as the number of warps allows.
  auto bands = [&](const Window &v, double cost) {
    return std::max(1, std::min(lattices[v.lat].ny, (int)std::ceil(v.total / cost)));
  };
  double most = 1.0;
  for (const Window &v : win) most = std::max(most, v.total);
  auto cheapest = [&](int n_max) {  // the least cost per cell that needs at most n_max cells
    double lo = 1.0, up = most;
    for (int k = 0; k < 40; ++k) {
      const double mid = 0.5 * (lo + up);
      long long n = 0;
      for (const Window &v : win) n += bands(v, mid);
      if (n <= n_max) up = mid;
      else lo = mid;
    }
    return up;
  };
  // Where few bands fit (wide lattices), a second or third cell per warp wastes
  // fewer of the warps: 40000 x 3000 has 667 windows, so three bands leave a
  // sixth of 2,432 warps idle and ran at 1324 us a step, seven at 964.
  double hi = cheapest(warps);
  for (int rounds = 2; rounds <= 3; ++rounds) {
    const double c = cheapest(rounds * warps);
    if (rounds * (c + kCellCost) < 0.95 * (hi + kCellCost) && (long long)rounds * warps <= cells_cap) {
      hi = c;
      break;
    }
  }
  std::vector<int4> cells;
  std::vector<double> place;  // a cell's height in its lattice
  for (const Window &v : win) {
    const int n = bands(v, hi), ny = lattices[v.lat].ny;
    int a = 0;
    for (int k = 1; k <= n; ++k) {
      double t = v.total * k / n / v.row;  // cost of the rows up to the band's end
      if (t > v.y0) t = t < v.y0 + kBodyCost * (v.y1 - v.y0) ? v.y0 + (t - v.y0) / kBodyCost : t - (kBodyCost - 1.0) * (v.y1 - v.y0);
      const int b = k == n ? ny : std::min(ny, (int)(t + 0.5));
      if (b > a) {
        cells.push_back(make_int4(v.lat << 16 | v.w, a, b, -1));
        place.push_back(v.lat + (double)a / ny);
      }
      a = std::max(a, b);
    }
  }
  const int n = (int)cells.size();
  if (n > cells_cap) return LBM_OK;
  // lattice by lattice, band by band: neighbouring windows side by side
  std::vector<int> order((size_t)n);
  for (int i = 0; i < n; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int l, int r) { return place[l] < place[r]; });
  std::vector<int4> sorted((size_t)n);
  for (int i = 0; i < n; ++i) sorted[i] = cells[order[i]];
  cells.swap(sorted);
  // Force slots of the cells that own links, case by case.
  std::vector<int2> ranges(lattices.size(), make_int2(0, 0));
  int slots = 0;
  for (int i = 0; i < n;) {
    const int l = cells[i].x >> 16;
    ranges[l].x = slots;
    for (; i < n && cells[i].x >> 16 == l; ++i) {
      const Geometry &g = *lattices[l].geo;
      const int o0 = (cells[i].x & 0xffff) * kPairOut - kPairMargin + 2;
      if (g.fx1 >= g.fx0 && o0 <= g.fx1 && o0 + kPairOut > g.fx0 && cells[i].y <= g.fy1 && cells[i].z > g.fy0)
        cells[i].w = slots++;
    }
    ranges[l].y = slots;
  }
  if (slots > slots_cap) return LBM_OK;
  // The cells whose nodes lie within two columns and two rows of a cell's own:
  // those it reads, and those that read it.
  std::vector<std::vector<int>> by_window(win.size());
  std::vector<int> base(lattices.size(), 0);
  for (size_t v = 0; v < win.size(); ++v)
    if (win[v].w == 0) base[win[v].lat] = (int)v;
  for (int i = 0; i < n; ++i) by_window[(size_t)base[cells[i].x >> 16] + (cells[i].x & 0xffff)].push_back(i);
  std::vector<int> deps((size_t)n * 32, -1);
  for (int i = 0; i < n; ++i) {
    const int l = cells[i].x >> 16, w = cells[i].x & 0xffff, ny = lattices[l].ny;
    const int windows = pair_windows(lattices[l].nx);
    int m = 0;
    for (int v = std::max(w - 1, 0); v <= std::min(w + 1, windows - 1); ++v) {
      const std::vector<int> &col = by_window[(size_t)base[l] + v];  // bottom to top
      for (int s = -1; s <= 1; ++s) {                                // periodic: the rows past the ends
        if (s != 0 && lattices[l].bc != LBM_BC_PERIODIC) continue;
        const int y0 = cells[i].y - 2 - s * ny, y1 = cells[i].z + 2 - s * ny;  // rows [y0, y1) of the window
        auto it = std::partition_point(col.begin(), col.end(), [&](int c) { return cells[c].z <= y0; });
        for (; it != col.end() && cells[*it].y < y1; ++it) {
          int *end = deps.data() + (size_t)i * 32 + m;
          if (*it == i || std::find(end - m, end, *it) != end) continue;
          if (m == 32) return LBM_OK;
          *end = *it;
          ++m;
        }
      }
    }
  }
  char *at = (char *)region;
  long long nodes = 0;
  for (const PairLattice &t : lattices) nodes += (long long)t.nx * t.ny;
  int4 *d_cells = (int4 *)at;
  at += part(cells_cap, sizeof(int4));
  int *d_deps = (int *)at;
  at += part((size_t)cells_cap * 32, sizeof(int));
  q->flags = (unsigned *)at;
  at += part(cells_cap, sizeof(unsigned));
  q->slots = (double2 *)at;
  at += part((size_t)2 * kPairMax * slots_cap, sizeof(double2));
  int2 *d_ranges = (int2 *)at;
  q->cells = d_cells;
  q->deps = d_deps;
  q->case_slots = d_ranges;
  q->ncells = n;
  q->nslots = slots;
  q->pairs = nodes < kPairManyNodes ? kPairMax : 1;
  q->parity = 0;
  q->fault_case = q->fault_row = -1;
  CK(cudaMemcpyAsync(d_cells, cells.data(), cells.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(d_deps, deps.data(), deps.size() * sizeof(int), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(d_ranges, ranges.data(), ranges.size() * sizeof(int2), cudaMemcpyHostToDevice, st));
  CK(cudaMemsetAsync(q->flags, 0, (size_t)n * sizeof(unsigned), st));
  CK(cudaStreamSynchronize(st));
  *grid = std::min(n, sms);
  return LBM_OK;
}

int64_t pair_steps_of(cudaStream_t st, int64_t n) {
  if (n < 2) return 0;
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &status) != cudaSuccess) cudaGetLastError();  // the launch reports it
  return n & ~(int64_t)(status == cudaStreamCaptureStatusNone ? 1 : 3);
}

}  // namespace gblbm
