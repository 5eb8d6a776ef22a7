// lbm_pair.cuh -- two steps of the lattice in one pass over memory, many passes
// per launch.
//
// The one-step kernel moves 2 x 9 values per node and step and runs at the
// copy bandwidth on a large lattice: the only way past it is to move less.
// step_pairs reads f*(n), keeps f*(n + 1) in registers and writes f*(n + 2), so
// a step costs 9 values per node instead of 18.  On a small lattice a step costs
// mostly its launch: here a launch runs up to kPairMax passes.
//
// Every warp works alone.  It owns a window of 64 columns, two adjacent nodes
// per lane, and marches up the rows of a cell: row i of f*(n) arrives by
// asynchronous copies (plane k: row i - c_ky) in the warp's own ring of staged
// rows, the warp computes row i of f*(n + 1) from it, then row i - 1 of
// f*(n + 2) from the rows i - 2, i - 1 and i of f*(n + 1), which it holds in
// registers.  A pull from the left or right neighbour is one shuffle per plane
// and pair of nodes.  Each stage loses a column on either side, so a window
// yields 60 columns; the nodes around a cell are computed twice, by neighbouring
// warps, with the same bits.  There is no barrier between warps: one that meets
// the body or the inlet delays nobody.
//
// The per-node arithmetic is that of the one-step kernels, on packed pairs: the
// populations are bit-identical to two of their steps; a force is a double sum of the
// same links in another order.
//
// Why a warp, 64 columns and registers: with a CTA per strip and f*(n + 1) in
// shared memory, the barrier of each row made every warp wait for the one with
// the body or the inlet; with four nodes a lane (128 columns) only two warps fit a
// scheduler and latency ruled (100 GLUPS on 8000 x 4000 against 136 with two).
// What bounds it now: instruction issue and latency (562 instructions for the 120
// node steps of a warp's row, issue slots 53 % used, DRAM 62 % busy on 8000 x 4000).
// Time per step, BGK, cylinder lattices, one-step kernel before and this now:
// 400 x 200 10.2 -> 4.6 us, 800 x 400 14.1 -> 6.1, 1600 x 800 21.2 -> 12.2,
// 3200 x 1600 66.4 -> 37.8, 8000 x 4000 357 -> 222, 16000 x 8000 1416 -> 1035.
#pragma once

#include <algorithm>

#include "lbm_kernels.cuh"

namespace gblbm {

// ---- lane arithmetic: two nodes in packed FP32 instructions ------------------
// The bits of the one-node lane LF.  A packed sum written as an add may be
// merged with the product it adds to, whatever its rounding modifier (seen on
// CUDA 13.0: about 1 % of results differ in the last bit), so sums are
// multiply-adds by a one the compiler cannot see through: exact, and nothing
// left to merge.
static __constant__ float2 kPairOne = {1.f, 1.f}, kPairMinusOne = {-1.f, -1.f};
struct LP2 { float2 v; };
__device__ __forceinline__ LP2 operator+(LP2 a, LP2 b) { return {__ffma2_rn(a.v, kPairOne, b.v)}; }
__device__ __forceinline__ LP2 operator-(LP2 a, LP2 b) { return {__ffma2_rn(b.v, kPairMinusOne, a.v)}; }
__device__ __forceinline__ LP2 operator*(LP2 a, LP2 b) { return {__fmul2_rn(a.v, b.v)}; }
__device__ __forceinline__ LP2 fma(LP2 a, LP2 b, LP2 c) { return {__ffma2_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ LP2 neg_recip(LP2 x) {
  const LP2 y{make_float2(rcp_estimate(-x.v.x), rcp_estimate(-x.v.y))};
  const LP2 e = fma(x, y, LP2{make_float2(1.f, 1.f)});
  return fma(y, e, y);
}
template <> __device__ __forceinline__ LP2 splat<LP2>(double c) { return {make_float2((float)c, (float)c)}; }
template <> __device__ __forceinline__ LP2 coef_at<LP2>(const StepParams &p, int i) {
  return {make_float2(p.kf[i], p.kf[i])};
}

// ---- staging ------------------------------------------------------------------
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

template <int NW, int STAGES>
struct PairLayout {
  static constexpr int TILE = 9 * kPairCols;  // values of one staged row
  static constexpr size_t WARP = (size_t)STAGES * TILE * sizeof(float);
  static constexpr size_t BYTES = NW * WARP;
};

// One plane of the lane's two nodes shifted by its c_kx: the lane's sources.
template <int K>
__device__ __forceinline__ float2 pair_shift(float2 v) {
  if constexpr (CX(K) == 0) return v;
  else if constexpr (CX(K) > 0) return make_float2(__shfl_up_sync(0xffffffffu, v.y, 1), v.x);
  else return make_float2(v.y, __shfl_down_sync(0xffffffffu, v.x, 1));
}
__device__ __forceinline__ float elem(float2 v, int j) { return j ? v.y : v.x; }
__device__ __forceinline__ void set_elem(float2 &v, int j, float s) {
  if (j) v.y = s;
  else v.x = s;
}

// Force sums of a row's links.  A double operation costs an SM 16 clocks a warp and a
// long wait, so a row is added in pairs of floats, and its sums go to the double totals
// once.  The pairs lose nothing while the terms lie within a factor of 2^15: up to 32 of
// them are multiples of the smallest one's last bit, their rounding errors below 2^-14 of
// the largest, and the sum of those fits a float's 24 bits.  Rows with other terms or near
// the ends of the float range are added in double; with an infinity or NaN among them the
// sum is one too, whatever it is added in.
struct LinkSum {
  LF xh{}, xl{}, yh{}, yl{};
  uint32_t most = 0, least = 0xffffffffu;  // largest term's bits; smallest nonzero one's, less 1
  __device__ __forceinline__ void see(float t) {
    const uint32_t bits = __float_as_uint(fabsf(t));
    most = max(most, bits);
    least = min(least, bits - 1u);
  }
  __device__ __forceinline__ void add(int k, float t) {  // along c_k
    LF e;
    if (CX(k)) {
      xh = two_sum(xh, LF{CX(k) > 0 ? t : -t}, e);
      xl = xl + e;
    }
    if (CY(k)) {
      yh = two_sum(yh, LF{CY(k) > 0 ? t : -t}, e);
      yl = yl + e;
    }
    see(t);
  }
  // Add the sums to the totals; false where they have to be added in double.
  __device__ __forceinline__ bool to(double &fx, double &fy) const {
    const bool exact = (most >> 23) < 248u && (most >> 23) <= ((least + 1u) >> 23) + 15u;
    const bool finite = most < 0x7f800000u;
    if (finite && !exact) return false;
    fx += (double)xh.v + (double)(finite ? xl.v : 0.f);
    fy += (double)yh.v + (double)(finite ? yl.v : 0.f);
    return true;
  }
};

// A sum in a pair of floats, 48 bits, without a branch on the terms (batches with BGK).
struct PairSum {
  LF hi{}, lo{};
  __device__ __forceinline__ void add(LF v) {
    LF e;
    hi = two_sum(hi, v, e);
    lo = lo + e;
  }
};
// The same in double, whatever the terms (an infinity or NaN is in hi alone).
__device__ __forceinline__ double total(const PairSum &s) {
  const bool finite = fabsf(s.hi.v) < __int_as_float(0x7f800000);
  return (double)s.hi.v + ((double)(finite ? s.lo.v : 0.f));
}

// The wall rules of boundaries() for a node of the bottom or top row.
__device__ __forceinline__ void pair_wall(int bc, bool bottom, float U, float (&v)[9]) {
  if (bc == BC_FREESLIP) {
    if (bottom) {
      v[2] = v[4];
      v[6] = v[7];
      v[5] = v[8];
    } else {
      v[4] = v[2];
      v[7] = v[6];
      v[8] = v[5];
    }
  } else if (bc == BC_ZOUHE) {
    const float d = 0.5f * (v[1] - v[3]);
    if (bottom) {
      const float m = 0.5f * (v[0] + v[1] + v[3] + 2.f * (v[4] + v[7] + v[8])) * U;
      v[2] = v[4];
      v[5] = v[7] - d + m;
      v[6] = v[8] + d - m;
    } else {
      const float m = 0.5f * (v[0] + v[1] + v[3] + 2.f * (v[2] + v[5] + v[6])) * U;
      v[4] = v[2];
      v[7] = v[5] + d - m;
      v[8] = v[6] - d + m;
    }
  }
}

// History entries of a launch: block c its case c, one warp per step, each
// step's slots of the case summed in slot order.  Clears the cells' flags for the
// next launch, whatever this one left of them (one that gave up leaves them uneven).
static __global__ void __launch_bounds__(1024) pair_finish(StepParams p0, const CaseDesc *cases, PairParams q) {
  const StepParams &p = cases ? cases[blockIdx.x].p : p0;
  const int2 range = q.case_slots ? q.case_slots[blockIdx.x] : make_int2(0, q.nslots);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < q.ncells; i += gridDim.x * blockDim.x) q.flags[i] = 0;
  const unsigned long long n0 = *p.step;
  for (int s = warp; s < 2 * q.pairs; s += 32) {
    double sx, sy;
    slot_sum(q.slots + (size_t)s * q.nslots + range.x, range.y - range.x, lane, sx, sy);
    if (lane == 0 && 2 * q.pairs - s <= p.hist_cap) {  // entries the ring still holds after the launch
      double *h = p.hist + 2 * ((n0 + (unsigned long long)s) % (unsigned long long)p.hist_cap);
      h[0] = sx + p.fconst_x;
      h[1] = sy + p.fconst_y;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) *p.step = n0 + 2ull * (unsigned long long)q.pairs;
}

template <int NW, int STAGES, int MRT, bool INTERP, bool BATCH>
__global__ void __launch_bounds__(NW * 32, 1)
    step_pairs(float *buf0, float *buf1, const __grid_constant__ StepParams p0, const CaseDesc *__restrict__ cases,
               PairParams q) {
  using Lay = PairLayout<NW, STAGES>;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ StepParams sp[BATCH ? NW : 1];  // the parameters of each warp's case

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // a CTA takes neighbouring cells: they share the columns at their edges
  const int per = min(NW, (q.ncells + (int)gridDim.x - 1) / (int)gridDim.x), stride = per * (int)gridDim.x;
  if (warp >= per) return;
  const int first = (int)blockIdx.x * per + warp;
  if (first >= q.ncells) return;
  // Zero.  Waiting for it here keeps a launch's warps in step, and with them the columns
  // and DRAM pages that neighbouring cells share: 64 batched cases with MRT, 76M nodes, ran
  // at 90 GLUPS without this load and at 112 with it.
  const unsigned base_pass = ld_relaxed_gpu(q.flags + first);
  const StepParams &p = BATCH ? sp[warp] : p0;
  float *tiles = reinterpret_cast<float *>(smem + warp * Lay::WARP);

#pragma unroll 1
  for (int pass = 0; pass < q.pairs; ++pass)
#pragma unroll 1
  for (int cell = first; cell < q.ncells; cell += stride) {
    const int4 cd = __ldg(q.cells + cell);
    const float *A = buf0;
    float *B = buf1;
    if constexpr (BATCH) {
      const CaseDesc *c = cases + (cd.x >> 16);
      const uint32_t *src = reinterpret_cast<const uint32_t *>(&c->p);
      uint32_t *dst = reinterpret_cast<uint32_t *>(&sp[warp]);
      __syncwarp();
      for (int k = lane; k < (int)(sizeof(StepParams) / 4); k += 32) dst[k] = __ldg(src + k);
      __syncwarp();
      A = (const float *)c->buf[q.parity];
      B = (float *)c->buf[q.parity ^ 1];
    }
    if (pass & 1) {
      float *t = const_cast<float *>(A);
      A = B;
      B = t;
    }
    if (pass > 0) {  // the neighbours' last pass
      const int dep = __ldg(q.deps + (size_t)cell * 32 + lane);
      const unsigned need = base_pass + (unsigned)pass;
      bool ok = dep < 0 || ld_relaxed_gpu(q.flags + max(dep, 0)) >= need;
      if (!__all_sync(0xffffffffu, ok)) {
        const unsigned long long t0 = global_ns(), lim = wait_limit(p.wait_ns);
        while (true) {
          if (!ok) ok = ld_relaxed_gpu(q.flags + dep) >= need;
          if (__all_sync(0xffffffffu, ok)) break;
          if (__any_sync(0xffffffffu, global_ns() - t0 > lim)) {
            if (lane == 0) atomicOr(p.err, ERR_TIMEOUT);
            return;  // with no copy in flight; the cells that wait for this one run out as well
          }
        }
      }
      fence_acq_rel_gpu();
      __syncwarp();
    }
    const bool wrap = p.bc == BC_PERIODIC;
    const int nx = p.nx, ny = p.ny;
    const int a = cd.y, b = cd.z;
    const int base = (cd.x & 0xffff) * kPairOut - kPairMargin, xl = base + 2 * lane;  // the lane's columns: xl, xl + 1
    const bool mine = lane >= 1 && lane <= 30;  // the columns this window yields
    // First-stage rows: [a - 1, b], clipped unless periodic.
    const int ta = wrap || a > 0 ? a - 1 : 0, tb = wrap || b < ny ? b : ny - 1;
    auto row_of = [&](int t) { return t < 0 ? t + ny : (t >= ny ? t - ny : t); };

    // ---- staging: lane l copies 16 bytes at column 4 (l mod 16) of the planes
    // l / 16, 2 + l / 16, ...; one group of copies per row (an empty group past
    // the last row)
    const int half = lane >> 4, ix = base + 4 * (lane & 15);
    const bool copies = (unsigned)ix < (unsigned)p.pitch;
    const int up = half ? -p.pitch : p.pitch;  // planes 4 and 5 lie a row above and below, 6 and 7 below and above
    int it = ta, ist = 0;
    auto stage_next = [&]() {
      if (it <= tb && copies) {
        const int y = row_of(it);
        const float *src = A + (size_t)y * p.pitch + (half ? p.plane : 0) + ix;
        const uint32_t dst = smem_addr(tiles + ist * Lay::TILE + half * kPairCols + 4 * (lane & 15));
        constexpr int step = 2 * kPairCols * 4;
        if (y > 0 && y < ny - 1) {
          cp_async16(dst, src);
          cp_async16(dst + step, src + 2 * p.plane - (half ? 0 : p.pitch));
          cp_async16(dst + 2 * step, src + 4 * p.plane + up);
          cp_async16(dst + 3 * step, src + 6 * p.plane - up);
          if (half == 0) cp_async16(dst + 4 * step, src + 8 * p.plane + up);
        } else {  // past a wall: wrapped, or (never used) the wall row itself
#pragma unroll 1
          for (int c = 0; c < 5 - half; ++c) {
            const int k = 2 * c + half;
            int sy = y - CY(k);
            sy = wrap ? row_of(sy) : min(max(sy, 0), ny - 1);
            cp_async16(dst + c * step, A + (size_t)k * p.plane + (size_t)sy * p.pitch + ix);
          }
        }
      }
      cp_async_commit();
      ++it;
      if (++ist == STAGES) ist = 0;
    };
#pragma unroll 1
    for (int k = 0; k < STAGES - 1; ++k) stage_next();

    const Coef<LP2> cf = make_coef<LP2>(p);
    const float U = (float)p.U;
    uint32_t worst = 0;                             // largest |u|^2 seen, as bits
    // this lane's links, per stage
    double fx[2] = {0.0, 0.0}, fy[2] = {0.0, 0.0};
    int st = 0;                                     // stage of the current row's tile
    const bool map_cols = p.lx0 < base + kPairCols && p.lx0 + p.lw > base;  // the window meets the link map
    const bool has_inlet = base <= 0, has_outlet = base + kPairCols >= nx;
    uint32_t valid[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) valid[j] = mine && xl + j >= 0 && xl + j < nx - 1 ? 0xffffffffu : 0u;
    uint32_t lm[2], lmp[2] = {0, 0};  // link masks of rows i and i - 1
    auto load_map = [&](int t) {
      const int y = row_of(t);
      const bool in = map_cols && (unsigned)(y - p.ly0) < (unsigned)p.lh;
#pragma unroll
      for (int j = 0; j < 2; ++j) lm[j] = in ? link_mask(p, xl + j, y) : 0u;
    };
    load_map(ta);
    float2 h[9], hp[9], hq[9];  // f*(n + 1): row i; row i - 1; of row i - 2 the planes with c_ky = 1
#pragma unroll
    for (int k = 0; k < 9; ++k) h[k] = hp[k] = hq[k] = make_float2(0.f, 0.f);

    auto wall_row = [&](int y) { return !wrap && (y == 0 || y == ny - 1); };
    auto any_link = [&](const uint32_t (&m)[2]) { return __any_sync(0xffffffffu, (m[0] | m[1]) != 0) != 0; };
    // One stage on the lane's nodes of row y: g holds every source as it lies
    // (from outside the lattice or the body: whatever lies there) and becomes
    // the post-collision state.  Without a branch per node: links take the node's
    // own value by selection, a wall row's rule runs on the whole row, and at the
    // inlet the three populations from outside are replaced by the rule (the
    // corner nodes of a Zou-He wall, whose rule reads them, take their own values
    // first).
    auto update = [&](float2 (&g)[9], int y, const uint32_t (&m)[2], bool links, const float2 (&own)[9], bool counts,
                      int s) {
      if (links) {
        [[maybe_unused]] LinkSum sum;  // interpolated links: the populations that leave and return
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (!__any_sync(0xffffffffu, (m[j] & LM_LINKS) != 0)) continue;
          float src[9];
#pragma unroll
          for (int k = 0; k < 9; ++k) src[k] = elem(g[k], j);
          const float *qn = INTERP ? p.qmap + ((size_t)(y - p.ly0) * p.lw + (xl + j - p.lx0)) * 8 : nullptr;
#pragma unroll
          for (int k = 1; k < 9; ++k) {
            const bool hit = (m[j] & (1u << k)) != 0;
            const float hi = elem(own[OPP(k)], j);
            if constexpr (!INTERP) {
              const float r = CX(k) ? hi + (float)(-6.0 * WD(k) * CX(k)) * U : hi;
              set_elem(g[k], j, hit ? r : src[k]);
            } else {
              if (hit) {
                float r;
                const float qf = __ldg(qn + (k - 1));
                float wref;
                if (qf < 0.5f) {
                  r = (2.f * qf) * hi + (1.f - 2.f * qf) * src[OPP(k)];  // the node behind, x + c_k
                  wref = 1.f;
                } else {
                  wref = 0.5f / qf;
                  r = wref * hi + (1.f - wref) * elem(own[k], j);
                }
                if (CX(k)) r += (float)(-6.0 * WD(k) * CX(k)) * U * wref;
                set_elem(g[k], j, r);
                sum.add(OPP(k), hi);
                sum.add(OPP(k), r);
              }
            }
          }
        }
        if constexpr (INTERP) {
          if (counts && mine) {
            if (!sum.to(fx[s], fy[s])) {
#pragma unroll 1
              for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int k = 1; k < 9; ++k)
                  if ((j ? m[1] : m[0]) & (1u << k)) {
                    const double t = (double)elem(own[OPP(k)], j) + (double)elem(g[k], j);
                    if (CX(k)) fx[s] += CX(k) < 0 ? t : -t;
                    if (CY(k)) fy[s] += CY(k) < 0 ? t : -t;
                  }
            }
          }
        }
      }
      if (wall_row(y)) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          float v[9];
#pragma unroll
          for (int k = 0; k < 9; ++k) v[k] = elem(g[k], j);
          if (p.bc == BC_MOVINGWALL) {
            float drho = 0.f;
#pragma unroll
            for (int k = 0; k < 9; ++k) drho += elem(own[k], j);
#pragma unroll
            for (int k = 1; k < 9; ++k)
              if (CY(k) == (y == 0 ? 1 : -1)) v[k] = elem(own[OPP(k)], j) + (float)(6.0 * WD(k) * CX(k)) * U * drho;
          } else if (xl + j == 0) {
            v[1] = elem(own[1], j);
            v[5] = elem(own[5], j);
            v[8] = elem(own[8], j);
          }
          pair_wall(p.bc, y == 0, U, v);
#pragma unroll
          for (int k = 0; k < 9; ++k) set_elem(g[k], j, v[k]);
        }
      }
      if (has_inlet && xl == 0) {
        float v[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) v[k] = g[k].x;
        inlet<float>(v, U);
#pragma unroll
        for (int k = 0; k < 9; ++k) g[k].x = v[k];
      }
      LP2 v[9];
#pragma unroll
      for (int k = 0; k < 9; ++k) v[k] = LP2{g[k]};
      const float2 uu = collide_model<MRT, LP2>(v, cf).v;
#pragma unroll
      for (int k = 0; k < 9; ++k) g[k] = v[k].v;
      uint32_t u[2] = {__float_as_uint(uu.x), __float_as_uint(uu.y)};
      if (links) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (m[j] & LM_SOLID) u[j] = 0;
#pragma unroll
          for (int k = 0; k < 9; ++k)
            if (m[j] & LM_SOLID) set_elem(g[k], j, 0.f);
        }
        if constexpr (!INTERP) {
          if (counts) {  // half-way links: the population leaves and returns (the factor 2 comes last)
            if constexpr (BATCH && !MRT) {
              // Without a branch: one in this place, or the registers of a longer sum, makes
              // the BGK batch spill in its marching loop (16 cases: 113 GLUPS as it is, 70
              // with the exact pairs below, 69 with triples of floats).  Scaled by 2^-8 the sums
              // stay within the float range.
              PairSum sx, sy;
#pragma unroll
              for (int k = 1; k < 9; ++k)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                  const float t = m[j] & (1u << OPP(k)) ? 0x1p-8f * elem(g[k], j) : 0.f;
                  if (CX(k)) sx.add(LF{CX(k) > 0 ? t : -t});
                  if (CY(k)) sy.add(LF{CY(k) > 0 ? t : -t});
                }
              if (mine) {
                fx[s] += 256.0 * total(sx);
                fy[s] += 256.0 * total(sy);
              }
            } else {
            // Per node one value for each pair of opposite directions (both seldom hold a
            // link), and no branch for a direction without links.
            float d[2][4];
            uint32_t both = 0;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              const uint32_t mj = mine ? m[j] : 0u;
              auto of = [&](int k) { return mj & (1u << OPP(k)) ? elem(g[k], j) : 0.f; };
              both |= mj & (mj >> 2) & 0x66u;  // directions 1 and 3, 2 and 4, 5 and 7, 6 and 8
              d[j][0] = of(1) - of(3);
              d[j][1] = of(2) - of(4);
              d[j][2] = of(5) - of(7);
              d[j][3] = of(6) - of(8);
            }
            LF t[4], l[4], e;  // the two nodes' values added
            LinkSum sum;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              t[c] = two_sum(LF{d[0][c]}, LF{d[1][c]}, l[c]);
              sum.see(d[0][c]);
              sum.see(d[1][c]);
            }
            sum.xh = two_sum(t[0], t[2], e);
            sum.xl = (l[0] + l[2]) + e;
            sum.xh = two_diff(sum.xh, t[3], e);
            sum.xl = sum.xl + (e - l[3]);
            sum.yh = two_sum(t[1], t[2], e);
            sum.yl = (l[1] + l[2]) + e;
            sum.yh = two_sum(sum.yh, t[3], e);
            sum.yl = sum.yl + (e + l[3]);
            if (both || !sum.to(fx[s], fy[s])) {
#pragma unroll 1
              for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int k = 1; k < 9; ++k)
                  if ((mine ? (j ? m[1] : m[0]) : 0u) & (1u << OPP(k))) {
                    const double t = j ? g[k].y : g[k].x;
                    if (CX(k)) fx[s] += CX(k) > 0 ? t : -t;
                    if (CY(k)) fy[s] += CY(k) > 0 ? t : -t;
                  }
            }
            }
          }
        }
      }
      // |u|^2 as bits: monotonic for numbers, above all of them for a NaN
      worst = max(worst, max(u[0] & valid[0], u[1] & valid[1]));
      if (has_outlet) {  // Eq. 13: column nx - 1 is column nx - 2
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          const float left = __shfl_up_sync(0xffffffffu, g[k].y, 1);
          if (xl + 1 == nx - 1) g[k].y = g[k].x;
          if (xl == nx - 1) g[k].x = left;
        }
      }
    };

#pragma unroll 1
    for (int i = ta; i <= b; ++i) {
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        if (CY(k) > 0) hq[k] = hp[k];
        hp[k] = h[k];
      }
      if (i <= tb) {  // ---- first stage, row i
        cp_async_wait<STAGES - 2>();
        __syncwarp();
        const float *tile = tiles + st * Lay::TILE + 2 * lane;
        auto at = [&](int k) { return *reinterpret_cast<const float2 *>(tile + k * kPairCols); };
        h[0] = pair_shift<0>(at(0));
        h[1] = pair_shift<1>(at(1));
        h[2] = pair_shift<2>(at(2));
        h[3] = pair_shift<3>(at(3));
        h[4] = pair_shift<4>(at(4));
        h[5] = pair_shift<5>(at(5));
        h[6] = pair_shift<6>(at(6));
        h[7] = pair_shift<7>(at(7));
        h[8] = pair_shift<8>(at(8));
        const int y = row_of(i);
        const bool links = any_link(lm);
        float2 own[9];
        if (links || wall_row(y)) {
          // A node's own value of plane k lies in the tile of row i + c_ky, or
          // past the ends of the cell in global memory.
          const int stm = st == 0 ? STAGES - 1 : st - 1, stp = st == STAGES - 1 ? 0 : st + 1;
          cp_async_wait<STAGES - 3>();
          __syncwarp();
          const float *row = A + (size_t)y * p.pitch + min(max(xl, 0), p.pitch - 2);
#pragma unroll
          for (int k = 0; k < 9; ++k) {
            const int t = i + CY(k), sk = CY(k) == 0 ? st : (CY(k) > 0 ? stp : stm);
            if (t < ta || t > tb) own[k] = __ldcg(reinterpret_cast<const float2 *>(row + (size_t)k * p.plane));
            else own[k] = *reinterpret_cast<const float2 *>(tiles + sk * Lay::TILE + k * kPairCols + 2 * lane);
          }
        }
        update(h, y, lm, links, own, i >= a && i < b, 0);
        if (++st == STAGES) st = 0;
        __syncwarp();
        stage_next();  // into the stage of row i - 1, which no lane reads any more
      }
      const uint32_t m[2] = {lmp[0], lmp[1]};
      lmp[0] = lm[0];
      lmp[1] = lm[1];
      if (i < tb) load_map(i + 1);
      if (i > a) {  // ---- second stage, row i - 1
        float2 g[9] = {pair_shift<0>(hp[0]), pair_shift<1>(hp[1]), pair_shift<2>(hq[2]),
                       pair_shift<3>(hp[3]), pair_shift<4>(h[4]),  pair_shift<5>(hq[5]),
                       pair_shift<6>(hq[6]), pair_shift<7>(h[7]),  pair_shift<8>(h[8])};
        update(g, i - 1, m, any_link(m), hp, true, 1);
        float *o = B + (size_t)(i - 1) * p.pitch + xl;
        // a node at column nx lies in the row's padding; the outlet column, a copy,
        // may follow the last column of the window
        if (mine ? xl >= 0 && xl < nx : lane == 31 && xl == nx - 1) {
#pragma unroll
          for (int k = 0; k < 9; ++k) *reinterpret_cast<float2 *>(o + (size_t)k * p.plane) = g[k];
        }
      }
    }
    if (__any_sync(0xffffffffu, worst > __float_as_uint(0.09f)) && lane == 0) atomicOr(p.err, ERR_UNSTABLE);
    if (cd.w >= 0) {  // the cell owns links: its force partials of the two steps
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const double c = INTERP ? 1.0 : 2.0;  // half-way links: the population leaves and returns
        const double sx = warp_sum(c * fx[s]), sy = warp_sum(c * fy[s]);
        if (lane == 0) __stcg(q.slots + (size_t)(2 * pass + s) * q.nslots + cd.w, make_double2(sx, sy));
      }
    }
    // the pass is done: this cell's nodes are written, its neighbours' are read
    cp_async_wait<0>();
    __syncwarp();
    if (lane == 0 && !(cd.x >> 16 == q.fault_case && a <= q.fault_row && q.fault_row < b)) {
      fence_acq_rel_gpu();
      st_relaxed_gpu(q.flags + cell, base_pass + (unsigned)pass + 1u);
    }
  }
}

// Launch q.pairs passes and the sums of their forces (mode 0), set the
// shared-memory limit (1) or query the resident CTAs per SM (2, into *occ).
// Single lattice: buf0, buf1, p; batch: cases, ncases.
template <int NW, int STAGES, bool INTERP, bool BATCH>
cudaError_t pair_one(int grid, float *buf0, float *buf1, const StepParams &p, const CaseDesc *cases, int ncases, int mrt,
                     const PairParams &q, cudaStream_t st, int mode, int *occ) {
  constexpr size_t smem = PairLayout<NW, STAGES>::BYTES;
  auto k0 = step_pairs<NW, STAGES, 0, INTERP, BATCH>;
  auto k1 = step_pairs<NW, STAGES, 1, INTERP, BATCH>;
  if (mode == 1) {
    const cudaError_t e = cudaFuncSetAttribute(k0, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  }
  if (mode == 2) {
    int n = 0, m = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k0, NW * 32, smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&m, k1, NW * 32, smem);
    *occ = n < m ? n : m;
    return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  // only the warps that get a cell, with their rings: launches of several small lattices
  // on streams of their own then share the SMs
  const int per = std::min(NW, (q.ncells + grid - 1) / grid);
  cfg.blockDim = dim3(per * 32);
  cfg.dynamicSmemBytes = per * PairLayout<NW, STAGES>::WARP;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, mrt ? k1 : k0, buf0, buf1, p, cases, q);
  if (e != cudaSuccess) return e;
  pair_finish<<<BATCH ? ncases : 1, 1024, 0, st>>>(p, BATCH ? cases : nullptr, q);
  return cudaGetLastError();
}

}  // namespace gblbm
