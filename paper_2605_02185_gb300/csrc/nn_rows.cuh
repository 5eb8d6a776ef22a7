// nn_rows.cuh -- 3x3 convolution of the layers with few channels (8 to 96 in, up
// to 96 out) on the tensor cores: included by nn_tc.cu.
//
// Such a layer is bound by moving data.  conv_tc_kernel copies the 128-pixel
// input tile once per tap and the weights once per tile: 90 KB of L2 traffic for
// 18 MMAs on a 32 -> 32 layer.  Here the weights stay in shared memory and a CTA
// marches down the image rows of one 128-pixel column, holding a ring of input
// rows (130 pixels wide): a tile needs one new row, and the nine taps are nine
// start addresses into the three rows it holds.  For that the rows lie
// unswizzled, [8-channel chunk][pixel][16 bytes] -- the core-matrix layout of
// tcgen05's no-swizzle mode with eight-pixel groups 128 bytes apart, linear in
// the pixel, so that a shift by a pixel is 16 bytes.
//
// Warps 0-3 read the accumulators back, warp 4 issues the MMAs, warps 5-8 copy
// the rows (cp.async, 16 bytes per thread and access, zero-filled outside the
// image).  The MMAs of a tile are issued in the order of conv_tc_kernel (of the
// mma.sync kernel for 8 channels, whose K steps of 16 are half zeros), so the
// sums are the same bits.  Every wait is bounded as in nn_tc.cu.
//
// 4 samples, us before (conv_tc_kernel; 8 channels: mma.sync) and now, both without a
// mask: 800 x 1600, forward 32 -> 32 457 and 169, 8 -> 32 594 and 122, 32 -> 8 457 and 126,
// 96 -> 32 700 and 655; gradient 32 -> 32 450 and 157, 32 -> 96 862 and 416; 400 x 800,
// 32 -> 64 162 and 104, 64 -> 64 154 and 105, its gradient 158 and 102.  Small images are
// left to conv_tc_kernel (nn_rows_rule.h).  What bounds
// it: 32 -> 32 DRAM at half its rate, with the latency of the read-back and the
// row copies of two resident CTAs; 96 -> 32 the MMAs, each reading 4 KB of A for 32
// columns.
#pragma once

constexpr int kRowPix = kTileM + 2;              // pixels of a staged row
constexpr int kRowChunk = kRowPix * 16;          // bytes of its 8-channel chunk
constexpr int kRowThreads = 288, kRowProducers = 128;

template <int BN, int CIN, int SLOTS>
struct RowLayout {
  static constexpr int C8 = CIN / 8;                   // chunks of a pixel in memory
  static constexpr int CH = C8 < 2 ? 2 : C8;           // chunks of a staged row (a zero chunk fills K = 16)
  static constexpr int KCH = 9 * CH;                   // chunks along K
  static constexpr int ROW = CH * kRowChunk;
  static constexpr int W_OFF = SLOTS * ROW;            // weights: [K chunk][BN][16 bytes]
  static constexpr int BIAS_OFF = W_OFF + KCH * BN * 16;
  static constexpr int BAR_OFF = BIAS_OFF + BN * 4;    // full[S], empty[S], acc_full[2], acc_empty[2], drain
  static constexpr int BYTES = BAR_OFF + (2 * SLOTS + 5) * 8 + 16;
  static constexpr uint32_t ACC_COLS = BN <= 32 ? 32 : BN <= 64 ? 64 : 128;
  static constexpr uint32_t NCOLS = 2 * ACC_COLS;
  static constexpr int ALLOC = BYTES + 128 > smem_floor(NCOLS) ? BYTES + 128 : smem_floor(NCOLS);
};

// Descriptor of an unswizzled K-major operand: core matrices of 8 rows x 16
// bytes, 128 bytes apart along M or N, lbo bytes apart along K.
__device__ __forceinline__ uint64_t plain_desc(uint32_t addr, uint32_t lbo) {
  uint64_t d = (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)(128u >> 4) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}
__device__ __forceinline__ void st_global_32(void *p, const uint32_t *v) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]),
               "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
// One lane of the converged warp.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r));
  return r;
}
__device__ __forceinline__ void umma_bf16_if(uint32_t issue, uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                             uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(issue)
      : "memory");
}
__device__ __forceinline__ void umma_commit_if(uint32_t issue, uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar),
      "r"(issue)
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void cp_async16_fill(uint32_t dst, const void *src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}

// Rows [h0, h1) of 128-pixel column `col` of the walk that falls to one CTA.
struct RowWalk {
  long long u, end;
  int H;
  __device__ RowWalk(long long units, int H_) : H(H_) {
    u = units * blockIdx.x / gridDim.x;
    end = units * (blockIdx.x + 1) / gridDim.x;
  }
  __device__ bool next(int &col, int &h0, int &h1) {
    if (u >= end) return false;
    col = (int)(u / H);
    h0 = (int)(u - (long long)col * H);
    h1 = end - u < H - h0 ? h0 + (int)(end - u) : H;
    u += h1 - h0;
    return true;
  }
};

template <int BN, int CIN, int SLOTS>
__global__ void __launch_bounds__(kRowThreads, BN <= 32 && CIN <= 32 ? 2 : 1)
    conv_rows_kernel(const bf16 *__restrict__ x, int xs, const bf16 *__restrict__ w, const float *__restrict__ bias,
                     bf16 *__restrict__ y, int ys, const bf16 *__restrict__ mask, int ms, int H, int W, int cout, int relu,
                     long long units) {
  using Lay = RowLayout<BN, CIN, SLOTS>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
  float *sbias = reinterpret_cast<float *>(smem + Lay::BIAS_OFF);
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + Lay::BAR_OFF);
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + Lay::BAR_OFF + (2 * SLOTS + 5) * 8);
  __shared__ int s_abort_store;
  volatile int *s_abort = &s_abort_store;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wtiles = (W + kTileM - 1) / kTileM;
  const uint32_t full0 = saddr(&bars[0]), empty0 = saddr(&bars[SLOTS]);
  const uint32_t accf0 = saddr(&bars[2 * SLOTS]), acce0 = saddr(&bars[2 * SLOTS + 2]);
  const uint32_t drain_bar = saddr(&bars[2 * SLOTS + 4]);

  if (threadIdx.x == 0) {
    for (int s = 0; s < SLOTS; ++s) {
      mbar_init(full0 + 8 * s, kRowProducers);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf0 + 8 * b, 1);
      mbar_init(acce0 + 8 * b, 4);
    }
    mbar_init(drain_bar, 1);
    *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // weights (zero beyond cout and beyond the layer's channels), bias, zero chunks
  for (int i = threadIdx.x; i < Lay::KCH * BN; i += kRowThreads) {
    const int q = i / BN, o = i - q * BN, tap = q / Lay::CH, c = q - tap * Lay::CH;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (o < cout && c < Lay::C8) v = __ldg(reinterpret_cast<const uint4 *>(w + ((size_t)o * 9 + tap) * CIN + 8 * c));
    *reinterpret_cast<uint4 *>(smem + Lay::W_OFF + i * 16) = v;
  }
  for (int o = threadIdx.x; o < BN; o += kRowThreads) sbias[o] = bias && o < cout ? bias[o] : 0.f;
  if constexpr (Lay::CH > Lay::C8) {
    for (int i = threadIdx.x; i < SLOTS * kRowPix; i += kRowThreads)
      *reinterpret_cast<uint4 *>(smem + (i / kRowPix) * Lay::ROW + kRowChunk + (i % kRowPix) * 16) = make_uint4(0, 0, 0, 0);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 4) {
    tmem_alloc(saddr(tmem_slot), Lay::NCOLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  RowWalk walk(units, H);
  int col, h0, h1;

  if (warp >= 5) {  // ---------------- producers: one input row after another
    const int tid = threadIdx.x - 160;
    int g = 0, arrived = 0;  // rows copied, rows handed over
    bool stop = false;
    auto hand_over = [&]() {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(full0 + 8 * (arrived % SLOTS));
      ++arrived;
    };
    while (!stop && walk.next(col, h0, h1)) {
      const int n = col / wtiles, w0 = (col - n * wtiles) * kTileM;
      for (int r = h0 - 1; r <= h1; ++r, ++g) {
        const int s = g % SLOTS;
        if (g >= SLOTS && !mbar_wait(empty0 + 8 * s, ((g / SLOTS) - 1) & 1, s_abort)) {
          if (!*s_abort) give_up(s_abort);
          stop = true;
          break;
        }
        const bool row_ok = (unsigned)r < (unsigned)H;
        const bf16 *src = x + ((size_t)n * H + (row_ok ? r : 0)) * W * xs;
        const uint32_t dst = saddr(smem + s * Lay::ROW);
#pragma unroll 4
        for (int i = tid; i < kRowPix * Lay::C8; i += kRowProducers) {
          const int px = i / Lay::C8, c = i - px * Lay::C8, gx = w0 - 1 + px;
          const bool ok = row_ok && (unsigned)gx < (unsigned)W;
          cp_async16_fill(dst + c * kRowChunk + px * 16, ok ? src + (size_t)gx * xs + 8 * c : x, ok);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (g - arrived >= 2) {
          asm volatile("cp.async.wait_group 2;" ::: "memory");
          hand_over();
        }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    while (arrived < g) hand_over();
  } else if (warp == 4) {  // ---------------- MMA issuer: the whole warp runs the loop, so that
    // its addresses stay in uniform registers; one lane issues
    const uint32_t leader = elect_one();
    constexpr uint32_t idesc = idesc_bf16(BN);
    const uint64_t bdesc = plain_desc(saddr(smem + Lay::W_OFF), BN * 16);
    const uint64_t adesc = plain_desc(saddr(smem), kRowChunk);
    int g = 0, i = 0, slot = 0;  // rows waited for; tiles; slot of row h - 1
    bool stop = false;
    while (!stop && walk.next(col, h0, h1)) {
      for (int h = h0; h < h1 && !stop; ++h, ++i) {
        const int b = i & 1;
        if (i >= 2 && !mbar_wait(acce0 + 8 * b, ((i >> 1) - 1) & 1, s_abort)) {
          if (!*s_abort) give_up(s_abort);
          stop = true;
        }
        for (int k = h == h0 ? 3 : 1; k > 0 && !stop; --k, ++g) {  // up to row h + 1
          if (!mbar_wait(full0 + 8 * (g % SLOTS), (g / SLOTS) & 1, s_abort)) {
            if (!*s_abort) give_up(s_abort);
            stop = true;
          }
        }
        stop = __any_sync(0xffffffffu, stop);
        if (stop) break;
        tc_fence_after();
        const uint32_t acc = tmem + (uint32_t)(b * Lay::ACC_COLS);
        const int s1 = slot + 1 < SLOTS ? slot + 1 : slot + 1 - SLOTS, s2 = slot + 2 < SLOTS ? slot + 2 : slot + 2 - SLOTS;
#pragma unroll
        for (int dy = 0; dy < 3; ++dy) {
          const uint64_t row = adesc + (uint64_t)((dy == 0 ? slot : dy == 1 ? s1 : s2) * (Lay::ROW >> 4));
          // K order of conv_tc_kernel: 64-channel layers tap by tap, others 32 channels of a kernel row at a time
          constexpr int GROUP = CIN % 64 == 0 ? Lay::CH : (Lay::CH < 4 ? Lay::CH : 4);
#pragma unroll
          for (int c0 = 0; c0 < Lay::CH; c0 += GROUP)
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)
#pragma unroll
              for (int c = c0; c < c0 + GROUP; c += 2)
                umma_bf16_if(leader, acc, row + (uint64_t)((c * kRowChunk + dx * 16) >> 4),
                             bdesc + (uint64_t)(((3 * dy + dx) * Lay::CH + c) * BN), idesc, (dy | c0 | dx | (c - c0)) != 0);
        }
        umma_commit_if(leader, empty0 + 8 * slot);  // row h - 1 is free once these MMAs have read it
        if (h == h1 - 1) {                          // the segment's last two rows with it
          umma_commit_if(leader, empty0 + 8 * s1);
          umma_commit_if(leader, empty0 + 8 * s2);
          slot = s2;
        }
        umma_commit_if(leader, accf0 + 8 * b);
        slot = slot + 1 < SLOTS ? slot + 1 : 0;
      }
    }
    if (i > 0) {  // every MMA done before the tensor memory is freed
      umma_commit_if(leader, drain_bar);
      const unsigned long long t0 = now_ns();
      while (!mbar_test(drain_bar, 0)) {
        if (now_ns() - t0 > kWaitNs) {
          give_up(s_abort);
          break;
        }
      }
    }
  } else {  // ---------------- epilogue warps 0..3
    const int m = 32 * warp + lane;
    const bool wide = ys % 16 == 0 && ((uintptr_t)y & 31) == 0;
    int i = 0;
    bool stop = false;
    while (!stop && walk.next(col, h0, h1)) {
      const int n = col / wtiles, px = (col - n * wtiles) * kTileM + m;
      for (int h = h0; h < h1; ++h, ++i) {
        const int b = i & 1;
        const size_t pix = ((size_t)n * H + h) * W + px;
        constexpr int STEP = BN < 32 ? 16 : 32, OUT = BN < 32 ? 8 : 32;  // columns read, channels stored
        uint4 next[OUT / 8];  // the mask of the channels to come, fetched ahead of their sums
        auto load_mask = [&](int j0) {
          if (mask && px < W) {
            const uint4 *mp = reinterpret_cast<const uint4 *>(mask + pix * ms + j0);
#pragma unroll
            for (int q = 0; q < OUT / 8; ++q) next[q] = __ldg(mp + q);
          }
        };
        load_mask(0);
        bool ok = mbar_wait(accf0 + 8 * b, (i >> 1) & 1, s_abort);
        if (!ok && !*s_abort) give_up(s_abort);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) {
          stop = true;
          break;
        }
        tc_fence_after();
#pragma unroll 1
        for (int j0 = 0; j0 < BN; j0 += STEP) {
          uint4 cur[OUT / 8];
#pragma unroll
          for (int q = 0; q < OUT / 8; ++q) cur[q] = next[q];
          if (j0 + STEP < BN) load_mask(j0 + STEP);
          uint32_t r[STEP];
          const uint32_t at = tmem + (uint32_t)(b * Lay::ACC_COLS) + ((uint32_t)(32 * warp) << 16) + (uint32_t)j0;
          if constexpr (STEP == 16) tmem_ld16(at, r);
          else tmem_ld32(at, r);
          tmem_ld_wait();
          if (px < W) {
            float v[OUT];
#pragma unroll
            for (int q = 0; q < OUT; ++q) v[q] = __uint_as_float(r[q]) + sbias[j0 + q];
            if (relu) {
#pragma unroll
              for (int q = 0; q < OUT; ++q) v[q] = fmaxf(v[q], 0.f);
            }
            if (mask) {
#pragma unroll
              for (int q = 0; q < OUT / 8; ++q) {
                const uint4 mv = cur[q];
                const uint32_t mw[4] = {mv.x, mv.y, mv.z, mv.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const __nv_bfloat162 mk = *reinterpret_cast<const __nv_bfloat162 *>(&mw[e]);
                  if (!(__bfloat162float(mk.x) > 0.f)) v[8 * q + 2 * e] = 0.f;
                  if (!(__bfloat162float(mk.y) > 0.f)) v[8 * q + 2 * e + 1] = 0.f;
                }
              }
            }
            uint32_t pk[OUT / 2];
#pragma unroll
            for (int e = 0; e < OUT / 2; ++e) {
              const __nv_bfloat162 b2 = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
              pk[e] = *reinterpret_cast<const uint32_t *>(&b2);
            }
            bf16 *yp = y + pix * ys + j0;
            if (OUT >= 16 && wide) {  // whole 32-byte sectors
#pragma unroll
              for (int q = 0; q + 8 <= OUT / 2; q += 8) st_global_32(yp + 2 * q, pk + q);
            } else {
#pragma unroll
              for (int q = 0; q < OUT / 2; q += 4)
                *reinterpret_cast<uint4 *>(yp + 2 * q) = make_uint4(pk[q], pk[q + 1], pk[q + 2], pk[q + 3]);
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acce0 + 8 * b);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 4) {
    tc_fence_after();
    tmem_dealloc(tmem, Lay::NCOLS);
  }
}

template <int BN, int CIN, int SLOTS>
cudaError_t launch_rows(const void *x, int xs, const void *w, const float *bias, void *y, int ys, const void *mask, int ms,
                        int N, int H, int W, int cout, int relu, cudaStream_t st) {
  using Lay = RowLayout<BN, CIN, SLOTS>;
  static_assert(Lay::ALLOC <= 227 * 1024, "shared memory");
  auto kern = conv_rows_kernel<BN, CIN, SLOTS>;
  static PerDevice resident;
  const int per_sm = resident.get(current_device(), [&] { return resident_ctas(kern, Lay::ALLOC, kRowThreads, Lay::NCOLS); });
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const long long units = (long long)N * ((W + kTileM - 1) / kTileM) * H;
  const long long most = (long long)per_sm * sm_count();
  kern<<<(int)(units < most ? units : most), kRowThreads, Lay::ALLOC, st>>>(
      (const bf16 *)x, xs, (const bf16 *)w, bias, (bf16 *)y, ys, (const bf16 *)mask, ms, H, W, cout, relu, units);
  return cudaGetLastError();
}

// kNotEligible where there is no row kernel for the channel counts or the
// alignment, or where the image is too small for it (nn_rows_rule.h); arguments as conv_fwd.  Layers of 8 channels only where `eight`: a
// caller that requires the tensor-core kernels by name is refused them.
int conv_rows(const void *x, int xs, const void *w, const float *bias, void *y, int ys, const void *mask, int ms, int N,
              int H, int W, int cin, int cout, int relu, bool eight, cudaStream_t st) {
  if (!eight && (cin == 8 || cout == 8)) return kNotEligible;
  if (xs % 8 || ys % 8 || (uintptr_t)x % 16 || (uintptr_t)w % 16 || (uintptr_t)y % 16) return kNotEligible;
  if (mask && ((uintptr_t)mask % 16 || ms % 8)) return kNotEligible;
  const long long columns = (long long)N * ((W + kTileM - 1) / kTileM);
  if (columns > 0x7fffffff || !rows_pay(cin, cout, columns * H, sm_count())) return kNotEligible;
  cudaError_t e;
#define GBNN_ROWS_CASE(CIN_, COUT_, BN_, SLOTS_)                                                            \
  if (cin == CIN_ && cout == COUT_)                                                                         \
    e = launch_rows<BN_, CIN_, SLOTS_>(x, xs, w, bias, y, ys, mask, ms, N, H, W, cout, relu, st);           \
  else
  GBNN_ROWS_CASE(8, 32, 32, 6)
  GBNN_ROWS_CASE(32, 8, 16, 6)
  GBNN_ROWS_CASE(32, 32, 32, 6)
  GBNN_ROWS_CASE(32, 64, 64, 6)
  GBNN_ROWS_CASE(32, 96, 96, 6)
  GBNN_ROWS_CASE(64, 32, 32, 6)
  GBNN_ROWS_CASE(64, 64, 64, 6)
  GBNN_ROWS_CASE(96, 32, 32, 5)
  return kNotEligible;
#undef GBNN_ROWS_CASE
  return e == cudaSuccess ? 0 : -2;
}
