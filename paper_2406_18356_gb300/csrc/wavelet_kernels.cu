// Dictionary kernels: W = [Psi_1 .. Psi_M], Psi_m the periodized orthonormal
// 2-D Daubechies db_m transform with J levels (Sect. 4.3, App. A.1; the
// closed-form Lipschitz constant of Sect. 3.4 assumes orthogonal bases with
// circular boundaries).
//
// One analysis level on an n x n block X is Y = T X T^T, T the periodized
// analysis matrix:
//   a_i = sum_k h_k x[(2i + k) mod n],  d_i = sum_k g_k x[(2i + k) mod n],
//   g_k = (-1)^k h_{L-1-k}.
// Mallat layout: [0,h)^2 approximation, rows [0,h) x cols [h,n) low-y/high-x,
// rows [h,n) x cols [0,h) high-y/low-x, [h,n)^2 high/high, h = n/2.
// Synthesis is the transpose X = T^T Y T.
//
// Nearly every level runs in small tiles (fine_levels.cuh).  The kernel of
// this file serves what is left: the analysis levels of FP64 images of more
// than 512 pixels, and subbands whose side is no multiple of four.  It is
// register-blocked: a thread slides over 8 outputs of one row or column with
// its inputs held in registers.  Each basis is a separate template instance so
// the filter taps are compile-time constant-bank operands.
//
// The analysis kernel of the minor cycle also does FISTA's step (Algorithm 1):
// its level-1 input is the gradient image 2 (K W alpha_k - b) of the
// extrapolated point, and at each coefficient it forms
// alpha = B_k + t (B_k - B_{k-1}) and writes
// B_{k+1} = soft(alpha - g/theta, lambda/theta), so gradient coefficients
// never reach global memory.

#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace ms {

__constant__ double c_hd[kMaxBases][kMaxTaps];
__constant__ double c_gd[kMaxBases][kMaxTaps];
// FP32 coefficient pairs for the packed filters: (h_k, g_k) of the analysis
// tap k, (h_2m, h_2m+1) and (g_2m, g_2m+1) of the synthesis output pair
__constant__ float2 c_hg2[kMaxBases][kMaxTaps];
__constant__ float2 c_hh2[kMaxBases][kMaxTaps / 2];
__constant__ float2 c_gg2[kMaxBases][kMaxTaps / 2];

void set_wavelet_filters(const double* h, const int* len, int nbases) {
  double hd[kMaxBases][kMaxTaps] = {}, gd[kMaxBases][kMaxTaps] = {};
  float hf[kMaxBases][kMaxTaps] = {}, gf[kMaxBases][kMaxTaps] = {};
  for (int m = 0; m < nbases; ++m) {
    for (int k = 0; k < len[m]; ++k) {
      hd[m][k] = h[m * kMaxTaps + k];
      gd[m][k] = ((k & 1) ? -1.0 : 1.0) * h[m * kMaxTaps + len[m] - 1 - k];
      hf[m][k] = (float)hd[m][k];
      gf[m][k] = (float)gd[m][k];
    }
  }
  cudaMemcpyToSymbol(c_hd, hd, sizeof(hd));
  cudaMemcpyToSymbol(c_gd, gd, sizeof(gd));
  float2 hg[kMaxBases][kMaxTaps] = {}, hh[kMaxBases][kMaxTaps / 2] = {},
         gg[kMaxBases][kMaxTaps / 2] = {};
  for (int m = 0; m < kMaxBases; ++m)
    for (int k = 0; k < kMaxTaps; ++k) {
      hg[m][k] = make_float2(hf[m][k], gf[m][k]);
      if (k % 2 == 0) {
        hh[m][k / 2] = make_float2(hf[m][k], hf[m][k + 1]);
        gg[m][k / 2] = make_float2(gf[m][k], gf[m][k + 1]);
      }
    }
  cudaMemcpyToSymbol(c_hg2, hg, sizeof(hg));
  cudaMemcpyToSymbol(c_hh2, hh, sizeof(hh));
  cudaMemcpyToSymbol(c_gg2, gg, sizeof(gg));
}

namespace {
// Filter pairs on the FP32 pipe's packed form (fma.rn.f32x2: two lanes of
// FP32 fused multiply-add per instruction, each lane rounded as fmaf): the
// two outputs of a filter step that share their input (analysis: the low and
// high band of tap k; synthesis: outputs 2m and 2m + 1), in the same order of
// operations as the scalar chains, so results are bit-identical.  The
// coefficient pairs come from constant memory as one 64-bit operand.
// Measured at 1024^2 (FP32, M = 8, J = 4), per FISTA iteration: synthesis
// levels 4..2 29.8 -> 26.8 us, level 1 36.0 -> 33.3 us, analysis levels 2..4
// 35.5 -> 33.6 us, level 1 37.1 -> 35.1 us (144.9 -> 136.0 us in all).
// (d.x, d.y) = (c.x x + acc.x, c.y x + acc.y), c a coefficient pair read from
// constant memory as one 64-bit operand
__device__ __forceinline__ float2 ffma2_cx(const float2& c, float x, float2 acc) {
  float2 d;
  const unsigned long long cc = *reinterpret_cast<const unsigned long long*>(&c);
  asm("{\n\t.reg .b64 rx, ra, rd;\n\t"
      "mov.b64 rx, {%3, %3};\n\tmov.b64 ra, {%4, %5};\n\t"
      "fma.rn.f32x2 rd, %2, rx, ra;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "l"(cc), "f"(x), "f"(acc.x), "f"(acc.y));
  return d;
}
// analysis tap k of basis MB on input x: (a, d) += (h_k, g_k) x
template <typename R, int MB>
__device__ __forceinline__ void tap_hg(int k, R x, R& a, R& d) {
  if constexpr (sizeof(R) == 4) {
    const float2 r = ffma2_cx(c_hg2[MB][k], x, make_float2(a, d));
    a = r.x;
    d = r.y;
  } else {
    a = fma(c_hd[MB][k], x, a);
    d = fma(c_gd[MB][k], x, d);
  }
}
// synthesis taps 2m, 2m + 1 of basis MB on low input x and high input y:
// (e, o) += (h_2m, h_2m+1) x, then (e, o) += (g_2m, g_2m+1) y
template <typename R, int MB>
__device__ __forceinline__ void tap_syn(int m, R x, R y, R& e, R& o) {
  if constexpr (sizeof(R) == 4) {
    float2 r = ffma2_cx(c_hh2[MB][m], x, make_float2(e, o));
    r = ffma2_cx(c_gg2[MB][m], y, r);
    e = r.x;
    o = r.y;
  } else {
    e = fma(c_hd[MB][2 * m], x, e);
    e = fma(c_gd[MB][2 * m], y, e);
    o = fma(c_hd[MB][2 * m + 1], x, o);
    o = fma(c_gd[MB][2 * m + 1], y, o);
  }
}

constexpr int kP = 8;   // outputs per thread and direction

__host__ __device__ constexpr int round4(int x) { return (x + 3) / 4 * 4; }

// Analysis geometry for subband tiles of side AT (per block and basis): the
// staged input window, the column-filtered rows ylo / yhi and the four output
// subbands, which alias the window.  Region sizes are multiples of 4 elements
// so every region starts 16-byte aligned.  Every geometry keeps 256 threads:
// the small levels run in one wave, and there the per-block critical path
// (not occupancy) sets the time, so more threads per tile is better.
template <int AT> struct AG {
  static constexpr int T = AT;
  static constexpr int In = 2 * AT + kMaxTaps - 2;   // window side: 78, 46, 30
  static constexpr int InS = round4(In + 2);         // window row stride: 80, 48, 32
  static constexpr int YS = In + 1;                  // odd row stride of ylo / yhi
  static constexpr int GS = AT + 4;                  // 16-byte row stride of the outputs
  static constexpr int InSz = round4(In * InS);
  static constexpr int YSz = round4(AT * YS);
#ifndef MS_ANA_SMALL_THREADS
  static constexpr int Threads = 256;
#else
  static constexpr int Threads = AT >= 32 ? 256 : MS_ANA_SMALL_THREADS;
#endif
  static_assert(4 * AT * GS <= InSz, "the outputs alias the input window");
  static_assert(2 * AT * (AT / kP) <= Threads, "one thread per row unit");
};
// the widest tiles; the TMA box of the level-1 window
constexpr int kAT = 32;

// The largest power of two <= the preferred side that divides the level's
// side (sides need not be powers of two: N = 48 gives 48, 24, 12, 6).
__host__ __device__ __forceinline__ int fit_tile(int t, int n) {
  int p = 1;
  while (2 * p <= t && n % (2 * p) == 0) p *= 2;
  return p;
}
__host__ __device__ __forceinline__ int ana_tile(int h) {   // subband side
  return fit_tile(kAT, h);
}
__device__ __forceinline__ int wrap(int i, int n) {
  i %= n;
  return i < 0 ? i + n : i;
}
// periodic index for i in [-n, 2n)
__device__ __forceinline__ int wrapc(int i, int n) {
  return i < 0 ? i + n : (i >= n ? i - n : i);
}

// u / d (integer quotient) for 0 <= u < 2^22, d >= 1, through the FP32
// reciprocal inv = 1 / d: (u + 0.5) / d lies at least 0.5 / d from an
// integer, and the two roundings move it by at most (u / d) 2^-23 < 0.5 / d,
// so truncation gives the quotient (a few instructions instead of an integer
// division)
__device__ __forceinline__ int div_small(int u, float inv) {
  return (int)(((float)u + 0.5f) * inv);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(bar)),
               "r"(count)
               : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, unsigned phase) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(bar);
  for (int it = 0; it < (1 << 22); ++it) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(a), "r"(phase)
        : "memory");
    if (ok) return true;
  }
  return false;
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
      "l"((unsigned long long)map), "r"(x), "r"(y),
      "r"((unsigned)__cvta_generic_to_shared(bar))
      : "memory");
}

// first 128-byte-aligned shared address at or after p
__device__ __forceinline__ unsigned char* smem_align128(unsigned char* p) {
  const unsigned pad = (128u - (saddr(p) & 127u)) & 127u;
  return p + pad;
}

// Tile sides up to MS_COMPACT_T use the compact filters (below).
#ifndef MS_COMPACT_T
#define MS_COMPACT_T 16   // tile sides up to this use the compact filters
#endif
template <int T> constexpr bool kCompact = T <= MS_COMPACT_T;

// 8 decimated outputs from 2*8 + L - 2 inputs held in registers
template <typename R, int MB>
__device__ __forceinline__ void fir_down8(const R* x, R* lo, R* hi) {
  constexpr int L = 2 * (MB + 1);
#pragma unroll
  for (int j = 0; j < kP; ++j) {
    R a = 0, d = 0;
#pragma unroll
    for (int k = 0; k < L; ++k) tap_hg<R, MB>(k, x[2 * j + k], a, d);
    lo[j] = a;
    hi[j] = d;
  }
}

// per-thread compensated sum of |x| in the working precision (Kahan), so the
// FP64 unit only sees one value per thread
template <typename R> struct KSum {
  R s = 0, c = 0;
  __device__ __forceinline__ void add(R v) {
    R y = v - c;
    R t = s + y;
    c = (t - s) - y;
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

template <typename R> struct Vec;
template <> struct Vec<float> { using T = float4; static constexpr int N = 4; };
template <> struct Vec<double> { using T = double2; static constexpr int N = 2; };
}  // namespace

namespace {
// the four output subbands alias the input window; + alignment slack,
// block-sum scratch, mbarrier and flags
template <int AT> size_t analysis_smem_bytes(size_t rsz) {
  return (size_t)(AG<AT>::InSz + 2 * AG<AT>::YSz) * rsz + 128 +
         (AG<AT>::Threads / 32) * sizeof(double) + sizeof(uint64_t) + 2 * sizeof(int);
}
}  // namespace

// ------------------------------------------------------------------ analysis
// Small tiles (the coarse levels) run the same filters with the output loop
// rolled and the inputs read from shared memory per tap: a few times more
// shared-memory loads, a fraction of the code.  A coarse level's blocks each
// execute one basis's filter once, so its time is set by the instruction
// fetch of that code, not by the loads.  The sums are formed in the same
// order as the register-blocked versions, so results are identical.

template <typename R, int MB, class G>
__device__ __forceinline__ void analysis_filter_compact(const R* sIn, R* ylo, R* yhi, R* gout,
                                                        int TOe, int lt) {
  constexpr int L = 2 * (MB + 1);
  const int tid = threadIdx.x;
  const int nparts = TOe >> 3;
  const int cols = 2 * TOe + L - 2;
  const float inv_cols = 1.0f / (float)cols;
  for (int u = tid; u < nparts * cols; u += G::Threads) {
    const int part = div_small(u, inv_cols);
    const int col = u - part * cols;
    const R* xc = sIn + (2 * kP * part) * G::InS + col;
#pragma unroll 1
    for (int r = 0; r < kP; ++r) {
      R a = 0, d = 0;
#pragma unroll
      for (int k = 0; k < L; ++k) {
        tap_hg<R, MB>(k, xc[(2 * r + k) * G::InS], a, d);
      }
      ylo[(kP * part + r) * G::YS + col] = a;
      yhi[(kP * part + r) * G::YS + col] = d;
    }
  }
  __syncthreads();
  const int lp = lt - 3;
  const int r = tid & (TOe - 1), seg = (tid >> lt) & (nparts - 1), src = tid >> (lt + lp);
  __syncthreads();   // (the barrier pair of the register-blocked version)
  if (src >= 2) return;
  const R* yrow = (src ? yhi : ylo) + r * G::YS + 2 * kP * seg;
  R* o_lo = gout + (src ? 2 : 0) * G::T * G::GS + r * G::GS + kP * seg;
  R* o_hi = gout + (src ? 3 : 1) * G::T * G::GS + r * G::GS + kP * seg;
#pragma unroll 1
  for (int q = 0; q < kP; ++q) {
    R a = 0, d = 0;
#pragma unroll
    for (int k = 0; k < L; ++k) {
      tap_hg<R, MB>(k, yrow[2 * q + k], a, d);
    }
    o_lo[q] = a;
    o_hi[q] = d;
  }
}

// Filtering of one basis on the staged input tile: columns (y) into
// ylo / yhi, then rows (x) into the four subbands gout[0..3] =
// (approximation, low-y/high-x, high-y/low-x, high/high), G::T x G::GS each.
// TOe (a power of two, 8..G::T) outputs per subband side, lt = log2(TOe).
template <typename R, int MB, class G>
__device__ __forceinline__ void analysis_filter(const R* sIn, R* ylo, R* yhi, R* gout, int TOe,
                                                int lt) {
  constexpr int L = 2 * (MB + 1);
  constexpr int NI = 2 * kP + L - 2;
  const int tid = threadIdx.x;
  const int nparts = TOe >> 3;
  const int cols = 2 * TOe + L - 2;
  if constexpr (kCompact<G::T>) {
    analysis_filter_compact<R, MB, G>(sIn, ylo, yhi, gout, TOe, lt);
  } else {
    const float inv_cols = 1.0f / (float)cols;
    for (int u = tid; u < nparts * cols; u += G::Threads) {
      int part = div_small(u, inv_cols);
      int col = u - part * cols;
      R xin[NI];
#pragma unroll
      for (int i = 0; i < NI; ++i) xin[i] = sIn[(2 * kP * part + i) * G::InS + col];
      R lo[kP], hi[kP];
      fir_down8<R, MB>(xin, lo, hi);
#pragma unroll
      for (int r = 0; r < kP; ++r) {
        ylo[(kP * part + r) * G::YS + col] = lo[r];
        yhi[(kP * part + r) * G::YS + col] = hi[r];
      }
    }
    __syncthreads();
    // rows: unit = (row r, segment, source); a warp takes consecutive rows of
    // one segment
    const int lp = lt - 3;   // log2(nparts)
    const int r = tid & (TOe - 1), seg = (tid >> lt) & (nparts - 1), src = tid >> (lt + lp);
    const bool active = src < 2;
    R xin[NI];
    if (active) {
      const R* yrow = (src ? yhi : ylo) + r * G::YS + 2 * kP * seg;
#pragma unroll
      for (int i = 0; i < NI; ++i) xin[i] = yrow[i];
    }
    __syncthreads();   // the outputs overwrite the input tile
    if (!active) return;
    R lo[kP], hi[kP];
    fir_down8<R, MB>(xin, lo, hi);
    R* o_lo = gout + (src ? 2 : 0) * G::T * G::GS + r * G::GS + kP * seg;
    R* o_hi = gout + (src ? 3 : 1) * G::T * G::GS + r * G::GS + kP * seg;
    using V = typename Vec<R>::T;
    constexpr int NV = Vec<R>::N;
#pragma unroll
    for (int q = 0; q < kP; q += NV) {
      *reinterpret_cast<V*>(o_lo + q) = *reinterpret_cast<const V*>(lo + q);
      *reinterpret_cast<V*>(o_hi + q) = *reinterpret_cast<const V*>(hi + q);
    }
  }
}

// shared-memory layout of an analysis block (after the 128-byte alignment)
template <typename R, class G> struct AnaSmem {
  R* sIn;        // [G::In][G::InS]; later the outputs [4][G::T][G::GS]
  R* ylo;        // [G::T][G::YS]
  R* yhi;
  double* red;   // [G::Threads / 32]
  uint64_t* bar;
  int* flags;    // [2]
  __device__ __forceinline__ explicit AnaSmem(unsigned char* base) {
    sIn = reinterpret_cast<R*>(base);
    ylo = sIn + G::InSz;
    yhi = ylo + G::YSz;
    red = reinterpret_cast<double*>(yhi + G::YSz);
    bar = reinterpret_cast<uint64_t*>(red + G::Threads / 32);
    flags = reinterpret_cast<int*>(bar + 1);
  }
};

// One analysis work item: subband tile `tile` (of side TO <= G::T) of level
// j for basis MB.  n = N >> (j-1) is the input side, h = n/2 the subband side.
// MODE 0: plain analysis (W^H x); input x (level 1) or LL_{j-1}.
// MODE 1: FISTA step; level 1 input is the gradient image 2 (K W alpha_k - b);
//         detail (and level-J approximation) outputs go through the prox into
//         B_{k+1} and |B_{k+1}| accumulates into l1.
// With the widest geometry, level 1 stages its 78 x 78 input window by one
// TMA tensor copy when the window lies inside the image (the caller has
// initialized the mbarrier and tracks its phase); other windows are staged by
// cp.async with periodic wrap.  Ends with a block barrier, so the caller may
// reuse the shared buffers.
template <typename R, int MODE, int MB, class G>
__device__ __forceinline__ void analysis_item(unsigned char* base, const CUtensorMap* xmap,
                                              bool use_tma, unsigned& phase, const R* x_in,
                                              const R* ll_in, R* ll_out, R* out_plain,
                                              const R* cur, const R* prev, R* next, R t, R mu,
                                              R thr, int N, int j, int J, int tile,
                                              FistaCtl* ctl, KSum<R>& l1, int tma_y0) {
  constexpr int m = MB;
  const AnaSmem<R, G> sm(base);
  R* sIn = sm.sIn;
  R* gout = sIn;

  const int n = N >> (j - 1), h = n / 2;
  const int TO = ana_tile(h);
  const int TOe = TO < kP ? kP : TO;             // outputs computed per side
  const int lt = 31 - __clz(TOe);
  const int lto = 31 - __clz(TO);
  const int ext = 2 * TOe + kMaxTaps - 2;        // staged input window side
  const int tiles_x = h / TO;
  const int o0y = (tile / tiles_x) * TO, o0x = (tile % tiles_x) * TO;
  const int p0y = 2 * o0y, p0x = 2 * o0x;
  constexpr int NV = Vec<R>::N;
  constexpr int LNV = NV == 4 ? 2 : 1;
  using V = typename Vec<R>::T;
  const bool vec = (TO % NV) == 0;
  const int64_t plane = (int64_t)m * N * N;
  // coefficient-plane offset of (subband s = 1..3, row, col) of this tile
  auto coef_off = [&](int s, int row, int col) -> int64_t {
    int rr = (s >= 2 ? h : 0) + o0y + row;
    int cc = (s & 1 ? h : 0) + o0x + col;
    return plane + (int64_t)rr * N + cc;
  };

  // The TMA copy is issued only after checking its alignment rules (128-byte
  // shared destination, 64-byte descriptor, 16-byte start column); a
  // violation is recorded in ctl->error (MS_ERR_UNSUPPORTED) and the window
  // is staged by cp.async instead.
  bool tma = G::T == kAT && use_tma && j == 1 && TO == kAT && p0x + G::InS <= n &&
             p0y + G::In <= n;
  if (tma) {
    if (threadIdx.x == 0) {
      const bool aligned = (saddr(sIn) & 127u) == 0 &&
                           (reinterpret_cast<uintptr_t>(xmap) & 63u) == 0 &&
                           ((p0x * (int)sizeof(R)) & 15) == 0;
      sm.flags[1] = aligned ? 1 : 0;
      if (aligned) {
        // order the block's earlier generic accesses of the window before
        // the asynchronous copy overwrites it
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(sm.bar, (unsigned)(G::In * G::InS * sizeof(R)));
        tma_load_2d(sIn, xmap, p0x, p0y + tma_y0, sm.bar);
      } else if (ctl) {
        atomicExch(&ctl->error, 8);
      }
    }
    __syncthreads();
    tma = sm.flags[1] != 0;
  }

  if (!tma) {
    // stage the input window with periodic wrap
    const R* src = (j == 1) ? x_in : ll_in + (int64_t)m * n * n;
    const bool cheap = n >= ext;   // positions lie in [0, n + ext)
    constexpr int V16 = 16 / (int)sizeof(R);
    const int nch = (ext + V16 - 1) / V16;
    if (p0x + nch * V16 <= n && (n % V16) == 0) {
      // the window's columns need no wrap: whole 16-byte chunks per row
      // (p0x = 2 o0x is a multiple of 16), rows wrap
      for (int e = threadIdx.x; e < ext * nch; e += G::Threads) {
        const int a = e / nch, c = e - a * nch;
        const int py = cheap ? wrapc(p0y + a, n) : wrap(p0y + a, n);
        cp_async<16>(sIn + a * G::InS + c * V16, src + (int64_t)py * n + p0x + c * V16);
      }
    } else {
      const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
      constexpr int NW = G::Threads / 32;
      for (int a = warp; a < ext; a += NW) {
        const int py = cheap ? wrapc(p0y + a, n) : wrap(p0y + a, n);
        const R* row = src + (int64_t)py * n;
        for (int b = lane; b < ext; b += 32) {
          const int px = cheap ? wrapc(p0x + b, n) : wrap(p0x + b, n);
          cp_async<sizeof(R)>(sIn + a * G::InS + b, row + px);
        }
      }
    }
    cp_async_commit();
  }

  bool skip = false;
  if (tma) {
    // bounded wait for the window; on time-out the tile is skipped (the
    // error is recorded) but every barrier is still passed
    const bool ok = mbar_wait_bounded(sm.bar, phase);
    phase ^= 1u;
    skip = __syncthreads_or(!ok) != 0;
    if (skip && threadIdx.x == 0 && ctl) atomicExch(&ctl->error, 5);
  } else {
    cp_async_wait<0>();
  }
  __syncthreads();
  if (!skip) {
    analysis_filter<R, MB, G>(sIn, sm.ylo, sm.yhi, gout, TOe, lt);
  } else {
    __syncthreads();   // the filter's two barriers
    __syncthreads();
  }
  __syncthreads();

  // write / update the tile's coefficients
  auto prox = [&](R g, R bc, R bp) -> R {
    R alpha = bc + t * (bc - bp);
    R z = alpha - mu * g;
    R az = fabs(z) - thr;
    R nb = az > (R)0 ? copysign(az, z) : (R)0;
    l1.add(fabs(nb));
    return nb;
  };
  if (skip) {
    // nothing is written for a tile whose window never arrived
  } else if (vec) {
    const int lpr = lto - LNV;    // log2(vectors per tile row)
    const int s_first = (j == J) ? 0 : 1;
    const int lsub = lto + lpr;   // log2(vectors per subband tile)
    const int items = (4 - s_first) << lsub;
    for (int e = threadIdx.x; e < items; e += G::Threads) {
      int s = s_first + (e >> lsub);
      int rem = e & ((1 << lsub) - 1);
      int row = rem >> lpr, c4 = (rem & ((1 << lpr) - 1)) << LNV;
      V gv = *reinterpret_cast<const V*>(gout + (s * G::T + row) * G::GS + c4);
      int64_t off = s ? coef_off(s, row, c4) : plane + (int64_t)(o0y + row) * N + o0x + c4;
      if (MODE == 0) {
        *reinterpret_cast<V*>(out_plain + off) = gv;
      } else {
        V cv = *reinterpret_cast<const V*>(cur + off);
        V pv = *reinterpret_cast<const V*>(prev + off);
        V nv;
        R* np = reinterpret_cast<R*>(&nv);
        const R* gp = reinterpret_cast<const R*>(&gv);
        const R* cp = reinterpret_cast<const R*>(&cv);
        const R* pp = reinterpret_cast<const R*>(&pv);
#pragma unroll
        for (int q = 0; q < NV; ++q) np[q] = prox(gp[q], cp[q], pp[q]);
        *reinterpret_cast<V*>(next + off) = nv;
      }
    }
    if (j < J) {   // approximation feeds the next level
      for (int e = threadIdx.x; e < (1 << lsub); e += G::Threads) {
        int row = e >> lpr, c4 = (e & ((1 << lpr) - 1)) << LNV;
        *reinterpret_cast<V*>(ll_out + (int64_t)m * h * h + (int64_t)(o0y + row) * h + o0x + c4) =
            *reinterpret_cast<const V*>(gout + row * G::GS + c4);
      }
    }
  } else {   // tiny levels: scalar path
    const int s_first = (j == J) ? 0 : 1;
    for (int e = threadIdx.x; e < 4 * TO * TO; e += G::Threads) {
      int s = e / (TO * TO);
      int row = (e / TO) % TO, col = e % TO;
      R gval = gout[(s * G::T + row) * G::GS + col];
      if (s == 0 && j < J) {
        ll_out[(int64_t)m * h * h + (int64_t)(o0y + row) * h + o0x + col] = gval;
        continue;
      }
      if (s < s_first) continue;
      int64_t off = s ? coef_off(s, row, col) : plane + (int64_t)(o0y + row) * N + o0x + col;
      if (MODE == 0)
        out_plain[off] = gval;
      else
        next[off] = prox(gval, cur[off], prev[off]);
    }
  }
  __syncthreads();
}

// MODE 1: level j of the minor cycle's analysis + FISTA update.  The spectral
// kernel of this pass has already advanced ctl->k, so this builds B_{k+1}
// with k = ctl->k - 1; each block leaves its sum of |B_{k+1}| over its tile
// in l1_parts[part_base + block] (the next spectral kernel adds them up, in a
// fixed order).  MODE 0: level j of plain = W^H a.grad.  blockIdx.x = subband
// tile, blockIdx.y = basis.
template <typename R, int MODE, int AT>
__global__ void __launch_bounds__(AG<AT>::Threads, 512 / AG<AT>::Threads)
    analysis_level_kernel(const __grid_constant__ CUtensorMap xmap, FistaPass<R> a_, R* plain,
                          int j, int use_tma, int part_base) {
  using G = AG<AT>;
  const FistaPass<R> a = job_slice(a_);   // blockIdx.z: the job (batched form)
  pdl_wait();
  pdl_trigger();
  R t = 0, mu = 0, thr = 0;
  const R *cur = nullptr, *prev = nullptr;
  R* next = nullptr;
  if (MODE == 1) {
    const int done = a.ctl->done;
    const int k = a.ctl->k - 1;
    if (done) return;   // uniform: `done` does not change during this kernel
    t = ctl_t<R>(a.ctl, k & 1);   // momentum t_k
    mu = ctl_mu<R>(a.ctl);        // 1 / theta
    thr = ctl_thr<R>(a.ctl);      // lambda / theta
    cur = k % 3 == 0 ? a.B0 : (k % 3 == 1 ? a.B1 : a.B2);
    prev = k % 3 == 0 ? a.B2 : (k % 3 == 1 ? a.B0 : a.B1);
    next = k % 3 == 0 ? a.B1 : (k % 3 == 1 ? a.B2 : a.B0);
  }
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* base = smem_align128(smem_raw);
  const AnaSmem<R, G> sm(base);
  const bool tma = G::T == kAT && use_tma != 0 && j == 1;
  if (tma && threadIdx.x == 0) mbar_init(sm.bar, 1);
  __syncthreads();
  unsigned phase = 0;
  KSum<R> l1;
  const int64_t half = (int64_t)a.M * (a.N / 2) * (a.N / 2);
  const R* ll_in = (j == 1) ? nullptr : a.tmp + ((j - 1) & 1) * half;
  R* ll_out = a.tmp + (j & 1) * half;
  switch (blockIdx.y) {
#define MS_ANA(MBV)                                                                            \
  case MBV:                                                                                    \
    analysis_item<R, MODE, MBV, G>(base, &xmap, tma, phase, a.grad, ll_in, ll_out, plain, cur, \
                                   prev, next, t, mu, thr, a.N, j, a.J, blockIdx.x,            \
                                   MODE == 1 ? a.ctl : nullptr, l1, (int)blockIdx.z * a.N);    \
    break;
    MS_ANA(0) MS_ANA(1) MS_ANA(2) MS_ANA(3) MS_ANA(4) MS_ANA(5) MS_ANA(6) MS_ANA(7)
#undef MS_ANA
  }
  if (MODE == 0) return;
  // block sum of |B_{k+1}|: error-free working-precision warp sums, FP64
  // once per warp
  R hi = l1.s, lo = -l1.c;
  warp_sum_comp<R>(hi, lo);
  if ((threadIdx.x & 31) == 0) sm.red[threadIdx.x >> 5] = (double)hi + (double)lo;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int q = 0; q < G::Threads / 32; ++q) sum += sm.red[q];
    a.l1_parts[part_base + (int64_t)blockIdx.y * gridDim.x + blockIdx.x] = sum;
  }
}

#include "fine_levels.cuh"

// ------------------------------------------------------------- dispatch
namespace {
// The kernel of an analysis level with subbands of side h.  Tiles of 16 (a
// thread forms 4 outputs of a row or column) where that makes a block for
// nearly every SM (8 bases x 16 tiles at h = 64), else tiles of 8 or 4 with
// an output per thread; FP64, whose time is the FP64 instructions of the
// busiest scheduler, takes tiles of 8 up to h = 128 and of 16 at 256, and
// above that the wide register-blocked tiles (fewest halo columns filtered
// twice).  Measured per level, us (this rule's | the alternatives'): FP32
// h = 512 27.7 | 31.7 (one block per tile over all bases); h = 256..64
// together 26 | 26.7 in one cooperative launch of full-width strips, and 120
// against 133 per iteration at 1024 px with both directions' coarse levels
// replaced; FP64, an iteration at 128 px with h = 64..8: 155 | 219, at 256
// px 301 | 337 with tiles of 16, at 1024 px with h = 512 wide 1549 | 1715
// with tiles of 16.  The plain FP64 transform has no prox operands in flight:
// tiles of 8 below h = 256 (8 bases, h = 192: 62 | 80 with 16; 256: 101 | 96),
// then of 16 (h = 384: 197 | 203 wide, 512: 346 | 352) until some 4500 wide
// tiles keep the SMs evenly busy (h = 768: 740 wide | 772; 4 bases 211 | 203).
enum class Ana { kWide, k16, k8, k4 };
Ana ana_kernel(bool f64, bool plain, int h, int M) {
  if (f64 && plain && h % 8 == 0 && h < 256) return Ana::k8;
  if (f64 && plain && h % 16 == 0 && (int64_t)h * h * M < 4500 * 32 * 32) return Ana::k16;
  if (f64 && h > 256) return h % 16 == 0 ? Ana::kWide : (h % 4 == 0 ? Ana::k4 : Ana::kWide);
  if (h % 16 == 0 && h >= (f64 ? 129 : 64)) return Ana::k16;
  if (h % 8 == 0) return Ana::k8;
  return h % 4 == 0 ? Ana::k4 : Ana::kWide;
}
int ana_side(bool f64, bool plain, int h, int M) {
  switch (ana_kernel(f64, plain, h, M)) {
    case Ana::k16: return 16;
    case Ana::k8: return 8;
    case Ana::k4: return 4;
    default: return ana_tile(h);
  }
}
// The kernel of a synthesis level j >= 2 with output side n, M bases and
// `jobs` jobs: tiles of 32 or 16 (4 or 2 output pairs per unit) where they
// make some 1000 or 500 blocks, else of 8.  Measured at 1024 px, FP32, one
// job, us an iteration: (n = 512, 256, 128) in tiles of (32, 16, 16) 128,
// (32, 32, 16) 132 and 136, (16, 16, 16) 134; 8 jobs: (32, 32, 32) 89.9 a
// job, (16, 16, 16) 95.1.  FP64: 32 (2 pairs, 256 threads) from 512 blocks on
// (8 bases, us a level, 32 | 16 | 8: n = 384 48 | 60 | 75, 512 81 | 103 | 132,
// 8 jobs at 128 54 | 62 | 71; n = 256, 512 blocks, 36 | 37 | 35), else 16 from
// 512 on and 8 below (the fewest instructions in the busiest scheduler).
enum class Syn { k32, k16, k8, k4, k2 };
Syn syn_kernel(bool f64, int n, int M, int jobs) {
  auto blocks = [&](int t) { return (int64_t)(n / t) * (n / t) * M * jobs; };
  const Syn small = n % 8 == 0 ? Syn::k8 : (n % 4 == 0 ? Syn::k4 : Syn::k2);
  if (f64 && n % 32 == 0 && blocks(32) >= 512) return Syn::k32;
  if (f64) return n >= 512 && n % 16 == 0 ? Syn::k16 : small;
  if (n % 32 == 0 && blocks(32) >= 1000) return Syn::k32;
  if (n % 16 == 0 && blocks(16) >= 500) return Syn::k16;
  return small;
}

template <typename R, int MODE>
cudaError_t launch_analysis_level(const FistaPass<R>& a, R* plain, const CUtensorMap* grad_map,
                                  int j, int part_base, cudaStream_t s) {
  const int h = a.N >> j, T = ana_side(sizeof(R) == 8, MODE == 0, h, a.M);
  const dim3 grid((h / T) * (h / T), a.M, a.js.jobs);
  switch (ana_kernel(sizeof(R) == 8, MODE == 0, h, a.M)) {
    case Ana::k16:
      return launch_pdl(fine_analysis_kernel<R, MODE, 16, 16, 4, 128>, grid, dim3(128), 0, s, a,
                        plain, j, part_base);
    case Ana::k8:
      return launch_pdl(fine_analysis_kernel<R, MODE, 8, 8, 1, 128>, grid, dim3(128), 0, s, a,
                        plain, j, part_base);
    case Ana::k4:
      return launch_pdl(fine_analysis_kernel<R, MODE, 4, 4, 1, 64>, grid, dim3(64), 0, s, a,
                        plain, j, part_base);
    default: break;
  }
  const CUtensorMap m = grad_map ? *grad_map : CUtensorMap{};
  auto go = [&](auto kern, int threads, size_t smem) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    return launch_pdl(kern, grid, dim3(threads), smem, s, m, a, plain, j, grad_map ? 1 : 0,
                      part_base);
  };
  if constexpr (sizeof(R) == 8) {   // (FP32: subbands no multiple of 4, tiles of 1 or 2)
    if (T >= 32)
      return go(analysis_level_kernel<R, MODE, 32>, AG<32>::Threads,
                analysis_smem_bytes<32>(sizeof(R)));
    if (T >= 16)
      return go(analysis_level_kernel<R, MODE, 16>, AG<16>::Threads,
                analysis_smem_bytes<16>(sizeof(R)));
  }
  return go(analysis_level_kernel<R, MODE, 8>, AG<8>::Threads, analysis_smem_bytes<8>(sizeof(R)));
}

// Level j of the synthesis of B_k (plain NULL) or of `plain` into a.x
template <typename R>
cudaError_t launch_synthesis_level(const FistaPass<R>& a, const R* plain, int j, cudaStream_t s) {
  const int n = 2 * (a.N >> j), jobs = a.js.jobs;
  const bool f64 = sizeof(R) == 8;
  if (j == 1) {
    // FP32 below 256 px, and FP64 below some 218 tiles of 32 pixels: a warp per
    // basis (at 128 px, FP64: 24.6 us an iteration less than one block per
    // 16-pixel tile).  FP64 above: the sum kernel, an output pair a thread (us
    // a level, 8 bases, warps | sum: 320 px 49 | 54, 448 px 90 | 100, 512 px
    // 118 | 100, 768 px 235 | 197, 2048 px 1595 | 1312; one basis at 1024 px 36
    // | 13; 8 jobs at 512 px 806 | 681).
    auto go = [&](auto kern, int ty, int tx, size_t elems) {
      const size_t smem = kMaxBases * elems * sizeof(R);
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      return launch_pdl(kern, dim3((n / ty) * (n / tx), 1, jobs), dim3(32 * kMaxBases), smem, s, a,
                        plain);
    };
    if (f64 && (int64_t)(n / 8) * (n / 16) * jobs < 256)
      return go(fine_synthesis_l1_kernel<R, 8, 16, 1>, 8, 16, FineSyn<8, 16>::Elems);
    const int64_t tiles = (int64_t)(n / 32) * (n / 32) * jobs;
    if (n < 256 || n % 32 || (f64 && tiles < 218))
      return go(fine_synthesis_l1_kernel<R, 16, 16, 2>, 16, 16, FineSyn<16, 16>::Elems);
    auto sum = [&](auto kern, int threads) {
      return launch_pdl(kern, dim3((n / 32) * (n / 32), 1, jobs), dim3(threads), 0, s, a, plain);
    };
    if constexpr (sizeof(R) == 8) {
      return sum(fine_synthesis_sum_kernel<R, 32, 32, 1, 512>, 512);
    } else {
      // 4 output pairs a thread (fewest shared-memory loads) where the tiles
      // occupy the SMs several times over, else 2 by twice the threads.
      // Measured, us an iteration and job (4 | 2): 256 px 58.6 | 44.9, 512 px
      // 73.6 | 65.1, 4 jobs at 512 px 30.5 | 31.1, 1024 px 109.4 | 110.7.
      if (tiles >= 1000) return sum(fine_synthesis_sum_kernel<R, 32, 32, 4, 128>, 128);
      return sum(fine_synthesis_sum_kernel<R, 32, 32, 2, 256>, 256);
    }
  }
  auto go = [&](auto kern, int t, int threads) {
    return launch_pdl(kern, dim3((n / t) * (n / t), a.M, jobs), dim3(threads), 0, s, a, plain, j);
  };
  switch (syn_kernel(f64, n, a.M, jobs)) {
    case Syn::k32:
      if constexpr (sizeof(R) == 4) return go(fine_synthesis_kernel<R, 32, 32, 4, 128>, 32, 128);
      else return go(fine_synthesis_kernel<R, 32, 32, 2, 256>, 32, 256);
    case Syn::k16: return go(fine_synthesis_kernel<R, 16, 16, 2, 128>, 16, 128);
    case Syn::k8: return go(fine_synthesis_kernel<R, 8, 8, 1, 128>, 8, 128);
    case Syn::k4: return go(fine_synthesis_kernel<R, 4, 4, 1, 64>, 4, 64);
    default: break;
  }
  return go(fine_synthesis_kernel<R, 2, 2, 1, 32>, 2, 32);
}
}  // namespace

int analysis_prox_partials(WaveletGeom g, size_t rsz) {
  int total = 0;
  for (int j = 1; j <= g.J; ++j) {
    const int h = g.N >> j, T = ana_side(rsz == 8, false, h, g.M);
    total += (h / T) * (h / T) * g.M;
  }
  return total;
}

namespace {
// a pass that only names the images and the geometry (plain transforms)
template <typename R> FistaPass<R> plain_pass(const R* grad, R* x, R* tmp, WaveletGeom g) {
  FistaPass<R> a{};
  a.grad = grad;
  a.x = x;
  a.tmp = tmp;
  a.N = g.N;
  a.J = g.J;
  a.M = g.M;
  return a;
}
}  // namespace

template <typename R>
cudaError_t launch_synthesis(const R* coef, R* x, R* tmp, WaveletGeom g, cudaStream_t s) {
  const FistaPass<R> a = plain_pass<R>(nullptr, x, tmp, g);
  for (int j = g.J; j >= 1; --j) {
    const cudaError_t e = launch_synthesis_level<R>(a, coef, j, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename R>
cudaError_t launch_analysis(const R* x, R* coef, R* tmp, WaveletGeom g, cudaStream_t s) {
  const FistaPass<R> a = plain_pass<R>(x, nullptr, tmp, g);
  for (int j = 1; j <= g.J; ++j) {
    const cudaError_t e = launch_analysis_level<R, 0>(a, coef, nullptr, j, 0, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// TMA box of the level-1 input window: {80 columns, 78 rows}
void analysis_window_box(unsigned* cols, unsigned* rows) {
  *cols = AG<kAT>::InS;
  *rows = AG<kAT>::In;
}

template <typename R>
cudaError_t launch_synthesis_pass(const FistaPass<R>& a, cudaStream_t s, int only_level) {
  for (int j = a.J; j >= 1; --j) {
    if (only_level > 0 && j != only_level) continue;
    if (only_level < 0 && j == 1) continue;
    const cudaError_t e = launch_synthesis_level<R>(a, nullptr, j, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename R>
cudaError_t launch_analysis_pass(const FistaPass<R>& a, const CUtensorMap* grad_map,
                                 cudaStream_t s, int only_level) {
  int part_base = 0;
  for (int j = 1; j <= a.J; ++j) {
    const int h = a.N >> j, T = ana_side(sizeof(R) == 8, false, h, a.M);
    if (only_level == 0 || j == only_level || (only_level < 0 && j > 1)) {
      const cudaError_t e = launch_analysis_level<R, 1>(a, nullptr, grad_map, j, part_base, s);
      if (e != cudaSuccess) return e;
    }
    part_base += (h / T) * (h / T) * a.M;
  }
  return cudaSuccess;
}

#define MS_INST(R)                                                                              \
  template cudaError_t launch_synthesis<R>(const R*, R*, R*, WaveletGeom, cudaStream_t);        \
  template cudaError_t launch_analysis<R>(const R*, R*, R*, WaveletGeom, cudaStream_t);         \
  template cudaError_t launch_synthesis_pass<R>(const FistaPass<R>&, cudaStream_t, int);        \
  template cudaError_t launch_analysis_pass<R>(const FistaPass<R>&, const CUtensorMap*,         \
                                               cudaStream_t, int);
MS_INST(float)
MS_INST(double)
#undef MS_INST

}  // namespace ms
