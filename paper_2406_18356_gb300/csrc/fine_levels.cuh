// Wavelet levels of the minor cycle in small tiles: one block per (tile,
// basis), threads that form a few outputs each.  Included by
// wavelet_kernels.cu, whose filter taps, wrapping and sums it uses.
//
// The register-blocked kernels give a thread 8 outputs of a row or column and
// a block a 16 to 64 pixel tile: right for wide levels, but a level of a few
// thousand coefficients then runs a handful of warps on a fraction of the
// SMs.  Here a unit of work is U outputs of one column or row, and tiles are
// small enough for every level to fill the SMs.  Every output is the same
// chain of multiply-adds in the same order, so coefficients and images do not
// depend on which kernel ran a level.

// exact quotient of 0 <= u < 2^22 by a compile-time divisor's reciprocal
template <int D> __device__ __forceinline__ int div_const(int u) {
  return (D & (D - 1)) == 0 ? u / D : div_small(u, 1.0f / (float)D);
}

// ------------------------------------------------------------- analysis
// Level j of basis MB on one subband tile of TY x TX outputs: input window by
// cp.async (periodic), columns into ylo / yhi, rows into the prox (or, at
// MODE 0, the coefficients).  As analysis_item; U outputs per unit.
template <int TY, int TX> struct FineAna {
  static constexpr int InY = 2 * TY + kMaxTaps - 2, InX = 2 * TX + kMaxTaps - 2;
  static constexpr int XS = round4(InX + 2);                 // window row stride
  // filtered-row stride 1 mod 8: rows and segments of 4 outputs then fall in
  // different banks (FP32)
  static constexpr int YS = (InX + 6) / 8 * 8 + 1;
  static constexpr int Elems = InY * XS + 2 * TY * YS;
};

template <typename R, int MODE, int MB, int TY, int TX, int U, int THREADS>
__device__ __forceinline__ void fine_analysis_item(R* smem, const R* __restrict__ src,
                                                   R* __restrict__ ll_out, R* __restrict__ out,
                                                   const R* __restrict__ cur,
                                                   const R* __restrict__ prev, R t, R mu, R thr,
                                                   int N, int n, bool last, int tile,
                                                   KSum<R>& l1) {
  using G = FineAna<TY, TX>;
  constexpr int L = 2 * (MB + 1);
  constexpr int rows_in = 2 * TY + L - 2, cols = 2 * TX + L - 2;
  R* sx = smem;
  R* ylo = sx + G::InY * G::XS;
  R* yhi = ylo + TY * G::YS;
  const int h = n / 2, tiles_x = h / TX;
  const int o0y = tile / tiles_x * TY, o0x = (tile - tile / tiles_x * tiles_x) * TX;
  const int p0y = 2 * o0y, p0x = 2 * o0x;
  const int tid = threadIdx.x;
  // the window: whole 16-byte chunks where no column wraps and rows start
  // aligned (n and TX multiples of the chunk), else element by element
  constexpr int V = 16 / (int)sizeof(R);
  constexpr int nch = (cols + V - 1) / V;
  if ((2 * TX) % V == 0 && n % V == 0 && p0x + nch * V <= n &&
      (reinterpret_cast<uintptr_t>(src) & 15) == 0) {
    for (int e = tid; e < rows_in * nch; e += THREADS) {
      const int a = div_const<nch>(e), c = e - a * nch;
      int py = p0y + a;
      py = py < 2 * n ? wrapc(py, n) : py % n;
      cp_async<16>(sx + a * G::XS + c * V, src + (int64_t)py * n + p0x + c * V);
    }
  } else {
    for (int e = tid; e < rows_in * cols; e += THREADS) {
      const int a = div_const<cols>(e), c = e - a * cols;
      int py = p0y + a, px = p0x + c;
      py = py < 2 * n ? wrapc(py, n) : py % n;
      px = px < 2 * n ? wrapc(px, n) : px % n;
      cp_async<sizeof(R)>(sx + a * G::XS + c, src + (int64_t)py * n + px);
    }
  }
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  // columns: unit = (column, group of U output rows)
  constexpr int NI = 2 * U + L - 2;
  for (int u = tid; u < (TY / U) * cols; u += THREADS) {
    const int g = div_const<cols>(u), x = u - g * cols;
    const R* s = sx + 2 * U * g * G::XS + x;
    R xin[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) xin[i] = s[i * G::XS];
#pragma unroll
    for (int r = 0; r < U; ++r) {
      R a = 0, d = 0;
#pragma unroll
      for (int k = 0; k < L; ++k) tap_hg<R, MB>(k, xin[2 * r + k], a, d);
      ylo[(U * g + r) * G::YS + x] = a;
      yhi[(U * g + r) * G::YS + x] = d;
    }
  }
  __syncthreads();
  // rows: unit = (segment of U outputs, row, source lo / hi), segments fastest
  constexpr int segs = TX / U;
  const int64_t plane = (int64_t)MB * N * N;
  for (int u = tid; u < 2 * TY * segs; u += THREADS) {
    const int seg = u % segs, r = u / segs % TY, hi = u / (segs * TY);
    const int row = o0y + r, col = o0x + U * seg;
    // a: approximation (lo) or high-y/low-x (hi); d: low-y/high-x or high/high
    const int64_t off_a = plane + (int64_t)(hi ? h + row : row) * N + col;
    const int64_t off_d = off_a + h;
    const bool keep_a = hi || last;
    // U * sizeof(R) bytes at a time: col, h and N are multiples of U
    struct alignas(U * sizeof(R) < 16 ? U * sizeof(R) : 16) Pack { R v[U]; };
    Pack ca{}, pa{}, cd{}, pd{};
    if (MODE == 1) {   // the prox operands, in flight while the filter runs
      cd = *reinterpret_cast<const Pack*>(cur + off_d);
      pd = *reinterpret_cast<const Pack*>(prev + off_d);
      if (keep_a) {
        ca = *reinterpret_cast<const Pack*>(cur + off_a);
        pa = *reinterpret_cast<const Pack*>(prev + off_a);
      }
    }
    const R* y = (hi ? yhi : ylo) + r * G::YS + 2 * U * seg;
    R xin[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) xin[i] = y[i];
    Pack a, d;
#pragma unroll
    for (int q = 0; q < U; ++q) {
      R s0 = 0, s1 = 0;
#pragma unroll
      for (int k = 0; k < L; ++k) tap_hg<R, MB>(k, xin[2 * q + k], s0, s1);
      a.v[q] = s0;
      d.v[q] = s1;
    }
    auto prox = [&](Pack& g, const Pack& c, const Pack& p) {
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const R alpha = c.v[q] + t * (c.v[q] - p.v[q]);
        const R z = alpha - mu * g.v[q];
        const R az = fabs(z) - thr;
        const R nb = az > (R)0 ? copysign(az, z) : (R)0;
        l1.add(fabs(nb));
        g.v[q] = nb;
      }
    };
    if (keep_a) {
      if (MODE == 1) prox(a, ca, pa);
      *reinterpret_cast<Pack*>(out + off_a) = a;
    } else {
      *reinterpret_cast<Pack*>(ll_out + (int64_t)MB * h * h + (int64_t)row * h + col) = a;
    }
    if (MODE == 1) prox(d, cd, pd);
    *reinterpret_cast<Pack*>(out + off_d) = d;
  }
}

// MODE 1: level j of the minor cycle's analysis + FISTA update (as
// analysis_level_kernel); MODE 0: of the plain analysis of a.grad into out.
// blockIdx.x = tile, blockIdx.y = basis, the longest filters first.
template <typename R, int MODE, int TY, int TX, int U, int THREADS>
__global__ void __launch_bounds__(THREADS)
    fine_analysis_kernel(FistaPass<R> a_, R* plain, int j, int part_base) {
  const FistaPass<R> a = job_slice(a_);   // blockIdx.z: the job (batched form)
  pdl_wait();
  pdl_trigger();
  R t = 0, mu = 0, thr = 0;
  const R *cur = nullptr, *prev = nullptr;
  R* next = plain;
  if (MODE == 1) {
    if (a.ctl->done) return;   // uniform: `done` does not change during this kernel
    const int k = a.ctl->k - 1;
    t = ctl_t<R>(a.ctl, k & 1);
    mu = ctl_mu<R>(a.ctl);
    thr = ctl_thr<R>(a.ctl);
    cur = k % 3 == 0 ? a.B0 : (k % 3 == 1 ? a.B1 : a.B2);
    prev = k % 3 == 0 ? a.B2 : (k % 3 == 1 ? a.B0 : a.B1);
    next = k % 3 == 0 ? a.B1 : (k % 3 == 1 ? a.B2 : a.B0);
  }
  __shared__ __align__(16) R smem[FineAna<TY, TX>::Elems];
  const int64_t half = (int64_t)a.M * (a.N / 2) * (a.N / 2);
  const int n = a.N >> (j - 1);
  const int m = a.M - 1 - (int)blockIdx.y;
  const R* src = j == 1 ? a.grad : a.tmp + ((j - 1) & 1) * half + (int64_t)m * n * n;
  R* ll_out = a.tmp + (j & 1) * half;
  KSum<R> l1;
  switch (m) {
#define MS_FA(MBV)                                                                               \
  case MBV:                                                                                      \
    fine_analysis_item<R, MODE, MBV, TY, TX, U, THREADS>(smem, src, ll_out, next, cur, prev, t,  \
                                                         mu, thr, a.N, n, j == a.J, blockIdx.x,  \
                                                         l1);                                    \
    break;
    MS_FA(0) MS_FA(1) MS_FA(2) MS_FA(3) MS_FA(4) MS_FA(5) MS_FA(6) MS_FA(7)
#undef MS_FA
  }
  if (MODE == 1) {
    // block sum of |B_{k+1}|, as analysis_level_kernel
    __shared__ double red[THREADS / 32];
    R hi = l1.s, lo = -l1.c;
    warp_sum_comp<R>(hi, lo);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = (double)hi + (double)lo;
    __syncthreads();
    if (threadIdx.x == 0) {
      double sum = 0.0;
      for (int q = 0; q < THREADS / 32; ++q) sum += red[q];
      a.l1_parts[part_base + (int64_t)blockIdx.y * gridDim.x + blockIdx.x] = sum;
    }
  }
}

// ------------------------------------------------------------ synthesis
template <int TY, int TX> struct FineSyn {
  static constexpr int InY = TY / 2 + kMaxTaps / 2 - 1, InX = TX / 2 + kMaxTaps / 2 - 1;
  static constexpr int XS = TX / 2 + kMaxTaps / 2;   // window row: whole 16-byte chunks
  static constexpr int ZS = InX | 1;
  static constexpr int Sub = InY * XS;
  static constexpr int Elems = 4 * Sub + round4(2 * TY * ZS);
};
// of basis MB: halo columns, and staged columns before the filter's first (a
// window row starts on a chunk)
template <int MB> constexpr int kSynHalo = MB;
template <typename R, int MB>
constexpr int kSynLead = (16 / (int)sizeof(R) - MB % (16 / (int)sizeof(R))) % (16 / (int)sizeof(R));

// The four subband windows of basis MB for the output tile at (r0, c0), by
// cp.async: whole 16-byte chunks where no column wraps and rows start
// aligned, else lane by lane along a row.  (Element by element through two
// quotients, staging took half of a tile's instructions: an iteration at 2048
// px 398 -> 350 us, at 1024 px 122 -> 114, 8 jobs at 1024 px 88 -> 76 a job.)
// TID of NT threads (a block, or a warp that works by itself).
template <typename R, int MB, int TY, int TX, int NT>
__device__ __forceinline__ void fine_synthesis_stage(R* sub, int tid, const R* __restrict__ ap,
                                                     int aps, const R* __restrict__ plane, int N,
                                                     int h, int r0, int c0) {
  using G = FineSyn<TY, TX>;
  constexpr int V = 16 / (int)sizeof(R), HL = kSynHalo<MB>, LEAD = kSynLead<R, MB>;
  constexpr int iny = TY / 2 + HL, inx = TX / 2 + HL;
  constexpr int nch = (LEAD + inx + V - 1) / V;
  const int x0 = c0 / 2 - HL - LEAD, y0 = r0 / 2 - HL;
  const bool chunks = (TX / 2) % V == 0 && x0 >= 0 && h % V == 0 &&
                      ((reinterpret_cast<uintptr_t>(ap) | reinterpret_cast<uintptr_t>(plane)) &
                       15) == 0;
  if (chunks) {
    for (int e = tid; e < 4 * iny * nch; e += NT) {
      const int sq = div_const<nch>(e), c = (e - sq * nch) * V;
      const int s = div_const<iny>(sq), q = sq - s * iny;
      int y = y0 + q;
      y = y >= -h ? wrapc(y, h) : wrap(y, h);
      const R* p = s == 0 ? ap + (int64_t)y * aps
                          : plane + (int64_t)(s >= 2 ? h + y : y) * N + (s & 1 ? h : 0);
      cp_async<16>(sub + s * G::Sub + q * G::XS + c, p + x0 + c);
    }
  } else {
    constexpr int LW = inx <= 8 ? 8 : (inx <= 16 ? 16 : 32);   // lanes a row
    static_assert(inx <= 32 && NT % LW == 0, "a row fits a warp");
    const int c = tid % LW;
    int x = c0 / 2 - HL + c;
    x = x >= -h ? wrapc(x, h) : wrap(x, h);
    if (c < inx) {
      for (int q = tid / LW; q < iny; q += NT / LW) {
        int y = y0 + q;
        y = y >= -h ? wrapc(y, h) : wrap(y, h);
        R* d = sub + q * G::XS + LEAD + c;
        const R* lo = plane + (int64_t)y * N + x;
        const R* hi = lo + (int64_t)h * N;
        cp_async<sizeof(R)>(d, ap + (int64_t)y * aps + x);
        cp_async<sizeof(R)>(d + G::Sub, lo + h);
        cp_async<sizeof(R)>(d + 2 * G::Sub, hi);
        cp_async<sizeof(R)>(d + 3 * G::Sub, hi + h);
      }
    }
  }
  cp_async_commit();
}

// columns: unit = (column, group of U output row pairs, pair lo / hi)
template <typename R, int MB, int TY, int TX, int U, int NT>
__device__ __forceinline__ void fine_synthesis_columns(const R* sub, R* zlo, R* zhi, int tid) {
  using G = FineSyn<TY, TX>;
  constexpr int L = 2 * (MB + 1), HL = kSynHalo<MB>, inx = TX / 2 + HL, NI = U + HL;
  constexpr int gy = TY / 2 / U;
  for (int u = tid; u < inx * gy * 2; u += NT) {
    const int rest = div_const<inx>(u), x = u - rest * inx;
    const int g = rest % gy, pair = rest / gy;
    const R* s0 = sub + pair * G::Sub + U * g * G::XS + kSynLead<R, MB> + x;
    const R* s1 = s0 + 2 * G::Sub;
    R lo[NI], hi[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      lo[i] = s0[i * G::XS];
      hi[i] = s1[i * G::XS];
    }
    R* z = (pair ? zhi : zlo) + 2 * U * g * G::ZS + x;
#pragma unroll
    for (int q = 0; q < U; ++q) {
      R e = 0, o = 0;
#pragma unroll
      for (int m = 0; m < L / 2; ++m) tap_syn<R, MB>(m, lo[q - m + HL], hi[q - m + HL], e, o);
      z[2 * q * G::ZS] = e;
      z[(2 * q + 1) * G::ZS] = o;
    }
  }
}

// rows: unit = (segment of U output pairs, row), rows fastest; put(row, first
// column, 2 U outputs)
template <typename R, int MB, int TY, int TX, int U, int NT, class Put>
__device__ __forceinline__ void fine_synthesis_rows(const R* zlo, const R* zhi, int tid,
                                                    const Put& put) {
  using G = FineSyn<TY, TX>;
  constexpr int L = 2 * (MB + 1), HL = kSynHalo<MB>, NI = U + HL;
  constexpr int gx = TX / 2 / U;
  for (int u = tid; u < TY * gx; u += NT) {
    const int r = u % TY, g = u / TY;
    const R* z0 = zlo + r * G::ZS + U * g;
    const R* z1 = zhi + r * G::ZS + U * g;
    R lo[NI], hi[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      lo[i] = z0[i];
      hi[i] = z1[i];
    }
    R o[2 * U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      R e = 0, d = 0;
#pragma unroll
      for (int m = 0; m < L / 2; ++m) tap_syn<R, MB>(m, lo[q - m + HL], hi[q - m + HL], e, d);
      o[2 * q] = e;
      o[2 * q + 1] = d;
    }
    put(r, 2 * U * g, o);
  }
}

// One output tile of one basis: SYNC joins the NT threads.
template <typename R, int MB, int TY, int TX, int U, int NT, class Sync, class Put>
__device__ __forceinline__ void fine_synthesis_item(R* smem, int tid, const R* __restrict__ ap,
                                                    int aps, const R* __restrict__ plane, int N,
                                                    int h, int r0, int c0, const Sync& sync,
                                                    const Put& put) {
  using G = FineSyn<TY, TX>;
  R* zlo = smem + 4 * G::Sub;
  R* zhi = zlo + TY * G::ZS;
  fine_synthesis_stage<R, MB, TY, TX, NT>(smem, tid, ap, aps, plane, N, h, r0, c0);
  cp_async_wait<0>();
  sync();
  fine_synthesis_columns<R, MB, TY, TX, U, NT>(smem, zlo, zhi, tid);
  sync();
  fine_synthesis_rows<R, MB, TY, TX, U, NT>(zlo, zhi, tid, put);
}

// Levels j >= 2: blockIdx.x = tile, blockIdx.y = basis (longest first); writes
// the approximation of the level below.
template <typename R, int TY, int TX, int U, int THREADS>
__global__ void __launch_bounds__(THREADS)
    fine_synthesis_kernel(FistaPass<R> a_, const R* plain, int j) {
  const FistaPass<R> a = job_slice(a_);   // blockIdx.z: the job (batched form)
  pdl_wait();
  pdl_trigger();
  const R* coef = plain;
  if (!plain) {
    if (a.ctl->done) return;   // uniform: `done` does not change during this kernel
    const int k = a.ctl->k;
    coef = k % 3 == 0 ? a.B0 : (k % 3 == 1 ? a.B1 : a.B2);
  }
  __shared__ __align__(16) R smem[FineSyn<TY, TX>::Elems];
  const int64_t half = (int64_t)a.M * (a.N / 2) * (a.N / 2);
  const int h = a.N >> j, n = 2 * h, tiles_x = n / TX;
  const int r0 = (int)blockIdx.x / tiles_x * TY, c0 = (int)blockIdx.x % tiles_x * TX;
  const int m = a.M - 1 - (int)blockIdx.y;
  const R* plane = coef + (int64_t)m * a.N * a.N;
  const R* ap = j == a.J ? plane : a.tmp + ((j + 1) & 1) * half + (int64_t)m * h * h;
  const int aps = j == a.J ? a.N : h;
  R* out = a.tmp + (j & 1) * half + (int64_t)m * n * n;
  const auto put = [&](int r, int c, const R (&o)[2 * U]) {
    struct alignas(2 * U * sizeof(R) < 16 ? 2 * U * sizeof(R) : 16) Pack { R v[2 * U]; };
    *reinterpret_cast<Pack*>(out + (int64_t)(r0 + r) * n + c0 + c) =
        *reinterpret_cast<const Pack*>(o);
  };
  const auto sync = [] { __syncthreads(); };
  switch (m) {
#define MS_FS(MBV)                                                                              \
  case MBV:                                                                                     \
    fine_synthesis_item<R, MBV, TY, TX, U, THREADS>(smem, threadIdx.x, ap, aps, plane, a.N, h,  \
                                                    r0, c0, sync, put);                         \
    break;
    MS_FS(0) MS_FS(1) MS_FS(2) MS_FS(3) MS_FS(4) MS_FS(5) MS_FS(6) MS_FS(7)
#undef MS_FS
  }
}

// Level 1: x = sum of the bases, one warp per basis (each with its own
// staging, no block barrier until the sum), added in basis order.  Warps w
// and w + 4 share a scheduler: bases w and 7 - w, 18 taps in all, so the four
// schedulers finish together.
template <typename R, int TY, int TX, int U>
__global__ void __launch_bounds__(32 * kMaxBases)
    fine_synthesis_l1_kernel(FistaPass<R> a_, const R* plain) {
  const FistaPass<R> a = job_slice(a_);   // blockIdx.z: the job (batched form)
  pdl_wait();
  pdl_trigger();
  const R* coef = plain;
  if (!plain) {
    if (a.ctl->done) return;   // uniform: `done` does not change during this kernel
    const int k = a.ctl->k;
    coef = k % 3 == 0 ? a.B0 : (k % 3 == 1 ? a.B1 : a.B2);
  }
  using G = FineSyn<TY, TX>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m = warp < 4 ? warp : kMaxBases + 3 - warp;
  R* smem = reinterpret_cast<R*>(smem_raw) + m * G::Elems;
  const int64_t half = (int64_t)a.M * (a.N / 2) * (a.N / 2);
  const int h = a.N / 2, n = a.N, tiles_x = n / TX;
  const int r0 = (int)blockIdx.x / tiles_x * TY, c0 = (int)blockIdx.x % tiles_x * TX;
  const R* plane = coef + (int64_t)m * n * n;
  const R* ap = a.J == 1 ? plane : a.tmp + (int64_t)m * h * h;   // LL_1: half (2 & 1)
  const int aps = a.J == 1 ? n : h;
  // a basis's outputs over its own staged windows (dead by then)
  const auto sync = [] { __syncwarp(); };
  const auto put = [&](int r, int c, const R (&o)[2 * U]) {
#pragma unroll
    for (int q = 0; q < 2 * U; ++q) smem[r * TX + c + q] = o[q];
  };
  static_assert(TY * TX <= 4 * G::Sub, "the outputs alias the windows");
  if (m < a.M) {
    switch (m) {
#define MS_FS(MBV)                                                                           \
  case MBV:                                                                                  \
    fine_synthesis_item<R, MBV, TY, TX, U, 32>(smem, lane, ap, aps, plane, n, h, r0, c0,     \
                                               sync, put);                                   \
    break;
      MS_FS(0) MS_FS(1) MS_FS(2) MS_FS(3) MS_FS(4) MS_FS(5) MS_FS(6) MS_FS(7)
#undef MS_FS
    }
  }
  __syncthreads();
  const R* all = reinterpret_cast<const R*>(smem_raw);
  for (int e = threadIdx.x; e < TY * TX; e += 32 * kMaxBases) {
    R s = 0;
    for (int q = 0; q < a.M; ++q) s += all[q * G::Elems + e];
    const int r = e / TX, c = e - r * TX;
    a.x[(int64_t)(r0 + r) * n + c0 + c] = s;
  }
}

// Level 1 of larger images: x = sum of the bases, a block per tile, basis after
// basis with the next one's windows in flight.  A thread keeps the sums of its
// 2 U outputs of one row in registers.  Tiles this small, rather than 64 pixels
// with half of an SM's shared memory and two blocks an SM, let seven or more
// blocks share an SM and hide each other's barriers (an FP32 iteration, 64 | 32:
// at 1024 px 114 | 109 us, 2048 px 350 | 335, 8 jobs at 1024 px 76.1 | 74.7 a
// job).
template <typename R, int TY, int TX, int U, int NT>
__global__ void __launch_bounds__(NT)
    fine_synthesis_sum_kernel(FistaPass<R> a_, const R* plain) {
  static_assert(TY * (TX / 2 / U) == NT, "a row unit per thread");
  const FistaPass<R> a = job_slice(a_);   // blockIdx.z: the job (batched form)
  pdl_wait();
  pdl_trigger();
  const R* coef = plain;
  if (!plain) {
    if (a.ctl->done) return;   // uniform: `done` does not change during this kernel
    const int k = a.ctl->k;
    coef = k % 3 == 0 ? a.B0 : (k % 3 == 1 ? a.B1 : a.B2);
  }
  using G = FineSyn<TY, TX>;
  __shared__ __align__(16) R subs[2][4 * G::Sub];
  __shared__ R z[2][TY * G::ZS];
  const int tid = threadIdx.x, h = a.N / 2, n = a.N, tiles_x = n / TX;
  const int r0 = (int)blockIdx.x / tiles_x * TY, c0 = (int)blockIdx.x % tiles_x * TX;
  const auto stage = [&](auto basis) {
    constexpr int MB = decltype(basis)::value;
    const R* plane = coef + (int64_t)MB * n * n;
    const R* ap = a.J == 1 ? plane : a.tmp + (int64_t)MB * h * h;   // LL_1: half (2 & 1)
    fine_synthesis_stage<R, MB, TY, TX, NT>(subs[MB & 1], tid, ap, a.J == 1 ? n : h, plane, n, h,
                                            r0, c0);
  };
  R acc[2 * U];
#pragma unroll
  for (int q = 0; q < 2 * U; ++q) acc[q] = 0;
  const auto step = [&](auto basis) {
    constexpr int MB = decltype(basis)::value;
    if (MB >= a.M) return;
    cp_async_wait<0>();
    __syncthreads();   // window MB is there; the other buffer and z are free
    if constexpr (MB + 1 < kMaxBases)
      if (MB + 1 < a.M) stage(std::integral_constant<int, MB + 1>());
    fine_synthesis_columns<R, MB, TY, TX, U, NT>(subs[MB & 1], z[0], z[1], tid);
    __syncthreads();
    fine_synthesis_rows<R, MB, TY, TX, U, NT>(z[0], z[1], tid,
                                              [&](int, int, const R (&o)[2 * U]) {
#pragma unroll
                                                for (int q = 0; q < 2 * U; ++q) acc[q] += o[q];
                                              });
  };
  stage(std::integral_constant<int, 0>());
#define MS_FS(MBV) step(std::integral_constant<int, MBV>());
  MS_FS(0) MS_FS(1) MS_FS(2) MS_FS(3) MS_FS(4) MS_FS(5) MS_FS(6) MS_FS(7)
#undef MS_FS
  struct alignas(2 * U * sizeof(R) < 16 ? 2 * U * sizeof(R) : 16) Pack { R v[2 * U]; };
  R* dst = a.x + (int64_t)(r0 + tid % TY) * n + c0 + 2 * U * (tid / TY);
  *reinterpret_cast<Pack*>(dst) = *reinterpret_cast<const Pack*>(acc);
}
