// The 2-D transforms of the measurement operator (Sect. 2: F Z D and Z^H D^H
// F^H) for image sides N a power of two, 16..4096, on the Ng = 2N grid.
//
// An image is real and fills a quarter of its padded grid, its grid is
// Hermitian, and visibilities reach only cells within `ext` of the origin
// (the plan's longest baseline).  So:
//   forward   N real rows (deapodized, padded) -> columns 0..ext of the half
//             plane; each column's transform of its N nonzero rows, written
//             to rows -ext..ext and, conjugated, to the column's mirror;
//   adjoint   Re(F^H g) needs the Hermitian part only: column u and the mirror
//             of column -u are added as they are read, transformed, and the N
//             image rows of the result kept; N real rows from the half plane,
//             cropped, deapodized and scaled as they are written.
// Each grid cell is written or read once, 8 to 32 bytes of a row by each block
// (ColBlock; blocks that share a sector run side by side and meet in L2);
// padding, cropping, deapodization and the grid's centring (cell k at index k
// + Ng / 2) cost no pass of their own.  A complex transform of the whole grid
// (2-D cuFFT between a padding and a cropping pass) moves 4 to 9 times the
// bytes.  Measured, both directions (own | cuFFT with the passes): N = 128 FP64
// 23 | 75 us, N = 1024 FP32 42 | 91, 16 grids of it 395 | 1166, N = 4096 697 |
// 1290.
//
// A sequence of 2^LOGN elements is held by 2^(LOGN - LE) threads, 2^LE
// elements each, through Stockham stages of radix up to 2^LE: inputs of the
// first stage come from global memory, outputs of the last one go there, and
// the stages between exchange through one padded shared-memory buffer
// (written and read on opposite sides of a barrier, so that four 4096-point
// columns fit a block).  LE is 4 for long FP32 sequences (fewest exchanges);
// FP64, bound by the FP64 instructions of its busiest warp at short lengths,
// spreads them over more threads (see fft_lrad of the spectral kernels).
//
// The kernels are launched with programmatic dependent launch and wait first
// of all: chains of short launches (the linear operator's six an iteration, a
// small image's four) then overlap each launch with its predecessor's end.
// 448 px linear minor cycle 10.65 -> 9.23 ms, residual image at 128 px, FP64, 143
// -> 137 us.
#include <algorithm>

#include "common.cuh"
#include "fft_radix.cuh"

namespace ms {
namespace {

// one sequence: v holds the inputs of the stage after sub-transforms of size
// 2^DONE; store(index, value) receives the outputs of the last stage
template <typename R, int LOGN, int LE, int DONE, bool INV, class Store>
__device__ __forceinline__ void run_stages(C2<R> (&v)[1 << LE], C2<R>* buf,
                                           const C2<R>* __restrict__ tw, int tw_step, int t,
                                           const Store& store) {
  constexpr int N = 1 << LOGN, TPS = N >> LE, EPT = 1 << LE;
  constexpr int LR = LOGN - DONE >= LE ? LE : LOGN - DONE;
  constexpr int Rd = 1 << LR, NS = 1 << DONE;
#pragma unroll
  for (int q = 0; q < EPT / Rd; ++q) {
    const int j = t + q * TPS, js = j & (NS - 1);
    C2<R> w[Rd];
#pragma unroll
    for (int r = 0; r < Rd; ++r) w[r] = v[q * Rd + r];
    if (NS > 1) {
      const int unit = js * (N / (NS * Rd)) * tw_step;
      // W^r: the powers of two from the table, the others products of two
      // smaller ones (a gather of 15 entries took longer than the butterfly:
      // N = 4096 row transforms 166 -> 117 and 124 -> 80 us)
      C2<R> pw[Rd];
#pragma unroll
      for (int r = 1; r < Rd; ++r) {
        const int top = r >= 8 ? 8 : (r >= 4 ? 4 : (r >= 2 ? 2 : 1));
        if (r == top) {
          pw[r] = tw[r * unit];
          if (INV) pw[r].y = -pw[r].y;
        } else {
          const C2<R> x = pw[top], y = pw[r - top];
          pw[r].x = x.x * y.x - x.y * y.y;
          pw[r].y = x.x * y.y + x.y * y.x;
        }
        const C2<R> z = pw[r];
        const C2<R> x = w[r];
        w[r].x = x.x * z.x - x.y * z.y;
        w[r].y = x.x * z.y + x.y * z.x;
      }
    }
    dft_reg<R, Rd, INV>(w);
    const int d0 = (j - js) * Rd + js;
#pragma unroll
    for (int r = 0; r < Rd; ++r) {
      if constexpr (DONE + LR == LOGN)
        store(d0 + r * NS, w[r]);
      else
        buf[padi(d0 + r * NS)] = w[r];
    }
  }
  if constexpr (DONE + LR < LOGN) {
    __syncthreads();
    constexpr int LR2 = LOGN - DONE - LR >= LE ? LE : LOGN - DONE - LR;
    constexpr int Rd2 = 1 << LR2;
#pragma unroll
    for (int q = 0; q < EPT / Rd2; ++q)
#pragma unroll
      for (int r = 0; r < Rd2; ++r) v[q * Rd2 + r] = buf[padi(t + q * TPS + r * (N / Rd2))];
    __syncthreads();
    run_stages<R, LOGN, LE, DONE + LR, INV>(v, buf, tw, tw_step, t, store);
  }
}

// transform of one sequence, load(index) -> store(index, value); tw[m
// tw_step] = exp(-2 pi i m / 2^LOGN)
template <typename R, int LOGN, int LE, bool INV, class Load, class Store>
__device__ __forceinline__ void transform(C2<R>* buf, const C2<R>* __restrict__ tw, int tw_step,
                                          int t, const Load& load, const Store& store) {
  constexpr int N = 1 << LOGN, TPS = N >> LE, EPT = 1 << LE;
  constexpr int Rd = LOGN >= LE ? EPT : N;
  static_assert(LOGN >= LE, "a thread's elements");
  C2<R> v[EPT];
#pragma unroll
  for (int r = 0; r < Rd; ++r) v[r] = load(t + r * TPS);
  run_stages<R, LOGN, LE, 0, INV>(v, buf, tw, tw_step, t, store);
}

// log2 of the elements per thread of a sequence of length 2^logn.  Measured,
// the operator's forward + adjoint transforms, us (rows N, columns 2N long):
// FP32 N = 1024 with 16 a thread from length 2048 on 25.4 + 23.8, with 8 28.8 +
// 27.6; N = 4096 388 + 302 | 463 + 378; N = 512 with 8 15.7 + 14.6, with 16 16.1
// + 16.6, with 4 16.8 + 14.8 (N = 64 to 256 would take 0.5 to 1.5 less with 4).
// FP64 with the elements below | twice | half: N = 128 16.3 + 14.6 | 18.4 + 18.0
// | -, N = 512 80 + 96 | 77 + 79 | 84 + 99, N = 1024 258 + 264 | 266 + 273 | 248
// + 250, N = 2048 984 + 1017 | 975 + 1018 | 999 + 1037 (two columns a block).
constexpr int elems_log(size_t rsz, int logn) {
  return rsz == 4 ? (logn >= 11 ? 4 : (logn >= 6 ? 3 : 2))
                  : (logn <= 9 ? 1 : (logn <= 11 ? 2 : 3));
}
// Sequences of length 2^logn of a block and its shared memory.  Rows: some 256
// threads, at most N / 128 rows.  Columns, as far as 1024 threads and the
// shared memory go: FP32 a 32-byte sector of each row from length 2048 on (N =
// 2048, 4 | 2 columns: 74 + 64 | 83 + 71 us), two at 1024 (N = 512, 2 | 1: 15.7
// + 14.6 | 17.9 + 14.1), else one, so that short columns make a block for each
// SM; FP64 one (N = 512, 1 | 2: 70 + 70 | 80 + 96, N = 1024 228 + 236 | 258 +
// 264; linear operator, 20 iterations and the step size, at 512 px 43.6 | 46.3
// ms, 1024 px 137 | 147), two at 4096 (2 | 1: 984 + 1017 | 963 + 977 us, but the
// linear operator at 2048 px 568 | 572 ms).
template <typename R, int LOGN> struct Seq {
  static constexpr int LE = elems_log(sizeof(R), LOGN);
  static constexpr int TPS = 1 << (LOGN - LE);
  static constexpr int P = padi(1 << LOGN) + 4;   // so that 4 columns' elements share no banks
};
template <typename R, int LOGN> struct ColBlock {
  using S = Seq<R, LOGN>;
  static constexpr int kWant = sizeof(R) == 4 ? (LOGN >= 11 ? 4 : (LOGN == 10 ? 2 : 1))
                                              : (LOGN >= 12 ? 2 : 1);
  static constexpr int kMax = 1024 / S::TPS;
  static constexpr int CB0 = kWant < kMax ? kWant : kMax;
  static constexpr int CB = S::TPS * CB0 < 32 ? 32 / S::TPS : CB0;
  static constexpr int THREADS = CB * S::TPS;
  static constexpr size_t SMEM = (size_t)CB * S::P * sizeof(C2<R>);
};
template <typename R, int LOGM> struct RowBlock {
  using S = Seq<R, LOGM>;
  static constexpr int N = 1 << LOGM;
  static constexpr int kThreads = 256 / S::TPS < 1 ? 1 : 256 / S::TPS;
  static constexpr int kRows = N / 128 < 1 ? 1 : N / 128;
  static constexpr int RB0 = kThreads < kRows ? kThreads : kRows;
  static constexpr int RB = S::TPS * RB0 < 32 ? 32 / S::TPS : RB0;
  static constexpr int THREADS = RB * S::TPS;
  static constexpr size_t SMEM = (size_t)RB * S::P * sizeof(C2<R>);
  static_assert(RB <= N, "rows of a block");
};

// the job of this block: blockIdx.y of the device table, or the one given
template <typename R> __device__ __forceinline__ OpFftJob<R> pick_job(const OpFftArgs<R>& a) {
  if (!a.jobs) return a.one;
  const BatchJob<R>& b = a.jobs[blockIdx.y];
  OpFftJob<R> o;
  o.image_in = b.image_in;
  o.image_out = b.image_out;
  o.grid = b.grid;
  o.scale = b.inv_n;
  o.half = a.one.half + (int64_t)blockIdx.y * a.N * a.pitch;
  return o;
}

// The spectrum out[0..last] of a real row of 2M elements from buf, the M-point
// transform of z_n = x_2n + i x_2n+1: X_k = E_k + W^k O_k, E, O the transforms
// of the even and odd elements (thread t of tps).
template <typename R, int M>
__device__ __forceinline__ void unpack_real_row(const C2<R>* buf, const C2<R>* __restrict__ tw,
                                                C2<R>* out, int last, int t, int tps) {
  for (int k = t; k <= last; k += tps) {
    const C2<R> zk = buf[padi(k == M ? 0 : k)], zm = buf[padi(k == 0 ? 0 : M - k)];
    const R ex = (R)0.5 * (zk.x + zm.x), ey = (R)0.5 * (zk.y - zm.y);
    const R ox = (R)0.5 * (zk.y + zm.y), oy = (R)-0.5 * (zk.x - zm.x);
    const C2<R> w = tw[k];
    C2<R> X;
    X.x = ex + (w.x * ox - w.y * oy);
    X.y = ey + (w.x * oy + w.y * ox);
    out[k] = X;
  }
}

// image row p, deapodized and centred -> its half-plane spectrum 0..ext
template <typename R, int LOGM>
__global__ void __launch_bounds__(RowBlock<R, LOGM>::THREADS)
    op_row_forward_kernel(OpFftArgs<R> a) {
  pdl_wait();
  pdl_trigger();
  using B = RowBlock<R, LOGM>;
  using S = typename B::S;
  constexpr int M = 1 << LOGM, N = M, H = N / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const OpFftJob<R> jb = pick_job(a);
  const int rr = threadIdx.x / S::TPS, t = threadIdx.x - rr * S::TPS;
  const int p = blockIdx.x * B::RB + rr;
  C2<R>* buf = reinterpret_cast<C2<R>*>(smem_raw) + rr * S::P;
  const R* row = jb.image_in + (int64_t)p * N;
  const R dp = a.psi[p];
  // z_n = x_2n + i x_2n+1 of the padded row; image column q sits at q - H mod 2N
  auto load = [&](int n) {
    C2<R> z;
    z.x = z.y = (R)0;
    if (n < H / 2 || n >= M - H / 2) {
      const int q = n < H / 2 ? 2 * n + H : 2 * n - (2 * N - H);
      z.x = row[q] / (dp * a.psi[q]);
      z.y = row[q + 1] / (dp * a.psi[q + 1]);
    }
    return z;
  };
  auto keep = [&](int k, C2<R> z) { buf[padi(k)] = z; };
  transform<R, LOGM, S::LE, false>(buf, a.tw, 2, t, load, keep);
  __syncthreads();
  unpack_real_row<R, M>(buf, a.tw, jb.half + (int64_t)p * a.pitch, a.ext, t, S::TPS);
}

// columns u of the half plane -> grid columns u and -u, rows -ext..ext
template <typename R, int LOGG>
__global__ void __launch_bounds__(ColBlock<R, LOGG>::THREADS)
    op_col_forward_kernel(OpFftArgs<R> a) {
  pdl_wait();
  pdl_trigger();
  using B = ColBlock<R, LOGG>;
  using S = typename B::S;
  constexpr int Ng = 1 << LOGG, N = Ng / 2, H = N / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const OpFftJob<R> jb = pick_job(a);
  const int c = threadIdx.x % B::CB, t = threadIdx.x / B::CB;
  const int u = blockIdx.x * B::CB + c;
  const bool live = u <= a.ext;
  C2<R>* buf = reinterpret_cast<C2<R>*>(smem_raw) + c * S::P;
  const C2<R>* col = jb.half + u;
  auto load = [&](int n) {
    C2<R> z;
    z.x = z.y = (R)0;
    if (live && (n < H || n >= Ng - H)) z = col[(int64_t)(n < H ? n + H : n - (Ng - H)) * a.pitch];
    return z;
  };
  C2<R>* g = jb.grid;
  const int iu = (N + u) & (Ng - 1), mu = N - u;   // grid columns of u and -u
  auto store = [&](int v, C2<R> z) {
    if (!live || (v > a.ext && v < Ng - a.ext)) return;
    g[(int64_t)((N + v) & (Ng - 1)) * Ng + iu] = z;
    if (mu != iu) {
      z.y = -z.y;
      g[(int64_t)((N - v) & (Ng - 1)) * Ng + mu] = z;
    }
  };
  transform<R, LOGG, S::LE, false>(buf, a.tw, 1, t, load, store);
}

// grid columns u and -u (their Hermitian part, doubled), rows -ext..ext -> the
// N image rows of the column's inverse transform
template <typename R, int LOGG>
__global__ void __launch_bounds__(ColBlock<R, LOGG>::THREADS)
    op_col_adjoint_kernel(OpFftArgs<R> a) {
  pdl_wait();
  pdl_trigger();
  using B = ColBlock<R, LOGG>;
  using S = typename B::S;
  constexpr int Ng = 1 << LOGG, N = Ng / 2, H = N / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const OpFftJob<R> jb = pick_job(a);
  const int c = threadIdx.x % B::CB, t = threadIdx.x / B::CB;
  const int u = blockIdx.x * B::CB + c;
  const bool live = u <= a.ext;
  C2<R>* buf = reinterpret_cast<C2<R>*>(smem_raw) + c * S::P;
  const C2<R>* g = jb.grid;
  const int iu = (N + u) & (Ng - 1), mu = N - u;   // grid columns of u and -u
  auto load = [&](int v) {
    C2<R> z;
    z.x = z.y = (R)0;
    if (live && (v <= a.ext || v >= Ng - a.ext)) {
      const C2<R> x = g[(int64_t)((N + v) & (Ng - 1)) * Ng + iu];
      const C2<R> y = g[(int64_t)((N - v) & (Ng - 1)) * Ng + mu];
      z.x = x.x + y.x;
      z.y = x.y - y.y;
    }
    return z;
  };
  C2<R>* col = jb.half + u;
  auto store = [&](int n, C2<R> z) {
    if (live && (n < H || n >= Ng - H)) col[(int64_t)(n < H ? n + H : n - (Ng - H)) * a.pitch] = z;
  };
  transform<R, LOGG, S::LE, true>(buf, a.tw, 1, t, load, store);
}

// half-plane row p (0..ext) -> image row p: cropped, deapodized, scaled
template <typename R, int LOGM>
__global__ void __launch_bounds__(RowBlock<R, LOGM>::THREADS)
    op_row_adjoint_kernel(OpFftArgs<R> a) {
  pdl_wait();
  pdl_trigger();
  using B = RowBlock<R, LOGM>;
  using S = typename B::S;
  constexpr int M = 1 << LOGM, N = M, H = N / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const OpFftJob<R> jb = pick_job(a);
  const int rr = threadIdx.x / S::TPS, t = threadIdx.x - rr * S::TPS;
  const int p = blockIdx.x * B::RB + rr;
  C2<R>* buf = reinterpret_cast<C2<R>*>(smem_raw) + rr * S::P;
  const C2<R>* in = jb.half + (int64_t)p * a.pitch;
  auto at = [&](int k) {
    C2<R> z;
    z.x = z.y = (R)0;
    if (k <= a.ext) z = in[k];
    if (k == 0 || k == M) z.y = (R)0;   // real up to rounding
    return z;
  };
  // Z'_k = (X_k + conj X_(M-k)) + i W^-k (X_k - conj X_(M-k))
  auto load = [&](int k) {
    const C2<R> x = at(k), y = at(M - k), w = a.tw[k];
    const R sx = x.x + y.x, sy = x.y - y.y, dx = x.x - y.x, dy = x.y + y.y;
    const R fx = w.x * dx + w.y * dy, fy = w.x * dy - w.y * dx;
    C2<R> z;
    z.x = sx - fy;
    z.y = sy + fx;
    return z;
  };
  R* row = jb.image_out + (int64_t)p * N;
  const R dp = a.psi[p], sc = (R)(0.5 * jb.scale);   // (the columns were doubled)
  auto store = [&](int n, C2<R> z) {
    if (n >= H / 2 && n < M - H / 2) return;
    const int q = n < H / 2 ? 2 * n + H : 2 * n - (2 * N - H);
    row[q] = z.x * sc / (dp * a.psi[q]);
    row[q + 1] = z.y * sc / (dp * a.psi[q + 1]);
  };
  transform<R, LOGM, S::LE, true>(buf, a.tw, 2, t, load, store);
}

template <typename R, int LOGG>
cudaError_t go(const OpFftArgs<R>& a, bool forward, int njobs, cudaStream_t s) {
  using C = ColBlock<R, LOGG>;
  using W = RowBlock<R, LOGG - 1>;
  auto run = [&](auto kern, int blocks, int threads, size_t smem) {
    if (smem > 48 * 1024) {
      const cudaError_t e =
          cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    return launch_pdl(kern, dim3(blocks, njobs), dim3(threads), smem, s, a);
  };
  const int rows = W::N / W::RB, cols = a.ext / C::CB + 1;
  cudaError_t e;
  if (forward) {
    e = run(op_row_forward_kernel<R, LOGG - 1>, rows, W::THREADS, W::SMEM);
    if (e == cudaSuccess) e = run(op_col_forward_kernel<R, LOGG>, cols, C::THREADS, C::SMEM);
  } else {
    e = run(op_col_adjoint_kernel<R, LOGG>, cols, C::THREADS, C::SMEM);
    if (e == cudaSuccess) e = run(op_row_adjoint_kernel<R, LOGG - 1>, rows, W::THREADS, W::SMEM);
  }
  return e;
}

// ------------------------------------------------ linear PSF operator
// out = scale (P F^-1(H^ . F(P^T x)) + add) on images of side N (even) by
// transforms of length L = 2^LOGL >= 2N: N real rows -> half plane (M = L / 2,
// M + 1 columns) -> each column's transform, product with H^ (column-major,
// 1 / L^2 included) and inverse in one kernel, N rows in and N out -> N real
// rows, cropped, scaled and added to as they are written.  Three launches and
// 4 N (N + M) values; padding, product and cropping as passes between cuFFT
// transforms of the whole L x L field take ten launches and move some 20 N L.
template <typename R, int LOGM>
__global__ void __launch_bounds__(RowBlock<R, LOGM>::THREADS)
    lin_row_forward_kernel(LinFftArgs<R> a) {
  pdl_wait();
  pdl_trigger();
  using B = RowBlock<R, LOGM>;
  using S = typename B::S;
  constexpr int M = 1 << LOGM;
  if (a.ctl && a.ctl->done) return;   // uniform: `done` does not change during this kernel
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int rr = threadIdx.x / S::TPS, t = threadIdx.x - rr * S::TPS;
  const int p = blockIdx.x * B::RB + rr;
  const bool live = p < a.N;
  C2<R>* buf = reinterpret_cast<C2<R>*>(smem_raw) + rr * S::P;
  // (N even: pairs of columns are aligned)
  const C2<R>* row = reinterpret_cast<const C2<R>*>(a.in + (int64_t)p * a.N);
  auto load = [&](int n) {   // z_n = x_2n + i x_2n+1 of the padded row
    C2<R> z;
    z.x = z.y = (R)0;
    if (live && 2 * n < a.N) z = row[n];
    return z;
  };
  auto keep = [&](int k, C2<R> z) { buf[padi(k)] = z; };
  transform<R, LOGM, S::LE, false>(buf, a.tw, 2, t, load, keep);
  __syncthreads();
  if (!live) return;
  unpack_real_row<R, M>(buf, a.tw, a.half + (int64_t)p * a.pitch, M, t, S::TPS);
}

template <typename R, int LOGL>
__global__ void __launch_bounds__(ColBlock<R, LOGL>::THREADS)
    lin_col_kernel(LinFftArgs<R> a) {
  pdl_wait();
  pdl_trigger();
  using B = ColBlock<R, LOGL>;
  using S = typename B::S;
  constexpr int L = 1 << LOGL, M = L / 2;
  if (a.ctl && a.ctl->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int c = threadIdx.x % B::CB, t = threadIdx.x / B::CB;
  const int u = blockIdx.x * B::CB + c;
  const bool live = u <= M;
  C2<R>* buf = reinterpret_cast<C2<R>*>(smem_raw) + c * S::P;
  C2<R>* col = a.half + u;
  const R* h = a.H + (int64_t)(live ? u : 0) * L;
  auto load = [&](int n) {
    C2<R> z;
    z.x = z.y = (R)0;
    if (live && n < a.N) z = col[(int64_t)n * a.pitch];
    return z;
  };
  auto mul = [&](int v, C2<R> z) {
    const R hv = h[v];
    z.x *= hv;
    z.y *= hv;
    buf[padi(v)] = z;
  };
  transform<R, LOGL, S::LE, false>(buf, a.tw, 1, t, load, mul);
  __syncthreads();
  C2<R> v[1 << S::LE];
#pragma unroll
  for (int r = 0; r < (1 << S::LE); ++r) v[r] = buf[padi(t + r * S::TPS)];
  __syncthreads();   // the first stage writes the buffer
  auto store = [&](int n, C2<R> z) {
    if (live && n < a.N) col[(int64_t)n * a.pitch] = z;
  };
  run_stages<R, LOGL, S::LE, 0, true>(v, buf, a.tw, 1, t, store);
}

template <typename R, int LOGM>
__global__ void __launch_bounds__(RowBlock<R, LOGM>::THREADS)
    lin_row_inverse_kernel(LinFftArgs<R> a) {
  pdl_wait();
  pdl_trigger();
  using B = RowBlock<R, LOGM>;
  using S = typename B::S;
  constexpr int M = 1 << LOGM;
  if (a.ctl && a.ctl->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int rr = threadIdx.x / S::TPS, t = threadIdx.x - rr * S::TPS;
  const int p = blockIdx.x * B::RB + rr;
  const bool live = p < a.N;
  C2<R>* buf = reinterpret_cast<C2<R>*>(smem_raw) + rr * S::P;
  const C2<R>* in = a.half + (int64_t)p * a.pitch;
  auto at = [&](int k) {
    C2<R> z;
    z.x = z.y = (R)0;
    if (live) z = in[k];
    if (k == 0 || k == M) z.y = (R)0;   // real up to rounding
    return z;
  };
  // Z'_k = (X_k + conj X_(M-k)) + i W^-k (X_k - conj X_(M-k))
  auto load = [&](int k) {
    const C2<R> x = at(k), y = at(M - k), w = a.tw[k];
    const R sx = x.x + y.x, sy = x.y - y.y, dx = x.x - y.x, dy = x.y + y.y;
    const R fx = w.x * dx + w.y * dy, fy = w.x * dy - w.y * dx;
    C2<R> z;
    z.x = sx - fy;
    z.y = sy + fx;
    return z;
  };
  const int64_t o = (int64_t)p * a.N;
  auto store = [&](int n, C2<R> z) {
    if (!live || 2 * n >= a.N) return;
    const int64_t q = o + 2 * n;
    if (a.add) {
      const C2<R> d = *reinterpret_cast<const C2<R>*>(a.add + q);
      z.x += d.x;
      z.y += d.y;
    }
    z.x *= a.scale;
    z.y *= a.scale;
    *reinterpret_cast<C2<R>*>(a.out + q) = z;
  };
  transform<R, LOGM, S::LE, true>(buf, a.tw, 2, t, load, store);
}

template <typename R, int LOGL> cudaError_t go_linear(const LinFftArgs<R>& a, cudaStream_t s) {
  using C = ColBlock<R, LOGL>;
  using W = RowBlock<R, LOGL - 1>;
  auto run = [&](auto kern, int blocks, int threads, size_t smem) {
    if (smem > 48 * 1024) {
      const cudaError_t e =
          cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    return launch_pdl(kern, dim3(blocks), dim3(threads), smem, s, a);
  };
  const int rows = (a.N + W::RB - 1) / W::RB, cols = W::N / C::CB + 1;
  cudaError_t e = run(lin_row_forward_kernel<R, LOGL - 1>, rows, W::THREADS, W::SMEM);
  if (e == cudaSuccess) e = run(lin_col_kernel<R, LOGL>, cols, C::THREADS, C::SMEM);
  if (e == cudaSuccess) e = run(lin_row_inverse_kernel<R, LOGL - 1>, rows, W::THREADS, W::SMEM);
  return e;
}

// H^ as lin_col_kernel reads it from H2, the real spectrum on the 2N x 2N
// field (L = 2N)
template <typename R>
__global__ void lin_spectrum_kernel(const R* __restrict__ H2, R* __restrict__ H, int L) {
  const int nc = L / 2 + 1;
  const double inv = 1.0 / ((double)L * L);
  const int64_t total = (int64_t)L * nc;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t u = k / L, v = k - u * L;
    H[k] = (R)((double)H2[v * nc + u] * inv);
  }
}

// H^ of the L x L field from the PSF image (plan time): rows, then columns, as
// the operator's transforms, whose tables and block shapes serve.  The image
// has side P = 2N and its origin at (0, 0); of the L-field only rows and
// columns at offsets below +-N are not zero, 2N - 1 of each.
template <typename R, int LOGM>
__global__ void __launch_bounds__(RowBlock<R, LOGM>::THREADS)
    lin_psf_row_kernel(const R* __restrict__ psf, C2<R>* __restrict__ half,
                       const C2<R>* __restrict__ tw, int N, int pitch) {
  using B = RowBlock<R, LOGM>;
  using S = typename B::S;
  constexpr int M = 1 << LOGM, L = 2 * M;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int rr = threadIdx.x / S::TPS, t = threadIdx.x - rr * S::TPS;
  const int p = blockIdx.x * B::RB + rr;
  const bool live = p < 2 * N - 1;
  C2<R>* buf = reinterpret_cast<C2<R>*>(smem_raw) + rr * S::P;
  // row p: offset p, or p - (2N - 1) from N on
  const R* row = psf + (int64_t)(p < N ? p : p + 1) * (2 * N);
  auto at = [&](int x) {
    return live && (x < N || x > L - N) ? row[x < N ? x : x - L + 2 * N] : (R)0;
  };
  auto load = [&](int n) {
    C2<R> z;
    z.x = at(2 * n);
    z.y = at(2 * n + 1);
    return z;
  };
  auto keep = [&](int k, C2<R> z) { buf[padi(k)] = z; };
  transform<R, LOGM, S::LE, false>(buf, tw, 2, t, load, keep);
  __syncthreads();
  if (live) unpack_real_row<R, M>(buf, tw, half + (int64_t)p * pitch, M, t, S::TPS);
}

template <typename R, int LOGL>
__global__ void __launch_bounds__(ColBlock<R, LOGL>::THREADS)
    lin_psf_col_kernel(const C2<R>* __restrict__ half, R* __restrict__ H,
                       const C2<R>* __restrict__ tw, int N, int pitch) {
  using B = ColBlock<R, LOGL>;
  using S = typename B::S;
  constexpr int L = 1 << LOGL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int c = threadIdx.x % B::CB, t = threadIdx.x / B::CB;
  const int u = blockIdx.x * B::CB + c;
  const bool live = u <= L / 2;
  C2<R>* buf = reinterpret_cast<C2<R>*>(smem_raw) + c * S::P;
  auto load = [&](int n) {
    C2<R> z;
    z.x = z.y = (R)0;
    if (live && (n < N || n > L - N))
      z = half[(int64_t)(n < N ? n : n - L + 2 * N - 1) * pitch + u];
    return z;
  };
  auto store = [&](int v, C2<R> z) {   // (L^2: a power of two)
    if (live) H[(int64_t)u * L + v] = z.x * ((R)1 / ((R)L * (R)L));
  };
  transform<R, LOGL, S::LE, false>(buf, tw, 1, t, load, store);
}

template <typename R, int LOGL>
cudaError_t go_psf(const R* psf, C2<R>* half, R* H, const C2<R>* tw, int N, int pitch,
                   cudaStream_t s) {
  using C = ColBlock<R, LOGL>;
  using W = RowBlock<R, LOGL - 1>;
  auto rows = lin_psf_row_kernel<R, LOGL - 1>;
  auto cols = lin_psf_col_kernel<R, LOGL>;
  cudaError_t e = cudaSuccess;
  if (W::SMEM > 48 * 1024)
    e = cudaFuncSetAttribute(rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)W::SMEM);
  if (e == cudaSuccess && C::SMEM > 48 * 1024)
    e = cudaFuncSetAttribute(cols, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
  if (e != cudaSuccess) return e;
  rows<<<(2 * N - 1 + W::RB - 1) / W::RB, W::THREADS, W::SMEM, s>>>(psf, half, tw, N, pitch);
  cols<<<W::N / C::CB + 1, C::THREADS, C::SMEM, s>>>(half, H, tw, N, pitch);
  return cudaGetLastError();
}
}  // namespace

bool op_fft_supported(int N) { return N >= 16 && N <= 4096 && (N & (N - 1)) == 0; }

// row pitch of the half plane: whole 32-byte sectors
int op_fft_pitch(int N) { return N + 4; }

template <typename R>
cudaError_t launch_op_fft(const OpFftArgs<R>& a, bool forward, int njobs, cudaStream_t s) {
  int l = 0;
  while ((1 << l) < 2 * a.N) ++l;
  switch (l) {
    case 5: return go<R, 5>(a, forward, njobs, s);
    case 6: return go<R, 6>(a, forward, njobs, s);
    case 7: return go<R, 7>(a, forward, njobs, s);
    case 8: return go<R, 8>(a, forward, njobs, s);
    case 9: return go<R, 9>(a, forward, njobs, s);
    case 10: return go<R, 10>(a, forward, njobs, s);
    case 11: return go<R, 11>(a, forward, njobs, s);
    case 12: return go<R, 12>(a, forward, njobs, s);
    case 13: return go<R, 13>(a, forward, njobs, s);
    default: return cudaErrorInvalidValue;
  }
}
template cudaError_t launch_op_fft<float>(const OpFftArgs<float>&, bool, int, cudaStream_t);
template cudaError_t launch_op_fft<double>(const OpFftArgs<double>&, bool, int, cudaStream_t);

// The transform length of the linear PSF operator's own kernels for image
// side N, or 0: cuFFT on the 2N x 2N field.  The next power of two where the
// extra columns cost less than the launches and passes saved: up to 8/5 of 2N
// in FP32, 4/3 in FP64.  Measured, step size and a minor cycle of 30
// iterations, ms (own | cuFFT): FP32 128 px 5.8 | 10.0, 320 px (L = 8/5 of 2N)
// 7.9 | 12.9, 384 px (4/3) 8.0 | 13.3, 448 px 9.5 | 16.2, 640 px (8/5) 12.1 |
// 21.6, 1024 px 15.5 | 23.8; FP64 128 px 10.5 | 23.1, 192 px (4/3) 17.3 | 37,
// 384 px (4/3) 46 | 65, 512 px 55 | 109, 640 px (8/5) 162 | 138, 1024 px 199 |
// 330.  Larger sides, the step size and 30 iterations of one basis: FP32 1280 px
// (8/5) 30 | 37, 2048 px 37 | 67, 2560 px (8/5, L = 8192) 151 | 137, 2624 px
// 152 | 266, 2816 px (16/11) 155 | 156, 3072 px (4/3) 161 | 203, 4096 px 187 |
// 246; FP64 1408 px (16/11) 547 | 518, 1536 px (4/3) 563 | 661, 2048 px 617 |
// 1200, 3072 px (4/3) 2379 | 2753, 4096 px 2611 | 4219.  So 8192 serves FP32
// below 8/5 only.
int lin_fft_length(int N, size_t rsz) {
  int L = 32;
  while (L < 2 * N) L *= 2;
  if (N % 2 || L > 8192) return 0;
  if (rsz == 8) return 3 * L <= 8 * N ? L : 0;
  return 5 * L < 16 * N + (L < 8192) ? L : 0;
}

template <typename R> cudaError_t launch_lin_fft(const LinFftArgs<R>& a, int L, cudaStream_t s) {
  switch (L) {
    case 32: return go_linear<R, 5>(a, s);
    case 64: return go_linear<R, 6>(a, s);
    case 128: return go_linear<R, 7>(a, s);
    case 256: return go_linear<R, 8>(a, s);
    case 512: return go_linear<R, 9>(a, s);
    case 1024: return go_linear<R, 10>(a, s);
    case 2048: return go_linear<R, 11>(a, s);
    case 4096: return go_linear<R, 12>(a, s);
    case 8192: return go_linear<R, 13>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

template <typename R>
void launch_lin_spectrum(const R* H2, R* H, int L, cudaStream_t s) {
  lin_spectrum_kernel<R><<<1024, 256, 0, s>>>(H2, H, L);
}
template <typename R>
cudaError_t launch_lin_psf(const R* psf, C2<R>* half, R* H, const C2<R>* tw, int N, int L,
                           int pitch, cudaStream_t s) {
  switch (L) {
    case 128: return go_psf<R, 7>(psf, half, H, tw, N, pitch, s);
    case 256: return go_psf<R, 8>(psf, half, H, tw, N, pitch, s);
    case 512: return go_psf<R, 9>(psf, half, H, tw, N, pitch, s);
    case 1024: return go_psf<R, 10>(psf, half, H, tw, N, pitch, s);
    case 2048: return go_psf<R, 11>(psf, half, H, tw, N, pitch, s);
    case 4096: return go_psf<R, 12>(psf, half, H, tw, N, pitch, s);
    case 8192: return go_psf<R, 13>(psf, half, H, tw, N, pitch, s);
    default: return cudaErrorInvalidValue;
  }
}
#define MS_INST(R)                                                                       \
  template cudaError_t launch_lin_fft<R>(const LinFftArgs<R>&, int, cudaStream_t);       \
  template void launch_lin_spectrum<R>(const R*, R*, int, cudaStream_t);                 \
  template cudaError_t launch_lin_psf<R>(const R*, C2<R>*, R*, const C2<R>*, int, int,   \
                                         int, cudaStream_t);
MS_INST(float)
MS_INST(double)
#undef MS_INST

}  // namespace ms
