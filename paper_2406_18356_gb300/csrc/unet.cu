// The learned warm start: a small U-Net mapping [step-one image, long-baseline
// dirty image] to a starting image for step two (Sect. 3.3), trained on pairs
// the method itself produces.  Activations and weights are bfloat16, every
// product accumulates in FP32 on the tensor cores (mma.sync m16n8k16), master
// weights and the Adam state are FP32, the loss reduces in FP64.
//
// Every convolution is a product over a 3 x 3 window,
//   forward        Y[p][co]  = sum_k X~[p][k] W[co][k],   k = tap Ci + ci
//   data gradient  dX[p][ci] = sum_tap sum_co dZ[p - tap][co] W[co][tap][ci]
//   weight grad.   dW[co][k] = sum_p dZ[p][co] X~[p][k]
// with X~ the window's values (zero outside the image).  None of the windows
// is written to memory: a block stages the pixels of its tile and the ring
// around it once in shared memory and reads the operand fragments from there
// at the offset of each k.  Channel counts are small (6 to 288 at the
// configured shape), so the layers are bound by what they move, and what a
// layer's output needs next (bias and ReLU, the 2 x 2 pooling, the
// concatenation, the ReLU's and the pooling's gradients) is done where the
// values are in registers.  Rounding points match the oracle: inputs, weights
// and stored activations (after ReLU, after pooling) are rounded to bfloat16,
// and so is every pre-activation gradient before it enters a product.
//
// Measured (6 levels, width 6): forward pass at 1024 x 1024 356 us, forward
// and backward pass with the gradients at 512 x 512 746 us; before, with the
// windows written out (im2col, 9 times the activations, and a transposed copy
// for the weight gradients) and one general product kernel: 4166 and 5449 us.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "mstep.h"

namespace ms {
namespace {
using bf16 = __nv_bfloat16;
constexpr int kT = 256;

// The network's kernels after the packing of the weights are launched early
// (programmatic dependent launch): a block stages its weights and computes
// its offsets while the layer before finishes, and waits here before it reads
// or writes anything else.  The next kernel is let go only after the wait, so
// when a kernel starts all kernels but its predecessor have completed: the
// packed weights, two or more launches back, may be read before the wait.
// (Forward pass at 1024 px 421 -> 360 us, gradients at 512 px 870 -> 750.)
__device__ __forceinline__ void after_predecessor() {
  pdl_wait();
  pdl_trigger();
}

int blocks(int64_t n, int cap = 0) {
  if (cap <= 0) cap = sm_count() * 16;
  int64_t b = (n + kT - 1) / kT;
  if (b > cap) b = cap;
  return b < 1 ? 1 : (int)b;
}
__host__ __device__ constexpr int pad16(int x) { return (x + 15) / 16 * 16; }

// ---------------------------------------------------------------- operands
__device__ __forceinline__ void mma16816(float (&d)[4], const unsigned (&a)[4], unsigned b0,
                                         unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
      "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// four 8 x 8 matrices of 16-bit values; lane l gives the address of row l mod
// 8 of matrix l / 8 (16-byte aligned)
__device__ __forceinline__ void ldsm4(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm4t(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm2(unsigned& r0, unsigned& r1, unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];"
               : "=r"(r0), "=r"(r1)
               : "r"(addr)
               : "memory");
}
// asynchronous copy of BYTES (4 or 16), zeros instead when !ok
template <int BYTES> __device__ __forceinline__ void cpz(void* dst, const void* src, bool ok) {
  const int n = ok ? BYTES : 0;
  if (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(saddr(dst)), "l"(src),
                 "r"(n)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(saddr(dst)), "l"(src),
                 "r"(n)
                 : "memory");
}

// A layer's input: the bf16 image a [H][W][ca] (cb = 0), or the concatenation
// of the nearest 2x upsampling of a [H/2][W/2][ca] and b [H][W][cb].
struct Act {
  const bf16* a = nullptr;
  const bf16* b = nullptr;
  int ca = 0, cb = 0;
};
__device__ __forceinline__ const bf16* act_at(const Act& x, int W, int y, int xx, int c) {
  if (x.cb == 0) return x.a + ((int64_t)y * W + xx) * x.ca + c;
  return c < x.ca ? x.a + ((int64_t)(y >> 1) * (W >> 1) + (xx >> 1)) * x.ca + c
                  : x.b + ((int64_t)y * W + xx) * x.cb + (c - x.ca);
}
// values that every aligned group of which lies in one pixel of one source:
// 8 (16-byte copies), 2 (4-byte) or 1
int act_vec(const Act& x) {
  const int g = x.ca | x.cb;
  return g % 8 == 0 ? 8 : (g % 2 == 0 ? 2 : 1);
}

// Stages channels [c0, c0 + n) of the (rows x cols) pixels from (y0, x0) on
// into dst [rows cols][stride], nst >= n values of each pixel written (zeros
// for rows and columns outside the image, and from n on).  VEC as act_vec (n,
// nst and c0 multiples of it).  The copies of VEC > 1 are asynchronous (the
// caller commits and waits).  A thread keeps its column and channels and goes
// down the rows, so the quotients and the choice of the source are taken once
// and a copy costs an add and a compare (element by element the index
// arithmetic took more instructions than the products: forward pass at
// 1024 px 481 -> 418 us with the other changes beside it, dw_kernel at 512 px
// 207 -> 136 with them).
template <int VEC>
__device__ __forceinline__ void stage_pixels(bf16* dst, int stride, int rows, int cols, int y0,
                                             int x0, int H, int W, int c0, int n, int nst,
                                             const Act& src) {
  const int nv = nst / VEC, len = cols * nv, nt = blockDim.x;
  // rows side by side where one takes fewer copies than there are threads
  const int par = len < nt ? nt / len : 1;
  const int r0 = len < nt ? (int)threadIdx.x / len : 0;
  if (r0 >= par) return;
  for (int e = threadIdx.x - r0 * len; e < len; e += nt) {
    const int px = e / nv, v = (e - px * nv) * VEC, x = x0 + px, c = c0 + v;
    const bool okx = x >= 0 && x < W && v < n;
    const bool up = src.cb != 0 && c < src.ca;
    const bf16* g;
    int64_t row;
    if (src.cb == 0 || up) {
      g = src.a + (int64_t)(up ? x >> 1 : x) * src.ca + c;
      row = (int64_t)(up ? W >> 1 : W) * src.ca;
    } else {
      g = src.b + (int64_t)x * src.cb + (c - src.ca);
      row = (int64_t)W * src.cb;
    }
    bf16* d = dst + (r0 * cols + px) * stride + v;
    for (int r = r0; r < rows; r += par, d += par * cols * stride) {
      const int y = y0 + r;
      const bool ok = okx && y >= 0 && y < H;
      const bf16* q = ok ? g + (up ? y >> 1 : y) * row : src.a;
      if constexpr (VEC == 8) cpz<16>(d, q, ok);
      else if constexpr (VEC == 2) cpz<4>(d, q, ok);
      else *d = ok ? *q : __float2bfloat16_rn(0.0f);
    }
  }
}

// Pixel tiles: a warp's m16 tile mt is 8 pixels wide and 2 high (fragment row
// r is pixel (r / 8, r mod 8)); a block takes 16 x 16 pixels (16 m-tiles) or,
// for images too small to fill the SMs that way, 8 x 8 (4 m-tiles).
template <bool BIG> struct Tile {
  static constexpr int S = BIG ? 16 : 8;        // pixels a side
  static constexpr int R = S + 2;               // with the ring
  static constexpr int MTILES = S * S / 16;
  __device__ static __forceinline__ int y(int mtile) { return BIG ? 2 * (mtile >> 1) : 2 * mtile; }
  __device__ static __forceinline__ int x(int mtile) { return BIG ? 8 * (mtile & 1) : 0; }
};

// --------------------------------------------------------------- forward
// Row stride of a pixel in shared memory: the operand reads of 8 neighbouring
// pixels (ldmatrix rows) fall in different banks when stride / 8 is odd.
__host__ __device__ constexpr int pix_stride(int c) {
  return c % 8 ? c + (c & 1) : (c / 8 % 2 ? c : c + 8);
}

struct ConvArgs {
  Act x;
  int H, W, ci, co;
  int kp, cop;              // row lengths of the packed weights (9 ci and co, padded to 16)
  const bf16* w;            // [co][kp]
  const bf16* wt;           // [9 ci][cop]
  const float* bias;
  bf16* out;                // [P][co] after the ReLU, or nullptr (the head)
  bf16* pooled;             // [P/4][co] 2 x 2 averages of out, or nullptr
  const float* head_in;     // head: the network's input [P][2]
  float* head_out;          // head: product + bias + the input's first channel
  int ck;                   // = ci (conv_kernel's loop over channels)
  int vec;                  // act_vec of x
};
// k of c channels, padded to whole steps, and shared memory
__host__ __device__ constexpr int conv_kl(int c) { return pad16(9 * c); }
template <bool BIG> size_t conv_smem(int c, int nt) {
  return ((size_t)Tile<BIG>::R * Tile<BIG>::R * pix_stride(c) + 16 + 8 +
          (size_t)nt * 8 * (conv_kl(c) + 8)) * sizeof(bf16) + (size_t)conv_kl(c) * sizeof(int);
}

// What a warp's sums become: bias and ReLU into out (and its 2 x 2 averages
// into pooled), or the head's output.  Its first m-tile, the tile's first pixel
// and its first channel; all lanes take part.
template <class TL, int MT, int NT>
__device__ __forceinline__ void conv_store(const ConvArgs& p, const float (&acc)[MT][NT][4],
                                           int mt0, int y0, int x0, int n0, int lane) {
  const int gid = lane >> 2, tig = lane & 3;
  // acc[.][.][q]: pixel row q / 2 of the m-tile's two, column gid, channel
  // 2 tig + (q & 1) of the n8 tile
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    const int mt = mt0 + i;
    const int y = y0 + TL::y(mt), x = x0 + TL::x(mt) + gid;
    const bool okx = x < p.W;
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      const int n = n0 + j * 8 + 2 * tig;
      if (p.out) {
        float v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int c = n + (q & 1);
          v[q] = fmaxf(acc[i][j][q] + (c < p.co ? p.bias[c] : 0.0f), 0.0f);
          v[q] = __bfloat162float(__float2bfloat16_rn(v[q]));   // exact in the stores below
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          if (!okx || y + r >= p.H || n >= p.co) continue;
          bf16* o = p.out + ((int64_t)(y + r) * p.W + x) * p.co + n;
          if (p.co % 2 == 0) {
            *reinterpret_cast<__nv_bfloat162*>(o) =
                __floats2bfloat162_rn(v[2 * r], v[2 * r + 1]);
          } else {
            o[0] = __float2bfloat16_rn(v[2 * r]);
            if (n + 1 < p.co) o[1] = __float2bfloat16_rn(v[2 * r + 1]);
          }
        }
        if (p.pooled) {
          // the pixel to the right is 4 lanes on; sides are even, so a 2 x 2
          // block lies in the image as a whole
          float s[2];
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const float right0 = __shfl_xor_sync(0xffffffffu, v[c], 4);
            const float right1 = __shfl_xor_sync(0xffffffffu, v[2 + c], 4);
            s[c] = 0.25f * (((v[c] + right0) + v[2 + c]) + right1);
          }
          if (okx && y < p.H && (gid & 1) == 0) {
            bf16* o = p.pooled + ((int64_t)(y >> 1) * (p.W >> 1) + (x >> 1)) * p.co + n;
            if (n < p.co) o[0] = __float2bfloat16_rn(s[0]);
            if (n + 1 < p.co) o[1] = __float2bfloat16_rn(s[1]);
          }
        }
      } else if (n == 0 && okx) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          if (y + r >= p.H) continue;
          const int64_t k = (int64_t)(y + r) * p.W + x;
          p.head_out[k] = (acc[i][j][2 * r] + p.bias[0]) + p.head_in[2 * k];
        }
      }
    }
  }
}

// One convolution on one pixel tile and NT n8 tiles of output channels.  VEC:
// act_vec of the input (8: operand rows by ldmatrix; else per-lane loads).
// The accumulation runs over k = tap ci + c in steps of 16, one chain per
// output.  The loop over channels makes one trip (p.ck = ci), which the compiler
// does not know: without the loop it schedules the k steps in fewer registers
// (NT = 2: 36 | 32) and small images take longer (6 levels of 6, forward pass:
// 128 px 82.2 | 85.2 us, 512 px 161.6 | 163.5).
template <bool BIG, int NT, int VEC>
__global__ void __launch_bounds__(128) conv_kernel(const ConvArgs p) {
  using TL = Tile<BIG>;
  constexpr int MT = TL::MTILES / 4;   // m-tiles per warp
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
  const int tiles_x = (p.W + TL::S - 1) / TL::S;
  const int ty = blockIdx.x / tiles_x, tx = blockIdx.x - ty * tiles_x;
  const int y0 = ty * TL::S, x0 = tx * TL::S, n0 = blockIdx.y * NT * 8;
  const int CS = pix_stride(p.ck), KS = conv_kl(p.ck) + 8;
  bf16* sx = reinterpret_cast<bf16*>(smem_raw);            // [R R][CS], then 16 zeros
  const int zero_off = (TL::R * TL::R * CS + 7) / 8 * 8;   // (16-byte aligned)
  bf16* sw = sx + zero_off + 16;                           // [NT 8][KS]
  int* koff = reinterpret_cast<int*>(sw + NT * 8 * KS);    // window offset of k (VEC > 1: k VEC)

  float acc[MT][NT][4];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;

  for (int c0 = 0; c0 < p.ci; c0 += p.ck) {
    const int ck = min(p.ck, p.ci - c0), kl = pad16(9 * ck);
    if (tid < 16) sx[zero_off + tid] = __float2bfloat16_rn(0.0f);
    for (int k = tid * VEC; k < kl; k += 128 * VEC) {
      const int tap = k / ck, c = k - tap * ck;
      // (k >= 9 ck: the padding reads zeros, whatever the window holds)
      koff[k / VEC] = tap < 9 ? ((tap / 3) * TL::R + tap % 3) * CS + c : -1;
    }
    const int nv = kl / 8;   // whole packed rows (kl = kp, a multiple of 16)
    const float inv = 1.0f / (float)nv;
    for (int e = tid; e < NT * 8 * nv; e += 128) {
      const int r = (int)(((float)e + 0.5f) * inv), v = (e - r * nv) * 8;
      const bool ok = n0 + r < p.co;
      cpz<16>(sw + r * KS + v, ok ? p.w + (int64_t)(n0 + r) * p.kp + v : p.w, ok);
    }
    after_predecessor();
    stage_pixels<VEC>(sx, CS, TL::R, TL::R, y0 - 1, x0 - 1, p.H, p.W, c0, ck, ck, p.x);
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();

    // this lane's pixel offsets: ldmatrix rows (VEC 8), or fragment row gid
    int base[MT];
#pragma unroll
    for (int i = 0; i < MT; ++i) {
      const int mt = warp * MT + i;
      const int yy = TL::y(mt) + (VEC == 8 ? (lane >> 3) & 1 : 0);
      const int xx = TL::x(mt) + (VEC == 8 ? lane & 7 : gid);
      base[i] = (yy * TL::R + xx) * CS;
    }
    const unsigned sx_a = saddr(sx), sw_a = saddr(sw);
    const unsigned zero_a = sx_a + 2u * zero_off;
    // B rows: matrix lane / 8 = (n8 tile of the pair, k half)
    const unsigned b_a = sw_a + 2u * (((lane >> 4) * 8 + (lane & 7)) * KS + ((lane >> 3) & 1) * 8);
    // one k step; PAD: it may hold k >= 9 ck
    const auto k_step = [&](int k0, auto last) {
      constexpr bool PAD = decltype(last)::value;
      unsigned b[NT][2];
#pragma unroll
      for (int j = 0; j + 1 < NT; j += 2) {
        unsigned r[4];
        ldsm4(r, b_a + 2u * (j * 8 * KS + k0));
        b[j][0] = r[0];
        b[j][1] = r[1];
        b[j + 1][0] = r[2];
        b[j + 1][1] = r[3];
      }
      if (NT & 1)
        ldsm2(b[NT - 1][0], b[NT - 1][1],
              sw_a + 2u * (((NT - 1) * 8 + (lane & 7)) * KS + ((lane >> 3) & 1) * 8 + k0));
      if constexpr (VEC == 8) {
        const int ko = koff[(k0 >> 3) + (lane >> 4)];
#pragma unroll
        for (int i = 0; i < MT; ++i) {
          unsigned a[4];
          ldsm4(a, !PAD || ko >= 0 ? sx_a + 2u * (base[i] + ko) : zero_a);
#pragma unroll
          for (int j = 0; j < NT; ++j) mma16816(acc[i][j], a, b[j][0], b[j][1]);
        }
      } else if constexpr (VEC == 2) {
        const int k_lo = koff[(k0 >> 1) + tig], k_hi = koff[(k0 >> 1) + 4 + tig];
        const int dy = TL::R * CS;
#pragma unroll
        for (int i = 0; i < MT; ++i) {
          unsigned a[4];
          const bf16* q = sx + (!PAD || k_lo >= 0 ? base[i] + k_lo : zero_off);
          const bf16* q1 = sx + (!PAD || k_lo >= 0 ? base[i] + dy + k_lo : zero_off);
          const bf16* h = sx + (!PAD || k_hi >= 0 ? base[i] + k_hi : zero_off);
          const bf16* h1 = sx + (!PAD || k_hi >= 0 ? base[i] + dy + k_hi : zero_off);
          a[0] = *reinterpret_cast<const unsigned*>(q);
          a[1] = *reinterpret_cast<const unsigned*>(q1);
          a[2] = *reinterpret_cast<const unsigned*>(h);
          a[3] = *reinterpret_cast<const unsigned*>(h1);
#pragma unroll
          for (int j = 0; j < NT; ++j) mma16816(acc[i][j], a, b[j][0], b[j][1]);
        }
      } else {
        int ko[4];   // k0 + 2 tig, + 1, + 8, + 9
#pragma unroll
        for (int q = 0; q < 4; ++q) ko[q] = koff[k0 + 2 * tig + (q & 1) + 8 * (q >> 1)];
#pragma unroll
        for (int i = 0; i < MT; ++i) {
          unsigned a[4];
#pragma unroll
          for (int f = 0; f < 4; ++f) {   // (row half f & 1, k half f >> 1)
            const int row = base[i] + (f & 1) * TL::R * CS;
            const int e0 = ko[2 * (f >> 1)], e1 = ko[2 * (f >> 1) + 1];
            const unsigned short l0 = *reinterpret_cast<const unsigned short*>(
                sx + (!PAD || e0 >= 0 ? row + e0 : zero_off));
            const unsigned short l1 = *reinterpret_cast<const unsigned short*>(
                sx + (!PAD || e1 >= 0 ? row + e1 : zero_off));
            a[f] = (unsigned)l0 | ((unsigned)l1 << 16);
          }
#pragma unroll
          for (int j = 0; j < NT; ++j) mma16816(acc[i][j], a, b[j][0], b[j][1]);
        }
      }
    };
    for (int k0 = 0; k0 < kl - 16; k0 += 16) k_step(k0, std::false_type());
    k_step(kl - 16, std::true_type());
  }

  conv_store<TL, MT, NT>(p, acc, warp * MT, y0, x0, n0, lane);
}

// Wider layers: a block takes 64 output channels of a pixel tile and walks over
// the input channels 16 at a time, the next ones' pixels and weights on their
// way (two buffers) while this one's nine taps are multiplied.  Half of the
// warps share each 32 channels; a warp's operand row then serves 4 n8 tiles and
// its weights 2 or 4 m-tiles, where conv_kernel, whose block holds the weights
// of all k at once, has room for one n8 tile beside some 400 channels and
// re-reads the pixels for each.  The weights come from the transposed copy,
// whose rows are aligned for any number of channels.  The sums run chunk by
// chunk, tap by tap, one chain per output.  Measured, forward pass of 2 levels
// of width 256 at 256 px: 1333 us (378 TFLOP/s); conv_kernel, channel chunks
// staged in turn, 32303; the products on written-out windows before it 6790.
constexpr int kWideN = 64, kWideC = 16;
constexpr int kWideXS = kWideC + 8, kWideWS = kWideN + 8;   // row strides (no bank conflicts)
template <bool BIG> struct Wide {
  static constexpr int Threads = BIG ? 256 : 128;
  static constexpr int X = Tile<BIG>::R * Tile<BIG>::R * kWideXS, W = 9 * kWideC * kWideWS;
  static constexpr size_t Smem = 2 * (size_t)(X + W) * sizeof(bf16);
};

template <bool BIG, int VEC>
__global__ void __launch_bounds__(Wide<BIG>::Threads, BIG ? 2 : 3)
    conv_wide_kernel(const ConvArgs p) {
  using TL = Tile<BIG>;
  using G = Wide<BIG>;
  constexpr int NW = G::Threads / 32, MT = TL::MTILES / (NW / 2), NT = kWideN / 16;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  bf16* buf = reinterpret_cast<bf16*>(smem_raw);   // two of (pixels [R R], weights [9][16][64])
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tiles_x = (p.W + TL::S - 1) / TL::S;
  const int ty = blockIdx.x / tiles_x, tx = blockIdx.x - ty * tiles_x;
  const int y0 = ty * TL::S, x0 = tx * TL::S, n0 = blockIdx.y * kWideN;
  const int mt0 = (warp >> 1) * MT, nw = (warp & 1) * NT * 8;   // this warp's share
  const auto stage_w = [&](int c0) {
    bf16* sw = buf + (c0 / kWideC & 1) * (G::X + G::W) + G::X;
    for (int e = tid; e < 9 * kWideC * (kWideN / 8); e += G::Threads) {
      const int r = e / (kWideN / 8), v = e % (kWideN / 8) * 8;
      const int tap = r / kWideC, c = c0 + r % kWideC;
      const bool ok = c < p.ci && n0 + v < p.cop;
      const bf16* q = ok ? p.wt + (int64_t)(tap * p.ci + c) * p.cop + n0 + v : p.wt;
      cpz<16>(sw + r * kWideWS + v, q, ok);
    }
  };
  const auto stage_x = [&](int c0) {
    stage_pixels<VEC>(buf + (c0 / kWideC & 1) * (G::X + G::W), kWideXS, TL::R, TL::R, y0 - 1,
                      x0 - 1, p.H, p.W, c0, min(kWideC, p.ci - c0), kWideC, p.x);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[MT][NT][4];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
  // ldmatrix rows: pixels (row half lane / 8 mod 2, k half lane / 16); weights,
  // transposed (n8 tile of the pair lane / 16, k half lane / 8 mod 2)
  unsigned a_o[MT];
#pragma unroll
  for (int i = 0; i < MT; ++i)
    a_o[i] = 2u * (((TL::y(mt0 + i) + ((lane >> 3) & 1)) * TL::R + TL::x(mt0 + i) + (lane & 7)) *
                       kWideXS + (lane >> 4) * 8);
  const unsigned b_o = 2u * (G::X + (lane & 15) * kWideWS + nw + (lane >> 4) * 8);
  stage_w(0);
  after_predecessor();
  stage_x(0);
  for (int c0 = 0; c0 < p.ci; c0 += kWideC) {
    if (c0 + kWideC < p.ci) {
      stage_w(c0 + kWideC);
      stage_x(c0 + kWideC);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const unsigned base = saddr(buf) + 2u * (c0 / kWideC & 1) * (G::X + G::W);
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) {
      unsigned b[NT][2];
#pragma unroll
      for (int j = 0; j < NT; j += 2) {
        unsigned r[4];
        ldsm4t(r, base + b_o + 2u * (tap * kWideC * kWideWS + j * 8));
        b[j][0] = r[0];
        b[j][1] = r[1];
        b[j + 1][0] = r[2];
        b[j + 1][1] = r[3];
      }
#pragma unroll
      for (int i = 0; i < MT; ++i) {
        unsigned a[4];
        ldsm4(a, base + a_o[i] + 2u * ((tap / 3) * TL::R + tap % 3) * kWideXS);
#pragma unroll
        for (int j = 0; j < NT; ++j) mma16816(acc[i][j], a, b[j][0], b[j][1]);
      }
    }
    __syncthreads();   // the buffer is staged again
  }
  conv_store<TL, MT, NT>(p, acc, mt0, y0, x0, n0 + nw, lane);
}

// ---------------------------------------------------------- data gradient
struct DxArgs {
  const bf16* dz;        // this layer's pre-activation gradient [P][co]
  const bf16* wt;        // [9 ci][cop]
  int H, W, ci, co, cop;
  int ck;                // output channels staged at a time (a multiple of 16, or co)
  // where the input's gradient goes (mode):
  //  0  through the ReLU of the layer before (out_a [P][ci]) into dz_a [P][ci]
  //  1  the input is a concatenation: its first ca channels, summed over each
  //     2 x 2 block, through the ReLU of the level below (out_a, dz_a
  //     [P/4][ca]), the others into skip_g [P][ci - ca] (FP32)
  //  2  the input is a pooled image: a quarter to each pixel of its 2 x 2
  //     block, plus skip_g [4 P][ci], through the ReLU of the level above
  //     (out_a, dz_a [4 P][ci])
  int mode, ca;
  const bf16* out_a;
  bf16* dz_a;
  float* skip_g;
};
template <bool BIG> size_t dx_smem(int ck, int nt) {
  const size_t ks = pad16(ck) + 8;
  return ((size_t)Tile<BIG>::R * Tile<BIG>::R * ks + (size_t)9 * nt * 8 * ks) * sizeof(bf16);
}
__device__ __forceinline__ bf16 relu_back(float g, bf16 out) {
  return __float2bfloat16_rn(__bfloat162float(out) > 0.0f ? g : 0.0f);
}

// Gradient of one convolution's input on one pixel tile and NT n8 tiles of
// input channels: the taps' products over the output channels, each one chain
// from zero, added in tap order.  VEC: alignment of dz's pixels (as act_vec).
template <bool BIG, int NT, int VEC>
__global__ void __launch_bounds__(BIG ? 256 : 128) dx_kernel(const DxArgs p) {
  using TL = Tile<BIG>;
  constexpr int NW = BIG ? 8 : 4, MT = TL::MTILES / NW;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
  const int tiles_x = (p.W + TL::S - 1) / TL::S;
  const int ty = blockIdx.x / tiles_x, tx = blockIdx.x - ty * tiles_x;
  const int y0 = ty * TL::S, x0 = tx * TL::S, n0 = blockIdx.y * NT * 8;
  const int KS = pad16(p.ck) + 8;
  bf16* sz = reinterpret_cast<bf16*>(smem_raw);   // [R R][KS]
  bf16* sw = sz + TL::R * TL::R * KS;             // [9][NT 8][KS]
  float sum[MT][NT][4];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) sum[i][j][q] = 0.0f;
  for (int c0 = 0; c0 < p.co; c0 += p.ck) {
    const int ck = min(p.ck, p.co - c0), kl = pad16(ck);
    if (c0) __syncthreads();
    const int nv = kl / 8;
    const float inv = 1.0f / (float)nv;
    for (int e = tid; e < 9 * NT * 8 * nv; e += NW * 32) {
      const int r = (int)(((float)e + 0.5f) * inv), v = (e - r * nv) * 8;
      const int tap = r / (NT * 8), c = n0 + r - tap * (NT * 8);
      const bool ok = c < p.ci;
      cpz<16>(sw + r * KS + v, ok ? p.wt + (int64_t)(tap * p.ci + c) * p.cop + c0 + v : p.wt, ok);
    }
    if (c0 == 0) after_predecessor();
    stage_pixels<VEC>(sz, KS, TL::R, TL::R, y0 - 1, x0 - 1, p.H, p.W, c0, ck, kl,
                      Act{p.dz, nullptr, p.co, 0});
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const unsigned sz_a = saddr(sz), sw_a = saddr(sw);
    const unsigned b_a = sw_a + 2u * (((lane >> 4) * 8 + (lane & 7)) * KS + ((lane >> 3) & 1) * 8);
    const unsigned b1_a = sw_a + 2u * (((NT - 1) * 8 + (lane & 7)) * KS + ((lane >> 3) & 1) * 8);
    unsigned a_a[MT];
#pragma unroll
    for (int i = 0; i < MT; ++i) {
      const int mt = warp * MT + i;
      const int px = (TL::y(mt) + ((lane >> 3) & 1)) * TL::R + TL::x(mt) + (lane & 7);
      a_a[i] = sz_a + 2u * (px * KS + (lane >> 4) * 8);
    }
#pragma unroll 1
    for (int tap = 0; tap < 9; ++tap) {
      // output pixel p - (ky - 1, kx - 1), in the staged tile (ring of one)
      const unsigned sh = 2u * (((2 - tap / 3) * TL::R + 2 - tap % 3) * KS);
      const unsigned wo = 2u * tap * NT * 8 * KS;
      float acc[MT][NT][4];
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
      for (int k0 = 0; k0 < kl; k0 += 16) {
        unsigned b[NT][2];
#pragma unroll
        for (int j = 0; j + 1 < NT; j += 2) {
          unsigned r[4];
          ldsm4(r, b_a + wo + 2u * (j * 8 * KS + k0));
          b[j][0] = r[0];
          b[j][1] = r[1];
          b[j + 1][0] = r[2];
          b[j + 1][1] = r[3];
        }
        if (NT & 1) ldsm2(b[NT - 1][0], b[NT - 1][1], b1_a + wo + 2u * k0);
#pragma unroll
        for (int i = 0; i < MT; ++i) {
          unsigned a[4];
          ldsm4(a, a_a[i] + sh + 2u * k0);
#pragma unroll
          for (int j = 0; j < NT; ++j) mma16816(acc[i][j], a, b[j][0], b[j][1]);
        }
      }
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int q = 0; q < 4; ++q) sum[i][j][q] += acc[i][j][q];
    }
  }
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    const int mt = warp * MT + i;
    const int y = y0 + TL::y(mt), x = x0 + TL::x(mt) + gid;
    const bool okx = x < p.W;
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int cc = 0; cc < 2; ++cc) {
        const int c = n0 + j * 8 + 2 * tig + cc;
        const float g0 = sum[i][j][cc], g1 = sum[i][j][2 + cc];   // rows y, y + 1
        if (p.mode == 1) {
          const float r0 = __shfl_xor_sync(0xffffffffu, g0, 4);
          const float r1 = __shfl_xor_sync(0xffffffffu, g1, 4);
          if (c >= p.ci || !okx || y >= p.H) continue;   // (H, W even)
          if (c < p.ca) {
            if (gid & 1) continue;
            const int64_t k = ((int64_t)(y >> 1) * (p.W >> 1) + (x >> 1)) * p.ca + c;
            p.dz_a[k] = relu_back(((g0 + r0) + g1) + r1, p.out_a[k]);
          } else {
            const int cs = p.ci - p.ca;
            const int64_t k = ((int64_t)y * p.W + x) * cs + c - p.ca;
            p.skip_g[k] = g0;
            p.skip_g[k + (int64_t)p.W * cs] = g1;
          }
          continue;
        }
        if (c >= p.ci || !okx) continue;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          if (y + r >= p.H) continue;
          const float g = r ? g1 : g0;
          if (p.mode == 0) {
            const int64_t k = ((int64_t)(y + r) * p.W + x) * p.ci + c;
            p.dz_a[k] = relu_back(g, p.out_a[k]);
          } else {
            const int64_t W2 = 2 * (int64_t)p.W;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int64_t k =
                  ((int64_t)(2 * (y + r) + (q >> 1)) * W2 + 2 * x + (q & 1)) * p.ci + c;
              p.dz_a[k] = relu_back(p.skip_g[k] + 0.25f * g, p.out_a[k]);
            }
          }
        }
      }
  }
}

// -------------------------------------------------------- weight gradients
// All layers' weight and bias gradients in one launch.  A block takes one
// unit of work of one layer: 16 output channels, 8 input channels (all nine
// taps: the same staged pixels serve them) and a range of 8 x 16 pixel tiles,
// whose four warps take 32 pixels of each tile.  The pixel sums of a block go to its slice of
// the partial sums; sum_partials_kernel adds a layer's slices in order.
// The sums' exchange shares the staging buffers, so four blocks fit an SM
// (registers; three before, 33 KB of shared memory each).
// A unit of 8 input channels (rather than more) leaves enough units at the
// coarse levels, where a layer has 256 pixels and up to 192 x 1728 weights.
constexpr int kMaxConvs = 24;   // 4 levels - 1 at most 6 levels
struct WLayer {
  Act x;
  const bf16* dz;
  int H, W, ci, co;
  int cob, cib, tiles_x, tiles, per;   // co / ci blocks, pixel tiles, tiles per unit
  int splits;
  int first;                            // its first block of the launch
  int vx, vz;                           // alignments of x and dz (act_vec)
  int64_t part;                         // its slices in the partial sums
  int64_t woff;                         // its weights and bias in the flat gradient
};
struct WArgs {
  WLayer l[kMaxConvs];
  int n;
  float* parts;
  float* grad;
  int64_t nparams;
};
constexpr int kWTileY = 8, kWTileX = 16;
constexpr int kWXP = (kWTileY + 2) * (kWTileX + 2);   // staged input pixels
constexpr int kWZS = 24;                              // row stride of a staged dz pixel (16 used)

template <int VEC>
__device__ __forceinline__ void w_stage_x(bf16* dst, const WLayer& l, int y0, int x0, int c0) {
  stage_pixels<VEC>(dst, 8, kWTileY + 2, kWTileX + 2, y0 - 1, x0 - 1, l.H, l.W, c0,
                    min(8, l.ci - c0), 8, l.x);
}
template <int VEC>
__device__ __forceinline__ void w_stage_z(bf16* dst, const WLayer& l, int y0, int x0, int c0) {
  stage_pixels<VEC>(dst, kWZS, kWTileY, kWTileX, y0, x0, l.H, l.W, c0, min(16, l.co - c0), 16,
                    Act{l.dz, nullptr, l.co, 0});
}

__global__ void __launch_bounds__(128, 4) dw_kernel(const __grid_constant__ WArgs p) {
  struct Stage {
    bf16 x[2][kWXP * 8], z[2][kWTileY * kWTileX * kWZS];
  };
  __shared__ __align__(16) union {
    Stage st;
    float red[3][10][32][4];   // the warps' sums, once the tiles are done
  } sm;
  after_predecessor();
  auto& sx = sm.st.x;
  auto& sz = sm.st.z;
  auto& red = sm.red;
  int li = 0;
  while (li + 1 < p.n && (int)blockIdx.x >= p.l[li + 1].first) ++li;
  const WLayer& l = p.l[li];
  int u = blockIdx.x - l.first;
  const int split = u / (l.cob * l.cib);
  u -= split * l.cob * l.cib;
  const int cb = u / l.cib, co0 = cb * 16, ci0 = (u - cb * l.cib) * 8;
  const int t_lo = split * l.per, t_hi = min(l.tiles, t_lo + l.per);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;

  auto stage = [&](int t) {
    const int ty = t / l.tiles_x, y0 = ty * kWTileY, x0 = (t - ty * l.tiles_x) * kWTileX;
    bf16* dx = sx[t & 1];
    bf16* dz = sz[t & 1];
    if (l.vx == 8) w_stage_x<8>(dx, l, y0, x0, ci0);
    else if (l.vx == 2) w_stage_x<2>(dx, l, y0, x0, ci0);
    else w_stage_x<1>(dx, l, y0, x0, ci0);
    if (l.vz == 8) w_stage_z<8>(dz, l, y0, x0, co0);
    else if (l.vz == 2) w_stage_z<2>(dz, l, y0, x0, co0);
    else w_stage_z<1>(dz, l, y0, x0, co0);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[10][4];   // nine taps, and the bias (a column of ones)
#pragma unroll
  for (int j = 0; j < 10; ++j)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[j][q] = 0.0f;
  const unsigned one = gid == 0 ? 0x3f803f80u : 0u;   // bf16 ones in the first column
  // row addresses of the transposed reads: pixel rows of 8 (matrix lane / 8)
  const int mi = lane >> 3, mr = lane & 7;
  if (t_lo < t_hi) stage(t_lo);
  for (int t = t_lo; t < t_hi; ++t) {
    if (t + 1 < t_hi) {
      stage(t + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const unsigned xa = saddr(sx[t & 1]), za = saddr(sz[t & 1]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {   // 16 pixels: one row of the tile
      const int py = warp * 2 + h;
      // A = dz^T (16 channels x 16 pixels): matrices (pixels 0-7 | 8-15) x
      // (channels 0-7 | 8-15), read transposed: a0 = channels 0-7 / pixels
      // 0-7, a1 = channels 8-15 / pixels 0-7, a2, a3 the other pixels
      unsigned a[4];
      ldsm4t(a, za + 2u * ((py * kWTileX + (mi >> 1) * 8 + mr) * kWZS + (mi & 1) * 8));
      mma16816(acc[9], a, one, one);
#pragma unroll
      for (int tp = 0; tp < 9; tp += 2) {
        // B (16 pixels x 8 channels) of taps tp, tp + 1: matrices (tap, pixel half)
        const int tap = min(tp + (mi >> 1), 8);
        unsigned b[4];
        ldsm4t(b, xa + 2u * (((py + tap / 3) * (kWTileX + 2) + (mi & 1) * 8 + mr + tap % 3) * 8));
        mma16816(acc[tp], a, b[0], b[1]);
        if (tp + 1 < 9) mma16816(acc[tp + 1], a, b[2], b[3]);
      }
    }
    __syncthreads();   // the buffer is staged again
  }
  // the warps' sums, in warp order
  if (warp > 0) {
#pragma unroll
    for (int j = 0; j < 10; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) red[warp - 1][j][lane][q] = acc[j][q];
  }
  __syncthreads();
  if (warp > 0) return;
  float* part = p.parts + l.part + (int64_t)split * l.co * (9 * l.ci + 1);
#pragma unroll
  for (int j = 0; j < 10; ++j)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float v = ((acc[j][q] + red[0][j][lane][q]) + red[1][j][lane][q]) + red[2][j][lane][q];
      const int co = co0 + gid + (q >> 1) * 8, cc = 2 * tig + (q & 1);
      if (co >= l.co) continue;
      if (j < 9) {
        if (ci0 + cc < l.ci) part[((int64_t)co * 9 + j) * l.ci + ci0 + cc] = v;
      } else if (cc == 0 && ci0 == 0) {
        part[(int64_t)l.co * 9 * l.ci + co] = v;
      }
    }
}

// the flat gradient (each layer's weights [co][9 ci], then its bias): a
// layer's slices added in order
__global__ void sum_partials_kernel(const __grid_constant__ WArgs p) {
  after_predecessor();
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < p.nparams;
       e += (int64_t)gridDim.x * blockDim.x) {
    int li = 0;
    while (li + 1 < p.n && e >= p.l[li + 1].woff) ++li;
    const WLayer& l = p.l[li];
    const int64_t n = (int64_t)l.co * (9 * l.ci + 1);
    const float* q = p.parts + l.part + (e - l.woff);
    float a = 0.0f;
#pragma unroll 16
    for (int s = 0; s < l.splits; ++s) a += q[s * n];   // (loads ahead of the sum)
    p.grad[e] = a;
  }
}

// ------------------------------------------------------------- small passes
__global__ void to_bf16_kernel(const float* __restrict__ in, int64_t n, bf16* __restrict__ out) {
  after_predecessor();
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x)
    out[e] = __float2bfloat16_rn(in[e]);
}

// weights: master [co][9 ci] (FP32) -> W [co][kp] and Wt [9 ci][cop] (bf16,
// zero padded); blockIdx.y = layer
struct PackLayer {
  const float* w;
  int co, k9, kp, cop;
  bf16 *wb, *wt;
};
struct PackArgs {
  PackLayer l[kMaxConvs];
};
__global__ void __launch_bounds__(kT) pack_weights_kernel(const __grid_constant__ PackArgs p) {
  // 32 x 32 tiles, turned in shared memory: both copies are written by rows
  __shared__ bf16 t[32][33];
  const PackLayer& l = p.l[blockIdx.y];
  const int tk = (l.kp + 31) / 32, tiles = tk * ((l.cop + 31) / 32);
  const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;
  for (int i = blockIdx.x; i < tiles; i += gridDim.x) {
    const int co0 = i / tk * 32, k0 = i % tk * 32;
    __syncthreads();
    for (int r = ly; r < 32; r += kT / 32) {
      const int co = co0 + r, k = k0 + lx;
      const bool ok = co < l.co && k < l.k9;
      const bf16 v = __float2bfloat16_rn(ok ? l.w[(int64_t)co * l.k9 + k] : 0.0f);
      if (co < l.co && k < l.kp) l.wb[(int64_t)co * l.kp + k] = v;
      t[r][lx] = v;
    }
    __syncthreads();
    for (int r = ly; r < 32; r += kT / 32) {
      const int co = co0 + lx, k = k0 + r;
      if (k < l.k9 && co < l.cop) l.wt[(int64_t)k * l.cop + co] = t[lx][r];
    }
  }
}

// the concatenation that a decoder level's first convolution reads, written
// out (for ms_unet_layer_tensor)
__global__ void cat_kernel(Act x, int H, int W, bf16* __restrict__ cat) {
  const int cc = x.ca + x.cb;
  const int64_t total = (int64_t)H * W * cc;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = e / cc;
    cat[e] = *act_at(x, W, (int)(p / W), (int)(p % W), (int)(e - p * cc));
  }
}

// the head's pre-activation gradient bf16(2 (y - t) / P) and per-block partial
// sums of (y - t)^2 in FP64
__global__ void mse_kernel(const float* y, const float* t, int64_t P,
                           bf16* __restrict__ dz, double* __restrict__ parts) {
  after_predecessor();
  __shared__ double red[kT / 32];
  double s = 0.0;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < P;
       p += (int64_t)gridDim.x * blockDim.x) {
    const float d = y[p] - t[p];
    dz[p] = __float2bfloat16_rn(2.0f * d / (float)P);
    s += (double)d * (double)d;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0;
    for (int w = 0; w < kT / 32; ++w) a += red[w];
    parts[blockIdx.x] = a;
  }
}

// Adam (Kingma and Ba 2015) on the FP32 master weights and biases
__global__ void adam_kernel(float* __restrict__ w, const float* __restrict__ gw, int64_t n,
                            float* __restrict__ m, float* __restrict__ v, float lr, float b1,
                            float b2, float c1, float c2, float eps) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const float g = gw[e];
    const float mm = b1 * m[e] + (1.0f - b1) * g;
    const float vv = b2 * v[e] + (1.0f - b2) * g * g;
    m[e] = mm;
    v[e] = vv;
    w[e] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
  }
}
}  // namespace
}  // namespace ms

// ====================================================================== host
using namespace ms;

namespace {
struct Layer {
  int ci, co, kp, cop, level;   // input / output channels, padded K and Co, resolution level
  bool relu;
  size_t woff;                  // offset of the weights in the master array (bias after)
  bf16 *Wb = nullptr, *Wt = nullptr;         // packed bf16 weights
  Act in;                                    // forward input (bf16 [P][ci])
  bf16* out = nullptr;                       // forward output (bf16 [P][co]) (not the head)
  bf16* dz = nullptr;                        // pre-activation gradient (bf16 [P][co])
};

struct Fail {
  ms_status st;
  std::string msg;
};
void ck(cudaError_t e, const char* what) {
  if (e != cudaSuccess)
    throw Fail{e == cudaErrorMemoryAllocation ? MS_ERR_OOM : MS_ERR_CUDA,
               std::string(what) + ": " + cudaGetErrorString(e)};
}
}  // namespace

struct ms_unet {
  int levels = 0, width = 0, max_side = 0, dev = 0;
  std::vector<Layer> L;
  size_t nparams = 0;
  float* master = nullptr;   // FP32 weights and biases, conv after conv
  float *grad = nullptr, *am = nullptr, *av = nullptr;   // gradient and Adam state, as master
  std::vector<void*> allocs;
  // activations (bf16): the layers' outputs, the network's input and the
  // pooled image of each encoder level
  bf16* xin = nullptr;
  std::vector<bf16*> pooled;
  float* head = nullptr;     // a training step's output
  float* wparts = nullptr;   // partial sums of the weight gradients
  int64_t wparts_n = 0;
  std::vector<float*> dskip; // skip gradients (FP32) of the encoder levels
  double* parts = nullptr;
  int adam_t = 0;
  bool keep = false;         // the checking aid is on
  bool kept = false;         // a backward pass has run with it on
  int last_h = 0, last_w = 0;   // image size of the last forward pass
  std::string msg;
  template <typename T> T* alloc(size_t n) {
    void* p = nullptr;
    ck(cudaMalloc(&p, sizeof(T) * (n ? n : 1)), "allocation");
    allocs.push_back(p);
    return (T*)p;
  }
  ~ms_unet() {
    for (void* p : allocs) cudaFree(p);
  }
};

int ms_unet_device_of(const ms_unet* net) { return net ? net->dev : -1; }

namespace {
template <typename F> ms_status guard(ms_unet* u, F&& f) {
  if (!u) return MS_ERR_ARG;
  try {
    u->msg.clear();
    f();
    return MS_OK;
  } catch (const Fail& e) {
    u->msg = e.msg;
    return e.st;
  }
}

void arg(bool ok, const char* what) {
  if (!ok) throw Fail{MS_ERR_ARG, what};
}

// ------------------------------------------------------------------ launches
constexpr size_t kSmemMax = 227 * 1024;   // a block's shared memory on sm_103a
// Above this a 16 x 16 tile leaves room for one block per SM: smaller tiles.
constexpr size_t kSmemBig = 110 * 1024;

// Tile side, n8 tiles per block and channels staged at a time of one layer
// (n output channels of the product, c channels staged, smem(big, ck, nt)).
// 16 x 16 pixels where two waves of them fill the SMs, else 8 x 8; then the
// most n8 tiles (fewest re-reads of the pixels) that divide the layer's, leave
// a block per SM and whose weights fit beside the pixels (288 -> 96 channels at
// 64 px: 3 n8 tiles a block 34.9 us, one 41).
struct Shape {
  bool big;
  int nt, ck;
};
template <class F> Shape pick_shape(int H, int W, int n, int c, F smem) {
  const int n8 = (n + 7) / 8;
  const int64_t tb = (int64_t)((H + 15) / 16) * ((W + 15) / 16);
  const int64_t ts = (int64_t)((H + 7) / 8) * ((W + 7) / 8);
  auto nt_for = [&](bool big, int64_t tiles, size_t limit) {
    for (int nt : {4, 3, 2})
      if (n8 % nt == 0 && tiles * (n8 / nt) >= sm_count() && smem(big, c, nt) <= limit) return nt;
    return 1;
  };
  Shape s{true, nt_for(true, tb, kSmemBig), c};
  if (tb * (n8 / s.nt) >= 2 * sm_count() && smem(true, c, s.nt) <= kSmemBig) return s;
  s = Shape{false, nt_for(false, ts, kSmemMax), c};
  if (smem(false, c, s.nt) <= kSmemMax) return s;
  while (smem(false, s.ck, 1) > kSmemMax) s.ck = (s.ck - 1) / 16 * 16;   // (16 channels fit)
  return s;
}

template <class K, class A>
void launch(K kern, dim3 grid, int threads, size_t smem, const A& p, cudaStream_t s) {
  if (smem > 48 * 1024)
    ck(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
       "shared memory");
  ck(launch_pdl(kern, grid, dim3(threads), smem, s, p), "launch");
}
#define MS_BY_NT(NTV, CALL)              \
  switch (NTV) {                         \
    case 1: { constexpr int NT = 1; CALL; break; } \
    case 2: { constexpr int NT = 2; CALL; break; } \
    case 3: { constexpr int NT = 3; CALL; break; } \
    default: { constexpr int NT = 4; CALL; break; } \
  }
#define MS_BY_VEC(VECV, CALL)            \
  switch (VECV) {                        \
    case 8: { constexpr int VEC = 8; CALL; break; } \
    case 2: { constexpr int VEC = 2; CALL; break; } \
    default: { constexpr int VEC = 1; CALL; break; } \
  }

// The layers of conv_wide_kernel: those whose channels conv_kernel cannot hold
// at once; from 96 input and 64 output channels on where 16 x 16 tiles make a
// block for every SM; and from 289 on (193 where the pixels are no whole 16-byte
// chunks, which costs conv_kernel an operand read per lane) where 8 x 8 tiles do
// for half of them.  Forward pass, us, this rule | conv_kernel throughout, in
// chunks of channels where it must | the products on written-out windows before
// both: 4 levels of width 64 at 512 px 1246 | 11100 | 8790, 3 of 128 at 128 px
// 531 | 2626 | 1430, 3 of 75 at 128 px 532 | 1039 | 884.  With fewer blocks
// conv_kernel's 8 channels a block win (6 levels of 10 at 256 px 158 | 196 wide
// from 193 on).  Narrower layers keep its order of summation: rounded to
// bfloat16 layer after layer, another order's last bits move a pass of the
// configured network by 1.5 %, half of its distance from exact arithmetic.
constexpr int kWideBig = 96, kWideSmall = 289, kWideSmallOdd = 193;
void conv_forward(ms_unet* u, Layer& l, const Act& x, int H, int W, bf16* pooled,
                  const float* head_in, float* head_out, cudaStream_t s) {
  l.in = x;
  const float* bias = u->master + l.woff + (size_t)l.co * 9 * l.ci;
  const ConvArgs p{x,    H,     W,      l.ci,    l.co,     l.kp, l.cop,    l.Wb, l.Wt,
                   bias, l.out, pooled, head_in, head_out, l.ci, act_vec(x)};
  const auto tiles = [&](int S) { return ((H + S - 1) / S) * ((W + S - 1) / S); };
  const int nw = (l.co + kWideN - 1) / kWideN;
  const bool big =
      l.ci >= kWideBig && l.co >= kWideN && (int64_t)tiles(16) * nw >= sm_count();
  const bool small = l.ci >= (p.vec == 8 ? kWideSmall : kWideSmallOdd) &&
                     (int64_t)tiles(8) * nw >= sm_count() / 2;
  if (l.out && (big || small || conv_smem<false>(l.ci, 1) > kSmemMax)) {
    const dim3 grid(tiles(big ? 16 : 8), nw);
    MS_BY_VEC(p.vec, {
      if (big)
        launch(conv_wide_kernel<true, VEC>, grid, Wide<true>::Threads, Wide<true>::Smem, p, s);
      else
        launch(conv_wide_kernel<false, VEC>, grid, Wide<false>::Threads, Wide<false>::Smem, p, s);
    })
    return;
  }
  const Shape sh = pick_shape(H, W, l.co, l.ci, [](bool big, int c, int nt) {
    return big ? conv_smem<true>(c, nt) : conv_smem<false>(c, nt);
  });
  const int n8 = (l.co + 7) / 8;
  const dim3 grid(tiles(sh.big ? 16 : 8), (n8 + sh.nt - 1) / sh.nt);
  const size_t smem = sh.big ? conv_smem<true>(l.ci, sh.nt) : conv_smem<false>(l.ci, sh.nt);
  MS_BY_VEC(p.vec, MS_BY_NT(sh.nt, {
    if (sh.big) launch(conv_kernel<true, NT, VEC>, grid, 128, smem, p, s);
    else launch(conv_kernel<false, NT, VEC>, grid, 128, smem, p, s);
  }))
}

// the input gradient of layer l, put where p (mode, out_a, dz_a, skip_g) says
void conv_backward(Layer& l, int H, int W, DxArgs p, cudaStream_t s) {
  p.dz = l.dz;
  p.wt = l.Wt;
  p.H = H;
  p.W = W;
  p.ci = l.ci;
  p.co = l.co;
  p.cop = l.cop;
  const Shape sh = pick_shape(H, W, l.ci, l.co, [](bool big, int c, int nt) {
    return big ? dx_smem<true>(c, nt) : dx_smem<false>(c, nt);
  });
  p.ck = sh.ck;
  const int S = sh.big ? 16 : 8, n8 = (l.ci + 7) / 8;
  const dim3 grid(((H + S - 1) / S) * ((W + S - 1) / S), (n8 + sh.nt - 1) / sh.nt);
  const size_t smem = sh.big ? dx_smem<true>(sh.ck, sh.nt) : dx_smem<false>(sh.ck, sh.nt);
  const Act dz{l.dz, nullptr, l.co, 0};
  MS_BY_VEC(act_vec(dz), MS_BY_NT(sh.nt, {
    if (sh.big) launch(dx_kernel<true, NT, VEC>, grid, 256, smem, p, s);
    else launch(dx_kernel<false, NT, VEC>, grid, 128, smem, p, s);
  }))
}

// The weight-gradient launch of the last backward pass's image size: units of
// at most kWUnitTiles pixel tiles (one FP32 chain of mma products covers at
// most 32 of their pixels each), fewer where a layer has few units.
constexpr int kWUnitTiles = 16;
WArgs weight_args(ms_unet* u, int H, int W, int* nblocks, int64_t* nparts) {
  WArgs a{};
  a.n = (int)u->L.size();
  a.parts = u->wparts;
  a.grad = u->grad;
  a.nparams = (int64_t)u->nparams;
  int first = 0;
  int64_t part = 0;
  for (int i = 0; i < a.n; ++i) {
    const Layer& l = u->L[i];
    WLayer& w = a.l[i];
    w.x = l.in;
    w.dz = l.dz;
    w.H = H >> l.level;
    w.W = W >> l.level;
    w.ci = l.ci;
    w.co = l.co;
    w.cob = (l.co + 15) / 16;
    w.cib = (l.ci + 7) / 8;
    w.tiles_x = (w.W + kWTileX - 1) / kWTileX;
    w.tiles = w.tiles_x * ((w.H + kWTileY - 1) / kWTileY);
    w.per = std::min(kWUnitTiles, w.tiles);
    w.splits = (w.tiles + w.per - 1) / w.per;
    w.first = first;
    w.vx = act_vec(l.in);
    w.vz = act_vec(Act{l.dz, nullptr, l.co, 0});
    w.part = part;
    w.woff = (int64_t)l.woff;
    first += w.splits * w.cob * w.cib;
    part += (int64_t)w.splits * l.co * (9 * l.ci + 1);
  }
  *nblocks = first;
  *nparts = part;
  return a;
}

void pack(ms_unet* u, cudaStream_t s) {
  PackArgs p{};
  int64_t most = 0;
  for (size_t i = 0; i < u->L.size(); ++i) {
    const Layer& l = u->L[i];
    p.l[i] = PackLayer{u->master + l.woff, l.co, 9 * l.ci, l.kp, l.cop, l.Wb, l.Wt};
    most = std::max(most, (int64_t)((l.kp + 31) / 32) * ((l.cop + 31) / 32));
  }
  pack_weights_kernel<<<dim3((unsigned)std::min<int64_t>(most, 1024), (unsigned)u->L.size()), kT,
                        0, s>>>(p);
}

// out = net(in) [H][W] (FP32)
void forward(ms_unet* u, const float* in, int H, int W, float* out, cudaStream_t s) {
  arg(H >= 4 && W >= 4 && H <= u->max_side && W <= u->max_side, "image side out of range");
  arg(H % (4 << (u->levels - 1)) == 0 && W % (4 << (u->levels - 1)) == 0,
      "image sides must be divisible by 4 * 2^(levels-1)");
  pack(u, s);
  u->last_h = H;
  u->last_w = W;
  const int Lv = u->levels;
  ck(launch_pdl(to_bf16_kernel, dim3(blocks((int64_t)H * W * 2)), dim3(kT), 0, s, in,
                (int64_t)H * W * 2, u->xin), "launch");
  size_t li = 0;
  Act x{u->xin, nullptr, 2, 0};
  int h = H, w = W;
  for (int lv = 0; lv < Lv; ++lv) {
    Layer& l0 = u->L[li++];
    conv_forward(u, l0, x, h, w, nullptr, nullptr, nullptr, s);
    Layer& l1 = u->L[li++];
    conv_forward(u, l1, Act{l0.out, nullptr, l0.co, 0}, h, w,
                 lv < Lv - 1 ? u->pooled[lv] : nullptr, nullptr, nullptr, s);
    if (lv < Lv - 1) {
      x = Act{u->pooled[lv], nullptr, l1.co, 0};
      h /= 2;
      w /= 2;
    }
  }
  const bf16* lo = u->L[li - 1].out;
  int clo = u->L[li - 1].co;
  for (int lv = Lv - 2; lv >= 0; --lv) {
    h *= 2;
    w *= 2;
    Layer& l0 = u->L[li++];
    conv_forward(u, l0, Act{lo, u->L[2 * lv + 1].out, clo, u->width << lv}, h, w, nullptr, nullptr,
                 nullptr, s);
    Layer& l1 = u->L[li++];
    conv_forward(u, l1, Act{l0.out, nullptr, l0.co, 0}, h, w, nullptr, nullptr, nullptr, s);
    lo = l1.out;
    clo = l1.co;
  }
  conv_forward(u, u->L[li], Act{lo, nullptr, clo, 0}, h, w, nullptr, in, out, s);
}

// gradients of the mean squared error of out = net(in) against target into
// u->grad; the loss's partial sums into u->parts (their number returned)
int backward(ms_unet* u, const float* target, int H, int W, const float* out, cudaStream_t s) {
  const int64_t P = (int64_t)H * W;
  const int nb = blocks(P, 1024);
  const int Lv = u->levels;
  int li = (int)u->L.size() - 1;
  ck(launch_pdl(mse_kernel, dim3(nb), dim3(kT), 0, s, out, target, P, u->L[li].dz, u->parts),
     "launch");
  auto through = [&](Layer& prev) {   // the input is prev's output
    DxArgs p{};
    p.mode = 0;
    p.out_a = prev.out;
    p.dz_a = prev.dz;
    return p;
  };
  conv_backward(u->L[li], H, W, through(u->L[li - 1]), s);   // head
  --li;
  int h = H, w = W;
  for (int lv = 0; lv <= Lv - 2; ++lv) {   // decoder, finest level first
    conv_backward(u->L[li], h, w, through(u->L[li - 1]), s);
    --li;
    Layer& below = u->L[li - 1];   // its output is upsampled into the concatenation
    DxArgs p{};
    p.mode = 1;
    p.ca = below.co;
    p.out_a = below.out;
    p.dz_a = below.dz;
    p.skip_g = u->dskip[lv];
    conv_backward(u->L[li], h, w, p, s);
    --li;
    h /= 2;
    w /= 2;
  }
  for (int lv = Lv - 1; lv >= 0; --lv) {   // bottom and encoder; h, w: level lv
    conv_backward(u->L[li], h, w, through(u->L[li - 1]), s);
    --li;
    if (lv > 0) {   // the input is level lv - 1's pooled output
      Layer& above = u->L[li - 1];
      DxArgs p{};
      p.mode = 2;
      p.out_a = above.out;
      p.dz_a = above.dz;
      p.skip_g = u->dskip[lv - 1];
      conv_backward(u->L[li], h, w, p, s);
    }
    --li;
    h *= 2;
    w *= 2;
  }
  int wb = 0;
  int64_t np = 0;
  const WArgs a = weight_args(u, H, W, &wb, &np);
  arg(np <= u->wparts_n, "weight-gradient partial sums");
  launch(dw_kernel, dim3(wb), 128, 0, a, s);
  launch(sum_partials_kernel, dim3(blocks(a.nparams)), kT, 0, a, s);
  if (u->keep) u->kept = true;
  return nb;
}

// the mean squared error from backward's partial sums (synchronizes)
double read_loss(ms_unet* u, int nb, int64_t P, cudaStream_t s) {
  std::vector<double> hp(nb);
  ck(cudaMemcpyAsync(hp.data(), u->parts, sizeof(double) * nb, cudaMemcpyDeviceToHost, s),
     "loss");
  ck(cudaStreamSynchronize(s), "synchronize");
  double sum = 0.0;
  for (double v : hp) sum += v;
  return sum / (double)P;
}
}  // namespace

extern "C" {

ms_status ms_unet_create(int32_t levels, int32_t width, int32_t max_side, uint64_t seed,
                         int32_t device, ms_unet** out) {
  if (!out || levels < 2 || levels > 6 || width < 1 || width > 256 || max_side < 8 ||
      max_side > 8192)
    return MS_ERR_ARG;
  *out = nullptr;
  ms_unet* u = new ms_unet();
  ms_status st = guard(u, [&] {
    u->levels = levels;
    u->width = width;
    u->max_side = max_side;
    u->dev = device;
    ck(cudaSetDevice(device), "set device");
    // layers in execution order: encoder + bottom, decoder, head
    auto add = [&](int co, int ci, int level, bool relu) {
      Layer l{};
      l.ci = ci;
      l.co = co;
      l.kp = pad16(9 * ci);
      l.cop = pad16(co);
      l.level = level;
      l.relu = relu;
      l.woff = u->nparams;
      u->nparams += (size_t)co * 9 * ci + co;
      u->L.push_back(l);
    };
    int cin = 2;
    for (int lv = 0; lv < levels; ++lv) {
      const int c = width << lv;
      add(c, cin, lv, true);
      add(c, c, lv, true);
      cin = c;
    }
    for (int lv = levels - 2; lv >= 0; --lv) {
      const int c = width << lv;
      add(c, (width << (lv + 1)) + c, lv, true);
      add(c, c, lv, true);
    }
    add(1, width, 0, false);
    u->master = u->alloc<float>(u->nparams);
    // He-normal initialization on the host (Box-Muller on a 64-bit LCG)
    std::vector<float> h(u->nparams, 0.0f);
    uint64_t st64 = seed * 6364136223846793005ULL + 1442695040888963407ULL;
    auto uni = [&]() {
      st64 = st64 * 6364136223846793005ULL + 1442695040888963407ULL;
      return ((st64 >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    };
    for (Layer& l : u->L) {
      // the head starts at zero: the untrained network returns its first
      // input channel (the step-one image) unchanged, and training learns a
      // correction to it
      if (!l.relu) continue;
      const double sd = std::sqrt(2.0 / (9.0 * l.ci));
      for (size_t i = 0; i < (size_t)l.co * 9 * l.ci; ++i) {
        const double r = std::sqrt(-2.0 * std::log(uni())), t = 6.283185307179586 * uni();
        h[l.woff + i] = (float)(sd * r * std::cos(t));
      }
    }
    ck(cudaMemcpy(u->master, h.data(), sizeof(float) * u->nparams, cudaMemcpyHostToDevice),
       "init");
    const int64_t P0 = (int64_t)max_side * max_side;
    u->grad = u->alloc<float>(u->nparams);
    u->am = u->alloc<float>(u->nparams);
    u->av = u->alloc<float>(u->nparams);
    ck(cudaMemset(u->am, 0, sizeof(float) * u->nparams), "memset");
    ck(cudaMemset(u->av, 0, sizeof(float) * u->nparams), "memset");
    for (Layer& l : u->L) {
      l.Wb = u->alloc<bf16>((size_t)l.co * l.kp);
      l.Wt = u->alloc<bf16>((size_t)9 * l.ci * l.cop);
      const int64_t Pl = P0 >> (2 * l.level);
      if (l.relu) l.out = u->alloc<bf16>((size_t)Pl * l.co);
      l.dz = u->alloc<bf16>((size_t)Pl * l.co);
    }
    u->xin = u->alloc<bf16>((size_t)P0 * 2);
    for (int lv = 0; lv < levels - 1; ++lv) {
      const int64_t Pl = P0 >> (2 * lv);
      const int c = width << lv;
      u->pooled.push_back(u->alloc<bf16>((size_t)(Pl / 4) * c));
      u->dskip.push_back(u->alloc<float>((size_t)Pl * c));
    }
    u->head = u->alloc<float>((size_t)P0);
    u->parts = u->alloc<double>(1024);
    // the most slices any image size takes (tiles cut at the sides add at
    // most one column and one row of them)
    for (const Layer& l : u->L) {
      const int64_t side = max_side >> l.level;
      const int64_t tiles = (side / kWTileX + 1) * (side / kWTileY + 1);
      u->wparts_n += (tiles / kWUnitTiles + 1) * l.co * (9 * (int64_t)l.ci + 1);
    }
    u->wparts = u->alloc<float>((size_t)u->wparts_n);
    ck(cudaDeviceSynchronize(), "create");
  });
  if (st != MS_OK) {
    delete u;
    return st;
  }
  *out = u;
  return MS_OK;
}

ms_status ms_unet_destroy(ms_unet* u) {
  if (!u) return MS_ERR_ARG;
  cudaSetDevice(u->dev);
  delete u;
  return MS_OK;
}

const char* ms_unet_last_error(const ms_unet* u) { return u ? u->msg.c_str() : "no network"; }

ms_status ms_unet_param_count(const ms_unet* u, int64_t* n) {
  if (!u || !n) return MS_ERR_ARG;
  *n = (int64_t)u->nparams;
  return MS_OK;
}

ms_status ms_unet_get_params(ms_unet* u, float* host, int64_t n) {
  return guard(u, [&] {
    arg(host && n == (int64_t)u->nparams, "host buffer of param_count floats required");
    ck(cudaSetDevice(u->dev), "set device");
    ck(cudaMemcpy(host, u->master, sizeof(float) * n, cudaMemcpyDeviceToHost), "copy");
  });
}

ms_status ms_unet_set_params(ms_unet* u, const float* host, int64_t n) {
  return guard(u, [&] {
    arg(host && n == (int64_t)u->nparams, "host buffer of param_count floats required");
    ck(cudaSetDevice(u->dev), "set device");
    ck(cudaMemcpy(u->master, host, sizeof(float) * n, cudaMemcpyHostToDevice), "copy");
    u->adam_t = 0;
    ck(cudaMemset(u->am, 0, sizeof(float) * n), "memset");
    ck(cudaMemset(u->av, 0, sizeof(float) * n), "memset");
  });
}

ms_status ms_unet_forward(ms_unet* u, const float* in, int32_t H, int32_t W, float* out,
                          void* stream) {
  return guard(u, [&] {
    arg(in && out, "in and out are required");
    ck(cudaSetDevice(u->dev), "set device");
    cudaStream_t s = (cudaStream_t)stream;
    forward(u, in, H, W, out, s);
    ck(cudaGetLastError(), "kernel launch");
  });
}

ms_status ms_unet_gradients(ms_unet* u, const float* in, const float* target, int32_t H,
                            int32_t W, float* out, float* grads_host, double* loss,
                            void* stream) {
  return guard(u, [&] {
    arg(in && target && out, "in, target and out are required");
    ck(cudaSetDevice(u->dev), "set device");
    cudaStream_t s = (cudaStream_t)stream;
    forward(u, in, H, W, out, s);
    const int nb = backward(u, target, H, W, out, s);
    if (grads_host)
      ck(cudaMemcpyAsync(grads_host, u->grad, sizeof(float) * u->nparams, cudaMemcpyDeviceToHost,
                         s),
         "copy gradients");
    const double l = read_loss(u, nb, (int64_t)H * W, s);   // (waits for the copy too)
    if (loss) *loss = l;
    ck(cudaGetLastError(), "kernel launch");
  });
}

ms_status ms_unet_keep_intermediates(ms_unet* u, int32_t keep) {
  return guard(u, [&] {
    u->keep = keep != 0;
  });
}

ms_status ms_unet_layer_tensor(ms_unet* u, int32_t layer, int32_t which, float* host, int64_t n) {
  return guard(u, [&] {
    arg(layer >= 0 && layer < (int)u->L.size(), "layer out of range");
    arg(which >= 0 && which <= 2, "which must be 0 (input), 1 (output) or 2 (gradient)");
    arg(u->last_h > 0, "no forward pass yet");
    const Layer& l = u->L[layer];
    const int64_t P = (int64_t)(u->last_h >> l.level) * (u->last_w >> l.level);
    const int c = which == 0 ? l.ci : l.co;
    arg(host && n == P * c, "host buffer of H_l W_l channels floats required");
    const bool have = which == 0 || (which == 1 ? l.out != nullptr : u->kept);
    arg(have, which == 1 ? "the head keeps no bfloat16 output"
                         : "no kept gradient: enable ms_unet_keep_intermediates "
                           "before ms_unet_gradients");
    ck(cudaSetDevice(u->dev), "set device");
    const bf16* src = which == 0 ? l.in.a : (which == 1 ? l.out : l.dz);
    bf16* cat = nullptr;
    if (which == 0 && l.in.cb) {   // a concatenation is read in place: write it out
      ck(cudaDeviceSynchronize(), "synchronize");
      ck(cudaMalloc(&cat, sizeof(bf16) * P * c), "allocation");
      cat_kernel<<<blocks(P * c), kT>>>(l.in, u->last_h >> l.level, u->last_w >> l.level, cat);
      src = cat;
    }
    std::vector<bf16> h((size_t)P * c);
    const cudaError_t e = cudaMemcpy(h.data(), src, sizeof(bf16) * h.size(),
                                     cudaMemcpyDeviceToHost);
    if (cat) cudaFree(cat);
    ck(e, "copy");
    for (size_t k = 0; k < h.size(); ++k) host[k] = __bfloat162float(h[k]);
  });
}

ms_status ms_unet_train_step(ms_unet* u, const float* in, const float* target, int32_t H,
                             int32_t W, float lr, double* loss, void* stream) {
  return guard(u, [&] {
    arg(in && target, "in and target are required");
    ck(cudaSetDevice(u->dev), "set device");
    cudaStream_t s = (cudaStream_t)stream;
    forward(u, in, H, W, u->head, s);
    const int nb = backward(u, target, H, W, u->head, s);
    const double l = read_loss(u, nb, (int64_t)H * W, s);
    if (loss) *loss = l;
    u->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - std::pow(b1, (float)u->adam_t);
    const float c2 = 1.0f - std::pow(b2, (float)u->adam_t);
    adam_kernel<<<blocks((int64_t)u->nparams), kT, 0, s>>>(
        u->master, u->grad, (int64_t)u->nparams, u->am, u->av, lr, b1, b2, c1, c2, 1e-8f);
    ck(cudaGetLastError(), "kernel launch");
  });
}

}  // extern "C"
