// The two convolution blocks of the paper's model class (see conv.cuh for the operation) in bf16 storage on the
// warp-level tensor-core instruction (mma m16n8k16, bf16 operands, fp32 accumulation): both blocks forward in one
// kernel, both backward in another; maps stay in shared memory, nothing is expanded to im2col rows.
//
//   forward   rows of the product = output pixels, columns = output channels, inner index = (dy, (dx, ci)): for one dy
//             the k Ci inputs of a pixel are contiguous in an [y][x][ci] map (padded to a multiple of 16 with zero
//             weights).  The 16 rows of a tile are 8 pooled pixels x 2 window columns, and the tiles of both window
//             rows run together, so a thread ends up with the four window positions of its pooled pixel and the row
//             operands of window row 1 at dy are those of window row 0 at dy + 1 (loaded once).
//   delta of the second block's input   rows = input pixels, inner index = (dy, dx, co), from the dense delta map with
//             a zero border; it is scattered straight to the first block's window positions.
//   weights   rows = (dy, dx, ci) (+ one row of ones: the bias), columns = co, inner index = output pixels, from
//             [ci][y][x] maps; pixel pairs need an even start, so a copy shifted by one element serves odd dx (in the
//             forward pass: odd x Ci).
// FP32-FMA kernels with one CTA per row spent 315 us of a 640-row round of the 32 x 32 x 3 network here (5 % of the
// FMA peak, bound by shared-memory reads per FMA); @@CONV@@
#pragma once
#include "common.cuh"
#include "outlayer.cuh"

namespace absb {
namespace cmma {

typedef __nv_bfloat16 bf16;
constexpr int NT = 256, NWARP = NT / 32;
constexpr int FR = 2;                    // gradient rows per CTA (divides the row padding unit)
constexpr int MT1 = 6;                   // most 16-row tiles of the first block's weight gradient (per warp)
constexpr int MT2 = 2;                   // ... of the second block's (16 tiles over 8 warps)

struct Block { int Hi, Wi, Ci, Ho, Wo, Ph, Pw, Co; size_t w_off; };
struct Args {
  DevState* st;
  RoundInfo* ri;
  const int* tile_slot;
  const int* row_idx;
  const void* ring; size_t slot_stride;
  int k;
  Block b[2];
  const bf16* X;                         // dataset images
  bf16* pool1; unsigned char* arg1;      // [rows][Ph1][Pw1][C1] pooled maps of the first block, position of each maximum
  bf16* feat; unsigned char* arg2;       // [rows][Ph2][Pw2][C2] the same of the second block: the features
  const bf16* dfeat;                     // [rows][...] delta of the features (zero where the feature is not positive)
  float* part[2];                        // [chunks of FR rows][k k Ci Co + Co] sums of the weight and bias gradient
};

__host__ __device__ inline int even(int n) { return (n + 1) & ~1; }

// ---- shared-memory layouts (byte offsets)
struct FwdLayout { int e1, o1, e2, o2, a1, f2, a2, row, b1, b2, bias, total; };
__host__ __device__ inline FwdLayout fwd_layout(int k, const Block& x, const Block& y) {
  FwdLayout f;
  int off = 0;
  auto take = [&](int bytes) { const int o = off; off += round_up(bytes, 16); return o; };
  const int m1 = 2 * (x.Hi * even(x.Wi * x.Ci) + 64), m2 = 2 * (y.Hi * even(y.Wi * y.Ci) + 64);
  f.e1 = take(m1); f.o1 = (x.Ci & 1) ? take(m1) : 0;
  f.e2 = take(m2); f.o2 = (y.Ci & 1) ? take(m2) : 0;
  f.a1 = take(x.Ph * x.Pw * x.Co);
  f.f2 = take(2 * y.Ph * y.Pw * y.Co);
  f.a2 = take(y.Ph * y.Pw * y.Co);
  f.row = off;                           // the maps of one gradient row; FR of them
  off *= FR;
  f.b1 = take(k * ((k * x.Ci + 15) / 16) * 256);
  f.b2 = take(k * ((k * y.Ci + 15) / 16) * ((y.Co + 7) / 8) * 256);
  f.bias = take(4 * (8 + 16));
  f.total = off;
  return f;
}
struct BwdLayout { int im, in2, dz1, dz2, dzb, a1, bd, pw1, pw2, total; int px1, px2, plane1, plane2, pz1, pz2, zw; };
// words between the channels of a dense delta map: 4 mod 8, so that 8 channels x 4 lanes hit 32 different banks
__host__ __device__ inline int dz_pitch(int pixels) { return round_up(round_up(pixels, 16) / 2, 8) + 4; }
__host__ __device__ inline BwdLayout bwd_layout(int k, const Block& x, const Block& y) {
  BwdLayout f;
  int off = 0;
  auto take = [&](int bytes) { const int o = off; off += round_up(bytes, 16); return o; };
  f.px1 = even(x.Wi); f.px2 = even(y.Wi);
  f.plane1 = x.Hi * f.px1; f.plane2 = y.Hi * f.px2;
  f.pz1 = dz_pitch(x.Ho * x.Wo); f.pz2 = dz_pitch(y.Ho * y.Wo);
  f.zw = y.Wo + 2 * (k - 1);
  f.im = take(2 * 2 * x.Ci * f.plane1 + 16);          // two copies, the second shifted by one element
  f.in2 = take(2 * 2 * y.Ci * f.plane2 + 16);
  f.dz1 = take(4 * 8 * f.pz1);
  f.dz2 = take(4 * 16 * f.pz2);
  f.dzb = take(2 * 24 * (y.Ho + 2 * (k - 1)) * f.zw);
  f.a1 = take(x.Ph * x.Pw * x.Co);
  f.bd = take(k * k * 256);
  f.pw1 = take(2 * (round_up(x.Ho * x.Wo, 16) / 2));
  f.pw2 = take(2 * (round_up(y.Ho * y.Wo, 16) / 2));
  f.total = off;
  const int red = 4 * NWARP * MT1 * 16 * 8;            // the first block's sums of the warps, over the maps at the end
  if (f.total < red) f.total = red;
  return f;
}
// model classes these kernels take
inline bool fits(int k, const Block& x, const Block& y) {
  return x.Co <= 8 && y.Co <= 16 && k * k * x.Ci + 1 <= 16 * MT1 && k * k * y.Ci + 1 <= 16 * MT2 * NWARP &&
         fwd_layout(k, x, y).total <= 110 * 1024 && bwd_layout(k, x, y).total <= 110 * 1024 &&
         x.Hi * even(x.Wi) < 65536 && y.Hi * even(y.Wi) < 65536;
}

__device__ __forceinline__ uint32_t join16(bf16 lo, bf16 hi) {
  return (uint32_t)*reinterpret_cast<unsigned short*>(&lo) | ((uint32_t)*reinterpret_cast<unsigned short*>(&hi) << 16);
}

// column operand of the forward products: fragment of inner step (dy, s) and column tile n: W[dy][16 s + ..][8 n + ..]
__device__ __forceinline__ void forward_weights(uint2* bf, const bf16* w, int k, int len, int Co, int n_ct) {
  const int ks = (len + 15) / 16;
  for (int e = threadIdx.x; e < k * ks * n_ct * 32; e += NT) {
    const int lane = e & 31, f = e >> 5, n = f % n_ct, step = f / n_ct;
    const int dy = step / ks, kk = (step - dy * ks) * 16 + 2 * (lane & 3), co = n * 8 + (lane >> 2);
    auto at = [&](int q) { return (q < len && co < Co) ? w[((size_t)dy * len + q) * Co + co] : (bf16)0.f; };
    bf[e] = make_uint2(join16(at(kk), at(kk + 1)), join16(at(kk + 8), at(kk + 9)));
  }
}

// One task of a forward block: 8 pooled pixels, all channels; results to `out` (pitch: elements between pooled rows) and
// `arg` ([pixel][Co]).
template <int NC>
__device__ __forceinline__ void forward_task(const Block& b, int k, const bf16* E, const bf16* O, const uint2* bf, const float* bias,
                                             int q0, bf16* out, int pitch, unsigned char* arg, int lane) {
  const int g = lane >> 2, t = lane & 3;
  const int P = even(b.Wi * b.Ci), ks = (k * b.Ci + 15) / 16, n_q = b.Ph * b.Pw;
  const int q = min(q0 + g, n_q - 1), py = q / b.Pw, px = q - py * b.Pw;
  const int at = 2 * py * P + 2 * px * b.Ci;          // even
  const uint32_t* p0 = reinterpret_cast<const uint32_t*>(E + at) + t;
  const uint32_t* p1 = reinterpret_cast<const uint32_t*>((b.Ci & 1) ? O + at + b.Ci - 1 : E + at + b.Ci) + t;
  float acc[2][NC][4];
#pragma unroll
  for (int w = 0; w < 2; ++w)
#pragma unroll
    for (int n = 0; n < NC; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[w][n][i] = 0.f;
  const uint2* bl = bf + lane;
  for (int i = 0; i <= k; ++i) {
#pragma unroll 2
    for (int s = 0; s < ks; ++s) {
      const int o = (i * P) / 2 + 8 * s;
      const uint32_t a[4] = {p0[o], p1[o], p0[o + 4], p1[o + 4]};
#pragma unroll
      for (int n = 0; n < NC; ++n) {
        if (i < k) {
          const uint2 w = bl[((i * ks + s) * NC + n) * 32];
          outl::mma16816(acc[0][n], a, w.x, w.y);
        }
        if (i > 0) {
          const uint2 w = bl[(((i - 1) * ks + s) * NC + n) * 32];
          outl::mma16816(acc[1][n], a, w.x, w.y);
        }
      }
    }
  }
  if (q0 + g >= n_q) return;
#pragma unroll
  for (int n = 0; n < NC; ++n)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int c = 8 * n + 2 * t + j;
      if (c < b.Co) {
        // stored ReLU outputs of the window in row-major order; the first maximum wins a tie
        const float bc = bias[c];
        bf16 best = __float2bfloat16_rn(fmaxf(acc[0][n][j] + bc, 0.f));
        int where = 0;
#pragma unroll
        for (int w = 1; w < 4; ++w) {
          const bf16 v = __float2bfloat16_rn(fmaxf(acc[w >> 1][n][2 * (w & 1) + j] + bc, 0.f));
          if (__bfloat162float(v) > __bfloat162float(best)) { best = v; where = w; }
        }
        out[py * pitch + px * b.Co + c] = best;
        arg[q * b.Co + c] = (unsigned char)where;
      }
    }
}

// O[i] = E[i + 1] for n elements (n even)
__device__ __forceinline__ void shift_copy(bf16* O, const bf16* E, int n) {
  const uint32_t* e = reinterpret_cast<const uint32_t*>(E);
  uint32_t* o = reinterpret_cast<uint32_t*>(O);
  for (int i = threadIdx.x; i < n / 2; i += NT) o[i] = __byte_perm(e[i], e[i + 1], 0x5432);
}

template <typename V, typename U>
__device__ __forceinline__ void copy_out(U* dst, const U* src, int n) {
  if ((n * (int)sizeof(U)) % sizeof(V) == 0) {
    for (int i = threadIdx.x; i < n * (int)sizeof(U) / (int)sizeof(V); i += NT) reinterpret_cast<V*>(dst)[i] = reinterpret_cast<const V*>(src)[i];
  } else {
    for (int i = threadIdx.x; i < n; i += NT) dst[i] = src[i];
  }
}

static __global__ void __launch_bounds__(NT) conv_fwd_mma_kernel(const __grid_constant__ Args a) {
  grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char cs[];
  const int r0 = (int)blockIdx.x * FR;
  const int status = a.st->status, n_rows = a.ri->n_rows, RB = a.st->RB;
  int s[FR];
  bool any = false;
#pragma unroll
  for (int j = 0; j < FR; ++j) s[j] = a.row_idx[r0 + j];
  if (status != ST_OK || r0 >= n_rows) return;
#pragma unroll
  for (int j = 0; j < FR; ++j) any |= s[j] >= 0;
  if (!any) return;                                   // padding rows: nothing reads more than finite values of them
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = a.k;
  const FwdLayout f = fwd_layout(k, a.b[0], a.b[1]);
  const Block &x = a.b[0], &y = a.b[1];
  const int slot = a.tile_slot[r0 / RB];
  const bf16* ring = (const bf16*)a.ring + (size_t)slot * a.slot_stride;
  const int n_in = x.Hi * x.Wi * x.Ci, P1 = even(x.Wi * x.Ci), P2 = even(y.Wi * y.Ci);
  const int n1 = x.Ph * x.Pw * x.Co, n2 = y.Ph * y.Pw * y.Co;
  auto map = [&](int j, int off) { return reinterpret_cast<bf16*>(cs + (size_t)j * f.row + off); };
  // ---- images, weights
#pragma unroll
  for (int j = 0; j < FR; ++j) {
    bf16* E = map(j, f.e1);
    const bf16* src = a.X + (size_t)max(s[j], 0) * n_in;
    if (P1 == x.Wi * x.Ci && n_in % 8 == 0) {
#pragma unroll 4
      for (int i = tid; i < n_in / 8; i += NT) reinterpret_cast<uint4*>(E)[i] = reinterpret_cast<const uint4*>(src)[i];
    } else {
      const int wc = x.Wi * x.Ci;
      for (int yy = warp; yy < x.Hi; yy += NWARP)
        for (int i = lane; i < P1; i += 32) E[yy * P1 + i] = i < wc ? src[(size_t)yy * wc + i] : (bf16)0.f;
    }
    // what a last pixel's padded inner steps may reach behind the maps meets zero weights: it has to be finite
    if (tid < 64) { E[x.Hi * P1 + tid] = (bf16)0.f; map(j, f.e2)[y.Hi * P2 + tid] = (bf16)0.f; }
    if (P2 != y.Wi * y.Ci && tid < y.Hi) map(j, f.e2)[tid * P2 + P2 - 1] = (bf16)0.f;
  }
  const int nc2 = (y.Co + 7) / 8;
  uint2* b1 = reinterpret_cast<uint2*>(cs + f.b1);
  uint2* b2 = reinterpret_cast<uint2*>(cs + f.b2);
  float* bias = reinterpret_cast<float*>(cs + f.bias);
  forward_weights(b1, ring + x.w_off, k, k * x.Ci, x.Co, 1);
  forward_weights(b2, ring + y.w_off, k, k * y.Ci, y.Co, nc2);
  if (tid < x.Co) bias[tid] = __bfloat162float(ring[x.w_off + (size_t)k * k * x.Ci * x.Co + tid]);
  if (tid < y.Co) bias[8 + tid] = __bfloat162float(ring[y.w_off + (size_t)k * k * y.Ci * y.Co + tid]);
  __syncthreads();
  if (x.Ci & 1) {
#pragma unroll
    for (int j = 0; j < FR; ++j) shift_copy(map(j, f.o1), map(j, f.e1), x.Hi * P1 + 62);
    __syncthreads();
  }
  // ---- first block
  const int g1 = (x.Ph * x.Pw + 7) / 8, g2 = (y.Ph * y.Pw + 7) / 8;
  for (int task = warp; task < FR * g1; task += NWARP) {
    const int j = task / g1;
    forward_task<1>(x, k, map(j, f.e1), map(j, f.o1), b1, bias, (task - j * g1) * 8, map(j, f.e2), P2, cs + (size_t)j * f.row + f.a1, lane);
  }
  __syncthreads();
  if (y.Ci & 1) {
#pragma unroll
    for (int j = 0; j < FR; ++j) shift_copy(map(j, f.o2), map(j, f.e2), y.Hi * P2 + 62);
    __syncthreads();
  }
  // ---- second block; the first one's results leave meanwhile
  for (int task = warp; task < FR * g2; task += NWARP) {
    const int j = task / g2, q0 = (task - j * g2) * 8;
    if (nc2 == 1) forward_task<1>(y, k, map(j, f.e2), map(j, f.o2), b2, bias + 8, q0, map(j, f.f2), y.Pw * y.Co, cs + (size_t)j * f.row + f.a2, lane);
    else forward_task<2>(y, k, map(j, f.e2), map(j, f.o2), b2, bias + 8, q0, map(j, f.f2), y.Pw * y.Co, cs + (size_t)j * f.row + f.a2, lane);
  }
#pragma unroll
  for (int j = 0; j < FR; ++j) {
    if (s[j] < 0) continue;
    const int r = r0 + j;
    if (P2 == y.Wi * y.Ci) copy_out<uint4>(a.pool1 + (size_t)r * n1, (const bf16*)map(j, f.e2), n1);
    else
      for (int i = tid; i < n1; i += NT) a.pool1[(size_t)r * n1 + i] = map(j, f.e2)[(i / (y.Wi * y.Ci)) * P2 + i % (y.Wi * y.Ci)];
    copy_out<uint2>(a.arg1 + (size_t)r * n1, (const unsigned char*)(cs + (size_t)j * f.row + f.a1), n1);
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < FR; ++j) {
    if (s[j] < 0) continue;
    const int r = r0 + j;
    copy_out<uint4>(a.feat + (size_t)r * n2, (const bf16*)map(j, f.f2), n2);
    copy_out<uint2>(a.arg2 + (size_t)r * n2, (const unsigned char*)(cs + (size_t)j * f.row + f.a2), n2);
  }
}

// [y][x][c] map in global memory -> [c][y][x] (pitch px) in shared memory
__device__ __forceinline__ void load_planar(bf16* dst, const bf16* src, int Hi, int Wi, int Ci, int px, int plane) {
  const int wpr = px / 2, words = Hi * wpr;
  for (int c = 0; c < Ci; ++c)
#pragma unroll 4
    for (int w = threadIdx.x; w < words; w += NT) {
      const int yy = w / wpr, xx = 2 * (w - yy * wpr);
      const bf16* p = src + ((size_t)yy * Wi + xx) * Ci + c;
      reinterpret_cast<uint32_t*>(dst + c * plane)[w] = join16(p[0], xx + 1 < Wi ? p[Ci] : (bf16)0.f);
    }
}
// word offset of weight-gradient row m (tap dy, dx of input channel ci) in the two planar copies
__device__ __forceinline__ int tap_offset(int m, int K, int k, int Ci, int px, int plane) {
  if (m >= K) return 0;                               // row of ones / padding rows: any finite value
  const int ci = m % Ci, tap = m / Ci, dx = tap % k, dy = tap / k;
  return ((dx & 1) * Ci * plane + ci * plane + dy * px + dx - (dx & 1)) / 2;
}

static __global__ void __launch_bounds__(NT, 2) conv_bwd_mma_kernel(const __grid_constant__ Args a) {
  grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char cs[];
  const int r0 = (int)blockIdx.x * FR;
  const int status = a.st->status, n_rows = a.ri->n_rows, RB = a.st->RB;
  int s[FR];
#pragma unroll
  for (int j = 0; j < FR; ++j) s[j] = a.row_idx[r0 + j];
  if (status != ST_OK || r0 >= n_rows) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = a.k;
  const int g = lane >> 2, t = lane & 3;
  const BwdLayout f = bwd_layout(k, a.b[0], a.b[1]);
  const Block &x = a.b[0], &y = a.b[1];
  const int slot = a.tile_slot[r0 / RB];
  const bf16* w2 = (const bf16*)a.ring + (size_t)slot * a.slot_stride + y.w_off;
  bf16* im = reinterpret_cast<bf16*>(cs + f.im);
  bf16* in2 = reinterpret_cast<bf16*>(cs + f.in2);
  uint32_t* dz1 = reinterpret_cast<uint32_t*>(cs + f.dz1);
  uint32_t* dz2 = reinterpret_cast<uint32_t*>(cs + f.dz2);
  bf16* dzb = reinterpret_cast<bf16*>(cs + f.dzb);
  unsigned char* arg1 = cs + f.a1;
  uint2* bd = reinterpret_cast<uint2*>(cs + f.bd);
  unsigned short* pw1 = reinterpret_cast<unsigned short*>(cs + f.pw1);
  unsigned short* pw2 = reinterpret_cast<unsigned short*>(cs + f.pw2);
  const int n1 = x.Ph * x.Pw * x.Co, n2 = y.Ph * y.Pw * y.Co, n_in = x.Hi * x.Wi * x.Ci;
  const int pix1 = x.Ho * x.Wo, pix2 = y.Ho * y.Wo, st1 = (pix1 + 15) / 16, st2 = (pix2 + 15) / 16;
  const int K1 = k * k * x.Ci, K2 = k * k * y.Ci;
  const int mt1 = K1 / 16 + 1, mt2 = K2 / 16 + 1;     // row tiles including the row of ones
  const int nc2 = (y.Co + 7) / 8;
  // ---- once per CTA: weights of the second block as column operand of the delta product, pixel tables, tap offsets
  for (int e = tid; e < k * k * 32; e += NT) {
    const int l = e & 31, tap = e >> 5, ci = l >> 2, co = 2 * (l & 3);
    auto at = [&](int q) { return (q < y.Co && ci < y.Ci) ? w2[((size_t)tap * y.Ci + ci) * y.Co + q] : (bf16)0.f; };
    bd[e] = make_uint2(join16(at(co), at(co + 1)), join16(at(co + 8), at(co + 9)));
  }
  for (int j = tid; j < st1 * 8; j += NT) pw1[j] = (unsigned short)(2 * j < pix1 ? ((2 * j / x.Wo) * f.px1 + 2 * j % x.Wo) / 2 : 0);
  for (int j = tid; j < st2 * 8; j += NT) pw2[j] = (unsigned short)(2 * j < pix2 ? ((2 * j / y.Wo) * f.px2 + 2 * j % y.Wo) / 2 : 0);
  int o1[MT1][2], o2[MT2][2];
#pragma unroll
  for (int m = 0; m < MT1; ++m)
#pragma unroll
    for (int h = 0; h < 2; ++h) o1[m][h] = tap_offset(16 * m + g + 8 * h, K1, k, x.Ci, f.px1, f.plane1);
#pragma unroll
  for (int m = 0; m < MT2; ++m)
#pragma unroll
    for (int h = 0; h < 2; ++h) o2[m][h] = tap_offset(16 * (warp + NWARP * m) + g + 8 * h, K2, k, y.Ci, f.px2, f.plane2);
  float c1[MT1][4], c2[MT2][2][4];
#pragma unroll
  for (int m = 0; m < MT1; ++m)
#pragma unroll
    for (int i = 0; i < 4; ++i) c1[m][i] = 0.f;
#pragma unroll
  for (int m = 0; m < MT2; ++m)
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) c2[m][n][i] = 0.f;
  constexpr uint32_t ONES = 0x3f803f80u;

  for (int j = 0; j < FR; ++j) {
    if (s[j] < 0) continue;                           // padding row (same decision in every thread)
    const int r = r0 + j;
    __syncthreads();                                  // the previous row's maps are no longer read
    // ---- maps of the row; empty delta maps
    load_planar(im, a.X + (size_t)s[j] * n_in, x.Hi, x.Wi, x.Ci, f.px1, f.plane1);
    load_planar(in2, a.pool1 + (size_t)r * n1, y.Hi, y.Wi, y.Ci, f.px2, f.plane2);
    for (int i = tid; i < n1; i += NT) arg1[i] = a.arg1[(size_t)r * n1 + i];
    for (int i = tid; i < (f.a1 - f.dz1) / 16; i += NT) reinterpret_cast<uint4*>(cs + f.dz1)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    // ---- shifted copies; the features' delta at the window positions that supplied the maxima
    shift_copy(im + x.Ci * f.plane1, im, x.Ci * f.plane1);
    shift_copy(in2 + y.Ci * f.plane2, in2, y.Ci * f.plane2);
    for (int e = tid; e < n2; e += NT) {
      const int co = e % y.Co, q = e / y.Co, px = q % y.Pw, py = q / y.Pw;
      const int w = a.arg2[(size_t)r * n2 + e], oy = 2 * py + (w >> 1), ox = 2 * px + (w & 1);
      const bf16 d = a.dfeat[(size_t)r * n2 + e];
      reinterpret_cast<bf16*>(dz2 + co * f.pz2)[oy * y.Wo + ox] = d;
      dzb[((oy + k - 1) * f.zw + ox + k - 1) * 24 + co] = d;
    }
    __syncthreads();
    // ---- delta of the second block's input, 16 pixels per task, scattered to the first block's window positions
    const int n_px = y.Hi * y.Wi;
    for (int p0 = warp * 16; p0 < n_px; p0 += NWARP * 16) {
      const int p = min(p0 + (lane & 15), n_px - 1), yy = p / y.Wi, xx = p - yy * y.Wi;
      const uint32_t base = outl::s_u32(dzb + ((yy + k - 1) * f.zw + xx + k - 1) * 24 + (lane >> 4) * 8);
      float d[4] = {0.f, 0.f, 0.f, 0.f};
      for (int dy = 0; dy < k; ++dy)
#pragma unroll 5
        for (int dx = 0; dx < k; ++dx) {
          uint32_t af[4];
          outl::ldsm4(base - (uint32_t)((dy * f.zw + dx) * 48), af);
          const uint2 b = bd[(dy * k + dx) * 32 + lane];
          outl::mma16816(d, af, b.x, b.y);
        }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int q = p0 + g + 8 * h;                 // pooled pixel of the first block
        if (q < n_px) {
          const int py = q / y.Wi, px = q - py * y.Wi;
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int c = 2 * t + i;
            if (c < y.Ci && __bfloat162float(in2[c * f.plane2 + py * f.px2 + px]) > 0.f) {
              const int w = arg1[q * y.Ci + c];
              reinterpret_cast<bf16*>(dz1 + c * f.pz1)[(2 * py + (w >> 1)) * x.Wo + 2 * px + (w & 1)] = __float2bfloat16_rn(d[2 * h + i]);
            }
          }
        }
      }
    }
    // ---- weight gradient of the second block: row tiles dealt to the warps
    {
      const uint32_t* iw = reinterpret_cast<const uint32_t*>(in2);
#pragma unroll 2
      for (int q = 0; q < st2; ++q) {
        const int u = pw2[8 * q + t], v = pw2[8 * q + t + 4];
        uint32_t b[2][2];
#pragma unroll
        for (int n = 0; n < 2; ++n) {
          b[n][0] = dz2[(8 * n + g) * f.pz2 + 8 * q + t];
          b[n][1] = dz2[(8 * n + g) * f.pz2 + 8 * q + t + 4];
        }
#pragma unroll
        for (int m = 0; m < MT2; ++m) {
          const int mt = warp + NWARP * m;
          if (mt < mt2) {
            uint32_t af[4] = {iw[o2[m][0] + u], iw[o2[m][1] + u], iw[o2[m][0] + v], iw[o2[m][1] + v]};
            if (16 * mt + g == K2) af[0] = af[2] = ONES;
            if (16 * mt + g + 8 == K2) af[1] = af[3] = ONES;
            outl::mma16816(c2[m][0], af, b[0][0], b[0][1]);
            if (nc2 > 1) outl::mma16816(c2[m][1], af, b[1][0], b[1][1]);
          }
        }
      }
    }
    __syncthreads();
    // ---- weight gradient of the first block: pixels dealt to the warps, all row tiles per warp
    {
      const uint32_t* iw = reinterpret_cast<const uint32_t*>(im);
      for (int q = warp; q < st1; q += NWARP) {
        const int u = pw1[8 * q + t], v = pw1[8 * q + t + 4];
        const uint32_t b0 = dz1[g * f.pz1 + 8 * q + t], b1 = dz1[g * f.pz1 + 8 * q + t + 4];
#pragma unroll
        for (int m = 0; m < MT1; ++m)
          if (m < mt1) {
            uint32_t af[4] = {iw[o1[m][0] + u], iw[o1[m][1] + u], iw[o1[m][0] + v], iw[o1[m][1] + v]};
            if (16 * m + g == K1) af[0] = af[2] = ONES;
            if (16 * m + g + 8 == K1) af[1] = af[3] = ONES;
            outl::mma16816(c1[m], af, b0, b1);
          }
      }
    }
  }
  // ---- this CTA's sums (row K of the product is the bias)
  {
    float* dst = a.part[1] + (size_t)blockIdx.x * (size_t)(K2 + 1) * y.Co;
#pragma unroll
    for (int m = 0; m < MT2; ++m)
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int row = 16 * (warp + NWARP * m) + g + 8 * (i >> 1), co = 8 * n + 2 * t + (i & 1);
          if (row <= K2 && co < y.Co) dst[row * y.Co + co] = c2[m][n][i];
        }
  }
  __syncthreads();
  float* red = reinterpret_cast<float*>(cs);          // [warp][MT1 * 16][8]
#pragma unroll
  for (int m = 0; m < MT1; ++m)
#pragma unroll
    for (int i = 0; i < 4; ++i) red[(warp * MT1 * 16 + 16 * m + g + 8 * (i >> 1)) * 8 + 2 * t + (i & 1)] = c1[m][i];
  __syncthreads();
  float* dst = a.part[0] + (size_t)blockIdx.x * (size_t)(K1 + 1) * x.Co;
  for (int e = tid; e < (K1 + 1) * 8; e += NT) {
    const int row = e >> 3, co = e & 7;
    if (co >= x.Co) continue;
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < NWARP; ++w) tot += red[(w * MT1 * 16 + row) * 8 + co];
    dst[row * x.Co + co] = tot;
  }
}

}  // namespace cmma
}  // namespace absb
