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
// The weights of every model version are also kept in the order of the products' column operands ("fragments"), written
// beside the ring by the Eq. 3 kernel, so that a CTA copies them instead of gathering 2-byte elements.
// FP32-FMA kernels with one CTA per row spent 315 us of a 640-row round of the 32 x 32 x 3 network here (5 % of the
// FMA peak, bound by shared-memory reads per FMA).  These: 16 us forward, 37 us backward; bound by the shared-memory bytes
// of the operand fragments (7000 shared-memory wavefronts per row backward) and the latency of their chains.
#pragma once
#include "common.cuh"
#include "outlayer.cuh"

namespace absb {
namespace cmma {

typedef __nv_bfloat16 bf16;
constexpr int NT = 256, NWARP = NT / 32;
constexpr int FR = 2;                    // gradient rows per CTA (divides the row padding unit)
constexpr int MT1 = 5;                   // most 16-row tiles of the first block's weight gradient (per warp)
constexpr int MT2 = 2;                   // ... of the second block's (16 tiles over 8 warps)

struct Block { int Hi, Wi, Ci, Ho, Wo, Ph, Pw, Co; size_t w_off; };
struct FwdLayout { int e1, o1, e2, o2, a1, f2, a2, row, b1, bias, total; };
struct BwdLayout {
  int im, in2, dz1, dz2, dzb, raw, raw2, a1, bd, pw, total;
  int px1, px2, plane1, plane2, copy1, copy2, pz1, pz2, zw, n_pw1, n_pw2;
};
struct Args {
  DevState* st;
  RoundInfo* ri;
  const int* tile_slot;
  const int* row_idx;
  const void* ring; size_t slot_stride;
  const bf16* frag; size_t frag_stride;  // [S+1][frag_stride] weights as column operands (see FragMap)
  int k, rb_shift;                       // rows per tile_slot entry = 1 << rb_shift
  Block b[2];
  const bf16* X;                         // dataset images
  bf16* pool1; unsigned char* arg1;      // [rows][Ph1][Pw1][C1] pooled maps of the first block, position of each maximum
  bf16* feat; unsigned char* arg2;       // [rows][Ph2][Pw2][C2] the same of the second block: the features
  const bf16* dfeat;                     // [rows][...] delta of the features (zero where the feature is not positive)
  float* part[2];                        // [chunks of FR rows][k k Ci Co + Co] sums of the weight and bias gradient
  // everything that follows from the shapes, worked out once by the host (in the kernels it was a third of all
  // instructions)
  FwdLayout fl;
  BwdLayout bl;
  int frag1, frag2;                      // elements of the first / second block's forward fragments
  FastDiv by_gr[2], by_pw[2], by_co2, by_wi2, by_wpr[2];
  const int* taps;                       // tables of the backward kernel, see table_words
};

__host__ __device__ inline int even(int n) { return (n + 1) & ~1; }

// ---- fragments of one model version: [first block forward | second block forward | second block for the input delta],
// each a list of 32-lane uint2 fragments {rows 2t, 2t+1 | rows 2t+8, 2t+9} of 16 x 8 operand tiles, zero-padded.
__host__ __device__ inline int frag_fwd(int k, const Block& b) { return k * ((k * b.Ci + 15) / 16) * ((b.Co + 7) / 8) * 128; }
__host__ __device__ inline int frag_delta(int k) { return k * k * 128; }
__host__ __device__ inline int frag_total(int k, const Block& x, const Block& y) { return frag_fwd(k, x) + frag_fwd(k, y) + frag_delta(k); }
struct FragMap { bf16* frag; size_t stride; int k; Block b[2]; };      // frag null: not kept
// element (row r, column c) of an operand tile
__device__ __forceinline__ int frag_at(int tile, int r, int c) { return ((tile * 32 + c * 4 + ((r & 7) >> 1)) * 2 + (r >> 3)) * 2 + (r & 1); }
// parameter j of block i (W[dy][dx][ci][co], then the bias, which has no place here) of the version in `slot`
__device__ __forceinline__ void frag_store(const FragMap& m, int slot, int i, int j, bf16 v) {
  const Block& b = m.b[i];
  const int co = j % b.Co, row = j / b.Co, ci = row % b.Ci, tap = row / b.Ci, dx = tap % m.k, dy = tap / m.k;
  if (dy >= m.k) return;
  bf16* f = m.frag + (size_t)slot * m.stride;
  const int kk = dx * b.Ci + ci, ks = (m.k * b.Ci + 15) / 16, nc = (b.Co + 7) / 8;
  f[(i ? frag_fwd(m.k, m.b[0]) : 0) + frag_at((dy * ks + kk / 16) * nc + co / 8, kk % 16, co % 8)] = v;
  if (i == 1) f[frag_fwd(m.k, m.b[0]) + frag_fwd(m.k, b) + frag_at(tap, co, ci)] = v;
}
// fragments of the model versions in slots 0 .. gridDim.y - 1 of the ring
static __global__ void frag_fill_kernel(FragMap m, const bf16* ring, size_t slot_stride) {
  const int slot = blockIdx.y;
  for (int i = 0; i < 2; ++i) {
    const int len = m.k * m.k * m.b[i].Ci * m.b[i].Co;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < len; j += gridDim.x * blockDim.x)
      frag_store(m, slot, i, j, ring[(size_t)slot * slot_stride + m.b[i].w_off + j]);
  }
}

// ---- shared-memory layouts (byte offsets)
inline FwdLayout fwd_layout(int k, const Block& x, const Block& y) {
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
  f.b1 = take(2 * (frag_fwd(k, x) + frag_fwd(k, y)));
  f.bias = take(4 * (8 + 16 + 8));
  f.total = off;
  return f;
}
// words between the channels of a dense delta map: 4 mod 8, so that 8 channels x 4 lanes hit 32 different banks
inline int dz_pitch(int pixels) { return round_up(round_up(pixels, 16) / 2, 8) + 4; }
inline BwdLayout bwd_layout(int k, const Block& x, const Block& y) {
  BwdLayout f;
  int off = 0;
  auto take = [&](int bytes) { const int o = off; off += round_up(bytes, 16); return o; };
  f.px1 = even(x.Wi); f.px2 = even(y.Wi);
  // elements between channels / between the two copies: 12 and 8 words mod 32, so that most of the eight taps x channels
  // a fragment reads at once start in different groups of four banks
  auto pad = [](int words, int want) { return 2 * (words + ((want - words % 32) + 32) % 32); };
  f.plane1 = pad(x.Hi * f.px1 / 2, 12); f.plane2 = pad(y.Hi * f.px2 / 2, 12);
  f.copy1 = pad(x.Ci * f.plane1 / 2, 8); f.copy2 = pad(y.Ci * f.plane2 / 2, 8);
  f.pz1 = dz_pitch(x.Ho * x.Wo); f.pz2 = dz_pitch(y.Ho * y.Wo);
  f.zw = y.Wo + 2 * (k - 1);
  f.im = take(2 * 2 * f.copy1);                        // two copies, the second shifted by one element
  f.in2 = take(2 * 2 * f.copy2);
  f.dz1 = take(4 * 8 * f.pz1);
  f.dz2 = take(4 * 16 * f.pz2);
  f.dzb = take(2 * 24 * (y.Ho + 2 * (k - 1)) * f.zw);
  f.raw = take(2 * x.Hi * x.Wi * x.Ci + 16);           // the next row's maps as stored
  f.raw2 = take(2 * y.Hi * y.Wi * y.Ci + 16);
  f.a1 = take(x.Ph * x.Pw * x.Co);
  f.bd = take(2 * frag_delta(k));
  f.n_pw1 = round_up(x.Ho * x.Wo, 16) / 2;
  f.n_pw2 = round_up(y.Ho * y.Wo, 16) / 2;
  f.pw = take(4 * (f.n_pw1 + f.n_pw2));
  f.total = off;
  const int red = 4 * NWARP * (MT1 * 16 + 1) * 8;            // the first block's sums of the warps, over the maps at the end
  if (f.total < red) f.total = red;
  return f;
}
// Tables of the backward kernel (bytes into the maps): [MT1 * 16] taps of the first block, [MT2 * 8 * 16] of the second,
// then the offset of every pixel pair of the first and of the second block (padded to whole steps of 16 pixels).
inline int table_words(const BwdLayout& f) { return 16 * MT1 + 16 * MT2 * NWARP + f.n_pw1 + f.n_pw2; }
inline void fill_tables(int* tab, int k, const Block& x, const Block& y, const BwdLayout& f) {
  auto taps = [&](int* t, int n, int Ci, int px, int plane, int copy) {
    for (int m = 0; m < n; ++m) {
      const int ci = m % Ci, tap = m / Ci, dx = tap % k, dy = tap / k;
      t[m] = dy < k ? 2 * ((dx & 1) * copy + ci * plane + dy * px + dx - (dx & 1)) : 0;     // padding rows: any finite value
    }
  };
  auto pixels = [](int* t, int n, int pix, int Wo, int px) {
    for (int j = 0; j < n; ++j) t[j] = 2 * j < pix ? 2 * ((2 * j / Wo) * px + 2 * j % Wo) : 0;
  };
  taps(tab, 16 * MT1, x.Ci, f.px1, f.plane1, f.copy1);
  tab += 16 * MT1;
  taps(tab, 16 * MT2 * NWARP, y.Ci, f.px2, f.plane2, f.copy2);
  tab += 16 * MT2 * NWARP;
  pixels(tab, f.n_pw1, x.Ho * x.Wo, x.Wo, f.px1);
  pixels(tab + f.n_pw1, f.n_pw2, y.Ho * y.Wo, y.Wo, f.px2);
}
inline void fill_shapes(Args* a) {
  const Block &x = a->b[0], &y = a->b[1];
  a->fl = fwd_layout(a->k, x, y);
  a->bl = bwd_layout(a->k, x, y);
  a->frag1 = frag_fwd(a->k, x);
  a->frag2 = frag_fwd(a->k, y);
  for (int i = 0; i < 2; ++i) {
    const Block& b = a->b[i];
    a->by_gr[i] = FastDiv((b.Ph * b.Pw + 7) / 8);
    a->by_pw[i] = FastDiv(b.Pw);
    a->by_wpr[i] = FastDiv(even(b.Wi) / 2);
  }
  a->by_co2 = FastDiv(y.Co);
  a->by_wi2 = FastDiv(y.Wi);
}
// model classes these kernels take
inline bool fits(int k, const Block& x, const Block& y) {
  return x.Co <= 8 && y.Co <= 16 && k * k * x.Ci <= 16 * MT1 && k * k * y.Ci <= 16 * MT2 * NWARP &&
         fwd_layout(k, x, y).total <= 110 * 1024 && bwd_layout(k, x, y).total <= 110 * 1024;
}

__device__ __forceinline__ uint32_t join16(bf16 lo, bf16 hi) {
  return (uint32_t)*reinterpret_cast<unsigned short*>(&lo) | ((uint32_t)*reinterpret_cast<unsigned short*>(&hi) << 16);
}

// n bytes to shared memory (16-byte aligned destination), asynchronously where the source allows it
__device__ __forceinline__ void fetch(void* dst, const void* src, int n) {
  if ((((uintptr_t)src | (uintptr_t)n) & 15) == 0) {
    for (int i = threadIdx.x * 16; i < n; i += NT * 16)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(outl::s_u32((char*)dst + i)), "l"((const char*)src + i) : "memory");
  } else if ((((uintptr_t)src | (uintptr_t)n) & 3) == 0) {
    for (int i = threadIdx.x * 4; i < n; i += NT * 4)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(outl::s_u32((char*)dst + i)), "l"((const char*)src + i) : "memory");
  } else {
    for (int i = threadIdx.x; i < n; i += NT) ((char*)dst)[i] = ((const char*)src)[i];
  }
}
__device__ __forceinline__ void fetch_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// G tasks of a forward block side by side (independent accumulators hide the latencies): 8 pooled pixels each, all
// channels; results to `out` (pitch: elements between pooled rows) and `arg` ([pixel][Co]).
struct FwdTask { const bf16 *E, *O; bf16* out; unsigned char* arg; int q0; };
template <int K, int NC, int G>
__device__ __forceinline__ void forward_tasks(const Block& b, int k_, const FwdTask (&task)[G], const uint2* bf, const float* bias,
                                              int pitch, const FastDiv& by_pw, int lane) {
  const int k = K ? K : k_;
  const int g = lane >> 2, t = lane & 3;
  const int P = even(b.Wi * b.Ci), ks = (k * b.Ci + 15) / 16, n_q = b.Ph * b.Pw;
  const uint32_t *p0[G], *p1[G];
  int py[G], px[G];
  float acc[G][2][NC][4];
#pragma unroll
  for (int u = 0; u < G; ++u) {
    const int q = min(task[u].q0 + g, n_q - 1);
    py[u] = by_pw.div(q);
    px[u] = q - py[u] * b.Pw;
    const int at = 2 * py[u] * P + 2 * px[u] * b.Ci;  // even
    p0[u] = reinterpret_cast<const uint32_t*>(task[u].E + at) + t;
    p1[u] = reinterpret_cast<const uint32_t*>((b.Ci & 1) ? task[u].O + at + b.Ci - 1 : task[u].E + at + b.Ci) + t;
#pragma unroll
    for (int w = 0; w < 2; ++w)
#pragma unroll
      for (int n = 0; n < NC; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[u][w][n][i] = 0.f;
  }
  const uint2* bl = bf + lane;
  for (int s = 0; s < ks; ++s) {
#pragma unroll
    for (int i = 0; i <= k; ++i) {
      const int o = (i * P) / 2 + 8 * s;
      uint32_t a[G][4];
#pragma unroll
      for (int u = 0; u < G; ++u) { a[u][0] = p0[u][o]; a[u][1] = p1[u][o]; a[u][2] = p0[u][o + 4]; a[u][3] = p1[u][o + 4]; }
#pragma unroll
      for (int n = 0; n < NC; ++n) {
        if (i < k) {
          const uint2 w = bl[((i * ks + s) * NC + n) * 32];
#pragma unroll
          for (int u = 0; u < G; ++u) outl::mma16816_rn(acc[u][0][n], a[u], w.x, w.y);
        }
        if (i > 0) {
          const uint2 w = bl[(((i - 1) * ks + s) * NC + n) * 32];
#pragma unroll
          for (int u = 0; u < G; ++u) outl::mma16816_rn(acc[u][1][n], a[u], w.x, w.y);
        }
      }
    }
  }
#pragma unroll
  for (int u = 0; u < G; ++u) {
    const int q = task[u].q0 + g;
    if (q >= n_q) continue;
#pragma unroll
    for (int n = 0; n < NC; ++n)
{
      const int c = 8 * n + 2 * t;
      if (c < b.Co) {
        // the window's stored values (ReLU, rounded; row-major order) of channels c and c + 1: bf16 patterns of
        // non-negative numbers order like integers, and 3 - position below them makes the first maximum win a tie
        const float b0 = bias[c], b1 = bias[c + 1];
        uint32_t lo = 0u, hi = 0u;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          const float* v = &acc[u][w >> 1][n][2 * (w & 1)];
          uint32_t pk;
          asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(pk) : "f"(v[1] + b1), "f"(v[0] + b0));
          lo = max(lo, (pk << 16) | (uint32_t)(3 - w));
          hi = max(hi, (pk & 0xffff0000u) | (uint32_t)(3 - w));
        }
        unsigned short* o = reinterpret_cast<unsigned short*>(task[u].out) + py[u] * pitch + px[u] * b.Co + c;
        unsigned char* ar = task[u].arg + q * b.Co + c;
        o[0] = (unsigned short)(lo >> 16);
        ar[0] = (unsigned char)(3u - (lo & 3u));
        if (c + 1 < b.Co) {
          o[1] = (unsigned short)(hi >> 16);
          ar[1] = (unsigned char)(3u - (hi & 3u));
        }
      }
    }
  }
}
// all tasks of a block for the CTA's rows
template <int K, int NC, int G, class F>
__device__ __forceinline__ void forward_block(const Block& b, int k, const FastDiv& by_gr, const FastDiv& by_pw, const uint2* bf,
                                              const float* bias, int pitch, int warp, int lane, F make) {
  const int gr = (b.Ph * b.Pw + 7) / 8, n = FR * gr;
  for (int t0 = warp; t0 < n; t0 += NWARP * G) {
    FwdTask task[G];
#pragma unroll
    for (int u = 0; u < G; ++u) {                     // (a task too many repeats the last one)
      const int q = min(t0 + u * NWARP, n - 1), j = by_gr.div(q);
      task[u] = make(j);
      task[u].q0 = (q - j * gr) * 8;
    }
    forward_tasks<K, NC, G>(b, k, task, bf, bias, pitch, by_pw, lane);
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

template <int K>
__global__ void __launch_bounds__(NT) conv_fwd_mma_kernel(const __grid_constant__ Args a) {
  grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char cs[];
  const int r0 = (int)blockIdx.x * FR;
  const int status = a.st->status, n_rows = a.ri->n_rows, slot = a.tile_slot[r0 >> a.rb_shift];
  int s[FR];
  bool any = false;
#pragma unroll
  for (int j = 0; j < FR; ++j) s[j] = a.row_idx[r0 + j];
  if (status != ST_OK || r0 >= n_rows) return;
#pragma unroll
  for (int j = 0; j < FR; ++j) any |= s[j] >= 0;
  if (!any) return;                                   // padding rows: nothing reads more than finite values of them
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = K ? K : a.k;
  const FwdLayout& f = a.fl;
  const Block &x = a.b[0], &y = a.b[1];
  const bf16* ring = (const bf16*)a.ring + (size_t)slot * a.slot_stride;
  const int n_in = x.Hi * x.Wi * x.Ci, P1 = even(x.Wi * x.Ci), P2 = even(y.Wi * y.Ci);
  const int n1 = x.Ph * x.Pw * x.Co, n2 = y.Ph * y.Pw * y.Co;
  auto map = [&](int j, int off) { return reinterpret_cast<bf16*>(cs + (size_t)j * f.row + off); };
  // ---- images, weights
  const bf16* frag = a.frag + (size_t)slot * a.frag_stride;
  uint2* b1 = reinterpret_cast<uint2*>(cs + f.b1);
  uint2* b2 = b1 + a.frag1 / 4;
  fetch(b1, frag, 2 * (a.frag1 + a.frag2));
#pragma unroll
  for (int j = 0; j < FR; ++j) {
    bf16* E = map(j, f.e1);
    const bf16* src = a.X + (size_t)max(s[j], 0) * n_in;
    if (P1 == x.Wi * x.Ci) {
      fetch(E, src, 2 * n_in);
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
  float* bias = reinterpret_cast<float*>(cs + f.bias);
  if (tid < 8) bias[tid] = tid < x.Co ? __bfloat162float(ring[x.w_off + (size_t)k * k * x.Ci * x.Co + tid]) : 0.f;
  else if (tid < 24) bias[tid] = tid - 8 < y.Co ? __bfloat162float(ring[y.w_off + (size_t)k * k * y.Ci * y.Co + tid - 8]) : 0.f;
  fetch_wait();
  __syncthreads();
  if (x.Ci & 1) {
#pragma unroll
    for (int j = 0; j < FR; ++j) shift_copy(map(j, f.o1), map(j, f.e1), x.Hi * P1 + 62);
    __syncthreads();
  }
  // ---- first block
  forward_block<K, 1, 2>(x, k, a.by_gr[0], a.by_pw[0], b1, bias, P2, warp, lane,
                         [&](int j) { return FwdTask{map(j, f.e1), map(j, f.o1), map(j, f.e2), cs + (size_t)j * f.row + f.a1, 0}; });
  __syncthreads();
  if (y.Ci & 1) {
#pragma unroll
    for (int j = 0; j < FR; ++j) shift_copy(map(j, f.o2), map(j, f.e2), y.Hi * P2 + 62);
    __syncthreads();
  }
  // ---- second block; the first one's results leave meanwhile
  auto second = [&](int j) { return FwdTask{map(j, f.e2), map(j, f.o2), map(j, f.f2), cs + (size_t)j * f.row + f.a2, 0}; };
  if (nc2 == 1) forward_block<K, 1, 1>(y, k, a.by_gr[1], a.by_pw[1], b2, bias + 8, y.Pw * y.Co, warp, lane, second);
  else forward_block<K, 2, 1>(y, k, a.by_gr[1], a.by_pw[1], b2, bias + 8, y.Pw * y.Co, warp, lane, second);
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

// [y][x][c] map in shared memory -> the two [c][y][x] copies (pitch px)
__device__ __forceinline__ void make_planar(bf16* dst, const bf16* src, int Hi, int Wi, int Ci, int px, int plane, int copy, const FastDiv& by_wpr) {
  const int wpr = px / 2;
  for (int w = threadIdx.x; w < Hi * wpr; w += NT) {
    const int yy = by_wpr.div(w), xx = 2 * (w - yy * wpr);
    const bf16* p = src + (yy * Wi + xx) * Ci;
    const bool has1 = xx + 1 < Wi, has2 = xx + 2 < Wi;
    uint32_t* d = reinterpret_cast<uint32_t*>(dst) + w;
    for (int c = 0; c < Ci; ++c) {
      const bf16 e0 = p[c], e1 = has1 ? p[Ci + c] : (bf16)0.f, e2 = has2 ? p[2 * Ci + c] : (bf16)0.f;
      d[c * plane / 2] = join16(e0, e1);
      d[copy / 2 + c * plane / 2] = join16(e1, e2);
    }
  }
}
template <int K>
__global__ void __launch_bounds__(NT, 3) conv_bwd_mma_kernel(const __grid_constant__ Args a) {
  grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char cs[];
  const int r0 = (int)blockIdx.x * FR;
  const int status = a.st->status, n_rows = a.ri->n_rows, slot = a.tile_slot[r0 >> a.rb_shift];
  int s[FR];
#pragma unroll
  for (int j = 0; j < FR; ++j) s[j] = a.row_idx[r0 + j];
  if (status != ST_OK || r0 >= n_rows) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = K ? K : a.k;
  const int g = lane >> 2, t = lane & 3;
  const BwdLayout& f = a.bl;
  const Block &x = a.b[0], &y = a.b[1];
  bf16* im = reinterpret_cast<bf16*>(cs + f.im);
  bf16* in2 = reinterpret_cast<bf16*>(cs + f.in2);
  uint32_t* dz1 = reinterpret_cast<uint32_t*>(cs + f.dz1);
  uint32_t* dz2 = reinterpret_cast<uint32_t*>(cs + f.dz2);
  bf16* dzb = reinterpret_cast<bf16*>(cs + f.dzb);
  unsigned char* arg1 = cs + f.a1;
  uint2* bd = reinterpret_cast<uint2*>(cs + f.bd);
  const int* pw1 = reinterpret_cast<const int*>(cs + f.pw);
  const int* pw2 = pw1 + f.n_pw1;
  const int n1 = x.Ph * x.Pw * x.Co, n2 = y.Ph * y.Pw * y.Co, n_in = x.Hi * x.Wi * x.Ci;
  const int st1 = f.n_pw1 / 8, st2 = f.n_pw2 / 8;
  const int K1 = k * k * x.Ci, K2 = k * k * y.Ci;
  const int mt1 = (K1 + 15) / 16, mt2 = (K2 + 15) / 16;
  const int nc2 = (y.Co + 7) / 8;
  // ---- once per CTA: weights of the second block as column operand of the delta product, pixel tables, tap offsets
  fetch(bd, a.frag + (size_t)slot * a.frag_stride + a.frag1 + a.frag2, 2 * frag_delta(k));
  fetch(cs + f.pw, a.taps + 16 * MT1 + 16 * MT2 * NWARP, 4 * (f.n_pw1 + f.n_pw2));
  // a row's maps as stored (the next row's while this one is worked on)
  auto fetch_maps = [&](int j) {
    if (j >= FR || s[j] < 0) return;
    fetch(cs + f.raw, a.X + (size_t)s[j] * n_in, 2 * n_in);
    fetch(cs + f.raw2, a.pool1 + (size_t)(r0 + j) * n1, 2 * n1);
  };
  fetch_maps(s[0] >= 0 ? 0 : 1);
  auto lds = [&](int off) { return *reinterpret_cast<const uint32_t*>(cs + off); };
  int o1[MT1][2], o2[MT2][2];                         // offsets of this thread's taps
#pragma unroll
  for (int m = 0; m < MT1; ++m)
#pragma unroll
    for (int h = 0; h < 2; ++h) o1[m][h] = f.im + a.taps[16 * m + g + 8 * h];
#pragma unroll
  for (int m = 0; m < MT2; ++m)
#pragma unroll
    for (int h = 0; h < 2; ++h) o2[m][h] = f.in2 + a.taps[16 * MT1 + 16 * (warp + NWARP * m) + g + 8 * h];
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
  const uint32_t ones[4] = {0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u};
  float s1[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f};     // bias sums: products with ones (every row the same)

  for (int j = 0; j < FR; ++j) {
    if (s[j] < 0) continue;                           // padding row (same decision in every thread)
    const int r = r0 + j;
    __syncthreads();                                  // the previous row's maps are no longer read
    // ---- maps of the row; empty delta maps
    fetch_wait();
    for (int i = tid; i < n1; i += NT) arg1[i] = a.arg1[(size_t)r * n1 + i];
    for (int i = tid; i < (f.raw - f.dz1) / 16; i += NT) reinterpret_cast<uint4*>(cs + f.dz1)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    make_planar(im, reinterpret_cast<const bf16*>(cs + f.raw), x.Hi, x.Wi, x.Ci, f.px1, f.plane1, f.copy1, a.by_wpr[0]);
    make_planar(in2, reinterpret_cast<const bf16*>(cs + f.raw2), y.Hi, y.Wi, y.Ci, f.px2, f.plane2, f.copy2, a.by_wpr[1]);
    // the features' delta at the window positions that supplied the maxima
    {
      for (int e = tid; e < n2; e += NT) {
        const int w = a.arg2[(size_t)r * n2 + e];
        const bf16 d = a.dfeat[(size_t)r * n2 + e];
        const int q = a.by_co2.div(e), co = e - q * y.Co, py = a.by_pw[1].div(q), px = q - py * y.Pw;
        const int oy = 2 * py + (w >> 1), ox = 2 * px + (w & 1);
        reinterpret_cast<bf16*>(dz2 + co * f.pz2)[oy * y.Wo + ox] = d;
        dzb[((oy + k - 1) * f.zw + ox + k - 1) * 24 + co] = d;
      }
    }
    __syncthreads();
    fetch_maps(j + 1);
    // ---- delta of the second block's input, 16 pixels per task, scattered to the first block's window positions
    const int n_px = y.Hi * y.Wi;
    for (int p0 = warp * 16; p0 < n_px; p0 += NWARP * 16) {
      const int p = min(p0 + (lane & 15), n_px - 1), yy = a.by_wi2.div(p), xx = p - yy * y.Wi;
      const uint32_t base = outl::s_u32(dzb + ((yy + k - 1) * f.zw + xx + k - 1) * 24 + (lane >> 4) * 8);
      float d[4] = {0.f, 0.f, 0.f, 0.f}, d2[4] = {0.f, 0.f, 0.f, 0.f};      // even / odd dx: two shorter chains
      for (int dy = 0; dy < k; ++dy) {
        if (K) {                                      // all operands of a kernel row first, then its products
          uint32_t af[K ? K : 1][4];
          uint2 b[K ? K : 1];
#pragma unroll
          for (int dx = 0; dx < K; ++dx) {
            outl::ldsm4(base - (uint32_t)((dy * f.zw + dx) * 48), af[dx]);
            b[dx] = bd[(dy * k + dx) * 32 + lane];
          }
#pragma unroll
          for (int dx = 0; dx < K; ++dx) {
            if (dx & 1) outl::mma16816_rn(d2, af[dx], b[dx].x, b[dx].y);
            else outl::mma16816_rn(d, af[dx], b[dx].x, b[dx].y);
          }
        } else {
          for (int dx = 0; dx < k; ++dx) {
            uint32_t af[4];
            outl::ldsm4(base - (uint32_t)((dy * f.zw + dx) * 48), af);
            const uint2 b = bd[(dy * k + dx) * 32 + lane];
            outl::mma16816_rn(d, af, b.x, b.y);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) d[i] += d2[i];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int q = p0 + g + 8 * h;                 // pooled pixel of the first block
        if (q < n_px) {
          const int py = a.by_wi2.div(q), px = q - py * y.Wi;
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
      for (int m = 0; m < MT2; ++m)
        if (warp + NWARP * m < mt2) {
          const uint32_t af[4] = {lds(o2[m][0] + u), lds(o2[m][1] + u), lds(o2[m][0] + v), lds(o2[m][1] + v)};
          outl::mma16816_rn(c2[m][0], af, b[0][0], b[0][1]);
          if (nc2 > 1) outl::mma16816_rn(c2[m][1], af, b[1][0], b[1][1]);
        }
      if (warp < nc2) {
        if (warp == 0) outl::mma16816_rn(s2, ones, b[0][0], b[0][1]);
        else outl::mma16816_rn(s2, ones, b[1][0], b[1][1]);
      }
    }
    __syncthreads();
    // ---- weight gradient of the first block: pixels dealt to the warps, all row tiles per warp
    for (int q = warp; q < st1; q += NWARP) {
      const int u = pw1[8 * q + t], v = pw1[8 * q + t + 4];
      const uint32_t b0 = dz1[g * f.pz1 + 8 * q + t], b1 = dz1[g * f.pz1 + 8 * q + t + 4];
#pragma unroll
      for (int m = 0; m < MT1; ++m)
        if (m < mt1) {
          const uint32_t af[4] = {lds(o1[m][0] + u), lds(o1[m][1] + u), lds(o1[m][0] + v), lds(o1[m][1] + v)};
          outl::mma16816_rn(c1[m], af, b0, b1);
        }
      outl::mma16816_rn(s1, ones, b0, b1);
    }
  }
  // ---- this CTA's sums: [k k Ci][Co], then the bias
  {
    float* dst = a.part[1] + (size_t)blockIdx.x * (size_t)(K2 + 1) * y.Co;
#pragma unroll
    for (int m = 0; m < MT2; ++m)
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int row = 16 * (warp + NWARP * m) + g + 8 * (i >> 1), co = 8 * n + 2 * t + (i & 1);
          if (row < K2 && co < y.Co) dst[row * y.Co + co] = c2[m][n][i];
        }
    if (warp < nc2 && g == 0)
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (8 * warp + 2 * t + i < y.Co) dst[K2 * y.Co + 8 * warp + 2 * t + i] = s2[i];
  }
  // a CTA whose rows are all padding has not waited for its copies yet: they must not land on the sums below
  fetch_wait();
  __syncthreads();
  constexpr int RW = (16 * MT1 + 1) * 8;              // floats per warp: [rows and bias][8 channels]
  float* red = reinterpret_cast<float*>(cs);
#pragma unroll
  for (int m = 0; m < MT1; ++m)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      *reinterpret_cast<float2*>(red + warp * RW + (16 * m + g + 8 * h) * 8 + 2 * t) = make_float2(c1[m][2 * h], c1[m][2 * h + 1]);
  if (g == 0) *reinterpret_cast<float2*>(red + warp * RW + 16 * MT1 * 8 + 2 * t) = make_float2(s1[0], s1[1]);
  __syncthreads();
  float* dst = a.part[0] + (size_t)blockIdx.x * (size_t)(K1 + 1) * x.Co;
  for (int e = tid; e < (K1 + 1) * 8; e += NT) {
    const int row = e >> 3, co = e & 7;
    if (co >= x.Co) continue;
    const float* p = red + (row < K1 ? row : 16 * MT1) * 8 + co;
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < NWARP; ++w) tot += p[w * RW];
    dst[row * x.Co + co] = tot;
  }
}

}  // namespace cmma
}  // namespace absb
