// The narrow output layer of a bf16 network in one pass over 64 gradient rows per CTA, with its
// three small contractions on the warp-level tensor-core instruction (mma.sync m16n8k16, bf16
// operands, fp32 accumulation):
//   logits  Z[r][c]   = sum_m H[r][m] W_s[m][c] + b_s[c]       soft-max cross-entropy loss and
//                                                              delta D = softmax(Z) - onehot(y)
//   weights G[m][c]   = sum_r H[r][m] D[r][c]  (+ bias row)    this CTA's share, Eq. 3 adds them up
//   below   Dl[r][m]  = (sum_c D[r][c] W_s[m][c]) [H[r][m] > 0]
// (Eq. 2 with U = 1 for the rows' model version s; D is rounded to bf16 like every stored delta.)
// The 64 input rows stay in shared memory for all three; the class count is padded to 16 with
// zero weights.  The work per CTA is a few hundred tensor-core instructions, so the kernel is
// bound by the round trip of its loads and stores: one wave of CTAs, every phase short.
#pragma once
#include "common.cuh"
#include "narrow.cuh"

namespace absb {
namespace outl {

constexpr int ROWS = 64;          // gradient rows per CTA
constexpr int THREADS = 256;
constexpr int CP = 16;            // padded class count
constexpr int WP = 24;            // shared-memory pitch (elements) of the [.][16] class rows: 48 bytes,
                                  // which spreads eight consecutive rows over all banks

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
// d += a (16 x 16, row) * b (16 x 8, col), bf16 in, fp32 accumulate
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// d += a * b with the addition to d rounded to nearest: the instruction itself truncates where it adds to a large
// accumulator, and stored (rounded) activations turn such errors into flipped ReLU / max-pool decisions.  It also leaves
// consecutive products independent of one another.  Sums over many products use it (gradients, back-propagated deltas, bias
// sums): the additions hide behind the operand reads (CNN 75.9 -> 75.7 us a round, 785-513-511-10 bf16 291 -> 296).  One
// step of the 32 x 32 x 3 CNN against binary64 with the same storage rounding, mean of four inputs: 4.6e-4 on the first
// convolution's weights (FP32 FMAs 6.8e-4), 7e-5 on the first affine layer's (2.7e-4): what flipped decisions leave.  Its
// parameters after 200 rounds: 3.65e-4 from binary64 (FP32 FMAs 3.64e-4, truncating chains 4.77e-4; binary64 itself from
// weights perturbed by 1e-7: 5.2e-4).
__device__ __forceinline__ void mma16816_rn(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  float p[4];
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
               : "=f"(p[0]), "=f"(p[1]), "=f"(p[2]), "=f"(p[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
#pragma unroll
  for (int i = 0; i < 4; ++i) d[i] += p[i];
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

inline size_t smem_bytes(int in, int C) {
  return (size_t)ROWS * (in + 8) * 2 + (size_t)(in + 8) * WP * 2 + (size_t)ROWS * WP * 2 + (size_t)4 * 32 * 8 * 4 +
         ((size_t)(in + 1) * C * 2 + 15) / 16 * 16 + 64;
}

// NT = in / 128: feature tiles (16 wide) per warp of the weight-gradient phase.
// part[cta][(in + 1) * C]: this CTA's share of the layer's gradient block (row `in` = bias sums).
template <int NT>
__global__ void __launch_bounds__(THREADS) out_layer_mma_kernel(NarrowArgs a, float* part, int has_dgrad) {
  grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char osm_raw[];
  DevState* st = a.st;
  RoundInfo* ri = a.ri;
  const int r0 = blockIdx.x * ROWS;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;
  // one wave of loads (the grid covers the row capacity, so every address exists); warp (mt, kh) finishes the soft-max of
  // rows 16 mt + 8 kh + g
  const int status = st->status, n_rows = ri->n_rows, t_round = ri->t, slot = a.tile_slot[r0 >> a.tile_shift];
  const int my_row = 16 * (warp & 3) + 8 * (warp >> 2) + g;
  const int my_idx = a.row_idx[r0 + my_row];
  if (status != ST_OK || r0 >= n_rows) return;
  constexpr int IN = NT * 128;
  constexpr int HP = IN + 8;                    // row pitch of the input rows (elements): 16 bytes of padding
  const int C = a.C;
  __nv_bfloat16* hs = reinterpret_cast<__nv_bfloat16*>(osm_raw);          // [ROWS][HP] input rows, later Dl
  __nv_bfloat16* ws = hs + (size_t)ROWS * HP;                             // [IN + 1 (+7)][WP] weights, row IN = bias
  __nv_bfloat16* d3s = ws + (size_t)(IN + 8) * WP;                        // [ROWS][WP] deltas of this layer
  float* lp = reinterpret_cast<float*>(d3s + (size_t)ROWS * WP);          // [4][32][8] logit partial sums
  __nv_bfloat16* wraw = reinterpret_cast<__nv_bfloat16*>(lp + 4 * 32 * 8);  // [IN + 1][C] weights + bias as stored

  // ---- loads: the 64 input rows (asynchronous 16-byte copies), the weights of the rows' version
  const __nv_bfloat16* src = (const __nv_bfloat16*)a.act_in + (size_t)r0 * IN;
  for (int item = tid; item < ROWS * (IN / 8); item += THREADS) {
    const int rr = item / (IN / 8), v = item - rr * (IN / 8);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s_u32(hs + (size_t)rr * HP + v * 8)),
                 "l"(src + (size_t)rr * IN + v * 8) : "memory");
  }
  const int lab = my_idx < 0 ? -1 : a.labels[my_idx];
  const float sa = sa_slot_weight(a.sa, a.S, t_round, slot);     // staleness-aware step size: weight of these rows in Eq. 3
  const __nv_bfloat16* Wm = (const __nv_bfloat16*)a.ring + (size_t)slot * a.slot_stride + a.w_off;
  {
    // weights + bias are contiguous and start on a 128-byte boundary: whole 16-byte pieces
    const int n16 = (int)(((size_t)(IN + 1) * C * 2 + 15) / 16);
    for (int i = tid; i < n16; i += THREADS)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s_u32(wraw + 8 * i)), "l"(Wm + 8 * i) : "memory");
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  for (int k = tid; k <= IN; k += THREADS) {                // class rows padded to 16 with zeros
    const unsigned short* src_k = reinterpret_cast<const unsigned short*>(wraw) + k * C;
    uint32_t v[CP / 2];
#pragma unroll
    for (int c = 0; c < CP; c += 2)
      v[c / 2] = (c < C ? src_k[c] : 0u) | (c + 1 < C ? (uint32_t)src_k[c + 1] << 16 : 0u);
    uint4* dst_k = reinterpret_cast<uint4*>(ws + k * WP);
    dst_k[0] = make_uint4(v[0], v[1], v[2], v[3]);
    dst_k[1] = make_uint4(v[4], v[5], v[6], v[7]);
  }
  __syncthreads();

  // ---- logits: warp = (row tile mt, half of the features kh)
  {
    const int mt = warp & 3, kh = warp >> 2;
    float acc[2][4];
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[n][i] = 0.f;
    const uint32_t a_base = s_u32(hs + (size_t)(16 * mt + (lane & 15)) * HP + (lane >> 4) * 8);
    const uint32_t b_base = s_u32(ws + (size_t)((lane & 7) + ((lane >> 3) & 1) * 8) * WP + (lane >> 4) * 8);
#pragma unroll 4
    for (int k0 = kh * (IN / 2); k0 < (kh + 1) * (IN / 2); k0 += 16) {
      uint32_t af[4], bf[4];
      ldsm4(a_base + k0 * 2, af);
      ldsm4t(b_base + k0 * WP * 2, bf);
      mma16816(acc[0], af, bf[0], bf[1]);
      mma16816(acc[1], af, bf[2], bf[3]);
    }
    // the halves exchange partial sums: kh = 0 keeps row g of the tile, kh = 1 row g + 8; the sum is always formed as
    // (first half + second half) + bias
    {
      float* to = lp + (mt * 32 + lane) * 8 + 4 * kh;
      *reinterpret_cast<float4*>(to) = kh ? make_float4(acc[0][0], acc[0][1], acc[1][0], acc[1][1])
                                          : make_float4(acc[0][2], acc[0][3], acc[1][2], acc[1][3]);
    }
    __syncthreads();
    {
      // thread: row g + 8 kh of the tile, classes 2t, 2t+1, 8+2t, 8+2t+1
      const float4 o4 = *reinterpret_cast<const float4*>(lp + (mt * 32 + lane) * 8 + 4 * (1 - kh));
      const float other[4] = {o4.x, o4.y, o4.z, o4.w};
      float z[4];
      int cls[4];
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int c = 8 * n + 2 * t + j, e = 2 * n + j;
          const float mine = kh ? acc[n][2 + j] : acc[n][j];
          cls[e] = c;
          z[e] = (kh ? other[e] + mine : mine + other[e]) + __bfloat162float(ws[IN * WP + c]);
          z[e] = c < C ? z[e] : NO_CLASS;                   // padded classes: exp(NO_CLASS - max) = 0
        }
      float zmax = fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3]));
      zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, 1));
      zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, 2));
      float se = 0.f, zy = 0.f, e[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        e[i] = expf(z[i] - zmax);
        se += e[i];
        zy = cls[i] == lab ? z[i] : zy;
      }
      se += __shfl_xor_sync(0xffffffffu, se, 1);
      se += __shfl_xor_sync(0xffffffffu, se, 2);
      zy += __shfl_xor_sync(0xffffffffu, zy, 1);
      zy += __shfl_xor_sync(0xffffffffu, zy, 2);
      const float inv = 1.f / se;
      float d[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        d[i] = (lab >= 0 && cls[i] < C) ? (e[i] * inv - (cls[i] == lab ? 1.f : 0.f)) * sa : 0.f;   // padding rows add nothing to Eq. 3
      *reinterpret_cast<uint32_t*>(d3s + my_row * WP + 2 * t) = pack_bf16(d[0], d[1]);
      *reinterpret_cast<uint32_t*>(d3s + my_row * WP + 8 + 2 * t) = pack_bf16(d[2], d[3]);
      if (t == 0) {
        const float loss = lab >= 0 ? logf(se) - (zy - zmax) : 0.f;
        a.row_loss[r0 + my_row] = loss;
        if (!isfinite(loss)) ri->diverged = 1;
      }
    }
    __syncthreads();
  }

  // ---- this CTA's share of the weight and bias gradient: warp w owns feature tiles w, w + 8, ...
  {
    float acc[NT][2][4];
#pragma unroll
    for (int m = 0; m < NT; ++m)
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[m][n][i] = 0.f;
    const uint32_t b_base = s_u32(d3s + (size_t)((lane & 7) + ((lane >> 3) & 1) * 8) * WP + (lane >> 4) * 8);
    const uint32_t a_base = s_u32(hs + (size_t)((lane & 7) + ((lane >> 4) & 1) * 8) * HP + ((lane >> 3) & 1) * 8);
    // bias sums: a product with ones (every row of it is the column sum)
    const uint32_t ones[4] = {0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u};
    float bias_sum[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int ks = 0; ks < ROWS / 16; ++ks) {
      uint32_t bf[4];
      ldsm4t(b_base + ks * 16 * WP * 2, bf);
      if (warp == 0) {
        mma16816_rn(bias_sum[0], ones, bf[0], bf[1]);
        mma16816_rn(bias_sum[1], ones, bf[2], bf[3]);
      }
#pragma unroll
      for (int m = 0; m < NT; ++m) {
        uint32_t af[4];
        ldsm4t(a_base + (uint32_t)(ks * 16 * HP + (warp + 8 * m) * 16) * 2, af);
        mma16816(acc[m][0], af, bf[0], bf[1]);
        mma16816(acc[m][1], af, bf[2], bf[3]);
      }
    }
    float* dst = part + (size_t)blockIdx.x * (size_t)(IN + 1) * C;
#pragma unroll
    for (int m = 0; m < NT; ++m)
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int f = (warp + 8 * m) * 16 + g + 8 * (i >> 1), c = 8 * n + 2 * t + (i & 1);
          if (c < C) dst[(size_t)f * C + c] = acc[m][n][i];
        }
    if (warp == 0 && g == 0) {
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int j = 0; j < 2; ++j)
          if (8 * n + 2 * t + j < C) dst[(size_t)IN * C + 8 * n + 2 * t + j] = bias_sum[n][j];
    }
  }
  if (!has_dgrad) return;
  __syncthreads();            // all reads of the input rows by the gradient phase are done

  // ---- delta of the layer below, written over the input rows: warp w owns features [w*IN/8, (w+1)*IN/8)
  {
    uint32_t af[ROWS / 16][4];
#pragma unroll
    for (int mt = 0; mt < ROWS / 16; ++mt)
      ldsm4(s_u32(d3s + (size_t)(16 * mt + (lane & 15)) * WP + (lane >> 4) * 8), af[mt]);
    const uint32_t b_base = s_u32(ws + (size_t)((lane & 7) + ((lane >> 4) & 1) * 8) * WP + ((lane >> 3) & 1) * 8);
#pragma unroll 2
    for (int f0 = warp * (IN / 8); f0 < (warp + 1) * (IN / 8); f0 += 16) {
      uint32_t bf[4];
      ldsm4(b_base + f0 * WP * 2, bf);
#pragma unroll
      for (int mt = 0; mt < ROWS / 16; ++mt)
#pragma unroll
        for (int n = 0; n < 2; ++n) {
          float d[4] = {0.f, 0.f, 0.f, 0.f};
          mma16816(d, af[mt], bf[2 * n], bf[2 * n + 1]);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t* hp = reinterpret_cast<uint32_t*>(hs + (size_t)(16 * mt + g + 8 * h) * HP + f0 + 8 * n + 2 * t);
            const float2 hv = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(hp));
            *hp = pack_bf16(hv.x > 0.f ? d[2 * h] : 0.f, hv.y > 0.f ? d[2 * h + 1] : 0.f);
          }
        }
    }
  }
  __syncthreads();
  __nv_bfloat16* out = (__nv_bfloat16*)a.delta_in + (size_t)r0 * IN;
  for (int item = tid; item < ROWS * (IN / 8); item += THREADS) {
    const int rr = item / (IN / 8), v = item - rr * (IN / 8);
    *reinterpret_cast<uint4*>(out + (size_t)rr * IN + v * 8) = *reinterpret_cast<const uint4*>(hs + (size_t)rr * HP + v * 8);
  }
}

}  // namespace outl
}  // namespace absb
