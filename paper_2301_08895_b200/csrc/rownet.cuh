// Networks without tcgen05 layers (fp32 storage, or bf16 widths TMA cannot address) and the fully connected part of
// the CNN, two kernels per round:
//   rows_fma_kernel / rows_mma_kernel   CTA = R gradient rows of one model version: all layers forward (Eq. 2 at the
//                     version the rows' workers hold), soft-max cross-entropy, all layers' deltas backward,
//   grad_step_kernel  weight and bias gradients of all layers, each 32 x 32 block summed over all rows of the round
//                     (Eq. 3), and the SGD step and ring write of that block in the same CTA.
// One launch per layer and direction would be bound by launch gaps and by grids of a few CTAs: rounds of this model
// class are a few hundred rows and 10^4 .. 10^6 parameters.
// Measured per round (one launch per layer and direction -> this): 300-123-57-7 fp32, 13 workers x 37 rows: 114 -> 18 us
// (11 -> 3 launches); 784-10 fp32, 16 x 64: 22 -> 14 us; the 400-120-84-10 part of the CNN, 640 rows: 13 -> 2 launches,
// 17 us for the row kernel between two events (28 us with FP32 FMAs for the bf16 products).
// Activations and deltas are rounded to the storage type where they are stored, sums are fp32 in a fixed order.
#pragma once
#include <algorithm>

#include "common.cuh"
#include "convmma.cuh"
#include "ctl.cuh"
#include "lsqpipe.cuh"
#include "narrow.cuh"
#include "outlayer.cuh"
#include "tc.cuh"

namespace absb {
namespace rnet {

using lsqp::f32x2;

constexpr int NW = 8;                    // compute warps of the row kernels
constexpr int NT = NW * 32;
constexpr int THREADS = NT + 32;         // and the warp that fetches the weights
constexpr int MAX_STAGES = 8;
constexpr int MMA_NW = 15;               // its compute warps: with the fetching warp 512 threads of up to 128 registers
constexpr int MMA_THREADS = MMA_NW * 32 + 32;

struct RowsArgs {
  DevState* st;
  RoundInfo* ri;
  const int* tile_slot;                  // ring slot of every R rows (the row padding unit)
  const int* row_idx;                    // sample index per gradient row, -1: padding
  const int* labels;
  const void* ring; size_t slot_stride;
  const int* job; u64* next_dur; int* dur_job; int W;    // duration look-ahead (see refresh_next_durations)
  const void* X; int gather;             // layer-0 input of row r: X[row_idx[r]] (gather) or X[r]
  void* act[ABS_MAX_LAYERS + 1];         // [rows][dims[l]] stored ReLU outputs, l = 1 .. n_layers - 1
  void* delta[ABS_MAX_LAYERS + 1];       // [rows][dims[l]] stored deltas, l = 1 .. n_layers; delta[0]: see want_d0
  float* row_loss;                       // [rows]
  size_t w_off[ABS_MAX_LAYERS];          // element offset of W[in][out]; the bias follows it as row `in`
  int n_layers, dims[ABS_MAX_LAYERS + 1];
  int sa, S;                             // DevState's staleness-aware step size and ring
  int want_d0;                           // also the delta of the layer-0 input (CNN features, masked by feature > 0)
  // Weights in shared memory.  resident: every layer is copied once and stays (stage l = layer l, the backward pass
  // reads it again); otherwise chunks of rpc[l] rows stream through `stages` stages, forward and again backward.
  int resident, stages, stage_bytes;
  int w_bytes;                           // ... all of them
  int w_res[ABS_MAX_LAYERS];             // byte offset of layer l (resident)
  int rpc[ABS_MAX_LAYERS];               // rows per chunk: a multiple of 16 (chunks start on 16 bytes), or all of them
  int act_off[ABS_MAX_LAYERS];           // element offset (T) of layer l's input behind the weights
  int out_off, red_off;                  // fma: logits [C] quads, partial sums (floats); mma: output delta (T), logits (bytes)
};

__host__ __device__ inline int mma_pitch(int n) { return round_up(n, 16) + 8; }   // bf16 row pitch, zero-padded to 16

// Shared-memory plan for R rows per CTA; false: does not fit.
inline bool plan_rows(RowsArgs* a, int R, int esz, size_t* smem) {
  const bool mma = esz == 2;
  int off = 0;
  for (int l = 0; l < a->n_layers; ++l) {
    if (a->dims[l + 1] > 1024) return false;           // columns all warps of a CTA can hold
    a->act_off[l] = off;
    off += mma ? R * mma_pitch(a->dims[l]) : (a->dims[l] + 1) * R;
  }
  a->out_off = off;
  const int C = a->dims[a->n_layers];
  size_t bytes;
  if (mma) {
    off += R * mma_pitch(C);
    a->red_off = round_up(2 * off, 16);
    bytes = (size_t)a->red_off + (size_t)4 * R * (C + 1);
  } else {
    off += C * R;
    a->red_off = round_up(off, 4);
    bytes = 4 * ((size_t)a->red_off + (size_t)NW * 128 * R);
  }
  bytes += 128;
  size_t all = 0, stage = 0;
  for (int l = 0; l < a->n_layers; ++l) {
    a->w_res[l] = (int)std::min<size_t>(all, 1u << 30);
    a->rpc[l] = a->dims[l] + 1;
    all += round_up_sz((size_t)(a->dims[l] + 1) * a->dims[l + 1] * esz, 128);
  }
  a->resident = all + bytes <= 220 * 1024;
  a->stages = a->n_layers;
  a->stage_bytes = 0;
  *smem = all + bytes;
  a->w_bytes = (int)std::min<size_t>(all, 1u << 30);
  if (a->resident) return true;
  for (int l = 0; l < a->n_layers; ++l) {
    const size_t row16 = (size_t)16 * a->dims[l + 1] * esz;
    a->rpc[l] = 16 * (int)std::max<size_t>(1, 24576 / row16);
    stage = std::max(stage, round_up_sz((size_t)a->rpc[l] * a->dims[l + 1] * esz, 128));
  }
  a->stage_bytes = (int)stage;
  for (a->stages = MAX_STAGES; a->stages >= 2; --a->stages) {
    *smem = (size_t)a->stages * stage + bytes;
    a->w_bytes = a->stages * (int)stage;
    if (*smem <= 220 * 1024) return true;
  }
  return false;
}

__device__ __forceinline__ void rows_sync() { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); }

// The weights of the CTA's model version, in shared memory (see RowsArgs::resident).
struct Weights {
  const RowsArgs& a;
  unsigned char* base;
  uint64_t *full, *empty;
  int* gave_up;
  int stage = 0;
  uint32_t phase = 0;
  __device__ __forceinline__ Weights(const RowsArgs& a_, unsigned char* b, uint64_t* f, uint64_t* e, int* g)
      : a(a_), base(b), full(f), empty(e), gave_up(g) {}
  // one thread: all copies, in the order the consumers take them
  template <typename T>
  __device__ __forceinline__ void produce(const T* ring) {
    const int L = a.n_layers, l_min = a.want_d0 ? 0 : 1;
    bool ok = true;
    for (int step = 0; step < (a.resident ? L : 2 * L - l_min) && ok; ++step) {
      const int l = step < L ? step : 2 * L - 1 - step;
      const int rows = a.dims[l] + 1, out = a.dims[l + 1], rpc = a.rpc[l];
      const T* w = ring + a.w_off[l];
      for (int k0 = 0; k0 < rows; k0 += rpc) {
        if (!a.resident) ok = tc::mbar_wait(&empty[stage], phase ^ 1u, gave_up);
        if (!ok) break;
        // (the last piece of a layer may run up to 12 bytes into the padding behind it)
        const uint32_t bytes = (uint32_t)round_up(min(rpc, rows - k0) * out * (int)sizeof(T), 16);
        tc::mbar_expect_tx(&full[stage], bytes);
        lsqp::bulk_row(base + (a.resident ? (size_t)a.w_res[l] : (size_t)stage * a.stage_bytes), w + (size_t)k0 * out, bytes, &full[stage]);
        if (++stage == a.stages) { stage = 0; phase ^= 1u; }
      }
    }
  }
  // consumers: the next chunk (of layer l); a wait that runs out ends the run at the end of the kernel
  __device__ __forceinline__ const void* take(int l) {
    if (a.resident) {
      tc::mbar_wait(&full[l], 0u, gave_up);
      return base + a.w_res[l];
    }
    tc::mbar_wait(&full[stage], phase, gave_up);
    return base + (size_t)stage * a.stage_bytes;
  }
  __device__ __forceinline__ void give(int lane) {
    if (a.resident) return;
    __syncwarp();
    if (lane == 0) tc::mbar_arrive(&empty[stage]);
    if (++stage == a.stages) { stage = 0; phase ^= 1u; }
  }
};

__device__ __forceinline__ void weights_init(const RowsArgs& a, uint64_t* full, uint64_t* empty, int* gave_up, int n_warps) {
  if (threadIdx.x == 0) {
    for (int s = 0; s < a.stages; ++s) { tc::mbar_init(&full[s], 1); tc::mbar_init(&empty[s], n_warps); }
    *gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
}
__device__ __forceinline__ void rows_end(const RowsArgs& a, const int* gave_up) {
  __syncthreads();
  if (threadIdx.x == 0 && *gave_up) {
    // let copies in flight land before the shared memory goes away
    const unsigned long long t0 = tc::global_ns();
    while (tc::global_ns() - t0 < 200000ull) {}
    a.st->timeout_where = 400;
    report(a.ri, RI_TIMEOUT);
  }
}

// Soft-max cross-entropy of one row by one warp: lane holds the logits of classes lane and lane + 32 (at most 64);
// returns their deltas (0 for a padding row, label -1) and publishes the loss.
template <typename T>
__device__ __forceinline__ float2 row_softmax(const RowsArgs& a, float z0, float z1, int r, int yl, float sa, int lane) {
  const int C = a.dims[a.n_layers];
  z0 = lane < C ? z0 : NO_CLASS;
  z1 = lane + 32 < C ? z1 : NO_CLASS;
  float zmax = fmaxf(z0, z1);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, o));
  const float e0 = expf(z0 - zmax), e1 = expf(z1 - zmax);
  float se = e0 + e1, zy = (lane == yl ? z0 : 0.f) + (lane + 32 == yl ? z1 : 0.f);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    se += __shfl_xor_sync(0xffffffffu, se, o);
    zy += __shfl_xor_sync(0xffffffffu, zy, o);
  }
  const float inv = 1.f / se;
  if (lane == 0) {
    const float loss = yl < 0 ? 0.f : logf(se) - (zy - zmax);
    a.row_loss[r] = loss;
    if (!isfinite(loss)) report(a.ri, RI_DIVERGED);
  }
  // a delta is a stored quantity; sa: staleness-aware step size (weight of these rows in Eq. 3)
  if (yl < 0) return make_float2(0.f, 0.f);
  return make_float2(round_store((e0 * inv - (lane == yl ? 1.f : 0.f)) * sa, (const T*)nullptr),
                     round_store((e1 * inv - (lane + 32 == yl ? 1.f : 0.f)) * sa, (const T*)nullptr));
}

// Sum over the lanes of 32 values per lane: afterwards lane l holds the sum of value l (31 exchanges; each halves the
// values a lane still carries).
__device__ __forceinline__ float lane_transpose_sum(float (&v)[32], int lane) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool hi = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (i < o) {
        const float send = hi ? v[i] : v[i + o], keep = hi ? v[i + o] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
  }
  return v[0];
}

// ---- fp32: rows kept as [R / 4][k][4], so that one 16-byte read serves four rows of an input (all lanes, forward) or of
// 32 columns (backward).
// Partial products of one chunk: lane owns columns n0 + CW j (j < CPT, CW lanes per group of columns), and takes every
// KGS-th weight row.  Per row and warp: CPT 4-byte and R / 4 16-byte shared-memory reads (1 and 2 cycles) for CPT R / 2
// packed FMAs (2 cycles on each of four schedulers): the reads bound it up to CPT = 2.
template <int R, int CPT, int CW>
__device__ __forceinline__ void fma_chunk(f32x2 (&z)[4][R / 2], const float* w, const float* x, int plane, int nk, int kg, int kgs,
                                          int out, int n0) {
  int col[CPT];
#pragma unroll
  for (int j = 0; j < CPT; ++j) col[j] = min(n0 + CW * j, out - 1);
  const float* wp = w + kg * out;
  const float* xp = x + kg * 4;
  const int ws = kgs * out, xs = kgs * 4;
  constexpr int UN = CPT == 4 ? 2 : 4;
  int k = kg;
  for (; k + (UN - 1) * kgs < nk; k += UN * kgs) {
    float wv[UN][CPT];
    ulonglong2 xv[UN][R / 4];
#pragma unroll
    for (int u = 0; u < UN; ++u) {
#pragma unroll
      for (int j = 0; j < CPT; ++j) wv[u][j] = wp[u * ws + col[j]];
#pragma unroll
      for (int q = 0; q < R / 4; ++q) xv[u][q] = *reinterpret_cast<const ulonglong2*>(xp + u * xs + q * plane);
    }
#pragma unroll
    for (int u = 0; u < UN; ++u)
#pragma unroll
      for (int j = 0; j < CPT; ++j) {
        const f32x2 p = lsqp::pack2(wv[u][j], wv[u][j]);
#pragma unroll
        for (int q = 0; q < R / 4; ++q) {
          lsqp::ffma2(z[j][2 * q], p, xv[u][q].x);
          lsqp::ffma2(z[j][2 * q + 1], p, xv[u][q].y);
        }
      }
    wp += UN * ws;
    xp += UN * xs;
  }
  for (; k < nk; k += kgs) {
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
      const float wv = wp[col[j]];
      const f32x2 p = lsqp::pack2(wv, wv);
#pragma unroll
      for (int q = 0; q < R / 4; ++q) {
        const ulonglong2 xv = *reinterpret_cast<const ulonglong2*>(xp + q * plane);
        lsqp::ffma2(z[j][2 * q], p, xv.x);
        lsqp::ffma2(z[j][2 * q + 1], p, xv.y);
      }
    }
    wp += ws;
    xp += xs;
  }
}

// Forward of one layer up to the partial sums red[KGS][NP][R] (NP = columns rounded up); returns KGS, NP.
template <int R, int CPT, int CW>
__device__ __forceinline__ int2 fma_layer(Weights& W, int l, const float* x, float* red, int warp, int lane) {
  const int rows = W.a.dims[l] + 1, out = W.a.dims[l + 1], rpc = W.a.rpc[l];
  constexpr int COLS = CPT * CW, SUB = 32 / CW;
  const int ncw = (out + COLS - 1) / COLS, wk = NW / ncw;     // warps across the columns / across the weight rows
  const int g = warp / ncw, cw = warp - g * ncw;
  const int kg = g * SUB + lane / CW, kgs = wk * SUB, n0 = cw * COLS + lane % CW;
  const int plane = rows * 4;
  f32x2 z[4][R / 2];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int q = 0; q < R / 2; ++q) z[j][q] = 0ull;
  for (int k0 = 0; k0 < rows; k0 += rpc) {
    const float* w = reinterpret_cast<const float*>(W.take(l));
    if (g < wk) fma_chunk<R, CPT, CW>(z, w, x + k0 * 4, plane, min(rpc, rows - k0), kg, kgs, out, n0);
    W.give(lane);
  }
  if (g < wk) {
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
      float* o = red + (size_t)(kg * ncw * COLS + n0 + CW * j) * R;
#pragma unroll
      for (int q = 0; q < R / 4; ++q) *reinterpret_cast<ulonglong2*>(o + 4 * q) = make_ulonglong2(z[j][2 * q], z[j][2 * q + 1]);
    }
  }
  return make_int2(kgs, ncw * COLS);
}

template <int R>
__global__ void __launch_bounds__(THREADS, 1) rows_fma_kernel(const __grid_constant__ RowsArgs a) {
  extern __shared__ __align__(128) unsigned char rsm[];
  __shared__ uint64_t full[MAX_STAGES], empty[MAX_STAGES];
  __shared__ int gave_up;
  __shared__ int lab[R];                             // label of each row, -1: padding
  weights_init(a, full, empty, &gave_up, NW);        // before the wait: touches nothing of the kernels in front
  grid_dependency_sync();
  DevState* st = a.st;
  RoundInfo* ri = a.ri;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = (int)blockIdx.x * R;
  // one wave of loads (the grid covers the row capacity, so every address exists)
  const int status = st->status, n_rows = ri->n_rows, t_round = ri->t, slot = a.tile_slot[blockIdx.x];
  const int my_idx = a.row_idx[r0 + lane % R];       // sample index of row lane % R
  if (status != ST_OK) return;
  // the fetching warps of the first CTAs also prepare job durations, off the critical path
  const int look = (int)blockIdx.x * 32 < a.W ? (int)blockIdx.x * 32 + lane : a.W;
  if (r0 >= n_rows) {
    if (warp == NW) refresh_next_durations(st, a.job, a.next_dur, a.dur_job, look);
    return;
  }
  const int L = a.n_layers;
  float* fs = reinterpret_cast<float*>(rsm + a.w_bytes);
  Weights W(a, rsm, full, empty, &gave_up);
  constexpr int RQ = R / 4;

  if (warp == NW) {
    if (lane == 0) W.produce((const float*)a.ring + (size_t)slot * a.slot_stride);
    __syncwarp();
    refresh_next_durations(st, a.job, a.next_dur, a.dur_job, look);
  } else {
    const int label = (tid < R && my_idx >= 0) ? a.labels[my_idx] : -1;       // stored when first needed
    // ------------------------------------------------------------------ input rows
    {
      const int in = a.dims[0];
      float* x = fs + a.act_off[0];
      const int rq = warp % RQ;                      // (RQ divides NW) four rows per warp
      const float* src[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = r0 + rq * 4 + j;
        const int s = __shfl_sync(0xffffffffu, my_idx, rq * 4 + j);
        src[j] = (a.gather && s < 0) ? nullptr : (const float*)a.X + (size_t)(a.gather ? s : r) * in;
      }
      // all loads of up to 32 / R x 256 features in flight at once: the rows come from all over the dataset (784
      // features, 8 rows: 6000 cycles with two iterations in flight)
      constexpr int KB = 8, KSTEP = NW / RQ * 32;
      for (int kb = (warp / RQ) * 32 + lane; kb < in; kb += KB * KSTEP) {
        float v[KB][4];
#pragma unroll
        for (int u = 0; u < KB; ++u)
#pragma unroll
          for (int j = 0; j < 4; ++j) v[u][j] = (src[j] && kb + u * KSTEP < in) ? src[j][kb + u * KSTEP] : 0.f;
#pragma unroll
        for (int u = 0; u < KB; ++u)
          if (kb + u * KSTEP < in)
            *reinterpret_cast<float4*>(x + (size_t)rq * (in + 1) * 4 + (kb + u * KSTEP) * 4) = make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
      }
      for (int e = tid; e < L * R; e += NT) {         // the input of the bias row
        const int l = e / R, q = e % R / 4;
        fs[a.act_off[l] + (q * (a.dims[l] + 1) + a.dims[l]) * 4 + (e & 3)] = 1.f;
      }
    }
    rows_sync();
    // ------------------------------------------------------------------ forward
    float* red = fs + a.red_off;
    for (int l = 0; l < L; ++l) {
      const int out = a.dims[l + 1];
      const bool last = l == L - 1;
      const float* x = fs + a.act_off[l];
      int2 kn;
      if (out > 64) kn = fma_layer<R, 4, 32>(W, l, x, red, warp, lane);
      else if (out > 32) kn = fma_layer<R, 2, 32>(W, l, x, red, warp, lane);
      else if (out > 16) kn = fma_layer<R, 1, 32>(W, l, x, red, warp, lane);
      else if (out > 8) kn = fma_layer<R, 1, 16>(W, l, x, red, warp, lane);
      else kn = fma_layer<R, 1, 8>(W, l, x, red, warp, lane);
      rows_sync();
      float* y = fs + (last ? a.out_off : a.act_off[l + 1]);
      const int y_plane = (last ? out : out + 1) * 4;
      float* ga = last ? nullptr : (float*)a.act[l + 1];
      for (int e = tid; e < out * RQ; e += NT) {      // partial sums in order, ReLU
        const int n = e / RQ, q = e % RQ;
        const float4* p = reinterpret_cast<const float4*>(red) + (size_t)n * RQ + q;
        float4 s = p[0];
#pragma unroll 4
        for (int g = 1; g < kn.x; ++g) {
          const float4 t = p[(size_t)g * kn.y * RQ];
          s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
        }
        if (!last) {
          s.x = fmaxf(s.x, 0.f); s.y = fmaxf(s.y, 0.f); s.z = fmaxf(s.z, 0.f); s.w = fmaxf(s.w, 0.f);
          const size_t o = (size_t)(r0 + 4 * q) * out + n;
          ga[o] = s.x; ga[o + out] = s.y; ga[o + 2 * (size_t)out] = s.z; ga[o + 3 * (size_t)out] = s.w;
        }
        *reinterpret_cast<float4*>(y + (size_t)q * y_plane + n * 4) = s;
      }
      if (last && tid < R) lab[tid] = label;
      rows_sync();
    }
    // ------------------------------------------------------------------ loss and delta of the output layer: warp = row
    {
      const int C = a.dims[L];
      float* z = fs + a.out_off;
      for (int rr = warp; rr < R; rr += NW) {
        float* zr = z + (rr / 4) * C * 4 + (rr & 3);
        const float2 d = row_softmax<float>(a, lane < C ? zr[lane * 4] : 0.f, lane + 32 < C ? zr[(lane + 32) * 4] : 0.f, r0 + rr, lab[rr],
                                            sa_slot_weight(a.sa, a.S, t_round, slot), lane);
        float* gd = (float*)a.delta[L] + (size_t)(r0 + rr) * C;
        if (lane < C) { zr[lane * 4] = d.x; gd[lane] = d.x; }
        if (lane + 32 < C) { zr[(lane + 32) * 4] = d.y; gd[lane + 32] = d.y; }
      }
    }
    rows_sync();
    // ------------------------------------------------------------------ backward: the delta of layer l's input takes the
    // place of that input (only its sign is still needed, by the lane that overwrites it)
    for (int l = L - 1; l >= (a.want_d0 ? 0 : 1); --l) {
      constexpr int MB = 32 / R;                     // weight rows per warp step
      const int in = a.dims[l], out = a.dims[l + 1], rpc = a.rpc[l];
      const float* dl = fs + (l == L - 1 ? a.out_off : a.act_off[l + 1]);
      const int d_plane = (l == L - 1 ? out : out + 1) * 4;
      float* h = fs + a.act_off[l];
      float* gd = (float*)a.delta[l];
      for (int k0 = 0; k0 < in + 1; k0 += rpc) {
        const float* w = reinterpret_cast<const float*>(W.take(l));
        const int nk = min(rpc, in - k0);
        for (int mb = warp * MB; mb < nk; mb += NW * MB) {
          f32x2 acc[MB][R / 2];
#pragma unroll
          for (int i = 0; i < MB; ++i)
#pragma unroll
            for (int j = 0; j < R / 2; ++j) acc[i][j] = 0ull;
          const float* wr[MB];
#pragma unroll
          for (int i = 0; i < MB; ++i) wr[i] = w + min(mb + i, nk - 1) * out;
#pragma unroll 2
          for (int n = lane; n < out; n += 32) {
            f32x2 d2[R / 2];
#pragma unroll
            for (int q = 0; q < RQ; ++q) {
              const ulonglong2 dv = *reinterpret_cast<const ulonglong2*>(dl + q * d_plane + n * 4);
              d2[2 * q] = dv.x;
              d2[2 * q + 1] = dv.y;
            }
#pragma unroll
            for (int i = 0; i < MB; ++i) {
              const float wv = wr[i][n];
              const f32x2 p = lsqp::pack2(wv, wv);
#pragma unroll
              for (int j = 0; j < R / 2; ++j) lsqp::ffma2(acc[i][j], p, d2[j]);
            }
          }
          float v[32];
#pragma unroll
          for (int i = 0; i < MB; ++i)
#pragma unroll
            for (int j = 0; j < R / 2; ++j) lsqp::unpack2(acc[i][j], v[i * R + 2 * j], v[i * R + 2 * j + 1]);
          const float s = lane_transpose_sum(v, lane);
          const int mi = mb + lane / R, rr = lane % R;
          if (mi < nk) {
            float* hp = h + (size_t)(rr / 4) * (in + 1) * 4 + (size_t)(k0 + mi) * 4 + (rr & 3);
            const float d = *hp > 0.f ? s : 0.f;
            *hp = d;
            gd[(size_t)(r0 + rr) * in + k0 + mi] = d;
          }
        }
        W.give(lane);
      }
      rows_sync();
    }
  }
  rows_end(a, &gave_up);
}

// ---- bf16: the same with the warp-level tensor-core instruction (mma m16n8k16, bf16 in, fp32 accumulate): the weights
// are the row operand (16 columns of a layer, backward 16 of its inputs), the CTA's gradient rows the column operand, 8
// or 16 kept as [row][k] (pitch: a multiple of 16 plus 8 elements, zero-padded).  Row i of an operand tile is column 2i of the
// layer, row i + 8 column 2i + 1, so that even widths are read as 4-byte pairs and results stored as pairs; the widths of
// this class rarely give the 16-byte rows of ldmatrix.  (tcgen05 tiles would be 128 rows; a round has a few hundred rows
// in groups of any size.)  Bound by shared-memory reads of the weights and the latency of the layers' chain.
// 400-120-84-10, 640 rows: 16.8 us with the rows as row operand and unrolled tiles, 12.7 us now (between launches).
__device__ __forceinline__ uint32_t pair16(const __nv_bfloat16* p, int stride) {          // p[0] | p[stride] << 16
  const uint32_t lo = *reinterpret_cast<const unsigned short*>(p), hi = *reinterpret_cast<const unsigned short*>(p + stride);
  return lo | (hi << 16);
}
// elements c and c + 1 of a row of n, clamped to the row (what lies behind it meets zeros)
template <bool EVEN>
__device__ __forceinline__ uint32_t pair_at(const __nv_bfloat16* row, int c, int n) {
  if (EVEN) return *reinterpret_cast<const uint32_t*>(row + min(c, n - 2));
  const int c0 = min(c, n - 1);
  return pair16(row + c0, min(c + 1, n - 1) - c0);
}
// One tile of 16 layer columns over rows [0, nk) of a chunk (n: this lane's two columns): the operands of the next 32 rows
// are read while these are multiplied.  Rows behind the last one meet zero activations.  RT: column tiles of 8 gradient
// rows, `xt` bytes apart.  UN: unrolled, for weights that come in many chunks; code that runs once or twice per CTA is
// bound by fetching its instructions and kept short instead (400-120-84-10, 640 rows: 16.7 us unrolled, 12.7 us).
template <bool EVEN, int RT, bool UN>
__device__ __forceinline__ void forward_tile(float (&acc)[RT][4], const __nv_bfloat16* w, uint32_t x, uint32_t xt, int n, int nk, int out, int t) {
  uint32_t b[RT][4], p[8];
  auto load = [&](int k) {
#pragma unroll
    for (int r = 0; r < RT; ++r) outl::ldsm4(x + r * xt + (uint32_t)k * 2u, b[r]);       // (columns behind the padding are not used)
#pragma unroll
    for (int i = 0; i < 8; ++i) p[i] = pair_at<EVEN>(w + min(k + 2 * t + (i >> 1) * 8 + (i & 1), nk - 1) * out, n, out);
  };
  auto multiply = [&](bool both) {
    uint32_t af[2][4];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int i = 0; i < 4; ++i) af[u][i] = __byte_perm(p[4 * u + (i & 2)], p[4 * u + (i & 2) + 1], (i & 1) ? 0x7632 : 0x5410);
#pragma unroll
    for (int r = 0; r < RT; ++r) outl::mma16816_rn(acc[r], af[0], b[r][0], b[r][1]);
    if (both)
#pragma unroll
      for (int r = 0; r < RT; ++r) outl::mma16816_rn(acc[r], af[1], b[r][2], b[r][3]);
  };
  int k = 0;
  if (UN) {
    const __nv_bfloat16* q = w + 2 * t * out;
#pragma unroll 2
    for (; k + 32 <= nk; k += 32) {
#pragma unroll
      for (int r = 0; r < RT; ++r) outl::ldsm4(x + r * xt + (uint32_t)k * 2u, b[r]);
#pragma unroll
      for (int i = 0; i < 8; ++i) p[i] = pair_at<EVEN>(q + ((i >> 1) * 8 + (i & 1)) * out, n, out);
      multiply(true);
      q += 32 * out;
    }
    if (k < nk) {
      load(k);
      multiply(k + 16 < nk);
    }
    return;
  }
  load(0);
#pragma unroll 1
  for (; k < nk; k += 32) {
    uint32_t af[2][4], c[RT][4];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int i = 0; i < 4; ++i) af[u][i] = __byte_perm(p[4 * u + (i & 2)], p[4 * u + (i & 2) + 1], (i & 1) ? 0x7632 : 0x5410);
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
      for (int i = 0; i < 4; ++i) c[r][i] = b[r][i];
    if (k + 32 < nk) load(k + 32);
#pragma unroll
    for (int r = 0; r < RT; ++r) outl::mma16816_rn(acc[r], af[0], c[r][0], c[r][1]);
    if (k + 16 < nk)
#pragma unroll
      for (int r = 0; r < RT; ++r) outl::mma16816_rn(acc[r], af[1], c[r][2], c[r][3]);
  }
}
// the same backward: 16 weight rows, of which wa, wb are this lane's, over the layer's columns
template <bool EVEN, int RT, bool UN>
__device__ __forceinline__ void backward_tile(float (&acc)[RT][4], const __nv_bfloat16* wa, const __nv_bfloat16* wb, uint32_t d, uint32_t dt, int out, int t) {
#pragma unroll UN ? 2 : 1
  for (int n = 0; n < out; n += 32) {
    uint32_t b[RT][4], p[8];
#pragma unroll
    for (int r = 0; r < RT; ++r) outl::ldsm4(d + r * dt + (uint32_t)n * 2u, b[r]);
#pragma unroll
    for (int i = 0; i < 8; ++i) p[i] = pair_at<EVEN>((i & 1) ? wb : wa, n + 2 * t + (i >> 1) * 8, out);
    const uint32_t a0[4] = {p[0], p[1], p[2], p[3]}, a1[4] = {p[4], p[5], p[6], p[7]};
#pragma unroll
    for (int r = 0; r < RT; ++r) outl::mma16816_rn(acc[r], a0, b[r][0], b[r][1]);
    if (n + 16 < out)
#pragma unroll
      for (int r = 0; r < RT; ++r) outl::mma16816_rn(acc[r], a1, b[r][2], b[r][3]);
  }
}

// rows [R][pitch] of shared memory -> rows of n elements: R = 8 two warps per row (one for the last), 16 one (two for the last)
template <int R>
__device__ __forceinline__ void copy_rows(__nv_bfloat16* dst, const __nv_bfloat16* src, int pitch, int n, int warp, int lane) {
  if (R == 16 && warp == 0) copy_rows<1>(dst + 15 * (size_t)n, src + 15 * pitch, pitch, n, 0, lane);      // (15 warps)
  const int rr = warp % R, at = warp / R, of = R == 8 && rr + R < MMA_NW ? 2 : 1;
  if ((n & 7) == 0) {
#pragma unroll 1
    for (int k = (at * 32 + lane) * 8; k < n; k += of * 256)
      *reinterpret_cast<uint4*>(dst + (size_t)rr * n + k) = *reinterpret_cast<const uint4*>(src + rr * pitch + k);
  } else {
#pragma unroll 1
    for (int k = at * 32 + lane; k < n; k += of * 32) dst[(size_t)rr * n + k] = src[rr * pitch + k];
  }
}

template <int R, bool RESIDENT>
__global__ void __launch_bounds__(MMA_THREADS, 1) rows_mma_kernel(const __grid_constant__ RowsArgs a) {
  extern __shared__ __align__(128) unsigned char rsm[];
  __shared__ uint64_t full[MAX_STAGES], empty[MAX_STAGES];
  __shared__ int gave_up;
  __shared__ int lab[R];                             // label of each row, -1: padding
  typedef __nv_bfloat16 T;
  constexpr int RT = R / 8, WPR = 16 / R, NWM = MMA_NW;
  weights_init(a, full, empty, &gave_up, NWM);       // before the wait: touches nothing of the kernels in front
  grid_dependency_sync();
  DevState* st = a.st;
  RoundInfo* ri = a.ri;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = (int)blockIdx.x * R;
  const int my_row = warp / WPR;                     // two warps (of 16) or one fetch a row
  // one wave of loads (the grid covers the row capacity, so every address exists)
  const int status = st->status, n_rows = ri->n_rows, t_round = ri->t, slot = a.tile_slot[blockIdx.x];
  const int my_idx = a.row_idx[r0 + my_row], lab_idx = tid < R ? a.row_idx[r0 + tid] : -1;
  if (status != ST_OK) return;
  const int look = (int)blockIdx.x * 32 < a.W ? (int)blockIdx.x * 32 + lane : a.W;
  if (r0 >= n_rows) {
    if (warp == NWM) refresh_next_durations(st, a.job, a.next_dur, a.dur_job, look);
    return;
  }
  const int g = lane >> 2, t = lane & 3;
  const int L = a.n_layers;
  T* ts = reinterpret_cast<T*>(rsm + a.w_bytes);
  Weights W(a, rsm, full, empty, &gave_up);
  auto sync_compute = [] { asm volatile("bar.sync 1, %0;" ::"n"(NWM * 32) : "memory"); };
  const T* w_ring = (const T*)a.ring + (size_t)slot * a.slot_stride;
  if (RESIDENT && tid == NWM * 32) W.produce(w_ring);
  __syncwarp();
  const int label = lab_idx >= 0 ? a.labels[lab_idx] : -1;       // stored when first needed
  {
    // ---------------------------------------------------------------- input row (part) of this warp; zero padding columns
    const int in = a.dims[0], part = warp % WPR;
    const T* src = (a.gather && my_idx < 0) ? nullptr : (const T*)a.X + (size_t)(a.gather ? my_idx : r0 + my_row) * in;
    T* x = ts + a.act_off[0] + my_row * mma_pitch(in);
    if ((in & 7) == 0) {                              // rows on 16-byte boundaries
#pragma unroll 4
      for (int k = (part * 32 + lane) * 8; k < in; k += 256 * WPR)
        *reinterpret_cast<uint4*>(x + k) = src ? *reinterpret_cast<const uint4*>(src + k) : make_uint4(0u, 0u, 0u, 0u);
    } else {
#pragma unroll 8
      for (int k = part * 32 + lane; k < in; k += 32 * WPR) x[k] = src ? src[k] : (T)0.f;
    }
    if (part == 0) {
#pragma unroll 1
      for (int l = 0; l <= L; ++l) {
        const int n = a.dims[l], p = mma_pitch(n);    // at most 8 + 15 padding columns
        if (n + lane < p) ts[(l < L ? a.act_off[l] : a.out_off) + my_row * p + n + lane] = (T)0.f;
      }
    }
  }
  __syncthreads();

  if (warp == NWM) {
    if (!RESIDENT && lane == 0) W.produce(w_ring);
    __syncwarp();
    refresh_next_durations(st, a.job, a.next_dur, a.dur_job, look);
  } else {
    const int sel = (lane & 7), sel_col = (lane >> 3) * 8;            // ldmatrix addresses: two inner steps of 16 at once
    // ------------------------------------------------------------------ forward: warp takes column tiles warp, warp + 15, ...
    float* logits = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(ts) + a.red_off);     // [R][C + 1]
    for (int l = 0; l < L; ++l) {
      const int in = a.dims[l], out = a.dims[l + 1], rpc = a.rpc[l], pitch = mma_pitch(in);
      const bool last = l == L - 1, even = (out & 1) == 0;
      const uint32_t x_base = outl::s_u32(ts + a.act_off[l] + sel * pitch + sel_col);
      const int n_ct = (out + 15) >> 4;
      auto tile = [&](float (&acc)[RT][4], const T* w, int ct, int k0, int nk) {
        if (even) forward_tile<true, RT, !RESIDENT>(acc, w, x_base + 2u * (uint32_t)k0, 16u * pitch, ct * 16 + 2 * g, nk, out, t);
        else forward_tile<false, RT, !RESIDENT>(acc, w, x_base + 2u * (uint32_t)k0, 16u * pitch, ct * 16 + 2 * g, nk, out, t);
      };
      auto finish = [&](const float (&acc)[RT][4], const T* bias, int ct) {
        const int n = ct * 16 + 2 * g;
        if (n >= out) return;
        const bool two = n + 1 < out;
        const float b0 = __bfloat162float(bias[n]), b1 = two ? __bfloat162float(bias[n + 1]) : 0.f;
#pragma unroll
        for (int h = 0; h < 2 * RT; ++h) {            // gradient row 2t + h % 2 of column tile h / 2
          const float v0 = acc[h >> 1][h & 1] + b0, v1 = acc[h >> 1][2 + (h & 1)] + b1;
          const int rr = 8 * (h >> 1) + 2 * t + (h & 1);
          if (last) {
            logits[rr * (out + 1) + n] = v0;
            if (two) logits[rr * (out + 1) + n + 1] = v1;
          } else {                                    // (the column behind an odd last one is padding and stays zero)
            *reinterpret_cast<uint32_t*>(ts + a.act_off[l + 1] + rr * mma_pitch(out) + n) =
                outl::pack_bf16(fmaxf(v0, 0.f), two ? fmaxf(v1, 0.f) : 0.f);
          }
        }
      };
      if (RESIDENT) {
        const T* w = reinterpret_cast<const T*>(W.take(l));
#pragma unroll 1
        for (int ct = warp; ct < n_ct; ct += NWM) {
          float acc[RT][4] = {};
          tile(acc, w, ct, 0, in);
          finish(acc, w + in * out, ct);
        }
      } else {
        // streamed weights come once, so a warp takes all its tiles along, chunk by chunk (1024 columns: 5 tiles per warp)
        constexpr int TP = 5;
        float acc[TP][RT][4] = {};
#pragma unroll 1
        for (int k0 = 0; k0 < in + 1; k0 += rpc) {
          const T* w = reinterpret_cast<const T*>(W.take(l));
          const int nk = min(rpc, in - k0);           // weight rows of this chunk (the bias row apart)
#pragma unroll
          for (int c = 0; c < TP; ++c)
            if (nk > 0 && warp + c * NWM < n_ct) tile(acc[c], w, warp + c * NWM, k0, nk);
          if (k0 + rpc >= in + 1) {                   // the last chunk ends with the bias row
#pragma unroll
            for (int c = 0; c < TP; ++c)
              if (warp + c * NWM < n_ct) finish(acc[c], w + nk * out, warp + c * NWM);
          }
          W.give(lane);
        }
      }
      if (last && tid < R) lab[tid] = label;
      sync_compute();
      if (!last) copy_rows<R>((T*)a.act[l + 1] + (size_t)r0 * out, ts + a.act_off[l + 1], mma_pitch(out), out, warp, lane);
    }
    // ------------------------------------------------------------------ loss and delta of the output layer
    {
      const int C = a.dims[L];
      T* dl = ts + a.out_off;
      for (int rr = warp; rr < R; rr += NWM) {
        const float* z = logits + rr * (C + 1);
        const float2 d = row_softmax<T>(a, lane < C ? z[lane] : 0.f, lane + 32 < C ? z[lane + 32] : 0.f, r0 + rr, lab[rr],
                                        sa_slot_weight(a.sa, a.S, t_round, slot), lane);
        T* gd = (T*)a.delta[L] + (size_t)(r0 + rr) * C;
        if (lane < C) { dl[rr * mma_pitch(C) + lane] = __float2bfloat16_rn(d.x); gd[lane] = __float2bfloat16_rn(d.x); }
        if (lane + 32 < C) { dl[rr * mma_pitch(C) + lane + 32] = __float2bfloat16_rn(d.y); gd[lane + 32] = __float2bfloat16_rn(d.y); }
      }
    }
    sync_compute();
    // ------------------------------------------------------------------ backward: tiles of 16 weight rows (= input columns)
    for (int l = L - 1; l >= (a.want_d0 ? 0 : 1); --l) {
      const int in = a.dims[l], out = a.dims[l + 1], rpc = a.rpc[l], pitch = mma_pitch(in);
      const T* dl = ts + (l == L - 1 ? a.out_off : a.act_off[l + 1]);
      const uint32_t d_base = outl::s_u32(dl + sel * mma_pitch(out) + sel_col);
      T* h = ts + a.act_off[l];
      const bool even = (out & 1) == 0;
      for (int k0 = 0; k0 < in + 1; k0 += rpc) {
        const T* w = reinterpret_cast<const T*>(W.take(l));
        const int nk = min(rpc, in - k0);
#pragma unroll 1
        for (int m0 = warp * 16; m0 < nk; m0 += NWM * 16) {
          float acc[RT][4] = {};
          const int mi = m0 + 2 * g;                  // this lane's weight rows: mi and mi + 1
          const T *wa = w + min(mi, nk - 1) * out, *wb = w + min(mi + 1, nk - 1) * out;
          if (even) backward_tile<true, RT, !RESIDENT>(acc, wa, wb, d_base, 16u * mma_pitch(out), out, t);
          else backward_tile<false, RT, !RESIDENT>(acc, wa, wb, d_base, 16u * mma_pitch(out), out, t);
          if (mi < nk) {                              // (the element behind an odd last one is padding and stays zero)
#pragma unroll
            for (int q = 0; q < 2 * RT; ++q) {
              uint32_t* hp = reinterpret_cast<uint32_t*>(h + (8 * (q >> 1) + 2 * t + (q & 1)) * pitch + k0 + mi);
              const float2 hv = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(hp));
              *hp = outl::pack_bf16(hv.x > 0.f ? acc[q >> 1][q & 1] : 0.f, hv.y > 0.f ? acc[q >> 1][2 + (q & 1)] : 0.f);
            }
          }
        }
        W.give(lane);
      }
      sync_compute();
      copy_rows<R>((T*)a.delta[l] + (size_t)r0 * in, h, pitch, in, warp, lane);
    }
  }
  rows_end(a, &gave_up);
}

// ---------------------------------------------------------------------------------------------
constexpr int GT = 32;                   // features x outputs per tile of grad_step_kernel
constexpr int GK = 64;                   // rows per pipeline step
constexpr int GP = GT + 4;               // shared-memory pitch
constexpr int MP = GT + 8;               // ... bf16 (five 16-byte units: ldmatrix reads without bank conflicts)

struct StepArgs {
  DevState* st;
  const RoundInfo* ri;
  const int* row_idx;
  const void* X; int gather;
  const void* act[ABS_MAX_LAYERS + 1];
  const void* delta[ABS_MAX_LAYERS + 1];
  float* master; void* ring; size_t d_pad;
  float lr;
  size_t w_off[ABS_MAX_LAYERS];
  int n_layers, dims[ABS_MAX_LAYERS + 1];
  int first_tile[ABS_MAX_LAYERS + 1];    // tiles of layer l: [first_tile[l], first_tile[l + 1])
  FastDiv nct[ABS_MAX_LAYERS];           // column tiles of layer l
  int Q, q_shift;                        // CTAs (a cluster, 2^q_shift) per tile: they share the rows
  int rows_cap;                          // rows the buffers hold
  // parts of the gradient left as per-chunk partial sums (the CNN's convolution blocks): blocks behind the tiles
  struct Region { const float* part; int len, chunk_rows; size_t off; int first_block; } region[2];
  int n_regions;
  cmma::FragMap frag;                    // region i = convolution block i: the weights also as operand fragments
};

// Four groups of 64 threads take 16 rows of a 64-row step each (fp32: 4 x 4 sums per thread, two 16-byte shared-memory
// reads for eight packed FMAs, two steps' rows in registers on the way; bf16: matrix instructions with the products added
// in fp32: the FMA form was bound by shared-memory reads; 201-133-10, 4096 rows: 60.7 -> 52.8 us a round, CNN 76.9 -> 75.5).  Groups are added in order, each CTA of a cluster
// hands its sums to the owner of their share (remote stores counted on the owner's barrier: a cluster barrier's release waits
// for all of a CTA's stores: 784-10 fp32, 1024 rows 13.74 -> 13.31 us a round, 59-10 10.39 -> 10.01), which adds them in order and applies Eq. 3.
// Bound by the chain of dependent latencies (indices, rows, exchange), so: the tile is found before the wait for the
// kernels in front, indices come with the round's sizes in one wave of loads, the weights a CTA updates are fetched
// before its sums exist.  784 x 10 fp32, 1024 rows: 6.4 -> 4 us
// with the row kernel's loads done likewise (19.3 -> 14.4 us a round); 300-123-57-7, 481 rows: 27.7 -> 18.3 us a round.
template <typename T, int DEPTH>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 2 : 3) grad_step_kernel(const __grid_constant__ StepArgs a) {
  constexpr bool MMA = sizeof(T) == 2;
  constexpr int P = MMA ? MP : GP;
  __shared__ __align__(16) T tiles[4][GK][P];        // two stages of inputs, two of deltas
  T (*As)[GK][P] = tiles, (*Ds)[GK][P] = tiles + 2;
  float (*red)[GT * GT] = reinterpret_cast<float (*)[GT * GT]>(tiles);     // sums of the four groups, at the end
  __shared__ __align__(16) float box[GT * GT];       // sums of this CTA's share: [CTA of the cluster][share]
  __shared__ uint64_t box_bar;                       // ... have arrived
  __shared__ int gave_up;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    tc::mbar_init(&box_bar, 1);
    gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tc::mbar_expect_tx(&box_bar, GT * GT * 4);
  }
  const int n_tiles = a.first_tile[a.n_layers];
  const int Q = a.Q, rank = (int)blockIdx.x & (Q - 1), tile = min((int)blockIdx.x >> a.q_shift, n_tiles - 1);
  int l = 0;
  while (tile >= a.first_tile[l + 1]) ++l;
  const int in = a.dims[l], out = a.dims[l + 1], lt = tile - a.first_tile[l];
  const int tm = a.nct[l].div(lt);
  const int m0 = tm * GT, n0 = (lt - tm * ((out + GT - 1) / GT)) * GT;
  const bool gather = l == 0 && a.gather;
  const T* A = (const T*)(l == 0 ? a.X : a.act[l]);
  const T* D = (const T*)a.delta[l + 1];
  const int m = m0 + lane, n = n0 + lane;
  grid_dependency_sync();
  DevState* st = a.st;
  const RoundInfo* ri = a.ri;
  // row 8 i + warp of a step is loaded by this warp; lane i < 8 holds its sample index
  auto load_idx = [&](int s) -> int {
    const int r = s * GK + 8 * lane + warp;
    return (lane < 8 && r < a.rows_cap) ? (gather ? a.row_idx[r] : r) : -1;
  };
  int ia = load_idx(rank), ib = DEPTH == 2 ? load_idx(rank + Q) : -1;
  const int status = st->status, diverged = ri->diverged, K = ri->K, n_rows = ri->n_rows, B = st->B, t = ri->t, S = st->S;
  if (status != ST_OK || diverged) return;
  const float step = __fdiv_rn(a.lr, (float)(K * B));
  const int slot = (t + 1) % (S + 1);
  T* dst = (T*)a.ring + (size_t)slot * a.d_pad;
  if ((int)blockIdx.x >= n_tiles * a.Q) {
    // region block: 32 parameters x 8 lanes over the chunks, fixed order
    float* part = &red[0][0];
    const int rb = (int)blockIdx.x - n_tiles * a.Q;
    const int q = (a.n_regions > 1 && rb >= a.region[1].first_block) ? 1 : 0;
    const StepArgs::Region& G = a.region[q];
    const int n_chunks = (n_rows + G.chunk_rows - 1) / G.chunk_rows;
    const int j = (rb - G.first_block) * 32 + lane;
    float acc = 0.f;
    if (j < G.len) {
#pragma unroll 8
      for (int c = warp; c < n_chunks; c += 8) acc += G.part[(size_t)c * G.len + j];
    }
    part[warp * 33 + lane] = acc;
    __syncthreads();
    if (warp == 0 && j < G.len) {
      float tot = 0.f;
#pragma unroll
      for (int c = 0; c < 8; ++c) tot += part[c * 33 + lane];
      const size_t e = G.off + (size_t)j;
      const float m = fmaf(-step, tot, a.master[e]);
      a.master[e] = m;
      stf(dst, e, m);
      if (sizeof(T) == 2 && a.frag.frag != nullptr) cmma::frag_store(a.frag, slot, q, j, __float2bfloat16_rn(m));
    }
    return;
  }
  const int n_steps = (n_rows + GK - 1) / GK;
  // Loads are unconditional (clamped addresses, selected when stored): a load and its conversion under a condition wait
  // for each other.  The mask has the rows that count; indices behind the round's rows are leftovers.
  struct Rows { T a[8], d[8]; unsigned ok; };
  const T zero = T(0.f), one = T(1.f);
  const T* Am = A + min(m, in - 1);
  const T* Dn = D + min(n, out - 1);
  auto load = [&](int s, int idx, Rows& p) {
    const int r0 = s * GK + warp;
    p.ok = __ballot_sync(0xffffffffu, idx >= 0 && r0 + 8 * lane < n_rows);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      p.a[i] = Am[(size_t)max(__shfl_sync(0xffffffffu, idx, i), 0) * in];
      p.d[i] = Dn[(size_t)min(r0 + 8 * i, a.rows_cap - 1) * out];
    }
  };
  Rows p0, p1;
  load(rank, ia, p0);
  if (DEPTH == 2) load(rank + Q, ib, p1);
  ia = load_idx(rank + DEPTH * Q);
  if (DEPTH == 2) ib = load_idx(rank + 3 * Q);
  // this CTA's share of the tile: elements e_0 + tid + 256 i
  const int share = (GT * GT) >> a.q_shift;
  float w[4];
  size_t o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int e = rank * share + tid + 256 * i, mm = m0 + e / GT, nn = n0 + e % GT;
    const bool mine = tid + 256 * i < share && mm <= in && nn < out;
    o[i] = mine ? a.w_off[l] + (size_t)mm * out + nn : (size_t)-1;
    w[i] = mine ? a.master[o[i]] : 0.f;
  }
  const int kg = tid >> 6, tx = tid & 7, ty = (tid >> 3) & 7;
  f32x2 acc[MMA ? 1 : 4][2] = {};                    // fp32: features 4 ty .., outputs 4 tx ..
  float acm[MMA ? 4 : 1][4] = {};                    // bf16: features 16 (warp & 1) .., four 8-output tiles
  auto one_step = [&](int s, int buf, int& idx, Rows& p) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const bool ok = (p.ok >> i & 1u) != 0;
      As[buf][8 * i + warp][lane] = m < in ? (ok ? p.a[i] : zero) : m == in ? one : zero;       // row `in`: the bias
      Ds[buf][8 * i + warp][lane] = ok && n < out ? p.d[i] : zero;
    }
    __syncthreads();
    if (s + DEPTH * Q < n_steps) {
      load(s + DEPTH * Q, idx, p);
      idx = load_idx(s + 2 * DEPTH * Q);
    }
    if constexpr (MMA) {
      uint32_t af[4], b[4];
      const int k0 = kg * 16, x = lane & 7, h = lane >> 3;
      outl::ldsm4t(outl::s_u32(&As[buf][k0 + (h >> 1) * 8 + x][(warp & 1) * 16 + (h & 1) * 8]), af);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        outl::ldsm4t(outl::s_u32(&Ds[buf][k0 + (h & 1) * 8 + x][16 * q + (h >> 1) * 8]), b);
        outl::mma16816_rn(acm[2 * q], af, b[0], b[1]);
        outl::mma16816_rn(acm[2 * q + 1], af, b[2], b[3]);
      }
    } else {
#pragma unroll
      for (int k = 0; k < GK / 4; ++k) {
        const float4 av = *reinterpret_cast<const float4*>(&As[buf][kg * (GK / 4) + k][4 * ty]);
        const ulonglong2 dv = *reinterpret_cast<const ulonglong2*>(&Ds[buf][kg * (GK / 4) + k][4 * tx]);
        const f32x2 p[4] = {lsqp::pack2(av.x, av.x), lsqp::pack2(av.y, av.y), lsqp::pack2(av.z, av.z), lsqp::pack2(av.w, av.w)};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          lsqp::ffma2(acc[i][0], p[i], dv.x);
          lsqp::ffma2(acc[i][1], p[i], dv.y);
        }
      }
    }
  };
#pragma unroll 1
  for (int s = rank; s < n_steps; s += 2 * Q) {
    one_step(s, 0, ia, p0);
    if (s + Q < n_steps) one_step(s + Q, 1, DEPTH == 2 ? ib : ia, DEPTH == 2 ? p1 : p0);
  }
  if (Q > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");       // (peers have started: see below)
  __syncthreads();
  if constexpr (MMA) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        *reinterpret_cast<float2*>(&red[kg][(16 * (warp & 1) + (lane >> 2) + 8 * h) * GT + 8 * q + 2 * (lane & 3)]) = make_float2(acm[q][2 * h], acm[q][2 * h + 1]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      *reinterpret_cast<ulonglong2*>(&red[kg][(4 * ty + i) * GT + 4 * tx]) = make_ulonglong2(acc[i][0], acc[i][1]);
  }
  __syncthreads();
  if (Q > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  {
    const int e = 4 * tid;                           // (a share is 128 elements or more)
    float4 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = *reinterpret_cast<const float4*>(&red[k][e]);
    const float4 s = make_float4((v[0].x + v[1].x) + (v[2].x + v[3].x), (v[0].y + v[1].y) + (v[2].y + v[3].y),
                                 (v[0].z + v[1].z) + (v[2].z + v[3].z), (v[0].w + v[1].w) + (v[2].w + v[3].w));
    if (Q > 1) {
      const uint32_t owner = (uint32_t)(e >> (10 - a.q_shift));       // (GT x GT = 2^10)
      tc::st_async4(tc::map_to_cta(tc::smem_u32(box + rank * share + (e & (share - 1))), owner), s, tc::map_to_cta(tc::smem_u32(&box_bar), owner));
      tc::wait_cluster(&box_bar, 0u, &gave_up);
      if (__syncthreads_or(gave_up)) {               // ends the run; all threads alike, so that no share is half applied
        tc::leave_cluster();
        // not st->status: a cluster that starts later must find the same status in all of its CTAs, or one of them leaves and
        // the others store to it.  The next control step and the host take the run for ended by this word.
        if (tid == 0) st->timeout_where = 500;
        return;
      }
    } else {
      *reinterpret_cast<float4*>(box + e) = s;
      __syncthreads();
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (o[i] == (size_t)-1) continue;
    float g = box[tid + 256 * i];
    if (Q > 1)
#pragma unroll
      for (int q = 1; q < 8; ++q)
        if (q < Q) g += box[q * share + tid + 256 * i];
    const float m_new = fmaf(-step, g, w[i]);
    a.master[o[i]] = m_new;
    stf(dst, o[i], m_new);
  }
}

}  // namespace rnet
}  // namespace absb
