// Local SGD inside a job (Eq. 2 with U > 1): a cluster of CTAs per selected worker (local_cluster_kernel), or one CTA
// (local_sgd_kernel: steps whose rows do not fit a cluster, tiny steps of many workers; see cluster_plan), runs the worker's U
// minibatch steps one after the other on the worker's own copy of the model, which starts at the version the
// worker holds (its ring slot) and lives in shared memory as fp32 (bf16 configurations compute each
// step with the bf16 rounding of that copy, as their tensor-core paths must).  Step u draws its minibatch from
// Philox blocks (n, j, 1, u * ceil(B/4) + b/4).  The upload is the sum over the steps of the
// per-sample gradient sums, G = (B / eta) (w^{.,0} - w^{.,U}), and the average of the U mean
// minibatch losses (Algorithm 1, last worker line); Eq. 3 then reads the K uploads like the
// partial sums of the U = 1 path.  Single-layer models only (least squares, soft-max regression
// with at most 16 classes): their parameter vector fits in shared memory twice.
// The chains of different workers are independent but each is strictly sequential, so the kernels
// are latency-bound by design; a step is B short dot products and one rank-B update.
#pragma once
#include <algorithm>

#include "common.cuh"
#include "ctl.cuh"
#include "narrow.cuh"
#include "lsqpipe.cuh"

namespace absb {
namespace local {

constexpr int MAX_PARAMS = 12288;     // fp32 parameters of the local model (twice in shared memory)
constexpr int MAX_C = 16;
constexpr int MAX_BC = 8192;          // B * C deltas of one step
constexpr int NT_MAX = 1024;          // threads per CTA: only K CTAs run, so a large model gets wide CTAs
inline int threads_for(int n_par) { return n_par >= 2048 ? NT_MAX : 256; }

struct Args {
  DevState* st;
  RoundInfo* ri;
  const int* sel; const int* job; const int* sel_tau;
  const int2* shard;                  // [W] first sample and length of each worker's shard
  const void* X; const void* y;       // y: float targets (least squares) or int labels
  const void* ring; size_t slot_stride;
  float* loss;                        // [W] uploaded loss of each selected worker
  float* G;                           // [W][slot_stride] uploaded gradient sums
  int lsq;                            // 1: least squares (C = 1, no bias)
  int in, C, U;
  float lr;
};

inline size_t smem_bytes(int n_par, int B, int C) {
  return sizeof(float) * ((size_t)2 * n_par + (size_t)B * C + B + 64) + sizeof(int) * (size_t)B;
}

// (d0, d1) += x * (w0, w1) as one packed binary32 FMA (each lane rounds like a scalar fma).
__device__ __forceinline__ void ffma2_bcast(float& d0, float& d1, float x, const float2 w) {
  asm("{\n\t.reg .b64 ra, rb, rc;\n\tmov.b64 ra, {%2, %2};\n\tmov.b64 rb, {%3, %4};\n\tmov.b64 rc, {%0, %1};\n\t"
      "fma.rn.f32x2 rc, ra, rb, rc;\n\tmov.b64 {%0, %1}, rc;\n\t}"
      : "+f"(d0), "+f"(d1) : "f"(x), "f"(w.x), "f"(w.y));
}

template <typename T>
__global__ void __launch_bounds__(NT_MAX) local_sgd_kernel(Args a) {
  grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char loc_raw[];
  DevState* st = a.st;
  RoundInfo* ri = a.ri;
  if (st->status != ST_OK) return;
  const int i = blockIdx.x;
  if (i >= ri->K) return;
  const int B = st->B, in = a.in, C = a.C, U = a.U, W = st->W;
  const int n_w = in * C, n_par = a.lsq ? in : n_w + C;
  float* wl = reinterpret_cast<float*>(loc_raw);        // [n_par] local model
  float* gs = wl + n_par;                                // [n_par] sum of the steps' gradient sums
  float* dl = gs + n_par;                                // [B][C] deltas of the step (residuals for least squares)
  float* rl = dl + (size_t)B * C;                        // [B] sample losses of the step
  float* red = rl + B;                                   // [64]
  int* sidx = reinterpret_cast<int*>(red + 64);          // [B] sample indices of the step
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int NT = (int)blockDim.x;
  const bool even_c = (C & 1) == 0;
  const int wn = a.sel[i], jb = a.job[wn];
  const int slot = (ri->t - a.sel_tau[i]) % (st->S + 1);
  const T* w0 = (const T*)a.ring + (size_t)slot * a.slot_stride;
  const T* X = (const T*)a.X;
  const i64 M = st->n_samples;
  const i64 lo = ((i64)wn * M) / W, hi = ((i64)(wn + 1) * M) / W;
  const u64 len = (u64)(hi - lo);
  const uint32_t key0 = st->key0, key1 = st->key1;
  const int nblk = (B + 3) >> 2;
  const float step = __fdiv_rn(a.lr, (float)B);
  for (int p = tid; p < n_par; p += NT) { wl[p] = ldf(w0, p); gs[p] = 0.f; }
  float loss_sum = 0.f;
  for (int u = 0; u < U; ++u) {
    for (int blk = tid; blk < nblk; blk += NT) {
      uint32_t w4[4];
      philox4x32_10((uint32_t)wn, (uint32_t)jb, 1u, (uint32_t)(u * nblk + blk), key0, key1, w4);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (blk * 4 + q < B) sidx[blk * 4 + q] = (int)lo + (int)(((u64)w4[q] * len) >> 32);
    }
    __syncthreads();
    // ---- forward at the local model: one warp per row
    for (int b = warp; b < B; b += NT / 32) {
      const T* x = X + (size_t)sidx[b] * in;
      float acc[MAX_C];
#pragma unroll
      for (int c = 0; c < MAX_C; ++c) acc[c] = 0.f;
#pragma unroll 8
      for (int m = lane; m < in; m += 32) {
        const float xv = ldf(x, m);
        if (even_c) {                 // class pairs: one 8-byte shared-memory read and one packed FMA per pair
          const float2* wp = reinterpret_cast<const float2*>(wl + m * C);
#pragma unroll
          for (int c = 0; c < MAX_C; c += 2)
            if (c < C) {
              float2 w = wp[c >> 1];
              w.x = round_store(w.x, (const T*)nullptr);
              w.y = round_store(w.y, (const T*)nullptr);
              ffma2_bcast(acc[c], acc[c + 1], xv, w);
            }
        } else {
#pragma unroll
          for (int c = 0; c < MAX_C; ++c)
            if (c < C) acc[c] = fmaf(xv, round_store(wl[m * C + c], (const T*)nullptr), acc[c]);
        }
      }
#pragma unroll
      for (int c = 0; c < MAX_C; ++c)
        if (c < C) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
        }
      if (a.lsq) {
        const float r = acc[0] - ((const float*)a.y)[sidx[b]];
        if (lane == 0) { dl[b] = r; rl[b] = 0.5f * r * r; }
      } else {
        const int y = ((const int*)a.y)[sidx[b]];
        float zmax = -3.0e38f, zy = 0.f;
#pragma unroll
        for (int c = 0; c < MAX_C; ++c)
          if (c < C) { acc[c] += round_store(wl[n_w + c], (const T*)nullptr); zmax = fmaxf(zmax, acc[c]); if (c == y) zy = acc[c]; }
        float se = 0.f;
#pragma unroll
        for (int c = 0; c < MAX_C; ++c)
          if (c < C) { acc[c] = expf(acc[c] - zmax); se += acc[c]; }
        const float inv = 1.f / se;
        float mine = 0.f;
#pragma unroll
        for (int c = 0; c < MAX_C; ++c)
          if (c == lane) mine = acc[c] * inv - (c == y ? 1.f : 0.f);
        // a delta is a stored quantity of the bf16 configurations: rounded like every other delta
        if (lane < C) dl[b * C + lane] = round_store(mine, (const T*)nullptr);
        if (lane == 0) rl[b] = logf(se) - (zy - zmax);
      }
    }
    __syncthreads();
    // ---- mean loss of the step (fixed order: strided partial sums, then a shuffle tree, then the warps in order)
    {
      float part = 0.f;
      for (int b = tid; b < B; b += NT) part += rl[b];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      if (lane == 0) red[warp] = part;
    }
    // ---- gradient sum of the step, one feature per thread (all classes), and the local step
    for (int m = tid; m < in; m += NT) {
      float acc[MAX_C];
#pragma unroll
      for (int c = 0; c < MAX_C; ++c) acc[c] = 0.f;
#pragma unroll 8
      for (int b = 0; b < B; ++b) {
        const float xv = ldf(X, (size_t)sidx[b] * in + m);
        if (even_c) {
          const float2* dp = reinterpret_cast<const float2*>(dl + b * C);
#pragma unroll
          for (int c = 0; c < MAX_C; c += 2)
            if (c < C) ffma2_bcast(acc[c], acc[c + 1], xv, dp[c >> 1]);
        } else {
#pragma unroll
          for (int c = 0; c < MAX_C; ++c)
            if (c < C) acc[c] = fmaf(xv, dl[b * C + c], acc[c]);
        }
      }
#pragma unroll
      for (int c = 0; c < MAX_C; ++c)
        if (c < C) {
          gs[m * C + c] += acc[c];
          wl[m * C + c] = fmaf(-step, acc[c], wl[m * C + c]);
        }
    }
    if (!a.lsq && tid < C) {
      float acc = 0.f;
      for (int b = 0; b < B; ++b) acc += dl[b * C + tid];
      gs[n_w + tid] += acc;
      wl[n_w + tid] = fmaf(-step, acc, wl[n_w + tid]);
    }
    __syncthreads();
    if (tid == 0) {
      float tot = 0.f;
      for (int q = 0; q < NT / 32; ++q) tot += red[q];
      loss_sum += __fdiv_rn(tot, (float)B);
    }
  }
  float* g = a.G + (size_t)i * a.slot_stride;
  const float sa = st->sa_penalty ? sa_weight(a.sel_tau[i]) : 1.f;   // staleness-aware step size: weight of the upload in Eq. 3
  for (int p = tid; p < n_par; p += NT) g[p] = gs[p] * sa;
  if (tid == 0) {
    const float loss = __fdiv_rn(loss_sum, (float)U);
    a.loss[i] = loss;
    if (!isfinite(loss)) ri->diverged = 1;
  }
}

// ---------------------------------------------------------------------------------------------
// The same local steps with a CLUSTER of Q CTAs per selected worker.  The one-CTA kernel above uses K of
// 148 SMs and walks every row twice through L2 with scalar loads; here CTA q of the cluster owns the features
// [q F, (q + 1) F) of the worker's model, which stay in its shared memory for the whole job, and the soft-max of the
// rows [q RQ, (q + 1) RQ) of every step:
//   - the slice of a step's B rows is copied once (asynchronously, one step ahead: a job's minibatches are known
//     from the counter-based generator) and serves both the forward pass and the gradient,
//   - each CTA sends its partial logits of a row to the row's owner and the owner sends the row's deltas to every CTA,
//     both as remote stores that complete on the receiver's mbarrier (st.async; launched as a cluster only, Q > 1): no
//     cluster barrier inside a step,
//   - the copies of the next rows and the draws of the step after that are issued while the exchange is on its way.
// A step is bound by its chain of phases, each of dependent shared-memory reads: 784 -> 10, 16 workers x 64 rows, cycles at 1.96
// GHz: partial logits 1930, sum and send 720, soft-max with the wait for the logits 1810, copies of the next rows 1190, wait for
// the deltas 160, gradient 1750, local step 1390, barriers 310: 9300.  With a cluster barrier and remote loads (2400 cycles: its
// release waits for all stores) and bulk copies of the row slices by one warp that also took part in the soft-max (64 copies:
// 6900 cycles) a step took 14000 (a round of ten steps 91.7 -> 73.1 us; 20 to 64 workers 74 us and 143 us; 2 to 16 classes, 87
// to 687 features 1.12 to 1.43 times as fast).  Of the kernel's 66 us the start-up (job, draws, model slice, first rows, cluster
// start) is 5 and the upload 1.4; the steps are 46 us in 14 of the 16 clusters, 53 and 59 in the two whose CTAs share SMs.
// Both buffers of the exchange are used again in the next step.  A CTA sends step u + 1's logits after it has all deltas of
// step u, so every owner has read its logits of step u; an owner sends step u + 1's deltas after every CTA has sent its
// logits of step u + 1, that is after the gradient of step u.
struct Geo {
  int Q;        // CTAs per worker (cluster width)
  int F;        // features per CTA (a multiple of 8)
  int RQ;       // rows of a step per CTA (soft-max)
  int pitch;    // elements between rows of the staged slices: an odd number of 16-byte groups, so that 16-byte
                // reads of one column group by consecutive rows fall into different banks
  int nbuf;     // row buffers (2: the next step's rows are copied during this one)
  int PZ, PG;   // partial sums per row (forward) / per feature group (gradient) inside a CTA
};

constexpr int CL_NT = 256;
template <typename T> __host__ __device__ constexpr int group_elems() { return 16 / (int)sizeof(T); }

// CTAs of the cluster kernel per SM: by the registers of one group's sums (ge elements x CP classes)
__host__ __device__ constexpr int cluster_ctas_per_sm(int ge, int CP) { return ge * CP < 64 ? 2 : 1; }

inline size_t cluster_smem(const Geo& g, int esz, int B, int CP) {
  const size_t zp = std::max((size_t)g.PZ * B * CP, (size_t)g.PG * g.F * CP);
  return (size_t)g.nbuf * B * g.pitch * esz +
         4 * ((size_t)(esz == 2 ? 3 : 2) * g.F * CP + zp + ((size_t)g.Q * g.RQ + B) * CP + (size_t)4 * round_up(B, 4) + 2 * round_up(g.RQ, 4) + 2 * 16) + 64;
}

// Cluster width and staging for a model of `in` features, C classes, W workers of which n run at once (K^0 where K is
// fixed, else all); Q = 0: the one-CTA kernel runs.
// Q: as many CTAs as the chip holds twice over when every worker is selected, slices of at least 32 features.
// The one-CTA kernel stays where the rows of a step do not fit a cluster's shared memory, and on batches of a few rows once
// the clusters of n workers take more than one wave: for models below 2048 parameters (its CTAs are 256 threads there, and
// several share an SM) and for large ones whose clusters of two take two partial waves.  us a round, one-CTA / cluster,
// U = 10, all workers selected: 64 -> 10 bf16, 1024 workers, 4 rows 176 / 282, 8 rows 204 / 292, 12 rows 274 / 293; 200
// workers, 6 rows 79 / 89, 8 rows 83 / 86, 10 rows 116 / 90; 64 -> 1 fp32, 512 workers, 4 rows 64 / 78, 8 rows 76 / 82, 12 rows
// 91 / 84; 784 -> 10 bf16, 100 workers, 8 rows 131 / 146, 10 rows 144 / 156, 12 rows 148 / 156, 14 rows 165 / 166, 16 rows 167 /
// 162; 148 workers, 8 rows 136 / 152, 12 rows 152 / 163; 784 -> 10 fp32, 145 workers, 64 rows 363 / 343.
inline Geo cluster_plan(int in, int C, int n_par, int B, int W, int n, int esz) {
  const int CP = round_up(C, 4), ge = 16 / esz;
  const int wave = PLAN_SMS * cluster_ctas_per_sm(ge, CP);
  auto geo = [&](int Q, int nbuf) {
    Geo g;
    g.Q = Q;
    g.F = round_up((in + Q - 1) / Q, 8);
    g.RQ = (B + Q - 1) / Q;
    const int groups = g.F / ge;
    g.pitch = (groups | 1) * ge;
    g.nbuf = nbuf;
    const int pairs = (B + 1) / 2;
    g.PZ = std::max(1, std::min(std::min(CL_NT / std::max(1, pairs), 16), groups));
    // (32 KB of partial gradients: two CTAs have to fit an SM, since the chip has no room for 16 clusters of eight with an SM
    // per CTA: with 48 KB the 16 workers above took two waves, 103 instead of 65 us)
    g.PG = std::max(1, std::min(std::min(CL_NT / groups, 8192 / (g.F * CP)), std::min(16, B / 4)));
    return g;
  };
  int first = 8;
  while (first > 1 && (W * first > 2 * PLAN_SMS || in / first < 32)) first /= 2;
  Geo none = geo(1, 1);
  none.Q = 0;
  if (n_par < 2048 && (B <= 8 ? n * first > wave : B <= 12 && wave == PLAN_SMS && n * first > 2 * wave)) return none;
  if (n_par > 6000 && B <= 12 && first == 2 && n * first > wave) return none;
  for (int nbuf = 2; nbuf >= 1; --nbuf)
    for (int Q = first; Q <= 8; Q *= 2) {
      const Geo g = geo(Q, nbuf);
      if (cluster_smem(g, esz, B, CP) <= 220 * 1024) return g;
    }
  return none;
}

__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ float4 add4(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }

// one 16-byte group of stored values as binary32
__device__ __forceinline__ void load_group(const float* p, float (&v)[4]) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void load_group(const __nv_bfloat16* p, float (&v)[8]) { load8(p, v); }

// CP: class count rounded up to a multiple of 4 (padded classes have zero weights and zero deltas)
template <typename T, int CP>
__global__ void __launch_bounds__(CL_NT, cluster_ctas_per_sm(group_elems<T>(), CP)) local_cluster_kernel(Args a, Geo geo) {
  grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char loc_raw[];
  using lsqp::f32x2;
  constexpr int NT = CL_NT, GE = group_elems<T>(), C4 = CP / 4;
  DevState* st = a.st;
  RoundInfo* ri = a.ri;
  const int Q = geo.Q, F = geo.F, RQ = geo.RQ, pitch = geo.pitch, PZ = geo.PZ, PG = geo.PG;
  const int i = (int)blockIdx.x / Q;                 // (< W: its entries exist whether or not it is selected)
  const int status = st->status, K = ri->K, t_round = ri->t, B = st->B, S = st->S, wn = a.sel[i], tau = a.sel_tau[i];
  const uint32_t key0 = st->key0, key1 = st->key1;
  if (status != ST_OK || i >= K) return;             // same decision in every CTA of the cluster
  const int rank = Q > 1 ? (int)tc::cluster_rank() : 0;
  const int in = a.in, C = a.C, U = a.U;
  const int n_w = in * C;
  const int m0 = rank * F, nf = max(0, min(F, in - m0));     // this CTA's features
  const int b_own = rank * RQ, n_own = max(0, min(RQ, B - b_own));      // rows whose soft-max it forms
  const int groups = F / GE, n_g = F * C4;           // 16-byte row groups; float4s of the slice's gradient
  const int Br = round_up(B, 4), Rr = round_up(RQ, 4);
  T* xs = reinterpret_cast<T*>(loc_raw);                                     // [nbuf][B][pitch]
  float* wl = reinterpret_cast<float*>(xs + (size_t)geo.nbuf * B * pitch);   // [F][CP] local model
  float* wq = sizeof(T) == 2 ? wl + (size_t)F * CP : wl;                     // ... as the forward pass reads it (bf16 values)
  float4* gs = reinterpret_cast<float4*>(wq + (size_t)F * CP);               // [GE * C4][groups] sum of the steps' gradient sums
  float* zp = reinterpret_cast<float*>(gs + n_g);                            // partial logits / partial gradients
  float* zin = zp + max((size_t)PZ * B * CP, (size_t)PG * F * CP);           // [Q][RQ][CP] the CTAs' partial logits of this CTA's rows
  float* dl = zin + (size_t)Q * RQ * CP;                                     // [B][CP] deltas, from the rows' owners
  float* rl = dl + (size_t)B * CP;                                           // [B] sample losses (first CTA)
  float* bs = rl + Br;                                                       // [16] bias, [16] its gradient sum
  int* sidx = reinterpret_cast<int*>(bs + 32);                               // [3][B] sample indices by step mod 3
  uint32_t* ys = reinterpret_cast<uint32_t*>(sidx + 3 * Br);                 // [2][RQ] targets / labels by step parity
  __shared__ uint64_t bar_z, bar_d;                  // logits / deltas of the step have arrived
  __shared__ int gave_up;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool last_warp = warp == NT / 32 - 1;
  const int jb = a.job[wn];
  const int2 shard = a.shard[wn];
  const int slot = (t_round - tau) % (S + 1);
  const T* w0 = (const T*)a.ring + (size_t)slot * a.slot_stride;
  const T* X = (const T*)a.X + m0;
  const int nblk = (B + 3) >> 2;
  const float step = __fdiv_rn(a.lr, (float)B);

  auto draw = [&](int u) {                           // sample indices of step u (last warp)
    int* dst = sidx + (u % 3) * Br;
    for (int blk = lane; blk < nblk; blk += 32) {
      uint32_t w4[4];
      philox4x32_10((uint32_t)wn, (uint32_t)jb, 1u, (uint32_t)(u * nblk + blk), key0, key1, w4);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (blk * 4 + q < B) dst[blk * 4 + q] = shard.x + (int)__umulhi(w4[q], (uint32_t)shard.y);
    }
  };
  // this CTA's slice of step u's rows, in the widest pieces the rows' starts allow (F is a multiple of 8), and the labels of
  // its own rows
  const int row_bytes_mod = (int)(((size_t)in * sizeof(T)) % 16);
  const int per = row_bytes_mod == 0 ? nf / GE : row_bytes_mod % 4 == 0 ? nf * (int)sizeof(T) / 4 : nf;
  const FastDiv by_per(max(per, 1));
  auto fetch = [&](int u) {
    const int* idx = sidx + (u % 3) * Br;
    T* dst = xs + (size_t)(u % geo.nbuf) * B * pitch;
    if (row_bytes_mod == 0) {
#pragma unroll 2
      for (int e = tid; e < B * per; e += NT) {
        const int b = by_per.div(e), v = (e - b * per) * GE;
        cp_async16(dst + b * pitch + v, X + (size_t)idx[b] * in + v);
      }
    } else if (row_bytes_mod % 4 == 0) {
      constexpr int E4 = 4 / (int)sizeof(T);         // (F and here `in` are even for 2-byte elements)
#pragma unroll 2
      for (int e = tid; e < B * per; e += NT) {
        const int b = by_per.div(e), v = (e - b * per) * E4;
        cp_async4(dst + b * pitch + v, X + (size_t)idx[b] * in + v);
      }
    } else {
      for (int e = tid; e < B * per; e += NT) {
        const int b = by_per.div(e), v = e - b * per;
        dst[b * pitch + v] = X[(size_t)idx[b] * in + v];
      }
    }
    for (int b = tid; b < n_own; b += NT) cp_async4(ys + (u & 1) * Rr + b, (const uint32_t*)a.y + idx[b_own + b]);
  };

  if (tid == 0) {
    tc::mbar_init(&bar_z, 1);
    tc::mbar_init(&bar_d, 1);
    gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (last_warp) {
    draw(0);
    if (U > 1) draw(1);
  }
  // columns behind the slice's features are read by the 16-byte groups but never copied: zero in every buffer
  for (int r = warp; r < geo.nbuf * B; r += NT / 32)
    for (int v = nf + lane; v < pitch; v += 32) stf(xs, (size_t)r * pitch + v, 0.f);
#pragma unroll 4
  for (int e = tid; e < F * CP; e += NT) {
    const int m = e / CP, c = e - m * CP;
    const float w = (m < nf && c < C) ? ldf(w0, (size_t)(m0 + m) * C + c) : 0.f;    // a stored model is already rounded
    wl[e] = w;
    wq[e] = w;
  }
  for (int e = tid; e < n_g; e += NT) gs[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (tid < 16) {
    bs[tid] = (!a.lsq && tid < C) ? ldf(w0, (size_t)n_w + tid) : 0.f;
    bs[16 + tid] = 0.f;
  }
  __syncthreads();
  fetch(0);
  float loss_sum = 0.f;                              // last warp of the first CTA
  if (Q > 1) tc::cluster_sync_all();                 // peers have started: their barriers and shared memory exist

  const uint32_t bar_z_a = tc::smem_u32(&bar_z), bar_d_a = tc::smem_u32(&bar_d);
  const uint32_t zin_a = tc::smem_u32(zin + (size_t)rank * RQ * CP), dl_a = tc::smem_u32(dl);
  // ---- logits, loss, deltas of this CTA's rows: four lanes per row, four classes each
  auto softmax = [&](int par, uint32_t parity) {
    if (warp * 8 >= n_own) return;
    if (Q > 1) tc::wait_cluster(&bar_z, parity, &gave_up);
#pragma unroll 1
    for (int b0 = 0; b0 + warp * 8 < n_own; b0 += NT / 4) {
      const int b = b0 + (tid >> 2), l = tid & 3;    // row b_own + b
      const bool have = b < n_own && l < C4;
      float z[4] = {0.f, 0.f, 0.f, 0.f};
      if (have) {
        const float* mine = zin + (size_t)b * CP + 4 * l;
        float4 p[8];                                 // the cluster's partial logits of these classes
#pragma unroll
        for (int q = 0; q < 8; ++q)
          p[q] = q < Q ? *reinterpret_cast<const float4*>(mine + (size_t)q * RQ * CP) : make_float4(0.f, 0.f, 0.f, 0.f);
        float4 s = p[0];
#pragma unroll
        for (int q = 1; q < 8; ++q) s = add4(s, p[q]);
        z[0] = s.x; z[1] = s.y; z[2] = s.z; z[3] = s.w;
      }
      float d[4] = {0.f, 0.f, 0.f, 0.f}, loss;
      const uint32_t yb = b < n_own ? ys[par * Rr + b] : 0u;
      if (a.lsq) {
        const float r = z[0] - __uint_as_float(yb);
        loss = 0.5f * r * r;
        if (l == 0) d[0] = r;
      } else {
        const int y = (int)yb;
        float zy = 0.f, se = 0.f;
        // padded classes: exp(NO_CLASS - max) = 0, and their delta is 0
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          z[k] = 4 * l + k < C ? z[k] : NO_CLASS;
          zy = 4 * l + k == y ? z[k] : zy;
        }
        float zmax = fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3]));
        zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, 1));
        zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, 2));
#pragma unroll
        for (int k = 0; k < 4; ++k) z[k] = expf(z[k] - zmax);
        se = (z[0] + z[1]) + (z[2] + z[3]);
        se += __shfl_xor_sync(0xffffffffu, se, 1);
        se += __shfl_xor_sync(0xffffffffu, se, 2);
        zy += __shfl_xor_sync(0xffffffffu, zy, 1);
        zy += __shfl_xor_sync(0xffffffffu, zy, 2);
        const float inv = 1.f / se;
        // a delta is a stored quantity of the bf16 configurations: rounded like every other delta
#pragma unroll
        for (int k = 0; k < 4; ++k) d[k] = round_store(z[k] * inv - (4 * l + k == y ? 1.f : 0.f), (const T*)nullptr);
        loss = logf(se) - (zy - zmax);
      }
      if (have) {
        const uint32_t off = (uint32_t)(((b_own + b) * CP + 4 * l) * 4);
        const float4 dv = make_float4(d[0], d[1], d[2], d[3]);
        if (Q > 1) {
#pragma unroll
          for (int q = 0; q < 8; ++q)
            if (q < Q) tc::st_async4(tc::map_to_cta(dl_a + off, (uint32_t)q), dv, tc::map_to_cta(bar_d_a, (uint32_t)q));
          if (l == 0) tc::st_async1(tc::map_to_cta(tc::smem_u32(rl + b_own + b), 0u), loss, tc::map_to_cta(bar_d_a, 0u));
        } else {
          *reinterpret_cast<float4*>(dl + (size_t)b * CP + 4 * l) = dv;
          if (l == 0) rl[b] = loss;
        }
      }
    }
  };

  const int n_pairs = (B + 1) / 2;
  const FastDiv by_pairs(n_pairs), by_groups(groups), by_rq(RQ);
  for (int u = 0; u < U; ++u) {
    const uint32_t parity = (uint32_t)u & 1u;
    if (Q > 1 && tid == 0) {                         // what this step's exchange brings
      tc::mbar_expect_tx(&bar_z, (uint32_t)(Q * n_own * CP * 4));
      tc::mbar_expect_tx(&bar_d, (uint32_t)(B * CP * 4 + (rank == 0 ? B * 4 : 0)));
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();                                 // rows of step u are here; the previous step is done with everything
    const T* xb = xs + (size_t)(u % geo.nbuf) * B * pitch;
    // ---- partial logits of this slice: item = (row pair, every PZ-th column group)
    for (int it = tid; it < n_pairs * PZ; it += NT) {
      const int part = by_pairs.div(it), r0 = it - part * n_pairs, r1 = r0 + n_pairs;
      const T* x0 = xb + r0 * pitch;
      const T* x1 = xb + min(r1, B - 1) * pitch;
      f32x2 z0[CP / 2], z1[CP / 2];
#pragma unroll
      for (int c = 0; c < CP / 2; ++c) z0[c] = z1[c] = 0ull;
      for (int g = part; g < groups; g += PZ) {
        float v0[GE], v1[GE];
        load_group(x0 + g * GE, v0);
        load_group(x1 + g * GE, v1);
        const float* w = wq + g * (GE * CP);
#pragma unroll
        for (int j = 0; j < GE; ++j) {
          const f32x2 p0 = lsqp::pack2(v0[j], v0[j]), p1 = lsqp::pack2(v1[j], v1[j]);
#pragma unroll
          for (int c = 0; c < C4; ++c) {
            const ulonglong2 ww = *reinterpret_cast<const ulonglong2*>(w + j * CP + 4 * c);
            lsqp::ffma2(z0[2 * c], p0, ww.x);
            lsqp::ffma2(z0[2 * c + 1], p0, ww.y);
            lsqp::ffma2(z1[2 * c], p1, ww.x);
            lsqp::ffma2(z1[2 * c + 1], p1, ww.y);
          }
        }
      }
      float* o = zp + ((size_t)part * B + r0) * CP;
#pragma unroll
      for (int c = 0; c < C4; ++c) {
        *reinterpret_cast<ulonglong2*>(o + 4 * c) = make_ulonglong2(z0[2 * c], z0[2 * c + 1]);
        if (r1 < B) *reinterpret_cast<ulonglong2*>(o + (size_t)n_pairs * CP + 4 * c) = make_ulonglong2(z1[2 * c], z1[2 * c + 1]);
      }
    }
    __syncthreads();
    for (int e = tid; e < B * C4; e += NT) {         // partial sums in order; the first CTA adds the bias
      float4 z = reinterpret_cast<const float4*>(zp)[e];
#pragma unroll 8
      for (int p = 1; p < PZ; ++p) z = add4(z, reinterpret_cast<const float4*>(zp + (size_t)p * B * CP)[e]);
      const int b = e / C4;
      if (rank == 0) {
        const float4 bq = reinterpret_cast<const float4*>(bs)[e - b * C4];
        z = add4(z, make_float4(round_store(bq.x, (const T*)nullptr), round_store(bq.y, (const T*)nullptr),
                                round_store(bq.z, (const T*)nullptr), round_store(bq.w, (const T*)nullptr)));
      }
      if (Q == 1) {
        reinterpret_cast<float4*>(zin)[e] = z;
        continue;
      }
      const int owner = by_rq.div(b);                // element e of the step is element e - owner RQ C4 of its owner's
      tc::st_async4(tc::map_to_cta(zin_a + (uint32_t)(e - owner * RQ * C4) * 16u, (uint32_t)owner), z, tc::map_to_cta(bar_z_a, (uint32_t)owner));
    }
    // the next rows are fetched while the exchange is on its way (behind the soft-max by the warps that form it)
    if (Q == 1) __syncthreads();
    const bool early = warp * 8 < n_own, ahead = geo.nbuf == 2 && u + 1 < U;
    if (ahead && !early) fetch(u + 1);
    softmax(u & 1, parity);
    if (ahead && early) fetch(u + 1);
    if (last_warp && u + 2 < U) draw(u + 2);
    if (Q > 1) tc::wait_cluster(&bar_d, parity, &gave_up);
    else __syncthreads();
    // ---- gradient of this slice: item = (column group, every PG-th row)
    for (int it = tid; it < groups * PG; it += NT) {
      const int part = by_groups.div(it), g = it - part * groups;
      f32x2 acc[GE][CP / 2];
#pragma unroll
      for (int j = 0; j < GE; ++j)
#pragma unroll
        for (int c = 0; c < CP / 2; ++c) acc[j][c] = 0ull;
#pragma unroll 2
      for (int b = part; b < B; b += PG) {
        float v[GE];
        load_group(xb + b * pitch + g * GE, v);
        f32x2 d2[CP / 2];
#pragma unroll
        for (int c = 0; c < C4; ++c) {
          const ulonglong2 dd = *reinterpret_cast<const ulonglong2*>(dl + b * CP + 4 * c);
          d2[2 * c] = dd.x;
          d2[2 * c + 1] = dd.y;
        }
#pragma unroll
        for (int j = 0; j < GE; ++j) {
          const f32x2 p = lsqp::pack2(v[j], v[j]);
#pragma unroll
          for (int c = 0; c < CP / 2; ++c) lsqp::ffma2(acc[j][c], p, d2[c]);
        }
      }
      ulonglong2* o = reinterpret_cast<ulonglong2*>(zp) + (size_t)part * n_g + g;
#pragma unroll
      for (int j = 0; j < GE; ++j)
#pragma unroll
        for (int c = 0; c < C4; ++c) o[(size_t)(j * C4 + c) * groups] = make_ulonglong2(acc[j][2 * c], acc[j][2 * c + 1]);
    }
    if (last_warp && rank == 0) {                    // mean loss and bias step (fixed orders)
      float part = 0.f;
      for (int b = lane; b < B; b += 32) part += rl[b];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      loss_sum += __fdiv_rn(part, (float)B);
      const int c = lane & 15;                       // two lanes per class, every second row each
      float s = 0.f;
      if (c < CP) {
#pragma unroll 8
        for (int b = lane >> 4; b < B; b += 2) s += dl[(size_t)b * CP + c];
      }
      s += __shfl_xor_sync(0xffffffffu, s, 16);
      if (!a.lsq && lane < C) {
        bs[16 + lane] += s;
        bs[lane] = fmaf(-step, s, bs[lane]);
      }
    }
    __syncthreads();
    // A wait of this step ran out: the run ends (below).  No further step, whose bytes would be announced on a barrier that still
    // waits for this step's; the peers' waits then run out as well.  (All waits lie behind the step's first barrier and before
    // this one, so all threads read the same.)
    if (gave_up) break;
    if (geo.nbuf == 1 && u + 1 < U) fetch(u + 1);    // the gradient has read the only row buffer
    // ---- the local step
    for (int e = tid; e < n_g; e += NT) {
      float4 s = reinterpret_cast<const float4*>(zp)[e];
#pragma unroll 8
      for (int p = 1; p < PG; ++p) s = add4(s, reinterpret_cast<const float4*>(zp)[(size_t)p * n_g + e]);
      gs[e] = add4(gs[e], s);
      const int jc = by_groups.div(e), g = e - jc * groups;
      const int m = g * GE + jc / C4, c4 = jc % C4;
      float4* w4 = reinterpret_cast<float4*>(wl + (size_t)m * CP) + c4;
      float4 w = *w4;
      w.x = fmaf(-step, s.x, w.x); w.y = fmaf(-step, s.y, w.y); w.z = fmaf(-step, s.z, w.z); w.w = fmaf(-step, s.w, w.w);
      *w4 = w;
      if (sizeof(T) == 2)
        reinterpret_cast<float4*>(wq + (size_t)m * CP)[c4] =
            make_float4(round_store(w.x, (const T*)nullptr), round_store(w.y, (const T*)nullptr),
                        round_store(w.z, (const T*)nullptr), round_store(w.w, (const T*)nullptr));
    }
  }
  if (gave_up) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    tc::leave_cluster();                             // (no peer stores to a CTA that has left)
  } else if (Q > 1) {
    tc::cluster_sync_all();
  } else {
    __syncthreads();
  }
  float* out = a.G + (size_t)i * a.slot_stride;
  const float sa = st->sa_penalty ? sa_weight(a.sel_tau[i]) : 1.f;   // staleness-aware step size: weight of the upload in Eq. 3
  for (int e = tid; e < nf * C; e += NT) {
    const int m = e / C, c = e - m * C;
    const float4 q = gs[(size_t)((m % GE) * C4 + c / 4) * groups + m / GE];
    const int k = c & 3;
    out[(size_t)m0 * C + e] = (k == 0 ? q.x : k == 1 ? q.y : k == 2 ? q.z : q.w) * sa;
  }
  if (rank == 0) {
    if (!a.lsq && tid < C) out[(size_t)n_w + tid] = bs[16 + tid] * sa;
    if (last_warp && lane == 0) {
      const float loss = __fdiv_rn(loss_sum, (float)U);
      a.loss[i] = loss;
      if (!isfinite(loss)) report(ri, RI_DIVERGED);
    }
  }
  if (tid == 0 && gave_up) {
    // not st->status: a cluster that starts later must find the same status in all of its CTAs
    st->timeout_where = 300;
    report(ri, RI_TIMEOUT);
  }
}

}  // namespace local
}  // namespace absb
