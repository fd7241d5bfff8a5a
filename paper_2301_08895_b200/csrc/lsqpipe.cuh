// Least squares on bf16 data, HBM-bound form: Eq. 2 (U = 1) for all selected workers of a round as
// one stream of bulk row copies.
//
// Work item = (selected worker i, group g of 8 minibatch rows).  Items are dealt round-robin to one
// persistent CTA per SM.  A producer warp copies an item's rows X[idx_b][:] (8 KB each at d = 4096)
// and the model vector of the worker's version into a ring of shared-memory stages with
// cp.async.bulk + mbarrier.  Two teams of 256 threads take four rows of every item each, a thread reading ITS
// columns of them once into registers (the 16-byte vectors tid and tid + 256 of every row), and from those
// registers form the partial dot products (team-reduced in a fixed order to the residuals
// r_b = x_b . w_v - y_b) and then the gradient contribution sum_b r_b x_b into accumulators that
// persist over all items of the CTA.  Every sample row is read from HBM exactly once and from
// shared memory exactly once.  Inside an item a team runs one chain (wait, reads, dots, exchange, residuals, gradient);
// the teams wait for nothing of each other but the stages, so one's arithmetic fills the other's latencies.  An item's 64 KB
// of rows per SM take 2880 cycles at the chip's copy rate (6552 GB/s; 1.947 GHz; a copy also writes); its 8 KB model vector comes
// from L2.  An item takes 2770 cycles, 6.8 TB/s of rows, where a CTA has 28 (mean over all CTAs), 2890 where it has 3 or 4; with
// one team of 512 threads 2900 to 3000.  The inner loops are packed FMAs on operands kept in 64-bit registers.  A round of a few items per CTA is its start-up, so nothing is staged for all of a CTA's items first (5600
// cycles for 4 items, 10600 for 28: the targets' loads queued behind the first items' copies): the producer's lanes draw four
// items' samples at a time, fetch what the draws of the next four need meanwhile, and a row's target arrives with its item,
// by an asynchronous copy counted on the same barrier.  Eq. 3 only
// needs the sum over workers: a CTA writes one partial sum, and one partial loss sum per item and team; the
// Eq. 3 kernel adds both up in a fixed order.
#pragma once
#include <algorithm>

#include "common.cuh"
#include "ctl.cuh"
#include "tc.cuh"

namespace absb {
namespace lsqp {

constexpr int GROUP = 8;                 // rows per item / stage
constexpr int TEAMS = 2;
constexpr int TROWS = GROUP / TEAMS;     // rows of an item per team
constexpr int TEAM = 256;                // threads of a team, two 16-byte column slices each: d <= 4096
constexpr int TWARPS = TEAM / 32;
constexpr int CONSUMERS = TEAMS * TEAM;
constexpr int THREADS = CONSUMERS + 64;  // + producer warp + a warp that prepares job durations
constexpr int BATCH = 32 / GROUP;        // items whose rows the producer's lanes hold
constexpr int MAX_STAGES = 6;
constexpr int SA_LEN = 8;                // weights of the stages, padded: what follows starts on a 16-byte boundary
constexpr int RS = 12;                   // floats between rows of the partial-dot table [TROWS][RS]: 16-byte reads of the rows'
                                         // halves by 8 lanes fall into different banks
constexpr int RED = 2 * TEAMS * TROWS * RS;      // ... of both teams, twice

struct Args {
  DevState* st;
  RoundInfo* ri;
  const int* sel; const int* job; const int* sel_tau;
  const int2* shard;
  u64* next_dur; int* dur_job;           // duration look-ahead (see refresh_next_durations)
  const __nv_bfloat16* X; const float* y;
  const __nv_bfloat16* ring; size_t slot_stride;
  float* loss_part;     // [K][ceil(B / TROWS)] sum over a team's rows of an item of 1/2 r_b^2
  float* G;             // [gridDim.x][slot_stride] per-CTA partial gradient sums
  int d;                // features, multiple of 8, at most 4096
  int stages;           // pipeline depth (2..MAX_STAGES)
  int groups;           // ceil(B / GROUP)
  FastDiv by_groups;
  int W, B, S, sa;      // constants of the run (sa: staleness-aware step size)
  uint32_t key0, key1;
};

inline size_t stage_bytes(int d) { return (size_t)(GROUP + 1) * d * 2; }
inline size_t smem_bytes(int d, int stages) {
  return std::max((size_t)stages * stage_bytes(d), (size_t)TEAM * 64) + (size_t)(MAX_STAGES * GROUP + SA_LEN + RED) * 4 +
         2 * MAX_STAGES * 8 + 64;
}

// Two binary32 values in one 64-bit register (first value in the low word).  The consumers are bound
// by instruction issue: a packed FMA (each half rounds like a scalar fma) halves their FMA count, and
// operands that are created, kept and consumed as 64-bit registers need no moves around it.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
// the two bf16 values of a 32-bit word as binary32 values (exact): element 0 (low half) first; a byte
// permute and a mask, both on the integer pipe, so that the FMA pipe is left to the packed FMAs
__device__ __forceinline__ f32x2 bf16x2_to_f32x2(uint32_t u) {
  f32x2 r;
  asm("{\n\t.reg .b32 lo, hi;\n\tprmt.b32 lo, %1, 0, 0x1044;\n\tand.b32 hi, %1, 0xffff0000;\n\tmov.b64 %0, {lo, hi};\n\t}"
      : "=l"(r) : "r"(u));
  return r;
}
__device__ __forceinline__ void ffma2(f32x2& d, f32x2 a, f32x2 b) {      // d += a * b, per half
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

__device__ __forceinline__ void bulk_row(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(tc::smem_u32(dst)), "l"(src), "r"(bytes), "r"(tc::smem_u32(bar)) : "memory");
}

// a row's target: a 4-byte asynchronous copy, and the lane's arrival on the item's barrier once its copies have landed
__device__ __forceinline__ void target(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void target_arrive(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}

__global__ void __launch_bounds__(THREADS, 1) lsq_pipe_kernel(const __grid_constant__ Args a) {
  extern __shared__ __align__(128) unsigned char lsm[];
  const int B = a.B, d = a.d, S = a.S, groups = a.groups, STAGES = a.stages;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nvec = d >> 3;
  const uint32_t row_bytes = (uint32_t)d * 2u;
  const size_t stg = (size_t)(GROUP + 1) * row_bytes;
  unsigned char* stage0 = lsm;                                             // (and the teams' exchange at the end)
  float* m_y = reinterpret_cast<float*>(lsm + max((size_t)STAGES * stg, (size_t)TEAM * 64));     // [MAX_STAGES][GROUP] targets
  float* m_sa = m_y + MAX_STAGES * GROUP;                                  // [MAX_STAGES] weight of the worker's gradient in Eq. 3
  float* red = m_sa + SA_LEN;                                              // [2][TEAMS][TROWS][RS] partial dots, [row][warp]
  uint64_t* full = reinterpret_cast<uint64_t*>(red + RED);                 // [STAGES]
  uint64_t* empty = full + MAX_STAGES;                                     // [STAGES]
  volatile int* abort = reinterpret_cast<volatile int*>(empty + MAX_STAGES);
  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) { tc::mbar_init(&full[s], 1 + GROUP); tc::mbar_init(&empty[s], CONSUMERS / 32); }
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  grid_dependency_sync();
  DevState* st = a.st;
  RoundInfo* ri = a.ri;
  const bool producer = warp == CONSUMERS / 32;
  // items of this CTA: it = blockIdx.x + q * gridDim.x, q = 0 .. my_items - 1.  The producer's lanes hold the rows of four of
  // them (a selected worker's entries exist whether or not it is selected this round).
  struct Draw { int i, wn, tau; };
  auto selected = [&](int q0) -> Draw {
    Draw w{a.by_groups.div((int)blockIdx.x + (q0 + (lane >> 3)) * (int)gridDim.x), 0, 0};
    if (w.i < a.W) { w.wn = a.sel[w.i]; w.tau = a.sel_tau[w.i]; }
    return w;
  };
  Draw cur{0, 0, 0}, nxt{0, 0, 0};
  if (producer) { cur = selected(0); nxt = selected(BATCH); }
  const int status = st->status, K = ri->K, t = ri->t;
  if (status != ST_OK) return;
  const int n_items = K * groups;
  const int my_items = n_items > (int)blockIdx.x ? (n_items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;

  f32x2 acc[2][4];                  // gradient sums of this thread's 2 x 8 columns (all-zero bits = two zeros)
#pragma unroll
  for (int v = 0; v < 2; ++v)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[v][j] = 0ull;
  int stage = 0, buf = 0;
  uint32_t phase = 0;
  bool ok = true;
  if (producer) {
    // ------------------------------------------------------------------ producer warp
    int2 shard = a.shard[cur.wn];
    int job = a.job[cur.wn];
    for (int q0 = 0; q0 < my_items && ok; q0 += BATCH) {
      const int2 shard_n = a.shard[nxt.wn];          // for the next four items
      const int job_n = a.job[nxt.wn];
      const Draw after = selected(q0 + 2 * BATCH);
      const int r = lane & 7, g = (int)blockIdx.x + (q0 + (lane >> 3)) * (int)gridDim.x - cur.i * groups;
      const int b = g * GROUP + r, rows = min(GROUP, B - g * GROUP);
      int idx = -1;
      if (q0 + (lane >> 3) < my_items && b < B) {    // Philox block b / 4, word b % 4
        uint32_t w4[4];
        philox4x32_10((uint32_t)cur.wn, (uint32_t)job, 1u, (uint32_t)(b >> 2), a.key0, a.key1, w4);
        const uint32_t wd = (b & 3) == 0 ? w4[0] : (b & 3) == 1 ? w4[1] : (b & 3) == 2 ? w4[2] : w4[3];
        idx = shard.x + (int)__umulhi(wd, (unsigned)shard.y);
      }
      const int slot = (t - cur.tau) % (S + 1);
#pragma unroll 1
      for (int e = 0; e < min(BATCH, my_items - q0); ++e) {
        if (lane == 0) ok = tc::mbar_wait(&empty[stage], phase ^ 1u, abort);
        ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
        if (!ok) break;
        if ((lane >> 3) == e) {                      // the lanes that hold the item's rows; the first also the weights
          unsigned char* sb = stage0 + (size_t)stage * stg;
          if (r == 0) {
            m_sa[stage] = a.sa ? sa_weight(cur.tau) : 1.f;       // staleness-aware step size
            tc::mbar_expect_tx(&full[stage], (uint32_t)(rows + 1) * row_bytes);
            bulk_row(sb + (size_t)GROUP * row_bytes, a.ring + (size_t)slot * a.slot_stride, row_bytes, &full[stage]);
          }
          if (idx >= 0) {
            target(m_y + stage * GROUP + r, a.y + idx);
            bulk_row(sb + (size_t)r * row_bytes, a.X + (size_t)idx * d, row_bytes, &full[stage]);
          }
          target_arrive(&full[stage]);
        }
        __syncwarp();
        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
      }
      cur = nxt; nxt = after; shard = shard_n; job = job_n;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else if (warp == CONSUMERS / 32 + 1) {
    // job durations: worker blockIdx.x + gridDim.x * lane
    refresh_next_durations(st, a.job, a.next_dur, a.dur_job, (int)blockIdx.x + (int)gridDim.x * lane);
  } else {
    // ------------------------------------------------------------------ consumers
    const int team = warp / TWARPS, tw = warp % TWARPS, r0 = team * TROWS;
    const int v0 = tid % TEAM, v1 = v0 + TEAM;     // the 16-byte column slices this thread owns
    const bool in0 = v0 < nvec, in1 = v1 < nvec;
    for (int q = 0; q < my_items; ++q) {
      // a wait that runs out ends the run (status below); the item is then formed on whatever is there
      tc::mbar_wait(&full[stage], phase, abort);
      const unsigned char* sb = stage0 + (size_t)stage * stg;
      const unsigned char* sx = sb + (size_t)r0 * row_bytes;
      const unsigned char* sw = sb + (size_t)GROUP * row_bytes;
      const int it = (int)blockIdx.x + q * (int)gridDim.x;
      const int i = a.by_groups.div(it), g = it - i * groups;
      const int rows = min(TROWS, B - g * GROUP - r0);     // may be negative: no row for this team
      uint4 xr[2][TROWS], wr[2];
      if (rows == TROWS && nvec == 2 * TEAM) {       // the usual case (uniform in the CTA): no predicates
        wr[0] = *reinterpret_cast<const uint4*>(sw + (size_t)v0 * 16);
        wr[1] = *reinterpret_cast<const uint4*>(sw + (size_t)v1 * 16);
#pragma unroll
        for (int r = 0; r < TROWS; ++r) {
          xr[0][r] = *reinterpret_cast<const uint4*>(sx + (size_t)r * row_bytes + (size_t)v0 * 16);
          xr[1][r] = *reinterpret_cast<const uint4*>(sx + (size_t)r * row_bytes + (size_t)v1 * 16);
        }
      } else {
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        wr[0] = in0 ? *reinterpret_cast<const uint4*>(sw + (size_t)v0 * 16) : zero;
        wr[1] = in1 ? *reinterpret_cast<const uint4*>(sw + (size_t)v1 * 16) : zero;
#pragma unroll
        for (int r = 0; r < TROWS; ++r) {
          xr[0][r] = (in0 && r < rows) ? *reinterpret_cast<const uint4*>(sx + (size_t)r * row_bytes + (size_t)v0 * 16) : zero;
          xr[1][r] = (in1 && r < rows) ? *reinterpret_cast<const uint4*>(sx + (size_t)r * row_bytes + (size_t)v1 * 16) : zero;
        }
      }
      // the rows are in registers now: hand the stage back to the producer
      const float yv = m_y[stage * GROUP + r0 + (lane & 3)], sa = m_sa[stage];
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&empty[stage]);
      if (++stage == STAGES) { stage = 0; phase ^= 1u; }
      // partial dot products of the team's rows over this thread's columns
      float pd[TROWS];
      {
        f32x2 s2[TROWS];               // (sum over even columns, sum over odd columns)
#pragma unroll
        for (int r = 0; r < TROWS; ++r) s2[r] = 0ull;
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          if (v == 1 && nvec <= TEAM) break;         // (short rows: uniform)
          const f32x2 w2[4] = {bf16x2_to_f32x2(wr[v].x), bf16x2_to_f32x2(wr[v].y), bf16x2_to_f32x2(wr[v].z), bf16x2_to_f32x2(wr[v].w)};
#pragma unroll
          for (int r = 0; r < TROWS; ++r) {
            ffma2(s2[r], bf16x2_to_f32x2(xr[v][r].x), w2[0]);
            ffma2(s2[r], bf16x2_to_f32x2(xr[v][r].y), w2[1]);
            ffma2(s2[r], bf16x2_to_f32x2(xr[v][r].z), w2[2]);
            ffma2(s2[r], bf16x2_to_f32x2(xr[v][r].w), w2[3]);
          }
        }
#pragma unroll
        for (int r = 0; r < TROWS; ++r) {
          float e0, e1;
          unpack2(s2[r], e0, e1);
          pd[r] = e0 + e1;
        }
      }
      // warp sum of the 4 values with 6 shuffles: the first two exchanges halve the rows a lane still carries;
      // afterwards lane l holds the warp's sum for row l >> 3
      float k1;
      {
        const bool hi = (lane & 16) != 0, h8 = (lane & 8) != 0;
        float k2[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float recv = __shfl_xor_sync(0xffffffffu, hi ? pd[e] : pd[e + 2], 16);
          k2[e] = (hi ? pd[e + 2] : pd[e]) + recv;
        }
        const float recv = __shfl_xor_sync(0xffffffffu, h8 ? k2[0] : k2[1], 8);
        k1 = (h8 ? k2[1] : k2[0]) + recv;
        k1 += __shfl_xor_sync(0xffffffffu, k1, 4);
        k1 += __shfl_xor_sync(0xffffffffu, k1, 2);
        k1 += __shfl_xor_sync(0xffffffffu, k1, 1);
      }
      float* rb = red + (buf * TEAMS + team) * (TROWS * RS);
      if ((lane & 7) == 0) rb[(lane >> 3) * RS + tw] = k1;
      asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(TEAM) : "memory");
      // every warp adds the 8 warps' sums of a row up in the same order: lane l takes row l & 3 and
      // the four warps of half (l >> 2) & 1 (one 16-byte load), then the halves are added across lanes
      const int row = lane & 3;
      const float4 four = *reinterpret_cast<const float4*>(rb + row * RS + 4 * ((lane >> 2) & 1));
      float mine = (four.x + four.y) + (four.z + four.w);
      mine += __shfl_xor_sync(0xffffffffu, mine, 4);
      mine = row < rows ? mine - yv : 0.f;
      float res[TROWS], lsum = 0.f;
#pragma unroll
      for (int r = 0; r < TROWS; ++r) {
        res[r] = __shfl_sync(0xffffffffu, mine, r);
        lsum += 0.5f * res[r] * res[r];
      }
      if (v0 == 0 && rows > 0) a.loss_part[(size_t)i * ((B + TROWS - 1) / TROWS) + g * TEAMS + team] = lsum;
#pragma unroll
      for (int r = 0; r < TROWS; ++r) {
        const float rr = res[r] * sa;
        const f32x2 r2 = pack2(rr, rr);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          if (v == 1 && nvec <= TEAM) break;
          ffma2(acc[v][0], bf16x2_to_f32x2(xr[v][r].x), r2);
          ffma2(acc[v][1], bf16x2_to_f32x2(xr[v][r].y), r2);
          ffma2(acc[v][2], bf16x2_to_f32x2(xr[v][r].z), r2);
          ffma2(acc[v][3], bf16x2_to_f32x2(xr[v][r].w), r2);
        }
      }
      buf ^= 1;
    }
  }
  ok = __syncthreads_and(*abort == 0) != 0;
  // the producer's copies have all been consumed (every full barrier was waited on), unless a wait
  // gave up: then let copies in flight land before the shared memory goes away
  if (!ok) {
    const unsigned long long t0 = tc::global_ns();
    while (tc::global_ns() - t0 < 200000ull) {}
    if (tid == 0) {
      st->timeout_where = 200;
      st->status = ST_TIMEOUT;
    }
    return;
  }
  // this CTA's partial sum: first team's + second team's
  f32x2* box = reinterpret_cast<f32x2*>(stage0);
  if (tid >= TEAM && tid < 2 * TEAM)
#pragma unroll
    for (int v = 0; v < 2; ++v)
#pragma unroll
      for (int j = 0; j < 4; j += 2)
        *reinterpret_cast<ulonglong2*>(box + ((v * 2 + j / 2) * TEAM + tid - TEAM) * 2) = make_ulonglong2(acc[v][j], acc[v][j + 1]);
  __syncthreads();
  if (tid < TEAM) {
    float* gout = a.G + (size_t)blockIdx.x * a.slot_stride;
#pragma unroll
    for (int v = 0; v < 2; ++v)
      if (tid + v * TEAM < nvec)
#pragma unroll
        for (int j = 0; j < 4; j += 2) {
          float4 g;
          unpack2(acc[v][j], g.x, g.y);
          unpack2(acc[v][j + 1], g.z, g.w);
          const float4 o = *reinterpret_cast<const float4*>(box + ((v * 2 + j / 2) * TEAM + tid) * 2);
          reinterpret_cast<float4*>(gout + (size_t)(tid + v * TEAM) * 8)[j / 2] = make_float4(g.x + o.x, g.y + o.y, g.z + o.z, g.w + o.w);
        }
  }
}

}  // namespace lsqp
}  // namespace absb
