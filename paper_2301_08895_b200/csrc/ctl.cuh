// Server-side integer engine of Algorithm 1: arrival selection, Eq. 4-6 bookkeeping,
// Philox job durations and minibatch indices.  One CTA of 1024 threads; every result is an
// integer decided by exact arithmetic, so the trace is reproducible bit for bit.
#pragma once
#include "common.cuh"

namespace absb {

// ---------------------------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32->64 multiplies, with the key
// advanced by Weyl constants between rounds.
__device__ __forceinline__ void philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                              uint32_t k0, uint32_t k1, uint32_t out[4]) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi_a = __umulhi(0xD2511F53u, c0), lo_a = 0xD2511F53u * c0;
    const uint32_t hi_b = __umulhi(0xCD9E8D57u, c2), lo_b = 0xCD9E8D57u * c2;
    const uint32_t n0 = hi_b ^ c1 ^ k0, n2 = hi_a ^ c3 ^ k1;
    c0 = n0; c1 = lo_b; c2 = n2; c3 = lo_a;
    k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
  }
  out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
}

// Series logarithm that defines the exponential job times: u = m 2^e with m in [sqrt(1/2),
// sqrt(2)), s = (m-1)/(m+1), ln u = e ln2 + 2s(1 + s^2/3 + ... + s^22/23).  Each step is one
// binary64 operation rounded to nearest (the _rn intrinsics are never contracted into FMAs).
__device__ __forceinline__ double ln_series(double u) {
  const u64 bits = (u64)__double_as_longlong(u);
  int e = (int)((bits >> 52) & 0x7FF) - 1023;
  double m = __longlong_as_double((i64)((bits & 0x000FFFFFFFFFFFFFull) | 0x3FF0000000000000ull));
  if (m >= 1.4142135623730951) { m = __dmul_rn(m, 0.5); e += 1; }
  const double s = __ddiv_rn(__dadd_rn(m, -1.0), __dadd_rn(m, 1.0));
  const double s2 = __dmul_rn(s, s);
  // the coefficients 1 / (2k + 1) are correctly rounded quotients of constants: compile-time values
  constexpr double INV_ODD[12] = {1.0 / 1.0,  1.0 / 3.0,  1.0 / 5.0,  1.0 / 7.0,  1.0 / 9.0,  1.0 / 11.0,
                                  1.0 / 13.0, 1.0 / 15.0, 1.0 / 17.0, 1.0 / 19.0, 1.0 / 21.0, 1.0 / 23.0};
  double p = INV_ODD[11];
#pragma unroll
  for (int k = 10; k >= 0; --k) {
    p = __dmul_rn(p, s2);
    p = __dadd_rn(p, INV_ODD[k]);
  }
  const double head = __dmul_rn((double)e, 0.6931471805599453);
  const double tail = __dmul_rn(__dmul_rn(2.0, s), p);
  return __dadd_rn(head, tail);
}

// Duration of job j of worker n in ticks (2^20 per time unit); 0 signals "out of range".
__device__ __forceinline__ u64 job_ticks(const TimeDist& d, uint32_t k0, uint32_t k1, int n, int j) {
  uint32_t w[4];
  philox4x32_10((uint32_t)n, (uint32_t)j, 0u, 0u, k0, k1, w);
  const double u = __dmul_rn(__dadd_rn((double)w[0], 0.5), 2.3283064365386963e-10);  // 2^-32
  double dur;
  if (d.kind == ABS_T_GAMMA) {
    // sum of `shape` exponential draws, left to right; draw i uses word i % 4 of block i / 4
    double total = -ln_series(u);
    for (int i = 1; i < d.shape; ++i) {
      if ((i & 3) == 0) philox4x32_10((uint32_t)n, (uint32_t)j, 0u, (uint32_t)(i >> 2), k0, k1, w);
      const uint32_t wi = (i & 3) == 0 ? w[0] : (i & 3) == 1 ? w[1] : (i & 3) == 2 ? w[2] : w[3];
      const double ui = __dmul_rn(__dadd_rn((double)wi, 0.5), 2.3283064365386963e-10);
      total = __dadd_rn(total, -ln_series(ui));
    }
    dur = __dadd_rn(d.shift, __ddiv_rn(total, d.rate));
  } else if (d.kind == ABS_T_CONST) dur = d.shift;
  else if (d.kind == ABS_T_EXP) dur = __ddiv_rn(-ln_series(u), d.rate);
  else if (d.kind == ABS_T_SHIFTED_EXP) dur = __dadd_rn(d.shift, __ddiv_rn(-ln_series(u), d.rate));
  else dur = __ddiv_rn(d.scale, __dsqrt_rn(u));
  if (d.slow_mod > 0 && n % d.slow_mod == d.slow_rem) dur = __dmul_rn(dur, d.slow_factor);
  const double scaled = __dmul_rn(dur, 1048576.0);
  if (!(scaled < 9007199254740992.0)) return 0ull;
  const u64 ticks = __double2ull_rd(scaled);
  return ticks < 1ull ? 1ull : ticks;
}

// The double-precision pipe of one SM is narrow, so the control CTA does not compute durations
// itself: the duration of the job a worker will start NEXT depends only on (worker, job index)
// and is prepared ahead of time by one warp of each of the first ceil(N/32) CTAs of a wide
// kernel that runs between two control kernels.  Only workers whose job index moved are redone.
__device__ __forceinline__ void refresh_next_durations(const DevState* st, const int* job, u64* next_dur,
                                                       int* dur_job, int n) {
  if (n >= st->W) return;
  const int j = job[n] + 1;
  if (dur_job[n] != j) {
    next_dur[n] = job_ticks(st->dist, st->key0, st->key1, n, j);
    dur_job[n] = j;
  }
}

// ---------------------------------------------------------------------------------------------
// Sort of n = 256 (NT < 1024), 512 or 1024 distinct 64-bit keys, one per thread, by ranking: inside a warp every key counts
// the smaller keys of its warp (31 shuffles, no dependent chain), which leaves sorted runs of 32.  Eight runs are merged at
// once: a key's place is the number of smaller keys in every other run, found by binary searches that run side by side (256
// keys: 1.5k cycles instead of 3.1k with pairwise merges); more runs are merged pairwise, where one search per key and
// level is less shared-memory traffic.  Returns the buffer (A or B) that holds the sorted keys.
template <int NT>
__device__ __forceinline__ u64* rank_merge_sort(u64 key, u64* A, u64* B, int n) {
  const int tid = threadIdx.x, lane = tid & 31;
  const bool active = tid < n;                 // whole warps
  if (active) {
    int rank = 0;
#pragma unroll
    for (int l = 0; l < 32; ++l) rank += (__shfl_sync(0xffffffffu, key, l) < key) ? 1 : 0;
    A[(tid - lane) + rank] = key;
  }
  __syncthreads();
  if (NT < 1024) {
    if (active) {
      const u64 k = A[tid];
      const int own = tid >> 5;
      int lo[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) lo[r] = 0;
#pragma unroll
      for (int step = 16; step > 0; step >>= 1)
#pragma unroll
        for (int r = 0; r < 8; ++r)
          lo[r] += A[r * 32 + lo[r] + step - 1] < k ? step : 0;     // at most 31 of a run after the last step
      int rank = 0;
#pragma unroll
      for (int r = 0; r < 8; ++r)
        rank += r == own ? lane : lo[r] + (A[r * 32 + lo[r]] < k ? 1 : 0);
      B[rank] = k;
    }
    __syncthreads();
    return B;
  }
  u64* src = A;
  u64* dst = B;
  for (int L = 32; L < n; L <<= 1) {
    if (active) {
      const u64 k = src[tid];
      const int pair_base = tid & ~(2 * L - 1);
      const int idx = tid - pair_base;
      const int own = idx & (L - 1);
      const u64* other = src + pair_base + ((idx < L) ? L : 0);
      int lo = 0, hi = L;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (other[mid] < k) lo = mid + 1; else hi = mid;
      }
      dst[pair_base + own + lo] = k;
    }
    __syncthreads();
    u64* tmp = src; src = dst; dst = tmp;
  }
  return src;
}

__device__ __forceinline__ int floor_div(int a, int b) {  // b > 0
  const int q = a / b;
  return (a % b != 0 && a < 0) ? q - 1 : q;
}

struct CtlShared {
  u64 keysA[1024], keysB[1024];        // (row losses of the open round before the sort)
  unsigned short wcnt[32][MAX_TAU];   // per-warp count of selected workers per staleness
  int cnt[MAX_TAU];                    // selected workers per staleness
  int grow0[MAX_TAU];                  // first row of each staleness group
  int row0[1024];                      // first gradient row of each selected worker
  float lossv[1024];                   // mean minibatch loss of each selected worker
  int version[1024], job[1024];        // per-worker state after the round's bookkeeping
  int sel_n[1024];                     // worker id of each arrival, in arrival order
  int2 shard[1024];                    // per worker: first sample and length of its shard
  float redf[32];
  int bad[32];
  int warp_tot[32];
  int scalar[8];
};

// A duration that was not prepared ahead of time (rare: kept out of the step's straight-line code)
static __device__ __noinline__ u64 job_ticks_call(const DevState* st, uint32_t key0, uint32_t key1, int n, int j) {
  return job_ticks(st->dist, key0, key1, n, j);
}

// Completes the open round (Eq. 5, Eq. 4, Eq. 6, trace row), then selects the arrivals of the
// next round and lays out its gradient rows.
//   do_finish: complete the open round if there is one
//   do_select: open the next round
// A lone CTA is bound by its chain of dependent phases: a global-memory access costs close to a microsecond, a block-wide
// barrier with what leads to it a few hundred cycles, and straight-line code that runs once a launch about ten cycles an
// instruction.  So everything a later phase needs is loaded up front in one wave (the run's constants come with the
// launch), sums over the arrivals and the rules that follow from them are formed by every warp itself instead of by one for
// all, rules that rarely change anything (Eq. 5 raising K, Eq. 4 after it) have a short test in front, and a worker's rank
// is counted.  16 workers x 64 rows: 5.7 -> 4.4 us; 64 workers 6.6 -> 4.9 us;
// 8 workers inside the persistent kernel, 200 rounds: 1.51 -> 1.39 ms a run (now 5.7 us a round in the kernel).
//   t_sel:     index of the round that follows the open one (the host counts rounds; parity of
//              t_sel - 1 / t_sel picks the layout copy of the open / the new round)
//   look_here: the workers that were renewed also get the duration of the job AFTER the one they
//              start now prepared here, at the end of the step (see refresh_next_durations), for
//              callers whose gradient kernel does not do it (2000 cycles of binary64 series)
//   late_status: when the step runs next to the Eq. 3 kernel of the round it finishes, a status it
//              raises must not be seen by that kernel's blocks (they would skip a valid step):
//              the status is left in *late_status (shared memory) for the caller to publish later
template <int NT>
__device__ __forceinline__ int ctl_round(const CtlArgs& a, CtlShared& sh, int do_finish, int do_select, int t_sel,
                                         int look_here = 0, int* late_status = nullptr) {
  constexpr int NWP = NT / 32;
  constexpr int ROWS = NT >= 1024 ? 4 : 8;            // row losses a thread fetches ahead of time
  DevState* st = a.st;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto raise = [&](int code) {
    if (late_status != nullptr) *late_status = code;
    else st->status = code;
  };
  // ---- one wave of loads (everything a later phase may need: all addresses exist whether or not a round is open)
  const CtlConst& k = a.k;
  const int W = k.W, S = k.S, B = k.B;
  const int po = (t_sel - 1) & 1, pn = t_sel & 1;     // layout copy of the open / of the new round
  const bool net = a.row_loss != nullptr;
  const bool ahead = net && do_finish && a.rows_cap <= ROWS * NT;      // all row losses fit
  int my_sel = 0, my_tau = 0, my_row0 = 0, my_version = 0, my_job = 0, my_dur_job = -1;
  float my_loss = 0.f;
  int2 my_shard = make_int2(0, 0);
  u64 my_c = 0, my_next_dur = 0;
  float rl[ROWS];
  if (ahead) {
#pragma unroll
    for (int u = 0; u < ROWS; ++u) rl[u] = tid + u * NT < a.rows_cap ? a.row_loss[tid + u * NT] : 0.f;
  }
  if (tid < W) {
    my_c = a.c[tid]; my_version = a.version[tid]; my_job = a.job[tid];
    my_dur_job = a.dur_job[tid]; my_next_dur = a.next_dur[tid];
    my_sel = a.sel[po][tid]; my_tau = a.sel_tau[po][tid]; my_row0 = a.sel_row0[po][tid];
    if (a.draw) my_shard = a.shard[tid];
    if (do_finish && !net && a.loss_part == nullptr) my_loss = a.loss[tid];
  }
  const int status0 = st->status, expired0 = st->timeout_where, open0 = st->open, diverged0 = a.ri[po].diverged;
  const u64 T_end0 = st->T_end;
  const float L0_prev = st->L0;
  const i64 sel_off = st->sel_total, rst_off = st->rst_total;
  const u64 comm0 = st->comm;
  const int last_id = st->last_id, theta0 = st->theta;
  int t = st->t, K = st->K;
  if (do_finish && !net && a.loss_part != nullptr && tid < W) {
    // the least-squares pipeline leaves per-group sums; same order and rounding as its Eq. 3 kernel
    const float* p = a.loss_part + (size_t)tid * a.loss_groups;
    float s = 0.f;
#pragma unroll 4
    for (int g = 0; g < a.loss_groups; ++g) s += p[g];
    my_loss = __fdiv_rn(s, (float)B);
  }
  if (status0 != ST_OK) return 1;
  if (expired0 != 0) {                                // (by a kernel that may not change the status while it runs)
    if (tid == 0) raise(ST_TIMEOUT);
    return 1;
  }
  const bool fin = do_finish && open0;

  int restart = 0, renewed = 0;                       // this thread's worker started a new job in the finish step
  int K_next = K, theta = theta0;
  float Lt = 0.f, L0 = 0.f;
  // ------------------------------------------------------------------ finish round t
  if (fin) {
    if (net) {
      // per-worker mean of the per-sample losses: TPW neighbouring threads share a worker, each
      // adds every TPW-th row (eight at a time), then the TPW partial sums are added by a
      // fixed shuffle tree
      float* rls = reinterpret_cast<float*>(sh.keysA);
      sh.row0[tid] = my_row0;
      if (ahead) {
#pragma unroll
        for (int u = 0; u < ROWS; ++u) rls[tid + u * NT] = rl[u];
      }
      __syncthreads();
      const int lg_k = max(5, 32 - __clz(K - 1)), lg_tpw = min(5, 31 - __clz(NT) - lg_k);      // (K >= 1; K = 1: clz(0) = 32)
      const int tpw = 1 << lg_tpw, i = tid >> lg_tpw, sub = tid & (tpw - 1);
      float acc = 0.f;
      if (i < K) {
        const float* src = (ahead ? rls : a.row_loss) + sh.row0[i];
#pragma unroll 1
        for (int b = sub; b < B; b += 8 * tpw) {
          float x[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) x[u] = b + u * tpw < B ? src[b + u * tpw] : 0.f;
#pragma unroll
          for (int u = 0; u < 8; ++u) acc += x[u];
        }
      }
#pragma unroll 1
      for (int o = tpw >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (i < K && sub == 0) sh.lossv[i] = __fdiv_rn(acc, (float)B);
    } else if (tid < K) {
      sh.lossv[tid] = my_loss;
    }
    __syncthreads();
    // loss estimate: adjacent-pair tree sum in binary32 over 1024 leaves (missing ones are zero), /K in binary32
    auto tree = [&](float v) {
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) v = __fadd_rn(v, __shfl_down_sync(0xffffffffu, v, o));
      return v;
    };
    float v = 0.f;
    int bad = 0;
    if (tid < K) my_loss = sh.lossv[tid];
    if (K <= 32) {
      if (lane < K) v = sh.lossv[lane];
      bad = __any_sync(0xffffffffu, !isfinite(v));
      v = tree(v);
    } else {
      if (tid < K) v = my_loss;
      bad = __any_sync(0xffffffffu, !isfinite(v));
      v = tree(v);
      if (lane == 0) { sh.redf[warp] = v; sh.bad[warp] = bad; }
      __syncthreads();
      v = lane < NWP ? sh.redf[lane] : 0.f;
      bad = __any_sync(0xffffffffu, lane < NWP && sh.bad[lane]);
      v = tree(v);
    }
    v = __shfl_sync(0xffffffffu, v, 0);
    if (bad || diverged0) {
      if (tid == 0) { raise(diverged0 & RI_TIMEOUT ? ST_TIMEOUT : ST_DIVERGED); st->open = 0; }
      return 1;
    }
    Lt = __fdiv_rn(v, (float)K);
    L0 = (t == 0) ? Lt : L0_prev;
    // Eq. 5 as an exact integer rule: the largest k with k^2 Lt <= K0^2 L0, if above K (binary64 products of a 20-bit
    // integer and a binary32 value are exact).  K + 1 is tested first; only when it passes, a binary32 estimate of
    // K0 sqrt(L0/Lt) is corrected with the exact test.
    if (k.k_mode == ABS_K_ADAPTIVE && K < W) {
      const double rhs = __dmul_rn((double)(k.K0 * k.K0), (double)L0), lt = (double)Lt;
      auto holds = [&](int n) { return __dmul_rn((double)(n * n), lt) <= rhs; };
      if (Lt <= 0.f) {
        K_next = W;
      } else if (holds(K + 1)) {
        const float est = (float)k.K0 * sqrtf(L0 / Lt);
        int n = (est >= (float)W) ? W : max(K + 1, (est >= 1.f) ? (int)est : 1);
        while (n < W && holds(n + 1)) ++n;
        while (!holds(n)) --n;                        // (ends at K + 1 at the latest)
        K_next = n;
      }
    }
    // Eq. 4 with a = S - N/K0, in integers: a function of K, so the last round's threshold stands while K does
    if (K_next != K || t == 0) {
      theta = k.theta_cap;
      if (k.bound_mode == ABS_BOUND_ADAPTIVE) {
        // (32-bit: at most 1024 workers)
        theta = min(theta, max(1, theta + floor_div(W * (k.K0 - K_next), K_next * k.K0)));
      } else if (k.bound_mode == ABS_BOUND_OFFSET) {     // Eq. 4 with a given: floor(N/K + a) = floor(N/K) + a
        theta = min(theta, max(1, W / K_next + k.bound_offset));
      }
    }
    // Eq. 6 in Algorithm 1's order: arrivals and over-stale workers get w^{t+1}.  The arrivals are the workers up to the last
    // one's (completion tick, id).
    int range_err = 0;
    if (tid < W) {
      const bool sel_me = ((my_c << 10) | (u64)tid) <= ((T_end0 << 10) | (u64)last_id);
      restart = !sel_me && !k.no_restart && (t + 1 - k.literal_eq6 - my_version) > theta;
      if (sel_me || restart) {
        const int j = my_job + 1;
        const u64 dt = (my_dur_job == j) ? my_next_dur : job_ticks_call(st, k.key0, k.key1, tid, j);
        const u64 cn = T_end0 + dt;
        if (dt == 0ull || cn >= (1ull << 53)) range_err = 1;
        my_job = j; my_version = t + 1; my_c = cn;
        renewed = 1;
        a.job[tid] = j;
        a.version[tid] = t + 1;
        a.c[tid] = cn;
      }
    }
    // (for the ascending list of restarted ids)
    const unsigned rb = __ballot_sync(0xffffffffu, restart), eb = __ballot_sync(0xffffffffu, range_err);
    if (lane == 0) sh.warp_tot[warp] = __popc(rb) | (eb != 0u ? 1 << 16 : 0);
  }
  if (do_select) {
    // unused slots get distinct keys above every real one
    sh.keysA[tid] = (tid < W) ? ((my_c << 10) | (u64)tid) : (0xFFFFFFFFFFFFFC00ull | (u64)tid);
    sh.version[tid] = my_version;
    sh.job[tid] = my_job;
    sh.shard[tid] = my_shard;
    if (net) for (int u = lane; u <= S; u += 32) sh.wcnt[warp][u] = 0;
  }
  __syncthreads();
  if (fin) {
    const int x = lane < NWP ? sh.warp_tot[lane] : 0;
    const int R = __reduce_add_sync(0xffffffffu, x & 0xffff);
    const bool range_err = __any_sync(0xffffffffu, x >> 16);
    if (R > 0) {                                      // ascending list of restarted ids
      const unsigned rb = __ballot_sync(0xffffffffu, restart);
      const int base = __reduce_add_sync(0xffffffffu, lane < warp ? x & 0xffff : 0);
      if (restart) a.tr_rst_id[rst_off + base + __popc(rb & ((1u << lane) - 1u))] = tid;
    }
    if (tid < K) {
      a.tr_sel_id[sel_off + tid] = my_sel;
      a.tr_sel_tau[sel_off + tid] = my_tau;
      a.tr_sel_loss[sel_off + tid] = my_loss;
    }
    if (tid == 0) {
      const u64 comm = comm0 + (u64)(K + R);
      a.tr_K[t] = K; a.tr_R[t] = R; a.tr_theta[t] = theta; a.tr_T[t] = T_end0;
      a.tr_loss[t] = Lt; a.tr_comm[t] = comm;
      a.tr_sel_off[t] = sel_off; a.tr_rst_off[t] = rst_off;
      a.tr_sel_off[t + 1] = sel_off + K; a.tr_rst_off[t + 1] = rst_off + R;
      st->sel_total = sel_off + K; st->rst_total = rst_off + R; st->comm = comm;
      st->L0 = L0; st->theta = theta; st->K = K_next; st->t = t + 1; st->open = 0;
      if (range_err) raise(ST_RANGE);
    }
    if (range_err) return 1;
    t = t + 1;
    K = K_next;
  }

  // duration of the job after the one just started, for the next control step to look up
  if (look_here && renewed) {
    a.next_dur[tid] = job_ticks_call(st, k.key0, k.key1, tid, my_job + 1);
    a.dur_job[tid] = my_job + 1;
  }
  // ------------------------------------------------------------------ select round t
  if (!do_select) return 1;
  if (t != t_sel) {                      // host and device disagree on the round index
    if (tid == 0) raise(ST_INTERNAL);
    return 1;
  }
  if (t >= k.max_rounds) {
    if (tid == 0) raise(ST_NOSPACE);
    return 1;
  }
  // arrivals: the K smallest (completion tick, worker id) keys
  const u64* sorted = sh.keysA;
  const bool count = NT < 1024 && W <= 128;
  if (count) {
    // the rank of a key is the number of smaller ones: 8, 4 or 2 lanes share a key and take every 8th, 4th, 2nd other (merging
    // sorted runs by binary search, in code for eight runs, took 3300 cycles for two; from 129 workers on comparing all pairs
    // would cost more)
    const int lg_p = W <= 32 ? 3 : W <= 64 ? 2 : 1, per = 256 >> (2 * lg_p);
    const int n = tid >> lg_p, part = tid & ((1 << lg_p) - 1);
    if (tid < 256) {
      const u64 mine = sh.keysA[n];
      int rank = 0;
      const u64* p = sh.keysA + part;
#pragma unroll 4
      for (int q = 0; q < per; ++q) rank += p[q << lg_p] < mine ? 1 : 0;
#pragma unroll 1
      for (int o = (1 << lg_p) >> 1; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
      if (part == 0 && rank < K) sh.sel_n[rank] = n;     // (n < W: the keys of unused slots rank behind)
    }
    __syncthreads();
  } else {
    sorted = rank_merge_sort<NT>(sh.keysA[tid], sh.keysA, sh.keysB, NT < 1024 ? 256 : W <= 512 ? 512 : 1024);
  }
  int n = -1, tau = -1;
  u64 T_end = 0ull;
  if (tid < K) {
    n = count ? sh.sel_n[tid] : (int)(sorted[tid] & 1023ull);
    tau = t - sh.version[n];
  }
  int last = 0;
  if (tid == 0) {
    last = count ? sh.sel_n[K - 1] : (int)(sorted[K - 1] & 1023ull);
    T_end = sorted[count ? last : K - 1] >> 10;
  }
  int rank_in_warp = 0;
  if (net) {
    // network models: group the arrivals by staleness (all members of a group read the same
    // ring slot); inside a group keep arrival order.  Least squares needs no row layout.
    const unsigned peers = __match_any_sync(0xffffffffu, tau);
    rank_in_warp = __popc(peers & ((1u << lane) - 1u));
    if (tau >= 0 && rank_in_warp == 0) sh.wcnt[warp][min(tau, S)] = (unsigned short)__popc(peers);
  }
  if (__syncthreads_or(tid < K && (tau < 0 || tau > S))) {
    // with forced restarts this cannot happen (consumed staleness <= threshold <= S); without
    // them the arrival's model version may have left the ring: the run ends here, before any
    // kernel reads the slot that was overwritten
    if (tid == 0) raise(k.no_restart ? ST_STALE : ST_INTERNAL);
    return 1;
  }
  int row0_me = tid * B, n_rows = K * B;
  if (net) {
    // every warp for itself: per staleness u its count in all warps and in the ones before this one, then first rows by a
    // scan over u (RB is a power of two)
    const int rb1 = (1 << k.rb_shift) - 1, nw = (K + 31) >> 5;
    int carry = 0;
    for (int u0 = 0; u0 <= S; u0 += 32) {
      const int u = u0 + lane;
      int c = 0, before = 0;
      if (u <= S) {
#pragma unroll 4
        for (int w = 0; w < nw; ++w) { const int x = sh.wcnt[w][u]; before += w < warp ? x : 0; c += x; }
      }
      const int rows = (c * B + rb1) & ~rb1;
      int sum = rows;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) { const int x = __shfl_up_sync(0xffffffffu, sum, o); if (lane >= o) sum += x; }
      const int first = carry + sum - rows;
      if (u <= S && warp == 0) { sh.cnt[u] = c; sh.grow0[u] = first; }
      const int mine = __shfl_sync(0xffffffffu, first + before * B, tau & 31);
      if (tau >= 0 && (tau & ~31) == u0) row0_me = mine + rank_in_warp * B;
      carry += __shfl_sync(0xffffffffu, sum, 31);
    }
    n_rows = carry;
  }
  if (tid < K) {
    a.sel[pn][tid] = n;
    a.sel_tau[pn][tid] = tau;
    a.sel_row0[pn][tid] = row0_me;
    sh.row0[tid] = row0_me;
    sh.sel_n[tid] = n;
  }
  if (tid == 0) {
    st->T_end = T_end;
    st->last_id = last;
    st->n_rows = n_rows;
    st->n_row_tiles = net ? n_rows >> k.rb_shift : K;
    st->open = 1;
    RoundInfo info;
    info.n_rows = n_rows; info.K = K; info.t = t; info.diverged = 0;
    a.ri[pn] = info;
    sh.scalar[4] = K; sh.scalar[5] = t;
  }
  if (!net) return 0;           // least squares: no row tiles, minibatches drawn by its own kernel
  __syncthreads();
  // ring slot of every row tile and padding rows, one warp per staleness group
  {
    const int sh_rb = k.rb_shift, RB = 1 << sh_rb, tm = t % (S + 1);
#pragma unroll 1
    for (int g = warp; g <= S; g += NWP) {
      const int c = sh.cnt[g];
      if (c == 0) continue;
      const int r0 = sh.grow0[g], p0 = r0 + c * B, p1 = r0 + ((c * B + RB - 1) & ~(RB - 1));
      const int slot = tm - g < 0 ? tm - g + S + 1 : tm - g;      // (t - g) mod (S + 1); g <= S
#pragma unroll 1
      for (int q = (r0 >> sh_rb) + lane; q < (p1 >> sh_rb); q += 32) {
        a.tile_slot[pn][q] = slot;
        a.tile_real[pn][q] = min(RB, p0 - (q << sh_rb));
      }
#pragma unroll 1
      for (int r = p0 + lane; r < p1; r += 32) a.row_idx[pn][r] = -1;
    }
  }
  if (!a.draw) return 0;
  // minibatch draws: sample b of job (n, j) = word b%4 of Philox block (n, j, 1, b/4),
  // mapped into the worker's shard [n M / N, (n+1) M / N)
  const int blocks_per = (B + 3) >> 2;
#pragma unroll 1
  for (int item = tid; item < K * blocks_per; item += NT) {
    const int i = a.by_blk.div(item), blk = item - i * blocks_per;
    const int wn = sh.sel_n[i];
    uint32_t w4[4];
    philox4x32_10((uint32_t)wn, (uint32_t)sh.job[wn], 1u, (uint32_t)blk, k.key0, k.key1, w4);
    const int2 shard = sh.shard[wn];
    const int row0 = sh.row0[i];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int b = blk * 4 + q;
      if (b < B) a.row_idx[pn][row0 + b] = shard.x + (int)__umulhi(w4[q], (unsigned)shard.y);
    }
  }
  return 0;
}

// pdl = 0: the step waits for the kernel in front of it before it starts.  pdl = 1: the kernel in
// front is the Eq. 3 step of the round being finished, which this step does not depend on (it reads
// the uploaded losses, which were complete before the Eq. 3 kernel passed its own wait, and the job
// durations, which it prepares itself (look, see ctl_round) or the round's gradient kernels have
// prepared: row kernels and least-squares pipeline): the two run side by side, and this kernel waits
// for the Eq. 3 kernel only at its end, so that whatever follows in the stream sees both complete.
// The Eq. 3 kernel does not touch the prepared durations on these paths.
__global__ void __launch_bounds__(1024, 1) abs_ctl_kernel(CtlArgs a, int do_finish, int do_select, int t_sel, int pdl, int look) {
  if (pdl) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  else grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char ctl_smem[];
  CtlShared& sh = *reinterpret_cast<CtlShared*>(ctl_smem);
  __shared__ int late;
  if (threadIdx.x == 0) late = ST_OK;
  ctl_round<1024>(a, sh, do_finish, do_select, t_sel, look, pdl ? &late : nullptr);
  if (pdl) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (threadIdx.x == 0 && late != ST_OK) a.st->status = late;      // the Eq. 3 kernel is done: publish
  }
}

// The same step with 256 threads for runs of at most 256 workers (one thread per worker is all the
// step needs; its block-wide barriers are cheaper with 8 warps than with 32).
__global__ void __launch_bounds__(256, 1) abs_ctl_small_kernel(CtlArgs a, int do_finish, int do_select, int t_sel, int pdl, int look) {
  if (pdl) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  else grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char ctl_smem[];
  CtlShared& sh = *reinterpret_cast<CtlShared*>(ctl_smem);
  __shared__ int late;
  if (threadIdx.x == 0) late = ST_OK;
  ctl_round<256>(a, sh, do_finish, do_select, t_sel, look, pdl ? &late : nullptr);
  if (pdl) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (threadIdx.x == 0 && late != ST_OK) a.st->status = late;      // the Eq. 3 kernel is done: publish
  }
}

// Duration look-ahead (see refresh_next_durations): one warp per 32 workers.
__global__ void abs_times_kernel(const DevState* st, const int* job, u64* next_dur, int* dur_job) {
  grid_dependency_sync();
  if (st->status != ST_OK) return;
  refresh_next_durations(st, job, next_dur, dur_job, blockIdx.x * 32 + threadIdx.x);
}

// Algorithm 1, initialisation: every worker holds w^0 and starts job 0 at tick 0.
__global__ void abs_init_state_kernel(CtlArgs a) {
  DevState* st = a.st;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  if (tid < st->W) {
    const u64 dt = job_ticks(st->dist, st->key0, st->key1, tid, 0);
    if (dt == 0ull) st->status = ST_RANGE;
    const i64 M = st->n_samples, lo = ((i64)tid * M) / st->W, hi = ((i64)(tid + 1) * M) / st->W;
    a.shard[tid] = make_int2((int)lo, (int)(hi - lo));
    a.c[tid] = dt;
    a.version[tid] = 0;
    a.job[tid] = 0;
    a.next_dur[tid] = job_ticks(st->dist, st->key0, st->key1, tid, 1);
    a.dur_job[tid] = 1;
  }
}

}  // namespace absb
