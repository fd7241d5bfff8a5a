// Stand-alone operation of the round loop: minibatch gradients of the least-squares model for
// several workers at one model, and their mean (Eq. 2 with U = 1, then the sum of Eq. 3).
#include <cstdarg>
#include <cstdio>
#include <mutex>
#include <string>

#include "common.cuh"

using namespace absb;

namespace absb {
void set_last_error(const char* text);   // abs_api.cu: text returned by abs_last_error()
}

namespace {

int op_fail(int code, const char* fmt, ...) {
  char buf[384];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  set_last_error(buf);
  return code;
}

// The workers are dealt to clusters of CL = 8 CTAs: Q CTAs share one worker's rows (Q = 1, 2, 4 or 8), so a cluster
// holds CL / Q workers, and its CTAs' gradient sums are added through distributed shared memory.  With at most CL / Q
// workers the one cluster's sum is the result (a single launch); otherwise every cluster leaves one partial sum and
// op_lsq_reduce_kernel adds those.  The operation is bound by the chain index -> row -> residual -> gradient, i.e. by
// two memory round trips per batch of rows, until n B d reaches a few million elements (then by HBM).
// Measured per call (two kernels with one CTA per worker and scalar loads -> now): n = 1, B = 256, d = 64 fp32 36 -> 8 us
// (host-bound from here on down); n = 64, B = 64, d = 512 fp32 27 -> 10; n = 8, B = 64, d = 4096 bf16 147 -> 10;
// n = 256, B = 256: d = 256 bf16 62 -> 12, d = 2048 bf16 399 -> 110, d = 4096 fp32 1245 -> 581.
constexpr int CL = 8, OP_NT = 256, OP_NW = OP_NT / 32;
constexpr int OP_SMEM_D = 8192;       // features whose per-CTA sum is kept in shared memory

struct OpArgs {
  const void* X; const float* y; const void* w; const int* idx;
  int n, B, d, Q;
  float* partial;                     // [clusters][d], or [workers][d] (Q = 1) when `direct`
  float* loss; float* g;
  int single;                         // one cluster: write g itself
  int direct;                         // d > OP_SMEM_D: no cluster, every CTA writes its worker's sum to `partial`
};

__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float ld_peer(const float* p, int rank) {       // *p of CTA `rank` of the cluster
  uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(r) : "memory");
  return v;
}

// VE consecutive stored values as loaded, and as binary32
template <typename T, int VE> struct Vec;
template <> struct Vec<float, 4> {
  float4 q;
  __device__ __forceinline__ void load(const float* p) { q = __ldg(reinterpret_cast<const float4*>(p)); }
  __device__ __forceinline__ void zero() { q = make_float4(0.f, 0.f, 0.f, 0.f); }
  __device__ __forceinline__ void get(float (&v)[4]) const { v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w; }
};
template <> struct Vec<__nv_bfloat16, 8> {
  uint4 q;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { q = __ldg(reinterpret_cast<const uint4*>(p)); }
  __device__ __forceinline__ void zero() { q = make_uint4(0u, 0u, 0u, 0u); }
  __device__ __forceinline__ void get(float (&v)[8]) const {
    const uint32_t u[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) { v[2 * j] = __uint_as_float(u[j] << 16); v[2 * j + 1] = __uint_as_float(u[j] & 0xffff0000u); }
  }
};
template <typename T> struct Vec<T, 1> {
  T q;
  __device__ __forceinline__ void load(const T* p) { q = *p; }
  __device__ __forceinline__ void zero() { q = (T)0.f; }
  __device__ __forceinline__ void get(float (&v)[1]) const { v[0] = (float)q; }
};

// End of both kernels: this CTA's loss share is the sum of lw[] over its warps, its gradient sum is red[0..d).
__device__ __forceinline__ void op_finish(const OpArgs& a, float* red, float* lw, float* lsum, int rank, int cluster) {
  const int tid = threadIdx.x;
  if (tid == 0) {
    float tot = 0.f;
    for (int q = 0; q < OP_NW; ++q) tot += lw[q];
    *lsum = tot;
  }
  cluster_sync();
  const int i = cluster * (CL / a.Q) + rank / a.Q;
  if (tid == 0 && rank % a.Q == 0 && i < a.n) {
    float tot = *lsum;
    for (int q = 1; q < a.Q; ++q) tot += ld_peer(lsum, rank + q);
    a.loss[i] = __fdiv_rn(tot, (float)a.B);
  }
  float* out = a.single ? a.g : a.partial + (size_t)cluster * a.d;
  const float div = (float)((long long)a.n * a.B);
  const int share = (a.d + CL - 1) / CL;
  for (int j = rank * share + tid; j < min(a.d, (rank + 1) * share); j += OP_NT) {
    float v[CL];
#pragma unroll
    for (int q = 0; q < CL; ++q) v[q] = ld_peer(red + j, q);
    float acc = 0.f;
#pragma unroll
    for (int q = 0; q < CL; ++q) acc += v[q];
    out[j] = a.single ? acc / div : acc;
  }
  cluster_sync();                     // nobody leaves while a peer reads its shared memory
}

// Rows in registers: a warp takes a row (lane l holds vectors l, l + 32, ... of VE elements), forms the residual and
// adds r x into its running sum; IT rows per warp are loaded back to back.  Every row is read once.
template <typename T, int VE, int NV>
__global__ void __launch_bounds__(OP_NT) op_lsq_rows_kernel(OpArgs a) {
  constexpr int IT = NV >= 8 ? 1 : 8 / NV;
  extern __shared__ float osm[];       // [OP_NW / 2][d] gradient sums of the warps
  __shared__ float lw[OP_NW], lsum;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)(blockIdx.x % CL), cluster = (int)(blockIdx.x / CL);
  const int Q = a.Q, B = a.B, d = a.d, nvec = d / VE;
  const int i = cluster * (CL / Q) + rank / Q, sub = rank % Q;
  const T* X = (const T*)a.X;
  const T* w = (const T*)a.w;
  grid_wait();
  grid_go();
  float acc[NV][VE];
#pragma unroll
  for (int k = 0; k < NV; ++k)
#pragma unroll
    for (int j = 0; j < VE; ++j) acc[k][j] = 0.f;
  float loss = 0.f;
  if (i < a.n) {
    Vec<T, VE> wv[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      if (lane + 32 * k < nvec) wv[k].load(w + (lane + 32 * k) * VE);
      else wv[k].zero();
    }
    const int* idx = a.idx + (size_t)i * B;
    for (int b0 = sub * OP_NW + warp; b0 < B; b0 += IT * Q * OP_NW) {
      // lane k fetches index and target of row b0 + k Q OP_NW
      const int mine = b0 + lane * Q * OP_NW;
      const int s = (lane < IT && mine < B) ? idx[mine] : -1;
      const float yv = s >= 0 ? a.y[s] : 0.f;
      Vec<T, VE> x[IT][NV];
#pragma unroll
      for (int t = 0; t < IT; ++t) {
        const int r = __shfl_sync(0xffffffffu, s, t);
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          if (r >= 0 && lane + 32 * k < nvec) x[t][k].load(X + (size_t)r * d + (lane + 32 * k) * VE);
          else x[t][k].zero();
        }
      }
#pragma unroll
      for (int t = 0; t < IT; ++t) {
        float dot = 0.f;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          float xv[VE], wf[VE];
          x[t][k].get(xv);
          wv[k].get(wf);
#pragma unroll
          for (int j = 0; j < VE; ++j) dot = fmaf(xv[j], wf[j], dot);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
        // (a row that is absent adds nothing, also where the weights are not finite and 0 w is a NaN)
        const float target = __shfl_sync(0xffffffffu, yv, t);
        const float res = __shfl_sync(0xffffffffu, s, t) >= 0 ? dot - target : 0.f;
        loss = fmaf(0.5f * res, res, loss);
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          float xv[VE];
          x[t][k].get(xv);
#pragma unroll
          for (int j = 0; j < VE; ++j) acc[k][j] = fmaf(res, xv[j], acc[k][j]);
        }
      }
    }
  }
  if (lane == 0) lw[warp] = loss;
  // warps 4..7 leave their sums, warps 0..3 add theirs, then the four are added in order
  float* mine = osm + (size_t)(warp & 3) * d;
#pragma unroll
  for (int h = 1; h >= 0; --h) {
    if ((warp >> 2) == h) {
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const int v = lane + 32 * k;
        if (v < nvec) {
#pragma unroll
          for (int j = 0; j < VE; ++j) mine[v * VE + j] = h ? acc[k][j] : acc[k][j] + mine[v * VE + j];
        }
      }
    }
    __syncthreads();
  }
  for (int j = tid; j < d; j += OP_NT) osm[j] = (osm[j] + osm[d + j]) + (osm[2 * d + j] + osm[3 * d + j]);
  op_finish(a, osm, lw, &lsum, rank, cluster);
}

// Rows too long for that: a residual pass (one warp per row) and a gradient pass (one thread per VE columns, all rows
// of the CTA; the rows come from L2 now).
template <typename T, int VE>
__global__ void __launch_bounds__(OP_NT) op_lsq_long_kernel(OpArgs a) {
  extern __shared__ float osm[];       // [d] gradient sum of the CTA (not when `direct`)
  __shared__ float res[1024];
  __shared__ int sidx[1024];
  __shared__ float lw[OP_NW], lsum;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = a.direct ? 0 : (int)(blockIdx.x % CL), cluster = (int)(blockIdx.x / CL);
  const int Q = a.Q, B = a.B, d = a.d, nvec = d / VE;
  const int i = a.direct ? (int)blockIdx.x : cluster * (CL / Q) + rank / Q, sub = rank % Q;
  const int nb = i < a.n ? (B - sub + Q - 1) / Q : 0;                 // rows sub, sub + Q, ... of worker i
  const T* X = (const T*)a.X;
  const T* w = (const T*)a.w;
  grid_wait();
  grid_go();
  for (int b = tid; b < nb; b += OP_NT) sidx[b] = a.idx[(size_t)i * B + sub + b * Q];
  __syncthreads();
  float loss = 0.f;
  for (int b = warp; b < nb; b += OP_NW) {
    const T* x = X + (size_t)sidx[b] * d;
    const float yv = a.y[sidx[b]];
    float dot = 0.f;
#pragma unroll 8
    for (int v = lane; v < nvec; v += 32) {
      Vec<T, VE> xq, wq;
      xq.load(x + v * VE);
      wq.load(w + v * VE);
      float xv[VE], wv[VE];
      xq.get(xv);
      wq.get(wv);
#pragma unroll
      for (int j = 0; j < VE; ++j) dot = fmaf(xv[j], wv[j], dot);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    const float r = dot - yv;
    if (lane == 0) res[b] = r;
    loss = fmaf(0.5f * r, r, loss);
  }
  if (lane == 0) lw[warp] = loss;
  __syncthreads();
  float* out = a.direct ? a.partial + (size_t)i * d : osm;
  for (int v = tid; v < nvec; v += OP_NT) {
    float acc[VE];
#pragma unroll
    for (int j = 0; j < VE; ++j) acc[j] = 0.f;
#pragma unroll 8
    for (int b = 0; b < nb; ++b) {
      Vec<T, VE> xq;
      xq.load(X + (size_t)sidx[b] * d + v * VE);
      float xv[VE];
      xq.get(xv);
#pragma unroll
      for (int j = 0; j < VE; ++j) acc[j] = fmaf(res[b], xv[j], acc[j]);
    }
#pragma unroll
    for (int j = 0; j < VE; ++j) out[v * VE + j] = acc[j];
  }
  if (a.direct) {
    if (tid == 0) {
      float tot = 0.f;
      for (int q = 0; q < OP_NW; ++q) tot += lw[q];
      a.loss[i] = __fdiv_rn(tot, (float)B);
    }
    return;
  }
  op_finish(a, osm, lw, &lsum, rank, cluster);
}

// g[j] = (1 / (n B)) sum_p partial[p][j]: block = 32 features x 8 lanes; lane w adds partials w, w + 8, ... in order,
// then the 8 lanes are added in order.
__global__ void __launch_bounds__(256) op_lsq_reduce_kernel(const float* partial, int parts, float div, int d, float* g) {
  __shared__ float red[8][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int j = blockIdx.x * 32 + lane;
  grid_wait();
  grid_go();
  float acc = 0.f;
  if (j < d) {
#pragma unroll 8
    for (int p = w; p < parts; p += 8) acc += partial[(size_t)p * d + j];
  }
  red[w][lane] = acc;
  __syncthreads();
  if (w == 0 && j < d) {
    float tot = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) tot += red[q][lane];
    g[j] = tot / div;
  }
}

int check_args(const void* X, const float* y, const void* w, const int* idx, int n, int B, int d, int dtype,
               const float* g_out, const float* loss_out) {
  if (!X || !y || !w || !idx || !g_out || !loss_out) return op_fail(ABS_EINVAL, "null pointer argument");
  if (n < 1 || n > ABS_MAX_WORKERS) return op_fail(ABS_EINVAL, "n %d outside [1, %d]", n, ABS_MAX_WORKERS);
  if (B < 1 || B > 1024) return op_fail(ABS_EINVAL, "B %d outside [1, 1024]", B);
  if (d < 1 || d > (1 << 20)) return op_fail(ABS_EINVAL, "d %d outside [1, 2^20]", d);
  if (dtype != ABS_FP32 && dtype != ABS_BF16_FP32MASTER) return op_fail(ABS_EUNSUPPORTED, "unknown dtype %d", dtype);
  return ABS_OK;
}

// Launch that may start while the kernel in front of it drains; all kernels of this file wait for it before they
// read anything.
template <typename... KArgs, typename... Args>
cudaError_t op_launch(void (*kernel)(KArgs...), int grid, size_t smem, int cluster, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(OP_NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// the kernel for rows of d elements in vectors of VE: rows in registers up to 32 x 8 vectors
template <typename T, int VE>
void (*op_kernel(int d, size_t* smem))(OpArgs) {
  const int nvec = d / VE;
  *smem = (size_t)OP_NW / 2 * d * 4;
  if (nvec <= 32) return op_lsq_rows_kernel<T, VE, 1>;
  if (nvec <= 64) return op_lsq_rows_kernel<T, VE, 2>;
  if (nvec <= 128) return op_lsq_rows_kernel<T, VE, 4>;
  if (nvec <= 256) return op_lsq_rows_kernel<T, VE, 8>;
  *smem = d <= OP_SMEM_D ? (size_t)d * 4 : 0;
  return op_lsq_long_kernel<T, VE>;
}

int run(const void* X, const float* y, const void* w, const int* idx, int n, int B, int d, int dtype, float* scratch,
        float* g_out, float* loss_out, cudaStream_t s) {
  const int esz = dtype == ABS_FP32 ? 4 : 2;
  const bool vec = (((uintptr_t)X | (uintptr_t)w | ((uintptr_t)d * esz)) & 15) == 0;    // rows on 16-byte boundaries
  OpArgs a = {X, y, w, idx, n, B, d, 1, scratch, loss_out, g_out, 0, d > OP_SMEM_D ? 1 : 0};
  // CTAs per worker: enough for two per SM, at least a row per warp
  while (!a.direct && a.Q < CL && n * a.Q * 2 <= 2 * PLAN_SMS && B >= 2 * a.Q * OP_NW) a.Q *= 2;
  const int per = CL / a.Q, clusters = (n + per - 1) / per;
  a.single = !a.direct && clusters == 1 ? 1 : 0;
  size_t smem = 0;
  void (*kernel)(OpArgs) =
      dtype == ABS_FP32 ? (vec ? op_kernel<float, 4>(d, &smem) : op_kernel<float, 1>(d, &smem))
                        : (vec ? op_kernel<__nv_bfloat16, 8>(d, &smem) : op_kernel<__nv_bfloat16, 1>(d, &smem));
  cudaError_t e = op_launch(kernel, a.direct ? n : clusters * CL, smem, a.direct ? 1 : CL, s, a);
  if (e == cudaSuccess && !a.single)
    e = op_launch(op_lsq_reduce_kernel, (d + 31) / 32, 0, 1, s, (const float*)scratch, a.direct ? n : clusters,
                  (float)((long long)n * B), d, g_out);
  if (e != cudaSuccess) return op_fail(ABS_ECUDA, "kernel launch: %s", cudaGetErrorString(e));
  return ABS_OK;
}

}  // namespace

extern "C" int abs_lsq_gradient(const void* X, const float* y, const void* w, const int* idx, int n, int B, int d,
                                int dtype, float* scratch, size_t scratch_floats, float* g_out, float* loss_out,
                                void* stream) {
  const int rc = check_args(X, y, w, idx, n, B, d, dtype, g_out, loss_out);
  if (rc != ABS_OK) return rc;
  if (!scratch) return op_fail(ABS_EINVAL, "scratch is null");
  if (scratch_floats < (size_t)n * d)
    return op_fail(ABS_ENOSPACE, "scratch holds %zu floats, n*d = %zu needed", scratch_floats, (size_t)n * d);
  return run(X, y, w, idx, n, B, d, dtype, scratch, g_out, loss_out, (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------------------------
// Variant for callers that cannot allocate device memory.  The per-worker partial sums live in a
// fixed array that is part of the loaded library image on every GPU (4 MiB, held until exit).
namespace {

constexpr size_t NOALLOC_MAX_FLOATS = 1u << 20;          // n * d limit of the no-allocation variant
static __device__ __align__(256) float g_noalloc_partials[NOALLOC_MAX_FLOATS];

constexpr int MAX_DEVICES = 64;
std::mutex g_noalloc_mutex;
float* g_noalloc_ptr[MAX_DEVICES] = {};                  // device address of the array, per device

// Device address of the array on the current device.  In host code the array's name is only a
// handle; the address a kernel can use comes from cudaGetSymbolAddress, looked up once per device.
int noalloc_scratch(float** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return op_fail(ABS_ECUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
  if (dev < 0 || dev >= MAX_DEVICES) return op_fail(ABS_EUNSUPPORTED, "device index %d not supported", dev);
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (!g_noalloc_ptr[dev]) {
    float* p = nullptr;
    e = cudaGetSymbolAddress((void**)&p, g_noalloc_partials);
    if (e != cudaSuccess || !p)
      return op_fail(ABS_ECUDA, "cudaGetSymbolAddress(partials): %s", cudaGetErrorString(e));
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return ABS_OK;
}

}  // namespace

extern "C" int abs_lsq_gradient_noalloc(const void* X, const float* y, const void* w, const int* idx, int n, int B,
                                        int d, int dtype, float* g_out, float* loss_out, void* stream) {
  const int rc = check_args(X, y, w, idx, n, B, d, dtype, g_out, loss_out);
  if (rc != ABS_OK) return rc;
  if ((size_t)n * (size_t)d > NOALLOC_MAX_FLOATS)
    return op_fail(ABS_ENOSPACE, "n*d = %zu exceeds the built-in limit of %zu floats; use abs_lsq_gradient with "
                   "caller scratch", (size_t)n * d, NOALLOC_MAX_FLOATS);
  float* scratch = nullptr;
  const int rs = noalloc_scratch(&scratch);
  if (rs != ABS_OK) return rs;
  // every partial that the reduction reads is written by the first kernel of this call, so the
  // previous call's leftovers in the shared array never need clearing
  return run(X, y, w, idx, n, B, d, dtype, scratch, g_out, loss_out, (cudaStream_t)stream);
}
