// Integrated autocorrelation time of many series on the device (the paper's
// comparison of samplers by the autocorrelation of the energy, Sec. III and
// Sec. IV).  Windowed estimator with Sokal's automatic window, per series
// x_0 .. x_{n-1}:
//   m = mean, G(t) = (1/n) sum_{s < n-t} (x_s - m)(x_{s+t} - m),
//   tau(W) = 1/2 + sum_{t=1}^{W} G(t)/G(0),  W = first W >= 1 with W >= c tau(W)
// (W <= n-1; a constant series gives tau = 1/2, W = 0).
// One CTA per series, the series (less its mean) in shared memory, up to 32 lags
// to a round until the window closes: the work is O(n W) per series, and what
// bounds it is the FP64 pipe (n W multiply-adds; a warp instruction holds its
// sub-partition's pipe for about 64 cycles).  Each warp takes 16 lags of a
// quarter of the series, a register accumulator per lag, so that the FP64
// additions that bring a round's sums together are 16 for each 16 n / 128
// multiply-adds of a warp instead of a block sum per lag.  1024 series of
// 2000 steps, W about 140: 1.03 ms with the copies (one lag at a time: 6.5 ms).
#include <mutex>

#include "crbm.h"
#include "crbm_device.cuh"
#include "crbm_kernels.h"

namespace crbm {

namespace {

constexpr int kTauThreads = 256;
constexpr int kTauStatic = 4096;                   // of a CTA's shared memory, for the static arrays

constexpr int kLags = 32;                          // lags of a full round
constexpr int kLagTile = 16;                       // most lags of a warp
constexpr int kWarps = kTauThreads / 32;
constexpr int kChunk = 2048;                       // steps staged at a time of a series beyond shared memory

// Sums of TILE accumulators over the warp: the lanes with lane / (32 / TILE) = l
// return accumulator l's total, halving the accumulators at every exchange.
template <int TILE>
__device__ __forceinline__ double warp_sums(double (&a)[TILE], int lane) {
  int o = 16;
#pragma unroll
  for (int h = TILE / 2; h > 0; h >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;               // this lane keeps the upper half
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double send = up ? a[i] : a[i + h], keep = up ? a[i + h] : a[i];
      a[i] = keep + __shfl_xor_sync(kFull, send, o);
    }
  }
#pragma unroll
  for (; o > 0; o >>= 1) a[0] += __shfl_xor_sync(kFull, a[0], o);
  return a[0];
}

// Parts of the sums over t of d_t d_(t + lag), lag = lag0 .. lag0 + TILE GROUPS - 1,
// d the series less its mean: a warp takes TILE lags of every (8 / GROUPS)-th 32
// steps.  SMEM: ds holds the whole series and TILE zeros; else chunks of it and of
// the series lag0 on are staged there (kChunk and kChunk + kLags doubles).
template <bool SMEM, int TILE, int GROUPS>
__device__ __forceinline__ void lag_round(double* ds, const double* col, long long ld, long long n, double m,
                                          long long lag0, double (*part)[kLags]) {
  constexpr int kParts = kWarps / GROUPS;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, grp = warp / kParts, prt = warp % kParts;
  double acc[TILE];
#pragma unroll
  for (int l = 0; l < TILE; ++l) acc[l] = 0.0;
  const long long pairs = n - lag0 - grp * TILE;   // of this warp's first lag
  auto run = [&](const double* a, const double* b, long long steps) {
    for (long long t = 32 * prt + lane; t < steps; t += 32 * kParts) {
      const double d = a[t];
      const double* e = b + t + grp * TILE;
#pragma unroll
      for (int l = 0; l < TILE; ++l) acc[l] = fma(d, e[l], acc[l]);
    }
  };
  if (SMEM) {
    run(ds, ds + lag0, pairs);
  } else {
    double* ds2 = ds + kChunk;
    for (long long c0 = 0; c0 < n - lag0; c0 += kChunk) {
      __syncthreads();
      for (int t = tid; t < kChunk + kLags; t += kTauThreads) {
        const long long t1 = c0 + t, t2 = t1 + lag0;
        if (t < kChunk) ds[t] = t1 < n ? col[t1 * ld] - m : 0.0;
        ds2[t] = t2 < n ? col[t2 * ld] - m : 0.0;
      }
      __syncthreads();
      run(ds, ds2, pairs - c0 < kChunk ? pairs - c0 : kChunk);
    }
  }
  const double tot = warp_sums<TILE>(acc, lane);
  if ((lane & (32 / TILE - 1)) == 0) part[prt][grp * TILE + lane / (32 / TILE)] = tot;
}

// Series j of a time-major [n][n_series] array.  SMEM: the series less its
// mean fits shared memory (n + kLagTile doubles, the last kLagTile zero);
// otherwise it is read from global memory.  Rounds of 4, 4, 8 and 16 lags
// come before those of 32: the window of a series of nearly independent steps closes
// within a few lags (200000 steps of white noise, W = 3, with the copies: 0.87 ms;
// 3.92 with rounds of 32 alone, 0.95 lag by lag).
template <bool SMEM>
__global__ void __launch_bounds__(kTauThreads) tau_kernel(const double* __restrict__ x, int n_series, long long n,
                                                         double c, double* tau_out, long long* w_out) {
  extern __shared__ __align__(16) double ds[];
  __shared__ double sc[kTauThreads / 32];
  __shared__ double part[kWarps][kLags];
  __shared__ double tau_sh;
  __shared__ long long w_sh;
  const int j = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double* col = x + j;
  const long long ld = n_series;
  double s = 0.0;
  for (long long t = tid; t < n; t += kTauThreads) {
    const double v = col[t * ld];
    if (SMEM) ds[t] = v;
    s += v;
  }
  const double m = block_sum(s, sc) / (double)n;
  double q = 0.0;
  for (long long t = tid; t < n; t += kTauThreads) {
    const double d = (SMEM ? ds[t] : col[t * ld]) - m;
    if (SMEM) ds[t] = d;
    q = fma(d, d, q);
  }
  if (SMEM && tid < kLagTile) ds[n + tid] = 0.0;
  const double g0 = block_sum(q, sc) / (double)n;
  double tau = 0.5;
  long long W = 0;
  if (n >= 2 && g0 != 0.0) {
    W = n - 1;
    int lags = 4;
    for (long long lag0 = 1; lag0 < n; lag0 += lags, lags = (int)(lag0 - 1 < kLags ? lag0 - 1 : kLags)) {
      if (lags == 4) lag_round<SMEM, 4, 1>(ds, col, ld, n, m, lag0, part);
      else if (lags == 8) lag_round<SMEM, 8, 1>(ds, col, ld, n, m, lag0, part);
      else if (lags == 16) lag_round<SMEM, 16, 1>(ds, col, ld, n, m, lag0, part);
      else lag_round<SMEM, kLagTile, 2>(ds, col, ld, n, m, lag0, part);
      __syncthreads();
      if (warp == 0) {
        // lane = lag: G(lag)/G(0), then the running sum over the lags
        const long long lag = lag0 + lane;
        const bool on = lane < lags && lag < n;
        double p = 0.0;
        for (int w = 0; w < (lags == kLags ? kWarps / 2 : kWarps); ++w) p += part[w][lane];
        double r = on ? (p / (double)n) / g0 : 0.0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const double y = __shfl_up_sync(kFull, r, o);
          if (lane >= o) r += y;
        }
        const double tl = tau + r;
        const unsigned closed = __ballot_sync(kFull, on && (double)lag >= c * tl);
        const int at = closed ? __ffs(closed) - 1 : 31;
        const double t_at = __shfl_sync(kFull, tl, at);
        if (lane == 0) {
          tau_sh = t_at;
          w_sh = closed ? lag0 + at : 0;
        }
      }
      __syncthreads();
      tau = tau_sh;
      if (w_sh != 0) {
        W = w_sh;
        break;
      }
    }
  }
  if (tid == 0) {
    tau_out[j] = tau;
    w_out[j] = W;
  }
}

// Fixed device scratch of the no-allocation variant (crbm_autocorr_noalloc):
// tau[kMaxNoAllocSeries] FP64 followed by W[kMaxNoAllocSeries] int64, 256 KiB
// per device.  Each call's kernel writes every entry that the call copies
// back before the copy, so nothing in it has to start at zero.  All calls on
// a device share it: calls that overlap in time race.
constexpr int kMaxNoAllocSeries = CRBM_AUTOCORR_NOALLOC_MAX_SERIES;
static __device__ __align__(256) unsigned char g_tau_scratch[kMaxNoAllocSeries * 16];

}  // namespace

// The kernel's limit is the process's, so it is set once to the most that any
// call takes (with a context's creation), not by each call to its own size:
// another thread's call between that and the launch would lower it.
cudaError_t tau_set_smem_limit(size_t optin) {
  return cudaFuncSetAttribute(tau_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)optin - kTauStatic);
}

static cudaError_t launch_tau_kernel(const double* x, int n_series, long long n, double c, double* tau, long long* w,
                                     cudaStream_t st) {
  // a series that does not fit the shared memory of a CTA is read from global memory
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  const long long bytes = (n + kLagTile) * 8;
  if (bytes > optin - kTauStatic) {
    tau_kernel<false><<<n_series, kTauThreads, (2 * kChunk + kLags) * 8, st>>>(x, n_series, n, c, tau, w);
    return cudaGetLastError();
  }
  tau_kernel<true><<<n_series, kTauThreads, (size_t)bytes, st>>>(x, n_series, n, c, tau, w);
  return cudaGetLastError();
}

cudaError_t launch_tau(const double* x, int n_series, long long n, double c, double* tau, long long* w,
                       cudaStream_t st) {
  if (n_series == 0) return cudaSuccess;
  return launch_tau_kernel(x, n_series, n, c, tau, w, st);
}

// Address of the scratch array on the current device, looked up once per
// device (cudaGetSymbolAddress; the first lookup on a device must not happen
// while a stream capture is in progress on it) and cached.
static cudaError_t tau_scratch(unsigned char** out) {
  constexpr int kMaxDevices = 64;
  static std::mutex mu;
  static unsigned char* addr[kMaxDevices] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_tau_scratch);
    if (e != cudaSuccess) return e;
    addr[dev] = (unsigned char*)p;
  }
  *out = addr[dev];
  return cudaSuccess;
}

cudaError_t launch_tau_noalloc(const double* x, int n_series, long long n, double c, double* tau_host,
                               int64_t* w_host, cudaStream_t st) {
  if (n_series <= 0) return cudaSuccess;
  if (n_series > kMaxNoAllocSeries) return cudaErrorInvalidValue;
  unsigned char* base = nullptr;
  cudaError_t e = tau_scratch(&base);
  if (e != cudaSuccess) return e;
  double* d_tau = (double*)base;
  long long* d_w = (long long*)(base + (size_t)kMaxNoAllocSeries * 8);
  e = launch_tau_kernel(x, n_series, n, c, d_tau, d_w, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(tau_host, d_tau, (size_t)n_series * 8, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(w_host, d_w, (size_t)n_series * 8, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e;
}

}  // namespace crbm

// ------------------------------------------------------------------ peak probes
// FMA throughput of the FP32 and FP64 pipes: every thread runs 8 independent
// dependency chains of fused multiply-adds (enough to hide the pipe latency),
// the grid fills every SM several times over; a checksum of all chains is
// stored so that the compiler keeps the work.
namespace crbm {
namespace {

template <typename R>
__global__ void __launch_bounds__(256) fma_probe_kernel(int iters, R a, R b, R* sink) {
  R x[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) x[c] = (R)(threadIdx.x + c) * (R)1e-3;
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int c = 0; c < 8; ++c) x[c] = x[c] * a + b;
  }
  R s = 0;
#pragma unroll
  for (int c = 0; c < 8; ++c) s += x[c];
  sink[blockIdx.x * blockDim.x + threadIdx.x] = s;
}

}  // namespace

// Measured FMA rate (TFLOP/s, 2 flops per FMA) of one precision on the current device.
template <typename R>
static cudaError_t probe_one(int sms, R* sink, cudaStream_t st, double* tflops) {
  const int blocks = sms * 8, threads = 256;
  const int iters = sizeof(R) == 8 ? 256 : 4096;     // about a second of FP64, a quarter of FP32
  cudaEvent_t e0, e1;
  cudaError_t e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  if (e != cudaSuccess) return e;
  fma_probe_kernel<R><<<blocks, threads, 0, st>>>(iters / 8, (R)0.999, (R)1e-4, sink);   // warm-up
  cudaEventRecord(e0, st);
  fma_probe_kernel<R><<<blocks, threads, 0, st>>>(iters, (R)0.999, (R)1e-4, sink);
  cudaEventRecord(e1, st);
  e = cudaEventSynchronize(e1);
  float ms = 0.0f;
  if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (e != cudaSuccess) return e;
  *tflops = 2.0 * 8.0 * (double)iters * blocks * threads / ((double)ms * 1e-3) / 1e12;
  return cudaGetLastError();
}

cudaError_t probe_fma_peaks(int device, double* fp32_tflops, double* fp64_tflops, cudaStream_t st) {
  int sms = 0;
  cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  if (e != cudaSuccess) return e;
  const size_t n = (size_t)sms * 8 * 256;
  double* sink = nullptr;
  e = cudaMalloc(&sink, n * sizeof(double));
  if (e != cudaSuccess) return e;
  e = probe_one<float>(sms, (float*)sink, st, fp32_tflops);
  if (e == cudaSuccess) e = probe_one<double>(sms, sink, st, fp64_tflops);
  cudaStreamSynchronize(st);
  cudaFree(sink);
  return e;
}

}  // namespace crbm
