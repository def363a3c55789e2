// The paper's CRBM trainer on the device (Sec. II, App. A, Algorithm 1):
// epochs of minibatch ADAM steps on the energy-matching loss
//   diff_i = t_i - F(x_i),  C = mean diff,  loss = mean (diff_i - C)^2,
//   d loss/d theta = (2/M) sum_i (diff_i - C) [ sum_ij sigma(a^f_ij) v_(i+a)(j+b),
//                                               sum_ij v_ij,  sum_ij sigma(a^f_ij) ]
// (the W, v_bias, h_bias components; sum_i (diff_i - C) = 0 removes C's own
// dependence on theta), then ADAM (Kingma & Ba 2014).  Everything is FP64.
//
// One cluster of CTAs per training problem (the paper trains one CRBM per
// temperature): minibatch steps depend on each other through the parameters,
// so a problem runs its steps in order, the samples of a minibatch divided
// over the cluster's CTAs; independent problems fill the GPU side by side.
// Every CTA keeps the parameters, ADAM moments and row-sum tables of the
// current filters in its own shared memory and updates them alike (the same
// additions in the same order), so that a step needs two cluster barriers:
// after F of every sample (read from the owners' shared memory) and after the
// CTAs' gradient sums.
//
// What bounds it: the FP64 pipe (a warp instruction holds its sub-partition's
// pipe for about 64 cycles on GB300) and the serial chain of a step.  Hence:
//   - the sum of log(1 + e^-|x|) of a warp's units is the log of their product:
//     two operations per unit (join_log1p) instead of a log1p;
//   - the gradient's sums over sites are exact 96-bit fixed-point additions of
//     the FP64 sigma(a) off the FP64 pipe (WideSum), in FP64 for samples with a
//     unit below their range;
//   - the bias corrections 1 / (1 - b^t) are taken for 32 steps at a time, one
//     step per lane (a pow per thread and step was a third of the epoch);
//   - the next minibatch's samples and targets are fetched during a step.
// K = 2 5x5, L = 8, 10^4 samples, batch 20: 24 problems 9.4 ms per epoch
// (one 512-thread CTA per problem, log1p and pow per unit and thread, FP64
// gradient sums: 69.3 ms).
#include <algorithm>

#include <cooperative_groups.h>

#include "crbm.h"
#include "crbm_device.cuh"
#include "crbm_kernels.h"

namespace crbm {

namespace {

namespace cg = cooperative_groups;

constexpr int kTrainThreads = 512;
constexpr int kTrainWarps = kTrainThreads / 32;
constexpr int kMaxCluster = 8;             // portable cluster size
constexpr int kMaxBatch = 64;
constexpr size_t kSigBudget = 96 * 1024;   // shared memory for hidden probabilities

struct TrainParams {
  int batch, per;                          // samples of a minibatch, of a CTA
  double lr, b1, b2, eps;
  crbm_train_problem pr[CRBM_TRAIN_MAX_PROBLEMS];
};

// Samples whose hidden probabilities fit the shared buffer at once.
__host__ __device__ inline int sig_capacity(int K, int N) {
  const size_t per = (size_t)K * N * 8;
  const size_t c = kSigBudget / per;
  return c < 1 ? 1 : (int)c;
}

// Shared memory of a CTA that takes `per` samples of each minibatch of M
// (offsets in bytes; 8-byte arrays first).
struct TrainLayout {
  int th, am, av, gr, tab, F, cw, tgt, spos, sprod, rbc, part, sig, ord, bits, total;
};
__host__ __device__ inline TrainLayout train_layout(int K, int k, int L, int M, int per) {
  const int N = L * L, P = K * k * k + 1 + K, Wd = (N + 31) / 32, cap = sig_capacity(K, N);
  TrainLayout y;
  int o = 0;
  auto take = [&](int bytes) {
    const int at = o;
    o += (bytes + 7) & ~7;
    return at;
  };
  y.th = take(P * 8);
  y.am = take(P * 8);
  y.av = take(P * 8);
  y.gr = take(P * 8);                                // this CTA's gradient sum
  y.tab = take(K * k * (1 << k) * 8);
  y.F = take(per * 8);
  y.cw = take(per * 8);                              // (2/M)(diff_i - C)
  y.tgt = take(2 * M * 8);                           // targets, this minibatch's and the next
  y.spos = take((kMaxBatch > kTrainWarps ? kMaxBatch : kTrainWarps) * 8);
  y.sprod = take((kMaxBatch > kTrainWarps ? kMaxBatch : kTrainWarps) * 8);
  y.rbc = take(2 * 32 * 8);                          // 1 / (1 - b^t) of 32 steps
  y.part = take(kTrainThreads * 8);                  // gradient partials
  y.sig = take((per < cap ? per : cap) * K * N * 8);
  y.ord = take(3 * M * 4);                           // visiting order of three minibatches
  y.bits = take(2 * (per * Wd + 1) * 4);             // lattices (one word of padding each)
  y.total = o;
  return y;
}

__device__ __forceinline__ double warp_sum64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "n"(BYTES)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Exact sum of up to 1024 FP64 values in [kWideMin, 1]: 96-bit fixed point in
// units of 2^-84, so every bit of every value counts whatever the others' size.  Ten
// integer instructions an addition, where an FP64 one holds the pipe for 64 cycles
// (epoch of 24 problems, K = 2 5x5, L = 8: 9.4 ms, about 12 with FP64 sums).
constexpr int kWideMinHi = (1023 - 31) << 20;      // high word of 2^-31
struct WideSum {
  uint32_t w1 = 0u, w2 = 0u, w3 = 0u;
  // adds x if on != 0
  __device__ __forceinline__ void add(double x, uint32_t on) {
    // the 53-bit mantissa, 32 zero bits below it, shifted down by 0 <= sh <= 31
    const uint32_t xh = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t sh = 1023u - (xh >> 20), hi = (xh & 0xFFFFFu) | 0x100000u;
    asm("{\n.reg .pred p;\nsetp.ne.u32 p, %6, 0;\n@p add.cc.u32 %0, %0, %3;\n@p addc.cc.u32 %1, %1, %4;\n@p addc.u32 %2, %2, %5;\n}\n"
        : "+r"(w1), "+r"(w2), "+r"(w3)
        : "r"(__funnelshift_r(0u, lo, sh)), "r"(__funnelshift_r(lo, hi, sh)), "r"(hi >> (sh & 31u)), "r"(on));
  }
  __device__ __forceinline__ double value() const {
    return fma((double)(((unsigned long long)w3 << 32) | w2), 0x1p-52, (double)w1 * 0x1p-84);
  }
};

// Warps per sample of unit_pass for ns samples, and the hidden units (a
// multiple of 32) each takes of the sample's K N.
__device__ __forceinline__ int segments(int ns) { return ns >= kTrainWarps ? 1 : kTrainWarps / ns; }

// Hidden units of samples [i0, i1): SEG warps per sample, lanes over its
// units (f, site).  sig[(i - i0) K N + unit] = sigma(a) of the
// samples below i0 + cap; with WANT_F also, per (sample, segment), softplus a =
// log(1 + e^a) as a product of the factors, less 1, in sprod, or, where a is above
// the bound that keeps the product below e^700, as a in spos and the factor
// 1 + e^-a (spos is rarely needed, and so is its sum over the lanes).  Segments
// longer than 960 units take their lanes' logs first.  Bit i of tiny: sample i
// holds a sigma below kWideMin.
template <bool WANT_F>
__device__ void unit_pass(const uint32_t* vb, int Wd, const double* tab, const double* hbias, int K, int k, int T,
                          int L, int i0, int i1, int cap, double* sig, double* spos, double* sprod, unsigned* tiny) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, N = L * L, U = K * N;
  const int SEG = segments(i1 - i0), span = ((U + SEG - 1) / SEG + 31) & ~31;
  // n factors of at most 1 + e^top < 2 e^top
  const double top = (double)(__fdividef(700.0f, (float)(span > 960 ? span / 32 : span)) - 0.7f);
  for (int task = warp; task < (i1 - i0) * SEG; task += kTrainWarps) {
    const int i = i0 + task / SEG, u0 = (task % SEG) * span, u1 = min(U, u0 + span);
    const uint32_t* v = vb + i * Wd;
    const bool keep = i - i0 < cap;
    double pos = 0.0, prod = 0.0;
    bool small = false;
    for (int u = u0 + lane; u < u1; u += 32) {
      const int f = u / N, s = u - f * N, si = s / L, sj = s - si * L;
      double x = hbias[f];
      for (int a = 0; a < k; ++a) {
        const int r = si + a < L ? si + a : si + a - L;
        x += tab[(f * k + a) * T + (int)row_window(v, L, r, sj, k)];
      }
      const bool up = x <= top;
      const double e = exp(up ? x : -x), d = 1.0 + e;
      if (keep) {
        const double y = (up ? e : 1.0) / d;
        sig[(size_t)(i - i0) * U + u] = y;
        small = small || __double2hiint(y) < kWideMinHi;
      }
      if (WANT_F) {
        if (!up) pos += x;
        prod = join_log1p(prod, e);
      }
    }
    if (__any_sync(kFull, small) && lane == 0) atomicOr(tiny + (i >> 5), 1u << (i & 31));
    if (WANT_F) {
      if (span > 960) {
        pos += log_joined(prod);
        prod = 0.0;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) prod = join_log1p(prod, __shfl_xor_sync(kFull, prod, o));
      if (__any_sync(kFull, pos != 0.0)) pos = warp_sum64(pos);
      if (lane == 0) {
        spos[task] = pos;
        sprod[task] = prod;
      }
    }
  }
}

__device__ __forceinline__ int count_ones(const uint32_t* v, int Wd) {
  int c = 0;
  for (int w = 0; w < Wd; ++w) c += __popc(v[w]);
  return c;
}

// Sum of sp[si L + j] over the sites of rows si = s0, s0 + step, .. whose bit j of
// row(si) is set.
template <class ROW>
__device__ __forceinline__ double site_sum(const double* sp, int L, int s0, int step, bool exact, ROW row) {
  WideSum wide;
  double sum = 0.0;
  for (int si = s0; si < L; si += step) {
    const double* x = sp + si * L;
    const uint32_t win = row(si);
    if (exact) {
#pragma unroll 8
      for (int j = 0; j < L; ++j) wide.add(x[j], win & (1u << j));
    } else {
      double part = 0.0;
      for (int j = 0; j < L; ++j)
        if ((win >> j) & 1u) part += x[j];
      sum += part;
    }
  }
  return exact ? wide.value() : sum;
}

__global__ void __launch_bounds__(kTrainThreads, 1) train_epoch_kernel(const __grid_constant__ TrainParams p) {
  cg::cluster_group cl = cg::this_cluster();
  const int CL = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const crbm_train_problem& q = p.pr[blockIdx.x / CL];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int K = q.K, k = q.k, L = q.L, N = L * L, T = 1 << k, Wd = (N + 31) / 32;
  const int nW = K * k * k, P = nW + 1 + K, nlut = K * k * T, U = K * N;
  const int M = p.batch, per = p.per, cap = sig_capacity(K, N);

  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned tiny[kMaxBatch / 32];
  const TrainLayout y = train_layout(K, k, L, M, per);
  double* th = (double*)(smem + y.th);
  double* am = (double*)(smem + y.am);
  double* av = (double*)(smem + y.av);
  double* gr = (double*)(smem + y.gr);
  double* tab = (double*)(smem + y.tab);
  double* Fs = (double*)(smem + y.F);
  double* cw = (double*)(smem + y.cw);
  double* tgt = (double*)(smem + y.tgt);
  double* spos = (double*)(smem + y.spos);
  double* sprod = (double*)(smem + y.sprod);
  double* rbc = (double*)(smem + y.rbc);
  double* part = (double*)(smem + y.part);
  double* sig = (double*)(smem + y.sig);
  int* ord = (int*)(smem + y.ord);
  uint32_t* bits = (uint32_t*)(smem + y.bits);

  const int nb = (q.n_samples + M - 1) / M;
  const int mine = rank * per;                        // this CTA's samples of a minibatch start here
  auto size_of = [&](int b) { return min(M, q.n_samples - b * M); };
  // lattices of this CTA's samples and every sample's target of minibatch b,
  // whose visiting order is in shared memory
  auto fetch = [&](int b) {
    const int Mb = size_of(b), ns = max(min(Mb, mine + per) - mine, 0), buf = b & 1;
    const int* o = ord + (b % 3) * M;
    uint32_t* dst = bits + buf * (per * Wd + 1);
    for (int e = tid; e < ns * Wd; e += kTrainThreads) {
      const int i = e / Wd, w = e - i * Wd;
      cp_async<4>(dst + e, q.samples + (size_t)o[mine + i] * Wd + w);
    }
    for (int i = tid; i < Mb; i += kTrainThreads) cp_async<8>(tgt + buf * M + i, q.targets + o[i]);
  };
  auto fetch_order = [&](int b) {
    for (int i = tid; i < size_of(b); i += kTrainThreads) cp_async<4>(ord + (b % 3) * M + i, q.order + (size_t)b * M + i);
  };

  for (int i = tid; i < P; i += kTrainThreads) {
    th[i] = q.theta[i];
    am[i] = q.adam_m[i];
    av[i] = q.adam_v[i];
  }
  if (tid < 2) bits[tid * (per * Wd + 1) + per * Wd] = 0u;
  const long long t0 = *q.adam_t;
  if (nb > 0) fetch_order(0);
  if (nb > 1) fetch_order(1);
  cp_async_wait();
  __syncthreads();
  if (nb > 0) fetch(0);
  cp_async_wait();
  __syncthreads();
  for (int b = 0; b < nb; ++b) {
    const int Mb = size_of(b), ns = max(min(Mb, mine + per) - mine, 0);
    const uint32_t* vb = bits + (b & 1) * (per * Wd + 1);
    const double* tg = tgt + (b & 1) * M;
    // the next minibatch's data and the order of the one after it (waited for at the step's end)
    if (b + 1 < nb) fetch(b + 1);
    if (b + 2 < nb) fetch_order(b + 2);
    if (tid < kMaxBatch / 32) tiny[tid] = 0u;
    // (1) row-sum tables of the current filters (bits summed in increasing b)
    for (int e = tid; e < nlut; e += kTrainThreads) {
      const int code = e % T, fa = e / T;
      double acc = 0.0;
      for (int bb = 0; bb < k; ++bb)
        if ((code >> bb) & 1) acc += th[fa * k + bb];
      tab[e] = acc;
    }
    if ((b & 31) == 0 && warp >= kTrainWarps - 2) {
      // bias corrections of steps t0 + b + 1 .. t0 + b + 32, one per lane
      const int which = warp - (kTrainWarps - 2);
      rbc[which * 32 + lane] = 1.0 / (1.0 - pow(which == 0 ? p.b1 : p.b2, (double)(t0 + b + 1 + lane)));
    }
    __syncthreads();
    const double vbias = th[nW];
    const double* hbias = th + nW + 1;
    // (2) F of this CTA's samples (and the hidden probabilities of the first chunk)
    if (ns > 0) unit_pass<true>(vb, Wd, tab, hbias, K, k, T, L, 0, ns, cap, sig, spos, sprod, tiny);
    __syncthreads();
    if (warp == 0) {
      const int SEG = ns > 0 ? segments(ns) : 1;
      for (int e = lane; e < ns * SEG; e += 32) spos[e] += log_joined(sprod[e]);
      __syncwarp();
      for (int i = lane; i < ns; i += 32) {
        double sp = 0.0;
        for (int g = 0; g < SEG; ++g) sp += spos[i * SEG + g];
        Fs[i] = -vbias * (double)count_ones(vb + i * Wd, Wd) - sp;
      }
    }
    cl.sync();
    if (warp == 0) {
      // C and the loss from every sample's F (from the owner's shared memory)
      double diff[kMaxBatch / 32], sum = 0.0;
#pragma unroll
      for (int h = 0; h < kMaxBatch / 32; ++h) {
        const int i = lane + 32 * h;
        diff[h] = 0.0;
        if (i < Mb) {
          diff[h] = tg[i] - cl.map_shared_rank(Fs, i / per)[i % per];
          sum += diff[h];
        }
      }
      const double C = warp_sum64(sum) / (double)Mb;
      double loss = 0.0;
#pragma unroll
      for (int h = 0; h < kMaxBatch / 32; ++h) {
        const int i = lane + 32 * h;
        const double d = diff[h] - C;
        if (i < Mb) {
          loss = fma(d, d, loss);
          if (i >= mine && i < mine + ns) cw[i - mine] = (2.0 / (double)Mb) * d;
        }
      }
      if (rank == 0 && q.losses) {
        loss = warp_sum64(loss);
        if (lane == 0) q.losses[b] = loss / (double)Mb;
      }
    }
    __syncthreads();
    // (3) this CTA's gradient sums, chunks of samples whose probabilities are
    // in shared memory: thread (parameter, sample group, every RS-th row), sites
    // exactly or, where one is too small for that, row by row in FP64, then cw_i
    // times the sum; the groups' partials added in order
    const int SG = max(1, min(ns, kTrainThreads / P)), RS = min(L, kTrainThreads / P / SG), groups = SG * RS;
    const int pp = tid % P, grp = tid / P, sg = grp % SG, row0 = grp / SG;
    double acc = 0.0;
    for (int i0 = 0; i0 < ns; i0 += cap) {
      const int i1 = min(ns, i0 + cap);
      if (i0 > 0) {
        // the first pass kept the probabilities of the first chunk only: recompute this one
        __syncthreads();
        unit_pass<false>(vb, Wd, tab, hbias, K, k, T, L, i0, i1, cap, sig, nullptr, nullptr, tiny);
        __syncthreads();
      }
      if (grp < groups) {
        for (int i = i0 + sg; i < i1; i += SG) {
          const uint32_t* v = vb + i * Wd;
          const bool exact = ((tiny[i >> 5] >> (i & 31)) & 1u) == 0u;
          if (pp == nW) {
            if (row0 == 0) acc = fma(cw[i], (double)count_ones(v, Wd), acc);
            continue;
          }
          // W^f_ab: the sites whose v at (si + a, j + b), periodic, is set; h_bias^f: all
          const bool tap = pp < nW;
          const int f = tap ? pp / (k * k) : pp - nW - 1, ab = tap ? pp - f * k * k : 0, a = ab / k, bb = ab - a * k;
          acc = fma(cw[i], site_sum(sig + (size_t)(i - i0) * U + f * N, L, row0, RS, exact, [&](int si) {
            const int r = si + a < L ? si + a : si + a - L;
            const uint32_t lo = row_window(v, L, r, bb, L < 16 ? L : 16);
            const uint32_t hi = L > 16 ? row_window(v, L, r, bb + 16 < L ? bb + 16 : bb + 16 - L, L - 16) : 0u;
            return tap ? lo | (hi << 16) : ~0u;
          }), acc);
        }
      }
    }
    if (grp < groups) part[grp * P + pp] = acc;
    __syncthreads();
    for (int i = tid; i < P; i += kTrainThreads) {
      double s = 0.0;
      for (int g = 0; g < groups; ++g) s += part[g * P + i];
      gr[i] = s;
    }
    cl.sync();
    // (4) the whole gradient (the CTAs' sums in rank order) and ADAM, alike in every CTA
    const double rb1 = rbc[b & 31], rb2 = rbc[32 + (b & 31)];
    for (int i = tid; i < P; i += kTrainThreads) {
      double g = 0.0;
      for (int r = 0; r < CL; ++r) g += cl.map_shared_rank(gr, r)[i];
      const double m = p.b1 * am[i] + (1.0 - p.b1) * g;
      const double w = p.b2 * av[i] + (1.0 - p.b2) * g * g;
      am[i] = m;
      av[i] = w;
      th[i] = th[i] - p.lr * (m * rb1) / (sqrt(w * rb2) + p.eps);
    }
    cp_async_wait();
    __syncthreads();
  }
  if (rank == 0) {
    for (int i = tid; i < P; i += kTrainThreads) {
      q.theta[i] = th[i];
      q.adam_m[i] = am[i];
      q.adam_v[i] = av[i];
    }
    if (tid == 0) *q.adam_t = t0 + nb;
  }
  cl.sync();        // no CTA leaves while another may read its shared memory
}

// CTAs per problem: as many as the SMs allow side by side (the FP64 pipe of an
// SM is what a step waits for, so two CTAs on one SM gain nothing), at most
// the portable cluster size, and no more than leave the largest share of a
// minibatch unchanged.
int cluster_size(int n, int batch) {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int most = std::max(1, std::min({kMaxCluster, sms / n, batch}));
  const int per = (batch + most - 1) / most;
  return (batch + per - 1) / per;
}

}  // namespace

// Shared memory of a CTA that takes a whole minibatch (the most any launch needs).
size_t train_smem_bytes(const crbm_train_problem& q, int batch) {
  return (size_t)train_layout(q.K, q.k, q.L, batch, batch).total;
}

// Once for the process (with a context's creation): a limit set by each call would
// be lowered by another thread's call between that and the launch.
cudaError_t train_set_smem_limit(size_t optin) {
  return cudaFuncSetAttribute(train_epoch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)optin - 1024);
}

cudaError_t launch_train(const crbm_train_problem* pr, int n, int batch, double lr, double b1, double b2,
                         double eps, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  TrainParams p;
  const int CL = cluster_size(n, batch);
  p.batch = batch;
  p.per = (batch + CL - 1) / CL;
  p.lr = lr;
  p.b1 = b1;
  p.b2 = b2;
  p.eps = eps;
  size_t smem = 0;
  for (int i = 0; i < n; ++i) {
    p.pr[i] = pr[i];
    smem = std::max(smem, (size_t)train_layout(pr[i].K, pr[i].k, pr[i].L, batch, p.per).total);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n * CL));
  cfg.blockDim = dim3(kTrainThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)CL;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, train_epoch_kernel, p);
}

}  // namespace crbm
