// Device-side building blocks of the CRBM proposal + Metropolis-Hastings step.
//
// Method: arXiv:2008.05401.  CRBM joint/free energy (Sec. II, Eqs. 12-13),
// Gibbs conditionals (App. B.1, Eqs. B1-B4), acceptance (App. B.2, Eq. B5),
// Ising energy (Sec. III, Eq. 14), Kitaev Majorana log-weight (Sec. IV,
// Eq. 16 and the free energy that follows it).
//
// Data layout in shared memory (one chain):
//   plane = ceil(L*L/32) + 1 uint32 words, site n = i*L + j is bit n%32 of
//   word n/32, the extra word is padding read (and masked) by row extraction.
//   Per chain: plane[0], plane[1] (current / proposed lattice, swapped on
//   accept), K hidden planes.
// Work unit: a block of 4 consecutive sites n = 4q..4q+3.  One Philox call
// gives the 4 uniforms of a unit for one tag, so a unit is owned by one thread.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace crbm {

constexpr int kMaxK = 8;
constexpr int kMaxk = 7;
constexpr int kMaxJobs = 16;
constexpr int kNobs = 4;
constexpr uint32_t kTagAcc = 0xFFFFFFFEu;
constexpr uint32_t kTagInit = 0xFFFFFFFFu;
constexpr uint32_t kTagSwap = 0xFFFFFFFDu;   // tempering: physical <-> RBM exchange
constexpr uint32_t kTagTemp = 0xFFFFFFFCu;   // tempering: neighbour temperature exchange
constexpr uint32_t kTagLocal = 0xFFFFFFFBu;  // local-update Metropolis sweeps
constexpr int kIsing = 0;
constexpr int kKitaev = 1;
constexpr int kFP64 = 0;
constexpr int kMixed = 1;
// Threads per CTA of the fused kernel and the CTAs per SM its register budget
// is sized for (compile-time; the defaults were chosen by measurement).
#ifndef CRBM_THREADS
#define CRBM_THREADS 256
#endif
#ifndef CRBM_MIN_BLOCKS
#define CRBM_MIN_BLOCKS 2
#endif
constexpr int kThreads = CRBM_THREADS;
constexpr unsigned kFull = 0xffffffffu;

enum DevErr : int { kErrNone = 0, kErrConfig = 1, kErrTimeout = 2 };

// Everything a kernel needs about one job; passed by value in the launch
// parameters.  Pointers into the job's caller-owned device memory.
struct JobDev {
  int kind, L, N, Wd, P, K, k, n_chains, nc;
  int nc64;                     // chains per CTA of the FP64 path (Ising)
  int lc_edge;                  // > 0: LCRBM with lc_edge unshared kernels per side; lattice open along j
  int ncls;                     // kernel classes in the tables: 2 lc_edge + 1, or 1
  int nhex;                     // Kitaev hexagons: N, or L (L-1) with open columns
  double vb;
  double hb[kMaxK];
  double J[3];
  float vb32;
  float hb32[kMaxK], hb_hi[kMaxK], hb_lo[kMaxK];
  float c0h, c0v, c1, csp;      // FP32 error-bound constants (see host code)
  float cdf;                    // per unit: |hi/lo-table pre-activation - FP64 path's|
  float fx_scale;               // 2^e: units of the mixed path's free-energy sums (FreeSum::fx) in 1
  double fx_unit;               // 2^-e
  const double* f64;            // [K][k][2^k] row-sum tables, see struct Tabs
  const double* b64;
  const float* fd;
  const float* bd;
  const float* fh;
  const float* fl;
  const float4* fd4;            // [k][2^k] filter-interleaved, K <= 4 (Tabs fdi, fhi, fli)
  const float4* fh4;
  const float4* fl4;
  // tensor-core form (Ising, L = 128, 64, 32 or 16, K <= 4, k <= 5; crbm_step_tc.cu):
  // operand images of the filter digits, null when the model has none
  const uint4* tcw;
  float tq2, tq1, tq0;          // digit scales qf 2^22, qf 2^11, qf
  float tc0h, tc0v, tc1, tcft;  // certified error constants of that form
  uint64_t seed, cid_base;
  uint32_t rk[20];              // Philox round keys (k0 + r W0, k1 + r W1), r = 0..9
  unsigned long long* step;     // device-resident step counter of the job (proposals made)
  uint32_t* bits;               // [n_chains][Wd]
  const double* T;              // [n_chains]
  double* F;                    // [n_chains]
  double* Fb;                   // [n_chains] bound on |F - F_fp64| (0: exact)
  double* Lb;                   // [n_chains] bound on |log pi - log pi_fp64| (0: exact)
  double* logpi;                // [n_chains]
  double* Ephys;                // [n_chains]
  double* obs_t;                // [n_chains][4] observables of the current lattice
  double* obs;                  // [n_chains][4] running sums
  unsigned long long* acc;      // [n_chains]
  unsigned long long* rec;      // [n_chains][2] FP64 recomputes: Bernoulli draws, MH decisions
  double* eps;                  // [n_chains][N] Kitaev: single-fermion energies of the current
                                // lattice, ascending (written by modes 1 and 2 only)
  double* trace;                // optional [trace_cap][n_chains]: E_phys after step t at row
  unsigned long long trace_base;  // t - trace_base, for 0 <= t - trace_base < trace_cap
  long long trace_cap;
};

// E_phys of chain c after step t into the job's trace, if one is set and t is inside it.
__device__ __forceinline__ void trace_store(const JobDev& jb, int c, unsigned long long t, double E) {
  if (jb.trace == nullptr) return;
  const long long r = (long long)(t - jb.trace_base);
  if (t >= jb.trace_base && r < jb.trace_cap) jb.trace[r * jb.n_chains + c] = E;
}

struct LaunchParams {
  // mode 0: S proposals; 1: evaluate the current state; 2: one uncorrected
  // proposal of the tempering RBM chains of job[0] and its exchange with the
  // physical chains of job[1] (n_jobs = 1);
  // 3: S local-update Metropolis sweeps (Kitaev), where correct = 1 adds each sweep's
  // observables to the sums (0: the exchange kernel that follows does)
  int n_jobs, S, g, correct, mode;
  int tile_begin[kMaxJobs + 1];
  int* err;
  // tensor-core kernel (persistent CTAs): work items 0 .. total_items - 1
  // handed out by the counter *queue (zero at launch, cleared after it);
  // every device-side wait gives up after wait_limit SM clock cycles
  int* queue;
  int total_items;
  long long wait_limit;
  JobDev job[kMaxJobs];
};

// ------------------------------------------------------------------ Philox
// Philox4x32-10 (Salmon et al., SC'11): per round the counter words x0, x2
// are multiplied (32x32 -> 64 bit) by M0, M1; the high halves are xored with
// the other two words and the key; the key is bumped by the Weyl constants.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c;
}

// Same rounds with the ten round keys precomputed (rk[2r], rk[2r+1]): the
// key schedule of a launch is fixed, so the kernels read it from the launch
// parameters instead of bumping the key in every call.
__device__ __forceinline__ uint4 philox4x32_10_rk(uint4 c, const uint32_t* rk) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ rk[2 * r], lo1, hi0 ^ c.w ^ rk[2 * r + 1], lo0);
  }
  return c;
}

__device__ __forceinline__ uint32_t pick(const uint4& w, int t) {
  return t == 0 ? w.x : (t == 1 ? w.y : (t == 2 ? w.z : w.w));
}

// ------------------------------------------------------- bit-row windows
// w bits (w <= 12) of row r starting at column c (0 <= c < L), periodic in the
// column: bit b of the result is site (r, (c + b) mod L).  Supports L <= 32
// and L a multiple of 32.
__device__ __forceinline__ uint32_t row_window(const uint32_t* __restrict__ bits, int L, int r,
                                               int c, int w) {
  uint32_t x;
  if ((L & 31) == 0) {
    const int WL = L >> 5, wi = c >> 5;
    const int wn = (wi + 1 == WL) ? 0 : wi + 1;
    x = __funnelshift_r(bits[r * WL + wi], bits[r * WL + wn], c & 31);
  } else {
    const int off = r * L;
    const uint32_t row =
        __funnelshift_r(bits[off >> 5], bits[(off >> 5) + 1], off & 31) & ((1u << L) - 1u);
    uint64_t rr = row;
    for (int s = L; s < 64; s += L) rr |= (uint64_t)row << s;
    x = (uint32_t)(rr >> c);
  }
  return x & ((1u << w) - 1u);
}

// Rows of planes whose side is not a multiple of 32 (L <= 31), each repeated
// with period L over 64 bits: a window of up to 33 - w columns past any start is
// one shift, where row_window on the packed plane has to cut the row out and
// repeat it (up to 60 instructions, taken K k times per site of a visible
// half-step).  Bound by instruction issue; 1024 chains of L = 24, K = 2, k = 5,
// 20 proposals: 1.26 -> 1.09 ms; 1024 Kitaev chains of L = 6, 8 proposals (with
// the warps of an idle unit range left out): 2.19 -> 1.92 ms.  (L >= 32 has rows
// of whole words, whose window is one funnel shift already.)  By the group's
// threads, from `planes` planes P words apart.
__device__ __forceinline__ void expand_rows(const uint32_t* plane, int P, uint64_t* ext, int L, int planes, int r,
                                            int tpc) {
  if ((L & 31) == 0) return;
  for (int e = r; e < planes * L; e += tpc) {
    const int f = e / L, off = (e - f * L) * L;
    const uint32_t* p = plane + f * P + (off >> 5);
    uint64_t x = __funnelshift_r(p[0], p[1], off & 31) & ((1u << L) - 1u);
    for (int s = L; s < 64; s *= 2) x |= x << s;
    ext[e] = x;
  }
}
// row_window of a plane with (L not a multiple of 32) or without expanded rows.
__device__ __forceinline__ uint32_t window(const uint32_t* bits, const uint64_t* ext, int L, int r, int c, int w) {
  if ((L & 31) == 0) return row_window(bits, L, r, c, w);
  return (uint32_t)(ext[r] >> c) & ((1u << w) - 1u);
}

__device__ __forceinline__ uint32_t site_bit(const uint32_t* bits, int n) {
  return (bits[n >> 5] >> (n & 31)) & 1u;
}

// Forward codes of unit q (sites n = 4q..4q+3): m[t][a] = a*T + (bits of
// sites (i_t + a, j_t + b), b = 0..k-1, as bit b) -- the offset of the
// row-sum table entry of kernel row a for the receptive field of hidden unit
// (i_t, j_t).  When L % 4 == 0 the 4 sites share a row and one window of
// k + 3 bits per kernel row serves all of them.  kC > 0 fixes k at compile time.
template <int kC>
__device__ __forceinline__ void fwd_codes(const uint32_t* bits, const uint64_t* ext, int L, int N, int k, int T, int q,
                                          uint32_t (&m)[4][kC ? kC : kMaxk]) {
  constexpr int kU = kC ? kC : kMaxk;
  const uint32_t mk = (1u << k) - 1u;
  if ((L & 3) == 0) {
    const int n0 = 4 * q, i = n0 / L, j0 = n0 - i * L;
#pragma unroll
    for (int a = 0; a < kU; ++a) {
      if (kC || a < k) {
        int r = i + a;
        if (r >= L) r -= L;
        const uint32_t win = window(bits, ext, L, r, j0, k + 3);
#pragma unroll
        for (int t = 0; t < 4; ++t) m[t][a] = (uint32_t)(a * T) + ((win >> t) & mk);
      }
    }
  } else {
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      int n = 4 * q + t;
      if (n >= N) n = 0;
      const int i = n / L, j = n - i * L;
#pragma unroll
      for (int a = 0; a < kU; ++a) {
        if (kC || a < k) {
          int r = i + a;
          if (r >= L) r -= L;
          m[t][a] = (uint32_t)(a * T) + window(bits, ext, L, r, j, k);
        }
      }
    }
  }
}

// ------------------------------------------------ Bernoulli decisions
// FP64: h = [u < sigma(x)], u = (w + 1/2) 2^-32 exactly (App. B.1 sampling),
// as u (1 + e^-x) < 1: no division on the FP64 pipe.
__device__ __forceinline__ uint32_t decide64(double x, uint32_t w) {
  const double u = ((double)w + 0.5) * 0x1p-32;
  return u * (1.0 + exp(-x)) < 1.0 ? 1u : 0u;
}

// Special-function-unit approximations (PTX ex2/rcp/lg2, flush-to-zero).
// Their error bounds are part of the certified margins below and are checked
// exhaustively on the device by the test-suite.
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// log u of an MH draw u = (w + 1/2) 2^-32 in FP32, within 2^-20 (1 + |log u|)
// of the exact value: u = m 2^e with m in [1, 2) split off its float exactly,
// lg2 of m from the special-function unit (absolute error 2^-22 on [1, 2]),
// the float rounding of u within 2^-23 relative, the sum and the ln 2
// product within 2^-24 relative each.
__device__ __forceinline__ float log_u32(uint32_t w) {
  const uint32_t ub = __float_as_uint(((float)w + 0.5f) * 0x1p-32f);
  const float lg2u = (float)((int)(ub >> 23) - 127) + lg2_approx(__uint_as_float((ub & 0x7FFFFFu) | 0x3F800000u));
  return lg2u * 0.69314718055994531f;
}

// sigma(x) in FP32: e = 2^(-x log2 e), p = 1/(1 + e).
__device__ __forceinline__ float sigmoid32(float x) {
  return rcp_approx(1.0f + ex2_approx(x * -1.4426950408889634f));
}

// FP32 decision with a certified margin: |p32 - p64| <= c0 + c1 |x| covers the
// FP32 pre-activation error, the ex2/rcp errors, the conversion of the Philox
// word, and the FP64 path's own rounding.  Returns 0/1 when the FP64 path
// takes the same decision, 2 when the FP64 code has to decide.
// The comparison runs in units of 2^-32 (p 2^32 against the Philox word), so
// c0 and c1 arrive pre-scaled by 2^32.
__device__ __forceinline__ uint32_t decide32(float x, uint32_t w, float c0, float c1) {
  const float d = fmaf(sigmoid32(x), 0x1p32f, -__uint2float_rn(w));
  const float delta = fmaf(c1, fabsf(x), c0);
  return fabsf(d) > delta ? (d > 0.0f ? 1u : 0u) : 2u;
}

// The same decision as decide32, returned as the FP32 bit and a flag that is
// 1 when the margin does not separate it (then the FP64 path decides).
__device__ __forceinline__ void decide32_split(float x, uint32_t w, float c0, float c1, uint32_t& bit,
                                               uint32_t& amb) {
  const float d = fmaf(sigmoid32(x), 0x1p32f, -__uint2float_rn(w));
  const float delta = fmaf(c1, fabsf(x), c0);
  bit = d > 0.0f ? 1u : 0u;
  amb = fabsf(d) > delta ? 0u : 1u;
}

// log(1 + e^x) in FP32 without overflow: max(x, 0) + ln 2 * log2(1 + 2^(-|x| log2 e)).
__device__ __forceinline__ float softplus32(float x) {
  const float e = ex2_approx(fabsf(x) * -1.4426950408889634f);
  return fmaxf(x, 0.0f) + 0.69314718055994531f * lg2_approx(1.0f + e);
}

// Store the 4-bit result of unit q: 8 consecutive lanes own the 8 units of
// one word and OR their nibbles together.  Every lane of the warp must call.
__device__ __forceinline__ void store_nibble(uint32_t* plane, int q, uint32_t nib, bool act) {
  uint32_t x = act ? (nib << (4 * (q & 7))) : 0u;
  x |= __shfl_xor_sync(kFull, x, 1);
  x |= __shfl_xor_sync(kFull, x, 2);
  x |= __shfl_xor_sync(kFull, x, 4);
  if (act && (q & 7) == 0) plane[q >> 3] = x;
}

// One chain's thread group: tpc threads (a power of two >= 8), rank r.
struct Grp {
  int c;          // chain index within the job
  int gl;         // group index within the CTA
  int r, tpc;
  bool active;    // c < n_chains
  uint32_t cid;   // chain id (Philox counter word 3)
};

// Deterministic sum of NV doubles over a chain's group; the result is valid in
// the leader (r == 0).  Every thread of the CTA must call (it may sync).
template <int NV>
__device__ __forceinline__ void grp_reduce(double (&x)[NV], const Grp& g, double* scratch) {
  const int span = g.tpc < 32 ? g.tpc : 32;
  for (int o = 1; o < span; o <<= 1) {
#pragma unroll
    for (int v = 0; v < NV; ++v) x[v] += __shfl_xor_sync(kFull, x[v], o);
  }
  if (g.tpc > 32) {
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
      for (int v = 0; v < NV; ++v) scratch[warp * NV + v] = x[v];
    }
    __syncthreads();
    if (g.r == 0) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        double s = 0.0;
        for (int w = 0; w < g.tpc / 32; ++w) s += scratch[(warp + w) * NV + v];
        x[v] = s;
      }
    }
    __syncthreads();
  }
}

// Barrier of one chain's thread group (warp-aligned groups of 32 .. blockDim
// threads): the CTA barrier when the group is the whole CTA, the warp's when it
// is one warp, else a named barrier of its own (id 1 + group index; a CTA holds
// at most 8 groups).  Only the group's threads take part, so groups may run
// different branches between two of their barriers.  MULTI = false: the
// caller's CTAs hold one group each, and this is the CTA barrier (code without
// named barriers, which would reserve all of the CTA's barrier slots).
template <bool MULTI>
__device__ __forceinline__ void grp_sync(const Grp& g) {
  if (!MULTI || g.tpc == (int)blockDim.x) {
    __syncthreads();
  } else if (g.tpc == 32) {
    __syncwarp();
  } else {
    asm volatile("bar.sync %0, %1;\n" :: "r"(1 + g.gl), "r"(g.tpc) : "memory");
  }
}

// Sums of a free-energy pass: F's softplus sum -- FP64 (s), or for the FP32
// pass the thread's sum as an integer in units of jb.fx_unit (fx: exact additions
// off the FP64 pipe, each thread's conversion within half a unit) with the data
// part of its error bound (b) -- and the lattice counts.  The unit is the power
// of two that leaves the largest sum the filters allow below 2^61 (fx_exponent):
// a fixed one would wrap for large filters, or round small sums.
struct FreeSum {
  double s;
  long long fx;
  float b;
  int ones, pairs;
};

// Deterministic sum over a chain's group, valid in its leader (r == 0).
// scratch: 3 doubles per warp of the CTA (MULTI: of the group, whose threads
// alone synchronise; else every thread of the CTA calls).
template <int PREC, bool MULTI>
__device__ __forceinline__ void reduce_free(FreeSum& x, const Grp& g, double* scratch) {
  const int span = g.tpc < 32 ? g.tpc : 32;
  for (int o = 1; o < span; o <<= 1) {
    if (PREC == kFP64) {
      x.s += __shfl_xor_sync(kFull, x.s, o);
    } else {
      x.fx += __shfl_xor_sync(kFull, x.fx, o);
      x.b += __shfl_xor_sync(kFull, x.b, o);
    }
    x.ones += __shfl_xor_sync(kFull, x.ones, o);
    x.pairs += __shfl_xor_sync(kFull, x.pairs, o);
  }
  if (g.tpc > 32) {
    const int warp = (MULTI ? g.r : (int)threadIdx.x) >> 5;
    double* mine = scratch + 3 * warp;
    if ((threadIdx.x & 31) == 0) {
      if (PREC == kFP64) mine[0] = x.s;
      else mine[0] = __longlong_as_double(x.fx);
      ((float*)mine)[2] = x.b;
      ((int*)mine)[3] = x.ones;
      ((int*)mine)[4] = x.pairs;
    }
    grp_sync<MULTI>(g);
    if (g.r == 0) {
      for (int w = 1; w < g.tpc / 32; ++w) {
        const double* o = mine + 3 * w;
        if (PREC == kFP64) x.s += o[0];
        else x.fx += __double_as_longlong(o[0]);
        x.b += ((const float*)o)[2];
        x.ones += ((const int*)o)[3];
        x.pairs += ((const int*)o)[4];
      }
    }
    grp_sync<MULTI>(g);
  }
}

// F (Eq. 13) from the group's sums.
template <int PREC>
__device__ __forceinline__ double free_value(const JobDev& jb, const FreeSum& x) {
  if (PREC == kFP64) return -jb.vb * (double)x.ones - x.s;
  return fma((double)x.fx, -jb.fx_unit, -jb.vb * (double)x.ones);
}

// Deterministic block-wide sum, result returned to every thread.
__device__ __forceinline__ double block_sum(double x, double* scratch) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) x += __shfl_xor_sync(kFull, x, o);
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) scratch[warp] = x;
  __syncthreads();
  double s = 0.0;
  for (int w = 0; w < nw; ++w) s += scratch[w];
  __syncthreads();
  return s;
}

// Row-sum tables of one model (index (f*k + a)*T + code, T = 2^k):
//   f64/b64   FP64, forward code / raw backward window (FP64 path; global
//             copies of them serve the mixed path's FP64 recomputes)
//   fd/bd     FP32 roundings of f64/b64 (mixed-path decisions)
//   fh/fl     hi/lo split of f64 (mixed-path free energy)
//   fdi/fhi/fli  the same forward tables with the filter index innermost
//             (global: (a*T + code)*4 + f for K <= 4, zero-padded), for K = 4 and,
//             Ising, K = 2: one 16- or 8-byte load serves all filters of a site.
//             In shared memory entry e is 32 floats, 32 / K copies of its K
//             values; thread t reads copy t % (32 / K) (the pointer includes its
//             offset, so entry e is at [32 e]): the threads one pass of a load
//             serves (a quarter or a half warp) hit distinct banks whatever
//             their codes, so it never conflicts
struct Tabs {
  const double* f64;
  const double* b64;
  const float* fd;
  const float* bd;
  const float* fh;
  const float* fl;
  const float *fdi, *fhi, *fli;
  int T;
};

// x_f += entry `code` of an interleaved table, all filters in one load.
template <int KC>
__device__ __forceinline__ void add_taps(float (&x)[KC], const float* table, uint32_t code) {
  static_assert(KC == 2 || KC == 4, "one 8- or 16-byte load");
  if constexpr (KC == 4) {
    const float4 e = *reinterpret_cast<const float4*>(table + 32 * code);
    x[0] += e.x;
    x[1] += e.y;
    x[2] += e.z;
    x[3] += e.w;
  } else {
    const float2 e = *reinterpret_cast<const float2*>(table + 32 * code);
    x[0] += e.x;
    x[1] += e.y;
  }
}

// FP64 recomputes of the mixed path (rare; kept out of line so that the FP32
// fast path keeps its registers).  Same tables (global copies), same order.
static __device__ __noinline__ uint32_t recompute_hidden(const JobDev& jb, int f, const uint32_t* m, int k,
                                                         int T, uint32_t w) {
  double x = jb.hb[f];
  const int base = f * k * T;
  for (int a = 0; a < k; ++a) x += __ldg(jb.f64 + base + m[a]);
  return decide64(x, w);
}

__device__ __forceinline__ int bwd_row(int i, int a, int L) {
  int r = i - a;
  return r < 0 ? r + L : r;
}

// This site's visible pre-activation with the FP64 tables, in the FP64 path's order.
static __device__ __noinline__ uint32_t recompute_visible(const JobDev& jb, const uint32_t* h, int P, int n,
                                                          uint32_t w) {
  const int L = jb.L, K = jb.K, k = jb.k, T = 1 << k;
  const int i = n / L, j = n - i * L;
  int c = j - (k - 1);
  if (c < 0) c += L;
  double x = jb.vb;
  for (int a = 0; a < k; ++a) {
    const int r = bwd_row(i, a, L);
    for (int f = 0; f < K; ++f) x += __ldg(jb.b64 + (f * k + a) * T + row_window(h + f * P, L, r, c, k));
  }
  return decide64(x, w);
}

// ------------------------------------------------- LCRBM (open columns)
// Column class of hidden column j: left edge columns 0..e-1, right edge
// columns e..2e-1, bulk 2e (Sec. IV, open boundary conditions).
__device__ __forceinline__ int lc_class(int j, int L, int e) {
  return j < e ? j : (j >= L - e ? e + (j - (L - e)) : 2 * e);
}

// FP64 pre-activation of filter f of an LCRBM at site n: the window is cut at
// the open column edge (bits b >= L - j dropped) and the table of the column's
// class is used.
__device__ __forceinline__ double lc_preact64(const JobDev& jb, const double* f64, int f, const uint32_t* v, int n,
                                              int k, int T) {
  const int L = jb.L, i = n / L, j = n - i * L;
  const int base = (lc_class(j, L, jb.lc_edge) * jb.K + f) * k * T;
  const uint32_t keep = (j + k > L) ? ((1u << (L - j)) - 1u) : 0xFFFFFFFFu;
  double x = jb.hb[f];
  for (int a = 0; a < k; ++a) {
    const int r = i + a < L ? i + a : i + a - L;
    x += f64[base + a * T + (int)(row_window(v, L, r, j, k) & keep)];
  }
  return x;
}

// FP64 visible pre-activation of an LCRBM at site n: v_bias plus, for every
// hidden unit (f, i-a, j-b) with j - b >= 0, its class kernel's weight
// W[c(j-b)][f][a][b] (the table entry of the single-bit code 1 << b) if set.
__device__ inline double lc_visible64(const JobDev& jb, const double* f64, const uint32_t* h, int P, int n,
                                      int k, int T) {
  const int L = jb.L, i = n / L, j = n - i * L;
  double x = jb.vb;
  for (int a = 0; a < k; ++a) {
    const int r = (i - a < 0) ? i - a + L : i - a;
    for (int f = 0; f < jb.K; ++f) {
      const uint32_t* pl = h + f * P;
      for (int b = 0; b < k && b <= j; ++b) {
        const int jc = j - b;
        if (site_bit(pl, r * L + jc))
          x += f64[((lc_class(jc, L, jb.lc_edge) * jb.K + f) * k + a) * T + (1 << b)];
      }
    }
  }
  return x;
}

// ------------------------------------------------- hidden half-step
// h^f_ij = [u < sigma(h_bias^f + sum_ab W^f_ab v_(i+a)(j+b))]  (Eq. B2, Eq. 12)
// FP64 order (shared with the mixed path's recompute): h_bias, then kernel
// rows a = 0..k-1.
// FP64 form: thread (filter, site), so that a warp's FP64 instructions (each
// holds the sub-partition's pipe for about 64 cycles whatever its active
// lanes) are full; the Philox block of four sites is drawn by each of them,
// integer work beside it.  sync: the group's barrier.
template <class SYNC>
__device__ void hidden_phase64(const JobDev& jb, const Tabs& tb, const Grp& g, const uint32_t* v, uint32_t* h, int P,
                               uint32_t step, int sub, SYNC sync) {
  const int L = jb.L, N = jb.N, K = jb.K, k = jb.k, T = tb.T;
  if (g.active)
    for (int w = g.r; w < K * P; w += g.tpc) h[w] = 0u;
  sync();
  if (!g.active) return;
  for (int e = g.r; e < K * N; e += g.tpc) {
    const int f = e / N, n = e - f * N, i = n / L, j = n - i * L;
    double x = jb.hb[f];
    if (jb.lc_edge) {
      x = lc_preact64(jb, tb.f64, f, v, n, k, T);
    } else {
      for (int a = 0; a < k; ++a) {
        const int r = i + a < L ? i + a : i + a - L;
        x += tb.f64[(f * k + a) * T + row_window(v, L, r, j, k)];
      }
    }
    const uint4 w = philox4x32_10_rk(make_uint4((uint32_t)(n >> 2), (uint32_t)(sub * (K + 1) + f), step, g.cid), jb.rk);
    if (decide64(x, pick(w, n & 3))) atomicOr(h + f * P + (n >> 5), 1u << (n & 31));
  }
}

// Mixed form: thread = unit of 4 sites, units q0 .. q1 - 1.  KC, kC > 0 fix K
// and k at compile time (0: runtime).
template <int KC, int kC>
__device__ void hidden_phase(const JobDev& jb, const Tabs& tb, const Grp& g, const uint32_t* v,
                             const uint64_t* ext, uint32_t* h, int P, uint32_t step, int sub, unsigned& nrec, int q0,
                             int q1) {
  constexpr int kU = kC ? kC : kMaxk;
  const int L = jb.L, N = jb.N, K = KC ? KC : jb.K, k = kC ? kC : jb.k, T = tb.T;
  const int iters = (q1 - q0 + g.tpc - 1) / g.tpc;
  for (int it = 0; it < iters; ++it) {
    const int q = q0 + g.r + it * g.tpc;
    const bool act = g.active && q < q1;
    uint32_t m[4][kU];
    if (!__any_sync(kFull, act)) continue;
    fwd_codes<kC>(v, ext, L, N, k, T, act ? q : 0, m);
    if constexpr (KC != 0) {
      // all filters per site from the filter-interleaved table
      uint4 w[KC];
#pragma unroll
      for (int f = 0; f < KC; ++f)
        w[f] = philox4x32_10_rk(make_uint4((uint32_t)q, (uint32_t)(sub * (KC + 1) + f), step, g.cid), jb.rk);
      uint32_t nib[KC] = {};
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        float x[KC];
#pragma unroll
        for (int f = 0; f < KC; ++f) x[f] = jb.hb32[f];
#pragma unroll
        for (int a = 0; a < kU; ++a) add_taps(x, tb.fdi, m[t][a]);
        const bool site = act && 4 * q + t < N;
#pragma unroll
        for (int f = 0; f < KC; ++f) {
          uint32_t bit = decide32(x[f], pick(w[f], t), jb.c0h, jb.c1);
          if (bit == 2u) {
            uint32_t mm[kMaxk];
#pragma unroll
            for (int a = 0; a < kU; ++a) mm[a] = m[t][a];
            bit = recompute_hidden(jb, f, mm, k, T, pick(w[f], t));
            if (site) ++nrec;
          }
          if (site) nib[f] |= bit << t;
        }
      }
#pragma unroll
      for (int f = 0; f < KC; ++f) store_nibble(h + f * P, q, nib[f], act);
      continue;
    }
    for (int f = 0; f < K; ++f) {
      const uint4 w = philox4x32_10_rk(make_uint4((uint32_t)q, (uint32_t)(sub * (K + 1) + f), step, g.cid), jb.rk);
      const int base = f * k * T;
      uint32_t nib = 0;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        float x = jb.hb32[f];
#pragma unroll
        for (int a = 0; a < kU; ++a) if (kC || a < k) x += tb.fd[base + m[t][a]];
        uint32_t bit = decide32(x, pick(w, t), jb.c0h, jb.c1);
        if (bit == 2u) {
          uint32_t mm[kMaxk];
#pragma unroll
          for (int a = 0; a < kU; ++a) mm[a] = m[t][a];
          bit = recompute_hidden(jb, f, mm, k, T, pick(w, t));
          if (act && 4 * q + t < N) ++nrec;
        }
        if (act && 4 * q + t < N) nib |= bit << t;
      }
      store_nibble(h + f * P, q, nib, act);
    }
  }
}

// ------------------------------------------------- visible half-step
// v'_ij = [u < sigma(v_bias + sum_f sum_ab W^f_ab h^f_(i-a)(j-b))]  (Eq. B3)
// The window of hidden row i - a starting at column j - (k-1) holds, as bit
// k-1-b, the unit h_(i-a)(j-b); the backward tables are indexed by that raw
// window.  Order: v_bias, then kernel rows a, then filters f.
// FP64 form: thread = site (see hidden_phase64).
template <class SYNC>
__device__ void visible_phase64(const JobDev& jb, const Tabs& tb, const Grp& g, const uint32_t* h, uint32_t* vp, int P,
                                uint32_t step, int sub, SYNC sync) {
  const int L = jb.L, N = jb.N, K = jb.K, k = jb.k, T = tb.T;
  if (g.active)
    for (int w = g.r; w < jb.Wd; w += g.tpc) vp[w] = 0u;
  sync();
  if (!g.active) return;
  for (int n = g.r; n < N; n += g.tpc) {
    double x = jb.vb;
    if (jb.lc_edge) {
      x = lc_visible64(jb, tb.f64, h, P, n, k, T);
    } else {
      const int i = n / L, j = n - i * L;
      int c = j - (k - 1);
      if (c < 0) c += L;
      for (int a = 0; a < k; ++a) {
        const int r = bwd_row(i, a, L);
        for (int f = 0; f < K; ++f) x += tb.b64[(f * k + a) * T + row_window(h + f * P, L, r, c, k)];
      }
    }
    const uint4 w = philox4x32_10_rk(make_uint4((uint32_t)(n >> 2), (uint32_t)(sub * (K + 1) + K), step, g.cid), jb.rk);
    if (decide64(x, pick(w, n & 3))) atomicOr(vp + (n >> 5), 1u << (n & 31));
  }
}

// Mixed form: thread = unit of 4 sites, units q0 .. q1 - 1.
template <int KC, int kC>
__device__ void visible_phase(const JobDev& jb, const Tabs& tb, const Grp& g, const uint32_t* h,
                              const uint64_t* ext, uint32_t* vp, int P, uint32_t step, int sub, unsigned& nrec, int q0,
                              int q1) {
  constexpr int kU = kC ? kC : kMaxk;
  constexpr int KU = KC ? KC : kMaxK;
  const int L = jb.L, N = jb.N, K = KC ? KC : jb.K, k = kC ? kC : jb.k, T = tb.T;
  const uint32_t mk = (1u << k) - 1u;
  const int iters = (q1 - q0 + g.tpc - 1) / g.tpc;
  const bool rows4 = (L & 3) == 0;
  for (int it = 0; it < iters; ++it) {
    const int q = q0 + g.r + it * g.tpc;
    const bool act = g.active && q < q1;
    if (!__any_sync(kFull, act)) continue;
    const int qq = act ? q : 0;
    float x32[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) x32[t] = jb.vb32;
    if (rows4) {
      const int n0 = 4 * qq, i = n0 / L, j0 = n0 - i * L;
      int c = j0 - (k - 1);
      if (c < 0) c += L;
#pragma unroll
      for (int a = 0; a < kU; ++a) {
        if (kC || a < k) {
          const int r = bwd_row(i, a, L);
          // word offsets of this window, shared by the K hidden planes
          const bool wide = (L & 31) == 0;
          const int WL = L >> 5, wi = c >> 5, o0 = r * WL + wi, o1 = r * WL + ((wi + 1 == WL) ? 0 : wi + 1);
#pragma unroll
          for (int f = 0; f < KU; ++f) {
            if (KC || f < K) {
              const uint32_t* pl = h + f * P;
              const uint32_t win = wide ? __funnelshift_r(pl[o0], pl[o1], c & 31) : (uint32_t)(ext[f * L + r] >> c);
              const int base = (f * k + a) * T;
#pragma unroll
              for (int t = 0; t < 4; ++t) {
                const uint32_t code = (win >> t) & mk;
                x32[t] += tb.bd[base + code];
              }
            }
          }
        }
      }
    } else {
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        int n = 4 * qq + t;
        if (n >= N) n = 0;
        const int i = n / L, j = n - i * L;
        int c = j - (k - 1);
        if (c < 0) c += L;
        for (int a = 0; a < k; ++a) {
          const int r = bwd_row(i, a, L);
          for (int f = 0; f < K; ++f) {
            const uint32_t code = window(h + f * P, ext + f * L, L, r, c, k);
            const int base = (f * k + a) * T;
            x32[t] += tb.bd[base + code];
          }
        }
      }
    }
    const uint4 w = philox4x32_10_rk(make_uint4((uint32_t)q, (uint32_t)(sub * (K + 1) + K), step, g.cid), jb.rk);
    uint32_t nib = 0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if (act && 4 * q + t < N) {
        uint32_t bit = decide32(x32[t], pick(w, t), jb.c0v, jb.c1);
        if (bit == 2u) {
          bit = recompute_visible(jb, h, P, 4 * q + t, pick(w, t));
          ++nrec;
        }
        nib |= bit << t;
      }
    }
    store_nibble(vp, q, nib, act);
  }
}

// ------------------------------------------------- free energy + lattice sums
// F(v) = -v_bias sum v - sum_{f,i,j} softplus(h_bias^f + (W^f * v)_ij)   (Eq. 13)
// Per-thread partial sums: softplus (FreeSum), the number of ones and of
// unequal nearest-neighbour pairs (Ising) or of hexagons with flux -1 (Kitaev).
// (1 + p)(1 + e) - 1: the sum of two log1p as the log1p of one number, which keeps
// its leading digits however small p and e are (1 + e would round them away).
__device__ __forceinline__ double join_log1p(double p, double e) { return fma(p, e, p + e); }
// log(1 + p), p >= 0, to p's own relative rounding: what u = 1 + p lost of p < 1 is
// below 2^-53 and enters with slope 1/u, 1 - 1/u <= p off 1 (a few FP64 operations
// cheaper than log1p: 100 proposals of 16 chains of L = 8 1.17 against 1.23 ms).
__device__ __forceinline__ double log_joined(double p) {
  const double u = 1.0 + p;
  return log(u) + (p < 1.0 ? p - (u - 1.0) : 0.0);
}

// FP64 form: thread (filter, site); the log(1 + e^-|x|) of a
// thread's units are the log of their product (factors in (1, 2], the log taken at
// least every 512), kept less 1.
__device__ inline FreeSum free_phase64(const JobDev& jb, const double* f64, const Grp& g, const uint32_t* v) {
  const int L = jb.L, N = jb.N, K = jb.K, k = jb.k, T = 1 << k;
  FreeSum out = {0.0, 0ll, 0.0f, 0, 0};
  if (!g.active) return out;
  double prod = 0.0;
  int held = 0;
  for (int e = g.r; e < K * N; e += g.tpc) {
    const int f = e / N, n = e - f * N, i = n / L, j = n - i * L;
    double x = jb.hb[f];
    if (jb.lc_edge) {
      x = lc_preact64(jb, f64, f, v, n, k, T);
    } else {
      for (int a = 0; a < k; ++a) {
        const int r = i + a < L ? i + a : i + a - L;
        x += f64[(f * k + a) * T + row_window(v, L, r, j, k)];
      }
    }
    out.s += fmax(x, 0.0);
    prod = join_log1p(prod, exp(-fabs(x)));
    if (++held == 512) {
      out.s += log_joined(prod);
      prod = 0.0;
      held = 0;
    }
  }
  if (held) out.s += log_joined(prod);
  for (int n = g.r; n < N; n += g.tpc) {
    const int i = n / L, j = n - i * L, jr = j + 1 == L ? 0 : j + 1;
    const uint32_t b0 = site_bit(v, n);
    out.ones += (int)b0;
    if (jb.kind == kIsing) {
      out.pairs += (int)(b0 ^ site_bit(v, i * L + jr)) + (int)(b0 ^ site_bit(v, (i + 1 == L ? 0 : i + 1) * L + j));
    } else if (!(jb.lc_edge && j + 1 == L)) {
      // the hexagon of cell r holds the z-bonds r and r - e1 + e2 (with
      // open columns the hexagons of column L-1 do not exist)
      out.pairs += (int)(b0 ^ site_bit(v, (i == 0 ? L - 1 : i - 1) * L + jr));
    }
  }
  return out;
}

// Bound on |F - F_fp64| of an FP32 free energy beyond the constant cst of
// free_constant: the summed data terms and F's own rounding.
__device__ __forceinline__ double free_bound(const FreeSum& x, double cst, double F) {
  return ((double)x.b * 1.001 + cst) + 1e-12 * fabs(F);
}
// Per unit the special-function and table errors, per thread the fixed-point conversion.
__device__ __forceinline__ double free_constant(const JobDev& jb, int tpc) {
  return (double)jb.K * (double)jb.N * (1.5 * 0x1p-23 + (double)jb.csp) + (double)tpc * (0.5 * jb.fx_unit);
}

// Mixed form: thread = unit of 4 sites, units q0 .. q1 - 1, FP32 with Kahan
// compensation.
template <int KC, int kC>
__device__ FreeSum free_phase(const JobDev& jb, const Tabs& tb, const Grp& g, const uint32_t* v,
                              const uint64_t* ext, int q0, int q1) {
  constexpr int kU = kC ? kC : kMaxk;
  const int L = jb.L, N = jb.N, K = KC ? KC : jb.K, k = kC ? kC : jb.k, T = tb.T;
  const int iters = (q1 - q0 + g.tpc - 1) / g.tpc;
  float s32 = 0.0f, c32 = 0.0f, sabs = 0.0f, ssp = 0.0f;
  int ones = 0, pairs = 0;
  for (int it = 0; it < iters; ++it) {
    const int q = q0 + g.r + it * g.tpc;
    const bool act = g.active && q < q1;
    if (!act) continue;
    uint32_t m[4][kU];
    fwd_codes<kC>(v, ext, L, N, k, T, q, m);
    if constexpr (KC != 0) {
      float sp[4][KC];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        float xh[KC], xl[KC];
#pragma unroll
        for (int f = 0; f < KC; ++f) {
          xh[f] = jb.hb_hi[f];
          xl[f] = jb.hb_lo[f];
        }
#pragma unroll
        for (int a = 0; a < kU; ++a) {
          add_taps(xh, tb.fhi, m[t][a]);
          add_taps(xl, tb.fli, m[t][a]);
        }
        const bool site = 4 * q + t < N;
#pragma unroll
        for (int f = 0; f < KC; ++f) {
          const float x = xh[f] + xl[f];
          sp[t][f] = site ? softplus32(x) : 0.0f;
          sabs += site ? fabsf(x) : 0.0f;
        }
      }
#pragma unroll
      for (int f = 0; f < KC; ++f) {
        const float us = (sp[0][f] + sp[1][f]) + (sp[2][f] + sp[3][f]);
        ssp += us;
        const float y = us - c32;          // Kahan summation of the unit sums
        const float tt = s32 + y;
        c32 = (tt - s32) - y;
        s32 = tt;
      }
    } else {
      for (int f = 0; f < K; ++f) {
        const int base = f * k * T;
        float sp[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          sp[t] = 0.0f;
          if (4 * q + t < N) {
            float xh = jb.hb_hi[f], xl = jb.hb_lo[f];
#pragma unroll
            for (int a = 0; a < kU; ++a) {
              if (kC || a < k) {
                xh += tb.fh[base + m[t][a]];
                xl += tb.fl[base + m[t][a]];
              }
            }
            const float x = xh + xl;
            sp[t] = softplus32(x);
            sabs += fabsf(x);
          }
        }
        const float us = (sp[0] + sp[1]) + (sp[2] + sp[3]);
        ssp += us;
        const float y = us - c32;
        const float tt = s32 + y;
        c32 = (tt - s32) - y;
        s32 = tt;
      }
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int n = 4 * q + t;
      if (n < N) {
        const int i = n / L, j = n - i * L;
        const uint32_t b0 = m[t][0] & 1u;
        ones += (int)b0;
        if (jb.kind == kIsing) {
          const uint32_t right = (k >= 2) ? ((m[t][0] >> 1) & 1u) : site_bit(v, i * L + (j + 1 == L ? 0 : j + 1));
          const uint32_t down = (k >= 2) ? ((m[t][kU > 1 ? 1 : 0] - (uint32_t)T) & 1u)
                                         : site_bit(v, (i + 1 == L ? 0 : i + 1) * L + j);
          pairs += (int)(b0 ^ right) + (int)(b0 ^ down);
        } else {
          // the hexagon of cell r holds the z-bonds r and r - e1 + e2 (with
          // open columns the hexagons of column L-1 do not exist)
          const int i2 = (i == 0) ? L - 1 : i - 1, j2 = (j + 1 == L) ? 0 : j + 1;
          if (!(jb.lc_edge && j + 1 == L)) pairs += (int)(b0 ^ site_bit(v, i2 * L + j2));
        }
      }
    }
  }
  FreeSum out;
  out.s = 0.0;
  out.fx = __float2ll_rn(s32 * jb.fx_scale);
  // x rounding + ex2 argument: 2^-23 |x|; pairwise, Kahan and final add: 6 2^-24 sp
  // (free_bound's factor covers the FP32 accumulation of these two sums themselves)
  out.b = sabs * 0x1p-23f + ssp * (6.0f * 0x1p-24f);
  out.ones = ones;
  out.pairs = pairs;
  return out;
}

// --------------------------------------------------- Kitaev log-weight
// Packed lower triangle of a symmetric N x N matrix: element (i, c), c <= i.
__device__ __forceinline__ int tri(int i, int c) { return i * (i + 1) / 2 + c; }
// Lanes per row of a group's matrix-vector product over m rows with nt
// threads: the largest power of two H <= 32 with H m <= nt (at least 1).
__device__ __forceinline__ int row_split(int m, int nt) {
  int H = 1;
  while (H < 32 && 2 * H * m <= nt) H <<= 1;
  return H;
}

// The same for the FP64 stage, which its pipe's warp instructions pace whatever
// lanes they fill: of that H and its two next, the one whose warps' steps, with the
// log2 H additions that join a row, are fewest (35 rows by 64 threads: 70 at H = 1,
// where the second warp takes 35 for three rows; 55 at H = 4).  Tempering of L = 8,
// six cycles of 2 x 1024 chains: 7.2 ms without it, 6.9 with.
__device__ __forceinline__ int row_lanes64(int m, int nt) {
  int H = row_split(min(m, nt), nt), best = H, cost = 1 << 30;
  for (int i = 0; i < 3 && H <= 8; ++i, H <<= 1) {
    const int t = ((m * H + 31) >> 5) * ((m + H - 1) / H + 31 - __clz(H));
    if (t < cost) {
      cost = t;
      best = H;
    }
  }
  return best;
}
// Element (c, l) of the rows and columns j1 .. of a packed lower triangle, on
// either side of its diagonal.  A warp of a matrix-vector product takes one loop
// over c with it: with a loop along the packed row and one down the packed column,
// each lane crossing over at its own diagonal, the warp took the longest of both
// (66 steps for the 35 of the first 32 rows at 35 columns).  Rows start at
// triangular numbers, distinct mod 16, columns are contiguous: no bank conflicts
// at one lane per row.  1024 chains of L = 6, mixed, eight proposals 1.92 -> 1.78
// ms, FP64, four 1.83 -> 1.74; tempering of L = 8 7.8 -> 6.9; 1024 open-boundary
// chains of L = 8, four proposals 8.7 -> 8.3; 683 mixed chains each of L = 8, 10,
// 12, three proposals 11.5 -> 11.1.
template <class T>
__device__ __forceinline__ T sym_at(const T* A, int j1, int c, int l) {
  return A[tri(j1 + max(c, l), j1) + min(c, l)];
}
// Lane h's share (columns h, h + H, ...) of row l of A22 x; mac(a, x, y): y += a x.
// (Loops of their own for the columns left and right of the warp's diagonals need
// no index arithmetic but are four times the code: 2.00 ms for the mixed L = 6.)
template <class T, class MAC>
__device__ __forceinline__ void sym_row(const T* A, const T* xs, int j1, int m, int l, int h, int H, T& y0, T& y1,
                                        MAC mac) {
  int c = h;
  for (; c + H < m; c += 2 * H) {
    mac(sym_at(A, j1, c, l), xs[c], y0);
    mac(sym_at(A, j1, c + H, l), xs[c + H], y1);
  }
  if (c < m) mac(sym_at(A, j1, c, l), xs[c], y0);
}

// Thread tid of nt visiting a packed triangle of R rows (row r: columns
// 0..r) with stride nt: rows p and R-1-p side by side form folded row p,
// R+1 long, so the thread's next element is a fixed step away in the folded
// rows (for odd R the middle row is the last folded row's first half).
// Every element is visited once, neighbouring threads take neighbouring
// elements, and no walk across the short rows is needed.
struct FoldWalk {
  int R, p, o, dp, dq;
  __device__ __forceinline__ FoldWalk(int rows, int tid, int nt) : R(rows) {
    p = tid / (rows + 1);
    o = tid - p * (rows + 1);
    dp = nt / (rows + 1);
    dq = nt - dp * (rows + 1);
  }
  __device__ __forceinline__ void rc(int& r, int& c) const {
    const bool first = o <= p;
    r = first ? p : R - 1 - p;
    c = first ? o : o - p - 1;
  }
  __device__ __forceinline__ void next() {
    o += dq;
    p += dp;
    if (o > R) {
      o -= R + 1;
      ++p;
    }
  }
};

struct KitaevWork {
  double* A;       // packed lower triangle, N (N+1) / 2 entries; reduced: d and e^2 scaled, the counts' grid
  double* d;       // N
  double* e;       // N
  double* uw;      // 2 N: (u, w) of the Householder step
  double* sc;      // 64 doubles
  double* xs;      // N + 8: the current column; reduced: the FP32 tridiagonal, padded to a multiple of 8 float2
};

// Number of eigenvalues below x of the symmetric tridiagonal (d, off-diagonal^2
// = e2): sign changes of p_{-1} = 1, p_0, ..., p_{N-1} with
// p_i = (d_i - x) p_{i-1} - e2_{i-1} p_{i-2} (Sturm).  A zero p_i takes the sign
// opposite to p_{i-1}.  The pair (p_i, p_{i-1}) is rescaled by 2^-+500 when
// it leaves [2^-500, 2^500].  Signs and exponents are read from the bit
// patterns with integer operations: only the recurrence itself uses the FP64
// pipe (three operations per step).
__device__ __forceinline__ int sturm_count(const double* d, const double* e2, int N, double x) {
  double pp = 1.0, p = d[0] - x;
  int hi = __double2hiint(p);
  uint32_t sprev = 0u;                                           // sign of p_{-1} = +1
  uint32_t s = ((hi & 0x7fffffff) | __double2loint(p)) == 0 ? 1u : ((uint32_t)hi >> 31);
  int cnt = (int)(s ^ sprev);
  sprev = s;
  for (int i = 1; i < N; ++i) {
    const double pn = fma(-e2[i - 1], pp, (d[i] - x) * p);
    pp = p;
    p = pn;
    hi = __double2hiint(p);
    const uint32_t zero = ((hi & 0x7fffffff) | __double2loint(p)) == 0;
    s = zero ? (sprev ^ 1u) : ((uint32_t)hi >> 31);
    cnt += (int)(s ^ sprev);
    sprev = s;
    const int ex = (hi >> 20) & 0x7ff;                           // biased exponent of p
    if (ex > 1023 + 500) {
      p *= 0x1p-500;
      pp *= 0x1p-500;
    } else if (ex < 1023 - 500 && ((__double2hiint(pp) >> 20) & 0x7ff) < 1023 - 500) {
      p *= 0x1p+500;
      pp *= 0x1p+500;
    }
  }
  return cnt;
}

// FP32 Sturm count of the scaled tridiagonal, entry i = (d_i, e_{i-1}^2),
// padded to a multiple of 8 with entries (2, 0), which change no sign (every
// x is below 2; the spectrum lies in [-1, 1], so nothing overflows): used only
// to isolate eigenvalues.
__device__ __forceinline__ int sturm_count32(const float2* de, int N, float x) {
  float pp = 0.0f, p = 1.0f;
  int cnt = 0;
  for (int i0 = 0; i0 < N; i0 += 8) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float2 t = de[i0 + i];
      const float pn = fmaf(-t.y, pp, (t.x - x) * p);
      cnt += (int)((__float_as_uint(pn) ^ __float_as_uint(p)) >> 31);
      pp = p;
      p = pn;
    }
    if (fmaxf(fabsf(p), fabsf(pp)) < 0x1p-50f) {
      p *= 0x1p+50f;
      pp *= 0x1p+50f;
    }
  }
  return cnt;
}

// Isolation of the eigenvalues of the scaled tridiagonal: G points strictly
// inside the Gershgorin interval (lo, hi), point k at lo + (k + 1) h with
// h = (hi - lo) / (G + 1), and the FP32 Sturm count at each, one point per
// thread of the group.  The count at a point is the number of eigenvalues
// below it, so eigenvalue idx lies between the last point whose count is
// <= idx and the next one: about log2(G + 1) rounds of bisection that every
// eigenvalue would otherwise repeat on its own are taken in one round.  The
// counts live in the reduced matrix's storage, free by then beyond the
// first 2N doubles (at most N^2 - 3N ints).
struct EigGrid {
  const float2* de;
  int* cnt;
  int N, G;
  float lo, hi, h;
  double glo, ghi;   // the interval widened by FP32's roundings: it holds the spectrum
  __device__ __forceinline__ EigGrid(const float2* de_, double* A, int n, float l, float u, int nt)
      : de(de_), cnt(reinterpret_cast<int*>(A + 2 * n)), N(n), G(min(nt, n * n - 3 * n)), lo(l), hi(u),
        h((u - l) / (float)(G + 1)) {
    const float out = 0x1p-20f * fmaxf(fabsf(l), fabsf(u));
    glo = (double)(l - out);
    ghi = (double)(u + out);
  }
  __device__ __forceinline__ float x(int k) const { return __fmaf_rn((float)(k + 1), h, lo); }
  // this thread's point (the caller syncs the group before the counts are read)
  __device__ __forceinline__ void fill(int tid) {
    if (tid < G) cnt[tid] = sturm_count32(de, N, x(tid));
  }
  // [a, b]: at most 2^-q of the interval wide (FP32 permitting), with
  // count(a) <= idx < count(b) as computed in FP32 (what it yields is certified
  // by the stage's own counts)
  __device__ __forceinline__ void isolate(int idx, float w, float& a, float& b) const {
    int i = 0, j = G;
    while (i < j) {
      const int mid = (i + j) >> 1;
      if (cnt[mid] > idx) j = mid; else i = mid + 1;
    }
    a = i == 0 ? lo : x(i - 1);
    b = i == G ? hi : x(i);
    for (int it = 0; it < 32 && b - a > w; ++it) {
      const float mid = 0.5f * (a + b);
      if (!(mid > a && mid < b)) break;
      if (sturm_count32(de, N, mid) > idx) b = mid; else a = mid;
    }
  }
};

// The leading 24 bits of an FP64 value as a float, by integer operations; 0
// below 2^-120 (|x| < 2^127).
__device__ __forceinline__ float lead32(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), e = (hi >> 20) & 0x7ffu;
  const uint32_t b = __funnelshift_l((uint32_t)__double2loint(x), hi, 3);
  return e < 1023 - 120 ? 0.0f : __uint_as_float(((b + 0x40000000u) & 0x7fffffffu) | (hi & 0x80000000u));
}
// x 2^k, k > 0, by its exponent field (0 stays 0).
__device__ __forceinline__ double shift_exponent(double x, int k) {
  const int hi = __double2hiint(x);
  return ((hi >> 20) & 0x7ff) == 0 ? x : __hiloint2double(hi + (k << 20), __double2loint(x));
}

// p_N(x) / p_N'(x) of the scaled tridiagonal: p in FP64 (three operations a
// step), its derivative in FP32 on the other pipe (the quotient needs no more
// than its leading digits).  An overflowing or lost value shows in the
// certification of the root.
__device__ __forceinline__ float newton_step64(const double* d, const double* e2, const float2* de, int N, double x) {
  const float xf = (float)x;
  double pp = 1.0, p = d[0] - x;
  float ppf = 1.0f, pf = lead32(p), dpp = 0.0f, dp = -1.0f;
  for (int i0 = 1; i0 < N; i0 += 4) {
    const int i1 = min(i0 + 4, N);
    for (int i = i0; i < i1; ++i) {
      const double pn = fma(-e2[i - 1], pp, (d[i] - x) * p);
      const float2 t = de[i];
      const float dpn = fmaf(-t.y, dpp, fmaf(t.x - xf, dp, -pf));
      dpp = dp;
      dp = dpn;
      pp = p;
      p = pn;
      ppf = pf;
      pf = lead32(p);
    }
    if (fmaxf(fabsf(pf), fabsf(ppf)) < 0x1p-30f) {
      p = shift_exponent(p, 30);
      pp = shift_exponent(pp, 30);
      pf = lead32(p);
      dp *= 0x1p+30f;
      dpp *= 0x1p+30f;
    }
  }
  return pf / dp;
}

// The eigenvalues of one warp's lanes, idx = its lane's index (N or more:
// none): FP32 isolation, Newton steps, then two of the stage's own counts
// certify each: count(x - tolc) <= idx < count(x + tolc), tolc several times
// the counts' own noise.  An eigenvalue that does not certify (clusters closer
// than FP32 separates, underflow) is found by the whole warp: 32 counts a round
// on points that span its bracket, which falls back to the Gershgorin interval
// where the bracket does not hold it, until it is tol wide (about 8 rounds,
// where one lane's bisection takes 40 counts); more than 6 of a warp bisect
// side by side.
// newton(x): refine a double; count(x): the stage's Sturm count.
template <class NEWTON, class COUNT>
__device__ __forceinline__ double warp_eigenvalues(const EigGrid& gr, int idx, float w, double tolc, double tol,
                                                   NEWTON newton, COUNT count) {
  const int lane = threadIdx.x & 31;
  const double glo = gr.glo, ghi = gr.ghi;
  float lo = gr.lo, hi = gr.hi;
  double x = 0.0;
  bool open = false;
  if (idx < gr.N) {
    gr.isolate(idx, w, lo, hi);
    x = newton(0.5f * (lo + hi));
    open = !(x >= glo && x <= ghi && count(x - tolc) <= idx && count(x + tolc) > idx);
  }
  unsigned left = __ballot_sync(kFull, open);
  if (__popc(left) > 6) {
    if (open) {
      double a = (double)lo, b = (double)hi;
      if (count(a) > idx) a = glo;
      if (count(b) <= idx) b = ghi;
      for (int it = 0; it < 64 && b - a > tol; ++it) {
        const double mid = 0.5 * (a + b);
        if (count(mid) > idx) b = mid; else a = mid;
      }
      x = 0.5 * (a + b);
    }
    left = 0u;
  }
  while (left) {
    const int who = __ffs(left) - 1, i = __shfl_sync(kFull, idx, who);
    left &= left - 1;
    const float pad = 0x1p-18f * (gr.hi - gr.lo);
    double a = fmax(glo, (double)(__shfl_sync(kFull, lo, who) - pad));
    double b = fmin(ghi, (double)(__shfl_sync(kFull, hi, who) + pad));
    bool below = false, above = false;                  // a, b known to enclose eigenvalue i
    for (int it = 0; it < 24 && (b - a > tol || !below || !above); ++it) {
      const double h = (b - a) * (1.0 / 31.0), at = lane < 31 ? fma((double)lane, h, a) : b;
      const unsigned over = __ballot_sync(kFull, count(at) > i);
      const int f = over ? __ffs(over) - 1 : 32;        // first point beyond eigenvalue i
      const double na = f > 0 ? __shfl_sync(kFull, at, f - 1) : (below ? a : glo);
      b = f < 32 ? __shfl_sync(kFull, at, f & 31) : (above ? b : ghi);
      a = na;
      below = above = true;
    }
    if (lane == who) x = 0.5 * (a + b);
  }
  return x;
}

// The Gershgorin interval of a group's tridiagonal: the least lo and the
// largest hi over its threads.  sc: 16 floats of the group.
template <bool MULTI>
__device__ __forceinline__ void group_interval(float& lo, float& hi, const Grp& g, float* sc) {
  const int tid = MULTI ? g.r : (int)threadIdx.x, nw = (MULTI ? g.tpc : (int)blockDim.x) >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(kFull, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(kFull, hi, o));
  }
  if ((tid & 31) == 0) {
    sc[2 * (tid >> 5)] = lo;
    sc[2 * (tid >> 5) + 1] = hi;
  }
  grp_sync<MULTI>(g);
  for (int w = 0; w < nw; ++w) {
    lo = fminf(lo, sc[2 * w]);
    hi = fmaxf(hi, sc[2 * w + 1]);
  }
}

// Sums of (lp, en, cf) and of a bound over a group, valid in its leader.  sc:
// 4 doubles per warp.
template <bool MULTI>
__device__ __forceinline__ void group_thermal(double& lp, double& en, double& cf, float& bd, const Grp& g, double* sc) {
  const int tid = MULTI ? g.r : (int)threadIdx.x, nw = (MULTI ? g.tpc : (int)blockDim.x) >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lp += __shfl_xor_sync(kFull, lp, o);
    en += __shfl_xor_sync(kFull, en, o);
    cf += __shfl_xor_sync(kFull, cf, o);
    bd += __shfl_xor_sync(kFull, bd, o);
  }
  if (nw == 1) return;
  grp_sync<MULTI>(g);
  if ((tid & 31) == 0) {
    double* mine = sc + 4 * (tid >> 5);
    mine[0] = lp;
    mine[1] = en;
    mine[2] = cf;
    *(float*)(mine + 3) = bd;
  }
  grp_sync<MULTI>(g);
  if (tid == 0)
    for (int w = 1; w < nw; ++w) {
      lp += sc[4 * w];
      en += sc[4 * w + 1];
      cf += sc[4 * w + 2];
      bd += *(const float*)(sc + 4 * w + 3);
    }
}

// Couplings scaled by a power of two so that the largest lies in [1, 2) (exact,
// undone at the end): FP32 helpers then never run out of exponents.  M's
// entries are the 2 J.  (Subnormal J: the least normal exponent, whose inverse
// times 2 is finite.)
__device__ __forceinline__ int coupling_exponent(const double* J) {
  const double m = fmax(fabs(J[0]), fmax(fabs(J[1]), fabs(J[2])));
  return m > 0.0 ? max((__double2hiint(m) >> 20) & 0x7ff, 1) - 1023 : 0;
}

// One single-fermion level's share of log pi, e and c_f (Sec. IV):
// log 2cosh x, -(eps/2) tanh x and x^2 sech^2 x with x = beta eps / 2.
__device__ __forceinline__ void thermal_add(double eps, double beta, double& lp, double& en, double& cf) {
  const double x = 0.5 * beta * eps;
  const double qx = exp(-2.0 * x), r = 1.0 / (1.0 + qx), t = x * r;
  lp += x + log1p(qx);
  en += -0.5 * eps * ((1.0 - qx) * r);
  cf += 4.0 * qx * (t * t);
}

// FP64 eigen-stage for one lattice: A = M^T M (Sec. IV, M_bw = 2 J_a u_bw) is
// reduced to tridiagonal form by Householder reflections, its eigenvalues
// mu_l = eps_l^2 found one per thread, and res = {log pi = sum_l
// log 2cosh(beta eps_l / 2), e, c_f}, valid in the group's leader (r == 0).
// eps_out (optional, device memory): the N energies eps, ascending.
// For periodic lattices (open ones: kitaev_logpi64_open).  Run by the chain's
// thread group g (warp-aligned) with its own work areas wk; every thread of the
// group calls, and only the group synchronises (MULTI: see grp_sync).
//
// Column j of the reduction, with x = A[j+1:, j], u = x - alpha e_1, tau = 2 /
// u^T u, p = tau A22 u, w = p - (tau p^T u / 2) u, A22 -= u w^T + w u^T, in three
// group barriers:
//   1. y = A22 x with H lanes per row, and per warp the partial of x^T y; beside
//      it one warp (each in turn) takes s = x^T x - x_0^2, alpha, u_0 and tau,
//      on which y does not wait;
//   2. u^T A22 u = x^T y - 2 alpha y_0 + alpha^2 a_00, p_l = tau (y_l - alpha
//      a_l0) and w;
//   3. the rank-2 update of the packed triangle, the first column (the next x)
//      into an array of its own.
// A column whose x is below 2^-59 ||A||_2 is taken as reduced.
// What bounds it: the FP64 pipe, which every warp instruction holds for about
// 64 cycles, so the count of FP64 instructions per warp -- hence the scalars in
// one warp instead of all, FP32 derivatives and two counts per eigenvalue
// (before: two counts, then Newton steps of five operations until one confirms
// the last), one Gershgorin interval in FP32 (before: a serial FP64 loop of one
// thread), and clusters found by the whole warp.  1024 chains of L = 6, four
// proposals: 1.74 ms (3.74); six tempering cycles of 1024 + 1024 chains of L = 8,
// four Gibbs steps each: 6.9 ms (15.0).
template <bool MULTI>
__device__ inline void kitaev_logpi64(const Grp& g, const uint32_t* v, int L, const double* J, double beta,
                               const KitaevWork& wk, double (&res)[3], double* eps_out = nullptr) {
  const int N = L * L, tid = MULTI ? g.r : (int)threadIdx.x, nt = MULTI ? g.tpc : (int)blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  double* A = wk.A;
  double2* uw = reinterpret_cast<double2*>(wk.uw);     // (u, w) of a row; .y holds y until w is known
  double* xs = wk.xs;
  const int kJ = coupling_exponent(J);
  const double sJ = ldexp(2.0, -kJ), tx = sJ * J[0], ty = sJ * J[1], tz = sJ * J[2];
  // A = M^T M, row w accumulated in a fixed order (z, x, y bond of w, then the
  // three whites of that black site)
  for (int e = tid; e < N * (N + 1) / 2; e += nt) A[e] = 0.0;
  grp_sync<MULTI>(g);
  for (int w = tid; w < N; w += nt) {
    double* row = A + tri(w, 0);                    // lower-triangle row w: columns 0..w
    const int i = w / L, j = w - i * L;
    for (int typ = 0; typ < 3; ++typ) {
      int bi = i, bj = j;
      if (typ == 1) bi = (i == 0) ? L - 1 : i - 1;
      if (typ == 2) bj = (j == 0) ? L - 1 : j - 1;
      const int b = bi * L + bj;
      const double mz = site_bit(v, b) ? tz : -tz;
      const double mw = (typ == 0) ? mz : (typ == 1 ? tx : ty);
      const int wz = b;
      const int wx = ((bi + 1 == L) ? 0 : bi + 1) * L + bj;
      const int wy = bi * L + ((bj + 1 == L) ? 0 : bj + 1);
      if (wz <= w) row[wz] += mw * mz;
      if (wx <= w) row[wx] += mw * tx;
      if (wy <= w) row[wy] += mw * ty;
    }
  }
  grp_sync<MULTI>(g);
  // sc: floats 0..15 partials of |x|^2 without x_0 (FP32, tells a reduced
  // column); doubles 16.. partials of x^T y; 48.. alpha, u_0, tau, y_0
  float* scS = reinterpret_cast<float*>(wk.sc);
  double* scQ = wk.sc + 16;
  double* scA = wk.sc + 48;
  auto column_sum = [&](float part) {           // this thread's share of |x|^2 - x_0^2
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(kFull, part, o);
    if (lane == 0) scS[warp] = part;
  };
  {
    float part = 0.0f;
    for (int r = tid; r < N - 1; r += nt) {
      const double a = A[tri(1 + r, 0)];
      const float f = lead32(a);
      xs[r] = a;
      if (r >= 1) part = fmaf(f, f, part);
    }
    column_sum(part);
  }
  grp_sync<MULTI>(g);
  const float amax = fabsf(lead32(tx)) + fabsf(lead32(ty)) + fabsf(lead32(tz));    // sqrt of a bound on ||A||_2
  const float tiny = 0x1p-118f * (amax * amax) * (amax * amax);
  for (int j = 0; j < N - 2; ++j) {
    const int m = N - j - 1, j1 = j + 1;
    float sf = 0.0f;
    for (int w = 0; w < nw; ++w) sf += scS[w];
    if (sf <= tiny) {
      // column already reduced: no reflection
      if (tid == 0) {
        wk.d[j] = A[tri(j, j)];
        wk.e[j] = xs[0];
      }
      grp_sync<MULTI>(g);
      float part = 0.0f;
      for (int r = tid; r < m - 1; r += nt) {
        const double a = A[tri(j1 + 1 + r, j1)];
        const float f = lead32(a);
        xs[r] = a;
        if (r >= 1) part = fmaf(f, f, part);
      }
      column_sum(part);
      grp_sync<MULTI>(g);
      continue;
    }
    // 1. y, x^T y; the scalars
    if (warp == j % nw) {
      double s = 0.0;
      for (int r = 1 + lane; r < m; r += 32) s = fma(xs[r], xs[r], s);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
      const double x0 = xs[0], sig = fma(x0, x0, s), nrm = sqrt(sig);
      const double alpha = (x0 >= 0.0) ? -nrm : nrm;
      // tau = 2 / (u_0^2 + s) = 1 / (|x|^2 + |x_0| |x|)
      const double tau = 1.0 / fma(fabs(x0), nrm, sig);
      if (lane == 0) {
        scA[0] = alpha;
        scA[1] = x0 - alpha;
        scA[2] = tau;
        wk.d[j] = A[tri(j, j)];
        wk.e[j] = alpha;
      }
    }
    double q = 0.0;
    const int H = row_lanes64(m, nt), h = lane & (H - 1);
    for (int lf = warp * (32 / H); lf < m; lf += nt / H) {
      const int lr = lf + lane / H, l = min(lr, m - 1);
      double y = 0.0, y1 = 0.0;
      sym_row(A, xs, j1, m, l, h, H, y, y1, [](double a, double x, double& t) { t = fma(a, x, t); });
      y += y1;
      for (int o = 1; o < H; o <<= 1) y += __shfl_xor_sync(kFull, y, o);
      if (lr < m && h == 0) {
        uw[l].y = y;
        if (l == 0) scA[3] = y;
        q = fma(xs[l], y, q);
      }
    }
    if (warp * (32 / H) < m) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(kFull, q, o);
    }
    if (lane == 0) scQ[warp] = q;
    grp_sync<MULTI>(g);
    // 2. u and w
    if (warp * 32 < m) {
      const double alpha = scA[0], u0 = scA[1], tau = scA[2];
      double xy = scQ[0];
      for (int w = 1; w < nw; ++w) xy += scQ[w];
      // K = tau^2 / 2 (x^T y + alpha (alpha a_00 - 2 y_0))
      const double uAu = fma(alpha, fma(alpha, A[tri(j1, j1)], -2.0 * scA[3]), xy);
      const double nK = (-0.5 * tau) * (tau * uAu);
      for (int l = tid; l < m; l += nt) {
        const double u = l == 0 ? u0 : xs[l];
        const double p = tau * fma(-alpha, A[tri(j1 + l, j1)], uw[l].y);
        uw[l] = make_double2(u, fma(nK, u, p));
      }
    }
    grp_sync<MULTI>(g);
    // 3. A22 -= u w^T + w u^T: the first column (the next x), then the rest of
    // the packed triangle (rows and columns 1..m-1) in the folded order of FoldWalk
    float part = 0.0f;
    const double2 c0 = uw[0];
    for (int r = tid; r < m; r += nt) {
      double* a = A + tri(j1 + r, j1);
      const double2 ur = uw[r];
      const double x = fma(-ur.x, c0.y, fma(-ur.y, c0.x, *a));
      if (r == 0) *a = x;
      else xs[r - 1] = x;
      if (r >= 2) {
        const float f = lead32(x);
        part = fmaf(f, f, part);
      }
    }
    const int ntri = (m - 1) * m / 2;
    FoldWalk fw(m - 1, tid, nt);
    for (int e = tid; e < ntri; e += nt, fw.next()) {
      int r, c;
      fw.rc(r, c);
      double* a = A + tri(j1 + 1 + r, j1 + 1 + c);
      const double2 ur = uw[r + 1], uc = uw[c + 1];
      *a = fma(-ur.x, uc.y, fma(-ur.y, uc.x, *a));
    }
    column_sum(part);
    grp_sync<MULTI>(g);
  }
  if (tid == 0) {
    wk.d[N - 2] = A[tri(N - 2, N - 2)];
    wk.d[N - 1] = A[tri(N - 1, N - 1)];
    wk.e[N - 2] = xs[0];
    wk.e[N - 1] = 0.0;
  }
  grp_sync<MULTI>(g);
  float lo = 3e38f, hi = -3e38f;
  for (int i = tid; i < N; i += nt) {
    const double d = wk.d[i], r = fabs(wk.e[i]) + (i > 0 ? fabs(wk.e[i - 1]) : 0.0);
    lo = fminf(lo, (float)(d - r));
    hi = fmaxf(hi, (float)(d + r));
  }
  group_interval<MULTI>(lo, hi, g, reinterpret_cast<float*>(scQ));
  // the tridiagonal scaled by 2^-ks to a spectrum inside [-1, 1]: d and e^2 in
  // the matrix's storage, FP32 copies for isolation
  const float big = fmaxf(fabsf(lo), fabsf(hi));
  const int ks = big > 0.0f ? (int)((__float_as_uint(big) >> 23) & 0xffu) - 127 + 2 : 0;
  const double s1 = ldexp(1.0, -ks);
  double* ds = A;
  double* es = A + N;
  float2* de = reinterpret_cast<float2*>(xs);
  for (int i = tid; i < ((N + 7) & ~7); i += nt) {
    float2 t = make_float2(2.0f, 0.0f);
    if (i < N) {
      const double d = wk.d[i] * s1, e = wk.e[i] * s1;
      ds[i] = d;
      es[i] = e * e;
      const double em = i > 0 ? wk.e[i - 1] * s1 : 0.0;
      t = make_float2((float)d, (float)(em * em));
    }
    de[i] = t;
  }
  grp_sync<MULTI>(g);
  EigGrid gr(de, A, N, lo * (float)s1, hi * (float)s1, nt);
  gr.fill(tid);
  grp_sync<MULTI>(g);
  const float range = gr.hi - gr.lo;
  const double tol = 0x1p-50 * (double)(range + fabsf(gr.lo)), back = ldexp(1.0, ks + 2 * kJ);
  // each step shrinks the error at least as it did the one before: done when the
  // next one would be below FP64's spacing
  auto newton = [&](float x0) {
    double x = (double)x0;
    float prev = 0.0f;
    for (int it = 0; it < 6; ++it) {
      const float step = newton_step64(ds, es, de, N, x);
      x -= (double)step;
      if (!(step * step > 0x1p-54f * range * prev)) break;
      prev = fabsf(step);
    }
    return x;
  };
  double lp = 0.0, en = 0.0, cf = 0.0;
  for (int base = 32 * warp; base < N; base += nt) {
    const int idx = base + lane;
    const double x = warp_eigenvalues(gr, idx, range * 0x1p-22f, 4.0 * tol, tol, newton,
                                      [&](double at) { return sturm_count(ds, es, N, at); });
    if (idx < N) {
      const double eps = sqrt(fmax(x, 0.0) * back);
      if (eps_out) eps_out[idx] = eps;
      thermal_add(eps, beta, lp, en, cf);
    }
  }
  float none = 0.0f;
  group_thermal<MULTI>(lp, en, cf, none, g, wk.sc);
  res[0] = lp;
  res[1] = en;
  res[2] = cf;
}

}  // namespace crbm
