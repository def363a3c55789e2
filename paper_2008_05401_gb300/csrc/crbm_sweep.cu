// Local-update Metropolis sweeps of the Ising model (the paper's baseline,
// Sec. III): checkerboard order, the sites with (i + j) even, then the odd
// ones (even L, so the sites of one colour never neighbour each other); site
// (i, j) with u unequal neighbours flips iff its uniform is below
// e^{-beta dE}, dE = 2 J (4 - 2u).  The uniform of site n is word n % 4 of
// Philox block n / 4 of tag kTagLocal at the sweep's step.
//
// The lattices stay packed in shared memory and a thread owns whole words of
// 32 sites: neighbours are funnel shifts of the packed rows, the four unequal
// bits of all 32 sites are counted with bit-sliced adders, and a word of the
// other colour's flips costs no loop over sites.  Each site's uniform meets
// the two thresholds that can reject it (u = 0, 1 for J > 0) in integers, by
// the borrow of a subtraction shifted into a mask; both colours use the same
// eight Philox blocks of a word, drawn once.  Energies and magnetisations
// follow from the flips (a flip changes the unequal pairs by 4 - 2u and the
// ones by 1 - 2v), exact integers; warps of their own turn them into the
// FP64 observables of each sweep, one sweep behind, so that no sweep waits on
// the FP64 pipe.  What bounds it is the issue of the Philox rounds (about 60
// of some 80 instructions per four sites).
// 512 chains of 64 x 64, 100 sweeps with the FP64 F of the last and the
// read-back: 0.52 ms (one site at a time, FP64 comparison, Philox per colour,
// counts by a pass over the sites: 4.32 ms).
#include <algorithm>

#include "crbm_device.cuh"
#include "crbm_kernels.h"

namespace crbm {

namespace {

constexpr int kMaxTpc = 512;      // most threads of a chain
constexpr int kWorkers = 128;     // least worker threads of a CTA

struct SweepParams {
  JobDev j;
  int S, tpc, nc;     // sweeps; worker threads per chain (a power of two); chains per CTA
  int add;            // 1: add each sweep's observables to the sums and the trace
};

// Accept rules of one chain.  Site word w against class c (0: the class of
// the largest dE > 0, 1: the next): accepted iff w <= t1 and on[c], which is
// (w + 1/2) 2^-32 < e^{-beta dE} exactly (nt1[c] = ~t1); the classes of two
// unequal neighbours and beyond (dE <= 0) by their masks.
struct Rule {
  uint32_t nt1[2], on[2], rest[3];
};

// 32 sites of the flat lattice from site o (0 <= o < N) on, periodic in N:
// bit b is site (o + b) mod N.  The word after the last is zero.
__device__ __forceinline__ uint32_t flat_window(const uint32_t* p, int o, int N, int Wd) {
  const int wi = o >> 5;
  if ((N & 31) == 0) return __funnelshift_r(p[wi], p[wi + 1 == Wd ? 0 : wi + 1], o & 31);
  if (N < 32) {       // L = 2 or 4: N divides 32
    uint32_t r = p[0];
    for (int s = N; s < 32; s <<= 1) r |= r << s;
    return __funnelshift_r(r, r, o);
  }
  const uint32_t x = __funnelshift_r(p[wi], p[wi + 1], o & 31);
  const int c = N - o;
  return c < 32 ? (x & ((1u << c) - 1u)) | (p[0] << c) : x;
}

struct Neighbours {
  uint32_t up, down, left, right;
};

// Neighbour bits of the 32 sites of word w; e0 / el: its sites in column 0 / L - 1.
__device__ __forceinline__ Neighbours neighbours(const uint32_t* p, int w, int L, int N, int Wd, uint32_t e0,
                                                 uint32_t el) {
  const int o = 32 * w;
  auto wrap = [&](int x) { return x < 0 ? x + N : (x >= N ? x - N : x); };
  Neighbours n;
  n.up = flat_window(p, wrap(o - L), N, Wd);
  n.down = flat_window(p, wrap(o + L), N, Wd);
  n.left = flat_window(p, wrap(o - 1), N, Wd);
  n.right = flat_window(p, wrap(o + 1), N, Wd);
  if (e0) n.left = (n.left & ~e0) | (flat_window(p, wrap(o + L - 1), N, Wd) & e0);
  if (el) n.right = (n.right & ~el) | (flat_window(p, wrap(o + 1 - L), N, Wd) & el);
  return n;
}

// reject = 2 reject + (w > t1), nt1 = ~t1: the carry of w + nt1 shifted into the mask.
__device__ __forceinline__ void push_reject(uint32_t& reject, uint32_t w, uint32_t nt1) {
  asm("{\n.reg .u32 d;\nadd.cc.u32 d, %1, %2;\naddc.u32 %0, %0, %0;\n}\n" : "+r"(reject) : "r"(w), "r"(nt1));
}

// WORDS: words of a thread (1 up to kMaxTpc words a chain; L = 256 has 2048).
template <int WORDS>
__global__ void __launch_bounds__(kMaxTpc + 32, 1) ising_sweep_kernel(const __grid_constant__ SweepParams p) {
  const JobDev& jb = p.j;
  const int L = jb.L, N = jb.N, Wd = jb.Wd, P = Wd + 1;
  const int tid = threadIdx.x, tpc = p.tpc, nc = p.nc, workers = tpc * nc;
  extern __shared__ __align__(16) uint32_t sweep_smem[];
  Rule* rules = (Rule*)sweep_smem;                         // nc
  int2* cnt = (int2*)(rules + nc + (nc & 1));              // [2][nc] changes of (pairs, ones), by sweep parity
  uint32_t* even = (uint32_t*)(cnt + 2 * nc);              // Wd: sites with (i + j) even
  uint32_t* col0 = even + Wd;                              // Wd: sites with j = 0
  uint32_t* colL = col0 + Wd;                              // Wd: sites with j = L - 1
  uint32_t* planes = colL + Wd;                            // [nc][P]

  const int c_first = (int)blockIdx.x * nc;
  for (int w = tid; w < Wd; w += blockDim.x) {
    uint32_t ev = 0u, e0 = 0u, el = 0u;
    for (int b = 0; b < 32; ++b) {
      const int n = 32 * w + b;
      if (n >= N) break;
      const int i = n / L, j = n - i * L;
      ev |= (uint32_t)(((i + j) & 1) == 0) << b;
      e0 |= (uint32_t)(j == 0) << b;
      el |= (uint32_t)(j == L - 1) << b;
    }
    even[w] = ev;
    col0[w] = e0;
    colL[w] = el;
  }
  for (int e = tid; e < nc * P; e += blockDim.x) {
    const int g = e / P, w = e - g * P;
    planes[e] = (w < Wd && c_first + g < jb.n_chains) ? jb.bits[(size_t)(c_first + g) * Wd + w] : 0u;
  }
  for (int e = tid; e < 2 * nc; e += blockDim.x) cnt[e] = make_int2(0, 0);
  for (int g = tid; g < nc; g += blockDim.x) {
    Rule r;
    const double beta = c_first + g < jb.n_chains ? 1.0 / jb.T[c_first + g] : 1.0;
    auto thr = [&](int u) { return exp(-beta * ((2.0 * jb.J[0]) * (double)(4 - 2 * u))) * 0x1p32; };
    const bool ferro = jb.J[0] >= 0.0;
    for (int c = 0; c < 2; ++c) {
      const double t = thr(ferro ? c : 4 - c);
      const double k = ceil(t - 0.5);                      // accepted words: 0 .. k - 1
      r.on[c] = t - 0.5 > 0.0 ? ~0u : 0u;
      r.nt1[c] = k >= 0x1p32 ? 0u : ~(r.on[c] ? (uint32_t)k - 1u : 0u);
    }
    for (int c = 0; c < 3; ++c) r.rest[c] = 0xFFFFFFFFp0 + 0.5 < thr(ferro ? 2 + c : 2 - c) ? ~0u : 0u;
    rules[g] = r;
  }
  __syncthreads();

  const unsigned long long step0 = *(volatile unsigned long long*)jb.step;
  if (tid < workers) {
    const int g = tid / tpc, r = tid - g * tpc, c = c_first + g;
    const bool active = c < jb.n_chains;
    const uint32_t cid = (uint32_t)(jb.cid_base + (uint64_t)c);
    uint32_t* v = planes + g * P;
    const bool ferro = jb.J[0] >= 0.0;
    const Rule rule = rules[g];
    const int span = tpc < 32 ? tpc : 32;
    auto reduce = [&](int x) {                             // over the chain's lanes of this warp
      if (span == 32) return __reduce_add_sync(kFull, x);
      for (int o = 1; o < span; o <<= 1) x += __shfl_xor_sync(kFull, x, o);
      return x;
    };
    // the chain's counts at the start, as the changes of "sweep -1" (parity 1)
    {
      int pairs = 0, ones = 0;
      if (active)
        for (int w = r; w < Wd; w += tpc) {
          const uint32_t x = v[w], live = 32 * w + 32 <= N ? ~0u : (1u << (N - 32 * w)) - 1u;
          const Neighbours nb = neighbours(v, w, L, N, Wd, col0[w], colL[w]);
          pairs += __popc((x ^ nb.right) & live) + __popc((x ^ nb.down) & live);
          ones += __popc(x);
        }
      pairs = reduce(pairs);
      ones = reduce(ones);
      if ((r & (span - 1)) == 0) {
        atomicAdd(&cnt[nc + g].x, pairs);
        atomicAdd(&cnt[nc + g].y, ones);
      }
    }
    __syncthreads();
    unsigned long long nacc = 0;
    for (int s = 0; s < p.S; ++s) {
      const uint32_t step = (uint32_t)(step0 + (uint64_t)s);
      uint32_t rej[WORDS][2];
      int dpairs = 0, dones = 0;
#pragma unroll
      for (int colour = 0; colour < 2; ++colour) {
#pragma unroll
        for (int q = 0; q < WORDS; ++q) {
          const int w = r + q * tpc;
          if (!active || w >= Wd) break;
          if (colour == 0) {
            rej[q][0] = rej[q][1] = 0u;
#pragma unroll 4
            for (int b = 7; b >= 0; --b) {
              const uint4 u = philox4x32_10_rk(make_uint4((uint32_t)(8 * w + b), kTagLocal, step, cid), jb.rk);
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                push_reject(rej[q][e], u.w, rule.nt1[e]);
                push_reject(rej[q][e], u.z, rule.nt1[e]);
                push_reject(rej[q][e], u.y, rule.nt1[e]);
                push_reject(rej[q][e], u.x, rule.nt1[e]);
              }
            }
          }
          const uint32_t x = v[w];
          const Neighbours nb = neighbours(v, w, L, N, Wd, col0[w], colL[w]);
          const uint32_t a = x ^ nb.up, d = x ^ nb.down, l = x ^ nb.left, t = x ^ nb.right;
          // u = a + d + l + t of every site: classes u = 0 .. 4
          const uint32_t odd = a ^ d ^ l ^ t, two = (a & d) | (l & t), both = a & d & l & t;
          const uint32_t c0 = ~(a | d | l | t), c1 = odd & ~two, c3 = odd & two, c4 = both,
                         c2 = ~(odd | c0 | c4);
          const uint32_t ext = ferro ? c0 : c4, mid = ferro ? c1 : c3, f3 = ferro ? c3 : c1, f4 = ferro ? c4 : c0;
          const uint32_t acc = (ext & ~rej[q][0] & rule.on[0]) | (mid & ~rej[q][1] & rule.on[1]) |
                               (c2 & rule.rest[0]) | (f3 & rule.rest[1]) | (f4 & rule.rest[2]);
          const uint32_t live = 32 * w + 32 <= N ? ~0u : (1u << (N - 32 * w)) - 1u;
          const uint32_t flip = acc & (colour == 0 ? even[w] : ~even[w]) & live;
          // only this thread writes word w, and the sites of this colour only:
          // what other threads read of it meanwhile does not change
          v[w] = x ^ flip;
          dpairs += 4 * (__popc(flip & c0) - __popc(flip & c4)) + 2 * (__popc(flip & c1) - __popc(flip & c3));
          const int nf = __popc(flip);
          dones += nf - 2 * __popc(flip & x);
          nacc += (unsigned long long)nf;
        }
        if (colour == 1) {
          dpairs = reduce(dpairs);
          dones = reduce(dones);
          if ((r & (span - 1)) == 0 && active) {
            atomicAdd(&cnt[(s & 1) * nc + g].x, dpairs);
            atomicAdd(&cnt[(s & 1) * nc + g].y, dones);
          }
        }
        __syncthreads();
      }
    }
    if (active) {
      for (int w = r; w < Wd; w += tpc) jb.bits[(size_t)c * Wd + w] = v[w];
      if (nacc) atomicAdd(&jb.acc[c], nacc);
    }
  } else {
    // four lanes per chain, one observable each: E, E^2, |M|, M^2
    const int e = tid - workers, g = e >> 2, o = e & 3, c = c_first + g;
    const bool on = g < nc && c < jb.n_chains;
    int pairs = 0, ones = 0;
    double E = 0.0, term = 0.0, sum = on ? jb.obs[(size_t)c * kNobs + o] : 0.0;
    __syncthreads();
    if (on) {
      pairs = cnt[nc + g].x;
      ones = cnt[nc + g].y;
    }
    __syncwarp();
    if (on && o == 0) cnt[nc + g] = make_int2(0, 0);
    for (int s = 0; s < p.S; ++s) {
      __syncthreads();
      __syncthreads();
      // the changes of sweep s; the workers add to this parity again two sweeps on
      if (on) {
        const int2 d = cnt[(s & 1) * nc + g];
        pairs += d.x;
        ones += d.y;
      }
      __syncwarp();
      if (on) {
        if (o == 0) cnt[(s & 1) * nc + g] = make_int2(0, 0);
        E = -jb.J[0] * (double)(2 * N - 2 * pairs);
        const double M = (double)(2 * ones - N), x = o < 2 ? E : fabs(M);
        term = (o & 1) ? x * x : x;
        sum += term;
        if (p.add && o == 0) trace_store(jb, c, step0 + (uint64_t)s, E);
      }
    }
    if (on) {
      jb.obs_t[(size_t)c * kNobs + o] = term;
      if (p.add) jb.obs[(size_t)c * kNobs + o] = sum;
      if (o == 0) {
        jb.Ephys[c] = E;
        jb.logpi[c] = -(1.0 / jb.T[c]) * E;
      }
    }
  }
}

__global__ void add_steps_kernel(unsigned long long* step, int S) { *step += (unsigned long long)S; }

}  // namespace

cudaError_t launch_ising_sweeps(const JobDev& j, int S, bool add, cudaStream_t st) {
  if (j.n_chains == 0 || S == 0) return cudaSuccess;
  SweepParams p;
  p.j = j;
  p.S = S;
  p.add = add ? 1 : 0;
  p.tpc = 1;
  while (p.tpc < j.Wd && p.tpc < kMaxTpc) p.tpc *= 2;
  p.nc = std::max(1, std::min(32, kWorkers / p.tpc));      // tpc nc: whole warps
  const int stat = (4 * p.nc + 31) / 32 * 32;
  const size_t smem = (size_t)(p.nc + (p.nc & 1)) * sizeof(Rule) + 2 * (size_t)p.nc * sizeof(int2) +
                      3 * (size_t)j.Wd * 4 + (size_t)p.nc * (j.Wd + 1) * 4;
  const int grid = (j.n_chains + p.nc - 1) / p.nc, nt = p.tpc * p.nc + stat;
  if (j.Wd <= kMaxTpc) ising_sweep_kernel<1><<<grid, nt, smem, st>>>(p);
  else ising_sweep_kernel<4><<<grid, nt, smem, st>>>(p);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  add_steps_kernel<<<1, 1, 0, st>>>(j.step, S);
  return cudaGetLastError();
}

}  // namespace crbm
