// Fused CRBM proposal + Metropolis-Hastings kernel (one launch runs S
// proposals; lattices stay in shared memory for the whole launch).
//
// Per proposal and chain (arXiv:2008.05401):
//   g x [hidden half-step (Eq. B2), visible half-step (Eq. B3)]   -> v'
//   F(v') (Eq. 13) and the lattice sums of v'
//   log pi(v'): Ising -beta E (Eq. 14) | Kitaev sum log 2cosh(beta eps/2) (Sec. IV)
//   log r = [log pi(v') - log pi(v)] + [F(v') - F(v)], accept iff log u < log r
//   (Eq. B5 with the pair (pi, P_CRBM); the Gibbs kernel is reversible w.r.t.
//   P_CRBM, App. B.1), then observables of the state after the decision.
// Template parameters: model kind, precision, and K, k fixed at compile time
// for the common filter banks (0 = runtime values).
#pragma once
#include "crbm_device.cuh"
#include "crbm_df64.cuh"
#include "crbm_open64.cuh"
#include "crbm_local.cuh"
#include "crbm_kernels.h"

#include <type_traits>

namespace crbm {

struct ChainSm {
  double F, Fb, lp, E;
  double ot[kNobs];      // observables of the current lattice
  double os[kNobs];      // running sums
  double Fp, Bp, lpp, Ep;
  double lpb, lppb;      // bounds on |log pi - FP64 path's log pi| (current, proposed)
  double cfp;            // Kitaev: c_f of the proposal
  double beta;
  double logu;           // log u of the current proposal's MH draw
  double cst, mgs;       // constant margin terms; tensor-core kernel: the current
                         // state's margin terms (both off the MH thread's path)
  unsigned long long acc, rec, rec_mh;
  int cur, flag_rec, flag_acc;
  int onesp, pairsp;     // lattice counts of the proposal
};

__host__ __device__ inline size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

// Shared-memory work areas of one Kitaev chain (one per thread group of the
// CTA): the packed lower triangle of A (N (N+1) / 2 FP64 or double-FP32
// entries), d, e, (u, w), 64 doubles of scratch, the current column (or the
// FP32 tridiagonal padded to a multiple of 8) and the proposed spectrum of a
// local sweep (N).
__host__ __device__ inline size_t kitaev_work_bytes(int N) {
  const size_t n = (size_t)N;
  return align16(n * (n + 1) / 2 * 8) + 2 * align16(n * 8) + n * 16 + align16(64 * 8) + align16((n + 8) * 8) +
         align16(n * 8);
}

// The mixed path's FP64 free energy (rare), out of line to spare registers.
static __device__ __noinline__ void free_energy64(const JobDev& jb, const Grp& g, const uint32_t* v, FreeSum* out) {
  *out = free_phase64(jb, jb.f64, g, v);
}

// F of a lattice by the threads of an FP64-path CTA and in their order of sums,
// valid in thread 0.  Every thread of the CTA (256 or more) calls.
static __device__ __noinline__ double path64_free(const JobDev& jb, const Grp& g, const uint32_t* v, double* scratch) {
  Grp q = g;
  q.r = (int)threadIdx.x;
  q.tpc = kThreads / jb.nc64;
  q.active = q.r < q.tpc;
  FreeSum f = free_phase64(jb, jb.f64, q, v);
  reduce_free<kFP64, false>(f, q, scratch);
  return free_value<kFP64>(jb, f);
}
// An Ising CTA's chains with flag_rec == flag, one after the other (rare): F of
// their proposals prop(i) as the FP64 path has it, and of the current lattices
// cur(i) whose F carries a bound.  Ends with a barrier.
template <class PROP, class CUR>
__device__ __forceinline__ void ising_redo64(const JobDev& jb, const Grp& g, ChainSm* cs, int flag, double* scratch,
                                             PROP prop, CUR cur) {
  for (int i = 0; i < jb.nc; ++i) {
    const bool redo = cs[i].Fb != 0.0;
    if (cs[i].flag_rec != flag) continue;
    const double Fp = path64_free(jb, g, prop(i), scratch), F = redo ? path64_free(jb, g, cur(i), scratch) : 0.0;
    __syncthreads();                // every thread has read the chain's flags
    if (threadIdx.x == 0) {
      cs[i].Fp = Fp;
      cs[i].Bp = 0.0;
      if (redo) {
        cs[i].F = F;
        cs[i].Fb = 0.0;
      }
    }
  }
  __syncthreads();
}

// Observables of a lattice: Ising from E and the number of ones; Kitaev from
// (e, c_f) of its spectrum and its count of hexagons with flux -1.
template <int KIND>
__device__ __forceinline__ void observables(const JobDev& jb, double E, double cf, int ones, int flux,
                                            double (&ot)[kNobs]) {
  ot[0] = E;
  ot[1] = E * E;
  if (KIND == kIsing) {
    const double M = (double)(2 * ones - jb.N);
    ot[2] = fabs(M);
    ot[3] = M * M;
  } else {
    ot[2] = cf;
    ot[3] = (double)flux / (double)jb.nhex;
  }
}
// Ising energy from the number of unequal nearest-neighbour pairs (2 N bonds).
__device__ __forceinline__ double ising_energy(const JobDev& jb, int pairs) {
  return -jb.J[0] * (double)(2 * jb.N - 2 * pairs);
}

// The mixed path's FP32 tables at sp (copied by the CTA's nt threads; a barrier
// before their first use is the caller's), their pointers into tb; returns the
// end of the area.
template <int KC>
__device__ __forceinline__ unsigned char* mixed_tables(const JobDev& jb, unsigned char* sp, Tabs& tb, int tid, int nt) {
  const int T = 1 << jb.k, nlut = jb.K * jb.k * T, nq = jb.k * T;   // nq: entries of a filter-interleaved table
  auto take = [&](size_t bytes) {
    unsigned char* at = sp;
    sp += align16(bytes);
    return at;
  };
  if constexpr (KC != 0) {
    // an entry is 32 / KC copies of its KC filters, 128 bytes: the lanes of a
    // quarter (KC = 4) or half warp (KC = 2), which one pass serves, read from
    // copies and so from banks of their own
    float* ti[3];
    for (int i = 0; i < 3; ++i) ti[i] = (float*)take((size_t)nq * 128);
    float* bd = (float*)take((size_t)nlut * 4);
    for (int i = tid; i < nlut; i += nt) bd[i] = jb.bd[i];
    const float *gd = (const float*)jb.fd4, *gh = (const float*)jb.fh4, *gl = (const float*)jb.fl4;
    for (int i = tid; i < nq * 32; i += nt) {
      const int e = (i >> 5) * 4 + (i & (KC - 1));
      ti[0][i] = gd[e];
      ti[1][i] = gh[e];
      ti[2][i] = gl[e];
    }
    const int copy = KC * (tid & (32 / KC - 1));
    tb.fdi = ti[0] + copy;
    tb.fhi = ti[1] + copy;
    tb.fli = ti[2] + copy;
    tb.bd = bd;
  } else {
    float* t[4];
    for (int i = 0; i < 4; ++i) t[i] = (float*)take((size_t)nlut * 4);
    for (int i = tid; i < nlut; i += nt) {
      t[0][i] = jb.fd[i];
      t[1][i] = jb.bd[i];
      t[2][i] = jb.fh[i];
      t[3][i] = jb.fl[i];
    }
    tb.fd = t[0];
    tb.bd = t[1];
    tb.fh = t[2];
    tb.fl = t[3];
  }
  return sp;
}

// n_gibbs block-Gibbs steps (Eqs. B2, B3) from v into vp through the hidden
// planes h; xv, xvp, xh: their expanded rows (xv given; xvp left behind).  sync:
// the group's barrier, also the last thing done.
template <int PREC, int KC, int kC, class SYNC>
__device__ __forceinline__ void gibbs_steps(const JobDev& jb, const Tabs& tb, const Grp& g, const uint32_t* v,
                                            uint32_t* vp, uint32_t* h, const uint64_t* xv, uint64_t* xvp, uint64_t* xh,
                                            int P, int n_gibbs, uint32_t step, unsigned& nrec, SYNC sync) {
  const int nblk = (jb.N + 3) >> 2, K = KC ? KC : jb.K;
  const bool narrow = (jb.L & 31) != 0;
  for (int sub = 0; sub < n_gibbs; ++sub) {
    if constexpr (PREC == kMixed) {
      hidden_phase<KC, kC>(jb, tb, g, v, xv, h, P, step, sub, nrec, 0, nblk);
      if (narrow) {
        sync();
        expand_rows(h, P, xh, jb.L, K, g.r, g.tpc);
      }
      sync();
      visible_phase<KC, kC>(jb, tb, g, h, xh, vp, P, step, sub, nrec, 0, nblk);
      if (narrow) {
        sync();
        expand_rows(vp, P, xvp, jb.L, 1, g.r, g.tpc);
      }
      xv = xvp;
    } else {
      hidden_phase64(jb, tb, g, v, h, P, step, sub, sync);
      sync();
      visible_phase64(jb, tb, g, h, vp, P, step, sub, sync);
    }
    sync();
    v = vp;
  }
}

// log pi, e and c_f of a Kitaev lattice in FP64, valid in the group's leader
// (the open lattices' jobs run in FP64 only).
template <int PREC, bool MULTI>
__device__ __forceinline__ void fp64_spectrum(const JobDev& jb, const Grp& g, const uint32_t* v, double beta,
                                              const KitaevWork& wk, double (&res)[3], double* eps_out) {
  if (PREC == kFP64 && jb.lc_edge) kitaev_logpi64_open<MULTI>(g, v, jb.L, jb.J, beta, wk, res, eps_out);
  else kitaev_logpi64<MULTI>(g, v, jb.L, jb.J, beta, wk, res, eps_out);
}

// AUX = 0: the proposal loop (mode 0) only; AUX = 1: modes 1-3.  Two kernels,
// so that the hot proposal loop carries none of the other modes' code and
// registers (with them it spilled).  MULTI (Kitaev, mode 0 only): CTAs hold
// several chain groups, which synchronise on named barriers of their own;
// without it every CTA holds one chain and uses the CTA barrier only.
template <int KIND, int PREC, int KC, int kC, int NT, int AUX, bool MULTI = false>
__global__ void __launch_bounds__(NT, CRBM_MIN_BLOCKS * 256 / NT) crbm_step_kernel(const __grid_constant__ LaunchParams prm) {
  int jid = 0;
  while (jid + 1 < prm.n_jobs && (int)blockIdx.x >= prm.tile_begin[jid + 1]) ++jid;
  const JobDev& jb = prm.job[jid];
  const int ltile = (int)blockIdx.x - prm.tile_begin[jid];
  const int tid = threadIdx.x;
  const int N = jb.N, nblk = (N + 3) >> 2, P = jb.P, K = jb.K, T = 1 << jb.k;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* sp = smem_raw;
  Tabs tb;
  tb.T = T;
  tb.f64 = tb.b64 = nullptr;
  tb.fd = tb.bd = tb.fh = tb.fl = nullptr;
  tb.fdi = tb.fhi = tb.fli = nullptr;
  if constexpr (PREC == kFP64) {
    // read through L1: the FP64 pipe, not the tables, paces the FP64 phases, and
    // an LCRBM's 36 KB of them per CTA left half of the chains waiting for an SM
    tb.f64 = jb.f64;
    tb.b64 = jb.b64;
  } else {
    sp = mixed_tables<KC>(jb, sp, tb, tid, NT);
  }
  ChainSm* cs = (ChainSm*)sp;
  sp += align16(jb.nc * sizeof(ChainSm));
  double* scratch = (double*)sp;
  sp += align16(64 * 8);
  unsigned char* kwork = sp;     // Kitaev: the work areas of the CTA's nc chains
  if (KIND == kKitaev) sp += (size_t)jb.nc * kitaev_work_bytes(N);
  uint32_t* planes = (uint32_t*)sp;

  Grp g;
  g.tpc = NT / jb.nc;
  g.gl = tid / g.tpc;
  g.r = tid - g.gl * g.tpc;
  g.c = ltile * jb.nc + g.gl;
  g.active = g.c < jb.n_chains;
  g.cid = (uint32_t)(jb.cid_base + (uint64_t)g.c);
  KitaevWork wk;
  double* eps_st = nullptr;     // Kitaev local sweeps: spectrum of the proposed lattice
  if (KIND == kKitaev) {
    unsigned char* kp = MULTI ? kwork + (size_t)g.gl * kitaev_work_bytes(N) : kwork;
    wk.A = (double*)kp;
    kp += align16((size_t)N * (N + 1) / 2 * 8);
    wk.d = (double*)kp;
    kp += align16((size_t)N * 8);
    wk.e = (double*)kp;
    kp += align16((size_t)N * 8);
    wk.uw = (double*)kp;
    kp += (size_t)N * 16;
    wk.sc = (double*)kp;
    kp += align16(64 * 8);
    wk.xs = (double*)kp;
    kp += align16((size_t)(N + 8) * 8);
    eps_st = (double*)kp;
  }
  uint32_t* my = planes + (size_t)g.gl * (2 + K) * P;
  // mixed: the chain's expanded rows (v, v', the hidden planes; see expand_rows)
  uint64_t* ex = PREC == kMixed ? (uint64_t*)((unsigned char*)planes + align16((size_t)jb.nc * (2 + K) * P * 4)) +
                                      (size_t)g.gl * (2 + K) * jb.L
                                : nullptr;
  ChainSm& ch = cs[g.gl];

  for (int i = tid; i < jb.nc * (2 + K) * P; i += NT) planes[i] = 0u;
  __syncthreads();
  if (g.r == 0) {
    // every slot, including the unused slots of a partial last tile, starts
    // from a defined state: the plane index `cur` addresses shared memory
    ch.F = ch.Fb = ch.lp = ch.E = 0.0;
    ch.lpb = ch.lppb = 0.0;
    for (int o = 0; o < kNobs; ++o) ch.ot[o] = ch.os[o] = 0.0;
    ch.beta = 1.0;
    ch.acc = 0ull;
    ch.rec = 0ull;
    ch.rec_mh = 0ull;
    ch.cur = 0;
    ch.flag_rec = 0;
    ch.flag_acc = 0;
  }
  if (g.active) {
    for (int w = g.r; w < jb.Wd; w += g.tpc) my[w] = jb.bits[(size_t)g.c * jb.Wd + w];
    if (g.r == 0) {
      ch.F = jb.F[g.c];
      ch.Fb = jb.Fb[g.c];
      ch.lpb = jb.Lb[g.c];
      ch.lp = jb.logpi[g.c];
      ch.E = jb.Ephys[g.c];
      for (int o = 0; o < kNobs; ++o) {
        ch.ot[o] = jb.obs_t[(size_t)g.c * kNobs + o];
        // sums continue in place: the same sequence of additions however a
        // run is split into launches or batched with other jobs
        ch.os[o] = jb.obs[(size_t)g.c * kNobs + o];
      }
      ch.beta = 1.0 / jb.T[g.c];
    }
  }
  __syncthreads();
  unsigned nrec = 0;
  if (PREC == kMixed) {
    expand_rows(my, P, ex, jb.L, 1, g.r, g.tpc);
    __syncthreads();
  }

  if (AUX && prm.mode == 1) {
    // evaluate F (FP64, or in the mixed path FP32 with its certified bound,
    // as after a mixed proposal), log pi and the observables (FP64) of the
    // current lattices
    FreeSum fs;
    if constexpr (PREC == kMixed) fs = free_phase<KC, kC>(jb, tb, g, my, ex, 0, nblk);
    else fs = free_phase64(jb, tb.f64, g, my);
    reduce_free<PREC, false>(fs, g, scratch);
    double kr[3] = {0.0, 0.0, 0.0};
    if (KIND == kKitaev)
      fp64_spectrum<PREC, MULTI>(jb, g, my, g.active ? ch.beta : 1.0, wk, kr, g.active ? jb.eps + (size_t)g.c * N : nullptr);
    if (g.active && g.r == 0) {
      const double F = free_value<PREC>(jb, fs);
      const double E = KIND == kIsing ? ising_energy(jb, fs.pairs) : kr[1];
      double ot[kNobs];
      observables<KIND>(jb, E, kr[2], fs.ones, fs.pairs, ot);
      jb.F[g.c] = F;
      jb.Fb[g.c] = PREC == kMixed ? free_bound(fs, free_constant(jb, g.tpc), F) : 0.0;
      jb.Lb[g.c] = 0.0;
      jb.logpi[g.c] = KIND == kIsing ? -ch.beta * E : kr[0];
      jb.Ephys[g.c] = E;
      for (int o = 0; o < kNobs; ++o) jb.obs_t[(size_t)g.c * kNobs + o] = ot[o];
    }
    return;
  }

  if (AUX && prm.mode == 2) {
    // tempering: the RBM chain makes g Gibbs steps without correction (Eq. B4),
    // then its new lattice y' and the physical chain x of the same slot (job
    // prm.job[1]) are exchanged with the Eq. (B5) probability for the pair
    // (pi, P_CRBM):  log a = [log pi(y') - log pi(x)] + [F(y') - F(x)].  In the
    // mixed path F(y') is the FP32 value with its certified bound and F(x) may
    // carry one too; a decision inside the bounds is redone with FP64 F.
    const JobDev& xj = prm.job[1];
    const uint32_t step = (uint32_t)*(volatile unsigned long long*)jb.step;
    const uint32_t cycle = (uint32_t)*(volatile unsigned long long*)xj.step;
    uint32_t* vp = my + P;
    uint32_t* h = my + 2 * P;
    gibbs_steps<PREC, KC, kC>(jb, tb, g, my, vp, h, ex, ex + jb.L, ex + 2 * jb.L, P, prm.g, step, nrec,
                              []() { __syncthreads(); });
    FreeSum fs;
    if constexpr (PREC == kMixed) fs = free_phase<KC, kC>(jb, tb, g, vp, ex + jb.L, 0, nblk);
    else fs = free_phase64(jb, tb.f64, g, vp);
    reduce_free<PREC, false>(fs, g, scratch);
    double kr[3] = {0.0, 0.0, 0.0};
    if (KIND == kKitaev)
      fp64_spectrum<PREC, MULTI>(jb, g, vp, g.active ? ch.beta : 1.0, wk, kr, g.active ? jb.eps + (size_t)g.c * N : nullptr);
    // the physical chain's lattice into the first hidden plane (free now)
    if (g.active)
      for (int w = g.r; w < jb.Wd; w += g.tpc) h[w] = xj.bits[(size_t)g.c * jb.Wd + w];
    if (g.active && g.r == 0) {
      ch.Fp = free_value<PREC>(jb, fs);
      ch.Bp = PREC == kMixed ? free_bound(fs, free_constant(jb, g.tpc), ch.Fp) : 0.0;
      ch.Ep = KIND == kIsing ? ising_energy(jb, fs.pairs) : kr[1];
      ch.lpp = KIND == kIsing ? -ch.beta * ch.Ep : kr[0];
      ch.cfp = kr[2];
      ch.onesp = fs.ones;
      ch.pairsp = fs.pairs;
      ch.F = xj.F[g.c];
      ch.Fb = xj.Fb[g.c];
      ch.lp = xj.logpi[g.c];
      const double loga = (ch.lpp - ch.lp) + (ch.Fp - ch.F);
      const uint4 w = philox4x32_10_rk(make_uint4(0u, kTagSwap, cycle, (uint32_t)(xj.cid_base + (uint64_t)g.c)),
                                       xj.rk);
      const double logu = log(((double)w.x + 0.5) * 0x1p-32);
      ch.flag_rec = 0;
      if (PREC == kFP64) {
        ch.flag_acc = logu < loga;
      } else {
        const double Mg = ch.Bp + ch.Fb + 1e-12 * (fabs(ch.lpp) + fabs(ch.lp) + fabs(ch.Fp) + fabs(ch.F)) + 1e-300;
        if (loga - logu > Mg) ch.flag_acc = 1;
        else if (logu - loga > Mg) ch.flag_acc = 0;
        else ch.flag_rec = 1;
      }
    }
    if (PREC == kMixed) {
      const int need = __syncthreads_or(g.active && g.r == 0 && ch.flag_rec);
      if (need) {
        // FP64 free energies of y' and (when only its FP32 value is known) of x
        Grp g2 = g;
        g2.active = g.active && ch.flag_rec;
        if constexpr (KIND == kIsing) {
          ising_redo64(jb, g, cs, 1, scratch, [&](int i) { return planes + (size_t)i * (2 + K) * P + (vp - my); },
                       [&](int i) { return planes + (size_t)i * (2 + K) * P + (h - my); });
        } else {
          FreeSum f1;
          free_energy64(jb, g2, vp, &f1);
          reduce_free<kFP64, false>(f1, g2, scratch);
          Grp g3 = g2;
          g3.active = g2.active && ch.Fb != 0.0;
          FreeSum f2;
          free_energy64(jb, g3, h, &f2);
          reduce_free<kFP64, false>(f2, g3, scratch);
          if (g2.active && g.r == 0) {
            ch.Fp = free_value<kFP64>(jb, f1);
            ch.Bp = 0.0;
            if (g3.active) {
              ch.F = free_value<kFP64>(jb, f2);
              ch.Fb = 0.0;
            }
          }
        }
        if (g2.active && g.r == 0) {
          const double loga = (ch.lpp - ch.lp) + (ch.Fp - ch.F);
          const uint4 w = philox4x32_10_rk(
              make_uint4(0u, kTagSwap, cycle, (uint32_t)(xj.cid_base + (uint64_t)g.c)), xj.rk);
          ch.flag_acc = log(((double)w.x + 0.5) * 0x1p-32) < loga;
          ch.rec_mh += 1ull;
        }
      }
    }
    if (nrec) atomicAdd(&ch.rec, (unsigned long long)nrec);
    __syncthreads();
    if (g.active) {
      const bool sw = ch.flag_acc != 0;
      const size_t c = (size_t)g.c;
      uint32_t* xb = xj.bits + c * jb.Wd;
      uint32_t* yb = jb.bits + c * jb.Wd;
      for (int w = g.r; w < jb.Wd; w += g.tpc) {
        if (sw) {
          xb[w] = vp[w];
          yb[w] = h[w];
        } else {
          yb[w] = vp[w];
        }
      }
      if (KIND == kKitaev && sw) {
        for (int l = g.r; l < N; l += g.tpc) {
          const double t = xj.eps[c * N + l];
          xj.eps[c * N + l] = jb.eps[c * N + l];
          jb.eps[c * N + l] = t;
        }
      }
      if (g.r == 0) {
        double otp[kNobs];
        observables<KIND>(jb, ch.Ep, ch.cfp, ch.onesp, ch.pairsp, otp);
        if (sw) {
          // the RBM slot takes x (read before the physical slot is overwritten)
          jb.F[c] = ch.F;
          jb.Fb[c] = ch.Fb;
          jb.Lb[c] = xj.Lb[c];
          jb.logpi[c] = ch.lp;
          jb.Ephys[c] = xj.Ephys[c];
          for (int o = 0; o < kNobs; ++o) jb.obs_t[c * kNobs + o] = xj.obs_t[c * kNobs + o];
          xj.F[c] = ch.Fp;
          xj.Fb[c] = ch.Bp;
          xj.Lb[c] = 0.0;
          xj.logpi[c] = ch.lpp;
          xj.Ephys[c] = ch.Ep;
          for (int o = 0; o < kNobs; ++o) xj.obs_t[c * kNobs + o] = otp[o];
          xj.acc[c] += 1ull;
        } else {
          jb.F[c] = ch.Fp;
          jb.Fb[c] = ch.Bp;
          jb.Lb[c] = 0.0;
          jb.logpi[c] = ch.lpp;
          jb.Ephys[c] = ch.Ep;
          for (int o = 0; o < kNobs; ++o) jb.obs_t[c * kNobs + o] = otp[o];
        }
        jb.rec[2 * c] += ch.rec;
        jb.rec[2 * c + 1] += ch.rec_mh;
      }
    }
    return;
  }

  if (AUX && KIND == kKitaev && prm.mode == 3) {
    // local-update Metropolis sweeps (Sec. IV baseline; the Ising kind's are crbm_sweep.cu's)
    const unsigned long long step0 = *(volatile unsigned long long*)jb.step;
    for (int s = 0; s < prm.S; ++s) {
      const uint32_t step = (uint32_t)(step0 + (uint64_t)s);
      // per chain group: every branch below is uniform in the group, and only
      // the group synchronises (a short last tile has groups without a chain)
      for (int n = 0; n < N; ++n) {
        const uint32_t* v = my + ch.cur * P;
        uint32_t* vp = my + (ch.cur ^ 1) * P;
        for (int w = g.r; w < jb.Wd; w += g.tpc) vp[w] = v[w] ^ ((w == (n >> 5)) ? (1u << (n & 31)) : 0u);
        grp_sync<MULTI>(g);
        double kr[4] = {0.0, 0.0, 0.0, 0.0};
        if (PREC == kMixed) {
          kitaev_logpi_df<MULTI>(g, vp, jb.L, jb.J, ch.beta, wk, kr);
        } else {
          double k3[3];
          fp64_spectrum<PREC, MULTI>(jb, g, vp, ch.beta, wk, k3, eps_st);
          kr[0] = k3[0];
          kr[1] = k3[1];
          kr[2] = k3[2];
        }
        if (g.r == 0) {
          const uint4 w = philox4x32_10_rk(make_uint4((uint32_t)(n >> 2), kTagLocal, step, g.cid), jb.rk);
          const double logu = log(((double)pick(w, n & 3) + 0.5) * 0x1p-32);
          const double logr = kr[0] - ch.lp;
          ch.lpp = kr[0];
          ch.lppb = kr[3];
          ch.Ep = kr[1];
          ch.cfp = kr[2];
          ch.flag_rec = 0;
          if (PREC == kFP64) {
            ch.flag_acc = logu < logr;
          } else {
            const double M = ch.lppb + ch.lpb + 1e-12 * (fabs(ch.lpp) + fabs(ch.lp)) + 1e-300;
            if (logr - logu > M) ch.flag_acc = 1;
            else if (logu - logr > M) ch.flag_acc = 0;
            else ch.flag_rec = 1;
          }
        }
        grp_sync<MULTI>(g);
        if (PREC == kMixed && ch.flag_rec) {
          // the FP64 eigen-stage of the proposal (and of the current lattice
          // when its log-weight came from the df64 stage)
          double k1v[3], k0v[3] = {0.0, 0.0, 0.0};
          const bool redo_v = ch.lpb != 0.0;
          fp64_spectrum<PREC, MULTI>(jb, g, vp, ch.beta, wk, k1v, eps_st);
          if (redo_v) fp64_spectrum<PREC, MULTI>(jb, g, v, ch.beta, wk, k0v, nullptr);
          if (g.r == 0) {
            ch.lpp = k1v[0];
            ch.lppb = 0.0;
            ch.Ep = k1v[1];
            ch.cfp = k1v[2];
            if (redo_v) {
              ch.lp = k0v[0];
              ch.lpb = 0.0;
            }
            const uint4 w = philox4x32_10_rk(make_uint4((uint32_t)(n >> 2), kTagLocal, step, g.cid), jb.rk);
            const double logu = log(((double)pick(w, n & 3) + 0.5) * 0x1p-32);
            ch.flag_acc = logu < ch.lpp - ch.lp;
            ch.rec_mh += 1ull;
          }
          grp_sync<MULTI>(g);
        }
        if (ch.flag_acc) {
          // the spectrum cache follows the lattice when the proposal's came from the FP64 stage
          if (g.active && (PREC == kFP64 || ch.flag_rec))
            for (int l = g.r; l < N; l += g.tpc) jb.eps[(size_t)g.c * N + l] = eps_st[l];
          grp_sync<MULTI>(g);
          if (g.r == 0) {
            ch.cur ^= 1;
            ch.lp = ch.lpp;
            ch.lpb = ch.lppb;
            ch.E = ch.Ep;
            ch.ot[0] = ch.Ep;
            ch.ot[1] = ch.Ep * ch.Ep;
            ch.ot[2] = ch.cfp;
            ch.acc += 1ull;
          }
        }
        grp_sync<MULTI>(g);
      }
      // observables of the lattice after the sweep
      double cn[1] = {flux_count(jb, g, my + ch.cur * P)};
      grp_reduce<1>(cn, g, scratch);
      if (g.active && g.r == 0) {
        ch.ot[3] = cn[0] / (double)jb.nhex;
        if (prm.correct) {
          for (int o = 0; o < kNobs; ++o) ch.os[o] += ch.ot[o];
          trace_store(jb, g.c, step0 + (uint64_t)s, ch.E);
        }
      }
      __syncthreads();
    }
    // FP64 free energy of the final lattices, then everything back to the job
    FreeSum fs;
    free_energy64(jb, g, my + ch.cur * P, &fs);
    reduce_free<kFP64, false>(fs, g, scratch);
    if (g.active) {
      const uint32_t* v = my + ch.cur * P;
      for (int w = g.r; w < jb.Wd; w += g.tpc) jb.bits[(size_t)g.c * jb.Wd + w] = v[w];
      if (g.r == 0) {
        jb.F[g.c] = free_value<kFP64>(jb, fs);
        jb.Fb[g.c] = 0.0;
        jb.Lb[g.c] = ch.lpb;
        jb.logpi[g.c] = ch.lp;
        jb.Ephys[g.c] = ch.E;
        for (int o = 0; o < kNobs; ++o) {
          jb.obs_t[(size_t)g.c * kNobs + o] = ch.ot[o];
          jb.obs[(size_t)g.c * kNobs + o] = ch.os[o];
        }
        jb.acc[g.c] += ch.acc;
        jb.rec[2 * (size_t)g.c + 1] += ch.rec_mh;
      }
    }
    return;
  }

  if (AUX) return;
  // The Kitaev kind's chain groups are warp-aligned and independent inside
  // the proposal loop: they synchronise and reduce on their own (a group whose
  // eigen-stage takes longer holds back no other chain of the CTA); the Ising
  // kind's groups may be smaller than a warp and use the CTA barrier.
  auto loop_sync = [&]() {
    if (KIND == kKitaev && MULTI) grp_sync<MULTI>(g);
    else __syncthreads();
  };
  auto loop_reduce = [&](FreeSum& x, const Grp& gg, auto prec) {
    reduce_free<decltype(prec)::value, KIND == kKitaev && MULTI>(x, gg, KIND == kKitaev && MULTI ? wk.sc : scratch);
  };
  // the step counter lives in device memory (advanced by advance_steps after
  // the launch), so a captured CUDA graph can be replayed
  const unsigned long long step0 = *(volatile unsigned long long*)jb.step;
  // What follows a decision (the accepted state's values, the running sums)
  // and the next proposal's log u are left to the group's last thread, which
  // takes them beside the hidden half-step: a single thread's FP64 instructions
  // hold their sub-partition's pipe as long as a full warp's, and the leader's
  // would hold up the whole group.
  const bool clerk = g.active && g.r == g.tpc - 1;
  auto settle = [&](unsigned long long t) {
    if (ch.flag_acc) {
      ch.F = ch.Fp;
      ch.Fb = ch.Bp;
      ch.lp = ch.lpp;
      ch.lpb = ch.lppb;
      ch.E = ch.Ep;
      observables<KIND>(jb, ch.Ep, ch.cfp, ch.onesp, ch.pairsp, ch.ot);
      ch.acc += 1ull;
    }
    for (int o = 0; o < kNobs; ++o) ch.os[o] += ch.ot[o];
    trace_store(jb, g.c, t, ch.E);
  };
  auto accept_word = [&](uint32_t step) {
    return philox4x32_10_rk(make_uint4(0u, kTagAcc, step, g.cid), jb.rk).x;
  };
  auto log_u64 = [&](uint32_t step) { return log(((double)accept_word(step) + 0.5) * 0x1p-32); };
  if (PREC == kMixed && g.active && g.r == 0) ch.cst = free_constant(jb, g.tpc);
  for (int s = 0; s < prm.S; ++s) {
    const uint32_t step = (uint32_t)(step0 + (uint64_t)s);
    const int cur = ch.cur;
    uint32_t* v = my + cur * P;
    uint32_t* vp = my + (cur ^ 1) * P;
    uint32_t* h = my + 2 * P;
    if (clerk) {
      if (s > 0) settle(step0 + (uint64_t)(s - 1));
      // mixed: in FP32, within 2^-20 (1 + |log u|), a term of the decision's margin
      if (prm.correct) ch.logu = PREC == kFP64 ? log_u64(step) : (double)log_u32(accept_word(step));
    }
    gibbs_steps<PREC, KC, kC>(jb, tb, g, v, vp, h, ex + cur * jb.L, ex + (cur ^ 1) * jb.L, ex + 2 * jb.L, P, prm.g, step,
                              nrec, loop_sync);
    FreeSum fs;
    if constexpr (PREC == kMixed) fs = free_phase<KC, kC>(jb, tb, g, vp, ex + (cur ^ 1) * jb.L, 0, nblk);
    else fs = free_phase64(jb, tb.f64, g, vp);
    loop_reduce(fs, g, std::integral_constant<int, PREC>());
    double kr[4] = {0.0, 0.0, 0.0, 0.0};
    if (KIND == kKitaev) {
      if (PREC == kMixed) {
        kitaev_logpi_df<MULTI>(g, vp, jb.L, jb.J, g.active ? ch.beta : 1.0, wk, kr);
      } else {
        double k3[3];
        fp64_spectrum<PREC, MULTI>(jb, g, vp, g.active ? ch.beta : 1.0, wk, k3, nullptr);
        kr[0] = k3[0];
        kr[1] = k3[1];
        kr[2] = k3[2];
      }
    }
    if (g.active && g.r == 0) {
      const double E = KIND == kIsing ? ising_energy(jb, fs.pairs) : kr[1];
      const double lpp = KIND == kIsing ? -ch.beta * E : kr[0];
      const double Fp = free_value<PREC>(jb, fs);
      ch.Ep = E;
      ch.lpp = lpp;
      ch.cfp = kr[2];
      ch.onesp = fs.ones;
      ch.pairsp = fs.pairs;
      ch.lppb = kr[3];
      ch.Fp = Fp;
      ch.Bp = PREC == kMixed ? free_bound(fs, ch.cst, Fp) : 0.0;
      ch.flag_rec = 0;
      if (!prm.correct) {
        ch.flag_acc = 1;
      } else {
        const double logu = ch.logu, logr = (lpp - ch.lp) + (Fp - ch.F);
        if (PREC == kFP64) {
          ch.flag_acc = logu < logr;
        } else {
          const double M = ch.Bp + ch.Fb + ch.lppb + ch.lpb +
                           1e-12 * (fabs(lpp) + fabs(ch.lp) + fabs(Fp) + fabs(ch.F)) +
                           0x1p-20 * (1.0 + fabs(logu)) + 1e-300;
          if (logr - logu > M) ch.flag_acc = 1;
          else if (logu - logr > M) ch.flag_acc = 0;
          else ch.flag_rec = 1;
        }
      }
      if (!ch.flag_rec && ch.flag_acc) ch.cur ^= 1;
    }
    int need = 0;
    if (PREC == kMixed && !(KIND == kKitaev && MULTI)) {
      need = __syncthreads_or(g.active && g.r == 0 && ch.flag_rec);
    } else {
      loop_sync();                 // the leader's decision, read by its whole group
      if (PREC == kMixed) need = g.active && ch.flag_rec;
    }
    if (PREC == kMixed && need) {
      // the chains (several per CTA: some of them) whose margin straddled the threshold
      Grp g2 = g;
      g2.active = g.active && ch.flag_rec != 0;
      loop_sync();
      const bool mine = g2.active && g.r == 0;
      if (KIND == kIsing) {
        // second level: F of v' (and of v when only an FP32 value of it is
        // known) with df64 softplus (bound ~1e-7); flag_rec = 2 sends a decision
        // that still straddles the threshold on to the FP64 path's code below
        Grp g3 = g2;
        g3.active = g2.active && ch.Fb != 0.0;
        double f1[3], f2[3];
        free_sum_df<KC ? KC : kMaxK>(jb, g2, vp, 0, N, f1);
        grp_reduce<3>(f1, g2, scratch);
        free_sum_df<KC ? KC : kMaxK>(jb, g3, v, 0, N, f2);
        grp_reduce<3>(f2, g3, scratch);
        if (mine) {
          ch.Fp = -jb.vb * f1[2] - f1[0];
          ch.Bp = f1[1] + 1e-15 * fabs(ch.Fp);
          if (g3.active) {
            ch.F = -jb.vb * f2[2] - f2[0];
            ch.Fb = f2[1] + 1e-15 * fabs(ch.F);
          }
          const double logr = (ch.lpp - ch.lp) + (ch.Fp - ch.F);
          const double lu = log_u64(step);
          const double Mg = ch.Bp + ch.Fb + 1e-12 * (fabs(ch.lpp) + fabs(ch.lp) + fabs(ch.Fp) + fabs(ch.F)) + 1e-300;
          if (logr - lu > Mg) ch.flag_acc = 1;
          else if (lu - logr > Mg) ch.flag_acc = 0;
          else ch.flag_rec = 2;
          ch.rec_mh += 1ull;
        }
        need = __syncthreads_or(mine && ch.flag_rec == 2);
      }
      if (need) {
        // the FP64 path's free energies of v' (and of v when only its FP32
        // value is known), computed by the same code and reduction order
        // (tables from global memory: the mixed kernel keeps only FP32 ones)
        if constexpr (KIND == kIsing) {
          ising_redo64(jb, g, cs, 2, scratch,
                       [&](int i) { return planes + (size_t)i * (2 + K) * P + (cs[i].cur ^ 1) * P; },
                       [&](int i) { return planes + (size_t)i * (2 + K) * P + cs[i].cur * P; });
        } else {
          FreeSum f1;
          free_energy64(jb, g2, vp, &f1);
          loop_reduce(f1, g2, std::integral_constant<int, kFP64>());
          Grp g3 = g2;
          g3.active = g2.active && ch.Fb != 0.0;
          FreeSum f2;
          free_energy64(jb, g3, v, &f2);
          loop_reduce(f2, g3, std::integral_constant<int, kFP64>());
          // the FP64 eigen-stage of v' (and of v when its log-weight came from
          // the df64 stage), by the group that needs it
          double k1v[3] = {0.0, 0.0, 0.0}, k0v[3] = {0.0, 0.0, 0.0};
          const bool redo_v = ch.lpb != 0.0;
          fp64_spectrum<PREC, MULTI>(jb, g, vp, ch.beta, wk, k1v, nullptr);
          if (redo_v) fp64_spectrum<PREC, MULTI>(jb, g, v, ch.beta, wk, k0v, nullptr);
          if (mine) {
            ch.Fp = free_value<kFP64>(jb, f1);
            ch.Bp = 0.0;
            if (g3.active) {
              ch.F = free_value<kFP64>(jb, f2);
              ch.Fb = 0.0;
            }
            ch.lpp = k1v[0];
            ch.lppb = 0.0;
            ch.Ep = k1v[1];
            ch.cfp = k1v[2];
            if (redo_v) {
              ch.lp = k0v[0];
              ch.lpb = 0.0;
            }
            ch.rec_mh += 1ull;      // Ising: counted at the df64 level
          }
        }
        if (mine && (KIND == kKitaev || ch.flag_rec == 2))
          ch.flag_acc = log_u64(step) < (ch.lpp - ch.lp) + (ch.Fp - ch.F);
      }
      if (mine && ch.flag_acc) ch.cur ^= 1;
      loop_sync();
    }
  }
  if (clerk && prm.S > 0) settle(step0 + (uint64_t)(prm.S - 1));

  if (nrec) atomicAdd(&ch.rec, (unsigned long long)nrec);
  __syncthreads();
  if (g.active) {
    const uint32_t* v = my + ch.cur * P;
    for (int w = g.r; w < jb.Wd; w += g.tpc) jb.bits[(size_t)g.c * jb.Wd + w] = v[w];
    if (g.r == 0) {
      jb.F[g.c] = ch.F;
      jb.Fb[g.c] = ch.Fb;
      jb.Lb[g.c] = ch.lpb;
      jb.logpi[g.c] = ch.lp;
      jb.Ephys[g.c] = ch.E;
      for (int o = 0; o < kNobs; ++o) {
        jb.obs_t[(size_t)g.c * kNobs + o] = ch.ot[o];
        jb.obs[(size_t)g.c * kNobs + o] = ch.os[o];
      }
      jb.acc[g.c] += ch.acc;
      jb.rec[2 * (size_t)g.c] += ch.rec;
      jb.rec[2 * (size_t)g.c + 1] += ch.rec_mh;
    }
  }
}


// After a launch of S proposals: every job's device step counter += S.
static __global__ void advance_steps_kernel(const __grid_constant__ LaunchParams p) {
  const int i = threadIdx.x;
  if (i < p.n_jobs) *p.job[i].step += (unsigned long long)p.S;
}

// Launch one instantiation; raise its dynamic shared-memory limit.  MULTI
// launches run mode 0 only.
template <int KIND, int PREC, int KC, int kC, int NT, bool MULTI = false>
cudaError_t launch_inst(const LaunchParams& p, int grid, size_t smem, cudaStream_t st) {
  if constexpr (MULTI) {
    crbm_step_kernel<KIND, PREC, KC, kC, NT, 0, true><<<grid, NT, smem, st>>>(p);
  } else {
    if (p.mode == 0) crbm_step_kernel<KIND, PREC, KC, kC, NT, 0><<<grid, NT, smem, st>>>(p);
    else crbm_step_kernel<KIND, PREC, KC, kC, NT, 1><<<grid, NT, smem, st>>>(p);
  }
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && p.mode != 1 && p.S > 0) {
    advance_steps_kernel<<<1, kMaxJobs, 0, st>>>(p);
    e = cudaGetLastError();
  }
  return e;
}

template <int KIND, int PREC, int KC, int kC, int NT>
cudaError_t limit_inst(size_t bytes) {
  cudaError_t e = cudaFuncSetAttribute(crbm_step_kernel<KIND, PREC, KC, kC, NT, 0>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(crbm_step_kernel<KIND, PREC, KC, kC, NT, 1>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  return e;
}

template <int KIND, int PREC, int NT>
cudaError_t launch_nt(int KC, int kC, const LaunchParams& p, int grid, size_t smem, cudaStream_t st) {
  if constexpr (PREC == kMixed) {
    if (KC == 4 && kC == 5) return launch_inst<KIND, PREC, 4, 5, NT>(p, grid, smem, st);
    if (KC == 4 && kC == 3) return launch_inst<KIND, PREC, 4, 3, NT>(p, grid, smem, st);
    if constexpr (KIND == kIsing) {
      if (KC == 2 && kC == 5) return launch_inst<KIND, PREC, 2, 5, NT>(p, grid, smem, st);
      if (KC == 2 && kC == 3) return launch_inst<KIND, PREC, 2, 3, NT>(p, grid, smem, st);
    }
  }
  return launch_inst<KIND, PREC, 0, 0, NT>(p, grid, smem, st);
}

template <int KIND, int PREC, int NT>
cudaError_t limit_nt(size_t bytes) {
  cudaError_t e = limit_inst<KIND, PREC, 0, 0, NT>(bytes);
  if constexpr (PREC == kMixed) {
    if (e == cudaSuccess) e = limit_inst<KIND, PREC, 4, 5, NT>(bytes);
    if (e == cudaSuccess) e = limit_inst<KIND, PREC, 4, 3, NT>(bytes);
    if constexpr (KIND == kIsing) {
      if (e == cudaSuccess) e = limit_inst<KIND, PREC, 2, 5, NT>(bytes);
      if (e == cudaSuccess) e = limit_inst<KIND, PREC, 2, 3, NT>(bytes);
    }
  }
  return e;
}

// The several-chains-per-CTA proposal kernel (mixed-size Kitaev batches).
template <int KIND, int PREC, int NT>
cudaError_t launch_multi(int KC, int kC, const LaunchParams& p, int grid, size_t smem, cudaStream_t st) {
  if constexpr (PREC == kMixed) {
    if (KC == 4 && kC == 5) return launch_inst<KIND, PREC, 4, 5, NT, true>(p, grid, smem, st);
    if (KC == 4 && kC == 3) return launch_inst<KIND, PREC, 4, 3, NT, true>(p, grid, smem, st);
  }
  return launch_inst<KIND, PREC, 0, 0, NT, true>(p, grid, smem, st);
}

template <int KIND, int PREC, int NT>
cudaError_t limit_multi(size_t bytes) {
  auto limit = [&](auto f) {
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
  cudaError_t e = limit(crbm_step_kernel<KIND, PREC, 0, 0, NT, 0, true>);
  if constexpr (PREC == kMixed) {
    if (e == cudaSuccess) e = limit(crbm_step_kernel<KIND, PREC, 4, 5, NT, 0, true>);
    if (e == cudaSuccess) e = limit(crbm_step_kernel<KIND, PREC, 4, 3, NT, 0, true>);
  }
  return e;
}

// One translation unit per (kind, precision, CTA size) instantiates the
// (K, k) variants (mixed: (4, 5), (4, 3) and runtime; FP64, whose phases wait
// on the FP64 pipe and not on their integer work: runtime alone): CTAs of 256 threads, plus 128,
// 64 and 32 threads for the Kitaev kind (small matrices); every CTA size gets
// the same 128-register budget.  Separate units compile in parallel.
#define CRBM_VARIANTS_NT(KIND, PREC, NT)                                                       \
  cudaError_t launch_##KIND##_##PREC##_##NT(int KC, int kC, const LaunchParams& p, int grid,   \
                                            size_t smem, cudaStream_t st) {                    \
    return launch_nt<KIND, PREC, NT>(KC, kC, p, grid, smem, st);                               \
  }                                                                                            \
  cudaError_t limit_##KIND##_##PREC##_##NT(size_t bytes) { return limit_nt<KIND, PREC, NT>(bytes); }

#define CRBM_VARIANTS_MULTI(KIND, PREC, NT)                                                    \
  cudaError_t launch_##KIND##_##PREC##_##NT##_multi(int KC, int kC, const LaunchParams& p, int grid, \
                                                    size_t smem, cudaStream_t st) {            \
    return launch_multi<KIND, PREC, NT>(KC, kC, p, grid, smem, st);                            \
  }                                                                                            \
  cudaError_t limit_##KIND##_##PREC##_##NT##_multi(size_t bytes) { return limit_multi<KIND, PREC, NT>(bytes); }

}  // namespace crbm
