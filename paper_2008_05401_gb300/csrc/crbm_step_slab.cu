// The table kernel's Ising proposals with a chain divided over a cluster of
// CTAs: mixed precision, lattice sides of whole words (L a multiple of 32),
// mode 0.  For launches whose chains are fewer than the SMs (a served request at
// a side the tensor-core form does not have): one CTA per chain would leave
// most SMs idle, and a chain's proposals are sequential.
//
// CTA `rank` of a chain's cluster owns rows L rank / CL .. L (rank + 1) / CL - 1
// (CL of 1 to 8, whatever the SMs of the GPCs hold side by side): their units'
// draws, decisions and sums are its own, with the table kernel's phases.  Every
// CTA has room for the whole packed lattices (8 KB a plane at L = 256), of which
// it keeps its rows and the neighbours' it reads: the k - 1 rows after them of v
// and v' (Eqs. B2, 13), the k - 1 rows before them of the hidden planes (Eq.
// B3), copied over distributed shared memory after the cluster barrier that ends
// the phase writing them.  The CTAs' sums are added in rank order by every CTA,
// so each takes the same decision and keeps the chain's values itself.
// Three cluster barriers per proposal of one Gibbs step; the rest is bound by
// instruction issue like the table kernel (59 % of the slots).  16 chains of
// L = 256, K = 4 5x5, 40 proposals and the read-back, in clusters of six: 1.74 ms
// (one CTA per chain: 12.5 ms).
#include <algorithm>

#include <cooperative_groups.h>

#include "crbm_step.cuh"

namespace crbm {

namespace {

namespace cg = cooperative_groups;

constexpr int kSlabThreads = 512;      // 16 warps at 128 registers: one CTA per SM
constexpr int kMaxSlabs = 8;           // the portable cluster size

// What a CTA contributes to a decision.
struct SlabSum {
  double d[3];         // second level: free_sum_df's sums; FP64: d[0]
  long long fx;        // first level: FreeSum
  float b;
  int ones, pairs;
};

// Sums over the cluster of the CTAs' contributions (valid in `mine` of thread
// 0), returned to the lanes of warp 0.  slots: two per CTA, taken in turn, so
// that a slot is written again only after a later barrier of the cluster.
__device__ __forceinline__ SlabSum cluster_sum(cg::cluster_group& cl, SlabSum mine, SlabSum* slots, int& turn) {
  SlabSum* slot = slots + turn;
  turn ^= 1;
  if (threadIdx.x == 0) *slot = mine;
  cl.sync();
  SlabSum x = {{0.0, 0.0, 0.0}, 0ll, 0.0f, 0, 0};
  if (threadIdx.x < 32) {
    if (threadIdx.x < cl.num_blocks()) x = *cl.map_shared_rank(slot, (int)threadIdx.x);
    for (int o = 1; o < kMaxSlabs; o <<= 1) {
      for (int i = 0; i < 3; ++i) x.d[i] += __shfl_xor_sync(kFull, x.d[i], o);
      x.fx += __shfl_xor_sync(kFull, x.fx, o);
      x.b += __shfl_xor_sync(kFull, x.b, o);
      x.ones += __shfl_xor_sync(kFull, x.ones, o);
      x.pairs += __shfl_xor_sync(kFull, x.pairs, o);
    }
  }
  return x;
}

// F of a lattice whose rows the cluster's CTAs hold, as the FP64 path has it, by
// every CTA on its own copy (out of line: rare).
__device__ __noinline__ double whole_free64(const JobDev& jb, const Grp& g, uint32_t* lattice, double* scratch) {
  cg::cluster_group cl = cg::this_cluster();
  const int CL = (int)cl.num_blocks(), rank = (int)cl.block_rank(), WL = jb.L >> 5;
  for (int w = threadIdx.x; w < jb.Wd; w += kSlabThreads) {
    const int owner = ((w / WL + 1) * CL - 1) / jb.L;
    if (owner != rank) lattice[w] = cl.map_shared_rank(lattice, owner)[w];
  }
  __syncthreads();
  return path64_free(jb, g, lattice, scratch);
}

template <int KC, int kC>
__global__ void __launch_bounds__(kSlabThreads, 1) slab_kernel(const __grid_constant__ LaunchParams prm) {
  cg::cluster_group cl = cg::this_cluster();
  const int CL = (int)cl.num_blocks(), rank = (int)cl.block_rank(), chain = (int)blockIdx.x / CL;
  int jid = 0;
  while (jid + 1 < prm.n_jobs && chain >= prm.tile_begin[jid + 1]) ++jid;
  const JobDev& jb = prm.job[jid];
  const int tid = threadIdx.x, L = jb.L, P = jb.P, K = jb.K, WL = L >> 5, Wd = jb.Wd;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ SlabSum slots[2];
  __shared__ ChainSm ch;
  __shared__ double scratch[64];
  Tabs tb;
  tb.T = 1 << jb.k;
  tb.f64 = tb.b64 = nullptr;
  tb.fd = tb.bd = tb.fh = tb.fl = nullptr;
  tb.fdi = tb.fhi = tb.fli = nullptr;
  uint32_t* my = (uint32_t*)mixed_tables<KC>(jb, smem_raw, tb, tid, kSlabThreads);

  Grp g;
  g.c = chain - prm.tile_begin[jid];
  g.gl = 0;
  g.r = tid;
  g.tpc = kSlabThreads;
  g.active = true;
  g.cid = (uint32_t)(jb.cid_base + (uint64_t)g.c);
  const int r0 = L * rank / CL, r1 = L * (rank + 1) / CL;       // this CTA's rows r0 .. r1 - 1
  const int q0 = r0 * (L >> 2), q1 = r1 * (L >> 2);             // their units, sites
  const int n0 = 4 * q0, n1 = 4 * q1;
  const int halo = max(1, (kC ? kC : jb.k) - 1);               // at most any CTA's rows (slab_most)
  const int next = rank + 1 == CL ? 0 : rank + 1, prev = rank == 0 ? CL - 1 : rank - 1;
  // `halo` rows from row r (mod L) of `planes` planes, from CTA `from`'s copies
  auto pull = [&](uint32_t* plane, int planes, int r, int from) {
    if (CL == 1) return;
    const uint32_t* theirs = cl.map_shared_rank(plane, from);
    const int n = halo * WL, w0 = (r < 0 ? r + L : (r >= L ? r - L : r)) * WL;
    for (int e = tid; e < planes * n; e += kSlabThreads) {
      const int f = e / n, w = w0 + e - f * n, at = f * P + (w >= Wd ? w - Wd : w);
      plane[at] = theirs[at];
    }
  };

  for (int i = tid; i < (2 + K) * P; i += kSlabThreads) my[i] = i < Wd ? jb.bits[(size_t)g.c * Wd + i] : 0u;
  if (tid == 0) {
    ch.F = jb.F[g.c];
    ch.Fb = jb.Fb[g.c];
    ch.lpb = jb.Lb[g.c];
    ch.lppb = 0.0;
    ch.lp = jb.logpi[g.c];
    ch.E = jb.Ephys[g.c];
    for (int o = 0; o < kNobs; ++o) {
      ch.ot[o] = jb.obs_t[(size_t)g.c * kNobs + o];
      ch.os[o] = jb.obs[(size_t)g.c * kNobs + o];
    }
    ch.beta = 1.0 / jb.T[g.c];
    ch.acc = ch.rec = ch.rec_mh = 0ull;
    ch.cur = ch.flag_rec = ch.flag_acc = 0;
    ch.cst = free_constant(jb, kSlabThreads * CL);
  }
  const unsigned long long step0 = *(volatile unsigned long long*)jb.step;
  unsigned nrec = 0;
  int turn = 0;
  cl.sync();

  // the clerk's work beside the hidden half-step, as in the table kernel
  const bool clerk = tid == kSlabThreads - 1;
  auto settle = [&](unsigned long long t) {
    if (ch.flag_acc) {
      ch.F = ch.Fp;
      ch.Fb = ch.Bp;
      ch.lp = ch.lpp;
      ch.E = ch.Ep;
      observables<kIsing>(jb, ch.Ep, 0.0, ch.onesp, ch.pairsp, ch.ot);
      ch.acc += 1ull;
    }
    for (int o = 0; o < kNobs; ++o) ch.os[o] += ch.ot[o];
    if (rank == 0) trace_store(jb, g.c, t, ch.E);
  };
  auto accept_word = [&](uint32_t step) {
    return philox4x32_10_rk(make_uint4(0u, kTagAcc, step, g.cid), jb.rk).x;
  };
  auto log_u64 = [&](uint32_t step) { return log(((double)accept_word(step) + 0.5) * 0x1p-32); };
  for (int s = 0; s < prm.S; ++s) {
    const uint32_t step = (uint32_t)(step0 + (uint64_t)s);
    const int cur = ch.cur;
    uint32_t* v = my + cur * P;
    uint32_t* vp = my + (cur ^ 1) * P;
    uint32_t* h = my + 2 * P;
    const uint32_t* src = v;
    if (clerk) {
      if (s > 0) settle(step0 + (uint64_t)(s - 1));
      if (prm.correct) ch.logu = (double)log_u32(accept_word(step));
    }
    for (int sub = 0; sub < prm.g; ++sub) {
      hidden_phase<KC, kC>(jb, tb, g, src, nullptr, h, P, step, sub, nrec, q0, q1);
      cl.sync();
      pull(h, K, r0 - halo, prev);
      __syncthreads();
      visible_phase<KC, kC>(jb, tb, g, h, nullptr, vp, P, step, sub, nrec, q0, q1);
      cl.sync();
      pull(vp, 1, r1, next);
      __syncthreads();
      src = vp;
    }
    FreeSum fs = free_phase<KC, kC>(jb, tb, g, vp, nullptr, q0, q1);
    reduce_free<kMixed, false>(fs, g, scratch);
    const SlabSum all = cluster_sum(cl, {{0.0, 0.0, 0.0}, fs.fx, fs.b, fs.ones, fs.pairs}, slots, turn);
    if (tid == 0) {
      fs.fx = all.fx;
      fs.b = all.b;
      fs.ones = all.ones;
      fs.pairs = all.pairs;
      const double E = ising_energy(jb, fs.pairs), lpp = -ch.beta * E, Fp = free_value<kMixed>(jb, fs);
      ch.Ep = E;
      ch.lpp = lpp;
      ch.onesp = fs.ones;
      ch.pairsp = fs.pairs;
      ch.Fp = Fp;
      ch.Bp = free_bound(fs, ch.cst, Fp);
      ch.flag_rec = 0;
      if (!prm.correct) {
        ch.flag_acc = 1;
      } else {
        const double logu = ch.logu, logr = (lpp - ch.lp) + (Fp - ch.F);
        const double M = ch.Bp + ch.Fb + 1e-12 * (fabs(lpp) + fabs(ch.lp) + fabs(Fp) + fabs(ch.F)) +
                         0x1p-20 * (1.0 + fabs(logu)) + 1e-300;
        if (logr - logu > M) ch.flag_acc = 1;
        else if (logu - logr > M) ch.flag_acc = 0;
        else ch.flag_rec = 1;
      }
      if (!ch.flag_rec && ch.flag_acc) ch.cur ^= 1;
    }
    // every CTA holds the same values, so the cluster takes these branches together
    if (__syncthreads_or(tid == 0 && ch.flag_rec)) {
      // df64 softplus: the CTAs' rows, summed over the cluster; FP64: the whole
      // lattice in every CTA, by the FP64 path's threads in its order, so that the
      // decision is that path's to the last bit (rare)
      auto level = [&](bool df64, uint32_t* lattice) {
        SlabSum mine = {{0.0, 0.0, 0.0}, 0ll, 0.0f, 0, 0};
        if (df64) {
          free_sum_df<KC ? KC : kMaxK>(jb, g, lattice, n0, n1, mine.d);
          grp_reduce<3>(mine.d, g, scratch);
          return cluster_sum(cl, mine, slots, turn);
        }
        mine.d[0] = -whole_free64(jb, g, lattice, scratch);      // F = -v_bias d[2] - d[0]
        return mine;
      };
      const bool redo_v = ch.Fb != 0.0;
      // second level: df64 softplus; then, inside its bound too, the FP64 path's own
      for (int lev = 0; lev < 2; ++lev) {
        const SlabSum f1 = level(lev == 0, vp);
        SlabSum f2 = f1;
        if (redo_v) f2 = level(lev == 0, v);
        if (tid == 0) {
          ch.Fp = -jb.vb * f1.d[2] - f1.d[0];
          ch.Bp = lev == 0 ? f1.d[1] + 1e-15 * fabs(ch.Fp) : 0.0;
          if (redo_v) {
            ch.F = -jb.vb * f2.d[2] - f2.d[0];
            ch.Fb = lev == 0 ? f2.d[1] + 1e-15 * fabs(ch.F) : 0.0;
          }
          const double logr = (ch.lpp - ch.lp) + (ch.Fp - ch.F), lu = log_u64(step);
          const double Mg =
              lev == 0 ? ch.Bp + ch.Fb + 1e-12 * (fabs(ch.lpp) + fabs(ch.lp) + fabs(ch.Fp) + fabs(ch.F)) + 1e-300 : 0.0;
          ch.flag_acc = lu < logr;
          ch.flag_rec = lev == 0 && !(fabs(logr - lu) > Mg);
          if (lev == 0) ch.rec_mh += 1ull;
          if (!ch.flag_rec && ch.flag_acc) ch.cur ^= 1;
        }
        if (!__syncthreads_or(tid == 0 && ch.flag_rec)) break;
      }
    }
  }
  if (clerk && prm.S > 0) settle(step0 + (uint64_t)(prm.S - 1));
  if (nrec) atomicAdd(&ch.rec, (unsigned long long)nrec);
  __syncthreads();
  const uint32_t* v = my + ch.cur * P;
  for (int w = r0 * WL + tid; w < r1 * WL; w += kSlabThreads) jb.bits[(size_t)g.c * Wd + w] = v[w];
  if (tid == 0) {
    if (ch.rec) atomicAdd(&jb.rec[2 * (size_t)g.c], ch.rec);
    if (rank == 0) {
      jb.F[g.c] = ch.F;
      jb.Fb[g.c] = ch.Fb;
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
  cl.sync();        // no CTA leaves while another may read its shared memory
}

// Launch (or, with `fit`, count the clusters that run side by side) of one instantiation.
template <int KC, int kC>
cudaError_t launch_inst(const LaunchParams* p, int chains, int CL, size_t smem, cudaStream_t st, int* fit) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(chains * CL));
  cfg.blockDim = dim3(kSlabThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)CL;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (fit) return cudaOccupancyMaxActiveClusters(fit, slab_kernel<KC, kC>, &cfg);
  return cudaLaunchKernelEx(&cfg, slab_kernel<KC, kC>, *p);
}

cudaError_t launch_any(int K, int k, const LaunchParams* p, int chains, int CL, size_t smem, cudaStream_t st, int* fit) {
  int KC, kC;
  specialisation(kIsing, K, k, KC, kC);
  if (KC == 4 && kC == 5) return launch_inst<4, 5>(p, chains, CL, smem, st, fit);
  if (KC == 4 && kC == 3) return launch_inst<4, 3>(p, chains, CL, smem, st, fit);
  if (KC == 2 && kC == 5) return launch_inst<2, 5>(p, chains, CL, smem, st, fit);
  if (KC == 2 && kC == 3) return launch_inst<2, 3>(p, chains, CL, smem, st, fit);
  return launch_inst<0, 0>(p, chains, CL, smem, st, fit);
}

template <int KC, int kC>
cudaError_t limit_inst(size_t bytes) {
  // the static arrays (chain values, scratch, slots) come out of the same limit
  return cudaFuncSetAttribute(slab_kernel<KC, kC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes - 2048);
}

}  // namespace

size_t slab_smem_bytes(int L, int K, int k) {
  int KC, kC;
  specialisation(kIsing, K, k, KC, kC);
  const size_t P = (size_t)L * L / 32 + 1, nlut = (size_t)K * k << k, nq = (size_t)k << k;
  return (KC != 0 ? 3 * align16(nq * 16 * 8) + align16(nlut * 4) : 4 * align16(nlut * 4)) + (2 + (size_t)K) * P * 4;
}

int slab_most(int L, int K, int k, size_t smem_limit) {
  if (L % 32 != 0 || slab_smem_bytes(L, K, k) + 2048 > smem_limit) return 0;
  return std::min(kMaxSlabs, L / std::max(1, k - 1));
}

cudaError_t slab_fit(int K, int k, int CL, size_t smem, int* clusters) {
  return launch_any(K, k, nullptr, 1, CL, smem, nullptr, clusters);
}

cudaError_t launch_slab(const LaunchParams& p, int chains, int CL, size_t smem, cudaStream_t st) {
  cudaError_t e = launch_any(p.job[0].K, p.job[0].k, &p, chains, CL, smem, st, nullptr);
  if (e == cudaSuccess) {
    advance_steps_kernel<<<1, kMaxJobs, 0, st>>>(p);
    e = cudaGetLastError();
  }
  return e;
}

cudaError_t slab_set_smem_limit(size_t bytes) {
  cudaError_t e = limit_inst<4, 5>(bytes);
  if (e == cudaSuccess) e = limit_inst<4, 3>(bytes);
  if (e == cudaSuccess) e = limit_inst<2, 5>(bytes);
  if (e == cudaSuccess) e = limit_inst<2, 3>(bytes);
  if (e == cudaSuccess) e = limit_inst<0, 0>(bytes);
  return e;
}

}  // namespace crbm
