// FP64 eigen-stage of the open-boundary Kitaev model (the LCRBM's lattices:
// open along j, the y-bonds from column L-1 to column 0 absent).
//
// The open edges carry modes in pairs far closer than FP32 separates.  The
// Newton iteration here may settle both of a pair on one root (a step that
// approaches it from the left ends there), which root depends on the last bits
// of the tridiagonal, and log pi and e are then off by up to 1e-5 of their size
// in single lattices.  Chains are continued and compared by these values, so
// the arithmetic of this stage -- its operations, their order, the sums over the
// group -- is kept to the bit; kitaev_logpi64 (periodic lattices), whose
// eigenvalues are certified, has no such error and would take less time (four
// proposals of 1024 chains of L = 8: 4.7 ms instead of 8.3), but gives other
// values on these lattices: the right ones.
#pragma once
#include "crbm_device.cuh"

namespace crbm {

struct OpenWork {
  double *A, *d, *e, *vv, *pw, *sc;
  float *d32, *e32;
};

// Deterministic sum over a chain's (warp-aligned) group, returned to every
// thread of it: a butterfly within each warp, then the warps' partials added
// in warp order -- the order of block_sum for a CTA of tpc threads, so a group
// gives the same bits as a CTA of its size.  scratch: 32 doubles of the group.
template <bool MULTI>
__device__ __forceinline__ double grp_sum(double x, const Grp& g, double* scratch) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) x += __shfl_xor_sync(kFull, x, o);
  const int r = MULTI ? g.r : (int)threadIdx.x, tpc = MULTI ? g.tpc : (int)blockDim.x;
  const int warp = r >> 5, nw = tpc >> 5;
  grp_sync<MULTI>(g);
  if ((r & 31) == 0) scratch[warp] = x;
  grp_sync<MULTI>(g);
  double s = 0.0;
  for (int w = 0; w < nw; ++w) s += scratch[w];
  grp_sync<MULTI>(g);
  return s;
}

// FP32 Sturm count (same recurrence, rescaled by 2^-+60): used only to
// isolate eigenvalues; every bracket it yields is checked with FP64 counts.
__device__ __forceinline__ int sturm_count32_open(const float* d, const float* e2, int N, float x) {
  float pp = 1.0f, p = d[0] - x;
  uint32_t b = __float_as_uint(p);
  uint32_t sprev = 0u;
  uint32_t s = (b << 1) == 0u ? 1u : (b >> 31);
  int cnt = (int)(s ^ sprev);
  sprev = s;
  for (int i = 1; i < N; ++i) {
    const float pn = fmaf(-e2[i - 1], pp, (d[i] - x) * p);
    pp = p;
    p = pn;
    b = __float_as_uint(p);
    s = (b << 1) == 0u ? (sprev ^ 1u) : (b >> 31);
    cnt += (int)(s ^ sprev);
    sprev = s;
    const int ex = (int)((b >> 23) & 0xffu);
    if (ex > 127 + 60) {
      p *= 0x1p-60f;
      pp *= 0x1p-60f;
    } else if (ex < 127 - 60 && (int)((__float_as_uint(pp) >> 23) & 0xffu) < 127 - 60) {
      p *= 0x1p+60f;
      pp *= 0x1p+60f;
    }
  }
  return cnt;
}

// Shared start of the eigenvalues' FP32 bisections: G points strictly inside
// the (FP32) Gershgorin interval, point k at lo + (k + 1) h with
// h = (hi - lo) / (G + 1), and the FP32 Sturm count at each, one point per
// thread of the group.  The count at a point is the number of eigenvalues
// below it, so eigenvalue idx lies between the last point whose count is
// <= idx and the next one: about log2(G + 1) rounds of bisection that every
// eigenvalue would otherwise repeat on its own are taken in one round.  The
// counts live in the reduced matrix's storage, free by then beyond the
// first 2N doubles (at most N^2 - 3N ints).
struct OpenGrid {
  const int* cnt;
  int G;
  float lo, hi, h;
  __device__ __forceinline__ float x(int k) const { return __fmaf_rn((float)(k + 1), h, lo); }
  // [lo32, hi32]: neighbouring grid points (or interval ends) with
  // count(lo32) <= idx < count(hi32) as computed; the bisection goes on from
  // there, and the verification after it falls back to the Gershgorin interval
  // should the FP32 counts not be monotone
  __device__ __forceinline__ void bracket(int idx, float& lo32, float& hi32) const {
    int a = 0, b = G;
    while (a < b) {
      const int mid = (a + b) >> 1;
      if (cnt[mid] > idx) b = mid; else a = mid + 1;
    }
    lo32 = a == 0 ? lo : x(a - 1);
    hi32 = a == G ? hi : x(a);
  }
};

// Fill the grid (every thread of the group calls; the caller syncs the group
// before the counts are read).  d32 / e32 and the interval must be final.
__device__ __forceinline__ OpenGrid open_grid(const OpenWork& wk, int N, double glo, double ghi, int tid, int nt) {
  OpenGrid gr;
  int* cnt = reinterpret_cast<int*>(wk.A + 2 * N);
  gr.cnt = cnt;
  gr.G = min(nt, N * N - 3 * N);
  gr.lo = (float)glo;
  gr.hi = (float)ghi;
  gr.h = (gr.hi - gr.lo) / (float)(gr.G + 1);
  if (tid < gr.G) cnt[tid] = sturm_count32_open(wk.d32, wk.e32, N, gr.x(tid));
  return gr;
}

// FP64 Sturm count together with p_N(x) and p_N'(x) (for a Newton step):
// p_i' = (d_i - x) p_{i-1}' - p_{i-1} - e2_{i-1} p_{i-2}', all four values of a
// step rescaled together.  Five FP64 operations per step.
struct SturmNewton {
  int cnt;
  double p, dp;
};

__device__ __forceinline__ SturmNewton sturm_newton(const double* d, const double* e2, int N, double x) {
  double pp = 1.0, p = d[0] - x, dpp = 0.0, dp = -1.0;
  int hi = __double2hiint(p);
  uint32_t sprev = 0u;
  uint32_t s = ((hi & 0x7fffffff) | __double2loint(p)) == 0 ? 1u : ((uint32_t)hi >> 31);
  int cnt = (int)(s ^ sprev);
  sprev = s;
  for (int i = 1; i < N; ++i) {
    const double dx = d[i] - x;
    const double pn = fma(-e2[i - 1], pp, dx * p);
    const double dpn = fma(-e2[i - 1], dpp, fma(dx, dp, -p));
    pp = p;
    p = pn;
    dpp = dp;
    dp = dpn;
    hi = __double2hiint(p);
    const uint32_t zero = ((hi & 0x7fffffff) | __double2loint(p)) == 0;
    s = zero ? (sprev ^ 1u) : ((uint32_t)hi >> 31);
    cnt += (int)(s ^ sprev);
    sprev = s;
    const int ex = max((hi >> 20) & 0x7ff, (__double2hiint(dp) >> 20) & 0x7ff);
    if (ex > 1023 + 500) {
      p *= 0x1p-500;
      pp *= 0x1p-500;
      dp *= 0x1p-500;
      dpp *= 0x1p-500;
    } else if (ex < 1023 - 500 && max((__double2hiint(pp) >> 20) & 0x7ff, (__double2hiint(dpp) >> 20) & 0x7ff) <
                                      1023 - 500) {
      p *= 0x1p+500;
      pp *= 0x1p+500;
      dp *= 0x1p+500;
      dpp *= 0x1p+500;
    }
  }
  return {cnt, p, dp};
}

// Eigenvalue idx (ascending) of the tridiagonal: FP32 bisection isolates it,
// two FP64 Sturm counts verify the bracket (falling back to the Gershgorin
// interval), then safeguarded Newton steps on p_N refine it in FP64; every
// iterate updates the bracket through its Sturm count, and a step that leaves
// the bracket is replaced by bisection.
__device__ __forceinline__ double eigen_idx_open(const OpenWork& wk, const OpenGrid& gr, int N, int idx,
                                                 double glo, double ghi) {
  const double range = fmax(ghi - glo, 1e-300);
  float lo32, hi32;
  gr.bracket(idx, lo32, hi32);
  const float w32 = (float)(range * 0x1p-20);
  for (int it = 0; it < 48 && hi32 - lo32 > w32; ++it) {
    const float mid = 0.5f * (lo32 + hi32);
    if (!(mid > lo32 && mid < hi32)) break;
    if (sturm_count32_open(wk.d32, wk.e32, N, mid) > idx) hi32 = mid; else lo32 = mid;
  }
  const double pad = 0x1p-14 * range;
  double lo = fmax(glo, (double)lo32 - pad), hi = fmin(ghi, (double)hi32 + pad);
  if (sturm_count(wk.d, wk.vv, N, lo) > idx) lo = glo;
  if (sturm_count(wk.d, wk.vv, N, hi) <= idx) hi = ghi;
  const double tol_abs = 1e-15 * range;
  double x = 0.5 * (lo + hi);
  for (int it = 0; it < 100; ++it) {
    const double tol = fmax(tol_abs, 4.0 * 2.220446049250313e-16 * fmax(fabs(lo), fabs(hi)));
    if (hi - lo <= tol) {
      x = 0.5 * (lo + hi);
      break;
    }
    const SturmNewton r = sturm_newton(wk.d, wk.vv, N, x);
    if (r.cnt > idx) hi = x; else lo = x;
    const double step = r.p / r.dp;
    double xn = x - step;
    // a Newton step below the tolerance that stays in the bracket has found
    // the root: stop before the bracket test below can turn it into bisection
    // (x may sit on the root itself, which then is one end of the bracket)
    if (fabs(step) <= tol && xn >= lo && xn <= hi) {
      x = xn;
      break;
    }
    if (!(xn > lo && xn < hi)) xn = 0.5 * (lo + hi);
    if (fabs(xn - x) <= tol) {
      x = xn;
      break;
    }
    x = xn;
  }
  return x;
}

// log pi, e and c_f of an open lattice (see kitaev_logpi64 for the arguments),
// valid in the group's leader.
template <bool MULTI>
static __device__ __noinline__ void kitaev_logpi64_open(const Grp& g, const uint32_t* v, int L, const double* J,
                                                        double beta, const KitaevWork& kw, double (&res)[3],
                                                        double* eps_out = nullptr) {
  const OpenWork wk = {kw.A, kw.d, kw.e, kw.uw, kw.uw + L * L, kw.sc, (float*)kw.xs, (float*)kw.xs + L * L};
  const int N = L * L, tid = MULTI ? g.r : (int)threadIdx.x, nt = MULTI ? g.tpc : (int)blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  double* A = wk.A;
  const double tx = 2.0 * J[0], ty = 2.0 * J[1], tz = 2.0 * J[2];
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
      if (typ == 2 && j == 0) continue;      // this y-bond crosses the open cut
      const int b = bi * L + bj;
      const double mz = site_bit(v, b) ? tz : -tz;
      const double mw = (typ == 0) ? mz : (typ == 1 ? tx : ty);
      const int wz = b;
      const int wx = ((bi + 1 == L) ? 0 : bi + 1) * L + bj;
      const int wy = bi * L + ((bj + 1 == L) ? 0 : bj + 1);
      if (wz <= w) row[wz] += mw * mz;
      if (wx <= w) row[wx] += mw * tx;
      if (wy <= w && bj + 1 < L) row[wy] += mw * ty;
    }
  }
  grp_sync<MULTI>(g);
  // Householder tridiagonalisation, column j: x = A[j+1:, j] -> alpha e_1 by
  // H = I - tau u u^T, u = x - alpha e_1.  Only the lower triangle of the
  // trailing block A22 (rows and columns j+1..N-1, m of them) is read and
  // updated; the product with A22 reads u from column j itself (u_0 = x_0 -
  // alpha, u_c = A[j+1+c][j]), which the step does not change, and stores it
  // in vv for the update.  Three group barriers per column: p = tau A22 u
  // with H lanes per row and, per warp, the partial of p^T u; then w = p -
  // (tau p^T u / 2) u; then A22 -= u w^T + w u^T, its first column (with
  // per-warp partials of the next step's s, the sum of squares below the
  // subdiagonal) and the rest of the packed triangle element by element over
  // the group's threads in the folded order of FoldWalk.  sc[0..31]: p^T u
  // partials, sc[32..63]: s.
  double* scP = wk.sc;
  double* scS = wk.sc + 32;
  double s;
  {
    double s0 = 0.0;
    for (int i = 2 + tid; i < N; i += nt) {
      const double a = A[tri(i, 0)];
      s0 = fma(a, a, s0);
    }
    s = grp_sum<MULTI>(s0, g, wk.sc);
  }
  for (int j = 0; j < N - 2; ++j) {
    const int m = N - j - 1, j1 = j + 1;
    const double x0 = A[tri(j1, j)];
    if (tid == 0) wk.d[j] = A[tri(j, j)];
    if (s == 0.0) {
      // column already reduced: no reflection; s of the next column directly
      if (tid == 0) wk.e[j] = x0;
      double s2 = 0.0;
      for (int i = j + 3 + tid; i < N; i += nt) {
        const double a = A[tri(i, j1)];
        s2 = fma(a, a, s2);
      }
      s = grp_sum<MULTI>(s2, g, wk.sc);
      continue;
    }
    const double nrm = sqrt(x0 * x0 + s);
    const double alpha = (x0 >= 0.0) ? -nrm : nrm;
    const double u0 = x0 - alpha;
    const double tau = 2.0 / (u0 * u0 + s);
    if (tid == 0) wk.e[j] = alpha;
    // p_l = tau sum_c A22[l][c] u_c, u_c = A[tri(j1 + c, j)] (c >= 1): H lanes
    // of a warp per row (H = 1, 2, 4, .. while H m still fits the group), lane
    // h of a row taking the columns c = h mod H -- the row part c <= l
    // (contiguous), then the column part c > l -- alternately into two
    // accumulators, the H lanes' sums then added by a butterfly.  One loop for
    // both parts (see sym_at): ea, eb take turns, and a lane whose column part
    // starts out of turn exchanges them there, so that every sum keeps its order
    const int H = row_split(m, nt), h = lane & (H - 1);
    double part = 0.0;
    for (int l0 = 0; l0 < m; l0 += nt / H) {
      const int l = l0 + warp * (32 / H) + lane / H, lc = min(l, m - 1);
      double e = 0.0;
      if (l0 + warp * (32 / H) < m) {
        int c = h == 0 ? H : h;
        // ea: the odd accumulator of the row part, which its first term goes to
        double ea = 0.0, eb = h == 0 ? A[tri(j1 + lc, j1)] * u0 : 0.0;
        const int turns = lc >= c ? (lc - c) / H + 1 : 0;       // of the row part
        const int cross = (turns & 1) ? -1 : c + turns * H;     // (an even turn, so ea's)
        for (; c < m; c += 2 * H) {
          if (c == cross) {
            const double t = ea;
            ea = eb;
            eb = t;
          }
          ea = fma(sym_at(A, j1, c, lc), A[tri(j1 + c, j)], ea);
          if (c + H < m) eb = fma(sym_at(A, j1, c + H, lc), A[tri(j1 + c + H, j)], eb);
        }
        e = ea + eb;
      }
      for (int o = 1; o < H; o <<= 1) e += __shfl_xor_sync(kFull, e, o);
      if (l < m && h == 0) {
        const double p = tau * e, ul = l == 0 ? u0 : A[tri(j1 + l, j)];
        wk.pw[l] = p;
        wk.vv[l] = ul;
        part = fma(p, ul, part);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(kFull, part, o);
    if (lane == 0) scP[warp] = part;
    grp_sync<MULTI>(g);
    double pv = 0.0;
    for (int w = 0; w < nw; ++w) pv += scP[w];
    const double Kc = 0.5 * tau * pv;
    for (int l = tid; l < m; l += nt) wk.pw[l] = fma(-Kc, wk.vv[l], wk.pw[l]);
    grp_sync<MULTI>(g);
    // A22 -= u w^T + w u^T (u in vv, w in pw): column 0 of A22 -- the next
    // step's column -- row r by thread r mod nt, with the partials of s; then
    // the rest of the packed triangle (rows and columns 1..m-1), in the
    // folded order of FoldWalk
    const double* uu = wk.vv;
    const double* ww = wk.pw;
    double sp = 0.0;
    for (int r = tid; r < m; r += nt) {
      double* a = A + tri(j1 + r, j1);
      const double x = fma(-uu[r], ww[0], fma(-ww[r], u0, *a));
      *a = x;
      if (r >= 2) sp = fma(x, x, sp);
    }
    const int ntri = (m - 1) * m / 2;
    FoldWalk fw(m - 1, tid, nt);
    for (int q = tid; q < ntri; q += nt, fw.next()) {
      int r, c;
      fw.rc(r, c);
      double* a = A + tri(j1 + 1 + r, j1 + 1 + c);
      *a = fma(-uu[r + 1], ww[c + 1], fma(-ww[r + 1], uu[c + 1], *a));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sp += __shfl_xor_sync(kFull, sp, o);
    if (lane == 0) scS[warp] = sp;
    grp_sync<MULTI>(g);
    s = 0.0;
    for (int w = 0; w < nw; ++w) s += scS[w];
  }
  if (tid == 0) {
    wk.d[N - 2] = A[tri(N - 2, N - 2)];
    wk.d[N - 1] = A[tri(N - 1, N - 1)];
    wk.e[N - 2] = A[tri(N - 1, N - 2)];
    wk.e[N - 1] = 0.0;
  }
  grp_sync<MULTI>(g);
  // Gershgorin interval
  double glo = 1e300, ghi = -1e300;
  for (int i = tid; i < N; i += nt) {
    const double r = fabs(wk.e[i]) + (i > 0 ? fabs(wk.e[i - 1]) : 0.0);
    glo = fmin(glo, wk.d[i] - r);
    ghi = fmax(ghi, wk.d[i] + r);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    glo = fmin(glo, __shfl_xor_sync(kFull, glo, o));
    ghi = fmax(ghi, __shfl_xor_sync(kFull, ghi, o));
  }
  if (lane == 0) {
    wk.sc[2 * warp] = glo;
    wk.sc[2 * warp + 1] = ghi;
  }
  grp_sync<MULTI>(g);
  for (int w = 0; w < nw; ++w) {
    glo = fmin(glo, wk.sc[2 * w]);
    ghi = fmax(ghi, wk.sc[2 * w + 1]);
  }
  // squared off-diagonals for the Sturm recurrence (reuse vv), FP32 copies
  for (int i = tid; i < N; i += nt) {
    wk.vv[i] = wk.e[i] * wk.e[i];
    wk.d32[i] = (float)wk.d[i];
    wk.e32[i] = (float)(wk.e[i] * wk.e[i]);
  }
  grp_sync<MULTI>(g);
  const OpenGrid gr = open_grid(wk, N, glo, ghi, tid, nt);
  grp_sync<MULTI>(g);
  double lp = 0.0, en = 0.0, cf = 0.0;
  for (int idx = tid; idx < N; idx += nt) {
    const double mu = fmax(eigen_idx_open(wk, gr, N, idx, glo, ghi), 0.0);
    const double eps = sqrt(mu);
    if (eps_out) eps_out[idx] = eps;
    thermal_add(eps, beta, lp, en, cf);
  }
  float none = 0.0f;
  group_thermal<MULTI>(lp, en, cf, none, g, wk.sc);
  res[0] = lp;
  res[1] = en;
  res[2] = cf;
}

}  // namespace crbm
