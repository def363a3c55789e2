// Local-update Metropolis sweeps of the Kitaev model (the paper's baseline,
// Sec. IV), run by the fused kernel in mode 3 with the lattices resident in
// shared memory (the Ising sweeps have a kernel of their own, crbm_sweep.cu).
//
// Kitaev: sites n = 0 .. N-1 in order; eta_n flips iff
// log u_site < log pi(eta with eta_n flipped) - log pi(eta), each proposal
// needing one eigen-stage.  The uniform of site n is word n % 4 of Philox
// block n / 4 of tag kTagLocal at the sweep's step.
#pragma once
#include "crbm_device.cuh"
#include "crbm_df64.cuh"

namespace crbm {

// Number of hexagons with flux -1 of lattice v: a per-thread partial.
__device__ inline double flux_count(const JobDev& jb, const Grp& g, const uint32_t* v) {
  const int L = jb.L, N = jb.N;
  int pairs = 0;
  if (g.active) {
    for (int n = g.r; n < N; n += g.tpc) {
      // the hexagon of cell r holds the z-bonds r and r - e1 + e2 (none in
      // column L-1 when the columns are open)
      const int i = n / L, j = n - i * L;
      const int i2 = (i == 0) ? L - 1 : i - 1, j2 = (j + 1 == L) ? 0 : j + 1;
      if (!(jb.lc_edge && j + 1 == L)) pairs += (int)(site_bit(v, n) ^ site_bit(v, i2 * L + j2));
    }
  }
  return (double)pairs;
}

}  // namespace crbm
