"""Parity of the CUDA path (through the C ABI) with the CPU oracle.

Every case runs the same chains, from the same packed lattices and Philox
streams, on both sides.  Lattices and accept counts must match bit for bit
unless the oracle reports a Bernoulli draw within 1e-12 of its threshold or an
MH decision within 1e-10 (relative) -- FP64 on the two sides uses different
exp/log implementations and summation orders, so only such draws may differ.
Floating results (log pi, F, observable sums) must agree to 1e-9 relative:
FP64 rounding over <= 2^16 terms of size O(1), well inside that.
"""
import numpy as np
import pytest

import crbm_workloads as wl
from _common import decisions_are_clear, gpu_ctx, oracle_chains, run_oracle

pytestmark = pytest.mark.gpu

SEED = 2008054010


@pytest.fixture(scope="module")
def ctx():
    c = gpu_ctx()
    yield c
    c.close()


def _compare(job, ref, worst, S, exact_floats=True):
    bits, step = job.state()
    lp, F, E = job.energies()
    sums, acc, rec = job.observables()
    assert step == S
    if not decisions_are_clear(worst):
        pytest.skip(f"oracle reports a decision inside the FP64 margin: {worst}")
    np.testing.assert_array_equal(bits, wl.pack_bits(ref.v))
    np.testing.assert_array_equal(acc, ref.accepts)
    np.testing.assert_allclose(lp, ref.logpi, rtol=1e-9, atol=1e-9)
    np.testing.assert_allclose(E, ref.E_phys, rtol=1e-9, atol=1e-9)
    np.testing.assert_allclose(sums, ref.obs, rtol=1e-9, atol=1e-9)
    if exact_floats:
        np.testing.assert_allclose(F, ref.F, rtol=1e-10, atol=1e-10)
    return bits, acc, rec, F


ISING_CASES = [
    # L, K, k, n, g, correct, std
    (4, 2, 3, 40, 1, True, 0.6),
    (6, 1, 2, 24, 1, True, 0.5),      # L % 4 != 0: ragged units across rows, N % 32 != 0
    (8, 2, 3, 16, 1, True, 0.1),      # the small Ising workload
    (8, 4, 5, 33, 2, True, 0.3),      # g = 2, ragged chain tail
    (12, 3, 4, 10, 1, False, 0.4),    # uncorrected Gibbs
    (16, 4, 5, 20, 1, True, 0.2),
    (24, 2, 7, 5, 1, True, 0.2),      # widest kernel
    (32, 4, 5, 6, 1, True, 0.15),
    (64, 4, 5, 3, 1, True, 0.1),      # several tiles of 4-site units, multi-word rows
    (96, 2, 3, 2, 1, True, 0.1),      # row of 3 words
    (256, 8, 6, 2, 1, True, 0.05),    # the largest lattice, K = 8 filters, K k 2^k = 3072 table entries
    (20, 4, 7, 3, 3, True, 0.1),      # k = 7 (largest kernel), g = 3
]


@pytest.mark.parametrize("L,K,k,n,g,correct,std", ISING_CASES)
def test_ising_matches_oracle(ctx, L, K, k, n, g, correct, std):
    from paper_2008_05401_gb300 import FP64, ISING, MIXED
    W, hb, vb = wl.gaussian_crbm(K, k, std, seed=L * 100 + K)
    T = wl.ising_ladder(n, 8)
    bits0 = wl.pack_bits(wl.random_lattices(n, L, seed=L))
    S = 12
    ref = oracle_chains("ising", W, hb, vb, L, T, (1.0,), SEED, n, bits0)
    worst = run_oracle(ref, S, g=g, correct=correct)
    mid = ctx.load_model(ISING, W, vb, hb)
    job = ctx.new_job(mid, ISING, L, T, (1.0,), SEED, 0, bits0, FP64)
    job.run(S, g=g, correct=correct, precision=FP64)
    bits64, acc64, rec64, F64 = _compare(job, ref, worst, S)
    assert rec64.sum() == 0
    # the mixed path takes exactly the FP64 path's decisions
    jm = ctx.new_job(mid, ISING, L, T, (1.0,), SEED, 0, bits0, MIXED)
    jm.run(S, g=g, correct=correct, precision=MIXED)
    bm, _ = jm.state()
    np.testing.assert_array_equal(bm, bits64)
    _, accm, recm = jm.observables()
    np.testing.assert_array_equal(accm, acc64)
    # read back in FP64 (crbm_read_energies re-evaluates a mixed job's lattices)
    lpm, Fm, Em = jm.energies()
    np.testing.assert_allclose(Fm, ref.F, rtol=1e-10, atol=1e-10)
    np.testing.assert_allclose(lpm, ref.logpi, rtol=1e-10, atol=1e-10)
    np.testing.assert_allclose(Em, ref.E_phys, rtol=1e-10, atol=1e-10)
    job.release()
    jm.release()


@pytest.mark.parametrize("L,K,k,n,g", [(2, 1, 2, 5003, 1), (4, 2, 3, 4999, 2), (6, 2, 3, 2501, 1), (8, 2, 3, 1301, 1),
                                       (12, 4, 3, 310, 1), (24, 2, 5, 307, 1)])
def test_many_ising_chains_match_oracle(ctx, L, K, k, n, g):
    """Enough chains for several to share a CTA, a warp or a word's lanes (the
    few chains of the cases above take a CTA each), a partly empty last CTA:
    both precisions against the oracle."""
    from paper_2008_05401_gb300 import FP64, ISING, MIXED
    W, hb, vb = wl.gaussian_crbm(K, k, 0.3, seed=L * 10 + K)
    T = wl.ising_ladder(n, 8)
    bits0 = wl.pack_bits(wl.random_lattices(n, L, seed=L))
    S = 3
    ref = oracle_chains("ising", W, hb, vb, L, T, (1.0,), SEED, n, bits0)
    worst = run_oracle(ref, S, g=g)
    mid = ctx.load_model(ISING, W, vb, hb)
    for prec in (FP64, MIXED):
        job = ctx.new_job(mid, ISING, L, T, (1.0,), SEED, 0, bits0, prec)
        job.run(S, g=g, precision=prec)
        _compare(job, ref, worst, S)
        job.release()


@pytest.mark.parametrize("L,K,k,n,g", [
    (3, 8, 3, 700, 2),       # a row repeated until it fills 64 bits; the window spans it
    (7, 3, 7, 200, 1),       # window as wide as the row
    (20, 4, 7, 40, 2),       # four sites of one row per unit, the widest window
    (28, 4, 5, 9, 1),
    (29, 4, 3, 9, 2),        # sites of two rows in a unit
    (31, 2, 5, 9, 1),        # the longest row
])
def test_repeated_rows_match_oracle(ctx, L, K, k, n, g):
    """Mixed precision at sides that are no multiple of 32, whose windows are
    taken from rows repeated over 64 bits: the oracle's chains."""
    from paper_2008_05401_gb300 import ISING, MIXED
    W, hb, vb = wl.gaussian_crbm(K, k, 0.2, seed=L * 10 + k)
    T = wl.ising_ladder(n, 8)
    bits0 = wl.pack_bits(wl.random_lattices(n, L, seed=L))
    S = 3
    ref = oracle_chains("ising", W, hb, vb, L, T, (1.0,), SEED, n, bits0)
    worst = run_oracle(ref, S, g=g)
    mid = ctx.load_model(ISING, W, vb, hb)
    job = ctx.new_job(mid, ISING, L, T, (1.0,), SEED, 0, bits0, MIXED)
    job.run(S, g=g, precision=MIXED)
    _compare(job, ref, worst, S)
    job.release()


@pytest.mark.parametrize("L,K,k,n,g,correct", [
    (32, 5, 3, 3, 1, True),      # clusters of 8, four rows per CTA
    (32, 2, 6, 2, 1, True),      # k - 1 = 5 rows of halo: clusters of 4
    (32, 2, 7, 30, 2, False),    # clusters of 4, two Gibbs steps, uncorrected
    (64, 8, 3, 40, 1, True),     # 40 chains: clusters of 2
    (96, 4, 5, 4, 2, True),      # rows of three words, twelve rows per CTA
    (96, 1, 1, 19, 1, True),     # one tap: the halo row only counts pairs; all 152 CTAs
    (96, 2, 5, 3, 1, True),      # two filters from one 8-byte table entry
    (160, 2, 3, 2, 1, True),
    (224, 4, 3, 2, 1, True),
    (256, 4, 5, 3, 1, True),
])
def test_divided_chains_match_oracle(ctx, L, K, k, n, g, correct):
    """Mixed-precision chains divided over a cluster's CTAs (few chains at a side
    or filter shape the tensor-core form does not have): the oracle's lattices,
    accepts, energies and sums."""
    from paper_2008_05401_gb300 import ISING, MIXED
    W, hb, vb = wl.gaussian_crbm(K, k, 0.15, seed=L + 10 * K + k)
    T = wl.ising_ladder(n, 8)
    bits0 = wl.pack_bits(wl.random_lattices(n, L, seed=L))
    S = 4
    ref = oracle_chains("ising", W, hb, vb, L, T, (1.0,), SEED, n, bits0)
    worst = run_oracle(ref, S, g=g, correct=correct)
    mid = ctx.load_model(ISING, W, vb, hb)
    job = ctx.new_job(mid, ISING, L, T, (1.0,), SEED, 0, bits0, MIXED)
    job.run(1, g=g, correct=correct, precision=MIXED)
    job.run(S - 1, g=g, correct=correct, precision=MIXED)
    _compare(job, ref, worst, S)
    job.release()


def test_divided_chains_in_a_batch_and_a_graph(ctx):
    """Jobs of several sides (clusters of 8 and 4 in one call), the same jobs in
    a call with too many chains for clusters, and a replayed graph: one result."""
    from paper_2008_05401_gb300 import ISING, MIXED
    W, hb, vb = wl.gaussian_crbm(2, 6, 0.15, seed=4)
    mid = ctx.load_model(ISING, W, vb, hb)

    def jobs(sizes):
        return [ctx.new_job(mid, ISING, L, wl.ising_ladder(n, 8), (1.0,), SEED, 100 * i,
                            wl.pack_bits(wl.random_lattices(n, L, seed=L)), MIXED) for i, (L, n) in enumerate(sizes)]
    sizes = [(32, 6), (96, 5), (160, 3)]
    a, b, c = jobs(sizes), jobs(sizes + [(64, 200)]), jobs(sizes)
    ctx.run_batch(a, 4, precision=MIXED)
    ctx.run_batch(b, 4, precision=MIXED)
    gr = ctx.graph(c, 2, precision=MIXED)
    gr.launch()
    gr.launch()
    for x, y, z in zip(a, b, c):
        sx, ax, _ = x.observables()
        for other in (y, z):
            so, ao, _ = other.observables()
            np.testing.assert_array_equal(other.state()[0], x.state()[0])
            np.testing.assert_array_equal(ao, ax)
            np.testing.assert_array_equal(so, sx)
    gr.destroy()
    for j in a + b + c:
        j.release()


@pytest.mark.parametrize("model,L,K,k,n,hb", [
    ("ising", 24, 2, 5, 40, 2e6),     # softplus sum 2.3e9, just past 2^31
    ("ising", 5, 3, 2, 40, 1e9),
    ("ising", 96, 2, 5, 12, 3e6),     # divided over clusters
    ("ising", 64, 8, 3, 12, 1e8),
    ("ising", 24, 2, 5, 40, -2e6),    # silent units: the sum vanishes
    ("kitaev", 4, 2, 3, 24, 2e8),
    ("ising", 16, 4, 5, 40, 3e6),     # a side and shape of the tensor-core form
    ("ising", 128, 2, 3, 12, 1e5),
    # F's own FP64 rounding of the size of the decisions: the same order of its sums too
    ("ising", 24, 2, 5, 40, 1e12),
    ("ising", 96, 2, 5, 12, 1e12),
    ("ising", 64, 8, 3, 40, 1e12),
    ("ising", 5, 3, 3, 1300, 1e12),   # other chains per CTA in FP64 than in mixed precision
    ("ising", 2, 8, 2, 701, 1e12),
])
def test_large_free_energies_keep_the_decisions(ctx, model, L, K, k, n, hb):
    """Filters whose free energy passes any fixed range of the mixed path's sums:
    its decisions are the FP64 path's whatever the size of F.  Weak filters and
    temperatures of the lattice's side keep F and log pi of two lattices within a
    few units, so that proposals are accepted and rejected."""
    from paper_2008_05401_gb300 import FP64, ISING, KITAEV, MIXED
    W, _, vb = wl.gaussian_crbm(K, k, 1.0 / (L * k), seed=L * 10 + K)
    kind, J = (ISING, (1.0,)) if model == "ising" else (KITAEV, (1.0, 1.0, 1.0))
    T = L * (wl.ising_ladder(n, 8) if model == "ising" else wl.kitaev_ladder(n, 8))
    bits0 = wl.pack_bits(wl.random_lattices(n, L, seed=L))
    mid = ctx.load_model(kind, W, vb, np.full(K, hb))
    S, got = 3, []
    for prec in (FP64, MIXED):
        job = ctx.new_job(mid, kind, L, T, J, SEED, 0, bits0, prec)
        job.run(S, precision=prec)
        got.append((job.state()[0], job.observables()[1]))
        job.release()
    assert 0 < got[0][1].sum() < n * S
    np.testing.assert_array_equal(got[1][0], got[0][0])
    np.testing.assert_array_equal(got[1][1], got[0][1])


@pytest.mark.parametrize("L,n,hb", [(8, 16, -25.0), (8, 16, -40.0), (24, 4, -60.0), (256, 1, -38.0), (3, 700, -300.0)])
def test_silent_units_keep_their_free_energy(ctx, L, n, hb):
    """F of a model whose units are all but off is the small sum of their softplus
    terms, to FP64's relative rounding (a few units of 2^-53 per term and
    addition), in an evaluation and at a run's end."""
    from oracle import crbm
    from paper_2008_05401_gb300 import FP64, ISING
    W, _, _ = wl.gaussian_crbm(2, 3, 0.3, seed=L)
    bits0 = wl.pack_bits(wl.random_lattices(n, L, seed=L))
    mid = ctx.load_model(ISING, W, 0.0, np.full(2, hb))
    job = ctx.new_job(mid, ISING, L, wl.ising_ladder(n, 8), (1.0,), SEED, 0, bits0, FP64)
    for S in (0, 2):
        job.run(S, precision=FP64)
        F = crbm.free_energy(wl.unpack_bits(job.state()[0], L), W, np.full(2, hb), 0.0)
        np.testing.assert_allclose(job.energies()[1], F, rtol=1e-12, atol=0.0)
    job.release()


KITAEV_CASES = [
    # L, K, k, n, correct
    (2, 2, 2, 6, True),
    (3, 4, 3, 8, True),    # odd L: N = 9, ragged units
    (4, 4, 3, 8, True),
    (6, 4, 3, 12, True),   # the small Kitaev workload geometry
    (5, 2, 3, 4, False),
    (8, 2, 5, 4, True),
    (12, 4, 3, 2, True),   # N = 144: largest matrix
]


@pytest.mark.parametrize("L,K,k,n,correct", KITAEV_CASES)
def test_kitaev_matches_oracle(ctx, L, K, k, n, correct):
    from paper_2008_05401_gb300 import FP64, KITAEV, MIXED
    W, hb, vb = wl.gaussian_crbm(K, k, 0.05, seed=L + 17)
    T = wl.kitaev_ladder(n, 24)
    J = (1.0, 1.0, 1.0) if L % 2 == 0 else (0.8, 1.1, 1.3)
    bits0 = wl.pack_bits(wl.random_lattices(n, L, seed=L + 3))
    S = 4
    ref = oracle_chains("kitaev", W, hb, vb, L, T, J, SEED, n, bits0)
    worst = run_oracle(ref, S, correct=correct)
    mid = ctx.load_model(KITAEV, W, vb, hb)
    job = ctx.new_job(mid, KITAEV, L, T, J, SEED, 0, bits0, FP64)
    job.run(S, correct=correct, precision=FP64)
    bits64, acc64, _, F64 = _compare(job, ref, worst, S)
    jm = ctx.new_job(mid, KITAEV, L, T, J, SEED, 0, bits0, MIXED)
    jm.run(S, correct=correct, precision=MIXED)
    bm, _ = jm.state()
    np.testing.assert_array_equal(bm, bits64)
    lpm, Fm, _ = jm.energies()
    np.testing.assert_allclose(Fm, ref.F, rtol=1e-10, atol=1e-10)
    np.testing.assert_allclose(lpm, ref.logpi, rtol=1e-10, atol=1e-9)
    job.release()
    jm.release()


@pytest.mark.parametrize("J", [(0.0, 0.0, 1.0), (0.7, 0.0, 1.2), (0.0, 0.9, 1.1)])
@pytest.mark.parametrize("L", [4, 6])
def test_kitaev_degenerate_couplings_match_oracle(ctx, L, J):
    """Vanishing couplings: with J_x = J_y = 0 the matrix M^T M is diagonal,
    so every column of the Householder reduction is already reduced (the
    step without a reflection) and the spectrum is N-fold degenerate; with
    one of them zero the lattice falls apart into chains (repeated
    eigenvalues, columns that vanish part-way through the reduction).  Both
    precisions against the oracle's singular values."""
    from paper_2008_05401_gb300 import FP64, KITAEV, MIXED
    W, hb, vb = wl.gaussian_crbm(4, 3, 0.05, seed=L + 29)
    n, S = 24, 3
    T = wl.kitaev_ladder(n, 24)
    bits0 = wl.pack_bits(wl.random_lattices(n, L, seed=L + 11))
    ref = oracle_chains("kitaev", W, hb, vb, L, T, J, SEED, n, bits0)
    worst = run_oracle(ref, S)
    mid = ctx.load_model(KITAEV, W, vb, hb)
    for prec in (FP64, MIXED):
        job = ctx.new_job(mid, KITAEV, L, T, J, SEED, 0, bits0, prec)
        job.run(S, precision=prec)
        _compare(job, ref, worst, S)
        job.release()


@pytest.mark.parametrize("scale", [1e-310, 1e-160, 1e-40])
def test_kitaev_tiny_couplings_match_oracle(ctx, scale):
    """Couplings far below the temperatures, down to subnormal numbers: every
    level's share of log pi is log 2 to rounding, in both precisions."""
    from paper_2008_05401_gb300 import FP64, KITAEV, MIXED
    W, hb, vb = wl.gaussian_crbm(2, 3, 0.05, seed=3)
    n, S, L, J = 12, 2, 4, (3 * scale, scale, 2 * scale)
    T = wl.kitaev_ladder(n, 12)
    bits0 = wl.pack_bits(wl.random_lattices(n, L, seed=L))
    ref = oracle_chains("kitaev", W, hb, vb, L, T, J, SEED, n, bits0)
    worst = run_oracle(ref, S)
    mid = ctx.load_model(KITAEV, W, vb, hb)
    for prec in (FP64, MIXED):
        job = ctx.new_job(mid, KITAEV, L, T, J, SEED, 0, bits0, prec)
        job.run(S, precision=prec)
        np.testing.assert_allclose(job.energies()[0], L * L * np.log(2.0), rtol=1e-12)
        _compare(job, ref, worst, S)
        job.release()


def test_random_init_matches_oracle(ctx):
    """init = 0 draws the lattices from the stream's init tag on the device."""
    from oracle import chain
    from paper_2008_05401_gb300 import FP64, ISING
    W, hb, vb = wl.gaussian_crbm(2, 3, 0.1)
    mid = ctx.load_model(ISING, W, vb, hb)
    for L, n, base in ((8, 5, 0), (6, 3, 1000), (64, 2, 2 ** 32 - 2)):
        job = ctx.new_job(mid, ISING, L, np.full(n, 2.0), (1.0,), 99, base, None, FP64)
        bits, _ = job.state()
        np.testing.assert_array_equal(bits, wl.pack_bits(chain.random_init(99, np.arange(base, base + n), L)))
        job.release()


def test_analytic_crbm_accepts_everything(ctx):
    """App. C: the analytic CRBM equals the Ising distribution, so every
    proposal is accepted, at any lattice size (here L = 128)."""
    from oracle import ising
    from paper_2008_05401_gb300 import FP64, ISING, MIXED
    beta = 1 / 2.269
    W, hb, vb = ising.analytic_crbm(beta, 3)
    mid = ctx.load_model(ISING, W, vb, hb)
    for prec in (FP64, MIXED):
        job = ctx.new_job(mid, ISING, 128, np.full(4, 1 / beta), (1.0,), SEED, 0, None, prec)
        job.run(10, precision=prec)
        _, acc, _ = job.observables()
        assert np.all(acc == 10)
        job.release()


@pytest.mark.parametrize("L,n,S", [(6, 24, 4), (10, 24, 4), (12, 24, 4), (6, 1024, 3), (12, 682, 2)])
def test_kitaev_mixed_df64_stage_matches_fp64(ctx, L, n, S):
    """The mixed path's df64 eigen-stage: lattices and acceptances identical to
    the FP64 path over the whole temperature ladder (down to T = 0.005), also
    at the Kitaev workloads' chain counts, and log-weights (read back in FP64)
    within 1e-10."""
    from paper_2008_05401_gb300 import FP64, KITAEV, MIXED
    W, hb, vb = wl.gaussian_crbm(4, 3, 0.05, seed=L + 99)
    T = wl.kitaev_ladder(n, 24)
    bits0 = wl.pack_bits(wl.random_lattices(n, L, seed=L + 5))
    mid = ctx.load_model(KITAEV, W, vb, hb)
    a = ctx.new_job(mid, KITAEV, L, T, (1.0, 1.0, 1.0), SEED, 0, bits0, FP64)
    b = ctx.new_job(mid, KITAEV, L, T, (1.0, 1.0, 1.0), SEED, 0, bits0, MIXED)
    a.run(S, precision=FP64)
    b.run(S, precision=MIXED)
    np.testing.assert_array_equal(a.state()[0], b.state()[0])
    _, acc_a, _ = a.observables()
    _, acc_b, rec_b = b.observables()
    np.testing.assert_array_equal(acc_a, acc_b)
    lp_a, _, E_a = a.energies()
    lp_b, _, E_b = b.energies()
    np.testing.assert_allclose(lp_b, lp_a, rtol=1e-10, atol=1e-9)
    np.testing.assert_allclose(E_b, E_a, rtol=1e-9, atol=1e-9)
    assert rec_b[:, 1].sum() <= n * S // 2          # MH recomputes stay the exception
    a.release()
    b.release()
