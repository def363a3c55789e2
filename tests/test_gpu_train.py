"""Parity of the CUDA trainer (crbm_train_epochs, trainer.algorithm1) with the
oracle's (Sec. II, App. A, Algorithm 1).

FP64 on both sides with different summation orders: parameters, ADAM moments
and minibatch losses agree to 1e-9 relative after whole epochs; the ADAM step
counter exactly.  Algorithm 1 adds sampling (Metropolis physical samples,
Gibbs buffer) whose lattices are bit-exact between the two sides.
"""
import numpy as np
import pytest

import crbm_workloads as wl
from _common import gpu_ctx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = gpu_ctx()
    yield c
    c.close()


PROBLEMS = [
    # K, k, L, n_samples
    (2, 2, 3, 512),      # the paper's Ising protocol size (all states of L = 3)
    (2, 5, 8, 97),       # the paper's Kitaev kernel shape 2x5x5 at L = 8, ragged last batch
    (4, 3, 16, 45),
]


def test_epochs_match_oracle(ctx):
    import torch
    from oracle import ising, train
    from paper_2008_05401_gb300 import trainer
    batch, epochs = 20, 2
    probs, ref, data = [], [], []
    for j, (K, k, L, n) in enumerate(PROBLEMS):
        v = ising.all_states(L) if n == 2 ** (L * L) else wl.random_lattices(n, L, seed=j + 1)
        t = ising.energy(v) / 2.2
        th0 = wl.init_train_params(K, k, seed=j + 7)
        probs.append(trainer.Problem.new(ctx, K, k, L, th0))
        ref.append([th0.copy(), train.Adam.zeros(len(th0)), []])
        data.append((v, t))
    for e in range(epochs):
        xs, ts, os_ = [], [], []
        for j, (v, t) in enumerate(data):
            order = wl.epoch_order(len(t), 3, e)
            xs.append(torch.tensor(wl.pack_bits(v).view(np.int32), device="cuda:0"))
            ts.append(torch.tensor(t, device="cuda:0"))
            os_.append(torch.tensor(order, device="cuda:0"))
            K, k, _, _ = PROBLEMS[j]
            th, ls = train.epoch(ref[j][0], ref[j][1], v, t, order, K, k, M=batch)
            ref[j][0] = th
            ref[j][2].append(ls)
        losses = trainer.train_epochs(ctx, probs, xs, ts, os_, batch)
        for j in range(len(PROBLEMS)):
            np.testing.assert_allclose(losses[j].cpu().numpy(), ref[j][2][-1], rtol=1e-9, atol=1e-12)
    for j, pr in enumerate(probs):
        np.testing.assert_allclose(pr.theta.cpu().numpy(), ref[j][0], rtol=1e-9, atol=1e-12)
        np.testing.assert_allclose(pr.m.cpu().numpy(), ref[j][1].m, rtol=1e-9, atol=1e-14)
        np.testing.assert_allclose(pr.v.cpu().numpy(), ref[j][1].v, rtol=1e-9, atol=1e-18)
        assert int(pr.t.item()) == ref[j][1].t


@pytest.mark.parametrize("model", ["ising", "kitaev"])
def test_algorithm1_matches_oracle(ctx, model):
    from oracle import chain, train
    from paper_2008_05401_gb300 import ISING, KITAEV, trainer
    if model == "ising":
        kind, okind, L, Ts, J, K, k = ISING, chain.ISING, 4, [2.2, 3.0], (1.0,), 2, 3
    else:
        kind, okind, L, Ts, J, K, k = KITAEV, chain.KITAEV, 3, [0.3], (1.0, 1.0, 1.0), 2, 2
    th0 = wl.init_train_params(K, k, seed=11)
    kw = dict(n_phys=24, phys_sweeps=6, phys_seed=5, n_train=30, ub=10, g=2, rbm_seed=6, epochs=3, M=8, lr=1e-2)
    probs, hist = trainer.algorithm1(ctx, kind, L, Ts, J, K, k, th0, order_fn=lambda n, e: wl.epoch_order(n, 4, e),
                                     **kw)
    for i, T in enumerate(Ts):
        th, st, losses = train.algorithm1(okind, L, T, J, K, k, th0, order_seed=4, **kw)
        np.testing.assert_allclose(probs[i].theta.cpu().numpy(), th, rtol=1e-8, atol=1e-11)
        np.testing.assert_allclose(hist[:, i], losses, rtol=1e-8, atol=1e-11)
        assert int(probs[i].t.item()) == st.t


@pytest.mark.parametrize("model", ["ising", "kitaev"])
def test_pretraining_matches_oracle(ctx, model):
    """Pre-training on random states (App. A; Sec. IV; App. D): the random
    lattices drawn on the device, their targets, the epochs and the stopping
    rule give the oracle's epoch losses, stopping epoch and kept parameters at
    every temperature."""
    from oracle import chain, train
    from paper_2008_05401_gb300 import ISING, KITAEV, trainer
    if model == "ising":
        kind, okind, L, Ts, J, K, k = ISING, chain.ISING, 6, [2.0, 2.5, 3.2], (1.0,), 2, 3
    else:
        kind, okind, L, Ts, J, K, k = KITAEV, chain.KITAEV, 4, [0.1, 0.5], (1.0, 1.0, 1.0), 2, 3
    th0 = wl.init_train_params(K, k, seed=13)
    kw = dict(n_random=1500, seed=21, max_epochs=12, M=20, patience=2, rel_tol=0.02)
    probs, hist = trainer.pretrain(ctx, kind, L, Ts, J, K, k, th0, order_fn=lambda n, e: wl.epoch_order(n, 6, e),
                                   **kw)
    stopped_early = 0
    for i, T in enumerate(Ts):
        th, st, losses, n = train.pretrain(okind, L, T, J, K, k, th0, order_seed=6, **kw)
        assert len(hist[i]) == n
        stopped_early += n < kw["max_epochs"]
        np.testing.assert_allclose(hist[i], losses, rtol=1e-9, atol=1e-12)
        np.testing.assert_allclose(probs[i].theta.cpu().numpy(), th, rtol=1e-9, atol=1e-12)
        assert losses.min() < losses[0]
    if model == "ising":
        assert stopped_early >= 1                    # the stopping rule itself is exercised


def test_algorithm1_with_pretraining_matches_oracle(ctx):
    from oracle import chain, train
    from paper_2008_05401_gb300 import ISING, trainer
    L, Ts, J, K, k = 4, [2.2, 3.0], (1.0,), 2, 3
    th0 = wl.init_train_params(K, k, seed=11)
    kw = dict(n_phys=24, phys_sweeps=6, phys_seed=5, n_train=30, ub=10, g=2, rbm_seed=6, epochs=3, M=8, lr=1e-2)
    probs, hist = trainer.algorithm1(ctx, ISING, L, Ts, J, K, k, th0, order_fn=lambda n, e: wl.epoch_order(n, 4, e),
                                     pre=dict(n_random=400, seed=31, max_epochs=6,
                                              order_fn=lambda n, e: wl.epoch_order(n, 8, e)), **kw)
    for i, T in enumerate(Ts):
        th, st, losses = train.algorithm1(chain.ISING, L, T, J, K, k, th0, order_seed=4,
                                          pre=dict(n_random=400, seed=31, max_epochs=6, order_seed=8), **kw)
        np.testing.assert_allclose(probs[i].theta.cpu().numpy(), th, rtol=1e-8, atol=1e-11)
        np.testing.assert_allclose(hist[:, i], losses, rtol=1e-8, atol=1e-11)


@pytest.mark.parametrize("n_problems,K,k,L,n,batch", [
    (1, 2, 5, 8, 41, 20),      # cluster of 7 CTAs, a last minibatch of one sample
    (1, 1, 2, 2, 9, 1),        # one sample per minibatch, the smallest lattice
    (3, 2, 3, 17, 70, 64),     # the largest minibatch, windows wider than 16 columns
    (2, 4, 3, 31, 9, 5),       # odd side, three chunks of probabilities for a CTA's sample at most
    (80, 2, 3, 32, 20, 20),    # more problems than half the SMs: one CTA each, chunked, segments of 2048 units
    (40, 8, 2, 12, 25, 10),    # K = 8, two or three CTAs per problem
])
def test_cluster_split_matches_oracle(ctx, n_problems, K, k, L, n, batch):
    """The division of minibatches over a cluster's CTAs (samples per CTA,
    warps per sample, chunks of probabilities) leaves the epoch's results.
    Both sides round F (|F| below about N K) to a few units of 2^-52 |F|; a
    gradient component is (2/M) sum_i (diff_i - C) S_i with 0 <= S_i <= N, so it
    is off by eg = 2 N (4 2^-52 N K) whatever it cancels to, a moment m by the
    same, v by 2 |g| eg, and an ADAM step by at most lr times m's relative error."""
    import torch
    from oracle import train
    from paper_2008_05401_gb300 import trainer
    v = wl.random_lattices(n, L, seed=L + n)
    rng = np.random.default_rng(batch)
    ts = [rng.normal(0.0, 3.0, n) for _ in range(n_problems)]
    orders = [wl.epoch_order(n, 5, i) for i in range(n_problems)]
    probs = [trainer.Problem.new(ctx, K, k, L, wl.init_train_params(K, k, seed=i)) for i in range(n_problems)]
    x = torch.tensor(wl.pack_bits(v).view(np.int32), device="cuda:0")
    losses = trainer.train_epochs(ctx, probs, [x] * n_problems, [torch.tensor(t, device="cuda:0") for t in ts],
                                  [torch.tensor(o, device="cuda:0") for o in orders], batch)
    N, steps = L * L, -(-n // batch)
    eg = 2.0 * N * (4.0 * 2.0 ** -52 * N * K)
    for i in {0, n_problems // 2, n_problems - 1}:
        st = train.Adam.zeros(K * k * k + 1 + K)
        th, ls = train.epoch(wl.init_train_params(K, k, seed=i), st, v, ts[i], orders[i], K, k, M=batch)
        np.testing.assert_allclose(losses[i].cpu().numpy(), ls, rtol=1e-9, atol=1e-12)
        assert np.all(np.abs(probs[i].m.cpu().numpy() - st.m) <= eg + 1e-9 * np.abs(st.m))
        assert np.all(np.abs(probs[i].v.cpu().numpy() - st.v) <= 2.0 * np.sqrt(st.v / 0.001) * eg + 1e-9 * st.v)
        step = 1e-3 * steps * np.minimum(2.0, 2.0 * eg / np.maximum(np.abs(st.m), 1e-300))
        assert np.all(np.abs(probs[i].theta.cpu().numpy() - th) <= step + 1e-12)
        assert int(probs[i].t.item()) == st.t == steps


@pytest.mark.parametrize("L,k,hb,vb,spread", [(8, 3, (0.0, -25.0), 0.1, 3.0), (8, 3, (0.0, -40.0), 0.1, 3.0),
                                                 (8, 3, (0.0, -20.0), 0.1, 3.0), (16, 3, (0.0, -21.5), 0.1, 3.0),   # on either side of 2^-31
                                                 (17, 2, (0.5, -60.0), 0.1, 3.0),
                                                 (8, 3, (25.0, -40.0), 0.1, 3.0), (17, 2, (60.0, 1.0), 0.1, 3.0),
                                                 (8, 3, (-30.0, -35.0), 0.0, 0.0),     # F itself that small
                                                 (31, 2, (-30.0, -38.0), 0.0, 0.0)])
def test_silent_filters_keep_their_gradient(ctx, L, k, hb, vb, spread):
    """A filter whose units are all but off has a gradient of its own (small)
    size, which ADAM's normalisation restores.  One minibatch from zero moments:
    m / (1 - b1) is the gradient (2/M) sum_i d_i S_i, d_i = t_i - F_i - C, S_i >= 0
    a sum of at most N sigmas.  FP64 leaves d_i within 1e-12 (|t_i| + |F_i|) and
    S_i within 1e-12 of itself (a few hundred units of 2^-53 each)."""
    import torch
    from oracle import train
    from paper_2008_05401_gb300 import trainer
    n, K = 20, len(hb)
    v = wl.random_lattices(n, L, seed=L)
    rng = np.random.default_rng(5)
    t = rng.normal(0.0, spread, n)
    th0 = np.concatenate([rng.normal(0.0, 0.3, K * k * k), [vb], hb])
    prob = trainer.Problem.new(ctx, K, k, L, th0)
    losses = trainer.train_epochs(ctx, [prob], [torch.tensor(wl.pack_bits(v).view(np.int32), device="cuda:0")],
                                  [torch.tensor(t, device="cuda:0")], [torch.arange(n, dtype=torch.int32, device="cuda:0")], n)
    F, G = train.free_energy_grad(v, th0, K, k)
    d = t - F - (t - F).mean()
    off = 1e-12 * (np.abs(t) + np.abs(F))
    off += off.mean()
    tol = (2.0 / n) * ((off + 1e-12 * np.abs(d))[:, None] * np.abs(G)).sum(0)
    g = -(2.0 / n) * (d[:, None] * G).sum(0)
    assert np.all(np.abs(prob.m.cpu().numpy() / (1.0 - 0.9) - g) <= tol + 1e-13 * np.abs(g))
    assert abs(losses[0].item() - (d * d).mean()) <= 2.0 * (np.abs(d) * off).mean() + 1e-13 * (d * d).mean()


def test_train_rejects_bad_shapes(ctx):
    import torch
    from paper_2008_05401_gb300 import CrbmError, trainer
    pr = trainer.Problem.new(ctx, 2, 3, 40, wl.init_train_params(2, 3))      # L = 40 > 32
    x = torch.zeros((4, 50), dtype=torch.int32, device="cuda:0")
    t = torch.zeros(4, dtype=torch.float64, device="cuda:0")
    o = torch.arange(4, dtype=torch.int32, device="cuda:0")
    with pytest.raises(CrbmError):
        trainer.train_epochs(ctx, [pr], [x], [t], [o])
