"""Which of two builds or layouts a launch takes must not show in its results:
the step kernels for up to 64 workers (and 256 mixture weights) against those
for up to 256, the walk's two register budgets, and counters that settle
before the last step of a call.  All compared bit for bit (the paths form the
same sums in the same order)."""
import numpy as np
import pytest
import torch

import paper_2110_04175_gb300 as rs
from paper_2110_04175_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _run(n, d, edges, steps, mix, mode=1, **kw):
    run = rs.RelayRun(n, d, edges, device="cuda:0", mode=mode, **kw)
    run.init(0.1, 3, mix, 1.0, 5, 0.05)
    for _ in range(steps):
        run.step(0.05, 3)
    return run


def _same(a, b):
    assert torch.equal(a.x[:, :a.d], b.x[:, :b.d])
    assert torch.equal(a.messages[:a.E, :a.d], b.messages[:b.E, :b.d])
    assert torch.equal(a.counts, b.counts)


# 64 workers with 4 and 5 dense centres: 256 and 320 weights; 65 workers take the larger build
@pytest.mark.parametrize("n,K", [(64, 4), (64, 5), (65, 3), (16, 16), (17, 16)])
@pytest.mark.parametrize("kernel", ["walk", "nodes"])
def test_capacity_of_the_launch_does_not_show(n, K, kernel):
    d = 1031
    mix = wl.dirichlet_mix(n, K, 5.0, seed=2)
    assert np.count_nonzero(mix) == n * K
    edges = wl.random_tree(n, 4)
    stored = _run(n, d, edges, 5, mix, kernel=kernel)
    generated = _run(n, d, edges, 5, mix, kernel=kernel, objective="generated")
    _same(stored, generated)
    other = _run(n, d, edges, 5, mix, kernel="nodes" if kernel == "walk" else "walk")
    _same(stored, other)


# grids of 1.6 waves (7 CTAs per SM) and of 0.96 and 3.2 waves (8 or 7) at 152 SMs
@pytest.mark.parametrize("d", [600_003, 1_000_003, 2_000_001])
@pytest.mark.parametrize("optimizer", [None, ("nesterov", 0.9), ("adam", 0.9, 0.999, 1e-8)])
def test_walk_register_budgets_give_the_same_bits(d, optimizer):
    n, edges = 5, wl.binary_tree(5)
    mix = wl.identity_mix(n)
    _same(_run(n, d, edges, 2, mix, kernel="walk", optimizer=optimizer),
          _run(n, d, edges, 2, mix, kernel="nodes", optimizer=optimizer))


@pytest.mark.parametrize("shape,n", [("chain", 9), ("star", 7), ("binary", 16), ("pair", 2), ("one", 1)])
@pytest.mark.parametrize("k", [1, 2, 8, 66])
@pytest.mark.parametrize("algorithm", ["relaysgd", "dme"])
def test_steps_from_any_counters(shape, n, k, algorithm):
    """relay_steps runs as many counter rounds as the tree's longest path has
    edges; k relay_step calls run k, whatever the counters before them."""
    edges = {"chain": wl.chain, "star": wl.star, "binary": wl.binary_tree, "pair": wl.chain, "one": wl.chain}[shape](n)
    rng = np.random.Generator(np.random.PCG64(n + k))
    lost = (rng.random(2 * (n - 1)) < 0.2).astype(np.uint8)
    start = torch.from_numpy(rng.integers(-1000, 1000, size=max(2 * (n - 1), 1)).astype(np.int32))
    runs = []
    for _ in range(2):
        run = rs.RelayRun(n, 77, edges, device="cuda:0", mode=1, kernel="nodes", algorithm=algorithm,
                          received_sums=False)
        run.init(0.1, 3, wl.identity_mix(n), 1.0, 5, 0.05)
        run.counts.copy_(start)
        if n > 1:
            run.set_lost(lost)
        runs.append(run)
    runs[0].steps(k, 0.05, 3)
    for _ in range(k):
        runs[1].step(0.05, 3)
    _same(*runs)
    if algorithm == "dme":
        assert torch.equal(runs[0].trees[0].dme_count, runs[1].trees[0].dme_count)


# 24 and 40 workers: warps whose workers differ in degree
@pytest.mark.parametrize("n", [2, 5, 24, 40])
def test_paths_agree_in_the_sign_of_zero(n):
    """Models, messages and centres at -0 and 0 without noise: the sums are
    zeros of either sign, and a lane with fewer neighbours than its warp's
    widest must add nothing for the missing ones."""
    d, edges = 77, wl.random_tree(n, 3)
    runs = {}
    for kernel in ("walk", "nodes", "steps"):
        run = rs.RelayRun(n, d, edges, device="cuda:0", mode=1, kernel="walk" if kernel == "walk" else "nodes",
                          received_sums=False)
        run.init(0.0, 3, wl.identity_mix(n), 0.0, 5, 0.0)
        run.mu.zero_()
        for t in (run.x, run.msg[0], run.msg[1]):
            t.fill_(-0.0)
        if kernel == "steps":
            run.steps(3, 0.05, 3)
        else:
            for _ in range(3):
                run.step(0.05, 3)
        runs[kernel] = run
    walk = runs["walk"]
    assert bool((walk.x[:, :d].view(torch.int32) != 0).any()) and not bool(walk.x[:, :d].any())
    for other in (runs["nodes"], runs["steps"]):
        for a, b in ((walk.x, other.x), (walk.messages[:walk.E], other.messages[:walk.E])):
            assert torch.equal(a[:, :d].view(torch.int32), b[:, :d].view(torch.int32))
