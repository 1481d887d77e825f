"""Convergence metrics (relay_metrics): the consensus distance and the
distance of the average model to the optimum, as in the paper's analysis."""
from fractions import Fraction

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


def _reference(x, mu):
    x, mu = np.asarray(x, np.float64), np.asarray(mu, np.float64)
    xbar = x.mean(axis=0)
    return ((x - xbar) ** 2).sum(axis=0).mean() / x.shape[0], ((xbar - mu.mean(axis=0)) ** 2).mean()


@pytest.mark.parametrize("d", [1, 7, 1031, 300_001])
def test_metrics_match_float64_definition(d):
    n = 9
    run = rs.RelayRun(n, d, wl.random_tree(n, 1), device="cuda:0")
    run.init(0.3, 4, wl.identity_mix(n), 2.0, 5, 0.5)
    for _ in range(3):
        run.step(0.2, 4)
    m = run.metrics()[0].cpu().numpy()
    want = _reference(run.x[:, :d].cpu().numpy(), run.mu[:, :d].cpu().numpy())
    assert np.allclose(m, want, rtol=1e-9, atol=0)
    # deterministic: the same bits on every call
    assert np.array_equal(run.metrics()[0].cpu().numpy(), m)


def test_metrics_with_regenerated_centres_equal_stored():
    n, d = 16, 50_000
    mix = wl.dirichlet_mix(n, 10, 0.1, seed=1)
    out = []
    for objective in ("stored", "generated"):
        run = rs.RelayRun(n, d, wl.chain(n), device="cuda:0", objective=objective)
        run.init(0.1, 0, mix, 1.0, 2, 0.05)
        for _ in range(4):
            run.step(0.05, 0)
        out.append(run.metrics()[0].cpu().numpy())
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("scale", [1.0, 10.0])
@pytest.mark.parametrize("shape", ["chain", "star", "binary"])
def test_noise_free_runs_converge_linearly(shape, scale):
    """sigma = 0: both metrics fall geometrically to zero whatever the spread
    of the centres (appendix "Independence of heterogeneity")."""
    n, d = 16, 4096
    edges = {"chain": wl.chain(n), "star": wl.star(n), "binary": wl.binary_tree(n)}[shape]
    run = rs.RelayRun(n, d, edges, device="cuda:0")
    run.init(0.0, 0, wl.identity_mix(n), scale, 3, 0.0)
    run.step(0.3, 0)
    first = run.metrics()[0].cpu().numpy()
    for _ in range(400):
        run.step(0.3, 0)
    last = run.metrics()[0].cpu().numpy()
    assert last[0] < 1e-9 * first[0] and last[1] < 1e-9 * max(first[1], 1e-30) + 1e-20


@pytest.mark.parametrize("shape,n", [("chain", 16), ("binary", 16), ("star", 16), ("torus", 16)])
def test_lr_correction_matches_oracle(shape, n):
    from oracle import oracle
    edges = {"chain": wl.chain(n), "binary": wl.binary_tree(n), "star": wl.star(n),
             "torus": wl.torus_spanning_tree(4, 4, 0)}[shape]
    alpha, limits = rs.lr_correction(n, edges, mode=1, device="cuda:0")
    E = 2 * (n - 1)
    x, mu = np.zeros((n, 1)), np.ones((n, 1))
    msg, c = np.zeros((E, 1)), np.zeros(E, np.int32)
    oracle.run(n, edges, x, mu, msg, c, 1.0, 0.0, 0, 0, 1, 1)
    oracle.run(n, edges, x, mu, msg, c, 0.0, 0.0, 0, 1, 5000, 1)
    assert abs(alpha - x[:, 0].mean()) < 1e-5
    assert 0.0 < alpha < 1.0


@pytest.mark.parametrize("n", [1, 2, 85])
@pytest.mark.parametrize("d", [5, 515, 120_001])
def test_metrics_at_the_edges_of_their_blocks(n, d):
    """One block and many, ragged last quads whose columns beyond d hold NaN.
    The bar is that of test_metrics_match_float64_definition."""
    run = rs.RelayRun(n, d, wl.random_tree(n, 2), device="cuda:0")
    run.init(0.3, 4, wl.identity_mix(n), 2.0, 5, 0.5)
    for _ in range(2):
        run.step(0.2, 4)
    run.x[:, d:] = float("nan")
    run.mu[:, d:] = float("nan")
    m = run.metrics()[0].cpu().numpy()
    assert np.allclose(m, _reference(run.x[:, :d].cpu().numpy(), run.mu[:, :d].cpu().numpy()), rtol=1e-9, atol=0)
    regenerated = rs.RelayRun(n, d, wl.random_tree(n, 2), device="cuda:0", objective="generated")
    regenerated.init(0.3, 4, wl.identity_mix(n), 2.0, 5, 0.5)
    for _ in range(2):
        regenerated.step(0.2, 4)
    assert np.array_equal(regenerated.metrics()[0].cpu().numpy(), m)


def _exact_distance(x, mu):
    """mean_c (xbar - mubar)^2 of float32 arrays in rational arithmetic."""
    diff = [sum(map(Fraction, map(float, x[:, c]))) - sum(map(Fraction, map(float, mu[:, c])))
            for c in range(x.shape[1])]
    return sum(v * v for v in diff) / (x.shape[0] ** 2 * x.shape[1])


def _metrics_of(x, mu):
    n, d = x.shape
    run = rs.RelayRun(n, d, wl.random_tree(n, 2), device="cuda:0")
    run.init(0.0, 4, wl.identity_mix(n), 0.0, 5, 0.0)
    run.x[:, :d] = torch.from_numpy(x)
    run.mu[:, :d] = torch.from_numpy(mu)
    return run.metrics()[0].cpu().numpy()


@pytest.mark.parametrize("n", [1, 3, 7, 24, 64])
@pytest.mark.parametrize("d", [5, 2051])
@pytest.mark.parametrize("gap", [1.0, 1e-4])
def test_distance_next_to_the_optimum(n, d, gap):
    """The average model close to the optimum, where a converging run ends.
    All values lie on a grid of 2^-20 below 8 and n <= 64, so the sums over
    the workers have at most 29 bits and their fp32 pairs are exact.  What
    remains is the rounding of the squares, of their sums (4 in a thread, 13
    over a block, 13 over the blocks) and of the scaling: under 40 roundings
    of 2^-53, all of positive terms."""
    rng = np.random.Generator(np.random.PCG64(n + d))
    grid = 2.0 ** -20
    mu = np.clip(rng.standard_normal((n, d)), -4, 4)
    x = mu.mean(axis=0) + gap * rng.standard_normal(d) + 1e-2 * rng.standard_normal((n, d))
    x, mu = (np.round(np.clip(v, -7.9, 7.9) / grid).astype(np.float64) * grid for v in (x, mu))
    x, mu = x.astype(np.float32), mu.astype(np.float32)
    want = _exact_distance(x, mu)
    got = Fraction(float(_metrics_of(x, mu)[1]))
    assert abs(got - want) <= 40 * Fraction(2) ** -53 * want, float((got - want) / want)


def test_distance_where_large_values_cancel():
    """A column's running sum (1e-3) ends below the rounding error that it
    gathered on the way (1.3): both are exact here, so the bar is the one
    above."""
    x = np.array([[1e8, 3e7, -2e8], [1.3, 0.7, 5.3], [-1e8, -3e7, 2e8], [1e-3, 2e-3, 3e-3]], np.float32)
    mu = np.zeros_like(x)
    want = _exact_distance(x, mu)
    got = Fraction(float(_metrics_of(x, mu)[1]))
    assert abs(got - want) <= 40 * Fraction(2) ** -53 * want, float((got - want) / want)


def test_distance_over_many_orders_of_magnitude():
    """Workers whose values differ by up to 2^40, so that a difference does
    not fit two fp32 values.  A worker sum gathers at most n rounding errors,
    each within 2^-24 of the largest partial sum, and rounds every addition of
    them: n^2 2^-48 sum_i |x_i| for its pair.  Behind that, the roundings of
    test_distance_next_to_the_optimum."""
    n, d = 6, 2051
    rng = np.random.Generator(np.random.PCG64(9))
    scale = np.exp2(-rng.integers(0, 41, size=(n, d)).astype(np.float64))
    x = (rng.standard_normal((n, d)) * scale).astype(np.float32)
    mu = (rng.standard_normal((n, d)) * scale[::-1]).astype(np.float32)
    want = _exact_distance(x, mu)
    diff = np.abs(x.astype(np.float64).sum(axis=0) - mu.astype(np.float64).sum(axis=0))
    delta = n ** 2 * 2.0 ** -48 * (np.abs(x).sum(axis=0, dtype=np.float64) + np.abs(mu).sum(axis=0, dtype=np.float64))
    bound = float(np.sum(2 * diff * delta + delta ** 2)) / (n * n * d) + 40 * 2.0 ** -53 * float(want)
    got = Fraction(float(_metrics_of(x, mu)[1]))
    assert abs(float(got - want)) <= bound, (float((got - want) / want), bound / float(want))


def test_distance_beyond_fp32_range():
    x = np.array([[3e38, 1.0, -3e38, 2e38]], np.float32)
    mu = np.array([[-3e38, 1.5, 3e38, 2e38]], np.float32)
    want = _exact_distance(x, mu)
    got = Fraction(float(_metrics_of(x, mu)[1]))
    assert abs(got - want) <= 40 * Fraction(2) ** -53 * want, float((got - want) / want)


def test_consensus_distance_of_a_quad_beyond_fp32_range():
    """Each coordinate's squares sum to 2e38, the four of a quad to 8e38.  The
    pair arithmetic is within 2^-40 for the two workers."""
    x = np.array([[1e19, -1e19, 1e19, 1e19], [-1e19, 1e19, -1e19, -1e19]], np.float32)
    got = _metrics_of(x, np.zeros_like(x))
    want = float(np.float32(1e19)) ** 2
    assert abs(got[0] - want) <= 2.0 ** -40 * want and got[1] == 0.0, got
