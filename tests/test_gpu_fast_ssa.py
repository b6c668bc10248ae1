"""The SSA without FP64 (csrc/ssa_fast.cuh) at the edges of its conditions,
against the oracle: counts that leave their caps (replayed), counts and
networks it does not take (the FP64 path), coarsely represented rates, states
with a vanishing or zero total propensity, observation times far from zero,
orders 0 to 2, every reaction tier, and budgets met inside an interval.  The
bar is that of test_gpu_parity.py: equal statuses, event counts and digests."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import pf_oracle

pytestmark = pytest.mark.gpu


def _net(rx, U):
    R = len(rx)
    reac, prod = np.zeros((R, U), np.int32), np.zeros((R, U), np.int32)
    for r, (a, b) in enumerate(rx):
        for u, n in a.items():
            reac[r, u] = n
        for u, n in b.items():
            prod[r, u] = n
    return {"reactants": reac, "products": prod, "rate_index": None}


def _random_net(seed, U, R):
    rng = np.random.default_rng(seed)
    rx = []
    for _ in range(R):
        a = {}
        for _ in range(int(rng.integers(0, 3))):
            u = int(rng.integers(U))
            a[u] = a.get(u, 0) + 1
        b = {int(u): 1 for u in rng.choice(U, size=int(rng.integers(0, 3)), replace=False)}
        rx.append((a, b))
    return _net(rx, U)


BD = _net([({}, {0: 1}), ({0: 1}, {})], 1)
CASES = {
    # from 0 to thousands inside the first interval: beyond 4 max + 1024
    "growth": (BD, [[5000.0, 0.01], [900.0, 0.1], [1100.0, 0.0]], [0], [1.0, 2.0, 2.5]),
    # a burst of 100 per event: the room between two looks at the caps
    "bursts": (_net([({}, {0: 100}), ({0: 1}, {})], 1), [[20.0, 1.0], [300.0, 0.5]], [3], [0.5, 1.5, 3.0]),
    "dimer": (_net([({0: 2}, {1: 1}), ({1: 1}, {0: 2}), ({0: 1, 1: 1}, {0: 1}), ({}, {0: 1})], 2),
              [[1e-3, 0.5, 1e-4, 30.0], [2.0, 5.0, 0.1, 3.0]], [300, 1], [0.1, 0.2, 1.0]),
    # X + X with counts whose square passes 32 bits: the FP64 path
    "large_counts": (_net([({0: 2}, {}), ({}, {0: 1})], 1), [[1e-8, 5.0]], [70000], [0.5, 1.0]),
    "count_near_cap_square": (_net([({0: 2}, {}), ({}, {0: 1})], 1), [[1e-7, 5.0]], [16100], [0.5, 1.0]),
    # five species change in one reaction: the FP64 path
    "five_changes": (_net([({0: 1}, {1: 1, 2: 1, 3: 2, 4: 1}), ({1: 1, 2: 1}, {0: 1}), ({3: 1}, {}), ({4: 1}, {0: 1})], 5),
                     [[1.0, 0.1, 0.5, 0.2]], [20, 1, 0, 0, 5], [0.5, 1.0]),
    # times far from zero: rounding of t + tau; then beyond the path's limit
    "late_times": (BD, [[30.0, 0.3]], [40], [1000.0, 1000.25, 1001.0]),
    "very_late_times": (BD, [[0.05, 1.0]], [40], [40000.0, 40000.5, 40001.0]),
    # rates over fourteen decades: absolute error of the coarse ones
    "wide_rates": (_net([({}, {0: 1}), ({0: 1}, {}), ({0: 1}, {0: 1, 1: 1}), ({1: 2}, {})], 2),
                   [[1e-9, 1e-3, 50.0, 1e5], [5.0, 1e-11, 2.0, 1e4], [1e-12, 1e-12, 1e-12, 1e-12]], [4, 2], [1.0, 4.0]),
    # everything dies out; a rate of zero; no reaction possible at all
    "absorbing": (_net([({0: 1}, {}), ({0: 1, 1: 1}, {1: 1}), ({1: 1}, {})], 2),
                  [[1.0, 0.5, 2.0], [0.0, 1.0, 3.0], [0.0, 0.0, 0.0]], [6, 3], [0.5, 5.0, 50.0]),
    "tier8": (_random_net(5, 4, 7), None, [10, 20, 3, 0], [0.3, 1.0, 1.2]),
    "tier16": (_random_net(6, 7, 13), None, [10, 20, 3, 0, 5, 9, 1], [0.3, 1.0, 1.2]),
    "tier32": (_random_net(7, 16, 32), None, [5] * 16, [0.2, 0.5]),
}


@pytest.mark.parametrize("N", [1, 33, 150])
@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("cluster", [0, 2])
def test_matches_the_oracle(name, N, cluster):
    from paper_1606_08281_gb300 import pf
    if cluster and N == 1:
        pytest.skip("a cluster needs a particle per block")
    net, thetas, x0, times = CASES[name]
    R, U = net["reactants"].shape
    if thetas is None:
        thetas = np.exp(np.random.default_rng(R).uniform(np.log(0.02), np.log(3.0), size=(3, R)))
        thetas[:, net["reactants"].sum(1) == 2] *= 0.02
    thetas = np.asarray(thetas, float)
    C = np.zeros((1, U))
    C[0, 0] = 1.0
    y = np.full((2, len(times), 1), float(x0[0]))
    args = (net, thetas, np.asarray(x0, np.int32), np.asarray(times), y, C, np.array([200.0]), N, 91 + N)
    for budget in (0, 37):
        g = pf.pf_loglik(*args, event_budget=budget, diagnostics=True, cluster_blocks=cluster)
        o = pf_oracle.pf_loglik(*args, budget=budget or pf_oracle.DEFAULT_BUDGET)
        assert (g["status"] == o["status"]).all()
        ok = o["status"] == 0
        assert (g["events"][ok] == o["events"][ok]).all()
        assert (g["digest"][ok] == o["digest"][ok]).all()
        np.testing.assert_allclose(g["loglik"][ok], o["loglik"][ok], rtol=1e-9, atol=0)


@pytest.mark.parametrize("sigma", [1e-4, 0.05, 3.0, 1e7])
@pytest.mark.parametrize("N", [1, 31, 32, 257, 700])
def test_weights_match_the_oracle(sigma, N):
    """The integer exponential of the weights: sharp densities (most weights
    0 and far below 2^-62), flat ones (all near 1), the particles that attain
    the maximum, several observed dimensions with coefficients and offsets."""
    from paper_1606_08281_gb300 import pf
    net = _net([({}, {0: 1}), ({0: 1}, {}), ({0: 1}, {1: 1})], 2)
    thetas = np.array([[30.0, 0.5, 0.7], [4.0, 0.1, 0.1]])
    times = np.array([0.0, 0.5, 1.0, 2.0])
    C = np.array([[1.0, 0.0], [-0.25, 2.5]])
    y = np.array([[[3.0, 1.0], [14.0, 20.0], [20.0, 40.0], [25.0, 60.0]]])
    args = (net, thetas, np.array([3, 1], np.int32), times, y, C, np.array([sigma, 4 * sigma]), N, 17)
    g = pf.pf_loglik(*args, diagnostics=True)
    o = pf_oracle.pf_loglik(*args)
    assert (g["status"] == o["status"]).all()
    ok = o["status"] == 0
    assert (g["digest"][ok] == o["digest"][ok]).all()
    np.testing.assert_allclose(g["loglik"][ok], o["loglik"][ok], rtol=1e-12, atol=1e-12)
    y[0, 1, 0] = np.nan
    assert (pf.pf_loglik(*args)["status"] == pf.PF_ST_NONFINITE).all()


@pytest.mark.parametrize("name,N", [("gene_expression", 512), ("cascade", 64)])
def test_launch_order_by_mean_field_does_not_change_results(name, N):
    """PF_SCHED_AUTO's order (more filters than two per SM) against row order,
    with rows that are invalid, zero and beyond any estimate among them."""
    from paper_1606_08281_gb300 import pf
    from paper_1606_08281_gb300 import workloads as W
    w = W.get(name).subset(T=4, K=2)
    th = w.thetas(90).copy()
    th[3, 0] = -1.0
    th[5] = 0.0
    th[7, 0] = np.nan
    th[9, 0] = 1e300
    args = (w.net, th, w.x0, w.obs_times, w.observations(), w.C, w.sigma, N, 5)
    a = pf.pf_loglik(*args, event_budget=4096, diagnostics=True)
    b = pf.pf_loglik(*args, event_budget=4096, diagnostics=True, schedule=pf.PF_SCHED_NATURAL)
    assert (a["status"] == b["status"]).all()
    assert a["status"][3] == a["status"][7] == pf.PF_ST_INVALID_THETA
    ok = a["status"] == 0
    assert ok.sum() > 60
    for k in ("loglik", "ll_traj", "events", "digest"):
        assert (a[k][ok] == b[k][ok]).all()
