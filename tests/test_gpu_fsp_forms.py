"""The forms of the exact likelihood's kernel -- reachable states, a window on
a one-species box, the box itself -- against the FSP oracle, at the sizes that
choose between them.  Tolerance as in test_gpu_fsp.py: 1e-9 relative."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import fsp

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


BD = _net([({}, {0: 1}), ({0: 1}, {})], 1)
BURST = _net([({}, {0: 7}), ({0: 1}, {}), ({0: 2}, {0: 1})], 1)
SWITCH = _net([({0: 1}, {1: 1}), ({1: 1}, {0: 1}), ({1: 1}, {1: 1, 2: 1}), ({2: 1}, {})], 3)
PAIR = _net([({0: 1, 1: 1}, {2: 1}), ({2: 1}, {0: 1, 1: 1}), ({0: 2}, {1: 2})], 3)
CASES = {
    # one species: below 256 states (reachable states), just above, large
    "bd_255": (BD, [[6.0, 0.5]], [3], [254], [0.5, 1.0, 2.0]),
    "bd_256": (BD, [[6.0, 0.5], [0.0, 0.5], [5.0, 0.0], [0.0, 0.0]], [3], [255], [0.0, 0.5, 1.0]),
    "bd_wide": (BD, [[150.0, 0.3], [40.0, 1.0]], [400], [900], [0.25, 1.0, 3.0]),
    "bd_at_the_edge": (BD, [[60.0, 0.1]], [290], [300], [0.5, 1.0]),
    "burst": (BURST, [[4.0, 0.6, 0.01], [0.2, 0.01, 0.5]], [40], [511], [0.25, 0.5, 2.0]),
    # conservation: two of the box's first two species' four states
    "switch": (SWITCH, [[0.3, 0.4, 5.0, 0.2], [1.0, 0.0, 2.0, 0.0]], [1, 0, 2], [1, 1, 60], [0.5, 2.0, 4.0]),
    "pair": (PAIR, [[0.05, 0.4, 0.02]], [9, 5, 1], [12, 12, 12], [0.5, 1.0]),
    # more states than a block's shared memory holds with their stencil
    "large_box": (SWITCH, [[0.3, 0.4, 5.0, 0.02]], [1, 0, 20], [1, 1, 2040], [0.05, 0.1]),
    "large_line": (BD, [[3.0, 0.002]], [2000], [8100], [0.05, 0.1]),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("spread", [0, 3])
def test_forms_match_the_oracle(name, spread):
    from paper_1606_08281_gb300 import pf
    net, thetas, x0, box, times = CASES[name]
    U = len(x0)
    C = np.zeros((1, U))
    C[0, U - 1] = 1.0
    x0 = np.asarray(x0, np.int32)
    y = np.full((1, len(times), 1), float(x0[U - 1]) + 1.5)
    model = None
    if spread:
        hi = x0.copy()
        hi[U - 1] = min(x0[U - 1] + spread, box[U - 1])
        model = {"x0_hi": hi}
    sigma = np.array([6.0])
    th = np.asarray(thetas, float)
    g = pf.pf_fsp_loglik(net, th, x0, np.asarray(box), np.asarray(times), y, C, sigma, model=model, diagnostics=True)
    want, _, leak = fsp.loglik_batch(net, th, x0, np.asarray(box), np.asarray(times), y, C, sigma, model=model)
    assert (g["status"] == 0).all()
    np.testing.assert_allclose(g["loglik"], want, rtol=1e-9, atol=0)
    np.testing.assert_allclose(g["leak"], leak, rtol=0, atol=1e-9)
