"""The Erk kernels' branch-free quotients: rows whose operands leave the range
in which they are used (an absolute tolerance below 2^-60 puts every error
quotient of the forms that are still zero outside it) take the IEEE division
and give the same likelihood as in-range rows within the solver's tolerance."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 37, 4000])
def test_out_of_range_operands_use_ieee_division(M):
    from oracle import ode
    from paper_1606_08281_gb300 import pf
    from paper_1606_08281_gb300 import workloads as W
    e = W.erk()
    K = 3 if M == 4000 else 6
    th = e.thetas(M)
    pats, times, y = e.patterns[:2], e.obs_times[:K], e.observations()[:2, :K]
    tiny = pf.pf_erk_loglik(th, pats, times, y, rtol=1e-10, atol=1e-25)
    ref = pf.pf_erk_loglik(th, pats, times, y, rtol=1e-12, atol=1e-15)
    assert (tiny["status"] == 0).all() and (ref["status"] == 0).all()
    # per-step relative error 1e-10, accumulated over at most a few hundred
    # steps; d ll / d R = (y - R) / sigma^2 <= 2500 over 12 readings
    np.testing.assert_allclose(tiny["loglik"], ref["loglik"], rtol=1e-6, atol=1e-4)
    for i in range(min(M, 2)):
        want = sum(ode.loglik(th[i], [p], times, y[j:j + 1])[0] for j, p in enumerate(pats))
        assert abs(tiny["loglik"][i] - want) <= 1e-6 * abs(want) + 1e-4
