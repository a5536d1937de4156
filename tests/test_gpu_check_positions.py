"""Where a solve with predicted residual checks stops.

The rule: a check every `check_every` = m iterations, except that a check
which finds the tolerance n < m iterations away by the rate since the check
before asks for ceil(1.03 n) + 1 iterations, rounded up to whole chunks (of m
here, since m <= 50) - which for n close to m passes over the next check.  The
residuals at the multiples of m come from solves that end there by max_iter;
they differ from the predicted solve's by the rounding of a few more folds
(1e-6 relative at most), so layouts whose decisions lie closer are left out."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

M, TOL = 10, 1e-6


def _solid(seed):
    from paper_1711_04471_gb300 import inputs
    return inputs.les_buildings(24, 20, 14, dx=4.0, seed=seed, cover=0.2, margin_cells=3)


def _stop(rho):
    """(iterations at which the rule stops, distance of its closest decision), rho[k] after k m iterations."""
    k, prev, margin = 0, 0, 1.0
    while True:
        margin = min(margin, abs(rho[k] / TOL - 1.0))
        if k and rho[k] <= TOL:
            return k * M, margin
        step = 1
        if k and rho[k] < rho[prev]:
            lg = math.log(rho[k] / rho[prev]) / ((k - prev) * M)
            n = math.log(TOL / rho[k]) / lg
            margin = min(margin, abs(n / M - 1.0))
            if n < M:
                margin = min(margin, abs(1.03 * n + 1 - M))
                step = -(-max(1, math.ceil(1.03 * n) + 1) // M)
        prev, k = k, k + step


def test_predicted_checks_stop_where_the_rule_says():
    import paper_1711_04471_gb300 as P
    P.build()
    from paper_1711_04471_gb300.les import LES
    compared = passed_over = 0
    for seed in range(24):
        with LES(24, 20, 14, _solid(seed), check_every=M, tol=TOL) as g:
            got = g.step(1)[0]["iters"]
        rho = [1.0]
        with LES(24, 20, 14, _solid(seed), check_every=M, tol=TOL) as g:
            start = g.get_state()
            for k in range(1, got // M + 3):
                g.set_solver(tol=1e-30, max_iter=k * M)
                g.set_state(start)
                rho.append(g.step(1)[0]["rel_res"])
        want, margin = _stop(rho)
        if margin < 1e-4:
            continue
        compared += 1
        passed_over += any(r <= TOL for r in rho[1:want // M])
        assert got == want, (seed, got, want)
    assert compared >= 12
    assert passed_over >= 1
