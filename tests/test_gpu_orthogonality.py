"""Orthogonality of the Krylov basis after a full cycle of 63 steps: every tile size of the
fused projection-and-dot pass (up to 7, 15, 31 and 63 vectors) contributes, on a field with
fewer tiles than SMs and on larger ones, in the single and in the lockstep solver.

kappa 0.25 lies far above critical, so no cycle ends early.  With two projections the basis is
orthogonal to the accuracy of the second one's dot products: a thread or lane adds at most 82
terms in FP32 before FP64 takes over, so |v_i . v_j| stays below 82 * 2^-24 = 5e-6 (a missing or
misplaced term would leave 1e-3 and more)."""
import re

import numpy as np
import pytest

import synth
from paper_1412_2629_gb300 import dd

from gpu_helpers import ctx_for, gauge

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,dom,m", [((8, 8, 4, 4), (4, 4, 2, 2), 63), ((8, 8, 8, 8), (4, 4, 4, 4), 63),
                                        ((16, 16, 8, 24), (4, 4, 4, 4), 35)], ids=["8x8x4x4", "8^4", "16x16x8x24"])
def test_basis_orthogonality(dims, dom, m, capfd, monkeypatch):
    monkeypatch.setenv("DD_TRACE", "2")
    U = gauge(dims, 0.6, 95)
    c = ctx_for(dims, dom, U, 0.25, 1.0)
    f = synth.gaussian_source(dims, 96)
    x = np.zeros_like(f)
    c.dd_solve(f, x, tol=1e-10, m=m, k=0, max_iter=m, i_schwarz=1, i_domain=1, check=False)
    got = re.findall(r"max\|V\^H V - I\| = (\S+) over (\d+) vectors", capfd.readouterr().err)
    assert got and int(got[-1][1]) == m + 1, got
    assert float(got[-1][0]) <= 82 * 2.0 ** -24


def test_lockstep_takes_the_same_steps():
    """Two right-hand sides in lockstep reach the residual that two single solves reach after
    the same number of steps (FP32 vectors: equal to rounding)."""
    dims, dom = (8, 8, 8, 8), (4, 4, 4, 4)
    U = gauge(dims, 0.6, 95)
    c = ctx_for(dims, dom, U, 0.13, 1.0)
    f = np.stack([synth.gaussian_source(dims, 97 + r) for r in range(2)])
    x = np.zeros_like(f)
    args = dict(tol=1e-10, m=40, k=0, i_schwarz=1, i_domain=2)
    both = c.dd_solve(f, x, nrhs=2, **args)
    its = 0
    for r in range(2):
        y = np.zeros_like(f[r])
        its += c.dd_solve(f[r], y, **args).iterations
        assert np.linalg.norm(x[r] - y) <= 1e-8 * np.linalg.norm(y)
    assert abs(both.iterations - its) <= 2
