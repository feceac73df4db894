"""The first residual of a solve: f itself for a zero guess (the operator is skipped on the device),
f - A x for any other, also one whose squares underflow.  Every solve ends at the oracle's true
residual 1e-10; started at its own solution it takes no step."""
import numpy as np
import pytest

import synth
from oracle import solve as S
from paper_1412_2629_gb300 import dd

from gpu_helpers import ctx_for, gauge

pytestmark = pytest.mark.gpu

DIMS, DOM, KAPPA, CSW = (8, 8, 8, 8), (4, 4, 4, 4), 0.13, 1.0


@pytest.mark.parametrize("nrhs", [1, 2])
@pytest.mark.parametrize("scale", [0.0, 1e-200, 1.0, -3.0])
def test_initial_guess(scale, nrhs):
    U = gauge(DIMS, 0.6, 61)
    c = ctx_for(DIMS, DOM, U, KAPPA, CSW)
    f = np.stack([synth.gaussian_source(DIMS, 62 + r) for r in range(nrhs)])
    x = np.ascontiguousarray(scale * np.stack([synth.gaussian_source(DIMS, 72 + r) for r in range(nrhs)]))
    args = dict(nrhs=nrhs, tol=1e-10, m=16, k=4, i_schwarz=4, i_domain=4)
    first = c.dd_solve(f, x, **args)
    assert first.iterations > 0
    for r in range(nrhs):
        assert S.true_residual(U, x[r], f[r], KAPPA, CSW) <= 1e-10
    assert c.dd_solve(f, x, **args).iterations == 0


def test_gcr_from_zero():
    U = gauge(DIMS, 0.6, 63)
    c = ctx_for(DIMS, DOM, U, KAPPA, CSW)
    f = synth.gaussian_source(DIMS, 64)
    x = np.zeros_like(f)
    c.dd_solve_gcr(f, x, tol=1e-10, m=16, i_schwarz=4, i_domain=4)
    assert S.true_residual(U, x, f, KAPPA, CSW) <= 1e-10
    assert c.dd_solve_gcr(f, x, tol=1e-10, m=16, i_schwarz=4, i_domain=4, storage_prec=dd.DD_PREC_FP32).iterations == 0
