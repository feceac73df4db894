"""Orthogonality of the Krylov basis after a full cycle of 63 steps: every tile size of the
fused projection-and-dot pass (up to 7, 15, 31, 51 and 63 vectors) contributes, on fields with fewer
tiles than SMs and on larger ones, in the single and in the lockstep solver.

No cycle ends early on these fields.  At kappa 0.25 the first projection cancels little and a
second one never runs; at 0.16 it runs in most steps, on the dots of the fused pass.  The basis is
orthogonal to the accuracy of the last projection's dot products: a thread or lane adds at most
82 terms in FP32 before FP64 (or a two-float sum) takes over, so |v_i . v_j| stays below
82 * 2^-24 = 5e-6 (a missing or misplaced term would leave 1e-3 and more)."""
import re

import numpy as np
import pytest
import torch

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


@pytest.mark.parametrize("fused", [True, False], ids=["fused", "apart"])
@pytest.mark.parametrize("dims,dom", [((4, 4, 8, 8), (2, 2, 4, 4)), ((8, 8, 8, 8), (4, 4, 4, 4)),
                                      ((24, 24, 24, 24), (4, 4, 4, 4))], ids=["4x4x8x8", "8^4", "24^4"])
def test_orthogonality_with_two_projections(dims, dom, fused, capfd, monkeypatch):
    """kappa 0.16, with the fused pass and with the two passes that stand in for it without tensor
    maps.  On 24^4 a group of warps hands its FP32 sums on in mid-run: every 2048 float4."""
    monkeypatch.setenv("DD_TRACE", "2")
    monkeypatch.setenv("DD_NO_TENSOR_MAPS", "0" if fused else "1")
    if dims[0] == 24:
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        assert np.prod(dims) * 6 // (4 * sms) > 2048, "too few tiles per group for a hand-over before the last one"
    U = gauge(dims, 0.6, 95)
    c = ctx_for(dims, dom, U, 0.16, 1.0)
    f = synth.gaussian_source(dims, 96)
    x = np.zeros_like(f)
    c.dd_solve(f, x, tol=1e-10, m=63, k=0, max_iter=63, i_schwarz=1, i_domain=1, check=False)
    err = capfd.readouterr().err
    second = re.findall(r"reorth (\d)", err)
    assert len(second) == 63
    for first, last in ((1, 7), (8, 15), (16, 31), (32, 51), (52, 63)):   # vectors per tile size
        assert "1" in second[first - 1:last], f"no second projection against {first} to {last} vectors"
    got = re.findall(r"max\|V\^H V - I\| = (\S+) over (\d+) vectors", err)
    assert int(got[-1][1]) == 64
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
