"""The clover build's two inversion paths: symmetric sweeps with natural pivots, and pivoted
Gauss-Jordan for the blocks where a natural pivot is too small.

With a random (width 2) gauge field a c_sw of 12 makes many 6x6 blocks indefinite with
off-diagonal entries above their pivots, c_sw = 1 none.  The inverse is seen through one Schwarz
application in FP32 storage (one sweep, one MR step), compared with the FP64 oracle; rounding the
stored inverse and clover to FP32 moves the result by about 2^-24 times the blocks' condition
number, twice over (odd residual and Schur complement), so the bar is 30 * 2^-24 * max cond."""
import numpy as np
import pytest
import torch

import synth
from oracle import dd as DD
from oracle import wilson as W
from paper_1412_2629_gb300 import dd

from gpu_helpers import apply_gpu, ctx_for, dev, gauge, host, rel

pytestmark = pytest.mark.gpu


def site_blocks(F, kappa, csw, shape):
    """[sites, 12, 12] diagonal blocks of A, column by column."""
    cols = []
    for s in range(4):
        for c in range(3):
            e = np.zeros(shape + (4, 3), dtype=complex)
            e[..., s, c] = 1
            cols.append(DD.diag_part(F, e, kappa, csw).reshape(-1, 12))
    return np.stack(cols, -1)


@pytest.mark.parametrize("csw", [1.0, 12.0])
@pytest.mark.parametrize("dims,dom", [((8, 8, 8, 8), (4, 4, 4, 4)), ((8, 8, 12, 24), (4, 4, 2, 4))],
                         ids=["8x8x8x8", "8x8x12x24"])
def test_clover_and_inverse(dims, dom, csw):
    kappa = 0.125
    U = gauge(dims, 2.0, 91)
    F = W.field_strength(U)
    blocks = site_blocks(F, kappa, csw, dims[::-1])
    diag = np.abs(np.einsum("nii->ni", blocks))
    off = np.abs(blocks) * (1 - np.eye(12))
    assert (off.max(-1) > 2 * diag).any() == (csw > 5), "the field does not reach the path it is meant for"
    c = ctx_for(dims, dom, U, kappa, csw)
    f = synth.gaussian_source(dims, 92)
    assert rel(apply_gpu(c, f, dd.DD_PREC_FP64), W.apply_A(U, f, kappa, csw, F)) <= 1e-13
    want = DD.sap(U, F, f, kappa, csw, DD.Domains(dims, dom), 1, 1)
    src = dev(f, torch.float32)
    out = torch.empty_like(src)
    c.dd_sap_precondition(src, out, 1, 1, dd.DD_PREC_FP32, dd.DD_LAYOUT_CANONICAL)
    assert rel(host(out), want) <= 30 * 2.0 ** -24 * np.linalg.cond(blocks).max()
