"""The two-threads-per-site Schwarz kernel at the edges of the domain shapes it accepts: the
smallest and largest domains, extents of 2 (both faces of a direction cover the domain) and
face blocks larger than the work buffers they are staged into.  Three right-hand sides in one
launch (the faces of the second and third are staged again), against the oracle at the bars
of the other Schwarz tests: MR step lengths compound FP32 rounding mildly (1e-5), FP16 storage
rounds every operand to 2^-11 (5e-3)."""
import pytest
import torch

import synth
from oracle import dd as DD
from oracle import wilson as W
from paper_1412_2629_gb300 import dd

from gpu_helpers import ctx_for, dev, gauge, host, rel

pytestmark = pytest.mark.gpu

SHAPES = [(2, 2, 4, 4), (4, 4, 2, 2), (2, 2, 2, 16), (16, 2, 2, 2), (4, 2, 8, 2), (2, 8, 4, 4), (8, 8, 2, 4), (2, 2, 2, 64),
          (8, 4, 4, 4), (4, 4, 4, 4)]


@pytest.mark.parametrize("additive", [0, 1])
@pytest.mark.parametrize("dom", SHAPES, ids=lambda b: "x".join(map(str, b)))
def test_domain_shapes_match_oracle(dom, additive):
    dims = tuple(2 * b for b in dom)
    kappa, csw, i_s, i_d, n = 0.124, 1.3, 2, 3, 3
    U = gauge(dims, 0.5, 71)
    F = W.field_strength(U)
    doms = DD.Domains(dims, dom)
    c = ctx_for(dims, dom, U, kappa, csw)
    nb = c.dd_spinor_bytes(dd.DD_PREC_FP32, dd.DD_LAYOUT_INTERNAL)
    src = torch.empty(n * nb, dtype=torch.uint8, device="cuda")
    out = torch.empty_like(src)
    want = []
    for r in range(n):
        f = synth.gaussian_source(dims, 80 + r)
        c.dd_pack_spinor(dev(f), dd.DD_PREC_FP64, src[r * nb:(r + 1) * nb], dd.DD_PREC_FP32)
        want.append((DD.sap_additive if additive else DD.sap)(U, F, f, kappa, csw, doms, i_s, i_d))
    for prec, bar in ((dd.DD_PREC_FP32, 1e-5), (dd.DD_PREC_FP16, 5e-3), (dd.DD_PREC_FP16_H2, 5e-3)):
        c.dd_sap_precondition_batch(src, out, n, i_s, i_d, prec, additive=additive)
        for r in range(n):
            z = torch.empty(dims[::-1] + (4, 3, 2), dtype=torch.float64, device="cuda")
            c.dd_unpack_spinor(out[r * nb:(r + 1) * nb], dd.DD_PREC_FP32, z, dd.DD_PREC_FP64)
            assert rel(host(z), want[r]) <= bar, (prec, r)
