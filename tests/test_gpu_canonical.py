"""The operator on canonical fields: read directly where the fields allow 16-byte accesses, through
the layout passes where they do not (fields at odd addresses, or input and output overlapping),
on extents that are odd multiples of the domain's, at the operator tests' bars; and the batch
operator on the field counts where its pairs leave one over."""
import pytest
import torch

import synth
from oracle import wilson as W
from paper_1412_2629_gb300 import dd

from gpu_helpers import ctx_for, dev, gauge, host, rel

pytestmark = pytest.mark.gpu

LATTICES = [((8, 8, 12, 24), (4, 4, 2, 4)), ((16, 8, 8, 24), (8, 4, 4, 4)), ((8, 24, 8, 8), (4, 4, 4, 4)),
            ((4, 4, 4, 16), (2, 2, 2, 8))]


@pytest.mark.parametrize("dims,dom", LATTICES, ids=lambda d: "x".join(map(str, d)))
def test_canonical_fields_at_any_address(dims, dom):
    U = gauge(dims, 0.5, 51)
    f = synth.gaussian_source(dims, 52)
    want = W.apply_A(U, f, 0.124, 1.3)
    c = ctx_for(dims, dom, U, 0.124, 1.3)
    for dtype, prec, bar in ((torch.float64, dd.DD_PREC_FP64, 1e-13), (torch.float32, dd.DD_PREC_FP32, 1e-6)):
        src = dev(f, dtype)
        for off_in, off_out in ((0, 0), (1, 0), (0, 1), (3, 5)):
            a = torch.zeros(src.numel() + 8, dtype=dtype, device="cuda")
            b = torch.zeros_like(a)
            a[off_in:off_in + src.numel()] = src.reshape(-1)
            i, o = a[off_in:off_in + src.numel()], b[off_out:off_out + src.numel()]
            c.dd_apply_D(i, o, prec, dd.DD_LAYOUT_CANONICAL)
            assert rel(host(o.reshape(src.shape)), want) <= bar, (prec, off_in, off_out)
            assert (b[:off_out] == 0).all() and (b[off_out + src.numel():] == 0).all()
            packed = torch.empty(c.dd_spinor_bytes(prec, dd.DD_LAYOUT_INTERNAL), dtype=torch.uint8, device="cuda")
            c.dd_pack_spinor(i, prec, packed, prec)
            c.dd_unpack_spinor(packed, prec, o, prec)
            assert torch.equal(o, i)
        both = src.clone()
        c.dd_apply_D(both, both, prec, dd.DD_LAYOUT_CANONICAL)
        assert rel(host(both), want) <= bar


@pytest.mark.parametrize("n", [1, 2, 5])
@pytest.mark.parametrize("dims,dom", LATTICES, ids=lambda d: "x".join(map(str, d)))
def test_batches_with_one_left_over(dims, dom, n):
    U = gauge(dims, 0.5, 53)
    c = ctx_for(dims, dom, U, 0.124, 1.3)
    for prec, bar in ((dd.DD_PREC_FP32, 1e-6), (dd.DD_PREC_FP16, 3e-3)):
        nb = c.dd_spinor_bytes(prec, dd.DD_LAYOUT_INTERNAL)
        src = torch.empty(n * nb, dtype=torch.uint8, device="cuda")
        out = torch.zeros((n + 1) * nb, dtype=torch.uint8, device="cuda")
        fs = [synth.gaussian_source(dims, 54 + r) for r in range(n)]
        for r, f in enumerate(fs):
            c.dd_pack_spinor(dev(f), dd.DD_PREC_FP64, src[r * nb:(r + 1) * nb], prec)
        c.dd_apply_D_batch(src, out, n, prec)
        assert (out[n * nb:] == 0).all()
        for r, f in enumerate(fs):
            z = torch.empty(dims[::-1] + (4, 3, 2), dtype=torch.float64, device="cuda")
            c.dd_unpack_spinor(out[r * nb:(r + 1) * nb], prec, z, dd.DD_PREC_FP64)
            assert rel(host(z), W.apply_A(U, f, 0.124, 1.3)) <= bar, (prec, r)
