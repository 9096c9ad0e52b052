"""Operator results written straight into the caller's FP64 buffer: equal, bit for bit, to those that
go through a field and the export pass, which a buffer off the 16-byte boundaries still takes."""
import ctypes

import pytest
import torch

from hisq_inputs import fields

hisq = pytest.importorskip("paper_2306_01098_gb300.hisq")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["F64X", "F32", "F16", "BF16"])
@pytest.mark.parametrize("dims,nrhs,shape", [((6, 4, 8, 10), 1, (1, 4, 1)), ((10, 4, 6, 4), 3, (1, 2, 1)),
                                             ((8, 8, 4, 6), 4, (2, 1, 2)), ((6, 4, 4, 4), 4, (4, 1, 1))])
def test_direct_and_exported_results_agree(dims, nrhs, shape, prec):
    p = getattr(hisq, prec)
    pv = hisq.F64X if prec == "F64X" else hisq.F32
    fat, lng = fields.recipe_links(dims, 0.5, 1400)
    b = torch.stack([fields.gaussian_source(dims, 2400 + r)[0] for r in range(nrhs)]).cuda()
    ctx = hisq.Context(dims, fat.cuda(), lng.cuda(), precs=(p,))
    ctx.tune_set(p, pv, nrhs, shape[0], shape[1])
    ctx.tune_set_groups(p, pv, nrhs, shape[2])
    n = b.numel() * 2
    flat = torch.empty(n + 1, dtype=torch.float64, device="cuda")
    L, st = hisq.lib(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    for call in (lambda o: L.hisq_dslash(ctx.h, 1, b.data_ptr(), o, nrhs, p, st),
                 lambda o: L.hisq_mdagm(ctx.h, ctypes.c_double(0.05), b.data_ptr(), o, nrhs, p, st)):
        direct = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
        flat.fill_(float("nan"))
        assert call(direct.data_ptr()) == 0
        assert call(flat.data_ptr() + 8) == 0
        torch.cuda.synchronize()
        assert torch.isfinite(direct).all()
        assert torch.equal(direct, flat[1:])
