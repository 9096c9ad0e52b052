"""Smearing of links that the fixed-point products cannot take, or not to FP64's precision, and of links
that start off the 16-byte boundaries."""
import ctypes

import numpy as np
import pytest
import torch

from hisq_inputs import fields
from test_gpu_smear import _links_extended

hisq = pytest.importorskip("paper_2306_01098_gb300.hisq")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps", [1e-1, 1e-3, 1e-6, 1e-9])
@pytest.mark.parametrize("dims", [(10, 4, 6, 4), (4, 4, 4, 6)])
def test_small_entries_near_unity(dims, eps):
    # links near unity: every path has off-diagonal entries of order eps, and FP64 sums of them err by 1e-13
    # of that size, as sums of order-one products do by 1e-13 (the tolerance of the other tests)
    thin, _ = fields.recipe_links(dims, eps, 1203)
    fat, lng = hisq.smear_links(dims, thin.cuda(), eps_naik=0.1)
    want = _links_extended(dims, thin.numpy(), 0.1)
    off = ~np.eye(3, dtype=bool)
    for got, ref, tol in zip((fat, lng), want, (1e-13, 1e-14)):
        err = np.abs(got.cpu().numpy() - ref)
        assert err.max() <= tol
        assert err[..., off].max() <= tol * np.abs(ref[..., off]).max()


@pytest.mark.parametrize("dims", [(10, 4, 6, 4), (4, 4, 4, 6)])
def test_links_out_of_the_fixed_point_range(dims):
    # links of zeros, links 2^-250 of the others, links with reals too far apart, among links of order one
    thin = fields.recipe_links(dims, 0.3, 1204)[0].numpy().copy()
    rng = np.random.default_rng(11)
    pick = rng.random(thin.shape[:2])
    thin[pick < 0.02] = 0.0
    thin[(pick > 0.02) & (pick < 0.04)] *= 2.0 ** -250
    far = (pick > 0.04) & (pick < 0.06)
    thin[far] *= np.exp2(-rng.integers(0, 45, (int(far.sum()), 3, 3)))
    fat, lng = hisq.smear_links(dims, torch.from_numpy(thin).cuda())
    want_fat, want_lng = _links_extended(dims, thin, 0.0)
    assert np.abs(fat.cpu().numpy() - want_fat).max() <= 1e-13
    assert np.abs(lng.cpu().numpy() - want_lng).max() <= 1e-14


def test_thin_links_off_the_16_byte_boundaries():
    dims = (6, 4, 8, 4)
    thin = fields.recipe_links(dims, 0.5, 1205)[0].cuda()
    want = hisq.smear_links(dims, thin)
    flat = torch.empty(thin.numel() * 2 + 1, dtype=torch.float64, device="cuda")
    flat[1:] = torch.view_as_real(thin).reshape(-1)
    got = [torch.full_like(w, float("nan")) for w in want]
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    rc = hisq.lib().hisq_smear_links((ctypes.c_int * 4)(*dims), ctypes.c_void_p(flat.data_ptr() + 8), ctypes.c_void_p(got[0].data_ptr()),
                                     ctypes.c_void_p(got[1].data_ptr()), ctypes.c_double(0.0), 1, st)
    assert rc == 0
    for g, w in zip(got, want):
        assert torch.equal(g, w)
