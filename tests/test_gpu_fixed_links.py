"""FP64 Dslash with links that the fixed-point format cannot hold, and with links of exact zeros."""
import numpy as np
import pytest
import torch

import oracle
from hisq_inputs import fields

hisq = pytest.importorskip("paper_2306_01098_gb300.hisq")

pytestmark = pytest.mark.gpu

SHAPES = [((6, 4, 4, 4), 1, (1, 1)), ((8, 8, 8, 8), 1, (1, 4)), ((4, 6, 8, 10), 3, (1, 2)), ((6, 4, 4, 4), 4, (4, 1)),
          ((8, 4, 4, 6), 2, (2, 2))]


def _apply(dims, fat, lng, b, shape, parity):
    ctx = hisq.Context(dims, torch.from_numpy(fat).cuda(), torch.from_numpy(lng).cuda(), precs=(hisq.F64,))
    ctx.tune_set(hisq.F64, hisq.F64, len(b), *shape)
    out = torch.full(b.shape, float("nan"), dtype=torch.complex128, device="cuda")
    ctx.dslash(parity, torch.from_numpy(b).cuda(), out)
    return out.cpu().numpy()


def _reached(dims, mask_fat, mask_lng, parity):
    """Sites of `parity` that have a marked link among their 16."""
    nx, ny, nz, nt = dims
    vh = nx * ny * nz * nt // 2
    t, z, y, x = np.meshgrid(np.arange(nt), np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    eo = ((x + nx * (y + ny * (z + nz * t))) // 2 + vh * ((x + y + z + t) % 2)).reshape(nt, nz, ny, nx)
    hit = np.zeros(2 * vh, dtype=bool)
    for mask, k in ((mask_fat, 1), (mask_lng, 3)):
        for mu in range(4):
            hit[eo.reshape(-1)] |= mask[mu][eo.reshape(-1)] | mask[mu][np.roll(eo, k, 3 - mu).reshape(-1)]
    return hit[parity * vh:(parity + 1) * vh]


@pytest.mark.parametrize("vector", ["zero", "point", "dense"])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("dims,nrhs,shape", SHAPES)
def test_links_that_are_not_finite(dims, nrhs, shape, value, vector):
    # FP64: 0 x NaN and 0 x infinity are NaN, so every site that such a link reaches shows it, whatever the
    # vector holds there; all other sites are untouched by it
    fat, lng = (a.numpy().copy() for a in fields.recipe_links(dims, 0.5, 1500))
    rng = np.random.default_rng(8)
    mask = [rng.random(a.shape[:2]) < 0.01 for a in (fat, lng)]
    for a, m in zip((fat, lng), mask):
        # one component of one entry, among the first three reals of the link too
        a.reshape(*a.shape[:2], 9)[m, rng.integers(0, 9)] = complex(value, 0.5) if rng.random() < 0.5 else complex(0.5, value)
    b = np.stack([fields.gaussian_source(dims, 2500 + r)[0].numpy() for r in range(nrhs)])
    if vector == "zero":
        b[:] = 0.0
    if vector == "point":
        b[:, 1:] = 0.0
    clean = [np.where(m[..., None, None], 0.0, a) for a, m in zip((fat, lng), mask)]
    for parity in (0, 1):
        got = _apply(dims, fat, lng, b, shape, parity)
        hit = _reached(dims, *mask, parity)
        assert hit.any() and not hit.all()
        assert (np.isfinite(got).all(-1) == ~hit).all()
        # without these links the other sites are the same to the last bit
        assert (_apply(dims, *clean, b, shape, parity)[:, ~hit] == got[:, ~hit]).all()


@pytest.mark.parametrize("dims,nrhs,shape", SHAPES)
def test_zeros_of_links_stay_zeros(dims, nrhs, shape):
    # diagonal links do not mix colours: exactly nothing arrives in the others, in FP64
    vol = int(np.prod(dims))
    fat = np.zeros((4, vol, 3, 3), dtype=np.complex128)
    fat[..., range(3), range(3)] = [1.0, 0.75, 1.0 / 3.0]
    lng = -0.125 * fat
    b = np.stack([fields.gaussian_source(dims, 2600 + r)[0].numpy() for r in range(nrhs)])
    for colour in range(3):
        v = np.zeros_like(b)
        v[..., colour] = b[..., colour]
        got = _apply(dims, fat, lng, v, shape, 1)
        others = [c for c in range(3) if c != colour]
        assert (got[..., others] == 0).all()
        v[..., colour].imag = 0.0
        assert (_apply(dims, fat, lng, v, shape, 1).imag == 0).all()
        want = np.stack([oracle.dslash(dims, fat, lng, v[r], 1) for r in range(nrhs)])
        # 16 products and sums of FP64, |U| <= 1
        assert np.abs(_apply(dims, fat, lng, v, shape, 1) - want).max() <= 32 * 2.0 ** -53 * 16 * np.abs(v).max()
