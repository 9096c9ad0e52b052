"""FP64 Dslash with 18-real links, component by component: no less precise than FP64 multiply-adds where the
reals of links and vectors are of very different sizes.

Tolerance of a component: 200 u S, u = 2^-53, S = sum over its hops of |Re U| |Re v| + |Im U| |Im v| (real
part; crosswise for the imaginary part).  Each side's sum of 96 products errs by at most 97 u S with FP64
operations (the staggered signs cost nothing), and the fixed-point sites are held to the same.
"""
import numpy as np
import pytest
import torch

import oracle
from hisq_inputs import fields

hisq = pytest.importorskip("paper_2306_01098_gb300.hisq")

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
SHAPES = [((4, 6, 8, 10), 1, (1, 1)), ((8, 8, 8, 8), 1, (1, 4)), ((10, 4, 6, 4), 3, (1, 2)), ((6, 4, 4, 4), 4, (4, 1)),
          ((8, 4, 4, 6), 2, (2, 2))]


def _links(dims, kind):
    fat, lng = (a.numpy().copy() for a in fields.recipe_links(dims, {"near unity": 1e-4}.get(kind, 0.5), 1600))
    rng = np.random.default_rng(9)
    if kind == "unit":
        fat[:], lng[:] = np.eye(3), np.eye(3) / -24
    if kind == "small entries":
        for a in (fat, lng):
            a *= np.exp2(-rng.integers(0, 60, a.shape) * (rng.random(a.shape) < 0.3))
            a[rng.random(a.shape[:2]) < 0.1, 0, 1] = 1e-19 / 3
    if kind == "scales":
        for a in (fat, lng):
            a *= np.exp2(rng.integers(-60, 61, a.shape[:2]))[..., None, None]
    return fat, lng


def _vectors(dims, nrhs, kind):
    b = np.stack([fields.gaussian_source(dims, 2700 + r)[0].numpy() for r in range(nrhs)])
    rng = np.random.default_rng(10)
    if kind == "colours":
        b *= [1.0, 1e-9, 1e-20]
    if kind == "parts":
        b.imag *= 1e-13
    if kind == "one colour":
        b[..., 1:] = 0.0
    if kind == "steep":
        b *= np.exp2(rng.integers(-40, 41, b.shape[:2]))[..., None]
    if kind == "decay":  # a site's neighbours within a factor of a few
        b *= np.exp(rng.normal(size=b.shape[:2]))[..., None]
    return b


def _sums(dims, fat, lng, b, parity):
    """S of every component: [nrhs][Vh][3] complex, real and imaginary parts apart."""
    vh = b.shape[1]
    nx, ny, nz, nt = dims
    t, z, y, x = np.meshgrid(np.arange(nt), np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    eo = ((x + nx * (y + ny * (z + nz * t))) // 2 + vh * ((x + y + z + t) % 2)).reshape(nt, nz, ny, nx)
    here = eo.reshape(-1)
    full = np.zeros((b.shape[0], 2 * vh, 3), dtype=np.complex128)
    full[:, (1 - parity) * vh:(2 - parity) * vh] = np.abs(b.real) + 1j * np.abs(b.imag)
    out = np.zeros_like(full)
    for links, k in ((fat, 1), (lng, 3)):
        for mu in range(4):
            fwd, bwd = np.roll(eo, -k, 3 - mu).reshape(-1), np.roll(eo, k, 3 - mu).reshape(-1)
            for m, nb in ((links[mu][here], fwd), (links[mu][bwd].transpose(0, 2, 1), bwd)):
                re, im, v = np.abs(m.real), np.abs(m.imag), full[:, nb]
                mul = lambda a, w: np.einsum("sij,rsj->rsi", a, w)  # noqa: E731
                out[:, here] += mul(re, v.real) + mul(im, v.imag) + 1j * (mul(re, v.imag) + mul(im, v.real))
    return out[:, parity * vh:(parity + 1) * vh]


@pytest.mark.parametrize("vectors", ["plain", "colours", "parts", "one colour", "steep", "decay"])
@pytest.mark.parametrize("links", ["plain", "near unity", "unit", "small entries", "scales"])
@pytest.mark.parametrize("dims,nrhs,shape", SHAPES)
def test_components(dims, nrhs, shape, links, vectors):
    fat, lng = _links(dims, links)
    b = _vectors(dims, nrhs, vectors)
    ctx = hisq.Context(dims, torch.from_numpy(fat).cuda(), torch.from_numpy(lng).cuda(), precs=(hisq.F64,))
    ctx.tune_set(hisq.F64, hisq.F64, nrhs, *shape)
    for parity in (0, 1):
        out = torch.full(b.shape, float("nan"), dtype=torch.complex128, device="cuda")
        ctx.dslash(parity, torch.from_numpy(b).cuda(), out)
        err = out.cpu().numpy() - np.stack([oracle.dslash(dims, fat, lng, b[r], parity) for r in range(nrhs)])
        S = _sums(dims, fat, lng, b, parity)
        assert (np.abs(err.real) <= 200 * U * S.real).all()
        assert (np.abs(err.imag) <= 200 * U * S.imag).all()


@pytest.mark.parametrize("links", ["plain", "small entries"])
def test_point_source_gives_the_links(links):
    # one column of one link at each of the 16 neighbours: nothing to add, so the links themselves, bit for bit
    dims = (6, 8, 4, 6)
    fat, lng = _links(dims, links)
    ctx = hisq.Context(dims, torch.from_numpy(fat).cuda(), torch.from_numpy(lng).cuda(), precs=(hisq.F64,))
    vh = int(np.prod(dims)) // 2
    for site in (0, 17, vh - 1):
        for colour in range(3):
            b = np.zeros((vh, 3), dtype=np.complex128)
            b[site, colour] = 1.0
            out = torch.empty(vh, 3, dtype=torch.complex128, device="cuda")
            ctx.dslash(1, torch.from_numpy(b).cuda(), out)
            got, want = out.cpu().numpy(), oracle.dslash(dims, fat, lng, b, 1)
            assert (got == want).all()
