"""The FP64 Dslash with 18-real links, computed in fixed point, where that can go wrong: vectors and
links of very different magnitudes, zeros, and values that have to be left to FP64.

Tolerance per site: 200 u S with u = 2^-53 and S = sum over the hops of |U|_F |v|.  The oracle's sum
of 48 complex products errs by at most about 100 u S; the fixed-point sum by 96 products of
2^-57 + 2^-58 + 2 2^-61 of max |U| max |v| each, below 10 u S, and one rounding.
"""
import numpy as np
import pytest
import torch

import oracle
from hisq_inputs import fields

hisq = pytest.importorskip("paper_2306_01098_gb300.hisq")

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def _links(dims, kind):
    fat, lng = (a.numpy().copy() for a in fields.recipe_links(dims, 0.5, 1300))
    rng = np.random.default_rng(5)
    if kind == "ranges":  # every link at its own scale, some far below the others, some zero
        for a in (fat, lng):
            a *= np.exp2(rng.integers(-40, 41, a.shape[:2]))[..., None, None]
            a[rng.random(a.shape[:2]) < 0.05] = 0.0
    if kind == "no long":
        lng[:] = 0.0
    if kind == "tiny":  # links below the format's range: kept as doubles
        fat[rng.random(fat.shape[:2]) < 0.02] *= 2.0 ** -1000
    return fat, lng


def _vectors(dims, nrhs, kind):
    b = np.stack([fields.gaussian_source(dims, 2300 + r)[0].numpy() for r in range(nrhs)])
    rng = np.random.default_rng(6)
    if kind == "ranges":
        b *= np.exp2(rng.integers(-60, 61, b.shape[:2]))[..., None]
        b[rng.random(b.shape) < 0.2] *= 2.0 ** -70  # components far below their site's largest
        b[rng.random(b.shape[:2]) < 0.1] = 0.0
    if kind == "point":
        keep = b[:, 7].copy()
        b[:] = 0.0
        b[:, 7] = keep
    if kind == "special":
        b[:, 3, 1] = np.inf
        b[:, 11, 0] = np.nan
        b[:, 20] *= 1e-300
        b[:, 31] = 3e-310
        b[:, 40] *= 1e300
        b[:, 50, 2] = -0.0
    return b


def _hop_sizes(dims, fat, lng, b, parity):
    """S of every output site and right-hand side: the oracle applied to norms, links as |U|_F times
    a matrix that adds up without signs."""
    vh = b.shape[1]
    nx, ny, nz, nt = dims
    t, z, y, x = np.meshgrid(np.arange(nt), np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    eo = ((x + nx * (y + ny * (z + nz * t))) // 2 + vh * ((x + y + z + t) % 2)).reshape(nt, nz, ny, nx)
    full = np.zeros((b.shape[0], 2 * vh))
    full[:, (1 - parity) * vh:(2 - parity) * vh] = np.sqrt((np.abs(b) ** 2).sum(-1))
    out = np.zeros((b.shape[0], 2 * vh))
    for links, k in ((fat, 1), (lng, 3)):
        norm = np.sqrt((np.abs(links) ** 2).sum((-1, -2)))
        for mu in range(4):
            fwd = np.roll(eo, -k, 3 - mu).reshape(-1)
            bwd = np.roll(eo, k, 3 - mu).reshape(-1)
            here = eo.reshape(-1)
            out[:, here] += norm[mu][here] * full[:, fwd] + norm[mu][bwd] * full[:, bwd]
    return out[:, parity * vh:(parity + 1) * vh]


@pytest.mark.parametrize("links,vectors", [("plain", "plain"), ("ranges", "ranges"), ("no long", "point"),
                                           ("plain", "special"), ("tiny", "ranges")])
@pytest.mark.parametrize("dims,nrhs,shape", [((4, 6, 8, 10), 1, (1, 1)), ((8, 8, 8, 8), 1, (1, 4)),
                                             ((10, 4, 6, 4), 3, (1, 2)), ((6, 4, 4, 4), 4, (4, 1)),
                                             ((8, 4, 4, 6), 2, (2, 4))])
def test_fixed_point_dslash(dims, nrhs, shape, links, vectors):
    fat, lng = _links(dims, links)
    b = _vectors(dims, nrhs, vectors)
    ctx = hisq.Context(dims, torch.from_numpy(fat).cuda(), torch.from_numpy(lng).cuda(), precs=(hisq.F64,))
    ctx.tune_set(hisq.F64, hisq.F64, nrhs, shape[0], shape[1])
    for parity in (0, 1):
        out = torch.full(b.shape, float("nan"), dtype=torch.complex128, device="cuda")
        ctx.dslash(parity, torch.from_numpy(b).cuda(), out)
        got = out.cpu().numpy()
        with np.errstate(all="ignore"):
            want = np.stack([oracle.dslash(dims, fat, lng, b[r], parity) for r in range(nrhs)])
            S = _hop_sizes(dims, fat, lng, b, parity)
            finite = np.isfinite(want).all(-1)
            assert (np.isfinite(got).all(-1) == finite).all()
            err = np.sqrt((np.abs(got - want) ** 2).sum(-1))
        # (the smallest normal number covers sums that underflow)
        assert (err[finite] <= 200 * U * S[finite] + 2.3e-308).all()
