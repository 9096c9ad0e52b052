"""The stored form of FP64 links (csrc/fixed.cuh), on the host: the doubles come back bit for bit whatever
they are, zeros stay zeros, and the limbs that the kernels multiply are the doubles cut to one unit."""
import os
import subprocess

import numpy as np
import pytest

build = pytest.importorskip("paper_2306_01098_gb300.build")

SOURCE = r"""
#include <cstdio>
#include "fixed.cuh"
int main()
{
    double d[18], back[18];
    while (fread(d, 8, 18, stdin) == 18) {
        uint32_t w[36];
        uint64_t rest;
        hisq::fx_encode_link(d, w, rest);
        hisq::fx_decode_link(w, rest, back);
        uint32_t f;
        const int32_t code = (int32_t)hisq::fx_take_code(w, f);
        fwrite(back, 8, 18, stdout);
        fwrite(w, 4, 36, stdout);
        fwrite(&code, 4, 1, stdout);
        fwrite(&f, 4, 1, stdout);
    }
}
"""


@pytest.fixture(scope="module")
def roundtrip(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    src, exe = d / "links.cu", d / "links"
    src.write_text(SOURCE)
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    subprocess.run([nvcc, *build.ARCH, *build.FLAGS, str(src), "-o", str(exe)], check=True, capture_output=True)

    def run(links):
        out = subprocess.run([str(exe)], input=np.ascontiguousarray(links, dtype=np.float64).tobytes(), check=True,
                             capture_output=True).stdout
        rec = np.frombuffer(out, dtype=[("back", "<f8", 18), ("w", "<i4", (18, 2)), ("code", "<i4"), ("f", "<i4")])
        assert len(rec) == len(links)
        return rec

    return run


def _links(kind, n=4000):
    rng = np.random.default_rng(17)
    d = rng.normal(size=(n, 18))
    if kind == "spread":  # reals down to 2^-40 of the largest
        d *= np.exp2(-rng.integers(0, 41, d.shape) * (rng.random(d.shape) < 0.1))
    if kind == "sparse":
        d[rng.random(d.shape) < 0.5] = 0.0
    if kind == "binade edges":
        d = np.exp2(rng.integers(-30, 1, d.shape)) * (1 - rng.integers(0, 2, d.shape) * 2.0 ** -53) * rng.choice([-1, 1], d.shape)
    if kind == "any bits":
        d = rng.integers(0, 2 ** 64, d.shape, dtype=np.uint64).view(np.float64)
    if kind == "special":
        pick = rng.random(d.shape)
        for v, x in enumerate((np.inf, -np.inf, np.nan, 5e-324, -3e-310, 0.0, -0.0, 1e-300, 1e300)):
            d[(pick > 0.02 * v) & (pick < 0.02 * (v + 1))] = x
    if kind == "named":
        d = np.zeros((6, 18))
        d[0, [0, 8, 16]] = 1.0
        d[1, :] = 1.0 / 3.0
        d[1, 2] = 1e-19 / 3
        d[2, :2] = 1.0, 1.0 / 3000.0
        d[3, 5] = np.inf
        d[4, :] = 1e-300
    return d


@pytest.mark.parametrize("kind", ["plain", "spread", "sparse", "binade edges", "any bits", "special", "named"])
def test_doubles_come_back(roundtrip, kind):
    d = _links(kind)
    rec = roundtrip(d)
    want, got = d.view(np.uint64).copy(), np.ascontiguousarray(rec["back"]).view(np.uint64)
    want[(d == 0) & (rec["code"] != 0xfff)[:, None]] = 0  # the sign of a zero is not kept in fixed point
    assert (got == want).all()
    fx = rec["code"] != 0xfff
    if kind in ("plain", "spread", "sparse", "binade edges"):
        assert fx.mean() > 0.9 or kind == "binade edges"
    # value of the limbs: cut towards zero by less than a unit, so exactly zero where the link is
    x = rec["w"][:, :, 1].astype(object) * 2 ** 32 + rec["w"][:, :, 0].astype(object)
    for i in np.nonzero(fx)[0][:500]:
        for k in range(18):
            unit = int(rec["code"][i]) - 1023 - 59
            exact = abs(float(d[i, k]))
            num, den = exact.as_integer_ratio()
            cut = num * 2 ** -unit // den if unit < 0 else num // (den * 2 ** unit)
            assert abs(int(x[i, k])) == cut and (cut == 0 or (int(x[i, k]) < 0) == (d[i, k] < 0))
    assert (np.abs(rec["w"][fx][:, :, 1]) <= 2 ** 28).all()


@pytest.mark.parametrize("kind", ["plain", "sparse", "spread", "binade edges", "named"])
def test_balance_of_a_link(roundtrip, kind):
    # f 2^e is no more than any row or column sum of |reals|, and as large as that allows (up to the cut)
    d = _links(kind)
    rec = roundtrip(d)
    fx = (rec["code"] != 0xfff) & (rec["code"] != 0)
    a = np.abs(d).reshape(-1, 3, 3, 2).sum(-1)
    least = np.minimum(a.sum(1).min(1), a.sum(2).min(1))[fx] / np.exp2(rec["code"][fx] - 1023.0)
    f = rec["f"][fx]
    assert (f <= least).all() and (f >= np.minimum(3, np.floor(least - 1e-7))).all()
    unitary = np.linalg.qr(np.random.default_rng(3).normal(size=(200, 3, 3, 2)).view(np.complex128)[..., 0])[0] * 0.3
    assert (roundtrip(unitary.reshape(200, 9).view(np.float64))["f"] >= 1).all()
