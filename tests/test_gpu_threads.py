"""Threads, each with a context and a stream of its own, launching the same kernel with blocks of
different sizes (and so with different amounts of shared memory)."""
import threading

import pytest
import torch

from hisq_inputs import fields

hisq = pytest.importorskip("paper_2306_01098_gb300.hisq")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,nrhs,n_inner", [("F64", 4, 4), ("F64", 1, 1), ("F32", 8, 8)])
def test_block_sizes_of_threads(prec, nrhs, n_inner):
    dims, p = (8, 8, 8, 8), getattr(hisq, prec)
    fat, lng = (a.cuda() for a in fields.recipe_links(dims, 0.5, 1700))
    b = torch.stack([fields.gaussian_source(dims, 2800 + r)[0] for r in range(nrhs)]).cuda()
    ctxs = []
    for block in (64, 256, 64, 256):
        c = hisq.Context(dims, fat, lng, precs=(p,))
        c.tune_set(p, p, nrhs, n_inner, 1)
        c.tune_set_block(p, p, nrhs, block)
        ctxs.append(c)
    want = torch.empty_like(b)
    ctxs[0].dslash(1, b, want, p)
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(len(ctxs))

    def work(ctx):
        try:
            st = torch.cuda.Stream()
            out = torch.empty_like(b)
            start.wait(30)
            for _ in range(20000):
                ctx.dslash(1, b, out, p, stream=st.cuda_stream)
            st.synchronize()
            assert torch.equal(out, want)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(c,)) for c in ctxs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
