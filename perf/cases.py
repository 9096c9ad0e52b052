"""Performance cases of the HISQ library: what a program that uses it has it do.

A program holds one lattice's links as a `hisq.Context` (plan and weights of this library),
calls the operator (`dslash`, `mdagm`) or a solver (`cg`, `multishift_cg`) on device vectors,
trains and applies the learned preconditioner (`Net`), and once per gauge configuration builds
the smeared links (`smear_links`).  Sizes run from the smallest lattice of the tests (8^4) to
the repository's batched workload (64^3 x 16), with extents that divide into nothing among
them.

Links are seeded random SU(3) matrices at the workloads' distance from unity (fat = U, long =
-1/24 U U U, the workload recipe), sources are Gaussian; both are drawn on the GPU.  Results
of a reduced precision are handed on in the type whose precision they carry (the conversion
from the library's complex128 buffers loses nothing): complex64 for the FP32-vector operators,
bfloat16 for the network.
"""
import math

import torch

from paper_2306_01098_gb300 import hisq

PREC = {"f64": hisq.F64, "f64x": hisq.F64X, "f32": hisq.F32, "f16": hisq.F16}
LINK_BYTES = {"f64": 144, "f64x": 144, "f32": 72, "f16": 36}
VEC_BYTES = {"f64": 48, "f64x": 48, "f32": 24, "f16": 24}
FLOPS_PER_SITE = 1146.0  # one Dslash, one right-hand side


# ---------------------------------------------------------------- the cases

def listed():
    op = dict(nreal=18, nrhs=1, mass=0.01, eps=0.5)
    cg = dict(op, tol=1e-10)
    return [
        # one operator call on the smallest lattice of the tests: latency and launches
        dict(name="dslash f64 8^4", kind="dslash", dims="8x8x8x8", prec="f64", **op),
        # the FP64 normal operator of the benchmark lattice (residuals, plain CG)
        dict(name="mdagm f64 32^3x8", kind="mdagm", dims="32x32x32x8", prec="f64", **op),
        # float-pair normal operator, three colour sources, ragged extents
        dict(op, name="mdagm f64x 18x22x14x10 x3", kind="mdagm", dims="18x22x14x10", prec="f64x", nrhs=3),
        # the operator in single precision on the large workload, links streaming from memory
        dict(name="dslash f32 64^3x16", kind="dslash", dims="64x64x64x16", prec="f32", **op),
        # many right-hand sides share the links
        dict(op, name="dslash f32 48^3x12 x8", kind="dslash", dims="48x48x48x12", prec="f32", nrhs=8),
        # the benchmark: mixed-precision CG to 1e-10, 16-bit links
        dict(cg, name="cg f16 32^3x8", kind="cg", dims="32x32x32x8", prec="f16"),
        # CG with the library's default options (FP64 throughout) on a ragged small lattice
        dict(cg, name="cg f64 12x16x20x10", kind="cg", dims="12x16x20x10", prec="f64", mass=0.05),
        # propagator production: eight sources in one mixed-precision solve
        dict(cg, name="cg f16 32^3x16 x8", kind="cg", dims="32x32x32x16", prec="f16", nrhs=8),
        # rational-function inversions: 14 log-spaced shifts
        dict(cg, name="multishift f32 32^3x8", kind="multishift", dims="32x32x32x8", prec="f32", nshift=14),
        # the learned preconditioner inside flexible CG
        dict(op, name="net apply 32^3x8", kind="net_apply", dims="32x32x32x8", prec="f16"),
        # one training sample of it: forward, backward, loss and weight gradient
        dict(op, name="net grad 16^3x8", kind="net_grad", dims="16x16x16x8", prec="f16"),
        # links of one gauge configuration: two levels of smearing and the projection
        dict(name="smear 24^3x8", kind="smear", dims="24x24x24x8", eps=0.5),
    ]


def _extents(rng, lo, hi):
    """Four even extents >= 4 with a volume spread over the logarithm of [lo, hi] sites."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        d = []
        for left in (4, 3, 2):
            side = v ** (1.0 / left) * math.exp(rng.uniform(-0.3, 0.3))
            d.append(max(4, 2 * round(side / 2)))
            v /= d[-1]
        d.append(max(4, 2 * round(v / 2)))
        if max(d) <= 96 and d[0] * d[1] * d[2] * d[3] <= hi:
            return "x".join(map(str, d))


def draw(rng):
    kind = rng.choice(["dslash", "dslash", "dslash", "mdagm", "mdagm", "cg", "cg", "multishift", "net_apply",
                       "net_grad", "smear"])
    eps = rng.choice([0.3, 0.5])
    if kind == "smear":
        return dict(kind=kind, dims=_extents(rng, 256, 24 ** 3 * 8), eps=eps)
    c = dict(kind=kind, nreal=18, nrhs=1, mass=0.01, eps=eps)
    if kind in ("dslash", "mdagm"):
        c["prec"] = rng.choice(["f64", "f64", "f64x", "f32", "f16"])
        c["nrhs"] = rng.choice([1, 1, 2, 3, 4, 8])
        if c["prec"] != "f64x" and rng.random() < 0.2:
            c["nreal"] = 12
        c["dims"] = _extents(rng, 4096, 64 ** 3 * 16 // c["nrhs"])
    elif kind == "cg":
        c.update(prec=rng.choice(["f64", "f64x", "f32", "f16"]), nrhs=rng.choice([1, 1, 2, 3, 8]), tol=1e-10)
        c["mass"] = rng.choice([0.02, 0.05, 0.1])
        c["dims"] = _extents(rng, 4096, 32 ** 3 * 16 // max(1, c["nrhs"] // 2))
    elif kind == "multishift":
        c.update(prec=rng.choice(["f64", "f32", "f16"]), nshift=rng.randint(3, 14), tol=1e-10, mass=0.02)
        c["dims"] = _extents(rng, 4096, 32 ** 3 * 8)
    else:
        c["prec"] = rng.choice(["f16", "f32"])
        c["dims"] = _extents(rng, 4096, 32 ** 3 * 8 if kind == "net_apply" else 16 ** 3 * 16)
    return c


# ---------------------------------------------------------------- inputs

def _dims(case):
    return tuple(int(n) for n in case["dims"].split("x"))


def _volume(dims):
    return dims[0] * dims[1] * dims[2] * dims[3]


def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + stream)


def _mul(a, b):
    """Products of 3x3 matrices, elementwise over the leading axes."""
    return sum(a[..., :, j, None] * b[..., j, None, :] for j in range(3))


def _thin(dims, eps, seed):
    """Random SU(3) links, lexicographic [4][Nt][Nz][Ny][Nx][3][3] complex128: 1 + i eps H + (i eps H)^2 / 2
    with Gaussian traceless hermitian H, made unitary by Gram-Schmidt."""
    nx, ny, nz, nt = dims
    g = _gen(seed, 1)
    out = torch.empty(4, nt, nz, ny, nx, 3, 3, dtype=torch.complex128, device="cuda")
    for mu in range(4):
        h = 0.5 * torch.randn(8, _volume(dims), dtype=torch.float64, device="cuda", generator=g)
        m = torch.zeros(_volume(dims), 3, 3, dtype=torch.complex128, device="cuda")
        for i, (a, b) in enumerate(((0, 1), (0, 2), (1, 2))):
            z = torch.complex(h[2 * i], -h[2 * i + 1])
            m[:, a, b], m[:, b, a] = z, z.conj()
        m[:, 0, 0], m[:, 1, 1], m[:, 2, 2] = h[6] + h[7] / 3 ** 0.5, h[7] / 3 ** 0.5 - h[6], -2 * h[7] / 3 ** 0.5
        m = 1j * eps * m
        m = torch.eye(3, dtype=m.dtype, device="cuda") + m + 0.5 * _mul(m, m)
        r0 = m[:, 0] / m[:, 0].abs().square().sum(-1, keepdim=True).sqrt()
        r1 = m[:, 1] - (r0.conj() * m[:, 1]).sum(-1, keepdim=True) * r0
        r1 = r1 / r1.abs().square().sum(-1, keepdim=True).sqrt()
        r2 = torch.stack([(r0[:, (k + 1) % 3] * r1[:, (k + 2) % 3] - r0[:, (k + 2) % 3] * r1[:, (k + 1) % 3]).conj()
                          for k in range(3)], -1)
        out[mu] = torch.stack([r0, r1, r2], 1).reshape(nt, nz, ny, nx, 3, 3)
    return out


def _lex_of_eo(dims):
    """Lexicographic site of every canonical even-odd slot (even sites first, both in lexicographic order)."""
    nx, ny, nz, nt = dims
    t, z, y, x = torch.meshgrid(*(torch.arange(n, device="cuda") for n in (nt, nz, ny, nx)), indexing="ij")
    par = ((x + y + z + t) % 2).reshape(-1)
    return torch.cat([torch.nonzero(par == 0)[:, 0], torch.nonzero(par == 1)[:, 0]])


def _canonical(dims, lex):
    """[4][lattice][3][3] in lexicographic order -> [4][V][3][3] in canonical order."""
    return lex.reshape(4, -1, 3, 3)[:, _lex_of_eo(dims)].contiguous()


def _links(dims, eps, seed):
    """(fat, long) of the workload recipe in canonical order."""
    u = _thin(dims, eps, seed)
    lng = torch.empty_like(u)
    for mu in range(4):
        hop = lambda k: u[mu].roll(-k, 3 - mu)  # noqa: E731
        lng[mu] = -1.0 / 24.0 * _mul(_mul(u[mu], hop(1)), hop(2))
    return _canonical(dims, u), _canonical(dims, lng)


def _source(dims, nrhs, seed, stream=2):
    z = torch.randn(nrhs, _volume(dims) // 2, 3, 2, dtype=torch.float64, device="cuda", generator=_gen(seed, stream))
    return torch.view_as_complex(z)


def _shifts(n):
    return [math.exp(math.log(1e-5) * (1 - i / (n - 1))) for i in range(n)]


def _net_weights(case, seed):
    """Weights of a network of the default shape (1 -> 8 -> 8 -> 8 -> 1 channels, 17 taps): the identity path
    plus random hops, as training leaves them."""
    g = _gen(seed, 3)
    ws = []
    for cout, cin in ((8, 1), (8, 8), (8, 8), (1, 8)):
        w = torch.view_as_complex(0.05 * torch.randn(17, cout, cin, 2, dtype=torch.float64, device="cuda", generator=g))
        w[0] += torch.eye(cout, cin, dtype=w.dtype, device="cuda")
        ws.append(w)
    return ws


def prepare(case, seed):
    dims, kind = _dims(case), case["kind"]
    if kind == "smear":
        return dict(kind=kind, dims=dims, thin=_canonical(dims, _thin(dims, case["eps"], seed)))
    prec = PREC[case["prec"]]
    precs = (prec,) if kind in ("dslash", "mdagm", "net_apply", "net_grad") else tuple(sorted({prec, hisq.F64}))
    fat, lng = _links(dims, case["eps"], seed)
    ctx = hisq.Context(dims, fat, lng, precs=precs, compression={prec: case["nreal"]})
    b = _source(dims, case["nrhs"], seed)
    s = dict(kind=kind, ctx=ctx, prec=prec, mass=case["mass"], b=b)
    if kind == "multishift":
        s["sigma"] = _shifts(case["nshift"])
        s["x"] = [torch.empty_like(b) for _ in s["sigma"]]
    else:
        s["x"] = torch.empty_like(b)
    if kind in ("cg", "multishift"):
        s["opts"] = ctx.solve_opts(tol=case["tol"], prec_sloppy=prec)
    if kind in ("net_apply", "net_grad"):
        s["net"] = hisq.Net(ctx, link_prec=prec)
        s["net"].set_weights(torch.cat([w.reshape(-1) for w in _net_weights(case, seed)]).cpu().numpy())
        if kind == "net_grad":
            s["x"].copy_(_source(dims, 1, seed, stream=4))
    return s


# ---------------------------------------------------------------- one pass

def _kept(prec, x):
    return x.to(torch.complex64) if prec in (hisq.F32, hisq.F16) else x


def run(state):
    kind = state["kind"]
    if kind == "smear":
        return hisq.smear_links(state["dims"], state["thin"])
    ctx, b, x = state["ctx"], state["b"], state["x"]
    if kind == "dslash":
        ctx.dslash(1, b, x, state["prec"])
        return _kept(state["prec"], x)
    if kind == "mdagm":
        ctx.mdagm(state["mass"], b, x, state["prec"])
        return _kept(state["prec"], x)
    if kind == "cg":
        ctx.cg(state["mass"], b, x, opts=state["opts"])
        return x
    if kind == "multishift":
        ctx.multishift_cg(state["mass"], state["sigma"], b, x, opts=state["opts"])
        return x
    if kind == "net_apply":
        state["net"].apply(b, x)
        return torch.view_as_real(x).to(torch.bfloat16)
    return state["net"].loss_grad(b, x)


# ---------------------------------------------------------------- work and exact results

# operator applications of a solve to 1e-10 at the masses of the cases (measured 200 at 0.01,
# falling slowly with the mass): what any conjugate gradient of this accuracy needs
_APPLICATIONS = 200


def work(case):
    dims, kind = _dims(case), case["kind"]
    vol = _volume(dims)
    vh = vol // 2
    if kind == "smear":
        # per link and level: 3-, 5- and 7-link staples built from each other (60 matrix
        # products of 198 flops), the second level's Lepage paths (12 more), projection and Naik
        return dict(bytes=3.0 * 4 * vol * 144, flops=4.0 * vol * 198 * (2 * 60 + 12 + 12))
    if kind in ("net_apply", "net_grad"):
        # transports of every channel (72 flops per matrix-vector product) and channel mixing
        per = 0.0
        for (cin, cout), sites in zip(((1, 8), (8, 8), (8, 8), (8, 1)), (vol, vol, vol, vh)):
            per += sites * (16 * 72.0 * min(cin, cout) + 17 * 24.0 * cin * cout)
        passes = 1 if kind == "net_apply" else 3
        return dict(bytes=32.0 * vh * LINK_BYTES[case["prec"]] / 2 + 96.0 * vh, flops=per * passes)
    links = 16.0 * vh * LINK_BYTES[case["prec"]] * case["nreal"] / 18
    vecs = 2.0 * 48 * vh * case["nrhs"]
    flops = FLOPS_PER_SITE * vh * case["nrhs"]
    if kind == "dslash":
        return dict(bytes=links + vecs, flops=flops)
    if kind == "mdagm":
        return dict(bytes=links + vecs, flops=2 * flops)
    out = vecs if kind == "cg" else 48.0 * vh * (1 + case["nshift"])
    return dict(bytes=links + 16.0 * vh * 144 * (case["prec"] != "f64") + out, flops=2 * flops * _APPLICATIONS)


class _Stencil:
    """The operator in plain torch, complex128: phases and the antiperiodic time boundary folded into
    the links, neighbours by index."""

    def __init__(self, dims, fat, lng):
        nx, ny, nz, nt = dims
        vol = _volume(dims)
        self.vh = vol // 2
        lex = _lex_of_eo(dims)
        eo = torch.empty_like(lex)
        eo[lex] = torch.arange(vol, device="cuda")
        grid = eo.reshape(nt, nz, ny, nx)
        x, y, z, t = lex % nx, lex // nx % ny, lex // (nx * ny) % nz, lex // (nx * ny * nz)
        eta = [torch.zeros_like(x), x, x + y, x + y + z]
        self.taps = []  # (links by canonical site of the hop's origin, hop length, direction)
        for links, k in ((fat, 1), (lng, 3)):
            for mu in range(4):
                neg = eta[mu] % 2
                if mu == 3:
                    neg = neg + (t + k >= nt)
                sign = (1 - 2 * (neg % 2)).to(torch.float64)
                fwd = grid.roll(-k, 3 - mu).reshape(-1)[lex]
                bwd = grid.roll(k, 3 - mu).reshape(-1)[lex]
                self.taps.append((links[mu] * sign[:, None, None], fwd, bwd))

    def hops(self, v, sites):
        """Both hops of every tap at canonical sites `sites` (a slice) of the full-lattice field v [..., V, 3]."""
        for u, fwd, bwd in self.taps:
            f, w = fwd[sites], bwd[sites]
            yield torch.einsum("vij,...vj->...vi", u[sites], v[..., f, :])
            yield torch.einsum("vji,...vj->...vi", u[w].conj(), v[..., w, :])

    def dslash(self, parity, v):
        """D_{parity, 1 - parity} of a half-lattice field [nrhs][Vh][3]."""
        full = torch.zeros(*v.shape[:-2], 2 * self.vh, 3, dtype=v.dtype, device=v.device)
        here, there = slice(parity * self.vh, (parity + 1) * self.vh), slice((1 - parity) * self.vh, (2 - parity) * self.vh)
        full[..., there, :] = v
        out = torch.zeros_like(v)
        for i, h in enumerate(self.hops(full, here)):
            out += h if i % 2 == 0 else -h
        return out

    def mdagm(self, m, v):
        return 4 * m * m * v - self.dslash(0, self.dslash(1, v))


def _dot(a, b):
    return (a.conj() * b).real.sum((-2, -1), keepdim=True)


def _solve(st, m, b, sigma):
    """(A + sigma_s) x_s = b for all shifts by multi-shift CG on the unshifted system, to 1e-13."""
    x = [torch.zeros_like(b) for _ in sigma]
    ps = [b.clone() for _ in sigma]
    base = min(sigma)
    zp, z = [torch.ones_like(_dot(b, b)) for _ in sigma], [torch.ones_like(_dot(b, b)) for _ in sigma]
    r, p = b.clone(), b.clone()
    rr = bb = _dot(b, b)
    a_old, beta = torch.ones_like(rr), torch.zeros_like(rr)
    for _ in range(3000):
        ap = st.mdagm(m, p) + base * p
        a = rr / _dot(p, ap)
        for i, s in enumerate(sigma):
            den = a * beta * (zp[i] - z[i]) + zp[i] * a_old * (1 + (s - base) * a)
            zn = z[i] * zp[i] * a_old / den
            x[i] += a * zn / z[i] * ps[i]
            zp[i], z[i] = z[i], zn
        r = r - a * ap
        new = _dot(r, r)
        a_old, beta = a, new / rr
        rr = new
        p = r + beta * p
        for i in range(len(sigma)):
            ps[i] = z[i] * r + beta * (z[i] / zp[i]) ** 2 * ps[i]
        if float((rr / bb).max()) < 1e-26:
            break
    return x


def _smear_exact(dims, thin, eps_naik=0.0):
    """HISQ links in plain torch (two levels, polar projection between them)."""
    vol = _volume(dims)
    nx, ny, nz, nt = dims
    lex_of = _lex_of_eo(dims)
    u = torch.empty_like(thin)
    u[:, lex_of] = thin
    u = u.reshape(4, nt, nz, ny, nx, 3, 3)
    dag = lambda a: a.conj().transpose(-1, -2)  # noqa: E731
    at = lambda a, d, k: a.roll(-k, 3 - d)  # noqa: E731

    def staple(g, f, mu, nu):
        up = _mul(_mul(g[nu], at(f, nu, 1)), dag(at(g[nu], mu, 1)))
        down = _mul(_mul(dag(g[nu]), f), at(g[nu], mu, 1))
        return up + at(down, nu, -1)

    def level(g, c1, cl):
        out = torch.empty_like(g)
        for mu in range(4):
            dirs = [d for d in range(4) if d != mu]
            s3 = {nu: staple(g, g[mu], mu, nu) for nu in dirs}
            acc = c1 * g[mu] + sum(s3.values()) / 16
            for rho in dirs:
                others = [d for d in dirs if d != rho]
                acc = acc + staple(g, s3[others[0]] + s3[others[1]], mu, rho) / 64
                inner = staple(g, s3[others[0]], mu, others[1]) + staple(g, s3[others[1]], mu, others[0])
                acc = acc + staple(g, inner, mu, rho) / 384
                if cl:
                    two = _mul(g[rho], at(g[rho], rho, 1))
                    up = _mul(_mul(two, at(g[mu], rho, 2)), dag(at(two, mu, 1)))
                    down = _mul(_mul(dag(two), g[mu]), at(two, mu, 1))
                    acc = acc + cl * (up + at(down, rho, -2))
            out[mu] = acc
        return out

    v = level(u, 0.125, 0.0)
    h = _mul(dag(v), v)
    lam, q = torch.linalg.eigh(h.reshape(-1, 3, 3).cpu())
    lam, q = lam.cuda(), q.cuda()
    w = _mul(v, (_mul(q * (lam ** -0.5)[:, None, :].to(q.dtype), dag(q))).reshape(v.shape))
    fat = level(w, 1.0, -0.125)
    lng = torch.stack([(-1.0 / 24 + eps_naik / 8) * _mul(_mul(w[mu], at(w[mu], mu, 1)), at(w[mu], mu, 2))
                       for mu in range(4)])
    return tuple(a.reshape(4, vol, 3, 3)[:, lex_of].contiguous() for a in (fat, lng))


def _net_exact(st, ws, b):
    """The network on the full lattice: source on even sites, output read on even sites."""
    act = torch.zeros(1, 2 * st.vh, 3, dtype=torch.complex128, device="cuda")
    act[:, :st.vh] = b
    for w in ws:
        out = torch.einsum("oc,cvi->ovi", w[0], act)
        for n, h in enumerate(st.hops(act, slice(0, 2 * st.vh))):
            out = out + torch.einsum("oc,cvi->ovi", w[1 + n], h)
        act = out
    return act[:, :st.vh]


def exact(case, seed):
    dims, kind = _dims(case), case["kind"]
    if kind == "smear":
        return _smear_exact(dims, _canonical(dims, _thin(dims, case["eps"], seed)))
    # a solve of several right-hand sides on a large lattice takes plain torch too long
    if kind in ("cg", "multishift") and _volume(dims) * case["nrhs"] > 32 ** 3 * 8:
        return None
    st = _Stencil(dims, *_links(dims, case["eps"], seed))
    b = _source(dims, case["nrhs"], seed)
    if kind == "dslash":
        return st.dslash(1, b)
    if kind == "mdagm":
        return st.mdagm(case["mass"], b)
    if kind == "cg":
        return _solve(st, case["mass"], b, [0.0])[0]
    if kind == "multishift":
        return _solve(st, case["mass"], b, _shifts(case["nshift"]))
    ws = _net_weights(case, seed)
    if kind == "net_apply":
        return torch.view_as_real(_net_exact(st, ws, b).reshape(b.shape))
    x = _source(dims, 1, seed, stream=4)
    ws = [w.requires_grad_() for w in ws]
    loss = (_net_exact(st, ws, b) - x).abs().square().sum() / x.abs().square().sum()
    # torch's gradient of a real loss is dL/dRe + i dL/dIm, the library's convention
    grads = torch.autograd.grad(loss, ws)
    return float(loss), torch.cat([g.reshape(-1) for g in grads]).cpu().numpy()
