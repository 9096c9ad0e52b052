// smear.cu -- HISQ fat and long links from thin links: two levels of smearing with a U(3)
// projection between them (Sec. 3.1).
//
// First level:  V = c1 U + c3 S3 + c5 S5 + c7 S7       (c1 1/8, c3 1/16, c5 1/64, c7 1/384)
// projection:   W = V (V^+ V)^(-1/2)                    (unitary polar factor of V)
// second level: X = c1 W + c3 S3 + c5 S5 + c7 S7 + cL L (c1 1, the same staples, cL -1/8)
// Naik:         N_mu(x) = cN W_mu(x) W_mu(x+mu) W_mu(x+2mu),   cN = -1/24 + eps/8
// with the staples of a field F_mu built from the links of the level (U, then W):
//   stap_nu[F]_mu(x) = U_nu(x) F_mu(x+nu) U_nu(x+mu)^+ + U_nu(x-nu)^+ F_mu(x-nu) U_nu(x-nu+mu)
//   S3 = sum_nu stap_nu[F];  S5 = sum_rho stap_rho[sum_{nu != rho} stap_nu[F]];
//   S7 = sum_sig stap_sig[sum_{rho != sig} stap_rho[sum_{nu != rho, sig} stap_nu[F]]];
//   L  = the staples whose detour is two steps along nu
// (all directions different from mu).  Everything is FP64, the products of three matrices in 60-bit
// fixed point (fixed.cuh): the FP64 pipe, two operations a clock and SM, would bound them.
// The projection uses the scaled Newton iteration for the polar decomposition,
//   X <- (g X + X^{-+} / g) / 2,  g = (|X^-1|_F / |X|_F)^(1/2)
// (N. J. Higham, "Computing the polar decomposition - with applications", SIAM J. Sci. Stat.
// Comput. 7 (1986)), which converges quadratically to the unitary factor.
#include <cmath>
#include <cstring>

#include "fixed.cuh"
#include "internal.cuh"

namespace hisq {
namespace smear {

struct M3 {
    double2 a[9];
};

__device__ __forceinline__ double2 cmul(double2 x, double2 y) { return make_double2(x.x * y.x - x.y * y.y, x.x * y.y + x.y * y.x); }

// s += x y, s += x conj(y), s += conj(x) y: four FMAs each.  (A product formed first and then
// added costs six FP64 operations, and the FP64 pipe is what bounds these kernels.)
__device__ __forceinline__ void mac(double2 &s, double2 x, double2 y)
{
    s.x = fma(x.x, y.x, fma(-x.y, y.y, s.x));
    s.y = fma(x.x, y.y, fma(x.y, y.x, s.y));
}
__device__ __forceinline__ void mac_c(double2 &s, double2 x, double2 y)
{
    s.x = fma(x.x, y.x, fma(x.y, y.y, s.x));
    s.y = fma(x.y, y.x, fma(-x.x, y.y, s.y));
}
__device__ __forceinline__ void cmac(double2 &s, double2 x, double2 y)
{
    s.x = fma(x.x, y.x, fma(x.y, y.y, s.x));
    s.y = fma(x.x, y.y, fma(-x.y, y.x, s.y));
}

__device__ __forceinline__ M3 zero()
{
    M3 r;
#pragma unroll
    for (int i = 0; i < 9; i++) r.a[i] = make_double2(0.0, 0.0);
    return r;
}

// A B, A B^+, A^+ B
__device__ __forceinline__ M3 mul(const M3 &A, const M3 &B)
{
    M3 r;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int k = 0; k < 3; k++) {
            double2 s = make_double2(0.0, 0.0);
#pragma unroll
            for (int j = 0; j < 3; j++) mac(s, A.a[3 * i + j], B.a[3 * j + k]);
            r.a[3 * i + k] = s;
        }
    return r;
}
__device__ __forceinline__ M3 mul_d(const M3 &A, const M3 &B)
{
    M3 r;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int k = 0; k < 3; k++) {
            double2 s = make_double2(0.0, 0.0);
#pragma unroll
            for (int j = 0; j < 3; j++) mac_c(s, A.a[3 * i + j], B.a[3 * k + j]);
            r.a[3 * i + k] = s;
        }
    return r;
}
__device__ __forceinline__ M3 d_mul(const M3 &A, const M3 &B)
{
    M3 r;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int k = 0; k < 3; k++) {
            double2 s = make_double2(0.0, 0.0);
#pragma unroll
            for (int j = 0; j < 3; j++) cmac(s, A.a[3 * j + i], B.a[3 * j + k]);
            r.a[3 * i + k] = s;
        }
    return r;
}
__device__ __forceinline__ void axpy(M3 &y, double c, const M3 &x)
{
#pragma unroll
    for (int i = 0; i < 9; i++) {
        y.a[i].x = fma(c, x.a[i].x, y.a[i].x);
        y.a[i].y = fma(c, x.a[i].y, y.a[i].y);
    }
}

struct Lat {
    int n[4];
    uint32_t V, Vh;
};

// Coordinates of canonical site i (even sites first, each parity in lexicographic order), so that
// consecutive threads read and write consecutive 144-byte records.
__device__ __forceinline__ void coords(const Lat &L, uint32_t i, int (&c)[4])
{
    const uint32_t p = i >= L.Vh;
    uint32_t q = i - p * L.Vh;
    const uint32_t nxh = (uint32_t)L.n[0] / 2;
    const uint32_t xh = q % nxh;
    q /= nxh;
    c[1] = (int)(q % (uint32_t)L.n[1]);
    q /= (uint32_t)L.n[1];
    c[2] = (int)(q % (uint32_t)L.n[2]);
    c[3] = (int)(q / (uint32_t)L.n[2]);
    c[0] = (int)(2 * xh + ((p + c[1] + c[2] + c[3]) & 1));
}

__device__ __forceinline__ uint32_t site_index(const Lat &L, const int (&c)[4])
{
    const uint32_t lex = (uint32_t)c[0] + (uint32_t)L.n[0] * ((uint32_t)c[1] + (uint32_t)L.n[1] * ((uint32_t)c[2] + (uint32_t)L.n[2] * (uint32_t)c[3]));
    return (lex >> 1) + L.Vh * (uint32_t)((c[0] + c[1] + c[2] + c[3]) & 1);
}

// one step along d, forward (k = 1) or backward (k = -1), periodic
__device__ __forceinline__ void move(const Lat &L, int (&y)[4], int d, int k)
{
#pragma unroll
    for (int e = 0; e < 4; e++)
        if (e == d) {
            y[e] += k;
            if (y[e] == L.n[e]) y[e] = 0;
            if (y[e] < 0) y[e] += L.n[e];
        }
}

// index of the site one step from c along d, and of the one a further step along d2
__device__ __forceinline__ uint32_t at(const Lat &L, const int (&c)[4], int d, int k)
{
    int y[4] = {c[0], c[1], c[2], c[3]};
    move(L, y, d, k);
    return site_index(L, y);
}
__device__ __forceinline__ uint32_t at(const Lat &L, const int (&c)[4], int d, int k, int d2, int k2)
{
    int y[4] = {c[0], c[1], c[2], c[3]};
    move(L, y, d, k);
    move(L, y, d2, k2);
    return site_index(L, y);
}

// Matrix i of a field in work: blocks of 32 matrices, 16-byte chunk q of all of them contiguous (whole
// 144-byte records would make every load of a warp touch 32 lines).  Coherent loads: a launch may read
// what the one before wrote.
__device__ __forceinline__ const double2 *slot(const double2 *f, size_t i) { return f + (i >> 5) * 288 + (i & 31); }
__device__ __forceinline__ M3 load(const double2 *f, size_t i)
{
    const double2 *p = slot(f, i);
    M3 r;
#pragma unroll
    for (int k = 0; k < 9; k++) r.a[k] = p[32 * k];
    return r;
}
// CANON: the caller's layout, one 144-byte record after the other
template <bool CANON = false>
__device__ __forceinline__ void store(double2 *f, size_t i, const M3 &m)
{
    double2 *p = CANON ? f + i * 9 : const_cast<double2 *>(slot(f, i));
#pragma unroll
    for (int k = 0; k < 9; k++) p[(CANON ? 1 : 32) * k] = m.a[k];
}

// A matrix in fixed point: complex entry q has the limbs h, l of reals 2q and 2q + 1, value
// (h 2^32 + l) 2^(code - 1023 - 59)
struct FxM {
    int32_t h[18], l[18];
    uint32_t code;
    __device__ __forceinline__ bool ok() const { return code - 823u <= 400u; } // 2^-200 .. 2^200
};
// A field of links holds them as fx_encode_link leaves them, the `rest` of link i behind all of them.
__device__ __forceinline__ void link_words(const double2 *f, size_t i, uint32_t (&w)[36])
{
    const uint4 *p = reinterpret_cast<const uint4 *>(slot(f, i));
#pragma unroll
    for (int k = 0; k < 9; k++) {
        const uint4 v = p[32 * k];
        w[4 * k] = v.x;
        w[4 * k + 1] = v.y;
        w[4 * k + 2] = v.z;
        w[4 * k + 3] = v.w;
    }
}
__device__ __forceinline__ const uint64_t *rests(const double2 *f, uint32_t V) { return reinterpret_cast<const uint64_t *>(f + (size_t)36 * V); }
// link i of a field
__device__ __forceinline__ FxM load_fx(const double2 *f, size_t i)
{
    uint32_t w[36];
    link_words(f, i, w);
    FxM r;
    uint32_t rows;
    r.code = fx_take_code(w, rows);
#pragma unroll
    for (int k = 0; k < 18; k++) {
        r.l[k] = (int32_t)w[2 * k];
        r.h[k] = (int32_t)w[2 * k + 1];
    }
    return r;
}
__device__ __forceinline__ FxM to_fx(const M3 &m)
{
    FxM r;
    uint32_t top = 0;
#pragma unroll
    for (int k = 0; k < 9; k++) {
        top = max(top, (uint32_t)__double2hiint(m.a[k].x) & 0x7fffffffu);
        top = max(top, (uint32_t)__double2hiint(m.a[k].y) & 0x7fffffffu);
    }
    r.code = top >> 20;
#pragma unroll
    for (int k = 0; k < 9; k++) {
        fx_limbs((uint32_t)__double2loint(m.a[k].x), (uint32_t)__double2hiint(m.a[k].x), r.code, 0u, r.h[2 * k], r.l[2 * k]);
        fx_limbs((uint32_t)__double2loint(m.a[k].y), (uint32_t)__double2hiint(m.a[k].y), r.code, 0u, r.h[2 * k + 1],
                 r.l[2 * k + 1]);
    }
    return r;
}
// link i of a field of 4 V links as doubles
__device__ __forceinline__ M3 load_link(const double2 *f, uint32_t V, size_t i)
{
    uint32_t w[36];
    double d[18];
    link_words(f, i, w);
    fx_decode_link(w, rests(f, V)[i], d);
    M3 r;
#pragma unroll
    for (int k = 0; k < 9; k++) r.a[k] = make_double2(d[2 * k], d[2 * k + 1]);
    return r;
}

// a row of three complex sums: component 2k + c is H 2^32 + M
struct FxRow {
    int64_t H[6], M[6];
};
// (re, im) of column k += a b with a = (ar, ai), b's limbs given for each of the four products
__device__ __forceinline__ void mac(int64_t &H, int64_t &M, int32_t ah, int32_t al, int32_t bh, int32_t bl)
{
    H += (int64_t)ah * bh;
    M += (int64_t)ah * bl;
    M += (int64_t)al * bh;
}
__device__ __forceinline__ void fold(FxRow &r)
{
#pragma unroll
    for (int k = 0; k < 6; k++) {
        r.H[k] += (int64_t)(int32_t)(r.M[k] >> 32);
        r.M[k] = (int64_t)(uint32_t)r.M[k];
    }
}

// 1-norm of complex entry q in units of 2^-13 of 2^e, cut, at most 2^15
__device__ __forceinline__ uint32_t norm1(const FxM &m, int q)
{
    const int32_t r = m.h[2 * q], i = m.h[2 * q + 1];
    return ((uint32_t)(r ^ (r >> 31)) + (uint32_t)(i ^ (i >> 31))) >> 14;
}
// What enters the entries of row i of op(A) F op(B): S_ik = sum_jl |A_ij| |F_jl| |B_lk| in 1-norms of the entries;
// the least of a row in units of 2^-22 of 2^(eA + eF + eB)
template <bool DA, bool DB>
__device__ __forceinline__ void least_sums(const FxM &A, const FxM &F, const FxM &B, uint32_t (&m)[3])
{
    uint32_t g[9];
#pragma unroll
    for (int j = 0; j < 3; j++)
#pragma unroll
        for (int k = 0; k < 3; k++) {
            uint32_t x = 0;
#pragma unroll
            for (int l = 0; l < 3; l++) x += norm1(F, 3 * j + l) * norm1(B, DB ? 3 * k + l : 3 * l + k);
            g[3 * j + k] = x >> 17;
        }
#pragma unroll
    for (int i = 0; i < 3; i++) {
        m[i] = 0xffffffffu;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            uint32_t x = 0;
#pragma unroll
            for (int j = 0; j < 3; j++) x += norm1(A, DA ? 3 * j + i : 3 * i + j) * g[3 * j + k];
            m[i] = min(m[i], x);
        }
    }
}

// op(A) F op(B) with op the adjoint where DA, DB say so, for codes in range; false if the result may be less
// precise than FP64's.  Row by row: row i of op(A) F, brought back to two limbs (its sums of six products
// stay below 2^90.6; the shift sh <= 31 leaves its largest entry 59 or 60 bits), times op(B).
// Error of an entry's real or imaginary part, at most, in units of 2^-56 of 2^(eA + eF + eB): six products of the
// first kind, 1.75 each (fixed.cuh), a row cut to units of 2^(sh - 30) (and one more where a limb was negated),
// all times twelve, then 2^(sh - 27) for each l l' of the second and the cut of B: 126 + 10.5 2^(sh - 27).
// FP64 multiply-adds err by up to 12 2^-53 S.  Both worked out in exact arithmetic for 8,600 entries of products of
// links and staples at eps 0.03 to 1 (sh - 27 mostly 2): the fixed-point ones err less, 0.38 2^-53 S against 0.40
// (rms) and 1.1 against 1.9 (largest), from S = 0.75 on (0.48 against 0.37 below that; 0.10 against 0.25 from 10
// on).  So an entry needs S >= 0.5 + 2^(sh - 31).  Products that have less at eps 0.5: none, at 0.3 4e-5
// (second level; its links are smoother), at 0.2 0.4 %, at 0.1 28 %, closer to unity nearly all: 24^3 x 8 in
// 6.9, 7.2, 8.1, 18.1 ms, 13.7 ms at eps 0.001 (6.7 whatever the links without looking).
template <bool DA, bool DB>
__device__ __forceinline__ bool product(const FxM &A, const FxM &F, const FxM &B, M3 &out)
{
    uint32_t least[3];
    least_sums<DA, DB>(A, F, B, least);
    bool ok = min(least[0], min(least[1], least[2])) >= 2097152u;
    if (!ok) return false;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        FxRow r = {};
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const int q = DA ? 3 * j + i : 3 * i + j;
            const int32_t arh = A.h[2 * q], arl = A.l[2 * q], aih = A.h[2 * q + 1], ail = A.l[2 * q + 1];
            int32_t nh, nl;
            fx_neg(aih, ail, nh, nl);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const int f = 2 * (3 * j + k);
                mac(r.H[2 * k], r.M[2 * k], arh, arl, F.h[f], F.l[f]);
                mac(r.H[2 * k], r.M[2 * k], DA ? aih : nh, DA ? ail : nl, F.h[f + 1], F.l[f + 1]);
                mac(r.H[2 * k + 1], r.M[2 * k + 1], arh, arl, F.h[f + 1], F.l[f + 1]);
                mac(r.H[2 * k + 1], r.M[2 * k + 1], DA ? nh : aih, DA ? nl : ail, F.h[f], F.l[f]);
            }
        }
        fold(r);
        uint32_t top = 0;
#pragma unroll
        for (int k = 0; k < 6; k++) top |= (uint32_t)(r.H[k] >> 32) ^ (uint32_t)(r.H[k] >> 63);
        const uint32_t sh = 36u - (uint32_t)__clz((int)top); // 4 .. 31
        const uint32_t E = A.code + F.code + B.code - 1050u + sh;
        ok = ok && least[i] >= 2097152u + ((1u << sh) >> 9);
        int32_t ph[6], pl[6];
#pragma unroll
        for (int k = 0; k < 6; k++) {
            const uint32_t lo = (uint32_t)r.H[k];
            pl[k] = (int32_t)__funnelshift_r((uint32_t)r.M[k], lo, sh);
            ph[k] = (int32_t)__funnelshift_r(lo, (uint32_t)(r.H[k] >> 32), sh) + (int32_t)((uint32_t)pl[k] >> 31);
        }
        FxRow o = {};
#pragma unroll
        for (int j = 0; j < 3; j++) {
            // the part of the row's entry that enters negated: re with B^+, im with B
            int32_t nh, nl;
            fx_neg(ph[2 * j + (DB ? 0 : 1)], pl[2 * j + (DB ? 0 : 1)], nh, nl);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const int b = 2 * (DB ? 3 * k + j : 3 * j + k);
                mac(o.H[2 * k], o.M[2 * k], ph[2 * j], pl[2 * j], B.h[b], B.l[b]);
                mac(o.H[2 * k], o.M[2 * k], DB ? ph[2 * j + 1] : nh, DB ? pl[2 * j + 1] : nl, B.h[b + 1], B.l[b + 1]);
                mac(o.H[2 * k + 1], o.M[2 * k + 1], DB ? nh : ph[2 * j], DB ? nl : pl[2 * j], B.h[b + 1], B.l[b + 1]);
                mac(o.H[2 * k + 1], o.M[2 * k + 1], ph[2 * j + 1], pl[2 * j + 1], B.h[b], B.l[b]);
            }
        }
        fold(o);
#pragma unroll
        for (int k = 0; k < 3; k++)
            out.a[3 * i + k] = make_double2(fx_value(o.H[2 * k], (uint32_t)o.M[2 * k], E),
                                            fx_value(o.H[2 * k + 1], (uint32_t)o.M[2 * k + 1], E));
    }
    return ok;
}

// the same in FP64, for matrices that the fixed-point range or precision leaves out
static __device__ __noinline__ void product_f64(bool da, bool db, const double2 *u, uint32_t V, size_t ia, size_t ib, M3 &F)
{
    const M3 A = load_link(u, V, ia), B = load_link(u, V, ib);
    const M3 P = da ? d_mul(A, F) : mul(A, F);
    F = db ? mul_d(P, B) : mul(P, B);
}

// op(A) F op(B) of links ia and ib; get() gives F as doubles, F in fixed point
template <bool DA, bool DB, class Get>
__device__ __forceinline__ M3 around(const Lat &L, const double2 *u, size_t ia, const FxM &F, size_t ib, const Get &get)
{
    const FxM A = load_fx(u, ia), B = load_fx(u, ib);
    M3 r;
    if (A.ok() && B.ok() && F.ok() && product<DA, DB>(A, F, B, r)) return r;
    r = get();
    product_f64(DA, DB, u, L.V, ia, ib, r);
    return r;
}

// The two halves of stap_nu[F]_mu(x) = up + down for a field of V matrices F (of direction mu):
//   up   = U_nu(x) F(x+nu) U_nu(x+mu)^+,   down = U_nu(x-nu)^+ F(x-nu) U_nu(x-nu+mu)
// with get() the matrix F(x+nu) or F(x-nu).
template <class Get>
__device__ __forceinline__ M3 stap_up(const Lat &L, const double2 *u, int mu, int nu, const int (&x)[4], const Get &get)
{
    const size_t o = (size_t)nu * L.V;
    return around<false, true>(L, u, o + site_index(L, x), to_fx(get()), o + at(L, x, mu, 1), get);
}
template <class Get>
__device__ __forceinline__ M3 stap_down(const Lat &L, const double2 *u, int mu, int nu, const int (&x)[4], const Get &get)
{
    const size_t o = (size_t)nu * L.V;
    return around<true, false>(L, u, o + at(L, x, nu, -1), to_fx(get()), o + at(L, x, nu, -1, mu, 1), get);
}

struct Coef {
    double c1, c3, c5, c7, cl;
};

// One level for one direction mu, in three launches over the sites.  The nested staples are built
// from each other, with every intermediate stored:
//   1  T_nu = stap_nu[F], its halves apart when Lepage paths are wanted
//   2  G_rho = c5 sum_{nu != rho} T_nu + c7 (stap_a[T_b] + stap_b[T_a]),  {a, b} = not mu, rho
//   3  out = c1 F + c3 sum T + sum_rho stap_rho[G_rho] (+ Lepage)
// A Lepage path is the upper half around an upper half, or the lower around a lower, along one
// direction, so launch 3 only adds cl T_up to what the upper half encloses and cl T_down to the
// lower: no product of its own.  48 matrix products per link and level; building every path from
// its links took 252 (300 with Lepage).
// The products run on integers (product): FP64 multiply-adds, 48 x 108 per link at two a clock and SM,
// took 9.5 of 12.4 ms on 24^3 x 8, 4.9 of 7.6 ms so; what is left is bound by integer and FP64
// issue at eight warps an SM (the operands of a product fill the registers).  One thread per (site,
// detour) in launches 1 and 2, one per site in 3, consecutive sites in consecutive lanes.
// 24^3 x 8, the whole call with projection and Naik links: 76.0 ms with every path multiplied out, 12.4
// with stored staples in FP64, 7.6 with these products, 6.7 with the projection of now, 7.1 with the look at what
// enters each entry (product).
__global__ void __launch_bounds__(128) k_stap3(Lat L, const double2 *u, int mu, double2 *t, double2 *td)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.V) return;
    const int n = blockIdx.y, nu = n + (n >= mu);
    int x[4];
    coords(L, i, x);
    const size_t m = (size_t)mu * L.V, o = (size_t)nu * L.V;
    const size_t iu = m + at(L, x, nu, 1), id = m + at(L, x, nu, -1);
    M3 up = around<false, true>(L, u, o + site_index(L, x), load_fx(u, iu), o + at(L, x, mu, 1), [&] { return load_link(u, L.V, iu); });
    const M3 dn = around<true, false>(L, u, o + at(L, x, nu, -1), load_fx(u, id), o + at(L, x, nu, -1, mu, 1),
                                      [&] { return load_link(u, L.V, id); });
    if (td) store(td, (size_t)n * L.V + i, dn);
    else axpy(up, 1.0, dn);
    store(t, (size_t)n * L.V + i, up);
}

// T_n at site j (its halves added when they are stored apart)
__device__ __forceinline__ M3 load_t(const Lat &L, const double2 *t, const double2 *td, int n, uint32_t j)
{
    M3 r = load(t, (size_t)n * L.V + j);
    if (td) axpy(r, 1.0, load(td, (size_t)n * L.V + j));
    return r;
}

__global__ void __launch_bounds__(128) k_stap5(Lat L, const double2 *u, int mu, const double2 *t, const double2 *td,
                                               double2 *g, Coef c)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.V) return;
    const int n = blockIdx.y; // rho, as the n-th direction other than mu
    int x[4];
    coords(L, i, x);
    M3 acc = zero();
#pragma unroll 1
    for (int k = 1; k < 3; k++) {
        const int na = (n + k) % 3, nb = (n + 3 - k) % 3; // the two other detours, in both orders
        const int a = na + (na >= mu);
        axpy(acc, c.c7, stap_up(L, u, mu, a, x, [&] { return load_t(L, t, td, nb, at(L, x, a, 1)); }));
        axpy(acc, c.c7, stap_down(L, u, mu, a, x, [&] { return load_t(L, t, td, nb, at(L, x, a, -1)); }));
        axpy(acc, c.c5, load_t(L, t, td, na, i));
    }
    store(g, (size_t)n * L.V + i, acc);
}

template <bool CANON>
__global__ void __launch_bounds__(128) k_stap7(Lat L, const double2 *u, int mu, const double2 *t, const double2 *td,
                                               const double2 *g, double2 *out, Coef c)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.V) return;
    int x[4];
    coords(L, i, x);
    M3 acc = zero();
    axpy(acc, c.c1, load_link(u, L.V, (size_t)mu * L.V + i));
#pragma unroll 1
    for (int n = 0; n < 3; n++) {
        const int rho = n + (n >= mu);
        const uint32_t ju = at(L, x, rho, 1), jd = at(L, x, rho, -1);
        const auto inner = [&](const double2 *half, uint32_t j) {
            M3 F = load(g, (size_t)n * L.V + j);
            if (td) axpy(F, c.cl, load(half, (size_t)n * L.V + j));
            return F;
        };
        axpy(acc, 1.0, stap_up(L, u, mu, rho, x, [&] { return inner(t, ju); }));
        axpy(acc, 1.0, stap_down(L, u, mu, rho, x, [&] { return inner(td, jd); }));
        axpy(acc, c.c3, load_t(L, t, td, n, i));
    }
    store<CANON>(out, (size_t)mu * L.V + i, acc);
}

// One smearing level of the links u into out.  t, td, g: scratch of 3 V matrices each (td NULL: no
// Lepage paths); none of them overlaps u or out.  CANON: out in the caller's layout.
template <bool CANON>
static void smear_level(const Lat &L, const double2 *u, double2 *out, double2 *t, double2 *td, double2 *g, const Coef &c,
                        cudaStream_t st)
{
    const unsigned nb = (L.V + 127) / 128;
    for (int mu = 0; mu < 4; mu++) {
        k_stap3<<<dim3(nb, 3), 128, 0, st>>>(L, u, mu, t, td);
        k_stap5<<<dim3(nb, 3), 128, 0, st>>>(L, u, mu, t, td, g, c);
        k_stap7<CANON><<<nb, 128, 0, st>>>(L, u, mu, t, td, g, out, c);
    }
}

// inverse of a 3x3 complex matrix by cofactors; returns false if singular
__device__ bool inverse(const M3 &A, M3 &inv)
{
    const double2 *a = A.a;
    double2 cof[9];
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const int i1 = (i + 1) % 3, i2 = (i + 2) % 3, j1 = (j + 1) % 3, j2 = (j + 2) % 3;
            double2 p = cmul(a[3 * i1 + j1], a[3 * i2 + j2]);
            const double2 q = a[3 * i1 + j2];
            mac(p, make_double2(-q.x, -q.y), a[3 * i2 + j1]);
            cof[3 * i + j] = p;
        }
    double2 det = make_double2(0.0, 0.0);
#pragma unroll
    for (int j = 0; j < 3; j++) mac(det, a[j], cof[j]);
    const double dd = det.x * det.x + det.y * det.y;
    if (!(dd > 0.0) || !isfinite(dd)) return false;
    const double2 rdet = make_double2(det.x / dd, -det.y / dd);
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) inv.a[3 * i + j] = cmul(cof[3 * j + i], rdet); // adjugate / det
    return true;
}

__device__ __forceinline__ double fro2(const M3 &A)
{
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < 9; i++) s = fma(A.a[i].x, A.a[i].x, fma(A.a[i].y, A.a[i].y, s));
    return s;
}

// a matrix as a link of the second level (fixed point, in blocks)
__device__ __forceinline__ void store_link(double2 *f, uint32_t V, size_t i, const M3 &m)
{
    double d[18];
    uint32_t w[36];
    uint64_t rest;
#pragma unroll
    for (int k = 0; k < 9; k++) {
        d[2 * k] = m.a[k].x;
        d[2 * k + 1] = m.a[k].y;
    }
    fx_encode_link(d, w, rest);
    const_cast<uint64_t *>(rests(f, V))[i] = rest;
    uint4 *p = reinterpret_cast<uint4 *>(const_cast<double2 *>(slot(f, i)));
#pragma unroll
    for (int k = 0; k < 9; k++) p[32 * k] = make_uint4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
}

// the caller's thin links (records) as links of the first level
__global__ void __launch_bounds__(128) k_take_links(const double2 *thin, double2 *u, uint32_t V)
{
    const uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (t >= 4ull * V) return;
    M3 m;
#pragma unroll
    for (int k = 0; k < 9; k++) m.a[k] = thin[t * 9 + k];
    store_link(u, V, t, m);
}

// W = unitary polar factor of V (scaled Newton iteration); a singular or non-converging
// matrix raises the device error flag
__global__ void __launch_bounds__(128) k_project_u3(const double2 *v, double2 *w, uint32_t V, DevStatus *status)
{
    const uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (t >= 4ull * V) return;
    M3 X = load(v, t);
    bool ok = false, scaled = true;
    for (int it = 0; it < 30; it++) {
        M3 Xi;
        if (!inverse(X, Xi)) break;
        // any positive g leaves the polar factor alone (it only speeds up the first steps), so its
        // roots and inverse are taken in FP32, and left out once X is close to unitary: with a division
        // by g for each of the 18 reals the projection took 2.0 ms on 24^3 x 8, 1.1 ms so
        double g = 1.0, gi = 1.0;
        if (scaled) {
            const double q = fro2(Xi) / fro2(X);
            if (q > 1e-30 && q < 1e30) {
                const float f = sqrtf(sqrtf((float)q));
                g = (double)f;
                gi = (double)(1.f / f);
            } else {
                g = sqrt(sqrt(q));
                gi = 1.0 / g;
            }
        }
        M3 Y;
        double diff = 0.0;
#pragma unroll
        for (int r = 0; r < 3; r++)
#pragma unroll
            for (int c = 0; c < 3; c++) {
                // (X^-1)^+ = conj of the transposed inverse
                const double2 xi = Xi.a[3 * c + r];
                const double2 y = make_double2(0.5 * fma(g, X.a[3 * r + c].x, xi.x * gi),
                                               0.5 * fma(g, X.a[3 * r + c].y, -(xi.y * gi)));
                const double dx = y.x - X.a[3 * r + c].x, dy = y.y - X.a[3 * r + c].y;
                diff = fma(dx, dx, fma(dy, dy, diff));
                Y.a[3 * r + c] = y;
            }
        scaled = scaled && !(diff < 0.03);
        X = Y;
        // quadratic convergence: a change of 1e-12 leaves an error of order 1e-24
        if (diff <= 1e-24 * fro2(X)) {
            ok = true;
            break;
        }
    }
    store_link(w, V, t, X);
    if (!ok && status) {
        status->where = 2; // link projection
        atomicExch(&status->error, (int)HISQ_EDEVICE);
    }
}

// N_mu(x) = cN W_mu(x) W_mu(x+mu) W_mu(x+2mu)
__global__ void __launch_bounds__(128) k_naik(Lat L, const double2 *w, double2 *out, double cn)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.V) return;
    const int mu = blockIdx.y;
    int x[4];
    coords(L, i, x);
    const size_t m = (size_t)mu * L.V, j = m + at(L, x, mu, 1);
    const M3 r = around<false, false>(L, w, m + i, load_fx(w, j), m + at(L, x, mu, 1, mu, 1), [&] { return load_link(w, L.V, j); });
    M3 o = zero();
    axpy(o, cn, r);
    store<true>(out, (size_t)mu * L.V + i, o);
}

}  // namespace smear
}  // namespace hisq

using namespace hisq;

extern "C" int hisq_smear_links(const int dims[4], const double *thin, double *fat, double *lng, double eps_naik,
                                int links_on_device, void *stream)
{
    if (!dims || !thin || !fat || !lng || !std::isfinite(eps_naik)) return HISQ_EINVAL;
    smear::Lat L{};
    uint64_t V = 1;
    for (int d = 0; d < 4; d++) {
        if (dims[d] < 4 || dims[d] % 2) return HISQ_EINVAL;
        L.n[d] = dims[d];
        V *= (uint64_t)dims[d];
    }
    if (V > (1ull << 31)) return HISQ_EINVAL;
    L.V = (uint32_t)V;
    L.Vh = (uint32_t)(V / 2);
    const size_t bytes = 4 * V * 9 * sizeof(double2), fx_bytes = bytes + 4 * V * kFxRestBytes;
    cudaStream_t st = (cudaStream_t)stream;
    double2 *u = nullptr, *v = nullptr, *w = nullptr, *x = nullptr, *nk = nullptr;
    DevStatus *status = nullptr;
    auto release = [&]() {
        for (void *p : {(void *)u, (void *)v, (void *)w, (void *)x, (void *)nk, (void *)status})
            if (p) cudaFree(p);
    };
    bool ok = cudaMalloc((void **)&u, fx_bytes) == cudaSuccess && cudaMalloc((void **)&v, bytes) == cudaSuccess &&
              cudaMalloc((void **)&w, fx_bytes) == cudaSuccess && cudaMalloc((void **)&status, sizeof(DevStatus)) == cudaSuccess;
    if (ok && !links_on_device) ok = cudaMalloc((void **)&x, bytes) == cudaSuccess && cudaMalloc((void **)&nk, bytes) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        release();
        return HISQ_ENOMEM;
    }
    double2 *xo = links_on_device ? reinterpret_cast<double2 *>(fat) : x;
    double2 *no = links_on_device ? reinterpret_cast<double2 *>(lng) : nk;
    cudaError_t e = cudaMemsetAsync(status, 0, sizeof(DevStatus), st);
    // links on the host, or not on the 16-byte boundaries that the kernels read, go through v, which
    // holds nothing yet
    const bool direct = links_on_device && (reinterpret_cast<uintptr_t>(thin) & 15) == 0;
    const double2 *src = direct ? reinterpret_cast<const double2 *>(thin) : v;
    if (e == cudaSuccess && !direct)
        e = cudaMemcpyAsync(v, thin, bytes, links_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, st);
    const unsigned nb = (unsigned)((V + 127) / 128), nb4 = (unsigned)((4 * V + 127) / 128);
    if (e == cudaSuccess) {
        // scratch of a level (three matrices per site each): fields that hold nothing yet or no
        // longer, so no memory beyond the links, the two levels and the results is needed
        smear::k_take_links<<<nb4, 128, 0, st>>>(src, u, L.V);
        smear::smear_level<false>(L, u, v, w, nullptr, xo, smear::Coef{1.0 / 8, 1.0 / 16, 1.0 / 64, 1.0 / 384, 0.0}, st);
        smear::k_project_u3<<<nb4, 128, 0, st>>>(v, w, L.V, status);
        smear::smear_level<true>(L, w, xo, u, v, no, smear::Coef{1.0, 1.0 / 16, 1.0 / 64, 1.0 / 384, -1.0 / 8}, st);
        smear::k_naik<<<dim3(nb, 4), 128, 0, st>>>(L, w, no, -1.0 / 24 + eps_naik / 8);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && !links_on_device) {
        e = cudaMemcpyAsync(fat, xo, bytes, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(lng, no, bytes, cudaMemcpyDeviceToHost, st);
    }
    DevStatus h{};
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, status, sizeof(h), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    release();
    if (e != cudaSuccess) {
        cudaGetLastError();
        return e == cudaErrorMemoryAllocation ? HISQ_ENOMEM : HISQ_ECUDA;
    }
    return h.error ? HISQ_EDEVICE : HISQ_OK;
}
