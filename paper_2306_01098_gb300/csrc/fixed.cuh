// fixed.cuh -- link times colour vector in 60-bit fixed point: the arithmetic of the FP64
// Dslash with 18-real links.
//
// This GPU issues two FP64 operations per clock and SM; the 576 multiply-adds of one Dslash
// site then take 288 clocks where its bytes take about 100.  Integer multiply-adds
// (32 x 32 + 64 -> 64 bits) issue many times faster, so the products are formed on integers:
//   a link is  Lambda 2^(e_L - 59),   Lambda integer, |Lambda| <= 2^60, 2^e_L <= max |entry| < 2^(e_L + 1)
//   a vector is     N 2^(e_v - 59)    likewise, made from its doubles when it is loaded
// both kept as two limbs, x = h 2^32 + l with -2^31 <= l < 2^31 and |h| <= 2^28.  A product is
//   h h' 2^64 + (h l' + l h') 2^32     (l l' is dropped: at most 2^62 of up to 2^120)
// i.e. three multiply-adds into two 64-bit sums, H and M.  Bounds: H adds 96 products of at most
// 2^56 per component and site (16 hops, 3 colours, re and im): < 2^62.6.  M adds 12 products of
// at most 2^59 per hop, and is folded into H after every hop: < 2^62.6 too.  Nothing is lost in
// the sums; all hops of a site are aligned to the largest exponent e_L + e_v met so far (H and M
// are shifted when a larger one comes).
// Error of one real product, in units of 2^E, E the largest e_L + e_v of the site: 2^-56 for l l', 2^-58
// each for the cut of the vector and of the link (one unit of 2^-59, against less than 2), 2^-58 where a limb
// of -2^31 was negated: below 1.75 2^-56; the sum is rounded to FP64 once.  A sum of n products formed
// with FP64 multiply-adds errs by up to n 2^-53 S, S = sum |U| |v| over the reals that enter the component.
// So the fixed-point sum is held to no less precision, component by component, where S >= 7/32 2^E for all six
// components of a site: the sites where that is not certain are computed in FP64 (a point source, colours of
// very different sizes among links that hardly mix them).  What is certain: a hop gives every S at
// least the smallest real of its vector times the link's smallest row or column sum of |reals|, 2^e_L f and more
// with f = 0 .. 3 kept beside the exponent (1 at least for any multiple of a unitary matrix).  The one-step hops are
// counted, some ten instructions each (the three-step links are a 24th of theirs).  Of Gaussian vectors on links of
// eps 0.1 to 1 no more than 4e-5 of the sites are left to FP64, likewise of a solve's vectors some 20 steps from a
// point or wall source.
// Measured (max over a field, relative to its largest entry): 2.4e-16 after the normal operator of a
// 32^3 x 8 lattice, 3.9e-16 with FP64 multiply-adds.  Time there, two Dslash launches: 280.8 us with
// FP64 multiply-adds (their pipe alone needs 250 us), 130 us in fixed point without a look at the components, 137 us so
// (the bytes need 93 us).
// Sites that meet anything this cannot hold (an infinity or NaN, a link or vector whose largest real is
// below about 1e-289, products outside about 1e-254 .. 1e287, a link whose reals lie too far apart) are
// computed in FP64 instead (fx_sites_f64), from the same doubles.
#pragma once

#include "internal.cuh"

namespace hisq {

// Stored link, 18 reals: word 2i the low limb of real i, word 2i + 1 its high limb in 30 bits.  The top two
// bits of the high words of reals 0 .. 6 hold, from real 0 on, the biased exponent e_L + 1023 (11 bits): 0 for a
// link of zeros, 0x7ff for one that the format cannot hold (an infinity or NaN, entries too small or too far
// apart), whose words are then the doubles themselves; above it f (2 bits).  Magnitudes are cut, not rounded, to units of
// 2^(e_L - 59), so that a real's position below e_L can be read off its leading bit, and what was cut is
// kept: the store holds 64 more bits for every link, `rest`, with the mantissa bits below the unit, real after
// real (a real 2^-k of the largest has lost its lowest k - 7), or the two bits of each high word that a
// link of doubles gave to the exponent.  The doubles can be had back exactly (fx_decode_link), zeros stay zeros.
constexpr int kFxMarked = 7;        // reals whose high words carry bits of the code
constexpr uint32_t kFxRaw = 0xfff;  // fx_take_code of a link of doubles
constexpr uint32_t kFxBalance = 7u << 15; // 7/32 in the units of FxAcc::B
constexpr uint32_t kFxMinExp = 64;  // smallest biased exponent of a link or vector in fixed point
constexpr int kFxRestBytes = 8;     // bytes of `rest` per link
// biased exponents of products (sum of two biased exponents) that the sums are formed with
// (results, whose last bit is 2^-85 of the largest product, stay normal numbers)
constexpr uint32_t kFxELo = 1200, kFxEHi = 3000;

__host__ __device__ __forceinline__ uint64_t fx_bits(double x)
{
    union { double d; uint64_t u; } c;
    c.d = x;
    return c.u;
}
// position of the leading bit of x != 0
__host__ __device__ __forceinline__ int fx_top(uint64_t x)
{
#ifdef __CUDA_ARCH__
    return 63 - __clzll((long long)x);
#else
    return 63 - __builtin_clzll(x);
#endif
}

// the low 30 bits as a signed number
__host__ __device__ __forceinline__ int32_t fx_low30(uint32_t x)
{
#ifdef __CUDA_ARCH__
    int32_t r;
    asm("bfe.s32 %0, %1, 0, 30;" : "=r"(r) : "r"(x));
    return r;
#else
    return (int32_t)(x << 2) >> 2;
#endif
}

__host__ __device__ inline void fx_encode_link(const double (&d)[18], uint32_t (&w)[36], uint64_t &rest)
{
    uint32_t em = 0;
    bool zero = true;
#pragma unroll
    for (int i = 0; i < 18; i++) {
        const uint64_t b = fx_bits(d[i]);
        const uint32_t e = (uint32_t)(b >> 52) & 0x7ffu;
        em = e > em ? e : em;
        zero = zero && (b << 1) == 0;
    }
    bool raw = !zero && (em < kFxMinExp || em == 0x7ffu);
    uint32_t used = 0;
    rest = 0;
#pragma unroll
    for (int i = 0; i < 18; i++) {
        const uint64_t b = fx_bits(d[i]);
        const uint32_t e = (uint32_t)(b >> 52) & 0x7ffu, s = em - e;
        int64_t x = 0;
        if ((b << 1) != 0 && !raw) {
            // 53-bit magnitude, shifted left by 7 (60 bits) and right by the distance to the largest exponent
            const uint64_t m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 7;
            const uint32_t n = s > 7 ? s - 7 : 0;
            if (e == 0 || s > 59 || used + n > 64) {
                raw = true;
            } else {
                if (n) rest |= ((m & ((1ull << s) - 1)) >> 7) << used;
                used += n;
                x = (int64_t)(m >> s);
                if (b >> 63) x = -x;
            }
        }
        const int32_t l = (int32_t)(uint32_t)x;
        w[2 * i] = (uint32_t)l;
        w[2 * i + 1] = (uint32_t)((x - l) >> 32);
    }
    // smallest row and column sum of |reals|, in units of 2^e_L
    uint32_t row[3] = {0u, 0u, 0u}, col[3] = {0u, 0u, 0u};
#pragma unroll
    for (int q = 0; q < 18; q++) {
        const int32_t h = (int32_t)w[2 * q + 1];
        const uint32_t a = h < 0 ? ~(uint32_t)h : (uint32_t)h; // (no more than |x| 2^-32)
        row[q / 6] += a;
        col[q / 2 % 3] += a;
    }
    uint32_t f = 3;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        f = row[k] >> 27 < f ? row[k] >> 27 : f;
        f = col[k] >> 27 < f ? col[k] >> 27 : f;
    }
    const uint32_t code = zero ? 0u : raw ? 0x7ffu : em | f << 11;
    if (raw) rest = 0;
#pragma unroll
    for (int i = 0; i < 18; i++) {
        if (raw) {
            const uint64_t b = fx_bits(d[i]);
            w[2 * i] = (uint32_t)b;
            w[2 * i + 1] = (uint32_t)(b >> 32);
            if (i < kFxMarked) rest |= (uint64_t)(w[2 * i + 1] >> 30) << (2 * i);
        }
        if (i < kFxMarked) w[2 * i + 1] = (w[2 * i + 1] & 0x3fffffffu) | ((code >> (2 * i)) & 3u) << 30;
    }
}

// biased exponent and f of a stored link (kFxRaw: doubles, which stay as stored); the words become the limbs
__host__ __device__ __forceinline__ uint32_t fx_take_code(uint32_t (&w)[36], uint32_t &f)
{
    uint32_t c = 0;
#pragma unroll
    for (int i = kFxMarked - 1; i >= 0; i--) {
        c = c << 2 | w[2 * i + 1] >> 30;
        w[2 * i + 1] = (uint32_t)fx_low30(w[2 * i + 1]);
    }
    f = c >> 11;
    c &= 0x7ffu;
    return c == 0x7ffu ? kFxRaw : c;
}

// the doubles of a stored link (its words as stored); no branches on the reals, whose bits then come together
// side by side: only the count of bits used passes from one to the next
__host__ __device__ inline void fx_decode_link(const uint32_t (&w)[36], uint64_t rest, double (&d)[18])
{
    uint32_t code = 0;
#pragma unroll
    for (int i = 0; i < kFxMarked; i++) code |= (w[2 * i + 1] >> 30) << (2 * i);
    code &= 0x7ffu;
    union { double d; uint64_t u; } c;
    if (code == 0x7ffu) {
#pragma unroll
        for (int i = 0; i < 18; i++) {
            const uint32_t hi = i < kFxMarked ? (w[2 * i + 1] & 0x3fffffffu) | ((uint32_t)(rest >> (2 * i)) & 3u) << 30 : w[2 * i + 1];
            c.u = (uint64_t)hi << 32 | w[2 * i];
            d[i] = c.d;
        }
        return;
    }
    uint32_t used = 0;
#pragma unroll
    for (int i = 0; i < 18; i++) {
        const int32_t h = i < kFxMarked ? fx_low30(w[2 * i + 1]) : (int32_t)w[2 * i + 1];
        const int64_t x = (int64_t)h * 4294967296ll + (int32_t)w[2 * i];
        const uint64_t a = (uint64_t)(x < 0 ? -x : x);
        const uint32_t s = 59u - (uint32_t)fx_top(a | 1u), n = a && s > 7 ? s - 7 : 0;
        const uint64_t m = a << s | ((rest >> (used & 63)) & ((1ull << n) - 1)) << 7;
        used += n;
        c.u = (x < 0 ? 1ull << 63 : 0ull) | (uint64_t)(code - s) << 52 | ((m >> 7) & 0xfffffffffffffull);
        d[i] = a ? c.d : 0.0;
    }
}

// running sums of one output vector: component k is (H[k] 2^32 + M[k]) 2^(E - 2046 - 118 + 32)
// E: largest sum of biased exponents so far; B: what the S of every component reaches at least, in units of
// 2^-20 of 2^E (below 2^27); bad: a value that the format cannot hold was met
struct FxAcc {
    int64_t H[6], M[6];
    uint32_t E, B;
    bool bad;
};

__device__ __forceinline__ void fx_zero(FxAcc &a)
{
#pragma unroll
    for (int k = 0; k < 6; k++) a.H[k] = a.M[k] = 0;
    a.E = kFxELo;
    a.B = 0;
    a.bad = false;
}

// sums >>= d (d > 0): H and the 32 bits of M, as one 96-bit number
__device__ __forceinline__ void fx_shift(FxAcc &a, uint32_t d)
{
#pragma unroll
    for (int k = 0; k < 6; k++) {
        const int64_t H = a.H[k];
        const uint32_t f = (uint32_t)a.M[k];
        if (d < 32) a.M[k] = (int64_t)__funnelshift_r(f, (uint32_t)H, d);
        else a.M[k] = (int64_t)(uint32_t)(H >> (d - 32 < 63 ? d - 32 : 63));
        a.H[k] = H >> (d < 63 ? d : 63);
    }
    a.B = __funnelshift_rc(a.B, 0u, d);
}

// the sums are no better than FP64 would be (or hold something that has no place in them)
__device__ __forceinline__ bool fx_left(const FxAcc &a) { return a.bad || (a.E > kFxELo && a.B < kFxBalance); }

// M's carry into H; its low 32 bits stay
__device__ __forceinline__ void fx_fold(FxAcc &a)
{
#pragma unroll
    for (int k = 0; k < 6; k++) {
        a.H[k] += (int64_t)(int32_t)(a.M[k] >> 32);
        a.M[k] = (int64_t)(uint32_t)a.M[k];
    }
}

// limbs of the double hi:lo for the biased exponent t (>= its own), negated if flip = ~0
__device__ __forceinline__ void fx_limbs(uint32_t lo, uint32_t hi, uint32_t t, uint32_t flip, int32_t &h, int32_t &l)
{
    const uint32_t s = t - ((hi >> 20) & 0x7ffu);
    const uint32_t mh = (hi & 0xfffffu) | 0x100000u;
    uint64_t m = (uint64_t)__funnelshift_l(lo, mh, 7) << 32 | (lo << 7);
    m = s < 64 ? m >> s : 0ull;
    const uint32_t sg = (uint32_t)((int32_t)(hi ^ flip) >> 31);
    const int64_t x = (int64_t)(m ^ ((uint64_t)sg << 32 | sg)) - (int64_t)(int32_t)sg;
    l = (int32_t)(uint32_t)x;
    h = (int32_t)(x >> 32) + (int32_t)((uint32_t)l >> 31);
}

// the limbs of the negative (-2^31 has none in 32 bits: its limb becomes 2^31 - 1, one unit of 2^-60 off)
__device__ __forceinline__ void fx_neg(int32_t h, int32_t l, int32_t &nh, int32_t &nl)
{
    nh = -h;
    nl = -max(-2147483647, l);
}

// a += U v (BACK = false) or a -= U^+ v (BACK = true); w: the link's limbs, code and f: its exponent and
// balance (fx_take_code), v: the words of the vector's six doubles
// COUNT: the hop counts towards B
template <bool BACK, bool COUNT>
__device__ __forceinline__ void fx_hop(FxAcc &a, const uint32_t (&w)[36], uint32_t code, uint32_t f, const uint32_t (&v)[12])
{
    uint32_t top = 0, low = 0x7fffffffu;
#pragma unroll
    for (int k = 0; k < 6; k++) {
        const uint32_t m = v[2 * k + 1] & 0x7fffffffu;
        top = max(top, m);
        if (COUNT) low = min(low, m);
    }
    const uint32_t ev = top >> 20, e = code ? code + ev : 0u;
    if (ev - kFxMinExp >= 0x7ffu - kFxMinExp || e - kFxELo - 1u > kFxEHi - kFxELo - 1u) {
        // a link of zeros, or a vector of zeros unless the link holds doubles (an infinity or NaN among them,
        // maybe), contributes nothing; anything else here is left to FP64
        uint32_t any = 0;
#pragma unroll
        for (int k = 0; k < 6; k++) any |= (v[2 * k + 1] & 0x7fffffffu) | v[2 * k];
        a.bad |= code == kFxRaw || (any != 0 && (code != 0 || ev == 0x7ffu));
        return;
    }
    if (e > a.E) {
        fx_shift(a, e - a.E);
        a.E = e;
    }
    const uint32_t t = a.E - code; // the vector's exponent in these sums, >= ev
    if (COUNT) a.B += f * __funnelshift_rc((low & 0xfffffu) | 0x100000u, 0u, t - (low >> 20));
    int32_t h[6], l[6], nh[3], nl[3];
#pragma unroll
    for (int k = 0; k < 6; k++) fx_limbs(v[2 * k], v[2 * k + 1], t, BACK ? 0xffffffffu : 0u, h[k], l[k]);
    // the component that enters with both signs, negated: im forward, re backward
#pragma unroll
    for (int j = 0; j < 3; j++) fx_neg(h[2 * j + (BACK ? 0 : 1)], l[2 * j + (BACK ? 0 : 1)], nh[j], nl[j]);
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const int q = BACK ? 3 * j + i : 3 * i + j;
            const int32_t url = (int32_t)w[4 * q], urh = (int32_t)w[4 * q + 1];
            const int32_t uil = (int32_t)w[4 * q + 2], uih = (int32_t)w[4 * q + 3];
            const int r = 2 * j, m = 2 * j + 1;
            // forward: re += ur vr + ui (-vi), im += ur vi + ui vr
            // backward (h, l hold -v): re += ur (-vr) + ui (-vi), im += ur (-vi) + ui vr
            const int32_t ah = BACK ? h[m] : nh[j], al = BACK ? l[m] : nl[j];
            const int32_t bh = BACK ? nh[j] : h[r], bl = BACK ? nl[j] : l[r];
            int64_t &Hr = a.H[2 * i], &Hi = a.H[2 * i + 1], &Mr = a.M[2 * i], &Mi = a.M[2 * i + 1];
            Hr += (int64_t)urh * h[r];
            Hr += (int64_t)uih * ah;
            Mr += (int64_t)urh * l[r];
            Mr += (int64_t)url * h[r];
            Mr += (int64_t)uih * al;
            Mr += (int64_t)uil * ah;
            Hi += (int64_t)urh * h[m];
            Hi += (int64_t)uih * bh;
            Mi += (int64_t)urh * l[m];
            Mi += (int64_t)url * h[m];
            Mi += (int64_t)uih * bl;
            Mi += (int64_t)uil * bh;
        }
    fx_fold(a);
}

// sum over the DS lanes that share a site (32 / DS apart), in every one of them
template <int DS>
__device__ __forceinline__ void fx_combine(FxAcc &a)
{
#pragma unroll
    for (int off = 16; off >= 32 / DS; off >>= 1) {
        const uint32_t eo = __shfl_xor_sync(0xffffffffu, a.E, off);
        a.bad |= __shfl_xor_sync(0xffffffffu, (int)a.bad, off) != 0;
        if (eo > a.E) {
            fx_shift(a, eo - a.E);
            a.E = eo;
        }
        a.B += __shfl_xor_sync(0xffffffffu, a.B, off);
#pragma unroll
        for (int k = 0; k < 6; k++) {
            a.H[k] += __shfl_xor_sync(0xffffffffu, a.H[k], off);
            a.M[k] += (int64_t)__shfl_xor_sync(0xffffffffu, (uint32_t)a.M[k], off);
        }
        fx_fold(a);
    }
}

// (H 2^32 + M) 2^(E - 2132) as a double, to nearest, on integers: FP64 operations (four per component with exact
// splittings of the words) took 13 % of the normal operator's time at 2 a clock and SM
__device__ __forceinline__ double fx_value(int64_t H, uint32_t M, uint32_t E)
{
    // magnitude of the 96-bit sum H 2^32 + M as words x2 x1 x0
    const uint32_t sg = (uint32_t)((int32_t)(H >> 32) >> 31);
    uint32_t x0 = M ^ sg;
    uint64_t xh = (uint64_t)H ^ ((uint64_t)sg << 32 | sg);
    xh += (uint64_t)(sg & (uint32_t)(x0 == 0xffffffffu)); // + 1, carried
    x0 -= sg;
    uint32_t x2 = (uint32_t)(xh >> 32), x1 = (uint32_t)xh;
    int top = 95;
#pragma unroll
    for (int i = 0; i < 2; i++) {
        const bool z = x2 == 0;
        x2 = z ? x1 : x2;
        x1 = z ? x0 : x1;
        x0 = z ? 0u : x0;
        top -= z ? 32 : 0;
    }
    const int lz = __clz((int)x2);
    const uint32_t m1 = __funnelshift_l(x1, x2, lz), m0 = __funnelshift_l(x0, x1, lz); // leading bit on top
    // (the leading bit adds one to the exponent field, a carry of the rounding another)
    const int e = (int)E + top - lz - 2132 + 1023 - 1;
    uint64_t m = (uint64_t)(m1 >> 11) << 32 | __funnelshift_r(m0, m1, 11);
    m += (m0 >> 10) & 1u;
    m += (uint64_t)((uint32_t)e << 20 | (sg & 0x80000000u)) << 32;
    return x2 ? __longlong_as_double((long long)m) : 0.0;
}
__device__ __forceinline__ double fx_value(const FxAcc &a, int k) { return fx_value(a.H[k], (uint32_t)a.M[k], a.E); }

}  // namespace hisq
