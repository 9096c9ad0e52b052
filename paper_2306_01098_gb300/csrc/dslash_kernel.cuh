// dslash_kernel.cuh -- the HISQ staggered Dslash (Sec. 5.1) on one parity, all storage precisions.
//
//   out(x) = sum_mu [ X_mu(x) phi(x+mu) - X_mu(x-mu)^+ phi(x-mu)
//                   + W_mu(x) phi(x+3mu) - W_mu(x-3mu)^+ phi(x-3mu) ]      (x of parity p)
// with the staggered phases and the antiperiodic time boundary folded into the stored
// links (18 reals) or applied here (12 reals: rows 0 and 1 carry the sign, row 2 is
// rebuilt and signed in registers).
//
// Work decomposition
//   * NR right-hand sides per thread (the paper's N_inner loop, Sec. 5.1): every link is
//     loaded once per NR vectors.  The groups of NR right-hand sides (N_outer) are the
//     fastest index of the block number, so the blocks that read one tile of links run
//     together and only the first takes the links from HBM.
//   * Launch order of the sites: storage order, or with z and t interchanged (t runs
//     fastest among the planes).  A site's +-1/+-3 neighbours along the slowest launch
//     dimension were touched 1 to 3 slowest-dimension slices earlier; interchanging z and
//     t when Nt < Nz shrinks that reuse distance, and with it the L2 footprint that keeps
//     neighbour spinors of many right-hand sides resident.  Link stores too large for L2
//     are then read with an evict-first policy so that the streamed links do not displace
//     the spinors, where links go through registers; copies to shared memory (PipeShape)
//     take the ordinary priority.
//   * DS threads per site (1, 2 or 4), each taking 4/DS of the directions; the partial sums
//     meet through warp shuffles.  On small lattices one thread per site leaves a single
//     short wave whose duration is the latency of 16 dependent gathers; splitting the
//     directions multiplies the loads in flight.
//   * Links (PL) stream through with L1-bypassing 16-byte loads, read once per application;
//     neighbour spinors (PV) are gathered through L1/L2, where their 16-fold reuse happens.
//     PL and PV differ only for 16-bit links with FP32 vectors.
//   * FP64 with 18 reals runs on integers (fixed.cuh), twice as fast as FP64 multiply-adds on
//     this GPU; sites whose components would be less precise than theirs go to FP64.  12 reals stay in
//     FP64 (their third row is rebuilt in it).
// Optional epilogue (normal operator, Sec. 3.2 applyMdaggM):
//   EPI = 1: out = m4 * p - D in,   and <p, out> reduced in FP64 per right-hand side;
//   EPI = 2: the same and also |r|^2, <r, out> and <out, out> (four values per right-hand
//            side, from which the CG finishing step gets alpha and the next |r|^2);
//   EPI = 3: out = m4 * p - D in as canonical FP64, no dot products (hisq_mdagm; a kernel of its own, as
//            its store cost the solvers' EPI = 1 up to 2 %: two sides, 16-bit links, 32^3 x 8, 15.6 against 15.3 ms).
// Batches: one launch over the lattices of a batch, each with its own geometry and links
// (one right-hand side per lattice); a block finds its lattice in the batch table.
#pragma once

#include <algorithm>

#include "arith.cuh"
#include "dslash.cuh"
#include "fixed.cuh"
#include "reduce.cuh"

namespace hisq {

// dot products per right-hand side reduced by an epilogue
template <int EPI> struct EpiDots { static constexpr int n = EPI == 2 ? 4 : 1; };

// the output is canonical FP64: EPI = 3, or a plain Dslash of one lattice that says so
template <int EPI, bool PLAIN64>
__device__ __forceinline__ bool canonical_out(const DslashArgs &a)
{
    if constexpr (EPI == 3) return true;
    else return EPI == 0 && PLAIN64 && a.out64;
}

// |v|^2 and |o|^2 of FP32 records in float arithmetic, returned as floats
__device__ __forceinline__ float vec_norm2f(const FloatArith::Vec &v)
{
    float d = 0.f;
#pragma unroll
    for (int i = 0; i < 6; i++) d = fmaf(v.v[i], v.v[i], d);
    return d;
}
__device__ __forceinline__ float acc_norm2f(const FloatArith::Acc &o)
{
    float d = 0.f;
#pragma unroll
    for (int i = 0; i < 6; i++) d = fmaf(o.v[i], o.v[i], d);
    return d;
}

// |v|^2 of a vector: float arithmetic for the float types, double otherwise
template <class T>
__device__ __forceinline__ double vec_norm2(const typename T::Vec &v)
{
    if constexpr (std::is_same<typename T::Vec, FloatArith::Vec>::value) {
        float d = 0.f;
#pragma unroll
        for (int i = 0; i < 6; i++) d = fmaf(v.v[i], v.v[i], d);
        return (double)d;
    } else {
        double d = 0.0;
#pragma unroll
        for (int i = 0; i < 6; i++) {
            const double c = T::vcomp(v, i);
            d = fma(c, c, d);
        }
        return d;
    }
}

// |o|^2 of an accumulator: float arithmetic for the float types, double otherwise
template <class T>
__device__ __forceinline__ double acc_norm2(const typename T::Acc &o)
{
    if constexpr (std::is_same<typename T::Acc, FloatArith::Acc>::value) {
        float d = 0.f;
#pragma unroll
        for (int i = 0; i < 6; i++) d = fmaf(o.v[i], o.v[i], d);
        return (double)d;
    } else {
        double d = 0.0;
#pragma unroll
        for (int i = 0; i < 6; i++) {
            const double c = T::comp(o, i);
            d = fma(c, c, d);
        }
        return d;
    }
}

// bytes between the right-hand sides of the output
template <int EPI, bool PLAIN64>
__device__ __forceinline__ size_t out_stride(const DslashArgs &a)
{
    return canonical_out<EPI, PLAIN64>(a) ? (size_t)a.g.Vh * 48 : a.rhs_bytes;
}

// vector load: the read-only path, or (COH) ordinary loads for vectors that other blocks of
// the same launch write between grid barriers
template <class T, bool COH>
__device__ __forceinline__ void vec_load(const char *base, uint32_t s, typename T::Vec &v)
{
    if constexpr (COH) T::load_coh(base, s, v);
    else T::load(base, s, v);
}

// ---------------------------------------------------------------- hops through shared memory
// The hops of a site, each thread for itself: the link and the NR vectors of a hop are copied
// asynchronously into the thread's part of one of ST stages, ST hops before they are used, so that
// the requests in flight cost no registers and nothing keeps a warp from running ahead.  No thread
// reads another's part: the only waits are the thread's own (cp.async groups, one per hop).
// Used where registers limit the warps in flight: the fixed-point FP64 sites (a hop's link is 36
// registers; 137 -> 131 us for the 32^3 x 8 normal operator, 905 -> 853 us for a 64^3 x 16 Dslash, both
// before their sums were held to FP64 component by component: 137 and 920 us now) and FP32 vectors with four or more right-hand sides a thread (or two, with
// the third rows of 12-real links to rebuild): 32^3 x 16, 16-bit links, 8 right-hand sides, 159 -> 142 ms
// a solve.  With one or two right-hand sides of 18-real links the extra trip costs more than the
// registers do (FP32 64^3 x 16 467 -> 479 us, float pairs 18 x 22 x 14 x 10, three sides, 83 -> 94 us).
// Two stages fill the memory pipe; with four threads per site (lattices that leave the chip half
// empty) all four hops of a thread are in flight at once.
template <int PL, int PV, int NREAL, int NR, int DS>
struct PipeShape {
    static constexpr bool FX = PL == HISQ_F64 && NREAL == 18;
    static constexpr bool on = FX || (PV != HISQ_F64 && PV != HISQ_F64X && NR >= (NREAL == 12 ? 2 : 4));
    static constexpr int LB = NREAL == 18 ? LinkBytes<PL>::b18 : LinkBytes<PL>::b12;
    static constexpr int VB = Prec<PV>::SB;
    static constexpr int stage = LB + NR * VB; // bytes per thread and stage
    static constexpr int ST = FX && NR == 1 && DS == 4 ? 4 : 2;
    static constexpr int bytes = on ? ST * stage : 0; // per thread
};

template <int PL, int PV, int NREAL, int NR, int DS, bool LL1>
__device__ __forceinline__ void pipe_issue(const DslashArgs &a, const Geom &g, const char *links, size_t slot_bytes,
                                           const char *in, const Site &c, uint32_t s, int mu, int h, char *st)
{
    using P = PipeShape<PL, PV, NREAL, NR, DS>;
    const uint32_t n = blockDim.x, t = threadIdx.x;
    const int k = h == 0 ? 1 : h == 1 ? -1 : h == 2 ? 3 : -3, type = h >> 1;
    const bool back = h & 1;
    uint32_t sn;
    if constexpr (DS > 1) {
        sn = neighbour_any(g, c, s, mu, k);
    } else {
        bool wrap;
        sn = neighbour(g, c, s, mu, k, wrap);
    }
    const int lp = back ? 1 - a.p : a.p;
    const uint32_t sl = back ? sn : s, lane = sl & 31;
    const char *blk = links + (size_t)((lp * 2 + type) * 4 + mu) * slot_bytes + (size_t)(sl >> 5) * (32 * P::LB);
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(st);
    constexpr int NQ = P::LB / 16, TB = P::LB % 16;
#pragma unroll
    for (int q = 0; q < NQ; q++) cp_async<16, LL1>(dst + (q * n + t) * 16, blk + q * 512 + lane * 16);
    if constexpr (TB > 0) cp_async<TB, true>(dst + NQ * n * 16 + t * TB, blk + NQ * 512 + lane * TB);
    constexpr int VQ = P::VB / 16, VT = P::VB % 16;
#pragma unroll
    for (int r = 0; r < NR; r++) {
        const char *v = in + (size_t)r * a.rhs_bytes;
        const uint32_t d = dst + n * (uint32_t)(P::LB + r * P::VB);
#pragma unroll
        for (int q = 0; q < VQ; q++) cp_async<16, true>(d + (q * n + t) * 16, v + Prec<PV>::chunk_off(sn, q));
        if constexpr (VT > 0) cp_async<VT, true>(d + VQ * n * 16 + t * VT, v + Prec<PV>::chunk_off(sn, VQ));
    }
}

// the stages of one site's hops: for m = 0 .. 4/DS - 1 and h = 0 .. 3 (hops +1, -1, +3, -3 along
// direction part 4/DS + m): link(h, w), vec(h, r, x) for every r, then next(m, h)
template <int PL, int PV, int NREAL, int NR, int DS, bool LL1>
struct HopPipe {
    using P = PipeShape<PL, PV, NREAL, NR, DS>;
    static constexpr int NMU = 4 / DS, ST = P::ST;
    const DslashArgs &a;
    const Geom &g;
    const char *links;
    size_t slot_bytes;
    const char *in;
    const Site &c;
    uint32_t s;
    int mu0;
    char *smem;

    __device__ __forceinline__ char *stage(int h) const { return smem + (size_t)(h % ST) * blockDim.x * P::stage; }
    __device__ __forceinline__ void issue(int mu, int h)
    {
        pipe_issue<PL, PV, NREAL, NR, DS, LL1>(a, g, links, slot_bytes, in, c, s, mu, h, stage(h));
    }
    __device__ __forceinline__ void start()
    {
#pragma unroll
        for (int h = 0; h < ST; h++) {
            issue(mu0, h);
            cp_commit();
        }
    }
    __device__ __forceinline__ void link(int h, uint32_t (&w)[P::LB / 4])
    {
        cp_wait<ST - 1>();
        stage_read<P::LB>(stage(h), blockDim.x, threadIdx.x, w);
    }
    __device__ __forceinline__ void vec(int h, int r, uint32_t (&x)[P::VB / 4])
    {
        stage_read<P::VB>(stage(h) + blockDim.x * (uint32_t)(P::LB + r * P::VB), blockDim.x, threadIdx.x, x);
    }
    // hop (m, h) has been used: its stage takes the one ST hops later
    __device__ __forceinline__ void next(int m, int h)
    {
        const int mn = m + ((h + ST) >> 2);
        if (mn < NMU) issue(mu0 + mn, (h + ST) & 3);
        cp_commit();
    }
};

// ---------------------------------------------------------------- FP64 sites in fixed point
// out += hop (mu, type, back) of D in at site s in FP64; the link as doubles, - U^+ v turned into U v for the same
// multiply-adds
static __device__ __forceinline__ void fx_hop_f64(const DslashArgs &a, const Geom &g, const char *links, size_t slot_bytes,
                                                  const char *in, uint32_t s, int mu, int type, bool back,
                                                  Prec<HISQ_F64>::Acc &out)
{
    const uint32_t sn = neighbour_any(g, site_coords(g, s, a.p), s, mu, back ? (type ? -3 : -1) : (type ? 3 : 1));
    const uint32_t sl = back ? sn : s;
    const char *slot = links + (size_t)(((back ? 1 - a.p : a.p) * 2 + type) * 4 + mu) * slot_bytes;
    uint32_t w[36];
    load_link_words<144>(slot, sl, w);
    Prec<HISQ_F64>::Link U;
    Prec<HISQ_F64>::Vec v;
    fx_decode_link(w, reinterpret_cast<const uint64_t *>(slot + (size_t)g.VhPad * 144)[sl], U.v);
    Prec<HISQ_F64>::load(in, sn, v);
    if (back) {
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = 0; j < i; j++)
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    const double x = U.v[2 * (3 * i + j) + k];
                    U.v[2 * (3 * i + j) + k] = U.v[2 * (3 * j + i) + k];
                    U.v[2 * (3 * j + i) + k] = x;
                }
#pragma unroll
        for (int i = 0; i < 9; i++) U.v[2 * i] = -U.v[2 * i];
    }
    Prec<HISQ_F64>::hop<false, false>(out, U, v);
}

// D in in FP64 at the sites of the warp's lanes in m (each lane's own s and in; all lanes call), for sites that
// hold what the fixed-point format cannot (infinities, NaN, extreme magnitudes) or whose components it does
// not hold to FP64's precision for certain.  Few sites (the rule): two at a time, a lane for every hop; a lane alone
// with its site's 16 hops keeps its block for 50 to 85 us (a fifth of the warps with such a site on 32^3 x 8:
// 163 us that way, 88 us so, 66 us without).  More than half of them (a vector of one colour): every lane its
// own site, as its links are then read as whole lines (214 us so, 364 us two at a time).
static __device__ __noinline__ void fx_sites_f64(const DslashArgs &a, const Geom &g, const char *links, size_t slot_bytes,
                                                 const char *in, uint32_t s, uint32_t m, double (&out)[6])
{
    const int lane = threadIdx.x & 31;
    Prec<HISQ_F64>::Acc acc;
    if (__popc(m) > 16) {
        if (!(m >> lane & 1u)) return;
        Prec<HISQ_F64>::zero(acc);
#pragma unroll 1
        for (int q = 0; q < 16; q++) fx_hop_f64(a, g, links, slot_bytes, in, s, q >> 2, (q >> 1) & 1, q & 1, acc);
#pragma unroll
        for (int k = 0; k < 6; k++) out[k] = acc.v[k];
        return;
    }
#pragma unroll 1
    while (m) {
        const int l0 = __ffs((int)m) - 1;
        m &= m - 1;
        const int l1 = m ? __ffs((int)m) - 1 : l0;
        m &= m - 1;
        const int src = lane < 16 ? l0 : l1;
        const uint32_t ss = __shfl_sync(0xffffffffu, s, src);
        const char *si = reinterpret_cast<const char *>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(in), src));
        Prec<HISQ_F64>::zero(acc);
        fx_hop_f64(a, g, links, slot_bytes, si, ss, (lane >> 2) & 3, (lane >> 1) & 1, lane & 1, acc);
#pragma unroll
        for (int k = 0; k < 6; k++) {
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) acc.v[k] += __shfl_xor_sync(0xffffffffu, acc.v[k], off);
            const double x0 = __shfl_sync(0xffffffffu, acc.v[k], 0), x1 = __shfl_sync(0xffffffffu, acc.v[k], 16);
            if (lane == l0) out[k] = x0;
            else if (lane == l1) out[k] = x1;
        }
    }
}

// D in at site s for NR right-hand sides in fixed point (fixed.cuh), the directions of one of DS
// threads per site, summed over these threads
template <int NR, int DS, bool LL1>
__device__ __forceinline__ void fx_site(const DslashArgs &a, const Geom &g, const char *links, size_t slot_bytes,
                                        const char *in, uint32_t s, bool live, int part,
                                        Prec<HISQ_F64>::Acc (&out)[NR])
{
    FxAcc acc[NR];
#pragma unroll
    for (int r = 0; r < NR; r++) fx_zero(acc[r]);
    if (live) {
        extern __shared__ __align__(16) char pipe_smem[];
        const Site c = site_coords(g, s, a.p);
        HopPipe<HISQ_F64, HISQ_F64, 18, NR, DS, LL1> pipe{a, g, links, slot_bytes, in, c, s, part * (4 / DS), pipe_smem};
        pipe.start();
#pragma unroll 1
        for (int m = 0; m < 4 / DS; m++)
#pragma unroll
            for (int h = 0; h < 4; h++) {
                uint32_t w[36];
                pipe.link(h, w);
                uint32_t f;
                const uint32_t code = fx_take_code(w, f);
#pragma unroll
                for (int r = 0; r < NR; r++) {
                    uint32_t x[12];
                    pipe.vec(h, r, x);
                    if (h == 0) fx_hop<false, true>(acc[r], w, code, f, x);
                    else if (h == 1) fx_hop<true, true>(acc[r], w, code, f, x);
                    else if (h == 2) fx_hop<false, false>(acc[r], w, code, f, x);
                    else fx_hop<true, false>(acc[r], w, code, f, x);
                }
                pipe.next(m, h);
            }
    }
    bool left = false;
#pragma unroll
    for (int r = 0; r < NR; r++) {
        if constexpr (DS > 1) fx_combine<DS>(acc[r]);
#pragma unroll
        for (int k = 0; k < 6; k++) out[r].v[k] = fx_value(acc[r], k);
        acc[r].bad = fx_left(acc[r]);
        left |= acc[r].bad;
    }
    if (__any_sync(0xffffffffu, left)) {
#pragma unroll
        for (int r = 0; r < NR; r++) {
            // (the first of a site's threads goes on with the result)
            const uint32_t m = __ballot_sync(0xffffffffu, acc[r].bad && part == 0);
            if (m) fx_sites_f64(a, g, links, slot_bytes, in + (size_t)r * a.rhs_bytes, s, m, out[r].v);
        }
    }
}

// One work item: the sites of one tile (a.bs threads, DS per site; this thread is
// number tid of the tile) for the NR right-hand sides whose vectors start at in/out/pv/rv
// (consecutive right-hand sides a.rhs_bytes apart); geometry g, link store `links`.
// Epilogue dot products are added to dots (value j of right-hand side r at
// dots[r * EpiDots<EPI>::n + j]).  With an epilogue, pv, rv and the output are addressed at
// site s - ebase (ebase = 0: the whole field; else a block's own range, e.g. in shared memory).
// PF: issue the loads of all four hops of a direction before their products (more requests
// in flight per thread, more registers).
// RG > 1 (with DS = 1): RG consecutive threads share a site, thread g of them taking the NR
// right-hand sides g NR .. g NR + NR - 1 from the given ones; their loads of the site's links
// are the same addresses in the same instruction (one request), so a link is fetched once
// for all NR RG right-hand sides with 1/RG of the accumulators per thread.
// LL1: links allocate in L1 (right-hand-side groups of one block read the same links).
// PIPE: the hops' operands come through shared memory (HopPipe); else through registers.
// PLAIN64: a plain Dslash may write canonical FP64 (DslashArgs::out64).
template <int PL, int PV, int NREAL, int NR, int EPI, int DS, bool COH = false, bool PF = false, int RG = 1,
          class DT = double, bool LL1 = false, bool PIPE = false, bool PLAIN64 = false>
__device__ __forceinline__ void dslash_item(const DslashArgs &a, const Geom &g, const char *links, size_t slot_bytes,
                                            std::conditional_t<std::is_same<DT, FF>::value, float, double> sc0,
                                            std::conditional_t<std::is_same<DT, FF>::value, float, double> sc1,
                                            const char *in, char *outp, const char *pvp,
                                            const char *rvp, const double *m4r, uint32_t tile,
                                            DT (&dots)[NR * EpiDots<EPI>::n], uint32_t tid = threadIdx.x,
                                            uint32_t ebase = 0)
{
    static_assert(RG == 1 || DS == 1, "right-hand side groups share a site only with one thread per direction set");
    constexpr int ND = EpiDots<EPI>::n;
    // DT = FF (FP32 vectors inside the persistent CG kernel): float-float dot sums, float
    // scales (sc0, sc1) and the float m4f, so that no FP64 conversion runs per site
    constexpr bool FFD = std::is_same<DT, FF>::value;
    static_assert(!FFD || std::is_same<typename Prec<PV>::Vec, FloatArith::Vec>::value,
                  "float-float dot sums are for FP32 iteration vectors");
    using T = Prec<PV>;  // vectors and arithmetic
    using TL = Prec<PL>; // link storage
    constexpr int LB = NREAL == 18 ? LinkBytes<PL>::b18 : LinkBytes<PL>::b12;
    constexpr bool TWO = (PL == HISQ_F16 || PL == HISQ_BF16 || NREAL == 12);
    // directions summed apart: always for float pairs; for FP32 with one or four right-hand sides (with
    // two, the registers would cost more than the additions: 14 shifts, FP32 32^3 x 8, 60 -> 67 ms), so that
    // a site's error depends less on how many threads share it (measured 1.9e-7 with one running
    // sum, 1.2e-7 apart; the gathers hide the 24 additions)
    constexpr bool SPLIT = T::kSplitDirections || (PL == HISQ_F32 && (NR == 1 || NR == 4) && !TWO && !COH && DS < 4);
    constexpr int NMU = 4 / DS;
    const uint32_t gt = tile * (uint32_t)a.bs + tid;
    // site number in launch order, and this thread's directions: with DS > 1 a warp holds 32 / DS
    // sites, lanes in groups of 32 / DS per part, so that a quarter-warp's 16-byte accesses still fall
    // into one line (lanes of one site side by side spread them over DS)
    constexpr uint32_t kSites = 32 / DS;
    const uint32_t u = DS > 1 ? (gt >> 5) * kSites + (gt & (kSites - 1)) : gt / RG;
    const int part = DS > 1 ? (int)((gt & 31) / kSites) : 0;
    if constexpr (RG > 1) {
        const size_t goff = (size_t)(gt % RG) * NR * a.rhs_bytes;
        in += goff;
        outp += (size_t)(gt % RG) * NR * out_stride<EPI, PLAIN64>(a);
        if (pvp) pvp += goff;
        if (rvp) rvp += goff;
        if (m4r) m4r += (gt % RG) * NR;
    }
    const bool live = u < g.Vh;
    uint32_t s = u;
    if (a.zt) { // u = ((z Nt + t) Ps + i)  ->  s = ((t Nz + z) Ps + i), Ps = sites of one plane
        const uint32_t plane = g.dp.div(u);
        const uint32_t z = g.dt.div(plane);
        s = ((plane - z * (uint32_t)g.n[3]) * (uint32_t)g.n[2] + z) * g.sz + (u - plane * g.sz);
    }
    typename T::Acc out[NR];
#pragma unroll
    for (int r = 0; r < NR; r++) T::zero(out[r]);

    // FP64 with 18 reals: in fixed point, summed over the site's threads there
    constexpr bool FX = PL == HISQ_F64 && NREAL == 18;
    static_assert(!FX || PIPE, "the fixed-point sites read their operands from shared memory");
    if constexpr (FX) fx_site<NR, DS, LL1>(a, g, links, slot_bytes, in, s, live, part, out);
    else if (live) {
        const Site c = site_coords(g, s, a.p);
        typename T::Acc acc[TWO ? 2 : 1][NR];
#pragma unroll
        for (int t = 0; t < (TWO ? 2 : 1); t++)
#pragma unroll
            for (int r = 0; r < NR; r++) T::zero(acc[t][r]);

        if constexpr (PIPE) {
            extern __shared__ __align__(16) char pipe_smem[];
            HopPipe<PL, PV, NREAL, NR, DS, LL1> pipe{a, g, links, slot_bytes, in, c, s, part * NMU, pipe_smem};
            pipe.start();
#pragma unroll 1
            for (int m = 0; m < NMU; m++) {
                typename T::Acc dacc[SPLIT ? NR : 1];
                if constexpr (SPLIT) {
#pragma unroll
                    for (int r = 0; r < NR; r++) T::zero(dacc[r]);
                }
#pragma unroll
                for (int h = 0; h < 4; h++) {
                    uint32_t w[LB / 4];
                    pipe.link(h, w);
                    typename T::Link U;
                    TL::template unpack<NREAL>(w, U);
                    if constexpr (NREAL == 12) {
                        const int mu = part * NMU + m;
                        bool wrap;
                        neighbour(g, c, s, mu, h == 0 ? 1 : h == 1 ? -1 : h == 2 ? 3 : -3, wrap);
                        T::rebuild(U, (eta_neg(c, mu) != 0) ^ (mu == 3 && wrap));
                    }
#pragma unroll
                    for (int r = 0; r < NR; r++) {
                        uint32_t x[T::SB / 4];
                        pipe.vec(h, r, x);
                        typename T::Vec v;
                        T::vec_words(x, v);
                        typename T::Acc &dst = SPLIT ? dacc[SPLIT ? r : 0] : acc[TWO ? h >> 1 : 0][r];
                        if (h & 1) T::template hop<true, true>(dst, U, v);
                        else T::template hop<false, false>(dst, U, v);
                    }
                    pipe.next(m, h);
                }
                if constexpr (SPLIT) {
#pragma unroll
                    for (int r = 0; r < NR; r++) T::add_acc(acc[0][r], dacc[r]);
                }
            }
        } else {
#pragma unroll
            for (int m = 0; m < NMU; m++) {
                const int mu = part * NMU + m;
                typename T::Acc dacc[SPLIT ? NR : 1];
                if constexpr (SPLIT) {
#pragma unroll
                    for (int r = 0; r < NR; r++) T::zero(dacc[r]);
                }
                if constexpr (PF) {
                    // the loads of all four hops first (8 to 12 independent requests per thread in
                    // flight at once), then their products
                    uint32_t w[4][LB / 4];
                    typename T::Vec v[4][NR];
                    bool wrap[4];
#pragma unroll
                    for (int h = 0; h < 4; h++) {
                        const int k = h == 0 ? 1 : h == 1 ? -1 : h == 2 ? 3 : -3;
                        const int type = h >> 1;
                        const bool back = h & 1;
                        const uint32_t sn = neighbour(g, c, s, mu, k, wrap[h]);
                        const int lp = back ? 1 - a.p : a.p;
                        const char *slot = links + (size_t)((lp * 2 + type) * 4 + mu) * slot_bytes;
                        load_link_words<LB, LL1>(slot, back ? sn : s, w[h], NR > 1 && a.stream_links != 0);
#pragma unroll
                        for (int r = 0; r < NR; r++) vec_load<T, COH>(in + (size_t)r * a.rhs_bytes, sn, v[h][r]);
                    }
#pragma unroll
                    for (int h = 0; h < 4; h++) {
                        const int type = h >> 1;
                        const bool back = h & 1;
                        typename T::Link U;
                        TL::template unpack<NREAL>(w[h], U);
                        if constexpr (NREAL == 12) T::rebuild(U, (eta_neg(c, mu) != 0) ^ (mu == 3 && wrap[h]));
#pragma unroll
                        for (int r = 0; r < NR; r++) {
                            typename T::Acc &dst = SPLIT ? dacc[SPLIT ? r : 0] : acc[TWO ? type : 0][r];
                            if (back) T::template hop<true, true>(dst, U, v[h][r]);
                            else T::template hop<false, false>(dst, U, v[h][r]);
                        }
                    }
                } else {
#pragma unroll
                    for (int h = 0; h < 4; h++) {
                        const int k = h == 0 ? 1 : h == 1 ? -1 : h == 2 ? 3 : -3;
                        const int type = h >> 1;
                        const bool back = h & 1;
                        bool wrap;
                        const uint32_t sn = neighbour(g, c, s, mu, k, wrap);
                        const int lp = back ? 1 - a.p : a.p;
                        const char *slot = links + (size_t)((lp * 2 + type) * 4 + mu) * slot_bytes;
                        uint32_t w[LB / 4];
                        load_link_words<LB, LL1>(slot, back ? sn : s, w, NR > 1 && a.stream_links != 0);
                        typename T::Link U;
                        TL::template unpack<NREAL>(w, U);
                        if constexpr (NREAL == 12) T::rebuild(U, (eta_neg(c, mu) != 0) ^ (mu == 3 && wrap));
#pragma unroll
                        for (int r = 0; r < NR; r++) {
                            typename T::Vec v;
                            vec_load<T, COH>(in + (size_t)r * a.rhs_bytes, sn, v);
                            typename T::Acc &dst = SPLIT ? dacc[SPLIT ? r : 0] : acc[TWO ? type : 0][r];
                            if (back) T::template hop<true, true>(dst, U, v);
                            else T::template hop<false, false>(dst, U, v);
                        }
                    }
                }
                if constexpr (SPLIT) {
#pragma unroll
                    for (int r = 0; r < NR; r++) {
                        if (m == 0) acc[0][r] = dacc[r];
                        else T::add_acc(acc[0][r], dacc[r]);
                    }
                }
            }
        }
#pragma unroll
        for (int r = 0; r < NR; r++) {
            if constexpr (TWO) {
                T::axpy_acc(out[r], (typename T::Real)sc0, acc[0][r]);
                T::axpy_acc(out[r], (typename T::Real)sc1, acc[1][r]);
            } else {
                out[r] = acc[0][r];
            }
        }
    }
    // partial sums of the DS threads of a site meet in every one of them
    if constexpr (DS > 1 && !FX) {
#pragma unroll
        for (int off = 16; off >= (int)kSites; off >>= 1)
#pragma unroll
            for (int r = 0; r < NR; r++) T::shfl_xor_add(out[r], off);
    }
    if (live && part == 0) {
#pragma unroll
        for (int r = 0; r < NR; r++) {
            if constexpr (EPI >= 1) {
                typename T::Vec pv;
                vec_load<T, COH>(pvp + (size_t)r * a.rhs_bytes, s - ebase, pv);
                if constexpr (FFD) {
                    T::mdagm_epilogue(out[r], m4r ? a.m4f + (float)m4r[r] : a.m4f, pv);
                    if constexpr (EPI != 3) ff_add(dots[r * ND], T::dotf(pv, out[r]));
                } else {
                    T::mdagm_epilogue(out[r], a.m4 + (m4r ? m4r[r] : 0.0), pv);
                    if constexpr (EPI != 3) dots[r * ND] += T::dot(pv, out[r]);
                }
                if constexpr (EPI == 2) {
                    typename T::Vec rv;
                    vec_load<T, COH>(rvp + (size_t)r * a.rhs_bytes, s - ebase, rv);
                    if constexpr (FFD) {
                        ff_add(dots[r * ND + 1], vec_norm2f(rv));
                        ff_add(dots[r * ND + 2], T::dotf(rv, out[r]));
                        ff_add(dots[r * ND + 3], acc_norm2f(out[r]));
                    } else {
                        dots[r * ND + 1] += vec_norm2<T>(rv);
                        dots[r * ND + 2] += T::dot(rv, out[r]);
                        dots[r * ND + 3] += acc_norm2<T>(out[r]);
                    }
                }
            }
            if (canonical_out<EPI, PLAIN64>(a)) { // the caller's FP64 buffer, without a pass of its own
                double2 *q = reinterpret_cast<double2 *>(outp + (size_t)r * out_stride<EPI, PLAIN64>(a) + (size_t)s * 48);
#pragma unroll
                for (int i = 0; i < 3; i++) q[i] = make_double2(T::canon(out[r], 2 * i), T::canon(out[r], 2 * i + 1));
            } else {
                T::store(outp + (size_t)r * a.rhs_bytes, EPI >= 1 ? s - ebase : s, out[r]);
            }
        }
    }
}

// block sums of the epilogue's dot products (valid on thread 0): float-float or FP64
template <bool FFK, int N, class D>
__device__ __forceinline__ void block_sum_dots(D (&d)[N])
{
    if constexpr (FFK) block_sum_ff<N>(d);
    else block_sum_multi<N>(d);
}
__device__ __forceinline__ double dot_value(const FF &x) { return ff_value(x); }
__device__ __forceinline__ double dot_value(double x) { return x; }

// 256-thread blocks per SM that the registers are limited for.  Left alone the compiler moves the
// loads of all 16 hops to the front of the site (250 registers, 8 warps an SM); the gathers want warps, the
// dot products want registers (limits that leave too few spill 170 to 380 bytes).  FP32 vectors, registers per
// kernel and us per iteration of a solve on 32^3 x 8 and x 16 (uneven batch of 32 lattices: ms):
//   no dot products     48 / 64 / 128 at 1 / 2 / 4 right-hand sides a thread (14-shift FP32 solve 32^3 x 8: 74 ms
//                       without limits, 63 ms with 64 / 80 / 128, 59 ms so)
//   EPI = 1, one side   16-bit links 64: 56.5, 84.1 (48: 59.8, 89.5; no limit 56.3, 86.3, but 422 for 8 groups of one
//                       on x 16, where 64 take 368); FP32 links no limit: 76.1, 124 (64: 76.9, 127; 48: 79.8, 135)
//   EPI = 1, two, four  64 / 128: FP32 links, two 86.8, 147 (80: 97.7, 155), four 123, 199 (no limit 131, 211)
//   EPI = 2, one, two   no limit: 16-bit links 54.3, 82.7 and 80.3, 123 (48: 62.0, 96.2; 64: 88.8, 128)
//   EPI = 2, four       128: 16-bit links, 8 sides 210, 310 (no limit 211, 337)
//   batch               FP32 links no limit: 57.3, EPI = 2 62.4 (48: 59.0, 71.3); 16-bit links 64: 42.6, 48.9 (48: 47.6,
//                       55.6); the kernel without dot products alike, as its time chooses the threads per site of all
// One block less for rebuilt third rows (their EPI = 1 too: FP32 links 64.5, 95.9, no limit 66.1, 95.5).  FP64 and
// float pairs: 128 at one side (float pairs, four sides in groups of one: 437, 802, no limit 520, 962; FP64 batch 133
// ms, no limit 150).
constexpr int min_blocks(int pl, int pv, int nreal, int nr, int epi, bool batch, int rg)
{
    if (pv == HISQ_F64 || pv == HISQ_F64X) return nr == 1 && !(pl == HISQ_F64 && nreal == 12) ? 2 : 1;
    const int less = nreal == 12 ? 1 : 0;
    if (batch) return pl == HISQ_F32 ? 1 : 4 - less;
    if (epi == 2 && nr <= 2) return 1;
    if (epi == 1 && nr <= 2 && rg > 1) return 1;
    if (epi == 1 && nr == 1 && nreal == 18) return pl == HISQ_F32 ? 1 : 4;
    return nr == 1 ? 5 - less : nr == 2 ? 4 - less : nr == 4 ? 2 : 1;
}

// BATCH: the lattices of a batch in one launch (NR = 1; right-hand side k is lattice k).
// RG: groups of right-hand sides sharing a site's threads (dslash_item).
// WG > 1 (no epilogue, one thread per site, RG = 1): the block's threads form WG slices of
// a.bs threads over the same sites, slice g taking the g-th of the block's WG groups of NR
// right-hand sides; their link loads allocate in L1, so one L2 read of a link serves the
// block's WG NR right-hand sides without the registers of WG NR accumulators per thread.
template <int PL, int PV, int NREAL, int NR, int EPI, int DS, bool BATCH, int RG = 1, int WG = 1>
__global__ void __launch_bounds__(kDslashMaxBlock, min_blocks(PL, PV, NREAL, NR, EPI, BATCH, RG)) k_dslash(const DslashArgs a)
{
    static_assert(WG == 1 || (EPI == 0 && DS == 1 && RG == 1 && !BATCH), "block slices: plain Dslash, one thread per site");
    using T = Prec<PV>;
    using TL = Prec<PL>;
    static_assert(std::is_same<typename T::Link, typename TL::Link>::value, "link and vector arithmetic must agree");
    static_assert(!BATCH || NR == 1, "batches take one right-hand side per lattice");
    if (a.skip) { // uniform over the grid: the scalars do not change during the launch
        bool any = false;
        for (int r = 0; r < a.nrhs; r++) any |= a.skip[r].active != 0;
        if (!any) {
            // A launch that carries the loop control (the single-reduction CG epilogue) still
            // closes the iteration: the iteration stamps advance as the finishing step would
            // advance them, so no earlier alpha counts as fresh for the update that follows,
            // and the device loop is told that nothing is active.
            if constexpr (EPI == 2) {
                if (a.red.partials && a.red.ctl && blockIdx.x == 0 && threadIdx.x == 0) {
                    for (int r = 0; r < a.nrhs; r++) a.red.sc[r].it_all++;
                    finish_control(a.red, a.nrhs);
                }
            }
            return;
        }
    }
    constexpr int ND = EpiDots<EPI>::n;
    // FP32 vectors: the epilogue's dot products in float-float pairs, float scales and m4
    // (no FP64 operation per site or per thread; one conversion per block and value)
    constexpr bool FFK = PV == HISQ_F32 && RG == 1;
    using DTK = std::conditional_t<FFK, FF, double>;
    DTK dots[NR * ND];
#pragma unroll
    for (int r = 0; r < NR * ND; r++) dots[r] = DTK{};
    if constexpr (BATCH) {
        // One block per tile; with the epilogue's reduction a resident grid whose blocks
        // stride over the tiles: each tile's dot products go to its own partial (the tile
        // number of its lattice), and a block arrives once, after its last tile, instead of
        // every tile paying the block sum's barriers and the arrival's round trip in a wave
        // of its own.
        __shared__ Geom sg;
        constexpr int d = DS == 1 ? 0 : DS == 2 ? 1 : 2;
        const BatchDesc &B = *a.batch;
        for (uint32_t item = blockIdx.x; item < a.items; item += gridDim.x) {
            int k = 0;
            while (k + 1 < B.n && B.tstart[d][k + 1] <= item) k++;
            const uint32_t tile = item - B.tstart[d][k];
            __syncthreads(); // the previous tile's readers of sg are done
            if (threadIdx.x == 0) sg = B.lat[k].g;
            __syncthreads();
            const size_t off = (size_t)k * a.rhs_bytes;
            const BatchLattice &L = B.lat[k];
            const auto sc0 = [&] { if constexpr (FFK) return L.scale_f[PL][0]; else return L.scale[PL][0]; }();
            const auto sc1 = [&] { if constexpr (FFK) return L.scale_f[PL][1]; else return L.scale[PL][1]; }();
            DTK td[ND];
#pragma unroll
            for (int j = 0; j < ND; j++) td[j] = DTK{};
            dslash_item<PL, PV, NREAL, 1, EPI, DS, false, false, 1, DTK, false, PipeShape<PL, PV, NREAL, 1, DS>::on>(
                a, sg, L.links[PL], L.slot_bytes[PL], sc0, sc1, a.in + off, a.out + off, EPI ? a.pv + off : nullptr,
                EPI == 2 ? a.rv + off : nullptr, a.shift ? a.shift + k : nullptr, tile, td);
            if constexpr (EPI >= 1) {
                if (a.red.partials) {
                    block_sum_dots<FFK, ND>(td);
                    if (threadIdx.x == 0) {
#pragma unroll
                        for (int j = 0; j < ND; j++)
                            a.red.partials[(size_t)(ND * k + j) * a.red.nblocks + tile] = dot_value(td[j]);
                        // partials of lattice k beyond its own tiles are zero
                        if (tile == 0)
                            for (int j = 0; j < ND; j++)
                                for (int i = (int)(B.tstart[d][k + 1] - B.tstart[d][k]); i < a.red.nblocks; i++)
                                    a.red.partials[(size_t)(ND * k + j) * a.red.nblocks + i] = 0.0;
                    }
                }
            }
        }
        if constexpr (EPI >= 1) {
            // the partials are in place: arrive (no values of its own), the last block finishes
            if (a.red.partials) grid_reduce<ND>(a.red, nullptr, 0, 0, ND * a.nrhs, 0);
        }
    } else {
        // gridDim.x is a multiple of the group count, so a block keeps one group of right-hand
        // sides while it strides over the work items (site tile, group)
        // (with WG slices, a block group is WG consecutive groups, slice g of the block taking
        // the g-th; a.bs is then the threads of one slice)
        const uint32_t ngroups = (uint32_t)(a.nrhs / (NR * RG * WG));
        const uint32_t slice = WG > 1 ? threadIdx.x / (uint32_t)a.bs : 0u;
        const uint32_t tid = WG > 1 ? threadIdx.x - slice * (uint32_t)a.bs : threadIdx.x;
        const int rhs0 = (int)((blockIdx.x % ngroups) * WG + slice) * NR * RG;
        const size_t off = (size_t)rhs0 * a.rhs_bytes;
        const auto sc0 = [&] { if constexpr (FFK) return a.scale_f[0]; else return a.scale[0]; }();
        const auto sc1 = [&] { if constexpr (FFK) return a.scale_f[1]; else return a.scale[1]; }();
        for (uint32_t item = blockIdx.x; item < a.items; item += gridDim.x)
            dslash_item<PL, PV, NREAL, NR, EPI, DS, false, false, RG, DTK, (WG > 1), PipeShape<PL, PV, NREAL, NR, DS>::on, true>(
                a, a.g, a.links, a.slot_bytes, sc0, sc1, a.in + off, a.out + (size_t)rhs0 * out_stride<EPI, true>(a), EPI ? a.pv + off : nullptr,
                EPI == 2 ? a.rv + off : nullptr, a.shift ? a.shift + rhs0 : nullptr, item / ngroups, dots, tid);
        if constexpr (EPI == 1 || EPI == 2) {
            if (a.red.partials) { // uniform over the grid
                if constexpr (RG == 1) {
                    block_sum_dots<FFK, NR * ND>(dots);
                    double dd[NR * ND];
#pragma unroll
                    for (int j = 0; j < NR * ND; j++) dd[j] = threadIdx.x == 0 ? dot_value(dots[j]) : 0.0; // read on thread 0
                    grid_reduce<NR * ND>(a.red, dd, NR * ND, ND * rhs0, ND * a.nrhs, (int)(blockIdx.x / ngroups));
                } else {
                    const double *sums = block_sum_groups<NR * ND, RG>(dots);
                    grid_reduce<NR * ND>(a.red, sums, RG * NR * ND, ND * rhs0, ND * a.nrhs,
                                         (int)(blockIdx.x / ngroups));
                }
            }
        }
    }
}

// ---------------------------------------------------------------- launch table
// Work items are (site tile of kDslashBlock threads, group of NR right-hand sides), the
// group fastest.  Without a reduction every item is a block of its own.  With the
// epilogue's reduction the grid holds at most as many blocks as are resident at once (a
// multiple of the group count, from the occupancy of this instantiation) and blocks
// stride over the items, so that there is one partial per block and right-hand side.
template <int PL, int PV, int NREAL, int NR, int EPI, int DS, bool BATCH, int RG = 1, int WG = 1>
static cudaError_t launch_one(const DslashArgs &a0, cudaStream_t st)
{
    DslashArgs a = a0;
    const int bs = BATCH ? kDslashBlock : a.bs;
    if (bs != 64 && bs != 128 && bs != 256) return cudaErrorInvalidValue;
    a.bs = bs;
    const size_t smem = (size_t)bs * PipeShape<PL, PV, NREAL, NR, DS>::bytes;
    if (smem > 32 * 1024) { // (48 KB with the static part)
        // The attribute belongs to the function and device, not to this launch: always the most that any block
        // size takes, so that no thread lowers it between another's setting and its launch.
        cudaError_t e = cudaFuncSetAttribute(k_dslash<PL, PV, NREAL, NR, EPI, DS, BATCH, RG, WG>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kDslashMaxBlock * PipeShape<PL, PV, NREAL, NR, DS>::bytes);
        if (e != cudaSuccess) return e;
    }
    static int occ[3] = {-1, -1, -1}; // resident blocks per SM of this instantiation, per block size
    const int bi = bs == 64 ? 0 : bs == 128 ? 1 : 2;
    if (occ[bi] < 0) {
        int o = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_dslash<PL, PV, NREAL, NR, EPI, DS, BATCH, RG, WG>, bs,
                                                          smem) != cudaSuccess ||
            o < 1)
            o = 1;
        occ[bi] = o;
    }
    if constexpr (BATCH) { // one block per tile of every lattice; a resident grid with a reduction
        constexpr int d = DS == 1 ? 0 : DS == 2 ? 1 : 2;
        const uint32_t items = a.batch_tiles[d];
        const uint32_t resident = (uint32_t)std::max(1, a.sm_count) * (uint32_t)occ[bi];
        const uint32_t blocks = a.red.partials ? std::min(items, resident) : items;
        a.items = items;
        a.red.nblocks = (int)a.batch_maxtiles[d]; // partials per lattice (zero beyond its tiles)
        a.red.ntotal = (int)blocks;
        k_dslash<PL, PV, NREAL, 1, EPI, DS, true><<<blocks, kDslashBlock, smem, st>>>(a);
        return cudaGetLastError();
    } else {
        const int ts = bs / WG; // threads over the sites of one tile (one slice of the block)
        if (ts < 32) return cudaErrorInvalidValue;
        a.bs = ts;
        const size_t tiles = ((size_t)a.g.Vh * DS * RG + ts - 1) / ts;
        const size_t ng = (size_t)(a.nrhs / (NR * RG * WG));
        const size_t items = tiles * ng;
        const size_t resident = std::max<size_t>(ng, (size_t)std::max(1, a.sm_count) * occ[bi] / ng * ng);
        const size_t blocks = a.red.partials ? std::min(items, resident) : items;
        if (items > 0xffffffffull) return cudaErrorInvalidValue;
        a.items = (uint32_t)items;
        a.red.nblocks = (int)(blocks / ng); // partials per right-hand side
        a.red.ntotal = (int)blocks;
        k_dslash<PL, PV, NREAL, NR, EPI, DS, false, RG, WG><<<(unsigned)blocks, bs, smem, st>>>(a);
        return cudaGetLastError();
    }
}

template <int PL, int PV, int NREAL, int EPI, int DS>
static cudaError_t launch_nr(const DslashArgs &a, int nr, int rg, cudaStream_t st)
{
    if (a.nrhs < 1 || a.nrhs % (nr * rg)) return cudaErrorInvalidValue;
    if (a.batch) { // one right-hand side per lattice, storage order
        if constexpr (EPI == 3) return cudaErrorInvalidValue;
        else {
            if (nr != 1 || rg != 1 || a.zt || a.nrhs != a.batch_n) return cudaErrorInvalidValue;
            return launch_one<PL, PV, NREAL, 1, EPI, DS, true>(a, st);
        }
    }
    if (a.zt && !a.g.zt_ok) return cudaErrorInvalidValue;
    if (a.wg > 1) { // slices of a block over the same sites: plain Dslash, one thread per site
        if constexpr (EPI == 0 && DS == 1) {
            if (rg == 1 && a.nrhs % (nr * a.wg) == 0) {
                switch (a.wg * 16 + nr) {
                case 2 * 16 + 1: return launch_one<PL, PV, NREAL, 1, 0, 1, false, 1, 2>(a, st);
                case 2 * 16 + 2: return launch_one<PL, PV, NREAL, 2, 0, 1, false, 1, 2>(a, st);
                case 2 * 16 + 4: return launch_one<PL, PV, NREAL, 4, 0, 1, false, 1, 2>(a, st);
                case 4 * 16 + 1: return launch_one<PL, PV, NREAL, 1, 0, 1, false, 1, 4>(a, st);
                case 4 * 16 + 2: return launch_one<PL, PV, NREAL, 2, 0, 1, false, 1, 4>(a, st);
                case 4 * 16 + 4: return launch_one<PL, PV, NREAL, 4, 0, 1, false, 1, 4>(a, st);
                }
            }
        }
        return cudaErrorInvalidValue;
    }
    if (rg != 1) { // groups of right-hand sides on one site's threads: one thread per site only
        if constexpr (DS == 1) {
            switch (rg * 16 + nr) {
            case 2 * 16 + 1: return launch_one<PL, PV, NREAL, 1, EPI, 1, false, 2>(a, st);
            case 2 * 16 + 2: return launch_one<PL, PV, NREAL, 2, EPI, 1, false, 2>(a, st);
            case 2 * 16 + 4: return launch_one<PL, PV, NREAL, 4, EPI, 1, false, 2>(a, st);
            case 4 * 16 + 1: return launch_one<PL, PV, NREAL, 1, EPI, 1, false, 4>(a, st);
            case 4 * 16 + 2: return launch_one<PL, PV, NREAL, 2, EPI, 1, false, 4>(a, st);
            case 4 * 16 + 4: return launch_one<PL, PV, NREAL, 4, EPI, 1, false, 4>(a, st);
            }
        }
        return cudaErrorInvalidValue;
    }
    switch (nr) {
    case 1: return launch_one<PL, PV, NREAL, 1, EPI, DS, false>(a, st);
    case 2: return launch_one<PL, PV, NREAL, 2, EPI, DS, false>(a, st);
    case 4: return launch_one<PL, PV, NREAL, 4, EPI, DS, false>(a, st);
    case 8:
        if constexpr (PV == HISQ_F64 || PV == HISQ_F64X) return cudaErrorInvalidValue;
        else return launch_one<PL, PV, NREAL, 8, EPI, DS, false>(a, st);
    default: return cudaErrorInvalidValue;
    }
}

template <int PL, int PV, int NREAL, int EPI>
static cudaError_t launch_ds(const DslashArgs &a, int nr, int ds, int rg, cudaStream_t st)
{
    switch (ds) {
    case 1: return launch_nr<PL, PV, NREAL, EPI, 1>(a, nr, rg, st);
    case 2: return launch_nr<PL, PV, NREAL, EPI, 2>(a, nr, rg, st);
    case 4: return launch_nr<PL, PV, NREAL, EPI, 4>(a, nr, rg, st);
    }
    return cudaErrorInvalidValue;
}

template <int PL, int PV, int EPI>
static cudaError_t launch_prec(const DslashArgs &a, int nreal, int nr, int ds, int rg, cudaStream_t st)
{
    if (nreal == 12) {
        if constexpr (PL == HISQ_F64X) return cudaErrorInvalidValue;
        else return launch_ds<PL, PV, 12, EPI>(a, nr, ds, rg, st);
    }
    return launch_ds<PL, PV, 18, EPI>(a, nr, ds, rg, st);
}

// Instantiate the launcher of one link precision with one vector precision.  Epilogues exist for the vector
// precisions that a solver iterates (not 16-bit); EPI = 3 for those that are not canonical by themselves.
#define HISQ_DSLASH_INSTANTIATE(PL, PV)                                                                  \
    cudaError_t dslash_launch_##PL##_##PV(int epi, const DslashArgs &a, int nreal, int nr, int ds, int rg, \
                                          cudaStream_t st)                                               \
    {                                                                                                    \
        if (epi == 0) return launch_prec<PL, PV, 0>(a, nreal, nr, ds, rg, st);                           \
        if constexpr (PV != HISQ_F16 && PV != HISQ_BF16) {                                               \
            if (epi == 1) return launch_prec<PL, PV, 1>(a, nreal, nr, ds, rg, st);                       \
            if (epi == 2) return launch_prec<PL, PV, 2>(a, nreal, nr, ds, rg, st);                       \
            if constexpr (PV != HISQ_F64)                                                                \
                if (epi == 3) return launch_prec<PL, PV, 3>(a, nreal, nr, ds, rg, st);                   \
        }                                                                                                \
        return cudaErrorInvalidValue;                                                                    \
    }

}  // namespace hisq
