// The FP64 operator in block fixed point: products of 62-bit fixed-point
// numbers on the integer multiply-add units.
//
// GB300 issues 2 FP64 fused multiply-adds per clock and SM, but 32 widening
// integer multiply-adds (32 x 32 + 64 bits; the first measured with eight
// independent chains per thread, the second from the busy cycles of the pipe).  A
// product of two-limb integers a = a1 2^32 + a0 whose low limbs are balanced (|a0| <= 2^31, random sign)
// needs three of them, hh += a1 b1 and mid += a1 b0 + a0 b1: the dropped a0 b0
// is below the last bit kept.  A multiply-add of more precision than FP64's
// therefore takes three instructions of 1/16 the cost, which turns the operator
// from one bound by the FP64 pipe into one bound by instruction issue and HBM.
//
// Scales.  kappa = k' 2^ek with 1/2 <= |k'| < 1.  The links are stored times k',
// q = k' u 2^60 (unitary to 1e-3, so |q| <= 2^60), the clover term as
// q = C 2^(60 - e_C - ek), e_C the site's exponent (|C| < 2^(e_C + ek)).  A thread
// adds its eight hops and the clover term in 64-bit integers in units of
// 2^(E + ek - 56), E at least the exponent of the largest component of psi at the
// nine sites: a neighbour's components are brought to that unit as they are read
// (Q = psi 2^(60 - E)), and where a neighbour exceeds E the sum is shifted down.
// The result is the sum times a power of two: one rounding.  Sum bounds: a hop's
// row has |sum| <= 4.9 2^E (unitary rows, |h| <= 2 2^E), eight of them 2^5.3 2^E,
// the clover term 2^5 2^E (E >= e_psi + room, a row's absolute sum of C below
// 2^(5 + room + ek); room = 0 for kappa near 1/8), together below 2^62.2 units;
// the middle sums stay below 2^62.9 (two-norm bound for the links; for the clover
// eleven terms of 2^59 with its low limbs, and 2^31 times the row sum 2^30 of its
// high limbs).  The dropped products a0 b0 are of random sign, 2^-57 of the
// largest product in the mean square.
//
// A site is computed with FP64 instructions instead (fix_fallback) when its own
// or a neighbour's components span more than 2^27, include some but not only
// zeros, are not finite, or lie outside 2^-894 .. 2^961 (infinities and NaN
// propagate, and no conversion needs a test of its own); and when a component of
// the sum is too small for the unit (below).
//
// Error.  The roundings of the sum (components, links and clover terms brought to
// their units, dropped products, each hop rounded, without bias: a mean error of
// half a unit, the same everywhere, is a smooth field that the solvers' low modes
// amplify) are a fixed number of units of 2^(E + ek - 56), 1.2 of them in the mean
// square, whatever a component's size; FP64's error of a component goes with the
// magnitudes of the terms that enter it.  So a site runs on fixed point only where
// every one of its twelve components is large enough: FixTerms adds up magnitudes of
// the hops' contributions to it, which with the sum's own (together at most twice the
// terms) must reach 2^54 units.  Gaussian fields stay, at kappa = 0.125 to 0.1365, on
// links near and far from 1, c_SW 0 and 1 (the median component has about 2^57.5; of
// 663,552 sites none leaves, of the operator's sites in solves 6 in 10^6); a field whose
// colours or spins differ by more than about 4 in scale without being mixed leaves.
// Measured for a colour scaled by 2^-p on unit links: its error is 1.4e-16 to
// 1.6e-16 at every p from 0 to 50, as with FP64 instructions (1.5e-16); without the
// test it was 1.1e-14 at p = 10.
// Against quadruple precision the operator is off by 5.4e-17 in the 2-norm
// (kappa = 0.126 to 0.1365, c_SW = 1), with FP64 instructions by 1.7e-16; the
// rounding of the exact result alone is 4.7e-17.
#pragma once

#include "hop.cuh"
#include "tma.cuh"

namespace mgc {

typedef long long fix_t;

constexpr int FIX_EMIN = 0x80;   // smallest biased exponent the fixed-point path takes
constexpr int FIX_EMAX = 0x7c0;  // first biased exponent it does not

// threads of the operator's blocks, and the 16-byte staging slots a thread has in
// shared memory (slot k of thread t at [k][t], NT threads): a neighbour's spinor
// and a link
constexpr int FIX_THREADS = 128;
constexpr int FIX_SPINOR_SLOTS = 12, FIX_LINK_SLOTS = 9;

// 16-byte asynchronous copies global -> shared, read back by the thread that
// issued them, so no barrier is involved
__device__ __forceinline__ void fix_copy16(int4 *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void fix_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void fix_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// links times k': the plane order of Gauge64, a complex entry as (re hi, re lo, im hi, im lo)
struct FixLinks {
    const int4 *p;
    int lvb;
    __device__ __forceinline__ const int4 *at(int i, int mu) const
    {
        return p + (((size_t)(i >> lvb) * 4 + mu) * 9 << lvb) + (i & ((1 << lvb) - 1));
    }
};

// C: the plane order of Clover64, every site's (exponent, room), and ek
struct FixClover {
    const int4 *p;
    const int2 *e;
    int ek;
    int lvb;
    __device__ __forceinline__ const int4 *at(int i) const
    {
        return p + ((size_t)(i >> lvb) * 36 << lvb) + (i & ((1 << lvb) - 1));
    }
};

__device__ __forceinline__ fix_t mac64(int a, int b, fix_t c) { return c + (fix_t)a * (fix_t)b; }
__device__ __forceinline__ fix_t mul64(int a, int b) { return (fix_t)a * (fix_t)b; }
// -x (and the limbs below) as 32-bit numbers of unknown origin: where the compiler
// can see them it sign-extends first and multiplies 64-bit numbers (850 of the
// 2,640 multiply-adds a site, 2,520 products and 120 joins, each in four instructions).  The products themselves
// stay in C: as mad.wide in inline PTX a third came out as a multiplication and
// a separate 64-bit addition.
__device__ __forceinline__ int fix_neg(int x)
{
    int r;
    asm("neg.s32 %0, %1;" : "=r"(r) : "r"(x));
    return r;
}

// largest and smallest magnitude of three words read as FP32 bit patterns: the
// high words of doubles order like the doubles; NaN patterns (exponents from
// 0x7f8 on) stay NaN in the maximum
__device__ __forceinline__ float max3abs(float a, float b, float c)
{
    float d;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float min3abs(float a, float b, float c)
{
    float d;
    asm("min.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// a packed FP64 spinor's words, and the biased exponents of its largest and
// smallest component
struct FixRaw {
    uint4 w[12];
    int emax, emin;
    __device__ __forceinline__ void load(const Spinor64 &in, int i)
    {
        const uint4 *q = reinterpret_cast<const uint4 *>(in.at(i));
#pragma unroll
        for (int k = 0; k < 12; ++k) w[k] = __ldg(q + ((size_t)k << in.lvb));
    }
    // from the thread's staging slots
    __device__ __forceinline__ void load_staged(const int4 *slot, int nt)
    {
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const int4 v = slot[k * nt];
            w[k] = make_uint4(v.x, v.y, v.z, v.w);
        }
    }
    __device__ __forceinline__ void range()
    {
        float mx = fabsf(__uint_as_float(w[0].y)), mn = mx;
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            mx = max3abs(mx, __uint_as_float(w[k].y), __uint_as_float(w[k].w));
            mn = min3abs(mn, __uint_as_float(w[k].y), __uint_as_float(w[k].w));
        }
        emax = __float_as_int(mx) >> 20;
        emin = __float_as_int(mn) >> 20;
    }
};

// Q = x 2^(60 - E) for a double x with |x| < 2^E, K = E's biased exponent + 4,
// valid while K - (x's biased exponent) < 32.
// Negative values come out one unit (2^-60) low: the sign is applied as a
// one's complement.  neg = ~0 negates x.
__device__ __forceinline__ fix_t fix_from(uint32_t lo, uint32_t hi, int K, uint32_t neg)
{
    const uint32_t u = __funnelshift_l(lo, hi, 11) | 0x80000000u, v = lo << 11;
    const int s = K - (int)(hi >> 20);  // the sign bit adds a multiple of 32
    const uint32_t sm = (uint32_t)((int)hi >> 31);
    const uint32_t ql = __funnelshift_r(v, u, s) ^ sm ^ neg;
    const uint32_t qh = __funnelshift_r(u, 0u, s) ^ sm ^ neg;
    return (fix_t)(((unsigned long long)qh << 32) | ql);
}

// Q of a double, K = the unit's biased exponent + 4: x = Q 2^(K - 1086) rounded
// towards zero, |x| < 2^(K - 1023) (|Q| < 2^63)
__device__ __forceinline__ fix_t fix_from_any(double x, int K)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int e = (int)(hi >> 20) & 0x7ff;
    const int s = K - e;
    unsigned long long m = ((unsigned long long)(__funnelshift_l(lo, hi, 11) | 0x80000000u) << 32) | (lo << 11);
    m = (e == 0 || s > 63) ? 0 : m >> s;
    return (int)hi < 0 ? -(fix_t)m : (fix_t)m;
}

// component k of the site in units of 2^(E - 60), K = E + 4
__device__ __forceinline__ Cx<fix_t> fix_component(const FixRaw &r, int k, int K, uint32_t neg = 0)
{
    return {fix_from(r.w[k].x, r.w[k].y, K, neg), fix_from(r.w[k].z, r.w[k].w, K, neg)};
}

// every component of the site is zero (emax == 0 leaves zeros and denormals)
__device__ __forceinline__ bool fix_all_zero(const FixRaw &r)
{
    if (r.emax != 0) return false;
    uint32_t any = 0;
#pragma unroll
    for (int k = 0; k < 12; ++k) any |= r.w[k].x | r.w[k].z | ((r.w[k].y | r.w[k].w) & 0x7fffffffu);
    return any == 0;
}

// the site's components can be converted to units of 2^(E - 60): all of them
// nonzero, in range and above 2^-27 of 2^E
__device__ __forceinline__ bool fix_in_range(const FixRaw &r, int E)
{
    return r.emax < FIX_EMAX && r.emax >= FIX_EMIN && E + 4 - r.emin < 32;
}

// limbs with a balanced low part
__device__ __forceinline__ void fix_limbs(fix_t q, int &hi, int &lo)
{
    lo = (int)q;
    hi = (int)((uint32_t)((unsigned long long)q >> 32) + ((uint32_t)lo >> 31));
    asm("" : "+r"(lo), "+r"(hi));  // 32-bit numbers of unknown origin (above)
}

// hh + mid 2^-32 in units of hh, rounded down (the sums start from half a unit)
__device__ __forceinline__ fix_t fix_join(fix_t hh, fix_t mid) { return mac64((int)(mid >> 32), 1, hh); }

// hh + mid 2^-32 in units of hh 2^-L, rounded down, 0 <= L < 32
__device__ __forceinline__ fix_t fix_join_bits(fix_t hh, fix_t mid, int L)
{
    const fix_t y = fix_join(hh, mid);
    return (fix_t)(((unsigned long long)__funnelshift_l((uint32_t)y, (uint32_t)(y >> 32), L) << 32) |
                   __funnelshift_l((uint32_t)mid, (uint32_t)y, L));
}

// (a, b) + sgn P (l0, l1) with P the spin map of direction MU: the projected
// half spinor of one colour
template <int MU, int SGN>
__device__ __forceinline__ void fix_project(Cx<fix_t> &a, Cx<fix_t> &b, Cx<fix_t> l0, Cx<fix_t> l1)
{
    Cx<fix_t> o0, o1;
    isigma<MU>(l0, l1, o0, o1);
    a = SGN > 0 ? a - o0 : a + o0;
    b = SGN > 0 ? b - o1 : b + o1;
}

// the lower spins of one colour reconstructed from (w0, w1), as reconstruct_add
template <int MU, int SGN>
__device__ __forceinline__ void fix_reconstruct(Cx<fix_t> &a, Cx<fix_t> &b, Cx<fix_t> w0, Cx<fix_t> w1)
{
    Cx<fix_t> o0, o1;
    isigma<MU>(w0, w1, o0, o1);
    if ((MU == 3) == (SGN > 0)) {
        a = a - o0;
        b = b - o1;
    } else {
        a = a + o0;
        b = b + o1;
    }
}

// a direction known at run time (the same for every thread), as a switch over
// its spin maps: m = 2 mu + (projector 1 + gamma)
#define MGC_FIX_SWITCH(m, CALL)        \
    switch (m) {                       \
    case 0: CALL(0, -1); break;        \
    case 1: CALL(0, +1); break;        \
    case 2: CALL(1, -1); break;        \
    case 3: CALL(1, +1); break;        \
    case 4: CALL(2, -1); break;        \
    case 5: CALL(2, +1); break;        \
    case 6: CALL(3, -1); break;        \
    default: CALL(3, +1); break;       \
    }

// The limbs of the half spinor projected for direction m (above) from the
// components q(k) of a neighbour, conjugated for a backward hop; colour by
// colour, so that few 64-bit intermediates live at a time
template <class Q>
__device__ __forceinline__ void fix_project_limbs(Q q, int m, bool back, int h1[12], int h0[12])
{
    const fix_t bm = back ? -1 : 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        Cx<fix_t> a = q(k), b = q(3 + k);
        const Cx<fix_t> l0 = q(6 + k), l1 = q(9 + k);
#define MGC_FIX_CALL(MU, SGN) fix_project<MU, SGN>(a, b, l0, l1)
        MGC_FIX_SWITCH(m, MGC_FIX_CALL)
#undef MGC_FIX_CALL
        a.i ^= bm;
        b.i ^= bm;
        fix_limbs(a.r, h1[2 * k], h0[2 * k]);
        fix_limbs(a.i, h1[2 * k + 1], h0[2 * k + 1]);
        fix_limbs(b.r, h1[2 * k + 6], h0[2 * k + 6]);
        fix_limbs(b.i, h1[2 * k + 7], h0[2 * k + 7]);
    }
}

// Lower bounds of the terms that enter a site's components, in counts of 2^32 units:
// per colour the sum over the hops of the smaller of the half spinor's two
// contributions, |re| + |im|, which bounds those to each of the four spins whatever
// the direction's spin map.  A contribution is at most 6.9 2^56 units, eight of them
// 2^61.8.  (Counts per spin took six registers, which the smoother has none to spare
// of: 18 % of its FP64 solve in spills.)
struct FixTerms {
    int n[3];
    int hops;  // those added, less NONE while the site itself adds nothing
    static constexpr int NONE = 16;
    __device__ __forceinline__ void clear(bool own)
    {
        n[0] = n[1] = n[2] = 0;
        hops = own ? 0 : -NONE;
    }
    // nothing has been added: the sum is zero
    __device__ __forceinline__ bool nothing() const { return hops == -NONE; }
    // the unit grows by 2^d
    __device__ __forceinline__ void shift(int d)
    {
#pragma unroll
        for (int a = 0; a < 3; ++a) n[a] >>= min(d, 31);
    }
    static __device__ __forceinline__ uint32_t size(Cx<fix_t> v)
    {
        return (uint32_t)abs((int)(v.r >> 32)) + (uint32_t)abs((int)(v.i >> 32));
    }
    // a hop's contributions to colour a
    __device__ __forceinline__ void add(int a, Cx<fix_t> w0, Cx<fix_t> w1) { n[a] += (int)min(size(w0), size(w1)); }
    __device__ __forceinline__ bool all_reach(int least) const { return min(min(n[0], n[1]), n[2]) >= least; }
    // component k of the sum, of value v, has `least` counts
    __device__ __forceinline__ bool reaches(int least, int k, Cx<fix_t> v) const
    {
        return (uint32_t)n[k % 3] + size(v) >= (uint32_t)least;
    }
    // whether every component of the sum acc has `least` counts
    __device__ __forceinline__ bool enough(int least, const Cx<fix_t> acc[12]) const
    {
        if (all_reach(least) || nothing()) return true;
        bool all = true;
#pragma unroll
        for (int k = 0; k < 12; ++k) all = all && reaches(least, k, acc[k]);
        return all;
    }
    // the counts that every component of the operator needs: 2^54 units for eight
    // hops (whose sum's error is 1.2 units), for fewer by the square root of their number
    __device__ __forceinline__ int least() const
    {
        const int h = hops & (NONE - 1);
        return h > 4 ? 1 << 22 : (h > 2 ? 0x2d4000 : (h > 1 ? 1 << 21 : 0x16a000));
    }
};

// The projected half spinor of direction m (above) from the spinor in the staging
// slots (negated where `flip`, conjugated where `back`), as limbs; raises E (and
// shifts acc and the terms down) where the neighbour exceeds it; FIX_LEAVE when the
// site needs FP64.
enum { FIX_LEAVE, FIX_ZERO, FIX_HOP };
__device__ __forceinline__ int fix_half_spinor(const int4 *slot, int nt, int m, bool back, bool flip, Cx<fix_t> acc[12],
                                                FixTerms &terms, int &E, int h1[12], int h0[12])
{
    FixRaw r;
    r.load_staged(slot, nt);
    r.range();
    if (r.emax > E) {
        const int d = min(r.emax - E, 62);
        const fix_t half = (fix_t)1 << (d - 1);
        E = r.emax;
        terms.shift(d);
#pragma unroll
        for (int k = 0; k < 12; ++k) acc[k] = Cx<fix_t>{(acc[k].r + half) >> d, (acc[k].i + half) >> d};
    }
    if (!fix_in_range(r, E)) return fix_all_zero(r) ? FIX_ZERO : FIX_LEAVE;
    const int K = E + 4;
    const uint32_t fm = flip ? ~0u : 0u;
    fix_project_limbs([&](int k) { return fix_component(r, k, K, fm); }, m, back, h1, h0);
    return FIX_HOP;
}

// acc += the hop of direction m from its projected half spinor h (conjugated for
// a backward hop) and the link whose entry k is at link[k stride] (shared or
// global memory).  U^dagger h is the conjugate
// of U^T conj(h): the backward hop reads the transposed entries and negates the
// imaginary parts on the way in and out, as one's complements (~w = -w - 1, which
// the rounding constant of the imaginary parts makes up for).
__device__ __forceinline__ void fix_hop(const int4 *link, int stride, int m, bool back, const int h1[12],
                                        const int h0[12], Cx<fix_t> acc[12], FixTerms &terms)
{
    const int sa = (back ? 1 : 3) * stride, sb = (back ? 3 : 1) * stride;
    const fix_t bm = back ? -1 : 0;
    const fix_t cr = 0x80000000LL, ci = (bm << 32) | 0x80000000LL;  // +- half a unit of hh
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        fix_t hr[2], hi[2], mr[2], mi[2];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int4 u = link[a * sa + b * sb];
            const int n1 = fix_neg(u.z), n0 = fix_neg(u.w);
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int k = 2 * (3 * s + b);
                const int x1 = h1[k], x0 = h0[k], y1 = h1[k + 1], y0 = h0[k + 1];
                hr[s] = mac64(n1, y1, b ? mac64(u.x, x1, hr[s]) : mul64(u.x, x1));
                mr[s] = mac64(u.y, x1, mac64(u.x, x0, b ? mr[s] : cr));
                mr[s] = mac64(n0, y1, mac64(n1, y0, mr[s]));
                hi[s] = mac64(u.z, x1, b ? mac64(u.x, y1, hi[s]) : mul64(u.x, y1));
                mi[s] = mac64(u.y, y1, mac64(u.x, y0, b ? mi[s] : ci));
                mi[s] = mac64(u.w, x1, mac64(u.z, x0, mi[s]));
            }
        }
        const Cx<fix_t> w0 = {fix_join(hr[0], mr[0]), fix_join(hi[0], mi[0]) ^ bm};
        const Cx<fix_t> w1 = {fix_join(hr[1], mr[1]), fix_join(hi[1], mi[1]) ^ bm};
        acc[a] = acc[a] + w0;
        acc[3 + a] = acc[3 + a] + w1;
        terms.add(a, w0, w1);
#define MGC_FIX_CALL(MU, SGN) fix_reconstruct<MU, SGN>(acc[6 + a], acc[9 + a], w0, w1)
        MGC_FIX_SWITCH(m, MGC_FIX_CALL)
#undef MGC_FIX_CALL
    }
}

// the neighbour of hop d (mu = d / 2, backward when odd), and whether the hop
// carries the boundary sign
__device__ __forceinline__ int fix_neighbour(const Geom &g, const int c[4], int d, bool &flip)
{
    const int step = d & 1 ? -1 : 1;
    int n[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        int v = c[k] + (k == (d >> 1) ? step : 0);
        const bool lo = v < 0, hi = v >= g.L[k];
        v = lo ? v + g.L[k] : (hi ? 0 : v);
        if (k == 3) flip = (lo || hi) && g.tbc < 0;
        n[k] = v;
    }
    return site_index(g, n);
}

// acc = C psi in the sum's unit, from psi's components q(k): the products'
// unit times 2^L, L < 32
template <class Q>
__device__ __forceinline__ void fix_clover(const FixClover &C, int i, Q psi, int L, Cx<fix_t> acc[12])
{
    const int4 *cp = C.at(i);
    const fix_t half = 0x80000000LL >> max(L, 0);  // half a unit of the sum
#pragma unroll
    for (int chi = 0; chi < 2; ++chi) {
        int v1[12], v0[12];
        fix_t hh[12], mid[12];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const Cx<fix_t> q = psi(6 * chi + k);
            fix_limbs(q.r, v1[2 * k], v0[2 * k]);
            fix_limbs(q.i, v1[2 * k + 1], v0[2 * k + 1]);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int4 d = __ldg(cp + ((size_t)(18 * chi + k) << C.lvb));
#pragma unroll
            for (int z = 0; z < 2; ++z) {
                hh[4 * k + z] = mul64(d.x, v1[4 * k + z]);
                mid[4 * k + z] = mac64(d.x, v0[4 * k + z], mac64(d.y, v1[4 * k + z], half));
                hh[4 * k + 2 + z] = mul64(d.z, v1[4 * k + 2 + z]);
                mid[4 * k + 2 + z] = mac64(d.z, v0[4 * k + 2 + z], mac64(d.w, v1[4 * k + 2 + z], half));
            }
        }
        int k = 3;
#pragma unroll
        for (int a = 1; a < 6; ++a)
#pragma unroll
            for (int b = 0; b < a; ++b) {
                const int4 l = __ldg(cp + ((size_t)(18 * chi + k++) << C.lvb));
                const int n1 = fix_neg(l.z), n0 = fix_neg(l.w);
                // o[a] += L v[b], o[b] += conj(L) v[a]
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const int o = 2 * (t ? b : a), x = 2 * (t ? a : b);
                    const int s1 = t ? l.z : n1, s0 = t ? l.w : n0;  // sign of the (im, im) product
                    const int c1 = t ? n1 : l.z, c0 = t ? n0 : l.w;
                    hh[o] = mac64(l.x, v1[x], hh[o]);
                    mid[o] = mac64(l.x, v0[x], mid[o]);
                    mid[o] = mac64(l.y, v1[x], mid[o]);
                    hh[o] = mac64(s1, v1[x + 1], hh[o]);
                    mid[o] = mac64(s1, v0[x + 1], mid[o]);
                    mid[o] = mac64(s0, v1[x + 1], mid[o]);
                    hh[o + 1] = mac64(l.x, v1[x + 1], hh[o + 1]);
                    mid[o + 1] = mac64(l.x, v0[x + 1], mid[o + 1]);
                    mid[o + 1] = mac64(l.y, v1[x + 1], mid[o + 1]);
                    hh[o + 1] = mac64(c1, v1[x], hh[o + 1]);
                    mid[o + 1] = mac64(c1, v0[x], mid[o + 1]);
                    mid[o + 1] = mac64(c0, v1[x], mid[o + 1]);
                }
            }
#pragma unroll
        for (int m = 0; m < 12; ++m) {
            const fix_t y = fix_join(hh[m], mid[m]);
            fix_t r;
            if (L >= 0) r = fix_join_bits(hh[m], mid[m], L);
            else r = y >> min(-L, 63);
            (m & 1 ? acc[6 * chi + (m >> 1)].i : acc[6 * chi + (m >> 1)].r) = r;
        }
    }
}

// limbs of a 3x3 complex matrix, entry k as (re hi, re lo, im hi, im lo)
struct FixM3 {
    int4 e[9];
    // a link or its dagger
    __device__ __forceinline__ void load(const FixLinks &U, int site, int mu, bool dag)
    {
        const int4 *q = U.at(site, mu);
        const int sm = dag ? -1 : 0, sa = dag ? 1 : 3, sb = dag ? 3 : 1;
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                int4 v = __ldg(q + ((a * sa + b * sb) << U.lvb));
                v.z = (v.z ^ sm) - sm;
                v.w = (v.w ^ sm) - sm;
                asm("" : "+r"(v.z), "+r"(v.w));  // 32-bit numbers of unknown origin (fix_neg)
                e[a * 3 + b] = v;
            }
    }
};

// (hr, mr) + i (hi, mi) += u x, u and x complex limbs
__device__ __forceinline__ void fix_cmac(int4 u, int4 x, fix_t &hr, fix_t &mr, fix_t &hi, fix_t &mi)
{
    const int n1 = fix_neg(u.z), n0 = fix_neg(u.w);
    hr = mac64(n1, x.z, mac64(u.x, x.x, hr));
    mr = mac64(u.y, x.x, mac64(u.x, x.y, mr));
    mr = mac64(n0, x.z, mac64(n1, x.w, mr));
    hi = mac64(u.z, x.x, mac64(u.x, x.z, hi));
    mi = mac64(u.y, x.z, mac64(u.x, x.w, mi));
    mi = mac64(u.w, x.x, mac64(u.z, x.y, mi));
}

// (D psi)(x) with FP64 instructions, for the sites the fixed-point path leaves
template <bool DAG>
__device__ __noinline__ void fix_fallback(Geom g, int i, Spinor64 in, Spinor64 out, Gauge64 U, Clover64 C, double kappa)
{
    int c[4];
    site_coords(g, i, c);
    const Spinor64 one[1] = {in};
    Cx<double> o[1][12];
    dirac_site_pair<DAG, 1>(g, c, i, one, 1, U, C, kappa, o);
    out.store(i, o[0]);
}

// (D psi)(i) = -2^(E + ek - 1078) acc in fixed point (E the biased exponent);
// false when the site needs FP64 for its inputs, which it also does unless `terms`
// are enough.  `slots` is the thread's column of the block's
// staging slots, nt its threads.  One copy of the hop's code serves all eight:
// unrolled per direction the kernel is 12,600 instructions long and waits on
// instruction fetch for half its time (1060 us on 24^3 x 48).  The next hop's
// spinor and link are copied to shared memory while this hop's products run;
// without that, loads were the first stall (433 us).
// CLOVER = false leaves the clover term out: kappa H psi = 2^(E + ek - 1078) acc.
template <bool DAG, bool CLOVER = true>
__device__ __forceinline__ bool fix_dirac_sum(const Geom &g, int i, const Spinor64 &in, const FixLinks &U,
                                              const FixClover &C, int4 *slots, int nt, Cx<fix_t> acc[12],
                                              FixTerms &terms, int &E)
{
    int4 *const ls = slots + FIX_SPINOR_SLOTS * nt;
    auto copy_spinor = [&](int j) {
        const double2 *q = in.at(j);
#pragma unroll
        for (int k = 0; k < FIX_SPINOR_SLOTS; ++k) fix_copy16(slots + k * nt, q + ((size_t)k << in.lvb));
    };
    auto copy_link = [&](int d, int j) {
        const int4 *q = U.at(d & 1 ? j : i, d >> 1);
#pragma unroll
        for (int k = 0; k < FIX_LINK_SLOTS; ++k) fix_copy16(ls + k * nt, q + ((size_t)k << U.lvb));
    };
    int c[4];
    site_coords(g, i, c);
    bool flip;
    int j = fix_neighbour(g, c, 0, flip);
    copy_spinor(j);
    fix_commit();
    copy_link(0, j);
    fix_commit();

    int state = FIX_HOP;
    terms.clear(false);
    if constexpr (CLOVER) {
        FixRaw r;
        r.load(in, i);
        r.range();
        const int2 eC = __ldg(C.e + i);
        const int ep = max(r.emax, FIX_EMIN);
        E = ep + eC.y;
        if (fix_in_range(r, ep)) {
            terms.clear(true);
            fix_clover(C, i, [&](int k) { return fix_component(r, k, ep + 4); }, eC.x - eC.y, acc);
        } else {
            state = fix_all_zero(r) ? FIX_ZERO : FIX_LEAVE;
#pragma unroll
            for (int k = 0; k < 12; ++k) acc[k] = Cx<fix_t>{0, 0};
        }
        // the sum is that of kappa H psi - C psi
#pragma unroll
        for (int k = 0; k < 12; ++k) acc[k] = -acc[k];
    } else {
        E = FIX_EMIN;
#pragma unroll
        for (int k = 0; k < 12; ++k) acc[k] = Cx<fix_t>{0, 0};
    }
#pragma unroll 1
    for (int d = 0; d < 8 && state != FIX_LEAVE; ++d) {
        const int m = (d & ~1) + (int)((bool)(d & 1) != DAG);
        int h1[12], h0[12];
        fix_wait<1>();  // this hop's spinor (its link may be in flight)
        state = fix_half_spinor(slots, nt, m, d & 1, flip, acc, terms, E, h1, h0);
        if (d < 7) {
            // every slot has been read: the test above depends on all of them
            j = fix_neighbour(g, c, d + 1, flip);
            copy_spinor(j);
        }
        fix_commit();
        fix_wait<1>();  // this hop's link
        if (state == FIX_HOP) {
            ++terms.hops;
            fix_hop(ls, nt, m, d & 1, h1, h0, acc, terms);
        }
        if (d < 7) copy_link(d + 1, j);
        fix_commit();
    }
    fix_wait<0>();
    return state != FIX_LEAVE;
}

// 2^(e - 1023) for a biased exponent 0 < e < 2047
__device__ __forceinline__ double fix_pow2(int e) { return __hiloint2double(e << 20, 0); }

// out(i) = (D psi)(i); false (nothing stored) when the site needs FP64
template <bool DAG>
__device__ __forceinline__ bool fix_dirac_site(const Geom &g, int i, const Spinor64 &in, const Spinor64 &out,
                                               const FixLinks &U, const FixClover &C, int4 *slots)
{
    Cx<fix_t> acc[12];
    FixTerms terms;
    int E;
    if (!fix_dirac_sum<DAG>(g, i, in, U, C, slots, FIX_THREADS, acc, terms, E)) return false;
    if (!terms.enough(terms.least(), acc)) return false;
    const double sc = -fix_pow2(E + C.ek - 55);
    Cx<double> o[12];
#pragma unroll
    for (int k = 0; k < 12; ++k)
        o[k] = Cx<double>{sc * __ll2double_rn(acc[k].r), sc * __ll2double_rn(acc[k].i)};
    out.store(i, o);
    return true;
}

}  // namespace mgc
