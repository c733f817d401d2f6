// Domain solves with two threads per site: thread q of a site's pair (adjacent
// lanes) carries spins q and 2 + q, six of the twelve components.  A hop's link
// product acts on the two components of the projected half spinor separately, so
// each thread multiplies one of them; its result goes to its own upper spin and,
// by the direction's spin map, to its own lower spin (z, t) or its partner's
// (x, y), exchanged once after all hops.  Each clover block's rows split the same
// way.  A pair reads a link entry with one broadcast.
//
// The even-odd domain solver uses it to keep every thread busy while only half of
// the sites are updated at a time.
#pragma once

#include "hop.cuh"

namespace mgc {

__device__ __forceinline__ unsigned split_mask()
{
    return blockDim.x >= 32 ? 0xffffffffu : (1u << blockDim.x) - 1u;
}

// in-domain neighbours of a site, forward in the low and backward in the high half
// of n[mu], 0xffff where the hop leaves the domain
__device__ __forceinline__ void split_neighbours(const Geom &g, const int lc[4], uint32_t n[4])
{
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        int t[4] = {lc[0], lc[1], lc[2], lc[3]};
        t[mu] = lc[mu] + 1;
        const uint32_t f = t[mu] < (1 << g.lb[mu]) ? (uint32_t)local_index(g, t) : 0xffffu;
        t[mu] = lc[mu] - 1;
        const uint32_t b = t[mu] >= 0 ? (uint32_t)local_index(g, t) : 0xffffu;
        n[mu] = f | (b << 16);
    }
}

// one hop of thread q: the half spinor's component q from rs[k vb + n], the link
// entries at sL[k vb + lk]; sg = 1 (q = 0) or -1.  up, lo: the thread's upper and
// lower spin, lx: its partner's lower spin
template <int MU, int SGN>
__device__ __forceinline__ void split_hop(const float2 *rs, int vb, int n, const float2 *sL, int lk, int q, float sg,
                                          Cx<float> up[3], Cx<float> lo[3], Cx<float> lx[3])
{
    const float2 *so = rs + 3 * q * vb + n, *sz = rs + (MU < 2 ? 9 - 3 * q : 6 + 3 * q) * vb + n;
    const float f = (SGN > 0 ? -1.f : 1.f) * (MU == 1 || MU == 2 ? sg : 1.f);
    Cx<float> h[3], w[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float2 s = so[c * vb], z = sz[c * vb];
        if (MU == 0 || MU == 2) h[c] = {fmaf(-f, z.y, s.x), fmaf(f, z.x, s.y)};  // s + f i z
        else h[c] = {fmaf(f, z.x, s.x), fmaf(f, z.y, s.y)};
    }
    const float2 *u = sL + MU * 9 * vb + lk;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        Cx<float> t = {0.f, 0.f};
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const float2 e = u[(SGN < 0 ? a * 3 + b : b * 3 + a) * vb];
            t = SGN < 0 ? cfma(Cx<float>{e.x, e.y}, h[b], t) : cjfma(Cx<float>{e.x, e.y}, h[b], t);
        }
        w[a] = t;
    }
    // the lower spins take the spin map of w with the projector's sign
    const float r = (MU == 3 ? (SGN > 0 ? -1.f : 1.f) : (SGN > 0 ? 1.f : -1.f)) *
                    (MU == 1 ? -sg : (MU == 2 ? sg : 1.f));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        up[c] = up[c] + w[c];
        Cx<float> &o = MU < 2 ? lx[c] : lo[c];
        if (MU == 0 || MU == 2) o = Cx<float>{fmaf(-r, w[c].i, o.r), fmaf(r, w[c].r, o.i)};
        else o = Cx<float>{fmaf(r, w[c].r, o.r), fmaf(r, w[c].i, o.i)};
    }
}

// the in-domain hops at site l into the thread's spins: v[0..2] upper, v[3..5] lower
__device__ __forceinline__ void split_hops(const float2 *rs, int vb, const float2 *sL, int l, const uint32_t n[4],
                                           int q, float sg, Cx<float> v[6])
{
    Cx<float> lx[3];
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] = Cx<float>{0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 3; ++k) lx[k] = Cx<float>{0.f, 0.f};
#define MGC_SPLIT_DIR(MU)                                                                        \
    {                                                                                            \
        const int f = n[MU] & 0xffffu, b = n[MU] >> 16;                                          \
        if (f != 0xffff) split_hop<MU, -1>(rs, vb, f, sL, l, q, sg, v, v + 3, lx);               \
        if (b != 0xffff) split_hop<MU, +1>(rs, vb, b, sL, b, q, sg, v, v + 3, lx);               \
    }
    MGC_SPLIT_DIR(0)
    MGC_SPLIT_DIR(1)
    MGC_SPLIT_DIR(2)
    MGC_SPLIT_DIR(3)
#undef MGC_SPLIT_DIR
    const unsigned mask = split_mask();
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        v[3 + c].r += __shfl_xor_sync(mask, lx[c].r, 1);
        v[3 + c].i += __shfl_xor_sync(mask, lx[c].i, 1);
    }
}

// out = C v for the thread's spins at site l, the 72 reals of C as pairs at
// sC[pair vb + l]; v holds the thread's own six components, the partner's come by
// shuffles (every lane of the warp takes part)
__device__ __forceinline__ void split_clover(const float2 *sC, int vb, int l, int q, float sg, const Cx<float> v[6],
                                             Cx<float> out[6])
{
    const unsigned mask = split_mask();
#pragma unroll
    for (int chi = 0; chi < 2; ++chi) {
        const Cx<float> *own = v + 3 * chi;
        Cx<float> *o = out + 3 * chi;
        Cx<float> oth[3];
#pragma unroll
        for (int c = 0; c < 3; ++c)
            oth[c] = {__shfl_xor_sync(mask, own[c].r, 1), __shfl_xor_sync(mask, own[c].i, 1)};
        const float2 d0 = sC[(18 * chi + 2 * q) * vb + l], d1 = sC[(18 * chi + 1) * vb + l];
        const float d[3] = {q ? d1.y : d0.x, q ? d0.x : d0.y, q ? d0.y : d1.x};
#pragma unroll
        for (int c = 0; c < 3; ++c) o[c] = d[c] * own[c];
        // within the spin: entries (1,0) (2,0) (2,1) or (4,3) (5,3) (5,4)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int a = k ? 2 : 1, b = k == 2 ? 1 : 0;
            const int idx = q ? (k == 0 ? 9 : 12 + k) : k;
            const float2 e = sC[(18 * chi + 3 + idx) * vb + l];
            const Cx<float> L = {e.x, e.y};
            o[a] = cfma(L, own[b], o[a]);
            o[b] = cjfma(L, own[a], o[b]);
        }
        // between the spins: X_ab = (3 + a, b) for q = 1, its adjoint for q = 0
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const int r = q ? a : b, c = q ? b : a;
                const float2 e = sC[(18 * chi + 6 + r * (r + 5) / 2 + c) * vb + l];
                o[a] = cfma(Cx<float>{e.x, -sg * e.y}, oth[b], o[a]);
            }
    }
}

// a thread's six components to and from the site-indexed array rs[k vb + l]
__device__ __forceinline__ void split_put(float2 *rs, int vb, int l, int q, const Cx<float> v[6])
{
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        rs[(3 * q + c) * vb + l] = make_float2(v[c].r, v[c].i);
        rs[(6 + 3 * q + c) * vb + l] = make_float2(v[3 + c].r, v[3 + c].i);
    }
}
__device__ __forceinline__ void split_get(const float2 *rs, int vb, int l, int q, Cx<float> v[6])
{
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float2 a = rs[(3 * q + c) * vb + l], b = rs[(6 + 3 * q + c) * vb + l];
        v[c] = {a.x, a.y};
        v[3 + c] = {b.x, b.y};
    }
}

}  // namespace mgc
