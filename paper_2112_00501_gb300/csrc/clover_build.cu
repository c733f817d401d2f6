// The clover term of Eq. (1) and its inverse, built on the GPU in FP64 from
// the gauge field (Sec. 2: C and C^-1 are computed from the gauge field).
//
//   F_{mu nu}(x) = (Q_{mu nu}(x) - Q_{mu nu}(x)^+) / 8,
//   Q_{mu nu}(x) = sum of the four plaquette leaves in the mu-nu plane that
//                  start and end at x (orientation mu then nu),
//   C = 1 + i kappa c_SW sum_{mu<nu} sigma_{mu nu} F_{mu nu}.
// In the chiral basis sigma_{mu nu} = diag(s+_{mu nu}, s-_{mu nu}) with 2x2
// blocks built from Pauli matrices (table below), so C = diag(C+, C-) with
// two 6x6 Hermitian blocks.  Each block is inverted by L D L^+ where it is positive
// definite and the links have a fixed-point copy, by Gauss-Jordan elimination with
// partial pivoting otherwise.
#include "fix64.cuh"
#include "mgc_host.h"
#include "sigma.cuh"

namespace mgc {

typedef Cx<double> cd;

__device__ void m3mul(const cd *a, const cd *b, cd *o)
{
    cd t[9];
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) {
            cd acc = a[i * 3] * b[j];
            acc = cfma(a[i * 3 + 1], b[3 + j], acc);
            acc = cfma(a[i * 3 + 2], b[6 + j], acc);
            t[i * 3 + j] = acc;
        }
    for (int k = 0; k < 9; ++k) o[k] = t[k];
}

__device__ void m3dag(const cd *a, cd *o)
{
    cd t[9];
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) t[i * 3 + j] = conj(a[j * 3 + i]);
    for (int k = 0; k < 9; ++k) o[k] = t[k];
}

__device__ int shifted_site(const Geom &g, const int c[4], int mu, int dm, int nu, int dn)
{
    int n[4] = {c[0], c[1], c[2], c[3]};
    n[mu] = (n[mu] + dm + g.L[mu]) % g.L[mu];
    n[nu] = (n[nu] + dn + g.L[nu]) % g.L[nu];
    return site_index(g, n);
}

// link U_dir(site), optionally daggered
__device__ void get_link(const Gauge64 &U, int site, int dir, bool dag, cd *o)
{
    U.load(site, dir, o);
    if (dag) m3dag(o, o);
}

// the sum of the four leaves of the mu-nu plane at site x (coordinates c)
__device__ void clover_leaves(const Geom &g, const Gauge64 &U, const int c[4], int x, int mu, int nu, cd *Q)
{
    const int xpm = shifted_site(g, c, mu, 1, nu, 0), xpn = shifted_site(g, c, mu, 0, nu, 1);
    const int xmm = shifted_site(g, c, mu, -1, nu, 0), xmn = shifted_site(g, c, mu, 0, nu, -1);
    const int xmmpn = shifted_site(g, c, mu, -1, nu, 1), xmmmn = shifted_site(g, c, mu, -1, nu, -1);
    const int xpmmn = shifted_site(g, c, mu, 1, nu, -1);
    cd P[9], A[9];
    for (int k = 0; k < 9; ++k) Q[k] = cd{0, 0};
    // U_mu(x) U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+
    get_link(U, x, mu, false, P);
    get_link(U, xpm, nu, false, A); m3mul(P, A, P);
    get_link(U, xpn, mu, true, A); m3mul(P, A, P);
    get_link(U, x, nu, true, A); m3mul(P, A, P);
    for (int k = 0; k < 9; ++k) Q[k] = Q[k] + P[k];
    // U_nu(x) U_mu(x-mu+nu)^+ U_nu(x-mu)^+ U_mu(x-mu)
    get_link(U, x, nu, false, P);
    get_link(U, xmmpn, mu, true, A); m3mul(P, A, P);
    get_link(U, xmm, nu, true, A); m3mul(P, A, P);
    get_link(U, xmm, mu, false, A); m3mul(P, A, P);
    for (int k = 0; k < 9; ++k) Q[k] = Q[k] + P[k];
    // U_mu(x-mu)^+ U_nu(x-mu-nu)^+ U_mu(x-mu-nu) U_nu(x-nu)
    get_link(U, xmm, mu, true, P);
    get_link(U, xmmmn, nu, true, A); m3mul(P, A, P);
    get_link(U, xmmmn, mu, false, A); m3mul(P, A, P);
    get_link(U, xmn, nu, false, A); m3mul(P, A, P);
    for (int k = 0; k < 9; ++k) Q[k] = Q[k] + P[k];
    // U_nu(x-nu)^+ U_mu(x-nu) U_nu(x-nu+mu) U_mu(x)^+
    get_link(U, xmn, nu, true, P);
    get_link(U, xmn, mu, false, A); m3mul(P, A, P);
    get_link(U, xpmmn, nu, false, A); m3mul(P, A, P);
    get_link(U, x, mu, true, A); m3mul(P, A, P);
    for (int k = 0; k < 9; ++k) Q[k] = Q[k] + P[k];
}

// pack a Hermitian 6x6 (row-major) into 36 reals: diagonal, then lower triangle
__device__ void pack_herm6(const cd *A, double *out)
{
    for (int a = 0; a < 6; ++a) out[a] = A[a * 6 + a].r;
    int k = 6;
    for (int a = 1; a < 6; ++a)
        for (int b = 0; b < a; ++b) {
            out[k++] = A[a * 6 + b].r;
            out[k++] = A[a * 6 + b].i;
        }
}

// inverse of a 6x6 complex matrix, Gauss-Jordan with partial pivoting;
// returns false on an exactly zero pivot
__device__ bool invert6(const cd *A, cd *Ai)
{
    cd M[6][12];
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 12; ++j)
            M[i][j] = (j < 6) ? A[i * 6 + j] : cd{(j - 6 == i) ? 1.0 : 0.0, 0.0};
    for (int col = 0; col < 6; ++col) {
        int piv = col;
        double best = norm2(M[col][col]);
        for (int r = col + 1; r < 6; ++r)
            if (norm2(M[r][col]) > best) { best = norm2(M[r][col]); piv = r; }
        if (best == 0.0) return false;
        if (piv != col)
            for (int j = 0; j < 12; ++j) { cd t = M[col][j]; M[col][j] = M[piv][j]; M[piv][j] = t; }
        const cd d = M[col][col];
        const double dn = norm2(d);
        const cd inv = {d.r / dn, -d.i / dn};
        for (int j = 0; j < 12; ++j) M[col][j] = M[col][j] * inv;
        for (int r = 0; r < 6; ++r) {
            if (r == col) continue;
            const cd f = M[r][col];
            for (int j = 0; j < 12; ++j) M[r][j] = M[r][j] - f * M[col][j];
        }
    }
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j) Ai[i * 6 + j] = M[i][6 + j];
    return true;
}

// The whole build with FP64 instructions, for links without a fixed-point copy
// (*no_fix == 0: k_clover_leaves and k_clover_assemble have built it).
__global__ void k_clover_build(Geom g, Gauge64 U, double kappa, double csw, double2 *C64, double2 *Ci64, int *bad,
                               const int *no_fix)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.V || (no_fix && *no_fix == 0)) return;
    int c[4];
    site_coords(g, x, c);
    cd F[6][9];
    int p = 0;
    for (int mu = 0; mu < 4; ++mu)
        for (int nu = mu + 1; nu < 4; ++nu, ++p) {
            cd Q[9];
            clover_leaves(g, U, c, x, mu, nu, Q);
            for (int k = 0; k < 9; ++k) {
                const cd qd = conj(Q[(k % 3) * 3 + k / 3]);
                F[p][k] = 0.125 * (Q[k] - qd);
            }
        }
    const double kc = kappa * csw;
    const size_t base = ((size_t)(x >> g.lvb) * 36 << g.lvb) + (x & ((1 << g.lvb) - 1));
    for (int chi = 0; chi < 2; ++chi) {
        cd A[36], Ai[36];
        for (int s = 0; s < 2; ++s)
            for (int a = 0; a < 3; ++a)
                for (int t = 0; t < 2; ++t)
                    for (int b = 0; b < 3; ++b) {
                        cd acc = {(s == t && a == b) ? 1.0 : 0.0, 0.0};
                        for (int q = 0; q < 6; ++q) {
                            const cd sg = {c_sigma[chi][q][s][t][0], c_sigma[chi][q][s][t][1]};
                            // i kappa c_SW sigma F
                            const cd term = sg * F[q][a * 3 + b];
                            acc = acc + kc * times_i(term);
                        }
                        A[(s * 3 + a) * 6 + (t * 3 + b)] = acc;
                    }
        double pk[36];
        pack_herm6(A, pk);
        for (int k = 0; k < 18; ++k) C64[base + ((size_t)(chi * 18 + k) << g.lvb)] = make_double2(pk[2 * k], pk[2 * k + 1]);
        if (!invert6(A, Ai)) atomicAdd(bad, 1);
        pack_herm6(Ai, pk);
        for (int k = 0; k < 18; ++k) Ci64[base + ((size_t)(chi * 18 + k) << g.lvb)] = make_double2(pk[2 * k], pk[2 * k + 1]);
    }
}

// ---- the build from the fixed-point links (fix64.cuh): the leaves' matrix
// products on the integer multiply-add units, one thread per site and plane, then
// C and C^-1 per site with FP64 instructions.  24^3 x 48: 2.2 and 2.3 ms (leaves of
// weak fields, which run on FP64 instructions, 8.8 ms), against 19.1 ms with FP64
// products, a generic sigma table and Gauss-Jordan elimination throughout, bound by
// the FP64 pipe.  Error of C^-1 against quadruple precision: 9.4e-17 (1.5e-16 by
// elimination).

// the links of the four leaves at x in the plane (mu, nu) in loop order: the
// shifts (dm, dn) of the link's site, its direction (0: mu, 1: nu), its dagger
struct LeafLink {
    signed char dm, dn, dir, dag;
};
__constant__ LeafLink c_leaves[4][4] = {
    {{0, 0, 0, 0}, {1, 0, 1, 0}, {0, 1, 0, 1}, {0, 0, 1, 1}},
    {{0, 0, 1, 0}, {-1, 1, 0, 1}, {-1, 0, 1, 1}, {-1, 0, 0, 0}},
    {{-1, 0, 0, 1}, {-1, -1, 1, 1}, {-1, -1, 0, 0}, {0, -1, 1, 0}},
    {{0, -1, 1, 1}, {0, -1, 0, 0}, {1, -1, 1, 0}, {0, 0, 0, 1}},
};

// a row of P (three complex limbs) times A, both in units of 2^-60: out in units of
// 2^-(56 + L), L < 32
__device__ __forceinline__ void fix_row_mul(const int4 p[3], const FixM3 &A, int L, Cx<fix_t> out[3])
{
    const fix_t half = 0x80000000LL >> L;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        fix_t hr = 0, hi = 0, mr = half, mi = half;
#pragma unroll
        for (int k = 0; k < 3; ++k) fix_cmac(A.e[k * 3 + j], p[k], hr, mr, hi, mi);
        out[j] = Cx<fix_t>{fix_join_bits(hr, mr, L), fix_join_bits(hi, mi, L)};
    }
}

// The magnitudes of the terms of the nine reals of Q - Q^+ (below) in the product
// P A, added to S in units of 2^-56 of the scaled links
__device__ __forceinline__ void leaf_terms(const FixM3 &P, const FixM3 &A, float *S, int stride)
{
    auto mag = [](int hi) { return (float)abs(hi); };
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            float re = 0.f, im = 0.f;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float pr = mag(P.e[3 * a + k].x), pi = mag(P.e[3 * a + k].z);
                const float ar = mag(A.e[3 * k + b].x), ai = mag(A.e[3 * k + b].z);
                if (a != b) re = fmaf(pr, ar, fmaf(pi, ai, re));
                im = fmaf(pr, ai, fmaf(pi, ar, im));
            }
            if (a == b) {
                S[a * stride] += 2.f * im;
            } else {
                const int hi = a > b ? a : b, lo = a > b ? b : a, o = 3 + 2 * (hi - 1 + lo);
                S[o * stride] += re;
                S[(o + 1) * stride] += im;
            }
        }
}

// The same nine reals with FP64 instructions from the links themselves, in units of
// 2^-59
__device__ __noinline__ void leaves_fp64(Geom g, Gauge64 U, int x, int mu, int nu, double *G)
{
    const double scale = 0x1p59;
    int c[4];
    site_coords(g, x, c);
    cd Q[9];
    clover_leaves(g, U, c, x, mu, nu, Q);
    for (int k = 0; k < 3; ++k) G[k] = scale * (2 * Q[4 * k].i);
    int o = 3;
    for (int a = 1; a < 3; ++a)
        for (int b = 0; b < a; ++b) {
            G[o++] = scale * (Q[3 * a + b].r - Q[3 * b + a].r);
            G[o++] = scale * (Q[3 * a + b].i + Q[3 * b + a].i);
        }
}

// Q - Q^+ of plane blockIdx.y at every site, Q the sum of its four leaves, from those
// of the scaled links times unscale = 1 / k'^4: three imaginary diagonals and the
// entries (1,0), (2,0), (2,1), nine reals in units of 2^-59, to F as reals 9 plane + k
// of a packed clover term.
// Their error is some units whatever their size, with FP64 instructions it goes with
// the terms' magnitudes: fields exp(i eps H) have the same error, 2.6e-16 of the
// off-diagonal reals, at eps = 0.11.  A site and plane with a real whose terms (those
// of the last products, leaf_terms) stay below LEAF_LEAST, which such fields do and
// fields of eps >= 0.3 do not (smallest of 1.5e5 reals 2^55.4; k' = 1/2, the worst),
// is computed with FP64 instructions.
constexpr float LEAF_LEAST = 0x1p52f;  // 2^55 units
__global__ void __launch_bounds__(128, 4) k_clover_leaves(Geom g, FixLinks U, Gauge64 Ud, double unscale, double *F,
                                                          const int *no_fix)
{
    __shared__ float terms[9 * 128];
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.V || *no_fix) return;
    const int p = blockIdx.y;
    const int mu = p < 3 ? 0 : (p < 5 ? 1 : 2);
    const int nu = p < 3 ? p + 1 : (p < 5 ? p - 1 : 3);
    int c[4];
    site_coords(g, x, c);
    fix_t G[9];
    float *const S = terms + threadIdx.x;  // this thread's
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        G[k] = 0;
        S[k * 128] = 0.f;
    }
#pragma unroll 1
    for (int leaf = 0; leaf < 4; ++leaf) {
        FixM3 P;
#pragma unroll 1
        for (int step = 0; step < 4; ++step) {
            const LeafLink w = c_leaves[leaf][step];
            int n[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                int v = c[k] + (k == mu ? w.dm : 0) + (k == nu ? w.dn : 0);
                v = v < 0 ? v + g.L[k] : (v >= g.L[k] ? 0 : v);
                n[k] = v;
            }
            const int site = site_index(g, n), dir = w.dir ? nu : mu;
            if (step == 0) {
                P.load(U, site, dir, w.dag);
                continue;
            }
            FixM3 A;
            A.load(U, site, dir, w.dag);
            if (step == 3) leaf_terms(P, A, S, 128);
            Cx<fix_t> r[9];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                fix_row_mul(P.e + 3 * a, A, step == 3 ? 3 : 4, r + 3 * a);
                if (step < 3)
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        int4 &o = P.e[3 * a + k];
                        fix_limbs(r[3 * a + k].r, o.x, o.y);
                        fix_limbs(r[3 * a + k].i, o.z, o.w);
                    }
            }
            if (step == 3) {
#pragma unroll
                for (int k = 0; k < 3; ++k) G[k] += 2 * r[4 * k].i;
                int o = 3;
#pragma unroll
                for (int a = 1; a < 3; ++a)
#pragma unroll
                    for (int b = 0; b < a; ++b) {
                        G[o++] += r[3 * a + b].r - r[3 * b + a].r;
                        G[o++] += r[3 * a + b].i + r[3 * b + a].i;
                    }
            }
        }
    }
    double *o = F + 2 * (((size_t)(x >> g.lvb) * 36 << g.lvb) + (x & ((1 << g.lvb) - 1)));
    auto put = [&](int k, double v) {
        const int r = 9 * p + k;
        o[((size_t)(r >> 1) << (g.lvb + 1)) + (r & 1)] = v;
    };
    bool fine = true;
#pragma unroll
    for (int k = 0; k < 9; ++k) fine = fine && S[k * 128] >= LEAF_LEAST;
    if (fine) {
#pragma unroll
        for (int k = 0; k < 9; ++k) put(k, unscale * __ll2double_rn(G[k]));
    } else {
        double D[9];
        leaves_fp64(g, Ud, x, mu, nu, D);
        for (int k = 0; k < 9; ++k) put(k, D[k]);
    }
}

// The inverse of a Hermitian positive definite 6x6 matrix from its lower triangle
// A[a(a+1)/2 + b], in place (A = L D L^+ without pivoting, which is stable for such
// matrices); false when a pivot is not positive.
__device__ __forceinline__ bool invert_hpd6(cd A[21])
{
    auto at = [](int a, int b) { return a * (a + 1) / 2 + b; };
    double id[6];
    bool ok = true;
    // A -> unit lower L (below the diagonal), 1/d in id
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const double d = A[at(j, j)].r;
        ok = ok && d > 0;
        id[j] = 1.0 / d;
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            const cd l = id[j] * A[at(i, j)];
            // the columns to the right: A_ik -= L_ij d conj(L_kj) = l conj(A_kj)
#pragma unroll
            for (int k = j + 1; k <= i; ++k) {
                const cd v = k == i ? A[at(i, j)] : A[at(k, j)];
                cd &t = A[at(i, k)];
                t.r = fma(-l.r, v.r, fma(-l.i, v.i, t.r));
                if (k < i) t.i = fma(-l.i, v.r, fma(l.r, v.i, t.i));
            }
        }
#pragma unroll
        for (int i = j + 1; i < 6; ++i) A[at(i, j)] = id[j] * A[at(i, j)];
    }
    // L -> L^-1
#pragma unroll
    for (int j = 0; j < 6; ++j)
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            cd t = A[at(i, j)];
#pragma unroll
            for (int k = j + 1; k < i; ++k) t = cfma(A[at(i, k)], A[at(k, j)], t);
            A[at(i, j)] = -t;
        }
    // A^-1 = L^-+ D^-1 L^-1
#pragma unroll
    for (int a = 0; a < 6; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b) {
            // sum over k >= a of conj(Li_ka) Li_kb / d_k
            cd t = a == b ? cd{id[a], 0.0} : id[a] * A[at(a, b)];
#pragma unroll
            for (int k = a + 1; k < 6; ++k) {
                const cd u = A[at(k, a)], v = id[k] * A[at(k, b)];
                t.r = fma(u.r, v.r, fma(u.i, v.i, t.r));
                if (a != b) t.i = fma(u.r, v.i, fma(-u.i, v.r, t.i));
            }
            // row a of L^-1 is still needed by rows above only through k > a
            A[at(a, b)] = t;
        }
    return ok;
}

// the packed Hermitian block pk[36] and its inverse, by elimination with pivoting
__device__ __noinline__ bool invert_general(const double *pk, double *out)
{
    cd A[36], I[36];
    for (int a = 0; a < 6; ++a) A[a * 7] = cd{pk[a], 0.0};
    int k = 6;
    for (int a = 1; a < 6; ++a)
        for (int b = 0; b < a; ++b, k += 2) {
            A[a * 6 + b] = cd{pk[k], pk[k + 1]};
            A[b * 6 + a] = cd{pk[k], -pk[k + 1]};
        }
    const bool ok = invert6(A, I);
    pack_herm6(I, out);
    return ok;
}

// C = 1 + f sum sigma i (Q - Q^+) and C^-1 from k_clover_leaves' reals, f = kappa
// c_SW 2^-62; Ci64 holds those reals on entry
__global__ void __launch_bounds__(128, 3) k_clover_assemble(Geom g, double f, double2 *C64, double2 *Ci64, int *bad,
                                                         const int *no_fix)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.V || *no_fix) return;
    const size_t blk = x >> g.lvb, l = x & ((1 << g.lvb) - 1);
    const size_t base = (blk * 36 << g.lvb) + l;
    double G[54];
#pragma unroll
    for (int k = 0; k < 27; ++k) {
        const double2 v = Ci64[base + ((size_t)k << g.lvb)];
        G[2 * k] = f * v.x;
        G[2 * k + 1] = f * v.y;
    }
#pragma unroll
    for (int chi = 0; chi < 2; ++chi) {
        cd A[21];
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int t = 0; t < 2; ++t)
#pragma unroll
                    for (int b = 0; b < 3; ++b) {
                        const int r = 3 * s + a, cc = 3 * t + b;
                        if (cc > r) continue;
                        cd acc = {r == cc ? 1.0 : 0.0, 0.0};
#pragma unroll
                        for (int p = 0; p < 6; ++p) {
                            const double sr = c_sigma[chi][p][s][t][0], si = c_sigma[chi][p][s][t][1];
                            if (sr == 0.0 && si == 0.0) continue;
                            // i (Q - Q^+)_ab: Hermitian; its lower triangle from G
                            cd h;
                            if (a == b) h = cd{-G[9 * p + a], 0.0};
                            else {
                                const int hi = a > b ? a : b, lo = a > b ? b : a, o = 3 + 2 * (hi - 1 + lo);
                                const double vr = G[9 * p + o], vi = G[9 * p + o + 1];
                                h = a > b ? cd{-vi, vr} : cd{-vi, -vr};
                            }
                            acc.r = sr != 0.0 ? acc.r + sr * h.r : acc.r - si * h.i;
                            if (r != cc) acc.i = sr != 0.0 ? acc.i + sr * h.i : acc.i + si * h.r;
                        }
                        A[r * (r + 1) / 2 + cc] = acc;
                    }
        double pk[36];
#pragma unroll
        for (int a = 0; a < 6; ++a) pk[a] = A[a * (a + 1) / 2 + a].r;
        int k = 6;
#pragma unroll
        for (int a = 1; a < 6; ++a)
#pragma unroll
            for (int b = 0; b < a; ++b) {
                pk[k++] = A[a * (a + 1) / 2 + b].r;
                pk[k++] = A[a * (a + 1) / 2 + b].i;
            }
#pragma unroll
        for (int m = 0; m < 18; ++m)
            C64[base + ((size_t)(chi * 18 + m) << g.lvb)] = make_double2(pk[2 * m], pk[2 * m + 1]);
    }
    // the inverses, from C64 again: both blocks' reals and a block do not fit the registers
#pragma unroll 1
    for (int chi = 0; chi < 2; ++chi) {
        double pk[36];
        auto get = [&]() {
#pragma unroll
            for (int m = 0; m < 18; ++m) {
                const double2 v = C64[base + ((size_t)(chi * 18 + m) << g.lvb)];
                pk[2 * m] = v.x;
                pk[2 * m + 1] = v.y;
            }
        };
        get();
        cd A[21];
#pragma unroll
        for (int a = 0; a < 6; ++a) A[a * (a + 1) / 2 + a] = cd{pk[a], 0.0};
        int k = 6;
#pragma unroll
        for (int a = 1; a < 6; ++a)
#pragma unroll
            for (int b = 0; b < a; ++b, k += 2) A[a * (a + 1) / 2 + b] = cd{pk[k], pk[k + 1]};
        if (invert_hpd6(A)) {
            // X <- 1 - B X with B = C - 1, which multiplies X's error by B: taken where
            // B's Frobenius norm, and with it its largest eigenvalue, is below one.
            // Emulated, elimination with pivoting 1.4e-16 to 1.7e-16: 5.5e-17 at a
            // squared norm of 0.07 (c_SW = 1), 1.0e-16 at 0.95; without the step
            // 1.2e-16 to 1.4e-16.
            cd X[21];
            double n = 0;
#pragma unroll
            for (int a = 0; a < 6; ++a) {
                cd B[6];
#pragma unroll
                for (int j = 0; j < 6; ++j) {
                    const int hi = a > j ? a : j, lo = a > j ? j : a, o = 6 + hi * (hi - 1) + 2 * lo;
                    if (a == j) B[j] = cd{pk[a] - 1.0, 0.0};
                    else B[j] = cd{pk[o], a > j ? pk[o + 1] : -pk[o + 1]};
                    n += norm2(B[j]);
                }
#pragma unroll
                for (int b = 0; b <= a; ++b) {
                    cd t = {0, 0};
#pragma unroll
                    for (int j = 0; j < 6; ++j) {
                        const cd x = j >= b ? A[j * (j + 1) / 2 + b] : conj(A[b * (b + 1) / 2 + j]);
                        t = j == b ? cd{fma(B[j].r, x.r, t.r), fma(B[j].i, x.r, t.i)} : cfma(B[j], x, t);
                    }
                    X[a * (a + 1) / 2 + b] = a == b ? cd{1.0 - t.r, 0.0} : -t;
                }
            }
            if (n < 1.0)
#pragma unroll
                for (int m = 0; m < 21; ++m) A[m] = X[m];
#pragma unroll
            for (int a = 0; a < 6; ++a) pk[a] = A[a * (a + 1) / 2 + a].r;
            k = 6;
#pragma unroll
            for (int a = 1; a < 6; ++a)
#pragma unroll
                for (int b = 0; b < a; ++b) {
                    pk[k++] = A[a * (a + 1) / 2 + b].r;
                    pk[k++] = A[a * (a + 1) / 2 + b].i;
                }
        } else {
            double in[36], out[36];
            get();
#pragma unroll
            for (int m = 0; m < 36; ++m) in[m] = pk[m];
            if (!invert_general(in, out)) atomicAdd(bad, 1);
#pragma unroll
            for (int m = 0; m < 36; ++m) pk[m] = out[m];
        }
#pragma unroll
        for (int m = 0; m < 18; ++m)
            Ci64[base + ((size_t)(chi * 18 + m) << g.lvb)] = make_double2(pk[2 * m], pk[2 * m + 1]);
    }
}

int launch_clover_build(const Geom &g, const double2 *U64, const int4 *UQ, double ks, const int *no_fix, double kappa,
                        double csw, double2 *C64, double2 *Ci64, int *d_bad, cudaStream_t s)
{
    if (UQ) {
        k_clover_leaves<<<dim3(grid_for(g.V, 128), 6), 128, 0, s>>>(g, FixLinks{UQ, g.lvb}, Gauge64{(double2 *)U64, g.lvb},
                                                                    1 / (ks * ks * ks * ks), (double *)Ci64, no_fix);
        k_clover_assemble<<<grid_for(g.V, 128), 128, 0, s>>>(g, kappa * csw * 0x1p-62, C64, Ci64, d_bad, no_fix);
        count(2, (double)g.V * (576.0 + 2 * 432.0 + 2 * 576.0));
    }
    k_clover_build<<<grid_for(g.V, 128), 128, 0, s>>>(g, Gauge64{(double2 *)U64, g.lvb}, kappa, csw, C64, Ci64, d_bad,
                                                      UQ ? no_fix : nullptr);
    MGC_CUDA(cudaGetLastError());
    count(1, UQ ? 0.0 : (double)g.V * (576.0 + 2 * 576.0));
    return MGC_OK;
}

// FP64 packed clover -> FP32 (18 float4 planes) or FP16 (9 x 8 halves + scale)
__global__ void k_clover_lowprec(Geom g, Clover64 C, int prec, void *out)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.V) return;
    double c[72];
    C.load(x, c);
    const size_t l = x & ((1 << g.lvb) - 1), blk = x >> g.lvb;
    if (prec == 32) {
        float4 *o = (float4 *)out + (blk * 18 << g.lvb) + l;
        for (int k = 0; k < 18; ++k)
            o[(size_t)k << g.lvb] = make_float4((float)c[4 * k], (float)c[4 * k + 1], (float)c[4 * k + 2], (float)c[4 * k + 3]);
    } else {
        float m = 0.f;
        for (int k = 0; k < 72; ++k) m = fmaxf(m, fabsf((float)c[k]));
        const float inv = m > 0.f ? 1.0f / m : 0.f;
        uint4 *o = (uint4 *)out + (blk * 9 << g.lvb) + l;
        float *sc = (float *)((uint4 *)out + (size_t)g.V * 9);
        for (int k = 0; k < 9; ++k) {
            const double *q = c + 8 * k;
            o[(size_t)k << g.lvb] = make_uint4(pack_half2((float)q[0] * inv, (float)q[1] * inv),
                                               pack_half2((float)q[2] * inv, (float)q[3] * inv),
                                               pack_half2((float)q[4] * inv, (float)q[5] * inv),
                                               pack_half2((float)q[6] * inv, (float)q[7] * inv));
        }
        sc[x] = m;
    }
}

int launch_clover_lowprec(const Geom &g, const double2 *C64, int prec, void *out, cudaStream_t s)
{
    k_clover_lowprec<<<grid_for(g.V, 256), 256, 0, s>>>(g, Clover64{(double2 *)C64, g.lvb}, prec, out);
    MGC_CUDA(cudaGetLastError());
    count(1, (double)g.V * (576.0 + clover_site_bytes(prec)));
    return MGC_OK;
}

// packed FP64 clover -> canonical [s][12][12] complex128
__global__ void k_clover_export(Geom g, Clover64 C, double2 *out)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.V) return;
    int c[4];
    site_coords(g, x, c);
    double d[72];
    C.load(x, d);
    double2 *o = out + canon_index(g, c) * 144;
    for (int k = 0; k < 144; ++k) o[k] = make_double2(0.0, 0.0);
    for (int chi = 0; chi < 2; ++chi) {
        const double *q = d + 36 * chi;
        const int off = 6 * chi;
        for (int a = 0; a < 6; ++a) o[(off + a) * 12 + off + a] = make_double2(q[a], 0.0);
        int k = 6;
        for (int a = 1; a < 6; ++a)
            for (int b = 0; b < a; ++b) {
                o[(off + a) * 12 + off + b] = make_double2(q[k], q[k + 1]);
                o[(off + b) * 12 + off + a] = make_double2(q[k], -q[k + 1]);
                k += 2;
            }
    }
}

int launch_clover_export(const Geom &g, const double2 *C64, double *out, cudaStream_t s)
{
    k_clover_export<<<grid_for(g.V, 128), 128, 0, s>>>(g, Clover64{(double2 *)C64, g.lvb}, (double2 *)out);
    MGC_CUDA(cudaGetLastError());
    count(1, (double)g.V * (576.0 + 144 * 16.0));
    return MGC_OK;
}

// max over links of max|U U^+ - 1| and |det U - 1|, for 12-real compression
__global__ void k_unitarity(long long nlinks, const double2 *__restrict__ canon, unsigned long long *maxerr)
{
    const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    double err = 0.0;
    if (n < nlinks) {
        cd u[9];
        for (int k = 0; k < 9; ++k) u[k] = cd{canon[n * 9 + k].x, canon[n * 9 + k].y};
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) {
                cd acc = {0, 0};
                for (int k = 0; k < 3; ++k) acc = cfma(u[i * 3 + k], conj(u[j * 3 + k]), acc);
                if (i == j) acc.r -= 1.0;
                err = fmax(err, sqrt(norm2(acc)));
            }
        cd det = u[0] * (u[4] * u[8] - u[5] * u[7]) - u[1] * (u[3] * u[8] - u[5] * u[6]) +
                 u[2] * (u[3] * u[7] - u[4] * u[6]);
        det.r -= 1.0;
        err = fmax(err, sqrt(norm2(det)));
        if (!(err == err)) err = 1e300;  // NaN
    }
    // non-negative doubles order like their bit patterns
    atomicMax(maxerr, (unsigned long long)__double_as_longlong(err));
}

int launch_unitarity(const Geom &g, const double *canon_dev, double *d_maxerr, cudaStream_t s)
{
    const long long n = (long long)g.V * 4;
    k_unitarity<<<grid_for(n, 256), 256, 0, s>>>(n, (const double2 *)canon_dev, (unsigned long long *)d_maxerr);
    MGC_CUDA(cudaGetLastError());
    count(1, (double)n * 144.0);
    return MGC_OK;
}

}  // namespace mgc
