// Batched multi-RHS D with FP64 storage: one launch of the fixed-point operator
// (fix64.cuh) where a lattice of the batch has its fixed-point copies, in which the
// lattices without take FP64 instructions at every site; FP64 instructions with links
// shared between right-hand sides (kernel in dirac_batch.cuh) where none has.  All are
// bit-identical to the single-lattice operator.  The mixed launch is no slower than
// one of each kind, FP64 instructions being what bounds it: two lattices 16^3 x 32
// with four right-hand sides each, one with copies, 1286 us against 1300 us.
#include "dirac_batch.cuh"
#include "fix64.cuh"

namespace mgc {

namespace {
// one right-hand side of one site per thread, thread blocks numbered as in DiracBatch
struct DiracBatchFix {
    int n;
    int rhs_fast;
    int end[MGC_BATCH_MAX];
    int nsb[MGC_BATCH_MAX];
    int nrhs[MGC_BATCH_MAX];
    Geom g[MGC_BATCH_MAX];
    Spinor64 in[MGC_BATCH_MAX], out[MGC_BATCH_MAX];
    FixLinks UQ[MGC_BATCH_MAX];
    FixClover CQ[MGC_BATCH_MAX];
    Gauge64 U[MGC_BATCH_MAX];
    Clover64 C[MGC_BATCH_MAX];
    double kappa[MGC_BATCH_MAX];
};

template <bool DAG, int LVB>
__global__ void __launch_bounds__(FIX_THREADS, 3) k_dirac_batch_fix(DiracBatchFix B)
{
    __shared__ int4 slots[(FIX_SPINOR_SLOTS + FIX_LINK_SLOTS) * FIX_THREADS];
    int k = 0;
    while (k < B.n - 1 && (int)blockIdx.x >= B.end[k]) ++k;
    const int local = blockIdx.x - (k ? B.end[k - 1] : 0);
    const int sb = B.rhs_fast ? local / B.nrhs[k] : local % B.nsb[k];
    const int r = B.rhs_fast ? local % B.nrhs[k] : local / B.nsb[k];
    Geom g = B.g[k];
    const int i = sb * FIX_THREADS + threadIdx.x;
    const unsigned lanes = __ballot_sync(0xffffffffu, i < g.V);
    if (i >= g.V) return;
    Spinor64 src = shift_rhs(B.in[k], r, g.V), dst = shift_rhs(B.out[k], r, g.V);
    FixLinks U = B.UQ[k];
    FixClover C = B.CQ[k];
    if (LVB > 0) {
        g.lvb = LVB;
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) g.lb[mu] = LVB / 4;
        src.lvb = dst.lvb = U.lvb = C.lvb = LVB;
    }
    const bool done = C.p && fix_dirac_site<DAG>(g, i, src, dst, U, C, slots + threadIdx.x);
    __syncwarp(lanes);
    if (!done)
        fix_fallback<DAG>(g, i, src, dst, B.U[k], B.C[k], B.kappa[k]);
}

int dirac_batch_fix(const BatchSpec &spec, bool dag, const void *const *in, void *const *out, cudaStream_t s)
{
    const Geom &g0 = spec.ops[0]->gauge->lat->g;
    const bool cube = g0.lb[0] == g0.lb[1] && g0.lb[1] == g0.lb[2] && g0.lb[2] == g0.lb[3];
    DiracBatchFix B;
    B.n = spec.n;
    B.rhs_fast = spec.rhs_fast;
    int acc = 0;
    for (int k = 0; k < spec.n; ++k) {
        const mgc_clover_s *op = spec.ops[k];
        const Geom &g = op->gauge->lat->g;
        B.g[k] = g;
        B.nrhs[k] = spec.nrhs[k];
        B.nsb[k] = grid_for(g.V, FIX_THREADS);
        acc += B.nsb[k] * spec.nrhs[k];
        B.end[k] = acc;
        B.in[k] = sp64(g, in[k]);
        B.out[k] = sp64(g, out[k]);
        B.UQ[k] = FixLinks{op->UQ, g.lvb};
        B.CQ[k] = FixClover{op->CQ, op->CE, op->fix_ek, g.lvb};
        B.U[k] = Gauge64{op->gauge->U64, g.lvb};
        B.C[k] = Clover64{op->C64, g.lvb};
        B.kappa[k] = op->kappa;
    }
#define MGC_DBF_LAUNCH(L)                                                          \
    do {                                                                           \
        if (dag) k_dirac_batch_fix<true, L><<<acc, FIX_THREADS, 0, s>>>(B);        \
        else k_dirac_batch_fix<false, L><<<acc, FIX_THREADS, 0, s>>>(B);           \
    } while (0)
    if (cube && g0.lvb == 8) MGC_DBF_LAUNCH(8);
    else if (cube && g0.lvb == 4) MGC_DBF_LAUNCH(4);
    else MGC_DBF_LAUNCH(0);
#undef MGC_DBF_LAUNCH
    MGC_CUDA(cudaGetLastError());
    return MGC_OK;
}
}  // namespace

int dirac_batch_64(const BatchSpec &spec, bool dag, const void *const *in, void *const *out, int rb, int threads,
                   cudaStream_t s)
{
    for (int k = 0; k < spec.n; ++k)
        if (spec.ops[k]->CQ) return dirac_batch_fix(spec, dag, in, out, s);
    DiracBatch<Spinor64, Gauge64, Clover64> B;
    for (int k = 0; k < spec.n; ++k) {
        const mgc_clover_s *op = spec.ops[k];
        const Geom &g = op->gauge->lat->g;
        B.in[k] = sp64(g, in[k]);
        B.out[k] = sp64(g, out[k]);
        B.U[k] = Gauge64{op->gauge->U64, g.lvb};
        B.C[k] = Clover64{op->C64, g.lvb};
    }
    return dirac_batch_rb(B, spec, dag, rb, threads, s);
}

}  // namespace mgc
