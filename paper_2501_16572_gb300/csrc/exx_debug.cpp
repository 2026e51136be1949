// Host-only inspection hooks (include/exx_debug.h).
#include "exx_internal.h"
#include "../../include/exx_debug.h"

#include <algorithm>

extern "C" {

int exx_debug_tc3_layout(int n1, int n2, int n3, int share01, int *out)
{
    if (n1 < 2 || n2 < 2 || n3 < 2 || n1 > 256 || n2 > 256 || n3 > 256 || !out) return EXX_ERR_INVALID_ARG;
    exx::tc3_debug_layout(n1, n2, n3, share01 != 0, out);
    return EXX_OK;
}

int exx_debug_tc3_direct(int n1, int n2, int n3, int share01, int *out)
{
    if (n1 < 2 || n2 < 2 || n3 < 2 || n1 > 256 || n2 > 256 || n3 > 256 || !out) return EXX_ERR_INVALID_ARG;
    exx::tc3_debug_direct(n1, n2, n3, share01 != 0, out);
    return EXX_OK;
}

int exx_debug_tc_passes(int prec, int Np, int *out)
{
    if (prec <= EXX_PREC_FP64 || prec >= EXX_PREC_BF16X7 || Np < 16 || Np > 256 || Np % 16 || !out) return EXX_ERR_INVALID_ARG;
    exx::tc_debug_passes(prec, Np, out);
    return EXX_OK;
}

int exx_debug_matrix_digits(int nout, int nk, const double *C, int WN, int Kp, int n0, int k0, float *digits,
                            float *scales)
{
    if (nout < 1 || nk < 1 || WN < 1 || Kp < 8 || Kp % 8 || WN % 8 || n0 < 0 || k0 < 0 || !C || !digits || !scales)
        return EXX_ERR_INVALID_ARG;
    exx::tc3_debug_matrix_digits(nout, nk, C, WN, Kp, n0, k0, digits, scales);
    return EXX_OK;
}

int exx_debug_fd_weights(int p, double *w)
{
    if (p < 1 || p > 12 || !w) return EXX_ERR_INVALID_ARG;
    exx::fd_weights(p, w);
    return EXX_OK;
}

int exx_debug_second_derivative(int n, double h, int bc, int p, double *D)
{
    if (n < 1 || p < 1 || p > 12 || !D || !(h > 0)) return EXX_ERR_INVALID_ARG;
    exx::second_derivative(n, h, bc, p, D);
    return EXX_OK;
}

int exx_debug_sym_eig(int n, const double *A, double *V, double *lam)
{
    if (n < 1 || !A || !V || !lam) return EXX_ERR_INVALID_ARG;
    return exx::sym_eig(n, A, V, lam) ? EXX_ERR_UNSUPPORTED : EXX_OK;
}

int exx_debug_schedule(int n_occ, int n_in, int aliased, int block, int max_pairs, long *npairs,
                       long *nbatches, long *nblocks, int *pairs, int *batches, int *blocks)
{
    if (n_occ < 1 || n_in < 1 || block < 1 || block > 32 || max_pairs < 1 || !npairs || !nbatches || !nblocks)
        return EXX_ERR_INVALID_ARG;
    exx::Schedule S = exx::build_schedule(n_occ, n_in, aliased != 0, block, max_pairs);
    *npairs = long(S.pairs.size());
    *nbatches = long(S.batches.size());
    *nblocks = long(S.blocks.size());
    if (pairs)
        for (size_t i = 0; i < S.pairs.size(); ++i) {
            pairs[2 * i] = S.pairs[i].x;
            pairs[2 * i + 1] = S.pairs[i].y;
        }
    if (batches)
        for (size_t i = 0; i < S.batches.size(); ++i) {
            batches[3 * i] = S.batches[i].nfields;
            batches[3 * i + 1] = S.batches[i].block0;
            batches[3 * i + 2] = S.batches[i].nblocks;
        }
    if (blocks)
        for (size_t i = 0; i < S.blocks.size(); ++i) {
            const exx::Block &b = S.blocks[i];
            int v[6] = {b.I0, b.nI, b.J0, b.nJ, b.kind, b.field0};
            std::copy(v, v + 6, blocks + 6 * i);
        }
    return EXX_OK;
}

int exx_debug_plan_schedule(long N, int prec, int world, int pairs_per_batch, int block_orbitals, int n_occ, int n_in,
                            int aliased, int *limits, long *nbatches, int *batches)
{
    if (N < 1 || world < 1 || pairs_per_batch < 0 || block_orbitals < 0 || block_orbitals > 32 || n_occ < 1 || n_in < 1 ||
        !limits || !nbatches)
        return EXX_ERR_INVALID_ARG;
    exx::schedule_limits(N, prec, world, pairs_per_batch, block_orbitals, limits[0], limits[1]);
    const exx::Schedule S = exx::build_schedule(n_occ, n_in, aliased != 0, limits[0], limits[1], world);
    *nbatches = long(S.batches.size());
    if (batches)
        for (size_t i = 0; i < S.batches.size(); ++i) {
            batches[2 * i] = S.batches[i].nfields;
            batches[2 * i + 1] = S.blocks[S.batches[i].block0].kind == exx::BLK_ONE_SIDE;
        }
    return EXX_OK;
}

int exx_debug_gemm_shape(long m, int n, long K, int ktri, int num_sms, long budget, long *out)
{
    if (m < 1 || n < 1 || K < 1 || num_sms < 1 || budget < 1 || !out) return EXX_ERR_INVALID_ARG;
    const exx::GemmShape g = exx::gemm_shape({m, n, K, ktri != 0}, num_sms, budget);
    const long v[] = {g.rt, g.nt, g.Nt, g.mslab, g.kslab, g.Zmax, g.ktri, long(g.offB), long(g.offSA),
                      long(g.offSB), long(g.offP), long(g.bytes)};
    std::copy(v, v + 12, out);
    return EXX_OK;
}

int exx_debug_limits(exx_plan plan, long gemm_budget, long workspace_cap)
{
    exx::Plan *P = reinterpret_cast<exx::Plan *>(plan);
    if (!P || gemm_budget < 0 || workspace_cap < 0) return EXX_ERR_INVALID_ARG;
    P->gemm_budget = gemm_budget ? gemm_budget : exx::Plan().gemm_budget;
    P->ws_cap = size_t(workspace_cap);
    return EXX_OK;
}

int exx_debug_tc_gemm(int tf32, int n, int k, const float *A, const float *B, float *D, int *err)
{
    if (!A || !B || !D || !err) return EXX_ERR_INVALID_ARG;
    return exx::tc_unit_gemm(tf32, n, k, A, B, D, err);
}

int exx_debug_fastdiv(unsigned d, int count, const unsigned *n, unsigned *q)
{
    if (d < 1 || count < 0 || (count > 0 && (!n || !q))) return EXX_ERR_INVALID_ARG;
    const exx::FastDiv f = exx::make_fastdiv(d);
    for (int i = 0; i < count; ++i) q[i] = exx::fast_div(n[i], f);
    return EXX_OK;
}

int exx_debug_wait_timeout(int *status_h)
{
    if (!status_h) return EXX_ERR_INVALID_ARG;
    return exx::tc_wait_timeout_probe(status_h);
}

int exx_debug_wait_warp(unsigned *went_on_h)
{
    if (!went_on_h) return EXX_ERR_INVALID_ARG;
    return exx::tc_wait_warp_probe(went_on_h);
}

}  // extern "C"
