/*
 * exx_debug.h -- host-only inspection hooks of libexx_gb300, for tests.
 *
 * These run entirely on the CPU (no CUDA call), so the plan-setup mathematics and the
 * pair scheduler can be checked on a machine without a GPU.  They have no counterpart
 * in the paper beyond the steps they expose (Eqs. 6-7 for the eigen-decomposition,
 * Sec. II.B's batches of right-hand sides for the schedule).
 */
#ifndef EXX_GB300_DEBUG_H
#define EXX_GB300_DEBUG_H
#include "exx.h"
#ifdef __cplusplus
extern "C" {
#endif

/* FD weights w[0..p] of the order-2p central second difference (host copy of what a plan uses). */
int exx_debug_fd_weights(int p, double *w);

/* 1D second-derivative operator (n x n column-major) as a plan assembles it. */
int exx_debug_second_derivative(int n, double h, int bc, int p, double *D);

/* The plan's symmetric eigensolver: A (n x n column-major) = V diag(lam) V^T, lam ascending. */
int exx_debug_sym_eig(int n, const double *A, double *V, double *lam);

/* Pair schedule of exx_apply.  First call with NULL arrays to get the sizes; then with
 * pairs (2 ints per pair: m, n), batches (3 ints: nfields, first block, nblocks) and
 * blocks (6 ints: I0, nI, J0, nJ, kind, field0) of at least those sizes. */
int exx_debug_schedule(int n_occ, int n_in, int aliased, int block, int max_pairs, long *npairs,
                       long *nbatches, long *nblocks, int *pairs, int *batches, int *blocks);

/* The batches that exx_apply runs on a plan of N points with these settings (exx_plan_set_precision,
 * _set_shard, _set_batch): limits = {orbitals per pair block, most pairs per batch}; batches (2 ints
 * each: pair fields, 1 when its outputs are those of one side only) may be NULL to get the number. */
int exx_debug_plan_schedule(long N, int prec, int world, int pairs_per_batch, int block_orbitals, int n_occ, int n_in,
                            int aliased, int *limits, long *nbatches, int *batches);

/* How an ACE product D (m x n) = A B^T with a contraction of K is cut when its digit planes may take
 * `budget` bytes: out (HOST long[12]) = rows of a tile, column tiles, columns of each, rows of a slab, 320-long
 * chunks of a slab, k splits, triangular limit in use, then the byte offsets of B's planes, the row
 * scales of A and of B, the split sums, and the total.  ktri: B(j, k) = 0 for k > j. */
int exx_debug_gemm_shape(long m, int n, long K, int ktri, int num_sms, long budget, long *out);

/* A plan's bytes for those digit planes (0 = the default), and the size above which a workspace that
 * has a smaller form counts as out of memory (0 = no such size). */
int exx_debug_limits(exx_plan plan, long gemm_budget, long workspace_cap);

/* One 128 x n x k tensor-core tile (tcgen05.mma, one bf16 or tf32 piece per operand,
 * FP32 accumulation): D (128 x n, row-major) = A (128 x k, row-major) B (n x k,
 * row-major)^T.  DEVICE pointers; n, k multiples of 16 in [16, 256].  Synchronizes the
 * device.  Checks the operand layout and descriptors of the split-precision path. */
int exx_debug_tc_gemm(int tf32, int n, int k, const float *A, const float *B, float *D, int *err);

/* Quotients n[i] / d by the multiply-shift division the pass kernels use for row ->
 * (field, row in field) (Granlund & Montgomery 1994, Fig. 4.1), host-side.  d >= 1. */
int exx_debug_fastdiv(unsigned d, int count, const unsigned *n, unsigned *q);

/* The BF16X7 (three-pass) layouts of the older kernel forms for an n1 x n2 x n3 grid (what a grid gets
 * whose x/y matrices do not stay resident, and hand-made settings), host-side (no device):
 * out (HOST int[16]) = supported; shared memory of pass A and pass C; pass A streams its x/y
 * matrices and their chunk width; the same for pass C; pass A pipelined; pass A staged; pass B
 * shared memory (0 = none fits); pass B K-chunks; its chunk or block width; its buffers; its
 * matrices resident; units per thread; the shared-memory limit.  share01 = 1 when x and y have
 * the same length and boundary condition (one image serves both).  Sizes in [2, 256]. */
int exx_debug_tc3_layout(int n1, int n2, int n3, int share01, int *out);

/* The layouts of the direct kernel forms, which a grid gets by itself (slices: where both matrices stay
 * resident), host-side (no device): out (HOST int[59]) = 20 values each for pass A and pass C and 18 for
 * pass B, in the order that tc3_debug_direct states, and the shared-memory limit. */
int exx_debug_tc3_direct(int n1, int n2, int n3, int share01, int *out);

/* The forms of the five-pass kernels of a split mode (not BF16X7) for blocks of Np points (a multiple of
 * 16), host-side: out (HOST int[36]) = for pass 1, 2, 3 in one kernel, one half of pass 3, 4 and 5 each:
 * fits, staging buffers, accumulator sets, TMEM columns they take, columns allocated, shared memory. */
int exx_debug_tc_passes(int prec, int Np, int *out);

/* The base-512 digit image of the 1D matrices, host-side: C (HOST, row-major nout x nk, row n =
 * output n, column k = contraction index k) cut for a WN x Kp block of rows n0.. and indices
 * k0.. (a K-chunk when k0 > 0 or Kp < nk), decoded from the tensor-core layout back to values:
 * digits (HOST float[4][WN][Kp]) holds the four weighted digits of every entry (their sum times
 * the row's scale is the entry), scales (HOST float[WN]) the column scales.  Every row is
 * scaled by the largest entry of the whole row, so the chunks of a row share one scale.
 * WN and Kp multiples of 8. */
int exx_debug_matrix_digits(int nout, int nk, const double *C, int WN, int Kp, int n0, int k0, float *digits,
                            float *scales);

/* Failure detection without a fault: launches one kernel whose two mbarrier waits (the
 * same bounded waits the pass kernels use: the polled one of the five-pass kernels, 4096
 * polls, and the wall-time one of the three-pass kernels, here 2 ms) wait on a barrier that
 * nothing completes.  Each limit runs out, the kernel records it in an error word and
 * returns; *status_h is then EXX_ERR_TIMEOUT when both waits gave up (EXX_OK otherwise).
 * The context stays usable.  Returns EXX_ERR_CUDA without a GPU. */
int exx_debug_wait_timeout(int *status_h);

/* The wait of the MMA-issuing warps: one kernel in which half of a warp's lanes run out of time
 * before their barrier completes and the other half do not.  *went_on_h (HOST) has a bit for
 * every lane that took the wait as completed: all or none. */
int exx_debug_wait_warp(unsigned *went_on_h);

#ifdef __cplusplus
}
#endif
#endif
