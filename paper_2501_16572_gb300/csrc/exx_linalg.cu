// FP64 reductions and dense linear algebra of the path: exchange energy, the ACE
// matrices of Sec. III.A (M = dV Psi^T W, Cholesky factor of -sym(M), its inverse,
// xi = W L^{-T}) and the ACE application of Sec. III.B.
#include "exx_internal.h"

#include <algorithm>
#include <mutex>

namespace exx {

namespace {

// Neumaier-compensated accumulator (s, c)
struct KSum {
    double s, c;
};
__device__ __forceinline__ void kadd(KSum &k, double x)
{
    double t = k.s + x;
    if (fabs(k.s) >= fabs(x)) k.c += (k.s - t) + x;
    else k.c += (x - t) + k.s;
    k.s = t;
}
__device__ __forceinline__ void kmerge(KSum &a, const KSum &b)
{
    kadd(a, b.s);
    a.c += b.c;
}

constexpr int kRedThreads = 256;
constexpr int kRedBlocks = 512;

// E partial sums over a fixed grid: thread t of T sums (f_c dV / 4) psi_c(r) v_c(r) over
// the columns c in order and its points r = t, t + T, ... in plain FP64 (n N / T terms,
// about 10^2..10^4: relative rounding far below 1e-13); the threads' sums are merged with
// Neumaier compensation in a fixed tree, then the blocks' (reduce_partials_kernel).
__global__ void __launch_bounds__(kRedThreads)
energy_partial_kernel(const double *psi, int n, long ld, const double *f, const double *v, long ldv,
                      long N, double dV, KSum *partials)
{
    __shared__ KSum sh[kRedThreads];
    KSum acc{0.0, 0.0};
    const long T = long(gridDim.x) * blockDim.x;
    const long t0 = long(blockIdx.x) * blockDim.x + threadIdx.x;
    if (t0 < N) {
        double s = 0.0;
        for (int c = 0; c < n; ++c) {
            const double *pc = psi + long(c) * ld, *vc = v + long(c) * ldv;
            const double w = 0.25 * f[c] * dV;
            for (long r = t0; r < N; r += T) s = fma(w * pc[r], vc[r], s);
        }
        acc.s = s;
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int stride = kRedThreads / 2; stride > 0; stride >>= 1) {
        if (threadIdx.x < stride) kmerge(sh[threadIdx.x], sh[threadIdx.x + stride]);
        __syncthreads();
    }
    if (threadIdx.x == 0) partials[blockIdx.x] = sh[0];
}

// The block partials merged in a fixed tree by one block of kRedThreads threads.
__global__ void __launch_bounds__(kRedThreads) reduce_partials_kernel(const KSum *partials, int np, double *out)
{
    __shared__ KSum sh[kRedThreads];
    KSum acc{0.0, 0.0};
    for (int i = threadIdx.x; i < np; i += kRedThreads) kmerge(acc, partials[i]);
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int stride = kRedThreads / 2; stride > 0; stride >>= 1) {
        if (threadIdx.x < stride) kmerge(sh[threadIdx.x], sh[threadIdx.x + stride]);
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = sh[0].s + sh[0].c;
}

// ---- FP64 GEMMs (DFMA; GB300's FP64 rate makes these compute-bound) -----------------
constexpr int kTile = 64, kKt = 16, kGemmThreads = 256;

// C_z[i][j] = sum_{r in chunk z} A(r, i) B(r, j); A(r, i) = A[r + lda*i] (the columns of
// A and B are orbitals, r runs over the grid).  Partial tiles go to ws[z].
__global__ void __launch_bounds__(kGemmThreads)
gemm_tn_partial_kernel(int na, int nb, long K, long kchunk, const double *A, long lda,
                       const double *B, long ldb, double *ws)
{
    __shared__ double As[kKt][kTile + 1];
    __shared__ double Bs[kKt][kTile + 1];
    const int i0 = blockIdx.x * kTile, j0 = blockIdx.y * kTile;
    const long k_begin = long(blockIdx.z) * kchunk;
    const long k_end = min(K, k_begin + kchunk);
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    double acc[4][4] = {};
    for (long k0 = k_begin; k0 < k_end; k0 += kKt) {
        for (int t = threadIdx.x; t < kKt * kTile; t += kGemmThreads) {
            int kk = t % kKt, ii = t / kKt;
            long r = k0 + kk;
            As[kk][ii] = (r < k_end && i0 + ii < na) ? A[r + lda * (i0 + ii)] : 0.0;
            Bs[kk][ii] = (r < k_end && j0 + ii < nb) ? B[r + ldb * (j0 + ii)] : 0.0;
        }
        __syncthreads();
#pragma unroll 4
        for (int kk = 0; kk < kKt; ++kk) {
            double a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                a[u] = As[kk][ty + 16 * u];
                b[u] = Bs[kk][tx + 16 * u];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int w = 0; w < 4; ++w) acc[u][w] = fma(a[u], b[w], acc[u][w]);
        }
        __syncthreads();
    }
    double *wz = ws + size_t(blockIdx.z) * na * nb;
    for (int u = 0; u < 4; ++u)
        for (int w = 0; w < 4; ++w) {
            int i = i0 + ty + 16 * u, j = j0 + tx + 16 * w;
            if (i < na && j < nb) wz[i + size_t(na) * j] = acc[u][w];
        }
}

__global__ void splitk_reduce_kernel(const double *ws, int nsplit, int na, int nb, double alpha,
                                     double *C, int ldc)
{
    const long e = long(blockIdx.x) * blockDim.x + threadIdx.x;
    if (e >= long(na) * nb) return;
    int i = int(e % na), j = int(e / na);
    double s = 0.0;
    for (int z = 0; z < nsplit; ++z) s += ws[size_t(z) * na * nb + e];
    C[i + size_t(ldc) * j] = alpha * s;
}

// C(r, j) = alpha * sum_k A(r, k) Bop(k, j), A(r, k) = A[r + lda*k],
// Bop(k, j) = B[j*sbj + k*sbk];  r < M (grid rows), j < Nc, k < K.
__global__ void __launch_bounds__(kGemmThreads)
gemm_rows_kernel(long M, int Nc, int K, const double *A, long lda, const double *B, long sbj,
                 long sbk, double alpha, double *C, long ldc)
{
    __shared__ double As[kKt][kTile + 1];
    __shared__ double Bs[kKt][kTile + 1];
    const long r0 = long(blockIdx.x) * kTile;
    const int j0 = blockIdx.y * kTile;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    double acc[4][4] = {};
    for (int k0 = 0; k0 < K; k0 += kKt) {
        for (int t = threadIdx.x; t < kKt * kTile; t += kGemmThreads) {
            int rr = t % kTile, kk = t / kTile;
            As[kk][rr] = (r0 + rr < M && k0 + kk < K) ? A[(r0 + rr) + lda * (k0 + kk)] : 0.0;
            int jj = t % kTile;
            Bs[kk][jj] = (j0 + jj < Nc && k0 + kk < K) ? B[(j0 + jj) * sbj + (k0 + kk) * sbk] : 0.0;
        }
        __syncthreads();
#pragma unroll 4
        for (int kk = 0; kk < kKt; ++kk) {
            double a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                a[u] = As[kk][tx + 16 * u];
                b[u] = Bs[kk][ty + 16 * u];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int w = 0; w < 4; ++w) acc[u][w] = fma(a[u], b[w], acc[u][w]);
        }
        __syncthreads();
    }
    for (int u = 0; u < 4; ++u)
        for (int w = 0; w < 4; ++w) {
            long r = r0 + tx + 16 * u;
            int j = j0 + ty + 16 * w;
            if (r < M && j < Nc) C[r + ldc * j] = alpha * acc[u][w];
        }
}

// ---- blocked Cholesky and triangular inverse --------------------------------------------
// A = -(M + M^T)/2 is factored in place, right-looking, in column blocks of kCb = 32:
//   diagonal block: A_kk = L_kk L_kk^T and D_k = L_kk^{-1} (one warp, rows and columns in registers);
//   panel:          L_ik = A_ik D_k^T for the rows below (a CTA per kPanel rows);
//   trailing:       A_ij -= L_ik L_jk^T for i >= j > k (a CTA per lower 32 x 32 tile).
// Then X = L^{-1} by doubling: with the inverses X11, X22 of neighbouring diagonal blocks of s
// points known, X21 = -X22 (L21 X11), all pairs of a level at once.
// Everything here is a chain of small steps on the FP64 pipe (2 FMA per clock and SM: a 64 x 64 x 64 tile
// takes one SM 65 us, a 32 x 32 x 32 tile 8 us), so the tiles are small, spread over the SMs, and the
// diagonal block runs on shuffles instead of 1024 threads and three barriers a column.
// ace_build of n = 512 (72 x 72 x 144): 16.40 -> 12.09 ms against 64-wide blocks on one CTA of 1024
// threads and block rows of X in sequence.
// A failed pivot sets info_d[0] = 1 + its index; every later kernel then returns at once.
constexpr int kCb = 32, kPanel = 8, kCholThreads = 256;

__global__ void chol_prep_kernel(int n, const double *M, double *A, double *X, int *info_d)
{
    for (long e = long(blockIdx.x) * blockDim.x + threadIdx.x; e < long(n) * n; e += long(gridDim.x) * blockDim.x) {
        const int i = int(e % n), j = int(e / n);
        A[e] = (i >= j) ? -0.5 * (M[i + size_t(n) * j] + M[j + size_t(n) * i]) : 0.0;
        X[e] = 0.0;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) info_d[0] = 0;
}

// One warp: the diagonal block at (k0, k0) of size b <= NB (padded with the identity): lane i holds
// row i.  Writes L_kk into A, D = L_kk^{-1} (leading dimension kCb, zeros above) into Dk and X.
// A matrix of one block is taken straight from M: no preparation, no workspace.  NB and the
// stop at row b keep small blocks short; a FULL one (b = NB) has no stops, which would keep the
// FP64 chains of neighbouring rows from overlapping.
template <int NB, bool FULL>
__global__ void __launch_bounds__(32) chol_diag_kernel(int n, const double *M, double *A, int k0, int b, double *Dk, double *X,
                                                       int *info_d)
{
    const int lane = threadIdx.x;
    if (M) {
        if (lane == 0) info_d[0] = 0;
    } else if (info_d[0]) {
        return;
    }
    double a[NB], dg = 1.0;   // dg: L(lane, lane)
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        a[j] = j == lane ? 1.0 : 0.0;
        if (lane < b && j <= lane)
            a[j] = M ? -0.5 * (M[lane + size_t(n) * j] + M[j + size_t(n) * lane]) : A[(k0 + lane) + size_t(n) * (k0 + j)];
    }
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        if (!FULL && j >= b) break;
        const double d = __shfl_sync(0xffffffffu, a[j], j);
        if (!(d > 0.0)) {   // uniform
            if (lane == 0) info_d[0] = k0 + j + 1;
            return;
        }
        const double djj = sqrt(d);
        if (lane == j) dg = djj;
        // the quotient from the rounded reciprocal and its remainder, correctly rounded (Markstein,
        // "Computation of elementary functions on the IBM RISC System/6000 processor", 1990): the
        // division took 8 us more per block of 32 columns
        const double r = 1.0 / djj, q = a[j] * r;
        const double l = lane == j ? djj : fma(fma(-djj, q, a[j]), r, q);
        a[j] = l;
#pragma unroll
        for (int k = j + 1; k < NB; ++k) a[k] = fma(-l, __shfl_sync(0xffffffffu, l, k), a[k]);
    }
    if (!M) {
#pragma unroll
        for (int j = 0; j < NB; ++j)
            if (lane < b && j <= lane) A[(k0 + lane) + size_t(n) * (k0 + j)] = a[j];
    }
    // column `lane` of the inverse by forward substitution
    const double rdg = 1.0 / dg;
    double x[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) x[i] = 0.0;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        if (!FULL && i >= b) break;
        double s0 = i == lane ? 1.0 : 0.0, s1 = 0.0;
#pragma unroll
        for (int k = 0; k < i; ++k) {
            const double t = __shfl_sync(0xffffffffu, a[k], i);
            if (k & 1) s1 = fma(-t, x[k], s1);
            else s0 = fma(-t, x[k], s0);
        }
        x[i] = (s0 + s1) * __shfl_sync(0xffffffffu, rdg, i);
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const double v = i < b && lane < b && i >= lane ? x[i] : 0.0;
        if (Dk) Dk[i + kCb * lane] = v;
        if (i < b && lane < b) X[(k0 + i) + size_t(n) * (k0 + lane)] = v;
    }
}

// panel: rows r0 .. r0 + 7 below the diagonal block, L(r, c) = sum_t A(r, k0 + t) D(c, t)
__global__ void __launch_bounds__(kCholThreads) chol_panel_kernel(int n, double *A, int k0, int b, const double *Dk, const int *info_d)
{
    __shared__ double D[kCb][kCb + 1], R[kPanel][kCb + 1];
    if (info_d[0]) return;
    const int r0 = k0 + b + blockIdx.x * kPanel;
    for (int e = threadIdx.x; e < kCb * kCb; e += kCholThreads) D[e / kCb][e % kCb] = Dk[e];   // D[t][c]
    const int r = threadIdx.x % kPanel, c = threadIdx.x / kPanel;
    const bool ok = r0 + r < n && c < b;
    double *at = A + (r0 + r) + size_t(n) * (k0 + c);
    R[r][c] = ok ? *at : 0.0;
    __syncthreads();
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int t = 0; t < kCb; t += 2) {
        s0 = fma(R[r][t], D[t][c], s0);
        s1 = fma(R[r][t + 1], D[t + 1][c], s1);
    }
    if (ok) *at = s0 + s1;
}

// A 32 x 32 tile sum_{t < K} P(r, t) Q(t, c), 2 x 2 outputs per thread: P(r, t) = Pm[r + ldp t];
// Q(t, c) = Qm[c ldc + t ldt].  Rows and columns past rows / cols count as zero.
__device__ __forceinline__ void tile32(int rows, int cols, int K, const double *Pm, long ldp, const double *Qm, long ldc,
                                       long ldt, double (&acc)[2][2])
{
    __shared__ double Ps[kCb][kCb + 1], Qs[kCb][kCb + 1];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    for (int k0 = 0; k0 < K; k0 += kCb) {
        for (int e = threadIdx.x; e < kCb * kCb; e += kCholThreads) {
            const int i = e % kCb, j = e / kCb;
            Ps[j][i] = i < rows && k0 + j < K ? Pm[i + ldp * (k0 + j)] : 0.0;   // [t][r], r consecutive
            if (ldt == 1) Qs[i][j] = j < cols && k0 + i < K ? Qm[j * ldc + k0 + i] : 0.0;
            else Qs[j][i] = i < cols && k0 + j < K ? Qm[i * ldc + (k0 + j) * ldt] : 0.0;
        }
        __syncthreads();
#pragma unroll 8
        for (int t = 0; t < kCb; ++t) {
            const double p0 = Ps[t][tx], p1 = Ps[t][tx + 16], q0 = Qs[t][ty], q1 = Qs[t][ty + 16];
            acc[0][0] = fma(p0, q0, acc[0][0]);
            acc[0][1] = fma(p0, q1, acc[0][1]);
            acc[1][0] = fma(p1, q0, acc[1][0]);
            acc[1][1] = fma(p1, q1, acc[1][1]);
        }
        __syncthreads();
    }
}

// trailing update of the lower triangle: tile (bi, bj), bi >= bj, of the part past k0 + b (the strict
// upper part of a diagonal tile is updated too; it is never read)
__global__ void __launch_bounds__(kCholThreads) chol_update_kernel(int n, double *A, int k0, int b, const int *info_d)
{
    const int bi = blockIdx.x, bj = blockIdx.y;
    if (info_d[0] || bi < bj) return;
    const int r0 = k0 + b + bi * kCb, c0 = k0 + b + bj * kCb;
    const int rows = min(kCb, n - r0), cols = min(kCb, n - c0);
    double acc[2][2] = {};
    tile32(rows, cols, b, A + r0 + size_t(n) * k0, n, A + c0 + size_t(n) * k0, 1, n, acc);
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int w = 0; w < 2; ++w) {
            const int r = tx + 16 * u, c = ty + 16 * w;
            if (r < rows && c < cols) A[(r0 + r) + size_t(n) * (c0 + c)] -= acc[u][w];
        }
}

// Doubling level s: pair blockIdx.z, tile (blockIdx.x, blockIdx.y) of the block below X11.
// step 0: T = L21 X11 (X11 lower: t >= c); step 1: X21 = -X22 T (X22 lower: t <= r).
__global__ void __launch_bounds__(kCholThreads) chol_double_kernel(int n, int s, int step, const double *L, double *X, double *T,
                                                                   const int *info_d)
{
    if (info_d[0]) return;
    const int base = blockIdx.z * 2 * s, r0 = base + s + blockIdx.x * kCb, c0 = base + blockIdx.y * kCb;
    if (r0 >= n) return;
    const int rows = min(kCb, min(n, base + 2 * s) - r0), cols = kCb;   // columns lie in a whole block
    double acc[2][2] = {};
    double *out;
    if (step == 0) {
        tile32(rows, cols, base + s - c0, L + r0 + size_t(n) * c0, n, X + c0 + size_t(n) * c0, n, 1, acc);
        out = T;
    } else {
        const int t0 = base + s;
        tile32(rows, cols, r0 + rows - t0, X + r0 + size_t(n) * t0, n, T + t0 + size_t(n) * c0, n, 1, acc);
        out = X;
    }
    const double sg = step ? -1.0 : 1.0;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int w = 0; w < 2; ++w) {
            const int r = tx + 16 * u, c = ty + 16 * w;
            if (r < rows && c < cols) out[(r0 + r) + size_t(n) * (c0 + c)] = sg * acc[u][w];
        }
}

}  // namespace

int energy_fp64(Plan &P, const double *psi, int n, long ld, const double *f, const double *v, long ld_v,
                double *E_h, cudaStream_t s)
{
    size_t need = kRedBlocks * sizeof(KSum) + 64;
    if (int rc = dev_reserve(P.red_ws, need)) return rc;
    KSum *parts = static_cast<KSum *>(P.red_ws.p);
    double *res = reinterpret_cast<double *>(static_cast<char *>(P.red_ws.p) + kRedBlocks * sizeof(KSum));
    int tb = timing_begin(P, EXX_TIMING_ENERGY, s);
    energy_partial_kernel<<<kRedBlocks, kRedThreads, 0, s>>>(psi, n, ld, f, v, ld_v, P.N, P.dV, parts);
    EXX_LAUNCH("energy_partial_kernel");
    reduce_partials_kernel<<<1, kRedThreads, 0, s>>>(parts, kRedBlocks, res);
    timing_end(P, tb, s);
    EXX_LAUNCH("reduce_partials_kernel");
    P.launches += 2;
    EXX_CUDA(cudaMemcpyAsync(E_h, res, sizeof(double), cudaMemcpyDeviceToHost, s));
    EXX_CUDA(cudaStreamSynchronize(s));
    return EXX_OK;
}

int gemm_fp64_tn_splitk(Plan &P, int na, int nb, int K, const double *A, long lda, const double *B,
                        long ldb, double alpha, double *C, int ldc, cudaStream_t s)
{
    const int gx = (na + kTile - 1) / kTile, gy = (nb + kTile - 1) / kTile;
    // enough CTAs to fill the GPU twice over, each with a K chunk of at least 256
    int nsplit = std::max(1, (2 * P.num_sms + gx * gy - 1) / (gx * gy));
    long kchunk = (long(K) + nsplit - 1) / nsplit;
    kchunk = ((kchunk + kKt - 1) / kKt) * kKt;
    if (kchunk < 256) kchunk = 256;
    nsplit = int((long(K) + kchunk - 1) / kchunk);
    if (int rc = dev_reserve(P.gemm_ws, size_t(nsplit) * na * nb * sizeof(double))) return rc;
    double *ws = static_cast<double *>(P.gemm_ws.p);
    int tb = timing_begin(P, EXX_TIMING_GEMM, s);
    gemm_tn_partial_kernel<<<dim3(gx, gy, nsplit), kGemmThreads, 0, s>>>(na, nb, K, kchunk, A, lda, B,
                                                                         ldb, ws);
    EXX_LAUNCH("gemm_tn_partial_kernel");
    long tot = long(na) * nb;
    splitk_reduce_kernel<<<unsigned((tot + 255) / 256), 256, 0, s>>>(ws, nsplit, na, nb, alpha, C, ldc);
    timing_end(P, tb, s);
    EXX_LAUNCH("splitk_reduce_kernel");
    P.launches += 2;
    return EXX_OK;
}

int gemm_fp64_nt(Plan &P, int M, int Nc, int K, const double *A, long lda, const double *B, long ldb,
                 double alpha, double *C, long ldc, cudaStream_t s)
{
    // Bop(k, j) = B(j, k) = B[j + ldb*k]
    dim3 grid(unsigned((long(M) + kTile - 1) / kTile), unsigned((Nc + kTile - 1) / kTile));
    int tb = timing_begin(P, EXX_TIMING_GEMM, s);
    gemm_rows_kernel<<<grid, kGemmThreads, 0, s>>>(M, Nc, K, A, lda, B, 1, ldb, alpha, C, ldc);
    timing_end(P, tb, s);
    EXX_LAUNCH("gemm_rows_kernel");
    P.launches++;
    return EXX_OK;
}

int gemm_fp64_nn(Plan &P, int M, int Nc, int K, const double *A, long lda, const double *B, long ldb,
                 double alpha, double *C, long ldc, cudaStream_t s)
{
    // Bop(k, j) = B(k, j) = B[k + ldb*j]
    dim3 grid(unsigned((long(M) + kTile - 1) / kTile), unsigned((Nc + kTile - 1) / kTile));
    int tb = timing_begin(P, EXX_TIMING_GEMM, s);
    gemm_rows_kernel<<<grid, kGemmThreads, 0, s>>>(M, Nc, K, A, lda, B, ldb, 1, alpha, C, ldc);
    timing_end(P, tb, s);
    EXX_LAUNCH("gemm_rows_kernel");
    P.launches++;
    return EXX_OK;
}

int cholesky_neg_sym_and_inverse(Plan &P, int n, const double *M, double *Linv, int *info_d,
                                 cudaStream_t s)
{
    int tb = timing_begin(P, EXX_TIMING_CHOL, s);
    auto diag = [&](const double *m, double *A, int k0, int b, double *Dk) -> int {
        auto kern = b == 8    ? chol_diag_kernel<8, true>
                    : b < 8   ? chol_diag_kernel<8, false>
                    : b == 16 ? chol_diag_kernel<16, true>
                    : b < 16  ? chol_diag_kernel<16, false>
                    : b < kCb ? chol_diag_kernel<kCb, false>
                              : chol_diag_kernel<kCb, true>;
        kern<<<1, 32, 0, s>>>(n, m, A, k0, b, b == kCb ? Dk : nullptr, Linv, info_d);   // a last, shorter block has no panel
        EXX_LAUNCH("chol_diag_kernel");
        P.launches++;
        return EXX_OK;
    };
    if (n <= kCb) {
        const int rc = diag(M, nullptr, 0, n, nullptr);
        timing_end(P, tb, s);
        return rc;
    }
    // workspace: A (n x n), the products of the doubling (n x n), one diagonal-block inverse
    const size_t nn = size_t(n) * n;
    if (int rc = dev_reserve(P.small_ws, (2 * nn + kCb * kCb) * sizeof(double))) return rc;
    double *A = static_cast<double *>(P.small_ws.p);
    double *T = A + nn, *Dk = T + nn;
    const int eg = std::min(4 * P.num_sms, int((nn + 255) / 256));
    chol_prep_kernel<<<eg, 256, 0, s>>>(n, M, A, Linv, info_d);
    EXX_LAUNCH("chol_prep_kernel");
    P.launches++;
    for (int k0 = 0; k0 < n; k0 += kCb) {
        const int b = std::min(kCb, n - k0), rest = n - k0 - b;
        if (int rc = diag(nullptr, A, k0, b, Dk)) return rc;
        if (rest == 0) break;
        chol_panel_kernel<<<(rest + kPanel - 1) / kPanel, kCholThreads, 0, s>>>(n, A, k0, b, Dk, info_d);
        EXX_LAUNCH("chol_panel_kernel");
        const unsigned nt = unsigned((rest + kCb - 1) / kCb);
        chol_update_kernel<<<dim3(nt, nt), kCholThreads, 0, s>>>(n, A, k0, b, info_d);
        EXX_LAUNCH("chol_update_kernel");
        P.launches += 2;
    }
    for (int sz = kCb; sz < n; sz *= 2) {
        const dim3 grid(unsigned(sz / kCb), unsigned(sz / kCb), unsigned((n - sz + 2 * sz - 1) / (2 * sz)));
        for (int step = 0; step < 2; ++step) {
            chol_double_kernel<<<grid, kCholThreads, 0, s>>>(n, sz, step, A, Linv, T, info_d);
            EXX_LAUNCH("chol_double_kernel");
            P.launches++;
        }
    }
    timing_end(P, tb, s);
    return EXX_OK;
}

// ---------------------------------------------------------------------------------------
// Allocation-free Gram matrix M = dV Psi^T W (exx_gram_noalloc in include/exx.h).
//
// Same split-K kernels as the ACE matrix above, but the partial tiles live in a fixed
// device array that is part of the loaded library, so the call needs no cudaMalloc and
// no plan.  It exists for callers that must not allocate device memory at the point of
// the call: callers whose device memory is owned by a pool or framework allocator that
// this library cannot use, memory-capped processes that reserve everything up front, and
// loops that must not stall (cudaMalloc and cudaFree can synchronize the whole device).
namespace {

constexpr int kGramNoAllocMaxN = 128;      // largest n accepted
constexpr int kGramNoAllocMaxSplit = 8;    // K chunks (partial tiles per entry)

// One copy per GPU that loads the library (1 MiB), held until the process exits.  Host
// code must not pass this name to a kernel: on the host it is only a stand-in symbol.
static __device__ __align__(256) double g_gram_partials[kGramNoAllocMaxSplit * kGramNoAllocMaxN * kGramNoAllocMaxN];

constexpr int kMaxDevices = 64;
std::mutex g_gram_mutex;
double *g_gram_addr[kMaxDevices] = {};     // device address of g_gram_partials, per device

// Device address of the scratch array on the current device (looked up once per device).
int gram_scratch(double **out)
{
    int dev = 0;
    EXX_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) {
        set_error("exx_gram_noalloc: device ordinal out of range");
        return EXX_ERR_UNSUPPORTED;
    }
    std::lock_guard<std::mutex> lock(g_gram_mutex);
    if (!g_gram_addr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_gram_partials);
        if (e != cudaSuccess) return cuda_fail(e, "exx_gram_noalloc: cudaGetSymbolAddress");
        g_gram_addr[dev] = static_cast<double *>(p);
    }
    *out = g_gram_addr[dev];
    return EXX_OK;
}

}  // namespace
}  // namespace exx

extern "C" int exx_gram_noalloc(int N, double dV, const double *Psi, int n, long ld, const double *W, long ld_w,
                                double *M, exx_stream_t stream)
{
    using namespace exx;
    if (!Psi || !W || !M) {
        set_error("exx_gram_noalloc: NULL array");
        return EXX_ERR_INVALID_ARG;
    }
    if (N < 1 || ld < N || ld_w < N) {
        set_error("exx_gram_noalloc: need N >= 1 and leading dimensions >= N");
        return EXX_ERR_INVALID_ARG;
    }
    if (n < 1 || n > kGramNoAllocMaxN) {
        set_error("exx_gram_noalloc: n must be in [1, 128] (the fixed scratch holds 8 partial 128 x 128 tiles)");
        return EXX_ERR_INVALID_ARG;
    }
    double *ws = nullptr;
    if (int rc = gram_scratch(&ws)) return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int g = (n + kTile - 1) / kTile;
    long kchunk = (long(N) + kGramNoAllocMaxSplit - 1) / kGramNoAllocMaxSplit;
    kchunk = std::max<long>(256, ((kchunk + kKt - 1) / kKt) * kKt);
    const int nsplit = int((long(N) + kchunk - 1) / kchunk);   // <= kGramNoAllocMaxSplit
    // every partial tile entry (z, i < n, j < n) is rewritten below, so nothing from an
    // earlier call survives into this one and no clearing is needed
    gemm_tn_partial_kernel<<<dim3(g, g, nsplit), kGemmThreads, 0, s>>>(n, n, N, kchunk, Psi, ld, W, ld_w, ws);
    EXX_LAUNCH("gemm_tn_partial_kernel (no-alloc)");
    const long tot = long(n) * n;
    splitk_reduce_kernel<<<unsigned((tot + 255) / 256), 256, 0, s>>>(ws, nsplit, n, n, dV, M, n);
    EXX_LAUNCH("splitk_reduce_kernel (no-alloc)");
    return EXX_OK;
}
