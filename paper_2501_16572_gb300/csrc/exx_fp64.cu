// FP64 path of the batched Kronecker Poisson solve (Sec. II.B) and of the
// exchange accumulation (Eq. 1), on the CUDA cores.
//
// GB300 runs FP64 at a small fraction of its FP32 rate (2 FMA per clock and SM), so these
// kernels are bound by the double-precision FMA pipe, not by memory.  Every 1D operator commutes
// with the reflection of its axis (Toeplitz or circulant, and symmetric), so its eigenvectors are
// taken even or odd: a forward contraction works on x_k + x_{n-1-k} for the even outputs and on
// x_k - x_{n-1-k} for the odd ones, an inverse one gives y_k and y_{n-1-k} as the sum and the
// difference of an even and an odd part: n flops a point instead of 2n.  Each thread owns one row (a
// pencil along the contracted axis) and produces up to 20 outputs at a time from the slice of
// the matrix staged in shared memory (every thread of a warp reads the same entry, a
// broadcast); the slice width is the one that pads the axis least.
// 28 x 30 x 33 points, 24 of 32 orbitals: 6.05 ms without the reflection and with slices of 16, 2.97 with both.
#include "exx_internal.h"

#include <algorithm>
#include <cmath>
#include <numeric>

namespace exx {

namespace {

constexpr int kThreads = 256;

struct Fp64PassArgs {
    int nfields, R, K;
    const double *in;            // field stride N
    double *out;                 // field stride N
    long N;
    const double *B;             // ne x K: B[k*K + j], modes j even (ne of them) then odd
    const double *F;             // [j][r] scaling (R*K values) or null
    const double *psi_a, *psi_b; // pair prologue: psi_a[m*lda + ...], psi_b[n*ldb + ...]
    long lda, ldb;
    const int2 *pairs;
};

// Forward: C modes of one parity per sweep over the row.  Inverse: C / 2 point pairs per sweep.
template <int LOAD, int STORE, bool SCALE, bool INV, int C>
__global__ void __launch_bounds__(kThreads) fp64_pass_kernel(Fp64PassArgs a)
{
    extern __shared__ double Bs[];   // [k][C]
    const int K = a.K, no = K / 2, ne = K - no;
    const long rows = long(a.nfields) * a.R;
    const long g = long(blockIdx.x) * blockDim.x + threadIdx.x;
    const bool active = g < rows;
    const int p = active ? int(g / a.R) : 0;
    const int r = active ? int(g - long(p) * a.R) : 0;
    const double *in = a.in + size_t(p) * a.N;
    const double *pa = nullptr, *pb = nullptr;
    if (LOAD == LOAD_PAIR && active) {
        int2 mn = a.pairs[p];
        pa = a.psi_a + size_t(mn.x) * a.lda;
        pb = a.psi_b + size_t(mn.y) * a.ldb;
    }
    double *out = a.out + size_t(p) * a.N;
    auto load = [&](int k) {
        if (LOAD == LOAD_PAIR) return pa[size_t(k) * a.R + r] * pb[size_t(k) * a.R + r];
        if (LOAD == LOAD_KSLOW) return in[size_t(k) * a.R + r];
        return in[size_t(r) * a.K + k];
    };
    auto store = [&](int j, double v) {
        if (SCALE) v *= a.F[size_t(j) * a.R + r];
        if (STORE == STORE_NSLOW) out[size_t(j) * a.R + r] = v;
        else out[size_t(r) * a.K + j] = v;
    };
    if (!INV) {
        for (int par = 0; par < 2; ++par) {
            const int first = par ? ne : 0, cnt = par ? no : ne;   // modes of this parity
            for (int j0 = 0; j0 < cnt; j0 += C) {
                __syncthreads();
                for (int i = threadIdx.x; i < ne * C; i += blockDim.x) {
                    const int k = i / C, j = i - k * C;
                    Bs[i] = j0 + j < cnt ? a.B[size_t(k) * K + first + j0 + j] : 0.0;
                }
                __syncthreads();
                if (!active) continue;
                double acc[C];
#pragma unroll
                for (int j = 0; j < C; ++j) acc[j] = 0.0;
                for (int k = 0; k < ne; ++k) {   // k = no < ne: the middle point of an odd axis (even modes only)
                    double x = load(k);
                    if (k < no) x += par ? -load(K - 1 - k) : load(K - 1 - k);
                    const double2 *bk = reinterpret_cast<const double2 *>(Bs + k * C);
#pragma unroll
                    for (int j = 0; j < C / 2; ++j) {
                        const double2 b = bk[j];
                        acc[2 * j] = fma(x, b.x, acc[2 * j]);
                        acc[2 * j + 1] = fma(x, b.y, acc[2 * j + 1]);
                    }
                }
#pragma unroll
                for (int j = 0; j < C; ++j)
                    if (j0 + j < cnt) store(first + j0 + j, acc[j]);
            }
        }
    } else {
        constexpr int H = C / 2;
        for (int k0 = 0; k0 < ne; k0 += H) {
            __syncthreads();
            for (int i = threadIdx.x; i < K * H; i += blockDim.x) {
                const int j = i / H, k = k0 + i - j * H;
                Bs[i] = k < ne ? a.B[size_t(k) * K + j] : 0.0;
            }
            __syncthreads();
            if (!active) continue;
            double ev[H], od[H];
#pragma unroll
            for (int k = 0; k < H; ++k) ev[k] = od[k] = 0.0;
            for (int j = 0; j < ne; ++j) {
                const double t = load(j);
#pragma unroll
                for (int k = 0; k < H; ++k) ev[k] = fma(t, Bs[j * H + k], ev[k]);
            }
            for (int j = ne; j < K; ++j) {
                const double t = load(j);
#pragma unroll
                for (int k = 0; k < H; ++k) od[k] = fma(t, Bs[j * H + k], od[k]);
            }
#pragma unroll
            for (int k = 0; k < H; ++k) {
                if (k0 + k >= ne) break;
                store(k0 + k, ev[k] + od[k]);                            // od = 0 at the middle point
                if (k0 + k < no) store(K - 1 - k0 - k, ev[k] - od[k]);
            }
        }
    }
}

// The slice width that pads `count` modes (or point pairs, half a width each) least, the widest of equals.
inline int slice_width(int count, bool inv)
{
    int best = 0, cost = 1 << 30;
    for (int c : {20, 18, 16, 14, 12}) {
        const int w = inv ? c / 2 : c;
        const int padded = (count + w - 1) / w * w;
        if (padded < cost) {
            cost = padded;
            best = c;
        }
    }
    return best;
}

template <int LOAD, int STORE, bool SCALE, bool INV>
int launch_pass(Plan &P, int kind, const Fp64PassArgs &a, cudaStream_t s)
{
    const long rows = long(a.nfields) * a.R;
    const int grid = int((rows + kThreads - 1) / kThreads);
    const int ne = a.K - a.K / 2, C = slice_width(ne, INV);
    const size_t smem = size_t(INV ? a.K * (C / 2) : ne * C) * sizeof(double);   // at most 20.5 KB
    auto kern = C == 20   ? fp64_pass_kernel<LOAD, STORE, SCALE, INV, 20>
                : C == 18 ? fp64_pass_kernel<LOAD, STORE, SCALE, INV, 18>
                : C == 16 ? fp64_pass_kernel<LOAD, STORE, SCALE, INV, 16>
                : C == 14 ? fp64_pass_kernel<LOAD, STORE, SCALE, INV, 14>
                          : fp64_pass_kernel<LOAD, STORE, SCALE, INV, 12>;
    int tb = timing_begin(P, kind, s);
    kern<<<grid, kThreads, smem, s>>>(a);
    timing_end(P, tb, s);
    EXX_LAUNCH("fp64_pass_kernel");
    return EXX_OK;
}

// out_t(r) += - sum over the block's contributions f_s psi_s(r) V_field(r), FP64.
struct Fp64AccArgs {
    long N;
    const double *psi_a, *psi_b;  // occupied (sources) / input orbitals
    long lda, ldb;
    const double *f;
    const Block *blocks;
    const double *V;              // fields of the batch
    double *out;
    long ldo;
};

__device__ __forceinline__ int diag_index(int i, int j, int nI)
{
    // index of (i <= j) in the row-major upper-triangle enumeration of an nI x nI block
    return i * nI - (i * (i - 1)) / 2 + (j - i);
}

__global__ void __launch_bounds__(kThreads) fp64_accum_kernel(Fp64AccArgs a)
{
    const Block b = a.blocks[blockIdx.y];
    const long r = long(blockIdx.x) * blockDim.x + threadIdx.x;
    if (r >= a.N) return;
    const double *V = a.V + size_t(b.field0) * a.N + r;
    if (b.kind == BLK_SYM_DIAG) {
        for (int t = 0; t < b.nI; ++t) {
            double acc = 0.0;
            for (int s = 0; s < b.nI; ++s) {
                int m = b.I0 + s;
                int fi = s <= t ? diag_index(s, t, b.nI) : diag_index(t, s, b.nI);
                acc = fma(-a.f[m] * a.psi_a[size_t(m) * a.lda + r], V[size_t(fi) * a.N], acc);
            }
            double *o = a.out + size_t(b.I0 + t) * a.ldo + r;
            *o += acc;
        }
        return;
    }
    // outputs of J (both kinds): sources m in I
    for (int j = 0; j < b.nJ; ++j) {
        double acc = 0.0;
        for (int i = 0; i < b.nI; ++i) {
            int m = b.I0 + i;
            acc = fma(-a.f[m] * a.psi_a[size_t(m) * a.lda + r], V[size_t(i * b.nJ + j) * a.N], acc);
        }
        double *o = a.out + size_t(b.J0 + j) * a.ldo + r;
        *o += acc;
    }
    if (b.kind == BLK_SYM_OFF) {
        // outputs of I: sources n in J (J occupied as well, same array)
        for (int i = 0; i < b.nI; ++i) {
            double acc = 0.0;
            for (int j = 0; j < b.nJ; ++j) {
                int n = b.J0 + j;
                acc = fma(-a.f[n] * a.psi_a[size_t(n) * a.lda + r], V[size_t(i * b.nJ + j) * a.N], acc);
            }
            double *o = a.out + size_t(b.I0 + i) * a.ldo + r;
            *o += acc;
        }
    }
}

}  // namespace

int fp64_solve_batch(Plan &P, const double *psi_occ, long ld_occ, const double *psi_in, long ld_in,
                     const int2 *pairs_d, int nfields, double *bufA, double *bufB, double **result,
                     cudaStream_t s)
{
    double *src = nullptr, *dst = bufA;
    for (int pass = 0; pass < 5; ++pass) {
        PassGeom g = pass_geom(P.n, pass);
        Fp64PassArgs a{};
        a.nfields = nfields;
        a.R = g.R;
        a.K = g.K;
        a.N = P.N;
        a.psi_a = psi_occ;
        a.psi_b = psi_in;
        a.lda = ld_occ;
        a.ldb = ld_in;
        a.pairs = pairs_d;
        int rc = EXX_OK;
        if (pass == 2) {
            // forward y with the Hadamard scaling by f(Lambda), then inverse y
            a.in = src;
            a.out = dst;
            a.B = static_cast<const double *>(P.B64[1].p);
            a.F = static_cast<const double *>(P.F64.p);
            rc = launch_pass<LOAD_KFAST, STORE_NFAST, true, false>(P, EXX_TIMING_PASS3, a, s);
            if (rc) return rc;
            P.launches++;
            std::swap(src, dst);
            a.in = src;
            a.out = dst;
            a.B = static_cast<const double *>(P.B64[1].p);
            a.F = nullptr;
            rc = launch_pass<LOAD_KFAST, STORE_NFAST, false, true>(P, EXX_TIMING_PASS3, a, s);
        } else {
            a.in = src;
            a.out = dst;
            a.B = static_cast<const double *>(P.B64[g.axis].p);
            if (pass == 0) rc = launch_pass<LOAD_PAIR, STORE_NSLOW, false, false>(P, EXX_TIMING_PASS1, a, s);
            else if (pass == 1) rc = launch_pass<LOAD_KFAST, STORE_NSLOW, false, false>(P, EXX_TIMING_PASS2, a, s);
            else if (pass == 3) rc = launch_pass<LOAD_KSLOW, STORE_NFAST, false, true>(P, EXX_TIMING_PASS4, a, s);
            else rc = launch_pass<LOAD_KSLOW, STORE_NSLOW, false, true>(P, EXX_TIMING_PASS5, a, s);
        }
        if (rc) return rc;
        P.launches++;
        src = dst;
        dst = (dst == bufA) ? bufB : bufA;
    }
    *result = src;   // the solutions, natural layout
    return EXX_OK;
}

int fp64_accumulate(Plan &P, const double *psi_occ, long ld_occ, const double *psi_in, long ld_in,
                    const double *f, const Block *blocks_d, int nblocks, const double *V, double *out,
                    long ld_out, cudaStream_t s)
{
    Fp64AccArgs a{};
    a.N = P.N;
    a.psi_a = psi_occ;
    a.psi_b = psi_in;
    a.lda = ld_occ;
    a.ldb = ld_in;
    a.f = f;
    a.blocks = blocks_d;
    a.V = V;
    a.out = out;
    a.ldo = ld_out;
    dim3 grid(unsigned((P.N + kThreads - 1) / kThreads), unsigned(nblocks));
    int tb = timing_begin(P, EXX_TIMING_ACCUM, s);
    fp64_accum_kernel<<<grid, kThreads, 0, s>>>(a);
    timing_end(P, tb, s);
    EXX_LAUNCH("fp64_accum_kernel");
    P.launches++;
    return EXX_OK;
}

// Even and odd eigenvectors of one axis, ne x n: B[k n + j] is mode j (the ne even ones, then the
// odd ones) at point k, over sqrt(2) except at the middle point of an odd axis; order[j] = the mode's
// place among the ascending eigenvalues.
static int fold_axis(const Plan &P, int d, std::vector<double> &B, std::vector<int> &order)
{
    const int n = P.n[d], no = n / 2, ne = n - no;
    std::vector<double> D(size_t(n) * n), lam(n);
    second_derivative(n, P.h, P.bc[d], P.fd_order / 2, D.data());
    B.assign(size_t(ne) * n, 0.0);
    const double r2 = std::sqrt(0.5);
    for (int par = 0; par < 2; ++par) {
        const int m = par ? no : ne, first = par ? ne : 0;
        if (m == 0) continue;
        std::vector<double> A(size_t(m) * m), U(size_t(m) * m);
        for (int l = 0; l < m; ++l)
            for (int k = 0; k < m; ++k) {
                const bool mk = k == no, ml = l == no;   // the middle point is its own mirror image
                const double direct = D[size_t(k) + size_t(n) * l];
                const double mirror = D[size_t(k) + size_t(n) * (n - 1 - l)];
                A[size_t(k) + size_t(m) * l] = mk && ml ? direct : (mk || ml) ? direct / r2 : par ? direct - mirror : direct + mirror;
            }
        if (sym_eig(m, A.data(), U.data(), lam.data() + first)) {
            set_error("exx_plan_create: eigen-decomposition did not converge");
            return EXX_ERR_UNSUPPORTED;
        }
        for (int j = 0; j < m; ++j)
            for (int k = 0; k < m; ++k) B[size_t(k) * n + first + j] = U[size_t(k) + size_t(m) * j] * (k == no ? 1.0 : r2);
    }
    std::vector<int> rank(n);
    std::iota(rank.begin(), rank.end(), 0);
    std::stable_sort(rank.begin(), rank.end(), [&](int x, int y) { return lam[x] < lam[y]; });
    order.resize(n);
    for (int i = 0; i < n; ++i) order[rank[i]] = i;
    return EXX_OK;
}

int fp64_upload(Plan &P)
{
    std::vector<int> order[3];
    for (int d = 0; d < 3; ++d) {
        std::vector<double> B;
        if (int rc = fold_axis(P, d, B, order[d])) return rc;
        if (int rc = dev_reserve(P.B64[d], B.size() * sizeof(double))) return rc;
        EXX_CUDA(cudaMemcpy(P.B64[d].p, B.data(), B.size() * sizeof(double), cudaMemcpyHostToDevice));
    }
    // F in the P3 layout: [b][a][c] -> F(a, b, c); FP64 in the folded order of the modes, the
    // FP32 planes (hi, then lo) of the five-pass split modes in ascending order
    const int n1 = P.n[0], n2 = P.n[1], n3 = P.n[2];
    std::vector<double> F3(size_t(P.N));
    std::vector<float> F3f(2 * size_t(P.N));
    for (int b = 0; b < n2; ++b)
        for (int a = 0; a < n1; ++a)
            for (int c = 0; c < n3; ++c) {
                size_t idx = size_t(b) * n1 * n3 + size_t(a) * n3 + c;
                F3[idx] = P.F[order[0][a] + size_t(n1) * (order[1][b] + size_t(n2) * order[2][c])];
                const double v = P.F[a + size_t(n1) * (b + size_t(n2) * c)];
                F3f[idx] = float(v);
                F3f[idx + size_t(P.N)] = float(v - double(float(v)));
            }
    if (int rc = dev_reserve(P.F64, F3.size() * sizeof(double))) return rc;
    EXX_CUDA(cudaMemcpy(P.F64.p, F3.data(), F3.size() * sizeof(double), cudaMemcpyHostToDevice));
    if (int rc = dev_reserve(P.F32, F3f.size() * sizeof(float))) return rc;
    EXX_CUDA(cudaMemcpy(P.F32.p, F3f.data(), F3f.size() * sizeof(float), cudaMemcpyHostToDevice));
    return EXX_OK;
}

}  // namespace exx
