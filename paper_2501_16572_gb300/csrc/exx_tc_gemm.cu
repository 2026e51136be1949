// Fixed-point split GEMM on the tcgen05 tensor cores for the ACE products of Sec. III
// (M = dV Psi^T W and xi = W L^{-T} in the construction, chi = xi^T Phi and -dV xi chi in
// the application), used by plans in a split-precision mode:
//
//     D(i, j) = alpha * sum_k A(i, k) B(j, k)
//
// with FP64 operands addressed through element strides, A(i, k) = A[i as_i + k as_k].
//
// Every 320-long chunk of k is exact up to the operand digits: within the chunk each row
// of A and each row of B gets a power-of-two scale from its largest entry, the scaled
// row is rounded to a 31-bit integer X and cut into four balanced base-256 digits,
//     X = d0 2^24 + d1 2^16 + d2 2^8 + d3,   |d0| <= 64, |d1|, |d2|, |d3| <= 128,
// each stored exactly as a bf16.  Digit products of one level (i + j = l, l <= 4) are
// summed in their own TMEM accumulator (5 levels x up to 48 output columns per tile, two sets of them); a level
// gains at most 3 * 2^14 per k, so the 320-term sums stay integers below 2^24 and the
// tensor core never rounds.  The levels of a chunk are combined into an FP32 hi + lo pair, and
// the chunks are summed in FP64.  Dropped digit products (i + j >= 5) weigh below 2^-37 of the
// row maxima; the rounding of X, 2^-31 of the row maxima, is the leading error.
//
// Two kernels.  gemm_cut_kernel cuts every operand element once into digit planes in device
// memory, already in the operand layout of the MMA, and records the row scales;
// tc_gemm_kernel then only streams 8-byte-per-element blocks of them through shared memory
// (bulk copies, a producer warp) into the MMAs (one issuing warp) while 8 or 12 warps combine
// finished chunks.  Cutting inside the GEMM repeated the integer work of every A row for each
// column tile and left the tensor cores idle meanwhile: both products of ace_apply at
// n = nphi = 512 on 72 x 72 x 144 points took 65.7 ms, 9.7 ms now (cuts 3.3 ms near the HBM
// rate, the GEMMs 6.4 ms, of which the tensor pipe's own 4.2).
#include "exx_internal.h"
#include "tc_ptx.cuh"

#include <algorithm>
#include <cmath>

namespace exx {

namespace {

constexpr int kT = 128;              // rows of A per tile (TMEM lanes)
constexpr int kTN = 48;              // most rows of B per tile (output columns): two sets of levels fill TMEM
constexpr int kLev = 5;              // level accumulators: digit products with i + j <= 4
constexpr int kDig = 4;
constexpr int kBlk = 32;             // k per operand block
constexpr int kBlks = 10;            // blocks per exact chunk
constexpr int kChunk = kBlk * kBlks; // 320: 4 levels x 320 x 3 * 2^14 < 2^24
constexpr uint64_t kGemmWaitNs = 1000000000ull;
constexpr uint32_t kSbo = kBlk * 16;           // bytes between 8-row groups of a digit plane
constexpr int kParts = 3;            // drain warps per 32 TMEM lanes (2 for tiles of up to 32 columns)
constexpr int kNarrow = 32;          // tiles of up to 32 columns: one set of levels, two CTAs per SM
constexpr int kCutWarps = kBlks;     // gemm_cut_kernel: a warp per k block of a chunk

__device__ __forceinline__ int exp_field(uint32_t hi) { return int((hi >> 20) & 0x7ffu); }

// Byte offset of (row, 8-k group c) in the digit planes of an operand whose tiles have `rt`
// rows: tile (row / rt), block kb of `nkb`, digit plane q, then the canonical K-major
// no-swizzle image (8 rows x 16 bytes per core matrix).
__device__ __forceinline__ size_t cut_off(long tile, int r, int rt, long kb, long nkb, int c)
{
    return (size_t(tile) * nkb + kb) * (size_t(rt) * kBlk * 2 * kDig) + size_t(r >> 3) * kSbo + size_t(c) * 128 +
           size_t(r & 7) * 16;
}

// Digits of eight consecutive k of one row (largest biased exponent E in its chunk), stored as
// 16 bytes in each of the four planes.  |x| < 2^(E-1022), X = x 2^(1052-E) rounded to even,
// |X| <= 2^30: the 53-bit mantissa, 64-bit aligned, shifted right by 2 + E - e (zeros and
// subnormals give X = 0), on the integer pipe: the FP64 unit converts two values per clock and
// SM.  Digit l is X rounded to a multiple of 2^(24 - 8 l) less the same rounding one digit up.
__device__ __forceinline__ void cut8(uint8_t *dst, size_t plane, const double (&x)[8], int E)
{
    uint32_t w[kDig][4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        float d[2][kDig];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const double v = x[2 * p + h];
            const uint32_t hi = uint32_t(__double2hiint(v)), lo = uint32_t(__double2loint(v));
            const int e = exp_field(hi);
            const uint32_t top = e ? (0x80000000u | (hi << 11) | (lo >> 21)) : 0u;
            const int s = 2 + E - e;                      // >= 2
            const uint32_t low = lo << 11;
            uint32_t q = s < 32 ? top >> s : 0u;
            const uint32_t fr = s <= 32 ? __funnelshift_rc(low, top, s) : 0u;   // the fraction below q
            const uint32_t rest = (fr << 1) | low;
            q += (fr >> 31) & ((q & 1u) | (rest != 0u ? 1u : 0u));
            const int sg = int(hi) >> 31;
            const int X = (int(q) ^ sg) - sg;
            const int R0 = (X + (1 << 23)) >> 24, R1 = (X + (1 << 15)) >> 16, R2 = (X + (1 << 7)) >> 8;
            // small integers to FP32 through the 1.5 * 2^23 offset
            d[h][0] = __int_as_float(0x4B400000 + R0) - 12582912.f;
            d[h][1] = __int_as_float(0x4B400000 + R1 - R0 * 256) - 12582912.f;
            d[h][2] = __int_as_float(0x4B400000 + R2 - R1 * 256) - 12582912.f;
            d[h][3] = __int_as_float(0x4B400000 + X - R2 * 256) - 12582912.f;
        }
#pragma unroll
        for (int l = 0; l < kDig; ++l)
            w[l][p] = __byte_perm(__float_as_uint(d[0][l]), __float_as_uint(d[1][l]), 0x7632);
    }
#pragma unroll
    for (int l = 0; l < kDig; ++l)
        *reinterpret_cast<uint4 *>(dst + l * plane) = make_uint4(w[l][0], w[l][1], w[l][2], w[l][3]);
}

struct CutArgs {
    const double *X;     // element (row, k) at X[row sr + k sk]
    long sr, sk;
    long rows, K;        // valid rows and k (zeros beyond)
    int rt;              // rows per tile
    long nkb;            // k blocks
    uint8_t *dig;
    int *sh;             // [chunk][prow]: largest biased exponent of the row in the chunk (>= 100)
    long prow;           // padded rows
    int vec;             // k-contiguous rows start 16-byte aligned
};

// KFAST (sk = 1): a CTA takes 8 rows x one chunk, lane = (row, 8-k group) of its warp's block:
// 64 contiguous bytes per lane in, whole 512-byte runs of a plane out.  Otherwise (sr = 1, or
// any strides): 32 rows x one chunk, lane = row, four 8-k groups per lane.  Memory bound: 8 B
// read and 8 B written per element.
template <bool KFAST>
__global__ void __launch_bounds__(32 * kCutWarps) gemm_cut_kernel(const CutArgs a)
{
    __shared__ int smax[kCutWarps][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long chunk = blockIdx.y;
    const long k0 = chunk * kChunk + warp * kBlk;
    constexpr int G = KFAST ? 1 : 4;       // 8-k groups per lane
    const long row = KFAST ? long(blockIdx.x) * 8 + (lane & 7) : long(blockIdx.x) * 32 + lane;
    const bool ok = row < a.rows;
    double x[G][8];
    uint32_t m = 0;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const long kg = k0 + 8 * (KFAST ? lane >> 3 : g);
        const double *p = a.X + (ok ? row * a.sr : 0) + kg * a.sk;
        if (KFAST && a.vec && ok && kg + 8 <= a.K) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const double2 v = *reinterpret_cast<const double2 *>(p + 2 * e);
                x[g][2 * e] = v.x;
                x[g][2 * e + 1] = v.y;
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) x[g][e] = (ok && kg + e < a.K) ? p[e * a.sk] : 0.0;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) m = max(m, uint32_t(__double2hiint(x[g][e])) & 0x7ff00000u);
    }
    if (KFAST) {   // the lanes of one row: lane, lane ^ 8, lane ^ 16
        m = max(m, __shfl_xor_sync(0xffffffffu, m, 8));
        m = max(m, __shfl_xor_sync(0xffffffffu, m, 16));
    }
    smax[warp][lane] = int(m >> 20);
    __syncthreads();
    int E = 100;   // rows below 2^-922 are zero rows
#pragma unroll
    for (int w = 0; w < kCutWarps; ++w)
        if (w < int(blockDim.x >> 5)) E = max(E, smax[w][lane]);   // a short contraction launches fewer warps
    if (row < a.prow && warp == 0 && (!KFAST || lane < 8)) a.sh[chunk * a.prow + row] = E;
    const long kb = chunk * kBlks + warp;
    if (kb >= a.nkb || row >= a.prow) return;
    const long tile = row / a.rt;
    const int r = int(row - tile * a.rt);
#pragma unroll
    for (int g = 0; g < G; ++g)
        cut8(a.dig + cut_off(tile, r, a.rt, kb, a.nkb, KFAST ? lane >> 3 : g), size_t(a.rt) * kBlk * 2, x[g], E);
}

struct GemmArgs {
    long m;
    int n;
    int rt, Nt, mt, nt;        // tile rows and columns, tiles
    long Z;                    // k splits
    long nkb, nchunks;         // blocks and chunks of this slab
    long cper;                 // chunks per split
    const uint8_t *digA, *digB;
    const int *shA, *shB;
    long prowA, prowB;
    double *D;                 // split z writes D + z dz
    long ds_i, ds_j, dz;
    int add;                   // add to D (a later slab of k without splits)
    int ktri;                  // B(j, k) = 0 for k > j: tiles stop at their last column
    double alpha;
    int stages;
    uint32_t stage_bytes, offB, offTab, offBar;
    int tmem_cols;
    int *err;
};

// (h + l) 2^ex rounded to a double, for a chunk's sum h + l: h is its FP32 rounding, l the rest,
// zero or 2^-32 <= |h| < 2^26.  On the integer pipe: GB300 converts to and from FP64 at two per
// clock and SM, two conversions and an addition for each of 128 x 96 sums would take 18 thousand
// cycles.
__device__ __forceinline__ double chunk_value(float h, float l, int ex)
{
    const uint32_t b = __float_as_uint(h), sign = b & 0x80000000u, m = (b & 0x7fffffu) | 0x800000u;
    const int e = int((b >> 23) & 0xffu);
    int ed = e - 127 + 1023 + ex;
    if (e == 0 || uint32_t(ed - 2) > 2044u) {   // zero, or near the ends of the range
        if (e == 0 || ex < -1022) return 0.0;
        return (double(h) + double(l)) * __hiloint2double((min(ex, 1023) + 1023) << 20, 0);
    }
    // the mantissa of h as that of a double, l added in units of its last bit
    const float lq = l * __uint_as_float((uint32_t(306 - e) << 23) | sign);
    long long M = static_cast<long long>((uint64_t(m >> 3) << 32) | uint32_t(m << 29)) + __float2int_rn(lq);
    if (M < (1LL << 52)) {   // below a power of two: half the unit
        M = (1LL << 53) + __float2int_rn(2.f * lq);
        --ed;
    }
    return __hiloint2double(int((uint32_t(M >> 32) + (uint32_t(ed - 1) << 20)) | sign), int(uint32_t(M)));
}

// The CTAs walk the items (split z, row tile, column tile), column tiles fastest so that concurrent
// CTAs read the same A blocks from L2.  13 digit products per k in 4 MMAs of up to 192 columns
// (neighbouring B digits feed neighbouring levels): 320 cycles of the tensor pipe per 16 k of a
// 128 x 48 tile, against 22.5 KB of operands.
//   * SETS = 2 (tiles of 48 columns), one CTA per SM: two sets of level accumulators, so that the
//     drain warps combine a finished chunk under the next chunk's MMAs: with one set of 96 columns it
//     was not overlapped, and both products of ace_apply at n = nphi = 512 on 72 x 72 x 144 points took
//     15.7 ms, now 9.7.  TMEM loads take about as long for 4 columns as for 8: in groups of 4 the
//     combination took longer than the MMAs (10.1 ms for that call; 160 columns on 80 x 80 x 60 at
//     n = 512 3.49 ms, 2.61 in groups of 8 that skip the columns past the last).
//   * SETS = 1 (tiles of up to 32 columns), two CTAs per SM: bound by the operand blocks' way from L2
//     and by the chain load - MMA - drain - store of one item.
// PARTS: drain warps per 32 TMEM lanes (two cost 160 columns 5% more than three, four nothing less).
template <int PARTS, int SETS>
__global__ void __launch_bounds__(128 * PARTS + 64, 3 - SETS) tc_gemm_kernel(const __grid_constant__ GemmArgs a)
{
    constexpr int kDrainWarps = 4 * PARTS;
    constexpr int GW = 8;                                                       // columns of a group
    constexpr int NH = ((SETS == 1 ? kNarrow : kTN) / GW + PARTS - 1) / PARTS * GW;   // most columns of a drain warp
    extern __shared__ __align__(1024) uint8_t smem[];
    int *eb = reinterpret_cast<int *>(smem + a.offTab);            // column exponents of a chunk, two sets
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + a.offBar);
    uint64_t *empty = full + a.stages;
    uint64_t *dfull = empty + a.stages, *dempty = dfull + 2;   // per accumulator set
    uint32_t *tslot = reinterpret_cast<uint32_t *>(dempty + 2);
    int *sflag = reinterpret_cast<int *>(tslot + 1);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform
    if (tid == 0) {
        for (int i = 0; i < a.stages; ++i) {
            tc::mbar_init(full + i, 1);
            tc::mbar_init(empty + i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(dfull + i, 1);
            tc::mbar_init(dempty + i, 1);
        }
        *sflag = 0;
    }
    if (warp == 0) tc::tmem_alloc(tslot, uint32_t(a.tmem_cols));
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);
    const long items = a.Z * a.mt * a.nt;
    const int Nt = a.Nt;
    const uint32_t a_bytes = uint32_t(a.rt) * kBlk * 2 * kDig, b_bytes = uint32_t(Nt) * kBlk * 2 * kDig;
    struct Item {
        long z, c0, c1;
        int mi, ni;
    };
    auto item_of = [&](long it) {
        Item t;
        t.ni = int(it % a.nt);
        const long q = it / a.nt;
        t.mi = int(q % a.mt);
        t.z = q / a.mt;
        t.c0 = t.z * a.cper;
        t.c1 = min(a.nchunks, t.c0 + a.cper);
        if (a.ktri) t.c1 = min(t.c1, long((t.ni + 1) * Nt + kChunk - 1) / kChunk);
        return t;
    };

    if (warp == kDrainWarps) {
        // ---- producer warp: one operand block pair per stage ----
        if (lane == 0) {
            // stage and its parity by increments: a division per stage would cost as much as its MMAs
            int st = 0, filled = 0;
            uint32_t par = 1;   // of the stage's last release; the first pass over the stages waits for none
            bool bad = false, first = true;
            for (long it = blockIdx.x; it < items && !bad; it += gridDim.x) {
                const Item t = item_of(it);
                const long kb1 = min(a.nkb, t.c1 * kBlks);
                for (long kb = t.c0 * kBlks; kb < kb1; ++kb) {
                    if (!first && !tc::mbar_wait_timed(empty + st, par, kGemmWaitNs)) {
                        atomicExch(sflag, 1);
                        bad = true;
                        break;
                    }
                    uint8_t *s = smem + size_t(st) * a.stage_bytes;
                    tc::mbar_arrive_expect_tx(full + st, a_bytes + b_bytes);
                    tc::bulk_load(s, a.digA + (size_t(t.mi) * a.nkb + kb) * a_bytes, a_bytes, full + st);
                    tc::bulk_load(s + a_bytes, a.digB + (size_t(t.ni) * a.nkb + kb) * b_bytes, b_bytes, full + st);
                    filled = max(filled, st + 1);
                    if (++st == a.stages) {
                        st = 0;
                        par ^= 1u;
                        first = false;
                    }
                }
            }
            // every issued copy has landed before exit: the last fill of a stage before `st` belongs
            // to this pass over the stages (parity par ^ 1), of the others to the one before
            for (int i = 0; i < filled; ++i)
                if (!tc::mbar_wait_timed(full + i, i < st ? par ^ 1u : par, kGemmWaitNs)) atomicExch(sflag, 1);
        }
    } else if (warp == kDrainWarps + 1) {
        // ---- MMA warp ----
        int st = 0, set = 0;
        uint32_t par = 0, dpar = 3;   // dpar: per accumulator set, of its last release (the first wait passes)
        bool bad = false;
        // operand and accumulator steps, fixed for the launch: the issue of one 16-k step is a
        // straight run of MMAs by the whole warp whose descriptors differ by additions (computed in
        // a loop by one lane, a step took 1340 cycles, twice the tensor pipe's time)
        const uint32_t step_a = uint32_t(a.rt) * kBlk * 2 / 16, step_b = uint32_t(Nt) * kBlk * 2 / 16;   // next digit, in 16 bytes
        uint32_t idesc[kDig + 1];
#pragma unroll
        for (int g = 1; g <= kDig; ++g) idesc[g] = tc::instr_desc(false, g * Nt);
        const uint32_t el = tc::elect_one();
        // A digit i with the B digits 0 .. 4 - i, neighbours of levels i .. 4, in one MMA
        auto step = [&](uint32_t d0, uint64_t ad0, uint64_t bd, bool first) {
#pragma unroll
            for (int i = 0; i < kDig; ++i) {
                const int nj = kDig < kLev - i ? kDig : kLev - i;
                const uint64_t ad = ad0 + i * step_a;
                const uint32_t d = d0 + uint32_t(i * Nt);
                if (i == 1 && first) {   // digit 0 has opened levels 0..3; level 4 starts here
                    tc::mma_bf16_warp(d, ad, bd, idesc[kDig - 1], 1u, el);
                    tc::mma_bf16_warp(d0 + uint32_t(4 * Nt), ad, bd + (kDig - 1) * step_b, idesc[1], 0u, el);
                } else {
                    tc::mma_bf16_warp(d, ad, bd, idesc[nj], i == 0 && first ? 0u : 1u, el);
                }
            }
        };
        for (long it = blockIdx.x; it < items && !bad; it += gridDim.x) {
            const Item t = item_of(it);
            for (long c = t.c0; c < t.c1 && !bad; ++c) {
                if (!tc::mbar_wait_warp(dempty + set, (dpar >> set) & 1u, kGemmWaitNs)) {
                    atomicExch(sflag, 1);
                    bad = true;
                    break;
                }
                dpar ^= 1u << set;
                tc::tc_fence_after();
                const uint32_t d0 = tmem + uint32_t(set * kLev * Nt);
                const long kb0 = c * kBlks, kb1 = min(a.nkb, kb0 + kBlks);
                for (long kb = kb0; kb < kb1; ++kb) {
                    if (!tc::mbar_wait_warp(full + st, par, kGemmWaitNs)) {
                        atomicExch(sflag, 1);
                        bad = true;
                        break;
                    }
                    tc::tc_fence_after();
                    const uint32_t sa = tc::smem_addr(smem) + uint32_t(st) * a.stage_bytes;
                    const uint64_t ad = tc::smem_desc(sa, 128u, kSbo), bd = tc::smem_desc(sa + a_bytes, 128u, kSbo);
                    step(d0, ad, bd, kb == kb0);
                    step(d0, ad + 16, bd + 16, false);
                    if (el) tc::mma_commit(empty + st);
                    __syncwarp();
                    if (++st == a.stages) {
                        st = 0;
                        par ^= 1u;
                    }
                }
                if (!bad && el) tc::mma_commit(dfull + set);
                __syncwarp();
                if (SETS == 2) set ^= 1;
            }
        }
    } else {
        // ---- drain warps: TMEM lane `row`, column groups of this warp's part ----
        const int quarter = warp & 3;
        const int row = quarter * 32 + lane;
        const uint32_t lane_q = uint32_t(quarter * 32) << 16;
        const int part = (Nt / GW + PARTS - 1) / PARTS * GW, cbase = (warp >> 2) * part, ncol = min(part, Nt - cbase);
        constexpr int NT = 128 * PARTS;
        int seq = 0;   // chunks drained so far
        bool stop = false;
        for (long it = blockIdx.x; it < items && !stop; it += gridDim.x) {
            const Item t = item_of(it);
            const long i = long(t.mi) * kT + row;
            const int j0 = t.ni * Nt;
            double acc[NH];
#pragma unroll
            for (int e = 0; e < NH; ++e) acc[e] = 0.0;
            // row and column exponents, asked for a chunk ahead
            auto row_exp = [&](long c) { return i < a.m ? a.shA[c * a.prowA + i] : 0; };
            auto col_exp = [&](long c) { return tid < Nt && j0 + tid < a.n ? a.shB[c * a.prowB + j0 + tid] : 0; };
            int ea_next = row_exp(t.c0), eb_next = col_exp(t.c0);
            for (long c = t.c0; c < t.c1; ++c, ++seq) {
                const int set = SETS == 2 ? seq & 1 : 0;
                int *ebc = eb + (seq & 1) * kTN;
                if (tid < Nt) ebc[tid] = eb_next;
                // x = X 2^(E - 1052), and level 0 holds X 2^-24: 2 x (24 - 1052)
                const int ea = ea_next - 2056;
                if (c + 1 < t.c1) {
                    ea_next = row_exp(c + 1);
                    eb_next = col_exp(c + 1);
                }
                // one warp polls, the others sleep in the barrier: polls take issue slots from the MMAs'
                if (warp == 0 && !tc::mbar_wait_timed(dfull + set, uint32_t(seq / SETS) & 1u, kGemmWaitNs)) atomicExch(sflag, 1);
                if (tc::bar_red_or(1, NT, *sflag != 0)) {   // also: ebc is complete
                    stop = true;
                    break;
                }
                tc::tc_fence_after();
                const uint32_t d0 = tmem + lane_q + uint32_t(set * kLev * Nt);
#pragma unroll
                for (int cg = 0; cg < NH / GW; ++cg) {
                    const int cc = cbase + cg * GW;
                    if (cg * GW >= ncol || j0 + cc >= a.n || i - lane >= a.m) break;   // uniform
                    uint32_t r[kLev][GW];
#pragma unroll
                    for (int l = 0; l < kLev; ++l) tc::tmem_ld8_issue(d0 + uint32_t(l * Nt + cc), r[l]);
                    tc::tmem_wait_ld();
#pragma unroll
                    for (int l = 0; l < kLev; ++l)
#pragma unroll
                        for (int e = 0; e < GW; ++e) tc::order_after_wait(r[l][e]);
#pragma unroll
                    for (int e = 0; e < GW; e += 2) {
                        // levels combined in FP32 down to level 1 (rounding ~2^-32 of level 0's
                        // scale), level 0 added with TwoSum, the pair summed over the chunks in FP64
                        auto lv = [&](int l) { return make_float2(__uint_as_float(r[l][e]), __uint_as_float(r[l][e + 1])); };
                        const float2 q = make_float2(1.f / 256.f, 1.f / 256.f), m1 = make_float2(-1.f, -1.f);
                        float2 tl = __ffma2_rn(lv(4), q, lv(3));
                        tl = __ffma2_rn(tl, q, lv(2));
                        tl = __ffma2_rn(tl, q, lv(1));
                        tl = __fmul2_rn(tl, q);
                        const float2 l0 = lv(0);
                        const float2 h = __fadd2_rn(l0, tl);
                        const float2 b0 = __ffma2_rn(l0, m1, h);
                        const float2 lo = __fadd2_rn(__ffma2_rn(__ffma2_rn(b0, m1, h), m1, l0), __ffma2_rn(b0, m1, tl));
                        const int2 ebv = *reinterpret_cast<const int2 *>(ebc + cc + e);
                        acc[cg * GW + e] += chunk_value(h.x, lo.x, ea + ebv.x);
                        acc[cg * GW + e + 1] += chunk_value(h.y, lo.y, ea + ebv.y);
                    }
                }
                tc::tc_fence_before();   // TMEM reads before a later chunk's MMAs overwrite them
                tc::bar_sync(1, NT);
                if (tid == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_addr(dempty + set)) : "memory");
            }
            if (stop) break;
            if (i < a.m) {
                double *D = a.D + t.z * a.dz + i * a.ds_i;
#pragma unroll
                for (int e = 0; e < NH; ++e) {
                    const int j = j0 + cbase + e;
                    if (e < ncol && j < a.n) {
                        double *dp = D + long(j) * a.ds_j;
                        *dp = a.add ? fma(a.alpha, acc[e], *dp) : a.alpha * acc[e];
                    }
                }
            }
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (tid == 0 && *sflag) atomicExch(a.err, 1);
    if (warp == 0) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, uint32_t(a.tmem_cols));
    }
}

// D(i, j) (+)= alpha sum_z W[z][i + m j] with the output strides: 32 entries per CTA, eight threads
// each take every eighth split, then a fixed order (one thread per entry left 116 loads in sequence:
// 20 us for 128 x 16).
constexpr int kRedZ = 8;
__global__ void __launch_bounds__(32 * kRedZ) tc_gemm_reduce_kernel(const double *W, int Z, long m, int n, double alpha, double *D,
                                                                    long ds_i, long ds_j, int add)
{
    __shared__ double sh[kRedZ][32];
    const long tot = m * n;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (long e0 = long(blockIdx.x) * 32; e0 < tot; e0 += long(gridDim.x) * 32) {
        const long e = e0 + tx;
        double s = 0.0;
        if (e < tot)
            for (int z = ty; z < Z; z += kRedZ) s += W[long(z) * tot + e];
        sh[ty][tx] = s;
        __syncthreads();
        if (ty == 0 && e < tot) {
            for (int z = 1; z < kRedZ; ++z) s += sh[z][tx];
            double *dp = D + (e % m) * ds_i + (e / m) * ds_j;
            *dp = add ? fma(alpha, s, *dp) : alpha * s;
        }
        __syncthreads();
    }
}

inline long ceil_div(long a, long b) { return (a + b - 1) / b; }
inline size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Rows past the last group of 8 (or 32) that holds a valid one are left as they are: a row of an
// operand only reaches its own row or column of the output, and those are never stored.
int launch_cut(Plan &P, const double *X, long sr, long sk, long rows, long K, int rt, long tiles, uint8_t *dig, int *sh,
               cudaStream_t s)
{
    CutArgs c{};
    c.X = X;
    c.sr = sr;
    c.sk = sk;
    c.rows = rows;
    c.K = K;
    c.rt = rt;
    c.nkb = ceil_div(K, kBlk);
    c.dig = dig;
    c.sh = sh;
    c.prow = tiles * rt;
    c.vec = ((reinterpret_cast<uintptr_t>(X) | uintptr_t(sr * 8)) & 15) == 0;
    const unsigned chunks = unsigned(ceil_div(K, kChunk));
    const int threads = 32 * int(std::min<long>(kCutWarps, c.nkb));
    const int tb = timing_begin(P, EXX_TIMING_GEMM, s);
    if (sk == 1)
        gemm_cut_kernel<true><<<dim3(unsigned(ceil_div(c.rows, 8)), chunks), threads, 0, s>>>(c);
    else
        gemm_cut_kernel<false><<<dim3(unsigned(ceil_div(c.rows, 32)), chunks), threads, 0, s>>>(c);
    timing_end(P, tb, s);
    EXX_LAUNCH("gemm_cut_kernel");
    P.launches++;
    return EXX_OK;
}

}  // namespace

// Tiles, slabs and workspace of one product whose digit planes may take `budget` bytes.
GemmShape gemm_shape(const GemmDims &d, int num_sms, long budget)
{
    GemmShape g{};
    // column tiles: as even as 16-column steps allow, at most 48 (two sets of 5 levels in 512 TMEM columns)
    g.nt = int(ceil_div(d.n, kTN));
    g.Nt = int(ceil_div(ceil_div(d.n, g.nt), 16) * 16);
    const long np = long(g.nt) * g.Nt;
    // slabs: the digit planes (8 B per element) of one slab stay within the budget, cut along m
    // when the contraction is short, along k when it is long
    const long chunks = ceil_div(d.K, kChunk);
    const long chunk_bytes = std::min(8L * kChunk, ceil_div(d.K, kBlk) * kBlk * 8);   // per row (and of a lone short chunk)
    g.rt = int(std::min<long>(kT, ceil_div(d.m, 8) * 8));   // a lone short tile holds, and moves, no more rows than it has
    const long mpad = ceil_div(d.m, g.rt) * g.rt;
    g.mslab = mpad;
    g.kslab = chunks;
    if (chunks > 64) {
        g.kslab = std::max(1L, budget / (chunk_bytes * (mpad + np)));
    } else {
        g.kslab = std::min(chunks, std::max(1L, budget / 2 / (chunk_bytes * std::max<long>(np, g.rt))));
        const long room = budget - std::min(budget / 2, chunk_bytes * g.kslab * np);
        g.mslab = std::max<long>(g.rt, room / (chunk_bytes * g.kslab) / g.rt * g.rt);
    }
    g.mslab = std::min(g.mslab, mpad);
    g.kslab = std::min(std::min(g.kslab, chunks), 65535L);
    g.kslab = ceil_div(chunks, ceil_div(chunks, g.kslab));                     // even slabs
    g.mslab = ceil_div(mpad / g.rt, ceil_div(mpad, g.mslab)) * g.rt;
    // k splits: items (tiles x splits) for a whole number of rounds over the SMs
    g.ktri = d.ktri && g.kslab == chunks;   // the limit counts chunks from k = 0
    g.slots = long(num_sms) * (g.Nt <= kNarrow ? 2 : 1);   // CTAs resident at once
    g.Zmax = 1;
    const long tiles = (g.mslab / g.rt) * g.nt;
    if (!g.ktri && g.kslab > 1 && tiles < 2 * g.slots) {
        const long round = std::max(1L, g.slots / tiles);
        const long slot = ceil_div(g.mslab, kT) * kT * d.n * long(sizeof(double));
        g.Zmax = std::min(g.kslab >= 8 * round ? 2 * round : round, g.kslab);
        g.Zmax = std::min(g.Zmax, std::max(1L, budget / 4 / slot));
    }
    g.offB = round_up(size_t(g.mslab) * chunk_bytes * g.kslab, 256);
    g.offSA = g.offB + round_up(size_t(np) * chunk_bytes * g.kslab, 256);
    g.offSB = g.offSA + round_up(size_t(g.mslab) * g.kslab * 4, 256);
    g.offP = g.offSB + round_up(size_t(np) * g.kslab * 4, 256);
    g.bytes = g.offP + (g.Zmax > 1 ? size_t(g.Zmax) * std::min(g.mslab, d.m) * d.n * sizeof(double) : 0);
    return g;
}

// One workspace for the products of a call.  A device too full for it gets smaller slabs, down to
// one tile and one chunk; the plan keeps the smaller budget.
int tc_gemm_reserve(Plan &P, const GemmDims *d, int count)
{
    for (;;) {
        size_t bytes = 0;
        bool least = true;
        for (int i = 0; i < count; ++i) {
            const GemmShape g = gemm_shape(d[i], P.num_sms, P.gemm_budget);
            bytes = std::max(bytes, g.bytes);
            least = least && g.mslab == g.rt && g.kslab == 1;
        }
        const int rc = plan_reserve(P, P.gemm_ws, bytes);
        if (rc != EXX_ERR_OOM || least || P.gemm_budget < 2) return rc;
        P.gemm_budget /= 2;
    }
}

int tc_gemm(Plan &P, long m, int n, long K, const double *A, long as_i, long as_k, const double *B, long bs_j,
            long bs_k, double alpha, double *D, long ds_i, long ds_j, cudaStream_t s, bool ktri)
{
    if (m < 1 || n < 1 || K < 1) return EXX_ERR_INVALID_ARG;
    if (!P.err_d.p) {
        if (int rc = dev_reserve(P.err_d, 16)) return rc;
        EXX_CUDA(cudaMemsetAsync(P.err_d.p, 0, 16, s));
    }
    const GemmDims dims{m, n, K, ktri};
    GemmShape g = gemm_shape(dims, P.num_sms, P.gemm_budget);
    if (P.gemm_ws.bytes < g.bytes) {
        if (int rc = tc_gemm_reserve(P, &dims, 1)) return rc;
        g = gemm_shape(dims, P.num_sms, P.gemm_budget);
    }
    uint8_t *ws = static_cast<uint8_t *>(P.gemm_ws.p);
    int *shA = reinterpret_cast<int *>(ws + g.offSA), *shB = reinterpret_cast<int *>(ws + g.offSB);
    const int rt = g.rt, nt = g.nt, Nt = g.Nt;
    const long np = long(nt) * Nt, mslab = g.mslab, kslab = g.kslab, chunks = ceil_div(K, kChunk);
    ktri = g.ktri;

    GemmArgs a{};
    a.n = n;
    a.rt = rt;
    a.Nt = Nt;
    a.nt = nt;
    a.digA = ws;
    a.digB = ws + g.offB;
    a.shA = shA;
    a.shB = shB;
    a.prowB = np;
    a.ktri = ktri ? 1 : 0;
    a.err = static_cast<int *>(P.err_d.p);
    a.stage_bytes = uint32_t(rt + Nt) * kBlk * 2 * kDig;
    const bool narrow = Nt <= kNarrow;
    a.stages = int(std::min<size_t>(8, (narrow ? 111 : 222) * 1024 / a.stage_bytes));
    a.offTab = uint32_t(a.stages) * a.stage_bytes;
    a.offBar = a.offTab + 2 * kTN * 4;
    a.tmem_cols = 32;
    while (a.tmem_cols < (narrow ? 1 : 2) * kLev * Nt) a.tmem_cols *= 2;
    size_t smem = a.offBar + (2 * size_t(a.stages) + 4) * 8 + 16;
    // the MMA reads 128 rows of every A digit: what lies past a short tile's, to lanes nobody reads
    smem = std::max(smem, size_t(a.stages - 1) * a.stage_bytes + (size_t(3) * rt + kT) * kBlk * 2);
    auto kern = narrow ? tc_gemm_kernel<2, 1> : tc_gemm_kernel<kParts, 2>;
    const int threads = 128 * (narrow ? 2 : kParts) + 64;
    EXX_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));

    for (long c0 = 0; c0 < chunks; c0 += kslab) {
        const long nch = std::min(kslab, chunks - c0);
        const long k0 = c0 * kChunk, kk = std::min(K - k0, nch * kChunk);
        if (int rc = launch_cut(P, B + k0 * bs_k, bs_j, bs_k, n, kk, Nt, nt, ws + g.offB, shB, s)) return rc;
        for (long i0 = 0; i0 < m; i0 += mslab) {
            const long mr = std::min(mslab, m - i0);
            a.mt = int(ceil_div(mr, rt));
            if (int rc = launch_cut(P, A + i0 * as_i + k0 * as_k, as_i, as_k, mr, kk, rt, a.mt, ws, shA, s)) return rc;
            a.m = mr;
            a.prowA = long(a.mt) * rt;
            a.nkb = ceil_div(kk, kBlk);
            a.nchunks = nch;
            a.Z = std::min(g.Zmax, nch);
            a.cper = ceil_div(nch, a.Z);
            a.Z = ceil_div(nch, a.cper);
            double *Dd = D + i0 * ds_i;
            a.alpha = a.Z > 1 ? 1.0 : alpha;   // split sums take it in the reduction
            if (a.Z > 1) {
                a.D = reinterpret_cast<double *>(ws + g.offP);
                a.ds_i = 1;
                a.ds_j = mr;
                a.dz = mr * n;
                a.add = 0;
            } else {
                a.D = Dd;
                a.ds_i = ds_i;
                a.ds_j = ds_j;
                a.dz = 0;
                a.add = c0 > 0;
            }
            const long items = a.Z * a.mt * a.nt;
            int tb = timing_begin(P, EXX_TIMING_GEMM, s);
            kern<<<unsigned(std::min<long>(items, g.slots)), threads, smem, s>>>(a);
            timing_end(P, tb, s);
            EXX_LAUNCH("tc_gemm_kernel");
            P.launches++;
            if (a.Z > 1) {
                const long tot = mr * n;
                tb = timing_begin(P, EXX_TIMING_GEMM, s);
                tc_gemm_reduce_kernel<<<unsigned(std::min<long>((tot + 31) / 32, 32L * P.num_sms)), 32 * kRedZ, 0, s>>>(
                    a.D, int(a.Z), mr, n, alpha, Dd, ds_i, ds_j, c0 > 0);
                timing_end(P, tb, s);
                EXX_LAUNCH("tc_gemm_reduce_kernel");
                P.launches++;
            }
        }
    }
    return EXX_OK;
}

}  // namespace exx
