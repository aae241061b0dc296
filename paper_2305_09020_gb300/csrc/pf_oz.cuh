// FP64 transform GEMM on the tensor cores (tcgen05 kind::f16, sm_103a): exact products of 8-bit digits.
//
// C[M x N] = A[M x K] * B[K x N] for the constant eigenbasis products of the Remark after Algorithm 2 in
// double precision.  The FP64 pipe of the GB300 runs 2 FMA per SM and cycle (1.1 TFLOP/s measured), the
// tensor cores 4096 FP16 products, and small integers multiply and add exactly there.  So each operand
// is written in fixed point (the integer splitting of Ozaki, Ogita, Oishi and Rump for matrix units), after
// the terms a_mk b_kn of a sum have been balanced by an exact power of two per k:
//   s_k             the largest biased exponent of B's row k less 1023 (a table of the basis; rows of zeros,
//                   the eigenbases' constrained nodes, are left out of A whatever A holds there),
//   row m of A:     a_mk 2^s_k = X 2^(E_m - 1084),  X = rint(a_mk 2^(s_k + 1084 - E_m)), |X| < 2^62,
//                   E_m the largest biased exponent of the balanced row,
//   column n of B:  b_kn 2^-s_k = Y 2^(F_n - 1084), the same,
//   X = sum_s x_s 256^(7-s), eight balanced digits -128 <= x_s <= 127 (|x_0| <= 64), stored as FP16 integers.
// X Y summed over k is sum_d 256^(14-d) v_d with the level sums v_d = sum_{s+t=d} sum_k x_s y_t.  Levels
// 0..7 (36 digit products) are kept: the first dropped level is about 2^-61 of the product of the largest
// balanced entries of row and column.  Over a group of 128 k every level sum is an integer of at most
// 128 (6 2^14 + 2 2^13) < 2^24, so the tensor core's FP32 accumulation is exact.  The drain of a group adds the
// levels into a 64-bit integer and a byte of fraction, in units of 256^8:
//   256 acc + frac += v_0 2^48 + v_1 2^40 + v_2 2^32 + v_3 2^24 + v_4 2^16 + v_5 2^8 + v_6 + rint(v_7 / 256),
// which is exact but for v_7; |acc| < 2^62 for K < 512.  The result is rounded to double once.
//
// The error is relative to the largest balanced entries, an FMA chain's to the sum of the terms' sizes.
// Balanced, the largest entry of A meets the largest entry of B's row, so that one term of the row of C is
// as large as their product, and eight digits leave 2^-61 of it where a chain leaves 2^-53 per term: no plane, row
// or column of the solves tested is further off than with the chains (even, cosine and geometric meshes to a ratio
// of 4^10 in size, values of 1e200 at constrained nodes).  Measured against extended precision, 105 x 43
// nodes on a cosine mesh, plane / worst row / worst column: chains 8.4e-16 / 1.3e-15 / 2.9e-15, seven digits
// without the balance 1.1e-15 / 6.1e-14 / 5.7e-15 (and no digit left for a value of 1e16 at a constrained node),
// seven with it 6e-16 / 1.6e-14 / 4e-15 (emulated), these 1.2e-16 / 2.0e-16 / 3.0e-16.
// What cannot be balanced per k is a basis of uncoupled pieces (zeros inside rows and columns that are not
// zero): entries of one piece would take digits from another.  The allocation-free solve, whose bases are the
// caller's, finds those on the device and takes the FMA kernels (pf_static.cu); a run's own have none.
//
// A row of A or a column of B with an infinity or NaN gives NaN results; other rows and columns are not
// affected.  Subnormal entries keep their bits; normal results are rounded to nearest, ties to even.
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "pf_tc.cuh"

namespace pf {

constexpr int OZ_S = 8;                       // digits per operand, levels of the product
constexpr int OZ_KC = 32;                     // K per stage: 64-byte rows of FP16
constexpr int OZ_BM = 128;                    // rows per unit = TMEM lanes
constexpr int OZ_MAXH = 16;                   // accumulator columns per drain thread: BN <= 64
constexpr int OZ_GRP = 4;                     // stages per accumulation group (128 k)
constexpr int OZ_MAXK = 480;                  // K bound of the 64-bit sums (< 512)
constexpr int OZ_SKIP = -(1 << 20);           // shift of a k whose row of B is zero
constexpr int OZ_NONFINITE = 1 << 20;         // exponent of a row or column with an infinity or NaN
constexpr int OZ_EPI_WARPS = 16;              // four warpgroups: a quarter of the columns each
constexpr int OZ_THREADS = 640;
// the launch holds 640 x 96 = 61440 registers: 512 x 104 + 128 x 64 = 61440
constexpr int OZ_REG_EPI = 104, OZ_REG_AUX = 64;
static_assert(512 * OZ_REG_EPI + 128 * OZ_REG_AUX <= OZ_THREADS * 96, "the setmaxnreg split must fit the launch's registers");
constexpr uint32_t OZ_ABYTES = OZ_S * OZ_BM * OZ_KC * 2;   // A digits of a stage
constexpr int OZ_OUTC = 4, OZ_OUTP = 5;       // columns (a word of fractions) and row pitch (doubles) of a drain warp's store block
constexpr size_t OZ_OUTBYTES = (size_t)OZ_EPI_WARPS * 32 * OZ_OUTP * 8;
constexpr size_t OZ_FIXED = 1024 + OZ_OUTBYTES + 512;      // alignment slack; store blocks; barriers, TMEM slot

struct OzArgs {
    int M, N, K;
    int BN;                   // column tile (multiple of 32, <= 4 OZ_MAXH)
    int ntn;                  // column tiles
    int BNlast;               // width of the last one (multiple of 32)
    int nst;                  // K stages
    int stages;               // shared-memory stages
    int tmem_cols;            // >= OZ_S BN: a region per level
    int nunits;               // row tiles x column tiles
    const int *E, *F;         // exponents of A's rows and B's columns
    // epilogue: row m = p R + r; store 0: C[m ldc + n]; store 1: C[(p N + n) ldr + r]
    int R, store, ldc, ldr;
    const double *lamN, *lamR, *cpl;   // optional division by lamN[n] + lamR[r] + cpl[p % cpl_mod]
    int cpl_mod;
    const double2 *rcp;       // its reciprocals (oz_recip) [mode][r][n], mode of plane p: 0 when rcp_modes == 1,
    int rcp_modes;            // else that of the packed Fourier plane p % cpl_mod; null: divide
    double *C;
    double *C2;               // optional C2[m ldc + n] = -m2x[n] m2y[r] C (+ face2[p N + n] on r == 0)
    const double *m2x, *m2y, *face2;
    const int *active;        // ensembles: per-run flags (0 = frozen), run = p % amod; null otherwise
    int amod;
    const int *skip_if;       // nullable: nothing is done where it holds a value that is not 0
    int *err;                 // error word; null: a call without one, whose results become NaN on a time-out
    unsigned long long wait_ns;
    int stall;                // test hook: wait on a barrier that nothing arrives at, report, return
};

constexpr size_t OZ_SMEM = 227 * 1024;
__host__ __device__ inline int oz_kpad(int k) { return (k + OZ_KC - 1) / OZ_KC * OZ_KC; }

// sizes of the product of `rows` rows with an N x N matrix: column tiles, stages, shared memory.  Column
// tiles: enough units for the chip, against the cycles of a unit: 72 MMAs a stage of 40 + BN/4 cycles and
// about 6000 + 130 per column around them.
inline OzArgs oz_plan(long long rows, int N, int sms, size_t *smem) {
    OzArgs a{};
    const int mt = (int)((rows + OZ_BM - 1) / OZ_BM);
    a.M = (int)rows; a.N = N; a.K = N;
    a.nst = oz_kpad(N) / OZ_KC;
    double best = 0;
    for (int nt = (N + 4 * OZ_MAXH - 1) / (4 * OZ_MAXH); nt <= (N + 31) / 32; ++nt) {
        const int bn = ((N + nt - 1) / nt + 31) / 32 * 32, tiles = (N + bn - 1) / bn;
        const double rounds = (double)(((long long)mt * tiles + sms - 1) / sms);
        const double t = rounds * (a.nst * (72.0 * (40.0 + 0.25 * bn)) + 6000.0 + 130.0 * bn);
        if (a.BN == 0 || t < 0.98 * best) { best = t; a.BN = bn; a.ntn = tiles; }
    }
    a.BNlast = ((N - (a.ntn - 1) * a.BN) + 31) / 32 * 32;
    a.tmem_cols = 512;
    const size_t stage = OZ_ABYTES + (size_t)OZ_S * a.BN * OZ_KC * 2, fit = (OZ_SMEM - OZ_FIXED) / stage;
    a.stages = fit < 4 ? (int)fit : 4;
    a.nunits = mt * a.ntn;
    *smem = a.stages * stage + OZ_FIXED;
    return a;
}

// digit planes [OZ_S][rows][Kpad], boxes of 32 x box_rows x 8
inline bool oz_encode(CUtensorMap *m, const __half *ptr, long long rows, int Kpad, int box_rows) {
    cuuint64_t dims[3] = {(cuuint64_t)Kpad, (cuuint64_t)rows, (cuuint64_t)OZ_S};
    cuuint64_t strides[2] = {(cuuint64_t)Kpad * 2, (cuuint64_t)Kpad * 2 * rows};
    cuuint32_t box[3] = {(cuuint32_t)OZ_KC, (cuuint32_t)box_rows, (cuuint32_t)OZ_S};
    cuuint32_t estr[3] = {1, 1, 1};
    return tc_encode()(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half *>(ptr), dims, strides, box, estr,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// K-major, 64-byte swizzle, 8-row atoms of 512 bytes
__device__ __forceinline__ uint64_t sdesc_sw64(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(512 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;
    return d;
}

// instruction descriptor: D = F32, A = B = F16, both K-major, shape M x N
__device__ __forceinline__ uint32_t idesc_f16(int M, int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int x, int y, int z, uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
            dst),
        "l"((unsigned long long)map), "r"(x), "r"(y), "r"(z), "r"(mbar)
        : "memory");
}

// biased fixed point of a double whose balanced exponent lies r >= 0 below its row's:
// X + 128 (256^7 + .. + 1), so that byte s from the top is digit x_s + 128
__host__ __device__ __forceinline__ unsigned long long oz_fixed(unsigned long long bits, int r) {
    unsigned long long m = bits & 0xFFFFFFFFFFFFFull;
    if ((bits >> 52) & 0x7FF) m |= 1ull << 52;
    if (r > 63) r = 63;
    m = (((m << 10) >> r) + 1) >> 1;
    const unsigned long long s = 0ull - (bits >> 63);
    return ((m ^ s) - s) + 0x8080808080808080ull;
}
// biased exponent of a double for oz_fixed (1 for subnormals), shifted; OZ_SKIP and less for 0 and a left-out k
__host__ __device__ __forceinline__ int oz_exp(unsigned long long bits, int sh) {
    const int e = (int)(bits >> 52) & 0x7FF;
    return (bits << 1) ? (e ? e : 1) + sh : 2 * OZ_SKIP;
}

// (acc 256 + frac) 2^sc rounded to nearest even: one conversion (a rounding to odd keeps what does not fit into
// 64 bits), the power of two added to its exponent.  Normalising by integer operations instead took
// about thirty: 1 to 3% of a step
__device__ __forceinline__ double oz_double(long long acc, int frac, int sc) {
    const bool fits = (unsigned long long)(acc + (1ll << 54)) < (1ull << 55);
    const long long v = fits ? acc * 256 + frac : (acc + (frac >> 8)) | ((frac & 0xFF) != 0);
    if (!fits) sc += 8;
    const double x = __ll2double_rn(v);
    const int hi = __double2hiint(x), e = ((hi >> 20) & 0x7FF) + sc;
    if (v == 0) return 0.0;
    if (e < 1 || e > 2046) {   // subnormal or overflowing results: by powers of two in range
        const int t = min(max(sc, -2200), 2200), t1 = t / 3, t2 = (t - t1) / 2, t3 = t - t1 - t2;
        return x * __longlong_as_double((long long)(1023 + t1) << 52) * __longlong_as_double((long long)(1023 + t2) << 52) *
               __longlong_as_double((long long)(1023 + t3) << 52);
    }
    return __hiloint2double(hi + (int)((unsigned)sc << 20), __double2loint(x));
}

// 1/d as a rounded reciprocal and what it leaves (0 for d = 0, whose quotients are 0), and x/d from them: the
// product with both is x/d to 2^-100 before it is rounded, once, as the division operator rounds.  The
// rounded reciprocal alone leaves up to 1.5 units in the last place.
__host__ __device__ __forceinline__ double2 oz_recip(double d) {
    if (d == 0.0) return double2{0.0, 0.0};
    const double r = 1.0 / d, lo = fma(-r, d, 1.0) * r;
    return double2{r, lo == lo ? lo : 0.0};
}
__host__ __device__ __forceinline__ double oz_quot(double x, double2 r) { return fma(x, r.x, x * r.y); }

#ifndef PF_OZ_HELPERS_ONLY
// ---- digits of A: one warp per row ----------------------------------------------------------------
// dig[d][m][Kpad] (FP16), E[m], of the values row[k ks] 2^(sg sh[k]) of row m.  NI = ceil(Kpad / 64) pairs a lane;
// sh holds Kpad shifts.  sparse (nullable) is set where a row that is not zero has a zero at a k that is not
// left out.
template <int NI>
__device__ __forceinline__ void oz_split_row(const double *__restrict__ row, int ks, const int *__restrict__ sh, int sg, int m,
                                             int M, int K, int Kpad, __half *__restrict__ dig, int *__restrict__ E, int *sparse) {
    const int lane = threadIdx.x & 31;
    double x[NI][2];
    int ex[NI][2], em = 2 * OZ_SKIP;
    bool bad = false, hole = false;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int k = 2 * (lane + 32 * i);
        x[i][0] = k < K ? row[(long long)k * ks] : 0.0;
        x[i][1] = k + 1 < K ? row[(long long)(k + 1) * ks] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int k = 2 * (lane + 32 * i);
        const int2 s = k < Kpad ? *reinterpret_cast<const int2 *>(sh + k) : make_int2(OZ_SKIP, OZ_SKIP);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int sj = j ? s.y : s.x;
            bad |= (__double2hiint(x[i][j]) & 0x7FF00000) == 0x7FF00000;
            if (sj == OZ_SKIP) x[i][j] = 0.0;
            hole |= sj != OZ_SKIP && x[i][j] == 0.0;
            ex[i][j] = oz_exp((unsigned long long)__double_as_longlong(x[i][j]), sg * sj);
            em = max(em, ex[i][j]);
        }
    }
    em = __reduce_max_sync(0xffffffffu, em);
    bad = __any_sync(0xffffffffu, bad);
    hole = __any_sync(0xffffffffu, hole);
    if (lane == 0) {
        E[m] = bad ? OZ_NONFINITE : max(em, OZ_SKIP);
        if (sparse && hole && em > OZ_SKIP) *sparse = 1;
    }
    const long long DS = (long long)M * Kpad / 2;     // words per digit plane
    uint32_t *dst = reinterpret_cast<uint32_t *>(dig) + (long long)m * (Kpad / 2) + lane;
    const __half2 bias = __half2half2(__ushort_as_half(0x6480));   // 1152
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        if (2 * (lane + 32 * i) >= Kpad) break;
        const unsigned long long ua = oz_fixed((unsigned long long)__double_as_longlong(x[i][0]), em - ex[i][0]);
        const unsigned long long ub = oz_fixed((unsigned long long)__double_as_longlong(x[i][1]), em - ex[i][1]);
        const uint32_t al = (uint32_t)ua, ah = (uint32_t)(ua >> 32), bl = (uint32_t)ub, bh = (uint32_t)(ub >> 32);
#pragma unroll
        for (int d = 0; d < OZ_S; ++d) {   // two FP16 words 1024 + digit + 128, less 1152
            const uint32_t v = (__byte_perm(d < 4 ? ah : al, d < 4 ? bh : bl, 0x0703 - 0x0101 * (d & 3)) & 0x00FF00FFu) | 0x64006400u;
            const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&v), bias);
            dst[d * DS + 32 * i] = *reinterpret_cast<const uint32_t *>(&h);
        }
    }
}

// Bound by its 8 bytes read and 16 written per value, most of them in L2; a pass of its own because inside the
// GEMM every column tile would split the rows again (measured there: 7,000 issue slots per 128 x 32 stage
// against 3,100 cycles of MMAs).
template <int NI>
__global__ void __launch_bounds__(256) k_oz_split(const double *__restrict__ A, int M, int K, int Kpad, const int *__restrict__ sh,
                                                  __half *__restrict__ dig, int *__restrict__ E, int R,
                                                  const int *__restrict__ active, int amod, const int *__restrict__ skip_if) {
    const int m = blockIdx.x * 8 + (threadIdx.x >> 5);
    tc_pdl_enter();
    if (m >= M || (skip_if && *skip_if)) return;
    if (active && !active[(m / R) % amod]) return;   // a frozen run's rows: their products are not used
    oz_split_row<NI>(A + (long long)m * K, 1, sh, 1, m, M, K, Kpad, dig, E, nullptr);
}

// launch of k_oz_split for the M rows of A (K <= OZ_MAXK values each); pdl: as a programmatic dependent launch;
// skip_if: as OzArgs
inline void oz_split(const double *A, int M, int K, const int *sh, __half *dig, int *E, int R, const int *active, int amod,
                     cudaStream_t st, bool pdl = false, const int *skip_if = nullptr) {
    const int Kpad = oz_kpad(K);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((M + 7) / 8));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    auto go = [&](void (*k)(const double *, int, int, int, const int *, __half *, int *, int, const int *, int, const int *)) {
        cudaLaunchKernelEx(&cfg, k, A, M, K, Kpad, sh, dig, E, R, active, amod, skip_if);   // errors: the caller's cudaGetLastError
    };
    switch ((Kpad + 63) / 64) {
        case 1: go(k_oz_split<1>); break;
        case 2: go(k_oz_split<2>); break;
        case 3: go(k_oz_split<3>); break;
        case 4: go(k_oz_split<4>); break;
        case 5: go(k_oz_split<5>); break;
        case 6: go(k_oz_split<6>); break;
        default: go(k_oz_split<8>);
    }
}

// ---- digits of a caller's bases (the allocation-free solve), all four in two launches -------------------
struct OzBases {
    const double *B[4];      // n x n, row-major
    int n[4];
    int *sh[4];              // shifts of the rows, oz_kpad(n) entries
    __half *dig[4];
    int *F[4];
    int *sparse;             // 1: a basis has zeros inside rows and columns that are not zero
};

// shifts: one warp per row of a basis.  Infinities and NaN (whose columns' results are NaN) set none.
static __global__ void __launch_bounds__(256) k_oz_rows(OzBases g) {
    const int b = blockIdx.y, k = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31, n = g.n[b];
    if (blockIdx.x == 0 && b == 0 && threadIdx.x == 0) *g.sparse = 0;
    if (k >= oz_kpad(n)) return;
    int e = OZ_SKIP;
    if (k < n)
        for (int j = lane; j < n; j += 32) {
            const unsigned long long u = (unsigned long long)__double_as_longlong(g.B[b][(long long)k * n + j]);
            if (((u >> 52) & 0x7FF) != 0x7FF) e = max(e, oz_exp(u, -1023));
        }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) g.sh[b][k] = e;
}

// digits: one warp per column, blockIdx.y the basis
template <int NI>
static __global__ void __launch_bounds__(256) k_oz_split_bases(OzBases g) {
    const int b = blockIdx.y, m = blockIdx.x * 8 + (threadIdx.x >> 5), n = g.n[b];
    if (m >= n) return;
    oz_split_row<NI>(g.B[b] + m, n, g.sh[b], -1, m, n, n, oz_kpad(n), g.dig[b], g.F[b], g.sparse);
}

inline void oz_split_bases(const OzBases &g, cudaStream_t st) {   // errors: the caller's cudaGetLastError
    int n = 0;
    for (int v : g.n) n = v > n ? v : n;
    k_oz_rows<<<dim3((unsigned)((oz_kpad(n) + 7) / 8), 4), 256, 0, st>>>(g);
    const dim3 grid((unsigned)((n + 7) / 8), 4);
    switch ((oz_kpad(n) + 63) / 64) {
        case 1: k_oz_split_bases<1><<<grid, 256, 0, st>>>(g); break;
        case 2: k_oz_split_bases<2><<<grid, 256, 0, st>>>(g); break;
        case 3: k_oz_split_bases<3><<<grid, 256, 0, st>>>(g); break;
        case 4: k_oz_split_bases<4><<<grid, 256, 0, st>>>(g); break;
        default: k_oz_split_bases<8><<<grid, 256, 0, st>>>(g);
    }
}

// reciprocals of the eigenvalue sums of one solve family, [mode][r][n]
static __global__ void k_oz_rcp(double2 *__restrict__ out, const double *__restrict__ lamN, const double *__restrict__ lamR,
                                const double *__restrict__ shift, int modes, int nz, int R, int N) {
    const long long n = (long long)modes * R * N;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(i / ((long long)R * N));
        const int r = (int)(i / N - (long long)k * R), c = (int)(i % N);
        const int p = modes == 1 ? 0 : k == 0 ? 0 : (k == nz / 2 ? 1 : 2 * k);   // a packed plane of mode k
        out[i] = oz_recip(lamN[c] + lamR[r] + shift[p]);
    }
}

__device__ __forceinline__ bool oz_frozen(const OzArgs &g, int mt) {
    if (!g.active) return false;
    const int p1 = (min((mt + 1) * OZ_BM, g.M) - 1) / g.R;
    for (int p = mt * OZ_BM / g.R; p <= p1; ++p)
        if (g.active[p % g.amod]) return false;
    return true;
}

// ---- the GEMM: persistent, warp-specialised; a CTA walks units of 128 rows x BN columns -------------
//   warp 16     TMA: per 32-wide K stage the digits of A (32 x 128 x 8) and of B (32 x BN x 8), one 3D box each
//   warps 17-18 issue the MMAs level by level (7 first), each level into a tensor-memory region of its own
//               that it accumulates over a group of four stages: levels 7, 6, 2 by one warp, 5, 4, 3, 1, 0 by
//               the other, 36 MMAs of a stage each.  The drain of a level overlaps the group's later
//               levels and the next group's first stage
//   warps 0-15  drain the regions into the 64-bit integers, then convert and store (the epilogues of
//               k_gemm).  Sixteen, because this code overflows the schedulers' instruction caches and its
//               fetches are shared by a scheduler's warps
// setmaxnreg moves registers from warps 16-19 to the drain warps.  Every mbarrier wait is bounded as in
// pf_tc.cuh: on time-out the error word is set, copies and MMAs in flight finish (bounded), tensor memory
// is freed and the kernel returns.
static __global__ void __launch_bounds__(OZ_THREADS, 1) k_gemm_oz(const __grid_constant__ CUtensorMap tmA,
                                                                  const __grid_constant__ CUtensorMap tmB, OzArgs g) {
    if (g.skip_if && *g.skip_if) return;
    extern __shared__ __align__(1024) unsigned char oz_raw[];
    unsigned char *base = (unsigned char *)(((uintptr_t)oz_raw + 1023) & ~(uintptr_t)1023);
    const int S = g.stages, BN = g.BN;
    const uint32_t BSL = (uint32_t)BN * OZ_KC * 2;            // bytes of one digit of B
    const uint32_t STAGE = OZ_ABYTES + OZ_S * BSL;
    double *outb = (double *)(base + (size_t)S * STAGE);
    uint64_t *bars = (uint64_t *)((unsigned char *)outb + OZ_OUTBYTES);
    // barriers: full[4] (a stage's digits landed), empty[4] (both issuers' MMAs done with it), rfull[8] /
    // rempty[8] (a level's group done / drained), fin[2]
    const uint32_t b_full = smem_u32(bars), b_empty = b_full + 32, b_rfull = b_empty + 32, b_rempty = b_rfull + 8 * OZ_S,
                   b_fin = b_rempty + 8 * OZ_S;
    uint32_t *tslot = (uint32_t *)(bars + 8 + 2 * OZ_S + 2);
    volatile int *abort_flag = (volatile int *)(tslot + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int s = 0; s < 4; ++s) {
            mbar_init(b_full + 8 * s, 1);
            mbar_init(b_empty + 8 * s, 2);
        }
        for (int r = 0; r < OZ_S; ++r) {
            mbar_init(b_rfull + 8 * r, 1);
            mbar_init(b_rempty + 8 * r, OZ_EPI_WARPS);
        }
        mbar_init(b_fin, 1);
        mbar_init(b_fin + 8, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (g.stall) {
        __syncthreads();
        tc_pdl_enter();
        if (tid == 0 && !mbar_wait(b_fin, 0u, abort_flag, g.wait_ns)) tc_report(g.err);
        __syncthreads();
        return;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(g.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tslot;
    tc_pdl_enter();   // everything above is this kernel's own
    auto fail = [&]() {
        if (!*abort_flag && g.err) tc_report(g.err);
        *abort_flag = 1;
    };
    const int ntn = g.ntn, nst = g.nst;

    if (warp >= OZ_EPI_WARPS) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(OZ_REG_AUX));
        if (warp == OZ_EPI_WARPS) {
            // ---- TMA producer -----------------------------------------------------------------------
            if (lane == 0) {
                int s = 0, issued = 0;
                uint32_t ph = 0;
                bool ok = true;
                for (int u = blockIdx.x; u < g.nunits && ok; u += gridDim.x) {
                    const int mt = u / ntn, nt = u - mt * ntn;
                    if (oz_frozen(g, mt)) continue;
                    for (int c = 0; c < nst; ++c) {
                        if (!mbar_wait(b_empty + 8 * s, ph ^ 1u, abort_flag, g.wait_ns)) { fail(); ok = false; break; }
                        const uint32_t sa = smem_u32(base + (size_t)s * STAGE);
                        mbar_expect_tx(b_full + 8 * s, STAGE);
                        tma_load_3d(sa, &tmA, c * OZ_KC, mt * OZ_BM, 0, b_full + 8 * s);
                        tma_load_3d(sa + OZ_ABYTES, &tmB, c * OZ_KC, nt * BN, 0, b_full + 8 * s);
                        ++issued;
                        if (++s == S) { s = 0; ph ^= 1u; }
                    }
                }
                // copies still in flight (only after an abort) finish before the CTA leaves
                for (int q = issued - 1; q >= 0 && q >= issued - S; --q)
                    mbar_wait(b_full + 8 * (q % S), (uint32_t)((q / S) & 1), nullptr, g.wait_ns);
            }
            __syncwarp();
        } else if (warp <= OZ_EPI_WARPS + 2) {
            // ---- MMA issuers: whole warps, one elected lane (see pf_tc.cuh) ---------------------------
            const int w = warp - (OZ_EPI_WARPS + 1);
            const uint32_t id_full = idesc_f16(OZ_BM, BN), id_last = idesc_f16(OZ_BM, g.BNlast);
            int s = 0;
            uint32_t ph = 0, gph = 1;   // stage phase; phase of the regions' drained barriers
            bool ok = true;
            for (int u = blockIdx.x; u < g.nunits && ok; u += gridDim.x) {
                const int mt = u / ntn, nt = u - mt * ntn;
                if (oz_frozen(g, mt)) continue;
                const uint32_t idesc = nt == ntn - 1 ? id_last : id_full;
                for (int c = 0; c < nst && ok; ++c) {
                    if (!mbar_wait_warp(b_full + 8 * s, ph, abort_flag, g.wait_ns)) { fail(); ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t sa = smem_u32(base + (size_t)s * STAGE);
                    const uint64_t da = sdesc_sw64(sa), db = sdesc_sw64(sa + OZ_ABYTES);
                    const bool two = g.K - c * OZ_KC > 16;   // the last stage may hold one 16-wide step only
                    const bool first = (c & (OZ_GRP - 1)) == 0, last = (c & (OZ_GRP - 1)) == OZ_GRP - 1 || c == nst - 1;
#pragma unroll
                    for (int d = OZ_S - 1; d >= 0; --d) {
                        const bool mine = (d == 7 || d == 6 || d == 2) ? w == 0 : w == 1;
                        if (!mine) continue;
                        if (first) {
                            if (!mbar_wait_warp(b_rempty + 8 * d, gph, abort_flag, g.wait_ns)) { fail(); ok = false; break; }
                            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        }
                        const uint32_t t = tmem + (uint32_t)(d * BN);
                        if (elect_one()) {
#pragma unroll
                            for (int x = 0; x <= d; ++x) {
                                const uint64_t a = da + (uint64_t)(x * ((OZ_BM * OZ_KC * 2) >> 4));
                                const uint64_t b = db + (uint64_t)((d - x) * (int)(BSL >> 4));
                                mma_f16(t, a, b, idesc, (x || !first) ? 1u : 0u);
                                if (two) mma_f16(t, a + 2, b + 2, idesc, 1u);   // the next 16 k: 32 bytes further
                            }
                            if (last) mma_commit(b_rfull + 8 * d);
                        }
                        __syncwarp();
                    }
                    if (!ok) break;
                    if (last) gph ^= 1u;
                    if (elect_one()) mma_commit(b_empty + 8 * s);
                    __syncwarp();
                    if (++s == S) { s = 0; ph ^= 1u; }
                }
            }
            // every MMA issued finishes before the tensor memory is released (also after an abort)
            __syncwarp();
            if (elect_one()) mma_commit(b_fin + 8 * w);
            mbar_wait(b_fin + 8 * w, 0u, nullptr, g.wait_ns);
            __syncwarp();
        }
    } else {
        // ---- drain, epilogue (warps 0-15) ------------------------------------------------------------------
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(OZ_REG_EPI));
        const int quarter = warp & 3, half = warp >> 2;   // 32 rows; which quarter of the columns
        long long acc[OZ_MAXH];
        uint32_t frac[OZ_MAXH / 4] = {};   // a byte per column
#pragma unroll
        for (int j = 0; j < OZ_MAXH; ++j) acc[j] = 0;
        uint32_t gph = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < g.nunits && (ok || !g.err); u += gridDim.x) {
            const int mt = u / ntn, nt = u - mt * ntn;
            if (oz_frozen(g, mt)) continue;
            const int hbn = (nt == ntn - 1 ? g.BNlast : BN) >> 2;   // columns per thread (8 or 16)
            const uint32_t lane0 = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * hbn);
            for (int c = 0; c < nst && ok; c += OZ_GRP, gph ^= 1u) {
                // levels 7 and 6 together: what they add to acc, and a byte of fraction that stays
                ok = mbar_wait(b_rfull + 8 * 7, gph, abort_flag, g.wait_ns) && mbar_wait(b_rfull + 8 * 6, gph, abort_flag, g.wait_ns);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int j0 = 0; j0 < OZ_MAXH; j0 += 8)
                    if (j0 < hbn) {
                        float lo[8], hi[8];
                        tmem_ld8(lane0 + (uint32_t)(7 * BN + j0), lo);
                        tmem_ld8(lane0 + (uint32_t)(6 * BN + j0), hi);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            uint32_t &f = frac[(j0 + j) >> 2];
                            const int sh = 8 * (j & 3), t = __float2int_rn(hi[j]) + ((__float2int_rn(lo[j]) + 128) >> 8) + (int)((f >> sh) & 0xFF);
                            acc[j0 + j] += t >> 8;
                            f = (f & ~(0xFFu << sh)) | ((uint32_t)(t & 0xFF) << sh);
                        }
                    }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(b_rempty + 8 * 7);
                    mbar_arrive(b_rempty + 8 * 6);
                }
#pragma unroll
                for (int d = 5; d >= 0; --d) {
                    if (!mbar_wait(b_rfull + 8 * d, gph, abort_flag, g.wait_ns)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t ta = lane0 + (uint32_t)(d * BN);
                    float v[OZ_MAXH];
                    tmem_ld8(ta, v);
                    if (hbn > 8) tmem_ld8(ta + 8u, v + 8);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(b_rempty + 8 * d);
#pragma unroll
                    for (int j0 = 0; j0 < OZ_MAXH; j0 += 8)
                        if (j0 < hbn) {
#pragma unroll
                            for (int j = j0; j < j0 + 8; ++j)   // integers
                                acc[j] += (long long)__float2int_rn(v[j]) * (1ll << (8 * (5 - d)));
                        }
                }
            }
            if (!ok) {
                fail();
                if (g.err) break;
            }
            // ---- epilogue: four columns per round, the rest moved down (a small loop: code is fetched at
            // about five cycles an instruction here) --------------------------------------------------
            const int m0 = mt * OZ_BM + quarter * 32, m = m0 + lane, nb = nt * BN + half * hbn;
            const int em = m < g.M ? g.E[m] : 1;
            const int p = m < g.M ? m / g.R : 0, rr = m < g.M ? m - p * g.R : 0;
            const int ncol = min(hbn, g.N - nb);
            const int fl = lane < ncol ? g.F[nb + lane] : 1;   // the exponents of the warp's columns, one per lane
            double *ob = outb + warp * (32 * OZ_OUTP);
            double *cb = g.C + ((long long)p * g.N + nb) * g.ldr + rr;   // store 1
            const bool nan = em == OZ_NONFINITE || !ok;
            // store 0: this lane's place in a round's block, rows 8 i + lane / 4, column lane % 4
            const int lr = lane >> 2, lc = lane & 3;
            int ro[4] = {-1, -1, -1, -1};   // the reciprocals of those rows at column lc (-1: none)
            if (g.rcp) {
                const int pl = p % g.cpl_mod, md = g.rcp_modes == 1 ? 0 : (pl == 1 ? g.cpl_mod / 2 : pl >> 1);
                const int q = m < g.M ? (md * g.R + rr) * g.N + nb : -1;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    ro[i] = __shfl_sync(0xffffffffu, q, 8 * i + lr);
                    if (ro[i] >= 0) ro[i] += lc;
                }
            }
#pragma unroll 1
            for (int j0 = 0; j0 < ncol; j0 += OZ_OUTC) {
                double v[OZ_OUTC];
                double2 rc[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {   // in flight during the conversions
                    rc[i] = double2{1.0, 0.0};
                    if (ro[i] >= 0 && j0 + lc < ncol) rc[i] = g.rcp[ro[i] + j0];
                }
#pragma unroll
                for (int j = 0; j < OZ_OUTC; ++j) {   // units 2^64 of X Y 2^(E + F - 2168)
                    const int fn = __shfl_sync(0xffffffffu, fl, j0 + j);
                    v[j] = oz_double(acc[j], (int)((frac[0] >> (8 * j)) & 0xFF), em + fn - 2168 + 64);
                    if (nan || fn == OZ_NONFINITE) v[j] = __longlong_as_double(0x7FF8000000000000ll);
                }
                if (g.store == 1) {             // lanes hold consecutive rows: coalesced as it is
#pragma unroll
                    for (int j = 0; j < OZ_OUTC; ++j, cb += g.ldr)
                        if (m < g.M && j0 + j < ncol) *cb = v[j];
                } else {                        // through shared memory: four lanes per row segment of 32 bytes
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < OZ_OUTC; ++j) ob[lane * OZ_OUTP + j] = v[j];
                    __syncwarp();
                    const int n = nb + j0 + lc;
                    const bool in = j0 + lc < ncol;
                    double *cr = g.C + (long long)(m0 + lr) * g.ldc + n;
                    const bool plain = !g.C2 && !(g.lamN && !g.rcp);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        v[i] = ob[(8 * i + lr) * OZ_OUTP + lc];
                        if (g.rcp) v[i] = oz_quot(v[i], rc[i]);
                    }
                    if (plain) {
#pragma unroll
                        for (int i = 0; i < 4; ++i, cr += 8 * (long long)g.ldc)
                            if (in && m0 + 8 * i + lr < g.M) *cr = v[i];
                    } else {
#pragma unroll 1
                        for (int i = 0; i < 4; ++i, cr += 8 * (long long)g.ldc) {
                            const int row = 8 * i + lr, mm = m0 + row;
                            const int pp = __shfl_sync(0xffffffffu, p, row), r2 = __shfl_sync(0xffffffffu, rr, row);
                            double x = v[0];
#pragma unroll
                            for (int q = 0; q < 3; ++q) v[q] = v[q + 1];
                            if (in && mm < g.M) {
                                if (g.lamN && !g.rcp) {
                                    const double dd = g.lamN[n] + g.lamR[r2] + g.cpl[pp % g.cpl_mod];
                                    x = (dd != 0.0) ? x / dd : 0.0;
                                }
                                *cr = x;
                                if (g.C2) {
                                    double w2 = -g.m2x[n] * g.m2y[r2] * x;
                                    if (g.face2 && r2 == 0) w2 += g.face2[(long long)pp * g.N + n];
                                    g.C2[(long long)mm * g.ldc + n] = w2;
                                }
                            }
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j + OZ_OUTC < OZ_MAXH; ++j) acc[j] = acc[j + OZ_OUTC];
#pragma unroll
                for (int j = 0; j + 1 < OZ_MAXH / 4; ++j) frac[j] = frac[j + 1];
            }
#pragma unroll
            for (int j = 0; j < OZ_MAXH; ++j) acc[j] = 0;
#pragma unroll
            for (int j = 0; j < OZ_MAXH / 4; ++j) frac[j] = 0;
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(g.tmem_cols) : "memory");
    }
}
#endif  // PF_OZ_HELPERS_ONLY

}  // namespace pf
