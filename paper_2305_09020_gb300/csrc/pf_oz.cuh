// FP64 transform GEMM on the tensor cores (tcgen05 kind::f16, sm_103a): exact products of 8-bit digits.
//
// C[M x N] = A[M x K] * B[K x N] for the constant eigenbasis products of the Remark after Algorithm 2 in
// double precision.  The FP64 pipe of the GB300 runs 2 FMA per SM and cycle (1.1 TFLOP/s measured), the
// tensor cores 4096 FP16 products, and small integers multiply and add exactly there.  So each operand
// is written in fixed point (the integer splitting of Ozaki, Ogita, Oishi and Rump for matrix units):
//   row m of A:     a = X 2^(E_m - 1077),  X = rint(a 2^(1077 - E_m)), |X| < 2^55,
//                   E_m the largest biased exponent of the row,
//   column n of B:  b = Y 2^(F_n - 1077), the same (split once on the host),
//   X = sum_s x_s 256^(6-s), seven balanced digits -128 <= x_s <= 128, stored as FP16 integers.
// X Y summed over k is sum_d 256^(12-d) v_d with the level sums v_d = sum_{s+t=d} sum_k x_s y_t.  Levels
// 0..6 (28 digit products) are kept: the first dropped level is 2^-56 of a product of two row maxima.
// Over a group of 128 k every level sum is an integer of at most 7 * 128 * 2^14 < 2^24, so the tensor core's
// FP32 accumulation is exact.  The drain of a group adds v_d, in units of 256^7, into 64-bit integers:
//   acc += v_0 2^40 + v_1 2^32 + v_2 2^24 + v_3 2^16 + v_4 2^8 + v_5 + rint(v_6 / 256),
// which also is exact but for v_6 and stays below 2^63 for K < 512.  The result is rounded to double once.
// Against FMA chains, whose rounding grows with K, the error is smaller.
//
// A row of A or a column of B with an infinity or NaN gives NaN results; other rows and columns are not
// affected.  Subnormal entries keep their bits; results are rounded to nearest, ties to even.
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "pf_tc.cuh"

namespace pf {

constexpr int OZ_S = 7;                       // digits per operand
constexpr int OZ_KC = 32;                     // K per stage: 64-byte rows of FP16
constexpr int OZ_BM = 128;                    // rows per unit = TMEM lanes
constexpr int OZ_MAXH = 16;                   // accumulator columns per drain thread: BN <= 64
constexpr int OZ_GRP = 4;                     // stages per accumulation group (128 k)
constexpr int OZ_MAXK = 480;                  // K bound of the 64-bit sums (< 512)
constexpr int OZ_EPI_WARPS = 16;              // four warpgroups: a quarter of the columns each
constexpr int OZ_THREADS = 640;
// the launch holds 640 x 96 = 61440 registers: 512 x 104 + 128 x 64 = 61440
constexpr int OZ_REG_EPI = 104, OZ_REG_AUX = 64;
static_assert(512 * OZ_REG_EPI + 128 * OZ_REG_AUX <= OZ_THREADS * 96, "the setmaxnreg split must fit the launch's registers");
constexpr uint32_t OZ_ABYTES = OZ_S * OZ_BM * OZ_KC * 2;   // A digits of a stage
constexpr int OZ_OUTC = 4, OZ_OUTP = 5;       // columns and row pitch (doubles) of a drain warp's store block
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
    const double *rcp;        // its reciprocals [mode][r][n], mode of plane p: 0 when rcp_modes == 1, else
    int rcp_modes;            // that of the packed Fourier plane p % cpl_mod; null: divide
    double *C;
    double *C2;               // optional C2[m ldc + n] = -m2x[n] m2y[r] C (+ face2[p N + n] on r == 0)
    const double *m2x, *m2y, *face2;
    const int *active;        // ensembles: per-run flags (0 = frozen), run = p % amod; null otherwise
    int amod;
    int *err;                 // error word; null: a call without one, whose results become NaN on a time-out
    unsigned long long wait_ns;
};

constexpr size_t OZ_SMEM = 227 * 1024;
inline int oz_kpad(int k) { return (k + OZ_KC - 1) / OZ_KC * OZ_KC; }

// sizes of the product of `rows` rows with an N x N matrix: column tiles, stages, shared memory.  Column
// tiles: enough units for the chip, against the cycles of a unit: 56 MMAs a stage of 40 + BN/4 cycles and
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
        const double t = rounds * (a.nst * (56.0 * (40.0 + 0.25 * bn)) + 6000.0 + 130.0 * bn);
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

// digit planes [OZ_S][rows][Kpad], boxes of 32 x box_rows x 7
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

// biased fixed point of a against the row exponent emax (>= a's): X + 128 (256^6 + .. + 1), so that byte s
// from the top (16 bits for s = 0) is digit x_s + 128
__host__ __device__ __forceinline__ unsigned long long oz_fixed(unsigned long long bits, int emax) {
    const int e = (int)(bits >> 52) & 0x7FF;
    unsigned long long m = bits & 0xFFFFFFFFFFFFFull;
    if (e) m |= 1ull << 52;
    int r = emax - (e ? e : 1);
    if (r > 60) r = 60;
    m = (((m << 3) >> r) + 1) >> 1;
    const unsigned long long s = 0ull - (bits >> 63);
    return ((m ^ s) - s) + 0x0080808080808080ull;
}

// v 2^sc rounded to nearest even: one conversion, the power of two added to its exponent (normalising by
// integer operations instead took about thirty: 1 to 3% of a step)
__device__ __forceinline__ double oz_double(long long v, int sc) {
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

#ifndef PF_OZ_HELPERS_ONLY
// ---- digits of A: one warp per row ----------------------------------------------------------------
// dig[d][m][Kpad] (FP16), E[m], of the rows A[m rs + k ks].  Bound by its 8 bytes read and 14 written per value, most of them in L2;
// a pass of its own because inside the GEMM every column tile would split the rows again (measured there:
// 7,000 issue slots per 128 x 32 stage against 3,100 cycles of MMAs).  NI = ceil(Kpad / 64) pairs a lane.
template <int NI>
__global__ void __launch_bounds__(256) k_oz_split(const double *__restrict__ A, long long rs, int ks, int M, int K, int Kpad,
                                                  __half *__restrict__ dig, int *__restrict__ E, int R, const int *__restrict__ active, int amod) {
    const int m = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    tc_pdl_enter();
    if (m >= M) return;
    if (active && !active[(m / R) % amod]) return;   // a frozen run's rows: their products are not used
    const double *row = A + m * rs;
    double x[NI][2];
    unsigned int e = 0;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int k = 2 * (lane + 32 * i);
        x[i][0] = k < K ? row[(long long)k * ks] : 0.0;
        x[i][1] = k + 1 < K ? row[(long long)(k + 1) * ks] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < NI; ++i)
        e = max(e, max((unsigned int)__double2hiint(x[i][0]) & 0x7FF00000u, (unsigned int)__double2hiint(x[i][1]) & 0x7FF00000u));
    const int em = max((int)(__reduce_max_sync(0xffffffffu, e) >> 20), 1);
    if (lane == 0) E[m] = em;
    const long long DS = (long long)M * Kpad / 2;     // words per digit plane
    uint32_t *dst = reinterpret_cast<uint32_t *>(dig) + (long long)m * (Kpad / 2) + lane;
    const __half2 bias = __half2half2(__ushort_as_half(0x6480));   // 1152
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        if (2 * (lane + 32 * i) >= Kpad) break;
        const unsigned long long ua = oz_fixed((unsigned long long)__double_as_longlong(x[i][0]), em);
        const unsigned long long ub = oz_fixed((unsigned long long)__double_as_longlong(x[i][1]), em);
        const uint32_t al = (uint32_t)ua, ah = (uint32_t)(ua >> 32), bl = (uint32_t)ub, bh = (uint32_t)(ub >> 32);
        auto put = [&](int d, uint32_t v) {   // v: two FP16 words 1024 + digit + 128
            const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&v), bias);
            dst[d * DS + 32 * i] = *reinterpret_cast<const uint32_t *>(&h);
        };
        put(0, __byte_perm(ah, bh, 0x7632) + 0x64006400u);
        put(1, (__byte_perm(ah, bh, 0x0501) & 0x00FF00FFu) | 0x64006400u);
        put(2, (__byte_perm(ah, bh, 0x0400) & 0x00FF00FFu) | 0x64006400u);
        put(3, (__byte_perm(al, bl, 0x0703) & 0x00FF00FFu) | 0x64006400u);
        put(4, (__byte_perm(al, bl, 0x0602) & 0x00FF00FFu) | 0x64006400u);
        put(5, (__byte_perm(al, bl, 0x0501) & 0x00FF00FFu) | 0x64006400u);
        put(6, (__byte_perm(al, bl, 0x0400) & 0x00FF00FFu) | 0x64006400u);
    }
}

// launch of k_oz_split for M rows of K <= OZ_MAXK values: row pitch rs, value pitch ks (1, n for the rows and
// columns of an n x n matrix); pdl: as a programmatic dependent launch
inline void oz_split(const double *A, long long rs, int ks, int M, int K, __half *dig, int *E, int R, const int *active, int amod,
                     cudaStream_t st, bool pdl = false) {
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
    auto go = [&](void (*k)(const double *, long long, int, int, int, int, __half *, int *, int, const int *, int)) {
        cudaLaunchKernelEx(&cfg, k, A, rs, ks, M, K, Kpad, dig, E, R, active, amod);   // errors: the caller's cudaGetLastError
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

// reciprocals of the eigenvalue sums of one solve family, [mode][r][n] (0 where a sum is 0)
static __global__ void k_oz_rcp(double *__restrict__ out, const double *__restrict__ lamN, const double *__restrict__ lamR,
                                const double *__restrict__ shift, int modes, int nz, int R, int N) {
    const long long n = (long long)modes * R * N;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(i / ((long long)R * N));
        const int r = (int)(i / N - (long long)k * R), c = (int)(i % N);
        const int p = modes == 1 ? 0 : k == 0 ? 0 : (k == nz / 2 ? 1 : 2 * k);   // a packed plane of mode k
        const double d = lamN[c] + lamR[r] + shift[p];
        out[i] = d != 0.0 ? 1.0 / d : 0.0;
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
//   warp 16     TMA: per 32-wide K stage the digits of A (32 x 128 x 7) and of B (32 x BN x 7), one 3D box each
//   warps 17-18 issue the MMAs level by level (6 first), each level into a tensor-memory region of its own
//               that it accumulates over a group of four stages: levels 6, 3, 2 by one warp, 5, 4, 1, 0 by
//               the other, 28 MMAs of a stage each.  The drain of a level overlaps the group's later
//               levels and the next group's first stage
//   warps 0-15  drain the regions into the 64-bit integers, then convert and store (the epilogues of
//               k_gemm).  Sixteen, because this code overflows the schedulers' instruction caches and its
//               fetches are shared by a scheduler's warps
// setmaxnreg moves registers from warps 16-19 to the drain warps.  Every mbarrier wait is bounded as in
// pf_tc.cuh: on time-out the error word is set, copies and MMAs in flight finish (bounded), tensor memory
// is freed and the kernel returns.
static __global__ void __launch_bounds__(OZ_THREADS, 1) k_gemm_oz(const __grid_constant__ CUtensorMap tmA,
                                                                  const __grid_constant__ CUtensorMap tmB, OzArgs g) {
    extern __shared__ __align__(1024) unsigned char oz_raw[];
    unsigned char *base = (unsigned char *)(((uintptr_t)oz_raw + 1023) & ~(uintptr_t)1023);
    const int S = g.stages, BN = g.BN;
    const uint32_t BSL = (uint32_t)BN * OZ_KC * 2;            // bytes of one digit of B
    const uint32_t STAGE = OZ_ABYTES + OZ_S * BSL;
    double *outb = (double *)(base + (size_t)S * STAGE);
    uint64_t *bars = (uint64_t *)((unsigned char *)outb + OZ_OUTBYTES);
    // barriers: full[4] (a stage's digits landed), empty[4] (both issuers' MMAs done with it), rfull[7] /
    // rempty[7] (a level's group done / drained), fin[2]
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
        if (!*abort_flag && g.err) atomicExch(g.err, TC_ERR_TIMEOUT);
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
                        const bool mine = (d == 6 || d == 3 || d == 2) ? w == 0 : w == 1;
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
        // ---- drain, epilogue (warps 0-7) ------------------------------------------------------------------
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(OZ_REG_EPI));
        const int quarter = warp & 3, half = warp >> 2;   // 32 rows; which quarter of the columns
        long long acc[OZ_MAXH];
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
#pragma unroll
                for (int d = OZ_S - 1; d >= 0; --d) {
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
                            for (int j = j0; j < j0 + 8; ++j) {
                                const int w = __float2int_rn(v[j]);   // an integer
                                if (d == 6) acc[j] += (long long)((w + 128) >> 8);
                                else acc[j] += (long long)w * (1ll << (8 * (5 - d)));
                            }
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
            const bool nan = em == 0x7FF || !ok;
            // store 0: this lane's place in a round's block, rows 8 i + lane / 4, column lane % 4
            const int lr = lane >> 2, lc = lane & 3;
            const double *rp[4] = {nullptr, nullptr, nullptr, nullptr};   // the reciprocals' rows
            double rc[4] = {1.0, 1.0, 1.0, 1.0};
            if (g.rcp) {
                const int pl = p % g.cpl_mod, md = g.rcp_modes == 1 ? 0 : (pl == 1 ? g.cpl_mod / 2 : pl >> 1);
                const int q = m < g.M ? md * g.R + rr : -1;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int row = __shfl_sync(0xffffffffu, q, 8 * i + lr);
                    if (row >= 0) {
                        rp[i] = g.rcp + (long long)row * g.N + nb + lc;
                        if (lc < ncol) rc[i] = *rp[i];
                    }
                }
            }
#pragma unroll 1
            for (int j0 = 0; j0 < ncol; j0 += OZ_OUTC) {
                double v[OZ_OUTC], rn[4] = {1.0, 1.0, 1.0, 1.0};
                if (g.rcp) {   // the next round's reciprocals in flight during this one
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (rp[i] && j0 + OZ_OUTC + lc < ncol) rn[i] = rp[i][j0 + OZ_OUTC];
                }
#pragma unroll
                for (int j = 0; j < OZ_OUTC; ++j) {   // units 2^56 of X Y 2^(E + F - 2154)
                    const int fn = __shfl_sync(0xffffffffu, fl, j0 + j);
                    v[j] = oz_double(acc[j], em + fn - 2154 + 56);
                    if (nan || fn == 0x7FF) v[j] = __longlong_as_double(0x7FF8000000000000ll);
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
                        if (g.rcp) v[i] *= rc[i];
                        rc[i] = rn[i];
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
            }
#pragma unroll
            for (int j = 0; j < OZ_MAXH; ++j) acc[j] = 0;
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
