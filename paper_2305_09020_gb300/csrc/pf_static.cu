// Allocation-free variant of the fast-diagonalisation solve (FP64).
//
// Some callers cannot allocate device memory at the point where they need a solve:
// code running inside a region that forbids or cannot afford cudaMalloc (it may
// synchronise the device), a memory-planned real-time loop, or a host library that
// brings its own allocator and must not see a second one.  For them,
// pf_fdm_solve_static takes every input and output as a caller-owned device pointer
// and keeps its two intermediate buffers in the file-scope array below, which every
// GPU that loads this library holds until the process exits.
#include <cuda_runtime.h>

#include <mutex>
#include <string>

#include "../../include/pf.h"
#include "pf_kernels.cuh"
#define PF_TC_HELPERS_ONLY
#include "pf_oz.cuh"

void pf_internal_set_error(const std::string &msg);   // pf_api.cu: message for pf_last_error(NULL)

namespace {

// Two scratch planes sets of PF_STATIC_MAX_VALUES doubles each (16 MiB in total).
static __device__ __align__(256) double g_fdm_scratch[2 * PF_STATIC_MAX_VALUES];

// Digits of the right-hand sides and of the four eigenbases for the tensor-core transforms
// (pf_oz.cuh), 49 MB in all: planes whose padded rows fit take those, others the FMA kernel.
constexpr size_t DIG_A = (size_t)pf::OZ_S << 21, DIG_B = (size_t)pf::OZ_S * pf::OZ_MAXK * pf::OZ_MAXK;
constexpr int DIG_ROWS = 1 << 16, DIG_MIN = 16;   // n_x, n_y >= 16: at most 2^16 rows of 2^20 values
struct Digits {
    __half a[DIG_A], b[4][DIG_B];
    int E[DIG_ROWS], F[4][pf::OZ_MAXK], sh[4][pf::OZ_MAXK], sparse;
};
static __device__ __align__(256) unsigned char g_fdm_digits[sizeof(Digits)];

std::mutex g_mu;
double *g_scratch_ptr[64] = {nullptr};   // device address of g_fdm_scratch, per device
Digits *g_digits_ptr[64] = {nullptr};    // device address of g_fdm_digits, per device
int g_sms[64] = {0};

// Device address of the scratch array on the current device, looked up once per device.
// Host code must not pass the symbol itself to a kernel: on the host it only names a
// stand-in object, not device memory.
int scratch_for_current_device(double **out, Digits **digits, int *sms) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        pf_internal_set_error(std::string("cudaGetDevice: ") + cudaGetErrorString(e));
        return PF_ECUDA;
    }
    if (dev < 0 || dev >= 64) {
        pf_internal_set_error("device index out of range for the static scratch table");
        return PF_EINVAL;
    }
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_scratch_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_fdm_scratch);
        if (e != cudaSuccess || !p) {
            pf_internal_set_error(std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
            return PF_ECUDA;
        }
        void *q = nullptr;
        int n = 0;
        e = cudaGetSymbolAddress(&q, g_fdm_digits);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute((const void *)pf::k_gemm_oz, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pf::OZ_SMEM);
        if (e != cudaSuccess) {
            pf_internal_set_error(std::string("digit scratch: ") + cudaGetErrorString(e));
            return PF_ECUDA;
        }
        g_digits_ptr[dev] = static_cast<Digits *>(q);
        g_sms[dev] = n;
        g_scratch_ptr[dev] = static_cast<double *>(p);
    }
    *out = g_scratch_ptr[dev];
    *digits = g_digits_ptr[dev];
    *sms = g_sms[dev];
    return PF_OK;
}

int launch_gemm(const double *A, const double *B, double *C, long long rows, int n, int R, int store,
                const double *lamN, const double *lamR, const double *cpl, int cpl_mod, cudaStream_t st,
                const int *only_if = nullptr) {
    pf::GemmArgs<double> g{A, B, C, rows, n, R, store, lamN, lamR, cpl, cpl_mod};
    g.only_if = only_if;
    dim3 grid((n + 63) / 64, (unsigned)((rows + 63) / 64));
    pf::k_gemm<double, 64, 64, 8, 4, 4><<<grid, 256, 0, st>>>(g);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        pf_internal_set_error(std::string("k_gemm launch: ") + cudaGetErrorString(e));
        return PF_ECUDA;
    }
    return PF_OK;
}

// C = A B through the digits of A and of B's transpose (b: which of the four eigenbases)
int launch_digits(Digits *D, int sms, const double *A, int b, double *C, long long rows, int n, int R, int store,
                  const double *lamN, const double *lamR, const double *cpl, int cpl_mod, cudaStream_t st) {
    size_t smem = 0;
    pf::OzArgs a = pf::oz_plan(rows, n, sms, &smem);
    a.E = D->E; a.F = D->F[b]; a.skip_if = &D->sparse;
    a.R = R; a.store = store; a.ldc = n; a.ldr = R;
    a.lamN = lamN; a.lamR = lamR; a.cpl = cpl; a.cpl_mod = cpl_mod;
    a.C = C;
    a.wait_ns = 1000000000ull;
    CUtensorMap ma, mb;
    if (!pf::oz_encode(&ma, D->a, rows, pf::oz_kpad(n), pf::OZ_BM) || !pf::oz_encode(&mb, D->b[b], n, pf::oz_kpad(n), a.BN)) {
        pf_internal_set_error("cuTensorMapEncodeTiled failed");
        return PF_ECUDA;
    }
    pf::oz_split(A, (int)rows, n, D->sh[b], D->a, D->E, R, nullptr, 1, st, false, &D->sparse);
    pf::k_gemm_oz<<<(unsigned)(a.nunits < sms ? a.nunits : sms), pf::OZ_THREADS, smem, st>>>(ma, mb, a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        pf_internal_set_error(std::string("k_gemm_oz launch: ") + cudaGetErrorString(e));
        return PF_ECUDA;
    }
    return PF_OK;
}

// The tensor-core transforms take ten launches (the eigenbases are split anew in each call: they
// are the caller's) and the four of the FMA kernels, which return at once unless a basis falls into uncoupled
// pieces, and are the faster ones from the smallest planes measured on (FMA kernels alone / these): 16 x 17 nodes,
// one plane 124 / 95 us; 32 x 17 158 / 101; 128 x 65, one plane 462 / 123, 64 planes 620 / 160; 240 x 145, 30 planes
// 1977 / 218.  A basis of uncoupled pieces pays 35 to 50 us for the launches that return at once.
bool digits_fit(int nx, int ny, long long total) {
    if (nx < DIG_MIN || ny < DIG_MIN || nx > pf::OZ_MAXK || ny > pf::OZ_MAXK || pf::tc_encode() == nullptr) return false;
    const long long P = total / ((long long)nx * ny);
    return P * ny * pf::oz_kpad(nx) <= (1ll << 21) && P * nx * pf::oz_kpad(ny) <= (1ll << 21);
}

}  // namespace

extern "C" int pf_fdm_solve_static(int nx, int ny, int nplanes, const double *Sx, const double *SxT,
                                   const double *lam_x, const double *Sy, const double *SyT,
                                   const double *lam_y, const double *shift, const double *rhs, double *out,
                                   void *cuda_stream) {
    if (nx < 1 || ny < 1 || nplanes < 1 || !Sx || !SxT || !lam_x || !Sy || !SyT || !lam_y || !shift || !rhs ||
        !out) {
        pf_internal_set_error("pf_fdm_solve_static: null pointer or non-positive size");
        return PF_EINVAL;
    }
    const long long total = (long long)nx * ny * nplanes;
    if (total > PF_STATIC_MAX_VALUES) {
        pf_internal_set_error("pf_fdm_solve_static: nx*ny*nplanes exceeds PF_STATIC_MAX_VALUES");
        return PF_EINVAL;
    }
    double *scratch = nullptr;
    Digits *D = nullptr;
    int sms = 0;
    int rc = scratch_for_current_device(&scratch, &D, &sms);
    if (rc != PF_OK) return rc;
    double *W1 = scratch, *W2 = scratch + PF_STATIC_MAX_VALUES;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const long long P = nplanes;
    const int *fma = nullptr;
    if (digits_fit(nx, ny, total)) {
        // shifts and digits of each eigenbasis by columns
        pf::OzBases g{{Sx, Sy, SyT, SxT}, {nx, ny, ny, nx}, {}, {}, {}, &D->sparse};
        for (int b = 0; b < 4; ++b) g.sh[b] = D->sh[b], g.dig[b] = D->b[b], g.F[b] = D->F[b];
        pf::oz_split_bases(g, st);
        if ((rc = launch_digits(D, sms, rhs, 0, W1, P * ny, nx, ny, 1, nullptr, nullptr, nullptr, 1, st)) != PF_OK) return rc;
        if ((rc = launch_digits(D, sms, W1, 1, W2, P * nx, ny, nx, 0, lam_y, lam_x, shift, nplanes, st)) != PF_OK) return rc;
        if ((rc = launch_digits(D, sms, W2, 2, W1, P * nx, ny, nx, 1, nullptr, nullptr, nullptr, 1, st)) != PF_OK) return rc;
        if ((rc = launch_digits(D, sms, W1, 3, out, P * ny, nx, ny, 0, nullptr, nullptr, nullptr, 1, st)) != PF_OK) return rc;
        fma = &D->sparse;   // the kernels below run only where a basis falls into uncoupled pieces
    }
    // the same four transforms as the handle's solves: x, y (+ eigenvalue division), y^T, x^T
    if ((rc = launch_gemm(rhs, Sx, W1, P * ny, nx, ny, 1, nullptr, nullptr, nullptr, 1, st, fma)) != PF_OK) return rc;
    if ((rc = launch_gemm(W1, Sy, W2, P * nx, ny, nx, 0, lam_y, lam_x, shift, nplanes, st, fma)) != PF_OK) return rc;
    if ((rc = launch_gemm(W2, SyT, W1, P * nx, ny, nx, 1, nullptr, nullptr, nullptr, 1, st, fma)) != PF_OK) return rc;
    return launch_gemm(W1, SxT, out, P * ny, nx, ny, 0, nullptr, nullptr, nullptr, 1, st, fma);
}
