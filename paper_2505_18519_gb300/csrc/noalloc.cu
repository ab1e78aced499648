// Local energies and force-bias values of a batch of (walker, trial sample)
// pairs with no device allocation at all: the intermediate matrices and
// per-spin log-determinants live in file-scope device arrays instead of a
// caller-provided workspace.
//
// Some callers cannot call cudaMalloc or hand the library a workspace: code
// embedded in another framework's custom-operator hook, where device memory may
// only come from that framework's own pool, and latency-critical loops where an
// allocation (which can synchronise the device) is not allowed.  They pass only
// their inputs and outputs.
//
// The arrays are shared by every call in the process, on every device that loads
// them, and keep the last call's contents.  Only the status word must
// start at zero, and each call clears it; every other element a call reads is
// first written by that same call.  Calls that overlap on the GPU (other
// streams, other host threads, the same device) race on them.
//
// The contraction runs as integer digit products on the tensor cores
// (contract_fp64d: the FP64 accuracy of the FP64 kernel) when the digits of h and L,
// formed again by every call, and the work of one walker fit the second array (noalloc_work.cu), else (for the
// smallest systems, and where the GPU had no room for that array at its first call) as the FP64 kernel.  On one GB300: 1024 pairs of 50
// orbitals, 32 per walker, 1.71 ms against 30.9 (1 per walker 11.7 against 30.9), one pair 0.34
// against 4.7; 150 pairs of 120 orbitals 7.5 against 116; 8 orbitals with 32 matrices, one pair 0.14 against
// 0.21; with 16 matrices, 32 pairs 0.120 against 0.111.
#include <stdio.h>

#include <algorithm>
#include <mutex>

#include "kernels.cuh"

using namespace afq;

// 32 MiB of scratch, resident on every GPU that loads the library until exit.
static constexpr size_t kNoallocScratchBytes = 32ull << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocScratchBytes];

static std::mutex g_noalloc_mu;
static void* g_noalloc_addr[256];        // device addresses of the arrays, per device ordinal
static void* g_noalloc_work_addr[256];   // null: no room for the digits' work space at the first call

// Bytes of the work space that hold the walkers worked on together, 0 where the sizes do not fit.
static size_t digit_chunk(const Dims& d) {
    const size_t least = contract_fp64d_work_bytes(d.N, d.nu, d.nd, d.G, d.W, d.P, 0);
    if (least == 0 || least > NOALLOC_WORK_BYTES) return 0;
    size_t chunk = NOALLOC_WORK_BYTES - least + 1;
    while (contract_fp64d_work_bytes(d.N, d.nu, d.nd, d.G, d.W, d.P, chunk) > NOALLOC_WORK_BYTES) chunk -= chunk / 8 + 1;
    return std::max<size_t>(chunk, 1);   // a chunk of one byte is one walker
}

static thread_local char g_noalloc_err[256] = "";
static thread_local uint32_t g_noalloc_polls = 0;   // limit of the calling thread's waits, 0: the default

// log<Phi|phi> of the pairs, and NaN in every output if a wait of the digit products ran out: nobody reads
// the status word, and what the kernels left out would be the values of an earlier call.
static __global__ void noalloc_finish_kernel(long long pairs, int G, const int* __restrict__ status,
                                             const double2* __restrict__ logdet, double2* __restrict__ logov,
                                             double2* __restrict__ e_local, double2* __restrict__ force_bias) {
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= pairs) return;
    if (!(*status & STATUS_TIMEOUT)) {
        logov[p] = cadd(logdet[2 * p], logdet[2 * p + 1]);
        return;
    }
    const double nan = __longlong_as_double(0x7FF8000000000000LL);
    logov[p] = e_local[p] = cmk(nan, nan);
    for (int g = 0; g < G; ++g) force_bias[p * G + g] = cmk(nan, nan);
}

static afqmc_status noalloc_fail(afqmc_status st, const char* msg, cudaError_t e = cudaSuccess) {
    if (e != cudaSuccess)
        snprintf(g_noalloc_err, sizeof g_noalloc_err, "%s: %s", msg, cudaGetErrorString(e));
    else
        snprintf(g_noalloc_err, sizeof g_noalloc_err, "%s", msg);
    return st;
}

extern "C" const char* afqmc_noalloc_last_error(void) { return g_noalloc_err; }

extern "C" size_t afqmc_noalloc_scratch_bytes(void) { return kNoallocScratchBytes; }

extern "C" afqmc_status afqmc_noalloc_wait_polls(int64_t polls) {
    if (polls < 0 || polls > (1ll << 31)) return noalloc_fail(AFQMC_ERR_ARG, "polls must be in [0, 2^31]");
    g_noalloc_polls = (uint32_t)polls;
    return AFQMC_OK;
}

extern "C" afqmc_status afqmc_local_energy_noalloc(int N, int n_up, int n_dn, int n_chol, int64_t n_pairs,
                                                   int pairs_per_walker, const double* h, const double* L,
                                                   const double* Phi, const double* phi, double* logov,
                                                   double* e_local, double* force_bias, void* stream) {
    if (N < 1 || N > 256 || n_up < 1 || n_up > N || n_up > 64 || n_dn < 0 || n_dn > n_up || n_chol < 1 ||
        n_pairs < 0 || pairs_per_walker < 1)
        return noalloc_fail(AFQMC_ERR_ARG, "invalid sizes");
    if (!h || !L || !Phi || !phi || !logov || !e_local || !force_bias)
        return noalloc_fail(AFQMC_ERR_ARG, "every array must be a device pointer (none may be NULL)");
    if (!contract_fp64_supported(N, n_up, n_dn))
        return noalloc_fail(AFQMC_ERR_ARG, "sizes too large for the FP64 contraction kernel");
    const int nt = n_up + n_dn;
    // Bound n_pairs before any product with it, so that no size below can wrap: every
    // pair takes N nt complex Theta entries and two complex log-determinants, and the
    // layout adds at most 255 bytes of alignment and the status word.
    const size_t per_pair = (size_t)N * nt * sizeof(double2) + 2 * sizeof(double2);
    const size_t fixed = 256 + sizeof(int);
    if (n_pairs > 0 && (uint64_t)n_pairs > (kNoallocScratchBytes - fixed) / per_pair) {
        snprintf(g_noalloc_err, sizeof g_noalloc_err,
                 "batch of %lld pairs needs more scratch than the fixed maximum of %zu bytes "
                 "(about n_pairs * (N * (n_up + n_dn) * 16 + 32)); split the batch",
                 (long long)n_pairs, kNoallocScratchBytes);
        return AFQMC_ERR_ARG;
    }
    if ((n_pairs + pairs_per_walker - 1) / pairs_per_walker > INT32_MAX)
        return noalloc_fail(AFQMC_ERR_ARG, "too many walkers in the batch");
    const size_t theta_bytes = (size_t)n_pairs * N * nt * sizeof(double2);
    const size_t logdet_off = (theta_bytes + 255) & ~(size_t)255;
    const size_t status_off = logdet_off + (size_t)n_pairs * 2 * sizeof(double2);
    if (n_pairs == 0) return AFQMC_OK;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return noalloc_fail(AFQMC_ERR_CUDA, "cudaGetDevice", e);
    if (dev < 0 || dev >= 256) return noalloc_fail(AFQMC_ERR_ARG, "device ordinal out of range");
    void *base = nullptr, *work = nullptr;
    {
        // Set-up, once per device, with that device current: the host-side name
        // of the array is not a device address, so ask the runtime for it.  The
        // address belongs to the device's primary context (the one the runtime
        // API uses); it is cached for the life of the process, so neither another
        // driver-API context made current nor a cudaDeviceReset after this first
        // call is supported.
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!g_noalloc_addr[dev]) {
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess) return noalloc_fail(AFQMC_ERR_CUDA, "cudaGetSymbolAddress", e);
            void* q = nullptr;
            e = noalloc_work(&q);
            if (e != cudaSuccess) {
                cudaGetLastError();
                if (e != cudaErrorMemoryAllocation) return noalloc_fail(AFQMC_ERR_CUDA, "cudaGetSymbolAddress", e);
                q = nullptr;
            }
            g_noalloc_work_addr[dev] = q;
            g_noalloc_addr[dev] = p;
        }
        base = g_noalloc_addr[dev];
        work = g_noalloc_work_addr[dev];
    }
    double2* Theta = reinterpret_cast<double2*>(base);
    double2* logdet = reinterpret_cast<double2*>(static_cast<char*>(base) + logdet_off);
    cudaStream_t s = (cudaStream_t)stream;
    Dims d{};   // value-initialised: launch shapes at their defaults
    d.N = N; d.nu = n_up; d.nd = n_dn; d.nt = nt; d.G = n_chol; d.K = 1;
    d.P = pairs_per_walker;
    d.W = (int)((n_pairs + pairs_per_walker - 1) / pairs_per_walker);
    d.pairs = n_pairs;
    if (g_noalloc_polls) d.wait_polls = g_noalloc_polls;
    // the overlap kernel flags singular overlaps in a status word, which lives in
    // the scratch too and is cleared first (a singular pair gets log|ov| = -inf)
    int* status = reinterpret_cast<int*>(static_cast<char*>(base) + status_off);
    e = cudaMemsetAsync(status, 0, sizeof(int), s);
    if (e != cudaSuccess) return noalloc_fail(AFQMC_ERR_CUDA, "clearing the status word", e);
    // whole walkers, then a last one with fewer pairs, which the digit products take as a batch of its own
    Dims part[2] = {d, d};
    part[0].W = (int)(n_pairs / pairs_per_walker);
    part[0].pairs = (long long)part[0].W * pairs_per_walker;
    part[1].W = part[0].W < d.W;
    part[1].P = std::max(1, (int)(n_pairs - part[0].pairs));
    part[1].pairs = n_pairs - part[0].pairs;
    // by the sizes of the system and the pairs per walker alone, so that part of a batch gives the bits of the whole:
    // a walker of as many pairs as the scratch takes has to fit, and fewer then do
    Dims full = d;
    full.W = 1;
    full.P = (int)std::min<size_t>(pairs_per_walker, (kNoallocScratchBytes - fixed) / per_pair);
    full.pairs = full.P;
    bool digits = work && (long long)N * n_chol > 128 && full.P > 0 && digit_chunk(full) > 0;
    size_t chunk[2] = {0, 0};
    for (int q = 0; q < 2; ++q)
        if (digits && part[q].W) digits = (chunk[q] = digit_chunk(part[q])) > 0;
    for (int spin = 0; spin < 2; ++spin) {
        e = overlap_lu(s, d, spin, Phi, (long long)N * n_up, reinterpret_cast<const double2*>(phi), logdet, Theta,
                       nullptr, status, n_pairs, pairs_per_walker, digits ? OVL_TRIAL : OVL_THETA);
        if (e != cudaSuccess) return noalloc_fail(AFQMC_ERR_CUDA, "overlap kernel", e);
    }
    double2* v = reinterpret_cast<double2*>(force_bias);
    double2* el = reinterpret_cast<double2*>(e_local);
    if (digits) {
        // the digits of h and L lie first in the work space, at the same place for both parts
        e = contract_fp64d_prepare(s, part[part[0].W == 0], h, L, work, chunk[part[0].W == 0]);
        for (int q = 0; q < 2 && e == cudaSuccess; ++q) {
            const long long p0 = q ? part[0].pairs : 0, w0 = q ? part[0].W : 0;
            if (part[q].W)
                e = contract_fp64d(s, part[q], work, Theta + p0 * N * nt, reinterpret_cast<const double2*>(phi) + w0 * N * nt,
                                   v + p0 * n_chol, el + p0, status, PairList(), chunk[q]);
        }
    } else {
        e = contract_fp64(s, d, h, L, Phi, Theta, v, el, n_pairs);
    }
    if (e != cudaSuccess) return noalloc_fail(AFQMC_ERR_CUDA, "contraction kernel", e);
    noalloc_finish_kernel<<<(unsigned)((n_pairs + 255) / 256), 256, 0, s>>>(n_pairs, n_chol, status, logdet,
                                                                            reinterpret_cast<double2*>(logov), el, v);
    count_launches(1);
    e = cudaGetLastError();
    if (e != cudaSuccess) return noalloc_fail(AFQMC_ERR_CUDA, "log-determinant kernel", e);
    return AFQMC_OK;
}
