// FP64 contraction on the tensor cores: the fused force-bias / local-energy
// contraction of Eq. (15), (16), (27) with FP64 accuracy, every matrix product as
// exact integer digit products (digits64.cuh).
//
// With B_p = Phi_p A_p^-T (written by the overlap kernel in place of Theta; conj(Phi_p)
// for complex trial samples) and Y_g = X_g phi_w (X_0 = h, X_g = L_g; one per walker),
//     Z_{p,g} = B_p^T Y_g = A_p^-1 (Phi_p^dagger X_g phi_w)
// is similar to M_{p,g} = Phi_p^dagger X_g Theta_p, so v_g = sum_s Tr Z and
// E_L = sum_s Tr Z_0 + 1/2 sum_g [v_g^2 - sum_s Tr Z_g^2].
//
// Two GEMMs, both 128-row tiles of tcgen05.mma (kind::f16, K-major operands in the
// 128-byte swizzled layout).  A tile's D digits of A meet the D digits of B laid
// side by side (B rows q NT + c): one MMA of A digit i against the B digits
// 0 .. D - 1 - i adds A_i B_j to accumulator i + j for every j, so the D orders of a
// 128 x NT tile fill D NT of the 512 tensor-memory columns.
//   fd_y_kernel  Y: rows (w, column, re/im) of every walker of the chunk laid end to
//                end, columns j of X_g; the epilogue adds the orders as 64-bit
//                integers (exact to their rounding), stores those and keeps the
//                largest of each (walker, spin, g);
//   contract_fp64d_kernel  Z of one walker and spin: rows (re/im, pair, a) of a tile of
//                PB pairs, [Re B | -Im B] and [Im B | Re B] over K = (re, im) x N;
//                columns (g, b).  Four warps turn the integers of Y into digits in
//                shared memory (8 bytes per value from L2 instead of the 16 of its
//                digits), the A digits stream through a ring of bulk copies, and
//                the epilogue adds the orders to 56-bit integers Z' and forms
//                Tr Z and Tr Z^2 from those exactly (64-bit products of their 28-bit
//                halves): FP64 arithmetic is left for the last sums only,
//                whose pipe (two multiply-adds per clock and SM) would otherwise
//                take as long as the MMAs.
// What bounds it: shared memory.  D (D + 1) / 2 digit products per product, each MMA
// reading A (32 clocks) and B (N / 4) and taking N / 2 clocks itself, and both operands'
// way in (the A digits of a tile of pairs, 0.25 MB at 50 orbitals, pass once per column
// tile); then the epilogue's 64-bit integer arithmetic, about 30 instructions per entry.
// Measured on one GB300, whole contraction against the FP64 kernels it replaces:
// 50 orbitals, 512 x 32 pairs 18.4 ms against 265 (contract_fp64z_kernel, 0.98 of the FP64
// pipe); 120 orbitals, 8 x 64 pairs 18 ms against 458 (contract_fp64_kernel); 37 orbitals,
// 24 x 9 pairs 0.18 ms against 1.07; 8 orbitals, 64 x 16 pairs 0.15 ms against 0.40: faster
// at every size it takes, so it takes all of those (fd_shape).  With a list of pairs (the mixed path's
// refinement, api.cu has the rule) blocks of walkers and tiles without listed pairs end at once.
//
// Accuracy: operands to 63 (62) bits of the largest entry of their group (a matrix
// X_g; a column of a walker; a pair's B with its columns in the units those leave; one walker's Y_g of one spin), products exact, Y rounded
// at 2^-57 (2^-55) of the product of its groups' largest entries, Z at 2^-56 of its
// bound for Tr Z^2 and up to four bits finer for Tr Z: below the rounding of an FP64 sum
// of the same length.  Against quad precision, 8 to 200 orbitals: pair energies 3e-17 to
// 3e-16 (the FP64 kernels 6e-17 to 6e-16), force bias 1e-16 to 2e-15 (1e-16 to 2e-15).
//
// Everything of one (pair, g) is exact up to its rounding to FP64 (v and Tr Z^2, stored), and
// the sums over g are taken by the last kernel in one order: results do not depend on how the work is split, on the
// other pairs or on the column tiles.
#include <algorithm>

#include "digits64.cuh"
#include "kernels.cuh"
#include "tcgen05.cuh"

namespace afq {

namespace {

constexpr int FD_EPI = 512;               // epilogue threads: four warps per tensor-memory quadrant
constexpr int FDY_THREADS = 64 + FD_EPI;  // warp 0 producer, warp 1 MMA issue, warps 2-17 epilogue
constexpr int FDZ_DIG = 256;              // threads that write the digits of Y
constexpr int FDZ_FIN = FDY_THREADS + FDZ_DIG;   // first thread of the warp that forms the FP64 sums
constexpr int FDZ_THREADS = FDZ_FIN + 32;
constexpr uint32_t FD_ADIG = 16384;       // one digit of a 64-element K chunk of a 128-row operand
constexpr int FD_MAXS = 9;                // stages of the A ring
constexpr size_t FD_SMEM_MAX = 225 * 1024;   // dynamic; static use is below 2 KB of 227 KB
constexpr int FD_RUN = 4;                 // column tiles of a block at least

// Byte offset of the 16-byte unit u (K elements 8u .. 8u + 7) of row r in a K-major
// 128-byte swizzled region.
__host__ __device__ __forceinline__ uint32_t fd_swz(int r, int u) {
    return (uint32_t)(r >> 3) * 1024u + (uint32_t)(r & 7) * 128u + (uint32_t)((u ^ (r & 7)) << 4);
}

// Bounded wait that records a timeout; after one every wait of the block gives up.
__device__ __forceinline__ bool fd_wait(uint64_t* bar, uint32_t parity, uint32_t lim, volatile int* fail) {
    if (tc::mbar_wait(bar, parity, 1)) return true;
    if (*fail) return false;
    if (tc::mbar_wait(bar, parity, lim)) return true;
    *fail = 1;
    return false;
}

// Digits of B in one MMA of at most 256 columns, a multiple of 16 columns when split.
__host__ __device__ __forceinline__ int fd_maxblk(int NT) { return (NT & 8) ? (256 / NT) & ~1 : 256 / NT; }
// Tensor-memory columns of a tile's accumulators (with NT an odd multiple of 8 an MMA of an odd
// number of digits ends 8 columns past them); shared-memory bytes of a chunk of its B digits.
__host__ __device__ constexpr int fd_cols(int D, int NT) { return (NT & 8) ? (D * NT + 8 + 15) & ~15 : D * NT; }
__host__ __device__ __forceinline__ uint32_t fd_bslot(int D, int NT) { return (uint32_t)fd_cols(D, NT) * 128u; }

// Named barrier `id` over `count` threads (whole warps); the _or form returns the OR of v.
__device__ __forceinline__ void fd_group_sync(int id, int count) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ bool fd_group_sync_or(int id, int count, bool v) {
    uint32_t r;
    asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.or.pred q, %2, %3, p;\nselp.u32 %0, 1, 0, q;\n}"
                 : "=r"(r)
                 : "r"((uint32_t)v), "r"(id), "r"(count)
                 : "memory");
    return r != 0;
}

// A ring slot and the parity its producer waits for before filling it again.
struct FdRing {
    int st;
    uint32_t ph;
    __device__ __forceinline__ void next(int S) {
        if (++st == S) { st = 0; ph ^= 1u; }
    }
};

struct FdPipe {
    uint64_t afull[FD_MAXS], aempty[FD_MAXS], bfull[2], bempty[2], dfull[2], dempty[2], drain;
    uint32_t tslot;
    int fail;
};

__device__ __forceinline__ void fd_pipe_init(FdPipe& p, int S, int bfull_count, int epi_warps) {
    for (int q = 0; q < S; ++q) {
        tc::mbar_init(&p.afull[q], 1);
        tc::mbar_init(&p.aempty[q], 1);
    }
    for (int q = 0; q < 2; ++q) {
        tc::mbar_init(&p.bfull[q], bfull_count);
        tc::mbar_init(&p.bempty[q], 1);
    }
    for (int q = 0; q < 2; ++q) {
        tc::mbar_init(&p.dfull[q], 1);
        tc::mbar_init(&p.dempty[q], epi_warps);
    }
    tc::mbar_init(&p.drain, 1);
    tc::mbar_fence_init();
    p.fail = 0;
}

// The MMA loop of one warp: `tiles` tiles of KC chunks; A digits (unit (tile, chunk,
// digit)) from the ring, B chunks from two slots.  ksteps: K steps of 16 in all.
// A tile's accumulators take fd_cols columns of one of nbuf buffers: every MMA of a
// tile ends at column D NT, or, rounded up to 16 columns, in the padding past it.  a_res: the A digits of all chunks
// stay in the ring (S >= KC D), loaded once.
// One lane's instructions feed the tensor core, and an MMA whose operands are not
// already in uniform registers costs 160 to 230 clocks to issue against 72 to
// execute (N = 144 on average): NT is a template parameter and the digits are
// unrolled, so descriptors differ by constants, and the whole warp runs the loop
// without a divergent exit.  Issued like that the pattern of MMAs runs at 90 % (NT =
// 32) to 97 % (NT = 64) of the tensor peak; each MMA takes max(N / 2, 32 + N / 4)
// clocks (A and B from shared memory).  After a timeout the waits return at once and
// nothing is issued or handed back any more (the block's results are void then): a slot
// whose copy has not landed must not go back to its producer, whose barrier would take an arrival too many.
template <int BITS, int NT>
__device__ __forceinline__ bool fd_mma_loop_nt(FdPipe& p, uint32_t taddr, const uint8_t* bslots, uint32_t bslot_bytes,
                                               const uint8_t* ring, int S, int tiles, int KC, int ksteps, int nbuf,
                                               bool a_res, uint32_t lim) {
    constexpr int D = Dg64<BITS>::D;
    constexpr int MB = (NT & 8) ? (256 / NT) & ~1 : 256 / NT;   // fd_maxblk
    constexpr uint32_t bufcols = fd_cols(D, NT);
    const uint64_t bd0 = tc::desc_sw128(tc::smem_u32(bslots));
    const uint32_t bdelta = bslot_bytes >> 4;
    const uint64_t ad0 = tc::desc_sw128(tc::smem_u32(ring));
    volatile int* fail = &p.fail;
    bool ok = true;
    int ub = 0, st = 0;
    uint32_t aph = 0;                                  // ring slot and phase of the next A digit
    for (int t = 0; t < tiles; ++t) {
        const int w = t - nbuf;                        // the tile that last held these accumulators
        if (w >= 0) ok &= fd_wait(&p.dempty[w & 1], (uint32_t)((w >> 1) & 1), lim, fail);
        const uint32_t tb = taddr + (nbuf == 2 && (t & 1) ? bufcols : 0u);
        for (int c = 0; c < KC; ++c, ++ub) {
            ok &= fd_wait(&p.bfull[ub & 1], (uint32_t)((ub >> 1) & 1), lim, fail);
            const uint64_t bd = bd0 + (uint64_t)((ub & 1) ? bdelta : 0u);
            const int ks = min(4, ksteps - 4 * c);
            const uint32_t accc = c > 0 ? 1u : 0u;
#pragma unroll
            for (int i = 0; i < D; ++i) {
                if (!a_res || t == 0) ok &= fd_wait(&p.afull[st], aph, lim, fail);
                tc::fence_after_sync();
                const uint64_t ad = ad0 + (uint64_t)((uint32_t)st * (FD_ADIG / 16));
                constexpr int cap = MB;
                const int n1 = D - i < cap ? D - i : cap, n2 = D - i - n1;
                __syncwarp();
                if (tc::elect_one() && ok) {
#pragma unroll
                    for (int s = 0; s < 4; ++s) {
                        if (s < ks) {
                            const uint32_t acc = (i > 0 || s > 0) ? 1u : accc;
                            tc::mma_f16(tb + (uint32_t)(i * NT), ad + 2 * s, bd + 2 * s,
                                        tc::idesc_f16_f32(128, (n1 * NT + 15) & ~15), acc);
                            if (n2 > 0)
                                tc::mma_f16(tb + (uint32_t)((i + MB) * NT), ad + 2 * s, bd + (uint64_t)(MB * NT * 8 + 2 * s),
                                            tc::idesc_f16_f32(128, (n2 * NT + 15) & ~15), acc);
                        }
                    }
                    if (!a_res) tc::mma_commit(&p.aempty[st]);
                    if (i == D - 1) {
                        tc::mma_commit(&p.bempty[ub & 1]);
                        if (c == KC - 1) tc::mma_commit(&p.dfull[t & 1]);
                    }
                }
                __syncwarp();
                if (++st == (a_res ? KC * D : S)) { st = 0; aph ^= 1u; }
            }
        }
    }
    if (tc::elect_one()) tc::mma_commit(&p.drain);     // every issued MMA completes before the block leaves
    __syncwarp();
    tc::mbar_wait(&p.drain, 0, 1u << 22);
    return ok;
}

// NT by its template (host side: multiples of 8 up to 64).
template <int BITS>
__device__ __forceinline__ bool fd_mma_loop(FdPipe& p, uint32_t taddr, const uint8_t* bslots, uint32_t bslot_bytes,
                                            const uint8_t* ring, int S, int tiles, int KC, int ksteps, int NT, int nbuf,
                                            bool a_res, uint32_t lim) {
    switch (NT) {
    case 8: return fd_mma_loop_nt<BITS, 8>(p, taddr, bslots, bslot_bytes, ring, S, tiles, KC, ksteps, nbuf, a_res, lim);
    case 16: return fd_mma_loop_nt<BITS, 16>(p, taddr, bslots, bslot_bytes, ring, S, tiles, KC, ksteps, nbuf, a_res, lim);
    case 24: return fd_mma_loop_nt<BITS, 24>(p, taddr, bslots, bslot_bytes, ring, S, tiles, KC, ksteps, nbuf, a_res, lim);
    case 32: return fd_mma_loop_nt<BITS, 32>(p, taddr, bslots, bslot_bytes, ring, S, tiles, KC, ksteps, nbuf, a_res, lim);
    case 40: return fd_mma_loop_nt<BITS, 40>(p, taddr, bslots, bslot_bytes, ring, S, tiles, KC, ksteps, nbuf, a_res, lim);
    case 48: return fd_mma_loop_nt<BITS, 48>(p, taddr, bslots, bslot_bytes, ring, S, tiles, KC, ksteps, nbuf, a_res, lim);
    case 56: return fd_mma_loop_nt<BITS, 56>(p, taddr, bslots, bslot_bytes, ring, S, tiles, KC, ksteps, nbuf, a_res, lim);
    default: return fd_mma_loop_nt<BITS, 64>(p, taddr, bslots, bslot_bytes, ring, S, tiles, KC, ksteps, nbuf, a_res, lim);
    }
}

// The largest |x| of a group as the bits of a double (the order of non-negative doubles is that of their
// bits): FP64 comparisons would take the FP64 pipe, 16 clocks a warp.  Infinities and NaN come out above all.
__device__ __forceinline__ unsigned long long fd_abs_bits(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}
constexpr unsigned long long FD_INF_BITS = 0x7FF0000000000000ull;

// 2^e, |e| <= 1000.
__device__ __forceinline__ double fd_p2(int e) {
    return __longlong_as_double((long long)(1023 + max(-1000, min(1000, e))) << 52);
}

}  // namespace

// ---------------------------------------------------------------- X image (once)
// exponent of matrix g from its largest |entry|
template <int BITS>
__global__ void fd_xexp_kernel(int N, const double* __restrict__ h, const double* __restrict__ L, int* xexp) {
    __shared__ double red[8];
    const int g = blockIdx.x, lane = threadIdx.x & 31;
    const double* X = g == 0 ? h : L + (long long)(g - 1) * N * N;
    double m = 0.0;
    bool bad = false;
    for (int e = threadIdx.x; e < N * N; e += blockDim.x) {
        const double v = fabs(X[e]);
        bad |= !isfinite(v);
        m = fmax(m, v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) red[threadIdx.x >> 5] = m;
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        for (int q = 1; q < 8; ++q) m = fmax(m, red[q]);
        xexp[g] = bad ? DG64_NAN : dg64_exp<BITS>(m);
    }
}

// Block ((g JT + jt) KCX + c): D digits of NTY rows j = jt NTY + r, K = i in [64c, 64c + 64).
template <int BITS>
__global__ void fd_x_image_kernel(int N, int KCX, int JT, int NTY, int G1, const double* __restrict__ h,
                                  const double* __restrict__ L, const int* __restrict__ xexp, uint8_t* __restrict__ out) {
    constexpr int D = Dg64<BITS>::D;
    const long long units = (long long)G1 * JT * KCX * NTY * 8;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < units; e += (long long)gridDim.x * blockDim.x) {
        const int u = (int)(e & 7);
        const int r = (int)((e >> 3) % NTY);
        const long long blk = (e >> 3) / NTY;
        const int c = (int)(blk % KCX);
        const int jt = (int)((blk / KCX) % JT);
        const int g = (int)(blk / KCX / JT);
        const double* X = g == 0 ? h : L + (long long)(g - 1) * N * N;
        const int j = jt * NTY + r, xe = xexp[g];
        long long F[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int i = c * 64 + 8 * u + t;
            F[t] = (j < N && i < N) ? dg64_fix(X[(long long)j * N + i], xe) : 0;
        }
        uint8_t* base = out + (size_t)blk * D * NTY * 128;
        dg64_unit<BITS>(F, [&](int q, uint4 v) { *reinterpret_cast<uint4*>(base + fd_swz(q * NTY + r, u)) = v; });
    }
}

// ---------------------------------------------------------------- digits of the walkers
// Block: 64 columns of the chunk's walkers laid end to end, rows r = 2 column + (Re, Im), K = i.
// A column has an exponent of its own, cexp[w nt + c]: Z D and D^-1 Z have the traces of Z, so the
// column taken as phi 2^cexp here and B's as B 2^-cexp leave them as they are, and no column loses
// digits to a longer one.  bad[w] (cleared before): a non-finite entry.
template <int BITS>
__global__ void __launch_bounds__(256) fd_phi_image_kernel(int N, int nt, int KCX, long long w0, long long wb,
                                                           const double2* __restrict__ phi, uint8_t* __restrict__ out,
                                                           int* __restrict__ cexp, unsigned int* __restrict__ bad) {
    constexpr int D = Dg64<BITS>::D;
    __shared__ unsigned long long smax[4][64];
    __shared__ int se[64];
    const int C0 = blockIdx.x * 64, cols = (int)wb * nt;               // fd_shape keeps them in 32 bits
    const int tid = threadIdx.x;
    {
        const int q = tid & 63, part = tid >> 6;
        const int C = C0 + q;
        unsigned long long m = 0;
        if (C < cols) {
            const double2* ph = phi + (w0 + C / nt) * (long long)N * nt + C % nt;
#pragma unroll 4
            for (int i = part; i < N; i += 4) {
                const double2 v = ph[(long long)i * nt];
                m = max(m, max(fd_abs_bits(v.x), fd_abs_bits(v.y)));
            }
        }
        smax[part][q] = m;
    }
    __syncthreads();
    if (tid < 64) {
        const unsigned long long m = max(max(smax[0][tid], smax[1][tid]), max(smax[2][tid], smax[3][tid]));
        const bool inf = m >= FD_INF_BITS;
        const int e = inf ? DG64_NAN : dg64_exp<BITS>(__longlong_as_double((long long)m));
        se[tid] = e;
        const int C = C0 + tid;
        if (C < cols) {
            cexp[C] = inf ? 0 : e;
            if (inf) bad[C / nt] = 1;
        }
    }
    __syncthreads();
    uint8_t* base = out + (size_t)blockIdx.x * KCX * D * FD_ADIG;
    for (int e = tid; e < KCX * 128 * 8; e += 256) {
        const int r = e & 127, u = (e >> 7) & 7, c = e >> 10;
        long long F[8];
        const int C = C0 + (r >> 1);
        const bool ok = C < cols;
        const int pe = ok ? se[r >> 1] : 0;
        const double2* ph = phi + (w0 + C / nt) * (long long)N * nt + C % nt;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int i = c * 64 + 8 * u + t;
            F[t] = 0;
            if (ok && i < N) {
                const double2 v = ph[(long long)i * nt];
                F[t] = dg64_fix((r & 1) ? v.y : v.x, pe);
            }
        }
        dg64_unit<BITS>(F, [&](int q, uint4 v) {
            *reinterpret_cast<uint4*>(base + ((size_t)c * D + q) * FD_ADIG + fd_swz(r, u)) = v;
        });
    }
}

// ---------------------------------------------------------------- GEMM-Y
// Block: row tile blockIdx.x / n_gblk, matrices [gb GPB, (gb + 1) GPB); tiles (g, jt).
// Y[s][((wl G1 + g) n_s + b) 2 + ri][i < N8], the pairs (i, i + 1) of i % 8 = 0 first, then those
// of 2, 4, 6 (GEMM-Z's threads take eight values each, neighbours 16 bytes apart), as integers in units of
// 2^(UNIT - XTRA - cexp - xexp[g]), cexp the column's; ymax[(wl 2 + s) G1 + g] = max |Y| >> 32.
template <int BITS>
__global__ void __launch_bounds__(FDY_THREADS, 1)
    fd_y_kernel(int N8, int nu, int nd, int G1, int KCX, int ksteps, int JT, int NTY, int nbuf, int S, int GPB, int n_gblk,
                int a_res, long long wb, const uint8_t* __restrict__ Pimg, const uint8_t* __restrict__ Ximg,
                long long* __restrict__ Y0, long long* __restrict__ Y1, unsigned int* __restrict__ ymax, int* status,
                uint32_t lim, const int* __restrict__ listed) {
    constexpr int D = Dg64<BITS>::D;
    if (listed) {                                      // no walker of the tile has a listed pair
        const long long wt = (long long)(blockIdx.x / n_gblk) * 128 / (2 * (nu + nd)) + threadIdx.x;
        const bool in = threadIdx.x < 65 && wt < wb && wt * 2 * (nu + nd) < ((long long)(blockIdx.x / n_gblk) + 1) * 128;
        if (!__syncthreads_or(in && listed[wt] > 0)) return;
    }
    extern __shared__ uint8_t smraw[];
    uint8_t* sm = (uint8_t*)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
    const uint32_t bbytes = (uint32_t)D * (uint32_t)NTY * 128u;
    uint8_t* ring = sm + 2 * (size_t)bbytes;
    __shared__ FdPipe pp;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // warp: uniform
    const long long tile = blockIdx.x / n_gblk;
    const int gb = blockIdx.x % n_gblk;
    const int g0 = gb * GPB, g1 = min(G1, g0 + GPB);
    const int tiles = max(0, g1 - g0) * JT;
    const int nt = nu + nd;
    if (warp == 1) {
        tc::tmem_alloc(&pp.tslot, 512);
        tc::tmem_relinquish();
    }
    if (tid == 0) fd_pipe_init(pp, S, 1, FD_EPI / 32);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t taddr = pp.tslot;
    volatile int* fail = &pp.fail;
    bool failed = false;
    if (warp == 0) {
        if (lane == 0) {
            const uint8_t* At = Pimg + (size_t)tile * KCX * D * FD_ADIG;
            int ua = 0, ub = 0;
            FdRing rg{0, 1u};
            const uint8_t* Bt = Ximg + (size_t)g0 * JT * KCX * bbytes;   // tiles (g, jt) follow one another
            for (int t = 0; t < tiles && !failed; ++t, Bt += (size_t)KCX * bbytes) {
                for (int c = 0; c < KCX && !failed; ++c, ++ub) {
                    if (ub >= 2 && !fd_wait(&pp.bempty[ub & 1], (uint32_t)(((ub >> 1) - 1) & 1), lim, fail)) { failed = true; break; }
                    tc::mbar_arrive_expect_tx(&pp.bfull[ub & 1], bbytes);
                    tc::bulk_g2s(sm + (size_t)(ub & 1) * bbytes, Bt + (size_t)c * bbytes, bbytes, &pp.bfull[ub & 1]);
                    if (a_res && t > 0) continue;
                    for (int i = 0; i < D; ++i, ++ua) {
                        if (ua >= S && !fd_wait(&pp.aempty[rg.st], rg.ph, lim, fail)) { failed = true; break; }
                        tc::mbar_arrive_expect_tx(&pp.afull[rg.st], FD_ADIG);
                        tc::bulk_g2s(ring + (size_t)rg.st * FD_ADIG, At + ((size_t)c * D + i) * FD_ADIG, FD_ADIG, &pp.afull[rg.st]);
                        rg.next(S);
                    }
                    if (failed) { ++ub; break; }
                }
            }
            // every issued copy lands before the block leaves
            for (int v = max(0, ua - S); v < ua; ++v) tc::mbar_wait(&pp.afull[v % S], (uint32_t)((v / S) & 1), 1u << 22);
            for (int v = max(0, ub - 2); v < ub; ++v) tc::mbar_wait(&pp.bfull[v & 1], (uint32_t)((v >> 1) & 1), 1u << 22);
            if (failed) atomicOr(status, STATUS_TIMEOUT);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (!fd_mma_loop<BITS>(pp, taddr, sm, bbytes, ring, S, tiles, KCX, ksteps, NTY, nbuf, a_res != 0, lim))
            atomicOr(status, STATUS_TIMEOUT);
        __syncwarp();
    } else {
        const int quad = warp & 3, set = (warp - 2) >> 2;
        const long long R = tile * 128 + 32 * quad + lane;
        const long long w = R / (2 * nt);
        const int cc = (int)(R % (2 * nt));
        const bool row_ok = w < wb;
        const int c = cc >> 1, s = c >= nu;
        const int ns = s ? nd : nu, b = s ? c - nu : c;
        long long* Yr = (s ? Y1 : Y0) + (((row_ok ? w : 0) * G1 * ns + b) * 2 + (cc & 1)) * (long long)N8;
        const uint32_t lb = taddr + ((uint32_t)(32 * quad) << 16);
        const unsigned key = row_ok ? (unsigned)(w * 2 + s) : 0xffffffffu;
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        unsigned mx = 0;
        for (int t = 0; t < tiles; ++t) {
            const int g = g0 + t / JT, jt = t % JT;
            const int buf = nbuf == 2 ? (t & 1) : 0;
            bool ok = true;
            if (lane == 0) ok = fd_wait(&pp.dfull[t & 1], (uint32_t)((t >> 1) & 1), lim, fail);
            if (__any_sync(0xffffffffu, !ok)) { failed = true; break; }
            tc::fence_after_sync();
            for (int col = set * 4; col < NTY; col += 16) {
                const int j = jt * NTY + col;
                if (j >= N8) break;                                // uniform
                float v[D][4];
#pragma unroll
                for (int q = 0; q < D; ++q) tc::tmem_ld4(lb + (uint32_t)(buf * fd_cols(D, NTY)) + (uint32_t)(q * NTY + col), v[q]);
                tc::tmem_ld_wait();
                long long I[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float a[D];
#pragma unroll
                    for (int q = 0; q < D; ++q) a[q] = v[q][k];
                    I[k] = dg64_sum_fine<BITS>(a);
                    mx = max(mx, (unsigned)((I[k] < 0 ? -I[k] : I[k]) >> 32));
                }
                if (row_ok) {
                    longlong2* dst = reinterpret_cast<longlong2*>(Yr + (long long)g * ns * 2 * N8) + (j >> 3);
#pragma unroll
                    for (int k = 0; k < 2; ++k)
                        dst[(((j & 7) >> 1) + k) * (N8 >> 3)] = make_longlong2(I[2 * k], I[2 * k + 1]);
                }
            }
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&pp.dempty[t & 1]);
            if (jt == JT - 1) {
                const unsigned m = __reduce_max_sync(peers, mx);
                if (row_ok && lane == __ffs(peers) - 1) atomicMax(&ymax[(w * 2 + s) * G1 + g], m);
                mx = 0;
            }
        }
        if (failed && lane == 0) atomicOr(status, STATUS_TIMEOUT);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) tc::tmem_dealloc(taddr, 512);
}

// ---------------------------------------------------------------- digits of B_p
// Block: walker w0 + blockIdx.x / MT, pairs m PB .. of the walker, one spin.  Row
// r = 64 ri + p_l n + a: [Re B[:, a] | -Im B[:, a]] (ri = 0), [Im B[:, a] | Re B[:, a]]
// (ri = 1), each half N8 elements of K; KC chunks of D digits.  bexp[pair]: the
// pair's exponent, that of the columns B 2^-cexp (the walkers' cexp); bsh[pair]: the right shift that brings its Z into 2^zbits.  With a list
// the walker's pairs are its listed ones, in the order of the list.
// A block reads its columns of B into shared memory in one go (staged; they fit but for the
// largest N) and forms exponents and digits from there: read from global memory column by
// column, the loads' latency bound it, and the
// FP64 pipe by the maxima's comparisons, integer ones now (48 blocks of 200 orbitals and 40 electrons 110 us,
// staged 75, with a thread per column for the exponents 67; 64 blocks of 8 and 4 20, 16 and 17).
constexpr int FDB_T = 512;
template <int BITS>
__global__ void __launch_bounds__(FDB_T) fd_b_image_kernel(int N, int N8, int nt, int col0, int n, int P, int PB, int MT,
                                                         int KC, int zbits, long long w0, const int* __restrict__ cexp,
                                                         const double2* __restrict__ Bm, uint8_t* __restrict__ out,
                                                         int* __restrict__ bexp, int* __restrict__ bsh, PairList list, int staged) {
    constexpr int D = Dg64<BITS>::D;
    extern __shared__ double2 sB[];                                    // column q (pair q / n, a = q % n) at q NS
    __shared__ unsigned long long smax[64];
    __shared__ double sl1[64];
    __shared__ int se[64], sce[64], scol[64];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long wl = blockIdx.x / MT;
    const int m = blockIdx.x % MT;
    const int np = min(PB, (list.count ? list.count[w0 + wl] : P) - m * PB);
    if (np <= 0) return;
    const long long lp0 = wl * P + (long long)m * PB;                  // first pair, in the chunk
    __shared__ long long spair[64];
    if (tid < n) sce[tid] = cexp[wl * nt + col0 + tid];
    if (tid < np) spair[tid] = list.count ? (long long)list.items[list.base[w0 + wl] + m * PB + tid] : w0 * P + lp0 + tid;
    __syncthreads();
    const double2* B0 = Bm + col0;
    const int NS = N | 1, Nn = N * n;
    if (staged) {
        for (int e = tid; e < np * Nn; e += FDB_T) {
            const int p = e / Nn, i = (e - p * Nn) / n, a = e - p * Nn - i * n;
            sB[(p * n + a) * NS + i] = B0[(spair[p] * N + i) * nt + a];
        }
        __syncthreads();
    }
    // column q: entry i at Bq[i step]
    const long long step = staged ? 1 : nt;
    auto column = [&](int q) { return staged ? sB + q * NS : B0 + spair[q / n] * N * nt + q % n; };
    for (int q = warp; q < np * n; q += FDB_T / 32) {
        const double2* Bq = column(q);
        unsigned long long mx = 0;
        double l1 = 0.0;
        for (int i = lane; i < N; i += 32) {
            const double2 v = Bq[i * step];
            mx = max(mx, max(fd_abs_bits(v.x), fd_abs_bits(v.y)));
            l1 += fabs(v.x) + fabs(v.y);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            l1 += __shfl_xor_sync(0xffffffffu, l1, o);
        }
        if (lane == 0) {
            smax[q] = mx;
            sl1[q] = l1;
        }
    }
    __syncthreads();
    if (tid < np * n)      // the column's exponent in the walker's units; zero columns above, non-finite ones below all
        scol[tid] = smax[tid] == 0 ? INT_MAX
                    : smax[tid] >= FD_INF_BITS ? DG64_NAN
                    : dg64_exp<BITS>(__longlong_as_double((long long)smax[tid])) + sce[tid % n];
    __syncthreads();
    if (tid < np * n) {
        const int p = tid / n;
        int e = INT_MAX;
        for (int a = 0; a < n; ++a) e = min(e, scol[p * n + a]);
        if (e == INT_MAX) e = 0;
        // the column's integers added up, over 2^(TOT - 1)
        const double m = __longlong_as_double((long long)smax[tid]);
        double b0 = 0.0;
        if (e != DG64_NAN && m > 0.0)
            b0 = fmin(sl1[tid] / m, 2.0 * N) * ldexp(m, e - sce[tid % n] - (Dg64<BITS>::TOT - 1));
        sl1[tid] = b0;
        if (tid == p * n) se[p] = e;
    }
    __syncthreads();
    if (tid < np) {
        // |Z'| <= b0 2^54 before the shift, b0 the largest of the pair's columns
        double b0 = 0.0;
        for (int a = 0; a < n; ++a) b0 = fmax(b0, sl1[tid * n + a]);
        bexp[lp0 + tid] = se[tid];
        bsh[lp0 + tid] = b0 > 0.0 ? max(0, ilogb(b0 * (1.0 + 1e-9)) + 1 + 54 - zbits) : 0;
    }
    __syncthreads();
    uint8_t* base = out + (size_t)blockIdx.x * KC * D * FD_ADIG;
    const int h8 = N8 >> 3;
    for (int e = tid; e < KC * 128 * 8; e += FDB_T) {
        const int r = e & 127, u = (e >> 7) & 7, c = e >> 10;
        const int ri = r >> 6, q = r & 63;
        const int k8 = c * 8 + u;
        const int kim = k8 >= h8;
        long long F[8];
        const bool ok = q < np * n && k8 < 2 * h8;
        const double2* Bq = column(ok ? q : 0);
        const int be = ok ? se[q / n] - sce[q % n] : 0;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int i = (k8 - (kim ? h8 : 0)) * 8 + t;
            F[t] = 0;
            if (ok && i < N) {
                const double2 v = Bq[i * step];
                const long long f = dg64_fix((ri ^ kim) ? v.y : v.x, be);
                F[t] = (kim && !ri) ? -f : f;
            }
        }
        dg64_unit<BITS>(F, [&](int q2, uint4 v) {
            *reinterpret_cast<uint4*>(base + ((size_t)c * D + q2) * FD_ADIG + fd_swz(r, u)) = v;
        });
    }
}

// ---------------------------------------------------------------- GEMM-Z and the traces
struct FdZArgs {
    int n, G1, N8, KC, ksteps, NT, nbuf, ngrp, GB, NCT, P, PB, MT, S, T, RUN, NRUN;
    const uint8_t* Bimg;
    const int *bexp, *bsh, *xexp;
    const unsigned int* bad;                // walkers with a non-finite entry
    const long long* Y;
    const unsigned int* ymax;               // of this spin: entry (wl 2) G1 + g
    double2 *vpart, *xpart;                 // Tr Z and Tr Z^2 of [pair][g]
    int* status;
    const int* listed;                      // nullable: pairs of each walker (of the chunk), P at most
};

// Left shift that brings one walker's Y_g of a spin (largest |Y| >> 32 = m) to 0.99 2^(TOT - 1).
template <int BITS>
__device__ __forceinline__ int fd_yshift(unsigned m) {
    return Dg64<BITS>::TOT - 33 - (32 - __clz(m + (m >> 6) + 2u));
}

// Z' of a tile is kept as high 2^(FD_LOW + x) + low with x = min(FD_XTRA, shift) more bits than
// the products use, for the trace itself, which is summed over fewer entries; Z' + 2^(x - 1) is
// stored, so that low >> x rounds.
constexpr int FD_LOW = 28, FD_XTRA = 4;

// Sums over the index pairs of one (pair, g): Tr Z' (high and low parts) and Tr Z'^2 (128-bit,
// two words).
struct FdRed {
    long long th, uh, tl, ul, rh, ih;
    unsigned long long rl, il;
};

// h 2^(2 FD_LOW) + m 2^FD_LOW + l as a 128-bit integer.
__device__ __forceinline__ void fd_join(long long h, long long m, long long l, long long& hi, unsigned long long& lo) {
    const __int128 x = ((__int128)h << (2 * FD_LOW)) + ((__int128)m << FD_LOW) + l;
    hi = (long long)(x >> 64);
    lo = (unsigned long long)x;
}

__device__ __forceinline__ void fd_add(long long& hi, unsigned long long& lo, long long h2, unsigned long long l2) {
    lo += l2;
    hi += h2 + (lo < l2 ? 1 : 0);
}

// Block: item = (walker, tile of pairs, run of column tiles).  Column tile t holds the
// columns (g_l, b), g = t GB + g_l; shared memory: two chunks of Y's digits (D NT rows of
// 128 bytes), the A ring, Z' of a tile (128 rows of (high, low) halves), the sums of the
// (pair, g) of two tiles, and the list of unordered index pairs (a, b).  T threads share
// the traces of one (pair, g); a warp of its own turns the sums into FP64 (on the
// epilogue's warps the conversions took as long as the rest of it).
template <int BITS>
__global__ void __launch_bounds__(FDZ_THREADS, 1) contract_fp64d_kernel(const __grid_constant__ FdZArgs A, uint32_t lim) {
    constexpr int D = Dg64<BITS>::D;
    extern __shared__ uint8_t smraw[];
    uint8_t* sm = (uint8_t*)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
    const int n = A.n, NT = A.NT, GB = A.GB, G1 = A.G1, KC = A.KC, S = A.S, nbuf = A.nbuf;
    const uint32_t bbytes = fd_bslot(D, NT);
    uint8_t* ring = sm + 2 * (size_t)bbytes;
    const int ldc = (GB * n) | 1;
    const int combos = A.PB * GB, parts = A.T > 32 ? A.T / 32 : 1;
    int2* Ms = reinterpret_cast<int2*>(ring + (size_t)S * FD_ADIG);
    FdRed* red = reinterpret_cast<FdRed*>(Ms + A.ngrp * 128 * (ldc + 1));   // [2][combos parts]
    uchar2* tab = reinterpret_cast<uchar2*>(red + 2 * combos * parts);
    __shared__ FdPipe pp;
    __shared__ uint64_t rfull[2], rempty[2];
    __shared__ int sbexp[64], sbsh[64];
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // warp: uniform
    const int run = blockIdx.x % A.NRUN;
    const long long wm = blockIdx.x / A.NRUN;          // (walker, tile)
    const long long wl = wm / A.MT;
    const int m = (int)(wm % A.MT);
    const int np = min(A.PB, (A.listed ? A.listed[wl] : A.P) - m * A.PB);
    if (np <= 0) return;                               // uniform
    const long long lp0 = wl * A.P + (long long)m * A.PB;
    const int t0 = run * A.RUN, t1 = min(A.NCT, t0 + A.RUN);
    const int tiles = t1 - t0;
    const int U = n * (n + 1) / 2;

    if (warp == 1) {
        tc::tmem_alloc(&pp.tslot, 512);
        tc::tmem_relinquish();
    }
    if (tid == 0) {
        for (int q = 0; q < 2; ++q) {
            tc::mbar_init(&rfull[q], FD_EPI / 32 / A.ngrp);
            tc::mbar_init(&rempty[q], 1);
        }
        fd_pipe_init(pp, S, FDZ_DIG / 32, FD_EPI / 32 / A.ngrp);
    }
    if (tid >= 64 && tid < 64 + np) {
        sbexp[tid - 64] = A.bexp[lp0 + tid - 64];
        sbsh[tid - 64] = A.bsh[lp0 + tid - 64];
    }
    for (int a = tid; a < n; a += FDZ_THREADS) {       // (a, a) first, then (a, b > a)
        tab[a] = make_uchar2((unsigned char)a, (unsigned char)a);
        int u = n + a * (n - 1) - a * (a - 1) / 2;
        for (int b = a + 1; b < n; ++b) tab[u++] = make_uchar2((unsigned char)a, (unsigned char)b);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t taddr = pp.tslot;
    volatile int* fail = &pp.fail;
    bool failed = false;
    const unsigned int* ymx = A.ymax + wl * 2 * G1;

    if (warp == 0) {
        // ---- producer of the A digits
        if (lane == 0) {
            const uint8_t* At = A.Bimg + (size_t)wm * KC * D * FD_ADIG;
            const int per = KC * D, total = tiles * per;
            FdRing rg{0, 1u};
            int ua = 0;
            for (int k = 0; ua < total; ++ua) {        // counters, no division: the loop sets the ring's pace
                if (ua >= S && !fd_wait(&pp.aempty[rg.st], rg.ph, lim, fail)) { failed = true; break; }
                tc::mbar_arrive_expect_tx(&pp.afull[rg.st], FD_ADIG);
                tc::bulk_g2s(ring + (size_t)rg.st * FD_ADIG, At + (size_t)k * FD_ADIG, FD_ADIG, &pp.afull[rg.st]);
                if (++k == per) k = 0;
                rg.next(S);
            }
            for (int v = max(0, ua - S); v < ua; ++v) tc::mbar_wait(&pp.afull[v % S], (uint32_t)((v / S) & 1), 1u << 22);
            if (failed) atomicOr(A.status, STATUS_TIMEOUT);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (!fd_mma_loop<BITS>(pp, taddr, sm, bbytes, ring, S, tiles, KC, A.ksteps, NT, nbuf, false, lim))
            atomicOr(A.status, STATUS_TIMEOUT);
        __syncwarp();
    } else if (warp >= FDZ_FIN / 32) {
        // ---- the sums of a tile to FP64: lane q takes the (pair, g) q, q + 32, ..
        const bool bad = A.bad[wl] != 0;
        for (int t = t0; t < t1; ++t) {
            const int rb = (t - t0) & 1, use = (t - t0) >> 1;
            const int gn = min(GB, G1 - t * GB);
            bool ok = true;
            if (lane == 0) ok = fd_wait(&rfull[rb], (uint32_t)(use & 1), lim, fail);
            if (__any_sync(0xffffffffu, !ok)) { failed = true; break; }
            for (int q = lane; q < combos; q += 32) {
                const int pl = q / GB, gl = q - pl * GB, g = t * GB + gl;
                if (pl >= np || gl >= gn) continue;
                const int xe = __ldg(A.xexp + g);
                const unsigned ym = __ldg(ymx + g);
                const FdRed* rp = red + (rb * combos + q) * parts;
                FdRed r = rp[0];
                for (int k = 1; k < parts; ++k) {
                    r.th += rp[k].th;
                    r.uh += rp[k].uh;
                    r.tl += rp[k].tl;
                    r.ul += rp[k].ul;
                    fd_add(r.rh, r.rl, rp[k].rh, rp[k].rl);
                    fd_add(r.ih, r.il, rp[k].ih, rp[k].il);
                }
                double2 v, ex;
                const int eb = sbexp[pl];
                if (xe == DG64_NAN || bad || eb == DG64_NAN) {
                    const double nan = __longlong_as_double(0x7FF8000000000000LL);
                    v = cmk(nan, nan);
                    ex = v;
                } else {
                    // value of Z' = 1: 2^(UNIT + shift - bexp - yexp), in two exact factors
                    const int ey = fd_yshift<BITS>(ym) - (Dg64<BITS>::UNIT - Dg64<BITS>::XTRA) + xe;
                    const int sc = Dg64<BITS>::UNIT + sbsh[pl] - eb - ey;
                    const double f1 = fd_p2(sc >> 1), f2 = fd_p2(sc - (sc >> 1));
                    const double el = fd_p2(-min(FD_XTRA, sbsh[pl])), eh = fd_p2(FD_LOW);
                    v = cmk(fma((double)r.th, eh, (double)r.tl * el) * f1 * f2, fma((double)r.uh, eh, (double)r.ul * el) * f1 * f2);
                    const double xr = fma((double)r.rh, 0x1p64, (double)r.rl), xi = fma((double)r.ih, 0x1p64, (double)r.il);
                    ex = cmk(xr * f1 * f2 * f1 * f2, xi * f1 * f2 * f1 * f2);
                }
                A.vpart[(lp0 + pl) * (long long)G1 + g] = v;
                A.xpart[(lp0 + pl) * (long long)G1 + g] = ex;
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&rempty[rb]);
        }
        if (failed && lane == 0) atomicOr(A.status, STATUS_TIMEOUT);
    } else if (warp >= FDY_THREADS / 32) {
        // ---- digits of Y: unit (column cl, 8 K elements), a column's units side by side; the next
        // unit's values are under way while this one's digits are formed
        const int dt = tid - FDY_THREADS, h8 = A.N8 >> 3;
        const uint32_t rcp = 65536u / (uint32_t)n + 1u;               // cl / n for cl < 64
        const long long* Yw = A.Y + wl * G1 * (long long)n * 2 * A.N8;
        longlong2 nx[4];
        unsigned nm = 0;
        auto fetch = [&](int t, int c, int e) {
            const int cl = e >> 3, k8 = c * 8 + (e & 7);
            if (t >= t1 || cl >= min(GB, G1 - t * GB) * n || k8 >= 2 * h8) return;
            const int ri = k8 >= h8;
            const longlong2* src = reinterpret_cast<const longlong2*>(
                Yw + ((long long)(t * GB * n + cl) * 2 + ri) * A.N8) + (k8 - (ri ? h8 : 0));
#pragma unroll
            for (int q = 0; q < 4; ++q) nx[q] = __ldg(src + q * h8);
            nm = __ldg(ymx + t * GB + (int)(((uint32_t)cl * rcp) >> 16));
        };
        fetch(t0, 0, dt);
        int ub = 0;
        for (int t = t0; t < t1 && !failed; ++t) {
            const int nunit = min(GB, G1 - t * GB) * n * 8;
            for (int c = 0; c < KC; ++c, ++ub) {
                uint8_t* slot = sm + (size_t)(ub & 1) * bbytes;
                bool ok = true;
                if (ub >= 2 && lane == 0) ok = fd_wait(&pp.bempty[ub & 1], (uint32_t)(((ub >> 1) - 1) & 1), lim, fail);
                if (__any_sync(0xffffffffu, !ok)) { failed = true; break; }
                for (int e = dt; ; e += FDZ_DIG) {
                    const int cl = e >> 3, u = e & 7;
                    const bool have = e < nunit && c * 8 + u < 2 * h8;  // beyond K no K step reads
                    long long F[8];
                    const int k = fd_yshift<BITS>(nm);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        F[2 * q] = nx[q].x;
                        F[2 * q + 1] = nx[q].y;
                    }
                    const bool more = e + FDZ_DIG < nunit;
                    if (more) fetch(t, c, e + FDZ_DIG);
                    else fetch(c + 1 < KC ? t : t + 1, c + 1 < KC ? c + 1 : 0, dt);
                    if (have) {
                        if (k >= 0) {
#pragma unroll
                            for (int q = 0; q < 8; ++q) F[q] = (long long)((unsigned long long)F[q] << k);
                        } else {
#pragma unroll
                            for (int q = 0; q < 8; ++q) F[q] = (F[q] + (1ll << (-k - 1))) >> (-k);
                        }
                        dg64_unit<BITS>(F, [&](int q, uint4 v) { *reinterpret_cast<uint4*>(slot + fd_swz(q * NT + cl, u)) = v; });
                    }
                    if (!more) break;
                }
                tc::fence_proxy_async();                              // the digits to the tensor cores
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&pp.bfull[ub & 1]);
            }
        }
        if (failed && lane == 0) atomicOr(A.status, STATUS_TIMEOUT);
    } else {
        // ---- epilogue: ngrp groups of warps take the tiles in turn, so that one group's reading of
        // tensor memory and the other's traces, both bound by latencies, overlap
        const int gw = FD_EPI / 32 / A.ngrp;                          // warps of a group
        const int grp = (warp - 2) / gw, set = (warp - 2 - grp * gw) >> 2, nset = gw >> 2;
        const int et = tid - 64 - grp * gw * 32, quad = warp & 3;
        const int r = 32 * quad + lane, q64 = r & 63;
        const bool row_ok = q64 < np * n;
        const int sh = row_ok ? sbsh[q64 / n] : 0;
        const int xs = min(FD_XTRA, sh), shx = sh - xs;
        const float rnd = (float)((shx > 0 ? 1 << (shx - 1) : 0) + (xs > 0 ? 1 << (sh - 1) : 0));
        const uint32_t lb = taddr + ((uint32_t)(32 * quad) << 16);
        const int T = A.T;
        const int combo = et / T, sub = et % T;
        const int pl = combo / GB, gl = combo % GB;
        const bool mine = combo < combos && pl < np;
        int2* Mg = Ms + grp * 128 * (ldc + 1);
        const int2* R0 = Mg + (size_t)(mine ? pl * n : 0) * ldc + (mine ? gl * n : 0);
        const int2* I0 = R0 + (size_t)64 * ldc;
        const int px = mine ? min(FD_XTRA, sbsh[pl]) : 0, prx = px > 0 ? 1 << (px - 1) : 0;
        // the stored 2^(x - 1) of a thread's diagonal entries, taken off their sum: a low half may be at the end of 32 bits
        const long long bias = mine && sub < n ? (long long)prx * ((n - sub + T - 1) / T) : 0;
        for (int t = t0 + grp; t < t1; t += A.ngrp) {
            const int tt = t - t0;
            const uint32_t tbuf = nbuf == 2 && (tt & 1) ? (uint32_t)fd_cols(D, NT) : 0u;
            const int gn = min(GB, G1 - t * GB), ncol = gn * n;
            bool ok = true;
            if (lane == 0) {
                ok = fd_wait(&pp.dfull[tt & 1], (uint32_t)((tt >> 1) & 1), lim, fail);
                if (tt >= 2 && ok) ok = fd_wait(&rempty[tt & 1], (uint32_t)(((tt >> 1) - 1) & 1), lim, fail);
            }
            if (fd_group_sync_or(1 + grp, gw * 32, !ok)) { failed = true; break; }   // also: Mg is free
            tc::fence_after_sync();
            // the orders added: Z' = high 2^(FD_LOW + x) + low, |low| <= 2^(FD_LOW + x - 1)
            for (int col = 4 * set; col < ncol; col += 4 * nset) {    // uniform
                float v[D][4];
#pragma unroll
                for (int q = 0; q < D; ++q) tc::tmem_ld4(lb + tbuf + (uint32_t)(q * NT + col), v[q]);
                tc::tmem_ld_wait();
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float a[D];
#pragma unroll
                    for (int q = 0; q < D; ++q) a[q] = v[q][k];
                    const long long z = dg64_sum<BITS>(a, rnd) >> shx;
                    const int lo = (int)((uint32_t)z << (FD_XTRA - xs)) >> (FD_XTRA - xs);
                    const int hi = (int)((z - lo) >> (FD_LOW + xs));
                    if (row_ok && col + k < ncol) Mg[(size_t)r * ldc + col + k] = make_int2(hi, lo);
                }
            }
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&pp.dempty[tt & 1]);
            fd_group_sync(1 + grp, gw * 32);                          // Mg holds the tile
            long long th = 0, uh = 0, tl = 0, ul = 0, hr = 0, mr = 0, lr = 0, hm = 0, mm = 0, lm = 0;
            if (mine && gl < gn) {
                // sum over unordered pairs: Z_ab Z_ba once for a = b, twice otherwise; at most
                // 16 terms a thread keeps every sum below 2^62
                for (int u = sub; u < U; u += T) {
                    const uchar2 ab = tab[u];
                    const int o1 = ab.x * ldc + ab.y, o2 = ab.y * ldc + ab.x;
                    int2 xr = R0[o1], xi = I0[o1];
                    int2 yr = R0[o2], yi = I0[o2];
                    if (u < n) {
                        th += xr.x;
                        uh += xi.x;
                        tl += xr.y;
                        ul += xi.y;
                    }
                    xr.y >>= px; xi.y >>= px; yr.y >>= px; yi.y >>= px;
                    if (u >= n) {
                        xr.x *= 2; xr.y *= 2; xi.x *= 2; xi.y *= 2;
                    }
                    const int nxx = -xi.x, nxy = -xi.y;
                    hr += (long long)xr.x * yr.x; hr += (long long)nxx * yi.x;
                    mr += (long long)xr.x * yr.y; mr += (long long)xr.y * yr.x;
                    mr += (long long)nxx * yi.y; mr += (long long)nxy * yi.x;
                    lr += (long long)xr.y * yr.y; lr += (long long)nxy * yi.y;
                    hm += (long long)xr.x * yi.x; hm += (long long)xi.x * yr.x;
                    mm += (long long)xr.x * yi.y; mm += (long long)xr.y * yi.x;
                    mm += (long long)xi.x * yr.y; mm += (long long)xi.y * yr.x;
                    lm += (long long)xr.y * yi.y; lm += (long long)xi.y * yr.y;
                }
            }
            FdRed s;
            s.th = th;
            s.uh = uh;
            s.tl = tl - bias;
            s.ul = ul - bias;
            fd_join(hr, mr, lr, s.rh, s.rl);
            fd_join(hm, mm, lm, s.ih, s.il);
            for (int o = min(T, 32) >> 1; o > 0; o >>= 1) {
                s.th += __shfl_xor_sync(0xffffffffu, s.th, o);
                s.uh += __shfl_xor_sync(0xffffffffu, s.uh, o);
                s.tl += __shfl_xor_sync(0xffffffffu, s.tl, o);
                s.ul += __shfl_xor_sync(0xffffffffu, s.ul, o);
                fd_add(s.rh, s.rl, __shfl_xor_sync(0xffffffffu, s.rh, o), __shfl_xor_sync(0xffffffffu, s.rl, o));
                fd_add(s.ih, s.il, __shfl_xor_sync(0xffffffffu, s.ih, o), __shfl_xor_sync(0xffffffffu, s.il, o));
            }
            if (mine && (sub & 31) == 0) red[((tt & 1) * combos + combo) * parts + (sub >> 5)] = s;
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&rfull[tt & 1]);
        }
        if (failed && lane == 0) atomicOr(A.status, STATUS_TIMEOUT);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) tc::tmem_dealloc(taddr, 512);
}

// ---------------------------------------------------------------- per pair: v_g and E_L
// One warp per pair of the chunk (pair0 the first): v_g = sum_s Tr Z_s (g >= 1),
// E_L = sum_s Tr Z_{s,0} + 1/2 sum_g [v_g^2 - sum_s Tr Z_{s,g}^2].  With a list (w0 the chunk's
// first walker) pair i of a walker is its listed pair i.
__global__ void fd_finish_kernel(long long pair0, long long pairs, int P, long long w0, PairList list, int G, int two_spins,
                                 const double2* __restrict__ vp0, const double2* __restrict__ vp1,
                                 const double2* __restrict__ ex0, const double2* __restrict__ ex1,
                                 double2* __restrict__ vpair, double2* __restrict__ epair) {
    const long long p = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (p >= pairs) return;
    long long out = pair0 + p;
    if (list.count) {
        const long long w = w0 + p / P;
        const int i = (int)(p % P);
        if (i >= list.count[w]) return;
        out = list.items[list.base[w] + i];
    }
    const double2 *a = vp0 + p * (G + 1), *b = vp1 + p * (G + 1);
    const double2 *xa = ex0 + p * (G + 1), *xb = ex1 + p * (G + 1);
    double2 s = cmk(0.0, 0.0);
    for (int g = 1 + lane; g <= G; g += 32) {
        double2 v = a[g], x = xa[g];
        if (two_spins) {
            v = cadd(v, b[g]);
            x = cadd(x, xb[g]);
        }
        vpair[out * G + (g - 1)] = v;
        const double2 v2 = cmul(v, v);
        s.x += v2.x - x.x;
        s.y += v2.y - x.y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
    }
    if (lane == 0) {
        double2 e = a[0];
        if (two_spins) e = cadd(e, b[0]);
        epair[out] = cmk(e.x + 0.5 * s.x, e.y + 0.5 * s.y);
    }
}

// ---------------------------------------------------------------- host side
namespace {

struct FdSpin {
    int n, PB, MT, GB, NT, nbuf, ngrp, NCT, S, T;
    size_t smem, aimg;          // A image bytes per walker
};

struct FdShape {
    int bits, D, N8, KC, zsteps, KCX, ysteps, NTY, ybuf, yres, JT, SY, G1, zbits;
    size_t smem_y;
    FdSpin sp[2];
    long long WB;               // walkers per chunk
    size_t ximg, pimg, y[2], aimg[2];
};

inline int fd_up(int x, int m) { return (x + m - 1) / m * m; }

size_t fd_z_smem(int D, int NT, int GB, int n, int PB, int T, int S, int ngrp) {
    return 1024 + 2 * (size_t)fd_bslot(D, NT) + (size_t)S * FD_ADIG + (size_t)ngrp * 128 * (((GB * n) | 1) + 1) * 8 +
           (size_t)PB * GB * (T > 32 ? T / 32 : 1) * 2 * sizeof(FdRed) + (size_t)fd_up(n * (n + 1), 16);
}

// Clocks per column of a column tile, by which tiles are compared (K step of 16): the
// MMAs, or what they and the copies move through shared memory at 128 bytes per
// clock (A once per MMA, B, and both operands' way in), and, with one accumulator
// buffer, the epilogue's reading of the tile, which no MMA overlaps then.
double fd_tile_cost(int D, int NT, int nbuf, int ngrp, int used, int ksteps) {
    const int pr = D * (D + 1) / 2, maxblk = fd_maxblk(NT);
    const int mmas = D + std::max(0, D - maxblk);
    const double mma = pr * NT * 0.5;
    const double smem = 32.0 * mmas + pr * NT * 0.25 + 32.0 * D + D * NT * 0.25;
    const double tile = ksteps * std::max(mma, smem), drain = ngrp * (1000.0 + 60.0 * used), trace = 2000.0 + 60.0 * used;
    return std::max(tile + (nbuf == 2 ? 0.0 : drain), (drain + trace) / ngrp) / used;
}

bool fd_spin(const FdShape& s, int n, int P, FdSpin& f) {
    f.n = n;
    if (n < 1 || n > 64) return false;
    f.PB = std::min(64 / n, P);
    f.MT = (P + f.PB - 1) / f.PB;
    f.aimg = (size_t)f.MT * s.KC * s.D * FD_ADIG;
    const int U = n * (n + 1) / 2;
    double best = 0.0;
    // column tiles whose accumulators fit tensor memory (twice: the epilogue then overlaps the
    // next tile's MMAs), whose (pair, g) sums fit the epilogue's threads, and whose digits,
    // A ring and Z' fit shared memory; the cheapest per column
    for (int gb = std::min(64 / n, s.G1); gb >= 1; --gb) {
        const int NT = fd_up(gb * n, 8), cols = fd_cols(s.D, NT);
        if (cols > 512 || f.PB * gb > FD_EPI / 2 || s.D > 2 * fd_maxblk(NT)) continue;
        const int nbuf = 2 * cols <= 512 ? 2 : 1;
        for (int ngrp = 2; ngrp >= 1; --ngrp) {
            int T = 1;
            while (f.PB * gb * T * 2 <= FD_EPI / ngrp) T *= 2;
            if ((U + T - 1) / T > 16) continue;
            int S = FD_MAXS;
            while (S >= 3 && fd_z_smem(s.D, NT, gb, n, f.PB, T, S, ngrp) > FD_SMEM_MAX) --S;
            if (S < 3) continue;
            const double c = fd_tile_cost(s.D, NT, nbuf, ngrp, gb * n, s.zsteps);
            if (best == 0.0 || c < best) {
                best = c;
                f.GB = gb; f.NT = NT; f.nbuf = nbuf; f.ngrp = ngrp; f.S = S; f.T = T;
                f.smem = fd_z_smem(s.D, NT, gb, n, f.PB, T, S, ngrp);
                f.NCT = (s.G1 + gb - 1) / gb;
            }
        }
    }
    return best > 0.0;
}

// Digits by the length of the products: K = 2 N8 of GEMM-Z (and N of GEMM-Y) terms at most.
bool fd_shape(int N, int nu, int nd, int G, long long W, int P, size_t chunk, FdShape& s) {
    if (N < 1 || nu < 1 || nd < 0 || nd > nu || W < 1 || P < 1) return false;
    s.N8 = fd_up(N, 8);
    // GEMM-Y: with one K chunk the A digits stay in shared memory and two accumulator
    // buffers overlap the epilogue; longer products stream them past wider tiles
    if (2 * s.N8 <= Dg64<8>::MAXK) { s.bits = 8; s.D = Dg64<8>::D; s.NTY = 32; s.ybuf = 2; s.yres = 1; }
    else if (2 * s.N8 <= Dg64<7>::MAXK) { s.bits = 7; s.D = Dg64<7>::D; s.NTY = 48; s.ybuf = 1; s.yres = 0; }
    else return false;
    s.G1 = G + 1;
    s.zsteps = 2 * s.N8 / 16;
    s.KC = (s.zsteps + 3) / 4;
    s.ysteps = fd_up(N, 16) / 16;
    s.KCX = (s.ysteps + 3) / 4;
    s.JT = (s.N8 + s.NTY - 1) / s.NTY;
    s.zbits = 56;
    if (!fd_spin(s, nu, P, s.sp[0])) return false;
    if (nd > 0 && !fd_spin(s, nd, P, s.sp[1])) return false;
    if (nd == 0) s.sp[1] = FdSpin{};
    for (s.SY = s.yres ? s.KCX * s.D : FD_MAXS; s.SY >= 2; --s.SY) {
        s.smem_y = 1024 + 2 * (size_t)fd_bslot(s.D, s.NTY) + (size_t)s.SY * FD_ADIG;
        if (s.smem_y <= FD_SMEM_MAX) break;
    }
    if (s.SY < (s.yres ? s.KCX * s.D : 2)) return false;
    s.ximg = (size_t)s.G1 * s.JT * s.KCX * s.D * s.NTY * 128;
    // Y and A digits of as many walkers as `chunk` bytes hold
    size_t per = 0;
    for (int q = 0; q < 2; ++q) {
        const size_t y = (size_t)s.G1 * s.sp[q].n * 2 * s.N8 * 8;
        per += y + s.sp[q].aimg + (size_t)P * 32 * s.G1;
    }
    s.WB = std::max(1LL, std::min(W, (long long)(chunk / per)));
    for (int q = 0; q < 2; ++q) {
        s.y[q] = (size_t)s.WB * s.G1 * s.sp[q].n * 2 * s.N8 * 8;
        s.aimg[q] = (size_t)s.WB * s.sp[q].aimg;
    }
    const int nt = nu + nd;
    s.pimg = (size_t)((s.WB * 2 * nt + 127) / 128) * s.KCX * s.D * FD_ADIG;
    return (s.WB * 2 * nt + 127) / 128 * 64 < INT32_MAX;
}

size_t fd_align(size_t x) { return (x + 255) & ~(size_t)255; }

struct FdWork {
    uint8_t *ximg, *pimg, *aimg[2];
    int *xexp, *cexp, *bexp[2], *bsh[2];
    long long* y[2];
    unsigned int *ymax, *bad;   // cleared together
    double2 *vpart[2], *xpart[2];
    size_t total;
};

FdWork fd_carve(void* work, const FdShape& s, int P) {
    FdWork w{};
    uint8_t* p = static_cast<uint8_t*>(work);
    auto take = [&](size_t bytes) {
        uint8_t* r = p;
        p += fd_align(bytes);
        w.total += fd_align(bytes);
        return r;
    };
    const size_t wp = (size_t)s.WB * P;
    w.ximg = take(s.ximg);
    w.xexp = reinterpret_cast<int*>(take((size_t)s.G1 * 4));
    w.pimg = take(s.pimg);
    w.cexp = reinterpret_cast<int*>(take((size_t)s.WB * (s.sp[0].n + s.sp[1].n) * 4));
    w.bad = reinterpret_cast<unsigned int*>(take((size_t)s.WB * (2 * s.G1 + 1) * 4));
    w.ymax = w.bad + s.WB;
    for (int q = 0; q < 2; ++q) {
        if (s.sp[q].n == 0) continue;
        w.y[q] = reinterpret_cast<long long*>(take(s.y[q]));
        w.aimg[q] = take(s.aimg[q]);
        w.bexp[q] = reinterpret_cast<int*>(take(wp * 4));
        w.bsh[q] = reinterpret_cast<int*>(take(wp * 4));
        w.vpart[q] = reinterpret_cast<double2*>(take(wp * s.G1 * 16));
        w.xpart[q] = reinterpret_cast<double2*>(take(wp * s.G1 * 16));
    }
    return w;
}

int fd_sms() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 152;
    return std::max(1, sms);
}

template <int BITS>
cudaError_t fd_run(cudaStream_t st, const Dims& d, const FdShape& s, const FdWork& w, const double2* Bm,
                   const double2* phi, double2* vpair, double2* epair, int* status, const PairList& list) {
    const long long W = d.pairs / d.P;
    const int sms = fd_sms();
    cudaError_t e = raise_smem_limit((const void*)fd_y_kernel<BITS>, s.smem_y);
    for (int q = 0; q < 2 && e == cudaSuccess; ++q)
        if (s.sp[q].n) e = raise_smem_limit((const void*)contract_fp64d_kernel<BITS>, s.sp[q].smem);
    size_t bsm[2] = {0, 0};                                            // B columns of a block, 0: not staged
    for (int q = 0; q < 2 && e == cudaSuccess; ++q) {
        const size_t b = (size_t)s.sp[q].PB * s.sp[q].n * (d.N | 1) * sizeof(double2);
        if (b > 220 * 1024) continue;
        bsm[q] = b;
        if (b) e = raise_smem_limit((const void*)fd_b_image_kernel<BITS>, b);
    }
    if (e != cudaSuccess) return e;
    for (long long w0 = 0; w0 < W; w0 += s.WB) {
        const long long wb = std::min(s.WB, W - w0);
        const long long rt = (wb * 2 * d.nt + 127) / 128;
        if ((e = cudaMemsetAsync(w.bad, 0, (size_t)(s.WB + wb * 2 * s.G1) * 4, st)) != cudaSuccess) return e;
        fd_phi_image_kernel<BITS><<<(unsigned)rt, 256, 0, st>>>(d.N, d.nt, s.KCX, w0, wb, phi, w.pimg, w.cexp, w.bad);
        count_launches(1);
        // runs of matrices: about four blocks per SM, at least four matrices each
        const int want = (int)std::max(1LL, std::min<long long>((4LL * sms + rt - 1) / rt, (s.G1 + 3) / 4));
        const int gpb = (s.G1 + want - 1) / want, ngb = (s.G1 + gpb - 1) / gpb;
        fd_y_kernel<BITS><<<(unsigned)(rt * ngb), FDY_THREADS, s.smem_y, st>>>(
            s.N8, d.nu, d.nd, s.G1, s.KCX, s.ysteps, s.JT, s.NTY, s.ybuf, s.SY, gpb, ngb, s.yres, wb, w.pimg, w.ximg, w.y[0], w.y[1],
            w.ymax, status, d.wait_polls, list.count ? list.count + w0 : nullptr);
        count_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        for (int q = 0; q < 2; ++q) {
            const FdSpin& f = s.sp[q];
            if (f.n == 0) continue;
            fd_b_image_kernel<BITS><<<(unsigned)(wb * f.MT), FDB_T, bsm[q], st>>>(d.N, s.N8, d.nt, q ? d.nu : 0, f.n, d.P, f.PB,
                                                                         f.MT, s.KC, s.zbits, w0, w.cexp, Bm, w.aimg[q],
                                                                         w.bexp[q], w.bsh[q], list, bsm[q] > 0);
            FdZArgs a;
            a.n = f.n; a.G1 = s.G1; a.N8 = s.N8; a.KC = s.KC; a.ksteps = s.zsteps; a.NT = f.NT; a.nbuf = f.nbuf; a.ngrp = f.ngrp; a.GB = f.GB;
            a.NCT = f.NCT; a.P = d.P; a.PB = f.PB; a.MT = f.MT; a.S = f.S; a.T = f.T;
            // column tiles of a block: FD_RUN at least, so that the waves of blocks (tensor memory holds one per SM) take the
            // least time, a block's start as one tile; a list's blocks are not known here, some eight per SM then.
            // Short products (one K chunk) are bound by the traces: a last tile of few pairs counts for those.  Against
            // every other number at 22 shapes the choice is within 1 % of the best at 20, 2 % at the others.
            const long long wm = wb * f.MT;
            const long long share = s.KC == 1 ? (wb * (d.P - (f.MT - 1) * f.PB) + f.PB - 1) / f.PB : wb;
            const long long full = wb * (f.MT - 1) + share;
            const int most = (int)std::max(1LL, std::min<long long>((f.NCT + FD_RUN - 1) / FD_RUN,
                                                                    ((list.count ? 8LL : 64LL) * sms + wm - 1) / wm));
            long long best = 0;
            for (int runs = list.count ? most : 1; runs <= most; ++runs) {
                const int run = (f.NCT + runs - 1) / runs, n = (f.NCT + run - 1) / run;
                const long long cost = (full * n + sms - 1) / sms * (run + 1);
                if (best == 0 || cost < best) {
                    best = cost;
                    a.RUN = run;
                    a.NRUN = n;
                }
            }
            a.Bimg = w.aimg[q]; a.bexp = w.bexp[q]; a.bsh = w.bsh[q]; a.bad = w.bad; a.xexp = w.xexp;
            a.Y = w.y[q]; a.ymax = w.ymax + (size_t)q * s.G1;
            a.vpart = w.vpart[q]; a.xpart = w.xpart[q]; a.status = status;
            a.listed = list.count ? list.count + w0 : nullptr;
            contract_fp64d_kernel<BITS><<<(unsigned)(wm * a.NRUN), FDZ_THREADS, f.smem, st>>>(a, d.wait_polls);
            count_launches(2);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        const long long pairs = wb * d.P;
        fd_finish_kernel<<<(unsigned)((pairs * 32 + 255) / 256), 256, 0, st>>>(
            w0 * d.P, pairs, d.P, w0, list, d.G, d.nd > 0, w.vpart[0], d.nd > 0 ? w.vpart[1] : w.vpart[0], w.xpart[0],
            d.nd > 0 ? w.xpart[1] : w.xpart[0], vpair, epair);
        count_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <int BITS>
cudaError_t fd_prepare(cudaStream_t st, int N, const FdShape& s, const FdWork& w, const double* h, const double* L) {
    fd_xexp_kernel<BITS><<<(unsigned)s.G1, 256, 0, st>>>(N, h, L, w.xexp);
    fd_x_image_kernel<BITS><<<1024, 256, 0, st>>>(N, s.KCX, s.JT, s.NTY, s.G1, h, L, w.xexp, w.ximg);
    count_launches(2);
    return cudaGetLastError();
}

}  // namespace

bool contract_fp64d_supported(int N, int nu, int nd, int G, long long W, int P) {
    FdShape s;
    return fd_shape(N, nu, nd, G, W, P, FD_CHUNK, s);
}

size_t contract_fp64d_work_bytes(int N, int nu, int nd, int G, long long W, int P, size_t chunk) {
    FdShape s;
    if (!fd_shape(N, nu, nd, G, W, P, chunk, s)) return 0;
    return fd_carve(nullptr, s, P).total;
}

cudaError_t contract_fp64d_prepare(cudaStream_t st, const Dims& d, const double* h, const double* L, void* work, size_t chunk) {
    FdShape s;
    if (!work || !fd_shape(d.N, d.nu, d.nd, d.G, d.pairs / d.P, d.P, chunk, s)) return cudaErrorInvalidValue;
    const FdWork w = fd_carve(work, s, d.P);
    return s.bits == 8 ? fd_prepare<8>(st, d.N, s, w, h, L) : fd_prepare<7>(st, d.N, s, w, h, L);
}

cudaError_t contract_fp64d(cudaStream_t st, const Dims& d, void* work, const double2* Bm, const double2* phi,
                           double2* vpair, double2* epair, int* status, const PairList& list, size_t chunk) {
    FdShape s;
    if (!work || d.P < 1 || d.pairs % d.P != 0) return cudaErrorInvalidValue;
    if (d.pairs == 0) return cudaSuccess;
    if (!fd_shape(d.N, d.nu, d.nd, d.G, d.pairs / d.P, d.P, chunk, s)) return cudaErrorInvalidValue;
    const FdWork w = fd_carve(work, s, d.P);
    return s.bits == 8 ? fd_run<8>(st, d, s, w, Bm, phi, vpair, epair, status, list)
                       : fd_run<7>(st, d, s, w, Bm, phi, vpair, epair, status, list);
}

}  // namespace afq
