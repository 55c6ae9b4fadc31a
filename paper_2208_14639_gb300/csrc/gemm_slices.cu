// The FP64 product C = A B^T of gemm_f64.cu on the tensor cores: both operands are cut into eight
// 8-bit integer slices (an Ozaki-style split) whose products tcgen05 kind::f16 sums exactly in FP32.
//
// GB300 runs FP64 at 1/64 of the FP32 rate, so an FP64 product of the AO assembly is bound by that
// pipe (hexamer, 54 trials, 78 basis functions: 154 ms at 57 % of it, 88 ms at all of it); the 36
// exact slice products take 36 FP16 flops per FP64 one, on a unit 1,500 times faster.
//
// Slices.  In a block of 128 k, a row of A or of B is scaled by the power of two of its largest
// element: x = 2^(E - 5) sum_p d_p 2^(-8 p), p = 0 .. 7, every digit d_p an integer in [-128, 127]
// (|d_0| <= 64), formed in integer arithmetic from the bits of x rounded to 2^(E - 61): exact down to
// 2^-8 of the row's largest element, then with an absolute error of 2^-62 of it.  The products with
// p + q <= 7 are formed; those left out are below 7 x 2^-60 of the two scales (rms 2^-60).  Each
// level l = p + q has its own accumulator over the block: a sum of integers below 2^23.9, which
// FP32 holds exactly whatever order or truncation the tensor core uses.
//
// Sums.  A block's levels are combined into two exact integers and these into one FP64 number, which
// is scaled by the two powers of two and added in FP64: two roundings per 128 k, where a chain of
// FMAs rounds at every k.  Against 80-bit and wider sums the assembled matrices are off by 1.5e-16 to
// 9e-16 in norm (1,500 to 40,000 points), those of the FMA chains by 3e-16 to 3.5e-15.
//
// The cuts are relative to the two rows' largest elements in a block, not to their products: an element
// of C is off by about 2^-56 of the sum over the blocks of max |a| max |b|.  With the points in grid order
// that is below the rounding (CPU model of the slices, water on 65,000 points with an oxygen core
// exponent of 116,506 and a diffuse 0.02: every element within 2.6e-15 of its sum of absolute terms, FP64
// within 1.7e-15).  With an atom's points in random order, so that core and outer points share blocks,
// elements between a core and a diffuse function are off by up to 1e-12 of theirs (in norm still 6e-16).
// Rows that mix columns of unlike scale in every block, as the two-column factors of the nuclear
// derivative of F do, do not come here.
//
// A row's 128 elements of which one is not finite, or 2^512 and more (the scales of two rows could
// overflow), have no digits: its exponent is stored as kGsPlain, its products are left out, and the
// reduction forms them by FP64 FMA, so that NaN and infinities end up where an FP64 product puts them.
// (At the other end block sums below 2^-978 are zero.)
//
// A CTA owns a 128 x 64 tile of C and a range of blocks.  Eight warps cut both operands' tiles of
// 32 k (8 rows per warp and pass, loads of 64 contiguous bytes; the rows' E from a pass of its own)
// into swizzled shared memory, double-buffered, while one thread issues the 72 MMAs of the 32 k
// before; once a block they combine its accumulators.  Per 128 k the MMAs take 14,000 cycles and
// the combination (four FP64 operations an element) up to 12,000; the eight levels' accumulators fill
// the TMEM (8 x 64 columns).  Measured: 131,008 points x 78 x 936 2.2 ms (FMA kernel 34), tensor pipe
// 23 %, issue 31 %: what is left is the latency of cutting, MMAs and combination in turn.
#include <cmath>
#include <cuda_fp16.h>

#include "common.cuh"
#include "kernels.hpp"
#include "tc.cuh"

namespace vv10 {

namespace {

constexpr int kGsM = 128, kGsN = 64, kGsK = 32;  // tile of C, k per stage
constexpr int kGsBlk = 4;                        // stages per block (one scale per row)
constexpr int kGsSlices = 8;
constexpr int kGsBig = 1023 + 511;               // largest biased exponent that is cut into digits
constexpr int kGsPlain = -4096;                  // the row's block is left to the reduction
constexpr int kGsWarps = 8;                      // worker warps; warp 8 issues the MMAs
constexpr int kGsThreads = 12 * 32;              // (three warps a scheduler: 168 registers a thread)
constexpr uint32_t kGsABytes = kGsM * 64, kGsBBytes = kGsN * 64;  // one slice: 64-byte rows
constexpr uint32_t kGsBufBytes = kGsSlices * (kGsABytes + kGsBBytes);
constexpr uint32_t kGsBarOff = 2 * kGsBufBytes;
constexpr uint32_t kGsSmem = kGsBarOff + 256 + 1024;  // barriers, slack for the 1024-B alignment

struct GsArgs {
    int M, N;
    int64_t K;
    int32_t n_blk, per_split;    // blocks in all, and of one split
    const double *A, *B;
    int64_t lda, ldb;
    const int32_t *ea, *eb;      // [block][row] biased exponent of the row's largest |element|, or kGsPlain
    int32_t* plain;              // [split][tile of C]: whether a row of its block range is kGsPlain
    double* part;                // [split][N][M]
    int* err;
};

__device__ __forceinline__ bool gs_wait(uint64_t* bar, uint32_t parity, int* err, volatile int* abort_flag) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > kSpinCycles) {
            atomicOr(err, DEVERR_TIMEOUT);
            *abort_flag = 1;
            return false;
        }
    }
    return true;
}

// Rows `row0 + (lane & 7)` of a tile (8 rows of this warp) x a stage's 32 k: slices into smem (slice p
// at base + p slice_bytes).  X: element (row, k) at k ld + row; emax: the block's exponents.  Returns
// whether this lane's row is kGsPlain.
__device__ __forceinline__ bool gs_cut(const double* __restrict__ X, int64_t ld, int rows, int first,
                                       int row0, int64_t k0, int64_t K, const int32_t* __restrict__ emax,
                                       uint8_t* base, uint32_t slice_bytes) {
    const int lane = threadIdx.x & 31;
    const int r = row0 + (lane & 7), kq = lane >> 3;
    double x[8];
    const int e = first + r < rows ? emax[first + r] : kGsPlain;
    const bool real = e >= 0;  // others: zeros
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int64_t k = k0 + 8 * kq + q;
        x[q] = real && k < K ? X[k * ld + first + r] : 0.0;
    }
    // digits + 128 in the bytes of b (byte 7 - p holds digit p)
    uint32_t lo[8], hi[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int h = __double2hiint(x[q]), ex = (h >> 20) & 0x7ff;
        uint64_t m = (static_cast<uint64_t>((h & 0xfffff) | 0x100000) << 41) |
                     (static_cast<uint64_t>(static_cast<uint32_t>(__double2loint(x[q]))) << 9);
        const int sh = min(e - ex, 63);
        m = ex == 0 ? 0 : (m + ((uint64_t(1) << sh) >> 1)) >> sh;  // to nearest (ties away from zero)
        const uint64_t b = (h < 0 ? 0 - m : m) + 0x8080808080808080ull;
        lo[q] = static_cast<uint32_t>(b);
        hi[q] = static_cast<uint32_t>(b >> 32);
    }
    const uint32_t at = smem_u32(base) + r * 64 + ((kq ^ ((r >> 1) & 3)) << 4);  // 64-byte swizzle
#pragma unroll
    for (int p = 0; p < kGsSlices; ++p) {
        const int i = 7 - p;  // byte
        uint32_t w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t a = i < 4 ? lo[2 * q] : hi[2 * q], c = i < 4 ? lo[2 * q + 1] : hi[2 * q + 1];
            const uint32_t sel = static_cast<uint32_t>((i & 3) | ((i & 3) << 4) | ((4 + (i & 3)) << 8) | ((4 + (i & 3)) << 12));
            // FP16 of bits 0x6400 + byte is 1024 + byte: minus 1152 leaves the digit, exactly
            const uint32_t t = (__byte_perm(a, c, sel) & 0x00ff00ffu) | 0x64006400u;
            const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&t), __half2half2(__ushort_as_half(0x6480)));
            w[q] = *reinterpret_cast<const uint32_t*>(&v);
        }
        tc::st_shared_v4(at + p * slice_bytes, w[0], w[1], w[2], w[3]);
    }
    return !real && first + r < rows;
}

__global__ void __launch_bounds__(kGsThreads, 1) k_gemm_slices(GsArgs args) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kGsBarOff);
    uint64_t* full = bars;           // [2] a stage's slices are in shared memory
    uint64_t* mma_done = bars + 2;   // [2]
    uint64_t* acc_free = bars + 4;   // the accumulators of a block are read
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 5);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + 6);
    volatile int* plain_flag = abort_flag + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        mbar_init(&full[0], kGsWarps);
        mbar_init(&full[1], kGsWarps);
        mbar_init(&mma_done[0], 1);
        mbar_init(&mma_done[1], 1);
        mbar_init(acc_free, kGsWarps);
        *abort_flag = 0;
        *plain_flag = 0;
        fence_mbar_init();
    }
    if (warp == kGsWarps) tc::tmem_alloc(tmem_slot, 512);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tmem_slot;
    const int m0 = blockIdx.x * kGsM, n0 = blockIdx.y * kGsN;
    const int b0 = blockIdx.z * args.per_split;
    const int ns = kGsBlk * min(args.per_split, args.n_blk - b0);  // stages, >= kGsBlk

    if (warp < kGsWarps) {
        const int quad = warp & 3, half = warp >> 2;
        const int m = m0 + quad * 32 + lane;
        const bool rows = m0 + quad * 32 < args.M;  // this warp's lanes hold rows of C
        double acc[32];
#pragma unroll
        for (int c = 0; c < 32; ++c) acc[c] = 0.0;
        auto combine = [&](int j) -> bool {  // block j (from 0): its accumulators into the sums
            const int s = kGsBlk * j + kGsBlk - 1;
            const bool got = gs_wait(&mma_done[s & 1], (s >> 1) & 1, args.err, abort_flag);
            if (!__all_sync(0xffffffffu, got)) return false;
            tc::fence_after();
            if (rows) {
                const int64_t blk = b0 + j;
                const int er = m < args.M ? args.ea[blk * args.M + m] - 2 * 1028 - 24 + 1023 : 0;
                const int32_t* ec = args.eb + blk * args.N + n0 + half * 32;
                const uint32_t t0 = tmem + (static_cast<uint32_t>(quad * 32) << 16) + half * 32;
#pragma unroll
                for (int c0 = 0; c0 < 32; c0 += 4) {
                    uint32_t r[kGsSlices][4];
#pragma unroll
                    for (int l = 0; l < kGsSlices; ++l) tc::ld_x4(t0 + l * kGsN + c0, r[l]);
                    tc::wait_ld();
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        auto L = [&](int l) { return static_cast<int64_t>(__float2int_rn(__uint_as_float(r[l][u]))); };
                        // L0 + L1 2^-8 + ... + L7 2^-56 in two exact integers, units of 2^-24 and
                        // 2^-56, below 2^44 and 2^48; as the low bits of 1.5 x 2^52 they are FP64
                        const int64_t vh = (L(0) << 24) + (L(1) << 16) + (L(2) << 8) + L(3);
                        const int64_t vl = (L(4) << 24) + (L(5) << 16) + (L(6) << 8) + L(7);
                        const double dh = __longlong_as_double(0x4338000000000000ll + vh) - 0x1.8p52;
                        const double dl = __longlong_as_double(0x4338000000000000ll + vl) - 0x1.8p52;
                        const double x = fma(dl, 0x1p-32, dh);
                        // times 2^(E_a + E_b - 2 (1023 + 5) - 24)
                        int e = er + (n0 + half * 32 + c0 + u < args.N ? ec[c0 + u] : 0);
                        e = e < 0 ? 0 : e;  // (kGsPlain: 0; at most 2 kGsBig - 1057)
                        acc[c0 + u] = fma(x, __hiloint2double(e << 20, 0), acc[c0 + u]);
                    }
                }
            }
            tc::fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_free);
            return true;
        };
        bool ok = true, plain = false;
        for (int s = 0; s < ns && ok; ++s) {
            const int64_t blk = b0 + s / kGsBlk;
            if (s >= 2) {  // the buffer is free once the MMAs of stage s - 2 are done
                const bool got = gs_wait(&mma_done[s & 1], ((s - 2) >> 1) & 1, args.err, abort_flag);
                if (!__all_sync(0xffffffffu, got)) {
                    ok = false;
                    break;
                }
            }
            uint8_t* buf = smem + (s & 1) * kGsBufBytes;
            const int64_t k0 = (blk * kGsBlk + s % kGsBlk) * kGsK;
            for (int r0 = 8 * warp; r0 < kGsM; r0 += 8 * kGsWarps)
                if (m0 + r0 < args.M || s < 2)  // rows past M: zeros, once per buffer
                    plain |= gs_cut(args.A, args.lda, args.M, m0, r0, k0, args.K, args.ea + blk * args.M, buf, kGsABytes);
            plain |= gs_cut(args.B, args.ldb, args.N, n0, 8 * warp, k0, args.K, args.eb + blk * args.N,
                            buf + kGsSlices * kGsABytes, kGsBBytes);
            tc::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[s & 1]);
            if (s > 0 && s % kGsBlk == 0) ok = combine(s / kGsBlk - 1);
        }
        if (plain) *plain_flag = 1;  // every writer the same value
        if (ok && combine(ns / kGsBlk - 1) && m < args.M) {
            double* out = args.part + static_cast<int64_t>(blockIdx.z) * args.M * args.N + m;
#pragma unroll
            for (int c = 0; c < 32; ++c) {
                const int n = n0 + half * 32 + c;
                if (n < args.N) out[static_cast<int64_t>(n) * args.M] = acc[c];
            }
        }
        tc::wait_ld();
    } else if (warp == kGsWarps && lane == 0) {
        const uint32_t idesc = tc::idesc_f16(kGsM, kGsN);
        int s = 0;
        for (; s < ns; ++s) {
            const int b = s & 1, first = s % kGsBlk == 0;
            if (!gs_wait(&full[b], (s >> 1) & 1, args.err, abort_flag)) break;
            if (first && !gs_wait(acc_free, ((s / kGsBlk) & 1) ^ 1, args.err, abort_flag)) break;
            tc::fence_after();
            const uint32_t base = smem_u32(smem + b * kGsBufBytes);
            for (int ks = 0; ks < 2; ++ks)
#pragma unroll
                for (int p = 0; p < kGsSlices; ++p)
#pragma unroll
                    for (int q = 0; p + q < kGsSlices; ++q) {
                        const uint64_t da = tc::sdesc_kmajor_sw64(base + p * kGsABytes) + 2u * ks;
                        const uint64_t db = tc::sdesc_kmajor_sw64(base + kGsSlices * kGsABytes + q * kGsBBytes) + 2u * ks;
                        tc::mma_f16_ss(tmem + (p + q) * kGsN, da, db, idesc, !first || ks > 0 || p > 0);
                    }
            tc::commit(&mma_done[b]);
        }
        // every MMA finished before TMEM is released (normally the workers have seen to it)
        if (s > 0) mbar_wait(&mma_done[(s - 1) & 1], ((s - 1) >> 1) & 1, args.err);
    }
    tc::fence_before();
    __syncthreads();
    if (threadIdx.x == 0)
        args.plain[(blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = *plain_flag;
    if (warp == kGsWarps) {
        tc::fence_after();
        tc::tmem_dealloc(tmem, 512);
    }
}

// emax[block][row] = biased exponent of the row's largest |element| in the block's 128 k, or kGsPlain.
__global__ void __launch_bounds__(256) k_exp_max(const double* __restrict__ X, int64_t ld, int rows, int64_t K,
                                                 int32_t* __restrict__ emax) {
    __shared__ int sh[4][64];
    const int c = threadIdx.x & 63, g = threadIdx.x >> 6;
    const int r = blockIdx.y * 64 + c;
    const int64_t k0 = static_cast<int64_t>(blockIdx.x) * (kGsBlk * kGsK) + g * kGsK;
    int e = 0;
    if (r < rows)
#pragma unroll 8
        for (int k = 0; k < kGsK; ++k)
            if (k0 + k < K) e = max(e, (__double2hiint(X[(k0 + k) * ld + r]) >> 20) & 0x7ff);
    sh[g][c] = e;
    __syncthreads();
    if (g == 0 && r < rows) {
        e = max(max(sh[0][c], sh[1][c]), max(sh[2][c], sh[3][c]));
        emax[static_cast<int64_t>(blockIdx.x) * rows + r] = e > kGsBig ? kGsPlain : e;
    }
}

// C[m + n ldc] = sum over the splits, in split order, and of the blocks that have no digits.
__global__ void k_slices_reduce(GsArgs a, int n_split, double* __restrict__ C, int64_t ldc) {
    const int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t mn = static_cast<int64_t>(a.M) * a.N;
    if (e >= mn) return;
    const int64_t n = e / a.M, m = e % a.M;
    const int tiles_m = (a.M + kGsM - 1) / kGsM, tiles = tiles_m * ((a.N + kGsN - 1) / kGsN);
    const int32_t* plain = a.plain + n / kGsN * tiles_m + m / kGsM;
    double s = 0.0;
    int any = 0;
    for (int z = 0; z < n_split; ++z) {
        s += a.part[z * mn + e];
        any |= plain[z * tiles];
    }
    if (any)
        for (int64_t b = 0; b < a.n_blk; ++b) {
            if (a.ea[b * a.M + m] >= 0 && a.eb[b * a.N + n] >= 0) continue;
            const int64_t k1 = min(a.K, (b + 1) * kGsBlk * kGsK);
            for (int64_t k = b * kGsBlk * kGsK; k < k1; ++k) s = fma(a.A[k * a.lda + m], a.B[k * a.ldb + n], s);
        }
    C[n * ldc + m] = s;
}

}  // namespace

// The rows' exponents, and `plain` of at most max(tiles of C, 8 n_sm) CTAs (gemm_slices_splits).
size_t gemm_slices_expo_ints(int64_t M, int64_t N, int64_t K, int n_sm) {
    const int64_t tiles = ((M + kGsM - 1) / kGsM) * ((N + kGsN - 1) / kGsN), cap = 8 * static_cast<int64_t>(n_sm);
    return static_cast<size_t>((M + N) * ((K + kGsBlk * kGsK - 1) / (kGsBlk * kGsK)) + (tiles > cap ? tiles : cap));
}

// From 512 k: four blocks and the two exponent passes cost less than the FMA kernel's steps at every M
// and N (1,487 points: Fock matrix of 11 functions 0.08 ms against 0.17; hexamer, 78, 0.67 against 4.6).
bool gemm_slices_applies(int64_t K) { return K >= 512; }

int gemm_slices_splits(int M, int N, int64_t K, int n_sm, size_t work_elems) {
    const int64_t tiles = static_cast<int64_t>((M + kGsM - 1) / kGsM) * ((N + kGsN - 1) / kGsN);
    const int64_t blocks = (K + kGsBlk * kGsK - 1) / (kGsBlk * kGsK);
    int64_t cap = static_cast<int64_t>(work_elems / (static_cast<size_t>(M) * static_cast<size_t>(N)));
    if (cap > blocks) cap = blocks;
    // whole waves of one CTA per SM; a split costs about half a block's time of its own
    int best = 1;
    double best_t = 1e300;
    for (int64_t s = 1; s <= cap && s * tiles <= 8 * static_cast<int64_t>(n_sm); ++s) {
        const double t = std::ceil(static_cast<double>(tiles * s) / n_sm) * ((blocks + s - 1) / s + 0.5);
        if (t < best_t) {
            best_t = t;
            best = static_cast<int>(s);
        }
    }
    return best;
}

cudaError_t launch_gemm_slices(int M, int N, int64_t K, const double* A, int64_t lda, const double* B,
                               int64_t ldb, double* C, int64_t ldc, double* work, int n_split,
                               int32_t* expo, int* launched, int* err, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_gemm_slices, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(kGsSmem));
    if (e != cudaSuccess) return e;
    GsArgs a{};
    a.M = M;
    a.N = N;
    a.K = K;
    a.n_blk = static_cast<int32_t>((K + kGsBlk * kGsK - 1) / (kGsBlk * kGsK));
    a.per_split = (a.n_blk + n_split - 1) / n_split;
    n_split = (a.n_blk + a.per_split - 1) / a.per_split;
    a.A = A;
    a.B = B;
    a.lda = lda;
    a.ldb = ldb;
    a.ea = expo;
    a.eb = expo + static_cast<int64_t>(a.n_blk) * M;
    a.part = work;
    a.err = err;
    const unsigned nb = static_cast<unsigned>(a.n_blk);
    int32_t* expo_b = expo + static_cast<int64_t>(nb) * M;
    a.plain = expo_b + static_cast<int64_t>(nb) * N;
    *launched += 4;
    k_exp_max<<<dim3(nb, static_cast<unsigned>((M + 63) / 64)), 256, 0, st>>>(A, lda, M, K, expo);
    k_exp_max<<<dim3(nb, static_cast<unsigned>((N + 63) / 64)), 256, 0, st>>>(B, ldb, N, K, expo_b);
    const dim3 grid(static_cast<unsigned>((M + kGsM - 1) / kGsM), static_cast<unsigned>((N + kGsN - 1) / kGsN),
                    static_cast<unsigned>(n_split));
    k_gemm_slices<<<grid, kGsThreads, kGsSmem, st>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int64_t mn = static_cast<int64_t>(M) * N;
    k_slices_reduce<<<static_cast<unsigned>((mn + 255) / 256), 256, 0, st>>>(a, n_split, C, ldc);
    return cudaGetLastError();
}

}  // namespace vv10
