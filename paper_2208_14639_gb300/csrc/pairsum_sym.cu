// K2 / K4 over unordered pairs: the double grid sums of pairsum.cu with every pair of points
// evaluated once and added to both of its points.
//
// What a pair (i, j) costs is mostly common to (i, j) and (j, i): R^2, g, g', s and the
// reciprocal are the same numbers (addition and multiplication commute bit for bit), only the
// weights and the per-row brackets differ.  For E/U/W that is 29 FP32 operations per unordered
// pair instead of 2 x 21, for the nine sums of the fused step 58 instead of 2 x 39.
//
// Tiles.  The kept points are cut into tiles of 32 R points (R rows per lane: 8 in FP32, 4, 2 or
// 1 in FP64).  Row tile I takes the column tiles I + 1 .. I + floor((nb - 1) / 2) (mod nb), and for an
// even tile count half of the row tiles also take I + nb / 2: each unordered pair of tiles occurs
// once and every row tile has the same work.  The diagonal tile (I, I) is evaluated for its rows
// only.  A warp walks a range of a row tile's column tiles as one stream of columns.
//
// Order of the sums.  In FP32 a tile's sum over its 256 points is formed in point order from
// zero and then added in FP64, for rows and columns alike, exactly as pairsum.cu does, so both
// kernels give the same FP32 tile sums.  Lane l holds rows R l .. R l + R - 1 and is one column
// behind lane l - 1: at step s it evaluates column s - l, receives that column's sums over the
// lower rows from lane l - 1 by shuffle, adds its own rows in order and passes them on; lane 31
// finishes a column each step.  The stream is continuous over column tiles, so the 31 steps of
// skew are paid once per stream.
//
// A lane's row sums are stashed in shared memory when it crosses into the next column tile (each
// lane at its own step) and added to the warp's FP64 totals once per tile; finished column sums
// are written as they stand (colpart) and added up by k_sym_reduce in two numbers of their own type
// (FP32: ~48 bits; 7 FP32 operations where a conversion and an FP64 add would wait for the
// narrow FP64 pipe).
//
// FP32 pairs run on packed FP32x2 instructions over two rows (the same roundings as scalar ones):
// the packed form halves the issue slots and leaves the FMA pipe as the bound.  -1/(g g' s)
// is formed instead of 1/(g g' s) (the Newton step needs no negated operand then), and the sums
// it makes negative are negated when they are written.
//
// What bounds it: FP32 the FMA pipe (80 % busy, of which the rest is fixed-latency waits of two or
// three warps a scheduler), FP64 the FP64 pipe (30 operations per unordered pair for E/U/W against
// 2 x 22).  Measured against the row-by-row kernel, milliseconds: 131,008 points FP32 E/U/W 8.4
// (12.5), with A/B/C 13.2 (16.7), gradient 10.1 (15.3), all nine 20.0 (22.7); 29,339 points
// FP64 24.7 (35.3), 36.8 (48.2), 27.3 (41.2), 47.6 (63.8).
#include <cmath>

#include "common.cuh"
#include "kernels.hpp"

namespace vv10 {

namespace {

// Independent warps per CTA.  FP64: one, so that a few hundred of them spread over the SMs evenly
// (an SM's FP64 pipe is what they share); FP32: one per scheduler.
template <class T> constexpr int sym_warps() { return sizeof(T) == 4 ? 4 : 1; }

// One launch: column offsets [d0, d1) of every row tile.  The nb (d1 - d0) tile pairs in the order
// (row tile, offset) are dealt to n_warp warps in equal contiguous shares.  FP32 takes a multiple
// of nb warps, so that a share stays in its row tile; an FP64 share may run over row tiles, one
// stream ("segment", at most max_seg a warp) per row tile.
struct SymGeom {
    int64_t nkp;      // padded points = nb x tile
    int32_t nb;       // tiles
    int32_t d0, d1;   // offsets of this launch (0 = the diagonal tile)
    int32_t n_warp, max_seg;
    __host__ __device__ int cbase() const { return d0 > 0 ? d0 : 1; }  // first offset with columns
    __host__ __device__ int64_t pairs() const { return static_cast<int64_t>(nb) * (d1 - d0); }
    __host__ __device__ int64_t first(int64_t w) const { return w * pairs() / n_warp; }  // share of warp w
    __host__ __device__ int64_t owner(int64_t t) const {  // the last w with first(w) <= t
        return ((t + 1) * n_warp - 1) / pairs();
    }
};

// Signs of the accumulated quantities (see pair functions): row and column sums of quantity q.
template <int MODE> __device__ __forceinline__ float row_sign(int q) {
    if (MODE == MODE_GRAD || q >= 6) return -1.f;
    if (MODE == MODE_ABC) return 1.f;
    return (q == 1 || q == 2) ? -1.f : 1.f;
}
template <int MODE> __device__ __forceinline__ float col_sign(int q) {
    return ((MODE == MODE_EUW || MODE == MODE_EUWABC || MODE == MODE_EUWABCG) && (q == 1 || q == 2)) ? -1.f : 1.f;
}

// ---- arithmetic on two FP32 rows (float2) or one FP64 row
template <class T> struct V;  // the vector type a lane computes with
template <> struct V<float> { using type = float2; static constexpr int n = 2; };
template <> struct V<double> { using type = double; static constexpr int n = 1; };

__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }

// -1/x.  FP32: the hardware approximation of 1/(-x) and one Newton step, the value of
// rcp_refined(x) negated.
__device__ __forceinline__ float2 neg_recip(float2 x) {
    float2 r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(-x.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(-x.y));
    const float2 e = __ffma2_rn(x, r, make_float2(1.0f, 1.0f));
    return __ffma2_rn(r, e, r);
}
__device__ __forceinline__ double neg_recip(double x) { return -recip(x); }

// Adds a column's terms of two rows (in row order) or of one row to its running sum.
__device__ __forceinline__ void col_add(float& s, float2 v) { s = (s + v.x) + v.y; }
__device__ __forceinline__ void col_add(double& s, double v) { s += v; }
__device__ __forceinline__ void col_fma(float& s, float2 a, float2 b) {
    s = __fmaf_rn(a.y, b.y, __fmaf_rn(a.x, b.x, s));
}
__device__ __forceinline__ void col_fma(double& s, double a, double b) { s = fma(a, b, s); }

// A column as the lanes read it from shared memory: every value once per row of a vector
// (x, y, z and c = -3/2 w rho, negated except c's own sign).
template <class VT> struct __align__(16) ColRec { VT nx, ny, nz, c, om, ka; };
template <class VT> struct RowRec { VT x, y, z, c, om, ka; };

// One vector of rows against one column: row sums into acc, and (COL) column sums into ca.
// All sums built on n = -1/(g g' s) an odd number of times come out negated (row_sign, col_sign).
template <class T, int MODE, bool COL, class VT>
__device__ __forceinline__ void sym_pair(const RowRec<VT>& r, const ColRec<VT>& c,
                                         VT (&acc)[pair_mode_nq(MODE)], T (&ca)[pair_mode_nq(MODE)]) {
    const VT dx = vadd(r.x, c.nx), dy = vadd(r.y, c.ny), dz = vadd(r.z, c.nz);
    VT r2 = vmul(dx, dx);
    r2 = vfma(dy, dy, r2);
    r2 = vfma(dz, dz, r2);
    const VT g = vfma(r.om, r2, r.ka);
    const VT gp = vfma(c.om, r2, c.ka);
    const VT s = vadd(g, gp);
    const VT ggp = vmul(g, gp);
    const VT n = neg_recip(vmul(ggp, s));
    const VT ph = vmul(c.c, n);  // w_j rho_j Phi_ij (c.c = +3/2 w rho)
    VT pc;
    if (COL) pc = vmul(r.c, n);  // w_i rho_i Phi_ij
    if constexpr (MODE == MODE_EUW) {
        const VT t = vmul(vmul(vadd(g, s), gp), n);  // -(1/s + 1/g)
        const VT pt = vmul(ph, t);
        acc[0] = vadd(acc[0], ph);
        acc[1] = vadd(acc[1], pt);
        acc[2] = vfma(pt, r2, acc[2]);
        if (COL) {
            const VT u = vmul(vmul(vadd(gp, s), g), n);  // -(1/s + 1/g')
            const VT pu = vmul(pc, u);
            col_add(ca[0], pc);
            col_add(ca[1], pu);
            col_fma(ca[2], pu, r2);
        }
    } else if constexpr (MODE == MODE_ABC) {
        const VT L = vmul(ggp, n), Gi = vmul(vmul(gp, s), n);  // -1/s, -1/g
        const VT v = vmul(ph, vfma(L, vadd(L, Gi), vmul(Gi, Gi)));
        acc[0] = vadd(acc[0], v);
        const VT v2 = vmul(v, r2);
        acc[1] = vadd(acc[1], v2);
        acc[2] = vfma(v2, r2, acc[2]);
        if (COL) {
            const VT Gj = vmul(vmul(g, s), n);
            const VT x = vmul(pc, vfma(L, vadd(L, Gj), vmul(Gj, Gj)));
            const VT x2 = vmul(x, r2);
            col_add(ca[0], x);
            col_add(ca[1], x2);
            col_fma(ca[2], x2, r2);
        }
    } else if constexpr (MODE == MODE_GRAD) {
        const VT a = vmul(r.om, gp), b = vadd(s, g), e = vmul(c.om, g), f = vadd(s, gp);
        const VT w = vmul(vmul(ph, n), vfma(a, b, vmul(e, f)));
        acc[0] = vfma(w, dx, acc[0]);
        acc[1] = vfma(w, dy, acc[1]);
        acc[2] = vfma(w, dz, acc[2]);
        if (COL) {
            const VT x = vmul(vmul(pc, n), vfma(e, f, vmul(a, b)));
            col_fma(ca[0], x, dx);
            col_fma(ca[1], x, dy);
            col_fma(ca[2], x, dz);
        }
    } else {
        const VT L = vmul(ggp, n), Gi = vmul(vmul(gp, s), n);
        const VT t = vadd(L, Gi);
        const VT pt = vmul(ph, t);
        acc[0] = vadd(acc[0], ph);
        acc[1] = vadd(acc[1], pt);
        acc[2] = vfma(pt, r2, acc[2]);
        const VT v = vmul(ph, vfma(L, t, vmul(Gi, Gi)));
        acc[3] = vadd(acc[3], v);
        const VT v2 = vmul(v, r2);
        acc[4] = vadd(acc[4], v2);
        acc[5] = vfma(v2, r2, acc[5]);
        VT Gj, q;
        if (COL || MODE == MODE_EUWABCG) Gj = vmul(vmul(g, s), n);
        if constexpr (MODE == MODE_EUWABCG) {
            // D = omega_i/g + omega_j/g' + (omega_i + omega_j)/s, each point's own term last
            q = vmul(vadd(r.om, c.om), L);
            const VT f = vmul(ph, vfma(r.om, Gi, vfma(c.om, Gj, q)));
            acc[6] = vfma(f, dx, acc[6]);
            acc[7] = vfma(f, dy, acc[7]);
            acc[8] = vfma(f, dz, acc[8]);
        }
        if (COL) {
            const VT u = vadd(L, Gj);
            const VT pu = vmul(pc, u);
            col_add(ca[0], pc);
            col_add(ca[1], pu);
            col_fma(ca[2], pu, r2);
            const VT x = vmul(pc, vfma(L, u, vmul(Gj, Gj)));
            const VT x2 = vmul(x, r2);
            col_add(ca[3], x);
            col_add(ca[4], x2);
            col_fma(ca[5], x2, r2);
            if constexpr (MODE == MODE_EUWABCG) {
                const VT f = vmul(pc, vfma(c.om, Gj, vfma(r.om, Gi, q)));
                col_fma(ca[6], f, dx);
                col_fma(ca[7], f, dy);
                col_fma(ca[8], f, dz);
            }
        }
    }
}

__device__ __forceinline__ void vset(float2& v, int k, float x) { (k ? v.y : v.x) = x; }
__device__ __forceinline__ void vset(double& v, int, double x) { v = x; }
__device__ __forceinline__ float vget(float2 v, int k) { return k ? v.y : v.x; }
__device__ __forceinline__ double vget(double v, int) { return v; }
__device__ __forceinline__ float2 vdup(float x) { return make_float2(x, x); }
__device__ __forceinline__ double vdup(double x) { return x; }
__device__ __forceinline__ void vzero(float2& v) { v = make_float2(0.f, 0.f); }
__device__ __forceinline__ void vzero(double& v) { v = 0.0; }

// A record load that stays where it is written (the compiler otherwise sinks it to its use after
// the 32 steps it is meant to overlap).
__device__ __forceinline__ float4 load_early(const float4* p) {
    float4 v;
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ double4 load_early(const double4* p) {
    double4 v;
    asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2 + 16];" : "=d"(v.z), "=d"(v.w) : "l"(p));
    return v;
}

// hi + lo += x without loss (TwoSum; lo itself is rounded).
template <class T>
__device__ __forceinline__ void acc_exact(T& hi, T& lo, T x) {
    const T s = hi + x, b = s - hi;
    lo += (hi - (s - b)) + (x - b);
    hi = s;
}
// FP64 row totals over the tiles of a share are kept as hi + lo: hundreds of tiles are added one
// after the other there, where the row-by-row kernel adds in splits.
template <class T> constexpr int row_parts() { return sizeof(T) == 8 ? 2 : 1; }

template <class T, int MODE, int R>
struct __align__(16) SymShared {
    using VT = typename V<T>::type;
    static constexpr int NQ = pair_mode_nq(MODE);
    ColRec<VT> col[64];          // columns of two 32-column blocks, slot = column mod 64
    T done[NQ][64];              // finished column sums, slot = column mod 64
    T stash[NQ * R][33];         // row sums of a finished column tile, [quantity x row][lane]
};

// Registers before occupancy: 6 values and NQ sums per row, and a column's.  FP32: 168 a thread
// for three sums, 255 for six and nine (four schedulers with three or two warps each keep the FMA
// pipe as busy as four at 128 registers do: hexamer E/U/W 8.6 against 9.0 ms, nine sums 19.0
// against 20.8).  FP64: eight warps an SM, twice what fills its pipe.
template <class T, int MODE>
constexpr int sym_min_ctas() { return sizeof(T) == 8 ? 8 : (pair_mode_nq(MODE) == 3 ? 3 : 2); }

template <class T, int MODE, int R>
__global__ void __launch_bounds__(32 * sym_warps<T>(), sym_min_ctas<T, MODE>())
k_pairsum_sym(const typename PairRecs<T>::A* __restrict__ ra, const typename PairRecs<T>::B* __restrict__ rb,
              SymGeom G, double* __restrict__ rowpart, T* __restrict__ colpart) {
    using VT = typename V<T>::type;
    constexpr int VN = V<T>::n, NV = R / VN, NQ = pair_mode_nq(MODE), TS = 32 * R;
    extern __shared__ __align__(16) unsigned char sym_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    SymShared<T, MODE, R>& S = reinterpret_cast<SymShared<T, MODE, R>*>(sym_smem)[warp];
    int64_t w = static_cast<int64_t>(blockIdx.x) * sym_warps<T>() + warp;
    if (w >= G.n_warp) return;  // whole warps; no block-wide sync below
    // FP32: neighbouring warps take neighbouring row tiles, whose column streams overlap
    if (sizeof(T) == 4) w = (w % G.nb) * (G.n_warp / G.nb) + w / G.nb;
    const int64_t t_end = G.first(w + 1);
    int64_t t = G.first(w);
    int seg = 0;
    do {
    const int I = static_cast<int>(t / (G.d1 - G.d0));
    int d_lo = G.d0 + static_cast<int>(t % (G.d1 - G.d0));
    int d_hi = static_cast<int>(d_lo + (t_end - t) < G.d1 ? d_lo + (t_end - t) : G.d1);
    t += d_hi - d_lo;
    if (2 * (d_hi - 1) == G.nb && I >= G.nb / 2) --d_hi;  // the half turn: once per pair of tiles

    RowRec<VT> row[NV];
    VT acc[NV][NQ];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
#pragma unroll
        for (int k = 0; k < VN; ++k) {
            const int64_t i = static_cast<int64_t>(I) * TS + lane * R + v * VN + k;
            const auto a = ra[i];
            const auto b = rb[i];
            vset(row[v].x, k, a.x);
            vset(row[v].y, k, a.y);
            vset(row[v].z, k, a.z);
            vset(row[v].c, k, -a.w);
            vset(row[v].om, k, b.x);
            vset(row[v].ka, k, b.y);
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) vzero(acc[v][q]);
    }
    // this segment's FP64 row totals, [q R + r][lane]
    double* rp = rowpart + (w * G.max_seg + seg) * (NQ * TS * row_parts<T>()) + lane;
    bool first = true;
    T ca[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) ca[q] = T(0);

    auto stash = [&]() {  // this lane's tile sums to shared memory, and from zero again
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
#pragma unroll
                for (int k = 0; k < VN; ++k) S.stash[q * R + v * VN + k][lane] = vget(acc[v][q], k);
                vzero(acc[v][q]);
            }
    };
    auto flush = [&]() {  // every lane's stash into the FP64 totals
#pragma unroll
        for (int e = 0; e < NQ * R; ++e) {
            const double x = static_cast<double>(S.stash[e][lane]) * row_sign<MODE>(e / R);
            if (sizeof(T) == 8) {
                double hi = first ? 0.0 : __ldcg(rp + e * 32), lo = first ? 0.0 : __ldcg(rp + (NQ * R + e) * 32);
                acc_exact(hi, lo, x);
                __stcg(rp + e * 32, hi);
                __stcg(rp + (NQ * R + e) * 32, lo);
            } else {
                __stcg(rp + e * 32, first ? x : __ldcg(rp + e * 32) + x);
            }
        }
        first = false;
    };
    auto put_col = [&](int slot, const typename PairRecs<T>::A& a, const typename PairRecs<T>::B& b) {
        ColRec<VT> c;
        c.nx = vdup(-a.x);
        c.ny = vdup(-a.y);
        c.nz = vdup(-a.z);
        c.c = vdup(-a.w);
        c.om = vdup(b.x);
        c.ka = vdup(b.y);
        S.col[slot] = c;
    };
    // a column that adds nothing and divides by nothing small
    const typename PairRecs<T>::A noneA{T(0), T(0), T(0), T(0)};
    const typename PairRecs<T>::B noneB{T(1), T(1), T(0), T(0)};

    if (d_lo == 0 && d_hi > 0) {  // the diagonal tile: rows only, columns in step over the lanes
        for (int k = 0; k < TS / 32; ++k) {
            const int64_t j = static_cast<int64_t>(I) * TS + 32 * k + lane;
            put_col(lane, ra[j], rb[j]);
            __syncwarp();
            for (int jj = 0; jj < 32; ++jj) {
                const ColRec<VT> c = S.col[jj];
#pragma unroll
                for (int v = 0; v < NV; ++v) sym_pair<T, MODE, false>(row[v], c, acc[v], ca);
            }
            __syncwarp();
        }
        stash();
        flush();  // each lane reads back what it wrote
        d_lo = 1;
    }
    if (d_hi > d_lo) {
        const int n_blk = (d_hi - d_lo) * R;  // 32-column blocks of the stream
        // column c of the stream is point (base + c) mod nkp
        int64_t src = (static_cast<int64_t>(I) + d_lo) * TS;
        if (src >= G.nkp) src -= G.nkp;
        put_col(lane, ra[src + lane], rb[src + lane]);  // block 0: slots 0 .. 31
        put_col(32 + lane, noneA, noneB);               // the columns before the stream
        int64_t out = src;                              // point of the next finished block's first column
        T* cp = colpart + static_cast<int64_t>(d_lo - G.cbase()) * NQ * G.nkp;
        for (int k = 0; k <= n_blk; ++k) {
            __syncwarp();
            auto na = noneA;
            auto nb_ = noneB;
            if (k + 1 < n_blk) {  // the next block, while this one is evaluated
                src += 32;
                if (src >= G.nkp) src -= G.nkp;
                na = load_early(ra + src + lane);
                nb_ = load_early(rb + src + lane);
            }
            const bool edge = (k % R) == 0 && k > 0;  // lanes enter the next column tile in this block
#pragma unroll 1
            for (int ss = 0; ss < 32; ++ss) {
                const int slot = (32 * k + ss - lane) & 63;
                const ColRec<VT> c = S.col[slot];
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const T up = __shfl_up_sync(0xffffffffu, ca[q], 1);
                    ca[q] = lane == 0 ? T(0) : up;
                }
                if (edge && ss == lane) stash();
#pragma unroll
                for (int v = 0; v < NV; ++v) sym_pair<T, MODE, true>(row[v], c, acc[v], ca);
                if (lane == 31) {
#pragma unroll
                    for (int q = 0; q < NQ; ++q) S.done[q][slot] = ca[q];
                }
            }
            __syncwarp();
            if (k >= 1) {  // columns 32 (k - 1) .. 32 k - 1 are finished
                const int slot = (32 * (k - 1) + lane) & 63;
#pragma unroll
                for (int q = 0; q < NQ; ++q)
                    __stcs(cp + q * G.nkp + out + lane, S.done[q][slot] * T(col_sign<MODE>(q)));
                out += 32;
                if (out >= G.nkp) out -= G.nkp;
                if (k % R == 0) cp += static_cast<int64_t>(NQ) * G.nkp;  // the next offset's columns
            }
            put_col((32 * (k + 1) + lane) & 63, na, nb_);
            if (edge) flush();
        }
    }
    if (first) {  // no tile in this segment
#pragma unroll
        for (int e = 0; e < NQ * R * row_parts<T>(); ++e) __stcg(rp + e * 32, 0.0);
    }
    __syncwarp();  // the shared columns are read before the next segment's
    ++seg;
    } while (sizeof(T) == 8 && t < t_end);
}

// total[q][p] (+)= the row totals of p's tile over its segments, and its column sums over the
// offsets of the launch, in a fixed order.
template <class T, int NQ, int R>
__global__ void __launch_bounds__(256)
k_sym_reduce(SymGeom G, const double* __restrict__ rowpart, const T* __restrict__ colpart, int add,
             double* __restrict__ total) {
    constexpr int TS = 32 * R;
    const int64_t p = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x;
    const int q = blockIdx.y;
    if (p >= G.nkp) return;
    const int J = static_cast<int>(p / TS), e = static_cast<int>(p % TS);
    T hi = T(0), lo = T(0);  // column sums
    double sum = add ? total[q * G.nkp + p] : 0.0;
    const int64_t off = G.d1 - G.d0, w0 = G.owner(J * off), w1 = G.owner((J + 1) * off - 1);
    int64_t seg = J - G.first(w0) / off;  // the first share may have begun in an earlier tile
    for (int64_t w = w0; w <= w1; ++w, seg = 0) {
        const double* r = rowpart + (w * G.max_seg + seg) * (NQ * TS * row_parts<T>()) + (q * R + e % R) * 32 + e / R;
        if constexpr (sizeof(T) == 8) {
            acc_exact(hi, lo, r[0]);
            lo += r[NQ * TS];
        } else {
            sum += r[0];
        }
    }
    int d1 = G.d1;
    if (2 * (d1 - 1) == G.nb && J < G.nb / 2) --d1;  // the half turn's columns are the upper tiles
    const int n = d1 - G.cbase();
    const T* c = colpart + q * G.nkp + p;
    const int64_t step = static_cast<int64_t>(NQ) * G.nkp;
#pragma unroll 8
    for (int d = 0; d < n; ++d) acc_exact(hi, lo, __ldcs(c + d * step));
    sum += static_cast<double>(hi) + static_cast<double>(lo);
    total[q * G.nkp + p] = sum;
}

template <class T, int MODE, int R>
constexpr size_t sym_smem_bytes() { return sizeof(SymShared<T, MODE, R>) * sym_warps<T>(); }

// Warps that the SMs hold at once.
template <class T, int MODE, int R>
int sym_resident(int n_sm) {
    int n = 0;
    if (cudaFuncSetAttribute(k_pairsum_sym<T, MODE, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(sym_smem_bytes<T, MODE, R>())) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_pairsum_sym<T, MODE, R>, 32 * sym_warps<T>(),
                                                      sym_smem_bytes<T, MODE, R>()) != cudaSuccess) {
        cudaGetLastError();
        n = 1;
    }
    return (n > 0 ? n : 1) * sym_warps<T>() * (n_sm > 0 ? n_sm : 1);
}

struct SymPlan {
    int32_t nb, d_end, offsets;  // tiles; all offsets; offsets per launch
    int32_t warps, split;        // FP64: warps of a launch; FP32: warps per row tile
    double cost;                 // estimated time, in steps of one row per lane
    size_t row_bytes, col_bytes;
    int launches() const { return (d_end + offsets - 1) / offsets; }
    SymGeom launch(int64_t nkp, int32_t d0) const {
        SymGeom g{nkp, nb, d0, d0 + offsets < d_end ? d0 + offsets : d_end, 0, 1};
        const int64_t pairs = g.pairs();
        if (split > 0) {
            g.n_warp = nb * (split < g.d1 - g.d0 ? split : g.d1 - g.d0);
        } else {
            g.n_warp = static_cast<int32_t>(pairs < warps ? pairs : warps);
            g.max_seg = static_cast<int32_t>((pairs / g.n_warp + 1) / (g.d1 - g.d0) + 2);
        }
        return g;
    }
};

// col_budget: bytes of column sums of a launch, which covers as many offsets as fit (at least four).
template <class T, int MODE, int R>
SymPlan sym_plan(int64_t nkp, int n_sm, size_t col_budget) {
    constexpr int TS = 32 * R, NQ = pair_mode_nq(MODE);
    const size_t per_d = sizeof(T) * NQ * static_cast<size_t>(nkp);
    SymPlan P{};
    P.nb = static_cast<int32_t>(nkp / TS);
    P.d_end = P.nb / 2 + 1;
    int64_t most = static_cast<int64_t>(col_budget / per_d);
    if (most < 4) most = 4;
    const int launches = static_cast<int>((P.d_end + most - 1) / most);
    P.offsets = (P.d_end + launches - 1) / launches;
    const int slots = sym_resident<T, MODE, R>(n_sm);
    if (sizeof(T) == 4) {
        // A share costs its columns' steps and 32 for the skew.  Several waves of short shares
        // keep three warps on every scheduler to the end (a scheduler favours its oldest warp, so
        // equal shares of one wave end apart: hexamer E/U/W 10.2 ms in four splits, 8.35 in 28).
        P.cost = 1e300;
        for (int s = 1; s <= P.offsets; ++s) {
            const double unit = static_cast<double>((P.offsets + s - 1) / s) * TS + 32.0;
            const double waves = P.nb * static_cast<double>(s) / slots;
            const double c = R * unit * (waves > 1.0 ? waves + 0.5 : 1.0);
            if (c < P.cost) {
                P.cost = c;
                P.split = s;
            }
        }
    } else {
        // One wave of equal shares: the warps of an SM share its FP64 pipe, so the SM with the
        // most of them sets the time.
        const int64_t pairs = static_cast<int64_t>(P.nb) * P.offsets;
        P.warps = static_cast<int32_t>(pairs < slots ? pairs : slots);
        const double share = std::ceil(static_cast<double>(pairs) / P.warps);
        P.cost = R * std::ceil(static_cast<double>(P.warps) / n_sm) * (share * TS + 32.0 * (1.0 + share / P.offsets));
    }
    for (int32_t d0 = 0; d0 < P.d_end; d0 += P.offsets) {
        const SymGeom g = P.launch(nkp, d0);
        const size_t rows = sizeof(double) * NQ * TS * row_parts<T>() * static_cast<size_t>(g.n_warp) * g.max_seg;
        if (rows > P.row_bytes) P.row_bytes = rows;
    }
    P.col_bytes = per_d * static_cast<size_t>(P.offsets);
    return P;
}

template <class T, int MODE, int R>
cudaError_t launch_sym(int64_t nkp, const typename PairRecs<T>::A* ra, const typename PairRecs<T>::B* rb,
                       const SymPlan& plan, void* work, double* total, cudaStream_t st) {
    constexpr int W = sym_warps<T>(), NQ = pair_mode_nq(MODE);
    double* rowpart = static_cast<double*>(work);
    T* colpart = reinterpret_cast<T*>(static_cast<char*>(work) + plan.row_bytes);
    for (int32_t d0 = 0; d0 < plan.d_end; d0 += plan.offsets) {
        const SymGeom g = plan.launch(nkp, d0);
        k_pairsum_sym<T, MODE, R><<<static_cast<unsigned>((g.n_warp + W - 1) / W), 32 * W,
                                    sym_smem_bytes<T, MODE, R>(), st>>>(ra, rb, g, rowpart, colpart);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        k_sym_reduce<T, NQ, R><<<dim3(static_cast<unsigned>((g.nkp + 255) / 256), NQ), 256, 0, st>>>(
            g, rowpart, colpart, d0 > 0 ? 1 : 0, total);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Plans (work = null) or runs a mode.  FP32: eight rows per lane (the order of its tile sums).
// FP64: four, or fewer where more and smaller tiles fill the SMs better.
template <int MODE>
cudaError_t sym_mode(const PointsDev* p, int64_t nkp, bool fp64, int n_sm, size_t cols, SymPlan* plan,
                     void* work, double* total, cudaStream_t st) {
    if (!fp64) {
        *plan = sym_plan<float, MODE, 8>(nkp, n_sm, cols);
        return work ? launch_sym<float, MODE, 8>(nkp, p->r32a, p->r32b, *plan, work, total, st) : cudaSuccess;
    }
    const SymPlan p4 = sym_plan<double, MODE, 4>(nkp, n_sm, cols), p2 = sym_plan<double, MODE, 2>(nkp, n_sm, cols),
                  p1 = sym_plan<double, MODE, 1>(nkp, n_sm, cols);
    if (p4.cost <= p2.cost && p4.cost <= p1.cost) {
        *plan = p4;
        return work ? launch_sym<double, MODE, 4>(nkp, p->r64a, p->r64b, p4, work, total, st) : cudaSuccess;
    }
    if (p2.cost <= p1.cost) {
        *plan = p2;
        return work ? launch_sym<double, MODE, 2>(nkp, p->r64a, p->r64b, p2, work, total, st) : cudaSuccess;
    }
    *plan = p1;
    return work ? launch_sym<double, MODE, 1>(nkp, p->r64a, p->r64b, p1, work, total, st) : cudaSuccess;
}

cudaError_t sym_any(const PointsDev* p, int64_t nkp, int mode, bool fp64, int n_sm, size_t cols, SymPlan* plan,
                    void* work, double* total, cudaStream_t st) {
    switch (mode) {
        case MODE_EUW: return sym_mode<MODE_EUW>(p, nkp, fp64, n_sm, cols, plan, work, total, st);
        case MODE_ABC: return sym_mode<MODE_ABC>(p, nkp, fp64, n_sm, cols, plan, work, total, st);
        case MODE_GRAD: return sym_mode<MODE_GRAD>(p, nkp, fp64, n_sm, cols, plan, work, total, st);
        case MODE_EUWABC: return sym_mode<MODE_EUWABC>(p, nkp, fp64, n_sm, cols, plan, work, total, st);
        default: return sym_mode<MODE_EUWABCG>(p, nkp, fp64, n_sm, cols, plan, work, total, st);
    }
}

}  // namespace

// FP32: a tile pair is one warp's work, so below some forty tiles the warps are too few.  Calls of three,
// six and nine sums, microseconds row by row and here: 8,684 points 104, 128, 200 and 103, 134, 209; 10,732
// points 135, 176, 259 and 135, 192, 285; 10,988 points 164, 233, 304 and 136, 190, 285; 15,852 points 266,
// 354, 468 and 224, 321, 462.  (Both kernels' times are stairs: at 12,780 to 13,036 points six sums are 12 %,
// and up to 15,340 nine sums 8 to 11 %, slower here.)  FP64: the tiles shrink with the system; the smallest
// systems take pairsum.cu's small FP64 kernel before this rule is asked.
bool pairsum_sym_applies(int64_t nk, bool fp64) { return nk > (fp64 ? 128 : 10752); }

size_t pairsum_sym_work(int64_t nk_pad, int mode, bool fp64, int n_sm, size_t col_budget, int* n_launch) {
    SymPlan p{};
    sym_any(nullptr, nk_pad, mode, fp64, n_sm, col_budget, &p, nullptr, nullptr, nullptr);
    *n_launch = p.launches();
    return p.row_bytes + p.col_bytes;
}

cudaError_t launch_pairsum_sym(const PointsDev& p, int mode, bool fp64, int n_sm, size_t col_budget, void* work,
                               double* total, cudaStream_t st) {
    if (p.nk == 0) return cudaSuccess;
    SymPlan plan{};
    return sym_any(&p, p.nk_pad, mode, fp64, n_sm, col_budget, &plan, work, total, st);
}

}  // namespace vv10
