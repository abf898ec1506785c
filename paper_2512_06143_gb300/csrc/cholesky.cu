// cholesky.cu -- tiled FP64 Cholesky factorisation L L^T and solve, in one kernel that runs its tiles as
// their inputs become ready, and the exact log-determinant and y solve built on it.
//
// The covariance is sparse, and so is its factor at the level of 32 x 32 tiles of Morton-consecutive
// rows: the tiles are ordered by minimum degree on their adjacency (host, once per pattern), the fill is
// found symbolically, and only the tiles of the factor are stored and computed.
//
// What bounds it: GB300 issues one FP64 warp instruction every 19 cycles per SM (64 cycles per warp
// scheduler, dependent or not), about 0.98 TFLOP/s for the whole chip, so a dense factorisation of n rows takes at
// least n^3 / 3 / 0.98 TFLOP/s (n = 4096: 23 ms) and a 32 x 32 x 32 tile product 10 us on its SM.
// Skipping absent tiles removes most of that (n = 4096 in 2-D: 11,000 tile products of 358,000), and what is
// left is the chain diagonal tile -> panel tile -> next diagonal tile.  Tiles of 32 keep that chain
// short (its length per tile column falls with the tile's size squared), and the ordering prefers
// tile columns that do not wait on others (a band of 63 tile columns becomes a chain of 11).  One kernel
// with a flag per tile takes the place of four launches per panel of the whole matrix.
// Measured: the FP64 LML of 4,096 points in 2-D 52.1 -> 3.16 ms, an MCMC evaluation of 2,000 points in 1-D
// 18.4 -> 0.74 ms, the allocation-free call at 301 points, all tiles present, 2.47 -> 0.45 ms; with the pivots'
// tests and reciprocals mostly off the FP64 pipe 2.74, 0.70 and 0.41 ms.
#include <algorithm>
#include <cmath>
#include <vector>

#include "gp2s_cholesky.cuh"
#include "gp2s_kernel_math.cuh"

namespace gp2s {

namespace {

constexpr int kCholThreads = 128;
// Polls of a flag before a wait gives up: several seconds (a poll and its sleep take about a microsecond).  The
// tile that is waited for is in work already, so a wait lasts no longer than that tile's own products, and those of
// the few earlier ones that it waits for in turn: a row of at most 5,900 tiles (exact_fits) at 10 us a product,
// six CTAs to an SM, is 0.35 s.  Full matrices of 32,768 rows (9.5 s) and 100,000 points in 3-D (12 s, 60 entries a
// row) run through.  With every tile present (at most 16 tile columns, under a millisecond) some 50 ms: calls
// that overlap on the allocation-free path's one scratch array clear each other's flags.
template <bool ALL> constexpr int kCholMaxSpins = ALL ? 1 << 16 : 1 << 23;
enum { CT_FACTOR = 0, CT_FORWARD = 1, CT_BACKWARD = 2 };

__device__ __forceinline__ int ld_acquire(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(int *p, int v)
{
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Bounded wait of one thread for *flag; false when it gave up or another CTA did.
template <bool ALL>
__device__ __forceinline__ bool chol_wait(const int *flag, const int *abort_word)
{
    for (int spin = 0; spin < kCholMaxSpins<ALL>; ++spin) {
        if (ld_acquire(flag)) return true;
        if ((spin & 63) == 63 && ld_acquire(abort_word)) return false;
        if (spin > 16) __nanosleep(100);
    }
    return false;
}

// A pivot d is usable when its sign bit is clear and it is neither zero, infinite nor NaN: read off its high
// word, since an FP64 comparison takes as long as an FP64 addition (64 cycles of the warp).
__device__ __forceinline__ bool chol_positive(double d)
{
    const int hi = __double2hiint(d);
    return hi < 0x7ff00000 && (hi > 0 || (hi == 0 && __double2loint(d) != 0));
}

template <bool ALL> struct CholMap;
template <> struct CholMap<false> {
    static __device__ __forceinline__ int4 task(const CholArgs &a, int t) { return a.tasks[t]; }
    static __device__ __forceinline__ int row_begin(const CholArgs &a, int i) { return a.rptr[i]; }
    static __device__ __forceinline__ int row_end(const CholArgs &a, int i) { return a.rptr[i + 1]; }
    static __device__ __forceinline__ int diag(const CholArgs &a, int j) { return a.colptr[j]; }
    static __device__ __forceinline__ int col_end(const CholArgs &a, int j) { return a.colptr[j + 1]; }
    static __device__ __forceinline__ int col_pos(const CholArgs &a, int, int s) { return a.rowpos[s]; }
    // column and slot of entry e of row i; the slot of (i, k), -1 where it is absent
    static __device__ __forceinline__ int row_col(const CholArgs &a, int, int e) { return a.rcol[e]; }
    static __device__ __forceinline__ int row_slot(const CholArgs &a, int, int e) { return a.rslot[e]; }
    static __device__ __forceinline__ int find(const CholArgs &a, int i, int k)
    {
        int lo = a.rptr[i], hi = a.rptr[i + 1];
        const int end = hi;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (a.rcol[mid] < k) lo = mid + 1; else hi = mid;
        }
        return lo < end && a.rcol[lo] == k ? a.rslot[lo] : -1;
    }
    static __device__ __forceinline__ int origin(const CholArgs &a, int j) { return a.perm[j]; }
};
template <> struct CholMap<true> {
    static __device__ __forceinline__ int slot(const CholArgs &a, int i, int j)
    {
        return j * a.nt - j * (j - 1) / 2 + (i - j);
    }
    // column by column: the diagonal tile, the forward solve's block, the tiles below; then the
    // backward blocks from the last to the first
    static __device__ __forceinline__ int4 task(const CholArgs &a, int t)
    {
        for (int j = 0; j < a.nt; ++j) {
            const int cnt = a.nt - j + a.solve;
            if (t < cnt) {
                if (a.solve && t == 1) return make_int4(CT_FORWARD, j, j, 0);
                const int i = j + (t > 1 ? t - a.solve : t);
                return make_int4(CT_FACTOR, i, j, slot(a, i, j));
            }
            t -= cnt;
        }
        return make_int4(CT_BACKWARD, a.nt - 1 - t, a.nt - 1 - t, 0);
    }
    static __device__ __forceinline__ int row_begin(const CholArgs &, int) { return 0; }
    static __device__ __forceinline__ int row_end(const CholArgs &, int i) { return i; }
    static __device__ __forceinline__ int diag(const CholArgs &a, int j) { return slot(a, j, j); }
    static __device__ __forceinline__ int col_end(const CholArgs &a, int j) { return slot(a, j, j) + a.nt - j; }
    static __device__ __forceinline__ int col_pos(const CholArgs &a, int j, int s) { return j + (s - slot(a, j, j)); }
    static __device__ __forceinline__ int row_col(const CholArgs &, int, int e) { return e; }
    static __device__ __forceinline__ int row_slot(const CholArgs &a, int i, int e) { return slot(a, i, e); }
    static __device__ __forceinline__ int find(const CholArgs &a, int i, int k) { return slot(a, i, k); }
    static __device__ __forceinline__ int origin(const CholArgs &, int j) { return j; }
};

using CholTile = double (*)[kCT + 1];

// A tile travels global -> registers -> shared memory so that the next one's loads run under the
// current one's product (L2 only: another SM wrote it).
struct TileRegs { double2 v[kCTElems / 2 / kCholThreads]; };
__device__ __forceinline__ void tile_load(TileRegs &t, const double *__restrict__ g)
{
#pragma unroll
    for (int u = 0; u < kCTElems / 2 / kCholThreads; ++u)
        t.v[u] = __ldcg(reinterpret_cast<const double2 *>(g) + threadIdx.x + u * kCholThreads);
}
__device__ __forceinline__ void tile_store(CholTile S, const TileRegs &t)
{
#pragma unroll
    for (int u = 0; u < kCTElems / 2 / kCholThreads; ++u) {
        const int e = 2 * ((int)threadIdx.x + u * kCholThreads);
        S[e / kCT][e % kCT] = t.v[u].x;
        S[e / kCT][e % kCT + 1] = t.v[u].y;
    }
}

// One CTA takes tasks in increasing order; a task waits only for tiles of earlier tasks, which
// CTAs that already run hold, so no CTA needs the others to be resident.
template <bool ALL>
__global__ void __launch_bounds__(kCholThreads)
k_chol(const CholArgs a)
{
    using Map = CholMap<ALL>;
    __shared__ double As_[kCT][kCT + 1], Bs_[kCT][kCT + 1];
    __shared__ double colbuf[2][kCT], vec[kCT];
    __shared__ int s_task, s_ok, s_next, s_cnt;
    __shared__ int s_qa[kWarp], s_qb[kWarp];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    int *done_y = a.flags + a.ntiles, *done_x = done_y + a.nt;
    int *ticket = done_x + a.nt, *abort_word = ticket + 1;
    // product layout: rows tr + 16 p, columns tc + 8 q; solve layout: row r4, columns q4 + 4 m
    const int tr = tid >> 3, tc = tid & 7;
    const int r4 = tid >> 2, q4 = tid & 3;
    // every thread learns whether thread 0's wait succeeded
    auto wait_all = [&](const int *f1, const int *f2) -> bool {
        if (tid == 0) {
            bool ok = chol_wait<ALL>(f1, abort_word);
            if (ok && f2) ok = chol_wait<ALL>(f2, abort_word);
            s_ok = ok;
        }
        __syncthreads();
        return s_ok != 0;
    };
    auto finish = [&](int *flag) {
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            st_release(flag, 1);
        }
    };
    bool ok = true;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_task = ok && !ld_acquire(abort_word) ? atomicAdd(ticket, 1) : a.ntasks;
        __syncthreads();
        if (s_task >= a.ntasks) break;
        const int4 task = Map::task(a, s_task);
        const int j = task.z;
        // rows of the matrix in tile row j: the identity rows past them have nothing to compute.  A full tile
        // pays for a test every 8 pivots and every 8 steps of a solve: the allocation-free call at 1, 2, 16, 33 and 100
        // points 58.6 -> 44.6, 60.2 -> 46.0, 62.8 -> 54.2, 105.7 -> 91.7, 184.9 -> 172.0 us, at 512 662.8 -> 663.8.  With a
        // test per row, and the origin's load for it, 40.2, 43.8, 55.1, 87.4, 170.6, but 669.7 at 512 and up to 2 % of
        // the exact evaluations of 1,000 to 4,000 points; every 4 steps and after 1, 2 and 4 pivots was no better there.
        const int rows = j == a.last ? a.n - (a.nt - 1) * kCT : kCT;
        if (task.x != CT_FACTOR && !a.solve) continue;
        if (task.x == CT_FACTOR) {
            const int i = task.y;
            const bool dg = i == j;
            double *tile = a.tiles + (size_t)task.w * kCTElems;
            double acc[2][4];
#pragma unroll
            for (int p = 0; p < 2; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[p][q] = __ldcg(tile + (tr + 16 * p) * kCT + tc + 8 * q);
            // updates from the columns k < j that hold both (i, k) and (j, k), in increasing k
            const int kb = Map::row_begin(a, j), ke = Map::row_end(a, j);
            for (int base = kb; ok && base < ke; base += kWarp) {
                __syncthreads();   // the previous list is read
                if (wid == 0) {
                    int sb = -1, sa = -1;
                    if (base + lane < ke) {
                        sb = Map::row_slot(a, j, base + lane);
                        sa = dg ? sb : Map::find(a, i, Map::row_col(a, j, base + lane));
                    }
                    const unsigned m = __ballot_sync(0xffffffffu, sa >= 0);
                    if (sa >= 0) {
                        const int at = __popc(m & ((1u << lane) - 1u));
                        s_qa[at] = sa;
                        s_qb[at] = sb;
                    }
                    if (lane == 0) s_cnt = __popc(m);
                }
                __syncthreads();
                const int cnt = s_cnt;
                TileRegs ra, rb;
                bool have = false;
                for (int e = 0; e < cnt; ++e) {
                    if (!have) {
                        ok = wait_all(a.flags + s_qa[e], dg ? nullptr : a.flags + s_qb[e]);
                        if (!ok) break;
                        tile_load(ra, a.tiles + (size_t)s_qa[e] * kCTElems);
                        if (!dg) tile_load(rb, a.tiles + (size_t)s_qb[e] * kCTElems);
                    }
                    tile_store(As_, ra);
                    if (!dg) tile_store(Bs_, rb);
                    if (tid == 0)
                        s_next = e + 1 < cnt && ld_acquire(a.flags + s_qa[e + 1]) &&
                                 (dg || ld_acquire(a.flags + s_qb[e + 1]));
                    __syncthreads();
                    have = s_next != 0;
                    if (have) {
                        tile_load(ra, a.tiles + (size_t)s_qa[e + 1] * kCTElems);
                        if (!dg) tile_load(rb, a.tiles + (size_t)s_qb[e + 1] * kCTElems);
                    }
                    CholTile B = dg ? As_ : Bs_;
                    if (dg) {
                        // rows below 16 have no columns from 16 on in the lower triangle
#pragma unroll 4
                        for (int l = 0; l < kCT; ++l) {
                            const double a0 = As_[tr][l], a1 = As_[tr + 16][l];
                            const double b0 = B[tc][l], b1 = B[tc + 8][l], b2 = B[tc + 16][l], b3 = B[tc + 24][l];
                            acc[0][0] = fma(-a0, b0, acc[0][0]);
                            acc[0][1] = fma(-a0, b1, acc[0][1]);
                            acc[1][0] = fma(-a1, b0, acc[1][0]);
                            acc[1][1] = fma(-a1, b1, acc[1][1]);
                            acc[1][2] = fma(-a1, b2, acc[1][2]);
                            acc[1][3] = fma(-a1, b3, acc[1][3]);
                        }
                    } else {
#pragma unroll 4
                        for (int l = 0; l < kCT; ++l) {
                            const double av[2] = {As_[tr][l], As_[tr + 16][l]};
                            const double bv[4] = {B[tc][l], B[tc + 8][l], B[tc + 16][l], B[tc + 24][l]};
#pragma unroll
                            for (int p = 0; p < 2; ++p)
#pragma unroll
                                for (int q = 0; q < 4; ++q) acc[p][q] = fma(-av[p], bv[q], acc[p][q]);
                        }
                    }
                    __syncthreads();
                }
            }
            if (!ok) continue;
            // to the solve layout
#pragma unroll
            for (int p = 0; p < 2; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) As_[tr + 16 * p][tc + 8 * q] = acc[p][q];
            double v[8];
            if (dg) {
                __syncthreads();
#pragma unroll
                for (int m = 0; m < 8; ++m) v[m] = As_[r4][q4 + 4 * m];
                // L D L^T by columns (one reciprocal per column), scaled to L L^T at the end
#pragma unroll
                for (int c = 0; c < kCT; ++c) {
                    if (c % 8 == 0 && c >= rows) break;
                    if (q4 == (c & 3)) colbuf[c & 1][r4] = v[c >> 2];
                    __syncthreads();
                    // rows up to c are finished (a warp holds eight rows)
                    if (8 * wid + 7 > c) {
                        double d = colbuf[c & 1][c];
                        if (!chol_positive(d)) d = 1.0;
                        const double w = colbuf[c & 1][r4] * rcp_pos(d);
#pragma unroll
                        for (int m = 0; m < 8; ++m)
                            if (4 * m > c || (4 * m + 3 > c && q4 + 4 * m > c)) v[m] = fma(-w, colbuf[c & 1][q4 + 4 * m], v[m]);
                    }
                }
                __syncthreads();
                // the diagonal, its reciprocal square roots, the scaled columns
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    if (r4 == q4 + 4 * m) vec[r4] = v[m];
                __syncthreads();
                if (wid == 0) {
                    double d = vec[lane];
                    if (!(d > 0.0)) {
                        atomicOr(a.bad, 1);
                        d = 1.0;
                    }
                    const double s = sqrt(d), inv = 1.0 / s;
                    colbuf[0][lane] = s;
                    colbuf[1][lane] = inv;
                    a.dinv[j * kCT + lane] = inv;
                }
                __syncthreads();
#pragma unroll
                for (int m = 0; m < 8; ++m) {
                    const int c = q4 + 4 * m;
                    v[m] = r4 == c ? colbuf[0][c] : (r4 > c ? v[m] * colbuf[1][c] : 0.0);
                }
            } else {
                // X = B L_jj^{-T}, row by row
                ok = wait_all(a.flags + Map::diag(a, j), nullptr);
                if (!ok) continue;
                TileRegs t;
                tile_load(t, a.tiles + (size_t)Map::diag(a, j) * kCTElems);
                tile_store(Bs_, t);
                if (tid < kCT) vec[tid] = __ldcg(a.dinv + j * kCT + tid);
                __syncthreads();
#pragma unroll
                for (int m = 0; m < 8; ++m) v[m] = As_[r4][q4 + 4 * m];
#pragma unroll
                for (int c = 0; c < kCT; ++c) {
                    const double own = v[c >> 2] * vec[c];
                    const double x = __shfl_sync(0xffffffffu, own, (lane & ~3) | (c & 3));
                    if (q4 == (c & 3)) v[c >> 2] = x;
#pragma unroll
                    for (int m = 0; m < 8; ++m)
                        if (4 * m > c || (4 * m + 3 > c && q4 + 4 * m > c)) v[m] = fma(-x, Bs_[q4 + 4 * m][c], v[m]);
                }
            }
#pragma unroll
            for (int m = 0; m < 8; ++m) __stcg(tile + r4 * kCT + q4 + 4 * m, v[m]);
            finish(a.flags + task.w);
        } else {
            // one block of the forward (L y = b) or backward (L^T x = y) solve
            const bool fw = task.x == CT_FORWARD;
            const int o = Map::origin(a, j) * kCT;
            double acc = 0.0;                       // row / column r4's sum over the lanes' q4
            if (fw) {
                const int kb = Map::row_begin(a, j), ke = Map::row_end(a, j);
                for (int e = kb; ok && e < ke; ++e) {
                    const int k = Map::row_col(a, j, e), s = Map::row_slot(a, j, e);
                    ok = wait_all(done_y + k, a.flags + s);
                    if (!ok) break;
                    const double *t = a.tiles + (size_t)s * kCTElems + r4 * kCT;
#pragma unroll
                    for (int m = 0; m < 8; ++m)
                        acc = fma(__ldcg(t + q4 + 4 * m), __ldcg(a.yv + k * kCT + q4 + 4 * m), acc);
                    __syncthreads();
                }
            } else {
                for (int s = Map::col_end(a, j) - 1; ok && s > Map::diag(a, j); --s) {
                    const int i = Map::col_pos(a, j, s);
                    ok = wait_all(done_x + i, nullptr);
                    if (!ok) break;
                    const double *t = a.tiles + (size_t)s * kCTElems + r4;
#pragma unroll
                    for (int m = 0; m < 8; ++m)
                        acc = fma(__ldcg(t + (q4 + 4 * m) * kCT), __ldcg(a.xv + i * kCT + q4 + 4 * m), acc);
                    __syncthreads();
                }
            }
            if (ok) ok = wait_all(a.flags + Map::diag(a, j), fw ? nullptr : done_y + j);
            if (!ok) continue;
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            acc += __shfl_xor_sync(0xffffffffu, acc, 2);
            if (q4 == 0) vec[r4] = acc;
            TileRegs t;
            tile_load(t, a.tiles + (size_t)Map::diag(a, j) * kCTElems);
            tile_store(Bs_, t);
            __syncthreads();
            if (wid == 0) {
                const double inv = __ldcg(a.dinv + j * kCT + lane);
                double v;
                if (fw) v = o + lane < a.n ? (a.bs ? a.bs[o + lane] : 1.0) * a.b[o + lane] : 0.0;
                else v = __ldcg(a.yv + j * kCT + lane);
                if (fw && a.bh && o + lane < a.n) a.bh[o + lane] = v;
                v -= vec[lane];
                if (fw) {
                    for (int c0 = 0; c0 < rows; c0 += 8) {
#pragma unroll
                        for (int c = c0; c < c0 + 8; ++c) {
                            const double x = __shfl_sync(0xffffffffu, v * inv, c);
                            if (lane == c) v = x;
                            else if (lane > c) v = fma(-x, Bs_[lane][c], v);
                        }
                    }
                    a.yv[j * kCT + lane] = v;
                } else {
                    for (int c0 = (rows - 1) / 8 * 8; c0 >= 0; c0 -= 8) {
#pragma unroll
                        for (int c = c0 + 7; c >= c0; --c) {
                            const double x = __shfl_sync(0xffffffffu, v * inv, c);
                            if (lane == c) v = x;
                            else if (lane < c) v = fma(-x, Bs_[c][lane], v);
                        }
                    }
                    a.xv[j * kCT + lane] = v;
                    if (o + lane < a.n) {
                        a.x[o + lane] = (a.bs ? a.bs[o + lane] : 1.0) * v;
                        if (a.xh) a.xh[o + lane] = v;
                    }
                }
            }
            finish((fw ? done_y : done_x) + j);
        }
    }
    if (!ok && tid == 0) {
        atomicOr(a.bad, 2);
        st_release(abort_word, 1);
    }
}

// Bit ti - tj - 1 of tile row ti (words of 32 bits) for every stored entry in a tile (ti, tj), ti > tj: a band
// takes one word or two per tile row.  `words` covers the longest distance of the pattern.
__global__ void k_chol_bits(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ col, int64_t n, int words,
                            unsigned *__restrict__ bits)
{
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = w0; i < n; i += nw) {
        const int ti = (int)(i / kCT);
        for (int p = rowptr[i] + lane; p < rowptr[i + 1]; p += kWarp) {
            const int at = ti - 1 - col[p] / kCT;
            if (at < 0 || at >= 32 * words) continue;
            unsigned *w = bits + (int64_t)ti * words + at / 32;
            const unsigned b = 1u << (at % 32);
            if (!(*reinterpret_cast<volatile unsigned *>(w) & b)) atomicOr(w, b);
        }
    }
}

// Scatter the CSR values of the lower triangle (in elimination order) into the tiles, which were
// zeroed; rows past n get a unit diagonal.
__global__ void k_chol_fill(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ col,
                            const double *__restrict__ val, int64_t n, CholArgs a, const int *__restrict__ pos)
{
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = w0; i < (int64_t)a.nt * kCT; i += nw) {
        const int pi = pos[i / kCT], r = (int)(i % kCT);
        if (i >= n) {
            if (lane == 0) a.tiles[(size_t)a.colptr[pi] * kCTElems + r * kCT + r] = 1.0;
            continue;
        }
        for (int p = rowptr[i] + lane; p < rowptr[i + 1]; p += kWarp) {
            const int j = col[p], pj = pos[j / kCT], c = j % kCT;
            if (pj > pi || (pj == pi && c > r)) continue;
            int lo = a.colptr[pj], hi = a.colptr[pj + 1];
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (a.rowpos[mid] < pi) lo = mid + 1; else hi = mid;
            }
            if (lo < a.colptr[pj + 1] && a.rowpos[lo] == pi) a.tiles[(size_t)lo * kCTElems + r * kCT + c] = val[p];
        }
    }
}

__global__ void k_chol_logdiag(CholArgs a, double *__restrict__ part)
{
    __shared__ double sh[8];
    double s = 0.0;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < a.nt * kCT; e += gridDim.x * blockDim.x) {
        const int j = e / kCT, c = e % kCT;
        if (a.perm[j] * kCT + c < a.n) s += log(a.tiles[(size_t)a.colptr[j] * kCTElems + c * kCT + c]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
        part[blockIdx.x] = t;
    }
}

// Elimination order and symbolic factorisation on the tile graph (host): minimum degree plus the
// height of the column's subtree, so that among columns of like fill those that wait on nothing go
// first (on a band of 63 tile columns the chain falls from 33 columns to 11, with 1.5 times the tiles;
// in 2-D and 3-D both orders give about the same fill).
struct CholPlan {
    std::vector<int> perm, colptr, rowpos, rptr, rcol, rslot, pos;
    std::vector<int4> tasks;
};

// `low` holds per tile row i a bit for each present tile (i, i - 1 - k), k < 32 words.
//
// A band of nt tile rows is the long case (a new pattern of a 1-D evaluation orders it with the GPU idle), so
// no step goes through all tiles: the next tile comes from a tree of minima, whose leaves hold (degree +
// height, height, tile) packed into one word, and a row of the adjacency is visited only between the first and
// the last word that it uses.  A band of 50 entries each side, on one host core: 1.4 ms at 100,000 rows and 2.9
// ms at 180,000 (16.6 and 52 ms with a scan of all tiles and whole rows per step); the order is the same.
void chol_order(int nt, int words, const std::vector<uint32_t> &low, CholPlan &P)
{
    const int W = (nt + 63) / 64;
    std::vector<uint64_t> adj((size_t)nt * W, 0), alive(W, 0);
    std::vector<int> first(nt, W), last(nt, -1);   // words of a row that may be nonzero
    auto set = [&](int i, int j) {
        adj[(size_t)i * W + j / 64] |= uint64_t(1) << (j % 64);
        first[i] = std::min(first[i], j / 64);
        last[i] = std::max(last[i], j / 64);
    };
    for (int i = 0; i < nt; ++i) {
        alive[i / 64] |= uint64_t(1) << (i % 64);
        for (int w = 0; w < words; ++w)
            for (uint32_t v = low[(size_t)i * words + w]; v; v &= v - 1) {
                const int j = i - 1 - (w * 32 + __builtin_ctz(v));
                set(i, j);
                set(j, i);
            }
    }
    std::vector<int> deg(nt), level(nt, 0);
    int leaves = 1;
    while (leaves < nt) leaves *= 2;
    std::vector<uint64_t> best(2 * (size_t)leaves, UINT64_MAX);
    auto key = [&](int i) { return (uint64_t)(deg[i] + level[i]) << 42 | (uint64_t)level[i] << 21 | (uint64_t)i; };
    auto place = [&](int i, uint64_t k) {
        size_t at = (size_t)leaves + i;
        best[at] = k;
        while (at > 1) {
            const uint64_t m = std::min(best[at], best[at ^ 1]);
            at /= 2;
            if (best[at] == m) break;
            best[at] = m;
        }
    };
    for (int i = 0; i < nt; ++i) {
        int d = 0;
        for (int w = first[i]; w <= last[i]; ++w) d += __builtin_popcountll(adj[(size_t)i * W + w]);
        deg[i] = d;
        best[(size_t)leaves + i] = key(i);
    }
    for (int i = leaves - 1; i > 0; --i) best[i] = std::min(best[2 * (size_t)i], best[2 * (size_t)i + 1]);
    std::vector<std::vector<int>> below(nt);   // by tile: the tiles that its column fills
    P.perm.clear();
    P.pos.assign(nt, 0);
    for (int step = 0; step < nt; ++step) {
        // least degree + height, then least height, then the first tile
        const int v = (int)(best[1] & ((1u << 21) - 1));
        place(v, UINT64_MAX);
        alive[v / 64] &= ~(uint64_t(1) << (v % 64));
        P.pos[v] = step;
        P.perm.push_back(v);
        uint64_t *av = &adj[(size_t)v * W];
        for (int w = first[v]; w <= last[v]; ++w)
            for (uint64_t b = av[w] & alive[w]; b; b &= b - 1) below[v].push_back(w * 64 + __builtin_ctzll(b));
        for (int u : below[v]) {
            uint64_t *au = &adj[(size_t)u * W];
            first[u] = std::min(first[u], first[v]);
            last[u] = std::max(last[u], last[v]);
            int d = 0;
            for (int w = first[u]; w <= last[u]; ++w) {
                au[w] = (au[w] | av[w]) & alive[w];
                d += __builtin_popcountll(au[w]);
            }
            au[u / 64] &= ~(uint64_t(1) << (u % 64));
            deg[u] = d - 1;
            level[u] = std::max(level[u], level[v] + 1);
            place(u, key(u));
        }
    }
    // columns in elimination order, their tiles by position; rows likewise
    P.colptr.assign(nt + 1, 0);
    P.rowpos.clear();
    std::vector<int> rcnt(nt + 1, 0);
    for (int j = 0; j < nt; ++j) {
        std::vector<int> r;
        for (int u : below[P.perm[j]]) r.push_back(P.pos[u]);
        std::sort(r.begin(), r.end());
        P.rowpos.push_back(j);
        for (int i : r) {
            P.rowpos.push_back(i);
            ++rcnt[i + 1];
        }
        P.colptr[j + 1] = (int)P.rowpos.size();
    }
    for (int i = 0; i < nt; ++i) rcnt[i + 1] += rcnt[i];
    P.rptr = rcnt;
    P.rcol.assign(rcnt[nt], 0);
    P.rslot.assign(rcnt[nt], 0);
    std::vector<int> at(rcnt.begin(), rcnt.end() - 1);
    for (int j = 0; j < nt; ++j)
        for (int s = P.colptr[j] + 1; s < P.colptr[j + 1]; ++s) {
            const int i = P.rowpos[s];
            P.rcol[at[i]] = j;
            P.rslot[at[i]++] = s;
        }
    // tasks: columns by their height, so that columns that wait on nothing are taken first; within a
    // column the diagonal tile, the forward block, then the tiles by position (the parent's first)
    std::vector<int> order(nt);
    for (int j = 0; j < nt; ++j) order[j] = j;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return level[P.perm[x]] < level[P.perm[y]]; });
    P.tasks.clear();
    for (int j : order)
        for (int s = P.colptr[j]; s < P.colptr[j + 1]; ++s) {
            P.tasks.push_back(make_int4(CT_FACTOR, P.rowpos[s], j, s));
            if (s == P.colptr[j]) P.tasks.push_back(make_int4(CT_FORWARD, j, j, 0));
        }
    for (int k = nt - 1; k >= 0; --k) P.tasks.push_back(make_int4(CT_BACKWARD, order[k], order[k], 0));
}

}  // namespace

cudaError_t chol_launch(const CholArgs &a, int num_sms, cudaStream_t stream)
{
    // up to six CTAs per SM (17 KB of shared memory each): tiles that wait leave the FP64 pipe to the others
    const int grid = std::max(1, std::min(a.ntasks, num_sms * 6));
    if (a.colptr) k_chol<false><<<grid, kCholThreads, 0, stream>>>(a);
    else k_chol<true><<<grid, kCholThreads, 0, stream>>>(a);
    return cudaGetLastError();
}

// The factorisation takes matrices whose dense form would fit in the device's memory (or in GP2S_MEM_LIMIT): the
// order of a larger tile graph would take the host minutes.
gp2s_status exact_fits(gp2s_ctx *c, bool *fits)
{
    if (!c->total_mem) {
        size_t free_b = 0;
        GP2S_CUDA(c, cudaMemGetInfo(&free_b, &c->total_mem));
    }
    const double n = (double)c->A.n;
    *fits = 8.0 * n * n <= (double)(c->mem_limit ? c->mem_limit : c->total_mem);
    return GP2S_OK;
}

// The plan of the current pattern in c->chol_ints, built when the pattern is new: the tile adjacency comes
// from the GPU, the order and the task list go back.
static gp2s_status chol_plan(gp2s_ctx *c)
{
    if (c->chol_plan_valid) return GP2S_OK;
    const int64_t n = c->A.n;
    bool fits = false;
    GP2S_TRY(exact_fits(c, &fits));
    if (!fits) return set_err(c, GP2S_ENOMEM, "exact log-determinant: n^2 doubles exceed the device memory");
    // an entry `band` below the diagonal lies at most ceil(band / kCT) tiles below it
    const int nt = (int)ceil_div(n, kCT), words = std::max(1, (int)ceil_div(ceil_div(c->A.band, kCT), 32));
    const size_t nbits = (size_t)nt * words;
    std::vector<uint32_t> low(nbits);
    if (nt > 1) {                                     // (one tile has no neighbours)
        GP2S_TRY(ensure(c, c->chol_ints, sizeof(unsigned) * nbits));
        GP2S_CUDA(c, cudaMemsetAsync(c->chol_ints.p, 0, sizeof(unsigned) * nbits, c->stream));
        const unsigned gb = (unsigned)std::min<int64_t>(ceil_div(n * 32, 256), 152 * 16);
        k_chol_bits<<<gb, 256, 0, c->stream>>>(c->rowptr.as<int32_t>(), c->col.as<int32_t>(), n, words,
                                               c->chol_ints.as<unsigned>());
        GP2S_LAUNCH(c);
        GP2S_CUDA(c, cudaMemcpyAsync(low.data(), c->chol_ints.p, sizeof(unsigned) * nbits, cudaMemcpyDeviceToHost,
                                     c->stream));
        GP2S_CUDA(c, cudaStreamSynchronize(c->stream));
    }
    CholPlan P;
    chol_order(nt, words, low, P);
    // one upload: tasks (16-byte aligned), then the int lists
    const size_t lists = P.colptr.size() + P.rowpos.size() + P.rptr.size() + P.rcol.size() + P.rslot.size() + P.perm.size() +
                         P.pos.size();
    const size_t total = 4 * P.tasks.size() + lists;
    std::vector<int> up;
    up.reserve(total);
    const int *t0 = reinterpret_cast<const int *>(P.tasks.data());
    up.insert(up.end(), t0, t0 + 4 * P.tasks.size());
    for (const std::vector<int> *v : {&P.colptr, &P.rowpos, &P.rptr, &P.rcol, &P.rslot, &P.perm, &P.pos})
        up.insert(up.end(), v->begin(), v->end());
    GP2S_TRY(ensure(c, c->chol_ints, sizeof(int) * total));
    GP2S_CUDA(c, cudaMemcpyAsync(c->chol_ints.p, up.data(), sizeof(int) * total, cudaMemcpyHostToDevice, c->stream));
    GP2S_CUDA(c, cudaStreamSynchronize(c->stream));   // `up` is this call's
    c->chol_nt = nt;
    c->chol_ntiles = (int)P.rowpos.size();
    c->chol_ntasks = (int)P.tasks.size();
    c->chol_last = P.pos[nt - 1];
    c->chol_plan_valid = true;
    return GP2S_OK;
}

gp2s_status exact_logdet_solve(gp2s_ctx *c, const double *y_sorted_dev, double *logdet_hat)
{
    const Assembled &A = c->A;
    const int64_t n = A.n;
    GP2S_TRY(chol_plan(c));
    CholArgs a{};
    a.nt = c->chol_nt;
    a.ntiles = c->chol_ntiles;
    a.n = (int)n;
    a.last = c->chol_last;
    a.solve = y_sorted_dev != nullptr;
    a.ntasks = c->chol_ntasks;
    a.tasks = c->chol_ints.as<int4>();
    a.colptr = reinterpret_cast<const int *>(a.tasks + c->chol_ntasks);
    a.rowpos = a.colptr + a.nt + 1;
    a.rptr = a.rowpos + a.ntiles;
    a.rcol = a.rptr + a.nt + 1;
    a.rslot = a.rcol + (a.ntiles - a.nt);
    a.perm = a.rslot + (a.ntiles - a.nt);
    const int *pos = a.perm + a.nt;
    const size_t tile_bytes = sizeof(double) * (size_t)a.ntiles * kCTElems;
    const size_t nv = (size_t)a.nt * kCT;
    const size_t flags = chol_flag_ints(a.ntiles, a.nt);
    GP2S_TRY(ensure(c, c->dense, tile_bytes + sizeof(double) * nv * 3 + sizeof(int) * (flags + 1)));
    a.tiles = c->dense.as<double>();
    a.dinv = a.tiles + (size_t)a.ntiles * kCTElems;
    a.yv = a.dinv + nv;
    a.xv = a.yv + nv;
    a.flags = reinterpret_cast<int *>(a.xv + nv);
    a.bad = a.flags + flags;
    if (a.solve) GP2S_TRY(ensure(c, c->vec64, sizeof(double) * (size_t)n * 4 + 256));
    GP2S_CUDA(c, cudaMemsetAsync(a.tiles, 0, tile_bytes, c->stream));
    GP2S_CUDA(c, cudaMemsetAsync(a.flags, 0, sizeof(int) * (flags + 1), c->stream));
    const unsigned gb = (unsigned)std::min<int64_t>(ceil_div((int64_t)nv * 32, 256), 152 * 16);
    k_chol_fill<<<gb, 256, 0, c->stream>>>(c->rowptr.as<int32_t>(), c->col.as<int32_t>(), c->val64.as<double>(), n, a, pos);
    GP2S_LAUNCH(c);
    // a = s * (Ah^{-1} (s * y)), vec64 slot 3; slots 0 and 1 hold s * y and Ah^{-1} (s * y) for the residual
    a.b = y_sorted_dev;
    a.bs = c->s64.as<double>();
    if (a.solve) {
        a.bh = c->vec64.as<double>();
        a.xh = a.bh + n;
        a.x = a.bh + 3 * n;
    }
    ++c->launches;
    GP2S_CUDA(c, chol_launch(a, c->num_sms, c->stream));
    const int nb = 64;
    GP2S_TRY(ensure(c, c->gpart, sizeof(double) * (2 * 304 + 8)));
    k_chol_logdiag<<<nb, 256, 0, c->stream>>>(a, c->gpart.as<double>());
    GP2S_LAUNCH(c);
    int hbad = 0;
    double part[nb];
    GP2S_CUDA(c, cudaMemcpyAsync(&hbad, a.bad, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    GP2S_CUDA(c, cudaMemcpyAsync(part, c->gpart.p, sizeof(part), cudaMemcpyDeviceToHost, c->stream));
    GP2S_CUDA(c, cudaStreamSynchronize(c->stream));
    if (hbad & 2) return set_err(c, GP2S_ETIMEOUT, "Cholesky: a tile did not complete (bounded wait gave up)");
    if (hbad) return set_err(c, GP2S_ENOTPD, "Cholesky: non-positive pivot");
    double half = 0.0;
    for (int k = 0; k < nb; ++k) half += part[k];
    *logdet_hat = 2.0 * half;
    c->have_exact = true;
    c->exact_lhat = *logdet_hat;
    if (y_sorted_dev) c->have_solution = true;
    return GP2S_OK;
}

void exact_release(gp2s_ctx *c)
{
    release(c, c->dense);
    release(c, c->chol_ints);
    c->chol_plan_valid = false;
    c->have_exact = false;
}

}  // namespace gp2s
