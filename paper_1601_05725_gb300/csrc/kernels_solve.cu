// kernels_solve.cu -- x = A^{-1} b with the factors of the BTF diagonal blocks.
//
// BTF back-substitution (Sec. II and III-B: only the diagonal blocks are
// factored; the off-diagonal blocks keep A's values and enter through a
// product): blocks from last to first, c_d -= sum_{e>d} B_de z_e, then
// L_d w = P_d c_d and U_d z_d = w.  Evaluated by rows in pivot-step space, one
// warp per row and direction, claimed in a topological order:
//   forward row i   w_i = c(prow i) - sum_k L(i,k) w_k, k ascending, after the
//                   coupling terms of row prow i (later blocks' final z_j)
//   backward row i  z_i = (w_i - sum_k U(i,k) z_k) / U(i,i), k descending
// Each term waits for the value it reads (point-to-point synchronisation, Sec.
// IV) with a bounded wait.  Per solution entry the fma
// sequence is the one of the column sweeps (ascending steps for L, descending for
// U), so the result does not depend on the schedule.
//
// What bounds it: the chains of rows, and a row's serial chain of fmas (about 70
// cycles a term with the next batch's values and terms on their way; 165 when each
// batch waited for its flags, its values and its terms in turn).  The 316 x 316
// grid's solve 2.1 ms, was 3.0; eight right-hand sides, a lane each, 3.4 ms, was 67
// when they ran one after the other through the same chains.
//
// The factors are kept by columns; after every factorization bk_launch_rows
// transposes them into rows (count, scan, scatter, and a rank sort per row).
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>

#include "basker_internal.h"
#include "device_util.cuh"
#include "solve_internal.h"
#include "solve_word.cuh"
#include "trace.cuh"

using namespace bk;

namespace {

// ---------------------------------------------------------------- factors by rows

template <typename V>
__global__ void bk_rows_count(bk_dev d, bk_rows r)
{
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    int32_t *lc = r.cnt, *uc = r.cnt + d.n + 1;
    for (int c = warp; c < d.n; c += nwarps) {
        const int64_t lb = d.Lbeg[c];
        const int ln = d.Lcnt[c];
        for (int t = lane; t < ln; t += 32) {
            const int i = d.pinv[d.Li[lb + t]];
            r.Ls[lb + t] = i;
            atomicAdd(lc + i, 1);
        }
        const int64_t ub = d.Ubeg[c];
        const int un = d.Ucnt[c];
        for (int t = lane; t < un - 1; t += 32) atomicAdd(uc + d.Ui[ub + t], 1);
        if (lane == 0) vals<V>(r.Ud)[c] = vals<V>(d.Ux)[ub + un - 1];
    }
}

// Exclusive scan of m counts into m + 1 starts: per-block sums, a scan of the
// block sums, then each block's scan plus its offset.
__device__ __forceinline__ int64_t block_exscan(int64_t v, int64_t *warp_tot, int64_t &total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(BK_FULL, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) warp_tot[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        int64_t t = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : 0;
        int64_t ti = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(BK_FULL, ti, o);
            if (lane >= o) ti += y;
        }
        warp_tot[lane] = ti - t;
        if (lane == 31) warp_tot[32] = ti;
    }
    __syncthreads();
    const int64_t ex = inc - v + warp_tot[wid];
    total = warp_tot[32];
    __syncthreads();
    return ex;
}

__global__ void __launch_bounds__(1024) bk_scan_sums(const int32_t *cnt, int32_t m, int64_t *part)
{
    __shared__ int64_t wt[33];
    const int i = blockIdx.x * 1024 + threadIdx.x;
    int64_t total;
    block_exscan(i < m ? cnt[i] : 0, wt, total);
    if (threadIdx.x == 0) part[blockIdx.x] = total;
}

__global__ void __launch_bounds__(1024) bk_scan_parts(int64_t *part, int32_t nb)
{
    __shared__ int64_t wt[33];
    int64_t carry = 0;
    for (int b0 = 0; b0 < nb; b0 += 1024) {
        const int i = b0 + threadIdx.x;
        const int64_t v = i < nb ? part[i] : 0;
        int64_t total;
        const int64_t ex = block_exscan(v, wt, total);
        if (i < nb) part[i] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) part[nb] = carry;
}

__global__ void __launch_bounds__(1024) bk_scan_apply(const int32_t *cnt, int32_t m, const int64_t *part,
                                                      int64_t *out)
{
    __shared__ int64_t wt[33];
    const int i = blockIdx.x * 1024 + threadIdx.x;
    int64_t total;
    const int64_t ex = block_exscan(i < m ? cnt[i] : 0, wt, total);
    if (i < m) out[i] = part[blockIdx.x] + ex;
    if (i == 0) out[m] = part[gridDim.x];
}

// Entries of L (which = 0) or U (which = 1) into the unsorted row buffer.
template <typename V>
__global__ void bk_rows_scatter(bk_dev d, bk_rows r, int which)
{
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    int32_t *cur = r.cnt + (which ? d.n + 1 : 0);
    const int64_t *rp = which ? r.Urp : r.Lrp;
    for (int c = warp; c < d.n; c += nwarps) {
        if (which == 0) {
            const int64_t lb = d.Lbeg[c];
            const int ln = d.Lcnt[c];
            for (int t = lane; t < ln; t += 32) {
                const int i = r.Ls[lb + t];             // bk_rows_count
                const int64_t pos = rp[i] + atomicAdd(cur + i, 1);
                r.tk[pos] = c;
                vals<V>(r.tx)[pos] = vals<V>(d.Lx)[lb + t];
            }
        } else {
            const int64_t ub = d.Ubeg[c];
            const int un = d.Ucnt[c];
            for (int t = lane; t < un - 1; t += 32) {
                const int i = d.Ui[ub + t];
                const int64_t pos = rp[i] + atomicAdd(cur + i, 1);
                r.tk[pos] = c;
                vals<V>(r.tx)[pos] = vals<V>(d.Ux)[ub + t];
            }
        }
    }
}

// Each row's entries in ascending (L) or descending (U) column order: the rank of
// an entry is the number of entries of its row that come before it.  A warp a row:
//   up to 32 entries     compared with each other by shuffles, as many as there are;
//   up to BK_LONG_ROW    the columns (distinct) set bits of a map in shared memory, over
//                        the range they span if that is RS_WORDS words at most, else (U)
//                        over the row's L-space (own columns, then the ancestors'); an
//                        entry's rank is the set bits before its own.  Linear in the
//                        row's length and the map;
//                        else compared with each other, four a shared load.
// Bound by the instructions of the long rows (a comparison of every pair by shuffles
// took 256 times 32 for 512 entries).  Measured, L and U: 316 x 316 mesh (3.75 and 3.82
// million entries) 0.92 -> 0.13 ms, 8192 blocks of up to 1024 rows 1.42 -> 0.44 ms.
constexpr int RS_WARPS = 8;
constexpr int RS_WORDS = 512;

template <typename V>
__global__ void __launch_bounds__(RS_WARPS * 32) bk_rows_sort(bk_dev d, const int64_t *rp, const int32_t *tk,
                                                              const V *tx, int32_t *ok, V *ox, int desc)
{
    __shared__ __align__(16) int32_t skey[RS_WARPS][BK_LONG_ROW];
    __shared__ uint32_t sbm[RS_WARPS][RS_WORDS];
    __shared__ uint16_t spre[RS_WARPS][RS_WORDS];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int warp = blockIdx.x * RS_WARPS + wid;
    const int nwarps = gridDim.x * RS_WARPS;
    const int sentinel = desc ? INT_MIN : INT_MAX;
    int32_t *const key = skey[wid];
    uint32_t *const bm = sbm[wid];
    uint16_t *const pre = spre[wid];
    for (int i = warp; i < d.n; i += nwarps) {
        const int64_t p0 = rp[i];
        const int len = (int)(rp[i + 1] - p0);
        if (len > BK_LONG_ROW) continue;          // bk_rows_sort_long
        if (len <= 32) {
            const bool mine = lane < len;
            const int myk = mine ? tk[p0 + lane] : sentinel;
            const V myx = mine ? tx[p0 + lane] : V(0);
            int rank = 0;
            for (int t = 0; t < len; t += 4)
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int kk = __shfl_sync(BK_FULL, myk, t + u);
                    rank += desc ? (kk > myk) : (kk < myk);
                }
            if (mine) {
                ok[p0 + rank] = myk;
                ox[p0 + rank] = myx;
            }
            continue;
        }
        __syncwarp();
        int lo = INT_MAX, hi = 0;
        for (int e = lane; e < len; e += 32) {
            const int c = tk[p0 + e];
            key[e] = c;
            lo = min(lo, c);
            hi = max(hi, c);
        }
        lo = __reduce_min_sync(BK_FULL, lo);
        hi = __reduce_max_sync(BK_FULL, hi);
        if (((hi - lo) >> 5) >= RS_WORDS && desc) {
            // over the L-space of the row's task, if all columns are in it
            const bk_task &T = d.tasks[d.col_task[i]];
            if (T.lspace <= 32 * RS_WORDS) {
                bool in = true;
                for (int e = lane; e < len; e += 32) in = in && slot_of(T, T.lo, key[e]) >= 0;
                if (__all_sync(BK_FULL, in)) {
                    for (int e = lane; e < len; e += 32) key[e] = slot_of(T, T.lo, key[e]);
                    lo = 0;
                    hi = T.lspace - 1;
                }
            }
        }
        const int W = ((hi - lo) >> 5) + 1;
        __syncwarp();
        if (W <= RS_WORDS) {
            for (int w = lane; w < W; w += 32) bm[w] = 0u;
            __syncwarp();
            for (int e = lane; e < len; e += 32) {
                const int off = key[e] - lo;
                atomicOr(bm + (off >> 5), 1u << (off & 31));
            }
            __syncwarp();
            int carry = 0;
            for (int w0 = 0; w0 < W; w0 += 32) {
                const int w = w0 + lane;
                const int n = w < W ? __popc(bm[w]) : 0;
                const int ex = warp_exscan(n, lane);
                if (w < W) pre[w] = (uint16_t)(carry + ex);
                carry += __shfl_sync(BK_FULL, ex + n, 31);
            }
            __syncwarp();
            for (int e = lane; e < len; e += 32) {
                const int off = key[e] - lo;
                const int r = pre[off >> 5] + __popc(bm[off >> 5] & ((1u << (off & 31)) - 1u));
                const int rank = desc ? len - 1 - r : r;
                ok[p0 + rank] = tk[p0 + e];
                ox[p0 + rank] = tx[p0 + e];
            }
        } else {
            for (int e = len + lane; e < ((len + 3) & ~3); e += 32) key[e] = sentinel;
            __syncwarp();
            for (int e = lane; e < len; e += 32) {
                const int myk = key[e];
                int rank = 0;
                for (int t = 0; t < len; t += 4) {
                    const int4 o = *reinterpret_cast<const int4 *>(key + t);
                    rank += desc ? (o.x > myk) + (o.y > myk) + (o.z > myk) + (o.w > myk)
                                 : (o.x < myk) + (o.y < myk) + (o.z < myk) + (o.w < myk);
                }
                ok[p0 + rank] = myk;
                ox[p0 + rank] = tx[p0 + e];
            }
        }
    }
}

__global__ void bk_rows_long_list(int32_t n, const int64_t *rp, int32_t *longs)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        if (rp[i + 1] - rp[i] > BK_LONG_ROW) longs[1 + atomicAdd(longs, 1)] = i;
}

// Long rows, one block a row: the row's columns (distinct) set bits of a bitmap
// over [cmin, cmax]; an entry's rank is the number of set bits before its own,
// a prefix sum of the words' popcounts plus the popcount within its word.
// Linear in the row's length and its column range.
template <typename V>
__global__ void __launch_bounds__(1024) bk_rows_sort_long(const int64_t *rp, const int32_t *tk, const V *tx,
                                                          int32_t *ok, V *ox, int desc, const int32_t *longs,
                                                          uint32_t *sbits, int32_t *spre, int64_t swords)
{
    __shared__ int64_t wt[33];
    __shared__ int red[2][32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    uint32_t *bm = sbits + (int64_t)blockIdx.x * swords;
    int32_t *pre = spre + (int64_t)blockIdx.x * swords;
    const int nlong = longs[0];
    for (int q = blockIdx.x; q < nlong; q += gridDim.x) {
        const int i = longs[1 + q];
        const int64_t p0 = rp[i];
        const int len = (int)(rp[i + 1] - p0);
        int lo = INT_MAX, hi = -1;
        for (int e = tid; e < len; e += blockDim.x) {
            const int c = tk[p0 + e];
            lo = min(lo, c);
            hi = max(hi, c);
        }
        lo = warp_min(lo);
        hi = warp_max_i(hi);
        if (lane == 0) { red[0][wid] = lo; red[1][wid] = hi; }
        __syncthreads();
        if (wid == 0) {
            lo = lane < (int)(blockDim.x >> 5) ? red[0][lane] : INT_MAX;
            hi = lane < (int)(blockDim.x >> 5) ? red[1][lane] : -1;
            lo = warp_min(lo);
            hi = warp_max_i(hi);
            if (lane == 0) { red[0][0] = lo; red[1][0] = hi; }
        }
        __syncthreads();
        const int cmin = red[0][0];
        const int W = ((red[1][0] - cmin) >> 5) + 1;
        for (int w = tid; w < W; w += blockDim.x) bm[w] = 0u;
        __syncthreads();
        for (int e = tid; e < len; e += blockDim.x) {
            const int off = tk[p0 + e] - cmin;
            atomicOr(bm + (off >> 5), 1u << (off & 31));
        }
        __syncthreads();
        int64_t carry = 0;
        for (int w0 = 0; w0 < W; w0 += blockDim.x) {
            const int w = w0 + tid;
            const int64_t v = w < W ? __popc(bm[w]) : 0;
            int64_t total;
            const int64_t ex = block_exscan(v, wt, total);
            if (w < W) pre[w] = (int32_t)(carry + ex);
            carry += total;
        }
        __syncthreads();
        for (int e = tid; e < len; e += blockDim.x) {
            const int c = tk[p0 + e];
            const int off = c - cmin;
            const int r = pre[off >> 5] + __popc(bm[off >> 5] & ((1u << (off & 31)) - 1u));
            const int rank = desc ? len - 1 - r : r;
            ok[p0 + rank] = c;
            ox[p0 + rank] = tx[p0 + e];
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- leaf order

// Orders of an ND leaf's rows.  Backward: U(i,k) != 0 makes column k depend on
// step i in the factorization, so the factorization's column levels (d.level,
// longest chain from a source, counting only the leaf's steps for a leaf
// column) taken in decreasing order are a valid order, and one with the most
// rows at each level.  Forward: the same levels in increasing order are valid
// when every L(i,k) != 0 of the leaf has level(k) < level(i) (true for
// symmetric patterns); a leaf where that fails keeps its step order.  Each leaf's
// rows are split over `chunks` blocks (block b: leaf b / chunks, chunk b % chunks).
__global__ void bk_leaf_check(bk_dev d, bk_solve_dev s, int chunks)
{
    const int leaf = blockIdx.x / chunks, chunk = blockIdx.x % chunks;
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const bk_task &T = d.tasks[s.leaf_tasks[leaf]];
    int bad = 0;
    for (int i = T.lo + chunk * nw + wid; i < T.hi; i += nw * chunks) {
        const int li = d.level[i];
        for (int64_t e = s.r.Lrp[i] + lane; e < s.r.Lrp[i + 1]; e += 32)
            if (d.level[s.r.Lrk[e]] >= li) bad = 1;
    }
    if (__any_sync(BK_FULL, bad) && lane == 0) s.leaf_bad[leaf] = 1;
}

// Sort key of leaf row i (both below the leaf's size).
__device__ __forceinline__ int leaf_key(const bk_dev &d, const bk_solve_dev &s, int leaf, int lo, int hi, int i,
                                        int dir)
{
    if (dir == 0) return s.leaf_bad[leaf] ? i - lo : d.level[i];
    return s.leaf_maxrows - d.level[i];
}

// Counting sort of all leaf rows by level into their places of the claim order
// (a thread a row; rows of one level take their places in any order).
__global__ void bk_leaf_count(bk_dev d, bk_solve_dev s, int chunks)
{
    const int leaf = blockIdx.x / chunks, chunk = blockIdx.x % chunks;
    const bk_task &T = d.tasks[s.leaf_tasks[leaf]];
    for (int i = T.lo + chunk * blockDim.x + threadIdx.x; i < T.hi; i += blockDim.x * chunks) {
        atomicAdd(s.lcnt + leaf_key(d, s, leaf, T.lo, T.hi, i, 0), 1);
        atomicAdd(s.lcnt + (s.leaf_maxrows + 1) + leaf_key(d, s, leaf, T.lo, T.hi, i, 1), 1);
    }
}

__global__ void __launch_bounds__(1024) bk_leaf_scan(bk_solve_dev s)
{
    // exclusive scan of both count arrays (one block; counts of at most leaf_maxrows levels)
    __shared__ int64_t wt[33];
    const int m = s.leaf_maxrows + 1;
    for (int dir = 0; dir < 2; dir++) {
        int32_t *c = s.lcnt + dir * m;
        int64_t carry = 0;
        for (int b0 = 0; b0 < m; b0 += 1024) {
            const int i = b0 + threadIdx.x;
            const int64_t v = i < m ? c[i] : 0;
            int64_t total;
            const int64_t ex = block_exscan(v, wt, total);
            if (i < m) c[i] = (int32_t)(carry + ex);
            carry += total;
        }
        __syncthreads();
    }
}

__global__ void bk_leaf_scatter(bk_dev d, bk_solve_dev s, int chunks)
{
    const int leaf = blockIdx.x / chunks, chunk = blockIdx.x % chunks;
    const bk_task &T = d.tasks[s.leaf_tasks[leaf]];
    const int m = s.leaf_maxrows + 1;
    for (int i = T.lo + chunk * blockDim.x + threadIdx.x; i < T.hi; i += blockDim.x * chunks) {
        s.items[s.leaf_f0 + atomicAdd(s.lcnt + leaf_key(d, s, leaf, T.lo, T.hi, i, 0), 1)] = i;
        s.items[s.leaf_b0 + atomicAdd(s.lcnt + m + leaf_key(d, s, leaf, T.lo, T.hi, i, 1), 1)] = ~i;
    }
}

// ---------------------------------------------------------------- the solve

// A value that is not final yet is a word of ones (solve_word.cuh): a reader polls
// the value itself, so a link of the dataflow is one access, without flag or fence.

// One lane's bounded wait for the value at p, sleeping between polls.  The word of
// ones again if the wait ran out (the timeout status is then set).
template <typename V>
__device__ __forceinline__ typename SvWord<V>::U await_value(const bk_dev &d, const typename SvWord<V>::U *p,
                                                             long long budget)
{
    typedef SvWord<V> SW;
    typename SW::U v = SW::load(p);
    if (v != SW::none) return v;
    const long long t0 = clock64();
    unsigned ns = 32;
    while ((v = SW::load(p)) == SW::none) {
        if (*reinterpret_cast<const volatile int *>(&d.status->timeout) || clock64() - t0 > budget) {
            atomicExch(&d.status->timeout, 1);
            return SW::none;
        }
        __nanosleep(ns);
        ns = min(ns * 2, 128u);
    }
    return v;
}

// z -= sum over the terms [e0, e1) of a row, a_e * v(k_e), in their order, one
// right-hand side (every lane computes the same chain): 32 terms a batch, a lane
// each; the next batch's values and the one after's terms are read while a batch is
// applied.  Terms are applied as soon as every earlier one is there; the first
// missing one is polled by its lane.  The terms end before the first k with
// (k < cut) != below (cut < 0: at e1).  False if a wait ran out.
template <typename V>
__device__ __forceinline__ bool row_terms(const bk_dev &d, const typename SvWord<V>::U *src, const int32_t *rk,
                                          const int32_t *pos, const V *rx, int64_t e0, int64_t e1, int cut, bool below,
                                          long long budget, V &z)
{
    typedef SvWord<V> SW;
    typedef typename SW::U U;
    const int lane = threadIdx.x & 31;
    auto read = [&](int64_t e, int &k, V &a) {
        const bool in = e + lane < e1;
        k = in ? rk[e + lane] : -1;
        a = in ? rx[pos ? (int64_t)pos[e + lane] : e + lane] : V(0);
        if (cut >= 0 && k >= 0 && (k < cut) != below) k = -1;
    };
    int k, k1, k2;
    V a, a1, a2;
    read(e0, k, a);
    read(e0 + 32, k1, a1);
    U v = k >= 0 ? SW::load(src + k) : U(0);
    for (int64_t e = e0; e < e1; e += 32) {
        const int cnt = __popc(__ballot_sync(BK_FULL, k >= 0));
        if (cnt == 0) return true;
        const U v1 = k1 >= 0 ? SW::load(src + k1) : U(0);
        read(e + 64, k2, a2);
        for (int done = 0;;) {
            const uint32_t nr = __ballot_sync(BK_FULL, k >= 0 && v == SW::none);
            const int upto = nr ? __ffs(nr) - 1 : cnt;
            const V vv = SW::value(v);
            int t = done;
            for (; t + 4 <= upto; t += 4) {
#pragma unroll
                for (int u = 0; u < 4; u++)
                    z = fma(-__shfl_sync(BK_FULL, a, t + u), __shfl_sync(BK_FULL, vv, t + u), z);
            }
            for (; t < upto; t++) z = fma(-__shfl_sync(BK_FULL, a, t), __shfl_sync(BK_FULL, vv, t), z);
            if (upto >= cnt) break;
            done = upto;
            if (v == SW::none && k >= 0) v = lane == done ? await_value<V>(d, src + k, budget) : SW::load(src + k);
            if (__shfl_sync(BK_FULL, v == SW::none, done)) return false;
        }
        if (cnt < 32) return true;
        k = k1;
        a = a1;
        v = v1;
        k1 = k2;
        a1 = a2;
    }
    return true;
}

// The same for R right-hand sides, the lane's one being q.  Every lane reads every
// term (the same address over the warp); three groups of eight are under way: one
// applied, one with its values coming, one with its terms coming.
template <typename V>
__device__ __forceinline__ bool row_terms_multi(const bk_dev &d, const typename SvWord<V>::U *src, const int32_t *rk,
                                                const int32_t *pos, const V *rx, int64_t e0, int64_t e1, int cut,
                                                bool below, int R, int q, long long budget, V &z)
{
    typedef SvWord<V> SW;
    typedef typename SW::U U;
    constexpr int G = 8;
    auto read = [&](int64_t e, int (&k)[G], V (&a)[G]) {
#pragma unroll
        for (int u = 0; u < G; u++) {
            const bool in = e + u < e1;
            k[u] = in ? rk[e + u] : -1;
            a[u] = in ? rx[pos ? (int64_t)pos[e + u] : e + u] : V(0);
        }
        if (cut >= 0)
#pragma unroll
            for (int u = 0; u < G; u++)
                if (k[u] >= 0 && (k[u] < cut) != below) k[u] = -1;
    };
    auto values = [&](const int (&k)[G], U (&v)[G]) {
#pragma unroll
        for (int u = 0; u < G; u++) v[u] = k[u] >= 0 ? SW::load(src + (int64_t)k[u] * R + q) : U(0);
    };
    int k0[G], k1[G], k2[G];
    V a0[G], a1[G], a2[G];
    U v0[G], v1[G];
    read(e0, k0, a0);
    read(e0 + G, k1, a1);
    values(k0, v0);
    for (int64_t e = e0; k0[0] >= 0; e += G) {
        values(k1, v1);
        read(e + 2 * G, k2, a2);
        bool miss = false;
#pragma unroll
        for (int u = 0; u < G; u++) miss = miss || v0[u] == SW::none;
        if (__any_sync(BK_FULL, miss)) {
#pragma unroll
            for (int u = 0; u < G; u++)
                if (k0[u] >= 0 && v0[u] == SW::none) v0[u] = await_value<V>(d, src + (int64_t)k0[u] * R + q, budget);
            miss = false;
#pragma unroll
            for (int u = 0; u < G; u++) miss = miss || v0[u] == SW::none;
            if (__any_sync(BK_FULL, miss)) return false;
        }
#pragma unroll
        for (int u = 0; u < G; u++)
            if (k0[u] >= 0) z = fma(-a0[u], SW::value(v0[u]), z);
#pragma unroll
        for (int u = 0; u < G; u++) {
            k0[u] = k1[u];
            a0[u] = a1[u];
            v0[u] = v1[u];
            k1[u] = k2[u];
            a1[u] = a2[u];
        }
    }
    return true;
}

// ---------------------------------------------------------------- separator sweeps
//
// One block solves a separator's own triangle, its rows' outside terms already
// applied (the rows' values in s.part; in zs, in shared memory or in place in global
// memory, while they are swept).  Forward: for k ascending, w_k = zs[k] is final and L(i,k) w_k is
// subtracted from the node's rows i > k; backward: for k descending, z_k =
// zs[k] / U(k,k) is final and U(j,k) z_k is subtracted from the node's rows
// j < k.  Per row the terms come in the order of the row sweeps (ascending k
// forward, descending backward), after the outside terms; each step's terms go
// to distinct rows, spread over the block's threads, with one barrier a step.
// A column's own entries (the first ones of L(:,k), the last ones above the
// diagonal of U(:,k)) are copied into shared memory SW_P - 1 steps ahead
// (cp.async, a ring of SW_P stages of sw_win entries), and the columns' extents
// 2 SW_P steps ahead, so that a step waits for no global load.
constexpr int SW_NT = 128;     // threads of a block (the kernel's block size)
constexpr int SW_P = 8;        // pipeline stages
constexpr int SW_MR = 4 * SW_P;  // ring of column extents
constexpr int SW_WMAX = 448;   // most entries of a column a stage holds
constexpr int SW_MAXB = 64;    // most sweeper blocks
constexpr int SEP_SMEM_ROWS = 1024;   // most rows of a node swept in shared memory
constexpr int SW_ZMAX = 15 * 1024;    // most values of a node swept in shared memory (rows times right-hand sides)

__host__ __device__ constexpr size_t sw_align(size_t b) { return (b + 15) & ~(size_t)15; }

struct SwLayout {
    size_t ri, rv, rd, mb, mc, total;
};

__host__ __device__ inline SwLayout sw_layout(int win, int zrows, size_t vsize)
{
    SwLayout L;
    L.ri = sw_align((size_t)zrows * vsize);
    L.rv = L.ri + (size_t)SW_P * win * 4;
    L.rd = L.rv + (size_t)SW_P * win * vsize;
    L.mb = L.rd + sw_align((size_t)SW_P * vsize);
    L.mc = L.mb + (size_t)SW_MR * 8;
    L.total = L.mc + (size_t)SW_MR * 4;
    return L;
}

__device__ __forceinline__ void sw_cp4(void *dst, const void *src)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sa), "l"(src) : "memory");
}

__device__ __forceinline__ void sw_cp8(void *dst, const void *src)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa), "l"(src) : "memory");
}

template <typename V>
__device__ __forceinline__ void sw_cpv(V *dst, const V *src)
{
    if (sizeof(V) == 8) sw_cp8(dst, src);
    else sw_cp4(dst, src);
}

__device__ __forceinline__ void sw_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int N>
__device__ __forceinline__ void sw_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <typename V, bool MULTI>
__device__ void sep_sweep_block(const bk_dev &d, const bk_solve_dev &s, int it, int R, double *x, int ldx,
                                long long budget, const int32_t *Qout, unsigned char *smem)
{
    const int tid = threadIdx.x;
    const bool fwd = it >= 0;
    const int t = (fwd ? it : ~it) - d.n;
    // right-hand side and entry (of SW_NT / R) of this thread
    const int rr = MULTI ? R : 1;
    const int q = MULTI ? tid % rr : 0, g0 = MULTI ? tid / rr : tid, gs = MULTI ? SW_NT / rr : SW_NT;
    const bool on = g0 < gs;
    const int lo = d.tasks[t].lo, hi = d.tasks[t].hi, m = hi - lo;
    if (m <= 0) return;
    const int W = s.sw_win;
    const V *const Lx = vals<V>(d.Lx);
    const V *const Ux = vals<V>(d.Ux);
    typedef SvWord<V> SW;
    typedef typename SW::U U;
    U *const gout = reinterpret_cast<U *>(vals<V>(fwd ? s.w : s.z)) + (int64_t)lo * rr;
    U *const part = reinterpret_cast<U *>(vals<V>(s.part)) + ((int64_t)s.sepix[lo] + (fwd ? 0 : s.nsep)) * rr;
    const SwLayout Ly = sw_layout(W, s.sw_zrows * rr, sizeof(V));
    V *const zsm = reinterpret_cast<V *>(smem);
    int32_t *const ri = reinterpret_cast<int32_t *>(smem + Ly.ri);
    V *const rv = reinterpret_cast<V *>(smem + Ly.rv);
    V *const rd = reinterpret_cast<V *>(smem + Ly.rd);
    int64_t *const mb = reinterpret_cast<int64_t *>(smem + Ly.mb);
    int32_t *const mc = reinterpret_cast<int32_t *>(smem + Ly.mc);
    BK_TSTART(t0);
    V *const zs = m <= s.sw_zrows ? zsm : reinterpret_cast<V *>(part);
    bool ok = true;
    for (int r = tid; r < m * rr && ok; r += SW_NT) {
        const U v = await_value<V>(d, part + r, budget);
        ok = v != SW::none;
        // in place too: the other threads read what this one stores before the barrier, not
        // what another block has stored (a relaxed poll orders nothing)
        zs[r] = SW::value(v);
    }
    if (__syncthreads_or(!ok)) return;
    BK_TPHASE0(tp);
    // the column at sweep position p, and its own entries held by a stage
    auto col_of = [&](int p) { return lo + (fwd ? p : m - 1 - p); };
    auto own_win = [&](int p, int cnt) {
        const int kl = fwd ? p : m - 1 - p;
        return fwd ? min(min(cnt, m - 1 - kl), W) : min(min(cnt - 1, kl), W);
    };
    auto issue = [&](int p) {
        const int slot = p % SW_MR, st = p % SW_P;
        const int64_t beg = mb[slot];
        const int cnt = mc[slot];
        const int wn = own_win(p, cnt);
        const int64_t g0 = fwd ? beg : beg + cnt - 1 - wn;
        for (int e = tid; e < wn; e += SW_NT) {
            sw_cp4(ri + st * W + e, (fwd ? s.r.Ls : d.Ui) + g0 + e);
            sw_cpv(rv + st * W + e, (fwd ? Lx : Ux) + g0 + e);
        }
        if (!fwd && tid == 0) sw_cpv(rd + st, Ux + beg + cnt - 1);
    };
    {
        for (int p = tid; p < min(2 * SW_P, m); p += SW_NT) {
            const int c = col_of(p);
            mb[p % SW_MR] = fwd ? d.Lbeg[c] : d.Ubeg[c];
            mc[p % SW_MR] = fwd ? d.Lcnt[c] : d.Ucnt[c];
        }
        __syncthreads();
        for (int p = 0; p < SW_P - 1; p++) {
            if (p < m) issue(p);
            sw_commit();
        }
        V zprev = V(0);
        int kprev = -1;
        for (int p = 0; p < m; p++) {
            sw_wait<SW_P - 2>();
            __syncthreads();
            // the previous step's z (backward) is stored once every thread read it
            if (kprev >= 0 && g0 == 0 && on) zs[kprev * rr + q] = zprev;
            const int kl = fwd ? p : m - 1 - p;
            const int st = p % SW_P, slot = p % SW_MR;
            const int cnt = mc[slot];
            const int64_t beg = mb[slot];
            V v = zs[kl * rr + q];
            if (!fwd) v = v / rd[st];
            const int wn = own_win(p, cnt);
            for (int e = on ? g0 : wn; e < wn; e += gs) {
                const int r = ri[st * W + e];
                if (fwd ? r < hi : r >= lo) {
                    const int at = (r - lo) * rr + q;
                    zs[at] = fma(-rv[st * W + e], v, zs[at]);
                }
            }
            // own entries past the stage's window, read directly
            const int own = fwd ? min(cnt, m - 1 - kl) : min(cnt - 1, kl);
            for (int e = on ? W + g0 : own; e < own; e += gs) {
                const int64_t g = fwd ? beg + e : beg + cnt - 2 - e;
                const int r = fwd ? s.r.Ls[g] : d.Ui[g];
                if (fwd ? r >= hi : r < lo) break;
                const int at = (r - lo) * rr + q;
                zs[at] = fma(-(fwd ? Lx[g] : Ux[g]), v, zs[at]);
            }
            if (!fwd) {
                zprev = v;
                kprev = kl;
            }
            // extents 2 SW_P positions ahead; entries SW_P - 1 positions ahead (into
            // the stage every thread finished reading in the previous step)
            if (tid == 0 && p + 2 * SW_P < m) {
                const int pn = p + 2 * SW_P, c = col_of(pn);
                sw_cp8(mb + pn % SW_MR, fwd ? d.Lbeg + c : d.Ubeg + c);
                sw_cp4(mc + pn % SW_MR, fwd ? d.Lcnt + c : d.Ucnt + c);
            }
            if (p + SW_P - 1 < m) issue(p + SW_P - 1);
            sw_commit();
        }
        sw_wait<0>();
        __syncthreads();
        if (kprev >= 0 && g0 == 0 && on) zs[kprev * rr + q] = zprev;
        __syncthreads();
        for (int r = tid; r < m * rr; r += SW_NT) {
            const V v = zs[r];
            U vb = SW::bits(v);
            if (vb == SW::none) vb = SW::plain_nan;
            SW::store(gout + r, vb);
            if (!fwd) {
                const int row = lo + r / rr;
                x[(int64_t)(r % rr) * ldx + (Qout ? Qout[row] : row)] = (double)v;
            }
        }
        __syncthreads();
    }
    if (tid == 0) BK_TREC(d.trace, BK_TR_SOLVE, fwd ? 2 : 3, t, t0);
    BK_TPHASE(d.trace, tp, fwd ? 10 : 11, t);     // the sweep itself
}

// MULTI: R right-hand sides, one a lane (R <= 32); else one.  w and z hold row i's
// values at [i * R, (i + 1) * R).
template <typename V, bool MULTI>
__global__ void __launch_bounds__(128) bk_solve_kernel(bk_dev d, bk_solve_dev s, int32_t R,
                                                       const double *__restrict__ b, int32_t ldb, double *x,
                                                       int32_t ldx, long long budget, int32_t *counter,
                                                       const int32_t *__restrict__ Pin,
                                                       const int32_t *__restrict__ Qout)
{
    typedef SvWord<V> SW;
    typedef typename SW::U U;
    extern __shared__ __align__(16) double solve_smem[];
    const int lane = threadIdx.x & 31;
    // the first blocks sweep the separators' own triangles, in claim order
    const int nsb = min(s.nsweeps, SW_MAXB);
    if ((int)blockIdx.x < nsb) {
        for (int k = blockIdx.x; k < s.nsweeps; k += nsb) {
            sep_sweep_block<V, MULTI>(d, s, s.sweeps[k], R, x, ldx, budget, Qout,
                                      reinterpret_cast<unsigned char *>(solve_smem));
            if (__syncthreads_or(*reinterpret_cast<const volatile int *>(&d.status->timeout) != 0)) return;
        }
        return;
    }
    const V *const Bx = vals<V>(d.Bx);
    const V *const Ud = vals<V>(s.r.Ud);
    U *const gw = reinterpret_cast<U *>(vals<V>(s.w));
    U *const gz = reinterpret_cast<U *>(vals<V>(s.z));
    U *const part = reinterpret_cast<U *>(vals<V>(s.part));
    const int rr = MULTI ? R : 1, q = MULTI ? min(lane, rr - 1) : 0;
    auto terms = [&](const U *src, const int32_t *rk, const int32_t *pos, const V *rx, int64_t e0, int64_t e1, int cut,
                     bool below, V &z) {
        return MULTI ? row_terms_multi<V>(d, src, rk, pos, rx, e0, e1, cut, below, rr, q, budget, z)
                     : row_terms<V>(d, src, rk, pos, rx, e0, e1, cut, below, budget, z);
    };
    for (;;) {
        int k = 0;
        if (lane == 0) k = atomicAdd(counter, 1);
        k = __shfl_sync(BK_FULL, k, 0);
        if (k >= s.nitems) break;
        const int it = s.items[k];
        BK_TSTART(t0);
        const bool fwd = it >= 0;
        const int i = fwd ? it : ~it;
        if (i >= d.n) continue;   // a separator's sweep (the sweeper blocks take it)
        // a separator's row takes only the terms from outside its node
        const int px = s.sepix[i];
        V z;
        if (fwd) {
            // forward row i: coupling terms of row prow i, then L(i,k) for k below the node (or all)
            const int r = d.prow[i];
            const int64_t l0 = s.r.Lrp[i], l1 = s.r.Lrp[i + 1];
            z = (V)b[(int64_t)q * ldb + (Pin ? Pin[r] : r)];
            if (s.coupling && !terms(gz, s.offj, s.offpos, Bx, s.offp[r], s.offp[r + 1], -1, false, z)) return;
            if (!terms(gw, s.r.Lrk, nullptr, vals<V>(s.r.Lrx), l0, l1, px >= 0 ? s.cutlo[i] : -1, true, z)) return;
        } else {
            // backward row i: its forward result, then U(i,k) for k above the node (or all), then the diagonal
            const int64_t u0 = s.r.Urp[i], u1 = s.r.Urp[i + 1];
            const V ud = Ud[i];
            const U w = await_value<V>(d, gw + (int64_t)i * rr + q, budget);
            if (__any_sync(BK_FULL, w == SW::none)) return;
            z = SW::value(w);
            if (!terms(gz, s.r.Urk, nullptr, vals<V>(s.r.Urx), u0, u1, px >= 0 ? s.cuthi[i] : -1, false, z)) return;
            if (px < 0) z = z / ud;
        }
        U zb = SW::bits(z);
        if (zb == SW::none) zb = SW::plain_nan;
        if (MULTI ? lane < rr : lane == 0) {
            U *const to = px >= 0 ? part + ((int64_t)px + (fwd ? 0 : s.nsep)) * rr : (fwd ? gw : gz) + (int64_t)i * rr;
            SW::store(to + q, zb);
            if (!fwd && px < 0) x[(int64_t)q * ldx + (Qout ? Qout[i] : i)] = (double)z;
        }
        if (lane == 0) BK_TREC(d.trace, BK_TR_SOLVE, fwd ? 0 : 1, i, t0);
    }
}

}  // namespace

int bk_solve_blocks()
{
    // computed once, thread-safely (a function-local static)
    static const int blocks = [] {
        int dev = 0, sms = 0, per = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, bk_solve_kernel<double, false>, 128,
                                                      4 * SEP_SMEM_ROWS * sizeof(double));
        return std::max(1, sms) * std::max(1, std::min(per, 8));
    }();
    return blocks;
}

void bk_solve_sweep_setup(bk_solve_dev &s, int32_t sw_maxm)
{
    const int own = std::max(1, sw_maxm - 1);
    s.sw_win = std::min(SW_WMAX, (own + 3) & ~3);
    s.sw_zrows = std::min(std::max(sw_maxm, 1), SEP_SMEM_ROWS);
    // the FP64 layout, the larger one, serves both kernels
    s.sw_smem = sw_layout(s.sw_win, s.sw_zrows, sizeof(double)).total;
    int dev = 0, sms = 0, per[2] = {0, 0};
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // the function attribute is shared by every handle: the largest layout, once
    static const bool raised = [] {
        const int most = (int)sw_layout(SW_WMAX, SW_ZMAX, sizeof(double)).total;
        cudaFuncSetAttribute(bk_solve_kernel<double, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        cudaFuncSetAttribute(bk_solve_kernel<float, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        cudaFuncSetAttribute(bk_solve_kernel<double, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        cudaFuncSetAttribute(bk_solve_kernel<float, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        return true;
    }();
    (void)raised;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per[0], bk_solve_kernel<double, false>, SW_NT, s.sw_smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per[1], bk_solve_kernel<float, false>, SW_NT, s.sw_smem);
    for (int k = 0; k < 2; k++) s.sw_cap[k] = std::max(1, sms) * std::max(1, std::min(per[k], 8));
}

namespace {

void launch_scan(const int32_t *cnt, int32_t m, int64_t *part, int64_t *out, cudaStream_t st)
{
    const int nb = std::max(1, (m + 1023) / 1024);
    bk_scan_sums<<<nb, 1024, 0, st>>>(cnt, m, part);
    bk_scan_parts<<<1, 1024, 0, st>>>(part, nb);
    bk_scan_apply<<<nb, 1024, 0, st>>>(cnt, m, part, out);
}

}  // namespace

void bk_launch_rows(const bk_dev &d, const bk_rows &r, void *stream)
{
    if (d.n <= 0) return;
    cudaStream_t st = (cudaStream_t)stream;
    const int n = d.n;
    const int blocks = std::max(1, std::min((n + 7) / 8, 152 * 8));
    cudaMemsetAsync(r.cnt, 0, sizeof(int32_t) * 2 * ((size_t)n + 1), st);
    if (d.prec)
        bk_rows_count<float><<<blocks, 256, 0, st>>>(d, r);
    else
        bk_rows_count<double><<<blocks, 256, 0, st>>>(d, r);
    launch_scan(r.cnt, n, r.part, r.Lrp, st);
    launch_scan(r.cnt + n + 1, n, r.part, r.Urp, st);
    cudaMemsetAsync(r.cnt, 0, sizeof(int32_t) * 2 * ((size_t)n + 1), st);
    const int lblocks = std::max(1, std::min((n + 255) / 256, 152 * 8));
    for (int which = 0; which < 2; which++) {
        const int64_t *rp = which ? r.Urp : r.Lrp;
        int32_t *ok = which ? r.Urk : r.Lrk;
        double *ox = which ? r.Urx : r.Lrx;
        cudaMemsetAsync(r.longs, 0, sizeof(int32_t), st);
        bk_rows_long_list<<<lblocks, 256, 0, st>>>(n, rp, r.longs);
        if (d.prec) {
            bk_rows_scatter<float><<<blocks, 256, 0, st>>>(d, r, which);
            bk_rows_sort<float><<<blocks, RS_WARPS * 32, 0, st>>>(d, rp, r.tk, vals<float>(r.tx), ok, vals<float>(ox), which);
            bk_rows_sort_long<float><<<BK_LONG_CTAS, 1024, 0, st>>>(rp, r.tk, vals<float>(r.tx), ok, vals<float>(ox),
                                                                     which, r.longs, r.sbits, r.spre, r.swords);
        } else {
            bk_rows_scatter<double><<<blocks, 256, 0, st>>>(d, r, which);
            bk_rows_sort<double><<<blocks, RS_WARPS * 32, 0, st>>>(d, rp, r.tk, r.tx, ok, ox, which);
            bk_rows_sort_long<double><<<BK_LONG_CTAS, 1024, 0, st>>>(rp, r.tk, r.tx, ok, ox, which, r.longs, r.sbits,
                                                                      r.spre, r.swords);
        }
    }
}

void bk_launch_leaf_order(const bk_dev &d, const bk_solve_dev &s, void *stream)
{
    if (s.tasks) {
        bk_launch_torder(d, s, stream);
        return;
    }
    if (s.nleaves <= 0) return;
    cudaStream_t st = (cudaStream_t)stream;
    // each leaf's rows over up to 32 blocks of 256 threads
    const int chunks = std::max(1, std::min((s.leaf_maxrows + 255) / 256, 32));
    const unsigned grid = (unsigned)s.nleaves * (unsigned)chunks;
    cudaMemsetAsync(s.leaf_bad, 0, sizeof(int32_t) * (size_t)s.nleaves, st);
    bk_leaf_check<<<grid, 256, 0, st>>>(d, s, chunks);
    cudaMemsetAsync(s.lcnt, 0, sizeof(int32_t) * 2 * ((size_t)s.leaf_maxrows + 1), st);
    bk_leaf_count<<<grid, 256, 0, st>>>(d, s, chunks);
    bk_leaf_scan<<<1, 1024, 0, st>>>(s);
    bk_leaf_scatter<<<grid, 256, 0, st>>>(d, s, chunks);
}

// Right-hand sides of a batch: a lane each, and every job's values in shared memory.
static int solve_batch(const bk_solve_dev &s, int32_t nrhs)
{
    int r = std::min(nrhs, 32);
    if (s.tasks) r = std::min<int>(r, std::max(1, (int)(BK_TSOLVE_SMEM / 8 / std::max(s.tmax, 1))));
    return r;
}

int bk_solve_kernels(const bk_solve_dev &s, int32_t nrhs)
{
    const int r = std::max(1, solve_batch(s, nrhs));
    const int each = (s.nitems > 0) + (s.tasks ? (s.njobs_a > 0) + (s.njobs_c > 0) : 0);
    return (nrhs + r - 1) / r * each;
}

void bk_launch_solve(const bk_dev &d, const bk_solve_dev &s0, int32_t nrhs, const double *b, int32_t ldb,
                     double *x, int32_t ldx, long long budget, void *stream, bool permute,
                     int max_ctas)
{
    const int32_t *Pin = permute ? d.P : nullptr, *Qout = permute ? d.Q : nullptr;
    cudaStream_t st = (cudaStream_t)stream;
    const int batch = solve_batch(s0, nrhs);
    int32_t *const counter = d.counter + 8;
    for (int32_t q0 = 0; q0 < nrhs; q0 += batch) {
        const int R = std::min(batch, nrhs - q0);
        bk_solve_dev s = s0;
        const double *const bq = b + (int64_t)q0 * ldb;
        double *const xq = x + (int64_t)q0 * ldx;
        cudaMemsetAsync(counter, 0, 3 * sizeof(int32_t), st);
        // no value yet (jobs without separators wait for one another only through
        // the coupling, by their solution)
        const size_t vs = d.prec ? sizeof(float) : sizeof(double);
        if (s.nitems > 0) {
            cudaMemsetAsync(s.w, 0xff, (size_t)d.n * R * vs, st);
            if (s.nsep > 0) cudaMemsetAsync(s.part, 0xff, (size_t)s.nsep * 2 * R * vs, st);
        }
        if (s.nitems > 0 || s.coupling) cudaMemsetAsync(s.z, 0xff, (size_t)d.n * R * vs, st);
        if (s.tasks)
            bk_launch_tsolve(d, s, s.jobs_a, s.njobs_a, counter, R, bq, ldb, xq, ldx, budget, permute, stream);
        if (s.nitems > 0) {
            // sweeper blocks first, then the row warps' blocks; every block co-resident
            const int nsb = std::min(s.nsweeps, SW_MAXB);
            int cap = s.sw_cap[d.prec ? 1 : 0];
            size_t smem = s.sw_smem;
            if (R > 1) {
                s.sw_zrows = std::min(s.sw_zrows, SW_ZMAX / R);
                smem = sw_layout(s.sw_win, s.sw_zrows * R, sizeof(double)).total;
                int dev = 0, sms = 0, per = 0;
                cudaGetDevice(&dev);
                cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
                if (d.prec) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, bk_solve_kernel<float, true>, SW_NT, smem);
                else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, bk_solve_kernel<double, true>, SW_NT, smem);
                cap = std::max(1, sms) * std::max(1, std::min(per, 8));
            }
            const int limit = max_ctas > 0 ? std::min(max_ctas, cap) : cap;
            const int ctas = nsb + std::max(1, std::min<int>((s.nitems + 3) / 4, limit - nsb));
            if (d.prec) {
                if (R > 1) bk_solve_kernel<float, true><<<ctas, SW_NT, smem, st>>>(d, s, R, bq, ldb, xq, ldx, budget, counter + 2, Pin, Qout);
                else bk_solve_kernel<float, false><<<ctas, SW_NT, smem, st>>>(d, s, R, bq, ldb, xq, ldx, budget, counter + 2, Pin, Qout);
            } else {
                if (R > 1) bk_solve_kernel<double, true><<<ctas, SW_NT, smem, st>>>(d, s, R, bq, ldb, xq, ldx, budget, counter + 2, Pin, Qout);
                else bk_solve_kernel<double, false><<<ctas, SW_NT, smem, st>>>(d, s, R, bq, ldb, xq, ldx, budget, counter + 2, Pin, Qout);
            }
        }
        if (s.tasks)
            bk_launch_tsolve(d, s, s.jobs_c, s.njobs_c, counter + 1, R, bq, ldb, xq, ldx, budget, permute,
                             stream);
    }
}
