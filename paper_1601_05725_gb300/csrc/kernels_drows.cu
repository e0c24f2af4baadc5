// kernels_drows.cu -- the in-node phase of an ND separator as a dense right-looking
// elimination with the block's rows dealt over a cluster of thread blocks.
//
// The computation is that of kernels_dense.cu (which stays for blocks too large for
// the cluster's shared memory): step k chooses column k's pivot (threshold partial
// pivoting, the preferred row first), divides, and updates the later columns whose
// pattern holds the pivot row, one fma an entry, in ascending step order: the factors
// are Algorithm 1's bit for bit.
//
// What bounds it.  The steps are a chain.  With whole columns dealt over the blocks a
// step was 10,000 cycles: the owner's five barriers around the pivot search, a cluster
// barrier, every block dividing the whole column again (an SM has two FP64 lanes a
// cycle, and a warp's FP64 instruction holds them for 16 to 19 cycles whatever its
// lanes, so work repeated in each warp or block is not free), and reads of the owner's
// memory behind the barrier.  Here row sl of the block belongs to block sl mod CN of the
// cluster, so that a step's division, its update of the next column and the pivot search
// are over lsp / CN rows in each block; the patterns (words, U counts) are kept by every
// block, which brings them up to date by itself.  Two messages a step cross the cluster,
// written into the other blocks' shared memory and counted by a barrier there (st.async,
// mbarrier) without a cluster-wide barrier: each block's best row, to all; and the pivot
// row, from the block that holds it, to all, during the division.  Step k:
//   X  warp 0: the best own row of column k -> all blocks; their rows; the pivot
//      the other warps: step k - 1 on the columns after k (a warp has 32 columns, or 32
//      rows, and every G-th row, or column); L(:, step k - 1) stored     block barrier
//   Y  DR_DIV warps: L = rows / pivot; the step on column k + 1 when the pivot row is there
//      the other warps: the holder sends the pivot row; patterns and U counts of the later
//      columns                                                           block barrier
// What is left of a step is the latency of its dependent instructions (shared loads of
// 60 to 85 cycles, reductions over a warp of 35 to 55, the division 575, a message 500):
// some 4,300 cycles in FP32 and, with the FP64 lanes shared by the later columns'
// update, 7,300 in FP64.
// Measured (a 316 x 316 mesh, 16 leaves: separators of 78, 157, 158 and 316 columns, FP64):
// 3.6 -> 2.6 ms a factorization; 149 x 149, 8 leaves, FP32: 1.27 -> 0.62; 61 x 61 (one
// block, 30 and 61 columns): 0.40 -> 0.26.  1,024 threads a block: 2.9, 0.74, 0.30 ms; 256:
// 3.5, 0.72, 0.28; clusters of 16 blocks were 12 % slower than of 8; the division and the
// pivot search run ahead of the block barrier, with the barriers of two groups of warps: no gain.
#include <cuda_runtime.h>

#include <climits>
#include <mutex>

#include <cooperative_groups.h>

#include "basker_internal.h"
#include "device_util.cuh"
#include "trace.cuh"

using namespace bk;
namespace cg = cooperative_groups;

namespace {

constexpr int DR_THREADS = 512;
constexpr int DR_WARPS = DR_THREADS / 32;
constexpr int DR_DIV = 4;                      // warps that divide

struct DrShared {
    bk_task T;
    unsigned long long mb1[2], mb2[2];   // arrivals of the best rows, of the pivot row (by step parity)
    int flag[2];                         // a U region is full (by step parity)
    int nrows[2];                        // own rows of the step's L column (by step parity)
    int cnt, lover;                      // column k: entries of its pattern, L region too small
    int stopreq;                         // an earlier failure elsewhere (block 0), or this block's wait budget is spent
    int stop;                            // leave
    int ok, ps, hnext;                   // the step's pivot: found, its slot, in the next column's pattern
    unsigned long long xp;               // its value
};

__device__ __forceinline__ uint32_t dr_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t dr_map(uint32_t a, int rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

// A value as a message's word, and back.
__device__ __forceinline__ unsigned long long dr_word(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ unsigned long long dr_word(float v) { return (unsigned)__float_as_int(v); }
template <typename V> __device__ __forceinline__ V dr_value(unsigned long long w);
template <> __device__ __forceinline__ double dr_value<double>(unsigned long long w)
{
    return __longlong_as_double((long long)w);
}
template <> __device__ __forceinline__ float dr_value<float>(unsigned long long w)
{
    return __int_as_float((int)(unsigned)w);
}

// The largest of the lanes' keys (integer reductions, high words first).
__device__ __forceinline__ unsigned long long dr_max(unsigned long long k)
{
    const unsigned hi = __reduce_max_sync(BK_FULL, (unsigned)(k >> 32));
    const unsigned lo = __reduce_max_sync(BK_FULL, (unsigned)(k >> 32) == hi ? (unsigned)k : 0u);
    return ((unsigned long long)hi << 32) | lo;
}

// two 8-byte words into block rank's shared memory (16-byte aligned), counted there
__device__ __forceinline__ void dr_send(const void *dst, const void *bar, int rank, unsigned long long a,
                                        unsigned long long b)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(
                     dr_map(dr_addr(dst), rank)),
                 "l"(a), "l"(b), "r"(dr_map(dr_addr(bar), rank))
                 : "memory");
}

__device__ __forceinline__ void dr_expect(const void *bar, int bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(dr_addr(bar)), "r"(bytes) : "memory");
}

// A step's messages.  A wait longer than the budget times the call out, but the messages
// are still taken: the block says so in its next one (stopreq), and every block leaves
// after the same step, with nothing under way to one that has left.  Only a message that
// never comes ends the wait itself, BK_DENSE_WAIT cycles later.  (The first look does not
// block, so that a budget of a few cycles is noticed.)
__device__ __forceinline__ bool dr_wait(const bk_dev &d, DrShared &S, const void *bar, int parity, long long budget)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(dr_addr(bar)), "r"(parity)
        : "memory");
    if (done) return true;
    const long long t0 = clock64();
    bool told = false;
    for (;;) {
        const long long t = clock64() - t0;
        if (t > budget) {
            if (!told) {
                atomicExch(&d.status->timeout, 1);
                S.stopreq = 1;
                told = true;
            }
            if (t - budget > BK_DENSE_WAIT) return false;
        }
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(dr_addr(bar)), "r"(parity)
            : "memory");
        if (done) return true;
    }
}

// a / b for 0 <= a < 4096, 0 < b < 64
__device__ __forceinline__ int dr_div(int a, int b) { return (int)__fdividef((float)a + 0.5f, (float)b); }

// Shared memory of a block with the node's rows dealt over cn blocks, in bytes.
__host__ __device__ inline size_t dr_bytes(int own, int lsp, int cn)
{
    const size_t nrw = ((size_t)lsp + 31) / 32, rl = ((size_t)lsp + cn - 1) / cn;
    const size_t words = 2 * 2 * ((size_t)cn + 1) + 2 * (((size_t)own + 3) & ~(size_t)1) + 4 * (size_t)own + rl +
                         rl * (size_t)(own | 1);
    return words * 8 + (2 * (size_t)own + rl + 2 * nrw + (size_t)own * nrw) * 4 + 2 * (size_t)own + 16;
}

template <typename V, int CN>
__global__ void __launch_bounds__(DR_THREADS, 1) bk_dense_rows_kernel(bk_dev d, const int32_t *__restrict__ task_ids,
                                                                   double tau, int pref_mode, long long budget)
{
    V *const Lx = vals<V>(d.Lx);
    V *const Ux = vals<V>(d.Ux);
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    __shared__ __align__(16) DrShared S;
    extern __shared__ __align__(16) unsigned char dsm[];
    const int tx = threadIdx.x, lane = tx & 31, wid = tx >> 5;
    const int tid = task_ids[blockIdx.x / CN];
    BK_TSTART(t0);
    if (wid == 0) load_task(S.T, d.tasks + tid, lane);
    if (tx == 0) {
        for (int i = 0; i < 2; i++) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(dr_addr(&S.mb1[i])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(dr_addr(&S.mb2[i])) : "memory");
            S.flag[i] = 0;
            S.nrows[i] = 0;
        }
        S.stop = S.stopreq = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const bk_task &T = S.T;
    const int nown = T.hi - T.lo, lsp = T.lspace, nrw = (lsp + 31) >> 5;
    const int Rl = (lsp + CN - 1) / CN;              // own rows, at most: slot rl * CN + rank
    const int ld = nown | 1;                         // odd: a column's rows on distinct banks
    const int nown2 = (nown + 3) & ~1;
    ulonglong2 *const msg = reinterpret_cast<ulonglong2 *>(dsm);                 // [2][CN + 1]
    unsigned long long *const mrow = reinterpret_cast<unsigned long long *>(msg + 2 * (CN + 1));     // [2][nown2]
    int64_t *const ubs = reinterpret_cast<int64_t *>(mrow + 2 * nown2);
    int64_t *const ues = ubs + nown;
    int64_t *const lbs = ues + nown;
    int64_t *const les = lbs + nown;
    V *const lcol = reinterpret_cast<V *>(les + nown);                           // [Rl], in 8-byte slots
    V *const loc = reinterpret_cast<V *>(les + nown + Rl);                       // [Rl][ld]
    int32_t *const nus = reinterpret_cast<int32_t *>(les + nown + Rl + (int64_t)Rl * ld);
    int32_t *const prs = nus + nown;
    int32_t *const rows = prs + nown;                                            // [Rl]
    int32_t *const wpre = rows + Rl;                                             // [2][nrw]
    uint32_t *const bits = reinterpret_cast<uint32_t *>(wpre + 2 * nrw);         // [nown][nrw]
    unsigned char *const hit = reinterpret_cast<unsigned char *>(bits + (int64_t)nown * nrw);
    unsigned char *const cbad = hit + nown;

    const V *const A = vals<V>(d.ahat) + T.ahoff;          // column k at A + k * lsp
    const uint32_t *const AB = d.abits + T.aboff;          // column k at AB + k * nrw
    for (int k = tx; k < nown; k += DR_THREADS) {
        const int c = T.lo + k;
        ubs[k] = d.Ubeg[c];
        ues[k] = d.Uend[c];
        lbs[k] = d.Lbeg[c];
        les[k] = d.Lend[c];
        nus[k] = d.dcnt[c];
        prs[k] = (pref_mode ? d.pref[c] : c) - T.lo;
        hit[k] = 0;
        cbad[k] = 0;
    }
    for (int64_t e = tx; e < (int64_t)nown * nrw; e += DR_THREADS) bits[e] = AB[e];
    __syncthreads();
    // (entries outside the patterns hold stale values: zero)
    for (int64_t e = tx; e < (int64_t)nown * Rl; e += DR_THREADS) {
        const int k = (int)(e / Rl), rl = (int)(e % Rl), sl = rl * CN + rank;
        V v = V(0);
        if (sl < lsp && ((bits[(int64_t)k * nrw + (sl >> 5)] >> (sl & 31)) & 1u)) v = A[(int64_t)k * lsp + sl];
        loc[(int64_t)rl * ld + k] = v;
    }
    // an earlier failure: the first messages say so, and no step runs
    if (rank == 0 && tx == 0 && should_stop(d, tid, T.lo)) S.stopreq = 1;
    cl.sync();

    // L(:, step j) from lcol, its pivot slot pp (the last DR_DIV warps)
    auto store_l = [&](int j, int pp) {
        const uint32_t *const jb = bits + (int64_t)j * nrw;
        for (int q = tx - 32 * (DR_WARPS - DR_DIV); q < S.nrows[j & 1]; q += 32 * DR_DIV) {
            const int rl = rows[q], sl = rl * CN + rank;
            const uint32_t w = jb[sl >> 5];
            const int64_t pos =
                lbs[j] + wpre[(j & 1) * nrw + (sl >> 5)] + __popc(w & ((1u << (sl & 31)) - 1u)) - (pp < sl);
            d.Li[pos] = row_of_lslot(T, sl);
            Lx[pos] = lcol[rl];
        }
    };
    int psp = -1;
    for (int k = 0; k < nown; ++k) {
        const int c = T.lo + k, b = k & 1, par = (k >> 1) & 1;
        const uint32_t *const kb = bits + (int64_t)k * nrw;
        const int pr = prs[k];
        const bool prefok = pr >= 0 && pr < nown && ((kb[pr >> 5] >> (pr & 31)) & 1u);
        // ---- X
        if (wid == 0) {
            if (lane == 0) dr_expect(&S.mb1[b], CN * 16 + (prefok ? 16 : 0));
            bool bad = cbad[k] != 0;
            unsigned long long kmax = 0;
            int best = INT_MAX;
            for (int rl = lane; rl < Rl; rl += 32) {
                const int sl = rl * CN + rank;
                if (sl >= lsp || !((kb[sl >> 5] >> (sl & 31)) & 1u)) continue;
                const unsigned long long key = mag_key(loc[rl * ld + k]);
                if (key >= key_inf<V>()) bad = true;
                if (sl < nown && (best == INT_MAX || key > kmax)) {
                    kmax = key;
                    best = sl;
                }
            }
            unsigned long long wmax = dr_max(best == INT_MAX ? 0 : kmax);
            best = __reduce_min_sync(BK_FULL, best != INT_MAX && kmax == wmax ? best : INT_MAX);
            bad = __any_sync(BK_FULL, bad);
            const bool leave = *reinterpret_cast<const volatile int *>(&S.stopreq) != 0;
            if (lane < CN) {
                dr_send(msg + b * (CN + 1) + rank, &S.mb1[b], lane,
                        best == INT_MAX ? 0ull : dr_word(loc[(best / CN) * ld + k]),
                        (unsigned)best | (bad ? 1ull << 32 : 0ull) | (leave ? 1ull << 33 : 0ull));
                if (prefok && pr % CN == rank)
                    dr_send(msg + b * (CN + 1) + CN, &S.mb1[b], lane, dr_word(loc[(pr / CN) * ld + k]), 0ull);
            }
            // every block's best row: the pivot
            bool ok = dr_wait(d, S, &S.mb1[b], par, budget);
            if (__all_sync(BK_FULL, ok)) {
                unsigned long long v = 0, meta = (unsigned)INT_MAX;
                if (lane < CN) {
                    const ulonglong2 w = msg[b * (CN + 1) + lane];
                    v = w.x;
                    meta = w.y;
                }
                const int slot = (int)(unsigned)meta;
                const unsigned long long key = slot == INT_MAX ? 0 : mag_key(dr_value<V>(v));
                wmax = dr_max(key);
                int ps = __reduce_min_sync(BK_FULL, slot != INT_MAX && key == wmax ? slot : INT_MAX);
                bad = __any_sync(BK_FULL, (meta >> 32) & 1ull);
                const bool stop = __any_sync(BK_FULL, (meta >> 33) & 1ull);
                ok = !stop && !bad && ps != INT_MAX && wmax > 0;
                if (ok) {
                    unsigned long long xw = __shfl_sync(BK_FULL, v, ps % CN);
                    if (prefok) {
                        const unsigned long long pw = msg[b * (CN + 1) + CN].x;
                        // (the preferred row holding the maximum needs no FP64 instruction)
                        if ((tau <= 1.0 && mag_key(dr_value<V>(pw)) == wmax) ||
                            (double)fabs(dr_value<V>(pw)) >= tau * (double)key_value<V>(wmax)) {
                            ps = pr;
                            xw = pw;
                        }
                    }
                    if (lane == 0) {
                        S.ps = ps;
                        S.xp = xw;
                        S.hnext = k + 1 < nown && ((kb[nrw + (ps >> 5)] >> (ps & 31)) & 1u);
                    }
                } else if (!stop && rank == 0 && lane == 0) {
                    report_fail(d.status, c, bad ? BK_CODE_NAN : BK_CODE_SINGULAR);
                }
            } else {
                ok = false;
            }
            if (lane == 0) S.ok = ok;
        } else {
            if (wid == 1) {
                // ranks of the column's pattern
                int carry = 0;
                for (int w0 = 0; w0 < nrw; w0 += 32) {
                    const int w = w0 + lane;
                    const int n = w < nrw ? __popc(kb[w]) : 0;
                    const int pre = warp_exscan(n, lane);
                    if (w < nrw) wpre[b * nrw + w] = carry + pre;
                    carry += __shfl_sync(BK_FULL, pre + n, 31);
                }
                if (lane == 0) {
                    S.cnt = carry;
                    S.lover = lbs[k] + carry - 1 > les[k];
                }
            } else if (wid == DR_WARPS - 1 && rank == 0 && lane == 0 && (k & 15) == 0 && k > 0) {
                if (should_stop(d, tid, c)) S.stopreq = 1;
            }
            if (k > 0) {
                // step k - 1 on the columns after k (column k has it): lanes over columns
                // or over rows, whichever fills the warps better (an FP64 instruction
                // costs the same for one lane as for 32)
                const unsigned long long *const mr = mrow + (b ^ 1) * nown2;
                if (wid >= DR_WARPS - DR_DIV) store_l(k - 1, psp);
                const int nr = S.nrows[b ^ 1], nc = nown - k - 1;
                const int nch = (nc + 31) >> 5, nrh = (nr + 31) >> 5;
                if (nch * nr <= nrh * nc) {
                    const int G = nch > 0 ? max(1, dr_div(DR_WARPS - 1, nch)) : 0;
                    for (int it = wid - 1; it < nch * G; it += DR_WARPS - 1) {
                        const int g = dr_div(it, nch), c2 = k + 1 + (it - g * nch) * 32 + lane;
                        const bool on = c2 < nown && hit[c2] != 0;
                        if (!__any_sync(BK_FULL, on)) continue;
                        const V m = on ? dr_value<V>(mr[c2]) : V(0);
                        if (on && g == 0 && mag_key(m) >= key_inf<V>()) cbad[c2] = 1;
                        V *const a = loc + (on ? c2 : k + 1);
                        int q = g;
                        for (; q + 3 * G < nr; q += 4 * G) {
                            int r[4];
                            V l[4], v[4];
#pragma unroll
                            for (int u = 0; u < 4; u++) r[u] = rows[q + u * G];
#pragma unroll
                            for (int u = 0; u < 4; u++) {
                                l[u] = lcol[r[u]];
                                v[u] = a[r[u] * ld];
                            }
#pragma unroll
                            for (int u = 0; u < 4; u++)
                                if (on) a[r[u] * ld] = fma(-l[u], m, v[u]);
                        }
                        for (; q < nr; q += G) {
                            const int r = rows[q];
                            if (on) a[r * ld] = fma(-lcol[r], m, a[r * ld]);
                        }
                    }
                } else {
                    const int G = max(1, dr_div(DR_WARPS - 1, nrh));
                    for (int it = wid - 1; it < nrh * G; it += DR_WARPS - 1) {
                        const int g = dr_div(it, nrh), q = (it - g * nrh) * 32 + lane;
                        const bool on = q < nr;
                        const int r = rows[on ? q : 0];
                        const V l = lcol[r];
                        V *const a = loc + r * ld;
                        for (int c0 = k + 1 + g; c0 < nown; c0 += 4 * G) {
                            V m[4], v[4];
                            bool h[4];
#pragma unroll
                            for (int u = 0; u < 4; u++) {
                                const int c2 = c0 + u * G;
                                h[u] = c2 < nown && hit[c2] != 0;
                                m[u] = h[u] ? dr_value<V>(mr[c2]) : V(0);
                                v[u] = h[u] ? a[c2] : V(0);
                            }
#pragma unroll
                            for (int u = 0; u < 4; u++) {
                                if (!h[u]) continue;
                                if (on) a[c0 + u * G] = fma(-l, m[u], v[u]);
                                if (q == 0 && mag_key(m[u]) >= key_inf<V>()) cbad[c0 + u * G] = 1;
                            }
                        }
                    }
                }
            }
        }
        __syncthreads();
        // ---- Y
        bool go = S.ok != 0;
        const int ps = go ? S.ps : 0;
        const V xp = dr_value<V>(S.xp);
        if (go && S.lover) {
            // the L region is too small (every block finds this): a larger one
            cl.sync();
            if (rank == 0 && tx == 0) {
                const int64_t cap = min((long long)(2 * (int64_t)(S.cnt - 1) + 16),
                                        (long long)((T.hi - c - 1) + (lsp - nown)));
                const int64_t nb = pool_alloc(d.pool, d.lpool_end, cap);
                if (nb < 0) report_overflow(d, T, tid, c, 1);
                else {
                    d.Lbeg[c] = nb;
                    d.Lend[c] = nb + cap;
                }
                for (int r = 0; r < CN; r++) {
                    if (nb < 0) *cl.map_shared_rank(&S.stop, r) = 1;
                    else *cl.map_shared_rank(lbs + k, r) = nb;
                }
            }
            cl.sync();
            if (S.stop) go = false;
        }
        const int psr = ps % CN;
        const int p0 = (k + 1) & ~1, np = nown > k + 1 ? (nown - p0 + 1) >> 1 : 0;    // the pivot row, in pairs
        if (go) {
            if (tx == 0) {
                dr_expect(&S.mb2[b], np * 16);
                S.flag[b ^ 1] = 0;
                S.nrows[b ^ 1] = 0;
            }
            const V *const pl = loc + (ps / CN) * ld;
            if (wid < DR_DIV) {
                // L(:,c) = x / pivot over the own rows of the pattern
                for (int r0 = 32 * wid; r0 < Rl; r0 += 32 * DR_DIV) {
                    const int rl = r0 + lane, sl = rl * CN + rank;
                    const uint32_t w = rl < Rl && sl < lsp ? kb[sl >> 5] : 0u;
                    const bool in = ((w >> (sl & 31)) & 1u) && sl != ps;
                    const uint32_t all = __ballot_sync(BK_FULL, in);
                    int at = 0;
                    if (lane == 0 && all) at = atomicAdd(&S.nrows[b], __popc(all));
                    if (in) lcol[rl] = loc[rl * ld + k] / xp;
                    at = __shfl_sync(BK_FULL, at, 0);
                    if (in) rows[at + __popc(all & ((1u << lane) - 1u))] = rl;
                }
                // the step on the next column, as soon as the pivot row is there
                go = dr_wait(d, S, &S.mb2[b], par, budget);
                if (go && S.hnext) {
                    const unsigned long long mw = mrow[b * nown2 + k + 1];
                    const V m = dr_value<V>(mw);
                    if (tx == 0 && mag_key(m) >= key_inf<V>()) cbad[k + 1] = 1;
                    for (int rl = tx; rl < Rl; rl += 32 * DR_DIV) {
                        const int sl = rl * CN + rank;
                        if (sl >= lsp || sl == ps || !((kb[sl >> 5] >> (sl & 31)) & 1u)) continue;
                        loc[rl * ld + k + 1] = fma(-lcol[rl], m, loc[rl * ld + k + 1]);
                    }
                }
            } else {
                if (rank == psr)
                    for (int it = tx - 32 * DR_DIV; it < np * CN; it += DR_THREADS - 32 * DR_DIV) {
                        const int q = it / CN, c2 = p0 + 2 * q;
                        dr_send(mrow + b * nown2 + c2, &S.mb2[b], it - q * CN, dr_word(pl[c2]),
                                c2 + 1 < nown ? dr_word(pl[c2 + 1]) : 0ull);
                    }
                if (rank == 0 && tx == DR_THREADS - 1) {
                    const int64_t u = ubs[k] + nus[k];
                    const int piv = T.lo + ps;
                    d.Ui[u] = c;
                    Ux[u] = xp;
                    d.Ucnt[c] = nus[k] + 1;
                    d.Lcnt[c] = S.cnt - 1;
                    d.pinv[piv] = c;
                    d.prow[c] = piv;
                    if (piv != c) atomicAdd(&d.status->offdiag, 1);
                }
                // the later columns whose pattern holds the pivot row take step k: U(k, c2)
                // (its entry, which leaves the column) and the pattern of L (8 lanes a column)
                const int l8 = lane & 7, pw = ps >> 5;
                const uint32_t pb = 1u << (ps & 31);
                for (int q0 = k + 1 + 4 * (wid - DR_DIV); q0 < nown; q0 += 4 * (DR_WARPS - DR_DIV)) {
                    const int c2 = q0 + (lane >> 3);
                    const bool in = c2 < nown;
                    uint32_t *const b2 = bits + (int64_t)(in ? c2 : k) * nrw;
                    const bool h = in && (b2[pw] & pb) != 0u;
                    __syncwarp();
                    if (h)
                        for (int w = l8; w < nrw; w += 8) {
                            const uint32_t v = b2[w] | kb[w];
                            b2[w] = w == pw ? v & ~pb : v;
                        }
                    if (in && l8 == 0) {
                        hit[c2] = h;
                        if (h) {
                            const int nu = nus[c2];
                            const int64_t u = ubs[c2] + nu;
                            nus[c2] = nu + 1;
                            if (u + 2 > ues[c2]) {
                                hit[c2] = 2;
                                S.flag[b] = 1;
                            } else if (rank == psr) {
                                d.Ui[u] = c;
                                Ux[u] = pl[c2];
                            }
                        }
                    }
                }
            }
        }
        if (__syncthreads_or(!go)) break;
        psp = ps;
        if (k == nown - 1 && wid >= DR_WARPS - DR_DIV) store_l(k, ps);
        if (S.flag[b]) {
            // U regions that are full (every block finds them): larger ones
            cl.sync();
            if (rank == 0)
                for (int c2 = k + 1 + tx; c2 < nown; c2 += DR_THREADS) {
                    if (hit[c2] != 2) continue;
                    const int nu = nus[c2] - 1;
                    const int64_t ub = ubs[c2], cap = grown_ucap(nu, (int64_t)(T.lo + c2 - T.sp_lo) + 1);
                    const int64_t nb = pool_alloc(d.pool + 1, d.upool_end, cap);
                    if (nb < 0) {
                        report_overflow(d, T, tid, T.lo + c2, 2);
                        for (int r = 0; r < CN; r++) *cl.map_shared_rank(&S.stop, r) = 1;
                        continue;
                    }
                    for (int q = 0; q < nu; q++) {
                        d.Ui[nb + q] = __ldcg(d.Ui + ub + q);
                        Ux[nb + q] = __ldcg(Ux + ub + q);
                    }
                    d.Ui[nb + nu] = c;
                    Ux[nb + nu] = dr_value<V>(mrow[b * nown2 + c2]);
                    d.Ubeg[T.lo + c2] = nb;
                    d.Uend[T.lo + c2] = nb + cap;
                    for (int r = 0; r < CN; r++) {
                        *cl.map_shared_rank(ubs + c2, r) = nb;
                        *cl.map_shared_rank(ues + c2, r) = nb + cap;
                    }
                }
            cl.sync();
            if (S.stop) break;
        }
    }
    // no block leaves while another may still write into its shared memory
    cl.sync();
    if (rank == 0 && tx == 0) BK_TREC(d.trace, BK_TR_DENSE, 0, tid, t0);
}

}  // namespace

size_t bk_dense_rows_smem(const bk_task &T, int cluster) { return dr_bytes(T.hi - T.lo, T.lspace, cluster); }

// task_ids: nodes whose rows fit the shared memory of `cluster` blocks
void bk_launch_dense_rows(const bk_dev &d, const int32_t *task_ids, int32_t ntasks, size_t smem, double tau,
                          int pref_mode, int cluster, long long budget, void *stream)
{
    if (ntasks <= 0) return;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaFuncSetAttribute(bk_dense_rows_kernel<double, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, BK_DENSE_SMEM);
        cudaFuncSetAttribute(bk_dense_rows_kernel<float, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, BK_DENSE_SMEM);
        cudaFuncSetAttribute(bk_dense_rows_kernel<double, BK_DENSE_CLUSTER>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, BK_DENSE_SMEM);
        cudaFuncSetAttribute(bk_dense_rows_kernel<float, BK_DENSE_CLUSTER>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, BK_DENSE_SMEM);
    });
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(ntasks * cluster));
    cfg.blockDim = dim3(DR_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto go = [&](auto kernel) { cudaLaunchKernelEx(&cfg, kernel, d, task_ids, tau, pref_mode, budget); };
    if (cluster == 1) {
        if (d.prec) go(bk_dense_rows_kernel<float, 1>);
        else go(bk_dense_rows_kernel<double, 1>);
    } else {
        if (d.prec) go(bk_dense_rows_kernel<float, BK_DENSE_CLUSTER>);
        else go(bk_dense_rows_kernel<double, BK_DENSE_CLUSTER>);
    }
}
