// kernels_tsolve.cu -- the solve of BTF blocks and ND leaves, a job per block of
// threads.
//
// A job is a run of steps [lo, hi): an ND leaf's forward or backward rows, a BTF
// block, or a run of small BTF blocks (forward and backward).  Its rows are taken
// in order by the warps of one block; a row's terms come from the job's own values
// in shared memory or, for the coupling to other jobs and for the ND separators,
// from global memory.  A value that is not final yet is a word of ones (a NaN that
// arithmetic does not make; a result with these bits is stored as the plain NaN),
// so a reader polls the value itself: no flag, no fence, one access a link.
// Every row's terms are applied one fma each in the order of the column sweeps
// (ascending steps for L, descending for U, coupling first), so results do not
// depend on the schedule.
//
// Several right-hand sides: one lane each; a term's coefficient is read once for
// all of them.
//
// What bounds it: the chains of dependent rows (a link is a poll in shared memory,
// about 190 cycles, the term's fma, a division for U, the store: 400 cycles forward
// and 1,000 backward).  As a row dataflow over the whole GPU with flags in global
// memory a link was about 1.5 us.  A solve of the 2,000-row circuit 0.79 ms, was
// 1.71; of the 20,011-row netlist 1.2 ms, was 2.8; of 150,001 rows 2.5 ms, was 6.0.
// Consecutive items on one warp, in place of one on each: 1.08 ms for the circuit.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <mutex>

#include "basker_internal.h"
#include "device_util.cuh"
#include "solve_internal.h"
#include "solve_word.cuh"

using namespace bk;

namespace {

constexpr int TS_NT = 512;

// Every lane walks its own rows: gs lanes a row (a power of two, the right-hand
// sides rounded up), the block's lane groups taking the job's items in turn.  Each
// pass of the loop, a lane whose next term has its value applies it; lanes of one
// warp can wait for each other (nothing in the loop blocks).  A warp instruction of
// the FP64 pipe costs the same for one lane as for 32 (about 19 cycles), which is
// why a lane, not a warp, has a row.  w and z hold row i's values at [i * R, (i + 1)
// * R).
template <typename V>
__global__ void __launch_bounds__(TS_NT, 1) bk_tsolve_kernel(bk_dev d, bk_solve_dev s, const bk_sjob *__restrict__ jobs,
                                                             int njobs, int32_t *counter, int R, int gs,
                                                             const double *__restrict__ b, int32_t ldb, double *x,
                                                             int32_t ldx, long long budget, int permute)
{
    typedef SvWord<V> SW;
    typedef typename SW::U U;
    extern __shared__ __align__(16) unsigned char tsm[];
    __shared__ int s_job;
    const V *const Bx = vals<V>(d.Bx);
    U *const gw = reinterpret_cast<U *>(vals<V>(s.w));
    U *const gz = reinterpret_cast<U *>(vals<V>(s.z));
    const int q = min((int)threadIdx.x & (gs - 1), R - 1);
    const bool writer = ((int)threadIdx.x & (gs - 1)) < R;
    const int ngrp = blockDim.x / gs;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_job = atomicAdd(counter, 1);
        __syncthreads();
        const int jb = s_job;
        if (jb >= njobs) return;
        const bk_sjob J = jobs[jb];
        const int m = J.hi - J.lo;
        volatile U *const xw = reinterpret_cast<volatile U *>(tsm);          // forward results
        volatile U *const xz = J.mode == 2 ? xw + (size_t)m * R : xw;        // solution
        for (int i = threadIdx.x; i < m * R * (J.mode == 2 ? 2 : 1); i += blockDim.x) xw[i] = SW::none;
        __syncthreads();
        // consecutive items go to different warps: a warp that has just finished one
        // is not the one the next waits for
        int p = J.i0 + (int)(threadIdx.x >> 5) + ((int)(threadIdx.x & 31) / gs) * (int)(blockDim.x >> 5);
        // a row: its item (i forward, ~i backward), its terms [t, len) (t < 0:
        // coupling forward, the forward result backward), the next two terms'
        // columns and coefficients.  The lane's next row is read while it works on
        // one, so that taking it waits for nothing.
        struct Row {
            int it, len, t, c1, out, k, k2;
            int64_t e0;
            V a, a2, z, dg;
        };
        Row c, nx;
        int4 h = make_int4(0, 0, 0, 0);      // the record of the row after the next
        int64_t he = 0;
        auto term = [&](const Row &r, int u, int &kk, V &aa) {
            const bool fw = r.it >= 0;
            if (u >= 0) {
                kk = (fw ? s.r.Lrk : s.r.Urk)[r.e0 + u];
                aa = vals<V>(fw ? s.r.Lrx : s.r.Urx)[r.e0 + u];
            } else if (fw) {
                kk = s.offj[r.c1 + u];
                aa = Bx[s.offpos[r.c1 + u]];
            } else {
                kk = ~r.it;
            }
        };
        // the row's entries toward L1: its first 32 when it is read, then 16 further on
        auto fetch = [&](const Row &r, int u) {
            if (u >= r.len) return;
            const int64_t e = r.e0 + u;
            const bool fw = r.it >= 0;
            asm volatile("prefetch.global.L1 [%0];" ::"l"((fw ? s.r.Lrk : s.r.Urk) + e));
            asm volatile("prefetch.global.L1 [%0];" ::"l"(vals<V>(fw ? s.r.Lrx : s.r.Urx) + e));
        };
        auto record = [&]() {
            if (p < J.i1) {
                h = s.trec[p];
                he = s.tent[p];
            } else {
                h.y = -1;
            }
            p += ngrp;
        };
        auto read_next = [&]() {
            nx.len = h.y;
            if (h.y < 0) return;
            nx.it = h.x;
            nx.e0 = he;
            nx.t = 0;
            nx.out = permute ? h.w : (h.x >= 0 ? h.z : ~h.x);
            if (h.x >= 0) {
                nx.z = (V)b[(int64_t)q * ldb + nx.out];
                if (s.coupling) {
                    nx.c1 = s.offp[h.z + 1];
                    nx.t = s.offp[h.z] - nx.c1;
                }
            } else {
                nx.dg = vals<V>(s.r.Ud)[~h.x];
                if (J.mode == 2) nx.t = -1;
                else nx.z = SW::value(SW::load(gw + (int64_t)(~h.x) * R + q));
            }
            fetch(nx, 0);
            fetch(nx, 8);
            fetch(nx, 24);
            record();
            nx.k = nx.k2 = 0;
            nx.a = nx.a2 = V(0);
            if (nx.t < nx.len) term(nx, nx.t, nx.k, nx.a);
            if (nx.t + 1 < nx.len) term(nx, nx.t + 1, nx.k2, nx.a2);
        };
        nx.it = nx.len = nx.t = nx.c1 = nx.out = nx.k = nx.k2 = 0;
        nx.e0 = 0;
        nx.a = nx.a2 = nx.z = V(0);
        nx.dg = V(1);
        record();
        read_next();
        c = nx;
        read_next();
        bool ok = true;
        int idle = 0;
        long long t0 = 0;
        // where the lane's next value appears: in shared memory (s_at) or global (g_at)
        const volatile U *s_at = xw;
        const U *g_at = nullptr;
        auto aim = [&]() {
            if (c.len < 0 || c.t >= c.len) return;
            const bool use_w = (c.it >= 0) == (c.t >= 0);
            const int jl = c.k - J.lo;
            if ((unsigned)jl < (unsigned)m) {
                s_at = (use_w ? xw : xz) + jl * R + q;
                g_at = nullptr;
            } else {
                g_at = (use_w ? gw : gz) + (int64_t)c.k * R + q;
            }
        };
        aim();
        bool live = __any_sync(BK_FULL, c.len >= 0);
        while (live) {
            // until some lane can move: its value is there, or its terms are done
            U v = 0;
            bool go;
            for (;;) {
                const bool want = c.len >= 0 && c.t < c.len;
                if (want) v = g_at ? SW::load(g_at) : *s_at;
                go = c.len >= 0 && (!want || v != SW::none);
                if (__any_sync(BK_FULL, go)) break;
                if ((++idle & 255) == 0) {
                    if (idle == 256) t0 = clock64();
                    const int why = clock64() - t0 > budget || *reinterpret_cast<const volatile int *>(&d.status->timeout);
                    if (__shfl_sync(BK_FULL, why, 0)) {
                        if ((threadIdx.x & 31) == 0) atomicExch(&d.status->timeout, 1);
                        ok = false;
                        break;
                    }
                }
            }
            if (!ok) break;
            idle = 0;
            const bool last = go && c.t + 1 >= c.len;          // the row is done after this term
            if (go && c.t < c.len) c.z = c.it < 0 && c.t < 0 ? SW::value(v) : fma(-c.a, SW::value(v), c.z);
            if (last) {
                const bool fwd = c.it >= 0;
                const int i = fwd ? c.it : ~c.it;
                if (!fwd) c.z = c.z / c.dg;
                U zb = SW::bits(c.z);
                if (zb == SW::none) zb = SW::plain_nan;
                if (writer) {
                    (fwd ? xw : xz)[(i - J.lo) * R + q] = zb;
                    const int64_t g = (int64_t)i * R + q;
                    if (fwd) {
                        if (J.mode == 0) gw[g] = zb;
                    } else {
                        SW::store(gz + g, zb);
                        x[(int64_t)q * ldx + c.out] = (double)c.z;
                    }
                }
                c = nx;
                read_next();
            } else if (go) {
                c.t++;
                c.k = c.k2;
                c.a = c.a2;
                if (c.t + 1 < c.len) term(c, c.t + 1, c.k2, c.a2);
                if ((c.t & 7) == 0) fetch(c, c.t + 32);
            }
            if (go) aim();
            if (__any_sync(BK_FULL, last)) live = __any_sync(BK_FULL, c.len >= 0);
        }
        if (__syncthreads_or(!ok)) return;
    }
}

// The items' records, in their order: (row forward / ~row backward, terms, row of B
// or -1, place in b or x) and the first term.
__global__ void bk_trec_kernel(bk_dev d, bk_solve_dev s, int nitems)
{
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < nitems; p += gridDim.x * blockDim.x) {
        const int it = s.titems[p];
        const bool fwd = it >= 0;
        const int i = fwd ? it : ~it;
        const int64_t *const rp = fwd ? s.r.Lrp : s.r.Urp;
        const int64_t e0 = rp[i];
        const int r = fwd ? d.prow[i] : -1;
        s.trec[p] = make_int4(it, (int)(rp[i + 1] - e0), r, fwd ? d.P[r] : d.Q[i]);
        s.tent[p] = e0;
    }
}

// An ND leaf's rows in order of its columns' levels in the factorization: rows of
// a level wait for no other row of it.  Backward (decreasing level) that holds by
// construction; forward when every L(i,k) != 0 has level(k) < level(i) (checked; a
// leaf where it fails keeps its step order).  One block a leaf; counts in smem when
// the leaf's rows fit (lvl at least the leaf's rows), else in global memory.
__global__ void __launch_bounds__(1024) bk_torder_kernel(bk_dev d, bk_solve_dev s, int smem_rows)
{
    extern __shared__ int32_t cnt_s[];
    __shared__ int wt[33];
    const bk_task &T = d.tasks[s.leaf_tasks[blockIdx.x]];
    const int lo = T.lo, m = T.hi - T.lo;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (m <= 0) return;
    int32_t *const cnt = m <= smem_rows ? cnt_s : s.tcnt + lo;
    for (int i = tid; i < m; i += blockDim.x) cnt[i] = 0;
    int bad = 0;
    for (int i = lo + wid; i < T.hi; i += blockDim.x >> 5) {
        const int li = d.level[i];
        for (int64_t e = s.r.Lrp[i] + lane; e < s.r.Lrp[i + 1]; e += 32)
            if (d.level[s.r.Lrk[e]] >= li) bad = 1;
    }
    bad = __syncthreads_or(bad);
    for (int i = tid; i < m; i += blockDim.x) atomicAdd(cnt + min(max(d.level[lo + i], 0), m - 1), 1);
    __syncthreads();
    int carry = 0;
    for (int b0 = 0; b0 < m; b0 += blockDim.x) {
        const int i = b0 + tid;
        const int v = i < m ? cnt[i] : 0;
        int inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(BK_FULL, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) wt[wid] = inc;
        __syncthreads();
        if (wid == 0) {
            const int t = lane < (int)(blockDim.x >> 5) ? wt[lane] : 0;
            int ti = t;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(BK_FULL, ti, o);
                if (lane >= o) ti += y;
            }
            wt[lane] = ti - t;
            if (lane == 31) wt[32] = ti;
        }
        __syncthreads();
        if (i < m) cnt[i] = carry + inc - v + wt[wid];
        carry += wt[32];
        __syncthreads();
    }
    int32_t *const fo = s.titems + s.tf0 + (lo - s.tnd0), *const bo = s.titems + s.tb0 + (lo - s.tnd0);
    for (int i = tid; i < m; i += blockDim.x) {
        const int at = atomicAdd(cnt + min(max(d.level[lo + i], 0), m - 1), 1);
        fo[bad ? i : at] = lo + i;
        bo[m - 1 - at] = ~(lo + i);
    }
}

}  // namespace

namespace {

template <typename V>
void tsolve_launch(const bk_dev &d, const bk_solve_dev &s, const bk_sjob *jobs, int njobs, int32_t *counter, int R,
                   const double *b, int32_t ldb, double *x, int32_t ldx, long long budget, bool permute,
                   cudaStream_t st)
{
    static std::once_flag once;
    std::call_once(once, [] {
        cudaFuncSetAttribute(bk_tsolve_kernel<V>, cudaFuncAttributeMaxDynamicSharedMemorySize, BK_TSOLVE_SMEM);
    });
    const size_t smem = (size_t)s.tmax * (size_t)R * sizeof(V);
    int gs = 1;
    while (gs < R) gs *= 2;
    // 16 warps a job while the jobs have an SM each, else 8 (three blocks an SM)
    const int nt = njobs <= 152 ? TS_NT : TS_NT / 2;
    bk_tsolve_kernel<V><<<std::min(njobs, 152 * 4), nt, smem, st>>>(d, s, jobs, njobs, counter, R, gs, b, ldb, x, ldx,
                                                                       budget, permute ? 1 : 0);
}

}  // namespace

void bk_launch_tsolve(const bk_dev &d, const bk_solve_dev &s, const bk_sjob *jobs, int32_t njobs, int32_t *counter,
                      int32_t R, const double *b, int32_t ldb, double *x, int32_t ldx, long long budget,
                      bool permute, void *stream)
{
    if (njobs <= 0) return;
    cudaStream_t st = (cudaStream_t)stream;
    if (d.prec) tsolve_launch<float>(d, s, jobs, njobs, counter, R, b, ldb, x, ldx, budget, permute, st);
    else tsolve_launch<double>(d, s, jobs, njobs, counter, R, b, ldb, x, ldx, budget, permute, st);
}

void bk_launch_torder(const bk_dev &d, const bk_solve_dev &s, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    if (s.nleaves > 0) {
        constexpr int rows = 11 * 1024;          // 44 KB of counts
        bk_torder_kernel<<<s.nleaves, 1024, (size_t)std::min(rows, s.leaf_maxrows) * 4, st>>>(d, s, rows);
    }
    if (s.ntitems > 0)
        bk_trec_kernel<<<std::min((s.ntitems + 255) / 256, 152 * 8), 256, 0, st>>>(d, s, s.ntitems);
}
