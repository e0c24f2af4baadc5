// kernels_team.cu -- Algorithm 1 on a task without descendants (an ND leaf or a
// BTF block) by a team: one block of threads per task, one warp per column, many
// columns in flight.
//
// Which rows are pivoted at column c is known only when every earlier column has
// chosen its pivot, so the columns decide in order; everything else of a column
// runs ahead of that.  A warp loads its column, applies the steps of all decided
// columns in its reach (lowest first), chooses its pivot tentatively, and then
// only watches the decisions of the columns still before it: a decision that
// takes no row of its pattern leaves its state and its tentative choice as they
// are (one bit test); one that takes a row of the pattern becomes its next step.
// Every update of a column is therefore applied in ascending step order, each
// once, with the operations of the column-by-column form: the factors are the
// same bit for bit.
//
// A column publishes, in shared memory: rec[c], its pivot row, as soon as it is
// chosen (every warp keeps the inverse map of the records it has seen itself, so
// nothing else has to be visible with it); its L column, up to TM_RING entries,
// in its warp's ring buffer, read by the columns that wait for it (a sequence word
// tells a reader that the warp went on to its next column; the reader then takes
// the stored column); and meta[c], where L(:,c) is stored, its length and the
// column's level in the column DAG.
//
// What bounds it: about 72 % of the columns of a netlist or grid leaf depend on
// the column just before them (postordered subtrees), so the time is the task's
// columns times the link from one decision to the next: the flag, the step's
// entries (shared memory), the pivot search, a division; about 4,000 cycles by the
// trace, 4,600 to 5,000 a column, of which an issue every 8 cycles a warp (dependent
// instructions) is the cause, not memory (DRAM 0.02 % of peak).  Measured against one warp walking the
// columns alone, a launch: leaves of 2,499 columns (20,011-row netlist) 5.5 ms, was
// 44; of 4,685 columns (150,001 rows) 11.2 ms, was 87; 4,096 blocks of up to 1,024
// rows 7.3 ms, was 41.
//
// Repair.  After a stored-pattern pass (kernels_static.cu) a team starts at its
// task's first rejected column.  A column stands if none of its steps was computed
// anew and none of its rows was pivoted by another column than before (tested
// against two bitmaps, in the order of the decisions); the others are computed as
// above.  One launch resolves every rejection of every task: on the power grid
// (316 x 316, 10 to 24 rejections a refactorization) 12 ms in place of 22 ms of
// host-driven rounds.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <mutex>

#include "basker_internal.h"
#include "device_util.cuh"

using namespace bk;

namespace {

constexpr int TM_PF = 2;            // entries a lane of the next step's L column read ahead
constexpr int TM_BATCH = 4;         // further entries a lane in flight
constexpr int TM_RING = 32 * TM_PF;         // entries of an L column handed on through shared memory
constexpr int TM_LIST = 1024;       // rows of a column's pattern listed, at most
constexpr uint32_t TM_NONE = 0xffffu;
constexpr unsigned long long TM_PUB = 1ull << 63;

__device__ __forceinline__ void cta_fence() { asm volatile("fence.acq_rel.cta;" ::: "memory"); }

// The steps still to apply to a column: a bitmap with a summary word per 32 words.
struct TeamSteps {
    volatile uint32_t *w, *sum;
    int nsum;
    __device__ __forceinline__ void set(int i)
    {
        const uint32_t old = atomicOr(const_cast<uint32_t *>(w) + (i >> 5), 1u << (i & 31));
        if (old == 0u) atomicOr(const_cast<uint32_t *>(sum) + (i >> 10), 1u << ((i >> 5) & 31));
    }
    __device__ __forceinline__ void clear(int i)             // one lane
    {
        const uint32_t v = w[i >> 5] & ~(1u << (i & 31));
        w[i >> 5] = v;
        if (!v) sum[i >> 10] = sum[i >> 10] & ~(1u << ((i >> 5) & 31));
    }
    __device__ __forceinline__ int lowest(int lane) const    // -1: none (warp-uniform)
    {
        for (int q = 0; q < nsum; q += 32) {
            const uint32_t v = q + lane < nsum ? sum[q + lane] : 0u;
            const uint32_t ball = __ballot_sync(BK_FULL, v != 0u);
            if (ball) {
                const int l = __ffs(ball) - 1;
                const uint32_t sv = __shfl_sync(BK_FULL, v, l);
                const int wd = ((q + l) << 5) + __ffs(sv) - 1;
                return (wd << 5) + __ffs(w[wd]) - 1;
            }
        }
        return -1;
    }
};

// A column's dense vector x keeps its pattern with its values: an entry outside the
// pattern is the word 0, an entry of the pattern is its value's bits XOR a key that
// no value's bits equal (a NaN with a payload that arithmetic does not make; one
// in the input is replaced by the plain NaN when the column is loaded).
template <typename V> struct XWord;
template <> struct XWord<double> {
    typedef unsigned long long U;
    static constexpr U key = 0x7ff8b5a5c3d2e1f0ull, plain_nan = 0x7ff8000000000000ull, exp = 0x7ff0000000000000ull;
    static __device__ __forceinline__ U bits(double v) { return (U)__double_as_longlong(v); }
    static __device__ __forceinline__ double value(U b) { return __longlong_as_double((long long)b); }
};
template <> struct XWord<float> {
    typedef uint32_t U;
    static constexpr U key = 0x7fd5a5c3u, plain_nan = 0x7fc00000u, exp = 0x7f800000u;
    static __device__ __forceinline__ U bits(float v) { return __float_as_uint(v); }
    static __device__ __forceinline__ float value(U b) { return __uint_as_float(b); }
};

// The largest key of the warp by two 32-bit reductions.
__device__ __forceinline__ unsigned long long max_key(unsigned long long k)
{
    const uint32_t hi = (uint32_t)(k >> 32);
    const uint32_t mh = __reduce_max_sync(BK_FULL, hi);
    const uint32_t ml = __reduce_max_sync(BK_FULL, hi == mh ? (uint32_t)k : 0u);
    return ((unsigned long long)mh << 32) | ml;
}

__host__ __device__ inline int team_words(int bits) { return (bits + 31) >> 5; }
__host__ __device__ inline int team_sums(int bits) { return (team_words(bits) + 31) >> 5; }
__host__ __device__ inline int team_list(int lsp) { return lsp < TM_LIST ? (lsp + 3) & ~3 : TM_LIST; }
// shared memory of the team's tables, and of one warp: x (XS), ring values, then
// step and row bitmaps, the list and the ring's slots
__host__ __device__ inline size_t team_tables(int nown)
{
    return (((size_t)((nown + 1) & ~1) * 8 + (size_t)((nown + 7) & ~7) * 4 + (size_t)team_words(nown) * 8) + 15) &
           ~(size_t)15;
}
__host__ __device__ inline size_t team_warp_bytes(int nown, int lsp, size_t xbytes)
{
    const size_t words = team_words(nown) + team_words(lsp) + team_sums(nown);
    return ((xbytes + 7) & ~(size_t)7) + TM_RING * 8 + ((words * 4 + (size_t)team_list(lsp) * 2 + TM_RING * 2 + 7) & ~(size_t)7);
}

template <typename V, bool XS>
__global__ void __launch_bounds__(512, 1) bk_team_kernel(bk_dev d, const int32_t *__restrict__ ids, int ntasks,
                                                         double tau, int pref_mode, long long budget, int repair)
{
    extern __shared__ __align__(16) unsigned char tsm[];
    __shared__ bk_task T;
    __shared__ volatile int s_abort;
    __shared__ volatile int rseq[16];       // per warp: the column its ring holds (-1: none)
    __shared__ volatile int rlev[16];       // and its rows and level
    typedef XWord<V> XW;
    typedef typename XW::U XU;
    const V *const Bx = vals<V>(d.Bx);
    V *const Lx = vals<V>(d.Lx);
    V *const Ux = vals<V>(d.Ux);
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    const int W = blockDim.x >> 5;          // a power of two
    const uint32_t lt = (1u << lane) - 1u;
    XU *const xg = reinterpret_cast<XU *>(d.wsd + (int64_t)(blockIdx.x * W + wid) * d.wsd_slice);

    for (int ti = blockIdx.x; ti < ntasks; ti += gridDim.x) {
        const int tid = ids[ti];
        // a repair starts at the task's first rejected column (none: nothing to do)
        const int f = repair ? d.task_fail[tid] : 0;
        if (repair && f >= d.tasks[tid].hi) continue;
        if (wid == 0) load_task(T, d.tasks + tid, lane);
        if (threadIdx.x == 0) s_abort = 0;
        if (lane == 0) rseq[wid] = -1;
        __syncthreads();
        const int base = T.lo;
        const int nown = T.hi - T.lo;
        const int lsp = T.lspace;
        volatile unsigned long long *const meta = reinterpret_cast<unsigned long long *>(tsm);
        volatile uint16_t *const rec = reinterpret_cast<uint16_t *>(tsm + (size_t)((nown + 1) & ~1) * 8);
        volatile uint16_t *const spinv = rec + ((nown + 7) & ~7);
        // a repair's steps computed anew, and rows pivoted by a column other than before
        volatile uint32_t *const dirty = reinterpret_cast<uint32_t *>(const_cast<uint16_t *>(spinv) + ((nown + 7) & ~7));
        volatile uint32_t *const touched = dirty + team_words(nown);
        const int c0 = repair ? max(f - base, 0) : 0;
        const size_t xbytes = XS ? (size_t)lsp * sizeof(V) : 0;
        const size_t wstride = team_warp_bytes(nown, lsp, xbytes);
        unsigned char *const wb0 = tsm + team_tables(nown);
        unsigned char *const wb = wb0 + (size_t)wid * wstride;
        const size_t roff = (xbytes + 7) & ~(size_t)7;               // ring values
        const int words = team_words(nown) + team_words(lsp) + team_sums(nown);
        const size_t woff = roff + TM_RING * 8;                      // bitmaps
        const size_t loff = woff + (size_t)words * 4;                // list
        const size_t soff = loff + (size_t)team_list(lsp) * 2;       // ring slots
        XU *const x = XS ? reinterpret_cast<XU *>(wb) : xg;
        uint32_t *const bw = reinterpret_cast<uint32_t *>(wb + woff);
        TeamSteps sb;
        sb.w = bw;
        volatile uint32_t *const rb = bw + team_words(nown);
        sb.sum = rb + team_words(lsp);
        sb.nsum = team_sums(nown);
        uint16_t *const list = reinterpret_cast<uint16_t *>(wb + loff);
        const int cap = team_list(lsp);
        const int nrw = team_words(lsp);
        for (int i = threadIdx.x; i < nown; i += blockDim.x) {
            meta[i] = 0ull;
            rec[i] = 0;
            spinv[i] = (uint16_t)TM_NONE;
        }
        for (int i = threadIdx.x; i < 2 * team_words(nown); i += blockDim.x) dirty[i] = 0u;
        for (int i = lane; i < words; i += 32) bw[i] = 0u;
        if (XS)
            for (int i = lane; i < lsp; i += 32) x[i] = 0;
        __syncthreads();

        if (c0 > 0) {
            // the columns before the first rejected one stand
            for (int i = threadIdx.x; i < c0; i += blockDim.x) {
                const int r = d.prow[base + i] - base;
                if ((unsigned)r >= (unsigned)nown) { report_internal(d.status, base + i, 55); continue; }
                rec[i] = (uint16_t)(r + 1);
                spinv[r] = (uint16_t)i;
                meta[i] = TM_PUB | ((unsigned long long)d.Lbeg[base + i] << 32) |
                          ((unsigned long long)d.Lcnt[base + i] << 16) | (unsigned long long)d.level[base + i];
            }
            __syncthreads();
        }
        int seen = c0;         // decisions this warp has taken into spinv
        int pubw = c0;         // columns known to be stored: all below this
        bool stop = false;
        auto abort_team = [&]() {
            if (lane == 0) s_abort = 1;
            stop = true;
        };
        // why: 0 go on waiting, 1 the team gave up, 2 this wait ran out of budget
        auto give_up = [&](int why) -> bool {
            if (why == 0) return true;
            if (why == 2) {
                if (lane == 0) atomicExch(&d.status->timeout, 1);
                abort_team();
            }
            stop = true;
            return false;
        };
        auto xval = [](XU w) { return XW::value(w ^ XW::key); };
        auto nonfinite = [](XU w) { return ((w ^ XW::key) & XW::exp) == XW::exp; };

        // the extents and first entries of the warp's next column, read ahead
        int n_e0 = 0, n_e1 = 0, n_pref = 0, n_r = -1;
        V n_v = V(0);
        auto next_extent = [&](int c) {
            if (c >= nown) return;
            const int gc = base + c;
            n_e0 = d.dstart[gc];
            n_e1 = d.Bp[gc + 1];
            n_pref = (pref_mode ? d.pref[gc] : gc) - base;
        };
        auto next_entries = [&](int c) {
            n_r = -1;
            if (c < nown && n_e0 + lane < n_e1) {
                n_r = d.Bi[n_e0 + lane];
                n_v = Bx[n_e0 + lane];
            }
        };
        const int cw = c0 + ((wid - c0) & (W - 1));      // the warp's first column
        next_extent(cw);
        next_entries(cw);

        for (int c = cw, it = 0; c < nown; c += W, it++) {
            const int gc = base + c;
            if ((it & 15) == 0 && __shfl_sync(BK_FULL, (int)should_stop(d, tid, gc), 0)) { abort_team(); break; }
            const int e0 = n_e0, e1 = n_e1, pref = n_pref;
            const int r_first = n_r;
            const V v_first = n_v;
            next_extent(c + W);
            int64_t ub = d.Ubeg[gc], ue = d.Uend[gc], lb = d.Lbeg[gc], le = d.Lend[gc];
            int cnt = 0;               // rows listed (in the pattern at some time)
            int npend = 0;             // steps still to apply (the bits set in sb)
            auto append = [&](bool isnew, int s) {
                const uint32_t m = __ballot_sync(BK_FULL, isnew);
                const int at = cnt + __popc(m & lt);
                if (isnew && at < cap) list[at] = (uint16_t)s;
                cnt += __popc(m);
            };
            // decisions published before now are known: no row is in the pattern yet
            for (;;) {
                const int k = seen + lane;
                const uint32_t r1 = k < c ? rec[k] : 0u;
                const uint32_t m = __ballot_sync(BK_FULL, r1 != 0u);
                const int n1 = m == BK_FULL ? 32 : __ffs(~m) - 1;
                if (lane < n1) spinv[r1 - 1] = (uint16_t)k;
                seen += n1;
                if (n1 < 32) break;
            }
            __syncwarp();
            const int pr0 = repair ? d.prow[gc] - base : -1;       // the pivot row of before
            if (repair && !d.col_fail[gc]) {
                // the stored column stands unless one of its steps was computed anew
                // or one of its rows was pivoted by an earlier column than before;
                // decisions still to come are tested as they are published
                cta_fence();
                const int us = d.Ucnt[gc] - 1, ls = d.Lcnt[gc];
                auto bit = [](const volatile uint32_t *w, int i) { return (w[i >> 5] >> (i & 31)) & 1u; };
                auto mark = [](const volatile uint32_t *w, int i) {
                    atomicOr(const_cast<uint32_t *>(w) + (i >> 5), 1u << (i & 31));
                };
                bool hit = false;
                for (int q = lane; q < us; q += 32) {
                    const int k = d.Ui[ub + q] - base;
                    if ((unsigned)k >= (unsigned)c) { report_internal(d.status, gc, 56); continue; }
                    if (bit(dirty, k)) hit = true;
                    else if (k >= seen) mark(sb.w, k);
                }
                for (int q = lane; q <= ls; q += 32) {
                    const int sl = q < ls ? d.Ls[lb + q] : pr0;
                    if ((unsigned)sl >= (unsigned)nown) continue;
                    if (bit(touched, sl)) hit = true;
                    mark(rb, sl);
                }
                __syncwarp();
                hit = __any_sync(BK_FULL, hit);
                long long w0 = 0;
                while (!hit && seen < c) {
                    const int k = seen + lane;
                    const uint32_t r1 = k < c ? rec[k] : 0u;
                    const uint32_t m = __ballot_sync(BK_FULL, r1 != 0u);
                    const int n1 = m == BK_FULL ? 32 : __ffs(~m) - 1;
                    if (n1 > 0) {
                        cta_fence();
                        if (lane < n1) {
                            const int r = (int)r1 - 1;
                            spinv[r] = (uint16_t)k;
                            hit = (bit(dirty, k) && bit(sb.w, k)) || (bit(touched, r) && bit(rb, r));
                        }
                        hit = __any_sync(BK_FULL, hit);
                        seen += n1;
                        w0 = 0;
                        __syncwarp();
                    } else {
                        if (w0 == 0) w0 = clock64();
                        const int why = s_abort ? 1 : clock64() - w0 > budget ? 2 : 0;
                        if (!give_up(__shfl_sync(BK_FULL, why, 0))) break;
                        if (c - seen > 2) __nanosleep(40);
                    }
                }
                if (stop) break;
                for (int q = lane; q < us; q += 32) {
                    const int k = d.Ui[ub + q] - base;
                    if ((unsigned)k < (unsigned)c) sb.w[k >> 5] = 0u;
                }
                for (int q = lane; q <= ls; q += 32) {
                    const int sl = q < ls ? d.Ls[lb + q] : pr0;
                    if ((unsigned)sl < (unsigned)nown) rb[sl >> 5] = 0u;
                }
                __syncwarp();
                if (!hit) {
                    if (lane == 0) {
                        meta[c] = TM_PUB | ((unsigned long long)lb << 32) | ((unsigned long long)ls << 16) |
                                  (unsigned long long)d.level[gc];
                        rec[c] = (uint16_t)(pr0 + 1);
                    }
                    next_entries(c + W);
                    continue;
                }
            }
            for (int eb = e0; eb < e1; eb += 32) {
                const int e = eb + lane;
                const int r = eb == e0 ? r_first : e < e1 ? d.Bi[e] : -1;
                const V v = eb == e0 ? v_first : e < e1 ? Bx[e] : V(0);
                const int s = e < e1 ? ((unsigned)(r - base) < (unsigned)nown ? r - base : slot_of(T, base, r)) : -1;
                if (e < e1 && s < 0) report_internal(d.status, gc, 51);
                bool isnew = false;
                if (s >= 0) {
                    const XU vb = XW::bits(v);
                    x[s] = (vb == XW::key ? XW::plain_nan : vb) ^ XW::key;
                    const uint32_t p = s < nown ? spinv[s] : TM_NONE;
                    isnew = p >= (uint32_t)seen;
                    if (!isnew) sb.set((int)p);
                }
                npend += __popc(__ballot_sync(BK_FULL, s >= 0 && !isnew));
                append(isnew, s);
            }
            __syncwarp();
            int nu = 0, nflushed = 0, lev = 0;
            int uj = 0;
            V um = V(0);
            bool bad = false, chosen = false;
            int total = 0, piv = -1;
            int sel_s = 0;                 // cnt <= 32: the lane's row and word at the choice
            XU sel_w = 0;
            auto flush = [&](int m) -> bool {
                if (ub + nflushed + m > ue) {
                    const int64_t ncap = max((long long)grown_ucap(nflushed + m, (int64_t)c + 1),
                                             (long long)(nflushed + m));
                    int64_t nb = 0;
                    if (lane == 0) nb = pool_alloc(d.pool + 1, d.upool_end, ncap);
                    nb = __shfl_sync(BK_FULL, nb, 0);
                    if (nb < 0) {
                        if (lane == 0) report_overflow(d, T, tid, gc, 2);
                        return false;
                    }
                    for (int k = lane; k < nflushed; k += 32) {
                        d.Ui[nb + k] = d.Ui[ub + k];
                        Ux[nb + k] = Ux[ub + k];
                    }
                    __syncwarp();
                    ub = nb;
                    ue = nb + ncap;
                    if (lane == 0) {
                        d.Ubeg[gc] = ub;
                        d.Uend[gc] = ue;
                    }
                }
                if (lane < m) {
                    d.Ui[ub + nflushed + lane] = uj;
                    Ux[ub + nflushed + lane] = um;
                }
                nflushed += m;
                return true;
            };
            // f(slot, word) over the pattern's unpivoted rows (once no step is left
            // to apply), all lanes together (word 0: none)
            auto for_rows = [&](auto &&f) {
                if (cnt <= cap) {
                    for (int i0 = 0; i0 < cnt; i0 += 32) {
                        const int s = i0 + lane < cnt ? list[i0 + lane] : 0;
                        f(s, i0 + lane < cnt ? x[s] : XU(0));
                    }
                } else {
                    for (int i0 = 0; i0 < lsp; i0 += 32) f(i0 + lane, i0 + lane < lsp ? x[i0 + lane] : XU(0));
                }
            };
            auto choose = [&]() {
                const XU wp = pref >= 0 && pref < nown ? x[pref] : XU(0);
                unsigned long long km = 0;
                bool bx = bad;
                if (cnt <= 32) {
                    // one row a lane
                    const int s = lane < cnt ? list[lane] : 0;
                    const XU w = lane < cnt ? x[s] : XU(0);
                    sel_s = s;
                    sel_w = w;
                    bx = bx || (w && nonfinite(w));
                    km = max_key(w && s < nown ? mag_key(xval(w)) : 0ull);
                    total = __popc(__ballot_sync(BK_FULL, w != 0));
                    if (!__any_sync(BK_FULL, bx)) {
                        if (wp && mag_key(xval(wp)) == km && km > 0) {
                            piv = pref;
                        } else if (wp && km > 0 && (double)fabs(xval(wp)) >= tau * (double)key_value<V>(km)) {
                            piv = pref;
                        } else {
                            piv = -1;
                            if (km > 0)
                                piv = (int)__reduce_min_sync(BK_FULL, w && s < nown && mag_key(xval(w)) == km
                                                                          ? (unsigned)s : 0xffffffffu);
                        }
                    } else {
                        piv = -2;
                    }
                    chosen = true;
                    return;
                }
                total = 0;
                for_rows([&](int s, XU w) {
                    if (w && nonfinite(w)) bx = true;
                    if (w && s < nown) km = key_max(km, mag_key(xval(w)));
                    total += __popc(__ballot_sync(BK_FULL, w != 0));
                });
                km = max_key(km);
                const V amax = key_value<V>(km);
                piv = -1;
                if (__any_sync(BK_FULL, bx)) {
                    piv = -2;
                } else if (km > 0) {          // a candidate of nonzero magnitude
                    if (wp && (double)fabs(xval(wp)) >= tau * (double)amax) {
                        piv = pref;
                    } else {
                        unsigned best = 0xffffffffu;
                        for_rows([&](int s, XU w) {
                            if (w && s < nown && mag_key(xval(w)) == km) best = min(best, (unsigned)s);
                        });
                        piv = (int)__reduce_min_sync(BK_FULL, best);
                    }
                }
                chosen = true;
            };

            // the column's steps, lowest first; the next one's entries read ahead
            int jb = npend ? sb.lowest(lane) : -1;
            int pj = -1;                    // the step whose entries are read ahead
            int pr[TM_PF];
            V pv[TM_PF];
            long long t0 = 0;
            while (!stop) {
                if (jb < 0) {
                    // no step left among the decided columns: take in the decisions
                    // published meanwhile; the lowest that pivots a row of the
                    // pattern is the next step
                    if (seen < c) {
                        const int k = seen + lane;
                        const uint32_t r1 = k < c ? rec[k] : 0u;
                        const uint32_t m = __ballot_sync(BK_FULL, r1 != 0u);
                        const int n1 = m == BK_FULL ? 32 : __ffs(~m) - 1;
                        if (n1 > 0) {
                            bool hit = false;
                            if (lane < n1) {
                                const int r = (int)r1 - 1;
                                spinv[r] = (uint16_t)k;
                                hit = x[r] != 0;
                            }
                            const uint32_t hits = __ballot_sync(BK_FULL, hit);
                            if (hits) {
                                if (hit) sb.set(k);
                                chosen = false;
                                npend = __popc(hits);
                                jb = seen + __ffs(hits) - 1;
                                t0 = 0;
                            }
                            seen += n1;
                            __syncwarp();
                            if (hits) continue;
                            if (n1 == 32) continue;
                        }
                    }
                    if (!chosen) {
                        choose();
                        continue;
                    }
                    if (seen == c) break;
                    if (t0 == 0) t0 = clock64();
                    const int why = s_abort ? 1 : clock64() - t0 > budget ? 2 : 0;
                    if (!give_up(__shfl_sync(BK_FULL, why, 0))) break;
                    if (c - seen > 2) __nanosleep(40);
                    continue;
                }
                const int j = jb;
                const int sp = (int)rec[j] - 1;
                if (nu > c || (unsigned)sp >= (unsigned)nown) {
                    if (lane == 0) report_internal(d.status, gc, 54);
                    abort_team();
                    break;
                }
                int ss[TM_PF];
                V ll[TM_PF];
                int jc = 0, jlev = 0;
                int64_t jl = 0;
                bool ring = false;
                if (j >= pubw) {
                    // recent: from the ring of its warp while that holds it, else stored
                    const int wj = j & (W - 1);
                    const long long w0 = clock64();
                    for (;;) {
                        const int why = s_abort ? 1 : clock64() - w0 > budget ? 2 : 0;
                        const int state = __shfl_sync(BK_FULL, why ? 4 + why : rseq[wj] == j ? 1 : meta[j] != 0ull ? 2 : 0, 0);
                        if (state == 0) continue;
                        if (state >= 4) { give_up(state - 4); break; }
                        cta_fence();
                        if (state == 1) {
                            const unsigned char *const wr = wb0 + (size_t)wj * wstride;
                            const volatile V *const rv = reinterpret_cast<const volatile V *>(wr + roff);
                            const volatile uint16_t *const rs = reinterpret_cast<const volatile uint16_t *>(wr + soff);
                            const int rl = rlev[wj];
#pragma unroll
                            for (int u = 0; u < TM_PF; u++) {
                                ss[u] = -1;
                                ll[u] = V(0);
                                if (u == 0 || (rl >> 16) > 32 * u) {
                                    const int s = rs[lane + 32 * u];
                                    ss[u] = s == 0xffff ? -1 : s;
                                    ll[u] = rv[lane + 32 * u];
                                }
                            }
                            jlev = rl & 0xffff;
                            __syncwarp();
                            cta_fence();
                            if (__any_sync(BK_FULL, rseq[wj] != j)) continue;     // overwritten meanwhile
                            ring = true;
                        }
                        break;
                    }
                    if (stop) break;
                    if (!ring) {
                        for (;;) {
                            const int k = pubw + lane;
                            const uint32_t m = __ballot_sync(BK_FULL, k < seen && meta[k] != 0ull);
                            const int n1 = m == BK_FULL ? 32 : __ffs(~m) - 1;
                            pubw += n1;
                            if (n1 < 32) break;
                        }
                        cta_fence();
                        __syncwarp();
                    }
                }
                if (!ring) {
                    const unsigned long long mt = meta[j];
                    jl = (int64_t)((mt & ~TM_PUB) >> 32);
                    jc = (int)(mt >> 16) & 0xffff;
                    jlev = (int)(mt & 0xffffull);
                    if (pj != j) {
#pragma unroll
                        for (int u = 0; u < TM_PF; u++) {
                            const int q = lane + 32 * u;
                            pr[u] = q < jc ? d.Ls[jl + q] : -1;
                            pv[u] = q < jc ? Lx[jl + q] : V(0);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < TM_PF; u++) {
                        ss[u] = pr[u];
                        ll[u] = pv[u];
                    }
                }
                // what the first entries need, read together
                const XU mw = x[sp];
                XU xw[TM_PF];
                uint32_t sv[TM_PF];
#pragma unroll
                for (int u = 0; u < TM_PF; u++) {
                    xw[u] = ss[u] >= 0 ? x[ss[u]] : XU(0);
                    sv[u] = (unsigned)ss[u] < (unsigned)nown ? spinv[ss[u]] : TM_NONE;
                }
                if (lane == 0) sb.clear(j);
                npend--;
                __syncwarp();
                if (lane == 0) x[sp] = 0;
                // the next step as known now: its first entries
                const int jn = npend ? sb.lowest(lane) : -1;
                int nr[TM_PF];
                V nv[TM_PF];
                const bool ahead = jn >= 0 && jn < pubw;
                if (ahead) {
                    const unsigned long long mn = meta[jn];
                    const int64_t nl = (int64_t)((mn & ~TM_PUB) >> 32);
                    const int nc = (int)(mn >> 16) & 0xffff;
#pragma unroll
                    for (int u = 0; u < TM_PF; u++) {
                        const int q = lane + 32 * u;
                        nr[u] = q < nc ? d.Ls[nl + q] : -1;
                        nv[u] = q < nc ? Lx[nl + q] : V(0);
                    }
                }
                const V m = xval(mw);
                if (nonfinite(mw)) bad = true;
                if ((nu & 31) == lane) {
                    uj = base + j;
                    um = m;
                }
                nu++;
                lev = max(lev, jlev + 1);
                unsigned newmin = 0xffffffffu;       // the lowest step the updates add
                int nadd = 0;
                // entry of slot s (word w, known decision sv): x -= l m; a new row of
                // the pattern is listed, or is a step
                auto apply = [&](int s, V l, XU w, uint32_t p) {
                    bool isnew = false, isstep = false;
                    if (s >= 0) {
                        x[s] = XW::bits(fma(-l, m, w ? xval(w) : V(0))) ^ XW::key;
                        if (!w) {
                            isnew = p >= (uint32_t)seen;
                            isstep = !isnew;
                            if (isstep) {
                                if ((int)p <= j) report_internal(d.status, gc, 53);
                                sb.set((int)p);
                                newmin = min(newmin, p);
                            }
                        }
                    }
                    nadd += __popc(__ballot_sync(BK_FULL, isstep));
                    append(isnew, s);
                };
#pragma unroll
                for (int u = 0; u < TM_PF; u++)
                    if (u == 0 || __any_sync(BK_FULL, ss[u] >= 0)) apply(ss[u], ll[u], xw[u], sv[u]);
                for (int q0 = 32 * TM_PF; q0 < jc; q0 += 32 * TM_BATCH) {
                    int sr[TM_BATCH];
                    V lr[TM_BATCH];
                    XU xr[TM_BATCH];
                    uint32_t vr[TM_BATCH];
#pragma unroll
                    for (int u = 0; u < TM_BATCH; u++) {
                        const int q = q0 + lane + 32 * u;
                        sr[u] = q < jc ? d.Ls[jl + q] : -1;
                        lr[u] = q < jc ? Lx[jl + q] : V(0);
                    }
#pragma unroll
                    for (int u = 0; u < TM_BATCH; u++) {
                        xr[u] = sr[u] >= 0 ? x[sr[u]] : XU(0);
                        vr[u] = (unsigned)sr[u] < (unsigned)nown ? spinv[sr[u]] : TM_NONE;
                    }
#pragma unroll
                    for (int u = 0; u < TM_BATCH; u++) apply(sr[u], lr[u], xr[u], vr[u]);
                }
                if ((nu & 31) == 0 && !flush(32)) { abort_team(); break; }
                if (nadd) newmin = __reduce_min_sync(BK_FULL, newmin);
                npend += nadd;
                __syncwarp();
                jb = newmin < (unsigned)(jn < 0 ? INT_MAX : jn) ? (int)newmin : jn;
                pj = -1;
                if (ahead && jb == jn) {
                    pj = jn;
#pragma unroll
                    for (int u = 0; u < TM_PF; u++) {
                        pr[u] = nr[u];
                        pv[u] = nv[u];
                    }
                }
            }
            if (!stop && piv < 0) {
                if (lane == 0) report_fail(d.status, gc, piv == -2 ? BK_CODE_NAN : BK_CODE_SINGULAR);
                abort_team();
            }
            if (stop) break;
            // the decision
            if (lane == 0) {
                if (repair) {
                    atomicOr(const_cast<uint32_t *>(dirty) + (c >> 5), 1u << (c & 31));
                    if (piv != pr0) atomicOr(const_cast<uint32_t *>(touched) + (piv >> 5), 1u << (piv & 31));
                    cta_fence();
                }
                rec[c] = (uint16_t)(piv + 1);
            }
            const V xp = xval(x[piv]);
            const int lcnt = total - 1;
            // the L column of a short pattern: values in registers and, for the
            // columns that wait for it, in the ring
            const bool thin = cnt <= TM_RING;
            int es[TM_PF];
            V el[TM_PF];
            if (thin) {
                V *const rv = reinterpret_cast<V *>(wb + roff);
                uint16_t *const rs = reinterpret_cast<uint16_t *>(wb + soff);
                if (lane == 0) rseq[wid] = -1;
#pragma unroll
                for (int u = 0; u < TM_PF; u++) es[u] = -1;
                if (cnt <= 32) {
                    if (sel_s == piv) sel_w = 0;
                    es[0] = sel_w ? sel_s : -1;
                    el[0] = sel_w ? xval(sel_w) / xp : V(0);
                } else {
#pragma unroll
                    for (int u = 0; u < TM_PF; u++) {
                        const int i = lane + 32 * u;
                        const int s = i < cnt ? list[i] : piv;
                        const XU w = s != piv ? x[s] : XU(0);
                        es[u] = w ? s : -1;
                        el[u] = w ? xval(w) / xp : V(0);
                    }
                }
                cta_fence();
                __syncwarp();
#pragma unroll
                for (int u = 0; u < TM_PF; u++) {
                    if (u > 0 && cnt <= 32 * u) break;
                    rs[lane + 32 * u] = (uint16_t)(es[u] < 0 ? 0xffff : es[u]);
                    rv[lane + 32 * u] = el[u];
                }
                if (lane == 0) rlev[wid] = (cnt << 16) | lev;
                __syncwarp();
                cta_fence();
                if (lane == 0) rseq[wid] = c;
            }
            next_entries(c + W);
            if ((nu & 31) == lane) {
                uj = gc;
                um = xp;
            }
            nu++;
            bool ok = flush(nu - nflushed);
            if (ok && lb + lcnt > le) {
                const int64_t ncap = min((long long)(2 * (int64_t)lcnt + 16),
                                         (long long)((nown - c - 1) + (lsp - nown)));
                int64_t nb = 0;
                if (lane == 0) nb = pool_alloc(d.pool, d.lpool_end, ncap);
                nb = __shfl_sync(BK_FULL, nb, 0);
                if (nb < 0) {
                    if (lane == 0) report_overflow(d, T, tid, gc, 1);
                    ok = false;
                } else {
                    lb = nb;
                    if (lane == 0) {
                        d.Lbeg[gc] = lb;
                        d.Lend[gc] = nb + ncap;
                    }
                }
            }
            if (!ok) {
                abort_team();
                break;
            }
            // L(:,c) = x / pivot over the pattern's rows in ascending order
            if (thin) {
                int rk[TM_PF];
#pragma unroll
                for (int u = 0; u < TM_PF; u++) rk[u] = 0;
                for (int i0 = 0; i0 < cnt; i0 += 32) {
                    const unsigned so = (unsigned)(i0 == 0 ? es[0] : es[1]);
#pragma unroll 8
                    for (int t = 0; t < 32; t++) {
                        const unsigned o = __shfl_sync(BK_FULL, so, t);
#pragma unroll
                        for (int u = 0; u < TM_PF; u++) rk[u] += o < (unsigned)es[u];
                    }
                }
#pragma unroll
                for (int u = 0; u < TM_PF; u++)
                    if (es[u] >= 0) {
                        const int s = es[u];
                        d.Li[lb + rk[u]] = s < nown ? base + s : row_of_lslot(T, s);
                        Lx[lb + rk[u]] = el[u];
                        d.Ls[lb + rk[u]] = s;
                        x[s] = 0;
                    }
                if (lane == 0) x[piv] = 0;
            } else {
                // the pattern as a bitmap, 32 words of it at a time listed in ascending order
                for_rows([&](int s, XU w) {
                    if (w) atomicOr(const_cast<uint32_t *>(rb) + (s >> 5), 1u << (s & 31));
                });
                __syncwarp();
                int done = 0;
                for (int w0 = 0; w0 < nrw; w0 += 32) {
                    const int w = w0 + lane;
                    uint32_t bits = w < nrw ? rb[w] : 0u;
                    if (bits) rb[w] = 0u;
                    const int n1 = __popc(bits);
                    const int pre = warp_exscan(n1, lane);
                    const int tot = __shfl_sync(BK_FULL, pre + n1, 31);
                    if (tot == 0) continue;
                    int o = pre;
                    while (bits) {
                        const int b = __ffs(bits) - 1;
                        bits &= bits - 1;
                        list[o++] = (uint16_t)((w << 5) + b);
                    }
                    __syncwarp();
                    for (int i = lane; i < tot; i += 32) {
                        const int s = list[i];
                        if (s != piv) {
                            const int64_t q = lb + done + i - (s > piv ? 1 : 0);
                            d.Li[q] = s < nown ? base + s : row_of_lslot(T, s);
                            Lx[q] = xval(x[s]) / xp;
                            d.Ls[q] = s;
                        }
                        x[s] = 0;
                    }
                    done += tot;
                    __syncwarp();
                }
            }
            if (lane == 0) {
                d.pinv[base + piv] = gc;
                d.prow[gc] = base + piv;
                d.Lcnt[gc] = lcnt;
                d.Ucnt[gc] = nu;
                d.level[gc] = lev;
                if (piv != c) atomicAdd(&d.status->offdiag, 1);
                if (repair || piv != pref) atomicAdd(&d.status->repaired, 1);
            }
            __syncwarp();
            if (lane == 0) {
                cta_fence();
                meta[c] = TM_PUB | ((unsigned long long)lb << 32) | ((unsigned long long)lcnt << 16) |
                          (unsigned long long)lev;
            }
            __syncwarp();
        }
        if (stop && !XS)       // leave x clean: the next task's columns start from zero
            for (int i = lane; i < lsp; i += 32) x[i] = 0;
        __syncwarp();
        __syncthreads();
    }
}

template <typename V, bool XS>
void team_launch(const bk_dev &d, const bk_team_group &g, double tau, int pref_mode, long long budget, int repair,
                 cudaStream_t s)
{
    static std::once_flag once;
    std::call_once(once, [] {
        cudaFuncSetAttribute(bk_team_kernel<V, XS>, cudaFuncAttributeMaxDynamicSharedMemorySize, BK_TEAM_SMEM);
    });
    bk_team_kernel<V, XS><<<g.blocks, g.W * 32, g.smem, s>>>(d, g.ids, g.ntasks, tau, pref_mode, budget, repair);
}

}  // namespace

size_t bk_team_smem(const bk_task &T, int W, bool xs)
{
    const int nown = T.hi - T.lo;
    return team_tables(nown) + (size_t)W * team_warp_bytes(nown, T.lspace, xs ? (size_t)T.lspace * 8 : 0);
}

void bk_launch_team(const bk_dev &d, const bk_team_group &g, double tau, int pref_mode, long long budget,
                    bool repair, void *stream)
{
    cudaStream_t s = (cudaStream_t)stream;
    if (g.ntasks <= 0) return;
    if (d.prec) {
        if (g.xs) team_launch<float, true>(d, g, tau, pref_mode, budget, repair ? 1 : 0, s);
        else team_launch<float, false>(d, g, tau, pref_mode, budget, repair ? 1 : 0, s);
    } else {
        if (g.xs) team_launch<double, true>(d, g, tau, pref_mode, budget, repair ? 1 : 0, s);
        else team_launch<double, false>(d, g, tau, pref_mode, budget, repair ? 1 : 0, s);
    }
}
