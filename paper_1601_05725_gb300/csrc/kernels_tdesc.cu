// kernels_tdesc.cu -- the reach of a separator's column over its descendants, a
// block of warps per column, the descendant nodes in parallel (Algorithm 4's solves
// with the descendants' L and the reductions into A-hat).
//
// A step of node N changes rows of N and of N's ancestors only.  So the nodes of
// one tree level run at once, a warp each: the node's pending steps, lowest first,
// applied to its own rows; what a step adds to rows above the node (the tail of its
// L column) goes to the node's log, in order, as (slot, l, m).  Before a node above
// the leaves starts its steps, and at the end for the separator's and its
// ancestors' rows, the logs of its descendants are applied to its rows, in
// postorder: every entry receives its updates one fma each in ascending step order,
// as in the column's own sweep (bk_gp_desc_kernel), with the same result bit for
// bit.  Log entries are taken 32 at a time; those that meet in a row follow one
// another by their place.
//
// A column whose log outgrows its room is listed for bk_gp_desc_kernel.
//
// In stages, where a separator has separators below it: its columns' steps in the leaves
// need the leaves alone.  So the first launch takes every separator column of the block
// through its leaves (level 1's columns whole) and keeps its vector, bitmaps and logs;
// each later level's launch goes on from there when the separators below are factored.
// One wave of leaf steps then takes the place of one a level, nearly all of a netlist
// column's steps being in one leaf.  (A problem whose regions would take more than 1 GB,
// or with one level of separators, takes the columns of a level whole, if at all.)
//
// What bounds it: a step's chain of dependent instructions and reads (about 2,500
// cycles; 3,000 in one warp alone), so the steps of the node that has most, and the
// walk over the logs.  Measured, the descendant phase of a factorization: 150,001-row
// netlist, 32 leaves, 7.6 ms one warp a column and level by level, 3.4 in stages (2.0 for
// the leaves); 20,011 rows, 8 leaves, 2.2 and 1.15; 100,003-row circuit with supply
// rails of up to 22,600 steps 37 (one warp), 14.6 (columns of a level whole, rails only),
// 12.8 in stages.  With columns of fewer than 128 symbolic steps above level 1 the stages'
// own work shows: 2,000-row circuit, 4 leaves, 0.10 ms a level in one warp, 0.16 here.
// 1,024 threads a block spill registers and put one block on an SM: 3.4 ms for the leaves.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <mutex>

#include "basker_internal.h"
#include "device_util.cuh"

using namespace bk;

namespace {

constexpr int TD_NT = 512;
constexpr int TD_W = TD_NT / 32;
constexpr int TD_CK = 64;              // entries of a log chunk

// The column's dense vector x is 0 outside its pattern, the bitmap pr (by slot).  sb: steps to apply, ap: steps applied (by
// step, both from the space's first row on).
template <typename V>
__global__ void __launch_bounds__(TD_NT) bk_tdesc_kernel(bk_dev d, const int32_t *__restrict__ cols, int32_t ncols,
                                                         int32_t *counter, const int32_t *__restrict__ ncols_dev,
                                                         int32_t *over, int32_t *nover, bk_tdesc_dev lg, int stage,
                                                         int first)
{
    if (ncols_dev) ncols = *ncols_dev;
    extern __shared__ __align__(16) uint32_t td_sm[];
    __shared__ bk_task T;
    __shared__ int s_col, s_chunks, s_wsum[TD_W];
    __shared__ volatile int s_bad, s_over;
    const V *const Bx = vals<V>(d.Bx);
    const V *const Lx = vals<V>(d.Lx);
    V *const Ux = vals<V>(d.Ux);
    V *const Ahat = vals<V>(d.ahat);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    // per descendant node two logs: to descendant rows (2 D), and to the separator's
    // and its ancestors' (2 D + 1): first chunk and entries
    int32_t *const nfirst = reinterpret_cast<int32_t *>(td_sm);
    int32_t *const ncnt = nfirst + 2 * lg.nodes;
    uint16_t *const next = reinterpret_cast<uint16_t *>(ncnt + 2 * lg.nodes);
    volatile uint32_t *const sb = td_sm + 4 * lg.nodes + ((lg.cap / TD_CK + 1) >> 1);
    for (;;) {
        __syncthreads();
        if (tid == 0) {
            s_col = atomicAdd(counter, 1);
            s_chunks = s_bad = s_over = 0;
        }
        __syncthreads();
        if (s_col >= ncols) return;
        const int ord = stage == 1 ? ncols - 1 - s_col : first + s_col;
        const int c = cols[stage == 1 ? ord : s_col];
        const int64_t lg0 = stage ? lg.loff[ord] : (int64_t)blockIdx.x * lg.cap;
        const int nchunks = (stage ? (int)(lg.loff[ord + 1] - lg0) : lg.cap) / TD_CK;
        int32_t *const log_s = lg.slot + lg0;
        V *const log_l = vals<V>(lg.l) + lg0;
        V *const log_m = vals<V>(lg.m) + lg0;
        V *const x = stage ? vals<V>(lg.x) + lg.xoff[ord] : reinterpret_cast<V *>(d.wsd + (int64_t)blockIdx.x * d.wsd_slice);
        uint32_t *const keep = lg.state + (int64_t)ord * lg.words;
        const int task = d.col_task[c];
        if (wid == 0) load_task(T, d.tasks + task, lane);
        __syncthreads();
        const bool quit = __syncthreads_or(tid == 0 && should_stop(d, task, c));
        if (quit && stage < 2) continue;
        const bool part = stage == 1 && T.level > 1;      // the leaves only, for stage 2
        const int base = T.sp_lo;
        const int ndesc = T.lo - base;
        const int lsp = T.lspace;
        const int nsw = (ndesc + 31) >> 5, npw = (ndesc + lsp + 31) >> 5;
        volatile uint32_t *const ap = sb + nsw;
        volatile uint32_t *const pr = ap + nsw;
        const int t0 = d.col_task[base];               // the descendants: tasks [t0, task)
        const int nn = task - t0;
        const int words = (int)(sb - td_sm) + 2 * nsw + npw;
        if (stage < 2) {
            for (int i = tid; i < 2 * nsw + npw; i += TD_NT) sb[i] = 0u;
            for (int i = tid; i < 2 * nn; i += TD_NT) {
                nfirst[i] = -1;
                ncnt[i] = 0;
            }
        } else {
            for (int i = tid; i < words; i += TD_NT) td_sm[i] = keep[4 + i];
            if (tid == 0) {
                s_chunks = (int)keep[0];
                s_bad = (int)keep[1];
                s_over = (int)keep[2];
            }
        }
        __syncthreads();
        auto bit_set = [](volatile uint32_t *w, int i) {
            atomicOr(const_cast<uint32_t *>(w) + (i >> 5), 1u << (i & 31));
        };
        auto bit = [](const volatile uint32_t *w, int i) { return (w[i >> 5] >> (i & 31)) & 1u; };
        for (int e = d.dstart[c] + tid; e < d.Bp[c + 1]; e += TD_NT) {
            const int r = d.Bi[e];
            const int s = slot_of(T, base, r);
            if (s < 0) { report_internal(d.status, c, 61); continue; }
            if (stage < 2) {
                x[s] = Bx[e];
                bit_set(pr, s);
            }
            // (the rows of separators below have their pivots by stage 2)
            if (s < ndesc && !quit && (stage == 0 || !(d.tasks[d.col_task[r]].level == 0 ? stage == 2 : part))) {
                const int p = d.pinv[r] - base;
                if ((unsigned)p < (unsigned)ndesc) bit_set(sb, p);
                else report_internal(d.status, c, 62);
            }
        }
        __syncthreads();

        // the updates of log g to the slots that want(slot) takes
        auto take_log = [&](int g, auto &&want, bool desc) {
            int chunk = nfirst[g];
            const int cnt = ncnt[g];
            auto place_of = [&](int o) { return (int64_t)chunk * TD_CK + (o & (TD_CK - 1)) + lane; };
            // the next 32 entries are read while 32 are applied
            int s1 = lane < cnt ? log_s[place_of(0)] : -1;
            V l1 = lane < cnt ? log_l[place_of(0)] : V(0), m1 = lane < cnt ? log_m[place_of(0)] : V(0);
            for (int o = 0; o < cnt; o += 32) {
                const int s = s1;
                const V l = l1, m = m1;
                const int on = o + 32;
                if (on < cnt) {
                    if ((on & (TD_CK - 1)) == 0) chunk = next[chunk];
                    const int64_t at = place_of(on);
                    s1 = on + lane < cnt ? log_s[at] : -1;
                    l1 = on + lane < cnt ? log_l[at] : V(0);
                    m1 = on + lane < cnt ? log_m[at] : V(0);
                }
                const bool sel = s >= 0 && want(s);
                if (__any_sync(BK_FULL, sel)) {
                    const uint32_t peers = __match_any_sync(BK_FULL, sel ? s : -1 - lane);
                    const int rank = __popc(peers & lt);
                    const int most = (int)__reduce_max_sync(BK_FULL, sel ? (unsigned)rank : 0u);
                    for (int k = 0; k <= most; k++) {
                        if (sel && rank == k) {
                            const bool in = bit(pr, s);
                            x[s] = fma(-l, m, in ? x[s] : V(0));
                            if (!in) {
                                bit_set(pr, s);
                                if (desc) {
                                    const int p = __ldcg(d.pinv + base + s) - base;
                                    if ((unsigned)p < (unsigned)ndesc) bit_set(sb, p);
                                    else report_internal(d.status, c, 63);
                                }
                            }
                        }
                        __syncwarp();
                    }
                }
            }
        };

        for (int h = stage == 2 ? 1 : 0; h < (quit ? 0 : part ? 1 : T.level); h++) {
            for (int D = wid; D < nn; D += TD_W) {
                const bk_task *const N = d.tasks + t0 + D;
                if (__any_sync(BK_FULL, N->level != h || s_over)) continue;
                const int nlo = N->lo - base, nhi = N->hi - base;     // the node's rows and steps
                const int f = N->sp_lo < N->lo ? d.col_task[N->sp_lo] - t0 : D;
                for (int e = f; e < D; e++) take_log(2 * e, [&](int s) { return s >= nlo && s < nhi; }, true);
                // the node's steps, lowest first; the step after the current one, as
                // known, has its place and its first 64 entries read meanwhile
                int wd = nlo >> 5;
                auto lowest = [&](int from) -> int {       // pending step at or after from, in the node
                    for (int w = max(wd, from >> 5); w <= (nhi - 1) >> 5; w += 32) {
                        uint32_t v = w + lane <= (nhi - 1) >> 5 ? sb[w + lane] : 0u;
                        if (w + lane == from >> 5) v &= ~0u << (from & 31);
                        if (w + lane == (nhi - 1) >> 5 && (nhi & 31)) v &= (1u << (nhi & 31)) - 1u;
                        const uint32_t ball = __ballot_sync(BK_FULL, v != 0u);
                        if (ball) {
                            const int l = __ffs(ball) - 1;
                            return ((w + l) << 5) + __ffs(__shfl_sync(BK_FULL, v, l)) - 1;
                        }
                    }
                    return -1;
                };
                // a step: its pivot row's slot, its L column's place and first 64 entries
                // (row, row as step, that step's L column, value)
                struct Step {
                    int j, sp, jc;
                    int64_t jl;
                    int r[2], p[2];
                    unsigned long long k[2];
                    V l[2];
                };
                auto place = [&](Step &S, int j) {
                    S.j = j;
                    if (j < 0) return;
                    S.sp = __ldcg(d.prow + base + j) - base;
                    S.jl = __ldcg(d.Lbeg + base + j);
                    S.jc = __ldcg(d.Lcnt + base + j);
                };
                auto entries = [&](Step &S) {
                    if (S.j < 0) return;
#pragma unroll
                    for (int u = 0; u < 2; u++) {
                        const int q = lane + 32 * u;
                        S.r[u] = q < S.jc ? d.Li[S.jl + q] : -1;
                        S.p[u] = q < S.jc ? d.Ls[S.jl + q] : -1;
                        S.k[u] = q < S.jc ? lg.link[S.jl + q] : 0ull;
                        S.l[u] = q < S.jc ? Lx[S.jl + q] : V(0);
                    }
                };
                int lchunk[2] = {-1, -1}, lcnt[2] = {0, 0};
                Step cur, nx;
                place(cur, nhi > nlo ? lowest(nlo) : -1);
                entries(cur);
                place(nx, cur.j >= 0 ? lowest(cur.j + 1) : -1);
                while (cur.j >= 0 && !__any_sync(BK_FULL, s_over)) {
                    const int j = cur.j;
                    if ((unsigned)cur.sp >= (unsigned)ndesc) {
                        if (lane == 0) report_internal(d.status, c, 64);
                        break;
                    }
                    wd = j >> 5;
                    entries(nx);
                    Step n2;
                    place(n2, nx.j >= 0 ? lowest(nx.j + 1) : -1);
                    const V m = x[cur.sp];
                    if (!isfinite(m)) s_bad = 1;
                    if (lane == 0) {
                        atomicAnd(const_cast<uint32_t *>(sb) + (j >> 5), ~(1u << (j & 31)));
                        bit_set(ap, j);
                    }
                    unsigned newmin = 0xffffffffu;      // the lane's lowest new step, its
                    unsigned long long nlink = 0ull;    // L column and its row's slot
                    int nslot = -1;
                    for (int q0 = 0; q0 < cur.jc; q0 += 32) {
                        int r, p;
                        unsigned long long k;
                        V l;
                        if (q0 < 64) {
                            r = q0 == 0 ? cur.r[0] : cur.r[1];
                            p = q0 == 0 ? cur.p[0] : cur.p[1];
                            k = q0 == 0 ? cur.k[0] : cur.k[1];
                            l = q0 == 0 ? cur.l[0] : cur.l[1];
                        } else {
                            const int q = q0 + lane;
                            r = q < cur.jc ? d.Li[cur.jl + q] : -1;
                            p = q < cur.jc ? d.Ls[cur.jl + q] : -1;
                            k = q < cur.jc ? lg.link[cur.jl + q] : 0ull;
                            l = q < cur.jc ? Lx[cur.jl + q] : V(0);
                        }
                        const int s0 = r - base;
                        const bool own = r >= 0 && s0 < nhi;
                        if (own) {
                            if (s0 < nlo) {
                                report_internal(d.status, c, 65);
                            } else {
                                const bool in = bit(pr, s0);
                                x[s0] = fma(-l, m, in ? x[s0] : V(0));
                                if (!in) {
                                    bit_set(pr, s0);
                                    const int st = p - base;
                                    if (st > j && st < nhi) {
                                        bit_set(sb, st);
                                        if ((unsigned)st < newmin) {
                                            newmin = (unsigned)st;
                                            nlink = k;
                                            nslot = s0;
                                        }
                                    } else {
                                        report_internal(d.status, c, 66);
                                    }
                                }
                            }
                        }
                        // above the node: to its logs, each with at most one new chunk
                        const int g = r >= 0 && !own ? (r >= T.lo ? 1 : 0) : -1;
                        bool full = false;
#pragma unroll
                        for (int t = 0; t < 2; t++) {
                            const uint32_t up = __ballot_sync(BK_FULL, g == t);
                            if (!up) continue;
                            const int add = __popc(up), off = lcnt[t] & (TD_CK - 1);
                            int fresh = -1;
                            if (off == 0 || off + add > TD_CK) {
                                if (lane == 0) {
                                    fresh = atomicAdd(&s_chunks, 1);
                                    if (fresh >= nchunks) {
                                        s_over = 1;
                                        fresh = -1;
                                    } else if (lcnt[t] == 0) {
                                        nfirst[2 * D + t] = fresh;
                                    } else {
                                        next[lchunk[t]] = (uint16_t)fresh;
                                    }
                                }
                                fresh = __shfl_sync(BK_FULL, fresh, 0);
                                if (fresh < 0) {
                                    full = true;
                                    break;
                                }
                            }
                            if (g == t) {
                                const int sl = r < T.hi ? r - base : slot_of(T, base, r);
                                if (sl < 0) report_internal(d.status, c, 67);
                                const int at0 = off + __popc(up & lt);
                                const bool here = off > 0 && at0 < TD_CK;
                                const int64_t at = (int64_t)(here ? lchunk[t] : fresh) * TD_CK + (at0 & (TD_CK - 1));
                                log_s[at] = sl;
                                log_l[at] = l;
                                log_m[at] = m;
                            }
                            lcnt[t] += add;
                            if (fresh >= 0) lchunk[t] = fresh;
                        }
                        if (full) break;
                    }
                    __syncwarp();
                    const unsigned mine = newmin;
                    newmin = __reduce_min_sync(BK_FULL, newmin);
                    if (newmin < (unsigned)(nx.j < 0 ? INT_MAX : nx.j)) {
                        // a step the current one added comes first: its place is
                        // with the entry that added it
                        const int old = nx.j;
                        const int from = __ffs(__ballot_sync(BK_FULL, mine == newmin)) - 1;
                        const unsigned long long lk = __shfl_sync(BK_FULL, nlink, from);
                        cur.j = (int)newmin;
                        cur.sp = __shfl_sync(BK_FULL, nslot, from);
                        cur.jl = (int64_t)(lk >> 20);
                        cur.jc = (int)(lk & 0xfffffull);
                        entries(cur);
                        // the steps after it: the lowest pending beyond it
                        const int after = lowest((int)newmin + 1);
                        if (after != old) place(nx, after);
                    } else {
                        cur = nx;
                        // n2 was found before the current step's additions
                        const int after = cur.j >= 0 && newmin != 0xffffffffu ? lowest(cur.j + 1) : n2.j;
                        if (after == n2.j) nx = n2;
                        else place(nx, after);
                    }
                }
                if (lane == 0) {
                    ncnt[2 * D] = lcnt[0];
                    ncnt[2 * D + 1] = lcnt[1];
                }
                __syncwarp();
            }
            __syncthreads();
        }
        if (part) {
            // the rest when the separators below are factored
            for (int i = tid; i < words; i += TD_NT) keep[4 + i] = td_sm[i];
            if (tid == 0) {
                keep[0] = (uint32_t)s_chunks;
                keep[1] = (uint32_t)s_bad;
                keep[2] = (uint32_t)s_over;
            }
            continue;
        }
        if (!s_over && !quit) {
            // the separator's and its ancestors' rows: a warp takes every TD_W-th slot
            for (int D = 0; D < nn; D++)
                take_log(2 * D + 1, [&](int s) { return (s & (TD_W - 1)) == wid; }, false);
        }
        __syncthreads();
        if (quit) {
        } else if (s_over) {
            if (tid == 0) over[atomicAdd(nover, 1)] = c;
        } else {
            // U(desc, c): the applied steps in ascending order, a run of words a thread
            const int per = (nsw + TD_NT - 1) / TD_NT, wa = min(nsw, tid * per), wz = min(nsw, wa + per);
            int mine = 0;
            for (int w = wa; w < wz; w++) mine += __popc(ap[w]);
            const int pre = warp_exscan(mine, lane);
            if (lane == 31) s_wsum[wid] = pre + mine;
            __syncthreads();
            int o = pre, nu = 0;
            for (int w = 0; w < TD_W; w++) {
                if (w < wid) o += s_wsum[w];
                nu += s_wsum[w];
            }
            __shared__ long long s_ub;
            if (tid == 0) {
                int64_t ub = d.Ubeg[c];
                if (ub + nu + 2 > d.Uend[c]) {
                    const int64_t cap = grown_ucap(nu, (int64_t)(c - T.sp_lo) + 1);
                    ub = pool_alloc(d.pool + 1, d.upool_end, cap);
                    if (ub >= 0) {
                        d.Ubeg[c] = ub;
                        d.Uend[c] = ub + cap;
                    }
                }
                s_ub = ub;
                d.dcnt[c] = nu;
                if (ub < 0) report_overflow(d, T, task, c, 2);
                else if (s_bad) report_fail(d.status, c, BK_CODE_NAN);
            }
            __syncthreads();
            const int64_t ub = s_ub;
            if (ub >= 0)
                for (int w = wa; w < wz; w++) {
                    uint32_t v = ap[w];
                    while (v) {
                        const int j = (w << 5) + __ffs(v) - 1;
                        v &= v - 1;
                        d.Ui[ub + o] = base + j;
                        Ux[ub + o] = x[__ldcg(d.prow + base + j) - base];
                        o++;
                    }
                }
            // A-hat(:,c) on the separator's and its ancestors' rows, and its pattern
            const int nrw = (lsp + 31) >> 5;
            V *const ah = Ahat + T.ahoff + (int64_t)(c - T.lo) * lsp;
            uint32_t *const ab = d.abits + T.aboff + (int64_t)(c - T.lo) * nrw;
            for (int ls = tid; ls < nrw * 32; ls += TD_NT) {
                const bool in = ls < lsp && bit(pr, ndesc + ls);
                const uint32_t word = __ballot_sync(BK_FULL, in);
                if (lane == 0) ab[ls >> 5] = word;
                if (in) ah[ls] = x[ndesc + ls];
            }
        }
        __syncthreads();
        // x clean again
        for (int w = tid; w < npw; w += TD_NT) {
            uint32_t v = pr[w];
            while (v) {
                x[(w << 5) + __ffs(v) - 1] = V(0);
                v &= v - 1;
            }
        }
    }
}

// The rows of the L columns of level `level` of the ND block as steps (rows pivoted
// by now; others -1), and where those steps' own L columns lie.
__global__ void bk_lsteps_kernel(bk_dev d, int c0, int c1, int level, unsigned long long *link)
{
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int c = c0 + ((blockIdx.x * blockDim.x + threadIdx.x) >> 5); c < c1; c += warps) {
        if (d.tasks[d.col_task[c]].level != level) continue;
        const int64_t lb = d.Lbeg[c];
        const int lc = d.Lcnt[c];
        for (int q = lane; q < lc; q += 32) {
            const int p = d.pinv[d.Li[lb + q]];
            d.Ls[lb + q] = p;
            link[lb + q] = p >= 0 ? ((unsigned long long)d.Lbeg[p] << 20) | (unsigned long long)d.Lcnt[p] : 0ull;
        }
    }
}

}  // namespace

size_t bk_tdesc_smem(const bk_tdesc_dev &lg, int64_t ndesc, int64_t space)
{
    const int64_t nchunks = lg.cap / TD_CK;
    return (size_t)(4 * lg.nodes + ((nchunks + 1) >> 1) + 2 * ((ndesc + 31) / 32) + (space + 31) / 32 + 4) * 4;
}

void bk_launch_lsteps(const bk_dev &d, const bk_tdesc_dev &lg, int32_t c0, int32_t c1, int32_t level, void *stream)
{
    if (c1 <= c0) return;
    bk_lsteps_kernel<<<std::max(1, std::min((c1 - c0 + 7) / 8, 152 * 8)), 256, 0, (cudaStream_t)stream>>>(d, c0, c1, level,
                                                                                                  lg.link);
}

void bk_launch_tdesc(const bk_dev &d, const bk_tdesc_dev &lg, const int32_t *cols, int32_t ncols, int32_t *counter,
                     const int32_t *ncols_dev, int32_t *over, int32_t *nover, size_t smem, int stage, int first,
                     void *stream)
{
    if (ncols <= 0) return;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaFuncSetAttribute(bk_tdesc_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, BK_TDESC_SMEM);
        cudaFuncSetAttribute(bk_tdesc_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, BK_TDESC_SMEM);
    });
    // staged: a region a column; else a region a block
    const int grid = stage ? std::min(ncols, 608) : std::min(std::min(ncols, lg.blocks), d.wsd_warps);
    cudaStream_t s = (cudaStream_t)stream;
    if (d.prec)
        bk_tdesc_kernel<float><<<grid, TD_NT, smem, s>>>(d, cols, ncols, counter, ncols_dev, over, nover, lg, stage, first);
    else
        bk_tdesc_kernel<double><<<grid, TD_NT, smem, s>>>(d, cols, ncols, counter, ncols_dev, over, nover, lg, stage, first);
}
