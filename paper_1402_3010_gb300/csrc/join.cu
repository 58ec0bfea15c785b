// The inverted-index join (Alg. 2, Find-Matches, with the all-pairs-2 bounds) and the
// output stage.
//
// One persistent launch takes every size class in turn, one CTA per SM. A join tile is one
// warp: it holds a dense score array A over a window of W candidate ids in its own part of
// shared memory (the paper's all-pairs-0-array accumulator, cut into windows because n floats
// do not fit on chip), so no step of a query vector waits for another warp and the warps of an
// SM hide one another's latency. For a query x (a whole vector of the set from a cost-ordered
// work list, or one part of its windows where x is among the heaviest) and each window of
// candidates y > x:
//   1. create: A[y] += x[i] * y[i] over the posting lists of x's components from its create
//      boundary on (remscore and norm bounds: a match has one of these in common with x). A
//      holds 32-bit fixed-point sums (products rounded up to multiples of 2^-30, at least one
//      unit), added with integer shared-memory atomics whose returned old value tells a slot's
//      first update: those slots go to the warp's candidate list. Entries with |y| below minsize
//      are skipped using the size class stored in the entry;
//   2. update: the same over x's earlier components, which only add where A is not zero;
//   3. filter: dot(x, y') <= ||x on the ranks before y's first indexed one|| * ||y'||
//      (Cauchy-Schwarz). Both of y's parts are in its one-byte code, x's norms in a table made
//      once per unit, so a candidate costs one byte of global memory;
//   4. verify the rest, one candidate per lane: the same bound with the exact norm, in a self-join
//      the paper's upperbound A[y] + min(|y'|, |x|) * maxweight(x) * maxweight(y') >= t, then
//      s = A[y] + dot(x, y') with y' the unindexed prefix of y; scores within a band of t are
//      recomputed in float64 and decided there. A match leaves its score in A and a bit in the
//      window's bitmap;
//   5. emit: the bitmap is walked in id order and the (y, score) go to the staging slab that
//      the warp reserves in bulk. The run of x (or of its part) is recorded at its slot.
// A window with more candidates than the list holds is filtered from A itself, in stretches
// of as many slots as the list has entries. (Such windows are dearer than they were with groups of
// warps, 1.3 to 1.8 times at loose thresholds or over a few dozen dimensions; scanning them in the
// filter's own loop was no better, 5.9 against 5.2 ms for 50,000 rows at t = 0.4.)
// What bounds it is the latency of its loads with the 24 warps that 80 registers a thread allow: at
// 50,000 rows a scheduler issues in half of the cycles (0.8 of its 6 warps ready), the top stall is the
// long scoreboard (3.7 cycles an issue), no pipe is above 30%, L1 at 40% and L2 at 17%.
// With groups of warps sharing a window, and barriers between these steps, and lists up
// to the split alone, the 200,000-row power-law set took 37.2 ms and a batch of 512 instances
// 58; 21.6 and 14.9 now. 4096 queries against a million rows take 7.1 ms a call (17.2).
// The output stage scans the per-slot counts and gathers the staged runs into (i, j, score)
// arrays, which are then in (i, j) order without a sort.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <system_error>
#include <thread>
#include <vector>

#include "index.cuh"

namespace aps {
namespace {

std::atomic<int64_t> g_stage_hint{0};
std::atomic<int64_t> g_stage_cap_once{0};  // test hook: staging room of the next self-join

struct JoinParams {
    const InstDesc *inst;
    const int32_t *vinst;
    const int32_t *items;
    int one;  // a single instance
    // classes, taken in order by one persistent launch: class c is the work-list range
    // [cls_begin[c], cls_begin[c + 1]) run with tile shape cls_G[c], or, when cls_G[c] is 0,
    // one warp per vector with one or two components. The first cls_heavy[c] items are cut
    // into `parts` parts of their windows.
    int ncls;
    int cls_G[JOIN_NCLS];
    int64_t cls_begin[JOIN_NCLS + 1];
    int64_t cls_heavy[JOIN_NCLS];
    int parts;
    const int2 *crow;    // rank-ordered rows {rank, value}
    const int4 *vmeta;   // {row offset, |x|, create boundary, maxweight(x)}
    const int4 *vcand;   // {row offset, |y'|, first rank after y', ||y'||_2 bound}
    const float *mwj;    // maxweight(y')
    const uint8_t *code; // per vector: octave of the first rank after y', 4-bit ||y'||_2 bound
    // dimension-block items (the vertical split with local pruning, Sec. 5.1): iblk[it] >= 0
    // makes work item it one of nblk blocks of the vector items[it]; null: none
    const int8_t *iblk;
    int nblk;
    // a block item's lists, boundaries and prefixes (up to the split alone)
    const int4 *vmeta_b, *vcand_b;
    const uint8_t *code_b;
    const int64_t *lptr_b;
    const uint32_t *wptr_b;
    const int2 *post_b;
    unsigned long long *sp_key;    // pairs found by block items: local x * n + local y
    uint32_t *sp_score;            // their float32 scores (bits)
    unsigned long long *sp_count;  // pairs reserved in sp_key / sp_score
    int64_t sp_cap;
    const int64_t *lptr;
    const uint32_t *wptr;
    const int2 *post;
    const uint64_t *wlist, *wlist_b;  // COARSE: the lists' places in wptr (in wptr_b)
    uint32_t flags;
    int2 *stage;
    int64_t stage_cap;
    unsigned long long *stage_count;  // staging slots handed out (whole slabs of stage_slab)
    int64_t stage_slab;
    Segment *segs;                    // [slots]: the first piece of a slot's run
    int2 *chain;                      // [stage_cap / stage_slab + 1]: later pieces, by slab
    int32_t *cntq;                    // [slots]: pairs
    unsigned long long *counters;  // visits, candidates, verified, pairs, band; [6] entries read
    unsigned long long *work;       // [ncls] work-list cursors
    int2 *scratch;                  // per-warp lists of the streamed class, JOIN_ECAP each
    // query mode: items are external query rows matched against every indexed vector
    const int2 *qcrow;    // query rows over the index's ranks
    const int4 *qvmeta;   // {row offset, |q|, create boundary, maxweight(q)}
    float qt;
};

__device__ __forceinline__ int64_t warp_incl_scan(int64_t v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int64_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

__device__ __forceinline__ int warp_excl_scan_int(int v, int lane, int *total) {
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    *total = __shfl_sync(0xffffffffu, inc, 31);
    return inc - v;
}

// Position of the first entry at or after `lo` of a rank-ordered row whose rank is >= r.
__device__ __forceinline__ int row_find(const int2 *row, int lo, int hi, const int r) {
#pragma unroll 1
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (row[mid].x < r) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// The value at rank r of a rank-ordered row (0 when it has none).
__device__ __forceinline__ float x_at(const int r, const int2 *xrow, const int xl) {
    const int p = row_find(xrow, 0, xl, r);
    if (p < xl) {
        const int2 e = xrow[p];
        if (e.x == r) return __int_as_float(e.y);
    }
    return 0.f;
}

// A warp's staging place and the pieces of the run that it is writing, in shared memory.
// Reservations are whole slabs, so a piece that
// begins a reservation is named by its slab. Nothing is left unused but the rest of the last one.
struct Stager {
    int64_t base;         // current reservation
    int64_t head;         // the run's first pair
    uint32_t used, size;  // of the reservation
    uint32_t piece_cnt, head_cnt, cnt;
    int32_t piece;        // slab of the current piece, -1: the run's first one
    int32_t head_next;
    // room handed out last: pair p goes to a + p for p < f, to b + p - f from there on
    uint32_t f;
    int64_t a, b;
};

// Work totals of a warp: visits, candidates, verified, pairs, band, entries read.
struct Totals {
    unsigned long long v[6];
};

// tot[k] += the warp's sum of v. Warp-collective.
__device__ __forceinline__ void count_add(Totals &S, const int k, const uint32_t v, const int lane) {
    const uint32_t s = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0) S.v[k] += s;
}

// Room for c more pairs of the run: S.a, S.f, S.b. One thread.
__device__ __forceinline__ void stage_take(Stager &S, const JoinParams &P, const uint32_t c) {
    const uint32_t f = min(c, S.size - S.used);
    const int64_t a = S.base + S.used;
    S.a = a;
    S.f = f;
    if (f == c) {
        if (S.cnt == 0) S.head = a;
        S.used += c;
        S.piece_cnt += c;
        S.cnt += c;
        return;
    }
    const uint32_t slab = (uint32_t)P.stage_slab;
    const uint32_t want = (c - f + slab - 1) / slab * slab;
    const int64_t b = (int64_t)atomicAdd(P.stage_count, (unsigned long long)want);
    S.b = b;
    if (S.cnt == 0 && f == 0) {  // the run begins here
        S.head = b;
        S.piece_cnt = c;
    } else {
        if (S.cnt == 0) S.head = a;
        const int32_t nx = (int32_t)(b / slab);
        if (S.piece < 0) {
            S.head_cnt = S.piece_cnt + f;
            S.head_next = nx;
        } else if ((int64_t)S.piece * slab < P.stage_cap) {
            P.chain[S.piece] = make_int2((int)(S.piece_cnt + f), nx);
        }
        S.piece = nx;
        S.piece_cnt = c - f;
    }
    S.base = b;
    S.size = want;
    S.used = c - f;
    S.cnt += c;
}

// The run is complete: its record at `slot`. One thread.
__device__ __forceinline__ void stage_close(Stager &S, const JoinParams &P, const int64_t slot, const int32_t id) {
    if (S.cnt == 0) return;
    P.cntq[slot] = (int32_t)S.cnt;
    Segment g;
    g.src = S.head;
    g.cnt = (int32_t)(S.piece < 0 ? S.piece_cnt : S.head_cnt);
    g.i = id;
    g.next = S.piece < 0 ? -1 : S.head_next;
    g._pad = 0;
    P.segs[slot] = g;
    if (S.piece >= 0 && (int64_t)S.piece * P.stage_slab < P.stage_cap)
        P.chain[S.piece] = make_int2((int)S.piece_cnt, -1);
    S.piece = -1;
    S.piece_cnt = S.cnt = 0;
}

__device__ __forceinline__ void stage_put(const JoinParams &P, const Stager &S, const uint32_t p, const int2 v) {
    const int64_t at = p < S.f ? S.a + p : S.b + (p - S.f);
    if (at < P.stage_cap) P.stage[at] = v;  // past the room: the host grows it and runs again
}

// First position in [a, b) of a posting list (ids increasing) whose id exceeds lx, or b
// when none does: a 32-way search by the whole warp (each step probes 32 evenly spaced
// entries and keeps the one gap that holds the answer).
__device__ __forceinline__ int64_t first_after(const int2 *__restrict__ post, int64_t a, int64_t b, const int32_t lx,
                                               const int32_t idmask, const int lane) {
    while (b - a > 32) {
        const int64_t step = (b - a + 31) >> 5;
        const int64_t pos = a + (int64_t)lane * step;
        const bool past = pos >= b || (__ldg(&post[pos].x) & idmask) > lx;
        const unsigned m = __ballot_sync(0xffffffffu, past);
        if (m & 1u) return a;  // the range's first entry is already after x
        if (m == 0u) {
            a += 31 * step + 1;  // every probe at or before x: the answer lies after the last one
        } else {
            const int f = __ffs(m) - 1;  // probe f is past x, probe f - 1 is not
            b = min(b, a + (int64_t)f * step);
            a += (int64_t)(f - 1) * step + 1;
        }
    }
    const int64_t pos = a + lane;
    const unsigned m = __ballot_sync(0xffffffffu, pos < b && (__ldg(&post[pos].x) & idmask) > lx);
    return m ? a + (__ffs(m) - 1) : b;
}

// First position of post in [lo, hi) (one list, ids increasing) whose id is at or past `bound`, or hi.
__device__ __forceinline__ uint32_t first_at(const int2 *__restrict__ post, uint32_t lo, uint32_t hi,
                                             const uint32_t bound, const int32_t idmask) {
#pragma unroll 1
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if ((uint32_t)(__ldg(&post[mid].x) & idmask) < bound) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// The part of the list of global rank R in window w, [s0, s1), where starts are stored by list
// (instance of nw windows of W ids). Returns the list's starts where it has every window's, else null.
__device__ __forceinline__ const uint32_t *list_range(const uint64_t *__restrict__ wlist,
                                                      const uint32_t *__restrict__ wptr,
                                                      const int64_t *__restrict__ lptr,
                                                      const int2 *__restrict__ post, const int64_t R, const int w,
                                                      const int nw, const int W, const int32_t idmask, uint32_t &s0,
                                                      uint32_t &s1) {
    const uint64_t d = __ldg(wlist + R);
    const int shift = (int)(d & 63u);
    const uint32_t *const starts = wptr + (d >> 6);
    const bool grouped = window_groups(nw, shift) > 1;
    if (grouped) {
        s0 = __ldg(starts + (w >> shift));
        s1 = __ldg(starts + (w >> shift) + 1);
        if (shift == 0) return starts;
    } else {
        s0 = (uint32_t)__ldg(lptr + R);
        s1 = (uint32_t)__ldg(lptr + R + 1);
    }
    const int within = (1 << shift) - 1;
    if (w & within) s0 = first_at(post, s0, s1, (uint32_t)w * (uint32_t)W, idmask);
    if (((w + 1) & within) && w + 1 < nw) s1 = first_at(post, s0, s1, (uint32_t)(w + 1) * (uint32_t)W, idmask);
    return nullptr;
}

// The part of a posting list after x: [first, end) of list rank r of instance I (the
// search starts in the window of x's successor, whose part of the list holds the answer
// or ends right before it).
template <bool COARSE>
__device__ __forceinline__ void list_after(const JoinParams &P, const InstDesc &I, const int r, const int32_t lx,
                                           const int wf, const int32_t idmask, const int lane, int64_t &first,
                                           int64_t &end) {
    const int64_t R = (int64_t)I.rbase + r;
    const int64_t ls = P.lptr[R];
    end = P.lptr[R + 1];
    int64_t a = ls, b = end;
    if (COARSE) {
        const uint64_t d = P.wlist[R];
        if (window_groups(I.nw, (int)(d & 63u)) > 1) {
            const uint32_t *wp = P.wptr + (d >> 6) + (wf >> (int)(d & 63u));
            a = wp[0];
            b = wp[1];
        }
    } else if (I.nw > 1) {
        const uint32_t *wp = P.wptr + I.wbase + (int64_t)r * (I.nw + 1);
        a = wp[wf];
        b = wp[wf + 1];
    }
    first = first_after(P.post, a, b, lx, idmask, lane);
}

// Number of the 32 values v held by the lanes (increasing with the lane, padded with
// INT_MAX) that are below key (LE: at or below key), by halving over the lanes.
template <bool LE>
__device__ __forceinline__ int count_below(const int v, const int key) {
    int c = 0;
#pragma unroll
    for (int h = 16; h; h >>= 1) {
        const int w = __shfl_sync(0xffffffffu, v, c + h - 1);
        if (LE ? w <= key : w < key) c += h;
    }
    const int w = __shfl_sync(0xffffffffu, v, 31);
    if (c == 31 && (LE ? w <= key : w < key)) c = 32;
    return c;
}

// The vectors with one or two components (Alg. 2 for |x| <= 2), one warp per vector, no
// accumulator and no windows.
//   |x| = 1 (rank r, value x0): every entry (y, w) of r's list with y after x and
//   |y| >= minsize is a candidate whose accumulated score x0 * w is its whole score (x has
//   no other component, and dot(x, y') = 0 since r lies in y's indexed part).
//   |x| = 2 (ranks r0 < r1, values x0, x1): the two lists after x are merged by id, 32
//   entries at a time. An id on both lists scores x0 * w0 + x1 * w1 (both ranks in y's
//   indexed part, so y's prefix holds neither); an id on r0's list alone scores x0 * w0
//   (y has no r1: it is not in the indexed part, and the prefix ranks lie below r0), and is
//   a candidate only if r0 may create (remscore); an id on r1's list alone scores
//   x1 * w1 + x0 * y[r0], where y[r0] can only sit in y's unindexed prefix (looked up there
//   unless the ||y'||_2 bound already rules the pair out).
// Each candidate is decided like the windowed path (float32 outside a band of beta around
// t, the exact float64 sum of the products inside it). The matches, in increasing y, go to
// the warp's scratch list and are then copied as x's run to the staging slab that the warp
// reserves in bulk; a vector with more matches than the scratch list holds is streamed a
// second time, writing them there directly.
template <bool COARSE>
__device__ __forceinline__ void stream_short(const JoinParams &P, unsigned long long *work, const int64_t item_begin,
                                          const int64_t item_end, const bool f_minsize, const bool f_remscore,
                                          Totals &tot, Stager &S) {
    const int lane = threadIdx.x & 31;
    struct {
        uint32_t visits = 0, cand = 0, verified = 0, band = 0;
    } ct;  // folded into the warp's totals after every item
    const unsigned lt_mask = (1u << lane) - 1u;
    int2 *const elist = P.scratch + ((size_t)blockIdx.x * JOIN_WARPS + (threadIdx.x >> 5)) * JOIN_ECAP;
    // the first item is this warp's own, the next ones are asked for one item ahead (lane 0)
    const unsigned long long nwarps = (unsigned long long)gridDim.x * JOIN_WARPS;
    unsigned long long nw = blockIdx.x + (unsigned long long)gridDim.x * (threadIdx.x >> 5);
    for (;;) {
        const int64_t it = (int64_t)__shfl_sync(0xffffffffu, nw, 0) + item_begin;
        count_add(tot, 0, ct.visits, lane);
        count_add(tot, 1, ct.cand, lane);
        count_add(tot, 2, ct.verified, lane);
        count_add(tot, 4, ct.band, lane);
        ct.visits = ct.cand = ct.verified = ct.band = 0;
        if (it >= item_end) break;
        if (lane == 0) nw = atomicAdd(work, 1ull) + nwarps;
        const int64_t x = P.items[it];
        const InstDesc I = P.inst[P.vinst[x]];
        const int32_t lx = (int32_t)(x - I.vbase);
        const int4 xm = P.vmeta[x];
        const int xl = xm.y;  // 1 or 2
        const int qs = f_remscore ? xm.z : 0;
        if (qs >= xl) continue;  // remscore < t from the first component on: no candidate
        const int2 xe0 = P.crow[xm.x];
        const int2 xe1 = xl == 2 ? P.crow[xm.x + 1] : make_int2(0, 0);
        const float x0 = __int_as_float(xe0.y), x1 = __int_as_float(xe1.y);
        const float t = I.t;
        const float beta = fmaxf(1e-5f, (float)(xl + 2) * 1.1920929e-7f);  // (|x| + 2) * 2^-23
        const float mwx = __int_as_float(xm.w);
        int smin = 0;  // minsize, bounded as in the windowed path
        if (f_minsize && I.packed && mwx > 0.f)
            smin = (int)ceilf(fminf(__fdiv_rd(__fsub_rd(t, beta), __fmul_ru(mwx, 1.0020001f)), 255.f));
        const uint32_t smin_tag = (uint32_t)max(smin, 0) << 24;
        const int32_t idmask = I.packed ? 0x00ffffff : 0x7fffffff;
        const int wf = (lx + 1) / I.W;  // the window of x's successor
        int64_t f0, e0, f1 = 0, e1 = 0;
        list_after<COARSE>(P, I, xe0.x, lx, wf, idmask, lane, f0, e0);
        if (xl == 2) list_after<COARSE>(P, I, xe1.x, lx, wf, idmask, lane, f1, e1);
        if (lane == 0) tot.v[5] += (unsigned long long)((e0 - f0) + (e1 - f1));
        // pass 0: count the matches, the first JOIN_ECAP into the scratch list; pass 1 (only
        // when there were more): write them all into the reserved run
        int cnt = 0;
        for (int pass = 0; pass < 2; pass++) {
            int k = 0;  // matches so far
            if (xl == 1) {
                for (int64_t p0 = f0; p0 < e0; p0 += 128) {
                    int2 e[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        const int64_t p = p0 + u * 32 + lane;
                        e[u] = p < e0 ? __ldg(&P.post[p]) : make_int2(0, 0);
                    }
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        const int64_t p = p0 + u * 32 + lane;
                        bool m = false;
                        float sc = 0.f;
                        if (p < e0 && (uint32_t)e[u].x >= smin_tag) {
                            if (pass == 0) { ct.visits++; ct.cand++; }
                            sc = x0 * __int_as_float(e[u].y);
                            if (sc >= t + beta) {
                                m = true;
                            } else if (sc > t - beta) {  // inside the band: the exact product decides
                                const double ex = (double)x0 * (double)__int_as_float(e[u].y);
                                if (pass == 0) ct.band++;
                                m = ex >= (double)t;
                                sc = (float)ex;
                            }
                        }
                        const unsigned bal = __ballot_sync(0xffffffffu, m);
                        if (m) {
                            const int at = k + __popc(bal & lt_mask);
                            const int2 v2 = make_int2(e[u].x & idmask, __float_as_int(sc));
                            if (pass == 1) stage_put(P, S, (uint32_t)at, v2);
                            else if (at < JOIN_ECAP) elist[at] = v2;
                        }
                        k += __popc(bal);
                    }
                }
            } else {
                // merge of the two lists after x, 32 merged entries per step: lane l holds
                // entry i + l of r0's list (a) and entry j + l of r1's list (b); an entry's
                // place in the merged order is its lane plus the other list's entries below
                // it (ties: a first, so an id on both lists gives a then b, adjacent)
                const int64_t n0 = e0 - f0, n1 = e1 - f1;
                int64_t i = 0, j = 0;
                const bool create0 = qs == 0;  // r0 may create candidates (remscore >= t)
                while (i < n0 || j < n1) {
                    const bool va = i + lane < n0, vb = j + lane < n1;
                    const int2 ea = va ? __ldg(&P.post[f0 + i + lane]) : make_int2(0x7fffffff, 0);
                    const int2 eb = vb ? __ldg(&P.post[f1 + j + lane]) : make_int2(0x7fffffff, 0);
                    const int ida = va ? (ea.x & idmask) : 0x7fffffff;
                    const int idb = vb ? (eb.x & idmask) : 0x7fffffff;
                    const int nb = count_below<false>(idb, ida);  // b entries below a
                    const int na = count_below<true>(ida, idb);   // a entries at or below b
                    const int ra = lane + nb, rb = lane + na;       // places in the merged order
                    const bool ina = va && ra < 32, inb = vb && rb < 32;
                    const float wbd = __int_as_float(__shfl_sync(0xffffffffu, eb.y, nb & 31));
                    // (every lane takes part in the shuffles; their results are used where valid)
                    const int idb_nb = __shfl_sync(0xffffffffu, idb, nb & 31);
                    const int ida_na = __shfl_sync(0xffffffffu, ida, (na - 1) & 31);
                    const bool dupa = va && nb < 32 && idb_nb == ida;
                    const bool dupb = vb && na > 0 && ida_na == idb;
                    const int ca = __popc(__ballot_sync(0xffffffffu, ina));
                    int cb = __popc(__ballot_sync(0xffffffffu, inb));
                    // an id on both lists whose a entry closes the step: its b entry goes too
                    {
                        const bool nd = __shfl_sync(0xffffffffu, dupb, cb & 31), nv2 = __shfl_sync(0xffffffffu, vb, cb & 31);
                        const int nna = __shfl_sync(0xffffffffu, na, cb & 31);
                        if (cb < 32 && nv2 && nd && nna <= ca) cb++;
                    }
                    // candidates: a entries (on both lists, or r0 may create), b entries alone
                    bool ma = false, mb = false;
                    float sa = 0.f, sbs = 0.f;
                    if (ina && (uint32_t)ea.x >= smin_tag) {
                        if (pass == 0) ct.visits += dupa ? 2u : 1u;  // the b entry of a shared id visits too
                        if (dupa || create0) {
                            if (pass == 0) ct.cand++;
                            const float wa = __int_as_float(ea.y), wb = dupa ? wbd : 0.f;
                            sa = fmaf(x1, wb, x0 * wa);
                            if (sa >= t + beta) {
                                ma = true;
                            } else if (sa > t - beta) {
                                const double ex = (double)x0 * (double)wa + (double)x1 * (double)wb;
                                if (pass == 0) ct.band++;
                                ma = ex >= (double)t;
                                sa = (float)ex;
                            }
                        }
                    }
                    if (inb && !dupb && (uint32_t)eb.x >= smin_tag) {
                        if (pass == 0) { ct.visits++; ct.cand++; }
                        const float wb = __int_as_float(eb.y);
                        const float s1 = x1 * wb;
                        float y0 = 0.f;
                        // y[r0] <= 1 + 1e-3 (the norm tolerance): most pairs stop here, unloaded
                        bool look = s1 + x0 * 1.0011f > t - beta;
                        int4 yc = make_int4(0, 0, 0, 0);  // {row offset, |y'|, rank after y', ||y'||_2 bound}
                        if (look) {
                            yc = __ldg(&P.vcand[I.vbase + idb]);
                            look = yc.y > 0 && xe0.x < yc.z && s1 + x0 * __int_as_float(yc.w) > t - beta;
                        }
                        if (look) {  // r0 in y's unindexed prefix?
                            if (pass == 0) ct.verified++;
                            y0 = x_at(xe0.x, P.crow + yc.x, yc.y);
                        }
                        sbs = fmaf(x0, y0, s1);
                        if (sbs >= t + beta) {
                            mb = true;
                        } else if (sbs > t - beta) {
                            const double ex = (double)x0 * (double)y0 + (double)x1 * (double)wb;
                            if (pass == 0) ct.band++;
                            mb = ex >= (double)t;
                            sbs = (float)ex;
                        }
                    }
                    // matches in merged order: a bit per place
                    const unsigned mm = __reduce_or_sync(0xffffffffu, (ma ? 1u << ra : 0u) | (mb ? 1u << rb : 0u));
                    if (ma) {  // (a lane may hold a match in both lists)
                        const int at = k + __popc(mm & ((1u << ra) - 1u));
                        const int2 v2 = make_int2(ida, __float_as_int(sa));
                        if (pass == 1) stage_put(P, S, (uint32_t)at, v2);
                        else if (at < JOIN_ECAP) elist[at] = v2;
                    }
                    if (mb) {
                        const int at = k + __popc(mm & ((1u << rb) - 1u));
                        const int2 v2 = make_int2(idb, __float_as_int(sbs));
                        if (pass == 1) stage_put(P, S, (uint32_t)at, v2);
                        else if (at < JOIN_ECAP) elist[at] = v2;
                    }
                    k += __popc(mm);
                    i += ca;
                    j += cb;
                }
            }
            if (pass == 0) {
                cnt = k;
                if (cnt == 0) break;
                __syncwarp();  // (the previous run's writers have read its place)
                if (lane == 0) {
                    stage_take(S, P, (uint32_t)cnt);
                    stage_close(S, P, x * P.parts, lx);
                    tot.v[3] += (unsigned long long)cnt;
                }
                __syncwarp();
                if (cnt <= JOIN_ECAP) {  // every match is in the scratch list
#pragma unroll 1
                    for (int q = lane; q < cnt; q += 32) stage_put(P, S, (uint32_t)q, elist[q]);
                    break;
                }
            }
        }
    }
}

// A warp's part of shared memory.
struct Tile {
    uint32_t *A;     // [tile_window(G)] accumulated scores, fixed point, units of 2^-30
    uint32_t *bm;    // [tile_window(G) / 32] the window's matches
    float *px;       // [64] norm of x on the rank buckets 0 .. b
    int4 *wait;      // [32] lists of a long x waiting for a walk: {first position, entries, x's value, -}
    int2 *seg;       // [32] the lists of a run: {first position - place in the run, x's value scaled by 2^30}
    int2 *xr;        // [JOIN_XCAP] x's row, where it fits
    uint16_t *list;  // [JOIN_LCAP] candidate slots
};

// What a walk needs beside its lists.
struct WinCtx {
    uint32_t smin_tag;
    int32_t idmask;
    int w0, first;  // first id of the window; first id after x
};

// Predicated single instructions for the walk's steps (the compiler turns the same conditions
// written in C++ into divergent branches, which cost more than the instruction they guard).
__device__ __forceinline__ uint32_t shl_clamped(const uint32_t v, const uint32_t by) {  // 0 from 32 on
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(by));
    return r;
}
__device__ __forceinline__ void ldg_if(const bool on, const int2 *p, int2 &v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p ld.global.nc.v2.u32 {%0, %1}, [%2];\n\t}"
                 : "+r"(v.x), "+r"(v.y)
                 : "l"(p), "r"((uint32_t)on));
}
__device__ __forceinline__ uint32_t atoms_add_if(const bool on, const uint32_t addr, const uint32_t q) {  // old, or 1
    uint32_t old;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\tmov.u32 %0, 1;\n\t@p atom.shared.add.u32 %0, [%1], %2;\n\t}"
                 : "=&r"(old)
                 : "r"(addr), "r"(q), "r"((uint32_t)on)
                 : "memory");
    return old;
}
__device__ __forceinline__ void reds_add_if(const bool on, const uint32_t addr, const uint32_t q) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p red.shared.add.u32 [%0], %1;\n\t}" ::"r"(addr), "r"(q),
                 "r"((uint32_t)on)
                 : "memory");
}
__device__ __forceinline__ uint32_t lds_if(const bool on, const uint32_t addr) {  // or 0
    uint32_t v;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\tmov.u32 %0, 0;\n\t@p ld.shared.u32 %0, [%1];\n\t}"
                 : "=&r"(v)
                 : "r"(addr), "r"((uint32_t)on)
                 : "memory");
    return v;
}
__device__ __forceinline__ void sts16_if(const bool on, const uint32_t addr, const uint32_t v) {
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b16 h;\n\tsetp.ne.u32 p, %2, 0;\n\tcvt.u16.u32 h, %1;\n\t@p st.shared.u16 [%0], h;\n\t}" ::"r"(addr),
                 "r"(v), "r"((uint32_t)on)
                 : "memory");
}

// 64 consecutive entries of a run, two per lane, and x's values for them.
struct Round {
    int2 ent[2];
    float xs[2];
};

// The entries of up to 32 lists (lane l: cnt entries from post[st] on, x's value xv) as one
// run, taken 32 consecutive entries per step whichever lists they belong to, two steps per round,
// the next round's loads in flight while a round is added, so that short lists leave no lanes
// idle. The lists of the first ncl lanes may create candidates (their slots go to the list, n its
// length; slots past its end are counted only); those of the others only add where A is already
// non-zero, and are left out while there is no candidate.
__device__ __forceinline__ void walk(const Tile &T, const int2 *__restrict__ post, const WinCtx &C, const int ncl,
                                     const uint32_t st, const int cnt, const float xv, const int lane, int &n,
                                     uint32_t &visits, Totals &tot) {
    const unsigned nonempty = __ballot_sync(0xffffffffu, cnt > 0);
    if (!nonempty) return;
    const unsigned lt_mask = (1u << lane) - 1u, le_mask = 2u * lt_mask + 1u;
    int total;
    int pre = warp_excl_scan_int(cnt, lane, &total);
    // entries before the first updating list
    const int cend = ncl >= 32 ? total : __shfl_sync(0xffffffffu, pre, ncl);
    __syncwarp();  // (the previous run's readers are done)
    if (cnt > 0)   // x's value scaled by 2^30 (exact)
        T.seg[__popc(nonempty & lt_mask)] = make_int2((int)(st - (uint32_t)pre), __float_as_int(xv * 1073741824.f));
    else
        pre = 0x7fffffff;  // begins in no step
    if (lane == 0) tot.v[5] += (unsigned long long)total;
    __syncwarp();
    const uint32_t abase = (uint32_t)__cvta_generic_to_shared(T.A) - 4u * (uint32_t)C.w0;  // slot of id 0
    const uint32_t lbase = (uint32_t)__cvta_generic_to_shared(T.list);
    int kb = -1;       // the list that holds the entry before the next step to load
    int lb = lane;     // this lane's place in that step
    int lpre = pre;    // pre minus the step's first place
    auto load = [&](Round &R) {
#pragma unroll
        for (int u = 0; u < 2; u++) {
            // the lists that begin in this step, a bit at their place
            const unsigned starts = __reduce_or_sync(0xffffffffu, shl_clamped(1u, (uint32_t)lpre));
            const int2 sg = T.seg[kb + __popc(starts & le_mask)];
            kb += __popc(starts);
            R.xs[u] = __int_as_float(sg.y);
            ldg_if(lb < total, post + (uint32_t)(sg.x + lb), R.ent[u]);
            lb += 32;
            lpre -= 32;
        }
    };
    auto add = [&](const Round &R, const int base) {
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int b = base + 32 * u, p = b + lane;
            const int id = R.ent[u].x & C.idmask;
            const bool ok = p < total && (uint32_t)R.ent[u].x >= C.smin_tag && id >= C.first;
            const uint32_t a = abase + 4u * (uint32_t)id;
            visits += (uint32_t)ok;  // an entry Alg. 2 visits: y after x, |y| >= minsize
            // rounded up, and at least one unit (the smallest addend keeps a tiny product from 0)
            const uint32_t q = __float2uint_ru(fmaf(R.xs[u], __int_as_float(R.ent[u].y), 1e-30f));
            if (b < cend) {
                const uint32_t old = atoms_add_if(ok && p < cend, a, q);
                const unsigned fresh = __ballot_sync(0xffffffffu, old == 0u);
                const int at = n + __popc(fresh & lt_mask);
                sts16_if(old == 0u && at < JOIN_LCAP, lbase + 2u * (uint32_t)at, (uint32_t)(id - C.w0));
                n += __popc(fresh);
                if (b + 32 >= cend) __syncwarp();  // creations land before updates
            }
            if (b + 32 > cend) {
                const uint32_t v = lds_if(ok && p >= cend, a);
                reds_add_if(v != 0u, a, q);
            }
        }
    };
    // one copy of the code for each: a join of a few thousand vectors runs it about once per warp,
    // and its time is then the instruction fetches
    Round R, N;
    N.ent[0] = N.ent[1] = make_int2(0, 0);
#pragma unroll 1
    for (int base = -64; base < total; base += 64) {
        if (base >= 0 && base >= cend && n == 0) break;
        R = N;
        if (base + 64 < total) load(N);
        if (base >= 0) add(R, base);
    }
}

// x * y in the units of A, to the nearest. dot(x, y') is summed in them like the entries of the
// lists, so that a score is rounded to float32 once, wherever y's prefix ends.
__device__ __forceinline__ uint32_t fixed_product(const float x, const float y) {
    return __float2uint_rn(x * 1073741824.f * y);
}

// One class of windowed items with tile shape G: every warp takes units (a vector, or one
// part of a heavy vector's windows) from the class's work list until it is empty.
template <bool QMODE, bool SPLIT, bool COARSE, bool NOUPPER>
__device__ __forceinline__ void join_class(const JoinParams &P, const int G, const int64_t item_begin,
                                           const int64_t item_end, const int64_t heavy, unsigned long long *const work,
                                           const bool f_minsize, const bool f_remscore, const bool f_upper,
                                           Stager &S, Totals &tot) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp >= tile_warps(G)) return;
    const int W = tile_window(G);
    const unsigned lt_mask = (1u << lane) - 1u;
    Tile T;
    T.A = reinterpret_cast<uint32_t *>(smem + (size_t)warp * tile_bytes(G));
    T.bm = T.A + W;
    T.px = reinterpret_cast<float *>(T.bm + W / 32);
    T.wait = reinterpret_cast<int4 *>(T.px + 64);
    T.seg = reinterpret_cast<int2 *>(T.wait + 32);
    T.xr = T.seg + 32;
    T.list = reinterpret_cast<uint16_t *>(T.xr + JOIN_XCAP);
#pragma unroll 1
    for (int i = lane; i < W + W / 32; i += 32) T.A[i] = 0u;
    __syncwarp();
    const uint32_t parts = (uint32_t)P.parts, ncut = (uint32_t)heavy * parts;
    const uint32_t nunits = (uint32_t)(item_end - item_begin) + (uint32_t)heavy * (parts - 1u);
    auto item_of = [&](const uint32_t unit) -> int64_t {
        return item_begin + (unit < ncut ? unit / parts : unit - (uint32_t)heavy * (parts - 1u));
    };
    // A warp's first two units are its own, dealt over the SMs; the others are asked for two ahead
    // and their work items read one ahead (lane 0). A small join thus runs without one atomic.
    const uint32_t nwarps = gridDim.x * (uint32_t)tile_warps(G);
    uint32_t u0 = blockIdx.x + gridDim.x * (uint32_t)warp, u1 = u0 + nwarps, x0 = 0;
    if (lane == 0 && u0 < nunits) x0 = QMODE ? (uint32_t)item_of(u0) : (uint32_t)P.items[item_of(u0)];
    for (;;) {
        const uint32_t unit = __shfl_sync(0xffffffffu, u0, 0);
        if (unit >= nunits) break;
        // x: a vector of the set (self-join: candidates are the later ids of its instance)
        // or an external query (all indexed vectors are candidates)
        const uint32_t x = __shfl_sync(0xffffffffu, x0, 0);
        if (lane == 0) {
            u0 = u1;
            if (u0 < nunits) {
                u1 = (uint32_t)min(atomicAdd(work, 1ull) + 2ull * nwarps, 0xffffffffull);
                x0 = QMODE ? (uint32_t)item_of(u0) : (uint32_t)P.items[item_of(u0)];
            }
        }
        const int blk = (SPLIT && P.iblk) ? (int)P.iblk[item_of(unit)] : -1;
        const InstDesc &I = P.inst[QMODE || P.one ? 0 : P.vinst[x]];
        const bool in_block = SPLIT && blk >= 0;
        const int4 xm = QMODE ? P.qvmeta[x] : (in_block ? P.vmeta_b : P.vmeta)[x];
        const uint32_t vbase = (uint32_t)I.vbase;
        const int32_t lx = QMODE ? -1 : (int32_t)(x - vbase);
        const int2 *xrow = (QMODE ? P.qcrow : P.crow) + (uint32_t)xm.x;
        const int32_t xl = xm.y;
        const int32_t qs = f_remscore ? xm.z : 0;
        const float mwx = __int_as_float(xm.w);
        const float t = QMODE ? P.qt : I.t;
        const float beta = fmaxf(1e-5f, (float)(xl + 2) * 1.1920929e-7f);  // (|x|+2) * 2^-23
        if (qs >= xl) continue;  // no component may create: x has no candidate at all
        // the windows of this unit: its share of those from x's successor on
        const int nw = I.nw, IW = I.W, In = I.n;
        int wfirst = 0;
        if (!QMODE && nw > 1) wfirst = (lx + 1) / IW;
        const uint32_t *const wp0 = (in_block ? P.wptr_b : P.wptr) + I.wbase;
        const int64_t *const lptr = in_block ? P.lptr_b : P.lptr;
        const int2 *const post = in_block ? P.post_b : P.post;
        const int32_t rbase = I.rbase;
        int wa = wfirst, wz = nw;
        uint32_t part = 0;
        if (unit < ncut && parts > 1u) {  // (nw * parts stays below 2^32: both are at most 2^31 / 1536, or small)
            part = unit % parts;
            wa = wfirst + (int)((uint32_t)(nw - wfirst) * (uint64_t)part / parts);
            wz = wfirst + (int)((uint32_t)(nw - wfirst) * (uint64_t)(part + 1u) / parts);
        }
        if (wa >= wz) continue;
        // A block item walks its share of x's creating components (every nblk-th, from its
        // block index on) and all of x's updating ones, which only add to candidates its
        // own creating components made.
        const int cstr = blk < 0 ? 1 : P.nblk, coff = blk < 0 ? 0 : blk;
        const int ncreate = blk < 0 ? xl - qs : (xl - qs > blk ? (xl - qs - blk + P.nblk - 1) / P.nblk : 0);
        if (ncreate == 0) continue;
        WinCtx C;
        // minsize: a match y needs |y| >= t / maxweight(x) (a margin of 1e-5 for rounding, over
        // the 1e-3 norm tolerances, so the bound can only come out below its exact value and
        // never prunes a match); the size class byte of each entry is compared with it
        int smin = 0;
        if (f_minsize && I.packed && mwx > 0.f)
            smin = (int)ceilf(fminf(__fdividef(t - beta, mwx) * 0.99799f, 255.f));
        C.smin_tag = (uint32_t)max(smin, 0) << 24;
        C.idmask = I.packed ? 0x00ffffff : 0x7fffffff;
        C.first = lx + 1;
        // x's norms up to each rank bucket, rounded up
        {
            uint32_t *pu = reinterpret_cast<uint32_t *>(T.px);
            pu[lane] = pu[lane + 32] = 0u;
            __syncwarp();
#pragma unroll 1
            for (int c = lane; c < xl; c += 32) {
                const int2 e = __ldg(xrow + c);
                const float v = __int_as_float(e.y);
                atomicAdd(&pu[rank_bucket(e.x)], __float2uint_ru(__fmul_ru(__fmul_ru(v, v), 1073741824.f)));
            }
            __syncwarp();
            const uint32_t p0 = pu[2 * lane], p1 = pu[2 * lane + 1];
            int sum;
            const uint32_t ex = (uint32_t)warp_excl_scan_int((int)(p0 + p1), lane, &sum);
            __syncwarp();
            // (the approximate square root is good to a few units in the last place)
            const float s0 = __uint2float_ru(ex + p0) * 9.31322574615478515625e-10f;
            const float s1 = __uint2float_ru(ex + p0 + p1) * 9.31322574615478515625e-10f;
            T.px[2 * lane] = s0 > 0.f ? s0 * rsqrtf(s0) * 1.00001f : 0.f;
            T.px[2 * lane + 1] = s1 > 0.f ? s1 * rsqrtf(s1) * 1.00001f : 0.f;
        }
        // A candidate is worth verifying when A[y] + ||x before y's lists|| * ||y'|| exceeds
        // t - beta. A block item keeps y by Lemma 1 (local pruning): a match scores
        // A + dot(x, y') >= t, the blocks that created y hold all of A between them, so one
        // of them has A_b >= (t - dot(x, y')) / nblk.
        const float scale = (SPLIT && blk >= 0 ? (float)P.nblk : 1.f) * 9.31322574615478515625e-10f * 1.000001f;
        const float floor_ = f_upper || blk >= 0 ? t - beta : -1.f;
        // x's row in shared memory where it fits (verification searches it)
        const int2 *xs = xrow;
        if (xl <= JOIN_XCAP || NOUPPER) {  // (NOUPPER: of a long row, the first components)
#pragma unroll 1
            for (int c = lane; c < min(xl, JOIN_XCAP); c += 32) T.xr[c] = __ldg(xrow + c);
            if (xl <= JOIN_XCAP) xs = T.xr;
            __syncwarp();
        }
        // x's first component from `at` on whose rank is at least r, and a component. Without the upper
        // bounds every candidate's prefix is looked up, and prefixes hold low ranks: the first components
        // of a long row are in shared memory then (the paper's all-pairs-1 on the 200k power-law set: 284
        // ms, 469 with long rows searched in global memory and empty prefixes verified).
        auto x_find = [&](int at, const int r) -> int {
            if (!NOUPPER) return row_find(xs, at, xl, r);
            if (at < JOIN_XCAP) at = row_find(T.xr, at, min(xl, JOIN_XCAP), r);
            return at < JOIN_XCAP ? at : row_find(xrow, at, xl, r);
        };
        auto x_comp = [&](const int at) -> int2 {
            return !NOUPPER ? xs[at] : at < JOIN_XCAP ? T.xr[at] : __ldg(xrow + at);
        };
        auto x_value = [&](const int r) -> float {
            if (!NOUPPER) return x_at(r, xs, xl);
            const int at = x_find(0, r);
            const int2 e = at < xl ? x_comp(at) : make_int2(-1, 0);
            return e.x == r ? __int_as_float(e.y) : 0.f;
        };
        // The lists of a short x stay in registers over the windows (a lane each, the creating
        // ones first), and so do their positions: a window's lists end where the next one's
        // begin, so each window loads one position per list, for the window after it.
        const bool shortx = ncreate + qs <= 32;
        auto list_at = [&](const int r, const int w) -> uint32_t {
            return nw > 1 ? __ldg(wp0 + (int64_t)r * (nw + 1) + w) : (uint32_t)__ldg(lptr + (rbase + r + w));
        };
        auto range_at = [&](const int r, const int w, uint32_t &s0, uint32_t &s1) {  // COARSE
            return list_range(in_block ? P.wlist_b : P.wlist, in_block ? P.wptr_b : P.wptr, lptr, post, (int64_t)rbase + r,
                              w, nw, IW, C.idmask, s0, s1);
        };
        int2 e0 = make_int2(0, 0);
        uint32_t p0 = 0, p1 = 0;
        // COARSE: a list with every window's start is read like the table; of another one, which holds
        // an entry in few windows, the id at p1 says whether there is anything to look for
        const uint32_t *starts = nullptr;
        uint32_t pend = 0, nextid = 0xffffffffu;
        auto id_at = [&](const uint32_t q) { return q < pend ? (uint32_t)(__ldg(&post[q].x) & C.idmask) : 0xffffffffu; };
        if (shortx && lane < ncreate + qs) {
            e0 = xs[lane < ncreate ? qs + coff + lane * cstr : lane - ncreate];
            if (COARSE) {
                starts = range_at(e0.x, wa, p0, p1);
                if (!starts) {
                    pend = (uint32_t)__ldg(lptr + (rbase + e0.x + 1));
                    nextid = id_at(p1);
                }
            } else {
                p0 = list_at(e0.x, wa);
                p1 = list_at(e0.x, wa + 1);
            }
        }
        uint32_t visits = 0;
#pragma unroll 1
        for (int w = wa; w < wz; w++) {
            const int w0 = w * IW;
            const int wn = min(IW, In - w0);
            C.w0 = w0;
            int n = 0;  // candidates
            // A short x: one walk, its creating lists first. A long one: create, then update (only
            // where there are candidates); the non-empty lists of the window are gathered over
            // blocks of 32 components and walked 32 at a time, because most lists of a long
            // vector have no entry in a given window.
            uint32_t p2 = p1;  // the next window's list ends
            if (shortx && w + 1 < wz && lane < ncreate + qs) {
                if (!COARSE) {
                    p2 = list_at(e0.x, w + 2);
                } else if (starts) {
                    p2 = __ldg(starts + w + 2);
                } else if (const uint32_t bound = (uint32_t)(w + 2) * (uint32_t)IW; nextid < bound) {
                    p2 = p1 + 1u;
                    nextid = id_at(p2);
                    if (nextid < bound) {
                        p2 = first_at(post, p2 + 1u, pend, bound, C.idmask);
                        nextid = id_at(p2);
                    }
                }
            }
            uint32_t st = p0;
            int cnt = (int)(p1 - p0), k0 = 0;
            float xv = __int_as_float(e0.y);
            for (int ph = 0;;) {
                if (!shortx) {
                    const bool create = ph == 0;
                    const int count = create ? ncreate : qs;
                    int qn = 0;  // lists gathered
#pragma unroll 1
                    for (; k0 < count; k0 += 32) {
                        int2 e = make_int2(0, 0);
                        uint32_t s0 = 0, s1 = 0;
                        if (k0 + lane < count) {
                            e = xs[create ? qs + coff + (k0 + lane) * cstr : k0 + lane];
                            if (COARSE) {
                                range_at(e.x, w, s0, s1);
                            } else {
                                s0 = list_at(e.x, w);
                                s1 = list_at(e.x, w + 1);
                            }
                        }
                        const unsigned have = __ballot_sync(0xffffffffu, s1 > s0);
                        if (qn + __popc(have) > 32) break;  // no room: this block again, after the walk
                        if (s1 > s0) T.wait[qn + __popc(have & lt_mask)] = make_int4((int)s0, (int)(s1 - s0), e.y, 0);
                        qn += __popc(have);
                    }
                    __syncwarp();
                    const int4 g = lane < qn ? T.wait[lane] : make_int4(0, 0, 0, 0);
                    st = (uint32_t)g.x;
                    cnt = g.y;
                    xv = __int_as_float(g.z);
                }
                walk(T, post, C, shortx ? ncreate : ph == 0 ? 32 : 0, st, cnt, xv, lane, n, visits, tot);
                __syncwarp();
                if (shortx) break;
                if (k0 >= (ph == 0 ? ncreate : qs)) {
                    if (ph == 1 || n == 0) break;
                    ph = 1;
                    k0 = 0;
                }
            }
            p0 = p1;
            p1 = p2;
            if (n == 0) continue;  // no candidate in this window
            __syncwarp();
            // ---------------- filter and verify: the candidate list at once, or, when it ran
            // over, the slots of the window in stretches of JOIN_LCAP
            const uint8_t *codes = (in_block ? P.code_b : P.code) + (vbase + (uint32_t)w0);
            const int4 *cands = (in_block ? P.vcand_b : P.vcand) + (vbase + (uint32_t)w0);
            const bool over = n > JOIN_LCAP;
            if (lane == 0) tot.v[1] += (unsigned long long)n;
            int nm = 0;  // matches
            for (int s0 = 0; s0 < (over ? wn : 1); s0 += JOIN_LCAP) {
                if (over) {
                    n = 0;
#pragma unroll 1
                    for (int q = s0; q < min(s0 + JOIN_LCAP, wn); q += 32) {
                        const bool on = q + lane < wn && T.A[q + lane] != 0u;
                        const unsigned bal = __ballot_sync(0xffffffffu, on);
                        if (on) T.list[n + __popc(bal & lt_mask)] = (uint16_t)(q + lane);
                        n += __popc(bal);
                    }
                    __syncwarp();
                }
                int ns = 0;
#pragma unroll 1
                for (int b = 0; b < n; b += 128) {  // four codes per lane in flight
                    int slot[4], code[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        slot[u] = -1;
                        code[u] = 0;
                        if (b + 32 * u + lane < n) {
                            slot[u] = T.list[b + 32 * u + lane];
                            code[u] = __ldg(codes + slot[u]);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        bool keep = false;
                        if (slot[u] >= 0) {
                            const float pn = (float)(code[u] & 15) * (PN4_STEP * 1.0001f);
                            // (no prefix: A is the whole score)
                            keep = fmaf(__uint2float_ru(T.A[slot[u]]), scale, T.px[(code[u] >> 4) * 4 + 3] * pn) >
                                   (NOUPPER && (code[u] & 15) == 0 ? t - beta : floor_);
                            if (!keep) T.A[slot[u]] = 0u;
                        }
                        const unsigned bal = __ballot_sync(0xffffffffu, keep);
                        if (keep) T.list[ns + __popc(bal & lt_mask)] = (uint16_t)slot[u];  // (already read)
                        ns += __popc(bal);
                    }
                    __syncwarp();
                }
#pragma unroll 1
                for (int b = 0; b < ns; b += 32) {
                    bool emit = false;
                    float sc = 0.f;
                    uint32_t sum = 0u;  // the score so far, in the units of A
                    int slot = 0;
                    int4 yc = make_int4(0, 0, 0, 0);  // {row offset, |y'|, first rank after y', ||y'||_2 bound}
                    // 0: rejected or emitted, 1: score known, 2: short dot(x, y') left, 3: long one
                    int stage = 0;
                    if (b + lane < ns) {
                        slot = T.list[b + lane];
                        sum = T.A[slot];
                        const float v = __uint2float_rn(sum) * 9.31322574615478515625e-10f;  // 2^-30
                        yc = __ldg(cands + slot);
                        if (SPLIT && blk >= 0) {  // a partial sum: y scored whole, in float64
                            stage = 4;
                        } else if (!f_upper || v + T.px[rank_bucket(yc.z)] * __int_as_float(yc.w) * 1.00001f > t - beta) {
                            stage = yc.y == 0 ? 1 : (yc.y <= 16 ? 2 : 3);
                            // The paper's upperbound. On the 200k power-law set it stops 4% of what gets
                            // here, at no cost to be seen; a batch of 4096 queries takes 2% longer with
                            // it (6.64 ms in the kernel without, 6.78 with), so queries go without.
                            if (!QMODE && f_upper && stage > 1) {
                                const float l1 = (float)min(yc.y, xl) * mwx;
                                // (maxweight(y') >= ||y'|| / sqrt(|y'|): not loaded where that is enough)
                                if (v + l1 * __int_as_float(yc.w) * rsqrtf((float)yc.y) * 0.998f < t - beta &&
                                    v + l1 * __ldg(P.mwj + (vbase + (uint32_t)(w0 + slot))) < t - beta)
                                    stage = 0;
                            }
                        }
                    }
                    {
                        const unsigned dots = __ballot_sync(0xffffffffu, stage == 2 || stage == 3);
                        if (lane == 0 && dots) tot.v[2] += (unsigned long long)__popc(dots);
                    }
                    if (stage == 2) {  // short prefixes: each lane its own candidate
                        const int2 *yr = P.crow + (uint32_t)yc.x;
                        int at = 0;  // both rows in rank order: x is searched from the last place on
#pragma unroll 1
                        for (int k = 0; k < yc.y && at < xl; k++) {
                            const int2 e = __ldg(yr + k);
                            at = x_find(at, e.x);
                            if (at < xl) {
                                const int2 xe = x_comp(at);
                                if (xe.x == e.x) sum += fixed_product(__int_as_float(xe.y), __int_as_float(e.y));
                            }
                        }
                        stage = 1;
                    }
                    // long prefixes: the whole warp takes one candidate at a time, its lanes
                    // reading y's prefix entries side by side
                    for (unsigned lm = __ballot_sync(0xffffffffu, stage == 3); lm; lm &= lm - 1u) {
                        const int src = __ffs(lm) - 1;
                        const uint32_t yo = (uint32_t)__shfl_sync(0xffffffffu, yc.x, src);
                        const int yl = __shfl_sync(0xffffffffu, yc.y, src);
                        uint32_t acc = 0u;
#pragma unroll 1
                        for (int k = lane; k < yl; k += 32) {
                            const int2 e = __ldg(&P.crow[yo + k]);
                            acc += fixed_product(x_value(e.x), __int_as_float(e.y));
                        }
                        acc = __reduce_add_sync(0xffffffffu, acc);
                        if (lane == src) {
                            sum += acc;
                            stage = 1;
                        }
                    }
                    if (stage == 1) {
                        sc = __uint2float_rn(sum) * 9.31322574615478515625e-10f;
                        if (sc >= t + beta) {
                            emit = true;
                            stage = 0;
                        } else if (sc <= t - beta) {
                            stage = 0;
                        }
                    }
                    if (stage == 4) stage = 1;
                    // inside the band: float64 dot(x, y) over all of y, one candidate at a
                    // time across the warp (exact products)
                    int yfull = 0;
                    if (stage == 1) yfull = __ldg(&P.vmeta[vbase + (uint32_t)(w0 + slot)]).y;
                    for (unsigned lm = __ballot_sync(0xffffffffu, stage == 1); lm; lm &= lm - 1u) {
                        const int src = __ffs(lm) - 1;
                        const uint32_t yo = (uint32_t)__shfl_sync(0xffffffffu, yc.x, src);
                        const int yl = __shfl_sync(0xffffffffu, yfull, src);
                        double acc = 0.0;
#pragma unroll 1
                        for (int k = lane; k < yl; k += 32) {
                            const int2 e = __ldg(&P.crow[yo + k]);
                            acc += (double)x_value(e.x) * (double)__int_as_float(e.y);
                        }
#pragma unroll
                        for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                        if (lane == 0) tot.v[4]++;
                        if (lane == src) {
                            emit = acc >= (double)t;
                            sc = (float)acc;
                        }
                    }
                    const unsigned bal = __ballot_sync(0xffffffffu, emit);
                    if (SPLIT && blk >= 0) {  // block items: pairs to the global list, merged after the join
                        unsigned long long g = 0;
                        if (lane == 0 && bal) g = atomicAdd(P.sp_count, (unsigned long long)__popc(bal));
                        g = __shfl_sync(0xffffffffu, g, 0) + (unsigned long long)__popc(bal & lt_mask);
                        if (emit && g < (unsigned long long)P.sp_cap) {
                            P.sp_key[g] = (unsigned long long)lx * (unsigned long long)In + (unsigned long long)(w0 + slot);
                            P.sp_score[g] = __float_as_uint(sc);
                        }
                        emit = false;
                    } else {
                        nm += __popc(bal);
                    }
                    if (b + lane < ns) {
                        T.A[slot] = emit ? __float_as_uint(sc) : 0u;
                        if (emit) atomicOr(&T.bm[slot >> 5], 1u << (slot & 31));
                    }
                }
                __syncwarp();
            }
            if (nm == 0) continue;
            // ---------------- emit the window's matches in id order
            if (lane == 0) {
                stage_take(S, P, (uint32_t)nm);
                tot.v[3] += (unsigned long long)nm;
            }
            __syncwarp();
            uint32_t at = 0;
#pragma unroll 1
            for (int q = lane; q - lane < (wn + 31) >> 5; q += 32) {
                uint32_t word = 0u;
                if (q < (wn + 31) >> 5) {
                    word = T.bm[q];
                    if (word) T.bm[q] = 0u;
                }
                int sum;
                uint32_t p = at + (uint32_t)warp_excl_scan_int(__popc(word), lane, &sum);
                at += (uint32_t)sum;
#pragma unroll 1
                for (; word; word &= word - 1u) {
                    const int slot = (q << 5) + __ffs(word) - 1;
                    stage_put(P, S, p++, make_int2(w0 + slot, (int)T.A[slot]));
                    T.A[slot] = 0u;
                }
            }
            __syncwarp();
        }
        if (lane == 0) stage_close(S, P, (int64_t)x * parts + part, QMODE ? (int32_t)x : lx);
        count_add(tot, 0, visits, lane);
        __syncwarp();
    }
}

// QMODE: external queries against the index; SPLIT: a self-join whose work list may hold
// dimension-block items (P.iblk); COARSE: window starts by list; NOUPPER: a self-join
// without the upper bounds (the others read the flag). Each is
// compiled separately, so that the plain self-join
// carries none of the other paths' state.
template <bool QMODE, bool SPLIT, bool COARSE, bool NOUPPER>
__global__ void __launch_bounds__(JOIN_THREADS, 1) join_kernel(const __grid_constant__ JoinParams P) {
    const bool f_minsize = !(P.flags & APS_NO_MINSIZE);
    const bool f_remscore = !(P.flags & APS_NO_REMSCORE);
    const bool f_upper = !NOUPPER && !(P.flags & APS_NO_UPPERBOUND);
    __shared__ Stager stagers[JOIN_WARPS];
    __shared__ Totals totals[JOIN_WARPS];
    const int warp = threadIdx.x >> 5;
    Stager &S = stagers[warp];
    Totals &tot = totals[warp];
    if ((threadIdx.x & 31) == 0) {
        memset(&tot, 0, sizeof(tot));
        memset(&S, 0, sizeof(S));
        S.piece = -1;
    }
    __syncwarp();
    // A warp that finds a class's work list empty waits for the CTA's other warps before the
    // next class's tiles take their place in shared memory: the classes share one launch and
    // one tail. (The streamed class needs no tile.)
    for (int cls = 0; cls < P.ncls; cls++) {
        const int64_t item_begin = P.cls_begin[cls], item_end = P.cls_begin[cls + 1];
        if (item_end <= item_begin) continue;
        const int G = P.cls_G[cls];
        unsigned long long *const work = P.work + cls;
        if (!QMODE && G == 0) {  // short vectors: one warp each
            stream_short<COARSE>(P, work, item_begin, item_end, f_minsize, f_remscore, tot, S);
            continue;
        }
        join_class<QMODE, SPLIT, COARSE, NOUPPER>(P, G, item_begin, item_end, P.cls_heavy[cls], work, f_minsize, f_remscore, f_upper, S,
                                 tot);
        bool later = false;  // another windowed class
        for (int c = cls + 1; c < P.ncls; c++) later = later || (P.cls_G[c] > 0 && P.cls_begin[c + 1] > P.cls_begin[c]);
        if (later) __syncthreads();
    }
    __syncwarp();
    // the warps' totals, one global atomic per counter and warp
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int k = 0; k < 6; k++)
            if (tot.v[k]) atomicAdd(&P.counters[k < 5 ? k : 6], tot.v[k]);
    }
}

// One warp per slot: copy its staged run, piece by piece, to the output at scan(counts)[slot].
__global__ void k_gather(const Segment *__restrict__ segs, const int2 *__restrict__ chain, int64_t slab,
                         const int32_t *__restrict__ cntq, int64_t nslots, const int2 *__restrict__ stage,
                         const int64_t *__restrict__ off, int32_t *__restrict__ oi, int32_t *__restrict__ oj,
                         float *__restrict__ os) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t q = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); q < nslots; q += nwarps) {
        if (cntq[q] == 0) continue;
        const Segment S = segs[q];
        int64_t dst = off[q], src = S.src;
        int cnt = S.cnt, next = S.next;
        for (;;) {
            for (int e = lane; e < cnt; e += 32) {
                const int2 v = stage[src + e];
                oi[dst + e] = S.i;
                oj[dst + e] = v.x;
                os[dst + e] = __int_as_float(v.y);
            }
            if (next < 0) break;
            dst += cnt;
            src = (int64_t)next * slab;
            const int2 c = chain[next];
            cnt = c.x;
            next = c.y;
        }
    }
}

__global__ void k_inst_offsets(const InstDesc *__restrict__ inst, int k, const int64_t *__restrict__ off, int parts,
                               int64_t nslots, int64_t *out) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= k; i += gridDim.x * blockDim.x)
        out[i] = i < k ? off[inst[i].vbase * parts] : off[nslots];
}

// The heaviest vectors of a class whose windows are cut into parts: enough units for every warp
// of the chip several times over. (Join ms with 1024 / 2048 / 8192 / 32768 of them: 30,000 power-law
// rows 2.8 / 2.27 / 1.75 / 1.65, 200,000 rows 22.3 / 21.55 / 21.6 / 21.75, 96 instances 1.92 / 1.92 /
// 1.96 / 2.09.)
constexpr int64_t JOIN_HEAVY = 8192;

int join_smem() {
    int b = 0;
    for (int G : {1, 2, 4, 8}) b = std::max(b, tile_bytes(G) * tile_warps(G));
    return b;
}

// The index's work-list classes as one launch's class list, the windows of the heaviest
// vectors in `parts` parts. Returns the CTA count (the units spread over the SMs, at most
// max_ctas CTAs).
int set_classes(JoinParams &P, const aps_index *ix, int parts, int max_ctas) {
    static const int Gs[JOIN_NCLS] = {1, 2, 4, 8, 0};
    P.ncls = JOIN_NCLS;
    P.parts = parts;
    int64_t ctas = 1;
    for (int c = 0; c < JOIN_NCLS; c++) {
        P.cls_G[c] = Gs[c];
        P.cls_begin[c] = ix->class_begin[c];
        const int64_t ni = ix->class_begin[c + 1] - ix->class_begin[c];
        P.cls_heavy[c] = Gs[c] > 0 ? std::min(ni, JOIN_HEAVY) : 0;
        ctas = std::max(ctas, ni + P.cls_heavy[c] * (parts - 1));
    }
    P.cls_begin[JOIN_NCLS] = ix->class_begin[JOIN_NCLS];
    return (int)std::min<int64_t>(max_ctas, ctas);
}

// The kernel for an index's self-join (split: with dimension-block items) or for queries of it.
using JoinKernel = void (*)(const JoinParams);
JoinKernel self_kernel(const aps_index *ix, uint32_t flags, bool split = false) {
    const bool by_list = ix->wper >= 0;
    if (split) return by_list ? join_kernel<false, true, true, false> : join_kernel<false, true, false, false>;
    if (by_list) return join_kernel<false, false, true, false>;
    return flags & APS_NO_UPPERBOUND ? join_kernel<false, false, false, true> : join_kernel<false, false, false, false>;
}
JoinKernel query_kernel(const aps_index *ix) {
    return ix->wper >= 0 ? join_kernel<true, false, true, false> : join_kernel<true, false, false, false>;
}
aps_status allow_smem(JoinKernel k) {  // (the same for every index: the limit is shared by all threads)
    APS_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, join_smem()));
    return APS_OK;
}

// What every join reads of an index.
void set_index(JoinParams &P, const aps_index *ix) {
    const IndexArrays &d = ix->d;
    memset(&P, 0, sizeof(P));
    P.inst = d.inst.p;
    P.vinst = d.vinst.p;
    P.items = ix->items.p;
    P.one = ix->k == 1;
    P.crow = d.crow.p;
    P.vmeta = d.vmeta.p;
    P.vcand = d.vcand.p;
    P.mwj = ix->l2 ? d.mwj.p : d.mwpre.p;
    P.code = d.code.p;
    P.nblk = 1;
    P.parts = 1;
    P.lptr = d.lptr.p;
    P.wptr = d.wptr.p;
    P.post = d.post.p;
    P.wlist = d.wlist.p;
}

// The join phase: reset the counters and the per-slot pair counts, then the persistent join.
// An index's first join launches the three directly: most indexes are joined once, and capturing,
// instantiating and destroying a graph costs the host some 100 us (a whole join of 2,000 vectors
// takes 600). From the second join on they are a CUDA graph, captured on a private stream, so any
// caller stream works, including the legacy default one, and replayed with the memset targets and
// the kernel's parameters and grid updated in place.
aps_status run_join_graph(aps_index *ix, JoinParams &P, int grid, int smem, unsigned long long *ctr, int32_t *cntq,
                          int64_t nslots, cudaStream_t s) {
    JoinGraph &G = ix->jgraph;
    const size_t ctr_bytes = 16 * sizeof(unsigned long long), cnt_bytes = sizeof(int32_t) * (size_t)nslots;
    const JoinKernel kernel = self_kernel(ix, P.flags);
    APS_TRY(allow_smem(kernel));
    if (G.launches++ == 0) {
        APS_CUDA(cudaMemsetAsync(ctr, 0, ctr_bytes, s));
        APS_CUDA(cudaMemsetAsync(cntq, 0, cnt_bytes, s));
        kernel<<<grid, JOIN_THREADS, smem, s>>>(P);
        APS_LAUNCH_CHECK();
        return APS_OK;
    }
    if (!G.exec) {
        cudaStream_t cs = nullptr;
        APS_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            cudaMemsetAsync(ctr, 0, ctr_bytes, cs);
            cudaMemsetAsync(cntq, 0, cnt_bytes, cs);
            kernel<<<grid, JOIN_THREADS, smem, cs>>>(P);
            cudaGraph_t g = nullptr;
            e = cudaStreamEndCapture(cs, &g);
            G.graph = g;
        }
        cudaStreamDestroy(cs);
        APS_CUDA(e);
        size_t nn = 0;
        APS_CUDA(cudaGraphGetNodes(G.graph, nullptr, &nn));
        std::vector<cudaGraphNode_t> nodes(nn);
        APS_CUDA(cudaGraphGetNodes(G.graph, nodes.data(), &nn));
        for (cudaGraphNode_t nd : nodes) {
            cudaGraphNodeType ty;
            APS_CUDA(cudaGraphNodeGetType(nd, &ty));
            if (ty == cudaGraphNodeTypeKernel) {
                G.join = nd;
            } else if (ty == cudaGraphNodeTypeMemset) {
                cudaMemsetParams mp;
                APS_CUDA(cudaGraphMemsetNodeGetParams(nd, &mp));
                if (mp.dst == ctr) G.reset_ctr = nd;
                if (mp.dst == cntq) G.reset_cnt = nd;
            }
        }
        if (nn != 3 || !G.join || !G.reset_ctr || !G.reset_cnt) {
            set_error("join graph: expected two memset nodes and one kernel node, captured %zu nodes", nn);
            return APS_ECUDA;
        }
        APS_CUDA(cudaGraphInstantiate(&G.exec, G.graph, 0));
    } else {
        cudaMemsetParams mp;
        APS_CUDA(cudaGraphMemsetNodeGetParams(G.reset_ctr, &mp));
        mp.dst = ctr;
        APS_CUDA(cudaGraphExecMemsetNodeSetParams(G.exec, G.reset_ctr, &mp));
        APS_CUDA(cudaGraphMemsetNodeGetParams(G.reset_cnt, &mp));
        mp.dst = cntq;
        APS_CUDA(cudaGraphExecMemsetNodeSetParams(G.exec, G.reset_cnt, &mp));
        void *args[1] = {&P};
        cudaKernelNodeParams kp;
        memset(&kp, 0, sizeof(kp));
        kp.func = reinterpret_cast<void *>(kernel);
        kp.gridDim = dim3((unsigned)grid);
        kp.blockDim = dim3(JOIN_THREADS);
        kp.sharedMemBytes = (unsigned)smem;
        kp.kernelParams = args;
        APS_CUDA(cudaGraphExecKernelNodeSetParams(G.exec, G.join, &kp));
    }
    APS_CUDA(cudaGraphLaunch(G.exec, s));
    count_launch();
    return APS_OK;
}

}  // namespace

namespace {

// The work list of a split join: the first `heavy` items of the list (the costliest
// vectors) become nblk block items each, the rest stay whole.
__global__ void k_split_items(const int32_t *__restrict__ items, int64_t nitems, int64_t heavy, int nblk,
                              int32_t *out, int8_t *blk) {
    const int64_t total = nitems + heavy * (nblk - 1);
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total; k += (int64_t)gridDim.x * blockDim.x) {
        if (k < heavy * nblk) {
            out[k] = items[k / nblk];
            blk[k] = (int8_t)(k % nblk);
        } else {
            out[k] = items[k - heavy * (nblk - 1)];
            blk[k] = -1;
        }
    }
}

// First occurrence of each key in a sorted list (the block items of one vector may find a
// pair twice, with the same score).
__global__ void k_first_of_key(const unsigned long long *__restrict__ key, int64_t n, int32_t *flag) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        flag[k] = (k == 0 || key[k] != key[k - 1]) ? 1 : 0;
}

// The split vectors' pairs (key = local x * n + local y, sorted, first occurrences at
// off[k]) into the staging buffer from `base` on, as the runs of their vectors' slots.
__global__ void k_split_place(const unsigned long long *__restrict__ key, const uint32_t *__restrict__ score,
                              const int32_t *__restrict__ flag, const int64_t *__restrict__ off, int64_t n,
                              const InstDesc *__restrict__ inst, int parts, int64_t base, int2 *stage,
                              Segment *segs, int32_t *cntq) {
    const InstDesc I = inst[0];
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        if (!flag[k]) continue;
        const unsigned long long kk = key[k];
        const int32_t lx = (int32_t)(kk / (unsigned long long)I.n), y = (int32_t)(kk % (unsigned long long)I.n);
        const int64_t qw = (I.vbase + lx) * parts;  // (a split vector has no run of its own in any part)
        const int64_t pos = base + off[k];
        stage[pos] = make_int2(y, (int)score[k]);
        atomicAdd(&cntq[qw], 1);
        bool first = k == 0;
        if (!first) {
            const unsigned long long pk = key[k - 1];
            first = (int32_t)(pk / (unsigned long long)I.n) != lx;
        }
        if (first) {
            Segment S;
            S.src = pos;
            S.cnt = 0;  // (the count is cntq's: k_split_counts)
            S.i = lx;
            S.next = -1;
            S._pad = 0;
            segs[qw] = S;
        }
    }
}

// The split vectors' piece lengths, once every pair is counted: a vector with no run of its
// own (it was joined by blocks) has its whole count in its one piece.
__global__ void k_split_counts(const unsigned long long *__restrict__ key, const int32_t *__restrict__ flag, int64_t n,
                               const InstDesc *__restrict__ inst, int parts, const int32_t *__restrict__ cntq, Segment *segs) {
    const InstDesc I = inst[0];
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t lx = (int64_t)(key[k] / (unsigned long long)I.n);
        if (k == 0 || (int64_t)(key[k - 1] / (unsigned long long)I.n) != lx)
            segs[(I.vbase + lx) * parts].cnt = cntq[(I.vbase + lx) * parts];
    }
}

}  // namespace

// Staging slots one CTA can reserve and leave unused: less than a slab per warp.
int64_t join_slab_slack() { return (int64_t)JOIN_WARPS * JOIN_STAGE_SLAB; }

void debug_stage_cap(int64_t pairs) { g_stage_cap_once.store(pairs > 0 ? pairs : 0); }

aps_status join_all_pairs(aps_index *ix, uint32_t flags, aps_pairs *out, std::vector<int64_t> *pair_offsets_h,
                          int nblk, int64_t heavy) {
    cudaStream_t s = ix->stream;
    IndexArrays &d = ix->d;
    const int sms = num_sms();
    cudaEvent_t ev[4];
    for (int i = 0; i < 4; i++) APS_CUDA(cudaEventCreate(&ev[i]));
    struct EvGuard {
        cudaEvent_t *e;
        ~EvGuard() {
            for (int i = 0; i < 4; i++) cudaEventDestroy(e[i]);
        }
    } evg{ev};
    const int need = join_smem();

    // the vertical split: the costliest `heavy` vectors as nblk dimension blocks each
    const bool split = nblk >= 2 && heavy > 0 && ix->k == 1;
    const int parts = ix->parts;
    const int64_t nslots = ix->N * parts;
    int split_cls = -1;
    int64_t nsplit = 0, sp_cap = 0;
    DBuf<int32_t> items2;
    DBuf<int8_t> iblk;
    DBuf<uint64_t> sp_key;
    DBuf<uint32_t> sp_score;
    BlockIndex bx;
    if (split) {
        // block items come from the windowed classes (G = 1 ... 8), never from the
        // streamed class (one- and two-component vectors) that follows them
        for (int c = 0; c < 4; c++)
            if (ix->class_begin[c + 1] > ix->class_begin[c]) split_cls = c;
        const int64_t nitems = ix->class_begin[JOIN_NCLS] - ix->class_begin[0];
        nsplit = std::min<int64_t>(heavy, ix->class_begin[4] - ix->class_begin[0]);
        if (nsplit > 0) {
            APS_TRY(allow_smem(self_kernel(ix, flags, true)));
            const int64_t total = nitems + nsplit * (nblk - 1);
            APS_TRY(items2.alloc((size_t)total, s));
            APS_TRY(iblk.alloc((size_t)total, s));
            k_split_items<<<grid_for(total, 256), 256, 0, s>>>(ix->items.p, nitems, nsplit, nblk, items2.p, iblk.p);
            APS_LAUNCH_CHECK();
            if (ix->l2) APS_TRY(build_block_index(ix, bx, s));
            sp_cap = std::max<int64_t>((int64_t)1 << 20, nsplit * 4096);
        }
    }

    DBuf<int32_t> cntq;
    DBuf<unsigned long long> ctr;  // 0..4 counters, 5 stage count, 6 entries read, 8..12 work, 13 split pairs
    APS_TRY(cntq.alloc((size_t)std::max<int64_t>(nslots, 1), s));
    APS_TRY(ctr.alloc(16, s));
    // Staging capacity: the index's own hint, else the last join of this process; a join
    // that still overflows is re-run with room for what it reserved plus one slab per
    // warp. First pieces are stored per slot and later ones per slab, so their tables never
    // overflow.
    int64_t stage_cap = std::max<int64_t>({ix->hint_pairs, g_stage_hint.load(), (int64_t)1 << 20, ix->nnz});
    if (ix->hint_pairs == 0 && g_stage_hint.load() == 0) {
        // no join of this process has sized the staging yet: take room for every possible
        // pair plus one slab per warp, but at most an eighth of the free device memory
        // and 2^28 pairs, so that a first join rarely has to run twice
        int64_t most = (int64_t)sms * join_slab_slack();
        for (const InstDesc &I : ix->inst_h) most += (int64_t)I.n * (I.n - 1) / 2;
        size_t fr = 0, tot = 0;
        if (cudaMemGetInfo(&fr, &tot) == cudaSuccess) {
            const int64_t room = std::min<int64_t>({most, (int64_t)(fr / 8 / sizeof(int2)), (int64_t)1 << 28});
            stage_cap = std::max(stage_cap, room);
        } else {
            cudaGetLastError();
        }
    }
    if (const int64_t once = g_stage_cap_once.exchange(0); once > 0) stage_cap = once;
    DBuf<int2> stage;
    DBuf<Segment> segs;
    DBuf<int2> scratch, chain;
    APS_TRY(scratch.alloc((size_t)sms * JOIN_WARPS * JOIN_ECAP, s));
    APS_TRY(segs.alloc((size_t)std::max<int64_t>(nslots, 1), s));
    int64_t total_pairs = 0, reserved = 0;
    unsigned long long ch[16];
    int reruns = 0;
    for (int attempt = 0; attempt < 3; attempt++) {
        APS_TRY(stage.alloc((size_t)stage_cap, s));
        APS_TRY(chain.alloc((size_t)(stage_cap / JOIN_STAGE_SLAB) + 1, s));
        if (nsplit > 0) {
            APS_TRY(sp_key.alloc((size_t)sp_cap, s));
            APS_TRY(sp_score.alloc((size_t)sp_cap, s));
        }
        if (ix->class_begin[JOIN_NCLS] <= ix->class_begin[0]) {  // nothing to join: just the resets
            APS_CUDA(cudaMemsetAsync(ctr.p, 0, 16 * sizeof(unsigned long long), s));
            if (nslots) APS_CUDA(cudaMemsetAsync(cntq.p, 0, sizeof(int32_t) * nslots, s));
            APS_CUDA(cudaEventRecord(ev[0], s));
        } else {
            JoinParams P;
            set_index(P, ix);
            const int grid = set_classes(P, ix, parts, sms);
            P.flags = flags | (ix->flags & (APS_NO_MINSIZE | APS_NO_REMSCORE | APS_NO_UPPERBOUND));
            P.stage = stage.p;
            P.stage_cap = stage_cap;
            P.stage_count = ctr.p + 5;
            P.stage_slab = JOIN_STAGE_SLAB;
            P.segs = segs.p;
            P.chain = chain.p;
            P.cntq = cntq.p;
            P.counters = ctr.p;
            P.work = ctr.p + 8;
            P.scratch = scratch.p;
            P.sp_count = ctr.p + 13;
            APS_CUDA(cudaEventRecord(ev[0], s));
            if (nsplit > 0) {  // the split work list, one direct launch
                P.items = items2.p;
                P.iblk = iblk.p;
                P.nblk = nblk;
                P.vmeta_b = ix->l2 ? bx.vmeta.p : P.vmeta;
                P.vcand_b = ix->l2 ? bx.vcand.p : P.vcand;
                P.code_b = ix->l2 ? bx.code.p : P.code;
                P.lptr_b = ix->l2 ? bx.lptr.p : P.lptr;
                P.wptr_b = ix->l2 ? bx.wptr.p : P.wptr;
                P.wlist_b = ix->l2 ? bx.wlist.p : P.wlist;
                P.post_b = ix->l2 ? bx.post.p : P.post;
                P.sp_key = reinterpret_cast<unsigned long long *>(sp_key.p);
                P.sp_score = sp_score.p;
                P.sp_cap = sp_cap;
                for (int c = split_cls + 1; c <= JOIN_NCLS; c++) P.cls_begin[c] += nsplit * (nblk - 1);
                // block items come first and are cut into parts as heavy vectors are: whole, the
                // longest of them would be one warp's tail (200 vectors in two blocks: 41.2 ms,
                // 23.8 cut)
                P.cls_heavy[split_cls] = std::min(P.cls_begin[split_cls + 1] - P.cls_begin[split_cls],
                                                  std::min(nsplit * nblk, 4 * JOIN_HEAVY) + JOIN_HEAVY);
                APS_CUDA(cudaMemsetAsync(ctr.p, 0, 16 * sizeof(unsigned long long), s));
                APS_CUDA(cudaMemsetAsync(cntq.p, 0, sizeof(int32_t) * std::max<int64_t>(nslots, 1), s));
                self_kernel(ix, flags, true)<<<grid, JOIN_THREADS, need, s>>>(P);
                APS_LAUNCH_CHECK();
            } else {
                APS_TRY(run_join_graph(ix, P, grid, need, ctr.p, cntq.p, nslots, s));
            }
        }
        APS_CUDA(cudaEventRecord(ev[1], s));
        APS_CUDA(cudaMemcpyAsync(ch, ctr.p, sizeof(ch), cudaMemcpyDeviceToHost, s));
        APS_CUDA(cudaStreamSynchronize(s));
        total_pairs = (int64_t)ch[3];
        reserved = (int64_t)ch[5];
        const int64_t sp_found = nsplit > 0 ? (int64_t)ch[13] : 0;
        if (reserved <= stage_cap && sp_found <= sp_cap) {
            if (sp_found > 0) {
                // the split vectors' pairs: sorted by (x, y), first occurrences kept, placed
                // after the join's staged runs as the runs of their slots
                const InstDesc &I0 = ix->inst_h[0];
                APS_TRY(sort_pairs(sp_key, sp_score, sp_found, bits_for((uint64_t)I0.n * (uint64_t)I0.n), s));
                const unsigned long long *const sp_sorted = reinterpret_cast<const unsigned long long *>(sp_key.p);
                DBuf<int32_t> flag;
                DBuf<int64_t> off;
                APS_TRY(flag.alloc((size_t)sp_found, s));
                APS_TRY(off.alloc((size_t)sp_found + 1, s));
                k_first_of_key<<<grid_for(sp_found, 256), 256, 0, s>>>(sp_sorted, sp_found, flag.p);
                APS_LAUNCH_CHECK();
                APS_TRY(scan_exclusive(flag.p, off.p, sp_found, s));
                int64_t nuniq = 0;
                APS_CUDA(cudaMemcpyAsync(&nuniq, off.p + sp_found, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
                APS_CUDA(cudaStreamSynchronize(s));
                if (reserved + nuniq > stage_cap) {  // room after the join's runs
                    DBuf<int2> grown;
                    APS_TRY(grown.alloc((size_t)(reserved + nuniq), s));
                    if (reserved > 0)
                        APS_CUDA(cudaMemcpyAsync(grown.p, stage.p, sizeof(int2) * reserved, cudaMemcpyDeviceToDevice, s));
                    std::swap(grown.p, stage.p);
                    std::swap(grown.n, stage.n);
                    stage_cap = reserved + nuniq;
                }
                k_split_place<<<grid_for(sp_found, 256), 256, 0, s>>>(sp_sorted, sp_score.p, flag.p, off.p, sp_found,
                                                                     d.inst.p, parts, reserved, stage.p, segs.p, cntq.p);
                APS_LAUNCH_CHECK();
                k_split_counts<<<grid_for(sp_found, 256), 256, 0, s>>>(sp_sorted, flag.p, sp_found, d.inst.p, parts,
                                                                      cntq.p, segs.p);
                APS_LAUNCH_CHECK();
                total_pairs += nuniq;
            }
            break;
        }
        if (sp_found > sp_cap) sp_cap = sp_found + sp_found / 8 + 1024;
        if (reserved <= stage_cap) {
            reruns++;
            if (attempt == 2) {
                set_error("split pair list overflow persisted");
                return APS_EOVERFLOW;
            }
            continue;
        }
        // the staging buffer was too small: grow it and run again
        reruns++;
        stage_cap = reserved + (int64_t)sms * join_slab_slack();  // plus every slab a CTA can leave unfilled
        if (attempt == 2) {
            set_error("pair staging overflow persisted");
            return APS_EOVERFLOW;
        }
    }
    ix->hint_pairs = reserved + reserved / 16 + 1024;
    g_stage_hint.store(ix->hint_pairs);
    APS_CUDA(cudaEventRecord(ev[3], s));

    // ---------------- output: scan counts, gather runs into (i, j, score)
    DBuf<int64_t> qwoff;
    APS_TRY(qwoff.alloc((size_t)nslots + 1, s));
    APS_TRY(scan_exclusive(cntq.p, qwoff.p, nslots, s));
    const int64_t npairs = total_pairs;
    PairsAlloc *pa = new PairsAlloc();
    pa->stream = s;
    const size_t bytes = (size_t)std::max<int64_t>(npairs, 1) * 12 + 256;
    aps_status st = dalloc(&pa->block, bytes, s);
    if (st != APS_OK) {
        delete pa;
        return st;
    }
    char *blk = static_cast<char *>(pa->block);
    int32_t *oi = reinterpret_cast<int32_t *>(blk);
    int32_t *oj = reinterpret_cast<int32_t *>(blk + (((size_t)npairs * 4 + 127) & ~(size_t)127));
    float *os = reinterpret_cast<float *>(blk + 2 * (((size_t)npairs * 4 + 127) & ~(size_t)127));
    if (npairs > 0) {
        k_gather<<<grid_for(nslots * 32, 256, (int64_t)sms * 32), 256, 0, s>>>(
            segs.p, chain.p, JOIN_STAGE_SLAB, cntq.p, nslots, stage.p, qwoff.p, oi, oj, os);
        APS_LAUNCH_CHECK();
    }
    if (pair_offsets_h) {
        DBuf<int64_t> offs;
        APS_TRY(offs.alloc((size_t)ix->k + 1, s));
        k_inst_offsets<<<grid_for(ix->k + 1, 256), 256, 0, s>>>(d.inst.p, ix->k, qwoff.p, parts, nslots, offs.p);
        APS_LAUNCH_CHECK();
        pair_offsets_h->assign((size_t)ix->k + 1, 0);
        APS_CUDA(cudaMemcpyAsync(pair_offsets_h->data(), offs.p, sizeof(int64_t) * (ix->k + 1),
                                 cudaMemcpyDeviceToHost, s));
    }
    APS_CUDA(cudaEventRecord(ev[2], s));
    APS_CUDA(cudaEventSynchronize(ev[2]));
    float ms_join = 0, ms_sort = 0;
    cudaEventElapsedTime(&ms_join, ev[0], ev[1]);
    cudaEventElapsedTime(&ms_sort, ev[3], ev[2]);
    std::lock_guard<std::mutex> lk(ix->stats_mu);  // queries may report meanwhile
    aps_stats &S = ix->stats;
    S.visits = (int64_t)ch[0];
    S.candidates = (int64_t)ch[1];
    S.verified = (int64_t)ch[2];
    S.pairs = total_pairs;
    S.band = (int64_t)ch[4];
    S.entries_read = (int64_t)ch[6];
    S.reruns = reruns;
    S.ms_join = ms_join;
    S.ms_sort = ms_sort;
    S.evaluations = 0;
    for (const InstDesc &I : ix->inst_h) S.evaluations += (int64_t)I.n * (I.n - 1) / 2;
    out->count = npairs;
    out->i = oi;
    out->j = oj;
    out->score = os;
    out->on_device = 1;
    out->_reserved = 0;
    out->_priv = pa;
    return APS_OK;
}

void pairs_release(aps_pairs *p) {
    if (!p || !p->_priv) return;
    PairsAlloc *pa = static_cast<PairsAlloc *>(p->_priv);
    if (--pa->refs <= 0) {
        if (pa->on_device)
            dfree(pa->block, pa->stream);
        else
            hfree(pa->block, pa->bytes);
        delete pa;
    }
    p->_priv = nullptr;
    p->i = p->j = nullptr;
    p->score = nullptr;
    p->count = 0;
}

namespace {

// Whether p is host memory, pinned or not (managed memory is left to the driver).
bool is_host(const void *p) {
    cudaPointerAttributes pa;
    if (cudaPointerGetAttributes(&pa, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return pa.type == cudaMemoryTypeUnregistered || pa.type == cudaMemoryTypeHost;
}

}  // namespace

aps_status pairs_copy(const aps_pairs *p, int32_t *i, int32_t *j, float *score, cudaStream_t s) {
    const size_t n = (size_t)std::max<int64_t>(p->count, 0);
    const void *src[3] = {p->i, p->j, p->score};
    void *dst[3] = {i, j, score};
    bool all_host = n && !p->on_device;
    for (int k = 0; k < 3 && all_host; k++) all_host = !dst[k] || is_host(dst[k]);
    if (all_host) {
        // A result in pinned host memory to plain host memory: the processor copies it (the driver
        // moves such copies at 9.5 GB/s), the three arrays side by side where they are large.
        APS_CUDA(cudaStreamSynchronize(s));
        std::thread side[2];
        int running = 0;
        int own[3], nown = 0;
        for (int k = 0; k < 3; k++) {
            if (!dst[k]) continue;
            if (nown > 0 && n >= ((size_t)1 << 18)) {
                try {
                    void *d = dst[k];
                    const void *a = src[k];
                    side[running] = std::thread([d, a, n] { memcpy(d, a, n * 4); });
                    running++;
                    continue;
                } catch (const std::system_error &) {  // no thread to be had: copied here
                }
            }
            own[nown++] = k;
        }
        for (int q = 0; q < nown; q++) memcpy(dst[own[q]], src[own[q]], n * 4);
        for (int q = 0; q < running; q++) side[q].join();
        return APS_OK;
    } else if (n) {
        for (int k = 0; k < 3; k++)
            if (dst[k]) APS_CUDA(cudaMemcpyAsync(dst[k], src[k], n * 4, cudaMemcpyDefault, s));
    }
    APS_CUDA(cudaStreamSynchronize(s));
    return APS_OK;
}

// Copy device pairs into one pinned host allocation (replacing the device one).
aps_status pairs_to_host(aps_pairs *p, cudaStream_t s) {
    if (!p->on_device) return APS_OK;
    PairsAlloc *pa = new PairsAlloc();
    pa->on_device = 0;
    pa->stream = s;
    // the three arrays as they lie on the device, so that one copy takes a few pairs over
    const size_t n = (size_t)p->count, seg = (n * 4 + 127) & ~(size_t)127;
    pa->bytes = std::max<size_t>(2 * seg + n * 4, 12);
    aps_status hst = halloc(&pa->block, pa->bytes);
    if (hst != APS_OK) {
        delete pa;
        return hst;
    }
    char *blk = static_cast<char *>(pa->block);
    int32_t *hi = reinterpret_cast<int32_t *>(blk);
    int32_t *hj = reinterpret_cast<int32_t *>(blk + seg);
    float *hs = reinterpret_cast<float *>(blk + 2 * seg);
    const char *di = reinterpret_cast<const char *>(p->i);
    if (n && reinterpret_cast<const char *>(p->j) == di + seg && reinterpret_cast<const char *>(p->score) == di + 2 * seg) {
        APS_CUDA(cudaMemcpyAsync(hi, di, 2 * seg + n * 4, cudaMemcpyDeviceToHost, s));
    } else if (n) {
        APS_CUDA(cudaMemcpyAsync(hi, p->i, n * 4, cudaMemcpyDeviceToHost, s));
        APS_CUDA(cudaMemcpyAsync(hj, p->j, n * 4, cudaMemcpyDeviceToHost, s));
        APS_CUDA(cudaMemcpyAsync(hs, p->score, n * 4, cudaMemcpyDeviceToHost, s));
    }
    APS_CUDA(cudaStreamSynchronize(s));
    pairs_release(p);
    p->count = (int64_t)n;
    p->i = hi;
    p->j = hj;
    p->score = hs;
    p->on_device = 0;
    p->_priv = pa;
    return APS_OK;
}

// ------------------------------------------------------------------ arena variant
// The same join and output kernels with every buffer carved out of a caller-provided
// device arena instead of allocated: counters, per-vector counts and offsets, the segment
// table, the streamed class's per-warp lists (for at most max_ctas CTAs) and, in what is
// left, the pair staging buffer. Pairs are gathered into the caller's (i, j, score) arrays.
namespace {

constexpr int SCAN1_THREADS = 1024;

// Exclusive prefix sum by a single CTA, tile by tile with a running carry (no scratch).
__global__ void __launch_bounds__(SCAN1_THREADS) k_scan_single(const int32_t *__restrict__ in, int64_t n,
                                                               int64_t *__restrict__ out) {
    __shared__ int64_t wt[SCAN1_THREADS / 32];
    __shared__ int64_t carry_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry_s = 0;
    __syncthreads();
    for (int64_t base = 0; base < n; base += (int64_t)SCAN1_THREADS * 4) {
        const int64_t i0 = base + (int64_t)threadIdx.x * 4;
        int64_t v[4], local = 0;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            v[k] = (i0 + k < n) ? (int64_t)in[i0 + k] : 0;
            local += v[k];
        }
        int64_t inc = warp_incl_scan(local, lane);
        if (lane == 31) wt[warp] = inc;
        __syncthreads();
        const int64_t wv = lane < SCAN1_THREADS / 32 ? wt[lane] : 0;
        const int64_t winc = warp_incl_scan(wv, lane);
        const int64_t before = __shfl_sync(0xffffffffu, winc - wv, warp);
        const int64_t tile = __shfl_sync(0xffffffffu, winc, 31);
        int64_t run = carry_s + before + inc - local;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            if (i0 + k < n) out[i0 + k] = run;
            run += v[k];
        }
        __syncthreads();
        if (threadIdx.x == 0) carry_s += tile;
        __syncthreads();
    }
    if (threadIdx.x == 0) out[n] = carry_s;
}

inline size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace

aps_status join_noalloc(aps_index *ix, unsigned char *arena, size_t arena_bytes, int max_ctas, int32_t *oi,
                        int32_t *oj, float *os, int64_t cap, int64_t *count, cudaStream_t s, int parts) {
    const int grid_max = std::max(1, std::min(num_sms(), max_ctas));
    // The documented limit: 28 bytes for each of the index's arena slots beside the fixed parts.
    const size_t limit = (size_t)std::max<int64_t>(ix->arena_slots, 1) * 28 + (size_t)max_ctas * 32 * 1408 * sizeof(int2);
    const int64_t slab = 32;  // small slabs: the arena's staging room is modest
    // The heaviest vectors' windows in parts, as in the allocating join, where their slots take no
    // more than a sixteenth of the arena; if the pairs then do not fit the rest, once more in one.
    const int64_t part_room = (int64_t)(arena_bytes / 16 / (sizeof(int32_t) + sizeof(int64_t) + sizeof(Segment)));
    if (parts < 0) parts = (int)std::max<int64_t>(1, std::min<int64_t>(ix->parts, part_room / std::max<int64_t>(ix->N, 1)));
    const int64_t nslots = std::max<int64_t>(ix->N * parts, 1);
    size_t off = 0;
    unsigned long long *ctr = reinterpret_cast<unsigned long long *>(arena + off);
    off = align256(off + 16 * sizeof(unsigned long long));
    int32_t *cntq = reinterpret_cast<int32_t *>(arena + off);
    off = align256(off + sizeof(int32_t) * nslots);
    int64_t *qwoff = reinterpret_cast<int64_t *>(arena + off);
    off = align256(off + sizeof(int64_t) * (nslots + 1));
    Segment *segs = reinterpret_cast<Segment *>(arena + off);
    off = align256(off + sizeof(Segment) * nslots);
    int2 *elists = reinterpret_cast<int2 *>(arena + off);
    off = align256(off + sizeof(int2) * (size_t)grid_max * JOIN_WARPS * JOIN_ECAP);
    if (limit >= arena_bytes || off + 4096 >= arena_bytes) {
        set_error("index too large for the %zu-byte arena: its %lld arena slots count as %zu bytes "
                  "before any pair is staged",
                  arena_bytes, (long long)ix->arena_slots, std::max(limit, off));
        return APS_EINVAL;
    }
    // the rest: staged pairs (8 bytes each) and a chain entry (8 bytes) for every slab of them
    const int64_t nslabs = (int64_t)((arena_bytes - off - 1024) / (sizeof(int2) * (slab + 1)));
    const int64_t stage_cap = nslabs * slab;
    int2 *chain = reinterpret_cast<int2 *>(arena + off);
    off = align256(off + sizeof(int2) * (nslabs + 1));
    int2 *stage = reinterpret_cast<int2 *>(arena + off);

    const int need = join_smem();
    const uint32_t flags = ix->flags & (APS_NO_MINSIZE | APS_NO_REMSCORE | APS_NO_UPPERBOUND);
    APS_TRY(allow_smem(self_kernel(ix, flags)));
    APS_CUDA(cudaMemsetAsync(ctr, 0, 16 * sizeof(unsigned long long), s));
    APS_CUDA(cudaMemsetAsync(cntq, 0, sizeof(int32_t) * nslots, s));
    if (ix->class_begin[JOIN_NCLS] > ix->class_begin[0]) {
        JoinParams P;
        set_index(P, ix);
        const int grid = set_classes(P, ix, parts, grid_max);
        P.flags = flags;
        P.stage = stage;
        P.stage_cap = stage_cap;
        P.stage_count = ctr + 5;
        P.stage_slab = slab;
        P.segs = segs;
        P.chain = chain;
        P.cntq = cntq;
        P.counters = ctr;
        P.work = ctr + 8;
        P.scratch = elists;
        self_kernel(ix, flags)<<<grid, JOIN_THREADS, need, s>>>(P);
        APS_LAUNCH_CHECK();
    }
    unsigned long long ch[16];
    APS_CUDA(cudaMemcpyAsync(ch, ctr, sizeof(ch), cudaMemcpyDeviceToHost, s));
    APS_CUDA(cudaStreamSynchronize(s));
    const int64_t total = (int64_t)ch[3];
    *count = total;
    if ((int64_t)ch[5] > stage_cap && parts > 1)
        return join_noalloc(ix, arena, arena_bytes, max_ctas, oi, oj, os, cap, count, s, 1);
    if ((int64_t)ch[5] > stage_cap) {
        set_error("%lld staged pairs (%lld emitted) exceed the arena's staging room of %lld pairs",
                  (long long)ch[5], (long long)total, (long long)stage_cap);
        return APS_EOVERFLOW;
    }
    if (total > cap) {
        set_error("%lld pairs do not fit the caller's capacity of %lld", (long long)total, (long long)cap);
        return APS_EOVERFLOW;
    }
    k_scan_single<<<1, SCAN1_THREADS, 0, s>>>(cntq, ix->N * parts, qwoff);
    APS_LAUNCH_CHECK();
    if (total > 0) {
        k_gather<<<grid_for(nslots * 32, 256, (int64_t)num_sms() * 32), 256, 0, s>>>(segs, chain, slab, cntq, nslots,
                                                                                    stage, qwoff, oi, oj, os);
        APS_LAUNCH_CHECK();
    }
    APS_CUDA(cudaStreamSynchronize(s));
    // the index's stats report the last join, whichever entry point ran it (no timings:
    // this path records no events)
    std::lock_guard<std::mutex> lk(ix->stats_mu);
    aps_stats &S = ix->stats;
    S.visits = (int64_t)ch[0];
    S.candidates = (int64_t)ch[1];
    S.verified = (int64_t)ch[2];
    S.pairs = (int64_t)ch[3];
    S.band = (int64_t)ch[4];
    S.entries_read = (int64_t)ch[6];
    S.reruns = 0;
    S.ms_join = S.ms_sort = S.ms_total = 0.f;
    S.evaluations = 0;
    for (const InstDesc &I : ix->inst_h) S.evaluations += (int64_t)I.n * (I.n - 1) / 2;
    return APS_OK;
}

// ------------------------------------------------------------------ external queries
aps_status join_queries(const aps_index *ix, const QueryArrays &qa, float t, uint32_t flags, cudaStream_t s,
                        aps_pairs *out, aps_stats *stats) {
    const IndexArrays &d = ix->d;
    const InstDesc &I = ix->inst_h[0];
    const int sms = num_sms();
    const int64_t nq = qa.nq;
    const int G = I.G;
    const int parts = query_parts(ix, nq);
    const int64_t nqw = std::max<int64_t>(nq * parts, 1);
    const int need = tile_bytes(G) * tile_warps(G);
    const int64_t slab = QUERY_SLAB;
    APS_TRY(allow_smem(query_kernel(ix)));
    cudaEvent_t ev[3];
    for (int i = 0; i < 3; i++) APS_CUDA(cudaEventCreate(&ev[i]));
    struct EvGuard {
        cudaEvent_t *e;
        ~EvGuard() {
            for (int i = 0; i < 3; i++) cudaEventDestroy(e[i]);
        }
    } evg{ev};
    const int64_t nitems = I.nw > 0 ? nq : 0;
    const int grid = query_ctas(ix, nq);
    DBuf<unsigned long long> ctr;  // 16 counters, then the pair counts of the query parts
    DBuf<int2> chain, stage;
    DBuf<Segment> segs;
    APS_TRY(ctr.alloc(16 + ((size_t)nqw + 1) / 2, s));
    int32_t *const cntq = reinterpret_cast<int32_t *>(ctr.p + 16);
    APS_TRY(segs.alloc((size_t)nqw, s));
    const int64_t slack = (int64_t)grid * JOIN_WARPS * slab;
    int64_t stage_cap = query_stage(ix, nq);
    unsigned long long ch[16];
    for (int attempt = 0; attempt < 2; attempt++) {
        APS_TRY(stage.alloc((size_t)stage_cap, s));
        APS_TRY(chain.alloc((size_t)(stage_cap / slab) + 1, s));
        APS_CUDA(cudaMemsetAsync(ctr.p, 0, sizeof(ch) + sizeof(int32_t) * nqw, s));
        APS_CUDA(cudaEventRecord(ev[0], s));
        if (nq > 0) {
            JoinParams P;
            set_index(P, ix);
            P.items = nullptr;
            P.ncls = 1;
            P.cls_G[0] = G;
            P.cls_begin[0] = 0;
            P.cls_begin[1] = nitems;
            P.cls_heavy[0] = nitems;
            P.parts = parts;
            P.flags = flags & (APS_NO_MINSIZE | APS_NO_REMSCORE | APS_NO_UPPERBOUND);
            P.stage = stage.p;
            P.stage_cap = stage_cap;
            P.stage_count = ctr.p + 5;
            P.stage_slab = slab;
            P.segs = segs.p;
            P.chain = chain.p;
            P.cntq = cntq;
            P.counters = ctr.p;
            P.work = ctr.p + 8;
            P.qcrow = qa.crow.p;
            P.qvmeta = qa.vmeta.p;
            P.qt = t;
            query_kernel(ix)<<<grid, JOIN_THREADS, need, s>>>(P);
            APS_LAUNCH_CHECK();
        }
        APS_CUDA(cudaEventRecord(ev[1], s));
        APS_CUDA(cudaMemcpyAsync(ch, ctr.p, sizeof(ch), cudaMemcpyDeviceToHost, s));
        APS_CUDA(cudaStreamSynchronize(s));
        if ((int64_t)ch[5] <= stage_cap) break;
        stage_cap = (int64_t)ch[5] + slack;  // what was reserved, plus one slab per warp
    }
    if (nq > 0) {  // remember what this batch needed (with a quarter more), for the next ones
        const int64_t need16 = (int64_t)ch[3] * 20 / nq;  // (the slabs' unused rests are the slack)
        int64_t cur = ix->q_ppq16.load(std::memory_order_relaxed);
        while (need16 > cur && !ix->q_ppq16.compare_exchange_weak(cur, need16, std::memory_order_relaxed)) {
        }
    }
    if ((int64_t)ch[5] > stage_cap) {
        set_error("pair staging overflow persisted");
        return APS_EOVERFLOW;
    }
    const int64_t npairs = (int64_t)ch[3];
    DBuf<int64_t> qwoff;
    APS_TRY(qwoff.alloc((size_t)nqw + 1, s));
    APS_TRY(scan_exclusive(cntq, qwoff.p, nqw, s));
    PairsAlloc *pa = new PairsAlloc();
    pa->stream = s;
    const size_t seg4 = ((size_t)npairs * 4 + 127) & ~(size_t)127;
    aps_status st = dalloc(&pa->block, std::max<size_t>(3 * seg4, 256), s);
    if (st != APS_OK) {
        delete pa;
        return st;
    }
    char *blk = static_cast<char *>(pa->block);
    int32_t *oi = reinterpret_cast<int32_t *>(blk);
    int32_t *oj = reinterpret_cast<int32_t *>(blk + seg4);
    float *os = reinterpret_cast<float *>(blk + 2 * seg4);
    if (npairs > 0) {
        k_gather<<<grid_for(nqw * 32, 256, (int64_t)sms * 32), 256, 0, s>>>(segs.p, chain.p, slab, cntq, nqw,
                                                                           stage.p, qwoff.p, oi, oj, os);
        APS_LAUNCH_CHECK();
    }
    APS_CUDA(cudaEventRecord(ev[2], s));
    APS_CUDA(cudaEventSynchronize(ev[2]));
    if (stats) {
        float mj = 0, mo = 0;
        cudaEventElapsedTime(&mj, ev[0], ev[1]);
        cudaEventElapsedTime(&mo, ev[1], ev[2]);
        memset(stats, 0, sizeof(*stats));
        stats->visits = (int64_t)ch[0];
        stats->candidates = (int64_t)ch[1];
        stats->verified = (int64_t)ch[2];
        stats->pairs = (int64_t)ch[3];
        stats->band = (int64_t)ch[4];
        stats->entries_read = (int64_t)ch[6];
        stats->evaluations = nq * (int64_t)I.n;
        stats->ms_join = mj;
        stats->ms_sort = mo;
    }
    out->count = npairs;
    out->i = oi;
    out->j = oj;
    out->score = os;
    out->on_device = 1;
    out->_reserved = 0;
    out->_priv = pa;
    return APS_OK;
}

}  // namespace aps
