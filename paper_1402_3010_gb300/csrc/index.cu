// Index build: input statistics, dimension ranking, canonical rows, partial-indexing
// split and the suffix inverted index (the preprocessing of all-pairs-1/2 and the
// index-insertion step of Alg. 1, done for all vectors at once).
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "index.cuh"

namespace aps {
namespace {

constexpr int T256 = 256;

__device__ __forceinline__ int inst_of_vec(const InstDesc *inst, int k, int64_t x) {
    // last instance whose vbase <= x (instances with n == 0 share the next vbase)
    int lo = 0, hi = k;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (inst[mid].vbase <= x) lo = mid + 1; else hi = mid;
    }
    return lo - 1;
}

__device__ __forceinline__ int inst_of_rank(const InstDesc *inst, int k, int64_t r) {
    int lo = 0, hi = k;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if ((int64_t)inst[mid].rbase <= r) lo = mid + 1; else hi = mid;
    }
    return lo - 1;
}

// The start of a build in one launch: the row pointers' copy, every vector's instance, empty
// dimension statistics and counters (err[0] all ones, the others 0) and, for a single instance,
// its description (by value: no copy from the host; its windows follow with the list pointers). A copy or a reset of its own costs its
// caller 3 to 15 us, a tenth of the smallest builds in all.
__global__ void k_setup(const int64_t *__restrict__ indptr, InstDesc one, InstDesc *inst, int k, int64_t N, int64_t M,
                        int64_t *cptr, int32_t *vinst, int32_t *nnz_d, float *mw_d, unsigned long long *err, int nerr) {
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    if (k == 1 && i0 == 0) inst[0] = one;
    if (i0 < nerr) err[i0] = i0 == 0 ? ~0ull : 0ull;
    for (int64_t x = i0; x <= N; x += step) {
        cptr[x] = indptr[x];
        if (x < N) vinst[x] = k == 1 ? 0 : inst_of_vec(inst, k, x);
    }
    for (int64_t d = i0; d < M; d += step) {
        nnz_d[d] = 0;
        mw_d[d] = 0.f;
    }
}

// Validation codes reported as (row << 8 | code) through atomicMin.
enum { E_PTR = 1, E_IDX_RANGE = 2, E_IDX_ORDER = 3, E_VALUE = 4, E_NORM = 5 };

// CTAs for a warp per row: some rounds of what is resident, so that the sums each CTA adds to one
// counter are few. With a warp for each of 1.9M rows, the 64-bit atomics on one address were most
// of the time of the kernels that have them (k_split took 3.1 ms, 1.4 with these grids).
unsigned rows_grid(int64_t rows) { return grid_for(rows * 32, 256, (int64_t)num_sms() * 64); }

// One warp per row: checks the row, records |x| and maxweight(x), and copies the values
// (scaled to unit norm with APS_NORMALIZE). The lanes read 32 components at a time; the
// error code is that of the row's first bad component (range before order before value,
// as for a sequential check). The float64 sum of squares is a warp tree sum.
__global__ void k_validate(const int64_t *__restrict__ indptr, const int32_t *__restrict__ idx,
                           const float *__restrict__ val, const int32_t *__restrict__ vinst,
                           const InstDesc *__restrict__ inst, int32_t m1, int64_t N, int64_t nnz, uint32_t flags,
                           int32_t *__restrict__ erow, float *__restrict__ vout, int32_t *__restrict__ len,
                           float *__restrict__ mw, unsigned long long *err,
                           unsigned long long *longest_out) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long longest = 0;  // the longest row this warp met (to *longest_out, when given)
    for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < N; x += nwarps) {
        const int64_t a = indptr[x], b = indptr[x + 1];
        if (a < 0 || b < a || b > nnz) {
            if (lane == 0) {
                atomicMin(err, ((unsigned long long)x << 8) | E_PTR);
                len[x] = 0;
                mw[x] = 0.f;
            }
            continue;
        }
        const int m = vinst ? inst[vinst[x]].m : m1;
        int code = 0, prev_last = -1;
        float s32 = 0.f;
        for (int64_t base = a; base < b; base += 32) {
            const int64_t p = base + lane;
            const int cnt = (int)min((int64_t)32, b - base);
            int d = 0;
            float v = 1.f;
            if (p < b) {
                d = idx[p];
                v = val[p];
                erow[p] = (int32_t)x;
            }
            int prevd = __shfl_up_sync(0xffffffffu, d, 1);
            if (lane == 0) prevd = prev_last;
            int ec = 0;
            if (p < b) {
                if (d < 0 || d >= m) ec = E_IDX_RANGE;
                else if (d <= prevd) ec = E_IDX_ORDER;
                else if (!(v > 0.f) || !isfinite(v)) ec = E_VALUE;
            }
            const unsigned bad = __ballot_sync(0xffffffffu, ec != 0);
            if (!code && bad) code = __shfl_sync(0xffffffffu, ec, __ffs(bad) - 1);
            if (p < b) s32 = fmaf(v, v, s32);
            prev_last = __shfl_sync(0xffffffffu, d, cnt - 1);
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) s32 += __shfl_xor_sync(0xffffffffu, s32, o);
        float best = 0.f;
        if (b > a && !code) {
            // float32 decides where its sum of squares, off by less than 3e-5 (L / 32 + 6 roundings
            // of at most 2^-24 each), lies clear of the norms 1 -+ 1e-3; the rest, and rows to be
            // scaled, take the float64 norm (for every one of 1.9M rows that took 3.5 ms, this 0.64)
            const bool clear = b - a <= 8192 && s32 <= 1.0019f && ((flags & APS_SUBUNIT_NORMS) || s32 >= 0.9981f);
            double nrm = 1.0;
            if ((flags & APS_NORMALIZE) || !clear) {
                double ss = 0.0;
                for (int64_t p = a + lane; p < b; p += 32) ss += (double)val[p] * (double)val[p];
#pragma unroll
                for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
                nrm = sqrt(ss);
                if (!(flags & APS_NORMALIZE) &&
                    ((flags & APS_SUBUNIT_NORMS) ? nrm > 1.0 + 1e-3 : fabs(nrm - 1.0) > 1e-3))
                    code = E_NORM;
            }
            for (int64_t p = a + lane; p < b; p += 32) {
                const float v = (flags & APS_NORMALIZE) ? (float)((double)val[p] / nrm) : val[p];
                vout[p] = v;
                best = fmaxf(best, v);
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
        }
        if (lane == 0) {
            if (code) atomicMin(err, ((unsigned long long)x << 8) | (unsigned long long)code);
            len[x] = (int32_t)(b - a);
            mw[x] = best;
            longest = max(longest, (unsigned long long)(b - a));
        }
    }
    if (longest_out) {
        __shared__ unsigned long long blongest;
        if (threadIdx.x == 0) blongest = 0ull;
        __syncthreads();
        if (lane == 0) atomicMax(&blongest, longest);
        __syncthreads();
        if (threadIdx.x == 0) atomicMax(longest_out, blongest);
    }
}

// The rank-ordered rows when no row is longer than 64 components: one warp per row sorts
// the row's (rank, value) pairs by a bitonic network over the lanes, two per lane (element
// k = 2 * lane + h; rows of at most 32, one per lane and six steps fewer), instead of the
// global sort by (row, rank) that longer rows need. Bound by the network's exchanges: 1.9M rows
// of 30 on average took 1.4 ms with 64 places for every row and a CTA for every eight, 1.06 now.
__global__ void k_canon_rows64(const int64_t *__restrict__ cptr, const int32_t *__restrict__ idx,
                               const float *__restrict__ vout, const int32_t *__restrict__ vinst,
                               const InstDesc *__restrict__ inst, const int32_t *__restrict__ rank_of_dim,
                               int64_t N, int32_t *crank, float *cval) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < N; x += nwarps) {
        const int64_t a = cptr[x];
        const int L = (int)(cptr[x + 1] - a);  // <= 64
        const int64_t rb = inst[vinst[x]].rbase;
        if (L <= 32) {
            int r = 0x7fffffff;  // padding sorts last
            float v = 0.f;
            if (lane < L) {
                r = rank_of_dim[rb + idx[a + lane]];
                v = vout[a + lane];
            }
#pragma unroll
            for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
                for (int j = size >> 1; j > 0; j >>= 1) {
                    const int pr = __shfl_xor_sync(0xffffffffu, r, j);
                    const float pv = __shfl_xor_sync(0xffffffffu, v, j);
                    const bool keep_min = ((lane & j) == 0) == ((lane & size) == 0);
                    if (keep_min ? pr < r : pr > r) {
                        r = pr;
                        v = pv;
                    }
                }
            }
            if (lane < L) {
                crank[a + lane] = r;
                cval[a + lane] = v;
            }
            continue;
        }
        const int k0 = 2 * lane, k1 = k0 + 1;
        int r0 = 0x7fffffff, r1 = 0x7fffffff;  // padding sorts last
        float v0 = 0.f, v1 = 0.f;
        if (k0 < L) {
            r0 = rank_of_dim[rb + idx[a + k0]];
            v0 = vout[a + k0];
        }
        if (k1 < L) {
            r1 = rank_of_dim[rb + idx[a + k1]];
            v1 = vout[a + k1];
        }
#pragma unroll
        for (int size = 2; size <= 64; size <<= 1) {
            // blocks of `size` elements ascending where bit `size` of k is 0, descending elsewhere
            const bool asc = (k0 & size) == 0;  // (k0 and k1 agree on it for size >= 2)
#pragma unroll
            for (int j = size >> 1; j > 0; j >>= 1) {
                if (j == 1) {  // elements k0, k1 of this lane
                    if ((r0 > r1) == asc) {
                        const int tr = r0;
                        r0 = r1;
                        r1 = tr;
                        const float tv = v0;
                        v0 = v1;
                        v1 = tv;
                    }
                } else {  // element k and k ^ j: the same slot of lane ^ (j / 2)
                    const int lm = j >> 1;
                    const int p0 = __shfl_xor_sync(0xffffffffu, r0, lm), p1 = __shfl_xor_sync(0xffffffffu, r1, lm);
                    const float q0 = __shfl_xor_sync(0xffffffffu, v0, lm), q1 = __shfl_xor_sync(0xffffffffu, v1, lm);
                    const bool keep_min = ((lane & lm) == 0) == asc;  // the lower element keeps the min when ascending
                    if (keep_min ? p0 < r0 : p0 > r0) {
                        r0 = p0;
                        v0 = q0;
                    }
                    if (keep_min ? p1 < r1 : p1 > r1) {
                        r1 = p1;
                        v1 = q1;
                    }
                }
            }
        }
        if (k0 < L) {
            crank[a + k0] = r0;
            cval[a + k0] = v0;
        }
        if (k1 < L) {
            crank[a + k1] = r1;
            cval[a + k1] = v1;
        }
    }
}

// Per-dimension non-zero count and maxweight_i(V) (positive floats order like ints).
__global__ void k_dimstats(const int32_t *__restrict__ idx, const float *__restrict__ vout,
                           const int32_t *__restrict__ erow, const int32_t *__restrict__ vinst,
                           const InstDesc *__restrict__ inst, int64_t nnz, int32_t *nnz_d, float *mw_d) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x) {
        int64_t D = (int64_t)inst[vinst[erow[p]]].rbase + idx[p];
        atomicAdd(&nnz_d[D], 1);
        atomicMax(reinterpret_cast<int *>(&mw_d[D]), __float_as_int(vout[p]));
    }
}

// The same for a batch of instances of at most DIMSTATS_DIMS dimensions each: one CTA per
// instance counts in shared memory (shared atomics instead of global ones on 25M
// dimensions), first the non-zeros, then the maxima, each written out once.
constexpr int DIMSTATS_DIMS = 56 * 1024;  // 224 KB of 32-bit counters
__global__ void __launch_bounds__(1024) k_dimstats_inst(const int64_t *__restrict__ cptr,
                                                        const int32_t *__restrict__ idx,
                                                        const float *__restrict__ vout,
                                                        const InstDesc *__restrict__ inst, int32_t *nnz_d,
                                                        float *mw_d) {
    extern __shared__ uint32_t dcnt[];  // [I.m]
    const InstDesc I = inst[blockIdx.x];
    const int64_t a = cptr[I.vbase], b = cptr[I.vbase + I.n];
    for (int pass = 0; pass < 2; pass++) {
        for (int d = threadIdx.x; d < I.m; d += blockDim.x) dcnt[d] = 0u;
        __syncthreads();
        for (int64_t p = a + threadIdx.x; p < b; p += blockDim.x) {
            if (pass == 0) atomicAdd(&dcnt[idx[p]], 1u);
            else atomicMax(&dcnt[idx[p]], __float_as_uint(vout[p]));  // positive floats order like their bits
        }
        __syncthreads();
        for (int d = threadIdx.x; d < I.m; d += blockDim.x) {
            if (pass == 0) nnz_d[(int64_t)I.rbase + d] = (int32_t)dcnt[d];
            else mw_d[(int64_t)I.rbase + d] = __uint_as_float(dcnt[d]);
        }
        __syncthreads();
    }
}

// Dimension order of all-pairs-1: decreasing non-zero count; the sort is stable and the
// input is in id order, so ties keep ascending dimension id.
template <class K>
__global__ void k_rank_keys(const int32_t *__restrict__ nnz_d, const InstDesc *__restrict__ inst, int k,
                            int64_t M, int nbits, uint64_t nmax, K *keys, uint32_t *vals) {
    for (int64_t D = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; D < M; D += (int64_t)gridDim.x * blockDim.x) {
        uint64_t ki = (uint64_t)inst_of_rank(inst, k, D);
        keys[D] = (K)((ki << nbits) | (nmax - (uint64_t)nnz_d[D]));
        vals[D] = (uint32_t)D;
    }
}

// The dimensions in rank order (vals): keys of 32 bits where they hold the instance and the count.
template <class K>
aps_status sort_dims(const aps_index *ix, int32_t maxn, DBuf<uint32_t> &vals, cudaStream_t s) {
    const IndexArrays &d = ix->d;
    const int nb = bits_for((uint64_t)maxn);
    DBuf<K> keys;
    APS_TRY(keys.alloc((size_t)ix->M, s));
    APS_TRY(vals.alloc((size_t)ix->M, s));
    k_rank_keys<K><<<grid_for(ix->M, T256), T256, 0, s>>>(d.nnz_d.p, d.inst.p, ix->k, ix->M, nb, (uint64_t)maxn, keys.p,
                                                          vals.p);
    APS_LAUNCH_CHECK();
    return sort_pairs(keys, vals, ix->M, nb + bits_for((uint64_t)(ix->k - 1)), s);
}

__global__ void k_rank_scatter(const uint32_t *__restrict__ vals, const InstDesc *__restrict__ inst, int k,
                               int64_t M, const float *__restrict__ mw_d, int32_t *rank_of_dim,
                               int32_t *dim_of_rank, float *mwr) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t D = vals[i];
        int ki = inst_of_rank(inst, k, i);
        rank_of_dim[D] = (int32_t)(i - inst[ki].rbase);
        dim_of_rank[i] = (int32_t)D;
        mwr[i] = mw_d[D];
    }
}

__global__ void k_canon_keys(const int32_t *__restrict__ idx, const int32_t *__restrict__ erow,
                             const int32_t *__restrict__ vinst, const InstDesc *__restrict__ inst,
                             const int32_t *__restrict__ rank_of_dim, int64_t nnz, int rb, uint64_t *keys,
                             uint32_t *vals) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x) {
        int64_t x = erow[p];
        int32_t r = rank_of_dim[(int64_t)inst[vinst[x]].rbase + idx[p]];
        keys[p] = ((uint64_t)x << rb) | (uint64_t)r;
        vals[p] = (uint32_t)p;
    }
}

__global__ void k_canon_gather(const uint64_t *__restrict__ keys, const uint32_t *__restrict__ vals,
                               const float *__restrict__ vout, int64_t nnz, uint64_t rmask, int32_t *crank,
                               float *cval) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nnz; q += (int64_t)gridDim.x * blockDim.x) {
        crank[q] = (int32_t)(keys[q] & rmask);
        cval[q] = vout[vals[q]];
    }
}

// Partial indexing (all-pairs-1): walking x's components in rank order, b accumulates
// x[i] * maxweight_i(V) in float64; qsplit = the first component where b >= t (the
// remscore boundary for x as a query). The index split is qsplit, or 0 without partial
// indexing, or, for a queryable index, the first component where ||x_prefix||_2 reaches
// t (with a margin for the 1e-3 norm tolerance). One warp per row: the lanes load 32
// components, form their products (exact in float64) and take the running sums by a warp
// prefix scan, carried from one 32-component step to the next. The scan associates the
// terms differently from a left-to-right sum, so where b comes within rounding of t the
// split may fall one component apart from a sequential one; either is a valid split (the
// bound of the unindexed prefix stays below t up to rounding, which the float64 band of
// the decisions covers).
//
// With l2, the join's own prefix and create boundary reach to the first component where the
// norm of the leading components, summed in float32 with every operation rounded up, can
// reach t (times 1.0025 in the square for the norm tolerance of both vectors): no row scores
// t on such a prefix, so a match has a later component in common. On the 200k power-law set
// this takes the visits from 1.2e10 to 2.2e9 and the candidates from 1.6e9 to 3.4e8.
__device__ __forceinline__ double warp_incl_scan_f64(double v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

__device__ __forceinline__ float warp_incl_scan_ru(float v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v = __fadd_ru(v, y);
    }
    return v;
}

// The smallest 4-bit code c with c * PN4_STEP >= pn (the bound stays a bound).
__device__ __forceinline__ int pn4_code(float pn) {
    int c = (int)ceilf(__fdiv_ru(pn, PN4_STEP));
    if (__fmul_rd((float)c, PN4_STEP) < pn) c++;
    return min(max(c, 0), 15);
}

// The remaining-score bound's sums in float32 are off by at most (1 + 5 + chunks of 32 so far)
// roundings of 2^-24 (all terms are positive), which stays below SPLIT_F32_EPS up to component
// SPLIT_F32_MAX. A row whose first sum at t (1 - eps) is also past t (1 + eps) splits there in
// float64 too; any other that comes near t is summed again in float64 (about one row in 10^4, or
// rows of equal weights that reach t exactly). A float64 instruction takes the SM some 15 cycles a
// warp: 58M components of 1.9M rows take 1.4 ms, 1.8 with the float64 scan for every row.
constexpr float SPLIT_F32_EPS = 1e-5f;
constexpr int SPLIT_F32_MAX = 2048;

__device__ __forceinline__ float warp_incl_scan(float v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// First component where sum c * maxweight reaches t, in float64 (L: none); term(p) is component
// p's pair of the two. All lanes call it.
template <class F>
__device__ __forceinline__ int32_t split_f64(F term, int32_t L, double t, int lane) {
    double bmw = 0.0;
#pragma unroll 1
    for (int32_t base = 0; base < L; base += 32) {
        const int32_t p = base + lane;
        double v = 0.0;
        if (p < L) {
            const float2 e = term(p);
            v = (double)e.x * (double)e.y;
        }
        const double bi = bmw + warp_incl_scan_f64(v, lane);
        const unsigned hit = __ballot_sync(0xffffffffu, p < L && bi >= t);
        if (hit) return base + __ffs(hit) - 1;
        bmw = __shfl_sync(0xffffffffu, bi, 31);
    }
    return L;
}

// One chunk of 32 of the same search in float32, bmw the sum before it (brought forward): the
// component, L + 1 where float64 finds that no component of the row reaches t, L to go on.
template <class F>
__device__ __forceinline__ int32_t split_step(float v, bool in, int32_t at, float &bmw, F term, int32_t L, float t,
                                              int lane) {
    const bool tiny = t < 1e-30f;  // (products might underflow)
    const float bi = bmw + warp_incl_scan(v, lane);
    const unsigned near = __ballot_sync(0xffffffffu, in && (tiny || bi >= t * (1.f - SPLIT_F32_EPS)));
    const unsigned past = __ballot_sync(0xffffffffu, in && !tiny && bi > t * (1.f + SPLIT_F32_EPS));
    bmw = __shfl_sync(0xffffffffu, bi, 31);
    if (near == 0 && at < SPLIT_F32_MAX) return L;
    if (past && __ffs(near) == __ffs(past) && at < SPLIT_F32_MAX) return at + __ffs(near) - 1;
    const int32_t q = split_f64(term, L, (double)t, lane);
    return q < L ? q : L + 1;
}

__global__ void k_split(const int64_t *__restrict__ cptr, const int32_t *__restrict__ crank,
                        const float *__restrict__ cval, const float *__restrict__ mwr,
                        const int32_t *__restrict__ vinst, const InstDesc *__restrict__ inst, int64_t N,
                        uint32_t flags, bool l2, const float *__restrict__ mw, int32_t *split, int32_t *qsplit,
                        float *mwpre, float *mwj, int4 *vmeta, int4 *vcand, uint8_t *code, int64_t M, uint32_t *pkeys,
                        uint32_t *pvals, unsigned long long *nsuf, unsigned long long *njoin) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long nsuf_w = 0, njoin_w = 0;  // this warp's indexed components (lane 0)
    for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < N; x += nwarps) {
        const InstDesc &I = inst[vinst[x]];
        const double t = (double)I.t;
        const float t2 = __fmul_rd(I.t, I.t);
        const int64_t a = cptr[x], b = cptr[x + 1];
        const int32_t L = (int32_t)(b - a);
        const bool need_cs = (flags & APS_QUERYABLE) != 0;  // the norm-bound split of queryable indexes
        const auto term = [&](int32_t p) {
            return make_float2(cval[a + p], mwr[(int64_t)I.rbase + crank[a + p]]);
        };
        int32_t qs = L, cs = L, ls = L;
        double ss = 0.0;  // sums of the components before this step
        float bmw = 0.f, ssu = 0.f;  // the remaining-score bound; the squares, rounded up
        for (int64_t base = a; base < b && (qs == L || (need_cs && cs == L) || (l2 && ls == L)); base += 32) {
            const int64_t p = base + lane;
            float c = 0.f, mwc = 0.f;
            if (p < b) {
                c = cval[p];
                mwc = mwr[(int64_t)I.rbase + crank[p]];
            }
            const int32_t at = (int32_t)(base - a);
            if (qs == L) qs = split_step(__fmul_rn(c, mwc), p < b, at, bmw, term, L, I.t, lane);
            if (need_cs && cs == L) {
                const double si = ss + warp_incl_scan_f64((double)c * (double)c, lane);
                const unsigned hc = __ballot_sync(0xffffffffu, p < b && si * (1.0 + 2e-3) >= t * t);
                if (hc) cs = at + __ffs(hc) - 1;
                ss = __shfl_sync(0xffffffffu, si, 31);
            }
            if (l2 && ls == L) {
                const float si = __fadd_ru(ssu, warp_incl_scan_ru(__fmul_ru(c, c), lane));
                const unsigned hl = __ballot_sync(0xffffffffu, p < b && __fmul_ru(si, 1.0025f) >= t2);
                if (hl) ls = at + __ffs(hl) - 1;
                ssu = __shfl_sync(0xffffffffu, si, 31);
            }
        }
        qs = min(qs, L);
        const int32_t sp = (flags & APS_NO_PARTIAL_INDEX) ? 0 : (need_cs ? cs : qs);
        // the join's prefix (external queries only obey the norm bound) and create boundary
        const int32_t js = (l2 && !need_cs) ? max(sp, ls) : sp;
        const int32_t jq = l2 ? max(qs, ls) : qs;
        // maxweight(x') of the split and of the join's prefix, and an upper bound of the join prefix's norm (float32 with
        // every operation rounded up, so the bound can only come out above the exact norm;
        // times 1 + 1.1e-3 for the 1e-3 norm tolerance of the vectors it will be dotted with)
        float best = 0.f, bestj = 0.f, pss = 0.f;
        for (int64_t p = a + lane; p < a + js; p += 32) {
            const float c = cval[p];
            if (p < a + sp) best = fmaxf(best, c);
            bestj = fmaxf(bestj, c);
            pss = __fmaf_ru(c, c, pss);
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
            bestj = fmaxf(bestj, __shfl_xor_sync(0xffffffffu, bestj, o));
            pss = __fadd_ru(pss, __shfl_xor_sync(0xffffffffu, pss, o));
        }
        if (lane == 0) {
            const float pn = js ? __fmul_ru(__fsqrt_ru(pss), 1.0011f) : 0.f;
            const int32_t rlim = js < L ? crank[a + js] : 0x7fffffff;
            split[x] = sp;
            qsplit[x] = qs;
            mwpre[x] = best;
            if (mwj) mwj[x] = bestj;
            vmeta[x] = make_int4((int32_t)a, L, jq, __float_as_int(mw[x]));
            vcand[x] = make_int4((int32_t)a, js, rlim, __float_as_int(pn));
            code[x] = (uint8_t)((rank_bucket(rlim) >> 2) << 4 | pn4_code(pn));
            nsuf_w += (unsigned long long)(L - sp);
            njoin_w += (unsigned long long)(L - js);
        }
        // the row's posting keys: an indexed entry its global rank, a prefix entry a sentinel
        // past the last rank (it sorts last); the value is the entry's index. The sort is
        // stable and entries arrive in row order, so every list comes out in increasing id.
        for (int64_t p = a + lane; p < b; p += 32) {
            pkeys[p] = (p - a >= js) ? (uint32_t)I.rbase + (uint32_t)crank[p] : (uint32_t)M;
            pvals[p] = (uint32_t)p;
        }
    }
    __shared__ unsigned long long bsum[2];
    if (threadIdx.x < 2) bsum[threadIdx.x] = 0ull;
    __syncthreads();
    if (lane == 0) {
        atomicAdd(&bsum[0], nsuf_w);
        atomicAdd(&bsum[1], njoin_w);
    }
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(nsuf, bsum[0]);
    if (threadIdx.x == 1) atomicAdd(njoin, bsum[1]);
}

// Posting keys by a given split (for the exported lists), one thread per component.
__global__ void k_post_keys(const int64_t *__restrict__ cptr, const int32_t *__restrict__ crank,
                            const int32_t *__restrict__ erow, const int32_t *__restrict__ vinst,
                            const InstDesc *__restrict__ inst, const int32_t *__restrict__ split, int64_t nnz,
                            int64_t M, uint32_t *pkeys, uint32_t *pvals) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x) {
        const int64_t x = erow[p];
        pkeys[p] = (p - cptr[x] >= split[x]) ? (uint32_t)inst[vinst[x]].rbase + (uint32_t)crank[p] : (uint32_t)M;
        pvals[p] = (uint32_t)p;
    }
}

// The row of every component.
__global__ void k_rows_of(const int64_t *__restrict__ cptr, int64_t N, int32_t *erow) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < N; x += nwarps)
        for (int64_t p = cptr[x] + lane; p < cptr[x + 1]; p += 32) erow[p] = (int32_t)x;
}

__global__ void k_post_fill(const uint32_t *__restrict__ vals, const int32_t *__restrict__ erow,
                            const float *__restrict__ cval, const int32_t *__restrict__ len,
                            const int32_t *__restrict__ vinst, const InstDesc *__restrict__ inst, int64_t nsuf,
                            int2 *post) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nsuf; q += (int64_t)gridDim.x * blockDim.x) {
        uint32_t p = vals[q];
        int64_t x = erow[p];
        const InstDesc &I = inst[vinst[x]];
        const int32_t lid = (int32_t)(x - I.vbase);
        const int32_t tag = I.packed ? (min(len[x], 255) << 24) : 0;
        post[q] = make_int2(lid | tag, __float_as_int(cval[p]));
    }
}

// List pointers from the sorted posting keys: lptr[R] = first suffix entry with key >= R
// (binary search; lptr[M] = nsuf).
// `inst`, when given, takes a single instance's description with its windows (no copy from the host).
__global__ void k_lptr(const uint32_t *__restrict__ keys, int64_t nsuf, int64_t M, int64_t *lptr, InstDesc one,
                       InstDesc *inst) {
    if (inst && blockIdx.x == 0 && threadIdx.x == 0) *inst = one;
    for (int64_t R = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; R <= M; R += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = nsuf;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (keys[mid] < (uint32_t)R) lo = mid + 1; else hi = mid;
        }
        lptr[R] = lo;
    }
}

// Interleaved rows read by the join.
__global__ void k_pack(const int32_t *__restrict__ crank, const float *__restrict__ cval, int64_t nnz, int2 *crow) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < nnz; p += stride)
        crow[p] = make_int2(crank[p], __float_as_int(cval[p]));
}

// Where the windows of a multi-window instance begin inside each list: w[i] = the position in
// post of list R's first entry with local id >= i * W (lists are in increasing id; binary
// search). One thread per window of a list, in the order they are stored, instances over
// blockIdx.y: with a warp per list, 12 windows left 20 lanes idle (25M lists of a batch of 512
// instances: 1.07 ms, 0.33 now).
__global__ void k_wptr(const InstDesc *__restrict__ inst, int k, const int64_t *__restrict__ lptr,
                       const int2 *__restrict__ post, uint32_t *wptr) {
    const int lane = threadIdx.x & 31;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int q = blockIdx.y; q < k; q += gridDim.y) {
        const InstDesc &I = inst[q];
        if (I.nw <= 1) continue;
        const int32_t idmask = I.packed ? 0x00ffffff : 0x7fffffff;
        const uint32_t per = (uint32_t)I.nw + 1u;
        const int64_t total = (int64_t)I.m * per;
        uint32_t *w = wptr + I.wbase;
        for (int64_t e0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; e0 < total; e0 += step) {
            const int64_t r0 = e0 / per;  // one long division a warp
            const uint32_t off = (uint32_t)(e0 - r0 * per) + (uint32_t)lane;
            const int64_t r = r0 + off / per, e = e0 + lane;
            if (e >= total) continue;
            const int64_t bound = (int64_t)(off % per) * I.W;
            int64_t lo = lptr[I.rbase + r], hi = lptr[I.rbase + r + 1];
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if ((post[mid].x & idmask) < bound) lo = mid + 1; else hi = mid;
            }
            w[e] = (uint32_t)lo;
        }
    }
}

dim3 wptr_grid(int32_t maxm, int32_t maxnw, int k) {
    const int64_t blocks = ((int64_t)maxm * (maxnw + 1) + T256 - 1) / T256;
    return dim3((unsigned)std::max<int64_t>(1, std::min<int64_t>(blocks, 65536 / k)), (unsigned)std::min(k, 65535));
}

// The same per list (wlist): how many starts each list has, where they begin, and the starts, one
// thread each.
__global__ void k_wlist_counts(const InstDesc *__restrict__ inst, int k, const int64_t *__restrict__ lptr, int64_t M,
                               int per, int32_t *cnt) {
    for (int64_t R = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; R < M; R += (int64_t)gridDim.x * blockDim.x) {
        const int nw = inst[inst_of_rank(inst, k, R)].nw;
        const int groups = window_groups(nw, list_shift(lptr[R + 1] - lptr[R], nw, per));
        cnt[R] = groups > 1 ? groups + 1 : 0;
    }
}

__global__ void k_wlist(const InstDesc *__restrict__ inst, int k, const int64_t *__restrict__ lptr,
                        const int64_t *__restrict__ off, int64_t M, int per, uint64_t *wlist) {
    for (int64_t R = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; R < M; R += (int64_t)gridDim.x * blockDim.x)
        wlist[R] = (uint64_t)off[R] << 6 |
                   (uint64_t)list_shift(lptr[R + 1] - lptr[R], inst[inst_of_rank(inst, k, R)].nw, per);
}

__global__ void k_wlist_starts(const InstDesc *__restrict__ inst, int k, const int64_t *__restrict__ lptr,
                               const int2 *__restrict__ post, const int64_t *__restrict__ off,
                               const uint64_t *__restrict__ wlist, int64_t M, int64_t total, uint32_t *wptr) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        int64_t a = 0, b = M;  // the last list that begins at or before e (those without starts begin where the next does)
        while (a < b) {
            const int64_t mid = (a + b) >> 1;
            if (off[mid] <= e) a = mid + 1; else b = mid;
        }
        const int64_t R = a - 1;
        const InstDesc &I = inst[inst_of_rank(inst, k, R)];
        const int32_t idmask = I.packed ? 0x00ffffff : 0x7fffffff;
        const int64_t bound = ((e - off[R]) << (wlist[R] & 63)) * I.W;
        int64_t lo = lptr[R], hi = lptr[R + 1];
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if ((post[mid].x & idmask) < bound) lo = mid + 1; else hi = mid;
        }
        wptr[e] = (uint32_t)lo;
    }
}

// The table of window starts of the lists (lptr, post), in the form that the build chose.
aps_status window_starts(const aps_index *ix, const DBuf<int64_t> &lptr, const DBuf<int2> &post, DBuf<uint32_t> &wptr,
                         DBuf<uint64_t> &wlist, cudaStream_t s) {
    const InstDesc *const inst = ix->d.inst.p;
    const int64_t M = ix->M;
    if (ix->wper < 0) {
        APS_TRY(wptr.alloc((size_t)std::max<int64_t>(ix->nwptr, 1), s));
        if (ix->nwptr) {
            k_wptr<<<wptr_grid(ix->maxm, ix->maxnw, ix->k), T256, 0, s>>>(inst, ix->k, lptr.p, post.p, wptr.p);
            APS_LAUNCH_CHECK();
        }
        return APS_OK;
    }
    DBuf<int32_t> cnt;
    DBuf<int64_t> off;
    APS_TRY(cnt.alloc((size_t)M, s));
    APS_TRY(off.alloc((size_t)M + 1, s));
    APS_TRY(wlist.alloc((size_t)M, s));
    k_wlist_counts<<<grid_for(M, T256), T256, 0, s>>>(inst, ix->k, lptr.p, M, ix->wper, cnt.p);
    APS_LAUNCH_CHECK();
    APS_TRY(scan_exclusive(cnt.p, off.p, M, s));
    int64_t total = 0;
    APS_CUDA(cudaMemcpyAsync(&total, off.p + M, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    APS_CUDA(cudaStreamSynchronize(s));
    APS_TRY(wptr.alloc((size_t)std::max<int64_t>(total, 1), s));
    k_wlist<<<grid_for(M, T256), T256, 0, s>>>(inst, ix->k, lptr.p, off.p, M, ix->wper, wlist.p);
    APS_LAUNCH_CHECK();
    if (total) {
        k_wlist_starts<<<grid_for(total, T256), T256, 0, s>>>(inst, ix->k, lptr.p, post.p, off.p, wlist.p, M, total,
                                                              wptr.p);
        APS_LAUNCH_CHECK();
    }
    return APS_OK;
}

// Join work list: every vector with later candidates in its instance, keyed by
// (class, decreasing estimated cost) so that the persistent join takes the most expensive
// queries first (least-loaded-first idea of the vertical algorithm's binning). Classes 0-3
// are the instance's tile shape (G = 1, 2, 4, 8); class 4 holds the vectors with one or two
// components, which the join streams one warp per vector.
constexpr int ITEM_COST_BITS = 13;
__global__ void k_item_keys(const int64_t *__restrict__ cptr, const int32_t *__restrict__ crank,
                            const int64_t *__restrict__ lptr, const int32_t *__restrict__ vinst,
                            const InstDesc *__restrict__ inst, int64_t N, uint32_t *keys, uint32_t *vals,
                            unsigned long long *class_count) {
    // one warp per vector: the lanes read its ranks side by side and look up their lists;
    // the class counts go through shared memory (one global atomic per class and block)
    __shared__ unsigned long long ccount[JOIN_NCLS];
    if (threadIdx.x < JOIN_NCLS) ccount[threadIdx.x] = 0ull;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < N; x += nwarps) {
        const InstDesc &I = inst[vinst[x]];
        const int64_t lx = x - I.vbase;
        if (lx >= (int64_t)I.n - 1) {  // no later candidates: after every class
            if (lane == 0) {
                keys[x] = (uint32_t)JOIN_NCLS << ITEM_COST_BITS;
                vals[x] = (uint32_t)x;
            }
            continue;
        }
        const int64_t a = cptr[x], b = cptr[x + 1];
        int64_t lsum = 0;  // total length of x's posting lists
        for (int64_t p = a + lane; p < b; p += 32) {
            const int64_t R = (int64_t)I.rbase + crank[p];
            lsum += lptr[R + 1] - lptr[R];
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        if (lane == 0) {
            const float later = (float)(I.n - 1 - lx);
            const float cost = (float)lsum * (later / (float)I.n) + later * 0.125f + 32.f;
            // decreasing cost inside the class: the exponent and seven bits of the mantissa (costs
            // are 32 to 2^63), so that the sort takes two passes instead of four
            const uint32_t c = min((__float_as_uint(cost) - __float_as_uint(32.f)) >> 16, (1u << ITEM_COST_BITS) - 1u);
            // (a merge of two long lists would be one warp's serial tail: those go by windows; 200,000
            // rows with the line at 1024 / 8192 / 65536 entries / none: 21.9 / 21.6 / 22.0 / 22.0 ms)
            const int cls = b - a <= 1 || (b - a == 2 && lsum <= 8192) ? 4 : I.G == 1 ? 0 : I.G == 2 ? 1 : I.G == 4 ? 2 : 3;
            keys[x] = ((uint32_t)cls << ITEM_COST_BITS) | ((1u << ITEM_COST_BITS) - 1u - c);
            vals[x] = (uint32_t)x;
            atomicAdd(&ccount[cls], 1ull);
        }
    }
    __syncthreads();
    if (threadIdx.x < JOIN_NCLS && ccount[threadIdx.x]) atomicAdd(&class_count[threadIdx.x], ccount[threadIdx.x]);
}

__global__ void k_take_vals(const uint32_t *__restrict__ vals, int64_t n, int32_t *out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (int32_t)vals[i];
}

const char *code_name(int c) {
    switch (c) {
        case E_PTR: return "row pointers decrease or exceed nnz";
        case E_IDX_RANGE: return "dimension index out of [0, m)";
        case E_IDX_ORDER: return "dimension indices not strictly increasing";
        case E_VALUE: return "value not finite and > 0";
        case E_NORM: return "row L2 norm differs from 1 by more than 1e-3 (pass APS_NORMALIZE), or exceeds 1 + 1e-3 "
                            "with APS_SUBUNIT_NORMS";
        default: return "invalid input";
    }
}

}  // namespace

namespace {

constexpr int64_t WPTR_LARGE = 64 << 20;  // (asking for the free memory takes the host some 10 us)

// Device memory that an allocation can have: free, or kept by the pool without being used.
size_t memory_at_hand() {
    size_t fr = 0, tot = 0;
    if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) {
        cudaGetLastError();
        return SIZE_MAX;
    }
    int dev = 0;
    cudaMemPool_t pool;
    uint64_t kept = 0, used = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess &&
        cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &kept) == cudaSuccess &&
        cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) == cudaSuccess && kept > used)
        fr += kept - used;
    return fr;
}

}  // namespace

aps_status build_index_device(aps_index *ix, const int64_t *indptr, const int32_t *idx, const float *val,
                              const std::vector<InstDesc> &inst_in, cudaStream_t s, const aps_tuning *tune) {
    const int k = (int)inst_in.size();
    ix->k = k;
    ix->stream = s;
    // ---- host-side layout of instances: ranks, windows, classes
    std::vector<InstDesc> inst = inst_in;
    int64_t N = 0, M = 0, arena_slots = 0;
    int32_t maxm = 1, maxn = 1;
    // tile shape per instance: G query groups per CTA from the size-bucket table (its
    // queryable column for indexes built to answer queries)
    const aps_tuning tu = tune ? *tune : tuning_current();
    const int32_t *gtab = (ix->flags & APS_QUERYABLE) ? tu.query_groups : tu.groups;
    for (int i = 0; i < k; i++) {
        InstDesc &I = inst[i];
        I.vbase = N;
        I.rbase = (int32_t)M;
        I.G = gtab[tune_bucket(I.n)];
        I.packed = I.n < (1 << 24) ? 1 : 0;
        arena_slots += (int64_t)I.n * (((int64_t)I.n * I.G + 40959) / 40960);
        N += I.n;
        M += I.m;
        maxm = std::max(maxm, I.m);
        maxn = std::max(maxn, I.n);
    }
    if (M >= (1ll << 31) || N >= (1ll << 31)) {
        set_error("too many vectors or dimensions (limit 2^31 - 1)");
        return APS_EINVAL;
    }
    ix->N = N;
    ix->M = M;
    ix->arena_slots = arena_slots;
    ix->maxm = maxm;
    // every bound on: the join may keep the norm-bounded prefixes to itself
    ix->l2 = !(ix->flags & (APS_NO_PARTIAL_INDEX | APS_NO_MINSIZE | APS_NO_REMSCORE | APS_NO_UPPERBOUND));
    IndexArrays &d = ix->d;

    // the first and the last row pointer, as one strided copy where its pitch may be that wide
    int64_t ends[2] = {0, 0};
    if (N >= 1 && N < ((int64_t)1 << 27)) {
        APS_CUDA(cudaMemcpy2DAsync(ends, sizeof(int64_t), indptr, sizeof(int64_t) * (size_t)N, sizeof(int64_t), 2,
                                   cudaMemcpyDeviceToHost, s));
    } else {
        APS_CUDA(cudaMemcpyAsync(&ends[0], indptr, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        APS_CUDA(cudaMemcpyAsync(&ends[1], indptr + N, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    }
    APS_CUDA(cudaStreamSynchronize(s));
    const int64_t first = ends[0], nnz = ends[1];
    if (first != 0 || nnz < 0 || nnz >= (1ll << 31)) {
        set_error("indptr[0] must be 0 and nnz in [0, 2^31); got indptr[0]=%lld nnz=%lld",
                  (long long)first, (long long)nnz);
        return APS_EINVAL;
    }
    ix->nnz = nnz;
    Carver cv;
    cv.s = s;
    for (int pass = 0; pass < 2; pass++) {
        cv.off = 0;
        cv.put(d.inst, (size_t)k);
        cv.put(d.vinst, (size_t)N);
        cv.put(d.cptr, (size_t)N + 1);
        cv.put(d.len, (size_t)N);
        cv.put(d.mw, (size_t)N);
        cv.put(d.split, (size_t)N);
        cv.put(d.qsplit, (size_t)N);
        cv.put(d.mwpre, (size_t)N);
        if (ix->l2) cv.put(d.mwj, (size_t)N);
        cv.put(d.crank, (size_t)nnz);
        cv.put(d.cval, (size_t)nnz);
        cv.put(d.nnz_d, (size_t)M);
        cv.put(d.mw_d, (size_t)M);
        cv.put(d.mwr, (size_t)M);
        cv.put(d.rank_of_dim, (size_t)M);
        cv.put(d.dim_of_rank, (size_t)M);
        cv.put(d.lptr, (size_t)M + 1);
        cv.put(d.vmeta, (size_t)N);
        cv.put(d.vcand, (size_t)N);
        cv.put(d.code, (size_t)N);
        if (pass == 0) {
            APS_TRY(d.block.alloc(cv.off, s));
            cv.base = d.block.p;
        }
    }
    DBuf<char> tblock;
    DBuf<int32_t> erow;
    DBuf<float> vout;
    DBuf<unsigned long long> err;  // {first bad row, components indexed by split, longest row, in the join's lists}, classes
    cv.base = nullptr;
    for (int pass = 0; pass < 2; pass++) {
        cv.off = 0;
        cv.put(erow, (size_t)nnz);
        cv.put(vout, (size_t)nnz);
        cv.put(err, 4 + JOIN_NCLS);
        if (pass == 0) {
            APS_TRY(tblock.alloc(cv.off, s));
            cv.base = tblock.p;
        }
    }
    if (k > 1) APS_CUDA(cudaMemcpyAsync(d.inst.p, inst.data(), sizeof(InstDesc) * k, cudaMemcpyHostToDevice, s));

    const unsigned gE = grid_for(nnz, T256), gM = grid_for(M, T256);
    // ---- a1: validation, |x|, maxweight(x), per-dimension statistics
    k_setup<<<grid_for(std::max<int64_t>(N + 1, M), T256), T256, 0, s>>>(
        indptr, inst[0], d.inst.p, k, N, M, d.cptr.p, d.vinst.p, d.nnz_d.p, d.mw_d.p, err.p, 4 + JOIN_NCLS);
    APS_LAUNCH_CHECK();
    k_validate<<<rows_grid(N), T256, 0, s>>>(indptr, idx, val, d.vinst.p, d.inst.p, 0, N, nnz, ix->flags, erow.p,
                                             vout.p, d.len.p, d.mw.p, err.p, err.p + 2);
    APS_LAUNCH_CHECK();
    unsigned long long e3[3] = {~0ull, 0ull, 0ull};  // first error, (unused here), longest row
    APS_CUDA(cudaMemcpyAsync(e3, err.p, sizeof(e3), cudaMemcpyDeviceToHost, s));
    APS_CUDA(cudaStreamSynchronize(s));
    const unsigned long long e_h = e3[0], longest_row = e3[2];
    if (e_h != ~0ull) {
        long long row = (long long)(e_h >> 8);
        int code = (int)(e_h & 0xff);
        int inst_id = 0;
        for (int i = 0; i < k; i++)
            if (inst[i].vbase <= row) inst_id = i;
        if (k > 1)
            set_error("invalid input in instance %d, row %lld: %s", inst_id, row - (long long)inst[inst_id].vbase,
                      code_name(code));
        else
            set_error("invalid input at row %lld: %s", row, code_name(code));
        return APS_EINVAL;
    }
    // windows, and the table of their starts with every window
    int64_t nwptr = 0;
    int32_t maxnw = 1;
    const auto set_windows = [&](int halvings) {
        nwptr = 0;
        maxnw = 1;
        for (InstDesc &I : inst) {
            I.W = tile_window(I.G) >> halvings;
            I.nw = I.n > 0 ? (int32_t)(((int64_t)I.n + I.W - 1) / I.W) : 0;
            I.wbase = nwptr;
            if (I.nw > 1) nwptr += (int64_t)I.m * (I.nw + 1);
            maxnw = std::max(maxnw, I.nw);
        }
    };
    int halvings = 0;
    while (halvings < WINDOW_HALVINGS && N < WINDOWS_LEAST * (tile_window(2) >> halvings)) halvings++;
    const bool uneven = longest_row > (unsigned long long)(8 * nnz / std::max<int64_t>(N, 1));
    if (uneven && halvings > 0) halvings = std::min(halvings + 1, WINDOW_HALVINGS);
    set_windows(halvings);
    if (maxnw < 4) set_windows(halvings = 0);  // (too few to be cut all the same)
    while (halvings > 0 && 4 * nwptr > window_bytes(nnz, M)) set_windows(--halvings);  // (wide tables: wide windows)
    ix->nwptr = nwptr;
    ix->maxnw = maxnw;
    // A heavy vector's windows go to several warps where there are few vectors (2M slots at most)
    // and enough windows for it: a vector's tables cost a unit about as much as a window does. (Join
    // ms with 1 / 4 / 8 / 16 / 32 parts: 30,000 power-law rows 5.6 / 2.2 / 1.68 / 1.75 / 1.78, 200,000
    // rows 26.1 / 22.1 / 21.7 / 21.6 / 21.6.)
    ix->parts = maxnw < 4 ? 1 : (int32_t)std::max<int64_t>(1, std::min<int64_t>({16, maxnw, ((int64_t)1 << 21) / std::max<int64_t>(N, 1)}));
    ix->inst_h = inst;
    // the table of window starts: every window's where that takes no more than its share and, when it
    // is large, an eighth of the memory at hand; else by list
    if (4 * nwptr > window_bytes(nnz, M) || (4 * nwptr > WPTR_LARGE && (uint64_t)nwptr > memory_at_hand() / 32)) {
        ix->wper = WLIST_ENTRIES;
        const uint64_t room = memory_at_hand() / 32;
        while (ix->wper > 0 && (uint64_t)ix->wper * (uint64_t)nnz * 4 > WPTR_LARGE && (uint64_t)ix->wper * (uint64_t)nnz > room)
            ix->wper /= 2;
    }
    if (nnz > 0 && k > 1 && maxm <= DIMSTATS_DIMS) {  // a batch of small instances: one CTA each
        const int sm = (int)(sizeof(uint32_t) * (size_t)maxm);
        // (the kernel's limit is shared by every thread: the same for every batch)
        APS_CUDA(cudaFuncSetAttribute(k_dimstats_inst, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)sizeof(uint32_t) * DIMSTATS_DIMS));
        k_dimstats_inst<<<k, 1024, sm, s>>>(d.cptr.p, idx, vout.p, d.inst.p, d.nnz_d.p, d.mw_d.p);
        APS_LAUNCH_CHECK();
    } else if (nnz > 0) {
        k_dimstats<<<gE, T256, 0, s>>>(idx, vout.p, erow.p, d.vinst.p, d.inst.p, nnz, d.nnz_d.p, d.mw_d.p);
        APS_LAUNCH_CHECK();
    }
    // ---- a2: dimension ranks and rank-ordered rows
    {
        DBuf<uint32_t> vals;
        if (bits_for((uint64_t)maxn) + bits_for((uint64_t)(k - 1)) <= 32)
            APS_TRY(sort_dims<uint32_t>(ix, maxn, vals, s));
        else
            APS_TRY(sort_dims<uint64_t>(ix, maxn, vals, s));
        k_rank_scatter<<<gM, T256, 0, s>>>(vals.p, d.inst.p, k, M, d.mw_d.p, d.rank_of_dim.p, d.dim_of_rank.p,
                                           d.mwr.p);
        APS_LAUNCH_CHECK();
    }
    if (nnz > 0 && longest_row <= 64) {  // every row sorted inside one warp
        k_canon_rows64<<<rows_grid(N), T256, 0, s>>>(d.cptr.p, idx, vout.p, d.vinst.p, d.inst.p,
                                                               d.rank_of_dim.p, N, d.crank.p, d.cval.p);
        APS_LAUNCH_CHECK();
    } else if (nnz > 0) {  // a global sort by (row, rank)
        DBuf<uint64_t> keys;
        DBuf<uint32_t> vals;
        APS_TRY(keys.alloc((size_t)nnz, s));
        APS_TRY(vals.alloc((size_t)nnz, s));
        int rb = bits_for((uint64_t)(maxm - 1));
        if (rb == 0) rb = 1;
        k_canon_keys<<<gE, T256, 0, s>>>(idx, erow.p, d.vinst.p, d.inst.p, d.rank_of_dim.p, nnz, rb, keys.p, vals.p);
        APS_LAUNCH_CHECK();
        APS_TRY(sort_pairs(keys, vals, nnz, rb + bits_for((uint64_t)(N - 1)), s));
        k_canon_gather<<<gE, T256, 0, s>>>(keys.p, vals.p, vout.p, nnz, (1ull << rb) - 1, d.crank.p, d.cval.p);
        APS_LAUNCH_CHECK();
    }
    // ---- a3: partial-indexing split
    // the split also writes each row's posting keys for a4 (and counts the indexed components)
    DBuf<uint32_t> pkeys;
    DBuf<uint32_t> pvals;
    APS_TRY(pkeys.alloc((size_t)std::max<int64_t>(nnz, 1), s));
    APS_TRY(pvals.alloc((size_t)std::max<int64_t>(nnz, 1), s));
    unsigned long long *nsuf_d = err.p + 1;
    k_split<<<rows_grid(N), T256, 0, s>>>(d.cptr.p, d.crank.p, d.cval.p, d.mwr.p, d.vinst.p, d.inst.p, N,
                                                    ix->flags, ix->l2, d.mw.p, d.split.p, d.qsplit.p, d.mwpre.p,
                                                    d.mwj.p, d.vmeta.p, d.vcand.p, d.code.p, M, pkeys.p, pvals.p, nsuf_d,
                                                    nsuf_d + 2);
    APS_LAUNCH_CHECK();
    // ---- a4: suffix inverted index
    {
        DBuf<uint32_t> &keys = pkeys;
        DBuf<uint32_t> &vals = pvals;
        unsigned long long cnt3[3] = {0, 0, 0};  // by split, (longest row), in the join's lists
        // (a batch's descriptions with their windows; waited for here, as `inst` goes with this call)
        if (k > 1) APS_CUDA(cudaMemcpyAsync(d.inst.p, inst.data(), sizeof(InstDesc) * k, cudaMemcpyHostToDevice, s));
        APS_CUDA(cudaMemcpyAsync(cnt3, nsuf_d, sizeof(cnt3), cudaMemcpyDeviceToHost, s));
        APS_CUDA(cudaStreamSynchronize(s));
        ix->nsuf = (int64_t)cnt3[0];
        ix->njoin = (int64_t)cnt3[2];
        if (nnz > 0) APS_TRY(sort_pairs(keys, vals, nnz, bits_for((uint64_t)M), s));
        APS_TRY(d.post.alloc((size_t)std::max<int64_t>(ix->njoin, 1), s));
        if (ix->njoin > 0) {
            k_post_fill<<<grid_for(ix->njoin, T256), T256, 0, s>>>(vals.p, erow.p, d.cval.p, d.len.p, d.vinst.p,
                                                                   d.inst.p, ix->njoin, d.post.p);
            APS_LAUNCH_CHECK();
        }
        k_lptr<<<grid_for(M + 1, T256), T256, 0, s>>>(keys.p, ix->njoin, M, d.lptr.p, inst[0], k == 1 ? d.inst.p : nullptr);
        APS_LAUNCH_CHECK();
        APS_TRY(window_starts(ix, d.lptr, d.post, d.wptr, d.wlist, s));
        APS_TRY(d.crow.alloc((size_t)std::max<int64_t>(nnz, 1), s));
        if (nnz > 0) {
            k_pack<<<gE, T256, 0, s>>>(d.crank.p, d.cval.p, nnz, d.crow.p);
            APS_LAUNCH_CHECK();
        }
    }
    // ---- join work list
    {
        DBuf<uint32_t> keys, vals;
        APS_TRY(keys.alloc((size_t)std::max<int64_t>(N, 1), s));
        APS_TRY(vals.alloc((size_t)std::max<int64_t>(N, 1), s));
        unsigned long long *cc = err.p + 4;  // one counter per class
        if (N > 0) {
            k_item_keys<<<rows_grid(N), T256, 0, s>>>(d.cptr.p, d.crank.p, d.lptr.p, d.vinst.p, d.inst.p,
                                                               N, keys.p, vals.p,
                                            cc);
            APS_LAUNCH_CHECK();
            APS_TRY(sort_pairs(keys, vals, N, 3 + ITEM_COST_BITS, s));
        }
        unsigned long long cnt_h[JOIN_NCLS] = {};
        APS_CUDA(cudaMemcpyAsync(cnt_h, cc, sizeof(cnt_h), cudaMemcpyDeviceToHost, s));
        APS_CUDA(cudaStreamSynchronize(s));
        int64_t acc = 0;
        for (int c = 0; c < JOIN_NCLS; c++) {
            ix->class_begin[c] = acc;
            acc += (int64_t)cnt_h[c];
        }
        ix->class_begin[JOIN_NCLS] = acc;
        APS_TRY(ix->items.alloc((size_t)std::max<int64_t>(acc, 1), s));
        if (acc > 0) {
            k_take_vals<<<grid_for(acc, T256), T256, 0, s>>>(vals.p, acc, ix->items.p);
            APS_LAUNCH_CHECK();
        }
    }
    APS_CUDA(cudaStreamSynchronize(s));
    return APS_OK;
}

aps_status export_postings(const aps_index *ix, DBuf<int64_t> &lptr, DBuf<int2> &post, cudaStream_t s) {
    const IndexArrays &d = ix->d;
    DBuf<uint32_t> keys, vals;
    DBuf<int32_t> erow;
    APS_TRY(keys.alloc((size_t)std::max<int64_t>(ix->nnz, 1), s));
    APS_TRY(vals.alloc((size_t)std::max<int64_t>(ix->nnz, 1), s));
    APS_TRY(erow.alloc((size_t)std::max<int64_t>(ix->nnz, 1), s));
    APS_TRY(lptr.alloc((size_t)ix->M + 1, s));
    APS_TRY(post.alloc((size_t)std::max<int64_t>(ix->nsuf, 1), s));
    if (ix->nnz > 0) {
        k_rows_of<<<grid_for(ix->N * 32, T256), T256, 0, s>>>(d.cptr.p, ix->N, erow.p);
        APS_LAUNCH_CHECK();
        k_post_keys<<<grid_for(ix->nnz, T256), T256, 0, s>>>(d.cptr.p, d.crank.p, erow.p, d.vinst.p, d.inst.p,
                                                             d.split.p, ix->nnz, ix->M, keys.p, vals.p);
        APS_LAUNCH_CHECK();
        APS_TRY(sort_pairs(keys, vals, ix->nnz, bits_for((uint64_t)ix->M), s));
    }
    if (ix->nsuf > 0) {
        k_post_fill<<<grid_for(ix->nsuf, T256), T256, 0, s>>>(vals.p, erow.p, d.cval.p, d.len.p, d.vinst.p, d.inst.p,
                                                              ix->nsuf, post.p);
        APS_LAUNCH_CHECK();
    }
    k_lptr<<<grid_for(ix->M + 1, T256), T256, 0, s>>>(keys.p, ix->nsuf, ix->M, lptr.p, ix->inst_h[0], nullptr);
    APS_LAUNCH_CHECK();
    return APS_OK;
}

aps_status build_block_index(const aps_index *ix, BlockIndex &b, cudaStream_t s) {
    const IndexArrays &d = ix->d;
    const int64_t N = ix->N, M = ix->M, nnz = ix->nnz;
    DBuf<int32_t> split, qsplit, erow;
    DBuf<float> mwpre;
    DBuf<uint32_t> keys, vals;
    DBuf<unsigned long long> sums;
    APS_TRY(split.alloc((size_t)N, s));
    APS_TRY(qsplit.alloc((size_t)N, s));
    APS_TRY(mwpre.alloc((size_t)N, s));
    APS_TRY(erow.alloc((size_t)nnz, s));
    APS_TRY(keys.alloc((size_t)nnz, s));
    APS_TRY(vals.alloc((size_t)nnz, s));
    APS_TRY(sums.alloc(2, s));
    APS_TRY(b.vmeta.alloc((size_t)N, s));
    APS_TRY(b.vcand.alloc((size_t)N, s));
    APS_TRY(b.code.alloc((size_t)N, s));
    APS_TRY(b.lptr.alloc((size_t)M + 1, s));
    APS_TRY(b.post.alloc((size_t)ix->nsuf, s));
    if (N == 0 || nnz == 0) return APS_OK;  // (nothing to join)
    APS_CUDA(cudaMemsetAsync(sums.p, 0, 2 * sizeof(unsigned long long), s));
    k_split<<<rows_grid(N), T256, 0, s>>>(d.cptr.p, d.crank.p, d.cval.p, d.mwr.p, d.vinst.p, d.inst.p, N, ix->flags,
                                          false, d.mw.p, split.p, qsplit.p, mwpre.p, nullptr, b.vmeta.p, b.vcand.p, b.code.p, M,
                                          keys.p, vals.p, sums.p, sums.p + 1);
    APS_LAUNCH_CHECK();
    k_rows_of<<<grid_for(N * 32, T256), T256, 0, s>>>(d.cptr.p, N, erow.p);
    APS_LAUNCH_CHECK();
    APS_TRY(sort_pairs(keys, vals, nnz, bits_for((uint64_t)M), s));
    if (ix->nsuf > 0) {  // (the components from the splits on, as counted by the build)
        k_post_fill<<<grid_for(ix->nsuf, T256), T256, 0, s>>>(vals.p, erow.p, d.cval.p, d.len.p, d.vinst.p, d.inst.p,
                                                              ix->nsuf, b.post.p);
        APS_LAUNCH_CHECK();
    }
    k_lptr<<<grid_for(M + 1, T256), T256, 0, s>>>(keys.p, ix->nsuf, M, b.lptr.p, ix->inst_h[0], nullptr);
    APS_LAUNCH_CHECK();
    return window_starts(ix, b.lptr, b.post, b.wptr, b.wlist, s);
}

// ------------------------------------------------------------------ external queries
namespace {

template <class K>
__global__ void k_q_keys(const int32_t *__restrict__ qidx, const int32_t *__restrict__ erow,
                         const int32_t *__restrict__ rank_of_dim, int64_t nnz, int rb, K *keys, uint32_t *vals) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x) {
        keys[p] = (K)(((uint64_t)erow[p] << rb) | (uint64_t)rank_of_dim[qidx[p]]);
        vals[p] = (uint32_t)p;
    }
}

template <class K>
__global__ void k_q_gather(const K *__restrict__ keys, const uint32_t *__restrict__ vals,
                           const float *__restrict__ vout, int64_t nnz, uint64_t rmask, int2 *crow) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nnz; q += (int64_t)gridDim.x * blockDim.x)
        crow[q] = make_int2((int32_t)(keys[q] & rmask), __float_as_int(vout[vals[q]]));
}

// The query rows over the index's ranks, in rank order (keys: row, rank).
template <class K>
aps_status sort_queries(const int32_t *qidx, const int32_t *erow, const int32_t *rank_of_dim, const float *vout,
                        int64_t nnz, int rb, int bits, int2 *crow, cudaStream_t s) {
    DBuf<K> keys;
    DBuf<uint32_t> vals;
    APS_TRY(keys.alloc((size_t)nnz, s));
    APS_TRY(vals.alloc((size_t)nnz, s));
    k_q_keys<K><<<grid_for(nnz, T256), T256, 0, s>>>(qidx, erow, rank_of_dim, nnz, rb, keys.p, vals.p);
    APS_LAUNCH_CHECK();
    APS_TRY(sort_pairs(keys, vals, nnz, bits, s));
    k_q_gather<K><<<grid_for(nnz, T256), T256, 0, s>>>(keys.p, vals.p, vout, nnz, (1ull << rb) - 1, crow);
    APS_LAUNCH_CHECK();
    return APS_OK;
}

// Remscore boundary of a query: the first rank-ordered component where
// sum x[i] * maxweight_i(V) reaches t (exact as float64 is, as for indexed vectors), or, with l2 and if
// that is later, where the norm of the leading components can reach t. One warp per query.
__global__ void k_q_split(const int64_t *__restrict__ qptr, const int2 *__restrict__ crow,
                          const float *__restrict__ mwr, const float *__restrict__ mw, int64_t nq, float t, bool l2,
                          int4 *vmeta) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const float t2 = __fmul_rd(t, t);
    for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < nq; x += nwarps) {
        const int64_t a = qptr[x], b = qptr[x + 1];
        const int32_t L = (int32_t)(b - a);
        const auto term = [&](int32_t p) {
            const int2 e = crow[a + p];
            return make_float2(__int_as_float(e.y), mwr[e.x]);
        };
        int32_t qs = L, ls = l2 ? L : 0;
        float bmw = 0.f, ssu = 0.f;
        for (int64_t base = a; base < b && (qs == L || ls == L); base += 32) {
            const int64_t p = base + lane;
            int2 e = make_int2(0, 0);
            float mwc = 0.f;
            if (p < b) {
                e = crow[p];
                mwc = mwr[e.x];
            }
            const float c = __int_as_float(e.y);
            if (qs == L) qs = split_step(__fmul_rn(c, mwc), p < b, (int32_t)(base - a), bmw, term, L, t, lane);
            const float si = __fadd_ru(ssu, warp_incl_scan_ru(__fmul_ru(c, c), lane));
            const unsigned hl = __ballot_sync(0xffffffffu, p < b && __fmul_ru(si, 1.0025f) >= t2);
            if (ls == L && hl) ls = (int32_t)(base - a) + __ffs(hl) - 1;
            ssu = __shfl_sync(0xffffffffu, si, 31);
        }
        if (lane == 0) vmeta[x] = make_int4((int32_t)a, L, max(min(qs, L), ls), __float_as_int(mw[x]));
    }
}

}  // namespace

aps_status prepare_queries(const aps_index *ix, const int64_t *qptr, const int32_t *qidx, const float *qval,
                           int32_t nq, float t, uint32_t flags, cudaStream_t s, QueryArrays &qa, int64_t nnz_known) {
    const IndexArrays &d = ix->d;
    int64_t nnz = nnz_known, first = 0;
    if (nnz_known < 0) {  // the row pointers live on the device only: read their ends back
        APS_CUDA(cudaMemcpyAsync(&nnz, qptr + nq, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        APS_CUDA(cudaMemcpyAsync(&first, qptr, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        APS_CUDA(cudaStreamSynchronize(s));
    }
    if (first != 0 || nnz < 0 || nnz >= (1ll << 31)) {
        set_error("query indptr[0] must be 0 and nnz in [0, 2^31)");
        return APS_EINVAL;
    }
    qa.nq = nq;
    qa.nnz = nnz;
    DBuf<int32_t> erow, len;
    DBuf<float> vout;
    DBuf<unsigned long long> err;
    APS_TRY(erow.alloc((size_t)std::max<int64_t>(nnz, 1), s));
    APS_TRY(vout.alloc((size_t)std::max<int64_t>(nnz, 1), s));
    APS_TRY(len.alloc((size_t)std::max<int64_t>(nq, 1), s));
    APS_TRY(qa.mw.alloc((size_t)std::max<int64_t>(nq, 1), s));
    APS_TRY(err.alloc(1, s));
    APS_CUDA(cudaMemsetAsync(err.p, 0xff, sizeof(unsigned long long), s));
    if (nq > 0) {
        // (the index's single instance gives the dimension space)
        k_validate<<<rows_grid(nq), T256, 0, s>>>(qptr, qidx, qval, nullptr, nullptr, ix->inst_h[0].m, nq, nnz, flags,
                                                  erow.p, vout.p, len.p, qa.mw.p, err.p, nullptr);
        APS_LAUNCH_CHECK();
    }
    unsigned long long e_h = ~0ull;
    APS_CUDA(cudaMemcpyAsync(&e_h, err.p, sizeof(e_h), cudaMemcpyDeviceToHost, s));
    APS_CUDA(cudaStreamSynchronize(s));
    if (e_h != ~0ull) {
        set_error("invalid query row %lld: %s", (long long)(e_h >> 8), code_name((int)(e_h & 0xff)));
        return APS_EINVAL;
    }
    APS_TRY(qa.crow.alloc((size_t)std::max<int64_t>(nnz, 1), s));
    if (nnz > 0) {
        const int rb = std::max(1, bits_for((uint64_t)(ix->maxm - 1)));
        const int bits = rb + bits_for((uint64_t)std::max(nq - 1, 0));
        if (bits <= 32)
            APS_TRY(sort_queries<uint32_t>(qidx, erow.p, d.rank_of_dim.p, vout.p, nnz, rb, bits, qa.crow.p, s));
        else
            APS_TRY(sort_queries<uint64_t>(qidx, erow.p, d.rank_of_dim.p, vout.p, nnz, rb, bits, qa.crow.p, s));
    }
    APS_TRY(qa.vmeta.alloc((size_t)std::max<int64_t>(nq, 1), s));
    if (nq > 0) {
        const bool l2 = !(flags & (APS_NO_MINSIZE | APS_NO_REMSCORE | APS_NO_UPPERBOUND));
        k_q_split<<<rows_grid(nq), T256, 0, s>>>(qptr, qa.crow.p, d.mwr.p, qa.mw.p, nq, t, l2,
                                                                    qa.vmeta.p);
        APS_LAUNCH_CHECK();
    }
    return APS_OK;
}

}  // namespace aps
