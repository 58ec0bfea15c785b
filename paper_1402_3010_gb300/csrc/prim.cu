// Error state, device memory and the generic device primitives (prefix sum, stable
// radix sort) used by the index build and the output stage.
#include <atomic>
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "aps_internal.cuh"

namespace aps {

// ------------------------------------------------------------------ error state
static thread_local char g_err[512] = "";

void set_error(const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
}

aps_status cuda_status(cudaError_t e, const char *what, const char *file, int line) {
    set_error("%s failed: %s (%s:%d)", what, cudaGetErrorString(e), file, line);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();  // clear the sticky-free allocation error
        return APS_ENOMEM;
    }
    return APS_ECUDA;
}

static std::atomic<int64_t> g_launches{0};
void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

// ------------------------------------------------------------------ memory
static std::mutex g_pool_mu;
static bool g_pool_ready[64];
// test hook: the k-th device allocation from now fails (atomic: serving slots allocate
// from their own threads)
static std::atomic<int64_t> g_alloc_fault{0};

void set_alloc_fault(int64_t k) { g_alloc_fault.store(k); }

static void pool_setup() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (g_pool_ready[dev]) return;
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
        uint64_t thr = UINT64_MAX;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
    }
    g_pool_ready[dev] = true;
}

aps_status dalloc(void **p, size_t bytes, cudaStream_t s) {
    *p = nullptr;
    if (g_alloc_fault.load() > 0 && g_alloc_fault.fetch_sub(1) == 1) {
        set_error("device allocation of %zu bytes failed (injected)", bytes);
        return APS_ENOMEM;
    }
    pool_setup();
    cudaError_t e = cudaMallocAsync(p, bytes ? bytes : 1, s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        set_error("device allocation of %zu bytes failed: %s", bytes, cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? APS_ENOMEM : APS_ECUDA;
    }
    return APS_OK;
}

void dfree(void *p, cudaStream_t s) {
    if (p) cudaFreeAsync(p, s);
}

// ------------------------------------------------------------------ pinned host blocks
static std::mutex g_host_mu;
static std::vector<void *> g_host_free[64];  // cached blocks by size class (2^c bytes)
static size_t g_host_cached = 0;
constexpr size_t HOST_CACHE_MAX = (size_t)8 << 30;

static int host_class(size_t bytes) {
    int c = 20;  // 1 MiB
    while (c < 63 && ((size_t)1 << c) < bytes) c++;
    return c;
}

aps_status halloc(void **p, size_t bytes) {
    *p = nullptr;
    const int c = host_class(bytes);
    {
        std::lock_guard<std::mutex> lk(g_host_mu);
        if (!g_host_free[c].empty()) {
            *p = g_host_free[c].back();
            g_host_free[c].pop_back();
            g_host_cached -= (size_t)1 << c;
            return APS_OK;
        }
    }
    cudaError_t e = cudaMallocHost(p, (size_t)1 << c);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return cuda_status(e, "cudaMallocHost", __FILE__, __LINE__);
    }
    return APS_OK;
}

void hfree(void *p, size_t bytes) {
    if (!p) return;
    const int c = host_class(bytes);
    {
        std::lock_guard<std::mutex> lk(g_host_mu);
        if (g_host_cached + ((size_t)1 << c) <= HOST_CACHE_MAX) {
            g_host_free[c].push_back(p);
            g_host_cached += (size_t)1 << c;
            return;
        }
    }
    cudaFreeHost(p);
}

// ------------------------------------------------------------------ prefix sum
namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

template <class T>
__global__ void scan_reduce_kernel(const T *__restrict__ in, int64_t n, int64_t *__restrict__ sums) {
    __shared__ int64_t warp_tot[SCAN_THREADS / 32];
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    int64_t acc = 0;
    for (int k = 0; k < SCAN_ITEMS; k++) {
        int64_t i = base + (int64_t)k * SCAN_THREADS + threadIdx.x;
        if (i < n) acc += (int64_t)in[i];
    }
    for (int o = 16; o; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) warp_tot[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t t = 0;
        for (int w = 0; w < SCAN_THREADS / 32; w++) t += warp_tot[w];
        sums[blockIdx.x] = t;
    }
}

// Each block scans its tile (thread t owns items [t*ITEMS, (t+1)*ITEMS) of the tile) and
// adds the scanned block offset.
template <class T>
__global__ void scan_down_kernel(const T *__restrict__ in, int64_t n, const int64_t *__restrict__ offs,
                                 int64_t *__restrict__ out) {
    __shared__ int64_t warp_tot[SCAN_THREADS / 32];
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    int64_t v[SCAN_ITEMS];
    int64_t local = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; k++) {
        int64_t i = base + k;
        v[k] = i < n ? (int64_t)in[i] : 0;
        local += v[k];
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t inc = local;
    for (int o = 1; o < 32; o <<= 1) {
        int64_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    int64_t wbase = 0;
    for (int w = 0; w < warp; w++) wbase += warp_tot[w];
    int64_t run = (offs ? offs[blockIdx.x] : 0) + wbase + inc - local;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; k++) {
        int64_t i = base + k;
        if (i < n) out[i] = run;
        run += v[k];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == SCAN_THREADS - 1) out[n] = run;
}

template <class T>
aps_status scan_impl(const T *in, int64_t *out, int64_t n, cudaStream_t s) {
    if (n <= 0) {
        APS_CUDA(cudaMemsetAsync(out, 0, sizeof(int64_t), s));
        return APS_OK;
    }
    int64_t nb = (n + SCAN_TILE - 1) / SCAN_TILE;
    DBuf<int64_t> offs;
    if (nb > 1) {
        DBuf<int64_t> sums;
        APS_TRY(sums.alloc((size_t)nb, s));
        scan_reduce_kernel<T><<<(unsigned)nb, SCAN_THREADS, 0, s>>>(in, n, sums.p);
        APS_LAUNCH_CHECK();
        APS_TRY(offs.alloc((size_t)nb + 1, s));
        APS_TRY(scan_impl<int64_t>(sums.p, offs.p, nb, s));
    }
    scan_down_kernel<T><<<(unsigned)nb, SCAN_THREADS, 0, s>>>(in, n, offs.p, out);
    APS_LAUNCH_CHECK();
    return APS_OK;
}

}  // namespace

aps_status scan_exclusive(const int32_t *in, int64_t *out, int64_t n, cudaStream_t s) {
    return scan_impl<int32_t>(in, out, n, s);
}
aps_status scan_exclusive(const int64_t *in, int64_t *out, int64_t n, cudaStream_t s) {
    return scan_impl<int64_t>(in, out, n, s);
}

// ------------------------------------------------------------------ radix sort
// Stable LSD radix sort, 8 bits a pass, by the single-pass method with decoupled look-back (Merrill and
// Garland's scan, 2016; Adinets and Merrill's sort, 2022). One kernel counts the digits of every pass; a pass is
// then one kernel that reads each item once and writes it once: a tile ranks its items by warp,
// publishes its digit counts, adds up the earlier tiles' by looking back over what they have
// published, and writes its items out in digit runs. 40M keys with a payload take 0.37 ms a pass
// and 0.12 for the counts, some 40% of the copy bandwidth (it was 0.50 with a histogram, a scan of
// three launches and a scatter for each pass). What bounds it is a tile's chain of steps: its reads,
// its ranks, the look-back (hundreds of tiles run side by side) and its writes. So the tiles are
// large (4096 items at three CTAs an SM beat 3072 at four, 0.42 ms, and 2048 at five, 0.43), and the
// payload is read after the look-back, which has its registers until then. Nine bits a pass, which
// saves 18-bit keys a pass, made each pass half again as long.
// Up to SMALL_MAX items one CTA sorts in shared memory, all passes in one launch.
namespace {

constexpr int RS_THREADS = 256;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_DIGITS = 256;
constexpr int RS_MAXPASS = 8;

template <class K>
__device__ __forceinline__ int digit_of(const K k, const int shift) {
    return (int)((k >> shift) & (K)0xff);
}

// Digit counts of all passes (gcount[pass][digit]); the last block to finish turns each pass's
// counts into the digits' first output positions.
template <class K>
__global__ void __launch_bounds__(RS_THREADS) rs_count_kernel(const K *__restrict__ keys, int64_t n, int passes,
                                                              unsigned long long *gcount, uint32_t *done) {
    __shared__ uint32_t h[RS_MAXPASS][RS_DIGITS];
    __shared__ unsigned long long wsum[RS_WARPS];
    __shared__ bool last;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int p = 0; p < passes; p++) h[p][t] = 0u;
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * RS_THREADS;
    for (int64_t i0 = (int64_t)blockIdx.x * RS_THREADS; i0 < n; i0 += stride) {
        const int64_t i = i0 + t;
        const bool valid = i < n;
        const K k = valid ? keys[i] : (K)0;
        for (int p = 0; p < passes; p++) {
            const int d = digit_of(k, 8 * p);
            const int d0 = __shfl_sync(0xffffffffu, d, 0);
            // (one digit for the whole warp is common in the high passes and among equal keys)
            const bool same = valid && d == d0;
            if (__all_sync(0xffffffffu, same)) {
                if (lane == 0) atomicAdd(&h[p][d], 32u);
            } else if (valid) {
                atomicAdd(&h[p][d], 1u);
            }
        }
    }
    __syncthreads();
    for (int p = 0; p < passes; p++)
        if (h[p][t]) atomicAdd(&gcount[p * RS_DIGITS + t], (unsigned long long)h[p][t]);
    __threadfence();
    __syncthreads();
    if (t == 0) last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int p = 0; p < passes; p++) {
        const unsigned long long c = *(volatile unsigned long long *)&gcount[p * RS_DIGITS + t];
        unsigned long long inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        for (int w = 0; w < warp; w++) inc += wsum[w];
        gcount[p * RS_DIGITS + t] = inc - c;
        __syncthreads();
    }
}

// Ranks of a warp's items among the items of the same digit of this warp so far (whist: the
// warp's digit counts). Warp-collective; invalid items take no part.
__device__ __forceinline__ uint32_t warp_rank(uint32_t *whist, const int d, const bool valid, const unsigned lt_mask) {
    // lanes with the same digit, one ballot per bit (the match instruction is slower than eight votes)
    unsigned peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
    for (int b = 0; b < 8; b++) {
        const bool bit = (d >> b) & 1;
        const unsigned m = __ballot_sync(0xffffffffu, bit);
        peers &= bit ? m : ~m;
    }
    const uint32_t before = (uint32_t)__popc(peers & lt_mask);
    uint32_t base = 0u;
    if (valid) base = whist[d];
    __syncwarp();
    if (valid && before == 0u) whist[d] = base + (uint32_t)__popc(peers);
    __syncwarp();
    return base + before;
}

constexpr unsigned long long RS_COUNT = 1ull << 62, RS_TOTAL = 2ull << 62, RS_VALUE = (1ull << 62) - 1ull;
constexpr int RS_SPINS = 1 << 14;  // polls without an answer before a tile is counted here

template <class K, bool VALS, int ITEMS>
constexpr int rs_smem() { return RS_THREADS * ITEMS * (int)(sizeof(K) + (VALS ? 4 : 0)); }

// One pass. Tiles are taken by ticket, so the earlier tiles that a tile looks back on have all
// been started. A tile that stays silent for RS_SPINS polls is counted from its keys instead, so
// the wait always ends.
template <class K, bool VALS, int ITEMS>
__global__ void __launch_bounds__(RS_THREADS, 3) rs_pass_kernel(const K *__restrict__ kin,
                                                             const uint32_t *__restrict__ vin, K *__restrict__ kout,
                                                             uint32_t *__restrict__ vout, int64_t n, int shift,
                                                             const unsigned long long *__restrict__ gbase,
                                                             unsigned long long *status, uint32_t *ticket) {
    constexpr int TILE = RS_THREADS * ITEMS;
    extern __shared__ __align__(16) unsigned char rs_mem[];
    K *sk = reinterpret_cast<K *>(rs_mem);
    uint32_t *sv = reinterpret_cast<uint32_t *>(sk + TILE);
    __shared__ uint32_t whist[RS_WARPS][RS_DIGITS];
    __shared__ int64_t gpos[RS_DIGITS];  // output position of the digit's items minus their place in the tile
    __shared__ uint32_t wsum[RS_WARPS];
    __shared__ uint32_t tile_s;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    if (t == 0) tile_s = atomicAdd(ticket, 1u);
    for (int w = 0; w < RS_WARPS; w++) whist[w][t] = 0u;
    __syncthreads();
    const int64_t tile = tile_s;
    const int tn = (int)min((int64_t)TILE, n - tile * TILE);  // items of the tile
    const int first = warp * (32 * ITEMS) + lane;             // this lane's first one
    const K *const kp = kin + tile * TILE + first;
    K k[ITEMS];
    uint32_t v[ITEMS], rank[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; i++) k[i] = first + 32 * i < tn ? kp[32 * i] : (K)0;
#pragma unroll
    for (int i = 0; i < ITEMS; i++)
        rank[i] = warp_rank(whist[warp], digit_of(k[i], shift), first + 32 * i < tn, lt_mask);
    __syncthreads();
    // thread t: digit t. The warps' counts become their offsets, the tile's count is published
    uint32_t c = 0;
#pragma unroll
    for (int w = 0; w < RS_WARPS; w++) {
        const uint32_t x = whist[w][t];
        whist[w][t] = c;
        c += x;
    }
    volatile unsigned long long *st = status;
    st[tile * RS_DIGITS + t] = (tile == 0 ? RS_TOTAL : RS_COUNT) | (unsigned long long)c;
    uint32_t inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    for (int w = 0; w < warp; w++) inc += wsum[w];
    const uint32_t lbase = inc - c;  // place of the digit's first item in the tile
    unsigned long long before = 0ull;  // the digit's items in earlier tiles
    // eight earlier tiles at a time: a step back costs a load's latency, and hundreds of tiles run
    // side by side without a total to stop at
    int spins = 0;
    for (int64_t q = tile - 1; q >= 0;) {
        unsigned long long x[8];
#pragma unroll
        for (int j = 0; j < 8; j++) {
            x[j] = RS_TOTAL + 0ull;
            if (q >= j) x[j] = st[(q - j) * RS_DIGITS + t];
        }
        int used = 0;
        bool total = false;
#pragma unroll
        for (int j = 0; j < 8; j++) {
            if (used == j && !total && (x[j] >> 62) != 0ull) {
                before += x[j] & RS_VALUE;
                total = (x[j] >> 62) == 2ull;
                used++;
            }
        }
        if (total) break;
        q -= used;
        if (used == 0) {
            if (++spins <= RS_SPINS) {
                __nanosleep(20);
            } else {
                for (int64_t e = q * TILE; e < (q + 1) * TILE; e++) before += digit_of(kin[e], shift) == t ? 1ull : 0ull;
                q--;
                spins = 0;
            }
        }
    }
    if (tile > 0) st[tile * RS_DIGITS + t] = RS_TOTAL | (before + (unsigned long long)c);
    gpos[t] = (int64_t)(gbase[t] + before) - (int64_t)lbase;
#pragma unroll
    for (int w = 0; w < RS_WARPS; w++) whist[w][t] += lbase;
    if (VALS) {  // (not earlier: the look-back keeps its registers)
        const uint32_t *const vp = vin + tile * TILE + first;
#pragma unroll
        for (int i = 0; i < ITEMS; i++) v[i] = first + 32 * i < tn ? vp[32 * i] : 0u;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
        if (first + 32 * i < tn) {
            const uint32_t q = whist[warp][digit_of(k[i], shift)] + rank[i];
            sk[q] = k[i];
            if (VALS) sv[q] = v[i];
        }
    }
    __syncthreads();
    for (int q = t; q < tn; q += RS_THREADS) {
        const K x = sk[q];
        const int64_t dst = gpos[digit_of(x, shift)] + q;
        kout[dst] = x;
        if (VALS) vout[dst] = sv[q];
    }
}

// Up to SMALL_MAX items: one CTA, every pass in shared memory.
constexpr int SMALL_THREADS = 1024;
constexpr int SMALL_WARPS = SMALL_THREADS / 32;
constexpr int SMALL_ITEMS = 8;
constexpr int SMALL_MAX = SMALL_THREADS * SMALL_ITEMS;

template <class K>
__global__ void __launch_bounds__(SMALL_THREADS) rs_small_kernel(K *keys, uint32_t *vals, int n, int passes) {
    extern __shared__ __align__(16) unsigned char rs_mem[];
    K *sk = reinterpret_cast<K *>(rs_mem);
    uint32_t *sv = reinterpret_cast<uint32_t *>(sk + SMALL_MAX);
    uint32_t(*whist)[RS_DIGITS] = reinterpret_cast<uint32_t(*)[RS_DIGITS]>(sv + SMALL_MAX);
    __shared__ uint32_t wsum[8];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    // rounds of 32 items a warp takes, and the warps that have any
    const int per = (n + SMALL_THREADS - 1) / SMALL_THREADS, used = (n + 32 * per - 1) / (32 * per);
    const int first = warp * (32 * per) + lane;
    K k[SMALL_ITEMS];
    uint32_t v[SMALL_ITEMS], rank[SMALL_ITEMS];
#pragma unroll
    for (int i = 0; i < SMALL_ITEMS; i++) {
        const int q = first + 32 * i;
        k[i] = i < per && q < n ? keys[q] : (K)0;
        v[i] = vals && i < per && q < n ? vals[q] : 0u;
    }
    for (int p = 0; p < passes; p++) {
        for (int i = t; i < used * RS_DIGITS; i += SMALL_THREADS) (&whist[0][0])[i] = 0u;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < SMALL_ITEMS; i++) {
            rank[i] = 0u;
            if (i < per && warp < used)  // (the same for the whole warp)
                rank[i] = warp_rank(whist[warp], digit_of(k[i], 8 * p), first + 32 * i < n, lt_mask);
        }
        __syncthreads();
        uint32_t c = 0, inc = 0;
        if (t < RS_DIGITS) {  // thread t: digit t
            for (int w = 0; w < used; w++) {
                const uint32_t x = whist[w][t];
                whist[w][t] = c;
                c += x;
            }
            inc = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            if (lane == 31) wsum[warp] = inc;
        }
        __syncthreads();
        if (t < RS_DIGITS) {
            for (int w = 0; w < warp; w++) inc += wsum[w];
            for (int w = 0; w < used; w++) whist[w][t] += inc - c;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < SMALL_ITEMS; i++) {
            if (i < per && first + 32 * i < n) {
                const uint32_t q = whist[warp][digit_of(k[i], 8 * p)] + rank[i];
                sk[q] = k[i];
                sv[q] = v[i];
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < SMALL_ITEMS; i++) {
            const int q = first + 32 * i;
            if (i < per && q < n) {
                k[i] = sk[q];
                v[i] = sv[q];
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < SMALL_ITEMS; i++) {
        const int q = first + 32 * i;
        if (i < per && q < n) {
            keys[q] = k[i];
            if (vals) vals[q] = v[i];
        }
    }
}

template <class K, bool VALS, int ITEMS>
aps_status sort_tiles(DBuf<K> &keys, DBuf<uint32_t> *vals, int64_t n, int passes, cudaStream_t s) {
    constexpr int TILE = RS_THREADS * ITEMS;
    constexpr int smem = rs_smem<K, VALS, ITEMS>();
    const int64_t nb = (n + TILE - 1) / TILE;
    DBuf<K> k2;
    DBuf<uint32_t> v2;
    // counts of every pass, then every pass's tile states, then the tickets and the done counter
    DBuf<unsigned long long> work;
    const size_t words = (size_t)passes * RS_DIGITS * (size_t)(nb + 1) + RS_MAXPASS;
    APS_TRY(k2.alloc((size_t)n, s));
    if (VALS) APS_TRY(v2.alloc((size_t)n, s));
    APS_TRY(work.alloc(words, s));
    APS_CUDA(cudaMemsetAsync(work.p, 0, words * sizeof(unsigned long long), s));
    unsigned long long *gcount = work.p, *status = work.p + (size_t)passes * RS_DIGITS;
    uint32_t *tickets = reinterpret_cast<uint32_t *>(work.p + words - RS_MAXPASS);
    APS_CUDA(cudaFuncSetAttribute(rs_pass_kernel<K, VALS, ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    rs_count_kernel<K><<<grid_for(n, RS_THREADS * (ITEMS == 4 ? 2 : 8), (int64_t)num_sms() * 8), RS_THREADS, 0, s>>>(
        keys.p, n, passes, gcount, tickets + RS_MAXPASS);
    APS_LAUNCH_CHECK();
    for (int p = 0; p < passes; p++) {
        rs_pass_kernel<K, VALS, ITEMS><<<(unsigned)nb, RS_THREADS, smem, s>>>(
            keys.p, VALS ? vals->p : nullptr, k2.p, VALS ? v2.p : nullptr, n, 8 * p, gcount + p * RS_DIGITS,
            status + (size_t)p * RS_DIGITS * nb, tickets + p);
        APS_LAUNCH_CHECK();
        std::swap(keys.p, k2.p);  // (the sorted items are the caller's, whatever the number of passes)
        std::swap(keys.n, k2.n);
        std::swap(keys.own, k2.own);
        if (VALS) {
            std::swap(vals->p, v2.p);
            std::swap(vals->n, v2.n);
            std::swap(vals->own, v2.own);
        }
    }
    return APS_OK;
}

template <class K, bool VALS>
aps_status sort_impl(DBuf<K> &keys, DBuf<uint32_t> *vals, int64_t n, int bits, cudaStream_t s) {
    if (n <= 1 || bits <= 0) return APS_OK;
    const int passes = (bits + 7) / 8;
    if (n <= SMALL_MAX) {
        constexpr int smem = SMALL_MAX * (int)(sizeof(K) + 4) + SMALL_WARPS * RS_DIGITS * 4;
        APS_CUDA(cudaFuncSetAttribute(rs_small_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        rs_small_kernel<K><<<1, SMALL_THREADS, smem, s>>>(keys.p, VALS ? vals->p : nullptr, (int)n, passes);
        APS_LAUNCH_CHECK();
        return APS_OK;
    }
    // Tiles of four items a thread while they leave an SM no more than one: a pass is then one
    // tile's chain of steps, and a shorter tile's is shorter (31,000 64-bit keys: counts and three
    // passes 24 us, 31 with the larger tiles).
    if (n <= (int64_t)num_sms() * RS_THREADS * 4) return sort_tiles<K, VALS, 4>(keys, vals, n, passes, s);
    return sort_tiles<K, VALS, sizeof(K) == 8 ? 16 : 20>(keys, vals, n, passes, s);
}

}  // namespace

aps_status sort_pairs(DBuf<uint64_t> &keys, DBuf<uint32_t> &vals, int64_t n, int bits, cudaStream_t s) {
    return sort_impl<uint64_t, true>(keys, &vals, n, bits, s);
}
aps_status sort_pairs(DBuf<uint32_t> &keys, DBuf<uint32_t> &vals, int64_t n, int bits, cudaStream_t s) {
    return sort_impl<uint32_t, true>(keys, &vals, n, bits, s);
}
aps_status sort_keys(DBuf<uint64_t> &keys, int64_t n, int bits, cudaStream_t s) {
    return sort_impl<uint64_t, false>(keys, nullptr, n, bits, s);
}

}  // namespace aps

extern "C" const char *aps_last_error(void) { return aps::g_err; }
extern "C" int64_t aps_launch_count(void) { return aps::g_launches.load(); }
