"""The host side of queries and of the request loop, on the CPU: serve.cu (which launches nothing
itself) compiled by the host compiler against a stand-in for the CUDA runtime whose copies read
their source only when their stream is waited for, as CUDA's documentation allows, and for the
kernels' entry points. Freed host memory is overwritten and never handed out again."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1402_3010_gb300", "csrc")
CUDA = next((d for d in ("/usr/local/cuda/include",) if os.path.exists(os.path.join(d, "cuda_runtime.h"))), None)

pytestmark = pytest.mark.skipif(CUDA is None or shutil.which("g++") is None, reason="needs g++ and the CUDA headers")

HARNESS = r"""
#include <algorithm>
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <malloc.h>
#include <map>
#include <mutex>
#include <new>
#include <thread>
#include <vector>
static inline int __clz(int x) { return x ? __builtin_clz((unsigned)x) : 32; }
using std::max;
using std::min;
#include "serve.cu"

void *operator new(size_t n) {
    void *p = malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void *p) noexcept { if (p) memset(p, 0xDD, malloc_usable_size(p)); }
void operator delete(void *p, size_t) noexcept { operator delete(p); }

// ---- the runtime: a copy is done when its stream is waited for
struct Copy { void *d; const void *s; size_t n; };
static std::mutex mu;
static std::map<cudaStream_t, std::vector<Copy>> inflight;
static void drain(cudaStream_t s) {
    std::vector<Copy> v;
    { std::lock_guard<std::mutex> lk(mu); v.swap(inflight[s]); }
    for (const Copy &c : v) memcpy(c.d, c.s, c.n);
}
static size_t pending(cudaStream_t s) { std::lock_guard<std::mutex> lk(mu); return inflight[s].size(); }
extern "C" {
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    std::lock_guard<std::mutex> lk(mu);
    inflight[st].push_back({d, s, n});
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { drain(s); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)malloc(16); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)malloc(16); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
const char *aps_last_error(void) { return ""; }
}

// ---- the rest of the library
static aps_status prepare_status = APS_OK;  // APS_ENOMEM: out of memory before the first wait
static std::vector<int64_t> want_ptr;
static std::vector<int32_t> want_idx;
static std::vector<float> want_val;
static int seen = 0, running = 0, most = 0, hold_for = 0;
static std::mutex jm;
static std::condition_variable jcv;
namespace aps {
void set_error(const char *, ...) {}
aps_status cuda_status(cudaError_t, const char *, const char *, int) { return APS_ECUDA; }
aps_status dalloc(void **p, size_t n, cudaStream_t) { *p = malloc(n); return *p ? APS_OK : APS_ENOMEM; }
void dfree(void *p, cudaStream_t) { free(p); }
void pairs_release(aps_pairs *) {}
aps_status pairs_to_host(aps_pairs *, cudaStream_t) { return APS_OK; }
aps_status prepare_queries(const aps_index *, const int64_t *p, const int32_t *i, const float *v, int32_t nq, float,
                           uint32_t, cudaStream_t s, QueryArrays &qa, int64_t nnz) {
    if (prepare_status != APS_OK) return prepare_status;
    drain(s);
    if (!want_ptr.empty()) {
        const bool same = nnz == (int64_t)want_idx.size() && !memcmp(p, want_ptr.data(), 8 * want_ptr.size()) &&
                          !memcmp(i, want_idx.data(), 4 * want_idx.size()) &&
                          !memcmp(v, want_val.data(), 4 * want_val.size());
        seen += same ? 1 : 1000;
    }
    qa.nq = nq;
    qa.nnz = nnz;
    return APS_OK;
}
aps_status join_queries(const aps_index *, const QueryArrays &, float, uint32_t, cudaStream_t, aps_pairs *, aps_stats *) {
    std::unique_lock<std::mutex> lk(jm);
    most = std::max(most, ++running);
    jcv.notify_all();
    if (hold_for) jcv.wait_for(lk, std::chrono::seconds(2), [] { return most >= hold_for; });
    running--;
    return APS_OK;
}
}  // namespace aps

static aps_index ix;
static void index_of(int n) {
    ix.flags = APS_QUERYABLE;
    ix.k = 1;
    ix.t = 0.5f;
    ix.inst_h.resize(1);
    ix.inst_h[0] = InstDesc{};
    ix.inst_h[0].n = n;
    ix.inst_h[0].m = 100;
    ix.inst_h[0].G = 2;
    ix.inst_h[0].W = tile_window(2);
    ix.inst_h[0].nw = (n + tile_window(2) - 1) / tile_window(2);
}
static void rows(int nq, int per) {
    want_ptr.clear(); want_idx.clear(); want_val.clear();
    for (int q = 0; q <= nq; q++) want_ptr.push_back((int64_t)q * per);
    for (int e = 0; e < nq * per; e++) { want_idx.push_back(e % per); want_val.push_back(0.25f + e); }
}
"""

MAINS = {
    # queries packed into one buffer (up to 32 KB) and copied from the caller's arrays: what the
    # device reads is what the caller gave
    "rows_arrive": r"""
int main() {
    const cudaStream_t s = (cudaStream_t)&ix;
    ix.stream = s;
    index_of(10000);
    int calls = 0;
    for (int per : {1, 10, 300, 5000})
        for (int nq : {1, 3}) {
            rows(nq, per);
            aps_pairs out;
            if (aps_query(&ix, want_ptr.data(), want_idx.data(), want_val.data(), nq, 0.5f, 0, &out) != APS_OK) return 1;
            calls++;
            if (pending(s) != 0) return 2;
        }
    printf("%d rows seen right in %d calls\n", seen, calls);
    return seen == calls ? 0 : 3;
}""",
    # out of memory before the first wait: no copy of the caller's arrays outlives the call
    "failure_leaves_no_copy": r"""
int main() {
    const cudaStream_t s = (cudaStream_t)&ix;
    ix.stream = s;
    index_of(10000);
    prepare_status = APS_ENOMEM;
    for (int per : {10, 5000}) {
        rows(2, per);
        aps_pairs out;
        if (aps_query(&ix, want_ptr.data(), want_idx.data(), want_val.data(), 2, 0.5f, 0, &out) != APS_ENOMEM) return 1;
        printf("%zu copies in flight\n", pending(s));
        if (pending(s) != 0) return 2;
    }
    return 0;
}""",
    # a last row pointer that no array can have is refused before a size is computed from it
    "huge_counts_are_refused": r"""
int main() {
    index_of(10000);
    aps_server *sv = nullptr;
    if (aps_server_create(&ix, 1 << 30, 1, &sv) != APS_OK) return 1;
    const int32_t id = 0;
    const float val = 1.f;
    int rc = 0;
    for (int64_t nnz : {(int64_t)1 << 31, (int64_t)1 << 60, (int64_t)1 << 61, (int64_t)1 << 62, INT64_MAX, (int64_t)-1}) {
        const int64_t ptr[2] = {0, nnz};
        aps_pairs out;
        if (aps_query(&ix, ptr, &id, &val, 1, 0.5f, 0, &out) != APS_EINVAL) rc = 2;
        const aps_query_req req = {ptr, &id, &val, 1, 0.5f};
        uint64_t ticket = 0;
        if (aps_stream_submit(sv, &req, &ticket) != APS_EINVAL) rc = 3;
    }
    aps_server_free(sv);
    return rc;
}""",
    # batches whose footprint leaves room for another run side by side: one query against a million rows
    # holds some 20 MB (its staging most of all)
    "small_batches_share_a_budget": r"""
int main() {
    index_of(1000000);
    const int32_t id[1] = {3};
    const float val[1] = {1.f};
    const int64_t ptr[2] = {0, 1};
    hold_for = 2;
    for (size_t budget : {(size_t)48 << 20, (size_t)1}) {  // room for two; for none: one at a time
        most = 0;
        if (budget == 1) hold_for = 0;
        aps_server *sv = nullptr;
        if (aps_server_create(&ix, budget, 2, &sv) != APS_OK) return 1;
        uint64_t tk[2];
        const aps_query_req req = {ptr, id, val, 1, 0.5f};
        for (uint64_t &t : tk)
            if (aps_stream_submit(sv, &req, &t) != APS_OK) return 2;
        for (uint64_t t : tk) {
            aps_pairs out;
            if (aps_stream_poll(sv, t, 10000000, &out) != APS_OK) return 3;
        }
        aps_server_free(sv);
        printf("budget %zu: %d at once\n", budget, most);
        if (most != (budget == 1 ? 1 : 2)) return 4;
    }
    return 0;
}""",
}


def _run(tmp_path, name):
    src = tmp_path / f"{name}.cc"
    src.write_text(HARNESS + MAINS[name])
    exe = tmp_path / name
    r = subprocess.run(["g++", "-std=c++17", "-O0", "-w", "-I", CUDA, "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                        str(src), "-o", str(exe), "-lpthread"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[:4000]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)


@pytest.mark.parametrize("name", sorted(MAINS))
def test_serve_host(tmp_path, name):
    _run(tmp_path, name)
