// Results and the pool of page-locked blocks: rn_api.cpp over fakes of the calls that a result makes,
// the copying launch failing or not.  Built as a shared library
// (the engine's functions stay unresolved) and run by tests/test_host_result.py.
#include <cstdlib>

#include <cuda_runtime.h>

#include "rn_internal.h"

static int allocations = 0;
static bool fails = true;  // the copying launch

extern "C" cudaError_t cudaHostAlloc(void **p, size_t bytes, unsigned) {
    allocations++;
    *p = std::malloc(bytes);
    return cudaSuccess;
}
extern "C" cudaError_t cudaFreeHost(void *p) {
    std::free(p);
    return cudaSuccess;
}
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }
extern "C" cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
extern "C" cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }

namespace rn {
void fail(rn_status s, const std::string &msg) { throw Error{s, msg}; }
void triple_to_host(const uint32_t *, const uint32_t *, const uint32_t *, uint64_t, uint32_t *, void *) {
    if (fails) fail(RN_ECUDA, "launch failed");
}
void to_host_pairs(const rn_dpairs &d, rn_pairs *out, void *stream);
}  // namespace rn

// Results that were not given back or not reported, and the blocks allocated for three results.
extern "C" int failed_results(int *blocks) {
    int bad = 0;
    for (int run = 0; run < 3; run++) {
        uint32_t word = 0;
        rn_dpairs d{&word, &word, &word, 8192, 8192};
        rn_pairs out{};
        bool threw = false;
        try {
            rn::to_host_pairs(d, &out, nullptr);
        } catch (const rn::Error &e) {
            threw = e.status == RN_ECUDA;
        }
        bad += !threw || out.u || out.v || out.d || out.n;
    }
    *blocks = allocations;
    return bad;
}

// The blocks allocated for `runs` results of n pairs, each freed before the next.
extern "C" int blocks_for_results(uint64_t n, int runs) {
    fails = false;
    allocations = 0;
    for (int run = 0; run < runs; run++) {
        uint32_t word = 0;
        rn_dpairs d{&word, &word, &word, n, n};
        rn_pairs out{};
        rn::to_host_pairs(d, &out, nullptr);
        rn_pairs_free(&out);
    }
    return allocations;
}
