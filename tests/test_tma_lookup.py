"""The driver's tensor-map encoder is looked up once: threads that ask while the first of them
is still looking wait for what it finds (without it, creating a surrogate network fails)."""
import pytest

import host_build

SRC = r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#include <cuda.h>
#include <cuda_runtime.h>
static int calls = 0;
// the driver's lookup, slow and always successful
static cudaError_t slow_lookup(const char*, void** p, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* q)
{
    ++calls;
    std::this_thread::sleep_for(std::chrono::milliseconds(300));
    *p = (void*)&calls;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
#define cudaGetDriverEntryPointByVersion slow_lookup
#include "salec_tma.cuh"
int main()
{
    std::vector<void*> got(8, nullptr);
    std::vector<std::thread> t;
    for (size_t k = 0; k < got.size(); ++k) t.emplace_back([&got, k] { got[k] = (void*)salec::tma_encode_tiled(); });
    for (auto& x : t) x.join();
    for (void* p : got) std::printf("%d ", p == (void*)&calls);
    std::printf("%d\n", calls);
}
"""


@pytest.mark.skipif(host_build.nvcc_missing(), reason="no nvcc")
def test_threads_wait_for_the_first_lookup(tmp_path):
    assert host_build.run(SRC, tmp_path).split() == ["1"] * 8 + ["1"]
