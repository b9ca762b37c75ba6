"""The descriptor arena on the host, against a CUDA runtime of plain memory: every table pushed inside a gather
scope is on the device after that scope's upload, whatever scopes and blocks it crosses."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2509_03024_gb300", "csrc")

RUNTIME = r"""
#include <cstdlib>
#include <cstring>
#include <cstdio>
#include "core.cuh"
static int copies = 0;
extern "C" {
cudaError_t cudaMallocHost(void** p, size_t n) { *p = std::calloc(n, 1); return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = std::calloc(n, 1); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memcpy(d, s, n);
    copies++;
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
}
namespace fhe {
void fail(int code, const std::string& msg) { throw FheException(code, msg); }
void cuda_check(cudaError_t, const char*) {}
}
using namespace fhe;
static std::vector<u64> table(u64 tag, size_t words) {
    std::vector<u64> t(words);
    for (size_t i = 0; i < words; i++) t[i] = tag * 1000003 + i;
    return t;
}
#define NEED(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
static bool there(const u64* d, const std::vector<u64>& t) { return std::memcmp(d, t.data(), t.size() * 8) == 0; }
"""

CASES = {
    "one_scope": """
    ArenaGather g(a);
    u64 *x = a.push_vec(A, 0), *y = a.push_vec(B, 0);
    NEED(copies == 0);
    g.upload(0);
    NEED(copies == 1 && there(x, A) && there(y, B));
    u64* z = a.push_vec(C, 0);            // after the upload the scope is over
    NEED(there(z, C));""",
    "nested": """
    ArenaGather g(a);
    u64 *x = a.push_vec(A, 0), *y, *z;
    {
        ArenaGather h(a);
        y = a.push_vec(B, 0);
        h.upload(0);
        NEED(there(y, B));
    }
    z = a.push_vec(C, 0);
    NEED(!there(z, C));                   // the outer scope still gathers
    g.upload(0);
    NEED(there(x, A) && there(y, B) && there(z, C));""",
    "nested_abandoned": """
    ArenaGather g(a);
    u64 *x = a.push_vec(A, 0), *z;
    try {
        ArenaGather h(a);
        a.push_vec(B, 0);
        fail(-1, "");
    } catch (const FheException&) {
    }
    z = a.push_vec(C, 0);
    g.upload(0);
    NEED(there(x, A) && there(z, C));""",
    "abandoned": """
    try {
        ArenaGather g(a);
        a.push_vec(A, 0);
        fail(-1, "");
    } catch (const FheException&) {
    }
    u64* z = a.push_vec(C, 0);
    NEED(there(z, C));
    ArenaGather h(a);
    u64* y = a.push_vec(B, 0);
    h.upload(0);
    NEED(there(y, B));""",
    "nested_over_blocks": """
    const std::vector<u64> big = table(9, (3u << 20) / 8);    // two of them need two blocks of 4 MiB
    for (int round = 0; round < 4; round++) {                 // rounds 2 and 3 reuse the blocks of 0 and 1
        a.reset(0);
        ArenaGather g(a);
        u64 *x = a.push_vec(A, 0), *b1 = a.push_vec(big, 0), *b2, *y;
        {
            ArenaGather h(a);
            b2 = a.push_vec(big, 0);
            y = a.push_vec(B, 0);
            h.upload(0);
            NEED(there(b2, big) && there(y, B));
        }
        u64 *b3 = a.push_vec(big, 0), *z = a.push_vec(C, 0);
        g.upload(0);
        NEED(there(x, A) && there(b1, big) && there(b3, big) && there(z, C));
        for (auto& hf : a.halves)
            for (auto& b : hf.blocks) std::memset(b.dev, 0, b.cap);
    }""",
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_gathered_tables_reach_the_device(name, tmp_path):
    src = tmp_path / "main.cpp"
    src.write_text(RUNTIME + "int main() {\n    Arena a;\n    const std::vector<u64> A = table(1, 100), B = table(2, 33), "
                             "C = table(3, 1);" + CASES[name] + "\n    return 0;\n}\n")
    exe = str(tmp_path / "arena")
    subprocess.run(["g++", "-std=c++17", "-I/usr/local/cuda/include", f"-I{CSRC}", str(src), "-x", "c++",
                    os.path.join(CSRC, "arena.cu"), "-o", exe], check=True)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stdout
