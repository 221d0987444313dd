"""The layer-level calls' scratch pool (csrc/scratch.h) over a fake of the CUDA calls it makes: a device of 400 MiB that fails like a full one."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

PROGRAM = r"""
#include "scratch.h"
#include <cstdio>
#include <cstdlib>
#include <map>
static const size_t CAPACITY = (size_t)400 << 20;
static std::map<void*, size_t> device_blocks; static size_t used; static int host_blocks; static bool host_fails; static cudaError_t last;
static cudaError_t fail() { return last = cudaErrorMemoryAllocation; }
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { if (used + n > CAPACITY) return fail(); *p = malloc(1); device_blocks[*p] = n; used += n; return cudaSuccess; }
cudaError_t cudaFree(void* p) { if (p) { used -= device_blocks.at(p); device_blocks.erase(p); free(p); } return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { if (host_fails) return fail(); *p = malloc(n); ++host_blocks; return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { if (p) { --host_blocks; free(p); } return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
}
#define CHECK(x) do { if (!(x)) { printf("failed at line %d: %s\n", __LINE__, #x); return 1; } } while (0)
static const size_t MB = (size_t)1 << 20;
int main() {
    { Scratch a(0); CHECK(a.take(100) == cudaSuccess && a.b.bytes == MB); }
    CHECK(used == MB && host_blocks == 1);
    { Scratch a(0); CHECK(a.take(MB) == cudaSuccess); }                              // the same block again
    CHECK(used == MB);
    { Scratch a(0), b(0), c(0); CHECK(a.take(60 * MB) == cudaSuccess && b.take(60 * MB) == cudaSuccess && c.take(60 * MB) == cudaSuccess); }
    CHECK(used == 193 * MB);                                                         // kept: 1 + 3 x 64
    { Scratch a(0); CHECK(a.take(300 * MB) == cudaSuccess && a.b.bytes == 300 * MB); CHECK(used == 300 * MB && last == cudaSuccess); }
    CHECK(used == 0 && host_blocks == 0);                                            // above the limit: not kept
    { Scratch a(0), b(0); CHECK(a.take(340 * MB) == cudaSuccess); CHECK(b.take(40 * MB) == cudaSuccess && b.b.bytes == 40 * MB); }      // no room for 64
    scratch_release();
    { Scratch a(0); CHECK(a.take(401 * MB) == cudaErrorMemoryAllocation && last == cudaSuccess && !a.b.dev); }
    host_fails = true;
    { Scratch a(0); CHECK(a.take(MB) == cudaErrorMemoryAllocation && last == cudaSuccess); }
    CHECK(used == 0 && host_blocks == 0);
    host_fails = false;
    {
        Scratch* s[24]; for (Scratch*& p : s) { p = new Scratch(0); CHECK(p->take(MB) == cudaSuccess); }
        for (Scratch* p : s) delete p;
        CHECK(used == 16 * MB && host_blocks == 16);                                 // no more than 16 blocks are kept
    }
    scratch_release();
    CHECK(used == 0 && host_blocks == 0);
    puts("ok");
}
"""


def test_scratch_pool_gives_its_idle_blocks_back_before_a_call_fails(tmp_path):
    src, exe = tmp_path / "pool.cpp", tmp_path / "pool"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(CUDA, "include"), "-I", os.path.join(ROOT, "paper_2107_00961_b200", "csrc"), "-o", exe, src, "-lpthread"])
    assert subprocess.run([exe], capture_output=True, text=True).stdout.strip() == "ok"
