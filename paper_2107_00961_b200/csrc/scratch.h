// Scratch of the layer-level calls.  cudaMalloc and cudaFree cost 100 to 300 us each (cudaFree also waits for the whole device), many
// times the kernels of a small layer, so a call borrows a block and hands it back once its work is done (every call
// synchronises its stream before it returns, so a block handed back is idle).  A block: device scratch plus pinned host memory for
// the descriptors, which go up in one asynchronous copy.  A borrowed block belongs to one call alone, so any number of threads and
// streams may be inside the calls.  Idle blocks are kept up to SCRATCH_IDLE_BYTES and SCRATCH_IDLE_BLOCKS over all devices, the rest is
// freed at once; scratch_release() gives back the idle ones, as does a call that finds no memory for its own.
#pragma once
#include <cuda_runtime.h>
#include <algorithm>
#include <cstring>
#include <mutex>

namespace {
constexpr size_t SCRATCH_IDLE_BYTES = (size_t)256 << 20, SCRATCH_HOST_BYTES = 16384;
constexpr int SCRATCH_IDLE_BLOCKS = 16;
struct ScratchBlock { char* dev = nullptr; char* host = nullptr; size_t bytes = 0; int device = -1; };
std::mutex g_scratch_mutex;
struct ScratchList {                                          // of fixed room: nothing here may throw
    ScratchBlock at[SCRATCH_IDLE_BLOCKS + 1]; int n = 0;
    void put(const ScratchBlock& b) { at[n++] = b; }
    ScratchBlock take(int i) { const ScratchBlock b = at[i]; at[i] = at[--n]; return b; }
};
ScratchList g_scratch_idle;                                   // guarded by the mutex

void scratch_free(const ScratchList& l) { for (int i = 0; i < l.n; ++i) { cudaFree(l.at[i].dev); cudaFreeHost(l.at[i].host); } }
void scratch_release() {
    ScratchList out;
    { std::lock_guard<std::mutex> lock(g_scratch_mutex); std::swap(out, g_scratch_idle); }
    scratch_free(out);
}

struct Scratch {
    ScratchBlock b;
    cudaStream_t st; size_t staged = 0; bool busy = false;
    explicit Scratch(cudaStream_t s) : st(s) {}
    Scratch(const Scratch&) = delete;
    cudaError_t allocate(size_t bytes, int dev) {
        b.bytes = bytes; b.device = dev;
        cudaError_t e = cudaMalloc(&b.dev, bytes);
        if (e == cudaSuccess) {
            e = cudaHostAlloc(&b.host, SCRATCH_HOST_BYTES, cudaHostAllocPortable);
            if (e != cudaSuccess) cudaFree(b.dev);
        }
        if (e != cudaSuccess) { cudaGetLastError(); b = ScratchBlock(); }      // the caller is told; nothing stays behind for a later check
        return e;
    }
    cudaError_t take(size_t bytes) {
        int dev = 0; cudaError_t e = cudaGetDevice(&dev); if (e != cudaSuccess) return e;
        {
            std::lock_guard<std::mutex> lock(g_scratch_mutex);
            int best = -1;
            for (int i = 0; i < g_scratch_idle.n; ++i)
                if (g_scratch_idle.at[i].device == dev && g_scratch_idle.at[i].bytes >= bytes && (best < 0 || g_scratch_idle.at[i].bytes < g_scratch_idle.at[best].bytes)) best = i;
            if (best >= 0) { b = g_scratch_idle.take(best); return cudaSuccess; }
        }
        size_t room = (size_t)1 << 20; while (room < bytes && room < ((size_t)64 << 20)) room *= 2;     // few sizes, so that blocks serve other layers too
        e = allocate(std::max(room, bytes), dev);
        if (e == cudaSuccess) return e;
        scratch_release();                                     // on a nearly full device the idle blocks, and the rounding up, may be what is in the way
        return allocate(bytes, dev);
    }
    // descriptors are laid out in the pinned memory at the offsets they have in the block, then sent as one copy
    void stage(size_t at, const void* what, size_t bytes) { memcpy(b.host + at, what, bytes); staged = std::max(staged, at + bytes); }
    cudaError_t send() { busy = true; return cudaMemcpyAsync(b.dev, b.host, staged, cudaMemcpyHostToDevice, st); }
    cudaError_t wait() { const cudaError_t e = cudaStreamSynchronize(st); busy = false; return e; }
    ~Scratch() {
        if (!b.dev) return;
        if (busy) cudaStreamSynchronize(st);                   // an error path left work in flight
        ScratchList out;
        {
            std::lock_guard<std::mutex> lock(g_scratch_mutex);
            g_scratch_idle.put(b);
            size_t total = 0; for (int i = 0; i < g_scratch_idle.n; ++i) total += g_scratch_idle.at[i].bytes;
            while (total > SCRATCH_IDLE_BYTES || g_scratch_idle.n > SCRATCH_IDLE_BLOCKS) {      // the largest goes first
                int big = 0; for (int i = 1; i < g_scratch_idle.n; ++i) if (g_scratch_idle.at[i].bytes > g_scratch_idle.at[big].bytes) big = i;
                total -= g_scratch_idle.at[big].bytes; out.put(g_scratch_idle.take(big));
            }
        }
        scratch_free(out);
    }
};
}
