// Memory behind the handles: a small cache of device blocks, and the copy of a large result into the caller's pageable
// memory.  Set-up work (quantising, exporting), where cudaMalloc / cudaFree (0.1 ms each, with a device-wide wait) and the
// driver's single-threaded staging of pageable copies (17 GB/s) cost several times what the kernels do.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>
#include <new>
#include <thread>
#include <utility>

#include "aq_internal.h"

namespace aq {

namespace {

// ---- device blocks ------------------------------------------------------------------
// A released block is kept for the next handle of about its size.  Bounded in bytes and number (a block counts with the bytes
// it was allocated with, however little its last owner asked for); a block that the next
// few releases have not found a use for goes back to the driver, and all of them do when an allocation fails.  Only idle
// blocks come in, so that a block may go to any stream; of the others cudaFree takes care, which waits for the device.  (The
// cache does not: a wait for the whole device ends every recording of a graph on it, another thread's included.)
struct Block {
    void* p;
    size_t bytes;
    int device;
    uint64_t stamp;
};
constexpr size_t CACHE_BYTES = 256u << 20;
constexpr size_t CACHE_BLOCKS = 16;
constexpr uint64_t CACHE_AGE = 16;      // releases

// (no container: nothing here may throw, the callers are C entry points)
struct Cache {
    std::mutex m;
    Block blocks[CACHE_BLOCKS + 1];     // in the order of their release
    size_t n = 0;
    uint64_t clock = 0;
    Block take(size_t i) {
        const Block b = blocks[i];
        std::copy(blocks + i + 1, blocks + n, blocks + i);
        --n;
        return b;
    }
};
Cache& cache() {
    alignas(Cache) static unsigned char memory[sizeof(Cache)];
    static Cache* c = new (memory) Cache;   // (outlives every handle: an interpreter may free some while it exits)
    return *c;
}

// `device` is the current one while this lives (the calling thread's own may be another).
struct OnDevice {
    int before = -1;
    bool changed = false;
    explicit OnDevice(int device) {
        if (cudaGetDevice(&before) != cudaSuccess) { cudaGetLastError(); before = -1; }
        if (before != device) changed = cudaSetDevice(device) == cudaSuccess;
    }
    ~OnDevice() { if (changed && before >= 0) cudaSetDevice(before); }
};

}  // namespace

void* device_alloc(size_t bytes, int device, size_t* held) {
    bytes = (bytes + 511) / 512 * 512;
    *held = bytes;
    Cache& c = cache();
    {
        std::lock_guard<std::mutex> lock(c.m);
        size_t best = c.n;
        for (size_t i = 0; i < c.n; ++i) {
            const Block& b = c.blocks[i];
            if (b.device == device && b.bytes >= bytes && b.bytes <= bytes + bytes / 4 && (best == c.n || b.bytes < c.blocks[best].bytes)) best = i;
        }
        if (best < c.n) {
            const Block b = c.take(best);
            *held = b.bytes;
            return b.p;
        }
    }
    OnDevice here(device);
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) == cudaSuccess) return p;
    cudaGetLastError();
    Block all[CACHE_BLOCKS + 1];
    size_t n = 0;
    {
        std::lock_guard<std::mutex> lock(c.m);
        std::copy(c.blocks, c.blocks + c.n, all);
        std::swap(n, c.n);
    }
    for (size_t i = 0; i < n; ++i) cudaFree(all[i].p);
    if (n > 0 && cudaMalloc(&p, bytes) == cudaSuccess) return p;
    cudaGetLastError();
    return nullptr;
}

void device_release(void* p, size_t held, int device, bool idle) {
    if (p == nullptr) return;
    void* out[CACHE_BLOCKS + 2];
    size_t n_out = 0;
    {
        Cache& c = cache();
        std::lock_guard<std::mutex> lock(c.m);
        ++c.clock;
        if (idle && held <= CACHE_BYTES) c.blocks[c.n++] = {p, held, device, c.clock};
        else out[n_out++] = p;
        size_t total = 0;
        for (size_t i = 0; i < c.n; ++i) total += c.blocks[i].bytes;
        while (c.n > 0 && (total > CACHE_BYTES || c.n > CACHE_BLOCKS || c.blocks[0].stamp + CACHE_AGE < c.clock)) {   // the oldest first
            total -= c.blocks[0].bytes;
            out[n_out++] = c.take(0).p;
        }
    }
    for (size_t i = 0; i < n_out; ++i) cudaFree(out[i]);
}

// ---- device -> pageable host ----------------------------------------------------------
namespace {
constexpr size_t CHUNK = 1u << 20;
constexpr int SLOTS = 8;                // 8 MB of pinned memory, kept
constexpr int MAX_THREADS = 4;
std::mutex g_stage_mutex;
uint8_t* g_stage = nullptr;
}  // namespace

// Copies bytes from device memory to pageable host memory after what `s` holds, and waits for it.  Large copies go
// through a ring of pinned chunks that a few threads empty while the next chunks arrive (22.5 MB: 1350 us as one
// pageable copy).  One such copy at a time; another thread's meanwhile, or a small one, is an ordinary copy.
cudaError_t copy_to_host(void* host, const void* dev, size_t bytes, cudaStream_t s) {
    const size_t n = (bytes + CHUNK - 1) / CHUNK;
    std::unique_lock<std::mutex> lock(g_stage_mutex, std::defer_lock);
    bool staged = n >= 4 && lock.try_lock();
    if (staged && g_stage == nullptr && cudaHostAlloc(reinterpret_cast<void**>(&g_stage), SLOTS * CHUNK, cudaHostAllocPortable) != cudaSuccess) {
        cudaGetLastError();
        g_stage = nullptr;
        staged = false;
    }
    cudaEvent_t ev[SLOTS];
    int n_ev = 0;
    for (; staged && n_ev < SLOTS; ++n_ev)
        if (cudaEventCreateWithFlags(&ev[n_ev], cudaEventDisableTiming) != cudaSuccess) { cudaGetLastError(); staged = false; break; }
    cudaError_t err = cudaSuccess;
    if (staged) {
        const int device = current_device();
        const unsigned cores = std::thread::hardware_concurrency();
        const int n_threads = cores >= 8 ? MAX_THREADS : cores >= 4 ? 2 : 1;   // (a divisor of SLOTS: a slot is always the same thread's)
        std::atomic<size_t> issued{0};
        std::atomic<size_t> emptied[SLOTS] = {};      // chunks of the slot so far
        std::atomic<bool> failed{false};
        auto empty_chunks = [&](size_t first) {
            cudaSetDevice(device);
            for (size_t i = first; i < n; i += (size_t)n_threads) {
                while (issued.load(std::memory_order_acquire) <= i) {
                    if (failed.load(std::memory_order_relaxed)) return;
                    std::this_thread::yield();
                }
                if (cudaEventSynchronize(ev[i % SLOTS]) != cudaSuccess) { failed.store(true); return; }
                std::memcpy(static_cast<uint8_t*>(host) + i * CHUNK, g_stage + (i % SLOTS) * CHUNK, std::min(CHUNK, bytes - i * CHUNK));
                emptied[i % SLOTS].fetch_add(1, std::memory_order_release);
            }
        };
        std::thread threads[MAX_THREADS];
        try {
            for (int t = 0; t < n_threads; ++t) threads[t] = std::thread(empty_chunks, (size_t)t);
        } catch (...) {   // the system has no thread to give: the ordinary copy below
            staged = false;
            failed.store(true);
        }
        for (size_t i = 0; i < n && staged && err == cudaSuccess; ++i) {
            while (emptied[i % SLOTS].load(std::memory_order_acquire) < i / SLOTS && !failed.load(std::memory_order_relaxed)) std::this_thread::yield();
            if (failed.load(std::memory_order_relaxed)) break;
            err = cudaMemcpyAsync(g_stage + (i % SLOTS) * CHUNK, static_cast<const uint8_t*>(dev) + i * CHUNK, std::min(CHUNK, bytes - i * CHUNK),
                                  cudaMemcpyDeviceToHost, s);
            if (err == cudaSuccess) err = cudaEventRecord(ev[i % SLOTS], s);
            if (err == cudaSuccess) issued.store(i + 1, std::memory_order_release);
        }
        if (err != cudaSuccess) failed.store(true);
        for (std::thread& t : threads)
            if (t.joinable()) t.join();
        if (failed.load()) cudaStreamSynchronize(s);   // chunks that were issued may be on their way into the ring, the next copy's
        if (staged && err == cudaSuccess && failed.load()) { err = cudaGetLastError(); if (err == cudaSuccess) err = cudaErrorUnknown; }
    }
    if (!staged) {
        err = cudaMemcpyAsync(host, dev, bytes, cudaMemcpyDeviceToHost, s);
        if (err == cudaSuccess) err = cudaStreamSynchronize(s);
    }
    for (int i = 0; i < n_ev; ++i) cudaEventDestroy(ev[i]);
    return err;
}

}  // namespace aq
