// Memory behind the handles: a small cache of device blocks, and the copy of a large result into the caller's pageable
// memory.  Set-up work (quantising, exporting), where cudaMalloc / cudaFree (0.1 ms each, with a device-wide wait) and the
// driver's single-threaded staging of pageable copies (17 GB/s) cost several times what the kernels do.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>
#include <thread>
#include <vector>

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

struct Cache {
    std::mutex m;
    std::vector<Block> blocks;
    uint64_t clock = 0;
};
Cache& cache() {
    static Cache* c = new Cache;        // (outlives every handle: an interpreter may free some while it exits)
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
        size_t best = c.blocks.size();
        for (size_t i = 0; i < c.blocks.size(); ++i) {
            const Block& b = c.blocks[i];
            if (b.device == device && b.bytes >= bytes && b.bytes <= bytes + bytes / 4 && (best == c.blocks.size() || b.bytes < c.blocks[best].bytes)) best = i;
        }
        if (best < c.blocks.size()) {
            void* p = c.blocks[best].p;
            *held = c.blocks[best].bytes;
            c.blocks.erase(c.blocks.begin() + best);
            return p;
        }
    }
    OnDevice here(device);
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) == cudaSuccess) return p;
    cudaGetLastError();
    std::vector<Block> all;
    {
        std::lock_guard<std::mutex> lock(c.m);
        all.swap(c.blocks);
    }
    for (const Block& b : all) cudaFree(b.p);
    if (!all.empty() && cudaMalloc(&p, bytes) == cudaSuccess) return p;
    cudaGetLastError();
    return nullptr;
}

void device_release(void* p, size_t held, int device, bool idle) {
    if (p == nullptr) return;
    std::vector<void*> out;
    {
        Cache& c = cache();
        std::lock_guard<std::mutex> lock(c.m);
        ++c.clock;
        if (idle && held <= CACHE_BYTES) c.blocks.push_back({p, held, device, c.clock});
        else out.push_back(p);
        size_t total = 0;
        for (const Block& b : c.blocks) total += b.bytes;
        // the oldest first: blocks are in the order of their release
        while (!c.blocks.empty() && (total > CACHE_BYTES || c.blocks.size() > CACHE_BLOCKS || c.blocks.front().stamp + CACHE_AGE < c.clock)) {
            total -= c.blocks.front().bytes;
            out.push_back(c.blocks.front().p);
            c.blocks.erase(c.blocks.begin());
        }
    }
    for (void* q : out) cudaFree(q);
}

// ---- device -> pageable host ----------------------------------------------------------
namespace {
constexpr size_t CHUNK = 1u << 20;
constexpr int SLOTS = 8;                // 8 MB of pinned memory, kept
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
        const int n_threads = cores >= 8 ? 4 : cores >= 4 ? 2 : 1;
        std::atomic<size_t> issued{0};
        std::atomic<bool> failed{false};
        std::vector<std::atomic<uint8_t>> done(n);
        for (auto& d : done) d.store(0, std::memory_order_relaxed);
        auto empty_chunks = [&](size_t first) {
            cudaSetDevice(device);
            for (size_t i = first; i < n; i += (size_t)n_threads) {
                while (issued.load(std::memory_order_acquire) <= i)
                    if (failed.load(std::memory_order_relaxed)) return;
                if (cudaEventSynchronize(ev[i % SLOTS]) != cudaSuccess) { failed.store(true); return; }
                std::memcpy(static_cast<uint8_t*>(host) + i * CHUNK, g_stage + (i % SLOTS) * CHUNK, std::min(CHUNK, bytes - i * CHUNK));
                done[i].store(1, std::memory_order_release);
            }
        };
        std::vector<std::thread> threads;
        for (int t = 0; t < n_threads; ++t) threads.emplace_back(empty_chunks, (size_t)t);
        for (size_t i = 0; i < n && err == cudaSuccess; ++i) {
            if (i >= SLOTS)
                while (!done[i - SLOTS].load(std::memory_order_acquire) && !failed.load(std::memory_order_relaxed)) std::this_thread::yield();
            if (failed.load(std::memory_order_relaxed)) break;
            err = cudaMemcpyAsync(g_stage + (i % SLOTS) * CHUNK, static_cast<const uint8_t*>(dev) + i * CHUNK, std::min(CHUNK, bytes - i * CHUNK),
                                  cudaMemcpyDeviceToHost, s);
            if (err == cudaSuccess) err = cudaEventRecord(ev[i % SLOTS], s);
            if (err == cudaSuccess) issued.store(i + 1, std::memory_order_release);
        }
        if (err != cudaSuccess) failed.store(true);
        for (std::thread& t : threads) t.join();
        if (err == cudaSuccess && failed.load()) { err = cudaGetLastError(); if (err == cudaSuccess) err = cudaErrorUnknown; }
    } else {
        err = cudaMemcpyAsync(host, dev, bytes, cudaMemcpyDeviceToHost, s);
        if (err == cudaSuccess) err = cudaStreamSynchronize(s);
    }
    for (int i = 0; i < n_ev; ++i) cudaEventDestroy(ev[i]);
    return err;
}

}  // namespace aq
