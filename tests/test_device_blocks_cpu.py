"""Host logic of `csrc/aq_memory.cu` (device blocks out of a bounded cache, copies into pageable memory), compiled with the
host compiler against a stand-in for the CUDA runtime that knows on which device a block lies and what was asked of it."""
import os
import shutil
import subprocess
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_24011_b200", "csrc")
pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host C++ compiler")

FAKE = textwrap.dedent(r"""
    #pragma once
    #include <atomic>
    #include <cstddef>
    #include <cstdint>
    #include <cstdio>
    #include <cstdlib>
    #include <cstring>
    #include <map>
    #include <mutex>
    typedef struct FakeStream* cudaStream_t;
    typedef struct FakeEvent* cudaEvent_t;
    enum cudaError_t { cudaSuccess = 0, cudaErrorMemoryAllocation = 2, cudaErrorUnknown = 999 };
    enum cudaMemcpyKind { cudaMemcpyDeviceToHost = 2 };
    constexpr unsigned cudaHostAllocPortable = 1, cudaEventDisableTiming = 2;
    namespace fake {
    struct Alloc { int device; size_t bytes; };
    inline std::mutex m;
    inline std::map<void*, Alloc> live;         // device blocks the driver has given out
    inline thread_local int current = 0;
    inline size_t limit = SIZE_MAX, used = 0;   // device memory
    inline int mallocs = 0, frees = 0, device_syncs = 0;
    inline std::atomic<int> stream_syncs{0}, copies{0}, copies_fail_from{1 << 30}, event_syncs_fail_from{1 << 30}, event_syncs{0};
    inline std::atomic<bool> unsynced{false};   // a copy was issued and its stream has not been waited for since
    }
    inline cudaError_t cudaGetDevice(int* d) { *d = fake::current; return cudaSuccess; }
    inline cudaError_t cudaSetDevice(int d) { fake::current = d; return cudaSuccess; }
    inline cudaError_t cudaGetLastError() { return cudaSuccess; }
    inline cudaError_t cudaDeviceSynchronize() { ++fake::device_syncs; return cudaSuccess; }
    inline cudaError_t cudaMalloc(void** p, size_t n) {
        std::lock_guard<std::mutex> l(fake::m);
        if (fake::used + n > fake::limit) return cudaErrorMemoryAllocation;
        *p = std::malloc(n);
        fake::live[*p] = {fake::current, n}; fake::used += n; ++fake::mallocs;
        return cudaSuccess;
    }
    inline cudaError_t cudaFree(void* p) {
        std::lock_guard<std::mutex> l(fake::m);
        auto it = fake::live.find(p);
        if (it == fake::live.end()) { std::printf("freed twice\n"); std::exit(1); }
        fake::used -= it->second.bytes; fake::live.erase(it); ++fake::frees;
        std::free(p);
        return cudaSuccess;
    }
    inline cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = std::malloc(n); return cudaSuccess; }
    inline cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = reinterpret_cast<cudaEvent_t>(std::malloc(1)); return cudaSuccess; }
    inline cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
    inline cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
    inline cudaError_t cudaEventSynchronize(cudaEvent_t) { return fake::event_syncs++ >= fake::event_syncs_fail_from ? cudaErrorUnknown : cudaSuccess; }
    inline cudaError_t cudaStreamSynchronize(cudaStream_t) { ++fake::stream_syncs; fake::unsynced = false; return cudaSuccess; }
    inline cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
        if (fake::copies++ >= fake::copies_fail_from) return cudaErrorUnknown;
        fake::unsynced = true;
        std::memcpy(d, s, n);
        return cudaSuccess;
    }
""")

MAIN = r"""
    #include "aq_memory.cu"
    namespace aq { int current_device() { int d = 0; cudaGetDevice(&d); return d; } }
    using namespace aq;
    #define CHECK(c) do { if (!(c)) { std::printf("FAIL line %d: %s\n", __LINE__, #c); return 1; } } while (0)
"""


def _run(tmp_path, body, before=""):
    (tmp_path / "cuda_runtime.h").write_text(FAKE)
    src = tmp_path / "t.cpp"
    src.write_text(textwrap.dedent(MAIN) + textwrap.dedent(before) + "int main() {\n" + textwrap.dedent(body) + '\n    std::printf("ok\\n");\n    return 0;\n}\n')
    exe = tmp_path / "t"
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", str(tmp_path), "-I", CSRC, str(src), "-o", str(exe), "-ldl"], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr


def test_a_block_lies_on_the_device_it_was_asked_for(tmp_path):
    _run(tmp_path, r"""
        fake::current = 1;
        size_t held;
        void* p = device_alloc(1 << 20, 0, &held);            // a handle of device 0 exported while device 1 is current
        CHECK(p && fake::live[p].device == 0 && fake::current == 1);
        device_release(p, held, 0, true);
        fake::current = 0;
        void* q = device_alloc(1 << 20, 0, &held);            // the next handle of device 0 may be built on that block
        CHECK(q && fake::live[q].device == 0);
        // the retry after the cache has been emptied looks at the device, too
        void* r = device_alloc(3 << 20, 0, &held);
        device_release(r, held, 0, true);
        fake::current = 1;
        fake::limit = fake::used;
        void* t = device_alloc(2 << 20, 0, &held);
        CHECK(t && fake::live[t].device == 0 && fake::current == 1);
    """)


def test_a_block_counts_with_the_bytes_it_has(tmp_path):
    """Ten blocks of 24 MB are handed out again for requests of 20 and 16 MB, two of 40 MB join: what the cache keeps with
    nothing in use stays within its 256 MB."""
    _run(tmp_path, r"""
        void* p[10];
        size_t held[10];
        for (size_t s : {24u << 20, 20u << 20, 16u << 20}) {
            for (int i = 0; i < 10; ++i) {
                p[i] = device_alloc(s, 0, &held[i]);
                CHECK(p[i] && held[i] == fake::live[p[i]].bytes && held[i] >= s);
            }
            for (int i = 0; i < 10; ++i) device_release(p[i], held[i], 0, true);
        }
        CHECK(fake::mallocs >= 10 && fake::used >= (200u << 20) && fake::used <= (256u << 20));
        void* q[2];
        size_t q_held[2];
        for (int i = 0; i < 2; ++i) q[i] = device_alloc(40u << 20, 0, &q_held[i]);
        for (int i = 0; i < 2; ++i) device_release(q[i], q_held[i], 0, true);
        CHECK(fake::used <= (256u << 20));
    """)


def test_a_busy_block_goes_to_the_driver_and_the_device_is_not_waited_for(tmp_path):
    _run(tmp_path, r"""
        size_t held;
        void* p = device_alloc(1 << 20, 0, &held);
        device_release(p, held, 0, false);
        CHECK(fake::frees == 1);
        p = device_alloc(1 << 20, 0, &held);
        CHECK(fake::mallocs == 2);
        device_release(p, held, 0, true);
        CHECK(device_alloc(1 << 20, 0, &held) == p && fake::mallocs == 2);
        CHECK(fake::device_syncs == 0);
    """)


THREADS = r"""
    #include <dlfcn.h>
    #include <errno.h>
    #include <pthread.h>
    static int threads_left = 1 << 30;              // what the system still gives
    extern "C" int pthread_create(pthread_t* t, const pthread_attr_t* a, void* (*f)(void*), void* x) {
        static auto real = reinterpret_cast<int (*)(pthread_t*, const pthread_attr_t*, void* (*)(void*), void*)>(dlsym(RTLD_NEXT, "pthread_create"));
        return threads_left-- > 0 ? real(t, a, f, x) : EAGAIN;
    }
    #include <vector>
    static std::vector<uint8_t> bytes_of(size_t n) {
        std::vector<uint8_t> v(n);
        for (size_t i = 0; i < n; ++i) v[i] = (uint8_t)(i * 2654435761u >> 13);
        return v;
    }
"""


def test_a_copy_without_threads_is_an_ordinary_copy(tmp_path):
    """The system refuses the first or a later helper thread: nothing is thrown out of the call, every byte arrives."""
    _run(tmp_path, r"""
        const auto from = bytes_of((21u << 20) + 5);
        for (int given = 0; given <= 4; ++given) {
            threads_left = given;
            std::vector<uint8_t> to(from.size(), 0);
            CHECK(aq::copy_to_host(to.data(), from.data(), from.size(), nullptr) == cudaSuccess && to == from);
        }
    """, before=THREADS)


def test_a_failed_copy_leaves_nothing_in_flight(tmp_path):
    """A chunk cannot be issued, or a helper's wait fails: the error is reported, and the ring is given up only after the
    stream has been waited for."""
    _run(tmp_path, r"""
        const auto from = bytes_of(21u << 20);
        std::vector<uint8_t> to(from.size());
        for (int at : {1, 7, 12, 20}) {
            fake::copies = 0; fake::copies_fail_from = at;
            CHECK(aq::copy_to_host(to.data(), from.data(), from.size(), nullptr) != cudaSuccess && !fake::unsynced);
        }
        fake::copies_fail_from = 1 << 30;
        for (int at : {0, 3, 15}) {
            fake::event_syncs = 0; fake::event_syncs_fail_from = at;
            CHECK(aq::copy_to_host(to.data(), from.data(), from.size(), nullptr) != cudaSuccess && !fake::unsynced);
        }
        fake::event_syncs_fail_from = 1 << 30;
        std::fill(to.begin(), to.end(), 0);
        CHECK(aq::copy_to_host(to.data(), from.data(), from.size(), nullptr) == cudaSuccess && to == from);
    """, before=THREADS)
