// Host check of the error words (csrc/vbq_error_words.h) against a fake CUDA
// runtime: words on one device survive a reset of another, live calls of many
// threads never share a line (also when there are more of them than lines),
// words start at zero, a kernel still to come is waited for before its words go
// back, and only the pages stay allocated.
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <memory>
#include <set>
#include <thread>
#include <vector>

#include "vbq_error_words.h"

static thread_local int t_device = 0;
static std::mutex g_mu;
static std::map<char*, std::pair<size_t, int>> g_allocs;      // live: size, device
static std::atomic<int> g_syncs{0};

cudaError_t cudaGetDevice(int* d) { *d = t_device; return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t bytes, unsigned int) {
    char* m = static_cast<char*>(std::malloc(bytes));
    std::memset(m, 0xA5, bytes);
    std::lock_guard<std::mutex> lock(g_mu);
    g_allocs[m] = {bytes, t_device};
    *p = m;
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_allocs.erase(static_cast<char*>(p))) return cudaErrorInvalidValue;
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { ++g_syncs; return cudaSuccess; }

// What a device reset does to pinned memory allocated in the device's context
// (the memory itself is kept here, so that a stray access is seen, not made).
static void reset_device(int dev) {
    std::lock_guard<std::mutex> lock(g_mu);
    for (auto it = g_allocs.begin(); it != g_allocs.end();) it = it->second.second == dev ? g_allocs.erase(it) : std::next(it);
}
static bool live(const void* p) {
    std::lock_guard<std::mutex> lock(g_mu);
    for (auto& a : g_allocs)
        if (p >= a.first && p < a.first + a.second.first) return true;
    return false;
}

static int faults = 0;
static void expect(bool ok, const char* what) {
    if (!ok) ++faults;
    std::printf("%s %s\n", ok ? "ok  " : "FAIL", what);
}

int main() {
    {   // the first call on device 0, the next on device 1, then device 0 is reset
        t_device = 0;
        { vbq::ErrorWords e; expect(e.get(nullptr) == cudaSuccess && live(e.arm(0)), "words on device 0"); e.settle(); }
        t_device = 1;
        { vbq::ErrorWords e; expect(e.get(nullptr) == cudaSuccess && live(e.arm(1)), "words on device 1"); e.settle(); }
        reset_device(0);
        vbq::ErrorWords e;
        expect(e.get(nullptr) == cudaSuccess && live(e.arm(0)), "words on device 1 after a reset of device 0");
        e.settle();
    }
    {   // more live calls than lines: no two on one line, zero at the start
        std::vector<std::unique_ptr<vbq::ErrorWords>> calls;
        std::set<uintptr_t> lines;
        bool zero = true, ok = true;
        for (int i = 0; i < 150; ++i) {
            calls.emplace_back(new vbq::ErrorWords());
            ok &= calls.back()->get(nullptr) == cudaSuccess;
            zero &= !calls.back()->set(0) && !calls.back()->set(1);
            uint32_t* w = calls.back()->arm(0);
            calls.back()->settle();
            ok &= live(w) && live(w + 1);
            lines.insert(reinterpret_cast<uintptr_t>(w));
            w[0] = w[1] = 7;
        }
        expect(ok && lines.size() == 150, "150 live calls on words of their own");
        expect(zero, "words start at zero");
        bool seen = true;
        for (auto& c : calls) seen &= c->set(0) && c->set(1);
        expect(seen, "an error is seen");
    }
    expect(g_allocs.size() == 1, "only device 1's page is left");
    {   // threads on two devices
        std::atomic<int> bad{0};
        std::vector<std::thread> ts;
        for (int t = 0; t < 90; ++t)
            ts.emplace_back([t, &bad] {
                t_device = 1 + t % 2;
                for (int i = 0; i < 300; ++i) {
                    vbq::ErrorWords e;
                    if (e.get(nullptr) != cudaSuccess || e.set(0) || e.set(1)) { ++bad; continue; }
                    volatile uint32_t* w = e.arm(0);
                    w[0] = (uint32_t)(t + 1);
                    w[1] = (uint32_t)i;
                    std::this_thread::yield();
                    if (w[0] != (uint32_t)(t + 1) || w[1] != (uint32_t)i) ++bad;
                    e.settle();
                }
            });
        for (auto& t : ts) t.join();
        expect(bad == 0, "90 threads never meet on a line");
        expect(g_allocs.size() == 2, "one page per device is left");
    }
    {   // an armed call that is not settled is waited for when it ends
        const int before = g_syncs;
        { vbq::ErrorWords e; e.get(nullptr); e.arm(0); }
        expect(g_syncs == before + 1, "a kernel still to come is waited for");
        { vbq::ErrorWords e; e.get(nullptr); e.arm(0); e.settle(); }
        expect(g_syncs == before + 2, "a settled call waits once");
        { vbq::ErrorWords e; e.get(nullptr); }
        expect(g_syncs == before + 2, "a call without a kernel does not wait");
    }
    std::printf("%s\n", faults ? "FAILED" : "ALL OK");
    return faults ? 1 : 0;
}
