// parallel_for when threads cannot be had: every allocation from the n-th on fails.  The work must be done all the same, and
// nothing may end the process (the callers are C entry points).  And no thread for less than `at_least` items.
#include <cstdio>
#include <cstdlib>
#include <new>

#include "prq_internal.h"

static std::atomic<bool> g_fail{false};
static std::atomic<int> g_left{0};
void* operator new(std::size_t n) {
    if (g_fail && --g_left < 0) throw std::bad_alloc();
    if (void* p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }

int main() {
    for (int left = 0; left < 12; ++left) {
        std::atomic<long> done{0};
        g_left = left;
        g_fail = true;
        prq::parallel_for(1000, [&](long lo, long hi) { done += hi - lo; });
        g_fail = false;
        if (done != 1000) { std::printf("%d allocations: %ld of 1000\n", left, done.load()); return 1; }
    }
    std::atomic<int> shares{0};
    prq::parallel_for(599, [&](long, long) { ++shares; }, 300);
    if (shares != 1) return 1;
    // an exception of the caller's own share arrives after the other shares are through
    std::atomic<long> done{0};
    bool caught = false;
    try {
        prq::parallel_for(1000, [&](long lo, long hi) { if (lo == 0) throw std::bad_alloc(); done += hi - lo; });
    } catch (const std::bad_alloc&) {
        caught = true;
    }
    return caught ? 0 : 1;
}
