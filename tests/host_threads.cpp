// Loops over the host's threads (run_ranges) under failures: the n-th
// allocation from here on throws, or the n-th thread cannot be started.  Every
// range has to run exactly once, or the caller to get the exception, with all
// threads ended.  Prints "ok" and counts.
#include <dlfcn.h>
#include <pthread.h>

#include <atomic>
#include <cerrno>
#include <cstdio>
#include <cstdlib>
#include <new>

#include "gks_internal.h"

static std::atomic<long> alloc_in{-1}, thread_in{-1};

void* operator new(std::size_t n) {
    if (alloc_in.load() >= 0 && alloc_in.fetch_sub(1) == 0) throw std::bad_alloc();
    if (void* p = std::malloc(n)) return p;
    throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }

extern "C" int pthread_create(pthread_t* t, const pthread_attr_t* a, void* (*f)(void*), void* x) {
    using Fn = int (*)(pthread_t*, const pthread_attr_t*, void* (*)(void*), void*);
    static const Fn real = reinterpret_cast<Fn>(dlsym(RTLD_NEXT, "pthread_create"));
    if (thread_in.load() >= 0 && thread_in.fetch_sub(1) == 0) return EAGAIN;
    return real(t, a, f, x);
}

static int done = 0, refused = 0;

// one loop of 4 ranges over 1,000 items, each range with an allocation of its own
static void loop() {
    static std::atomic<int> seen[1000];
    for (auto& s : seen) s = 0;
    bool threw = false;
    try {
        gks::run_ranges(1000, 4, [&](int64_t, int64_t lo, int64_t hi) {
            std::vector<int> own((size_t)(hi - lo), 1);
            for (int64_t i = lo; i < hi; ++i) seen[i] += own[(size_t)(i - lo)];
        });
    } catch (const std::bad_alloc&) {
        threw = true;
    }
    alloc_in = thread_in = -1;
    for (auto& s : seen)
        if (s > 1 || (s == 0 && !threw)) {
            std::puts("a range ran twice or not at all");
            std::exit(1);
        }
    (threw ? refused : done)++;
}

int main() {
    for (int rep = 0; rep < 50; ++rep) {
        for (int n = 0; n < 12; ++n) {
            alloc_in = n;
            loop();
        }
        for (int n = 0; n < 4; ++n) {
            thread_in = n;
            loop();
        }
    }
    std::printf("ok %d %d\n", done, refused);
}
