// Builds the edge table with no thread to be had beyond the first few, and with every k-th host
// allocation refused for growing k: a table that answers as the one built freely, or EAT_ERR_OOM;
// never an exception (the library's entry points are C).
#include <dlfcn.h>
#include <pthread.h>

#include <atomic>
#include <cerrno>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <random>

#include "eat_internal.h"

static std::atomic<long> allocations{-1}, threads{-1};      // left to give, < 0 = no limit

static bool take(std::atomic<long> &left) {
    long x = left.load();
    while (x >= 0) {
        if (x == 0) return false;
        if (left.compare_exchange_weak(x, x - 1)) return true;
    }
    return true;
}

void *operator new(size_t n) {
    void *p = take(allocations) ? std::malloc(n ? n : 1) : nullptr;
    if (!p) throw std::bad_alloc();
    return p;
}
void *operator new(size_t n, const std::nothrow_t &) noexcept { return take(allocations) ? std::malloc(n ? n : 1) : nullptr; }
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }

extern "C" int pthread_create(pthread_t *t, const pthread_attr_t *a, void *(*f)(void *), void *arg) {
    using Create = int (*)(pthread_t *, const pthread_attr_t *, void *(*)(void *), void *);
    static const Create real = (Create)dlsym(RTLD_NEXT, "pthread_create");
    return take(threads) ? real(t, a, f, arg) : EAGAIN;
}

namespace eat {
static int last;
int fail(int code, const std::string &) { return last = code; }
void clear_error() {}
}  // namespace eat

using namespace eat;

static int build(HostNet &h, long limit, long n_threads) {
    std::mt19937 rng(7);
    std::vector<int32_t> c[4];
    for (int i = 0; i < 3000; ++i) {
        const int u = (int)(rng() % 60), v = (int)(rng() % 60);
        for (int x[] = {u, v, (int)(rng() % 5000), (int)(1 + rng() % 900)}, k = 0; k < 4; ++k) c[k].push_back(x[k]);
    }
    eat_connections in{60, 3000, c[0].data(), c[1].data(), c[2].data(), c[3].data(), nullptr};
    if (build_host(&in, 3600, 0, h) || build_fused(h)) std::exit(2);
    allocations = limit;
    threads = n_threads;
    const int rc = build_edges(h);
    allocations = threads = -1;
    return rc;
}

static bool same(const HostNet &a, const HostNet &b) {
    return a.er == b.er && a.erow == b.erow && a.ex == b.ex && a.ee_words == b.ee_words &&
           !std::memcmp(a.ee.get(), b.ee.get(), a.ee_words * 4);
}

int main() {
    HostNet free;
    if (build(free, -1, -1)) return 1;
    for (long n : {0L, 1L, 2L}) {
        HostNet h;
        if (build(h, -1, n) || !same(h, free)) return 1;
    }
    int refused = 0;
    for (long n = 0;; n += 1 + n / 8) {
        HostNet h;
        const int rc = build(h, n, -1);
        if (rc == EAT_OK) {
            if (!same(h, free)) return 1;
            break;
        }
        if (rc != EAT_ERR_OOM) return 1;
        ++refused;
    }
    std::printf("%d builds refused\n", refused);
    return refused > 10 ? 0 : 1;
}
