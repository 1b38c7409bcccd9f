// klmc_cluster_histogram while the process has no host memory to give: operator new of this
// program throws when told to, in the library too.
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <new>
#include <vector>

#include "klmc.h"

static bool refuse = false;

void *operator new(size_t n)
{
    void *p = refuse ? nullptr : std::malloc(n);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }

int main()
{
    klmc_ctx *c = nullptr;
    if (klmc_create(&c, 64, 0.4, 0.6, 5) != KLMC_OK) return 2;
    std::vector<int64_t> s(100), n(100), s2(100), n2(100);
    int64_t k = 0, k2 = 0;
    if (klmc_cluster_histogram(c, 1, s.data(), n.data(), 100, &k) != KLMC_OK) return 3;
    refuse = true;
    const klmc_status st = klmc_cluster_histogram(c, 1, s2.data(), n2.data(), 100, &k2);
    refuse = false;
    if (st != KLMC_OK || k != k2 || k < 1 || s != s2 || n != n2) return 4;
    std::puts("same");
    return klmc_destroy(c) == KLMC_OK ? 0 : 5;
}
