// Host allocations that fail on demand, for the library that fake_cuda.cpp is linked into (the linker binds
// these to that library alone).
#include <cstdint>
#include <cstdlib>
#include <new>

static int64_t until_throw = -1;   // allocations until one throws (-1: none does)

extern "C" void fake_throw_after(int64_t allocations) { until_throw = allocations; }

void* operator new(size_t size)
{
    if (until_throw >= 0 && until_throw-- == 0)
        throw std::bad_alloc();
    void* p = std::malloc(size ? size : 1);
    if (!p)
        throw std::bad_alloc();
    return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }
