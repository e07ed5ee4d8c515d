// Owners of device memory (csrc/devmem.cuh) on a fake allocator that refuses
// what is asked to: after a refusal every array is live memory or empty, and
// a smaller request serves from live memory.
#include <cstdio>
#include <cstdlib>
#include <map>

#include "devmem.cuh"

static std::map<char*, size_t> live;  // blocks given out and not given back
static size_t largest = SIZE_MAX;     // requests above this are refused

static cudaError_t last_error = cudaSuccess;
extern "C" cudaError_t cudaGetLastError() {
    const cudaError_t e = last_error;
    last_error = cudaSuccess;
    return e;
}
extern "C" cudaError_t cudaMalloc(void** p, size_t bytes) {
    *p = nullptr;
    if (bytes > largest) return last_error = cudaErrorMemoryAllocation;
    char* q = static_cast<char*>(std::malloc(bytes));
    live[q] = bytes;
    *p = q;
    return cudaSuccess;
}
// the bytes stay reserved, so that a later block never has an old address
extern "C" cudaError_t cudaFree(void* p) {
    if (p && !live.erase(static_cast<char*>(p))) return cudaErrorInvalidValue;
    return cudaSuccess;
}

static int bad = 0;
template <class T>
static void check(const char* what, const lbmdem::DBuf<T>& b, size_t need) {
    const char* q = reinterpret_cast<const char*>(b.p);
    bool ok = b.p == nullptr && b.n == 0 && need == 0;
    for (const auto& l : live) ok |= q >= l.first && q + sizeof(T) * b.n <= l.first + l.second && b.n >= need;
    if (!ok) {
        std::printf("%s: %p, %zu elements, %zu needed, not in a live block\n", what, (const void*)q, b.n, need);
        bad = 1;
    }
}

static void cells(const char* what, const lbmdem::CellBufs& c, size_t np, size_t ncell) {
    check(what, c.of, np);
    check(what, c.order, np);
    check(what, c.count, ncell ? ncell + 1 : 0);
    check(what, c.start, ncell ? ncell + 1 : 0);
    check(what, c.fill, ncell);
}

// two arrays in a slab, as a packing's neighbour lists are kept: made again
// when the last of them is too small
struct Lists {
    lbmdem::Slab slab;
    lbmdem::DBuf<int> a, a2;
    lbmdem::DBuf<float> b;
    cudaError_t ensure(size_t n) {
        if (b.n >= n && b.p) return cudaSuccess;
        auto parts = [&] {
            slab.take(a, n);
            slab.take(a2, n);
            slab.take(b, n);
        };
        slab.measure();
        parts();
        if (cudaError_t e = slab.reserve()) return e;
        parts();
        return cudaSuccess;
    }
};

int main() {
    {
        lbmdem::CellBufs c;
        if (c.ensure(100, 60)) bad = 1;
        cells("a first packing", c, 100, 60);
        if (c.ensure(80, 60)) bad = 1;  // kept
        cells("a smaller packing", c, 80, 60);
        largest = 100000;
        if (c.ensure(100000, 60) != cudaErrorMemoryAllocation) bad = 1;
        cells("after a refusal", c, 0, 0);
        if (c.ensure(50, 30)) bad = 1;
        cells("a packing after a refusal", c, 50, 30);
        largest = SIZE_MAX;
        if (c.ensure(100000, 90)) bad = 1;
        cells("a larger packing", c, 100000, 90);
    }
    {
        Lists l;
        if (l.ensure(1000)) bad = 1;
        l.a.swap(l.a2);
        if (l.ensure(2000)) bad = 1;
        check("lists", l.a, 2000);
        check("lists", l.a2, 2000);
        // an array of its own in the place of a part is its owner's to keep
        if (l.a.alloc(3000)) bad = 1;
        largest = 10000;
        if (l.ensure(4000) != cudaErrorMemoryAllocation) bad = 1;
        check("its own array after a refusal", l.a, 3000);
        check("lists after a refusal", l.a2, 0);
        check("lists after a refusal", l.b, 0);
        if (l.ensure(500)) bad = 1;
        check("lists", l.a2, 500);
        check("lists", l.b, 500);
        largest = SIZE_MAX;
    }
    {
        lbmdem::ConversionBufs<int> f;
        auto whole = [&](const char* what, size_t n) {
            check(what, f.rec, 2 * n);
            check(what, f.scratch, 9 * n);
            check(what, f.valid, 3 * n);
        };
        if (f.ensure(100, 3)) bad = 1;
        whole("conversions", 100);
        largest = 20000;  // the queue fits, the populations do not
        if (f.ensure(1000, 3) != cudaErrorMemoryAllocation) bad = 1;
        if (f.ensure(100, 3)) bad = 1;
        whole("conversions after a refusal", 100);
        largest = SIZE_MAX;
    }
    if (last_error != cudaSuccess) {
        std::printf("a refusal is left for a later check to find\n");
        bad = 1;
    }
    if (!live.empty()) {
        std::printf("%zu blocks not given back\n", live.size());
        bad = 1;
    }
    if (!bad) std::printf("ok\n");
    return bad;
}
