// devmem.cuh -- owners of device memory: single arrays, several arrays in one
// block, and the groups of arrays a context keeps from one packing to the
// next.  Host code without kernels.
//
// A call that needs memory may be refused it, and the context goes on with the
// next call: whatever an owner holds after a refusal is either live memory or
// nothing (p null, n 0), never a part of a block that was given back.
#pragma once
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <utility>
#include <vector>

namespace lbmdem {

template <class T>
struct DBuf {
    T* p = nullptr;
    size_t n = 0;
    bool own = true;  // false: a part of a Slab
    DBuf() = default;
    DBuf(const DBuf&) = delete;
    DBuf& operator=(const DBuf&) = delete;
    ~DBuf() { release(); }
    cudaError_t alloc(size_t count) {
        release();
        if (count == 0) count = 1;
        cudaError_t e = cudaMalloc((void**)&p, sizeof(T) * count);
        if (e != cudaSuccess) {
            cudaGetLastError();  // reported here: not again after a later launch
            p = nullptr;
            n = 0;
            return e;
        }
        n = count;
        return cudaSuccess;
    }
    cudaError_t ensure(size_t count) { return count <= n && p ? cudaSuccess : alloc(count + count / 8); }
    void release() {
        if (p && own) cudaFree(p);
        p = nullptr;
        n = 0;
        own = true;
    }
    void view(T* q, size_t count) {
        release();
        p = q;
        n = count;
        own = false;
    }
    void swap(DBuf& o) {
        std::swap(p, o.p);
        std::swap(n, o.n);
        std::swap(own, o.own);
    }
};

// Several arrays in one device allocation: an allocation and its release take
// 65 us here whatever its size up to some 100 MB, and a context holds some
// sixty arrays.  take() is called in two passes over the same arrays: a first
// one that measures, then, after reserve(), one that hands the parts out.  The
// arrays live as long as the slab and swap their parts among themselves only.
struct Slab {
    struct Part {
        void* buf;
        void (*drop)(void*);
    };
    DBuf<uint8_t> mem;
    size_t off = 0;
    bool measuring = true;
    std::vector<Part> parts;  // the arrays that hold a part of mem
    void measure() {
        off = 0;
        measuring = true;
    }
    // Takes back every part handed out, then keeps a block that is large enough
    // or replaces it.
    cudaError_t reserve() {
        for (const Part& q : parts) q.drop(q.buf);
        parts.clear();
        cudaError_t e = off <= mem.n ? cudaSuccess : mem.alloc(off);
        off = 0;
        measuring = false;
        return e;
    }
    template <class T>
    void take(DBuf<T>& b, size_t count) {
        count = std::max<size_t>(count, 1);
        off = (off + 255) / 256 * 256;
        if (!measuring) {
            b.view(reinterpret_cast<T*>(mem.p + off), count);
            parts.push_back({&b, [](void* q) {
                                 DBuf<T>& d = *static_cast<DBuf<T>*>(q);
                                 if (!d.own) d.release();  // not one allocated anew since
                             }});
        }
        off += sizeof(T) * count;
    }
};

// cell-list buffers (per-sphere cell, per-cell counts, starts, fill cursors
// and the spheres in cell order)
struct CellBufs {
    Slab slab;
    DBuf<int> of, count, start, fill, order;
    cudaError_t ensure(size_t np, size_t ncell) {
        if (of.n >= np && fill.n >= ncell && of.p) return cudaSuccess;
        auto parts = [&] {
            slab.take(of, np);
            slab.take(order, np);
            slab.take(count, ncell + 1);
            slab.take(start, ncell + 1);
            slab.take(fill, ncell);
        };
        slab.measure();
        parts();
        cudaError_t e = slab.reserve();
        if (e == cudaSuccess) parts();
        return e;
    }
};

// scratch of the node conversions: `cap` conversions per step, queued by step
// parity, each with q x q gathered populations
template <class Rec>
struct ConversionBufs {
    DBuf<Rec> rec;
    DBuf<float> scratch;
    DBuf<uint8_t> valid;
    uint32_t cap = 0;  // 0 until all three are there
    cudaError_t ensure(uint32_t want, size_t q) {
        if (want == cap) return cudaSuccess;
        cap = 0;
        cudaError_t e = rec.alloc(2 * (size_t)want);
        if (e == cudaSuccess) e = scratch.alloc(want * q * q);
        if (e == cudaSuccess) e = valid.alloc(want * q);
        if (e == cudaSuccess) cap = want;
        return e;
    }
};

}  // namespace lbmdem
