// Device scratch that grows with the number of densities. Host code without
// CUDA calls of its own, so that a failing allocation can be tested on a CPU.
#pragma once
#include <cstddef>

// One region per molecule in one buffer; `unit` is the number of elements that
// one density takes in the regions before it. Offsets follow from what the
// buffer holds, so a growth that failed leaves an empty buffer and no offset
// into another one.
template <class T> struct JkPerMol {
    T *base = nullptr;
    size_t ndm = 0;   // densities per molecule it holds

    T *at(size_t unit) const { return base + ndm * unit; }
    // room for n densities of `total` elements each (contents are not kept);
    // alloc(bytes, &p) and its error code, 0 for success
    template <class Alloc, class Free> int grow(size_t n, size_t total, Alloc alloc, Free release)
    {
        if (ndm >= n) return 0;
        release(base);
        base = nullptr;
        ndm = 0;
        void *p = nullptr;
        const size_t elems = n * total;
        if (int e = alloc(sizeof(T) * (elems ? elems : 1), &p)) return e;
        base = static_cast<T *>(p);
        ndm = n;
        return 0;
    }
};
