// Elementwise passes over the cells of a grid between its padded layout and dense arrays: a flat numbering of 16-byte groups.
#pragma once

#include <initializer_list>
#include <type_traits>

#include "hg_internal.cuh"

namespace hg {

// Flat numbering of the groups of W consecutive cells of a row (row j, plane k): all threads busy whatever nx is, and
// neighbouring threads on neighbouring groups.  W is 16 bytes of the dense array where its rows allow such accesses
// (dense_width), else 1 (coalesced single elements: groups of 4 with element stores touch every sector four times).
// I is 32 bits wide unless the grid needs more.
template <typename I>
struct Group {
    int i0, j, k;
    long long dense;  // index of its first cell in a dense array
};
template <int W, typename I>
__device__ __forceinline__ Group<I> group_of(const Layout& L, I t, unsigned gpr) {
    const I row = t / gpr;
    Group<I> g;
    g.i0 = (int)(t - row * gpr) * W;
    const I k = row / (unsigned)L.ny;
    g.j = (int)(row - k * (unsigned)L.ny);
    g.k = (int)k;
    g.dense = (long long)row * L.nx + g.i0;
    return g;
}
template <int W, typename I, class F>
__device__ __forceinline__ void for_groups(const Layout& L, F&& f) {
    const unsigned gpr = (unsigned)(L.nx / W);  // W divides nx
    const I total = (I)gpr * (unsigned)L.ny * (unsigned)L.nz;
    for (I t = blockIdx.x * (I)blockDim.x + threadIdx.x; t < total; t += (I)gridDim.x * blockDim.x)
        f(group_of<W, I>(L, t, gpr));
}

template <typename T, int W>
struct alignas(sizeof(T) * W <= 16 ? sizeof(T) * W : 16) Vec {
    T v[W];
};
template <typename T, int W>
__device__ __forceinline__ Vec<T, W> ldv(const T* p) {
    return *reinterpret_cast<const Vec<T, W>*>(p);
}
template <typename T, int W>
__device__ __forceinline__ void stv(T* p, const Vec<T, W>& x) {
    *reinterpret_cast<Vec<T, W>*>(p) = x;
}

// elements per 16-byte word of a dense array of type T if its rows hold whole words on 16-byte boundaries, else 1
template <typename T>
int dense_width(const Layout& L, std::initializer_list<const void*> ptrs) {
    constexpr int W = 16 / sizeof(T);
    uintptr_t bits = 0;
    for (const void* p : ptrs) bits |= (uintptr_t)p;
    return L.nx % W == 0 && bits % 16 == 0 ? W : 1;
}
// groups of `w` cells are numbered in 32 bits (with room for the grid stride's overshoot)
inline bool fits32(const Layout& L) { return (long long)L.nx * L.ny * L.nz < (1LL << 31); }
inline unsigned group_blocks(const Layout& L, int w) {
    const long long n = ((long long)L.nx * L.ny * L.nz / w + 256 - 1) / 256;
    return (unsigned)(n < (1LL << 22) ? n : 1LL << 22);
}
// call f with the group width (1 or the word's elements) and the index type as compile-time values
template <typename T, class F>
void dispatch_groups(const Layout& L, int w, F&& f) {
    constexpr int W = 16 / sizeof(T);
    using One = std::integral_constant<int, 1>;
    using Word = std::integral_constant<int, W>;
    if (fits32(L)) {
        if (w == W) f(Word(), 0u);
        else f(One(), 0u);
    } else {
        if (w == W) f(Word(), 0ull);
        else f(One(), 0ull);
    }
}

}  // namespace hg
