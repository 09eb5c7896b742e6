// rism_grow.h -- buffers that only grow, with the capacity they share.
//
// Pointers and capacity change together.  A group that is too small gives back its memory and has capacity 0 until every
// one of its allocations has succeeded: after a failure the next call, however small its need, allocates again instead of
// passing the capacity test over null pointers.  No CUDA here: the allocator is a parameter (DeviceMem of
// rism_internal.cuh), and a host test gives one that fails.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace rism {

// One buffer of a group: the pointer and the elements it needs.
template <typename T>
struct Buf {
    T*& p;
    size_t count;
};
template <typename T>
Buf<T> buf(T*& p, int64_t count) {
    return Buf<T>{p, (size_t)(count > 0 ? count : 1)};
}

// Makes the group hold `need` (at least 1) of whatever its capacity counts.  Mem::alloc(void**, bytes) returns 0 or an
// error, Mem::release(void*) takes null.
template <typename Mem, typename Cap, typename... T>
auto grow_with(Cap& cap, int64_t need, Buf<T>... b) {
    decltype(Mem::alloc(nullptr, size_t{})) e{};
    if (need < 1) need = 1;
    if (need <= (int64_t)cap) return e;
    cap = 0;
    ((Mem::release(b.p), b.p = nullptr), ...);
    auto one = [&](auto& x) {
        void* v = nullptr;
        e = Mem::alloc(&v, x.count * sizeof(*x.p));
        if (e == decltype(e){}) x.p = static_cast<decltype(+x.p)>(v);
        return e == decltype(e){};
    };
    if ((one(b) && ...)) cap = (Cap)need;
    return e;
}

}  // namespace rism
