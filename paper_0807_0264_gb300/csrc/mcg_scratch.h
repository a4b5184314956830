// Named, grow-only buffers, kept between calls until clear(): the library's scratch
// on a device or in pinned host memory.  Mem gives the memory: static int
// alloc(void**, size_t) (0 or an error), free(void*), sync() (waits for everything
// that may use a buffer) and available() (free bytes).
//
// Required buffers are what a call cannot do without.  Optional ones buy speed: a
// request takes at most a quarter of the free memory, and all of them give way
// when a required buffer (or, through clear(), the caller) needs theirs.  A
// pointer from get_optional holds until the next get().
#pragma once

#include <algorithm>
#include <cstddef>
#include <map>
#include <string>

namespace mcg {

template <class Mem>
class ScratchCache {
    struct Buf {
        void* p = nullptr;
        size_t bytes = 0;
        bool optional = false;
    };
    std::map<std::string, Buf> bufs;

    static void drop(Buf& b) {
        if (b.p) {
            Mem::sync();
            Mem::free(b.p);
        }
        b.p = nullptr;
        b.bytes = 0;
    }

public:
    // null and *err set when there is no memory
    void* get(const char* name, size_t bytes, int* err) {
        Buf& b = bufs[name];
        b.optional = false;
        if (b.bytes >= bytes && b.p) return b.p;
        drop(b);
        bytes = std::max<size_t>(bytes, 256);
        *err = Mem::alloc(&b.p, bytes);
        if (*err && drop_optional()) *err = Mem::alloc(&b.p, bytes);
        if (*err) {
            b.p = nullptr;
            return nullptr;
        }
        b.bytes = bytes;
        return b.p;
    }

    // null when it would take more than its share or there is no memory (the old
    // buffer, if any, is kept)
    void* get_optional(const char* name, size_t bytes) {
        Buf& b = bufs[name];
        if (b.bytes >= bytes && b.p) return b.p;
        if (bytes > Mem::available() / 4) return nullptr;
        void* p = nullptr;
        bytes = std::max<size_t>(bytes, 256);
        if (Mem::alloc(&p, bytes)) return nullptr;
        drop(b);
        b.p = p;
        b.bytes = bytes;
        b.optional = true;
        return p;
    }

    // bytes that get_optional(name) would give
    size_t optional_room(const char* name) {
        const auto it = bufs.find(name);
        return std::max(it == bufs.end() ? 0 : it->second.bytes, Mem::available() / 4);
    }

    // frees the optional buffers; whether there were any
    bool drop_optional() {
        bool any = false;
        for (auto& kv : bufs)
            if (kv.second.optional && kv.second.p) {
                drop(kv.second);
                any = true;
            }
        return any;
    }

    void clear() {
        for (auto& kv : bufs) drop(kv.second);
        bufs.clear();
    }
};

}  // namespace mcg
