// spa_host_rules.h -- host-side decisions of the entry points as plain C++ (no CUDA headers), so that
// they can be compiled and checked where there is no GPU.
#pragma once

#include <cstddef>
#include <cstdint>
#include <mutex>
#include <vector>

namespace spa {

// What the driver knows of the allocation that a pointer lies in.
struct MemoryFacts {
    bool device = false;  // device memory (not managed, not host)
    int ordinal = -1;     // the device it belongs to
    uintptr_t begin = 0;  // the allocation's range
    size_t bytes = 0;
};

// Whether the likelihood entry points may read the caller's device particles [N][p] at `b` where they
// lie: they are in one allocation of the context's device, which holds all of them; rows read 16 bytes
// at a time are aligned; and nothing that the call writes ([out, out + out_bytes)) overlaps them.
// Everything else is left to the copy, which takes memory of another device, managed and host memory,
// and answers a pointer that it does not know with an error.
inline bool particles_in_place(const MemoryFacts& m, int ctx_device, uintptr_t b, int64_t N, int64_t p, uintptr_t out,
                               size_t out_bytes)
{
    const size_t bytes = sizeof(float) * (size_t)N * (size_t)p;
    if (!m.device || m.ordinal != ctx_device) return false;
    if (b < m.begin || bytes > m.bytes || b - m.begin > m.bytes - bytes) return false;
    if ((b & 3u) != 0 || ((p & 3) == 0 && (b & 15u) != 0)) return false;
    return out == 0 || out + out_bytes <= b || b + bytes <= out;
}

// Whether work may still run on a context's own stream, which a call on another stream has to wait for
// because both use the context's buffers. Busy from the moment the stream is handed out to be worked
// on, whatever becomes of the call, until the host has waited for that very stream.
struct OwnStream {
    const void* handle = nullptr;
    bool busy = true;
    void handed_out(const void* stream)
    {
        if (stream == handle) busy = true;
    }
    void waited_for(const void* stream)
    {
        if (stream == handle) busy = false;
    }
    bool holds_up(const void* stream) const { return busy && stream != handle; }
};

// Words of page-locked host memory for the contexts of a process, 64 to a page of 4 KB, a cache line
// each. A page of its own costs a context 125 us when it is made and 175 when it is destroyed (n = 200,
// p = 10: 192 and 96 us without). A page belongs to one CUDA context, given by its unique ID, and is
// never used by another: a device reset ends the CUDA context and the page with it. A page whose last
// word comes back is freed, except the only one of its CUDA context. Any thread may call.
class PinnedWords {
public:
    static constexpr size_t LINE = 64, WORDS = 64, PAGE = LINE * WORDS;
    // alloc(PAGE) returns page-locked memory of the current CUDA context, `owner`, or nullptr.
    template <typename Alloc>
    uint32_t* take(unsigned long long owner, Alloc alloc)
    {
        std::lock_guard<std::mutex> lock(mu_);
        for (Page& g : pages_)
            if (g.owner == owner && ~g.used != 0)
                for (size_t k = 0; k < WORDS; ++k)
                    if (!(g.used >> k & 1u)) {
                        g.used |= (uint64_t)1 << k;
                        return reinterpret_cast<uint32_t*>(g.base + LINE * k);
                    }
        char* base = static_cast<char*>(alloc(PAGE));
        if (!base) return nullptr;
        pages_.push_back(Page{owner, base, 1});
        return reinterpret_cast<uint32_t*>(base);
    }
    // free(page) is called for a page to be given back, and only if `owner` is `current`, the CUDA context
    // of the calling thread.
    template <typename Free>
    void give(uint32_t* word, unsigned long long owner, unsigned long long current, Free free)
    {
        std::lock_guard<std::mutex> lock(mu_);
        char* w = reinterpret_cast<char*>(word);
        size_t same = 0;
        for (const Page& g : pages_) same += g.owner == owner;
        for (size_t q = 0; q < pages_.size(); ++q) {
            Page& g = pages_[q];
            if (g.owner != owner || w < g.base || w >= g.base + PAGE) continue;
            g.used &= ~((uint64_t)1 << ((size_t)(w - g.base) / LINE));
            if (g.used == 0 && same > 1 && owner == current) {
                free(g.base);
                pages_.erase(pages_.begin() + (ptrdiff_t)q);
            }
            return;
        }
    }
    size_t pages()
    {
        std::lock_guard<std::mutex> lock(mu_);
        return pages_.size();
    }

private:
    struct Page {
        unsigned long long owner;
        char* base;
        uint64_t used;  // bit k: word k is taken
    };
    std::mutex mu_;
    std::vector<Page> pages_;
};

}  // namespace spa
