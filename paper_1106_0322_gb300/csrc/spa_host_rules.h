// spa_host_rules.h -- host-side decisions of the entry points as plain C++ (no CUDA headers), so that
// they can be compiled and checked where there is no GPU.
#pragma once

#include <cstddef>
#include <cstdint>

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

}  // namespace spa
