// state_source.h -- where a state array passed as a device pointer lies, and
// whether the state set-up kernel may read it there.  Plain C++.
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace mfc5 {

// What the driver says of an address.  Zeros: it knows nothing of it.
struct PointerInfo {
    bool device_memory;   // allocated on a device, not managed
    int device;           // that device
    uintptr_t range;      // the allocation (or reservation) the address lies in
    size_t range_bytes;
    uintptr_t map;        // the mapping behind it, where the driver reports one
    size_t map_bytes;
};

inline bool covers(uintptr_t base, size_t size, uintptr_t addr, size_t bytes) {
    return addr >= base && addr - base <= size && bytes <= size - (addr - base);
}

// The kernel dereferences the address on `device` as doubles, so it takes only
// memory of that device, aligned, and known to hold the whole array.  Anything
// else -- another device's memory, host or managed memory, an array longer than
// its allocation, a misaligned one -- goes through cudaMemcpyAsync first, which
// copies it or refuses it with an error.
inline bool read_in_place(const PointerInfo& p, uintptr_t addr, size_t bytes, int device) {
    return p.device_memory && p.device == device && addr % sizeof(double) == 0 &&
           covers(p.range, p.range_bytes, addr, bytes) &&
           (p.map_bytes == 0 || covers(p.map, p.map_bytes, addr, bytes));
}

}  // namespace mfc5
