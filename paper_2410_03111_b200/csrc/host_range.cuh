// Whether kernels may access a host buffer directly.  Plain C++, so that the decision can be tested without a GPU.
#pragma once

#include <stdint.h>

// What the driver knows about the first byte of a buffer (cuPointerGetAttributes).
struct LorcHostRange {
    unsigned type;          // CU_MEMORYTYPE_*; 0: memory the driver does not know (pageable)
    unsigned managed;
    uint64_t device;        // the byte's device address; 0: not mapped
    uint64_t start, size;   // the allocation or registration that holds the byte (device addresses)
};

// Device address of the buffer of `bytes` bytes whose first byte `r` describes, or 0 unless it is pinned and mapped host
// memory, 16-byte aligned, and lies inside ONE allocation or registration.  (Looking at its two ends is not enough: under
// unified addressing they are `bytes - 1` apart also where the memory between two registrations is pageable.)
inline uint64_t lorc_mapped_address(const LorcHostRange& r, uint64_t host, uint64_t bytes) {
    if (r.type != 1 /* CU_MEMORYTYPE_HOST */ || r.managed || !r.device || (host & 15) || (r.device & 15)) return 0;
    if (r.device < r.start || bytes > r.size || r.device - r.start > r.size - bytes) return 0;
    return r.device;
}
