// May a kernel write a caller's host buffer?  The decision alone, without CUDA: hbf_api.cu asks the driver for the facts.
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace hbf {

// what the driver knows of an address: kind of memory (1: host), the device's address of it (0: none), the allocation or
// registration it lies in, and what the device may do there (bit 0: read, bit 1: write)
struct HostMemory { uint32_t type; uint64_t device, start; size_t size; uint64_t access; };

// Every byte has to lie in one range that the device may write, at the address the host uses, and 8-byte stores have to be
// aligned: a buffer of which only a part is registered, or registered for reading, is left to the runtime's copies.
inline bool device_may_write(const HostMemory &m, const void *at, size_t bytes) {
    const uint64_t p = (uint64_t)(uintptr_t)at;
    return m.type == 1u && m.device == p && (p & 7u) == 0u && (m.access & 2u) != 0u && p >= m.start && p - m.start <= m.size && bytes <= m.size - (p - m.start);
}

}  // namespace hbf
