// Which of a caller's host buffers a kernel may store into (plain C++: no CUDA header).
#pragma once
#include <cstddef>
#include <cstdint>

// FP64 values at this address can be stored one by one (a copy takes any address)
inline bool doubles_aligned(uintptr_t at) { return at % sizeof(double) == 0; }

// one allocation or registration, size bytes from start on, holds all of the buffer (two
// registrations at its ends may have pageable memory between them)
inline bool allocation_holds(uintptr_t start, size_t size, uintptr_t at, size_t bytes) {
    return at >= start && at - start <= size && bytes <= size - (at - start);
}
