// Which of a caller's host buffers a kernel may store into (plain C++: no CUDA header).
#pragma once
#include <cstddef>
#include <cstdint>

// FP64 values at this address can be stored one by one (a copy takes any address)
inline bool doubles_aligned(uintptr_t at) { return at % sizeof(double) == 0; }
