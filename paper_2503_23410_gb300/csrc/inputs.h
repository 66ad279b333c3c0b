// inputs.h -- when the scene build reads a device input where it lies instead of
// copying it first (plain C++: compiled into the library and by the tests).
#pragma once

#include <cstddef>
#include <cstdint>

namespace vafr {

// `bytes` bytes of floats at address `at`, which the driver says lie in an
// allocation of `size` bytes at `base`.  A kernel may read them in place when they
// are on the device it runs on, whole floats, and all inside that allocation.
// Whatever else the caller passes goes through a copy: it fetches another
// device's memory and float data between two floats' addresses, and refuses a
// range that is not the caller's, which a kernel would fault on.
inline bool readable_in_place(bool on_this_device, uintptr_t at, size_t bytes, uintptr_t base, size_t size) {
    return on_this_device && at % sizeof(float) == 0 && at >= base && at - base <= size && bytes <= size - (at - base);
}

}  // namespace vafr
