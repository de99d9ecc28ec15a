// How a caller's array of sphere values is reached: host code without CUDA
// headers, so that the rule can be tried for memory no test machine has.
#pragma once

#include <cstdint>

namespace lbm {

enum class Mem { pageable, pinned, device, managed };

// An array of a call: what kind of memory it lies in, whether that is of the
// handle's device (pinned memory: allocated beside it), and its address for
// kernels.
struct ArrayAt {
    Mem mem;
    bool here;
    std::uintptr_t at;
};

// kernel: a kernel reads or writes it in place; staged: through the handle's
// pinned memory; copy: by a copy of its own.
enum class Route { kernel, staged, copy };

// A kernel takes whole doubles of its own device's memory only: an array of
// another device, or host memory in a call that says device memory (a mixed
// set of arrays), is the copy's business, which knows where both ends lie.
inline Route route_device(const ArrayAt &a) {
    return a.mem == Mem::device && a.here && a.at % 8 == 0 ? Route::kernel : Route::copy;
}

// Outputs of a call that says host memory, `have_stage`: its values fit the
// handle's pinned memory.  Pinned arrays are written in place; device memory
// among them cannot be filled by the host.
inline Route route_host(const ArrayAt &a, bool have_stage) {
    if (a.mem == Mem::pinned && a.here && a.at && a.at % 8 == 0) return Route::kernel;
    return a.mem != Mem::device && have_stage ? Route::staged : Route::copy;
}

}  // namespace lbm
