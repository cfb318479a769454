// host_rules.cuh -- decisions of the C ABI's host side that are taken on plain
// values, apart from the CUDA calls that supply them (plain C++, so that a host
// compiler can run them too).
#pragma once
#include <cstddef>
#include <cstdint>

namespace ih {

// What is known about an array that a caller passed.
struct CallerArray {
    enum Kind { kOther, kDevice, kManaged };   // host memory, registered or not, is kOther
    Kind kind = kOther;
    int device = -1;          // where kDevice memory lives
    uintptr_t at = 0;         // the array
    size_t bytes = 0;
    uintptr_t base = 0;       // the allocation that holds it (size 0: not known)
    size_t size = 0;
};

// Whether a kernel launched on a stream of launch_device, with current_device
// current, may touch the array: a handle's own memory is on handle_device, so the
// launch has to be there (a copy call takes any current device and any stream), and
// the array has to lie inside one allocation (a copy call refuses an array that
// ends past its allocation; a kernel would fault on it).
inline bool kernel_may_touch(const CallerArray &a, int handle_device, int current_device, int launch_device) {
    if (current_device != handle_device || launch_device != handle_device) return false;
    if (a.kind == CallerArray::kOther || (a.kind == CallerArray::kDevice && a.device != handle_device)) return false;
    return a.at >= a.base && a.bytes <= a.size && a.at - a.base <= a.size - a.bytes;
}

}  // namespace ih
