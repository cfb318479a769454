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

// The length of the adjoint's segments between checkpoints, longer than the caller's K
// where that can be had: the largest of ceil(H / 1), ceil(H / 2), ... above K whose
// scratch of need(k) floats is within the budget and is held already or can be
// reserved (0: none, or `failed`). A size that could not be reserved is written to
// `refused` and neither it nor a larger one is asked for again while the caller
// keeps `refused`: a repeated call then neither looks at the device's free memory nor
// allocates.
enum class Reserve { kDone, kNoMemory, kFailed };
template <typename Need, typename Try>
int longer_segment(int H, int K, size_t budget, const size_t &held, size_t &refused, bool &failed, Need need, Try reserve) {
    failed = false;
    for (int segs = 1, k = H; k > K; ++segs, k = (H + segs - 1) / segs) {
        const size_t f = need(k);
        if (f > budget) continue;
        if (f <= held) return k;
        if (f >= refused) continue;
        const Reserve r = reserve(f);
        if (r == Reserve::kDone) return k;
        if (r == Reserve::kFailed) {
            failed = true;
            return 0;
        }
        refused = f;
    }
    return 0;
}

}  // namespace ih
