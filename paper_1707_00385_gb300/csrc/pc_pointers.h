// pc_pointers.h -- the device-pointer checks of one call (host code only).
#pragma once
#include <cstddef>
#include <cstdint>

namespace pcurv {

// The device pointers of one call.  A pointer inside an allocation that holds
// another pointer of the call needs no query of its own: a batch of frames cut
// from a few allocations asks the driver a few times instead of four times a
// frame.  An allocation counts when its last byte is a device pointer too.
// Nothing is kept from one call for the next.
//
// Driver::is_device(p): whether p is device memory.  Driver::range(p, &base,
// &size): the allocation that holds p, false when it is not known.  (The driver
// gives the one mapping around p where an address reservation is mapped in
// parts, so a hole between two mappings is in neither range.)
template <typename Driver>
class DevicePointers {
  public:
    bool operator()(const void* p) {
        const uintptr_t a = (uintptr_t)p;
        for (int i = 0; i < used_; i++)
            if (a >= lo_[i] && a < hi_[i]) return true;
        if (!Driver::is_device(p)) return false;
        uintptr_t base = 0;
        size_t size = 0;
        if (Driver::range(p, &base, &size) && size > 0 && a >= base && a - base < size &&
            Driver::is_device((const void*)(base + size - 1))) {
            const int i = used_ < MAX ? used_++ : next_++ % MAX;
            lo_[i] = base;
            hi_[i] = base + size;
        }
        return true;
    }

  private:
    static constexpr int MAX = 8;
    uintptr_t lo_[MAX], hi_[MAX];
    int used_ = 0, next_ = 0;
};

}  // namespace pcurv
