// smem_seen.h -- which amount of dynamic shared memory each kernel may take,
// per device.  Host only, no CUDA calls.
#pragma once

#include <atomic>
#include <cstddef>
#include <mutex>

namespace vx {

constexpr int kMaxDevices = 64;

// One kernel's table.  allowed[] only grows and is what the kernel's attribute
// was last set to: under `growing` from the second look to the store, since
// the attribute is a value that a smaller one set later would lower.
struct SmemSeen {
    std::atomic<size_t> allowed[kMaxDevices] = {};
    std::mutex growing;
};

// Makes `bytes` allowed on device `dev`: set(bytes), a call that costs as much
// as a launch, is made when the device first needs that much.  Returns what
// set returned, or a value-initialised result.
template <class Set>
auto grow_allowed(SmemSeen &seen, int dev, size_t bytes, Set set) -> decltype(set(bytes))
{
    decltype(set(bytes)) ok{};
    const bool known = dev >= 0 && dev < kMaxDevices;
    if (known && seen.allowed[dev].load(std::memory_order_acquire) >= bytes) return ok;
    std::lock_guard<std::mutex> lk(seen.growing);
    if (known && seen.allowed[dev].load(std::memory_order_relaxed) >= bytes) return ok;
    const auto e = set(bytes);
    if (e == ok && known) seen.allowed[dev].store(bytes, std::memory_order_release);
    return e;
}

}  // namespace vx
