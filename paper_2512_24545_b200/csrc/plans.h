// Decisions of the host side that need no GPU, in plain C++ so that they can be checked on the CPU.
#pragma once

#include <cstddef>
#include <cstdint>

namespace mdbf {

// What the driver says about a host address: whether it lies in pinned memory, the device's address of it, and the one mapping
// (allocation or registration) it belongs to.
struct HostRange {
    bool pinned;
    uint64_t device, start;
    size_t size;
};
// The device's address of `bytes` bytes of host memory from there on, or 0 where not all of them lie in that mapping (a registered part
// of a larger array, say): what is behind it is not the device's to touch.
inline uint64_t host_view(const HostRange &r, size_t bytes) {
    if (!r.pinned || r.device == 0 || r.device < r.start) return 0;
    const uint64_t off = r.device - r.start;
    return off <= r.size && bytes <= r.size - off ? r.device : 0;
}
// Whether a kernel may store y (bytes of `es`-byte elements, T tokens) at this device address of host memory itself: whole elements on
// their own boundary (a copy takes any address, so a slice of a byte arena is a valid y_host), and at most as many tokens as the kernels
// with plain stores take - beyond that y leaves through a tensor map, and those are made over device memory only.
constexpr int kHostStoreMaxT = 64;
inline bool host_store_direct(uint64_t device, size_t es, int T) { return device != 0 && device % es == 0 && T <= kHostStoreMaxT; }

// CTAs of the cooperative orthogonalisation of n rows in chunks of `chunk`: at most `most`, and one per SM, so that all of them run at once
// on any device (a cooperative launch with more than that is refused).
inline int orth_ctas(int n, int chunk, int most, int sms) {
    const int chunks = (n + chunk - 1) / chunk, limit = sms < most ? sms : most;
    return chunks < limit ? chunks : limit;
}

}  // namespace mdbf
