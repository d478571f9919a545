// Page-locked host ranges as a kernel may address them. Host arithmetic only: the lookup of one
// address is the caller's, so that this part is checked without a GPU.
#pragma once
#include <cstddef>

namespace cp {

// What a host address belongs to: one page-locked allocation or registration.
struct PinnedSpan {
    char *device;  // the address as the device sees it
    size_t left;   // bytes from it to the end of that allocation or registration
};

// Device-side address of the host range [p, p + bytes), or nullptr unless every byte of it is page-locked
// and its device addresses are consecutive. The range may run through several registrations that
// follow one another (a large buffer registered in pieces). Looking at both ends is not enough: two
// registrations with a pageable hole between them look the same there, because a host address and
// its device address are mostly equal.
// span_at(q, span): fills the span of host address q; false if q is not page-locked.
template <class SpanAt>
void *pinned_view(void *p, size_t bytes, SpanAt span_at) {
    char *const host = static_cast<char *>(p);
    char *device = nullptr;
    for (size_t done = 0; done < bytes;) {
        PinnedSpan s;
        if (!span_at(host + done, s) || !s.device || s.left == 0) return nullptr;
        if (done == 0) device = s.device;
        else if (s.device != device + done) return nullptr;
        done += s.left < bytes - done ? s.left : bytes - done;
    }
    return device;
}

}  // namespace cp
