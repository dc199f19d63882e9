// Which host frames a tick may work on in place. (Plain C++: what the driver
// knows of an address comes in as a function.)
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace gmmlib {

// The page-locked bytes around an address that the device reaches at the same
// addresses: one allocation or registration. None: lo == hi.
struct HostSpan {
    uintptr_t lo, hi;
};

// Whether every byte of [q, q + bytes) is such memory. span_of(q): the span
// that holds q. Each byte counts, not the two ends: ordinary memory may lie
// between two registrations.
template <class SpanOf> bool all_page_locked(uintptr_t q, size_t bytes, SpanOf span_of) {
    const uintptr_t end = q + bytes;
    while (q < end) {
        const HostSpan s = span_of(q);
        if (s.lo > q || s.hi <= q)
            return false;
        q = s.hi;
    }
    return true;
}

// Whether a tick may read a frame of `pixels` pixels from r and d, and write
// the mask to m, in place: all of it page-locked, aligned as the kernels need
// it, the mask apart from the frame, and the direct kernel's to tick (the
// staged one's frames are uploaded: its stages wait for bulk copies of whole
// tiles of a frame, and that over the host link was not measured).
template <class SpanOf>
bool frame_in_place(bool staged, uintptr_t r, uintptr_t d, uintptr_t m, size_t pixels,
                    size_t mask_bytes, SpanOf span_of) {
    if (staged || d % 2 || m % 4)
        return false;
    const uintptr_t r1 = r + 3 * pixels, d1 = d + 2 * pixels, m1 = m + mask_bytes;
    if ((r < m1 && m < r1) || (d < m1 && m < d1))
        return false;
    return all_page_locked(r, 3 * pixels, span_of) && all_page_locked(d, 2 * pixels, span_of) &&
           all_page_locked(m, mask_bytes, span_of);
}

} // namespace gmmlib
