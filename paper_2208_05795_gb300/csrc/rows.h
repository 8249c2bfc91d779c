// rows.h -- rows of a device buffer to the host (host code).
#pragma once
#include <cstddef>

namespace tsx {

// A 2-D copy takes a pitch up to the device's limit, 2^31 - 1 bytes; a list's pitch is four bytes a
// record it has room for, so from 2^29 records on its rows go one by one.  The line is
// at half the limit: beside the transfer of such rows a few calls more cost nothing.
constexpr size_t kMaxRowPitch = size_t(1) << 30;

// rows of width bytes, pitch bytes apart at src, to dst, one after the other.  copy2d(dst, dst pitch, src, src
// pitch, width, rows) and copy(dst, src, bytes) return 0 or an error, which is returned.
template <class Copy2d, class Copy>
int copy_rows(void *dst, const void *src, size_t pitch, size_t width, size_t rows, Copy2d copy2d, Copy copy) {
    if (pitch <= kMaxRowPitch) return copy2d(dst, width, src, pitch, width, rows);
    for (size_t r = 0; r < rows; r++) {
        const int e = copy((char *)dst + r * width, (const char *)src + r * pitch, width);
        if (e) return e;
    }
    return 0;
}

}  // namespace tsx
