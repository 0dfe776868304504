// Length of a launch of marching tile blocks, in plane-times of one block.
#pragma once

#include <algorithm>

namespace kin {

// cols blocks per z chunk of zc planes, issued chunk by chunk (the grid's z
// index varies slowest), each to the slot that frees first, occupying it for its
// planes plus `prologue`.  All chunks but the last are equal, so whole waves are
// counted and only the last chunk's blocks are placed, on the slots of the last
// incomplete wave that are free earlier.
inline double tile_schedule(long long cols, int N, int zc, long long slots, double prologue) {
    const int full = N / zc, rest = N - full * zc;
    const double a = zc + prologue, b = rest + prologue;
    const long long late = cols * full % slots;  // slots one wave ahead of the others
    double early_at = (double)(cols * full / slots) * a, late_at = early_at + a;
    double end = late > 0 ? late_at : early_at;
    for (long long left = rest > 0 ? cols : 0; left > 0;) {
        if (late == 0 || early_at <= late_at) {
            left -= slots - late;
            early_at += b;
            end = std::max(end, early_at);
        } else {
            left -= late;
            late_at += b;
            end = std::max(end, late_at);
        }
    }
    return end;
}

}  // namespace kin
