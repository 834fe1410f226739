// Indices of a packed lower triangle (row-major, diagonal included).  No CUDA header is needed: the host checks it alone.
#pragma once

#include <math.h>

namespace infft {

__host__ __device__ __forceinline__ long long tri(long long r, long long c) { return r * (r + 1) / 2 + c; }

// (row, column) of entry e of a packed lower triangle (e = r (r + 1) / 2 + c, c <= r): a
// float estimate of the row, corrected by integer steps (in 32 bits where the index allows; unsigned, since
// (r + 1) (r + 2) passes 2^31 from e = 1,073,720,970 on)
__host__ __device__ __forceinline__ void tri_rc(long long e, long long* r_out, long long* c_out) {
    if (e < (1 << 30)) {
        const unsigned e32 = (unsigned)e;
        unsigned r = (unsigned)((sqrtf(8.f * (float)e32 + 1.f) - 1.f) * 0.5f);
        while (r * (r + 1) / 2 > e32) --r;
        while ((r + 1) * (r + 2) / 2 <= e32) ++r;
        *r_out = r;
        *c_out = e32 - r * (r + 1) / 2;
        return;
    }
    long long r = (long long)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    while (r * (r + 1) / 2 > e) --r;
    while ((r + 1) * (r + 2) / 2 <= e) ++r;
    *r_out = r;
    *c_out = e - r * (r + 1) / 2;
}

}  // namespace infft
