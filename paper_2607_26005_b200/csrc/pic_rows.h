// Which grid rows a view's footprint crosses, and when a walk over them ends (internal; device code, and host code that checks it).
#pragma once
#include <math.h>

#ifdef __CUDACC__
#define PIC_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define PIC_HOST_DEVICE inline
#endif

namespace pic {

constexpr int ROW_PASS = 32;     // rows looked at together, a lane each

// The rows from floor f0 to floor f1 of a grid of ny rows, both cut to the grid: lo in [0, ny], hi in [-1, ny - 1], hi < lo
// if none is crossed.  A pose may be any finite number, so f0 and f1 may be far outside the integers (or NaN, for poses whose
// differences overflow: then all rows); cut like this, lo + lane and hi - lo cannot overflow.
PIC_HOST_DEVICE void clamp_rows(float f0, float f1, unsigned ny, int& lo, int& hi) {
    lo = (int)fminf(fmaxf(f0, 0.f), (float)ny);
    hi = (int)fmaxf(fminf(f1, (float)ny - 1.f), -1.f);
}

// Are there rows after the pass that begins at row r0?
PIC_HOST_DEVICE bool rows_after(int r0, int hi) { return hi - r0 >= ROW_PASS; }

}  // namespace pic
