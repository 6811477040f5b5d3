// localmax.cuh -- the strict 26-neighbour maxima of a map (Sec. 3.4), used by
// Find Peaks and by block processing.
#pragma once

#include "ttm_internal.h"

namespace ttm {

// Candidates at z in [cz0, cz1) and y, x in the box, neighbours within
// z in [nz0, nz1) and the same y, x box, of a map with rows of X and planes
// of Y rows; indices are written as ((z + zoff) Yt + y) Xt + x.
struct LmGeom {
    int Y, X;
    int cz0, cz1, nz0, nz1, y0, y1, x0, x1;
    int64_t zoff;
    int Yt, Xt;
    int zchunk;  // planes per warp (set by localmax_run)
};

// appends the maxima (ties go to the lower linear index; NaN is never a
// peak and never beats one) to idx / val, at most cap of them, counting all
// of them in *count
void localmax_run(int num_sms, const float* d_map, LmGeom g, int64_t cap, int64_t* idx, float* val,
                  unsigned long long* count, cudaStream_t st);

}  // namespace ttm
