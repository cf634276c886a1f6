// boundary.h -- where a ghost cell outside the domain takes its values from.
#pragma once

#ifdef __CUDACC__
#define TSU_HD __host__ __device__ __forceinline__
#else
#define TSU_HD inline
#endif

namespace tsu {

// The cell whose values global index I, -2 <= I < n + 2, takes along one axis of n
// cells with the boundary rules lo and hi (0: wall, the mirror image across the
// domain's edge; else extrapolation, the edge's cell).  Always inside the domain, also
// on an axis of one cell, where the image of the second ghost cell lies past the other
// edge and is taken on by that edge's rule.  flip: the values' normal momentum changes
// sign (once for each wall).  Returns whether I lies outside.
TSU_HD bool boundary_source(int I, int n, int lo, int hi, int &src, bool &flip)
{
    flip = false;
    src = I;
    if (I < 0) {
        flip = lo == 0;
        src = lo == 0 ? -1 - I : 0;
        if (src >= n) {   // (one cell, I = -2: its image is cell 1)
            flip = flip != (hi == 0);
            src = n - 1;
        }
    } else if (I >= n) {
        flip = hi == 0;
        src = hi == 0 ? 2 * n - 1 - I : n - 1;
        if (src < 0) {    // (one cell, I = 2: its image is cell -1)
            flip = flip != (lo == 0);
            src = 0;
        }
    }
    return I < 0 || I >= n;
}

}  // namespace tsu
