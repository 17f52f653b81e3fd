// Whether a box of C components over z by x by y nodes fits in CAP words of shared memory.
// Plain C++ as well as device code.
#pragma once

#ifdef __CUDACC__
#define PIC_HD __host__ __device__
#else
#define PIC_HD
#endif

namespace pic {

// A chunk of sparse particles can span the whole grid, and pic_create accepts grids of close to 2^31 cells:
// the full product does not fit in 32 bits.  Each extent is held against CAP before it is multiplied, so
// no product here exceeds C CAP^2 < 2^31.  Extents are positive.
template <int C, int CAP>
PIC_HD constexpr bool box_fits(int z, int x, int y = 1) {
    static_assert((long long)C * CAP * CAP < (1LL << 31), "the products fit in 32 bits");
    return z <= CAP && x <= CAP && z * x <= CAP && y <= CAP && C * (z * x) * y <= CAP;
}

}  // namespace pic
