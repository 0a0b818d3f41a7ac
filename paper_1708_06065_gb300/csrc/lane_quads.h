// lane_quads.h -- the lanes of a warp in groups of four consecutive ones. Plain C++ as well as CUDA, so that the host
// can evaluate it.
#pragma once

#ifdef __CUDACC__
#define LAIR_HD __host__ __device__ __forceinline__
#else
#define LAIR_HD inline
#endif

namespace lair {

// The first lane of the first group at or after lane p (a multiple of 4, at most 32) of which any lane is in `lanes`,
// or 32. The mask is shifted by less than its width only: by 32, which p reaches when one of lanes 28 to 31 is in the
// mask, a shift is undefined (the GPU's gives 0, x86's leaves the mask as it is).
LAIR_HD constexpr int next_lane_quad(unsigned lanes, int p) {
    while (p < 32 && ((lanes >> p) & 15u) == 0) p += 4;
    return p;
}

}  // namespace lair
