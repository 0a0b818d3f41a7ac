// lane_quads.h -- the lanes of a warp in groups of four consecutive ones. Plain C++ as well as CUDA, so that the host
// can evaluate it.
#pragma once

#ifdef __CUDACC__
#define LAIR_HD __host__ __device__ __forceinline__
#else
#define LAIR_HD inline
#endif

namespace lair {

// A walk over the groups that have a lane in the mask:
//   for (int p = 0; lanes_from(lanes, p); p += 4) if (lane_quad(lanes, p)) ...
// The mask is shifted by less than its width only: by 32, which p reaches when one of lanes 28 to 31 is in the mask, a
// shift is undefined (the GPU's gives 0, x86's leaves the mask as it is).
LAIR_HD constexpr bool lanes_from(unsigned lanes, int p) { return p < 32 && lanes >> p != 0; }
LAIR_HD constexpr bool lane_quad(unsigned lanes, int p) { return ((lanes >> p) & 15u) != 0; }   // p < 32

}  // namespace lair
