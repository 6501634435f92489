// The node stack of the FP32-mixed gravity walk (k_walk32 in sph_gravity.cu): how
// many nodes a warp takes per turn, and the room their children need.
#pragma once

#ifdef __CUDACC__
#define SPH_WALK __host__ __device__ __forceinline__
#else
#define SPH_WALK inline
#endif

namespace sph {
namespace grav {

constexpr int kStack32 = 384;
constexpr int kChildren = 8;      // at most, per node
constexpr int kLevels = 8;        // Morton bits per axis: levels 0 (root) to 8

// Nodes to take off a stack of sp: as many as leave room for their children and
// for a depth-first walk from there (a node at a time: 7 more per level, at most
// kLevels of them).
SPH_WALK int walk_take(int sp) {
  const int room = (kStack32 - 8 * kLevels - sp) / (kChildren - 1);
  const int most = room < 1 ? 1 : (room > 32 ? 32 : room);
  return sp < most ? sp : most;
}

// Whether a walk goes on at sp: nodes are left, and the children of those that
// walk_take takes fit.  A walk that ends with nodes left has overrun the stack, which
// a tree of kLevels levels cannot; one comparison per turn guards it (a check at each
// push took 2% of the call).
SPH_WALK bool walk_on(int sp) {
  return (unsigned)(sp - 1) < (unsigned)(kStack32 - (kChildren - 1));
}

}  // namespace grav
}  // namespace sph
