// Exchange of halo rows between the tiles of the shared-memory SOR solve.
// With one grid barrier per sweep a block may publish sweep k while another has
// not yet loaded what sweep k starts from, so the rows go through two copies of
// the potential in turn (0: phi itself, which holds the starting guess): sweep k
// loads the copy that sweep k - 1 published and publishes the other, whose last
// readers passed the barrier before.  Plain C++, for host and device.
#pragma once
#if defined(__CUDACC__)
#define EKL_RIM_HD __host__ __device__
#else
#define EKL_RIM_HD
#endif

namespace ekl {

EKL_RIM_HD inline int rim_load_copy(int sweep) { return sweep & 1; }
EKL_RIM_HD inline int rim_store_copy(int sweep) { return (sweep & 1) ^ 1; }

}  // namespace ekl
