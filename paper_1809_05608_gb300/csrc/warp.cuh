// Which lanes take part in a warp operation, by arithmetic that the host can check.
#pragma once

namespace mgfld {

// The lanes of a warp that hold rows of one group of n consecutive rows, `lane` holding row k of it and the warp
// having `live` lanes: the members of a reduction over the group's part of the warp, known without asking which
// lanes happen to be converged.
__host__ __device__ constexpr unsigned group_lanes(int lane, int k, int n, int live) {
  const int lo = lane - k > 0 ? lane - k : 0;
  const int hi = lane - k + n < live ? lane - k + n - 1 : live - 1;
  return (0xffffffffu >> (31 - hi)) & (0xffffffffu << lo);
}

// A wait that a whole warp goes through together: one look, then the bounded wait.  The copy may complete between
// the looks of two lanes, so nothing but the votes tells a lane whether the others have seen it, and every lane takes
// part in as many of them.
template <class Look, class Bounded, class All>
__host__ __device__ inline bool warp_wait(Look look, Bounded bounded, All all) {
  if (all(look())) return true;
  return all(bounded());
}

// The last ring use whose copy has been issued when a warp waits for use u of NU, in a ring of S: the first S go out up
// front, use u - 1's steps issue one more once they hold the last rows of use u - 2.
__host__ __device__ constexpr int ring_last_issued(int u, int S, int NU) {
  const int v = u == 0 ? S - 1 : u + S - 2;
  return v < NU ? v : NU - 1;
}

}  // namespace mgfld
