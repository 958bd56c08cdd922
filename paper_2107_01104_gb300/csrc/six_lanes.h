// Lane arithmetic of the groups of six lanes (float64 steps, I = 6), in plain
// C++: the kernels and a host check use the same lines.
//
// Five groups take lanes 0..29; lanes 30 and 31 repeat lanes 24 and 25 in
// everything: what they compute, what they read from other lanes, and what they
// store to the group's weight buffer, so that both stores of an entry carry the
// same value.
#pragma once

#ifdef __CUDACC__
#define TRK_LANES_HD __host__ __device__
#else
#define TRK_LANES_HD
#endif

namespace trk {

struct SixLanes {
    int group, u, base;   // the lane's group, its place (stencil column) there, the group's first lane
    TRK_LANES_HD constexpr explicit SixLanes(int lane) : group(lane / 6 < 4 ? lane / 6 : 4), u(lane % 6), base(6 * group) {}

    // Sums of three values over the group: lanes 2 q and 2 q + 1 add the even and the
    // odd columns of value q.  Column next(1) of value q comes from lane pair next(1), to
    // whom q is next(2), and the other way round.
    TRK_LANES_HD constexpr int value() const { return u >> 1; }
    TRK_LANES_HD constexpr int next(int k) const { return (value() + k) % 3; }
    TRK_LANES_HD constexpr int partner(int k) const { return base + 2 * next(k) + (u & 1); }
    // a lane that holds the sum of value i
    TRK_LANES_HD constexpr int holder(int i) const { return base + 2 * i; }
};

}  // namespace trk
