// Index arithmetic of the tracking kernel, in plain C++ so that host programs can
// check it.
#pragma once
#include <math.h>

#ifdef __CUDACC__
#define DGF_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define DGF_HOST_DEVICE inline
#endif

namespace dgf {

// Rows of a warp's reduction scratch: one per lane, kRowStride floats apart. The lanes
// of a group (G consecutive ones) own the G rows from 20 g0 on, g0 being the warp lane of
// the group's lane 0, and no group touches another's: the groups of a warp need no
// barrier between a reduction of one and one of the other kind of its neighbour.
constexpr int kRowStride = 20;

// Place of value i of warp lane wl in the 4-value reduction, inside the group's own rows
// (the last is 20 g0 + 24 + 40 * 3 + 7 < 20 (g0 + 8)). A value's lanes lie side by side,
// values 40 floats apart and groups G floats past their rows' start, so that a value's
// 4-byte stores of all groups hit distinct banks, and so do the 16-byte reads of eight
// consecutive lanes.
DGF_HOST_DEVICE int short_place(int wl, int lane, int i) { return kRowStride * (wl - lane) + 40 * i + wl; }

// First of the four places lane reads: value lane & 3 of lanes 4 (lane >> 2) .. + 3.
DGF_HOST_DEVICE int short_read(int wl, int lane) { return short_place(wl & ~3, lane & ~3, lane & 3); }

// First tap column (or row) of the support of radius R around a position whose rounded
// down coordinate on an axis of n pixels is floor_p. Positions are the caller's and may lie
// anywhere: ones more than kFar pixels outside the axis, infinities and NaN are brought
// to kFar pixels outside it, where every tap clamps to the border pixel all the same, so
// that no index computed from the origin leaves the range of int.
constexpr int kFar = 64;
DGF_HOST_DEVICE int tap_origin(float floor_p, int R, int n)
{
    return (int)fminf(fmaxf(floor_p, -(float)kFar), (float)n + (float)kFar) - R;
}

// Whether the taps first .. first + count - 1 lie within an axis of n pixels and its
// replicated border.
DGF_HOST_DEVICE bool taps_inside(int first, int count, int n, int border)
{
    return first >= -border && first + count <= n + border;
}

}  // namespace dgf
