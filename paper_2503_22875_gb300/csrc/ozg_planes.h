// Layout of a set of digit planes (host and device).
#pragma once

namespace ozg {

// Difference planes.  For up to kd slices a plane set holds, in blocks t = 1 .. kd, the digit plane
// t and then the planes of digit p minus digit q for p < q, p + q = t + 1 (p = 1, 2, ..): the
// planes that slice count t adds to t - 1.  Digit planes above kd follow without differences.
__host__ __device__ inline int kd_plane_base(int t) { return (t - 1) + (t - 1) * (t - 1) / 4; }  // first of block t
// index of digit plane t in a set with differences up to kd (kd = 0: digit planes only)
__host__ __device__ inline int kd_plane(int t, int kd) {
  return t <= kd ? kd_plane_base(t) : kd_plane_base(kd + 1) + (t - kd - 1);
}
// planes of a set of s digit planes
__host__ __device__ inline int kd_planes(int s, int kd) { return kd_plane(s, kd) + (s <= kd ? 1 + s / 2 : 1); }
constexpr int kKdMax = 12;  // largest slice count with difference planes

}  // namespace ozg
