// Layout of a set of digit planes (host and device), and the memory a larger layout may take.
#pragma once
#include <cstddef>
#include <cstdint>

namespace ozg {

// Row pitch of a digit plane in elements (fp16): whole 128-byte lines, so that the 128-byte row of a
// TMA box is one line.  With rows only 16-byte aligned every box row straddles two: 1537 x
// 2001 with k = 1111, s = 10 took 639 us instead of 540, the learned batch of 2048 uneven calls 28.4
// ms instead of 27.4.  tight: 16-byte rows, for calls whose workspace does not have the room (a short
// k's planes take up to eight times the space on whole lines).
inline int64_t plane_pitch(int64_t k, bool tight) { return tight ? (k + 7) / 8 * 8 : (k + 63) / 64 * 64; }

// Size a workspace is allocated with when it has to hold `bytes`.
inline size_t workspace_size(size_t bytes) { return (bytes + bytes / 8 + ((size_t)1 << 20) - 1) >> 20 << 20; }
// Whether a workspace that now has cap bytes may be one for `bytes`, where a call needs no more than
// `lean`: difference planes, window words and whole-line rows make a call faster at up to eight times the
// workspace, which the context then keeps.  Beyond what the lean layout takes they may have a quarter of
// the memory that it leaves free, so that a program that shares the device keeps most of it.
inline bool layout_room(size_t cap, size_t lean, size_t bytes, size_t free_bytes) {
  if (bytes <= cap) return true;
  const size_t least = lean > cap ? workspace_size(lean) : cap, want = workspace_size(bytes);
  if (want <= least) return true;
  return least <= cap + free_bytes && want - least <= (cap + free_bytes - least) / 4;
}

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
