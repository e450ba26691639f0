// Which form the Arnoldi step takes, by what the device has room for (plain C++).
#pragma once

namespace vie {

constexpr int kMaxCluster = 16;  // blocks of the cluster form

// What a device (or the part of it a process sees) offers the one-launch step.
struct ArnoldiRoom {
  int cluster;   // largest cluster of its CTAs: 16, 8 (portable), or 0
  int resident;  // its CTAs resident at once over all SMs
};

// Blocks of one cluster of a step over `blocks` blocks per right-hand side:
// with 16 of them a batch puts two in a CTA.
inline int arnoldi_cluster(int blocks, int R) { return R > 1 && blocks == kMaxCluster ? blocks / 2 : blocks; }

// One launch: always with one block; as a cluster per right-hand side up to
// kMaxCluster blocks; above, for a single right-hand side, with every block
// resident.  Else the separate launches, which wait for no other block.
inline bool arnoldi_one_launch(int blocks, int R, const ArnoldiRoom &room) {
  if (blocks == 1) return true;
  if (blocks <= kMaxCluster) return arnoldi_cluster(blocks, R) <= room.cluster;
  return R == 1 && blocks <= room.resident;
}

}  // namespace vie
