// Tables of a decode step in three launches over all groups (gsi_flat.cu).
#pragma once

#include "gsi_umma.cuh"   // WideGroup

namespace gsi {

constexpr int kFlatMaxGroups = 512;   // (prefix sums in shared memory)
constexpr int kFlatMaxSlots = 64;     // CTAs that share the rows of one basis (their partials are added by each of them)
constexpr int kFlatMaxGrid = 160;
constexpr int kFlatMaxD = 16384;      // sixteen warps share a row of W

// Rows [r0, r1) of a group's basis, in units of 16, are one CTA's; its partial sums are number `slot`.
struct FlatShare {
  int group, r0, r1, slot;
};

// A group's shares are [first, first + slots) of the list, in the order of their rows.
struct FlatGroup {
  int first, slots;
  int O, k, d;
  float eps;
  unsigned flags;
  int unused;
};

struct FlatParams {
  const WideGroup* table;    // [n] (without tensor maps)
  const int* first;          // [grid + 1]: every CTA's first share
  const FlatShare* shares;
  const FlatGroup* groups;   // [n]
  float2* norms;             // [shares]: ||r||^2 and ||x||^2 of their rows
  int n, n_shares;
  int use_counter;
  int* step;                 // moved on by the last launch if use_counter
  int* arrived;              // its CTAs that have read it
};

cudaError_t launch_flat_step(const FlatParams& p, int grid, int most_k, cudaStream_t st);

}  // namespace gsi
