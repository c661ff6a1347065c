// Neighbours in a zincblende block by bit operations on the site number, shared by the H·X and
// valence-force-field kernels.
#pragma once

#include <cuda_runtime.h>

#include "sk_device.cuh"

// Whether component i of bond direction k is minus: the sign of p_i and of the i-th t2g orbital.
__host__ __device__ constexpr bool dir_minus(int k, int i) {
  return k != 0 && i != k - 1;   // (1,1,1), (1,-1,-1), (-1,1,-1), (-1,-1,1)
}

// Where the bonds of one atom lead.  With the four A sites (000), (022), (202), (220) and the B
// sites those plus (111), direction k joins A site s with B site s^k, and crosses into the next
// cell down (seen from A; up from B) along each axis where dir_k is minus and the site's
// coordinate is 0 (B: 3).  So an atom has one possible step per axis, the same for all its bonds.
struct Steps {
  int d[3];        // cell index change of the step along each axis (0: this site never steps there)
  unsigned bits;   // bit d: that step crosses a face of the block; bit 4 + d: and leaves a hard wall
};

__device__ __forceinline__ Steps steps_of(const Geo& g, int b, int ix, int iy, int iz) {
  const bool is_a = b < 4;
  const int s = b & 3;
  const int at[3] = {ix, iy, iz}, ext[3] = {g.nx, g.ny, g.nz}, str[3] = {1, g.nx, g.nx * g.ny};
  Steps t;
  t.bits = 0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const bool can = is_a ? (s == 0 || s == d + 1) : (s != 0 && s != d + 1);
    const bool edge = is_a ? at[d] == 0 : at[d] == ext[d] - 1;
    const int down = edge ? (ext[d] - 1) * str[d] : -str[d];   // of an A atom; a B atom's is the opposite
    t.d[d] = can ? (is_a ? down : -down) : 0;
    if (can && edge) t.bits |= (g.periodic[d] == OMEN_HARD_WALL ? 17u : 1u) << d;
  }
  return t;
}

struct Neighbour {
  int atom;
  int slot;        // bond slot (the A end's)
  unsigned wrap;   // bit d: the bond crosses a face along d (downwards from an A atom)
  bool ok;         // false: the bond leaves a hard wall
};

__device__ __forceinline__ Neighbour neighbour_of(const Geo& g, const Steps& t, int b, int k, int cell) {
  const bool is_a = b < 4;
  const int s = b & 3;
  int cell2 = cell;
  unsigned mask = 0;
#pragma unroll
  for (int d = 0; d < 3; ++d)
    if (dir_minus(k, d)) {
      cell2 += t.d[d];
      mask |= 1u << d;
    }
  Neighbour n;
  n.wrap = t.bits & mask;
  n.ok = (t.bits & (mask << 4)) == 0;
  n.atom = ((s ^ k) + (is_a ? 4 : 0)) * g.ncells + cell2;
  n.slot = is_a ? (k * 4 + s) * g.ncells + cell : (k * 4 + (s ^ k)) * g.ncells + cell2;
  return n;
}
