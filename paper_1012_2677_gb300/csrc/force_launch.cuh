// Launches of k_force_tile for one precision and list form: included by the translation unit that
// builds the form (one each, so that they compile in parallel).
#pragma once

#include "tile.cuh"

namespace ljmd {

template <bool MIXED, bool HALF, bool WHOLE, bool LONGLIST, int LANES, bool ENERGY>
static void force_tile_launch(const ForceLaunch& a) {
  set_smem(k_force_tile<MIXED, LANES, HALF, ENERGY, WHOLE, LONGLIST>, a.smem);
  k_force_tile<MIXED, LANES, HALF, ENERGY, WHOLE, LONGLIST><<<a.grid, kTileThreads, a.smem, a.s>>>(
      a.pos, a.cs, a.N, a.g, a.ta, a.c, a.rows, a.tile_list, a.ent, a.f, a.part, a.status, a.nbuf, a.skip);
}

template <bool MIXED, bool HALF, bool WHOLE, bool LONGLIST, int LANES>
static void force_tile_energy(const ForceLaunch& a) {
  if (a.energy) force_tile_launch<MIXED, HALF, WHOLE, LONGLIST, LANES, true>(a);
  else force_tile_launch<MIXED, HALF, WHOLE, LONGLIST, LANES, false>(a);
}

template <bool MIXED, bool HALF, bool WHOLE, bool LONGLIST>
static void force_tile_lanes(const ForceLaunch& a) {
  switch (a.lanes) {
    case 1: force_tile_energy<MIXED, HALF, WHOLE, LONGLIST, 1>(a); break;
    case 2: force_tile_energy<MIXED, HALF, WHOLE, LONGLIST, 2>(a); break;
    case 4: force_tile_energy<MIXED, HALF, WHOLE, LONGLIST, 4>(a); break;
    case 8: force_tile_energy<MIXED, HALF, WHOLE, LONGLIST, 8>(a); break;
    case 16: force_tile_energy<MIXED, HALF, WHOLE, LONGLIST, 16>(a); break;
    default: force_tile_energy<MIXED, HALF, WHOLE, LONGLIST, 32>(a); break;
  }
}

// The mixed form: whole box, tiles with long segments, tiles.
template <bool HALF>
static void force_tile_mixed(const ForceLaunch& a) {
  if (a.ta.whole) force_tile_lanes<true, HALF, true, false>(a);
  else if (a.ta.list_cap < a.ta.max_list) force_tile_lanes<true, HALF, false, true>(a);  // some beyond the staged capacity
  else force_tile_lanes<true, HALF, false, false>(a);
}

}  // namespace ljmd
