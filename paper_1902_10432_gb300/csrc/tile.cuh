// Bodies' phase-field tiles on the device: coordinates, overlap, and the launch geometry that the tile
// kernels (phase.cu, lbm.cu) share.
#pragma once

#include "cbl_dev.cuh"

namespace cbl {

// A phase counts as present where phi > PHI_EPS; the clamp sets phi < PHI_EPS to 0 and
// phi > 1 - PHI_EPS to 1. This keeps "present" (which sets N in the kinetics) from hinging on the
// last bit of a rounding, and keeps the support of a moving field compact.
constexpr double PHI_EPS = 1e-12;

// the clamp, on bit patterns (a NaN goes to 0, as by fmax)
__device__ __forceinline__ long long phi_clamp(long long b) {
  if (b < dbits(PHI_EPS) || b > 0x7FF0000000000000LL) return 0;
  return b > dbits(1.0 - PHI_EPS) ? dbits(1.0) : b;
}

// Launch geometry of the tile kernels: block (x, y, z) takes cells [256 x, 256 x + 256) of the tile's
// planes Z y .. Z y + Z - 1 of body z. One division per thread gives its column (a flat cell index needs
// three), and what depends on the column is computed once for Z cells. Most cells of a tile need nothing
// (phi is 0 around a body and 1 inside it); a kernel writes those at once, collects the others in shared
// memory (TileList) and works on them in full warps, because GB300 issues FP64 at 1/64 of the FP32 rate
// and a warp instruction holds that pipe for all its lanes, active or not. Z = 4 where that leaves a
// few blocks per SM, else 1 (tile_planes): with few blocks the one with most interface cells sets the time.
constexpr int TILE_T = 256, TILE_Z = 4;

inline int tile_planes(const ChainLaunch& c, int sms) {
  const long long xy = (c.max_xy + TILE_T - 1) / TILE_T, z = (c.max_z + TILE_Z - 1) / TILE_Z;
  return xy * z * c.bodies >= 4LL * sms ? TILE_Z : 1;
}

struct TileList {
  unsigned short id[TILE_T * TILE_Z];
  int n;
};

// every thread of the block: append `id` where want (warp-aggregated)
__device__ __forceinline__ void tile_append(TileList& l, bool want, int id) {
  const unsigned m = __ballot_sync(0xffffffffu, want);
  if (!m) return;
  const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(&l.n, __popc(m));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (want) l.id[base + __popc(m & ((1u << lane) - 1u))] = (unsigned short)id;
}

// the body of this block, and the context it belongs to: a single context is a kernel argument, a batch's
// are in a table, its bodies numbered over all of them
template <bool B>
__device__ __forceinline__ const TileSet& tile_set(const TileSet& one, const TileSet* __restrict__ sets,
                                                   const int2* __restrict__ items, int& self) {
  if constexpr (B) {
    const int2 it = items[blockIdx.z];
    self = it.y;
    return sets[it.x];
  } else {
    self = blockIdx.z;
    return one;
  }
}

struct TileCell {
  int i0, i1, i2;  // tile-local
  int gx, gy, gz;  // global (wrapped)
};

__device__ __forceinline__ TileCell tile_at(const BodyDev& b, int i0, int i1, int i2, const Lat& lat) {
  TileCell c;
  c.i0 = i0;
  c.i1 = i1;
  c.i2 = i2;
  c.gx = wrapi_near(b.o[0] + i0, lat.nx);
  c.gy = wrapi_near(b.o[1] + i1, lat.ny);
  c.gz = wrapi_near(b.o[2] + i2, lat.nz);
  return c;
}

__device__ __forceinline__ TileCell tile_cell(const BodyDev& b, long long t, const Lat& lat) {
  const unsigned u = (unsigned)t, L0 = (unsigned)b.L[0], L1 = (unsigned)b.L[1];  // tiles hold < 2^31 cells
  const unsigned r = u / L0;
  return tile_at(b, (int)(u - r * L0), (int)(r % L1), (int)(r / L1), lat);
}

__device__ __forceinline__ long long lat_index(const TileCell& c, const Lat& lat) {
  return c.gx + (long long)lat.nx * (c.gy + (long long)lat.ny * c.gz);
}

// the outer two layers of a tile, its stencils' halo (none along an axis that the tile spans)
__device__ __forceinline__ bool tile_halo(const BodyDev& b, const int nn[3], int i0, int i1, int i2) {
  return (b.L[0] < nn[0] && (i0 < 2 || i0 >= b.L[0] - 2)) || (b.L[1] < nn[1] && (i1 < 2 || i1 >= b.L[1] - 2)) ||
         (b.L[2] < nn[2] && (i2 < 2 || i2 >= b.L[2] - 2));
}

// local index of global cell g in a tile with origin o, or -1 if outside
__device__ __forceinline__ long long tile_index(const int o[3], const int L[3], int gx, int gy, int gz, const Lat& lat) {
  int a = wrapi_near(gx - o[0], lat.nx), b = wrapi_near(gy - o[1], lat.ny), c = wrapi_near(gz - o[2], lat.nz);
  if (a >= L[0] || b >= L[1] || c >= L[2]) return -1;
  return (long long)a + (long long)L[0] * ((long long)b + (long long)L[1] * c);
}

__device__ __forceinline__ bool covered_by_lower_body(const BodyDev* bodies, const BodyDev& b, int self, int gx, int gy,
                                                      int gz, const Lat& lat) {
  for (int k = 0; k < b.nnb; ++k) {
    int o = b.nbl[k];
    if (o >= self) break;
    if (tile_index(bodies[o].o, bodies[o].L, gx, gy, gz, lat) >= 0) return true;
  }
  return false;
}

}  // namespace cbl
