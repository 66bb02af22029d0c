// tiles.h -- node tables of the FP32 J V's element tiles.
//
// A tile is the run of elements (Morton order) that one block of the J V kernel works on:
// 64 hexahedra have 125 to 160 different corner nodes for their 512 corners.  With a table
// of those nodes a block brings every node once into shared memory (instead of 4 times from
// L2), interpolates a hanging node once, and adds a node's shares of all corners before an
// atomic leaves the SM (instead of 4).  On the uniform level-7 cube the corners' own float4
// gathers and atomics take 62 us of a launch, their scalar atomics 150 us.  Small meshes take
// smaller tiles (block_threads).
//
// The nodes' values lie in shared memory by slots: an entry's slot modulo 2^dim is its first
// corner's index xor its element's, the parity of the node's coordinates where the mesh is
// uniform.  The 16-byte loads of eight lanes (a cell's nodes) then meet different banks:
// 4.0 wavefronts per load of a warp on a uniform mesh and 4.1 on the membrane-band octree,
// 6.5 and 7.0 with the slots in the order of the entries.
//
// Record of a tile, all that a block needs to know of the mesh (16-byte aligned, `bytes`):
//   int32  id[cap]     node of entry u, or -(h+1) for hanging node h (ascending; `cnt` used)
//   uint16 seg[cap]    the corners of entry u: ord[seg[u]] .. ord[end - 1], end = seg[u + 1],
//                      or the tile's corners for the last entry
//   uint16 slot[cap]   slot of entry u, below `slots`
//   uint8  face[cap]   boundary-face bits of entry u's node
//   uint16 loc[corners]  slot of a corner (element-major)
//   uint16 ord[corners]  the corners ordered by entry, each by the place of its share
//                      (tile_share)
//   uint8  level[corners / 2^dim], padded to 16
//   int32  par[4 hcap], uint8 pface[4 hcap]  of the hanging entries (the first ones): the
//                      parents (two: the third is -1) and their boundary-face bits
//   int32  cnt, corners in use (2 more unused)
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

struct TileTab {
  const uint8_t* rec = nullptr;
  int64_t n = 0;      // tiles
  int threads = 0;    // per block of the kernel
  int corners = 0;    // per tile
  int cap = 0;        // entries at most, a multiple of 16
  int hcap = 0;       // hanging entries at most, a multiple of 4
  int slots = 0;      // slots at most
  int bytes = 0;      // of a record
  int blocks[2] = {0, 0};  // of the J V's persistent grid, without and with advection
};

// offsets in a record of the fields after the 4-byte and 2-byte ones of an entry
__host__ __device__ inline int tile_level_at(int corners, int cap) { return 9 * cap + 4 * corners; }
__host__ __device__ inline int tile_par_at(int corners, int nc, int cap) {
  return tile_level_at(corners, cap) + (corners / nc + 15) / 16 * 16;
}
__host__ __device__ inline int tile_bytes(int corners, int nc, int cap, int hcap) {
  return tile_par_at(corners, nc, cap) + 20 * hcap + 16;
}
// Place of a corner's share of the element vectors.  Hexahedra have two threads (by z) with
// four corners (x + 2 y) each: share j of a thread lies in row j, and the threads' order in a
// row is such that the shares of a 2 x 2 x 2 block's nodes from the same corner of their
// elements are in different banks.
__host__ __device__ inline int tile_share(int corner, int nc, int corners) {
  if (nc == 4) return corner;
  const int t = corner / 4;
  return (corner & 3) * (corners / 4) + (t ^ (t >> 3 & 1));
}

// Counts (rec null: the largest counts of entries, slots and hanging entries into
// most[0 .. 2], zeroed by the caller) or builds (rec) the records of a mesh (device tables conn [E][2^dim], level, faces).
struct TileMeshTables {
  int64_t n_elem;
  const int32_t *conn, *hang_par;
  const uint8_t *level, *faces, *hang_np;
};
cudaError_t launch_build_tiles(int dim, const TileMeshTables& M, int corners, int cap, int hcap, uint8_t* rec,
                               int* most, cudaStream_t s);

#ifdef __CUDACC__
// the record at p (shared memory)
struct TileView {
  const uint8_t* p;
  int cnt, corners;
  __device__ __forceinline__ int32_t id(const TileTab&, int u) const { return reinterpret_cast<const int32_t*>(p)[u]; }
  __device__ __forceinline__ const uint16_t* seg(const TileTab& t) const {
    return reinterpret_cast<const uint16_t*>(p + 4 * t.cap);
  }
  __device__ __forceinline__ int slot(const TileTab& t, int u) const { return seg(t)[t.cap + u]; }
  __device__ __forceinline__ uint8_t face(const TileTab& t, int u) const { return p[8 * t.cap + u]; }
  __device__ __forceinline__ const uint16_t* loc(const TileTab& t) const {
    return reinterpret_cast<const uint16_t*>(p + 9 * t.cap);
  }
  __device__ __forceinline__ const uint16_t* ord(const TileTab& t) const { return loc(t) + t.corners; }
  __device__ __forceinline__ int level(const TileTab& t, int e) const { return p[tile_level_at(t.corners, t.cap) + e]; }
  // of a hanging entry
  __device__ __forceinline__ int4 parents(const TileTab& t, int u) const {
    return reinterpret_cast<const int4*>(p + t.bytes - 16 - 20 * t.hcap)[u];
  }
  __device__ __forceinline__ uchar4 parent_faces(const TileTab& t, int u) const {
    return reinterpret_cast<const uchar4*>(p + t.bytes - 16 - 4 * t.hcap)[u];
  }
};
__device__ __forceinline__ TileView tile_view(const uint8_t* p, const TileTab& t) {
  const int2 n = *reinterpret_cast<const int2*>(p + t.bytes - 16);
  return TileView{p, n.x, n.y};
}
#endif
