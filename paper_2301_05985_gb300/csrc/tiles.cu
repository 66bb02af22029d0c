// tiles.cu -- the node tables of the element tiles (tiles.h): one block per tile, a thread per
// corner.
#include "kernels.h"
#include "tiles.h"

namespace {

// The nodes of a tile meet in a hash table in shared memory (twice as many places as corners);
// entries are ranked by node id and an entry's corners by index, by counting the smaller ones,
// so that a table does not depend on the order of the atomics.  (Ids in order: entries in the
// order of their first corners made the J V 6 % slower on the uniform level-7 cube, its loads
// and atomics touch more sectors.)  There, 32,768 tiles: 156 us to count, 412 us to build; sorting the
// (node, corner) pairs took 475 and 539 us.
constexpr int kMaxCorners = 512, kEmpty = INT32_MIN;
__global__ void __launch_bounds__(kMaxCorners)
    k_build_tiles(TileMeshTables M, int nc, int cap, int hcap, uint8_t* __restrict__ rec, int* __restrict__ most) {
  __shared__ int node[2 * kMaxCorners], first[2 * kMaxCorners];
  __shared__ uint16_t entry_of[2 * kMaxCorners], slot_of[kMaxCorners], list[kMaxCorners], rank_of[kMaxCorners];
  __shared__ int count[kMaxCorners], start[kMaxCorners + 1];
  // the record, written out as a whole (field by field its 2-byte stores took most of the time)
  __shared__ uint4 image[(29 * kMaxCorners + 4 * kMaxCorners + kMaxCorners / 4 + 32) / 16];
  __shared__ int heads[33][9];  // per warp, then before it: heads of each class, heads
  __shared__ __align__(16) int head_id[kMaxCorners + 4];
  const int tl = blockDim.x, i = threadIdx.x, lane = i & 31, warp = i >> 5, n_warps = tl >> 5;
  const int64_t L = M.n_elem * nc, t0 = (int64_t)blockIdx.x * tl, t = t0 + i;
  const int used = (int)(L - t0 < tl ? L - t0 : tl);
  for (int h = i; h < 2 * tl; h += tl) {
    node[h] = kEmpty;
    first[h] = tl;
  }
  count[i] = 0;
  __syncthreads();
  const int32_t id = i < used ? M.conn[t] : 0;
  int h = 0;
  if (i < used) {
    h = (int)((uint32_t)id * 2654435769u >> 12) & (2 * tl - 1);
    for (;;) {
      const int was = atomicCAS(node + h, kEmpty, id);
      if (was == kEmpty || was == id) break;
      h = (h + 1) & (2 * tl - 1);
    }
    atomicMin(first + h, i);
  }
  __syncthreads();
  const bool head = i < used && first[h] == i;
  const int cls = (i / nc ^ i) & (nc - 1);
  const unsigned before = (1u << lane) - 1;
  int rank = 0;
  for (int c = 0; c < nc; ++c) {
    const unsigned m = __ballot_sync(0xFFFFFFFFu, head && cls == c);
    if (cls == c) rank = __popc(m & before);
    if (lane == 0) heads[warp][c] = __popc(m);
  }
  const unsigned hm = __ballot_sync(0xFFFFFFFFu, head);
  if (lane == 0) heads[warp][nc] = __popc(hm);
  const int n_hang = __syncthreads_count(head && id < 0);
  if (i <= nc) {
    int sum = 0;
    for (int w = 0; w < n_warps; ++w) {
      const int x = heads[w][i];
      heads[w][i] = sum;
      sum += x;
    }
    heads[32][i] = sum;
    if (i < nc && !rec) atomicMax(most + 1, sum * nc);
  }
  __syncthreads();
  const int cnt = heads[32][nc];
  if (!rec) {
    if (i == 0) {
      atomicMax(most, cnt);
      atomicMax(most + 2, n_hang);
    }
    return;
  }
  const int sl = (heads[warp][cls] + rank) * nc + cls;  // of a head
  const int packed = heads[warp][nc] + __popc(hm & before);  // of a head: ranked by packed threads
  if (head) head_id[packed] = id;
  if (i < 4) head_id[cnt + i] = INT32_MAX;
  __syncthreads();
  if (i < cnt) {
    const int mine = head_id[i];
    int n = 0;
    for (int k = 0; k < cnt; k += 4) {
      const int4 o = *reinterpret_cast<const int4*>(head_id + k);
      n += (o.x < mine) + (o.y < mine) + (o.z < mine) + (o.w < mine);
    }
    rank_of[i] = (uint16_t)n;
  }
  __syncthreads();
  if (head) {
    entry_of[h] = rank_of[packed];
    slot_of[rank_of[packed]] = (uint16_t)sl;
  }
  __syncthreads();
  const int u = i < used ? entry_of[h] : 0;
  const int place = i < used ? atomicAdd(count + u, 1) : 0;
  __syncthreads();
  // start[u]: corners of the entries before u
  {
    const int c = count[i];
    int x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) heads[warp][0] = x;
    __syncthreads();
    int sum = 0;
    for (int w = 0; w < warp; ++w) sum += heads[w][0];
    start[i] = sum + x - c;
    if (i == tl - 1) start[tl] = sum + x;
  }
  __syncthreads();
  if (i < used) list[start[u] + place] = (uint16_t)i;
  __syncthreads();
  int at = i < used ? start[u] : 0;  // of corner i in its entry's list
  if (i < used)
    for (int k = start[u]; k < start[u + 1]; ++k) at += list[k] < i;
  const int bytes = tile_bytes(tl, nc, cap, hcap);
  uint8_t* r = reinterpret_cast<uint8_t*>(image);
  int32_t* id_of = reinterpret_cast<int32_t*>(r);
  uint16_t *seg = reinterpret_cast<uint16_t*>(r + 4 * cap), *slot = seg + cap,
           *loc = reinterpret_cast<uint16_t*>(r + 9 * cap), *ord = loc + tl;
  uint8_t *face = r + 8 * cap, *lev = r + tile_level_at(tl, cap);
  int4* par = reinterpret_cast<int4*>(r + tile_par_at(tl, nc, cap));
  uchar4* pface = reinterpret_cast<uchar4*>(par + hcap);
  if (i < used) {
    loc[i] = slot_of[u];
    ord[at] = (uint16_t)tile_share(i, nc, tl);
    if (head) {
      id_of[u] = id;
      seg[u] = (uint16_t)start[u];
      slot[u] = (uint16_t)sl;
      face[u] = id >= 0 ? M.faces[id] : 0;
      if (id < 0) {
        const int32_t* p = M.hang_par + 4 * (int64_t)(-id - 1);
        const bool four = M.hang_np[-id - 1] != 2;
        par[u] = make_int4(p[0], p[1], four ? p[2] : -1, four ? p[3] : -1);
        pface[u] = make_uchar4(M.faces[p[0]], M.faces[p[1]], four ? M.faces[p[2]] : 0, four ? M.faces[p[3]] : 0);
      }
    }
  } else {
    loc[i] = slot_of[0];  // corners past the end read entry 0
    ord[i] = 0;
  }
  if (i < (tl / nc + 15) / 16 * 16) {
    const int64_t e = t0 / nc + i;
    lev[i] = i < tl / nc && e < M.n_elem ? M.level[e] : 0;
  }
  for (int w = cnt + i; w < cap; w += tl) {
    id_of[w] = 0;
    seg[w] = slot[w] = 0;
    face[w] = 0;
  }
  for (int w = n_hang + i; w < hcap; w += tl) {
    par[w] = make_int4(0, 0, 0, 0);
    pface[w] = make_uchar4(0, 0, 0, 0);
  }
  if (i == 0) {
    int32_t* tail = reinterpret_cast<int32_t*>(pface + hcap);
    tail[0] = cnt;
    tail[1] = used;
    tail[2] = tail[3] = 0;
  }
  __syncthreads();
  uint4* out = reinterpret_cast<uint4*>(rec + (int64_t)blockIdx.x * bytes);
  for (int k = i; k < bytes / 16; k += tl) out[k] = image[k];
}

}  // namespace

cudaError_t launch_build_tiles(int dim, const TileMeshTables& M, int corners, int cap, int hcap, uint8_t* rec,
                               int* most, cudaStream_t s) {
  if (M.n_elem == 0) return cudaSuccess;
  if (corners > kMaxCorners || cap > kMaxCorners || hcap > kMaxCorners) return cudaErrorInvalidValue;
  const unsigned n = (unsigned)(((M.n_elem << dim) + corners - 1) / corners);
  k_build_tiles<<<n, corners, 0, s>>>(M, 1 << dim, cap, hcap, rec, most);
  note_launch();
  return cudaGetLastError();
}
