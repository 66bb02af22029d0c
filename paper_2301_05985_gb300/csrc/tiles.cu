// tiles.cu -- the node tables of the element tiles (tiles.h): one block per tile sorts its
// (node, corner) pairs in shared memory.
#include "kernels.h"
#include "tiles.h"

namespace {

// Key: uint32_t while (nodes + hanging) x corners fits, else uint64_t.  The sort of 32-bit
// keys takes a third of the instructions.
template <typename Key>
__global__ void __launch_bounds__(1024)
    k_build_tiles(TileMeshTables M, int nc, int cap, int hcap, uint8_t* __restrict__ rec, int* __restrict__ most) {
  __shared__ Key key[1024];
  __shared__ uint16_t slot_of[1024];
  // per warp: heads (entries that start there), and heads of each class; then sums before it
  __shared__ int heads[33], cls_heads[32][8];
  const int tl = blockDim.x, i = threadIdx.x, lane = i & 31, warp = i >> 5, n_warps = tl >> 5;
  const int64_t L = M.n_elem * nc, t0 = (int64_t)blockIdx.x * tl, t = t0 + i;
  const int used = (int)(L - t0 < tl ? L - t0 : tl), bits = 31 - __clz(tl);
  const int n_hanging = (int)M.n_hanging;
  // ascending by signed id, then by corner; corners past the end last.  Bitonic, a pair's
  // exchange within a warp by shuffles
  Key mine = i < used ? (Key)((Key)(M.conn[t] + n_hanging) << bits | (Key)i) : ~Key(0);
  for (int k = 2; k <= tl; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      Key other;
      if (j < 32) {
        other = __shfl_xor_sync(0xFFFFFFFFu, mine, j);
      } else {
        __syncthreads();
        key[i] = mine;
        __syncthreads();
        other = key[i ^ j];
      }
      const bool low = ((i & j) == 0) == ((i & k) == 0);  // keeps the smaller one
      mine = low ? min(mine, other) : max(mine, other);
    }
  __syncthreads();
  key[i] = mine;
  __syncthreads();
  const int corner = (int)(mine & (Key)(tl - 1)), cls = (corner / nc ^ corner) & (nc - 1);
  const bool head = i < used && (i == 0 || (key[i - 1] >> bits) != (mine >> bits));
  const unsigned before = (1u << lane) - 1, hm = __ballot_sync(0xFFFFFFFFu, head);
  int rank = 0;
  for (int c = 0; c < nc; ++c) {
    const unsigned m = __ballot_sync(0xFFFFFFFFu, head && cls == c);
    if (cls == c) rank = __popc(m & before);
    if (lane == 0) cls_heads[warp][c] = __popc(m);
  }
  if (lane == 0) heads[warp] = __popc(hm);
  __syncthreads();
  if (i <= nc) {  // sums over the warps: thread c < nc of class c, thread nc of all
    int sum = 0;
    for (int w = 0; w < n_warps; ++w) {
      int* p = i < nc ? &cls_heads[w][i] : &heads[w];
      const int x = *p;
      *p = sum;
      sum += x;
    }
    if (i == nc) heads[n_warps] = sum;
    else if (!rec) atomicMax(most + 1, sum * nc);
  }
  __syncthreads();
  const int cnt = heads[n_warps];
  // hanging entries come first
  const int n_hang = __syncthreads_count(head && (int64_t)(mine >> bits) < n_hanging);
  if (!rec) {
    if (i == 0) {
      atomicMax(most, cnt);
      atomicMax(most + 2, n_hang);
    }
    return;
  }
  const int u = heads[warp] + __popc(hm & (before | 1u << lane)) - 1;  // entry of this pair
  const int sl = (cls_heads[warp][cls] + rank) * nc + cls;             // of a head
  if (head) slot_of[u] = (uint16_t)sl;
  __syncthreads();
  uint8_t* r = rec + (int64_t)blockIdx.x * tile_bytes(tl, nc, cap, hcap);
  int32_t* id = reinterpret_cast<int32_t*>(r);
  uint16_t *seg = reinterpret_cast<uint16_t*>(r + 4 * cap), *slot = seg + cap,
           *loc = reinterpret_cast<uint16_t*>(r + 9 * cap), *ord = loc + tl;
  uint8_t *face = r + 8 * cap, *lev = r + tile_level_at(tl, cap);
  int4* par = reinterpret_cast<int4*>(r + tile_par_at(tl, nc, cap));
  uchar4* pface = reinterpret_cast<uchar4*>(par + hcap);
  if (i < used) {
    loc[corner] = slot_of[u];
    ord[i] = (uint16_t)tile_share(corner, nc, tl);
    if (head) {
      const int32_t nid = (int32_t)(mine >> bits) - n_hanging;
      id[u] = nid;
      seg[u] = (uint16_t)i;
      slot[u] = (uint16_t)sl;
      face[u] = nid >= 0 ? M.faces[nid] : 0;
      if (nid < 0) {
        const int32_t* p = M.hang_par + 4 * (int64_t)(-nid - 1);
        const bool four = M.hang_np[-nid - 1] != 2;
        par[u] = make_int4(p[0], p[1], four ? p[2] : -1, four ? p[3] : -1);
        pface[u] = make_uchar4(M.faces[p[0]], M.faces[p[1]], four ? M.faces[p[2]] : 0, four ? M.faces[p[3]] : 0);
      }
    }
  } else {
    loc[i] = slot_of[0];  // corners past the end read entry 0
    ord[i] = 0;
  }
  if (i < tl / nc) {
    const int64_t e = t0 / nc + i;
    lev[i] = e < M.n_elem ? M.level[e] : 0;
  }
  for (int w = cnt + i; w < cap; w += tl) {
    id[w] = 0;
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
  }
}

}  // namespace

cudaError_t launch_build_tiles(int dim, const TileMeshTables& M, int corners, int cap, int hcap, uint8_t* rec,
                               int* most, cudaStream_t s) {
  if (M.n_elem == 0) return cudaSuccess;
  if (corners > 1024) return cudaErrorInvalidValue;
  const unsigned n = (unsigned)(((M.n_elem << dim) + corners - 1) / corners);
  if ((M.n_nodes + M.n_hanging) * corners < int64_t(0xFFFFFFFF))
    k_build_tiles<uint32_t><<<n, corners, 0, s>>>(M, 1 << dim, cap, hcap, rec, most);
  else
    k_build_tiles<uint64_t><<<n, corners, 0, s>>>(M, 1 << dim, cap, hcap, rec, most);
  note_launch();
  return cudaGetLastError();
}
