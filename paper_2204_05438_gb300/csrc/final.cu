// Output CSR (the paper's Mesh and Position arrays, Section 2).  Every output
// polygon already sits in the vertex pool in its final vertex order (written by
// the thread or block that walked it); the order of the polygons is fixed here:
// traversal polygons in seed order, each split polygon replaced in place by its
// pieces.  One single-pass scan over the polygons' (piece count, vertex count)
// replaces the paper's AtomicAdd on i_Gmesh / i_Gpos, and each polygon's pieces
// are copied to their offsets in the same pass.
#include "walk.cuh"

namespace polylla {

__device__ __forceinline__ void out_counts(const PolyArrays& P, long long i, long long* c,
                                           long long* l) {
  const int pc = P.pcnt[i];
  *c = pc == 0 ? 1 : pc;
  *l = P.flen[i];
}

// Every polygon's output -- its pieces in order, for a split one -- lies in one
// contiguous stretch of the pool, and the output of a warp's 32 polygons is one
// contiguous stretch of the CSR.  The warp copies that stretch flat, a lane per vertex:
// the vertex's polygon is the number of polygons that start at or before it (a bit per
// polygon start in a 32-vertex window), and each polygon has one distance from its
// place in the stretch to its place in the pool.  kOutLoads windows are loaded before
// any is stored, so that a warp's ten windows take two round trips to L2, however its
// polygons lie in the pool.
//
// What bounds it: latency (a tile's records, its look-back, its copies).  Copying one
// after another the runs that are contiguous in the pool as well took a round trip per
// run, and the polygons that splits take out of the walk's order leave five or so of
// them to a warp.  Times before and after, us: gmm16-10m 135 and 115, 1M uniform points
// 35 and 28, 200,000 mixture points 29 and 14, 20,000 points with holes 22 and 11.
//
// A block takes SUB consecutive 256-polygon sub-tiles per ticket (one look-back tile):
// four on large meshes, so that one look-back serves 1024 polygons (gmm16-10m 115 us
// against 158 with one), one on small meshes, whose tiles would leave SMs idle (20,000
// points: 11 us against 17; at 1M points, kOutSmall, 28 against 31).  The tile
// offsets come from a look-back over `status` in the same pass (tiles in ticket
// order; one word per tile packs the piece count << 33 | vertex count, exact
// within the mesh size limits), and the last tile writes the totals and the CSR
// end marker.  The status words clean themselves: the block that finishes the last
// tile (C->out_done counts them) clears them and the count.
constexpr int kOutLoads = 6;
constexpr long long kOutSmall = 1ll << 21;  // triangles: 1,230 tiles of 256 polygons

// Every frontier half-edge's turn ends, checked by the whole grid (a corrupt mesh
// only: out of line, so that the copy kernel does not pay registers for it).
__device__ __noinline__ void check_turns(const int* tf, int H, Counters* C) {
  for (long long h = blockIdx.x * (long long)blockDim.x + threadIdx.x; h < H;
       h += (long long)gridDim.x * blockDim.x) {
    if (tf[h] >= 0) continue;
    long long steps = 0;
    if (turn_tf(tf, (int)h, H, steps, H) < 0) set_error(C, POLYLLA_ERR_LIMIT, 50);
  }
}


template <int SUB>
__global__ void __launch_bounds__(kBlock, SUB == 4 ? 6 : 5) k_final_write(DevMesh M, const int* tf, PolyArrays P,
                                                        FinalPieces F, Pool pool,
                                                        unsigned long long* status,
                                                        long long* __restrict__ off,
                                                        int* __restrict__ vtx,
                                                        long long* __restrict__ obase,
                                                        Counters* C) {
  constexpr int kWarps = kBlock / 32;
  constexpr long long kOutTile = SUB * kPolyTile;
  constexpr long long kLen = (1ll << 33) - 1;  // counts << 33 | vertices
  static_assert(SUB * kWarps <= 32, "one warp scans the warps' totals");
  const long long m = M.m;
  __shared__ long long s_src[SUB][kBlock], s_x[SUB][kBlock];  // pool place; in-warp sums
  __shared__ int s_len[SUB][kBlock], s_pc[SUB][kBlock];
  __shared__ long long s_sum[SUB * kWarps];  // per sub-tile and warp: total, then offsets
  __shared__ long long s_dist[kWarps][32];
  __shared__ long long s_tile;
  __shared__ int s_clear;
  const long long n = C->n_seeds;
  if (C->n_vtx_trav != C->n_front) check_turns(tf, (int)(3 * m), C);
  const long long ntiles = (n + kOutTile - 1) / kOutTile;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (;;) {
    if (threadIdx.x == 0)
      s_tile = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(&C->ticket), 1ull);
    __syncthreads();
    const long long tile = s_tile;
    if (tile >= ntiles) break;
    // this thread's polygon in each sub-tile; every load issued before any use
    int pcj[SUB], lj[SUB];
#pragma unroll
    for (int j = 0; j < SUB; ++j) {
      const long long i = tile * kOutTile + (long long)j * kPolyTile + threadIdx.x;
      pcj[j] = i < n ? P.pcnt[i] : 0;
      lj[j] = i < n ? P.flen[i] : 0;
    }
#pragma unroll
    for (int j = 0; j < SUB; ++j) {
      const long long i = tile * kOutTile + (long long)j * kPolyTile + threadIdx.x;
      long long src = -1;
      if (i < n) {
        if (pcj[j] == 0) {
          src = P.pos[i];
        } else {
          const long long fb = P.pbase[i];
          if (pcj[j] > 0 && fb >= 0 && fb + pcj[j] <= F.cap) src = F.pos[fb];
          else pcj[j] = lj[j] = 0;  // (reported with the polygon's missing source)
        }
        if (lj[j] < 0) lj[j] = 0;
      }
      s_src[j][threadIdx.x] = src;
      s_len[j][threadIdx.x] = lj[j];
      s_pc[j][threadIdx.x] = pcj[j];
      // the polygon's first vertex (and its line) to L2 while the tile waits for its
      // look-back
      if (src >= 0 && src < pool.cap) asm volatile("prefetch.global.L2 [%0];" ::"l"(pool.v + src));
      const long long own = i < n ? (long long)max(pcj[j], 1) << 33 | lj[j] : 0;
      long long x = own;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
      }
      s_x[j][threadIdx.x] = x - own;
      if (lane == 31) s_sum[j * kWarps + warp] = x;
    }
    __syncthreads();
    if (warp == 0) {
      const long long own = lane < SUB * kWarps ? s_sum[lane] : 0;
      long long x = own;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
      }
      const long long all = __shfl_sync(0xffffffffu, x, 31);
      const long long ex = lookback_warp(status, tile, all, C);
      if (lane < SUB * kWarps) s_sum[lane] = ex + x - own;
      if (lane == 0 && tile == ntiles - 1) {
        const long long np = (ex + all) >> 33, nv = (ex + all) & kLen;
        C->n_poly = np;
        C->n_vtx = nv;
        if (np <= m) off[np] = nv;
        else set_error(C, POLYLLA_ERR_LIMIT, 82);
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int j = 0; j < SUB; ++j) {
      const long long i = tile * kOutTile + (long long)j * kPolyTile + threadIdx.x;
      const long long at = s_sum[j * kWarps + warp] + s_x[j][threadIdx.x];
      const long long pb = at >> 33, vb = at & kLen;
      const int pc = s_pc[j][threadIdx.x];
      const long long l = s_len[j][threadIdx.x], src = s_src[j][threadIdx.x];
      long long sj = -1;
      if (i < n) {
        if (pb + max(pc, 1) > m || vb + l > 3 * m) {
          set_error(C, POLYLLA_ERR_LIMIT, 80);
        } else {
          if (obase) obase[i] = pb;
          off[pb] = vb;
          if (src < 0 || src + l > pool.cap) set_error(C, POLYLLA_ERR_LIMIT, 81);
          else sj = src;
        }
      }
      // the offsets of the further pieces: pieces lie back to back in the pool
      for (unsigned left = __ballot_sync(0xffffffffu, sj >= 0 && pc > 1); left; left &= left - 1) {
        const int a = __ffs(left) - 1;
        const int pa = __shfl_sync(0xffffffffu, pc, a);
        const long long p0 = __shfl_sync(0xffffffffu, pb, a), v0 = __shfl_sync(0xffffffffu, vb, a);
        const long long q0 = __shfl_sync(0xffffffffu, sj, a);
        const long long fb = __shfl_sync(0xffffffffu, (long long)(pc > 1 ? P.pbase[i] : 0), a);
        for (int r = 1 + lane; r < pa; r += 32) off[p0 + r] = v0 + (F.pos[fb + r] - q0);
      }
      // the copy: start is the polygon's place in the warp's stretch
      const long long w0 = __shfl_sync(0xffffffffu, vb, 0);
      const long long total = __shfl_sync(0xffffffffu, vb + l, 31) - w0;
      const int E = total <= 3 * m ? (int)total : 0;  // (more only after an error)
      const int start = (int)(vb - w0);
      const bool some = l > 0;
      const unsigned um = __ballot_sync(0xffffffffu, some);
      if (some)
        s_dist[warp][__popc(um & ((1u << lane) - 1u))] = sj >= 0 ? sj - start : -(1ll << 40);
      __syncwarp();
      const unsigned upto = (2u << lane) - 1u;
      int* const to = vtx + w0;
      int before = -1;
      for (int e0 = 0; e0 < E; e0 += 32 * kOutLoads) {
        int v[kOutLoads];
        unsigned ok = 0;
#pragma unroll
        for (int u = 0; u < kOutLoads; ++u) {
          const int wu = e0 + 32 * u;
          if (wu < E) {
            const unsigned starts =
                __reduce_or_sync(0xffffffffu, some && start >> 5 == wu >> 5 ? 1u << (start & 31) : 0u);
            const long long src = s_dist[warp][before + __popc(starts & upto)] + (wu + lane);
            before += __popc(starts);
            if (wu + lane < E && src >= 0) {
              v[u] = pool.v[src];
              ok |= 1u << u;
            }
          }
        }
#pragma unroll
        for (int u = 0; u < kOutLoads; ++u)
          if (ok >> u & 1u) to[e0 + 32 * u + lane] = v[u];
      }
      __syncwarp();
    }
    if (threadIdx.x == 0) {
      // the last tile to finish clears the status words for the next pass; the fence
      // keeps this tile's own word from arriving after that
      __threadfence();
      const unsigned long long done =
          atomicAdd(reinterpret_cast<unsigned long long*>(&C->out_done), 1ull);
      s_clear = done == (unsigned long long)(ntiles - 1);
    }
    __syncthreads();
    if (s_clear) {
      for (long long q = threadIdx.x; q < ntiles; q += kBlock) status[q] = 0;
      if (threadIdx.x == 0) C->out_done = 0;
    }
  }
}

cudaError_t launch_final_write(const DevMesh& M, const int* tf, const PolyArrays& P,
                               const FinalPieces& F, const Pool& pool, unsigned long long* status,
                               long long* off, int* vtx, long long* obase, Counters* C, int grid,
                               cudaStream_t s) {
  // seeds are about a seventh of the triangles, and never more than all of them
  static std::atomic<int> cap1{0}, cap4{0};
  if (M.m <= kOutSmall) {
    grid = resident_grid(reinterpret_cast<const void*>(k_final_write<1>), kBlock, 0, grid, &cap1);
    k_final_write<1><<<grid, kBlock, 0, s>>>(M, tf, P, F, pool, status, off, vtx, obase, C);
  } else {
    grid = resident_grid(reinterpret_cast<const void*>(k_final_write<4>), kBlock, 0, grid, &cap4);
    k_final_write<4><<<grid, kBlock, 0, s>>>(M, tf, P, F, pool, status, off, vtx, obase, C);
  }
  return cudaGetLastError();
}

}  // namespace polylla
