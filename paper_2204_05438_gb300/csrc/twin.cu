// The twin array from the triangles alone (the step before the paper's input: its
// Neighbor array, Section 2, comes from the triangulator).  Half-edge h = 3t + k
// runs from tri[h] to tri[3t + (k+1) % 3]; its twin is the half-edge running the
// other way, or -1.
//
// One pass over tiles of kTwinTile triangles:
//   in shared memory, each half-edge writes itself to its edge's slot and reads what
//   stands there: of two twins one has lost the slot to the other and has found it.  Those
//   that lost to another edge try a second slot;
//   in a table of half-edges in memory, one word per edge, the half-edges left take a
//   free word or find their twin in it, and for each pair of a tile its later half-edge
//   takes a word, closed.  A third half-edge of an edge, or a second in the same
//   direction, meets one of the others in a slot or a word: POLYLLA_ERR_TOPOLOGY.
#include "polylla_internal.cuh"

namespace polylla {

// What bounds it: the compare-and-swaps in L2 and their latency, one or two per edge, a
// chain of about four for the longest of a warp, and the issue slots of the tiles' part.
// Tiles: in an order with locality (a space-filling curve, a triangulator's insertion
// order) 94 % of the half-edges have their twin among 512 triangles; those need neither a
// second compare-and-swap nor the other's vertices from memory.  1,024 triangles: 96 %,
// but fewer warps in flight; 256: 92 %.
// Table: a word is a half-edge, whose vertices are looked up in tri, not a pair of
// vertices.  An edge's words are near those of its region: 8 words, a sector, per vertex
// (3 edges on average, those of which the vertex is the owner), then words anywhere,
// then all in turn; the table is larger than the number of half-edges, so that a search
// always ends.
// Before: lists of half-edges per origin, searched for the twin (count, tile sums, scan,
// first slots, fill, match).  With the launches and the wait, before and now: 4.0M
// triangles of a mixture 227 us, 180; 400,000 of them 49, 31; 1,981 of a uniform mesh
// 29, 20; 2.0M in random order (nothing to find in a tile) 222, 155; a fan of 100,000
// (its hub's list) 5,540, 131.  The table alone, without tiles: 212, 36, 19, 107, 230.  A list
// per owner with a warp matching 32 of them in shared memory: 204, 53, 35, 162.
constexpr int kTwinTile = 512;  // triangles
constexpr int kTwinEdges = 3 * kTwinTile;
constexpr int kTwinPer = kTwinTile / kBlock;  // triangles of a thread
constexpr unsigned kTwinSlots = 4096;         // of a tile: more than twice its edges
constexpr unsigned kTwinGroup = 8;            // words of a vertex
constexpr unsigned kTwinRandom = 64;          // words tried anywhere
constexpr unsigned kTwinFree = 0xffffffffu;
constexpr unsigned kTwinClosed = 0x80000000u;

// (the multipliers here and in tile_slot: a prime next to 2^32 over the golden ratio, and the
// low word of 2^64 over it; the two of MurmurHash3's 32-bit finaliser, A. Appleby, public
// domain; 0x7feb352d from C. Wellons' search for 32-bit mixers, public domain)
__device__ __forceinline__ unsigned twin_hash(unsigned a, unsigned b, unsigned i) {
  unsigned x = a * 0x9e3779b1u ^ (b + i * 0x7f4a7c15u) * 0x85ebca6bu;
  x ^= x >> 15;
  x *= 0xc2b2ae35u;
  return x ^ x >> 13;
}

// The i-th word tried for an edge of lo and hi, beyond its owner's group.
__device__ __noinline__ unsigned twin_far(unsigned lo, unsigned hi, unsigned i, unsigned words) {
  i -= kTwinGroup;
  const unsigned r =
      (unsigned)((unsigned long long)twin_hash(lo, hi, min(i, kTwinRandom)) * words >> 32);
  return i <= kTwinRandom ? r : (unsigned)(((unsigned long long)r + (i - kTwinRandom)) % words);
}

// The i-th word tried for the edge of u and v; scale: groups per vertex, 32.32.
__device__ __forceinline__ unsigned twin_word(int u, int v, unsigned i, unsigned words,
                                              unsigned long long scale) {
  // the owner: either vertex, so that a hub or a low id owns half of its edges
  const unsigned lo = min(u, v), hi = max(u, v);
  const bool low = (lo ^ hi) & 1;
  if (i >= kTwinGroup) return twin_far(lo, hi, i, words);
  return (unsigned)((low ? lo : hi) * scale >> 32) * kTwinGroup + ((low ? hi : lo) + i) % kTwinGroup;
}

// A vertex out of range is reported whatever else is wrong with the mesh.
__device__ __forceinline__ void set_range_error(Counters* C) {
  const int was = atomicCAS(&C->error, 0, (int)POLYLLA_ERR_RANGE);
  if (was == (int)POLYLLA_ERR_TOPOLOGY) atomicCAS(&C->error, was, (int)POLYLLA_ERR_RANGE);
  if (was == 0 || was == (int)POLYLLA_ERR_TOPOLOGY) C->err_info = 140;
}

// A slot of the tile's table for an edge: round r = 0, 1.
__device__ __forceinline__ unsigned tile_slot(int u, int v, int r) {
  const unsigned lo = min(u, v), hi = max(u, v);
  const unsigned x = r ? lo * 0x85ebca6bu + hi * 0xc2b2ae35u : lo * 0x9e3779b1u + hi * 0x7feb352du;
  return x / (unsigned)(0x100000000ull / kTwinSlots);
}

// Half-edge l = u -> v of a tile: its twin, when the edge's slot holds it (a half-edge
// and the next of its triangle, 16 bits each).
__device__ __forceinline__ void match_in_tile(const int* s_v, int* s_mate, int l, int u, int v,
                                              unsigned slot, Counters* C) {
  const int o = (int)(slot & 0xffff);
  if (o == l) return;
  const int a = s_v[o], b = s_v[slot >> 16];
  if (a == v && b == u && u != v) {
    s_mate[l] = o;
    if (atomicExch(s_mate + o, l) != -1) set_error(C, POLYLLA_ERR_TOPOLOGY, 141);
  } else if (a == u && b == v) {
    set_error(C, POLYLLA_ERR_TOPOLOGY, 141);
  }
}

// (6 blocks an SM, 40 registers: 180 us at 4.0M triangles; 4 blocks, nothing spilled: 208)
__global__ void __launch_bounds__(kBlock, 6) k_twin_build(const int* __restrict__ tri, long long m,
                                                          long long n, int* __restrict__ twin,
                                                          unsigned* __restrict__ table,
                                                          unsigned words, unsigned long long scale,
                                                          Counters* C) {
  __shared__ int s_v[kTwinEdges];
  __shared__ int s_mate[kTwinEdges];
  __shared__ unsigned s_slot[kTwinSlots];
  __shared__ unsigned short s_list[kTwinEdges];
  __shared__ int s_open;
  const int lane = threadIdx.x & 31;
  for (long long t0 = (long long)blockIdx.x * kTwinTile; t0 < m;
       t0 += (long long)gridDim.x * kTwinTile) {
    const int base = (int)(3 * t0), count = (int)min((long long)kTwinEdges, 3 * (m - t0));
    int v[kTwinPer][3];
#pragma unroll
    for (int j = 0; j < kTwinPer; ++j) {
      const int l = 3 * (threadIdx.x + j * kBlock);
#pragma unroll
      for (int k = 0; k < 3; ++k) v[j][k] = l < count ? __ldg(tri + base + l + k) : -1;
    }
    if (threadIdx.x == 0) s_open = 0;
#pragma unroll
    for (int j = 0; j < kTwinPer; ++j) {
      const int l = 3 * (threadIdx.x + j * kBlock);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (l < count && (v[j][k] < 0 || v[j][k] >= n)) {
          set_range_error(C);
          v[j][k] = -1;
        }
        s_v[l + k] = v[j][k];
        s_mate[l + k] = -1;
      }
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (min(v[j][k], v[j][(k + 1) % 3]) >= 0)
          s_slot[tile_slot(v[j][k], v[j][(k + 1) % 3], 0)] = (l + k) | (l + (k + 1) % 3) << 16;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kTwinPer; ++j) {
      const int l = 3 * (threadIdx.x + j * kBlock);
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (min(v[j][k], v[j][(k + 1) % 3]) >= 0)
          match_in_tile(s_v, s_mate, l + k, v[j][k], v[j][(k + 1) % 3],
                        s_slot[tile_slot(v[j][k], v[j][(k + 1) % 3], 0)], C);
    }
    __syncthreads();
    // the half-edges that lost their slot to another edge, and those without a twin here
#pragma unroll
    for (int j = 0; j < kTwinPer; ++j) {
      const int l = 3 * (threadIdx.x + j * kBlock);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const bool open = min(v[j][k], v[j][(k + 1) % 3]) >= 0 && s_mate[l + k] < 0;
        const unsigned who = __ballot_sync(0xffffffffu, open);
        int at = 0;
        if (lane == 0 && who) at = atomicAdd(&s_open, __popc(who));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (open) s_list[at + __popc(who & ((1u << lane) - 1))] = (unsigned short)(l + k);
      }
    }
    __syncthreads();
    const int opens = s_open;
    for (int j = threadIdx.x; j < opens; j += kBlock) {
      const int l = s_list[j], ln = he_next(l);
      s_slot[tile_slot(s_v[l], s_v[ln], 1)] = l | ln << 16;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < opens; j += kBlock) {
      const int l = s_list[j], u = s_v[l], w = s_v[he_next(l)];
      match_in_tile(s_v, s_mate, l, u, w, s_slot[tile_slot(u, w, 1)], C);
    }
    __syncthreads();
    for (int l = threadIdx.x; l < count; l += kBlock) {
      const int mate = s_mate[l];
      twin[base + l] = mate >= 0 ? base + mate : -1;
    }
    __threadfence();  // the words of twin before their half-edges can be found
    __syncthreads();
    // the half-edges left, and the later one of each pair, into the table
    unsigned open = 0, closed = 0;
#pragma unroll
    for (int j = 0; j < kTwinPer; ++j) {
      const int l = 3 * (threadIdx.x + j * kBlock);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int mate = s_mate[l + k];
        if (min(v[j][k], v[j][(k + 1) % 3]) >= 0 && l + k > mate) open |= 1u << (3 * j + k);
        if (mate >= 0) closed |= 1u << (3 * j + k);
      }
    }
    for (unsigned i = 0; open; ++i) {
      unsigned o[kTwinPer][3];
#pragma unroll
      for (int j = 0; j < kTwinPer; ++j)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const unsigned bit = 1u << (3 * j + k);
          if (!(open & bit)) continue;
          const unsigned h = base + 3 * (threadIdx.x + j * kBlock) + k;
          o[j][k] = atomicCAS(table + twin_word(v[j][k], v[j][(k + 1) % 3], i, words, scale),
                              kTwinFree, closed & bit ? h | kTwinClosed : h);
        }
#pragma unroll
      for (int j = 0; j < kTwinPer; ++j)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const unsigned bit = 1u << (3 * j + k);
          if (!(open & bit)) continue;
          if (o[j][k] == kTwinFree) {
            open &= ~bit;
            continue;
          }
          const int g = (int)(o[j][k] & ~kTwinClosed), u = v[j][k], w = v[j][(k + 1) % 3];
          const int a = __ldg(tri + g), b = __ldg(tri + he_next(g));
          if (a == w && b == u && u != w && !(closed & bit) && !(o[j][k] & kTwinClosed)) {
            const int h = base + 3 * (threadIdx.x + j * kBlock) + k;
            if (atomicCAS(twin + g, -1, h) != -1) set_error(C, POLYLLA_ERR_TOPOLOGY, 141);
            twin[h] = g;
            open &= ~bit;
          } else if ((a == u && b == w) || (a == w && b == u)) {
            set_error(C, POLYLLA_ERR_TOPOLOGY, 141);
            open &= ~bit;
          }
        }
    }
#pragma unroll
    for (int j = 0; j < kTwinPer; ++j)
#pragma unroll
      for (int k = 0; k < 3; ++k)  // an edge from a vertex to itself
        if (v[j][k] >= 0 && v[j][k] == v[j][(k + 1) % 3]) {
          const int h = base + 3 * (threadIdx.x + j * kBlock) + k;
          twin[h] = h;
        }
    __syncthreads();  // (the next tile's vertices)
  }
}

cudaError_t launch_build_twin(const int* tri, long long m, long long n, int* twin, int* table,
                              Counters* C, cudaStream_t s) {
  const long long tiles = (m + kTwinTile - 1) / kTwinTile;
  const long long words = twin_words(m);
  const unsigned long long scale =
      ((unsigned long long)(words / kTwinGroup) << 32) / (unsigned long long)n;
  cudaError_t e = cudaMemsetAsync(table, 0xff, sizeof(int) * (size_t)words, s);
  if (e != cudaSuccess) return e;
  static std::atomic<int> cap{0};
  const int g = resident_grid(reinterpret_cast<const void*>(k_twin_build), kBlock, 0, tiles, &cap);
  k_twin_build<<<g, kBlock, 0, s>>>(tri, m, n, twin, reinterpret_cast<unsigned*>(table),
                                    (unsigned)words, scale, C);
  return cudaGetLastError();
}

}  // namespace polylla

namespace polylla {

// ------------------------------------------------------------------ Neighbor array
// The twin array from the triangulator's Neighbor array (Section 2): nb[3t + j] is
// the triangle across edge j of t, or -1 on the border.  Edge j is the one
// opposite vertex j (convention 0, the layout of Triangle's .neigh files) or the
// one from vertex j to vertex j+1 (convention 1).  The twin of h = 3t + k (from
// u = tri[h] to v = tri[3t + (k+1) % 3]) is the half-edge v -> u of that
// neighbour; a neighbour id outside [-1, m) is POLYLLA_ERR_RANGE, a neighbour
// without the reversed edge POLYLLA_ERR_TOPOLOGY (the twin is then -1).
__global__ void __launch_bounds__(kBlock) k_twin_from_neighbor(const int* __restrict__ tri,
                                                               const int* __restrict__ nb,
                                                               long long m, int convention,
                                                               int* __restrict__ twin,
                                                               Counters* C) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < m;
       t += (long long)gridDim.x * blockDim.x) {
    const int a[3] = {__ldg(tri + 3 * t), __ldg(tri + 3 * t + 1), __ldg(tri + 3 * t + 2)};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int j = convention ? k : (k + 2) % 3;  // the edge u -> v is opposite vertex k+2
      const int u = __ldg(nb + 3 * t + j);
      int g = -1;
      if (u >= 0 && u < m) {
        const int from = a[(k + 1) % 3], to = a[k];  // the twin runs v -> u
#pragma unroll
        for (int q = 0; q < 3; ++q)
          if (__ldg(tri + 3LL * u + q) == from && __ldg(tri + 3LL * u + (q + 1) % 3) == to)
            g = 3 * u + q;
        if (g < 0) set_error(C, POLYLLA_ERR_TOPOLOGY, 150);
      } else if (u < -1 || u >= m) {
        set_error(C, POLYLLA_ERR_RANGE, 151);
      }
      twin[3 * t + k] = g;
    }
  }
}

cudaError_t launch_twin_from_neighbor(const int* tri, const int* nb, long long m, int convention,
                                      int* twin, Counters* C, int grid, cudaStream_t s) {
  static std::atomic<int> cap{0};
  grid = resident_grid(reinterpret_cast<const void*>(k_twin_from_neighbor), kBlock, 0, grid, &cap);
  k_twin_from_neighbor<<<grid, kBlock, 0, s>>>(tri, nb, m, convention, twin, C);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ Trivertex
// The Trivertex array (Section 2: one element incident to each vertex; the
// paper's reparation reaches a tip's fan through it): for every vertex, the
// smallest half-edge leaving it, or -1 for a vertex no triangle uses.  tv starts
// as all ones (0xffffffff = -1); each half-edge lowers its origin's word.
__global__ void __launch_bounds__(kBlock) k_trivertex(const int* __restrict__ tri, long long m,
                                                      long long n, unsigned* __restrict__ tv,
                                                      Counters* C) {
  const long long H = 3 * m;
  for (long long h = blockIdx.x * (long long)blockDim.x + threadIdx.x; h < H;
       h += (long long)gridDim.x * blockDim.x) {
    const int v = __ldg(tri + h);
    if (v < 0 || v >= n) {
      set_error(C, POLYLLA_ERR_RANGE, 152);
      continue;
    }
    atomicMin(tv + v, (unsigned)h);
  }
}

cudaError_t launch_trivertex(const int* tri, long long m, long long n, int* tv, Counters* C,
                             int grid, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(tv, 0xff, sizeof(int) * (size_t)n, s);
  if (e != cudaSuccess) return e;
  static std::atomic<int> cap{0};
  grid = resident_grid(reinterpret_cast<const void*>(k_trivertex), kBlock, 0, grid, &cap);
  k_trivertex<<<grid, kBlock, 0, s>>>(tri, m, n, reinterpret_cast<unsigned*>(tv), C);
  return cudaGetLastError();
}

}  // namespace polylla
