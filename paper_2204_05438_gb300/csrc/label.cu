// Label phase (Section 3.2.1, Algorithm 2) and seed compaction.
//
//   k_label_max    LabelMax: per triangle, the index of its longest edge.
//   k_label_class  LabelSeed + LabelFrontier fused: per triangle, the frontier
//                  flag of each edge, "longest edge is terminal" and the seed
//                  flag.
//   k_seed_write   the Seed array compacted in ascending order, the tile
//                  offsets by a decoupled look-back in the same pass.
//
// All three are HBM streams over the triangle arrays (tri / twin: 12 bytes per
// triangle each, read as 3 x int4 per thread of 4 triangles) with gathers of
// vertex coordinates (LabelMax) or of neighbour label bytes (LabelSeed /
// LabelFrontier) that hit L2 on spatially ordered meshes.  Every id read from the
// input is range-checked before it is dereferenced; a bad id sets the handle's
// error word and the element is skipped.
#include "polylla_internal.cuh"

namespace polylla {

// ------------------------------------------------------------------ validation
__global__ void __launch_bounds__(kBlock) k_validate(DevMesh M, Counters* C) {
  const long long n = M.n, m = M.m, H = 3 * m;
  const long long lim = n > H ? n : H;
  const long long kMaxCoord = 1ll << 30;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < lim;
       i += (long long)gridDim.x * blockDim.x) {
    if (i < n) {
      const long long x = M.xy[2 * i], y = M.xy[2 * i + 1];
      if (x < 0 || x >= kMaxCoord || y < 0 || y >= kMaxCoord) set_error(C, POLYLLA_ERR_RANGE, 1);
    }
    if (i < H) {
      const int h = (int)i;
      const int v = M.tri[h];
      const int w = M.tri[he_next(h)];
      if (v < 0 || v >= n) {
        set_error(C, POLYLLA_ERR_RANGE, 2);
      }
      const int g = M.twin[h];
      if (g < -1 || g >= H) {
        set_error(C, POLYLLA_ERR_RANGE, 3);
      } else if (g >= 0) {
        if (g == h || M.twin[g] != h || M.tri[g] != w || M.tri[he_next(g)] != v)
          set_error(C, POLYLLA_ERR_TOPOLOGY, 4);
      }
    }
    if (i < m) {
      const int a = M.tri[3 * i], b = M.tri[3 * i + 1], c = M.tri[3 * i + 2];
      if (a < 0 || a >= n || b < 0 || b >= n || c < 0 || c >= n) continue;  // reported above
      const long long ax = M.xy[2 * a], ay = M.xy[2 * a + 1];
      const long long bx = M.xy[2 * b], by = M.xy[2 * b + 1];
      const long long cx = M.xy[2 * c], cy = M.xy[2 * c + 1];
      if (ax < 0 || ax >= kMaxCoord || ay < 0 || ay >= kMaxCoord || bx < 0 || bx >= kMaxCoord ||
          by < 0 || by >= kMaxCoord || cx < 0 || cx >= kMaxCoord || cy < 0 || cy >= kMaxCoord)
        continue;  // reported by the vertex check
      const long long orient = (bx - ax) * (cy - ay) - (by - ay) * (cx - ax);
      if (orient <= 0) set_error(C, POLYLLA_ERR_TOPOLOGY, 5);
    }
  }
}

cudaError_t launch_validate(const DevMesh& M, Counters* C, int grid, cudaStream_t s) {
  k_validate<<<grid, kBlock, 0, s>>>(M, C);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ loads
// The 12 ints of triangles 4g .. 4g+3 (3 x int4 when the group is complete;
// scalar loads, zero-filled, for the ragged last group).
__device__ __forceinline__ void load_tri_group(const int* __restrict__ a, long long g, long long m,
                                               int v[12]) {
  const long long t0 = 4 * g;
  if (t0 + 4 <= m) {
    const int4* p = reinterpret_cast<const int4*>(a) + 3 * g;
    const int4 x = __ldg(p), y = __ldg(p + 1), z = __ldg(p + 2);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
    v[8] = z.x; v[9] = z.y; v[10] = z.z; v[11] = z.w;
  } else {
#pragma unroll
    for (int j = 0; j < 12; ++j) v[j] = (3 * t0 + j < 3 * m) ? __ldg(a + 3 * t0 + j) : 0;
  }
}

__device__ __forceinline__ long long sqdist(longlong2 p, longlong2 q) {
  const long long dx = q.x - p.x, dy = q.y - p.y;
  return dx * dx + dy * dy;
}

// ------------------------------------------------------------------ LabelMax
// Longest edge by (exact squared length, then lower undirected id min(h, twin(h))).
// The twin array is read only for triangles whose longest length is tied.
// With len, also the longest edge of each kLenChunk triangles, and of all of them in
// C->max_len: what k_seed_write finds the long terminal edges by.
// (5 blocks an SM then: with the 42 registers of 6 blocks it spills, 31.0 us against 27.5 at
// 2M triangles in random order; 8M in order 49 us, 45 without len)
template <bool LEN>
__global__ void __launch_bounds__(kBlock, LEN ? 5 : 6) k_label_max(DevMesh M, uint8_t* __restrict__ lab,
                                                         unsigned* __restrict__ len, Counters* C) {
  pdl_launch_dependents();
  const long long m = M.m, n = M.n;
  const long long ngroups = (m + 3) / 4;
  unsigned seen = 0;  // the longest edge of this warp's triangles so far
  const longlong2* __restrict__ xy2 = reinterpret_cast<const longlong2*>(M.xy);
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < ngroups;
       g += (long long)gridDim.x * blockDim.x) {
    int v[12];
    load_tri_group(M.tri, g, m, v);
    unsigned packed = 0;
    unsigned longest = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const long long t = 4 * g + j;
      if (t >= m) break;
      const int a = v[3 * j], b = v[3 * j + 1], c = v[3 * j + 2];
      if ((unsigned)a >= (unsigned long long)n || (unsigned)b >= (unsigned long long)n ||
          (unsigned)c >= (unsigned long long)n) {
        set_error(C, POLYLLA_ERR_RANGE, 10);
        continue;
      }
      const longlong2 pa = __ldg(xy2 + a), pb = __ldg(xy2 + b), pc = __ldg(xy2 + c);
      const long long l0 = sqdist(pa, pb), l1 = sqdist(pb, pc), l2 = sqdist(pc, pa);
      const long long lmax = max(l0, max(l1, l2));
      if (LEN) longest = max(longest, len_key(lmax));
      const int cnt = (l0 == lmax) + (l1 == lmax) + (l2 == lmax);
      int k;
      if (cnt == 1) {
        k = (l0 == lmax) ? 0 : ((l1 == lmax) ? 1 : 2);
      } else {
        // tie at the maximum: the lower undirected edge id wins
        const long long l[3] = {l0, l1, l2};
        int best_e = 0x7fffffff;
        k = 0;
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          if (l[e] != lmax) continue;
          const int h = (int)(3 * t + e);
          const int tw = __ldg(M.twin + h);
          const int eid = (tw >= 0 && tw < h) ? tw : h;
          if (eid < best_e) {
            best_e = eid;
            k = e;
          }
        }
      }
      packed |= (unsigned)k << (8 * j);
    }
    const long long t0 = 4 * g;
    if (t0 + 4 <= m) {
      reinterpret_cast<unsigned*>(lab)[g] = packed;
    } else {
      for (int j = 0; t0 + j < m; ++j) lab[t0 + j] = (uint8_t)(packed >> (8 * j));
    }
    if (LEN) {  // the longest edge of the warp's kLenChunk triangles, and of all
      const long long lanes = ngroups - (g - g % 32);
      const unsigned here =
          __reduce_max_sync(lanes < 32 ? (1u << lanes) - 1u : 0xffffffffu, longest);
      if (g % 32 == 0) {
        len[g / 32] = here;
        seen = max(seen, here);
      }
    }
  }
  if (LEN) {  // one atomic per block: one per warp took 6 us at 2M triangles in random order
    __shared__ unsigned s_seen[kBlock / 32];
    if (threadIdx.x % 32 == 0) s_seen[threadIdx.x / 32] = seen;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
      for (int w = 1; w < kBlock / 32; ++w) seen = max(seen, s_seen[w]);
      atomicMax(&C->max_len, seen);
    }
  }
}

template <bool LEN>
cudaError_t launch_label_max_t(const DevMesh& M, uint8_t* lab, unsigned* len, Counters* C, int grid,
                               cudaStream_t s) {
  static std::atomic<int> cap{0};
  grid = resident_grid(reinterpret_cast<const void*>(k_label_max<LEN>), kBlock, 0, grid, &cap);
  k_label_max<LEN><<<grid, kBlock, 0, s>>>(M, lab, len, C);
  return cudaGetLastError();
}

cudaError_t launch_label_max(const DevMesh& M, uint8_t* lab, unsigned* len, Counters* C, int grid,
                             cudaStream_t s) {
  return (len ? launch_label_max_t<true> : launch_label_max_t<false>)(M, lab, len, C, grid, s);
}

// ------------------------------------------------------------------ LabelSeed + LabelFrontier
// Per triangle t with longest edge k* and twins g_k:
//   frontier(k)  <=> g_k < 0  or  (k != k*  and  edge g_k is not the longest of its triangle)
//   terminal     <=> g_k* < 0 or  edge g_k* is the longest of its triangle
//   seed         <=> terminal and (g_k* < 0 or t < triangle(g_k*))
// Neighbour label bytes are read while other threads rewrite them; only their
// bits 0-1 (the Max array, written by the previous kernel) are used, and every
// rewrite keeps those bits, so any version of a byte gives the same answer.
// When tf is given, also writes tf[h] = twin(h) with bit 31 set iff h is frontier
// (0x7fffffff as the twin of a border half-edge): one load then tells both
// whether a walk stops at h and where it turns next.  No barrier: each thread's 4
// triangles are independent.
__global__ void __launch_bounds__(kBlock, 5) k_label_class(DevMesh M, uint8_t* lab,
                                                           int* __restrict__ tf, Counters* C) {
  pdl_wait();  // the Max array
  pdl_launch_dependents();
  const long long m = M.m;
  const long long H = 3 * m;
  const long long ntiles = (m + kTriTile - 1) / kTriTile;
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const long long g = tile * kBlock + threadIdx.x;  // group of 4 triangles
    const long long t0 = 4 * g;
    if (t0 < m) {
      int tw[12];
      load_tri_group(M.twin, g, m, tw);
      const bool full = t0 + 4 <= m;
      unsigned own = 0;
      if (full) {
        own = *reinterpret_cast<const unsigned*>(lab + t0);
      } else {
        for (int j = 0; t0 + j < m; ++j) own |= (unsigned)lab[t0 + j] << (8 * j);
      }
      unsigned out = 0;
      int tfo[12];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const long long t = t0 + j;
        if (t >= m) break;
        const int kst = (own >> (8 * j)) & 3;
        unsigned byte = (unsigned)kst;
        unsigned nbm = 0;  // bit k: edge k is also the longest edge of the neighbour
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          if (tw[3 * j + k] >= H) {  // a border edge from here on: every tf word is frontier or a twin
            set_error(C, POLYLLA_ERR_RANGE, 11);
            tw[3 * j + k] = -1;
          }
          const int gk = tw[3 * j + k];
          if (gk >= 0) {
            const int gt = gk / 3;
            const int nb = lab[gt] & 3;
            nbm |= (unsigned)(nb == gk - 3 * gt) << k;
          }
          const bool fr = (gk < 0) || (k != kst && !((nbm >> k) & 1u));
          byte |= (unsigned)fr << (2 + k);
          tfo[3 * j + k] = (gk & 0x7fffffff) | (fr ? (int)0x80000000u : 0);
        }
        const int gs = (kst == 0) ? tw[3 * j] : ((kst == 1) ? tw[3 * j + 1] : tw[3 * j + 2]);
        const bool terminal = (gs < 0) || ((nbm >> kst) & 1u);
        const bool seed = terminal && (gs < 0 || t < gs / 3);
        byte |= (unsigned)terminal << 6;
        byte |= (unsigned)seed << 5;
        out |= byte << (8 * j);
      }
      if (full) {
        *reinterpret_cast<unsigned*>(lab + t0) = out;
        if (tf) {
          int4* q = reinterpret_cast<int4*>(tf) + 3 * g;
          q[0] = make_int4(tfo[0], tfo[1], tfo[2], tfo[3]);
          q[1] = make_int4(tfo[4], tfo[5], tfo[6], tfo[7]);
          q[2] = make_int4(tfo[8], tfo[9], tfo[10], tfo[11]);
        }
      } else {
        for (int j = 0; t0 + j < m; ++j) {
          lab[t0 + j] = (uint8_t)(out >> (8 * j));
          if (tf)
            for (int k = 0; k < 3; ++k) tf[3 * (t0 + j) + k] = tfo[3 * j + k];
        }
      }
    }
  }
}

cudaError_t launch_label_class(const DevMesh& M, uint8_t* lab, int* tf, Counters* C, int grid,
                               cudaStream_t s, bool pdl) {
  static std::atomic<int> cap{0};
  grid = resident_grid(reinterpret_cast<const void*>(k_label_class), kBlock, 0, grid, &cap);
  return launch_chain(k_label_class, grid, kBlock, 0, s, pdl, M, lab, tf, C);
}

// ------------------------------------------------------------------ seed compaction
// The Seed array compacted in ascending order in one pass: a block takes, in
// ticket order, tiles of kSeedSub sub-tiles of kSeedSpan triangles (16 per thread
// and sub-tile, one 16-byte label load each), counts their seeds (label bit 5),
// gets the tile's offset by a decoupled look-back over `status` (one word per
// tile), and writes each sub-tile's seeds -- staged in shared memory -- coalesced.
// The last tile writes the seed count to C->n_seeds.  The status words clean
// themselves: the block that finishes the last tile (C->seed_done counts
// them) clears them and the count, so nothing has to be zeroed before the next
// run; the ticket counter C->seed_ticket starts at zero with the label phase's
// counters.
// With `entry` non-null, also the terminal half-edge 3t + k of each seed t (label
// bits 0-1), where the walk enters its region.  The frontier half-edges (label bits
// 2-4) are counted in C->n_front.
// With `early`, the seeds whose regions may be long are listed (their entries carry
// kEarlyBit): those whose terminal edge is a border edge (the label's frontier bit of
// the longest edge; the slivers along a hull), and those whose terminal edge is at least a
// 16th of the mesh's longest edge (the gaps between clusters).  Counted on the host on
// uniform and mixture meshes of 1,000 to 1M points: 13-42 seeds of the first kind, and of
// the second 15-45 on mixtures, 184-237 on 1,000 uniform points, 28 or fewer on 5,000 and
// none from 20,000 on; every region of more than kWalkCap boundary edges is among them.  A
// kind with more than kEarlyMost seeds says nothing, and its seeds are the walk's like all
// others: a mesh of edges all alike, or the border kind of a domain with holes (120-218
// seeds at 20,000 uniform points, 295 at 60,000, 339 at 100,000), whose long regions are
// then walked after the others as on larger meshes.
constexpr int kSeedPer = 16;
constexpr int kSeedSpan = kBlock * kSeedPer;   // triangles per sub-tile
// Sub-tiles per look-back tile: 4, or 1 on meshes of at most kSeedSmall triangles, where
// 4 leave most of the GPU idle (us with 4 and 1, this kernel and the run: 29,667 triangles
// with holes 22 and 12, 75 and 63; 400,000 of a mixture 16 and 12, 93 and 90; 1.4M 20 and
// 15, 136 and 131; 2.0M uniform 21 and 19, 174 and 175).
constexpr int kSeedSub = 4;
constexpr long long kSeedSmall = 1 << 21;

__device__ __forceinline__ void list_early(int* early, int kind, long long i, Counters* C) {
  const long long at =
      (long long)atomicAdd(reinterpret_cast<unsigned long long*>(&C->n_early[kind]), 1ull);
  if (at < kEarlyMost) early[kind * kEarlyMost + at] = (int)i;
}

template <int kSeedSub, bool EARLY>
__global__ void __launch_bounds__(kBlock) k_seed_write(const uint8_t* __restrict__ lab, long long m,
                                                       unsigned long long* status,
                                                       int* __restrict__ seeds,
                                                       int* __restrict__ entry,
                                                       DevMesh M, const unsigned* __restrict__ len,
                                                       int* __restrict__ early, Counters* C) {
  constexpr int kSeedTile = kSeedSub * kSeedSpan;
  __shared__ int sw[kSeedSub][kBlock / 32];
  __shared__ int s_seed[kSeedSpan], s_entry[kSeedSpan];
  __shared__ long long s_tile, s_base;
  __shared__ int s_clear;
  pdl_wait();  // the label bytes
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long nbt = (m + kSeedTile - 1) / kSeedTile;
  const bool aligned16 = (reinterpret_cast<uintptr_t>(lab) & 15u) == 0;
  const unsigned longest = EARLY ? C->max_len : 0;
  const unsigned far = longest > kLenFar ? longest - kLenFar : 0;
  for (;;) {
    if (threadIdx.x == 0)
      s_tile = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(&C->seed_ticket), 1ull);
    __syncthreads();
    const long long bt = s_tile;
    if (bt >= nbt) break;
    // this thread's 16 label bytes of each sub-tile (every load issued first)
    unsigned w[kSeedSub][4];
    unsigned smask[kSeedSub];
    unsigned near = 0;  // bit j: the chunk of the sub-tile's 16 triangles has a long edge
    int incl[kSeedSub], cnt[kSeedSub];
#pragma unroll
    for (int j = 0; j < kSeedSub; ++j) {
      const long long t0 = ((bt * kSeedSub + j) * kBlock + threadIdx.x) * kSeedPer;
      w[j][0] = w[j][1] = w[j][2] = w[j][3] = 0;
      if constexpr (EARLY)
        if (t0 < m) near |= (unsigned)(len[t0 / kLenChunk] >= far) << j;
      if (t0 + kSeedPer <= m && aligned16) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(lab) + (t0 / kSeedPer));
        w[j][0] = v.x;
        w[j][1] = v.y;
        w[j][2] = v.z;
        w[j][3] = v.w;
      } else if (t0 + kSeedPer <= m) {  // a caller's label array aligned to 4 bytes only
        const unsigned* l4 = reinterpret_cast<const unsigned*>(lab + t0);
#pragma unroll
        for (int q = 0; q < 4; ++q) w[j][q] = __ldg(l4 + q);
      } else {
        for (int i = 0; i < kSeedPer && t0 + i < m; ++i)
          w[j][i >> 2] |= (unsigned)__ldg(lab + t0 + i) << (8 * (i & 3));
      }
    }
#pragma unroll
    for (int j = 0; j < kSeedSub; ++j) {
      unsigned sm = 0;  // bit i: triangle t0 + i is a seed
#pragma unroll
      for (int i = 0; i < kSeedPer; ++i) sm |= ((w[j][i >> 2] >> (8 * (i & 3) + 5)) & 1u) << i;
      smask[j] = sm;
      cnt[j] = __popc(sm);
      int x = cnt[j];
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
      }
      incl[j] = x;
      if (lane == 31) sw[j][warp] = x;
    }
    __syncthreads();
    unsigned nf = 0;
#pragma unroll
    for (int j = 0; j < kSeedSub; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) nf += __popc(w[j][q] & 0x1c1c1c1cu);
    nf = __reduce_add_sync(0xffffffffu, nf);
    if (lane == 0 && nf)
      atomicAdd(reinterpret_cast<unsigned long long*>(&C->n_front), (unsigned long long)nf);
    int sub_total[kSeedSub];
    int total = 0;
#pragma unroll
    for (int j = 0; j < kSeedSub; ++j) {
      int t = 0;
#pragma unroll
      for (int v = 0; v < kBlock / 32; ++v) t += sw[j][v];
      sub_total[j] = t;
      total += t;
    }
    if (warp == 0) {
      const long long ex = lookback_warp(status, bt, total, C);
      if (lane == 0) {
        s_base = ex;
        if (bt == nbt - 1) C->n_seeds = ex + total;
      }
    }
    __syncthreads();
    long long base = s_base;
#pragma unroll
    for (int j = 0; j < kSeedSub; ++j) {
      const long long t0 = ((bt * kSeedSub + j) * kBlock + threadIdx.x) * kSeedPer;
      int before = 0;
#pragma unroll
      for (int v = 0; v < kBlock / 32; ++v) before += (v < warp) ? sw[j][v] : 0;
      int pos = before + incl[j] - cnt[j];
      unsigned sm = smask[j];
      while (sm) {  // the seeds only, in increasing order
        const int i = __ffs(sm) - 1;
        sm &= sm - 1;
        const unsigned wq = i < 8 ? (i < 4 ? w[j][0] : w[j][1]) : (i < 12 ? w[j][2] : w[j][3]);
        const int t = (int)(t0 + i);
        const unsigned byte = wq >> (8 * (i & 3)), k = byte & 3u;
        const bool border = EARLY && (byte >> (2 + k) & 1u);  // its terminal edge
        s_seed[pos] = t | (near >> j & 1u ? (int)kEarlyBit : 0);
        s_entry[pos] = (3 * t + (int)k) | (border ? (int)kEarlyBit : 0);
        ++pos;
      }
      __syncthreads();
      for (int k = threadIdx.x; k < sub_total[j]; k += kBlock) {
        const int t = s_seed[k] & ~(int)kEarlyBit;
        int e = s_entry[k];
        seeds[base + k] = t;
        if constexpr (EARLY) {
          if (e < 0) {
            list_early(early, 0, base + k, C);
          } else if (s_seed[k] < 0 && *const_cast<volatile long long*>(&C->n_early[1]) <= kEarlyMost) {
            const int a = M.tri[e], b = M.tri[he_next(e)];
            if ((unsigned)a < (unsigned long long)M.n && (unsigned)b < (unsigned long long)M.n) {
              const longlong2* xy2 = reinterpret_cast<const longlong2*>(M.xy);
              if (len_key(sqdist(__ldg(xy2 + a), __ldg(xy2 + b))) >= far) {
                list_early(early, 1, base + k, C);
                e |= (int)kEarlyBit;
              }
            }
          }
        }
        if (entry) entry[base + k] = e;
      }
      base += sub_total[j];
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      // the last tile to finish clears the status words for the next run; the fence
      // keeps this tile's own word from arriving after that
      __threadfence();
      const unsigned long long done =
          atomicAdd(reinterpret_cast<unsigned long long*>(&C->seed_done), 1ull);
      s_clear = done == (unsigned long long)(nbt - 1);
    }
    __syncthreads();
    if (s_clear) {
      for (long long q = threadIdx.x; q < nbt; q += kBlock) status[q] = 0;
      if (threadIdx.x == 0) C->seed_done = 0;
    }
  }
}

template <int SUB, bool EARLY>
cudaError_t launch_seed_write_t(const uint8_t* lab, long long m, unsigned long long* status,
                                int* seeds, int* entry, const DevMesh& M, const unsigned* len,
                                int* early, Counters* C, cudaStream_t s, bool pdl) {
  static std::atomic<int> cap{0};
  const int grid = resident_grid(reinterpret_cast<const void*>(k_seed_write<SUB, EARLY>), kBlock, 0,
                                 (m + SUB * kSeedSpan - 1) / (SUB * kSeedSpan), &cap);
  return launch_chain(k_seed_write<SUB, EARLY>, grid, kBlock, 0, s, pdl, lab, m, status, seeds, entry, M,
                      len, early, C);
}

cudaError_t launch_seed_write(const uint8_t* lab, long long m, unsigned long long* status,
                              int* seeds, int* entry, const DevMesh& M, const unsigned* len,
                              int* early, bool small, Counters* C, cudaStream_t s, bool pdl) {
  const bool one = small && m <= kSeedSmall;
  const auto launch =
      early ? (one ? launch_seed_write_t<1, true> : launch_seed_write_t<kSeedSub, true>)
            : (one ? launch_seed_write_t<1, false> : launch_seed_write_t<kSeedSub, false>);
  return launch(lab, m, status, seeds, entry, M, len, early, C, s, pdl);
}

long long seed_tiles(long long m, bool small) {
  const long long large = (m + kSeedSub * kSeedSpan - 1) / (kSeedSub * kSeedSpan);
  const long long n = small ? (std::min(m, kSeedSmall) + kSeedSpan - 1) / kSeedSpan : 0;
  return std::max(large, n);
}

}  // namespace polylla
