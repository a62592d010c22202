// Traversal (Section 3.2.2, Algorithms 3 and 4) and, for ordinary polygons,
// reparation (Section 3.2.3, Algorithm 5) in one pass.
//
//   k_walk  a warp takes 32 seeds: the triangles of their regions, from each terminal
//           edge down the region's longest-edge tree, then every boundary edge's
//           place in its polygon (at most kWalkCap vertices) from the subtree sizes,
//           the canonical starts and the tips.  A polygon without tips (or any, when
//           no reparation is asked for) is copied, rotated to its canonical start,
//           into the vertex pool, whose space is handed out per warp.  A polygon
//           with tips is listed -- one tip (about 90% of them) or several -- so that
//           the dependent loads of a split do not stall its warp; a longer one is
//           left to one thread block (long.cu).
//   k_repair_one    one thread per polygon with one tip: split it and cut the
//           two pieces out of the vertex sequence the walk left in the pool.
//   k_repair_multi  one thread per polygon with several tips: the cycle becomes
//           a linked list of nodes in shared memory, and each split (smallest tip
//           of the current piece first) adds two chord nodes and relinks four
//           pointers.
// The paper's AtomicAdd on i_Gmesh / i_Gpos is replaced by the output scan
// (final.cu); the pool order does not matter.
#include "walk.cuh"

#include <cstddef>

namespace polylla {

// Warp-aggregated allocation: each lane asks for `need` entries; one atomic per
// warp.  All 32 lanes must call it.
__device__ __forceinline__ long long warp_alloc(long long* counter, int need) {
  const int lane = threadIdx.x & 31;
  int incl = need;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += y;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  unsigned long long base = 0;
  if (lane == 31 && total > 0)
    base = atomicAdd(reinterpret_cast<unsigned long long*>(counter), (unsigned long long)total);
  base = __shfl_sync(0xffffffffu, base, 31);
  return (long long)base + incl - need;
}


// Polygons with more tips than this are split by one thread re-walking its pieces
// (repair_seq); those with 2..kRsMaxSplit tips get the walk's tip records and the
// several-tip kernel's node list.
constexpr int kRsMaxSplit = 8;

// The walk of 32 seeds by a warp.  The non-frontier edges of a region form its
// longest-edge tree (every triangle but the terminal pair hangs from the neighbour
// across its longest edge), so the boundary cycle is the tree's tour: the subtree of
// the seed's triangle, entered through its terminal edge e0, then the one across e0
// (only e0 itself when e0 is a border edge).  A triangle entered through half-edge e
// contributes the boundary across n1 = next(e), then across n2 = prev(e): the edge
// itself if it is frontier, else the subtree behind it.  The warp does not follow the
// tour; it places every boundary edge by the sizes of the subtrees before it:
//
//   1. the triangles of the 32 regions go through one queue in shared memory, 32 a
//      pass, one lane each: two independent loads (tf[n1], tf[n2]), the children
//      appended (their queue indices in link[]);
//   2. the passes backwards: each triangle's boundary edges, from its children's;
//   3. the passes forwards: each triangle's place in its polygon, its children's, and
//      its frontier edges into he[], polygon after polygon;
//   4. the origins gathered, a lane per boundary edge; a lane per polygon scans them
//      for the smallest (origin, half-edge) and the tips; then every lane stores its
//      edges' origins, each polygon turned to start there, in one stretch of the pool.
//
// What bounds it: the latency of the queue's passes, ten on average for the 212
// triangles of 32 regions, and the instructions issued (3,000 a warp and 32 seeds, 60
// % of the issue slots); DRAM is at a quarter.  One lane per polygon that follows
// precomputed successors runs as long as the longest of its warp's 32 polygons (21
// steps where the mean is 8.6) with scattered loads at every step, and the successors
// took a pass of their own.  gmm16-10m (20M triangles): 0.369 ms, against 0.188 ms for
// the successors and 0.338 ms for that walk; 1M uniform points 0.062 against 0.087 ms;
// the same with shuffled triangles 0.072 against 0.103; 200,000 mixture points 0.029
// against 0.038.  A lane (or two) per polygon on the tour itself took 0.58-0.65 ms.
// A warp whose regions do not fit the queue (0.3 %) leaves out those already too long
// for a walk, or takes half as many seeds at a time.
constexpr int kWalkWarps = kWalkThreads / 32;
constexpr int kWalkQ = 288;              // triangles of a warp's regions
constexpr int kWalkE = kWalkQ + 2 * 32;  // a region of T triangles has T + 2 boundary edges
constexpr int kWalkPasses = 64;          // one region of at most kWalkCap - 2 triangles fits
constexpr int kWalkLeast = 16;           // seeds a warp on a small mesh
constexpr int kGather = 5;               // loads in flight a lane in step 4
constexpr int kTipSlots = 48;            // tips of a warp's polygons (two on average)
constexpr unsigned kKidA = 0x400, kKidB = 0x800;  // link: children, below them (10 bits)
constexpr int kCorner = 12;  // the first child's queue index, above them the entry's corner
static_assert(kWalkQ + 64 < (int)kKidA && kWalkQ >= kWalkCap && 2 * kWalkQ >= kWalkE &&
                  kWalkPasses >= kWalkCap,
              "links hold queue indices, any one region fits, the vertices fit v");

struct WalkBuf {
  int he[kWalkE];  // boundary half-edges, polygon after polygon
  union {
    struct {
      int e[kWalkQ];                // the queue: entry half-edge of each triangle,
      unsigned short link[kWalkQ];  // its children and its corner,
      unsigned short cp[kWalkQ];    // its subtree's boundary edges, then its place
    } q;
    int v[kWalkE];  // step 4: origins of he
  } u;
  unsigned short p0[kWalkPasses];  // first queue index of each pass
  int tip_h[kTipSlots];  // tips (candidates, then -1 if none): half-edge,
  int tip_at[kTipSlots]; // polygon << 16 | place in the polygon
  // per polygon that is not empty, in lane order: its tips, its place (and length << 10),
  // its smallest vertex, where that is, its lane
  int nt[32], info[32], least[32], rank[32];
  unsigned char lane[32];
  unsigned starts[kWalkE / 32 + kGather];  // bit j: a polygon starts at place j
  int one[64], multi[64];        // polygons with one tip, with several, to be listed
  int tn;
};

// The warp's n buffered polygons appended to a list, one atomic for all; returns 0.
__device__ __forceinline__ int list_flush(const int* buf, int n, const LongList& D,
                                          long long* counter, Counters* C) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  unsigned long long at = 0;
  if (lane == 0)
    at = atomicAdd(reinterpret_cast<unsigned long long*>(counter), (unsigned long long)n);
  at = __shfl_sync(0xffffffffu, at, 0);
  if ((long long)at + n > D.cap) set_error(C, POLYLLA_ERR_LIMIT, 55);
  for (int k = lane; k < n; k += 32)
    if ((long long)at + k < D.cap) D.poly[at + k] = buf[k];
  __syncwarp();
  return 0;
}

__global__ void __launch_bounds__(kWalkThreads, 4) k_walk(DevMesh M, const int* __restrict__ tf,
                                                          const int* __restrict__ entry,
                                                          PolyArrays P, Pool pool, LongList Lg,
                                                          LongList D1, LongList Dm, int cap,
                                                          int repair, int tips_to_long,
                                                          Counters* C) {
  extern __shared__ __align__(16) unsigned char walk_smem[];
  pdl_wait();  // the tf words, seeds and entries
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned full = 0xffffffffu, lt = (1u << lane) - 1u;
  WalkBuf& B = reinterpret_cast<WalkBuf*>(walk_smem)[warp];
  const int* __restrict__ tri = M.tri;
  const int n = (int)C->n_seeds;  // below 2^29
  const int H = (int)(3 * M.m);
  // polygons with 2 to this many tips get tip records
  const int most_rec = tips_to_long > 0 ? min(tips_to_long - 1, kRsMaxSplit) : kRsMaxSplit;
  unsigned st_len = 0, st_tips = 0, st_tippolys = 0;
  // 32 seeds a warp and round, or fewer while that leaves no warp without any: on a
  // small mesh a warp's chain of passes is the kernel's time (200,000 mixture points, 60,204
  // seeds: 28.7 us against 39 with 32 seeds a warp)
  const int warps = (int)gridDim.x * kWalkWarps;
  int per = 32;
  while (per > kWalkLeast && n <= (per >> 1) * warps) per >>= 1;
  int width = per;  // seeds taken at a time
  int n1 = 0, nm = 0;  // entries of the warp's list buffers
  for (int base = ((int)blockIdx.x * kWalkWarps + warp) * per; base < n; base += warps * per) {
    const int i = base + lane;
    const int e0 = lane < per && i < n ? __ldg(entry + i) : -1;
    int x0 = e0 >= 0 ? __ldg(tf + e0) : -1;
    bool big = false;  // too long for a walk: left to a thread block
    for (int b0 = 0; b0 < per && base + b0 < n;) {
      const bool taken = e0 >= 0 && lane >= b0 && lane < b0 + width;
      if (taken && x0 >= H) {
        set_error(C, POLYLLA_ERR_LIMIT, 52);
        x0 = -1;
      }
      const bool mine = taken && !big;
      const bool inner = mine && x0 >= 0;  // the terminal edge has a far side
      const unsigned ma = __ballot_sync(full, mine), mb = __ballot_sync(full, inner);
      const int ra = __popc(ma & lt), rb = __popc(ma) + __popc(mb & lt);  // the roots
      int hi = __popc(ma) + __popc(mb);
      if (mine) B.u.q.e[ra] = e0;
      if (inner) B.u.q.e[rb] = x0;
      B.nt[lane] = 0;
      if (lane < kWalkE / 32 + kGather) B.starts[lane] = 0;
      if (lane == 0) B.tn = 0;
      __syncwarp();
      // ---- 1. the queue
      int np = 0, lo = 0;
      bool overflow = false;
      while (lo < hi) {
        if (lane == 0) B.p0[np] = (unsigned short)lo;
        const int x = lo + lane;
        int a = -1, b = -1, k = 0;
        if (x < hi) {
          const int e = B.u.q.e[x];
          k = (int)((unsigned)e % 3u);
          a = __ldg(tf + (k == 2 ? e - 2 : e + 1));
          b = __ldg(tf + (k == 0 ? e + 2 : e - 1));
          if (max(a, b) >= H) {
            set_error(C, POLYLLA_ERR_LIMIT, 52);
            a = b = -1;
          }
        }
        const unsigned da = __ballot_sync(full, a >= 0), db = __ballot_sync(full, b >= 0);
        const int ca = hi + __popc(da & lt) + __popc(db & lt);  // the first child
        const int cb = ca + (a >= 0);
        const int end = hi + __popc(da) + __popc(db);
        if (end > kWalkQ || np == kWalkPasses - 1) {
          overflow = true;
          break;
        }
        if (x < hi)
          B.u.q.link[x] = (unsigned short)(ca | (a >= 0 ? kKidA : 0) | (b >= 0 ? kKidB : 0) |
                                           k << kCorner);
        if (a >= 0) B.u.q.e[ca] = a;
        if (b >= 0) B.u.q.e[cb] = b;
        __syncwarp();
        lo = min(lo + 32, hi);
        hi = end;
        ++np;
      }
      if (overflow) {  // the triangles not followed count as leaves
        for (int x = lo + lane; x < hi; x += 32) B.u.q.cp[x] = 2;
        __syncwarp();
      }
      // ---- 2. boundary edges of every subtree
      for (int p = np - 1, end = overflow ? lo : hi; p >= 0; --p) {
        const int first = B.p0[p];
        const int x = first + lane;
        if (x < end) {
          const unsigned l = B.u.q.link[x];
          const unsigned ca = l & (kKidA - 1), cb = ca + (l & kKidA ? 1 : 0);
          int c = 2;
          if (l & kKidA) c += B.u.q.cp[ca] - 1;
          if (l & kKidB) c += B.u.q.cp[cb] - 1;
          B.u.q.cp[x] = (unsigned short)c;
        }
        end = first;
        __syncwarp();
      }
      // ---- the polygons' lengths and places
      const int na = mine ? B.u.q.cp[ra] : 0;
      int L = mine ? na + (inner ? B.u.q.cp[rb] : 1) : 0;
      const bool over = L > cap;
      big |= over;
      if (overflow) {
        if (!__any_sync(full, over)) {
          if (width == 1) big |= taken;  // (a single region that fits never gets here)
          else width >>= 1;
        }
        __syncwarp();
        continue;
      }
      if (over) L = 0;
      int first = L;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(full, first, d);
        if (lane >= d) first += y;
      }
      const int E = __shfl_sync(full, first, 31);
      first -= L;
      long long off = 0;
      if (lane == 0 && E > 0)
        off = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(&C->pool_alloc),
                                   (unsigned long long)E);
      if (mine) {
        B.u.q.cp[ra] = over ? 0xffff : (unsigned short)first;
        if (inner) B.u.q.cp[rb] = over ? 0xffff : (unsigned short)(first + na);
        else if (!over) B.he[first + na] = e0;
      }
      __syncwarp();
      // ---- 3. the boundary edges in order
      for (int p = 0; p < np; ++p) {
        const int x = B.p0[p] + lane;
        if (x < (p + 1 < np ? (int)B.p0[p + 1] : hi)) {
          const unsigned l = B.u.q.link[x];
          const unsigned ca = l & (kKidA - 1), cb = ca + (l & kKidA ? 1 : 0), k = l >> kCorner;
          const int at = B.u.q.cp[x];
          const int e = B.u.q.e[x];
          int bt = at;
          if (at != 0xffff) {
            if (l & kKidA) bt += B.u.q.cp[ca];
            else B.he[bt++] = k == 2 ? e - 2 : e + 1;
            if (!(l & kKidB)) B.he[bt] = k == 0 ? e + 2 : e - 1;
          }
          if (l & kKidA) B.u.q.cp[ca] = (unsigned short)at;
          if (l & kKidB) B.u.q.cp[cb] = (unsigned short)bt;
        }
        __syncwarp();
      }
      // ---- 4. the vertices.  The polygon of place j is the number of polygons that
      //         start at or before it (starts: a bit per place)
      const unsigned some = __ballot_sync(full, L > 0);
      const int ord = __popc(some & lt);
      if (L) {
        B.info[ord] = first | L << 10;
        B.least[ord] = 0x7fffffff;
        B.rank[ord] = 0;
        atomicOr(&B.starts[first >> 5], 1u << (first & 31));
      }
      __syncwarp();
      const unsigned upto = lt << 1 | 1u;
      for (int j0 = 0, poly = -1; j0 < E; j0 += 32 * kGather) {
        int o[kGather];
#pragma unroll
        for (int w = 0; w < kGather; ++w) {
          const int j = j0 + 32 * w + lane;
          if (j < E) o[w] = __ldg(tri + B.he[j]);
        }
#pragma unroll
        for (int w = 0; w < kGather; ++w) {
          const int j = j0 + 32 * w + lane;
          const unsigned starts = B.starts[(j0 >> 5) + w];
          if (j < E) {
            B.u.v[j] = o[w];
            atomicMin(&B.least[poly + __popc(starts & upto)], o[w]);
          }
          poly += __popc(starts);
        }
      }
      __syncwarp();
      // where each polygon's smallest vertex is (count << 16 | place in the polygon),
      // and where a vertex repeats two steps on: a tip a, b, a if its half-edge a->b is
      // followed by its twin
#pragma unroll 1
      for (int j0 = 0, poly = -1; j0 < E; j0 += 32) {
        const unsigned starts = B.starts[j0 >> 5];
        const int j = j0 + lane;
        if (j < E) {
          const int s = poly + __popc(starts & upto);
          const int inf = B.info[s];
          const int p0 = inf & 1023, l = inf >> 10;
          const int v = B.u.v[j];
          int j2 = j + 2;
          if (j2 >= p0 + l) j2 -= l;
          if (v == B.least[s]) atomicAdd(&B.rank[s], 0x10000 + j - p0);
          if (v == B.u.v[j2]) {
            const int k = atomicAdd(&B.tn, 1);
            if (k < kTipSlots) B.tip_at[k] = s << 16 | (j - p0);
          }
        }
        poly += __popc(starts);
      }
      __syncwarp();
      int rank = L ? B.rank[ord] : 0;
      if (rank >> 16 > 1) {  // it repeats: the smallest half-edge
        const int least = B.least[ord];
        int h = 0x7fffffff;
        for (int q = 0; q < L; ++q)
          if (B.u.v[first + q] == least && B.he[first + q] < h) {
            h = B.he[first + q];
            rank = q;
          }
      }
      rank &= 0xffff;
      const int tn = B.tn;
      const int start = L ? B.he[first + rank] : 0;
      for (int t0 = 0; t0 < min(tn, kTipSlots); t0 += 32) {
        const int t = t0 + lane;
        const bool live = t < min(tn, kTipSlots);
        if (live) {
          const int at = B.tip_at[t], inf = B.info[at >> 16];
          const int q = at & 0xffff, p0 = inf & 1023, l = inf >> 10;
          const int h = B.he[p0 + q];
          const bool tip = tf_twin(__ldg(tf + h)) == B.he[p0 + (q + 1 < l ? q + 1 : 0)];
          B.tip_h[t] = tip ? h : -1;
          if (tip) atomicAdd(&B.nt[at >> 16], 1);
        }
      }
      __syncwarp();
      // the lists of polygons to split, kept in the warp's buffers until one is half full
      const int ntips = L ? B.nt[ord] : 0;
      // several tips on a small mesh: the block kernel splits them in parallel; it
      // also takes the polygons of a warp whose tip list is full
      const bool many =
          L && (tn > kTipSlots || (repair && tips_to_long > 0 && ntips >= tips_to_long));
      const bool is_long = taken && (big || many);
      const bool split = repair && ntips > 0 && !many;
      const bool rec = split && ntips >= 2 && ntips <= most_rec;
      const unsigned m1 = __ballot_sync(full, split && ntips == 1);
      const unsigned mm = __ballot_sync(full, split && ntips > 1);
      if (split) {
        if (ntips == 1) B.one[n1 + __popc(m1 & lt)] = i;
        else B.multi[nm + __popc(mm & lt)] = i;
      }
      n1 += __popc(m1);
      nm += __popc(mm);
      // to the pool, each polygon turned to its canonical start: the polygon of an
      // edge is the number of polygons that start at or before it
      if (L) {
        B.rank[ord] = rank;
        B.lane[ord] = (unsigned char)lane;
      }
      __syncwarp();
      off = __shfl_sync(full, off, 0);
      const bool fits = off + E <= pool.cap;
      if (!fits && lane == 0) set_error(C, POLYLLA_ERR_LIMIT, 53);
      if (fits) {
        int* out = pool.v + off;
#pragma unroll 1
        for (int j0 = 0, poly = -1; j0 < E; j0 += 32) {
          const unsigned starts = B.starts[j0 >> 5];
          const int j = j0 + lane;
          if (j < E) {
            const int s = poly + __popc(starts & upto);
            const int inf = B.info[s];
            int at = j - B.rank[s];
            if (at < (inf & 1023)) at += inf >> 10;
            out[at] = B.u.v[j];
          }
          poly += __popc(starts);
        }
      }
      // ---- records and lists
      long long roff = off + first;
      if (__any_sync(full, rec)) {
        // several tips: the sequence and the records (rotated tip index, tip
        // half-edge) get space of their own, which the pieces overwrite
        const long long o = warp_alloc(&C->pool_alloc, rec ? L + 2 * ntips : 0);
        if (rec) roff = o;
      }
      // an entry of a list whose sequence is not in the pool is one of length 0,
      // which the split kernels skip
      const bool kept = fits && (!rec || roff + L + 2 * ntips <= pool.cap);
      if (rec && !kept) set_error(C, POLYLLA_ERR_LIMIT, 53);
      for (unsigned left = __ballot_sync(full, rec && kept); left; left &= left - 1) {
        const int s = __ffs(left) - 1;
        const int p0 = __shfl_sync(full, first, s), l = __shfl_sync(full, L, s);
        const int pr = __shfl_sync(full, rank, s);
        const long long po = __shfl_sync(full, roff, s);
        for (int q = lane; q < l; q += 32)
          pool.v[po + (q >= pr ? q - pr : q - pr + l)] = B.u.v[p0 + q];
      }
      if (repair) {
        for (int t0 = 0; t0 < min(tn, kTipSlots); t0 += 32) {
          const int t = t0 + lane;
          const bool live = t < min(tn, kTipSlots) && B.tip_h[t] >= 0;
          const int at = live ? B.tip_at[t] : 0;
          const int s = at >> 16, owner = live ? B.lane[s] : 0;
          const long long po = __shfl_sync(full, roff, owner);
          const int how = __shfl_sync(full, (int)(split && kept) | (int)rec << 1, owner);
          if (live && (how & 1)) {
            const int inf = B.info[s], pr = B.rank[s];
            const int p0 = inf & 1023, l = inf >> 10;
            const int q = at & 0xffff;
            const int b = B.u.v[p0 + (q + 1 < l ? q + 1 : 0)];  // the tip vertex
            int order = 0;
            bool lowest = true;
            const bool one = B.nt[s] == 1;
            for (int k = 0; k < min(tn, kTipSlots) && !one; ++k) {
              if (B.tip_at[k] >> 16 != s || B.tip_h[k] < 0) continue;
              const int qk = B.tip_at[k] & 0xffff;
              order += k < t;
              lowest &= B.u.v[p0 + (qk + 1 < l ? qk + 1 : 0)] >= b;
            }
            const int rot = q >= pr ? q - pr : q - pr + l;
            const int ip = base + owner;
            if (how & 2) {
              pool.v[po + l + 2 * order] = rot;
              pool.v[po + l + 2 * order + 1] = B.tip_h[t];
            }
            if (lowest) {
              P.tip_h[ip] = B.tip_h[t];
              if (one) P.pbase[ip] = rot;  // the tip's index in the sequence
            }
          }
        }
      }
      if (taken) {
        P.pcnt[i] = 0;
        P.flen[i] = split || is_long || !fits ? 0 : L;
        if (is_long) {
          const long long d =
              (long long)atomicAdd(reinterpret_cast<unsigned long long*>(&C->n_long), 1ull);
          if (d < Lg.cap) Lg.poly[d] = i;
        } else {
          P.pos[i] = roff;
          st_len += L;
          st_tips += ntips;
          st_tippolys += ntips > 0;
        }
        if (split) {
          P.start[i] = start;
          P.len[i] = kept ? L : 0;
          P.ntip[i] = ntips;
          if (ntips > 1) P.pbase[i] = rec ? 1 : 0;  // several tips: records at pos, or none
        }
      }
      __syncwarp();
      if (n1 > 32) n1 = list_flush(B.one, n1, D1, &C->n_defer, C);
      if (nm > 32) nm = list_flush(B.multi, nm, Dm, &C->n_multi, C);
      b0 += width;
    }
    width = min(per, 2 * width);
  }
  if (n1) list_flush(B.one, n1, D1, &C->n_defer, C);
  if (nm) list_flush(B.multi, nm, Dm, &C->n_multi, C);
  st_len = __reduce_add_sync(0xffffffffu, st_len);
  st_tips = __reduce_add_sync(0xffffffffu, st_tips);
  st_tippolys = __reduce_add_sync(0xffffffffu, st_tippolys);
  if ((threadIdx.x & 31) == 0) {
    if (st_len) atomicAdd(reinterpret_cast<unsigned long long*>(&C->n_vtx_trav), (unsigned long long)st_len);
    if (st_tips) atomicAdd(reinterpret_cast<unsigned long long*>(&C->n_tips), (unsigned long long)st_tips);
    if (st_tippolys)
      atomicAdd(reinterpret_cast<unsigned long long*>(&C->n_tip_polys), (unsigned long long)st_tippolys);
  }
}

cudaError_t launch_walk(const DevMesh& M, const int* tf, const int* entry, const PolyArrays& P,
                        const Pool& pool, const LongList& Lg, const LongList& D1,
                        const LongList& Dm, int cap, int repair, int tips_to_long, Counters* C,
                        int grid, cudaStream_t s, bool pdl) {
  if (cap < 16 || cap > kWalkCap || cap % 16) return cudaErrorInvalidValue;
  constexpr size_t smem = sizeof(WalkBuf) * kWalkWarps;
  static std::atomic<bool> attr[kMaxDevices];
  const cudaError_t e = smem_limit_once(reinterpret_cast<const void*>(k_walk), (int)smem, attr);
  if (e != cudaSuccess) return e;
  static std::atomic<int> resident{0};
  grid = resident_grid(reinterpret_cast<const void*>(k_walk), kWalkThreads, smem, grid, &resident);
  return launch_chain(k_walk, grid, kWalkThreads, smem, s, pdl, M, tf, entry, P, pool, Lg, D1, Dm,
                      cap, repair, tips_to_long, C);
}

__device__ __forceinline__ unsigned long long vkey(int origin, int h) {
  return ((unsigned long long)(unsigned)origin << 32) | (unsigned)h;
}

constexpr int kSeqChunk = 4;  // sequence entries loaded at a time by the split kernels

// One tip p = a->b, split along oj = b->x (tw = x->b), with q = turn(oj) and
// pn = twin(p) = b->a.  The two pieces are
//     oj, q, turn(q), ..., p          and          tw, pn, turn(pn), ..., pred(q)
// (the boundary walk with oj, tw frontier); the other frontier half-edges keep
// their turns.  The walk left the polygon's vertex sequence v (from its canonical
// start) in the pool and the tip's index t in it (v[t] = a, v[t+1] = b).  When x
// occurs once in v, at u, q is the half-edge leaving x there, and the pieces are
//     b, v[u], ..., v[t]          and          x, v[t+1], ..., v[u-1]
// (indices cyclic); each is written from its smallest vertex when that vertex
// occurs once in it (then it is the canonical start).  Otherwise (x, or a piece's
// smallest vertex, repeated: the canonical start needs half-edge ids) the two arcs
// of the cycle are walked by turning, staged over v (arc 1 from the front, arc 2
// from the back), and each piece is copied from its canonical start.
// Pool space: L + 2 for the pieces.
__global__ void __launch_bounds__(kBlock) k_repair_one(DevMesh M, uint8_t* lab, int* tf,
                                                       PolyArrays P, FinalPieces F, Pool pool,
                                                       LongList D1, int rare, Counters* C) {
  pdl_wait();  // the walk's lists, records and sequences
  const long long nd = min(C->n_defer, D1.cap);
  const int H = (int)(3 * M.m);
  const long long limit = 3 * M.m + 3;
  unsigned st_bad = 0, st_chase = 0;
  for (long long base = (long long)blockIdx.x * blockDim.x; base < nd;
       base += (long long)gridDim.x * blockDim.x) {
    const long long d = base + threadIdx.x;
    const long long i = (d < nd) ? D1.poly[d] : -1;
    const int L = (i >= 0) ? P.len[i] : 0;
    const long long off = warp_alloc(&C->pool_alloc, i >= 0 ? L + 2 : 0);
    const long long foff = warp_alloc(&C->fslot_alloc, i >= 0 ? 2 : 0);
    if (i < 0) continue;
    if (off + L + 2 > pool.cap || foff + 2 > F.cap || L < 3) {
      set_error(C, POLYLLA_ERR_LIMIT, 56);
      continue;
    }
    const int tp = P.tip_h[i];
    const int t = P.pbase[i];
    const long long vpos = P.pos[i];
    if ((unsigned)tp >= (unsigned)H || (unsigned)t >= (unsigned)L || vpos < 0 ||
        vpos + L > pool.cap) {
      set_error(C, POLYLLA_ERR_LIMIT, 57);
      continue;
    }
    int* v = pool.v + vpos;
    const int pn = tf_twin(tf[tp]);
    const int b = M.tri[he_next(tp)];
    const int oj = split_edge(tf, tp, H);
    if (oj < 0 || pn >= H) {
      set_error(C, POLYLLA_ERR_LIMIT, 54);
      continue;
    }
    const int tw = tf_twin(tf[oj]);
    const int x = M.tri[he_next(oj)];
    if (tw >= H) {
      set_error(C, POLYLLA_ERR_LIMIT, 54);
      continue;
    }
    set_frontier(lab, tf, oj);
    set_frontier(lab, tf, tw);
    int* out = pool.v + off;
    // the passes over the sequence load kSeqChunk entries at a time, so that
    // their latencies overlap
    int u = -1, nx = 0;
    for (int q0 = 0; q0 < L; q0 += kSeqChunk) {
      int w[kSeqChunk];
#pragma unroll
      for (int k = 0; k < kSeqChunk; ++k) w[k] = (q0 + k < L) ? v[q0 + k] : -1;
#pragma unroll
      for (int k = 0; k < kSeqChunk; ++k) {
        if (w[k] == x) {
          u = q0 + k;
          ++nx;
        }
      }
    }
    bool fast = nx == 1 && !rare;
    int l1 = 0, l2 = 0, r1 = 0, r2 = 0;
    if (fast) {
      const int n1 = (t >= u ? t - u : t - u + L) + 1;  // v[u..t]
      l1 = n1 + 1;
      l2 = L - n1 + 1;
      int m1 = b, c1 = 1, m2 = x, c2 = 1;
      for (int j0 = 0; j0 < L; j0 += kSeqChunk) {  // v[u + j], j = 0..L-1
        int w[kSeqChunk];
#pragma unroll
        for (int k = 0; k < kSeqChunk; ++k) {
          int q = u + j0 + k;
          if (q >= L) q -= L;
          w[k] = (j0 + k < L) ? v[q] : 0;
        }
#pragma unroll
        for (int k = 0; k < kSeqChunk; ++k) {
          const int j = j0 + k, o = w[k];
          if (j >= L) break;
          if (j < n1) {
            if (o < m1) {
              m1 = o;
              c1 = 1;
              r1 = 1 + j;
            } else if (o == m1) {
              ++c1;
            }
          } else if (o < m2) {
            m2 = o;
            c2 = 1;
            r2 = 1 + j - n1;
          } else if (o == m2) {
            ++c2;
          }
        }
      }
      fast = c1 == 1 && c2 == 1;
      if (fast) {
        // piece 1: index k >= 1 is v[u + k - 1]; piece 2: index k >= 1 is v[t + k]
        for (int q0 = 0; q0 < l1 + l2; q0 += kSeqChunk) {
          int w[kSeqChunk];
#pragma unroll
          for (int c = 0; c < kSeqChunk; ++c) {
            const int q = q0 + c;
            int val = 0;
            if (q < l1) {
              int k = r1 + q;
              if (k >= l1) k -= l1;
              int z = u + k - 1;
              if (z >= L) z -= L;
              val = k ? v[z] : b;
            } else if (q < l1 + l2) {
              int k = r2 + (q - l1);
              if (k >= l2) k -= l2;
              int z = t + k;
              if (z >= L) z -= L;
              val = k ? v[z] : x;
            }
            w[c] = val;
          }
#pragma unroll
          for (int c = 0; c < kSeqChunk; ++c)
            if (q0 + c < l1 + l2) out[q0 + c] = w[c];
        }
      }
    }
    if (!fast) {
      ++st_chase;
      long long steps = 0;
      const int g = turn_tf(tf, oj, H, steps, limit);
      if (g < 0 || g == tw || g == pn) {
        set_error(C, POLYLLA_ERR_LIMIT, 54);
        continue;
      }
      int* stage = v;  // the sequence is not read again
      int c1 = g, c2 = pn, n1 = 0, n2 = 0;
      bool a1 = true, a2 = true;
      unsigned long long b1 = vkey(b, oj), b2 = vkey(x, tw);
      for (int it = 0; (a1 || a2) && it < L; ++it) {
        if (a1) {
          const int o1 = M.tri[c1];
          stage[n1] = o1;
          const unsigned long long k = vkey(o1, c1);
          ++n1;
          if (k < b1) {
            b1 = k;
            r1 = n1;
          }
          if (c1 == tp) a1 = false;
          else c1 = turn_tf(tf, c1, H, steps, limit);
        }
        if (a2) {
          const int o2 = M.tri[c2];
          ++n2;
          stage[L - n2] = o2;
          const unsigned long long k = vkey(o2, c2);
          if (k < b2) {
            b2 = k;
            r2 = n2;
          }
          c2 = turn_tf(tf, c2, H, steps, limit);
          if (c2 == tw) a2 = false;
        }
        if (c1 < 0 || c2 < 0) break;
      }
      if (a1 || a2 || n1 + n2 != L) {
        ++st_bad;
        continue;
      }
      // piece 1 = [b, stage[0..n1)], piece 2 = [x, stage[L-1], ..., stage[L-n2]]
      l1 = n1 + 1;
      l2 = n2 + 1;
      int k = r1;
      for (int q = 0; q < l1; ++q) {
        out[q] = k ? stage[k - 1] : b;
        if (++k == l1) k = 0;
      }
      k = r2;
      for (int q = 0; q < l2; ++q) {
        out[l1 + q] = k ? stage[L - k] : x;
        if (++k == l2) k = 0;
      }
    }
    F.pos[foff] = off;
    F.len[foff] = l1;
    F.pos[foff + 1] = off + l1;
    F.len[foff + 1] = l2;
    P.pcnt[i] = 2;
    P.pbase[i] = (int)foff;
    P.flen[i] = L + 2;
  }
  if (st_bad) set_error(C, POLYLLA_ERR_LIMIT, 58);
  st_chase = __reduce_add_sync(0xffffffffu, st_chase);
  if ((threadIdx.x & 31) == 0 && st_chase)
    atomicAdd(reinterpret_cast<unsigned long long*>(&C->n_one_chase), (unsigned long long)st_chase);
  // one split per polygon of this list
  if (blockIdx.x == 0 && threadIdx.x == 0 && nd > 0)
    atomicAdd(reinterpret_cast<unsigned long long*>(&C->n_splits), (unsigned long long)nd);
}

// Linked-list reparation of one polygon with several tips per thread.
//
// Nodes 0..L-1 are the polygon's frontier half-edges in boundary order from its
// canonical start (bit 31 set on a barrier-edge tip a->b, i.e. the node followed
// by twin(a->b)); nodes kWalkCap.. are chord half-edges added by splits.  Each
// node keeps its half-edge, its origin vertex and next/prev links, all in shared
// memory, transposed ([node][thread]) so that lanes at the same step hit distinct
// banks.  The pieces form an ordered list of start nodes, as in repair_seq: the
// first piece with a tip is split at its smallest tip b (the destination of tip
// node p) along oj = split_edge(), and is replaced by the piece from oj (b->x)
// followed by the piece from tw = twin(oj) (x->b).  With q the node of turn(oj)
// -- the first frontier half-edge after oj around x -- and qp its predecessor:
//     p -> oj -> q   and   qp -> tw -> next(p),
// which is the boundary that walking the region with the new frontier edge gives.
// A split removes the tip at p, and the one at qp if x was a tip, and creates
// none (x always has a frontier edge of the region besides the chord), so only
// those two flags change.
//
// The node list comes from the walk's records (the origins from the canonical
// start, and each tip's index and half-edge): the other nodes' half-edges stay
// unknown (kSuccMask) unless needed.  q is the piece's
// only node with origin x; when x occurs more than once in the piece, q is the
// one whose successor's origin is dest(turn(oj)) (a directed edge occurs once in
// a boundary).  A finished piece starts at its smallest vertex; when that vertex
// occurs more than once, the piece's half-edges are found by turning from a node
// whose half-edge is known (a chord), and the smallest (origin, half-edge) key
// decides.  The pieces are written over the records (as long as the polygon and
// its tip records, at least its final length).
constexpr int kRsThreads = 64;
constexpr int kRsNodes = kWalkCap + 2 * kRsMaxSplit;
constexpr int kRsList = kRsMaxSplit + 2;
constexpr size_t kRsSmem =
    (size_t)kRsThreads * (kRsNodes * (2 * sizeof(int) + 2) + kRsList);

__global__ void __launch_bounds__(kRsThreads) k_repair_multi(DevMesh M, uint8_t* lab, int* tf,
                                                             PolyArrays P, FinalPieces F,
                                                             Pool pool, LongList Dm, int rare,
                                                             Counters* C) {
  extern __shared__ int rs_smem[];
  int* nh = rs_smem;                                   // [kRsNodes][kRsThreads]
  int* no = nh + kRsNodes * kRsThreads;                // origins
  uint8_t* nx = reinterpret_cast<uint8_t*>(no + kRsNodes * kRsThreads);
  uint8_t* pv = nx + kRsNodes * kRsThreads;
  uint8_t* ps = pv + kRsNodes * kRsThreads;            // [kRsList][kRsThreads]
  const int t = threadIdx.x;
#define NH(j) nh[(j) * kRsThreads + t]
#define NO(j) no[(j) * kRsThreads + t]
#define NX(j) nx[(j) * kRsThreads + t]
#define PV(j) pv[(j) * kRsThreads + t]
#define PS(j) ps[(j) * kRsThreads + t]
  const long long nd = min(C->n_multi, Dm.cap);
  const int H = (int)(3 * M.m);
  const long long limit = 3 * M.m + 3;
  unsigned st_splits = 0, st_seq = 0, st_turn = 0;
  for (long long base = (long long)blockIdx.x * blockDim.x; base < nd;
       base += (long long)gridDim.x * blockDim.x) {
    const long long d = base + t;
    const long long i = (d < nd) ? Dm.poly[d] : -1;
    const int L = (i >= 0) ? P.len[i] : 0;
    const int nt = (i >= 0) ? P.ntip[i] : 0;
    const bool listed = nt <= kRsMaxSplit && L <= kWalkCap;
    const bool rec = i >= 0 && listed && nt >= 2 && L >= 3 && P.pbase[i] == 1;
    const long long off0 = warp_alloc(&C->pool_alloc, i >= 0 && !rec ? L + 2 * nt : 0);
    const long long foff = warp_alloc(&C->fslot_alloc, i >= 0 ? nt + 1 : 0);
    if (i < 0) continue;
    const long long off = rec ? P.pos[i] : off0;
    if (L < 3 || off < 0 || off + L + 2 * nt > pool.cap || foff + nt + 1 > F.cap) {
      set_error(C, POLYLLA_ERR_LIMIT, 56);
      continue;
    }
    int cnt;
    if (!listed) {
      ++st_seq;
      const Cyc first{P.start[i], L, P.tip_h[i], nt, true};
      cnt = repair_seq(M.tri, tf, lab, first, nt + 1, H, limit, F.h + foff, F.pos + foff,
                       F.len + foff, pool.v + off, off, L + 2 * nt);
    } else {
      cnt = -1;
      bool bad = false;
      if (!rec) {
        bad = true;  // the walk leaves records for every such polygon
      } else {
        const int* rv = pool.v + off;
        for (int j0 = 0; j0 < L; j0 += kSeqChunk) {
          int w[kSeqChunk];
#pragma unroll
          for (int k = 0; k < kSeqChunk; ++k) w[k] = (j0 + k < L) ? rv[j0 + k] : 0;
#pragma unroll
          for (int k = 0; k < kSeqChunk; ++k) {
            const int j = j0 + k;
            if (j >= L) break;
            NH(j) = kSuccMask;
            NO(j) = w[k];
            NX(j) = (uint8_t)(j + 1 == L ? 0 : j + 1);
            PV(j) = (uint8_t)(j == 0 ? L - 1 : j - 1);
          }
        }
        for (int k = 0; k < nt; ++k) {
          const int ix = rv[L + 2 * k], hh = rv[L + 2 * k + 1];
          if ((unsigned)ix >= (unsigned)L || (unsigned)hh >= (unsigned)H) {
            bad = true;
            break;
          }
          NH(ix) = hh | kTipFlag;
        }
      }
      int nn = kWalkCap;  // next chord node
      int count = 1;
      PS(0) = 0;
      long long acc = 0;
      int j = 0;
      while (!bad && j < count) {
        const int s0 = PS(j);
        // the piece: its smallest tip, its smallest vertex and how often it occurs
        int tb = 0x7fffffff, tipn = -1, mo = 0x7fffffff, mn = s0, mc = 0, len = 0;
        int v = s0;
        do {
          const int x = NH(v);
          const int nv = NX(v);
          if (x < 0) {
            const int b = NO(nv);
            if (b < tb) {
              tb = b;
              tipn = v;
            }
          }
          const int o = NO(v);
          if (o < mo) {
            mo = o;
            mn = v;
            mc = 1;
          } else if (o == mo) {
            ++mc;
          }
          ++len;
          v = nv;
        } while (v != s0 && len <= kRsNodes);
        if (len > kRsNodes) {
          bad = true;
          break;
        }
        if (tipn < 0) {  // finished piece: its origins from the canonical start
          if (mc > 1 || rare) {  // the smallest vertex repeats: compare (origin, half-edge)
            ++st_turn;
            int c0 = -1;
            v = s0;
            for (int k = 0; k < len && c0 < 0; ++k, v = NX(v))
              if ((NH(v) & kSuccMask) != kSuccMask) c0 = v;
            if (c0 < 0) {
              bad = true;
              break;
            }
            v = c0;
            for (int k = 0; k + 1 < len && !bad; ++k) {  // unknown half-edges by turning
              const int nv = NX(v);
              if ((NH(nv) & kSuccMask) == kSuccMask) {
                long long steps = 0;
                const int g = turn_tf(tf, NH(v) & kSuccMask, H, steps, limit);
                if (g < 0) bad = true;
                else NH(nv) = g;
              }
              v = nv;
            }
            if (bad) break;
            unsigned long long best = ~0ull;
            v = s0;
            for (int k = 0; k < len; ++k, v = NX(v)) {
              const unsigned long long key = vkey(NO(v), NH(v) & kSuccMask);
              if (key < best) {
                best = key;
                mn = v;
              }
            }
          }
          int* out = pool.v + off + acc;
          v = mn;
          for (int k = 0; k < len; ++k) {
            out[k] = NO(v);
            v = NX(v);
          }
          F.pos[foff + j] = off + acc;
          F.len[foff + j] = len;
          acc += len;
          ++j;
          continue;
        }
        if (count + 1 > nt + 1 || nn + 2 > kRsNodes) {
          bad = true;
          break;
        }
        const int oj = split_edge(tf, NH(tipn) & kSuccMask, H);
        if (oj < 0) {
          bad = true;
          break;
        }
        const int tw = tf_twin(tf[oj]);
        if (tw >= H) {
          bad = true;
          break;
        }
        set_frontier(lab, tf, oj);
        set_frontier(lab, tf, tw);
        const int x = M.tri[tw];  // origin of tw = dest(oj)
        // q: the piece's node leaving x at turn(oj)
        int q = -1, nq = 0;
        v = s0;
        for (int k = 0; k < len; ++k, v = NX(v)) {
          if (NO(v) == x) {
            q = v;
            ++nq;
          }
        }
        if (nq != 1 || rare) {  // x repeats: the node whose edge is x -> dest(turn(oj))
          long long steps = 0;
          const int g = turn_tf(tf, oj, H, steps, limit);
          if (g < 0 || g == tw) {
            bad = true;
            break;
          }
          const int y = M.tri[he_next(g)];
          q = -1;
          v = s0;
          for (int k = 0; k < len; ++k, v = NX(v))
            if (NO(v) == x && NO(NX(v)) == y) q = v;
          if (q < 0) {
            bad = true;
            break;
          }
          if ((NH(q) & kSuccMask) == kSuccMask) NH(q) = g;
        }
        const int qp = PV(q);
        const int pn = NX(tipn);
        const int u = nn, w = nn + 1;
        nn += 2;
        NH(u) = oj;
        NO(u) = tb;
        NH(w) = tw;
        NO(w) = x;
        NX(tipn) = (uint8_t)u;
        PV(u) = (uint8_t)tipn;
        NX(u) = (uint8_t)q;
        PV(q) = (uint8_t)u;
        NX(qp) = (uint8_t)w;
        PV(w) = (uint8_t)qp;
        NX(w) = (uint8_t)pn;
        PV(pn) = (uint8_t)w;
        NH(tipn) &= kSuccMask;
        NH(qp) &= kSuccMask;
        for (int k = count; k > j + 1; --k) PS(k) = PS(k - 1);
        PS(j) = (uint8_t)u;
        PS(j + 1) = (uint8_t)w;
        ++count;
      }
      if (!bad) cnt = count;
    }
#undef NH
#undef NO
#undef NX
#undef PV
#undef PS
    if (cnt < 0) {
      set_error(C, POLYLLA_ERR_LIMIT, 54);
      continue;
    }
    P.pcnt[i] = cnt;
    P.pbase[i] = (int)foff;
    P.flen[i] = L + 2 * (cnt - 1);
    st_splits += cnt - 1;
  }
  st_splits = __reduce_add_sync(0xffffffffu, st_splits);
  st_seq = __reduce_add_sync(0xffffffffu, st_seq);
  if ((threadIdx.x & 31) == 0 && st_splits)
    atomicAdd(reinterpret_cast<unsigned long long*>(&C->n_splits), (unsigned long long)st_splits);
  if ((threadIdx.x & 31) == 0 && st_seq)
    atomicAdd(reinterpret_cast<unsigned long long*>(&C->n_multi_seq), (unsigned long long)st_seq);
  st_turn = __reduce_add_sync(0xffffffffu, st_turn);
  if ((threadIdx.x & 31) == 0 && st_turn)
    atomicAdd(reinterpret_cast<unsigned long long*>(&C->n_multi_turn), (unsigned long long)st_turn);
}

cudaError_t launch_repair_one(const DevMesh& M, uint8_t* lab, int* tf, const PolyArrays& P,
                              const FinalPieces& F, const Pool& pool,
                              const LongList& D1, int rare, Counters* C, int sms,
                              cudaStream_t s, bool pdl) {
  static std::atomic<int> cap{0};
  const int grid = resident_grid(reinterpret_cast<const void*>(k_repair_one), kBlock, 0,
                                 (long long)sms * 8, &cap);
  return launch_chain(k_repair_one, grid, kBlock, 0, s, pdl, M, lab, tf, P, F, pool, D1, rare, C);
}

cudaError_t launch_repair_multi(const DevMesh& M, uint8_t* lab, int* tf, const PolyArrays& P,
                                const FinalPieces& F, const Pool& pool,
                                const LongList& Dm, int rare, Counters* C, int sms,
                                cudaStream_t s) {
  static std::atomic<bool> attr[kMaxDevices];
  const cudaError_t e =
      smem_limit_once(reinterpret_cast<const void*>(k_repair_multi), (int)kRsSmem, attr);
  if (e != cudaSuccess) return e;
  const int per_sm = (int)((220 * 1024) / (kRsSmem + 1024));
  const int grid = sms * (per_sm < 1 ? 1 : per_sm);
  k_repair_multi<<<grid, kRsThreads, kRsSmem, s>>>(M, lab, tf, P, F, pool, Dm, rare, C);
  return cudaGetLastError();
}

}  // namespace polylla
