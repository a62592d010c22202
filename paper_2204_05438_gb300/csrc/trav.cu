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
//           left to one thread block (long.cu), and a seed listed by the seed pass,
//           whose region may be long, to a block that runs beside the walk.
//   k_repair_one    one thread per polygon with one tip: split it and cut the
//           two pieces out of the vertex sequence the walk left in the pool.
//   k_repair_multi  one warp per polygon with several tips: all split edges at once,
//           then the pieces as the cycles of the new successors.
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
//   4. the origins gathered, a lane per boundary edge, and compared in shared memory:
//      each polygon's smallest vertex and where it is (the half-edges only if it
//      repeats), and the vertices that repeat two steps on, which tips do; then every
//      lane stores its edges' origins, each polygon turned to start at its smallest,
//      in one stretch of the pool.
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
                                                          int beside, Counters* C) {
  extern __shared__ __align__(16) unsigned char walk_smem[];
  pdl_wait();  // the tf words, seeds and entries
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned full = 0xffffffffu, lt = (1u << lane) - 1u;
  WalkBuf& B = reinterpret_cast<WalkBuf*>(walk_smem)[warp];
  const int* __restrict__ tri = M.tri;
  const int n = (int)C->n_seeds;  // below 2^29
  const int H = (int)(3 * M.m);
  const bool early0 = beside && C->n_early[0] <= kEarlyMost,
             early1 = beside && C->n_early[1] <= kEarlyMost;
  // polygons with 2 to this many tips leave their half-edges to the several-tip kernel
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
    const bool any = lane < per && i < n;
    const int raw = any ? __ldg(entry + i) : 0;
    int e0 = any ? raw & ~(int)kEarlyBit : -1;
    if (e0 >= H) {  // (no seed pass writes one)
      set_error(C, POLYLLA_ERR_LIMIT, 51);
      e0 = -1;
    }
    // A listed seed of a kind the blocks have is theirs.  The kind comes from the twin array,
    // which nothing writes: the blocks mark split edges in tf at the same time, and one may be
    // a listed region's own terminal edge, whose word then looks like a border's.
    if (raw < 0 && e0 >= 0) {
      const int g = __ldg(M.twin + e0);  // (out of range: a border's, to the label pass)
      if (g < 0 || g >= H ? early0 : early1) e0 = -1;
    }
    int x0 = e0 >= 0 ? __ldg(tf + e0) : -1;  // (of regions that only the walk has)
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
        // several tips: the half-edges get space of their own, which the pieces
        // overwrite
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
          pool.v[po + (q >= pr ? q - pr : q - pr + l)] = B.he[p0 + q];
      }
      if (repair) {
        for (int t0 = 0; t0 < min(tn, kTipSlots); t0 += 32) {
          const int t = t0 + lane;
          const bool live = t < min(tn, kTipSlots) && B.tip_h[t] >= 0;
          const int at = live ? B.tip_at[t] : 0;
          const int s = at >> 16, owner = live ? B.lane[s] : 0;
          const bool listed = __shfl_sync(full, (int)(split && kept), owner) != 0;
          if (live && listed) {
            const int inf = B.info[s], pr = B.rank[s];
            const int p0 = inf & 1023, l = inf >> 10;
            const int q = at & 0xffff;
            const int b = B.u.v[p0 + (q + 1 < l ? q + 1 : 0)];  // the tip vertex
            bool lowest = true;
            const bool one = B.nt[s] == 1;
            for (int k = 0; k < min(tn, kTipSlots) && !one; ++k) {
              if (B.tip_at[k] >> 16 != s || B.tip_h[k] < 0) continue;
              const int qk = B.tip_at[k] & 0xffff;
              lowest &= B.u.v[p0 + (qk + 1 < l ? qk + 1 : 0)] >= b;
            }
            if (lowest) {
              P.tip_h[base + owner] = B.tip_h[t];
              if (one) P.pbase[base + owner] = q >= pr ? q - pr : q - pr + l;  // its index
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
          if (ntips > 1) P.pbase[i] = rec ? 1 : 0;  // several tips: half-edges at pos, or none
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
                        const LongList& Dm, int cap, int repair, int tips_to_long, int beside,
                        Counters* C, int grid, cudaStream_t s, bool pdl) {
  if (cap < 16 || cap > kWalkCap || cap % 16) return cudaErrorInvalidValue;
  constexpr size_t smem = sizeof(WalkBuf) * kWalkWarps;
  static std::atomic<bool> attr[kMaxDevices];
  const cudaError_t e = smem_limit_once(reinterpret_cast<const void*>(k_walk), (int)smem, attr);
  if (e != cudaSuccess) return e;
  static std::atomic<int> resident{0};
  grid = resident_grid(reinterpret_cast<const void*>(k_walk), kWalkThreads, smem, grid, &resident);
  return launch_chain(k_walk, grid, kWalkThreads, smem, s, pdl, M, tf, entry, P, pool, Lg, D1, Dm,
                      cap, repair, tips_to_long, beside, C);
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

// Reparation of one polygon with 2 to kRsMaxSplit tips by a warp.
//
// The walk left the polygon's half-edges in boundary order from its canonical start.
// A lane per tip finds its split edge from the labels as they are (a tip's fan changes
// only through a split edge that ends at the tip, which removes it as a tip), and the
// rule's order -- the first piece with a tip is split at its smallest tip -- comes to
// all tips in increasing vertex order, leaving out those a smaller tip's split edge
// ends on.  With the kept split edges marked frontier, the nodes are the polygon's
// half-edges and two per split edge (oj = b->x and tw = x->b); a node's successor is
// the next half-edge, unless a split edge ends at its destination: then it is found by
// turning.  A lane per side of each split edge walks its piece, the piece's smallest
// such node names it, and the pieces' order is the rule's tree of splits: the two sides
// of each split joined, the largest tip first, the side of oj on the left.
//
// What bounds it: the chain of dependent loads of one polygon (its records, the fans,
// the turns), about 17 us; the one-thread form split tip by tip, walking its pieces
// in between.  Before and after, us: gmm16-10m (19,880 polygons) 71 and 57, 200,000
// mixture points (416) 65 and 18, where it was the longest of the three kernels that
// run side by side (the run: 122 and 104).
constexpr int kRsThreads = 128;
constexpr int kRsWarps = kRsThreads / 32;
constexpr int kRsNodes = kWalkCap + 2 * kRsMaxSplit;
constexpr int kRsRounds = (kRsNodes + 31) / 32;
static_assert(kWalkCap == 64 && kRsNodes < 256 && 2 * kRsMaxSplit <= 32 &&
                  4 * (kRsMaxSplit + 1) <= 64,
              "two half-edges a lane, a lane per side, a piece order of 4-bit numbers");

struct SplitBuf {
  int h[kRsNodes], v[kRsNodes];  // nodes: half-edge, origin
  int end[2 * kRsMaxSplit];      // the split edges' end vertices
  unsigned char nx[kRsNodes], todo[kRsNodes];
  unsigned char tip[kRsMaxSplit];
  unsigned char pstart[kRsMaxSplit + 1], plen[kRsMaxSplit + 1];
};

// Returns the number of pieces (their records in F from *foff), or -1; every lane of
// the warp calls it.  *by_half_edge grows by the pieces whose smallest vertex repeats (all,
// if rare).  hs: the polygon's L half-edges, overwritten with the pieces.
__device__ __forceinline__ int split_by_warp(const DevMesh& M, uint8_t* lab, int* tf, SplitBuf& B,
                                             int L, int nt, int* hs, long long off,
                                             const FinalPieces& F, int rare, Counters* C,
                                             long long* foff, unsigned* by_half_edge) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int H = (int)(3 * M.m);
  const long long limit = 3 * M.m + 3;
  bool bad = false;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int q = lane + 32 * r;
    if (q < L) {
      const int h = hs[q];
      bad |= (unsigned)h >= (unsigned)H;
      B.h[q] = h;
    }
  }
  if (__any_sync(full, bad)) return -1;
  __syncwarp();
  // origins, and the tips: half-edges followed by their twins
  int found = 0;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int q = lane + 32 * r;
    bool tip = false;
    if (q < L) {
      const int h = B.h[q];
      B.v[q] = M.tri[h];
      tip = tf_twin(tf[h]) == B.h[q + 1 < L ? q + 1 : 0];
    }
    const unsigned t = __ballot_sync(full, tip);
    const int k = found + __popc(t & lt);
    if (tip && k < kRsMaxSplit) B.tip[k] = (unsigned char)q;
    found += __popc(t);
  }
  __syncwarp();
  if (found != nt) return -1;
  // a lane per tip b: its split edge oj = b->x
  int b = 0x7fffffff, oj = -1, tw = -1, x = -1;
  if (lane < nt) {
    const int q = B.tip[lane];
    b = B.v[q + 1 < L ? q + 1 : 0];
    oj = split_edge(tf, B.h[q], H);
    tw = oj >= 0 ? tf_twin(tf[oj]) : H;
    if (tw < H) x = M.tri[tw];
    else bad = true;
  }
  if (__any_sync(full, bad)) return -1;
  // in increasing vertex order; a split edge that ends on a larger tip removes it
  int rank = 0, hit = -1;
  for (int k = 0; k < nt; ++k) rank += __shfl_sync(full, b, k) < b;
  for (int k = 0; k < nt; ++k) {
    const int bk = __shfl_sync(full, b, k), rk = __shfl_sync(full, rank, k);
    if (bk == x && bk > b) hit = rk;
  }
  unsigned gone = 0;
  for (int r = 0; r < nt; ++r) {
    const unsigned at = __ballot_sync(full, lane < nt && rank == r);
    if (!at) return -1;  // (a vertex twice among the tips: a corrupt mesh)
    const int to = __shfl_sync(full, hit, __ffs(at) - 1);
    if (!(gone >> r & 1u) && to >= 0) gone |= 1u << to;
  }
  const bool keep = lane < nt && !(gone >> rank & 1u);
  const int chord = __popc(~gone & ((1u << rank) - 1u));  // among the kept, by vertex
  const int ns = __popc(__ballot_sync(full, keep)), N = L + 2 * ns;
  if (keep) {
    B.h[L + 2 * chord] = oj;
    B.v[L + 2 * chord] = b;
    B.h[L + 2 * chord + 1] = tw;
    B.v[L + 2 * chord + 1] = x;
    B.end[2 * chord] = b;
    B.end[2 * chord + 1] = x;
    set_frontier(lab, tf, oj);
    set_frontier(lab, tf, tw);
  }
  __syncwarp();
  // successors: the next half-edge, or by turning where a split edge ends
  int ntodo = 0;
#pragma unroll
  for (int r = 0; r < kRsRounds; ++r) {
    const int a = lane + 32 * r;
    bool turn = a >= L && a < N;
    if (a < L) {
      const int nx = a + 1 < L ? a + 1 : 0;
      const int d = B.v[nx];
      B.nx[a] = (unsigned char)nx;
      turn = rare != 0;
      for (int k = 0; k < 2 * ns; ++k) turn |= B.end[k] == d;
    }
    const unsigned t = __ballot_sync(full, turn);
    if (turn) B.todo[ntodo + __popc(t & lt)] = (unsigned char)a;
    ntodo += __popc(t);
  }
  __syncwarp();
  for (int t = lane; t < ntodo; t += 32) {
    const int a = B.todo[t];
    long long steps = 0;
    const int g = turn_tf(tf, B.h[a], H, steps, limit);
    int c = 0;
    while (c < N && B.h[c] != g) ++c;
    if (g < 0 || c == N) bad = true;
    else B.nx[a] = (unsigned char)c;
  }
  if (__any_sync(full, bad)) return -1;
  __syncwarp();
  // a lane per side of each split edge walks its piece
  const bool side = lane < 2 * ns;
  int name = 255, len = 0, least = 0x7fffffff, start = 0;
  bool again = false;  // the smallest vertex repeats
  if (side) {
    int a = L + lane;
    do {
      const int o = B.v[a];
      again = o == least || (again && o > least);
      if (o < least || (o == least && B.h[a] < B.h[start])) {
        least = o;
        start = a;
      }
      if (a >= L && a < name) name = a;
      a = B.nx[a];
    } while (++len <= N && a != L + lane);
    bad = len > N;
  }
  if (__any_sync(full, bad)) return -1;
  const unsigned owners = __ballot_sync(full, side && name == L + lane);
  const int np = __popc(owners);
  if (np != ns + 1) return -1;
  *by_half_edge += __popc(owners & __ballot_sync(full, again || rare));
  // the piece of each side, numbered by name; each piece's start and length
  const int piece = side ? __popc(owners & ((1u << (name - L)) - 1u)) : 0;
  if (owners >> lane & 1u) {
    B.pstart[piece] = (unsigned char)start;
    B.plen[piece] = (unsigned char)len;
  }
  __syncwarp();
  // the tree of splits: lane p holds the group of piece p and, as a group's first
  // piece, the group's pieces in order (4 bits each) and their number
  int group = lane, count = 1;
  unsigned long long order = (unsigned)lane & 15u;
  for (int k = ns - 1; k >= 0; --k) {
    const int ga = __shfl_sync(full, group, __shfl_sync(full, piece, 2 * k));
    const int gb = __shfl_sync(full, group, __shfl_sync(full, piece, 2 * k + 1));
    if (ga == gb) return -1;
    const unsigned long long ob = __shfl_sync(full, order, gb);
    const int cb = __shfl_sync(full, count, gb);
    if (lane == ga) {
      order |= ob << (4 * count);
      count += cb;
    }
    if (group == gb) group = ga;
  }
  order = __shfl_sync(full, order, __shfl_sync(full, group, 0));
  // the pieces, a lane each, from their canonical starts
  const int p = lane < np ? (int)(order >> (4 * lane) & 15u) : 0;
  const int l = lane < np ? B.plen[p] : 0;
  int at = l;
#pragma unroll
  for (int d = 1; d < 16; d <<= 1) {
    const int y = __shfl_up_sync(full, at, d);
    if (lane >= d) at += y;
  }
  at -= l;
  long long f = 0;
  if (lane == 0)
    f = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(&C->fslot_alloc),
                             (unsigned long long)np);
  f = __shfl_sync(full, f, 0);
  if (f + np > F.cap) return -1;
  if (lane < np) {
    F.pos[f + lane] = off + at;
    F.len[f + lane] = l;
    int a = B.pstart[p];
    for (int k = 0; k < l; ++k) {
      hs[at + k] = B.v[a];
      a = B.nx[a];
    }
  }
  *foff = f;
  return np;
}

__global__ void __launch_bounds__(kRsThreads) k_repair_multi(DevMesh M, uint8_t* lab, int* tf,
                                                             PolyArrays P, FinalPieces F,
                                                             Pool pool, LongList Dm, int rare,
                                                             Counters* C) {
  __shared__ SplitBuf s_buf[kRsWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long nd = min(C->n_multi, Dm.cap);
  const int H = (int)(3 * M.m);
  const long long limit = 3 * M.m + 3;
  unsigned st_splits = 0, st_seq = 0, st_turn = 0;
  for (long long d = (long long)blockIdx.x * kRsWarps + warp; d < nd;
       d += (long long)gridDim.x * kRsWarps) {
    const int i = Dm.poly[d];
    const int L = P.len[i], nt = P.ntip[i];
    int cnt = -1;
    long long foff = 0;
    if (nt >= 2 && nt <= kRsMaxSplit && L >= 3 && L <= kWalkCap && P.pbase[i] == 1) {
      const long long off = P.pos[i];
      if (off >= 0 && off + L + 2 * nt <= pool.cap)
        cnt = split_by_warp(M, lab, tf, s_buf[warp], L, nt, pool.v + off, off, F, rare, C, &foff,
                            &st_turn);
    } else if (nt > kRsMaxSplit && L >= 3) {
      if (lane == 0) {  // more tips than the nodes hold: one thread, piece by piece
        ++st_seq;
        const long long off = (long long)atomicAdd(
            reinterpret_cast<unsigned long long*>(&C->pool_alloc), (unsigned long long)(L + 2 * nt));
        foff = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(&C->fslot_alloc),
                                    (unsigned long long)(nt + 1));
        if (off + L + 2 * nt <= pool.cap && foff + nt + 1 <= F.cap) {
          const Cyc first{P.start[i], L, P.tip_h[i], nt, true};
          cnt = repair_seq(M.tri, tf, lab, first, nt + 1, H, limit, F.h + foff, F.pos + foff,
                           F.len + foff, pool.v + off, off, L + 2 * nt);
        }
      }
    }
    if (lane == 0) {
      if (cnt < 0) {
        set_error(C, POLYLLA_ERR_LIMIT, 54);
      } else {
        P.pcnt[i] = cnt;
        P.pbase[i] = (int)foff;
        P.flen[i] = L + 2 * (cnt - 1);
        st_splits += cnt - 1;
      }
    }
    __syncwarp();
  }
  if (lane == 0) {
    if (st_splits)
      atomicAdd(reinterpret_cast<unsigned long long*>(&C->n_splits), (unsigned long long)st_splits);
    if (st_seq)
      atomicAdd(reinterpret_cast<unsigned long long*>(&C->n_multi_seq), (unsigned long long)st_seq);
    if (st_turn)
      atomicAdd(reinterpret_cast<unsigned long long*>(&C->n_multi_turn), (unsigned long long)st_turn);
  }
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
  static std::atomic<int> cap{0};
  const int grid = resident_grid(reinterpret_cast<const void*>(k_repair_multi), kRsThreads, 0,
                                 (long long)sms * 16, &cap);
  k_repair_multi<<<grid, kRsThreads, 0, s>>>(M, lab, tf, P, F, pool, Dm, rare, C);
  return cudaGetLastError();
}

}  // namespace polylla
