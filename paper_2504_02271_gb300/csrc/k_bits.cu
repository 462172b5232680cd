// Step two by bit rows: the closure of one hyperedge u (Sec. 3.2-3.3) without looking its
// neighbours' lists up.
//
// Every hyper-triangle {e_u, e_v, e_w} is owned by its lowest-ranked member u (see
// k_close.cu), and v, w are out-neighbours of u that share a vertex.  So the triangles of u
// are the intersecting pairs of out(u), and whether and how two of them intersect follows
// from the vertices of the hyperedges in out(u) alone.  A team lays them out as a 0/1
// matrix: one row per out-neighbour, one column per vertex that lies in e_u or in at least
// two of the hyperedges of out(u) (a vertex of one of them only is private to it).  A
// column is stored as a bit row over out(u), S_y = {w in out(u) : y in e_w}.  For
// an out-neighbour v, 32 pairs (v, w) at a time,
//   g = OR of S_y over y in e_u cap e_v          d = OR of ~S_y over the same
//   f = OR of S_y over y in e_u \ e_v            a = OR of ~S_y over the same
//   t = number of S_y, y in e_v \ e_u, holding w (bit-sliced: one bit plane per binary digit)
//   e = t > 0       b = some y in e_v \ e_u is private or has ~S_y
//   c = w has a private vertex or t differs from w's number of shared vertices outside e_u
// are the seven Venn regions of Sec. 2, and the pair is a hyper-triangle when g or e is
// set.  Classes without inclusion (9-20, nearly all) are counted by population counts of
// 12 bit expressions; a pair with an inclusion is put in its labelled-mask bin by itself.
//
// Work per out-neighbour v: its |e_v| vertices (one dictionary access each), and per 32
// out-neighbours |e_u| words of e_u's columns and one word per shared vertex of e_v outside e_u,
// against one hash lookup and about 71 lane instructions per entry of out(v) for the list walk
// (95 entries of out(v) per out-neighbour on the co-authorship workload, 1,350 on the tag-shaped
// prefix of 40,000 hyperedges).  The closure there went from 8.0 to 6.0 ms and from 145 to 46
// ms, on 2,000 uniform hyperedges over 1,000 vertices from 2.2 to 0.5 ms.  Owners whose
// neighbourhoods are sparse, or large hyperedges over few others, walk (list_of in
// k_close.cu); an owner whose tables overflow goes back to the walking team of its shape.  The
// small teams are bound by instruction issue and their barriers (10,000-20,000 warp
// instructions a team), the large ones by the shared-memory reads of the column words (half of
// their time) and by the vertices read from memory (a third).
#include <type_traits>

#include "hg_internal.cuh"

namespace hg {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kBins = 128;
constexpr int kPlanes = kBitPlanes;
constexpr int kClasses = 12;          // classes counted in registers
constexpr int kMaxProbes = 256;       // dictionary probes of one vertex
constexpr uint32_t kShared = 1u << 31;   // dictionary key seen at least twice (or in e_u)

// labelled masks (bit r = region r of a..g) standing for the classes of patterns 9-20 in
// the order of bit_step's counters, then of patterns 1-8; any labelling of the class does
// (the host folds the six orders of a mask)
__constant__ uint8_t c_class_mask[kClasses + 8] = {71, 79, 93, 95, 120, 121, 123, 127,
                                                   56, 57, 59, 63,
                                                   73, 67, 75, 88, 90, 77, 89, 91};

constexpr uint32_t kPad = ~0u;   // list entry that is no vertex
constexpr int kWideMean = 8;         // mean column list from which a step takes four words

__device__ __forceinline__ uint32_t slot_of(uint32_t y, int log2) {
  return (y * 0x9E3779B1u) >> (32 - log2);
}

template <int NW>
__device__ __forceinline__ void team_sync() {
  if (NW == 1) __syncwarp();
  else __syncthreads();
}

// Vertex dictionary of a team.  Hash: key[slot] = y, bit 31 once y is shared, val[slot] its
// column (valid once shared).  Direct (few vertices): two bit maps, seen and shared, and
// val[y].  touch() returns the handle stored in the column list.
template <bool DIRECT>
struct Dict {
  uint32_t* key;    // direct: the seen map, then the shared map
  uint16_t* val;
  int log2;
  int words;
  // *full is set when a key finds no slot within kMaxProbes (the owner is then given back)
  __device__ __forceinline__ uint32_t touch(uint32_t y, int* ncol, int* full) const {
    if (DIRECT) {
      const uint32_t b = 1u << (y & 31u);
      uint32_t* shared_map = key + words;
      volatile uint32_t* sh = shared_map + (y >> 5);
      if (*sh & b) return y;
      if (atomicOr(&key[y >> 5], b) & b) {
        if (!(atomicOr(&shared_map[y >> 5], b) & b)) val[y] = (uint16_t)atomicAdd(ncol, 1);
      }
      return y;
    }
    const uint32_t mask = (1u << log2) - 1u;
    uint32_t h = slot_of(y, log2);
    for (int probe = 0; probe < kMaxProbes; ++probe) {
      uint32_t cur = *(volatile uint32_t*)&key[h];
      if (cur == ~0u) cur = atomicCAS(&key[h], ~0u, y);
      if (cur == ~0u) return h;
      if ((cur & ~kShared) == y) {
        if (!(cur & kShared) && !(atomicOr(&key[h], kShared) & kShared))
          val[h] = (uint16_t)atomicAdd(ncol, 1);
        return h;
      }
      h = (h + 1u) & mask;
    }
    *full = 1;
    return 0;
  }
  // vertex number p of e_u: column p
  __device__ __forceinline__ void own(uint32_t y, int p) const {
    if (DIRECT) {
      const uint32_t b = 1u << (y & 31u);
      atomicOr(&key[y >> 5], b);
      atomicOr(&key[words + (y >> 5)], b);
      val[y] = (uint16_t)p;
      return;
    }
    const uint32_t mask = (1u << log2) - 1u;
    uint32_t h = slot_of(y, log2);
    // the table is at most half full, so a free slot exists
    while (atomicCAS(&key[h], ~0u, y | kShared) != ~0u) h = (h + 1u) & mask;
    val[h] = (uint16_t)p;
  }
  // column of a vertex that was touched, -1 when it is private
  __device__ __forceinline__ int find(uint32_t y) const {
    if (DIRECT) return col(y);
    const uint32_t mask = (1u << log2) - 1u;
    uint32_t h = slot_of(y, log2);
    for (int probe = 0; probe < kMaxProbes; ++probe) {
      const uint32_t cur = key[h];
      if ((cur & ~kShared) == y) return cur & kShared ? (int)val[h] : -1;
      h = (h + 1u) & mask;
    }
    return -1;
  }
  // column of a handle, -1 when its vertex is private
  __device__ __forceinline__ int col(uint32_t h) const {
    if (DIRECT) return (key[words + (h >> 5)] >> (h & 31u)) & 1u ? (int)val[h] : -1;
    return key[h] & kShared ? (int)val[h] : -1;
  }
};

// What the row step reads: the team's matrix.
struct BitRows {
  const uint2* rows;        // [du] column list of every out-neighbour: start, entries
  const uint16_t* csr;      // columns (outside e_u, shared), starts at multiples of four
  const uint32_t* m;        // [szu][W] columns of e_u
  const uint32_t* s;        // [ncol][cw] the other columns, words c0 .. c0 + cw - 1
  const uint32_t* priv;     // [W] out-neighbours with a private vertex
  const uint32_t* plane;    // [kPlanes][W] digits of the shared counts
  int W, du, szu, np, cw, c0;
};

__device__ __forceinline__ uint32_t maj(uint32_t a, uint32_t b, uint32_t c) {
  return (a & b) | (c & (a | b));
}

// Rows k0 .. k0 + 32 / WL - 1 against the words j0 .. j0 + WL - 1 of the chunk: lane =
// (row, word), so that the lanes of a row read consecutive words of a column and share its
// column list.
template <int WL, int NP>
__device__ __forceinline__ void bit_step(const BitRows& t, int k0, int j0, int n_max,
                                         uint32_t (&cls)[kClasses], uint32_t* hist, int lane) {
  const int j = j0 + lane % WL, k = k0 + lane / WL;
  const int jend = t.c0 + t.cw < t.W ? t.c0 + t.cw : t.W;   // words of the chunk
  const int jc = j < jend ? j : jend - 1;   // a word to read for lanes past the last one
  const int kc = k < t.du ? k : t.du - 1, i = kc >> 5;
  const uint2 row = t.rows[kc];
  const bool valid = k < t.du && j < jend && i <= j;
  // the pairs of this word: w after v in out(u)
  uint32_t want = t.du - 32 * jc >= 32 ? ~0u : (1u << (t.du - 32 * jc)) - 1u;
  if (!valid) want = 0;
  if (i == j) want &= 0xfffffffeu << (k & 31);
  uint32_t ra = 0, rd = 0, rf = 0, rg = 0;
  {
    const uint32_t* mi = t.m + i;
    const uint32_t* mj = t.m + jc;
    for (int p = 0; p < t.szu; ++p, mi += t.W, mj += t.W) {   // columns of e_u
      const uint32_t x = *mj, in = (uint32_t)((int32_t)(*mi << (31 - (kc & 31))) >> 31);
      rg |= x & in;
      rd |= in & ~x;
      rf |= x & ~in;
      ra |= ~(x | in);
    }
  }
  // columns outside e_u: t in bit planes (np of them can be reached), b
  const int n = valid ? (int)row.y : 0;
  const int np = n_max ? 32 - __clz(n_max) : 0;
  const uint16_t* cl = t.csr + row.x;
  const uint32_t* S = t.s + (jc - t.c0);
  uint32_t T[NP];
#pragma unroll
  for (int q = 0; q < NP; ++q) T[q] = 0;
  for (int x = 0; x < n; x += 4) {   // four columns at a time (lists are padded to that)
    const uint2 c4 = *reinterpret_cast<const uint2*>(cl + x);
    const uint32_t v0 = S[(c4.x & 0xffffu) * t.cw], v1 = S[(c4.x >> 16) * t.cw];
    const uint32_t v2 = S[(c4.y & 0xffffu) * t.cw], v3 = S[(c4.y >> 16) * t.cw];
    const uint32_t s01 = T[0] ^ v0 ^ v1, c01 = maj(T[0], v0, v1);
    const uint32_t c23 = maj(s01, v2, v3);
    T[0] = s01 ^ v2 ^ v3;
    uint32_t carry = maj(T[1], c01, c23);
    T[1] ^= c01 ^ c23;
#pragma unroll
    for (int q = 2; q < NP; ++q) {
      if (q >= np) break;
      const uint32_t up = T[q] & carry;
      T[q] ^= carry;
      carry = up;
    }
  }
  // e: t > 0; b: v has a private vertex or t differs from its count; c: the same of w
  uint32_t re = 0, rb = 0u - ((t.priv[i] >> (kc & 31)) & 1u), rc = t.priv[jc];
  if (np > 0) {
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      if (q >= np) break;
      re |= T[q];
      rb |= T[q] ^ (0u - ((uint32_t)n >> q & 1u));
      rc |= T[q] ^ t.plane[q * t.W + jc];
    }
  }
  for (int q = np; q < t.np; ++q) rc |= t.plane[q * t.W + jc];   // counts t cannot reach
  const uint32_t tri = (rg | re) & want;
  // The class of a pair follows from the number of pairwise regions (d, e, f), of single
  // regions (a, b, c) and g: none pairwise: 2 or 3 singles (patterns 2, 9); one: 1, 2, 3
  // singles (1, 3 or 6, 10), 6 when the single region opposite the pair is there; two: 0 to
  // 3 singles (4, 5 or 7, 8 or 11, 12), 5 and 8 when the single region of the hyperedge in
  // both pairs is there; three: 13-16 with g, 17-20 without.
  const uint32_t p0 = rd ^ re ^ rf, p1 = maj(rd, re, rf);
  const uint32_t s0 = ra ^ rb ^ rc, s1 = maj(ra, rb, rc);
  const uint32_t none = tri & ~p1 & ~p0, one = tri & ~p1 & p0, two = tri & p1 & ~p0;
  const uint32_t three = tri & p1 & p0, tg = three & rg, tn = three & ~rg;
  const uint32_t mid = (rc & ~rd) | (ra & ~re) | (rb & ~rf);
  const uint32_t c9 = none & s0, c10 = one & s1 & s0, c11 = two & s1 & ~s0 & ~mid;
  const uint32_t c12 = two & s1 & s0;
  cls[0] += __popc(c9);
  cls[1] += __popc(c10);
  cls[2] += __popc(c11);
  cls[3] += __popc(c12);
  cls[4] += __popc(tg & ~s1 & ~s0);
  cls[5] += __popc(tg & ~s1 & s0);
  cls[6] += __popc(tg & s1 & ~s0);
  cls[7] += __popc(tg & s1 & s0);
  cls[8] += __popc(tn & ~s1 & ~s0);
  cls[9] += __popc(tn & ~s1 & s0);
  cls[10] += __popc(tn & s1 & ~s0);
  cls[11] += __popc(tn & s1 & s0);
  const uint32_t rest = tri & ~(three | c9 | c10 | c11 | c12);
  if (__any_sync(kFull, rest != 0)) {   // patterns 1-8 (an inclusion among the three)
    const uint32_t opp = (rd & rc) | (re & ra) | (rf & rb);
    const uint32_t w8[8] = {one & ~s1 & s0, none & ~s0,        one & s1 & ~s0 & ~opp,
                            two & ~s1 & ~s0, two & ~s1 & s0 & mid, one & s1 & ~s0 & opp,
                            two & ~s1 & s0 & ~mid, two & s1 & ~s0 & mid};
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const uint32_t c = __reduce_add_sync(kFull, (uint32_t)__popc(w8[q]));
      if (lane == q && c) atomicAdd(&hist[c_class_mask[kClasses + q]], c);
    }
  }
}

// Every pair of a row and a word of the chunk on or above the diagonal, the row groups
// of all words dealt to the warps in turn.
template <int WL, int NW>
__device__ __forceinline__ void bit_rows(const BitRows& t, uint32_t (&cls)[kClasses],
                                         uint32_t* hist, int lane, int w) {
  constexpr int RG = 32 / WL;
  const int jend = t.c0 + t.cw < t.W ? t.c0 + t.cw : t.W;
  int first = w;   // this warp's first row group of the word group
  for (int j0 = t.c0; j0 < jend; j0 += WL) {
    const int kend = t.du < 32 * (j0 + WL) ? t.du : 32 * (j0 + WL);
    const int groups = (kend + RG - 1) / RG;
    int q = first;
    for (; q < groups; q += NW) {
      const int k = q * RG + lane / WL;
      // (lists of rows below the diagonal are not walked; they only widen the digits)
      const int n_max = __reduce_max_sync(kFull, k < t.du ? (int)t.rows[k].y : 0);
      if (n_max < 256) bit_step<WL, 8>(t, q * RG, j0, n_max, cls, hist, lane);
      else bit_step<WL, kPlanes>(t, q * RG, j0, n_max, cls, hist, lane);
    }
    first = q - groups;
  }
}

// Long column lists (wide) take four words of a row at a time, so that a list entry is read
// once for them; short ones one word per lane and 32 rows, which wastes least below the
// diagonal.
template <int NW>
__device__ __forceinline__ void chunk_rows(const BitRows& t, bool wide, uint32_t (&cls)[kClasses],
                                           uint32_t* hist, int lane, int w) {
  if (wide && t.cw >= 4) bit_rows<4, NW>(t, cls, hist, lane, w);
  else bit_rows<1, NW>(t, cls, hist, lane, w);
}

__device__ __forceinline__ void copy4(uint32_t* dst, const int32_t* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Per-block counters of both kernels and the flush of their bins.
struct TeamBlock {
  uint32_t hist[kBins];
  unsigned long long work[kCloseBuckets][3];
  unsigned long long probes;
  int32_t next;   // next owner, -1 after the last
  int ncol, most, used, full, inc, ncand;
  int bins[32];
};

template <int NW>
__device__ __forceinline__ void flush_bins(TeamBlock& b, uint32_t (&cls)[kClasses],
                                           unsigned long long* __restrict__ out, int lane) {
#pragma unroll
  for (int q = 0; q < kClasses; ++q) {
    const uint32_t x = __reduce_add_sync(kFull, cls[q]);
    if (lane == 0 && x) atomicAdd(&b.hist[c_class_mask[q]], x);
    cls[q] = 0;
  }
  team_sync<NW>();
  for (int k = threadIdx.x; k < kBins; k += NW * 32) {
    const uint32_t x = b.hist[k];
    if (x) atomicAdd(&out[k], (unsigned long long)x);
    b.hist[k] = 0;
  }
  team_sync<NW>();
}

// Bin of a shared count in the row order.
__device__ __forceinline__ int count_bin(uint32_t c) {
  return c < 16u ? (int)c : (c < 16u + 8u * 15u ? 16 + (int)((c - 16u) >> 3) : 31);
}

// Rows in their final order with the digits of their shared counts, their private flags
// (alone(k)) and the columns of e_u (has(p, k): row k has vertex p of e_u).  sort: rows by
// ascending count, so that the rows of a step have lists of like length and the pair (v, w)
// walks the shorter one (v before w); else as they are.  Column lists are padded to a multiple
// of four with the empty column ncol.  np: digits of the largest count.  Synchronises at the
// end.
template <int NW, class Alone, class Has>
__device__ __forceinline__ void finish_rows(TeamBlock& tb, const uint32_t* cnt, const uint2* in,
                                            uint2* out, uint16_t* csr, int ncol, uint32_t* m,
                                            uint16_t* order, uint32_t* plane, int du, int W,
                                            int szu, int np, bool sort, int lane, int w,
                                            Alone alone, Has has) {
  if (sort) {
    if (threadIdx.x < 32) tb.bins[threadIdx.x] = 0;
    team_sync<NW>();
    for (int k = threadIdx.x; k < du; k += NW * 32) atomicAdd(&tb.bins[count_bin(cnt[k])], 1);
    team_sync<NW>();
    if (w == 0) {
      const int x = tb.bins[lane];
      int incl = x;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int up = __shfl_up_sync(kFull, incl, d);
        if (lane >= d) incl += up;
      }
      tb.bins[lane] = incl - x;
    }
    team_sync<NW>();
    for (int k = threadIdx.x; k < du; k += NW * 32)
      order[atomicAdd(&tb.bins[count_bin(cnt[k])], 1)] = (uint16_t)k;
    team_sync<NW>();
  }
  for (int k0 = w * 32; k0 < du; k0 += NW * 32) {
    const int k = k0 + lane, i = k0 >> 5;
    const int old = k < du ? (sort ? (int)order[k] : k) : 0;
    const uint32_t c = k < du ? cnt[old] : 0u;
    const uint32_t pw = __ballot_sync(kFull, k < du && alone(old));
    if (lane == 0) plane[kPlanes * W + i] = pw;
    for (int q = 0; q < np; ++q) {
      const uint32_t dw = __ballot_sync(kFull, (c >> q) & 1u);
      if (lane == 0) plane[q * W + i] = dw;
    }
    if (k < du) {
      const uint32_t at = in[old].x;
      out[k] = make_uint2(at, c);
      for (uint32_t e = c; e & 3u; ++e) csr[at + e] = (uint16_t)ncol;   // the empty column
    }
    for (int p = 0; p < szu; ++p) {
      const uint32_t mw = __ballot_sync(kFull, k < du && has(p, old));
      if (lane == 0) m[p * W + i] = mw;
    }
  }
  team_sync<NW>();
}

// The words c0 .. c0 + cw - 1 of every column, from the column lists of their rows (G lanes
// per row).  The store is empty before; synchronises at the end.
template <int NW, int G>
__device__ __forceinline__ void fill_chunk(uint32_t* S, const uint2* rows, const uint16_t* csr,
                                           int du, int c0, int cw) {
  const int kend = du < 32 * (c0 + cw) ? du : 32 * (c0 + cw);
  for (int k = 32 * c0 + (int)threadIdx.x / G; k < kend; k += NW * 32 / G) {
    const uint2 row = rows[k];
    for (int e = (int)threadIdx.x % G; e < (int)row.y; e += G)
      atomicOr(&S[(int)csr[row.x + e] * cw + ((k >> 5) - c0)], 1u << (k & 31));
  }
  team_sync<NW>();
}

// ------------------------------------------------------------------ small teams
//
// Everything in shared memory, |e_u| <= 32.  The vertices of out(u)'s hyperedges are copied
// there (asynchronously, four lanes per hyperedge) as one list, in groups of four entries of
// one hyperedge, and all threads take it group by group: a hashed bit map finds the entries
// whose vertex may occur twice or lie in e_u, and only those go through the exact dictionary
// (on the tiny_plain workload a third of them).

struct SmallLayout {
  int icap, dcap, mwords, swords, slots_log2, bits_log2;
  uint32_t off_y, off_map, off_list, off_key, off_val, off_src, off_rows, off_cnt, off_mask,
      off_prow, off_plane, off_m, off_s, bytes;
};

// The next owner, fetched by one thread while the team works on the current one.
struct NextOwner {
  int32_t r, u;
  __device__ __forceinline__ void fetch(int32_t* counter) { r = atomicAdd(counter, 1); }
  __device__ __forceinline__ void find(const OwnerList& list, int32_t n) {
    u = r < n ? list.get(r) : -1;
  }
};

// An owner that a team cannot hold goes back to the walking team of its label (to the
// global-table blocks when every owner is to be handed over).
__device__ __forceinline__ void give_back(const ReturnLists& ret, const OwnerList& handed,
                                          int handover, int label, int32_t u) {
  const bool all = handover && label < kWideBucket;
#pragma unroll
  for (int k = 0; k < kCloseBuckets; ++k)   // (the lists are kernel parameters: no indexing)
    if (!all && k == label) ret.back[k].put(u);
  if (all) handed.put(u);
}

template <int NW, int MINB, bool PACKED, typename ROW>
__global__ void __launch_bounds__(NW * 32, MINB)
    k_bits_small(DevGraph g, Oriented o, SmallLayout ly, OwnerList list,
                 unsigned long long* __restrict__ hist_out, unsigned long long* __restrict__ work,
                 TeamRule rule, int32_t* __restrict__ counter, ReturnLists ret, OwnerList handed,
                 int handover) {
  constexpr int NT = NW * 32, G = 4;
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ TeamBlock tb;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, tid = threadIdx.x;
  uint32_t* y = reinterpret_cast<uint32_t*>(dyn + ly.off_y);
  uint4* y4 = reinterpret_cast<uint4*>(y);
  uint32_t* map1 = reinterpret_cast<uint32_t*>(dyn + ly.off_map);
  uint32_t* map2 = map1 + ((1u << ly.bits_log2) >> 5);
  uint16_t* csr = reinterpret_cast<uint16_t*>(dyn + ly.off_map);   // once the maps are dead
  uint16_t* cand = reinterpret_cast<uint16_t*>(dyn + ly.off_list);
  Dict<false> dict;
  dict.key = reinterpret_cast<uint32_t*>(dyn + ly.off_key);
  dict.val = reinterpret_cast<uint16_t*>(dyn + ly.off_val);
  dict.words = 0;
  uint4* src = reinterpret_cast<uint4*>(dyn + ly.off_src);
  uint2* rows = reinterpret_cast<uint2*>(dyn + ly.off_rows);   // place in the list, |e_v|
  uint2* rows2 = reinterpret_cast<uint2*>(src);                // once the list is copied
  uint16_t* order = reinterpret_cast<uint16_t*>(rows2 + ly.dcap);
  uint32_t* cnt = reinterpret_cast<uint32_t*>(dyn + ly.off_cnt);
  uint32_t* mask = reinterpret_cast<uint32_t*>(dyn + ly.off_mask);   // e_u cap e_v
  ROW* prow = reinterpret_cast<ROW*>(dyn + ly.off_prow);   // per group of four entries
  uint32_t* plane = reinterpret_cast<uint32_t*>(dyn + ly.off_plane);
  uint32_t* m = reinterpret_cast<uint32_t*>(dyn + ly.off_m);
  uint32_t* S = reinterpret_cast<uint32_t*>(dyn + ly.off_s);
  for (int k = tid; k < kBins; k += NT) tb.hist[k] = 0;
  for (int k = tid; k < kCloseBuckets * 3; k += NT) (&tb.work[0][0])[k] = 0;
  const int32_t n = *list.n;
  uint32_t cls[kClasses];
#pragma unroll
  for (int q = 0; q < kClasses; ++q) cls[q] = 0;
  unsigned long long since_flush = 0;
  int32_t cur = 0;
  NextOwner next{0, -1};
  if (tid == 0) {
    next.fetch(counter);
    next.find(list, n);
    tb.next = next.u;
  }
  team_sync<NW>();
  int32_t u = tb.next;
  while (u >= 0) {
    const uint4 hu = g.rec[u];
    const int64_t bu = o.row_ptr[u];
    const int32_t entries = g.osum[u];
    if (tid == 0) next.fetch(counter);
    const int32_t mem = member_of(g, u);
    if (mem != cur || since_flush > (1ull << 30)) {   // 32-bit bins stay far from overflow
      flush_bins<NW>(tb, cls, hist_out + (size_t)cur * kBins, lane);
      cur = mem;
      since_flush = 0;
    }
    // 0. empty maps
    {
      uint4* mv = reinterpret_cast<uint4*>(map1);
      for (int k = tid; k < (2 << ly.bits_log2) / 128; k += NT) mv[k] = make_uint4(0, 0, 0, 0);
    }
    const int32_t du = (int32_t)hu.w, szu = (int32_t)hu.z;
    const int64_t eb = (int64_t)(((unsigned long long)hu.y << 32) | hu.x);
    const int W = (du + 31) >> 5;
    since_flush += (unsigned long long)du * (unsigned long long)du / 2;
    // empty dictionary (slots: at least the entries and e_u; a shared vertex has two
    // entries, so at most about half are taken)
    int lg = 32 - __clz(entries + szu);
    lg = lg < 6 ? 6 : (lg > ly.slots_log2 ? ly.slots_log2 : lg);
    dict.log2 = lg;
    {
      uint4* kv = reinterpret_cast<uint4*>(dict.key);
      for (int k = tid; k < (1 << lg) / 4; k += NT) kv[k] = make_uint4(~0u, ~0u, ~0u, ~0u);
    }
    if (tid == 0) {
      tb.used = tb.full = tb.inc = tb.ncand = tb.most = 0;
      tb.probes = 0;
      tb.ncol = szu;
    }
    team_sync<NW>();
    // 1. where each hyperedge of out(u) lies and its place in the list; e_u's vertices
    for (int k0 = w * 32; k0 < du; k0 += NT) {
      const int k = k0 + lane;
      uint4 rx = make_uint4(0, 0, 0, 0);
      if (k < du) {
        const int32_t x = PACKED ? (int32_t)(__ldg(o.packed + bu + k) >> 8) : __ldg(o.nbr + bu + k);
        rx = g.rec[x];
      }
      const int room = (int)((rx.z + 3u) & ~3u);
      int incl = room;
      const uint32_t out_x = __reduce_add_sync(kFull, rx.w);
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int up = __shfl_up_sync(kFull, incl, d);
        if (lane >= d) incl += up;
      }
      int at = 0;
      if (lane == 31) {
        at = atomicAdd(&tb.used, incl);
        atomicAdd(&tb.probes, (unsigned long long)out_x);
      }
      at = __shfl_sync(kFull, at, 31) + incl - room;
      rx.w = (uint32_t)at;
      if (k < du) {
        src[k] = rx;
        rows[k] = make_uint2((uint32_t)at, rx.z);
        cnt[k] = 0;
        mask[k] = 0;
      }
    }
    for (int p = tid; p < szu; p += NT) {
      const uint32_t v = (uint32_t)__ldg(g.e_idx + eb + p), h = slot_of(v, ly.bits_log2);
      dict.own(v, p);
      atomicOr(&map2[h >> 5], 1u << (h & 31u));
    }
    if (tid == 0) next.find(list, n);
    team_sync<NW>();
    // 2. the list: vertices, and the row of every group of four
    for (int k = tid / G; k < du; k += NT / G) {
      const uint4 rx = src[k];
      const int32_t* from = g.e_idx + (int64_t)(((unsigned long long)rx.y << 32) | rx.x);
      const int gl = tid % G;
      int left = (int)rx.z - gl;   // entries from this lane's on
      uint32_t* to = y + rx.w + gl;
      ROW* pr = prow + (rx.w >> 2);
      from += gl;
      for (; left > -gl; left -= G, from += G, to += G, ++pr) {
        if (left > 0) copy4(to, from);
        else *to = kPad;
        if (gl == 0) *pr = (ROW)k;
      }
    }
    copy_wait();
    team_sync<NW>();
    const int groups = tb.used >> 2;
    for (int f = tid; f < groups; f += NT) {   // vertices seen twice, or hashed like one
      const uint4 v = y4[f];
      const uint32_t h0 = slot_of(v.x, ly.bits_log2), h1 = slot_of(v.y, ly.bits_log2);
      const uint32_t h2 = slot_of(v.z, ly.bits_log2), h3 = slot_of(v.w, ly.bits_log2);
      const uint32_t b0 = 1u << (h0 & 31u), b1 = 1u << (h1 & 31u);
      const uint32_t b2 = 1u << (h2 & 31u), b3 = 1u << (h3 & 31u);
      // (padding hashes too: it can only add candidates)
      const uint32_t o0 = atomicOr(&map1[h0 >> 5], b0), o1 = atomicOr(&map1[h1 >> 5], b1);
      const uint32_t o2 = atomicOr(&map1[h2 >> 5], b2), o3 = atomicOr(&map1[h3 >> 5], b3);
      if (o0 & b0) atomicOr(&map2[h0 >> 5], b0);
      if (o1 & b1) atomicOr(&map2[h1 >> 5], b1);
      if (o2 & b2) atomicOr(&map2[h2 >> 5], b2);
      if (o3 & b3) atomicOr(&map2[h3 >> 5], b3);
    }
    team_sync<NW>();
    for (int f0 = w * 32; f0 < groups; f0 += NT) {   // candidates; the others are private
      const int f = f0 + lane;
      const uint4 v = f < groups ? y4[f] : make_uint4(kPad, kPad, kPad, kPad);
      auto twice = [&](uint32_t x) {
        const uint32_t h = slot_of(x, ly.bits_log2);
        return x != kPad && ((map2[h >> 5] >> (h & 31u)) & 1u);
      };
      const bool c0 = twice(v.x), c1 = twice(v.y), c2 = twice(v.z), c3 = twice(v.w);
      const unsigned q0 = __ballot_sync(kFull, c0), q1 = __ballot_sync(kFull, c1);
      const unsigned q2 = __ballot_sync(kFull, c2), q3 = __ballot_sync(kFull, c3);
      const int n0 = __popc(q0), n1 = n0 + __popc(q1), n2 = n1 + __popc(q2);
      int at = 0;
      if (lane == 0) at = atomicAdd(&tb.ncand, n2 + __popc(q3));
      at = __shfl_sync(kFull, at, 0);
      const unsigned lt = (1u << lane) - 1u;
      if (c0) cand[at + __popc(q0 & lt)] = (uint16_t)(4 * f);
      if (c1) cand[at + n0 + __popc(q1 & lt)] = (uint16_t)(4 * f + 1);
      if (c2) cand[at + n1 + __popc(q2 & lt)] = (uint16_t)(4 * f + 2);
      if (c3) cand[at + n2 + __popc(q3 & lt)] = (uint16_t)(4 * f + 3);
    }
    if (tid == 0) tb.next = next.u;
    team_sync<NW>();
    const int ncand = tb.ncand;
    for (int c = tid; c < ncand; c += NT) {   // handles in place of the vertices
      const int f = cand[c];
      y[f] = dict.touch(y[f], &tb.ncol, &tb.full);
    }
    team_sync<NW>();
    const int ncol = tb.ncol - szu;   // columns outside e_u
    // words per chunk: all, or the power of two that the column store holds
    const int scol = ncol + 1;        // and the empty one
    int cw = W;
    if (scol * cw > ly.swords) {
      cw = 8;
      while (cw > 1 && scol * cw > ly.swords) cw >>= 1;
    }
    const bool over = handover || tb.full != 0 || scol * cw > ly.swords;
    if (over) {   // the same on every thread: a walking team takes u
      if (tid == 0) give_back(ret, handed, handover, rule.label(du, szu), u);
    } else {
      for (int k = tid; k < scol * cw; k += NT) S[k] = 0;
      team_sync<NW>();
      // 3. masks over e_u, columns (first chunk), column lists of the rows
      int inc = 0, most = 0;
      for (int q = tid; q < ncand; q += NT) {
        const int f = cand[q], k = (int)prow[f >> 2];
        const int c = dict.col(y[f]);
        if (c >= szu) {
          if ((k >> 5) < cw) atomicOr(&S[(c - szu) * cw + (k >> 5)], 1u << (k & 31));
          const int e = (int)atomicAdd(&cnt[k], 1u);
          csr[rows[k].x + e] = (uint16_t)(c - szu);
          ++inc;
          most = e + 1 > most ? e + 1 : most;
        } else if (c >= 0) {
          atomicOr(&mask[k], 1u << c);
        }
      }
      inc = __reduce_add_sync(kFull, inc);
      most = __reduce_max_sync(kFull, most);
      if (lane == 0 && inc) {
        atomicAdd(&tb.inc, inc);
        atomicMax(&tb.most, most);
      }
      team_sync<NW>();
      if (tid == 0) {
        const int label = rule.label(du, szu);
        tb.work[label][0] += tb.probes;
        tb.work[label][1] += (unsigned long long)(g.cand[u] + szu);
        tb.work[label][2] += (unsigned long long)du;
      }
      const bool sort = tb.inc >= 2 * du;
      BitRows t;
      t.np = tb.most ? 32 - __clz(tb.most) : 0;
      // (the list sources are dead: their place takes the rows)
      finish_rows<NW>(
          tb, cnt, rows, rows2, csr, ncol, m, order, plane, du, W, szu, t.np, sort, lane, w,
          [&](int k) { return (int)rows[k].y - __popc(mask[k]) - (int)cnt[k] > 0; },
          [&](int p, int k) { return (mask[k] >> p & 1u) != 0u; });
      t.rows = rows2;
      t.csr = csr;
      t.m = m;
      t.s = S;
      t.priv = plane + kPlanes * W;
      t.plane = plane;
      t.W = W;
      t.du = du;
      t.szu = szu;
      t.cw = cw;
      // 4. rows against the columns, a chunk of cw words at a time
      for (int c0 = 0; c0 < W; c0 += cw) {
        t.c0 = c0;
        if (c0 > 0 || sort) {   // (unsorted, the first chunk is there)
          team_sync<NW>();
          for (int k = tid; k < scol * cw; k += NT) S[k] = 0;
          team_sync<NW>();
          if (ncol > 0) fill_chunk<NW, G>(S, rows2, csr, du, c0, cw);
        }
        chunk_rows<NW>(t, tb.inc >= kWideMean * du, cls, tb.hist, lane, w);
      }
    }
    u = tb.next;          // written before the barriers above
    team_sync<NW>();      // every reader is done before the next owner's writes
  }
  flush_bins<NW>(tb, cls, hist_out + (size_t)cur * kBins, lane);
  if (tid < kCloseBuckets * 3) {
    const unsigned long long x = (&tb.work[0][0])[tid];
    if (x) atomicAdd(&work[tid], x);
  }
}

// ------------------------------------------------------------------ large teams
//
// One block of 32 warps per SM.  The list does not fit beside the columns, so the
// hyperedges of out(u) are read twice, one warp per hyperedge with the next one's vertices
// in flight: once to find the shared vertices, once to write the column lists.  The vertex
// dictionary is a direct map while |V| allows, its columns in shared memory up to
// kBitDirectVertices and in scratch (L2) up to kBitMapVertices, else a hash.  Column lists stay in
// shared memory when they fit behind the dictionary, else in the block's slice of global
// scratch; the columns then take the dictionary's place.

constexpr int kLargeWarps = 32;

// f(k, place, vertex) for every hyperedge k of out(u), 32 of its vertices at a time (-1 on
// lanes past the last), one warp per hyperedge.  Four hyperedges' first 32 vertices are in
// flight at once, and the next 32 of a longer one while the current ones are used.
template <int NW, class F>
__device__ __forceinline__ void for_each_row(const DevGraph& g, const uint4* src, int du, int lane,
                                             int w, F f) {
  constexpr int U = 4;
  for (int k0 = w; k0 < du; k0 += NW * U) {
    int32_t v[U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const int k = k0 + q * NW;
      v[q] = -1;
      if (k < du) {
        const uint4 r = src[k];
        const int64_t at = (int64_t)(((unsigned long long)r.y << 32) | r.x);
        if (lane < (int)r.z) v[q] = __ldg(g.e_idx + at + lane);
      }
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const int k = k0 + q * NW;
      if (k >= du) break;
      const uint4 r = src[k];
      const int32_t* e = g.e_idx + (int64_t)(((unsigned long long)r.y << 32) | r.x);
      const int size = (int)r.z;
      int32_t x = v[q];
      for (int b = 32;; b += 32) {
        const int32_t more = b + lane < size ? __ldg(e + b + lane) : -1;
        f(k, r.w, x);
        if (b >= size) break;
        x = more;
      }
    }
  }
}

// Where the vertex dictionary of a large team lives: a hash; bit maps and columns by vertex in
// shared memory; or the bit maps there and the columns in the block's slice of scratch.
enum { kDictHash, kDictDirect, kDictMaps };

template <bool PACKED, int DICT>
__global__ void __launch_bounds__(kLargeWarps * 32, 1)
    k_bits_large(DevGraph g, Oriented o, int slots_log2, OwnerList list,
                 char* __restrict__ scratch, int64_t slice, int64_t dmax,
                 unsigned long long* __restrict__ hist_out, unsigned long long* __restrict__ work,
                 TeamRule rule, int32_t* __restrict__ counter, ReturnLists ret, OwnerList handed,
                 int handover) {
  constexpr int NW = kLargeWarps, NT = NW * 32, G = 8;
  constexpr bool DIRECT = DICT != kDictHash;
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ TeamBlock tb;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, tid = threadIdx.x;
  uint4* gsrc = reinterpret_cast<uint4*>(scratch + slice * blockIdx.x);   // [dmax]
  uint16_t* gcsr = reinterpret_cast<uint16_t*>(gsrc + dmax);
  uint16_t* gval = reinterpret_cast<uint16_t*>(scratch + slice * (blockIdx.x + 1) -
                                               bits_val_bytes(g.nv));
  for (int k = tid; k < kBins; k += NT) tb.hist[k] = 0;
  for (int k = tid; k < kCloseBuckets * 3; k += NT) (&tb.work[0][0])[k] = 0;
  const int32_t n = *list.n;
  uint32_t cls[kClasses];
#pragma unroll
  for (int q = 0; q < kClasses; ++q) cls[q] = 0;
  unsigned long long since_flush = 0;
  int32_t cur = 0;
  NextOwner next{0, -1};
  if (tid == 0) {
    next.fetch(counter);
    next.find(list, n);
    tb.next = next.u;
  }
  __syncthreads();
  int32_t u = tb.next;
  while (u >= 0) {
    const uint4 hu = g.rec[u];
    const int64_t bu = o.row_ptr[u];
    if (tid == 0) next.fetch(counter);
    const int32_t mem = member_of(g, u);
    if (mem != cur || since_flush > (1ull << 30)) {
      flush_bins<NW>(tb, cls, hist_out + (size_t)cur * kBins, lane);
      cur = mem;
      since_flush = 0;
    }
    const int32_t du = (int32_t)hu.w, szu = (int32_t)hu.z;
    const int64_t eb = (int64_t)(((unsigned long long)hu.y << 32) | hu.x);
    const int W = (du + 31) >> 5;
    since_flush += (unsigned long long)du * (unsigned long long)du / 2;
    // layout of this u: digits and flags, columns of e_u, rows, then the region X
    uint32_t at = 0;
    auto take = [&](uint32_t bytes) {
      const uint32_t p = at;
      at += (bytes + 15u) & ~15u;
      return p;
    };
    uint32_t* plane = reinterpret_cast<uint32_t*>(dyn + take(4u * (kPlanes + 1) * W));
    uint32_t* m = reinterpret_cast<uint32_t*>(dyn + take(4u * szu * W));
    uint32_t* m2 = reinterpret_cast<uint32_t*>(dyn + take(4u * szu * W));
    uint2* rows = reinterpret_cast<uint2*>(dyn + take(8u * du));
    uint2* rows2 = reinterpret_cast<uint2*>(dyn + take(8u * du));
    uint32_t* cnt = reinterpret_cast<uint32_t*>(dyn + take(4u * du));
    uint16_t* order = reinterpret_cast<uint16_t*>(dyn + take(2u * du));
    uint8_t* priv = reinterpret_cast<uint8_t*>(dyn + take(du));
    const uint32_t x0 = at;
    Dict<DIRECT> dict;
    dict.log2 = slots_log2;
    dict.words = (g.nv + 31) / 32;
    const uint32_t key_bytes = DIRECT ? 8u * (uint32_t)dict.words : 4u << slots_log2;
    dict.key = reinterpret_cast<uint32_t*>(dyn + take(key_bytes));
    dict.val = DICT == kDictMaps
                   ? gval
                   : reinterpret_cast<uint16_t*>(
                         dyn + take(DIRECT ? 2u * (uint32_t)g.nv : 2u << slots_log2));
    // the hyperedges' places in e_idx: in X when they fit, else in global scratch
    const uint32_t src_at = take(16u * du);
    const bool src_in = at <= (uint32_t)kBitSmem;
    if (!src_in) at = src_at;
    uint4* src = src_in ? reinterpret_cast<uint4*>(dyn + src_at) : gsrc;
    const bool fits = at <= (uint32_t)kBitSmem;
    // 0.
    if (fits) {
      for (uint32_t k = tid; k < key_bytes / 4u; k += NT) dict.key[k] = DIRECT ? 0u : ~0u;
      for (int k = tid; k < szu * W; k += NT) m[k] = 0;
    }
    if (tid == 0) {
      tb.ncol = szu;
      tb.most = tb.full = tb.used = tb.inc = 0;
      tb.probes = 0;
    }
    __syncthreads();
    // 1. rows and their places in the column lists; e_u's vertices
    if (fits) {
      for (int p = tid; p < szu; p += NT) dict.own((uint32_t)__ldg(g.e_idx + eb + p), p);
      for (int k0 = w * 32; k0 < du; k0 += NT) {
        const int k = k0 + lane;
        uint4 rx = make_uint4(0, 0, 0, 0);
        if (k < du) {
          const int32_t x = PACKED ? (int32_t)(__ldg(o.packed + bu + k) >> 8)
                                   : __ldg(o.nbr + bu + k);
          rx = g.rec[x];
        }
        const int room = (int)((rx.z + 3u) & ~3u);
        unsigned long long out_x = rx.w;
        int incl = room;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int up = __shfl_up_sync(kFull, incl, d);
          if (lane >= d) incl += up;
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) out_x += __shfl_down_sync(kFull, out_x, d);
        int before = 0;
        if (lane == 31) before = atomicAdd(&tb.used, incl);
        before = __shfl_sync(kFull, before, 31) + incl - room;
        if (lane == 0) atomicAdd(&tb.probes, out_x);
        rx.w = (uint32_t)before;
        if (k < du) src[k] = rx;
      }
    }
    if (tid == 0) next.find(list, n);
    __syncthreads();
    bool over = !fits || handover;
    const int used = tb.used;
    // column lists at the end of shared memory when the region X holds them too
    const uint32_t csr_bytes = (2u * (uint32_t)used + 15u) & ~15u;
    const bool inside = at + csr_bytes <= (uint32_t)kBitSmem;
    uint16_t* csr = inside ? reinterpret_cast<uint16_t*>(dyn + kBitSmem - csr_bytes) : gcsr;
    const int swords = (int)(((uint32_t)kBitSmem - (inside ? csr_bytes : 0u) - x0) / 4u);
    uint32_t* S = reinterpret_cast<uint32_t*>(dyn + x0);
    int ncol = 0, cw = 1;
    BitRows t;
    if (!over) {
      // 2. shared vertices
      for_each_row<NW>(g, src, du, lane, w, [&](int, uint32_t, int32_t v) {
        // (once a hash is full, every further vertex would take all its probes for nothing)
        if (v >= 0 && (DIRECT || !*(volatile int*)&tb.full))
          dict.touch((uint32_t)v, &tb.ncol, &tb.full);
      });
      if (tid == 0) tb.next = next.u;
      __syncthreads();
      over = tb.full != 0;
    } else if (tid == 0) {
      tb.next = next.u;
    }
    if (!over) {
      // 3. column lists, columns of e_u, private flags
      int last = -1, c_n = 0, inc = 0, most = 0;   // entries of row `last` so far
      for_each_row<NW>(g, src, du, lane, w, [&](int k, uint32_t place, int32_t v) {
        if (k != last) {
          last = k;
          c_n = 0;
          if (lane == 0) priv[k] = 0;
        }
        const int c = v >= 0 ? dict.find((uint32_t)v) : 0;
        const bool alone = v >= 0 && c < 0, own = v >= 0 && c >= 0 && c < szu, out = c >= szu;
        const unsigned bal = __ballot_sync(kFull, out);
        if (__any_sync(kFull, alone) && lane == 0) priv[k] = 1;
        if (own) atomicOr(&m[c * W + (k >> 5)], 1u << (k & 31));
        if (out) csr[place + c_n + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(c - szu);
        c_n += __popc(bal);
        inc += __popc(bal);
        most = c_n > most ? c_n : most;
        if (lane == 0) {
          rows[k] = make_uint2(place, 0);
          cnt[k] = (uint32_t)c_n;
        }
      });
      if (lane == 0) {
        atomicAdd(&tb.inc, inc);
        atomicMax(&tb.most, most);
      }
      __syncthreads();
      t.np = tb.most ? 32 - __clz(tb.most) : 0;
      ncol = tb.ncol - szu;
      finish_rows<NW>(
          tb, cnt, rows, rows2, csr, ncol, m2, order, plane, du, W, szu, t.np, true, lane, w,
          [&](int k) { return priv[k] != 0; },
          [&](int p, int k) { return (m[p * W + (k >> 5)] >> (k & 31) & 1u) != 0u; });
      // words per chunk: a multiple of 4 while that fits
      cw = swords / (ncol + 1);
      if (cw >= W) cw = W;
      else if (cw >= 4) cw &= ~3;
      over = cw < 1;
    }
    if (over) {
      if (tid == 0) give_back(ret, handed, handover, rule.label(du, szu), u);
    } else {
      if (tid == 0) {
        const int label = rule.label(du, szu);
        tb.work[label][0] += tb.probes;
        tb.work[label][1] += (unsigned long long)(g.cand[u] + szu);
        tb.work[label][2] += (unsigned long long)du;
      }
      t.rows = rows2;
      t.csr = csr;
      t.m = m2;
      t.s = S;
      t.priv = plane + kPlanes * W;
      t.plane = plane;
      t.W = W;
      t.du = du;
      t.szu = szu;
      t.cw = cw;
      for (int c0 = 0; c0 < W; c0 += cw) {
        t.c0 = c0;
        for (int k = tid; k < (ncol + 1) * cw; k += NT) S[k] = 0;
        __syncthreads();
        fill_chunk<NW, G>(S, rows2, csr, du, c0, cw);
        chunk_rows<NW>(t, tb.inc >= kWideMean * du, cls, tb.hist, lane, w);
        __syncthreads();
      }
    }
    __syncthreads();
    u = tb.next;
    __syncthreads();
  }
  flush_bins<NW>(tb, cls, hist_out + (size_t)cur * kBins, lane);
  if (tid < kCloseBuckets * 3) {
    const unsigned long long x = (&tb.work[0][0])[tid];
    if (x) atomicAdd(&work[tid], x);
  }
}

// ------------------------------------------------------------------ shapes

struct Shape {
  int nw;           // warps
  int minb;         // blocks per SM the registers are held to
  int icap_log2, map_log2, slots_log2, dcap, mwords, swords;
};
// Teams of the list classes kListBits .. kListBits + 4 (bit_class_of has the same limits).
// map_log2: bits of one seen-twice map, 16 per entry (one unshared entry in 16 passes) while
// that fits, 8 for the largest; the two maps later hold the column lists (2 bytes per entry).
constexpr Shape kShapes[kBitClasses - 1] = {
    {2, 16, 9, 13, 9, 64, 128, 512},
    {4, 8, 10, 14, 10, 128, 256, 1536},
    {8, 4, 11, 15, 11, 256, 512, 3072},
    {16, 2, 12, 15, 12, 512, 1024, 8192},
    {32, 1, 13, 16, 13, 1024, 2048, 10240},
};

constexpr SmallLayout small_layout(int c) {
  const Shape sh = kShapes[c];
  SmallLayout l{};
  l.icap = 1 << sh.icap_log2;
  l.dcap = sh.dcap;
  l.mwords = sh.mwords;
  l.swords = sh.swords;
  l.slots_log2 = sh.slots_log2;
  l.bits_log2 = sh.map_log2;
  const uint32_t icap = (uint32_t)l.icap, dcap = (uint32_t)l.dcap;
  const uint32_t sizes[13] = {4u * icap,                          // list
                              (2u << l.bits_log2) / 8u,           // two maps, column lists
                              2u * icap,                          // candidates
                              4u << l.slots_log2, 2u << l.slots_log2,   // dictionary
                              16u * dcap, 8u * dcap, 4u * dcap, 4u * dcap,   // per row
                              (dcap <= 256 ? 1u : 2u) * icap / 4u,      // row of every group
                              4u * (kPlanes + 1) * ((dcap + 31u) / 32u),
                              4u * (uint32_t)sh.mwords, 4u * (uint32_t)sh.swords};
  uint32_t off[13] = {}, at = 0;
  for (int k = 0; k < 13; ++k) {
    off[k] = at;
    at += (sizes[k] + 15u) & ~15u;
  }
  l.off_y = off[0];
  l.off_map = off[1];
  l.off_list = off[2];
  l.off_key = off[3];
  l.off_val = off[4];
  l.off_src = off[5];
  l.off_rows = off[6];
  l.off_cnt = off[7];
  l.off_mask = off[8];
  l.off_prow = off[9];
  l.off_plane = off[10];
  l.off_m = off[11];
  l.off_s = off[12];
  l.bytes = at;
  return l;
}

template <int C, bool PACKED>
void launch_small(const CloseRun& r, const OwnerList& list, int32_t n, const ReturnLists& ret,
                  unsigned long long* work, const TeamRule& rule, int32_t* counter) {
  constexpr Shape sh = kShapes[C];
  using ROW = typename std::conditional<(sh.dcap <= 256), uint8_t, uint16_t>::type;
  auto kern = k_bits_small<sh.nw, sh.minb, PACKED, ROW>;
  constexpr SmallLayout ly = small_layout(C);
  static_assert(ly.bytes <= (uint32_t)kBitSmem, "shared memory of a block");
  static_assert((2u << ly.bits_log2) / 8u >= 2u * (uint32_t)ly.icap, "column lists in the maps");
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ly.bytes);
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, sh.nw * 32, ly.bytes);
  if (per_sm < 1) per_sm = 1;
  const int blocks = n < per_sm * r.nsm ? n : per_sm * r.nsm;
  note_launch();
  kern<<<blocks, sh.nw * 32, ly.bytes, r.s>>>(r.g, r.o, ly, list, r.hist, work, rule, counter, ret,
                                              r.over, r.handover);
}

template <bool PACKED, int DICT>
void launch_large(const CloseRun& r, const OwnerList& list, int32_t n, const ReturnLists& ret,
                  void* scratch, int64_t slice, int64_t dmax, int blocks,
                  unsigned long long* work, const TeamRule& rule, int32_t* counter) {
  auto kern = k_bits_large<PACKED, DICT>;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kBitSmem);
  note_launch();
  kern<<<blocks < n ? blocks : n, kLargeWarps * 32, kBitSmem, r.s>>>(
      r.g, r.o, kBitLargeSlots, list, (char*)scratch, slice, dmax, r.hist, work, rule, counter, ret,
      r.over, r.handover);
}

}  // namespace

int64_t bits_slice_bytes(int64_t dmax, int64_t imax, int64_t nv) {
  return 16 * ((dmax + 15) / 16 * 16) + (2 * imax + 255) / 256 * 256 + bits_val_bytes(nv);
}

cudaError_t launch_close_bits(int c, const CloseRun& r, const OwnerList& list, int32_t n,
                              const ReturnLists& ret, void* scratch, int64_t slice, int64_t dmax,
                              int blocks_max, unsigned long long* work, const TeamRule& rule,
                              int32_t* counter) {
  if (n <= 0) return cudaSuccess;
#define HG_SMALL(C)                                                                     \
  (r.packed ? launch_small<C, true>(r, list, n, ret, work, rule, counter)               \
            : launch_small<C, false>(r, list, n, ret, work, rule, counter))
#define HG_LARGE(D)                                                                              \
  (r.packed ? launch_large<true, D>(r, list, n, ret, scratch, slice, dmax, blocks_max, work, rule, \
                                    counter)                                                     \
            : launch_large<false, D>(r, list, n, ret, scratch, slice, dmax, blocks_max, work,    \
                                     rule, counter))
  switch (c) {
    case 0: HG_SMALL(0); break;
    case 1: HG_SMALL(1); break;
    case 2: HG_SMALL(2); break;
    case 3: HG_SMALL(3); break;
    case 4: HG_SMALL(4); break;
    default:
      if (r.g.nv <= kBitDirectVertices) HG_LARGE(kDictDirect);
      else if (r.g.nv <= kBitMapVertices) HG_LARGE(kDictMaps);
      else HG_LARGE(kDictHash);
  }
#undef HG_SMALL
#undef HG_LARGE
  return cudaGetLastError();
}

}  // namespace hg
