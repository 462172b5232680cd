// Internal declarations shared by the CUDA translation units of libhg.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "hg.h"

namespace hg {

constexpr int kWarp = 32;

// Error words written by kernels (first writer wins via atomicCAS).
enum DevErr : int {
  DE_OK = 0,
  DE_EMPTY = 1,
  DE_RANGE = 2,
  DE_DUPV = 3,
  DE_UNSORTED = 4,
  DE_DUPEDGE = 5,
  DE_PTR = 6,       // edge_ptr not monotone / out of [0, nnz]
  DE_INTERNAL = 7,  // a kernel-side consistency check failed
  DE_LIMIT = 8,     // an input row beyond a kernel's fixed capacity
  DE_TIMEOUT = 9,   // a bounded device wait gave up
};

__device__ __forceinline__ void dev_fail(int* err, int code) { atomicCAS(err, 0, code); }

// Oriented wedge entries.  Packed: (nbr << 8) | omega, used when |E| < 2^24 and
// every omega < 256; otherwise nbr and omega live in two int32 arrays.
struct Oriented {
  int64_t* row_ptr;   // [ne+1] start of row i (capacity deg(i))
  int32_t* dplus;     // [ne] used length of row i
  uint32_t* packed;   // [2W] packed entries, or nullptr
  int32_t* nbr;       // [2W] wide entries, or nullptr
  int32_t* omega;     // [2W]
  int64_t slots;      // entries the arrays hold (0 = not recorded)
};

struct DevGraph {
  int32_t nv, ne;
  int64_t nnz;
  const int64_t* e_ptr;
  const int32_t* e_idx;
  const int32_t* esize;
  const int64_t* v_ptr;
  const int32_t* v_idx;
  // a batch of disjoint member hypergraphs: member m owns hyperedges
  // [m_eoff[m], m_eoff[m+1]); nm == 0 for a single hypergraph
  const int32_t* m_eoff;
  int32_t nm;
  // step two, set once the build is done (null before): per hyperedge x its start in e_idx
  // (two words), |e_x| and its out-degree in one 16-byte record; osum[u] = sum over
  // x in out(u) of |e_x| rounded up to a multiple of four, dsum[u] = the sum of their degrees
  // (both at most 2^31 - 1); cand[u] = sum over its vertices of |E_y| - 1
  const uint4* rec;
  const int32_t* osum;
  const int32_t* dsum;
  const int64_t* cand;
};

// member owning hyperedge u (0 for a single hypergraph)
__device__ __forceinline__ int32_t member_of(const DevGraph& g, int32_t u) {
  int32_t lo = 0, hi = g.nm > 0 ? g.nm - 1 : 0;
  while (lo < hi) {
    const int32_t mid = (lo + hi + 1) >> 1;
    if (__ldg(g.m_eoff + mid) <= u) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// ---------------- launch wrappers (implemented in the .cu files) ----------------

// process-wide count of kernel launches made by the library (defined in hg_api.cu)
void note_launch(int n = 1);

// k_scan.cu
// out[0..n] = exclusive prefix sums of in[0..n) (out[n] = total); tmp >= scan_tmp_bytes(n).
size_t scan_tmp_bytes(int64_t n);
void scan_i32_to_i64(const int32_t* in, int64_t* out, int64_t n, void* tmp, cudaStream_t s);
void scan_i64_to_i64(const int64_t* in, int64_t* out, int64_t n, void* tmp, cudaStream_t s);
// acc[0] += sum C(x,2), acc[1] = max x, acc[2] += sum x over x in deg (dplus) [0..n), and
// ds[i] = (deg[i], esize[i]) (rec[i] = (e_ptr[i] in two words, esize[i], dplus[i]))
void launch_deg_stats(const int32_t* deg, const int32_t* esize, int64_t n,
                      unsigned long long* acc, int2* ds, cudaStream_t s);
void launch_out_stats(const int32_t* dplus, const int64_t* e_ptr, const int32_t* esize, int64_t n,
                      unsigned long long* acc, uint4* rec, cudaStream_t s);

// k_load.cu
// One thread waits until *flag != 0, at most limit_ns of the global timer (and a bounded
// number of polls), else records DE_TIMEOUT in *err.
void launch_wait_flag(const int32_t* flag, int64_t limit_ns, int* err, cudaStream_t s);
void launch_check_ptr(const int64_t* e_ptr, int32_t ne, int64_t nnz, int* err, cudaStream_t s);
void launch_validate_rows(const DevGraph& g, int32_t* esize, int32_t* vdeg, int* err,
                          cudaStream_t s);
void launch_scatter(const DevGraph& g, int32_t* cursor, int32_t* v_idx, const int* err,
                    cudaStream_t s);
// cand[i] = sum_{v in e_i} (|E_v| - 1); also bucket rows by cand into lists
void launch_candidates(const DevGraph& g, int64_t* cand, unsigned long long* max_cand,
                       int32_t* max_size, const int* err, cudaStream_t s);

// k_dense.cu: heavy x heavy omega on the tensor cores
struct DenseInfo {
  const int32_t* heavy_idx;   // [ne] position in the heavy list or -1; nullptr = no dense path
  const int32_t* ids;         // [nh] hyperedge id of each heavy position
  const uint16_t* omega;      // [rows_pad x rows_pad] omega of heavy pairs
  int64_t ld;                 // row stride of omega
  int32_t nh;
  const int2* hrange;         // a batch: [first, end) heavy positions of every member; else null
};
size_t dense_smem_bytes();
int64_t dense_round_rows(int64_t n);
int64_t dense_round_k(int64_t k);
void launch_size_hist(const int32_t* esize, int32_t ne, int32_t max_bin, unsigned long long* hist,
                      cudaStream_t s);
// heavy: min_size <= |e_i| <= max_size, at most cap of them
void launch_pick_heavy(const int32_t* esize, int32_t ne, int32_t min_size, int32_t max_size,
                       int32_t cap, int32_t* heavy_idx, int32_t* ids, int32_t* count,
                       cudaStream_t s);
// omega values the tile kernel writes exactly (uint16 output)
constexpr int32_t kDenseMaxOmega = 65535;
// the same for a batch, member by member: flag[i], then (rank = prefix sums of flag) places and
// every member's range of heavy positions (hrange cleared before)
void launch_heavy_flags(const int32_t* esize, int32_t ne, int32_t min_size, int32_t max_size,
                        int32_t* flag, cudaStream_t s);
void launch_heavy_place(const DevGraph& g, const int32_t* flag, const int64_t* rank, int32_t cap,
                        int32_t* heavy_idx, int32_t* ids, int32_t* count, int2* hrange,
                        cudaStream_t s);
// a batch's tiles with work (at most dense_tiles(rows_pad)) and their number
int64_t dense_tiles(int64_t rows_pad);
void launch_tile_list(const DevGraph& g, const int32_t* ids, int32_t nh, const int32_t* voff,
                      int64_t rows_pad, int4* list, int32_t* list_n, cudaStream_t s);
// voff: member vertex offsets (columns are member-local then), or null
void launch_fill_dense(const DevGraph& g, const int32_t* ids, int32_t nh, uint8_t* a, int64_t lda,
                       const int32_t* voff, cudaStream_t s);
// list, list_n: launch_tile_list's, or null (every tile, every step of K)
cudaError_t launch_dense_omega(const uint8_t* a, int64_t rows, int64_t rows_pad, int64_t k_pad,
                               const int4* list, const int32_t* list_n, uint16_t* omega, int* err,
                               cudaStream_t s);

// k_wedge.cu
struct WedgeBuckets {
  int32_t* rows[3];  // light (warp), medium (block, smem), heavy (block, global scratch)
  int32_t* count;    // [3] device counters
};
// rows gathering at most light_max incidences take one warp (light_max <= wedge_light_max_cand)
void launch_bucket_rows(const int64_t* cand, int32_t ne, WedgeBuckets b, int light_max,
                        cudaStream_t s);
// the largest gather count of a one-warp row in the packed (1) or unpacked (0) layout
int wedge_light_max_cand(int packed);
int wedge_medium_max_cand();
// Per-row outputs of the count pass (each may be null): upc[i] = |{j > i}|,
// wcr[i] = |{j > i : omega_ij = min(|e_i|, |e_j|)}| (inclusion-type hyperwedges).
struct RowCounts {
  int32_t* upc;
  int32_t* wcr;
};

// The gather pass of step one: deg(i), RowCounts, W_c into *wc, the duplicate check,
// and every (j, omega_ij) of row i written from rows.row_ptr[i] (a capacity layout:
// room for cap[i] = min(gathered incidences, |E| - 1) entries, see launch_cap_rows).
void launch_wedge_rows(const DevGraph& g, const WedgeBuckets& b, const int32_t* nb,
                       int64_t heavy_max_cand, const int64_t* cand, int32_t* deg,
                       unsigned long long* wc, const Oriented& rows, int packed,
                       unsigned long long* scratch, int* err, int32_t* work_counter,
                       const DenseInfo& dense, RowCounts rc, cudaStream_t s, int nsm);
void launch_cap_rows(const int64_t* cand, int32_t ne, int32_t* cap, cudaStream_t s);
// Filter rows of the capacity layout (len[i] entries from src_ptr[i]) into an exact layout
// (row i from dst_ptr[i]), order kept: keep 0 = j ranked above i in (deg, id), 1 = j > i,
// 2 = all.  count_only: write the number kept to cnt[i] instead.
// ds: (deg, |e|) of every hyperedge (keep 0 only); osum, dsum (keep 0, may be null): see
// DevGraph.
void launch_filter_rows(int keep, bool count_only, const int64_t* src_ptr, const int32_t* len,
                        const Oriented& src, const int2* ds, int32_t ne, int packed,
                        const int64_t* dst_ptr, const Oriented& dst, int32_t* cnt,
                        int32_t* osum, int32_t* dsum, cudaStream_t s);

// hg_api.cu: allocations of the calling thread skip the caller-installed hooks
void alloc_bypass_hooks(bool on);
// Device memory of a built handle: what it holds, how much of that is rows of packed entries
// (twice as large unpacked), and what a count of it would take beside.  The last finds the
// owners of every closure list on the device; a count made before is forgotten.
struct HandleBytes {
  size_t held = 0, packed_rows = 0, count = 0;
};
hg_status handle_bytes(hg_graph* g, HandleBytes* out);

// k_batch.cu
void launch_sub_base(int64_t* e_ptr, int32_t ne, int64_t base, cudaStream_t s);
void launch_add_member_base(int64_t* e_ptr, int32_t ne, const int32_t* m_eoff, int32_t nm,
                            const int64_t* noff, cudaStream_t s);
void launch_localize(const DevGraph& g, const int32_t* m_voff, int32_t* e_idx, int* err,
                     cudaStream_t s);
void launch_member_stats(const DevGraph& g, const int32_t* deg, const int32_t* wcr,
                         unsigned long long* out, cudaStream_t s);

// k_sample.cu
int sample_sort_max_log2();
void sample_set_lut(const uint8_t lut[128], cudaStream_t s);
// max_len: an upper bound of the row lengths
cudaError_t launch_sort_upper(const int64_t* up_ptr, int32_t ne, const Oriented& up, int packed,
                              uint64_t max_len, int* err, cudaStream_t s, int nsm);
// Bucket index of a row-pointer array of `entries` entries over ne rows (sampler row
// searches): row_index_buckets(entries, row_index_shift(entries, ne)) + 1 int32.
int row_index_shift(uint64_t entries, int32_t rows);
int64_t row_index_buckets(uint64_t entries, int shift);
void launch_row_index(const int64_t* ptr, int32_t ne, uint64_t entries, int32_t* first,
                      cudaStream_t s);
// work (may be null): [0] row-pointer reads, [1] upper-row entries read, [2] vertex ids merged;
// up_index (may be null): the bucket index of up_ptr
void launch_sample(const DevGraph& g, const int64_t* up_ptr, const int32_t* up_index,
                   const Oriented& up, int packed, uint64_t W, uint64_t seed, uint64_t first,
                   uint64_t num, unsigned long long* raw, unsigned long long* work, cudaStream_t s,
                   int nsm);
// Appro-adv (Algorithm 7)
void launch_type_counts(const int32_t* upc, const int32_t* wcr, int32_t ne, int32_t* cnt_t,
                        cudaStream_t s);
void launch_split_types(const DevGraph& g, const int64_t* up_ptr, const Oriented& up, int packed,
                        const int64_t* t_ptr, const Oriented& t, const int64_t* c_ptr,
                        const Oriented& c, cudaStream_t s);
void launch_sample_adv(const DevGraph& g, const int64_t* set_ptr, const int32_t* set_index,
                       const Oriented& set_ent, uint64_t Wx, int type, int cls, uint32_t stream,
                       const int64_t* full_ptr, const Oriented& full, int packed, uint64_t seed,
                       uint64_t first, uint64_t num, unsigned long long* raw, cudaStream_t s,
                       int nsm);
// single-pattern enumeration over the upper rows
void launch_enumerate(const DevGraph& g, const int64_t* up_ptr, const int32_t* up_index,
                      const Oriented& up, int packed, uint64_t W, int target, int32_t* out,
                      unsigned long long cap, unsigned long long* count, cudaStream_t s, int nsm);
// the sub-hypergraph G' of Algorithms 6-7 (sigma < 1)
void launch_priority(int32_t ne, uint64_t seed, unsigned long long* pr, cudaStream_t s);
void launch_digit_hist(const unsigned long long* pr, int32_t ne, int shift,
                       unsigned long long pmask, unsigned long long prefix, unsigned int* hist,
                       cudaStream_t s);
void launch_equal_flags(const unsigned long long* pr, int32_t ne, unsigned long long T,
                        int32_t* eq, cudaStream_t s);
void launch_keep_flags(const unsigned long long* pr, int32_t ne, unsigned long long T,
                       const int64_t* eq_rank, int64_t need, int32_t* keep, cudaStream_t s);
void launch_compact_kept(const int32_t* keep, const int64_t* pos, const int32_t* esize, int32_t ne,
                         int32_t* ids, int32_t* sizes, cudaStream_t s);
void launch_gather_rows(const int64_t* e_ptr, const int32_t* e_idx, const int32_t* ids, int32_t nk,
                        const int64_t* sub_ptr, int32_t* sub_idx, cudaStream_t s);
size_t wedge_heavy_scratch_bytes(int64_t heavy_max_cand, int nsm);

// Step two.  Shapes a caller sees (hg_close_stats): by out-degree and |e_u|, see
// TeamRule::label.  Lists of owners the kernels take: one per kernel shape.
constexpr int kCloseBuckets = 8;
constexpr int kWideBucket = 6;
constexpr int kClusterBucket = 7;
constexpr int kWideLargeMin = 4096;
constexpr int kWarpMaskBits = 32;         // one-word masks of the warp teams
constexpr int kBlockMaxPacked = 6144;
constexpr int kBlockMaxUnpacked = 4096;

struct TeamRule {
  int all_wide;    // every owner to the global-table blocks
  int warp_max;    // largest out-degree labelled a warp team (64, 128 or 256)
  int block_max;   // largest out-degree labelled a block team
  // shape of an owner with out-degree d and sz vertices (-1: it closes nothing)
  __host__ __device__ int label(int32_t d, int32_t sz) const {
    if (d < 2) return -1;
    if (all_wide) return kWideBucket;
    if (sz <= kWarpMaskBits && d <= warp_max) return d <= 64 ? 0 : (d <= 128 ? 1 : 2);
    if (sz <= kWarpMaskBits && d <= 1024) return 3;
    if (sz <= kWarpMaskBits && d <= 2048) return 4;
    if (sz <= kWarpMaskBits && d <= block_max) return 5;
    return d > kWideLargeMin ? kClusterBucket : kWideBucket;
  }
};

// Lists of owners: the walking teams by label (warp teams 0-2, block teams with shared tables
// 3-5, global-table blocks and clusters), the bit-row classes, and the owners that a walking
// team handed over to the global-table blocks.
constexpr int kListWide = kWideBucket;
constexpr int kListCluster = kClusterBucket;
constexpr int kListBits = kCloseBuckets;
constexpr int kBitClasses = 6;
constexpr int kListOver = kListBits + kBitClasses;
constexpr int kLists = kListOver + 1;

// A list of owners on the device: entry k at at[k * step], its length at *n.  Two lists share
// an array of |E| entries where no owner can be in both, one from each end.
struct OwnerList {
  int32_t* at;
  int32_t step;
  int32_t* n;
#ifdef __CUDACC__
  __device__ __forceinline__ int32_t get(int32_t k) const { return at[(int64_t)k * step]; }
  __device__ __forceinline__ void put(int32_t u) const {
    at[(int64_t)atomicAdd(n, 1) * step] = u;
  }
#endif
};
constexpr int kWalkRatio0 = 8, kWalkRatio3 = 40, kWalkRatio4 = 80;   // see list_of in k_close.cu
constexpr int kWalkRatioWide = 8;
constexpr int kBitMaxOut = 8192;             // bit rows: out-degree, column-list entries
constexpr int kBitMaxEntries = 1 << 22;
// Direct vertex map up to kBitDirectVertices; its bit maps alone in shared memory up to
// kBitMapVertices (at most 64 KB, less than the hash), its columns in global scratch.  Beyond,
// a hash of 16,384 vertices: closure of a tag shape of 200,000 hyperedges over 40,000 vertices
// 1.56 with the hash and 0.35 s with the maps, of 300,000 over 100,000 3.79 and 0.52 (block
// teams: 1.08, 1.57).  An owner that fills the hash goes to the block teams after its vertices
// were read, so the hash is tried up to kBitHashEntries of osum + |e_u| (closure of 60,000 and
// 300,000 tag-shaped hyperedges over 300,000 vertices, ms: never 195, 1,389; 16,384 190, 1,356;
// 32,768 155, 1,170; 65,536 126, 1,248; 131,072 130, 1,441).
constexpr int kBitDirectVertices = 32768;
constexpr int kBitMapVertices = 262144;
constexpr int kBitHashEntries = 65536;

constexpr int kBitSmem = 232448 - 2048;      // dynamic shared memory a block may take
constexpr int kBitPlanes = 16;               // digits of a shared count (<= 65,535)
constexpr int kBitLargeSlots = 14;           // log2 slots of the last class's hash dictionary

// Shared memory of the last class: digits and flags, e_u's columns twice and the rows, then the
// vertex dictionary, whose place the columns take later.
__host__ __device__ inline int64_t bit_rows_bytes(int64_t du, int64_t szu) {
  const int64_t W = (du + 31) / 32;
  return 4 * (kBitPlanes + 1) * W + 8 * szu * W + 23 * du + 256;
}
__host__ __device__ inline int64_t bit_large_bytes(int64_t du, int64_t szu, int64_t nv) {
  return bit_rows_bytes(du, szu) +
         (nv <= kBitMapVertices ? 8 * ((nv + 31) / 32) + (nv <= kBitDirectVertices ? 2 * nv : 0)
                                : 6ll << kBitLargeSlots);
}

// Global scratch of a block for the columns by vertex.
__host__ __device__ inline int64_t bits_val_bytes(int64_t nv) {
  return nv > kBitDirectVertices && nv <= kBitMapVertices ? (2 * nv + 255) / 256 * 256 : 0;
}

// Smallest bit-row class that holds an owner (k_bits.cu, kShapes), -1 for none.  osum: see
// DevGraph (an upper bound of the column list, and with szu of the dictionary's keys).
__host__ __device__ inline int bit_class_of(int64_t du, int64_t szu, int64_t osum, int64_t nv) {
  const int64_t mw = szu * ((du + 31) / 32), e = osum + szu;
  if (szu <= kWarpMaskBits) {
    if (du <= 64 && e <= 512 && mw <= 128) return 0;
    if (du <= 128 && e <= 1024 && mw <= 256) return 1;
    if (du <= 256 && e <= 2048 && mw <= 512) return 2;
    if (du <= 512 && e <= 4096 && mw <= 1024) return 3;
    if (du <= 1024 && e <= 8192 && mw <= 2048) return 4;
  }
  // (32 KB of columns at least)
  if (du <= kBitMaxOut && e <= kBitMaxEntries && szu <= 4096 &&
      bit_large_bytes(du, szu, nv) <= kBitSmem - 32768)
    return 5;
  return -1;
}

// k_close.cu
struct CloseLists {
  OwnerList list[kLists];
  int32_t* labels;        // [kCloseBuckets] owners per label
  unsigned long long* maxima;   // largest [0] out-degree, [1] |e_u| of the labels 6 and 7,
                                // [2], [3] of the others, [4] osum, [5] out-degree of the
                                // last bit class
};
// sel: NULL, or one byte per hyperedge; then only the hyperedges u with sel[u] != 0
// get a team (the hyper-triangles they own).
void launch_bucket_close(const DevGraph& g, const Oriented& o, CloseLists b, const TeamRule& rule,
                         const uint8_t* sel, cudaStream_t s);
// What every kernel of a count shares.
struct CloseRun {
  DevGraph g;
  Oriented o;
  int packed;
  unsigned long long* hist;
  OwnerList over;   // owners that the walking teams' tables cannot hold (every one of the warp,
  int handover;     // block and bit-row teams when handover is set)
  cudaStream_t s;
  int nsm;
};
// Scratch of the global-table teams.
struct WideSpace {
  int64_t cap = 16, words = 1, dmax = 1;
  void* scratch = nullptr;
};
// list_id: a walking team's list or kListOver; n: its length, or an upper bound (sizes the
// grid; the kernel reads the length on the device); counter: zeroed fetch counter; work[0] +=
// probes, work[1] += E_y entries, work[2] += out-entries (hg_close_stats)
cudaError_t launch_close(int list_id, const CloseRun& r, const OwnerList& list, int32_t n,
                         const WideSpace& w, unsigned long long* work, int32_t* counter);
// k_bits.cu: the owners of bit-row class c.  work: [kCloseBuckets][3] as above, by label.
// back[label]: the walking team's list that an owner whose tables overflow goes to.  The last
// class keeps `slice` bytes of scratch per block, at most blocks_max blocks.
struct ReturnLists {
  OwnerList back[kCloseBuckets];
};
int64_t bits_slice_bytes(int64_t dmax, int64_t imax, int64_t nv);
cudaError_t launch_close_bits(int c, const CloseRun& r, const OwnerList& list, int32_t n,
                              const ReturnLists& ret, void* scratch, int64_t slice, int64_t dmax,
                              int blocks_max, unsigned long long* work, const TeamRule& rule,
                              int32_t* counter);
size_t close_wide_scratch_bytes(int64_t cap, int64_t words, int64_t dmax, int nsm);

}  // namespace hg
