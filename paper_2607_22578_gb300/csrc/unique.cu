// K2-K4: exact unique-with-inverse over fingerprinted rows — the merge step of
// topological fusion within a time window (Section 3.3, "Dynamic Fusion and
// Reuse Mechanism" (I)) and the merge sets M(v*) of Appendix A.2.
//
// The window's matching of a new node against the nodes already seen is a
// lookup by signature; here it is a device hash table keyed by the 64-bit
// fingerprint, whose value is the smallest row index carrying that key:
//   1. insert: every row offers (fp, i); equal fingerprints within a warp are
//      combined first, the slot keeps the minimum index (atomicMin);
//   2. lookup + verify: rep[i] = the slot's index; a row with rep[i] != i is
//      compared in full (length + tokens) with row rep[i]: the pairs of a warp's
//      rows as one flat list of pieces, or, in the one-launch path, two pairs per
//      warp round of 16 lanes each.  A mismatch — rows with equal fingerprints
//      but different contents — sends the row to a collision list;
//   3. collision list (empty unless fingerprints collide): exact regrouping
//      in linear work — the listed rows are grouped again by a second key
//      (a different hash of the row, mixed with its fingerprint) in the now
//      free table, and each is compared with the smallest listed row of its
//      group; rows that collide in both keys (practically never) are peeled:
//      the smallest unassigned one becomes a representative and every one
//      equal to it joins it;
//   4. exclusive sum-scan of "row is its own representative" gives each
//      group its ordinal in first-occurrence order (single pass, decoupled
//      look-back with bounded spins); the final kernel writes unique_idx and
//      inverse.
// Up to kSmallRows rows, one launch of one cluster does it all.
#include <mutex>
#include <type_traits>

#include "fnv.cuh"
#include "hs_internal.cuh"
#include "row_table.cuh"

namespace hs {
namespace {

using namespace table;

constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;
static_assert(kScanThreads % 32 == 0 && kScanThreads <= 1024, "scan block: whole warps, at most 32");
constexpr int64_t kSmallRows = 4096;    // single-launch path: 1024 threads, four rows each
constexpr int kResolveThreads = 512;    // one block for the collision list

constexpr size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct Layout {
  int log2T;
  // zero-initialised region first, then the region set to all-ones bytes
  size_t ctr, scan_status, zero_end;
  size_t keys, idx, ones_end;
  size_t rep, uid, coll_list, total;
};

// Counters (uint32 each) in the zeroed region.
constexpr int kCtrColl = 0;   // collision list length
constexpr int kCtrScan = 1;   // scan tile ticket

constexpr Layout layout(int64_t n) {
  Layout L{};
  L.log2T = table_log2(n);
  const size_t T1 = (size_t(1) << L.log2T) + 1;   // + the slot of fingerprint kEmpty
  const int64_t tiles = (n + kScanTile - 1) / kScanTile;
  size_t o = 0;
  L.ctr = o;          o += align256(sizeof(uint32_t) * 16);
  L.scan_status = o;  o += align256(sizeof(uint64_t) * (size_t)tiles);
  L.zero_end = o;
  L.keys = o;         o += align256(sizeof(uint64_t) * T1);
  L.idx = o;          o += align256(sizeof(uint32_t) * T1);
  L.ones_end = o;
  L.rep = o;          o += align256(sizeof(int32_t) * (size_t)n);
  L.uid = o;          o += align256(sizeof(int32_t) * (size_t)n);
  L.coll_list = o;    o += align256(sizeof(int32_t) * (size_t)n);
  L.total = o;
  return L;
}

// The workspace's cleared part, both regions in one launch that is scheduled
// while the work before it ends and lets the next one be.  Bound by its launch
// up to some 100,000 rows (3.1 MB), by its writes beyond (400,000 rows: 12.6 MB,
// in L2).  hs_merge_rows of 5000 rows of 256 tokens 25.6 -> 22.0 us, of 65,536
// rows 45.8 -> 41.9, against two memset nodes, which nothing overlaps.
__global__ void __launch_bounds__(256) clear_kernel(uint4* __restrict__ p, int64_t zeros,
                                                    int64_t total) {
  pdl_wait();
  pdl_trigger();
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += step) {
    const uint32_t v = i < zeros ? 0u : ~0u;
    p[i] = make_uint4(v, v, v, v);
  }
}

// ---- row comparison ---------------------------------------------------------------------------
__device__ __forceinline__ int32_t clamp_len(const int32_t* lens, int64_t r, int32_t stride,
                                             unsigned* err) {
  int32_t L = lens ? __ldg(lens + r) : stride;
  if (L < 0 || L > stride) {
    set_error(err, kErrInvalidArg);
    L = L < 0 ? 0 : stride;
  }
  return L;
}

// Half-warp: do rows a and b differ in their first len tokens?  16 lanes, up
// to six 16-byte pieces of each row per lane in flight per round trip.
template <bool VEC>
__device__ __forceinline__ bool half_rows_differ(const int32_t* __restrict__ tokens,
                                                 int32_t stride, int64_t a, int64_t b, int32_t len,
                                                 int hl) {
  const int32_t* ra = tokens + a * (int64_t)stride;
  const int32_t* rb = tokens + b * (int64_t)stride;
  bool diff = false;
  int32_t done = 0;
  if (VEC) {
    const int32_t pieces = len >> 2;
    const int4* pa = reinterpret_cast<const int4*>(ra);
    const int4* pb = reinterpret_cast<const int4*>(rb);
    for (int32_t j0 = 0; j0 < pieces; j0 += 96) {
      int4 x[6], y[6];
#pragma unroll
      for (int u = 0; u < 6; ++u) {
        const int32_t j = j0 + u * 16 + hl;
        if (j < pieces) {
          x[u] = __ldg(pa + j);
          y[u] = __ldg(pb + j);
        }
      }
#pragma unroll
      for (int u = 0; u < 6; ++u) {
        const int32_t j = j0 + u * 16 + hl;
        if (j < pieces)
          diff |= (x[u].x != y[u].x) | (x[u].y != y[u].y) | (x[u].z != y[u].z) | (x[u].w != y[u].w);
      }
    }
    done = pieces << 2;
  }
  for (int32_t t = done + hl; t < len; t += 16) diff |= (__ldg(ra + t) != __ldg(rb + t));
  return diff;
}

// Whole warp: lane l holds a pair (a, b) with `need` set if the rows must be
// compared (their lengths, la, are equal).  Pairs are compared two at a time
// (one per half-warp).  Returns, to each lane, whether its pair differs.
template <bool VEC>
__device__ __forceinline__ bool warp_pairs_differ(const int32_t* __restrict__ tokens,
                                                  int32_t stride, bool need, int64_t a, int64_t b,
                                                  int32_t la) {
  const int lane = threadIdx.x & 31, half = lane >> 4, hl = lane & 15;
  unsigned todo = __ballot_sync(0xffffffffu, need);
  unsigned differ = 0u;
  while (todo != 0u) {
    const int j0 = __ffs(todo) - 1;
    todo &= todo - 1;
    int j1 = -1;
    if (todo != 0u) {
      j1 = __ffs(todo) - 1;
      todo &= todo - 1;
    }
    const int j = half == 0 ? j0 : j1;
    const int src = j < 0 ? 0 : j;
    const int64_t aj = __shfl_sync(0xffffffffu, a, src);
    const int64_t bj = __shfl_sync(0xffffffffu, b, src);
    const int32_t lj = __shfl_sync(0xffffffffu, la, src);
    const bool diff = j >= 0 && half_rows_differ<VEC>(tokens, stride, aj, bj, lj, hl);
    const unsigned dm = __ballot_sync(0xffffffffu, diff);
    if ((dm & 0xffffu) != 0u) differ |= 1u << j0;
    if (j1 >= 0 && (dm >> 16) != 0u) differ |= 1u << j1;
  }
  return (differ >> lane) & 1u;
}

// Whole warp: are rows a and b equal (same length, same tokens below it)?
template <bool VEC>
__device__ __forceinline__ bool rows_equal_warp(const int32_t* __restrict__ tokens, int32_t stride,
                                const int32_t* __restrict__ lens, int64_t a, int64_t b,
                                unsigned* err) {
  const int lane = threadIdx.x & 31;
  const int32_t la = clamp_len(lens, a, stride, err);
  const int32_t lb = clamp_len(lens, b, stride, err);
  if (la != lb) return false;
  const int32_t* ra = tokens + a * (int64_t)stride;
  const int32_t* rb = tokens + b * (int64_t)stride;
  bool diff = false;
  int32_t done = 0;
  if (VEC) {
    const int32_t pieces = la >> 2;
    const int4* pa = reinterpret_cast<const int4*>(ra);
    const int4* pb = reinterpret_cast<const int4*>(rb);
    for (int32_t j = lane; j < pieces; j += 32) {
      const int4 x = __ldg(pa + j), y = __ldg(pb + j);
      diff |= (x.x != y.x) | (x.y != y.y) | (x.z != y.z) | (x.w != y.w);
    }
    done = pieces << 2;
  }
  for (int32_t t = done + lane; t < la; t += 32) diff |= (__ldg(ra + t) != __ldg(rb + t));
  return !__any_sync(0xffffffffu, diff);
}

// Verify the 32 rows [p0, p0+32) of one warp against their tentative
// representatives r (lane = row).  Returns, per lane, whether the row stays
// merged with r (true for a row that is its own representative).
template <bool VEC>
__device__ __forceinline__ bool verify_warp(const int32_t* __restrict__ tokens, int32_t stride,
                                            const int32_t* __restrict__ lens, bool valid,
                                            int64_t a, int64_t r, unsigned* err) {
  const bool self = !valid || r == a;
  const int32_t la = valid ? clamp_len(lens, a, stride, err) : 0;
  const int32_t lr = self ? la : clamp_len(lens, r, stride, err);
  const bool need = !self && la == lr;
  const bool differ = warp_pairs_differ<VEC>(tokens, stride, need, a, r, la);
  return self || (need && !differ);
}

// Second grouping key of row a for the collision list: a multiply-xorshift
// hash over its length and tokens (structurally unlike FNV-1a, so rows whose
// fingerprints collide almost never collide here too), mixed with the row's
// fingerprint.  Rows with equal contents get equal keys, because their
// fingerprints are equal.  The key only groups rows for the comparison that
// follows, so exactness does not depend on it.
template <bool VEC>
__device__ __forceinline__ uint64_t regroup_key(const uint64_t* __restrict__ fp, const int32_t* __restrict__ tokens,
                                int32_t stride, const int32_t* __restrict__ lens, int64_t a,
                                unsigned* err) {
  constexpr uint64_t kMul = 0x9E3779B97F4A7C15ull, kFin = 0xD6E8FEB86659FD93ull;
  const int32_t len = clamp_len(lens, a, stride, err);
  const int32_t* row = tokens + a * (int64_t)stride;
  uint64_t h = 0x243F6A8885A308D3ull ^ (uint64_t)(uint32_t)len;
  int32_t t = 0;
  if (VEC) {
    const int4* p = reinterpret_cast<const int4*>(row);
#pragma unroll 1
    for (; t + 4 <= len; t += 4) {
      const int4 v = __ldg(p + (t >> 2));
      h = (h ^ (uint32_t)v.x) * kMul;
      h ^= h >> 29;
      h = (h ^ (uint32_t)v.y) * kMul;
      h ^= h >> 29;
      h = (h ^ (uint32_t)v.z) * kMul;
      h ^= h >> 29;
      h = (h ^ (uint32_t)v.w) * kMul;
      h ^= h >> 29;
    }
  }
#pragma unroll 1
  for (; t < len; ++t) {
    h = (h ^ (uint32_t)__ldg(row + t)) * kMul;
    h ^= h >> 29;
  }
  h ^= __ldg(fp + a) * kFin;
  h ^= h >> 32;
  h *= kFin;
  return h ^ (h >> 29);
}

// Exact regrouping of the m listed rows (rep == -1: each differs from the
// smallest row with its fingerprint, so it can only equal other listed
// rows) in linear work; one block.  The listed rows are grouped by
// regroup_key in the table keys/idx (any contents; it needs
// 2^table_log2(m) + 1 slots), each row is compared in full with the
// smallest listed row of its group and joins it if equal (the smallest row
// of a group is its own representative: every row equal to it is listed and
// in its group).  A row that differs from its group's smallest row as well
// goes to list2; returns their number, the same in every thread.
template <bool VEC>
__device__ __forceinline__ uint32_t regroup_block(const uint64_t* __restrict__ fp,
                                  const int32_t* __restrict__ tokens, int32_t stride,
                                  const int32_t* __restrict__ lens, int32_t* rep,
                                  const int32_t* list, uint32_t m, uint64_t* keys, uint32_t* idx,
                                  int32_t* list2, unsigned* err) {
  __shared__ uint32_t s_m2;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5;
  const int log2M = table_log2(m);
  const uint32_t T1 = (1u << log2M) + 1u;
  for (uint32_t s = tid; s < T1; s += blockDim.x) {
    keys[s] = kEmpty;
    idx[s] = kNoRow;
  }
  if (tid == 0) s_m2 = 0;
  __syncthreads();
  for (uint32_t c = tid; c < m; c += blockDim.x) {   // list order is arbitrary: no combining
    const int32_t a = list[c];
    const uint32_t s = insert_key(keys, regroup_key<VEC>(fp, tokens, stride, lens, a, err), log2M);
    atomicMin(idx + s, (uint32_t)a);
  }
  __syncthreads();
  for (uint32_t b = (uint32_t)w * 32u; b < m; b += (uint32_t)nw * 32u) {
    const uint32_t c = b + lane;
    const bool valid = c < m;
    const int64_t a = valid ? list[c] : 0;
    int64_t r = a;
    if (valid) {
      const uint64_t k2 = regroup_key<VEC>(fp, tokens, stride, lens, a, err);
      const uint32_t v = idx[find_key(keys, k2, log2M)];
      if (v != kNoRow) r = v;
    }
    const bool merged = verify_warp<VEC>(tokens, stride, lens, valid, a, r, err);
    if (valid) {
      if (merged)
        rep[a] = (int32_t)r;
      else
        list2[atomicAdd(&s_m2, 1u)] = (int32_t)a;
    }
  }
  __syncthreads();
  return s_m2;
}

// Exact regrouping of the listed rows (rep == -1) by peeling; one block.
// Listed rows differ from the representative of their fingerprint, so they
// can only equal each other; the smallest unassigned row of each content
// becomes its representative.  rep may be in shared or global memory.
template <bool VEC>
__device__ __forceinline__ void peel_block(const uint64_t* __restrict__ fp, const int32_t* __restrict__ tokens,
                           int32_t stride, const int32_t* __restrict__ lens, int32_t* rep,
                           const int32_t* coll_list, uint32_t m, unsigned* err) {
  __shared__ int32_t s_first;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5;
  for (;;) {
    if (tid == 0) s_first = 0x7fffffff;
    __syncthreads();
    int32_t mine = 0x7fffffff;
    for (uint32_t c = tid; c < m; c += blockDim.x) {
      const int32_t a = coll_list[c];
      if (*reinterpret_cast<volatile int32_t*>(rep + a) == -1 && a < mine) mine = a;
    }
    if (mine != 0x7fffffff) atomicMin(&s_first, mine);
    __syncthreads();
    const int32_t a0 = s_first;
    if (a0 == 0x7fffffff) break;
    const uint64_t f0 = fp[a0];
    for (uint32_t c = w; c < m; c += nw) {
      const int32_t b = coll_list[c];
      if (b == a0 || *reinterpret_cast<volatile int32_t*>(rep + b) != -1 || fp[b] != f0) continue;
      if (rows_equal_warp<VEC>(tokens, stride, lens, a0, b, err) && lane == 0) rep[b] = a0;
    }
    __syncthreads();
    if (tid == 0) rep[a0] = a0;
    __syncthreads();
  }
}

// ---- multi-kernel path ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) insert_kernel(const uint64_t* __restrict__ fp, int64_t n,
                                                     uint64_t* keys, uint32_t* idx, int log2T) {
  pdl_wait();
  pdl_trigger();
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n;
       base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = base + threadIdx.x;
    const bool valid = i < n;
    insert_row(keys, idx, log2T, valid, valid ? __ldg(fp + i) : 0ull, (uint32_t)i);
  }
}

// The collision list, after verify: the table is free again (verify was its
// last reader) and so is uid (the scan writes it next), which holds list2.
template <bool VEC>
__global__ void __launch_bounds__(kResolveThreads) resolve_kernel(
    const uint64_t* __restrict__ fp, const int32_t* __restrict__ tokens, int32_t stride,
    const int32_t* __restrict__ lens, int32_t* rep, const int32_t* coll_list,
    const uint32_t* ctr, uint64_t* keys, uint32_t* idx, int32_t* list2, unsigned* err) {
  pdl_wait();
  pdl_trigger();
  const uint32_t m = ctr[kCtrColl];
  if (m == 0) return;
  const uint32_t m2 = regroup_block<VEC>(fp, tokens, stride, lens, rep, coll_list, m, keys, idx,
                                         list2, err);
  if (m2 > 0) peel_block<VEC>(fp, tokens, stride, lens, rep, list2, m2, err);
}

// Single-pass exclusive sum-scan of "rep[i] == i" with decoupled look-back;
// the last tile writes the total (the group count).  A warp looks back over 32
// predecessors per round trip, so tiles can be small enough to spread a batch
// over the SMs (400,000 rows: 98 tiles of 4096).  A predecessor's status is
// awaited for at most limit_ns of %globaltimer; then the wait gives up, sets
// kErrTimeout and counts the predecessor as a zero prefix (the call's outputs
// are then unspecified, but every write stays in bounds).
// Bound by its chain of round trips: 65,536 rows 5.2 us cold (7.2 us in tiles
// of 16,384 with eight predecessors at a time).
__device__ __forceinline__ uint64_t wait_status(const volatile unsigned long long* p,
                                                unsigned* err, uint64_t limit_ns) {
  unsigned long long s = *p;
  if (s >> 32) return s;
  const uint64_t t0 = globaltimer_ns();
  for (uint32_t it = 1;; ++it) {
    s = *p;
    if (s >> 32) return s;
    if ((it & 31u) == 0) {
      __nanosleep(64);
      if (globaltimer_ns() - t0 > limit_ns) {
        set_error(err, kErrTimeout);
        return 2ull << 32;  // give up: treat as a zero prefix
      }
    }
  }
}

__global__ void __launch_bounds__(kScanThreads) scan_kernel(
    const int32_t* __restrict__ rep, int64_t n, int32_t* __restrict__ uid,
    unsigned long long* status, uint32_t* ctr, int32_t* total_out, unsigned* err,
    uint64_t limit_ns, int64_t withhold_tile) {
  pdl_wait();
  pdl_trigger();
  constexpr int kWarps = kScanThreads / 32;
  __shared__ uint32_t s_tile;
  __shared__ int32_t s_warp[kWarps];
  __shared__ int32_t s_prefix;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid == 0) s_tile = atomicAdd(ctr + kCtrScan, 1u);
  __syncthreads();
  const uint32_t tile = s_tile;
  const int64_t base = (int64_t)tile * kScanTile + (int64_t)tid * kScanItems;
  int32_t r[kScanItems];
  if (base + kScanItems <= n) {
#pragma unroll
    for (int i = 0; i < kScanItems; i += 4) {
      const int4 v = *reinterpret_cast<const int4*>(rep + base + i);
      r[i] = v.x;
      r[i + 1] = v.y;
      r[i + 2] = v.z;
      r[i + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) r[i] = base + i < n ? rep[base + i] : 0;
  }
  int32_t run = 0;
  uint32_t own = 0;                            // bit i: row base + i is its own representative
#pragma unroll
  for (int i = 0; i < kScanItems; ++i)
    if (base + i < n && r[i] == (int32_t)(base + i)) {
      own |= 1u << i;
      ++run;
    }
  int32_t incl = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_warp[w] = incl;
  __syncthreads();
  if (w == 0) {
    const int32_t v = lane < kWarps ? s_warp[lane] : 0;
    int32_t iv = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, iv, o);
      if (lane >= o) iv += y;
    }
    if (lane < kWarps) s_warp[lane] = iv - v;  // exclusive warp offsets
    const int32_t tile_total = __shfl_sync(0xffffffffu, iv, 31);
    // A withheld tile (test hook, -1 in normal use) never publishes, so its
    // successors' waits run out.
    volatile unsigned long long* st = status;
    const bool publish = lane == 0 && (int64_t)tile != withhold_tile;
    if (publish) st[tile] = ((tile == 0 ? 2ull : 1ull) << 32) | (uint32_t)tile_total;
    int32_t prefix = 0;
    bool done = tile == 0;
    for (int64_t j0 = (int64_t)tile - 1; !done; j0 -= 32) {
      const int64_t j = j0 - lane;             // before the first tile: a zero prefix
      const uint64_t sv = j >= 0 ? wait_status(st + j, err, limit_ns) : 2ull << 32;
      const unsigned ends = __ballot_sync(0xffffffffu, (sv >> 32) == 2ull);
      const int last = ends ? __ffs(ends) - 1 : 31;
      prefix += __reduce_add_sync(0xffffffffu, lane <= last ? (int32_t)(uint32_t)sv : 0);
      done = ends != 0u;
    }
    if (lane == 0) {
      if (publish && tile > 0) st[tile] = (2ull << 32) | (uint32_t)(prefix + tile_total);
      s_prefix = prefix;
      const int64_t tiles = (n + kScanTile - 1) / kScanTile;
      if ((int64_t)tile == tiles - 1) *total_out = prefix + tile_total;
    }
  }
  __syncthreads();
  int32_t acc = s_prefix + s_warp[w] + incl - run;
  int32_t u[kScanItems];
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    u[i] = acc;
    acc += (own >> i) & 1u;
  }
  if (base + kScanItems <= n) {
#pragma unroll
    for (int i = 0; i < kScanItems; i += 4)
      *reinterpret_cast<int4*>(uid + base + i) = make_int4(u[i], u[i + 1], u[i + 2], u[i + 3]);
  } else {
#pragma unroll
    for (int i = 0; i < kScanItems; ++i)
      if (base + i < n) uid[base + i] = u[i];
  }
}

__global__ void __launch_bounds__(256) finalize_kernel(const int32_t* __restrict__ rep,
                                                       const int32_t* __restrict__ uid, int64_t n,
                                                       const int32_t* __restrict__ n_unique,
                                                       int32_t* __restrict__ unique_idx,
                                                       int32_t* __restrict__ inverse) {
  pdl_wait();
  pdl_trigger();
  const int64_t nu = *n_unique;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r = rep[i];
    inverse[i] = uid[r];
    if (r == (int32_t)i) unique_idx[uid[i]] = (int32_t)i;
    if (i >= nu) unique_idx[i] = 0;     // the tail is a valid row map too
  }
}

// ---- verify over flat piece lists ------------------------------------------------------------
// Verify of up to 32 consecutive rows per warp against their representatives (the
// table's smallest row with the same fingerprint).  The rows that need a
// comparison (representative another row, lengths equal) are compared as
// one flat list of piece pairs: the warp's pairs are laid end to end (a
// prefix sum of their piece counts in shared memory), and each lane takes
// every 32nd piece pair, kPieces of them in flight per round, so a warp's
// rows cost about as many round trips as their bytes need whatever their
// lengths.  VEC: pieces of 16 bytes (16-byte aligned rows, stride % 4 == 0),
// the tokens of a pair's last piece past its length masked.  Otherwise the
// rows may start on any word and a piece is one word, coalesced over the
// lanes: 20,011 rows at a stride of 333, a third of them copies, take 21 us cold (40
// us as two rows per warp round).  Eight of these are in flight per lane; four in
// rows of fewer than 64, where the registers of eight cost a block in six and more
// than they give.  Fingerprints to inverse, us, four / eight: 1,000,000 rows of 31, a
// tenth copies, 96 / 106; 400,000 of 64, half copies, 59.4 / 58.8; 200,000 of 128 54.2 /
// 49.2, of 333 102 / 90.  Batches that do not fill the GPU with 32 rows per warp take
// fewer, down to 4, so a warp's chain of rounds is shorter: with the scan's smaller
// tiles 20,011 rows take 25 us from fingerprints to inverse (35), 65,536 rows of 256
// tokens 33 (38).
constexpr int kVerifyThreads = 256;

// Do the first `live` tokens of two 16-byte pieces, or two words, differ?
__device__ __forceinline__ bool piece_differs(const uint4& x, const uint4& y, int live) {
  return (x.x != y.x) | ((live > 1) & (x.y != y.y)) | ((live > 2) & (x.z != y.z)) |
         ((live > 3) & (x.w != y.w));
}
__device__ __forceinline__ bool piece_differs(uint32_t x, uint32_t y, int) { return x != y; }

template <bool VEC, int kPieces>
__global__ void __launch_bounds__(kVerifyThreads) verify_flat_kernel(
    const uint64_t* __restrict__ fp, uint64_t key_mask, int64_t n,
    const uint64_t* __restrict__ keys, const uint32_t* __restrict__ idx, int log2T,
    const int32_t* __restrict__ tokens, int32_t stride, const int32_t* __restrict__ lens,
    int rows_per_warp, int32_t* __restrict__ rep, int32_t* coll_list, uint32_t* ctr,
    unsigned* err) {
  pdl_wait();
  pdl_trigger();
  __shared__ int32_t s_pre[kVerifyThreads / 32][32];
  __shared__ int32_t s_a[kVerifyThreads / 32][32];
  __shared__ int32_t s_b[kVerifyThreads / 32][32];
  __shared__ int32_t s_len[kVerifyThreads / 32][32];
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  for (int64_t p0 = w * rows_per_warp; p0 < n; p0 += warps * rows_per_warp) {
    const int64_t a = p0 + lane;
    const bool valid = lane < rows_per_warp && a < n;
    int64_t r = a;
    int32_t la = 0, lr = 0;
    if (valid) {
      const uint32_t v = idx[find_key(keys, __ldg(fp + a) & key_mask, log2T)];
      if (v < (uint32_t)n) r = v;
      else set_error(err, kErrInvalidArg);   // not reached: every row was inserted
      la = clamp_len(lens, a, stride, err);
      lr = r != a ? clamp_len(lens, r, stride, err) : la;
    }
    const bool need = valid && r != a && la == lr;
    // The list's length fits 32 bits: this path takes more than 4096 rows,
    // so 32 of them hold less than 2^31 words in any memory there is.
    int32_t incl = need ? (VEC ? (la + 3) >> 2 : la) : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    s_pre[wl][lane] = incl;
    s_a[wl][lane] = (int32_t)a;
    s_b[wl][lane] = (int32_t)r;
    s_len[wl][lane] = la;
    const int32_t total = __shfl_sync(0xffffffffu, incl, 31);
    __syncwarp();
    uint32_t differ = 0;                       // bit t: a piece of pair t differs
    int t = 0;                                 // this lane's current pair (only moves forward)
    for (int32_t g0 = 0; g0 < total; g0 += 32 * kPieces) {
      using Piece = typename std::conditional<VEC, uint4, uint32_t>::type;
      Piece x[kPieces], y[kPieces];
      int tt[kPieces], vt[kPieces];
#pragma unroll
      for (int u = 0; u < kPieces; ++u) {
        const int32_t g = g0 + u * 32 + lane;
        tt[u] = -1;
        if (g < total) {
          while (s_pre[wl][t] <= g) ++t;
          const int32_t j = g - (t > 0 ? s_pre[wl][t - 1] : 0);
          x[u] = __ldg(reinterpret_cast<const Piece*>(tokens + (int64_t)s_a[wl][t] * stride) + j);
          y[u] = __ldg(reinterpret_cast<const Piece*>(tokens + (int64_t)s_b[wl][t] * stride) + j);
          tt[u] = t;
          vt[u] = s_len[wl][t] - 4 * j;        // VEC: live tokens in this piece (>= 1)
        }
      }
#pragma unroll
      for (int u = 0; u < kPieces; ++u)
        if (tt[u] >= 0 && piece_differs(x[u], y[u], vt[u])) differ |= 1u << tt[u];
    }
    differ = __reduce_or_sync(0xffffffffu, differ);
    __syncwarp();                              // shared lists free for the next rows
    if (valid) {
      const bool merged = r == a || (need && !((differ >> lane) & 1u));
      rep[a] = merged ? (int32_t)r : -1;
      if (!merged) coll_list[atomicAdd(ctr + kCtrColl, 1u)] = (int32_t)a;
    }
  }
}

// ---- hs_merge_rows: second pass of the fingerprint, fused with the insert ---------------------
// One thread per row finishes the fingerprint (the last L mod 32 tokens, from the
// state the chunk kernel left in fp_out, or all of a row shorter than 32 tokens;
// the chunk kernel runs where any row can be as long), writes it, and offers
// (fp & key_mask, row) to the table in the same pass: rows of a warp with equal
// keys are combined and the smallest index inserts (atomicMin), as insert_kernel
// does.  An invalid length sets the error word and a zero fingerprint, as
// hs_fingerprint does.
__global__ void __launch_bounds__(256) tails_insert_kernel(
    const int32_t* __restrict__ tokens, int64_t n, int32_t stride,
    const int32_t* __restrict__ lens, uint64_t seed, uint64_t key_mask,
    uint64_t* __restrict__ fp_out, uint64_t* keys, uint32_t* idx, int log2T, unsigned* err) {
  pdl_wait();
  pdl_trigger();
  constexpr int T = 32;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n;
       base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = base + threadIdx.x;
    const bool valid = r < n;
    uint64_t f = 0;
    if (valid) {
      const int32_t L = lens ? __ldg(lens + r) : stride;
      if (L < 0 || L > stride) {
        set_error(err, kErrInvalidArg);
      } else {
        const int32_t rest = L % T;
        f = L >= T ? fp_out[r] : seed;
        if (rest > 0) {
          uint32_t lo = (uint32_t)f, hi = (uint32_t)(f >> 32);
          fnv::hash_tokens<T, true>(lo, hi, tokens + r * (int64_t)stride + (L - rest), rest);
          f = ((uint64_t)hi << 32) | lo;
        }
      }
      fp_out[r] = f;
    }
    insert_row(keys, idx, log2T, valid, f & key_mask, (uint32_t)r);
  }
}

// ---- single-launch path (n <= kSmallRows) ----------------------------------------------------
// One cluster of CTAs, each of which builds the whole table in its own shared
// memory (the same table in each), verifies its share of the rows, and, once
// the cluster's barrier has shown that no keys collided, scans the whole batch
// and writes its share of the outputs.  The barrier is the only dependency
// between CTAs, so the call needs no counters in memory and nothing cleared.
// A collision list (its length in the first CTA's shared memory) is regrouped
// by that CTA, which then writes all outputs.  THREADS threads of up to ROWS
// rows each.
//
// Bound by its chain of round trips and barriers.  Fingerprints to inverse, us
// (CTAs without a cluster, whose last one to finish scanned and wrote alone,
// after a memset of its counters): 64 rows 5.1 (12.3), 512 rows of 384 words
// 7.5 (12.7), 2048 rows 14.9 (21.0), 4096 rows of 128 words 23.5 (26.7).
// Dynamic shared memory: keys[T + 1], idx[T + 1], rep[n], uid[n] (T = 2^log2T).
constexpr size_t small_smem(int64_t n) {
  const size_t T1 = (size_t(1) << table_log2(n)) + 1;
  return T1 * 8 + T1 * 4 + (size_t)n * 8 + 16;
}
static_assert(small_smem(kSmallRows) + 256 <= 232448,
              "one-launch path: the table, rep and uid fit one CTA's shared memory");

template <bool VEC, int THREADS, int ROWS>
__global__ void __launch_bounds__(THREADS, 1) unique_small_kernel(
    const uint64_t* __restrict__ fp, int n, const int32_t* __restrict__ tokens, int32_t stride,
    const int32_t* __restrict__ lens, int32_t* __restrict__ n_unique,
    int32_t* __restrict__ unique_idx, int32_t* __restrict__ inverse, int32_t* coll_list,
    unsigned* err) {
  extern __shared__ __align__(16) uint8_t sm[];
  __shared__ uint32_t s_ncoll;
  __shared__ int32_t s_warp[THREADS / 32];
  const int log2T = table_log2(n);
  const uint32_t T1 = (1u << log2T) + 1u;
  uint64_t* keys = reinterpret_cast<uint64_t*>(sm);
  uint32_t* idx = reinterpret_cast<uint32_t*>(keys + T1);
  int32_t* rep = reinterpret_cast<int32_t*>(idx + T1);
  int32_t* uid = rep + n;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  constexpr int kWarps = THREADS / 32;
  const int ctas = (int)gridDim.x, rank = (int)blockIdx.x;   // the grid is one cluster

  // 1. the table for all rows (the same in every CTA)
  for (uint32_t s = tid; s < T1; s += THREADS) {
    keys[s] = kEmpty;
    idx[s] = kNoRow;
  }
  if (tid == 0) s_ncoll = 0;
  pdl_wait();
  pdl_trigger();
  __syncthreads();
  if (ctas > 1) cluster_sync();                // the first CTA's counter is 0
  uint64_t f[ROWS];                            // all of the thread's rows at once
#pragma unroll
  for (int u = 0; u < ROWS; ++u) f[u] = u * THREADS + tid < n ? __ldg(fp + u * THREADS + tid) : 0ull;
#pragma unroll
  for (int u = 0; u < ROWS; ++u)
    if (u * THREADS < n)
      insert_row(keys, idx, log2T, u * THREADS + tid < n, f[u], (uint32_t)(u * THREADS + tid));
  __syncthreads();
#pragma unroll
  for (int u = 0; u < ROWS; ++u) {
    const int i = u * THREADS + tid;
    if (i < n) {
      const uint32_t v = idx[find_key(keys, f[u], log2T)];
      rep[i] = v < (uint32_t)n ? (int32_t)v : i;
    }
  }
  __syncthreads();

  // 2. verify this CTA's rows: rounds of 8 rows per warp (a round is a chain
  //    of memory round trips, two rows at a time), dealt over all warps
  constexpr int kRound = 8;
  const uint32_t count = cluster_smem_addr(&s_ncoll, 0);
  const int rounds = (n + kRound - 1) / kRound;
  for (int rd = w * ctas + rank; rd < rounds; rd += ctas * kWarps) {
    const int a = rd * kRound + lane;
    const bool valid = lane < kRound && a < n;
    const int64_t r = valid ? rep[a] : a;
    const bool merged = verify_warp<VEC>(tokens, stride, lens, valid, a, r, err);
    if (valid && !merged) coll_list[cluster_atomic_inc(count)] = a;
  }
  __syncthreads();
  if (ctas > 1) cluster_sync();                // every row is verified
  uint32_t m = ld_cluster(count);
  if (ctas > 1) cluster_sync();                // the counter is read: its CTA may leave
  if (m > 0) {
    if (rank != 0) return;
    __threadfence();
    for (uint32_t c = tid; c < m; c += THREADS) rep[__ldcg(coll_list + c)] = -1;
    __syncthreads();
    // the table and uid are free here: uid holds the rows left for peeling
    const uint32_t m2 =
        regroup_block<VEC>(fp, tokens, stride, lens, rep, coll_list, m, keys, idx, uid, err);
    if (m2) peel_block<VEC>(fp, tokens, stride, lens, rep, uid, m2, err);
    __syncthreads();
  }

  // 3. exclusive scan of rep[i] == i: contiguous items per thread
  const int per = (n + THREADS - 1) / THREADS;
  const int b0 = min(n, tid * per), b1 = min(n, b0 + per);
  int32_t run = 0;
  for (int i = b0; i < b1; ++i) run += rep[i] == i;
  int32_t incl = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_warp[w] = incl;
  __syncthreads();
  int32_t off = 0, total = 0;
#pragma unroll
  for (int i = 0; i < kWarps; ++i) {
    off += i < w ? s_warp[i] : 0;
    total += s_warp[i];
  }
  int32_t acc = off + incl - run;
  for (int i = b0; i < b1; ++i) {
    uid[i] = acc;
    acc += rep[i] == i;
  }
  __syncthreads();

  // 4. the outputs, every CTA its share
  const int shares = m > 0 ? 1 : ctas;
  for (int i = rank * THREADS + tid; i < n; i += shares * THREADS) {
    const int32_t r = rep[i];
    inverse[i] = uid[r];
    if (r == i) unique_idx[uid[i]] = i;
    if (i >= total) unique_idx[i] = 0;
  }
  if (rank == 0 && tid == 0) *n_unique = total;
}

// Test hook of the look-back's bounded wait (hs_debug_scan_wait): the wait
// limit and a tile that does not publish its status (-1: none).
std::atomic<uint64_t> g_scan_wait_limit_ns{kWaitLimitNs};
std::atomic<int64_t> g_scan_withhold_tile{-1};

unsigned grid_for(int64_t items, int per_block, int max_blocks) {
  int64_t b = (items + per_block - 1) / per_block;
  if (b < 1) b = 1;
  if (b > max_blocks) b = max_blocks;
  return (unsigned)b;
}

void launch_clear(char* w, const Layout& L, int sms, cudaStream_t stream) {
  const int64_t total = (int64_t)(L.ones_end / sizeof(uint4));
  launch_pdl(clear_kernel, dim3(grid_for(total, 1024, sms * 8)), dim3(256), 0, stream,
             reinterpret_cast<uint4*>(w), (int64_t)(L.zero_end / sizeof(uint4)), total);
}

// Rows per warp of the verify: 32, or fewer while that leaves over half of the
// GPU's warps (32 per SM) without any.
int verify_rows(int64_t n, int sms) {
  int r = 32;
  while (r > 4 && n < (int64_t)sms * 16 * r) r /= 2;
  return r;
}

template <bool VEC, int THREADS, int ROWS>
hs_status launch_small(const uint64_t* fp, const int32_t* tokens, int64_t n, int32_t stride,
                       const int32_t* lens, int32_t* n_unique, int32_t* unique_idx,
                       int32_t* inverse, int32_t* coll_list, unsigned* err, cudaStream_t stream) {
  auto* kernel = unique_small_kernel<VEC, THREADS, ROWS>;
  const size_t smem = small_smem(n);
  static std::atomic<uint64_t> configured{0};
  if (smem > 48 * 1024) {
    const hs_status cst = once_per_device(configured, [] {
      return cuda_fail(cudaFuncSetAttribute(unique_small_kernel<VEC, THREADS, ROWS>,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)small_smem(THREADS * ROWS)),
                       "unique smem attribute");
    });
    if (cst != HS_OK) return cst;
  }
  // A CTA per 64 rows, at most the portable cluster size.
  unsigned ctas = 1;
  while (ctas < 8 && (int64_t)ctas * 64 < n) ctas *= 2;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = ctas;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cuda_fail(cudaLaunchKernelEx(&cfg, kernel, fp, (int)n, tokens, stride,
                                      lens, n_unique, unique_idx, inverse, coll_list, err),
                   "unique launch");
}

}  // namespace

size_t unique_inverse_workspace(int64_t n) { return n <= 0 ? 256 : layout(n).total; }

hs_status launch_unique_inverse(const uint64_t* fp, const int32_t* tokens, int64_t n,
                                int32_t stride, const int32_t* lens, int32_t* n_unique_dev,
                                int32_t* unique_idx, int32_t* inverse, void* ws,
                                cudaStream_t stream) {
  unsigned* err = device_error_word();
  if (!err) return fail(HS_ERR_CUDA, "could not resolve the device error word");
  const Layout L = layout(n);
  char* w = static_cast<char*>(ws);
  uint32_t* ctr = reinterpret_cast<uint32_t*>(w + L.ctr);
  auto* status = reinterpret_cast<unsigned long long*>(w + L.scan_status);
  uint64_t* keys = reinterpret_cast<uint64_t*>(w + L.keys);
  uint32_t* idx = reinterpret_cast<uint32_t*>(w + L.idx);
  int32_t* rep = reinterpret_cast<int32_t*>(w + L.rep);
  int32_t* uid = reinterpret_cast<int32_t*>(w + L.uid);
  int32_t* coll_list = reinterpret_cast<int32_t*>(w + L.coll_list);
  const bool vec = ((reinterpret_cast<uintptr_t>(tokens) & 15u) == 0) && (stride % 4 == 0);
  const int sms = num_sms();

  if (n <= kSmallRows) {
    // Twice the threads once there are more than four rows for each of 512
    // (us, 512 / 1024 threads: 512 rows 7.5 / 8.6, 4096 ragged rows 33.5 / 29.4).
    auto* launch = n <= 2048 ? (vec ? launch_small<true, 512, 4> : launch_small<false, 512, 4>)
                             : (vec ? launch_small<true, 1024, 4> : launch_small<false, 1024, 4>);
    const hs_status st = launch(fp, tokens, n, stride, lens, n_unique_dev, unique_idx, inverse,
                                coll_list, err, stream);
    if (st == HS_OK) count_launches(1);
    return st;
  }
  launch_clear(w, L, sms, stream);
  launch_pdl(insert_kernel, dim3(grid_for(n, 256, sms * 8)), dim3(256), 0, stream, fp, n, keys, idx,
             L.log2T);
  const int vr = verify_rows(n, sms);
  launch_pdl(vec           ? verify_flat_kernel<true, 4>
             : stride < 64 ? verify_flat_kernel<false, 4>
                           : verify_flat_kernel<false, 8>,
             dim3(grid_for(n, vr * (kVerifyThreads / 32), sms * 8)), dim3(kVerifyThreads), 0, stream,
             fp, ~0ull, n, (const uint64_t*)keys, (const uint32_t*)idx, L.log2T, tokens, stride,
             lens, vr, rep, coll_list, ctr, err);
  if (vec)
    launch_pdl(resolve_kernel<true>, dim3(1), dim3(kResolveThreads), 0, stream, fp, tokens, stride,
               lens, rep, coll_list, ctr, keys, idx, uid, err);
  else
    launch_pdl(resolve_kernel<false>, dim3(1), dim3(kResolveThreads), 0, stream, fp, tokens,
               stride, lens, rep, coll_list, ctr, keys, idx, uid, err);
  const int64_t tiles = (n + kScanTile - 1) / kScanTile;
  launch_pdl(scan_kernel, dim3((unsigned)tiles), dim3(kScanThreads), 0, stream, rep, n, uid, status,
             ctr, n_unique_dev, err, g_scan_wait_limit_ns.load(), g_scan_withhold_tile.load());
  launch_pdl(finalize_kernel, dim3(grid_for(n, 256, sms * 8)), dim3(256), 0, stream, rep, uid, n,
             n_unique_dev, unique_idx, inverse);
  count_launches(6);  // clear, insert, verify, resolve, scan, finalize
  return cuda_fail(cudaGetLastError(), "unique_inverse launch");
}

hs_status launch_fingerprint(const int32_t*, int64_t, int32_t, const int32_t*, uint64_t,
                             uint64_t*, cudaStream_t);
hs_status launch_fingerprint_chunks(const int32_t*, int64_t, int32_t, const int32_t*, uint64_t,
                                    uint64_t*, cudaStream_t);

// Test hook of hs_merge_rows (hs_debug_merge_key_mask): the table key is
// fp & mask, so a narrow mask forces fingerprint collisions.
std::atomic<uint64_t> g_merge_key_mask{~0ull};

size_t merge_rows_workspace(int64_t n) { return unique_inverse_workspace(n); }

// hs_merge_rows: the fingerprint's chunk pass, then one pass that finishes
// the fingerprints and inserts them (no separate insert pass), then the
// verify, collision resolve, scan and finalize of hs_unique_inverse.
hs_status launch_merge_rows(const int32_t* tokens, int64_t n, int32_t stride, const int32_t* lens,
                            uint64_t seed, uint64_t* fp_out, int32_t* n_unique_dev,
                            int32_t* unique_idx, int32_t* inverse, void* ws, cudaStream_t stream) {
  const bool vec = ((reinterpret_cast<uintptr_t>(tokens) & 15u) == 0) && (stride % 4 == 0);
  const uint64_t mask = g_merge_key_mask.load();
  if (n <= kSmallRows || !vec) {   // few rows, or rows not 16-byte aligned: the two calls
    hs_status st = launch_fingerprint(tokens, n, stride, lens, seed, fp_out, stream);
    if (st != HS_OK) return st;
    return launch_unique_inverse(fp_out, tokens, n, stride, lens, n_unique_dev, unique_idx,
                                 inverse, ws, stream);
  }
  unsigned* err = device_error_word();
  if (!err) return fail(HS_ERR_CUDA, "could not resolve the device error word");
  const Layout L = layout(n);
  char* w = static_cast<char*>(ws);
  uint32_t* ctr = reinterpret_cast<uint32_t*>(w + L.ctr);
  auto* status = reinterpret_cast<unsigned long long*>(w + L.scan_status);
  uint64_t* keys = reinterpret_cast<uint64_t*>(w + L.keys);
  uint32_t* idx = reinterpret_cast<uint32_t*>(w + L.idx);
  int32_t* rep = reinterpret_cast<int32_t*>(w + L.rep);
  int32_t* uid = reinterpret_cast<int32_t*>(w + L.uid);
  int32_t* coll_list = reinterpret_cast<int32_t*>(w + L.coll_list);
  const int sms = num_sms();
  launch_clear(w, L, sms, stream);
  const hs_status st = launch_fingerprint_chunks(tokens, n, stride, lens, seed, fp_out, stream);
  if (st != HS_OK) return st;
  launch_pdl(tails_insert_kernel, dim3(grid_for(n, 256, sms * 16)), dim3(256), 0, stream, tokens, n,
             stride, lens, seed, mask, fp_out, keys, idx, L.log2T, err);
  const int vr = verify_rows(n, sms);
  launch_pdl(verify_flat_kernel<true, 4>, dim3(grid_for(n, vr * (kVerifyThreads / 32), sms * 8)),
             dim3(kVerifyThreads), 0, stream, (const uint64_t*)fp_out, mask, n,
             (const uint64_t*)keys, (const uint32_t*)idx, L.log2T, tokens, stride, lens, vr, rep,
             coll_list, ctr, err);
  launch_pdl(resolve_kernel<true>, dim3(1), dim3(kResolveThreads), 0, stream,
             (const uint64_t*)fp_out, tokens, stride, lens, rep, (const int32_t*)coll_list,
             (const uint32_t*)ctr, keys, idx, uid, err);
  const int64_t tiles = (n + kScanTile - 1) / kScanTile;
  launch_pdl(scan_kernel, dim3((unsigned)tiles), dim3(kScanThreads), 0, stream,
             (const int32_t*)rep, n, uid, status, ctr, n_unique_dev, err,
             g_scan_wait_limit_ns.load(), g_scan_withhold_tile.load());
  launch_pdl(finalize_kernel, dim3(grid_for(n, 256, sms * 8)), dim3(256), 0, stream,
             (const int32_t*)rep, (const int32_t*)uid, n, (const int32_t*)n_unique_dev,
             unique_idx, inverse);
  count_launches(6);  // clear, tails+insert, verify, resolve, scan, finalize (the chunk
                      // launcher counts its own)
  return cuda_fail(cudaGetLastError(), "merge_rows launch");
}

}  // namespace hs

// ---- allocation-free entry point -------------------------------------------------------------
// Some callers cannot allocate device memory at the moment they merge rows:
// code that runs while a CUDA graph is being captured (an allocation there
// would be recorded into, or break, the graph), plugins and embedded runtimes
// that are handed a fixed memory budget and may not touch the allocator, and
// latency-critical request paths where an allocator call (or a pool that has
// to grow) is an unbounded stall.  hs_unique_inverse_noalloc serves them with
// a scratch area that is part of the library's own module memory: a
// file-scope device array sized for kNoAllocMaxRows rows (2,360,320 bytes),
// which every GPU that loads the library holds until the process exits.
namespace hs {
namespace {
constexpr int64_t kNoAllocMaxRows = 65536;
constexpr size_t kNoAllocBytes = layout(kNoAllocMaxRows).total;
static_assert(kNoAllocBytes == 2360320, "the scratch size stated in hs.h");
static __device__ __align__(256) unsigned char g_noalloc_ws[kNoAllocBytes];
constexpr int kNoAllocDevices = 64;
void* g_noalloc_addr[kNoAllocDevices] = {};
std::mutex g_noalloc_mu;

// Device address of this device's copy of the scratch array.  In host code
// the array's name is only a host-side stand-in, so the address is looked up
// once per device, with that device current, and cached.
hs_status noalloc_scratch(void** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev < 0 || dev >= kNoAllocDevices) return fail(HS_ERR_UNSUPPORTED, "device index %d", dev);
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_ws);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(scratch)");
    g_noalloc_addr[dev] = p;
  }
  *out = g_noalloc_addr[dev];
  return HS_OK;
}
}  // namespace
}  // namespace hs

extern "C" hs_status hs_debug_scan_wait(uint64_t limit_ns, int64_t withhold_tile) {
  using namespace hs;
  clear_last_error();
  if (limit_ns > kWaitLimitNs)
    return fail(HS_ERR_INVALID_ARG, "wait limit above the default of %llu ns",
                (unsigned long long)kWaitLimitNs);
  if (withhold_tile < -1) return fail(HS_ERR_INVALID_ARG, "withhold_tile < -1");
  g_scan_wait_limit_ns.store(limit_ns == 0 ? kWaitLimitNs : limit_ns);
  g_scan_withhold_tile.store(withhold_tile);
  return HS_OK;
}

extern "C" hs_status hs_debug_merge_key_mask(uint64_t mask) {
  hs::clear_last_error();
  hs::g_merge_key_mask.store(mask == 0 ? ~0ull : mask);
  return HS_OK;
}

extern "C" hs_status hs_unique_inverse_noalloc(const uint64_t* fp, const int32_t* tokens,
                                               int64_t n_rows, int32_t row_stride,
                                               const int32_t* lens, int32_t* n_unique_dev,
                                               int32_t* unique_idx_out, int32_t* inverse_out,
                                               hs_stream_t stream) {
  using namespace hs;
  clear_last_error();
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (n_rows < 0 || n_rows > kNoAllocMaxRows)
    return fail(HS_ERR_INVALID_ARG, "n_rows outside [0, %lld], the allocation-free limit",
                (long long)kNoAllocMaxRows);
  if (row_stride < 0) return fail(HS_ERR_INVALID_ARG, "row_stride < 0");
  if (!n_unique_dev) return fail(HS_ERR_INVALID_ARG, "n_unique_dev is NULL");
  if (reinterpret_cast<uintptr_t>(n_unique_dev) % 4)
    return fail(HS_ERR_INVALID_ARG, "n_unique_dev misaligned");
  if (n_rows == 0)
    return cuda_fail(cudaMemsetAsync(n_unique_dev, 0, sizeof(int32_t), s), "n_unique clear");
  if (!fp || !unique_idx_out || !inverse_out || (!tokens && row_stride > 0))
    return fail(HS_ERR_INVALID_ARG, "NULL input or output pointer");
  if (reinterpret_cast<uintptr_t>(fp) % 8 || reinterpret_cast<uintptr_t>(tokens) % 4 ||
      (lens && reinterpret_cast<uintptr_t>(lens) % 4) ||
      reinterpret_cast<uintptr_t>(unique_idx_out) % 4 ||
      reinterpret_cast<uintptr_t>(inverse_out) % 4)
    return fail(HS_ERR_INVALID_ARG, "misaligned pointer");
  void* scratch = nullptr;
  const hs_status st = noalloc_scratch(&scratch);
  if (st != HS_OK) return st;
  // launch_unique_inverse clears the parts of the scratch that must start at
  // zero on every call, so what an earlier call left there does not matter.
  return launch_unique_inverse(fp, tokens, n_rows, row_stride, lens, n_unique_dev,
                               unique_idx_out, inverse_out, scratch, s);
}
