// K6/K7: dense retrieval with a fused per-query top-k — the vector-retrieval
// node shared by merged queries (Section 4.1, "Workloads": embed, retrieve the
// top-k chunks; Section 3.3: merged nodes execute once).
//
//   S = Q * C^T   (bf16 x bf16 -> fp32), per query keep the k best (S, j),
//   ordered by score descending, ties to the lower corpus index j.
//
// K6 (retrieve_kernel) is a persistent, warp-specialised tcgen05 kernel:
//   warp 0      TMA producer: 128x64 query tile + 256x64 corpus tile per
//               stage (CTA pair: + the 128x64 half of it), 128-byte swizzle,
//               4-stage (pair: 6-stage) mbarrier ring;
//   warp 1      MMA issuer: 4 x tcgen05.mma (M=128 or pair M=256, N=256,
//               K=16) per stage into a double-buffered fp32 accumulator in
//               tensor memory (2 x 256 columns), tcgen05.commit releases
//               smem stages;
//   warps 2-9   epilogue: two warps per TMEM lane quarter, each reading half
//               of the 128 x 256 score tile with tcgen05.ld; thread = (query,
//               column half); threshold filter + per-query top-k.
// With two or more query blocks the CTAs run as pairs (clusters of two,
// cta_group::2): the even CTA issues M = 256 MMAs that take the two CTAs'
// query blocks as the two halves of A and the two 128-row halves of the
// corpus tile, one staged in each CTA, as B.  Each CTA's tensor memory holds
// the scores of its own query block against the whole tile, so each SM
// stages half of every corpus tile and reads half as much shared memory per
// MMA as a single CTA would.  The producer of each CTA loads its own query
// tile and corpus half; both complete on the even CTA's barrier.
// The Q x N score matrix never leaves the SM.  Work is split into units
// (query block pair, corpus split); units that share a corpus split run at
// the same time on different SMs, so each corpus tile is read from HBM about
// once and served to the other query blocks from L2.
//
// Top-k state per (query, half): a sorted list in registers (KREG = 8 to 32
// slots; more than 16 results are first looked for in lists shorter than k, and
// what such a list may have cut off in one more pass over its rows).
// A 32-column chunk whose maximum beats no lane's threshold costs one
// max-reduction; otherwise the chunk is staged in shared memory and every lane
// inserts its candidates in one converged loop, so the warp pays for the
// largest candidate count of a lane, not for the sum over lanes.  Where k > 32
// and such lists do not suffice, a 16-entry candidate buffer per thread in
// shared memory is sorted and merged into a sorted list in global scratch
// whenever a buffer fills.  Each unit writes its k best per (query, half); K7
// merges the sorted lists of each query: by ranking what can be among the k
// best (few rows), or one warp per query takes the largest head of its lists
// k times (packed (score, index) keys).
#include <float.h>

#include <algorithm>

#include "hs_internal.cuh"

namespace hs {
namespace {

constexpr int BM = 128;               // queries per tile: UMMA M = TMEM lanes
constexpr int BN = 256;               // corpus rows per tile: UMMA N
constexpr int BK = 64;                // K per stage: one 128-byte swizzle row
constexpr int UK = 16;                // K per tcgen05.mma, kind::f16
constexpr int kEpiWarps = 8;
constexpr int kEpi = kEpiWarps * 32;  // epilogue threads
constexpr int kThreads = 64 + kEpi;
constexpr uint32_t kABytes = BM * BK * 2;
constexpr uint32_t kBBytes = BN * BK * 2;
constexpr int kCap = 16;              // candidate buffer per thread (large-k path)
constexpr int kMergeMax = 16384;      // bound on lists * k per query (the merge's candidates)
constexpr size_t kBarBytes = 256;
constexpr size_t kEpiSmem = (size_t)kEpi * 32 * 4;  // 32 KB: staging or candidate buffer
static_assert((size_t)kCap * kEpi * 8 == kEpiSmem, "candidate buffer size");
// Shared-memory ring per CTA.  Single CTA: a 128-row query tile and the
// whole 256-row corpus tile per stage, 4 stages.  CTA pair (cta_group::2):
// each CTA stages its own query tile and its 128-row half of the corpus
// tile, so a stage is 32 KB and 6 fit.
template <int CL>
struct Ring {
  static constexpr int stages = CL == 2 ? 6 : 4;
  static constexpr uint32_t b_bytes = kBBytes / CL;
  static constexpr uint32_t stage_bytes = kABytes + b_bytes;
  static constexpr size_t smem = 1024 + (size_t)stages * stage_bytes + kBarBytes + kEpiSmem;
};
// Resident queries (17 to 64 of them, single CTAs): the query block is kept in
// shared memory, 64 rows of 128 bytes per 64 dimensions, and the ring carries
// corpus boxes of RN rows only.  The MMA reads 128 query rows all the same:
// rows 64-127 of a block are whatever follows it (the next block, or the
// ring), and the scores they give lie in lanes nobody reads.
constexpr int RQ = 64;                   // queries
constexpr int kResMaxKb = 16;            // d <= 1024 ...
constexpr int kResMaxKbWide = 12;        // ... and 768 for tiles of 256 rows
constexpr int kResMaxStages = 12;
constexpr uint32_t kResQBytes = RQ * BK * 2;
constexpr size_t kResEpiSmem = (size_t)4 * 32 * 32 * 4;   // staging of the four warps with queries
__host__ __device__ constexpr int res_stages(int rn, int kb) {
  const int64_t room =
      232448 - 1024 - (int64_t)kBarBytes - (int64_t)kResEpiSmem - (int64_t)kb * kResQBytes;
  const int64_t n = room / (rn * BK * 2);
  return (int)(n < kResMaxStages ? n : kResMaxStages);
}
constexpr size_t res_smem(int rn, int kb) {
  return 1024 + (size_t)kb * kResQBytes + (size_t)res_stages(rn, kb) * rn * BK * 2 + kBarBytes +
         kResEpiSmem;
}
static_assert(res_stages(128, kResMaxKb) >= 4 && res_stages(256, kResMaxKbWide) >= 3,
              "resident queries: a ring of a few stages");
static_assert(128 * BK * 2 >= (int)kResQBytes, "rows past the last query block lie in the ring");
static_assert(8 * (2 * kResMaxStages + 4 + 2) + 8 + 8 <= kBarBytes, "barrier area");
// The pass over cut lists: 128 queries and 128 corpus rows per stage.
constexpr int kCutRows = 128, kCutStages = 5;
constexpr uint32_t kCutStageBytes = kABytes + kCutRows * BK * 2;
static_assert(Ring<1>::smem <= 232448 && Ring<2>::smem <= 232448, "shared memory per CTA");
static_assert(8 * (2 * Ring<2>::stages + 4) + 8 + 8 <= kBarBytes, "barrier area");

// Lists of a query at most: kMaxListsPerLane per lane of the warp merge, and two
// (one per column half) per split.
constexpr int kMaxListsPerLane = 10;
constexpr int kMaxLists = 32 * kMaxListsPerLane;

// Queries of which a first pass's list may have been cut, by list: queue[l][0,
// count[l]), in no order; count[kMaxLists] is the sum.
struct CutQueues {
  uint32_t *count, *queue;              // [kMaxLists + 1], [kMaxLists][Q]
  int64_t Q, tiles;                     // the first pass: queries, tiles of ...
  const int32_t* count_dev;             // (as in Params)
  int32_t tile_rows, list_k;            // ... so many rows, a list's slots, ...
  int32_t slots, cl;                    // ... executors, CTAs of each
  int32_t most_parts;                   // parts that a list's rows are taken in, at most
};

// The same as work: list l's queries are the rows [row[l], row[l + 1]) of the pass
// over cut lists, in the blocks of BM [block[l], block[l + 1]).
struct CutTable {
  uint32_t blocks, parts, lists, rows;
  uint32_t row[kMaxLists + 1], block[kMaxLists + 1];
};
struct Params {
  int64_t Qmax, N, tiles;
  const int32_t* count_dev;  // queries to process: min(*count_dev, Qmax); NULL: Qmax
  int32_t k, kb_count;
  int32_t slots;             // concurrent unit executors the plan targets (CTAs / cl)
  int32_t cl;                // CTAs per cluster: 1, or 2 forming a CTA pair (M = 256 MMA)
  float* part_s;     // [Q][2 * nsplit][k]: one list per (split, column half)
  int32_t* part_i;
  float* list_s;     // large-k: [grid][kEpi][2][k]
  int32_t* list_i;
  unsigned* err;
  // Optional per-query floor, a score that k rows of the query are known to
  // reach (order-preserving uint32 code of the float, 0 = none): lower scores
  // are not kept, which prunes without changing the result.  Zero before the
  // call's first pass; the merge of a pass whose lists may be cut hands its k-th
  // best score on in it.  With raise_floor set every list of the query raises
  // it with atomicMax to its own last entry, and reads it once per tile.  (Not
  // where lists are shorter than k: their last entries bound nothing.)
  uint32_t* qfloor;
  int32_t raise_floor;
  // Optional, one word per query block: a unit whose query blocks are all 0
  // here is skipped (the exact large-k pass re-runs only the flagged blocks).
  const uint32_t* only;
  CutQueues cut;             // what the pass over cut lists (CUT kernels) runs
  // Bounded waits of retrieve_kernel: give up after wait_limit_ns.  With
  // withhold_first set (a test hook) every CTA skips the loads of its first
  // stage, so that stage never fills and the waits run out.
  uint64_t wait_limit_ns;
  int32_t withhold_first;
};

// Rows the merge writes: with inv NULL one per query (row q = query q);
// otherwise n_out rows, row o holding the results of query inv[o] — the
// fan-out of each merged query's results to every row merged into it.
struct OutRows {
  const int32_t* inv;
  int64_t n_out;
};

__device__ __forceinline__ uint32_t float_code(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float code_float(uint32_t c) {
  return __uint_as_float((c & 0x80000000u) ? (c ^ 0x80000000u) : ~c);
}

__host__ __device__ inline int64_t gcd64(int64_t a, int64_t b) {
  while (b) {
    const int64_t t = a % b;
    a = b;
    b = t;
  }
  return a;
}

// Largest split count a plan may use: every split needs a corpus tile, and
// the merge sorts 2 * nsplit * k candidates per query.
__host__ __device__ inline int64_t max_splits(int64_t sms, int64_t tiles, int32_t k) {
  int64_t ns = sms;
  if (ns > tiles) ns = tiles;
  if (ns > kMergeMax / (2 * k)) ns = kMergeMax / (2 * k);
  return ns < 1 ? 1 : ns;
}

// Work decomposition for Q queries: query blocks of 128, grouped by cl (the
// CTAs of a cluster take adjacent query blocks over the same corpus tiles),
// and corpus splits; units = groups * nsplit is a multiple of the number of
// unit executors (slots) when the caps allow.  Host and device evaluate the
// same function, so a launch can take its query count from device memory.
struct SplitPlan {
  int32_t qblocks, groups, nsplit;
};
__host__ __device__ inline SplitPlan split_plan(int64_t Q, int64_t tiles, int32_t k,
                                                int64_t slots, int32_t cl) {
  SplitPlan sp;
  sp.qblocks = (int32_t)((Q + BM - 1) / BM);
  sp.groups = (sp.qblocks + cl - 1) / cl;
  int64_t ns = slots / gcd64(slots, sp.groups > 0 ? sp.groups : 1);
  const int64_t cap = max_splits(slots, tiles, k);
  if (ns > cap) ns = cap;
  sp.nsplit = (int32_t)ns;
  return sp;
}

__device__ __forceinline__ int64_t query_count(const Params& p) {
  if (!p.count_dev) return p.Qmax;
  const int64_t c = *p.count_dev;
  return c < 0 ? 0 : (c > p.Qmax ? p.Qmax : c);
}

// Unit u's queries [q0, q1) (CUT: rows of the pass, and where they are in the
// queue), lists and tiles.
struct Unit {
  int64_t q0, q1, t0, t1, queue;
  int32_t split, half;
};
__device__ __forceinline__ Unit unit_coords(const SplitPlan& sp, int64_t Q, int64_t tiles,
                                            int64_t u, int rank, int cl) {
  Unit un;
  un.q0 = ((u % sp.groups) * cl + rank) * BM;
  un.q1 = Q;
  un.queue = un.half = 0;
  un.split = (int)(u / sp.groups);
  un.t0 = (int64_t)un.split * tiles / sp.nsplit;
  un.t1 = (int64_t)(un.split + 1) * tiles / sp.nsplit;
  return un;
}

// The table, in shared memory, by one warp.  The parts of a list's rows spread what
// there is over the SMs, in as few rounds as their number allows.
__device__ __forceinline__ void make_cut_table(const CutQueues& c, CutTable& t, int sms) {
  const int lane = threadIdx.x & 31;
  const int64_t n_dev = c.count_dev ? *c.count_dev : c.Q;
  const SplitPlan sp = split_plan(n_dev < 0 ? 0 : (n_dev > c.Q ? c.Q : n_dev), c.tiles, c.list_k,
                                  c.slots, c.cl);
  // A lane takes `per` lists in a row: their sums, then the warp's.
  const int lists = 2 * sp.nsplit, per = (lists + 31) / 32, first = lane * per;
  uint32_t n[kMaxListsPerLane], rows = 0, blocks = 0;
#pragma unroll
  for (int j = 0; j < kMaxListsPerLane; ++j) {
    n[j] = j < per && first + j < lists ? c.count[first + j] : 0u;
    rows += n[j];
    blocks += (n[j] + BM - 1) / BM;
  }
  uint32_t r = rows, b = blocks;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t yr = __shfl_up_sync(0xffffffffu, r, o);
    const uint32_t yb = __shfl_up_sync(0xffffffffu, b, o);
    if (lane >= o) {
      r += yr;
      b += yb;
    }
  }
  const uint32_t all = __shfl_sync(0xffffffffu, b, 31);
  const int room = max(1, min(c.most_parts, sp.nsplit * 3 / 8));       // at most 8
  const uint32_t parts = lane + 1;
  const uint32_t cost =
      (int)parts <= room ? (all * parts + sms - 1) / sms * 840u / parts : ~0u >> 5;  // lcm(1 ... 8)
  const uint32_t best = __reduce_min_sync(0xffffffffu, cost * 32 + lane);
  if (lane == 31) {
    t.row[lists] = t.rows = r;
    t.block[lists] = t.blocks = b;
    t.lists = lists;
    t.parts = (best & 31) + 1;
  }
  r -= rows;
  b -= blocks;
#pragma unroll
  for (int j = 0; j < kMaxListsPerLane; ++j)
    if (j < per && first + j < lists) {
      t.row[first + j] = r;
      t.block[first + j] = b;
      r += n[j];
      b += (n[j] + BM - 1) / BM;
    }
}

// The pass over cut lists is bound by its reading of their rows, and with few of them
// by its launch: every list of 300 queries over 262,144 x 384 cut, 44 us, 4.6 TB/s,
// tensor pipe 24 %, 3 us where nothing is cut.  It kept lists of 32 in registers at
// first, whose insertions, 20 neighbours in a row in one lane, bounded it (1000
// queries over 262,144 x 384, k = 17, the whole call 361 us, 323 now); and it went by
// split, not by half a split, which reads twice the rows for half the units (2000
// over 262,144 x 768, 1 in 100 cut: 589 us, 555 now).
//
// Unit u of the pass over cut lists: block u / parts, part u % parts (which may be
// empty) of its list's tiles; tile t is the 128 rows from
// t * tile_rows + half * tile_rows / 2 on, `half` the list's.
__device__ __forceinline__ Unit cut_unit(const CutTable& t, const CutQueues& c, int64_t u) {
  const uint32_t b = (uint32_t)(u / t.parts), part = (uint32_t)(u % t.parts);
  int lo = 0, hi = (int)t.lists;         // block[lo] <= b < block[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) / 2;
    if (t.block[mid] <= b)
      lo = mid;
    else
      hi = mid;
  }
  Unit un;
  const int64_t at = (int64_t)(b - t.block[lo]) * BM;
  un.q0 = t.row[lo] + at;
  un.q1 = t.row[lo + 1];
  un.queue = lo * c.Q + at;
  un.split = (int)part;
  un.half = lo & 1;
  const int64_t nsplit = t.lists / 2, a = (lo / 2) * c.tiles / nsplit;
  const int64_t n = (lo / 2 + 1) * c.tiles / nsplit - a;
  un.t0 = a + part * n / t.parts;
  un.t1 = a + (part + 1) * n / t.parts;
  return un;
}

// True when `only` is set and no query block of unit u's group is flagged.
// Every role of a CTA pair evaluates it for the same units, so all skip alike.
__device__ __forceinline__ bool unit_skipped(const Params& p, const SplitPlan& sp, int64_t u,
                                             int cl) {
  if (!p.only) return false;
  const int g = (int)(u % sp.groups);
  for (int r = 0; r < cl; ++r) {
    const int qb = g * cl + r;
    if (qb < sp.qblocks && p.only[qb] != 0u) return false;
  }
  return true;
}

__device__ __forceinline__ float max3f(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Maximum of 32 scores as a tree of three-input maxima (17 operations; the
// maximum is exact, so the order does not change the result).
__device__ __forceinline__ float chunk_max(const uint32_t (&r)[32]) {
  float m[11];
#pragma unroll
  for (int j = 0; j < 10; ++j)
    m[j] = max3f(__uint_as_float(r[3 * j]), __uint_as_float(r[3 * j + 1]),
                 __uint_as_float(r[3 * j + 2]));
  m[10] = fmaxf(__uint_as_float(r[30]), __uint_as_float(r[31]));
  const float a = max3f(m[0], m[1], m[2]), b = max3f(m[3], m[4], m[5]);
  const float c = max3f(m[6], m[7], m[8]), e = fmaxf(m[9], m[10]);
  return fmaxf(max3f(a, b, c), e);
}

// Sort N (a power of two) values in descending order: a bitonic network.
template <int N>
__device__ __forceinline__ void sort_desc(float (&v)[N]) {
#pragma unroll
  for (int size = 2; size <= N; size *= 2)
#pragma unroll
    for (int d = size / 2; d > 0; d /= 2)
#pragma unroll
      for (int i = 0; i < N; ++i)
        if ((i & d) == 0) {
          const float hi = fmaxf(v[i], v[i | d]), lo = fminf(v[i], v[i | d]);
          const bool down = (i & size) == 0;
          v[i] = down ? hi : lo;
          v[i | d] = down ? lo : hi;
        }
}

// Insert (s, idx) into a list sorted by score descending.  idx is larger than
// every index already present, so on equal scores it goes after them.
template <int KREG>
__device__ __forceinline__ void list_insert(float (&ls)[KREG], int32_t (&li)[KREG], float s,
                                            int32_t idx) {
#pragma unroll
  for (int i = KREG - 1; i > 0; --i) {
    const bool up = s > ls[i - 1];
    const bool here = !up && s > ls[i];
    ls[i] = up ? ls[i - 1] : (here ? s : ls[i]);
    li[i] = up ? li[i - 1] : (here ? idx : li[i]);
  }
  if (s > ls[0]) {
    ls[0] = s;
    li[0] = idx;
  }
}

// ---- large-k helpers (per thread, serial) ---------------------------------------------
__device__ void flush_candidates(float* cs, int32_t* ci, int et, int& cnt, float* Ls, int32_t* Li,
                                 int k, int& cur, float& theta, float floor_theta, float& kth) {
  if (cnt == 0) return;
  // Stable insertion sort of the buffer, score descending (buffer order is
  // ascending corpus index, so ties keep the lower index first).
  for (int a = 1; a < cnt; ++a) {
    const float s = cs[a * kEpi + et];
    const int32_t i = ci[a * kEpi + et];
    int b = a - 1;
    while (b >= 0 && s > cs[b * kEpi + et]) {
      cs[(b + 1) * kEpi + et] = cs[b * kEpi + et];
      ci[(b + 1) * kEpi + et] = ci[b * kEpi + et];
      --b;
    }
    cs[(b + 1) * kEpi + et] = s;
    ci[(b + 1) * kEpi + et] = i;
  }
  // Merge with the current list (all of whose entries have lower corpus
  // indices: on equal scores the list entry wins).  The list is consumed in
  // order, so its addresses are known ahead of the comparisons: it is read in
  // windows of 8 with the next window in flight, not one dependent load at a
  // time.
  constexpr int Wn = 8;
  const float* As = Ls + (size_t)cur * k;
  const int32_t* Ai = Li + (size_t)cur * k;
  float* Os = Ls + (size_t)(cur ^ 1) * k;
  int32_t* Oi = Li + (size_t)(cur ^ 1) * k;
  float wa[Wn];
  int32_t wi[Wn];
#pragma unroll
  for (int e = 0; e < Wn; ++e) {
    wa[e] = e < k ? As[e] : -FLT_MAX;
    wi[e] = e < k ? Ai[e] : -1;
  }
  int b = 0, o = 0;
  float sb = cs[et];
  int32_t ib = ci[et];
  float last = -FLT_MAX;
  for (int a0 = 0; a0 < k && o < k; a0 += Wn) {
    float na[Wn];
    int32_t ni[Wn];
    const bool more = a0 + Wn < k;
    if (more) {
#pragma unroll
      for (int e = 0; e < Wn; ++e) {
        const bool in = a0 + Wn + e < k;
        na[e] = in ? As[a0 + Wn + e] : -FLT_MAX;
        ni[e] = in ? Ai[a0 + Wn + e] : -1;
      }
    }
#pragma unroll
    for (int e = 0; e < Wn; ++e) {
      while (b < cnt && o < k && sb > wa[e]) {
        Os[o] = sb;
        Oi[o] = ib;
        last = sb;
        ++o;
        ++b;
        if (b < cnt) {
          sb = cs[b * kEpi + et];
          ib = ci[b * kEpi + et];
        }
      }
      if (o < k && a0 + e < k) {
        Os[o] = wa[e];
        Oi[o] = wi[e];
        last = wa[e];
        ++o;
      }
    }
    if (more) {
#pragma unroll
      for (int e = 0; e < Wn; ++e) {
        wa[e] = na[e];
        wi[e] = ni[e];
      }
    }
  }
  cur ^= 1;
  kth = last;                        // the k-th entry of the new list (-FLT_MAX if not full)
  theta = fmaxf(last, floor_theta);  // ... not below the floor
  cnt = 0;
}

// RN > 0: resident queries (CL = 1) and corpus tiles of RN rows.  CUT: the units
// are those of p.cut, single CTAs.
template <int KREG, int CL, int RN, bool CUT>
__global__ void __launch_bounds__(kThreads, 1)
    retrieve_kernel(const __grid_constant__ CUtensorMap tmap_q,
                    const __grid_constant__ CUtensorMap tmap_c, const Params p) {
  constexpr bool RES = RN > 0;
  static_assert(!RES || (CL == 1 && KREG > 0), "resident queries: single CTAs, register lists");
  static_assert(!CUT || (CL == 1 && !RES && KREG == 0), "cut lists: lists in memory");
  constexpr int BN = RES ? RN : CUT ? kCutRows : hs::BN;
  constexpr int kHalfCols = BN / 2;     // columns per epilogue thread per tile
  constexpr uint32_t kTmemCols = 2 * BN;
  const int kStages = RES ? res_stages(RN, p.kb_count) : CUT ? kCutStages : Ring<CL>::stages;
  constexpr uint32_t kBLocal = RES ? RN * BK * 2 : CUT ? kCutRows * BK * 2 : Ring<CL>::b_bytes;
  constexpr uint32_t kStageBytes = RES ? RN * BK * 2 : CUT ? kCutStageBytes : Ring<CL>::stage_bytes;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = smem;
  uint8_t* sB = smem + (RES ? p.kb_count * kResQBytes : kStages * kABytes);
  uint8_t* bar_base = RES ? sB + kStages * kStageBytes : smem + kStages * kStageBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(bar_base);
  uint64_t* full = bars;
  uint64_t* empty = bars + kStages;
  uint64_t* tfull = bars + 2 * kStages;
  uint64_t* tempty = tfull + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  uint64_t* drain = tempty + 3;          // after tmem_slot and abort_flag: the MMA drain
  uint64_t* qfull = drain + 1;           // resident queries are there
  uint8_t* epi_smem = bar_base + kBarBytes;
  const uint64_t lim = p.wait_limit_ns ? p.wait_limit_ns : kWaitLimitNs;

  // A pass over what an earlier one flagged, of which there is mostly nothing,
  // then ends here (every CTA sees the same): 3.4 us cold, 5 to 7.5 where it
  // found no unit after the setup.
  if (CUT || p.only) {
    pdl_wait();
    bool any = CUT && p.cut.count[kMaxLists] != 0u;
    if (!CUT)
      for (int64_t b = threadIdx.x; b < (p.Qmax + BM - 1) / BM; b += kThreads) any |= p.only[b] != 0u;
    if (!__syncthreads_or(any)) return;
  }

  // CTA pair: the even CTA (rank 0) owns the full and tempty barriers that
  // both CTAs' loads and epilogues signal, and issues every MMA.
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull + a, 1);
      mbar_init(tempty + a, kEpiWarps * CL);
    }
    mbar_init(drain, 1);
    if (RES) mbar_init(qfull, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    prefetch_tmap(&tmap_q);
    prefetch_tmap(&tmap_c);
  }
  if (warp == 1) {
    if (CL == 2) {
      tmem_alloc_pair(tmem_slot, kTmemCols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(tmem_slot, kTmemCols);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (CL > 1) cluster_sync();            // the pair's barriers exist before any remote signal
  const uint32_t tmem_base = *tmem_slot;
  const int rank = CL > 1 ? (int)cluster_ctarank() : 0;
  // Everything above touched only shared memory, TMEM and the kernel
  // parameters; global memory (the query count, queries, corpus) waits for
  // the previous kernel on the stream.
  pdl_wait();
  pdl_trigger();
  const CutTable& cut = *reinterpret_cast<const CutTable*>(epi_smem + hs::kEpiSmem);
  if (CUT) {
    if (warp == 0)
      make_cut_table(p.cut, *reinterpret_cast<CutTable*>(epi_smem + hs::kEpiSmem), gridDim.x);
    __syncthreads();
  }
  const int64_t Q = query_count(p);
  const SplitPlan sp = CUT ? SplitPlan{0, 0, (int32_t)cut.parts}
                           : split_plan(Q, p.tiles, p.k, p.slots, CL);
  const int64_t units = CUT     ? (int64_t)cut.blocks * cut.parts
                        : Q > 0 ? (int64_t)sp.groups * sp.nsplit
                                : 0;
  const int64_t u0 = blockIdx.x / CL, ustep = gridDim.x / CL;
  auto tile_row = [&](const Unit& un, int64_t t) {   // a tile's first corpus row
    return CUT ? t * p.cut.tile_rows + un.half * (p.cut.tile_rows / 2) : t * BN;
  };
  auto unit_of = [&](int64_t u, int rank) {
    return CUT ? cut_unit(cut, p.cut, u) : unit_coords(sp, Q, p.tiles, u, rank, CL);
  };

  if (CUT && warp == 0) {
    // ------------------------------------------------------------ TMA producer
    // of cut queries: each lane takes four of a block's rows from their places
    // (whole rows of four; the rest of the 128 is whatever was there, in lanes
    // nobody reads), lane 0 the corpus tile.
    const uint64_t pol_c = policy_evict_first();
    uint32_t stage = 0, phase = 0;
    int64_t issued = 0;
    bool ok = true;
    for (int64_t u = u0; u < units && ok; u += ustep) {
      const Unit un = unit_of(u, 0);
      const int live = (int)min((int64_t)BM, un.q1 - un.q0), fours = (live + 3) / 4;
      const uint32_t* qs = p.cut.queue + un.queue;
      int4 mine = make_int4(0, 0, 0, 0);
      if (lane < fours)
        mine = make_int4((int)qs[4 * lane], (int)qs[min(4 * lane + 1, live - 1)],
                         (int)qs[min(4 * lane + 2, live - 1)], (int)qs[min(4 * lane + 3, live - 1)]);
      for (int64_t t = un.t0; t < un.t1 && ok; ++t) {
        for (int kb = 0; kb < p.kb_count; ++kb) {
          ok = __all_sync(0xffffffffu, mbar_wait_limit(empty + stage, phase ^ 1u, abort_flag, lim));
          if (!ok) break;
          if (!p.withhold_first || issued > 0) {   // (test hook: that stage never fills)
            if (lane == 0) {
              mbar_arrive_expect_tx(full + stage, (uint32_t)fours * 4 * BK * 2 + kBLocal);
              const int64_t cy = tile_row(un, t);    // past the last row: any, masked
              tma_load_2d_hint(sB + stage * kBLocal, &tmap_c, full + stage, kb * BK,
                               (int32_t)(cy < p.N ? cy : 0), pol_c);
            }
            __syncwarp();
            if (lane < fours)
              tma_gather4(sA + stage * kABytes + lane * 4 * BK * 2, &tmap_q, full + stage, kb * BK,
                          mine);
          }
          ++issued;
          if (++stage == kStages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
    }
    if (lane == 0) {                       // no copy in flight when the CTA leaves, as below
      volatile int keep_going = 0;
      for (int64_t i = issued > kStages ? issued - kStages : 0; i < issued; ++i) {
        if (p.withhold_first && i == 0) continue;
        if (!mbar_wait_limit(full + (int)(i % kStages), (uint32_t)((i / kStages) & 1), &keep_going,
                             lim))
          break;
      }
    }
    __syncwarp();
  } else if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      const uint64_t pol_c = policy_evict_first();
      const uint64_t pol_q = policy_evict_last();
      uint32_t stage = 0, phase = 0;
      int64_t issued = 0;                 // stages armed (or withheld) so far
      const bool queries = RES && u0 < units;
      if (queries) {
        mbar_arrive_expect_tx(qfull, (uint32_t)p.kb_count * kResQBytes);
        for (int kb = 0; kb < p.kb_count; ++kb)
          tma_load_2d(sA + kb * kResQBytes, &tmap_q, qfull, kb * BK, 0);
      }
      for (int64_t u = u0; u < units; u += ustep) {
        if (!CUT && unit_skipped(p, sp, u, CL)) continue;
        const Unit un = unit_of(u, rank);
        for (int64_t t = un.t0; t < un.t1; ++t) {
          for (int kb = 0; kb < p.kb_count; ++kb) {
            if (!mbar_wait_limit(empty + stage, phase ^ 1u, abort_flag, lim)) goto producer_done;
            if (p.withhold_first && issued == 0) {   // test hook: this stage never fills
              ++issued;
              if (++stage == kStages) {
                stage = 0;
                phase ^= 1u;
              }
              continue;
            }
            ++issued;
            // A query block past the last addressable row is loaded from
            // row 0 instead: its scores are masked, and no box lies wholly
            // outside the tensor.
            const int32_t qy = un.q0 < p.Qmax ? (int32_t)un.q0 : 0;
            if (RES) {
              mbar_arrive_expect_tx(full + stage, kStageBytes);
              tma_load_2d_hint(sB + stage * kBLocal, &tmap_c, full + stage, kb * BK,
                               (int32_t)(t * BN), pol_c);
            } else if (CL == 1) {
              mbar_arrive_expect_tx(full + stage, kStageBytes);
              tma_load_2d_hint(sA + stage * kABytes, &tmap_q, full + stage, kb * BK, qy, pol_q);
              tma_load_2d_hint(sB + stage * kBLocal, &tmap_c, full + stage, kb * BK,
                               (int32_t)(t * BN), pol_c);
            } else {
              // Both CTAs' bytes complete on the even CTA's full barrier,
              // armed there for the pair.  A corpus half past the last row
              // re-reads the tile's first half (masked).
              if (rank == 0) mbar_arrive_expect_tx(full + stage, 2 * kStageBytes);
              const uint32_t bar = cluster_smem_addr(full + stage, 0);
              const int64_t cy = t * BN + rank * (BN / CL);
              tma_load_2d_pair_hint(sA + stage * kABytes, &tmap_q, bar, kb * BK, qy, pol_q);
              tma_load_2d_pair_hint(sB + stage * kBLocal, &tmap_c, bar, kb * BK,
                                    (int32_t)(cy < p.N ? cy : t * BN), pol_c);
            }
            if (++stage == kStages) {
              stage = 0;
              phase ^= 1u;
            }
          }
        }
      }
    producer_done:
      // Before it leaves, the even CTA (whose full barriers count both CTAs'
      // bytes) waits, bounded, for every stage it armed that may still be in
      // flight, so no copy lands in shared memory after the CTAs exit, even
      // when some role gave up.  In a normal run these phases have completed
      // or complete within the last tile.
      if (rank == 0) {
        volatile int keep_going = 0;
        if (queries) mbar_wait_limit(qfull, 0u, &keep_going, lim);
        for (int64_t i = issued > kStages ? issued - kStages : 0; i < issued; ++i) {
          if (p.withhold_first && i == 0) continue;           // never armed
          if (!mbar_wait_limit(full + (int)(i % kStages), (uint32_t)((i / kStages) & 1),
                               &keep_going, lim))
            break;
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0 && rank == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(BM * CL, BN);
      uint32_t stage = 0, phase = 0, tile_i = 0;
      bool any_mma = false;
      if (RES && u0 < units && !mbar_wait_limit(qfull, 0u, abort_flag, lim)) goto mma_done;
      for (int64_t u = u0; u < units; u += ustep) {
        if (!CUT && unit_skipped(p, sp, u, CL)) continue;
        const Unit un = unit_of(u, rank);
        for (int64_t t = un.t0; t < un.t1; ++t, ++tile_i) {
          const uint32_t acc = tile_i & 1u, aphase = (tile_i >> 1) & 1u;
          if (!mbar_wait_limit(tempty + acc, aphase ^ 1u, abort_flag, lim)) goto mma_done;
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + acc * BN;
          for (int kb = 0; kb < p.kb_count; ++kb) {
            if (!mbar_wait_limit(full + stage, phase, abort_flag, lim)) goto mma_done;
            tc_fence_after();
            any_mma = true;
            const uint64_t a0 =
                smem_desc_k_sw128(smem_u32(sA + (RES ? kb * kResQBytes : stage * kABytes)));
            const uint64_t b0 = smem_desc_k_sw128(smem_u32(sB + stage * kBLocal));
#pragma unroll
            for (int kk = 0; kk < BK / UK; ++kk) {
              const uint64_t koff = (uint64_t)(kk * UK * 2 / 16);
              if (CL == 1)
                umma_bf16(d_tmem, a0 + koff, b0 + koff, idesc, (kb | kk) != 0 ? 1u : 0u);
              else
                umma_bf16_pair(d_tmem, a0 + koff, b0 + koff, idesc, (kb | kk) != 0 ? 1u : 0u);
            }
            if (CL == 1)
              umma_commit(empty + stage);
            else
              umma_commit_pair_mc(empty + stage, 0x3);
            if (++stage == kStages) {
              stage = 0;
              phase ^= 1u;
            }
          }
          if (CL == 1)
            umma_commit(tfull + acc);
          else
            umma_commit_pair_mc(tfull + acc, 0x3);
        }
      }
    mma_done:
      // Every MMA this thread issued completes before the teardown frees
      // tensor memory, even when some role gave up (one commit to the drain
      // barrier; in a normal run the last tile's MMAs are all it waits for).
      if (any_mma) {
        if (CL == 1)
          umma_commit(drain);
        else
          umma_commit_pair_mc(drain, 0x1);
        volatile int keep_going = 0;
        mbar_wait_limit(drain, 0u, &keep_going, lim);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    const int ew = warp - 2;                  // 0..7
    const int quarter = warp & 3;             // TMEM lanes [32*quarter, 32*quarter+32)
    const int half = ew >> 2;                 // columns [half*128, half*128+128) of a tile
    const int row = quarter * 32 + lane;      // query within the block
    // Epilogue thread index, 0..255; with resident queries those of quarters 0
    // and 1, the ones that have queries, are 0..127 (the others stage nothing).
    const int et = RES ? ((half * 2 + (quarter & 1)) * 32 + lane) : ew * 32 + lane;
    constexpr int kEpi = RES ? 128 : hs::kEpi;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const int k = p.k;
    const int lists = 2 * sp.nsplit;
    uint32_t tile_i = 0;
    float* stage_f = reinterpret_cast<float*>(epi_smem);            // KREG: [8][kEpi][4]
    float* cand_s = reinterpret_cast<float*>(epi_smem);             // large k: [kCap][kEpi]
    int32_t* cand_i = reinterpret_cast<int32_t*>(epi_smem + (size_t)kCap * kEpi * 4);
    float* Ls = p.list_s + ((size_t)blockIdx.x * kEpi + et) * 2 * (size_t)k;
    int32_t* Li = p.list_i + ((size_t)blockIdx.x * kEpi + et) * 2 * (size_t)k;
    for (int64_t u = u0; u < units; u += ustep) {
      if (!CUT && unit_skipped(p, sp, u, CL)) continue;
      const Unit un = unit_of(u, rank);
      const int64_t t0 = un.t0, t1 = un.t1, q = un.q0 + row;
      const bool valid_q = q < un.q1;
      const int64_t qcall = CUT && valid_q ? (int64_t)p.cut.queue[un.queue + row] : q;
      const bool warp_has_query = __any_sync(0xffffffffu, valid_q);
      float theta = -FLT_MAX;
      // Register list (k <= 32): KREG slots sorted descending, the first
      // KREG - k holding +FLT_MAX sentinels that never move, so the last
      // slot is always the k-th best score seen: the list's own threshold.
      float ls[KREG > 0 ? KREG : 1];
      int32_t li[KREG > 0 ? KREG : 1];
      int cnt = 0, cur = 0;
#pragma unroll
      for (int i = 0; i < (KREG > 0 ? KREG : 1); ++i) {
        ls[i] = (KREG > 0 && i < KREG - k) ? FLT_MAX : -FLT_MAX;
        li[i] = -1;
      }
      // The query's shared floor, as a threshold that keeps ties with it
      // (another list may hold an equal score at a higher index).
      uint32_t qf_seen = 0, qf_next = 0;
      float qf_theta = -FLT_MAX;
      float list_kth = -FLT_MAX;               // large k: this list's k-th best so far
      const size_t list = ((size_t)q * lists + 2 * un.split + half) * k;
      // Cut lists: few scores reach the floor that they start with, most of them
      // together, so they are kept in no order, in place, and the least is looked
      // for only once there are k.
      int at_least = 0;
      auto keep = [&](float sc, int32_t idx) {
        float* os = p.part_s + list;
        int32_t* oi = p.part_i + list;
        const int at = cnt < k ? cnt++ : at_least;
        os[at] = sc;
        oi[at] = idx;
        if (cnt < k) return;
        float ls0 = INFINITY;
        int32_t li0 = -1;
        for (int i = 0; i < k; ++i) {
          const float s = os[i];
          const int32_t j = oi[i];
          if (s < ls0 || (s == ls0 && j > li0) || i == 0) {
            ls0 = s;
            li0 = j;
            at_least = i;
          }
        }
        list_kth = ls0;
        theta = fmaxf(theta, ls0);
      };
      if (valid_q && p.qfloor) {               // an earlier pass or other lists may have set it
        qf_seen = *reinterpret_cast<volatile uint32_t*>(p.qfloor + qcall);
        if (qf_seen) qf_theta = nextafterf(code_float(qf_seen), -INFINITY);
      }
      if (KREG == 0 && !CUT && valid_q) {
        for (int i = 0; i < k; ++i) {
          Ls[i] = -FLT_MAX;
          Li[i] = -1;
        }
      }
      // A list that starts with no threshold would take nearly every score of
      // its first tile in turn.  The maxima of 16 groups of columns give it one:
      // the k-th largest is reached by k columns, so the k best of the tile are
      // not below it (ties with it are kept).  A 17 to 128 query batch over 4096
      // x 384, k = 10: 31 to 35 -> 22 to 25 us.  (Lists of 32 slots have no
      // registers for it: the large corpus with k = 100 took 1 % more.)
      if (KREG > 0 && KREG < 32 && __any_sync(0xffffffffu, valid_q && qf_seen == 0u)) {
        const uint32_t acc = tile_i & 1u, aphase = (tile_i >> 1) & 1u;
        if (!mbar_wait_limit(tfull + acc, aphase, abort_flag, lim)) goto epi_done;
        tc_fence_after();
        const int64_t col0 = t0 * BN + half * kHalfCols;
        const bool tail = col0 + kHalfCols > p.N;
        constexpr int kGroups = 16, kEach = kHalfCols / kGroups;
        float gm[kGroups];
#pragma unroll
        for (int c = 0; c < kHalfCols / 32; ++c) {
          uint32_t r[32];
          tmem_ld_32x32b_x32(tmem_base + lane_addr + acc * BN + half * kHalfCols + c * 32, r);
          tmem_ld_wait();
#pragma unroll
          for (int g = 0; g < 32 / kEach; ++g) {
            float m = -FLT_MAX;
#pragma unroll
            for (int e = 0; e < kEach; ++e)
              if (!tail || col0 + c * 32 + g * kEach + e < p.N)
                m = fmaxf(m, __uint_as_float(r[g * kEach + e]));
            gm[c * (32 / kEach) + g] = m;
          }
        }
        tc_fence_before();
        sort_desc<kGroups>(gm);
        float kth = INFINITY;                  // the least of the first k, not gm[k - 1]:
#pragma unroll                                 // an index would put gm in local memory
        for (int i = 0; i < kGroups; ++i) kth = i < k ? fminf(kth, gm[i]) : kth;
        if (kth > -FLT_MAX) qf_theta = fmaxf(qf_theta, nextafterf(kth, -INFINITY));
      }
      for (int64_t t = t0; t < t1; ++t, ++tile_i) {
        const uint32_t acc = tile_i & 1u, aphase = (tile_i >> 1) & 1u;
        if (!mbar_wait_limit(tfull + acc, aphase, abort_flag, lim)) goto epi_done;
        tc_fence_after();
        const int64_t col0 = tile_row(un, t) + half * kHalfCols;
        const bool tail = col0 + kHalfCols > p.N;
        // Register lists: the candidates of the staged chunk (if any) of every
        // lane, inserted in one converged loop (the warp pays for the largest
        // candidate count of a lane); thresholds are re-read per insert.
        bool pending = false;
        int32_t pending_base = 0;
        auto drain = [&]() {
          uint32_t m = 0;
          if (pending) {
#pragma unroll
            for (int v = 0; v < 8; ++v) {
              const uint4 x = reinterpret_cast<const uint4*>(stage_f)[v * kEpi + et];
              m |= (__uint_as_float(x.x) > theta ? 1u : 0u) << (4 * v);
              m |= (__uint_as_float(x.y) > theta ? 1u : 0u) << (4 * v + 1);
              m |= (__uint_as_float(x.z) > theta ? 1u : 0u) << (4 * v + 2);
              m |= (__uint_as_float(x.w) > theta ? 1u : 0u) << (4 * v + 3);
            }
          }
          const int most = __reduce_max_sync(0xffffffffu, (unsigned)__popc(m));
          for (int it = 0; it < most; ++it) {
            const int j = m ? __ffs(m) - 1 : 0;
            const float sc = m ? stage_f[((j >> 2) * kEpi + et) * 4 + (j & 3)] : -FLT_MAX;
            m &= m - 1;
            if (sc > theta) {
              list_insert<(KREG > 0 ? KREG : 1)>(ls, li, sc, pending_base + j);
              theta = fmaxf(ls[(KREG > 0 ? KREG : 1) - 1], qf_theta);
            }
          }
          pending = false;
          __syncwarp();
        };
        // One 32-column chunk: mask columns past N, then the threshold test
        // and candidate handling.
        auto do_chunk = [&](uint32_t(&r)[32], int c) {
          const int32_t cbase = (int32_t)(col0 + c * 32);
          if (tail) {                           // zero-filled rows past N never qualify
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if ((int64_t)cbase + j >= p.N) r[j] = __float_as_uint(-FLT_MAX);
          }
          if (KREG > 0) {
            // A chunk with a candidate is staged in the lane's slot; drain()
            // inserts the staged candidates of all lanes in one converged
            // loop.  Long lists (32 slots, costly inserts) defer it to the end
            // of the tile, so the lanes' candidates of several chunks share
            // one pass (a lane whose slot is taken drains first); short lists
            // drain at once.
            const float mx = chunk_max(r);
            const bool any = valid_q && mx > theta;   // padding query rows never insert
            if (KREG >= 32) {
              if (__any_sync(0xffffffffu, any && pending)) drain();
              if (any) {
#pragma unroll
                for (int v = 0; v < 8; ++v)
                  reinterpret_cast<uint4*>(stage_f)[v * kEpi + et] =
                      make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
                pending = true;
                pending_base = cbase;
              }
            } else if (__any_sync(0xffffffffu, any)) {
              // Short lists: this chunk's candidates at once, the mask built
              // from the registers.
              uint32_t m = 0;
              if (any) {
#pragma unroll
                for (int j = 0; j < 32; ++j) m |= (__uint_as_float(r[j]) > theta ? 1u : 0u) << j;
#pragma unroll
                for (int v = 0; v < 8; ++v)
                  reinterpret_cast<uint4*>(stage_f)[v * kEpi + et] =
                      make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
              }
              const int most = __reduce_max_sync(0xffffffffu, (unsigned)__popc(m));
              for (int it = 0; it < most; ++it) {
                const int j = m ? __ffs(m) - 1 : 0;
                const float sc = m ? stage_f[((j >> 2) * kEpi + et) * 4 + (j & 3)] : -FLT_MAX;
                m &= m - 1;
                if (sc > theta) {
                  list_insert<(KREG > 0 ? KREG : 1)>(ls, li, sc, cbase + j);
                  theta = fmaxf(ls[(KREG > 0 ? KREG : 1) - 1], qf_theta);
                }
              }
              __syncwarp();
            }
          } else if (CUT) {
            const bool any = valid_q && chunk_max(r) > theta;
            if (__any_sync(0xffffffffu, any)) {
              uint32_t m = 0;
              if (any) {
#pragma unroll
                for (int j = 0; j < 32; ++j) m |= (__uint_as_float(r[j]) > theta ? 1u : 0u) << j;
#pragma unroll
                for (int v = 0; v < 8; ++v)
                  reinterpret_cast<uint4*>(stage_f)[v * kEpi + et] =
                      make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
              }
              for (; m; m &= m - 1) {
                const int j = __ffs(m) - 1;
                const float sc = stage_f[((j >> 2) * kEpi + et) * 4 + (j & 3)];
                if (sc > theta) keep(sc, cbase + j);
              }
              __syncwarp();
            }
          } else {
            // Same first test as above: a chunk whose maximum beats no
            // lane's threshold costs one max-reduction and a vote.
            const float mx = chunk_max(r);
            if (__any_sync(0xffffffffu, valid_q && mx > theta)) {
#pragma unroll
              for (int j0 = 0; j0 < 32; j0 += 4) {
#pragma unroll
                for (int j = j0; j < j0 + 4; ++j) {
                  const float s = __uint_as_float(r[j]);
                  if (valid_q && s > theta) {
                    cand_s[cnt * kEpi + et] = s;
                    cand_i[cnt * kEpi + et] = cbase + j;
                    ++cnt;
                  }
                }
                if (__any_sync(0xffffffffu, cnt > kCap - 4))
                  flush_candidates(cand_s, cand_i, et, cnt, Ls, Li, k, cur, theta, qf_theta,
                                   list_kth);
              }
            }
          }
        };
        // The floor asked for at the end of the last tile; its round trip has
        // passed in the wait for this tile's scores.
        if (qf_next > qf_seen) {
          qf_seen = qf_next;
          qf_theta = nextafterf(code_float(qf_next), -INFINITY);  // keep s >= floor
        }
        theta = fmaxf(theta, qf_theta);
        // Lists of up to 16 slots: two chunks per TMEM round trip (both loads,
        // one wait).  Longer lists and large k keep one: they need the
        // registers.
        // A warp whose 32 query rows are all padding has nothing to read.
#pragma unroll 1
        for (int c = 0; c < kHalfCols / 32 && warp_has_query; c += (KREG > 0 && KREG < 32 ? 2 : 1)) {
          const uint32_t ta = tmem_base + lane_addr + acc * BN + half * kHalfCols + c * 32;
          uint32_t ra[32];
          if (KREG > 0 && KREG < 32) {
            uint32_t rb[32];
            tmem_ld_32x32b_x32(ta, ra);
            tmem_ld_32x32b_x32(ta + 32, rb);
            tmem_ld_wait();
            do_chunk(ra, c);
            do_chunk(rb, c + 1);
          } else {
            tmem_ld_32x32b_x32(ta, ra);
            tmem_ld_wait();
            do_chunk(ra, c);
          }
        }
        if (KREG >= 32 && __any_sync(0xffffffffu, pending)) drain();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {                       // the scores are read: the next MMA may have them
          if (CL == 1)
            mbar_arrive(tempty + acc);
          else
            mbar_arrive_cluster(cluster_smem_addr(tempty + acc, 0));
        }
        if (valid_q && p.raise_floor) {
          // Publish this list's k-th best if it raises the query's floor,
          // and fetch the floor for the next tile.  With narrow rows a tile
          // takes little longer than this round trip: not waiting for it, and
          // giving the scores' place back before it, 2000 queries over 524,288
          // x 128, k = 1: 340 -> 318 us, k = 10 500 -> 480; x 384 487 -> 468,
          // 650 -> 635.
          const float kth = KREG > 0 ? ls[(KREG > 0 ? KREG : 1) - 1] : list_kth;
          const uint32_t mine = kth > -FLT_MAX ? float_code(kth) : 0u;
          if (mine > qf_seen) atomicMax(p.qfloor + qcall, mine);
          qf_next = *reinterpret_cast<volatile uint32_t*>(p.qfloor + qcall);
        }
      }
      if (valid_q) {
        float* os = p.part_s + list;
        int32_t* oi = p.part_i + list;
        if (CUT) {                             // the least of a full list goes last
          if (cnt == k) {
            const float sl = os[at_least];
            const int32_t il = oi[at_least];
            os[at_least] = os[k - 1];
            oi[at_least] = oi[k - 1];
            os[k - 1] = sl;
            oi[k - 1] = il;
          }
          for (int i = cnt; i < k; ++i) {
            os[i] = -FLT_MAX;
            oi[i] = -1;
          }
        } else if (KREG > 0) {
#pragma unroll
          for (int i = 0; i < (KREG > 0 ? KREG : 1); ++i)
            if (i >= KREG - k) {
              os[i - (KREG - k)] = ls[i];
              oi[i - (KREG - k)] = li[i];
            }
        } else {
          flush_candidates(cand_s, cand_i, et, cnt, Ls, Li, k, cur, theta, qf_theta,
                           list_kth);
          for (int i = 0; i < k; ++i) {
            os[i] = Ls[(size_t)cur * k + i];
            oi[i] = Li[(size_t)cur * k + i];
          }
        }
      }
    }
  epi_done:;
  }

  tc_fence_before();
  __syncthreads();
  if (CL > 1) cluster_sync();            // the pair's MMAs and remote signals are done
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    if (CL == 2)
      tmem_dealloc_pair(tmem_base, kTmemCols);
    else
      tmem_dealloc(tmem_base, kTmemCols);
  }
  if (CL > 1) cluster_sync();            // no CTA leaves while its peer may still signal it
  if (threadIdx.x == 0 && *abort_flag) set_error(p.err, kErrTimeout);
}

// ---- K7: merge of the per-split lists ----------------------------------------------------
// What a merge does with a query of which a list may have been cut, that is a
// full list whose last entry is not below the k-th best: it flags the query's
// block, or (pairs set) notes, once, which lists were cut, for the pass over
// them.  No more than k entries are that good and a cut list has p.k of
// them, so at most `most` = k / p.k of a query's lists are cut.  The k-th
// best score, which k rows reach, is the later passes' floor (of every query,
// as a flagged block is run whole).
struct CutOut {
  uint32_t* block;
  uint32_t* floor;                      // by query
  uint32_t* pairs;                      // by query: lists cut
  uint2* at;                            // [query][most]: the list, the place in its queue
  int32_t most;
  CutQueues queues;
};

__device__ __forceinline__ void add_pair(const CutOut& c, int64_t q, int32_t i, int32_t list) {
  if (i >= c.most) return;              // not reached, but after a wait that ran out
  const uint32_t at = atomicAdd(c.queues.count + list, 1u);
  atomicAdd(c.queues.count + kMaxLists, 1u);
  c.queues.queue[(size_t)list * c.queues.Q + at] = (uint32_t)q;
  c.at[(size_t)q * c.most + i] = make_uint2((uint32_t)list, at);
}

// Keys order as the lists do: scores are sums that start from +0, so none is -0.
__device__ __forceinline__ uint64_t pack_key(float s, int32_t idx) {
  uint32_t u = __float_as_uint(s);
  u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  return ((uint64_t)u << 32) | (uint64_t)(0xffffffffu - (uint32_t)idx);
}

__device__ __forceinline__ void unpack_key(uint64_t key, float& s, int32_t& idx) {
  uint32_t u = (uint32_t)(key >> 32);
  u = (u & 0x80000000u) ? (u ^ 0x80000000u) : ~u;
  s = __uint_as_float(u);
  idx = (int32_t)(0xffffffffu - (uint32_t)key);
}

// Is it a row's key (a list's unused entries have none)?
__device__ __forceinline__ bool real_key(uint64_t key) { return (uint32_t)key != 0u; }

// The floor that a k-th pick is: its score's code (a key's upper half), or 0
// where it is none, with fewer rows than k in the lists.
__device__ __forceinline__ uint32_t key_floor(uint64_t key) {
  return real_key(key) ? (uint32_t)(key >> 32) : 0u;
}

// Largest key of the warp's: the largest high word, then the largest low word
// among the lanes holding it (two warp reductions).
__device__ __forceinline__ uint64_t warp_max_key(uint64_t key) {
  const uint32_t hi = (uint32_t)(key >> 32);
  const uint32_t mhi = __reduce_max_sync(0xffffffffu, hi);
  const uint32_t mlo = __reduce_max_sync(0xffffffffu, hi == mhi ? (uint32_t)key : 0u);
  return ((uint64_t)mhi << 32) | mlo;
}

// One warp per query runs a tournament over the sorted lists.
// Lane l owns lists l, l+32, ...; it keeps each list's head and the entry
// after it (prefetched) in registers.  Each round the warp takes the largest
// head (keys are unique: a corpus row lives in exactly one list; padding
// keys tie, and the lowest such lane advances), so kout rounds give the kout
// best in order.
//
// Any kout: picks 0..31 are kept one per lane and written together when
// kout <= 32; for larger kout each pick is written as it is made.  With
// p.only set, rows whose query block is not flagged there are skipped.  With CUT and
// cut_out.floor set, a query is handed on to `cut_out` when one of its lists may have cut off a member
// of the top kout: a full list whose last (k-th) entry is not below the union's
// kout-th pick.  A list whose last entry is below it holds every row of its
// range that can be in the top kout, so with no list cut the union's first kout
// entries are exact.  LPL lists per lane at most (the launch's bound on 2 *
// nsplit / 32, rounded up); slots past the query's list count are skipped
// warp-uniformly, so the per-round work and the registers follow the lists a
// launch can have, not the largest count.
template <int LPL, bool CUT>
__global__ void __launch_bounds__(256) merge_warp_kernel(const Params p, float* __restrict__ out_s,
                                                         int32_t* __restrict__ out_i,
                                                         int32_t kout, OutRows rows,
                                                         const CutOut cut_out) {
  pdl_wait();
  pdl_trigger();
  const int64_t Q = query_count(p);
  const SplitPlan sp = split_plan(Q, p.tiles, p.k, p.slots, p.cl);
  const int k = p.k;
  const int lists = 2 * sp.nsplit;
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t R = rows.inv ? rows.n_out : Q;
  for (int64_t o = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; o < R; o += nwarps) {
    const int64_t q = rows.inv ? (int64_t)__ldg(rows.inv + o) : o;
    if (q < 0 || q >= Q) {                         // warp-uniform
      if (lane == 0) set_error(p.err, kErrInvalidArg);
      continue;
    }
    if (p.only && p.only[q / BM] == 0u) continue;  // warp-uniform
    const float* __restrict__ ps = p.part_s + (size_t)q * lists * k;
    const int32_t* __restrict__ pi = p.part_i + (size_t)q * lists * k;
    uint64_t head[LPL], next[LPL];
    int pos[LPL];
#pragma unroll
    for (int j = 0; j < LPL; ++j) {
      const int l = j * 32 + lane;
      pos[j] = 0;
      head[j] = next[j] = 0ull;
      if (j * 32 < lists) {                        // warp-uniform
        if (l < lists) head[j] = pack_key(ps[(size_t)l * k], pi[(size_t)l * k]);
        if (l < lists && k > 1) next[j] = pack_key(ps[(size_t)l * k + 1], pi[(size_t)l * k + 1]);
      }
    }
    float my_s = -FLT_MAX;
    int32_t my_i = -1;
    uint64_t last = 0ull;                          // key of the latest pick
    for (int r = 0; r < kout; ++r) {
      uint64_t best = 0ull;
      int bj = 0;
#pragma unroll
      for (int j = 0; j < LPL; ++j)
        if (j * 32 < lists && head[j] > best) {    // the first test is warp-uniform
          best = head[j];
          bj = j;
        }
      const uint64_t mx = warp_max_key(best);
      const unsigned win = __ballot_sync(0xffffffffu, best == mx && mx != 0ull);
      last = mx;
      if (kout <= 32) {
        if (lane == r && mx != 0ull) unpack_key(mx, my_s, my_i);
      } else if (lane == 0) {
        float sc = -FLT_MAX;
        int32_t id = -1;
        if (mx != 0ull) unpack_key(mx, sc, id);
        out_s[(size_t)o * kout + r] = sc;
        out_i[(size_t)o * kout + r] = id;
      }
      if (win != 0u && lane == __ffs(win) - 1) {
#pragma unroll
        for (int j = 0; j < LPL; ++j)
          if (j == bj) {
            const int l = j * 32 + lane;
            ++pos[j];
            head[j] = next[j];
            next[j] = pos[j] + 1 < k ? pack_key(ps[(size_t)l * k + pos[j] + 1],
                                                pi[(size_t)l * k + pos[j] + 1])
                                     : 0ull;
          }
      }
    }
    if (kout <= 32 && lane < kout) {
      out_s[(size_t)o * kout + lane] = my_s;
      out_i[(size_t)o * kout + lane] = my_i;
    }
    if (CUT && cut_out.floor) {
      if (lane == 0) cut_out.floor[q] = key_floor(last);
      auto cut = [&](int l) {                      // is list l?
        if (l >= lists) return false;
        const uint64_t key = pack_key(ps[(size_t)l * k + k - 1], pi[(size_t)l * k + k - 1]);
        return real_key(key) && key >= last;
      };
      bool any = false;
#pragma unroll 1
      for (int l = lane; l < lists; l += 32) any |= cut(l);
      if (!__any_sync(0xffffffffu, any)) continue;
      if (!cut_out.pairs) {
        if (lane == 0) atomicOr(cut_out.block + q / BM, 1u);
      } else if (__shfl_sync(0xffffffffu, lane == 0 ? atomicCAS(cut_out.pairs + q, 0u, ~0u) : 0u,
                             0) == 0u) {
        int32_t n = 0;
#pragma unroll 1
        for (int l0 = 0; l0 < lists; l0 += 32) {
          const uint32_t m = __ballot_sync(0xffffffffu, cut(l0 + lane));
          if ((m >> lane) & 1u) add_pair(cut_out, q, n + __popc(m & lanemask_lt()), l0 + lane);
          n += __popc(m);
        }
        if (lane == 0) cut_out.pairs[q] = min(n, cut_out.most);
      }
    }
  }
}

// A block per row, and no tournament.  The first `depth` entries of the lists,
// as many as it takes to have kout of them, are ranked by counting; the
// kout-th best bounds the result from below, so only lists whose depth-th entry
// reaches it can hold more.  What is left of these, with the first entries
// above the bound little more than kout, is ranked by counting again, and an
// entry's rank is its place.  Two round trips to memory and two loops over
// shared memory in place of kout dependent rounds.  64 rows of 304 lists, k =
// 10: 11 us cold, 14.4 with a warp each; 24 rows, k = 50: 27.8 -> 8.4 (32 lists of
// 32 entries before, 64 of 12 now); 100 rows, k = 100: 66.9 -> 16.8.
// Lists of at most 32 entries (p.k); CAP >= kout * p.k.  cut_out as above.
constexpr int kMrThreads = 256;
constexpr int kMrLists = kMaxLists;
constexpr int kMrMaxK = 128;
static_assert(kMrLists <= 2 * kMrThreads, "two heads per thread");
static_assert(kMrLists >= 2 * kMrMaxK, "lists * depth < kout + lists <= kMrLists");

template <int CAP>
__global__ void __launch_bounds__(kMrThreads) merge_rank_kernel(const Params p,
                                                                float* __restrict__ out_s,
                                                                int32_t* __restrict__ out_i,
                                                                int32_t kout, OutRows rows,
                                                                const CutOut cut_out) {
  pdl_wait();
  pdl_trigger();
  __shared__ uint64_t s_head[kMrLists], s_cand[CAP], s_kth;
  __shared__ int32_t s_sel[kMrLists];
  __shared__ int s_nsel, s_ncand, s_npairs;
  const int64_t Q = query_count(p);
  const SplitPlan sp = split_plan(Q, p.tiles, p.k, p.slots, p.cl);
  const int k = p.k, lists = 2 * sp.nsplit, tid = threadIdx.x;
  const int depth = min((kout + lists - 1) / lists, k);
  const int heads = lists * depth;               // entry e of list l: head e * lists + l
  const int64_t R = rows.inv ? rows.n_out : Q;
  for (int64_t o = blockIdx.x; o < R; o += gridDim.x) {
    const int64_t q = rows.inv ? (int64_t)__ldg(rows.inv + o) : o;
    if (q < 0 || q >= Q) {                         // block-uniform
      if (tid == 0) set_error(p.err, kErrInvalidArg);
      continue;
    }
    if (p.only && p.only[q / BM] == 0u) continue;  // block-uniform
    const float* __restrict__ ps = p.part_s + (size_t)q * lists * k;
    const int32_t* __restrict__ pi = p.part_i + (size_t)q * lists * k;
    uint64_t mine[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int h = j * kMrThreads + tid;
      mine[j] = 0ull;
      if (h < heads) {
        const size_t e = (size_t)(h % lists) * k + h / lists;
        const uint64_t key = pack_key(ps[e], pi[e]);
        s_head[h] = mine[j] = real_key(key) ? key : 0ull;
      }
    }
    if (tid == 0) {
      s_nsel = s_ncand = 0;
      s_kth = 0ull;                                // stays 0 when there are not kout entries
    }
    __syncthreads();
    int rank[2] = {0, 0};
#pragma unroll 8
    for (int h = 0; h < heads; ++h) {              // (missing entries are alike)
      const uint64_t y = s_head[h];
      rank[0] += (y > mine[0]) | ((y == mine[0]) & (h < tid));
      rank[1] += (y > mine[1]) | ((y == mine[1]) & (h < tid + kMrThreads));
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
      if (mine[j] != 0ull && rank[j] == kout - 1) s_kth = mine[j];
    __syncthreads();
    // the kout-th best head; with fewer entries than that every one counts
    const uint64_t bound = s_kth;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int h = j * kMrThreads + tid;
      if (mine[j] != 0ull && rank[j] < kout) {
        s_cand[atomicAdd(&s_ncand, 1)] = mine[j];
        if (h / lists == depth - 1) s_sel[atomicAdd(&s_nsel, 1)] = h % lists;
      }
    }
    __syncthreads();
    const int rest = k - depth, more = s_nsel * rest;
    for (int i = tid; i < more; i += kMrThreads) {
      const size_t e = (size_t)s_sel[i / rest] * k + depth + i % rest;
      const uint64_t key = pack_key(ps[e], pi[e]);
      if (real_key(key) && key >= bound) s_cand[atomicAdd(&s_ncand, 1)] = key;
    }
    if (tid == 0) s_kth = 0ull;
    __syncthreads();
    const int c = s_ncand;
    for (int i = c + tid; i < kout; i += kMrThreads) {       // fewer rows than results
      out_s[(size_t)o * kout + i] = -FLT_MAX;
      out_i[(size_t)o * kout + i] = -1;
    }
    for (int i = tid; i < c; i += kMrThreads) {
      const uint64_t key = s_cand[i];
      int r = 0;
#pragma unroll 8
      for (int j = 0; j < c; ++j) r += s_cand[j] > key;
      if (r < kout) {
        float sc;
        int32_t id;
        unpack_key(key, sc, id);
        out_s[(size_t)o * kout + r] = sc;
        out_i[(size_t)o * kout + r] = id;
        if (r == kout - 1) s_kth = key;
      }
    }
    __syncthreads();                               // read before the next row's lists come in
    if (cut_out.floor) {
      const uint64_t kth = s_kth;
      if (tid == 0) cut_out.floor[q] = key_floor(kth);
      uint32_t cut = 0;                            // bit j: list j * kMrThreads + tid is
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int l = j * kMrThreads + tid;
        if (l < lists) {
          const uint64_t key = pack_key(ps[(size_t)l * k + k - 1], pi[(size_t)l * k + k - 1]);
          if (real_key(key) && key >= kth) cut |= 1u << j;
        }
      }
      if (__syncthreads_or(cut)) {                 // block-uniform
        if (tid == 0) {
          s_npairs = cut_out.pairs ? (int)(atomicCAS(cut_out.pairs + q, 0u, ~0u) != 0u) : -1;
          if (!cut_out.pairs) atomicOr(cut_out.block + q / BM, 1u);
        }
        __syncthreads();
        const bool first = s_npairs == 0;          // block-uniform
        __syncthreads();
        for (int j = 0; j < 2 && first; ++j)
          if ((cut >> j) & 1u)
            add_pair(cut_out, q, atomicAdd(&s_npairs, 1), j * kMrThreads + tid);
        __syncthreads();
        if (first && tid == 0) cut_out.pairs[q] = min(s_npairs, cut_out.most);
      }
    }
  }
}

// ---- the pass over cut lists, its merge ---------------------------------------------------
constexpr int kCutThreads = 256;
// The results of the cut queries: the first pass's k best, and what their cut
// lists, run again, have above the k-th of them.  A row met twice (in the results,
// or in tiles that overlap) counts once.  More new rows than the block holds, or
// (k > 32) a list cut again, flag the query's block.  Bound by its round trips and
// barriers: 300 queries with 20 new rows each 9.4 us cold, 2.4 where nothing is cut.
constexpr int kCutNew = 3072;
constexpr int kMaxK = HS_TOPK_MAX_K;

__global__ void __launch_bounds__(kCutThreads) cut_merge_kernel(
    const Params p, float* __restrict__ out_s, int32_t* __restrict__ out_i, int32_t kout,
    OutRows rows, const CutOut cut, int sms) {
  pdl_wait();
  pdl_trigger();
  if (cut.queues.count[kMaxLists] == 0u) return;
  __shared__ uint64_t s_res[kMaxK], s_new[kCutNew], s_kth;
  __shared__ uint8_t s_dup[kCutNew];
  __shared__ int s_n;
  __shared__ CutTable t;
  if (threadIdx.x < 32) make_cut_table(cut.queues, t, sms);
  __syncthreads();
  const int tid = threadIdx.x, k = p.k, per = 2 * (int)t.parts * k;
  const int64_t n_queries = cut.queues.Q, R = rows.inv ? rows.n_out : n_queries;
  for (int64_t o = blockIdx.x; o < R; o += gridDim.x) {
    const int64_t q = rows.inv ? (int64_t)__ldg(rows.inv + o) : o;
    const int np = q >= 0 && q < n_queries ? (int)cut.pairs[q] : 0;   // block-uniform
    if (np == 0) continue;
    for (int i = tid; i < kout; i += kCutThreads) {
      const uint64_t key = pack_key(out_s[(size_t)o * kout + i], out_i[(size_t)o * kout + i]);
      s_res[i] = real_key(key) ? key : 0ull;
    }
    if (tid == 0) {
      s_n = 0;
      s_kth = 0ull;
    }
    __syncthreads();
    const uint64_t kth = s_res[kout - 1];
    for (int i = tid; i < np * per; i += kCutThreads) {
      const uint2 at = cut.at[(size_t)q * cut.most + i / per];
      const size_t e = ((size_t)t.row[at.x] + at.y) * per + i % per;
      const uint64_t key = pack_key(p.part_s[e], p.part_i[e]);
      if (!real_key(key) || key <= kth) continue;
      int lo = 0, hi = kout;                       // the first result not above it
      while (lo < hi) {
        const int mid = (lo + hi) / 2;
        if (s_res[mid] > key)
          lo = mid + 1;
        else
          hi = mid;
      }
      if (lo < kout && s_res[lo] == key) continue;
      const int n = atomicAdd(&s_n, 1);
      if (n < kCutNew) s_new[n] = key;
    }
    __syncthreads();
    const int n = min(s_n, kCutNew);
    const bool over = s_n > kCutNew;               // k > 32: k <= 32 has 1024 at most
    for (int i = tid; i < n; i += kCutThreads) {
      bool dup = false;
      for (int j = 0; j < i; ++j) dup |= s_new[j] == s_new[i];
      s_dup[i] = dup;
    }
    __syncthreads();
    for (int i = tid; i < kout + n && !over; i += kCutThreads) {
      const bool is_new = i >= kout;
      const uint64_t key = is_new ? s_new[i - kout] : s_res[i];
      if (key == 0ull || (is_new && s_dup[i - kout])) continue;
      int r = is_new ? 0 : i;
      if (is_new)
        for (int j = 0; j < kout; ++j) r += s_res[j] > key;
      for (int j = 0; j < n; ++j) r += s_new[j] > key && !s_dup[j];
      if (r >= kout) continue;
      float sc;
      int32_t id;
      unpack_key(key, sc, id);
      out_s[(size_t)o * kout + r] = sc;
      out_i[(size_t)o * kout + r] = id;
      if (r == kout - 1) s_kth = key;
    }
    __syncthreads();
    if (kout > 32) {
      const uint64_t best = s_kth;
      bool again = over;
      for (int l = tid; l < np * (per / k); l += kCutThreads) {
        const uint2 at = cut.at[(size_t)q * cut.most + l / (per / k)];
        const size_t e = ((size_t)t.row[at.x] + at.y) * per + (l % (per / k)) * k + k - 1;
        const uint64_t key = pack_key(p.part_s[e], p.part_i[e]);
        again |= real_key(key) && key >= best;
      }
      if (__syncthreads_or(again) && tid == 0) atomicOr(cut.block + q / BM, 1u);
      if (tid == 0 && !over) cut.floor[q] = key_floor(best);
    }
    __syncthreads();                               // read before the next row's
  }
}

// ---- K6s: small batches (at most 16 queries) -------------------------------------------
// With few queries the query block of the main kernel is mostly padding and
// is re-streamed with every corpus stage.  Here the roles are swapped: the
// corpus tile is the MMA's M operand (128 rows) and the queries, padded to
// 16, are its N operand, loaded once and kept in shared memory.  The ring
// then carries only corpus boxes (10 stages of 16 KB), which is what an
// HBM-bound pass needs.  TMEM holds four 128 x 16 fp32 accumulators.
//
// Epilogue (warps 2-5, one per TMEM lane quarter): thread = corpus row of the
// tile, holding its 16 scores.  A score above its query's threshold is
// appended to that query's candidate buffer in shared memory; after each
// tile a warp merges each non-empty buffer with the query's sorted top-k list
// (a few candidates are put in their places by a ballot each, many go through
// k rounds of a warp-wide maximum over packed (score, ~row) keys) and resets
// the threshold to the new k-th best.  Each CTA covers a contiguous range of
// 128-row tiles and writes one sorted list per query, in the layout of the
// main kernel's lists, so the same merge kernels finish the job.  With k rounds
// for every buffer these bounded the kernel: 16 queries, k = 10, 2,097,152 x
// 768: 680 -> 476 us; k = 32, 1,048,576 x 1024: 1602 -> 353 us.
constexpr int SQ_N = 16;                    // queries per MMA (N)
constexpr int SQ_BM = 128;                  // corpus rows per tile (M)
constexpr int SQ_STAGES = 10;
constexpr int SQ_MAXKB = 16;                // d <= 1024
constexpr int SQ_TBUF = 4;                  // TMEM accumulators
constexpr uint32_t SQ_TMEM_COLS = 64;       // SQ_TBUF * SQ_N
constexpr int SQ_CAP = SQ_BM;               // candidates per query per tile: at most one per row
constexpr int SQ_INSERT = 16;               // candidates inserted one by one; more are selected
constexpr int SQ_THREADS = 64 + 128;        // producer, MMA, 4 epilogue warps
constexpr uint32_t SQ_ABYTES = SQ_BM * BK * 2;   // 16 KB
constexpr uint32_t SQ_QBYTES = SQ_N * BK * 2;    // 2 KB per k-block
constexpr size_t SQ_EPI_BYTES = (size_t)SQ_N * (SQ_CAP + 32) * 8 + SQ_N * 8;
constexpr size_t SQ_SMEM = 1024 + (size_t)SQ_MAXKB * SQ_QBYTES + (size_t)SQ_STAGES * SQ_ABYTES +
                           256 + SQ_EPI_BYTES;
static_assert(SQ_SMEM <= 232448, "small-batch kernel shared memory");
static_assert(8 * (2 * SQ_STAGES + 1 + 2 * SQ_TBUF) + 8 + 8 <= 256, "small-batch barrier area");

__global__ void __launch_bounds__(SQ_THREADS, 1)
    retrieve_small_kernel(const __grid_constant__ CUtensorMap tmap_q,
                          const __grid_constant__ CUtensorMap tmap_c, const Params p,
                          int64_t tiles128) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* sQ = smem;
  uint8_t* sA = sQ + SQ_MAXKB * SQ_QBYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sA + SQ_STAGES * SQ_ABYTES);
  uint64_t* full = bars;
  uint64_t* empty = bars + SQ_STAGES;
  uint64_t* qfull = bars + 2 * SQ_STAGES;
  uint64_t* tfull = qfull + 1;
  uint64_t* tempty = tfull + SQ_TBUF;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + SQ_TBUF);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  uint64_t* drain = tempty + SQ_TBUF + 1;    // after tmem_slot and abort_flag: the MMA drain
  const uint64_t lim = p.wait_limit_ns ? p.wait_limit_ns : kWaitLimitNs;
  uint64_t* lists = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(bars) + 256);  // [16][32]
  uint64_t* cands = lists + SQ_N * 32;                                                    // [16][128]
  float* theta = reinterpret_cast<float*>(cands + SQ_N * SQ_CAP);                          // [16]
  int32_t* cnt = reinterpret_cast<int32_t*>(theta + SQ_N);                                 // [16]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < SQ_STAGES; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    mbar_init(qfull, 1);
    for (int b = 0; b < SQ_TBUF; ++b) {
      mbar_init(tfull + b, 1);
      mbar_init(tempty + b, 4);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    prefetch_tmap(&tmap_q);
    prefetch_tmap(&tmap_c);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, SQ_TMEM_COLS);
    tmem_relinquish();
  }
  for (int i = threadIdx.x; i < SQ_N * 32; i += SQ_THREADS) lists[i] = 0ull;
  if (threadIdx.x < SQ_N) {
    theta[threadIdx.x] = -FLT_MAX;
    cnt[threadIdx.x] = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();                            // global memory only after the previous kernel
  pdl_trigger();
  const int64_t Q = query_count(p);
  const int k = p.k;
  const int64_t t0 = (int64_t)blockIdx.x * tiles128 / gridDim.x;
  const int64_t t1 = (int64_t)(blockIdx.x + 1) * tiles128 / gridDim.x;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0 && Q > 0) {
      const uint64_t pol_c = policy_evict_first();
      mbar_arrive_expect_tx(qfull, (uint32_t)p.kb_count * SQ_QBYTES);
      for (int kb = 0; kb < p.kb_count; ++kb)
        tma_load_2d(sQ + kb * SQ_QBYTES, &tmap_q, qfull, kb * BK, 0);
      uint32_t stage = 0, phase = 0;
      int64_t issued = 0;                 // corpus stages armed (or withheld) so far
      for (int64_t t = t0; t < t1; ++t) {
        for (int kb = 0; kb < p.kb_count; ++kb) {
          if (!mbar_wait_limit(empty + stage, phase ^ 1u, abort_flag, lim)) goto sq_producer_done;
          if (p.withhold_first && issued == 0) {   // test hook: this stage never fills
            ++issued;
            if (++stage == SQ_STAGES) {
              stage = 0;
              phase ^= 1u;
            }
            continue;
          }
          ++issued;
          mbar_arrive_expect_tx(full + stage, SQ_ABYTES);
          tma_load_2d_hint(sA + stage * SQ_ABYTES, &tmap_c, full + stage, kb * BK,
                           (int32_t)(t * SQ_BM), pol_c);
          if (++stage == SQ_STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
    sq_producer_done:
      // Before it leaves, the producer waits, bounded, for the query copies
      // and every corpus stage it armed that may still be in flight, so no
      // copy lands in shared memory after the CTA exits, even when some role
      // gave up (in a normal run these phases have completed or complete
      // within the last tile).
      {
        volatile int keep_going = 0;
        mbar_wait_limit(qfull, 0u, &keep_going, lim);
        for (int64_t i = issued > SQ_STAGES ? issued - SQ_STAGES : 0; i < issued; ++i) {
          if (p.withhold_first && i == 0) continue;           // never armed
          if (!mbar_wait_limit(full + (int)(i % SQ_STAGES), (uint32_t)((i / SQ_STAGES) & 1),
                               &keep_going, lim))
            break;
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0 && Q > 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(SQ_BM, SQ_N);
      uint32_t stage = 0, phase = 0, tile_i = 0;
      bool any_mma = false;
      if (!mbar_wait_limit(qfull, 0u, abort_flag, lim)) goto sq_mma_done;
      tc_fence_after();
      for (int64_t t = t0; t < t1; ++t, ++tile_i) {
        const uint32_t b = tile_i % SQ_TBUF, bphase = (tile_i / SQ_TBUF) & 1u;
        if (!mbar_wait_limit(tempty + b, bphase ^ 1u, abort_flag, lim)) goto sq_mma_done;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + b * SQ_N;
        for (int kb = 0; kb < p.kb_count; ++kb) {
          if (!mbar_wait_limit(full + stage, phase, abort_flag, lim)) goto sq_mma_done;
          tc_fence_after();
          any_mma = true;
          const uint64_t a0 = smem_desc_k_sw128(smem_u32(sA + stage * SQ_ABYTES));
          const uint64_t b0 = smem_desc_k_sw128(smem_u32(sQ + kb * SQ_QBYTES));
#pragma unroll
          for (int kk = 0; kk < BK / UK; ++kk)
            umma_bf16(d_tmem, a0 + (uint64_t)(kk * UK * 2 / 16), b0 + (uint64_t)(kk * UK * 2 / 16),
                      idesc, (kb | kk) != 0 ? 1u : 0u);
          umma_commit(empty + stage);
          if (++stage == SQ_STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
        umma_commit(tfull + b);
      }
    sq_mma_done:
      // Every MMA this thread issued completes before the teardown frees
      // tensor memory (one commit to the drain barrier).
      if (any_mma) {
        umma_commit(drain);
        volatile int keep_going = 0;
        mbar_wait_limit(drain, 0u, &keep_going, lim);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    const int ew = warp - 2;                     // 0..3, merges queries q = ew (mod 4)
    const int quarter = warp & 3;                // TMEM lanes [32*quarter, 32*quarter+32)
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const int nq = (int)(Q < SQ_N ? Q : SQ_N);
    uint32_t tile_i = 0;
    for (int64_t t = t0; t < t1 && nq > 0; ++t, ++tile_i) {
      const uint32_t b = tile_i % SQ_TBUF, bphase = (tile_i / SQ_TBUF) & 1u;
      // On a timeout every later wait fails at once; the named barriers
      // below stay paired because all four warps walk every tile.
      const bool ok = mbar_wait_limit(tfull + b, bphase, abort_flag, lim);
      tc_fence_after();
      uint32_t r[16];
      tmem_ld_32x32b_x16(tmem_base + lane_addr + b * SQ_N, r);
      tmem_ld_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty + b);
      const int64_t row = t * SQ_BM + quarter * 32 + lane;
      if (ok && row < p.N) {
#pragma unroll
        for (int q = 0; q < SQ_N; ++q) {
          const float sc = __uint_as_float(r[q]);
          if (q < nq && sc > theta[q]) {
            const int slot = atomicAdd(cnt + q, 1);
            if (slot < SQ_CAP) cands[q * SQ_CAP + slot] = pack_key(sc, (int32_t)row);
          }
        }
      }
      named_bar_sync(1, 128);
      // Merge: list (k sorted keys) + candidates -> the k best, per query.
      for (int q = ew; q < nq; q += 4) {
        const int c = min(cnt[q], SQ_CAP);
        if (c == 0) continue;
        uint64_t mine = lane < k ? lists[q * 32 + lane] : 0ull;
        if (c <= SQ_INSERT) {
          // A few: each goes to its place in the sorted list (keys differ).
          for (int e = 0; e < c; ++e) {
            const uint64_t x = cands[q * SQ_CAP + e];
            const int at = __popc(__ballot_sync(0xffffffffu, mine > x));
            const uint64_t up = __shfl_up_sync(0xffffffffu, mine, 1);
            if (lane >= at) mine = lane == at ? x : up;
          }
          if (lane >= k) mine = 0ull;
        } else {
          uint64_t held[1 + SQ_CAP / 32];
          held[0] = mine;
          mine = 0ull;
#pragma unroll
          for (int j = 0; j < SQ_CAP / 32; ++j) {
            const int e = j * 32 + lane;
            held[1 + j] = e < c ? cands[q * SQ_CAP + e] : 0ull;
          }
          for (int rd = 0; rd < k; ++rd) {
            uint64_t best = held[0];
            int bj = 0;
#pragma unroll
            for (int j = 1; j < 1 + SQ_CAP / 32; ++j)
              if (held[j] > best) {
                best = held[j];
                bj = j;
              }
            const uint64_t mx = warp_max_key(best);
            if (mx == 0ull) break;                 // warp-uniform: nothing left
            if (lane == rd) mine = mx;
            if (best == mx) {                      // one lane: keys differ
#pragma unroll
              for (int j = 0; j < 1 + SQ_CAP / 32; ++j)
                if (j == bj) held[j] = 0ull;
            }
          }
        }
        if (lane < k) lists[q * 32 + lane] = mine;
        const uint64_t kth = __shfl_sync(0xffffffffu, mine, k - 1);
        if (lane == 0) {
          float sk = -FLT_MAX;
          int32_t ik;
          if (kth != 0ull) unpack_key(kth, sk, ik);
          theta[q] = sk;
          cnt[q] = 0;
        }
      }
      named_bar_sync(1, 128);
    }
    // This CTA's list per query (list index = blockIdx.x of 2 * nsplit).
    const int nlists = (int)gridDim.x;
    for (int q = ew; q < nq; q += 4) {
      if (lane < k) {
        const uint64_t key = lists[q * 32 + lane];
        float sc = -FLT_MAX;
        int32_t id = -1;
        if (key != 0ull) unpack_key(key, sc, id);
        const size_t o = ((size_t)q * nlists + blockIdx.x) * k + lane;
        p.part_s[o] = sc;
        p.part_i[o] = id;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, SQ_TMEM_COLS);
  }
  if (threadIdx.x == 0 && *abort_flag) set_error(p.err, kErrTimeout);
}

// ---- host side ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

bool make_map(CUtensorMap* map, const uint16_t* base, int64_t rows, int32_t d, uint32_t box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)d * 2};
  const cuuint32_t box[2] = {(cuuint32_t)BK, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t*>(base), dims, strides,
            box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Test hook of the main kernel's bounded waits (hs_debug_retrieve_wait): the
// wait limit (0: 2 s) and whether every CTA withholds its first stage.
std::atomic<uint64_t> g_ret_wait_limit_ns{0};
std::atomic<int> g_ret_withhold{0};

// The pass over cut lists: the ring, as the others', and the table.
constexpr size_t kCutSmem = 1024 + (size_t)kCutStages * kCutStageBytes + kBarBytes + kEpiSmem +
                            sizeof(CutTable);
static_assert(kCutSmem <= 232448 && sizeof(CutTable) % 4 == 0, "shared memory per CTA");
static_assert(8 * (2 * kCutStages + 4 + 2) + 8 + 8 <= kBarBytes, "barrier area");

template <int KREG, int CL, int RN, bool CUT = false>
hs_status configure_kernel() {
  static std::atomic<uint64_t> done{0};
  return once_per_device(done, [] {
    return cuda_fail(cudaFuncSetAttribute(retrieve_kernel<KREG, CL, RN, CUT>,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          RN > 0 ? 232448 : CUT ? (int)kCutSmem : (int)Ring<CL>::smem),
                     "retrieve smem attribute");
  });
}

// Clusters of two that can be resident at once (one CTA per SM; pairs must
// share a GPC), cached per kernel variant.
template <int KREG>
int64_t max_pairs() {
  static std::atomic<int64_t> per_device[kMaxDeviceOrdinals];   // 0: not yet queried
  const int dev = device_ordinal();
  int64_t cached = dev >= 0 ? per_device[dev].load() - 1 : -1;
  if (cached < 0) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(num_sms() & ~1), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = Ring<2>::smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, retrieve_kernel<KREG, 2, 0, false>, &cfg) != cudaSuccess) n = 0;
    cached = n;
    if (dev >= 0) per_device[dev].store(cached + 1);
  }
  return cached;
}

template <int KREG, int CL, int RN, bool CUT = false>
hs_status launch_kernel(const CUtensorMap& mq, const CUtensorMap& mc, const Params& prm,
                        int64_t grid, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = CL;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = RN > 0 ? res_smem(RN, prm.kb_count) : CUT ? kCutSmem : Ring<CL>::smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = CL > 1 ? 2 : 1;
  return cuda_fail(cudaLaunchKernelEx(&cfg, retrieve_kernel<KREG, CL, RN, CUT>, mq, mc, prm),
                   "retrieve launch");
}

// Unit executors of a launch: pairs of CTAs where there are two query blocks (they
// share corpus tiles) and pairs can be resident, else single CTAs; at most kMaxLists
// / 2, so every query's lists (2 per split, nsplit <= slots) fit the merges.
struct Executors {
  int cl;
  int64_t slots;
};
template <int KREG>
hs_status executors(int64_t Qmax, Executors* out) {
  const int64_t sms = num_sms();
  hs_status st = configure_kernel<KREG, 1, 0>();
  if (st != HS_OK) return st;
  *out = Executors{1, std::min<int64_t>(sms, kMaxLists / 2)};
  if (Qmax > BM) {
    st = configure_kernel<KREG, 2, 0>();
    if (st != HS_OK) return st;
    const int64_t pairs =
        std::min<int64_t>(std::min<int64_t>(max_pairs<KREG>(), sms / 2), kMaxLists / 2);
    if (pairs >= 1) *out = Executors{2, pairs};
  }
  return HS_OK;
}

// Plan and launch for one register-list size.
template <int KREG>
hs_status launch_variant(const uint16_t* corpus, int64_t N, int32_t d, const CUtensorMap& mq,
                         Params& prm, cudaStream_t stream) {
  Executors ex;
  const hs_status st = executors<KREG>(prm.Qmax, &ex);
  if (st != HS_OK) return st;
  const int cl = ex.cl;
  const int64_t slots = ex.slots;
  CUtensorMap mc;
  if (!make_map(&mc, corpus, N, d, BN / cl))
    return fail(HS_ERR_CUDA, "cuTensorMapEncodeTiled failed (driver entry point or arguments)");
  prm.slots = (int32_t)slots;
  prm.cl = cl;
  // With a host-known count the grid covers only the plan's units; with a
  // device count every slot gets a CTA (or pair) and idle ones exit.
  int64_t execs = slots;
  if (!prm.count_dev) {
    const SplitPlan sp = split_plan(prm.Qmax, prm.tiles, prm.k, slots, cl);
    const int64_t units = (int64_t)sp.groups * sp.nsplit;
    if (units < execs) execs = units;
  }
  if (execs < 1) execs = 1;
  return cl == 2 ? launch_kernel<KREG, 2, 0>(mq, mc, prm, execs * 2, stream)
                 : launch_kernel<KREG, 1, 0>(mq, mc, prm, execs, stream);
}

// The same with resident queries.  One query block, so the plan has a split
// per CTA.
template <int KREG, int RN>
hs_status launch_resident(const uint16_t* queries, const uint16_t* corpus, int64_t N, int32_t d,
                          Params& prm, cudaStream_t stream) {
  const hs_status st = configure_kernel<KREG, 1, RN>();
  if (st != HS_OK) return st;
  CUtensorMap mq, mc;
  if (!make_map(&mq, queries, prm.Qmax, d, RQ) || !make_map(&mc, corpus, N, d, RN))
    return fail(HS_ERR_CUDA, "cuTensorMapEncodeTiled failed (driver entry point or arguments)");
  prm.tiles = (N + RN - 1) / RN;
  prm.slots = (int32_t)std::min<int64_t>(num_sms(), kMaxLists / 2);
  prm.cl = 1;
  const SplitPlan sp = split_plan(1, prm.tiles, prm.k, prm.slots, 1);
  return launch_kernel<KREG, 1, RN>(mq, mc, prm, sp.nsplit, stream);
}

}  // namespace

// The fewest lists that a query gets from these executors; with a count that only
// the device knows, over every count up to Q.
static int64_t fewest_lists(int64_t Q, bool device_count, int64_t tiles, const Executors& ex) {
  const int64_t groups = ((Q + BM - 1) / BM + ex.cl - 1) / ex.cl;
  auto lists = [&](int64_t q) { return 2 * split_plan(q, tiles, 16, ex.slots, ex.cl).nsplit; };
  int64_t fewest = lists(Q);
  for (int64_t g = 1; device_count && g < std::min(groups, ex.slots + 1); ++g)
    fewest = std::min<int64_t>(fewest, lists(g * BM * ex.cl));
  return fewest;
}

// One of the two arrays of lists.  Batches of up to RQ queries may be split
// into tiles of 128 rows.
static size_t part_bytes(int64_t Q, int64_t N, int32_t k, int64_t sms) {
  const int64_t few = std::min<int64_t>(Q, RQ) * max_splits(sms, (N + 127) / 128, k);
  const int64_t lists = std::max<int64_t>(Q * max_splits(sms, (N + BN - 1) / BN, k), few);
  return (((size_t)lists * 2 * k * 4) + 255) & ~(size_t)255;
}

// Workspace: lists, large-k lists, then what is cleared (floors, block flags, and
// for k > 16 how many lists of each query and queries of each list were cut), and
// for k > 16 which they were.
// Upper bound over every query count up to Q: a plan's split count is at most
// max_splits() and the grid is at most the SM count, so one workspace serves
// every batch of at most Q queries.
struct Workspace {
  size_t part, list;                    // sizes: two of each, at 0 and 2 * part
  size_t floor, flags, pairs, count, clear_end, queue, at, total;
};
constexpr int kFewSlots = 12;           // of a first pass's lists, at the fewest
static Workspace workspace(int64_t Q, int64_t N, int32_t k) {
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const int64_t sms = num_sms();
  Workspace w{};
  w.part = part_bytes(Q, N, k, sms);
  w.list = k <= 32 ? 0 : up((size_t)sms * kEpi * 2 * k * 4);
  const bool cut = k > 16;
  size_t o = 2 * w.part + 2 * w.list;
  w.floor = o;       o += up((size_t)Q * 4);
  w.flags = o;       o += up((size_t)((Q + BM - 1) / BM) * 4);
  w.pairs = o;       o += cut ? up((size_t)Q * 4) : 0;
  w.count = o;       o += cut ? up((kMaxLists + 1) * 4) : 0;
  w.clear_end = o;
  w.queue = o;       o += cut ? up((size_t)kMaxLists * Q * 4) : 0;
  w.at = o;          o += cut ? up((size_t)Q * (k / kFewSlots) * sizeof(uint2)) : 0;
  w.total = o;
  return w;
}

size_t retrieve_topk_workspace(int64_t Q, int64_t N, int32_t d, int32_t k) {
  if (Q <= 0 || N <= 0 || k <= 0) return 256;
  (void)d;
  return workspace(Q, N, k).total;
}

// Qmax rows of `queries` are addressable; the kernels process the first
// count of them, count = *count_dev (clamped to [0, Qmax]) or Qmax if
// count_dev is NULL.  With inv NULL, scores_out / ids_out get one row per
// query; otherwise n_out rows, row o holding the results of query inv[o].
hs_status launch_retrieve_topk(const uint16_t* queries, int64_t Qmax, const int32_t* count_dev,
                               const int32_t* inv, int64_t n_out, const uint16_t* corpus,
                               int64_t N, int32_t d, int32_t k, float* scores_out,
                               int32_t* ids_out, void* ws, size_t ws_bytes, cudaStream_t stream) {
  unsigned* err = device_error_word();
  if (!err) return fail(HS_ERR_CUDA, "could not resolve the device error word");
  const int64_t sms = num_sms();
  const int64_t tiles = (N + BN - 1) / BN;
  const Workspace L = workspace(Qmax, N, k);
  if (ws_bytes < L.total)
    return fail(HS_ERR_WORKSPACE, "retrieve workspace too small: %zu < %zu", ws_bytes, L.total);
  CUtensorMap mq;
  if (!make_map(&mq, queries, Qmax, d, BM))
    return fail(HS_ERR_CUDA, "cuTensorMapEncodeTiled failed (driver entry point or arguments)");
  char* w = static_cast<char*>(ws);
  Params prm{};
  prm.Qmax = Qmax;
  prm.N = N;
  prm.tiles = tiles;
  prm.count_dev = count_dev;
  prm.k = k;
  prm.kb_count = (d + BK - 1) / BK;
  prm.wait_limit_ns = g_ret_wait_limit_ns.load();
  prm.withhold_first = g_ret_withhold.load();
  prm.part_s = reinterpret_cast<float*>(w);
  prm.part_i = reinterpret_cast<int32_t*>(w + L.part);
  prm.list_s = reinterpret_cast<float*>(w + 2 * L.part);
  prm.list_i = reinterpret_cast<int32_t*>(w + 2 * L.part + L.list);
  prm.qfloor = reinterpret_cast<uint32_t*>(w + L.floor);
  prm.raise_floor = 1;
  uint32_t* block_flags = reinterpret_cast<uint32_t*>(w + L.flags);
  prm.err = err;
  const bool small = Qmax <= SQ_N && k <= 32 && prm.kb_count <= SQ_MAXKB;
  // Up to 64 queries stay in shared memory, which leaves the ring to the
  // corpus.  Tiles of 256 rows cost less per row, tiles of 128 spread a small
  // corpus over twice the SMs and leave wide rows a ring.  us, k = 10, a 128-row
  // query block streamed beside the corpus / resident with tiles of 128 / of
  // 256: 17 queries, 1,000,000 x 768 313 / 237 / 233, 2,000,000 x 256 222 / 172 /
  // 168; 64 queries, 4096 x 384 24.5 / 22.5 / 24.2, 20,000 x 768 30.1 / 34.8 /
  // 30.5, 2,000,000 x 256 177 to 187 / 189 / 173, 1,000,000 x 768 235 to 255 /
  // 240 / 236 to 241.  A stage's batch of 64 over 2,097,152 x 768: 508 -> 475.
  // Where the merge takes k rounds over its lists, tiles of 128 are taken only if
  // those of 256 give as many lists, or too few for short ones (3 queries, 32,768 x
  // 1024, k = 500: 296 with 304 lists, 238 with 256; 1 query, 4096 x 1024, k = 200:
  // 107 with 64 lists of 16, 125 with 32 of 32).
  const bool wide = prm.kb_count <= kResMaxKbWide && (N + 127) / 128 > sms;
  const bool resident = !small && Qmax <= RQ && prm.kb_count <= kResMaxKb &&
                        (wide || k <= kMrMaxK || tiles >= sms || (int64_t)k > 7 * tiles);
  const OutRows rows{inv, n_out};
  const int64_t R = inv ? n_out : Qmax;             // rows the final merge writes
  auto merge = [&](const Params& pm, int32_t kout, float* os, int32_t* oi, OutRows orows,
                   const CutOut cut = CutOut{}) -> hs_status {
    const int64_t nr = orows.inv ? orows.n_out : Qmax;
    if (nr == 0) return HS_OK;
    // Every plan caps its executors (slots) at kMaxLists / 2: the warp merge takes
    // every launch.
    if (2 * (int64_t)pm.slots > kMaxLists)
      return fail(HS_ERR_UNSUPPORTED, "more lists per query than the merge takes");
    // Up to 32 results: a block per row while there is an SM for each (256 rows
    // of 152 lists take 1 to 2 us more than with a warp each), and k is worth it:
    // a block ranks the lists' heads, a warp takes k rounds.  us, block / warp, after
    // the small-batch kernel: 16 lists, k = 4 7.4 / 7.3; 64, k = 6 9.2 / 9.0, k = 8
    // 9.5 / 9.8; 152, k = 8 23.6 / 22.9, k = 16 28.3 / 29.4; after the main kernel:
    // 30, k = 4 16.4 / 16.5; 152, k = 6 61.7 / 62.5; 304, k = 8 43.2 to 47.2 / 41.2 to
    // 46.9, k = 10 48.1 to 53.0 / 47.5 to 53.4, k = 16 67.8 / 71.2.
    // More results: up to twelve rows per SM (1000 rows, k = 50 and 100, 8 and 19
    // us less than with a warp each; 4000 rows 15 more).
    // After the main kernel it is launched in plain stream order: with its
    // blocks waiting beside it, their shared memory cost the next retrieval up to
    // 45 us.  After the small-batch kernel it is launched early, 0.4 us less, but
    // not where that leaves too few SMs free for a block each, as all of them then
    // wait there (8 queries over 19,000 x 128, k = 16: 27.0 early, 17.2 plain).
    const int64_t lists = 2 * split_plan(Qmax, pm.tiles, pm.k, pm.slots, pm.cl).nsplit;
    const bool ranked = small ? 30 * (int64_t)(kout - 4) >= lists : 60 * (int64_t)(kout - 3) >= lists;
    if (ranked && kout <= 32 && nr <= sms) {
      if (small && (lists >= sms || nr <= sms - lists))
        launch_pdl(merge_rank_kernel<32 * 32>, dim3((unsigned)nr), dim3(kMrThreads), 0, stream, pm,
                   os, oi, kout, orows, cut);
      else
        merge_rank_kernel<32 * 32><<<dim3((unsigned)nr), dim3(kMrThreads), 0, stream>>>(
            pm, os, oi, kout, orows, cut);
      return cuda_fail(cudaGetLastError(), "merge launch");
    }
    if (kout > 32 && kout <= kMrMaxK && pm.k <= 32 && nr <= 12 * sms) {
      const int64_t blocks = std::min<int64_t>(nr, 6 * sms);
      merge_rank_kernel<32 * kMrMaxK><<<dim3((unsigned)blocks), dim3(kMrThreads), 0, stream>>>(
          pm, os, oi, kout, orows, cut);
      return cuda_fail(cudaGetLastError(), "merge launch");
    }
    {
      const int64_t blocks = (nr + 7) / 8;          // one warp per row
      const dim3 grid((unsigned)(blocks < sms * 16 ? blocks : sms * 16));
      // lists per query <= 2 * slots (nsplit <= slots): lanes need that / 32
      const int64_t lpl = (2 * (int64_t)pm.slots + 31) / 32;
      // The hand-on costs only the longest lists registers that they need: without
      // it <5> has 78 instead of 114, a third block fits an SM, and the blocks that
      // wait for a retrieval's first free SMs crowd there (256 queries over 20,000 x
      // 384, k = 10: 39.6 us, 37.7 with 114).
      auto* kernel = lpl <= 2    ? merge_warp_kernel<2, true>
                     : lpl <= 3  ? merge_warp_kernel<3, true>
                     : lpl <= 5  ? merge_warp_kernel<5, true>
                     : cut.floor ? merge_warp_kernel<kMaxListsPerLane, true>
                                 : merge_warp_kernel<kMaxListsPerLane, false>;
      launch_pdl(kernel, grid, dim3(256), 0, stream, pm, os, oi, kout, orows, cut);
      return cuda_fail(cudaGetLastError(), "merge launch");
    }
  };
  hs_status st;
  if (small) {
    // Small batch: corpus as the M operand, queries resident (swap-AB).
    CUtensorMap mq16, mc128;
    if (!make_map(&mq16, queries, Qmax, d, SQ_N) || !make_map(&mc128, corpus, N, d, SQ_BM))
      return fail(HS_ERR_CUDA, "cuTensorMapEncodeTiled failed (driver entry point or arguments)");
    static std::atomic<uint64_t> sq_configured{0};
    const hs_status cst = once_per_device(sq_configured, [] {
      return cuda_fail(cudaFuncSetAttribute(retrieve_small_kernel,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)SQ_SMEM),
                       "retrieve smem attribute");
    });
    if (cst != HS_OK) return cst;
    // Lists per query = 2 * nsplit of the plan the merge kernel recomputes
    // (one query block, one group: nsplit = min(slots, tiles, 8192 / k)).
    prm.slots = (int32_t)std::max<int64_t>(1, std::min<int64_t>(sms / 2, kMaxLists / 2));
    prm.cl = 1;
    const SplitPlan sp = split_plan(1, tiles, k, prm.slots, 1);
    const int64_t grid = 2 * (int64_t)sp.nsplit;
    launch_pdl(retrieve_small_kernel, dim3((unsigned)grid), dim3(SQ_THREADS), SQ_SMEM, stream,
               mq16, mc128, prm, (N + SQ_BM - 1) / SQ_BM);
    st = cuda_fail(cudaGetLastError(), "retrieve launch");
  } else {
    // k > 16: how many of a query's k best one of its lists holds on average bounds
    // the slots that a list needs.
    int64_t lists = 0;
    if (k > 16) {
      Executors ex{1, std::min<int64_t>(sms, kMaxLists / 2)};
      if (!resident) {
        st = executors<16>(Qmax, &ex);
        if (st != HS_OK) return st;
      }
      lists = fewest_lists(Qmax, !resident && count_dev,
                           resident && !wide ? (N + 127) / 128 : tiles, ex);
    }
    const int32_t few = 4 * (int64_t)k <= 5 * lists ? kFewSlots : 2 * (int64_t)k <= 7 * lists ? 16 : 32;
    const bool guess = k > 32 ? (int64_t)k <= 32 * tiles : k > 16 && few < 32;
    // The shared per-query floors of the register-list passes start empty, and
    // no query or block is flagged.
    const size_t clear = guess ? L.clear_end - L.floor : (size_t)Qmax * 4;
    const cudaError_t ze = cudaMemsetAsync(prm.qfloor, 0, clear, stream);
    if (ze != cudaSuccess) return cuda_fail(ze, "floor clear");
    // Whole-corpus pass of register lists.
    auto pass = [&](Params& pm, int32_t slots) -> hs_status {
      if (resident) {
        auto* launch = slots <= 8    ? (wide ? launch_resident<8, 256> : launch_resident<8, 128>)
                       : slots <= 12 ? (wide ? launch_resident<12, 256> : launch_resident<12, 128>)
                       : slots <= 16 ? (wide ? launch_resident<16, 256> : launch_resident<16, 128>)
                                     : (wide ? launch_resident<32, 256> : launch_resident<32, 128>);
        return launch(queries, corpus, N, d, pm, stream);
      }
      return slots <= 8    ? launch_variant<8>(corpus, N, d, mq, pm, stream)
             : slots <= 12 ? launch_variant<12>(corpus, N, d, mq, pm, stream)
             : slots <= 16 ? launch_variant<16>(corpus, N, d, mq, pm, stream)
                           : launch_variant<32>(corpus, N, d, mq, pm, stream);
    };
    st = HS_OK;
    if (guess) {
      // More than 16 results: unless the corpus has few tiles an optimistic
      // pass runs first: the register-list kernel (no shared floor: a floor
      // that bounds the list's last entry would cut rows of the top k) over the
      // whole corpus with as many slots as a list is likely to need, merged to
      // the first k of the union of its lists.  A list whose last entry is
      // below the union's k-th best holds every row of its range that can be in
      // the top k, so where no list of a query is cut that way the union's
      // first k are exact.  The merge flags the query blocks where some list
      // may have been cut, and every later kernel skips the others.
      // With rows in no special order a list's share is binomial: 12 slots for
      // an average of 1.25, 16 for 3.5 and 32 for 16 (k = 32 tiles, two lists a
      // tile) leave one of 128 queries cut once in 1,000 batches or less, but
      // for the last (one in 20).  Queries whose best rows lie side by side in
      // the corpus, as chunks of a document do, are cut more often.  Their cut
      // lists alone are run again, the queries of each taken from their places
      // side by side, over that list's rows, from the k-th best score so far as
      // a floor; with min(k, 32) slots they are enough for k <= 32.  The blocks of
      // queries cut again, or at first with 32 slots, are run exactly, from the
      // floor too.  300 queries over 131,072 x 384, 20 neighbours among the best of
      // none, 1 in 100, all of the queries, us: k = 17 94 / 110 / 132, k = 32 101 /
      // 117 / 138 (32 slots from the start 145 / 145 / 146 and 199 / 199 / 205),
      // k = 50 of all 132 (986 with 32 slots, then exactly); 2000 over 262,144 x
      // 768, k = 17 513 / 555 / 709 (558 / 560 / 643), k = 100 of all 868 (6100).
      // What it can cost is one more reading of the corpus, where some query's best
      // crowd in nearly every list: 256 over 262,144 x 1536, k = 17 all 243 (192); and
      // two launches that find work, where a call is short: 256 over 12,000 x 768,
      // k = 17 of half 84 (65).
      // The slots decide the time, as a list starts by taking nearly all it
      // sees: 300 queries over 131,072 x 384, k = 50: 237 us with 32 slots, 146
      // with 16, 126 with 12 (105 with the merge by rank and skipped passes that
      // end at once), k = 32: 199 -> 104; over 4096 x 128, k = 32: 73 -> 41;
      // 1000 over 524,288 x 384, k = 100: 637 -> 450.
      Params pa = prm;
      pa.k = few;
      pa.qfloor = nullptr;
      pa.raise_floor = 0;
      CutOut cut{};
      cut.block = block_flags;
      cut.floor = prm.qfloor;
      if (few < 32) {
        cut.pairs = reinterpret_cast<uint32_t*>(w + L.pairs);
        cut.at = reinterpret_cast<uint2*>(w + L.at);
        cut.most = k / few;
      }
      st = pass(pa, few);
      if (few < 32) {
        CutQueues& c = cut.queues;
        c.count = reinterpret_cast<uint32_t*>(w + L.count);
        c.queue = reinterpret_cast<uint32_t*>(w + L.queue);
        c.list_k = few;
        c.slots = pa.slots;
        c.cl = pa.cl;
        c.tiles = pa.tiles;
        c.Q = Qmax;
        c.count_dev = count_dev;
        c.tile_rows = resident && !wide ? 128 : BN;
        // The lists of this pass go where the first pass's were: at most
        // Q * k / few * 2 * parts of 32 entries, where max_splits() * 2 * Q * k fit.
        c.most_parts = (int32_t)std::min<int64_t>(8, max_splits(sms, tiles, k) * 3 / 8);
      }
      if (st == HS_OK) st = merge(pa, k, scores_out, ids_out, rows, cut);
      if (st != HS_OK) return st;
      count_launches(2);
      if (few < 32) {
        CUtensorMap mq1, mc;
        if (!make_map(&mq1, queries, Qmax, d, 1) || !make_map(&mc, corpus, N, d, kCutRows))
          return fail(HS_ERR_CUDA, "cuTensorMapEncodeTiled failed (driver entry point or arguments)");
        Params pc = prm;
        pc.k = k <= 32 ? k : 32;
        pc.raise_floor = k <= 32;
        pc.cut = cut.queues;
        st = configure_kernel<0, 1, 0, true>();
        if (st == HS_OK) st = launch_kernel<0, 1, 0, true>(mq1, mc, pc, sms, stream);
        if (st != HS_OK) return st;
        launch_pdl(cut_merge_kernel,
                   dim3((unsigned)std::min<int64_t>(std::max<int64_t>(R, 1), 4 * sms)),
                   dim3(kCutThreads), 0, stream, pc, scores_out, ids_out, k, rows, cut, (int)sms);
        st = cuda_fail(cudaGetLastError(), "cut merge launch");
        if (st != HS_OK) return st;
        count_launches(2);
        if (k <= 32) return HS_OK;
      }
      prm.only = block_flags;
    }
    if (k <= 32) {
      st = pass(prm, k);
    } else {
      // The exact path of large k: of the flagged blocks, whose queries start
      // with the floor that the merges gave, or of all.
      st = launch_variant<0>(corpus, N, d, mq, prm, stream);
    }
  }
  if (st != HS_OK) return st;
  st = merge(prm, k, scores_out, ids_out, rows);
  if (st != HS_OK) return st;
  count_launches(R > 0 ? 2 : 1);  // retrieve_kernel + merge_warp_kernel
  return HS_OK;
}

}  // namespace hs

/*
 * Diagnostics only (declared in hs.h as hs_debug_retrieve_wait).
 */
extern "C" hs_status hs_debug_retrieve_wait(uint64_t limit_ns, int32_t withhold_first) {
  hs::clear_last_error();
  if (limit_ns > hs::kWaitLimitNs) return hs::fail(HS_ERR_INVALID_ARG, "limit above 2 s");
  if (withhold_first < 0 || withhold_first > 1)
    return hs::fail(HS_ERR_INVALID_ARG, "withhold_first must be 0 or 1");
  hs::g_ret_wait_limit_ns.store(limit_ns);
  hs::g_ret_withhold.store(withhold_first);
  return HS_OK;
}
