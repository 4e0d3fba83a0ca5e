// K1 + K2 + K5 fused for a small query batch: fingerprint every query row,
// merge exactly-equal rows into unique queries with an inverse map, and
// gather the unique rows for retrieval — one launch.
//
// Paper: the signature of a node (Section 3.3, Eq. 2), the merge of a node
// into an equal node already in the window (Section 3.3, "Dynamic Fusion and
// Reuse Mechanism" (I)) and the merge sets M(v*) executed once (Appendix A.2).
// The results are those of hs_fingerprint, hs_unique_inverse and
// hs_scatter_results(queries, unique_idx) called in turn.
//
// Small batches are latency-bound: each of those calls is a few microseconds
// of launch and dependency latency around very little work.  Here every merging
// CTA runs the whole merge on its own — a key of every row, the hash table in
// shared memory, the verification, the scan — so the CTAs never wait for one
// another, and they split only the final gather.  The redundant work is cheap
// at these sizes: at most 256 rows, read from L2.  CTA 0 alone writes
// unique_idx, inverse and the unique count.
//
// The merge does not need the fingerprints, whose hash is the longest chain
// here (a warp per row, fnv_warp.cuh): its key is a hash of the whole row that
// a warp takes in one round of loads (multiply-xorshift of each 16-byte piece
// with its place, added up), and further CTAs of the same launch compute the
// fingerprints meanwhile.  Given fingerprints are taken as the keys.
//
// Bound by the launch and its dependent round trips (keys, verify, gather); at
// 256 rows of 768 by each CTA's reading of all rows.  us with the launch, where
// one thread hashed each row first: 1 row of 768 3.6 (15.0), 64 rows 7.0
// (17.6), 256 rows 16.6 (28.1).
//
// Exactness: rows are grouped by key (the table keeps the smallest row index
// per key), then every row whose group leader is another row is compared with
// it in full.  A row that differs from its leader (a collision) is re-grouped
// by a warp in ascending row order: its leader is the first earlier row with
// the same key that leads its own group and has equal contents, else itself.
#include "fnv_warp.cuh"
#include "hs_internal.cuh"
#include "row_table.cuh"

namespace hs {
namespace {

using namespace table;

constexpr int kQmMaxRows = 256;             // the first threads take a row each
static_assert(kQmMaxRows <= 256 && kQmMaxRows >= HS_MERGE_QUERIES_MAX, "a thread per row");
constexpr int kQmLog2 = table_log2(kQmMaxRows);
constexpr int kQmSlots = (1 << kQmLog2) + 1;
constexpr int kQmMaxCtas = 32;
constexpr int kQmRows = 4;                  // rows a group takes side by side for their keys
constexpr int kQmPieces = 3;                // 16-byte pieces per lane and row in flight
constexpr int kQmUnroll = 4;                // independent 16-byte copies in flight per thread

__device__ __forceinline__ bool same4(const uint4& a, const uint4& b) {
  return a.x == b.x && a.y == b.y && a.z == b.z && a.w == b.w;
}

// Hash of one 16-byte piece at place v of its row; a row's key is the sum of
// its pieces' hashes, so lanes and rounds add up in any order.
__device__ __forceinline__ uint64_t piece_key(const uint4& x, int v) {
  constexpr uint64_t kMul = 0x9E3779B97F4A7C15ull, kFin = 0xD6E8FEB86659FD93ull;
  uint64_t h = ((((uint64_t)x.y << 32) | x.x) ^ ((uint64_t)(v + 1) * kFin)) * kMul;
  h = (h ^ (h >> 32) ^ (((uint64_t)x.w << 32) | x.z)) * kMul;
  return h ^ (h >> 29);
}

// CTAs [0, merge_ctas) merge; the others hash rows (fp_in NULL, fp_out not).
template <int THREADS>
__global__ void __launch_bounds__(THREADS) merge_queries_kernel(
    const uint4* __restrict__ q, int n, int nv, uint64_t seed, const uint64_t* __restrict__ fp_in,
    uint64_t* __restrict__ fp_out, int32_t* __restrict__ n_unique,
    int32_t* __restrict__ unique_idx, int32_t* __restrict__ inverse, uint4* __restrict__ uq,
    int merge_ctas) {
  pdl_wait();
  pdl_trigger();
  if ((int)blockIdx.x >= merge_ctas) {
    const int warps = ((int)gridDim.x - merge_ctas) * (THREADS / 32);
    for (int r = ((int)blockIdx.x - merge_ctas) * (THREADS / 32) + (int)(threadIdx.x >> 5);
         r < n; r += warps) {
      const uint64_t h = fnv::hash_row_warp<true>(
          reinterpret_cast<const uint32_t*>(q + (size_t)r * nv), nv * 4, seed);
      if ((threadIdx.x & 31) == 0) fp_out[r] = h;
    }
    return;
  }
  __shared__ uint64_t s_fp[kQmMaxRows];
  __shared__ uint64_t s_keys[kQmSlots];
  __shared__ uint32_t s_idx[kQmSlots];
  __shared__ int32_t s_rep[kQmMaxRows];
  __shared__ int32_t s_uid[kQmMaxRows];
  __shared__ int32_t s_uidx[kQmMaxRows];
  __shared__ int32_t s_list[kQmMaxRows];
  __shared__ uint8_t s_diff[kQmMaxRows];
  __shared__ int32_t s_warp[THREADS / 32];
  __shared__ int32_t s_nlist, s_ncoll;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int log2T = table_log2(n);
  const int T1 = (1 << log2T) + 1;
  const bool row = tid < n;

  for (int s = tid; s < T1; s += THREADS) {
    s_keys[s] = kEmpty;
    s_idx[s] = kNoRow;
  }
  if (tid < kQmMaxRows) s_diff[tid] = 0;
  if (tid == 0) s_nlist = s_ncoll = 0;

  // 1. every row's key
  if (fp_in) {
    if (row) {
      s_fp[tid] = __ldg(fp_in + tid);
      if (blockIdx.x == 0 && fp_out) fp_out[tid] = s_fp[tid];
    }
  } else {
    // A group of lanes per row (fewer than 32 for short rows), and kQmRows
    // rows side by side.
    int group = 32;
    while (group > 1 && group / 2 >= nv) group /= 2;
    const int groups = THREADS / group, gl = tid & (group - 1);
    for (int base = 0; base < n; base += groups * kQmRows) {     // the same for every lane
      const int r0 = base + tid / group;
      uint64_t h[kQmRows];
#pragma unroll
      for (int r = 0; r < kQmRows; ++r) h[r] = 0;
      for (int v0 = 0; v0 < nv; v0 += group * kQmPieces) {
        uint4 x[kQmRows][kQmPieces];
#pragma unroll
        for (int r = 0; r < kQmRows; ++r)
#pragma unroll
          for (int p = 0; p < kQmPieces; ++p) {
            const int v = v0 + p * group + gl;
            if (r0 + r * groups < n && v < nv)
              x[r][p] = __ldg(q + (size_t)(r0 + r * groups) * nv + v);
          }
#pragma unroll
        for (int r = 0; r < kQmRows; ++r)
#pragma unroll
          for (int p = 0; p < kQmPieces; ++p) {
            const int v = v0 + p * group + gl;
            if (r0 + r * groups < n && v < nv) h[r] += piece_key(x[r][p], v);
          }
      }
#pragma unroll
      for (int r = 0; r < kQmRows; ++r) {
        if (base + r * groups >= n) break;
        for (int o = group / 2; o > 0; o >>= 1) h[r] += __shfl_xor_sync(0xffffffffu, h[r], o);
        if (gl == 0 && r0 + r * groups < n) s_fp[r0 + r * groups] = h[r];
      }
    }
  }
  __syncthreads();
  const uint64_t f = row ? s_fp[tid] : 0ull;

  // 2. table: each key's smallest row index; rep = that row
  insert_row(s_keys, s_idx, log2T, row, f, (uint32_t)tid);
  __syncthreads();
  int32_t rep = tid;
  if (row) {
    const uint32_t v = s_idx[find_key(s_keys, f, log2T)];
    rep = v < (uint32_t)n ? (int32_t)v : tid;
    s_rep[tid] = rep;
    if (rep != tid) s_list[atomicAdd(&s_nlist, 1)] = tid;
  }
  __syncthreads();

  // 3. verify every listed row against its leader, all 16-byte pairs in flight
  const int m = s_nlist;
  const int items = m * nv;
  for (int b = tid; b < items; b += THREADS * kQmUnroll) {
    uint4 x[kQmUnroll], y[kQmUnroll];
    int ra[kQmUnroll];
#pragma unroll
    for (int u = 0; u < kQmUnroll; ++u) {
      const int it = b + u * THREADS;
      ra[u] = -1;
      if (it < items) {
        const int li = it / nv, v = it - li * nv;
        ra[u] = s_list[li];
        x[u] = __ldg(q + (size_t)ra[u] * nv + v);
        y[u] = __ldg(q + (size_t)s_rep[ra[u]] * nv + v);
      }
    }
#pragma unroll
    for (int u = 0; u < kQmUnroll; ++u)
      if (ra[u] >= 0 && !same4(x[u], y[u])) s_diff[ra[u]] = 1;
  }
  __syncthreads();
  if (row && s_diff[tid]) atomicAdd(&s_ncoll, 1);
  __syncthreads();

  // 4. collisions (rows that differ from their leader): warp 0, ascending
  if (s_ncoll > 0 && warp == 0) {
    for (int a0 = 0; a0 < n; a0 += 32) {
      unsigned cm = __ballot_sync(0xffffffffu, a0 + lane < n && s_diff[a0 + lane]);
      while (cm) {
        const int a = a0 + __ffs(cm) - 1;
        cm &= cm - 1;
        const uint64_t fa = s_fp[a];
        int found = a;
        for (int j0 = 0; j0 < a && found == a; j0 += 32) {
          const int j = j0 + lane;
          unsigned cand = __ballot_sync(0xffffffffu, j < a && s_fp[j] == fa && s_rep[j] == j);
          while (cand && found == a) {
            const int jj = j0 + __ffs(cand) - 1;
            cand &= cand - 1;
            bool eq = true;
            for (int v = lane; v < nv; v += 32)
              eq &= same4(__ldg(q + (size_t)jj * nv + v), __ldg(q + (size_t)a * nv + v));
            if (__all_sync(0xffffffffu, eq)) found = jj;
          }
        }
        if (lane == 0) s_rep[a] = found;
        __syncwarp();
      }
    }
  }
  __syncthreads();

  // 5. ordinals in first-occurrence order
  if (row) rep = s_rep[tid];
  const bool lead = row && rep == tid;
  const unsigned bal = __ballot_sync(0xffffffffu, lead);
  if (lane == 0) s_warp[warp] = __popc(bal);
  __syncthreads();
  int32_t off = 0, total = 0;
#pragma unroll
  for (int w = 0; w < THREADS / 32; ++w) {
    off += w < warp ? s_warp[w] : 0;
    total += s_warp[w];
  }
  if (lead) {
    const int32_t u = off + __popc(bal & ((1u << lane) - 1u));
    s_uid[tid] = u;
    s_uidx[u] = tid;
  }
  __syncthreads();
  if (blockIdx.x == 0 && row) {
    inverse[tid] = s_uid[rep];
    unique_idx[tid] = tid < total ? s_uidx[tid] : 0;
    if (tid == 0) *n_unique = total;
  }

  // 6. gather the unique rows, split over the CTAs
  const int gitems = total * nv;
  const int gstride = merge_ctas * THREADS;
  for (int b = blockIdx.x * THREADS + tid; b < gitems; b += gstride * kQmUnroll) {
    uint4 x[kQmUnroll];
    int dst[kQmUnroll];
#pragma unroll
    for (int u = 0; u < kQmUnroll; ++u) {
      const int it = b + u * gstride;
      dst[u] = -1;
      if (it < gitems) {
        const int g = it / nv, v = it - g * nv;
        x[u] = __ldg(q + (size_t)s_uidx[g] * nv + v);
        dst[u] = it;
      }
    }
#pragma unroll
    for (int u = 0; u < kQmUnroll; ++u)
      if (dst[u] >= 0) uq[dst[u]] = x[u];
  }
}

}  // namespace

hs_status launch_merge_queries(const uint16_t* queries, int64_t n, int32_t dim, uint64_t seed,
                               const uint64_t* fp_in, uint64_t* fp_out, int32_t* n_unique,
                               int32_t* unique_idx, int32_t* inverse, uint16_t* uq,
                               cudaStream_t stream) {
  if (n == 0)
    return cuda_fail(cudaMemsetAsync(n_unique, 0, sizeof(int32_t), stream), "n_unique clear");
  const int nv = dim / 8;                     // 16-byte vectors per row
  const int64_t work = n * (int64_t)nv;
  // Few pieces leave most of 512 threads idle at every barrier.  us, 256 / 512: 1 row
  // of 8 3.1 / 3.4, 64 of 16 4.0 / 4.2, 7 of 768 (672 pieces) 4.0 / 4.1, 64 of 128 (1024)
  // 5.1 / 4.9, 64 of 768 9.4 / 7.3.
  const int threads = work <= 640 ? 256 : 512;
  int64_t grid = (work + threads * kQmUnroll - 1) / (threads * kQmUnroll);
  grid = grid < 1 ? 1 : (grid > kQmMaxCtas ? kQmMaxCtas : grid);
  const int hash = !fp_in && fp_out ? (int)((n + threads / 32 - 1) / (threads / 32)) : 0;
  launch_pdl(threads == 256 ? merge_queries_kernel<256> : merge_queries_kernel<512>,
             dim3((unsigned)(grid + hash)), dim3(threads), 0, stream,
             reinterpret_cast<const uint4*>(queries), (int)n, nv, seed, fp_in, fp_out, n_unique,
             unique_idx, inverse, reinterpret_cast<uint4*>(uq), (int)grid);
  count_launches(1);
  return cuda_fail(cudaGetLastError(), "merge_queries launch");
}

}  // namespace hs
