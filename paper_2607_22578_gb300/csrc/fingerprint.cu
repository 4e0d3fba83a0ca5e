// K1: per-row 64-bit FNV-1a fingerprints over int32 token rows — the D_in
// part of the node semantic signature Sig(v) (Section 3.3, Eq. 2).
//
// FNV-1a is a serial chain over the octets of one row, so parallelism comes
// from rows: each lane of a warp owns one row at a time and hashes it in
// chunks of 32 tokens, straight-line from registers.
// The octet rounds themselves are in fnv.cuh.
#include <algorithm>

#include "fnv_warp.cuh"
#include "hs_internal.cuh"

namespace hs {
namespace {

using namespace fnv;

// A lane loads its next chunk of T = 32 tokens with 16- or 32-byte loads
// straight into registers one chunk ahead of the chunk it hashes (NB register
// buffers).  A lane that has issued its row's last chunk claims the next
// unclaimed row of its warp's range (lengths prefetched 64 rows ahead and
// handed out by shuffle).
//
// Chunks start on a 16-byte boundary, so a row that does not gets up to three
// tokens of the chunk before its first, and its last chunk may run past its
// length.  Both are hashed as zeros: a round on a zero octet is a plain
// multiply by the prime, which is odd and so has an inverse mod 2^64.  The
// state is multiplied by the inverse once per padding octet (a table of
// powers), before a row's first chunk and after its last, and comes out
// exactly as if the padding had not been there.  So every lane runs the same
// straight-line hash whatever its row's start and length, in one pass.
//
// Where there are rows enough, 16 warps an SM (all that the two buffers' registers
// leave) share their time between a chunk's arrival and its chain: issue slots 56 to
// 59 % busy, DRAM at 3.2 to 4.2 TB/s (400,000 unaligned rows of 333 words, aligned
// ones of 64 to 256).  200,000 rows of 512 tokens: 81 us, 5.0 TB/s; 400,000 of 8 to 36: 19.6 us
// (23.6 as a pass over full chunks and a second one over the rests); 20,011 rows at a
// stride of 333: 19 us (75 hashing word by word), where the chain bounds it.  Rests
// queued and hashed 32 at a time, masks or steps left out by a vote of the warp
// (400,000 rows of 64 to 512: 113 -> 125), and loads with a 256-byte prefetch or a
// bulk prefetch to L2 were each slower.  Long rows of unequal lengths go in those two
// passes (two_passes below), rows of less than a chunk to the second alone.
//
// A chunk whose tokens are all below 65536 (in every live lane) takes the
// two-round small-token hash; otherwise the whole chunk takes the octet-wise
// rounds, which are exact for every token.

template <int VB>
__device__ __forceinline__ void load_vec(const int32_t* p, uint32_t* x) {
  if constexpr (VB == 32) {
    asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]),
                   "=r"(x[6]), "=r"(x[7])
                 : "l"(p));
  } else {
    asm volatile("ld.global.nc.L1::no_allocate.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3])
                 : "l"(p));
  }
}

constexpr int kChunk = 32;      // T: tokens per chunk
constexpr int kFpThreads = 256;

// kUnpad.v[t] = prime^-(4 t): undoes t zero tokens.
struct Unpad {
  uint64_t v[kChunk + 1];
};
constexpr Unpad make_unpad() {
  Unpad u{};
  u.v[0] = 1;
  for (int t = 1; t <= kChunk; ++t) u.v[t] = u.v[t - 1] * power(inverse_prime(), 4);
  return u;
}
static_assert(make_unpad().v[1] * kPrime * kPrime * kPrime * kPrime == 1, "inverse of the prime");
__constant__ Unpad kUnpad = make_unpad();

// VB bytes per load, K loads per chunk, NB register buffers; stride >= T.  MASK: a
// chunk may hold tokens that are not the row's (lengths, or a stride that is no
// multiple of T); HEAD: and rows may start off a 16-byte boundary (4-byte
// aligned), VB is then 16.
template <int VB, int K, int NB, bool MASK, bool HEAD>
__global__ void __launch_bounds__(kFpThreads) fingerprint_kernel(
    const int32_t* __restrict__ tokens, int64_t n, int32_t stride,
    const int32_t* __restrict__ lens, uint64_t seed, uint64_t* __restrict__ fp_out,
    int64_t rows_per_warp, unsigned* err) {
  pdl_wait();
  pdl_trigger();
  constexpr int W = VB / 4;  // tokens per vector load
  constexpr int T = W * K;   // tokens per chunk
  static_assert(T == kChunk && (!HEAD || (MASK && W == 4)), "chunk of 32 tokens, offsets below 4");
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t r_begin = warp * rows_per_warp;
  if (r_begin >= n) return;
  const int64_t r_end = min(n, r_begin + rows_per_warp);
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t seed_lo = (uint32_t)seed, seed_hi = (uint32_t)(seed >> 32);
  const int32_t* const tokens_end = tokens + n * (int64_t)stride;

  // Issue side: the row being loaded, its next chunk's first token (-3 ... -1
  // in a first chunk that starts before the row), its length.
  int64_t irow = -1;
  int32_t ipos = 0, ilen = 0;
  uint32_t buf[NB][T];
  int64_t brow[NB];
  int32_t bend[NB];              // tokens [pad, bend) of the buffer are the row's ...
  int32_t bpos[NB];              // ... with pad = max(0, -bpos)
  bool blast[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    brow[b] = -1;
    bend[b] = bpos[b] = 0;
    blast[b] = false;
  }
  uint32_t lo = seed_lo, hi = seed_hi;

  int64_t next = r_begin;
  int64_t wbase = r_begin;
  auto len_of = [&](int64_t r) -> int32_t {
    return r < r_end ? (lens ? __ldg(lens + r) : stride) : 0;
  };
  int32_t len_a = len_of(wbase + lane), len_b = len_of(wbase + 32 + lane);

  auto claim = [&]() {
    unsigned need = __ballot_sync(0xffffffffu, irow < 0);
    while (need != 0u && next < r_end) {
      const int64_t avail = r_end - next;
      const int rank = __popc(need & lanemask_lt());
      const int off = (int)(next - wbase) + (irow < 0 ? rank : 0);
      const int32_t La = __shfl_sync(0xffffffffu, len_a, off & 31);
      const int32_t Lb = __shfl_sync(0xffffffffu, len_b, off & 31);
      if (irow < 0 && rank < avail) {
        const int32_t L = off < 32 ? La : Lb;
        if (L < 0 || L > stride) {                       // reported, fingerprint 0
          set_error(err, kErrInvalidArg);
          fp_out[next + rank] = 0ull;
        } else if (L == 0) {
          fp_out[next + rank] = seed;
        } else {
          irow = next + rank;
          ilen = L;
          ipos = 0;
          if (HEAD)
            ipos = -(int32_t)((reinterpret_cast<uintptr_t>(tokens + irow * (int64_t)stride) >> 2) & 3u);
        }
      }
      next += min((int64_t)__popc(need), avail);
      if (next - wbase >= 32) {
        wbase += 32;
        len_a = len_b;
        len_b = len_of(wbase + 32 + lane);
      }
      need = __ballot_sync(0xffffffffu, irow < 0);
    }
  };

  // Load this lane's next chunk into buffer b: the pieces that hold one of
  // the row's tokens.  A piece that would leave the token array (only before
  // the first row's start and past the last row's end) is read word by word.
  auto issue = [&](int b) {
    brow[b] = irow;
    if (irow >= 0) {
      const int32_t* src = tokens + irow * (int64_t)stride + ipos;
#pragma unroll
      for (int j = 0; j < K; ++j) {
        const int32_t* p = src + j * W;
        if (!MASK || ipos + j * W < ilen) {
          if (!HEAD || (p >= tokens && p + W <= tokens_end)) {
            load_vec<VB>(p, &buf[b][j * W]);
          } else {
#pragma unroll
            for (int i = 0; i < W; ++i)
              buf[b][j * W + i] = p + i >= tokens && p + i < tokens_end ? (uint32_t)__ldg(p + i) : 0u;
          }
        }
      }
      bpos[b] = ipos;
      bend[b] = min(T, ilen - ipos);
      ipos += T;
      blast[b] = ipos >= ilen;
      if (blast[b]) irow = -1;
    }
  };

  // Hash buffer b (every lane, live or not: an idle lane's result is dropped).
  auto consume = [&](int b) {
    const bool live = brow[b] >= 0, first = live && bpos[b] <= 0;
    lo = first ? seed_lo : lo;
    hi = first ? seed_hi : hi;
    if (HEAD && first) {
      const uint64_t h = seed * kUnpad.v[-bpos[b]];
      lo = (uint32_t)h;
      hi = (uint32_t)(h >> 32);
    }
    if (MASK) {
      uint32_t own = bend[b] >= T ? 0xffffffffu : (1u << bend[b]) - 1u;
      if (HEAD && bpos[b] < 0) own &= 0xffffffffu << -bpos[b];
#pragma unroll
      for (int t = 0; t < T; ++t)
        if (!((own >> t) & 1u)) buf[b][t] = 0u;
    }
    uint32_t any = 0;
#pragma unroll
    for (int t = 0; t < T; ++t) any |= buf[b][t];
    if (__all_sync(0xffffffffu, !live || (any >> 16) == 0u)) {
#pragma unroll
      for (int t = 0; t < T; ++t) hash_word_small(lo, hi, buf[b][t]);
    } else {
#pragma unroll
      for (int t = 0; t < T; ++t) hash_word_full(lo, hi, buf[b][t]);
    }
    if (live && blast[b]) {
      const uint64_t h = ((uint64_t)hi << 32) | lo;
      fp_out[brow[b]] = MASK ? h * kUnpad.v[T - bend[b]] : h;
    }
    brow[b] = -1;
  };

  // Chunks 0 .. NB-2 in flight before the first hash; then each step loads
  // chunk c + NB - 1 and hashes chunk c.
#pragma unroll
  for (int b = 0; b < NB - 1; ++b) {
    claim();
    issue(b);
  }
  for (;;) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      claim();
      issue((b + NB - 1) % NB);
      consume(b);
    }
    bool pending = irow >= 0;
#pragma unroll
    for (int b = 0; b < NB; ++b) pending |= brow[b] >= 0;
    if (!__any_sync(0xffffffffu, pending) && next >= r_end) break;
  }
}

// ---- few rows: a warp per row -------------------------------------------------------------
// Bound by the latency of one row, which a warp cuts to eight prefix xors and
// 32 rounds per 1024 octets (fnv_warp.cuh).  It costs about three times the
// instructions of a lane per row, so it is for batches that leave most of the
// GPU idle.  A row of 1536 octets takes 3.5 us with its launch where the chain takes 14.4.
template <bool VEC>
__global__ void __launch_bounds__(128) fingerprint_warp_kernel(
    const int32_t* __restrict__ tokens, int64_t n, int32_t stride,
    const int32_t* __restrict__ lens, uint64_t seed, uint64_t* __restrict__ fp_out,
    unsigned* err) {
  pdl_wait();
  pdl_trigger();
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n; r += warps) {
    const int32_t L = lens ? __ldg(lens + r) : stride;
    const bool bad = L < 0 || L > stride;                  // reported, fingerprint 0
    uint64_t h = 0;
    if (!bad)
      h = hash_row_warp<VEC>(reinterpret_cast<const uint32_t*>(tokens + r * (int64_t)stride), L,
                             seed);
    if ((threadIdx.x & 31) == 0) {
      if (bad) set_error(err, kErrInvalidArg);
      fp_out[r] = h;
    }
  }
}

// ---- the tokens past a row's full chunks, or all of a short row: a thread per row ------
// MAX tokens at most.  The chunk pass below has left the state of rows of a chunk and
// more, where there can be any.
template <int MAX, bool VEC>
__global__ void __launch_bounds__(kFpThreads) fingerprint_rests_kernel(
    const int32_t* __restrict__ tokens, int64_t n, int32_t stride,
    const int32_t* __restrict__ lens, uint64_t seed, uint64_t* __restrict__ fp_out,
    unsigned* err) {
  pdl_wait();
  pdl_trigger();
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int32_t L = lens ? __ldg(lens + r) : stride;
    if (L < 0 || L > stride) {                             // reported, fingerprint 0
      set_error(err, kErrInvalidArg);
      fp_out[r] = 0ull;
      continue;
    }
    const int32_t rest = L % kChunk;
    if (L >= kChunk && rest == 0) continue;
    const uint64_t h = L >= kChunk ? fp_out[r] : seed;
    uint32_t lo = (uint32_t)h, hi = (uint32_t)(h >> 32);
    hash_tokens<MAX, VEC>(lo, hi, tokens + r * (int64_t)stride + (L - rest), rest);
    fp_out[r] = ((uint64_t)hi << 32) | lo;
  }
}

// ---- full chunks only (the first pass of hs_merge_rows) -----------------------------------
template <int VB, int K, int NB>
__global__ void __launch_bounds__(256) fingerprint_chunks_kernel(
    const int32_t* __restrict__ tokens, int64_t n, int32_t stride,
    const int32_t* __restrict__ lens, uint64_t seed, uint64_t* __restrict__ fp_out,
    int64_t rows_per_warp) {
  pdl_wait();
  pdl_trigger();
  constexpr int W = VB / 4;  // tokens per vector load
  constexpr int T = W * K;   // tokens per chunk
  static_assert(T == kChunk, "chunk size shared with the tail pass");
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t r_begin = warp * rows_per_warp;
  if (r_begin >= n) return;
  const int64_t r_end = min(n, r_begin + rows_per_warp);
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t seed_lo = (uint32_t)seed, seed_hi = (uint32_t)(seed >> 32);

  // Issue side: the row being loaded, the next chunk's start, the end of its
  // full chunks.
  int64_t irow = -1;
  int32_t ipos = 0, iend = 0;
  uint32_t buf[NB][T];
  int64_t brow[NB];
  bool bfirst[NB], blast[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    brow[b] = -1;
    bfirst[b] = blast[b] = false;
  }
  uint32_t lo = seed_lo, hi = seed_hi;

  int64_t next = r_begin;
  int64_t wbase = r_begin;
  auto len_of = [&](int64_t r) -> int32_t {
    return r < r_end ? (lens ? __ldg(lens + r) : stride) : 0;
  };
  int32_t len_a = len_of(wbase + lane), len_b = len_of(wbase + 32 + lane);

  auto claim = [&]() {
    unsigned need = __ballot_sync(0xffffffffu, irow < 0);
    while (need != 0u && next < r_end) {
      const int64_t avail = r_end - next;
      const int rank = __popc(need & lanemask_lt());
      const int off = (int)(next - wbase) + (irow < 0 ? rank : 0);
      const int32_t La = __shfl_sync(0xffffffffu, len_a, off & 31);
      const int32_t Lb = __shfl_sync(0xffffffffu, len_b, off & 31);
      if (irow < 0 && rank < avail) {
        const int32_t L = off < 32 ? La : Lb;
        if (L >= T && L <= stride) {
          irow = next + rank;
          ipos = 0;
          iend = (L / T) * T;
        }
      }
      next += min((int64_t)__popc(need), avail);
      if (next - wbase >= 32) {
        wbase += 32;
        len_a = len_b;
        len_b = len_of(wbase + 32 + lane);
      }
      need = __ballot_sync(0xffffffffu, irow < 0);
    }
  };

  // Load this lane's next full chunk into buffer b.
  auto issue = [&](int b) {
    brow[b] = irow;
    if (irow >= 0) {
      const int32_t* src = tokens + irow * (int64_t)stride + ipos;
#pragma unroll
      for (int j = 0; j < K; ++j) load_vec<VB>(src + j * W, &buf[b][j * W]);
      bfirst[b] = ipos == 0;
      ipos += T;
      blast[b] = ipos == iend;
      if (blast[b]) irow = -1;
    }
  };

  // Hash buffer b (every lane, live or not: an idle lane's result is dropped).
  auto consume = [&](int b) {
    const bool live = brow[b] >= 0;
    lo = (live && bfirst[b]) ? seed_lo : lo;
    hi = (live && bfirst[b]) ? seed_hi : hi;
    uint32_t any = 0;
#pragma unroll
    for (int t = 0; t < T; ++t) any |= buf[b][t];
    if (__all_sync(0xffffffffu, !live || (any >> 16) == 0u)) {
#pragma unroll
      for (int t = 0; t < T; ++t) hash_word_small(lo, hi, buf[b][t]);
    } else {
#pragma unroll
      for (int t = 0; t < T; ++t) hash_word_full(lo, hi, buf[b][t]);
    }
    if (live && blast[b]) fp_out[brow[b]] = ((uint64_t)hi << 32) | lo;
    brow[b] = -1;
  };

  // Chunks 0 .. NB-2 in flight before the first hash; then each step loads
  // chunk c + NB - 1 and hashes chunk c.
#pragma unroll
  for (int b = 0; b < NB - 1; ++b) {
    claim();
    issue(b);
  }
  for (;;) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      claim();
      issue((b + NB - 1) % NB);
      consume(b);
    }
    bool pending = irow >= 0;
#pragma unroll
    for (int b = 0; b < NB; ++b) pending |= brow[b] >= 0;
    if (!__any_sync(0xffffffffu, pending) && next >= r_end) break;
  }
}

template <int VB, int K, int NB, bool MASK, bool HEAD>
hs_status launch_rows(const int32_t* tokens, int64_t n, int32_t stride, const int32_t* lens,
                      uint64_t seed, uint64_t* fp_out, unsigned* err, cudaStream_t stream) {
  // Resident warps per SM at this kernel's register count (queried once per
  // device).
  static std::atomic<int> per_device[kMaxDeviceOrdinals];
  const int dev = device_ordinal();
  int warps_per_sm = dev >= 0 ? per_device[dev].load() : 0;
  if (warps_per_sm == 0) {
    int blocks = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &blocks, fingerprint_kernel<VB, K, NB, MASK, HEAD>, kFpThreads, 0);
    if (e != cudaSuccess) return cuda_fail(e, "fingerprint occupancy");
    warps_per_sm = blocks > 0 ? blocks * (kFpThreads / 32) : 8;
    if (dev >= 0) per_device[dev].store(warps_per_sm);
  }
  const int64_t sms = num_sms();
  const int64_t warps_target = sms * warps_per_sm;
  int64_t rpw = (n + warps_target - 1) / warps_target;
  if (rpw < 32) rpw = 32;
  const int64_t warps = (n + rpw - 1) / rpw;
  // Few warps: one-warp blocks, so they spread over all SMs.
  const int threads = warps >= sms * 8 ? kFpThreads : 32;
  const int64_t blocks = (warps * 32 + threads - 1) / threads;
  launch_pdl(fingerprint_kernel<VB, K, NB, MASK, HEAD>, dim3((unsigned)blocks), dim3(threads), 0, stream,
             tokens, n, stride, lens, seed, fp_out, rpw, err);
  count_launches(1);
  return cuda_fail(cudaGetLastError(), "fingerprint launch");
}

template <int VB, int K, int NB>
hs_status launch_chunks(const int32_t* tokens, int64_t n, int32_t stride, const int32_t* lens,
                        uint64_t seed, uint64_t* fp_out, int64_t sms, cudaStream_t stream) {
  // Resident warps per SM at this kernel's register count (queried once per
  // device; the kernel uses no shared memory).
  static std::atomic<int> per_device[kMaxDeviceOrdinals];
  const int dev = device_ordinal();
  int warps_per_sm = dev >= 0 ? per_device[dev].load() : 0;
  if (warps_per_sm == 0) {
    int blocks = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &blocks, fingerprint_chunks_kernel<VB, K, NB>, 256, 0);
    if (e != cudaSuccess) return cuda_fail(e, "fingerprint occupancy");
    warps_per_sm = blocks > 0 ? blocks * 8 : 8;
    if (dev >= 0) per_device[dev].store(warps_per_sm);
  }
  const int64_t warps_target = sms * warps_per_sm;
  int64_t rpw = (n + warps_target - 1) / warps_target;
  if (rpw < 32) rpw = 32;
  const int64_t warps = (n + rpw - 1) / rpw;
  // Few warps: one-warp blocks, so they spread over all SMs.
  const int threads = warps >= sms * 8 ? 256 : 32;
  const int64_t blocks = (warps * 32 + threads - 1) / threads;
  launch_pdl(fingerprint_chunks_kernel<VB, K, NB>, dim3((unsigned)blocks), dim3(threads), 0, stream,
             tokens, n, stride, lens, seed, fp_out, rpw);
  count_launches(1);
  return HS_OK;
}

}  // namespace

// The full 32-token chunks only (the first pass of hs_merge_rows, whose
// second pass finishes the tails; nothing where no row can have one): 16-byte
// aligned rows with stride % 4 == 0.
hs_status launch_fingerprint_chunks(const int32_t* tokens, int64_t n, int32_t stride,
                                    const int32_t* lens, uint64_t seed, uint64_t* fp_out,
                                    cudaStream_t stream) {
  if (stride < kChunk) return HS_OK;
  const bool vec32 = (reinterpret_cast<uintptr_t>(tokens) & 31u) == 0 && stride % 8 == 0;
  const int64_t sms = num_sms();
  return vec32 ? launch_chunks<32, 4, 2>(tokens, n, stride, lens, seed, fp_out, sms, stream)
               : launch_chunks<16, 8, 2>(tokens, n, stride, lens, seed, fp_out, sms, stream);
}

// Aligned rows in a pass over full chunks and one over the rests, or in one that
// masks: masks cost every step of a chain, the second pass a launch and its own
// reads.  us, one pass / two: lengths up to 1024, 12,000 rows 27.7 / 26.0, 40,000
// 57.1 / 49.3, 200,000 117 / 108; up to 512, 12,000 15.4 / 16.0, 40,000 30.1 / 28.0,
// 400,000 105 / 101; up to 256, 65,536 16.9 / 19.5, 100,000 23.6 / 22.2, 400,000 58.5 /
// 58.2; up to 128, 100,000 14.8 / 16.1, 700,000 53.8 / 59.8; all of 36 tokens, 40,000
// 6.9 / 8.6, 400,000 26.8 / 22.4, 700,000 38.3 / 36.8; all of 200, 6500 8.2 / 8.3, 40,000
// 15.8 / 13.3, 400,000 75.9 / 72.8, 700,000 114 / 118.
bool two_passes(int64_t n, int32_t stride, bool lens) {
  if (stride >= 640) return true;
  if (n > 80000) return lens ? stride >= 256 && n <= 1000 * (int64_t)stride : n < 600000;
  return n >= 16384 && stride >= (lens ? 512 : 200);
}

// 32-byte loads where every row starts on such a boundary, else 16-byte loads.
hs_status launch_fingerprint(const int32_t* tokens, int64_t n, int32_t stride,
                             const int32_t* lens, uint64_t seed, uint64_t* fp_out,
                             cudaStream_t stream) {
  unsigned* err = device_error_word();
  if (!err) return fail(HS_ERR_CUDA, "could not resolve the device error word");
  const uintptr_t base = reinterpret_cast<uintptr_t>(tokens);
  const bool vec16 = (base & 15u) == 0 && stride % 4 == 0;
  auto rests = [&] {
    auto* kernel = vec16 ? (stride <= 8    ? fingerprint_rests_kernel<8, true>
                            : stride <= 16 ? fingerprint_rests_kernel<16, true>
                            : stride <= 24 ? fingerprint_rests_kernel<24, true>
                                           : fingerprint_rests_kernel<kChunk, true>)
                         : (stride <= 8    ? fingerprint_rests_kernel<8, false>
                            : stride <= 16 ? fingerprint_rests_kernel<16, false>
                            : stride <= 24 ? fingerprint_rests_kernel<24, false>
                                           : fingerprint_rests_kernel<kChunk, false>);
    launch_pdl(kernel,
               dim3((unsigned)std::min<int64_t>((n + kFpThreads - 1) / kFpThreads, num_sms() * 64)),
               dim3(kFpThreads), 0, stream, tokens, n, stride, lens, seed, fp_out, err);
    count_launches(1);
    return cuda_fail(cudaGetLastError(), "fingerprint launch");
  };
  // Rows of fewer tokens than a chunk have a thread each: 1,000,000 rows of up to 4
  // tokens 7 us (20 in the lanes' chunks), of 8 8.7 to 9.4 (19 to 26), of 16 15 to 21
  // (24 to 32), of 28 31 to 41 (33 to 40).  Few rows of more than 16 have a warp
  // (100 rows of 31: 3.1 us, 3.8 with a thread).
  if (stride <= 16) return rests();
  // A warp per row takes 0.7 ns per row and 256 tokens at full size; a lane per
  // row the chain of the longest row while that many lanes fit the GPU, 17 to 23 ns
  // per token (50 where rows are not aligned).  us, warp / lane: aligned, 4096 rows
  // of 256 tokens 4.9 / 6.6, 8192 7.4 / 6.6, 2048 of 384 (octet-wise) 5.1 / 14.4; on
  // any word, all of 333 10,000 rows 15.9 / 18.9, 12,288 19.0 / 18.9, 16,384 24.0 /
  // 18.9, of 128 10,000 9.0 / 9.9, 12,288 10.6 / 9.8, of 1024 16,384 44.9 / 51.0, 20,011
  // 54.2 / 54.0.
  const int64_t work = n * (((int64_t)stride + 255) / 256);
  if (n < (1 << 20) && work <= (vec16 ? 24 : 72) * (int64_t)stride) {
    const int64_t blocks = (n + 3) / 4;
    launch_pdl(vec16 ? fingerprint_warp_kernel<true> : fingerprint_warp_kernel<false>,
               dim3((unsigned)std::min<int64_t>(blocks, num_sms() * 64)), dim3(128), 0, stream,
               tokens, n, stride, lens, seed, fp_out, err);
    count_launches(1);
    return cuda_fail(cudaGetLastError(), "fingerprint launch");
  }
  if (stride < kChunk) return rests();
  const bool whole = !lens && stride % kChunk == 0 && stride > 0;   // no masks needed
  if (vec16 && !whole && two_passes(n, stride, lens != nullptr)) {
    const hs_status st = launch_fingerprint_chunks(tokens, n, stride, lens, seed, fp_out, stream);
    return st == HS_OK ? rests() : st;
  }
  if ((base & 31u) == 0 && stride % 8 == 0)
    return whole ? launch_rows<32, 4, 2, false, false>(tokens, n, stride, lens, seed, fp_out, err, stream)
                 : launch_rows<32, 4, 2, true, false>(tokens, n, stride, lens, seed, fp_out, err, stream);
  if (vec16)
    return launch_rows<16, 8, 2, true, false>(tokens, n, stride, lens, seed, fp_out, err, stream);
  return launch_rows<16, 8, 2, true, true>(tokens, n, stride, lens, seed, fp_out, err, stream);
}

}  // namespace hs
