// Lookups on the sorted output (Section IV-C: the library lets its users
// binary-search the sorted data and find every entry's previous processor and
// index).  C ABI: pgs_search, pgs_provenance (declared in include/pgs.h).
#include "pgs_host.cuh"

namespace pgs {
namespace {

constexpr int kSearchNT = 256;
// Threads of an indexed search's CTA (26 registers each, 38 with interpolation),
// CTAs per SM, and the heap nodes that tell whether keys repeat.
constexpr int index_threads(bool step) { return step ? 1024 : 768; }
constexpr int kSearchMB = 2;
constexpr uint64_t kSearchCtas = 152 * kSearchMB;
constexpr uint32_t kSpread = 512;

// Last b in [0, P) with e[b] <= pos, for pos < e[P] (the bucket holding pos).
__device__ __forceinline__ uint32_t bucket_holding(const uint64_t* e, uint32_t P, uint64_t pos) {
  if (pos >= e[P]) return P;
  uint32_t a = 0, z = P;                                // e[a] <= pos < e[z]
  while (z - a > 1) {
    const uint32_t mid = (a + z) >> 1;
    if (e[mid] <= pos) a = mid; else z = mid;
  }
  return a;
}

// One thread per query: lower (RIGHT = false) or upper bound of the query in
// the sorted keys, by key order (float32 by totalOrder of its bits).
template <typename K, bool RIGHT>
__global__ void __launch_bounds__(kSearchNT)
k_search(const K* __restrict__ keys, uint64_t n, const K* __restrict__ queries, uint64_t m, int f32,
         const uint64_t* __restrict__ e, uint32_t P, uint64_t* __restrict__ pos_out, uint32_t* __restrict__ bucket_out) {
  const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (i >= m) return;
  const K v = to_order<K>(queries[i], f32);
  uint64_t lo = 0, hi = n;
  while (lo < hi) {
    const uint64_t mid = lo + ((hi - lo) >> 1);
    const K k = to_order<K>(__ldg(keys + mid), f32);
    if (RIGHT ? !(v < k) : (k < v)) lo = mid + 1; else hi = mid;
  }
  pos_out[i] = lo;
  if (bucket_out) bucket_out[i] = bucket_holding(e, P, lo);
}

// Indexed search.  Random DRAM accesses bound it: a plain bisection of a large
// array misses in L2 on most of its lower levels.  The index is a compact copy of
// every kStride-th key (1/64 of the array, L2-resident); each CTA keeps every
// 2^top_log-th of its entries in shared memory, which take the top levels of the
// bisection.  Between two of those, interpolation picks one 32-byte group of the
// index to look at before bisection goes on, and inside the block of kStride keys
// the 64-byte line to read first, then the one next to it, then bisection.  A warp
// interpolates only if all its queries lie strictly between the entries on either
// side: among equal keys the values say nothing of the position.  Interpolation
// only chooses where to look; every bound is a comparison of keys, so any order of
// keys ends, in range.
// Two cases bisect index and block a key at a time (STEP, and `step` found by each
// CTA): arrays of up to kStepBytes, whose lines L2 and L1 hold, so that a look
// saves no more than its arithmetic costs, and keys of which more than a quarter of
// the spread top entries equal their neighbour, where looks miss.  CTAs are large,
// so that few copies of the top take room from L1.
// Measured, against index and block bisected from the start (us; 256-thread CTAs
// that always interpolate, 8 KB tops, in brackets), with 17 to 64 buckets.
// 2^24 queries in 2^26 keys: u64 uniform 1972 -> 963 (988), normal/lognormal 1963 ->
// 1088 (1152), Zipf 902 -> 676 (608), u32 uniform 1230 -> 627 (661), f32 Zipf 703 ->
// 480 (497).  2^22 queries: in 190,000 keys u64 uniform 127 -> 115 (126), Zipf 90 ->
// 84 (112), u32 uniform 107 -> 87 (127), f32 Zipf 87 -> 64 (104); in 1,100,003 keys
// 160 -> 138 (140), 100 -> 108 (127), 135 -> 108 (137), 96 -> 73 (118); in 12,000,017
// keys 228 -> 163 (167), 127 -> 143 (144), 198 -> 147 (159), 108 -> 100 (117).  What
// is still slower than at first: u64 queries that are mostly equal and not among the
// keys, from 10^6 keys on where their number is no power of two (by 5 to 16 %; where
// it is one, 164 -> 98 in 2^20).  The line of kStepBytes: u64 uniform keys 122 by
// steps, 129 with looks at 400,003, 138 and 136 at 2^20, 149 and 137 at 1,100,003; u32
// 106 and 122 at 2^20, 128 and 129 at 3*10^6.  For 2^26 keys: without the look at the
// index u64 takes a fifth more, with 128-byte lines half as much again; eight lanes
// sharing 128-byte nodes of a 16-ary tree move as few bytes but spend 3.8 ms in
// instructions.  What is left: 181 bytes of DRAM lines a query and the latency of
// four dependent looks.
constexpr uint64_t kStride = 64;
constexpr int kTopBytes = 16384, kLineBytes = 64;
constexpr uint64_t kStepBytes = 8 << 20;
// Fewer queries than this bisect the array itself: the index costs a DRAM sector
// for every kStride keys, in every call.  Plainly and with it, us: 2^18 queries in
// 2^20, 2^22 u64 keys 20 and 22, 22 and 26, 393216 queries 39 and 26, 43 and 29; in
// 2^24 keys 196608 queries 21 and 22, 2^18 24 and 28, 393216 51 and 30; in 2^26 keys
// 131072 44 and 46, 196608 63 and 48; in 2^28 keys 1024 queries 12 and 105, 196608
// 92 and 116, 2^18 116 and 131, 393216 198 and 139.
constexpr uint64_t kIndexQueries = 3 << 17, kIndexQueriesLarge = 3 << 16, kIndexLarge = 1 << 24;
constexpr uint32_t kSearchBounds = 1024;             // bucket bounds kept in shared memory

template <typename K>
__global__ void __launch_bounds__(kSearchNT)
k_search_index(const K* __restrict__ keys, uint64_t n, int f32, K* __restrict__ index, uint64_t I) {
  const uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (j < I) index[j] = to_order<K>(keys[j * kStride], f32);
}

// How many of a line's keys that lie before `end` pass the test, which holds on
// a prefix of them; all loads in flight together.
template <typename K, typename Test>
__device__ __forceinline__ uint32_t line_prefix(const K* p, const K* end, bool aligned, const Test& test) {
  constexpr int F = kLineBytes / sizeof(K), E = 16 / sizeof(K);
  uint32_t c = 0;
  if (aligned && p + F <= end) {
    union { uint4 v[kLineBytes / 16]; K k[F]; } u;
#pragma unroll
    for (int i = 0; i < F / E; ++i) u.v[i] = __ldg(reinterpret_cast<const uint4*>(p) + i);
#pragma unroll
    for (int i = 0; i < F; ++i) c += test(u.k[i]);
  } else {
    for (int i = 0; i < F; ++i) c += p + i < end && test(__ldg(p + i));
  }
  return c;
}

template <typename K, bool RIGHT, bool STEP>
__global__ void __launch_bounds__(index_threads(STEP), kSearchMB)
k_search_indexed(const K* __restrict__ keys, uint64_t n, const K* __restrict__ index, uint32_t I, int top_log,
                 const K* __restrict__ queries, uint64_t m, int f32, const uint64_t* __restrict__ e, uint32_t P,
                 uint64_t* __restrict__ pos_out, uint32_t* __restrict__ bucket_out) {
  constexpr int NT = index_threads(STEP), F = kLineBytes / sizeof(K), LINES = (int)(kStride / F), G = 32 / sizeof(K);
  // The top in heap order (the children of node x are 2 x and 2 x + 1): a sorted
  // array's power-of-two strides would put a whole level into one bank.
  __shared__ K s_top[kTopBytes / sizeof(K)];
  extern __shared__ uint64_t s_e[];
  const uint32_t ntop = ((I - 1) >> top_log) + 1;
  const int depth = 32 - __clz(max(ntop, 2u) - 1);      // entries 1 .. 2^depth - 1 cover 1 .. ntop - 1
  bool same = false;                                    // nodes 1 .. kSpread - 1: equal to the entry before
  for (uint32_t x = 1 + threadIdx.x; x < 1u << depth; x += NT) {
    const int level = 31 - __clz(x);
    const uint32_t entry = (2 * (x - (1u << level)) + 1) << (depth - 1 - level);
    s_top[x] = entry < ntop ? index[(uint64_t)entry << top_log] : ~K(0);
    if (!STEP && x < kSpread) same = entry < ntop && s_top[x] == index[(uint64_t)(entry - 1) << top_log];
  }
  const bool near = bucket_out && P < kSearchBounds;
  if (near)
    for (uint32_t i = threadIdx.x; i <= P; i += NT) s_e[i] = e[i];
  const bool step = __syncthreads_count(same) > (int)(kSpread * ntop >> depth) / 4 || STEP;
  const bool aligned = (reinterpret_cast<uintptr_t>(keys) & 15) == 0;
  const bool index_aligned = (reinterpret_cast<uintptr_t>(index) & 15) == 0;
  // All lanes of a warp stay in the loop together (those past the last query
  // repeat it), so that every vote is one of the whole warp.
  constexpr uint32_t WARP = 0xFFFFFFFFu;
  for (uint64_t i = blockIdx.x * (uint64_t)NT + threadIdx.x; i - (threadIdx.x & 31) < m; i += (uint64_t)gridDim.x * NT) {
    const K v = to_order<K>(queries[umin(i, m - 1)], f32);
    auto before = [&](K k) { return RIGHT ? !(v < k) : k < v; };
    // The block c is the number of index entries 1, 2, ... before v: the answer
    // lies among the keys of block c or right after them.
    uint32_t x = 1;
    for (int l = 0; l < depth; ++l) x = 2 * x + before(s_top[x]);
    const uint32_t cell = min(x - (1u << depth), ntop - 1);  // pads are before the greatest key's upper bound
    // Entry c (0: none) is before v and entry c_end (I: none) is not.
    uint32_t c = cell << top_log, c_end = I - c > 1u << top_log ? c + (1u << top_log) : I;
    auto in_block = [&] {
      const K* block = keys + c * kStride;
      uint32_t a = 0, z = (uint32_t)umin(kStride, n - c * kStride);
      while (a < z) {
        const uint32_t mid = (a + z) >> 1;
        if (before(to_order<K>(__ldg(block + mid), f32))) a = mid + 1;
        else z = mid;
      }
      return c * kStride + a;
    };
    uint64_t pos;
    if (step) {
      while (c + 1 < c_end) {
        const uint32_t g = c + (c_end - c) / 2;
        if (before(__ldg(index + g))) c = g;
        else c_end = g;
      }
      pos = in_block();
    } else {
      // lo and hi: the nearest entries on either side, between which the position
      // is interpolated.
      auto top_entry = [&](uint32_t j) {
        const int t = __ffs(j) - 1;
        return s_top[(1u << (depth - 1 - t)) + (j >> (t + 1))];
      };
      K lo = cell > 0 ? top_entry(cell) : index[0], hi = cell + 1 < ntop ? top_entry(cell + 1) : index[I - 1];
      auto between = [&] { return lo < v && v < hi; };
      bool look = __all_sync(WARP, index_aligned && between()), smooth = true;
      while (c + 1 < c_end) {
        uint32_t g = c + (c_end - c) / 2;
        if (look) {
          look = false;
          g = c + min((uint32_t)(__fdividef((float)(v - lo), (float)(hi - lo)) * (float)(c_end - c)), c_end - c - 1);
          g = g / G * G;
          if (I - g >= G) {
            union { uint4 v[2]; K k[G]; } u;
            u.v[0] = __ldg(reinterpret_cast<const uint4*>(index + g));
            u.v[1] = __ldg(reinterpret_cast<const uint4*>(index + g) + 1);
            int below = 0;
#pragma unroll
            for (int j = 0; j < G; ++j) below += before(u.k[j]);
#pragma unroll
            for (int j = 0; j < G; ++j) {
              if (j + 1 == below && g + j > c) c = g + j, lo = u.k[j];
              if (j == below && g + j < c_end) c_end = g + j, hi = u.k[j];
            }
            smooth = c + 1 >= c_end;
            continue;
          }
          g = c + (c_end - c) / 2;
        }
        const K k = __ldg(index + g);
        if (before(k)) lo = k, c = g;
        else hi = k, c_end = g;
      }
      // Where few of the warp's looks at the index hit, the keys are not smooth.
      const bool inside = __all_sync(WARP, between()), hit = __popc(__ballot_sync(WARP, smooth)) >= 8;
      if (inside && hit) {
        int first = 0, last = LINES - 1;
        int line = min((int)(__fdividef((float)(v - lo), (float)(hi - lo)) * LINES), last);
        for (int look = 0;; ++look) {
          const uint64_t at = c * kStride + line * F;
          const uint32_t below =
              at < n ? line_prefix<K>(keys + at, keys + n, aligned, [&](K k) { return before(to_order<K>(k, f32)); }) : 0;
          pos = umin(at + below, n);
          if (below == 0 && line > first) last = line - 1, line = look ? (first + last) >> 1 : last;
          else if (below == (uint32_t)F && line < last) first = line + 1, line = look ? (first + last) >> 1 : first;
          else break;
        }
      } else {
        pos = in_block();
      }
    }
    if (i < m) {
      pos_out[i] = pos;
      if (bucket_out) bucket_out[i] = near ? bucket_holding(s_e, P, pos) : bucket_holding(e, P, pos);
    }
  }
}

// Run r of the floor split holds input positions [floor(r n / P), floor((r+1) n / P)).
__global__ void __launch_bounds__(kSearchNT)
k_provenance(const uint32_t* __restrict__ vals, uint64_t m, uint64_t n, uint64_t P, uint32_t* __restrict__ run_out,
             uint64_t* __restrict__ index_out) {
  const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (i >= m) return;
  const uint64_t v = vals[i];
  uint64_t r;
  if (v >= n) {
    r = P;                                              // not an input position
  } else {
    // Largest r with floor(r n / P) <= v is ceil((v + 1) P / n) - 1; then check.
    r = (uint64_t)(((unsigned __int128)(v + 1) * P + n - 1) / n) - 1;
    if (r >= P) r = P - 1;
    while (r > 0 && run_start(r, n, P) > v) --r;
    while (r + 1 < P && run_start(r + 1, n, P) <= v) ++r;
  }
  if (run_out) run_out[i] = (uint32_t)r;
  if (index_out) index_out[i] = v - (r < P ? run_start(r, n, P) : n);
}

bool on_device(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Bytes of workspace the indexed search uses for n keys of w bytes (0: none).
inline size_t search_index_bytes(uint64_t n, int w) {
  return n >= kStride * 1024 ? (size_t)ceil_div(n, kStride) * w : 0;
}

template <typename K>
int launch_search(const K* keys, uint64_t n, const K* q, uint64_t m, int side, int f32, const uint64_t* e,
                  uint32_t P, uint64_t* pos, uint32_t* bucket, void* ws, size_t ws_bytes, cudaStream_t st) {
  const size_t need = search_index_bytes(n, sizeof(K));
  if (need && ws && ws_bytes >= need && m >= (n >= kIndexLarge ? kIndexQueriesLarge : kIndexQueries) && n < kStride << 31) {
    K* index = static_cast<K*>(ws);
    const uint64_t I = ceil_div(n, kStride);
    int top_log = 0;
    while (ceil_div(I, 1ull << top_log) * sizeof(K) > kTopBytes) ++top_log;
    k_search_index<K><<<(unsigned)ceil_div(I, kSearchNT), kSearchNT, 0, st>>>(keys, n, f32, index, I);
    // Dynamic shared memory: the bucket bounds, where they are looked up and fit.
    const size_t smem = bucket && P < kSearchBounds ? (P + 1) * sizeof(uint64_t) : 0;
    auto run = [&](auto* kernel, int threads) {
      kernel<<<(unsigned)std::min<uint64_t>(ceil_div(m, threads), kSearchCtas), threads, smem, st>>>(
          keys, n, index, (uint32_t)I, top_log, q, m, f32, e, P, pos, bucket);
    };
    if (n * sizeof(K) <= kStepBytes)
      run(side ? k_search_indexed<K, true, true> : k_search_indexed<K, false, true>, index_threads(true));
    else
      run(side ? k_search_indexed<K, true, false> : k_search_indexed<K, false, false>, index_threads(false));
    PGS_CUDA(cudaGetLastError());
    return PGS_OK;
  }
  const unsigned grid = (unsigned)ceil_div(m, kSearchNT);
  if (side)
    k_search<K, true><<<grid, kSearchNT, 0, st>>>(keys, n, q, m, f32, e, P, pos, bucket);
  else
    k_search<K, false><<<grid, kSearchNT, 0, st>>>(keys, n, q, m, f32, e, P, pos, bucket);
  PGS_CUDA(cudaGetLastError());
  return PGS_OK;
}

}  // namespace
}  // namespace pgs

using namespace pgs;

extern "C" {

int pgs_search(const void* keys, uint64_t n, const void* queries, uint64_t m, int side,
               const uint64_t* bucket_bounds, uint32_t P, uint64_t* pos_out, uint32_t* bucket_out, void* stream,
               const pgs_config* cfg) {
  Options o;
  int rc = read_options(cfg, &o);
  if (rc) return rc;
  if (side != 0 && side != 1) return PGS_ERR_INVALID;
  if ((bucket_bounds == nullptr) != (bucket_out == nullptr)) return PGS_ERR_INVALID;
  if (bucket_bounds && P == 0) return PGS_ERR_INVALID;
  if (m == 0) return PGS_OK;
  if (!queries || !pos_out || (n > 0 && !keys)) return PGS_ERR_INVALID;
  if (n >= (1ull << 40) || m >= (1ull << 40)) return PGS_ERR_UNSUPPORTED;
  if (!on_device(queries) || !on_device(pos_out) || (n > 0 && !on_device(keys)) ||
      (bucket_bounds && (!on_device(bucket_bounds) || !on_device(bucket_out))))
    return PGS_ERR_INVALID;
  if (ceil_div(m, kSearchNT) > 0x7FFFFFFFull) return PGS_ERR_UNSUPPORTED;
  DeviceGuard dg;
  PGS_TRY(dg.use_device_of(pos_out));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int f32 = o.dtype == PGS_F32;
  if (o.workspace && (!on_device(o.workspace) || (reinterpret_cast<uintptr_t>(o.workspace) % kAlign) != 0))
    return PGS_ERR_WORKSPACE;
  if (o.dtype == PGS_U64)
    return launch_search<uint64_t>(static_cast<const uint64_t*>(keys), n, static_cast<const uint64_t*>(queries), m,
                                   side, 0, bucket_bounds, P, pos_out, bucket_out, o.workspace, o.workspace_bytes,
                                   st);
  return launch_search<uint32_t>(static_cast<const uint32_t*>(keys), n, static_cast<const uint32_t*>(queries), m,
                                 side, f32, bucket_bounds, P, pos_out, bucket_out, o.workspace, o.workspace_bytes,
                                 st);
}

size_t pgs_search_workspace_bytes(uint64_t n, const pgs_config* cfg) {
  Options o;
  if (read_options(cfg, &o) != PGS_OK) return 0;
  return search_index_bytes(n, key_bytes(o.dtype));
}

int pgs_provenance(const uint32_t* vals, uint64_t m, uint64_t n, uint32_t P, uint32_t* run_out,
                   uint64_t* index_out, void* stream) {
  if (P == 0) return PGS_ERR_INVALID;
  if (m == 0) return PGS_OK;
  if (!vals || (!run_out && !index_out)) return PGS_ERR_INVALID;
  if (n >= (1ull << 40) || m >= (1ull << 40)) return PGS_ERR_UNSUPPORTED;
  if (!on_device(vals) || (run_out && !on_device(run_out)) || (index_out && !on_device(index_out)))
    return PGS_ERR_INVALID;
  if (ceil_div(m, kSearchNT) > 0x7FFFFFFFull) return PGS_ERR_UNSUPPORTED;
  DeviceGuard dg;
  PGS_TRY(dg.use_device_of(vals));
  const uint64_t Peff = n == 0 ? 1 : std::max<uint64_t>(1, std::min<uint64_t>(P, n));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  k_provenance<<<(unsigned)ceil_div(m, kSearchNT), kSearchNT, 0, st>>>(vals, m, n, Peff, run_out, index_out);
  PGS_CUDA(cudaGetLastError());
  return PGS_OK;
}

}  // extern "C"
