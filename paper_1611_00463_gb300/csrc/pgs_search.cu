// Lookups on the sorted output (Section IV-C: the library lets its users
// binary-search the sorted data and find every entry's previous processor and
// index).  C ABI: pgs_search, pgs_provenance (declared in include/pgs.h).
#include "pgs_host.cuh"

namespace pgs {
namespace {

constexpr int kSearchNT = 256;
constexpr int kSearchOcc = 6;                         // CTAs of an indexed search per SM (40 registers a thread)
constexpr uint64_t kSearchCtas = 152 * kSearchOcc;

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
// Measured, 2^24 queries in 2^26 sorted keys, with buckets, against index and
// block bisected a key at a time: u64 uniform 2.03 -> 0.98 ms, normal/lognormal
// 1.99 -> 1.15, u32 uniform 1.29 -> 0.74; Zipf keys, where most blocks hold one
// value, u64 0.94 -> 0.90, f32 0.74 -> 0.63; 2^22 queries in 2^20 keys u64 232 ->
// 150 us, Zipf f32 124 -> 115.  Without the look at the index u64 takes 1.18, with
// two looks 0.96 (but Zipf 0.95 and u32 0.81), with 128-byte lines 1.62; a 16 KB
// top gains 1 %; interpolation by each lane for itself costs Zipf f32 1.29.  Eight
// lanes sharing 128-byte nodes of a 16-ary tree move as few bytes but spend 3.8 ms
// in instructions.  What is left: 161 bytes of DRAM lines a query and the latency
// of four dependent looks.
constexpr uint64_t kStride = 64;
constexpr int kTopBytes = 8192, kLineBytes = 64;
// Fewer queries than this bisect the array itself: the index costs a DRAM sector
// for every kStride keys, in every call.  1024 queries in 2^26 (2^28) u64 keys
// take 23 (25) us plainly and 47 (117) with the index, 2^18 queries 81 (115) and
// 64 (142), 2^20 queries 277 (398) and 108 (202); in 2^20 and 2^22 keys 2^18
// queries take 23 and 27 us plainly, 27 and 31 with it, 2^19 44 and 50, 36 and 40.
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

template <typename K, bool RIGHT>
__global__ void __launch_bounds__(kSearchNT, kSearchOcc)
k_search_indexed(const K* __restrict__ keys, uint64_t n, const K* __restrict__ index, uint32_t I, int top_log,
                 const K* __restrict__ queries, uint64_t m, int f32, const uint64_t* __restrict__ e, uint32_t P,
                 uint64_t* __restrict__ pos_out, uint32_t* __restrict__ bucket_out) {
  constexpr int F = kLineBytes / sizeof(K), LINES = (int)(kStride / F), G = 32 / sizeof(K);
  // The top in heap order (the children of node x are 2 x and 2 x + 1): a sorted
  // array's power-of-two strides would put a whole level into one bank.
  __shared__ K s_top[kTopBytes / sizeof(K)];
  extern __shared__ uint64_t s_e[];
  const uint32_t ntop = ((I - 1) >> top_log) + 1;
  const int depth = 32 - __clz(max(ntop, 2u) - 1);      // entries 1 .. 2^depth - 1 cover 1 .. ntop - 1
  for (uint32_t x = 1 + threadIdx.x; x < 1u << depth; x += kSearchNT) {
    const int level = 31 - __clz(x);
    const uint32_t entry = (2 * (x - (1u << level)) + 1) << (depth - 1 - level);
    s_top[x] = entry < ntop ? index[(uint64_t)entry << top_log] : ~K(0);
  }
  const K first_entry = index[0], last_entry = index[I - 1];
  const bool near = bucket_out && P < kSearchBounds;
  if (near)
    for (uint32_t i = threadIdx.x; i <= P; i += kSearchNT) s_e[i] = e[i];
  __syncthreads();
  const bool aligned = (reinterpret_cast<uintptr_t>(keys) & 15) == 0;
  const bool index_aligned = (reinterpret_cast<uintptr_t>(index) & 15) == 0;
  // All lanes of a warp stay in the loop together (those past the last query
  // repeat it), so that every vote is one of the whole warp.
  constexpr uint32_t WARP = 0xFFFFFFFFu;
  for (uint64_t i = blockIdx.x * (uint64_t)kSearchNT + threadIdx.x; i - (threadIdx.x & 31) < m;
       i += (uint64_t)gridDim.x * kSearchNT) {
    const K v = to_order<K>(queries[umin(i, m - 1)], f32);
    auto before = [&](K k) { return RIGHT ? !(v < k) : k < v; };
    // The block c is the number of index entries 1, 2, ... before v: the answer
    // lies among the keys of block c or right after them.  lo and hi: the nearest
    // entries on either side, between which the position is interpolated.
    uint32_t x = 1;
    for (int l = 0; l < depth; ++l) x = 2 * x + before(s_top[x]);
    const uint32_t cell = min(x - (1u << depth), ntop - 1);  // pads are before the greatest key's upper bound
    auto top_entry = [&](uint32_t j) {
      const int t = __ffs(j) - 1;
      return s_top[(1u << (depth - 1 - t)) + (j >> (t + 1))];
    };
    K lo = cell > 0 ? top_entry(cell) : first_entry, hi = cell + 1 < ntop ? top_entry(cell + 1) : last_entry;
    auto between = [&] { return lo < v && v < hi; };
    // Entry c (0: none) is before v and entry c_end (I: none) is not.
    uint32_t c = cell << top_log, c_end = I - c > 1u << top_log ? c + (1u << top_log) : I;
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
    uint64_t pos;
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
      const K* block = keys + c * kStride;
      uint32_t a = 0, z = (uint32_t)umin(kStride, n - c * kStride);
      while (a < z) {
        const uint32_t mid = (a + z) >> 1;
        if (before(to_order<K>(__ldg(block + mid), f32))) a = mid + 1;
        else z = mid;
      }
      pos = c * kStride + a;
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
    const unsigned grid = (unsigned)std::min<uint64_t>(ceil_div(m, kSearchNT), kSearchCtas);
    // Dynamic shared memory: the bucket bounds, where they are looked up and fit.
    const size_t smem = bucket && P < kSearchBounds ? (P + 1) * sizeof(uint64_t) : 0;
    if (side)
      k_search_indexed<K, true><<<grid, kSearchNT, smem, st>>>(keys, n, index, (uint32_t)I, top_log, q, m, f32, e, P,
                                                               pos, bucket);
    else
      k_search_indexed<K, false><<<grid, kSearchNT, smem, st>>>(keys, n, index, (uint32_t)I, top_log, q, m, f32, e, P,
                                                               pos, bucket);
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
