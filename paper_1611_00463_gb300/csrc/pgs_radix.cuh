// Device code of the radix form of the sort: the stable order of Section IV's
// six steps by least-significant-digit passes over run-tagged keys, and the
// method's splitters, bucket bounds and cut matrix read off the sorted order.
//
// Why it gives the six steps' results.  Steps 1, 5 and 6 (local sorts, the
// exchange, the balanced merge) end in the stable sort of the whole input, and
// that order is unique, so any stable sort reaches it.  Every key carries its
// run (the paper's "previous processor") through the passes.  In the sorted
// order the keys of run r appear in run r's own sorted order, so a key's
// position in its sorted run is the number of keys of run r before it, and
// steps 2-4 need no sorted runs:
//  - a key is a regular sample iff that position is one of the sample positions;
//  - the samples in sorted order are the samples in position order (ties by run
//    and position are already in place), so splitter t_b is the sample number
//    floor(b S / P) - 1 along the output;
//  - L_b and L_b + G_b are the bounds of t_b in the output, e_b follows by the
//    investigator's rule, and cut[r][b] is the number of keys of run r among
//    the first e_b outputs.
// (The LOCAL investigator's order is not the stable sort, and a learned model
// is evaluated on sorted runs: those sorts run the merge pipeline.)
#pragma once

#include <type_traits>

#include "pgs_kernels.cuh"

namespace pgs {

constexpr int kRadixBits = 8;
constexpr int kRadixBins = 1 << kRadixBits;
template <typename K> constexpr int radix_digits() { return (int)sizeof(K); }   // one pass per byte

// Threads, keys per thread and CTAs per SM of a pass's tile.  Larger tiles write
// longer runs of each digit, more CTAs overlap their phases; shared memory and
// registers trade one for the other.  Measured (ms per 2^27-key move, u64 + u32
// payload + tag / u32 + u32 payload + tag): 384 x 16 0.715 / 0.645, 384 x 20 (one
// CTA per SM for u64) 0.995 / 0.618, 384 x 12 0.817 / 0.741, 256 x 16 with 3 CTAs
// 0.848 / 0.678, 512 x 14 1.051 / 0.639, 448 x 16 1.038 / 0.647, 320 x 18 0.823 / 0.672.
#ifndef PGS_RADIX_NT8
#define PGS_RADIX_NT8 384
#define PGS_RADIX_VT8 16
#define PGS_RADIX_MB8 2
#define PGS_RADIX_NT4 384
#define PGS_RADIX_VT4 20
#define PGS_RADIX_MB4 2
#endif
template <int W> struct RadixShape;
template <> struct RadixShape<8> { static constexpr int NT = PGS_RADIX_NT8, VT = PGS_RADIX_VT8, MB = PGS_RADIX_MB8; };
template <> struct RadixShape<4> { static constexpr int NT = PGS_RADIX_NT4, VT = PGS_RADIX_VT4, MB = PGS_RADIX_MB4; };
constexpr uint32_t radix_tile(int w) {
  return w == 8 ? (uint32_t)(RadixShape<8>::NT * RadixShape<8>::VT) : (uint32_t)(RadixShape<4>::NT * RadixShape<4>::VT);
}

// A tile of a pass, and the chunk of tiles one counting CTA takes (batches; a
// single sort's are closed form).
struct RadixTile {
  uint64_t start;          // first key
  uint32_t cnt;            // keys
  uint32_t inst;           // instance
  uint64_t chunk;          // the tile's chunk
};
struct RadixChunk {
  uint64_t start;          // first key
  uint64_t tile;           // first tile
  uint32_t cnt;            // keys
  uint32_t inst;           // instance
};

// What travels with a key besides its payload, its tag.
//  Id8   the run (P <= 256) in the low byte and the next pass's digit in the
//        high byte, so that the next count reads two bytes a key, not the key;
//  Id16  the run;
//  Dig   the next pass's digit (nothing asked for depends on the runs, wide keys);
//  None  nothing (the same, narrow keys: the count reads the key).
struct Id8 { using Tag = uint16_t; static constexpr int bytes = 2; static constexpr bool run = true, digit = true; };
struct Id16 { using Tag = uint16_t; static constexpr int bytes = 2; static constexpr bool run = true, digit = false; };
struct Dig { using Tag = uint8_t; static constexpr int bytes = 1; static constexpr bool run = false, digit = true; };
struct None { using Tag = uint8_t; static constexpr int bytes = 0; static constexpr bool run = false, digit = false; };

// A pass's digit and run of a tag, and the tag for the next pass.
template <typename ID> __device__ __forceinline__ uint32_t tag_digit(uint32_t t) { return ID::run ? t >> 8 : t; }
template <typename ID> __device__ __forceinline__ uint32_t next_tag(uint32_t t, uint32_t digit) {
  if (!ID::digit) return t;
  return ID::run ? (t & 0xFF) | (digit << 8) : digit;
}

// One pass, a stable counting sort by one byte of the key: count every tile's
// digits, scan the counts, move.  The move reads and writes each key, payload
// and tag once, tile by tile in order, so that neighbouring tiles' writes to a
// digit's range meet in L2.  (A single kernel that finds each tile's place by
// look-back over its predecessors saves the count and loses more to waiting:
// at 22 tiles a microsecond the nearest tile that knows its prefix is some 50
// tiles back, 1.13 against 1.02 ms per 2^27-key u64 pass.)
template <typename K>
struct RadixPass {
  const K* ksrc;
  K* kdst;
  const uint32_t* vsrc;
  uint32_t* vdst;
  const void* tsrc;                // tags; NULL in the first pass (runs worked out from the position)
  void* tdst;
  uint32_t* cnt;                   // tiles x 256: the digits of the chunk's earlier tiles
  uint64_t* pre;                   // chunks x 256: a chunk's digits, then those of the instance's earlier chunks
  uint64_t* total;                 // instances x 256: digit totals
  const RadixTile* tiles;          // NULL: a single sort
  const RadixChunk* chunks;
  const uint64_t* koff;            // instances' first keys and partition counts (runs)
  const uint32_t* P;
  uint32_t* err;
  uint64_t n, wait_ns;
  uint32_t chunk_tiles;            // tiles of a single sort's chunk
  int byte, f32_in, f32_out;
  int last;                        // no next pass: tags are runs alone
};

// Byte `sel` of a key, for the pass's uniform byte number.
__device__ __forceinline__ uint32_t radix_digit(uint32_t k, uint32_t sel) { return __byte_perm(k, 0, 0x4440 | sel); }
__device__ __forceinline__ uint32_t radix_digit(uint64_t k, uint32_t sel) {
  const uint32_t w = sel & 4 ? (uint32_t)(k >> 32) : (uint32_t)k;
  return __byte_perm(w, 0, 0x4440 | (sel & 3));
}

// One CTA per chunk: each tile's row of counts, of the chunk's tiles before
// it, and the chunk's totals.  With tags that hold it, the digit comes from there.
constexpr int kCountNT = 512;

template <typename K, typename ID, bool TAGS>
__global__ void __launch_bounds__(kCountNT)
k_radix_count(RadixPass<K> a) {
  pdl_enter();
  constexpr uint32_t T = radix_tile((int)sizeof(K));
  __shared__ uint32_t s_cnt[kRadixBins];
  uint64_t start, tile;
  uint32_t left;
  if (a.chunks) {
    const RadixChunk c = a.chunks[blockIdx.x];
    start = c.start;
    tile = c.tile;
    left = c.cnt;
  } else {
    tile = (uint64_t)blockIdx.x * a.chunk_tiles;
    start = tile * T;
    left = (uint32_t)umin((uint64_t)a.chunk_tiles * T, a.n - start);
  }
  if (threadIdx.x < kRadixBins) s_cnt[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t sel = a.byte;
  auto digit = [&](uint64_t i) -> uint32_t {
    if (TAGS) return tag_digit<ID>(static_cast<const typename ID::Tag*>(a.tsrc)[i]);
    return radix_digit(to_order<K>(a.ksrc[i], a.f32_in), sel);
  };
  for (; left > 0; ++tile, start += T) {
    const uint32_t cnt = left < T ? left : T;
    left -= cnt;
    if (threadIdx.x < kRadixBins) a.cnt[tile * kRadixBins + threadIdx.x] = s_cnt[threadIdx.x];
    __syncthreads();
    if (cnt == T) {
      constexpr int U = (T + kCountNT - 1) / kCountNT;
      uint32_t d[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (u * kCountNT + threadIdx.x < T) d[u] = digit(start + u * kCountNT + threadIdx.x);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (u * kCountNT + threadIdx.x < T) atomicAdd(&s_cnt[d[u]], 1u);
    } else {
      for (uint32_t i = threadIdx.x; i < cnt; i += kCountNT) atomicAdd(&s_cnt[digit(start + i)], 1u);
    }
    __syncthreads();
  }
  if (threadIdx.x < kRadixBins) a.pre[(uint64_t)blockIdx.x * kRadixBins + threadIdx.x] = s_cnt[threadIdx.x];
}

// Exclusive prefixes of every digit's chunk totals, in place, and the digit
// totals, for a single sort of `rows` chunks: CTA = 8 digits x 128 parts of
// the rows (8 digits are one 64-byte piece of a row).
static __global__ void __launch_bounds__(1024)
k_radix_scan_wide(uint64_t* pre, uint64_t* total, uint64_t rows) {
  pdl_enter();
  constexpr int D = 8, PARTS = 1024 / D;
  __shared__ uint64_t s_sum[PARTS][D];
  const uint32_t x = threadIdx.x % D, part = threadIdx.x / D;
  const uint64_t per = (rows + PARTS - 1) / PARTS, lo = umin(part * per, rows), hi = umin(lo + per, rows);
  uint64_t* c = pre + blockIdx.x * D + x;
  uint64_t sum = 0;
#pragma unroll 8
  for (uint64_t r = lo; r < hi; ++r) sum += c[r * kRadixBins];
  s_sum[part][x] = sum;
  __syncthreads();
  // Thread (digit w) of warp w / 4 ... : an inclusive scan over the parts by one warp per digit.
  if (threadIdx.x < 32 * D) {
    const uint32_t d = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint64_t carry = 0;
#pragma unroll
    for (int k = 0; k < PARTS / 32; ++k) {
      const uint64_t v = s_sum[k * 32 + lane][d];
      uint64_t inc = v;
#pragma unroll
      for (int s = 1; s < 32; s <<= 1) {
        const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, inc, s);
        if (lane >= s) inc += y;
      }
      s_sum[k * 32 + lane][d] = carry + inc - v;
      carry += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
    if (lane == 0) total[blockIdx.x * D + d] = carry;
  }
  __syncthreads();
  uint64_t run = s_sum[part][x];
#pragma unroll 8
  for (uint64_t r = lo; r < hi; ++r) {
    const uint64_t v = c[r * kRadixBins];
    c[r * kRadixBins] = run;
    run += v;
  }
}

// The same for a batch: one CTA per instance, one thread per digit, over the
// instance's chunks [first[i], first[i + 1]).
static __global__ void __launch_bounds__(kRadixBins)
k_radix_scan_batch(uint64_t* pre, uint64_t* total, const uint64_t* __restrict__ first) {
  pdl_enter();
  uint64_t run = 0;
#pragma unroll 8
  for (uint64_t r = first[blockIdx.x]; r < first[blockIdx.x + 1]; ++r) {
    uint64_t* c = pre + r * kRadixBins + threadIdx.x;
    const uint64_t v = *c;
    *c = run;
    run += v;
  }
  total[(uint64_t)blockIdx.x * kRadixBins + threadIdx.x] = run;
}

// Lanes of the warp whose digit equals this lane's: one ballot per bit, kept
// or complemented by the lane's own bit (predicated, four instructions a bit;
// the C form of the same costs half again as many, match.any four times).
__device__ __forceinline__ uint32_t match_digit(uint32_t d) {
  uint32_t m = 0xFFFFFFFFu;
#pragma unroll
  for (int b = 0; b < kRadixBits; ++b) {
    uint32_t v;
    asm("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t"
        "and.b32 t, %1, %2;\n\tsetp.ne.u32 p, t, 0;\n\t"
        "vote.sync.ballot.b32 %0, p, 0xffffffff;\n\t@!p not.b32 %0, %0;\n\t}"
        : "=r"(v)
        : "r"(d), "r"(1u << b));
    m &= v;
  }
  return m;
}

// OFF: the type of output positions (uint32_t up to 2^32 keys).
template <typename K, bool V, typename ID, typename OFF>
struct RadixSmem {
  static constexpr int NT = RadixShape<(int)sizeof(K)>::NT, VT = RadixShape<(int)sizeof(K)>::VT;
  static constexpr int T = NT * VT, NW = NT / 32;
  // Keys, payloads and tags as they came (bulk copies widened to 16-byte
  // boundaries: up to 32 bytes more each), the source position of every tile
  // slot, the warps' digit counters, the digits' output positions.
  static constexpr size_t val = (size_t)T * sizeof(K) + 32;
  static constexpr size_t tag = val + (V ? (size_t)T * 4 + 32 : 0);
  static constexpr size_t perm = tag + (ID::bytes ? (size_t)T * ID::bytes + 32 : 0);
  static constexpr size_t warp = perm + (size_t)T * 2;
  static constexpr size_t base = warp + (size_t)NW * kRadixBins * 4;
  static constexpr size_t bar = base + kRadixBins * sizeof(OFF);
  static constexpr size_t bytes = bar + 16;
  static_assert(T <= 65536 && T % 16 == 0, "16-bit source positions, aligned copies");
  static_assert(warp % 16 == 0 && bar % 8 == 0, "aligned parts");
};

// Exclusive scan over 256 values by threads 0..255 (others pass); s_warp: 8 entries.
template <typename T>
__device__ __forceinline__ T digit_scan(T x, T* s_warp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T inc = x;
#pragma unroll
  for (int s = 1; s < 32; s <<= 1) {
    const T y = __shfl_up_sync(0xFFFFFFFFu, inc, s);
    if (lane >= s) inc += y;
  }
  if (lane == 31) s_warp[warp] = inc;
  asm volatile("bar.sync 1, %0;" ::"n"(kRadixBins) : "memory");
  T off = 0;
#pragma unroll
  for (int w = 0; w < kRadixBins / 32; ++w) off += w < warp ? s_warp[w] : 0;
  return off + inc - x;
}

// The move of one tile per CTA.  The load/store unit bounds it (75 % of its data
// pipe, 29 to 32 shared-memory wavefronts per 32 keys, most of them random
// accesses that 32 banks serve in 3.5 cycles; DRAM at 65 %), so the tile costs it
// as little as it can: keys, payloads and tags arrive by bulk copy and stay where
// they came; each warp counts its digits, ranks its keys by ballots (no shared
// memory) and scatters only 16-bit source positions; the way out reads them in
// slot order, gathers, and writes runs of 24 to 30 keys per digit.  5.1 TB/s at
// 2^28 u64 keys + payloads + tags (1.48 ms, 0.75 of the measured copy), 4.4 TB/s
// at 2^30 u32 (4.9 ms).
template <typename K, bool V, typename ID, typename OFF>
__global__ void __launch_bounds__(RadixShape<(int)sizeof(K)>::NT, RadixShape<(int)sizeof(K)>::MB)
k_radix_move(RadixPass<K> a) {
  pdl_enter();
  using L = RadixSmem<K, V, ID, OFF>;
  constexpr int NT = L::NT, VT = L::VT, T = L::T, NW = L::NW;
  using Tag = typename ID::Tag;
  constexpr bool TAGS = ID::bytes != 0;
  static_assert(NT >= kRadixBins && NT % 32 == 0, "a thread per digit");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint16_t* s_perm = reinterpret_cast<uint16_t*>(smem_raw + L::perm);
  uint32_t* s_all = reinterpret_cast<uint32_t*>(smem_raw + L::warp);
  OFF* s_base = reinterpret_cast<OFF*>(smem_raw + L::base);     // digit d's output position of tile slot 0
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw + L::bar);
  __shared__ uint32_t s_warp[kRadixBins / 32];
  __shared__ uint64_t s_warp64[kRadixBins / 32];
  __shared__ int s_stop;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t tile = blockIdx.x;
  uint64_t start, chunk;
  uint32_t cnt, inst;
  if (a.tiles) {
    const RadixTile t = a.tiles[tile];
    start = t.start;
    cnt = t.cnt;
    inst = t.inst;
    chunk = t.chunk;
  } else {
    start = tile * T;
    cnt = (uint32_t)umin(T, a.n - start);
    inst = 0;
    chunk = tile / a.chunk_tiles;
  }
  const Span16 ks = widen16(a.ksrc + start, cnt);
  Span16 vs{nullptr, 0, 0}, ts{nullptr, 0, 0};
  if (V) vs = widen16(a.vsrc + start, cnt);
  if (TAGS && a.tsrc) ts = widen16(static_cast<const Tag*>(a.tsrc) + start, cnt);
  if (tid == 0) {
    s_stop = poisoned(a.err) ? 1 : 0;
    mbar_init(bar, 1);
    fence_barrier_init();
    if (!s_stop) {
      mbar_arrive_expect_tx(bar, ks.bytes + vs.bytes + ts.bytes);
      bulk_load(smem_raw, ks.base, ks.bytes, bar);
      if (vs.bytes) bulk_load(smem_raw + L::val, vs.base, vs.bytes, bar);
      if (ts.bytes) bulk_load(smem_raw + L::tag, ts.base, ts.bytes, bar);
    }
  }
  const K* s_key = reinterpret_cast<const K*>(smem_raw) + ks.skip;
  const uint32_t* s_val = reinterpret_cast<const uint32_t*>(smem_raw + L::val) + vs.skip;
  Tag* s_tag = reinterpret_cast<Tag*>(smem_raw + L::tag) + ts.skip;
  uint32_t* wc = s_all + warp * kRadixBins;         // the warp's digit counters
#pragma unroll
  for (int i = 0; i < kRadixBins / 32; ++i) wc[i * 32 + lane] = 0;
  const uint64_t k0 = a.koff[inst];
  const uint32_t wbase = warp * 32 * VT + lane;     // tile position of item 0; item i sits 32 i further
  uint64_t next = 0;                                // thread d: output position of the tile's first key of digit d
  if (tid < kRadixBins)
    next = k0 + digit_scan<uint64_t>(a.total[(uint64_t)inst * kRadixBins + tid], s_warp64) +
           a.pre[chunk * kRadixBins + tid] + a.cnt[tile * kRadixBins + tid];
  if (ID::run && !a.tsrc) {
    // Run ids of the first pass come from the positions: run r owns
    // [floor(r n / P), floor((r + 1) n / P)), so position x is in run
    // floor(((x + 1) P - 1) / n) and the next run starts at the next bound.
    const uint64_t ni = a.tiles ? a.koff[inst + 1] - k0 : a.n, P = a.P[inst];
    uint64_t x = start - k0 + wbase;
    uint64_t r = umin(((x + 1) * P - 1) / ni, P - 1), bound = run_start(r + 1, ni, P);
#pragma unroll 1
    for (int i = 0; i < VT; ++i) {
      while (x >= bound && r + 1 < P) {
        ++r;
        bound = run_start(r + 1, ni, P);
      }
      s_tag[wbase + i * 32] = (Tag)r;
      x += 32;
    }
  }
  __syncthreads();
  if (s_stop) return;
  if (!mbar_wait(bar, 0, a.wait_ns)) {              // gave up: flag it, let copies in flight land
    atomicOr(a.err, kErrWaitTimeout);
    s_stop = 1;
    mbar_wait(bar, 0, a.wait_ns);
  }

  // This warp's digits, in position order; pads past the end rank last.
  const uint32_t sel = a.byte;
  uint32_t dig[VT];
#pragma unroll
  for (int i = 0; i < VT; ++i) {
    const uint32_t p = wbase + i * 32;
    if (ID::digit && a.tsrc) dig[i] = tag_digit<ID>(s_tag[p]);
    else dig[i] = radix_digit(to_order<K>(s_key[p], a.f32_in), sel);
    if (p >= cnt) dig[i] = kRadixBins - 1;
  }
#pragma unroll
  for (int i = 0; i < VT; ++i) atomicAdd(&wc[dig[i]], 1u);
  __syncthreads();
  if (s_stop) return;

  // Digit d (thread d): the counts of every warp become the tile slots where
  // each warp's keys of the digit start.
  if (tid < kRadixBins) {
    uint32_t c[NW], total = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      c[w] = s_all[w * kRadixBins + tid];
      total += c[w];
    }
    uint32_t run = digit_scan(total, s_warp);
    s_base[tid] = (OFF)(next - run);
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      s_all[w * kRadixBins + tid] = run;
      run += c[w];
    }
  }
  __syncthreads();

  // Tile slot of every key, in position order within its digit.
  const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
  for (int i = 0; i < VT; ++i) {
    const uint32_t m = match_digit(dig[i]);
    const uint32_t below = __popc(m & lt);
    const int lead = 31 - __clz(m);                 // the last of the equal lanes counts them
    uint32_t old = 0;
    if ((m >> lane) == 1u) old = atomicAdd(&wc[dig[i]], below + 1);
    const uint32_t slot = __shfl_sync(0xFFFFFFFFu, old, lead) + below;
    s_perm[slot] = (uint16_t)(wbase + i * 32);
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < VT; ++i) {
    const uint32_t j = i * NT + tid;
    if (j < cnt) {
      const uint32_t p = s_perm[j];
      const K k = to_order<K>(s_key[p], a.f32_in);
      const OFF g = s_base[radix_digit(k, sel)] + (OFF)j;
      a.kdst[g] = from_order<K>(k, a.f32_out);
      if (V) a.vdst[g] = s_val[p];
      if (TAGS && (ID::run || !a.last))
        static_cast<Tag*>(a.tdst)[g] = (Tag)next_tag<ID>(ID::run ? s_tag[p] : 0, a.last ? 0 : radix_digit(k, sel + 1));
    }
  }
}

// ---------------------------------------------------------------------------
// Steps 2-4 on the sorted order.  The run ids of the output are cut into
// groups of kRunGroup tiles of `tile` ids (a power of two; run_tile): cnt
// holds, per tile, the ids of every run before the tile inside its group;
// gpre, per group, the ids of every run before the group.
// ---------------------------------------------------------------------------

constexpr uint32_t kRunGroup = 32;

// Ids per tile for P runs: the tile's row of P counts stays a small share of
// the ids it covers.
__host__ __device__ constexpr uint32_t run_tile(uint32_t P) {
  uint32_t t = 512;
  while (t < 32u * P && t < 32768u) t *= 2;
  return t;
}

struct RunGroup {          // one group (batches; a single sort's groups are closed form)
  uint32_t inst, g;        // instance, group within it
};

// Where an instance's rows are: cnt rows of P entries from cnt_off, gpre rows from gpre_off.
struct RunTables {
  const RunGroup* groups;      // NULL: a single sort
  const uint64_t* cnt_off;     // per instance (NULL: 0)
  const uint64_t* gpre_off;
  uint32_t* cnt;
  uint64_t* gpre;
};

constexpr int kRunHistNT = 256;

// One CTA per group: its tiles' rows of counts and the group's totals (into gpre).
static __global__ void __launch_bounds__(kRunHistNT)
k_run_hist(const uint16_t* __restrict__ ids, Geo geo, RunTables rt) {
  pdl_enter();
  extern __shared__ uint32_t s_cnt[];
  const uint32_t inst = rt.groups ? rt.groups[blockIdx.x].inst : 0;
  const uint32_t g = rt.groups ? rt.groups[blockIdx.x].g : blockIdx.x;
  const uint64_t k0 = geo.koff[inst], n = geo.koff[inst + 1] - k0;
  const uint32_t P = geo.P[inst], tl = run_tile(P);
  const uint64_t tiles = (n + tl - 1) / tl;
  uint32_t* cnt = rt.cnt + (rt.cnt_off ? rt.cnt_off[inst] : 0);
  uint64_t* gpre = rt.gpre + (rt.gpre_off ? rt.gpre_off[inst] : 0);
  for (uint32_t r = threadIdx.x; r < P; r += kRunHistNT) s_cnt[r] = 0;
  __syncthreads();
  const uint16_t* src = ids + k0;
  for (uint32_t k = 0; k < kRunGroup; ++k) {
    const uint64_t t = (uint64_t)g * kRunGroup + k;
    if (t >= tiles) break;
    for (uint32_t r = threadIdx.x; r < P; r += kRunHistNT) cnt[t * P + r] = s_cnt[r];
    __syncthreads();
    const uint64_t lo = t * tl, hi = umin(lo + tl, n);
    for (uint64_t i = lo + threadIdx.x; i < hi; i += kRunHistNT) atomicAdd(&s_cnt[src[i]], 1u);
    __syncthreads();
  }
  for (uint32_t r = threadIdx.x; r < P; r += kRunHistNT) gpre[(uint64_t)g * P + r] = s_cnt[r];
}

// Column-wise exclusive scan of an instance's group totals, in place: CTA
// (instance, block of 32 runs), 32 rows at a time by each of 32 warps' threads.
static __global__ void __launch_bounds__(1024)
k_run_scan(Geo geo, RunTables rt) {
  pdl_enter();
  __shared__ uint64_t s_sum[32][33];
  const uint32_t inst = blockIdx.x;
  const uint64_t n = geo.koff[inst + 1] - geo.koff[inst];
  const uint32_t P = geo.P[inst];
  const uint32_t c = blockIdx.y * 32 + (threadIdx.x & 31);
  if (P < 2 || blockIdx.y * 32 >= P) return;
  const uint64_t tiles = (n + run_tile(P) - 1) / run_tile(P);
  const uint64_t rows = (tiles + kRunGroup - 1) / kRunGroup;
  uint64_t* gpre = rt.gpre + (rt.gpre_off ? rt.gpre_off[inst] : 0);
  const uint32_t part = threadIdx.x >> 5;
  const uint64_t per = (rows + 31) / 32, lo = umin(part * per, rows), hi = umin(lo + per, rows);
  uint64_t sum = 0;
  if (c < P)
    for (uint64_t r = lo; r < hi; ++r) sum += gpre[r * P + c];
  s_sum[part][threadIdx.x & 31] = sum;
  __syncthreads();
  uint64_t pre = 0;
  for (uint32_t p = 0; p < part; ++p) pre += s_sum[p][threadIdx.x & 31];
  if (c < P)
    for (uint64_t r = lo; r < hi; ++r) {
      const uint64_t v = gpre[r * P + c];
      gpre[r * P + c] = pre;
      pre += v;
    }
}

// Samples of a sorted run of nr keys (s of them, at positions
// floor((i + 1) nr / s) - 1) among its first x keys: floor(((x + 1) s - 1) / nr).
__device__ __forceinline__ uint64_t samples_before(uint64_t x, uint64_t s, uint64_t nr) {
  if (nr <= 0xFFFFFFFFull) return ((x + 1) * s - 1) / nr;                 // s <= nr: the product fits
  return (uint64_t)(((unsigned __int128)(x + 1) * s - 1) / nr);
}

constexpr int kFindNT = 256;
constexpr int kFindNW = kFindNT / 32;

// One instance as the splitter search sees it.
struct RunView {
  uint64_t n, s, tiles;
  uint32_t P, tl;
  const uint32_t* cnt;
  const uint64_t* gpre;
};

// Sum over the runs of the samples before the given counts, by one warp.
template <typename F>
__device__ __forceinline__ uint64_t warp_samples(const RunView& v, const F& before) {
  uint64_t sum = 0;
  for (uint32_t r = threadIdx.x & 31; r < v.P; r += 32) {
    const uint64_t nr = run_start(r + 1, v.n, v.P) - run_start(r, v.n, v.P);
    sum += samples_before(before(r), umin(v.s, nr), nr);
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, d);
  return sum;
}

// The last row in [lo, hi) whose sample count is at most k (row lo's is): nine-way
// search, one candidate row per warp.
template <typename F>
__device__ __forceinline__ uint64_t find_row(const RunView& v, uint64_t lo, uint64_t hi, uint64_t k, uint64_t* s_c,
                                             const F& before_row) {
  const uint32_t w = threadIdx.x >> 5;
  while (hi - lo > 1) {
    const uint64_t span = hi - lo;
    const uint64_t m = span <= kFindNW + 1 ? lo + 1 + w : lo + (span * (w + 1)) / (kFindNW + 1);
    if (m < hi) {
      const uint64_t c = warp_samples(v, [&](uint32_t r) { return before_row(m, r); });
      if ((threadIdx.x & 31) == 0) s_c[w] = c;
    }
    __syncthreads();
    uint64_t nlo = lo, nhi = hi;
    for (uint32_t x = 0; x < kFindNW; ++x) {
      const uint64_t mx = span <= kFindNW + 1 ? lo + 1 + x : lo + (span * (x + 1)) / (kFindNW + 1);
      if (mx >= hi) break;
      if (s_c[x] <= k) nlo = mx;
      else if (mx < nhi) nhi = mx;
    }
    lo = nlo;
    hi = nhi;
    __syncthreads();
  }
  return lo;
}

// cut[.][b] = the keys of every run among the first e outputs.
__device__ __forceinline__ void write_cuts(const RunView& v, const uint16_t* __restrict__ ids, uint64_t e, uint32_t b,
                                           uint32_t* s_c, uint64_t* __restrict__ cut) {
  const uint64_t t = umin(e / v.tl, v.tiles - 1), g = t / kRunGroup;
  for (uint32_t r = threadIdx.x; r < v.P; r += kFindNT) s_c[r] = 0;
  __syncthreads();
  for (uint64_t i = t * v.tl + threadIdx.x; i < e; i += kFindNT) atomicAdd(&s_c[ids[i]], 1u);
  __syncthreads();
  for (uint32_t r = threadIdx.x; r < v.P; r += kFindNT)
    cut[(uint64_t)r * (v.P + 1) + b] = v.gpre[g * v.P + r] + v.cnt[t * v.P + r] + s_c[r];
}

// Steps 3 and 4 for bucket boundary b of one instance (one CTA each): the
// splitter t_b, and unless variant is EQUAL (which needs every splitter first)
// the bound e_b and column b of the cut matrix.  The CTAs of b = 0 write the
// fixed cuts.  keys: the sorted output (float bits if f32).
template <typename K>
__global__ void __launch_bounds__(kFindNT)
k_run_splitters(const K* __restrict__ keys, const uint16_t* __restrict__ ids_all, Geo geo, RunTables rt, int f32, int variant,
                K* __restrict__ t_out, K* __restrict__ user_out, uint64_t* __restrict__ cut, uint64_t* __restrict__ e,
                const uint32_t* err) {
  pdl_enter();
  if (cta_poisoned(err)) return;
  extern __shared__ __align__(8) unsigned char s_dyn[];
  __shared__ uint64_t s_c[kFindNW];
  __shared__ uint64_t s_pos, s_e;
  __shared__ uint32_t s_ids[kFindNT];
  const uint32_t beta = blockIdx.x, inst = geo.run_inst[beta], b = beta - geo.R0[inst];
  const uint64_t k0 = geo.koff[inst];
  RunView v;
  v.n = geo.koff[inst + 1] - k0;
  v.P = geo.P[inst];
  v.s = geo.s[inst];
  v.tl = run_tile(v.P);
  v.tiles = (v.n + v.tl - 1) / v.tl;
  v.cnt = rt.cnt + (rt.cnt_off ? rt.cnt_off[inst] : 0);
  v.gpre = rt.gpre + (rt.gpre_off ? rt.gpre_off[inst] : 0);
  const uint16_t* ids = ids_all + k0;
  uint64_t* ei = e + geo.R0[inst] + inst;
  uint64_t* ci = cut ? cut + geo.mat[inst] : nullptr;          // NULL: no cut matrix asked for
  if (b == 0) {
    for (uint32_t r = threadIdx.x; ci && r < v.P; r += kFindNT) {
      ci[(uint64_t)r * (v.P + 1)] = 0;
      ci[(uint64_t)r * (v.P + 1) + v.P] = run_start(r + 1, v.n, v.P) - run_start(r, v.n, v.P);
    }
    if (threadIdx.x == 0) {
      ei[0] = 0;
      ei[v.P] = v.n;
    }
    return;
  }
  uint64_t* s_pre = reinterpret_cast<uint64_t*>(s_dyn);         // P: keys of every run before the window
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(s_pre + v.P);   // P
  const uint64_t S = v.s >= (v.n + v.P - 1) / v.P ? v.n : v.s * v.P;
  const uint64_t k = (uint64_t)(((unsigned __int128)b * S) / v.P) - 1;
  const uint64_t groups = (v.tiles + kRunGroup - 1) / kRunGroup;
  const uint64_t g = find_row(v, 0, groups, k, s_c, [&](uint64_t m, uint32_t r) { return v.gpre[m * v.P + r]; });
  const uint64_t t = find_row(v, g * kRunGroup, umin((g + 1) * kRunGroup, v.tiles), k, s_c,
                              [&](uint64_t m, uint32_t r) { return v.gpre[g * v.P + r] + v.cnt[m * v.P + r]; });
  for (uint32_t r = threadIdx.x; r < v.P; r += kFindNT) {
    s_pre[r] = v.gpre[g * v.P + r] + v.cnt[t * v.P + r];
    s_cnt[r] = 0;
  }
  __syncthreads();
  // Halve the tile until a window of one id per thread holds sample k.
  auto before = [&](uint32_t r) { return s_pre[r] + s_cnt[r]; };
  auto cta_samples = [&]() {
    uint64_t sum = 0;
    for (uint32_t r = threadIdx.x; r < v.P; r += kFindNT) {
      const uint64_t nr = run_start(r + 1, v.n, v.P) - run_start(r, v.n, v.P);
      sum += samples_before(before(r), umin(v.s, nr), nr);
    }
    uint64_t tot;
    block_exclusive_scan(sum, &tot);
    return tot;
  };
  uint64_t lo = t * v.tl, hi = umin(lo + v.tl, v.n);
  while (hi - lo > kFindNT) {
    const uint64_t mid = lo + (hi - lo) / 2;
    for (uint64_t i = lo + threadIdx.x; i < mid; i += kFindNT) atomicAdd(&s_cnt[ids[i]], 1u);
    __syncthreads();
    if (cta_samples() <= k) {                                  // (ends with a barrier)
      lo = mid;
    } else {
      for (uint64_t i = lo + threadIdx.x; i < mid; i += kFindNT) atomicSub(&s_cnt[ids[i]], 1u);
      hi = mid;
      __syncthreads();
    }
  }
  const uint64_t f0 = cta_samples();
  const uint32_t len = (uint32_t)(hi - lo), x = threadIdx.x;
  uint32_t my = 0;
  if (x < len) {
    my = ids[lo + x];
    s_ids[x] = my;
  }
  __syncthreads();
  uint64_t is = 0;
  if (x < len) {
    uint32_t same = 0;
    for (uint32_t y = 0; y < x; ++y) same += s_ids[y] == my;
    const uint64_t pos = before(my) + same;                    // position in its sorted run
    const uint64_t nr = run_start(my + 1, v.n, v.P) - run_start(my, v.n, v.P), s = umin(v.s, nr);
    is = samples_before(pos + 1, s, nr) - samples_before(pos, s, nr);
  }
  if (x == 0) s_pos = umin(hi, v.n) - 1;                       // always found below
  __syncthreads();
  const uint64_t at = f0 + block_exclusive_scan(is, nullptr);
  if (is && at == k) s_pos = lo + x;
  __syncthreads();
  const K* ks = keys + k0;
  const K tb = to_order<K>(ks[s_pos], f32);
  if (x == 0) {
    t_out[beta] = tb;
    if (user_out && geo.I == 1) user_out[b - 1] = from_order<K>(tb, f32);
  }
  if (variant == 1) return;
  // e_b: the target rank, clamped to the range of keys equal to t_b (RANK), or
  // that range's end (OFF).
  if (x < 32) {
    const uint64_t target = (uint64_t)(((unsigned __int128)b * v.n) / v.P);
    const K kt = to_order<K>(ks[target], f32);
    uint64_t eb = target;
    if (variant == 2 || kt > tb)
      eb = warp_partition_point(0, v.n, [&](uint64_t m) { return to_order<K>(ks[m], f32) <= tb; });
    else if (kt < tb)
      eb = warp_partition_point(target, v.n, [&](uint64_t m) { return to_order<K>(ks[m], f32) < tb; });
    if (x == 0) {
      s_e = eb;
      ei[b] = eb;
    }
  }
  __syncthreads();
  if (ci) write_cuts(v, ids, s_e, b, s_cnt, ci);
}

// The EQUAL investigator: a group of k equal splitters divides the range of
// its value into k equal parts.
template <typename K>
__global__ void __launch_bounds__(kFindNT)
k_run_cuts_equal(const K* __restrict__ keys, const uint16_t* __restrict__ ids_all, Geo geo, RunTables rt, int f32,
                 const K* __restrict__ t_in, uint64_t* __restrict__ cut, uint64_t* __restrict__ e, const uint32_t* err) {
  pdl_enter();
  if (cta_poisoned(err)) return;
  extern __shared__ __align__(8) unsigned char s_dyn[];
  __shared__ uint64_t s_e;
  const uint32_t beta = blockIdx.x, inst = geo.run_inst[beta], b = beta - geo.R0[inst];
  if (b == 0) return;
  const uint64_t k0 = geo.koff[inst];
  RunView v;
  v.n = geo.koff[inst + 1] - k0;
  v.P = geo.P[inst];
  v.s = geo.s[inst];
  v.tl = run_tile(v.P);
  v.tiles = (v.n + v.tl - 1) / v.tl;
  v.cnt = rt.cnt + (rt.cnt_off ? rt.cnt_off[inst] : 0);
  v.gpre = rt.gpre + (rt.gpre_off ? rt.gpre_off[inst] : 0);
  const K* ks = keys + k0;
  const K* ti = t_in + geo.R0[inst];
  if (threadIdx.x < 32) {
    const K tb = ti[b];
    const uint64_t L = warp_partition_point(0, v.n, [&](uint64_t m) { return to_order<K>(ks[m], f32) < tb; });
    const uint64_t U = warp_partition_point(L, v.n, [&](uint64_t m) { return to_order<K>(ks[m], f32) <= tb; });
    const uint64_t g0 = partition_point(1, v.P, [&](uint64_t m) { return ti[m] < tb; });
    const uint64_t g1 = partition_point(g0, v.P, [&](uint64_t m) { return ti[m] <= tb; });
    if (threadIdx.x == 0) {
      s_e = L + ((U - L) * (b - g0 + 1)) / (g1 - g0);
      e[geo.R0[inst] + inst + b] = s_e;
    }
  }
  __syncthreads();
  if (cut) write_cuts(v, ids_all + k0, s_e, b, reinterpret_cast<uint32_t*>(s_dyn), cut + geo.mat[inst]);
}

}  // namespace pgs
