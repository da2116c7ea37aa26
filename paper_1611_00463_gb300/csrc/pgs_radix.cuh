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

// Which bytes the passes of an instance of 8-byte keys take, found on the device
// ("Passes that are left out" below).
struct RadixPlan {
  uint64_t diff;                   // bits in which the instance's keys differ (set by the first count)
  uint32_t lo;                     // the first pass's byte; the order below it is k_radix_finish's
  uint32_t pad;
};

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
  uint64_t n, ntiles, wait_ns;
  uint32_t chunk_tiles;            // tiles of a single sort's chunk
  int byte, next, f32_in, f32_out; // this pass's byte and the next one's
  int last;                        // no next pass: tags are runs alone
  // With plans: the pass's number; its bytes and buffers follow on the device.
  RadixPlan* plan;                 // per instance
  const K* kin;
  const uint32_t* vin;
  K *kout, *kalt;
  uint32_t *vout, *valt;
  void *tag_a, *tag_b;
  const uint32_t* most;            // batches: passes of the instance that has most
  int pass;
  int even;                        // an output shares memory with an input (radix_steps)
  int fault;                       // testing only: tile 0 announces its copies and issues none
};

// The bytes a plan's passes take, as a bit mask, and their number (made even,
// with a last pass that moves nothing out of order, where an output shares memory
// with an input: the first pass, which scatters while other tiles are still to be
// read, then writes the workspace).
struct RadixSteps {
  uint32_t bytes, passes;
};
__device__ __forceinline__ RadixSteps radix_steps(uint64_t diff, uint32_t lo, bool even) {
  RadixSteps st{0, 0};
#pragma unroll
  for (int b = 0; b < 8; ++b) st.bytes |= (uint32_t)(((diff >> (8 * b)) & 0xFF) != 0) << b;
  st.bytes = (st.bytes & (0xFFu << lo)) | 1u << lo;
  st.passes = __popc(st.bytes);
  if (even) st.passes += st.passes & 1;
  return st;
}
__device__ __forceinline__ RadixSteps radix_steps(const RadixPlan* plan, bool even) {
  return radix_steps(plan->diff, plan->lo, even);
}
// Byte of pass p (8: none, whose digit is 0).
__device__ __forceinline__ int step_byte(uint32_t bytes, int p) {
  for (; p > 0; --p) bytes &= bytes - 1;
  return bytes ? __ffs((int)bytes) - 1 : 8;
}
// Fills in a planned pass of one instance; false: there is no such pass.  Every
// pass changes buffers, and the last one lands in kout, vout and tag_b.
template <typename K>
__device__ __forceinline__ bool plan_pass(RadixPass<K>& a, uint32_t inst) {
  if (sizeof(K) != 8 || !a.plan) return true;
  const RadixSteps st = radix_steps(a.plan + inst, a.even);
  if (a.pass >= (int)st.passes) return false;
  const bool to_out = ((st.passes - 1 - a.pass) & 1) == 0;
  a.byte = step_byte(st.bytes, a.pass);
  a.next = step_byte(st.bytes, a.pass + 1);
  a.last = a.pass + 1 == (int)st.passes;
  a.ksrc = a.pass == 0 ? a.kin : to_out ? a.kalt : a.kout;
  a.vsrc = a.pass == 0 ? a.vin : to_out ? a.valt : a.vout;
  a.tsrc = a.pass == 0 ? nullptr : to_out ? a.tag_a : a.tag_b;
  a.kdst = to_out ? a.kout : a.kalt;
  a.vdst = to_out ? a.vout : a.valt;
  a.tdst = to_out ? a.tag_b : a.tag_a;
  return true;
}

// True if no instance has this pass (batches: as k_radix_scan_batch found).
template <typename K>
__device__ __forceinline__ bool no_pass(const RadixPass<K>& a) {
  return sizeof(K) == 8 && a.plan && a.pass > 0 && a.most && a.pass >= (int)*a.most;
}

// Byte `sel` of a key, for the pass's uniform byte number.
__device__ __forceinline__ uint32_t radix_digit(uint32_t k, uint32_t sel) { return __byte_perm(k, 0, 0x4440 | sel); }
__device__ __forceinline__ uint32_t radix_digit(uint64_t k, uint32_t sel) {
  const uint32_t w = sel & 4 ? (uint32_t)(k >> 32) : (uint32_t)k;
  return __byte_perm(w, 0, 0x4440 | (sel < 8 ? sel & 3 : 4));        // byte 8: digit 0
}

// One CTA per chunk: each tile's row of counts, of the chunk's tiles before
// it, and the chunk's totals.  With tags that hold it, the digit comes from there.
constexpr int kCountNT = 512;

template <typename K, typename ID, bool TAGS>
__global__ void __launch_bounds__(kCountNT)
k_radix_count(RadixPass<K> a) {
  pdl_enter();
  if (no_pass(a)) return;
  constexpr uint32_t T = radix_tile((int)sizeof(K));
  __shared__ uint32_t s_cnt[kRadixBins];
  __shared__ unsigned long long s_diff;
  uint64_t start, tile;
  uint32_t left, inst = 0;
  if (a.chunks) {
    const RadixChunk c = a.chunks[blockIdx.x];
    inst = c.inst;
    start = c.start;
    tile = c.tile;
    left = c.cnt;
  } else {
    tile = (uint64_t)blockIdx.x * a.chunk_tiles;
    start = tile * T;
    left = (uint32_t)umin((uint64_t)a.chunk_tiles * T, a.n - start);
  }
  const bool first = sizeof(K) == 8 && !TAGS && a.plan && a.pass == 0;   // finds the keys' differing bits, too
  K base = 0, diff = 0;
  if (first) {
    a.byte = a.plan[inst].lo;
    base = a.ksrc[a.chunks ? a.koff[inst] : 0];
  } else if (!plan_pass(a, inst)) {
    return;
  }
  if (threadIdx.x < kRadixBins) s_cnt[threadIdx.x] = 0;
  if (threadIdx.x == 0) s_diff = 0;
  __syncthreads();
  const uint32_t sel = a.byte;
  auto digit = [&](uint64_t i) -> uint32_t {
    if (TAGS) return tag_digit<ID>(static_cast<const typename ID::Tag*>(a.tsrc)[i]);
    const K k = to_order<K>(a.ksrc[i], a.f32_in);
    if (first) diff |= k ^ base;
    return radix_digit(k, sel);
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
  if (first) {
    const uint64_t d = (uint64_t)diff;
    const uint64_t all = (uint64_t)__reduce_or_sync(0xFFFFFFFFu, (uint32_t)(d >> 32)) << 32 |
                         __reduce_or_sync(0xFFFFFFFFu, (uint32_t)d);
    if ((threadIdx.x & 31) == 0) atomicOr(&s_diff, (unsigned long long)all);
    __syncthreads();
    if (threadIdx.x == 0 && (s_diff & ~__ldcg(&a.plan[inst].diff)))  // most CTAs add nothing
      atomicOr(reinterpret_cast<unsigned long long*>(&a.plan[inst].diff), s_diff);
  }
}

// Exclusive prefixes of every digit's chunk totals, in place, and the digit
// totals, for a single sort of `rows` chunks: CTA = 8 digits x 128 parts of
// the rows (8 digits are one 64-byte piece of a row).
// Latency bounds it: with a thread's rows kept in registers and at
// most 1216 of them the four scans of 1.7*10^7 keys take 14 us less of 470.
constexpr int kScanRows = 10, kScanParts = 128;          // at most 1280 rows
static __global__ void __launch_bounds__(1024)
k_radix_scan_wide(uint64_t* pre, uint64_t* total, uint32_t rows, const RadixPlan* plan, int pass, int even) {
  pdl_enter();
  if (plan && pass >= (int)radix_steps(plan, even).passes) return;
  constexpr int D = 8, PARTS = kScanParts;
  static_assert(D * PARTS == 1024, "a thread for each part of a digit's rows");
  __shared__ uint64_t s_sum[PARTS][D];
  const uint32_t x = threadIdx.x % D, part = threadIdx.x / D;
  const uint32_t per = (rows + PARTS - 1) / PARTS, lo = part * per, mine = lo < rows ? min(per, rows - lo) : 0;
  uint64_t* c = pre + (uint64_t)lo * kRadixBins + blockIdx.x * D + x;
  uint64_t sum = 0, v[kScanRows];
#pragma unroll
  for (uint32_t k = 0; k < kScanRows; ++k) v[k] = k < mine ? c[k * kRadixBins] : 0;
#pragma unroll
  for (uint32_t k = 0; k < kScanRows; ++k) sum += v[k];
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
#pragma unroll
  for (uint32_t k = 0; k < kScanRows; ++k) {
    if (k < mine) c[k * kRadixBins] = run;
    run += v[k];
  }
}

// The same for a batch: one CTA per instance, one thread per digit, over the
// instance's chunks [first[i], first[i + 1]).
static __global__ void __launch_bounds__(kRadixBins)
k_radix_scan_batch(uint64_t* pre, uint64_t* total, const uint64_t* __restrict__ first, const RadixPlan* plan, int pass,
                   int even, uint32_t* most) {
  pdl_enter();
  if (plan) {
    const uint32_t passes = radix_steps(plan + blockIdx.x, even).passes;
    if (pass == 0 && threadIdx.x == 0) atomicMax(most, passes);
    if (pass >= (int)passes) return;
  }
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
// or complemented by the lane's own bit (the masks of a warp-level multisplit,
// Ashkiani et al., GPU Multisplit, 2016; in CUB a test, a ballot and a predicated
// complement do it, and here too).  ms a move of 2^28 u64 keys: 1.466; with the ballot
// xor-ed with a mask selected by the bit 1.48, the mask by a shift 1.59, left to the
// compiler 1.78; match.any takes four times as long.
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

// The slot of this lane's key of digit d, and the warp's counters wc moved past
// the warp's 32 keys: equal digits take consecutive slots in lane order.
__device__ __forceinline__ uint32_t warp_slot(uint32_t* wc, uint32_t d) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t m = match_digit(d);
  const uint32_t below = __popc(m & ((1u << lane) - 1u));
  const int lead = 31 - __clz(m);                   // the last of the equal lanes counts them
  uint32_t old = 0;
  if ((m >> lane) == 1u) old = atomicAdd(&wc[d], below + 1);
  return __shfl_sync(0xFFFFFFFFu, old, lead) + below;
}

// Digit threadIdx.x (< 256): the NW warps' counts of it become the slots where
// each warp's keys of the digit start.  Gives the digit's first slot and its keys.
template <int NW>
__device__ __forceinline__ void digit_starts(uint32_t* counters, uint32_t* s_warp, uint32_t& slot0, uint32_t& total) {
  uint32_t* wc = counters + threadIdx.x;
  uint32_t c[NW];
  total = 0;
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    c[w] = wc[w * kRadixBins];
    total += c[w];
  }
  slot0 = digit_scan(total, s_warp);
  uint32_t run = slot0;
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    wc[w * kRadixBins] = run;
    run += c[w];
  }
}

// OFF: the type of output positions (uint32_t up to 2^32 keys).
template <typename K, bool V, typename ID, typename OFF, int NT_, int VT_>
struct RadixSmem {
  static constexpr int NT = NT_, VT = VT_;
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
  static_assert(NT >= kRadixBins && NT % 32 == 0, "a thread per digit");
  static_assert(warp % 16 == 0 && bar % 8 == 0, "aligned parts");
};

constexpr int kAnyPass = 0, kFirstPass = 1, kLaterPass = 2;

// A tile's work, step by step (all NT threads of the CTA; the caller's barriers
// lie between the steps).
template <typename K, bool V, typename ID, typename OFF, int NT, int VT>
struct RadixTileWork {
  using L = RadixSmem<K, V, ID, OFF, NT, VT>;
  using Tag = typename ID::Tag;
  static constexpr int T = L::T, NW = L::NW;
  static constexpr bool TAGS = ID::bytes != 0;
  unsigned char* smem;
  Span16 ks, vs, ts;
  uint32_t cnt;
  uint32_t dig[VT];                                 // this warp's digits, in position order

  __device__ uint64_t* bar() const { return reinterpret_cast<uint64_t*>(smem + L::bar); }
  __device__ uint32_t* counters() const { return reinterpret_cast<uint32_t*>(smem + L::warp); }
  __device__ OFF* base() const { return reinterpret_cast<OFF*>(smem + L::base); }   // digit d's output position of slot 0
  __device__ const K* keys() const { return reinterpret_cast<const K*>(smem) + ks.skip; }
  __device__ Tag* tags() const { return reinterpret_cast<Tag*>(smem + L::tag) + ts.skip; }
  // Tile position of this thread's item 0; item i sits 32 i further.
  __device__ static uint32_t first_item() { return (threadIdx.x >> 5) * 32 * VT + (threadIdx.x & 31); }

  // Where the tile [start, start + cnt) lies; thread 0 sends for it.
  __device__ void locate(const RadixPass<K>& a, uint64_t start, uint32_t count) {
    cnt = count;
    ks = widen16(a.ksrc + start, cnt);
    vs = ts = Span16{nullptr, 0, 0};
    if (V) vs = widen16(a.vsrc + start, cnt);
    if (TAGS && a.tsrc) ts = widen16(static_cast<const Tag*>(a.tsrc) + start, cnt);
  }
  __device__ void send(bool lost) const {
    mbar_arrive_expect_tx(bar(), ks.bytes + vs.bytes + ts.bytes);
    if (lost) return;                               // fault injection: nothing is in flight, the wait runs out
    bulk_load(smem, ks.base, ks.bytes, bar());
    if (vs.bytes) bulk_load(smem + L::val, vs.base, vs.bytes, bar());
    if (ts.bytes) bulk_load(smem + L::tag, ts.base, ts.bytes, bar());
  }
  // Clears the warp's digit counters.
  __device__ void clear() const {
    uint32_t* wc = counters() + (threadIdx.x >> 5) * kRadixBins;
#pragma unroll
    for (int i = 0; i < kRadixBins / 32; ++i) wc[i * 32 + (threadIdx.x & 31)] = 0;
  }
  // Run ids of the first pass, from the positions (x of an instance of n keys):
  // run r owns [floor(r n / P), floor((r + 1) n / P)), so position x is in run
  // floor(((x + 1) P - 1) / n) and the next run starts at the next bound.  A tile
  // no longer than a run meets one bound at most: a compare with it is the id.
  // Shorter runs' ids are written to the tags.
  __device__ void find_runs(uint64_t x0, uint64_t n, uint64_t P, uint32_t* s_run) const {
    if (n / P >= T) {
      if (threadIdx.x == NT - 1) {
        const uint64_t r = umin(((x0 + 1) * P - 1) / n, P - 1);
        s_run[0] = (uint32_t)r;
        s_run[1] = r + 1 < P ? (uint32_t)umin(run_start(r + 1, n, P) - x0, T) : (uint32_t)T;
      }
      return;
    }
    if (threadIdx.x == NT - 1) s_run[1] = 0;                 // the tags tell
    Tag* s_tag = tags();
    const uint32_t w = first_item();
    uint64_t x = x0 + w;
    uint64_t r = umin(((x + 1) * P - 1) / n, P - 1), bound = run_start(r + 1, n, P);
#pragma unroll 1
    for (int i = 0; i < VT; ++i) {
      while (x >= bound && r + 1 < P) {
        ++r;
        bound = run_start(r + 1, n, P);
      }
      s_tag[w + i * 32] = (Tag)r;
      x += 32;
    }
  }
  // Once the tile has landed: digits (pads past the end rank last) and the
  // warp's counts of them.  PASS: the first (no tags yet), a later one, or either.
  template <int PASS = kAnyPass>
  __device__ void count(const RadixPass<K>& a) {
    uint32_t* wc = counters() + (threadIdx.x >> 5) * kRadixBins;
    const uint32_t w = first_item(), sel = a.byte;
    const K* s_key = keys();
    const Tag* s_tag = tags();
#pragma unroll
    for (int i = 0; i < VT; ++i) {
      const uint32_t p = w + i * 32;
      if (ID::digit && (PASS == kLaterPass || (PASS == kAnyPass && a.tsrc))) dig[i] = tag_digit<ID>(s_tag[p]);
      else dig[i] = radix_digit(to_order<K>(s_key[p], a.f32_in), sel);
      if (p >= cnt) dig[i] = kRadixBins - 1;
    }
#pragma unroll
    for (int i = 0; i < VT; ++i) atomicAdd(&wc[dig[i]], 1u);
  }
  // Digit d (thread d < 256): the tile slots where each warp's keys of the digit
  // start; the digit's first slot and its keys in the tile (pads included).
  __device__ void starts(uint32_t* s_warp, uint32_t& slot0, uint32_t& total) const {
    digit_starts<NW>(counters(), s_warp, slot0, total);
  }
  // Tile slot of every key, in position order within its digit: the slot gets
  // the key's tile position.
  __device__ void rank() const {
    uint32_t* wc = counters() + (threadIdx.x >> 5) * kRadixBins;
    uint16_t* s_perm = reinterpret_cast<uint16_t*>(smem + L::perm);
    const uint32_t w = first_item();
#pragma unroll
    for (int i = 0; i < VT; ++i) s_perm[warp_slot(wc, dig[i])] = (uint16_t)(w + i * 32);
  }
  // The way out, in slot order.  s_run: the tile's first run and where the next
  // one starts, or a 0 there (find_runs).
  template <int PASS = kAnyPass>
  __device__ void write(const RadixPass<K>& a, const uint32_t* s_run) const {
    if (ID::run && (PASS == kFirstPass || (PASS == kAnyPass && !a.tsrc)) && s_run[1]) {
      const uint32_t run = s_run[0], bound = s_run[1];
      write_out(a, [=](uint32_t p) { return run + (p >= bound); });
    } else {
      const Tag* s_tag = tags();
      write_out(a, [=](uint32_t p) { return ID::run ? (uint32_t)s_tag[p] : 0u; });
    }
  }
  template <typename F>
  __device__ void write_out(const RadixPass<K>& a, const F& tag) const {
    const uint16_t* s_perm = reinterpret_cast<const uint16_t*>(smem + L::perm);
    const uint32_t* s_val = reinterpret_cast<const uint32_t*>(smem + L::val) + vs.skip;
    const K* s_key = keys();
    const OFF* s_base = base();
    const uint32_t sel = a.byte;
#pragma unroll
    for (int i = 0; i < VT; ++i) {
      const uint32_t j = i * NT + threadIdx.x;
      if (j < cnt) {
        const uint32_t p = s_perm[j];
        const K k = to_order<K>(s_key[p], a.f32_in);
        const OFF g = s_base[radix_digit(k, sel)] + (OFF)j;
        a.kdst[g] = from_order<K>(k, a.f32_out);
        if (V) a.vdst[g] = s_val[p];
        if (TAGS && (ID::run || !a.last))
          static_cast<Tag*>(a.tdst)[g] = (Tag)next_tag<ID>(tag(p), a.last ? 0 : radix_digit(k, a.next));
      }
    }
  }
};

// The move of one tile per CTA.  The load/store unit bounds it (75 % of its data
// pipe, 29 to 32 shared-memory wavefronts per 32 keys, most of them random
// accesses that 32 banks serve in 3.5 cycles; DRAM at 65 %), so the tile costs it
// as little as it can: keys, payloads and tags arrive by bulk copy and stay where
// they came; each warp counts its digits, ranks its keys by ballots (no shared
// memory) and scatters only 16-bit source positions; the way out reads them in
// slot order, gathers, and writes runs of 24 to 30 keys per digit.  5.1 TB/s at
// 2^28 u64 keys + payloads + tags (1.48 ms, 0.75 of the measured copy), 4.4 TB/s
// at 2^30 u32 (4.8 ms).
// LOOP: a few CTAs take all tiles in turn, for passes that are mostly left out
// (an empty CTA of this size costs 1.9 ns, 82 us a pass of 2^28 keys; a pass that
// is run takes 1.98 ms so, 1.45 with a CTA per tile).
// PASS: the first pass works the runs out and reads its digits from the keys, the
// later ones find both in the tags; in one kernel each slows the other down (2^29
// f32 keys, ms: 2.83 and 2.23 as one, 2.53 and 2.28 with the two ways out as
// branches).
template <typename K, bool V, typename ID, typename OFF, int PASS, bool LOOP>
__global__ void __launch_bounds__(RadixShape<(int)sizeof(K)>::NT, RadixShape<(int)sizeof(K)>::MB)
k_radix_move(RadixPass<K> a) {
  pdl_enter();
  if (LOOP && no_pass(a)) return;
  using W = RadixTileWork<K, V, ID, OFF, RadixShape<(int)sizeof(K)>::NT, RadixShape<(int)sizeof(K)>::VT>;
  constexpr int T = W::T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t s_warp[kRadixBins / 32];
  __shared__ uint64_t s_warp64[kRadixBins / 32];
  __shared__ int s_stop, s_lost;                    // the call has failed; the tile's copies never came
  __shared__ uint32_t s_run[2];
  const int tid = threadIdx.x;
  W w;
  w.smem = smem_raw;
  uint32_t waits = 0;
  for (uint64_t tile = blockIdx.x; !LOOP || tile < a.ntiles; tile += gridDim.x) {
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
    if (!plan_pass(a, inst)) {
      if (!LOOP || !a.tiles) return;
      continue;
    }
    if (LOOP && waits) {                            // the last tile's shared memory is read
      asm volatile("fence.proxy.async;" ::: "memory");
      __syncthreads();
    }
    w.locate(a, start, cnt);
    if (tid == 0) {
      if (waits == 0) {
        s_stop = poisoned(a.err) ? 1 : 0;
        s_lost = 0;
        mbar_init(w.bar(), 1);
        fence_barrier_init();
      }
      if (!s_stop) w.send(PASS == kFirstPass && a.fault && tile == 0);
    }
    w.clear();
    const uint64_t k0 = a.koff[inst];
    uint64_t next = 0;                              // thread d: output position of the tile's first key of digit d
    if (tid < kRadixBins)
      next = k0 + digit_scan<uint64_t>(a.total[(uint64_t)inst * kRadixBins + tid], s_warp64) +
             a.pre[chunk * kRadixBins + tid] + a.cnt[tile * kRadixBins + tid];
    if (ID::run && PASS == kFirstPass) w.find_runs(start - k0, a.tiles ? a.koff[inst + 1] - k0 : a.n, a.P[inst], s_run);
    __syncthreads();
    if (s_stop) return;
    if (!mbar_wait_copies(w.bar(), waits & 1, a.wait_ns, a.err)) s_lost = 1;
    w.template count<PASS>(a);
    __syncthreads();
    if (s_lost) return;
    if (tid < kRadixBins) {
      uint32_t slot0, total;
      w.starts(s_warp, slot0, total);
      w.base()[tid] = (OFF)(next - slot0);
    }
    __syncthreads();
    w.rank();
    __syncthreads();
    w.template write<PASS>(a, s_run);
    if (!LOOP) return;
    ++waits;
  }
}

// ---------------------------------------------------------------------------
// Passes that are left out (8-byte keys).  A pass costs the same whatever its
// byte holds, and most of eight bytes hold nothing: the top ones are often
// constant, and once a few have told nearly all keys apart the rest only order
// the few that are left.  So a sample of the keys says from which byte `lo` on
// the keys are (nearly) told apart, the passes take the bytes from lo up that
// differ at all (the first count finds them, exactly), and k_radix_finish puts
// the keys that agree above lo in order, stably, in place, with one read of the
// keys and little else.  A segment of more than kFinishReach such keys that is
// out of order is left to k_radix_redo.  The order is right whatever the sample
// says; it decides only what is done where.
// Measured against eight passes: 2^28 normal/lognormal keys with payloads, P =
// 128, 13.5 -> 8.7 ms (four passes and counts 6.7, the finish 1.5, the plan 0.06,
// the passes left out 0.15); 2*10^7 keys alone 1.11 -> 0.69 ms; a batch of 2000
// uneven instances (uniform, exponential, Zipf), 4.5*10^8 keys, 20.1 -> 11.3.
// ---------------------------------------------------------------------------

constexpr int kPickNT = 1024, kPickVT = 8, kPlanKeys = kPickNT * kPickVT;
constexpr int kFinishNT = 640, kFinishVT = 10, kFinishReach = 256;
static_assert(kFinishNT * kFinishVT == radix_tile(8) + kFinishReach, "a pass's tile and its reach");
// Unlike keys a key may agree with on average: six cost the finish about what the
// pass they would save costs (6 ps a key).
constexpr float kPlanMates = 6.0f;
constexpr size_t kFinishSmem = 8 + kFinishNT * kFinishVT * (8 + 2);
constexpr size_t kPickSmem = kPlanKeys * 8 + kPickNT / 32 * kRadixBins * 4;

struct RadixSeg {
  uint64_t start, end;
  uint64_t what;           // low byte: the instance's lo; above it, the bits in which the keys differ (k_radix_redo)
};

// Keys sampled of an instance of n: one pair of them that agree then stands for
// some eight unlike keys that a key agrees with.
__device__ __forceinline__ uint32_t plan_keys(uint64_t n) {
  uint32_t m = kPickNT;
  while (m < kPlanKeys && 4ull * m * m < n) m += kPickNT;
  return m;
}

__device__ __forceinline__ uint64_t plan_hash(uint32_t i) {
  uint64_t h = (i + 1) * 0x9E3779B97F4A7C15ull;            // splitmix64's finalizer
  h = (h ^ (h >> 30)) * 0xBF58476D1CE4E5B9ull;
  h = (h ^ (h >> 27)) * 0x94D049BB133111EBull;
  return h ^ (h >> 31);
}

// Positions of a uniform sample, one in each of m equal parts.
__device__ __forceinline__ uint64_t plan_position(uint32_t i, uint64_t n, uint32_t m) {
  const uint64_t a = i * n / m, b = (i + 1) * n / m;        // n < 2^40
  return a + plan_hash(i) % (b - a);
}

// Such a sample is blind to keys that lie closer together in the input than its
// parts are long, where those of a nearly sorted one have their mates.  So sampled
// keys are compared with one further on, too, at a distance d of 1 to a part's
// length, its logarithm uniform: each unlike pair that descends and agrees above so
// many bytes then stands for d log(length) mates on one side, and as many keys that
// ascend (sorted input, which leaves the finish nothing to do, has none that
// descend).  Timestamps a microsecond apart in order, give or take 65, P = 4, by
// merges / without / with this: 10^6 133 / 171 / 133 us, 2*10^6 179 / 225 / 167, 3*10^7
// 1745 / 1937 / 1350.
constexpr uint32_t kBesidePairs = 3;                        // fewer are chance
struct Beside {
  uint32_t pairs[9], mates[9];                               // by the bytes in which a pair differs; d added up
};
__device__ __forceinline__ float beside_length(uint64_t n, uint32_t m) { return fminf((float)n / (float)m, 0x1p20f); }
__device__ __forceinline__ uint32_t beside_distance(uint32_t i, float length) {
  const float u = (float)(uint32_t)(plan_hash(i) >> 40) * 0x1p-24f;
  return max(1u, (uint32_t)exp2f(u * log2f(length)));          // length below 1: 1
}
__device__ __forceinline__ void see_beside(Beside* s, uint64_t k, uint64_t after, uint32_t d) {
  const uint64_t x = k ^ after;
  if (after >= k || x >> 56) return;
  const int b = (71 - __clzll((long long)x)) / 8;
  atomicAdd(&s->pairs[b], 1u);
  atomicAdd(&s->mates[b], d);
}
// The largest byte up to lo above which `count` compared keys have few such mates.
__device__ __forceinline__ uint32_t lo_beside(const Beside& s, uint32_t lo, uint32_t count, float length) {
  for (; lo > 0; --lo) {
    uint32_t pairs = 0, mates = 0;
    for (uint32_t b = 1; b <= lo; ++b) pairs += s.pairs[b];
    if (pairs < kBesidePairs) break;
    for (uint32_t b = 1; b <= lo; ++b) mates += s.mates[b];
    if (4.0f * logf(length) * (float)mates <= kPlanMates * (float)count) break;
  }
  return lo;
}

// The lo of up to kFewKeys keys, by kFewNT threads of a CTA (the others only pass
// its barriers): one sampled key a thread, each compared with half of the others;
// 3 us, where sorting a sample takes 15.  The rule is k_radix_plan's, with a
// byte's margin where the sample holds kFewDups equal pairs or more: a value that
// many keys share makes a long segment of any other that agrees with it, and so
// small a sample misses most values.
constexpr uint32_t kFewNT = 384, kFewDups = 24;
constexpr uint64_t kFewKeys = 1 << 18;
__device__ __forceinline__ uint32_t few_plan(const uint64_t* __restrict__ keys, uint64_t n, uint64_t* s_key,
                                             uint32_t* s_pairs, uint32_t* s_crowd) {
  constexpr uint32_t M = kFewNT;
  __shared__ Beside s_beside;
  const uint32_t tid = threadIdx.x;
  uint64_t k = 0, after = 0;
  const float length = beside_length(n, M);
  uint32_t d = 0;
  if (tid < M) {
    const uint64_t p = n >= M ? plan_position(tid, n, M) : tid % n;
    d = beside_distance(tid, length);
    after = keys[umin(p + d, n - 1)];
    s_key[tid] = k = keys[p];
  }
  if (tid < 9) s_pairs[tid] = s_crowd[tid] = s_beside.pairs[tid] = s_beside.mates[tid] = 0;
  __syncthreads();
  if (tid < M) {
    see_beside(&s_beside, k, after, d);
    uint64_t levels = 0;                                     // 8 bits a level: pairs that agree above so many bytes
    uint32_t at = tid;
#pragma unroll 4
    for (uint32_t j = 0; j < M / 2; ++j) {
      at = at + 1 == M ? 0 : at + 1;
      const uint64_t x = k ^ s_key[at];
      if (x >> 56 == 0) levels += x ? 1ull << (56 - (__clzll((long long)x) & ~7)) : 1ull << 56;   // level 8: equal
    }
    for (uint32_t b = 1; b <= 8; ++b) {
      const uint32_t pairs = (uint32_t)(levels >> (8 * (b - 1))) & 0xFF;
      if (pairs) atomicAdd(&s_pairs[b], pairs);
      if (pairs > 2) s_crowd[b] = 1;
    }
  }
  __syncthreads();
  uint32_t lo = 0, pairs = 0;
  for (uint32_t b = 1; b < 8; ++b) {
    pairs += s_pairs[b];
    if (s_crowd[b] || 2.0f * (float)pairs * (float)n > kPlanMates * (float)M * (float)M) break;
    lo = b;
  }
  if (s_pairs[8] == M * (M / 2)) return 0;                   // one value: the bytes that differ at all are few
  return lo_beside(s_beside, lo > 0 && s_pairs[8] >= kFewDups ? lo - 1 : lo, M, length);
}

// Chooses an instance's lo from a sample of its keys (a CTA an instance) and
// clears the rest of the plan and the segments' marks.  lo is the largest byte
// above which a key agrees with fewer than kPlanMates unlike keys on average, as
// the sample's pairs have it, and no part of the sample hints at a large crowd:
// no four keys that agree and are not all equal, no such pair of values with
// more than two pairs of keys between them.  The sample is sorted like a tile
// of a pass, in the bytes in which its keys differ.
static __global__ void __launch_bounds__(kPickNT)
k_radix_plan(const uint64_t* __restrict__ keys_all, const uint64_t* __restrict__ koff, RadixPlan* plan, uint32_t* bits,
             uint64_t words) {
  pdl_enter();
  extern __shared__ __align__(8) unsigned char s_dyn[];
  uint64_t* s = reinterpret_cast<uint64_t*>(s_dyn);
  uint32_t* counters = reinterpret_cast<uint32_t*>(s + kPlanKeys);
  __shared__ uint32_t s_warp[kRadixBins / 32], s_pairs[9], s_crowd[9], s_diff[2];
  __shared__ Beside s_beside;
  constexpr uint32_t HOT = 64;
  __shared__ uint64_t s_hot[HOT];                             // hot values, up to so many
  __shared__ uint32_t s_nhot, s_near[9], s_runs[3];           // values seen, once, twice; the once's agreements with hot ones
  const int tid = threadIdx.x;
  const uint64_t k0 = koff[blockIdx.x], n = koff[blockIdx.x + 1] - k0;
  const uint64_t* keys = keys_all + k0;
  const uint32_t m = plan_keys(n);
  const int vt = m / kPickNT;
  for (uint64_t i = blockIdx.x * (uint64_t)kPickNT + tid; i < words; i += (uint64_t)gridDim.x * kPickNT) bits[i] = 0;
  if (n <= kFewKeys) {
    const uint32_t lo = n ? few_plan(keys, n, s, s_pairs, s_crowd) : 7;
    if (tid == 0) plan[blockIdx.x] = RadixPlan{0, lo, 0};
    return;
  }
  if (tid < 9) s_pairs[tid] = s_crowd[tid] = s_near[tid] = 0;
  if (tid < 2) s_diff[tid] = 0;
  if (tid < 3) s_runs[tid] = 0;
  if (tid == 0) s_nhot = 0;
  if (tid < 9) s_beside.pairs[tid] = s_beside.mates[tid] = 0;
  const float length = beside_length(n, m);                   // the first kPickNT keys are compared
  const uint32_t d = beside_distance(tid, length);
  const uint64_t p = plan_position(tid, n, m), after = keys[umin(p + d, n - 1)];
  uint64_t k[kPickVT];
  const uint64_t k_first = keys[0];
  k[0] = keys[p];
#pragma unroll
  for (int i = 1; i < kPickVT; ++i) {
    const uint32_t x = i * kPickNT + tid;
    k[i] = k_first;
    if (x < m) k[i] = keys[plan_position(x, n, m)];
  }
  __syncthreads();
  see_beside(&s_beside, k[0], after, d);
  uint64_t diff = 0;
#pragma unroll
  for (int i = 0; i < kPickVT; ++i) {
    diff |= k[i] ^ k_first;
    const uint32_t x = i * kPickNT + tid;
    if (i < vt) s[x] = k[i];
  }
  const uint32_t d0 = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)diff), d1 = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)(diff >> 32));
  if ((tid & 31) == 0) {
    atomicOr(&s_diff[0], d0);
    atomicOr(&s_diff[1], d1);
  }
  __syncthreads();
  diff = (uint64_t)s_diff[1] << 32 | s_diff[0];
  uint32_t* wc = counters + (tid >> 5) * kRadixBins;
  const uint32_t w = (tid >> 5) * 32 * vt + (tid & 31);
  for (int b = 0; b < 8; ++b) {
    if (((diff >> (8 * b)) & 0xFF) == 0) continue;
    uint32_t d[kPickVT];
#pragma unroll
    for (int i = 0; i < kRadixBins / 32; ++i) wc[i * 32 + (tid & 31)] = 0;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < kPickVT; ++i)
      if (i < vt) {
        k[i] = s[w + i * 32];
        d[i] = radix_digit(k[i], b);
        atomicAdd(&wc[d[i]], 1u);
      }
    __syncthreads();
    if (tid < kRadixBins) {
      uint32_t slot0, total;
      digit_starts<kPickNT / 32>(counters, s_warp, slot0, total);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kPickVT; ++i)
      if (i < vt) s[warp_slot(wc, d[i])] = k[i];
    __syncthreads();
  }
  auto bytes = [](uint64_t x) { return (71 - __clzll((long long)x)) / 8; };   // x's significant bytes
  // A value seen so often makes a segment that is long.
  const uint32_t often = min(max(3u, (uint32_t)((uint64_t)kFinishReach * m / n)), 8u);
  for (uint32_t i = tid; i < m; i += kPickNT) {
    const uint64_t x = i + 1 < m ? s[i] ^ s[i + 1] : 1;
    if (x) {                                                // the last of its value
      uint32_t l = 1, r = 1;
      while (l < 8 && i >= l && s[i - l] == s[i]) ++l;
      atomicAdd(&s_runs[0], 1u);
      if (l <= 2) atomicAdd(&s_runs[l], 1u);
      if (l >= often) {
        const uint32_t at = atomicAdd(&s_nhot, 1u);
        if (at < HOT) s_hot[at] = s[i];
      }
      if (i + 1 == m) break;
      // Unlike neighbours: they agree above bytes(x).
      while (r < 8 && i + 1 + r < m && s[i + 1 + r] == s[i + 1]) ++r;
      atomicAdd(&s_pairs[bytes(x)], l * r);
      if (l * r > 2) s_crowd[bytes(x)] = 1;
    }
    if (i + 3 < m && s[i] != s[i + 3]) s_crowd[bytes(s[i] ^ s[i + 3])] = 1;
  }
  __syncthreads();
  const uint32_t hot = min(s_nhot, HOT);
  for (uint32_t i = tid; hot && i < m; i += kPickNT) {
    if ((i > 0 && s[i - 1] == s[i]) || (i + 1 < m && s[i + 1] == s[i])) continue;
    uint64_t levels = 0;                                    // a value seen once: the hot ones it agrees with above so many bytes
    for (uint32_t h = 0; h < hot; ++h) levels += 1ull << (8 * bytes(s[i] ^ s_hot[h]) - 8);
    for (uint32_t b = 1; b <= 8; ++b)
      if (const uint32_t c = (uint32_t)(levels >> (8 * b - 8)) & 0xFF) atomicAdd(&s_near[b], c);
  }
  __syncthreads();
  if (tid == 0) {
    uint32_t lo = 0, pairs = 0;
    for (uint32_t b = 1; b < 8; ++b) {
      pairs += s_pairs[b];
      if (s_crowd[b] || 2.0f * (float)pairs * (float)n > kPlanMates * (float)m * (float)m) break;
      lo = b;
    }
    // A hot value makes a long segment of any other value that agrees with it,
    // and the sample has not seen all values.  Those seen once and twice tell how
    // many there are (Chao's estimate; at most the keys that the once's share of
    // the sample stands for), the once's agreements with hot values, a byte's
    // 256th for each byte further up, how many to expect: bytes are added while
    // it is more than one in a hundred (a batch of instances takes the risk often).
    const float once = (float)s_runs[1], twice = (float)s_runs[2];
    if (hot && once > 0.0f) {
      float values = once * (float)n / (float)m;
      if (twice > 0.0f) values = fminf(values, once * once / (2.0f * twice));
      for (; lo > 0; --lo) {
        float expect = values, share = 1.0f / 256.0f;
        uint32_t agree = 0;
        for (uint32_t b = 1; b <= lo; ++b) agree += s_near[b];
        for (uint32_t b = lo + 1; b <= 8; ++b, share /= 256.0f) {
          agree += s_near[b];
          expect = fminf(expect, values * ((float)agree + 0.5f) / once * share);
        }
        if (expect <= 0.01f) break;
      }
    }
    lo = lo_beside(s_beside, lo, kPickNT, length);
    if (s_runs[0] == 1) lo = 0;                             // one value: the bytes that differ at all are few
    plan[blockIdx.x] = RadixPlan{0, lo, 0};
  }
}

struct RadixFinish {
  uint64_t* keys;                  // sorted by the bytes from lo up
  uint32_t* vals;
  uint16_t* tags;
  uint64_t* kalt;
  uint32_t* valt;
  uint16_t* talt;
  const RadixTile* tiles;          // NULL: a single sort
  const uint64_t* koff;
  RadixPlan* plan;
  RadixSeg* segs;                  // segments left to k_radix_redo
  uint64_t cap;
  uint32_t* bits;                  // bit p / kFinishReach: the segment that starts at p is listed
  uint32_t* listed;                // segments listed
  const uint32_t* most;            // batches: the most passes an instance has
  uint32_t* passes;                // passes made, for the statistics
  int even;
  uint32_t* rows;
  uint32_t* err;
  uint32_t* barrier;               // k_radix_redo's arrivals, zero at the call's start and no other kernel's
  uint64_t n, wait_ns;
  int fault;                       // testing only: k_radix_redo's CTA 0 waits for arrivals that never come
};

// The order below byte lo, tile by tile (the passes' tiles).  Keys that agree
// from lo up lie together; a segment of them belongs to the tile it starts in,
// which reads kFinishReach keys past its end, and one out of order is ranked by
// comparing its keys with one another.  Ballot words of the segments' starts and
// of the descents inside them tell in a few bit operations that most keys have
// nothing to do.  Other tiles' keys may be permuted while they are read, but
// only inside a segment, where all agree on what is looked at.  Instructions
// bound it (77 % of the issue slots; 1.52 ms at 2^28 normal/lognormal keys, half
// of which sit with one or two others, 76 us at 2*10^7, which mostly sit alone;
// DRAM floors 0.6 and 0.024): unrolled over a thread's keys the look at a segment
// overflows the instruction cache (2.4 ms), and a list of the segments, one
// thread each, leaves lanes idle (2.2).
template <bool V, bool RUN>
__global__ void __launch_bounds__(kFinishNT, 3)
k_radix_finish(RadixFinish f) {
  pdl_enter();
  constexpr int NT = kFinishNT, VT = kFinishVT, WORDS = NT * VT / 32, REACH = kFinishReach / 32 + 1;
  constexpr uint32_t T = radix_tile(8);
  extern __shared__ __align__(8) unsigned char s_dyn[];
  uint64_t* s_key = reinterpret_cast<uint64_t*>(s_dyn) + 1;          // [-1]: the key before the tile
  uint16_t* s_to = reinterpret_cast<uint16_t*>(s_key + NT * VT);      // where each key goes
  __shared__ uint32_t s_start[WORDS], s_desc[WORDS];
  uint64_t start = blockIdx.x * (uint64_t)T, k0 = 0, k1 = f.n;
  uint32_t cnt = (uint32_t)umin(T, k1 - start), inst = 0;
  if (f.tiles) {
    const RadixTile t = f.tiles[blockIdx.x];
    inst = t.inst;
    start = t.start;
    cnt = t.cnt;
    k0 = f.koff[t.inst];
    k1 = f.koff[t.inst + 1];
  }
  const uint32_t lo = f.plan[inst].lo;
  if (lo == 0 || cta_poisoned(f.err)) return;
  const int sh = 8 * lo;
  const uint32_t len = (uint32_t)umin(cnt + kFinishReach, k1 - start);
#pragma unroll
  for (int u = 0; u < VT; ++u) {
    const uint32_t i = u * NT + threadIdx.x;
    if (i < len) s_key[i] = f.keys[start + i];
  }
  // Before the instance's first key: one that differs from it above lo.
  if (threadIdx.x == 0) s_key[-1] = start > k0 ? f.keys[start - 1] : ~f.keys[start];
  __syncthreads();
  uint32_t any = 0;
  auto words = [&](auto agree) {                             // agree(k, before): equal from lo up
#pragma unroll
    for (int u = 0; u < VT; ++u) {
      const uint32_t i = u * NT + threadIdx.x;
      const uint64_t k = s_key[i], before = s_key[(int)i - 1];
      const bool same = agree(k, before) && i < len;
      const uint32_t dw = __ballot_sync(0xFFFFFFFFu, same && k < before);
      const uint32_t fw = ~__ballot_sync(0xFFFFFFFFu, same);
      any |= dw;
      if ((threadIdx.x & 31) == 0) {
        s_start[i / 32] = fw;
        s_desc[i / 32] = dw;
      }
    }
  };
  if (lo >= 4)
    words([=](uint64_t k, uint64_t b) { return (((uint32_t)(k >> 32) ^ (uint32_t)(b >> 32)) >> (sh - 32)) == 0; });
  else
    words([=](uint64_t k, uint64_t b) { return ((k ^ b) >> sh) == 0; });
  if (!__syncthreads_or(any != 0)) return;
  // The segment of key i, as far as the tile's words tell: its start (-1: not
  // within reach) and the next segment's (0: not within reach).
  auto seg_start = [&](uint32_t i) {
    int w = i / 32;
    uint32_t m = s_start[w] & (0xFFFFFFFFu >> (31 - i % 32));
    for (int r = 0; r < REACH && m == 0 && w > 0; ++r) m = s_start[--w];
    return m ? w * 32 + 31 - __clz(m) : -1;
  };
  auto seg_end = [&](uint32_t i) {
    int w = i / 32;
    uint32_t m = s_start[w] & ~(0xFFFFFFFFu >> (31 - i % 32));
    for (int r = 0; r < REACH && m == 0 && w + 1 < WORDS; ++r) m = s_start[++w];
    const uint32_t e = m ? w * 32 + __ffs(m) - 1 : w + 1 == WORDS ? WORDS * 32 : 0;
    return e < len || start + len == k1 ? (int)e : 0;
  };
  uint32_t moved = 0;                                        // bit u: this thread's u-th key
#pragma unroll 1
  for (uint32_t i = threadIdx.x, bit = 1; i < len; i += NT, bit *= 2) {
    // Starts and descents of the 32 keys up to i and of the 32 after it.
    const int w = i / 32, q = i % 32;
    const uint32_t back = __funnelshift_l(w > 0 ? s_start[w - 1] : 0, s_start[w], 31 - q);
    const uint32_t ahead = __funnelshift_rc(s_start[w], w + 1 < WORDS ? s_start[w + 1] : 0, q + 1);
    if ((back >> 31) && (ahead & 1)) continue;               // a segment of one key
    int s, e;
    bool desc;
    if (back && ahead) {                                     // nearly always
      s = i - __clz(back);
      e = i + __ffs(ahead);
      const uint32_t dback = __funnelshift_l(w > 0 ? s_desc[w - 1] : 0, s_desc[w], 31 - q);
      const uint32_t dahead = __funnelshift_rc(s_desc[w], w + 1 < WORDS ? s_desc[w + 1] : 0, q + 1);
      desc = (dback >> (31 - __clz(back))) || (dahead & ((1u << (e - i - 1)) - 1));
    } else {
      s = seg_start(i);
      e = seg_end(i);
      desc = false;
      if (s >= 0 && e > 0)
        for (int x = s / 32; x <= (e - 1) / 32 && !desc; ++x) {
          uint32_t m = s_desc[x];
          if (x == s / 32) m &= ~0u << (s % 32);
          if (x == (e - 1) / 32) m &= 0xFFFFFFFFu >> (31 - (e - 1) % 32);
          desc = m != 0;
        }
    }
    if (s >= (int)cnt) continue;                             // the next tile's
    if (s >= 0 && e > 0 && e - s <= kFinishReach) {
      if (!desc) continue;
      uint32_t to = s;
      if (lo <= 4) {                                         // they differ in the low word alone
        const uint32_t* low = reinterpret_cast<const uint32_t*>(s_key);
        const uint32_t k = low[2 * i];
#pragma unroll 4
        for (int j = s; j < e; ++j) to += low[2 * j] < k || (j < (int)i && low[2 * j] == k);
      } else {
        const uint64_t k = s_key[i];
        for (int j = s; j < e; ++j) to += s_key[j] < k || (j < (int)i && s_key[j] == k);
      }
      if (to != i) {
        s_to[i] = (uint16_t)to;
        moved |= bit;
      }
    } else if (i < cnt && (s_desc[w] >> q & 1)) {
      // A descent in a segment that is long, or starts in an earlier tile (which
      // then orders it, if it is short).  The first such tile lists it.
      const uint64_t pre = s_key[i] >> sh;
      uint64_t a = start + s, z = start + e;
      if (s < 0) {
        a = k0;
        for (uint64_t h = start + i; a < h;) {
          const uint64_t mid = a + (h - a) / 2;
          if (f.keys[mid] >> sh < pre) a = mid + 1;
          else h = mid;
        }
      }
      if (e == 0) {
        z = start + i;
        for (uint64_t h = k1; z < h;) {
          const uint64_t mid = z + (h - z) / 2;
          if (f.keys[mid] >> sh <= pre) z = mid + 1;
          else h = mid;
        }
      }
      if (z - a <= kFinishReach) continue;
      uint32_t* word = f.bits + a / kFinishReach / 32;
      const uint32_t mark = 1u << (a / kFinishReach % 32);
      if ((__ldcg(word) & mark) || (atomicOr(word, mark) & mark)) continue;
      const uint64_t at = atomicAdd(f.listed, 1u);
      if (at < f.cap) f.segs[at] = RadixSeg{a, z, lo};
      else atomicOr(f.err, kErrBadTile);
    }
  }
  // Payloads and tags of the keys that move are all read before any is written.
  uint32_t val[VT], tag[VT];
  __syncthreads();
#pragma unroll
  for (int u = 0; u < VT; ++u) {
    const uint32_t i = u * NT + threadIdx.x;
    if (moved >> u & 1) {
      if (V) val[u] = f.vals[start + i];
      if (RUN) tag[u] = f.tags[start + i];
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < VT; ++u) {
    const uint32_t i = u * NT + threadIdx.x;
    if (moved >> u & 1) {
      const uint64_t g = start + s_to[i];
      f.keys[g] = s_key[i];
      if (V) f.vals[g] = val[u];
      if (RUN) f.tags[g] = (uint16_t)tag[u];
    }
  }
}

// ---------------------------------------------------------------------------
// Small sorts: every pass in one cooperative launch, one tile per CTA, all
// tiles resident.  A pass is a tile's count, a grid barrier (every tile's
// counts are published), each tile's place from the rows of counts, the move,
// and a grid barrier (the next pass reads what every tile wrote).  Against
// three launches a pass, whose latencies bound a sort of this size: 2^20 u32
// keys 133.6 -> 88.9 us for the whole call, 2^16 keys 107 -> 58.  A pass of 43
// tiles of 4 keys a thread takes 7.0 us: landing 0.6, counting and publishing
// 0.7, the tile's own ranks 1.3 (they cover the first barrier), rows and scan
// 0.8, the way out 0.8, the second barrier 2.3.  8-byte keys leave passes out as
// larger sorts do (few_plan in every CTA, the differing bits with the first counts):
// against merges, P = 24, 2^20 keys 178 -> 130 us and 8192 keys 89 -> 60, where
// eight passes took 178 and 76.
// ---------------------------------------------------------------------------

constexpr int kSmallNT = 384, kSmallMB = 2;

template <typename K>
struct RadixSmall {
  RadixPass<K> pass;               // first pass; the others follow from the buffers below
  K *kout, *kalt;
  uint32_t *vout, *valt;
  void *tag_a, *tag_b;
  uint16_t* rows;                  // tiles x 256 digit counts, digit d at (d % 32) * 8 + d / 32
  uint32_t* barrier;               // arrivals of the call's grid barriers, zero at the start
  uint64_t* diff;                  // 8-byte keys: bits in which they differ, zero at the start
  RadixPlan* plan;                 // and what k_radix_finish is told
  uint32_t* bits;
  uint32_t words;
  int f32;
  int fault;                       // testing only: CTA 0 waits for arrivals that never come
};

constexpr uint32_t kNeverArrives = 1u << 30;                // fault injection: more than any call's arrivals

// A grid barrier in two halves: every CTA's writes before its arrival are
// visible to every CTA after the wait (BULK: to the bulk copies that its thread
// 0 issues, too: a proxy fence on both sides).
template <bool BULK>
__device__ __forceinline__ void grid_arrive(uint32_t* counter) {
  if (BULK) asm volatile("fence.proxy.async;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
}
// False (for the whole CTA): the wait gave up.
template <bool BULK>
__device__ __forceinline__ bool grid_wait(uint32_t* counter, uint32_t target, uint32_t* err, uint64_t wait_ns,
                                          int* s_stop) {
  if (threadIdx.x == 0) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
    if (v < target) {
      const uint64_t t0 = global_timer_ns();
      const uint64_t limit = wait_ns ? wait_ns : kWaitLimitNs;
      while (true) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
        if (v >= target) break;
        if (poisoned(err) || global_timer_ns() - t0 > limit) {
          atomicOr(err, kErrWaitTimeout);
          *s_stop = 1;
          break;
        }
      }
    }
    if (BULK) asm volatile("fence.proxy.async;" ::: "memory");
  }
  __syncthreads();
  return *s_stop == 0;
}

template <typename K, bool V, typename ID, int VT>
__global__ void __launch_bounds__(kSmallNT, kSmallMB)
k_radix_small(RadixSmall<K> p) {
  using W = RadixTileWork<K, V, ID, uint32_t, kSmallNT, VT>;
  constexpr int D = (int)sizeof(K), T = W::T, NW = W::NW;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t s_warp[kRadixBins / 32];
  __shared__ uint32_t s_before[kRadixBins], s_total[kRadixBins];
  __shared__ int s_stop;
  __shared__ uint32_t s_run[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t tiles = gridDim.x, tile = blockIdx.x;
  RadixPass<K> a = p.pass;
  const uint64_t start = (uint64_t)tile * T;
  const uint32_t cnt = (uint32_t)umin(T, a.n - start);
  W w;
  w.smem = smem_raw;
  if (tid == 0) {
    s_stop = 0;
    mbar_init(w.bar(), 1);
    fence_barrier_init();
  }
  __syncthreads();
  uint32_t arrivals = 0;
  constexpr bool PLAN = sizeof(K) == 8;
  uint32_t lo = 0;
  RadixSteps st{0, D};
  if (PLAN) {
    static_assert(kFewNT == kSmallNT, "a key a thread");
    lo = few_plan(reinterpret_cast<const uint64_t*>(a.ksrc), a.n, reinterpret_cast<uint64_t*>(smem_raw), s_before, s_total);
    for (uint32_t i = tid; tile == 0 && i < p.words; i += kSmallNT) p.bits[i] = 0;
    asm volatile("fence.proxy.async;" ::: "memory");       // bulk copies write over the sample
    __syncthreads();
  }
#pragma unroll 1
  for (int d = 0; d < (int)st.passes; ++d) {
    if (d > 0) {
      const bool from_alt = ((st.passes - 1 - d) & 1) == 0;
      a.ksrc = from_alt ? p.kalt : p.kout;
      a.vsrc = from_alt ? p.valt : p.vout;
      a.tsrc = ID::bytes ? (from_alt ? p.tag_a : p.tag_b) : nullptr;
    }
    a.byte = PLAN ? (d ? step_byte(st.bytes, d) : (int)lo) : d;
    a.f32_in = d == 0 ? p.f32 : 0;
    w.locate(a, start, cnt);
    if (tid == 0) w.send(a.fault && d == 0 && tile == 0);
    w.clear();
    if (tid < kRadixBins) s_before[tid] = s_total[tid] = 0;
    if (ID::run && !a.tsrc) w.find_runs(start, a.n, a.P[0], s_run);
    __syncthreads();
    if (!mbar_wait_copies(w.bar(), d & 1, a.wait_ns, a.err)) s_stop = 1;
    w.count(a);
    if (PLAN && d == 0) {                               // and the bits in which the keys differ
      const uint64_t base = reinterpret_cast<const uint64_t*>(p.pass.ksrc)[0];
      uint64_t diff = 0;
#pragma unroll
      for (int i = 0; i < VT; ++i)
        if (w.first_item() + i * 32 < cnt) diff |= (uint64_t)w.keys()[w.first_item() + i * 32] ^ base;
      const uint64_t all = (uint64_t)__reduce_or_sync(0xFFFFFFFFu, (uint32_t)(diff >> 32)) << 32 |
                           __reduce_or_sync(0xFFFFFFFFu, (uint32_t)diff);
      if (lane == 0 && (all & ~__ldcg(p.diff))) atomicOr(reinterpret_cast<unsigned long long*>(p.diff), all);
    }
    __syncthreads();
    if (s_stop) return;
    // The counts are published, and the keys ranked inside the tile while the
    // other tiles' counts come in.
    if (tid < kRadixBins) {
      uint32_t total = 0;
#pragma unroll
      for (int x = 0; x < NW; ++x) total += w.counters()[x * kRadixBins + tid];
      p.rows[tile * kRadixBins + (tid % 32) * 8 + tid / 32] =
          (uint16_t)(total - (tid == kRadixBins - 1 ? T - cnt : 0));              // without the pads
    }
    arrivals += tiles;
    grid_arrive<false>(p.barrier);
    uint32_t slot0 = 0;
    if (tid < kRadixBins) {
      uint32_t total;
      w.starts(s_warp, slot0, total);
    }
    __syncthreads();
    w.rank();
    if (!grid_wait<false>(p.barrier, arrivals + (p.fault && tile == 0 ? kNeverArrives : 0), a.err, a.wait_ns, &s_stop)) return;
    if (PLAN && d == 0) st = radix_steps(__ldcg(p.diff), lo, p.pass.even);
    const bool to_out = ((st.passes - 1 - d) & 1) == 0; // the last pass lands in the caller's output
    a.kdst = to_out ? p.kout : p.kalt;
    a.vdst = to_out ? p.vout : p.valt;
    a.tdst = to_out ? p.tag_b : p.tag_a;
    a.next = PLAN ? step_byte(st.bytes, d + 1) : d + 1;
    a.last = d + 1 == (int)st.passes;
    a.f32_out = a.last ? p.f32 : 0;
    // Keys of each digit in all tiles and in the tiles before this one: a warp
    // reads a row with one 16-byte load per lane (lane l: digits l, 32 + l, ...).
    uint32_t before[8] = {}, all[8] = {};
    constexpr int B = 4;
    for (uint32_t r0 = warp; r0 < tiles; r0 += B * NW) {
      uint4 v[B];
#pragma unroll
      for (int k = 0; k < B; ++k) {
        const uint32_t r = r0 + k * NW;
        v[k] = r < tiles ? __ldcg(reinterpret_cast<const uint4*>(p.rows) + r * 32 + lane) : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int k = 0; k < B; ++k) {
        const uint32_t x[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
        const bool mine = r0 + k * NW < tile;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const uint32_t c = (x[q / 2] >> (16 * (q % 2))) & 0xFFFF;
          all[q] += c;
          before[q] += mine ? c : 0;
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      atomicAdd(&s_total[q * 32 + lane], all[q]);
      atomicAdd(&s_before[q * 32 + lane], before[q]);
    }
    __syncthreads();
    if (tid < kRadixBins) w.base()[tid] = digit_scan(s_total[tid], s_warp) + s_before[tid] - slot0;
    __syncthreads();
    w.write(a, s_run);
    if (a.last) break;
    arrivals += tiles;
    grid_arrive<true>(p.barrier);
    if (!grid_wait<true>(p.barrier, arrivals, a.err, a.wait_ns, &s_stop)) return;
  }
  if (PLAN && tile == 0 && tid == 0) *p.plan = RadixPlan{*p.diff, lo, 0};
}

// ---------------------------------------------------------------------------
// The segments k_radix_finish lists, sorted by their bytes below lo: rare, so
// kept simple.  One cooperative launch; a large segment is taken by all CTAs
// together (some 12 us a pass more than its keys need), the others by one CTA
// each (1 ns a key and pass): from 2^14 keys if there are few, else from 2^17.
// Bytes in which all of a segment's keys agree are left out.  2^26 u64 keys, half
// of them of one value with 10^-5 in its neighbourhood, which a sample misses: 3.36
// ms (4.96 with all bytes passed over and an add a key to one counter; by merges 4.07).
// ---------------------------------------------------------------------------

constexpr int kRedoNT = 512, kRedoVT = 8, kRedoCtas = 152;
constexpr uint64_t kRedoFew = 16, kRedoBigFew = 1 << 14, kRedoBig = 1 << 17;

// One pass over segment [s, e) by CTA `me` of `ctas`, whose keys are a
// contiguous part of it; `back`: they are in the alternate buffers.  False: a
// wait gave up.
template <bool V, bool RUN>
__device__ bool redo_pass(const RadixFinish& f, uint64_t s, uint64_t e, int byte, bool back, uint32_t me, uint32_t ctas,
                          uint32_t* counters, uint64_t* s_base, uint32_t* s_hist, uint32_t& arrivals, int* s_stop) {
  constexpr int NT = kRedoNT, VT = kRedoVT, NW = NT / 32, CH = NT * VT;
  __shared__ uint32_t s_warp[kRadixBins / 32];
  __shared__ uint64_t s_warp64[kRadixBins / 32];
  const uint64_t* ksrc = back ? f.kalt : f.keys;
  const uint32_t* vsrc = back ? f.valt : f.vals;
  const uint16_t* tsrc = back ? f.talt : f.tags;
  uint64_t* kdst = back ? f.keys : f.kalt;
  uint32_t* vdst = back ? f.vals : f.valt;
  uint16_t* tdst = back ? f.tags : f.talt;
  const int tid = threadIdx.x;
  const uint64_t per = ((e - s + ctas - 1) / ctas + CH - 1) / CH * CH;
  const uint64_t lo = umin(s + me * per, e), hi = umin(lo + per, e);
  if (tid < kRadixBins) s_hist[tid] = 0;
  __syncthreads();
  // Many keys of a segment are mostly of one value: a warp whose digits agree adds once.
  for (uint64_t i0 = lo + (tid & ~31); i0 < hi; i0 += VT * NT) {
    uint32_t d[VT];
#pragma unroll
    for (int i = 0; i < VT; ++i) {
      const uint64_t at = i0 + i * NT + (tid & 31);
      d[i] = at < hi ? radix_digit(__ldcg(ksrc + at), byte) : kRadixBins;
    }
#pragma unroll
    for (int i = 0; i < VT; ++i) {
      const uint32_t first = __shfl_sync(0xFFFFFFFFu, d[i], 0);
      const uint32_t live = __ballot_sync(0xFFFFFFFFu, d[i] < kRadixBins);
      if (__all_sync(0xFFFFFFFFu, d[i] == first || d[i] == kRadixBins)) {
        if ((tid & 31) == 0 && live) atomicAdd(&s_hist[first], __popc(live));
      } else if (d[i] < kRadixBins) {
        atomicAdd(&s_hist[d[i]], 1u);
      }
    }
  }
  __syncthreads();
  if (ctas > 1) {
    if (tid < kRadixBins) f.rows[me * kRadixBins + tid] = s_hist[tid];
    arrivals += ctas;
    grid_arrive<false>(f.barrier);
    if (!grid_wait<false>(f.barrier, arrivals + (f.fault && me == 0 ? kNeverArrives : 0), f.err, f.wait_ns, s_stop)) return false;
  }
  if (tid < kRadixBins) {
    uint64_t before = 0, all = s_hist[tid];
    if (ctas > 1) {
      all = 0;
      for (uint32_t c = 0; c < ctas; ++c) {
        const uint32_t x = __ldcg(f.rows + c * kRadixBins + tid);
        all += x;
        before += c < me ? x : 0;
      }
    }
    s_base[tid] = s + digit_scan<uint64_t>(all, s_warp64) + before;
  }
  uint32_t* wc = counters + (tid >> 5) * kRadixBins;
  for (uint64_t c0 = lo; c0 < hi; c0 += CH) {
    const uint32_t cnt = (uint32_t)umin(CH, hi - c0), w = (tid >> 5) * 32 * VT + (tid & 31);
    uint64_t k[VT];
    uint32_t d[VT];
#pragma unroll
    for (int i = 0; i < kRadixBins / 32; ++i) wc[i * 32 + (tid & 31)] = 0;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < VT; ++i) {
      k[i] = w + i * 32 < cnt ? __ldcg(ksrc + c0 + w + i * 32) : ~0ull;      // pads rank last
      d[i] = w + i * 32 < cnt ? radix_digit(k[i], byte) : kRadixBins - 1;
      atomicAdd(&wc[d[i]], 1u);
    }
    __syncthreads();
    uint64_t next = 0;
    if (tid < kRadixBins) {
      uint32_t slot0, total;
      digit_starts<NW>(counters, s_warp, slot0, total);
      next = s_base[tid] + total - (tid == kRadixBins - 1 ? CH - cnt : 0);
      s_base[tid] -= slot0;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < VT; ++i) {
      const uint64_t g = s_base[d[i]] + warp_slot(wc, d[i]);
      if (w + i * 32 < cnt) {
        kdst[g] = k[i];
        if (V) vdst[g] = __ldcg(vsrc + c0 + w + i * 32);
        if (RUN) tdst[g] = __ldcg(tsrc + c0 + w + i * 32);
      }
    }
    __syncthreads();
    if (tid < kRadixBins) s_base[tid] = next;
    __syncthreads();
  }
  if (ctas > 1) {
    arrivals += ctas;
    grid_arrive<false>(f.barrier);
    return grid_wait<false>(f.barrier, arrivals, f.err, f.wait_ns, s_stop);
  }
  __syncthreads();
  return true;
}

// The bits in which the segment's keys differ (all of them below byte lo), found
// by CTA `me` of `ctas`.  False: a wait gave up.
__device__ __forceinline__ bool redo_diff(const RadixFinish& f, RadixSeg* seg, uint64_t s, uint64_t e, uint32_t me,
                                          uint32_t ctas, uint32_t& arrivals, int* s_stop, uint64_t& diff) {
  constexpr int NT = kRedoNT, VT = kRedoVT;
  __shared__ unsigned long long s_diff;
  const uint64_t base = __ldcg(f.keys + s);
  uint64_t d = 0;
  if (threadIdx.x == 0) s_diff = 0;
  __syncthreads();
  for (uint64_t i = s + me * (uint64_t)(VT * NT) + threadIdx.x; i < e; i += (uint64_t)ctas * (VT * NT)) {
#pragma unroll
    for (int u = 0; u < VT; ++u) d |= (i + u * NT < e ? __ldcg(f.keys + i + u * NT) : base) ^ base;
  }
  const uint64_t all = (uint64_t)__reduce_or_sync(0xFFFFFFFFu, (uint32_t)(d >> 32)) << 32 |
                       __reduce_or_sync(0xFFFFFFFFu, (uint32_t)d);
  if ((threadIdx.x & 31) == 0) atomicOr(&s_diff, (unsigned long long)all);
  __syncthreads();
  diff = s_diff;
  if (ctas == 1) return true;
  if (threadIdx.x == 0) atomicOr(reinterpret_cast<unsigned long long*>(&seg->what), (unsigned long long)diff << 8);
  arrivals += ctas;
  grid_arrive<false>(f.barrier);
  if (!grid_wait<false>(f.barrier, arrivals, f.err, f.wait_ns, s_stop)) return false;
  diff = __ldcg(&seg->what) >> 8;
  return true;
}

// Segment [s, e) from the alternate buffers, by CTA `me` of `ctas`.
template <bool V, bool RUN>
__device__ void redo_copy(const RadixFinish& f, uint64_t s, uint64_t e, uint32_t me, uint32_t ctas) {
  for (uint64_t i = s + me * kRedoNT + threadIdx.x; i < e; i += (uint64_t)ctas * kRedoNT) {
    f.keys[i] = __ldcg(f.kalt + i);
    if (V) f.vals[i] = __ldcg(f.valt + i);
    if (RUN) f.tags[i] = __ldcg(f.talt + i);
  }
}

template <bool V, bool RUN>
__global__ void __launch_bounds__(kRedoNT)
k_radix_redo(RadixFinish f) {
  __shared__ uint32_t s_counters[kRedoNT / 32 * kRadixBins], s_hist[kRadixBins];
  __shared__ uint64_t s_base[kRadixBins];
  __shared__ int s_stop;
  if (blockIdx.x == 0 && threadIdx.x == 0) *f.passes = f.most ? *f.most : radix_steps(f.plan, f.even).passes;
  const uint32_t segs = *f.listed;
  if (segs == 0 || cta_poisoned(f.err)) return;
  if (threadIdx.x == 0) s_stop = 0;
  __syncthreads();
  uint32_t arrivals = 0;
  for (int big = 1; big >= 0; --big)                          // the shared ones first: their waits stay short
    for (uint32_t j = big ? 0 : blockIdx.x; j < segs; j += big ? 1 : gridDim.x) {
      const RadixSeg x = f.segs[j];
      if ((x.end - x.start > (segs <= kRedoFew ? kRedoBigFew : kRedoBig)) != (big != 0)) continue;
      const uint32_t me = big ? blockIdx.x : 0, ctas = big ? gridDim.x : 1;
      uint64_t diff;
      if (!redo_diff(f, f.segs + j, x.start, x.end, me, ctas, arrivals, &s_stop, diff)) return;
      bool back = false;
      for (int d = 0; d < (int)(x.what & 0xFF); ++d) {
        if (((diff >> (8 * d)) & 0xFF) == 0) continue;
        if (!redo_pass<V, RUN>(f, x.start, x.end, d, back, me, ctas, s_counters, s_base, s_hist, arrivals, &s_stop))
          return;
        back = !back;
      }
      if (back) redo_copy<V, RUN>(f, x.start, x.end, me, ctas);
    }
}

// ---------------------------------------------------------------------------
// Steps 2-4 on the sorted order.  The run ids of the output are cut into
// groups of tiles of `tile` ids (a power of two; run_tile): cnt
// holds, per tile, the ids of every run before the tile inside its group;
// gpre, per group, the ids of every run before the group.
// ---------------------------------------------------------------------------

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
  uint32_t group;              // tiles per group
};

// Adds `delta` to s_cnt[id] for every id in [p, p + n), by all NT threads: 16
// bytes (8 ids) a load, four loads in flight (a scalar loop waits for each id).
// Ids are not checked against P.  find_runs gives none above P - 1, the passes
// carry them unchanged and the last one leaves nothing else in the tags, as long
// as none has failed: after a wait that ran out the tags hold an earlier pass's
// (run and digit) or what was in the workspace, so the callers return at entry
// once the error word is set.
template <int NT>
__device__ __forceinline__ void count_ids(const uint16_t* __restrict__ p, uint32_t n, uint32_t* s_cnt, uint32_t delta) {
  const uint32_t head = min(n, (uint32_t)((16 - (reinterpret_cast<uintptr_t>(p) & 15)) & 15) / 2);
  if (threadIdx.x < head) atomicAdd(&s_cnt[p[threadIdx.x]], delta);
  const uint4* v = reinterpret_cast<const uint4*>(p + head);
  const uint32_t vecs = (n - head) / 8;
  auto add = [&](uint32_t w) {
    atomicAdd(&s_cnt[w & 0xFFFF], delta);
    atomicAdd(&s_cnt[w >> 16], delta);
  };
  constexpr int U = 4;
  for (uint32_t i = threadIdx.x; i < vecs; i += U * NT) {
    uint4 x[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i + u * NT < vecs) x[u] = __ldg(v + i + u * NT);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i + u * NT < vecs) {
        add(x[u].x);
        add(x[u].y);
        add(x[u].z);
        add(x[u].w);
      }
  }
  const uint32_t tail = head + vecs * 8;
  if (threadIdx.x < n - tail) atomicAdd(&s_cnt[p[tail + threadIdx.x]], delta);
}

constexpr int kRunHistNT = 256;

// One CTA per group: its tiles' rows of counts and the group's totals (into gpre).
static __global__ void __launch_bounds__(kRunHistNT)
k_run_hist(const uint16_t* __restrict__ ids, Geo geo, RunTables rt, const uint32_t* err) {
  pdl_enter();
  extern __shared__ uint32_t s_cnt[];
  __shared__ int s_stop;
  if (threadIdx.x == 0) s_stop = poisoned(err) ? 1 : 0;
  const uint32_t inst = rt.groups ? rt.groups[blockIdx.x].inst : 0;
  const uint32_t g = rt.groups ? rt.groups[blockIdx.x].g : blockIdx.x;
  const uint64_t k0 = geo.koff[inst], n = geo.koff[inst + 1] - k0;
  const uint32_t P = geo.P[inst], tl = run_tile(P);
  const uint64_t tiles = (n + tl - 1) / tl;
  uint32_t* cnt = rt.cnt + (rt.cnt_off ? rt.cnt_off[inst] : 0);
  uint64_t* gpre = rt.gpre + (rt.gpre_off ? rt.gpre_off[inst] : 0);
  for (uint32_t r = threadIdx.x; r < P; r += kRunHistNT) s_cnt[r] = 0;
  __syncthreads();
  if (s_stop) return;
  const uint16_t* src = ids + k0;
  for (uint32_t k = 0; k < rt.group; ++k) {
    const uint64_t t = (uint64_t)g * rt.group + k;
    if (t >= tiles) break;
    for (uint32_t r = threadIdx.x; r < P; r += kRunHistNT) cnt[t * P + r] = s_cnt[r];
    __syncthreads();
    const uint64_t lo = t * tl, hi = umin(lo + tl, n);
    count_ids<kRunHistNT>(src + lo, (uint32_t)(hi - lo), s_cnt, 1u);
    __syncthreads();
  }
  for (uint32_t r = threadIdx.x; r < P; r += kRunHistNT) gpre[(uint64_t)g * P + r] = s_cnt[r];
}

// Column-wise exclusive scan of an instance's group totals, in place: CTA
// (instance, block of 32 runs), 32 rows at a time by each of 32 warps' threads.
// Two rounds of loads bound it, so a thread's rows stay in registers where 608
// groups suffice (a 2^20-key sort 88.2 -> 86.2 us).
constexpr int kRunScanRows = 19;                         // 608 groups by 32 parts
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
  const uint64_t rows = (tiles + rt.group - 1) / rt.group;
  uint64_t* gpre = rt.gpre + (rt.gpre_off ? rt.gpre_off[inst] : 0);
  const uint32_t part = threadIdx.x >> 5;
  const uint64_t per = (rows + 31) / 32, lo = umin(part * per, rows), hi = umin(lo + per, rows);
  uint64_t sum = 0, v[kRunScanRows];
  const bool held = per <= kRunScanRows;                // a thread's rows stay in registers
  if (held) {
#pragma unroll
    for (int k = 0; k < kRunScanRows; ++k) v[k] = c < P && lo + k < hi ? gpre[(lo + k) * P + c] : 0;
#pragma unroll
    for (int k = 0; k < kRunScanRows; ++k) sum += v[k];
  } else if (c < P) {
#pragma unroll 8
    for (uint64_t r = lo; r < hi; ++r) sum += gpre[r * P + c];
  }
  s_sum[part][threadIdx.x & 31] = sum;
  __syncthreads();
  uint64_t pre = 0;
  for (uint32_t p = 0; p < part; ++p) pre += s_sum[p][threadIdx.x & 31];
  if (held) {
#pragma unroll
    for (int k = 0; k < kRunScanRows; ++k) {
      if (c < P && lo + k < hi) gpre[(lo + k) * P + c] = pre;
      pre += v[k];
    }
  } else if (c < P) {
#pragma unroll 8
    for (uint64_t r = lo; r < hi; ++r) {
      const uint64_t x = gpre[r * P + c];
      gpre[r * P + c] = pre;
      pre += x;
    }
  }
}

// Samples of a sorted run of nr keys (s of them, at positions
// floor((i + 1) nr / s) - 1) among its first x keys: floor(((x + 1) s - 1) / nr).
__device__ __forceinline__ uint64_t samples_before(uint64_t x, uint64_t s, uint64_t nr) {
  if (((nr + 1) * s >> 32) == 0 && nr <= 0xFFFFFFFEull)                  // a short division where it fits
    return ((uint32_t)(x + 1) * (uint32_t)s - 1u) / (uint32_t)nr;
  if (nr <= 0xFFFFFFFFull) return ((x + 1) * s - 1) / nr;                 // s <= nr: the product fits
  return (uint64_t)(((unsigned __int128)(x + 1) * s - 1) / nr);
}

constexpr int kFindNT = 256;
constexpr int kFindNW = kFindNT / 32;

// One instance as the splitter search sees it.
struct RunView {
  uint64_t n, s, tiles;
  uint32_t P, tl, group;
  const uint32_t* cnt;
  const uint64_t* gpre;
  const uint64_t* ro;      // the runs' first keys
};

// Sum over the runs of the samples before the given counts, by one warp.
template <typename F>
__device__ __forceinline__ uint64_t warp_samples(const RunView& v, const F& before) {
  uint64_t sum = 0;
  for (uint32_t r = threadIdx.x & 31; r < v.P; r += 32) {
    const uint64_t nr = v.ro[r + 1] - v.ro[r];
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
  const uint64_t t = umin(e / v.tl, v.tiles - 1), g = t / v.group;
  for (uint32_t r = threadIdx.x; r < v.P; r += kFindNT) s_c[r] = 0;
  __syncthreads();
  count_ids<kFindNT>(ids + t * v.tl, (uint32_t)(e - t * v.tl), s_c, 1u);
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
  v.group = rt.group;
  v.ro = geo.run_off + geo.R0[inst];
  v.tiles = (v.n + v.tl - 1) / v.tl;
  v.cnt = rt.cnt + (rt.cnt_off ? rt.cnt_off[inst] : 0);
  v.gpre = rt.gpre + (rt.gpre_off ? rt.gpre_off[inst] : 0);
  const uint16_t* ids = ids_all + k0;
  uint64_t* ei = e + geo.R0[inst] + inst;
  uint64_t* ci = cut ? cut + geo.mat[inst] : nullptr;          // NULL: no cut matrix asked for
  if (b == 0) {
    for (uint32_t r = threadIdx.x; ci && r < v.P; r += kFindNT) {
      ci[(uint64_t)r * (v.P + 1)] = 0;
      ci[(uint64_t)r * (v.P + 1) + v.P] = v.ro[r + 1] - v.ro[r];
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
  const uint64_t groups = (v.tiles + v.group - 1) / v.group;
  const uint64_t g = find_row(v, 0, groups, k, s_c, [&](uint64_t m, uint32_t r) { return v.gpre[m * v.P + r]; });
  const uint64_t t = find_row(v, g * v.group, umin((g + 1) * v.group, v.tiles), k, s_c,
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
      const uint64_t nr = v.ro[r + 1] - v.ro[r];
      sum += samples_before(before(r), umin(v.s, nr), nr);
    }
    uint64_t tot;
    block_exclusive_scan(sum, &tot);
    return tot;
  };
  uint64_t lo = t * v.tl, hi = umin(lo + v.tl, v.n);
  while (hi - lo > kFindNT) {
    const uint64_t mid = lo + (hi - lo) / 2;
    count_ids<kFindNT>(ids + lo, (uint32_t)(mid - lo), s_cnt, 1u);
    __syncthreads();
    if (cta_samples() <= k) {                                  // (ends with a barrier)
      lo = mid;
    } else {
      count_ids<kFindNT>(ids + lo, (uint32_t)(mid - lo), s_cnt, ~0u);
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
    const uint64_t nr = v.ro[my + 1] - v.ro[my], s = umin(v.s, nr);
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
  v.group = rt.group;
  v.ro = geo.run_off + geo.R0[inst];
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

// ---------------------------------------------------------------------------
// Tiny sorts: one CTA, one launch for the whole call.  The keys stay where they
// were loaded, in order form; every pass permutes 16-bit positions.  One more
// pass by run lists each run's keys in sorted order, from which samples,
// splitters, bounds and cuts follow as above.  Bound by the latencies of one
// CTA's barriers: 2000 u32 keys on 4 partitions 54 us (eleven launches of merge
// rounds and their planning) -> 19.5 us.
// ---------------------------------------------------------------------------

constexpr int kTinyVT = 8;
constexpr uint32_t kTinyMaxP = 256;

template <typename K>
struct RadixTiny {
  const K* kin;
  const uint32_t* vin;
  K* kout;
  uint32_t* vout;
  uint64_t* bounds;          // optional outputs, as the call asks for them
  uint64_t* cuts;
  K* splitters;
  DevStats* stats;
  uint64_t s;                // samples per run
  uint32_t n, P;
  int f32, variant, want;    // want: any of bounds, cuts, splitters, stats
};

template <typename K, int NT>
struct TinySmem {
  static constexpr int T = NT * kTinyVT, NW = NT / 32;
  static constexpr size_t ord = (size_t)T * sizeof(K);
  static constexpr size_t ord2 = ord + (size_t)T * 2;
  static constexpr size_t warp = ord2 + (size_t)T * 2;
  static constexpr size_t flag = warp + (size_t)NW * kRadixBins * 4;
  static constexpr size_t spl = flag + (size_t)T;
  static constexpr size_t e = spl + kTinyMaxP * sizeof(K);
  static constexpr size_t bytes = e + (kTinyMaxP + 1) * 4 + 16;
  static_assert(ord % 4 == 0 && warp % 16 == 0 && spl % 8 == 0, "aligned parts");
};

template <typename K, bool V, int NT>
__global__ void __launch_bounds__(NT)
k_radix_tiny(RadixTiny<K> a) {
  pdl_enter();
  using L = TinySmem<K, NT>;
  constexpr int VT = kTinyVT, NW = L::NW, D = (int)sizeof(K);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  K* s_key = reinterpret_cast<K*>(smem_raw);
  uint16_t* s_from = reinterpret_cast<uint16_t*>(smem_raw + L::ord);
  uint16_t* s_to = reinterpret_cast<uint16_t*>(smem_raw + L::ord2);
  uint32_t* s_all = reinterpret_cast<uint32_t*>(smem_raw + L::warp);
  uint8_t* s_flag = smem_raw + L::flag;
  K* s_spl = reinterpret_cast<K*>(smem_raw + L::spl);          // t_b at [b]
  uint32_t* s_e = reinterpret_cast<uint32_t*>(smem_raw + L::e);
  __shared__ uint32_t s_warp[kRadixBins / 32];
  __shared__ uint32_t s_max, s_min;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t n = a.n, P = a.P;
  const uint32_t w0 = warp * 32 * VT + lane;        // position of item 0; item i sits 32 i further
  uint32_t* wc = s_all + warp * kRadixBins;
#pragma unroll
  for (int i = 0; i < VT; ++i) {
    const uint32_t p = w0 + i * 32;
    if (p < n) s_key[p] = to_order<K>(a.kin[p], a.f32);
    s_from[p] = (uint16_t)p;
  }
  if (tid == 0) {
    s_max = 0;
    s_min = 0xFFFFFFFFu;
  }
  // One stable pass by `digit(position)`, from s_from to s_to, pads last;
  // thread d gets the first slot of digit d.
  auto pass = [&](auto digit) -> uint32_t {
#pragma unroll
    for (int i = 0; i < kRadixBins / 32; ++i) wc[i * 32 + lane] = 0;
    __syncthreads();
    uint32_t dig[VT], from[VT];
#pragma unroll
    for (int i = 0; i < VT; ++i) {
      const uint32_t p = w0 + i * 32;
      from[i] = s_from[p];
      dig[i] = p < n ? digit(from[i]) : kRadixBins - 1;
      atomicAdd(&wc[dig[i]], 1u);
    }
    __syncthreads();
    uint32_t slot0 = 0, total;
    if (tid < kRadixBins) digit_starts<NW>(s_all, s_warp, slot0, total);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < VT; ++i) s_to[warp_slot(wc, dig[i])] = (uint16_t)from[i];
    __syncthreads();
    return slot0;
  };
  auto flip = [&]() {
    uint16_t* x = s_from;
    s_from = s_to;
    s_to = x;
  };
#pragma unroll 1
  for (int d = 0; d < D; ++d) {
    pass([&](uint32_t p) { return radix_digit(s_key[p], d); });
    flip();
  }
  const uint16_t* s_ord = s_from;                   // sorted position -> input position
  uint32_t val[V ? VT : 1];
  if (V) {                                          // every payload is read before any is written (in place)
#pragma unroll
    for (int i = 0; i < VT; ++i) {
      const uint32_t j = i * NT + tid;
      if (j < n) val[i] = a.vin[s_ord[j]];
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < VT; ++i) {
    const uint32_t j = i * NT + tid;
    if (j < n) {
      a.kout[j] = from_order<K>(s_key[s_ord[j]], a.f32);
      if (V) a.vout[j] = val[i];
    }
  }
  if (!a.want) return;
  auto key_at = [&](uint32_t j) { return s_key[s_ord[j]]; };
  const uint32_t s = (uint32_t)umin(a.s, 0xFFFFFFFFull);
  auto run_first = [&](uint32_t r) { return (r * n) / P; };             // n P < 2^32
  auto run_of = [&](uint32_t p) { return ((p + 1) * P - 1) / n; };
  if (P > 1) {
    // The list of every run's keys, runs in order: slot run_first(r) + i holds the
    // sorted position of run r's i-th key.  A pass over sorted positions.
    uint16_t* s_list = s_to;
#pragma unroll
    for (int i = 0; i < kRadixBins / 32; ++i) wc[i * 32 + lane] = 0;
    __syncthreads();
    uint32_t dig[VT];
#pragma unroll
    for (int i = 0; i < VT; ++i) {
      const uint32_t j = w0 + i * 32;
      dig[i] = j < n ? run_of(s_ord[j]) : kRadixBins - 1;
      atomicAdd(&wc[dig[i]], 1u);
    }
    __syncthreads();
    if (tid < kRadixBins) {
      uint32_t slot0, total;
      digit_starts<NW>(s_all, s_warp, slot0, total);
    }
    __syncthreads();
    // A key is a sample iff its position in its run is one of the run's sample positions.
#pragma unroll
    for (int i = 0; i < VT; ++i) {
      const uint32_t j = w0 + i * 32, slot = warp_slot(wc, dig[i]);
      s_list[slot] = (uint16_t)j;
      uint8_t flag = 0;
      if (j < n) {
        const uint32_t r0 = run_first(dig[i]), nr = run_first(dig[i] + 1) - r0, x = slot - r0, sr = min(s, nr);
        flag = (uint8_t)(samples_before(x + 1, sr, nr) - samples_before(x, sr, nr));
      }
      s_flag[j] = flag;
    }
    __syncthreads();
    // Splitter t_b is the sample number floor(b S / P) - 1 along the sorted keys.
    const uint32_t S = s >= (n + P - 1) / P ? n : s * P;
    uint32_t mine = 0;
    const uint32_t j0 = tid * VT;                   // blocked: thread t owns [t VT, t VT + VT)
    for (int i = 0; i < VT; ++i) mine += s_flag[j0 + i];
    uint32_t at = (uint32_t)block_exclusive_scan(mine, nullptr);
    for (int i = 0; i < VT; ++i) {
      if (s_flag[j0 + i]) {
        const uint32_t b = (uint32_t)(((uint64_t)(at + 1) * P + S - 1) / S);   // the only b that can fit
        if (b < P && (uint32_t)(((uint64_t)b * S) / P) - 1 == at) s_spl[b] = key_at(j0 + i);
        ++at;
      }
    }
    __syncthreads();
    // e_b by the investigator's rule.
    if (tid > 0 && tid < (int)P) {
      const uint32_t b = tid, target = (b * n) / P;
      const K t = s_spl[b];
      auto lower = [&](uint32_t lo, uint32_t hi) {
        return (uint32_t)partition_point(lo, hi, [&](uint64_t m) { return key_at((uint32_t)m) < t; });
      };
      auto upper = [&](uint32_t lo, uint32_t hi) {
        return (uint32_t)partition_point(lo, hi, [&](uint64_t m) { return key_at((uint32_t)m) <= t; });
      };
      uint32_t eb = target;
      if (a.variant == 1) {
        const uint32_t lo = lower(0, n), up = upper(lo, n);
        const uint64_t g0 = partition_point(1, P, [&](uint64_t m) { return s_spl[m] < t; });
        const uint64_t g1 = partition_point(g0, P, [&](uint64_t m) { return s_spl[m] <= t; });
        eb = lo + (uint32_t)(((uint64_t)(up - lo) * (b - g0 + 1)) / (g1 - g0));
      } else if (a.variant == 2 || key_at(target) > t) {
        eb = upper(0, n);
      } else if (key_at(target) < t) {
        eb = lower(target, n);
      }
      s_e[b] = eb;
      if (a.splitters) a.splitters[b - 1] = from_order<K>(t, a.f32);
    }
    if (tid == 0) {
      s_e[0] = 0;
      s_e[P] = n;
    }
    __syncthreads();
    if (a.cuts) {
      for (uint32_t x = tid; x < P * (P + 1); x += NT) {
        const uint32_t r = x / (P + 1), b = x % (P + 1);
        const uint32_t r0 = run_first(r), r1 = run_first(r + 1), eb = s_e[b];
        a.cuts[x] = partition_point(r0, r1, [&](uint64_t m) { return s_list[m] < eb; }) - r0;
      }
    }
  } else {
    if (tid == 0) {
      s_e[0] = 0;
      s_e[1] = n;
      if (a.cuts) {
        a.cuts[0] = 0;
        a.cuts[1] = n;
      }
    }
    __syncthreads();
  }
  if (a.bounds)
    for (uint32_t b = tid; b <= P; b += NT) a.bounds[b] = s_e[b];
  if (a.stats) {
    for (uint32_t b = tid; b < P; b += NT) {
      const uint32_t size = s_e[b + 1] - s_e[b];
      atomicMax(&s_max, size);
      atomicMin(&s_min, size);
    }
    __syncthreads();
    if (tid == 0) {
      DevStats st{};
      st.n = n;
      st.P = P;
      st.s = s;
      st.max_bucket = s_max;
      st.min_bucket = s_min;
      st.passes = D;
      st.launches = 1;
      st.max_over_mean = (float)((double)s_max * P / (double)n);
      *a.stats = st;
    }
  }
}

}  // namespace pgs
