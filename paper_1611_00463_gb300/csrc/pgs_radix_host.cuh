// Launch sequence of the radix form of the sort (pgs_radix.cuh), and the rule
// that picks it.
#pragma once

#include "pgs_host.cuh"

namespace pgs {

// Sorts from these sizes run the radix form whatever P is.  Its time hardly
// depends on P, the merge pipeline's does (the bucket rounds plan P^2
// segments): at P = 16 they meet near 2^19 keys of 4 bytes (107 against 109
// us) and 2^22 keys of 8 (403 against 393 us; 651 against 733 at 2^23), at
// P = 300 the radix form takes 111 against 479 us at 2^16 keys of 4 bytes and
// 162 against 528 us of 8.
constexpr uint64_t kRadixMinKeys4 = 1ull << 19;
constexpr uint64_t kRadixMinKeys8 = 1ull << 22;
constexpr uint32_t kRadixMinP = 65;
// A batch needs tiles filled to this share: 2000 instances of 4266 keys on
// average take 354 against 440 us (4 bytes) and 730 against 590 us (8 bytes),
// of 1876 keys 265 against 231 and 520 against 297 us, of 12,288 keys (200
// instances) 105 against 200 and 228 against 241 us.
constexpr double kRadixMinFill4 = 0.4, kRadixMinFill8 = 0.6;

// Calls that run the radix form.  Asking for a merge width, a merge tile shape,
// an exchange or the merge kernels' fault injection asks for the merge
// pipeline; the LOCAL investigator's order is not the stable sort; a learned
// model is trained on and evaluated over sorted runs (beyond kLearnedMaxP
// partitions no model is trained and the sampled cuts stand).
inline bool use_radix(const Shape& sh, const Options& o) {
  if (!sh.radix || o.merge_ways != 0 || o.tile_variant != 0 || o.exchange != PGS_EXCHANGE_AUTO ||
      o.fault_inject != 0 || o.investigator == PGS_INVESTIGATOR_LOCAL)
    return false;
  if (sh.learned && (o.model || sh.R <= kLearnedMaxP)) return false;
  if (sh.batch) {
    const double fill = (double)sh.n / ((double)sh.rtiles * radix_tile(sh.w));
    return fill >= (sh.w == 8 ? kRadixMinFill8 : kRadixMinFill4);
  }
  return sh.R >= kRadixMinP || sh.n >= (sh.w == 8 ? kRadixMinKeys8 : kRadixMinKeys4);
}

// Dynamic shared memory of the splitter search for P runs.
inline size_t run_splitters_smem(uint32_t P) { return (size_t)P * 12; }

template <typename K, bool V, typename ID>
inline int set_radix_move_attr(const Shape& sh) {
  if (sh.n <= 0xFFFFFFFFull)
    PGS_CUDA(cudaFuncSetAttribute(k_radix_move<K, V, ID, uint32_t>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)RadixSmem<K, V, ID, uint32_t>::bytes));
  else
    PGS_CUDA(cudaFuncSetAttribute(k_radix_move<K, V, ID, uint64_t>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)RadixSmem<K, V, ID, uint64_t>::bytes));
  return PGS_OK;
}

// Tags of a sort whose results do not depend on the runs.
template <typename K> using NoRun = typename std::conditional<sizeof(K) == 8, Dig, None>::type;

// Opt in to more than 48 KB of dynamic shared memory (set on every call, as
// set_smem_attrs does).
template <typename K, bool V>
inline int set_radix_attrs(const Shape& sh) {
  PGS_TRY((set_radix_move_attr<K, V, NoRun<K>>(sh)));
  if (sh.Pmax == 1) return PGS_OK;
  if (sh.Pmax <= 256) PGS_TRY((set_radix_move_attr<K, V, Id8>(sh)));
  else PGS_TRY((set_radix_move_attr<K, V, Id16>(sh)));
  PGS_CUDA(cudaFuncSetAttribute(k_run_splitters<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)run_splitters_smem(kMaxP)));
  return PGS_OK;
}

// Steps 2-4 on the sorted keys and run ids.
template <typename K>
int radix_cuts(const Shape& sh, const Options& o, const K* kout, const uint16_t* ids, Ctx& c, const Buffers& b) {
  const Geo g = b.geo(sh);
  const RunTables rt{b.rgroups, b.rcnt_off, b.rgpre_off, b.run_cnt, b.run_gpre};
  const int f32 = o.dtype == PGS_F32;
  uint64_t* cut = o.cuts && !sh.batch ? b.cut : nullptr;
  PGS_TRY(launch(c, PGS_KERNEL_RUN_COUNTS, 2, 2 * sh.n + 4 * sh.rcnt, [&] {
    klaunch(c.st, c.pdl, k_run_hist, (unsigned)sh.rgroups, kRunHistNT, (size_t)sh.Pmax * 4, ids, g, rt);
  }));
  PGS_TRY(launch(c, PGS_KERNEL_SCAN, 2, 16 * sh.rgpre, [&] {
    klaunch(c.st, c.pdl, k_run_scan, dim3(sh.I, (unsigned)ceil_div(sh.Pmax, 32)), 1024, 0, g, rt);
  }));
  PGS_TRY(launch(c, PGS_KERNEL_SPLITTERS, 3, 8 * sh.MAT, [&] {
    klaunch(c.st, c.pdl, k_run_splitters<K>, sh.R, kFindNT, run_splitters_smem(sh.Pmax), kout, ids, g, rt, f32,
            o.investigator, static_cast<K*>(b.spl), static_cast<K*>(o.splitters), cut, b.e, b.err);
  }));
  if (o.investigator == PGS_INVESTIGATOR_EQUAL)
    PGS_TRY(launch(c, PGS_KERNEL_INVESTIGATOR, 4, 8 * sh.MAT, [&] {
      klaunch(c.st, c.pdl, k_run_cuts_equal<K>, sh.R, kFindNT, (size_t)sh.Pmax * 4, kout, ids, g, rt, f32,
              static_cast<const K*>(b.spl), cut, b.e, b.err);
    }));
  return PGS_OK;
}

// The passes, least significant byte first.  Tags change buffers with the keys;
// the last pass leaves the runs in tag_b.
template <typename K, bool V, typename ID, typename OFF>
int radix_passes(const Shape& sh, const Options& o, const K* kin, const uint32_t* vin, K* kout, uint32_t* vout,
                 Ctx& c, const Buffers& b) {
  using L = RadixSmem<K, V, ID, OFF>;
  constexpr int D = (int)sizeof(K);
  const int f32 = o.dtype == PGS_F32;
  K* alt_k = static_cast<K*>(b.alt_k);
  RadixPass<K> a{};
  a.cnt = b.rcnt;
  a.pre = b.rpre;
  a.total = b.rtotal;
  a.tiles = b.rtiles;
  a.chunks = b.rchunks;
  a.koff = b.koff;
  a.P = b.Pt;
  a.err = b.err;
  a.n = sh.n;
  a.wait_ns = o.spin_limit;
  a.chunk_tiles = (uint32_t)sh.rchunk_tiles;
  for (int d = 0; d < D; ++d) {
    const bool to_out = (D - 1 - d) % 2 == 0;           // the last pass lands in the caller's output
    a.ksrc = d == 0 ? kin : to_out ? alt_k : kout;
    a.vsrc = d == 0 ? vin : to_out ? b.alt_v : vout;
    a.tsrc = d == 0 || ID::bytes == 0 ? nullptr : d % 2 ? b.tag_a : b.tag_b;
    a.kdst = to_out ? kout : alt_k;
    a.vdst = to_out ? vout : b.alt_v;
    a.tdst = d % 2 ? b.tag_b : b.tag_a;
    a.byte = d;
    a.f32_in = d == 0 ? f32 : 0;
    a.f32_out = d == D - 1 ? f32 : 0;
    a.last = d == D - 1;
    const bool tags = ID::digit && d > 0;
    PGS_TRY(launch(c, PGS_KERNEL_RADIX_COUNT, 1, sh.n * (tags ? ID::bytes : (int)sizeof(K)), [&] {
      if (tags)
        klaunch(c.st, c.pdl, k_radix_count<K, ID, ID::digit>, (unsigned)sh.rchunks, kCountNT, 0, a);
      else
        klaunch(c.st, c.pdl, k_radix_count<K, ID, false>, (unsigned)sh.rchunks, kCountNT, 0, a);
    }));
    PGS_TRY(launch(c, PGS_KERNEL_SCAN, 1, 16 * sh.rchunks * kRadixBins, [&] {
      if (sh.batch)
        klaunch(c.st, c.pdl, k_radix_scan_batch, sh.I, kRadixBins, 0, b.rpre, b.rtotal, b.rfirst);
      else
        klaunch(c.st, c.pdl, k_radix_scan_wide, kRadixBins / 8, 1024, 0, b.rpre, b.rtotal, sh.rchunks);
    }));
    PGS_TRY(launch(c, PGS_KERNEL_RADIX_MOVE, 1, 2 * sh.n * (sizeof(K) + (V ? 4 : 0) + ID::bytes), [&] {
      klaunch(c.st, c.pdl, k_radix_move<K, V, ID, OFF>, (unsigned)sh.rtiles, L::NT, L::bytes, a);
    }));
  }
  return PGS_OK;
}

template <typename K, bool V, typename ID>
int radix_passes(const Shape& sh, const Options& o, const K* kin, const uint32_t* vin, K* kout, uint32_t* vout,
                 Ctx& c, const Buffers& b) {
  if (sh.n <= 0xFFFFFFFFull) return radix_passes<K, V, ID, uint32_t>(sh, o, kin, vin, kout, vout, c, b);
  return radix_passes<K, V, ID, uint64_t>(sh, o, kin, vin, kout, vout, c, b);
}

template <typename K, bool V>
int run_radix(const Shape& sh, const Options& o, const K* kin, const uint32_t* vin, K* kout, uint32_t* vout, Ctx& c,
              const Buffers& b) {
  cudaStream_t st = c.st;
  c.pdl = sh.n <= kPdlMaxKeys;
  const Geo g = b.geo(sh);
  PGS_CUDA(cudaMemsetAsync(b.err, 0, sizeof(uint32_t), st));
  // The runs matter only to what is read off the sorted order.
  const bool bounds = o.stats || (!sh.batch && (o.bucket_bounds || o.cuts || o.splitters));
  if (!bounds || sh.Pmax == 1)
    PGS_TRY((radix_passes<K, V, NoRun<K>>(sh, o, kin, vin, kout, vout, c, b)));
  else if (sh.Pmax <= 256)
    PGS_TRY((radix_passes<K, V, Id8>(sh, o, kin, vin, kout, vout, c, b)));
  else
    PGS_TRY((radix_passes<K, V, Id16>(sh, o, kin, vin, kout, vout, c, b)));
  if (bounds && sh.Pmax > 1)
    PGS_TRY((radix_cuts<K>(sh, o, kout, reinterpret_cast<const uint16_t*>(b.tag_b), c, b)));
  else if (bounds)
    PGS_TRY(launch(c, PGS_KERNEL_INVESTIGATOR, 4, 24 * (uint64_t)sh.R, [&] {
      klaunch(st, c.pdl, k_cut_edges, grid_for(sh.R, 256), 256, 0, g, sh.batch ? nullptr : b.cut, b.e);
    }));
  if (sh.learned)
    PGS_TRY(launch(c, PGS_KERNEL_SPLITTERS, 3, 8, [&] {
      klaunch(st, c.pdl, k_learned_skip, 1, 256, 0, b.fallback, b.learned_ratio, o.model_out);
    }));
  if (!bounds) return PGS_OK;
  if (o.cuts && sh.I == 1)
    PGS_CUDA(cudaMemcpyAsync(o.cuts, b.cut, sizeof(uint64_t) * sh.MAT, cudaMemcpyDeviceToDevice, st));
  const uint32_t launches = c.launches + 1;             // including the statistics kernel
  return launch(c, PGS_KERNEL_STATS, 0, 8 * ((uint64_t)sh.R + sh.I), [&] {
    klaunch(st, c.pdl, k_stats, 1, 256, 0, g, b.e, sh.n, (uint32_t)std::min<uint64_t>(sh.s, 0xFFFFFFFFu),
            sh.learned ? PGS_SPLITTERS_LEARNED : PGS_SPLITTERS_SAMPLED, (uint32_t)sizeof(K), launches, b.err, b.fallback,
            b.learned_ratio, static_cast<DevStats*>(o.stats), o.bucket_bounds, b.max_ratio);
  });
}

}  // namespace pgs
