// Launch sequence of the radix form of the sort (pgs_radix.cuh).
#pragma once

#include "pgs_host.cuh"

namespace pgs {

// Dynamic shared memory of the splitter search for P runs.
inline size_t run_splitters_smem(uint32_t P) { return (size_t)P * 12; }

template <typename K, bool V, typename ID, typename OFF>
using MoveSmem = RadixSmem<K, V, ID, OFF, RadixShape<(int)sizeof(K)>::NT, RadixShape<(int)sizeof(K)>::VT>;

// Keys per thread of the small form's tiles (0: too large a sort): the smallest
// that gives at most 128 tiles, since every tile reads every tile's row of
// counts (171 tiles of 4 keys a thread take 10.9 us a pass, 86 of 8 take 8.4),
// else the largest, up to the tiles that are resident (2 CTAs per SM).
inline int small_vt(const Shape& sh) {
  if (sh.batch) return 0;
  const int most = sh.w == 8 ? kSmallVT8 : kSmallVT4;
  if (ceil_div(sh.n, (uint64_t)kSmallNT * most) > kSmallTiles) return 0;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 0;
  const uint64_t resident = std::min<uint64_t>(kSmallTiles, (uint64_t)sms * kSmallMB);   // a slice of a GPU has fewer
  for (int vt : {4, 8, 12})
    if (ceil_div(sh.n, (uint64_t)kSmallNT * vt) <= std::min<uint64_t>(128, resident)) return vt;
  return ceil_div(sh.n, (uint64_t)kSmallNT * most) <= resident ? most : 0;
}

// Passes of 8-byte keys from this one on are mostly left out (RadixPlan).
constexpr int kLoopPass = 5;
constexpr uint64_t kLoopCtas = 2 * 152;

template <typename K, bool V, typename ID>
inline int set_radix_move_attr(const Shape& sh) {
  auto set = [](auto* kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
  constexpr bool LOOP = sizeof(K) == 8;
  if (sh.n <= 0xFFFFFFFFull) {
    PGS_CUDA(set(k_radix_move<K, V, ID, uint32_t, kFirstPass, false>, MoveSmem<K, V, ID, uint32_t>::bytes));
    PGS_CUDA(set(k_radix_move<K, V, ID, uint32_t, kLaterPass, false>, MoveSmem<K, V, ID, uint32_t>::bytes));
    PGS_CUDA(set(k_radix_move<K, V, ID, uint32_t, kLaterPass, LOOP>, MoveSmem<K, V, ID, uint32_t>::bytes));
  } else {
    PGS_CUDA(set(k_radix_move<K, V, ID, uint64_t, kFirstPass, false>, MoveSmem<K, V, ID, uint64_t>::bytes));
    PGS_CUDA(set(k_radix_move<K, V, ID, uint64_t, kLaterPass, false>, MoveSmem<K, V, ID, uint64_t>::bytes));
    PGS_CUDA(set(k_radix_move<K, V, ID, uint64_t, kLaterPass, LOOP>, MoveSmem<K, V, ID, uint64_t>::bytes));
  }
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
  const RunTables rt{b.rgroups, b.rcnt_off, b.rgpre_off, b.run_cnt, b.run_gpre, sh.rgroup};
  const int f32 = o.dtype == PGS_F32;
  uint64_t* cut = o.cuts && !sh.batch ? b.cut : nullptr;
  PGS_TRY(launch(c, PGS_KERNEL_RUN_COUNTS, 2, 2 * sh.n + 4 * sh.rcnt, [&] {
    klaunch(c.st, c.pdl, k_run_hist, (unsigned)sh.rgroups, kRunHistNT, (size_t)sh.Pmax * 4, ids, g, rt,
            static_cast<const uint32_t*>(b.err));
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

// Whether an output shares memory with an input: keys and payloads may each be
// sorted in place, with the other one or not.
template <typename K>
bool outputs_on_inputs(uint64_t n, const K* kin, const uint32_t* vin, const K* kout, const uint32_t* vout) {
  auto meet = [n](const void* a, size_t aw, const void* b, size_t bw) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return a && b && x < y + n * bw && y < x + n * aw;
  };
  return meet(kin, sizeof(K), kout, sizeof(K)) || meet(vin, 4, vout, 4) || meet(kin, sizeof(K), vout, 4) ||
         meet(vin, 4, kout, sizeof(K));
}

// The order below the passes' bytes.
template <bool V, bool RUN>
int radix_finish(const Shape& sh, const Options& o, uint64_t* kout, uint32_t* vout, bool even, Ctx& c,
                 const Buffers& b) {
  RadixFinish f{};
  f.keys = kout;
  f.vals = vout;
  f.tags = reinterpret_cast<uint16_t*>(b.tag_b);
  f.kalt = static_cast<uint64_t*>(b.alt_k);
  f.valt = b.alt_v;
  f.talt = reinterpret_cast<uint16_t*>(b.tag_a);
  f.tiles = b.rtiles;
  f.koff = b.koff;
  f.plan = static_cast<RadixPlan*>(b.plan);
  f.segs = static_cast<RadixSeg*>(b.segs);
  f.cap = sh.seg_cap();
  f.bits = b.seg_bits;
  f.listed = b.seg_bits + sh.seg_words();
  f.most = sh.batch ? f.listed + 1 : nullptr;
  f.passes = f.listed + 2;
  f.even = even;
  f.rows = b.seg_rows;
  f.err = b.err;
  f.barrier = b.err + 4;
  f.n = sh.n;
  f.wait_ns = o.spin_limit;
  f.fault = o.fault_inject == PGS_FAULT_RADIX_BARRIER;
  PGS_CUDA(cudaFuncSetAttribute(k_radix_finish<V, RUN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kFinishSmem));
  PGS_TRY(launch(c, PGS_KERNEL_RADIX_MOVE, 1, 8 * sh.n, [&] {
    klaunch(c.st, c.pdl, k_radix_finish<V, RUN>, (unsigned)sh.rtiles, kFinishNT, kFinishSmem, f);
  }));
  int dev = 0, sms = 0;
  PGS_CUDA(cudaGetDevice(&dev));
  PGS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  return launch(c, PGS_KERNEL_RADIX_MOVE, 1, 0, [&] {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = (unsigned)std::min(kRedoCtas, sms);
    cfg.blockDim = kRedoNT;
    cfg.stream = c.st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_radix_redo<V, RUN>, f);
  });
}

// The passes, least significant byte first.  Tags change buffers with the keys;
// the last pass leaves the runs in tag_b.
template <typename K, bool V, typename ID, typename OFF>
int radix_passes(const Shape& sh, const Options& o, const K* kin, const uint32_t* vin, K* kout, uint32_t* vout,
                 Ctx& c, const Buffers& b) {
  using L = MoveSmem<K, V, ID, OFF>;
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
  a.ntiles = sh.rtiles;
  uint32_t* most = nullptr;
  a.even = outputs_on_inputs(sh.n, kin, vin, kout, vout);
  a.wait_ns = o.spin_limit;
  a.chunk_tiles = (uint32_t)sh.rchunk_tiles;
  if constexpr (D == 8) {                               // the bytes and buffers of a pass follow on the device
    a.plan = static_cast<RadixPlan*>(b.plan);
    a.kin = kin;
    a.vin = vin;
    a.kout = kout;
    a.vout = vout;
    a.kalt = alt_k;
    a.valt = b.alt_v;
    a.tag_a = b.tag_a;
    a.tag_b = b.tag_b;
    most = b.seg_bits + sh.seg_words() + 1;
    if (sh.batch) a.most = most;
    PGS_CUDA(cudaFuncSetAttribute(k_radix_plan, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPickSmem));
    PGS_TRY(launch(c, PGS_KERNEL_SAMPLE, 1, (uint64_t)sh.I * kPlanKeys * 8, [&] {
      klaunch(c.st, c.pdl, k_radix_plan, sh.I, kPickNT, kPickSmem, reinterpret_cast<const uint64_t*>(kin), b.koff, a.plan,
              b.seg_bits, sh.seg_words() + 2);
    }));
  }
  for (int d = 0; d < D; ++d) {
    const bool to_out = (D - 1 - d) % 2 == 0;           // the last pass lands in the caller's output
    a.ksrc = d == 0 ? kin : to_out ? alt_k : kout;
    a.vsrc = d == 0 ? vin : to_out ? b.alt_v : vout;
    a.tsrc = d == 0 || ID::bytes == 0 ? nullptr : d % 2 ? b.tag_a : b.tag_b;
    a.kdst = to_out ? kout : alt_k;
    a.vdst = to_out ? vout : b.alt_v;
    a.tdst = d % 2 ? b.tag_b : b.tag_a;
    a.byte = d;
    a.next = d + 1;
    a.pass = d;
    a.f32_in = d == 0 ? f32 : 0;
    a.f32_out = d == D - 1 ? f32 : 0;
    a.last = d == D - 1;
    a.fault = d == 0 && o.fault_inject == PGS_FAULT_RADIX_COPIES;
    const bool tags = ID::digit && d > 0;
    PGS_TRY(launch(c, PGS_KERNEL_RADIX_COUNT, 1, sh.n * (tags ? ID::bytes : (int)sizeof(K)), [&] {
      if (tags)
        klaunch(c.st, c.pdl, k_radix_count<K, ID, ID::digit>, (unsigned)sh.rchunks, kCountNT, 0, a);
      else
        klaunch(c.st, c.pdl, k_radix_count<K, ID, false>, (unsigned)sh.rchunks, kCountNT, 0, a);
    }));
    PGS_TRY(launch(c, PGS_KERNEL_SCAN, 1, 16 * sh.rchunks * kRadixBins, [&] {
      if (sh.batch)
        klaunch(c.st, c.pdl, k_radix_scan_batch, sh.I, kRadixBins, 0, b.rpre, b.rtotal, b.rfirst, a.plan, d, a.even, most);
      else
        klaunch(c.st, c.pdl, k_radix_scan_wide, kRadixBins / 8, 1024, 0, b.rpre, b.rtotal, (uint32_t)sh.rchunks, a.plan, d,
                a.even);
    }));
    PGS_TRY(launch(c, PGS_KERNEL_RADIX_MOVE, 1, 2 * sh.n * (sizeof(K) + (V ? 4 : 0) + ID::bytes), [&] {
      if (d == 0)
        klaunch(c.st, c.pdl, k_radix_move<K, V, ID, OFF, kFirstPass, false>, (unsigned)sh.rtiles, L::NT, L::bytes, a);
      else if (D == 8 && d >= kLoopPass)
        klaunch(c.st, c.pdl, k_radix_move<K, V, ID, OFF, kLaterPass, D == 8>,
                (unsigned)std::min<uint64_t>(sh.rtiles, kLoopCtas), L::NT, L::bytes, a);
      else
        klaunch(c.st, c.pdl, k_radix_move<K, V, ID, OFF, kLaterPass, false>, (unsigned)sh.rtiles, L::NT, L::bytes, a);
    }));
  }
  if constexpr (D == 8) return radix_finish<V, ID::run>(sh, o, reinterpret_cast<uint64_t*>(kout), vout, a.even, c, b);
  return PGS_OK;
}

// Every pass of a small sort in one cooperative launch.
template <typename K, bool V, typename ID, int VT>
int radix_small(const Shape& sh, const Options& o, const K* kin, const uint32_t* vin, K* kout, uint32_t* vout, Ctx& c,
                const Buffers& b) {
  using L = RadixSmem<K, V, ID, uint32_t, kSmallNT, VT>;
  static_assert((L::bytes + 4096) * kSmallMB <= 227 * 1024, "the tiles of a small sort are resident");
  PGS_CUDA(cudaFuncSetAttribute(k_radix_small<K, V, ID, VT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)L::bytes));
  RadixSmall<K> p{};
  p.pass.ksrc = kin;
  p.pass.vsrc = vin;
  p.pass.koff = b.koff;
  p.pass.P = b.Pt;
  p.pass.err = b.err;
  p.pass.n = sh.n;
  p.pass.wait_ns = o.spin_limit;
  p.pass.even = outputs_on_inputs(sh.n, kin, vin, kout, vout);
  p.kout = kout;
  p.vout = vout;
  p.kalt = static_cast<K*>(b.alt_k);
  p.valt = b.alt_v;
  p.tag_a = b.tag_a;
  p.tag_b = b.tag_b;
  p.rows = b.rrows;
  p.barrier = b.err + 1;
  p.diff = reinterpret_cast<uint64_t*>(b.err + 2);
  p.plan = static_cast<RadixPlan*>(b.plan);
  p.bits = b.seg_bits;
  p.words = (uint32_t)(sh.seg_words() + 2);
  p.f32 = o.dtype == PGS_F32;
  p.pass.fault = o.fault_inject == PGS_FAULT_RADIX_COPIES;
  p.fault = o.fault_inject == PGS_FAULT_RADIX_BARRIER;
  const unsigned tiles = (unsigned)ceil_div(sh.n, (uint64_t)L::T);
  PGS_TRY(launch(c, PGS_KERNEL_RADIX_MOVE, 1, 2 * sh.n * sizeof(K) * (sizeof(K) + (V ? 4 : 0) + ID::bytes), [&] {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = tiles;
    cfg.blockDim = kSmallNT;
    cfg.dynamicSmemBytes = L::bytes;
    cfg.stream = c.st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_radix_small<K, V, ID, VT>, p);
  }));
  if constexpr (sizeof(K) == 8) return radix_finish<V, ID::run>(sh, o, reinterpret_cast<uint64_t*>(kout), vout, p.pass.even, c, b);
  return PGS_OK;
}

template <typename K, bool V, typename ID>
int radix_passes(const Shape& sh, const Options& o, const K* kin, const uint32_t* vin, K* kout, uint32_t* vout,
                 Ctx& c, const Buffers& b) {
  switch (small_vt(sh)) {
    case 4: return radix_small<K, V, ID, 4>(sh, o, kin, vin, kout, vout, c, b);
    case 8: return radix_small<K, V, ID, 8>(sh, o, kin, vin, kout, vout, c, b);
    case 12: return radix_small<K, V, ID, 12>(sh, o, kin, vin, kout, vout, c, b);
    case 0: break;
    default: return radix_small<K, V, ID, sizeof(K) == 8 ? kSmallVT8 : kSmallVT4>(sh, o, kin, vin, kout, vout, c, b);
  }
  if (sh.n <= 0xFFFFFFFFull) return radix_passes<K, V, ID, uint32_t>(sh, o, kin, vin, kout, vout, c, b);
  return radix_passes<K, V, ID, uint64_t>(sh, o, kin, vin, kout, vout, c, b);
}

// A tiny sort, the whole call in one launch.
template <typename K, bool V, int NT>
int radix_tiny(const Shape& sh, const Options& o, const K* kin, const uint32_t* vin, K* kout, uint32_t* vout, Ctx& c) {
  using L = TinySmem<K, NT>;
  PGS_CUDA(cudaFuncSetAttribute(k_radix_tiny<K, V, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes));
  RadixTiny<K> a{};
  a.kin = kin;
  a.vin = vin;
  a.kout = kout;
  a.vout = vout;
  a.bounds = o.bucket_bounds;
  a.cuts = o.cuts;
  a.splitters = static_cast<K*>(o.splitters);
  a.stats = static_cast<DevStats*>(o.stats);
  a.s = sh.s;
  a.n = (uint32_t)sh.n;
  a.P = sh.R;
  a.f32 = o.dtype == PGS_F32;
  a.variant = o.investigator;
  a.want = o.bucket_bounds || o.cuts || o.splitters || o.stats;
  return launch(c, PGS_KERNEL_RADIX_MOVE, 1, 2 * sh.n * (sizeof(K) + (V ? 4 : 0)), [&] {
    klaunch(c.st, c.pdl, k_radix_tiny<K, V, NT>, 1, NT, L::bytes, a);
  });
}

template <typename K, bool V>
int run_radix(const Shape& sh, const Options& o, const K* kin, const uint32_t* vin, K* kout, uint32_t* vout, Ctx& c,
              const Buffers& b) {
  cudaStream_t st = c.st;
  c.pdl = sh.n <= kPdlMaxKeys;
  const Geo g = b.geo(sh);
  PGS_CUDA(cudaMemsetAsync(b.err, 0, kErrWords * sizeof(uint32_t), st));
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
            b.learned_ratio, static_cast<DevStats*>(o.stats), o.bucket_bounds, b.max_ratio, sh.w == 8 ? b.seg_bits + sh.seg_words() + 2 : nullptr);
  });
}

}  // namespace pgs
