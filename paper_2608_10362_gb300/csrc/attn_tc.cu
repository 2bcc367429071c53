// attn_tc.cu - attention of many query vectors per KV head (batched verify, prefill,
// GQA) on tcgen05: one CTA, or a cluster that shares the keys, per (request, KV head,
// row block).
//
// On mma.sync (attn_body.cuh) the launch was bound by instruction issue with 64 vectors
// a CTA, blocks of 8 vectors re-read a head's keys once per block, and one CTA combined
// its unit's splits.  Here the vectors of a unit (heads of the KV head x rows, at most
// 128) are the 128 rows of an MMA:
//   S = Q K^T    A = Q (shared memory), B = a tile of 128 keys as TMA left it
//   O += P V     A = P (tensor memory, over S), B = the V tile, N-major
// P in two bf16 planes (hi + lo), Q in three, S and O fp32 in tensor memory.  (The lo
// plane's rounding of Q is most of the error that two planes leave, and the tensor core's
// chain of 8 sums at hd 128 added 1-4% to it; with three the output's error against 64
// bits is 3.2e-6 to 4.6e-6 where mma.sync's two planes had 4.3e-6 to 6.7e-6, hd 64 and
// 128, 300 to 3000 keys.)  A thread owns an MMA
// row, so the softmax has no cross-lane step; its running max only follows a tile's
// when that is more than 2^8 larger (exact: every use of it cancels), which leaves
// rescaling O to a few tiles (as published for FlashAttention-4; two softmax groups
// that alternate, below: FlashAttention-3).  Units of fewer vectors repeat them: with kKG = 64 (32)
// keys per thread the 128 rows are 2 (4) copies of up to 64 (32) vectors, copy j takes
// keys [j kKG, (j + 1) kKG) of each tile and has zeros for the others in P.
// Two softmax warpgroups take the even and the odd tiles, each with its own S, O, max
// and sum, so that one's softmax runs during the other's MMAs.  At the end the CTA's
// partial rows (2 warpgroups x copies) are reduced in shared memory, the cluster's over
// distributed shared memory, each CTA finishing a share of the vectors; sums run in
// ascending order of warpgroup, copy and CTA.
//
// Measured (GB300; us per launch in its pass, the mma.sync kernel / now): 8B target, 16
// requests x 9 rows, 512..4096 keys 101 / 45 (a tile of 128 keys takes 1.55, 2560 cycles
// of it MMAs, 152 SMs' share of HBM allows 1.5; the longest request's CTAs set the
// time); 7B target, 256 prefill rows at up to 2048 keys 26 (128 rows: 72 / 24); 7B, 5
// rows at 2048 keys 15.5 / 11.5.  Passes: 8B verify 7.15 / 5.63 ms, 7B verify 2.71 /
// 2.66, 1.1B verify of 6 rows 0.820 / 0.804, 160M draft of 4 tokens 1.27 / 1.205.
// Code that each launch fetches anew costs as much as it computes: with 128 keys
// unrolled and no dry run a prefill launch took 39, a first tile alone 10.
// Tried instead: the planes of P in the two copies' rows, which saves half of P V's MMAs
// but gives every thread 128 keys: 0.34 ms more for the 8B verify; P V of two tiles and
// then S of two (8B verify 5.85 ms); the tiles of all units dealt to one CTA per SM in
// equal runs, units in several CTAs finished by the last to arrive: 8B at 512..4096 keys
// 1.551 -> 1.548 ms in 8 layers, but at 16 x 3000 keys 1.513 -> 1.572 (a segment costs 5
// us besides its tiles), parts of units as CTAs of their own in order of size 1.573 ->
// 1.604.
//
// Roles (384 threads): warps 0-3, 4-7 softmax, 8 copies, 9 MMAs of S, 11 of P V; warp 10 runs the softmax
// code and the reduction once, dry (no store, no barrier), while the others wait for their
// predecessor and the first tiles: code that each launch fetches anew.  K and V tiles pass
// through one ring in the order of their use: K0 K1 V0 K2 V1 ...  Every wait is bounded.
#include <cuda_bf16.h>

#include <type_traits>

#include "internal.h"
#include "ptx.cuh"

namespace memspec {

namespace {

constexpr int kThreads = 384;
constexpr int kTile = 128;        // keys per tile
constexpr int kRows = 128;        // MMA rows
constexpr int kMaxSlots = 8;
constexpr int kQPlanes = 3;       // bf16 planes of Q

template <int HD>
struct Cfg {
  static constexpr int kSlotBytes = kTile * HD * 2;
  static constexpr int kPlaneBytes = kRows * HD * 2;
  static constexpr int kSlots = HD == 128 ? 4 : 8;
  static constexpr int kSmem = 1024 + kSlots * kSlotBytes + kQPlanes * kPlaneBytes;
  // the partial rows of both warpgroups reuse the ring
  static_assert(kSlots * kSlotBytes >= 2 * kRows * HD * 4, "reduction buffer");
};

struct Ctl {
  uint64_t full[kMaxSlots], empty[kMaxSlots];
  uint64_t q_full;
  uint64_t s_full[2];    // S of the warpgroup's tile is complete
  uint64_t p_full[2];    // ... its P is written (4 warps)
  uint64_t o_full[2];    // ... its P V is complete
  uint64_t drain[2];
  uint32_t tmem_base;
  int abort_flag;
  int at[kRows];         // vector -> its offset in q and out, in heads
};

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
  const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&t);
}
// the two floats of a bf16 pair
__device__ __forceinline__ float2 unpack2(uint32_t x) {
  return make_float2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u));
}

// 32 TMEM lanes x n consecutive 32-bit columns, one lane per thread: load (and wait) ...
__device__ __forceinline__ void tmem_ld_x32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {"
      "%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
// ... and store (tmem_st_wait completes it).
__device__ __forceinline__ void tmem_st_x32(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {"
      "%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 3-D box (64 columns, 128 rows, hd / 64 halves)
__device__ __forceinline__ void tma_load_3d(void* smem_dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar,
                                            uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(smem_addr(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar)), "l"(policy)
      : "memory");
}

// D[tmem] (+)= A[tmem] * B[smem], issued by one thread.
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
__device__ __forceinline__ float2 ld_cluster_f2(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}

__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); }

// Index (floats) of features d..d+3 of partial row r: 16-byte chunks rotated by the
// row, so that 32 threads storing one row each meet no bank conflicts.
template <int HD>
__device__ __forceinline__ int red_at(int r, int d) {
  return r * HD + ((((d >> 2) ^ r) & 7) << 2) + (d & ~31);
}

template <int HD, int KG>
__global__ void __launch_bounds__(kThreads, 1) attn_tc_kernel(const __grid_constant__ AttnArgs a) {
  using C = Cfg<HD>;
  constexpr int kNS = C::kSlots;
  constexpr int kVR = KG;                 // vectors per copy (rows of the copy)
  constexpr int kCopies = kRows / kVR;
  constexpr uint32_t kO = 256;            // TMEM: S of the two warpgroups, then their O
  constexpr uint32_t kTmemCols = 512;
  __shared__ Ctl ctl;
  extern __shared__ uint8_t dsmem_raw[];
  uint8_t* ring = dsmem_raw + ((1024u - (smem_addr(dsmem_raw) & 1023u)) & 1023u);
  uint8_t* qs = ring + kNS * C::kSlotBytes;
  // once every MMA has completed, where Q was: (max, sum) of each partial row
  // [2][kRows], then of each vector in this CTA
  float2* ml = reinterpret_cast<float2*>(qs);
  float2* cml = ml + 2 * kRows;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int lin = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  unsigned long long* trace = a.trace != nullptr && lin < a.trace_ctas ? a.trace + lin * 16 : nullptr;
  if (threadIdx.x == 0) {
    trace_at(trace, 0);
    for (int s = 0; s < kNS; ++s) {
      mbar_init(&ctl.full[s], 1);
      mbar_init(&ctl.empty[s], 1);
    }
    mbar_init(&ctl.q_full, 256);
    for (int w = 0; w < 2; ++w) {
      mbar_init(&ctl.s_full[w], 1);
      mbar_init(&ctl.p_full[w], 4);
      mbar_init(&ctl.o_full[w], 1);
    }
    mbar_init(&ctl.drain[0], 1);
    mbar_init(&ctl.drain[1], 1);
    ctl.abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 9) {
    tmem_alloc(&ctl.tmem_base, kTmemCols);
    tmem_relinquish();
  }
  if (threadIdx.x == 256) {
    tma_prefetch_desc(&a.kmap);
    tma_prefetch_desc(&a.vmap);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctl.tmem_base;
  volatile int* abort_flag = &ctl.abort_flag;
  const bool dry = warp == 10, soft = warp < 8 || dry;

  const bool early = a.ctx_early != 0;
  if (!early) pdl_wait();
  const RowPlan* plan = a.plan;
  const int g = blockIdx.z, split = blockIdx.x, n_cta = gridDim.x;
  const int kvh = blockIdx.y / a.row_blocks, rb = blockIdx.y - kvh * a.row_blocks;
  const int n_groups = plan->n_groups, R = plan->rows_per_group, req = plan->req[g], valid = plan->valid[g];
  const int pos0 = plan->pos0[g], tree = plan->tree;
  const int r_lo = rb * a.rows_per_block;
  const int nr = min(r_lo + a.rows_per_block, valid) - r_lo;
  const int gs = a.H / a.Hkv;
  const int nq = gs * nr;
  const int kmax = pos0 + r_lo + nr - 1;
  bool work = g < n_groups && nr > 0;   // the same in every CTA of the cluster
  if (work && (pos0 < 0 || kmax >= a.max_seq || gs > 64 || nq > kVR)) {   // reported, never read
    if (threadIdx.x == 0 && split == 0) atomicOr(a.status, 0x4u);
    work = false;
  }
  // the tiles of keys 0..kmax, spread evenly over the cluster
  const int all_tiles = kmax / kTile + 1;
  const int per_cta = (all_tiles + n_cta - 1) / n_cta;
  const int n_active = work ? (all_tiles + per_cta - 1) / per_cta : 0;
  const int k0 = split * per_cta * kTile;
  const int n = work ? max(0, min(per_cta, all_tiles - split * per_cta)) : 0;   // this CTA's tiles
  const int k1 = min(k0 + n * kTile, kmax + 1);

  if (warp == 8) {
    // ------------------------------------------------ copies
    if (lane == 0) {
      const uint64_t pol = l2_policy_evict_first();
      const int row0 = (req * a.Hkv + kvh) * a.max_seq + k0;
      const int loads = 2 * n;
      // load i: K0, then K(t + 1) and V(t) in turn, last V(n - 1)
      auto is_v = [&](int i) { return i == loads - 1 || (i > 0 && (i & 1) == 0); };
      auto tile_of = [&](int i) { return i == loads - 1 ? n - 1 : is_v(i) ? i / 2 - 1 : (i + 1) / 2; };
      auto load = [&](int i, int s) {
        mbar_arrive_expect_tx(&ctl.full[s], C::kSlotBytes);
        tma_load_3d(ring + s * C::kSlotBytes, is_v(i) ? &a.vmap : &a.kmap, 0, row0 + tile_of(i) * kTile, 0,
                    &ctl.full[s], pol);
      };
      int i = 0;
      if (early) {   // tiles of cached keys alone
        for (; i < loads && i < kNS && k0 + (tile_of(i) + 1) * kTile <= pos0; ++i) load(i, i);
        pdl_wait();
      }
      pdl_launch_dependents();   // after the wait: see ptx.cuh
      trace_at(trace, 13);
      bool ok = true;
      for (; i < loads; ++i) {
        const int s = i % kNS;
        if (i >= kNS && !mbar_wait_bounded(&ctl.empty[s], static_cast<uint32_t>(i / kNS - 1) & 1u, abort_flag, a.status)) {
          ok = false;
          break;
        }
        load(i, s);
      }
      // the CTA leaves when the last MMAs have signalled their slots; after a wait that ran
      // out, when no copy is in flight
      for (int j = max(0, i - kNS); j < i; ++j)
        mbar_wait_drain(ok ? &ctl.empty[j % kNS] : &ctl.full[j % kNS], static_cast<uint32_t>(j / kNS) & 1u);
    }
    __syncwarp();
  } else if (warp == 9 || warp == 11) {
    // ------------------------------------------------ MMAs: warp 9 S, warp 11 P V.  The warps
    // stay converged, one lane issues.  A tcgen05 fence after a wait holds a thread until
    // its own earlier MMAs have completed (470 cycles of a drained pipe, measured): hence two
    // threads, and none after the waits for copies, which need none
    const bool lead = elect_one();
    bool ok = n > 0;
    auto wait = [&](uint64_t* bar, int phase) {
      ok = ok && __all_sync(0xffffffffu, mbar_wait_bounded(bar, static_cast<uint32_t>(phase) & 1u, abort_flag, a.status));
      return ok;
    };
    if (warp == 9) {
      constexpr uint32_t kIdS = make_idesc_bf16_f32(kRows, kTile);
      const uint64_t qdesc = make_smem_desc_sw128(smem_addr(qs));
      const uint64_t kdesc0 = make_smem_desc_sw128(smem_addr(ring));
      wait(&ctl.q_full, 0);
      for (int t = 0; t < n && ok; ++t) {
        const int i = t == 0 ? 0 : 2 * t - 1, s = i % kNS;   // load of K(t)
        if (t >= 2) {   // P of tile t - 2 lies where S of tile t goes
          if (!wait(&ctl.o_full[t & 1], (t - 2) >> 1)) break;
          tc_fence_after();
        }
        if (!wait(&ctl.full[s], i / kNS)) break;
        if (lead) {
          const uint64_t kd = kdesc0 + static_cast<uint32_t>(s * (C::kSlotBytes >> 4));
          const uint32_t d = tmem + static_cast<uint32_t>((t & 1) * 128);
#pragma unroll
          for (int pl = kQPlanes - 1; pl >= 0; --pl)   // small terms first: fewer roundings at full size
#pragma unroll
            for (int ks = 0; ks < HD / 16; ++ks) {
              const uint32_t off = static_cast<uint32_t>(((ks >> 2) * kTile * 128 + (ks & 3) * 32) >> 4);
              tc_mma_bf16(d, qdesc + pl * (C::kPlaneBytes >> 4) + off, kd + off, kIdS,
                          pl < kQPlanes - 1 || ks > 0 ? 1u : 0u);
            }
          tc_commit(&ctl.empty[s]);
          tc_commit(&ctl.s_full[t & 1]);
        }
        __syncwarp();
      }
    } else {
      constexpr uint32_t kIdO = make_idesc_bf16_f32(kRows, HD) | (1u << 16);   // B N-major
      // V tile, N-major: 64-feature columns kTile x 128 bytes apart, 8-key groups 1024
      const uint64_t vdesc0 = (make_smem_desc_sw128(smem_addr(ring)) & ~(0xFFFFull << 16)) |
                              (static_cast<uint64_t>((kTile * 128) >> 4) << 16);
      for (int t = 0; t < n && ok; ++t) {
        const int i = t == n - 1 ? 2 * n - 1 : 2 * t + 2, s = i % kNS;   // load of V(t)
        if (!wait(&ctl.full[s], i / kNS) || !wait(&ctl.p_full[t & 1], t >> 1)) break;
        tc_fence_after();
        if (lead) {
          const uint64_t vd = vdesc0 + static_cast<uint32_t>(s * (C::kSlotBytes >> 4));
          const uint32_t d = tmem + kO + static_cast<uint32_t>((t & 1) * HD);
          const uint32_t p = tmem + static_cast<uint32_t>((t & 1) * 128);
#pragma unroll
          for (int pl = 0; pl < 2; ++pl)
#pragma unroll
            for (int ks = 0; ks < kTile / 16; ++ks)
              mma_ts(d, p + (ks >> 1) * 32 + pl * 16 + (ks & 1) * 8, vd + static_cast<uint32_t>((ks * 2048) >> 4), kIdO,
                     t >= 2 || pl + ks > 0 ? 1u : 0u);
          tc_commit(&ctl.empty[s]);
          tc_commit(&ctl.o_full[t & 1]);
        }
        __syncwarp();
      }
    }
    if (!ok && n > 0 && lead) {   // every MMA issued completes before the CTA leaves
      uint64_t* drain = &ctl.drain[warp == 9 ? 0 : 1];
      tc_commit(drain);
      mbar_wait_drain(drain, 0);
    }
    __syncwarp();
  } else {
    // ------------------------------------------------ softmax
    const int w = dry ? 0 : warp >> 2;
    const int row = (warp & 3) * 32 + lane;            // MMA row = TMEM lane
    const int copy = row / kVR, v = row % kVR;         // (copy: the same in the whole warp)
    const int rr = v < nq ? v % nr : 0;
    if (w == 0 && copy == 0 && !dry && v < nq) ctl.at[v] = (g * R + r_lo + rr) * a.H + kvh * gs + v / nr;
    if (!dry) named_bar_sync(1, 256);
    if (early && !dry) pdl_wait();
    if (threadIdx.x == 0) trace_at(trace, 2);
    if (n > 0 && !dry) {
      // Q, scaled, in its planes, K-major with the 128-byte swizzle; every copy.  Rows
      // without a vector keep what the memory holds: no other row's result sees them.
      // Eight features are 32 bytes of q and 16 of each plane: they land where planes 1
      // and 2 of them go, all of the CTA's in one round trip
      const int items = nq * (HD / 8);
      auto slot = [&](int vv, int ch) { return qs + (ch >> 3) * (kRows * 128) + vv * 128 + (((ch ^ vv) & 7) << 4); };
#pragma unroll 2
      for (int idx = threadIdx.x; idx < items; idx += 256) {
        const int vv = idx / (HD / 8), ch = idx % (HD / 8);
        const float* src = a.q + static_cast<size_t>(ctl.at[vv]) * HD + ch * 8;
        const uint32_t dst = smem_addr(slot(vv, ch)) + C::kPlaneBytes;
        asm volatile("cp.async.cg.shared.global [%0], [%2], 16;\n\tcp.async.cg.shared.global [%1], [%3], 16;" ::"r"(dst),
                     "r"(dst + C::kPlaneBytes), "l"(src), "l"(src + 4)
                     : "memory");
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll 1
      for (int idx = threadIdx.x; idx < items; idx += 256) {
        const int vv = idx / (HD / 8), ch = idx % (HD / 8);
        uint8_t* at = slot(vv, ch);
        const float4 x0 = *reinterpret_cast<const float4*>(at + C::kPlaneBytes);
        const float4 x1 = *reinterpret_cast<const float4*>(at + 2 * C::kPlaneBytes);
        const float xs[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
        uint32_t pq[kQPlanes][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float y0 = xs[2 * e] * a.scale_log2, y1 = xs[2 * e + 1] * a.scale_log2;
#pragma unroll
          for (int pl = 0; pl < kQPlanes; ++pl) {
            pq[pl][e] = bf16x2(y0, y1);
            const float2 h = unpack2(pq[pl][e]);
            y0 -= h.x;
            y1 -= h.y;
          }
        }
#pragma unroll
        for (int c = 0; c < kCopies; ++c)   // (a copy's rows are a multiple of the swizzle's eight apart)
#pragma unroll
          for (int pl = 0; pl < kQPlanes; ++pl)
            *reinterpret_cast<uint4*>(at + c * kVR * 128 + pl * C::kPlaneBytes) =
                make_uint4(pq[pl][0], pq[pl][1], pq[pl][2], pq[pl][3]);
      }
      fence_proxy_async_smem();
      mbar_arrive(&ctl.q_full);
    }
    const int p_row = v < nq ? pos0 + r_lo + rr : -1;              // last key the row sees
    const uint32_t amask = tree && v < nq && r_lo + rr < kTreeRows ? plan->anc[r_lo + rr] : 0u;
    const uint32_t lanes = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t s_at = tmem + lanes + static_cast<uint32_t>(w * 128);
    const uint32_t o_at = tmem + lanes + kO + static_cast<uint32_t>(w * HD);
    float m = -INFINITY, l = 0.f;
    bool ok = true;
    for (int t = w; t < (dry ? 1 : n); t += 2) {
      ok = dry || __all_sync(0xffffffffu, mbar_wait_bounded(&ctl.s_full[w], static_cast<uint32_t>(t >> 1) & 1u, abort_flag, a.status));
      if (!ok) break;
      tc_fence_after();
      if (t == 0 && threadIdx.x == 0) trace_at(trace, 10);
      const int kt0 = k0 + t * kTile;
      const int key0 = kt0 + copy * KG;
      const bool part = dry || key0 + KG > min(pos0, k1);   // holds keys that some row does not see
      const int lim = min(p_row, k1 - 1);
      auto mask = [&](float* x, int key1) {
        if (!part) return;
        if (!tree) {
#pragma unroll
          for (int e = 0; e < 32; ++e) x[e] = key1 + e <= lim ? x[e] : -INFINITY;
          return;
        }
#pragma unroll
        for (int e = 0; e < 32; ++e) {
          const int rel = key1 + e - pos0;
          const bool vis = key1 + e <= lim && (rel < 0 || (rel < kTreeRows && ((amask >> rel) & 1u) != 0u));
          x[e] = vis ? x[e] : -INFINITY;
        }
      };
      // 32 columns at a time; more than 32 are read again for P
      float s[32];
      float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll 1
      for (int c = 0; c < KG; c += 32) {
        tmem_ld_x32(s_at + copy * KG + c, s);
        mask(s, key0 + c);
#pragma unroll
        for (int e = 0; e < 32; ++e) mx[e & 3] = fmaxf(mx[e & 3], s[e]);
      }
      const float mt = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
      if (t < 2) {
        m = mt;
      } else {
        const bool up = v < nq && mt > m + 8.f;
        if (__any_sync(0xffffffffu, up)) {
          const float f = up ? ex2(m - mt) : 1.f;   // m = -inf: 0
          m = up ? mt : m;
          l *= f;
#pragma unroll 1
          for (int c = 0; c < HD / 32; ++c) {
            float o[32];
            uint32_t u[32];
            tmem_ld_x32(o_at + c * 32, o);
#pragma unroll
            for (int e = 0; e < 32; ++e) u[e] = __float_as_uint(o[e] * f);
            tmem_st_x32(o_at + c * 32, u);
          }
        }
      }
      const float mu = m == -INFINITY ? 0.f : m;
      float sum[4] = {0.f, 0.f, 0.f, 0.f};
      // P over S, 32 keys in the columns of their scores: 16 columns of the hi plane,
      // 16 of the lo plane, two keys a column
#pragma unroll 1
      for (int c = 0; c < KG; c += 32) {
        if constexpr (KG > 32) {
          tmem_ld_x32(s_at + copy * KG + c, s);
          mask(s, key0 + c);
        }
        uint32_t p[32];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const float p0 = ex2(s[2 * e] - mu), p1 = ex2(s[2 * e + 1] - mu);
          sum[(2 * e) & 3] += p0;
          sum[(2 * e + 1) & 3] += p1;
          p[e] = bf16x2(p0, p1);
          const float2 h = unpack2(p[e]);
          p[16 + e] = bf16x2(p0 - h.x, p1 - h.y);
        }
        if (!dry) tmem_st_x32(s_at + copy * KG + c, p);
      }
      l += (sum[0] + sum[1]) + (sum[2] + sum[3]);
      if constexpr (kCopies > 1) {   // zeros for the other copies' keys
        uint32_t z[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) z[e] = 0u;
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (c / (KG / 32) != copy && !dry) tmem_st_x32(s_at + c * 32, z);
      }
      tmem_st_wait();
      if (kt0 + kTile > k1 && !dry) {   // V rows past the last key hold anything: zeros
        const int i = 2 * n - 1;
        ok = __all_sync(0xffffffffu, mbar_wait_bounded(&ctl.full[i % kNS], static_cast<uint32_t>(i / kNS) & 1u, abort_flag, a.status));
        if (!ok) break;
        uint8_t* vs = ring + (i % kNS) * C::kSlotBytes;
        const int nk = k1 - kt0;
        for (int idx = row; idx < (kTile - nk) * (HD / 8); idx += 128) {
          const int kr = nk + idx / (HD / 8), ch = idx % (HD / 8);
          *reinterpret_cast<uint4*>(vs + (ch >> 3) * (kTile * 128) + kr * 128 + ((ch & 7) << 4)) = make_uint4(0u, 0u, 0u, 0u);
        }
        fence_proxy_async_smem();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0 && !dry) mbar_arrive(&ctl.p_full[w]);
    }
    const int mine = (n - w + 1) >> 1;   // tiles of this warpgroup
    if (ok && mine > 0 && !dry)
      ok = __all_sync(0xffffffffu, mbar_wait_bounded(&ctl.o_full[w], static_cast<uint32_t>(mine - 1) & 1u, abort_flag, a.status));
    tc_fence_after();
    if (threadIdx.x == 0) trace_at(trace, 9);
    // the CTA's partial rows: weights against the vector's max, then the sum
    if (n > 0) {
      float* red = reinterpret_cast<float*>(ring);
      if (!dry) {
        named_bar_sync(1, 256);   // every MMA of the CTA has completed: the ring and Q are free
        ml[w * kRows + row] = make_float2(m, l);
        named_bar_sync(1, 256);
      }
      float M = -INFINITY, L = 0.f;
#pragma unroll
      for (int q = 0; q < 2 * kCopies; ++q) M = fmaxf(M, ml[q / kCopies * kRows + (q % kCopies) * kVR + v].x);
#pragma unroll
      for (int q = 0; q < 2 * kCopies; ++q) {
        const float2 x = ml[q / kCopies * kRows + (q % kCopies) * kVR + v];
        if (x.x != -INFINITY) L += ex2(x.x - M) * x.y;
      }
      if (w == 0 && copy == 0 && !dry) cml[v] = make_float2(M, n_cta == 1 ? 1.f / L : L);
      const float f = m == -INFINITY ? 0.f : ex2(m - M);
#pragma unroll 1
      for (int c = 0; c < HD / 32; ++c) {
        float o[32];
        tmem_ld_x32(o_at + c * 32, o);
        if (v < nq && !dry) {
#pragma unroll
          for (int e = 0; e < 32; e += 4) {
            const bool z = m == -INFINITY;   // no visible key, or no tile: O holds anything
            *reinterpret_cast<float4*>(red + red_at<HD>(w * kRows + row, c * 32 + e)) =
                z ? make_float4(0.f, 0.f, 0.f, 0.f)
                  : make_float4(f * o[e], f * o[e + 1], f * o[e + 2], f * o[e + 3]);
          }
        }
      }
      tc_fence_before();
    }
  }

  // every CTA of the cluster: reduce its own rows, then finish a share of the vectors
  float* red = reinterpret_cast<float*>(ring);
  constexpr int kV4 = HD / 4;
  const int tid = dry ? lane : static_cast<int>(threadIdx.x);
  auto emit = [&](int vv, int d, float4 o, float li) {   // li: 1 / sum
    const size_t oi = static_cast<size_t>(ctl.at[vv]) * HD + d;
    const float y[4] = {o.x * li, o.y * li, o.z * li, o.w * li};
    __nv_bfloat16 hv[4], lv[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) split_bf16(y[e], hv[e], lv[e]);
    if (dry) return;
    *reinterpret_cast<uint2*>(a.out + oi) = *reinterpret_cast<const uint2*>(hv);
    if (a.out_lo != nullptr) *reinterpret_cast<uint2*>(a.out_lo + oi) = *reinterpret_cast<const uint2*>(lv);
  };
  if (soft && n > 0) {
    if (!dry) named_bar_sync(1, 256);
    const bool good = !*abort_flag;
#pragma unroll 2
    for (int idx = tid; idx < (!good ? 0 : dry ? kV4 : nq * kV4); idx += 256) {
      const int vv = idx / kV4, d = (idx % kV4) * 4;
      float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int q = 0; q < 2 * kCopies; ++q) {
        const float4 x = *reinterpret_cast<const float4*>(red + red_at<HD>((q / kCopies) * kRows + (q % kCopies) * kVR + vv, d));
        o.x += x.x;
        o.y += x.y;
        o.z += x.z;
        o.w += x.w;
      }
      if (n_cta == 1)
        emit(vv, d, o, cml[vv].y);
      else if (!dry)
        *reinterpret_cast<float4*>(red + red_at<HD>(vv, d)) = o;   // this thread alone reads that place
    }
  }
  if (n_cta > 1) {
    if (!dry) {
      cluster_arrive_release();
      cluster_wait_acquire();
    }
    if (threadIdx.x == 0) trace_at(trace, 6);
    if (soft && work) {
      const uint32_t red_addr = smem_addr(red), cml_addr = smem_addr(cml);
      const int lo = nq * split / n_cta, hi = dry ? lo + 1 : nq * (split + 1) / n_cta;
      const int n_src = dry ? 1 : n_active, src0 = dry ? split : 0;   // (dry: this CTA's own memory)
      // kB x four features of this CTA's vectors from kQ CTAs in one round trip
      auto combine = [&](auto q_c, auto b_c) {
        constexpr int kQ = decltype(q_c)::value, kB = decltype(b_c)::value;
        for (int base = lo * kV4 + tid; base < hi * kV4; base += 256 * kB) {
          float2 st[kB][kQ];
          float4 x[kB][kQ];
#pragma unroll
          for (int b = 0; b < kB; ++b) {
            const int idx = min(base + b * 256, hi * kV4 - 1);
            const int vv = idx / kV4, at = red_at<HD>(vv, (idx % kV4) * 4) * 4;
#pragma unroll
            for (int q = 0; q < kQ; ++q)
              if (q < n_src) {
                st[b][q] = ld_cluster_f2(mapa_shared(cml_addr + vv * 8, src0 + q));
                x[b][q] = ld_cluster_f4(mapa_shared(red_addr + at, src0 + q));
              }
          }
#pragma unroll
          for (int b = 0; b < kB; ++b) {
            const int idx = base + b * 256;
            if (idx >= hi * kV4) break;
            float M = -INFINITY, L = 0.f;
#pragma unroll
            for (int q = 0; q < kQ; ++q)
              if (q < n_src) M = fmaxf(M, st[b][q].x);
            float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int q = 0; q < kQ; ++q)
              if (q < n_src) {
                const float f = st[b][q].x == -INFINITY ? 0.f : ex2(st[b][q].x - M);
                L += f * st[b][q].y;
                o.x += f * x[b][q].x;
                o.y += f * x[b][q].y;
                o.z += f * x[b][q].z;
                o.w += f * x[b][q].w;
              }
            emit(idx / kV4, (idx % kV4) * 4, o, 1.f / L);
          }
        }
      };
      if (n_cta == 2)
        combine(std::integral_constant<int, 2>{}, std::integral_constant<int, 4>{});
      else if (n_cta == 8)
        combine(std::integral_constant<int, 8>{}, std::integral_constant<int, 1>{});
      else
        combine(std::integral_constant<int, 4>{}, std::integral_constant<int, 2>{});
    }
    if (dry) {
      cluster_arrive_release();
      cluster_wait_acquire();
    }
    cluster_arrive_relaxed();   // no CTA leaves while another reads its rows (all were used)
    cluster_wait_acquire();
  }
  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
  if (threadIdx.x == 0) trace_at(trace, 1);
}

template <int HD>
const void* kernel_of(int qmax) {
  if (qmax <= 32) return reinterpret_cast<const void*>(attn_tc_kernel<HD, 32>);
  if (qmax <= 64) return reinterpret_cast<const void*>(attn_tc_kernel<HD, 64>);
  return reinterpret_cast<const void*>(attn_tc_kernel<HD, 128>);
}

}  // namespace

cudaError_t attn_tc_set_max_smem() {
  for (int qmax : {32, 64, 128}) {
    cudaError_t e = cudaFuncSetAttribute(kernel_of<64>(qmax), cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<64>::kSmem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kernel_of<128>(qmax), cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<128>::kSmem);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

namespace {
void tc_config(const AttnArgs& a, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
  cfg->blockDim = dim3(kThreads);
  cfg->dynamicSmemBytes = a.hd == 64 ? Cfg<64>::kSmem : Cfg<128>::kSmem;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = a.n_splits;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
}
const void* kernel_for(int hd, int qmax) { return hd == 64 ? kernel_of<64>(qmax) : kernel_of<128>(qmax); }
}  // namespace

int attn_tc_max_clusters(int hd, int qmax, int C) {
  AttnArgs a{};
  a.hd = hd;
  a.n_splits = C;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3(C);
  tc_config(a, &cfg, attr);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel_for(hd, qmax), &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t launch_attn_tc(const AttnArgs& a, int n_groups, cudaStream_t s, bool pdl) {
  if ((a.hd != 64 && a.hd != 128) || a.qmax > kRows || a.n_splits < 1 || a.n_splits > 8) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  tc_config(a, &cfg, attr);
  cfg.gridDim = dim3(a.n_splits, a.Hkv * a.row_blocks, n_groups);
  cfg.stream = s;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  if (pdl) cfg.numAttrs = 2;
  AttnArgs copy = a;
  void* args[] = {&copy};
  return cudaLaunchKernelExC(&cfg, kernel_for(a.hd, a.qmax), args);
}

}  // namespace memspec
