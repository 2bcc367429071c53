// gemm_pair.cu - the projection GEMM for many activation rows (batched verify,
// prefill, memspec_op_linear): two CTAs of a cluster work on one 256-feature tile.
//
// gemm.cu's kernel gives every CTA its own copy of the activation tile: at 128
// rows in two bf16 planes that is 32 KB fetched from L2 for each 16 KB of weights,
// and the launch is bound by L2 and by the few ring stages that fit.  Here
// tcgen05.mma.cta_group::2 takes M = 256 features (a 128-row weight tile from each
// CTA) against N activation rows of which each CTA holds half, so a CTA's stage is
// half as large and the activation traffic is halved:
//   one plane                  N = n_pad,     CTA r loads rows [r n_pad/2, + n_pad/2)
//   hi + lo, 2 n_pad <= 256    N = 2 n_pad,   CTA 0 loads the hi plane, CTA 1 the lo
//   hi + lo, larger            N = n_pad twice, halves of both: into one accumulator, or
//                              (prefill) two that are added at the end
// Each CTA's tensor memory receives its own 128 features.  In one accumulator the chain
// of sums is twice as long and a lo product, 2^-9 of its hi product, is cut at the hi
// sum's last bit: of a 256-row pass's V (d = 4096) 1.36e-3 of the values are not the
// rounded 64-bit ones, with two 0.67e-3, as with 128 rows side by side.  Two fill the
// tensor memory, so that a segment's MMAs wait until the last one's sums are drained: 2047
// prompt tokens of the 7B 48.1 ms (with one 46.9), 8 layers of the 8B verify of 144 rows
// 1.37 (1.30; with 32 columns of both planes per load in the drain no less: the stores
// bound it).  Prefill takes two, so that its keys and values are as exact in passes of 256
// rows as in passes of 128.
//
// Roles (192 threads per CTA): warp 0 copies its CTA's weights and half of the
// activations, both CTAs' bytes completing on CTA 0's barrier (.cta_group::2; a
// thread of CTA 1 that passed its own barrier on with a release arrive held the
// loop at 1 us per tile); warp 1 of CTA 0 issues every MMA; warps 2-5 drain the
// accumulator (double-buffered where two fit).  Stream-K over pairs; split tiles are left as fp32
// partials for gemm_finish.cu, and so are whole ones but those of the fp32-output
// epilogue (a fused epilogue in here, by four warps, took 20 us for a whole tile of
// 144 rows at the end of some CTAs' ranges).  Every wait is bounded.
//
// Measured (GB300, in a pass, us, gemm.cu's kernel before / this one now; with the
// finishing launch before / now):
//   8B target, 144 rows  gate/up 77.6 / 47.1 (5.0 TB/s of weights), QKV 19.7 / 15.1,
//                        down 39.4 / 32.8; finishing 9-16 / 5-6
//   7B target, 128 rows  gate/up 63.2 / 33.0 (5.5 TB/s), QKV 29.0 / 20.5, down 32.5 /
//                        23.3, O 13.3 / 10.4; finishing 9-15 / 5-6.5
//   7B target, 256 rows  gate/up 48 (1.9 PFLOP/s), QKV 29 (1.8), down 28 (1.6), O 15.5
//                        (one accumulator; prefill's two take 1 to 1.5 more)
#include <cuda_bf16.h>

#include "gemm_epi.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace memspec {

namespace {

using namespace gemm;

constexpr int kPairThreads = 192;
constexpr int kPairMaxStages = 8;

struct PairCtl {
  uint64_t full[kPairMaxStages];        // CTA 0: the stage has landed in both CTAs
  uint64_t empty[kPairMaxStages];       // each CTA: its stage has been read
  uint64_t acc_full[2];
  uint64_t acc_empty[2];                // CTA 0: drained by the eight epilogue warps of the pair
  uint64_t drain;
  uint32_t tmem_base;
  int abort_flag;
  int wait_ok;
};

__device__ __forceinline__ void tmem_alloc_pair(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(dst_smem)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void mma_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// 2-D box into this CTA's shared memory, completing on the barrier at shared::cluster
// address `bar` (CTA 0's).
__device__ __forceinline__ void load_pair(void* dst, const CUtensorMap* map, int x, int y, uint32_t bar,
                                          uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(smem_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar), "l"(policy)
      : "memory");
}
// Arrive once on `bar` of both CTAs when every MMA issued so far has completed.
__device__ __forceinline__ void commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_addr(bar)),
      "h"(static_cast<uint16_t>(3))
      : "memory");
}
// Arrive on `bar` of cluster CTA `rank` (release at cluster scope).
__device__ __forceinline__ void arrive_at(uint64_t* bar, uint32_t rank) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(
                   mapa_shared(smem_addr(bar), rank))
               : "memory");
}

// hi and lo planes as two MMAs, accumulator columns as kWide's
constexpr int kApart = 3;
__host__ __device__ inline int pair_layout(int n_pad, int split, int apart) {
  return !split ? kPlain : (2 * n_pad <= 256 ? kWide : (apart ? kApart : kTwice));
}
// activation bytes of one stage in one CTA
__host__ __device__ inline int pair_b_bytes(int n_pad, int split) { return n_pad * (split ? 128 : 64); }

// Columns col..col+15 of the warp's lanes, plus (lo != 0) the columns lo further.
__device__ __forceinline__ void tmem_ld_sum(uint32_t taddr, uint32_t lo, float* v) {
  uint32_t r[32];
  if (lo == 0) {
    tmem_ld_32x32b_x16(taddr, v);
    return;
  }
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%33];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr), "r"(taddr + lo)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]) + __uint_as_float(r[16 + i]);
}

// F32: the fp32-output epilogue (op_linear, LM head) for tiles owned whole.
template <bool F32>
__global__ void __launch_bounds__(kPairThreads, 1) gemm_pair_kernel(const __grid_constant__ GemmArgs a) {
  __shared__ PairCtl ctl;
  extern __shared__ uint8_t dsmem_raw[];
  uint8_t* dsmem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(dsmem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int S = a.stages;
  const int b_bytes = pair_b_bytes(a.n_pad, a.split);
  const uint32_t stage_tx = static_cast<uint32_t>(kABytes + b_bytes);
  uint8_t* smem_a = dsmem;
  uint8_t* smem_b = dsmem + static_cast<size_t>(S) * kABytes;
  [[maybe_unused]] float* rms = reinterpret_cast<float*>(smem_b + static_cast<size_t>(S) * b_bytes);   // F32
  [[maybe_unused]] EpiCtx* ectx = reinterpret_cast<EpiCtx*>(rms + kMaxRows);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int KT = a.k_tiles;
  const int T = (a.row_tiles + 1) / 2 * KT;      // tiles of row-tile pairs
  const int G = gridDim.x >> 1, c = blockIdx.x >> 1;
  const int t_begin = sk_begin(c, T, G), t_end = sk_begin(c + 1, T, G);
  const int layout = pair_layout(a.n_pad, a.split, a.apart);
  const bool sums = layout == kWide || layout == kApart;   // hi in columns [0, n_pad), lo in the next n_pad
  const int acols = sums ? 2 * a.n_pad : a.n_pad;
  const int bufs = layout == kApart ? 1 : 2;               // accumulators that fit (512 columns)
  const uint32_t tmem_cols = layout == kApart ? 512 : tmem_cols_for(acols);

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&ctl.full[s], 1);
      mbar_init(&ctl.empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&ctl.acc_full[b], 1);
      mbar_init(&ctl.acc_empty[b], 8);
    }
    mbar_init(&ctl.drain, 1);
    ctl.abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    __syncwarp();
    tmem_alloc_pair(&ctl.tmem_base, tmem_cols);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // both CTAs' barriers and tensor memory exist before either touches the other's
  cluster_arrive_release();
  cluster_wait_acquire();
  const uint32_t tmem_base = ctl.tmem_base;
  unsigned long long* trace = a.trace != nullptr ? a.trace + blockIdx.x * 16 : nullptr;
  if (threadIdx.x == 64) trace_at(trace, 0);
  volatile int* abort_flag = &ctl.abort_flag;

  if (warp == 0) {
    // ------------------------------------------------ copies
    if (lane == 0) {
      tma_prefetch_desc(&a.map_a);
      tma_prefetch_desc(&a.map_b);
      if (a.split) tma_prefetch_desc(&a.map_b2);
      const uint64_t pol = a.l2_hint == L2_EVICT_FIRST ? l2_policy_evict_first() : l2_policy_evict_normal();
      const uint64_t pol_b = l2_policy_evict_last();   // activations are re-read by every pair
      const uint32_t full0 = mapa_shared(smem_addr(&ctl.full[0]), 0);
      // an odd last row tile is paired with itself (its second result is dropped)
      auto row_tile = [&](int pt) { return min(2 * pt + rank, a.row_tiles - 1); };
      auto load_a = [&](int slot, int pt, int kt) {
        uint8_t* dst = smem_a + static_cast<size_t>(slot) * kABytes;
        const int rt = row_tile(pt);
        if (a.a_packed != nullptr)   // a packed tile is 32 rows of 512 bytes of the map
          load_pair(dst, &a.map_a, 0, (rt * KT + kt) * 32, full0 + slot * 8, pol);
        else
          load_pair(dst, &a.map_a, kt * kTileK, rt * kTileM, full0 + slot * 8, pol);
      };
      const int half = a.n_pad / 2;
      auto load_b = [&](int slot, int kt) {
        uint8_t* dst = smem_b + static_cast<size_t>(slot) * b_bytes;
        if (layout == kWide) {
          load_pair(dst, rank == 0 ? &a.map_b : &a.map_b2, kt * kTileK, 0, full0 + slot * 8, pol_b);
        } else {
          load_pair(dst, &a.map_b, kt * kTileK, rank * half, full0 + slot * 8, pol_b);
          if (a.split) load_pair(dst + half * 128, &a.map_b2, kt * kTileK, rank * half, full0 + slot * 8, pol_b);
        }
      };
      // CTA 0 announces the bytes of both (CTA 1's may land before that)
      auto expect = [&](int slot) {
        if (rank == 0) mbar_arrive_expect_tx(&ctl.full[slot], 2 * stage_tx);
      };
      uint32_t issued_mask = 0, last_par = 0;
      bool ok = true;
      const int n_pre = min(S, t_end - t_begin);
      int pt = t_begin / KT, kt = t_begin - pt * KT;
      const int kt_first = kt;
      if (a.w_after_wait) pdl_wait();
      // weights do not depend on the previous launch: requested before its end
      for (int p = 0; p < n_pre; ++p) {
        expect(p);
        load_a(p, pt, kt);
        issued_mask |= 1u << p;
        if (++kt == KT) {
          kt = 0;
          ++pt;
        }
      }
      pdl_wait();
      pdl_launch_dependents();   // after the wait: see ptx.cuh
      trace_at(trace, 2);
      for (int p = 0, k2 = kt_first; p < n_pre; ++p) {
        load_b(p, k2);
        if (++k2 == KT) k2 = 0;
      }
      int s = n_pre == S ? 0 : n_pre;
      uint32_t ph = n_pre == S ? 1u : 0u;
      for (int t = t_begin + n_pre; t < t_end; ++t) {
        if (!mbar_wait_bounded(&ctl.empty[s], ph ^ 1u, abort_flag, a.status)) {
          ok = false;
          break;
        }
        expect(s);
        load_a(s, pt, kt);
        load_b(s, kt);
        issued_mask |= 1u << s;
        last_par = (last_par & ~(1u << s)) | (ph << s);
        if (++kt == KT) {
          kt = 0;
          ++pt;
        }
        if (++s == S) {
          s = 0;
          ph ^= 1u;
        }
      }
      // the CTA leaves after its copies have landed and the last MMAs have signalled
      // its barriers (a wait that ran out: CTA 0 waits for the copies of both, CTA 1
      // for CTA 0 at the end)
      for (int q = 0; q < S; ++q)
        if ((issued_mask & (1u << q)) && (ok || rank == 0))
          mbar_wait_drain(ok ? &ctl.empty[q] : &ctl.full[q], (last_par >> q) & 1u);
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ---------------------------------------------- CTA 0: MMAs
      // The whole warp walks the tiles and one elected lane issues, so that descriptors
      // and loop counters stay in uniform registers.
      const bool lead = elect_one();
      const uint32_t idesc = make_idesc_bf16_f32(2 * kTileM, layout == kWide ? 2 * a.n_pad : a.n_pad);
      const uint64_t adesc0 = make_smem_desc_sw128(smem_addr(smem_a));
      const uint64_t bdesc0 = make_smem_desc_sw128(smem_addr(smem_b));
      const uint32_t a_step = kABytes >> 4, b_step = static_cast<uint32_t>(b_bytes) >> 4;
      // kTwice, kApart: the lo plane and its accumulator
      const uint32_t p_step = static_cast<uint32_t>(a.n_pad / 2 * 128) >> 4;
      const uint32_t lo_col = layout == kApart ? a.n_pad : 0;
      int s = 0, seg = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = t_begin; t < t_end && ok; ++seg) {
        const int seg_end = min(t_end, (t / KT + 1) * KT);
        const int buf = seg & (bufs - 1), use = seg >> (bufs - 1);
        if (use > 0) {
          ok = __all_sync(0xffffffffu,
                          mbar_wait_cluster_bounded(&ctl.acc_empty[buf], static_cast<uint32_t>(use - 1) & 1u,
                                                    abort_flag, a.status));
          if (!ok) break;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(buf * acols);
        for (int tt = t; tt < seg_end; ++tt) {
          ok = __all_sync(0xffffffffu, mbar_wait_bounded(&ctl.full[s], ph, abort_flag, a.status));
          if (!ok) break;
          tc_fence_after();
          const uint64_t ad = adesc0 + static_cast<uint32_t>(s) * a_step;
          const uint64_t bd = bdesc0 + static_cast<uint32_t>(s) * b_step;
          const uint32_t acc0 = tt > t ? 1u : 0u;
          if (lead) {
            if (tt == t_begin) trace_at(trace, 3);
            if (layout < kTwice) {
#pragma unroll
              for (int kk = 0; kk < kTileK / 16; ++kk)
                mma_pair(d_tmem, ad + 2 * kk, bd + 2 * kk, idesc, kk > 0 ? 1u : acc0);
            } else {
#pragma unroll
              for (int kk = 0; kk < kTileK / 16; ++kk) {
                mma_pair(d_tmem, ad + 2 * kk, bd + 2 * kk, idesc, kk > 0 ? 1u : acc0);
                mma_pair(d_tmem + lo_col, ad + 2 * kk, bd + p_step + 2 * kk, idesc, kk > 0 || lo_col == 0 ? 1u : acc0);
              }
            }
            commit_pair(&ctl.empty[s]);
          }
          __syncwarp();
          if (++s == S) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (!ok) break;
        if (lead) commit_pair(&ctl.acc_full[buf]);
        __syncwarp();
        t = seg_end;
      }
      if (!ok && lead) {   // every MMA issued completes before the pair leaves
        commit_pair(&ctl.drain);
        mbar_wait_drain(&ctl.drain, 0);
      }
    }
  } else {
    // ------------------------------------------------ drain (warps 2-5)
    const int ew = warp & 3;
    const int et = ew * 32 + lane;   // tile feature == TMEM lane
    pdl_wait();                      // the partials may still be read by an earlier launch
    if (threadIdx.x == 64) trace_at(trace, 13);
    if constexpr (F32) {
      if (a.rms) rms_prologue(a, rms, et);
      epi_prologue<EPI_F32>(a, ectx, et);
    }
    int seg = 0;
    for (int t = t_begin; t < t_end; ++seg) {
      const int pt = t / KT, rt = 2 * pt + rank;
      const int seg_end = min(t_end, (pt + 1) * KT);
      [[maybe_unused]] const bool whole = t == pt * KT && seg_end == (pt + 1) * KT;
      const int slot = pair_slot(a, pt, c, rank, seg == 0 ? 0 : 1);
      const int buf = seg & (bufs - 1);
      if (threadIdx.x == 64)
        ctl.wait_ok =
            mbar_wait_bounded(&ctl.acc_full[buf], static_cast<uint32_t>(seg >> (bufs - 1)) & 1u, abort_flag, a.status) ? 1 : 0;
      named_bar_sync(1, 128);
      const int ok = ctl.wait_ok;
      named_bar_sync(1, 128);
      if (!ok) break;
      tc_fence_after();
      if (rt < a.row_tiles) {
        const uint32_t tbase =
            tmem_base + (static_cast<uint32_t>(ew * 32) << 16) + static_cast<uint32_t>(buf * acols);
        const int chunks = (a.rows_total + 15) / 16;
        for (int chunk = 0; chunk < chunks; ++chunk) {
          float v[16];
          tmem_ld_sum(tbase + chunk * 16, sums ? a.n_pad : 0, v);
          if constexpr (F32) {
            if (whole) {
              const int f = rt * kTileM + et;
              if (f < a.n_out) {
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                  const int r = chunk * 16 + j;
                  const float y = a.rms ? v[j] * rms[r] : v[j];
                  if (a.last_only) {
                    if (ctx_bit(ectx->last, r)) a.out[ectx->grp[r] * a.out_group_stride + f] = y;
                  } else if (ctx_bit(ectx->valid, r)) {
                    a.out[static_cast<size_t>(r) * a.out_ld + f] = y;
                  }
                }
              }
              continue;
            }
          }
          float* dst = a.partials + part_offset(slot, chunks, chunk, et);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            *reinterpret_cast<float4*>(dst + q * kTileM * 4) =
                make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) arrive_at(&ctl.acc_empty[buf], 0);
      if (threadIdx.x == 64) trace_at(trace, 4);
      t = seg_end;
    }
  }

  // neither CTA frees its tensor memory or leaves while the other may still use it
  // or signal its barriers
  tc_fence_before();
  __syncthreads();
  cluster_arrive_release();
  cluster_wait_acquire();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, tmem_cols);
  }
  if (threadIdx.x == 64) trace_at(trace, 1);
}

constexpr int kPairSmemF32 = 222 * 1024;   // dynamic shared memory, most of it the ring
constexpr int kPairSmem = 196 * 1024;      // leaves room for the next launch's first CTAs
int pair_fixed_bytes(int epi) {
  return 1024 + (epi == EPI_F32 ? kMaxRows * 4 + static_cast<int>(sizeof(EpiCtx)) : 0);
}

}  // namespace

// An MMA's N (n_pad, or 2 n_pad for two planes side by side) is a multiple of 32.
int gemm_pair_pad(int rows, int split) {
  const int m = split && rows <= 128 ? 16 : 32;
  return (rows + m - 1) / m * m;
}

int gemm_pair_box_rows(int n_pad, int split) {
  return pair_layout(n_pad, split, 0) == kWide ? n_pad : n_pad / 2;
}

int gemm_pair_stages(int n_pad, int split, int epi) {
  const int budget = (epi == EPI_F32 ? kPairSmemF32 : kPairSmem) - pair_fixed_bytes(epi);
  const int s = budget / (kABytes + pair_b_bytes(n_pad, split));
  return s < kPairMaxStages ? s : kPairMaxStages;
}

cudaError_t gemm_pair_set_max_smem() {
  cudaError_t e = cudaFuncSetAttribute(gemm_pair_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmemF32);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_pair_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem);
  return e;
}

cudaError_t launch_gemm_pair(const GemmArgs& a, cudaStream_t s, bool pdl) {
  if (a.n_pad != gemm_pair_pad(a.rows_total, a.split) || a.n_pad > kMaxRows || a.stages < 2 || (a.pair && a.a_packed == nullptr))
    return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * a.pairs);
  cfg.blockDim = dim3(kPairThreads);
  cfg.dynamicSmemBytes = static_cast<size_t>(a.stages) * (kABytes + pair_b_bytes(a.n_pad, a.split)) +
                         pair_fixed_bytes(a.epi);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return a.epi == EPI_F32 ? cudaLaunchKernelEx(&cfg, gemm_pair_kernel<true>, a)
                          : cudaLaunchKernelEx(&cfg, gemm_pair_kernel<false>, a);
}

}  // namespace memspec
