// gemm.cu - weight-streaming projection GEMM with fp32 output (memspec_op_linear from
// 17 to 160 rows, memspec_op_linear_noalloc); the persistent pass kernel streams its
// projections the same way.
//
// Y[rows][n_out] = X[rows][k] . W[n_out][k]^T with rows <= 256.  At these row counts
// every projection reads each weight exactly once and is bound by HBM bandwidth, so
// the kernel is organised around streaming weights:
//
//  * swap-AB: the weight tile is the MMA's M=128 operand, the activation rows
//    are its N (16..256) operand; tcgen05.mma.kind::f16 (bf16 in, fp32 out)
//    accumulates in TMEM;
//  * weight tiles [128 rows x 64 k] and activation tiles [n_pad rows x 64 k] arrive
//    by TMA (128-byte swizzle) into a multi-stage ring, a stage's copies on one
//    mbarrier, all after griddepcontrol.wait;
//  * stream-K: the (row-tile, k-tile) space is cut into one contiguous range
//    per CTA, one CTA per SM; a row tile split over several CTAs is reduced by
//    the last-arriving CTA in ascending CTA order (deterministic, no float
//    atomics) from an fp32 partial buffer;
#include <cuda_bf16.h>

#include <cstdlib>

#include "gemm_epi.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace memspec {

namespace {

using namespace gemm;

constexpr int kThreads = 192;   // warp 0 TMA, warp 1 MMA, warps 2-5 epilogue

struct SmemCtl {
  uint64_t full[kMaxStages];
  uint64_t empty[kMaxStages];
  uint64_t acc_full[2];
  uint64_t acc_empty[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort_flag;
  int reduce_flag;
  int wait_ok;
  float red[4][16];
};

__global__ void __launch_bounds__(kThreads, 1) gemm_stream_kernel(const __grid_constant__ GemmArgs a) {
  __shared__ SmemCtl ctl;
  extern __shared__ uint8_t dsmem_raw[];
  uint8_t* dsmem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(dsmem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int S = a.stages;
  const int b_bytes = a.n_pad * 128;                  // [n_pad][64] bf16 activations
  const uint32_t stage_tx = static_cast<uint32_t>(kABytes + b_bytes);
  uint8_t* smem_a = dsmem;
  uint8_t* smem_b = dsmem + static_cast<size_t>(S) * kABytes;
  float* stage = reinterpret_cast<float*>(smem_b + static_cast<size_t>(S) * b_bytes);
  float* rms = stage + kStageFloats;
  EpiCtx* ectx = reinterpret_cast<EpiCtx*>(rms + kMaxRows);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int T = a.row_tiles * a.k_tiles;
  const int G = gridDim.x, c = blockIdx.x;
  const int t_begin = sk_begin(c, T, G), t_end = sk_begin(c + 1, T, G);
  const int KT = a.k_tiles;
  const int acols = acc_cols(a, kPlain);                 // accumulator columns per buffer
  const uint32_t tmem_cols = tmem_cols_for(acols);

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&ctl.full[s], 1);
      mbar_init(&ctl.empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&ctl.acc_full[b], 1);
      mbar_init(&ctl.acc_empty[b], 4);
    }
    mbar_init(&ctl.drain, 1);
    ctl.abort_flag = 0;
    ctl.reduce_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    __syncwarp();
    tmem_alloc(&ctl.tmem_base, tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = ctl.tmem_base;
  // optional trace (16 slots per CTA): 0 entry, 13 dependency released,
  // 2 activation loads issued, 3 first MMA, 4..11 epilogue, 1 exit
  unsigned long long* trace = a.trace != nullptr ? a.trace + blockIdx.x * 16 : nullptr;
  if (threadIdx.x == 64) trace_at(trace, 0);
  volatile int* abort_flag = &ctl.abort_flag;

  if (warp == 0) {
    // ------------------------------------------------ TMA producer
    // The weights' maps point at the caller's matrix, which earlier work on the stream may
    // write: every copy comes after the wait.
    if (lane == 0) {
      tma_prefetch_desc(&a.map_a);
      tma_prefetch_desc(&a.map_b);
      const uint64_t pol = l2_policy_evict_first();
      const uint64_t pol_b = l2_policy_evict_last();   // activations are re-read by every CTA
      uint32_t issued_mask = 0, last_par = 0;
      bool ok = true;
      const int n_pre = min(S, t_end - t_begin);
      // One thread issues every copy, so the loop is lean: the ring position and
      // the tile coordinates advance incrementally (no division per tile).
      int rt = t_begin / KT, kt = t_begin - rt * KT;
      auto load_a = [&](int slot) {
        tma_load_2d(smem_a + static_cast<size_t>(slot) * kABytes, &a.map_a, kt * kTileK, rt * kTileM, &ctl.full[slot], pol);
      };
      auto load_b = [&](int slot, int k_tile) {
        tma_load_2d(smem_b + static_cast<size_t>(slot) * b_bytes, &a.map_b, k_tile * kTileK, 0, &ctl.full[slot], pol_b);
      };
      pdl_wait();
      pdl_launch_dependents();   // after the wait: see ptx.cuh
      trace_at(trace, 2);
      // the first n_pre tiles (the ring is empty: no wait needed)
      for (int p = 0; p < n_pre; ++p) {
        mbar_arrive_expect_tx(&ctl.full[p], stage_tx);
        load_a(p);
        load_b(p, kt);
        issued_mask |= 1u << p;
        if (++kt == KT) {
          kt = 0;
          ++rt;
        }
      }
      int s = n_pre == S ? 0 : n_pre;
      uint32_t ph = n_pre == S ? 1u : 0u;   // phase of the fill the next wait is for
      for (int t = t_begin + n_pre; t < t_end; ++t) {
        if (!mbar_wait_bounded(&ctl.empty[s], ph ^ 1u, abort_flag, a.status)) {
          ok = false;
          break;
        }
        mbar_arrive_expect_tx(&ctl.full[s], stage_tx);
        load_a(s);
        load_b(s, kt);
        issued_mask |= 1u << s;
        last_par = (last_par & ~(1u << s)) | (ph << s);
        if (++kt == KT) {
          kt = 0;
          ++rt;
        }
        if (++s == S) {
          s = 0;
          ph ^= 1u;
        }
      }
      if (!ok) {  // tear-down: let every copy still in flight land before exit
        for (int s = 0; s < S; ++s)
          if (issued_mask & (1u << s)) mbar_wait_drain(&ctl.full[s], (last_par >> s) & 1u);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer
    // The whole warp walks the tiles and one elected lane issues, so that descriptors
    // and loop counters stay in uniform registers.
    const bool lead = elect_one();
    const uint32_t idesc = make_idesc_bf16_f32(kTileM, a.n_pad);
    // descriptors of stage 0; a stage's (and a k-step's) are offsets in the
    // start-address field (address >> 4, 14 bits: shared memory < 256 KB)
    const uint64_t adesc0 = make_smem_desc_sw128(smem_addr(smem_a));
    const uint64_t bdesc0 = make_smem_desc_sw128(smem_addr(smem_b));
    const uint32_t a_step = kABytes >> 4, b_step = static_cast<uint32_t>(b_bytes) >> 4;
    int s = 0, seg = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int t = t_begin; t < t_end && ok; ++seg) {
      const int seg_end = min(t_end, (t / KT + 1) * KT);
      const int buf = seg & 1;
      if (seg >= 2) {
        ok = __all_sync(0xffffffffu, mbar_wait_bounded(&ctl.acc_empty[buf], static_cast<uint32_t>((seg >> 1) - 1) & 1u,
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
#pragma unroll
          for (int kk = 0; kk < kTileK / 16; ++kk)
            tc_mma_bf16(d_tmem, ad + 2 * kk, bd + 2 * kk, idesc, kk > 0 ? 1u : acc0);
          tc_commit(&ctl.empty[s]);
        }
        __syncwarp();
        if (++s == S) {
          s = 0;
          ph ^= 1u;
        }
      }
      if (!ok) break;
      if (lead) tc_commit(&ctl.acc_full[buf]);
      __syncwarp();
      t = seg_end;
    }
    if (!ok && lead) {  // tear-down: wait for every MMA already issued
      tc_commit(&ctl.drain);
      mbar_wait_drain(&ctl.drain, 0);
    }
  } else {
    // ------------------------------------------------ epilogue (warps 2-5)
    // a warp may only read TMEM lanes 32*(warp % 4) .. +31: that is its feature block
    const int ew = warp & 3;
    const int et = ew * 32 + lane;  // tile feature == TMEM lane
    pdl_wait();
    if (threadIdx.x == 64) trace_at(trace, 13);
    epi_prologue<EPI_F32>(a, ectx, et);
    int seg = 0;
    for (int t = t_begin; t < t_end; ++seg) {
      const int rt = t / KT;
      const int k0 = t - rt * KT;
      const int seg_end = min(t_end, (rt + 1) * KT);
      const int k1 = seg_end - rt * KT;
      const int buf = seg & 1;
      // one thread waits; the four epilogue warps follow (or stop) together
      if (threadIdx.x == 64)
        ctl.wait_ok = mbar_wait_bounded(&ctl.acc_full[buf], static_cast<uint32_t>(seg >> 1) & 1u,
                                        abort_flag, a.status)
                          ? 1
                          : 0;
      named_bar_sync(1, 128);
      const int ok = ctl.wait_ok;
      named_bar_sync(1, 128);
      if (!ok) break;
      tc_fence_after();
      epilogue_segment<EPI_F32>(a, ectx, kPlain, acols, tmem_base, buf, seg, c, G, rt, k0, k1, stage, rms, ctl.red,
                            &ctl.reduce_flag, ctl.acc_empty, et, ew, lane, threadIdx.x == 64 ? trace : nullptr);
      t = seg_end;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, tmem_cols);
  }
  if (threadIdx.x == 64) trace_at(trace, 1);
}

}  // namespace

// Shared-memory budget of the stage ring.  A deep ring keeps more weight bytes
// in flight per SM; a budget under ~110 KB lets the next kernel's CTA start on
// the same SM early (programmatic dependent launch).  MEMSPEC_GEMM_SMEM_KB
// overrides the default (for measurement).
static int gemm_budget_bytes() {
  static int env_kb = -1;
  if (env_kb < 0) {
    const char* e = std::getenv("MEMSPEC_GEMM_SMEM_KB");
    env_kb = e != nullptr ? std::atoi(e) : 0;
  }
  if (env_kb > 0) return env_kb * 1024;
  return 200 * 1024;
}

int gemm_pick_stages(int n_pad) {
  const int stage = kABytes + n_pad * 128;
  const int budget = gemm_budget_bytes();
  const int fixed = kTileM * kStagePitch * 4 + kMaxRows * 4 + static_cast<int>(sizeof(EpiCtx)) + 1024;
  int s = (budget - fixed) / stage;
  if (s > kMaxStages) s = kMaxStages;
  if (s < 2) s = 2;
  return s;
}

size_t gemm_smem_bytes(int n_pad, int stages) {
  return static_cast<size_t>(stages) * (kABytes + n_pad * 128) + kTileM * kStagePitch * 4 +
         kMaxRows * 4 + sizeof(EpiCtx) + 1024;
}

cudaError_t gemm_set_max_smem() {
  // 227 KB per block minus the kernel's static shared memory
  return cudaFuncSetAttribute(gemm_stream_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
}

cudaError_t launch_gemm(const GemmArgs& a, int grid, size_t smem, cudaStream_t s, bool pdl) {
  if (a.epi != EPI_F32) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, gemm_stream_kernel, a);
}

}  // namespace memspec
