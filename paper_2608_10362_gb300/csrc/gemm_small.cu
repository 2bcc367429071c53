// gemm_small.cu - projection GEMM for the rows of a decode pass: up to 8 activation
// rows in two bf16 planes (verify and draft passes), up to 16 in one
// (memspec_op_linear).
//
// gemm.cu's weight stream (128 x 64 tiles by 16 KB copies into an mbarrier ring,
// tcgen05 MMA with the weights as M = 128, stream-K over one CTA per SM) with what
// bounds such a launch beside the stream cut down:
//  * the activations of a k tile are one 2 KB MMA operand of N = 16 rows, hi plane in
//    rows 0..7 and lo plane in rows 8..15, and arrive as one box of a 4-D map
//    {64 columns, 8 rows, 2 planes, k tiles}; the boxes of the ring's first fill, which
//    wait for the previous launch, cover four k tiles each.  A TMA request costs an SM
//    about 100 ns whatever its size: with two per tile the first MMAs of a launch,
//    their weights long in shared memory, came 225 ns apart;
//  * the tail handles 8 rows: the residual rows and the gain are requested before the
//    accumulator is waited for, the tile is turned in shared memory so that a thread
//    finishes eight features of one row (four wide stores instead of 24 narrow ones),
//    and the partial sums exchanged between contributors are half as large.
// A row tile split over several CTAs is reduced in ascending CTA order: by the first
// contributor from partials pushed into its shared memory where they share a cluster
// (CSK), else by the last to arrive, from global memory.
//
// Measured (GB300; us from the previous launch's end, gemm.cu's kernel before / now):
//   7B target, 5 rows    QKV 21.8 / 16.4 (6.1 TB/s), O 14.5 / 7.7, gate/up 31.0 / 28.2
//                        (6.4 TB/s), down 20.0 / 15.4; verify pass 3.28 / 2.73 ms
//   1.1B target, 6 rows  QKV 10.5 / 4.6, O 10.5 / 5.2, down 14.3 / 7.9; 1.31 / 0.90 ms
//   alone, 5 rows        2304 x 768 8.5 / 4.2, 4096 x 4096 13.9 / 8.6, 28672 x 4096 44.5 /
//                        38.2 (6.2 TB/s); without the launch overlapping the previous one's
//                        end (set-up, dry run; every read stays behind the wait) 5.6, 10.1,
//                        39.3
// Tried instead: the features of a launch dealt to CTAs in any number over all of k,
// without split-K (mma.sync from registers or from row runs of the packed tiles): 2 to 3
// TB/s, a run of 27 rows is 3.4 KB a k tile.
#include <cuda_bf16.h>

#include "gemm_epi.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace memspec {

namespace {

using namespace gemm;

constexpr int kThreads = 192;    // warp 0 copies, warp 1 MMA, warps 2-5 epilogue
constexpr int kN = 16;           // MMA N
constexpr int kBBytes = kN * 128;
constexpr int kSmallStages = 12;
constexpr int kXGroup = 4;       // k tiles of a first-fill activation box

// The rows of the pass and, for QKV, their RoPE factors.
struct SmallRows {
  int pos[8], req[8], grp[8];
  uint32_t valid, last;          // bit r: row r is valid / the last valid row of its group
  float rc[8][64], rs[8][64];
};

struct SmallCtl {
  uint64_t full[kSmallStages];
  uint64_t empty[kSmallStages];
  uint64_t acc_full[2];
  uint64_t acc_empty[2];
  uint64_t drain;
  uint64_t recv;                 // CSK: partials pushed by peers (one phase)
  uint32_t tmem_base;
  int abort_flag;
  int reduce_flag;
  int wait_ok;
  int recv_pending;
  float scale[8];                // RMSNorm scale of each row
};

// Rows of y per thread: 8, or 16 of one plane.
template <int PLANES>
constexpr int rows_of() {
  return PLANES == 2 ? 8 : 16;
}

// The 128 epilogue threads; no barrier at the end.
template <int EPI>
__device__ __forceinline__ void small_rows(const GemmArgs& a, SmallRows& sr, int et) {
  const RowPlan* plan = a.plan;
  if (et < 32) {
    const int r = et;
    bool valid = false, last = false;
    int g = 0, pos = 0, req = 0;
    if (r < 8 && r < a.rows_total) {
      valid = last = true;
      if (plan != nullptr) {
        const int R = plan->rows_per_group;
        g = r / R;
        const int i = r - g * R;
        const int nv = plan->valid[g];
        valid = i < nv;
        last = i == nv - 1;
        pos = plan->pos0[g] + i;
        req = plan->req[g];
      }
    }
    const uint32_t vb = __ballot_sync(0xffffffffu, valid), lb = __ballot_sync(0xffffffffu, last);
    if (r < 8) {
      sr.pos[r] = pos;
      sr.req[r] = req;
      sr.grp[r] = g;
    }
    if (r == 0) {
      sr.valid = vb;
      sr.last = lb;
    }
  }
  if constexpr (EPI == EPI_QKV) {
    // thread (row et / 16, pairs et % 16 + 16 i): the factors at the row's position
    const int r = et >> 4, half = a.head_dim >> 1;
    int pos = -1;
    if (r < a.rows_total) {
      const int R = plan->rows_per_group, g = r / R, i = r - g * R;
      pos = plan->pos0[g] + i;
      if (i >= plan->valid[g] || pos < 0 || pos >= a.max_seq)
        pos = -1;
      else if (plan->tree && i < kTreeRows)
        pos = plan->pos0[g] + plan->rope_off[i];
    }
    for (int ip = et & 15; ip < half; ip += 16) {
      sr.rc[r][ip] = pos >= 0 ? a.rope_cos[static_cast<size_t>(pos) * half + ip] : 0.f;
      sr.rs[r][ip] = pos >= 0 ? a.rope_sin[static_cast<size_t>(pos) * half + ip] : 0.f;
    }
  }
}

// RMSNorm scales: warp w of the four takes rows w and w + 4.
__device__ __forceinline__ void small_scales(const GemmArgs& a, float* scale, int et) {
  const int w = et >> 5, lane = et & 31;
  float ss[2] = {0.f, 0.f};
#pragma unroll
  for (int q = 0; q < 2; ++q)
    if (w + 4 * q < a.rows_total)
      for (int i = lane; i < a.ss_count; i += 32) ss[q] += __ldcg(a.ss + static_cast<size_t>(i) * a.ss_stride + w + 4 * q);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ss[0] += __shfl_xor_sync(0xffffffffu, ss[0], o);
    ss[1] += __shfl_xor_sync(0xffffffffu, ss[1], o);
  }
  if (lane < 2) scale[w + 4 * lane] = rsqrtf((lane ? ss[1] : ss[0]) / static_cast<float>(a.k_in) + a.eps);
}

// The finishing threads of a tile (two planes): thread et takes row et / 16 and the
// tile's features 4 c .. 4 c + 3 and 64 + 4 c .. + 3, c = et % 16: a row's sum of
// squares is one half-warp's, a SwiGLU pair and (head_dim 128) a RoPE pair are one
// thread's, and stores are 16 or 8 bytes.
struct EpiPre {          // what they need beside the sums, requested before them
  float4 h[2];           // EPI_RESIDUAL: residual and gain
  uint2 gain[2];
};
template <int EPI>
__device__ __forceinline__ void small_pre(const GemmArgs& a, int rt, int et, EpiPre& p) {
  if constexpr (EPI == EPI_RESIDUAL) {
    const int r = et >> 4;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int f = rt * kTileM + 64 * q + 4 * (et & 15);
      p.h[q] = make_float4(0.f, 0.f, 0.f, 0.f);
      p.gain[q] = make_uint2(0u, 0u);
      if (r < a.rows_total) {
        p.h[q] = __ldcg(reinterpret_cast<const float4*>(a.h + static_cast<size_t>(r) * a.h_ld + f));
        if (a.gain_next != nullptr) p.gain[q] = *reinterpret_cast<const uint2*>(a.gain_next + f);
      }
    }
  }
}

__device__ __forceinline__ uint2 pack_bf16x4(float x, float y, float z, float w) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(x, y), hi = __floats2bfloat162_rn(z, w);
  return make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}
__device__ __forceinline__ float bf_at(uint2 v, int i) {
  const uint32_t w = i < 2 ? v.x : v.y;
  return __uint_as_float(i & 1 ? w & 0xffff0000u : w << 16);
}
// Four consecutive values as hi and lo planes.
__device__ __forceinline__ void store_split4(bf16* hi_p, bf16* lo_p, const float (&y)[4]) {
  const uint2 hi = pack_bf16x4(y[0], y[1], y[2], y[3]);
  *reinterpret_cast<uint2*>(hi_p) = hi;
  *reinterpret_cast<uint2*>(lo_p) =
      pack_bf16x4(y[0] - bf_at(hi, 0), y[1] - bf_at(hi, 1), y[2] - bf_at(hi, 2), y[3] - bf_at(hi, 3));
}

constexpr int kStageLd = kTileM + 4;   // staged tile: [8 rows][128 features], padded

// Epilogue of row tile rt: v = the sums of feature et (= TMEM lane) of the tile.  The
// 128 epilogue threads together; dry: nothing is stored.  Inlined at its one call: a
// called function reads the launch parameters through memory, not the constant bank,
// which took 0.5 us of the tail.
template <int EPI, int PLANES>
__device__ __forceinline__ void small_epilogue(const GemmArgs& a, const SmallRows& sr, const float* scale, float* stage,
                                               int rt, int et, const float* v, const EpiPre& pre,
                                               unsigned long long* ts, bool dry) {
  constexpr int NR = rows_of<PLANES>();
  if constexpr (EPI == EPI_F32) {   // out rows of any length and alignment: a feature per thread
    const int f = rt * kTileM + et;
    if (f < a.n_out && !dry) {
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const float y = PLANES == 2 && a.rms ? v[r] * scale[r] : v[r];
        if constexpr (PLANES == 1) {
          if (r < a.rows_total) a.out[static_cast<size_t>(r) * a.out_ld + f] = y;
        } else if (a.last_only) {
          if ((sr.last >> r) & 1u) a.out[sr.grp[r] * a.out_group_stride + f] = y;
        } else if ((sr.valid >> r) & 1u) {
          a.out[static_cast<size_t>(r) * a.out_ld + f] = y;
        }
      }
    }
    return;
  }
#pragma unroll
  for (int r = 0; r < 8; ++r) stage[r * kStageLd + et] = v[r];
  named_bar_sync(1, 128);
  const int r = et >> 4, c4 = 4 * (et & 15);
  const float* row = stage + r * kStageLd;
  float x[2][4];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const float4 t = *reinterpret_cast<const float4*>(row + 64 * q + c4);
    const float sc = a.rms ? scale[r] : 1.f;
    x[q][0] = t.x * sc;
    x[q][1] = t.y * sc;
    x[q][2] = t.z * sc;
    x[q][3] = t.w * sc;
  }
  const bool store = r < a.rows_total && !dry;
  if constexpr (EPI == EPI_RESIDUAL) {   // n_out is a multiple of 128 (d_model)
    float sq = 0.f;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float hv[4] = {pre.h[q].x, pre.h[q].y, pre.h[q].z, pre.h[q].w};
      float g[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        x[q][i] += hv[i];
        sq += x[q][i] * x[q][i];
        g[i] = x[q][i] * bf_at(pre.gain[q], i);
      }
      const size_t o = static_cast<size_t>(r) * a.h_ld + rt * kTileM + 64 * q + c4;
      if (store) {
        *reinterpret_cast<float4*>(a.h + o) = make_float4(x[q][0], x[q][1], x[q][2], x[q][3]);
        if (a.gain_next != nullptr) store_split4(a.xg_out + o, a.xg_lo_out + o, g);
      }
    }
    trace_at(ts, 12);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (store && c4 == 0) a.ss_out[static_cast<size_t>(rt) * a.ss_stride + r] = sq;
  }
  if constexpr (EPI == EPI_SWIGLU) {   // features 0..63 of the tile are gate rows, 64..127 the same up rows
    float y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) y[i] = x[0][i] / (1.0f + expf(-x[0][i])) * x[1][i];
    const int fo = rt * 64 + c4;   // n_out (d_ffn) is a multiple of 8
    const size_t o = static_cast<size_t>(r) * a.act_ld + fo;
    if (store && fo < a.n_out) store_split4(a.act + o, a.act_lo + o, y);
  }
  if constexpr (EPI == EPI_QKV) {   // RoPE on q and k, K/V appended to the cache; a tile is all q, k or v
    const int f0 = rt * kTileM, hd = a.head_dim;
    const int seg = f0 < a.q_dim ? 0 : (f0 < a.q_dim + a.kv_dim ? 1 : 2);
    const int fs = f0 - (seg == 0 ? 0 : (seg == 1 ? a.q_dim : a.q_dim + a.kv_dim));
    if (seg < 2) {
      if (hd == 128) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float c = sr.rc[r][c4 + i], s = sr.rs[r][c4 + i], lo = x[0][i], hi = x[1][i];
          x[0][i] = lo * c - hi * s;
          x[1][i] = lo * s + hi * c;
        }
      } else {   // 64: features 64 q + c4 + i, partner 32 away
        const float sc = a.rms ? scale[r] : 1.f;
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int ip = (c4 + i) & 31;
            const float c = sr.rc[r][ip], s = sr.rs[r][ip], o = row[64 * q + ((c4 + i) ^ 32)] * sc;
            x[q][i] = c4 < 32 ? x[q][i] * c - o * s : o * s + x[q][i] * c;
          }
      }
    }
    const int pos = sr.pos[r];
    // invalid positions were flagged by the embedding kernel: skip the row
    if (!dry && ((sr.valid >> r) & 1u) && pos >= 0 && pos < a.max_seq) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int d = fs + 64 * q + c4;   // within q, k or v
        if (seg == 0) {
          *reinterpret_cast<float4*>(a.q_out + static_cast<size_t>(r) * a.q_dim + d) =
              make_float4(x[q][0], x[q][1], x[q][2], x[q][3]);
        } else {
          const int head = d / hd;
          bf16* cache = (seg == 1 ? a.kcache : a.vcache) +
                        ((static_cast<size_t>(sr.req[r]) * a.n_kv_heads + head) * a.max_seq + pos) * hd + (d - head * hd);
          *reinterpret_cast<uint2*>(cache) = pack_bf16x4(x[q][0], x[q][1], x[q][2], x[q][3]);
        }
      }
    }
  }
  named_bar_sync(1, 128);   // stage is reused by the next tile
}

// Partial of slot `slot` (2 CTA + (0: the CTA's first row tile, 1: its last)): rows
// 4 q .. 4 q + 3 of feature et, a warp's accesses contiguous.
template <int NR>
__device__ __forceinline__ float* part_ptr(const GemmArgs& a, int slot, int q, int et) {
  return a.partials + (static_cast<size_t>(slot) * (NR / 4) + q) * (kTileM * 4) + et * 4;
}

template <int EPI, bool CSK, int PLANES>
__global__ void __launch_bounds__(kThreads, 1) gemm_small_kernel(const __grid_constant__ GemmArgs a) {
  constexpr int NR = rows_of<PLANES>();
  __shared__ SmallCtl ctl;
  extern __shared__ uint8_t dsmem_raw[];
  uint8_t* dsmem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(dsmem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int S = a.stages;
  uint8_t* smem_a = dsmem;
  uint8_t* smem_b = dsmem + static_cast<size_t>(S) * kABytes;
  float* stage = reinterpret_cast<float*>(smem_b + static_cast<size_t>(S) * kBBytes);   // [8][kStageLd]
  SmallRows& sr = *reinterpret_cast<SmallRows*>(stage + 8 * kStageLd);
  float* recv = reinterpret_cast<float*>(
      (reinterpret_cast<uintptr_t>(&sr + 1) + 15) & ~static_cast<uintptr_t>(15));       // [csk - 1][NR / 4][128][4]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int KT = a.k_tiles, T = a.row_tiles * KT;
  const int G = gridDim.x, c = blockIdx.x;
  const int t_begin = sk_begin(c, T, G), t_end = sk_begin(c + 1, T, G);
  constexpr uint32_t kTmemCols = 32;   // two accumulators of 16 columns

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
    mbar_init(&ctl.recv, 1);
    ctl.recv_pending = 0;
    ctl.abort_flag = 0;
    ctl.reduce_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    __syncwarp();
    tmem_alloc(&ctl.tmem_base, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // the barriers above are initialised before any peer pushes (every thread arrives
  // here; a thread waits before its first push)
  if constexpr (CSK) cluster_arrive_release();
  const uint32_t tmem_base = ctl.tmem_base;
  // optional trace (16 slots per CTA): 0 entry, 13 dependency released,
  // 2 activation loads issued, 3 first MMA, 4..12 epilogue, 1 exit
  unsigned long long* trace = a.trace != nullptr ? a.trace + blockIdx.x * 16 : nullptr;
  if (threadIdx.x == 64) trace_at(trace, 0);
  volatile int* abort_flag = &ctl.abort_flag;

  if (warp == 0) {
    // ------------------------------------------------ copies
    if (lane == 0) {
      if (a.a_packed == nullptr) tma_prefetch_desc(&a.map_a);
      tma_prefetch_desc(&a.map_b);
      tma_prefetch_desc(&a.map_b2);
      const uint64_t pol = a.l2_hint == L2_EVICT_FIRST ? l2_policy_evict_first() : l2_policy_evict_normal();
      const uint64_t pol_b = l2_policy_evict_last();   // activations are re-read by every CTA
      uint32_t issued_mask = 0, last_par = 0;
      bool ok = true;
      const int n_pre = min(S, t_end - t_begin);
      const uint8_t* wsrc = a.a_packed != nullptr ? a.a_packed + static_cast<size_t>(t_begin) * kABytes : nullptr;
      int rt = t_begin / KT, kt = t_begin - rt * KT;
      auto load_a = [&](int slot) {
        uint8_t* dst = smem_a + static_cast<size_t>(slot) * kABytes;
        if (wsrc != nullptr) {
          bulk_load(dst, wsrc, kABytes, &ctl.full[slot], pol);
          wsrc += kABytes;
        } else {
          tma_load_2d(dst, &a.map_a, kt * kTileK, rt * kTileM, &ctl.full[slot], pol);
        }
      };
      // activations of one k tile (4-D map map_b, or where k is not whole k tiles two
      // 2-D maps map_b, map_b2 of a plane each), or of kXGroup (4-D map map_b2)
      auto load_b = [&](int slot, int k_tile) {
        uint8_t* dst = smem_b + static_cast<size_t>(slot) * kBBytes;
        if (a.x4d) {
          tma_load_4d(dst, &a.map_b, 0, 0, 0, k_tile, &ctl.full[slot], pol_b);
        } else {
          tma_load_2d(dst, &a.map_b, k_tile * kTileK, 0, &ctl.full[slot], pol_b);
          if (PLANES == 2) tma_load_2d(dst + kBBytes / 2, &a.map_b2, k_tile * kTileK, 0, &ctl.full[slot], pol_b);
        }
      };
      auto group_at = [&](int p, int k_tile) {   // k tiles of the box that starts at stage p of the first fill
        return a.x4d && p + kXGroup <= n_pre && k_tile + kXGroup <= KT ? kXGroup : 1;
      };
      auto next_tile = [&] {
        if (++kt == KT) {
          kt = 0;
          ++rt;
        }
      };
      // first fill: the weights do not depend on earlier launches and are requested
      // before the wait (a group's activations complete on its first stage's barrier:
      // stages are read in order)
      const int kt_first = kt;
      if (a.w_after_wait) pdl_wait();
      for (int p = 0, left = 0; p < n_pre; ++p) {
        uint32_t bytes = kABytes;
        if (left == 0) {
          left = group_at(p, kt);
          bytes += left * kBBytes;
        }
        --left;
        mbar_arrive_expect_tx(&ctl.full[p], bytes);
        load_a(p);
        issued_mask |= 1u << p;
        next_tile();
      }
      pdl_wait();
      pdl_launch_dependents();   // after the wait: see ptx.cuh
      trace_at(trace, 2);
      for (int p = 0, k2 = kt_first; p < n_pre;) {
        const int n = group_at(p, k2);
        if (n > 1)
          tma_load_4d(smem_b + static_cast<size_t>(p) * kBBytes, &a.map_b2, 0, 0, 0, k2, &ctl.full[p], pol_b);
        else
          load_b(p, k2);
        p += n;
        k2 += n;
        if (k2 == KT) k2 = 0;
      }
      int s = n_pre == S ? 0 : n_pre;
      uint32_t ph = n_pre == S ? 1u : 0u;   // phase of the fill the next wait is for
      for (int t = t_begin + n_pre; t < t_end; ++t) {
        if (!mbar_wait_bounded(&ctl.empty[s], ph ^ 1u, abort_flag, a.status)) {
          ok = false;
          break;
        }
        mbar_arrive_expect_tx(&ctl.full[s], kABytes + kBBytes);
        load_a(s);
        load_b(s, kt);
        issued_mask |= 1u << s;
        last_par = (last_par & ~(1u << s)) | (ph << s);
        next_tile();
        if (++s == S) {
          s = 0;
          ph ^= 1u;
        }
      }
      if (!ok) {   // every copy in flight lands before the CTA leaves
        for (int q = 0; q < S; ++q)
          if (issued_mask & (1u << q)) mbar_wait_drain(&ctl.full[q], (last_par >> q) & 1u);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer
    // The whole warp walks the tiles and one elected lane issues, so that descriptors
    // and loop counters stay in uniform registers.
    const bool lead = elect_one();
    const uint32_t idesc = make_idesc_bf16_f32(kTileM, kN);
    const uint64_t adesc0 = make_smem_desc_sw128(smem_addr(smem_a));
    const uint64_t bdesc0 = make_smem_desc_sw128(smem_addr(smem_b));
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
      const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(buf * kN);
      for (int tt = t; tt < seg_end; ++tt) {
        ok = __all_sync(0xffffffffu, mbar_wait_bounded(&ctl.full[s], ph, abort_flag, a.status));
        if (!ok) break;
        tc_fence_after();
        const uint64_t ad = adesc0 + static_cast<uint32_t>(s) * (kABytes >> 4);
        const uint64_t bd = bdesc0 + static_cast<uint32_t>(s) * (kBBytes >> 4);
        const uint32_t acc0 = tt > t ? 1u : 0u;
        if (lead) {
          if (tt == t_begin) trace_at(trace, 3);
#pragma unroll
          for (int kk = 0; kk < kTileK / 16; ++kk)
            tc_mma_bf16(d_tmem, ad + 2 * kk, bd + 2 * kk, idesc, kk > 0 ? 1u : acc0);
          if (tt + S < t_end) tc_commit(&ctl.empty[s]);   // else the slot is not filled again
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
    if (!ok && lead) {   // wait for every MMA already issued
      tc_commit(&ctl.drain);
      mbar_wait_drain(&ctl.drain, 0);
    }
  } else {
    // ------------------------------------------------ epilogue (warps 2-5)
    // a warp may only read TMEM lanes 32*(warp % 4) .. +31: that is its feature block
    const int ew = warp & 3;
    const int et = ew * 32 + lane;   // tile feature == TMEM lane
    unsigned long long* ts = threadIdx.x == 64 ? trace : nullptr;
    // cluster exchange: the first contributor of the row tile this range ends in
    // expects its peers' partials (arrival count 1: this arrive; bytes may land first)
    if (CSK && t_end > t_begin && threadIdx.x == 64) {
      const int rt_last = (t_end - 1) / KT;
      const int cf = sk_cta_of(rt_last * KT, T, G), cl = sk_cta_of((rt_last + 1) * KT - 1, T, G);
      if (cf == c && cl > c && cf / a.csk == cl / a.csk) {
        mbar_arrive_expect_tx(&ctl.recv, static_cast<uint32_t>((cl - cf) * kTileM * NR * 4));
        ctl.recv_pending = 1;
      }
    }
    float v[NR];
    EpiPre pre;
    if (a.ctx_early) small_rows<EPI>(a, sr, et);
    // The first turn of the loop is a dry run of the epilogue while the previous launch
    // ends: the code runs once per tile, and cold its instructions are fetched one miss
    // after another.
    if (!a.ctx_early) {   // the plan is not final yet: stand-ins
      if (et < 8) sr.pos[et] = sr.req[et] = sr.grp[et] = 0;
      if (et == 0) sr.valid = sr.last = 0u;
    }
    if (et < 8) ctl.scale[et] = 0.f;
    named_bar_sync(1, 128);
#pragma unroll
    for (int r = 0; r < NR; ++r) v[r] = 0.f;
    pre.h[0] = pre.h[1] = make_float4(0.f, 0.f, 0.f, 0.f);
    pre.gain[0] = pre.gain[1] = make_uint2(0u, 0u);
    int t = t_begin;
    for (int seg = -1;; ++seg) {
      int rt = 0;
      bool finish = true;          // this CTA runs the tile's epilogue
      if (seg >= 0) {
        if (t >= t_end) break;
        rt = t / KT;
        const int k0 = t - rt * KT;
        const int seg_end = min(t_end, (rt + 1) * KT);
        const bool full = k0 == 0 && seg_end == (rt + 1) * KT;
        const int c_first = sk_cta_of(rt * KT, T, G), c_last = sk_cta_of((rt + 1) * KT - 1, T, G);
        const bool dsm = CSK && !full && c_first / a.csk == c_last / a.csk;
        const int buf = seg & 1;
        small_pre<EPI>(a, rt, et, pre);
        if (threadIdx.x == 64)
          ctl.wait_ok =
              mbar_wait_bounded(&ctl.acc_full[buf], static_cast<uint32_t>(seg >> 1) & 1u, abort_flag, a.status) ? 1 : 0;
        named_bar_sync(1, 128);
        const int ok = ctl.wait_ok;
        named_bar_sync(1, 128);
        if (!ok) break;
        tc_fence_after();
        {
          float d[kN];
          tmem_ld_32x32b_x16(tmem_base + (static_cast<uint32_t>(ew * 32) << 16) + static_cast<uint32_t>(buf * kN), d);
#pragma unroll
          for (int r = 0; r < NR; ++r) v[r] = PLANES == 2 ? d[r] + d[(8 + r) % kN] : d[r];
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl.acc_empty[buf]);
        t = seg_end;
        if (CSK && dsm) {
          trace_at(ts, 4);
          if (c != c_first) {
            const uint32_t rank = static_cast<uint32_t>(c_first % a.csk);
            float* slot = recv + static_cast<size_t>(c - c_first - 1) * kTileM * NR + et * 4;
            const uint32_t raddr = mapa_shared(smem_addr(slot), rank);
            const uint32_t rbar = mapa_shared(smem_addr(&ctl.recv), rank);
#pragma unroll
            for (int q = 0; q < NR / 4; ++q)
              st_async_f4(raddr + q * kTileM * 16, v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3], rbar);
            finish = false;
          } else {
            // every thread acquires the peers' bytes itself; a wait that runs out ends
            // the epilogue of the whole CTA
            const bool got = mbar_wait_cluster_bounded(&ctl.recv, 0, abort_flag, a.status);
            if (!got) ctl.wait_ok = 0;
            named_bar_sync(1, 128);
            if (!ctl.wait_ok) break;
            trace_at(ts, 5);
            for (int k = 0; k < c_last - c_first; ++k) {
              const float* src = recv + static_cast<size_t>(k) * kTileM * NR + et * 4;
#pragma unroll
              for (int q = 0; q < NR / 4; ++q) {
                const float4 x = *reinterpret_cast<const float4*>(src + q * kTileM * 4);
                v[4 * q] += x.x;
                v[4 * q + 1] += x.y;
                v[4 * q + 2] += x.z;
                v[4 * q + 3] += x.w;
              }
            }
          }
        } else if (!full) {
#pragma unroll
          for (int q = 0; q < NR / 4; ++q)
            *reinterpret_cast<float4*>(part_ptr<NR>(a, 2 * c + (seg == 0 ? 0 : 1), q, et)) =
                make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
          trace_at(ts, 4);
          // The barrier orders this CTA's partial stores before thread 0's arrival, whose
          // release (acq_rel, GPU scope) publishes them; the last contributor's acquire
          // and the second barrier order every other contributor's partials before its
          // loads (which bypass L1).
          named_bar_sync(1, 128);
          if (et == 0) {
            // counted at the first contributor, whose range ends in this tile: no other
            // split tile has the same one
            ctl.reduce_flag = atom_add_acq_rel_gpu(&a.counters[c_first], 1) == c_last - c_first ? 1 : 0;
            if (ctl.reduce_flag) a.counters[c_first] = 0;
          }
          named_bar_sync(1, 128);
          trace_at(ts, 5);
          finish = ctl.reduce_flag != 0;
          if (finish) {
            // ascending CTA order, two contributors fetched at once
            float sum[NR];
#pragma unroll
            for (int r = 0; r < NR; ++r) sum[r] = 0.f;
            for (int cc0 = c_first; cc0 <= c_last; cc0 += 2) {
              float4 x[2][NR / 4];
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                const int cc = min(cc0 + i, c_last);
                const int sl = sk_begin(cc, T, G) >= rt * KT ? 0 : 1;
#pragma unroll
                for (int q = 0; q < NR / 4; ++q) x[i][q] = ld_cg_f4(part_ptr<NR>(a, 2 * cc + sl, q, et));
              }
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                if (cc0 + i > c_last) break;
#pragma unroll
                for (int q = 0; q < NR / 4; ++q) {
                  sum[4 * q] += x[i][q].x;
                  sum[4 * q + 1] += x[i][q].y;
                  sum[4 * q + 2] += x[i][q].z;
                  sum[4 * q + 3] += x[i][q].w;
                }
              }
            }
#pragma unroll
            for (int r = 0; r < NR; ++r) v[r] = sum[r];
          }
        }
        if (finish && ts != nullptr) trace_after(ts, 6, v[0] + v[NR - 1]);
      }
      if (finish) small_epilogue<EPI, PLANES>(a, sr, ctl.scale, stage, rt, et, v, pre, seg >= 0 ? ts : nullptr, seg < 0);
      if (seg >= 0) {
        trace_at(ts, 7);
        continue;
      }
      pdl_wait();
      if constexpr (CSK) cluster_wait_acquire();
      trace_at(ts, 13);
      if (PLANES == 2 && a.rms) small_scales(a, ctl.scale, et);
      if (!a.ctx_early) small_rows<EPI>(a, sr, et);
      named_bar_sync(1, 128);
    }
  }

  // a CTA that expects pushed partials leaves only after they landed (they do at
  // once unless a peer stopped early; the wait is bounded)
  if constexpr (CSK) {
    if (threadIdx.x == 64 && ctl.recv_pending) mbar_wait_drain(&ctl.recv, 0);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
  if (threadIdx.x == 64) trace_at(trace, 1);
}

constexpr int kSmallSmem = 212 * 1024;

int small_fixed_bytes(int planes, int csk) {
  return 1024 + 8 * (kTileM + 4) * 4 + static_cast<int>(sizeof(SmallRows)) +
         (csk > 1 ? (csk - 1) * kTileM * (planes == 2 ? 8 : 16) * 4 + 16 : 0);
}

template <bool CSK>
const void* small_kernel_for(int epi, int planes) {
  if (planes == 1)
    return epi == EPI_F32 ? reinterpret_cast<const void*>(gemm_small_kernel<EPI_F32, CSK, 1>) : nullptr;
  switch (epi) {
    case EPI_F32: return reinterpret_cast<const void*>(gemm_small_kernel<EPI_F32, CSK, 2>);
    case EPI_RESIDUAL: return reinterpret_cast<const void*>(gemm_small_kernel<EPI_RESIDUAL, CSK, 2>);
    case EPI_SWIGLU: return reinterpret_cast<const void*>(gemm_small_kernel<EPI_SWIGLU, CSK, 2>);
    case EPI_QKV: return reinterpret_cast<const void*>(gemm_small_kernel<EPI_QKV, CSK, 2>);
    default: return nullptr;
  }
}

void cluster_attr(cudaLaunchAttribute* attr, int csk) {
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = csk;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
}

}  // namespace

int gemm_small_stages(int planes, int csk) {
  const int budget = 200 * 1024 - small_fixed_bytes(planes, csk);
  const int s = budget / (kABytes + kBBytes);
  return s < kSmallStages ? s : kSmallStages;
}

size_t gemm_small_smem(int planes, int csk) {
  return static_cast<size_t>(gemm_small_stages(planes, csk)) * (kABytes + kBBytes) + small_fixed_bytes(planes, csk);
}

int gemm_small_x_group() { return kXGroup; }

cudaError_t gemm_small_set_max_smem() {
  for (int planes = 1; planes <= 2; ++planes)
    for (int epi : {EPI_F32, EPI_RESIDUAL, EPI_SWIGLU, EPI_QKV})
      for (const void* f : {small_kernel_for<false>(epi, planes), small_kernel_for<true>(epi, planes)}) {
        if (f == nullptr) continue;
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmem);
        if (e != cudaSuccess) return e;
      }
  return cudaSuccess;
}

int gemm_small_max_clusters(int epi, int planes, int csk) {
  const void* fn = small_kernel_for<true>(epi, planes);
  if (fn == nullptr || csk < 2 || csk > 8) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(csk);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = gemm_small_smem(planes, csk);
  cudaLaunchAttribute attr[1];
  cluster_attr(attr, csk);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t launch_gemm_small(const GemmArgs& a, int grid, cudaStream_t s, bool pdl) {
  const int planes = a.split ? 2 : 1;
  const void* fn = a.csk > 1 ? small_kernel_for<true>(a.epi, planes) : small_kernel_for<false>(a.epi, planes);
  if (fn == nullptr || a.rows_total < 1 || a.rows_total > (planes == 2 ? 8 : 16) || a.n_pad != kN ||
      (a.pair && a.a_packed == nullptr) || (a.csk > 1 && (a.csk > 8 || grid % a.csk != 0)))
    return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = gemm_small_smem(planes, a.csk);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int n_attr = 0;
  if (pdl) {
    attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
    ++n_attr;
  }
  if (a.csk > 1) cluster_attr(&attr[n_attr++], a.csk);
  cfg.attrs = attr;
  cfg.numAttrs = n_attr;
  GemmArgs args = a;
  void* params[] = {&args};
  return cudaLaunchKernelExC(&cfg, fn, params);
}

}  // namespace memspec
