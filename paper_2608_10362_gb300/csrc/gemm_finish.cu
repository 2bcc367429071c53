// gemm_finish.cu - the second launch of a GEMM over more activation rows than
// gemm_small.cu takes: sums the stream-K partials of a row tile and runs the epilogue.
//
// CTA (row tile, 16-row chunk), 128 threads; the sums are formed with a thread per
// feature of the tile, then the tile is turned in shared memory and a thread finishes
// four times four (SwiGLU: eight) features of one row with wide loads and stores.  One
// CTA folding every chunk of a tile in turn would hold the GEMM for tens of
// microseconds past its last MMA; here the whole chip does it.  Bound by latency:
// everything that is final before the GEMM ends - the chunk's rows of the row plan,
// the RoPE table - is read before griddepcontrol.wait, everything else in one round
// trip to L2 after it.
// Many rows are bound by issue slots and latency together (7B, 256 rows, gate/up: 2752
// CTAs, 14 us, 34 MB).  Turned, with 8 to 16 bytes per access, against a thread per
// feature with 2 and 4: 2047 prompt tokens of the 7B 48.9 -> 47.5 ms, the 8B verify of
// 144 rows 5.64 -> 5.61.
// Tried instead: fewer CTAs that take several chunks in turn (7B prefill 49.1 -> 49.8
// to 61 ms with 16 to 3 CTAs per SM).
#include <cuda_bf16.h>

#include "gemm_epi.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace memspec {

namespace {

using namespace gemm;

constexpr int kRows = 16;          // rows of a chunk
constexpr int kPitch = kRows + 1;  // staged tile: [128 features][16 rows], padded

// The chunk's rows of the row plan.
struct ChunkRows {
  int pos[kRows], rpos[kRows], req[kRows], grp[kRows];
  uint32_t valid, last;   // bit j: row j is valid / the last valid row of its group
};

__device__ __forceinline__ void chunk_rows(const GemmArgs& a, ChunkRows& cr, int r0, int lane) {
  // lanes 0..15 of warp 0
  const RowPlan* plan = a.plan;
  const int r = r0 + (lane & 15);
  bool valid = false, last = false;
  int g = 0, pos = 0, rpos = 0, req = 0;
  if (r < a.rows_total) {
    if (plan == nullptr) {
      valid = true;
    } else {
      const int R = plan->rows_per_group;
      g = r / R;
      const int i = r - g * R;
      const int nv = plan->valid[g];
      valid = i < nv;
      last = i == nv - 1;
      pos = plan->pos0[g] + i;
      rpos = (plan->tree && i < kTreeRows) ? plan->pos0[g] + plan->rope_off[i] : pos;
      req = plan->req[g];
    }
  }
  const uint32_t vb = __ballot_sync(0xffffffffu, valid), lb = __ballot_sync(0xffffffffu, last);
  if (lane < kRows) {
    cr.pos[lane] = pos;
    cr.rpos[lane] = rpos;
    cr.req[lane] = req;
    cr.grp[lane] = g;
  }
  if (lane == 0) {
    cr.valid = vb & 0xffffu;
    cr.last = lb & 0xffffu;
  }
}

__device__ __forceinline__ float bf_lo(uint32_t x) { return __uint_as_float(x << 16); }
__device__ __forceinline__ float bf_hi(uint32_t x) { return __uint_as_float(x & 0xffff0000u); }
// Four neighbours, hi and (unless null) lo plane, 8 bytes each.
__device__ __forceinline__ void store4(bf16* hi_p, bf16* lo_p, float a, float b, float c, float d) {
  const float y[4] = {a, b, c, d};
  __nv_bfloat16 h[4], l[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) split_bf16(y[e], h[e], l[e]);
  *reinterpret_cast<uint2*>(hi_p) = *reinterpret_cast<const uint2*>(h);
  if (lo_p != nullptr) *reinterpret_cast<uint2*>(lo_p) = *reinterpret_cast<const uint2*>(l);
}

template <int EPI>
__global__ void __launch_bounds__(128, EPI == EPI_QKV || EPI == EPI_RESIDUAL ? 6 : 8)
gemm_split_epi_kernel(const __grid_constant__ GemmArgs a, int gemm_grid) {
  __shared__ ChunkRows cr;
  __shared__ float stage[EPI == EPI_F32 ? 1 : kTileM * kPitch];
  __shared__ float scale[kRows];
  __shared__ float red[4][kRows];
  const int rt = blockIdx.x, chunk = blockIdx.y, et = threadIdx.x;
  const int warp = et >> 5, lane = et & 31;
  const int KT = a.k_tiles, G = gemm_grid, r0 = chunk * kRows;
  const int nr = min(kRows, a.rows_total - r0);   // rows of the chunk
  // stream-K tiles: row tiles, or (gemm_pair.cu, G its CTA pairs) pairs of them
  const int T = (a.pairs ? (a.row_tiles + 1) / 2 : a.row_tiles) * KT, unit = a.pairs ? rt >> 1 : rt;
  const int c_first = sk_cta_of(unit * KT, T, G), c_last = sk_cta_of((unit + 1) * KT - 1, T, G);
  // optional trace (a.trace: 16 slots per CTA, CTAs in launch order up to the row's
  // width): 0 entry, 13 dependency released, 2 partials summed, 1 done
  const int lin = blockIdx.y * gridDim.x + blockIdx.x;
  unsigned long long* ts = (a.trace != nullptr && et == 0 && lin < a.trace_ctas) ? a.trace + lin * 16 : nullptr;
  trace_at(ts, 0);
  // row tiles that a CTA owned whole were finished by it (gemm_pair.cu: with the
  // fp32-output epilogue only)
  if ((!a.pairs || EPI == EPI_F32) && c_first == c_last) return;
  if (!a.ctx_early) pdl_wait();
  if (warp == 0) chunk_rows(a, cr, r0, lane);
  // this thread's feature
  const int f = rt * kTileM + et;
  // the turned tile: row tr of the chunk, features 4 tq + 32 i .. + 3 of the tile
  const int tr = et >> 3, tq = et & 7;
  [[maybe_unused]] uint2 gain[4];
  if constexpr (EPI == EPI_RESIDUAL) {
    if (a.gain_next != nullptr)   // weights: never written
#pragma unroll
      for (int i = 0; i < 4; ++i)
        gain[i] = *reinterpret_cast<const uint2*>(a.gain_next + rt * kTileM + 4 * tq + 32 * i);
  }
  // QKV: segment (q, k, v) and first head of the tile (segments are whole tiles), and
  // the row's rotations; at hd 64 the tile holds two heads
  [[maybe_unused]] int seg = 0, fs = 0;
  [[maybe_unused]] float4 rc[2], rs[2];
  if constexpr (EPI == EPI_QKV) {
    const int f0 = rt * kTileM, half = a.head_dim >> 1;
    seg = f0 < a.q_dim ? 0 : (f0 < a.q_dim + a.kv_dim ? 1 : 2);
    fs = f0 - (seg == 0 ? 0 : (seg == 1 ? a.q_dim : a.q_dim + a.kv_dim));
    __syncthreads();
    const int pos = cr.pos[tr];
    const bool ok = seg < 2 && ((cr.valid >> tr) & 1u) && pos >= 0 && pos < a.max_seq;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      rc[i] = rs[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (ok && 32 * i < half) {
        const size_t ri = static_cast<size_t>(cr.rpos[tr]) * half + 4 * tq + 32 * i;
        rc[i] = *reinterpret_cast<const float4*>(a.rope_cos + ri);
        rs[i] = *reinterpret_cast<const float4*>(a.rope_sin + ri);
      }
    }
  }
  if (a.ctx_early) pdl_wait();
  pdl_launch_dependents();   // after the wait: see ptx.cuh
  trace_at(ts, 13);
  // ---- one round trip: sums of squares, residual rows, partials
  float ss = 0.f;
  if (a.rms) {   // thread (row et % 16, part et / 16): every eighth partial sum of the row
    const int r = r0 + (et & 15);
    float t[4];
    for (int i0 = et >> 4; i0 < a.ss_count; i0 += 32) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        t[q] = (r < a.rows_total && i0 + 8 * q < a.ss_count)
                   ? __ldcg(a.ss + static_cast<size_t>(i0 + 8 * q) * a.ss_stride + r)
                   : 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q) ss += t[q];
    }
  }
  [[maybe_unused]] float4 h[4];
  if constexpr (EPI == EPI_RESIDUAL) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      h[i] = tr < nr ? ld_cg_f4(a.h + static_cast<size_t>(r0 + tr) * a.h_ld + rt * kTileM + 4 * tq + 32 * i)
                     : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float v[kRows];
  reduce_partials<2>(a, rt, c_first, c_last, chunk, et, T, G, v);
  if (ts != nullptr) trace_after(ts, 2, v[0] + v[15]);
  if (a.rms) {
    // parts of a row: lanes l and l + 16, then the warps in order
    ss += __shfl_xor_sync(0xffffffffu, ss, 16);
    if (lane < kRows) red[warp][lane] = ss;
    __syncthreads();
    if (et < kRows)
      scale[et] = rsqrtf((((red[0][et] + red[1][et]) + red[2][et]) + red[3][et]) / static_cast<float>(a.k_in) + a.eps);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kRows; ++j) v[j] *= scale[j];
  } else {
    __syncthreads();   // cr
  }

  if constexpr (EPI == EPI_F32) {
    if (f < a.n_out) {
#pragma unroll
      for (int j = 0; j < kRows; ++j) {
        if (a.last_only) {
          if ((cr.last >> j) & 1u) a.out[cr.grp[j] * a.out_group_stride + f] = v[j];
        } else if ((cr.valid >> j) & 1u) {
          a.out[static_cast<size_t>(r0 + j) * a.out_ld + f] = v[j];
        }
      }
    }
  }
  if constexpr (EPI != EPI_F32) {
#pragma unroll
    for (int j = 0; j < kRows; ++j) stage[et * kPitch + j] = v[j];
    __syncthreads();
  }
  // features 4 tq + 32 i + (0..3) of row tr
  [[maybe_unused]] auto turned = [&](int i) {
    const float* s = stage + (4 * tq + 32 * i) * kPitch + tr;
    return make_float4(s[0], s[kPitch], s[2 * kPitch], s[3 * kPitch]);
  };
  if constexpr (EPI == EPI_RESIDUAL) {   // n_out is a multiple of 128 (d_model)
    float sq = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 x = turned(i);
      h[i].x += x.x;
      h[i].y += x.y;
      h[i].z += x.z;
      h[i].w += x.w;
      sq += (h[i].x * h[i].x + h[i].y * h[i].y) + (h[i].z * h[i].z + h[i].w * h[i].w);
      if (tr < nr) {
        const size_t o = static_cast<size_t>(r0 + tr) * a.h_ld + rt * kTileM + 4 * tq + 32 * i;
        *reinterpret_cast<float4*>(a.h + o) = h[i];
        if (a.gain_next != nullptr)
          store4(a.xg_out + o, a.xg_lo_out != nullptr ? a.xg_lo_out + o : nullptr, h[i].x * bf_lo(gain[i].x),
                 h[i].y * bf_hi(gain[i].x), h[i].z * bf_lo(gain[i].y), h[i].w * bf_hi(gain[i].y));
      }
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (tq == 0 && tr < nr) a.ss_out[static_cast<size_t>(rt) * a.ss_stride + r0 + tr] = sq;
  }
  if constexpr (EPI == EPI_SWIGLU) {
    // features 0..63 of the tile are gate rows, 64..127 the same up rows; a thread
    // finishes features 4 tq + 32 i of its row, i = 0, 1
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int fo = rt * 64 + 4 * tq + 32 * i;
      const float4 g = turned(i), u = turned(i + 2);
      auto act = [](float x, float y) { return x / (1.0f + expf(-x)) * y; };
      if (tr < nr && fo < a.n_out) {
        const size_t o = static_cast<size_t>(r0 + tr) * a.act_ld + fo;
        const float y[4] = {act(g.x, u.x), act(g.y, u.y), act(g.z, u.z), act(g.w, u.w)};
        bf16* lo = a.act_lo != nullptr ? a.act_lo + o : nullptr;
        if (fo + 3 < a.n_out && (a.act_ld & 3) == 0)
          store4(a.act + o, lo, y[0], y[1], y[2], y[3]);
        else
          for (int e = 0; e < 4 && fo + e < a.n_out; ++e)
            store_split_bf16(a.act + o + e, lo != nullptr ? lo + e : nullptr, y[e]);
      }
    }
  }
  if constexpr (EPI == EPI_QKV) {   // RoPE on q and k, K/V appended to the cache
    const int pos = cr.pos[tr];
    // invalid positions were flagged by the embedding kernel: skip the row
    if (((cr.valid >> tr) & 1u) && pos >= 0 && pos < a.max_seq) {
      bf16* cache = seg == 1 ? a.kcache : a.vcache;
      const int step = a.head_dim >> 6;   // half a head, in groups of 32 features
      float4 x[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] = turned(i);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float4 y = x[i];
        if (seg < 2) {
          const bool lo = (i & step) == 0;
          const float4 p = step == 1 ? x[i ^ 1] : x[i ^ 2];
          const float4 c = step == 1 ? rc[0] : rc[i & 1], n = step == 1 ? rs[0] : rs[i & 1];
          // low half: x c - x' s, high half: x' s + x c
          y.x = lo ? (x[i].x * c.x - p.x * n.x) : (p.x * n.x + x[i].x * c.x);
          y.y = lo ? (x[i].y * c.y - p.y * n.y) : (p.y * n.y + x[i].y * c.y);
          y.z = lo ? (x[i].z * c.z - p.z * n.z) : (p.z * n.z + x[i].z * c.z);
          y.w = lo ? (x[i].w * c.w - p.w * n.w) : (p.w * n.w + x[i].w * c.w);
        }
        const int ft = fs + 4 * tq + 32 * i;   // feature of the segment
        if (seg == 0) {
          *reinterpret_cast<float4*>(a.q_out + static_cast<size_t>(r0 + tr) * a.q_dim + ft) = y;
        } else {
          const int head = ft >> (step == 1 ? 6 : 7), dd = ft & (a.head_dim - 1);   // head_dim 64 or 128
          const __nv_bfloat162 b0 = __floats2bfloat162_rn(y.x, y.y), b1 = __floats2bfloat162_rn(y.z, y.w);
          *reinterpret_cast<uint2*>(
              cache + ((static_cast<size_t>(cr.req[tr]) * a.n_kv_heads + head) * a.max_seq + pos) * a.head_dim + dd) =
              make_uint2(*reinterpret_cast<const uint32_t*>(&b0), *reinterpret_cast<const uint32_t*>(&b1));
        }
      }
    }
  }
  trace_at(ts, 1);
}

}  // namespace

cudaError_t launch_gemm_split_epi(const GemmArgs& a, int gemm_grid, cudaStream_t s, bool pdl) {
  if (a.n_pad % 16 != 0 || a.n_pad > kMaxRows) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.row_tiles, (a.rows_total + kRows - 1) / kRows);
  cfg.blockDim = dim3(128);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  switch (a.epi) {
    case EPI_F32: return cudaLaunchKernelEx(&cfg, gemm_split_epi_kernel<EPI_F32>, a, gemm_grid);
    case EPI_RESIDUAL: return cudaLaunchKernelEx(&cfg, gemm_split_epi_kernel<EPI_RESIDUAL>, a, gemm_grid);
    case EPI_SWIGLU: return cudaLaunchKernelEx(&cfg, gemm_split_epi_kernel<EPI_SWIGLU>, a, gemm_grid);
    case EPI_QKV: return cudaLaunchKernelEx(&cfg, gemm_split_epi_kernel<EPI_QKV>, a, gemm_grid);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace memspec
