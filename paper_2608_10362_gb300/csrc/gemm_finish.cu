// gemm_finish.cu - the second launch of a GEMM over more than 16 activation rows:
// sums the stream-K partials of a row tile and runs the fused epilogue.
//
// CTA (row tile, 16-row chunk), 128 threads, thread = feature within the tile.  One
// CTA folding every chunk of a tile in turn would hold the GEMM for tens of
// microseconds past its last MMA; here the whole chip does it.  Bound by latency:
// everything that is final before the GEMM ends - the chunk's rows of the row plan,
// the RoPE table - is read before griddepcontrol.wait, everything else in one round
// trip to L2 after it.
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

template <int EPI>
__global__ void __launch_bounds__(128, EPI == EPI_QKV ? 5 : (EPI == EPI_RESIDUAL ? 6 : 8))
gemm_split_epi_kernel(const __grid_constant__ GemmArgs a, int gemm_grid) {
  __shared__ ChunkRows cr;
  __shared__ float stage[(EPI == EPI_QKV || EPI == EPI_SWIGLU) ? kTileM * kPitch : 1];
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
  [[maybe_unused]] float gain = 0.f;
  if constexpr (EPI == EPI_RESIDUAL) {
    if (a.gain_next != nullptr) gain = __bfloat162float(a.gain_next[f]);   // weights: never written
  }
  // QKV: segment (q, k, v), head, element of the head, rotation pair
  [[maybe_unused]] int seg = 0, head = 0, dd = 0, ip = 0;
  [[maybe_unused]] float rc[kRows], rs[kRows];
  if constexpr (EPI == EPI_QKV) {
    const int hd = a.head_dim;
    seg = f < a.q_dim ? 0 : (f < a.q_dim + a.kv_dim ? 1 : 2);
    const int fs = f - (seg == 0 ? 0 : (seg == 1 ? a.q_dim : a.q_dim + a.kv_dim));
    head = fs / hd;
    dd = fs - head * hd;
    ip = dd < hd / 2 ? dd : dd - hd / 2;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      const int pos = cr.pos[j];
      const bool ok = seg < 2 && ((cr.valid >> j) & 1u) && pos >= 0 && pos < a.max_seq;
      const size_t ri = ok ? static_cast<size_t>(cr.rpos[j]) * (hd >> 1) + ip : 0;
      rc[j] = seg < 2 ? a.rope_cos[ri] : 0.f;
      rs[j] = seg < 2 ? a.rope_sin[ri] : 0.f;
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
  [[maybe_unused]] float h[kRows];
  if constexpr (EPI == EPI_RESIDUAL) {
#pragma unroll
    for (int j = 0; j < kRows; ++j) h[j] = j < nr ? __ldcg(a.h + static_cast<size_t>(r0 + j) * a.h_ld + f) : 0.f;
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
  if constexpr (EPI == EPI_RESIDUAL) {   // n_out is a multiple of 128 (d_model)
    float sq[kRows];
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      h[j] += v[j];
      sq[j] = j < nr ? h[j] * h[j] : 0.f;
      if (j < nr) {
        const size_t o = static_cast<size_t>(r0 + j) * a.h_ld + f;
        a.h[o] = h[j];
        if (a.gain_next != nullptr)
          store_split_bf16(a.xg_out + o, a.xg_lo_out != nullptr ? a.xg_lo_out + o : nullptr, h[j] * gain);
      }
    }
    // the sixteen rows' sums over the warp's features together: each halving step
    // keeps half the rows, so lane l ends with row l / 2
    int row = 0;
#pragma unroll
    for (int o = 16, n = kRows; o > 1; o >>= 1, n >>= 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int j = 0; j < kRows / 2; ++j)
        if (j < n / 2) {
          const float give = up ? sq[j] : sq[j + n / 2];
          const float keep = up ? sq[j + n / 2] : sq[j];
          sq[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
      if (up) row += n / 2;
    }
    sq[0] += __shfl_xor_sync(0xffffffffu, sq[0], 1);
    if ((lane & 1) == 0) red[warp][row] = sq[0];
    __syncthreads();
    if (et < nr)
      a.ss_out[static_cast<size_t>(rt) * a.ss_stride + r0 + et] =
          ((red[0][et] + red[1][et]) + red[2][et]) + red[3][et];
  }
  if constexpr (EPI == EPI_SWIGLU) {
    // features 0..63 of the tile are gate rows, 64..127 the same up rows; thread
    // et < 64 finishes rows 0..7 of feature et, thread et + 64 rows 8..15
    const bool up = et >= 64;
    const int e = et & 63;
#pragma unroll
    for (int j = 0; j < 8; ++j) stage[et * kPitch + j] = up ? v[j] : v[8 + j];
    __syncthreads();
    const int fo = rt * 64 + e;
    if (fo < a.n_out) {
      const float* other = stage + (up ? e : e + 64) * kPitch;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int row = (up ? 8 : 0) + j;
        const float g = up ? other[j] : v[j], u = up ? v[8 + j] : other[j];
        if (row < nr) {
          const float y = g / (1.0f + expf(-g)) * u;
          const size_t o = static_cast<size_t>(r0 + row) * a.act_ld + fo;
          store_split_bf16(a.act + o, a.act_lo != nullptr ? a.act_lo + o : nullptr, y);
        }
      }
    }
  }
  if constexpr (EPI == EPI_QKV) {   // RoPE on q and k, K/V appended to the cache
#pragma unroll
    for (int j = 0; j < kRows; ++j) stage[et * kPitch + j] = v[j];
    __syncthreads();
    const int half = a.head_dim >> 1;
    const bool lo = dd < half;
    const float* other = stage + (lo ? et + half : et - half) * kPitch;   // seg < 2: in this tile
    bf16* cache = seg == 1 ? a.kcache : a.vcache;
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      const int pos = cr.pos[j];
      // invalid positions were flagged by the embedding kernel: skip the row
      if (!((cr.valid >> j) & 1u) || pos < 0 || pos >= a.max_seq) continue;
      float y = v[j];
      if (seg < 2) y = lo ? (v[j] * rc[j] - other[j] * rs[j]) : (other[j] * rs[j] + v[j] * rc[j]);
      if (seg == 0)
        a.q_out[static_cast<size_t>(r0 + j) * a.q_dim + f] = y;
      else
        cache[((static_cast<size_t>(cr.req[j]) * a.n_kv_heads + head) * a.max_seq + pos) * a.head_dim + dd] =
            __float2bfloat16_rn(y);
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
