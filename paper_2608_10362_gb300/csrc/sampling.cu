// sampling.cu - the draft-token sampler and the acceptance / resample / commit
// kernel (the latter's algorithm in sample_body.cuh).
//
// Sampler (draft tokens of the per-op passes, the rows of a tree step,
// memspec_op_sample): one cluster of C = 1, 2, 4 or 8 CTAs per row, each CTA
// reading its contiguous slice of the row once.  Each of a CTA's sixteen warps
// streams its own 128-id tiles without waiting for the others: the tiles' weight
// sums are taken relative to that warp's maximum of the round they were loaded in.
// Then the tile sums are brought to the slice's maximum (by warp 0, or of a slice of
// several rounds by all), and warp 0 scans them, trades (max, first argmax, sum) with
// the other slices through distributed shared memory and, where its slice holds
// u * total, finds the tile and the id.  Bound by latency for a few rows and by HBM for
// many; sample_shape() has the measurements.  Ids that differ from the ones of 64-bit
// sums (u within a rounding of a boundary): 25 of 11232 over five shapes of 64 to 256
// rows, with one CTA per row 25.
#include "internal.h"
#include "ptx.cuh"
#include "sample_body.cuh"

namespace memspec {

namespace {

using namespace smp;

constexpr int kSThreads = 512;   // accept kernel; compute threads of the sampler
constexpr int kSWarps = kSThreads / 32;
constexpr int kMaxCluster = 8;
constexpr int kTileIds = 128;    // ids of one weight tile: 4 per lane

constexpr int kMaxVocab = 131072;

struct ClSampleSmem {
  float4 peer[kMaxCluster];      // slices' (max, first argmax, weight sum), pushed by the CTAs
  uint64_t peer_bar;
  float wmax[kMaxVocab / 4096][kSWarps];   // [round][warp]; a round is at least 4096 ids
  int warg[kSWarps];             // first id of the warp's maximum over its rounds
  float wbest[kSWarps];
  float tiles[kMaxVocab / kTileIds];
};

// Maximum and first id of (bm, ba) over groups of `width` lanes.
template <int WIDTH>
__device__ __forceinline__ void lane_argmax(float& bm, int& ba) {
#pragma unroll
  for (int o = WIDTH / 2; o > 0; o >>= 1) {
    const float om = __shfl_xor_sync(0xffffffffu, bm, o);
    const int oa = __shfl_xor_sync(0xffffffffu, ba, o);
    if (om > bm || (om == bm && oa < ba)) {
      bm = om;
      ba = oa;
    }
  }
}

// The lane whose range (excl, incl) holds r; failing that (rounding at the end)
// the last lane with mass, or -1.
__device__ __forceinline__ int claim_lane(float own, float excl, float incl, float r) {
  const unsigned claim = __ballot_sync(0xffffffffu, own > 0.f && excl <= r && r < incl);
  const unsigned mass = __ballot_sync(0xffffffffu, own > 0.f);
  return claim ? __ffs(claim) - 1 : (mass ? 31 - __clz(mass) : -1);
}
__device__ __forceinline__ void lane_scan(float own, int lane, float& excl, float& incl) {
  incl = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float nb = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += nb;
  }
  excl = __shfl_up_sync(0xffffffffu, incl, 1);
  if (lane == 0) excl = 0.f;
}
// First of the N weights whose running sum from `cum` passes r, else the last
// with mass (-1: none); cum becomes the sum before it.
template <int N>
__device__ __forceinline__ int pick_in(const float (&wt)[N], float r, float& cum) {
  int sel = -1;
  float before = cum;
  bool done = false;
#pragma unroll
  for (int t = 0; t < N; ++t) {
    if (!done && wt[t] > 0.f) {
      sel = t;
      before = cum;
      done = cum + wt[t] > r;
    }
    cum += wt[t];
  }
  cum = before;
  return sel;
}

// A CTA's slice of one row: whole tiles, ids [base, end).  Ids are shifted by the
// row's misalignment (up to 3 floats) so that every vector load is aligned, where
// the shifted row still fits the cluster (else vec is false: single loads).
struct Slice {
  const float* z;
  int base, end;
  bool vec;
};
__device__ __forceinline__ Slice slice_of(const SampleArgs& a, int g, int rank, int C) {
  Slice s;
  s.z = a.logits + g * a.row_stride;
  const int mis = static_cast<int>((reinterpret_cast<uintptr_t>(s.z) >> 2) & 3);
  const int shift = a.vocab + mis <= kMaxVocab ? mis : 0;
  s.vec = shift == mis;
  const int len = (a.vocab + shift + C * kTileIds - 1) / (C * kTileIds) * kTileIds;
  s.base = rank * len - shift;
  s.end = min(s.base + len, a.vocab);
  return s;
}
__device__ __forceinline__ bool in_slice(const Slice& s, int x) { return x >= 0 && x < s.end; }

// NV float4 per thread and round, kAhead: the next round's loads are issued before a
// round is summed; thread (warp w, lane l) has ids 4 l .. 4 l + 3 of the slice's tiles
// t * 16 + w, t = 0, 1, ...
template <int NV, bool kAhead>
__global__ void __launch_bounds__(kSThreads, NV > 2 ? 2 : 3) sample_kernel(const __grid_constant__ SampleArgs a,
                                                                          int C) {
  __shared__ ClSampleSmem sm;
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int rank = static_cast<int>(cluster_ctarank()), g = blockIdx.x / C;
  const bool greedy = a.greedy != 0;
  const float it = a.inv_temp;
  if (C > 1) {
    if (tid == 0) {
      mbar_init(&sm.peer_bar, 1);
      fence_mbar_init();
      mbar_arrive_expect_tx(&sm.peer_bar, static_cast<uint32_t>(C) * 16);
    }
    cluster_arrive_release();   // waited for before the first push
  }
  pdl_wait();
  pdl_launch_dependents();
  const Slice s = slice_of(a, g, rank, C);
  const int off0 = s.base + w * kTileIds + lane * 4;
  float best = -INFINITY;
  int arg = 0x7fffffff;
  int round = 0;
  constexpr int kRound = NV * kSThreads * 4;
  auto load = [&](float (&v)[NV][4], int x00) {
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int x = x00 + j * kSThreads * 4;
      if (s.vec && x >= 0 && x + 3 < s.end) {
        const float4 t = __ldcg(reinterpret_cast<const float4*>(s.z + x));
        v[j][0] = t.x;
        v[j][1] = t.y;
        v[j][2] = t.z;
        v[j][3] = t.w;
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) v[j][q] = in_slice(s, x + q) ? __ldcg(s.z + x + q) : -INFINITY;
      }
    }
  };
  float nx[kAhead ? NV : 1][4];   // the next round's, under way while this one is summed
  if constexpr (kAhead) load(nx, off0);
  for (int x00 = off0; x00 - off0 < s.end - s.base; x00 += kRound, ++round) {
    float v[NV][4];
    if constexpr (kAhead) {
#pragma unroll
      for (int j = 0; j < NV; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) v[j][q] = nx[j][q];
      if (x00 + kRound - off0 < s.end - s.base) load(nx, x00 + kRound);
    } else {
      load(v, x00);
    }
    float bm = -INFINITY;
    int ba = 0x7fffffff;
#pragma unroll
    for (int j = 0; j < NV; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (v[j][q] > bm) {
          bm = v[j][q];
          ba = x00 + j * kSThreads * 4 + q;
        }
    lane_argmax<32>(bm, ba);
    if (bm > best) {   // rounds ascend in id
      best = bm;
      arg = ba;
    }
    if (greedy) continue;
    const float m = bm * it;
    float own[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int x = x00 + j * kSThreads * 4;
      float e[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) e[q] = __expf(v[j][q] * it - m);
      // ids outside the slice, or a round without any weight
      if (x < 0 || x + 3 >= s.end || bm == -INFINITY) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (!in_slice(s, x + q) || bm == -INFINITY) e[q] = 0.f;
      }
      own[j] = (e[0] + e[1]) + (e[2] + e[3]);
    }
    // the NV tiles' sums over the lanes together: each of the first log2(NV) steps
    // keeps half the tiles, the rest sum the remaining lanes
    int tile = 0;
#pragma unroll
    for (int o = 16, n = NV; o > 0; o >>= 1, n = n > 1 ? n / 2 : 1) {
      if (n > 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int j = 0; j < NV / 2; ++j)
          if (j < n / 2) {
            const float give = up ? own[j] : own[j + n / 2];
            const float keep = up ? own[j + n / 2] : own[j];
            own[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
          }
        if (up) tile += n / 2;
      } else {
        own[0] += __shfl_xor_sync(0xffffffffu, own[0], o);
      }
    }
    if ((lane & (32 / NV - 1)) == 0) sm.tiles[(round * NV + tile) * kSWarps + w] = own[0];
    if (lane == 0) sm.wmax[round][w] = bm;
  }
  if (lane == 0) {
    sm.wbest[w] = best;
    sm.warg[w] = arg;
  }
  __syncthreads();
  // the tile sums relative to the slice's maximum: by all threads where there are many
  const int n_tiles = round * NV * kSWarps;
  auto rescale = [&](int idx, float m) {   // tile (round, j, warp)
    const float x = sm.tiles[idx];
    return x == 0.f ? 0.f : x * __expf(sm.wmax[idx / (NV * kSWarps)][idx & (kSWarps - 1)] * it - m * it);
  };
  if constexpr (kAhead) {
    if (!greedy) {
      float m = sm.wbest[lane & (kSWarps - 1)];
#pragma unroll
      for (int o = kSWarps / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      for (int idx = tid; idx < n_tiles; idx += kSThreads) sm.tiles[idx] = rescale(idx, m);
      __syncthreads();
    }
  }
  if (w != 0) return;
  // -------------------------------------------------- warp 0: the decision
  float u = 0.f;
  if (!greedy) {
    if (a.u_explicit != nullptr)
      u = a.u_explicit[g];
    else if (a.row_slots != nullptr)   // tree step: rows of request 0
      u = philox_uniform(a.seeds[0], 0, a.seq_state[2], a.slot + a.row_slots[g]);
    else
      u = philox_uniform(a.seeds[g], g, a.seq_state[g * kStateInts + 2], a.slot);
  }
  float bm = sm.wbest[lane & (kSWarps - 1)];
  int ba = sm.warg[lane & (kSWarps - 1)];
  lane_argmax<kSWarps>(bm, ba);
  // the scan of the tile sums (a lane's tiles are consecutive)
  const int tpl = (n_tiles + 31) / 32;
  float ls = 0.f, excl = 0.f, incl = 0.f;
  if (!greedy) {
    for (int t = 0; t < tpl; ++t) {
      const int idx = lane * tpl + t;
      if constexpr (!kAhead) sm.tiles[idx] = rescale(idx, bm);
      ls += sm.tiles[idx];
    }
    lane_scan(ls, lane, excl, incl);
  }
  const float tot = __shfl_sync(0xffffffffu, incl, 31);
  // lane c: slice c's (max, argmax, sum)
  float4 p = make_float4(-INFINITY, __int_as_float(0x7fffffff), 0.f, 0.f);
  if (C > 1) {
    cluster_wait_acquire();
    if (lane < C)
      st_async_f4(mapa_shared(smem_addr(&sm.peer[rank]), lane), bm, __int_as_float(ba), tot, 0.f,
                  mapa_shared(smem_addr(&sm.peer_bar), lane));
    // the CTA leaves only after every peer's push into it has landed
    const bool ok = mbar_wait_cluster_bounded(&sm.peer_bar, 0, nullptr, a.status);
    if (!__all_sync(0xffffffffu, ok)) return;
    if (lane < C) p = sm.peer[lane];
  } else if (lane == 0) {
    p = make_float4(bm, __int_as_float(ba), tot, 0.f);
  }
  // the same arithmetic in every CTA of the cluster
  const float m_own = bm;
  bm = p.x;
  ba = __float_as_int(p.y);
  lane_argmax<32>(bm, ba);
  int tok = ba;
  bool mine = rank == 0;
  if (!greedy) {
    const float t = p.z == 0.f ? 0.f : p.z * __expf(p.x * it - bm * it);
    float s_excl, s_incl;
    lane_scan(t, lane, s_excl, s_incl);
    const float total = __shfl_sync(0xffffffffu, s_incl, 31);
    if (total > 0.f) {   // else no mass, or a NaN among the weights: the argmax
      const float target = u * total;
      const int owner = claim_lane(t, s_excl, s_incl, target);
      mine = owner == rank;
      if (!mine) return;
      // r: the rest of the target in weights relative to the slice's maximum
      const float r = (target - __shfl_sync(0xffffffffu, s_excl, owner)) *
                      (tot / __shfl_sync(0xffffffffu, t, owner));
      const int src = claim_lane(ls, excl, incl, r);
      int sel = -1;
      float before = 0.f;
      if (lane == src) {   // the first tile whose running sum passes r, else the last with mass
        float cum = excl;
        for (int k = 0; k < tpl; ++k) {
          const float y = sm.tiles[src * tpl + k];
          if (y > 0.f) {
            sel = src * tpl + k;
            before = cum;
            if (cum + y > r) break;
          }
          cum += y;
        }
      }
      if (src >= 0) {
        sel = __shfl_sync(0xffffffffu, sel, src);
        before = __shfl_sync(0xffffffffu, before, src);
        // the tile's ids again (they are in L2)
        const int x0 = s.base + sel * kTileIds + lane * 4;
        float wv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) wv[q] = in_slice(s, x0 + q) ? __ldcg(s.z + x0 + q) : -INFINITY;
#pragma unroll
        for (int q = 0; q < 4; ++q) wv[q] = in_slice(s, x0 + q) ? __expf(wv[q] * it - m_own * it) : 0.f;
        const float own = (wv[0] + wv[1]) + (wv[2] + wv[3]);
        float e_excl, e_incl;
        lane_scan(own, lane, e_excl, e_incl);
        const int who = claim_lane(own, e_excl, e_incl, r - before);
        float c = e_excl;
        const int q = pick_in(wv, r - before, c);
        if (who >= 0) tok = __shfl_sync(0xffffffffu, x0 + q, who);
      }
    }
  }
  if (mine && lane == 0) a.out_tok[static_cast<size_t>(g) * a.out_stride] = tok;
}

// grid (2K+1 rows, groups): row statistics per CTA; the last CTA of a group decides
__global__ void __launch_bounds__(kSThreads) accept_kernel(const __grid_constant__ AcceptArgs a) {
  __shared__ SampleSmem sm;
  pdl_wait();
  pdl_launch_dependents();
  accept_row<kSThreads>(a, blockIdx.x, blockIdx.y, sm, threadIdx.x, [] { __syncthreads(); });
}

// CTAs per row and float4 per thread and round.  A row is cut in two while the
// launch's CTAs still fit the chip at two per SM and a CTA keeps 2048 ids.  A slice
// of one round is taken at once (2, or 8 for a few rows), a longer one in rounds of 4
// with the next one's loads under way.
// Measured (GB300, kernel alone, T = 1; before: one CTA per row, which read its row
// twice): 1 x 32000 18.5 -> 3.3 us, 1 x 128256 57.5 -> 4.9, 32 x 128256 75.8 -> 7.7,
// 144 x 128256 77.3 -> 18.6 (4.0 TB/s; T = 0 13.2), 256 x 128256 101 -> 33.6.  With the
// tile sums rescaled by warp 0 alone 19.4 and 36.0; without the loads ahead too, rounds
// of 8, 20.8 and 36.7 - but 1 x 128256 5.1 in rounds of 4.  The scan over the tiles by all
// warps took 17.9 and 30.8, but adds them in another order.  Clusters of
// eight whatever the row count: 144 x 128256 36 us (four waves of short CTAs); a
// persistent grid that copies its next row while it reduces one: 35 us.
struct SampleShape {
  int C, nv;
};
SampleShape sample_shape(int rows, int vocab) {
  int C = 1;
  while (C < kMaxCluster && rows * C * 2 <= 304 && vocab >= 2 * C * 2048) C *= 2;
  const int round = C * kSThreads * 4;   // one float4 per thread
  return {C, vocab + 3 <= 2 * round ? 2 : (rows <= 8 && vocab + 3 <= 8 * round ? 8 : 4)};
}

}  // namespace

cudaError_t launch_sample(const SampleArgs& a, cudaStream_t s, bool pdl) {
  if (a.vocab > kMaxVocab) return cudaErrorInvalidValue;
  const SampleShape sh = sample_shape(a.n_groups, a.vocab);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(a.n_groups) * sh.C);
  cfg.blockDim = dim3(kSThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = sh.C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return sh.nv == 2   ? cudaLaunchKernelEx(&cfg, sample_kernel<2, false>, a, sh.C)
         : sh.nv == 8 ? cudaLaunchKernelEx(&cfg, sample_kernel<8, false>, a, sh.C)
                      : cudaLaunchKernelEx(&cfg, sample_kernel<4, true>, a, sh.C);
}

cudaError_t launch_accept(const AcceptArgs& a, cudaStream_t s, bool pdl) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * a.K + 1, a.n_groups);
  cfg.blockDim = dim3(kSThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, accept_kernel, a);
}

}  // namespace memspec
