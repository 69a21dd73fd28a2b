// Speculative-sampling acceptance of a chain proposal (the acceptance strategy
// that Section 2 names and Section 4.1 uses for GliDe alone): position i
// accepts x_i when u_i * p_D,i(x_i) < p_T,i(x_i), with p_T = SoftMax(target
// logits); after the first rejection (position i) one more token is drawn from
// max(0, p_T,i - p_D,i), else from p_T,gamma+1, by inverse CDF with v: the
// first token whose running weight exceeds v * (total weight).
//
// What bounds it: latency.  A sequence's rows are a few hundred KB, a
// microsecond of one GPC's share of the bandwidth, and what the draw reads
// depends on every row's decision.  So a cluster of C CTAs serves a sequence
// and its warps meet twice at the cluster barrier, through distributed shared
// memory, instead of counting rows in through global memory:
// 1. each row is cut into 32 parts, each part an online (max, sum of exp) by one
//    warp, the (gamma + 1) x 32 parts dealt over the cluster's warps; a part's
//    result goes to every CTA, and each CTA merges the parts of a row in order
//    and decides every position.  The loads a decision needs (the draft's token,
//    its logit and probability, u) are issued before the rows;
// 2. the row of the first rejection is cut into 32 contiguous segments, a warp
//    each, whose weights are summed with unit-stride loads and kept in shared
//    memory; the segments' sums go to every CTA, a scan places them on the
//    running total, and the warp whose segment reaches past v * total walks it in
//    32-token groups (a shuffle scan per group) to the first token past the
//    target.
// The parts, the segments and the order of every sum do not depend on C.
// Measured over three sets in turn, with a CTA per row, a global counter and a
// second pass by one CTA -> this (us): 1 sequence, gamma 4, 32000 tokens 12.0 ->
// 7.3; 4 sequences, gamma 5 12.8 -> 8.6, gamma 4, 50257 tokens 17.3 -> 11.8; 16,
// gamma 8 13.5 -> 12.0; 64, gamma 4 27.8 -> 18.6.
// Floating point decides integers here (a decision, a token), in fp32 with
// this kernel's summation order; an exact real-number computation can differ
// only where u * p_D(x) or v * total lies within rounding of its threshold.
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include "attn_common.cuh"
#include "device.h"
#include "kernels.h"

namespace glide {
namespace {

constexpr int kParts = 32;                // parts of a row, and segments of the drawn row
constexpr int kWarps = 20;                // per CTA
constexpr int kThreads = kWarps * 32;
constexpr int kChunk = 16;                // floats of a row that a lane loads at once
constexpr int kGrp = 32;                  // draw: 32-token groups whose loads are issued together
constexpr int kWalk = 8;                  // walk: groups scanned together
constexpr int kKeep = 1632;               // weights of a segment that stay in shared memory
constexpr int kMaxRowsS = kMaxTree;       // gamma + 1 at most
constexpr int kMaxCluster = 16;
constexpr int kPortable = 8;              // every device runs clusters of this size

struct SampleParams {
  const int32_t* draft;    // [B, gamma]
  const float* q;          // [B, gamma, V]
  const float* logits;     // [B, gamma + 1, V]
  const float* u;          // [B, gamma + 1]
  int32_t* n_acc;          // [B]
  int32_t* next_tok;       // [B]
  int gamma, V, C;
};

// The running (max, sum of 2^((x - max) log2 e)) takes one more value, or another
// running pair, without a branch: the smaller maximum's side is rescaled.
__device__ __forceinline__ void online_add(float& m, float& s, float x) {
  const bool up = x > m;
  const float e = fast_exp2(-fabsf(x - m) * kLog2e);
  s = fmaf(up ? s : 1.f, e, up ? 1.f : s);
  m = up ? x : m;
}
__device__ __forceinline__ void online_merge(float& m, float& s, float m2, float s2) {
  const bool up = m2 > m;
  const float e = fast_exp2(-fabsf(m2 - m) * kLog2e);
  if (m2 != -CUDART_INF_F) s = fmaf(up ? s : s2, e, up ? s2 : s);
  m = up ? m2 : m;
}

// A value of this CTA's address in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void store_peer(float2* p, uint32_t rank, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(peer_addr(p, rank)), "f"(v.x), "f"(v.y) : "memory");
}

// The (max, sum) of parts first, first + every, ... of the `total` parts of the
// rows of n units of kVec floats; a part is the units part x 32 + lane, + 1024, ...
// in turn.  Two chunks of kChunk floats a lane are in flight, the later one
// under the arithmetic of the earlier, across the ends of parts.
template <int kVec, class F>
__device__ __forceinline__ void scan_parts(const float* rows, int n, int first, int every, int total, int lane, F finish) {
  constexpr int kUnits = kChunk / kVec, kSpan = kUnits * kParts * 32;
  float x[2][kChunk];
  auto start = [&](int k) { return k % kParts * 32 + lane; };
  auto load = [&](float (&v)[kChunk], int k, int j) {
    const float* row = rows + (size_t)(k / kParts) * n * kVec;
#pragma unroll
    for (int e = 0; e < kUnits; ++e) {
      const int u = j + e * kParts * 32;
      if constexpr (kVec == 4) {
        if (u < n) {
          const float4 f = __ldcg(reinterpret_cast<const float4*>(row) + u);
          v[4 * e] = f.x;
          v[4 * e + 1] = f.y;
          v[4 * e + 2] = f.z;
          v[4 * e + 3] = f.w;
        }
      } else {
        if (u < n) v[e] = __ldcg(row + u);
      }
    }
  };
  // the chunk after (k, j): the part's next, else the next part's first
  auto advance = [&](int& k, int& j) {
    j += kSpan;
    if (j - lane >= n) {  // the same for all lanes
      k += every;
      j = start(k);
    }
  };
  int k0 = first, j0 = start(first);
  if (k0 >= total) return;
  int k1 = k0, j1 = j0;
  load(x[0], k0, j0);
  advance(k1, j1);
  if (k1 < total) load(x[1], k1, j1);
  float m = -CUDART_INF_F, s = 0.f;
#pragma unroll 1
  while (k0 < total) {
#pragma unroll
    for (int e = 0; e < kUnits; ++e)
      if (j0 + e * kParts * 32 < n) {
#pragma unroll
        for (int c = 0; c < kVec; ++c) online_add(m, s, x[0][kVec * e + c]);
      }
    if (k1 != k0) {
      finish(k0, m, s);
      m = -CUDART_INF_F;
      s = 0.f;
    }
#pragma unroll
    for (int e = 0; e < kChunk; ++e) x[0][e] = x[1][e];
    k0 = k1;
    j0 = j1;
    advance(k1, j1);
    if (k1 < total) load(x[1], k1, j1);
  }
}

__global__ void __launch_bounds__(kThreads, 1) spec_sample_kernel(const SampleParams p) {
  extern __shared__ float keep[];                // weights of this CTA's segments, kKeep of each
  __shared__ float2 red[kMaxRowsS][kParts];      // (max, sum) of every part of every row
  __shared__ float2 segs[kParts];                // (sum of weights, last token with one) of every segment
  __shared__ float2 stats[kMaxRowsS];
  __shared__ int accepted[kMaxRowsS];
  cluster_arrive();  // no CTA writes into one that has not started
  pdl_wait();
  const int G1 = p.gamma + 1, V = p.V;
  const int rank = (int)cluster_rank(), b = blockIdx.x / p.C;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* rows = p.logits + (size_t)b * G1 * V;
  const float* probs = p.q + (size_t)b * p.gamma * V;

  // what the decision of row `warp` needs
  float lx = 0.f, qx = 0.f, ux = 0.f;
  auto fetch = [&](int i) {
    if (i >= p.gamma || lane != 0) return;
    int x = __ldcg(p.draft + (size_t)b * p.gamma + i);
    ux = __ldcg(p.u + (size_t)b * G1 + i);
    x = x < 0 ? 0 : (x >= V ? V - 1 : x);
    lx = __ldcg(rows + (size_t)i * V + x);
    qx = __ldcg(probs + (size_t)i * V + x);
  };
  fetch(warp);
  const float v = __ldcg(p.u + (size_t)b * G1 + p.gamma);

  // ---- 1. (max, sum) of every part
  bool started = false;
  auto finish = [&](int k, float m, float s) {
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, m, off), s2 = __shfl_xor_sync(0xffffffffu, s, off);
      online_merge(m, s, m2, s2);
    }
    m = __shfl_sync(0xffffffffu, m, 0);  // lane 0's order of merges
    s = __shfl_sync(0xffffffffu, s, 0);
    if (!started) cluster_wait();
    started = true;
    if (lane < p.C) store_peer(&red[k / kParts][k % kParts], lane, make_float2(m, s));
  };
  if ((V & 3) == 0)
    scan_parts<4>(rows, V / 4, rank * kWarps + warp, p.C * kWarps, G1 * kParts, lane, finish);
  else
    scan_parts<1>(rows, V, rank * kWarps + warp, p.C * kWarps, G1 * kParts, lane, finish);
  if (!started) cluster_wait();
  cluster_arrive();
  cluster_wait();

  // ---- the rows' statistics: parts 0, 1, ... merged in order, and the decisions
  for (int i = warp; i < G1; i += kWarps) {
    if (i != warp) fetch(i);
    const float2 r = red[i][lane];
    float before = r.x;  // the maximum of the parts before this one
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float y = __shfl_up_sync(0xffffffffu, before, off);
      if (lane >= off) before = fmaxf(before, y);
    }
    const float M = __shfl_sync(0xffffffffu, before, 31);
    before = __shfl_up_sync(0xffffffffu, before, 1);
    const float e = fast_exp2(-fabsf(r.x - before) * kLog2e);
    const unsigned up = __ballot_sync(0xffffffffu, r.x > before);
    const unsigned take = __ballot_sync(0xffffffffu, r.x != -CUDART_INF_F);
    float S = __shfl_sync(0xffffffffu, r.y, 0);
#pragma unroll
    for (int w = 1; w < kParts; ++w) {
      const float ew = __shfl_sync(0xffffffffu, e, w), sw = __shfl_sync(0xffffffffu, r.y, w);
      const bool u = (up >> w) & 1u;
      if ((take >> w) & 1u) S = fmaf(u ? S : sw, ew, u ? sw : S);
    }
    if (lane == 0) {
      stats[i] = make_float2(M, S);
      if (i < p.gamma) {
        const float pt = fast_exp2((lx - M) * kLog2e) / S;
        accepted[i] = (ux * qx < pt) ? 1 : 0;
      }
    }
  }
  __syncthreads();

  // ---- 2. the first rejection and the extra token
  int n = 0;
  while (n < p.gamma && accepted[n]) ++n;
  const float2 st = stats[n];
  const float* L = rows + (size_t)n * V;
  const float* Q = n < p.gamma ? probs + (size_t)n * V : nullptr;  // null: draw from p_T
  const float inv = 1.f / st.y;
  const int seg = (V + kParts - 1) / kParts;  // contiguous tokens per segment

  // Inverse-CDF draw from the current weights: the warp with the winning segment
  // writes the token.  False, in every warp of the cluster, when they sum to 0.
  auto draw = [&]() -> bool {
#pragma unroll 1
    for (int sl = warp; rank + sl * p.C < kParts; sl += kWarps) {  // segments rank, rank + C, ... are this CTA's
      const int sg = rank + sl * p.C, x0 = min(V, sg * seg), x1 = min(V, x0 + seg);
      float part = 0.f;
      int lastpos = -1;
#pragma unroll 1
      for (int base = x0; base < x1; base += 32 * kGrp) {
        float lv[kGrp], qv[kGrp];
#pragma unroll
        for (int k = 0; k < kGrp; ++k) {
          const int x = base + 32 * k + lane;
          lv[k] = x < x1 ? __ldcg(L + x) : 0.f;
          qv[k] = (Q && x < x1) ? __ldcg(Q + x) : 0.f;
        }
#pragma unroll
        for (int k = 0; k < kGrp; ++k) {
          const int x = base + 32 * k + lane;
          const float pt = fast_exp2((lv[k] - st.x) * kLog2e) * inv;
          const float w = x < x1 ? (Q ? fmaxf(0.f, pt - qv[k]) : pt) : 0.f;
          if (x - x0 < kKeep) keep[sl * kKeep + x - x0] = w;
          part += w;
          if (w > 0.f) lastpos = x;
        }
      }
      const float segsum = warp_sum(part);
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) lastpos = max(lastpos, __shfl_xor_sync(0xffffffffu, lastpos, off));
      if (lane < p.C) store_peer(&segs[sg], lane, make_float2(segsum, __int_as_float(lastpos)));
    }
    cluster_arrive();
    cluster_wait();
    const float2 sv = segs[lane];
    float t = sv.x;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float y = __shfl_up_sync(0xffffffffu, t, off);
      if (lane >= off) t += y;
    }  // t: upper end of segment `lane` on the running total
    const float total = __shfl_sync(0xffffffffu, t, 31);
    if (!(total > 0.f)) return false;
    const float target = v * total;
    const unsigned past = __ballot_sync(0xffffffffu, t > target);
    // no segment past the target: rounding at the very end, the row's last token
    const int last = __reduce_max_sync(0xffffffffu, __float_as_int(sv.y));
    const int win = past ? __ffs(past) - 1 : 0;
    if (win % p.C != rank || win / p.C % kWarps != warp) return true;
    int tok = -1;
    if (past) {
      const int sl = win / p.C, x0 = min(V, win * seg), x1 = min(V, x0 + seg);
      float running = __shfl_sync(0xffffffffu, t, win > 0 ? win - 1 : 0);
      if (win == 0) running = 0.f;
#pragma unroll 1
      for (int base = x0; base < x1 && tok < 0; base += 32 * kWalk) {
        float w[kWalk], incl[kWalk];
#pragma unroll
        for (int k = 0; k < kWalk; ++k) {
          const int x = base + 32 * k + lane;
          w[k] = 0.f;
          if (x < x1) {
            if (x - x0 < kKeep) {
              w[k] = keep[sl * kKeep + x - x0];
            } else {
              const float pt = fast_exp2((__ldcg(L + x) - st.x) * kLog2e) * inv;
              w[k] = Q ? fmaxf(0.f, pt - __ldcg(Q + x)) : pt;
            }
          }
          incl[k] = w[k];
        }
#pragma unroll
        for (int off = 1; off < 32; off <<= 1)
#pragma unroll
          for (int k = 0; k < kWalk; ++k) {
            const float y = __shfl_up_sync(0xffffffffu, incl[k], off);
            if (lane >= off) incl[k] += y;
          }
#pragma unroll
        for (int k = 0; k < kWalk; ++k) {
          const unsigned hit = __ballot_sync(0xffffffffu, running + incl[k] > target && w[k] > 0.f);
          if (tok < 0 && hit) tok = base + 32 * k + __ffs(hit) - 1;
          running += __shfl_sync(0xffffffffu, incl[k], 31);
        }
      }
      // rounding can leave the walk just short of the target: the segment's last token
      if (tok < 0) tok = __float_as_int(__shfl_sync(0xffffffffu, sv.y, win));
    }
    if (tok < 0) tok = last;
    if (lane == 0) p.next_tok[b] = tok;
    return true;
  };

  bool drawn = draw();
  if (!drawn) {  // max(0, p_T - p_D) summed to 0 in fp32: draw from p_T instead
    Q = nullptr;
    cluster_arrive();  // every warp has read the first draw's sums
    cluster_wait();
    drawn = draw();
  }
  if (rank == 0 && threadIdx.x == 0) {
    p.n_acc[b] = n;
    if (!drawn) p.next_tok[b] = -1;
  }
}

size_t keep_bytes(int C) { return (size_t)((kParts + C - 1) / C) * kKeep * sizeof(float); }

cudaLaunchConfig_t config(int B, int C, cudaStream_t st, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(B * C));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = keep_bytes(C);
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)C;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}

// How many clusters of each size the current device runs at once (0: none).
struct Room {
  int clusters[kMaxCluster + 1] = {};
};
cudaError_t find_room(Room& r) {
  cudaError_t e = cudaFuncSetAttribute(spec_sample_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)keep_bytes(1));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(spec_sample_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  for (int C = 1; C <= kMaxCluster; ++C) {
    if (C > kPortable && C < kMaxCluster) continue;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = config(1, C, nullptr, attr);
    cfg.attrs = attr + 1;  // the cluster's size alone
    cfg.numAttrs = 1;
    e = cudaOccupancyMaxActiveClusters(&r.clusters[C], spec_sample_kernel, &cfg);
    if (e == cudaSuccess) continue;
    cudaGetLastError();
    r.clusters[C] = 0;
    if (e != cudaErrorInvalidClusterSize) return e;
  }
  return cudaSuccess;
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

// The call's workspace, as its callers allocate it; this kernel's warps meet in distributed shared
// memory and leave it alone.
size_t sample_workspace_bytes(int B, int gamma) {
  return 256 + align256((size_t)B * 4) + align256((size_t)B * (gamma + 1) * 8) + align256((size_t)B * gamma * 4);
}

cudaError_t launch_spec_sample(const SampleArgs& a, cudaStream_t st) {
  static PerDevice<Room> rooms;
  Room room;  // unknown: one CTA per sequence
  if (rooms.get(room, find_room) != cudaSuccess) room = Room();
  // CTAs per sequence: as many as let all sequences run at once (a second wave
  // costs as much as the first: 16 sequences, gamma 4, C = 6 and 8: 10.2 and 13.3
  // us).  Sixteen only where they save a round of parts (4 sequences, gamma 8,
  // C = 8 and 16: 10.2 and 8.9 us; gamma 4: 7.95 and 8.1).
  int C = kPortable;
  while (C > 1 && a.B > room.clusters[C]) --C;
  if (C == kPortable && (a.gamma + 1) * kParts > C * kWarps && a.B <= room.clusters[kMaxCluster]) C = kMaxCluster;
  SampleParams p;
  p.draft = a.draft; p.q = a.q; p.logits = a.logits; p.u = a.u;
  p.n_acc = a.n_acc; p.next_tok = a.next_tok;
  p.gamma = a.gamma; p.V = a.V; p.C = C;
  if ((long long)a.B * C > 0x7fffffffLL) return cudaErrorInvalidValue;
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = config(a.B, C, st, attr);
  return cudaLaunchKernelEx(&cfg, spec_sample_kernel, p);
}

}  // namespace glide
