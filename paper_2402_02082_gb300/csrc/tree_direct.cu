// fp32 verification, and grouped-query cross-attention, straight from global
// memory to registers (Section 3.2; without tree keys Section 3.1).
//
// What bounds it.  fp32 is what small checks and comparisons run in: a few
// heads, up to a thousand keys and a few query rows, a microsecond of bytes and
// arithmetic.  The streaming kernel (tree_attn_fma.cu) gives each warp a fixed
// set of rows and every key, so a slab's keys pass through shared memory once
// per row, and a share's start (table, ring, ancestor walk through global
// memory) and split merge come on top.  Here, as in cross_direct.cu, a cluster
// of C CTAs serves kRows query rows of one slab (sequence, cached head): its
// 8 C warps take the 16-key tiles in turn, a warp holds a tile's keys and values
// in registers and uses them for all the rows, and the partial results meet in
// shared and distributed shared memory in a fixed order.  Row tiles re-read the
// keys from L2; where there are SMs to spare a tile is a single row.
// Measured back to back over three sets in turn, streaming kernel -> this one
// (us): 4 heads, D = 64, 778 keys, 5 nodes 13.8 -> 5.0, 16 nodes 25.2 -> 6.3;
// D = 128, 4 / 2 heads, 1024 keys, 16 nodes 88.2 -> 8.5, cross-attention 12.1 ->
// 4.5; 32 heads, 2048 keys, 6 nodes 58.5 -> 23.5, 33 nodes 257 -> 81; 8 x 40
// heads, 1024 keys, 33 nodes 1161 -> 423.
#include <math_constants.h>

#include "attn_common.cuh"
#include "common.cuh"
#include "device.h"
#include "kernels.h"

namespace glide {
namespace {

constexpr int kTK = 16;    // keys per tile
constexpr int kWarps = 8;  // warps per CTA
constexpr int kThreads = kWarps * 32;
constexpr int kRows = 4;   // query rows per CTA: their outputs take as many registers as a tile's keys
constexpr int kMaxCluster = 8;

struct TreeDirectParams {
  const float* q;
  const float* K;
  const float* V;
  const int* kv_len;
  const int* parent;
  float* out;
  int H, Hkv, S_cap, max_kv_len;
  int n;      // query nodes
  int group;  // query heads per cached head
  int rows;   // n x group, node-major
  int R;      // row tiles per slab
  int tile_rows;  // rows per tile, <= kRows
  int tree;   // the n tree keys follow the prefix
  int C;      // CTAs of a cluster
  float scale_log2;
};

template <int D>
__global__ void __launch_bounds__(kThreads, D == 64 ? 2 : 1) tree_direct_kernel(const TreeDirectParams p) {
  using G = GroupMap<float, D>;
  __shared__ __align__(16) float sq[kRows][D];
  __shared__ float red[kWarps][kRows][D];
  __shared__ float2 stat[kWarps][kRows];
  __shared__ float part[kRows][D + 2];  // this CTA's (max, sum, o) for its peers
  __shared__ int par[kMaxTree];
  pdl_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank();
  const int tile = blockIdx.x / p.C, bh = tile / p.R, b = bh / p.Hkv, h = bh - b * p.Hkv;
  const int row0 = (tile - bh * p.R) * p.tile_rows, rows_here = min(p.tile_rows, p.rows - row0);
  int plen = p.kv_len[b];
  plen = plen < 0 ? 0 : (plen > p.max_kv_len ? p.max_kv_len : plen);
  const int len = plen + (p.tree ? p.n : 0);
  const int sub = lane & 7, g4 = (lane >> 3) * 4;  // lane group g takes keys 4g..4g+3 of each tile
  const uint64_t pol = policy_evict_first();
  const float* Kg = p.K + (size_t)bh * p.S_cap * D;
  const float* Vg = p.V + (size_t)bh * p.S_cap * D;

  // this lane's chunks of the group's four rows of a tile; rows past the end
  // (the cache may hold anything there, or end) are zeros
  auto load = [&](uint4 (&r)[4][G::kNC], const float* base, int key0) {
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
#pragma unroll
      for (int c = 0; c < G::kNC; ++c) {
        r[kk][c] = make_uint4(0u, 0u, 0u, 0u);
        if (key0 + g4 + kk < len)
          r[kk][c] = load_once(base + (size_t)(key0 + g4 + kk) * D + (sub + 8 * c) * 4, pol);
      }
  };
  const int step = p.C * kWarps * kTK;
  int key0 = (rank * kWarps + warp) * kTK;
  uint4 kr[4][G::kNC], vr[4][G::kNC];
  load(kr, Kg, key0);

  if (threadIdx.x < rows_here * (D / 4)) {
    const int r = threadIdx.x / (D / 4), c = threadIdx.x - r * (D / 4);
    const size_t row = out_row(b, h, row0 + r, p.rows, p.group, p.H);
    *reinterpret_cast<float4*>(&sq[r][4 * c]) = __ldcg(reinterpret_cast<const float4*>(p.q + row * D) + c);
  }
  if (p.tree && threadIdx.x < p.n) par[threadIdx.x] = p.parent[(size_t)b * p.n + threadIdx.x];
  __syncthreads();
  // the rows' ancestor-or-self sets; a parent outside [-1, j) ends the walk
  uint64_t anc[kRows] = {};
  if (p.tree) {
    uint64_t mine = 0;
    int j = lane < rows_here ? (row0 + lane) / p.group : -1;
    while (j >= 0) {
      mine |= 1ull << j;
      const int pj = par[j];
      j = pj < j ? pj : -1;
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) anc[r] = __shfl_sync(0xffffffffu, mine, r);
  }

  float m[kRows], l[kRows];
  uint64_t o2[kRows][G::kPairs];
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    m[r] = -CUDART_INF_F;
    l[r] = 0.f;
#pragma unroll
    for (int e = 0; e < G::kPairs; ++e) o2[r][e] = 0ull;
  }
#pragma unroll 1
  for (; key0 < len; key0 += step) {
    load(vr, Vg, key0);
    const int key = key0 + (lane >> 1);  // the key whose score this lane gets
    float sc[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      if (r < rows_here) {
        float s4[4], acc[4][2] = {};
#pragma unroll
        for (int c = 0; c < G::kNC; ++c) {
          const uint4 qc = *reinterpret_cast<const uint4*>(&sq[r][(sub + 8 * c) * 4]);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) dot_chunk<float>(qc, kr[kk][c], acc[kk]);
        }
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) s4[kk] = acc[kk][0] + acc[kk][1];
        sc[r] = group8_reduce4(s4, lane) * p.scale_log2;
        if (key >= plen && (key >= len || !((anc[r] >> (key - plen)) & 1ull))) sc[r] = -CUDART_INF_F;
      }
    }
    load(kr, Kg, key0 + step);  // the next tile's keys, under this one's softmax and values
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      if (r < rows_here) {
        const float m_new = fmaxf(m[r], warp_max(sc[r]));
        const float ref = m_new == -CUDART_INF_F ? 0.f : m_new;  // nothing visible so far: weights 0
        const float corr = fast_exp2(m[r] - ref);
        const float pe = fast_exp2(sc[r] - ref);
        l[r] = l[r] * corr + ((lane & 1) ? 0.f : pe);  // each key is held by two lanes: count it once
        const uint64_t corr2 = f2pack(corr, corr);
#pragma unroll
        for (int e = 0; e < G::kPairs; ++e) o2[r][e] = f2mul(o2[r][e], corr2);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const float pk = __shfl_sync(0xffffffffu, pe, (lane & ~7) + 2 * kk);
          const uint64_t p2 = f2pack(pk, pk);
#pragma unroll
          for (int c = 0; c < G::kNC; ++c) axpy_chunk<float>(p2, vr[kk][c], o2[r] + c * G::kPairsPerChunk);
        }
        m[r] = m_new;
      }
    }
  }

  // the warp's results: lane groups merged, lanes 0-7 hold o
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    if (r < rows_here) {
      const float L = warp_sum(l[r]);
#pragma unroll
      for (int e = 0; e < G::kPairs; ++e) {
        float2 v = f2unpack(o2[r][e]);
        v.x += __shfl_xor_sync(0xffffffffu, v.x, 8);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, 8);
        v.x += __shfl_xor_sync(0xffffffffu, v.x, 16);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, 16);
        const int d = (sub + 8 * (e / G::kPairsPerChunk)) * G::kChunkElems + 2 * (e % G::kPairsPerChunk);
        if (lane < 8) *reinterpret_cast<float2*>(&red[warp][r][d]) = v;
      }
      if (lane == 0) stat[warp][r] = make_float2(m[r], L);
    }
  }
  __syncthreads();
  // the CTA's: a warp without a tile has max -inf, weight 0 and zeros
  for (int i = threadIdx.x; i < rows_here * D; i += kThreads) {
    const int r = i / D, d = i - r * D;
    float M = -CUDART_INF_F, L = 0.f, O = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) M = fmaxf(M, stat[w][r].x);
    const float ref = M == -CUDART_INF_F ? 0.f : M;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const float f = fast_exp2(stat[w][r].x - ref);
      L += f * stat[w][r].y;
      O += f * red[w][r][d];
    }
    part[r][2 + d] = O;
    if (d == 0) {
      part[r][0] = M;
      part[r][1] = L;
    }
  }
  cluster_arrive();
  cluster_wait();
  // the cluster's: CTA k writes dims k D / C .. of every row
  const int dims = D / p.C;
  for (int i = threadIdx.x; i < rows_here * dims; i += kThreads) {
    const int r = i / dims, d = rank * dims + i - r * dims;
    float M = -CUDART_INF_F, L = 0.f, O = 0.f;
    float pm[kMaxCluster], pl[kMaxCluster], po[kMaxCluster];
#pragma unroll
    for (int c = 0; c < kMaxCluster; ++c) {
      // no CTA c: nothing, not CTA 0's values at weight 0 (0 times an infinity is a NaN)
      pm[c] = c < p.C ? load_peer(&part[r][0], c) : -CUDART_INF_F;
      pl[c] = c < p.C ? load_peer(&part[r][1], c) : 0.f;
      po[c] = c < p.C ? load_peer(&part[r][2 + d], c) : 0.f;
      M = fmaxf(M, pm[c]);
    }
    const float ref = M == -CUDART_INF_F ? 0.f : M;
#pragma unroll
    for (int c = 0; c < kMaxCluster; ++c) {
      const float f = c < p.C ? fast_exp2(pm[c] - ref) : 0.f;
      L += f * pl[c];
      O += f * po[c];
    }
    const size_t row = out_row(b, h, row0 + r, p.rows, p.group, p.H);
    p.out[row * D + d] = len == 0 ? 0.f : O / L;  // no cached keys: an empty softmax, zero
  }
  cluster_arrive();  // a CTA's shared memory stays until its peers have read it
  cluster_wait();
}

template <int D>
cudaError_t launch_d(const AttnArgs& a, int tile_rows, int C, cudaStream_t st) {
  TreeDirectParams p;
  p.q = static_cast<const float*>(a.q);
  p.K = static_cast<const float*>(a.K);
  p.V = static_cast<const float*>(a.V);
  p.kv_len = a.kv_len; p.parent = a.parent; p.out = a.out;
  p.H = a.H; p.Hkv = a.Hkv; p.S_cap = a.S_cap; p.max_kv_len = a.max_kv_len;
  p.n = a.nq; p.group = a.H / a.Hkv; p.rows = a.nq * p.group; p.tree = a.tree; p.C = C;
  p.tile_rows = tile_rows;
  p.R = (p.rows + tile_rows - 1) / tile_rows;
  p.scale_log2 = a.scale * kLog2e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.B * a.Hkv * p.R * C));
  cfg.blockDim = dim3(kThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)C;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, tree_direct_kernel<D>, p);
}

}  // namespace

cudaError_t launch_tree_direct(const AttnArgs& a, cudaStream_t st) {
  if (a.dtype != 1) return cudaErrorNotSupported;
  const int rows = a.nq * (a.H / a.Hkv), keys = a.max_kv_len + (a.tree ? a.nq : 0);
  // The tile's rows and the cluster's CTAs by what they cost: a CTA takes ~3.3
  // us and per round of its warps 0.55 us and 0.33 us a row; a wave holds two
  // CTAs an SM (D = 64) or one, but clusters of 8 find room in the GPCs for
  // about half of that.  Over 100 shapes the choice is within 10% of the best
  // of the 16 (two of them 8 and 24% off).
  int best_rows = 1, best_C = 1;
  float best = 0.f;
  for (int C = 1; C <= kMaxCluster; C *= 2) {
    const long long slots = (a.D == 64 ? 2LL : 1LL) * sm_count() / (C == kMaxCluster ? 2 : 1);
    const int rounds = (keys + C * kWarps * kTK - 1) / (C * kWarps * kTK);
    for (int t = 1; t <= kRows; ++t) {
      const long long ctas = (long long)a.B * a.Hkv * ((rows + t - 1) / t) * C;
      const float cost = (float)((ctas + slots - 1) / slots) * (3.3f + (float)rounds * (0.55f + 0.33f * (float)t));
      if (best == 0.f || cost < best) {
        best = cost;
        best_rows = t;
        best_C = C;
      }
    }
  }
  const long long ctas = (long long)a.B * a.Hkv * ((rows + best_rows - 1) / best_rows) * best_C;
  // Over a very long cache one or two slabs' clusters leave the chip idle, and the
  // streaming kernel, which spreads the keys over all SMs, catches up with its
  // later start (more than four rows of 64 floats: its merge takes longer).  Its
  // time and this kernel's over long caches, as measured from 32000 to 100000 keys
  // (us, this kernel / there, 65536 keys, D = 64: one slab, two rows 72.1 / 46.7,
  // five rows 72.1 / 66.1, nine rows 71.6 / 107.4; two slabs, one row 76.7 / 62.9;
  // four slabs 78.5 / 105.9; D = 128: one slab, two rows 80.0 / 59.6, two slabs, one
  // row 86.0 / 81.9).
  if (keys > 32768 && rows <= 8) {
    const float slabs = (float)((long long)a.B * a.Hkv);
    const float start = rows * a.D <= 256 ? 11.f + 13.f / slabs : 20.f + (a.D == 64 ? 22.f : 42.f) / slabs;
    const float there = start + slabs * (float)keys * (a.D == 64 ? 0.00036f : 0.000485f);
    const float here = best * ((a.D == 64 ? 1.13f : 1.28f) + 0.07f * slabs);
    if (there < here) return cudaErrorNotSupported;
  }
  // The streaming kernel also honours a bound on the CTAs.
  if (a.max_ctas > 0 && ctas > a.max_ctas) return cudaErrorNotSupported;
  if (ctas > 0x7fffffffLL) return cudaErrorNotSupported;  // grid
  if (a.D == 128) return launch_d<128>(a, best_rows, best_C, st);
  if (a.D == 64) return launch_d<64>(a, best_rows, best_C, st);
  return cudaErrorNotSupported;
}

}  // namespace glide
