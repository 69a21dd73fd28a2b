// GliDe cross-attention (Section 3.1): one draft query per (sequence, head)
// attends to every cached key, straight from global memory to registers.
//
// What bounds it.  The step reads every K and V byte once at ~1 flop per byte,
// so HBM bounds long caches and the fixed parts of a call bound short ones (a
// single user's decode: 32 heads, 2048 keys, 33 MB, 5 us of bytes).  The
// streaming kernel of cross_attn.cu spends ~7 us beside the bytes on a chunk
// table, run-time claims, shared-memory rings and a second kernel for the split
// merge.  Here a call is one kernel with little to start up:
// * a cluster of C CTAs serves one (b, h); its 8 C warps take the 16-key tiles
//   in turn.  A warp loads a tile's 8 KB into registers, the next keys while it
//   works on this tile's values; two CTAs an SM keep ~200 KB an SM in flight
//   without barriers or rings;
// * the warps' partial softmax results meet in shared memory, the C CTAs' in
//   distributed shared memory, so nothing passes through global memory and the
//   workspace is not used.  The order of all sums is fixed: repeated calls are
//   bit-identical;
// * the hardware hands the clusters to the SMs as they free up, which evens out
//   what the SMs are served where there are enough clusters for it (`pick`).
// Measured back to back over three caches in turn, streaming kernel -> this one
// (us): 32 heads, 2048 keys 11.8 -> 7.8; 128 keys 6.9 -> 3.7; 4 x 32 heads,
// 4096 keys 47.1 -> 40.9; ragged 32.8 -> 29.3; 4 x 52 heads, 16384 keys
// 249.8 -> 239.3 (7.3 TB/s), ragged 157.9 -> 154.1; D = 64, 4 x 32 heads,
// 2048 keys 25.2 -> 13.5.
#include <cuda_bf16.h>
#include <math.h>
#include <math_constants.h>

#include "attn_common.cuh"
#include "common.cuh"
#include "device.h"
#include "kernels.h"

namespace glide {
namespace {

constexpr int kTK = 16;       // keys per tile
constexpr int kWarps = 8;     // warps per CTA
constexpr int kThreads = kWarps * 32;
constexpr int kMaxCluster = 8;

struct DirectParams {
  const void* q;
  const void* K;
  const void* V;
  const int* kv_len;
  float* out;
  int H, S_cap, max_kv_len;
  int C;  // CTAs of a cluster
  float scale_log2;
};

template <typename T, int D>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 2 ? 2 : 1) cross_direct_kernel(const DirectParams p) {
  using G = GroupMap<T, D>;
  __shared__ float red[kWarps][D];
  __shared__ float2 stat[kWarps];
  __shared__ float part[D + 2];  // this CTA's (max, sum, o) for its peers
  pdl_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank();
  const int bh = blockIdx.x / p.C, b = bh / p.H;
  int n = p.kv_len[b];
  n = n < 0 ? 0 : (n > p.max_kv_len ? p.max_kv_len : n);
  const int sub = lane & 7, g4 = (lane >> 3) * 4;  // lane group g takes keys 4g..4g+3 of each tile
  const float sl2 = p.scale_log2;
  const uint64_t pol = policy_evict_first();
  const size_t slab = (size_t)bh * p.S_cap * D * sizeof(T);
  const unsigned char* Kg = static_cast<const unsigned char*>(p.K) + slab;
  const unsigned char* Vg = static_cast<const unsigned char*>(p.V) + slab;
  uint4 qc[G::kNC];
  {
    const unsigned char* qrow = static_cast<const unsigned char*>(p.q) + (size_t)bh * G::kRowBytes;
#pragma unroll
    for (int m = 0; m < G::kNC; ++m) qc[m] = __ldcg(reinterpret_cast<const uint4*>(qrow + (sub + 8 * m) * 16));
  }
  float m = -CUDART_INF_F, l = 0.f;
  uint64_t o2[G::kPairs];
#pragma unroll
  for (int e = 0; e < G::kPairs; ++e) o2[e] = 0ull;

  // this lane's chunks of the group's four rows of a tile; rows past the end
  // (the cache may hold anything there, or end) are zeros
  auto load = [&](uint4 (&r)[4][G::kNC], const unsigned char* base, int key0) {
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
#pragma unroll
      for (int c = 0; c < G::kNC; ++c) {
        r[kk][c] = make_uint4(0u, 0u, 0u, 0u);
        if (key0 + g4 + kk < n)
          r[kk][c] = load_once(base + (size_t)(key0 + g4 + kk) * G::kRowBytes + (sub + 8 * c) * 16, pol);
      }
  };
  const int step = p.C * kWarps * kTK;
  int key0 = (rank * kWarps + warp) * kTK;
  uint4 kr[4][G::kNC], vr[4][G::kNC];
  load(kr, Kg, key0);
#pragma unroll 1
  for (; key0 < n; key0 += step) {
    load(vr, Vg, key0);
    // partial scores of this group's 4 keys over this lane's dims
    float s4[4];
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      float acc[2] = {0.f, 0.f};
#pragma unroll
      for (int c = 0; c < G::kNC; ++c) dot_chunk<T>(qc[c], kr[kk][c], acc);
      s4[kk] = acc[0] + acc[1];
    }
    load(kr, Kg, key0 + step);  // the next tile's keys, under this one's softmax and values
    float sc = group8_reduce4(s4, lane) * sl2;  // score of key lane / 2 of the tile
    if (key0 + (lane >> 1) >= n) sc = -CUDART_INF_F;
    const float m_new = fmaxf(m, warp_max(sc));
    const float ref = m_new == -CUDART_INF_F ? 0.f : m_new;  // scores of -inf weigh 0; a NaN stays one
    const float corr = fast_exp2(m - ref);
    const float pe = fast_exp2(sc - ref);
    l = l * corr + ((lane & 1) ? 0.f : pe);  // each key is held by two lanes: count it once
    const uint64_t corr2 = f2pack(corr, corr);
#pragma unroll
    for (int e = 0; e < G::kPairs; ++e) o2[e] = f2mul(o2[e], corr2);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      const float pk = __shfl_sync(0xffffffffu, pe, (lane & ~7) + 2 * kk);
      const uint64_t p2 = f2pack(pk, pk);
#pragma unroll
      for (int c = 0; c < G::kNC; ++c) axpy_chunk<T>(p2, vr[kk][c], o2 + c * G::kPairsPerChunk);
    }
    m = m_new;
  }

  // the warp's result: lane groups merged, lanes 0-7 hold o
  l = warp_sum(l);
#pragma unroll
  for (int e = 0; e < G::kPairs; ++e) {
    float2 v = f2unpack(o2[e]);
    v.x += __shfl_xor_sync(0xffffffffu, v.x, 8);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, 8);
    v.x += __shfl_xor_sync(0xffffffffu, v.x, 16);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, 16);
    const int d = (sub + 8 * (e / G::kPairsPerChunk)) * G::kChunkElems + 2 * (e % G::kPairsPerChunk);
    if (lane < 8) *reinterpret_cast<float2*>(&red[warp][d]) = v;
  }
  if (lane == 0) stat[warp] = make_float2(m, l);
  __syncthreads();
  // the CTA's: a warp without a tile has max -inf, weight 0 and zeros
  if (threadIdx.x < D) {
    float M = -CUDART_INF_F, L = 0.f, O = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) M = fmaxf(M, stat[w].x);
    const float ref = M == -CUDART_INF_F ? 0.f : M;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const float f = fast_exp2(stat[w].x - ref);
      L += f * stat[w].y;
      O += f * red[w][threadIdx.x];
    }
    part[2 + threadIdx.x] = O;
    if (threadIdx.x == 0) {
      part[0] = M;
      part[1] = L;
    }
  }
  cluster_arrive();
  cluster_wait();
  // the cluster's: CTA r writes dims r dims .. of ceil(D / C) each
  const int dims = (D + p.C - 1) / p.C, d = rank * dims + threadIdx.x;
  if (threadIdx.x < dims && d < D) {
    float M = -CUDART_INF_F, L = 0.f, O = 0.f;
    float pm[kMaxCluster], pl[kMaxCluster], po[kMaxCluster];
#pragma unroll
    for (int c = 0; c < kMaxCluster; ++c) {
      // no CTA c: nothing, not CTA 0's values at weight 0 (0 times an infinity is a NaN)
      pm[c] = c < p.C ? load_peer(&part[0], c) : -CUDART_INF_F;
      pl[c] = c < p.C ? load_peer(&part[1], c) : 0.f;
      po[c] = c < p.C ? load_peer(&part[2 + d], c) : 0.f;
      M = fmaxf(M, pm[c]);
    }
    const float ref = M == -CUDART_INF_F ? 0.f : M;
#pragma unroll
    for (int c = 0; c < kMaxCluster; ++c) {
      const float f = c < p.C ? fast_exp2(pm[c] - ref) : 0.f;
      L += f * pl[c];
      O += f * po[c];
    }
    p.out[(size_t)bh * D + d] = M == -CUDART_INF_F ? 0.f : O / L;  // no cached keys: an empty softmax, zero
  }
  cluster_arrive();  // a CTA's shared memory stays until its peers have read it
  cluster_wait();
}

// How many clusters of each size the current device runs at once (0: none).
struct Room {
  int clusters[kMaxCluster + 1] = {};
};

cudaLaunchConfig_t config(long long slabs, int C, cudaStream_t st, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(slabs * C));
  cfg.blockDim = dim3(kThreads);
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}

template <typename T, int D>
cudaError_t find_room(Room& r) {
  for (int C = 1; C <= kMaxCluster; ++C) {
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = config(1, C, nullptr, attr);
    cfg.numAttrs = 1;  // the cluster's size alone
    const cudaError_t e = cudaOccupancyMaxActiveClusters(&r.clusters[C], cross_direct_kernel<T, D>, &cfg);
    if (e == cudaSuccess) continue;
    cudaGetLastError();
    return e;
  }
  return cudaSuccess;
}

// CTAs per slab (a slab: the keys of one (sequence, head)) by the slots of the
// chip alone: as many as one wave holds (each wave costs its start, ~3 us: 2 x 32
// heads, 512 keys, C = 4 and 8: 4.7 and 7.9 us), but no more than there are
// tiles.  Long caches: shorter CTAs in more waves, so that the SMs end together (4
// x 52 heads, 16384 keys, C = 1 and 4: 243.2 and 239.3 us, ragged 172.7 and
// 154.1).  More than a wave of slabs needs it sooner, and where one CTA each
// leaves a thin last wave, two fill it (8 x 40 heads, 2048 keys, C = 1 and 2: 65.0
// and 59.9 us; 16 x 32 heads, whose waves are as full with one: 79.7 and 85.0).
int usual(long long slabs, long long slots, int keys) {
  auto rounds = [&](int C) { return (keys + C * kWarps * kTK - 1LL) / (C * kWarps * kTK); };  // tiles per warp
  auto fill = [&](int C) {  // how full the waves are
    const double waves = (double)(slabs * C) / (double)slots;
    return waves / (double)((slabs * C + slots - 1) / slots);
  };
  int C = kMaxCluster;
  while (C > 1 && (slabs * C > slots || C * kWarps * kTK >= 2LL * keys)) C >>= 1;
  if (rounds(C) >= (slabs > slots ? 32 : 64)) {
    if (C < 4) C = 4;
  } else if (slabs > slots && rounds(C) >= 16 && fill(2) > fill(1) + 0.05) {
    C = 2;
  }
  return C;
}

// CTAs per slab for up to `keys` keys; 0: the streaming kernel.
//
// `usual` leaves bands of shapes badly split: one CTA a slab in a single wave that
// fills 53 to 90% of the slots, where the longest slab of a ragged batch runs on
// alone (up to 1.35 times the streaming kernel's time), or a last wave of a few
// clusters.  So every C is costed (us) relative to the streaming kernel, as the
// weighted sum of three calls, since only the bound is known here: all slabs at
// the bound, most of them far shorter (mean 0.42), and all at a sixteenth.  A wave
// of x of its full size takes `alone` + (1 - alone) x (0.7 + 0.3 x) of a full
// wave's time (few CTAs have the memory to themselves), each wave adds its start,
// and a long slab that starts late adds a little more.  What makes the ragged call
// slower than the streaming kernel counts threefold.  `usual` stands unless another
// C is 5% cheaper, and the streaming kernel is taken where it is 3% cheaper than
// that (fp32 only: its one CTA an SM leaves the start of every wave uncovered).
//
// The constants are fitted as a whole to some 650 calls of each type and head size (8
// to 520 slabs, 384 to 16384 keys, equal and ragged, every C), over which the
// choice is within 1 to 1.5% of the best C in the mean.  Streaming kernel /
// `usual` / this (us; ragged: down to an eighth), bf16, D = 128: 3 x 52 heads, 8000
// keys, ragged 71.9 / 78.6 / 67.2; 6 x 32, 6000, ragged 63.1 / 67.8 / 58.8; 4 x 40,
// 16384, equal 194.7 / 206.4 / 188.5; 5 x 16, 16384, equal 106.6 / 121.6 / 98.1;
// fp32, D = 64, 6 x 16, 6000, ragged 34.0 / 43.6 / 30.6.  Over 900 random calls the
// slowest against the streaming kernel were at 0.97 (fp32), 0.98 and 0.98 of its
// speed.  Under a bound of 4 or 16 times the lengths (176 calls) the slowest were
// 8 x 40 heads of 512 and 128 keys, 16 times: 24.3 / 25.4 / 25.5, 13.1 / 13.5 / 13.5.
int pick(const Room& room, long long slabs, bool several, float bytes_per_key, float stream_rate, float alone, int keys) {
  constexpr float kRate = 8.8f, kStart = 0.8f, kWave = 2.4f;  // MB/us; us; us
  constexpr float kStreamStart = 7.4f, kMean = 0.417f, kSpread = 0.37f, kLate = 0.1f;
  constexpr float kShort = 1.f / 16.f, kShortWeight = 0.15f;
  // Long caches of a few slabs do not fill the SMs even with eight CTAs each: the
  // streaming kernel spreads them over all (8 slabs, 8192 and 16384 keys, here
  // 11.6 and 20.4 us, there 13.0 and 20.4; fewer are faster there).
  if (slabs < 12 && keys > 8192) return 0;
  const float slots = (float)room.clusters[1], mb = (float)keys * bytes_per_key * 1e-6f, n = (float)slabs;
  const float per_wave = slots > (float)sm_count() ? kWave : 1.15f * kWave;  // one CTA an SM: no start under another's work
  const float weight = several ? 0.8f : 0.f;  // of the ragged call
  auto streaming = [&](float part) { return kStreamStart + part * n * mb / stream_rate; };
  auto shape = [](float x) { return x * (0.7f + 0.3f * x); };
  float cost[kMaxCluster + 1], judged[kMaxCluster + 1];
  int most = 1, best = 1;
  for (int C = 1; C <= kMaxCluster; ++C) {
    if (C > 1 && ((long long)(C - 1) * kWarps * kTK >= keys || room.clusters[C] < 1)) break;
    most = C;
    const float at_once = (float)room.clusters[C];
    const float wave = mb / (float)C * slots / kRate * sqrtf(at_once * (float)C / slots);
    const long long full = slabs / room.clusters[C], rest = slabs - full * room.clusters[C];
    const float start = kStart + per_wave * (float)(full + (rest ? 1 : 0));
    const float all = wave * ((float)full + (rest ? alone + (1.f - alone) * shape((float)rest / at_once) : 0.f));
    const float before = full ? (n - at_once) / at_once * kMean + (n > at_once ? kLate * alone : 0.f) : 0.f;
    const float ragged = wave * (before + alone + (1.f - alone) * kSpread * shape(full ? 1.f : n / at_once));
    const float rel = (start + ragged) / streaming(kMean);
    cost[C] = (start + all) / streaming(1.f) + weight * rel + kShortWeight * (start + kShort * all) / streaming(kShort);
    judged[C] = cost[C] + (several && rel > 1.f ? 2.f * (rel - 1.f) : 0.f);
    if (judged[C] < judged[best]) best = C;
  }
  int C = usual(slabs, room.clusters[1], keys);
  if (C > most) C = most;
  if (judged[best] < 0.95f * judged[C]) C = best;
  // below 1024 keys the streaming kernel's start is the call; what a few slabs cost
  // is not in the fit (2 slabs of 8000 keys: here 6.2 us, there 11.6)
  return slabs >= 64 && keys >= 1024 && cost[C] > 1.03f * (1.f + weight + kShortWeight) ? 0 : C;
}

template <typename T, int D>
cudaError_t launch_typed(const AttnArgs& a, cudaStream_t st) {
  static PerDevice<Room> rooms;
  Room room;
  if (rooms.get(room, find_room<T, D>) != cudaSuccess) return cudaErrorNotSupported;
  const long long slabs = (long long)a.B * a.H;
  const float stream_rate = sizeof(T) == 4 ? 7.1f : D == 128 ? 6.6f : 3.8f;  // of the streaming kernel, MB/us
  const float alone = sizeof(T) * D == 128 ? 0.45f : 0.37f;  // rows of 128 bytes: fewer bytes in flight a CTA
  const int C = pick(room, slabs, a.B > 1, 2.f * D * sizeof(T), stream_rate, alone, a.max_kv_len);
  if (C == 0) return cudaErrorNotSupported;
  if (a.max_ctas > 0 && slabs * C > a.max_ctas) return cudaErrorNotSupported;  // the streaming kernel honours the bound
  if (slabs * C > 0x7fffffffLL) return cudaErrorNotSupported;  // grid
  DirectParams p;
  p.q = a.q; p.K = a.K; p.V = a.V; p.kv_len = a.kv_len; p.out = a.out;
  p.H = a.H; p.S_cap = a.S_cap; p.max_kv_len = a.max_kv_len;
  p.C = C;
  p.scale_log2 = a.scale * kLog2e;
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = config(slabs, C, st, attr);
  return cudaLaunchKernelEx(&cfg, cross_direct_kernel<T, D>, p);
}

}  // namespace

cudaError_t launch_cross_direct(const AttnArgs& a, cudaStream_t st) {
  if (a.dtype == 0 && a.D == 128) return launch_typed<__nv_bfloat16, 128>(a, st);
  if (a.dtype == 0 && a.D == 64) return launch_typed<__nv_bfloat16, 64>(a, st);
  if (a.dtype == 1 && a.D == 128) return launch_typed<float, 128>(a, st);
  if (a.dtype == 1 && a.D == 64) return launch_typed<float, 64>(a, st);
  return cudaErrorNotSupported;
}

}  // namespace glide
