// Tree verification attention in 128-row tiles on the tcgen05 tensor cores,
// for grouped-query slabs (Section 3.2's verification of a CaPE tree, under
// the ancestor-or-self mask, on a target with fewer cached heads than query
// heads such as Mistral-7B, Section 4.1) and any slab of more than 64 query
// rows; without tree keys (a prefix-only mode) the same kernel serves the
// draft's grouped-query cross-attention (Section 3.1), the group's queries as
// a slab's rows.
//
// A slab is a (sequence, cached head) with n tree nodes x H / H_kv query
// heads as its rows, node-major: a 33-node CaPE tree on Mistral-7B's 32 query
// over 8 cached heads has 132.  The 64-row kernel serves such a slab in three
// row tiles whose CTAs each run the whole 64-key tile loop (the softmax chain
// sets a ~1400-cycle period per tile), so the work grows with the row tiles
// while the bytes stay the same.  Here a row tile is 128 rows and a key tile
// 128 keys, the shape of the training-time block-mask kernel:
//   S = Q K^T : M = 128 query rows, N = 128 keys, K = D, operands in shared memory
//   O += P V  : M = 128, N = D, K = 128 keys, P in tensor memory
// which does four times the (row, key) pairs of a 64 x 64 tile per softmax
// pass.  Tensor memory holds three S buffers of 128 columns (S of tile i + 3
// waits for P.V of tile i) and the O accumulator.  Two softmax groups of four
// warps take the tiles in turn, one thread per row: the softmax of a tile is a
// serial chain of ~1500 cycles and each group has two tile periods for it.  The
// reference max of the online softmax passes from tile to tile, so from group
// to group, through shared memory; a group keeps its own row sum and takes it
// to the segment's last reference at the end.  P overwrites the first 64
// columns of its S buffer.
//
// Code size counts like a resource here (see the 64-row kernel): the loops are
// rolled 64 scores at a time, the share is looked up once per CTA, waits are
// small: 99 KB of code became 63 KB.  Measured on Mistral-7B's 32 over 8 heads
// (16384 keys, 4 sequences), bursts of a few ms back to back: the 33-node tree,
// two row tiles (132 rows of 256), 72.4 -> 57.6 us (62.7 before the epilogue's
// exchange of rows; sustained over a second 74.0 -> 64.1); the draft step, 4 rows,
// 48.1 -> 45.7; 2 sequences of 211 keys, one node, 11.2 -> 8.9; one sequence of
// 13645 keys, 3 nodes, 21.9 -> 18.7 (before: the groups on the two key halves of
// every tile, meeting in an exchange of the row max).
//
// Work: the slabs' 128-key tiles are cut into G shares of equal cost (a
// segment switch counted as kSegWeight tiles), and R = ceil(rows / 128)
// adjacent CTAs serve each share, CTA x * R + y taking row tile y of every
// slab in share x: the R CTAs stream the same K/V tiles at about the same
// time, so DRAM serves each tile about once and L2 the other reads.  A slab
// whose keys all fall in one share is written out directly; a split slab
// leaves one partial (max, sum, o) per share and row, and the split merge
// kernel, launched as a programmatic dependent, combines them.
//
// Q comes by 3-D TMA: the [B n, H, D] queries as a box of 128 / group nodes x
// group heads x 64 head dims is exactly the 128 node-major rows of a row tile
// (so group must divide 128).  Rows past the slab's n x group are padding:
// whatever they read (another sequence's queries or the zero fill), their
// results are never written.
//
// Roles (384 threads, one CTA per SM):
//   warps 0-7  softmax and the segment epilogues: warp w reads TMEM lane
//              quarter w % 4 (one thread per row) of the tiles of parity w / 4.
//   warp 8     the K ring, warp 11 the V ring (2-D TMA by lane 0, 128-byte
//              swizzle); warp 11's lanes clear the V rows past a slab's end.
//   warp 9     lane 0: the queries of each segment, S issue; the TMEM allocation.
//   warp 10    P.V issue (lane 0).
//
// Masking: keys below the sequence's prefix length are visible to every row;
// tree key c (at prefix + c) is visible to the rows of node i iff c is an
// ancestor-or-self of i (the set built from the parent array by pointer
// jumping, at the start of a segment that reaches the tree keys); keys past the
// prefix and the n tree keys are masked, and their V rows are zeroed in
// shared memory before P.V (the cache beyond them may hold anything).  In the
// prefix-only mode a sequence without cached keys gets zeros.
// Online softmax in the log2 domain with a lazy reference max: O is rescaled
// in TMEM only when a tile's max exceeds the reference by more than 8.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math_constants.h>

#include "attn_common.cuh"
#include "device.h"
#include "kernels.h"
#include "tc_attn.cuh"
#include "tc_ptx.cuh"
#include "tensor_map.h"

namespace glide {
namespace {

constexpr int kBM = 128;          // query rows per row tile (MMA rows, TMEM lanes)
constexpr int kBN = 128;          // keys per tile
constexpr int kMaxStages = 4;     // K/V ring stages (the launch picks as many as fit)
constexpr int kSoftWarps = 8;     // two groups of four: the even and the odd tiles
constexpr int kFewRows = 24;      // a warp's rows up to which the epilogue stores them as they are (its comment)
constexpr int kKProdWarp = 8;     // the K ring
constexpr int kSWarp = 9;         // the queries and S
constexpr int kPVWarp = 10;
constexpr int kVProdWarp = 11;
constexpr int kThreads = 384;
constexpr int kTmemCols = 512;
constexpr int kSBufs = 3;                   // S / P buffers at columns 0, 128, 256
constexpr uint32_t kTmemO = kSBufs * kBN;   // the O accumulator from column 384
constexpr uint32_t kAtom = 128 * 128;       // one 128-byte-swizzle atom of 128 rows
constexpr float kRescaleLog2 = 8.0f;
// What a switch from one slab to the next costs a CTA, in 128-key tiles (the
// segment's epilogue and the pipeline start of the next, with its queries).
constexpr int kSegWeight = 4;

// ODONE has four slots (tile mod 4).  P.V completions are waited on only now
// and then (a rescale, the epilogue), when up to three products may still be
// in flight: P.V of tile i - 3 has completed once S of tile i has been read,
// but those of tiles i - 2 .. i may not have.  Four slots keep every such wait
// within one phase of its barrier; with two, a wait for tile i could pass on
// the completion of tile i - 2 (measured: the last tiles of a segment missing
// from O when the values arrived late from DRAM).
constexpr int B_KFULL = 0, B_KEMPTY = 4, B_VFULL = 8, B_VEMPTY = 12, B_QFULL = 16, B_QEMPTY = 17, B_SFULL = 18,
              B_PFULL = 21, B_BFREE = 24, B_ODONE = 27, B_MDONE = 31, B_OFREE = 33, B_VCLR = 34, kNumBars = 38;

template <int D>
struct WideCfg {
  static constexpr int kHalves = D / 64;                // swizzle atoms across the head dim
  static constexpr uint32_t kQBytes = kHalves * kAtom;  // 128 rows x D
  static constexpr uint32_t kKV = kHalves * kAtom;      // 128 keys x D
  static constexpr uint32_t off_Q = 0;
  static constexpr uint32_t off_K = kQBytes;
  // K ring of nk stages, then the V ring of nv, barriers, misc, row sums, batch table
  static __host__ __device__ uint32_t off_V(int nk) { return off_K + nk * kKV; }
  static __host__ __device__ uint32_t off_bar(int nk, int nv) { return off_V(nk) + nv * kKV; }
  // TMEM slot, abort flag, share start
  static __host__ __device__ uint32_t off_misc(int nk, int nv) { return off_bar(nk, nv) + kNumBars * 8; }
  // [2][row]: during a segment, [0] holds the running reference max of every
  // row; at its end, both hold the groups' row sums
  static __host__ __device__ uint32_t off_row(int nk, int nv) { return off_misc(nk, nv) + 32; }
  static __host__ __device__ uint32_t off_tab(int nk, int nv) { return off_row(nk, nv) + 2 * kBM * 4; }
  static size_t smem_bytes(int B, int nk, int nv) {
    return 1024 + off_tab(nk, nv) + (size_t)(B + 1) * 8 + (size_t)(4 * B + 1) * 4;
  }
  static_assert(kTmemO + D <= kTmemCols, "TMEM columns");
  static_assert(kNumBars % 2 == 0, "alignment");
};

struct WideParams {
  const int* kv_len;
  const int* parent;
  float* out;
  unsigned* status;
  int2* ranges;      // per slab: the share range of a split slab, (-1, -1) otherwise
  float* partials;
  int B, H, Hkv, group, S_cap, max_kv_len, n;
  int rows;          // query rows per slab: n nodes x group heads, node-major
  int R;             // row tiles of 128 per slab
  int tree;          // 1: the n tree keys follow the prefix (verification); 0: prefix only
  int nk, nv;        // K and V ring stages
  float scale_log2;
};

// The hand-over of a tile's reference max between the two warps (one of each
// softmax group) of a TMEM lane quarter: named barriers 8-15, per quarter and
// tile parity; the tile's warp arrives, the next tile's warp waits.
__device__ __forceinline__ void turn_pass(int quarter, unsigned tile) {
  asm volatile("bar.arrive %0, 64;" ::"r"(8 + 2 * quarter + (int)(tile & 1)) : "memory");
}
__device__ __forceinline__ void turn_wait(int quarter, unsigned tile) {
  asm volatile("bar.sync %0, 64;" ::"r"(8 + 2 * quarter + (int)(tile & 1)) : "memory");
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
    tree_attn_wide_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                          const __grid_constant__ CUtensorMap tmV, const WideParams p) {
  using C = WideCfg<D>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int nk = p.nk, nv = p.nv;  // K and V ring depths
  const uint32_t off_V = C::off_V(nk);
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + C::off_bar(nk, nv));
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base + C::off_misc(nk, nv));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base + C::off_misc(nk, nv) + 4);
  ShareStart* share = reinterpret_cast<ShareStart*>(base + C::off_misc(nk, nv) + 16);
  float* rowbuf = reinterpret_cast<float*>(base + C::off_row(nk, nv));
  BatchTiles bt;
  bt.start = reinterpret_cast<long long*>(base + C::off_tab(nk, nv));
  bt.len = reinterpret_cast<int*>(bt.start + p.B + 1);
  bt.ntiles = bt.len + p.B;
  bt.plen = bt.ntiles + p.B;
  bt.sidx = bt.plen + p.B;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Shared-memory set-up and the tensor-map fetches come before the wait for
  // the previous kernel; every global access and the TMEM allocation after it.
  if (threadIdx.x == 0) {
    tc::prefetch_tmap(&tmQ);
    tc::prefetch_tmap(&tmK);
    tc::prefetch_tmap(&tmV);
#pragma unroll 1
    for (int b = 0; b < kNumBars; ++b)
      mbar_init(&bars[b], b >= B_PFULL && b < B_PFULL + kSBufs ? kSoftWarps / 2 : b == B_OFREE ? kSoftWarps : 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  // this CTA: share x of the key tiles, row tile y of every slab in it
  const int G = gridDim.x / p.R, x = blockIdx.x / p.R, y = blockIdx.x - x * p.R;
  const int row0 = y * kBM;
  // one reader per tile: evict it first; R row tiles read each tile R times
  const uint64_t kv_pol = p.R == 1 ? policy_evict_first() : policy_evict_normal();
  auto load_tile = [&](const CUtensorMap* map, uint64_t* full, unsigned char* dst, int row) {
    mbar_arrive_expect_tx(full, C::kKV);
    for (int hd = 0; hd < C::kHalves; ++hd) tc::tma_load_2d(dst + hd * kAtom, map, hd * 64, row, full, kv_pol);
  };
  auto load_q = [&](int b, int h) {
    mbar_arrive_expect_tx(&bars[B_QFULL], C::kQBytes);
    const int z = b * p.n + row0 / p.group;  // the row tile's first node in [B n, H, D]
    for (int hd = 0; hd < C::kHalves; ++hd)
      tc::tma_load_3d(base + C::off_Q + hd * kAtom, &tmQ, hd * 64, h * p.group, z, &bars[B_QFULL], policy_evict_first());
  };
  if (warp == 0) {
    wait_and_build_share(bt, p.kv_len, p.B, p.Hkv, p.max_kv_len, p.tree ? p.n : 0, kBN, G, kSegWeight, x, share);
    if (lane == 0 && share->tiles > 0) {  // the first loads at once, not after the roles have found their way
      const int row = (share->b * p.Hkv + share->h) * p.S_cap + share->t0 * kBN;
      load_tile(&tmK, &bars[B_KFULL], base + C::off_K, row);
      load_q(share->b, share->h);
      load_tile(&tmV, &bars[B_VFULL], base + off_V, row);
    }
    __syncwarp();
  } else {
    pdl_wait();
  }
  if (warp == kSWarp) {
    tc::tmem_alloc(tmem_slot, kTmemCols);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  SegWalk s;
  s.start(bt, *share);

  if (warp == kKProdWarp || warp == kVProdWarp) {
    // ----------------------------------------------------------- producers
    // Warp 8 the keys, warp 11 the values: one loop, so that its code is there
    // once.  Lane 0 issues; the other lanes are there to clear the rows past a
    // slab's last key in its last V tile.
    const bool keys = warp == kKProdWarp;
    const CUtensorMap* map = keys ? &tmK : &tmV;
    unsigned char* ring = base + (keys ? C::off_K : off_V);
    uint64_t* full = &bars[keys ? B_KFULL : B_VFULL];
    uint64_t* empty = &bars[keys ? B_KEMPTY : B_VEMPTY];
    const int depth = keys ? nk : nv;
    int st = 0, issued = 0;
    uint32_t phase = 1;  // the stage's parity as the waiter sees it
    bool ok = true;
    for (; s.any() && ok; s.next(bt, p.Hkv)) {
      int row = (s.b * p.Hkv + s.h) * p.S_cap + s.t0 * kBN;
      const int len = bt.len[s.b];
      for (int t = s.t0; t < s.t1; ++t, row += kBN) {
        ok = warp_wait_small(&empty[st], phase, abort_flag);
        if (!ok) break;
        unsigned char* dst = ring + st * C::kKV;
        if (lane == 0 && issued > 0) load_tile(map, &full[st], dst, row);  // the share's first tile is on its way already
        __syncwarp();
        ++issued;
        const int vrows = len - t * kBN;
        if (!keys && vrows < kBN) {  // the slab's last tile: clear its V rows past the last key
          ok = warp_wait_small(&full[st], phase ^ 1, abort_flag);
          if (!ok) break;
#pragma unroll 1
          for (int idx = vrows * C::kHalves * 8 + lane; idx < kBN * C::kHalves * 8; idx += 32)
            *reinterpret_cast<uint4*>(dst + ((idx >> 3) % C::kHalves) * kAtom + idx / (C::kHalves * 8) * 128 +
                                      (idx & 7) * 16) = make_uint4(0u, 0u, 0u, 0u);
          tc::fence_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars[B_VCLR + st]);
        }
        if (++st == depth) {
          st = 0;
          phase ^= 1;
        }
      }
    }
    if (!ok && lane == 0)  // aborted: let issued loads land before the CTA exits
      for (int j = (issued > depth ? issued - depth : 0); j < issued; ++j)
        mbar_drain(&full[j % depth], (j / depth) & 1);
  } else if (warp == kSWarp || warp == kPVWarp) {
    // ----------------------------------------------------------- MMA issue
    // The P.V warp has time until the first probabilities.
    if (warp == kPVWarp && y == 0) write_ranges(bt, p.B, p.Hkv, G, kSegWeight, p.ranges, x * 32 + lane, G * 32);
    __syncwarp();
    // Ring positions are counted, not divided out.
    if (lane == 0) {
      bool ok = true;
      int bi = 0, st = 0, seg = 0;  // S buffer, ring stage, segment
      uint32_t col = tmem, phase = 0;
      if (warp == kSWarp) {
        // S(i) = Q K(i)^T into buffer i % 3, once P.V of tile i - 3 has read
        // that buffer; the segment's queries first, once S of the last segment
        // has read the previous ones
        constexpr uint32_t idS = tc::idesc_bf16_f32(kBM, kBN, false, false);
        const uint64_t dQ = tc::sw128_desc(smem_u32(base + C::off_Q), 16, 1024);
        const uint64_t dK0 = tc::sw128_desc(smem_u32(base + C::off_K), 16, 1024);
        uint32_t b_phase = 1;
        bool q_loading = false;
        for (; s.any() && ok; s.next(bt, p.Hkv), ++seg) {
          if (seg > 0) ok = mbar_wait_small(&bars[B_QEMPTY], (seg - 1) & 1, abort_flag);
          if (!ok) break;
          if (seg > 0) load_q(s.b, s.h);
          q_loading = true;
          ok = mbar_wait_small(&bars[B_QFULL], seg & 1, abort_flag);
          if (ok) q_loading = false;
#pragma unroll 1
          for (int t = s.t1 - s.t0; ok && t > 0; --t) {
            ok = mbar_wait_small(&bars[B_KFULL + st], phase, abort_flag) &&
                 mbar_wait_small(&bars[B_BFREE + bi], b_phase, abort_flag);
            if (!ok) break;
            tc::fence_after_sync();
            const uint64_t dK = dK0 + (uint64_t)st * desc_step(C::kKV);
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
              const uint64_t step = desc_step((ks >> 2) * kAtom + (ks & 3) * 32);
              tc::mma_bf16(col, dQ + step, dK + step, idS, ks > 0 ? 1u : 0u);
            }
            tc::mma_commit(&bars[B_SFULL + bi]);
            tc::mma_commit(&bars[B_KEMPTY + st]);
            if (t == 1) tc::mma_commit(&bars[B_QEMPTY]);
            if (++st == nk) {
              st = 0;
              phase ^= 1;
            }
            col += kBN;
            if (++bi == kSBufs) {
              bi = 0;
              b_phase ^= 1;
              col = tmem;
            }
          }
        }
        if (q_loading) mbar_drain(&bars[B_QFULL], seg & 1);  // aborted: let the queries land
        tc::mma_commit(&bars[B_MDONE]);  // every MMA finished before TMEM is released
        mbar_drain(&bars[B_MDONE], 0);
      } else {
        // O (+)= P(i) V(i), P in the first 64 columns of buffer i % 3; the
        // segment's first tile starts O, once its last value is read
        constexpr uint32_t idO = tc::idesc_bf16_f32(kBM, D, false, true);
        const uint64_t dV0 = tc::sw128_desc(smem_u32(base + off_V), kAtom, 1024);
        uint32_t p_phase = 0, cleared = 0;  // cleared: bit s, parity of the clears of V stage s so far
        int od = 0;
        for (; s.any() && ok; s.next(bt, p.Hkv), ++seg) {
          if (seg > 0) ok = mbar_wait_small(&bars[B_OFREE], (seg - 1) & 1, abort_flag);
          const bool partial = s.t1 == bt.ntiles[s.b] && bt.len[s.b] < s.t1 * kBN;  // its last V tile gets cleared rows
          uint32_t acc = 0;
#pragma unroll 1
          for (int t = s.t1 - s.t0; ok && t > 0; --t) {
            ok = mbar_wait_small(&bars[B_VFULL + st], phase, abort_flag);
            if (ok && t == 1 && partial) {
              ok = mbar_wait_small(&bars[B_VCLR + st], (cleared >> st) & 1, abort_flag);
              cleared ^= 1u << st;
            }
            ok = ok && mbar_wait_small(&bars[B_PFULL + bi], p_phase, abort_flag);
            if (!ok) break;
            tc::fence_after_sync();
            const uint64_t dV = dV0 + (uint64_t)st * desc_step(C::kKV);
#pragma unroll
            for (int ks = 0; ks < kBN / 16; ++ks)
              tc::mma_bf16_ts(tmem + kTmemO, col + ks * 8, dV + desc_step(ks * 16 * 128), idO, ks > 0 ? 1u : acc);
            acc = 1;
            tc::mma_commit(&bars[B_BFREE + bi]);
            tc::mma_commit(&bars[B_VEMPTY + st]);
            tc::mma_commit(&bars[B_ODONE + od]);
            od = (od + 1) & 3;
            if (++st == nv) {
              st = 0;
              phase ^= 1;
            }
            col += kBN;
            if (++bi == kSBufs) {
              bi = 0;
              p_phase ^= 1;
              col = tmem;
            }
          }
        }
        tc::mma_commit(&bars[B_MDONE + 1]);
        mbar_drain(&bars[B_MDONE + 1], 0);
      }
    }
  } else {
    // ----------------------------------------------- softmax and epilogues
    const int grp = warp >> 2, quarter = warp & 3;  // this group's tiles: CTA-local index parity grp
    const int r = quarter * 32 + lane;  // this thread's row in the tile (its TMEM lane)
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    const float sl2 = p.scale_log2;
    const uint64_t sc2 = f2(sl2, sl2);
    const int qrow = row0 + r;  // the slab's query row
    const bool valid = qrow < p.rows;
    const int node = valid ? qrow / p.group : 0;
    const int q_rel = node * p.H + qrow - node * p.group;  // its place in a sequence's [node, head] rows of out
    bool dead = false;

    // Zeros for a prefix-only call's sequences without cached keys (an empty softmax).
    constexpr int kST = kSoftWarps * 32;
    if (!p.tree)
      zero_empty(bt, p.B, (long long)p.n * p.H * D, p.out, (int)blockIdx.x * kST + (int)threadIdx.x,
                 (int)gridDim.x * kST);

    unsigned i = 0;  // CTA-local index of the segment's first tile
    for (; s.any(); s.next(bt, p.Hkv)) {
      const int plen = bt.plen[s.b], nt = s.t1 - s.t0;
      const unsigned jl = i + nt - 1;  // the segment's last tile
      // this row's node's ancestor-or-self set, if this group has a tile with tree
      // keys, while the segment's first scores are on their way
      uint64_t anc = 0;
      int t_tree = plen / kBN - s.t0;  // the segment's first tile with tree keys
      t_tree = t_tree < 0 ? 0 : t_tree;
      t_tree += (int)((i + t_tree) ^ grp) & 1;
      if (p.tree && t_tree < nt)
        anc = ancestors(parents_of(p.parent + (size_t)s.b * p.n, p.n, lane), p.n, node, valid, lane);
      float m_own = -CUDART_INF_F, l = 0.f;  // the sum over this group's tiles and the reference it is taken against
      for (int t = (int)((i ^ grp) & 1u); t < nt; t += 2) {
        const unsigned j = i + t, bi = j % kSBufs;
        const uint32_t s_col = lane_base + bi * kBN;
        if (!opaque(dead)) dead = !warp_wait_small(&bars[B_SFULL + bi], (j / kSBufs) & 1, abort_flag);
        tc::fence_after_sync();
        // keys this row does not see (tree keys that are no ancestors, and what
        // lies past the tree): -inf, written back to the S buffer
        const int k0 = (s.t0 + t) * kBN - plen;  // the tile's first key, past the prefix
        if (k0 + kBN > 0) {
#pragma unroll 1
          for (int c = 0; c < opaque(kBN / 32); ++c) {
            uint32_t o[32];
            tc::tmem_ld32(s_col + c * 32, o);
            tc::tmem_wait_ld();
            const uint32_t vis = (uint32_t)visible_keys(anc, k0 + c * 32);
#pragma unroll
            for (int e = 0; e < 32; ++e) o[e] = (vis & (1u << e)) ? o[e] : 0xff800000u;
            tc::tmem_st32(s_col + c * 32, o);
          }
          tc::tmem_wait_st();
        }
        // The scores are read from TMEM twice, 64 at a time in rolled loops
        // (row max, then exponentials): unrolled over a whole 128-key row the
        // loop body outgrows the instruction cache.
        float mx[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
#pragma unroll 1
        for (int hf = 0; hf < opaque(2); ++hf) {
          uint32_t sv[64];
          tc::tmem_ld32(s_col + hf * 64, *reinterpret_cast<uint32_t(*)[32]>(sv));
          tc::tmem_ld32(s_col + hf * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(sv + 32));
          tc::tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 64; e += 8)
#pragma unroll
            for (int q = 0; q < 4; ++q)
              mx[q] = fmax3(mx[q], __uint_as_float(sv[e + 2 * q]), __uint_as_float(sv[e + 2 * q + 1]));
        }
        const float tmax = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * sl2;
        // The reference max passes from tile to tile, so from group to group
        // (one slot: a thread reads its row's before it writes the next).
        float m_prev = -CUDART_INF_F;
        if (t > 0) {
          turn_wait(quarter, j - 1);
          m_prev = rowbuf[r];
        }
        const bool need = tmax > m_prev + kRescaleLog2;
        const float m_used = need ? tmax : m_prev;
        rowbuf[r] = m_used;
        turn_pass(quarter, j);
        if (__any_sync(0xffffffffu, need) && t > 0 && !dead) {
          // O holds the P.V of this segment's earlier tiles, the other group's last one included: rescale it
          dead = !warp_wait_small(&bars[B_ODONE + ((j - 1) & 3)], ((j - 1) >> 2) & 1, abort_flag);
          const float f = need ? fast_exp2(m_prev - m_used) : 1.f;
          tc::fence_after_sync();
#pragma unroll 1
          for (int c = 0; c < opaque(D / 32); ++c) {
            uint32_t o[32];
            tc::tmem_ld32(lane_base + kTmemO + c * 32, o);
            tc::tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * f);
            tc::tmem_st32(lane_base + kTmemO + c * 32, o);
          }
          tc::tmem_wait_st();
        }
        if (m_own != m_used) {
          l *= fast_exp2(m_own - m_used);  // 0 while there is no sum
          m_own = m_used;
        }
        const float m_eff = m_used == -CUDART_INF_F ? 0.f : m_used;
        const uint64_t nm2 = f2(-m_eff, -m_eff);
        uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll 1
        for (int hf = 0; hf < opaque(2); ++hf) {
          uint32_t sv[64], pk[32];
          tc::tmem_ld32(s_col + hf * 64, *reinterpret_cast<uint32_t(*)[32]>(sv));
          tc::tmem_ld32(s_col + hf * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(sv + 32));
          tc::tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            float x0, x1;
            unf2(ffma2(f2(__uint_as_float(sv[2 * e]), __uint_as_float(sv[2 * e + 1])), sc2, nm2), x0, x1);
            const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
            acc[e & 3] = fadd2(acc[e & 3], f2(p0, p1));
            pk[e] = pack_bf16x2(p0, p1);
          }
          tc::tmem_st32(s_col + hf * 32, pk);  // over scores already read
        }
        tc::tmem_wait_st();
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars[B_PFULL + bi]);
        float a0, a1, b0, b1;
        unf2(fadd2(acc[0], acc[1]), a0, a1);
        unf2(fadd2(acc[2], acc[3]), b0, b1);
        l += (a0 + a1) + (b0 + b1);
      }

      // ---- segment epilogue: the row sum over both groups, then each writes
      // its half of the head dims, O / l or a split partial.  The group that did
      // not do the last tile takes its sum to that tile's reference first, and
      // leaves it where the reference was.
      const bool mine = ((jl ^ grp) & 1u) == 0;
      if (!mine) {
        turn_wait(quarter, jl);
        const float m_last = rowbuf[r];
        if (m_own != m_last) l *= fast_exp2(m_own - m_last);
        m_own = m_last;
      }
      rowbuf[(mine ? kBM : 0) + r] = l;
      pair_sync(quarter);
      const float L = rowbuf[r] + rowbuf[kBM + r];
      pair_sync(quarter);  // read, before the next segment's reference goes in
      if (!dead) dead = !warp_wait_small(&bars[B_ODONE + (jl & 3)], (jl >> 2) & 1, abort_flag);
      tc::fence_after_sync();
      // Output rows of the whole slab in this share, else the share's partial [max,
      // sum, o] (a partial row is 8-byte aligned).  A thread holds one row's columns;
      // stored so, each 8 bytes of a warp's store lie in another sector, and 128 rows
      // took 4400 cycles, 9900 on the last CTAs.  Eight lanes exchange their rows
      // first, so that a store writes 64 consecutive bytes of four rows (32 / 8 heads:
      // 4 x 2048 keys, 33 nodes 24.5 -> 19.6 us, 4 x 16384 63.1 -> 58.0).  A few rows
      // are stored as they are (24: 11.5 us for 2048 keys, exchanged 11.8; 64: 13.5
      // and 12.7).
      const bool whole = s.whole(bt);
      float* dst = whole ? p.out + ((long long)s.b * p.n * p.H + s.h * p.group) * D
                         : partial_slot(p.partials, x + s.b * p.Hkv + s.h, p.rows, D) + 2;
      const int rel = !valid || dead ? -1 : whole ? q_rel * D : qrow * (D + 2);
      if (rel >= 0 && !whole && grp == 0) *reinterpret_cast<float2*>(dst + rel - 2) = make_float2(m_own, L);
      const float scale = !whole ? 1.f : L > 0.f ? 1.f / L : 0.f;
      const int warp_rows = p.rows - row0 - quarter * 32;
      dst += grp * (D / 2);
      auto load8 = [&](int c, float2 (&v)[8]) {
        uint32_t o[16];
        tc::tmem_ld16(lane_base + kTmemO + grp * (D / 2) + c * 16, o);
        tc::tmem_wait_ld();
#pragma unroll
        for (int k = 0; k < 8; ++k)
          v[k] = make_float2(__uint_as_float(o[2 * k]) * scale, __uint_as_float(o[2 * k + 1]) * scale);
      };
      if (warp_rows > kFewRows) {
        dst += 2 * (lane & 7);
#pragma unroll 1
        for (int c = 0; c < opaque(D / 32); ++c, dst += 16) {
          float2 v[8];  // 8 x 8 pairs over 8 lanes, to be transposed
          load8(c, v);
#pragma unroll
          for (int st = 4; st >= 1; st >>= 1)
#pragma unroll
            for (int k = 0; k < 8; ++k)
              if (!(k & st)) {
                const bool up = (lane & st) != 0;
                const float2 send = up ? v[k] : v[k | st];
                const float2 got =
                    make_float2(__shfl_xor_sync(0xffffffffu, send.x, st), __shfl_xor_sync(0xffffffffu, send.y, st));
                if (up) v[k] = got; else v[k | st] = got;
              }
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int to = __shfl_sync(0xffffffffu, rel, (lane & 24) + k);
            if (to >= 0) *reinterpret_cast<float2*>(dst + to) = v[k];
          }
        }
      } else if (warp_rows > 0) {
        dst += rel;
#pragma unroll 1
        for (int c = 0; c < opaque(D / 32); ++c, dst += 16) {
          float2 v[8];
          load8(c, v);
          if (rel >= 0)
#pragma unroll
            for (int k = 0; k < 8; ++k) *reinterpret_cast<float2*>(dst + 2 * k) = v[k];
        }
      }
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars[B_OFREE]);
      i += nt;
    }
  }

  __syncwarp();  // the MMA warps reconverge after their single-lane loops
  tc::fence_before_sync();
  __syncthreads();
  if (threadIdx.x == 0) record_abort(abort_flag, p.status);
  if (warp == kSWarp) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, kTmemCols);
  }
}

// ------------------------------------------------------------------- host
template <int D>
cudaError_t launch_typed(const AttnArgs& a, cudaStream_t st) {
  using C = WideCfg<D>;
  static PerDevice<int> allowed;
  const int limit = smem_optin_bytes();
  cudaError_t e = allow_smem(allowed, tree_attn_wide_kernel<D>, limit);
  if (e != cudaSuccess) return e;
  // As many stages as fit, the K ring first: S runs up to three tiles ahead of
  // P.V, so the keys are needed earlier than the values.
  int nk = kMaxStages, nv = kMaxStages;
  while ((nk > 2 || nv > 2) && C::smem_bytes(a.B, nk, nv) > (size_t)limit) {
    if (nv >= nk && nv > 2)
      --nv;
    else
      --nk;
  }
  if (C::smem_bytes(a.B, nk, nv) > (size_t)limit) return cudaErrorNotSupported;
  const int group = a.H / a.Hkv;
  CUtensorMap mq, mk, mv;
  const long long kv_rows = (long long)a.B * a.Hkv * a.S_cap;
  if (!make_bf16_rows3_map(&mq, a.q, D, a.H, (long long)a.B * a.nq, group, kBM / group) ||
      !make_bf16_map(&mk, a.K, kv_rows, D, D, kBN) || !make_bf16_map(&mv, a.V, kv_rows, D, D, kBN))
    return cudaErrorNotSupported;
  WideParams p;
  p.kv_len = a.kv_len;
  p.parent = a.parent;
  p.out = a.out;
  unsigned char* ws = static_cast<unsigned char*>(a.ws);
  p.status = reinterpret_cast<unsigned*>(ws);
  p.ranges = reinterpret_cast<int2*>(ws + WsLayout::ranges_off(a.B, a.H));
  p.partials = reinterpret_cast<float*>(ws + WsLayout::partials_off(a.B, a.H));
  p.B = a.B; p.H = a.H; p.Hkv = a.Hkv; p.group = group; p.S_cap = a.S_cap;
  p.max_kv_len = a.max_kv_len; p.n = a.nq;
  p.rows = a.nq * group;
  p.R = (p.rows + kBM - 1) / kBM;
  p.tree = a.tree;
  p.nk = nk;
  p.nv = nv;
  p.scale_log2 = a.scale * kLog2e;
  // G shares of the key tiles, R CTAs (row tiles) per share
  const long long tiles_ub = (long long)a.B * a.Hkv * ((a.max_kv_len + (a.tree ? a.nq : 0) + kBN - 1) / kBN);
  long long G = a.max_ctas > 0 ? a.max_ctas : sm_count() / p.R;
  if (G > kMaxCtas) G = kMaxCtas;
  if (G > tiles_ub) G = tiles_ub;
  if (G < 1) G = 1;
  e = launch_pdl(tree_attn_wide_kernel<D>, dim3((unsigned)(G * p.R)), dim3(kThreads),
                             C::smem_bytes(a.B, nk, nv), st, mq, mk, mv, p);
  if (e != cudaSuccess) return e;
  return launch_tree_merge<D>(p.ranges, p.partials, p.out, a.B * a.Hkv, p.rows, group, a.H, a.Hkv, st);
}

}  // namespace

cudaError_t launch_tree_attn_wide(const AttnArgs& a, cudaStream_t st) {
  if (a.dtype != 0 || (a.D != 128 && a.D != 64) || a.Hkv < 1) return cudaErrorNotSupported;
  const int group = a.H / a.Hkv;
  // Grouped-query slabs, and any slab of more than 64 rows; multi-head slabs
  // of up to 64 rows stream faster through the 64-row kernel's deeper rings.
  if ((group == 1 && a.nq <= 64) || a.nq * group > kMaxRows || kBM % group != 0) return cudaErrorNotSupported;
  // 32-bit TMA coordinates, including a tile's reach past the last row
  if ((long long)a.B * a.Hkv * a.S_cap + kBN > 0x7fffffffLL || (long long)a.B * a.nq + kBM > 0x7fffffffLL)
    return cudaErrorNotSupported;
  if (a.D == 128) return launch_typed<128>(a, st);
  return launch_typed<64>(a, st);
}

}  // namespace glide
