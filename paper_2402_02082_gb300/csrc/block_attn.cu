// The draft's cross-attention at training time under the block-wise mask
// (Section 3.1, "Block-wise Attention Mask") on the tcgen05 tensor cores.
//
// Position j of a training sequence attends to the target's keys and values
// of the positions k < L * (j / L), the blocks before its own.  Over T
// positions that is a lower-triangular attention of about T^2 / 2 (query,
// key) pairs at 4 D flops each: a compute-bound product, unlike the
// memory-bound decoding kernels.  Both products run on the tensor cores:
//   S = Q K^T   : M = 128 positions, N = 128 keys, K = D, operands in shared memory
//   O += P V    : M = 128, N = D, K = 128 keys, P in tensor memory, V in shared memory
// Q and K sit in shared memory in the 128-byte-swizzled K-major layout, V in
// the M/N-major layout.  Tensor memory (TMEM, 512 columns) holds three S
// buffers of 128 columns and the O accumulator (D columns).
//
// What bounds it.  The two products of a 128 x 128 tile take the tensor pipe
// ~1050 cycles; a softmax warp takes ~1500 on its 32 rows (S from TMEM, row
// max, 128 exponentials a row, P back), a serial chain whatever runs beside
// it.  Two softmax groups therefore take the tiles in turn, one thread per
// position with its whole 128-key row: each has two tile periods for its chain.
// A tile takes ~1400 cycles (the groups on the two key halves of every tile,
// meeting in a row-max exchange: ~2200): still the chain, with the round trips
// of S and P between the roles, not the pipe, which is 54% busy over a call.  The
// reference max of the online softmax passes from tile to tile, so from group to
// group, through shared memory right after a tile's row
// max is known; a group keeps its own row sum and takes it to the item's last
// reference at the end.  P (bf16 pairs) overwrites the first 64 columns of its
// S buffer.  S of tile i + 3 reuses the buffer of tile i, so it waits for the
// completion of P.V of tile i; three buffers keep that off the softmax's path.
//
// Code size.  Every role's loop competes for the instruction cache: with the
// softmax unrolled over a whole row the same schedule took 190 us, with the
// loops below 64 scores at a time, rolled, 139 us at the shape below (stalls
// for want of an instruction: 26% of all, then 4%).  So loops are rolled where
// they can be, waits are small, and the optimizer is kept from copying them.
//
// At an item's end everything hangs on how soon the next one starts: the
// epilogue warps read all of O at once (168 registers a thread) before they
// store it, Q has two buffers, and the rows of the last V tile past the item's
// keys are cleared by the value producer's idle lanes.  K and V rings of two
// stages each (D = 128) are what fits beside that; the epilogue stages O / l in
// 4 KB boxes of shared memory (the 128-byte swizzle) and writes them with bulk
// tensor stores, which drain while the warps go on.
//
// Measured at B = 4, T = 2048, 32 heads, D = 128, L = 5: 139.6 -> 112.7 us in
// bursts of a few ms, 65% of the measured bf16 rate, 142.6 -> 122.2 us (60%)
// sustained over a second; B = 5, T = 1818, 32 over 8 heads, L = 4, ragged:
// 165.9 -> 127.4 us.  What is left: ~1500 cycles of every item's switch, waits
// for K and V tiles that the other SMs' traffic delays, and CTAs with one pair
// more than others.
//
// Work item: (sequence b, query head h, tile of 128 positions).  Tile x of a
// (b, h) sees about x + 1 key tiles, so tile x is paired with tile
// T/128 - 1 - x and every pair carries the same number of key tiles.  CTA c
// runs pairs c, c + G, c + 2G, ... in (b, h)-major order: the CTAs that run at
// the same time read the keys and values of a few heads, which stay in L2.
//
// Roles (512 threads, one CTA per SM):
//   warps 0-7   softmax, two groups of four: warp w reads TMEM lane quarter
//               w % 4 of the tiles of parity w / 4; at the end of an item it
//               hands its row sums to the epilogue warps.
//   warp 8      producer of Q and K, warp 11 of V (2-D TMA by lane 0).
//   warp 9      S issue (lane 0) and the TMEM allocation.
//   warp 10     P.V issue (lane 0).  Separate issuers keep S of later tiles
//               from queueing behind the wait for this tile's P.
//   warps 12-15 epilogue: warp 12 + q reads lane quarter q of O once the
//               item's last P.V is done, frees O for the next item and writes
//               O / l, while the softmax warps are already on the next item.
//
// Online softmax in the log2 domain with a lazy reference max: O is rescaled
// in TMEM only when a tile's max exceeds the reference by more than 8 (factor
// 256); the final division by the sum taken against the same reference makes
// the result exact up to rounding.  Keys past the item's last visible key are
// masked, and their V rows are zeroed in shared memory before P.V (the cache
// beyond a sequence may hold anything, even NaN); positions at or past the
// sequence's length are written as zeros whatever their queries hold.
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

constexpr int kBM = 128;          // positions per work item (MMA rows, TMEM lanes)
constexpr int kBN = 128;          // keys per tile
constexpr int kSoftWarps = 8;     // two groups of four: the even and the odd tiles
constexpr int kProdWarp = 8;
constexpr int kSWarp = 9;
constexpr int kPVWarp = 10;
constexpr int kVProdWarp = 11;
constexpr int kEpiWarp0 = 12;    // warps 12-15: the item epilogues, one per TMEM lane quarter
constexpr int kEpiWarps = 4;
constexpr int kThreads = 512;
constexpr int kTmemCols = 512;
constexpr int kSBufs = 3;                   // S / P buffers at columns 0, 128, 256
constexpr uint32_t kTmemO = kSBufs * kBN;   // the O accumulator from column 384
constexpr uint32_t kAtom = 128 * 128;       // one 128-byte-swizzle atom of 128 rows
constexpr float kRescaleLog2 = 8.0f;

// ODONE has four slots (tile mod 4).  P.V completions are waited on only now
// and then (a rescale, the epilogue), when up to three products may still be
// in flight: P.V of tile i - 3 has completed once S of tile i has been read,
// but those of tiles i - 2 .. i may not have.  Four slots keep every such wait
// within one phase of its barrier; with two, a wait for tile i could pass on
// the completion of tile i - 2 (measured: the last tiles of a segment missing
// from O when the values arrived late from DRAM).
constexpr int B_KFULL = 0, B_KEMPTY = 4, B_VFULL = 8, B_VEMPTY = 12, B_QFULL = 16, B_SFULL = 18,
              B_PFULL = 21, B_BFREE = 24, B_ODONE = 27, B_OFREE = 31, B_MDONE = 32, B_LREADY = 34, B_LFREE = 35, B_VCLR = 36, B_QEMPTY = 40,
              kNumBars = 42;

template <int D>
struct BlkCfg {
  static constexpr int kHalves = D / 64;                // swizzle atoms across the head dim
  static constexpr uint32_t kQBytes = kHalves * kAtom;  // 128 positions x D
  static constexpr uint32_t kKV = kHalves * kAtom;      // 128 keys x D
  static constexpr uint32_t off_Q = 0;                  // two items' queries
  // epilogue staging: per epilogue warp two boxes of 32 positions x 32 fp32
  // outputs (4 KB each, 128-byte swizzle): the D/32 chunks go through them in
  // rounds of two
  static constexpr uint32_t kStage = kEpiWarps * 2 * 4096;
  static constexpr uint32_t off_stg = off_Q + 2 * kQBytes;
  static constexpr uint32_t off_K = off_stg + kStage;
  // The K ring, then the V ring, as many stages as fit.  The depths are
  // compile-time constants: a division by a run-time depth costs an issuing
  // thread ~100 cycles each.
  static constexpr unsigned kNK = D == 128 ? 2 : 4, kNV = D == 128 ? 2 : 4;
  static constexpr uint32_t off_V = off_K + kNK * kKV;
  static constexpr uint32_t off_bar = off_V + kNV * kKV;
  static constexpr uint32_t off_misc = off_bar + kNumBars * 8;
  // the item's row sums, [group][position], from the softmax to the epilogue warps
  static constexpr uint32_t off_lsum = off_misc + 16;
  // the running reference max of every position, from one softmax group to the other
  static constexpr uint32_t off_mref = off_lsum + 2 * kBM * 4;
  static constexpr size_t kSmem = 1024 + off_mref + kBM * 4;
  static_assert(kTmemO + D <= kTmemCols, "TMEM columns");
  static_assert(kSmem <= 227 * 1024, "shared memory");
};

// Division of a non-negative int below 2^31 by a fixed positive divisor d as
// one multiply and shift (Granlund and Montgomery, "Division by invariant
// integers using multiplication", 1994): with l = ceil(log2 d) and
// m = ceil(2^(31+l) / d) < 2^32, n / d = (m n) >> (31 + l) for 0 <= n < 2^31.
struct FastDiv {
  uint32_t m, s;
  int d;
  __device__ __forceinline__ int div(int n) const { return (int)(((uint64_t)m * (uint32_t)n) >> s); }
  static FastDiv make(int d) {
    int l = 0;
    while ((1ll << l) < d) ++l;
    FastDiv f;
    f.m = (uint32_t)(((1ull << (31 + l)) + (uint64_t)d - 1) / (uint64_t)d);
    f.s = 31 + l;
    f.d = d;
    return f;
  }
};

struct BlkParams {
  const int* seq_len;
  float* out;
  unsigned* status;
  int B, H, Hkv, T, S_cap, L;
  FastDiv by_L, by_H, by_group, by_npb;
  int nqt;             // position tiles per sequence
  int npb;             // tile pairs per (b, h)
  int npairs;          // B * H * npb (below 2^31)
  float scale_log2;
};

// One work item and its keys: positions j0 .. j0+127 of sequence b, query head
// h; keys [0, klen) are visible to some position of the tile, keys [0, mlim)
// to every position below the sequence's length n; nt key tiles.
struct Item {
  int b, h, j0, n, klen, mlim, nt;
};

// The items of this CTA in order: pairs blockIdx.x, +G, ...; in each pair the
// later (larger) tile first.  Items with no visible key are included.
struct Walker {
  int pair, e;
  int cb, cn;  // the last sequence looked up and its clamped length
  __device__ void start() {
    pair = blockIdx.x;
    e = 0;
    cb = -1;
    cn = 0;
  }
  __device__ bool next(const BlkParams& p, Item& it) {
    while (pair < p.npairs) {
      const int bh = p.by_npb.div(pair);
      const int k = pair - bh * p.npb;
      const int qa = p.nqt - 1 - k, qb = k;
      const int e0 = e;
      if (e == 0) {
        e = 1;
      } else {
        e = 0;
        pair += gridDim.x;
      }
      if (e0 == 1 && qb >= qa) continue;  // a pair of one tile (the middle of an odd count)
      it.b = p.by_H.div(bh);
      it.h = bh - it.b * p.H;
      if (it.b != cb) {  // consecutive pairs mostly share the sequence: one load per change
        const int n = p.seq_len[it.b];
        cb = it.b;
        cn = n < 0 ? 0 : (n > p.T ? p.T : n);
      }
      const int n = cn;
      it.n = n;
      it.j0 = (e0 == 0 ? qa : qb) * kBM;
      if (it.j0 < n) {
        const int jl = (it.j0 + kBM < n ? it.j0 + kBM : n) - 1;
        it.klen = p.L * p.by_L.div(jl);
        it.mlim = p.L * p.by_L.div(it.j0);
      } else {
        it.klen = 0;
        it.mlim = 0;
      }
      it.nt = (it.klen + kBN - 1) / kBN;
      return true;
    }
    return false;
  }
};


// One 32 x 32 fp32 box of this warp's staging (rows of 128 bytes, 16-byte
// chunk e of row r at chunk e ^ (r & 7): the 128-byte swizzle) to the output
// at (x, y, z) by a bulk tensor store from lane 0; the staging box stays in
// use until the store has read it (tc::bulk_wait_read_all).
__device__ __forceinline__ void store_box(const CUtensorMap* map, const unsigned char* box, int x, int y, int z,
                                          int lane) {
  tc::fence_async_smem();  // this lane's shared-memory writes, visible to the bulk copy
  __syncwarp();
  if (lane == 0) {
    tc::tma_store_3d(map, x, y, z, box);
    tc::bulk_commit();
  }
}

// Until the bulk store from this warp's staging box has read it.
__device__ __forceinline__ void staging_free(int lane) {
  if (lane == 0) tc::bulk_wait_read_all();
  __syncwarp();
}

// Warpgroup register split (setmaxnreg), 512 x 128 registers in all as the
// block is launched: 136 a thread for the two softmax warpgroups, 168 for the
// epilogue's (a whole row of O), 72 for the producers' and MMA issuers'.
template <int N>
__device__ __forceinline__ void regs_up() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N) : "memory");
}
template <int N>
__device__ __forceinline__ void regs_down() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N) : "memory");
}

// The hand-over of a tile's reference max between the two warps (one of each
// softmax group) of a TMEM lane quarter: named barriers 1-8, per quarter and
// tile parity; the tile's warp arrives, the next tile's warp waits.
__device__ __forceinline__ void turn_pass(int quarter, unsigned tile) {
  asm volatile("bar.arrive %0, 64;" ::"r"(1 + 2 * quarter + (int)(tile & 1)) : "memory");
}
__device__ __forceinline__ void turn_wait(int quarter, unsigned tile) {
  asm volatile("bar.sync %0, 64;" ::"r"(1 + 2 * quarter + (int)(tile & 1)) : "memory");
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
    block_attn_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                      const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO,
                      const BlkParams p) {
  using C = BlkCfg<D>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  constexpr unsigned k_stages = C::kNK, v_stages = C::kNV;  // K and V ring depths
  constexpr uint32_t off_V = C::off_V;
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + C::off_bar);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base + C::off_misc);
  float* lsum = reinterpret_cast<float*>(base + C::off_lsum);
  float* mref = reinterpret_cast<float*>(base + C::off_mref);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base + C::off_misc + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
#pragma unroll 1
    for (int b = 0; b < kNumBars; ++b) {
      const bool four = (b >= B_PFULL && b < B_PFULL + kSBufs) || b == B_OFREE || b == B_LFREE;
      mbar_init(&bars[b], b == B_LREADY ? kSoftWarps : four ? 4 : 1);  // the warps that arrive
    }
    *abort_flag = 0;
    fence_barrier_init();
  }
  pdl_wait();  // every global access and the TMEM allocation come after it
  if (warp == kSWarp) {
    tc::tmem_alloc(tmem_slot, kTmemCols);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  if (warp >= kSoftWarps && warp < kEpiWarp0) {
  regs_down<72>();
  if (warp == kProdWarp || warp == kVProdWarp) {
    // ----------------------------------------------------------- producers
    // Warp 8 loads the queries and the keys, warp 11 the values: one loop, so
    // that its code is there once.  Lane 0 issues; the other lanes are there to
    // clear the rows past an item's last visible key in its last V tile.
    const bool keys = warp == kProdWarp;
    const uint64_t pol_q = policy_evict_first(), pol_kv = policy_evict_last();
    const CUtensorMap* map = keys ? &tmK : &tmV;
    if (lane == 0) {
      tc::prefetch_tmap(map);
      if (keys) tc::prefetch_tmap(&tmQ);
    }
    unsigned char* ring = base + (keys ? C::off_K : off_V);
    uint64_t* full = &bars[keys ? B_KFULL : B_VFULL];
    uint64_t* empty = &bars[keys ? B_KEMPTY : B_VEMPTY];
    const unsigned depth = keys ? k_stages : v_stages;
    unsigned st = 0, phase = 1;  // stage and its parity as the waiter sees it
    unsigned issued = 0, q_issued = 0;
    Walker w;
    w.start();
    Item it, nx;
    nx.nt = 0;
    bool has = true, ok = true;
    while (has && ok) {
      it = nx;
      has = w.next(p, nx);
      if (it.nt == 0) continue;
      if (keys) {
        const unsigned qb = q_issued & 1;
        ok = warp_wait_small(&bars[B_QEMPTY + qb], ((q_issued >> 1) & 1) ^ 1, abort_flag);
        if (!ok) break;
        if (lane == 0) {
          mbar_arrive_expect_tx(&bars[B_QFULL + qb], C::kQBytes);
          for (int hd = 0; hd < C::kHalves; ++hd) {
            tc::tma_load_2d(base + C::off_Q + qb * C::kQBytes + hd * kAtom, &tmQ, it.h * D + hd * 64, it.b * p.T + it.j0,
                            &bars[B_QFULL + qb], pol_q);
            // the next item's Q into L2, an item ahead of its load
            if (has) tc::tma_prefetch_l2_2d(&tmQ, nx.h * D + hd * 64, nx.b * p.T + nx.j0);
          }
        }
        ++q_issued;
      }
      int row = (it.b * p.Hkv + p.by_group.div(it.h)) * p.S_cap;
      for (int t = 0; t < it.nt; ++t, row += kBN) {
        ok = warp_wait_small(&empty[st], phase, abort_flag);
        if (!ok) break;
        unsigned char* dst = ring + st * C::kKV;
        if (lane == 0) {
          mbar_arrive_expect_tx(&full[st], C::kKV);
          for (int hd = 0; hd < C::kHalves; ++hd)
            tc::tma_load_2d(dst + hd * kAtom, map, hd * 64, row, &full[st], pol_kv);
        }
        __syncwarp();
        ++issued;
        const int vrows = it.klen - t * kBN;
        if (!keys && vrows < kBN) {  // the item's last V tile: clear its rows past the last visible key
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
    if (!ok && lane == 0) {  // aborted: let issued loads land before the CTA exits
      for (unsigned j = (issued > depth ? issued - depth : 0); j < issued; ++j)
        mbar_drain(&full[j % depth], (j / depth) & 1);
      for (unsigned j = (q_issued > 2 ? q_issued - 2 : 0); j < q_issued; ++j)
        mbar_drain(&bars[B_QFULL + (j & 1)], (j >> 1) & 1);
    }
  } else if (warp == kSWarp || warp == kPVWarp) {
    // ----------------------------------------------------------- MMA issue
    // Ring positions are counted up, not divided out, and the loops hold little
    // but waits and products: the two threads' time per tile is what the tensor
    // pipe waits for between their batches.
    if (lane == 0) {
      bool ok = true;
      Walker w;
      w.start();
      Item it;
      unsigned bi = 0;  // S buffer of the tile
      uint32_t col = tmem;
      unsigned items = 0;
      if (warp == kSWarp) {
        // S(i) = Q K(i)^T into buffer i % 3, once P.V of tile i - 3 has read that buffer
        constexpr uint32_t idS = tc::idesc_bf16_f32(kBM, kBN, false, false);
        const uint64_t dQ0 = tc::sw128_desc(smem_u32(base + C::off_Q), 16, 1024);
        const uint64_t dK0 = tc::sw128_desc(smem_u32(base + C::off_K), 16, 1024);
        uint64_t dK = dK0;
        unsigned st = 0, k_phase = 0, b_phase = 1;
        while (ok && w.next(p, it)) {
          if (it.nt == 0) continue;
          const uint64_t dQ = dQ0 + (items & 1) * desc_step(C::kQBytes);
          ok = mbar_wait_small(&bars[B_QFULL + (items & 1)], (items >> 1) & 1, abort_flag);
          ++items;
#pragma unroll 1
          for (int t = it.nt; ok && t > 0; --t) {
            ok = mbar_wait_small(&bars[B_KFULL + st], k_phase, abort_flag) &&
                 mbar_wait_small(&bars[B_BFREE + bi], b_phase, abort_flag);
            if (!ok) break;
            tc::fence_after_sync();
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
              const uint64_t step = desc_step((ks >> 2) * kAtom + (ks & 3) * 32);
              tc::mma_bf16(col, dQ + step, dK + step, idS, ks > 0 ? 1u : 0u);
            }
            tc::mma_commit(&bars[B_SFULL + bi]);
            tc::mma_commit(&bars[B_KEMPTY + st]);
            if (t == 1) tc::mma_commit(&bars[B_QEMPTY + ((items - 1) & 1)]);
            dK += desc_step(C::kKV);
            if (++st == k_stages) {
              st = 0;
              k_phase ^= 1;
              dK = dK0;
            }
            col += kBN;
            if (++bi == kSBufs) {
              bi = 0;
              b_phase ^= 1;
              col = tmem;
            }
          }
        }
        tc::mma_commit(&bars[B_MDONE]);  // every MMA finished before TMEM is released
        mbar_drain(&bars[B_MDONE], 0);
      } else {
        // O (+)= P(i) V(i), P in the first 64 columns of buffer i % 3
        constexpr uint32_t idO = tc::idesc_bf16_f32(kBM, D, false, true);
        const uint64_t dV0 = tc::sw128_desc(smem_u32(base + off_V), kAtom, 1024);
        uint64_t dV = dV0;
        unsigned st = 0, v_phase = 0, p_phase = 0, od = 0;
        unsigned cleared = 0;  // bit s: parity of the clears of V stage s so far
        while (ok && w.next(p, it)) {
          if (it.nt == 0) continue;
          if (items > 0) ok = mbar_wait_small(&bars[B_OFREE], (items - 1) & 1, abort_flag);
          ++items;
          const bool partial = it.klen < it.nt * kBN;  // rows of the last V tile get cleared
          uint32_t acc = 0;
#pragma unroll 1
          for (int t = it.nt; ok && t > 0; --t) {
            ok = mbar_wait_small(&bars[B_VFULL + st], v_phase, abort_flag);
            if (ok && t == 1 && partial) {
              ok = mbar_wait_small(&bars[B_VCLR + st], (cleared >> st) & 1, abort_flag);
              cleared ^= 1u << st;
            }
            ok = ok && mbar_wait_small(&bars[B_PFULL + bi], p_phase, abort_flag);
            if (!ok) break;
            tc::fence_after_sync();
#pragma unroll
            for (int ks = 0; ks < kBN / 16; ++ks)
              tc::mma_bf16_ts(tmem + kTmemO, col + ks * 8, dV + desc_step(ks * 16 * 128), idO, ks > 0 ? 1u : acc);
            acc = 1;
            tc::mma_commit(&bars[B_BFREE + bi]);
            tc::mma_commit(&bars[B_VEMPTY + st]);
            tc::mma_commit(&bars[B_ODONE + od]);
            od = (od + 1) & 3;
            dV += desc_step(C::kKV);
            if (++st == v_stages) {
              st = 0;
              v_phase ^= 1;
              dV = dV0;
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
  }
  } else if (warp >= kEpiWarp0) {
    regs_up<168>();
    // ------------------------------------------------------------ epilogue
    // Warp 12 + q writes positions 32q .. 32q+31 of every item: O / (l_0 + l_1)
    // from TMEM lane quarter q, staged in D/32 boxes and written with bulk
    // tensor stores.  The softmax warps go on with the next item meanwhile; its
    // first P.V waits until O has been read here, so a whole row is read at once.
    const int quarter = warp - kEpiWarp0;
    const int r = quarter * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    unsigned char* stg = base + C::off_stg + quarter * 2 * 4096;  // this warp's two boxes
    bool dead = false;
    Walker w;
    w.start();
    Item it;
    unsigned i = 0, ke = 0;
    while (!dead && w.next(p, it)) {
      const int j = it.j0 + r;
      if (it.nt == 0) {  // no visible key anywhere in the tile: zeros
#pragma unroll 1
        for (int row = it.j0 + quarter * 32; row < p.T && row < it.j0 + quarter * 32 + 32; ++row)
          for (int c = lane; c < D / 4; c += 32)
            reinterpret_cast<float4*>(p.out + (((long long)it.b * p.T + row) * p.H + it.h) * D)[c] =
                make_float4(0.f, 0.f, 0.f, 0.f);
        continue;
      }
      i += it.nt;
      const unsigned jl = i - 1;  // the item's last tile
      // a position that saw no key, or past the sequence: zeros
      const bool has_value = j < it.n && p.L * p.by_L.div(j) > 0;
      dead = !warp_wait_small(&bars[B_LREADY], ke & 1, abort_flag);
      if (dead) break;
      const float inv = 1.f / (lsum[r] + lsum[kBM + r]);
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars[B_LFREE]);
      dead = !warp_wait_small(&bars[B_ODONE + (jl & 3)], (jl >> 2) & 1, abort_flag);
      if (dead) break;
      tc::fence_after_sync();
      uint32_t o[D];
#pragma unroll
      for (int c = 0; c < D / 32; ++c)
        tc::tmem_ld32(lane_base + kTmemO + c * 32, *reinterpret_cast<uint32_t(*)[32]>(o + 32 * c));
      tc::tmem_wait_ld();
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars[B_OFREE]);
      // through the two boxes in turn, and out
#pragma unroll
      for (int c = 0; c < D / 32; ++c) {
        unsigned char* box = stg + (c & 1) * 4096;
        if ((c & 1) == 0) staging_free(lane);  // the stores before have read the boxes
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const uint32_t* a = o + 32 * c + 4 * q;
          float4 v = make_float4(__uint_as_float(a[0]) * inv, __uint_as_float(a[1]) * inv,
                                 __uint_as_float(a[2]) * inv, __uint_as_float(a[3]) * inv);
          if (!has_value) v = make_float4(0.f, 0.f, 0.f, 0.f);
          *reinterpret_cast<float4*>(box + lane * 128 + ((q ^ (lane & 7)) << 4)) = v;
        }
        store_box(&tmO, box, it.h * D + c * 32, it.j0 + quarter * 32, it.b, lane);
      }
      ++ke;
    }
    if (lane == 0) tc::bulk_wait_all();  // the output stores have landed
  } else {
  regs_up<136>();
    // ------------------------------------------------------------- softmax
    const int grp = warp >> 2, quarter = warp & 3;  // this group's tiles: CTA-local index parity grp
    const int r = quarter * 32 + lane;  // this thread's position in the tile (its TMEM lane)
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    const float sl2 = p.scale_log2;
    const uint64_t sc2 = f2(sl2, sl2);
    bool dead = false;
    Walker w;
    w.start();
    Item it;
    unsigned i = 0, ke = 0;  // CTA-local tile, items with keys
    while (w.next(p, it)) {
      if (it.nt == 0) continue;  // no visible key anywhere in the tile: the epilogue warps write zeros
      const int j = it.j0 + r;
      const int rowlim = j < it.n ? p.L * p.by_L.div(j) : 0;  // keys below it are visible to this position
      float m_own = -CUDART_INF_F, l = 0.f;  // the sum over this group's tiles and the reference it is taken against
      for (int t = (int)((i ^ grp) & 1u); t < it.nt; t += 2) {
        const unsigned ti = i + t;
        const unsigned bi = ti % kSBufs;
        const uint32_t s_col = lane_base + bi * kBN;
        if (!opaque(dead)) dead = !warp_wait_small(&bars[B_SFULL + bi], (ti / kSBufs) & 1, abort_flag);
        tc::fence_after_sync();
        // keys at or past this position's limit: -inf (a suffix of the tile),
        // written back to the S buffer in the 32-key chunks that have one
        if ((t + 1) * kBN > it.mlim) {
          const int nv = rowlim - t * kBN, nv_min = __reduce_min_sync(0xffffffffu, nv);
#pragma unroll 1
          for (int c = nv_min < 0 ? 0 : nv_min >> 5; c < opaque(kBN / 32); ++c) {
            uint32_t o[32];
            tc::tmem_ld32(s_col + c * 32, o);
            tc::tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 32; ++e) o[e] = 32 * c + e < nv ? o[e] : 0xff800000u;
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
          turn_wait(quarter, ti - 1);
          m_prev = mref[r];
        }
        const bool need = tmax > m_prev + kRescaleLog2;
        const float m_used = need ? tmax : m_prev;
        mref[r] = m_used;
        turn_pass(quarter, ti);
        if (__any_sync(0xffffffffu, need) && t > 0 && !dead) {
          // O holds the P.V of this item's earlier tiles, the other group's last one included: rescale it
          dead = !warp_wait_small(&bars[B_ODONE + ((ti - 1) & 3)], ((ti - 1) >> 2) & 1, abort_flag);
          if (!dead) {
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
        }
        if (m_own != m_used) {
          l *= fast_exp2(m_own - m_used);  // m_used > m_own: 0 while there is no sum
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
      i += it.nt;
      if (((i ^ grp) & 1u) == 0) {  // the other group did the last tile: take this sum to its reference
        turn_wait(quarter, i - 1);
        const float m_last = mref[r];
        if (m_own != m_last) l *= fast_exp2(m_own - m_last);
      }

      // This group's sums to the epilogue warps (the buffer is free once they
      // have read the previous item's).
      if (!dead) dead = !warp_wait_small(&bars[B_LFREE], (ke & 1) ^ 1, abort_flag);
      lsum[grp * kBM + r] = l;
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars[B_LREADY]);
      ++ke;
    }
  }

  __syncwarp();  // the producer and MMA warps reconverge after their single-lane loops
  tc::fence_before_sync();
  __syncthreads();
  if (threadIdx.x == 0) record_abort(abort_flag, p.status);
  if (warp == kSWarp) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, kTmemCols);
  }
}

template <int D>
cudaError_t launch_typed(const AttnArgs& a, cudaStream_t st) {
  using C = BlkCfg<D>;
  static PerDevice<int> allowed;
  const int limit = smem_optin_bytes();
  cudaError_t e = allow_smem(allowed, block_attn_kernel<D>, limit);
  if (e != cudaSuccess) return e;
  if (C::kSmem > (size_t)limit) return cudaErrorNotSupported;
  CUtensorMap mq, mk, mv, mo;
  const long long kv_rows = (long long)a.B * a.Hkv * a.S_cap;
  if (!make_bf16_map(&mq, a.q, (long long)a.B * a.T, (long long)a.H * D, (long long)a.H * D, kBM) ||
      !make_bf16_map(&mk, a.K, kv_rows, D, D, kBN) || !make_bf16_map(&mv, a.V, kv_rows, D, D, kBN) ||
      !make_f32_seq_map(&mo, a.out, a.B, a.T, (long long)a.H * D))
    return cudaErrorNotSupported;
  BlkParams p;
  p.seq_len = a.kv_len;
  p.out = a.out;
  p.status = reinterpret_cast<unsigned*>(a.ws);
  p.B = a.B; p.H = a.H; p.Hkv = a.Hkv; p.T = a.T; p.S_cap = a.S_cap; p.L = a.block_L;
  p.by_L = FastDiv::make(a.block_L);
  p.by_H = FastDiv::make(a.H);
  p.by_group = FastDiv::make(a.H / a.Hkv);
  p.nqt = (a.T + kBM - 1) / kBM;
  p.npb = (p.nqt + 1) / 2;
  if ((long long)a.B * a.H * p.npb > 0x7fffffffLL) return cudaErrorNotSupported;
  p.npairs = a.B * a.H * p.npb;
  p.by_npb = FastDiv::make(p.npb);
  p.scale_log2 = a.scale * kLog2e;
  int G = a.max_ctas > 0 ? a.max_ctas : sm_count();
  if (G > p.npairs) G = p.npairs;
  if (G < 1) G = 1;
  if ((long long)p.npairs + G > 0x7fffffffLL) return cudaErrorNotSupported;  // a CTA's pair index steps by G
  return launch_pdl(block_attn_kernel<D>, dim3((unsigned)G), dim3(kThreads), C::kSmem, st, mq, mk, mv, mo, p);
}

}  // namespace

cudaError_t launch_block_attn(const AttnArgs& a, cudaStream_t st) {
  if (a.dtype != 0 || (a.D != 128 && a.D != 64) || a.block_L < 1 || a.T < 1) return cudaErrorNotSupported;
  if (reinterpret_cast<uintptr_t>(a.out) & 15) return cudaErrorNotSupported;  // bulk tensor stores
  // 32-bit TMA row coordinates, including a tile's reach past the last row
  if ((long long)a.B * a.T + kBM > 0x7fffffffLL || (long long)a.B * a.Hkv * a.S_cap + kBN > 0x7fffffffLL)
    return cudaErrorNotSupported;
  if (a.D == 128) return launch_typed<128>(a, st);
  return launch_typed<64>(a, st);
}

}  // namespace glide
