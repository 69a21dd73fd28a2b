// Checks build_share (common.cuh), which tells every CTA of the verification kernels where its share of the
// key tiles starts, against CostPartition, which the merge's bookkeeping uses (itself checked on the host by
// partition_check.cu): for seeded random batches, below and above the 32 sequences at which the lookup
// changes, with empty sequences, every share's start and size, and the batch table.  Prints "ok <cases>" and
// exits 0, or says what differs and exits 1.
#include <cstdio>
#include <random>
#include <vector>

#include "common.cuh"

namespace {

constexpr int kMostB = 80;

struct Table {
  long long start[kMostB + 1];
  int len[kMostB], ntiles[kMostB], plen[kMostB], sidx[kMostB + 1];
};

__global__ void __launch_bounds__(32) share_kernel(const int* kv_len, int B, int H, int most, int extra, int TK, int w,
                                                   glide::ShareStart* out, Table* table) {
  __shared__ Table t;
  __shared__ glide::ShareStart s;
  glide::BatchTiles bt;
  bt.start = t.start;
  bt.len = t.len;
  bt.ntiles = t.ntiles;
  bt.plen = t.plen;
  bt.sidx = t.sidx;
  glide::build_share(bt, kv_len, B, H, most, extra, TK, gridDim.x, w, blockIdx.x, &s);
  __syncwarp();
  if (threadIdx.x == 0) {
    out[blockIdx.x] = s;
    if (blockIdx.x == 0) *table = t;
  }
}

}  // namespace

int main() {
  std::mt19937 rng(20261205);
  auto pick = [&](std::initializer_list<int> v) { return *(v.begin() + rng() % v.size()); };
  int* kv;
  glide::ShareStart* out;
  Table* table;
  if (cudaMallocManaged(&kv, kMostB * sizeof(int)) != cudaSuccess ||
      cudaMallocManaged(&out, 1024 * sizeof(*out)) != cudaSuccess ||
      cudaMallocManaged(&table, sizeof(*table)) != cudaSuccess)
    return 2;
  int cases = 0, failures = 0;
  for (int it = 0; it < 600 && failures < 10; ++it, ++cases) {
    const int B = pick({1, 2, 3, 8, 31, 32, 33, 64, 80}), H = pick({1, 2, 8, 32, 52});
    const int TK = pick({64, 128}), extra = pick({0, 1, 6, 33, 64}), most = pick({1, 100, 700, 5000});
    const int G = pick({1, 2, 7, 100, 152, 1000}), w = pick({1, 4, 5, 8});
    for (int b = 0; b < B; ++b) kv[b] = pick({0, 0, 1, 63, 64, 65, 4096, (int)(rng() % 5200), -3});
    share_kernel<<<G, 32>>>(kv, B, H, most, extra, TK, w, out, table);
    if (cudaDeviceSynchronize() != cudaSuccess) return 2;
    // the table, and the partition over it
    std::vector<long long> start(B + 1);
    std::vector<int> nt(B), sidx(B + 1), len(B), plen(B);
    long long T = 0;
    int k = 0;
    bool ok = true;
    for (int b = 0; b < B; ++b) {
      plen[b] = kv[b] < 0 ? 0 : (kv[b] > most ? most : kv[b]);
      len[b] = plen[b] + extra;
      nt[b] = (len[b] + TK - 1) / TK;
      start[b] = T;
      sidx[b] = k;
      T += (long long)H * nt[b];
      if (nt[b] > 0) k += H;
      ok = ok && table->plen[b] == plen[b] && table->len[b] == len[b] && table->ntiles[b] == nt[b] &&
           table->start[b] == start[b] && table->sidx[b] == sidx[b];
    }
    start[B] = T;
    sidx[B] = k;
    ok = ok && table->start[B] == T && table->sidx[B] == k;
    if (!ok) std::printf("case %d (B=%d H=%d): batch table\n", it, B, H);
    glide::BatchTiles bt;
    bt.start = start.data();
    bt.len = len.data();
    bt.ntiles = nt.data();
    bt.plen = plen.data();
    bt.sidx = sidx.data();
    glide::CostPartition P;
    P.init(bt, B, H, G, w);
    for (int x = 0; x < G && ok; ++x) {
      const long long g0 = P.begin(x), g1 = P.end(x);
      glide::ShareStart want = {0, 0, 0, (int)(g1 - g0)};
      if (g1 > g0) {
        int b = 0;
        while (b + 1 < B && start[b + 1] <= g0) ++b;
        want.b = b;
        want.h = (int)((g0 - start[b]) / nt[b]);
        want.t0 = (int)(g0 - start[b]) - want.h * nt[b];
      }
      const glide::ShareStart& s = out[x];
      ok = s.b == want.b && s.h == want.h && s.t0 == want.t0 && s.tiles == want.tiles;
      if (!ok)
        std::printf("case %d (B=%d H=%d G=%d w=%d): share %d starts at (%d, %d, %d) with %d tiles, not (%d, %d, %d) with %d\n",
                    it, B, H, G, w, x, s.b, s.h, s.t0, s.tiles, want.b, want.h, want.t0, want.tiles);
    }
    if (!ok) ++failures;
  }
  if (failures) return 1;
  std::printf("ok %d\n", cases);
  return 0;
}
