// Host-side print of which kernel takes an fp32 verification or grouped-query call (runtime faked): reads
// "B H H_kv D keys n tree" lines, prints the CTAs of tree_direct.cu's launch, 0 for the streaming kernel.
#include "fake_cudart.cuh"

#include "kernels.h"
#include "tree_direct.cu"

int main() {
  alignas(16) static unsigned char buffer[64];
  int B, H, Hkv, D, keys, n, tree;
  while (std::scanf("%d %d %d %d %d %d %d", &B, &H, &Hkv, &D, &keys, &n, &tree) == 7) {
    glide::AttnArgs a{};
    a.q = a.K = a.V = buffer;
    a.kv_len = a.parent = reinterpret_cast<const int*>(buffer);
    a.out = reinterpret_cast<float*>(buffer);
    a.B = B;
    a.H = H;
    a.Hkv = Hkv;
    a.D = D;
    a.dtype = 1;
    a.S_cap = keys + n;
    a.max_kv_len = keys;
    a.nq = n;
    a.tree = tree;
    fake::launches.clear();
    const cudaError_t e = glide::launch_tree_direct(a, nullptr);
    if (e != cudaSuccess && e != cudaErrorNotSupported) return 1;
    std::printf("%u\n", fake::launches.empty() ? 0u : fake::launches[0].grid);
  }
  return 0;
}
