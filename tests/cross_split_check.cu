// Host-side print of how cross_direct.cu splits a call (runtime faked, a GB300's room for clusters):
// reads "B H D f32 keys max_ctas" lines, prints the CTAs per (sequence, head), 0 for the streaming kernel.
#include "fake_cudart.cuh"

#include "kernels.h"
#include "cross_direct.cu"

int main() {
  // clusters of each size that run at once with two CTAs an SM, and with one
  const int two[9] = {0, 304, 152, 97, 74, 58, 46, 38, 36}, one[9] = {0, 152, 76, 46, 36, 28, 23, 15, 15};
  alignas(16) static unsigned char buffer[64];
  int B, H, D, f32, keys, max_ctas;
  while (std::scanf("%d %d %d %d %d %d", &B, &H, &D, &f32, &keys, &max_ctas) == 6) {
    fake::device = f32 && D == 128 ? 1 : 0;
    fake::sms[1] = fake::sms[0];
    for (int c = 1; c <= 8; ++c) fake::room[fake::device][c] = (fake::device ? one : two)[c];
    glide::AttnArgs a{};
    a.q = a.K = a.V = buffer;
    a.kv_len = reinterpret_cast<const int*>(buffer);
    a.out = reinterpret_cast<float*>(buffer);
    a.B = B;
    a.H = a.Hkv = H;
    a.D = D;
    a.dtype = f32;
    a.S_cap = a.max_kv_len = keys;
    a.nq = 1;
    a.max_ctas = max_ctas;
    fake::launches.clear();
    const cudaError_t e = glide::launch_cross_direct(a, nullptr);
    if (e == cudaErrorNotSupported && fake::launches.empty()) {
      std::printf("0\n");
      continue;
    }
    if (e != cudaSuccess || fake::launches.size() != 1) return 1;
    const fake::Launch& l = fake::launches[0];
    if ((long long)l.cluster * B * H != (long long)l.grid) return 1;
    std::printf("%u\n", l.cluster);
  }
  return 0;
}
