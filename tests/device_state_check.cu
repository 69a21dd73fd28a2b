// Host-side check of what the launchers keep between calls: it belongs to the device that was current,
// not to the process.  UNIT is the csrc file, LAUNCH its number below.  Each launcher is called on
// device 0, on device 1 (fewer SMs, less room for clusters) and on device 0 again; every launch has to
// be one that its device takes.  Prints "ok" and exits 0, or says what was refused and exits 1.
#include "fake_cudart.cuh"

#include "kernels.h"
#include UNIT

namespace {

int failures = 0;
void expect(bool ok, const char* what) {
  if (ok) return;
  std::printf("%s on device %d\n", what, fake::device);
  ++failures;
}

alignas(16) unsigned char buffer[64];

[[maybe_unused]] glide::AttnArgs attention(int dtype, int D, int nq, int H, int Hkv) {
  glide::AttnArgs a{};
  a.q = a.K = a.V = buffer;
  a.kv_len = a.parent = reinterpret_cast<const int*>(buffer);
  a.out = reinterpret_cast<float*>(buffer);
  a.ws = buffer;
  a.B = 2;
  a.H = H;
  a.Hkv = Hkv;
  a.D = D;
  a.S_cap = 4096;
  a.nq = nq;
  a.max_kv_len = 2048;
  a.tree = 1;
  a.block_L = 5;
  a.T = 300;
  a.dtype = dtype;
  a.scale = 1.f;
  return a;
}

void call() {
#if LAUNCH == 0  // the runtime's own figures
  expect(glide::sm_count() == fake::sms[fake::device], "another device's SM count");
#elif LAUNCH == 1
  for (int dtype = 0; dtype < 2; ++dtype)
    for (int D = 64; D <= 128; D += 64)
      expect(glide::launch_cross_attn(attention(dtype, D, 1, 8, 8), nullptr) == cudaSuccess, "cross_attn refused");
#elif LAUNCH == 2
  for (int dtype = 0; dtype < 2; ++dtype)
    for (int D = 64; D <= 128; D += 64)
      expect(glide::launch_tree_attn_fma(attention(dtype, D, 5, 8, 8), nullptr) == cudaSuccess, "tree_attn_fma refused");
#elif LAUNCH == 3
  for (int D = 64; D <= 128; D += 64)
    expect(glide::launch_tree_attn_tc(attention(0, D, 5, 8, 8), nullptr) == cudaSuccess, "tree_attn_tc refused");
#elif LAUNCH == 4
  for (int D = 64; D <= 128; D += 64)
    expect(glide::launch_tree_attn_wide(attention(0, D, 33, 8, 2), nullptr) == cudaSuccess, "tree_attn_wide refused");
#elif LAUNCH == 5
  for (int D = 64; D <= 128; D += 64)
    expect(glide::launch_block_attn(attention(0, D, 1, 8, 8), nullptr) == cudaSuccess, "block_attn refused");
#elif LAUNCH == 6
  glide::AcceptArgs a{};
  a.logits = reinterpret_cast<const float*>(buffer);
  a.ws = buffer;
  a.B = 2;
  a.n = 5;
  a.V = 1000;
  expect(glide::launch_tree_accept(a, nullptr) == cudaSuccess, "tree_accept refused");
#elif LAUNCH == 7
  glide::SampleArgs a{};
  a.logits = a.q = a.u = reinterpret_cast<const float*>(buffer);
  a.ws = buffer;
  a.B = 4;
  a.gamma = 8;
  a.V = 1000;
  expect(glide::launch_spec_sample(a, nullptr) == cudaSuccess, "spec_sample refused");
  const fake::Launch& l = fake::launches.back();
  expect((int)(l.grid / l.cluster) <= fake::room[fake::device][l.cluster], "more clusters than the device has room for");
  expect(l.cluster > 1 || fake::device == 3, "clusters not used");
#endif
}

}  // namespace

int main() {
  for (int c = 1; c <= 16; ++c) {
    fake::room[0][c] = 304 / c;
    fake::room[1][c] = c <= 8 ? 40 / c : 0;
  }
  fake::failing_queries = LAUNCH == 7 ? 100 : 0;
#if LAUNCH == 7
  // queries that fail leave nothing behind: the call itself still works, and the next one asks again
  glide::SampleArgs a{};
  a.logits = a.q = a.u = reinterpret_cast<const float*>(buffer);
  a.ws = buffer;
  a.B = 4;
  a.gamma = 8;
  a.V = 1000;
  expect(glide::launch_spec_sample(a, nullptr) == cudaSuccess, "spec_sample without an answer refused");
  fake::failing_queries = 0;
#endif
  for (int d : {0, 1, 0, 1}) {
    fake::device = d;
    call();
  }
  const int first = fake::attribute_calls;
  for (int d : {0, 1}) {
    fake::device = d;
    call();
  }
  expect(fake::attribute_calls == first, "attributes set again");
  if (failures) return 1;
  std::printf("ok\n");
  return 0;
}
