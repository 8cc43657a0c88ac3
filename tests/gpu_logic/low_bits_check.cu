// Sorts by the low nbits of keys that carry other things above them: order,
// stability and the whole keys against the host, keys alone and with values.
// Usage: low_bits_check N SEED; prints "ok" or the first difference.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <numeric>
#include <random>
#include <vector>

#include "pj_prims.cuh"

using pj::Ctx;
using pj::DBuf;
typedef unsigned long long u64;

static bool sorts(size_t n, int nbits, bool values, std::mt19937_64& rng) {
  const Ctx c{};
  const u64 low = (1ull << nbits) - 1;
  std::vector<u64> k(n), want(n);
  for (auto& x : k) x = (rng() & ~low) | (rng() % 3 ? rng() & low : rng() & low & 7u);
  std::vector<uint32_t> v(n), order(n);
  std::iota(v.begin(), v.end(), 0u);
  std::iota(order.begin(), order.end(), 0u);
  std::stable_sort(order.begin(), order.end(), [&](uint32_t a, uint32_t b) { return (k[a] & low) < (k[b] & low); });
  for (size_t i = 0; i < n; ++i) want[i] = k[order[i]];
  DBuf<u64> k0(c, n), k1(c, n);
  DBuf<uint32_t> v0(c, n), v1(c, n);
  cudaMemcpy(k0.p, k.data(), n * 8, cudaMemcpyHostToDevice);
  cudaMemcpy(v0.p, v.data(), n * 4, cudaMemcpyHostToDevice);
  const bool second = pj::radix_sort_pairs_dn<u64>(c, k0.p, values ? v0.p : nullptr, k1.p, values ? v1.p : nullptr, n,
                                                   nullptr, nbits);
  c.sync();
  cudaMemcpy(k.data(), second ? k1.p : k0.p, n * 8, cudaMemcpyDeviceToHost);
  cudaMemcpy(v.data(), second ? v1.p : v0.p, n * 4, cudaMemcpyDeviceToHost);
  if (k == want && (!values || v == order)) return true;
  printf("%zu keys by %d bits, values %d: differs\n", n, nbits, (int)values);
  return false;
}

int main(int argc, char** argv) {
  const size_t n = strtoull(argv[1], nullptr, 10);
  std::mt19937_64 rng(strtoull(argv[2], nullptr, 10));
  bool ok = true;
  try {
    for (const int nbits : {1, 5, 8, 12, 41, 57, 58, 63})
      for (const bool values : {true, false}) ok = sorts(n, nbits, values, rng) && ok;
  } catch (const pj::Error& e) {
    printf("error: %s\n", e.msg.c_str());
    return 1;
  }
  if (ok) printf("ok\n");
  return ok ? 0 : 1;
}
