// The device primitives against the host: exclusive sums, stable sorts by
// nbits (values follow their keys, so stability shows in them), keys alone,
// and sorts by chosen bits; with the count on the host and on the device.
// Usage: prims_check N SEED; prints "ok" or the first difference.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <numeric>
#include <random>
#include <vector>

#include "pj_prims.cuh"

using pj::Ctx;
using pj::DBuf;
typedef unsigned long long u64;

static bool same(const char* what, const void* got, const void* want, size_t bytes) {
  if (memcmp(got, want, bytes) == 0) return true;
  printf("%s differs\n", what);
  return false;
}

template <class T>
static void up(const Ctx& c, DBuf<T>& d, const std::vector<T>& h) {
  d.reset(c, h.size());
  cudaMemcpy(d.p, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice);
}
template <class T>
static std::vector<T> down(const T* p, size_t n) {
  std::vector<T> h(n);
  cudaMemcpy(h.data(), p, n * sizeof(T), cudaMemcpyDeviceToHost);
  return h;
}

template <class T>
static bool scans(const Ctx& c, size_t n, size_t cap, std::mt19937_64& rng, T top) {
  std::vector<T> in(cap), want(n);
  for (auto& x : in) x = (T)(rng() % top);
  u64 sum = 0;
  for (size_t k = 0; k < n; ++k) {
    want[k] = (T)sum;
    sum += in[k];
  }
  DBuf<T> d, o;
  DBuf<u64> nd(c, 1), tot(c, 1);
  up(c, d, in);
  o.reset(c, cap);
  const u64 n64 = n;
  cudaMemcpy(nd.p, &n64, 8, cudaMemcpyHostToDevice);
  pj::exclusive_scan_dn<T>(c, d.p, o.p, cap, cap == n ? nullptr : nd.p, tot.p);
  c.sync();
  const auto got = down(o.p, n);
  const auto t = down(tot.p, 1);
  return same("scan", got.data(), want.data(), n * sizeof(T)) && same("total", t.data(), &sum, 8);
}

// keys with `distinct` different values below 2^nbits
static bool sorts(const Ctx& c, size_t n, size_t cap, int nbits, u64 distinct, bool values, std::mt19937_64& rng) {
  std::vector<u64> k(cap), alphabet(std::min<u64>(distinct, 1u << 16));
  for (auto& x : alphabet) x = rng() & (nbits == 64 ? ~0ull : (1ull << nbits) - 1);
  for (auto& x : k) x = distinct > alphabet.size() ? rng() & (nbits == 64 ? ~0ull : (1ull << nbits) - 1)
                                                   : alphabet[rng() % alphabet.size()];
  std::vector<uint32_t> v(cap), order(n);
  for (size_t i = 0; i < cap; ++i) v[i] = (uint32_t)i;
  std::iota(order.begin(), order.end(), 0u);
  std::stable_sort(order.begin(), order.end(), [&](uint32_t a, uint32_t b) { return k[a] < k[b]; });
  std::vector<u64> want(n);
  for (size_t i = 0; i < n; ++i) want[i] = k[order[i]];
  DBuf<u64> k0, k1(c, cap), nd(c, 1);
  DBuf<uint32_t> v0, v1(c, cap);
  up(c, k0, k);
  up(c, v0, v);
  const u64 n64 = n;
  cudaMemcpy(nd.p, &n64, 8, cudaMemcpyHostToDevice);
  const bool second = pj::radix_sort_pairs_dn<u64>(c, k0.p, values ? v0.p : nullptr, k1.p, values ? v1.p : nullptr, cap,
                                                   cap == n ? nullptr : nd.p, nbits);
  c.sync();
  const auto gk = down(second ? k1.p : k0.p, n);
  const auto gv = down(second ? v1.p : v0.p, n);
  return same("keys", gk.data(), want.data(), n * 8) && (!values || same("values", gv.data(), order.data(), n * 4));
}

// keys whose differing bits are `bits`
static bool bit_sort(const Ctx& c, size_t n, u64 bits, std::mt19937_64& rng) {
  std::vector<u64> k(n);
  for (auto& x : k) x = rng() & bits;
  std::vector<uint32_t> v(n), order(n);
  std::iota(v.begin(), v.end(), 0u);
  std::iota(order.begin(), order.end(), 0u);
  std::stable_sort(order.begin(), order.end(), [&](uint32_t a, uint32_t b) { return k[a] < k[b]; });
  DBuf<u64> dk;
  DBuf<uint32_t> dv;
  up(c, dk, k);
  up(c, dv, v);
  pj::radix_sort_bits<u64>(c, dk.p, dv.p, n, bits);
  c.sync();
  const auto got = down(dv.p, n);
  return same("bit sort", got.data(), order.data(), n * 4);
}

int main(int argc, char** argv) {
  const size_t n = strtoull(argv[1], nullptr, 10);
  std::mt19937_64 rng(strtoull(argv[2], nullptr, 10));
  const Ctx c{};
  bool ok = true;
  try {
    for (const size_t cap : {n, n + 1, 3 * n + 5000}) {
      ok = ok && scans<uint32_t>(c, n, cap, rng, 5) && scans<u64>(c, n, cap, rng, 1ull << 40);
      for (const bool values : {true, false}) {
        ok = ok && sorts(c, n, cap, 41, ~0ull, values, rng) && sorts(c, n, cap, 64, 3, values, rng) &&
             sorts(c, n, cap, 5, ~0ull, values, rng) && sorts(c, n, cap, 16, 1, values, rng);
      }
    }
    ok = ok && bit_sort(c, n, ~0ull << 32 | 0x3F07ull, rng) && bit_sort(c, n, ~0ull << 32 | 0x1FF3Full, rng);
    c.sync();
  } catch (const pj::Error& e) {
    printf("error: %s\n", e.msg.c_str());
    return 1;
  }
  if (ok) printf("ok\n");
  return ok ? 0 : 1;
}
