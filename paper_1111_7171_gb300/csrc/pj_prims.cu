// Exclusive scan and stable LSD radix sort, written for this library.
//
// Every kernel also takes an optional device-resident item count (n_dev):
// the launch is sized for a capacity, and the kernels read the actual count
// (clamped to the capacity) when they start.  Tiles past the count exit at
// once.  This lets a captured CUDA graph run the primitives on sizes that are
// only known on the device.
//
// Scan: one kernel, each value read and written once.  A tile's start comes
// from a decoupled look-back over the tiles before it (pj_lookback.cuh).
// Up to SCAN_SMALL values are scanned by one block, without status words.
//
// Radix sort: 8-bit digits.  One kernel counts the digits of every pass at
// once; then one kernel per pass ranks a tile in shared memory, finds by
// look-back, one thread per digit, how many items of each digit the tiles
// before it hold, and writes the tile out digit by digit.  Inside a tile each
// warp owns consecutive items, handled 32 at a time; lanes holding the same
// digit find each other with eight ballots, so the rank of an item among
// equal digits follows input order and the sort is stable.  Up to RSS_TILE
// items are sorted by one block that keeps them in shared memory over all
// passes.
//
// The methods: look-back after D. Merrill and M. Garland, "Single-pass
// Parallel Prefix Scan with Decoupled Look-back" (2016); one counting kernel
// and one look-back per pass after A. Adinets and D. Merrill, "Onesweep: A
// Faster Least Significant Digit Radix Sort for GPUs" (2022).
//
// What bounds it: the ranking's instructions and the look-back's loads, not
// HBM (1.6 ms per pass over 2.17e8 8-byte keys, 0.52 ms of it by bytes).
// Ballots, because match.any takes 260 cycles per warp for random 8-bit
// digits here against about 3 per ballot; look-back, because it takes the
// counting kernel and the scan out of every pass.  Measured, before (count,
// scan and scatter kernels per pass) / now: 2.17e8 keys of 40 bits 11.0 /
// 8.7 ms, 5e6 pairs of 48 bits 484 / 406 us, 1e6 pairs of 64 bits 281 / 180
// us, 6e4 pairs of 48 bits 160 / 85 us, 6e3 pairs of 64 bits 140 / 57 us;
// sums of 2.5e7 words 152 / 91 us, of 1e4 words 14.9 / 7 us.  Blocks of 512
// threads with 8 items each: with 256 threads and 16 items the large sort
// takes 8.1 ms, but the small ones 7 to 20% more.
#include "pj_prims.cuh"

#include <algorithm>

#include "pj_lookback.cuh"

namespace pj {

namespace {

// A scan tile is 8 warps x 4 rounds x 32 lanes x 4 values; a lane's 4 values
// are one or two 16-byte loads.
constexpr int SCAN_THREADS = 256;
constexpr int SCAN_VEC = 4;
constexpr int SCAN_ROUNDS = 4;
constexpr int SCAN_WARP = 32 * SCAN_VEC * SCAN_ROUNDS;
static_assert(SCAN_TILE == SCAN_THREADS / 32 * SCAN_WARP, "scan tile");
constexpr int SCAN_SMALL_THREADS = 1024;
static_assert(SCAN_SMALL == SCAN_SMALL_THREADS / 32 * SCAN_WARP, "small scan");

__device__ __forceinline__ size_t dev_count(size_t cap, const unsigned long long* n_dev) {
  return n_dev ? (size_t)min((unsigned long long)cap, *n_dev) : cap;
}

// A lane's 4 values from p (`left` of them exist); vec: 16-byte loads are
// aligned.
__device__ __forceinline__ void vec4(const uint32_t* p, uint32_t (&v)[SCAN_VEC]) {
  const uint4 a = *reinterpret_cast<const uint4*>(p);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
template <class T>
__device__ __forceinline__ void vec4(const T* p, T (&v)[SCAN_VEC]) {
  const ulonglong2 a = reinterpret_cast<const ulonglong2*>(p)[0], b = reinterpret_cast<const ulonglong2*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void put4(uint32_t* p, const uint32_t (&v)[SCAN_VEC]) {
  *reinterpret_cast<uint4*>(p) = make_uint4(v[0], v[1], v[2], v[3]);
}
template <class T>
__device__ __forceinline__ void put4(T* p, const T (&v)[SCAN_VEC]) {
  reinterpret_cast<ulonglong2*>(p)[0] = make_ulonglong2(v[0], v[1]);
  reinterpret_cast<ulonglong2*>(p)[1] = make_ulonglong2(v[2], v[3]);
}

template <class T>
__device__ __forceinline__ void load4(const T* p, size_t left, bool vec, T (&v)[SCAN_VEC]) {
  if (vec && left >= SCAN_VEC) {
    vec4(p, v);
  } else {
#pragma unroll
    for (int k = 0; k < SCAN_VEC; ++k) v[k] = (size_t)k < left ? p[k] : T(0);
  }
}

template <class T>
__device__ __forceinline__ void store4(T* p, size_t left, bool vec, const T (&v)[SCAN_VEC]) {
  if (vec && left >= SCAN_VEC) {
    put4(p, v);
  } else {
#pragma unroll
    for (int k = 0; k < SCAN_VEC; ++k)
      if ((size_t)k < left) p[k] = v[k];
  }
}

// One tile per block of WARPS warps; a single block (status NULL) covers the
// whole input.
template <class T, int WARPS>
__global__ void __launch_bounds__(WARPS * 32) k_scan(const T* __restrict__ in, T* __restrict__ out, size_t n,
                                                     const unsigned long long* __restrict__ n_dev,
                                                     unsigned long long* __restrict__ status,
                                                     unsigned long long* __restrict__ total, bool vec) {
  constexpr size_t TILE = (size_t)WARPS * SCAN_WARP;
  __shared__ unsigned long long wsum[WARPS], before;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  n = dev_count(n, n_dev);
  const unsigned tile = blockIdx.x;
  if ((size_t)tile * TILE >= n) {  // the whole block past the count
    if (total && tile == 0 && threadIdx.x == 0) *total = 0;
    return;
  }
  const size_t base = (size_t)tile * TILE + (size_t)warp * SCAN_WARP + (size_t)lane * SCAN_VEC;
  T v[SCAN_ROUNDS][SCAN_VEC];
#pragma unroll
  for (int r = 0; r < SCAN_ROUNDS; ++r) {
    const size_t i = base + (size_t)r * 32 * SCAN_VEC;
    load4(in + i, i < n ? n - i : 0, vec, v[r]);
  }
  // v becomes the exclusive sums inside the warp's items
  unsigned long long run = 0;
#pragma unroll
  for (int r = 0; r < SCAN_ROUNDS; ++r) {
    T sum = 0;
#pragma unroll
    for (int k = 0; k < SCAN_VEC; ++k) {
      const T x = v[r][k];
      v[r][k] = sum;
      sum += x;
    }
    const T incl = warp_incl_scan(sum);
    const T add = (T)run + (incl - sum);
#pragma unroll
    for (int k = 0; k < SCAN_VEC; ++k) v[r][k] += add;
    run += __shfl_sync(FULL, incl, 31);
  }
  if (lane == 31) wsum[warp] = run;
  __syncthreads();
  if (warp == 0) {
    const unsigned long long w = lane < WARPS ? wsum[lane] : 0ull;
    const unsigned long long incl = warp_incl_scan(w);
    const unsigned long long all = __shfl_sync(FULL, incl, 31);
    if (lane < WARPS) wsum[lane] = incl - w;
    unsigned long long b = 0;
    if (status) {
      if (lane == 0) lb_store(status + tile, (tile ? LB_SUM : LB_PREFIX) | all);
      if (tile) {
        b = lookback_warp(status, tile, [&](unsigned p) {
          unsigned long long s = 0;
          for (size_t i = (size_t)p * TILE + lane; i < (size_t)(p + 1) * TILE; i += 32) s += in[i];
          return warp_sum(s);
        });
        if (lane == 0) lb_store(status + tile, LB_PREFIX | (b + all));
      }
    }
    if (lane == 0) {
      before = b;
      if (total && (size_t)(tile + 1) * TILE >= n) *total = b + all;
    }
  }
  __syncthreads();
  const T add = (T)(before + wsum[warp]);
#pragma unroll
  for (int r = 0; r < SCAN_ROUNDS; ++r) {
    const size_t i = base + (size_t)r * 32 * SCAN_VEC;
#pragma unroll
    for (int k = 0; k < SCAN_VEC; ++k) v[r][k] += add;
    store4(out + i, i < n ? n - i : 0, vec, v[r]);
  }
}

__global__ void k_widen(const uint32_t* __restrict__ in, uint64_t* __restrict__ out, size_t n) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = in[i];
}

// The digits of a sort's passes: pass p takes mask[p], at most 8 bits wide,
// from shift[p] (digits that are the same in every key are left out by the
// caller).  The mask cuts the last digit to the bits that are sorted by: keys
// may carry other things above them (the packed accepted matches).
struct Digits {
  int n;
  int shift[8];
  unsigned mask[8];
};

template <class K>
__device__ __forceinline__ unsigned digit_of(K key, int shift, unsigned mask) {
  return (unsigned)(key >> shift) & mask;
}

// Counts of every pass's digits: hist[pass * 256 + digit] (zero before).
template <class K>
__global__ void __launch_bounds__(256) k_rs_hist(const K* __restrict__ keys, size_t n, Digits dg,
                                                 uint32_t* __restrict__ hist,
                                                 const unsigned long long* __restrict__ n_dev) {
  __shared__ uint32_t h[8 * 256];
  n = dev_count(n, n_dev);
  if ((size_t)blockIdx.x * 256 >= n) return;
  for (int k = threadIdx.x; k < dg.n * 256; k += 256) h[k] = 0;
  __syncthreads();
  for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (size_t)gridDim.x * 256) {
    const K key = keys[i];
#pragma unroll
    for (int p = 0; p < 8; ++p)
      if (p < dg.n) atomicAdd(&h[p * 256 + digit_of(key, dg.shift[p], dg.mask[p])], 1u);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < dg.n * 256; k += 256)
    if (h[k]) atomicAdd(&hist[k], h[k]);
}

constexpr int RS_THREADS = 512;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_ROUNDS = RS_TILE / RS_THREADS;  // items per lane
constexpr int RS_WARP_ITEMS = 32 * RS_ROUNDS;
static_assert(RS_THREADS >= 256, "one thread per digit");

// The ranks of a warp's items among its items of the same digit, in input
// order: rank[r] for this lane's item of round r, counted in cnt[digit].
template <int ROUNDS, class Digit>
__device__ __forceinline__ void warp_ranks(uint32_t* cnt, Digit digit, uint32_t (&rank)[ROUNDS]) {
  const unsigned lt = lanemask_lt();
  const unsigned gt = ~(lt | 1u << (threadIdx.x & 31));
  volatile uint32_t* const c = cnt;
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const unsigned d = digit(r);
    unsigned peers = FULL;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const unsigned m = __ballot_sync(FULL, (d >> b) & 1u);
      const unsigned no = ~(unsigned)((int)(d << (31 - b)) >> 31);  // all ones where the bit is clear
      peers &= m ^ no;
    }
    rank[r] = c[d] + (uint32_t)__popc(peers & lt);
    __syncwarp();
    if (!(peers & gt)) c[d] = rank[r] + 1;  // the digit's last lane
    __syncwarp();
  }
}

// Exclusive scan of one value per thread over the block's first 256 threads;
// every thread of the block calls it.
__device__ __forceinline__ uint32_t block_excl_256(uint32_t v, uint32_t* wsum) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t incl = warp_incl_scan(v);
  if (lane == 31 && warp < 8) wsum[warp] = incl;
  __syncthreads();
  uint32_t before = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) before += w < warp ? wsum[w] : 0u;
  __syncthreads();
  return before + incl - v;
}

template <class K>
constexpr size_t rs_shared() {
  return RS_TILE * sizeof(K) + (RS_WARPS + 2) * 256 * 4;
}

// One pass, a tile per block.  VALS false: keys only.
// Places past the count hold all-ones keys: they rank last in the last tile
// and are not written.
template <class K, bool VALS>
__global__ void __launch_bounds__(RS_THREADS, 3) k_rs_pass(const K* __restrict__ kin,
                                                           const uint32_t* __restrict__ vin, K* __restrict__ kout,
                                                           uint32_t* __restrict__ vout, size_t n, int shift,
                                                           unsigned mask, const uint32_t* __restrict__ hist,
                                                           unsigned long long* __restrict__ status,
                                                           const unsigned long long* __restrict__ n_dev) {
  extern __shared__ __align__(16) unsigned char smem[];
  K* const stage = reinterpret_cast<K*>(smem);
  uint32_t* const vstage = reinterpret_cast<uint32_t*>(smem);
  uint32_t* const wcnt = reinterpret_cast<uint32_t*>(stage + RS_TILE);  // [warp][digit]
  uint32_t* const local_start = wcnt + RS_WARPS * 256;
  uint32_t* const out_start = local_start + 256;
  __shared__ uint32_t wsum[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  n = dev_count(n, n_dev);
  const unsigned tile = blockIdx.x;
  const size_t tbase = (size_t)tile * RS_TILE;
  if (tbase >= n) return;
  const int items = (int)min((size_t)RS_TILE, n - tbase);
  kin += tbase;
  for (int d = tid; d < RS_WARPS * 256; d += RS_THREADS) wcnt[d] = 0;
  const int wbase = warp * RS_WARP_ITEMS + lane;
  K key[RS_ROUNDS];
#pragma unroll
  for (int r = 0; r < RS_ROUNDS; ++r) key[r] = wbase + r * 32 < items ? kin[wbase + r * 32] : ~K(0);
  __syncthreads();
  uint32_t rank[RS_ROUNDS];
  warp_ranks(wcnt + warp * 256, [&](int r) { return digit_of(key[r], shift, mask); }, rank);
  __syncthreads();
  // one thread per digit
  const int d = tid;
  uint32_t cnt = 0;
  unsigned long long* const mine = status + (size_t)tile * 256 + (d & 255);
  if (d < 256) {
#pragma unroll
    for (int w = 0; w < RS_WARPS; ++w) {  // the warps' starts inside the digit
      const uint32_t t = wcnt[w * 256 + d];
      wcnt[w * 256 + d] = cnt;
      cnt += t;
    }
    lb_store(mine, (tile ? LB_SUM : LB_PREFIX) | cnt);
  }
  const uint32_t start = block_excl_256(cnt, wsum);
  const uint32_t digit_start = block_excl_256(d < 256 ? hist[d] : 0u, wsum);
  if (d < 256) {
    local_start[d] = start;
    // items of digit d in the tiles before this one, four tiles a step
    unsigned long long before = 0;
    bool done = tile == 0;
    for (int hi = (int)tile - 1; !done; hi -= 4) {
      unsigned long long s[4];
      const unsigned long long* at = mine - (size_t)((int)tile - hi) * 256;
#pragma unroll
      for (int k = 0; k < 4; ++k) s[k] = hi - k >= 0 ? lb_load(at - k * 256) : LB_PREFIX;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (done) continue;
        for (int poll = 0; poll < LB_POLLS && (s[k] >> 62) == 0; ++poll) s[k] = lb_load(at - k * 256);
        if ((s[k] >> 62) == 0) {  // not published: count the digit in that tile's input
          unsigned c = 0;
          const K* in = kin - (size_t)((int)tile - (hi - k)) * RS_TILE;
#pragma unroll 1
          for (unsigned i = 0; i < RS_TILE; ++i) c += digit_of(in[i], shift, mask) == (unsigned)d;
          s[k] = LB_SUM | c;
        }
        before += s[k] & LB_VALUE;
        done = (s[k] >> 62) == 2;
      }
    }
    if (tile) lb_store(mine, LB_PREFIX | (before + cnt));
    // where the tile's item at position j (by digit) goes: out_start + j
    out_start[d] = digit_start + (uint32_t)before - start;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < RS_ROUNDS; ++r) {
    const unsigned k = digit_of(key[r], shift, mask);
    rank[r] += local_start[k] + wcnt[warp * 256 + k];
    stage[rank[r]] = key[r];
  }
  __syncthreads();
  uint32_t to[VALS ? RS_ROUNDS : 1];
#pragma unroll
  for (int r = 0; r < RS_ROUNDS; ++r) {
    const int j = r * RS_THREADS + tid;
    if (j < items) {
      const K k = stage[j];
      const uint32_t pos = out_start[digit_of(k, shift, mask)] + (uint32_t)j;
      kout[pos] = k;
      if (VALS) to[r] = pos;
    }
  }
  if (VALS) {
    vin += tbase;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r)
      if (wbase + r * 32 < items) vstage[rank[r]] = vin[wbase + r * 32];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) {
      const int j = r * RS_THREADS + tid;
      if (j < items) vout[to[r]] = vstage[j];
    }
  }
}

// All passes over at most RSS_TILE items by one block; the items stay in
// shared memory and leave in the input arrays' places.
constexpr int RSS_THREADS = 1024;
constexpr int RSS_WARPS = RSS_THREADS / 32;
constexpr int RSS_ROUNDS = RSS_TILE / RSS_THREADS;

template <class K>
constexpr size_t rss_shared(bool vals) {
  return (size_t)RSS_TILE * (sizeof(K) + (vals ? 4 : 0)) + RSS_WARPS * 256 * 4 + 256 * 4;
}

template <class K, bool VALS, int ROUNDS>
__global__ void __launch_bounds__(RSS_THREADS) k_rs_small(K* __restrict__ keys, uint32_t* __restrict__ vals, int n,
                                                          Digits dg) {
  extern __shared__ __align__(16) unsigned char smem[];
  K* const sk = reinterpret_cast<K*>(smem);
  uint32_t* const start = reinterpret_cast<uint32_t*>(sk + RSS_TILE);
  uint32_t* const sv = start + 256;
  uint32_t* const wcnt = sv + (VALS ? RSS_TILE : 0);
  __shared__ uint32_t wsum[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wbase = warp * ROUNDS * 32 + lane;
  K key[ROUNDS];
  uint32_t val[ROUNDS];
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const int i = wbase + r * 32;
    key[r] = i < n ? keys[i] : ~K(0);  // past the count: last in every pass
    val[r] = VALS && i < n ? vals[i] : 0u;
  }
  for (int p = 0; p < dg.n; ++p) {
    const int shift = dg.shift[p];
    const unsigned mask = dg.mask[p];
    for (int k = tid; k < RSS_WARPS * 256; k += RSS_THREADS) wcnt[k] = 0;
    __syncthreads();
    uint32_t rank[ROUNDS];
    warp_ranks(wcnt + warp * 256, [&](int r) { return digit_of(key[r], shift, mask); }, rank);
    __syncthreads();
    uint32_t cnt = 0, incl = 0;
    if (tid < 256) {
#pragma unroll
      for (int w = 0; w < RSS_WARPS; ++w) {
        const uint32_t t = wcnt[w * 256 + tid];
        wcnt[w * 256 + tid] = cnt;
        cnt += t;
      }
      incl = warp_incl_scan(cnt);
      if (lane == 31) wsum[warp] = incl;
    }
    __syncthreads();
    if (tid < 256) {
      uint32_t before = 0;
#pragma unroll
      for (int w = 0; w < 8; ++w) before += w < warp ? wsum[w] : 0u;
      start[tid] = before + incl - cnt;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
      const unsigned d = digit_of(key[r], shift, mask);
      const uint32_t at = start[d] + wcnt[warp * 256 + d] + rank[r];
      sk[at] = key[r];
      if (VALS) sv[at] = val[r];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
      key[r] = sk[wbase + r * 32];
      if (VALS) val[r] = sv[wbase + r * 32];
    }
  }
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const int i = wbase + r * 32;
    if (i < n) {
      keys[i] = key[r];
      if (VALS) vals[i] = val[r];
    }
  }
}

// 8-bit digits over the set bits of `bits`, from the lowest up.
Digits digits_of(unsigned long long bits) {
  Digits dg{};
  for (int s = 0; s < 64;) {
    if (!((bits >> s) & 1ull)) {
      ++s;
      continue;
    }
    if (dg.n == 8) fail(PJ_EINVAL, "radix sort: more than 8 digits");
    dg.shift[dg.n] = s;
    dg.mask[dg.n++] = (unsigned)(bits >> s) & 0xFFu;
    s += 8;
  }
  return dg;
}

template <class K, bool VALS, int ROUNDS>
void sort_small(const Ctx& c, K* keys, uint32_t* vals, int n, const Digits& dg) {
  constexpr int bytes = (int)rss_shared<K>(VALS);
  PJ_CUDA(cudaFuncSetAttribute(k_rs_small<K, VALS, ROUNDS>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  k_rs_small<K, VALS, ROUNDS><<<1, RSS_THREADS, bytes, c.stream>>>(keys, vals, n, dg);
  PJ_LAUNCHED("k_rs_small");
}

template <class K, bool VALS>
void sort_small(const Ctx& c, K* keys, uint32_t* vals, size_t n, const Digits& dg) {
  if (n <= RSS_THREADS) sort_small<K, VALS, 1>(c, keys, vals, (int)n, dg);
  else if (n <= 3 * RSS_THREADS) sort_small<K, VALS, 3>(c, keys, vals, (int)n, dg);
  else sort_small<K, VALS, RSS_ROUNDS>(c, keys, vals, (int)n, dg);
}

}  // namespace

template <class T>
void exclusive_scan_dn(const Ctx& c, const T* in, T* out, size_t cap, const unsigned long long* n_dev,
                       unsigned long long* total) {
  if (cap == 0) {
    if (total) PJ_CUDA(cudaMemsetAsync(total, 0, sizeof(*total), c.stream));
    return;
  }
  const bool vec = ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
  if (cap <= SCAN_SMALL) {
    k_scan<T, SCAN_SMALL_THREADS / 32><<<1, SCAN_SMALL_THREADS, 0, c.stream>>>(in, out, cap, n_dev, nullptr, total, vec);
    PJ_LAUNCHED("k_scan");
    return;
  }
  const unsigned tiles = ceil_div(cap, SCAN_TILE);
  DBuf<unsigned long long> status(c, tiles);
  PJ_CUDA(cudaMemsetAsync(status.p, 0, status.bytes(), c.stream));
  k_scan<T, SCAN_THREADS / 32><<<tiles, SCAN_THREADS, 0, c.stream>>>(in, out, cap, n_dev, status.p, total, vec);
  PJ_LAUNCHED("k_scan");
}

template <class T>
void exclusive_scan(const Ctx& c, const T* in, T* out, size_t n) {
  if (n == 0) return;
  exclusive_scan_dn<T>(c, in, out, n, nullptr, nullptr);
}

template <class K>
bool radix_sort_bits_dn(const Ctx& c, K* keys, uint32_t* vals, K* keys2, uint32_t* vals2, size_t cap,
                        const unsigned long long* n_dev, unsigned long long bits) {
  if (cap == 0 || bits == 0) return false;
  if (cap > 0xFFFFFFFFull) fail(PJ_EINVAL, "radix sort: more than 2^32 items");
  const Digits dg = digits_of(bits);
  if (cap <= RSS_TILE && !n_dev) {
    if (vals) sort_small<K, true>(c, keys, vals, cap, dg);
    else sort_small<K, false>(c, keys, nullptr, cap, dg);
    return false;
  }
  const unsigned ntiles = ceil_div(cap, RS_TILE);
  // one clear for the counts of every pass and their status words
  const size_t per_pass = (size_t)256 * ntiles;
  DBuf<unsigned long long> work(c, RS_HIST_WORDS + per_pass * dg.n);
  uint32_t* hist = reinterpret_cast<uint32_t*>(work.p);
  PJ_CUDA(cudaMemsetAsync(work.p, 0, work.bytes(), c.stream));
  const unsigned gh = std::min<unsigned>(ceil_div(cap, 256 * 8), sm_grid_cap(8));
  k_rs_hist<K><<<gh, 256, 0, c.stream>>>(keys, cap, dg, hist, n_dev);
  PJ_LAUNCHED("k_rs_hist");
  constexpr int bytes = (int)rs_shared<K>();
  if (vals) PJ_CUDA(cudaFuncSetAttribute(k_rs_pass<K, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  else PJ_CUDA(cudaFuncSetAttribute(k_rs_pass<K, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  K* ka = keys;
  uint32_t* va = vals;
  K* kb = keys2;
  uint32_t* vb = vals2;
  for (int p = 0; p < dg.n; ++p) {
    unsigned long long* status = work.p + RS_HIST_WORDS + per_pass * p;
    if (vals)
      k_rs_pass<K, true><<<ntiles, RS_THREADS, bytes, c.stream>>>(ka, va, kb, vb, cap, dg.shift[p], dg.mask[p],
                                                              hist + 256 * p, status, n_dev);
    else
      k_rs_pass<K, false><<<ntiles, RS_THREADS, bytes, c.stream>>>(ka, nullptr, kb, nullptr, cap, dg.shift[p], dg.mask[p],
                                                               hist + 256 * p, status, n_dev);
    PJ_LAUNCHED("k_rs_pass");
    K* tk = ka; ka = kb; kb = tk;
    uint32_t* tv = va; va = vb; vb = tv;
  }
  return ka != keys;
}

template <class K>
bool radix_sort_pairs_dn(const Ctx& c, K* keys, uint32_t* vals, K* keys2, uint32_t* vals2, size_t cap,
                         const unsigned long long* n_dev, int nbits) {
  if (nbits <= 0) return false;
  return radix_sort_bits_dn<K>(c, keys, vals, keys2, vals2, cap, n_dev, nbits >= 64 ? ~0ull : (1ull << nbits) - 1);
}

template <class K>
void radix_sort_bits(const Ctx& c, K* keys, uint32_t* vals, size_t n, unsigned long long bits) {
  if (n <= 1 || bits == 0) return;
  const bool small = n <= RSS_TILE;  // sorted in place
  DBuf<K> k2;
  DBuf<uint32_t> v2;
  if (!small) {
    k2.reset(c, n);
    v2.reset(c, n);
  }
  if (radix_sort_bits_dn<K>(c, keys, vals, k2.p, v2.p, n, nullptr, bits)) {
    PJ_CUDA(cudaMemcpyAsync(keys, k2.p, n * sizeof(K), cudaMemcpyDeviceToDevice, c.stream));
    PJ_CUDA(cudaMemcpyAsync(vals, v2.p, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, c.stream));
  }
}

template <class K>
void radix_sort_pairs(const Ctx& c, K* keys, uint32_t* vals, size_t n, int nbits) {
  if (nbits <= 0) return;
  radix_sort_bits<K>(c, keys, vals, n, nbits >= 64 ? ~0ull : (1ull << nbits) - 1);
}

void widen_u32(const Ctx& c, const uint32_t* in, uint64_t* out, size_t n) {
  if (n == 0) return;
  k_widen<<<ceil_div(n, 256), 256, 0, c.stream>>>(in, out, n);
  PJ_LAUNCHED("k_widen");
}

template void exclusive_scan_dn<uint32_t>(const Ctx&, const uint32_t*, uint32_t*, size_t,
                                          const unsigned long long*, unsigned long long*);
template void exclusive_scan_dn<unsigned long long>(const Ctx&, const unsigned long long*, unsigned long long*, size_t,
                                                    const unsigned long long*, unsigned long long*);
template bool radix_sort_pairs_dn<unsigned long long>(const Ctx&, unsigned long long*, uint32_t*, unsigned long long*,
                                                      uint32_t*, size_t, const unsigned long long*, int);
template void exclusive_scan<uint32_t>(const Ctx&, const uint32_t*, uint32_t*, size_t);
template void exclusive_scan<uint64_t>(const Ctx&, const uint64_t*, uint64_t*, size_t);
template void exclusive_scan<unsigned long long>(const Ctx&, const unsigned long long*, unsigned long long*, size_t);
template void radix_sort_pairs<uint32_t>(const Ctx&, uint32_t*, uint32_t*, size_t, int);
template void radix_sort_pairs<unsigned long long>(const Ctx&, unsigned long long*, uint32_t*, size_t, int);
template void radix_sort_bits<unsigned long long>(const Ctx&, unsigned long long*, uint32_t*, size_t,
                                                  unsigned long long);

}  // namespace pj
