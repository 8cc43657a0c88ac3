// The screen-and-verify queues shared by the extension-mode kernels, and the
// one-launch query kernel built on them.
#pragma once

#include "pj_internal.cuh"
#include "pj_probe.cuh"

namespace pj {

struct Counters {
  unsigned long long accepted;
  unsigned long long lookups;
  unsigned long long candidates;
  unsigned long long cells;
  unsigned long long fallback;
  unsigned long long hits;
  unsigned long long err;  // bit 0: run or posting outside the index; bit 1: probe limit
  unsigned long long filtered;  // candidates rejected by the character-count bound
  unsigned long long tasks;     // parts of long runs that a query batch set aside (k_query_fused)
};

struct AccOut {
  unsigned long long* key;
  uint32_t* ed;
  unsigned long long cap;
};

__device__ __forceinline__ void add_counter(unsigned long long* c, unsigned long long v) {
  if (v) atomicAdd(c, v);
}

// The same by a whole warp, one atomic for its lanes' sum.  An atomic per lane
// on one address, half a million of them for a full grid with four counters,
// takes some 100 us: a plan's batch of 64 queries 244 us, 152 us by warps.
__device__ __forceinline__ void warp_add_counter(unsigned long long* c, unsigned long long v) {
  __syncwarp();
  v = warp_sum(v);
  if ((threadIdx.x & 31u) == 0) add_counter(c, v);
}

// Sizes that a kernel reads from device memory when it starts: the launch
// covers a capacity `cap`, n_dev (if not NULL) holds the actual count.
__device__ __forceinline__ unsigned long long dev_count(unsigned long long cap, const unsigned long long* n_dev) {
  return n_dev ? min(cap, *n_dev) : cap;
}

constexpr int Q_BLOCK = 256;
constexpr int Q_WARPS = Q_BLOCK / 32;
constexpr int S_RUN = 8;                 // candidates one lane screens per step
constexpr int Q_CAP = 32 * S_RUN + 32;   // < 32 left + up to 32 * S_RUN new
constexpr int Q_SECOND = 64;             // < 32 left + up to 32 new
constexpr unsigned long long Q_CHUNK = 8ull * 32 * S_RUN;  // candidates a warp takes at a time
constexpr unsigned long long Q_CHUNK_MIN = 128;            // ... in launches too small to fill the warps

// Extension verification of one queue entry: probe q, indexed sid r, and
// the match's position, segment and threshold packed in pi.
template <int MAXW, bool SELF, bool MULTI>
__device__ __forceinline__ void verify_queued_entry(const ProbeView& v, uint32_t q, uint32_t r, uint32_t pi,
                                                    AccOut out, Counters* ctr, unsigned long long& cells) {
  const ProbeView vt = MULTI ? view_for_tau(v, (int)(pi >> 24)) : v;
  HitCtx hc;
  hc.q = q;
  hc.begin = 0;
  hc.p = (int)(pi & 0xFFFFu);
  hc.i = (int)((pi >> 16) & 0xFFu);
  if (vt.pref) {
    const unsigned long long ref = vt.pref[q];
    hc.ls = (int)(ref & 0xFFFFu);
    hc.s = vt.pbytes + (ref >> 16);
  } else {
    hc.ls = (int)vt.plen[q];
    hc.s = vt.pbytes + vt.poff[q];
  }
  unsigned long long key = 0;
  int ed = 0;
  if (verify_screened<MAXW>(vt, SELF, hc, r, key, ed, cells)) {
    const unsigned long long pos = atomicAdd(&ctr->accepted, 1ull);
    if (pos < out.cap) {
      out.key[pos] = key;
      out.ed[pos] = (uint32_t)ed;
    }
  }
}

// A warp's queues in shared memory.  A screened match waits in the first
// until 32 of them are verified together; with bit planes (short strings, tau
// <= 4) that is only the side with the smaller threshold, and the matches
// whose first side passed (its distance in place of the left limit) wait in
// the second until 32 of them can have the other side verified: most matches
// fail on the first side, and lanes with nothing left to do would idle through
// the second side's wider band.
struct SecondQueue {
  uint32_t q[Q_SECOND], sid[Q_SECOND], pi[Q_SECOND], lim[Q_SECOND];
};
struct QueueWarp {
  uint32_t q[Q_CAP], sid[Q_CAP], pi[Q_CAP], lim[Q_CAP];
  SecondQueue second;
};

// First side of one match per lane (`in` lanes have one).  Matches without
// planes (lengths 0 in lim) are verified as a whole.  n2: the second queue's
// size, the same in every lane.
template <int MAXW, bool SELF, bool MULTI>
__device__ __forceinline__ void verify_first(const ProbeView& v, SecondQueue& w, bool in, uint32_t q, uint32_t r,
                                             uint32_t pi, uint32_t lim, int& n2, AccOut out, Counters* ctr,
                                             unsigned long long& cells) {
  bool pass = false;
  uint32_t d1 = 0;
  if (in) {
    if (MAXW <= 5 && v.pplanes && lim >> 16) {
      const ProbeView vt = MULTI ? view_for_tau(v, (int)(pi >> 24)) : v;
      const PlaneMatch m = plane_match(vt, q, r, pi, lim);
      const int tl = m.i - 1, tr = m.tau + 1 - m.i;
      unsigned c = 0;
      if (m.li <= SEG_EXACT_MAX || plane_segment(m)) {
        const bool right = tr < tl;
        d1 = (uint32_t)plane_side<(MAXW - 1) / 2>(m, right, c);
        pass = (int)d1 <= (right ? tr : tl);
      }
      cells += c;
    } else {
      verify_queued_entry<MAXW, SELF, MULTI>(v, q, r, pi, out, ctr, cells);
    }
  }
  if (MAXW <= 5) {
    __syncwarp();
    const unsigned b = __ballot_sync(FULL, pass);
    if (pass) {
      const int slot = n2 + __popc(b & lanemask_lt());
      w.q[slot] = q;
      w.sid[slot] = r;
      w.pi[slot] = pi;
      w.lim[slot] = (lim & ~0xFFu) | d1;
    }
    n2 += __popc(b);
    __syncwarp();
  }
}

// Second side of the second queue's last min(n2, 32) entries.
template <int MAXW, bool SELF, bool MULTI>
__device__ __forceinline__ void verify_second(const ProbeView& v, SecondQueue& w, int& n2, AccOut out, Counters* ctr,
                                              unsigned long long& cells) {
  const int lane = (int)(threadIdx.x & 31u);
  const int n = ::min(n2, 32);
  n2 -= n;
  const int e = n2 + (lane < n ? lane : 0);
  const uint32_t q = w.q[e], r = w.sid[e], pi = w.pi[e], lim = w.lim[e];
  __syncwarp();  // taken before any later write
  if (lane < n) {
    const ProbeView vt = MULTI ? view_for_tau(v, (int)(pi >> 24)) : v;
    const PlaneMatch m = plane_match(vt, q, r, pi, lim);
    const int tl = m.i - 1, tr = m.tau + 1 - m.i;
    const bool right = !(tr < tl);
    unsigned c = 0;
    const int d2 = plane_side<MAXW - 1>(m, right, c);
    cells += c;
    if (d2 <= (right ? tr : tl)) {
      const unsigned long long pos = atomicAdd(&ctr->accepted, 1ull);
      if (pos < out.cap) {
        out.key[pos] = match_key(v, SELF, q, r);
        out.ed[pos] = (lim & 0xFFu) + (uint32_t)d2;
      }
    }
  }
}

// A query batch (R != S) in two launches, with nothing but the long posting
// runs in between in device memory: k_query_fused does selection, lookups,
// screen and extension verification; runs longer than RUN_PART postings (the
// few-character segments of a large index have runs of tens of thousands) are
// set aside in parts, which k_query_tasks deals evenly to all warps.
//
// Against two probe passes, two scans, candidate offsets and the queued kernel
// this saves six launches, two host reads of sizes and the hit array; a lane
// computes its substring's key afresh where the passes roll it along the
// window.  Bound by the latency of dependent lookups at small batches and by
// the screen's issue slots at large ones.
constexpr uint32_t RUN_PART = 256;
constexpr int STEP_MOST = 512;       // candidates a warp walks itself in one step ...
constexpr uint32_t RUN_KEEP = 32;    // ... or else only its runs of at most so many
constexpr int WALK = 4;  // records a lane loads at once

struct WalkWarp {
  uint32_t q[32 * WALK + 32], sid[32 * WALK + 32], pi[32 * WALK + 32], lim[32 * WALK + 32];
  SecondQueue second;
};

// What a lane counts, and its warp's queue sizes (the same in every lane).
struct WalkState {
  unsigned long long cells, filtered;
  int err, qn, n2;
};

template <int MAXW, bool MULTI>
__device__ __forceinline__ void walk_verify(const ProbeView& v, WalkWarp& w, WalkState& st, int n, AccOut out,
                                            Counters* ctr) {
  const int lane = (int)(threadIdx.x & 31u);
  __syncwarp();
  st.qn -= n;
  const int e = st.qn + (lane < n ? lane : 0);
  verify_first<MAXW, false, MULTI>(v, w.second, lane < n, w.q[e], w.sid[e], w.pi[e], w.lim[e], st.n2, out, ctr,
                                   st.cells);
  if (MAXW <= 5 && st.n2 >= 32) verify_second<MAXW, false, MULTI>(v, w.second, st.n2, out, ctr, st.cells);
  __syncwarp();  // the entries were taken before the next write
}

// Screens one posting record per lane (`in` lanes have one) against hit; the
// survivors wait in the queue.
template <bool MULTI>
__device__ __forceinline__ void walk_screen(const ProbeView& v, WalkWarp& w, WalkState& st, bool in, const Hit& hit,
                                            const PostRec& rec) {
  const uint32_t r = rec_sid(rec);
  bool pass = false;
  if (in) {
    if (r >= v.n_index) {
      st.err |= 1;
    } else {
      if (v.hit_sides) {
        unsigned dl, dr;
        side_distances(hit.sides, rec.sides, dl, dr);
        pass = dl <= (hit.lim & 0xFFu) && dr <= (hit.lim >> 8 & 0xFFu);
      } else {
        pass = !(v.pbm && signature_bound(v.pbm[hit.q], v.ibm[r]) > (MULTI ? (int)(hit.pi >> 24) : v.tau));
      }
      st.filtered += !pass;
    }
  }
  __syncwarp();
  const unsigned b = __ballot_sync(FULL, pass);
  if (pass) {
    const int at = st.qn + __popc(b & lanemask_lt());
    w.q[at] = hit.q;
    w.sid[at] = r;
    w.pi[at] = hit.pi;
    w.lim[at] = hit.lim;
  }
  st.qn += __popc(b);
}

// The postings of one hit, by the whole warp; every lane has the same hit.
template <int MAXW, bool MULTI>
__device__ __forceinline__ void walk_run(const ProbeView& v, WalkWarp& w, WalkState& st, const Hit& hit, AccOut out,
                                         Counters* ctr) {
  const unsigned lane = threadIdx.x & 31u;
  const PostRec* precs = (MULTI ? v.parts[hit.pi >> 24].precs : v.precs) + hit.begin;
  for (uint32_t k0 = 0; k0 < hit.count; k0 += 32 * WALK) {
    PostRec rec[WALK];
#pragma unroll
    for (int j = 0; j < WALK; ++j) rec[j] = precs[min(k0 + 32u * j + lane, hit.count - 1)];
#pragma unroll
    for (int j = 0; j < WALK; ++j) {
      if (k0 + 32u * j >= hit.count) break;  // the same in every lane
      walk_screen<MULTI>(v, w, st, k0 + 32u * j + lane < hit.count, hit, rec[j]);
    }
    while (st.qn >= 32) walk_verify<MAXW, MULTI>(v, w, st, 32, out, ctr);
  }
}

// The postings of every lane's own hit (count 0: none), the runs laid end to
// end so that a step takes 32 postings whatever the runs' lengths.
template <int MAXW, bool MULTI>
__device__ __forceinline__ void walk_runs(const ProbeView& v, WalkWarp& w, WalkState& st, const Hit& mine, AccOut out,
                                          Counters* ctr) {
  const unsigned lane = threadIdx.x & 31u;
  const int incl = warp_incl_scan((int)mine.count);  // at most 32 * RUN_PART
  const int total = __shfl_sync(FULL, incl, 31);
  const uint32_t base = mine.begin + mine.count - (uint32_t)incl;  // posting of item f of this lane's run: base + f
  for (int f0 = 0; f0 < total; f0 += 32 * WALK) {
    PostRec rec[WALK];
    int src[WALK];
#pragma unroll
    for (int j = 0; j < WALK; ++j) {
      const int f = min(f0 + 32 * j + (int)lane, total - 1);
      src[j] = warp_owner(incl, f);
      const uint32_t at = __shfl_sync(FULL, base, src[j]) + (uint32_t)f;
      const PostRec* precs = v.precs;
      if (MULTI) precs = v.parts[__shfl_sync(FULL, mine.pi, src[j]) >> 24].precs;
      rec[j] = precs[at];
    }
#pragma unroll
    for (int j = 0; j < WALK; ++j) {
      if (f0 + 32 * j >= total) break;  // the same in every lane
      Hit hit;
      hit.begin = hit.count = 0;
      hit.q = __shfl_sync(FULL, mine.q, src[j]);
      hit.pi = __shfl_sync(FULL, mine.pi, src[j]);
      hit.lim = __shfl_sync(FULL, mine.lim, src[j]);
#pragma unroll
      for (int k = 0; k < 3; ++k) hit.sides.w[k] = __shfl_sync(FULL, mine.sides.w[k], src[j]);
      walk_screen<MULTI>(v, w, st, f0 + 32 * j + (int)lane < total, hit, rec[j]);
    }
    while (st.qn >= 32) walk_verify<MAXW, MULTI>(v, w, st, 32, out, ctr);
  }
}

// What is left in the queues, and the counters.
template <int MAXW, bool MULTI>
__device__ __forceinline__ void walk_end(const ProbeView& v, WalkWarp& w, WalkState& st, AccOut out, Counters* ctr) {
  __syncwarp();
  if (st.qn) walk_verify<MAXW, MULTI>(v, w, st, st.qn, out, ctr);
  if (MAXW <= 5) {
    while (st.n2) {
      verify_second<MAXW, false, MULTI>(v, w.second, st.n2, out, ctr, st.cells);
      __syncwarp();
    }
  }
  warp_add_counter(&ctr->cells, st.cells);
  warp_add_counter(&ctr->filtered, st.filtered);
  if (st.err) atomicOr(&ctr->err, (unsigned long long)st.err);
}

// A lane takes one window position of one (query, length, segment) group, W =
// tau + 1 lanes a group, up to 32 / W groups a step and one when there are too
// few groups to fill the warps; then the whole warp walks the runs that its
// lanes found.  n_dev: the group count, if only the device knows it.  tasks:
// room for task_cap parts of long runs (without room a run is walked here).
template <int MAXW, bool MULTI>
__global__ void __launch_bounds__(Q_BLOCK) k_query_fused(const ProbeView v, unsigned long long n_groups,
                                                         const unsigned long long* __restrict__ n_dev,
                                                         Hit* __restrict__ tasks, unsigned long long task_cap,
                                                         AccOut out, Counters* ctr) {
  __shared__ WalkWarp queues[Q_WARPS];
  n_groups = dev_count(n_groups, n_dev);
  const unsigned lane = threadIdx.x & 31u;
  WalkWarp& w = queues[threadIdx.x >> 5];
  const unsigned long long warp = ((unsigned long long)blockIdx.x * Q_BLOCK + threadIdx.x) >> 5;
  const unsigned long long n_warps = ((unsigned long long)gridDim.x * Q_BLOCK) >> 5;
  const unsigned W = (unsigned)v.tau + 1;  // the largest window
  const unsigned most = W >= 32 ? 1u : 32u / W;
  const unsigned long long rounds = max(1ull, (n_groups + n_warps * most - 1) / (n_warps * most));
  const unsigned per =  // as many as make the rounds even, rather than a last one for a few warps
      (unsigned)min((unsigned long long)most, max(1ull, (n_groups + n_warps * rounds - 1) / (n_warps * rounds)));
  unsigned long long lookups = 0, cand = 0, n_hits = 0;
  WalkState st{0ull, 0ull, 0, 0, 0};
  for (unsigned long long t0 = warp * per; t0 < n_groups; t0 += n_warps * per) {
    for (unsigned s0 = 0; s0 < per * W; s0 += 32) {
      const unsigned slot = s0 + lane;
      const unsigned long long t = t0 + slot / W;
      Hit mine{0u, 0u, 0u, 0u, {{0u, 0u, 0u}}, 0u};
      if (slot < per * W && t < n_groups) {
        uint32_t q;
        int g;
        if (MULTI) {
          uint32_t lo = 0, hi = v.pcount;  // last q with qgoff[q] <= t
          while (hi - lo > 1) {
            const uint32_t mid = lo + ((hi - lo) >> 1);
            if (v.qgoff[mid] <= t) lo = mid; else hi = mid;
          }
          q = lo;
          g = (int)(t - v.qgoff[q]);
        } else {
          const unsigned G = (unsigned)groups_per_probe(v.tau, false);
          q = (uint32_t)(t / G);
          g = (int)(t - (unsigned long long)q * G);
        }
        const ProbeView vt = MULTI ? view_for_tau(v, v.ptau[q]) : v;
        const int ls = (int)vt.plen[q];
        int l, i, P, li, lo, hi;
        if (group_window(vt, false, q, ls, g, l, i, P, li, lo, hi) && lo + (int)(slot % W) <= hi) {
          const int p = lo + (int)(slot % W);
          const uint8_t* s = vt.pbytes + vt.poff[q];
          ++lookups;
          uint32_t b;
          const uint32_t c = lookup_key(vt, false, q, ls, l, seg_key(s + p, li, l, i), b, st.err);
          if (c) {
            mine = Hit{q, b, c, (uint32_t)p | (uint32_t)i << 16 | (MULTI ? (uint32_t)vt.tau << 24 : 0u),
                       {{0u, 0u, 0u}}, 0u};
            if (vt.hit_sides) {
              mine.sides = side_pair(side_signature(s, p), side_signature(s + p + li, ls - p - li));
              mine.lim = hit_limits(vt.tau, i, ls, l, p, P, li);
            }
            cand += c;
            ++n_hits;
          }
        }
      }
      __syncwarp();
      // runs to set aside: the long ones, and in a step of many candidates all
      // but the shortest, in parts that the whole step reserves at once
      const int here = warp_sum(mine.count <= RUN_PART ? (int)mine.count : 0);  // the same in every lane
      const uint32_t cut = task_cap && here > STEP_MOST ? RUN_KEEP : RUN_PART;
      const bool aside = mine.count > cut;
      if (__any_sync(FULL, aside)) {
        const unsigned long long parts = aside ? (mine.count + (unsigned long long)RUN_PART - 1) / RUN_PART : 0ull;
        const unsigned long long incl = warp_incl_scan(parts);
        const unsigned long long all = __shfl_sync(FULL, incl, 31);
        unsigned long long at = task_cap;
        if (lane == 0 && task_cap) at = atomicAdd(&ctr->tasks, all);
        at = __shfl_sync(FULL, at, 0);
        const bool room = at + all <= task_cap;  // the same in every lane
        if (parts == 1 && at + incl - 1 < task_cap) {
          Hit part = mine;
          if (!room) part.count = 0u;  // empty where not all parts have room
          tasks[at + incl - 1] = part;
        }
        if (parts == 1 && room) mine.count = 0;
        for (unsigned found = __ballot_sync(FULL, parts > 1); found; found &= found - 1) {  // long runs
          const int src = __ffs((int)found) - 1;
          Hit hit;
          hit.q = __shfl_sync(FULL, mine.q, src);
          hit.begin = __shfl_sync(FULL, mine.begin, src);
          hit.count = __shfl_sync(FULL, mine.count, src);
          hit.pi = __shfl_sync(FULL, mine.pi, src);
          hit.lim = __shfl_sync(FULL, mine.lim, src);
#pragma unroll
          for (int k = 0; k < 3; ++k) hit.sides.w[k] = __shfl_sync(FULL, mine.sides.w[k], src);
          if ((int)lane == src) mine.count = 0;
          const unsigned long long np = __shfl_sync(FULL, parts, src);
          const unsigned long long first = at + __shfl_sync(FULL, incl, src) - np;
          for (unsigned long long k = lane; k < np && first + k < task_cap; k += 32) {
            Hit part = hit;
            part.begin = hit.begin + (uint32_t)k * RUN_PART;
            part.count = room ? min(RUN_PART, hit.count - (uint32_t)k * RUN_PART) : 0u;
            tasks[first + k] = part;
          }
          __syncwarp();
          if (!room) walk_run<MAXW, MULTI>(v, w, st, hit, out, ctr);
        }
      }
      walk_runs<MAXW, MULTI>(v, w, st, mine, out, ctr);
    }
  }
  walk_end<MAXW, MULTI>(v, w, st, out, ctr);
  warp_add_counter(&ctr->lookups, lookups);
  warp_add_counter(&ctr->candidates, cand);
  warp_add_counter(&ctr->hits, n_hits);
}

// The parts that k_query_fused set aside, a warp a part.
template <int MAXW, bool MULTI>
__global__ void __launch_bounds__(Q_BLOCK) k_query_tasks(const ProbeView v, const Hit* __restrict__ tasks,
                                                         unsigned long long task_cap, AccOut out, Counters* ctr) {
  __shared__ WalkWarp queues[Q_WARPS];
  WalkWarp& w = queues[threadIdx.x >> 5];
  const unsigned long long n = min(task_cap, ctr->tasks);
  const unsigned long long warp = ((unsigned long long)blockIdx.x * Q_BLOCK + threadIdx.x) >> 5;
  const unsigned long long n_warps = ((unsigned long long)gridDim.x * Q_BLOCK) >> 5;
  if (warp >= n) return;  // the whole warp
  WalkState st{0ull, 0ull, 0, 0, 0};
  for (unsigned long long t = warp; t < n; t += n_warps) {
    const Hit hit = tasks[t];
    if (hit.count) walk_run<MAXW, MULTI>(v, w, st, hit, out, ctr);
  }
  walk_end<MAXW, MULTI>(v, w, st, out, ctr);
}

}  // namespace pj
