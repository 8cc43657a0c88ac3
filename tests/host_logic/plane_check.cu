// The bit-plane verification against the plain DP, on the host: sides of
// every length up to PLANE_LEN - 1 and every threshold 0..4, cut out of longer
// strings at random places, over alphabets whose characters differ in 1 to 8
// bits, with characters that the planes' bits do not cover (marked), and the
// segment comparison.  Also the side limits of a hit against side_distances.
#include <cstdio>
#include <random>
#include <string>
#include <vector>

#include "pj_probe.cuh"

static int ed(const std::string& a, const std::string& b) {
  std::vector<int> p(b.size() + 1), c(b.size() + 1);
  for (size_t j = 0; j <= b.size(); ++j) p[j] = (int)j;
  for (size_t i = 1; i <= a.size(); ++i) {
    c[0] = (int)i;
    for (size_t j = 1; j <= b.size(); ++j)
      c[j] = std::min(std::min(p[j] + 1, c[j - 1] + 1), p[j - 1] + (a[i - 1] != b[j - 1] ? 1 : 0));
    std::swap(p, c);
  }
  return p[b.size()];
}

static pj::ByteBits bits_of(const std::string& alphabet) {
  pj::ByteBits b{255u, 0u};
  for (unsigned char c : alphabet) {
    b.andd &= c;
    b.orr |= c;
  }
  return b;
}

int main() {
  std::mt19937 g(11);
  std::vector<std::string> alphabets = {"ab", "aq", "abcdefghijklmnopqrstuvwxyz ", "ACGT", std::string("\0\x80\x40\xff", 4)};
  std::string all;
  for (int c = 0; c < 256; ++c) all += (char)c;
  alphabets.push_back(all);
  long bad = 0, within = 0, sides = 0;
  for (const std::string& A : alphabets) {
    const pj::ByteBits bb = bits_of(A);
    for (int it = 0; it < 60000; ++it) {
      // whole strings: left side, segment, right side
      const int tau = 4, i = 1 + (int)(g() % 5), li = 1 + (int)(g() % 6);
      const int room = pj::PLANE_LEN - li;
      const int P = (int)(g() % (room + 1)), tail = (int)(g() % (room - P + 1));
      auto draw = [&](int n) {
        std::string s;
        for (int k = 0; k < n; ++k) s += A[g() % A.size()];
        return s;
      };
      std::string yl = draw(P), seg = draw(li), yr = draw(tail), xl = yl, xr = yr;
      for (std::string* s : {&xl, &xr})  // edits
        for (int e = (int)(g() % 6); e > 0; --e) {
          const unsigned kind = g() % 3;
          const size_t at = s->empty() ? 0 : g() % s->size();
          if (kind == 0) s->insert(at, 1, g() % 8 ? A[g() % A.size()] : (char)(g() & 255));
          else if (kind == 1 && !s->empty()) s->erase(at, 1);
          else if (!s->empty()) (*s)[at] = g() % 8 ? A[g() % A.size()] : (char)(g() & 255);
        }
      if ((int)(xl.size() + li + xr.size()) > pj::PLANE_LEN) continue;
      const bool same_seg = g() % 4 != 0;
      std::string xseg = seg;
      if (!same_seg) xseg[g() % li] = (char)(g() & 255);
      const std::string x = xl + xseg + xr, y = yl + seg + yr;
      pj::PlaneMatch m;
      const pj::Planes px = pj::string_planes((const uint8_t*)x.data(), (int)x.size(), bb);
      const pj::Planes py = pj::string_planes((const uint8_t*)y.data(), (int)y.size(), bb);
      for (int b = 0; b < 8; ++b) {
        m.X[b] = px.w[b];
        m.Y[b] = py.w[b];
      }
      m.ls = (int)x.size();
      m.lr = (int)y.size();
      m.p = (int)xl.size();
      m.P = P;
      m.li = li;
      m.tau = tau;
      m.i = i;
      m.wide = pj::planes_used(bb, false) > 6;
      if (pj::plane_segment(m) != (xseg == seg)) ++bad;
      unsigned dl = 0, dr = 0;
      const uint32_t lim = pj::hit_limits(tau, i, m.ls, m.lr, m.p, P, li);
      pj::side_distances(
          pj::side_pair(pj::side_signature((const uint8_t*)xl.data(), (int)xl.size()),
                        pj::side_signature((const uint8_t*)xr.data(), (int)xr.size())),
          pj::side_pair(pj::side_signature((const uint8_t*)yl.data(), (int)yl.size()),
                        pj::side_signature((const uint8_t*)yr.data(), (int)yr.size())), dl, dr);
      for (int right = 0; right < 2; ++right) {
        const int t = right ? tau + 1 - i : i - 1;
        const int want = std::min(t + 1, right ? ed(xr, yr) : ed(xl, yl));
        unsigned cells = 0;
        const int got = std::min(t + 1, pj::plane_side<4>(m, right != 0, cells));
        ++sides;
        if (got != want) {
          if (bad < 5) printf("t=%d got %d want %d\n", t, got, want);
          ++bad;
        }
        if (want <= t) {
          ++within;
          if ((right ? dr : dl) > (right ? lim >> 8 & 255u : lim & 255u)) ++bad;  // the screen dropped a similar side
        }
      }
    }
  }
  printf("bad=%ld within=%ld sides=%ld\n", bad, within, sides);
  return 0;
}
