// Host-side check of the sub-walks that the row gather's lanes follow
// (tests/test_walk_split_cpu.py).
//
// Reads a mesh as tests/walk_replay.cu does, encodes every row's walk, cuts it
// with the library's split_walk into 1, 2, 4 and 8 sub-walks and replays each
// sub-walk as a lane runs it: segments of two filling bytes (with the element
// count) and one byte per element, the next node read before the leaving one
// is written back, M = -c_c carried, a plane of accumulators per sub-walk.
// The planes' sums must equal direct sums over the star, the bytes must stay
// within the row's and every slot within the row's off-diagonal entries.
#include "../paper_2111_05651_gb300/csrc/nsi_create.cu"

namespace nsi {
int gather_kernel_regs(int) { return 64; }
}  // namespace nsi

using nsi::V3;
using D3 = V3<double>;

int main(int argc, char** argv) {
  FILE* fp = argc < 2 ? nullptr : std::fopen(argv[1], "rb");
  if (!fp) return 2;
  int64_t n = 0, E = 0;
  if (std::fread(&n, 8, 1, fp) != 1 || std::fread(&E, 8, 1, fp) != 1) return 2;
  std::vector<D3> X(n), U(n);
  std::vector<int32_t> ln(4 * E);
  if (std::fread(X.data(), 24, n, fp) != (size_t)n || std::fread(ln.data(), 4, 4 * E, fp) != (size_t)(4 * E) ||
      std::fread(U.data(), 24, n, fp) != (size_t)n)
    return 2;
  std::fclose(fp);
  std::vector<std::vector<std::pair<int64_t, int>>> inc(n);
  for (int64_t e = 0; e < E; ++e)
    for (int a = 0; a < 4; ++a) inc[ln[4 * e + a]].push_back({e, a});
  static const int EVEN[4][3] = {{1, 2, 3}, {0, 3, 2}, {3, 0, 1}, {2, 1, 0}};
  const double kmu = 1e-3;
  double worst = 0.0;
  long long elems = 0, longest = 0;
  nsi::WalkWork ws;
  auto fail = [](int64_t i, int nsub, const char* what) {
    std::printf("FAIL row %lld, %d sub-walks: %s\n", (long long)i, nsub, what);
    return 1;
  };
  for (int64_t i = 0; i < n; ++i) {
    std::vector<int32_t> col;
    for (auto& ea : inc[i])
      for (int a = 0; a < 4; ++a) col.push_back(ln[4 * ea.first + a]);
    std::sort(col.begin(), col.end());
    col.erase(std::unique(col.begin(), col.end()), col.end());
    if (col.empty()) continue;
    auto pos = [&](int32_t j) { return (int)(std::lower_bound(col.begin(), col.end(), j) - col.begin()); };
    const int dp = pos((int32_t)i), ns = (int)col.size() - 1;
    std::vector<uint16_t> tri;
    for (auto& ea : inc[i]) {
      unsigned w = 0;
      for (int m = 0; m < 3; ++m) w |= unsigned(pos(ln[4 * ea.first + EVEN[ea.second][m]])) << (5 * m);
      tri.push_back((uint16_t)w);
    }
    std::vector<uint8_t> steps;
    if (!nsi::encode_walk(tri.data(), (int)tri.size(), dp, steps, ws)) return fail(i, 0, "not encoded");
    auto node = [&](int slot) { return col[slot + (slot >= dp)]; };
    std::vector<double> A(ns, 0.0), Gx(ns, 0.0);
    double D = 0.0, sa = 0.0, sg = 0.0;
    for (uint16_t w : tri) {
      int sl[3];
      D3 d[3], us{2 * U[i].x, 2 * U[i].y, 2 * U[i].z};
      for (int b = 0; b < 3; ++b) {
        const int p = (w >> (5 * b)) & 31;
        sl[b] = p - (p > dp);
        d[b] = sub(X[col[p]], X[i]);
        us = add(us, U[col[p]]);
      }
      const D3 c[3] = {cross(d[1], d[2]), cross(d[2], d[0]), cross(d[0], d[1])};
      const double det = dot(d[0], c[0]);
      const D3 ci{-(c[0].x + c[1].x + c[2].x), -(c[0].y + c[1].y + c[2].y), -(c[0].z + c[1].z + c[2].z)};
      const double kv = kmu / det;
      sg = std::max(sg, std::sqrt(dot(ci, ci)));
      const D3 w3{us.x + kv * ci.x, us.y + kv * ci.y, us.z + kv * ci.z};
      for (int b = 0; b < 3; ++b) {
        A[sl[b]] += dot(w3, c[b]);
        Gx[sl[b]] += ci.x;
      }
      D += det;
    }
    for (int s = 0; s < ns; ++s) sa = std::max(sa, std::fabs(A[s]));
    for (int nsub : {1, 2, 4, 8}) {
      std::vector<uint8_t> b;
      if (!nsi::split_walk(steps.data(), (int)steps.size(), dp, nsub, b)) return fail(i, nsub, "not split");
      longest = std::max(longest, (long long)b.size());
      std::vector<double> rA(ns, 0.0), rG(ns, 0.0);
      double rD = 0.0;
      int count = 0;
      size_t at = nsub;
      for (int k = 0; k < nsub; ++k) {
        const size_t end = at + b[k];
        if (end > b.size()) return fail(i, nsub, "bytes past the row");
        struct Node {
          int k;
          D3 d, v;
          double a, g;
        };
        std::vector<double> pA(ns, 0.0), pG(ns, 0.0);
        std::vector<int> held(ns, 0);
        bool bad = false;
        auto load = [&](unsigned w) {
          const int s = (int)(w & nsi::WALK_POS);
          if (s >= ns || held[s]) {
            bad = true;
            return Node{};
          }
          ++held[s];
          return Node{s, sub(X[node(s)], X[i]), U[node(s)], pA[s], pG[s]};
        };
        auto store = [&](const Node& nd) {
          --held[nd.k];
          pA[nd.k] = nd.a;
          pG[nd.k] = nd.g;
        };
        while (at < end && !bad) {
          const int cnt = (b[at] >> 5) | ((b[at + 1] >> 5) << 3);
          if (cnt < 1 || at + 2 + cnt > end) return fail(i, nsub, "segment past its sub-walk");
          Node p = load(b[at]), q = load(b[at + 1]), c = load(b[at + 2]);
          D3 M = cross(q.d, p.d);
          for (int s = 0; s < cnt && !bad; ++s) {
            const unsigned w = b[at + 2 + s];
            Node nx{};
            if (s + 1 < cnt) nx = load(b[at + 3 + s]);
            const bool neg = w & nsi::WALK_NEG, evq = w & nsi::WALK_EVQ;
            const double f = neg ? -1.0 : 1.0;
            const D3 cp = cross(q.d, c.d), cq = cross(c.d, p.d);
            const double det = dot(p.d, cp), kv = kmu / det;
            const D3 ci{M.x - cp.x - cq.x, M.y - cp.y - cq.y, M.z - cp.z - cq.z};
            const D3 w3{2 * U[i].x + p.v.x + q.v.x + c.v.x + kv * ci.x, 2 * U[i].y + p.v.y + q.v.y + c.v.y + kv * ci.y,
                        2 * U[i].z + p.v.z + q.v.z + c.v.z + kv * ci.z};
            p.a += f * dot(w3, cp);
            q.a += f * dot(w3, cq);
            c.a -= f * dot(w3, M);
            p.g += f * ci.x;
            q.g += f * ci.x;
            c.g += f * ci.x;
            rD += f * det;
            ++count;
            if (evq) {
              store(q);
              M = cq;
            } else {
              store(p);
              p = q;
              M = D3{-cp.x, -cp.y, -cp.z};
            }
            q = c;
            c = nx;
          }
          if (bad) break;
          store(p);
          store(q);
          at += 2 + cnt;
        }
        if (bad) return fail(i, nsub, "a slot outside the row or still held");
        if (at != end) return fail(i, nsub, "sub-walk length");
        for (int s = 0; s < ns; ++s) rA[s] += pA[s], rG[s] += pG[s];
      }
      if (at != b.size() || count != (int)tri.size()) return fail(i, nsub, "elements walked");
      elems += count;
      for (int s = 0; s < ns; ++s)
        worst = std::max({worst, std::fabs(rA[s] - A[s]) / sa, std::fabs(rG[s] - Gx[s]) / sg});
      worst = std::max(worst, std::fabs(rD - D) / D);
    }
  }
  std::printf("elements=%lld longest=%lld worst=%.3g\n", elems, longest, worst);
  return worst <= 1e-12 ? 0 : 1;
}
