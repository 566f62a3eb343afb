// Host harness of test_quad_sums.py (no device code runs).  For each density vector A of
// a file it evaluates phi_1, phi_2 of a seeded basis from the library's own tables: in
// long double, in float as the record-wise kernel adds them (per-thread compensated
// sums over the records, a plain sum over the block), and in float as the quadratic
// kernel does (plain over a row's columns in table order, compensated over the rows,
// exact over the block), the last also with the columns by their index.  Prints one line
// per vector: the errors of the records, of the quadratic form, of the columns by index.
#include <algorithm>
#include <array>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <string>
#include <vector>

#include "apip_internal.h"
#include "gaunt_layout.h"

using namespace apip;

struct Kahan {   // s - c is the sum
  volatile float s = 0.f, c = 0.f;
  void take(float y) { const volatile float t = s + y, d = t - s; c = d - y; s = t; }   // y = value - c
};

int main(int, char** v) {
  const int nm = std::atoi(v[1]), lm = std::atoi(v[2]), nlm = (lm + 1) * (lm + 1);
  const int64_t nb = basis_size(nm, lm, 4);
  std::mt19937_64 gen(2);
  std::vector<double> c1(nb), c2(nb);
  for (int64_t k = 0; k < nb; ++k)
    for (auto* c : {&c1, &c2}) (*c)[k] = 0.2 * ((double)gen() / 18446744073709551616.0 - 0.5);
  HostAce h;
  HostQuad q;
  std::string err;
  std::vector<double> ga(kGaunt4Total);
  gaunt4_fill(ga.data());
  if (!build_coupled(nm, lm, 4, c1.data(), c2.data(), nb, &h, &err) || !build_quad(nm, lm, c1.data(), c2.data(), nb, &q, &err))
    return 1;
  std::FILE* f = std::fopen(v[3], "rb");
  std::vector<float> A(h.nA);
  while (f && std::fread(A.data(), 4, A.size(), f) == A.size()) {
    std::vector<long double> X(h.npool, 1.0L);
    std::vector<float> x(h.npool, 1.f);
    for (int c = 0; c < h.nA; ++c) X[1 + c] = x[1 + c] = A[c];
    for (int c = 0; c < h.nC; ++c) {
      const uint32_t k = h.comp[2 * c], g0 = h.comp[2 * c + 1] >> 8, g1 = g0 + (h.comp[2 * c + 1] & 255u);
      long double S = 0;
      float s = 0.f;
      for (uint32_t e = g0; e < g1; ++e) {
        const uint32_t i = (k & 0xffffu) + (h.gkey[e] & 255u), j = (k >> 16) + (h.gkey[e] >> 8);
        S += h.gval[e] * X[i] * X[j];
        s = std::fmaf((float)h.gval[e] * x[i], x[j], s);
      }
      X[1 + h.nA + c] = S;
      x[1 + h.nA + c] = s;
    }
    long double phi[2] = {0, 0};
    std::vector<Kahan> rec[2] = {std::vector<Kahan>(kAceThreads), std::vector<Kahan>(kAceThreads)};
    for (size_t r = 0; r < h.fkey.size(); ++r) {
      long double D = 0;
      float d = 0.f;
      for (uint32_t m = 0; m < h.flen[r]; ++m) {
        const uint32_t i = (h.fkey[r] & 0xffffu) + m, j = (h.fkey[r] >> 16) + m;
        D += X[i] * X[j];
        d = std::fmaf(x[i], x[j], d);
      }
      phi[0] += h.f1[r] * D;
      phi[1] += h.f2[r] * D;
      Kahan &a = rec[0][r % kAceThreads], &b = rec[1][r % kAceThreads];
      a.take((float)h.f1[r] * d - a.c);
      b.take((float)h.f2[r] * d - b.c);
    }
    double e[6];
    for (int ch = 0; ch < 2; ++ch) {
      float s = 0.f;
      for (int w = 0; w < kAceThreads; w += 32) {   // the warps' shuffles, then their sums
        std::vector<float> t(32), u(32);
        for (int l = 0; l < 32; ++l) t[l] = rec[ch][w + l].s;
        for (int o = 16; o; o >>= 1, t = u)
          for (int l = 0; l < 32; ++l) u[l] = t[l] + t[l ^ o];
        s += t[0];
      }
      e[ch] = (double)(s - phi[ch]);
    }
    std::vector<Kahan> sum[2][2];   // [columns by index][channel]
    for (auto& o : sum)
      for (auto& c : o) c.resize(kQuadThreads);
    for (int L = 0; L <= 2 * lm; ++L) {
      const int nc = q.hdr[4 * L], na = q.hdr[4 * L + 1], nM = 2 * L + 1;
      std::vector<float> y((size_t)(nc + na + 1) * nM, 1.f);
      for (int l1 = 0; l1 <= lm; ++l1)
        for (int l2 = l1; l2 <= lm; ++l2)
          for (int n = 0; n < nm * nm; ++n) {
            const int n1 = n / nm, n2 = n % nm;
            const int row = q.map[(size_t)L * kQuadMap + ((l1 * (kLmaxCap + 1) + l2) * kNmaxCap + n1) * kNmaxCap + n2];
            if (row < 0 || (l1 == l2 && n1 > n2)) continue;
            for (int M = 0; M < nM; ++M) y[(size_t)row * nM + M] = 0.f;
            int g = gaunt4_offset(l1, l2, L);
            for (int i = 0; i < 2 * l1 + 1; ++i)
              for (int j = 0; j < 2 * l2 + 1; ++j)
                for (int c = 0; c < 2; ++c) {
                  const int M = gaunt_cand(i - l1, j - l2, c, L);
                  if (M == kNoM) continue;
                  float& t = y[(size_t)row * nM + M + L];
                  t = std::fmaf((float)ga[g++] * A[n1 * nlm + l1 * l1 + i], A[n2 * nlm + l2 * l2 + j], t);
                }
          }
      for (int n = 0; n < na; ++n)
        for (int M = 0; M < nM; ++M) y[(size_t)(nc + n) * nM + M] = A[n * nlm + L * L + M];
      for (int it = 0; it < q.hdr[4 * L + 3] * nM; ++it)
        for (int pass = 0; pass < 2; ++pass) {
          const int M = it % nM, *t = q.tile.data() + 8 * (q.hdr[4 * L + 2] + it / nM), unit = pass ? 4 : 2;
          std::vector<std::array<int, 2>> col;   // (row of X, place in the list)
          for (int k = 0; k < t[4 * pass + 2]; ++k)
            col.push_back({(int)q.col[t[4 * pass + 1] + k / unit * kQuadBundle * unit + k % unit] / (nM * kQuadAtoms), k});
          for (int by_index = 0; by_index < 2; ++by_index) {
            if (by_index) std::sort(col.begin(), col.end());
            float z[kQuadTile] = {};
            for (const auto& c : col)
              for (int r = 0; r < kQuadTile; ++r) {
                const int st = c[1] / unit, w = c[1] % unit * (16 / unit) + (pass ? r : 2 * r);
                z[r] = std::fmaf(q.val[4 * (size_t)(t[4 * pass] + (st * 4 + w / 4) * kQuadBundle) + w % 4],
                                 y[(size_t)c[0] * nM + M], z[r]);
              }
            Kahan& a = sum[by_index][pass][it % kQuadThreads];
            for (int r = 0; r < t[7]; ++r) a.take(std::fmaf(y[(size_t)(t[3] + r) * nM + M], z[r], -a.c));
          }
        }
    }
    for (int k = 0; k < 4; ++k) {
      double s = 0;
      for (const Kahan& a : sum[k / 2][k % 2]) s += (double)a.s - (double)a.c;
      e[2 + k] = (double)((float)(k % 2 == 0 ? 0.5 * s : s) - phi[k % 2]);
    }
    std::printf("%.9g %.9g %.9g %.9g %.9g %.9g\n", e[0], e[1], e[2], e[3], e[4], e[5]);
  }
  return 0;
}
