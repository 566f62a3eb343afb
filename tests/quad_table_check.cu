// Host harness of test_quad_table_check.py (no device code runs): builds the quadratic
// tables of a few bases, checks that they pass, then corrupts one entry of each kind and
// checks that validate_quad rejects it; and compares the quadratic forms with the pool's
// records in double.  Prints one line per case: "<name> ok" or "<name> FAIL".
#include <cmath>
#include <cstdio>
#include <functional>
#include <random>
#include <string>
#include <vector>

#include "apip_internal.h"
#include "gaunt_layout.h"

using namespace apip;

static void report(const std::string& name, bool pass) { std::printf("%s %s\n", name.c_str(), pass ? "ok" : "FAIL"); }

int main() {
  const int bases[][2] = {{1, 0}, {1, 4}, {3, 2}, {5, 3}, {7, 3}, {8, 4}};
  std::string err;
  for (const auto& b : bases) {
    const int64_t nb = basis_size(b[0], b[1], 4);
    std::mt19937_64 gen(5);
    auto u = [&] { return 2.0 * (double)gen() / 18446744073709551616.0 - 1.0; };
    std::vector<double> c1(nb), c2(nb);
    for (int64_t k = 0; k < nb; ++k) { c1[k] = (double)(float)u(); c2[k] = (double)(float)u(); }
    HostQuad h;
    HostAce p;
    const std::string tag = std::to_string(b[0]) + std::to_string(b[1]);
    const bool built = build_quad(b[0], b[1], c1.data(), c2.data(), nb, &h, &err) &&
                       build_coupled(b[0], b[1], 4, c1.data(), c2.data(), nb, &p, &err);
    report("valid_" + tag, built && validate_quad(h, &err));
    // phi_1 = sum 1/2 X S1 X, phi_2 = sum X K2 X and the records' phi, all in double
    const int nlm = (b[1] + 1) * (b[1] + 1);
    std::vector<double> X(p.npool, 1.0), ga(kGaunt4Total);
    gaunt4_fill(ga.data());
    for (int c = 0; c < p.nA; ++c) X[1 + c] = u();
    for (int c = 0; c < p.nC; ++c) {
      const uint32_t k = p.comp[2 * c], g0 = p.comp[2 * c + 1] >> 8, g1 = g0 + (p.comp[2 * c + 1] & 255u);
      double s = 0;
      for (uint32_t e = g0; e < g1; ++e) s += p.gval[e] * X[(k & 0xffffu) + (p.gkey[e] & 255u)] * X[(k >> 16) + (p.gkey[e] >> 8)];
      X[1 + p.nA + c] = s;
    }
    double ref[2] = {0, 0}, mag = 0, got[2] = {0, 0};
    for (size_t r = 0; r < p.fkey.size(); ++r) {
      double d = 0;
      for (uint32_t m = 0; m < p.flen[r]; ++m) d += X[(p.fkey[r] & 0xffffu) + m] * X[(p.fkey[r] >> 16) + m];
      ref[0] += p.f1[r] * d;
      ref[1] += p.f2[r] * d;
      mag += std::fabs(d);
    }
    for (int L = 0; L <= 2 * b[1]; ++L) {
      const int nc = h.hdr[4 * L], na = h.hdr[4 * L + 1], nM = 2 * L + 1;
      std::vector<double> x((size_t)(nc + na + 1) * nM, 1.0);
      for (int l1 = 0; l1 <= b[1]; ++l1)
        for (int l2 = l1; l2 <= b[1]; ++l2)
          for (int n = 0; n < b[0] * b[0]; ++n) {
            const int n1 = n / b[0], n2 = n % b[0];
            const int row = h.map[(size_t)L * kQuadMap + ((l1 * (kLmaxCap + 1) + l2) * kNmaxCap + n1) * kNmaxCap + n2];
            if (row < 0 || (l1 == l2 && n1 > n2)) continue;
            for (int M = 0; M < nM; ++M) x[(size_t)row * nM + M] = 0.0;
            int g = gaunt4_offset(l1, l2, L);
            for (int i = 0; i < 2 * l1 + 1; ++i)
              for (int j = 0; j < 2 * l2 + 1; ++j)
                for (int c = 0; c < 2; ++c) {
                  const int M = gaunt_cand(i - l1, j - l2, c, L);
                  if (M != kNoM)
                    x[(size_t)row * nM + M + L] += ga[g++] * X[1 + n1 * nlm + l1 * l1 + i] * X[1 + n2 * nlm + l2 * l2 + j];
                }
          }
      for (int n = 0; n < na; ++n)
        for (int M = 0; M < nM; ++M) x[(size_t)(nc + n) * nM + M] = X[1 + n * nlm + L * L + M];
      for (int t = h.hdr[4 * L + 2]; t < h.hdr[4 * L + 2] + h.hdr[4 * L + 3]; ++t)
        for (int pass = 0; pass < 2; ++pass) {
          const int *tl = h.tile.data() + 8 * t, unit = pass ? 4 : 2;
          for (int k = 0; k < tl[4 * pass + 2]; ++k) {
            const int st = k / unit, w0 = k % unit * (16 / unit);
            const int col = h.col[tl[4 * pass + 1] + st * kQuadBundle * unit + k % unit] / (nM * kQuadAtoms);
            for (int r = 0; r < tl[7]; ++r) {
              const int w = w0 + (pass ? r : 2 * r);
              const double v = h.val[4 * (size_t)(tl[4 * pass] + (st * 4 + w / 4) * kQuadBundle) + w % 4];
              for (int M = 0; M < nM; ++M)
                got[pass] += (pass ? 1.0 : 0.5) * v * x[(size_t)(tl[3] + r) * nM + M] * x[(size_t)col * nM + M];
            }
          }
        }
    }
    // coefficients are floats here, so only double rounding is left
    report("forms_" + tag, std::fabs(got[0] - ref[0]) <= 1e-12 * mag && std::fabs(got[1] - ref[1]) <= 1e-12 * mag);
    if (b[0] != 5) continue;
    auto bad = [&](const char* name, const std::function<void(HostQuad&)>& f) {
      HostQuad x = h;
      f(x);
      report(name, !validate_quad(x, &err));
    };
    bad("degree_rows", [](HostQuad& x) { x.hdr[4 * 6] = x.rows; });
    bad("degree_tiles", [](HostQuad& x) { x.hdr[4 * 6 + 3] += 1; });
    bad("row_map", [](HostQuad& x) { x.map[(size_t)2 * kQuadMap] = (short)x.hdr[4 * 2]; });
    bad("row_map_negative", [](HostQuad& x) { x.map[0] = -2; });
    bad("tile_first_row", [](HostQuad& x) { x.tile[3] = x.hdr[0] + x.hdr[1] + 1; });
    bad("tile_rows", [](HostQuad& x) { x.tile[7] = kQuadTile + 1; });
    bad("tile_values", [](HostQuad& x) { x.tile[x.tile.size() - 8] = (int)(x.val.size() / 4); });
    bad("tile_columns", [](HostQuad& x) { x.tile[x.tile.size() - 7] = (int)x.col.size(); });
    bad("tile_length", [](HostQuad& x) { x.tile[2] = (int)x.col.size() / kQuadBundle * 2; });
    bad("tile_alignment", [](HostQuad& x) { x.tile[2] += 1; });
    bad("column_past_rows", [](HostQuad& x) { x.col[0] = (uint32_t)((x.hdr[0] + x.hdr[1] + 1) * kQuadAtoms); });
    bad("column_between_rows", [](HostQuad& x) { x.col[0] += 1; });
    bad("end_of_values", [](HostQuad& x) { x.val.resize(x.val.size() - 16 * kQuadBundle); });
    bad("end_of_columns", [](HostQuad& x) { x.col.resize(x.col.size() - 4 * kQuadBundle); });
  }
  return 0;
}
