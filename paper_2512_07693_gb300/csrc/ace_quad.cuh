// ACE evaluation for large bases of body order 4 in float32 (the quadratic kernel).  A block takes
// 8 compacted atoms at a time.  For one degree L, the couplings
//   C_{(p q) L M} = sum G(l_p m1, l_q m2, L M) A_{p m1} A_{q m2},
// the segments A_{n L} and, for L = 0, the constant 1 are the rows of X_L (one value
// per M and atom), and all basis functions of that degree are entries of matrices
// shared by all atoms (build_quad):
//   phi_c = sum_L 1/2 X_L . (S_L^c X_L),   dE/dX_L = S_L^1 X_L + F'(phi_2) S_L^2 X_L.
//  1. A (ace_device.cuh);
//  2. for every L: X_L from A (unrolled per (l1, l2, L)), then phi_2 += X_L . (K2_L X_L),
//     which gives F'(phi_2);
//  3. for every L: X_L again, S_L^1 X_L and S_L^2 X_L in packed float pairs, phi_1,
//     dE/dX_L, and that back onto A, each thread owning one segment A_{n l} of an atom;
//  4. pair forces (ace_device.cuh).
// No atomics, so the sums have a fixed order.  The sum over a row's columns is plain, in
// an order that puts the columns expected to be large last (build_quad); the rows'
// contributions to phi are compensated per thread, and the block adds them up in
// float-float.  In a restatement of the sums on the densities of cracked, void, vacancy
// and bulk crystals (bases 4/4 to 8/4) the RMS error of phi against 64 bits is 0.42 to
// 0.85 of the record-wise kernel's, which compensates per record; with the columns by
// index and plain sums over rows and block it was 1.3 and 1.4 times as large (8/4, a
// crack's faces).  Compensating within a row (every 16 or 32 columns) cost half and a
// third more time for nothing beyond that.
//
// What bounds it: the matrix products, 3.47 M multiply-adds per atom for n_max 8, l_max 4
// (2.95 M on entries that are not zero), one barrier after another: a degree's items do
// not fill the rounds of 384 threads evenly, and the warps wait at the barriers for 4.1 of
// some 8 cycles per issued instruction (FMA pipe 31 %, L1 42 %, L2 4 % busy, a crack of
// 126 k atoms).  The record-wise pool kernel (ace_pool.cuh) reads its 16-byte records,
// 5 MB forward and 20 MB back, once per group of 1 to 4 atoms through L2; here 2.1 MB of
// values serve 8 atoms.  A thread's tile is 4 rows (both channels) by the 8 atoms of one
// M: 32 packed multiply-adds for two uniform 16-byte loads of values and two of X from
// shared memory (8 rows by 4 atoms: four and one, which took 15 % longer).  8 atoms are
// what X_L and dE/dX_L of the largest degree leave room for (2 x 89 KB); step 2 before
// step 3 instead of both channels' dE/dX_L kept apart costs a fifth more multiply-adds
// and saves twice that space.  Prefetching the values into L1 one to six steps ahead
// changed nothing.
#pragma once

#include "ace_device.cuh"
#include "gaunt_layout.h"
#include "pair2.cuh"

namespace apip {

// Dynamic shared memory: X_L and dE/dX_L (step 1 stages R, Y there), A, dE/dA and the
// per-warp sums (high and low parts).
template <int LMAX>
__host__ __device__ inline size_t ace_quad_smem(int nA, int rows) {
  const int xy = 2 * rows * kQuadAtoms, ry = (ry_elems<LMAX, kQuadThreads>() + 3) / 4 * 4;
  return sizeof(float) * (size_t)((xy > ry ? xy : ry) + 2 * nA * kQuadAtoms + 2 * (kQuadThreads / 32) * kQuadAtoms);
}

// X_L and dE/dX_L: value M (of NM) of a row for atom k.  Four atoms lie together, so that
// the lanes of a warp, on consecutive M, read consecutive 16 bytes.
template <int NM>
__device__ __forceinline__ int quad_at(int row, int M, int k) {
  return (row * 2 + (k >> 2)) * (NM * 4) + M * 4 + (k & 3);
}

// Rows C_{(n1 L1)(n2 L2) LL} of X: four (n1, n2) and the 8 atoms per warp, chunk by chunk.
template <typename K, int L1, int L2, int LL>
__device__ __forceinline__ void quad_form(const float* A, float* X, const short* map, int n_max, int nlm, int chunk) {
  constexpr int N1 = 2 * L1 + 1, N2 = 2 * L2 + 1, NM = 2 * LL + 1, G0 = gaunt4_offset(L1, L2, LL);
  const int lane = threadIdx.x & 31, k = lane & 7, q = 4 * chunk + (lane >> 3);
  const int n1 = q / n_max, n2 = q - n1 * n_max;
  if (n1 >= n_max || (L1 == L2 && n1 > n2)) return;
  const int row = map[((L1 * (kLmaxCap + 1) + L2) * kNmaxCap + n1) * kNmaxCap + n2];
  if (row < 0) return;
  float x1[N1], x2[N2], C[NM];
#pragma unroll
  for (int i = 0; i < N1; ++i) x1[i] = A[(n1 * nlm + L1 * L1 + i) * kQuadAtoms + k];
#pragma unroll
  for (int j = 0; j < N2; ++j) x2[j] = A[(n2 * nlm + L2 * L2 + j) * kQuadAtoms + k];
#pragma unroll
  for (int M = 0; M < NM; ++M) C[M] = 0.f;
  int e = G0;
#pragma unroll
  for (int i = 0; i < N1; ++i)
#pragma unroll
    for (int j = 0; j < N2; ++j)
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const int M = gaunt_cand(i - L1, j - L2, v, LL);
        if (M != kNoM) {
          C[M + LL] += K::gaunt(e) * x1[i] * x2[j];
          ++e;
        }
      }
#pragma unroll
  for (int M = 0; M < NM; ++M) X[quad_at<NM>(row, M, k)] = C[M];
}

// The part of dE/dA_{(n l)} (l = LT) that comes through its couplings of degree LL with
// the segments of degree LO: g[i] += sum over the partners n' of G dE/dC A_{(n' LO)}.
template <typename K, int LT, int LO, int LL>
__device__ __forceinline__ void quad_back(const float* A, const float* Y, const short* map, int n, int n_max, int nlm,
                                          float (&g)[2 * LT + 1]) {
  constexpr int L1 = LT < LO ? LT : LO, L2 = LT < LO ? LO : LT;
  constexpr int NO = 2 * LO + 1, NM = 2 * LL + 1, G0 = gaunt4_offset(L1, L2, LL);
  const int k = threadIdx.x & 7;
  const short* m = map + (LT * (kLmaxCap + 1) + LO) * kNmaxCap * kNmaxCap + n * kNmaxCap;
#pragma unroll 1
  for (int o = 0; o < n_max; ++o) {
    const int row = m[o];
    if (row < 0) continue;
    const float two = (LT == LO && o == n) ? 2.f : 1.f;   // both factors are this segment
    float x[NO], y[NM];
#pragma unroll
    for (int j = 0; j < NO; ++j) x[j] = two * A[(o * nlm + LO * LO + j) * kQuadAtoms + k];
#pragma unroll
    for (int M = 0; M < NM; ++M) y[M] = Y[quad_at<NM>(row, M, k)];
    int e = G0;
#pragma unroll
    for (int i1 = 0; i1 < 2 * L1 + 1; ++i1)
#pragma unroll
      for (int i2 = 0; i2 < 2 * L2 + 1; ++i2)
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const int M = gaunt_cand(i1 - L1, i2 - L2, v, LL);
          if (M != kNoM) {
            const int i = LT < LO ? i1 : i2, j = LT < LO ? i2 : i1;
            g[i] += K::gaunt(e) * y[M + LL] * x[j];
            ++e;
          }
        }
  }
}

// acc[r][j] += value(r) . X(column, atom j) over the columns of a tile; F2 rows are the
// two channels of one row of S (NP = 4) or two rows of K2 (NP = 2).  Xq: the thread's M
// in the first row, its last four atoms half further.  The values of the next step (2
// or 4 columns) and their columns are loaded while these are used.
template <int NP>
__device__ __forceinline__ void quad_tile(const ulonglong2* val, const uint32_t* col, int len, const float* Xq, int half,
                                          F2 (&acc)[NP][kQuadAtoms]) {
  constexpr int U = 8 / NP;   // columns per step (64 bytes of values)
  ulonglong2 vn[4];
  uint32_t cn[U];
  auto fetch = [&](int st) {
#pragma unroll
    for (int q = 0; q < 4; ++q) vn[q] = __ldg(val + (size_t)(st * 4 + q) * kQuadBundle);
    if constexpr (U == 2) {
      const uint2 c = __ldg(reinterpret_cast<const uint2*>(col + (size_t)st * kQuadBundle * U));
      cn[0] = c.x; cn[1] = c.y;
    } else {
      const uint4 c = __ldg(reinterpret_cast<const uint4*>(col + (size_t)st * kQuadBundle * U));
      cn[0] = c.x; cn[1] = c.y; cn[2] = c.z; cn[3] = c.w;
    }
  };
  fetch(0);
#pragma unroll 1
  for (int st = 0; st < len / U; ++st) {
    ulonglong2 v[4];
    uint32_t c[U];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = vn[q];
#pragma unroll
    for (int u = 0; u < U; ++u) c[u] = cn[u];
    fetch(st + 1);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float4 x = *reinterpret_cast<const float4*>(Xq + c[u]), y = *reinterpret_cast<const float4*>(Xq + c[u] + half);
      const F2 xd[kQuadAtoms] = {f2(x.x), f2(x.y), f2(x.z), f2(x.w), f2(y.x), f2(y.y), f2(y.z), f2(y.w)};
#pragma unroll
      for (int r = 0; r < NP; ++r) {
        const ulonglong2 w = v[(u * NP + r) / 2];
        const F2 a{(r & 1) ? w.y : w.x};
#pragma unroll
        for (int j = 0; j < kQuadAtoms; ++j) acc[r][j] = fma2(a, xd[j], acc[r][j]);
      }
    }
  }
}

// X_L of the block's atoms (the caller's barrier follows).
template <typename K, int LMAX>
__device__ __forceinline__ void quad_rows(const AceDev<float>& t, int L, const float* A, float* X) {
  constexpr int NLM = (LMAX + 1) * (LMAX + 1), NW = kQuadThreads / 32;
  const int warp = threadIdx.x >> 5, n_max = t.n_max;
  const short* map = t.qmap + L * kQuadMap;
  const int chunks = (n_max * n_max + 3) / 4;
  int w = warp;   // the next work item of this warp, counted from the current type
#define APIP_FORM(l1, l2, LL)                                                                                  \
  if constexpr (l2 <= LMAX) {                                                                                  \
    for (; w < chunks; w += NW) quad_form<K, l1, l2, LL>(A, X, map, n_max, NLM, w);                            \
    w -= chunks;                                                                                               \
  }
  switch (L) {
    case 0: { APIP_GAUNT4_L0(APIP_FORM) } break;
    case 1: { APIP_GAUNT4_L1(APIP_FORM) } break;
    case 2: { APIP_GAUNT4_L2(APIP_FORM) } break;
    case 3: { APIP_GAUNT4_L3(APIP_FORM) } break;
    case 4: { APIP_GAUNT4_L4(APIP_FORM) } break;
    case 5: { APIP_GAUNT4_L5(APIP_FORM) } break;
    case 6: { APIP_GAUNT4_L6(APIP_FORM) } break;
    case 7: { APIP_GAUNT4_L7(APIP_FORM) } break;
    default: { APIP_GAUNT4_L8(APIP_FORM) } break;
  }
#undef APIP_FORM
  const int4 h = __ldg(t.qhdr + L);
  const int len = (2 * L + 1) * kQuadAtoms;
  for (int q = threadIdx.x; q < h.y * len; q += kQuadThreads) {
    const int n = q / len, M = (q - n * len) / kQuadAtoms, k = q % kQuadAtoms;
    X[((h.x + n) * 2 + (k >> 2)) * (len / 2) + M * 4 + (k & 3)] = A[(n * NLM + L * L + M) * kQuadAtoms + k];
  }
  if (L == 0 && threadIdx.x < kQuadAtoms) X[(h.x + h.y) * kQuadAtoms + threadIdx.x] = 1.f;
}

// dE/dA += what dE/dX_L (Y) gives, one segment (n, l) and atom per thread: a warp takes
// four n of one l, so that it runs one unrolled body at a time.
template <typename K, int LMAX>
__device__ __forceinline__ void quad_onto_a(const AceDev<float>& t, int L, const float* A, const float* Y, float* W) {
  constexpr int NLM = (LMAX + 1) * (LMAX + 1), NW = kQuadThreads / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, k = lane & 7, n_max = t.n_max;
  const short* map = t.qmap + L * kQuadMap;
  const int4 h = __ldg(t.qhdr + L);
  const int per_l = (n_max + 3) / 4;
  // the largest degrees have the most partners: they start first
  for (int u = warp; u < per_l * (LMAX + 1); u += NW) {
    const int l = LMAX - u / per_l, n = (u % per_l) * 4 + (lane >> 3);
    if (n >= n_max) continue;
    auto add = [&](auto lt) {
      constexpr int LT = decltype(lt)::value;
      float g[2 * LT + 1];
#pragma unroll
      for (int i = 0; i < 2 * LT + 1; ++i) g[i] = 0.f;
#define APIP_BACK(l1, l2, LL)                                                                         \
  if constexpr (l2 <= LMAX && l1 == LT) quad_back<K, LT, l2, LL>(A, Y, map, n, n_max, NLM, g);          \
  if constexpr (l2 <= LMAX && l2 == LT && l1 != l2) quad_back<K, LT, l1, LL>(A, Y, map, n, n_max, NLM, g);
      switch (L) {
        case 0: { APIP_GAUNT4_L0(APIP_BACK) } break;
        case 1: { APIP_GAUNT4_L1(APIP_BACK) } break;
        case 2: { APIP_GAUNT4_L2(APIP_BACK) } break;
        case 3: { APIP_GAUNT4_L3(APIP_BACK) } break;
        case 4: { APIP_GAUNT4_L4(APIP_BACK) } break;
        case 5: { APIP_GAUNT4_L5(APIP_BACK) } break;
        case 6: { APIP_GAUNT4_L6(APIP_BACK) } break;
        case 7: { APIP_GAUNT4_L7(APIP_BACK) } break;
        default: { APIP_GAUNT4_L8(APIP_BACK) } break;
      }
#undef APIP_BACK
      const bool direct = L == LT && n < h.y;   // the segment's own row of X_L
#pragma unroll
      for (int i = 0; i < 2 * LT + 1; ++i) {
        float v = W[(n * NLM + LT * LT + i) * kQuadAtoms + k] + g[i];
        if (direct) v += Y[quad_at<2 * LT + 1>(h.x + n, i, k)];
        W[(n * NLM + LT * LT + i) * kQuadAtoms + k] = v;
      }
    };
    if (l == 0) add(std::integral_constant<int, 0>{});
    if constexpr (LMAX >= 1) { if (l == 1) add(std::integral_constant<int, 1>{}); }
    if constexpr (LMAX >= 2) { if (l == 2) add(std::integral_constant<int, 2>{}); }
    if constexpr (LMAX >= 3) { if (l == 3) add(std::integral_constant<int, 3>{}); }
    if constexpr (LMAX >= 4) { if (l == 4) add(std::integral_constant<int, 4>{}); }
  }
}

// Sums of f (pairs of atoms) over the block per atom, with what the compensated sums
// still have to give back, in red[0 .. 7] after the barrier.  Each exchange within a warp
// halves the atoms that a lane keeps (9 float-float additions; 40 with all 8 on every
// lane).
__device__ __forceinline__ void quad_sum(const Acc2 (&f)[kQuadAtoms / 2], float* red) {
  constexpr int NW = kQuadThreads / 32;
  static_assert(kQuadAtoms == 8 && NW % 4 == 0, "three halvings; a quarter of the warps per lane");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  auto other = [](FF v, int o) { return FF{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)}; };
  FF v[kQuadAtoms];
#pragma unroll
  for (int j = 0; j < kQuadAtoms; ++j) {
    const float2 s = f2_get(f[j / 2].s), n = f2_get(f[j / 2].n);
    v[j] = (j & 1) ? FF{s.y, n.y} : FF{s.x, n.x};
  }
#pragma unroll
  for (int o = 16, keep = 4; keep > 0; o >>= 1, keep >>= 1)
#pragma unroll
    for (int j = 0; j < keep; ++j) {
      const bool up = (lane & o) != 0;
      const FF mine = up ? v[j + keep] : v[j];
      v[j] = ff_add(mine, other(up ? v[j] : v[j + keep], o));
    }
#pragma unroll
  for (int o = 2; o > 0; o >>= 1) v[0] = ff_add(v[0], other(v[0], o));
  if ((lane & 3) == 0) {   // lane 4 a: atom a
    red[warp * kQuadAtoms + lane / 4] = v[0].hi;
    red[(NW + warp) * kQuadAtoms + lane / 4] = v[0].lo;
  }
  __syncthreads();
  FF t{0.f, 0.f};
  if (warp == 0) {
    for (int w = lane / kQuadAtoms; w < NW; w += 32 / kQuadAtoms)
      t = ff_add(t, FF{red[w * kQuadAtoms + lane % kQuadAtoms], red[(NW + w) * kQuadAtoms + lane % kQuadAtoms]});
#pragma unroll
    for (int o = kQuadAtoms; o < 32; o <<= 1) t = ff_add(t, other(t, o));
  }
  __syncthreads();
  if (tid < kQuadAtoms) red[tid] = t.hi + t.lo;
  __syncthreads();
}

template <typename K, int LMAX>
__global__ void __launch_bounds__(kQuadThreads, 1) k_ace_quad(Args<float> a, AceDev<float> t) {
  pdl_begin();
  // every list-build kernel of this call has completed: block 0 clears the
  // trigger (and, after a build, the binning counts) for the next step
  if (blockIdx.x == 0) end_list_build(a.flags, a.cell_count, a.ncell);
  constexpr int NAT = kQuadAtoms, NT = kQuadThreads;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ AceGroup<float, NAT> g;
  const int tid = threadIdx.x, nA = t.nA;
  float* A = reinterpret_cast<float*>(smem_raw);   // A[c * 8 + k], then omega
  float* W = A + nA * NAT;                         // dE/dA
  float* red = W + nA * NAT;
  float* X = red + 2 * (NT / 32) * NAT;                  // X_L, then dE/dX_L (step 1 stages R, Y there)
  float* Y = X + t.qrows * NAT;
  const int count = a.counts[0];
  const int ngroups = count > t.split ? (count + NAT - 1) / NAT : 0;   // (else the pool kernel's)
  double e_part = 0.0;

  for (int grp = blockIdx.x; grp < ngroups; grp += gridDim.x) {
    group_setup<float, NAT>(a, grp, count, g);
    refine_switch<float, NAT, NT>(a, g);
    for (int c = tid; c < nA * NAT; c += NT) { A[c] = 0.f; W[c] = 0.f; }
    __syncthreads();
    densities<float, K, LMAX, NAT, NT>(a, t, g, A, X);

    // 2. phi_2 and F'(phi_2)
    {
      Acc2 f[NAT / 2];
      for (int L = 0; L <= 2 * LMAX; ++L) {
        const int4 h = __ldg(t.qhdr + L);
        quad_rows<K, LMAX>(t, L, A, X);
        __syncthreads();
        const int nm = 2 * L + 1, half = 4 * nm;
        for (int it = tid; it < h.w * nm; it += NT) {
          const int tl = it / nm, M = it - tl * nm;
          const int4 rb = __ldg(t.qtile + 2 * (h.z + tl)), ra = __ldg(t.qtile + 2 * (h.z + tl) + 1);
          if (ra.z == 0) continue;
          F2 acc[2][NAT];
#pragma unroll
          for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int j = 0; j < NAT; ++j) acc[r][j] = f2(0.f);
          quad_tile<2>(t.qval + ra.x, t.qcol + ra.y, ra.z, X + 4 * M, half, acc);
#pragma unroll
          for (int r = 0; r < kQuadTile; ++r) {
            if (r < ra.w) {
              const float* xp = X + (rb.w + r) * 2 * half + 4 * M;
#pragma unroll
              for (int b = 0; b < 2; ++b) {
                const float4 x = *reinterpret_cast<const float4*>(xp + b * half);
                float z[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  const float2 u = f2_get(acc[r / 2][4 * b + j]);
                  z[j] = (r & 1) ? u.y : u.x;
                }
                f[2 * b].add_prod(f2(x.x, x.y), f2(z[0], z[1]));
                f[2 * b + 1].add_prod(f2(x.z, x.w), f2(z[2], z[3]));
              }
            }
          }
        }
        __syncthreads();
      }
      quad_sum(f, red);
    }
    if (tid < NAT) {
      const float p2 = red[tid], q2 = sqrt(p2 * p2 + t.eps * t.eps);
      g.dfs[tid] = 0.5f * p2 / (q2 * sqrt(q2));
      g.e[tid] = p2;
    }
    __syncthreads();

    // 3. phi_1 and the adjoint
    {
      Acc2 f[NAT / 2];   // of 2 phi_1
      for (int L = 0; L <= 2 * LMAX; ++L) {
        const int4 h = __ldg(t.qhdr + L);
        quad_rows<K, LMAX>(t, L, A, X);   // (dE/dX of the degree before is read only from Y)
        __syncthreads();
        const int nm = 2 * L + 1, half = 4 * nm;
        for (int it = tid; it < h.w * nm; it += NT) {
          const int tl = it / nm, M = it - tl * nm;
          const int4 rb = __ldg(t.qtile + 2 * (h.z + tl));
          const int nr = __ldg(reinterpret_cast<const int*>(t.qtile + 2 * (h.z + tl) + 1) + 3);
          F2 acc[kQuadTile][NAT];
#pragma unroll
          for (int r = 0; r < kQuadTile; ++r)
#pragma unroll
            for (int j = 0; j < NAT; ++j) acc[r][j] = f2(0.f);
          quad_tile<kQuadTile>(t.qval + rb.x, t.qcol + rb.y, rb.z, X + 4 * M, half, acc);
#pragma unroll
          for (int r = 0; r < kQuadTile; ++r) {
            if (r < nr) {
              const int o = (rb.w + r) * 2 * half + 4 * M;
#pragma unroll
              for (int b = 0; b < 2; ++b) {
                const float4 x = *reinterpret_cast<const float4*>(X + o + b * half);
                float z[4], y[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  const float2 u = f2_get(acc[r][4 * b + j]);
                  z[j] = u.x;
                  y[j] = u.x + g.dfs[4 * b + j] * u.y;
                }
                f[2 * b].add_prod(f2(x.x, x.y), f2(z[0], z[1]));
                f[2 * b + 1].add_prod(f2(x.z, x.w), f2(z[2], z[3]));
                *reinterpret_cast<float4*>(Y + o + b * half) = make_float4(y[0], y[1], y[2], y[3]);
              }
            }
          }
        }
        __syncthreads();
        quad_onto_a<K, LMAX>(t, L, A, Y, W);
      }
      quad_sum(f, red);
    }
    if (tid < NAT) atom_scalars<float, NAT>(a, t, tid, 0.5f * red[tid], g.e[tid], g);
    __syncthreads();
    for (int item = tid; item < nA * NAT; item += NT)
      W[item] *= t.a_scale * (a.force_mix ? 1.f : g.lam[item % NAT]);
    __syncthreads();
    e_part += pair_forces<float, K, LMAX, NAT, NT>(a, t, g, W);
  }
  block_energy<float, NAT>(a, g, e_part);
}

// launch, or occupancy query (resident blocks per SM, 0 if it does not fit)
template <typename K, int LMAX>
int quad_l(const Args<float>* a, const AceDev<float>& t, int blocks, cudaStream_t s, bool query) {
  const size_t bytes = ace_quad_smem<LMAX>(t.nA, t.qrows);
  if (query) return resident_blocks(k_ace_quad<K, LMAX>, kQuadThreads, bytes);
  launch_pdl(k_ace_quad<K, LMAX>, blocks, kQuadThreads, bytes, s, *a, t);
  return 0;
}

template <typename K>
int quad_dispatch(const Args<float>* a, const AceDev<float>& t, int blocks, cudaStream_t s, bool query) {
  switch (t.l_max) {
    case 0: return quad_l<K, 0>(a, t, blocks, s, query);
    case 1: return quad_l<K, 1>(a, t, blocks, s, query);
    case 2: return quad_l<K, 2>(a, t, blocks, s, query);
    case 3: return quad_l<K, 3>(a, t, blocks, s, query);
    default: return quad_l<K, 4>(a, t, blocks, s, query);
  }
}

}  // namespace apip
