// All-atom passes of the adaptive-precision force pipeline: position
// preparation, the cell-binned neighbour list, the one-off CSP pair detection,
// pass 1 (EAM density and CSP^list g), pass 2 (switch, unweighted EAM force and
// stream compaction of lam > 0), the CSP part of the grad-lambda force, the
// float64 reductions and the velocity-Verlet kernels.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "kernels.h"
#include "pair2.cuh"

namespace apip {

namespace {

__device__ __forceinline__ double wrap1(double x, double L, double invL) {
  double w = x - L * floor(x * invL);
  if (w >= L) w -= L;
  if (w < 0.0) w += L;
  return w;
}

// The rare branch of wrap_near, kept out of line so that the compiler cannot
// turn it into predicated float64 instructions issued for every atom.
__device__ __noinline__ double wrap1_slow(double x, double L, double invL) { return wrap1(x, L, invL); }

// wrap1 for a position that is normally already in [0, L) (the drift of one
// step): the range test is made on the bit patterns (non-negative doubles order
// as integers), which keeps it off the float64 pipe.
__device__ __forceinline__ double wrap_near(double x, double L, double invL) {
  const long long b = __double_as_longlong(x), bl = __double_as_longlong(L);
  if (b >= 0 && b < bl) return x;
  return wrap1_slow(x, L, invL);
}

// isfinite from the exponent bits.
__device__ __forceinline__ bool finite_bits(double x) {
  return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;
}

__device__ __forceinline__ int cell_of(double xw, double L, int nc) {
  int c = (int)(xw * ((double)nc / L));
  return c < 0 ? 0 : (c >= nc ? nc - 1 : c);
}

// Duties shared by k_prep and the drift of the Verlet kernels for atom i at
// position (x, y, z): finiteness and id checks, the id -> index map, the
// fixed-point coordinates (FP32 path) and the neighbour-list trigger
// (displacement since the last build > skin / 2).  In the FP32 path the
// displacement is taken from the fixed-point coordinates (integer differences),
// which keeps float64 arithmetic out of this per-atom work; ``wrapped`` says that
// (x, y, z) already lie in [0, L).
template <typename T>
__device__ __forceinline__ float prep_atom(const Args<T>& a, int i, double x, double y, double z,
                                           bool wrapped = false) {
  if (!finite_bits(x) || !finite_bits(y) || !finite_bits(z)) atomicOr(&a.status[ST_BAD_INPUT], 1);
  const int idv = a.id[i];
  if (idv < 0 || idv >= a.nmax) atomicOr(&a.status[ST_BAD_INPUT], 1);
  else a.id2idx[idv] = i;
  if (sizeof(T) == 4) {
    const double xs[3] = {x, y, z};
    unsigned int q[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
      q[k] = fixed_coord(wrapped ? xs[k] : wrap1(xs[k], a.geo.L[k], a.geo.invL[k]), a.geo.unit_m[k], a.geo.unit_s[k]);
    a.posq[i] = make_uint4(q[0], q[1], q[2], 0u);
    const uint4 r = a.posq_ref[i];
    const float ex = (float)(int)(q[0] - r.x) * a.geo.unit[0], ey = (float)(int)(q[1] - r.y) * a.geo.unit[1],
                ez = (float)(int)(q[2] - r.z) * a.geo.unit[2];
    const float e2 = ex * ex + ey * ey + ez * ez;
    if (e2 > a.skin_half2_f) atomicOr(&a.flags[0], 1);
    return e2;
  }
  double dx = x - a.pos_ref[3 * i], dy = y - a.pos_ref[3 * i + 1], dz = z - a.pos_ref[3 * i + 2];
  dx -= a.geo.L[0] * rint(dx * a.geo.invL[0]);
  dy -= a.geo.L[1] * rint(dy * a.geo.invL[1]);
  dz -= a.geo.L[2] * rint(dz * a.geo.invL[2]);
  if (dx * dx + dy * dy + dz * dz > a.skin_half2) atomicOr(&a.flags[0], 1);
  return 0.f;
}

// FP32 path: the block's largest squared displacement since the list build into
// the running maximum flags[1] (float bits; non-negative floats order as
// integers), one atomic per block.  Called by every thread of the block.
template <typename T>
__device__ __forceinline__ void note_displacement(const Args<T>& a, float e2) {
  if constexpr (sizeof(T) == 4) {
    __shared__ int wmax[kBlock / 32];
    const int m = __reduce_max_sync(0xffffffffu, __float_as_int(e2));
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
      int b = wmax[0];
      for (int w = 1; w < (int)(blockDim.x >> 5); ++w) b = max(b, wmax[w]);
      atomicMax(&a.flags[1], b);
    }
  }
}

template <typename T>
__global__ void k_prep(Args<T> a) {
  pdl_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) a.counts[0] = a.counts[1] = 0;
  float e2 = 0.f;
  if (i < a.n) e2 = prep_atom(a, i, a.pos[3 * i], a.pos[3 * i + 1], a.pos[3 * i + 2]);
  note_displacement(a, e2);
}

// ------------------------------------------------------------ neighbour list
// Two launches per list build (binning, fill), each returning at once when no
// build is due: cell_count is zero before a build (zeroed on allocation, and after
// each build by end_list_build, which also clears the trigger).

// The cell of atom i and what its candidates are tested against.  FP32 path: from
// the fixed-point coordinates (integer arithmetic, floor(q nc / 2^32); rel: the exact
// fraction within the cell).  FP64 path: from the wrapped position; rel is the float
// position relative to the cell's lower corner.  w: the cell's edges.
template <typename T>
__device__ __forceinline__ void atom_in_cell(const Args<T>& a, int i, int c[3], float rel[3], float w[3]) {
  if constexpr (sizeof(T) == 4) {
    const uint4 q = a.posq[i];
    const unsigned qq[3] = {q.x, q.y, q.z};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const unsigned long long x = (unsigned long long)qq[k] * (unsigned)a.geo.nc[k];
      c[k] = (int)(x >> 32);
      w[k] = a.geo.csf[k];
      rel[k] = (float)(unsigned)x * (w[k] * 0x1p-32f);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double x = wrap1(a.pos[3 * i + k], a.geo.L[k], a.geo.invL[k]);
      c[k] = cell_of(x, a.geo.L[k], a.geo.nc[k]);
      w[k] = a.geo.csf[k];
      rel[k] = (float)(x - (double)c[k] * a.geo.cs[k]);
    }
  }
}

// Binning: each atom takes a slot of its cell (the order of the slots follows
// the atomics, so neighbour order within a cell is not fixed and every sum over
// neighbours is order-independent up to rounding, unless the deterministic mode
// sorts the cells).  The member's record is all that the fill's distance test needs:
// FP32 path its fixed-point position, FP64 path its float position relative to the
// cell's corner; the index rides in .w.
template <typename T>
__global__ void k_bin(Args<T> a) {
  pdl_begin();
  if (!a.flags[0]) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  int c[3];
  float rel[3], w[3];
  atom_in_cell(a, i, c, rel, w);
  const int cell = (c[2] * a.geo.nc[1] + c[1]) * a.geo.nc[0] + c[0];
  const int slot = atomicAdd(&a.cell_count[cell], 1);
  if (slot < a.cell_cap) {
    uint4 rec;
    if constexpr (sizeof(T) == 4) rec = a.posq[i];
    else rec = make_uint4(__float_as_uint(rel[0]), __float_as_uint(rel[1]), __float_as_uint(rel[2]), 0u);
    rec.w = (unsigned)i;
    a.cell_q[(size_t)cell * a.cell_cap + slot] = rec;
  } else {
    atomicOr(&a.status[ST_CELL_OVERFLOW], 1);
    atomicMax(&a.status[ST_MAX_CELL], slot + 1);
  }
}

// Deterministic mode, on a build: each cell's members sorted by atom index (one
// thread per cell, insertion sort: a cell holds a few atoms), so that the list's
// order, and with it every sum over neighbours, does not depend on the order of
// the binning atomics.
template <typename T>
__global__ void k_cell_sort(Args<T> a) {
  pdl_begin();
  if (!a.flags[0]) return;
  const int cell = blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= a.ncell) return;
  const int m = min(a.cell_count[cell], a.cell_cap);
  uint4* v = a.cell_q + (size_t)cell * a.cell_cap;
  for (int k = 1; k < m; ++k) {
    const uint4 x = v[k];
    int p = k;
    for (; p > 0 && v[p - 1].w > x.w; --p) v[p] = v[p - 1];
    v[p] = x;
  }
}

// The list of atom i: every atom within r_list, in three classes of the build
// distance (0 within the EAM cutoff, 1 within the EAM cutoff + skin, 2 beyond), each
// in cell order.  The passes' EAM sums stop at nnb_e (classes 0 and 1: a pair now
// within the EAM cutoff was within cutoff + skin at the build, since each atom has
// moved less than skin / 2), and the class order keeps the lanes of a warp on the
// same branch of those sums.
//
// What bounds it: the instructions per candidate (the 27 cells hold 6 times the
// atoms of the sphere), the float64 pipe in the FP64 path, and, in a small system,
// the length of one thread's scan.
//  - LANES = 4 or 8 threads share an atom where there are too few atoms to fill the
//    GPU (atom_lanes): they test LANES members of a cell at a time, take their
//    places in the scratch column from a ballot, and class the ~60 kept entries in a
//    second round (2 k atoms: 102 -> 27 us; four 2 k-atom label calls, whole pass
//    1357 -> 1050 us).
//  - FP64 path: the scan tests float positions relative to the cell (the bound is
//    2e-5 wider than r_list, far above their rounding); only the kept entries see
//    float64 arithmetic (249 k atoms: 3870 -> 650 us per build).
//  - FP32 path, one thread per atom: k_nbfill_one below.
constexpr unsigned kClassShift = 30;   // n_atoms_max <= 2^30: two bits are free above an index
template <typename T>
__device__ __forceinline__ int build_class(const Args<T>& a, T r2) {
  if constexpr (sizeof(T) == 4) {
    // against r_list^2 rounded up: the list holds every pair whose float distance is
    // below r_list (and perhaps a few at r_list)
    return r2 < a.r_e_in2f ? 0 : (r2 < a.r_e_mid2f ? 1 : (r2 < a.r_list2f ? 2 : 3));
  } else {
    return r2 < a.r_e_in2 ? 0 : (r2 < a.r_e_mid2 ? 1 : (r2 < a.r_list2 ? 2 : 3));
  }
}

template <typename T, int LANES>
__global__ void __launch_bounds__(kBlock) k_nbfill(Args<T> a) {
  pdl_begin();
  if (!a.flags[0]) return;
  // the new list's reference positions are the current ones: no displacement yet
  if (blockIdx.x == 0 && threadIdx.x == 0) a.flags[1] = 0;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const bool own = t / LANES < a.n;
  if (LANES == 1 && !own) return;
  const int i = own ? t / LANES : a.n - 1;   // (LANES > 1: the warp stays whole for its ballots)
  const int g = LANES == 1 ? 0 : (int)(threadIdx.x % LANES);
  const unsigned gshift = LANES == 1 ? 0u : (threadIdx.x & 31u) / LANES * LANES;
  constexpr unsigned gmask = LANES >= 32 ? 0xffffffffu : (1u << LANES) - 1u;
  const unsigned below = (1u << g) - 1u;
  int c[3];
  float rel[3], w[3];
  atom_in_cell(a, i, c, rel, w);
  const auto si = a.pv.self(i);
  int n0 = 0, n1 = 0, n2 = 0;   // class counts
  T min1 = T(INFINITY);         // least squared distance in class 1
  int k0, k1, k2;               // entries kept of each class: the first max_nb in class order
  // a cell whose nearest face is beyond the bound holds no candidate (1e-5 covers the
  // rounding of the gaps; with three or more cells per axis no member of a neighbour
  // cell is within r_list through the other side of the box)
  const float lim = sizeof(T) == 4 ? a.r_list2f : a.r_scan2f, prune2 = lim * 1.00001f;
  float lo2[3], hi2[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    lo2[k] = rel[k] * rel[k];
    hi2[k] = (w[k] - rel[k]) * (w[k] - rel[k]);
  }
  int* tmp = a.nbl_tmp + i;
  int m = 0;            // indices kept by the scan (beyond max_nb: counted, not written)
  auto gap = [&](int k, int d) { return d < 0 ? lo2[k] : (d > 0 ? hi2[k] : 0.f); };
  for (int dz = -1; dz <= 1; ++dz) {
    const int cz = (c[2] + dz + a.geo.nc[2]) % a.geo.nc[2];
    for (int dy = -1; dy <= 1; ++dy) {
      const int cy = (c[1] + dy + a.geo.nc[1]) % a.geo.nc[1];
      const float gzy = gap(2, dz) + gap(1, dy);
      for (int dx = -1; dx <= 1; ++dx) {
        const bool skip = gzy + gap(0, dx) > prune2;
        if (LANES == 1 && skip) continue;
        const int cx = (c[0] + dx + a.geo.nc[0]) % a.geo.nc[0];
        const int cell = APIP_CHK(a.status, BND_CELL, (cz * a.geo.nc[1] + cy) * a.geo.nc[0] + cx, a.ncell);
        const int cnt = skip ? 0 : min(a.cell_count[cell], a.cell_cap);
        const uint4* cq = a.cell_q + (size_t)cell * a.cell_cap;
        auto dist2 = [&](const uint4& o) {
          if constexpr (sizeof(T) == 4) {
            const V3<float> d = a.pv.vec_of(si, o);
            return dot3(d, d);
          } else {
            const float ex = __uint_as_float(o.x) - (rel[0] - (float)dx * w[0]),
                        ey = __uint_as_float(o.y) - (rel[1] - (float)dy * w[1]),
                        ez = __uint_as_float(o.z) - (rel[2] - (float)dz * w[2]);
            return ex * ex + ey * ey + ez * ez;
          }
        };
        if constexpr (LANES == 1) {
#pragma unroll 4
          for (int k = 0; k < cnt; ++k) {
            const uint4 o = cq[k];
            const int j = (int)o.w;
            if (dist2(o) < lim && j != i) {
              if (m < a.max_nb) tmp[(size_t)m * a.nmax] = APIP_CHK(a.status, BND_CELL, j, a.n);
              ++m;
            }
          }
        } else {
          const int most = __reduce_max_sync(0xffffffffu, cnt);
          for (int k = g; k < most + g; k += LANES) {
            bool in = false;
            int j = 0;
            if (k < cnt) {
              const uint4 o = cq[k];
              j = APIP_CHK(a.status, BND_CELL, (int)o.w, a.n);
              in = dist2(o) < lim && j != i;
            }
            const unsigned bal = (__ballot_sync(0xffffffffu, in) >> gshift) & gmask;
            const int at = m + __popc(bal & below);
            if (in && own && at < a.max_nb) tmp[(size_t)at * a.nmax] = j;
            m += __popc(bal);
          }
        }
      }
    }
  }
  if constexpr (LANES > 1) __syncwarp();
  if (own && m <= a.max_nb) {   // (only its own threads read a column: they tag its entries here)
    // exact classes; every kept index fits the scratch column
    if constexpr (LANES == 1) {
      int rest = 0;
      constexpr int B = 4;   // entries in flight
      for (int s0 = 0; s0 < m; s0 += B) {
        int js[B];
        typename PosView<T>::Rec rec[B];
#pragma unroll
        for (int q = 0; q < B; ++q) js[q] = tmp[(size_t)min(s0 + q, m - 1) * a.nmax];
#pragma unroll
        for (int q = 0; q < B; ++q) rec[q] = a.pv.fetch(js[q]);
#pragma unroll
        for (int q = 0; q < B; ++q) {
          if (s0 + q >= m) break;
          const auto d = a.pv.vec_of(si, rec[q]);
          const T r2 = dot3(d, d);
          const int cls = build_class(a, r2);
          if (cls == 0) {
            a.nbl[(size_t)n0 * a.nmax + i] = js[q];
            ++n0;
          } else if (cls < 3) {
            tmp[(size_t)rest * a.nmax] = (int)((unsigned)js[q] | ((unsigned)cls << kClassShift));
            ++rest;
            if (cls == 1) {
              ++n1;
              min1 = r2 < min1 ? r2 : min1;
            }
          }
        }
      }
      n2 = rest - n1;
      int p1 = n0, p2 = n0 + n1;
      for (int s = 0; s < rest; ++s) {
        const unsigned v = (unsigned)tmp[(size_t)s * a.nmax];
        const bool first = (v >> kClassShift) == 1u;
        a.nbl[(size_t)(first ? p1 : p2) * a.nmax + i] = (int)(v & ((1u << kClassShift) - 1u));
        p1 += first ? 1 : 0;
        p2 += first ? 0 : 1;
      }
    } else {
      for (int s = g; s < m; s += LANES) {
        const int j = tmp[(size_t)s * a.nmax];
        const auto d = a.pv.vec(si, j);
        const T r2 = dot3(d, d);
        const int cls = build_class(a, r2);
        if (own) tmp[(size_t)s * a.nmax] = (int)((unsigned)j | ((unsigned)cls << kClassShift));
        n0 += cls == 0;
        n1 += cls == 1;
        n2 += cls == 2;
        if (cls == 1) min1 = r2 < min1 ? r2 : min1;
      }
    }
  }
  if constexpr (LANES > 1) {
    __syncwarp();
#pragma unroll
    for (int o = 1; o < LANES; o <<= 1) {
      n0 += __shfl_xor_sync(0xffffffffu, n0, o);
      n1 += __shfl_xor_sync(0xffffffffu, n1, o);
      n2 += __shfl_xor_sync(0xffffffffu, n2, o);
      const T v = __shfl_xor_sync(0xffffffffu, min1, o);
      min1 = v < min1 ? v : min1;
    }
    const int mm = own && m <= a.max_nb ? m : 0;
    const int most = __reduce_max_sync(0xffffffffu, mm);
    int p0 = 0, p1 = n0, p2 = n0 + n1;
    for (int s = g; s < most + g; s += LANES) {
      const unsigned v = s < mm ? (unsigned)tmp[(size_t)s * a.nmax] : 0xffffffffu;
      const int cls = (int)(v >> kClassShift);
      const unsigned b0 = (__ballot_sync(0xffffffffu, cls == 0) >> gshift) & gmask;
      const unsigned b1 = (__ballot_sync(0xffffffffu, cls == 1) >> gshift) & gmask;
      const unsigned b2 = (__ballot_sync(0xffffffffu, cls == 2) >> gshift) & gmask;
      const int at = cls == 0 ? p0 + __popc(b0 & below) : (cls == 1 ? p1 + __popc(b1 & below) : p2 + __popc(b2 & below));
      if (own && cls < 3) a.nbl[(size_t)at * a.nmax + i] = (int)(v & ((1u << kClassShift) - 1u));
      p0 += __popc(b0);
      p1 += __popc(b1);
      p2 += __popc(b2);
    }
    if (!own || g != 0) return;
  }
  k0 = n0;
  k1 = n1;
  k2 = n2;
  if (m > a.max_nb) {
    // more kept by the scan than the column holds (an overflow, or a list at its very
    // capacity): one thread scans again, class by class, with the exact test
    n0 = n1 = n2 = 0;
    min1 = T(INFINITY);
    int kept = 0;
    for (int cls = 0; cls < 3; ++cls) {
      int found = 0;
      for (int q = 0; q < 27; ++q) {
        const int x = (c[0] + q % 3 - 1 + a.geo.nc[0]) % a.geo.nc[0], y = (c[1] + q / 3 % 3 - 1 + a.geo.nc[1]) % a.geo.nc[1],
                  z = (c[2] + q / 9 - 1 + a.geo.nc[2]) % a.geo.nc[2];
        const int cell = (z * a.geo.nc[1] + y) * a.geo.nc[0] + x;
        const int cnt = min(a.cell_count[cell], a.cell_cap);
        for (int k = 0; k < cnt; ++k) {
          const int j = APIP_CHK(a.status, BND_CELL, (int)a.cell_q[(size_t)cell * a.cell_cap + k].w, a.n);
          if (j == i) continue;
          const auto d = a.pv.vec(si, j);
          const T r2 = dot3(d, d);
          if (build_class(a, r2) != cls) continue;
          if (cls == 1) min1 = r2 < min1 ? r2 : min1;
          if (kept < a.max_nb) a.nbl[(size_t)kept++ * a.nmax + i] = j;
          ++found;
        }
      }
      (cls == 0 ? n0 : (cls == 1 ? n1 : n2)) = found;
    }
    k0 = min(n0, a.max_nb);
    k1 = min(n1, a.max_nb - k0);
    k2 = min(n2, a.max_nb - k0 - k1);
    const int cnt = n0 + n1 + n2;
    if (cnt > a.max_nb) {
      atomicOr(&a.status[ST_NB_OVERFLOW], 1);
      atomicMax(&a.status[ST_MAX_NNB], cnt);
    }
  }
  a.nnb[i] = k0 + k1 + k2;
  a.nnb_e[i] = k0 + k1;
  a.nnb_0[i] = k0;
  if constexpr (sizeof(T) == 4) a.mind1[i] = k1 < n1 ? 0.f : min1;   // a class-1 entry dropped on overflow: never skip class 1
  // the positions of this build: the FP64 path's displacement reference, and in
  // both paths what a checkpoint keeps to rebuild the same list on resume
  if (sizeof(T) == 4) a.posq_ref[i] = a.posq[i];
  a.pos_ref[3 * i] = a.pos[3 * i];
  a.pos_ref[3 * i + 1] = a.pos[3 * i + 1];
  a.pos_ref[3 * i + 2] = a.pos[3 * i + 2];
}

// The same, FP32 path, one thread per atom: class 0 goes straight to the list, classes
// 1 and 2 to the two ends of the scratch column, copied behind class 0 at the end.
// (The two-round form of k_nbfill was slower here, 281 -> 440 us at 249 k atoms: each
// lane's stores go to rows of their own, and it makes 150 of them per atom, not 90.)
__global__ void k_nbfill_one(Args<float> a) {
  pdl_begin();
  if (!a.flags[0]) return;
  // the new list's reference positions are the current ones: no displacement yet
  if (blockIdx.x == 0 && threadIdx.x == 0) a.flags[1] = 0;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  int c[3];
  const auto si = a.pv.self(i);
  const unsigned qq[3] = {si.q.x, si.q.y, si.q.z};
#pragma unroll
  for (int k = 0; k < 3; ++k) c[k] = (int)(((unsigned long long)qq[k] * (unsigned)a.geo.nc[k]) >> 32);
  const float rin2 = a.r_e_in2f, rmid2 = a.r_e_mid2f;
  int n0 = 0, n1 = 0, n2 = 0;   // class counts
  int w1 = 0, w2 = 0;           // class 1, 2 entries written to the scratch ends
  float min1 = INFINITY;        // least squared distance in class 1
  auto keep = [&](int j, float r2) {
    if (r2 < rin2) {
      if (n0 < a.max_nb) a.nbl[(size_t)n0 * a.nmax + i] = j;
      ++n0;
    } else if (r2 < rmid2) {
      if (w1 + w2 < a.max_nb) a.nbl_tmp[(size_t)(w1++) * a.nmax + i] = j;   // the ends meet only on overflow
      min1 = r2 < min1 ? r2 : min1;
      ++n1;
    } else {
      if (w1 + w2 < a.max_nb) a.nbl_tmp[(size_t)(a.max_nb - 1 - w2++) * a.nmax + i] = j;
      ++n2;
    }
  };
  // the squared distance from the atom to the nearest face of the neighbour cell at
  // offset -1, 0, +1 along each axis, from the atom's fraction within its own cell
  // (the low 32 bits of q * nc, exact); a cell whose nearest point is beyond r_list
  // (with a 1e-5 relative margin, far above the rounding of these gaps) holds no
  // candidate and is skipped.  Only with at least 5 cells per axis, where no member of
  // a neighbour cell is nearer through the other side of the box.
  float lo2[3] = {0.f, 0.f, 0.f}, hi2[3] = {0.f, 0.f, 0.f};
  float prune2 = INFINITY;
  if (a.geo.nc[0] >= 5 && a.geo.nc[1] >= 5 && a.geo.nc[2] >= 5) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const unsigned frac = (unsigned)((unsigned long long)qq[k] * (unsigned)a.geo.nc[k]);
      const float w = a.pv.unit[k] / (float)a.geo.nc[k];
      const float lo = (float)frac * w, hi = (4294967296.0f - (float)frac) * w;
      lo2[k] = lo * lo;
      hi2[k] = hi * hi;
    }
    prune2 = (float)(a.r_list2 * (1.0 + 1e-5));
  }
  auto gap = [&](int k, int d) { return d < 0 ? lo2[k] : (d > 0 ? hi2[k] : 0.f); };
  for (int dz = -1; dz <= 1; ++dz) {
    const int cz = (c[2] + dz + a.geo.nc[2]) % a.geo.nc[2];
    for (int dy = -1; dy <= 1; ++dy) {
      const int cy = (c[1] + dy + a.geo.nc[1]) % a.geo.nc[1];
      const float gzy = gap(2, dz) + gap(1, dy);
      for (int dx = -1; dx <= 1; ++dx) {
        if (gzy + gap(0, dx) > prune2) continue;
        const int cx = (c[0] + dx + a.geo.nc[0]) % a.geo.nc[0];
        const int cell = APIP_CHK(a.status, BND_CELL, (cz * a.geo.nc[1] + cy) * a.geo.nc[0] + cx, a.ncell);
        const int m = min(a.cell_count[cell], a.cell_cap);
        // float comparison against r_list^2 rounded up: the list holds every pair whose
        // float distance is below r_list (and perhaps a few at r_list)
        const uint4* cq = a.cell_q + (size_t)cell * a.cell_cap;
        const float rl2 = a.r_list2f;
#pragma unroll 2
        for (int k = 0; k < m; ++k) {
          const uint4 o = cq[k];
          const float ex = (float)(int)(o.x - si.q.x) * a.pv.unit[0];
          const float ey = (float)(int)(o.y - si.q.y) * a.pv.unit[1];
          const float ez = (float)(int)(o.z - si.q.z) * a.pv.unit[2];
          const float r2 = ex * ex + ey * ey + ez * ez;
          if (r2 < rl2 && (int)o.w != i) keep(APIP_CHK(a.status, BND_CELL, (int)o.w, a.n), r2);
        }
      }
    }
  }
  const int cnt = n0 + n1 + n2;
  if (cnt > a.max_nb) {
    atomicOr(&a.status[ST_NB_OVERFLOW], 1);
    atomicMax(&a.status[ST_MAX_NNB], cnt);
  }
  // the kept entries: the first max_nb in class order
  const int k0 = min(n0, a.max_nb), k1 = min(w1, a.max_nb - k0), k2 = min(w2, a.max_nb - k0 - k1);
  for (int s = 0; s < k1; ++s) a.nbl[(size_t)(k0 + s) * a.nmax + i] = a.nbl_tmp[(size_t)s * a.nmax + i];
  for (int s = 0; s < k2; ++s)
    a.nbl[(size_t)(k0 + k1 + s) * a.nmax + i] = a.nbl_tmp[(size_t)(a.max_nb - 1 - s) * a.nmax + i];
  a.nnb[i] = k0 + k1 + k2;
  a.nnb_e[i] = k0 + k1;
  a.nnb_0[i] = k0;
  a.mind1[i] = k1 < n1 ? 0.f : min1;   // a class-1 entry dropped on overflow: never skip class 1
  // the positions of this build: the displacement reference, and what a checkpoint
  // keeps to rebuild the same list on resume
  a.posq_ref[i] = si.q;
  a.pos_ref[3 * i] = a.pos[3 * i];
  a.pos_ref[3 * i + 1] = a.pos[3 * i + 1];
  a.pos_ref[3 * i + 2] = a.pos[3 * i + 2];
}

// -------------------------------------------------------------- CSP pairs
// Detection at t = 0 (Eq. B3): the csp_nnb nearest neighbours within
// csp_rcut (ordered by squared distance, ties by id) are paired greedily by
// ascending |r_ia + r_ib|^2 (ties by rank).  All float64 operations are
// explicitly rounded (no contraction) so the pairing is reproducible.
__device__ __forceinline__ double sq_rn(double x, double y, double z) {
  return __dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z));
}

__device__ __forceinline__ double minimg_rn(double d, double L) {
  return __dsub_rn(d, __dmul_rn(L, rint(__ddiv_rn(d, L))));
}

__global__ void k_csp_init(Args<double> a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  double r2s[kCspCap], rv[kCspCap][3];
  int ids[kCspCap];
  int m = 0;
  const int K = a.csp_nnb;
  const double xi = a.pos[3 * i], yi = a.pos[3 * i + 1], zi = a.pos[3 * i + 2];
  const int cnt = APIP_CHK(a.status, BND_LIST_LEN, a.nnb[i], a.max_nb + 1);
  for (int s = 0; s < cnt; ++s) {
    const int j = APIP_CHK(a.status, BND_NEIGHBOUR, a.nbl[(size_t)s * a.nmax + i], a.n);
    const double dx = minimg_rn(__dsub_rn(a.pos[3 * j], xi), a.geo.L[0]);
    const double dy = minimg_rn(__dsub_rn(a.pos[3 * j + 1], yi), a.geo.L[1]);
    const double dz = minimg_rn(__dsub_rn(a.pos[3 * j + 2], zi), a.geo.L[2]);
    const double r2 = sq_rn(dx, dy, dz);
    if (!(r2 < a.csp_rcut2)) continue;
    const int idj = a.id[j];
    // insert into the sorted list of the K best (r2, id)
    if (m == K && !(r2 < r2s[K - 1] || (r2 == r2s[K - 1] && idj < ids[K - 1]))) continue;
    if (m < K) ++m;
    int p = m - 1;
    while (p > 0 && (r2 < r2s[p - 1] || (r2 == r2s[p - 1] && idj < ids[p - 1]))) {
      r2s[p] = r2s[p - 1]; ids[p] = ids[p - 1];
      rv[p][0] = rv[p - 1][0]; rv[p][1] = rv[p - 1][1]; rv[p][2] = rv[p - 1][2];
      --p;
    }
    r2s[p] = r2; ids[p] = idj; rv[p][0] = dx; rv[p][1] = dy; rv[p][2] = dz;
  }
  const int idv = a.id[i];   // rows are kept by atom id, so atoms may be reordered later
  if (idv < 0 || idv >= a.nmax) return;   // reported by prep (ST_BAD_INPUT)
  int* out = a.csp + (size_t)idv * kCspCap;
  for (int k = 0; k < kCspCap; ++k) out[k] = -1;
  bool used[kCspCap];
  for (int k = 0; k < kCspCap; ++k) used[k] = false;
  for (int k = 0; 2 * k < K; ++k) {
    double best = 0.0;
    int bp = -1, bq = -1;
    for (int p = 0; p < m; ++p) {
      if (used[p]) continue;
      for (int q = p + 1; q < m; ++q) {
        if (used[q]) continue;
        const double s2 = sq_rn(__dadd_rn(rv[p][0], rv[q][0]), __dadd_rn(rv[p][1], rv[q][1]),
                                __dadd_rn(rv[p][2], rv[q][2]));
        if (bp < 0 || s2 < best) { best = s2; bp = p; bq = q; }
      }
    }
    if (bp < 0) break;
    used[bp] = used[bq] = true;
    out[2 * k] = ids[bp];
    out[2 * k + 1] = ids[bq];
  }
}

// Restored partner ids: the row of atom id i (kCspCap entries) from
// src[i * nnb .. + nnb), -1 beyond.
__global__ void k_set_csp(const int32_t* src, int* dst, int n, int nnb) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
#pragma unroll
  for (int k = 0; k < kCspCap; ++k) dst[(size_t)i * kCspCap + k] = k < nnb ? src[(size_t)i * nnb + k] : -1;
}

// The passes over the neighbour list: LANES threads share an atom (1 in a large
// system; 4 or 8 where one thread per atom would leave most of the GPU idle and
// each thread's chain of some 60 entries would be the pass's whole time: pass 1 and
// pass 2 at 2 k atoms 21 + 21 -> 9 + 10 us, at 27 k atoms 24 + 25 -> 13 + 14 us).  Thread g
// of an atom takes the entries s0 + g, s0 + g + LANES, ...
//
// FP32 path: two entries at a time, packed (pair2.cuh), the records of the next two
// in flight meanwhile (pass 2 at 249 k atoms: 70 -> 56 us).  f(s of the first, record, record, count of valid entries: 1 or 2).
template <int LANES, typename L, typename F>
__device__ __forceinline__ void walk_pairs(const int* nb, int nmax, int s0, int s1, int g, int* status, int n, L&& load,
                                           F&& f) {
  (void)status;
  (void)n;
  int s = s0 + g;
  if (s >= s1) return;
  const size_t step = (size_t)LANES * nmax;
  const int* p = nb + (size_t)s * nmax;
  int ja = APIP_CHK(status, BND_NEIGHBOUR, p[0], n), jb = s + LANES < s1 ? APIP_CHK(status, BND_NEIGHBOUR, p[step], n) : ja;
  auto ra = load(ja), rb = load(jb);
  p += 2 * step;
  ja = s + 2 * LANES < s1 ? APIP_CHK(status, BND_NEIGHBOUR, p[0], n) : ja;
  jb = s + 3 * LANES < s1 ? APIP_CHK(status, BND_NEIGHBOUR, p[step], n) : ja;
  for (; s < s1; s += 2 * LANES) {
    const auto ca = ra, cb = rb;
    ra = load(ja);
    rb = load(jb);
    p += 2 * step;
    if (s + 4 * LANES < s1) ja = APIP_CHK(status, BND_NEIGHBOUR, p[0], n);
    if (s + 5 * LANES < s1) jb = APIP_CHK(status, BND_NEIGHBOUR, p[step], n);
    f(s, ca, cb, s + LANES < s1 ? 2 : 1);
  }
}

// Separations of two neighbours, their r^2 and (1/r, r); an invalid second entry
// is put at r^2 = far2, outside every cutoff.
struct Sep2 { F2 x, y, z, r2, r, ir; };
__device__ __forceinline__ Sep2 sep2(const PosView<float>& pv, const PosView<float>::Self& s, const uint4& a,
                                     const uint4& b, int valid, float far2) {
  Sep2 d;
  d.x = mul2(f2((float)(int)(a.x - s.q.x), (float)(int)(b.x - s.q.x)), f2(pv.unit[0]));
  d.y = mul2(f2((float)(int)(a.y - s.q.y), (float)(int)(b.y - s.q.y)), f2(pv.unit[1]));
  d.z = mul2(f2((float)(int)(a.z - s.q.z), (float)(int)(b.z - s.q.z)), f2(pv.unit[2]));
  // (the order in which the compiler contracts dot3, so that both give the same bits)
  d.r2 = fma2(d.z, d.z, fma2(d.x, d.x, mul2(d.y, d.y)));
  if (valid < 2) d.r2 = f2(f2_get(d.r2).x, far2);
  d.ir = rsqrt2(d.r2);
  d.r = mul2(d.r2, d.ir);
  return d;
}

// The EAM terms of one float32 neighbour in scalar form (entries beyond class 0 that
// have come within the cutoff: rare), the same operations as the packed forms.
struct EamTerm { float rho, phi, drho, dphi; };
__device__ __noinline__ EamTerm eam_rare(const PassK<float>& k, float r) {
  float dfc;
  const float fc = ftrans(r, k.eam_rc_lo, k.eam_rc, k.eam_inv_w, &dfc);
  const float er = k.eam_A * fexp(-k.eam_beta * (r - k.eam_re));
  const float x = fexp(-k.eam_alpha * (r - k.eam_r0));
  return {er * fc, k.eam_D * (x * x - 2.f * x) * fc, er * (dfc - k.eam_beta * fc),
          k.eam_D * (2.f * k.eam_alpha * (x - x * x) * fc + (x * x - 2.f * x) * dfc)};
}

// ------------------------------------------------------------------ pass 1
// zeta_i and E_i^EAM (Eq. B1, S8), xi'(zeta_i), and g_i = CSP^list_i (Eq. B3).
// The EAM sums read only the first nnb_e list entries (the pairs that can be
// within the EAM cutoff).  FP32 path: also writes posg[i] = (posq[i], g_i) for
// pass 2.
// FP64 path: with one thread per atom bound by the float64 pipe, some 65 operations a
// pair with exp_tab's table in shared memory (tab), 100 with the library's exponential
// (249 k atoms, pass 1 and pass 2 with the shorter taper and smaller blocks: the step
// 3.16 -> 2.81 ms).  A small system is not bound by it and loses more by the table's
// loads and barrier in front of each short kernel (2 k atoms: 318 us a step without,
// 355 with it).
__device__ double2 g_exp_tab[kExpTab];
template <typename T, int LANES>
__host__ __device__ constexpr bool exp_by_table() { return sizeof(T) == 8 && LANES == 1; }

template <typename T, int LANES>
__device__ __forceinline__ void eam_sums(const Args<T>& a, int i, int g, const double2* tab, T* zeta_out, T* pair_out) {
  const auto si = a.pv.self(i);
  const int end0 = APIP_CHK(a.status, BND_LIST_LEN, a.nnb_0[i], a.max_nb + 1);
  int end = APIP_CHK(a.status, BND_LIST_LEN, a.nnb_e[i], a.max_nb + 1);
  if constexpr (sizeof(T) == 4) {
    // a class-1 entry (build distance r_b in [rc, rc + skin)) is now at
    // r >= r_b - d_i - d_j, where d_i is this atom's displacement since the build
    // and d_j <= the largest one (flags[1]); when the least r_b of the atom's
    // class-1 entries is at least rc + d_i + d_max (+ a rounding margin), none of
    // them is within the cutoff and the sums stop after class 0
    const float dmax2 = __int_as_float(a.flags[1]);   // NaN (-1) before the first build: no skip
    const uint4 r = a.posq_ref[i];
    const float ex = (float)(int)(si.q.x - r.x) * a.pv.unit[0], ey = (float)(int)(si.q.y - r.y) * a.pv.unit[1],
                ez = (float)(int)(si.q.z - r.z) * a.pv.unit[2];
    const float lim = a.k.eam_rc + sqrtf(ex * ex + ey * ey + ez * ez) + sqrtf(dmax2) + 1e-3f;
    if (a.mind1[i] >= lim * lim) end = end0;
    const float rc2 = a.k.eam_rc2, far2 = 4.f * rc2;
    const F2 tc = f2(a.k.eam_rc + a.k.eam_rc_lo), tw = f2(a.k.eam_inv_w);
    Acc2 zeta, pair;
    auto load = [&](int j) { return a.pv.fetch(j); };
    walk_pairs<LANES>(a.nbl + i, a.nmax, 0, end0, g, a.status, a.n, load,
                      [&](int, const uint4& oa, const uint4& ob, int valid) {
                        const Sep2 d = sep2(a.pv, si, oa, ob, valid, far2);
                        const F2 fc = taper_f(taper_t(d.r, tc, tw));   // 0 beyond the cutoff
                        const F2 er = exp2x(mul2(f2(-a.k.eam_beta), sub2(d.r, f2(a.k.eam_re))));
                        const F2 x = exp2x(mul2(f2(-a.k.eam_alpha), sub2(d.r, f2(a.k.eam_r0))));
                        zeta.add_prod(mul2(f2(a.k.eam_A), er), fc);
                        pair.add_prod(mul2(f2(a.k.eam_D), fma2(x, x, mul2(f2(-2.f), x))), fc);
                      });
    walk_pairs<LANES>(a.nbl + i, a.nmax, end0, end, g, a.status, a.n, load,
                      [&](int, const uint4& oa, const uint4& ob, int valid) {
                        const Sep2 d = sep2(a.pv, si, oa, ob, valid, far2);
                        const float2 r2 = f2_get(d.r2);
                        if (r2.x < rc2 || r2.y < rc2) {
                          const float2 r = f2_get(d.r);
                          const EamTerm u = r2.x < rc2 ? eam_rare(a.k, r.x) : EamTerm{}, v = r2.y < rc2 ? eam_rare(a.k, r.y) : EamTerm{};
                          zeta.add(f2(u.rho, v.rho));
                          pair.add(f2(u.phi, v.phi));
                        }
                      });
    *zeta_out = zeta.template value<LANES>();
    *pair_out = pair.template value<LANES>();
  } else {
    const T rc2 = a.k.eam_rc2, rc = a.k.eam_rc, rlo = a.k.eam_rc_lo, inv_w = a.k.eam_inv_w;
    T zeta = T(0), pair = T(0);
    const int cached = min(end0, a.pair_rows);
    for (int s = g; s < end; s += LANES) {
      const int j = APIP_CHK(a.status, BND_NEIGHBOUR, a.nbl[(size_t)s * a.nmax + i], a.n);
      const auto d = a.pv.vec(si, j);
      const T r2 = dot3(d, d);
      double2 keep = make_double2(0.0, 0.0);
      if (less_pos(r2, rc2)) {
        T r, ir;
        len_inv(r2, &r, &ir);
        T fc = T(1), dfc = T(0);
        if (!less_pos(r, rlo)) fc = ftrans_in(r, rlo, rc, inv_w, &dfc);
        auto expo = [&](T v) { return exp_by_table<T, LANES>() ? exp_tab(tab, v) : fexp(v); };
        const T er = a.k.eam_A * expo(-a.k.eam_beta * (r - a.k.eam_re));
        const T x = expo(-a.k.eam_alpha * (r - a.k.eam_r0));
        const T q = x * x - T(2) * x;
        zeta += er * fc;
        pair += a.k.eam_D * q * fc;
        keep.x = er * (dfc - a.k.eam_beta * fc) * ir;
        keep.y = a.k.eam_D * (T(2) * a.k.eam_alpha * (x - x * x) * fc + q * dfc) * ir;
      }
      if (s < cached) a.pair_keep[(size_t)s * a.nmax + i] = keep;
    }
#pragma unroll
    for (int o = 1; o < LANES; o <<= 1) {
      zeta += __shfl_xor_sync(0xffffffffu, zeta, o);
      pair += __shfl_xor_sync(0xffffffffu, pair, o);
    }
    *zeta_out = zeta;
    *pair_out = pair;
  }
}

// g_i = sum over the partner pairs of |r_ia + r_ib|^2 (Eq. B3).  The partner ids come
// from the row of this atom's id; their indices from the cache of the last call
// (valid while the atom at index i keeps its id and its partners keep their
// indices), checked against the ids, else from the id -> index map, and the cache
// rewritten (idx = -1: no partner, -2: id out of range).  Thread g of an atom takes
// the pairs g, g + LANES, ... (the sum is made in pair order by every thread).
template <typename T, int LANES>
__device__ __forceinline__ T csp_g(const Args<T>& a, int i, int g) {
  static_assert(kCspCap == 8, "four pairs of partner ids");
  constexpr int NP = kCspCap / 2, MINE = LANES >= NP ? 1 : NP / LANES;
  const auto si = a.pv.self(i);
  const int idv = a.id[i], own = a.csp_owner[i];
  const bool idok = idv >= 0 && idv < a.nmax;   // an invalid id: reported by prep, no partners
  const int2* ids = reinterpret_cast<const int2*>(a.csp + (size_t)(idok ? idv : 0) * kCspCap);
  int2* at = reinterpret_cast<int2*>(a.csp_idx + (size_t)i * kCspCap);
  int2 pid[MINE], idx[MINE];
  if constexpr (LANES == 1) {   // whole rows, two 16-byte loads each
#pragma unroll
    for (int u = 0; u < NP; u += 2) {
      const int4 p = idok ? reinterpret_cast<const int4*>(ids)[u / 2] : make_int4(-1, -1, -1, -1);
      const int4 q = reinterpret_cast<const int4*>(at)[u / 2];
      pid[u] = make_int2(p.x, p.y);
      pid[u + 1] = make_int2(p.z, p.w);
      idx[u] = make_int2(q.x, q.y);
      idx[u + 1] = make_int2(q.z, q.w);
    }
  }
#pragma unroll
  for (int u = 0; u < MINE; ++u) {
    const int k = g + u * LANES;
    if constexpr (LANES > 1) {
      pid[u] = k < NP && idok ? ids[k] : make_int2(-1, -1);
      idx[u] = k < NP ? at[k] : make_int2(-1, -1);
    }
    if (2 * k >= a.csp_nnb) pid[u].x = -1;
    if (2 * k + 1 >= a.csp_nnb) pid[u].y = -1;
  }
  // a partner entry holds: its index, checked against the ids, -1 for no partner, -2
  // for an id out of range
  auto holds = [&](int p, int x) {
    if (p < 0) return x == -1;
    if (p >= a.nmax) return x == -2;
    return x >= 0 && x < a.n && a.id[x] == p;
  };
  bool hit = own == idv;
#pragma unroll
  for (int u = 0; u < MINE; ++u)
    if (g + u * LANES < NP) hit = hit && holds(pid[u].x, idx[u].x) && holds(pid[u].y, idx[u].y);
#pragma unroll
  for (int o = 1; o < LANES; o <<= 1) hit = (__shfl_xor_sync(0xffffffffu, (int)hit, o) != 0) && hit;
  if (!hit) {
    auto find = [&](int p) { return p < 0 ? -1 : (p >= a.nmax ? -2 : a.id2idx[p]); };
#pragma unroll
    for (int u = 0; u < MINE; ++u) {
      if (g + u * LANES >= NP) continue;
      idx[u] = make_int2(find(pid[u].x), find(pid[u].y));
      at[g + u * LANES] = idx[u];
    }
    if (g == 0) a.csp_owner[i] = idv;
  }
  int bad = 0;
  T val[MINE];
  int ok[MINE];
#pragma unroll
  for (int u = 0; u < MINE; ++u) {
    val[u] = T(0);
    ok[u] = 0;
    if (pid[u].x < 0 || pid[u].y < 0) continue;
    // the index must hold that partner now: the id -> index map keeps the entries of
    // ids that are no longer present
    if (idx[u].x < 0 || idx[u].y < 0 || !(hit || (holds(pid[u].x, idx[u].x) && holds(pid[u].y, idx[u].y)))) {
      bad = 1;
      continue;
    }
    const V3<T> v = csp_vec(a.pv, si, idx[u].x, idx[u].y);
    val[u] = dot3(v, v);
    ok[u] = 1;
  }
  Acc<T> gs;
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    const int u = k / LANES;
    T v = val[u];
    int o = ok[u];
    if (LANES > 1) {
      const int src = ((int)(threadIdx.x & 31u) / LANES) * LANES + k % LANES;
      v = __shfl_sync(0xffffffffu, v, src);
      o = __shfl_sync(0xffffffffu, o, src);
    }
    if (o) gs.add(v);
  }
#pragma unroll
  for (int o = 1; o < LANES; o <<= 1) bad |= __shfl_xor_sync(0xffffffffu, bad, o);
  if (bad && g == 0) {
    atomicOr(&a.status[ST_BAD_PARTNER], 1);
    a.csp_owner[i] = -2;   // looked up again next call
  }
  return gs.value();
}

template <typename T, int LANES>
__global__ void __launch_bounds__(kBlock) k_pass1(Args<T> a) {
  pdl_begin();
  __shared__ double sh[32];
  __shared__ double2 tab[exp_by_table<T, LANES>() ? kExpTab : 1];
  if constexpr (exp_by_table<T, LANES>()) {
    for (int k = threadIdx.x; k < kExpTab; k += blockDim.x) tab[k] = g_exp_tab[k];
    __syncthreads();
  }
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int g = LANES == 1 ? 0 : (int)(threadIdx.x % LANES);
  const bool active = t / LANES < a.n;
  T e_out = T(0);
  if (LANES > 1 || active) {
    const int i = LANES == 1 ? t : min(t / LANES, a.n - 1);   // (LANES > 1: the warp stays whole for its shuffles)
    T z, pair;
    eam_sums<T, LANES>(a, i, g, tab, &z, &pair);
    const T gi = a.lam_mode == APIP_LAM_PAPER ? csp_g<T, LANES>(a, i, g) : T(0);
    if (active && g == 0) {
      const T sz = z > T(0) ? sqrt(z) : T(0);
      const T e = -sz + T(0.5) * pair;
      a.zeta[i] = z;
      a.xi_p[i] = z > T(0) ? T(-0.5) / sz : T(0);
      a.e_eam[i] = e;
      const double e_ind = ind_energy(a, i);   // the external indenter, if any
      if (a.e_atom) a.e_atom[i] = (double)e + e_ind;
      e_out = e + (T)e_ind;
      a.g[i] = gi;
      if constexpr (sizeof(T) == 4) {
        const uint4 q = a.posq[i];
        a.posg[i] = make_uint4(q.x, q.y, q.z, __float_as_uint(gi));
      }
    }
  }
  const double tot = block_sum_t(e_out, sh);
  if (threadIdx.x == 0) a.partials[blockIdx.x] = tot;
}

// ------------------------------------------------------------------ pass 2
// Switch (Eq. 6, Eq. 2 with lam = 1 - f_trans), the EAM force with unit weights
// F_i = sum_k [(xi'_i + xi'_k) rho'(r_ik) + Phi'(r_ik)] e_ik  (S13; the lam-
// dependent part of S12 is added by the ACE kernel for the atoms with lam > 0),
// and warp-ballot compaction of {i : lam_i > 0} into ace_list.
//
// The force components keep compensated sums (their rounding decides how well the
// float32 path conserves the total momentum); w-bar and sum g w are plain: they
// decide the compaction here, and the ACE kernel recomputes them in float64 for the
// transition atoms, where their rounding would reach the energy.
template <typename T>
struct Pass2Sums { T wbar, S, fx, fy, fz; };   // without the atom's own term

template <bool PAPER, int LANES>
__device__ __forceinline__ Pass2Sums<float> pass2_sums(const Args<float>& a, int i, int g) {
  const auto si = a.pv.self(i);
  const PassK<float>& k = a.k;
  const float rw2 = k.sw_r_w2, rc2 = k.eam_rc2, far2 = 4.f * fmaxf(rc2, rw2);
  const F2 wc = f2(k.sw_r_w + k.sw_r_w_lo), ww = f2(k.sw_inv_w);
  const F2 tc = f2(k.eam_rc + k.eam_rc_lo), tw = f2(k.eam_inv_w), dw = f2(-2.f * k.eam_inv_w);
  const float xi_i = a.xi_p[i];
  const bool force = a.eam_force != 0;
  F2 wbar = f2(0.f), S = f2(0.f);
  Acc2 fx, fy, fz;
  auto weigh = [&](const Sep2& d, unsigned ga, unsigned gb) {
    const float2 r2 = f2_get(d.r2);
    const F2 w = taper_f(taper_t(d.r, wc, ww));   // 0 beyond r_w, where g is not looked at
    wbar = add2(wbar, w);
    S = fma2(f2(r2.x < rw2 ? __uint_as_float(ga) : 0.f, r2.y < rw2 ? __uint_as_float(gb) : 0.f), w, S);
  };
  const int cnt = APIP_CHK(a.status, BND_LIST_LEN, a.nnb[i], a.max_nb + 1);
  const int cnt_0 = APIP_CHK(a.status, BND_LIST_LEN, a.nnb_0[i], cnt + 1);
  const int cnt_e = APIP_CHK(a.status, BND_LIST_LEN, a.nnb_e[i], cnt + 1);
  // class 0: switch and force
  struct RecE { uint4 o; float xi; };
  walk_pairs<LANES>(a.nbl + i, a.nmax, 0, cnt_0, g, a.status, a.n, [&](int j) { return RecE{a.posg[j], a.xi_p[j]}; },
                    [&](int, const RecE& ea, const RecE& eb, int valid) {
                      const Sep2 d = sep2(a.pv, si, ea.o, eb.o, valid, far2);
                      if (PAPER) weigh(d, ea.o.w, eb.o.w);
                      if (!force) return;
                      const F2 t = taper_t(d.r, tc, tw);
                      const F2 fc = taper_f(t), dfc = taper_df(t, dw);
                      const F2 er = mul2(f2(k.eam_A), exp2x(mul2(f2(-k.eam_beta), sub2(d.r, f2(k.eam_re)))));
                      const F2 drho = mul2(er, fma2(f2(-k.eam_beta), fc, dfc));
                      const F2 x = exp2x(mul2(f2(-k.eam_alpha), sub2(d.r, f2(k.eam_r0))));
                      const F2 q = fma2(x, x, mul2(f2(-2.f), x));
                      const F2 xm = fma2(mul2(x, f2(-1.f)), x, x);
                      const F2 z = fma2(q, dfc, mul2(mul2(f2(2.f * k.eam_alpha), xm), fc));
                      const F2 xs = add2(f2(xi_i), f2(ea.xi, eb.xi));
                      const F2 sc = mul2(fma2(xs, drho, mul2(f2(k.eam_D), z)), d.ir);
                      const float2 r2 = f2_get(d.r2), sv = f2_get(sc);
                      const F2 sm = f2(r2.x < rc2 ? sv.x : 0.f, r2.y < rc2 ? sv.y : 0.f);
                      fx.add_prod(sm, d.x);
                      fy.add_prod(sm, d.y);
                      fz.add_prod(sm, d.z);
                    });
  // classes 1 and 2: the switch, and the force of the few class-1 entries that have
  // come within the cutoff
  walk_pairs<LANES>(a.nbl + i, a.nmax, cnt_0, PAPER ? cnt : cnt_e, g, a.status, a.n, [&](int j) { return a.posg[j]; },
                    [&](int s, const uint4& oa, const uint4& ob, int valid) {
                      const Sep2 d = sep2(a.pv, si, oa, ob, valid, far2);
                      if (PAPER) weigh(d, oa.w, ob.w);
                      const float2 r2 = f2_get(d.r2);
                      if (force && s < cnt_e && (r2.x < rc2 || r2.y < rc2)) {
                        const float2 r = f2_get(d.r), ir = f2_get(d.ir);
                        float sc[2] = {0.f, 0.f};
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                          if (!((q ? r2.y : r2.x) < rc2)) continue;
                          const int j = APIP_CHK(a.status, BND_NEIGHBOUR, a.nbl[(size_t)(s + q * LANES) * a.nmax + i], a.n);
                          const EamTerm u = eam_rare(k, q ? r.y : r.x);
                          sc[q] = ((xi_i + a.xi_p[j]) * u.drho + u.dphi) * (q ? ir.y : ir.x);
                        }
                        const F2 sm = f2(sc[0], sc[1]);
                        fx.add_prod(sm, d.x);
                        fy.add_prod(sm, d.y);
                        fz.add_prod(sm, d.z);
                      }
                    });
  return {PAPER ? sum2<LANES>(wbar) : 0.f, PAPER ? sum2<LANES>(S) : 0.f, fx.value<LANES>(), fy.value<LANES>(),
          fz.value<LANES>()};
}

// FP64 path.  What bounds it: the float64 pipe (two operations a cycle and SM).  So
// ranges are tested on the bit patterns, the EAM pair terms come from pass 1
// (pair_keep), a distance is only formed where the switch's taper needs it (249 k
// atoms: 2196 -> 1052 us; 2 k atoms, with eight threads per atom: 322 -> 35 us).
template <bool PAPER, int LANES>
__device__ __forceinline__ Pass2Sums<double> pass2_sums(const Args<double>& a, int i, int g) {
  const auto si = a.pv.self(i);
  const PassK<double>& k = a.k;
  const double rw2 = k.sw_r_w2, rc2 = k.eam_rc2, one2 = k.sw_r_w_lo * k.sw_r_w_lo;
  const double xi_i = a.xi_p[i];
  const bool force = a.eam_force != 0;
  const int cnt = APIP_CHK(a.status, BND_LIST_LEN, a.nnb[i], a.max_nb + 1);
  const int cnt_0 = APIP_CHK(a.status, BND_LIST_LEN, a.nnb_0[i], cnt + 1);
  const int cnt_e = APIP_CHK(a.status, BND_LIST_LEN, a.nnb_e[i], cnt + 1);
  const int kept = min(cnt_0, a.pair_rows), end = PAPER ? cnt : cnt_e;
  double wbar = 0.0, S = 0.0, fx = 0.0, fy = 0.0, fz = 0.0;
  int whole = 0;   // neighbours of weight exactly 1
  for (int s = g; s < end; s += LANES) {
    const int j = APIP_CHK(a.status, BND_NEIGHBOUR, a.nbl[(size_t)s * a.nmax + i], a.n);
    const auto d = a.pv.vec(si, j);
    const double r2 = dot3(d, d);
    if (PAPER && less_pos(r2, rw2)) {
      const double gj = a.g[j];
      if (!less_pos(one2, r2)) {
        ++whole;
        S += gj;
      } else {
        double r, ir, dw;
        len_inv(r2, &r, &ir);
        const double w = ftrans_in(r, k.sw_r_w_lo, k.sw_r_w, k.sw_inv_w, &dw);
        wbar += w;
        S += gj * w;
      }
    }
    if (force && s < cnt_e) {
      double sc = 0.0;
      if (s < kept) {
        const double2 u = a.pair_keep[(size_t)s * a.nmax + i];
        sc = (xi_i + a.xi_p[j]) * u.x + u.y;
      } else if (less_pos(r2, rc2)) {
        double r, ir, dfc;
        len_inv(r2, &r, &ir);
        const double fc = ftrans(r, k.eam_rc_lo, k.eam_rc, k.eam_inv_w, &dfc);
        const double er = k.eam_A * fexp(-k.eam_beta * (r - k.eam_re));
        const double x = fexp(-k.eam_alpha * (r - k.eam_r0));
        const double dphi = k.eam_D * (2.0 * k.eam_alpha * (x - x * x) * fc + (x * x - 2.0 * x) * dfc);
        sc = ((xi_i + a.xi_p[j]) * (er * (dfc - k.eam_beta * fc)) + dphi) * ir;
      } else {
        continue;
      }
      fx += sc * d.x;
      fy += sc * d.y;
      fz += sc * d.z;
    }
  }
#pragma unroll
  for (int o = 1; o < LANES; o <<= 1) {
    if (PAPER) {
      wbar += __shfl_xor_sync(0xffffffffu, wbar, o);
      S += __shfl_xor_sync(0xffffffffu, S, o);
      whole += __shfl_xor_sync(0xffffffffu, whole, o);
    }
    fx += __shfl_xor_sync(0xffffffffu, fx, o);
    fy += __shfl_xor_sync(0xffffffffu, fy, o);
    fz += __shfl_xor_sync(0xffffffffu, fz, o);
  }
  return {wbar + (double)whole, S, fx, fy, fz};
}

//
// With several threads per atom the ACE kernel's blocks are let onto the SMs only when
// those of this pass have ended.  Let in before, they go in twos and threes to the SMs
// that are free first while others stay empty, and an ACE block beside another takes up
// to 1.5 times as long: 40 compacted atoms of 8192, body order 4 on basis 7/3: 244 to 300
// -> 190 us; float64: 472 -> 358 us; 27 k-atom step 85.9 -> 83.5 us.  In a large system
// it gains nothing (249 k atoms: 177 us either way).
template <typename T, bool PAPER, int LANES>
__global__ void __launch_bounds__(kBlock, 3) k_pass2(Args<T> a) {
  if (LANES == 1) pdl_begin();
  else pdl_wait();
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int g = LANES == 1 ? 0 : (int)(threadIdx.x % LANES);
  const bool active = t / LANES < a.n && g == 0;
  const int i = LANES == 1 ? t : min(t / LANES, a.n - 1);   // (LANES > 1: the warp stays whole for its shuffles)
  T lam = T(0);
  double ind_fv = 0.0;   // this atom's indenter force . centre velocity
  Pass2Sums<T> u{};
  if (LANES > 1 || active) u = pass2_sums<PAPER, LANES>(a, i, g);
  if (active) {
    T dv = T(0), dl = T(0), wb = T(1);
    if (PAPER) {
      wb = T(1) + u.wbar;   // the atom's own term, w(0) = 1
      // (two atoms at one place, r = NaN in float32: the clamped taper lost it, zeta did not)
      if (sizeof(T) == 4 && a.zeta[i] != a.zeta[i]) wb = a.zeta[i];
      dv = (a.g[i] + u.S) / wb - a.k.sw_d0;
      lam = ftrans_c(dv, a.k.sw_d_lo, a.k.sw_d_hi, a.k.sw_inv_d, &dl);
    } else {
      lam = a.lam_mode == APIP_LAM_CONST1 ? T(1) : T(0);
    }
    if (a.lam_fixed) {
      const double f = a.lam_fixed[i];
      if (f == f) {   // not NaN: constant lam on this atom (Appendix B)
        lam = T(f);
        dl = T(0);
      }
    }
    a.lam[i] = lam;
    a.dlam[i] = dl;
    a.wbar[i] = wb;
    a.dd[i] = dv;
    if (a.force) {
      // force mixing (Eq. 3): this atom's EAM force enters with (1 - lam_i) from the
      // fast model plus, when the precise model contains the EAM, lam_i from it
      const T wf = a.force_mix ? T(1) - lam + (a.precise_adds_eam ? lam : T(0)) : T(1);
      double gx = (double)(wf * u.fx), gy = (double)(wf * u.fy), gz = (double)(wf * u.fz);
      double fi[3], ei;
      if (a.ind_on && ind_term(a, i, &ei, fi)) {   // indenter: K (R - r)^2 (x_i - c) / r
        gx += fi[0];
        gy += fi[1];
        gz += fi[2];
        ind_fv = fi[0] * a.ind_v[0] + fi[1] * a.ind_v[1] + fi[2] * a.ind_v[2];
      }
      a.force[3 * i] = fix_put(gx, a.det);
      a.force[3 * i + 1] = fix_put(gy, a.det);
      a.force[3 * i + 2] = fix_put(gz, a.det);
    }
  }
  if (a.ind_on && __syncthreads_or(ind_fv != 0.0)) {
    __shared__ double shw[32];
    const double w = block_sum(ind_fv, shw);
    if (threadIdx.x == 0) scatter_add(&a.ind_acc[2], w, a.det);
  }
  const bool pred = active && lam > T(0);
  if (a.det) {   // the block's count (k_blk_scan and k_compact_det write the list in index order; LANES is 1)
    const int cnt = __syncthreads_count(pred);
    if (threadIdx.x == 0) {
      a.blk_cnt[blockIdx.x] = cnt;
      if (cnt) atomicAdd(&a.counts[0], cnt);
    }
    return;
  }
  const unsigned mask = __ballot_sync(0xffffffffu, pred);
  const int lane = threadIdx.x & 31;
  int base = 0;
  if (lane == 0 && mask) base = atomicAdd(&a.counts[0], __popc(mask));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (pred) a.ace_list[base + __popc(mask & ((1u << lane) - 1u))] = i;
}

// Deterministic mode: pass 2's per-block counts turned into exclusive offsets, in
// place (one block; each thread a contiguous run of counts, then a scan of the
// run totals).
__global__ void __launch_bounds__(1024) k_blk_scan(int* cnt, int nb) {
  pdl_begin();
  __shared__ int sc[1024];
  const int per = (nb + blockDim.x - 1) / blockDim.x;
  const int b0 = min((int)threadIdx.x * per, nb), b1 = min(b0 + per, nb);
  int run = 0;
  for (int b = b0; b < b1; ++b) run += cnt[b];
  sc[threadIdx.x] = run;
  __syncthreads();
  for (int o = 1; o < (int)blockDim.x; o <<= 1) {   // inclusive scan of the run totals
    const int v = (int)threadIdx.x >= o ? sc[threadIdx.x - o] : 0;
    __syncthreads();
    sc[threadIdx.x] += v;
    __syncthreads();
  }
  int off = sc[threadIdx.x] - run;
  for (int b = b0; b < b1; ++b) {
    const int v = cnt[b];
    cnt[b] = off;
    off += v;
  }
}

// Deterministic mode: the compacted list {i : lam_i > 0} in index order, each
// block at the offset k_blk_scan computed for it.
template <typename T>
__global__ void __launch_bounds__(kBlock) k_compact_det(Args<T> a) {
  pdl_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool pred = i < a.n && a.lam[i] > T(0);
  const unsigned mask = __ballot_sync(0xffffffffu, pred);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ int wc[kBlock / 32];
  if (lane == 0) wc[warp] = __popc(mask);
  __syncthreads();
  int off = a.blk_cnt[blockIdx.x];
  for (int w = 0; w < warp; ++w) off += wc[w];
  if (pred) a.ace_list[APIP_CHK(a.status, BND_COMPACT, off + __popc(mask & ((1u << lane) - 1u)), a.n)] = i;
}

// Deterministic mode: the force array, summed as 64-bit fixed point by pass 2 and
// the scattering kernels, back to float64.
__global__ void k_fix_finish(double* force, int n3) {
  pdl_begin();
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n3) force[k] = fix_get(force + k, 1);
}

// Indenter work by the midpoint rule over one step (dt > 0), or just the shift of
// the last (sum F).v (dt = 0, a plain force evaluation).  acc[2] holds fixed point
// in deterministic mode.
__global__ void k_ind_work(double* acc, double dt, int det) {
  pdl_begin();
  const double f = fix_get(acc + 2, det);
  acc[0] += 0.5 * dt * (acc[1] + f);
  acc[1] = f;
  acc[2] = 0.0;
}

// -------------------------------------------- grad-lambda force, CSP part
// F -= grad sum_j c_j g_j (Eq. S25-S27) for the atoms with c_j != 0, where
// c_j = sum_k Et_k w(r_kj) was accumulated by the ACE kernel; resets c_j.  One
// thread per atom in index order: the few atoms with c_j != 0 lie near the
// transition region, and neighbouring threads then gather and scatter near one
// another (a list of them in the ACE kernel's first-touch order measured slower).
template <typename T>
__global__ void k_csp_force(Args<T> a) {
  pdl_begin();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= a.n) return;
  // c == +-0 tested on the bits (off the float64 pipe; a zero fixed-point slot has
  // the bits of +0), so that only the few atoms with c != 0 convert it
  const double raw = a.cvec[j];
  if ((__double_as_longlong(raw) << 1) == 0) return;
  const double c = a.det ? fix_get(&raw, 1) : raw;
  a.cvec[j] = 0.0;
  const auto sj = a.pv.self(j);
  // the partners' indices as pass 1 of this call checked them (cached by atom
  // index); a row pass 1 found bad is skipped (the error is reported)
  if (a.csp_owner[j] != a.id[j]) return;
  static_assert(kCspCap == 8, "two int4 rows of partner indices");
  const int4* c4 = reinterpret_cast<const int4*>(a.csp_idx + (size_t)j * kCspCap);
  const int4 q0 = c4[0], q1 = c4[1];
  const int idx[kCspCap] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
  bool ok[kCspCap / 2];
#pragma unroll
  for (int k = 0; k < kCspCap / 2; ++k) {
    const int ia = idx[2 * k], ib = idx[2 * k + 1];
    ok[k] = ia >= 0 && ib >= 0 && ia < a.n && ib < a.n;
  }
  double fj[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int k = 0; k < kCspCap / 2; ++k) {
    if (!ok[k]) continue;
    const int ia = idx[2 * k], ib = idx[2 * k + 1];
    const V3<T> uv = csp_vec(a.pv, sj, ia, ib);
    const double u[3] = {(double)uv.x, (double)uv.y, (double)uv.z};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      scatter_add(&a.force[3 * ia + q], -2.0 * c * u[q], a.det);
      scatter_add(&a.force[3 * ib + q], -2.0 * c * u[q], a.det);
      fj[q] += 4.0 * c * u[q];
    }
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) scatter_add(&a.force[3 * j + q], fj[q], a.det);
}

// ------------------------------------------------------------- reductions
__device__ __forceinline__ void neumaier(double& s, double& c, double v) {
  const double t = s + v;
  c += (fabs(s) >= fabs(v)) ? (s - t) + v : (v - t) + s;
  s = t;
}

// The float64 sums of a step, in one launch of many small blocks: the energy
// partials (value 0) and, with thermo, the four kinetic-energy and momentum
// partials per block of the Verlet kernel (values 1..4).
//
// What bounds it: an SM does two float64 additions a cycle, so one block that sums
// everything (972 x 5 partials for 249 k atoms, 15 600 x 5 for 4 M) takes its time in
// its own float64 pipe: 23 us at 249 k atoms.  With a partial or two per thread in
// 64-thread blocks over all SMs (whole step with thermo output, same run: 225.1 ->
// 217.5 us at 249 k atoms, 2.307 -> 2.163 ms at 4 M) the additions cost nothing;
// what is left is the latency of two dependent passes.  Each warp leaves its
// compensated sums (s, c) in scratch[warp][value][2]; the block that draws the last
// ticket adds them in warp order, so the sum does not depend on the order of the
// blocks.
__global__ void __launch_bounds__(kFinalThreads)
    k_final(const double* partials, int n_part, double* e_total, double* e_pot_slot, const double* thermo_part,
            int n_tb, double* thermo_slot, int* flags, const int* counts, int64_t* n_ace_out, int* cell_count, int ncell,
            double* scratch, int* ticket) {
  pdl_begin();
  if (flags && blockIdx.x == 0) end_list_build(flags, cell_count, ncell);
  constexpr int kWarps = kFinalThreads / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int t0 = blockIdx.x * kFinalThreads + threadIdx.x, stride = gridDim.x * kFinalThreads;
  double s[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, c[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int k = t0; k < n_part; k += stride) neumaier(s[0], c[0], partials[k]);
  if (thermo_part)
    for (int k = t0; k < n_tb; k += stride) {
      const double2 u = reinterpret_cast<const double2*>(thermo_part)[2 * k];
      const double2 v = reinterpret_cast<const double2*>(thermo_part)[2 * k + 1];
      neumaier(s[1], c[1], u.x);
      neumaier(s[2], c[2], u.y);
      neumaier(s[3], c[3], v.x);
      neumaier(s[4], c[4], v.y);
    }
  const int nq = thermo_part ? 5 : 1;
  for (int q = 0; q < nq; ++q) {
    const double ts = warp_sum(s[q]);
    const double tc = warp_sum(c[q]);
    if (lane == 0) {
      double* out = scratch + ((size_t)(blockIdx.x * kWarps + warp) * 5 + q) * 2;
      out[0] = ts;
      out[1] = tc;
    }
  }
  __shared__ int last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  const int nw = gridDim.x * kWarps;
  for (int q = warp; q < nq; q += kWarps) {
    double ts = 0.0, tc = 0.0;
    for (int w = lane; w < nw; w += 32) {
      const double* in = scratch + ((size_t)w * 5 + q) * 2;
      neumaier(ts, tc, __ldcg(in));
      tc += __ldcg(in + 1);
    }
    const double tot = warp_sum(ts) + warp_sum(tc);
    if (lane != 0) continue;
    if (q == 0) {
      if (e_total) *e_total = tot;
      if (e_pot_slot) *e_pot_slot = tot;
    } else {
      thermo_slot[q] = q == 1 ? 0.5 * tot : tot;   // partials hold 2 E_kin
    }
  }
  if (threadIdx.x == 0) {
    if (n_ace_out) *n_ace_out = (int64_t)counts[0];
    *ticket = 0;
  }
}

// ----------------------------------------------------------------- Verlet
// MODE 0: kick + drift (the first half step of a call); MODE 1: kick + kick +
// drift (the second half of step s fused with the first half of step s + 1);
// MODE 2: the final kick.  THERMO: the kinetic-energy and momentum partials of
// the step that the first kick ends (MODE 1, 2).  Both are template parameters:
// float64 arithmetic is slow on this GPU, and a run-time test would leave the
// compiler free to issue the float64 work of the other modes as predicated-off
// instructions on every atom.
template <typename T, int MODE, bool THERMO>
__global__ void __launch_bounds__(kBlock) k_verlet(Args<T> a, double* pos, double* vel, const double* force,
                                                   const double* inv_mass, double dt, double half_dt,
                                                   double* thermo_part) {
  pdl_begin();
  static_assert(!(THERMO && MODE == 0), "no thermo output before the first force");
  __shared__ double sh4[4 * 32];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (MODE != 2 && i == 0) a.counts[0] = a.counts[1] = 0;
  double ke = 0.0, p[3] = {0.0, 0.0, 0.0};   // ke: 2 E_kin of the atom (v . p; halved after the sums)
  float e2 = 0.f;                            // squared displacement since the list build (FP32 path)
  if (i < a.n) {
    const double im = inv_mass[i];
    const double h = half_dt * im;
    double f[3], v[3], x[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) f[q] = force[3 * i + q];
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q] = vel[3 * i + q] + h * f[q];
    if constexpr (THERMO) {
      // mass = 1/inv_mass: exact in the float64 path; a float reciprocal (relative
      // error ~1e-7 on each atom's E_kin and momentum) in the float32 path, where
      // a float64 division per atom would cost more than the rest of the kernel
      const double mass = sizeof(T) == 8 ? 1.0 / im : (double)(1.0f / (float)im);
#pragma unroll
      for (int q = 0; q < 3; ++q) p[q] = v[q] * mass;
      ke = v[0] * p[0] + v[1] * p[1] + v[2] * p[2];
    }
    if constexpr (MODE == 1) {
#pragma unroll
      for (int q = 0; q < 3; ++q) v[q] += h * f[q];
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) vel[3 * i + q] = v[q];
    if constexpr (MODE != 2) {
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        x[q] = wrap_near(pos[3 * i + q] + dt * v[q], a.geo.L[q], a.geo.invL[q]);
        pos[3 * i + q] = x[q];
      }
      e2 = prep_atom(a, i, x[0], x[1], x[2], true);
    }
  }
  if constexpr (MODE != 2) note_displacement(a, e2);
  if constexpr (THERMO) {
    const double vals[4] = {ke, p[0], p[1], p[2]};
    double tot[4];
    block_sum4(vals, sh4, tot);
    if (threadIdx.x == 0)
      for (int q = 0; q < 4; ++q) thermo_part[4 * blockIdx.x + q] = tot[q];
  }
}

// ------------------------------------------------------------ inspection
template <typename T>
__global__ void k_get_field(Args<T> a, int field, void* dst) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  double* dd = (double*)dst;
  long long* di = (long long*)dst;
  switch (field) {
    case APIP_FIELD_G: dd[i] = (double)a.g[i]; break;
    case APIP_FIELD_D: dd[i] = (double)a.dd[i]; break;
    case APIP_FIELD_WBAR: dd[i] = (double)a.wbar[i]; break;
    case APIP_FIELD_LAM: dd[i] = (double)a.lam[i]; break;
    case APIP_FIELD_DLAM: dd[i] = (double)a.dlam[i]; break;
    case APIP_FIELD_E_EAM: dd[i] = (double)a.e_eam[i]; break;
    case APIP_FIELD_E_ACE: dd[i] = a.lam[i] > T(0) ? (double)a.e_ace[i] : 0.0; break;
    case APIP_FIELD_ZETA: dd[i] = (double)a.zeta[i]; break;
    case APIP_FIELD_ACE_LIST: di[i] = i < a.counts[0] ? (long long)a.ace_list[i] : -1; break;
    case APIP_FIELD_NNB: di[i] = a.nnb[i]; break;
    case APIP_FIELD_NBLIST:
      for (int s = 0; s < a.max_nb; ++s)
        di[(size_t)i * a.max_nb + s] = s < a.nnb[i] ? (long long)a.nbl[(size_t)s * a.nmax + i] : -1;
      break;
    case APIP_FIELD_CSP:
      // row i: the partners of the atom whose id is i (the rows are kept by id)
      for (int s = 0; s < a.csp_nnb; ++s) di[(size_t)i * a.csp_nnb + s] = a.csp[(size_t)i * kCspCap + s];
      break;
    case APIP_FIELD_BUILD_POS:
      for (int q = 0; q < 3; ++q) dd[3 * i + q] = a.pos_ref[3 * i + q];
      break;
    default: break;
  }
}

inline int nblocks(int n, int b = kBlock) { return (n + b - 1) / b > 0 ? (n + b - 1) / b : 1; }

}  // namespace

// ---------------------------------------------------------------- launchers
template <typename T> void launch_prep(const Args<T>& a, cudaStream_t s) {
  launch_pdl(k_prep<T>, nblocks(a.n), kBlock, 0, s, a);
}

template <typename T> void launch_neighbors(const Args<T>& a, int ncell, cudaStream_t s) {
  (void)ncell;
  launch_pdl(k_bin<T>, nblocks(a.n), kBlock, 0, s, a);
  if (a.det) launch_pdl(k_cell_sort<T>, nblocks(a.ncell), kBlock, 0, s, a);
  if (a.lanes == 8) launch_pdl(k_nbfill<T, 8>, nblocks(8 * a.n), kBlock, 0, s, a);
  else if (a.lanes == 4) launch_pdl(k_nbfill<T, 4>, nblocks(4 * a.n), kBlock, 0, s, a);
  else if constexpr (sizeof(T) == 4) launch_pdl(k_nbfill_one, nblocks(a.n), kBlock, 0, s, a);
  else launch_pdl(k_nbfill<T, 1>, nblocks(a.n), kBlock, 0, s, a);
}

void launch_set_csp(const int32_t* src, int* dst, int n, int nnb, cudaStream_t s) {
  k_set_csp<<<nblocks(n), kBlock, 0, s>>>(src, dst, n, nnb);
}

void launch_csp_init(const Args<double>& a, cudaStream_t s) {
  k_csp_init<<<nblocks(a.n, 128), 128, 0, s>>>(a);
}

template <typename T> void launch_pass1(const Args<T>& a, cudaStream_t s) {
  const int pt = pass_threads(sizeof(T), a.lanes);
  if (a.lanes == 8) launch_pdl(k_pass1<T, 8>, nblocks(8 * a.n, pt), pt, 0, s, a);
  else if (a.lanes == 4) launch_pdl(k_pass1<T, 4>, nblocks(4 * a.n, pt), pt, 0, s, a);
  else launch_pdl(k_pass1<T, 1>, nblocks(a.n, pt), pt, 0, s, a);
}

// The table of exp_tab on the current device.
cudaError_t exp_table_set() {
  std::vector<double2> h(kExpTab);
  exp_table_fill(h.data());
  return cudaMemcpyToSymbol(g_exp_tab, h.data(), sizeof(double2) * kExpTab);
}

// Force mixing: the precise model's forces on the atoms with lam > 0 need E^prec
// of every atom within the ACE cutoff of them; those with lam = 0 are appended
// to the compacted list after pass 2.
template <typename T>
__global__ void __launch_bounds__(kBlock) k_fm_buffer(Args<T> a) {
  pdl_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  bool pred = false;
  if (i < a.n && a.lam[i] == T(0)) {
    const auto si = a.pv.self(i);
    const T rc2 = a.ace_rc * a.ace_rc;
    const int cnt = APIP_CHK(a.status, BND_LIST_LEN, a.nnb[i], a.max_nb + 1);
    const int* nb = a.nbl + i;
    for (int s = 0; s < cnt && !pred; ++s, nb += a.nmax) {
      const int j = APIP_CHK(a.status, BND_NEIGHBOUR, *nb, a.n);
      if (a.lam[j] > T(0)) {
        const auto d = a.pv.vec(si, j);
        pred = dot3(d, d) < rc2;
      }
    }
  }
  const unsigned mask = __ballot_sync(0xffffffffu, pred);
  const int lane = threadIdx.x & 31;
  int base = 0;
  if (lane == 0 && mask) base = atomicAdd(&a.counts[0], __popc(mask));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (pred) a.ace_list[base + __popc(mask & ((1u << lane) - 1u))] = i;
}

void launch_ind_work(double* acc, double dt, int det, cudaStream_t s) {
  launch_pdl(k_ind_work, 1, 1, 0, s, acc, dt, det);
}

void launch_fix_finish(double* force, int n, cudaStream_t s) {
  launch_pdl(k_fix_finish, nblocks(3 * n), kBlock, 0, s, force, 3 * n);
}

template <typename T> void launch_fm_buffer(const Args<T>& a, cudaStream_t s) {
  launch_pdl(k_fm_buffer<T>, nblocks(a.n), kBlock, 0, s, a);
}

template <typename T> void launch_pass2(const Args<T>& a, cudaStream_t s) {
  // (the deterministic mode's compaction counts per 256 atoms: one thread per atom)
  const int lanes = a.det ? 1 : a.lanes;
  const bool paper = a.lam_mode == APIP_LAM_PAPER || a.lam_mode == APIP_LAM_LEARNED;
  const int pt = pass_threads(sizeof(T), lanes);
  if (lanes == 8) launch_pdl(paper ? k_pass2<T, true, 8> : k_pass2<T, false, 8>, nblocks(8 * a.n, pt), pt, 0, s, a);
  else if (lanes == 4) launch_pdl(paper ? k_pass2<T, true, 4> : k_pass2<T, false, 4>, nblocks(4 * a.n, pt), pt, 0, s, a);
  else launch_pdl(paper ? k_pass2<T, true, 1> : k_pass2<T, false, 1>, nblocks(a.n, pt), pt, 0, s, a);
  if (a.det) {
    launch_pdl(k_blk_scan, 1, 1024, 0, s, a.blk_cnt, nblocks(a.n));
    launch_pdl(k_compact_det<T>, nblocks(a.n), kBlock, 0, s, a);
  }
}

template <typename T> void launch_csp_force(const Args<T>& a, cudaStream_t s) {
  launch_pdl(k_csp_force<T>, nblocks(a.n), kBlock, 0, s, a);
}

void launch_final(double* partials, int n_part, double* e_total, double* e_pot_slot,
                  const double* thermo_part, int n_tblocks, double* thermo_slot, int* flags,
                  const int* counts, int64_t* n_ace_out, int* cell_count, int ncell, double* scratch, int* ticket,
                  cudaStream_t s) {
  const int most = n_part > n_tblocks ? n_part : n_tblocks;
  const int grid = std::min(nblocks(most, kFinalThreads), kFinalBlocks);
  launch_pdl(k_final, grid, kFinalThreads, 0, s, partials, n_part, e_total, e_pot_slot, thermo_part, n_tblocks,
             thermo_slot, flags, counts, n_ace_out, cell_count, ncell, scratch, ticket);
}

template <typename T> void launch_verlet(const Args<T>& a, int mode, double* pos, double* vel,
                                         const double* force, const double* inv_mass, double dt,
                                         double* thermo_part, cudaStream_t s) {
  const bool th = mode != 0 && thermo_part != nullptr;
  auto k = mode == 0 ? k_verlet<T, 0, false>
                     : (mode == 1 ? (th ? k_verlet<T, 1, true> : k_verlet<T, 1, false>)
                                  : (th ? k_verlet<T, 2, true> : k_verlet<T, 2, false>));
  launch_pdl(k, nblocks(a.n), kBlock, 0, s, a, pos, vel, force, inv_mass, dt, 0.5 * dt, thermo_part);
}

template <typename T> void launch_get_field(const Args<T>& a, int field, void* dst, cudaStream_t s) {
  k_get_field<T><<<nblocks(a.n), kBlock, 0, s>>>(a, field, dst);
}

#define APIP_INST(T)                                                                              \
  template void launch_prep<T>(const Args<T>&, cudaStream_t);                                     \
  template void launch_neighbors<T>(const Args<T>&, int, cudaStream_t);                           \
  template void launch_pass1<T>(const Args<T>&, cudaStream_t);                                    \
  template void launch_pass2<T>(const Args<T>&, cudaStream_t);                                    \
  template void launch_fm_buffer<T>(const Args<T>&, cudaStream_t);                                \
  template void launch_csp_force<T>(const Args<T>&, cudaStream_t);                                \
  template void launch_verlet<T>(const Args<T>&, int, double*, double*, const double*,            \
                                 const double*, double, double*, cudaStream_t);                   \
  template void launch_get_field<T>(const Args<T>&, int, void*, cudaStream_t);
APIP_INST(double)
APIP_INST(float)
#undef APIP_INST

}  // namespace apip
