// md.cu -- MD-scale force call: one large periodic cell, one parameter set, neighbour rebuild by a
// cell list plus energy, forces and virial (Eq. 1-14 of arXiv:1909.11474), every call.
//
// Coordinates. Every atom's cell coordinate w = x H^-1 nc is split into its floor C and an in-cell
// coordinate u = w - C in [0, 1), and C into an integer wrap m and a cell index c (C = m nc + c). The
// atom is kept as its in-cell Cartesian position X = u E (FP32; E = the cell edge vectors H_k / nc_k
// as rows). A bond to an atom of a neighbouring cell (offset o in {-1,0,1}^3) is d = o E + (X_j - X_i),
// in FP32 and accurate to ~1e-6 A whatever the box size; its image shift is n = kw + m_i - m_j (kw =
// the periodic wrap of the neighbouring cell). Membership uses an FP32 distance (the search forms it from
// positions relative to a brick's centre) where it is farther than a rounding margin from R2, and the
// exact FP64 test of the batched build otherwise: every decision is the exact one, whatever the rounding,
// so the two atoms of a pair agree and the lists equal the batched build's bit for bit; they are sorted to
// the same (j, n) order. The force kernel's FP32 d of (j, i) is exactly the negation of that of (i, j).
#include <math.h>

#include <algorithm>
#include <cmath>
#include <string>

#include "batch_kernel.cuh"
#include "common.cuh"
#include "ctx.hpp"

namespace tsf {

constexpr int kMdCap = 16;    // atom slots per cell
constexpr int kMdMaxM = 8;    // neighbours per atom handled by the force kernel
constexpr int kMdThreads = 128;
constexpr int kMdForceAtoms = kMdThreads / 4;   // atoms per block of the FP64 force kernel (four lanes each)
// Bricks of the pair search: 4 x 4 x 6 interior cells (the third axis, along which cells are
// consecutive, the longest), and the cells around them
constexpr int kBX = 4, kBY = 4, kBZ = 6;
constexpr int kHX = kBX + 2, kHY = kBY + 2, kHZ = kBZ + 2;
constexpr int kHaloCells = kHX * kHY * kHZ;       // 288
constexpr int kBrickCells = kBX * kBY * kBZ;      // 96
constexpr int kStageCap = 1024;                   // halo atoms staged in shared memory
constexpr int kSearchThreads = 192;               // about the atoms of a brick of a solid
constexpr int kCandCap = 12;                      // candidates (r^2 below the band's upper edge) kept per atom

struct MdGeom {
  double H[9], Hinv[9];
  int nc[3];
  int diag;                   // H (and so H^-1) diagonal: cell coordinates need 3 products, not 9
  double Hn[9];               // H^-1 with column k scaled by nc_k: x Hn = cell coordinates
  float Hnh[9], Hnl[9];       // Hn as FP32 head + tail (Hn = Hnh + Hnl to ~2^-48 relative)
  float E[9];                 // cell edge vectors, row k = H_k / nc_k
  float cut2_lo, cut2_hi;     // FP32 decision band around R2^2
  float scan_cut;             // cut2_hi + the rounding of the search's distance filter
  double R1, R2, R2sq;
  double inv_w, fcp_k;        // 1 / (R2 - R1) and -pi / (2 (R2 - R1)) (Eq. 9)
  float R1f, R2f, inv_wf, fcp_kf;
};

// Cartesian vector of a separation v in cell units: v0 E_0 + v1 E_1 + v2 E_2.
__device__ __forceinline__ float3 md_cart(const MdGeom &G, float v0, float v1, float v2) {
  return make_float3(v0 * G.E[0] + v1 * G.E[3] + v2 * G.E[6], v0 * G.E[1] + v1 * G.E[4] + v2 * G.E[7],
                     v0 * G.E[2] + v1 * G.E[5] + v2 * G.E[8]);
}

// Cell of every atom; the cell's slots hold (X, atom index) so the search reads one record per
// candidate. An atom that gets no slot (non-finite position, full cell) gets cell index -1 and an
// empty list here; no other atom sees it, and the call is flagged. The search writes every other count.
//
// The cell coordinates w = x Hn are formed in FP32 head + tail arithmetic (products split exactly by
// FMA, sums by two-sum), accurate to ~2^-44 |w|; below |w| = 2^16 cells that is under the FP32 rounding
// of u itself. Other positions take FP64 arithmetic. The floor C is then that of head + tail, and
// u = w - C is rounded once to FP32: any consistent (C, u) serves the search and the bond vectors.
__device__ __forceinline__ void md_bin_atom(int i, double x, double y, double z, const MdGeom &G,
                                            int *__restrict__ cellcnt, float4 *__restrict__ cellx,
                                            float4 *__restrict__ x4, int4 *__restrict__ m4, int *cnt, unsigned *status) {
  float xh[3], xl[3];
  bool fast = split_f64(x, xh[0], xl[0]);
  fast = split_f64(y, xh[1], xl[1]) && fast;
  fast = split_f64(z, xh[2], xl[2]) && fast;
  int Ci[3];
  float uu[3];
  if (fast) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float wh, wl;
      if (G.diag) {
        const float a = G.Hnh[4 * k], b = G.Hnl[4 * k];
        const float p = xh[k] * a;
        wl = __fmaf_rn(xh[k], a, -p) + __fmaf_rn(xh[k], b, xl[k] * a);
        wh = p;
      } else {
        float p[3], q = 0.f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const float h = G.Hnh[3 * a + k], l = G.Hnl[3 * a + k];
          p[a] = xh[a] * h;
          q += __fmaf_rn(xh[a], h, -p[a]) + __fmaf_rn(xh[a], l, xl[a] * h);
        }
        float s1, t1, s2, t2;
        two_sum(p[0], p[1], s1, t1);
        two_sum(s1, p[2], s2, t2);
        wh = s2;
        wl = q + t1 + t2;
      }
      // normalise (|wl| <= ulp(wh) / 2), then C = floor(wh) + floor(frac(wh) + wl)
      float h2, t2;
      two_sum(wh, wl, h2, t2);
      wh = h2;
      wl = t2;
      fast = fast && fabsf(wh) < 65536.f;
      const float ch = floorf(wh);
      const float s = (wh - ch) + wl;
      const float cl = floorf(s);
      uu[k] = s - cl;
      Ci[k] = (int)ch + (int)cl;
    }
  }
  if (!fast) {
    // FP64 cell coordinates: w = s nc (nc folded into the inverse box), its floor C, u = w - C
    double w[3];
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      w[k] = G.diag ? (k == 0 ? x : (k == 1 ? y : z)) * G.Hn[4 * k]
                    : x * G.Hn[k] + y * G.Hn[3 + k] + z * G.Hn[6 + k];
      ok = ok && fabs(w[k]) < 1e9;                 // false for NaN and inf
    }
    if (!ok) {
      set_status(status, TERSOFF_STATUS_NONFINITE);
      x4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      m4[i] = make_int4(0, 0, 0, -1);
      cnt[i] = 0;
      return;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double C = floor(w[k]);
      uu[k] = (float)(w[k] - C);
      Ci[k] = (int)C;
    }
  }
  int mm[3], cc[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {   // the integer split C = m nc + c
    const int n = G.nc[k];
    const int m = Ci[k] >= 0 ? Ci[k] / n : -((n - 1 - Ci[k]) / n);
    mm[k] = m;
    cc[k] = Ci[k] - m * n;
  }
  const int cell = (cc[0] * G.nc[1] + cc[1]) * G.nc[2] + cc[2];
  const float3 X = md_cart(G, uu[0], uu[1], uu[2]);
  x4[i] = make_float4(X.x, X.y, X.z, 0.f);
  const int slot = atomicAdd(&cellcnt[cell], 1);
  if (slot < kMdCap) {
    // the record's index carries in its sign bit whether the atom has a nonzero wrap m (lies outside
    // the primary box), so that the search loads m only for those atoms
    const int tag = i | ((mm[0] | mm[1] | mm[2]) ? (int)0x80000000u : 0);
    cellx[cell * kMdCap + slot] = make_float4(X.x, X.y, X.z, __int_as_float(tag));
  } else {
    set_status(status, TERSOFF_STATUS_NBR_OVERFLOW);
    cnt[i] = 0;
  }
  m4[i] = make_int4(mm[0], mm[1], mm[2], slot < kMdCap ? cell : -1);
}
__global__ void md_cells_kernel(int N, const double *__restrict__ pos, const __grid_constant__ MdGeom G,
                                int *__restrict__ cellcnt, float4 *__restrict__ cellx,
                                float4 *__restrict__ x4, int4 *__restrict__ m4, int *__restrict__ cnt,
                                unsigned *status) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  pdl_trigger();   // every MD kernel lets the next one launch at once; each waits for its predecessor's end here
  pdl_wait();
  if (i < N) md_bin_atom(i, pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], G, cellcnt, cellx, x4, m4, cnt, status);
}

// Offset code of a neighbouring cell o in {-1,0,1}^3: (o0+1) << 4 | (o1+1) << 2 | (o2+1). The code of
// -o is 42 - code.
constexpr unsigned kOffNeg = 42u;

// FP32 separation d = o E + (X_j - X_i) of an atom j of the neighbouring cell with offset code `code`
// (the products o_k E_k are exact, the sums rounded in a fixed order), so the d of (j, i) is exactly
// the negation of that of (i, j).
__device__ __forceinline__ float3 md_sep(const MdGeom &G, unsigned code, float4 xi, float4 xj) {
  const float o0 = (float)((int)(code >> 4) - 1), o1 = (float)((int)((code >> 2) & 3u) - 1),
              o2 = (float)((int)(code & 3u) - 1);
  const float3 b = md_cart(G, o0, o1, o2);
  return make_float3(__fadd_rn(b.x, __fsub_rn(xj.x, xi.x)), __fadd_rn(b.y, __fsub_rn(xj.y, xi.y)),
                     __fadd_rn(b.z, __fsub_rn(xj.z, xi.z)));
}

// Periodic wrap of the coordinate a = c + o (o in {-1, 0, 1}) on an axis of n cells: -1, 0 or 1, and
// the wrapped coordinate g.
__device__ __forceinline__ int md_wrap(int a, int n, int &g) {
  if (a < 0) {
    g = a + n;
    return -1;
  }
  if (a >= n) {
    g = a - n;
    return 1;
  }
  g = a;
  return 0;
}

// Membership of a candidate at FP32 separation d: the FP32 distance decides outside the rounding band
// around R2^2, the exact FP64 test of the batched build inside it (image shift n = wrap + m_i - m_j),
// so that every decision is the exact one.
__device__ __forceinline__ bool md_pair_in(const MdGeom &G, const double *__restrict__ pos,
                                           const int4 *__restrict__ m4, int i, int j, int4 mi, int w0, int w1,
                                           int w2, float3 d) {
  const float r2 = __fmaf_rn(d.z, d.z, __fmaf_rn(d.y, d.y, __fmul_rn(d.x, d.x)));
  if (r2 > G.cut2_hi) return false;
  if (r2 < G.cut2_lo) return true;
  const int4 mj = m4[j];
  const ExactPair e = exact_pair(pos[3 * j], pos[3 * j + 1], pos[3 * j + 2], pos[3 * i], pos[3 * i + 1],
                                 pos[3 * i + 2], G.H, w0 + mi.x - mj.x, w1 + mi.y - mj.y, w2 + mi.z - mj.z);
  return e.r2 < G.R2sq;
}

// The full shell of atom i (cell index mi.w, in-cell position xi): every record of the 27 cells around
// its own but i's own is a candidate; visit(key) is called for each member, key = j << 6 | offset code.
// The shell runs as 9 rows (o0, o1) of three cells along the third axis, each row one loop over its
// cells' records in turn (so that the lanes of a warp diverge by row lengths, not cell by cell). The
// FP32 separation here is (o E - X_i) + X_j; any rounding within the band serves, since the band
// sends every near-cutoff candidate to the exact test.
template <typename Visit>
__device__ __forceinline__ void md_shell(const MdGeom &G, const double *__restrict__ pos,
                                         const int4 *__restrict__ m4, const int *__restrict__ cellcnt,
                                         const float4 *__restrict__ cellx, int i, int4 mi, float4 xi,
                                         Visit &&visit) {
  const int nc0 = G.nc[0], nc1 = G.nc[1], nc2 = G.nc[2];
  const int c2 = mi.w % nc2, c1 = (mi.w / nc2) % nc1, c0 = mi.w / (nc2 * nc1);
  int g2[3], w2[3];
#pragma unroll
  for (int o = 0; o < 3; ++o) w2[o] = md_wrap(c2 + o - 1, nc2, g2[o]);
#pragma unroll 1
  for (int ab = 0; ab < 9; ++ab) {
    const int a = ab / 3, b = ab - 3 * a;
    int g0, g1;
    const int w0 = md_wrap(c0 + a - 1, nc0, g0), w1 = md_wrap(c1 + b - 1, nc1, g1);
    const int row = (g0 * nc1 + g1) * nc2;
    const int n0 = min(cellcnt[row + g2[0]], kMdCap), n1 = min(cellcnt[row + g2[1]], kMdCap),
              n2 = min(cellcnt[row + g2[2]], kMdCap);
    // the row's offset o E for o2 = -1, less X_i; o2 = 0 and 1 add the third edge once and twice
    const float fa = (float)(a - 1), fb = (float)(b - 1);
    const float bx = fa * G.E[0] + fb * G.E[3] - G.E[6] - xi.x;
    const float by = fa * G.E[1] + fb * G.E[4] - G.E[7] - xi.y;
    const float bz = fa * G.E[2] + fb * G.E[5] - G.E[8] - xi.z;
    const int n01 = n0 + n1, T = n01 + n2;
    for (int q = 0; q < T; ++q) {
      const int c = q < n0 ? 0 : (q < n01 ? 1 : 2);
      const int slot = q - (c == 0 ? 0 : (c == 1 ? n0 : n01));
      const float4 r = cellx[(size_t)(row + g2[c]) * kMdCap + slot];
      const int j = __float_as_int(r.w) & 0x7fffffff;
      const float fc = (float)c;
      const float dx = __fadd_rn(__fmaf_rn(fc, G.E[6], bx), r.x);
      const float dy = __fadd_rn(__fmaf_rn(fc, G.E[7], by), r.y);
      const float dz = __fadd_rn(__fmaf_rn(fc, G.E[8], bz), r.z);
      if (j != i && md_pair_in(G, pos, m4, i, j, mi, w0, w1, w2[c], make_float3(dx, dy, dz)))
        visit(((unsigned)j << 6) | (unsigned)((a << 4) | (b << 2) | c));
    }
  }
}

// Keys of the lists while a thread collects them: j << 7 | offset code << 1 | (partner j has a nonzero wrap m), which
// orders as (j, code) does (an entry's two keys differ above the mark).
__device__ __forceinline__ unsigned md_sort_key(unsigned key, bool wrapped) { return (key << 1) | (wrapped ? 1u : 0u); }

// key into the ascending list k[0 .. kMdMaxM - 1] (free places ~0u): one compare-exchange a place, no branches.
__device__ __forceinline__ void md_insert(unsigned (&k)[kMdMaxM], unsigned key) {
#pragma unroll
  for (int e = 0; e < kMdMaxM; ++e) {
    const unsigned lo = min(k[e], key);
    key = max(k[e], key);
    k[e] = lo;
  }
}

// List entry (j, n) of sort key `key` of atom i (wraps m_i, cell (c0, c1, c2)): n = wrap + m_i - m_j (m_j is loaded only
// where the mark is set). plain: no wrap anywhere near and m_i = 0, so that n = -m_j.
__device__ __forceinline__ void md_write_entry(const MdGeom &G, const int4 *__restrict__ m4, int4 mi, int c0, int c1,
                                               int c2, bool plain, unsigned key, size_t at, int *__restrict__ nbr,
                                               char4 *__restrict__ shift) {
  const int j = (int)(key >> 7);
  int n0 = 0, n1 = 0, n2 = 0;
  if (!plain) {
    int g;
    n0 = md_wrap(c0 + (int)((key >> 5) & 3u) - 1, G.nc[0], g) + mi.x;
    n1 = md_wrap(c1 + (int)((key >> 3) & 3u) - 1, G.nc[1], g) + mi.y;
    n2 = md_wrap(c2 + (int)((key >> 1) & 3u) - 1, G.nc[2], g) + mi.z;
  }
  if (key & 1u) {
    const int4 mj = m4[j];
    n0 -= mj.x;
    n1 -= mj.y;
    n2 -= mj.z;
  }
  nbr[at] = j;
  shift[at] = make_char4((signed char)n0, (signed char)n1, (signed char)n2, 0);
}

// The list of atom i from its members' sorted keys k (count of them; at most kMdMaxM kept): the count, the keys into the
// rows of `keys` and the entries (j, n) into the lists. (With at most one image of any j, plane spacings of at least
// 3 R2, the key order is the (j, n) order.)
__device__ __forceinline__ void md_emit(int N, int M, int i, int4 mi, int c0, int c1, int c2, bool plain, const MdGeom &G,
                                        const int4 *__restrict__ m4, const unsigned (&k)[kMdMaxM], int count,
                                        int *__restrict__ cnt, unsigned *__restrict__ keys, int *__restrict__ nbr,
                                        char4 *__restrict__ shift, unsigned *status) {
  cnt[i] = count;
  if (count > M) set_status(status, TERSOFF_STATUS_NBR_OVERFLOW);
  const int cm = min(count, M);
#pragma unroll
  for (int e = 0; e < kMdMaxM; ++e)
    if (e < cm) {
      keys[(size_t)e * N + i] = k[e] >> 1;
      md_write_entry(G, m4, mi, c0, c1, c2, plain, k[e], (size_t)e * N + i, nbr, shift);
    }
}

// The whole search of atom i from the cell arrays in global memory (md_shell): the path of bricks
// whose surroundings exceed the stage and of atoms with more than kMdMaxM members. Such an atom
// enumerates its shell a second time, keeps the first M members found in its row of `keys` and
// writes each at its rank among them (the row itself stays in the order found: the force kernel
// flags the atom and gives it no forces).
__device__ __noinline__ void md_search_atom(int N, int M, int i, const double *__restrict__ pos, const MdGeom &G,
                                               const float4 *__restrict__ x4, const int4 *__restrict__ m4,
                                               const int *__restrict__ cellcnt, const float4 *__restrict__ cellx,
                                               int *__restrict__ cnt, unsigned *__restrict__ keys,
                                               int *__restrict__ nbr, char4 *__restrict__ shift, unsigned *status) {
  const int4 mi = m4[i];
  const float4 xi = x4[i];
  const int nc2 = G.nc[2], nc1 = G.nc[1];
  const int c2 = mi.w % nc2, c1 = (mi.w / nc2) % nc1, c0 = mi.w / (nc2 * nc1);
  unsigned k[kMdMaxM];
#pragma unroll
  for (int u = 0; u < kMdMaxM; ++u) k[u] = 0xffffffffu;
  int count = 0;
  md_shell(G, pos, m4, cellcnt, cellx, i, mi, xi, [&](unsigned key) {
    md_insert(k, md_sort_key(key, true));          // the partner's m is loaded
    ++count;
  });
  if (count <= kMdMaxM) {
    md_emit(N, M, i, mi, c0, c1, c2, false, G, m4, k, count, cnt, keys, nbr, shift, status);
    return;
  }
  cnt[i] = count;
  if (count > M) set_status(status, TERSOFF_STATUS_NBR_OVERFLOW);
  const int cm = min(count, M);
  int p = 0;
  md_shell(G, pos, m4, cellcnt, cellx, i, mi, xi, [&](unsigned key) {
    if (p < M) keys[(size_t)p * N + i] = key;
    ++p;
  });
  for (int e = 0; e < cm; ++e) {
    const unsigned key = keys[(size_t)e * N + i];
    int rank = 0;
    for (int f = 0; f < cm; ++f) rank += keys[(size_t)f * N + i] < key ? 1 : 0;
    md_write_entry(G, m4, mi, c0, c1, c2, false, md_sort_key(key, true), (size_t)rank * N + i, nbr, shift);
  }
}

// Neighbour lists by bricks of 4x4x6 cells, full shell, no atomics: a CTA stages the records of its brick and of the
// cells around it (6x6x8) in shared memory, as positions x from the brick's centre with q = |x|^2, two records a pair
// of 16-byte words, so that one atom's test of a pair is two loads and four packed FP32 operations:
//   t = q_j + (|x_i|^2 - c) - 2 x_i . x_j = |x_j - x_i|^2 - c,   c = G.scan_cut, above the rounding band's upper edge by
// what bounds the rounding of t (a filter: it decides nothing but which records are looked at). One thread per atom of
// the brick tests the 9 rows (o0, o1) of its shell; the three cells of a row lie consecutively in the stage, so a row is
// one run of records, taken in blocks of four pairs: the sign bits of t are shifted into a word, whose set bits give the
// candidates. Members (FP32 below the band, the exact test in it) are inserted into a sorted list in registers as they
// are found. The scan is bound by instruction issue: tested a record at a time from three coordinate arrays and
// appended to a list without branches it took ~26 instructions a pair where this takes ~10 (67.8 -> 62 us for
// 512,000 atoms, 52.9 M -> 39.7 M warp instructions); what bounds it now is the shared-memory pipe (504 wavefronts a
// warp, 55 % of the time) and the latency of the staging phases. A brick whose surroundings hold more than kStageCap atoms, and an atom with more than kCandCap
// candidates or kMdMaxM members, take the global-memory path (md_search_atom).
__global__ void __launch_bounds__(kSearchThreads, 5) md_search_kernel(
    int N, int M, const double *__restrict__ pos, const __grid_constant__ MdGeom G, const float4 *__restrict__ x4,
    const int4 *__restrict__ m4, const int *__restrict__ cellcnt, const float4 *__restrict__ cellx,
    int *__restrict__ cnt, unsigned *__restrict__ keys, int *__restrict__ nbr, char4 *__restrict__ shift,
    unsigned *status) {
  // pair p of records (2p, 2p + 1): (x, x', y, y') and (z, z', q, q'); a block of four pairs may reach past the last
  __shared__ __align__(16) float4 s_xy[kStageCap / 2 + 4], s_zq[kStageCap / 2 + 4];
  __shared__ int s_sj[kStageCap];   // atom index; sign bit: a nonzero wrap m
  __shared__ unsigned char s_code[kStageCap];       // 16 h0 + 4 h1 + h2 of each staged record's halo cell
  __shared__ unsigned s_int[kStageCap];             // the brick's own atoms, cell by cell: staged record | halo cell << 16
  // candidates of each thread, [u][tid]
  __shared__ unsigned short s_cand[kCandCap * kSearchThreads];
  __shared__ int s_cnt[kHaloCells], s_start[kHaloCells + 1], s_gcell[kHaloCells];
  __shared__ int s_ipre[kBrickCells + 1];
  const int tid = threadIdx.x, lane = tid & 31;
  const int nb2 = (G.nc[2] + kBZ - 1) / kBZ, nb1 = (G.nc[1] + kBY - 1) / kBY;
  const int o0 = (blockIdx.x / (nb2 * nb1)) * kBX, o1 = ((blockIdx.x / nb2) % nb1) * kBY,
            o2 = (blockIdx.x % nb2) * kBZ;   // first interior cell of the brick
  // a brick none of whose halo cells lies beyond a face: no periodic wrap in any of its bonds
  const bool inside = o0 > 0 && o1 > 0 && o2 > 0 && o0 + kBX < G.nc[0] && o1 + kBY < G.nc[1] && o2 + kBZ < G.nc[2];
  pdl_trigger();
  pdl_wait();
  // 1. counts of the halo cells; a halo cell beyond nc is next to no interior cell and stays empty
  for (int h = tid; h < kHaloCells; h += kSearchThreads) {
    const int h0 = h / (kHY * kHZ), h1 = (h / kHZ) % kHY, h2 = h % kHZ;
    const int c0 = o0 + h0 - 1, c1 = o1 + h1 - 1, c2 = o2 + h2 - 1;
    int n = 0, g = 0;
    if (c0 <= G.nc[0] && c1 <= G.nc[1] && c2 <= G.nc[2]) {
      int g0, g1, g2;
      md_wrap(c0, G.nc[0], g0);
      md_wrap(c1, G.nc[1], g1);
      md_wrap(c2, G.nc[2], g2);
      g = (g0 * G.nc[1] + g1) * G.nc[2] + g2;
      n = min(cellcnt[g], kMdCap);
    }
    s_cnt[h] = n;
    s_gcell[h] = g;
  }
  __syncthreads();
  // 2. exclusive sums over the halo cells (warp 0, 9 per lane) and over the interior cells (warp 1, 3 per lane)
  static_assert(kHaloCells == 9 * 32 && kBrickCells == 3 * 32, "the scans map 9 and 3 cells onto each lane");
  if (tid < 32) {
    int a[9], tot = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      a[k] = s_cnt[9 * lane + k];
      tot += a[k];
    }
    int inc = tot;
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, off);
      if (lane >= off) inc += v;
    }
    int run = inc - tot;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      s_start[9 * lane + k] = run;
      run += a[k];
    }
    if (lane == 31) s_start[kHaloCells] = inc;
  } else if (tid < 64) {
    int b[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int q = 3 * lane + k, q0 = q / (kBY * kBZ), q1 = (q / kBZ) % kBY, q2 = q % kBZ;
      const bool in = o0 + q0 < G.nc[0] && o1 + q1 < G.nc[1] && o2 + q2 < G.nc[2];
      b[k] = in ? s_cnt[((q0 + 1) * kHY + q1 + 1) * kHZ + q2 + 1] : 0;
    }
    const int t2 = b[0] + b[1] + b[2];
    int inc2 = t2;
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc2, off);
      if (lane >= off) inc2 += v;
    }
    s_ipre[3 * lane] = inc2 - t2;
    s_ipre[3 * lane + 1] = inc2 - t2 + b[0];
    s_ipre[3 * lane + 2] = inc2 - t2 + b[0] + b[1];
    if (lane == 31) s_ipre[kBrickCells] = inc2;
  }
  __syncthreads();
  // 3. stage the records, one thread per halo cell (its first four records loaded together)
  const int total = s_start[kHaloCells], A = s_ipre[kBrickCells];
  const bool staged = total <= kStageCap;
  if (staged) {
    for (int h = tid; h < kHaloCells; h += kSearchThreads) {
      const int n = s_cnt[h];
      if (n == 0) continue;
      const int h0 = h / (kHY * kHZ), h1 = (h / kHZ) % kHY, h2 = h % kHZ;
      // the halo cell's offset from the brick's centre
      const float3 B = md_cart(G, (float)h0 - 0.5f * kHX, (float)h1 - 0.5f * kHY, (float)h2 - 0.5f * kHZ);
      const float4 *src = cellx + (size_t)s_gcell[h] * kMdCap;
      const int t0 = s_start[h];
      const int q0 = h0 - 1, q1 = h1 - 1, q2 = h2 - 1;
      const bool own = q0 >= 0 && q0 < kBX && q1 >= 0 && q1 < kBY && q2 >= 0 && q2 < kBZ && o0 + q0 < G.nc[0] &&
                       o1 + q1 < G.nc[1] && o2 + q2 < G.nc[2];
      const int i0 = own ? s_ipre[(q0 * kBY + q1) * kBZ + q2] : 0;
      auto put = [&](int q, const float4 &v) {
        const int t = t0 + q;
        const float x = B.x + v.x, y = B.y + v.y, z = B.z + v.z;
        float *xy = reinterpret_cast<float *>(s_xy) + 4 * (t >> 1) + (t & 1);
        float *zq = reinterpret_cast<float *>(s_zq) + 4 * (t >> 1) + (t & 1);
        xy[0] = x;
        xy[2] = y;
        zq[0] = z;
        zq[2] = x * x + y * y + z * z;
        s_sj[t] = __float_as_int(v.w);
        s_code[t] = (unsigned char)(16 * h0 + 4 * h1 + h2);
        if (own) s_int[i0 + q] = (unsigned)t | (unsigned)h << 16;
      };
      float4 r[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < n) r[q] = src[q];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < n) put(q, r[q]);
      for (int q = 4; q < n; ++q) put(q, src[q]);
    }
  }
  __syncthreads();
  // 4. one thread per atom of the brick
  for (int a = tid; a < A; a += kSearchThreads) {
    if (!staged) {
      int k = 0;                                   // interior cell of atom a
      for (int step = 64; step > 0; step >>= 1)
        if (k + step < kBrickCells && s_ipre[k + step] <= a) k += step;
      const int hi = ((k / (kBY * kBZ) + 1) * kHY + (k / kBZ) % kBY + 1) * kHZ + k % kBZ + 1;
      const int i = __float_as_int(cellx[(size_t)s_gcell[hi] * kMdCap + a - s_ipre[k]].w) & 0x7fffffff;
      md_search_atom(N, M, i, pos, G, x4, m4, cellcnt, cellx, cnt, keys, nbr, shift, status);
      continue;
    }
    const unsigned own = s_int[a];                 // staged record and halo cell of the atom
    const int slot = (int)(own & 0xffffu), hi = (int)(own >> 16), code = s_code[slot];
    const float *xyi = reinterpret_cast<const float *>(s_xy) + 4 * (slot >> 1) + (slot & 1);
    const float *zqi = reinterpret_cast<const float *>(s_zq) + 4 * (slot >> 1) + (slot & 1);
    const float xi = xyi[0], yi = xyi[2], zi = zqi[0];
    const int itag = s_sj[slot], i = itag & 0x7fffffff;
    const float2 ax = f2(-2.f * xi), ay = f2(-2.f * yi), az = f2(-2.f * zi), ac = f2(zqi[2] - G.scan_cut);
    int nc = 0;
#pragma unroll 1
    for (int ab = 0; ab < 9; ++ab) {
      const int ra = ab / 3, rb = ab - 3 * ra;
      const int hc = hi + ((ra - 1) * kHY + (rb - 1)) * kHZ;   // the row's middle cell
      const int p0 = s_start[hc - 1], pend = s_start[hc + 2];
      for (int kb = p0 >> 1; 2 * kb < pend; kb += 4) {
        unsigned w = 0;                            // sign bits of the block's eight records, the first one on top
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 u = s_xy[kb + q], v = s_zq[kb + q];
          float2 t = __fadd2_rn(make_float2(v.z, v.w), ac);
          t = __ffma2_rn(make_float2(u.x, u.y), ax, t);
          t = __ffma2_rn(make_float2(u.z, u.w), ay, t);
          t = __ffma2_rn(make_float2(v.x, v.y), az, t);
          w = __funnelshift_l(__float_as_uint(t.x), w, 1);
          w = __funnelshift_l(__float_as_uint(t.y), w, 1);
        }
        // the records of the run only: first .. last of the block's eight
        const int first = max(p0 - 2 * kb, 0), last = min(pend - 2 * kb, 8);
        unsigned hits = w & (0xffu >> first) & (0xff00u >> last);
        while (hits) {
          const int bit = 31 - __clz(hits);
          hits ^= 1u << bit;
          if (nc < kCandCap) s_cand[nc * kSearchThreads + tid] = (unsigned short)(2 * kb + 7 - bit);
          ++nc;
        }
      }
    }
    if (nc > kCandCap) {
      md_search_atom(N, M, i, pos, G, x4, m4, cellcnt, cellx, cnt, keys, nbr, shift, status);
      continue;
    }
    // members among the candidates: the FP32 distance decides below the band, the exact test in it
    const int4 mi = itag < 0 ? m4[i] : make_int4(0, 0, 0, 0);
    const int k0 = hi / (kHY * kHZ) - 1, k1 = (hi / kHZ) % kHY - 1, k2 = hi % kHZ - 1;
    const int c0 = o0 + k0, c1 = o1 + k1, c2 = o2 + k2;
    const int ci = code - (16 + 4 + 1);            // code of the shell's first cell: j's less it is its offset code
    unsigned kk[kMdMaxM];
#pragma unroll
    for (int u = 0; u < kMdMaxM; ++u) kk[u] = 0xffffffffu;
    int count = 0;
    for (int u = 0; u < nc; ++u) {
      const int p = s_cand[u * kSearchThreads + tid];
      if (p == slot) continue;
      const float *xyj = reinterpret_cast<const float *>(s_xy) + 4 * (p >> 1) + (p & 1);
      const float dx = __fsub_rn(xyj[0], xi), dy = __fsub_rn(xyj[2], yi),
                  dz = __fsub_rn(reinterpret_cast<const float *>(s_zq)[4 * (p >> 1) + (p & 1)], zi);
      const int jtag = s_sj[p], j = jtag & 0x7fffffff;
      const unsigned oc = (unsigned)((int)s_code[p] - ci);   // 16 (d0 + 1) + 4 (d1 + 1) + (d2 + 1)
      const float r2 = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
      bool in = r2 < G.cut2_lo;
      if (!in && r2 <= G.cut2_hi) {   // in the rounding band: the exact test, with the neighbouring cell's periodic wrap
        int g;
        const int w0 = md_wrap(c0 + (int)(oc >> 4) - 1, G.nc[0], g), w1 = md_wrap(c1 + (int)((oc >> 2) & 3u) - 1, G.nc[1], g),
                  w2 = md_wrap(c2 + (int)(oc & 3u) - 1, G.nc[2], g);
        in = md_pair_in(G, pos, m4, i, j, mi, w0, w1, w2, make_float3(dx, dy, dz));
      }
      if (in) {
        md_insert(kk, md_sort_key(((unsigned)j << 6) | oc, jtag < 0));
        ++count;
      }
    }
    if (count > kMdMaxM) {
      md_search_atom(N, M, i, pos, G, x4, m4, cellcnt, cellx, cnt, keys, nbr, shift, status);
      continue;
    }
    md_emit(N, M, i, mi, c0, c1, c2, inside && itag >= 0, G, m4, kk, count, cnt, keys, nbr, shift, status);
  }
}

// Fixed-order block sum of n values per quantity, src[k * stride + q] (q < n, k < K): a strided sum
// per thread (loads in flight together), a butterfly over each warp's lanes, then the warps in order
// (through `red`, [warps][8]); thread k < K returns quantity k.
template <int K, int TH>
__device__ __forceinline__ double md_block_sum(const double *src, size_t stride, int n, double (*red)[8]) {
  const int tid = threadIdx.x;
  double acc[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    acc[k] = 0.0;
#pragma unroll 4
    for (int q = tid; q < n; q += TH) acc[k] += __ldcg(&src[k * stride + q]);
    for (int off = 16; off > 0; off >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], off);
  }
  __syncthreads();                                 // earlier readers of red are done
  if ((tid & 31) == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) red[tid >> 5][k] = acc[k];
  __syncthreads();
  double s = 0.0;
  if (tid < K)
    for (int w = 0; w < TH / 32; ++w) s += red[w][tid];
  return s;
}

// Deterministic in-kernel sum of per-block partials [K][nblk] (FP64; blocks of TH threads): the last block of each
// group of md_group(nblk) blocks to finish sums its group into [K][ngroups], and the last group to finish sums the
// groups, both in a fixed order; quantity 0 goes to *out0 and quantity k >= 1 to out_rest[k - 1]. Up to 256 blocks are
// one group, whose sum is the result (an NVE step with one level against groups of 64: FP32 at 108, 172 and 256 blocks
// 35.0, 42.0 and 47.7 us against 40.4, 45.6 and 51.0; FP64 at 128 and 250 blocks 41.9 and 56.3 against 45.4 and 57.4).
// Beyond 256 neither is the better one throughout: one level took 3.8 us off a step at 365 blocks and 2.3 at 1,024, and
// added 1.5 at 432 and 3.0 at 1,458; 666 and 977 within 2 us. The group sums
// follow the partials; the counters [ngroups + 1] are zero before the launch and left zero by it. The threads that
// wrote the block's partials have fenced before the call.
__host__ __device__ inline int md_group(int nblk) { return nblk <= 256 ? 256 : 64; }
__host__ __device__ inline int md_ngroups(int nblk) { return (nblk + md_group(nblk) - 1) / md_group(nblk); }
template <int K, int TH>
__device__ __forceinline__ void md_grouped_sum(double *partial, unsigned *counter, int nblk, int b, double *out0,
                                               double *out_rest, double (*red)[8]) {
  __shared__ int s_last;
  const int tid = threadIdx.x, gsz = md_group(nblk), ngroups = md_ngroups(nblk);
  double *gpart = partial + (size_t)K * nblk;
  const int g = b / gsz, g0 = g * gsz, gn = min(gsz, nblk - g0);
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&counter[g], 1u) == (unsigned)(gn - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (tid == 0) counter[g] = 0u;                   // no block of the group is left to count
  double t = md_block_sum<K, TH>(partial + g0, (size_t)nblk, gn, red);
  if (ngroups > 1) {
    if (tid < K) {
      gpart[(size_t)tid * ngroups + g] = t;
      __threadfence();
    }
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&counter[ngroups], 1u) == (unsigned)(ngroups - 1);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid == 0) counter[ngroups] = 0u;
    t = md_block_sum<K, TH>(gpart, (size_t)ngroups, ngroups, red);
  }
  if (tid == 0) *out0 = t;
  else if (tid < K) out_rest[tid - 1] = t;
}

// Bytes of the partial-sum area of K quantities over nblk blocks: partials, group sums, counters.
inline size_t md_sum_bytes(int K, int nblk) {
  const int ngroups = md_ngroups(nblk);
  return ((size_t)nblk + ngroups) * K * sizeof(double) + (ngroups + 1) * sizeof(unsigned);
}
inline size_t md_counter_offset(int K, int nblk) {
  const int ngroups = md_ngroups(nblk);
  return ((size_t)nblk + ngroups) * K * sizeof(double);
}

// Slot of the reverse entry of key (j << 6 | offset code) of atom i: rank * N + j, the rank of
// (i, -o) among j's keys being its place in j's sorted list; -1 when j's list is not handled (more
// than kMdMaxM entries: flagged by the force kernel) or does not hold it (a truncated list: flagged).
__device__ __forceinline__ int md_reverse_slot(int N, int M, int i, unsigned key, const int *__restrict__ cnt,
                                               const unsigned *__restrict__ keys, unsigned *status) {
  const int j = (int)(key >> 6);
  // the partner's first four keys are loaded beside its count, not after it (entries past the count
  // are ignored below)
  unsigned q[kMdMaxM];
#pragma unroll
  for (int f = 0; f < 4; ++f) q[f] = f < M ? keys[(size_t)f * N + j] : 0xffffffffu;
  const int cj = cnt[j];
  if (cj > kMdMaxM) return -1;
  const int cjm = min(cj, M);
#pragma unroll
  for (int f = 4; f < kMdMaxM; ++f) q[f] = f < cjm ? keys[(size_t)f * N + j] : 0xffffffffu;
  const unsigned want = ((unsigned)i << 6) | (kOffNeg - (key & 63u));
  int rank = 0;
  bool found = false;
#pragma unroll
  for (int f = 0; f < kMdMaxM; ++f)
    if (f < cjm) {
      rank += q[f] < want ? 1 : 0;
      found = found || q[f] == want;
    }
  if (!found) {
    set_status(status, TERSOFF_STATUS_NBR_OVERFLOW);
    return -1;
  }
  return rank * N + j;
}

// Passes 1-2 of one atom per thread, M = the warp's largest neighbour count; bonds e >= m of this
// thread are phantoms (f_C = f_C' = 0, unit vector 0), which contribute exactly zero.
template <int M>
__device__ __forceinline__ void md_atom(const float (&ux)[M], const float (&uy)[M], const float (&uz)[M], const float (&r)[M],
                                        const float (&ir)[M], const float (&fc)[M], const float (&fcp)[M],
                                        const PConsts<float> &K, float &U, float (&Wv)[6], float (&Px)[M], float (&Py)[M],
                                        float (&Pz)[M]) {
  constexpr int NP = M * (M - 1) / 2;
  float cs[NP > 0 ? NP : 1], tq[NP > 0 ? NP : 1];
  float fR[M], fA[M], zeta[M];
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const float x = ex2((r[j] - K.k0) * K.k1);   // r - r0 exact in FP32 near r0
    const float Dx = K.D0 * x;
    fR[j] = Dx * x;
    fA[j] = Dx + Dx;
    zeta[j] = 0.f;
  }
  {
    int q = 0;
#pragma unroll
    for (int j = 0; j < M; ++j)
#pragma unroll
      for (int k = j + 1; k < M; ++k) {
        cs[q] = ux[j] * ux[k] + uy[j] * uy[k] + uz[j] * uz[k];
        const float u = cs[q] - K.h;
        const float t = K.beta * u;
        const float g = t * u;
        tq[q] = t;
        zeta[j] += fc[k] * g;
        zeta[k] += fc[j] * g;
        ++q;
      }
  }
  float cc[M], rad[M];
#pragma unroll
  for (int j = 0; j < M; ++j) {
    float b, bp;
    bond_order(zeta[j], K, b, bp);
    const float e = fR[j] - b * fA[j];
    U += 0.5f * fc[j] * e;
    cc[j] = -0.5f * fc[j] * fA[j] * bp;
    const float de = 2.f * K.mha * (fR[j] + e);    // f_R' - b f_A' = -alpha (f_R + e)
    rad[j] = 0.5f * (fcp[j] * e + fc[j] * de);
  }
  float Ax[M], Ay[M], Az[M], s[M], Rg[M];
#pragma unroll
  for (int j = 0; j < M; ++j) {
    Ax[j] = 0.f; Ay[j] = 0.f; Az[j] = 0.f; s[j] = 0.f; Rg[j] = 0.f;
  }
  {
    int q = 0;
#pragma unroll
    for (int j = 0; j < M; ++j)
#pragma unroll
      for (int k = j + 1; k < M; ++k) {
        const float w = (cc[j] * fc[k] + cc[k] * fc[j]) * tq[q];
        Ax[j] += w * ux[k]; Ay[j] += w * uy[k]; Az[j] += w * uz[k];
        Ax[k] += w * ux[j]; Ay[k] += w * uy[j]; Az[k] += w * uz[j];
        const float wc = w * cs[q];
        s[j] += wc;
        s[k] += wc;
        const float g = tq[q] * (cs[q] - K.h);
        Rg[j] += cc[k] * g;
        Rg[k] += cc[j] * g;
        ++q;
      }
  }
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const float ir2 = ir[j] + ir[j];
    const float coef = rad[j] + fcp[j] * Rg[j] - s[j] * ir2;
    Px[j] = coef * ux[j] + ir2 * Ax[j];
    Py[j] = coef * uy[j] + ir2 * Ay[j];
    Pz[j] = coef * uz[j] + ir2 * Az[j];
    const float dx = r[j] * ux[j], dy = r[j] * uy[j], dz = r[j] * uz[j];
    Wv[0] -= dx * Px[j]; Wv[1] -= dy * Py[j]; Wv[2] -= dz * Pz[j];
    Wv[3] -= dx * Py[j]; Wv[4] -= dy * Pz[j]; Wv[5] -= dz * Px[j];
  }
}

// FP32, a thread an atom. Passes 1-2 of atom i (m entries) with arrays for M >= m bonds (Mw = the warp's largest
// count): the bond geometry (the search's separation), md_atom, and the P_ij of every entry: summed over the entries in order into Fo (atom i's own part of F_i), and stored
// at the reverse entry's slot (rank, j) of Prev, so that the gather reads atom i's rows in order.
template <int Mw>
__device__ __forceinline__ void md_force_atom(int N, int M, int i, int m, const MdGeom &G, const PConsts<float> &K,
                                              const float4 *__restrict__ x4, const unsigned *__restrict__ keys,
                                              const int *__restrict__ cnt, float4 xi, float4 *__restrict__ Prev,
                                              unsigned *status, float &U, float (&Wv)[6], float (&Fo)[3]) {
  constexpr int M_ = Mw;
  float ux[M_], uy[M_], uz[M_], r[M_], ir[M_], fc[M_], fcp[M_];
  int rs[M_];
#pragma unroll
  for (int e = 0; e < M_; ++e) {
    ux[e] = 0.f; uy[e] = 0.f; uz[e] = 0.f; r[e] = 1.f; ir[e] = 0.f; fc[e] = 0.f; fcp[e] = 0.f;
    rs[e] = -1;
    if (e < m) {
      const unsigned key = keys[(size_t)e * N + i];
      rs[e] = md_reverse_slot(N, M, i, key, cnt, keys, status);
      // the search's FP32 separation: neighbouring-cell offset and in-cell positions
      const float3 d = md_sep(G, key & 63u, xi, x4[key >> 6]);
      const float dx = d.x, dy = d.y, dz = d.z;
      const float rr = sqrtf(dx * dx + dy * dy + dz * dz);
      ir[e] = 1.f / rr;
      r[e] = rr;
      ux[e] = dx * ir[e];
      uy[e] = dy * ir[e];
      uz[e] = dz * ir[e];
      if (rr <= G.R1f) {
        fc[e] = 1.f;
      } else if (rr < G.R2f) {
        const float w = (rr - G.R1f) * G.inv_wf;
        fc[e] = 0.5f * (1.f + cospif(w));
        fcp[e] = G.fcp_kf * sinpif(w);
      }
    }
  }
  float Px[M_], Py[M_], Pz[M_];
  md_atom<M_>(ux, uy, uz, r, ir, fc, fcp, K, U, Wv, Px, Py, Pz);
#pragma unroll
  for (int e = 0; e < M_; ++e)
    if (e < m) {
      Fo[0] += Px[e];
      Fo[1] += Py[e];
      Fo[2] += Pz[e];
      if (rs[e] >= 0) Prev[rs[e]] = make_float4(Px[e], Py[e], Pz[e], 0.f);
    }
}

// The same for the long lists (5-8 entries) as a called function: its many live values do not raise
// the register count of the kernel, which the short lists of solids need.
struct MdSums {
  float U, W[6], F[3];
};
template <int Mw>
__device__ __noinline__ MdSums md_force_atom_long(int N, int M, int i, int m, const MdGeom &G,
                                                     const PConsts<float> &K, const float4 *__restrict__ x4, const unsigned *__restrict__ keys,
                                                     const int *__restrict__ cnt, float4 xi,
                                                 float4 *__restrict__ Prev, unsigned *status) {
  MdSums o;
  o.U = 0.f;
#pragma unroll
  for (int k = 0; k < 6; ++k) o.W[k] = 0.f;
  o.F[0] = o.F[1] = o.F[2] = 0.f;
  md_force_atom<Mw>(N, M, i, m, G, K, x4, keys, cnt, xi, Prev, status, o.U, o.W, o.F);
  return o;
}

__global__ void __launch_bounds__(kMdThreads, 8) md_force_kernel(
    int N, int M, const MdGeom G, const PConsts<float> K, const float4 *__restrict__ x4,
    const unsigned *__restrict__ keys, const int *__restrict__ cnt, float4 *__restrict__ Fown, float4 *__restrict__ Prev,
    double *__restrict__ partial, unsigned *counters, double *__restrict__ E, double *__restrict__ W,
    int *__restrict__ zero_cells, int ncells, unsigned *status) {
  __shared__ double red[kMdThreads / 32][8];
  const int i = blockIdx.x * kMdThreads + threadIdx.x;
  const bool valid = i < N;
  pdl_trigger();
  pdl_wait();
  // NVE steps: the cell counts, last read by the search before this kernel, are zeroed for the next step's binning
  if (zero_cells)
    for (int c = i; c < ncells; c += (int)(gridDim.x * kMdThreads)) zero_cells[c] = 0;
  int m = valid ? min(cnt[i], M) : 0;   // a truncated list (count > M) is flagged; its row holds M entries
  if (m > kMdMaxM) {
    set_status(status, TERSOFF_STATUS_MANY_NBRS);
    m = 0;
  }
  float4 xi = make_float4(0.f, 0.f, 0.f, 0.f);
  if (valid) xi = x4[i];
  float U = 0.f, Wv[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, Fo[3] = {0.f, 0.f, 0.f};
  // arrays sized by the warp's largest neighbour count, so that the common short lists keep few
  // values live
  const int Mw = __reduce_max_sync(0xffffffffu, (unsigned)m);
  switch (Mw) {
#define TSF_MDCASE(MM) \
    case MM: md_force_atom<MM>(N, M, i, m, G, K, x4, keys, cnt, xi, Prev, status, U, Wv, Fo); break;
#define TSF_MDLONG(MM)                                                                      \
    case MM: {                                                                              \
      const MdSums o = md_force_atom_long<MM>(N, M, i, m, G, K, x4, keys, cnt, xi, Prev, status); \
      U = o.U;                                                                              \
      for (int k = 0; k < 6; ++k) Wv[k] = o.W[k];                                           \
      for (int k = 0; k < 3; ++k) Fo[k] = o.F[k];                                           \
      break;                                                                                \
    }
    TSF_MDCASE(1) TSF_MDCASE(2) TSF_MDCASE(3) TSF_MDCASE(4) TSF_MDLONG(5) TSF_MDLONG(6) TSF_MDLONG(7)
    TSF_MDLONG(8)
#undef TSF_MDCASE
#undef TSF_MDLONG
    default: break;
  }
  if (valid) {
    float4 f;
    f.x = Fo[0];
    f.y = Fo[1];
    f.z = Fo[2];
    f.w = 0.f;
    Fown[i] = f;
  }
  // per-warp sums in R, per-block FP64 partial sums of U and W, stored [7][blocks]
  float v[7] = {U, Wv[0], Wv[1], Wv[2], Wv[3], Wv[4], Wv[5]};
#pragma unroll
  for (int k = 0; k < 7; ++k)
    for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], off);
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int k = 0; k < 7; ++k) red[warp][k] = (double)v[k];
  __syncthreads();
  const int nblk = gridDim.x, b = blockIdx.x, tid = threadIdx.x;
  if (tid < 7) {
    double s = 0.0;
    for (int w = 0; w < kMdThreads / 32; ++w) s += red[w][tid];
    partial[(size_t)tid * nblk + b] = s;
    __threadfence();                               // the partial before this block's count
  }
  md_grouped_sum<7, kMdThreads>(partial, counters, nblk, b, E, W, red);
}

// FP64, four lanes an atom. One bond: its exact FP64 vector as unit vector, length, 2/r, f_C and
// f_C', and the slot of its reverse entry. A lane without a bond keeps a phantom (u = 0, r = 1, f = f' = 2/r = 0),
// which contributes exactly zero to every sum.
struct MdBond {
  double ux, uy, uz, r, ir2, fc, fcp;
  int rs;
};
__device__ __forceinline__ MdBond md_bond(int N, int M, int i, int e, bool real, const MdGeom &G,
                                          const double *__restrict__ pos, const unsigned *__restrict__ keys,
                                          const int *__restrict__ cnt, const int *__restrict__ nbr,
                                          const char4 *__restrict__ shift, unsigned *status) {
  MdBond o = {0.0, 0.0, 0.0, 1.0, 0.0, 0.0, 0.0, -1};
  if (!real) return o;
  const unsigned key = keys[(size_t)e * N + i];
  const int j = nbr[(size_t)e * N + i];
  const char4 n = shift[(size_t)e * N + i];
  double dx = pos[3 * j] - pos[3 * i], dy = pos[3 * j + 1] - pos[3 * i + 1], dz = pos[3 * j + 2] - pos[3 * i + 2];
  if ((n.x | n.y | n.z) != 0) {   // an image shift (atoms near a face); t is exactly zero without one
    const ExactPair p = exact_pair(pos[3 * j], pos[3 * j + 1], pos[3 * j + 2], pos[3 * i], pos[3 * i + 1],
                                   pos[3 * i + 2], G.H, n.x, n.y, n.z);
    dx = p.dx;
    dy = p.dy;
    dz = p.dz;
  }
  o.rs = md_reverse_slot(N, M, i, key, cnt, keys, status);
  const double r2 = dx * dx + dy * dy + dz * dz, ir = rsqrt64(r2);
  double rr = 0.0;                                 // coincident atoms: r = 0, as the square root gives
  if (__double_as_longlong(r2) != 0) {             // r2 ir and one Newton step of the square root: r to half an ulp
    rr = r2 * ir;
    rr = __fma_rn(scale2(ir, -1), __fma_rn(-rr, rr, r2), rr);
  }
  o.r = rr;
  o.ir2 = scale2(ir, 1);
  o.ux = dx * ir;
  o.uy = dy * ir;
  o.uz = dz * ir;
  if (__double_as_longlong(rr) <= __double_as_longlong(G.R1)) {   // both positive: ordered as integers
    o.fc = 1.0;
  } else if (rr < G.R2) {
    const double w = (rr - G.R1) * G.inv_w;
    o.fc = 0.5 * (1.0 + cospi(w));
    o.fcp = G.fcp_k * sinpi(w);
  }
  return o;
}

// Passes 1 and 2 (batch_kernel.cuh) with four lanes an atom: lane b of the group holds the bonds b and, where NB = 2,
// b + 4, and takes what it needs of the others by shuffles. U, W += sum u (x) T (to be scaled by -2) and P per bond, as
// atom_core_f64. INNER: every lane has a bond inside R1 (f_C = 1, f_C' = 0).
template <int NB, bool INNER>
__device__ __forceinline__ void md_bond_core(const MdBond (&B)[NB], const PConsts<double> &K, const LaneOrder<double> &order,
                                             double &U, double (&W)[6], double (&P)[NB][3]) {
  const int lane = threadIdx.x & 31, b = lane & 3, base = lane & ~3;
  constexpr unsigned kAll = 0xffffffffu;
  double px[NB][4], py[NB][4], pz[NB][4], pf[NB][4];    // the group's bonds, rotated so that t = 0 is this lane's own
#pragma unroll
  for (int q = 0; q < NB; ++q)
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int src = base + ((b + t) & 3);
      px[q][t] = t ? __shfl_sync(kAll, B[q].ux, src) : B[q].ux;
      py[q][t] = t ? __shfl_sync(kAll, B[q].uy, src) : B[q].uy;
      pz[q][t] = t ? __shfl_sync(kAll, B[q].uz, src) : B[q].uz;
      pf[q][t] = INNER ? 1.0 : (t ? __shfl_sync(kAll, B[q].fc, src) : B[q].fc);
    }
  double u[NB][NB][4], S[NB], cc[NB], rad[NB];          // u = cos - h of own bond s and partner (q, t)
#pragma unroll
  for (int s = 0; s < NB; ++s) {
    S[s] = 0.0;
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        u[s][q][t] = 0.0;
        if (q == s && t == 0) continue;
        const double c = B[s].ux * px[q][t] + B[s].uy * py[q][t] + B[s].uz * pz[q][t];
        u[s][q][t] = c - K.h;
        if constexpr (INNER) S[s] += u[s][q][t] * u[s][q][t];
        else S[s] += pf[q][t] * (u[s][q][t] * u[s][q][t]);
      }
    const FxBond f = fx_bond_any<false>(B[s].r, S[s], *order.lane, *order.tab, order.kc);
    cc[s] = f.cc;
    const double e = f.fR - 2.0 * f.bh, mde = K.mha * (f.fR + e);             // f_R - b f_A and half of its r-derivative
    if constexpr (INNER) {
      U += e;
      rad[s] = mde;
    } else {
      U += B[s].fc * e;
      cc[s] *= B[s].fc;
      rad[s] = 0.5 * B[s].fcp * e + B[s].fc * mde;
    }
  }
  double pc[NB][4];
#pragma unroll
  for (int q = 0; q < NB; ++q)
#pragma unroll
    for (int t = 0; t < 4; ++t) pc[q][t] = t ? __shfl_sync(kAll, cc[q], base + ((b + t) & 3)) : cc[q];
  bool sw = false;   // the f_C' g terms of bonds inside the switching region
  if constexpr (!INNER) {
#pragma unroll
    for (int s = 0; s < NB; ++s) sw |= B[s].fcp != 0.0;
    sw = __any_sync(kAll, sw);
  }
#pragma unroll
  for (int s = 0; s < NB; ++s) {
    double ax = 0.0, ay = 0.0, az = 0.0, rg = 0.0;
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        if (q == s && t == 0) continue;
        const double w = (INNER ? cc[s] + pc[q][t] : cc[s] * pf[q][t] + pc[q][t] * B[s].fc) * u[s][q][t];
        ax += w * px[q][t];
        ay += w * py[q][t];
        az += w * pz[q][t];
        if (!INNER && sw) rg += pc[q][t] * (u[s][q][t] * u[s][q][t]);
      }
    double rd = rad[s];
    if constexpr (!INNER) rd += B[s].fcp * rg;
    const double sj = B[s].ux * ax + B[s].uy * ay + B[s].uz * az;
    const double c = rd * scale2(B[s].r, -1) - sj;
    const double tx = c * B[s].ux + ax, ty = c * B[s].uy + ay, tz = c * B[s].uz + az;
    P[s][0] = B[s].ir2 * tx;
    P[s][1] = B[s].ir2 * ty;
    P[s][2] = B[s].ir2 * tz;
    W[0] += B[s].ux * tx;
    W[1] += B[s].uy * ty;
    W[2] += B[s].uz * tz;
    W[3] += B[s].ux * ty;
    W[4] += B[s].uy * tz;
    W[5] += B[s].uz * tx;
  }
}

// Bonds b, b + 4, ... of the lane's atom, the core, and the results: P at the reverse entry's slot (rank, j) of Prev, so
// that the gather reads atom i's rows in order, and the group's sum of P (atom i's own part of F_i) in Fo of every lane.
template <int NB>
__device__ __forceinline__ void md_force_atom64(int N, int M, int i, int m, const MdGeom &G, const PConsts<double> &K,
                                                const double *__restrict__ pos, const unsigned *__restrict__ keys,
                                                const int *__restrict__ cnt, const int *__restrict__ nbr,
                                                const char4 *__restrict__ shift, dvec4 *__restrict__ Prev, const LaneOrder<double> &order,
                                              unsigned *status, double &U, double (&W)[6], double (&Fo)[3]) {
  const int b = threadIdx.x & 3;
  MdBond B[NB];
  bool inner = NB == 1;
#pragma unroll
  for (int s = 0; s < NB; ++s) {
    B[s] = md_bond(N, M, i, b + 4 * s, b + 4 * s < m, G, pos, keys, cnt, nbr, shift, status);
    inner = inner && __double_as_longlong(B[s].fc) == 0x3ff0000000000000ll && (__double_as_longlong(B[s].fcp) << 1) == 0;
  }
  double P[NB][3];
  if (NB == 1 && __all_sync(0xffffffffu, inner)) md_bond_core<NB, NB == 1>(B, K, order, U, W, P);
  else md_bond_core<NB, false>(B, K, order, U, W, P);
#pragma unroll
  for (int s = 0; s < NB; ++s)
    if (B[s].rs >= 0) {
      // two 16-byte stores: one 32-byte store of a called function has come out wrong (nvcc 13.0)
      double2 *o = reinterpret_cast<double2 *>(Prev + B[s].rs);
      o[0] = make_double2(P[s][0], P[s][1]);
      o[1] = make_double2(P[s][2], 0.0);
    }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    Fo[k] = NB == 2 ? P[0][k] + P[NB - 1][k] : P[0][k];
    Fo[k] += __shfl_xor_sync(0xffffffffu, Fo[k], 1);
    Fo[k] += __shfl_xor_sync(0xffffffffu, Fo[k], 2);
  }
}

// Four lanes an atom, a lane a bond. A scheduler's FP64 unit takes 64 cycles a warp instruction, so what counts for a
// small system is how many schedulers have work and how few FP64 instructions stand in one warp's line: 4,096 atoms reach
// 512 schedulers with ~65 each instead of 128 with ~300 (51.2 us with the library's functions and a thread an atom, 32 us
// with fx64.cuh, 15.9 us so); for a large one the live values of one bond a lane leave room for 16 warps an SM instead of
// 8 (512,000 atoms: 997 -> 419 us). In FP32, issue-bound, the shuffles cost more than they bring (46.7 against 55 us).
__global__ void __launch_bounds__(kMdThreads, 4) md_force64_kernel(
    int N, int M, const __grid_constant__ MdGeom G, const __grid_constant__ PConsts<double> K, const double *__restrict__ pos,
    const unsigned *__restrict__ keys, const int *__restrict__ cnt,
    const int *__restrict__ nbr, const char4 *__restrict__ shift, dvec4 *__restrict__ Fown,
    dvec4 *__restrict__ Prev, double *__restrict__ partial, unsigned *counters, double *__restrict__ E,
    double *__restrict__ W, int *__restrict__ zero_cells, int ncells, unsigned *status) {
  __shared__ double red[kMdThreads / 32][8];
  __shared__ FxTables s_fx;
  const int tid = threadIdx.x, i = blockIdx.x * kMdForceAtoms + (tid >> 2);
  const bool valid = i < N;
  pdl_trigger();
  fx_load_tables(s_fx);
  pdl_wait();
  // NVE steps: the cell counts, last read by the search before this kernel, are zeroed for the next step's binning
  if (zero_cells)
    for (int c = blockIdx.x * kMdThreads + tid; c < ncells; c += (int)(gridDim.x * kMdThreads)) zero_cells[c] = 0;
  __syncthreads();
  const FxLane fxl = fx_lane_of<false>(&K.D0, s_fx);   // the first eight constants are laid out as prep_kernel's
  const LaneOrder<double> order = {&fxl, &s_fx, &K.D0};
  int m = valid ? min(cnt[i], M) : 0;   // a truncated list (count > M) is flagged; its row holds M entries
  if (m > kMdMaxM) {
    set_status(status, TERSOFF_STATUS_MANY_NBRS);
    m = 0;
  }
  double U = 0.0, Wv[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0}, Fo[3];
  if (__all_sync(0xffffffffu, m <= 4))
    md_force_atom64<1>(N, M, i, m, G, K, pos, keys, cnt, nbr, shift, Prev, order, status, U, Wv, Fo);
  else
    md_force_atom64<2>(N, M, i, m, G, K, pos, keys, cnt, nbr, shift, Prev, order, status, U, Wv, Fo);
  if (valid && (tid & 3) == 0) {
    dvec4 f;
    f.x = Fo[0];
    f.y = Fo[1];
    f.z = Fo[2];
    f.w = 0.0;
    Fown[i] = f;
  }
  // per-warp sums, per-block FP64 partial sums of U_i = U/2 and W = -2 Wv, stored [7][blocks]
  double v[8] = {U, Wv[0], Wv[1], Wv[2], Wv[3], Wv[4], Wv[5], 0.0};
  const double t = warp_sums8(v);
  if ((tid & 3) == 0) red[tid >> 5][(tid >> 2) & 7] = t;
  __syncthreads();
  const int nblk = gridDim.x, b = blockIdx.x;
  if (tid < 7) {
    double s = 0.0;
    for (int w = 0; w < kMdThreads / 32; ++w) s += red[w][tid];
    partial[(size_t)tid * nblk + b] = s * (tid == 0 ? 0.5 : -2.0);
    __threadfence();                               // the partial before this block's count
  }
  md_grouped_sum<7, kMdThreads>(partial, counters, nblk, b, E, W, red);
}

// F_i = sum_e P_ij - sum_e P_ji over atom i's entries e = (j, n): the first sum from Fown (the force
// kernel's), P_ji from Prev row e (written there by atom j). An atom with more than kMdMaxM entries
// has no P (the force kernel flags it) and gets F = 0.
template <typename R>
__device__ __forceinline__ void md_gather_atom(int N, int M, int i, int ci,
                                               const typename Vec4<R>::T *__restrict__ Fown,
                                               const typename Vec4<R>::T *__restrict__ Prev, R &Fx, R &Fy, R &Fz) {
  const int m = ci <= kMdMaxM ? min(ci, M) : 0;
  const auto f = Fown[i];
  Fx = f.x;
  Fy = f.y;
  Fz = f.z;
#pragma unroll
  for (int e = 0; e < kMdMaxM; ++e)
    if (e < m) {
      const auto b = Prev[(size_t)e * N + i];
      Fx -= b.x;
      Fy -= b.y;
      Fz -= b.z;
    }
}
template <typename R>
__global__ void md_gather_kernel(int N, int M, const int *__restrict__ cnt, const typename Vec4<R>::T *__restrict__ Fown,
                                 const typename Vec4<R>::T *__restrict__ Prev, R *__restrict__ F) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  pdl_trigger();
  pdl_wait();
  if (i >= N) return;
  R Fx, Fy, Fz;
  md_gather_atom<R>(N, M, i, cnt[i], Fown, Prev, Fx, Fy, Fz);
  F[3 * (size_t)i] = Fx;
  F[3 * (size_t)i + 1] = Fy;
  F[3 * (size_t)i + 2] = Fz;
}

// ---------------------------------------------------------------------------------------------
// Launches of the MD calls for one (N, box, parameters): the geometry, the workspaces and the kernels' arguments.
struct MdRun {
  int N, M, precision, nblk, fblk, ncells;
  bool pdl;
  MdGeom G;
  const double *pos;
  float4 *x4, *cells;
  int4 *m4;
  int *cellcnt, *cnt, *nbr;
  char4 *shift;
  unsigned *keys, *status, *sum_counters;
  double *red;
  void *Fown, *Prev;
  PConsts<double> K64;
  PConsts<float> K32;
};

int md_prepare(Ctx &c, int N, const double *pos, const double *boxh, const double *x, double R1, double R2, int M,
               int precision, cudaStream_t s, MdRun &r, std::string &err) {
  MdGeom &G = r.G;
  for (int k = 0; k < 9; ++k) G.H[k] = boxh[k];
  const double *H = G.H;
  const double bxc[3] = {H[4] * H[8] - H[5] * H[7], H[5] * H[6] - H[3] * H[8], H[3] * H[7] - H[4] * H[6]};
  const double cxa[3] = {H[7] * H[2] - H[8] * H[1], H[8] * H[0] - H[6] * H[2], H[6] * H[1] - H[7] * H[0]};
  const double axb[3] = {H[1] * H[5] - H[2] * H[4], H[2] * H[3] - H[0] * H[5], H[0] * H[4] - H[1] * H[3]};
  const double det = H[0] * bxc[0] + H[1] * bxc[1] + H[2] * bxc[2];
  if (!std::isfinite(det) || det == 0.0) {
    err = "singular or non-finite box";
    return TERSOFF_E_ARG;
  }
  for (int mu = 0; mu < 3; ++mu) {
    G.Hinv[3 * mu + 0] = bxc[mu] / det;
    G.Hinv[3 * mu + 1] = cxa[mu] / det;
    G.Hinv[3 * mu + 2] = axb[mu] / det;
  }
  const double vol = std::fabs(det);
  const double gap[3] = {vol / std::sqrt(bxc[0] * bxc[0] + bxc[1] * bxc[1] + bxc[2] * bxc[2]),
                         vol / std::sqrt(cxa[0] * cxa[0] + cxa[1] * cxa[1] + cxa[2] * cxa[2]),
                         vol / std::sqrt(axb[0] * axb[0] + axb[1] * axb[1] + axb[2] * axb[2])};
  double esum = 0.0;
  for (int k = 0; k < 3; ++k) {
    G.nc[k] = (int)std::floor(gap[k] / R2);
    if (G.nc[k] < 3) {
      err = "every plane spacing of the box must be at least 3*R2";
      return TERSOFF_E_ARG;
    }
    double en = 0.0;
    for (int mu = 0; mu < 3; ++mu) {
      G.E[3 * k + mu] = (float)(H[3 * k + mu] / G.nc[k]);
      en += G.E[3 * k + mu] * (double)G.E[3 * k + mu];
    }
    esum += std::sqrt(en);
  }
  // FP32 distance error: positions from a brick's centre (at most 4 sums of the cell edges in size), the in-cell part and
  // the cell's offset each rounded, then added and subtracted, stay within ~35 ulp of that sum (on the global-memory path,
  // from offsets of one cell, within ~12); the band is 128 ulp wide
  const double margin = 128.0 * 1.2e-7 * esum * 2.0 * R2 + 1e-6;
  G.diag = 1;
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b)
      if (a != b && (H[3 * a + b] != 0.0 || G.Hinv[3 * a + b] != 0.0)) G.diag = 0;
  for (int a = 0; a < 3; ++a)
    for (int k = 0; k < 3; ++k) {
      G.Hn[3 * a + k] = G.Hinv[3 * a + k] * (double)G.nc[k];
      G.Hnh[3 * a + k] = (float)G.Hn[3 * a + k];
      G.Hnl[3 * a + k] = (float)(G.Hn[3 * a + k] - (double)G.Hnh[3 * a + k]);
    }
  G.R1 = R1;
  G.R2 = R2;
  G.R2sq = R2 * R2;
  G.inv_w = 1.0 / (R2 - R1);
  G.fcp_k = -0.5 * M_PI / (R2 - R1);
  G.R1f = (float)R1;
  G.R2f = (float)R2;
  G.inv_wf = (float)G.inv_w;
  G.fcp_kf = (float)G.fcp_k;
  G.cut2_lo = (float)(R2 * R2 - margin);
  G.cut2_hi = (float)(R2 * R2 + margin);
  // the filter |x_j - x_i|^2 - c from |x|^2 and x_j . x_i of positions at most X from a brick's centre: four rounded
  // operations on terms of at most 4 X^2 and the rounding of |x|^2 stay below 2e-6 X^2; four times that
  double X = 0.0;
  const int halo[3] = {kHX, kHY, kHZ};
  for (int k = 0; k < 3; ++k) {
    double en = 0.0;
    for (int mu = 0; mu < 3; ++mu) en += G.E[3 * k + mu] * (double)G.E[3 * k + mu];
    X += 0.5 * halo[k] * std::sqrt(en);
  }
  G.scan_cut = (float)(R2 * R2 + margin + 8e-6 * X * X);
  const long ncells = (long)G.nc[0] * G.nc[1] * G.nc[2];
  if (ncells > (1L << 26)) {
    err = "too many cells";
    return TERSOFF_E_ARG;
  }
  const int nblk = (N + kMdThreads - 1) / kMdThreads;
  const int fblk = precision == 64 ? (N + kMdForceAtoms - 1) / kMdForceAtoms : nblk;   // blocks of the force kernel
  const int ngroups = md_ngroups(fblk);
  const size_t rs = precision == 64 ? 8 : 4;
  if (c.md_cellcnt.ensure((ncells + ngroups + 1) * sizeof(int)) || c.md_cells.ensure(ncells * kMdCap * sizeof(float4)) ||
      c.md_pos.ensure((size_t)N * (sizeof(float4) + sizeof(int4))) || c.md_cnt.ensure((size_t)N * sizeof(int)) ||
      c.md_nbr.ensure((size_t)N * M * sizeof(int)) || c.md_shift.ensure((size_t)N * M * sizeof(char4)) ||
      c.md_keys.ensure((size_t)N * M * sizeof(unsigned)) || c.md_Pij.ensure((size_t)N * (kMdMaxM + 1) * 4 * rs) ||
      c.md_red.ensure(md_sum_bytes(7, fblk))) {
    err = "device allocation failed";
    return TERSOFF_E_CUDA;
  }
  c.md_N = N;
  c.md_M = M;
  r.N = N;
  r.M = M;
  r.precision = precision;
  // Programmatic launch overlaps a kernel's start with its predecessor's last blocks (512,000 atoms, FP32: 142.9 -> 135.5 us
  // a call, back to back). The line was drawn from two sizes, on a first reading of 66 us without it and 73 with it at 4,500
  // atoms, which later measurements of both sides in turn do not bear out: 512 atoms 39.1 -> 33.2 us, 4,096 38.8 -> 29.4,
  // 21,952 41.1 -> 38.3, 64,000 53.2 -> 46.5, 125,000 63.1 -> 52.9 (a call waited for by itself: 54 -> 47, 53 -> 45,
  // 56 -> 50, 67 -> 61, 78 -> 70; FP64 alike or equal). Nothing speaks for the line any more. The steps of a run take
  // it at every size (md_nve sets it)
  r.pdl = c.pdl && N >= 131072;
  r.nblk = nblk;
  r.fblk = fblk;
  r.ncells = (int)ncells;
  r.pos = pos;
  r.x4 = c.md_pos.as<float4>();
  r.m4 = reinterpret_cast<int4 *>(r.x4 + N);
  r.cells = c.md_cells.as<float4>();
  r.cellcnt = c.md_cellcnt.as<int>();
  r.sum_counters = c.md_cellcnt.as<unsigned>() + ncells;
  r.cnt = c.md_cnt.as<int>();
  r.nbr = c.md_nbr.as<int>();
  r.shift = c.md_shift.as<char4>();
  r.keys = c.md_keys.as<unsigned>();
  r.status = c.status.as<unsigned>();
  r.red = c.md_red.as<double>();
  r.Fown = c.md_Pij.p;
  r.Prev = static_cast<char *>(c.md_Pij.p) + (size_t)N * 4 * rs;
  const double D0 = x[0], al = x[1], r0 = x[2], be = x[3], n = x[4], h = x[5];
  const double log2e = 1.4426950408889634;
  r.K64 = PConsts<double>{D0, -al * log2e, r0, -0.5 * al, be, h, n, -0.5 / n};
  r.K32 = PConsts<float>{(float)D0, (float)(-al * log2e), (float)r0, (float)(-0.5 * al), (float)be, (float)h,
                         (float)n, (float)(-0.5 / n)};
  // cell counts and the force kernel's sum counters, both zero at the start of the call: one memset
  if (cudaMemsetAsync(c.md_cellcnt.p, 0, (ncells + ngroups + 1) * sizeof(int), s) != cudaSuccess) {
    err = "CUDA error in the workspace reset";
    return TERSOFF_E_CUDA;
  }
  return TERSOFF_OK;
}

// One MD kernel with programmatic stream serialization (unless the context's launch mode has it off): it may become
// resident while its predecessor in the call drains, which it waits for before its first access (pdl_wait). The
// caller checks the launches (launched).
template <typename... P, typename... A>
void md_launch(const MdRun &r, void (*kern)(P...), unsigned grid, unsigned threads, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = r.pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  (void)cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

void md_launch_cells(const MdRun &r, cudaStream_t s) {
  md_launch(r, md_cells_kernel, r.nblk, kMdThreads, s, r.N, r.pos, r.G, r.cellcnt, r.cells, r.x4, r.m4, r.cnt, r.status);
}

// Search and force kernels; the P_ij are left for the gather. zero_cells: also zero the cell counts for the next binning.
void md_launch_search_force(const MdRun &r, double *E, double *W, bool zero_cells, cudaStream_t s) {
  const int *nc = r.G.nc;
  const long nbricks = (long)((nc[0] + kBX - 1) / kBX) * ((nc[1] + kBY - 1) / kBY) * ((nc[2] + kBZ - 1) / kBZ);
  md_launch(r, md_search_kernel, (unsigned)nbricks, kSearchThreads, s, r.N, r.M, r.pos, r.G, r.x4, r.m4, r.cellcnt, r.cells, r.cnt,
                                                               r.keys, r.nbr, r.shift, r.status);
  int *zc = zero_cells ? r.cellcnt : nullptr;
  if (r.precision == 64) {
    md_launch(r, md_force64_kernel, r.fblk, kMdThreads, s, r.N, r.M, r.G, r.K64, r.pos, r.keys, r.cnt, r.nbr, r.shift,
                                                    static_cast<dvec4 *>(r.Fown), static_cast<dvec4 *>(r.Prev), r.red,
                                                    r.sum_counters, E, W, zc, r.ncells, r.status);
  } else {
    md_launch(r, md_force_kernel, r.fblk, kMdThreads, s, r.N, r.M, r.G, r.K32, r.x4, r.keys, r.cnt, static_cast<float4 *>(r.Fown),
                                                  static_cast<float4 *>(r.Prev), r.red, r.sum_counters, E, W, zc, r.ncells,
                                                  r.status);
  }
}

int md_force(Ctx &c, int N, const double *pos, const double *boxh, const double *x, double R1, double R2,
             int M, int precision, double *E, void *F, double *W, cudaStream_t s, std::string &err) {
  MdRun r;
  if (const int rc = md_prepare(c, N, pos, boxh, x, R1, R2, M, precision, s, r, err)) return rc;
  md_launch_cells(r, s);
  md_launch_search_force(r, E, W, false, s);
  if (precision == 64)
    md_launch(r, md_gather_kernel<double>, r.nblk, kMdThreads, s, N, M, r.cnt, static_cast<const dvec4 *>(r.Fown),
                                                           static_cast<const dvec4 *>(r.Prev), static_cast<double *>(F));
  else
    md_launch(r, md_gather_kernel<float>, r.nblk, kMdThreads, s, N, M, r.cnt, static_cast<const float4 *>(r.Fown),
                                                          static_cast<const float4 *>(r.Prev), static_cast<float *>(F));
  const cudaError_t e = launched(4);   // cells, search, force (with the sums), gather
  if (e != cudaSuccess) {
    err = std::string("CUDA error: ") + cudaGetErrorString(e);
    return TERSOFF_E_CUDA;
  }
  return TERSOFF_OK;
}

// ---------------------------------------------------------------------------------------------
// Velocity-Verlet NVE on the MD-scale force call (units eV, A, amu, fs). The integrator is not part
// of the paper's method; it drives the force call the way an MD code does.
constexpr double kAccel = 9.648533215665e-3;      // 1 eV / (A amu) in A / fs^2 (CODATA 2018)
constexpr double kKinetic = 103.6426965268;       // 1 amu A^2 / fs^2 in eV

// a_i = (1 eV / (A amu)) / m_i in A / fs^2 per eV / A, once per run (the device's FP64 divide is slow).
__global__ void md_accel_kernel(int N, const double *__restrict__ mass, double *__restrict__ acc) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) acc[i] = kAccel / mass[i];
}

// One step's per-atom work between two searches, in one kernel: F_i from the P_ij (md_gather_kernel), the second half
// kick v += a F h of the step just evaluated (none before the first), the kinetic energy sum_i m v^2 / 2 into *Ekin
// in a fixed order, and, but after the last step, the first half kick v += a F dt/2 and the drift x += v dt of the
// next one with the binning of the new position. Every part is local to the atom, so a step is three launches
// (search, force, this) instead of eight with two memsets.
template <typename R>
__global__ void __launch_bounds__(kMdThreads) md_advance_kernel(
    int N, int M, const __grid_constant__ MdGeom G, int *cnt, const typename Vec4<R>::T *__restrict__ Fown,
    const typename Vec4<R>::T *__restrict__ Prev, R *__restrict__ F, double *__restrict__ pos, double *__restrict__ vel,
    const double *__restrict__ mass, const double *__restrict__ acc, double dt_kick, double dt_next,
    double *__restrict__ partial, unsigned *counters, double *__restrict__ Ekin, int *__restrict__ cellcnt,
    float4 *__restrict__ cellx, float4 *__restrict__ x4, int4 *__restrict__ m4, unsigned *status) {
  __shared__ double red[kMdThreads / 32][8];
  const int i = blockIdx.x * blockDim.x + threadIdx.x, tid = threadIdx.x;
  pdl_trigger();
  pdl_wait();
  double ke = 0.0;
  if (i < N) {
    R f[3];
    md_gather_atom<R>(N, M, i, cnt[i], Fown, Prev, f[0], f[1], f[2]);
    const double ai = acc[i], h = 0.5 * dt_kick * ai;
    double v[3], v2 = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      v[k] = vel[3 * i + k];
      if (dt_kick > 0.0) v[k] += h * (double)f[k];   // not with 0 times a force that may not be finite
      v2 += v[k] * v[k];
    }
    ke = (0.5 * kKinetic) * mass[i] * v2;
    if (dt_next > 0.0) {
      const double hn = 0.5 * dt_next * ai;
      double x[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        v[k] = v[k] + hn * (double)f[k];
        x[k] = pos[3 * i + k] + v[k] * dt_next;
        pos[3 * i + k] = x[k];
      }
      md_bin_atom(i, x[0], x[1], x[2], G, cellcnt, cellx, x4, m4, cnt, status);   // cnt[i] only, read above
    } else {
#pragma unroll
      for (int k = 0; k < 3; ++k) F[3 * (size_t)i + k] = f[k];
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) vel[3 * i + k] = v[k];
  }
  for (int off = 16; off > 0; off >>= 1) ke += __shfl_xor_sync(0xffffffffu, ke, off);
  if ((tid & 31) == 0) red[tid >> 5][0] = ke;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int w = 0; w < kMdThreads / 32; ++w) s += red[w][0];
    partial[blockIdx.x] = s;
    __threadfence();
  }
  md_grouped_sum<1, kMdThreads>(partial, counters, gridDim.x, blockIdx.x, Ekin, nullptr, red);
}

int md_nve(Ctx &c, int N, double *pos, double *vel, const double *mass, const double *boxh, const double *x,
           double R1, double R2, int M, int precision, double dt, int nsteps, double *Epot, double *Ekin,
           void *F, double *W, cudaStream_t s, std::string &err) {
  const int nblk = (N + kMdThreads - 1) / kMdThreads;
  const size_t sum_bytes = (md_sum_bytes(1, nblk) + 15) / 16 * 16;
  if (c.md_ke.ensure(sum_bytes + (size_t)N * sizeof(double))) {
    err = "device allocation failed";
    return TERSOFF_E_CUDA;
  }
  double *part = c.md_ke.as<double>();
  unsigned *counters = reinterpret_cast<unsigned *>(static_cast<char *>(c.md_ke.p) + md_counter_offset(1, nblk));
  double *acc = reinterpret_cast<double *>(static_cast<char *>(c.md_ke.p) + sum_bytes);
  MdRun r;
  if (const int rc = md_prepare(c, N, pos, boxh, x, R1, R2, M, precision, s, r, err)) return rc;
  r.pdl = c.pdl;
  if (cudaMemsetAsync(counters, 0, (md_ngroups(nblk) + 1) * sizeof(unsigned), s) != cudaSuccess) {
    err = "CUDA error in the workspace reset";
    return TERSOFF_E_CUDA;
  }
  md_accel_kernel<<<nblk, kMdThreads, 0, s>>>(N, mass, acc);
  md_launch_cells(r, s);
  cudaError_t e = launched(2);
  for (int k = 0; k <= nsteps && e == cudaSuccess; ++k) {
    const bool last = k == nsteps;
    md_launch_search_force(r, Epot + k, W, !last, s);
    const double kick = k == 0 ? 0.0 : dt, next = last ? 0.0 : dt;
    if (precision == 64)
      md_launch(r, md_advance_kernel<double>, nblk, kMdThreads, s, 
          N, M, r.G, r.cnt, static_cast<const dvec4 *>(r.Fown), static_cast<const dvec4 *>(r.Prev), static_cast<double *>(F),
          pos, vel, mass, acc, kick, next, part, counters, Ekin + k, r.cellcnt, r.cells, r.x4, r.m4, r.status);
    else
      md_launch(r, md_advance_kernel<float>, nblk, kMdThreads, s, 
          N, M, r.G, r.cnt, static_cast<const float4 *>(r.Fown), static_cast<const float4 *>(r.Prev), static_cast<float *>(F),
          pos, vel, mass, acc, kick, next, part, counters, Ekin + k, r.cellcnt, r.cells, r.x4, r.m4, r.status);
    e = launched(3);   // search, force, advance
  }
  if (e != cudaSuccess) {
    err = std::string("CUDA error: ") + cudaGetErrorString(e);
    return TERSOFF_E_CUDA;
  }
  return TERSOFF_OK;
}

}  // namespace tsf
