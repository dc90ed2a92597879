// atom64.cuh -- the per-atom core of the potential in FP64 (passes 1 and 2 of batch_kernel.cuh), written for a
// device whose FP64 unit issues one warp instruction in 16 cycles per multiprocessor: the transcendentals run on
// the integer units (fx64.cuh), the cutoff factors fold away where every bond lies inside R1, and the virial and
// the forces share their products. About 170 FP64 instructions per atom of four bonds and parameter set, from about
// 550 with the library's exp2 and log2 and the formulas term by term. Fitness of 73 sets on 100 64-atom cells (with the
// 8-wide tiles of batch_launch.cuh): 889 -> 290 us; ncu has the FP64 pipe active 66 % of the time at 235 instructions an
// evaluation, tile sums and gather included; the rest is the latency of two warps a scheduler.
#pragma once

#include "common.cuh"
#include "ctx.hpp"
#include "fx64.cuh"

namespace tsf {

#include "fx64_tables.inc"

// Fills a kernel's table copy in shared memory (all threads; the caller synchronises).
__device__ __forceinline__ void fx_load_tables(FxTables &t) {
  constexpr int n = sizeof(FxTables) / sizeof(uint4);
  const uint4 *src = reinterpret_cast<const uint4 *>(&kFxTables);
  uint4 *dst = reinterpret_cast<uint4 *>(&t);
#pragma unroll 10
  for (int k = threadIdx.x; k < n; k += blockDim.x) dst[k] = src[k];   // one warp: ten loads in flight
}

// f_R, b f_A / 2 and the coefficient cc of fx_bond.
struct FxBond {
  double fR, bh, cc;
};
// The library's functions, for what lies beyond the fixed-point ranges (far-off parameters, infinities, NaN). kc: the
// parameter set's constants as prep_kernel lays them out.
template <bool GEN>
__device__ __noinline__ FxBond fx_bond_slow(double r, double S, const double *kc) {
  FxBond o;
  const double D0 = kc[0], k1 = kc[1], r0 = kc[2], n = kc[6], minus_inv2n = kc[7], B = GEN ? 1.0 : kc[4];
  const double x = exp2((r - r0) * k1), hA = D0 * x, zr = B * S, z = zr > 1e-30 ? zr : 1e-30;
  const double zn = exp2(n * log2(z)), u2 = zn * 2.0 + 2.0;
  o.fR = GEN ? kc[8] * exp2((r - r0) * kc[9]) : hA * x;
  o.bh = exp2(minus_inv2n * log2(u2) - minus_inv2n) * hA;
  o.cc = B * (o.bh * zn / (z * u2));
  return o;
}
template <bool GEN>
__device__ __forceinline__ FxBond fx_bond_any(double r, double S, const FxLane &o, const FxTables &t, const double *kc) {
  FxBond v;
  if (!fx_bond(r, S, o, t, v.fR, v.bh, v.cc)) v = fx_bond_slow<GEN>(r, S, kc);
  return v;
}
// The same as a called function: some 420 integer instructions that need not be repeated for every bond of every
// list length and tile.
template <bool GEN>
__device__ __noinline__ FxBond fx_bond_call(double r, double S, const FxLane *o, const FxTables *t, const double *kc) {
  return fx_bond_any<GEN>(r, S, *o, *t, kc);
}
// The lane's fixed-point constants from the constants of its parameter set (prep_kernel's layout).
template <bool GEN>
__device__ __forceinline__ FxLane fx_lane_of(const double *kc, const FxTables &t) {
  return GEN ? fx_lane(kc[2], kc[1], kc[9], kc[0], kc[8], 1.0, kc[6], kc[7], t)
             : fx_lane(kc[2], kc[1], 2.0 * kc[1], kc[0], kc[0], kc[4], kc[6], kc[7], t);
}

// x 2^k for a normal x whose result is normal, on the integer unit.
__device__ __forceinline__ double scale2(double x, int k) {
  return fx_from_bits(fx_bits(x) + ((uint64_t)(int64_t)k << 52));
}

// 1/x to within 0.5002 ulp (a divide: 0.5), from the FP32 reciprocal (e = 1 - x y0 is exact and below 2^-22, the cubic
// step leaves e^3, and only its last operation rounds).
__device__ __forceinline__ double rcp64(double x) {
  const int e = (int)((fx_bits(x) >> 52) & 0x7ffu) - 1023;
  if (e < -100 || e > 100) return 1.0 / x;
  const double y0 = widen(rcp((float)x));
  const double d = __fma_rn(-x, y0, 1.0);
  return __fma_rn(y0, __fma_rn(d, d, d), y0);
}

// 1/sqrt(x) to within 1.0002 ulp (the reciprocal of a rounded square root: 1.5), likewise; here x y0 is rounded.
__device__ __forceinline__ double rsqrt64(double x) {
  const int e = (int)((fx_bits(x) >> 52) & 0x7ffu) - 1023;
  if (e < -100 || e > 100) return rsqrt(x);
  const double y0 = widen(rsqrtf((float)x));
  const double d = __fma_rn(-(x * y0), y0, 1.0);
  return __fma_rn(y0 * d, __fma_rn(d, 0.375, 0.5), y0);
}

// atom_core of batch_kernel.cuh in FP64: U = sum_j f_C (f_R - b f_A), P_j = dU_i/dd_ij, and sum_j u_j (x) T_j added
// to Wt (xx, yy, zz, xy, yz, zx), where P_j = (2/r_j) T_j, so that the atom's virial -sum_j d_j (x) P_j is -2 of it.
// T_j = (rad_j r_j/2 - u_j . A_j) u_j + A_j with the A_j, rad_j of atom_core. INNER: every bond is inside R1.
// CALL: the bond functions as a called function (long lists, and where the code would repeat them too often).
// kc: the constants of the parameter set (fx_bond_slow).
template <int M, bool INNER, bool GEN, bool CALL, typename K_>
__device__ __forceinline__ void atom_core_f64(const double (&ux)[M], const double (&uy)[M], const double (&uz)[M],
                                              const double (&r)[M], const double (&ir2)[M], const double (&fc)[M],
                                              const double (&fcp)[M], const double *cs, const K_ &K,
                                              const FxLane &lane, const FxTables &tab, const double *kc, double &U, double (&Wt)[6],
                                              double (&Px)[M], double (&Py)[M], double (&Pz)[M]) {
  constexpr int NP = M * (M - 1) / 2, NQ = NP > 0 ? NP : 1;
  double zeta[M], tq[NQ], gq[GEN ? NQ : 1];        // tq: g'/2 (Tersoff form), u with g' = 2 beta u (minimal form)
#pragma unroll
  for (int j = 0; j < M; ++j) zeta[j] = 0.0;
  {
    int q = 0;
#pragma unroll
    for (int j = 0; j < M; ++j)
#pragma unroll
      for (int k = j + 1; k < M; ++k) {
        const double u = cs[q] - K.h;
        double g;
        if constexpr (GEN) {
          const double u2 = u * u, iv = rcp64(u2 + K.d2);
          g = __fma_rn(K.gcd, u2 * iv, K.g0);
          tq[q] = K.gc2 * u * (iv * iv);
          gq[q] = g;
        } else {
          tq[q] = u;
          g = u;
        }
        if constexpr (INNER && !GEN) {
          zeta[j] = __fma_rn(u, u, zeta[j]);
          zeta[k] = __fma_rn(u, u, zeta[k]);
        } else {
          const double gg = GEN ? g : u * u;
          zeta[j] = INNER ? zeta[j] + gg : __fma_rn(fc[k], gg, zeta[j]);
          zeta[k] = INNER ? zeta[k] + gg : __fma_rn(fc[j], gg, zeta[k]);
        }
        ++q;
      }
  }
  double cc[M], rad[M];
  U = 0.0;
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const FxBond f = CALL ? fx_bond_call<GEN>(r[j], zeta[j], &lane, &tab, kc) : fx_bond_any<GEN>(r[j], zeta[j], lane, tab, kc);
    const double e = __fma_rn(f.bh, -2.0, f.fR);   // f_R - b f_A
    double mde;
    if constexpr (GEN) mde = __fma_rn(K.hl, f.fR, K.mha * f.bh);
    else mde = K.mha * (f.fR + e);
    if constexpr (INNER) {
      U += e;
      cc[j] = f.cc;
      rad[j] = mde;
    } else {
      U = __fma_rn(fc[j], e, U);
      cc[j] = fc[j] * f.cc;
      rad[j] = __fma_rn(0.5 * fcp[j], e, fc[j] * mde);
    }
  }
  double Ax[M], Ay[M], Az[M];
#pragma unroll
  for (int j = 0; j < M; ++j) Ax[j] = Ay[j] = Az[j] = 0.0;
  {
    int q = 0;
#pragma unroll
    for (int j = 0; j < M; ++j)
#pragma unroll
      for (int k = j + 1; k < M; ++k) {
        const double w = (INNER ? cc[j] + cc[k] : __fma_rn(cc[j], fc[k], cc[k] * fc[j])) * tq[q];
        Ax[j] = __fma_rn(w, ux[k], Ax[j]);
        Ay[j] = __fma_rn(w, uy[k], Ay[j]);
        Az[j] = __fma_rn(w, uz[k], Az[j]);
        Ax[k] = __fma_rn(w, ux[j], Ax[k]);
        Ay[k] = __fma_rn(w, uy[j], Ay[k]);
        Az[k] = __fma_rn(w, uz[j], Az[k]);
        ++q;
      }
  }
  if constexpr (!INNER) {   // the f_C' g terms of bonds inside the switching region
    bool sw = false;
#pragma unroll
    for (int j = 0; j < M; ++j) sw |= (__double_as_longlong(fcp[j]) << 1) != 0;
    if (__any_sync(0xffffffffu, sw)) {
      double Rg[M];
#pragma unroll
      for (int j = 0; j < M; ++j) Rg[j] = 0.0;
      int q = 0;
#pragma unroll
      for (int j = 0; j < M; ++j)
#pragma unroll
        for (int k = j + 1; k < M; ++k) {
          const double g = GEN ? gq[GEN ? q : 0] : tq[q] * tq[q];   // cc carries beta in the minimal form
          Rg[j] = __fma_rn(cc[k], g, Rg[j]);
          Rg[k] = __fma_rn(cc[j], g, Rg[k]);
          ++q;
        }
#pragma unroll
      for (int j = 0; j < M; ++j) rad[j] = __fma_rn(fcp[j], Rg[j], rad[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const double s = __fma_rn(uz[j], Az[j], __fma_rn(uy[j], Ay[j], ux[j] * Ax[j]));
    const double c = __fma_rn(rad[j], scale2(r[j], -1), -s);
    const double tx = __fma_rn(c, ux[j], Ax[j]), ty = __fma_rn(c, uy[j], Ay[j]), tz = __fma_rn(c, uz[j], Az[j]);
    Px[j] = ir2[j] * tx;
    Py[j] = ir2[j] * ty;
    Pz[j] = ir2[j] * tz;
    Wt[0] = __fma_rn(ux[j], tx, Wt[0]);
    Wt[1] = __fma_rn(uy[j], ty, Wt[1]);
    Wt[2] = __fma_rn(uz[j], tz, Wt[2]);
    Wt[3] = __fma_rn(ux[j], ty, Wt[3]);
    Wt[4] = __fma_rn(uy[j], tz, Wt[4]);
    Wt[5] = __fma_rn(uz[j], tx, Wt[5]);
  }
}

}  // namespace tsf
