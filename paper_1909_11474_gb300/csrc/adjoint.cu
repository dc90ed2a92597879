// adjoint.cu -- gradient of the fitness loss with respect to the parameters, x = [D0, alpha, r0,
// beta, n, h] (Eq. 16) of the minimal potential or x = [D0, alpha, r0, S, n, h, gamma, c, d] of the
// Tersoff form (Eq. 8, free S), for many parameter sets at once.
//
// For one parameter set the loss terms are S_e = sum_c (E_c/N_c - E*_c)^2,
// S_v = sum_c sum_k (W_ck/N_c - W*_ck)^2 and S_f = sum_i |F_i - F*_i|^2 (Eq. 17-19 before the square
// root). Their gradients are
//   dS_e/dx = sum_c a_e dE/dx,               a_e = 2 (E/N - E*) / N,
//   dS_v/dx = sum_c sum_k a_k dW_k/dx = -d/dx sum_ij P_ij . (B d_ij),   a_k = 2 (W_k/N - W*_k) / N,
//   dS_f/dx = sum_i v_i . dF_i/dx = -d/dx sum_ij P_ij . (v_j - v_i),   v_i = 2 (F_i - F*_i),
// with P_ij = dU_i/dd_ij and (B d)_nu = sum_{k = (mu, nu)} a_k d_mu. The virial and force terms are
// derivatives of the site energies along fixed directions q_ij of the bonds, so an atom needs nothing
// but its own bonds, its weights and the v of its neighbours. Two steps:
//  * the batched kernel (gradient mode) evaluates every (parameter set, configuration) and leaves v,
//    the weights a_e, a_k and the residual terms;
//  * tangent_kernel forms, for every (atom, parameter set), the derivative of the site energy along the
//    two directions and the derivatives of that number with respect to the parameters, in closed form.
//
// Closed form. With R = f_R, T = b f_A, rho_j = u_j . q_j and cdot_jk = d cos_jk / dt along q,
//   zeta_j = sum_k f_k g_jk,   zdot_j = sum_k (f'_k rho_k g_jk + f_k g'_jk cdot_jk),
//   U_i   = 1/2 sum_j f_j (R_j - T_j),
//   Udot  = 1/2 sum_j [ Y_j R_j - X_j T_j - f_j T_j B_j zdot_j ],
//   X = rho (f' - mu f),  Y = rho (f' - lambda f),  B = b'/b,
// (f = f_C). The parameters enter through R and T (D0, alpha, r0, S), through zeta and zdot (the angular
// parameters) and through b(zeta; n):
//   dUdot/dzeta_j = -1/2 T B [X + f zdot (B + (n/(1 + zeta^n) - 1)/zeta)],   dUdot/dzdot_j = -1/2 f T B,
//   dUdot/dn      = -1/2 [X T b_n/b + f T B zdot b'_n/b'],
// and zeta and zdot are linear in beta (in gamma and gamma c^2/d^2). About 800 FLOP and 25 SFU operations
// per atom of four bonds, against ~9,300 FLOP for forward-mode dual numbers over the same per-atom core.
#include <math.h>

#include <algorithm>

#include "batch_kernel.cuh"

namespace tsf {

constexpr int kTanWarps = 8;
constexpr int kTanThreads = kTanWarps * 32;

struct TangentParams {
  int P;
  int64_t Ntot, ldP;              // ldP: parameter-set stride of v and aw
  int iters;                      // atoms per warp and atom slot
  int nchunks;                    // CTAs along the atoms
  const float *consts;            // [P][8] PConsts<float> ([P][16] in the Tersoff form)
  const double *params;           // [P][9] raw parameters (Tersoff form)
  const int *atom_cfg, *atom_off, *boff, *poff, *ameta;
  const float4 *gA, *gB;
  const float *gcos;
  const float *v;                 // [Ntot][3][ldP]
  const float *aw;                // [C][7][ldP]: a_e, a_k (k = xx .. zx)
  double *gsum;                   // [P][nchunks][NG]: gradient terms of every CTA's atoms
};

// Constants of one parameter set (one per lane). The sums of tangent_atom carry no D0; tangent_map applies
// it. kl = lambda / alpha, km = mu / alpha; beta sits in gcd (minimal form: zeta = gcd A1).
template <bool GEN>
struct TanConsts {
  float D0, k1, r0, h, n, inv2n, lam, mu, kl, km, gcd;
  float kR1, pR, pA, S, g0, d2, d, c;   // Tersoff form: f_R exponent, prefactors 1/(S-1), S/(S-1)
};

// Raw sums per loss term: 0 Y R, 1 X T + f T B zdot, 2 R (dr Y + rho f), 3 dr (X T + f T B zdot) + rho f T
// (dr = r - r0), 4 the n term, 5 and 6 the zeta terms over hc and over its u-derivative, and in the Tersoff
// form 7 over the constant term of g and 8 over the d-derivative. The parameter derivatives are linear in
// them (tangent_map), so the sums over atoms run over these few numbers.
template <bool GEN>
constexpr int kTanNS = GEN ? 9 : 7;
template <bool GEN>
constexpr int kTanNX = GEN ? 9 : 6;

// One atom (per atom slot) with bond arrays for M bonds; bonds past the atom's own count are phantoms
// (f = f' = 0, u = 0, r = 1), which contribute exactly zero. a: a_e, a_xx .. a_zx of the atom's
// configuration; jv: offset of v_j of each bond's partner in v; vx, vy, vz: v_i. G: the lane's
// sums [3 NS] in shared memory, 32 apart (in registers they cost spills at 128 registers). INNER: every bond is inside R1
// (f = 1, f' = 0).
template <int M, bool INNER, bool GEN>
__device__ __forceinline__ void tangent_atom(const float (&ux)[M], const float (&uy)[M], const float (&uz)[M],
                                             const float (&r)[M], const float (&ir2)[M], const float (&fc)[M],
                                             const float (&fcp)[M], const float *cs, const TanConsts<GEN> &K,
                                             const float (&a)[7], const float *__restrict__ v, int64_t ldP,
                                             const int64_t (&jv)[M], float vx, float vy, float vz,
                                             float *G) {
  constexpr int NS = kTanNS<GEN>, NP = M * (M - 1) / 2, NQ = NP > 0 ? NP : 1;
  // ---- angular sums over the other bonds: A1 = sum f hc, AH = sum f hp; minimal form hc = u^2, hp = u (half
  // of dhc/du); Tersoff form hc = u^2 / (d^2 + u^2), hp = dhc/du, A0 = sum f, AD = sum f dhc/dd
  float A1[M], AH[M], A0[GEN ? M : 1], AD[GEN ? M : 1], iv[GEN ? NQ : 1];
#pragma unroll
  for (int j = 0; j < M; ++j) {
    A1[j] = AH[j] = 0.f;
    if constexpr (GEN) A0[j] = AD[j] = 0.f;
  }
  {
    int q = 0;
#pragma unroll
    for (int j = 0; j < M; ++j)
#pragma unroll
      for (int k = j + 1; k < M; ++k) {
        const float u = cs[q] - K.h;
        float hc, hp;
        if constexpr (GEN) {
          iv[q] = rcp(u * u + K.d2);
          hc = u * u * iv[q];
          hp = 2.f * K.d2 * u * iv[q] * iv[q];
          const float hd = -2.f * K.d * hc * iv[q];
          A0[j] += fc[k];
          A0[k] += fc[j];
          AD[j] += fc[k] * hd;
          AD[k] += fc[j] * hd;
        } else {
          hc = u * u;
          hp = u;
        }
        A1[j] += fc[k] * hc;
        A1[k] += fc[j] * hc;
        AH[j] += fc[k] * hp;
        AH[k] += fc[j] * hp;
        ++q;
      }
  }
  // ---- per bond: R, T, dr, f T B, b_n/b, b'_n/b', kz = B + (n / (1 + zeta^n) - 1) / zeta; the energy term
  float R[M], T[M], dr[M], B[M], kz[M], bn[M], bpn[M];
  float s[NS];
#pragma unroll
  for (int k = 0; k < NS; ++k) s[k] = 0.f;
#pragma unroll
  for (int j = 0; j < M; ++j) {
    dr[j] = r[j] - K.r0;
    const float x = ex2(dr[j] * K.k1);
    float A, zr;
    if constexpr (GEN) {
      A = K.pA * x;
      R[j] = K.pR * ex2(dr[j] * K.kR1);
      zr = K.g0 * A0[j] + K.gcd * A1[j];
    } else {
      A = x + x;
      R[j] = x * x;
      zr = K.gcd * A1[j];
    }
    const bool live = zr > 1e-30f;                 // a vanishing zeta has no derivative terms (see bond_order)
    const float z = live ? zr : 1e-30f, iz = live ? rcp(z) : 0.f;
    const float L = lg2(z), zn = ex2(K.n * L), w = 1.f + zn, l2 = lg2(w), sw = rcp(w);
    T[j] = ex2(K.inv2n * l2) * A;
    B[j] = -0.5f * zn * sw * iz;
    kz[j] = B[j] + (K.n * sw - 1.f) * iz;
    const float sl = sw * L;
    bn[j] = 0.6931471806f * K.inv2n * (2.f * K.inv2n * l2 + zn * sl);
    bpn[j] = bn[j] + 0.6931471806f * sl;
    const float fR = fc[j] * R[j], fT = fc[j] * T[j], fTB = fT * B[j];
    s[0] += fR;
    s[1] += fT;
    s[2] += dr[j] * fR;
    s[3] += dr[j] * fT;
    s[4] += fT * bn[j];
    s[5] += fTB * A1[j];
    s[6] += fTB * AH[j];
    if constexpr (GEN) {
      s[7] += fTB * A0[j];
      s[8] += fTB * AD[j];
    }
  }
#pragma unroll
  for (int k = 0; k < NS; ++k) G[32 * k] += a[0] * s[k];
  // the f'-terms only exist for bonds beyond R1; the vote keeps them off the common path
  bool sw = false;
  if constexpr (!INNER) {
#pragma unroll
    for (int j = 0; j < M; ++j) sw |= (fcp[j] != 0.f);
    sw = __any_sync(0xffffffffu, sw);
  }
  // ---- the virial and the force direction
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    // rho_j and cd_jk = d cos_jk / dt, one bond's direction q_j at a time
    float rho[M], cd[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) cd[q] = 0.f;
#pragma unroll
    for (int j = 0; j < M; ++j) {
      float qx, qy, qz;
      if (t == 0) {   // W_xx, W_yy, W_zz, W_xy, W_yz, W_zx = -sum d_mu P_nu
        const float dx = r[j] * ux[j], dy = r[j] * uy[j], dz = r[j] * uz[j];
        qx = a[1] * dx + a[6] * dz;
        qy = a[2] * dy + a[4] * dx;
        qz = a[3] * dz + a[5] * dy;
      } else {
        qx = v[jv[j]] - vx;
        qy = v[jv[j] + ldP] - vy;
        qz = v[jv[j] + 2 * ldP] - vz;
      }
      rho[j] = qx * ux[j] + qy * uy[j] + qz * uz[j];
      const float hir = 0.5f * ir2[j];
#pragma unroll
      for (int k = 0; k < M; ++k)
        if (k != j) {
          const int lo = j < k ? j : k, hi = j < k ? k : j, q = lo * M - (lo * (lo + 1)) / 2 - lo - 1 + hi;
          cd[q] += hir * (qx * ux[k] + qy * uy[k] + qz * uz[k] - rho[j] * cs[q]);
        }
    }
    float B1[M], BH[M], B0[GEN ? M : 1], BD[GEN ? M : 1];
#pragma unroll
    for (int j = 0; j < M; ++j) {
      B1[j] = BH[j] = 0.f;
      if constexpr (GEN) B0[j] = BD[j] = 0.f;
    }
    int q = 0;
#pragma unroll
    for (int j = 0; j < M; ++j)
#pragma unroll
      for (int k = j + 1; k < M; ++k) {
        const float u = cs[q] - K.h;
        if constexpr (GEN) {
          const float v2 = iv[q] * iv[q], hc = u * u * iv[q], hp = 2.f * K.d2 * u * v2;
          const float hpp = 2.f * K.d2 * v2 * (1.f - 4.f * hc);
          const float hpd = 4.f * K.d * u * v2 * (1.f - 2.f * K.d2 * iv[q]);   // dhp/dd
          const float c1 = hp * cd[q], cH = hpp * cd[q], cD = hpd * cd[q];
          B1[j] += fc[k] * c1;
          B1[k] += fc[j] * c1;
          BH[j] += fc[k] * cH;
          BH[k] += fc[j] * cH;
          BD[j] += fc[k] * cD;
          BD[k] += fc[j] * cD;
          if (sw) {
            const float hd = -2.f * K.d * hc * iv[q], pj = fcp[j] * rho[j], pk = fcp[k] * rho[k];
            B0[j] += pk;
            B0[k] += pj;
            B1[j] += pk * hc;
            B1[k] += pj * hc;
            BH[j] += pk * hp;
            BH[k] += pj * hp;
            BD[j] += pk * hd;
            BD[k] += pj * hd;
          }
        } else {
          const float c1 = 2.f * u * cd[q];
          B1[j] += fc[k] * c1;
          B1[k] += fc[j] * c1;
          BH[j] += fc[k] * cd[q];
          BH[k] += fc[j] * cd[q];
          if (sw) {
            const float pj = fcp[j] * rho[j] * u, pk = fcp[k] * rho[k] * u;
            B1[j] += pk * u;
            B1[k] += pj * u;
            BH[j] += pk;
            BH[k] += pj;
          }
        }
        ++q;
      }
#pragma unroll
    for (int k = 0; k < NS; ++k) s[k] = 0.f;
#pragma unroll
    for (int j = 0; j < M; ++j) {
      float zd;
      if constexpr (GEN) zd = K.g0 * B0[j] + K.gcd * B1[j];
      else zd = K.gcd * B1[j];
      const float rf = rho[j] * fc[j], fz1 = fc[j] * zd;
      const float X = rho[j] * fcp[j] - K.mu * rf, Y = rho[j] * fcp[j] - K.lam * rf;
      const float TB = T[j] * B[j], Zd = fz1 * TB, Q = X * T[j] + Zd;
      s[0] += Y * R[j];
      s[1] += Q;
      s[2] += R[j] * (dr[j] * Y + rf);
      s[3] += dr[j] * Q + rf * T[j];
      s[4] += X * T[j] * bn[j] + Zd * bpn[j];
      const float w1 = TB * (X + fz1 * kz[j]), w2 = TB * fc[j];
      s[5] += w1 * A1[j] + w2 * B1[j];
      s[6] += w1 * AH[j] + w2 * BH[j];
      if constexpr (GEN) {
        s[7] += w1 * A0[j] + w2 * B0[j];
        s[8] += w1 * AD[j] + w2 * BD[j];
      }
    }
#pragma unroll
    for (int k = 0; k < NS; ++k) G[32 * ((1 + t) * NS + k)] += s[k];
  }
}

// The parameter derivatives of one loss term from its raw sums (sign included: the virial and force terms
// are minus the directional derivatives).
template <bool GEN>
__device__ __forceinline__ void tangent_map(const float *s, const TanConsts<GEN> &K, float sign,
                                            float (&g)[kTanNX<GEN>]) {
  const float c = 0.5f * sign, cD = c * K.D0;
  g[0] = c * (s[0] - s[1]);
  g[1] = cD * (K.km * s[3] - K.kl * s[2]);
  g[2] = cD * (K.lam * s[0] - K.mu * s[1]);
  if constexpr (GEN) {   // [D0, alpha, r0, S, n, h, gamma, c, d]
    const float iS1 = 1.f / (K.S - 1.f), i2S = 0.5f / K.S;
    g[3] = cD * (-iS1 * s[0] + 2.f * i2S * iS1 * s[1] - i2S * (K.lam * s[2] + K.mu * s[3]));
    g[4] = -cD * s[4];
    g[5] = cD * K.gcd * s[6];
    const float c2 = K.c * K.c, id = 1.f / K.d, id2 = 1.f / K.d2;
    g[6] = -cD * (s[7] + c2 * id2 * s[5]);
    g[7] = -cD * (2.f * K.g0 * K.c * id2) * s[5];
    g[8] = -cD * (K.gcd * s[8] - 2.f * K.gcd * id * s[5]);
  } else {               // [D0, alpha, r0, beta, n, h]
    g[3] = -cD * s[5];
    g[4] = -cD * s[4];
    g[5] = 2.f * cD * K.gcd * s[6];
  }
}

// Loads of one atom per atom slot (m bonds of its own, m <= M) and tangent_atom. EXACT: m = M.
template <int M, bool EXACT, bool INNER, bool GEN>
__device__ __forceinline__ void tangent_load(const TangentParams &a, int64_t i, int m, int cb, int64_t a0, int64_t p,
                                             const TanConsts<GEN> &K, const float (&aw)[7],
                                             float *G) {
  constexpr int NP = M * (M - 1) / 2;
  float ux[M], uy[M], uz[M], r[M], ir2[M], fc[M], fcp[M], cs[NP > 0 ? NP : 1];
  int64_t jv[M];
  const float *vi = a.v + i * 3 * a.ldP + p;
  const float vx = vi[0], vy = vi[a.ldP], vz = vi[2 * a.ldP];
#pragma unroll
  for (int j = 0; j < M; ++j) {
    ux[j] = uy[j] = uz[j] = ir2[j] = fc[j] = fcp[j] = 0.f;
    r[j] = 1.f;
    jv[j] = i * 3 * a.ldP + p;                     // a phantom bond's direction is zero
    if (EXACT || j < m) {
      const float4 A = a.gA[cb + j], Bv = a.gB[cb + j];
      ux[j] = A.x; uy[j] = A.y; uz[j] = A.z; r[j] = A.w;
      ir2[j] = Bv.x;
      fc[j] = INNER ? 1.f : Bv.y;
      fcp[j] = INNER ? 0.f : Bv.z;
      jv[j] = (a0 + (__float_as_int(Bv.w) >> 16)) * 3 * a.ldP + p;
    }
  }
  const float *gc = a.gcos + a.poff[i];
  if constexpr (EXACT) {
    constexpr int NP4 = (NP + 3) / 4;
    const float4 *c4 = reinterpret_cast<const float4 *>(gc);
#pragma unroll
    for (int q = 0; q < NP4; ++q) {
      const float4 v = c4[q];
      const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (4 * q + k < NP) cs[4 * q + k] = w[k];
    }
  } else {
    int q = 0;
#pragma unroll
    for (int j = 0; j < M; ++j)
#pragma unroll
      for (int k = j + 1; k < M; ++k) {
        cs[q] = k < m ? gc[j * m - (j * (j + 1)) / 2 - j - 1 + k] : 0.f;
        ++q;
      }
  }
  tangent_atom<M, INNER, GEN>(ux, uy, uz, r, ir2, fc, fcp, cs, K, aw, a.v, a.ldP, jv, vx, vy, vz, G);
}

// The long lists (5 to 8 bonds, rare in solids) as called functions, so that their arrays do not raise the
// register count of the kernel.
template <int M, bool GEN>
__device__ __noinline__ void tangent_long(const TangentParams &a, int64_t i, int m, int cb, int64_t a0, int64_t p,
                                          const TanConsts<GEN> &K, const float (&aw)[7], float *G) {
  tangent_load<M, false, false, GEN>(a, i, m, cb, a0, p, K, aw, G);
}

// Grid (chunks of kTanWarps * 32/PT * iters consecutive atoms, parameter tiles). A warp's lanes are 32/PT atom
// slots x PT parameter sets (PT = 16 or 8 for few or awkward numbers of sets). No shared-memory staging: bond
// records come through L1 as broadcasts, v is read in rows of parameter sets, and only the final sum over the
// CTA's warps goes through shared memory, so two CTAs of eight warps fit an SM (128 registers). Bound by
// instruction issue and FP32 latency.
template <int PT, bool GEN>
__global__ void __launch_bounds__(kTanThreads, 2) tangent_kernel(const TangentParams a) {
  constexpr int APW = 32 / PT, NX = kTanNX<GEN>, NS = kTanNS<GEN>, NG = 3 * NX;
  __shared__ float acc[kTanWarps][3 * NS][32];      // the lanes' sums, then the warps' gradient terms
  static_assert(NG <= 3 * NS, "the gradient terms replace the sums");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, slot = lane / PT, pl = lane % PT;
  const int64_t p = (int64_t)blockIdx.y * PT + pl;
  pdl_wait();                                      // constants, v and weights of the kernels before
  TanConsts<GEN> K = {};
  {
    const int64_t pc = p < a.P ? p : a.P - 1;
    const float4 *kc = reinterpret_cast<const float4 *>(a.consts) + (GEN ? 4 : 2) * pc;
    const float4 k0 = kc[0], k1 = kc[1];
    K.k1 = k0.y; K.r0 = k0.z; K.h = k1.y; K.n = k1.z; K.inv2n = k1.w;
    if constexpr (GEN) {
      const float4 k2 = kc[2], k3 = kc[3];
      const double *x = a.params + 9 * pc;
      K.D0 = (float)x[0];
      K.S = (float)x[3];
      K.c = (float)x[7];
      K.d = (float)x[8];
      K.pR = 1.f / (K.S - 1.f);
      K.pA = K.S * K.pR;
      K.kl = sqrtf(2.f * K.S);
      K.km = sqrtf(2.f / K.S);
      K.mu = k0.w;
      K.lam = -2.f * k2.w;
      K.kR1 = k2.y;
      K.g0 = k3.x; K.d2 = k3.z; K.gcd = k3.w;
    } else {
      K.D0 = k0.x;
      K.gcd = k1.x;
      K.mu = -2.f * k0.w;                          // alpha
      K.lam = K.mu + K.mu;
      K.kl = 2.f;
      K.km = 1.f;
    }
  }
  float *G = &acc[warp][0][lane];
#pragma unroll
  for (int k = 0; k < 3 * NS; ++k) G[32 * k] = 0.f;
  const int64_t i0 = (int64_t)blockIdx.x * (kTanWarps * APW) * a.iters + warp * APW;
  for (int t = 0; t < a.iters; ++t) {
    const int64_t w0 = i0 + (int64_t)t * (kTanWarps * APW);
    if (w0 >= a.Ntot) break;                       // whole warps
    const bool valid = w0 + slot < a.Ntot;
    const int64_t i = valid ? w0 + slot : a.Ntot - 1;
    const int am = a.ameta[i], c = a.atom_cfg[i], cb = a.boff[i];
    const int m = valid ? am & 0xffff : 0;         // an atom beyond the end: phantoms only
    const int64_t a0 = a.atom_off[c];
    float aw[7];
    const float *wp = a.aw + (int64_t)c * 7 * a.ldP + p;
#pragma unroll
    for (int k = 0; k < 7; ++k) aw[k] = wp[k * a.ldP];
    const int Mw = PT == 32 ? m : (int)__reduce_max_sync(0xffffffffu, (unsigned)m);
    const bool inner = PT == 32 && (am >> 16) == 0;   // every bond inside R1 (one atom per warp)
    switch (Mw) {
#define TSF_TAN(MM)                                                                              \
  case MM:                                                                                       \
    if (inner) tangent_load<MM, true, PT == 32, GEN>(a, i, m, cb, a0, p, K, aw, G);              \
    else tangent_load<MM, PT == 32, false, GEN>(a, i, m, cb, a0, p, K, aw, G);                   \
    break;
      TSF_TAN(1) TSF_TAN(2) TSF_TAN(3) TSF_TAN(4)
#undef TSF_TAN
      case 5: case 6: tangent_long<6, GEN>(a, i, m, cb, a0, p, K, aw, G); break;
      case 7: case 8: tangent_long<8, GEN>(a, i, m, cb, a0, p, K, aw, G); break;
      default: break;                              // no bonds (more than 8 were refused before the launch)
    }
  }
  // the lanes of one parameter set over the atom slots, the parameter derivatives, then the warps' FP32 sums
  // added exactly and rounded once to FP64
  float sums[3 * NS];
#pragma unroll
  for (int k = 0; k < 3 * NS; ++k) sums[k] = sum_over_atom_slots<PT>(G[32 * k]);
  __syncwarp();
  if (slot == 0) {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      float g[NX];
      tangent_map<GEN>(sums + q * NS, K, q == 0 ? 1.f : -1.f, g);
#pragma unroll
      for (int x = 0; x < NX; ++x) G[32 * (q * NX + x)] = g[x];
    }
  }
  __syncthreads();
  for (int t = tid; t < NG * PT; t += kTanThreads) {
    const int lp = t / NG, k = t % NG;
    const int64_t pp = (int64_t)blockIdx.y * PT + lp;
    float xw[kTanWarps];
#pragma unroll
    for (int w = 0; w < kTanWarps; ++w) xw[w] = acc[w][k][lp];
    if (pp < a.P) a.gsum[(pp * a.nchunks + blockIdx.x) * NG + k] = exact_sum<kTanWarps>(xw);
  }
}

// One CTA per parameter set: S_q and D_q over the configurations, G_q = dS_q/dx over the chunks (FP64, a fixed
// order: each thread strided, then the threads' sums in order), then L and dL/dx for the squared loss
// (w_q S_q / D_q) or Z (w_q sqrt(S_q / D_q)). One warp per set with all its sums in registers took 24 us at
// P = 64, C = 100 (13 to 64 warps on the whole chip, a serial chain of FP64 additions each), 9.6 with every lane of eight
// warps adding all six sums, 8.1 so (warp_sums8).
constexpr int kGradFinThreads = 256;
template <int NX>
__global__ void __launch_bounds__(kGradFinThreads) grad_finalize_kernel(
    int P, int C, int nchunks, const double *__restrict__ part, const double *__restrict__ dpart,
    const double *__restrict__ gsum, double we, double wv, double wf, int loss, double *__restrict__ L,
    double *__restrict__ dL) {
  constexpr int NG = 3 * NX, kRows = kGradFinThreads / NG, kWarps = kGradFinThreads / 32;
  __shared__ double s_g[kRows][NG], s_sd[kWarps][6], s_c[3];
  __shared__ int s_finite;
  pdl_wait();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, p = blockIdx.x;
  double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};    // S_e, S_v, S_f, D_e, D_v, D_f
  for (int c = tid; c < C; c += kGradFinThreads)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      v[q] += part[((size_t)p * C + c) * 3 + q];
      v[3 + q] += dpart[(size_t)c * 3 + q];
    }
  double w8[8] = {v[0], v[1], v[2], v[3], v[4], v[5], 0.0, 0.0};
  const double t8 = warp_sums8(w8);
  if ((lane & 3) == 0 && lane < 24) s_sd[warp][lane >> 2] = t8;
  if (tid < kRows * NG) {                          // consecutive threads read consecutive terms of the chunks
    double g = 0.0;
    const double *src = gsum + (size_t)p * nchunks * NG;
#pragma unroll 4
    for (int64_t t = tid; t < (int64_t)nchunks * NG; t += kRows * NG) g += src[t];
    s_g[tid / NG][tid % NG] = g;
  }
  __syncthreads();
  if (tid < 3) {
    double s = 0.0, d = 0.0;
    for (int w = 0; w < kWarps; ++w) {
      s += s_sd[w][tid];
      d += s_sd[w][3 + tid];
    }
    const double wq = tid == 0 ? we : tid == 1 ? wv : wf;
    double l = 0.0, cq = 0.0;
    if (d > 0.0) {
      if (loss == TERSOFF_LOSS_SQ) {
        cq = wq / d;
        l = wq * s / d;
      } else {
        l = wq * sqrt(s / d);
        cq = s > 0.0 ? wq / (2.0 * sqrt(s * d)) : 0.0;
      }
    }
    s_c[tid] = cq;
    const bool finite = __all_sync(0x7u, isfinite(s));
    const double l1 = __shfl_sync(0x7u, l, 1), l2 = __shfl_sync(0x7u, l, 2);
    if (tid == 0) {
      s_finite = finite;
      L[p] = finite ? (l + l1) + l2 : INFINITY;
    }
  }
  if (tid >= 32 && tid < 32 + NG) {
    double g = 0.0;
    for (int w = 0; w < kRows; ++w) g += s_g[w][tid - 32];
    s_g[0][tid - 32] = g;
  }
  __syncthreads();
  if (tid < NX) {
    double gx = 0.0;
    for (int q = 0; q < 3; ++q) gx += s_c[q] * s_g[0][q * NX + tid];
    dL[(size_t)p * NX + tid] = s_finite ? gx : __longlong_as_double(0x7ff8000000000000ll);
  }
}

// ---------------------------------------------------------------------------------------------
// Parameter sets per tile of the tangent kernel: the width with the least padded work. Narrow tiles read their
// geometry per atom slot instead of as broadcasts and run the longest list of their slots; at P = 13 (one Newton
// iteration) a 16-wide tile does 16 lanes' work instead of 32. What narrow tiles cost, on full ones of 32, 16 and 8 sets
// (192 sets): 61.0, 63.2 and 65.2 us on 100 cells of 64 atoms, 134, 130 and 157 us on 100 mixed cells; with 96 sets 37.8,
// 37.4 and 35.8, and 74.9, 73.8 and 87.8 us. The weights 1.08 and 1.15 are at the upper end of the first and about the
// second, so a narrower tile is taken only where it saves more lanes than that.
static int tangent_tile(int P) {
  const double c32 = (P + 31) / 32 * 32, c16 = 1.08 * ((P + 15) / 16 * 16), c8 = 1.15 * ((P + 7) / 8 * 8);
  return c32 <= c16 && c32 <= c8 ? 32 : (c16 <= c8 ? 16 : 8);
}

template <int PT, bool GEN>
static cudaError_t launch_tangent(const TangentParams &a, dim3 grid, bool pdl, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kTanThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, tangent_kernel<PT, GEN>, a);
  if (e == cudaSuccess) count_launches(1);
  return e;
}

// Parameter sets handled by one launch sequence: all of them, or blocks of a multiple of 32 so that v stays
// within 1 GiB and the tiles (32 wide for blocks of that size) within a grid's 65,535 rows.
int grad_block(int64_t Ntot, int P) {
  const int64_t most = std::min<int64_t>(65535, std::max<int64_t>(1, (int64_t{1} << 30) / (Ntot * 12 * 32))) * 32;
  return (int)std::min<int64_t>(P, most);
}
GradPlan grad_plan(const Ctx &ctx, int P) {
  GradPlan g;
  g.block = grad_block(ctx.Ntot, P);
  g.tile = tangent_tile(g.block);
  g.ldP = (int64_t)(g.block + g.tile - 1) / g.tile * g.tile;
  // atoms per warp and slot: as many as leave about four CTAs per SM (two run at a time), at most eight
  const int64_t apc = (int64_t)kTanWarps * (32 / g.tile), ntiles = g.ldP / g.tile;
  const int64_t ctas = (ctx.Ntot + apc - 1) / apc * ntiles;
  g.iters = (int)std::min<int64_t>(8, std::max<int64_t>(1, ctas / (4 * ctx.nsm)));
  g.nchunks = (int)((ctx.Ntot + apc * g.iters - 1) / (apc * g.iters));
  return g;
}

// The gradient of the parameter sets p0 .. p0 + P - 1 (P <= the plan's block).
cudaError_t launch_param_grad(const Ctx &ctx, const GradPlan &gp, const double *params, int P, const BatchOut &o,
                              const double *w, int loss, double *gsum, double *L, double *dL, cudaStream_t s) {
  cudaError_t e = launch_batch(ctx, ctx.plan32, params, P, kModeGrad, o, s);
  if (e != cudaSuccess) return e;
  const bool gen = ctx.form == kFormTersoff;
  TangentParams a = {};
  a.P = P;
  a.Ntot = ctx.Ntot;
  a.ldP = gp.ldP;
  a.iters = gp.iters;
  a.nchunks = gp.nchunks;
  a.consts = reinterpret_cast<const float *>(o.consts);
  a.params = params;
  a.atom_cfg = ctx.atom_cfg.as<int>();
  a.atom_off = ctx.atom_off.as<int>();
  a.boff = ctx.boff.as<int>();
  a.poff = ctx.poff.as<int>();
  a.ameta = ctx.ameta.as<int>();
  a.gA = ctx.gA32.as<float4>();
  a.gB = ctx.gB32.as<float4>();
  a.gcos = ctx.gcos32.as<float>();
  a.v = static_cast<const float *>(o.F);
  a.aw = o.aw;
  a.gsum = gsum;
  const dim3 grid((unsigned)gp.nchunks, (unsigned)((P + gp.tile - 1) / gp.tile));
  if (gp.tile == 32) e = gen ? launch_tangent<32, true>(a, grid, o.pdl, s) : launch_tangent<32, false>(a, grid, o.pdl, s);
  else if (gp.tile == 16) e = gen ? launch_tangent<16, true>(a, grid, o.pdl, s) : launch_tangent<16, false>(a, grid, o.pdl, s);
  else e = gen ? launch_tangent<8, true>(a, grid, o.pdl, s) : launch_tangent<8, false>(a, grid, o.pdl, s);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)P);
  cfg.blockDim = dim3(kGradFinThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = o.pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = gen ? cudaLaunchKernelEx(&cfg, grad_finalize_kernel<9>, P, ctx.C, gp.nchunks, (const double *)o.part,
                               (const double *)o.dpart, (const double *)gsum, w[0], w[1], w[2], loss, L, dL)
          : cudaLaunchKernelEx(&cfg, grad_finalize_kernel<6>, P, ctx.C, gp.nchunks, (const double *)o.part,
                               (const double *)o.dpart, (const double *)gsum, w[0], w[1], w[2], loss, L, dL);
  if (e == cudaSuccess) count_launches(1);
  return e;
}

}  // namespace tsf
