// Device functions shared by the brick kernels (bm_kernels.cu: any particle
// arrangement; bm_lattice.cu: particles on a lattice): B-spline weights,
// stresses, contact, side labels, brick geometry and the per-particle work
// ahead of P2G.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "bm_internal.cuh"

#define FULL 0xffffffffu

namespace {

// --------------------------------------------------------------------------
// quadratic B-spline of Eq. 1: weight and d/dxl of node base+o, o in {0,1,2},
// for a particle at fractional offset f = xl - base in [0.5, 1.5)
// --------------------------------------------------------------------------
template <int O>
__device__ __forceinline__ void bs(float f, float &w, float &dw) {
  if (O == 0) {
    float t = 1.5f - f;
    w = 0.5f * t * t;
    dw = -t;
  } else if (O == 1) {
    float t = f - 1.0f;
    w = 0.75f - t * t;
    dw = -2.0f * t;
  } else {
    float t = f - 0.5f;
    w = 0.5f * t * t;
    dw = t;
  }
}

__device__ __forceinline__ void bs_rt(int o, float f, float &w, float &dw) {
  if (o == 0) bs<0>(f, w, dw);
  else if (o == 1) bs<1>(f, w, dw);
  else bs<2>(f, w, dw);
}

__device__ __forceinline__ bool conflict(uint32_t a1, uint32_t a2, uint32_t b1, uint32_t b2) {
  return ((a1 & b2) | (a2 & b1)) != 0u;
}

// --------------------------------------------------------------------------
// neo-Hookean first Piola-Kirchhoff stress, P = mu (F - F^-T) + lam ln J F^-T
// --------------------------------------------------------------------------
__device__ __forceinline__ bool piola(const float F[9], float mu, float lam, float P[9]) {
  float c[9];
  c[0] = F[4] * F[8] - F[5] * F[7];
  c[1] = F[5] * F[6] - F[3] * F[8];
  c[2] = F[3] * F[7] - F[4] * F[6];
  c[3] = F[2] * F[7] - F[1] * F[8];
  c[4] = F[0] * F[8] - F[2] * F[6];
  c[5] = F[1] * F[6] - F[0] * F[7];
  c[6] = F[1] * F[5] - F[2] * F[4];
  c[7] = F[2] * F[3] - F[0] * F[5];
  c[8] = F[0] * F[4] - F[1] * F[3];
  float J = F[0] * c[0] + F[1] * c[1] + F[2] * c[2];
  bool clamped = false;
  if (!(J > 1e-6f)) {
    J = 1e-6f;
    clamped = true;
  }
  float iJ = 1.0f / J;
  float lj = logf(J);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    float FinvT = c[k] * iJ;
    P[k] = mu * (F[k] - FinvT) + lam * lj * FinvT;
  }
  return clamped;
}

// --------------------------------------------------------------------------
// fixed-corotated stress, P = 2 mu (F - R) + lam (J - 1) J F^-T, with the
// rotation R of the polar decomposition F = R S from Newton's iteration
// R <- (g R + R^-T / g) / 2 (g = (|R^-1| / |R|)^(1/2), Frobenius norms),
// which converges quadratically to R for det F > 0.
// --------------------------------------------------------------------------
__device__ __forceinline__ void cof3(const float F[9], float c[9]) {
  c[0] = F[4] * F[8] - F[5] * F[7];
  c[1] = F[5] * F[6] - F[3] * F[8];
  c[2] = F[3] * F[7] - F[4] * F[6];
  c[3] = F[2] * F[7] - F[1] * F[8];
  c[4] = F[0] * F[8] - F[2] * F[6];
  c[5] = F[1] * F[6] - F[0] * F[7];
  c[6] = F[1] * F[5] - F[2] * F[4];
  c[7] = F[2] * F[3] - F[0] * F[5];
  c[8] = F[0] * F[4] - F[1] * F[3];
}

__device__ bool piola_fcr(const float F[9], float mu, float lam, float P[9]) {
  float c[9];
  cof3(F, c);
  const float J = F[0] * c[0] + F[1] * c[1] + F[2] * c[2];
  const bool clamped = !(J > 1e-6f);
  float R[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) R[k] = F[k];
  for (int it = 0; it < 16; ++it) {
    float q[9];
    cof3(R, q);
    const float d = R[0] * q[0] + R[1] * q[1] + R[2] * q[2];  // R^-T = cof(R) / det R
    if (d == 0.0f) break;
    const float id = 1.0f / d;
    float nr = 0.f, ni = 0.f;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      q[k] *= id;
      nr += R[k] * R[k];
      ni += q[k] * q[k];
    }
    const float g = sqrtf(sqrtf(ni / nr));
    const float ig = 1.0f / g;
    float dif = 0.f;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const float r = 0.5f * (g * R[k] + ig * q[k]);
      dif += (r - R[k]) * (r - R[k]);
      R[k] = r;
    }
    if (dif <= 1e-13f) break;
  }
  const float jl = lam * (J - 1.0f);
#pragma unroll
  for (int k = 0; k < 9; ++k) P[k] = 2.0f * mu * (F[k] - R[k]) + jl * c[k];
  return clamped;
}

__device__ __forceinline__ void mat3mul(const float A[9], const float B[9], float C[9]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) C[3 * i + j] = A[3 * i] * B[j] + A[3 * i + 1] * B[3 + j] + A[3 * i + 2] * B[6 + j];
}

// symmetric 3x3 eigen-decomposition A = V diag(w) V^T by cyclic Jacobi
// rotations (float32, at most 10 sweeps)
__device__ void sym_eig3(const float Ain[9], float V[9], float w[3]) {
  float A[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    A[k] = Ain[k];
    V[k] = (k % 4 == 0) ? 1.0f : 0.0f;
  }
  for (int sweep = 0; sweep < 10; ++sweep) {
    const float off = A[1] * A[1] + A[2] * A[2] + A[5] * A[5];
    const float dg = A[0] * A[0] + A[4] * A[4] + A[8] * A[8];
    if (!(off > 1e-14f * dg)) break;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int p = r == 2 ? 1 : 0, q = r == 0 ? 1 : 2;
      const float apq = A[3 * p + q];
      if (apq == 0.0f) continue;
      const float th = (A[3 * q + q] - A[3 * p + p]) / (2.0f * apq);
      const float t = copysignf(1.0f, th) / (fabsf(th) + sqrtf(th * th + 1.0f));
      const float c = 1.0f / sqrtf(t * t + 1.0f), sn = t * c;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float akp = A[3 * k + p], akq = A[3 * k + q];
        A[3 * k + p] = c * akp - sn * akq;
        A[3 * k + q] = sn * akp + c * akq;
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float apk = A[3 * p + k], aqk = A[3 * q + k];
        A[3 * p + k] = c * apk - sn * aqk;
        A[3 * q + k] = sn * apk + c * aqk;
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float vkp = V[3 * k + p], vkq = V[3 * k + q];
        V[3 * k + p] = c * vkp - sn * vkq;
        V[3 * k + q] = sn * vkp + c * vkq;
      }
    }
  }
  w[0] = A[0];
  w[1] = A[4];
  w[2] = A[8];
}

// von Mises plasticity: radial return of the deviatoric principal Hencky
// strains e of Fe onto sqrt(3/2) |2 mu e| = sigma_y (isochoric).  Returns
// whether Fe was projected.
__device__ bool vonmises(float Fe[9], float mu, float sy) {
  float C[9];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) C[3 * i + j] = Fe[i] * Fe[j] + Fe[3 + i] * Fe[3 + j] + Fe[6 + i] * Fe[6 + j];
  float V[9], w[3];
  sym_eig3(C, V, w);
  if (!(w[0] > 0.f) || !(w[1] > 0.f) || !(w[2] > 0.f)) return false;
  float sg[3], e[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    sg[k] = sqrtf(w[k]);
    e[k] = logf(sg[k]);
  }
  const float mean = (e[0] + e[1] + e[2]) * (1.0f / 3.0f);
#pragma unroll
  for (int k = 0; k < 3; ++k) e[k] -= mean;
  const float q = 2.4494897f * mu * sqrtf(e[0] * e[0] + e[1] * e[1] + e[2] * e[2]);  // sqrt(6) mu |e|
  if (!(q > sy)) return false;
  const float sc = sy / q;
  float rt[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) rt[k] = expf(mean + sc * e[k]) / sg[k];
  float M[9];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      M[3 * i + j] = V[3 * i] * rt[0] * V[3 * j] + V[3 * i + 1] * rt[1] * V[3 * j + 1] +
                     V[3 * i + 2] * rt[2] * V[3 * j + 2];
  float out[9];
  mat3mul(Fe, M, out);
#pragma unroll
  for (int k = 0; k < 9; ++k) Fe[k] = out[k];
  return true;
}

// Stress of a particle of a scene with plasticity or viscosity (kept out of
// line so that the elastic path keeps its registers): plastic projection of
// Fe = F Fp^-1 with Fp^-1 = F^-1 Fe stored back, P = P(Fe) Fp^-T, and the
// viscous part J eta (L + L^T) F^-T with L = dF/dt F^-1 of the last substep.
__device__ __noinline__ bool inelastic_stress(const DevScene &sc, const PPool &P, int p, const float F[9],
                                              float Pk[9]) {
  bool clamped = false;
  if (sc.yield_stress > 0.0f) {
    // Fe = F Fp^-1, projected; Fp^-1 = F^-1 Fe; P = P(Fe) Fp^-T
    float Fpi[9], Fe[9], Pe[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) Fpi[k] = P.Fpi[k][p];
    mat3mul(F, Fpi, Fe);
    if (vonmises(Fe, sc.mu, sc.yield_stress)) {
      float c[9];
      cof3(F, c);
      const float d = F[0] * c[0] + F[1] * c[1] + F[2] * c[2];
      if (d != 0.0f) {
        const float id = 1.0f / d;
        float Fi[9] = {c[0] * id, c[3] * id, c[6] * id, c[1] * id, c[4] * id,
                       c[7] * id, c[2] * id, c[5] * id, c[8] * id};  // F^-1 = cof(F)^T / det F
        mat3mul(Fi, Fe, Fpi);
#pragma unroll
        for (int k = 0; k < 9; ++k) P.Fpi[k][p] = Fpi[k];
      }
    }
    clamped |= sc.model == BM_MODEL_FIXED_COROTATED ? piola_fcr(Fe, sc.mu, sc.lam, Pe)
                                                    : piola(Fe, sc.mu, sc.lam, Pe);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        Pk[3 * i + j] = Pe[3 * i] * Fpi[3 * j] + Pe[3 * i + 1] * Fpi[3 * j + 1] + Pe[3 * i + 2] * Fpi[3 * j + 2];
  } else {
    clamped |= sc.model == BM_MODEL_FIXED_COROTATED ? piola_fcr(F, sc.mu, sc.lam, Pk)
                                                    : piola(F, sc.mu, sc.lam, Pk);
  }
  if (sc.viscosity > 0.0f) {
    // Cauchy eta (L + L^T), L = dF/dt F^-1 (last substep), as J sigma F^-T = sigma cof(F)
    float c[9], Fd[9], L[9];
    cof3(F, c);
    const float d = F[0] * c[0] + F[1] * c[1] + F[2] * c[2];
    if (d != 0.0f) {
      const float id = 1.0f / d;
      const float Fi[9] = {c[0] * id, c[3] * id, c[6] * id, c[1] * id, c[4] * id,
                           c[7] * id, c[2] * id, c[5] * id, c[8] * id};
#pragma unroll
      for (int k = 0; k < 9; ++k) Fd[k] = P.Fdot[k][p];
      mat3mul(Fd, Fi, L);
      float sv[9];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) sv[3 * i + j] = sc.viscosity * (L[3 * i + j] + L[3 * j + i]);
      float add[9];
      mat3mul(sv, c, add);
#pragma unroll
      for (int k = 0; k < 9; ++k) Pk[k] += add[k];
    }
  }
  return clamped;
}

// --------------------------------------------------------------------------
// Eq. 12: spring-history Coulomb friction (float32)
// --------------------------------------------------------------------------
__device__ __forceinline__ void friction(const float uh[3], const float n[3], const float vrel[3],
                                         float fn, float meff, float dt, float gk, float gc,
                                         float mus, float mud, float ft[3], float un[3]) {
  float udn = uh[0] * n[0] + uh[1] * n[1] + uh[2] * n[2];
  float ul = sqrtf(uh[0] * uh[0] + uh[1] * uh[1] + uh[2] * uh[2]);
  float tu[3] = {uh[0] - udn * n[0], uh[1] - udn * n[1], uh[2] - udn * n[2]};
  float tl = sqrtf(tu[0] * tu[0] + tu[1] * tu[1] + tu[2] * tu[2]);
  float sc = tl > 0.0f ? ul / tl : 0.0f;
  float ut[3] = {tu[0] * sc, tu[1] * sc, tu[2] * sc};
  float vn = vrel[0] * n[0] + vrel[1] * n[1] + vrel[2] * n[2];
  float vt[3] = {vrel[0] - vn * n[0], vrel[1] - vn * n[1], vrel[2] - vn * n[2]};
  float kt = gk * meff / (dt * dt);
  float ct = 2.0f * gc * sqrtf(meff * kt);
  float ftr[3] = {-kt * ut[0] - ct * vt[0], -kt * ut[1] - ct * vt[1], -kt * ut[2] - ct * vt[2]};
  float fl = sqrtf(ftr[0] * ftr[0] + ftr[1] * ftr[1] + ftr[2] * ftr[2]);
  if (fl <= mus * fn) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      ft[i] = ftr[i];
      un[i] = ut[i] + dt * vt[i];
    }
  } else {
    float s = mud * fn / fl;
    float ikt = 1.0f / kt;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      ft[i] = s * ftr[i];
      un[i] = -(ft[i] + ct * vt[i]) * ikt;
    }
  }
}

// --------------------------------------------------------------------------
// blade box: closest point, outward normal, sphere gap (float32)
// --------------------------------------------------------------------------
__device__ __forceinline__ void box_closest(const DevScene &sc, const float x[3], float R,
                                            float xc[3], float nB[3], float &phi) {
  const float *ax[3] = {sc.fn, sc.fe, sc.fd};
  float r[3] = {x[0] - sc.fc[0], x[1] - sc.fc[1], x[2] - sc.fc[2]};
  float q[3], qc[3], nl[3] = {0.f, 0.f, 0.f};
  bool outside = false;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    q[a] = r[0] * ax[a][0] + r[1] * ax[a][1] + r[2] * ax[a][2];
    outside |= fabsf(q[a]) > sc.fhext[a];
  }
  if (outside) {
    float diff[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      qc[a] = fminf(fmaxf(q[a], -sc.fhext[a]), sc.fhext[a]);
      diff[a] = q[a] - qc[a];
    }
    float dist = sqrtf(diff[0] * diff[0] + diff[1] * diff[1] + diff[2] * diff[2]);
    float id = 1.0f / dist;
#pragma unroll
    for (int a = 0; a < 3; ++a) nl[a] = diff[a] * id;
    phi = dist - R;
  } else {
    int best = 0;
    float bd = sc.fhext[0] - fabsf(q[0]);
#pragma unroll
    for (int a = 1; a < 3; ++a) {
      float dd = sc.fhext[a] - fabsf(q[a]);
      if (dd < bd) {
        bd = dd;
        best = a;
      }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) qc[a] = q[a];
    float sg = q[best] < 0.0f ? -1.0f : 1.0f;
    qc[best] = sg * sc.fhext[best];
    nl[best] = sg;
    phi = -bd - R;
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    xc[i] = sc.fc[i] + qc[0] * ax[0][i] + qc[1] * ax[1][i] + qc[2] * ax[2][i];
    nB[i] = nl[0] * ax[0][i] + nl[1] * ax[1][i] + nl[2] * ax[2][i];
  }
}

// --------------------------------------------------------------------------
// Eq. 3, 4, 6 side label.  float32 filter with a forward-error bound; within
// the bound of any threshold the decision is re-taken in float64 with every
// operation rounded separately, in the order of a plain double evaluation:
// r = x - x_e; s = (r0 n0 + r1 n1) + r2 n2; (same for l, f);
// u_c = ((ve0-v0) d0 + (ve1-v1) d1) + (ve2-v2) d2; lowb = -b_back - max(u_c dt, 0).
// --------------------------------------------------------------------------
__device__ __noinline__ int side_label_exact(const DevScene &sc, const float xf[3],
                                             const float vf[3]) {
  double x0 = xf[0], x1 = xf[1], x2 = xf[2];
  double r0 = __dsub_rn(x0, sc.dxe[0]), r1 = __dsub_rn(x1, sc.dxe[1]), r2 = __dsub_rn(x2, sc.dxe[2]);
  double s = __dadd_rn(__dadd_rn(__dmul_rn(r0, sc.dn[0]), __dmul_rn(r1, sc.dn[1])), __dmul_rn(r2, sc.dn[2]));
  double l = __dadd_rn(__dadd_rn(__dmul_rn(r0, sc.de[0]), __dmul_rn(r1, sc.de[1])), __dmul_rn(r2, sc.de[2]));
  double f = __dadd_rn(__dadd_rn(__dmul_rn(r0, sc.dd[0]), __dmul_rn(r1, sc.dd[1])), __dmul_rn(r2, sc.dd[2]));
  double u0 = __dsub_rn(sc.dve[0], (double)vf[0]);
  double u1 = __dsub_rn(sc.dve[1], (double)vf[1]);
  double u2 = __dsub_rn(sc.dve[2], (double)vf[2]);
  double uc = __dadd_rn(__dadd_rn(__dmul_rn(u0, sc.dd[0]), __dmul_rn(u1, sc.dd[1])), __dmul_rn(u2, sc.dd[2]));
  double ucdt = __dmul_rn(uc, sc.dt_d);
  double lowb = __dsub_rn(-sc.b_back_d, ucdt > 0.0 ? ucdt : 0.0);
  bool band = fabs(s) <= sc.h_d && fabs(l) <= sc.L_d && lowb <= f && f <= sc.b_lead_d;
  if (!band || !(f <= 0.0)) return 0;
  return s < 0.0 ? 1 : 2;
}

__device__ __forceinline__ int side_label(const DevScene &sc, const float x[3], const float v[3]) {
  const float r0 = x[0] - sc.fxe[0], r1 = x[1] - sc.fxe[1], r2 = x[2] - sc.fxe[2];
  const float s = r0 * sc.fn[0] + r1 * sc.fn[1] + r2 * sc.fn[2];
  // forward-error bounds (2^-20 = 16 u, generous over the ~5 u analysis)
  const float k = 9.5367431640625e-07f;
  const float mag = fabsf(x[0]) + fabsf(x[1]) + fabsf(x[2]) +
                    2.0f * (fabsf(sc.fxe[0]) + fabsf(sc.fxe[1]) + fabsf(sc.fxe[2]));
  const float E = k * mag + 1e-30f;
  const float as = fabsf(s);
  // beyond the band's half-width by more than the bound: outside the band
  // in float64 too (the decision below and the exact path both give 0)
  if (as > sc.h + (E + k * sc.h)) return 0;
  const float l = r0 * sc.fe[0] + r1 * sc.fe[1] + r2 * sc.fe[2];
  const float f = r0 * sc.fd[0] + r1 * sc.fd[1] + r2 * sc.fd[2];
  const float uc = (sc.fve[0] - v[0]) * sc.fd[0] + (sc.fve[1] - v[1]) * sc.fd[1] +
                   (sc.fve[2] - v[2]) * sc.fd[2];
  const float ucdt = uc * sc.dt;
  const float lowb = -sc.b_back - fmaxf(ucdt, 0.0f);
  const float Eu = k * ((fabsf(sc.fve[0]) + fabsf(sc.fve[1]) + fabsf(sc.fve[2]) + fabsf(v[0]) +
                         fabsf(v[1]) + fabsf(v[2])) * sc.dt + sc.b_back + fabsf(ucdt));
  const float al = fabsf(l);
  const bool near = as <= E || fabsf(as - sc.h) <= E + k * sc.h || fabsf(al - sc.fL) <= E + k * sc.fL ||
                    fabsf(f) <= E || fabsf(f - sc.b_lead) <= E + k * sc.b_lead ||
                    fabsf(f - lowb) <= E + Eu;
  if (near) return side_label_exact(sc, x, v);
  const bool band = as <= sc.h && al <= sc.fL && lowb <= f && f <= sc.b_lead;
  if (!band || !(f <= 0.0f)) return 0;
  return s < 0.0f ? 1 : 2;
}

// exclusive block scan of one int per thread (fixed order); total in all threads
__device__ __forceinline__ int block_excl_scan(int v, int *sm, int &total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(FULL, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();
  if (lane == 31) sm[wid] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int i = 0; i < nw; ++i) {
      int t = sm[i];
      sm[i] = acc;
      acc += t;
    }
    sm[nw] = acc;
  }
  __syncthreads();
  total = sm[nw];
  return x - v + sm[wid];
}

// --------------------------------------------------------------------------
// Brick geometry.  Particles are stored brick-major: bricks of 4x4x4 base
// cells, cells x-fastest inside a brick, so a brick's particles form one
// contiguous range.  A brick's particles touch the 6x6x6 node tile starting
// at its first cell (quadratic stencil: nodes base..base+2).
// --------------------------------------------------------------------------
#define BR 4
#define BR3 64
#define TE 6
#define TN 216
#define TSCAP BM_TILE_SLOTS

// Index of particle j of cell c in a brick's [particle-in-cell][cell]
// staging in shared memory.  The cell column is XOR-swizzled by the particle
// index, so that both the staging stores (consecutive particles of a few
// cells) and the per-cell reads (consecutive cells, one particle index) fall
// on distinct banks.
__device__ __forceinline__ int pic(int j, int c) { return j * BR3 + (c ^ ((j & 7) << 2)); }

#define BT 192  // threads per brick CTA: 64 cells x 3 z-offsets
// Sets of few bricks leave most of the chip idle and a brick's CTA is a chain
// of latencies.  Their CTAs have several groups of threads (WIDE of BT in the
// P2G and the general kernels): the particles take a third or less of the
// rounds, and the scatter's sums go side by side, momentum and force as well
// as the codes, each by one thread in the narrow form's order.
#define WIDE 4
// Lattice forms: substep of one cut scene, us, narrow -> wide: 80 bricks
// 77 -> 66, 210: 81 -> 74, 336: 86 -> 84, 432: 89 -> 96.
#define WIDE_BRICKS_LAT (2 * 152)

__device__ __forceinline__ void node_coords(const DevScene &sc, int li, int &ix, int &iy, int &iz) {
  ix = li % sc.nn[0];
  int r = li / sc.nn[0];
  iy = r % sc.nn[1];
  iz = r / sc.nn[1];
}

// brick-major index of base cell (bx, by, bz), scene-local coordinates
__device__ __forceinline__ int cell_index(const DevScene &sc, int bx, int by, int bz) {
  const int b = ((bz >> 2) * sc.nbr[1] + (by >> 2)) * sc.nbr[0] + (bx >> 2);
  return b * BR3 + (((bz & 3) * BR + (by & 3)) * BR + (bx & 3));
}

// The cell (0..63) of the brick's particle i: particles are sorted by cell,
// so it is the last cell whose range (cs: the brick's 65 cell starts,
// relative to its first particle) starts at or before i.
__device__ __forceinline__ int cell_of(const int *cs, int i) {
  int c = 0;
#pragma unroll
  for (int step = 32; step > 0; step >>= 1)
    if (cs[c + step] <= i) c += step;
  return c;
}

__device__ __forceinline__ void particle_base(uint32_t b, int &bx, int &by, int &bz) {
  bx = (int)(b & 1023u);
  by = (int)((b >> 10) & 1023u);
  bz = (int)((b >> 20) & 1023u);
}

__device__ __forceinline__ void brick_coords(const DevScene &sc, int lb, int &c0x, int &c0y, int &c0z) {
  c0x = (lb % sc.nbr[0]) * BR;
  c0y = ((lb / sc.nbr[0]) % sc.nbr[1]) * BR;
  c0z = (lb / (sc.nbr[0] * sc.nbr[1])) * BR;
}

// --------------------------------------------------------------------------
// The node tile of one brick: for each of its 6x6x6 nodes the first pool
// slot, the first tile slot (the node's logical grids laid out node by node
// in each node's own slot order) and the slot count; and, for the codes of
// the brick's particles (BPool::bcode; PPool::cid is a particle's index in
// the list), the slot (index at its node) of each code at each node.  Looked
// up in this table, a particle of a brick at a cut finds its 27 slots with
// one byte each; comparing its code with the slots' codes took two to four
// 8-byte reads a node.
// --------------------------------------------------------------------------
#define BRICK_SLOT_CODES 8  // codes with a slot table in shared memory (further codes compare)
#define NOSLOT 0xff

struct BrickTile {
  uint2 bcode[BM_BRICK_CODES];
  int goff[TN];
  uint16_t lo[TN];
  uint8_t cnt[TN];
  uint8_t slot[BRICK_SLOT_CODES][TN];
};

// slot of the brick's code b at tile node t (an index at the node), or NOSLOT
__device__ __forceinline__ int brick_slot(const World &w, const BrickTile &T, int nbc, int b, int t) {
  if (nbc <= BRICK_SLOT_CODES) return T.slot[b][t];
  const uint2 k = T.bcode[b];
  for (int a = 0; a < T.cnt[t]; ++a) {
    const uint2 c = w.S.code[T.goff[t] + a];
    if (c.x == k.x && c.y == k.y) return a;
  }
  return NOSLOT;
}

// Tile and codes of brick `brick` (nt threads); ends without a barrier.
__device__ __forceinline__ void brick_tile(const World &w, int brick, int nbc, BrickTile &T, int nt) {
  const int tid = threadIdx.x;
  for (int t = tid; t < TN; t += nt) {
    const int d = w.B.tdesc[(size_t)brick * TN + t];
    T.lo[t] = (uint16_t)(d & 0xffff);
    T.cnt[t] = (uint8_t)(d >> 16);
    T.goff[t] = w.B.tgoff[(size_t)brick * TN + t];  // valid where the count is not zero
  }
  if (tid < nbc) T.bcode[tid] = w.B.bcode[(size_t)brick * BM_BRICK_CODES + tid];
}

// Slot table of a brick with several codes or slots (after a barrier on
// brick_tile).  Slots whose code no particle of the brick carries get zero
// partial sums, mass and momentum and with FORCE the force too (pbase < 0:
// none are written).
template <bool FORCE>
__device__ __forceinline__ void brick_slots(const World &w, BrickTile &T, int nbc, int pbase, int nt) {
  for (int t = threadIdx.x; t < TN; t += nt) {
    const int n = T.cnt[t], g = T.goff[t];
    if (nbc <= BRICK_SLOT_CODES)
      for (int b = 0; b < nbc; ++b) T.slot[b][t] = NOSLOT;
    for (int a = 0; a < n; ++a) {
      const uint2 c = w.S.code[g + a];
      int id = -1;
      for (int b = 0; b < nbc; ++b)
        if (T.bcode[b].x == c.x && T.bcode[b].y == c.y) id = b;
      if (id >= 0) {
        if (nbc <= BRICK_SLOT_CODES) T.slot[id][t] = (uint8_t)a;
      } else if (pbase >= 0) {
        const size_t e = (size_t)pbase + T.lo[t] + a;
        w.B.pm[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (FORCE) w.B.pd[e] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  }
}

// What a brick kernel needs to know of its brick (of at most `places` particles).
struct BrickInfo {
  int nbc;        // distinct codes of the brick's particles
  bool single;    // no tile node holds several logical grids
  bool uniform;   // and at most one code: one pass, no code tests
  bool mask;      // empty places or several codes
  int pbase;      // partial-sum range (negative: pool overflow)
  int npass;      // a brick without particles still runs one pass: it writes zeros to its tile
  __device__ __forceinline__ BrickInfo(const World &w, const int4 &bt, int places) {
    const int info = w.B.binfo[bt.y];
    nbc = info & 0xff;
    single = (info >> 8) != 0;
    uniform = single && nbc <= 1;
    mask = bt.w < places || nbc > 1;
    pbase = w.B.poff[bt.y];
    npass = max(nbc, 1);
  }
  // slot of pass b's code at tile node t (an index at the node), or NOSLOT
  __device__ __forceinline__ int slot(const World &w, const BrickTile &T, int b, int t) const {
    return T.cnt[t] == 0 ? NOSLOT : uniform ? 0 : nbc == 0 ? NOSLOT : brick_slot(w, T, nbc, b, t);
  }
  // partial-sum entry of that slot, or -1
  __device__ __forceinline__ long long entry(const World &w, const BrickTile &T, int b, int t) const {
    const int sl = slot(w, T, b, t);
    return sl == NOSLOT || pbase < 0 ? -1 : (long long)pbase + T.lo[t] + sl;
  }
};

// --------------------------------------------------------------------------
// Per-particle work ahead of P2G (one thread per particle, inside the P2G
// brick kernel): tool and floor contact (Eq. 14-15 with friction Eq. 12),
// cutting progress D and release (Eq. 5), reaction wrench (Eq. 16), side
// label for the next substep (Eq. 3, 4, 6), and the P2G inputs
// A = -dt V0 P(F) / dx and the particle's total impulse J.
// --------------------------------------------------------------------------
// Whether the blade box is farther from the particle than one substep of
// relative motion can close: d > R_p + 2 dt (|v| + |v_B| + |w_B| r_max) (1-norms
// bound the speeds; r_max bounds the reach of the box from the blade's
// reference point), so that the predicted gap phi_hat = phi + dt min(v_n, 0)
// of the contact test is positive with a margin far above rounding.
__device__ __forceinline__ bool blade_out_of_reach(const DevScene &sc, const float x[3], const float v[3]) {
  const float *ax[3] = {sc.fn, sc.fe, sc.fd};
  const float r[3] = {x[0] - sc.fc[0], x[1] - sc.fc[1], x[2] - sc.fc[2]};
  float d2 = 0.f;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float q = r[0] * ax[a][0] + r[1] * ax[a][1] + r[2] * ax[a][2];
    const float e = fmaxf(fabsf(q) - sc.fhext[a], 0.0f);
    d2 += e * e;
  }
  const float rmax = fabsf(sc.fc[0] - sc.fxB[0]) + fabsf(sc.fc[1] - sc.fxB[1]) + fabsf(sc.fc[2] - sc.fxB[2]) +
                     sc.fhext[0] + sc.fhext[1] + sc.fhext[2];
  const float vb = fabsf(v[0]) + fabsf(v[1]) + fabsf(v[2]) + fabsf(sc.fvB[0]) + fabsf(sc.fvB[1]) +
                   fabsf(sc.fvB[2]) + (fabsf(sc.fwB[0]) + fabsf(sc.fwB[1]) + fabsf(sc.fwB[2])) * rmax;
  const float reach = sc.Rp * 1.0001f + 2.0f * sc.dt * vb;
  return d2 > reach * reach;
}

// INELASTIC: the launch set holds a scene with plasticity or viscosity (the
// elastic instantiation carries no trace of those paths)
template <bool INELASTIC>
__device__ __forceinline__ void pre_particle(const DevScene &sc, const PPool &P, int p, uint8_t tf, const float x[3],
                                             const float v[3], uint32_t s1, uint32_t s2, float A[9], float J[3],
                                             float wr[6], bool &clamped, bool &anyc) {
  const float dt = sc.dt, mp = sc.mp;
  const int cut = sc.cut;
  J[0] = J[1] = J[2] = 0.f;
  // most particles never touch the blade: D and u_t are read only where the
  // flag says they may be nonzero (both are exactly zero where it is clear)
  const float D0 = tf ? P.D[p] : 0.0f;
  float D = sc.reset_D ? 0.0f : D0;
  const float u00 = tf ? P.ut[0][p] : 0.0f, u01 = tf ? P.ut[1][p] : 0.0f, u02 = tf ? P.ut[2][p] : 0.0f;
  float uh[3] = {u00, u01, u02};
  if (sc.has_blade && sc.tool_contact_on && blade_out_of_reach(sc, x, v)) {
    uh[0] = uh[1] = uh[2] = 0.0f;  // as on the no-contact branch below
  } else if (sc.has_blade && sc.tool_contact_on) {
    float xc[3], nB[3], phi;
    box_closest(sc, x, sc.Rp, xc, nB, phi);
    float rc[3] = {xc[0] - sc.fxB[0], xc[1] - sc.fxB[1], xc[2] - sc.fxB[2]};
    float wr3[3] = {sc.fwB[1] * rc[2] - sc.fwB[2] * rc[1], sc.fwB[2] * rc[0] - sc.fwB[0] * rc[2],
                    sc.fwB[0] * rc[1] - sc.fwB[1] * rc[0]};
    float vrel[3] = {v[0] - (sc.fvB[0] + wr3[0]), v[1] - (sc.fvB[1] + wr3[1]), v[2] - (sc.fvB[2] + wr3[2])};
    float vn = vrel[0] * nB[0] + vrel[1] * nB[1] + vrel[2] * nB[2];
    float phihat = phi + dt * fminf(vn, 0.0f);
    // no predicted overlap: J_n = 0 below, and the impulse, reaction and
    // friction history come out as on the no-contact branch
    if (!(phihat < 0.0f)) {
      uh[0] = uh[1] = uh[2] = 0.0f;
      goto contact_done;
    }
    {
    float wB = 0.0f;
    if (sc.finv_mass > 0.0f) {
      float rn[3] = {rc[1] * nB[2] - rc[2] * nB[1], rc[2] * nB[0] - rc[0] * nB[2], rc[0] * nB[1] - rc[1] * nB[0]};
      float q0 = sc.fIinv[0] * rn[0] + sc.fIinv[1] * rn[1] + sc.fIinv[2] * rn[2];
      float q1 = sc.fIinv[3] * rn[0] + sc.fIinv[4] * rn[1] + sc.fIinv[5] * rn[2];
      float q2 = sc.fIinv[6] * rn[0] + sc.fIinv[7] * rn[1] + sc.fIinv[8] * rn[2];
      wB = sc.finv_mass + rn[0] * q0 + rn[1] * q1 + rn[2] * q2;
    }
    float meff = 1.0f / (1.0f / mp + wB);
    float Jn = sc.s_n * meff / dt * fmaxf(-phihat, 0.0f);
    float JB[3] = {0.f, 0.f, 0.f};
    if (Jn > 0.0f) {
      float ft[3], un[3];
      friction(uh, nB, vrel, Jn / dt, meff, dt, sc.gamma_k, sc.gamma_c, sc.fmu_s, sc.fmu_d, ft, un);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        JB[a] = Jn * nB[a] + dt * ft[a];
        uh[a] = un[a];
      }
      if (cut >= 0) {  // Eq. 5: front band, advancing cut
        float r[3] = {x[0] - sc.fxe[0], x[1] - sc.fxe[1], x[2] - sc.fxe[2]};
        float sp = r[0] * sc.fn[0] + r[1] * sc.fn[1] + r[2] * sc.fn[2];
        float lp = r[0] * sc.fe[0] + r[1] * sc.fe[1] + r[2] * sc.fe[2];
        float fp = r[0] * sc.fd[0] + r[1] * sc.fd[1] + r[2] * sc.fd[2];
        float uc = (sc.fve[0] - v[0]) * sc.fd[0] + (sc.fve[1] - v[1]) * sc.fd[1] + (sc.fve[2] - v[2]) * sc.fd[2];
        bool front = fabsf(sp) <= sc.h && fabsf(lp) <= sc.fL && fp >= 0.0f && fp <= sc.b_lead && uc > sc.u_min;
        if (front) {
          float Jc = fmaxf(JB[0] * sc.fd[0] + JB[1] * sc.fd[1] + JB[2] * sc.fd[2], 0.0f);
          if (D < 1.0f) {
            D = fminf(D + Jc * uc / sc.Wth, 1.0f);
          } else {
#pragma unroll
            for (int a = 0; a < 3; ++a) JB[a] -= Jc * sc.fd[a];
          }
        }
      }
    } else {
      uh[0] = uh[1] = uh[2] = 0.0f;
    }
    const float idt = 1.0f / dt;
    const float FB[3] = {-JB[0] * idt, -JB[1] * idt, -JB[2] * idt};
    anyc |= Jn > 0.0f;
    wr[0] += FB[0];
    wr[1] += FB[1];
    wr[2] += FB[2];
    wr[3] += rc[1] * FB[2] - rc[2] * FB[1];
    wr[4] += rc[2] * FB[0] - rc[0] * FB[2];
    wr[5] += rc[0] * FB[1] - rc[1] * FB[0];
    J[0] += JB[0];
    J[1] += JB[1];
    J[2] += JB[2];
    }
  contact_done:;
  }
  if (sc.floor_on) {
    const float phi = x[2] - sc.floor_z - sc.Rp;
    const float phihat = phi + dt * fminf(v[2], 0.0f);
    J[2] += sc.s_n * mp / dt * fmaxf(-phihat, 0.0f);
  }
  if (sc.pair_on) {
    J[0] += P.J[0][p];
    J[1] += P.J[1][p];
    J[2] += P.J[2][p];
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) J[a] += mp * sc.g[a] * dt;
  uint8_t pend = 0;
  if (cut >= 0 && ((s1 | s2) & (1u << cut)) == 0u) pend = (uint8_t)side_label(sc, x, v);
  float F[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) F[k] = P.F[k][p];
  float Pk[9];
  if (INELASTIC && (sc.yield_stress > 0.0f || sc.viscosity > 0.0f))
    clamped |= inelastic_stress(sc, P, p, F, Pk);
  else
    clamped |= sc.model == BM_MODEL_FIXED_COROTATED ? piola_fcr(F, sc.mu, sc.lam, Pk) : piola(F, sc.mu, sc.lam, Pk);
  const float cA = -dt * sc.V0 * sc.inv_dx;  // grad N is applied per axis in units of 1/dx
#pragma unroll
  for (int k = 0; k < 9; ++k) A[k] = cA * Pk[k];
  // cutting progress and friction history are written back only when they
  // change (most particles touch no tool in a substep)
  if (!(D == D0)) P.D[p] = D;
  if (!(uh[0] == u00 && uh[1] == u01 && uh[2] == u02)) {
    P.ut[0][p] = uh[0];
    P.ut[1][p] = uh[1];
    P.ut[2][p] = uh[2];
  }
  // cleared only when the values in memory are zero: a value equal to zero
  // (either sign) was either written above or already held as zero
  const uint8_t nf = (D != 0.0f || uh[0] != 0.0f || uh[1] != 0.0f || uh[2] != 0.0f) ? 1 : 0;
  if (nf != tf) P.tflag[p] = nf;
  P.pend[p] = pend;
}

// Per-particle reaction wrenches of a brick (wrc[k][i], rows of `stride`, one
// per particle) as the sums that BT threads striding over the particles would
// hold; for CTAs of more threads.  Thread t < BT returns its sums in wr.
__device__ __forceinline__ void stride_wrench(const float *wrc, int stride, int n, float wr[6]) {
  for (int i = threadIdx.x; i < n && threadIdx.x < BT; i += BT)
#pragma unroll
    for (int k = 0; k < 6; ++k) wr[k] += wrc[k * stride + i];
}

// Per-brick wrench partial of this substep: float32 sums inside the brick
// (fixed shuffle tree, warps in order), one double per component; bricks
// without tool contact write zeros.  All threads of the CTA call it; those of
// its first W warps hold sums.
template <int W>
__device__ __forceinline__ void brick_wrench(const World &w, int brick, const float wr[6], bool anyc,
                                             float (*red)[W]) {
  const int tid = threadIdx.x;
  if (__syncthreads_or(anyc)) {
    const int lane = tid & 31, wid = tid >> 5;
    if (wid < W)
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        float v = wr[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(FULL, v, o);
        if (lane == 0) red[k][wid] = v;
      }
    __syncthreads();
    if (tid < 6) {
      double s = 0.0;
      for (int q = 0; q < W; ++q) s += (double)red[tid][q];
      w.wpart[(size_t)brick * 6 + tid] = s;
    }
  } else if (tid < 6) {
    w.wpart[(size_t)brick * 6 + tid] = 0.0;
  }
}

// --------------------------------------------------------------------------
// Terms of the transfer sums, with the rounding of every operation spelled
// out: left to the compiler, a product and a sum are contracted in one
// instantiation of a kernel (a launch bound, a particle count, general or
// lattice) and not in another, and the forms of a kernel must agree bit for bit.
// --------------------------------------------------------------------------
// weight N = wx (wy wz) and a sum's next term
__device__ __forceinline__ float weight(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_term(float sum, float N, float v) { return __fmaf_rn(N, v, sum); }
// Eq. 17: v' = beta (v - v_old) + v_new, x' = x + dt v_new
__device__ __forceinline__ float next_v(float beta, float v, float so, float sn) {
  return __fmaf_rn(beta, __fsub_rn(v, so), sn);
}
__device__ __forceinline__ float next_x(float x, float dt, float sn) { return __fmaf_rn(dt, sn, x); }
// One component of A grad N + N J = wx (A1 dyz + A2 wyd + J wyz) + dwx (A0 wyz)
// in P2G
__device__ __forceinline__ float force_u(float A1, float dyz, float A2, float wyd, float J, float wyz) {
  return __fmaf_rn(J, wyz, __fmaf_rn(A1, dyz, __fmul_rn(A2, wyd)));
}
__device__ __forceinline__ float force_acc(float q, float w, float U, float d, float V) {
  return __fadd_rn(q, __fmaf_rn(w, U, __fmul_rn(d, V)));
}

// --------------------------------------------------------------------------
// From per-cell sums to the node tile
// --------------------------------------------------------------------------
// Reduction of per-(cell, z-offset) sums to per-node sums inside a warp.
// Cells are x-fastest in a brick and a warp holds 32 consecutive cells of one
// z-offset, so the 4 cells of an x-row are adjacent lanes and the 4 rows of a
// z-layer are 4 lanes apart.  On entry a[i][j][k] is value k of the thread's
// own cell for node (cx + j, cy + i, cz + oz).  The x pass adds, for node
// cx, the contributions of cells cx - 1 and cx - 2 (shuffles); the lane at
// the row's end also keeps the row's sums for the two node columns beyond it
// (nodes 4 and 5 of the tile's 6).  The y pass does the same along y.  On
// exit lane (cx, cy) holds, for its z-layer, the sums over the layer's cells
// of nodes (tx, ty) = (cx + j, cy + i), with j > 0 only at cx = 3 and i > 0
// only at cy = 3 (zeros elsewhere).  Each sum is taken in a fixed order (own
// cell, then the one before, then the one before that).
template <int NV>
__device__ __forceinline__ void xy_reduce(float (&a)[3][3][NV], int cx, int cy) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const float t1 = __shfl_up_sync(FULL, a[i][1][k], 1);
      const float t2 = __shfl_up_sync(FULL, a[i][2][k], 2);
      const float t3 = __shfl_up_sync(FULL, a[i][2][k], 1);
      float sum = a[i][0][k];
      if (cx >= 1) sum += t1;
      if (cx >= 2) sum += t2;
      a[i][0][k] = sum;
      a[i][1][k] = cx == 3 ? a[i][1][k] + t3 : 0.f;
      a[i][2][k] = cx == 3 ? a[i][2][k] : 0.f;
    }
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const float t1 = __shfl_up_sync(FULL, a[1][j][k], 4);
      const float t2 = __shfl_up_sync(FULL, a[2][j][k], 8);
      const float t3 = __shfl_up_sync(FULL, a[2][j][k], 4);
      float sum = a[0][j][k];
      if (cy >= 1) sum += t1;
      if (cy >= 2) sum += t2;
      a[0][j][k] = sum;
      a[1][j][k] = cy == 3 ? a[1][j][k] + t3 : 0.f;
      a[2][j][k] = cy == 3 ? a[2][j][k] : 0.f;
    }
}

// The layer sums of xy_reduce into the z stage, value k of tile node (tx,
// ty, cz + oz) from the cells of z-layer cz: with ZN = TN at sz[k][oz][t] (t
// the tile node), with ZN = TZ at sz[k][oz][(cz * TE + ty) * TE + tx] (a
// z-offset reaches 4 of the tile's 6 node layers, so each offset keeps
// 4 x 36 entries; the compact stage lets P2G run 4 CTAs per SM).  Each (node,
// oz) entry that the tile gather reads has exactly one writer.
#define TZ (BR * TE * TE)
template <int NV, int ZN>
__device__ __forceinline__ void stage_layer(float (*sz)[3][ZN], const float (&a)[3][3][NV], int cx, int cy,
                                            int cz, int oz) {
  const int lz = ZN == TN ? cz + oz : cz;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if ((i > 0 && cy != 3) || (j > 0 && cx != 3)) continue;
      const int e = (lz * TE + cy + i) * TE + cx + j;
#pragma unroll
      for (int k = 0; k < NV; ++k) sz[k][oz][e] = a[i][j][k];
    }
}

// Sums of tile node t over the z-offsets of the z stage (<= 3 terms, in
// ascending offset order); in the compact stage offset o holds node t at
// entry t - o * 36.
template <int NV, int ZN>
__device__ __forceinline__ void gather_z(const float (*sz)[3][ZN], int t, float (&acc)[NV]) {
  const int tz = t / (TE * TE);
  const int o0 = max(0, tz - (BR - 1)), o1 = min(2, tz);
#pragma unroll
  for (int k = 0; k < NV; ++k) acc[k] = 0.f;
  for (int o = o0; o <= o1; ++o)
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] += sz[k][o][ZN == TN ? t : t - o * TE * TE];
}

}  // namespace
