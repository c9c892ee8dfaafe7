// Adjoint (reverse mode) of the batched track fit.  Included after
// fit_core.cuh by the same kernel module, so that the forward recomputation
// uses the module's own arithmetic bit for bit.
//
// Objective: L = sum_i g_i chi2_i, chi2_i the inward-refit chi2 of track i.
// Gradients: dL/dm_h for every cluster measurement m_h = (y - dy, z - dz)
// (hence dL/d(dy, dz)[sector][row] = -sum over the clusters with that key),
// and dL/dseed_i.  The outward pass feeds the inward one through its final
// state (the covariance is reset, the outward chi2 is not part of L).
//
// Tape: the forward leaves the filter states of both passes on a tape, laid out
// so that a warp reads a state of its 32 tracks as contiguous rows, and the
// backward reverses the steps one by one from it (recomputing each step's
// intermediates from the state before it).
//
// Checkpoints, where there is no place on the tape: the forward writes the filter
// state before every kCkptEvery-th step of each pass.  The backward walks the
// segments of a track in reverse: it recomputes a segment's steps from its
// checkpoint into a per-warp segment store, then reverses them.  States carry y and
// z as residuals from the current cluster's measurement, like the fit.
#pragma once

namespace tpcfit {
namespace TPCFIT_NS {


struct JacBar {
  float yy, ys, yq, zy, zs, zt, zq, sy, ss, sq;
};

// d/du of asinc_f(u), consistent with the branch asinc_f takes.
__device__ __forceinline__ float asinc_deriv(float u) {
  const float au = u < 0.0f ? -u : u;
#if !TPCFIT_DET
  if (au < 0.05f) {  // derivative of the three-term fast-mode polynomial
    const float q = u * u;
    return (2.0f * u) * (static_cast<float>(1.0 / 6.0) +
                         q * (2.0f * static_cast<float>(3.0 / 40.0) + q * (3.0f * static_cast<float>(5.0 / 112.0))));
  }
#endif
  if (au <= 0.25f) {
    const float c1 = static_cast<float>(1.0 / 6.0);
    const float c2 = static_cast<float>(3.0 / 40.0);
    const float c3 = static_cast<float>(5.0 / 112.0);
    const float c4 = static_cast<float>(35.0 / 1152.0);
    const float c5 = static_cast<float>(63.0 / 2816.0);
    const float c6 = static_cast<float>(231.0 / 13312.0);
    const float q = u * u;
    float acc = 6.0f * c6;
    acc = acc * q + 5.0f * c5;
    acc = acc * q + 4.0f * c4;
    acc = acc * q + 3.0f * c3;
    acc = acc * q + 2.0f * c2;
    acc = acc * q + c1;
    return (2.0f * u) * acc;
  }
#if TPCFIT_DET
  const double ud = (double)u;
  const double sq = sqrt((1.0 - ud) * (1.0 + ud));
  return (float)((ud / sq - asin_f64(ud)) / (ud * ud));
#else
  return (u * rsqrtf((1.0f - u) * (1.0f + u)) - asinf(u)) / (u * u);
#endif
}

// Reverse of scalar_update<H>.  p, L: state before the update; b_p, b_L: in =
// adjoint after the update, out = adjoint before; b_chi: adjoint of chi2 (the
// same before and after).  b_m receives the adjoint of the measured value.
template <int H>
__device__ __forceinline__ void scalar_update_rev(const GeoRef& G, const float p[5], const float L[5][5], float mv, float b_p[5],
                                                  float b_L[5][5], float b_chi, float& b_m) {
  const float v = G.v_meas;
  float a[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) a[c] = L[H][c];
  float s2 = v + a[0] * a[0];
#pragma unroll
  for (int c = 1; c < 5; ++c) s2 = s2 + a[c] * a[c];
  float alpha, beta, gamma;
  potter_coeffs(s2, v, G.sqrt_v, alpha, beta, gamma);
  const float r = mv - p[H];
  float la[5], K[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    float acc = L[i][0] * a[0];
#pragma unroll
    for (int c = 1; c < 5; ++c) acc = acc + L[i][c] * a[c];
    la[i] = acc;
    K[i] = acc * alpha;
  }
  // p' = p + K r ; chi2' = chi2 + r^2 alpha
  float b_K[5], b_a[5];
  float b_r = 0.0f, b_alpha = 0.0f, b_gamma = 0.0f, b_beta = 0.0f;
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    b_K[i] = r * b_p[i];
    b_r += K[i] * b_p[i];
  }
  b_r += 2.0f * r * alpha * b_chi;
  b_alpha += r * r * b_chi;
#pragma unroll
  for (int c = 0; c < 5; ++c) b_a[c] = 0.0f;
  // L'_i = L_i - (gamma K_i) a (i != H)
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    if (i == H) continue;
    const float gk = gamma * K[i];
    float b_gk = 0.0f;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      b_gk -= b_L[i][c] * a[c];
      b_a[c] -= gk * b_L[i][c];
    }
    b_gamma += K[i] * b_gk;
    b_K[i] += gamma * b_gk;
  }
  // L'_H = beta a
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    b_a[c] += beta * b_L[H][c];
    b_beta += a[c] * b_L[H][c];
  }
  // gamma = 1/(1 + beta)
  b_beta -= gamma * gamma * b_gamma;
  // K_i = la_i alpha
  float b_la[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    b_la[i] = alpha * b_K[i];
    b_alpha += la[i] * b_K[i];
  }
  // r = m - p_H
  b_m = b_r;
  b_p[H] -= b_r;
  // alpha = 1/s2, beta = sqrt(v/s2)
  const float b_s2 = -(alpha * alpha) * b_alpha - 0.5f * (beta * alpha) * b_beta;
  // la_i = L_i . a (i != H); la_H = a . a
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    if (i == H) continue;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      b_L[i][c] += a[c] * b_la[i];
      b_a[c] += L[i][c] * b_la[i];
    }
  }
#pragma unroll
  for (int c = 0; c < 5; ++c) b_a[c] += 2.0f * a[c] * (b_la[H] + b_s2);
  // a = L_H: row H enters only through a
#pragma unroll
  for (int c = 0; c < 5; ++c) b_L[H][c] = b_a[c];
}

// Reverse of transport (L' = J L): b_L in = adjoint of L', out = adjoint of L;
// bJ = adjoint of the Jacobian entries.  L: the factor before the transport.
__device__ __forceinline__ void transport_rev(const float L[5][5], const Jac& J, float b_L[5][5], JacBar& bJ) {
  bJ.yy = bJ.ys = bJ.yq = bJ.zy = bJ.zs = bJ.zt = bJ.zq = bJ.sy = bJ.ss = bJ.sq = 0.0f;
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    const float b0 = b_L[0][c], b1 = b_L[1][c], b2 = b_L[2][c];
    bJ.ys += b0 * L[2][c];
    bJ.yq += b0 * L[4][c];
    bJ.zs += b1 * L[2][c];
    bJ.zt += b1 * L[3][c];
    bJ.zq += b1 * L[4][c];
    bJ.sq += b2 * L[4][c];
    b_L[3][c] += J.zt * b1;
    b_L[4][c] += J.yq * b0 + J.zq * b1 + J.sq * b2;
    if (!J.rot) {
      b_L[2][c] = b2 + J.ys * b0 + J.zs * b1;
    } else {
      bJ.yy += b0 * L[0][c];
      bJ.zy += b1 * L[0][c];
      bJ.sy += b2 * L[0][c];
      bJ.ss += b2 * L[2][c];
      b_L[0][c] = J.yy * b0 + J.zy * b1 + J.sy * b2;
      b_L[2][c] = J.ys * b0 + J.zs * b1 + J.ss * b2;
    }
  }
}

// Reverse of predict_t<FIELD> (FIELD 0: uniform field, 1: the map): b_po =
// adjoint of the predicted state, bJ = adjoint of the Jacobian entries; b_pi
// receives the adjoint of the state before the step (t, q: its tan(lambda) and
// q/pt).  With the map the curvature depends on the step's midpoint, hence on
// y, z, s, t and on the offsets (yo, zo) of residual coordinates, whose
// adjoints go to b_yo, b_zo (zero without the map).
template <int FIELD = 0>
__device__ __forceinline__ void predict_rev(const GeoRef& G, const PredTape& tp, const Jac& J, float t, float q, const float b_po[5],
                                            const JacBar& bJ, float b_pi[5], float& b_yo, float& b_zo) {
  const float kappa = FIELD == 1 ? tp.kap : G.kappa;
  float b_kap = 0.0f;  // adjoint of the curvature per unit q/pt (map only)
  const float dx = tp.dx, s1 = tp.s1, s2 = tp.s2, ic1 = tp.ic1, ic2 = tp.ic2, Tm = tp.Tm, tt = tp.tt;
  float b_t = b_po[3], b_q = b_po[4], b_s2 = b_po[2];
  float b_s1 = 0.0f, b_dx = 0.0f, b_k = 0.0f, b_kdx = 0.0f, b_ic1 = 0.0f, b_ic2 = 0.0f, b_c1 = 0.0f, b_c2 = 0.0f;
  float b_Tm = 0.0f, b_tt = 0.0f, b_dl = 0.0f, b_w = 0.0f, b_rr = 0.0f;
  float bJys0 = bJ.ys, bJzs0 = bJ.zs;
  if (J.rot) {
    const float rr = J.ss;
    b_rr = bJ.ss + bJ.ys * tp.Jys0 + bJ.zs * tp.Jzs0;
    bJys0 = bJ.ys * rr;
    bJzs0 = bJ.zs * rr;
    b_k -= tp.sa * bJ.sy;
    b_t -= tp.sa * ic2 * bJ.zy;
    b_ic2 -= tp.sa * t * bJ.zy;
    b_s2 -= tp.sa * ic2 * bJ.yy;
    b_ic2 -= tp.sa * s2 * bJ.yy;
  }
  // Jsq = dx kappa ; Jzq = (t kappa) Lk
  b_dx += kappa * bJ.sq;
  b_t += kappa * tp.Lk * bJ.zq;
  const float b_Lk = t * kappa * bJ.zq;
  if (FIELD == 1) b_kap += tp.dx * bJ.sq + (t * tp.Lk) * bJ.zq;
  if (tp.series) {
    const float i2 = ic1 * ic1, i3 = i2 * ic1, i5 = i3 * i2, i7 = i5 * i2, s1s = s1 * s1;
    const float a1 = (s1 * i3) * 0.5f;
    const float a2 = ((1.0f + 2.0f * s1s) * i5) * static_cast<float>(1.0 / 3.0);
#if TPCFIT_DET
    const float a3 = ((s1 * (3.0f + 2.0f * s1s)) * i7) * 0.125f;
#else
    const float a3 = 0.0f;  // the fast forward keeps two terms of the series
#endif
    const float kdx = tp.kdx, Q = a2 + kdx * a3, P = a1 + kdx * Q;
    b_dx += 2.0f * dx * P * b_Lk;
    const float b_P = dx * dx * b_Lk;
    const float b_a1 = b_P;
    b_kdx += Q * b_P;
    const float b_Q = kdx * b_P;
    const float b_a2 = b_Q;
    b_kdx += a3 * b_Q;
    const float b_a3 = kdx * b_Q;
    float b_s1s = 0.0f, b_i2 = 0.0f, b_i3 = 0.0f, b_i5 = 0.0f, b_i7 = 0.0f;
    b_s1 += 0.5f * i3 * b_a1;
    b_i3 += 0.5f * s1 * b_a1;
    b_s1s += static_cast<float>(2.0 / 3.0) * i5 * b_a2;
    b_i5 += (1.0f + 2.0f * s1s) * static_cast<float>(1.0 / 3.0) * b_a2;
    b_s1 += 0.125f * (3.0f + 2.0f * s1s) * i7 * b_a3;
    b_s1s += 0.25f * s1 * i7 * b_a3;
    b_i7 += 0.125f * s1 * (3.0f + 2.0f * s1s) * b_a3;
    b_s1 += 2.0f * s1 * b_s1s;
    b_i5 += i2 * b_i7;
    b_i2 += i5 * b_i7;
    b_i3 += i2 * b_i5;
    b_i2 += i3 * b_i5;
    b_i2 += ic1 * b_i3;
    b_ic1 += i2 * b_i3;
    b_ic1 += 2.0f * ic1 * b_i2;
  } else {
    const float k = tp.k;
    const float b_D = b_Lk / k;
    b_k -= tp.Lk / k * b_Lk;
    b_dx += ic2 * b_D;
    b_ic2 += dx * b_D;
    b_dl -= b_D;
  }
  b_dl += bJ.zt;  // Jzt = dl
  {  // Jzs0 = (t dx) (Tm (ic1 ic2))
    const float E = ic1 * ic2, F = Tm * E, G = t * dx;
    const float b_G = F * bJzs0, b_F = G * bJzs0, b_E = Tm * b_F;
    b_Tm += E * b_F;
    b_ic1 += ic2 * b_E;
    b_ic2 += ic1 * b_E;
    b_t += dx * b_G;
    b_dx += t * b_G;
  }
  {  // Jyq = ((dx kappa) dx) (tt (ic2 / 2))
    const float M = (dx * kappa) * dx;
    b_dx += 2.0f * kappa * dx * (tt * (ic2 * 0.5f)) * bJ.yq;
    b_tt += ic2 * 0.5f * M * bJ.yq;
    b_ic2 += tt * 0.5f * M * bJ.yq;
    if (FIELD == 1) b_kap += (dx * dx) * (tt * (ic2 * 0.5f)) * bJ.yq;
  }
  {  // Jys0 = (dx tt) ((ic1 + ic2) / 2)
    const float Hh = (ic1 + ic2) * 0.5f;
    b_dx += tt * Hh * bJys0;
    b_tt += dx * Hh * bJys0;
    b_ic1 += 0.5f * dx * tt * bJys0;
    b_ic2 += 0.5f * dx * tt * bJys0;
  }
  b_Tm += 2.0f * Tm * b_tt;  // tt = 1 + Tm^2
  // z2 = z1 + t dl ; y2 = y1 + dx Tm
  b_t += tp.dl * b_po[1];
  b_dl += t * b_po[1];
  b_dx += Tm * b_po[0];
  b_Tm += dx * b_po[0];
  // dl = (dx w) A ; A = asinc(sig) ; sig = kdx w
  const float b_A = dx * tp.w * b_dl;
  b_dx += tp.w * tp.A * b_dl;
  b_w += dx * tp.A * b_dl;
  const float b_sig = asinc_deriv(tp.sig) * b_A;
  b_kdx += tp.w * b_sig;
  b_w += tp.kdx * b_sig;
  // w = c1 + s1 Tm
  b_c1 += b_w;
  b_s1 += Tm * b_w;
  b_Tm += s1 * b_w;
  // Tm = (s1 + s2) / den, den = c1 + c2
  const float b_num = b_Tm / tp.den;
  const float b_den = -Tm * b_Tm / tp.den;
  b_s1 += b_num;
  b_s2 += b_num;
  b_c1 += b_den;
  b_c2 += b_den;
  // (c, 1/c) = sqrt_and_inv(u), u = (1 - s)(1 + s)
  const float b_u2 = 0.5f * ic2 * (b_c2 - ic2 * ic2 * b_ic2);
  const float b_u1 = 0.5f * ic1 * (b_c1 - ic1 * ic1 * b_ic1);
  b_s2 -= 2.0f * s2 * b_u2;
  b_s1 -= 2.0f * s1 * b_u1;
  // s2 = s1 + kdx ; kdx = k dx ; k = q kappa
  b_s1 += b_s2;
  b_kdx += b_s2;
  b_k += dx * b_kdx;
  b_dx += tp.k * b_kdx;
  b_q += kappa * b_k;
  // the map: kappa = kappa0 (1 + f_r (xm^2 + ym^2) + f_z zm^2) at the midpoint of
  // a straight half step, xm = x1 + dx/2, ym = (yo + y1) + (dx/2) s1/c1,
  // zm = (zo + z1) + (dx/2) t/c1
  float b_y1 = b_po[0], b_z1 = b_po[1], b_xm = 0.0f;
  b_yo = 0.0f;
  b_zo = 0.0f;
  if (FIELD == 1) {
    b_kap += q * b_k;
    const float k0 = 2.0f * G.kappa;
    b_xm = (k0 * G.f_r) * tp.xm * b_kap;
    const float b_ym = (k0 * G.f_r) * tp.ym * b_kap;
    const float b_zm = (k0 * G.f_z) * tp.zm * b_kap;
    const float hdx = 0.5f * dx, ic1c = ic1 * ic1 * ic1;
    b_yo = b_ym;
    b_zo = b_zm;
    b_y1 += b_ym;
    b_z1 += b_zm;
    b_t += (hdx * ic1) * b_zm;
    b_s1 += hdx * ic1c * (b_ym + (t * s1) * b_zm);  // d(s/c)/ds = 1/c^3, d(1/c)/ds = s/c^3
    b_dx += 0.5f * (b_xm + (s1 * ic1) * b_ym + (t * ic1) * b_zm);
  }
  // dx = X - x1
  const float b_x1 = b_xm - b_dx;
  if (J.rot) {
    // x1 = x ca + y sa ; y1 = y ca - x sa ; s1 = s ca - c sa ; cr = c ca + s sa ;
    // rr = cr / c ; c = sqrt((1 - s)(1 + s))
    const float rr = J.ss;
    const float b_cr = b_rr / tp.c;
    float b_c = -rr * b_rr / tp.c;
    b_pi[0] = tp.sa * b_x1 + tp.ca * b_y1;
    float b_s = tp.ca * b_s1;
    b_c -= tp.sa * b_s1;
    b_c += tp.ca * b_cr;
    b_s += tp.sa * b_cr;
    b_s -= (tp.s / tp.c) * b_c;
    b_pi[2] = b_s;
  } else {
    b_pi[0] = b_y1;
    b_pi[2] = b_s1;
  }
  b_pi[1] = b_z1;
  b_pi[3] = b_t;
  b_pi[4] = b_q;
}

// ---------------------------------------------------------------- backward kernel
struct StepState {
  float p[5];
  float L[5][5];
  float x;
  int sec;
};

// A checkpoint of the U-D fit, loaded as if it held L (u in rows 0-1, d in
// row 2): turned into the square-root factor L = U sqrt(D), upper triangular.
__device__ __forceinline__ void sqrt_from_ud_ckpt(StepState& S) {
  float u[10], sd[5];
#pragma unroll
  for (int e = 0; e < 10; ++e) u[e] = S.L[e / 5][e % 5];
#pragma unroll
  for (int c = 0; c < 5; ++c) sd[c] = sqrtf(S.L[2][c]);
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int c = 0; c < 5; ++c) S.L[i][c] = c < i ? 0.0f : (c == i ? sd[c] : u[4 * i - (i * (i - 1)) / 2 + (c - i - 1)] * sd[c]);
}

// One cluster as stored (y, z, packed row/sector), loaded ahead of its use.
template <class A>
__device__ __forceinline__ RecordedTrack recorded_track(const A& a, int32_t trk) {
  return tpcfit::recorded_track(a.off, a.n_hits, a.ndf, a.ck_last, trk);
}

struct HitRaw {
  float y, z;
  int rs;
};

__device__ __forceinline__ HitRaw load_hit(const float* y, const float* z, const uint16_t* rowsec, int h) {
  HitRaw r;
  r.y = __ldg(y + h);
  r.z = __ldg(z + h);
  r.rs = (int)__ldg(rowsec + h);
  return r;
}
__device__ __forceinline__ HitRaw load_hit(const BwdArgs& a, int h) { return load_hit(a.y, a.z, a.rowsec, h); }

// Measurement (alignment subtracted), row and sector of a loaded cluster.  Row
// and sector are clamped into the table: the recorded fit has validated them,
// the clamp only keeps a mismatched call inside shared memory.
__device__ __forceinline__ void decode_hit(const float* align, const HitRaw& r, float& m0, float& m1, int& row,
                                           int& sec) {
  row = min(r.rs >> 6, kMaxRows - 1);
  sec = min(r.rs & 63, kNSectors - 1);
  const float2 d = reinterpret_cast<const float2*>(align)[sec * kMaxRows + row];
  m0 = r.y - d.x;
  m1 = r.z - d.y;
}

// States between checkpoints: 8 float4 (p 5, L 25, x, sector bits), stored
// lane-interleaved ([float4 j][lane]) so that a warp's stores and copies coalesce.
constexpr int kStateF4 = 8;

__device__ __forceinline__ void pack_state(const StepState& S, float v[32]) {
#pragma unroll
  for (int c = 0; c < 5; ++c) v[c] = S.p[c];
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int c = 0; c < 5; ++c) v[5 + 5 * i + c] = S.L[i][c];
  v[30] = S.x;
  v[31] = __int_as_float(S.sec);
}

__device__ __forceinline__ void unpack_state(const float v[32], StepState& S) {
#pragma unroll
  for (int c = 0; c < 5; ++c) S.p[c] = v[c];
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int c = 0; c < 5; ++c) S.L[i][c] = v[5 + 5 * i + c];
  S.x = v[30];
  S.sec = __float_as_int(v[31]);
}

// dst[j * kWarp] = float4 j of the state (dst already offset by the lane).
__device__ __forceinline__ void store_state(float4* dst, const StepState& S) {
  float v[32];
  pack_state(S, v);
#pragma unroll
  for (int j = 0; j < kStateF4; ++j) dst[j * kWarp] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
}

// The same read, but never merged with an earlier one: the state is read again
// from shared memory where it is needed instead of being kept in registers.
__device__ __forceinline__ float4 lds_volatile(const float4* p) {
  float4 r;
  asm volatile("ld.volatile.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n"
               : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w)
               : "r"((unsigned)__cvta_generic_to_shared(p)));
  return r;
}

__device__ __forceinline__ void reread_state(const float4* src, StepState& S) {
  float v[32];
#pragma unroll
  for (int j = 0; j < kStateF4; ++j) {
    const float4 f = lds_volatile(src + j * kWarp);
    v[4 * j] = f.x;
    v[4 * j + 1] = f.y;
    v[4 * j + 2] = f.z;
    v[4 * j + 3] = f.w;
  }
  unpack_state(v, S);
}

__device__ __forceinline__ void read_state(const float4* src, StepState& S) {
  float v[32];
#pragma unroll
  for (int j = 0; j < kStateF4; ++j) {
    const float4 f = src[j * kWarp];
    v[4 * j] = f.x;
    v[4 * j + 1] = f.y;
    v[4 * j + 2] = f.z;
    v[4 * j + 3] = f.w;
  }
  unpack_state(v, S);
}

// One lane's state: F4 float4 from a lane-interleaved global slot into its
// lane-interleaved shared slot, as one commit group.
template <int F4 = kStateF4>
__device__ __forceinline__ void fetch_state(float4* sdst, const float4* gsrc) {
#pragma unroll
  for (int j = 0; j < F4; ++j) cp_async16(sdst + j * kWarp, gsrc + j * kWarp);
  cp_async_commit();
}

// A checkpoint (32 contiguous floats, 16-byte aligned: the
// state) into a lane-interleaved shared slot, as one commit group.
__device__ __forceinline__ void fetch_ckpt(float4* sdst, const float* ck) {
  const float4* g = reinterpret_cast<const float4*>(ck);
#pragma unroll
  for (int j = 0; j < kStateF4; ++j) cp_async16(sdst + j * kWarp, g + j);
  cp_async_commit();
}

// Forward of one step on a StepState (the same operations as the fit, in
// residual coordinates).  my, mz: measurement of the previous cluster on
// entry, of this cluster on exit.  conv: the first step of the outward pass,
// whose state is the seed in absolute coordinates.
// MAT: the material layers of the rows; FIELD as for predict_t (the smoother
// follows both; the adjoint runs without either).
template <bool MAT = false, int FIELD = 0>
__device__ __forceinline__ void step_fwd(const GeoRef& G, const SmemTables& T, StepState& S, float& my, float& mz, bool first, bool conv,
                                         int row, int sec18, float m0, float m1) {
  float chi2 = 0.0f;
  if (first) {
    S.x = T.row_x[row];
    S.sec = sec18;
    if (conv) {
      S.p[0] = S.p[0] - m0;
      S.p[1] = S.p[1] - m1;
    }
  } else {
    float pn[5];
    Jac J;
    PredTape tp;
    MatNoise N;
    if (MAT && !conv) {  // inward: the layer of the row left
      material_step(G, S.p, -1, N);
      material_factor(S.L, N);
    }
    predict_residual<FIELD>(G, T, S.p, S.x, S.sec, my, mz, sec18, T.row_x[row], m0, m1, pn, J, tp);
    if (MAT && conv) material_step(G, pn, 1, N);
#pragma unroll
    for (int c = 0; c < 5; ++c) S.p[c] = pn[c];
    S.x = T.row_x[row];
    S.sec = sec18;
    transport(S.L, J);
    if (MAT && conv) material_factor(S.L, N);
  }
  my = m0;
  mz = m1;
  scalar_update<0>(G, S.p, S.L, chi2, 0.0f);
  scalar_update<1>(G, S.p, S.L, chi2, 0.0f);
}

// Reverse of one step from the state before it, which sits in shared memory
// at src ([float4 j][lane]; read twice so that it need not stay in registers
// through the update reverses).  my_prev, mz_prev: measurement of the previous
// cluster.  b_p, b_L: in = adjoint after the step, out = adjoint before it.
// The measurements enter only through the residual shifts: b_mc = adjoint of
// this cluster's (y, z), b_mp = of the previous one's.
template <int FIELD = 0>
__device__ __forceinline__ void step_rev(const GeoRef& G, const SmemTables& T, const float4* src, float my_prev, float mz_prev,
                                         bool first, bool conv, int row, int sec18, float m0, float m1, float b_p[5],
                                         float b_L[5][5], float b_chi, float b_mc[2], float b_mp[2]) {
  StepState S0;
  read_state(src, S0);
  float p1[5];
  Jac J;
  float L[5][5];
  PredTape tp;
  if (first) {
#pragma unroll
    for (int c = 0; c < 5; ++c) p1[c] = S0.p[c];
    if (conv) {
      p1[0] = S0.p[0] - m0;
      p1[1] = S0.p[1] - m1;
    }
  } else {
    predict_residual<FIELD>(G, T, S0.p, S0.x, S0.sec, my_prev, mz_prev, sec18, T.row_x[row], m0, m1, p1, J, tp);
  }
  // the factor before the y update (kept) and before the z update
  float p2[5];
  float chi_dummy = 0.0f, b_dummy = 0.0f;
#pragma unroll
  for (int c = 0; c < 5; ++c) p2[c] = p1[c];
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int c = 0; c < 5; ++c) L[i][c] = S0.L[i][c];
  if (!first) transport(L, J);
  float L2[5][5];
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int c = 0; c < 5; ++c) L2[i][c] = L[i][c];
  scalar_update<0>(G, p2, L2, chi_dummy, 0.0f);
  scalar_update_rev<1>(G, p2, L2, 0.0f, b_p, b_L, b_chi, b_dummy);
  scalar_update_rev<0>(G, p1, L, 0.0f, b_p, b_L, b_chi, b_dummy);
  // b_p is now the adjoint of the predicted (shifted) state p1
  b_mc[0] = -b_p[0];
  b_mc[1] = -b_p[1];
  b_mp[0] = 0.0f;
  b_mp[1] = 0.0f;
  if (first) {
    if (!conv) b_mc[0] = b_mc[1] = 0.0f;  // the inward pass starts from residuals already
    return;
  }
  reread_state(src, S0);
  JacBar bJ;
  transport_rev(S0.L, J, b_L, bJ);
  const bool rot = S0.sec != sec18;
  if (!rot) {
    b_mp[0] = b_p[0];
    b_mp[1] = b_p[1];
  }
  // the prediction's intermediates (tp, J) are those of the forward above
  float b_pi[5], b_yo, b_zo;
  predict_rev<FIELD>(G, tp, J, S0.p[3], S0.p[4], b_p, bJ, b_pi, b_yo, b_zo);
  if (rot) {
    b_mp[0] = b_pi[0];
    b_mp[1] = b_pi[1];
  } else if (FIELD == 1) {  // the map's midpoint sits at the previous cluster plus the residual
    b_mp[0] += b_yo;
    b_mp[1] += b_zo;
  }
#pragma unroll
  for (int c = 0; c < 5; ++c) b_p[c] = b_pi[c];
}

// Reverse of material_step for a step that was taken.  p: the state before it;
// b_p in: adjoint of the state after, out: of the state before; bN: adjoints of
// the terms it handed on (qq, b_s, b_t, b_q).  Only s, t and q enter.
__device__ __forceinline__ void material_step_rev(const GeoRef& G, const float p[5], int dir, const MatNoise& bN, float b_p[5]) {
  const float s = p[2], t = p[3], q = p[4];
  const float q2 = q * q;
  if (!(q2 > 0.0f)) return;  // no material effect: nothing depends on the state
  const float tt1 = 1.0f + t * t;
  const float c = sqrtf((1.0f - s) * (1.0f + s));
  const float st1 = sqrtf(tt1);
  const float ell = (G.d_row * st1) / c;
  const float p2 = tt1 / q2;
  const float e2 = p2 + G.mass2;
  const float kx = static_cast<float>(0.0136 * 0.0136) * G.x0_inv;
  const float ip2 = 1.0f / p2;
  const float th2 = (kx * ell) * (e2 * (ip2 * ip2));
  const float e = sqrtf(e2);
  const float de = (G.dedx * ell) * (e2 * ip2);
  const float en = dir > 0 ? e - de : e + de;
  const float pn2 = en * en - G.mass2;
  const float ratio = sqrtf(p2 / pn2);
  const float qo = q * ratio;
  const float th = sqrtf(th2);
  // b_s = th c st1, b_t = th tt1, b_q = th qo t, qq = ratio, q' = q ratio
  const float b_qo = b_p[4] + (bN.b_q * th) * t;
  float b_t = b_p[3] + (bN.b_q * th) * qo;
  const float b_th = (bN.b_s * c) * st1 + bN.b_t * tt1 + (bN.b_q * qo) * t;
  float b_c = (bN.b_s * th) * st1;
  float b_st1 = (bN.b_s * th) * c;
  float b_tt1 = bN.b_t * th;
  const float b_ratio = bN.qq + b_qo * q;
  float b_q = b_qo * ratio;
  const float b_th2 = th > 0.0f ? 0.5f * b_th / th : 0.0f;
  // ratio = sqrt(u), u = p2 / pn2; pn2 = en^2 - m^2; en = e -+ de; e = sqrt(e2)
  const float b_u = 0.5f * b_ratio / ratio;
  const float ipn2 = 1.0f / pn2;
  float b_p2 = b_u * ipn2;
  const float b_pn2 = -(b_u * (p2 * ipn2)) * ipn2;
  const float b_en = 2.0f * en * b_pn2;
  float b_e2 = 0.5f * b_en / e;
  const float b_de = dir > 0 ? -b_en : b_en;
  // de = (dedx ell) (e2 / p2); th2 = (kx ell) (e2 / p2^2); e2 = p2 + m^2
  float b_ell = (G.dedx * (e2 * ip2)) * b_de + (kx * (e2 * (ip2 * ip2))) * b_th2;
  b_e2 += ((G.dedx * ell) * ip2) * b_de + ((kx * ell) * (ip2 * ip2)) * b_th2;
  b_p2 -= ((G.dedx * ell) * (e2 * (ip2 * ip2))) * b_de + 2.0f * ((kx * ell) * (e2 * (ip2 * ip2 * ip2))) * b_th2;
  b_p2 += b_e2;
  // p2 = tt1 / q^2; ell = d st1 / c; st1 = sqrt(tt1); c = sqrt((1 - s)(1 + s)); tt1 = 1 + t^2
  b_tt1 += b_p2 / q2;
  b_q += 2.0f * q * (-(b_p2 * p2) / q2);
  b_st1 += (G.d_row / c) * b_ell;
  b_c -= (ell / c) * b_ell;
  b_tt1 += 0.5f * b_st1 / st1;
  b_t += 2.0f * t * b_tt1;
  b_p[2] = b_p[2] - (s / c) * b_c;
  b_p[3] = b_t;
  b_p[4] = b_q;
}

// Reverse of material_factor.  Lin: the factor it was given (row q not yet
// scaled by qq); F: the factor it returned, lower triangular with
// F F^T = M = G G^T + B B^T, G = diag(1, 1, 1, 1, qq) Lin, B the noise columns
// (b_s in row s; b_t, b_q in rows t, q).  bL in: adjoint of F (its lower
// triangle; the rest of F is structurally zero), out: adjoint of Lin; bN
// receives the adjoints of qq, b_s, b_t, b_q.  From dM = dF F^T + F dF^T with
// F^-1 dF lower triangular: F^-1 dF = Phi(F^-1 dM F^-T), Phi keeping the lower
// triangle with the diagonal halved, hence b_M = F^-T Phi(F^T b_F) F^-1, and
// b_G = (b_M + b_M^T) G, b_B = (b_M + b_M^T) B.  (The Householder arithmetic
// of the forward is not reversed step by step: this is the derivative of the
// map it computes.)
__device__ __forceinline__ void material_factor_rev(const float Lin[5][5], const MatNoise& N, const float F[5][5],
                                                    float bL[5][5], MatNoise& bN) {
  float Fi[5][5];  // F^-1, lower triangular
#pragma unroll
  for (int i = 0; i < 5; ++i) Fi[i][i] = 1.0f / F[i][i];
#pragma unroll
  for (int i = 1; i < 5; ++i)
#pragma unroll
    for (int j = 0; j < i; ++j) {
      float acc = F[i][j] * Fi[j][j];
#pragma unroll
      for (int k = j + 1; k < i; ++k) acc = acc + F[i][k] * Fi[k][j];
      Fi[i][j] = -(acc * Fi[i][i]);
    }
  // P = Phi(F^T b_F): P_ij = sum_{k >= i} F_ki bF_kj (i >= j), diagonal halved
  float P[5][5];
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int j = 0; j <= i; ++j) {
      float acc = F[i][i] * bL[i][j];
#pragma unroll
      for (int k = i + 1; k < 5; ++k) acc = acc + F[k][i] * bL[k][j];
      P[i][j] = i == j ? 0.5f * acc : acc;
    }
  // T = P F^-1 (lower), then b_M = F^-T T
  float Tm[5][5];
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int j = 0; j <= i; ++j) {
      float acc = P[i][j] * Fi[j][j];
#pragma unroll
      for (int k = j + 1; k <= i; ++k) acc = acc + P[i][k] * Fi[k][j];
      Tm[i][j] = acc;
    }
  float Sm[5][5];  // b_M + b_M^T
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      const int k0 = i > j ? i : j;
      float acc = Fi[k0][i] * Tm[k0][j];
#pragma unroll
      for (int k = k0 + 1; k < 5; ++k) acc = acc + Fi[k][i] * Tm[k][j];
      Sm[i][j] = acc;
    }
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int j = 0; j < i; ++j) {
      const float v = Sm[i][j] + Sm[j][i];
      Sm[i][j] = v;
      Sm[j][i] = v;
    }
#pragma unroll
  for (int i = 0; i < 5; ++i) Sm[i][i] = 2.0f * Sm[i][i];
  // b_G = Sm G, G = D Lin
  float qsum = 0.0f;
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      float acc = Sm[i][0] * Lin[0][c];
#pragma unroll
      for (int j = 1; j < 4; ++j) acc = acc + Sm[i][j] * Lin[j][c];
      acc = acc + Sm[i][4] * (N.qq * Lin[4][c]);
      if (i == 4) {
        qsum = qsum + Lin[4][c] * acc;
        bL[i][c] = N.qq * acc;
      } else {
        bL[i][c] = acc;
      }
    }
  bN.qq = qsum;
  bN.b_s = Sm[2][2] * N.b_s;
  bN.b_t = Sm[3][3] * N.b_t + Sm[3][4] * N.b_q;
  bN.b_q = Sm[4][3] * N.b_t + Sm[4][4] * N.b_q;
}

// step_rev with the material layers of the rows.  Outward (conv): prediction,
// layer crossed on arrival (material_step on the predicted state), transport,
// noise folded (material_factor), updates.  Inward: the layer of the row left
// undone first (on the state before the step), then prediction, transport and
// updates.  Arguments as for step_rev.
template <int FIELD = 0>
__device__ __forceinline__ void step_rev_mat(const GeoRef& G, const SmemTables& T, const float4* src, float my_prev, float mz_prev,
                                             bool first, bool conv, int row, int sec18, float m0, float m1,
                                             float b_p[5], float b_L[5][5], float b_chi, float b_mc[2],
                                             float b_mp[2]) {
  StepState S0;
  read_state(src, S0);
  float p1[5];   // the state the updates start from
  float pb[5];   // outward: predicted state before the layer; inward: S0.p after undoing it
  float Lb[5][5];  // outward: transported factor before the noise; inward: S0.L after the layer
  Jac J;
  float L[5][5];
  PredTape tp;
  MatNoise N;
  if (first) {
#pragma unroll
    for (int c = 0; c < 5; ++c) p1[c] = S0.p[c];
    if (conv) {
      p1[0] = S0.p[0] - m0;
      p1[1] = S0.p[1] - m1;
    }
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
      for (int c = 0; c < 5; ++c) L[i][c] = S0.L[i][c];
  } else if (conv) {
    predict_residual<FIELD>(G, T, S0.p, S0.x, S0.sec, my_prev, mz_prev, sec18, T.row_x[row], m0, m1, p1, J, tp);
#pragma unroll
    for (int c = 0; c < 5; ++c) pb[c] = p1[c];
    material_step(G, p1, 1, N);
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
      for (int c = 0; c < 5; ++c) L[i][c] = S0.L[i][c];
    transport(L, J);
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
      for (int c = 0; c < 5; ++c) Lb[i][c] = L[i][c];
    material_factor(L, N);
  } else {
#pragma unroll
    for (int c = 0; c < 5; ++c) pb[c] = S0.p[c];
    material_step(G, pb, -1, N);
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
      for (int c = 0; c < 5; ++c) Lb[i][c] = S0.L[i][c];
    material_factor(Lb, N);
    predict_residual<FIELD>(G, T, pb, S0.x, S0.sec, my_prev, mz_prev, sec18, T.row_x[row], m0, m1, p1, J, tp);
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
      for (int c = 0; c < 5; ++c) L[i][c] = Lb[i][c];
    transport(L, J);
  }
  float p2[5];
  float chi_dummy = 0.0f, b_dummy = 0.0f;
#pragma unroll
  for (int c = 0; c < 5; ++c) p2[c] = p1[c];
  float L2[5][5];
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int c = 0; c < 5; ++c) L2[i][c] = L[i][c];
  scalar_update<0>(G, p2, L2, chi_dummy, 0.0f);
  scalar_update_rev<1>(G, p2, L2, 0.0f, b_p, b_L, b_chi, b_dummy);
  scalar_update_rev<0>(G, p1, L, 0.0f, b_p, b_L, b_chi, b_dummy);
  // b_p: adjoint of the (shifted) state the updates started from; the layers
  // change only q, so its y, z entries are those of the prediction
  b_mc[0] = -b_p[0];
  b_mc[1] = -b_p[1];
  b_mp[0] = 0.0f;
  b_mp[1] = 0.0f;
  if (first) {
    if (!conv) b_mc[0] = b_mc[1] = 0.0f;
    return;
  }
  reread_state(src, S0);
  const bool rot = S0.sec != sec18;
  JacBar bJ;
  MatNoise bN;
  float b_pi[5], b_yo, b_zo;
  if (conv) {
    material_factor_rev(Lb, N, L, b_L, bN);
    material_step_rev(G, pb, 1, bN, b_p);
    if (!rot) {
      b_mp[0] = b_p[0];
      b_mp[1] = b_p[1];
    }
    transport_rev(S0.L, J, b_L, bJ);
    predict_rev<FIELD>(G, tp, J, S0.p[3], S0.p[4], b_p, bJ, b_pi, b_yo, b_zo);
  } else {
    if (!rot) {
      b_mp[0] = b_p[0];
      b_mp[1] = b_p[1];
    }
    transport_rev(Lb, J, b_L, bJ);
    predict_rev<FIELD>(G, tp, J, pb[3], pb[4], b_p, bJ, b_pi, b_yo, b_zo);
    material_factor_rev(S0.L, N, Lb, b_L, bN);
    material_step_rev(G, S0.p, -1, bN, b_pi);
  }
  if (rot) {
    b_mp[0] = b_pi[0];
    b_mp[1] = b_pi[1];
  } else if (FIELD == 1) {
    b_mp[0] += b_yo;
    b_mp[1] += b_zo;
  }
#pragma unroll
  for (int c = 0; c < 5; ++c) b_p[c] = b_pi[c];
}

}  // namespace TPCFIT_NS
}  // namespace tpcfit

#include "ud_core.cuh"

namespace tpcfit {
namespace TPCFIT_NS {

// Fire-and-forget global float add (no value returned, nothing to wait for).
// No kernel reads the sums back, so the add carries no ordering constraint
// (no memory clobber): the compiler may schedule other accesses around it.
__device__ __forceinline__ void red_add(float* p, float v) {
  asm volatile("red.global.add.f32 [%0], %1;\n" ::"l"(__cvta_generic_to_global(p)), "f"(v));
}
// The same for two adjacent floats at an 8-byte-aligned address (each element
// added atomically): half the atomic operations at the alignment table, whose
// keys several lanes hit at once.
__device__ __forceinline__ void red_add2(float* p, float v0, float v1) {
  asm volatile("red.global.add.v2.f32 [%0], {%1, %2};\n" ::"l"(__cvta_generic_to_global(p)), "f"(v0), "f"(v1));
}

// prev: what the inward pass left at cluster h (read ahead by the caller; only
// the outward pass, pass 0, adds to it).  The clusters that no step of a fitted track
// reaches were cleared before (launch_clear_gradients).
__device__ __forceinline__ void accumulate_meas_grad(const BwdArgs& a, int pass, int h, int row, int sec, float g0,
                                                     float g1, float2 prev) {
  if (a.grad_meas) {
    float2* gm = reinterpret_cast<float2*>(a.grad_meas) + h;
    if (pass == 1) {
      *gm = make_float2(g0, g1);
    } else {
      *gm = make_float2(prev.x + g0, prev.y + g1);
    }
  }
  if (a.grad_align_atomic) {
    float* dst = a.grad_align_atomic + (sec * kMaxRows + row) * 2;
    if ((reinterpret_cast<uintptr_t>(dst) & 7u) == 0) {
      red_add2(dst, -g0, -g1);  // one atomic for the key's (dy, dz) pair
    } else {
      red_add(dst, -g0);
      red_add(dst + 1, -g1);
    }
  }
}

// Shared memory of a backward block (from checkpoints): geometry tables, the alignment table
// and, per warp, a double buffer for the state before the step being reversed
// and a buffer for the next segment's checkpoint (all [float4 j][lane]).
struct BwdSmem {
  SmemTables T;
  float align[kAlignFloats];
};
// F4: float4 per stored state (kStateF4 for the square-root form, kUDStateF4
// for U-D); the checkpoint buffer always holds kStateF4.
template <int F4 = kStateF4>
struct BwdWarpBufsT {
  float4 st[2][F4][kWarp];
  float4 ck[kStateF4][kWarp];
};
using BwdWarpBufs = BwdWarpBufsT<>;

template <int WARPS, int FORM = 0>
constexpr size_t backward_smem_bytes() {
  return sizeof(BwdSmem) + WARPS * sizeof(BwdWarpBufsT<FORM ? kUDStateF4 : kStateF4>);
}

// Per track, per pass (inward reversed first), segment by segment from the
// last: recompute the segment from its checkpoint, storing the state before
// each step in the warp's global segment store; then reverse the steps, last
// first, each state copied into shared memory asynchronously one step ahead.
// Clusters are loaded one step ahead as well; the next segment's checkpoint
// is copied while the current segment is reversed.
// Fast mode without material layers.  PHYS: bit 2 the field map.  FORM: the factor
// the segments are recomputed in, 0 the fit's square-root factor L, 1 U-D (a
// checkpoint's L is converted where a segment starts).
template <int WARPS, int PHYS, int FORM = 0>
__global__ void __launch_bounds__(WARPS * 32, 1) backward_kernel(const __grid_constant__ BwdArgs a) {
  const GeoRef& G = a.geo;
  constexpr int FIELD = (PHYS & 2) ? 1 : 0;
  constexpr int F4 = FORM ? kUDStateF4 : kStateF4;
  using State = typename std::conditional<FORM == 1, UDState, StepState>::type;
  // after a taped fit only the items that found no room on the tape are left
  // (none, unless tracks overlap or have more than 255 clusters)
  if (a.tape_item && a.work[kWorkMissing] == 0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  BwdSmem& B = *reinterpret_cast<BwdSmem*>(smem_raw);
  load_block_tables(G, B.T, B.align, a.align);
  const SmemTables& T = B.T;
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  BwdWarpBufsT<F4>& W = reinterpret_cast<BwdWarpBufsT<F4>*>(smem_raw + sizeof(BwdSmem))[warp];
  // this warp's segment store: [step kk][float4 j][lane]
  float4* const gs = a.seg + ((int64_t)blockIdx.x * WARPS + warp) * (kCkptEvery * F4 * kWarp) + lane;
  const int64_t n_items = ((int64_t)a.n_tracks + a.item_tracks - 1) / a.item_tracks;
  const int64_t N = a.n_tracks;
#pragma unroll 1
  for (bool first = true;; first = false) {
    const int64_t item = next_item(a.work, n_items, first);
    if (item < 0) break;
    if (a.tape_item && a.tape_item[item].x >= 0) continue;
    const int64_t slot = item * a.item_tracks + lane;
    if (lane >= a.item_tracks || slot >= N) continue;
    const int32_t trk = a.perm ? a.perm[slot] : (int32_t)slot;
    const float g = __ldg(a.grad_chi2 + trk);
    const RecordedTrack track = recorded_track(a, trk);
    const int begin = track.begin, steps = track.steps;
    float b_p[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    if (steps > 0) {
      const int last = steps - 1;
      float b_L[5][5];         // FORM 0: adjoint of the square-root factor
      float b_u[10], b_d[5];   // FORM 1: adjoint of the U-D factor
#pragma unroll 1
      for (int pass = 1; pass >= 0; --pass) {
#pragma unroll
        for (int i = 0; i < 5; ++i)
#pragma unroll
          for (int c = 0; c < 5; ++c) b_L[i][c] = 0.0f;
#pragma unroll
        for (int e = 0; e < 10; ++e) b_u[e] = 0.0f;
#pragma unroll
        for (int c = 0; c < 5; ++c) b_d[c] = 0.0f;
        const float b_chi = pass == 1 ? g : 0.0f;
        const int nseg = (steps + kCkptEvery - 1) / kCkptEvery;
        // hit index of step i of this pass
        const int h0 = pass == 0 ? begin : begin + last;
        const int hd = pass == 0 ? 1 : -1;
        const float* ckp = a.ck + ((int64_t)pass * a.ck_slots + (begin >> kCkptShift) + trk) * kCkptFloats;
        float pend0 = 0.0f, pend1 = 0.0f;  // gradient owed to the measurement of the step before
        // the outward pass adds to the inward pass's gradient of each cluster:
        // that value is read one reversed step ahead
        const float2* const gmr = reinterpret_cast<const float2*>(a.grad_meas);
        const bool addg = pass == 0 && gmr != nullptr;
        float2 gnx = addg ? gmr[h0 + hd * (steps - 1)] : make_float2(0.0f, 0.0f);
        fetch_ckpt(&W.ck[0][lane], ckp + (int64_t)(nseg - 1) * kCkptFloats);
        // a segment's first cluster and the one before it, loaded a segment
        // ahead; pv: the reverse's previous cluster, carried across segments
        HitRaw seg_first = load_hit(a, h0 + hd * ((nseg - 1) * kCkptEvery));
        HitRaw seg_prev{};
        if (nseg > 1) seg_prev = load_hit(a, h0 + hd * ((nseg - 1) * kCkptEvery - 1));
        HitRaw pv{};
#pragma unroll 1
        for (int s = nseg - 1; s >= 0; --s) {
          const int i0 = s * kCkptEvery;
          const int cnt = min(kCkptEvery, steps - i0);
          State S;
          float my = 0.0f, mz = 0.0f;
          HitRaw nx = seg_first;
          if (i0 > 0) {
            int row, sec;
            decode_hit(B.align, seg_prev, my, mz, row, sec);
          }
          cp_async_wait<0>();
          if constexpr (FORM == 1) {
            StepState C;
            read_state(&W.ck[0][lane], C);
            ud_state_from(C, a.ck_form == 1, S);
          } else {
            read_state(&W.ck[0][lane], S);
          }
          // level 1: the segment, storing the state before each step
          float m0 = 0.0f, m1 = 0.0f;
          int row = 0, sec = 0;
#pragma unroll 1
          for (int kk = 0; kk < cnt; ++kk) {
            const int i = i0 + kk;
            const HitRaw cur = nx;
            if (kk + 1 < cnt) nx = load_hit(a, h0 + hd * (i + 1));
            decode_hit(B.align, cur, m0, m1, row, sec);
            store_state(gs + kk * (F4 * kWarp), S);
            if constexpr (FORM == 1)
              step_fwd_ud<FIELD>(G, T, S, my, mz, i == 0, pass == 0, T.row_x[row], side_sector(sec), m0, m1);
            else
              step_fwd<false, FIELD>(G, T, S, my, mz, i == 0, pass == 0, row, side_sector(sec), m0, m1);
          }
          // the states just stored are read back by this thread's copies below
          __threadfence_block();
          // the next segment's checkpoint travels while this one is reversed.
          // Copy groups complete in order, so it is committed after the
          // loop's first state copy: the first reverse step then waits only
          // for its own state (a one-step segment commits it here)
          const bool ck_next = s > 0;
          if (ck_next && cnt == 1) fetch_ckpt(&W.ck[0][lane], ckp + (int64_t)(s - 1) * kCkptFloats);
          // reverse; (m0, m1, row, sec) hold the segment's last cluster, which is
          // the current cluster of its last step; each step's previous cluster
          // becomes the current one of the step before it
          fetch_state<F4>(&W.st[(cnt - 1) & 1][0][lane], gs + (cnt - 1) * (F4 * kWarp));
          // (in later segments the reverse of the segment after this one left
          // this cluster in pv)
          if (s == nseg - 1 && i0 + cnt - 1 > 0) pv = load_hit(a, h0 + hd * (i0 + cnt - 2));
          if (s > 0) {
            seg_first = load_hit(a, h0 + hd * (i0 - kCkptEvery));
            if (i0 - kCkptEvery > 0) seg_prev = load_hit(a, h0 + hd * (i0 - kCkptEvery - 1));
          }
#pragma unroll 1
          for (int kk = cnt - 1; kk >= 0; --kk) {
            const int i = i0 + kk;
            const int h = h0 + hd * i;
            if (kk > 0) {
              fetch_state<F4>(&W.st[(kk - 1) & 1][0][lane], gs + (kk - 1) * (F4 * kWarp));
              if (ck_next && kk == cnt - 1) {
                fetch_ckpt(&W.ck[0][lane], ckp + (int64_t)(s - 1) * kCkptFloats);
                cp_async_wait<2>();
              } else {
                cp_async_wait<1>();
              }
            } else {
              cp_async_wait<0>();
            }
            float mpy = 0.0f, mpz = 0.0f;
            int prow = 0, psec = 0;
            if (i > 0) {
              const HitRaw pc = pv;
              if (i > 1) pv = load_hit(a, h - 2 * hd);
              decode_hit(B.align, pc, mpy, mpz, prow, psec);
            }
            const float2 gcur = gnx;
            if (addg && i > 0) gnx = gmr[h - hd];
            float b_mc[2], b_mp[2];
            if constexpr (FORM == 1) {
              step_rev_ud<FIELD>(G, T, &W.st[kk & 1][0][lane], mpy, mpz, T.row_x[prow], side_sector(psec), i == 0,
                                 pass == 0, T.row_x[row], side_sector(sec), m0, m1, b_p, b_u, b_d, b_chi,
                                 [&](float g0, float g1) {
                                   accumulate_meas_grad(a, pass, h, row, sec, g0 + pend0, g1 + pend1, gcur);
                                 },
                                 b_mp);
            } else {
              step_rev<FIELD>(G, T, &W.st[kk & 1][0][lane], mpy, mpz, i == 0, pass == 0, row, side_sector(sec), m0, m1,
                              b_p, b_L, b_chi, b_mc, b_mp);
              accumulate_meas_grad(a, pass, h, row, sec, b_mc[0] + pend0, b_mc[1] + pend1, gcur);
            }
            pend0 = b_mp[0];
            pend1 = b_mp[1];
            m0 = mpy;
            m1 = mpz;
            row = prow;
            sec = psec;
          }
        }
        // the inward pass starts from the outward result with the factor reset:
        // b_p carries over, b_L does not
      }
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) a.grad_seeds[(int64_t)c * N + trk] = b_p[c];
  }
}

// ---------------------------------------------------------------- the tape
// Reverse of both passes from the recorded fit's tape (inward pass first).  The
// states are copied into shared memory ahead of their use, as contiguous rows.
// The steps of a pass run over the warp's longest track for all its lanes
// together (a lane of a shorter track joins when its last step comes), so that
// lanes of different lengths stay converged.

// The lane's float4 of row 0 of an item.
__device__ __forceinline__ const float4* tape_row0(const float4* tape, int2 place, int pitch, int lane) {
  return tape + (int64_t)place.x * pitch + lane;
}

template <int ROWS>
__device__ __forceinline__ void copy_rows(float4* sdst, const float4* src, int pitch) {
#pragma unroll
  for (int j = 0; j < ROWS; ++j) cp_async16(sdst + j * kWarp, src + j * pitch);
}

// U-D form (fast mode without material layers).  The fit stores the state before
// every EVERY-th step; with EVERY = 2 the odd states are recomputed from the even
// ones.  Per warp, EVERY steps ("a group") at a time: three groups in shared
// memory, the one being reversed, the one before it (its last cluster is the
// previous cluster of this one's first step) and one on its way.
//
// EVERY = 1 writes and reads 176 bytes a cluster and recomputes nothing: for
// batches that wait for their longest tracks rather than for memory.  EVERY = 2
// halves the states: the fit of 400,000 tracks writes at 4 TB/s, which with every
// state takes 1.54 ms (0.73 unrecorded).  Clusters are stored once for both
// passes, with the alignment taken off, so the reverse needs neither the hits nor
// the alignment table.
template <int EVERY>
struct TapeGroup {
  float4 state[kUDRows][kWarp];
  float4 cluster[EVERY][kWarp];
};
template <int EVERY>
struct TapeWarpUD {
  TapeGroup<EVERY> g[3];
  float4 odd[EVERY - 1 ? kUDRows : 1][kWarp];  // the recomputed state
};
template <>
struct TapeWarpUD<1> {
  TapeGroup<1> g[3];
};

template <int WARPS, int PHYS, int EVERY>
__global__ void __launch_bounds__(WARPS * 32, 1) tape_reverse_ud_kernel(const __grid_constant__ BwdArgs a) {
  const GeoRef& G = a.geo;
  constexpr int FIELD = (PHYS & 2) ? 1 : 0;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmemTables& T = *reinterpret_cast<SmemTables*>(smem_raw);
  load_tables(G, T);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  TapeWarpUD<EVERY>& W = reinterpret_cast<TapeWarpUD<EVERY>*>(smem_raw + sizeof(SmemTables))[threadIdx.x >> 5];
  const int pitch = a.item_tracks;
  const int64_t n_items = ((int64_t)a.n_tracks + pitch - 1) / pitch;
  const int64_t N = a.n_tracks;
#pragma unroll 1
  for (bool first = true;; first = false) {
    const int64_t item = next_item(a.work, n_items, first);
    if (item < 0) break;
    const int2 place = a.tape_item[item];
    if (place.x < 0) continue;  // left to backward_kernel
    const int64_t slot = item * pitch + lane;
    const bool have = lane < pitch && slot < N;
    const int32_t trk = have ? (a.perm ? a.perm[slot] : (int32_t)slot) : 0;
    const RecordedTrack track = have ? recorded_track(a, trk) : RecordedTrack();
    const int begin = track.begin, steps = track.steps;
    const float g = steps > 0 ? __ldg(a.grad_chi2 + trk) : 0.0f;
    const int most = __reduce_max_sync(0xffffffffu, steps);
    const float4* const row0 = tape_row0(a.tape, place, pitch, lane);
    float b_p[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
    for (int pass = 1; pass >= 0; --pass) {
      float b_u[10], b_d[5];
#pragma unroll
      for (int e = 0; e < 10; ++e) b_u[e] = 0.0f;
#pragma unroll
      for (int c = 0; c < 5; ++c) b_d[c] = 0.0f;
      const float b_chi = pass == 1 ? g : 0.0f;
      // the outward pass adds to the inward pass's gradient of each cluster:
      // that value is read one reversed step ahead
      const bool addg = pass == 0 && a.grad_meas != nullptr;
      const float2* const gmr = reinterpret_cast<const float2*>(a.grad_meas);
      const int h0 = pass == 0 ? begin : begin + steps - 1, hd = pass == 0 ? 1 : -1;
      float2 gnx = addg && steps > 0 ? gmr[h0 + hd * (steps - 1)] : make_float2(0.0f, 0.0f);
      float pend0 = 0.0f, pend1 = 0.0f;  // gradient owed to the measurement of the step before
      // step i of the pass: cluster row c0 + cd i, state i / EVERY
      const float4* const clusters = row0 + (pass == 0 ? 0 : steps - 1) * pitch;
      const int cd = hd * pitch;
      const float4* const states = row0 + (place.y + kUDRows * pass * (int)tape_states(place.y, EVERY)) * pitch;
      auto fetch = [&](TapeGroup<EVERY>& to, int grp) {
        const int i = grp * EVERY;
        if (i >= 0 && i < steps) {
          copy_rows<kUDRows>(&to.state[0][lane], states + grp * (kUDRows * pitch), pitch);
#pragma unroll
          for (int k = 0; k < EVERY; ++k)
            if (k == 0 || i + k < steps) cp_async16(&to.cluster[k][lane], clusters + (i + k) * cd);
        }
        cp_async_commit();
      };
      const int last_grp = most > 0 ? (most - 1) / EVERY : -1;
      fetch(W.g[0], last_grp);
      fetch(W.g[1], last_grp - 1);
      int s0 = 0, s1 = 1, s2 = 2;  // places of groups grp, grp - 1, grp - 2
#pragma unroll 1
      for (int i = most - 1; i >= 0; --i) {
        const int k = EVERY == 1 ? 0 : i & 1;  // place in the group
        if (EVERY == 1 || k == 1 || i == most - 1) {
          fetch(W.g[s2], i / EVERY - 2);
          cp_async_wait<1>();  // groups i / EVERY and the one before are in place
        }
        if (i < steps) {
          const float4* src = &W.g[s0].state[0][lane];
          const float4 cur = W.g[s0].cluster[k][lane];
          float4 prv = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          if (k > 0)
            prv = W.g[s0].cluster[0][lane];
          else if (i > 0)
            prv = W.g[s1].cluster[EVERY - 1][lane];
          const int rs = __float_as_int(cur.w);
          if constexpr (EVERY == 2) {
            if (k == 1) {  // the state before this step: forward of the step before it (cluster prv)
              UDState S;
              read_state_ud<false>(src, S);
              float4 pp = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
              if (i > 1) pp = W.g[s1].cluster[EVERY - 1][lane];
              S.x = pp.z;
              S.sec = side_sector(__float_as_int(pp.w) & 63);
              step_fwd_ud<FIELD>(G, T, S, pp.x, pp.y, i == 1, pass == 0, prv.z,
                                 side_sector(__float_as_int(prv.w) & 63), prv.x, prv.y);
              src = &W.odd[0][lane];
              store_state(&W.odd[0][lane], S);
            }
          }
          const float2 gcur = gnx;
          const int h = h0 + hd * i;
          if (addg && i > 0) gnx = gmr[h - hd];
          float b_mp[2];
          step_rev_ud<FIELD>(G, T, src, prv.x, prv.y, prv.z, side_sector(__float_as_int(prv.w) & 63), i == 0,
                             pass == 0, cur.z, side_sector(rs & 63), cur.x, cur.y, b_p, b_u, b_d, b_chi,
                             [&](float g0, float g1) {
                               accumulate_meas_grad(a, pass, h, rs >> 6, rs & 63, g0 + pend0, g1 + pend1, gcur);
                             },
                             b_mp);
          pend0 = b_mp[0];
          pend1 = b_mp[1];
        }
        if (k == 0) {
          const int t = s0;
          s0 = s1;
          s1 = s2;
          s2 = t;
        }
      }
      // the inward pass starts from the outward result with the factor reset:
      // b_p carries over, b_u and b_d do not
      cp_async_wait<0>();
    }
    if (!have) continue;
#pragma unroll
    for (int c = 0; c < 5; ++c) a.grad_seeds[(int64_t)c * N + trk] = b_p[c];
  }
}

constexpr size_t kTapeWarpSmemSqrt = sizeof(float4) * 2 * kSqrtRows * kWarp;

// The states of steps [i0, i0 + cnt) of a pass, recomputed from the checkpoint of
// step i0 into the warp's segment store (gs: this lane's float4 0 of it).  h: the
// cluster of step 0, hd: from one step's cluster to the next.  Not inlined: it
// runs for the items without a place on the tape only.
template <bool MAT, int FIELD>
__device__ __noinline__ void recompute_segment(const BwdArgs& a, const SmemTables& T, const float* align,
                                               const float* ck, float4* gs, int h, int hd, int i0, int cnt, bool conv) {
  StepState S;
  {
    const float4* c4 = reinterpret_cast<const float4*>(ck);
    float v[32];
#pragma unroll
    for (int j = 0; j < kStateF4; ++j) {
      const float4 f = __ldg(c4 + j);
      v[4 * j] = f.x;
      v[4 * j + 1] = f.y;
      v[4 * j + 2] = f.z;
      v[4 * j + 3] = f.w;
    }
    unpack_state(v, S);
  }
  float my = 0.0f, mz = 0.0f;
  if (i0 > 0) {
    int row, sec;
    decode_hit(align, load_hit(a, h + hd * (i0 - 1)), my, mz, row, sec);
  }
#pragma unroll 1
  for (int kk = 0; kk < cnt; ++kk) {
    float m0, m1;
    int row, sec;
    decode_hit(align, load_hit(a, h + hd * (i0 + kk)), m0, m1, row, sec);
    store_state(gs + kk * (kStateF4 * kWarp), S);
    step_fwd<MAT, FIELD>(a.geo, T, S, my, mz, i0 + kk == 0, conv, row, side_sector(sec), m0, m1);
  }
}

// Square-root form (deterministic mode; material layers).  An item without a place
// on the tape is recomputed segment by segment instead, in the same reverse loop.
template <int WARPS, int PHYS>
__global__ void __launch_bounds__(WARPS * 32, 1) tape_reverse_kernel(const __grid_constant__ BwdArgs a) {
  const GeoRef& G = a.geo;
  constexpr bool MAT = (PHYS & 1) != 0;
  constexpr int FIELD = (PHYS & 2) ? 1 : 0;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  BwdSmem& B = *reinterpret_cast<BwdSmem*>(smem_raw);
  load_block_tables(G, B.T, B.align, a.align);
  const SmemTables& T = B.T;
  const int lane = threadIdx.x & 31;
  float4 (*const st)[kSqrtRows][kWarp] =
      reinterpret_cast<float4 (*)[kSqrtRows][kWarp]>(smem_raw + sizeof(BwdSmem)) + 2 * (threadIdx.x >> 5);
  float4* const gs =
      a.seg + ((int64_t)blockIdx.x * WARPS + (threadIdx.x >> 5)) * (kCkptEvery * kStateF4 * kWarp) + lane;
  const int pitch = a.item_tracks;
  const int64_t n_items = ((int64_t)a.n_tracks + pitch - 1) / pitch;
  const int64_t N = a.n_tracks;
#pragma unroll 1
  for (bool first = true;; first = false) {
    const int64_t item = next_item(a.work, n_items, first);
    if (item < 0) break;
    const int2 place = a.tape_item ? a.tape_item[item] : make_int2(-1, 0);
    const bool taped = place.x >= 0;
    const int64_t slot = item * pitch + lane;
    const bool have = lane < pitch && slot < N;
    const int32_t trk = have ? (a.perm ? a.perm[slot] : (int32_t)slot) : 0;
    const RecordedTrack track = have ? recorded_track(a, trk) : RecordedTrack();
    const int begin = track.begin, steps = track.steps;
    const float g = steps > 0 ? __ldg(a.grad_chi2 + trk) : 0.0f;
    const int most = __reduce_max_sync(0xffffffffu, steps);
    float b_p[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
    for (int pass = 1; pass >= 0; --pass) {
      float b_L[5][5];
#pragma unroll
      for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int c = 0; c < 5; ++c) b_L[i][c] = 0.0f;
      const float b_chi = pass == 1 ? g : 0.0f;
      const int h0 = pass == 0 ? begin : begin + steps - 1, hd = pass == 0 ? 1 : -1;
      const bool addg = pass == 0 && a.grad_meas != nullptr;
      const float2* const gmr = reinterpret_cast<const float2*>(a.grad_meas);
      float2 gnx = addg && steps > 0 ? gmr[h0 + hd * (steps - 1)] : make_float2(0.0f, 0.0f);
      float pend0 = 0.0f, pend1 = 0.0f;  // gradient owed to the measurement of the step before
      float m0 = 0.0f, m1 = 0.0f;
      int row = 0, sec = 0;
      if (steps > 0) decode_hit(B.align, load_hit(a, h0 + hd * (steps - 1)), m0, m1, row, sec);
      HitRaw pv{};
      if (steps > 1) pv = load_hit(a, h0 + hd * (steps - 2));
      // steps [lo, hi) at a time: the whole pass from the tape, else a segment
      int hi = most;
#pragma unroll 1
      while (hi > 0) {
        int lo = 0;
        const float4* sp = gs;  // this lane's float4 0 of step lo
        int sp_pitch = kWarp;
        if (taped) {
          sp = tape_row0(a.tape, place, pitch, lane) + kSqrtRows * pass * place.y * pitch;
          sp_pitch = pitch;
        } else {
          lo = (hi - 1) & ~(kCkptEvery - 1);
          if (lo < steps)
            recompute_segment<MAT, FIELD>(
                a, T, B.align,
                a.ck + ((int64_t)pass * a.ck_slots + (begin >> kCkptShift) + trk + (lo >> kCkptShift)) * kCkptFloats, gs,
                h0, hd, lo, min(hi, steps) - lo, pass == 0);
          __threadfence_block();  // the states just stored are read back by this thread's copies below
        }
        const int step_f4 = kSqrtRows * sp_pitch;
        if (hi - 1 < steps) copy_rows<kSqrtRows>(&st[(hi - 1) & 1][0][lane], sp + (hi - 1 - lo) * step_f4, sp_pitch);
        cp_async_commit();
#pragma unroll 1
        for (int i = hi - 1; i >= lo; --i) {
          if (i > lo && i - 1 < steps)
            copy_rows<kSqrtRows>(&st[(i - 1) & 1][0][lane], sp + (i - 1 - lo) * step_f4, sp_pitch);
          cp_async_commit();
          cp_async_wait<1>();
          if (i < steps) {
            const int h = h0 + hd * i;
            float mpy = 0.0f, mpz = 0.0f;
            int prow = 0, psec = 0;
            if (i > 0) {
              const HitRaw pc = pv;
              if (i > 1) pv = load_hit(a, h - 2 * hd);
              decode_hit(B.align, pc, mpy, mpz, prow, psec);
            }
            const float2 gcur = gnx;
            if (addg && i > 0) gnx = gmr[h - hd];
            float b_mc[2], b_mp[2];
            if (MAT)
              step_rev_mat<FIELD>(G, T, &st[i & 1][0][lane], mpy, mpz, i == 0, pass == 0, row, side_sector(sec), m0,
                                  m1, b_p, b_L, b_chi, b_mc, b_mp);
            else
              step_rev<FIELD>(G, T, &st[i & 1][0][lane], mpy, mpz, i == 0, pass == 0, row, side_sector(sec), m0, m1,
                              b_p, b_L, b_chi, b_mc, b_mp);
            accumulate_meas_grad(a, pass, h, row, sec, b_mc[0] + pend0, b_mc[1] + pend1, gcur);
            pend0 = b_mp[0];
            pend1 = b_mp[1];
            m0 = mpy;
            m1 = mpz;
            row = prow;
            sec = psec;
          }
        }
        hi = lo;
        cp_async_wait<0>();
      }
      // the inward pass starts from the outward result with the factor reset:
      // b_p carries over, b_L does not
    }
    if (!have) continue;
#pragma unroll
    for (int c = 0; c < 5; ++c) a.grad_seeds[(int64_t)c * N + trk] = b_p[c];
  }
}

// Persistent launch of a kernel with up to `warps` warps per block, `block_smem`
// bytes of shared memory per block and `warp_smem` per warp.
template <class K, class A>
cudaError_t launch_persistent(K kernel, Resident& r, int warps, size_t block_smem, size_t warp_smem, const A& a,
                              cudaStream_t s) {
  cudaError_t e = resident_blocks(kernel, warps * kWarp, block_smem + warps * warp_smem, r);
  if (e != cudaSuccess) return e;
  const WorkShape w = work_shape(a.n_tracks, r.blocks, warps, r.sms);
  A b = a;
  b.item_tracks = w.tracks;
  if (needs_work_counter(w)) e = cudaMemsetAsync(a.work, 0, sizeof(unsigned int), s);
  if (e != cudaSuccess) return e;
  kernel<<<w.blocks, w.warps * kWarp, block_smem + w.warps * warp_smem, s>>>(b);
  return cudaGetLastError();
}

// Blocks of the one-kernel backward resident at once.
template <int WARPS, int PHYS, int FORM>
Resident& backward_resident() {
  static Resident r;
  return r;
}

template <int WARPS, int PHYS, int FORM>
cudaError_t backward_store_cfg(int64_t& float4s) {
  Resident& r = backward_resident<WARPS, PHYS, FORM>();
  cudaError_t e = resident_blocks(backward_kernel<WARPS, PHYS, FORM>, WARPS * kWarp, backward_smem_bytes<WARPS, FORM>(), r);
  float4s = (int64_t)r.blocks * WARPS * kCkptEvery * (FORM ? kUDStateF4 : kStateF4) * kWarp;
  return e;
}

template <int WARPS, int PHYS, int FORM>
cudaError_t launch_backward_cfg(const BwdArgs& a, cudaStream_t s) {
  return launch_persistent(backward_kernel<WARPS, PHYS, FORM>, backward_resident<WARPS, PHYS, FORM>(), WARPS,
                           sizeof(BwdSmem), sizeof(BwdWarpBufsT<FORM ? kUDStateF4 : kStateF4>), a, s);
}

#if !TPCFIT_DET
// The fast backward from checkpoints without material layers: in a uniform field
// every compiled block shape, with the field map 8 warps.
template <class F>
cudaError_t for_backward_shape(int warps, int phys, F&& f) {
  using std::integral_constant;
  if (phys == 2) return f(integral_constant<int, 8>(), integral_constant<int, 2>());
  if (phys != 0) return cudaErrorInvalidValue;
  switch (warps) {
    case 4: return f(integral_constant<int, 4>(), integral_constant<int, 0>());
    case 8: return f(integral_constant<int, 8>(), integral_constant<int, 0>());
    case 10: return f(integral_constant<int, 10>(), integral_constant<int, 0>());
    case 12: return f(integral_constant<int, 12>(), integral_constant<int, 0>());
    default: return cudaErrorInvalidValue;
  }
}

inline cudaError_t launch_checkpoint_backward(const BwdArgs& a, int warps, cudaStream_t s) {
  return for_backward_shape(warps, a.phys, [&](auto w, auto p) {
    return a.form == 1 ? launch_backward_cfg<w(), p(), 1>(a, s) : launch_backward_cfg<w(), p(), 0>(a, s);
  });
}

// The U-D reverse from the tape: 12 warps (168 registers) where there is work for
// them (400,000 tracks, every state on the tape: 1.96 ms against 2.20 with 8, 212
// registers), 8 otherwise (1,000 tracks: 304 us against 326).
template <int PHYS>
cudaError_t launch_tape_ud(const BwdArgs& a, cudaStream_t s) {
  static Resident r1, r2;
  if (a.tape_every == 1)
    return launch_persistent(tape_reverse_ud_kernel<8, PHYS, 1>, r1, 8, sizeof(SmemTables), sizeof(TapeWarpUD<1>), a, s);
  return launch_persistent(tape_reverse_ud_kernel<12, PHYS, 2>, r2, 12, sizeof(SmemTables), sizeof(TapeWarpUD<2>), a, s);
}
#endif

constexpr int kTapeSqrtWarps = 8;
template <int PHYS>
Resident& tape_sqrt_resident() {
  static Resident r;
  return r;
}
template <int PHYS>
cudaError_t tape_sqrt_store(int64_t& float4s) {
  Resident& r = tape_sqrt_resident<PHYS>();
  const cudaError_t e = resident_blocks(tape_reverse_kernel<kTapeSqrtWarps, PHYS>, kTapeSqrtWarps * kWarp,
                                        sizeof(BwdSmem) + kTapeSqrtWarps * kTapeWarpSmemSqrt, r);
  float4s = (int64_t)r.blocks * kTapeSqrtWarps * kCkptEvery * kStateF4 * kWarp;
  return e;
}
template <int PHYS>
cudaError_t launch_tape_sqrt(const BwdArgs& a, cudaStream_t s) {
  return launch_persistent(tape_reverse_kernel<kTapeSqrtWarps, PHYS>, tape_sqrt_resident<PHYS>(), kTapeSqrtWarps,
                           sizeof(BwdSmem), kTapeWarpSmemSqrt, a, s);
}

// Segment store (float4 count) the backward needs: in fast mode without material
// (form 0 square root, 1 U-D) for the reverse from checkpoints in `warps`-warp
// blocks, otherwise for the items that the tape has no room for.
inline cudaError_t backward_store(int warps, int phys, int form, int64_t& float4s) {
#if !TPCFIT_DET
  if (!(phys & 1))
    return for_backward_shape(warps, phys, [&](auto w, auto p) {
      return form == 1 ? backward_store_cfg<w(), p(), 1>(float4s) : backward_store_cfg<w(), p(), 0>(float4s);
    });
#endif
  switch (phys) {
#if TPCFIT_DET
    case 0: return tape_sqrt_store<0>(float4s);
    case 2: return tape_sqrt_store<2>(float4s);
#endif
    case 1: return tape_sqrt_store<1>(float4s);
    case 3: return tape_sqrt_store<3>(float4s);
    default: return cudaErrorInvalidValue;
  }
}

inline cudaError_t launch_backward(const BwdArgs& a, int warps, cudaStream_t s) {
  if (a.n_tracks <= 0) return cudaSuccess;
#if !TPCFIT_DET
  if (!(a.phys & 1)) {
    // from the tape where the fit left one; the kernel from checkpoints then looks
    // after the items that found no room on it
    if (a.tape) {
      const cudaError_t e = a.phys == 2 ? launch_tape_ud<2>(a, s) : launch_tape_ud<0>(a, s);
      if (e != cudaSuccess) return e;
    }
    return launch_checkpoint_backward(a, warps, s);
  }
#endif
  switch (a.phys) {
#if TPCFIT_DET
    case 0: return launch_tape_sqrt<0>(a, s);
    case 2: return launch_tape_sqrt<2>(a, s);
#endif
    case 1: return launch_tape_sqrt<1>(a, s);
    case 3: return launch_tape_sqrt<3>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace TPCFIT_NS
}  // namespace tpcfit
