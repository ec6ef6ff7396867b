// Reverse mode (adjoint) of one explicit step, for gradients of a loss with
// respect to the initial state, the bed z and Manning's n (through g n^2).
//
// One step maps U^n to U^{n+1} with a fixed dt (Sec. 2.2, Eq. 4 and the
// semi-implicit friction):
//   U*_i     = U^n_i - (dt / Omega_i) R_i,  R_i = sum over faces of s l (F + P n)
//   U^{n+1}_i = friction(U*_i)              (clip of h at 0, momentum / d)
// Given lambda = dL/dU^{n+1},
//   mu_i  = dL/dU*_i          (friction transposed; needs only U^{n+1}, g n^2, dt)
//   rho_i = dL/dR_i = -(dt / Omega_i) mu_i
// and per face the vector-Jacobian product of its two residual contributions
// with (rho_A, rho_B), giving dL/d(h, u, v, z) of both sides; then
//   dL/dU^n_i = mu_i + sum over the cell's faces of its side's part
//               (velocities taken back to hu, hv once per cell),
//   dL/dz_i  += sum of the z parts,  dL/d(g n^2)_i += friction part.
// What a step hands to the one before it is mu, not lambda: the cell's own
// thread has its U^n staged anyway and transposes the friction of step n - 1
// right there, so no step reads U^{n+1} and a halo cell costs its U^n, mu and
// area only.
// Every branch (wet/dry tests, the HLLC case, the min/max of the wave-speed
// estimates and of the reconstruction) is taken as the forward step takes
// it; where the forward picks between two equal values (a tie of max(zA, zB)
// or of the speed estimates) the derivative follows the first argument, the
// convention of the FP64 reference the gradients are checked against.
//
// The friction factor d is recovered from U^{n+1}: with c = dt g n^2 h^{-7/3}
// and q1 = |q^{n+1}|, d = 1 + c |q*| = 1 / (1 - c q1) exactly, so the adjoint
// needs no per-step copy of U* (relative error about eps * d).
// A depth clipped at 0 (never under the CFL step; the forward counts it) is
// differentiated as if it were not clipped.
#pragma once

#include "swe_kernels.cuh"

namespace swe {

// Signs and orders of doubles from their bit patterns (a comparison costs as
// much of the FP64 pipe as a multiply-add).
__device__ __forceinline__ bool below0(double x) {
  return (unsigned long long)__double_as_longlong(x) > 0x8000000000000000ull;
}
__device__ __forceinline__ bool above0(double x) { return __double_as_longlong(x) > 0; }
// a >= b
__device__ __forceinline__ bool at_least(double a, double b) {
  const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
  const long long ka = ia ^ ((ia >> 63) & 0x7fffffffffffffffll);
  const long long kb = ib ^ ((ib >> 63) & 0x7fffffffffffffffll);
  return ka >= kb || ((ia | ib) << 1) == 0;  // -0 and +0 are equal
}
// 2 x for a normal x > 0 (or 0 with pos false)
__device__ __forceinline__ double twice(double x, bool pos) {
  return pos ? __hiloint2double(__double2hiint(x) + 0x00100000, __double2loint(x)) : 0.0;
}

// dL/dU* of one cell from its post-step state (h1, q1x, q1y) and lambda:
// mu (3 values) and the derivative with respect to its g n^2. r1: 1 / h1 of a
// wet cell, which the FP64 form takes (FP32 divides).
__device__ __forceinline__ void cell_vjp(float h1, float q1x, float q1y, float, float lh, float lx,
                                         float ly, float gn2, float dt, const Num& num, float& mh,
                                         float& mx, float& my, float& bgn2) {
  using O = Ops<float>;
  const float zero = 0.0f;
  if (O::wet(h1, num)) {
    const float q1n = O::sqrt_(q1x * q1x + q1y * q1y);
    const float ch = O::friction(dt, 1.0f, 1.0f, h1);  // dt h^{-7/3}
    const float c = ch * gn2;
    const float cq = c * q1n;        // (d - 1) / d
    const float rd = 1.0f - cq;   // 1 / d
    const float ql = q1x * lx + q1y * ly;
    const float k = q1n > zero ? O::div(c * ql, q1n) : zero;
    mx = rd * (lx - k * q1x);
    my = rd * (ly - k * q1y);
    mh = lh + float(7.0 / 3.0) * O::div(cq, h1) * ql;
    bgn2 = -q1n * ch * ql;
  } else {
    mh = lh;
    mx = zero;
    my = zero;
    bgn2 = zero;
  }
}

// FP64: fewer FP64 instructions; the last output is left 0 where g n^2 is 0
// (it only enters dL/dn, multiplied by n).
__device__ __forceinline__ void cell_vjp(double h1, double q1x, double q1y, double r1, double lh,
                                         double lx, double ly, double gn2, double dt, const Num& num,
                                         double& mh, double& mx, double& my, double& bgn2) {
  using O = Ops<double>;
  const double zero = 0.0;
  mh = lh;
  mx = zero;
  my = zero;
  bgn2 = zero;
  if (!O::wet(h1, num)) return;
  mx = lx;
  my = ly;
  if (!above0(gn2)) return;
  const double q1n = O::sqrt_(fma_rn(q1x, q1x, q1y * q1y));
  const double ch = mul_rn(dt, O::pow_m73(h1));
  const double c = ch * gn2;
  const double cq = c * q1n;        // (d - 1) / d
  const double rd = 1.0 - cq;   // 1 / d
  const double ql = fma_rn(q1x, lx, q1y * ly);
  const double k = above0(q1n) ? O::div(c * ql, q1n) : zero;
  mx = rd * fma_rn(-k, q1x, lx);
  my = rd * fma_rn(-k, q1y, ly);
  mh = fma_rn((7.0 / 3.0) * (cq * r1), ql, lh);
  bgn2 = -(q1n * ch) * ql;
}

// Vector-Jacobian product of one face, with both sides' contributions:
// inputs the sides' cells as staged, the geometry, and rho = dL/dR of side A
// (the face adds c_A to R_A) and side B (the face subtracts c_B from R_B);
// outputs gA, gB through this face. FP32: cells (h, hu, hv, z), outputs
// dL/d(h, hu, hv, z). FP64: cells (h, u, v, z), velocities formed once per
// cell (0 on a dry one), outputs dL/d(h, u, v, z), taken back to hu, hv once
// per cell. The face is the clamped form of the flux the tiled steps compute
// (face_flux_f32, face_flux_f64): one HLL formula with the clamped speeds
// S- = min(S_A, 0), S+ = max(S_B, 0), the dry side's normal velocity replaced
// by un_B - 2 c_B (or un_A + 2 c_A) in the wave-speed estimates, the
// transverse momentum upwinded by the sign of F0. It is the same function of
// the inputs as the HLLC case analysis (the clamped speeds reproduce the
// supersonic cases: with S_A >= 0, S- = 0 and F = F_A, whose derivative with
// respect to S_A is 0), so the derivatives agree with the case analysis's
// away from ties; it has no case branches. Ties follow fixed conventions:
// max(zA, zB) and the speed estimates take the first argument, S_A = 0 counts
// as S_A >= 0 and S_B = 0 as S_B <= 0. For a wall B is ignored (the mirror of
// A folds into gA, gB = 0).
//
// FP32 differentiates the formulas as they stand: the shorter FP64 form below
// was no faster in FP32 (29.2 and 29.3 us per step of 1.0M cells), whose bound
// is not its arithmetic.
template <bool Wall>
__device__ __forceinline__ void face_vjp(const V4<float>& A, const V4<float>& B, float nx, float ny,
                                         float len, const Num& num, float rA0, float rA1, float rA2,
                                         float rB0, float rB1, float rB2, float gA[4], float gB[4]) {
  using O = Ops<float>;
  const float zero = 0.0f, half = 0.5f, quarter = 0.25f;
  const float g = float(num.g), hg = half * g;
  // ---- forward, keeping what the reverse sweep needs
  const float rA = O::wet(A.x, num) ? O::div(1.0f, A.x) : zero;  // 0 on a dry cell
  const float uA = A.y * rA, vA = A.z * rA;
  const float unA = uA * nx + vA * ny;
  const float utA = vA * nx - uA * ny;
  float hB, zB, unB, utB, uB = zero, vB = zero, rB = zero;
  if (Wall) {
    hB = A.x; zB = A.w; unB = -unA; utB = utA;
  } else {
    rB = O::wet(B.x, num) ? O::div(1.0f, B.x) : zero;
    uB = B.y * rB;
    vB = B.z * rB;
    hB = B.x; zB = B.w;
    unB = uB * nx + vB * ny;
    utB = vB * nx - uB * ny;
  }
  const bool zsA = A.w >= zB;  // max(zA, zB) taken from A on a tie
  const float zs = zsA ? A.w : zB;
  const float xA = A.x + A.w - zs, xB = hB + zB - zs;
  const bool wetA = O::wet(xA, num), wetB = O::wet(xB, num);  // reconstructed sides wet
  const float hAs = wetA ? xA : zero, hBs = wetB ? xB : zero;
  const float cA = O::sqrt_(g * hAs), cB = O::sqrt_(g * hBs);
  const float vnA = wetA ? unA : unB - 2.0f * cB;
  const float vnB = wetB ? unB : unA + 2.0f * cA;
  const float us = (vnA + vnB) * half + cA - cB;
  const float cs = (cA + cB) * half + (vnA - vnB) * quarter;
  const float a1 = vnA - cA, a2 = us - cs, b1 = vnB + cB, b2 = us + cs;
  const bool firstA = a1 <= a2, firstB = b1 >= b2;
  const float SA = firstA ? a1 : a2, SB = firstB ? b1 : b2;
  const bool negA = SA < zero, posB = SB > zero;
  const float Sm = negA ? SA : zero, Sp = posB ? SB : zero;
  const float qA = hAs * unA, qB = hBs * unB;
  const float FA1 = qA * unA + hg * hAs * hAs, FB1 = qB * unB + hg * hBs * hBs;
  const bool live = wetA || wetB;  // both sides dry: F = 0 whatever the speeds
  const float inv = live ? O::div(1.0f, Sp - Sm) : zero;
  const float SS = Sm * Sp, dh = hBs - hAs, dq = qB - qA;
  const float N0 = Sp * qA - Sm * qB + SS * dh;
  const float N1 = Sp * FA1 - Sm * FB1 + SS * dq;
  const float F0 = N0 * inv;
  const bool upA = F0 >= zero;  // transverse momentum from A where F0 >= 0

  // ---- reverse sweep
  // residual contributions: A gets +l (F0, Fx + PA nx, Fy + PA ny), B gets
  // -l (F0, Fx + PB nx, Fy + PB ny), Fx = F1 nx - F2 ny, Fy = F1 ny + F2 nx
  const float bFx = len * (rA1 - rB1), bFy = len * (rA2 - rB2);
  const float bF1 = bFx * nx + bFy * ny;
  float bF0 = zero, bF2 = zero;
  if (!Wall) {
    bF0 = len * (rA0 - rB0);
    bF2 = bFy * nx - bFx * ny;
  }
  const float bPA = len * (rA1 * nx + rA2 * ny);
  const float bPB = Wall ? zero : -len * (rB1 * nx + rB2 * ny);
  // P = g/2 (h^2 - h*^2)
  float bhA = g * A.x * bPA, bhB = g * hB * bPB;
  float bhAs = -g * hAs * bPA, bhBs = -g * hBs * bPB;
  // F2 = F0 ut
  bF0 += bF2 * (upA ? utA : utB);
  const float but = bF2 * F0;
  float butA = upA ? but : zero, butB = upA ? zero : but;
  // F0 = N0 / D, F1 = N1 / D, D = S+ - S-
  const float bN0 = bF0 * inv, bN1 = bF1 * inv;
  const float bD = -(bF0 * N0 + bF1 * N1) * inv * inv;
  const float bSp = bD + bN0 * (qA + Sm * dh) + bN1 * (FA1 + Sm * dq);
  const float bSm = -bD + bN0 * (Sp * dh - qB) + bN1 * (Sp * dq - FB1);
  float bqA = bN0 * Sp - bN1 * SS, bqB = bN1 * SS - bN0 * Sm;
  bhBs += bN0 * SS;
  bhAs -= bN0 * SS;
  const float bFA1 = bN1 * Sp, bFB1 = -bN1 * Sm;
  // F1 of each side = q un + g/2 h*^2, q = h* un
  bqA += bFA1 * unA;
  bqB += bFB1 * unB;
  float bunA = bFA1 * qA + bqA * hAs, bunB = bFB1 * qB + bqB * hBs;
  bhAs += bFA1 * g * hAs + bqA * unA;
  bhBs += bFB1 * g * hBs + bqB * unB;
  // S- = min(S_A, 0), S+ = max(S_B, 0); the speed estimates
  const float bSA = negA ? bSm : zero, bSB = posB ? bSp : zero;
  float bvnA = zero, bvnB = zero, bcA = zero, bcB = zero, bus = zero, bcs = zero;
  if (firstA) { bvnA += bSA; bcA -= bSA; } else { bus += bSA; bcs -= bSA; }
  if (firstB) { bvnB += bSB; bcB += bSB; } else { bus += bSB; bcs += bSB; }
  bvnA += half * bus + quarter * bcs;
  bvnB += half * bus - quarter * bcs;
  bcA += bus + half * bcs;
  bcB += half * bcs - bus;
  // a dry side's velocity in the estimates
  if (wetA) { bunA += bvnA; } else { bunB += bvnA; bcB -= 2.0f * bvnA; }
  if (wetB) { bunB += bvnB; } else { bunA += bvnB; bcA += 2.0f * bvnB; }
  // c = sqrt(g h*): dc/dh* = g / (2 c) on a wet side (c = 0 and no term on a dry one)
  if (wetA) bhAs += bcA * O::div(hg, cA);
  if (wetB) bhBs += bcB * O::div(hg, cB);
  // reconstruction h* = h + z - max(zA, zB) where it stays wet
  float bzA = zero, bzB = zero, bzs = zero;
  if (wetA) { bhA += bhAs; bzA += bhAs; bzs -= bhAs; }
  if (wetB) { bhB += bhBs; bzB += bhBs; bzs -= bhBs; }
  if (zsA) bzA += bzs; else bzB += bzs;
  if (Wall) {  // B mirrors A: hB = hA, zB = zA, unB = -unA, utB = utA
    bhA += bhB;
    bzA += bzB;
    bunA -= bunB;
    butA += butB;
  }
  // face frame -> x, y velocities -> conserved variables (u = hu r, r = 1/h
  // on a wet cell, 0 on a dry one)
  const float buA = bunA * nx - butA * ny, bvA = bunA * ny + butA * nx;
  gA[0] = bhA - (buA * uA + bvA * vA) * rA;
  gA[1] = buA * rA;
  gA[2] = bvA * rA;
  gA[3] = bzA;
  if (Wall) {
    gB[0] = zero; gB[1] = zero; gB[2] = zero; gB[3] = zero;
  } else {
    const float buB = bunB * nx - butB * ny, bvB = bunB * ny + butB * nx;
    gB[0] = bhB - (buB * uB + bvB * vB) * rB;
    gB[1] = buB * rB;
    gB[2] = bvB * rB;
    gB[3] = bzB;
  }
}

// FP64: the FP64 pipe bounds the adjoint as it bounds the step, so the sweep
// is arranged for few FP64 instructions (115 of them; about 175 when each
// face formed its velocities and differentiated N / D):
//   - with D = S+ - S-, and w- = S- / D, w+ = S+ / D, w = S- S+ / D, F_k of
//     side values f and states q is w+ f_A - w- f_B + w (q_B - q_A), and its
//     derivatives are dF/dS+ = w- (df - S- dq) / D and dF/dS- = -w+ (df - S+ dq) / D
//     (df, dq: B minus A), so neither numerator is formed;
//   - the wave speeds as in face_flux_f64, from their distance to un -+ c;
//   - z enters through the higher side only: one side's part, negated for
//     the other;
//   - signs and orders from bit patterns.
template <bool Wall>
__device__ __forceinline__ void face_vjp(const V4<double>& A, const V4<double>& B, double nx, double ny,
                                         double len, const Num& num, double rA0, double rA1, double rA2,
                                         double rB0, double rB1, double rB2, double gA[4], double gB[4]) {
  using O = Ops<double>;
  const double zero = 0.0, k34 = 0.75, two = 2.0;
  const double g = num.g, hg = 0.5 * g;
  // ---- forward
  const double unA = fma_rn(A.y, nx, A.z * ny);
  const double hB = Wall ? A.x : B.x, zB = Wall ? A.w : B.w;
  const double unB = Wall ? -unA : fma_rn(B.y, nx, B.z * ny);
  const bool zsA = Wall || at_least(A.w, zB);  // max(zA, zB) taken from A on a tie
  const double zs = zsA ? A.w : zB;
  const double xA = sub_rn(add_rn(A.x, A.w), zs), xB = Wall ? xA : sub_rn(add_rn(hB, zB), zs);
  const bool wetA = O::wet(xA, num), wetB = O::wet(xB, num);  // reconstructed sides wet
  const double hAs = wetA ? xA : zero, hBs = wetB ? xB : zero;
  const double pA = hg * hAs, pB = Wall ? pA : hg * hBs;
  const double cA = O::sqrt_(twice(pA, wetA)), cB = Wall ? cA : O::sqrt_(twice(pB, wetB));
  double vnA = unA, vnB = unB;
  if (!(wetA && wetB)) {
    if (!wetA) vnA = fma_rn(-two, cB, unB);
    if (!wetB) vnB = fma_rn(two, cA, unA);
  }
  const double dv = vnB - vnA, dc = cA - cB;
  const double eA = fma_rn(two, dc, dv), eB = fma_rn(two, dc, -dv);
  const bool secA = below0(eA), secB = above0(eB);  // the star-region estimate is the extreme one
  const double SA = fma_rn(k34, secA ? eA : zero, vnA - cA);
  const double SB = fma_rn(k34, secB ? eB : zero, vnB + cB);
  const bool negA = below0(SA), posB = above0(SB);
  const double Sm = negA ? SA : zero, Sp = posB ? SB : zero;
  const double qA = hAs * unA, qB = hBs * unB;
  const double dh = hBs - hAs, dq = qB - qA;
  const double dF = Wall ? zero : fma_rn(qB, unB, pB * hBs) - fma_rn(qA, unA, pA * hAs);
  const bool live = wetA || wetB;  // both sides dry: F = 0 whatever the speeds
  const double inv = live ? O::rcp(Sp - Sm) : zero;
  const double wm = Sm * inv, wp = Sp * inv, ws = Sm * wp;

  // ---- reverse sweep
  // residual contributions: A gets +l (F0, Fx + PA nx, Fy + PA ny), B gets
  // -l (F0, Fx + PB nx, Fy + PB ny), Fx = F1 nx - F2 ny, Fy = F1 ny + F2 nx
  const double gx = len * nx, gy = len * ny;
  const double d1 = Wall ? rA1 : rA1 - rB1, d2 = Wall ? rA2 : rA2 - rB2;
  const double bF1 = fma_rn(d1, gx, d2 * gy);
  // P = g/2 (h^2 - h*^2)
  const double gPA = g * (Wall ? bF1 : fma_rn(rA1, gx, rA2 * gy));
  const double gPB = Wall ? zero : -g * fma_rn(rB1, gx, rB2 * gy);
  double bF0 = zero, but = zero;
  bool upA = true;
  if (!Wall) {
    // F2 = F0 ut, ut of the upwind side
    const double F0 = fma_rn(ws, dh, fma_rn(wp, qA, -(wm * qB)));
    upA = !below0(F0);
    const double uu = upA ? A.y : B.y, vv = upA ? A.z : B.z;
    const double bF2 = fma_rn(d2, gx, -(d1 * gy));
    bF0 = fma_rn(bF2, fma_rn(vv, nx, -(uu * ny)), len * (rA0 - rB0));
    but = bF2 * F0;
  }
  // F0 (states q, h) and F1 (states F, q) of the two sides and the speeds
  const double P = Wall ? zero : fma_rn(bF1, dF, bF0 * dq) * inv;
  const double Q = (Wall ? bF1 * dq : fma_rn(bF1, dq, bF0 * dh)) * inv;
  const double bSB = posB ? wm * fma_rn(-Sm, Q, P) : zero;
  const double bSA = negA ? wp * fma_rn(Sp, Q, -P) : zero;
  const double bFA = bF1 * wp, bFB = -(bF1 * wm), s1 = bF1 * ws, s0 = Wall ? zero : bF0 * ws;
  const double bqA = fma_rn(bFA, unA, Wall ? -s1 : fma_rn(bF0, wp, -s1));
  const double bqB = fma_rn(bFB, unB, Wall ? s1 : fma_rn(-bF0, wm, s1));
  double bunA = fma_rn(bqA, hAs, bFA * qA), bunB = fma_rn(bqB, hBs, bFB * qB);
  double bhAs = fma_rn(fma_rn(g, bFA, -gPA), hAs, fma_rn(bqA, unA, -s0));
  double bhBs = fma_rn(Wall ? g * bFB : fma_rn(g, bFB, -gPB), hBs, fma_rn(bqB, unB, s0));
  // the speed estimates
  const double tA = secA ? k34 * bSA : zero, tB = secB ? k34 * bSB : zero;
  const double td = tA - tB, ts = tA + tB;
  const double bvA = bSA - td, bvB = bSB + td;
  double bcA = fma_rn(two, ts, -bSA), bcB = fma_rn(-two, ts, bSB);
  if (wetA && wetB) {
    bunA += bvA;
    bunB += bvB;
  } else {  // a dry side's velocity in the estimates
    if (wetA) { bunA += bvA; } else { bunB += bvA; bcB = fma_rn(-two, bvA, bcB); }
    if (wetB) { bunB += bvB; } else { bunA += bvB; bcA = fma_rn(two, bvB, bcA); }
  }
  // c = sqrt(g h*): dc/dh* = g / (2 c) on a wet side (c = 0 and no term on a dry one)
  bhAs = wetA ? fma_rn(bcA * hg, O::rcp(cA), bhAs) : zero;
  bhBs = wetB ? fma_rn(bcB * hg, Wall ? O::rcp(cA) : O::rcp(cB), bhBs) : zero;
  // reconstruction h* = h + z - max(zA, zB) where it stays wet
  double bhA = fma_rn(A.x, gPA, bhAs);
  if (Wall) {  // B mirrors A: hB = hA, zB = zA, unB = -unA, utB = utA
    bhA += bhBs;
    bunA -= bunB;
  }
  // face frame -> x, y
  const double tx = but * ny, ty = but * nx;
  gA[0] = bhA;
  gA[1] = Wall ? bunA * nx : fma_rn(bunA, nx, upA ? -tx : zero);
  gA[2] = Wall ? bunA * ny : fma_rn(bunA, ny, upA ? ty : zero);
  gA[3] = Wall ? zero : (zsA ? -bhBs : bhAs);
  if (Wall) {
    gB[0] = zero; gB[1] = zero; gB[2] = zero; gB[3] = zero;
  } else {
    gB[0] = fma_rn(hB, gPB, bhBs);
    gB[1] = fma_rn(bunB, nx, upA ? zero : -tx);
    gB[2] = fma_rn(bunB, ny, upA ? zero : ty);
    gB[3] = zsA ? bhBs : -bhAs;
  }
}

// Loss seeds of the gauges: the ncells distinct cells that hold gauges,
// ascending, those of tile t at tile_first[t] .. tile_first[t + 1] - 1, and for
// each the gauges in it (index[first[c]] .. index[first[c + 1] - 1], in
// ascending order); seed[k G + j] is dL/d(depth at gauge j after step k).
struct GaugeSeeds {
  const int32_t* cells;
  const int32_t* first;
  const int32_t* index;
  const int32_t* tile_first;
  const double* seed;
  int G, ncells;
};

// The seeds of step k of distinct gauge cell c, added to v in a fixed order.
template <typename Real>
__device__ __forceinline__ Real add_seeds(Real v, const GaugeSeeds& g, long long k, int c) {
  for (int q = g.first[c]; q < g.first[c + 1]; ++q) v += Real(g.seed[k * g.G + g.index[q]]);
  return v;
}

// Inputs and outputs of one adjoint launch, step n (interleaved cells,
// internal order, padded to whole tiles).
template <typename Real>
struct AdjArgs {
  const Real* un;      // U^n (h, hu, hv, z)
  const Real* mu_in;   // mu of step n (h, hu, hv), accumulated dL/dz
  Real* mu_out;        // the same of step n - 1; for n = 0 dL/dU^0 and dL/dz
  const Real* gn2;     // g n^2 per cell
  Real* dgn2;          // accumulated dL/d(g n^2) per cell (read-modify-write)
  Real dt, dt_prev;    // time steps of steps n and n - 1
  int split;           // parts per tile (Parts; see k_tiled_adjoint)
  int last;            // 1: n = 0
  int* err;            // kErr* bits (timeouts)
  // Gauge seeds of U^n, added to dL/dh of their cells before the transposed
  // friction of step n - 1 (by the cell's own thread: one thread for all of
  // them at the end of the launch cost 16 us per step with 64 gauges, a
  // dependent trip to L2 each); gstep < 0 adds nothing.
  GaugeSeeds gauges;
  long long gstep;
};

// Shared-memory plan of k_tiled_adjoint. Per stage: the tile's and its
// halo's cells of U^n, the face records with their geometry, the halo list.
// After the stages: rho per tile and halo cell (a halo cell's mu lands here
// and is scaled in place), the halo cells' areas, the face slots
// (dh, du, dv, dz) per face of each tile cell, face-major (placed as the
// step's, see kSlotPad), and the NS mbarriers.
struct AdjLayout {
  uint32_t ext, rec_cap, halo_cap;
  uint32_t off_un, off_tS, off_g0, off_g1, off_g2, off_hidx;
  uint32_t stage;
  uint32_t off_rho, off_harea, off_list, off_slots, off_bars, total;
};

inline AdjLayout make_adj_layout(uint32_t w, uint32_t geo_arrays, uint32_t tc, uint32_t ns,
                                 uint32_t rec_cap, uint32_t halo_cap) {
  auto a16 = [](uint32_t x) { return (x + 15u) & ~15u; };
  AdjLayout L{};
  L.rec_cap = rec_cap;
  L.halo_cap = halo_cap;
  L.ext = tc + halo_cap;
  uint32_t o = 0;
  L.off_un = o; o += a16(L.ext * 4 * w);
  if (w == 4) {  // FP32: interleaved 16-byte records
    L.off_tS = o; o += a16(rec_cap * 16);
    L.off_g0 = L.off_g1 = L.off_g2 = o;
  } else {
    L.off_tS = o; o += a16(rec_cap * 4);
    L.off_g0 = o; o += a16(rec_cap * w);
    L.off_g1 = o; o += a16(rec_cap * w);
    L.off_g2 = o; o += geo_arrays > 2 ? a16(rec_cap * w) : 0u;
  }
  L.off_hidx = o; o += a16(halo_cap * 4);
  L.stage = o;
  o = ns * L.stage;
  L.off_rho = o; o += a16(L.ext * 4 * w);
  L.off_harea = o; o += a16(halo_cap * w);
  L.off_list = o; o += w == 8 ? a16(rec_cap * 2) : 0u;
  L.off_slots = o; o += a16(3 * (tc + kSlotPad) * 4 * w);
  L.off_bars = o; o += a16(ns * 8);
  L.total = o;
  return L;
}

// Transposed friction of the last step, where the sweep starts: lambda of
// U^{n+1} (u1) becomes mu in place (n cells), and dgn2 gets its first part.
template <typename Real>
__global__ void __launch_bounds__(256)
    k_adjoint_start(const Real* u1, Real* lam, const Real* gn2, Real* dgn2, Real dt, Num num,
                    int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const V4<Real> c = ld4(u1 + 4 * i), l = ld4(lam + 4 * i);
    Real mh, mx, my, b;
    const Real r1 = sizeof(Real) == 8 && Ops<Real>::wet(c.x, num) ? Ops<Real>::rcp(c.x) : Real(0);
    cell_vjp(c.x, c.y, c.z, r1, l.x, l.y, l.z, gn2[i], dt, num, mh, mx, my, b);
    st4(lam + 4 * i, mh, mx, my, l.w);
    dgn2[i] = b;
  }
}

// Tiled adjoint of one step over the same tiles and records as k_tiled_step
// (interleaved tile walk, NS-stage TMA pipeline with the halo gathered by
// cp.async), on its own chunk table. Per tile:
//   (A) rho of every tile and halo cell in shared memory, and the staged
//       cells (h, hu, hv, z) turned into (h, u, v, z) in place; mu of the
//       thread's own cells stays in registers;
//   (B) the vector-Jacobian product of every face record into the slots of
//       the tile's cells (a face shared with another tile gives only this
//       tile's side, as in the forward);
//   (C) each cell: dL/dU^n = mu + its three slots in face order, the z parts
//       added to the running dL/dz; then the transposed friction of step
//       n - 1, whose part of dL/d(g n^2) is accumulated.
// (A) of the next tile runs right after (C), so two block barriers per tile.
//
// Parts (FP64): whole tiles of a small mesh leave SMs idle (40 tiles on 152
// SMs), so a unit of work is one of `split` parts of a tile: the block stages
// the whole tile and forms rho of all of it (cheap), lists the records that
// touch a cell of its part while it does so, and goes through those records
// and its part's cells only. Faces between two parts are computed twice.
// adjoint_split chooses.
//
// Measured per adjoint step (checkpoints at every step, 64 gauges; before:
// lambda and U^{n+1} read by every step, friction redone for halo cells,
// FP64 velocities per face, gauges by one thread at the end): FP32 1.0M cells
// 54.3 -> 29.3 us, 160,000 cells 28.0 -> 11.3, 10,000 cells 12.2 -> 8.7; FP64
// (16 gauges) 79,806 cells 153 -> 82, 10,000 cells 58 -> 25. FP64 is bound by
// the FP64 pipe, and by tiles not dividing over the SMs on small meshes; FP32
// by instruction issue and the two barriers per tile.
//
// Registers are capped so that 640 FP32 threads (5 blocks of 128 with
// 256-cell tiles, which their shared memory also allows) share an SM.
template <typename Real, int NT>
constexpr int adjoint_min_blocks() { return (sizeof(Real) == 4 ? 640 : 256) / NT; }

template <typename Real, int NT, int NS, int CPT, bool Parts = false>
__global__ void __launch_bounds__(NT, adjoint_min_blocks<Real, NT>())
    k_tiled_adjoint(DevMesh<Real> m, AdjArgs<Real> A, Num num, AdjLayout L) {
  constexpr int TC = NT * CPT;
  constexpr bool kF64 = sizeof(Real) == 8;  // velocities per cell, 1 / area from the mesh
  __shared__ int s_nrec[NS], s_nh[NS];
  extern __shared__ __align__(128) unsigned char smem[];
  Real* rho = reinterpret_cast<Real*>(smem + L.off_rho);      // [ext][4]
  Real* harea = reinterpret_cast<Real*>(smem + L.off_harea);  // [halo_cap]
  Real* slots = reinterpret_cast<Real*>(smem + L.off_slots);  // [3 (TC + kSlotPad)][4]
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + L.off_bars);
  const Real* __restrict__ area = kF64 ? m.rarea : m.area;

  const Chunk ch = m.chunks[blockIdx.x];
  // units (tiles, or parts of tiles) ch.tile0 + k ch.stride
  const int n_tiles = ch.ntiles, split = Parts ? A.split : 1;
  auto unit = [&](int k) { return ch.tile0 + k * ch.stride; };
  auto tile_of = [&](int k) { return Parts ? unit(k) / split : unit(k); };
  // cells [lo, hi) of the tile belong to unit k's part, whole warps of them
  auto part_of = [&](int k, int& lo, int& hi) {
    const int p = unit(k) % split;
    lo = (TC / 32 * p / split) * 32;
    hi = (TC / 32 * (p + 1) / split) * 32;
  };
  uint16_t* list = reinterpret_cast<uint16_t*>(smem + L.off_list);
  __shared__ int s_list[2];  // records listed for units k, k + 1
  const int cell_end = ch.cell_end;
  const Real dt = A.dt;
  const int tid = threadIdx.x;

  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < NS; ++i) mbar_init(&bar[i], 1);
    fence_mbar_init();
    s_list[0] = s_list[1] = 0;
  }
  __syncthreads();

  uint32_t parity_bits = 0, pending = 0;
  auto issue = [&](int st, int t) {
    unsigned char* p = smem + st * L.stage;
    const int64_t base = (int64_t)t * TC;
    const int64_t r0 = m.toff[t], h0 = m.hoff[t];
    const uint32_t nrec = (uint32_t)(m.toff[t + 1] - r0);
    const uint32_t nh = (uint32_t)(m.hoff[t + 1] - h0);
    const uint32_t cells = TC * 4 * (uint32_t)sizeof(Real);
    s_nrec[st] = (int)nrec;
    s_nh[st] = (int)nh;
    const uint32_t rb = nrec * (uint32_t)sizeof(Real);
    fence_proxy_async();
    mbar_expect_tx(&bar[st], cells + nrec * rec_bytes<Real>() + nh * 4);
    bulk_g2s(p + L.off_un, A.un + 4 * base, cells, &bar[st]);
    if constexpr (sizeof(Real) == 4) {
      bulk_g2s(p + L.off_tS, m.trec + r0, nrec * 16, &bar[st]);
    } else {
      bulk_g2s(p + L.off_tS, m.tS + r0, nrec * 4, &bar[st]);
      bulk_g2s(p + L.off_g0, m.tg0 + r0, rb, &bar[st]);
      bulk_g2s(p + L.off_g1, m.tg1 + r0, rb, &bar[st]);
      bulk_g2s(p + L.off_g2, m.tg2 + r0, rb, &bar[st]);
    }
    if (nh > 0) bulk_g2s(p + L.off_hidx, m.hidx + h0, nh * 4, &bar[st]);
    pending |= 1u << st;
  };
  auto wait_stage = [&](int st) -> bool {
    const bool ok = mbar_wait(&bar[st], (parity_bits >> st) & 1u, num.wait_rounds);
    if (ok) {
      parity_bits ^= 1u << st;
      pending &= ~(1u << st);
    }
    return ok;
  };
  // halo cells of stage st: U^n into the stage, mu and area into the block's
  // single rho and area arrays (free once the previous tile's faces are done)
  auto gather_halo = [&](int st) {
    unsigned char* p = smem + st * L.stage;
    const int32_t* hl = reinterpret_cast<const int32_t*>(p + L.off_hidx);
    Real* dun = reinterpret_cast<Real*>(p + L.off_un) + 4 * TC;
    const int nh = s_nh[st];
    constexpr int kV = 16 / (int)sizeof(Real);  // values per 16-byte copy
    for (int q = tid; q < nh; q += NT) {
      const int64_t c = hl[q];
#pragma unroll
      for (int b = 0; b < 4 / kV; ++b) {
        cp_async16(dun + 4 * q + b * kV, A.un + 4 * c + b * kV);
        cp_async16(rho + 4 * (TC + q) + b * kV, A.mu_in + 4 * c + b * kV);
      }
      cp_async(harea + q, area + c);
    }
  };

  // Per-cell inputs of the thread's own cells for (A), loaded one tile ahead
  // into registers (their latency hides behind the previous tile's face
  // loop): the area (mesh data) and mu (the previous launch's output).
  V4<Real> nmu[CPT];
  Real nar[CPT];
  auto load_area = [&](int t) {
    const int64_t b0 = (int64_t)t * TC;
#pragma unroll
    for (int cc = 0; cc < CPT; ++cc) nar[cc] = area[b0 + tid + cc * NT];
  };
  auto load_mu = [&](int t) {
    const int64_t b0 = (int64_t)t * TC;
#pragma unroll
    for (int cc = 0; cc < CPT; ++cc) nmu[cc] = ld4(A.mu_in + 4 * (b0 + tid + cc * NT));
  };
  auto scale = [&](Real a) { return kF64 ? -(dt * a) : -Ops<Real>::div(dt, a); };
  // (A) of a tile: the thread's own cells from the registers load_area and
  // load_mu filled, and the halo cells this thread gathered (gather_halo's
  // assignment, so no barrier is needed after its own copies land).
  V4<Real> mu[CPT];
  // FP64: 1 / h of a wet cell, else 0, and (hu, hv), which the staged cells
  // lose to their velocities (h u would differ from hu by two roundings)
  Real rh[CPT], mqx[CPT], mqy[CPT];
  auto phase_a = [&](int st, int k) {
    const int tile = tile_of(k);
    if constexpr (Parts) {  // the part's records
      int lo, hi;
      part_of(k, lo, hi);
      const int32_t* codes = reinterpret_cast<const int32_t*>(smem + st * L.stage + L.off_tS);
      const int nrec = s_nrec[st], lane = tid & 31;
      auto mine = [&](int code) {  // a cell of the part (padding and walls are no cells)
        const int j = (-1 - code) & (TC - 1);
        return code < 0 && code != kSideWall && j >= lo && j < hi;
      };
      for (int r0 = tid & ~31; r0 < nrec; r0 += NT) {
        const int r = r0 + lane;
        const int packed = r < nrec ? codes[r] : 0;
        const bool take = r < nrec && (mine(packed >> 16) || mine((int)(int16_t)(packed & 0xffff)));
        const unsigned m = __ballot_sync(0xffffffffu, take);
        int at = 0;
        if (lane == 0 && m) at = atomicAdd(&s_list[k & 1], __popc(m));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (take) list[at + __popc(m & ((1u << lane) - 1u))] = (uint16_t)r;
      }
    }
    Real* sun = reinterpret_cast<Real*>(smem + st * L.stage + L.off_un);
    auto to_velocity = [&](Real* c) -> Real {
      const V4<Real> x = ld4(c);
      const Real r = Ops<Real>::wet(x.x, num) ? Ops<Real>::rcp(x.x) : Real(0);
      st4(c, x.x, x.y * r, x.z * r, x.w);
      return r;
    };
    const int nc = min(TC, cell_end - tile * TC);
#pragma unroll
    for (int cc = 0; cc < CPT; ++cc) {
      const int j = tid + cc * NT;
      mu[cc] = nmu[cc];
      const Real a = j < nc ? scale(nar[cc]) : Real(0);  // padding: area 0
      st4(rho + 4 * j, a * mu[cc].x, a * mu[cc].y, a * mu[cc].z, Real(0));
      if constexpr (kF64) {
        mqx[cc] = sun[4 * j + 1];
        mqy[cc] = sun[4 * j + 2];
        rh[cc] = to_velocity(sun + 4 * j);
      }
    }
    const int nh = s_nh[st];
    for (int q = tid; q < nh; q += NT) {
      const int j = TC + q;
      const V4<Real> c = ld4(rho + 4 * j);
      const Real a = scale(harea[q]);
      st4(rho + 4 * j, a * c.x, a * c.y, a * c.z, Real(0));
      if constexpr (kF64) to_velocity(sun + 4 * j);
    }
  };
  int timeout = 0;
  // Programmatic dependent launch: the first tiles' tape states, records and
  // halo lists and the own cells' areas are fetched while the previous
  // adjoint step finishes; mu and dL/d(g n^2), its output, only after
  // griddepcontrol.wait.
  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < NS - 1; ++i)
      if (i < n_tiles) issue(i, tile_of(i));
  }
  if (n_tiles > 0) load_area(tile_of(0));
  pdl_trigger();
  pdl_wait();
  if (n_tiles > 0) load_mu(tile_of(0));
  if (n_tiles > 0) {
    const bool ok = (tid == 0) ? wait_stage(0) : true;
    if (__syncthreads_or(!ok)) {
      timeout = 1;
    } else {
      gather_halo(0);
      cp_async_wait_all();
      phase_a(0, 0);
      __syncthreads();
    }
  }
  // Each iteration: (B) the faces of tile k, then (C) its cells followed by
  // (A) of tile k+1 (rho is free once every face of tile k is done). Two
  // block barriers per tile.
  for (int k = 0; !timeout && k < n_tiles; ++k) {
    const int st = k % NS;
    const int tile = tile_of(k);
    const bool has_next = k + 1 < n_tiles;
    if (tid == 0 && k + NS - 1 < n_tiles) issue((k + NS - 1) % NS, tile_of(k + NS - 1));
    const unsigned char* p = smem + st * L.stage;
    const Real* sun = reinterpret_cast<const Real*>(p + L.off_un);
    const int32_t* rS = reinterpret_cast<const int32_t*>(p + L.off_tS);
    const Real* rg0 = reinterpret_cast<const Real*>(p + L.off_g0);
    const Real* rg1 = reinterpret_cast<const Real*>(p + L.off_g1);
    const Real* rg2 = reinterpret_cast<const Real*>(p + L.off_g2);
    const int base = tile * TC;
    const int nc = min(TC, cell_end - base);
    const int nrec = s_nrec[st];
    // what (C) and the next (A) need, into registers while the faces run
    // (cell arrays are padded to whole tiles, so the loads are in bounds)
    Real gn2[CPT], dg[CPT];
#pragma unroll
    for (int cc = 0; cc < CPT; ++cc) {
      gn2[cc] = A.gn2[base + tid + cc * NT];
      dg[cc] = A.dgn2[base + tid + cc * NT];
    }
    if (has_next) {
      load_area(tile_of(k + 1));
      load_mu(tile_of(k + 1));
    }
    int g0 = 0, g1 = 0;  // the tile's gauge cells
    if (A.gstep >= 0) {
      g0 = A.gauges.tile_first[tile];
      g1 = A.gauges.tile_first[tile + 1];
    }
    int lo = 0, hi = TC, n_faces = nrec;
    if constexpr (Parts) {
      part_of(k, lo, hi);
      n_faces = s_list[k & 1];
      if (tid == 0) s_list[(k + 1) & 1] = 0;
    }

    // (B) face records
    for (int q = tid; q < n_faces; q += NT) {
      const int r = Parts ? (int)list[q] : q;
      int32_t packed;
      Real nx, ny, len;
      if constexpr (sizeof(Real) == 4) {
        rec_f32(rS, r, packed, nx, ny, len);
      } else {
        packed = rS[r];
        Geo<Real>::get(rg0, rg1, rg2, r, nx, ny, len);
      }
      const int a = packed >> 16;
      if (a == kSideWall) continue;  // padding record
      const int b = (int)(int16_t)(packed & 0xffff);
      Real gA[4], gB[4];
      if (b == kSideWall) {  // wall: side A is the tile cell owning the edge
        const int ia = (-1 - a) & (TC - 1);
        const V4<Real> UA = ld4(sun + 4 * ia);
        const V4<Real> RA = ld4(rho + 4 * ia);
        face_vjp<true>(UA, UA, nx, ny, len, num, RA.x, RA.y, RA.z, Real(0), Real(0), Real(0),
                             gA, gB);
        st4(slots + 4 * slot_pad<TC>(-1 - a), gA[0], gA[1], gA[2], gA[3]);
        continue;
      }
      const int ia = a < 0 ? ((-1 - a) & (TC - 1)) : a;
      const int ib = b < 0 ? ((-1 - b) & (TC - 1)) : b;
      const V4<Real> UA = ld4(sun + 4 * ia);
      const V4<Real> UB = ld4(sun + 4 * ib);
      const V4<Real> RA = ld4(rho + 4 * ia);
      const V4<Real> RB = ld4(rho + 4 * ib);
      face_vjp<false>(UA, UB, nx, ny, len, num, RA.x, RA.y, RA.z, RB.x, RB.y, RB.z, gA, gB);
      if (a < 0) st4(slots + 4 * slot_pad<TC>(-1 - a), gA[0], gA[1], gA[2], gA[3]);
      if (b < 0) st4(slots + 4 * slot_pad<TC>(-1 - b), gB[0], gB[1], gB[2], gB[3]);
    }
    const bool ok = (tid == 0 && has_next) ? wait_stage((k + 1) % NS) : true;
    if (__syncthreads_or(!ok)) {
      timeout = 1;
      break;
    }
    if (has_next) gather_halo((k + 1) % NS);

    // (C) cells
#pragma unroll
    for (int cc = 0; cc < CPT; ++cc) {
      const int j = tid + cc * NT;
      if (j >= nc) break;
      if (Parts && (j < lo || j >= hi)) continue;
      const V4<Real> f0 = ld4(slots + 4 * j);
      const V4<Real> f1 = ld4(slots + 4 * (TC + kSlotPad + j));
      const V4<Real> f2 = ld4(slots + 4 * (2 * (TC + kSlotPad) + j));
      const V4<Real> c = ld4(sun + 4 * j);
      Real lh, lx, ly, qx = c.y, qy = c.z;
      if constexpr (kF64) {  // velocities' derivatives back to (hu, hv)
        const Real su = f0.y + f1.y + f2.y, sv = f0.z + f1.z + f2.z, r = rh[cc];
        lh = mu[cc].x + (f0.x + f1.x + f2.x - r * fma_rn(su, c.y, sv * c.z));
        lx = fma_rn(su, r, mu[cc].y);
        ly = fma_rn(sv, r, mu[cc].z);
        qx = mqx[cc];
        qy = mqy[cc];
      } else {
        lh = mu[cc].x + f0.x + f1.x + f2.x;
        lx = mu[cc].y + f0.y + f1.y + f2.y;
        ly = mu[cc].z + f0.z + f1.z + f2.z;
      }
      const Real lz = mu[cc].w + f0.w + f1.w + f2.w;
      for (int g = g0; g < g1; ++g)
        if (A.gauges.cells[g] == base + j) lh = add_seeds(lh, A.gauges, A.gstep, g);
      if (!A.last) {
        Real b;
        cell_vjp(c.x, qx, qy, kF64 ? rh[cc] : Real(0), lh, lx, ly, gn2[cc], A.dt_prev, num, lh, lx, ly,
                 b);
        A.dgn2[base + j] = dg[cc] + b;
      }
      st4(A.mu_out + 4 * (int64_t)(base + j), lh, lx, ly, lz);
    }
    cp_async_wait_all();
    if (has_next) phase_a((k + 1) % NS, k + 1);
    __syncthreads();
  }
  if (timeout && tid == 0) {
#pragma unroll
    for (int i = 0; i < NS; ++i)
      if ((pending >> i) & 1u) mbar_wait(&bar[i], (parity_bits >> i) & 1u);
    atomicOr(A.err, kErrTimeout);
  }
}

// Adds the gauge seeds of step k to lam, one thread per distinct cell.
template <typename Real>
__global__ void k_inject_gauges(Real* lam, GaugeSeeds g, long long k) {
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < g.ncells; c += gridDim.x * blockDim.x) {
    Real* p = lam + 4 * (int64_t)g.cells[c];
    *p = add_seeds(*p, g, k, c);
  }
}

}  // namespace swe
