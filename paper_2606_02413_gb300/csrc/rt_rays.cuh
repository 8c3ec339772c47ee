// The persistent one-thread-per-bundle ray kernel (step-wise magnification
// with 0, 2, 4 or 8 neighbours; Sec. 2.1 Eqs. 4-12, Sec. 3.2).
//
// Each thread owns one ray bundle at a time: the central ray of a (pixel,
// frequency) and its NB step-wise neighbours.  Per central step i it
//   (a) advances the central ray one RK4 step from node i (Eq. 4), with the
//       stage-1 sample giving n_e and T_e at node i;
//   (b) settles the transfer of segment i-1 -> i (Eq. 2 with Eq. 12, front to
//       back) and the TAU_STOP / STEP_LIMIT terminations;
//   (c) completes step i: chord t^i, transverse basis and eps (Eqs. 5, 6, 8),
//       the new node, and the clip tests against the inner and outer spheres;
//   (d) accumulates ln M^{i+1} (Eqs. 9-11): from the field's second
//       derivatives at the central ray's stage points while the neighbours
//       stay in those points' cells (kCurv, curvature_ln_m), else from a
//       retrace of step i for every neighbour, seeded at r^i +- eps e_j with
//       the central k^i (Eq. 7);
//   (e) on a clipped last step, closes the path at the crossing point.
// This is the order of the paper's per-step description.
//
// Why one thread per bundle.  The per-step bookkeeping (basis, ln M,
// absorption, transfer, termination, compensated updates) is scalar per
// bundle; with the bundle spread over NB + 1 lanes it ran on one lane of
// NB + 1 and took a third of the warp's issue slots.  Here every lane of a
// warp does useful work in every instruction, and a neighbour needs only the
// first three RK4 stages (its separation depends on its end position, which
// does not involve the fourth stage), so a retraced step costs 4 + 3 NB field
// evaluations instead of 4 (NB + 1), and one clear of the faces 4.
//
// Precision (kMixed) and the offset form of the separations are those of
// rt_bundle.cuh: d_j = eps e_j + h^2/12 (G_{+j} - G_{-j}) for a +-e_j pair,
// ln M = log1p(c1.e1 + c2.e2 + t.(c1 x c2)) with c_j = (d_j - eps e_j) / eps.
#pragma once
#include "rt_bundle.cuh"

namespace rt {

// __launch_bounds__ occupancy target (128-thread blocks).  At 4 blocks (16
// warps per SM, up to 128 registers) the step keeps its values in registers
// instead of recomputing or spilling them; the kernel is bound by issue, not
// latency, and 4 measured faster than 6, 5, 3 or 2 (without magnification
// too: 128^2 x 8 maps 11.6 ms, 5 blocks 12.6, 6 blocks 12.9).
#ifndef RT_RAY_MIN_BLOCKS
#define RT_RAY_MIN_BLOCKS 4
#endif
constexpr int kRayMinBlocks = RT_RAY_MIN_BLOCKS;

// The sum G = a1 + a2 + a3 of the first three RK4 stages from (p, k): a
// neighbour's end position is p + h k + h^2/6 G (the fourth stage enters only
// the wave vector).  Rounded operation by operation, so that the forms below
// agree bit for bit.
__device__ __forceinline__ Vec scaled(float kf, const Sample& s) {
  return {__fmul_rn(kf, s.gx), __fmul_rn(kf, s.gy), __fmul_rn(kf, s.gz)};
}
__device__ __forceinline__ Vec sum3(const Vec& a, const Vec& b, const Vec& c) {
  return {__fadd_rn(__fadd_rn(a.x, b.x), c.x), __fadd_rn(__fadd_rn(a.y, b.y), c.y),
          __fadd_rn(__fadd_rn(a.z, b.z), c.z)};
}
// stage 3 at p + h/2 (k + h/2 a1)
__device__ __forceinline__ Vec stage3_force(const GridDev& G, float kf, float hh, const Vec& p, const Vec& k,
                                            const Vec& a1) {
  const float qx = fmaf(hh, a1.x, k.x), qy = fmaf(hh, a1.y, k.y), qz = fmaf(hh, a1.z, k.z);
  return scaled(kf, eval_field_t<false>(G, fmaf(hh, qx, p.x), fmaf(hh, qy, p.y), fmaf(hh, qz, p.z), false));
}
__device__ __forceinline__ Vec rk4_g3(const GridDev& G, float kf, float h, const Vec& p, const Vec& k) {
  const float hh = 0.5f * h;
  // stages 1 and 2 are independent (stage 2 sits at p + h/2 k)
  const Vec a1 = scaled(kf, eval_field_t<false>(G, p.x, p.y, p.z, false));
  const Vec a2 = scaled(kf, eval_field_t<false>(G, fmaf(hh, k.x, p.x), fmaf(hh, k.y, p.y), fmaf(hh, k.z, p.z), false));
  return sum3(a1, a2, stage3_force(G, kf, hh, p, k, a1));
}
// The same by two adjacent lanes, each with the same p and k: the even lane
// takes stage 1 and the odd one stage 2 at the same time.
__device__ __forceinline__ Vec rk4_g3_halves(const GridDev& G, float kf, float h, const Vec& p, const Vec& k) {
  const float hh = 0.5f * h;
  const int lane = threadIdx.x & 31;
  const bool odd = lane & 1;
  const Vec q{odd ? fmaf(hh, k.x, p.x) : p.x, odd ? fmaf(hh, k.y, p.y) : p.y, odd ? fmaf(hh, k.z, p.z) : p.z};
  const Vec a = scaled(kf, eval_field_t<false>(G, q.x, q.y, q.z, false));
  const Vec a1{__shfl_sync(kFull, a.x, lane & ~1), __shfl_sync(kFull, a.y, lane & ~1), __shfl_sync(kFull, a.z, lane & ~1)};
  const Vec a2{__shfl_sync(kFull, a.x, lane | 1), __shfl_sync(kFull, a.y, lane | 1), __shfl_sync(kFull, a.z, lane | 1)};
  return sum3(a1, a2, stage3_force(G, kf, hh, p, k, a1));
}

// One central RK4 step (see Rk4Out) with the stage-1 sample including T_e;
// stages 1 and 2, and then 3 and 4, are independent of each other.  kCurv:
// also the second derivatives at the first two stage points (cv[0], cv[1]),
// which the neighbours' retrace needs, and those points' clearance.  The third
// stage point lies h^2/4 |a_1| from the second (1e-6 R_sun at h = 2e-3), where
// they are the same; d3: that distance squared (step_clear looks at it).
struct StagePoints {
  Curv cv[2];
  float x2, y2, z2, x3, y3, z3, x4, y4, z4;  // stage points 2 to 4
  float d3;
};
template <bool kCurv = false>
__device__ __forceinline__ Rk4Out rk4_central(const GridDev& G, float kf, float h, float px, float py, float pz,
                                              float kx, float ky, float kz, float off_r = 0.f, float off = 0.f,
                                              StagePoints* sp = nullptr) {
  Rk4Out o;
  const float hh = 0.5f * h;
  const float x2 = fmaf(hh, kx, px), y2 = fmaf(hh, ky, py), z2 = fmaf(hh, kz, pz);
  const Sample s1 = eval_field_t<true, kCurv>(G, px, py, pz, true, off_r, off, kCurv ? &sp->cv[0] : nullptr);
  const Sample s2 = eval_field_t<false, kCurv>(G, x2, y2, z2, false, off_r, off, kCurv ? &sp->cv[1] : nullptr);
  o.ne1 = s1.ne;
  o.te1 = s1.te;
  const float a1x = kf * s1.gx, a1y = kf * s1.gy, a1z = kf * s1.gz;
  const float a2x = kf * s2.gx, a2y = kf * s2.gy, a2z = kf * s2.gz;
  o.Gx = a1x; o.Gy = a1y; o.Gz = a1z;
  o.Ax = a1x; o.Ay = a1y; o.Az = a1z;
  o.Gx += a2x; o.Gy += a2y; o.Gz += a2z;
  o.Ax = fmaf(2.f, a2x, o.Ax); o.Ay = fmaf(2.f, a2y, o.Ay); o.Az = fmaf(2.f, a2z, o.Az);
  // stage 3 at p + h/2 (k + h/2 a1), stage 4 at p + h (k + h/2 a2)
  const float qx = fmaf(hh, a1x, kx), qy = fmaf(hh, a1y, ky), qz = fmaf(hh, a1z, kz);
  const float q3x = fmaf(hh, a2x, kx), q3y = fmaf(hh, a2y, ky), q3z = fmaf(hh, a2z, kz);
  const float x3 = fmaf(hh, qx, px), y3 = fmaf(hh, qy, py), z3 = fmaf(hh, qz, pz);
  const Sample s3 = eval_field_t<false>(G, x3, y3, z3, false);
  const float x4 = fmaf(h, q3x, px), y4 = fmaf(h, q3y, py), z4 = fmaf(h, q3z, pz);
  const Sample s4 = eval_field_t<false>(G, x4, y4, z4, false);
  const float a3x = kf * s3.gx, a3y = kf * s3.gy, a3z = kf * s3.gz;
  o.Gx += a3x; o.Gy += a3y; o.Gz += a3z;
  o.Ax = fmaf(2.f, a3x, o.Ax); o.Ay = fmaf(2.f, a3y, o.Ay); o.Az = fmaf(2.f, a3z, o.Az);
  o.Ax = fmaf(kf, s4.gx, o.Ax); o.Ay = fmaf(kf, s4.gy, o.Ay); o.Az = fmaf(kf, s4.gz, o.Az);
  if (sp) {
    sp->x2 = x2; sp->y2 = y2; sp->z2 = z2;
    sp->x3 = x3; sp->y3 = y3; sp->z3 = z3;
    sp->x4 = x4; sp->y4 = y4; sp->z4 = z4;
    const float dx = x3 - x2, dy = y3 - y2, dz = z3 - z2;
    sp->d3 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
  }
  return o;
}

// How far a step's neighbours reach radially: they sit eps off the path
// across the chord, so eps sin(angle of the ray to the radius), where the wave
// vector at the node stands for the chord.  `pad` (of eps, in Clear) covers
// what that leaves out: the chord's turn and the third stage's shift, which
// step_clear bounds, the radius's turn over half a step and the second order
// eps^2 / 2r.
__device__ __forceinline__ float radial_reach(const Clear& c, float px, float py, float pz, float kx, float ky, float kz) {
  const float pk = fmaf(px, kx, fmaf(py, ky, pz * kz));
  const float pp = fmaf(px, px, fmaf(py, py, pz * pz)), kk = fmaf(kx, kx, fmaf(ky, ky, kz * kz));
  const float c2 = __fdividef(pk * pk, pp * kk);
  return c.reach * (__fsqrt_rn(fmaxf(1.f - c2, 0.f)) + c.pad);
}

// Trace of the field's Hessian across the direction t at the point (x, y, z):
// sum_j e_j.H e_j over a transverse basis = tr H - t.H t.  f: t in the
// spherical frame there.
__device__ __forceinline__ float transverse_trace(const Curv& c, float x, float y, float z, const Vec& t, Vec& f) {
  const float xt = fmaf(x, t.x, y * t.y);
  f.x = fmaf(z, t.z, xt) * c.inv_r;
  f.y = fmaf(z * c.inv_rho, xt, -c.rho * t.z) * c.inv_r;
  f.z = fmaf(x, t.y, -y * t.x) * c.inv_rho;
  const float cross = fmaf(f.x, fmaf(f.y, c.hrt, f.z * c.hrp), f.y * f.z * c.htp);
  return fmaf(-2.f, cross, fmaf(c.htt, fmaf(-f.y, f.y, 1.f), c.hpp * fmaf(-f.z, f.z, 1.f)));
}

// "+" seed offset of neighbour pair j from the node: eps e1, eps e2, and (8
// neighbours) eps (e1 + e2)/sqrt2, eps (e2 - e1)/sqrt2; the "-" member of the
// pair sits at minus that offset.  a = eps e1, b = eps e2.
__device__ __forceinline__ Vec pair_offset(int j, const Vec& a, const Vec& b) {
  const float s2 = 0.70710678118654752f;
  if (j == 0) return a;
  if (j == 1) return b;
  if (j == 2) return {s2 * (a.x + b.x), s2 * (a.y + b.y), s2 * (a.z + b.z)};
  return {s2 * (b.x - a.x), s2 * (b.y - a.y), s2 * (b.z - a.z)};
}

// Completes a central RK4 step from node (p, k) (Eq. 4 in increment form):
// the chord dr = h (k + kl) + h^2/6 G, dk = h/6 A, and the next node
// (rn, kn).  kMixed carries the rounding of both updates in (rl, kl)
// (Fast2Sum); the plain form leaves them at zero.  The forward kernel and the
// adjoint's recomputation share it, so both follow the same path.
__device__ __forceinline__ Vec chord(float h, float h2_6, const Rk4Out& o, float kx, float ky, float kz, float klx,
                                     float kly, float klz) {
  return {fmaf(h, kx + klx, h2_6 * o.Gx), fmaf(h, ky + kly, h2_6 * o.Gy), fmaf(h, kz + klz, h2_6 * o.Gz)};
}
template <bool kMixed>
__device__ __forceinline__ void complete_step(float h_6, const Rk4Out& o, const Vec& dr, float px, float py, float pz,
                                              float kx, float ky, float kz, float& rlx, float& rly, float& rlz,
                                              float& klx, float& kly, float& klz, Vec& rn, Vec& kn) {
  const Vec dk{h_6 * o.Ax, h_6 * o.Ay, h_6 * o.Az};
  if (kMixed) {
    fast_two_sum(px, dr.x + rlx, rn.x, rlx);
    fast_two_sum(py, dr.y + rly, rn.y, rly);
    fast_two_sum(pz, dr.z + rlz, rn.z, rlz);
    fast_two_sum(kx, dk.x + klx, kn.x, klx);
    fast_two_sum(ky, dk.y + kly, kn.y, kly);
    fast_two_sum(kz, dk.z + klz, kn.z, klz);
  } else {
    rn = {px + dr.x, py + dr.y, pz + dr.z};
    kn = {kx + dk.x, ky + dk.y, kz + dk.z};
  }
}

// The step-wise retrace of one central step (Eqs. 5-11): chord direction t,
// transverse basis (e1, e2), eps, the scaled separations c1, c2 of the
// +-e1, +-e2 pairs (2 neighbours: one-sided against the central G0), and
// ln M.  With 8 neighbours the 45-degree pairs give a second estimate and M
// is the mean of the two.
struct Retrace {
  Vec t, e1, e2, c1, c2;
  float eps, lm;
};

// Chord direction, transverse basis and eps of a step (Eqs. 5, 6, 8).
__device__ __forceinline__ void chord_frame(Retrace& R, float eta, float eps_fixed, const Vec& dr) {
  const float d2n = dot3(dr, dr);
  const float ids = rsqrtf(d2n);
  R.t = {dr.x * ids, dr.y * ids, dr.z * ids};
  basis(R.t, R.e1, R.e2);
  R.eps = (eps_fixed > 0.f) ? eps_fixed : eta * (d2n * ids);
}

// Whether the step's neighbours stay in the cells of the stage points: these
// are clear of the faces by reach (and radial_reach of it), no offset is
// longer than that, the third stage lies near the second, and the chord has
// turned little from the wave vector (by about h^2/2 |a| / |dr|, twice the third
// stage's distance over the chord): Clear's limits on that distance.
__device__ __forceinline__ bool step_clear(const Clear& c, const StagePoints& sp, const Retrace& R, const Vec& dr) {
  // all at once, no short circuit (97x61 x 3 maps with 8 neighbours: 8.0 ms, with && 8.3)
  return sp.cv[0].clear & sp.cv[1].clear & (sp.d3 <= fminf(c.d3, c.d3_chord * dot3(dr, dr))) & (R.eps <= c.reach);
}

// c1, c2 and ln M from the raw separations D (NB >= 4: D_j = G_{+j} - G_{-j}
// over the +-pair j; NB == 2: D_j = G_j).
template <int NB>
__device__ __forceinline__ void finish_retrace(Retrace& R, const Vec* D, float h2_6, float h2_12, const Vec& G0) {
  constexpr int NP = (NB >= 4) ? NB / 2 : 2;
  if (NB == 2) {  // one-sided: d_j = eps e_j + h^2/6 (G_j - G_0)
    const float sc = h2_6 / R.eps;
    R.c1 = {sc * (D[0].x - G0.x), sc * (D[0].y - G0.y), sc * (D[0].z - G0.z)};
    R.c2 = {sc * (D[1].x - G0.x), sc * (D[1].y - G0.y), sc * (D[1].z - G0.z)};
  } else {        // central difference: d = eps e + h^2/12 (G_+ - G_-)
    const float sc = h2_12 / R.eps;
    R.c1 = {sc * D[0].x, sc * D[0].y, sc * D[0].z};
    R.c2 = {sc * D[1].x, sc * D[1].y, sc * D[1].z};
  }
  const float m = tube_m1(R.c1, R.c2, R.e1, R.e2, R.t);
  R.lm = log1p_small(m);
  if (NB == 8) {
    const float s2 = 0.70710678118654752f, sc = h2_12 / R.eps;
    const Vec g1{s2 * (R.e1.x + R.e2.x), s2 * (R.e1.y + R.e2.y), s2 * (R.e1.z + R.e2.z)};
    const Vec g2{s2 * (R.e2.x - R.e1.x), s2 * (R.e2.y - R.e1.y), s2 * (R.e2.z - R.e1.z)};
    const Vec c3{sc * D[2 % NP].x, sc * D[2 % NP].y, sc * D[2 % NP].z};
    const Vec c4{sc * D[3 % NP].x, sc * D[3 % NP].y, sc * D[3 % NP].z};
    // M = (M_e + M_g) / 2, taken before the logarithm: the mean of two
    // logarithms' exponentials would round ln M (~1e-7 a step) at ln 2's ulp
    const float m2 = tube_m1(c3, c4, g1, g2, R.t);
    R.lm = (m > -1.f && m2 > -1.f) ? log1p_small(0.5f * (m + m2))
                                   : __logf(0.5f * (fabsf(1.f + m) + fabsf(1.f + m2)));
  }
}

template <int NB>
__device__ __forceinline__ Retrace retrace_step(const GridDev& G, float kf, float h, float h2_6, float h2_12,
                                                float eta, float eps_fixed, float px, float py, float pz, float kx,
                                                float ky, float kz, const Vec& dr, const Vec& G0) {
  Retrace R;
  chord_frame(R, eta, eps_fixed, dr);
  const Vec sa{R.eps * R.e1.x, R.eps * R.e1.y, R.eps * R.e1.z}, sb{R.eps * R.e2.x, R.eps * R.e2.y, R.eps * R.e2.z};
  // neighbour q is the "+" (even q) or "-" (odd q) member of pair q / 2.
  // One retrace per loop trip keeps the code small.
  constexpr int NP = (NB >= 4) ? NB / 2 : 2;
  Vec D[NP];
#pragma unroll
  for (int m = 0; m < NP; ++m) D[m] = {0.f, 0.f, 0.f};
#pragma unroll 1
  for (int q = 0; q < NB; ++q) {
    const int j = (NB >= 4) ? (q >> 1) : q;
    const float sgn = (NB >= 4 && (q & 1)) ? -1.f : 1.f;
    const Vec off = (NB >= 4) ? pair_offset(j, sa, sb) : ((j == 0) ? sa : sb);
    const Vec g = rk4_g3(G, kf, h, Vec{fmaf(sgn, off.x, px), fmaf(sgn, off.y, py), fmaf(sgn, off.z, pz)},
                         Vec{kx, ky, kz});
#pragma unroll
    for (int m = 0; m < NP; ++m)
      if (m == j) D[m] = {fmaf(sgn, g.x, D[m].x), fmaf(sgn, g.y, D[m].y), fmaf(sgn, g.z, D[m].z)};
  }
  finish_retrace<NB>(R, D, h2_6, h2_12, G0);
  return R;
}

// ln M of a step whose neighbours all stay in the cells of the central ray's
// own stage points.  There a +-pair's separation is, to its third order in
// eps, the Hessian's: G_+ - G_- = 2 eps kf sum_s H(P_s) e over the three
// stage points P_s of the central ray, so with C = h^2/6 kf sum_s H(P_s)
//   ln M = tr_t C - tr_t C^2 / 2 + (tr C^2 - |C t|^2) / 6 + O(C^3),
// tr_t the trace across t; the last term is the third stage's own shift by
// h^2/4 a_1.  The same for 4 and for 8 neighbours and for any eps: no
// neighbour is evaluated.  The second order (formed at the middle stage
// point) is skipped where |C| <= 1e-5: it is below 1e-10 there; c2 = |C|^2: a
// step with |C| > 1e-3 retraces its neighbours.
// Why: the neighbours' 12 (24) of a step's 16 (28) field evaluations were
// three quarters of the kernel's instructions, and it is bound by issue.
// A few second derivatives at two points whose cell and fractions the central
// ray has anyway cost less than one evaluation.  One GB300, 4 neighbours, global
// corona 128^2 x 16 frequencies: 660 ms -> 332 ms; 64^2 x 1 on a 64x32x64
// corona 14.3 -> 7.9 ms; 8 neighbours, 97x61 x 3: 37.5 -> 11.6 ms (300, 5.5 and
// 7.7 ms with the steps that came after).  Paths, optical depths and step
// counts are bit-identical to the retraced form's; ln S differs by 5.6e-8 (rms)
// on the global corona.
__device__ __forceinline__ float curvature_ln_m(const StagePoints& sp, float px, float py, float pz, const Vec& t,
                                                float h2_6kf, float& c2) {
  Vec f1, f2;
  const float q2 = transverse_trace(sp.cv[1], sp.x2, sp.y2, sp.z2, t, f2);
  const float q = fmaf(2.f, q2, transverse_trace(sp.cv[0], px, py, pz, t, f1));  // the third stage is the second
  const Curv& c = sp.cv[1];
  const float off = fmaf(c.hrt, c.hrt, fmaf(c.hrp, c.hrp, c.htp * c.htp));
  const float h2 = fmaf(2.f, off, fmaf(c.htt, c.htt, c.hpp * c.hpp));  // tr H^2
  const float s2 = 9.f * h2_6kf * h2_6kf;                              // C = 3 h^2/6 kf H there
  c2 = s2 * h2;
  float lm = h2_6kf * q;
  if (c2 > 1e-10f) {
    const float gr = fmaf(c.hrt, f2.y, c.hrp * f2.z), gt = fmaf(c.hrt, f2.x, fmaf(c.htt, f2.y, c.htp * f2.z)),
                gp = fmaf(c.hrp, f2.x, fmaf(c.htp, f2.y, c.hpp * f2.z));
    const float g2 = fmaf(gr, gr, fmaf(gt, gt, gp * gp));              // |H t|^2
    const float th = c.htt + c.hpp - q2;                               // t.H t
    lm = fmaf(s2, fmaf(1.f / 6.f, h2 - g2, -0.5f * fmaf(th, th, fmaf(-2.f, g2, h2))), lm);
  }
  return lm;
}

// The neighbours of a step that comes too near a face (about one step in
// ten on a 64x32x64 corona at h = 2e-3, one in twenty on the global one) are
// retraced; almost every warp has such a lane, so a branch per lane would pay
// for all of them.  A warp's lanes retrace together the neighbours of the lanes
// that ask for it (slow): NB lanes per asking lane, one neighbour each, 32 / NB
// asking lanes at a time; while at most half of those ask, two lanes per
// neighbour, which take its first two stages at once (global corona 128^2 x 16:
// 314 -> 300 ms, 40 small requests 27.1 -> 25.7 ms).  The arithmetic of each is
// retrace_step's.  Every lane of the warp calls it; R.t, e1, e2, eps hold the
// asking lane's frame, and its ln M comes back in R.lm.  Measured and not kept:
// lanes that wait until a pass fills (rays that run along a face ask at every
// step and stall: 332 -> 362 ms), and differences at the stages near a face
// only (3% faster, but points formed in another order move ln S of single rays
// by up to 1e-3).
template <int NB>
struct RetraceSlot {
  float v[(NB == 8) ? 16 : 13];  // p, k, eps e1, eps e2, kf; then D_1 ... D_{NB/2}
};
template <int NB>
__device__ __forceinline__ void retrace_shared(const GridDev& G, RetraceSlot<NB>* slots, bool slow, float kf, float h,
                                               float h2_6, float h2_12, float px, float py, float pz, float kx,
                                               float ky, float kz, Retrace& R) {
  constexpr int PER = 32 / NB;
  const int lane = threadIdx.x & 31;
  unsigned todo = __ballot_sync(kFull, slow);
  while (todo) {
    const int rank = __popc(todo & ((1u << lane) - 1u));
    const bool mine = slow && rank < PER;
    if (mine) {
      float* v = slots[rank].v;
      v[0] = px; v[1] = py; v[2] = pz;
      v[3] = kx; v[4] = ky; v[5] = kz;
      v[6] = R.eps * R.e1.x; v[7] = R.eps * R.e1.y; v[8] = R.eps * R.e1.z;
      v[9] = R.eps * R.e2.x; v[10] = R.eps * R.e2.y; v[11] = R.eps * R.e2.z;
      v[12] = kf;
    }
    __syncwarp();
    // with few asking lanes each neighbour has two, a stage each
    const int asking = min(__popc(todo), PER);
    const bool two = asking <= PER / 2;
    const int n = two ? lane >> 1 : lane, q = n % NB, group = n / NB;
    // groups past the last asking lane repeat it (the lookups stay in bounds, nothing is written)
    float* v = slots[min(group, asking - 1)].v;
    const float sgn = (q & 1) ? -1.f : 1.f;
    const Vec off = pair_offset(q >> 1, Vec{v[6], v[7], v[8]}, Vec{v[9], v[10], v[11]});
    const Vec p{fmaf(sgn, off.x, v[0]), fmaf(sgn, off.y, v[1]), fmaf(sgn, off.z, v[2])}, k{v[3], v[4], v[5]};
    const float kfq = v[12];
    const Vec g = two ? rk4_g3_halves(G, kfq, h, p, k) : rk4_g3(G, kfq, h, p, k);
    const int step = two ? 2 : 1;
    const Vec d{g.x - __shfl_down_sync(kFull, g.x, step), g.y - __shfl_down_sync(kFull, g.y, step),
                g.z - __shfl_down_sync(kFull, g.z, step)};
    __syncwarp();
    if (group < asking && !(q & 1) && !(two && (lane & 1))) {
      float* w = v + 3 * (q >> 1);
      w[0] = d.x; w[1] = d.y; w[2] = d.z;
    }
    __syncwarp();
    if (mine) {
      Vec D[NB / 2];
#pragma unroll
      for (int m = 0; m < NB / 2; ++m)
        D[m] = {slots[rank].v[3 * m], slots[rank].v[3 * m + 1], slots[rank].v[3 * m + 2]};
      finish_retrace<NB>(R, D, h2_6, h2_12, Vec{0.f, 0.f, 0.f});
      slow = false;
    }
    __syncwarp();  // the slots are read: the next lanes may fill them
    todo = __ballot_sync(kFull, slow);
  }
}

template <int NB, bool kMixed, bool kCurv>
__global__ void __launch_bounds__(kThreads, kRayMinBlocks) trace_rays(const __grid_constant__ TraceParams P) {
  const int lane = threadIdx.x & 31;
  const float h = P.h;

  // per-ray state; what is touched only when a ray starts or ends lives in
  // shared memory (it would otherwise hold registers through every step)
  struct Cold {
    float* out;
    RayDiag* dg;
    unsigned long long steps_done, rays_done;
    unsigned int item;
    int ck_last;  // tape: the ray's last checkpoint slot (-1: none)
  };
  __shared__ Cold cold[kThreads];
  static_assert(!kCurv || NB >= 4, "the Hessian form stands for +-pairs");
  constexpr int kSlots = kCurv ? 32 / (NB > 0 ? NB : 1) : 1;
  __shared__ RetraceSlot<(NB > 0 ? NB : 4)> slots[kThreads / 32][kSlots];
  Cold& C = cold[threadIdx.x];
  C.out = nullptr;
  C.dg = nullptr;
  C.steps_done = 0;
  C.rays_done = 0;
  C.item = 0;
  C.ck_last = -1;
  int step = 0;
  bool active = false, exhausted = lane >= P.lanes;
  float px = 0.f, py = 0.f, pz = 0.f, kx = 0.f, ky = 0.f, kz = 0.f;
  float rlx = 0.f, rly = 0.f, rlz = 0.f, klx = 0.f, kly = 0.f, klz = 0.f;  // compensation (kMixed)
  float kf = 0.f, kap_c = 0.f, ln_f = 0.f;
  float tau_hi = 0.f, tau_lo = 0.f, lns_hi = 0.f, lns_lo = 0.f, tb_hi = 0.f, tb_lo = 0.f;
  float kap_prev = 0.f, te_prev = 0.f;

  auto finish = [&](int st, float ex, float ey, float ez) {
    *C.out = tb_hi + tb_lo;
    RayDiag* dg = C.dg;
    if (dg) {
      RayDiag d;
      d.exit_pos[0] = ex; d.exit_pos[1] = ey; d.exit_pos[2] = ez;
      d.tau = tau_hi + tau_lo;
      d.ln_s = lns_hi + lns_lo;
      d.steps = step;
      d.status = st;
      *dg = d;
    }
    if (P.ck_last) P.ck_last[C.item] = C.ck_last;
    C.steps_done += (unsigned long long)step;
    C.rays_done += 1;
    active = false;
  };

  // One central step of this thread's bundle.  Every lane of the warp runs
  // it while any lane holds a ray: a lane without one (only when the ticket
  // pool is exhausted) computes on its stale state, whose lookups stay in
  // bounds, and writes nothing.  Keeping the evaluations out of divergent
  // branches lets warp-uniform values (grid and step parameters) live in
  // uniform registers.
  auto step_once = [&]() {
    // ---------------------------------------------- (a) central RK4 step
    StagePoints sp;
    const float off_r = kCurv ? radial_reach(P.clear, px, py, pz, kx, ky, kz) : 0.f;
    const Rk4Out o = rk4_central<kCurv>(P.G, kf, h, px, py, pz, kx, ky, kz, off_r, P.clear.reach, &sp);
    const Vec dr = chord(h, P.h2_6, o, kx, ky, kz, klx, kly, klz);

    // ---------------------------------------------- (d) ln M of step `step`
    float lm = 0.f;
    if constexpr (kCurv) {
      Retrace R;
      chord_frame(R, P.eta, P.eps_fixed, dr);
      float c2;
      R.lm = curvature_ln_m(sp, px, py, pz, R.t, P.h2_6 * kf, c2);
      const bool fast = step_clear(P.clear, sp, R, dr) && c2 <= 1e-6f;
      retrace_shared<NB>(P.G, slots[threadIdx.x >> 5], active && !fast, kf, h, P.h2_6, P.h2_12, px, py, pz, kx, ky, kz,
                         R);
      lm = R.lm;
    } else if (NB > 0) {
      lm = retrace_step<(NB > 0 ? NB : 4)>(P.G, kf, h, P.h2_6, P.h2_12, P.eta, P.eps_fixed, px, py, pz, kx, ky, kz, dr,
                                           Vec{o.Gx, o.Gy, o.Gz}).lm;
    }
    if (!active) return;

    // ---------------------------------------------- (b) segment step-1 -> step
    const float kap = P.emission ? kappa_vac(o.ne1, o.te1, kap_c, ln_f) : 0.f;
    if (step >= 1) {
      const float dt = 0.5f * (kap_prev + kap) * P.hrsun;
      const float tbar = 0.5f * (te_prev + o.te1);
      const float tau0 = tau_hi + tau_lo;
      acc_add<kMixed>(tb_hi, tb_lo, tbar * one_minus_exp_neg(dt) * __expf((lns_hi + lns_lo) - tau0));
      acc_add<kMixed>(tau_hi, tau_lo, dt);
      int stop = 0;  // TAU_STOP or STEP_LIMIT: the path ends at node `step`
      if (P.tau_stop > 0.f && tau_hi + tau_lo >= P.tau_stop) stop = kTauStop;
      else if (step >= P.max_steps) stop = kStepLimit;
      if (stop != 0) {
        finish(stop, px, py, pz);
        return;
      }
    }
    if (P.ckpt && (step % kCkptEvery) == 0) {
      // state at node `step` for the adjoint's recomputation: in the ray's
      // own slots, or (a tape) in the next pool slot, linked to its previous
      unsigned long long slot;
      bool ok;
      if (P.ck_prev) {
        slot = atomicAdd(P.pool_counter, 1ull);
        ok = slot < P.pool_cap;  // an overflowing tape is detected from the counter
      } else {
        const unsigned int item = C.item;
        slot = P.ck_off[item] + (unsigned long long)(step / kCkptEvery);
        ok = slot < P.ck_off[item + 1];
      }
      if (ok) {
        Ckpt& c = P.ckpt[slot];
        c.r[0] = px; c.r[1] = py; c.r[2] = pz;
        c.k[0] = kx; c.k[1] = ky; c.k[2] = kz;
        c.rl[0] = rlx; c.rl[1] = rly; c.rl[2] = rlz;
        c.kl[0] = klx; c.kl[1] = kly; c.kl[2] = klz;
        c.tau_hi = tau_hi; c.tau_lo = tau_lo;
        c.lns_hi = lns_hi; c.lns_lo = lns_lo;
        c.step = step;
        if (P.ck_prev) {
          P.ck_prev[slot] = C.ck_last;
          C.ck_last = (int)slot;
        }
      }
    }

    // ---------------------------------------------- (c) complete step `step`
    Vec rn, kn;
    complete_step<kMixed>(P.h_6, o, dr, px, py, pz, kx, ky, kz, rlx, rly, rlz, klx, kly, klz, rn, kn);
    kap_prev = kap;
    te_prev = o.te1;
    const float rr2 = dot3(rn, rn);
    int term = 0;  // 0: carry on; else the status of a last step
    if (rr2 < P.G.r_min * P.G.r_min) term = kHitInner;
    else if (rr2 > P.G.r_max * P.G.r_max && dot3(rn, kn) > 0.f) term = kExitOuter;
    else if (!isfinite(rr2 + kn.x + kn.y + kn.z)) term = kNan;
    if (NB > 0 && term != kNan) acc_add<kMixed>(lns_hi, lns_lo, lm);

    // ---------------------------------------------- (e) next node, or the end of the path
    step += 1;
    if (term == 0) {
      px = rn.x; py = rn.y; pz = rn.z;
      kx = kn.x; ky = kn.y; kz = kn.z;
    } else if (term == kNan) {
      finish(kNan, rn.x, rn.y, rn.z);
    } else {
      // clipped last segment + boundary term (Eq. 2 front to back); the
      // crossing point closes the path
      const Vec here{px, py, pz};
      const float a = chord_crossing(here, dr, (term == kHitInner) ? P.G.r_min : P.G.r_max, term == kExitOuter);
      const float cx = fmaf(a, dr.x, px), cy = fmaf(a, dr.y, py), cz = fmaf(a, dr.z, pz);
      const Sample s = eval_field_t<true>(P.G, cx, cy, cz, true);
      const float kap_e = P.emission ? kappa_vac(s.ne, s.te, kap_c, ln_f) : 0.f;
      const float dt = 0.5f * (kap_prev + kap_e) * P.hrsun * a;
      const float tbar = 0.5f * (te_prev + s.te);
      const float lns = lns_hi + lns_lo;
      acc_add<kMixed>(tb_hi, tb_lo, tbar * one_minus_exp_neg(dt) * __expf(lns - (tau_hi + tau_lo)));
      acc_add<kMixed>(tau_hi, tau_lo, dt);
      float tbc = 0.f;
      if (term == kHitInner) tbc = (P.tbc_mode == 1) ? P.tbc_K : s.te;
      if (tbc != 0.f) acc_add<kMixed>(tb_hi, tb_lo, tbc * __expf(lns - (tau_hi + tau_lo)));
      finish(term, cx, cy, cz);
    }
  };

  while (true) {
    // ------------------------------------------------------------ refill
    bool need = !active && !exhausted;
    unsigned needmask = __ballot_sync(kFull, need);
    while (needmask) {
      const int leader = __ffs(needmask) - 1;
      unsigned int first = 0;
      if (lane == leader) first = atomicAdd(P.counter, (unsigned)__popc(needmask));
      first = __shfl_sync(kFull, first, leader);
      if (need) {
        const unsigned int item = first + __popc(needmask & ((1u << lane) - 1u));
        if (item >= P.total) {
          exhausted = true;
          need = false;
        } else {
          const RayStart rs = start_ray(P, item);
          C.item = item;
          C.out = rs.out;
          C.dg = rs.dg;
          C.ck_last = -1;
          if (rs.valid) {  // a ragged chunk tail has no ray behind the ticket: take another
            kf = P.straight ? 0.f : rs.F->kf;
            kap_c = rs.F->kap_c;
            ln_f = rs.F->ln_f;
            step = 0;
            tau_hi = tau_lo = lns_hi = lns_lo = tb_hi = tb_lo = 0.f;
            rlx = rly = rlz = klx = kly = klz = 0.f;
            kap_prev = te_prev = 0.f;
            if (!rs.enter) {
              finish(kMiss, rs.px, rs.py, rs.pz);
            } else {
              px = rs.px; py = rs.py; pz = rs.pz;
              kx = rs.kx; ky = rs.ky; kz = rs.kz;
              active = true;
              need = false;
            }
          }
        }
      }
      needmask = __ballot_sync(kFull, need);
    }
    if (!__any_sync(kFull, active)) break;
    step_once();
  }

  // ---- statistics
  unsigned long long steps_done = C.steps_done, rays_done = C.rays_done;
  for (int off = 16; off > 0; off >>= 1) {
    steps_done += __shfl_down_sync(kFull, steps_done, off);
    rays_done += __shfl_down_sync(kFull, rays_done, off);
  }
  if (lane == 0 && P.stats) {
    atomicAdd(P.stats, steps_done);
    atomicAdd(P.stats + 1, rays_done);
  }
}

}  // namespace rt

namespace rt {

// One node of a recorded ray path (rt_path_node).
struct PathNode {
  float r[3];
  float ln_s;     // ln(S / S_0) at the node
  float dlns_ds;  // ln M of the step arriving at the node over its chord length (0 at node 0)
  float tau;      // optical depth from the entry to the node
  float ne, te;   // the interpolated n_e and T_e at the node
};

// Ray-fan diagnostics (Sec. 3.2, Figs. 4 and 6): the rays of the given pixels
// at one frequency, one thread each, stepped exactly as trace_rays steps
// them (the same step code in the same order), recording every node.  A warp
// takes P.lanes rays (as few as fill the schedulers): where one lane retraces
// its neighbours the warp's others wait.  One GB300, 64x32x64 corona, 16, 256
// and 4096 rays with 4 neighbours: 9.5, 10.9 and 23.1 ms with full warps and
// every neighbour retraced, 4.7, 6.2 and 19.9 ms so.
// The first `cap` nodes of ray i go to path[i * cap ...], its node count to
// count[i], and its T_b and diagnostics to tb[i] and diag[i].
constexpr int kPathThreads = 64;
template <int NB, bool kMixed, bool kCurv>
__global__ void __launch_bounds__(kPathThreads)
    trace_paths(const __grid_constant__ TraceParams P, const int* __restrict__ pix, int n, int cap,
                PathNode* __restrict__ path, int* __restrict__ count, float* __restrict__ tb,
                RayDiag* __restrict__ diag) {
  const int lane = threadIdx.x & 31;
  const int i = (blockIdx.x * (kPathThreads / 32) + (threadIdx.x >> 5)) * P.lanes + lane;
  if (lane >= P.lanes || i >= n) return;
  const float h = P.h;
  RayStart rs;
  rs.V = &P.view;
  rs.F = &P.freq[0];
  ray_entry(P, rs.V, rs.F, pix[i], rs);
  PathNode* out = path + (size_t)i * cap;
  int nodes = 0;
  auto record = [&](float x, float y, float z, float lns, float dls, float tau, float ne, float te) {
    if (nodes < cap) {
      PathNode& q = out[nodes];
      q.r[0] = x; q.r[1] = y; q.r[2] = z;
      q.ln_s = lns; q.dlns_ds = dls; q.tau = tau; q.ne = ne; q.te = te;
    }
    ++nodes;
  };
  float tb_hi = 0.f, tb_lo = 0.f, tau_hi = 0.f, tau_lo = 0.f, lns_hi = 0.f, lns_lo = 0.f;
  int step = 0, status = kMiss;
  float ex = rs.px, ey = rs.py, ez = rs.pz;
  if (rs.enter) {
    const float kf = P.straight ? 0.f : rs.F->kf, kap_c = rs.F->kap_c, ln_f = rs.F->ln_f;
    float px = rs.px, py = rs.py, pz = rs.pz, kx = rs.kx, ky = rs.ky, kz = rs.kz;
    float rlx = 0.f, rly = 0.f, rlz = 0.f, klx = 0.f, kly = 0.f, klz = 0.f;
    float kap_prev = 0.f, te_prev = 0.f, dls = 0.f;
    while (true) {
      StagePoints sp;
      const float off_r = kCurv ? radial_reach(P.clear, px, py, pz, kx, ky, kz) : 0.f;
      const Rk4Out o = rk4_central<kCurv>(P.G, kf, h, px, py, pz, kx, ky, kz, off_r, P.clear.reach, &sp);
      // the step's end and ln M before the transfer, as in trace_rays: neither
      // waits for its exponentials (256 rays, 4 neighbours: 6.35 -> 6.17 ms)
      const Vec dr = chord(h, P.h2_6, o, kx, ky, kz, klx, kly, klz);
      Vec rn, kn;
      complete_step<kMixed>(P.h_6, o, dr, px, py, pz, kx, ky, kz, rlx, rly, rlz, klx, kly, klz, rn, kn);
      const float rr2 = dot3(rn, rn);
      float lm = 0.f;
      if (NB > 0) {
        Retrace R;
        bool fast = false;
        if (kCurv) {
          chord_frame(R, P.eta, P.eps_fixed, dr);
          float c2;
          R.lm = curvature_ln_m(sp, px, py, pz, R.t, P.h2_6 * kf, c2);
          fast = step_clear(P.clear, sp, R, dr) && c2 <= 1e-6f;
        }
        if (!fast)
          R = retrace_step<(NB > 0 ? NB : 4)>(P.G, kf, h, P.h2_6, P.h2_12, P.eta, P.eps_fixed, px, py, pz, kx, ky,
                                              kz, dr, Vec{o.Gx, o.Gy, o.Gz});
        lm = R.lm;
      }
      const float kap = P.emission ? kappa_vac(o.ne1, o.te1, kap_c, ln_f) : 0.f;
      if (step >= 1) {
        const float dt = 0.5f * (kap_prev + kap) * P.hrsun;
        const float tbar = 0.5f * (te_prev + o.te1);
        const float tau0 = tau_hi + tau_lo;
        acc_add<kMixed>(tb_hi, tb_lo, tbar * one_minus_exp_neg(dt) * __expf((lns_hi + lns_lo) - tau0));
        acc_add<kMixed>(tau_hi, tau_lo, dt);
      }
      record(px, py, pz, lns_hi + lns_lo, dls, tau_hi + tau_lo, o.ne1, o.te1);
      ex = px; ey = py; ez = pz;
      if (step >= 1 && P.tau_stop > 0.f && tau_hi + tau_lo >= P.tau_stop) { status = kTauStop; break; }
      if (step >= 1 && step >= P.max_steps) { status = kStepLimit; break; }
      kap_prev = kap;
      te_prev = o.te1;
      int term = 0;
      if (rr2 < P.G.r_min * P.G.r_min) term = kHitInner;
      else if (rr2 > P.G.r_max * P.G.r_max && dot3(rn, kn) > 0.f) term = kExitOuter;
      else if (!isfinite(rr2 + kn.x + kn.y + kn.z)) term = kNan;
      dls = 0.f;
      if (NB > 0 && term != kNan) {
        acc_add<kMixed>(lns_hi, lns_lo, lm);
        dls = lm * rsqrtf(dot3(dr, dr));
      }
      if (term == 0) {
        px = rn.x; py = rn.y; pz = rn.z;
        kx = kn.x; ky = kn.y; kz = kn.z;
        step += 1;
        continue;
      }
      step += 1;
      status = term;
      if (term == kNan) { ex = rn.x; ey = rn.y; ez = rn.z; break; }
      const Vec here{px, py, pz};
      const float a = chord_crossing(here, dr, (term == kHitInner) ? P.G.r_min : P.G.r_max, term == kExitOuter);
      const float cx = fmaf(a, dr.x, px), cy = fmaf(a, dr.y, py), cz = fmaf(a, dr.z, pz);
      const Sample s = eval_field(P.G, cx, cy, cz, true);
      const float kap_e = P.emission ? kappa_vac(s.ne, s.te, kap_c, ln_f) : 0.f;
      const float dt = 0.5f * (kap_prev + kap_e) * P.hrsun * a;
      const float tbar = 0.5f * (te_prev + s.te);
      const float lns = lns_hi + lns_lo;
      acc_add<kMixed>(tb_hi, tb_lo, tbar * one_minus_exp_neg(dt) * __expf(lns - (tau_hi + tau_lo)));
      acc_add<kMixed>(tau_hi, tau_lo, dt);
      float tbc = 0.f;
      if (term == kHitInner) tbc = (P.tbc_mode == 1) ? P.tbc_K : s.te;
      if (tbc != 0.f) acc_add<kMixed>(tb_hi, tb_lo, tbc * __expf(lns - (tau_hi + tau_lo)));
      record(cx, cy, cz, lns, dls, tau_hi + tau_lo, s.ne, s.te);
      ex = cx; ey = cy; ez = cz;
      break;
    }
  }
  count[i] = nodes;
  tb[i] = tb_hi + tb_lo;
  if (diag) {
    RayDiag d;
    d.exit_pos[0] = ex; d.exit_pos[1] = ey; d.exit_pos[2] = ez;
    d.tau = tau_hi + tau_lo;
    d.ln_s = lns_hi + lns_lo;
    d.steps = step;
    d.status = status;
    diag[i] = d;
  }
}

}  // namespace rt
