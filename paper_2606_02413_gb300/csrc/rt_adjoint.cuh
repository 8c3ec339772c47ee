// Reverse-mode (adjoint) building blocks and the adjoint ray-bundle kernel.
//
// The adjoint differentiates the discrete forward computation (Sec. 2.1
// Eqs. 4-12, Sec. 3.2) with respect to the grid node values of n_e and T_e,
// holding the discrete events fixed (cell indices, the basis axis branch,
// the step count and the termination step), the convention of the FP64
// oracle's tape adjoint.
//
// Interpolant derivatives used here, for a cell with corner values N_c and
// trilinear weights w_c(u, v, w):
//   value       f = sum_c w_c N_c,     d f / d N_c = w_c,     grad f as forward
//   gradient    g = sum_c grad w_c N_c, lambda . d g / d N_c = lambda . grad w_c
//               = sum_a (lambda . grad a) d w_c / d a   (a = u, v, w)
//   position    d (lambda . g) / d x = H lambda, the Hessian of the interpolant
//               applied to lambda, from its components in the spherical frame
//               (cell held fixed).
//   tube area   ln M = h^2/6 kf sum_s Q(P_s), Q = tr H - t.H t at the central
//               stage points, where the step stays clear of the cells' faces
//               (curvature_ln_m): with (r, theta, phi) partials f_i of the
//               interpolant Q = sum_i alpha_i f_i, the alpha functions of the
//               position and of t alone, so d Q / d N_c, d Q / d x and
//               d Q / d t = -2 H t come in closed form at the cell that the
//               central ray's own adjoint visits.
#pragma once
#include "rt_rays.cuh"

namespace rt {

// --------------------------------------------------------- cell geometry
struct CellGeom {
  int i, j, k, k1;           // cell and wrapped phi neighbour
  float u, v, w;             // fractions
  Vec du, dv, dw;            // Cartesian gradients of u, v, w (dv = 0 in the clamped theta caps)
  bool vac;                  // beyond the outer band
};

__device__ __forceinline__ CellGeom cell_geom(const GridDev& G, float x, float y, float z) {
  CellGeom c;
  const float rho2 = fmaf(x, x, y * y);
  const float r2 = fmaf(z, z, rho2);
  const float inv_r = rsqrtf(r2);
  const float r = r2 * inv_r;
  c.vac = !(r <= G.r_vac);
  if (c.vac) {
    c.i = c.j = c.k = c.k1 = 0;
    c.u = c.v = c.w = 0.f;
    c.du = c.dv = c.dw = {0.f, 0.f, 0.f};
    return c;
  }
  float2 rc;
  c.i = radial_lookup(G, r, rc.x, rc.y);
  c.u = (r - rc.x) * rc.y;
  const float inv_rho = (rho2 > 0.f) ? rsqrtf(rho2) : 0.f;
  const float rho = rho2 * inv_rho;
  // theta cell as in the field evaluation: clamped to the outermost cells,
  // where the fraction sticks at 0 or 1 and the theta derivative is off
  const float tt = (atan2_grid<true>(rho, z) - G.t0) * G.t_inv;
  c.j = min(max(__float2int_rd(tt), 0), G.n_t - 2);
  c.v = fminf(fmaxf(tt - (float)c.j, 0.f), 1.f);
  const float tsel = (tt > 0.f && tt < G.t_last) ? 1.f : 0.f;
  float ph = atan2_grid(y, x) - G.p0;
  if (ph < 0.f) ph += kTwoPiF;
  if (ph >= kTwoPiF) ph -= kTwoPiF;
  const float pp = ph * G.p_inv;
  c.k = min(max(__float2int_rd(pp), 0), G.n_p - 1);
  c.w = pp - (float)c.k;
  c.k1 = (c.k + 1 == G.n_p) ? 0 : c.k + 1;
  // grad u = r_hat / dr; grad v = theta_hat / (r dtheta); grad w = phi_hat / (rho dphi)
  const float a = rc.y * inv_r;
  c.du = {a * x, a * y, a * z};
  const float ir2 = inv_r * inv_r;
  const float bt = tsel * G.t_inv * ir2;
  c.dv = {bt * z * x * inv_rho, bt * z * y * inv_rho, -bt * rho};
  const float bp = G.p_inv * inv_rho * inv_rho;
  c.dw = {-bp * y, bp * x, 0.f};
  return c;
}

__device__ __forceinline__ long node_index(const GridDev& G, const CellGeom& c, int a, int b, int cc) {
  return ((long)(c.i + a) * G.n_t + (c.j + b)) * G.n_p + (cc ? c.k1 : c.k);
}

// Value scatter: d/dN_c of (lam_ne n_e + lam_te T_e) = w_c (lam_ne, lam_te);
// returns lam_ne grad n_e + lam_te grad T_e (the position adjoint).
__device__ __forceinline__ Vec value_adjoint(const GridDev& G, float x, float y, float z, float lam_ne, float lam_te,
                                             float* dne, float* dte) {
  const CellGeom c = cell_geom(G, x, y, z);
  if (c.vac) return {0.f, 0.f, 0.f};
  const int cell = (c.i * (G.n_t - 1) + c.j) * G.n_p + c.k;
  const float4 n0 = __ldg(G.ne + 2 * cell), n1 = __ldg(G.ne + 2 * cell + 1);
  const float4 t0 = __ldg(G.te + 2 * cell), t1 = __ldg(G.te + 2 * cell + 1);
  const float nv[8] = {n0.x, n0.z, n1.x, n1.z, n0.y, n0.w, n1.y, n1.w};  // [a][b][c]
  const float tv[8] = {t0.x, t0.z, t1.x, t1.z, t0.y, t0.w, t1.y, t1.w};
  const float wu[2] = {1.f - c.u, c.u}, wv[2] = {1.f - c.v, c.v}, ww[2] = {1.f - c.w, c.w};
  const float sg[2] = {-1.f, 1.f};
  float fu = 0.f, fv = 0.f, fw = 0.f, tu = 0.f, tvv = 0.f, tw = 0.f;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int cc = 0; cc < 2; ++cc) {
        const int q = a * 4 + b * 2 + cc;
        const float wgt = wu[a] * wv[b] * ww[cc];
        const long id = node_index(G, c, a, b, cc);
        if (lam_ne != 0.f) atomicAdd(dne + id, lam_ne * wgt);
        if (lam_te != 0.f) atomicAdd(dte + id, lam_te * wgt);
        const float gu = sg[a] * wv[b] * ww[cc], gv = wu[a] * sg[b] * ww[cc], gw = wu[a] * wv[b] * sg[cc];
        fu = fmaf(gu, nv[q], fu); fv = fmaf(gv, nv[q], fv); fw = fmaf(gw, nv[q], fw);
        tu = fmaf(gu, tv[q], tu); tvv = fmaf(gv, tv[q], tvv); tw = fmaf(gw, tv[q], tw);
      }
  const float an = lam_ne * fu + lam_te * tu, bn = lam_ne * fv + lam_te * tvv, cn = lam_ne * fw + lam_te * tw;
  return {an * c.du.x + bn * c.dv.x + cn * c.dw.x, an * c.du.y + bn * c.dv.y + cn * c.dw.y,
          an * c.du.z + bn * c.dv.z + cn * c.dw.z};
}

// Per-thread accumulator of the node adjoints of one cell, in shared memory
// laid out [corner][thread] (a warp's accesses hit distinct banks): n_e's and,
// after them, T_e's.  The adjoints of a step lie within a few 1e-3 R_sun of
// its node, and mostly in the node's cell: they add here, and the sums reach
// the grid with 16 atomics when the node moves to another cell or the ray
// ends, instead of 8 or 16 per adjoint.  Stage points in another cell scatter
// directly.
template <int kThreadsAcc>
struct NodeAcc {
  static constexpr int T = kThreadsAcc;
  float* v;    // v[q * T], corner q = 4 a + 2 b + c of n_e, 8 + q of T_e
  int* key;    // the cell held (-1: none)
};

template <int T>
__device__ __forceinline__ void acc_flush(const GridDev& G, const NodeAcc<T>& A, float* dne, float* dte) {
  const int cell = *A.key;
  if (cell < 0) return;
  // node (i, j, k) of the cell's corner (0, 0, 0): one theta row more per shell than cells
  const long b0 = (long)cell + (long)(cell / ((G.n_t - 1) * G.n_p)) * G.n_p, sr = (long)G.n_t * G.n_p;
  const int dk = (cell % G.n_p + 1 == G.n_p) ? 1 - G.n_p : 1;  // k1 - k: back across the phi seam
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const long id = b0 + (q >> 2) * sr + ((q >> 1) & 1) * G.n_p + (q & 1) * dk;
    const float x = A.v[q * T], y = A.v[(8 + q) * T];
    if (x != 0.f) atomicAdd(dne + id, x);
    if (y != 0.f) atomicAdd(dte + id, y);
    A.v[q * T] = 0.f;
    A.v[(8 + q) * T] = 0.f;
  }
  *A.key = -1;
}

// Adjoint of the field's use at one RK4 stage point p.  Given lam = dL/da of
// the force a = kf grad n_e(p) and lq = dL/dQ of the tube area's Q(p; t) (0:
// none), scatters
//   kf lam . grad w_c + lq d Q / d N_c
// to the n_e nodes (through the accumulator A when p lies in its cell; adopt:
// p is a node, whose cell the accumulator takes over) and returns the position
// adjoint kf H(p) lam + lq d Q / d p.  value (p is a node): also the adjoints
// (lam_ne, lam_te) of the interpolated n_e and T_e themselves, w_c (lam_ne,
// lam_te) to the nodes and lam_ne grad n_e + lam_te grad T_e to the position.
// All uses share the cell, its corners and one scatter.  on = false: a lane
// that only keeps the warp together.  kShare: the four lanes of an aligned group
// reverse the four neighbours of one ray, acc is that ray's accumulator, and
// what of the group falls into its cell is summed over the group before it is
// added, two corners a lane: the parts of a +-pair nearly cancel, and must not
// meet in other sums first (scattered by each lane on its own, n_e's gradient
// on 5x3x4 cells was 2e-5 off, relative L2, where it is 2e-6 now).
template <bool kShare, int T>
__device__ __forceinline__ Vec stage_adjoint(const GridDev& G, float kf, float x, float y, float z, const Vec& lam,
                                             float lq, const Vec& t, float* dne, float* dte, const NodeAcc<T>& acc,
                                             bool adopt, bool value, float lam_ne, float lam_te, bool on) {
  const float rho2 = fmaf(x, x, y * y);
  const float r2 = fmaf(z, z, rho2);
  const float inv_r = rsqrtf(r2);
  const float r = r2 * inv_r;
  float R, inv_dr;
  const int i = radial_lookup(G, r, R, inv_dr);  // n_r - 1: the vacuum shell, all zero
  const float u = (r - R) * inv_dr;
  const float inv_rho = (rho2 > 0.f) ? rsqrtf(rho2) : 0.f;
  const float rho = rho2 * inv_rho;
  const float tt = (atan2_grid<true>(rho, z) - G.t0) * G.t_inv;
  const int j = min(max(__float2int_rd(tt), 0), G.n_t - 2);
  const float v = fminf(fmaxf(tt - (float)j, 0.f), 1.f);
  const float ti = (tt > 0.f && tt < G.t_last) ? G.t_inv : 0.f;  // no theta derivative in the clamped caps
  float ph = atan2_grid(y, x) - G.p0;
  if (ph < 0.f) ph += kTwoPiF;
  if (ph >= kTwoPiF) ph -= kTwoPiF;
  const float pp = ph * G.p_inv;
  const int k = min(max(__float2int_rd(pp), 0), G.n_p - 1);
  const float w = pp - (float)k;
  const int cell = (i * (G.n_t - 1) + j) * G.n_p + k;
  const bool scatter = on && i < G.n_r - 1;

  // partials of the interpolant in (u, v, w), then in (r, theta, phi)
  float n000, n001, n010, n011, n100, n101, n110, n111;
  ldg8(G.ne + 2 * cell, n000, n100, n001, n101, n010, n110, n011, n111);
  const float d00 = n001 - n000, d01 = n011 - n010, d10 = n101 - n100, d11 = n111 - n110;
  const float a00 = fmaf(w, d00, n000), a01 = fmaf(w, d01, n010), a10 = fmaf(w, d10, n100), a11 = fmaf(w, d11, n110);
  const float e0 = a01 - a00, e1 = a11 - a10;
  const float q0 = d01 - d00, q1 = d11 - d10;
  const float g0 = fmaf(v, q0, d00), g1 = fmaf(v, q1, d10);
  const float f_r = (fmaf(v, e1, a10) - fmaf(v, e0, a00)) * inv_dr;
  const float f_t = fmaf(u, e1 - e0, e0) * ti;
  const float f_p = fmaf(u, g1 - g0, g0) * G.p_inv;
  const float f_rt = (e1 - e0) * inv_dr * ti;
  const float f_rp = (g1 - g0) * inv_dr * G.p_inv;
  const float f_tp = fmaf(u, q1 - q0, q0) * ti * G.p_inv;
  const float f_rtp = (q1 - q0) * inv_dr * ti * G.p_inv;

  // the Hessian in the spherical frame (H_rr = 0) and lam there
  const float cot = z * inv_rho, cs = z * inv_r;  // cot and cos of theta
  const float htt = f_r * inv_r;
  const float hpp = fmaf(f_t * cot, inv_r * inv_r, htt);
  const float hrt = inv_r * fmaf(-f_t, inv_r, f_rt);
  const float hrp = inv_rho * fmaf(-f_p, inv_r, f_rp);
  const float htp = inv_r * inv_rho * fmaf(-cot, f_p, f_tp);
  const float xl = fmaf(x, lam.x, y * lam.y);
  const float lr = fmaf(z, lam.z, xl) * inv_r;
  const float lt = fmaf(cot, xl, -rho * lam.z) * inv_r;
  const float lp = fmaf(x, lam.y, -y * lam.x) * inv_rho;
  float pr = kf * fmaf(hrt, lt, hrp * lp);                    // position adjoint in the frame
  float pt = kf * fmaf(hrt, lr, fmaf(htt, lt, htp * lp));
  float pf = kf * fmaf(hrp, lr, fmaf(htp, lt, hpp * lp));
  // node coefficients of w_c's partials: first (from lam) and mixed
  float cu = kf * lr * inv_dr, cv = kf * lt * inv_r * ti, cw = kf * lp * inv_rho * G.p_inv;
  float cuv = 0.f, cuw = 0.f, cvw = 0.f;
  if (lq != 0.f) {
    const float xt = fmaf(x, t.x, y * t.y);
    const float tr = fmaf(z, t.z, xt) * inv_r;
    const float th = fmaf(cot, xt, -rho * t.z) * inv_r;
    const float tp = fmaf(x, t.y, -y * t.x) * inv_rho;
    const float is = r * inv_rho, sn = rho * inv_r;       // 1 / sin theta, sin theta
    const float m = fmaf(cot, th, tr);                    // (t_r sin + t_th cos) / sin
    const float ir2 = inv_r * inv_r;
    const float omp = fmaf(-tp, tp, 1.f);
    // Q = sum alpha_i f_i
    const float c1 = fmaf(tr, tr, 1.f) * inv_r;
    const float c2 = fmaf(cot, omp, 2.f * tr * th) * ir2;
    const float c3 = 2.f * tp * m * is * ir2;
    const float c4 = -2.f * tr * th * inv_r;
    const float c5 = -2.f * tr * tp * is * inv_r;
    const float c6 = -2.f * th * tp * is * ir2;
    // d Q / d r: the partials' own change, and the alphas' (powers of r)
    const float dr_f = fmaf(c2, f_rt, fmaf(c3, f_rp, c6 * f_rtp));
    const float dr_a = -inv_r * (fmaf(c1, f_r, fmaf(c4, f_rt, c5 * f_rp)) +
                                 2.f * fmaf(c2, f_t, fmaf(c3, f_p, c6 * f_tp)));
    // d Q / d theta with t fixed in space: d t_r = t_th, d t_th = -t_r
    const float dt2 = fmaf(th, th, -tr * tr);
    const float dt_f = fmaf(c1, f_rt, fmaf(c3, f_tp, c5 * f_rtp));
    const float dt_a = 2.f * tr * th * inv_r * f_r + ir2 * fmaf(2.f, dt2, -omp * is * is) * f_t -
                       2.f * cot * c3 * f_p - 2.f * dt2 * inv_r * f_rt -
                       2.f * tp * is * fmaf(-cot, tr, th) * inv_r * f_rp + c3 * f_tp;
    // d Q / d phi: d t_r = sin t_p, d t_th = cos t_p, d t_p = -(sin t_r + cos t_th)
    const float dp_f = fmaf(c1, f_rp, fmaf(c2, f_tp, c4 * f_rtp));
    const float b = 2.f * tp * fmaf(sn, th, cs * tr);
    const float dp_a = 2.f * tr * sn * tp * inv_r * f_r + ir2 * fmaf(2.f * cs * tp, m, b) * f_t +
                       2.f * ir2 * fmaf(tp * is, tp * is, -m * m) * f_p - b * inv_r * f_rt -
                       2.f * inv_r * fmaf(tp, tp, -tr * m) * f_rp - 2.f * ir2 * fmaf(cot * tp, tp, -th * m) * f_tp;
    pr = fmaf(lq, dr_f + dr_a, pr);
    pt = fmaf(lq * inv_r, dt_f + dt_a, pt);
    pf = fmaf(lq * inv_rho, dp_f + dp_a, pf);
    cu = fmaf(lq * c1, inv_dr, cu);
    cv = fmaf(lq * c2, ti, cv);
    cw = fmaf(lq * c3, G.p_inv, cw);
    cuv = lq * c4 * inv_dr * ti;
    cuw = lq * c5 * inv_dr * G.p_inv;
    cvw = lq * c6 * ti * G.p_inv;
  }

  // node scatter: w_c = U_a V_b W_c
  if (adopt && scatter && cell != *acc.key) {
    acc_flush(G, acc, dne, dte);
    *acc.key = cell;
  }
  float wn = 0.f;  // weight of w_c itself
  if (value) {
    wn = lam_ne;
    float m000, m001, m010, m011, m100, m101, m110, m111;
    ldg8(G.te + 2 * cell, m000, m100, m001, m101, m010, m110, m011, m111);
    const float b00 = fmaf(w, m001 - m000, m000), b01 = fmaf(w, m011 - m010, m010);
    const float b10 = fmaf(w, m101 - m100, m100), b11 = fmaf(w, m111 - m110, m110);
    const float t_r = (fmaf(v, b11 - b10, b10) - fmaf(v, b01 - b00, b00)) * inv_dr;
    const float t_t = fmaf(u, (b11 - b10) - (b01 - b00), b01 - b00) * ti;
    const float h0 = fmaf(v, (m011 - m010) - (m001 - m000), m001 - m000);
    const float h1 = fmaf(v, (m111 - m110) - (m101 - m100), m101 - m100);
    const float t_p = fmaf(u, h1 - h0, h0) * G.p_inv;
    pr += fmaf(lam_ne, f_r, lam_te * t_r);
    pt += fmaf(lam_ne, f_t, lam_te * t_t) * inv_r;
    pf += fmaf(lam_ne, f_p, lam_te * t_p) * inv_rho;
    // T_e's nodes: the node's own cell, which the accumulator holds
    const bool te = scatter && lam_te != 0.f;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const float uv = te ? lam_te * ((a ? u : 1.f - u) * (b ? v : 1.f - v)) : 0.f;
        acc.v[(8 + a * 4 + b * 2) * T] += uv * (1.f - w);
        acc.v[(8 + a * 4 + b * 2 + 1) * T] += uv * w;
      }
  }
  const bool hit = scatter && cell == *acc.key;
  const bool miss = scatter && !hit;
  float* nb = dne + (((long)i * G.n_t + j) * G.n_p + k);
  const long sr = (long)G.n_t * G.n_p;
  const int dk = (k + 1 == G.n_p) ? 1 - G.n_p : 1;
  float part[8];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const float U = a ? u : 1.f - u, V = b ? v : 1.f - v;
      const float su = a ? 1.f : -1.f, sv = b ? 1.f : -1.f;
      const float X = fmaf(U * V, wn, fmaf(su * V, cu, fmaf(sv * U, cv, su * sv * cuv)));
      const float Y = fmaf(U * V, cw, fmaf(su * V, cuw, sv * U * cvw));
      const float v0 = fmaf(X, 1.f - w, -Y), v1 = fmaf(X, w, Y);
      // both branches as straight-line code: the shared adds take 0 on a
      // miss, the atomics are predicated (no divergence among the corners)
      const int q = a * 4 + b * 2;
      if (kShare) {
        part[q] = hit ? v0 : 0.f;
        part[q + 1] = hit ? v1 : 0.f;
      } else {
        acc.v[q * T] += hit ? v0 : 0.f;
        acc.v[(q + 1) * T] += hit ? v1 : 0.f;
      }
      if (miss) {
        atomicAdd(nb + a * sr + b * G.n_p, v0);
        atomicAdd(nb + a * sr + b * G.n_p + dk, v1);
      }
    }
  if (kShare) {  // the group's sums, halved between the lanes along phi and then along theta
    const bool c1 = threadIdx.x & 1, b1 = threadIdx.x & 2;
    float half[4];  // corners (a, b, c1) over the pair
#pragma unroll
    for (int n = 0; n < 4; ++n)
      half[n] = (c1 ? part[2 * n + 1] : part[2 * n]) + __shfl_xor_sync(kFull, c1 ? part[2 * n] : part[2 * n + 1], 1);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const float sum = (b1 ? half[2 * a + 1] : half[2 * a]) + __shfl_xor_sync(kFull, b1 ? half[2 * a] : half[2 * a + 1], 2);
      if (on) acc.v[(a * 4 + (threadIdx.x & 2) + (threadIdx.x & 1)) * T] += sum;
    }
  }
  // back to Cartesian
  const float rr = pr * inv_r, tq = pt * inv_r, pq = pf * inv_rho;
  const float h = fmaf(tq, cot, rr);
  return {fmaf(h, x, -pq * y), fmaf(h, y, pq * x), fmaf(rr, z, -tq * rho)};
}

// Reverse of one RK4 step from (p, k) (rk4_central, or rk4_g3 for a
// neighbour's retrace), given the adjoints of its outputs: lr = dL/dr',
// lk = dL/dk' and lg on G = a1 + a2 + a3; lq = dL/dQ of the tube area at a
// stage point (0: none; the second stage's also stands for the third), t its
// direction.  With
// r' = r + h k + h^2/6 G and k' = k + h/6 (a1 + 2 a2 + 2 a3 + a4), the stage
// points are P1 = p, P2 = p + h/2 k, P3 = p + h/2 k2, P4 = p + h k3 with
// k2 = k + h/2 a1, k3 = k + h/2 a2, and a_s = kf grad n_e(P_s); P3 and P4 come
// from the recomputation.  value: the adjoints lam_ne, lam_te of n_e and T_e at
// the node p join its stage.
// kStages = 4 (central ray) or 3 (a neighbour: lr = lk = 0 and the fourth
// stage has no adjoint).  Adds dL/dp to lp and dL/dk to lko and scatters the
// n_e nodes.  The stages are reversed in one loop around a single adjoint
// (the kernel's instruction footprint, not its arithmetic, bounds it).
template <int kStages, int T>
__device__ __forceinline__ void rk4_reverse(const GridDev& G, float kf, float h, const Vec& p, const Vec& k,
                                            const Vec& P3, const Vec& P4, const Vec& lr, const Vec& lk,
                                            const Vec& lg, float lq, const Vec& t, bool value, float lam_ne,
                                            float lam_te, Vec& lp, Vec& lko, float* dne, float* dte,
                                            const NodeAcc<T>& A, bool on) {
  const float hh = 0.5f * h, h6 = h / 6.f, h3 = h / 3.f;
  const Vec P2{fmaf(hh, k.x, p.x), fmaf(hh, k.y, p.y), fmaf(hh, k.z, p.z)};
  // adjoints of the accelerations and velocities from the outputs
  // (k4 = k + h a3 enters r' only: its adjoint h/6 lr is applied at once)
  Vec La1{fmaf(h6, lk.x, lg.x), fmaf(h6, lk.y, lg.y), fmaf(h6, lk.z, lg.z)};
  Vec La2{fmaf(h3, lk.x, lg.x), fmaf(h3, lk.y, lg.y), fmaf(h3, lk.z, lg.z)};
  Vec La3{fmaf(h * h6, lr.x, La2.x), fmaf(h * h6, lr.y, La2.y), fmaf(h * h6, lr.z, La2.z)};
  const Vec La4{h6 * lk.x, h6 * lk.y, h6 * lk.z};
  Vec Lk2{h3 * lr.x, h3 * lr.y, h3 * lr.z}, Lk3 = Lk2;  // adjoints of k2, k3
  Vec Lp{lr.x, lr.y, lr.z};
  Vec Lk{lk.x + 2.f * h6 * lr.x, lk.y + 2.f * h6 * lr.y, lk.z + 2.f * h6 * lr.z};  // k itself and k4 = k + h a3
#pragma unroll 1
  for (int s = kStages - 1; s >= 0; --s) {
    const Vec pt = (s == 3) ? P4 : (s == 2) ? P3 : (s == 1) ? P2 : p;
    const Vec la = (s == 3) ? La4 : (s == 2) ? La3 : (s == 1) ? La2 : La1;
    // the central ray's stage 1 is the node: the accumulator follows it
    const Vec LP = stage_adjoint<kStages == 3>(G, kf, pt.x, pt.y, pt.z, la,
                                 (s >= 2) ? 0.f : (s == 1) ? 2.f * lq : lq, t, dne, dte, A,
                                 kStages == 4 && s == 0, kStages == 4 && s == 0 && value, lam_ne, lam_te, on);
    Lp = {Lp.x + LP.x, Lp.y + LP.y, Lp.z + LP.z};
    if (s == 3) {         // P4 = p + h k3, k3 = k + h/2 a2
      Lk3 = {fmaf(h, LP.x, Lk3.x), fmaf(h, LP.y, Lk3.y), fmaf(h, LP.z, Lk3.z)};
      Lk = {Lk.x + Lk3.x, Lk.y + Lk3.y, Lk.z + Lk3.z};
      La2 = {fmaf(hh, Lk3.x, La2.x), fmaf(hh, Lk3.y, La2.y), fmaf(hh, Lk3.z, La2.z)};
    } else if (s == 2) {  // P3 = p + h/2 k2, k2 = k + h/2 a1
      Lk2 = {fmaf(hh, LP.x, Lk2.x), fmaf(hh, LP.y, Lk2.y), fmaf(hh, LP.z, Lk2.z)};
      Lk = {Lk.x + Lk2.x, Lk.y + Lk2.y, Lk.z + Lk2.z};
      La1 = {fmaf(hh, Lk2.x, La1.x), fmaf(hh, Lk2.y, La1.y), fmaf(hh, Lk2.z, La1.z)};
    } else if (s == 1) {  // P2 = p + h/2 k
      Lk = {fmaf(hh, LP.x, Lk.x), fmaf(hh, LP.y, Lk.y), fmaf(hh, LP.z, Lk.z)};
    }
  }
  lp = {lp.x + Lp.x, lp.y + Lp.y, lp.z + Lp.z};
  lko = {lko.x + Lk.x, lko.y + Lk.y, lko.z + Lk.z};
}

// sum over the stage points of -2 H t (the second stands for the third),
// Cartesian: d (sum_s Q_s) / d t.
__device__ __forceinline__ Vec curvature_dt(const StagePoints& sp, float px, float py, float pz, const Vec& t) {
  const float xs[2] = {px, sp.x2}, ys[2] = {py, sp.y2}, zs[2] = {pz, sp.z2};
  Vec o{0.f, 0.f, 0.f};
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const Curv& c = sp.cv[s];
    const float x = xs[s], y = ys[s], z = zs[s];
    const float cot = z * c.inv_rho, xt = fmaf(x, t.x, y * t.y);
    const float tr = fmaf(z, t.z, xt) * c.inv_r;
    const float tt = fmaf(cot, xt, -c.rho * t.z) * c.inv_r;
    const float tp = fmaf(x, t.y, -y * t.x) * c.inv_rho;
    const float hr = fmaf(c.hrt, tt, c.hrp * tp) * c.inv_r;
    const float ht = fmaf(c.hrt, tr, fmaf(c.htt, tt, c.htp * tp)) * c.inv_r;
    const float hp = fmaf(c.hrp, tr, fmaf(c.htp, tt, c.hpp * tp)) * c.inv_rho;
    const float m = fmaf(ht, cot, hr);
    const float n = (s == 1) ? -4.f : -2.f;
    o = {fmaf(n, fmaf(m, x, -hp * y), o.x), fmaf(n, fmaf(m, y, hp * x), o.y), fmaf(n, fmaf(hr, z, -ht * c.rho), o.z)};
  }
  return o;
}

// d kappa_vac / d n_e and d kappa_vac / d T_e (see kappa_vac).
__device__ __forceinline__ void kappa_partials(float ne, float te, float kap_c, float ln_f, float& dk_dne,
                                               float& dk_dte) {
  dk_dne = dk_dte = 0.f;
  if (!(ne > 0.f) || !(te > 0.f)) return;
  const float lnT = __logf(te);
  const bool hot = te > 2e5f;
  const float g = hot ? (24.5f + lnT - ln_f) : fmaf(1.5f, lnT, 18.2f - ln_f);
  const float rs = rsqrtf(te);
  const float base = (kap_c * ne) * (rs * rs * rs);  // kap_c n_e T^-1.5
  dk_dne = 2.f * base * g;
  dk_dte = base * ne * ((hot ? 1.f : 1.5f) - 1.5f * g) / te;
}

// ------------------------------------------------------------ the kernel
struct AdjParams {
  GridDev G;
  float h, h2_6, h_6, h2_12, hrsun, eta, eps_fixed, tbc_K;
  Clear clear;
  int tbc_mode, emission, curv;
  ViewDev view;
  int nf;
  FreqDev freq[kMaxFreq];
  const RayDiag* diag;         // forward diagnostics (steps, status), output order
  const float* dL_dTb;         // [nf][npix], output order
  const Ckpt* ckpt;
  const unsigned long long* ck_off;  // ray t owns ckpt[ck_off[t] .. ck_off[t+1]); or, a tape:
  const int* ck_prev;                // the pool's links to each ray's previous checkpoint
  const int* ck_last;                // and each ray's last checkpoint
  float* dne;
  float* dte;
  unsigned int* counter;
  unsigned int total;
  int lanes;                     // rays of a warp (32 unless the launch has fewer rays than thread slots)
  unsigned long long* mismatch;  // rays whose step count does not match their checkpoint allocation
};

// One recomputed step of a segment (node m = m0 + j), in the thread's local
// memory (the reverse reads it back last to first).
struct StepRec {
  float r[3], k[3], dr[3];     // node state and the chord increment of step m
  float p3[3], p4[3];          // its stage points 3 and 4
  float kap, te, ne;           // node transfer values
  float sw;                    // ln S at node m+1 minus the optical depth at node m
  float c1[3], c2[3], lnm;     // a retraced step: scaled separations of the +-e1, +-e2 pairs and ln M; else in
                               // c1 d (sum Q_s) / d t (ln M came from the second derivatives)
  int retraced;
};

// What a lane hands to the lanes that reverse its neighbours' retraces, and
// what comes back from them.
struct AdjointSlot {
  union {
    struct {
      float r[3], k[3], e1[3], e2[3];  // node, wave vector, transverse basis
      float l1[3], l2[3];              // adjoints of G on the "+" member of each pair
      float eps, kf;
      int thread;                      // the asking lane's
    } in;
    float out[4][6];                 // dL/dp, dL/dk of each neighbour
  };
};

// The adjoint of the forward (trace_rays), one thread per ray bundle.  Per
// ray, segment by segment from the last: recompute the segment's K central
// steps from its checkpoint with the forward's own step code, then reverse it
// step by step: (A) the transfer of the segment and the tube area of the step
// (Eqs. 2, 9-12), (B) the neighbours' retraces (RK4 stages 1-3) of a step that
// retraced them, (C) the central RK4 step with its chord, basis and eps (Eqs.
// 4-8) and, where ln M came from the field's second derivatives, their adjoint
// at the same three stage points.  Supported forms: step-wise with 4
// neighbours, or magnification off (NB = 0).
//
// The lanes of a warp go through their segments together (one without a step
// to do computes on stale state and writes nothing), because (B) is shared:
// the few lanes of a warp that retraced hand their four neighbours to the
// other lanes, as in the forward.  A step takes its ln M from the second
// derivatives here where |C| <= 1e-4, so that the first order's derivative
// errs by less than that (gradients over steps up to 8e-3 R_sun are as far from
// 64 bits as with every step retraced); one that the forward took so with a
// larger |C| is replayed from a retrace, equal to the third order in C.
//
// One block holds all the warps of an SM (T / 32 of them at most, see
// launch_adjoint_rays) and keeps them in the same phase (one
// barrier between recomputation and reverse, one per reversed step): the
// kernel's code is larger than the instruction caches near the schedulers, and
// warps in different phases waited 2.0 of 5.7 stall cycles per issued
// instruction for it.  One GB300, 128x90x180 corona, 128^2 x 8 frequencies,
// forward with tape and reverse sweep: 328 ms with 16 force adjoints a step and
// 128-thread blocks, 223 ms with the second derivatives, 173 ms with one block
// an SM and the value adjoints in the node's own stage, 150 ms with 12 or 16
// warps by rounds and each ray's retraces summed into its own accumulator.
// Bound by latency and issue (54% of the slots): 194 warp-instructions per
// ray-step (466 before), of which the shared retraces take about a third.  Where every step is retraced (dtau
// 1e-2, 64x32x64 corona, 320^2 x 2 maps) the reverse sweep takes 60 ms (75 ms
// with a ray's neighbours one after the other in its own lane).
template <int NB, bool kMixed, int T>
__global__ void __launch_bounds__(T, 1) adjoint_rays(const __grid_constant__ AdjParams P) {
  static_assert(NB == 0 || NB == 4, "adjoint: 4 step-wise neighbours or none");
  constexpr int K = kCkptEvery;
  constexpr int kPer = 8;  // lanes that four neighbours each fill a warp
  const int lane = threadIdx.x & 31;
  const float h = P.h;
  StepRec R[K];
  __shared__ float acc_v[16 * T];
  __shared__ int acc_key[T];
  // a warp's slots: the recomputation's or the reverse's
  __shared__ union Slots {
    RetraceSlot<4> f[NB ? kPer : 1];
    AdjointSlot a[NB ? kPer : 1];
    __device__ Slots() {}
  } slots_of[T / 32];
  Slots& S = slots_of[threadIdx.x >> 5];
  const NodeAcc<T> A{acc_v + threadIdx.x, acc_key + threadIdx.x};
#pragma unroll
  for (int q = 0; q < 16; ++q) A.v[q * T] = 0.f;
  *A.key = -1;

  // per-ray state of the reverse sweep
  unsigned int item = 0;
  bool active = false, exhausted = lane >= P.lanes;
  int N = 0, status = 0, seg = 0;
  int slot = -1;  // tape: the pool slot of segment seg's checkpoint
  bool clipped = false;
  float kf = 0.f, kn2 = 0.f, kap_c = 0.f, ln_f = 0.f, lamT = 0.f, alpha = 1.f;
  float Wsuf = 0.f;                   // weight of everything beyond the node (sum of later terms)
  Vec Lr{0.f, 0.f, 0.f}, Lk{0.f, 0.f, 0.f};  // adjoints of the node state (r, k)
  float lkap = 0.f, lte = 0.f;        // partial adjoints of kappa and T_e at the node
  float px = 0.f, py = 0.f, pz = 0.f, kx = 0.f, ky = 0.f, kz = 0.f;  // state of the recomputed step

  // The block's warps meet here (when measured: tape and reverse of 128^2 x 8
  // rays 204 ms on their own, 165 ms together; 40^2 x 2 rays, one warp a
  // scheduler, 40.3 and 36.6 ms).  The result passes through a vote, so that the
  // compiler knows it uniform (the barrier's own: 166 and 37.2 ms).
  auto any = [&](bool v) { return __any_sync(kFull, __syncthreads_or(v)); };

  while (true) {
    // ---------------------------------------------------------- refill
    bool need = !active && !exhausted;
    unsigned needmask = __ballot_sync(kFull, need);
    while (needmask) {
      const int leader = __ffs(needmask) - 1;
      unsigned int first = 0;
      if (lane == leader) first = atomicAdd(P.counter, (unsigned)__popc(needmask));
      first = __shfl_sync(kFull, first, leader);
      if (need) {
        item = first + __popc(needmask & ((1u << lane) - 1u));
        if (item >= P.total) {
          exhausted = true;
          need = false;
        } else {
          const int fi = item / P.view.tickets;
          const int pix = item - fi * P.view.tickets;
          const FreqDev& F = P.freq[fi];
          const size_t o = (size_t)F.out_slab * P.view.npix + pix;
          const RayDiag d = P.diag[o];
          const float lw = P.dL_dTb[o];
          // the checkpoints were sized from a step count: it must be this ray's
          const unsigned long long n_ck =
              (d.steps > 0 && lw != 0.f) ? (unsigned long long)((d.steps - 1) / K + 1) : 0ull;
          // a tape's chain is checked segment by segment (the checkpoint's step)
          const bool fits = P.ck_prev ? true : P.ck_off[item + 1] - P.ck_off[item] == n_ck;
          if (!fits) atomicAdd(P.mismatch, 1ull);
          if (P.ck_prev) slot = P.ck_last[item];
          if (fits && d.steps > 0 && d.status >= kExitOuter && d.status <= kStepLimit && lw != 0.f) {
            N = d.steps;
            status = d.status;
            clipped = (d.status == kExitOuter || d.status == kHitInner);
            seg = (d.steps - 1) / K;
            kf = F.kf; kn2 = F.kn2; kap_c = F.kap_c; ln_f = F.ln_f;
            lamT = lw;
            alpha = 1.f;
            Wsuf = 0.f;
            Lr = {0.f, 0.f, 0.f};
            Lk = {0.f, 0.f, 0.f};
            lkap = lte = 0.f;
            active = true;
            need = false;
          }
        }
      }
      needmask = __ballot_sync(kFull, need);
    }
    if (!any(active)) break;

    // ---------------------------------------------- recompute the segment
    if (active && P.ck_prev && (slot < 0 || P.ckpt[slot].step != seg * K)) {
      // the tape does not hold this segment: the diagnostics belong to another forward
      atomicAdd(P.mismatch, 1ull);
      acc_flush(P.G, A, P.dne, P.dte);
      active = false;
    }
    const int m0 = seg * K;
    const int n_s = active ? min(K, N - m0) : 0;
    const bool last_seg = (m0 + n_s == N);
    float rlx = 0.f, rly = 0.f, rlz = 0.f, klx = 0.f, kly = 0.f, klz = 0.f, tau = 0.f, lns = 0.f;
    if (active) {
      const Ckpt& c = P.ckpt[P.ck_prev ? (unsigned long long)slot : P.ck_off[item] + seg];
      px = c.r[0]; py = c.r[1]; pz = c.r[2];
      kx = c.k[0]; ky = c.k[1]; kz = c.k[2];
      rlx = c.rl[0]; rly = c.rl[1]; rlz = c.rl[2];
      klx = c.kl[0]; kly = c.kl[1]; klz = c.kl[2];
      tau = c.tau_hi + c.tau_lo;
      lns = c.lns_hi + c.lns_lo;
    }
    const int n_all = __reduce_max_sync(kFull, n_s);
    float kap_prev = 0.f;
    for (int j = 0; j < n_all; ++j) {
      const bool live = j < n_s;
      StagePoints sp;
      Rk4Out o;
      if (NB > 0) {
        const float off_r = radial_reach(P.clear, px, py, pz, kx, ky, kz);
        o = rk4_central<true>(P.G, kf, h, px, py, pz, kx, ky, kz, off_r, P.clear.reach, &sp);
      } else {
        o = rk4_central<false>(P.G, kf, h, px, py, pz, kx, ky, kz, 0.f, 0.f, &sp);
      }
      const float kap = P.emission ? kappa_vac(o.ne1, o.te1, kap_c, ln_f) : 0.f;
      if (j > 0) tau += 0.5f * (kap_prev + kap) * P.hrsun;
      kap_prev = kap;
      StepRec& rc = R[min(j, K - 1)];
      if (live) {
        rc.r[0] = px; rc.r[1] = py; rc.r[2] = pz;
        rc.k[0] = kx; rc.k[1] = ky; rc.k[2] = kz;
        rc.p3[0] = sp.x3; rc.p3[1] = sp.y3; rc.p3[2] = sp.z3;
        rc.p4[0] = sp.x4; rc.p4[1] = sp.y4; rc.p4[2] = sp.z4;
        rc.kap = kap; rc.te = o.te1; rc.ne = o.ne1;
      }
      const Vec dr = chord(h, P.h2_6, o, kx, ky, kz, klx, kly, klz);
      Vec rn, kn;
      complete_step<kMixed>(P.h_6, o, dr, px, py, pz, kx, ky, kz, rlx, rly, rlz, klx, kly, klz, rn, kn);
      if (live) { rc.dr[0] = dr.x; rc.dr[1] = dr.y; rc.dr[2] = dr.z; }
      if constexpr (NB > 0) {
        Retrace Q;
        chord_frame(Q, P.eta, P.eps_fixed, dr);
        float c2;
        Q.lm = curvature_ln_m(sp, px, py, pz, Q.t, P.h2_6 * kf, c2);
        const bool slow = live && !(P.curv && step_clear(P.clear, sp, Q, dr) && c2 <= 1e-8f);
        Q.c1 = curvature_dt(sp, px, py, pz, Q.t);
        Q.c2 = {0.f, 0.f, 0.f};
        retrace_shared<NB>(P.G, S.f, slow, kf, h, P.h2_6, P.h2_12, px, py, pz, kx, ky, kz, Q);
        lns += Q.lm;
        if (live) {
          rc.c1[0] = Q.c1.x; rc.c1[1] = Q.c1.y; rc.c1[2] = Q.c1.z;
          rc.c2[0] = Q.c2.x; rc.c2[1] = Q.c2.y; rc.c2[2] = Q.c2.z;
          rc.lnm = Q.lm;
          rc.retraced = slow ? 1 : 0;
        }
      }
      if (live) {
        rc.sw = lns - tau;
        px = rn.x; py = rn.y; pz = rn.z;
        kx = kn.x; ky = kn.y; kz = kn.z;
      }
    }
    // the closing node of the segment: node m0 + n_s (the crossing point on a clipped last step)
    float kap_end = 0.f, te_end = 0.f, ne_end = 0.f;
    Vec p_end{px, py, pz};
    if (active) {
      const StepRec& rp = R[n_s - 1];
      if (last_seg && clipped) {
        const Vec rr{rp.r[0], rp.r[1], rp.r[2]}, dr{rp.dr[0], rp.dr[1], rp.dr[2]};
        const float a = (status == kHitInner) ? chord_crossing(rr, dr, P.G.r_min, false)
                                              : chord_crossing(rr, dr, P.G.r_max, true);
        alpha = a;
        p_end = {fmaf(a, dr.x, rr.x), fmaf(a, dr.y, rr.y), fmaf(a, dr.z, rr.z)};
      }
      const Sample s = eval_field_t<true>(P.G, p_end.x, p_end.y, p_end.z, true);
      kap_end = P.emission ? kappa_vac(s.ne, s.te, kap_c, ln_f) : 0.f;
      te_end = s.te;
      ne_end = s.ne;
      if (last_seg) {
        const float al = clipped ? alpha : 1.f;
        const float sN = __expf(rp.sw - 0.5f * (rp.kap + kap_end) * P.hrsun * al);
        float tbc = 0.f;
        if (status == kHitInner) tbc = (P.tbc_mode == 1) ? P.tbc_K : s.te;
        Wsuf = tbc * sN;  // the boundary term
        if (status == kHitInner && P.tbc_mode == 0) lte = lamT * sN;
      }
    }
    __syncthreads();

    // ------------------------------------------------ reverse the segment
    // The transfer of one segment (Eq. 2 front to back, differentiated), from
    // the values at its two nodes: the adjoints of n_e and T_e at the far node
    // are then complete (lam_ne, lam_te), those at the near one begun (lkap,
    // lte), and lLnM, lalpha are the adjoints of ln M and of the clip.
    float lam_ne = 0.f, lam_te = 0.f, lalpha = 0.f, lLnM = 0.f;
    auto transfer = [&](const StepRec& near, float kap_f, float te_f, float ne_f, float al) {
      float dkn, dkt;
      kappa_partials(ne_f, te_f, kap_c, ln_f, dkn, dkt);
      if (!P.emission) { dkn = 0.f; dkt = 0.f; }
      const float kap_sum = near.kap + kap_f;
      const float dt = 0.5f * kap_sum * P.hrsun * al;
      const float tbar = 0.5f * (near.te + te_f);
      const float qv = __expf(near.sw);
      const float om = one_minus_exp_neg(dt);
      const float W = tbar * om * qv;
      const float lDt = lamT * (tbar * __expf(-dt) * qv - Wsuf);
      const float lTbar = lamT * om * qv;
      lLnM = lamT * (W + Wsuf);
      Wsuf += W;
      const float lk_node = 0.5f * P.hrsun * al * lDt;
      lalpha = 0.5f * kap_sum * P.hrsun * lDt;
      const float lkap_f = lkap + lk_node;
      lam_ne = lkap_f * dkn;
      lam_te = lte + 0.5f * lTbar + lkap_f * dkt;
      lkap = lk_node;
      lte = 0.5f * lTbar;
    };
    // The last segment of nodes m0 + n_s - 1, m0 + n_s: the far node belongs to
    // no step of this segment, its value adjoints go alone.
    Vec lpc{0.f, 0.f, 0.f};
    if (active) {
      const bool clip = last_seg && clipped;
      transfer(R[n_s - 1], kap_end, te_end, ne_end, clip ? alpha : 1.f);
      const Vec lpos = value_adjoint(P.G, p_end.x, p_end.y, p_end.z, lam_ne, lam_te, P.dne, P.dte);
      if (clip) lpc = lpos;                                       // the crossing point closes the path
      else Lr = {Lr.x + lpos.x, Lr.y + lpos.y, Lr.z + lpos.z};    // the node's full adjoint
    }
    // Step t (node m = m0 + t): (B) the neighbours' retraces of step m, (C) the
    // central step m.  Before its node's stage the transfer of segment m - 1
    // completes the node's value adjoints, which join that stage; the segment's
    // first node waits for the segment before it.
    for (int it = 0; any(active && it < n_s); ++it) {
      const int t = n_s - 1 - it;
      const bool stepping = active && t >= 0;
      if (!__any_sync(kFull, stepping)) continue;  // a warp that waits for the block's others leaves them the SM
      const StepRec rc = R[max(t, 0)];
      const bool clip = last_seg && it == 0 && clipped;

      // tube area of step m (Eqs. 9-11, differentiated)
      const Vec rr{rc.r[0], rc.r[1], rc.r[2]}, rk{rc.k[0], rc.k[1], rc.k[2]};
      const Vec dr{rc.dr[0], rc.dr[1], rc.dr[2]};
      Vec slp{0.f, 0.f, 0.f}, slk{0.f, 0.f, 0.f};   // sums of the seed adjoints
      Vec ldr{0.f, 0.f, 0.f}, t3{0.f, 0.f, 0.f};
      float lq = 0.f;  // dL/dQ_s
      if constexpr (NB > 0) {
        const float ids = rsqrtf(dot3(dr, dr));
        t3 = {dr.x * ids, dr.y * ids, dr.z * ids};
        const bool slow = stepping && rc.retraced != 0;
        Vec lt{0.f, 0.f, 0.f};
        float lds = 0.f;
        if (stepping && !slow) {
          lq = lLnM * P.h2_6 * kf;
          lt = {lq * rc.c1[0], lq * rc.c1[1], lq * rc.c1[2]};
        }
        unsigned todo = __ballot_sync(kFull, slow);
        if (todo) {
          // (B) the neighbours' retraces: seeds r_m +- eps e_j with k = k_m; the
          // G of a "+" ("-") member enters D_j with +1 (-1)
          Vec e1, e2, le1, le2;
          basis(t3, e1, e2);
          const float eps = (P.eps_fixed > 0.f) ? P.eps_fixed : P.eta * (dot3(dr, dr) * ids);
          const float sc = P.h2_12 / eps;
          const Vec c1{rc.c1[0], rc.c1[1], rc.c1[2]}, c2{rc.c2[0], rc.c2[1], rc.c2[2]};
          const float lm1 = lLnM * __expf(-rc.lnm);  // d ln(1 + m1) / d m1 = 1 / M
          const Vec c2xt{c2.y * t3.z - c2.z * t3.y, c2.z * t3.x - c2.x * t3.z, c2.x * t3.y - c2.y * t3.x};
          const Vec txc1{t3.y * c1.z - t3.z * c1.y, t3.z * c1.x - t3.x * c1.z, t3.x * c1.y - t3.y * c1.x};
          const Vec lc1{lm1 * (e1.x + c2xt.x), lm1 * (e1.y + c2xt.y), lm1 * (e1.z + c2xt.z)};
          const Vec lc2{lm1 * (e2.x + txc1.x), lm1 * (e2.y + txc1.y), lm1 * (e2.z + txc1.z)};
          le1 = {lm1 * c1.x, lm1 * c1.y, lm1 * c1.z};
          le2 = {lm1 * c2.x, lm1 * c2.y, lm1 * c2.z};
          float leps = -(dot3(c1, lc1) + dot3(c2, lc2)) / eps;
          // one neighbour's adjoints come back: sums over the seeds, and those of the frame
          auto fold = [&](int n, const Vec& lpn, const Vec& lkn) {
            const float sn = (n & 1) ? -1.f : 1.f;
            slp = {slp.x + lpn.x, slp.y + lpn.y, slp.z + lpn.z};
            slk = {slk.x + lkn.x, slk.y + lkn.y, slk.z + lkn.z};
            leps += sn * dot3((n < 2) ? e1 : e2, lpn);
            Vec& le = (n < 2) ? le1 : le2;
            le = {fmaf(sn * eps, lpn.x, le.x), fmaf(sn * eps, lpn.y, le.y), fmaf(sn * eps, lpn.z, le.z)};
          };
          AdjointSlot* slots = S.a;
          const int q = lane & 3, group = lane >> 2;
          const float sgn = (q & 1) ? -1.f : 1.f;
          bool left = slow;
          while (todo) {
            const int rank = __popc(todo & ((1u << lane) - 1u));
            const bool mine = left && rank < kPer;
            if (mine) {
              auto& in = slots[rank].in;
              in.r[0] = rr.x; in.r[1] = rr.y; in.r[2] = rr.z;
              in.k[0] = rk.x; in.k[1] = rk.y; in.k[2] = rk.z;
              in.e1[0] = e1.x; in.e1[1] = e1.y; in.e1[2] = e1.z;
              in.e2[0] = e2.x; in.e2[1] = e2.y; in.e2[2] = e2.z;
              in.l1[0] = sc * lc1.x; in.l1[1] = sc * lc1.y; in.l1[2] = sc * lc1.z;
              in.l2[0] = sc * lc2.x; in.l2[1] = sc * lc2.y; in.l2[2] = sc * lc2.z;
              in.eps = eps;
              in.kf = kf;
              in.thread = threadIdx.x;
            }
            __syncwarp();
            // groups past the last asking lane repeat it (the lookups stay in bounds, nothing is written)
            const int asking = min(__popc(todo), kPer);
            const bool on = group < asking;
            const auto& in = slots[min(group, asking - 1)].in;
            const float* ev = (q < 2) ? in.e1 : in.e2;
            const float* lv = (q < 2) ? in.l1 : in.l2;
            const float se = sgn * in.eps, kfq = in.kf;
            const Vec base{fmaf(se, ev[0], in.r[0]), fmaf(se, ev[1], in.r[1]), fmaf(se, ev[2], in.r[2])};
            const Vec kk{in.k[0], in.k[1], in.k[2]}, lg{sgn * lv[0], sgn * lv[1], sgn * lv[2]};
            const NodeAcc<T> Aq{acc_v + in.thread, acc_key + in.thread};
            const Vec zero{0.f, 0.f, 0.f};
            Vec lp_o = zero, lk_o = zero;
            const float hh = 0.5f * h;
            const Sample s1 = eval_field_t<false>(P.G, base.x, base.y, base.z, false);
            const Vec p3{fmaf(hh, fmaf(hh, kfq * s1.gx, kk.x), base.x), fmaf(hh, fmaf(hh, kfq * s1.gy, kk.y), base.y),
                         fmaf(hh, fmaf(hh, kfq * s1.gz, kk.z), base.z)};
            rk4_reverse<3>(P.G, kfq, h, base, kk, p3, zero, zero, zero, lg, 0.f, zero, false, 0.f, 0.f, lp_o, lk_o,
                           P.dne, P.dte, Aq, on);
            __syncwarp();
            if (on) {
              float* out = slots[group].out[q];
              out[0] = lp_o.x; out[1] = lp_o.y; out[2] = lp_o.z;
              out[3] = lk_o.x; out[4] = lk_o.y; out[5] = lk_o.z;
            }
            __syncwarp();
            if (mine) {
#pragma unroll
              for (int n = 0; n < 4; ++n) {
                const float* out = slots[rank].out[n];
                fold(n, Vec{out[0], out[1], out[2]}, Vec{out[3], out[4], out[5]});
              }
              left = false;
            }
            __syncwarp();  // the slots are read: the next lanes may fill them
            todo = __ballot_sync(kFull, left);
          }
          if (slow) {
            lt = {lm1 * (c1.y * c2.z - c1.z * c2.y), lm1 * (c1.z * c2.x - c1.x * c2.z),
                  lm1 * (c1.x * c2.y - c1.y * c2.x)};
            // e2 = t x e1
            lt = {lt.x + (e1.y * le2.z - e1.z * le2.y), lt.y + (e1.z * le2.x - e1.x * le2.z),
                  lt.z + (e1.x * le2.y - e1.y * le2.x)};
            le1 = {le1.x + (le2.y * t3.z - le2.z * t3.y), le1.y + (le2.z * t3.x - le2.x * t3.z),
                   le1.z + (le2.x * t3.y - le2.y * t3.x)};
            // e1 = c / |c|, c = a x t
            const Vec av = (fabsf(t3.z) <= 0.9f) ? Vec{0.f, 0.f, 1.f} : Vec{0.f, 1.f, 0.f};
            const Vec cv{av.y * t3.z - av.z * t3.y, av.z * t3.x - av.x * t3.z, av.x * t3.y - av.y * t3.x};
            const float ic = rsqrtf(dot3(cv, cv));
            const float pe = dot3(e1, le1);
            const Vec lc{(le1.x - pe * e1.x) * ic, (le1.y - pe * e1.y) * ic, (le1.z - pe * e1.z) * ic};
            lt = {lt.x + (lc.y * av.z - lc.z * av.y), lt.y + (lc.z * av.x - lc.x * av.z),
                  lt.z + (lc.x * av.y - lc.y * av.x)};
            lds = (P.eps_fixed > 0.f) ? 0.f : P.eta * leps;  // eps = eta |dr| (Eq. 8)
          }
        }
        // t = dr / |dr| (Eq. 5)
        const float pt = dot3(t3, lt);
        ldr = {(lt.x - pt * t3.x) * ids + t3.x * lds, (lt.y - pt * t3.y) * ids + t3.y * lds,
               (lt.z - pt * t3.z) * ids + t3.z * lds};
      }

      // (C) the central step
      Vec lp_o = slp, lk_o = slk, lr_in = Lr, lk_in = Lk;
      if (clip) {
        // crossing point pc = r_m + alpha dr with |pc| = R:
        // d alpha = -(pc . (d r_m + alpha d dr)) / (pc . dr)
        const Vec pc = p_end;
        const float den = dot3(pc, dr);
        const float la = lalpha + dot3(lpc, dr);
        const float g = (den != 0.f) ? la / den : 0.f;
        lp_o = {lp_o.x + lpc.x - g * pc.x, lp_o.y + lpc.y - g * pc.y, lp_o.z + lpc.z - g * pc.z};
        ldr = {ldr.x + alpha * (lpc.x - g * pc.x), ldr.y + alpha * (lpc.y - g * pc.y),
               ldr.z + alpha * (lpc.z - g * pc.z)};
        lr_in = {0.f, 0.f, 0.f};  // the unclipped node is used only through the chord
      }
      // dr = r' - r_m
      lr_in = {lr_in.x + ldr.x, lr_in.y + ldr.y, lr_in.z + ldr.z};
      lp_o = {lp_o.x - ldr.x, lp_o.y - ldr.y, lp_o.z - ldr.z};
      const bool value = stepping && t > 0;
      if (value) transfer(R[t - 1], rc.kap, rc.te, rc.ne, 1.f);
      rk4_reverse<4>(P.G, kf, h, rr, rk, Vec{rc.p3[0], rc.p3[1], rc.p3[2]}, Vec{rc.p4[0], rc.p4[1], rc.p4[2]}, lr_in,
                     lk_in, Vec{0.f, 0.f, 0.f}, lq, t3, value, lam_ne, lam_te, lp_o, lk_o, P.dne, P.dte, A, stepping);
      if (stepping) {
        Lr = lp_o;  // node m, complete but for the value adjoints of the segment's first node
        Lk = lk_o;
      }
    }
    if (active && seg == 0) {
      // node 0 on the outer sphere: its transfer values and k0 = n(r0) (-o)
      const StepRec& r0 = R[0];
      float dkn, dkt;
      kappa_partials(r0.ne, r0.te, kap_c, ln_f, dkn, dkt);
      if (!P.emission) { dkn = 0.f; dkt = 0.f; }
      lam_ne = lkap * dkn;
      lam_te = lte + lkap * dkt;
      const Vec k0{r0.k[0], r0.k[1], r0.k[2]};
      const float n0 = sqrtf(dot3(k0, k0));
      if (n0 > 0.f) lam_ne += dot3(Lk, k0) / n0 * kn2 / (2.f * n0);
      value_adjoint(P.G, r0.r[0], r0.r[1], r0.r[2], lam_ne, lam_te, P.dne, P.dte);
    }

    // ------------------------------------------------ next segment / done
    if (active) {
      if (seg == 0) {
        acc_flush(P.G, A, P.dne, P.dte);
        active = false;
      } else {
        seg -= 1;
        if (P.ck_prev) slot = P.ck_prev[slot];
      }
    }
  }
}

}  // namespace rt
