// Derivatives of the per-record yarn BYSDF (device): the gradient of
// sum_c g_c f_c with respect to the material parameters (KB_BASIC, KB_EXT,
// KB_L2) or to the record's directions (KB_DIRS).
//
// The value is one number per record, so the lobes, the shading state and the
// aggregation of the nodes are differentiated backwards: one sweep gives the
// adjoints of the nodes' summed normal, tangent, hit point and shadowing,
// whatever the number of parameters.  In front of them stands the geometry,
// which only three scalars move: the helix angles alpha_p and alpha_f, or the
// ray's slope kappa for the directions.  It carries their tangents forwards,
// in closed form:
//   ply trace    the hit's in-plane distance t and the ply's phase psi; one
//                factor per update maps psi' to t';
//   frame        (n_p, t_p, e_p) is orthonormal, so its tangent is a
//                rotation: beta' about the yarn axis and -A' about n_p; the
//                fiber twist turns about n_p, the deviation delta about t_f;
//   shadowing    linear in (t', psi') and in the shadow ray's azimuth.
// The other parameters have closed forms in the lobe values.
//
// Against dual numbers through the whole record (two tangents; six in the
// lobes of the direction products) this leaves out the products with tangents
// that are zero and the copies of the lobes' algebra per tangent.
#pragma once

#include "bysdf_model.cuh"

namespace bysdf {

// Every product that meets a sum is written out, as a fused multiply-add or
// rounded by itself: left to the compiler, the choice depends on the code
// around it, and the derivatives of a ray that grazes its ply amplify one
// rounding of the trace without bound.
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
// a b + c d, the first product fused
__device__ __forceinline__ float mad2(float a, float b, float c, float d) {
  return fmaf(a, b, mul(c, d));
}
__device__ __forceinline__ float inv(float x) { return 1.0f / x; }
__device__ __forceinline__ float dotf(const V3<float>& a, const V3<float>& b) {
  return fmaf(a.z, b.z, mad2(a.x, b.x, a.y, b.y));
}
__device__ __forceinline__ V3<float> crossf(const V3<float>& a, const V3<float>& b) {
  return mk3<float>(mad2(a.y, b.z, -a.z, b.y), mad2(a.z, b.x, -a.x, b.z),
                    mad2(a.x, b.y, -a.y, b.x));
}
__device__ __forceinline__ V3<float> scale(const V3<float>& a, float s) {
  return mk3<float>(mul(a.x, s), mul(a.y, s), mul(a.z, s));
}
// s x + y
__device__ __forceinline__ V3<float> axpy(float s, const V3<float>& x, const V3<float>& y) {
  return mk3<float>(fmaf(s, x.x, y.x), fmaf(s, x.y, y.y), fmaf(s, x.z, y.z));
}
// a s + b t, a's products fused
__device__ __forceinline__ V3<float> comb(const V3<float>& a, float s, const V3<float>& b,
                                          float t) {
  return axpy(s, a, scale(b, t));
}
__device__ __forceinline__ V3<float> comb3(const V3<float>& a, float s, const V3<float>& b,
                                           float t, const V3<float>& c, float u) {
  return axpy(s, a, comb(b, t, c, u));
}
__device__ __forceinline__ V3<float> local(const V3<float>& w, const V3<float>& t,
                                           const V3<float>& b, const V3<float>& n) {
  return mk3<float>(dotf(w, t), dotf(w, b), dotf(w, n));
}

// Reciprocal as an instruction of its own (the compiler may join 1 / sqrt(x)
// into the reciprocal square root).
__device__ __forceinline__ float rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// 1 / sqrt(x): the parameter gradients take the reciprocal square root, the
// direction products the reciprocal of the root (one rounding apart, and each
// result as it has been).
template <bool DIRS>
__device__ __forceinline__ float inv_root(float x) {
  return DIRS ? rcp(sqrtf(x)) : rsqrtf(x);
}

// The scalars whose tangents the geometry carries: the helix angles, or the
// ray's slope (DIRS).
enum { T_ALPHA_P = 0, T_ALPHA_F = 1, T_KAPPA = 0 };
template <bool DIRS> struct GradDims {
  static constexpr int all = DIRS ? 1 : 2;
};

// The nodes of a record (Sec. 4.2): sums over the hit nodes and their
// tangents.
template <bool DIRS>
struct GeoGrad {
  static constexpr int NT = GradDims<DIRS>::all;
  V3<float> n, t;             // sums of the nodes' fiber normals and tangents
  float x, y, g;              // sums of the hit points (in plane) and of G_p G_f
  V3<float> dn[NT], dt[NT];
  float dx, dy, dg[NT];       // (alpha_f does not move the hit point)
  float dg_dsig;              // d(sum G_p G_f) / d sigma_s
  float dg_dphi;              // by the azimuth of the shadow ray (DIRS)
  int nis, nhit;
};

// A fiber map lookup (Sec. 3.5.1) with the maps' slopes in the fiber phase w.
struct FiberTap {
  float delta, of, ddelta, dof;
};
__device__ __forceinline__ FiberTap fiber_tap(const float2* map, int T, float w) {
  const float wv = w + 0.5f;
  const float a = w + (0.5f - floorf(wv));
  const float tau = fmaf(a, (float)T, -0.5f);
  const float fl = floorf(tau);
  const float f = tau - fl;
  int i0 = (int)fl;
  i0 = i0 < 0 ? i0 + T : (i0 >= T ? i0 - T : i0);
  BY_BOUNDS(i0 >= 0 && i0 < T, i0 = 0);
  const int i1 = i0 + 1 == T ? 0 : i0 + 1;
  const float2 t0 = map[i0], t1 = map[i1];
  const float sd = t1.x - t0.x, so = t1.y - t0.y;
  FiberTap r;
  r.delta = fmaf(f, sd, t0.x);
  r.of = fmaf(f, so, t0.y);
  r.ddelta = mul((float)T, sd);
  r.dof = mul((float)T, so);
  return r;
}

// Fiber migration (Sec. 3.5; migration_maps): the segment of height v + dz,
// the neighbour it blends with, the neighbour's weight (0 outside the blend
// zones) and the weight's slope in the segment fraction.
struct MigSpot {
  int seg, nb;
  float wgt, slope;
};
__device__ __forceinline__ MigSpot migration_spot(const MatDev& m, float v, float dz) {
  const MigMap* m1 = mig_map(m, 1);
  const float ph = mul(v, m.mig_inv_len);
  const float pe = fmaf(v, m1->aux, fmaf(v, m.mig_inv_len, -ph));
  float nf = floorf(ph);
  float t = fmaf(dz, m.mig_inv_len, (ph - nf) + pe);
  const float kf2 = floorf(t);
  t = t - kf2;
  nf += kf2;
  MigSpot r;
  r.seg = (int)(((int64_t)nf % kMigPeriod + kMigPeriod) % kMigPeriod);
  r.nb = r.seg;
  r.wgt = r.slope = 0.f;
  if (t < m.mig_blend) {
    r.wgt = fmaf(-t, m.mig_inv_2b, 0.5f);
    r.slope = -m.mig_inv_2b;
    r.nb = r.seg == 0 ? kMigPeriod - 1 : r.seg - 1;
  } else if (t > 1.0f - m.mig_blend) {
    r.wgt = fmaf(t - 1.0f, m.mig_inv_2b, 0.5f);
    r.slope = m.mig_inv_2b;
    r.nb = r.seg == kMigPeriod - 1 ? 0 : r.seg + 1;
  }
  BY_BOUNDS(r.seg >= 0 && r.seg < kMigPeriod, r.seg = 0);
  BY_BOUNDS(r.nb >= 0 && r.nb < kMigPeriod, r.nb = 0);
  return r;
}

// delta and o_f of a migrating ply (Sec. 3.5) and their derivatives by the
// ply azimuth u, the height z of the hit and alpha_f.
struct FiberGrad {
  float delta, of;
  float d_u, d_z, d_af;  // of delta
  float o_u, o_z, o_af;  // of o_f
};
__device__ __forceinline__ void fiber_of_map(const MatDev& m, const float2* map0, int k,
                                             float u_ply, float v, float dz, float w0,
                                             FiberGrad& r) {
  const float2* mp = map0;
  float mu = m.m_over_2pi, kf = m.kf_hi + m.kf_lo, dkf = m.dkf, w = w0;
  if (k != 0) {
    const MigMap* mk = mig_map(m, k);
    mp = reinterpret_cast<const float2*>(mk + 1);
    mu = mk->m_over_2pi;
    kf = mk->kf_hi + mk->kf_lo;
    dkf = mk->dkf;
    w = fmaf(-kf, dz, fmaf(u_ply, mu, -frac_prod(mk->kf_hi, mk->kf_lo, v)));
  }
  const FiberTap f = fiber_tap(mp, m.T, w);
  const float waf = mul(-dkf, v + dz);
  r.delta = f.delta;
  r.of = f.of;
  r.d_u = mul(f.ddelta, mu);
  r.d_z = mul(-f.ddelta, kf);
  r.d_af = mul(f.ddelta, waf);
  r.o_u = mul(f.dof, mu);
  r.o_z = mul(-f.dof, kf);
  r.o_af = mul(f.dof, waf);
}
__device__ __forceinline__ void fiber_grad(const MatDev& m, const float2* map0, float u_ply,
                                           float v, float dz, float w0, FiberGrad& r) {
  if (m.mig_maps <= 1) {
    fiber_of_map(m, map0, 0, u_ply, v, dz, w0, r);
    return;
  }
  const MigSpot sp = migration_spot(m, v, dz);
  const uint8_t* tab = mig_table(m);
  int k0 = tab[sp.seg], k1 = tab[sp.nb];
  BY_BOUNDS(k0 < m.mig_maps, k0 = 0);
  BY_BOUNDS(k1 < m.mig_maps, k1 = 0);
  fiber_of_map(m, map0, k0, u_ply, v, dz, w0, r);
  if (!(sp.wgt > 0.f)) return;
  FiberGrad q;
  fiber_of_map(m, map0, k1, u_ply, v, dz, w0, q);
  const float wz = mul(sp.slope, m.mig_inv_len);
  const float ed = q.delta - r.delta, eo = q.of - r.of;
  r.d_z = fmaf(wz, ed, fmaf(sp.wgt, q.d_z - r.d_z, r.d_z));
  r.o_z = fmaf(wz, eo, fmaf(sp.wgt, q.o_z - r.o_z, r.o_z));
  r.d_u = fmaf(sp.wgt, q.d_u - r.d_u, r.d_u);
  r.o_u = fmaf(sp.wgt, q.o_u - r.o_u, r.o_u);
  r.d_af = fmaf(sp.wgt, q.d_af - r.d_af, r.d_af);
  r.o_af = fmaf(sp.wgt, q.o_af - r.o_af, r.o_af);
  r.delta = fmaf(sp.wgt, ed, r.delta);
  r.of = fmaf(sp.wgt, eo, r.of);
}

// One node of the ray on its closest ply (picked by the float trace), with
// tangents, added to the record's sums.  The trace runs all N_it updates, the
// last one with sincospif; a ray that grazes the ply within rounding has no
// derivative there and the node is dropped.
template <bool DIRS>
__device__ __forceinline__ void node_grad(const MatDev& m, const float2* map, float X0x,
                                          float X0y, float ex, float ey, float v, float kappa,
                                          float wx, float wy, float s0v, float c0v,
                                          float phase_f_v, int ply, int ni, GeoGrad<DIRS>& G) {
  const float Rp = m.Rp, Rc = m.Rc;
  const float kp = m.kp_hi + m.kp_lo, kf = m.kf_hi + m.kf_lo;
  const float ck = mad2(c0v, m.rot_c[ply], -s0v, m.rot_s[ply]);
  const float sk = mad2(s0v, m.rot_c[ply], c0v, m.rot_s[ply]);
  const float w2kp = mul(2.0f * kPi, kp), w2dkp = mul(2.0f * kPi, m.dkp);
  const int n_upd = m.nit;
  float t = 0.f, cx = 0.f, cy = 0.f, s = 0.f, c = 1.f;
  float t1 = 0.f, p1 = 0.f;  // t', psi' by alpha_p, or by kappa (DIRS)
  bool grazed = false;
#pragma unroll 1
  for (int i = 0; i < n_upd; ++i) {
    float sd, cd;
    const float turns = mul(kp, mul(t, kappa));
    if (i + 1 < n_upd) {
      xsincos_turns_fast(turns, &sd, &cd);
    } else {
      xsincos_turns(turns, &sd, &cd);
    }
    // psi = 2 pi kp (v + kappa t)
    p1 = DIRS ? mul(w2kp, fmaf(kappa, t1, t))
              : mad2(mul(w2kp, kappa), t1, w2dkp, fmaf(kappa, t, v));
    c = mad2(ck, cd, -sk, sd);
    s = mad2(sk, cd, ck, sd);
    cx = mul(c, Rc);
    cy = mul(s, Rc);
    const float qx = X0x - cx, qy = X0y - cy;
    const float b = mad2(qy, ey, qx, ex);
    const float perp = mad2(-qy, ex, qx, ey);
    const float disc = mul(Rp - perp, Rp + perp);
    grazed = grazed || !(disc > 0.f);
    const float sq = sqrtf(xmax0(disc));
    const float tn = -b - sq;
    t = xmax0(tn);
    // b' = R_c psi' (s e_x - c e_y), perp' = R_c psi' (s e_y + c e_x)
    const float e1 = mad2(s, ex, -c, ey), e2 = mad2(s, ey, c, ex);
    const float gain = tn < 0.f ? 0.f : mul(Rc, fmaf(mul(perp, inv(sq)), e2, -e1));
    t1 = mul(gain, p1);
  }
  if (grazed) return;
  const float xx = fmaf(t, ex, X0x), xy = fmaf(t, ey, X0y);
  const float dz = mul(t, kappa);
  const float dx = xx - cx, dy = xy - cy;
  const float inv_dl = rsqrtf(mad2(dx, dx, dy, dy));
  const V3<float> np = mk3<float>(mul(dx, inv_dl), mul(dy, inv_dl), 0.f);
  const float wp = mul(kp, 2.0f * kPi);
  const V3<float> traw = mk3<float>(-mul(wp, xy), mul(wp, xx), 1.f);
  const float tn = mad2(traw.x, np.x, traw.y, np.y);
  const V3<float> tv = axpy(-tn, np, traw);
  const float il = rsqrtf(dotf(tv, tv));
  const V3<float> tp = scale(tv, il);
  const V3<float> ep = crossf(tp, np);
  const float u_ply = xatan2(mad2(c, np.y, -s, np.x), mad2(c, np.x, s, np.y));
  const float w = fmaf(-kf, dz, fmaf(u_ply, m.m_over_2pi, -phase_f_v));
  FiberGrad fg;
  fiber_grad(m, map, u_ply, v, dz, w, fg);
  const V3<float> tf = comb(tp, m.cos_af, ep, m.sin_af);
  float sd, cd;
  xsincos(fg.delta, &sd, &cd);
  const V3<float> ef = crossf(tf, np);
  const V3<float> nf = comb(np, cd, ef, sd);
  // shadowing: occ = sum of chords; occ' = at t' + ap psi' (and aph per
  // radian of the shadow ray's azimuth)
  float occ = 0.f, at = 0.f, ap = 0.f, aph = 0.f;
  const float eb = mad2(ex, wx, ey, wy), epp = mad2(ex, wy, -ey, wx);
#pragma unroll 1
  for (int j = 1; j < m.np; ++j) {
    const float rc = m.rot_c[j], rs = m.rot_s[j];
    const float cjx = mad2(cx, rc, -cy, rs);
    const float cjy = DIRS ? mad2(cx, rs, cy, rc) : mad2(cy, rc, cx, rs);
    const float qx = xx - cjx, qy = xy - cjy;
    const float b = mad2(qx, wx, qy, wy);
    const float perp = mad2(qx, wy, -qy, wx);
    const float disc = mul(Rp - perp, Rp + perp);
    if (disc > 0.f) {
      const float sq = sqrtf(disc);
      const float s2 = sq - b;
      if (s2 > 0.f) {
        const float s1 = -b - sq;
        const bool whole = !(s1 < 0.f);  // the whole chord lies ahead
        occ = occ + (s2 - xmax0(s1));
        const float cb = whole ? 0.f : -1.f;
        const float cp = mul(mul(whole ? -2.f : -1.f, perp), inv(sq));
        at += mad2(cb, eb, cp, epp);
        ap += mad2(cb, mad2(cjy, wx, -cjx, wy), cp, mad2(cjy, wy, cjx, wx));
        if (DIRS) aph += mad2(cp, b, -cb, perp);
      }
    }
  }
  const float occ_all = fmaf(occ, m.inv_2Rp, fg.of);
  const float g = xexp(-mul(occ_all, m.sigma_s));
  const float gs = mul(-g, m.sigma_s);
  // values
  G.nhit += 1;
  G.nis += ni;
  G.n = G.n + nf;
  G.t = G.t + tf;
  G.x += xx;
  G.y += xy;
  G.g += g;
  G.dg_dsig = fmaf(-occ_all, g, G.dg_dsig);
  if (DIRS) G.dg_dphi = fmaf(mul(gs, m.inv_2Rp), aph, G.dg_dphi);
  // tangents: the frame turns by beta' about the axis and -A' about n_p, the
  // normal also by delta' about t_f
  const V3<float> md = comb(ef, cd, np, -sd);
  const float xn = mad2(xx, np.x, xy, np.y), en = mad2(ex, np.x, ey, np.y);
  // n_p' = beta' (-n_y, n_x), from the hit and the ply centre
  const float ddx = mad2(t1, ex, cy, p1), ddy = mad2(t1, ey, -cx, p1);
  const float be = mul(mad2(np.x, ddy, -np.y, ddx), inv_dl);
  // tan A = in-plane part of the helix direction across n_p
  const float q0 = mul(mul(wp, t1), en);
  const float q1 = fmaf(-be, tn, DIRS ? q0 : fmaf(w2dkp, xn, q0));
  const float A = mul(mul(q1, il), il);
  const float u1 = be - p1, z1 = DIRS ? fmaf(kappa, t1, t) : mul(kappa, t1);
  const float d1 = mad2(fg.d_u, u1, fg.d_z, z1), o1 = mad2(fg.o_u, u1, fg.o_z, z1);
  const V3<float> om = mk3<float>(mul(-A, np.x), mul(-A, np.y), be);
  G.dt[0] = G.dt[0] + crossf(om, tf);
  G.dn[0] = G.dn[0] + axpy(d1, md, crossf(om, nf));
  G.dx = fmaf(t1, ex, G.dx);
  G.dy = fmaf(t1, ey, G.dy);
  G.dg[0] = fmaf(gs, fmaf(mad2(at, t1, ap, p1), m.inv_2Rp, o1), G.dg[0]);
  if constexpr (!DIRS) {
    G.dt[T_ALPHA_F] = G.dt[T_ALPHA_F] + ef;
    G.dn[T_ALPHA_F] = axpy(fg.d_af, md, axpy(-sd, tf, G.dn[T_ALPHA_F]));
    G.dg[T_ALPHA_F] = fmaf(gs, fg.o_af, G.dg[T_ALPHA_F]);
  }
}

// The record's ray in the yarn frame.
struct RayGrad {
  float kappa, wx, wy, inv_l, width;
};

// All nodes of a record; false where no node hits.
template <bool DIRS>
__device__ __forceinline__ bool geometry_grad(const MatDev& m, const float2* map,
                                              const Record& q, RayGrad& r, GeoGrad<DIRS>& G) {
  const Footprint fp = footprint(q.h, q.ratio, m.kmax);
  r.width = fp.width;
  float sU, cU;
  sincosf(q.u, &sU, &cU);
  const float ch = sqrtf(fmaxf(0.f, fmaf(-q.h, q.h, 1.0f)));
  const float su = mad2(sU, ch, -cU, q.h), cu = mad2(cU, ch, sU, q.h);
  const float ex = -cu, ey = -su;
  const float l2 = mad2(q.wi[0], q.wi[0], q.wi[1], q.wi[1]);
  if (!(sqrtf(l2) >= 1e-7f)) return false;
  r.inv_l = inv_root<DIRS>(l2);
  r.kappa = mul(-q.wi[2], r.inv_l);
  r.wx = mul(q.wi[0], r.inv_l);
  r.wy = mul(q.wi[1], r.inv_l);
  float s0v, c0v;
  xsincos_turns(frac_prod(m.kp_hi, m.kp_lo, q.v), &s0v, &c0v);
  const float phase_f_v = frac_prod(m.kf_hi, m.kf_lo, q.v);
  G.n = G.t = mk3<float>(0.f, 0.f, 0.f);
  G.x = G.y = G.g = G.dx = G.dy = G.dg_dsig = G.dg_dphi = 0.f;
  G.nis = G.nhit = 0;
#pragma unroll
  for (int k = 0; k < GradDims<DIRS>::all; ++k) {
    G.dn[k] = G.dt[k] = mk3<float>(0.f, 0.f, 0.f);
    G.dg[k] = 0.f;
  }
  const MatVars mv = mat_vars(m);
  const bool near = fp.K == 1 && fp.width == 0.0f;
#pragma unroll 1
  for (int j = 0; j < fp.K; ++j) {
    float X0x, X0y;
    if (near) {
      X0x = cU;
      X0y = sU;
    } else {
      const float hj = fp.h1 + mul((float)j + 0.5f, fp.width) / (float)fp.K;
      const float cj = sqrtf(fmaxf(0.f, fmaf(-hj, hj, 1.0f)));
      X0x = mad2(cu, cj, -su, hj);
      X0y = mad2(su, cj, cu, hj);
    }
    X0x = mul(X0x, m.R);
    X0y = mul(X0y, m.R);
    // derivatives follow the branch the values take: a float pass over all
    // plies (one per pass: fewer live registers) picks the closest and N_i
    NodeGeo pick;
    node_geometry<1>(m, map, mv, X0x, X0y, ex, ey, q.v, r.kappa, r.wx, r.wy, s0v, c0v, phase_f_v,
                     pick, true);
    if (!pick.hit) continue;
    node_grad<DIRS>(m, map, X0x, X0y, ex, ey, q.v, r.kappa, r.wx, r.wy, s0v, c0v, phase_f_v,
                    pick.ply, pick.ni, G);
  }
  return G.nhit != 0;
}

// Fresnel reflectance at cosine ci >= 0 and its derivative.
__device__ __forceinline__ float fresnel_grad(float ci, float eta, float* dF) {
  const float ie2 = 1.0f / (eta * eta);
  const float s2t = mul(fmaf(-ci, ci, 1.0f), ie2);
  *dF = 0.f;
  if (!(s2t < 1.0f)) return 1.f;
  const float ct = sqrtf(1.0f - s2t);
  const float dct = mul(mul(ci, ie2), inv(ct));
  const float is = inv(fmaf(ct, eta, ci)), ip = inv(fmaf(ci, eta, ct));
  const float rs = mul(fmaf(-ct, eta, ci), is), rp = mul(fmaf(ci, eta, -ct), ip);
  const float ed = mul(eta, dct);
  const float ds = mul(fmaf(-rs, 1.0f + ed, 1.0f - ed), is);
  const float dp = mul(fmaf(-rp, eta + dct, eta - dct), ip);
  *dF = mad2(rs, ds, rp, dp);
  return mul(0.5f, mad2(rs, rs, rp, rp));
}

// Smith G1 terms of a direction in the microfacet frame: r as in G1 = 2 an /
// (an + r), and d ln G1 by the local components (z: of G1 / |w.z| when
// over_cos) and by the roughness.
struct G1Grad {
  float an, r;
  V3<float> d;
  float dat, dab;
};
__device__ __forceinline__ G1Grad g1_grad(const V3<float>& w, float at, float ab, bool over_cos) {
  G1Grad g;
  g.an = w.z < 0.f ? -w.z : w.z;
  const float ax = mul(w.x, at), ay = mul(w.y, ab);
  g.r = sqrtf(fmaf(ay, ay, mad2(g.an, g.an, ax, ax)));
  const float ir = inv(g.r);
  const float k = mul(ir, inv(g.an + g.r));
  g.dat = mul(mul(-ax, w.x), k);
  g.dab = mul(mul(-ay, w.y), k);
  float dz = -ir;
  if (!over_cos) dz += inv(g.an);
  g.d = mk3<float>(mul(mul(-at, ax), k), mul(mul(-ab, ay), k), w.z < 0.f ? -dz : dz);
  return g;
}

// Gradient columns: the 8 of the basic set, or the 15 of the extended set;
// KB_L2 also takes the upstream gradient from an L2 loss against target
// radiance, whose value is a ninth column.  KB_DIRS has the direction
// products instead.
enum { KB_BASIC = 0, KB_EXT = 1, KB_L2 = 2, KB_DIRS = 3 };
template <int KIND> struct KbCols {
  static constexpr int grad = KIND == KB_EXT ? 15 : 8;            // gradient columns
  static constexpr int acc = KIND == KB_L2 ? 9 : grad;             // accumulated columns
};

// Gradient of sum_c g_c f_c of one record.  upstream(f, g): g_c from the
// record's f_c (KB_L2 returns the loss, else 0).  gout: the columns
// accumulated per material ([0..2] moves both body colours in the basic
// set), or for KB_DIRS the six products with omega_i and omega_o.
template <int KIND, class Up>
__device__ __forceinline__ void record_grad(const MatDev& m, const float2* map, const Record& q,
                                            Up&& upstream, float* gout) {
  constexpr bool EXT = KIND == KB_EXT, DIRS = KIND == KB_DIRS;
  constexpr int NT = GradDims<DIRS>::all;
  RayGrad ray;
  GeoGrad<DIRS> G;
  if (!geometry_grad<DIRS>(m, map, q, ray, G)) return;
  const V3<float> wi = mk3<float>(q.wi[0], q.wi[1], q.wi[2]);
  const V3<float> wo = mk3<float>(q.wo[0], q.wo[1], q.wo[2]);
  // aggregation (Eqs. 9-11): n = ns / |ns|, t orthogonalised against it
  const float inv_hit = 1.0f / (float)G.nhit;
  const float nn = dotf(G.n, G.n);
  if (!(sqrtf(nn) > 1e-9f * (float)G.nhit)) return;
  const float inl = inv_root<DIRS>(nn);
  const V3<float> ng = scale(G.n, inl);
  const float tn = dotf(G.t, ng);
  const V3<float> tperp = axpy(-tn, ng, G.t);
  const float tt2 = dotf(tperp, tperp);
  if (!(sqrtf(tt2) > 1e-9f * (float)G.nhit)) return;
  const float itl = inv_root<DIRS>(tt2);
  const V3<float> t = scale(tperp, itl);
  const float px = mul(G.x, inv_hit), py = mul(G.y, inv_hit);
  const float g = mul(G.g, inv_hit);
  const float ni = mul((float)G.nis, inv_hit);
  // shading state (two-sided)
  V3<float> n = ng, b = crossf(ng, t);
  const bool flip = dotf(wi, n) < 0.f;
  if (flip) {
    n = -n;
    b = -b;
  }
  const float mui = dotf(wi, n), muo = dotf(wo, n);
  const float hw = 0.5f * ray.width;
  const float at = clamp_alpha(m.beta_t + hw), ab = clamp_alpha(m.beta_b + hw);
  const bool at_free = at == m.beta_t + hw, ab_free = ab == m.beta_b + hw;
  const bool refl = muo > 0.f;
  float dfr;
  const float fr = fresnel_grad(mui, m.eta, &dfr);
  // body lobe (Eqs. 5-6) per unit (r B) or ((1 - r) B), with its derivatives
  // by mu_i and mu_o
  float body_w = 0.f, bw_i = 0.f, bw_o = 0.f;
  const bool lit = mui > 0.f && (refl || muo < 0.f);
  if (lit) {
    if (refl) {
      const float lg = xlog(1.0f + inv(mui));
      const float ia = inv(fmaf(0.5f, fmaf(-mui, lg, 1.0f), 1.0f));
      const float x0 = mul(g, ia);
      const float iss = inv(mui + muo);
      const float ls = 1.0f / (4.0f * kPi);
      const float xb = mul(x0, fmaf(ls, iss, 1.0f / kPi));
      const float xs = mul(mul(mul(x0, mul(ls, iss)), iss), muo);
      body_w = mul(xb, muo);
      bw_o = xb - xs;
      // a'(mu) = -(ln(1 + 1/mu) - 1/(1 + mu)) / 2
      bw_i = fmaf(mul(body_w, 0.5f), mul(lg - inv(1.0f + mui), ia), -xs);
    } else {
      bw_o = -mul(g, 1.0f / kPi);
      body_w = mul(bw_o, muo);
    }
  }
  const float body_k = refl ? mul(m.r, m.B) : mul(1.0f - m.r, m.B);
  const float body = mul(body_k, body_w);
  // transmission path: smooth refraction at x, straight to y (Eq. 3 / 4)
  const float ie = m.inv_eta;
  V3<float> iy = mk3<float>(0.f, 0.f, 0.f);
  float nyx = 1.f, nyy = 0.f, sy = 0.f, s_y = 1.f, il_y = 1.f, kref = 0.f, dkref = 0.f;
  float tau = 0.f, tx = 0.f;
  bool tt = false, sy_free = false;
  const float s2t = mul(fmaf(-mui, mui, 1.0f), mul(ie, ie));
  if (lit && !refl && s2t < 1.0f) {
    const float ct = sqrtf(1.0f - s2t);
    kref = fmaf(mui, ie, -ct);
    dkref = fmaf(-mui, mul(mul(ie, ie), inv(ct)), ie);
    V3<float> din = comb(wi, -ie, n, kref);
    if (DIRS) {
      din.x = fmaf(n.x, kref, mul(wi.x, -ie));
      din.y = fmaf(n.y, kref, mul(wi.y, -ie));
    }
    const float a = mad2(din.x, din.x, din.y, din.y);
    if (a > 1e-12f) {
      const float bq = mad2(px, din.x, py, din.y);
      const float c = fmaf(-m.R, m.R, mad2(px, px, py, py));
      const float disc = xmax0(mad2(bq, bq, -a, c));
      s_y = sqrtf(disc);
      const float raw = mul(s_y - bq, inv(a));
      sy = xmax0(raw);
      sy_free = !(raw < 0.f) && disc > 0.f;
      const float yx = fmaf(din.x, sy, px), yy = fmaf(din.y, sy, py);
      il_y = rsqrtf(mad2(yx, yx, yy, yy));
      nyx = mul(yx, il_y);
      nyy = mul(yy, il_y);
      iy = -din;
      tau = xexp(-mul(mul(ni, m.sigma_t), sy));
      tx = 1.0f - fr;
      tt = true;
    }
  }
  // the microfacet lobe that applies to omega_o (Eq. 2 at x, Eq. 3 at y), in
  // its frame: D at the half vector, G1 of both directions, Fresnel
  const V3<float> fz = mk3<float>(0.f, 0.f, 1.f);
  const V3<float> ny = mk3<float>(nyx, nyy, 0.f);
  const V3<float> fn = vsel(refl, n, ny);
  const V3<float> ft = vsel(refl, t, fz);
  const V3<float> fb = vsel(refl, b, mk3<float>(nyy, -nyx, 0.f));
  const V3<float> vi = vsel(refl, wi, iy);
  float spec = 0.f, spec_u = 0.f, dln_at = 0.f, dln_ab = 0.f;
  V3<float> h = fz, lh = fz, li = fz, lo = fz;
  float h_il = 0.f, h_sg = 1.f, ih = 0.f, oh = 0.f, k_ih = 0.f, k_oh = 0.f;
  float u_tx = 0.f, u_ih = 0.f;  // by tx; F's own share by i.h
  bool on = lit && (refl || (tt && dotf(iy, ny) < 0.f && dotf(wo, ny) > 0.f));
  if (on) {
    const V3<float> hv = refl ? wi + wo : -axpy(m.eta, iy, wo);
    h_il = rsqrtf(dotf(hv, hv));
    h = scale(hv, h_il);
    if (dotf(h, fn) < 0.f) {
      h = -h;
      h_sg = -1.f;
    }
    ih = dotf(vi, h);
    oh = dotf(wo, h);
    on = refl || (ih < 0.f && oh > 0.f);
  }
  if (on) {
    const V3<float> hl = local(h, ft, fb, fn), il = local(vi, ft, fb, fn),
                    ol = local(wo, ft, fb, fn);
    const float iat = 1.0f / at, iab = 1.0f / ab;
    const float mx = mul(hl.x, iat), my = mul(hl.y, iab);
    const float qd = fmaf(hl.z, hl.z, mad2(mx, mx, my, my));
    const float D = hl.z > 0.f ? mul(1.0f / kPi, inv(mul(mul(qd, mul(at, ab)), qd))) : 0.f;
    const G1Grad gi = g1_grad(il, at, ab, true), go = g1_grad(ol, at, ab, false);
    const float g1i = mul(ih, il.z) > 0.f ? mul(2.0f, inv(gi.an + gi.r)) : 0.f;
    const float g1o = mul(oh, ol.z) > 0.f ? mul(mul(go.an, 2.0f), inv(go.an + go.r)) : 0.f;
    float dF;
    const float F = fresnel_grad(refl ? ih : -ih, refl ? m.eta : ie, &dF);
    if (refl) {
      const float qq = mul(mul(g1i, D), 0.25f);
      spec_u = mul(mul(F, g1o), qq);
      u_ih = mul(mul(g1o, qq), dF);
    } else {
      const float den = fmaf(ih, m.eta, oh);
      const float iden = inv(den);
      const float qq = mul(mul(mul(mul(g1i, -ih), D), oh), mul(iden, iden));
      const float gq = mul(g1o, mul(tau, qq));
      u_tx = mul(1.0f - F, gq);
      spec_u = mul(tx, u_tx);
      u_ih = mul(mul(tx, dF), gq);
      k_ih = fmaf(mul(-2.0f, m.eta), iden, inv(ih));
      k_oh = fmaf(-2.0f, iden, inv(oh));
    }
    on = spec_u != 0.f;
    spec = mul(m.ks, spec_u);
    if (on) {
      const float q4 = mul(4.0f, inv(qd));
      lh = mk3<float>(-mul(mul(q4, mx), iat), -mul(mul(q4, my), iab), -mul(q4, hl.z));
      li = gi.d;
      lo = go.d;
      dln_at = fmaf(mul(mul(q4, mx), mx), iat, -iat) + gi.dat + go.dat;
      dln_ab = fmaf(mul(mul(q4, my), my), iab, -iab) + gi.dab + go.dab;
    }
  }
  // f_c = spec + k^B_c body, with k^B = k^B_x (reflection side) or k^B_y
  const bool rf = refl || !lit;
  const float* kb = rf ? m.alb : m.alb_y;
  float fc[3], gc[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) fc[c] = fmaf(kb[c], body, spec);
  const float loss = upstream(fc, gc);
  if (KIND == KB_L2) gout[8] = loss;
  const float gs = gc[0] + gc[1] + gc[2];
  const float gb = fmaf(gc[2], kb[2], mad2(gc[0], kb[0], gc[1], kb[1]));
  const float ig = g > 0.f ? inv(g) : 0.f;
  if constexpr (!DIRS) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float v = mul(gc[c], body);
      gout[c] = EXT && !rf ? 0.f : v;
      if constexpr (EXT) gout[9 + c] = rf ? 0.f : v;
    }
    // roughness: d spec / d beta = spec d ln spec / d alpha, unless clamped
    gout[3] = at_free ? mul(mul(gs, spec), dln_at) : 0.f;
    gout[4] = ab_free ? mul(mul(gs, spec), dln_ab) : 0.f;
    // shadow density: the body lobes are proportional to G
    gout[7] = mul(mul(gb, body), mul(mul(G.dg_dsig, inv_hit), ig));
    if constexpr (EXT) {
      // body = r B body_w (reflection side) or (1 - r) B body_w; spec = (1 - B)
      // k_spec spec_u; the transmission lobe carries tau = exp(-sigma_t N_i
      // |x - y|) (Eq. 4)
      gout[8] = mul(mul(gb, rf ? m.B : -m.B), body_w);
      gout[12] = rf ? 0.f : mul(mul(gs, spec), -mul(ni, sy));
      gout[13] = mad2(mul(gb, rf ? m.r : 1.0f - m.r), body_w, mul(-gs, m.k_spec), spec_u);
      gout[14] = mul(mul(gs, 1.0f - m.B), spec_u);
    }
  }
  if (!lit) return;
  // ---- reverse sweep: adjoints of n, t, b, the hit point, G and mu_i ----
  const float gbk = mul(gb, body_k);
  float a_mui = mul(gbk, bw_i);
  const float a_muo = mul(gbk, bw_o);
  const float a_g = mul(mul(gbk, body_w), ig);
  const V3<float> zero = mk3<float>(0.f, 0.f, 0.f);
  V3<float> a_n = scale(wo, a_muo), a_t = zero, a_b = zero, a_wi = zero, a_wo = zero;
  if (DIRS) a_wo = scale(n, a_muo);
  float a_px = 0.f, a_py = 0.f;
  if (on) {
    const float S = mul(gs, spec), kS = mul(gs, m.ks);
    const float a_ih = mad2(S, k_ih, kS, u_ih), a_oh = mul(S, k_oh);
    lh = scale(lh, S);
    li = scale(li, S);
    lo = scale(lo, S);
    V3<float> a_fn = comb3(h, lh.z, vi, li.z, wo, lo.z);
    const V3<float> a_fb = comb3(h, lh.y, vi, li.y, wo, lo.y);
    V3<float> a_vi = comb3(ft, li.x, fb, li.y, fn, li.z);
    V3<float> a_v = zero;
    if (DIRS || !refl) {
      const V3<float> a_h =
          axpy(a_oh, wo, axpy(a_ih, vi, comb3(ft, lh.x, fb, lh.y, fn, lh.z)));
      a_v = scale(axpy(-dotf(h, a_h), h, a_h), mul(h_il, h_sg));
      a_vi = axpy(a_ih, h, a_vi);
    }
    if (DIRS) {
      const V3<float> a_ol = axpy(a_oh, h, comb3(ft, lo.x, fb, lo.y, fn, lo.z));
      a_wo = a_wo + a_ol + (refl ? a_v : -a_v);
    }
    if (refl) {
      a_n = a_n + a_fn;
      a_b = a_fb;
      a_t = comb3(h, lh.x, vi, li.x, wo, lo.x);
      if (DIRS) a_wi = a_vi + a_v;
    } else {
      // through the exit point y = x + s_y d and the refraction d
      V3<float> a_din = -axpy(-m.eta, a_v, a_vi);
      // b_y = (n_y, -n_x); only the part across n_y moves the unit normal
      a_fn.x -= a_fb.y;
      a_fn.y += a_fb.x;
      const float ac = mul(mad2(a_fn.y, nyx, -a_fn.x, nyy), il_y);
      a_px = mul(-nyy, ac);
      a_py = mul(nyx, ac);
      a_din.x = fmaf(sy, a_px, a_din.x);
      a_din.y = fmaf(sy, a_py, a_din.y);
      if (sy_free) {
        // |x + s_y d| = R: d s_y = -(y . dx + s_y y . dd) / (y . d), with
        // y . d = sqrt(disc)
        const float a_sy = fmaf(mul(-m.sigma_t, ni), S, -mad2(a_px, iy.x, a_py, iy.y));
        const float k = mul(mul(-a_sy, inv(s_y)), inv(il_y));
        a_px = fmaf(k, nyx, a_px);
        a_py = fmaf(k, nyy, a_py);
        a_din.x = fmaf(mul(k, sy), nyx, a_din.x);
        a_din.y = fmaf(mul(k, sy), nyy, a_din.y);
      }
      if (DIRS) a_wi = scale(a_din, -ie);
      a_n = axpy(kref, a_din, a_n);
      a_mui += mad2(dkref, dotf(a_din, n), mul(-dfr, kS), u_tx);
    }
  }
  a_n = axpy(a_mui, wi, a_n);
  if (DIRS) a_wi = axpy(a_mui, n, a_wi);
  // b = n x t; then the two-sided flip, t's orthogonalisation, the norms
  if (flip) {
    a_n = -a_n;
    a_b = -a_b;
  }
  a_n = a_n + crossf(t, a_b);
  a_t = a_t + crossf(a_b, ng);
  const V3<float> a_tp = scale(axpy(-dotf(t, a_t), t, a_t), itl);
  const float nt = dotf(ng, a_tp);
  a_n = axpy(-nt, G.t, axpy(-tn, a_tp, a_n));
  const V3<float> a_ts = axpy(-nt, ng, a_tp);
  const V3<float> a_ns = scale(axpy(-dotf(ng, a_n), ng, a_n), inl);
  const float hx = mul(a_px, inv_hit), hy = mul(a_py, inv_hit), hg = mul(a_g, inv_hit);
  float d[NT];
#pragma unroll
  for (int k = 0; k < NT; ++k)
    d[k] = fmaf(hg, G.dg[k], dotf(a_ts, G.dt[k])) + dotf(a_ns, G.dn[k]);
  d[0] += mad2(hx, G.dx, hy, G.dy);
  if constexpr (DIRS) {
    // kappa = -w_z / l and the shadow ray's azimuth of (w_x, w_y) / l
    const float dk = mul(d[T_KAPPA], ray.inv_l), dp = mul(mul(hg, G.dg_dphi), ray.inv_l);
    const float dkk = mul(dk, ray.kappa);
    gout[0] = a_wi.x - mad2(dkk, ray.wx, dp, ray.wy);
    gout[1] = a_wi.y - mad2(dkk, ray.wy, -dp, ray.wx);
    gout[2] = a_wi.z - dk;
    gout[3] = a_wo.x;
    gout[4] = a_wo.y;
    gout[5] = a_wo.z;
  } else {
    gout[5] = d[T_ALPHA_P];
    gout[6] = d[T_ALPHA_F];
  }
}

}  // namespace bysdf
