// nyx_pair32.cuh -- the FP32 arithmetic of the task form (nyx_fused2.cuh),
// on pairs of values: f32x2 instructions add, multiply and fuse two floats in
// one issue slot.  A face's solve keeps its left and right states as a pair; a
// trace pairs (rho, p) and the two tangential velocities.  Selections, minima
// and the special functions have no pair form and stay per value, and so do
// products with a constant (a constant pair costs two moves).  216 boxes of
// 32^3, per advance: 3.45 ms with every operation on single values, 3.32 ms
// with pairs.
//
// The scheme is that of nyx_scheme.cuh (PPM or PLM profiles, characteristic
// tracing with a reference state, corner coupling, two-shock solver), with
// the profiles written as deviations from the cell value,
//   a = s_i - s_L,  b = s_R - s_i,  w = b - a  (w = s_6 / -3),
// in which
//   * the CW84 parabola limiter is a' = minmod(a, 2b), b' = minmod(b, 2a):
//     for b > 0 its test D M > D^2 / 6 reads a > 2b, its other one b > 2a,
//     and an extremum is a b <= 0;
//   * the average of the parabola over the fraction sigma of the cell next to
//     the high face is s_i + (1 - sigma)(b - sigma w), next to the low face
//     s_i - (1 - sigma)(a + sigma w);
//   * a wave that moves away from a face takes its reference's sigma, which
//     makes its amplitude vanish exactly, so no selection per variable is
//     left, and of the reference state only p and u_n enter.
// Deviations are also the more exact form: the 1 / 2^24 roundings scale with
// the differences between cells and not with the values.
#pragma once
#include "nyx_scheme.cuh"

namespace NYX_NS {

// ---------------------------------------------------------------- pairs
__device__ __forceinline__ float2 mk2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n"
      " add.rn.ftz.f32x2 z, x, y;\n mov.b64 {%0, %1}, z;\n}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n"
      " mul.rn.ftz.f32x2 z, x, y;\n mov.b64 {%0, %1}, z;\n}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{\n .reg .b64 x, y, z, w;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n"
      " mov.b64 z, {%6, %7};\n fma.rn.ftz.f32x2 w, x, y, z;\n mov.b64 {%0, %1}, w;\n}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n"
      " sub.rn.ftz.f32x2 z, x, y;\n mov.b64 {%0, %1}, z;\n}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
// by a constant: a constant operand costs a scalar instruction nothing, a pair
// of it two moves
__device__ __forceinline__ float2 mulc(float2 a, float k) { return mk2(a.x * k, a.y * k); }

__device__ __forceinline__ float rcpa(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rsqa(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float2 rcpa2(float2 a) { return mk2(rcpa(a.x), rcpa(a.y)); }
__device__ __forceinline__ float2 rsqa2(float2 a) { return mk2(rsqa(a.x), rsqa(a.y)); }
// n / d with the approximate reciprocal's error taken off once
__device__ __forceinline__ float div_refined(float n, float d) {
  const float r = rcpa(d), q = n * r;
  return fmaf(fmaf(-d, q, n), r, q);
}
// NaN if either operand is (a limited edge next to a NaN stays NaN)
__device__ __forceinline__ float min_nan(float a, float b) {
  float r;
  asm("min.NaN.ftz.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// the floors: a NaN stays one
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.ftz.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// ---------------------------------------------------------------- profiles
// Twice the MC-limited slope from the differences x, y to the two neighbours.
__device__ __forceinline__ float mc2_one(float x, float y) {
  const float t = x + y;
  const float q = fminf(fabsf(t), 4.0f * fminf(fabsf(x), fabsf(y)));
  return (x * y > 0.0f) ? copysignf(q, t) : 0.0f;
}
__device__ __forceinline__ float2 mc2_pair(float2 x, float2 y) {
  const float2 t = add2(x, y), p = mul2(x, y);
  const float qx = fminf(fabsf(t.x), 4.0f * fminf(fabsf(x.x), fabsf(y.x)));
  const float qy = fminf(fabsf(t.y), 4.0f * fminf(fabsf(x.y), fabsf(y.y)));
  return mk2((p.x > 0.0f) ? copysignf(qx, t.x) : 0.0f, (p.y > 0.0f) ? copysignf(qy, t.y) : 0.0f);
}

// Deviations a, b of the cell's profile from the five cell values.
__device__ __forceinline__ void profile_one(bool plm, float s0, float s1, float s2, float s3,
                                            float s4, float &a, float &b) {
  const float e1 = s2 - s1, e2 = s3 - s2;
  const float D0 = mc2_one(e1, e2);
  if (plm) {
    a = b = 0.25f * D0;
    return;
  }
  const float Dm = mc2_one(s1 - s0, e1), Dp = mc2_one(e2, s4 - s3);
  const float ra = 0.5f * e1 + (D0 - Dm) * (1.0f / 12.0f);
  const float rb = 0.5f * e2 + (D0 - Dp) * (1.0f / 12.0f);
  const bool ext = ra * rb <= 0.0f;
  const float qa = min_nan(fabsf(ra), fabsf(2.0f * rb)), qb = min_nan(fabsf(rb), fabsf(2.0f * ra));
  a = ext ? 0.0f : copysignf(qa, ra);
  b = ext ? 0.0f : copysignf(qb, rb);
}
__device__ __forceinline__ void profile_pair(bool plm, float2 s0, float2 s1, float2 s2, float2 s3,
                                             float2 s4, float2 &a, float2 &b) {
  const float2 e1 = sub2(s2, s1), e2 = sub2(s3, s2);
  const float2 D0 = mc2_pair(e1, e2);
  if (plm) {
    a = b = mulc(D0, 0.25f);
    return;
  }
  const float2 Dm = mc2_pair(sub2(s1, s0), e1), Dp = mc2_pair(e2, sub2(s4, s3));
  const float2 da = sub2(D0, Dm), db = sub2(D0, Dp);
  const float2 ra = mk2(0.5f * e1.x + da.x * (1.0f / 12.0f), 0.5f * e1.y + da.y * (1.0f / 12.0f));
  const float2 rb = mk2(0.5f * e2.x + db.x * (1.0f / 12.0f), 0.5f * e2.y + db.y * (1.0f / 12.0f));
  const float2 p = mul2(ra, rb), a2 = add2(ra, ra), b2 = add2(rb, rb);
  const float qax = min_nan(fabsf(ra.x), fabsf(b2.x)), qay = min_nan(fabsf(ra.y), fabsf(b2.y));
  const float qbx = min_nan(fabsf(rb.x), fabsf(a2.x)), qby = min_nan(fabsf(rb.y), fabsf(a2.y));
  const bool ex = p.x <= 0.0f, ey = p.y <= 0.0f;
  a = mk2(ex ? 0.0f : copysignf(qax, ra.x), ey ? 0.0f : copysignf(qay, ra.y));
  b = mk2(ex ? 0.0f : copysignf(qbx, rb.x), ey ? 0.0f : copysignf(qby, rb.y));
}

// ---------------------------------------------------------------- tracing
// Traced states of one cell along its direction n (tangential axes t1 < t2):
// rp[o] = (rho, p), tt[o] = (u_t1, u_t2), un[o] at cells i-2 .. i+2;
// gn, gt: gravity.  Out (rho, u_n, u_t1, u_t2, p) at the low (qm) and the
// high face (qp).
__device__ __forceinline__ void trace_pair(const Eos<float> &E, const float2 (&rp)[5],
                                           const float2 (&tt)[5], const float (&un)[5], float gn,
                                           float2 gt, float dtdx, const TraceSrc<float> &src,
                                           float fl, float (&qm)[5], float (&qp)[5]) {
  float2 arp, brp, att, btt;
  float an, bn;
  profile_pair(E.plm, rp[0], rp[1], rp[2], rp[3], rp[4], arp, brp);
  profile_pair(E.plm, tt[0], tt[1], tt[2], tt[3], tt[4], att, btt);
  profile_one(E.plm, un[0], un[1], un[2], un[3], un[4], an, bn);
  if (E.flat) {  // shock flattening: profiles pulled toward the cell value
    arp = mulc(arp, fl);
    brp = mulc(brp, fl);
    att = mulc(att, fl);
    btt = mulc(btt, fl);
    an = an * fl;
    bn = bn * fl;
  }
  const float rho = rp[2].x, p = rp[2].y, u = un[2];
  const float ir = rcpa(rho);
  const float cs2 = E.gamma * p * ir;
  const float rs = rsqa(cs2), c = cs2 * rs, ic2 = rs * rs;
  const float l0 = u - c, l2 = u + c;
  // fractions of the cell that reach the faces; a wave moving away takes its
  // face's reference fraction
  const float s2 = fmaxf(l2, 0.0f) * dtdx, s0 = fmaxf(-l0, 0.0f) * dtdx, s1 = u * dtdx;
  const float s1h = (u > 0.0f) ? s1 : s2, s1l = (u < 0.0f) ? -s1 : s0;
  const float2 wrp = sub2(brp, arp), wtt = sub2(btt, att);
  const float wn = bn - an;
  const float2 vt = mk2((tt[2].x + src.hdtp * gt.x) - src.src_u * tt[2].x,
                        (tt[2].y + src.hdtp * gt.y) - src.src_u * tt[2].y);
  const float vn = (u + src.hdtp * gn) - src.src_u * u;
  const float vp = p - src.src_p * p;
  {  // high face
    const float o2 = 1.0f - s2, o1 = 1.0f - s1h;
    float rfp = o2 * (brp.y - s2 * wrp.y), rfn = o2 * (bn - s2 * wn);
    const float2 m1 = dup2(-s1h);
    const float2 oo = dup2(o1);
    const float2 er = mul2(fma2(wrp, m1, brp), oo), et = mul2(fma2(wtt, m1, btt), oo);
    float dr = er.x + (rfp - er.y) * ic2;
    if (l0 > 0.0f) {  // the slow acoustic wave reaches the high face too
      const float s = l0 * dtdx, o = 1.0f - s;
      const float dp = rfp - o * (brp.y - s * wrp.y), dn = rfn - o * (bn - s * wn);
      const float bm = (dp - rho * c * dn) * (0.5f * ic2);
      dr = dr - bm;
      rfn = rfn + c * ir * bm;
      rfp = rfp - cs2 * bm;
    }
    const float2 qt = add2(vt, et);
    qp[0] = max_nan(rho + dr, E.small_dens);
    qp[1] = vn + rfn;
    qp[2] = qt.x;
    qp[3] = qt.y;
    qp[4] = max_nan(vp + rfp, E.small_pres);
  }
  {  // low face: deviations of the opposite sign
    const float o0 = s0 - 1.0f, o1 = s1l - 1.0f;
    float rfp = o0 * (arp.y + s0 * wrp.y), rfn = o0 * (an + s0 * wn);
    const float2 m1 = dup2(s1l);
    const float2 oo = dup2(o1);
    const float2 er = mul2(fma2(wrp, m1, arp), oo), et = mul2(fma2(wtt, m1, att), oo);
    float dr = er.x + (rfp - er.y) * ic2;
    if (l2 < 0.0f) {
      const float s = -l2 * dtdx, o = s - 1.0f;
      const float dp = rfp - o * (arp.y + s * wrp.y), dn = rfn - o * (an + s * wn);
      const float bp = (dp + rho * c * dn) * (0.5f * ic2);
      dr = dr - bp;
      rfn = rfn - c * ir * bp;
      rfp = rfp - cs2 * bp;
    }
    const float2 qt = add2(vt, et);
    qm[0] = max_nan(rho + dr, E.small_dens);
    qm[1] = vn + rfn;
    qm[2] = qt.x;
    qm[3] = qt.y;
    qm[4] = max_nan(vp + rfp, E.small_pres);
  }
}

// ---------------------------------------------------------------- Riemann
// A pair of states (left, right) in the face's normal frame; ir = 1 / rho.
struct Pair5 {
  float2 r, ir, n, t1, t2, p;
};

// The solution sampled from side o (s = +1 left, -1 right), as
// sample_side_fast of nyx_scheme.cuh, with the side's sign folded into the
// wave speeds.
__device__ __forceinline__ void sample_pair(const Eos<float> &E, float ro, float iro, float uo,
                                            float po, float Wo, float iWo, float co, float s,
                                            float ps, float us, float (&g)[3]) {
  const float dp = ps - po;
  const float d = E.linear ? rcpa(ro + dp * rcpa(co * co)) : iro - dp * (iWo * iWo);
  const float rq = div_refined(1.0f, d);
  const bool low = !(rq >= E.small_dens);
  const float rst = low ? E.small_dens : rq;
  const float ird = low ? 1.0f / E.small_dens : d;
  const float cs2 = E.gamma * ps * ird;
  const float cs = cs2 * rsqa(cs2);
  const bool shock = ps > po;
  const float so = s * uo, ss = s * us;
  const float S = so - Wo * iro, Hd = so - co, T = ss - cs;
  const bool star = shock ? (S < 0.0f) : (!(Hd >= 0.0f) && T < 0.0f);
  const bool fan = !shock && !(Hd >= 0.0f) && !(T < 0.0f);
  const float w = Hd * rcpa(Hd - T), v = 1.0f - w;
  g[0] = fan ? v * ro + w * rst : (star ? rst : ro);
  g[1] = fan ? v * uo + w * us : (star ? us : uo);
  g[2] = fan ? v * po + w * ps : (star ? ps : po);
}

// Two-shock (or linearised) solve of a pair; out = (F_rho, F_mn, F_mt1,
// F_mt2, F_rhoE, F_rhoe, u_g, p_g), the iteration of riemann_fast.
__device__ __forceinline__ void riemann_pair(const Eos<float> &E, const Pair5 &q, float (&out)[8]) {
  const float2 c2 = mul2(mulc(q.p, E.gamma), q.ir);
  const float2 rs = rsqa2(c2);
  const float2 c = mul2(c2, rs), C = mul2(q.r, c), iC = mul2(q.ir, rs);
  const float2 k = mulc(rcpa2(q.p), E.kshock);
  const float du = q.n.y - q.n.x;
  float p;
  {
    // acoustic estimate as a deviation from p_L
    p = q.p.x + ((q.p.y - q.p.x) * iC.y - du) * rcpa(iC.x + iC.y);
    p = max_nan(p, E.small_pres);
  }
  // Newton iteration.  Three steps in four lanes out of five and four in most
  // warps: the first three are taken without a test, which spares their
  // divergent loop ends (a lane that had converged only repeats its last bit).
  auto newton = [&](float p0) {
    const float2 dp = mk2(p0 - q.p.x, p0 - q.p.y);
    const float2 x = mk2(fmaxf(dp.x * k.x + 1.0f, 1e-10f), fmaxf(dp.y * k.y + 1.0f, 1e-10f));
    const float2 r = rsqa2(x);
    const float2 w = mul2(r, iC);
    const float2 t = mul2(dp, w);
    // twice the slopes: (x + 1) r^3 / C
    const float2 z = mul2(mul2(mk2(x.x + 1.0f, x.y + 1.0f), mul2(r, r)), w);
    return max_nan(p0 - ((t.x + t.y) + du) * (2.0f * rcpa(z.x + z.y)), E.small_pres);
  };
  if (!E.linear) {
    int it = 0;
    if (E.max_iter > 3) {
      p = newton(newton(newton(p)));
      it = 3;
    }
    for (; it < E.max_iter; ++it) {
      const float pn = newton(p);
      const bool conv = fabsf(pn - p) <= E.tol * pn;
      p = pn;
      if (conv) break;
    }
  }
  float2 W = C, iW = iC;
  if (!E.linear) {
    const float2 x = mk2(fmaxf((p - q.p.x) * k.x + 1.0f, 1e-10f),
                         fmaxf((p - q.p.y) * k.y + 1.0f, 1e-10f));
    const float2 r = rsqa2(x);
    W = mul2(mul2(C, x), r);
    iW = mul2(iC, r);
  }
  const float us = q.n.x + div_refined((q.p.x - q.p.y) + W.y * du, W.x + W.y);
  float g[3];
  const bool rt = us < 0.0f;
  sample_pair(E, rt ? q.r.y : q.r.x, rt ? q.ir.y : q.ir.x, rt ? q.n.y : q.n.x, rt ? q.p.y : q.p.x,
              rt ? W.y : W.x, rt ? iW.y : iW.x, rt ? c.y : c.x, rt ? -1.0f : 1.0f, p, us, g);
  float t1 = rt ? q.t1.y : q.t1.x, t2 = rt ? q.t2.y : q.t2.x;
  if (us == 0.0f) {  // the mean of both sides
    float h[3];
    sample_pair(E, q.r.y, q.ir.y, q.n.y, q.p.y, W.y, iW.y, c.y, -1.0f, p, us, h);
#pragma unroll
    for (int v = 0; v < 3; ++v) g[v] = 0.5f * (g[v] + h[v]);
    t1 = 0.5f * (t1 + q.t1.y);
    t2 = 0.5f * (t2 + q.t2.y);
  }
  const float rg = max_nan(g[0], E.small_dens), ug = g[1], pg = max_nan(g[2], E.small_pres);
  const float fr = rg * ug;
  const float re = pg * E.igm1;
  const float ke = 0.5f * rg * (ug * ug + t1 * t1 + t2 * t2);
  out[0] = fr;
  out[1] = fr * ug + pg;
  out[2] = fr * t1;
  out[3] = fr * t2;
  out[4] = ug * (re + ke + pg);
  out[5] = ug * re;
  out[6] = ug;
  out[7] = pg;
}

// ---------------------------------------------------------------- corner coupling
// Conserved form (rho, m, rho e) of a pair of edge states while the
// transverse flux differences of their cells are taken off.
struct Cons5 {
  float2 r, n, t1, t2, e;
};
__device__ __forceinline__ Cons5 to_cons(const Eos<float> &E, float2 r, float2 n, float2 t1,
                                         float2 t2, float2 p) {
  Cons5 u;
  u.r = r;
  u.n = mul2(r, n);
  u.t1 = mul2(r, t1);
  u.t2 = mul2(r, t2);
  u.e = mulc(p, E.igm1);
  return u;
}
// Back to primitives, from the corrected state.
__device__ __forceinline__ Pair5 from_cons(const Eos<float> &E, const Cons5 &u) {
  Pair5 o;
  o.r = u.r;
  o.ir = rcpa2(u.r);
  o.n = mul2(u.n, o.ir);
  o.t1 = mul2(u.t1, o.ir);
  o.t2 = mul2(u.t2, o.ir);
  o.p = mk2(max_nan(u.e.x * E.gm1, E.small_pres), max_nan(u.e.y * E.gm1, E.small_pres));
  return o;
}

}  // namespace NYX_NS
