// mw_adjoint.cuh -- adjoint of the forces for force-matching fits.
//
// The paper fits lambda, epsilon and sigma by scans (Sec. II.D); this is the
// gradient-based counterpart.  Given w = dL/dF (one vector per atom) let
//   D(x, theta) = sum_i w_i . grad_i E.
// Because F = -grad E:
//   dL/dx       = -grad_x D = -H w                (H = Hessian of E)
//   dL/depsilon = -D / epsilon                     (E is linear in epsilon)
//   dL/dlambda  = -D3 / lambda                     (E3 is linear in lambda)
//   dL/dsigma   = (D + sum_terms sum_legs r_leg . dD_term/dr_leg) / sigma
// the last from the reduced form E = epsilon E~(x / sigma) of Sec. II.A.
// Each term of E depends on its leg vectors r (centre -> partner); D_term =
// sum_legs dw_leg . dterm/dr_leg with dw = w_partner - w_centre, and
// dD_term/dr_leg is the forward-mode tangent of dterm/dr_leg along dw
// (H_term dw).  The leg and triplet quantities are recomputed here from the
// positions and the current neighbour list, never stored between calls.
//
// Layout mirrors k_force: kG lanes per centre compact its legs into a
// shared-memory table (stage_legs), then two passes over the legs, each lane
// its own.  Pass B takes a leg's terms (leg_terms, as the forces do), its
// tangents du = (dw - (u.dw) u)/r, rdot = u.dw and the pair part, and adds
// the leg to the centre's moments S0 = sum e, s = sum e u, M = sum e u u^T
// and to their tangents (edot = -nde rdot e).  Pass C forms each leg's
// three-body gradient G_j = dE3_i/dr_j and its tangent H_j from the moments
// in O(1): with A_j, B_j, C_j of k_force (sums over k != j that are affine in
// the moments, the k = j term taken back out),
//   G_j = e_j [tr (A_j - B_j u_j) - nde C_j u_j],
//   H_j = (edot_j / e_j) G_j + e_j [trdot (A_j - B_j u_j) + tr (Adot_j - Bdot_j u_j - B_j du_j)
//         - (ndedot C_j + nde Cdot_j) u_j - nde C_j du_j],
// where Adot_j, Bdot_j, Cdot_j are the same sums with one factor replaced by
// its tangent.  This is the sum over ordered leg pairs reordered, O(n) per
// centre instead of O(n^2).
//
// Bound by instruction issue: about 330 FP32 operations per leg.  On 64 boxes
// of 4096 atoms (262144) the kernel takes 97 us (fit of 64 frames); the loop over
// ordered leg pairs that it replaced took 234 us.
#pragma once

#include "mw_device.cuh"

namespace mw {

struct AdjTable {
  float4 ue[kFAtoms * kLMax];   // pass A: dx, dy, dz, j; then ux, uy, uz, e
  float4 aux[kFAtoms * kLMax];  // nde, 1/r, t = 1/(r - a sig), j (int bits)
  float4 dw[kFAtoms * kLMax];   // dw (x, y, z), r
};

constexpr int kAdjSums = 4;  // D2, D3, RH and one unused (a power of two reduces by butterfly)

struct AdjDev {
  const float4* w;   // dL/dF in sorted order
  float4* gx;        // dL/dx accumulator, sorted order
  double* acc;       // per box: kAdjSums sums
  float4* lrel;      // per box: relative rounding error of Lq (x, y, z)
};

// d^2 phi2 / dr^2 of a leg from its terms (FP32).  With E = A eps exp(sig t),
// t = 1/(r - a sig), and h = sig t^2 (E' = -h E, h' = -2 t h),
//   phi2'' = E f'' - 2 h E f' + h (h + 2 t) E f,   f = B (sig/r)^p - (sig/r)^q.
// For (p, q) = (4, 0), E f = phi2 and E B (sig/r)^4 = phi2 + E come from
// leg_terms, which carries them to about an ulp.
__device__ __forceinline__ float phi2_d2(const FParams& P, const LegTerms& lt) {
  const float t2 = lt.t * lt.t;
  const float h = fmaf(P.sig, t2, P.sig_lo * t2);
  const float hh = h * fmaf(2.0f, lt.t, h);
  if (P.p == 4 && P.q == 0) {
    const float yr = (lt.phi + lt.ae2) * lt.invr;  // E B (sig/r)^4 / r
    return fmaf(yr, fmaf(20.0f, lt.invr, 8.0f * h), lt.phi * hh);
  }
  const float sr = P.sig * lt.invr;
  const float srp = powi(sr, P.p), srq = powi(sr, P.q);
  const float f1 = ((float)(-P.p) * P.B * srp + (float)P.q * srq) * lt.invr;
  const float f2 = ((float)(P.p * (P.p + 1)) * P.B * srp - (float)(P.q * (P.q + 1)) * srq) * lt.invr * lt.invr;
  return fmaf(lt.ae2, fmaf(-2.0f * f1, h, f2), lt.phi * hh);
}

// Whole contribution of a centre with more than kLMax legs (rare): legs in
// local memory, ordered leg pairs.  Called by the centre's group leader, out
// of line so that its local arrays stay off the common path.
__device__ __noinline__ void adjoint_overflow_item(const Dev& d, const AdjDev& A, const FParams& P, int i) {
  const uint4 qi = d.q[i];
  const int b = (int)qi.w;
  const Box& bx = d.box[b];
  const float4 wi = A.w[i];
  int cnt = d.nbr_cnt[i];
  if (cnt > d.W) cnt = d.W;
  float4 U[kMaxLegsOverflow], X[kMaxLegsOverflow], V[kMaxLegsOverflow];
  int nl = 0;
  float d2s = 0.f, d3s = 0.f, rhs = 0.f, cx = 0.f, cy = 0.f, cz = 0.f;
  for (int s = 0; s < cnt; ++s) {
    const int j = d.nbr[(size_t)i * d.W + s];
    const uint4 qj = d.q[j];
    const float dx = fix_diff(qi.x, qj.x, bx.Lq[0]), dy = fix_diff(qi.y, qj.y, bx.Lq[1]),
                dz = fix_diff(qi.z, qj.z, bx.Lq[2]);
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    if (r2 >= P.rc2) continue;
    LegTerms lt;
    if (!leg_terms<true>(r2, P, lt)) continue;  // (edges' rounding left in: a rare path)
    if (nl >= kMaxLegsOverflow) {
      set_status(d.g, ST_LEGS);
      d.g->err_index = i;
      return;
    }
    const float ux = dx * lt.invr, uy = dy * lt.invr, uz = dz * lt.invr;
    const float4 wj = A.w[j];
    const float wx = wj.x - wi.x, wy = wj.y - wi.y, wz = wj.z - wi.z;
    const float rd = fmaf(ux, wx, fmaf(uy, wy, uz * wz));
    U[nl] = make_float4(ux, uy, uz, P.sle * lt.e3);
    X[nl] = make_float4(2.0f * lt.invr, lt.nde, lt.t, __int_as_float(j));
    V[nl] = make_float4((wx - rd * ux) * lt.invr, (wy - rd * uy) * lt.invr, (wz - rd * uz) * lt.invr, rd);
    const float d2r = phi2_d2(P, lt) * rd;
    cx = fmaf(d2r, ux, fmaf(lt.dphi, V[nl].x, cx));
    cy = fmaf(d2r, uy, fmaf(lt.dphi, V[nl].y, cy));
    cz = fmaf(d2r, uz, fmaf(lt.dphi, V[nl].z, cz));
    d2s = fmaf(0.5f * lt.dphi, rd, d2s);
    rhs = fmaf(0.5f * lt.r, d2r, rhs);
    ++nl;
  }
  for (int jj = 0; jj < nl; ++jj) {
    const float4 uj = U[jj], xj = X[jj], vj = V[jj];
    const float trj = xj.x, ndej = xj.y, tj = xj.z, rdj = vj.w;
    const float trdot = -0.5f * trj * trj * rdj;
    const float ndedot = -2.0f * ndej * tj * rdj;
    float Gx = 0.f, Gy = 0.f, Gz = 0.f, hx = 0.f, hy = 0.f, hz = 0.f;
    for (int k = 0; k < nl; ++k) {
      if (k == jj) continue;
      const float4 uk = U[k], vk = V[k];
      const float ndek = X[k].y;
      const float c = fmaf(uj.x, uk.x, fmaf(uj.y, uk.y, uj.z * uk.z));
      const float cd = fmaf(vj.x, uk.x, fmaf(vj.y, uk.y, fmaf(vj.z, uk.z,
                       fmaf(uj.x, vk.x, fmaf(uj.y, vk.y, uj.z * vk.z)))));
      const float D = c - P.c0;
      const float pk = uj.w * uk.w;
      const float gg = pk * D;
      const float gd = fmaf(-gg, fmaf(ndej, rdj, ndek * vk.w), pk * cd);
      const float av = gg * trj;
      const float ad = fmaf(gd, trj, gg * trdot);
      const float qv = fmaf(c, trj, D * ndej);
      const float qd = fmaf(cd, trj + ndej, fmaf(c, trdot, D * ndedot));
      const float bv = gg * qv;
      const float bd = fmaf(gd, qv, gg * qd);
      Gx = fmaf(av, uk.x, fmaf(-bv, uj.x, Gx));
      Gy = fmaf(av, uk.y, fmaf(-bv, uj.y, Gy));
      Gz = fmaf(av, uk.z, fmaf(-bv, uj.z, Gz));
      hx = fmaf(ad, uk.x, fmaf(av, vk.x, fmaf(-bd, uj.x, fmaf(-bv, vj.x, hx))));
      hy = fmaf(ad, uk.y, fmaf(av, vk.y, fmaf(-bd, uj.y, fmaf(-bv, vj.y, hy))));
      hz = fmaf(ad, uk.z, fmaf(av, vk.z, fmaf(-bd, uj.z, fmaf(-bv, vj.z, hz))));
    }
    const float rj = 2.0f / trj;
    const float wx = fmaf(rj, vj.x, rdj * uj.x), wy = fmaf(rj, vj.y, rdj * uj.y), wz = fmaf(rj, vj.z, rdj * uj.z);
    d3s = fmaf(wx, Gx, fmaf(wy, Gy, fmaf(wz, Gz, d3s)));
    rhs = fmaf(rj, fmaf(uj.x, hx, fmaf(uj.y, hy, uj.z * hz)), rhs);
    red_add_v4(A.gx + __float_as_int(xj.w), -hx, -hy, -hz);
    cx += hx;
    cy += hy;
    cz += hz;
  }
  red_add_v4(A.gx + i, cx, cy, cz);
  atomicAdd(&A.acc[kAdjSums * b], (double)d2s);
  atomicAdd(&A.acc[kAdjSums * b + 1], (double)d3s);
  atomicAdd(&A.acc[kAdjSums * b + 2], (double)rhs);
}

__device__ void adjoint_block(const Dev& d, const AdjDev& A, const FParams& P, AdjTable& T, int blk) {
  const int g = threadIdx.x & (kG - 1);
  const int a = threadIdx.x / kG;
  const int sw = (a * kG) & 7;  // the row's bank-group swizzle, as in k_force
  auto at = [&](int l) { return a * kLMax + (l ^ sw); };
  const int i = blk * kFAtoms + a;
  const bool valid = i < d.N;
  float acc[kAdjSums] = {0.f, 0.f, 0.f, 0.f};  // D2, D3, RH
  float px = 0.f, py = 0.f, pz = 0.f;  // dL/dx_i
  uint4 qi = make_uint4(0u, 0u, 0u, 0u);
  float4 wi = make_float4(0.f, 0.f, 0.f, 0.f);
  int cnt = 0, b = -1;
  float L0 = 0.f, L1 = 0.f, L2 = 0.f;
  float4 lrel = make_float4(0.f, 0.f, 0.f, 0.f);
  if (valid) {
    qi = d.q[i];
    b = (int)qi.w;
    wi = A.w[i];
    lrel = A.lrel[b];
    cnt = min(d.nbr_cnt[i], d.W);
    const Box& bx = d.box[b];
    L0 = bx.Lq[0];
    L1 = bx.Lq[1];
    L2 = bx.Lq[2];
  }
  const int nl = stage_legs<kG, kLMax>(d, P.rc2, T.ue, at, T.aux + (threadIdx.x >> 5) * kWAtoms * kLMax, qi, L0, L1, L2,
                                         d.nbr + (size_t)(valid ? i : 0) * d.W, cnt);
  __syncwarp();
  const int nstage = nl <= kLMax ? nl : 0;  // larger centres: adjoint_overflow_item does everything
  // moments S0, s, M (xx yy zz xy xz yz) and their tangents
  float m[10] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  float md[10] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (int l = g; l < nstage; l += kG) {
    const float4 rec = T.ue[at(l)];
    const float r2 = fmaf(rec.x, rec.x, fmaf(rec.y, rec.y, rec.z * rec.z));
    // the FP32 rounding of the edges (up to 6e-8) stretches every leg alike,
    // and dL/dsigma and dL/dlambda amplify it twentyfold: taken out here
    const float x2 = rec.x * rec.x, y2 = rec.y * rec.y, z2 = rec.z * rec.z;
    const float stretch = fmaf(x2, lrel.x, fmaf(y2, lrel.y, z2 * lrel.z)) * rcp_approx(r2);
    const float4 wj = A.w[__float_as_int(rec.w)];
    LegTerms lt;
    if (!leg_terms<true>(r2, P, lt, stretch)) {
      T.ue[at(l)] = make_float4(0.f, 0.f, 0.f, 0.f);
      continue;
    }
    const float ux = rec.x * lt.invu, uy = rec.y * lt.invu, uz = rec.z * lt.invu;
    const float wx = wj.x - wi.x, wy = wj.y - wi.y, wz = wj.z - wi.z;
    const float rd = fmaf(ux, wx, fmaf(uy, wy, uz * wz));
    const float vx = fmaf(-rd, ux, wx) * lt.invr, vy = fmaf(-rd, uy, wy) * lt.invr, vz = fmaf(-rd, uz, wz) * lt.invr;
    // pair: dD/dr = phi'' rdot u + phi' du ; dL/dx_i = +dD/dr (owner)
    const float d2r = phi2_d2(P, lt) * rd;
    px = fmaf(d2r, ux, fmaf(lt.dphi, vx, px));
    py = fmaf(d2r, uy, fmaf(lt.dphi, vy, py));
    pz = fmaf(d2r, uz, fmaf(lt.dphi, vz, pz));
    acc[0] = fmaf(0.5f * lt.dphi, rd, acc[0]);
    acc[2] = fmaf(0.5f * lt.r, d2r, acc[2]);
    const float e = P.sle * lt.e3;
    const float ed = -lt.nde * rd * e;
    T.ue[at(l)] = make_float4(ux, uy, uz, e);
    T.aux[at(l)] = make_float4(lt.nde, lt.invr, lt.t, rec.w);
    T.dw[at(l)] = make_float4(wx, wy, wz, lt.r);
    const float ex = e * ux, ey = e * uy, ez = e * uz;
    const float fx = fmaf(ed, ux, e * vx), fy = fmaf(ed, uy, e * vy), fz = fmaf(ed, uz, e * vz);  // tangent of e u
    m[0] += e;
    m[1] += ex;
    m[2] += ey;
    m[3] += ez;
    m[4] = fmaf(ex, ux, m[4]);
    m[5] = fmaf(ey, uy, m[5]);
    m[6] = fmaf(ez, uz, m[6]);
    m[7] = fmaf(ex, uy, m[7]);
    m[8] = fmaf(ex, uz, m[8]);
    m[9] = fmaf(ey, uz, m[9]);
    md[0] += ed;
    md[1] += fx;
    md[2] += fy;
    md[3] += fz;
    md[4] = fmaf(fx, ux, fmaf(ex, vx, md[4]));
    md[5] = fmaf(fy, uy, fmaf(ey, vy, md[5]));
    md[6] = fmaf(fz, uz, fmaf(ez, vz, md[6]));
    md[7] = fmaf(fx, uy, fmaf(ex, vy, md[7]));
    md[8] = fmaf(fx, uz, fmaf(ex, vz, md[8]));
    md[9] = fmaf(fy, uz, fmaf(ey, vz, md[9]));
  }
#pragma unroll
  for (int k = 0; k < 10; ++k) {
#pragma unroll
    for (int o = 1; o < kG; o <<= 1) {
      m[k] += __shfl_xor_sync(kFull, m[k], o);
      md[k] += __shfl_xor_sync(kFull, md[k], o);
    }
  }
  __syncwarp();  // the group's table entries are complete
  const float c0 = P.c0;
  const float cc = c0 * c0, ccl = fmaf(c0, c0, -cc);  // c0^2 as hi + lo
  const int n3 = nstage > 1 ? nstage : 0;  // one leg: no three-body term
  for (int l = g; l < n3; l += kG) {
    const float4 u = T.ue[at(l)];
    const float4 x = T.aux[at(l)];
    const float4 w = T.dw[at(l)];
    const float e = u.w, nde = x.x, invr = x.y, t = x.z, r = w.w;
    if (e == 0.f) continue;
    const float rd = fmaf(u.x, w.x, fmaf(u.y, w.y, u.z * w.z));
    const float3 v = make_float3(fmaf(-rd, u.x, w.x) * invr, fmaf(-rd, u.y, w.y) * invr, fmaf(-rd, u.z, w.z) * invr);
    const float mx = fmaf(m[4], u.x, fmaf(m[7], u.y, m[8] * u.z));  // M u
    const float my = fmaf(m[7], u.x, fmaf(m[5], u.y, m[9] * u.z));
    const float mz = fmaf(m[8], u.x, fmaf(m[9], u.y, m[6] * u.z));
    const float qm = fmaf(u.x, mx, fmaf(u.y, my, u.z * mz));              // u.M u
    const float ps = fmaf(u.x, m[1], fmaf(u.y, m[2], u.z * m[3]));        // u.s
    const float cjj = fmaf(u.x, u.x, fmaf(u.y, u.y, u.z * u.z));
    const float djj = cjj - c0;
    const float self = e * djj;
    const float Bj = fmaf(-c0, ps, qm) - self * cjj;
    const float Cj = fmaf(-2.0f * c0, ps, fmaf(cc, m[0], fmaf(ccl, m[0], qm))) - self * djj;
    const float Ax = fmaf(-c0, m[1], mx) - self * u.x;
    const float Ay = fmaf(-c0, m[2], my) - self * u.y;
    const float Az = fmaf(-c0, m[3], mz) - self * u.z;
    // tangents: Md u, M v, and the scalars built from them
    const float dx = fmaf(md[4], u.x, fmaf(md[7], u.y, md[8] * u.z));
    const float dy = fmaf(md[7], u.x, fmaf(md[5], u.y, md[9] * u.z));
    const float dz = fmaf(md[8], u.x, fmaf(md[9], u.y, md[6] * u.z));
    const float nx = fmaf(m[4], v.x, fmaf(m[7], v.y, m[8] * v.z));
    const float ny = fmaf(m[7], v.x, fmaf(m[5], v.y, m[9] * v.z));
    const float nz = fmaf(m[8], v.x, fmaf(m[9], v.y, m[6] * v.z));
    const float qd = fmaf(u.x, dx, fmaf(u.y, dy, u.z * dz)) + 2.0f * fmaf(v.x, mx, fmaf(v.y, my, v.z * mz));
    const float pd = fmaf(v.x, m[1], fmaf(v.y, m[2], v.z * m[3])) + fmaf(u.x, md[1], fmaf(u.y, md[2], u.z * md[3]));
    const float cd = 2.0f * fmaf(u.x, v.x, fmaf(u.y, v.y, u.z * v.z));  // of c_jj (rounding only)
    const float ed = -nde * rd * e;
    const float selfd = fmaf(ed, djj, e * cd);
    const float Bd = fmaf(-c0, pd, qd) - fmaf(selfd, cjj, self * cd);
    const float Cd = fmaf(-2.0f * c0, pd, fmaf(cc, md[0], fmaf(ccl, md[0], qd))) - fmaf(selfd, djj, self * cd);
    const float Adx = fmaf(-c0, md[1], dx + nx) - fmaf(selfd, u.x, self * v.x);
    const float Ady = fmaf(-c0, md[2], dy + ny) - fmaf(selfd, u.y, self * v.y);
    const float Adz = fmaf(-c0, md[3], dz + nz) - fmaf(selfd, u.z, self * v.z);
    const float tr = 2.0f * invr;
    const float trd = -0.5f * tr * tr * rd;
    const float nded = -2.0f * nde * t * rd;
    // G = e (tr (A - B u) - nde C u), H its tangent
    const float k1 = fmaf(tr, Bj, nde * Cj);
    const float Gx = e * fmaf(tr, Ax, -k1 * u.x), Gy = e * fmaf(tr, Ay, -k1 * u.y), Gz = e * fmaf(tr, Az, -k1 * u.z);
    const float k2 = fmaf(trd, Bj, fmaf(tr, Bd, fmaf(nded, Cj, nde * Cd)));
    const float ndr = -nde * rd;  // edot / e
    const float hx = fmaf(ndr, Gx, e * fmaf(trd, Ax, fmaf(tr, Adx, fmaf(-k1, v.x, -k2 * u.x))));
    const float hy = fmaf(ndr, Gy, e * fmaf(trd, Ay, fmaf(tr, Ady, fmaf(-k1, v.y, -k2 * u.y))));
    const float hz = fmaf(ndr, Gz, e * fmaf(trd, Az, fmaf(tr, Adz, fmaf(-k1, v.z, -k2 * u.z))));
    acc[1] = fmaf(w.x, Gx, fmaf(w.y, Gy, fmaf(w.z, Gz, acc[1])));
    acc[2] = fmaf(r, fmaf(u.x, hx, fmaf(u.y, hy, u.z * hz)), acc[2]);
    red_add_v4(A.gx + __float_as_int(x.w), -hx, -hy, -hz);
    px += hx;
    py += hy;
    pz += hz;
  }
#pragma unroll
  for (int o = 1; o < kG; o <<= 1) {
    px += __shfl_xor_sync(kFull, px, o);
    py += __shfl_xor_sync(kFull, py, o);
    pz += __shfl_xor_sync(kFull, pz, o);
  }
  if (valid && g == 0) {
    if (nl > kLMax)
      adjoint_overflow_item(d, A, P, i);
    else
      red_add_v4(A.gx + i, px, py, pz);
  }
  box_accumulate<kAdjSums>(acc, b, [&](int bb) { return &A.acc[kAdjSums * bb]; });
}

constexpr int kAdjBlocksPerSm = 6;  // 80 registers a thread, 36.9 KB of shared memory a block

__global__ void __launch_bounds__(kFThreads, kAdjBlocksPerSm) k_adjoint(const __grid_constant__ Dev d, const __grid_constant__ AdjDev A,
                                                                          const __grid_constant__ FParams P) {
  if (block_stop(d)) return;
  __shared__ AdjTable T;
  adjoint_block(d, A, P, T, blockIdx.x);
}

// dL/dF (caller's order, floats) -> sorted float4; clear outputs and counters.
__global__ void k_adj_prep(Dev d, AdjDev A, const float* __restrict__ w_user) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < kAdjSums * d.nbox) A.acc[i] = 0.0;
  if (i < d.nbox) {
    const Box& bx = d.box[i];
    float e[3];
    for (int k = 0; k < 3; ++k) e[k] = (float)(bx.L[k] * 2.3283064365386963e-10 / (double)bx.Lq[k] - 1.0);  // 2^-32
    A.lrel[i] = make_float4(e[0], e[1], e[2], 0.f);
  }
  if (i >= d.N) return;
  const int u = d.id[i];
  ((float4*)A.w)[i] = make_float4(w_user[3 * (size_t)u], w_user[3 * (size_t)u + 1], w_user[3 * (size_t)u + 2], 0.f);
  A.gx[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// dL/dx sorted -> caller's order.
__global__ void k_adj_out(Dev d, AdjDev A, float* __restrict__ g_user) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= d.N) return;
  const int u = d.id[i];
  const float4 v = A.gx[i];
  g_user[3 * (size_t)u] = v.x;
  g_user[3 * (size_t)u + 1] = v.y;
  g_user[3 * (size_t)u + 2] = v.z;
}

}  // namespace mw
