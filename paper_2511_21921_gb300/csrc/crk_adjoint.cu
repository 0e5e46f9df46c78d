// crk_adjoint.cu -- (d) vector-Jacobian product of the rates (dv/dt, du/dt)
// with respect to positions, velocities, internal energies and smoothing
// lengths.
//
// The paper has no adjoint; this is the reverse of the forward chain
//   x,h,m -> V (Eq. Vg) -> moments -> A,B,grad A,grad B (Eq. RK)
//         -> rho (Eq. rhow), grad v (Eq. gradv) -> P, c -> pair rates
// taken sweep by sweep in reverse order: c2^T, EOS^T, c1^T (+ coefficient^T),
// b2^T, b1^T.  Each sweep is gather-only: a thread accumulates only its own
// particle's adjoints.  For every list entry it takes both roles of the pair --
// its own outputs (gather flag) and its contribution to the neighbor's outputs
// (scatter flag) -- so no atomics and no per-pair storage are needed.  Neighbor
// sets, image shifts, relaxation flags and limiter branches are held fixed.
#include <cstring>

#include "crk_sweep.cuh"

namespace crk {

// (1/r) dg/dr of the Wendland C4 kernel: -30 c_g / h^7 (1-q)^4  (smooth at r = 0)
template <class R> __device__ __forceinline__ R wendland_gg(R r, R ih) {
  R q = r * ih;
  R om = R(1) - q;
  om = om > R(0) ? om : R(0);
  R om2 = om * om;
  R ih2 = ih * ih;
  return R(-30.0 * Wend<R>::cg) * (ih2 * ih2 * ih2 * ih) * (om2 * om2);
}

// Adjoint of (W, g) = wendland(|d|, 1/h) with cotangents (Wb, gb): adds the
// separation part to db and returns the h part.
//   dW/dd = g d,  dg/dd = gg d,  dW/dh = -(3W + g r^2)/h,  dg/dh = -(5g + gg r^2)/h
template <class R>
__device__ __forceinline__ R wendland_rev(R Wb, R gb, R W, R g, R gg, R r2, R ih, const R* d,
                                          R* db) {
  const R c = Wb * g + gb * gg;
#pragma unroll
  for (int k = 0; k < 3; ++k) db[k] += c * d[k];
  return -ih * (Wb * (R(3) * W + g * r2) + gb * (R(5) * g + gg * r2));
}

// Adjoint of rk_gradient: adds to Cb (coefficients), xb (separation), Wb, gb.
template <class R>
__device__ __forceinline__ void rk_gradient_rev(const R* C, const R* x, R W, R g, bool rk,
                                                const R* Gb, R* Cb, R* xb, R& Wb, R& gb) {
  if (!rk) {
    gb += Gb[0] * x[0] + Gb[1] * x[1] + Gb[2] * x[2];
#pragma unroll
    for (int k = 0; k < 3; ++k) xb[k] += g * Gb[k];
    return;
  }
  const R A = C[0];
  const R lin = R(1) + (C[1] * x[0] + C[2] * x[1] + C[3] * x[2]);
  const R linW = lin * W, AW = A * W, Alg = A * (lin * g);
  R linWb = R(0), AWb = R(0), Algb = R(0);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const R dBx = C[7 + 3 * k] * x[0] + C[8 + 3 * k] * x[1] + C[9 + 3 * k] * x[2];
    linWb += Gb[k] * C[4 + k];
    AWb += Gb[k] * (dBx + C[1 + k]);
    Algb += Gb[k] * x[k];
    Cb[4 + k] += Gb[k] * linW;
    Cb[1 + k] += Gb[k] * AW;
    const R dBxb = Gb[k] * AW;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      Cb[7 + 3 * k + a] += dBxb * x[a];
      xb[a] += dBxb * C[7 + 3 * k + a];
    }
    xb[k] += Gb[k] * Alg;
  }
  Cb[0] += Algb * (lin * g) + AWb * W;
  const R linb = Algb * (A * g) + linWb * W;
  gb += Algb * (A * lin);
  Wb += AWb * A + linWb * lin;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    Cb[1 + a] += linb * x[a];
    xb[a] += linb * C[1 + a];
  }
}

// Adjoint of rk_coefficients: reduced-moment cotangents mb[29] from the
// coefficient cotangents Cb[16], with the inverse of m2, u and A the forward
// coefficient step stored beside the moments (arithmetic in R throughout).
template <class R>
__device__ void rk_coefficients_rev(const R* mom, const R* Cb, R* mb) {
#pragma unroll
  for (int k = 0; k < 29; ++k) mb[k] = R(0);
  if (mom[kMomSing] != R(0)) return;  // constant fallback: no gradient
  // m2^-1, u = m2^-1 m1 and A as the forward coefficient step formed them
  const R Ar = mom[kMomA];
  R Mr[3][3], u[3];
  Mr[0][0] = mom[kMomInv + 0];
  Mr[0][1] = Mr[1][0] = mom[kMomInv + 1];
  Mr[0][2] = Mr[2][0] = mom[kMomInv + 2];
  Mr[1][1] = mom[kMomInv + 3];
  Mr[1][2] = Mr[2][1] = mom[kMomInv + 4];
  Mr[2][2] = mom[kMomInv + 5];
#pragma unroll
  for (int i = 0; i < 3; ++i) u[i] = mom[kMomU + i];
  const R m0r = mom[0];
  const R* m1r = mom + 1;
  const R* S0 = mom + 10;
  const R* S2 = mom + 13;
  const R* S3 = mom + 19;
  R ub[3] = {R(0), R(0), R(0)};
  R Mb[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) Mb[i][k] = R(0);
  R Ab = Cb[0];
#pragma unroll
  for (int g = 0; g < 3; ++g) {
    R d1[3], t[3], d2[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i) d1[i] = S2[s6(i, g)] + (i == g ? m0r : R(0));
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      R acc = R(0);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        d2[i][k] = S3[s10(i, k, g)] + (i == g ? m1r[k] : R(0)) + (k == g ? m1r[i] : R(0));
        acc += d2[i][k] * u[k];
      }
      t[i] = acc;
    }
    const R sdot = S0[g] - R(2) * (u[0] * d1[0] + u[1] * d1[1] + u[2] * d1[2]) +
                   (u[0] * t[0] + u[1] * t[1] + u[2] * t[2]);
    const R w[3] = {t[0] - d1[0], t[1] - d1[1], t[2] - d1[2]};
    // dB_g = M w
    const R* dBb = Cb + 7 + 3 * g;
    R wb[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      wb[k] = Mr[0][k] * dBb[0] + Mr[1][k] * dBb[1] + Mr[2][k] * dBb[2];
#pragma unroll
      for (int i = 0; i < 3; ++i) Mb[i][k] += dBb[i] * w[k];
    }
    R tb[3] = {wb[0], wb[1], wb[2]};
    R d1b[3] = {-wb[0], -wb[1], -wb[2]};
    // dA_g = -A^2 sdot
    const R dAb = Cb[4 + g];
    Ab += dAb * (R(-2) * Ar * sdot);
    const R sb = -(Ar * Ar) * dAb;
    // sdot = S0_g - 2 u.d1 + u.t
    mb[10 + g] += sb;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      ub[k] += sb * (t[k] - R(2) * d1[k]);
      d1b[k] += R(-2) * sb * u[k];
      tb[k] += sb * u[k];
    }
    // t = d2 u
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const R d2b = tb[i] * u[k];
        ub[k] += d2[i][k] * tb[i];
        mb[19 + s10(i, k, g)] += d2b;
        if (i == g) mb[1 + k] += d2b;
        if (k == g) mb[1 + i] += d2b;
      }
    // d1_i = S2_{ig} + delta_ig m0
#pragma unroll
    for (int i = 0; i < 3; ++i) mb[13 + s6(i, g)] += d1b[i];
    mb[0] += d1b[g];
  }
  // A = 1/(m0 - m1.u), B = -u, u = M m1, M = m2^{-1}
  const R* m1 = mom + 1;
  const R a0b = -Ar * Ar * Ab;
  R ubd[3], Mbd[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) ubd[k] = ub[k] - a0b * m1[k] - Cb[1 + k];
  mb[0] += a0b;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    R t = -a0b * u[k];
#pragma unroll
    for (int i = 0; i < 3; ++i) t += Mr[i][k] * ubd[i];
    mb[1 + k] += t;
  }
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) Mbd[i][k] = Mb[i][k] + ubd[i] * m1[k];
  R T[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k)
      T[i][k] = Mr[i][0] * Mbd[0][k] + Mr[i][1] * Mbd[1][k] + Mr[i][2] * Mbd[2][k];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const R v = -(T[i][0] * Mr[0][k] + T[i][1] * Mr[1][k] + T[i][2] * Mr[2][k]);
      mb[4 + s6(i, k)] += v;
    }
}

// ===========================================================================
// prologue: alpha = g_dvdt / m, beta = g_dudt / (2 m) in sorted order
// ===========================================================================
template <class R>
__global__ void k_adj_prep(const R* __restrict__ gdv, const R* __restrict__ gdu,
                           const R* __restrict__ ms, const int32_t* __restrict__ perm, int64_t n,
                           R* __restrict__ rec_ab) {
  int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const int64_t p = perm[s];
  const R im = R(1) / ms[s];
  R r[4] = {gdv[p] * im, gdv[n + p] * im, gdv[2 * n + p] * im, R(0.5) * gdu[p] * im};
  store_rec<4>(rec_ab, s, r);
}

// ===========================================================================
// c2^T: reverse of the pair rates.  For the unordered pair {i, j},
//   L_ij = F.(alpha_i - alpha_j) + 2 (beta_i f_ij + beta_j f_ji) E_ij,
//   E_ij = F.(v_j - v_i)   (f = 1/2 unless the energy split is on)
// and thread i takes the derivative with respect to its own variables (the
// share's u_i dependence included; the sign of E_ij is held, as every branch).
// ===========================================================================
template <class R, bool VAR = false> struct PassA2 {
  // VAR: the formulation variants (per-side viscosity, energy split) are
  // compiled in; the default form is compiled without them so that its
  // register allocation is not affected.
  static constexpr bool GATHER = false;
  static constexpr int BLOCK = 64;
  static constexpr int MB0 = 1, MB1 = 5, MB2 = 6;  // resident-block variants
  static constexpr int DEEP = 3;  // register buffers of load mode 4
  static constexpr int QUEUE = Q_A_C2;
  using Real = R;
  static constexpr int SW0 = Rec<R>::C2, SW1 = 4;  // words staged per neighbor
  static constexpr bool LPT = true;   // items longest first
  static constexpr bool BALANCE = true;   // full sweep takes the length-balanced work list
  using RC = Rec<R>;
  using AR = ARec<R>;
  struct Args {
    Common c;
    const R* __restrict__ rec_c2;
    const R* __restrict__ rec_ab;
    const R* __restrict__ rhos;
    const R* __restrict__ us;
    const R* __restrict__ Ds;
    const R* __restrict__ ms;
    const R* __restrict__ coef;
    R* rec_a1;
    R* acc;
    R* cbar;
    AVParams<R> av;
    R Cl, Cq, gm1, ggm1;
    // optional: the forward rates, accumulated from the same pair forces
    // (the fused forward + adjoint sweep of crk_rates_adjoint)
    R* dvdt;
    R* dudt;
  };
  using D2 = P2<R>;
  struct State {
    R ri[RC::C2];  // own record, columns negated (load_own_rates_record)
    R ab[4];
    R L, halfL;
    int64_t s;
    // sums over the pairs; the factors that depend on this particle alone are
    // applied in end()
    D2 xb01, vb01;
    R xb2, vb2;
    R h1;        // -(1/h) times this is the h part through W, g and mu
    R h2;        // -(1/h)^2 times this is the h part through eta
    R Vb, Pb;    // Vb: times -1/2
    R q1, q2;    // sum of Qb mu, of Qb mu^2
    R u, ubs;    // specific energy and its cotangent through the energy split
    D2 K[8];     // minus the cotangents of M's constant column; those of its others
    D2 gvb00, gvb2;    // (00, 01), (02, 12)
    R gvb11, gvb22;
    R fa[3];
    Acc<R> fe;
  };
  __device__ static void begin(const Args& a, int64_t s, State& st) {
    load_own_rates_record<R>(a.rec_c2, s, st.ri);
    load_rec<4>(a.rec_ab, s, st.ab);
    const double L = a.c.box_L[a.c.boxid[s]];
    st.L = (R)L;
    st.halfL = (R)(0.5 * L);
    st.s = s;
    const D2 zero = dup2(R(0));
    st.xb01 = st.vb01 = st.gvb00 = st.gvb2 = zero;
    st.xb2 = st.vb2 = st.h1 = st.h2 = st.Vb = st.Pb = st.q1 = st.q2 = R(0);
    st.gvb11 = st.gvb22 = R(0);
    st.u = VAR ? a.us[s] : R(0);
    st.ubs = R(0);
#pragma unroll
    for (int k = 0; k < 8; ++k) st.K[k] = zero;
    st.fa[0] = st.fa[1] = st.fa[2] = R(0);
    st.fe = Acc<R>();
  }
  __device__ static const R* src0(const Args& a) { return a.rec_c2; }
  __device__ static const R* src1(const Args& a) { return a.rec_ab; }
  // (grad v + grad v^T) e from grad v e
  __device__ static __forceinline__ void both_gradv(const R* rec, const R* e, const R* gve, R* o) {
#pragma unroll
    for (int q = 0; q < 3; ++q)
      o[q] = fma_(rec[c2_gv(2, q)], e[2],
                  fma_(rec[c2_gv(1, q)], e[1], fma_(rec[c2_gv(0, q)], e[0], gve[q])));
  }
  __device__ static void pair_s(const Args& a, State& st, const R* rj, const R* abj, uint32_t j,
                                uint32_t) {
    const R* ri = st.ri;
    PairC2<R> p;
    p.template forward<VAR>(ri, rj, st.L, st.halfL, a.av);
    const bool qside = VAR && a.av.q_side;
    R f = R(0.5), dfdui = R(0), E = R(0);
    if (VAR || a.dvdt) E = p.work();
    if (VAR && a.av.energy_split) {
      const R uj = a.us[j];
      f = energy_share(true, E, st.u, uj);
      const R su = st.u + uj;
      if (su > R(0) && E != R(0)) dfdui = (E > R(0) ? -uj : uj) / (su * su);
    }
    if (a.dvdt) {  // forward rates from the same force (fused sweep)
#pragma unroll
      for (int k = 0; k < 3; ++k) st.fa[k] += p.F[k];
      st.fe.add(f * E);
    }
    // beta = g_dudt / (2 m), so the energy term of the pair is c E with
    // c = 2 (beta_i f_ij + beta_j f_ji) (beta_i + beta_j for halves)
    R csum;
    if (VAR && a.av.energy_split) {
      csum = R(2) * (st.ab[3] * f + abj[3] * (R(1) - f));
      st.ubs += R(2) * (st.ab[3] - abj[3]) * E * dfdui;
    } else {
      csum = st.ab[3] + abj[3];
    }
    R Fb[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) Fb[k] = fma_(-csum, p.vij[k], st.ab[k] - abj[k]);
    // cotangents of G_i (qi) and, negated, of G_j (qj), and of Q_i, Q_j
    R qi[3], qj[3], Qib, Qjb;
    const R Vj = rj[RC::C2_V];
    if (qside) {
      // F = VV [PP dG + 2 (Q_i G_i - Q_j G_j)]
      R VVb = R(0), FdG = R(0), FGi = R(0), FGj = R(0);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        VVb += Fb[k] * (p.PP * p.dG[k] + R(2) * (p.Qi * p.Gi[k] - p.Qj * p.Gj[k]));
        FdG += Fb[k] * p.dG[k];
        FGi += Fb[k] * p.Gi[k];
        FGj += Fb[k] * p.Gj[k];
        qi[k] = p.VV * (p.PP + R(2) * p.Qi) * Fb[k];
        qj[k] = p.VV * (p.PP + R(2) * p.Qj) * Fb[k];
      }
      Qib = R(2) * p.VV * FGi;
      Qjb = R(-2) * p.VV * FGj;
      st.Vb = fma_(VVb, Vj, st.Vb);
      st.Pb += p.VV * FdG;
    } else {
      const R preb = dot3(Fb, p.dG);
      const R pre = p.VV * p.Pi;
      const R pv = preb * Vj;
#pragma unroll
      for (int k = 0; k < 3; ++k) qi[k] = pre * Fb[k];
      qj[0] = qi[0];
      qj[1] = qi[1];
      qj[2] = qi[2];
      st.Vb = fma_(pv, p.Pi, st.Vb);
      Qib = Qjb = pv * (R(-0.5) * ri[RC::C2_V]);
      st.Pb += Qib;
    }
    // ---- viscosity: Q = mu (QB mu + QA'), mu = min(0, t), t = vx ih / D
    R mui, muj, ti, tj;
    get2(p.mu, mui, muj);
    get2(p.t, ti, tj);
    const R y1 = Qib * mui;
    st.q1 += y1;
    st.q2 = fma_(y1, mui, st.q2);
    R mbi, mbj;
    get2(mul2(mk2(Qib, Qjb), fma2(mk2(ri[RC::C2_QB], rj[RC::C2_QB]), p.mu, p.qs)), mbi, mbj);
    const D2 mb = mk2(ti < R(0) ? mbi : R(0), tj < R(0) ? mbj : R(0));
    const R vxb = hadd2(mul2(mb, p.hD));
    // dt/d(r^2) = -t ih^2/D, dt/d(ih) = (t/ih) (1 - 2 r^2 ih^2/D)
    const D2 zt = mul2(mb, p.t);
    const D2 zw = mul2(zt, mul2(p.ih2, p.iD));
    const R r2b = -hadd2(zw);
    const R h1a = fma_(R(-2) * p.r2, lo2(zw), lo2(zt));
    // ---- limiter: vx = v_ij.d - phi (pa + pb)/2
    const R sm = p.pa + p.pb;
    const R hphi = R(-0.5) * p.phi;
    const R phib = R(-0.5) * (vxb * sm);
    R ki = vxb * hphi, kj = ki, rb = R(0);  // cotangents of pa and pb
    if (a.av.limiter) {
      // d phi0/d pa = 4 pb (pb - pa)/(pa + pb)^3
      const R c4 = R(4) * (phib * p.damp) * p.is * ((p.pb - p.pa) * p.is);
      ki = fma_(c4, p.pb * p.is, ki);
      kj = fma_(-c4, p.pa * p.is, kj);
      // eta = r min(1/h_i, 1/h_j), z = (eta - eta_crit)/eta_fold where negative
      const R etab = phib * p.phi * (R(-2) * p.z) * a.av.inv_fold;
      rb = etab * p.ihmin;
      const R ihi = ri[RC::C2_IH], ihj = rj[RC::C2_IH];
      const bool own = (ihi < ihj) || (ihi == ihj && st.s < (int64_t)j);
      st.h2 = fma_(own ? etab : R(0), p.r, st.h2);
    }
    // grad v cotangent k_i d d^T, symmetric
    const D2 ke01 = mul2(dup2(ki), p.e01);
    const R ke2 = ki * p.e[2];
    st.gvb00 = fma2(dup2(lo2(ke01)), p.e01, st.gvb00);
    st.gvb2 = fma2(ke01, p.e2, st.gvb2);
    st.gvb11 = fma_(hi2(ke01), p.e[1], st.gvb11);
    st.gvb22 = fma_(ke2, p.e[2], st.gvb22);
    R wi[3], wj[3];
    both_gradv(ri, p.e, p.gie, wi);
    both_gradv(rj, p.e, p.gje, wj);
    // ---- corrected gradients: Y = minus the cotangent of (u, lin) of i, plus j's
    R Wi, Wj, gi, gj;
    get2(p.W, Wi, Wj);
    get2(p.g, gi, gj);
    const R tei = dot3(qi, p.e), tej = qside ? dot3(qj, p.e) : tei;
    const D2 qi01 = mk2(qi[0], qi[1]), qj01 = mk2(qj[0], qj[1]);
    D2 Yi01 = mul2(dup2(-Wi), qi01), Yi2l = mk2(-Wi * qi[2], gi * tei);
    D2 Yj01 = mul2(dup2(Wj), qj01), Yj2l = mk2(Wj * qj[2], gj * tej);
    if (a.av.relax && !(ri[RC::C2_FLAG] == R(0) && rj[RC::C2_FLAG] == R(0)))
      Yi01 = Yi2l = Yj01 = Yj2l = dup2(R(0));
    // cotangents of W: q.u for i, -q.u for j; of g: -lin (q.e) for both
    const R Wib = fma_(lo2(p.ui2l), qi[2], hadd2(mul2(p.ui01, qi01)));
    const R Wjb = -fma_(lo2(p.uj2l), qj[2], hadd2(mul2(p.uj01, qj01)));
    const D2 Wb = mk2(Wib, Wjb);
    const D2 gb = mk2(-hi2(p.ui2l) * tei, -hi2(p.uj2l) * tej);
    // gg = (1/r) dg/dr = -30 c_g / h^7 (1-q)^4
    const D2 gg = mul2(mul2(mul2(p.ih2, mul2(p.ih2, p.ih2)), mul2(p.ih, p.om4)),
                       dup2(R(-30.0 * Wend<R>::cg)));
    const D2 cr = fma2(gb, gg, mul2(Wb, p.g));
    st.h1 += h1a + fma_(Wib, fma_(gi, p.r2, R(3) * Wi),
                        lo2(gb) * fma_(lo2(gg), p.r2, R(5) * gi));
    // everything along e (d = -e): W, g, the viscosity's r^2 and eta's r
    const R along = -(hadd2(cr) + fma_(R(2), r2b, rb * p.ir));
    const D2 ea[3] = {p.e0, p.e1, p.e2};
    st.K[0] = add2(st.K[0], Yi01);
    st.K[1] = add2(st.K[1], Yi2l);
    R Yx[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const R* Mi = ri + RC::C2_M + 4 + 4 * k;
      const R* Mj = rj + RC::C2_M + 4 + 4 * k;
      Yx[k] = hadd2(fma2(mk2(Mj[2], Mj[3]), Yj2l,
                         fma2(mk2(Mj[0], Mj[1]), Yj01,
                              fma2(mk2(Mi[2], Mi[3]), Yi2l, mul2(mk2(Mi[0], Mi[1]), Yi01)))));
      st.K[2 + 2 * k] = fma2(Yi01, ea[k], st.K[2 + 2 * k]);
      st.K[3 + 2 * k] = fma2(Yi2l, ea[k], st.K[3 + 2 * k]);
    }
    R gq[3];
    if (qside) {
#pragma unroll
      for (int k = 0; k < 3; ++k) gq[k] = p.gli * qi[k] + p.glj * qj[k];
    } else {
      const R gl = p.gli + p.glj;
#pragma unroll
      for (int k = 0; k < 3; ++k) gq[k] = gl * qi[k];
    }
    const D2 w01i = mk2(wi[0], wi[1]), w01j = mk2(wj[0], wj[1]);
    const D2 vij01 = mk2(p.vij[0], p.vij[1]);
    D2 db01 = add2(mk2(Yx[0], Yx[1]), mk2(gq[0], gq[1]));
    db01 = fma2(dup2(vxb), vij01, db01);
    db01 = fma2(dup2(-ki), w01i, db01);
    db01 = fma2(dup2(-kj), w01j, db01);
    db01 = fma2(dup2(along), p.e01, db01);
    st.xb01 = add2(st.xb01, db01);
    const R db2 = fma_(along, p.e[2],
                       fma_(-kj, wj[2], fma_(-ki, wi[2], fma_(vxb, p.vij[2], Yx[2] + gq[2]))));
    st.xb2 += db2;
    // v_ij enters through vx (along d) and the pair work
    st.vb01 = fma2(dup2(-vxb), p.e01, fma2(dup2(-csum), mk2(p.F[0], p.F[1]), st.vb01));
    st.vb2 = fma_(-vxb, p.e[2], fma_(-csum, p.F[2], st.vb2));
  }
  __device__ static void end(const Args& a, int64_t s, State& st) {
    using A_ = ARec<R>;
    if (a.dvdt) {
      const R im = R(1) / a.ms[s];
      const int64_t p = a.c.perm[s];
#pragma unroll
      for (int k = 0; k < 3; ++k) a.dvdt[k * a.c.n + p] = st.fa[k] * im;
      a.dudt[p] = st.fe.s * im;
    }
    const R u = a.us[s], rho = a.rhos[s];
    const R cs = sqrt_(a.ggm1 * u);
    // Q = rho (Cq mu^2 - Cl c mu); EOS: P = (gamma-1) rho u, c = sqrt(gamma (gamma-1) u)
    const R rhob = a.Cq * st.q2 - a.Cl * cs * st.q1 + a.gm1 * u * st.Pb;
    const R cb = -a.Cl * rho * st.q1;
    const R ub = a.gm1 * rho * st.Pb + (cs > R(0) ? cb * a.ggm1 / (R(2) * cs) : R(0)) + st.ubs;
    // rho = N / D
    const R D = a.Ds[s];
    const R Nb = rhob / D, Db = -rhob * rho / D;
    R C[16];
    load_rec<16>(a.coef, s, C);
    const R ih = st.ri[RC::C2_IH];
    R r[A_::A1];
#pragma unroll
    for (int k = 0; k < A_::A1; ++k) r[k] = R(0);
#pragma unroll
    for (int k = 0; k < RC::XW; ++k) r[k] = st.ri[RC::C2_X + k];
    r[A_::A1_IH] = ih;
    r[A_::A1_V] = st.ri[RC::C2_V];
    r[A_::A1_M] = a.ms[s];
#pragma unroll
    for (int k = 0; k < 3; ++k) r[A_::A1_VEL + k] = st.ri[RC::C2_VEL + k];
#pragma unroll
    for (int k = 0; k < 16; ++k) r[A_::A1_C + k] = C[k];
    r[A_::A1_NB] = Nb;
    r[A_::A1_DB] = Db;
    R gvb[9];
    get2(st.gvb00, gvb[0], gvb[1]);
    get2(st.gvb2, gvb[2], gvb[5]);
    gvb[3] = gvb[1];
    gvb[6] = gvb[2];
    gvb[7] = gvb[5];
    gvb[4] = st.gvb11;
    gvb[8] = st.gvb22;
#pragma unroll
    for (int k = 0; k < 9; ++k) r[A_::A1_GVB + k] = gvb[k];
    store_rec<A_::A1>(a.rec_a1, s, r);
    R ac[A_::ACC];
#pragma unroll
    for (int k = 0; k < A_::ACC; ++k) ac[k] = R(0);
    get2(st.xb01, ac[A_::XB], ac[A_::XB + 1]);
    ac[A_::XB + 2] = st.xb2;
    get2(st.vb01, ac[A_::VB], ac[A_::VB + 1]);
    ac[A_::VB + 2] = st.vb2;
    ac[A_::HB] = -ih * (st.h1 + ih * st.h2);
    ac[A_::UB] = ub;
    ac[A_::VVB] = R(-0.5) * st.Vb;
    store_rec<A_::ACC>(a.acc, s, ac);
    // cotangents of c_k = dA_k + A B_k, E_ka = A dB_ka + dA_k B_a, b_a = A B_a and
    // lin's constant A, taken to those of A, B, grad A, grad B (C[7 + 3 k + a])
    R cc[4], cm[3][4], Cb[16];
    get2(st.K[0], cc[0], cc[1]);
    get2(st.K[1], cc[2], cc[3]);
#pragma unroll
    for (int k = 0; k < 4; ++k) cc[k] = -cc[k];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      get2(st.K[2 + 2 * k], cm[k][0], cm[k][1]);
      get2(st.K[3 + 2 * k], cm[k][2], cm[k][3]);
    }
    R Ab = cc[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      R t = cc[k];
      Ab += cc[k] * C[1 + k] + cm[k][3] * C[1 + k];
      R bb = C[0] * (cc[k] + cm[k][3]);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        t += cm[q][k] * C[1 + q];         // E_kq's share of dA_k
        bb += cm[k][q] * C[4 + q];        // E_qk's share of B_k
        Ab += cm[q][k] * C[7 + 3 * k + q];
        Cb[7 + 3 * k + q] = C[0] * cm[q][k];
      }
      Cb[4 + k] = t;
      Cb[1 + k] = bb;
    }
    Cb[0] = Ab;
    store_rec<16>(a.cbar, s, Cb);
  }
};

// ===========================================================================
// c1^T: reverse of density and velocity gradient, then of the coefficients
// ===========================================================================
template <class R> struct PassA1 {
  static constexpr bool GATHER = false;
  static constexpr int BLOCK = 64;
  static constexpr int MB0 = 1, MB1 = 6, MB2 = 8;  // resident-block variants
  static constexpr int DEEP = 3;  // register buffers of load mode 4
  static constexpr int QUEUE = Q_A_C1;
  using Real = R;
  static constexpr int SW0 = ARec<R>::A1, SW1 = 0;  // words staged per neighbor
  static constexpr bool LPT = false;  // queue order (longest first measured slower here)
  static constexpr bool BALANCE = true;   // full sweep takes the length-balanced work list
  using AR = ARec<R>;
  struct Args {
    Common c;
    const R* __restrict__ rec_a1;
    const R* __restrict__ mom;
    const R* __restrict__ cbar;
    R* rec_a2;
    R* acc;
  };
  struct State {
    R ra[AR::A1];
    R L, halfL;
    R xb[3], vb[3], hb, ub, Vb;
    R Cb[16];
  };
  __device__ static void begin(const Args& a, int64_t s, State& st) {
    load_rec<AR::A1>(a.rec_a1, s, st.ra);
    R ac[AR::ACC];
    load_rec<AR::ACC>(a.acc, s, ac);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      st.xb[k] = ac[AR::XB + k];
      st.vb[k] = ac[AR::VB + k];
    }
    st.hb = ac[AR::HB];
    st.ub = ac[AR::UB];
    st.Vb = ac[AR::VVB];
#pragma unroll
    for (int k = 0; k < 16; ++k) st.Cb[k] = R(0);
    const double L = a.c.box_L[a.c.boxid[s]];
    st.L = (R)L;
    st.halfL = (R)(0.5 * L);
  }
  // one side: particle "o" (record ro) owns the sums; the other particle has
  // mass mo, volume Vo and velocity vo; dd = x_o - x_other.  Returns the
  // cotangents of the separation (ddb) and of the other's volume and
  // velocity difference; coefficient cotangents go to Cb when non-null.
  __device__ static __forceinline__ void side(const R* ro, const R* dd, R r2, R mo_other,
                                              R V_other, const R* vdiff, R* Cb, R* ddb, R& hb,
                                              R& Vb_other, R* vdiffb) {
    const R* C = ro + AR::A1_C;
    const R ih = ro[AR::A1_IH];
    const R r = radius(r2);
    R W, g;
    wendland(r, ih, W, g);
    const R gg = wendland_gg(r, ih);
    const R lin = R(1) + (C[1] * dd[0] + C[2] * dd[1] + C[3] * dd[2]);
    const R WR = C[0] * lin * W;
    R G[3];
    rk_gradient(C, dd, W, g, true, G);
    const R Nb = ro[AR::A1_NB], Db = ro[AR::A1_DB];
    const R* gvb = ro + AR::A1_GVB;
    const R WRb = Nb * mo_other * V_other + Db * V_other * V_other;
    R Gb[3];
    R gvG = R(0);
#pragma unroll
    for (int q = 0; q < 3; ++q)
      Gb[q] = -V_other * (gvb[q] * vdiff[0] + gvb[3 + q] * vdiff[1] + gvb[6 + q] * vdiff[2]);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const R t = gvb[3 * p] * G[0] + gvb[3 * p + 1] * G[1] + gvb[3 * p + 2] * G[2];
      vdiffb[p] = -V_other * t;
      gvG += vdiff[p] * t;
    }
    Vb_other = Nb * mo_other * WR + R(2) * Db * V_other * WR - gvG;
    R Wb = WRb * C[0] * lin, gb = R(0);
    const R linb = WRb * C[0] * W;
    if (Cb) Cb[0] += WRb * lin * W;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (Cb) Cb[1 + k] += linb * dd[k];
      ddb[k] += linb * C[1 + k];
    }
    R Cdummy[16];
    rk_gradient_rev(C, dd, W, g, true, Gb, Cb ? Cb : Cdummy, ddb, Wb, gb);
    hb += wendland_rev(Wb, gb, W, g, gg, r2, ih, dd, ddb);
  }
  __device__ static const R* src0(const Args& a) { return a.rec_a1; }
  __device__ static const R* src1(const Args&) { return nullptr; }
  __device__ static void pair_s(const Args& a, State& st, const R* rj, const R*, uint32_t j,
                                uint32_t e) {
    R d[3];
    separation(st.ra, rj, st.L, st.halfL, d);
    const R r2 = dot3(d, d);
    if (e & kGatherBit) {  // own outputs: pair (k, j), d = x_k - x_j
      R vd[3], vdb[3], db[3] = {R(0), R(0), R(0)}, Vjb;
#pragma unroll
      for (int p = 0; p < 3; ++p) vd[p] = st.ra[AR::A1_VEL + p] - rj[AR::A1_VEL + p];
      side(st.ra, d, r2, rj[AR::A1_M], rj[AR::A1_V], vd, st.Cb, db, st.hb, Vjb, vdb);
#pragma unroll
      for (int p = 0; p < 3; ++p) {
        st.xb[p] += db[p];
        st.vb[p] += vdb[p];
      }
    }
    if (e & kScatterBit) {  // j's outputs: pair (j, k), dd = x_j - x_k = -d
      const R dd[3] = {-d[0], -d[1], -d[2]};
      R vd[3], vdb[3], ddb[3] = {R(0), R(0), R(0)}, Vkb, hdummy = R(0);
#pragma unroll
      for (int p = 0; p < 3; ++p) vd[p] = rj[AR::A1_VEL + p] - st.ra[AR::A1_VEL + p];
      side(rj, dd, r2, st.ra[AR::A1_M], st.ra[AR::A1_V], vd, nullptr, ddb, hdummy, Vkb, vdb);
      st.Vb += Vkb;
#pragma unroll
      for (int p = 0; p < 3; ++p) {
        st.xb[p] -= ddb[p];
        st.vb[p] -= vdb[p];
      }
    }
  }
  __device__ static void end(const Args& a, int64_t s, State& st) {
    const R* ra = st.ra;
    const R ih = ra[AR::A1_IH], V = ra[AR::A1_V], m = ra[AR::A1_M];
    const R W0 = wendland0(ih);
    const R A = ra[AR::A1_C];
    const R Nb = ra[AR::A1_NB], Db = ra[AR::A1_DB];
    // self terms N += m V A W0, D += V^2 A W0
    st.Vb += Nb * m * A * W0 + R(2) * Db * V * A * W0;
    const R wsum = Nb * m * V + Db * V * V;
    st.Cb[0] += wsum * W0;
    st.hb += wsum * A * (R(-3) * W0 * ih);
    // coefficients -> reduced moments
    R cb2[16];
    load_rec<16>(a.cbar, s, cb2);
#pragma unroll
    for (int k = 0; k < 16; ++k) cb2[k] += st.Cb[k];
    R mom[kMomW];
    load_rec<kMomW>(a.mom, s, mom);
    R r[AR::A2];
#pragma unroll
    for (int k = 0; k < AR::A2; ++k) r[k] = R(0);
    rk_coefficients_rev<R>(mom, cb2, r + AR::A2_MB);
#pragma unroll
    for (int k = 0; k < AR::XW; ++k) r[k] = ra[k];
    r[AR::A2_IH] = ih;
    r[AR::A2_V] = V;
    store_rec<AR::A2>(a.rec_a2, s, r);
    R ac[AR::ACC];
#pragma unroll
    for (int k = 0; k < AR::ACC; ++k) ac[k] = R(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      ac[AR::XB + k] = st.xb[k];
      ac[AR::VB + k] = st.vb[k];
    }
    ac[AR::HB] = st.hb;
    ac[AR::UB] = st.ub;
    ac[AR::VVB] = st.Vb;
    store_rec<AR::ACC>(a.acc, s, ac);
  }
};

// ===========================================================================
// b2^T: reverse of the moment sums (V_j held as a variable)
// ===========================================================================
template <class R> struct PassAB2 {
  static constexpr bool GATHER = false;
  static constexpr int BLOCK = 64;
  static constexpr int MB0 = 1, MB1 = 10, MB2 = 12;  // resident-block variants
  static constexpr int DEEP = 3;  // register buffers of load mode 4
  static constexpr int QUEUE = Q_A_B2;
  using Real = R;
  static constexpr int SW0 = ARec<R>::A2, SW1 = 0;  // words staged per neighbor
  static constexpr bool LPT = false;  // queue order (longest first measured slower here)
  static constexpr bool BALANCE = true;   // full sweep takes the length-balanced work list
  using AR = ARec<R>;
  struct Args {
    Common c;
    const R* __restrict__ rec_a2;
    const R* __restrict__ ms;
    R* rec_a3;
    R* acc;
  };
  struct State {
    R ra[AR::A2];
    R L, halfL;
    R xb[3], hb, Vb;
  };
  __device__ static void begin(const Args& a, int64_t s, State& st) {
    load_rec<AR::A2>(a.rec_a2, s, st.ra);
    R ac[AR::ACC];
    load_rec<AR::ACC>(a.acc, s, ac);
#pragma unroll
    for (int k = 0; k < 3; ++k) st.xb[k] = R(0);
    st.hb = R(0);
    st.Vb = R(0);
    const double L = a.c.box_L[a.c.boxid[s]];
    st.L = (R)L;
    st.halfL = (R)(0.5 * L);
  }
  // Sums of particle o over its gather set, one term: w = V W, gam = V g
  // with the other particle's volume Vother.  Adds the separation cotangent to
  // ddb and returns the h part; Vb_other receives d/dV_other.
  __device__ static __forceinline__ R side(const R* ro, const R* d, R r2, R Vother, R* ddb,
                                           R& Vb_other) {
    const R* mb = ro + AR::A2_MB;
    const R ih = ro[AR::A2_IH];
    const R r = radius(r2);
    R W, g;
    wendland(r, ih, W, g);
    const R gg = wendland_gg(r, ih);
    const R w = Vother * W, gam = Vother * g;
    const R xx[6] = {d[0] * d[0], d[0] * d[1], d[0] * d[2], d[1] * d[1], d[1] * d[2], d[2] * d[2]};
    const R xxx[10] = {xx[0] * d[0], xx[0] * d[1], xx[0] * d[2], xx[1] * d[1], xx[1] * d[2],
                       xx[2] * d[2], xx[3] * d[1], xx[3] * d[2], xx[4] * d[2], xx[5] * d[2]};
    const R* m1b = mb + 1;
    const R* m2b = mb + 4;
    const R* S0b = mb + 10;
    const R* S2b = mb + 13;
    const R* S3b = mb + 19;
    R wb = mb[0], gamb = R(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      wb += m1b[k] * d[k];
      gamb += S0b[k] * d[k];
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      wb += m2b[k] * xx[k];
      gamb += S2b[k] * xx[k];
    }
#pragma unroll
    for (int k = 0; k < 10; ++k) gamb += S3b[k] * xxx[k];
    // explicit dependence on d
    R Q[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) Q[k] = w * m2b[k] + gam * S2b[k];
    R db[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      R t = w * m1b[c] + gam * S0b[c] + R(2) * Q[s6(c, c)] * d[c];
#pragma unroll
      for (int b2 = 0; b2 < 3; ++b2)
        if (b2 != c) t += Q[s6(c, b2)] * d[b2];
      db[c] = t;
    }
    const R* S = S3b;
    db[0] += gam * (R(3) * S[0] * xx[0] + R(2) * S[1] * xx[1] + R(2) * S[2] * xx[2] + S[3] * xx[3] +
                    S[4] * xx[4] + S[5] * xx[5]);
    db[1] += gam * (S[1] * xx[0] + R(2) * S[3] * xx[1] + S[4] * xx[2] + R(3) * S[6] * xx[3] +
                    R(2) * S[7] * xx[4] + S[8] * xx[5]);
    db[2] += gam * (S[2] * xx[0] + S[4] * xx[1] + R(2) * S[5] * xx[2] + S[7] * xx[3] +
                    R(2) * S[8] * xx[4] + R(3) * S[9] * xx[5]);
    Vb_other = wb * W + gamb * g;
    const R hpart = wendland_rev(wb * Vother, gamb * Vother, W, g, gg, r2, ih, d, db);
#pragma unroll
    for (int k = 0; k < 3; ++k) ddb[k] += db[k];
    return hpart;
  }
  __device__ static const R* src0(const Args& a) { return a.rec_a2; }
  __device__ static const R* src1(const Args&) { return nullptr; }
  __device__ static void pair_s(const Args& a, State& st, const R* rj, const R*, uint32_t j,
                                uint32_t e) {
    R d[3];
    separation(st.ra, rj, st.L, st.halfL, d);
    const R r2 = dot3(d, d);
    if (e & kGatherBit) {
      R db[3] = {R(0), R(0), R(0)}, Vjb;
      st.hb += side(st.ra, d, r2, rj[AR::A2_V], db, Vjb);
#pragma unroll
      for (int p = 0; p < 3; ++p) st.xb[p] += db[p];
    }
    if (e & kScatterBit) {
      const R dd[3] = {-d[0], -d[1], -d[2]};
      R ddb[3] = {R(0), R(0), R(0)}, Vkb;
      (void)side(rj, dd, r2, st.ra[AR::A2_V], ddb, Vkb);
      st.Vb += Vkb;
#pragma unroll
      for (int p = 0; p < 3; ++p) st.xb[p] -= ddb[p];
    }
  }
  __device__ static void end(const Args& a, int64_t s, State& st) {
    const R* ra = st.ra;
    const R ih = ra[AR::A2_IH], V = ra[AR::A2_V];
    const R mb0 = ra[AR::A2_MB];
    const R W0 = wendland0(ih);
    R ac[AR::ACC];
    load_rec<AR::ACC>(a.acc, s, ac);
    // self term of m0: V W0
    R Vb = ac[AR::VVB] + st.Vb + mb0 * W0;
    R hb = ac[AR::HB] + st.hb + mb0 * V * (R(-3) * W0 * ih);
#pragma unroll
    for (int k = 0; k < 3; ++k) ac[AR::XB + k] += st.xb[k];
    ac[AR::HB] = hb;
    ac[AR::VVB] = Vb;
    store_rec<AR::ACC>(a.acc, s, ac);
    // V = m / s  ->  sbar = -Vbar V^2 / m
    const R m = a.ms[s];
    R r[AR::A3];
#pragma unroll
    for (int k = 0; k < AR::A3; ++k) r[k] = R(0);
#pragma unroll
    for (int k = 0; k < AR::XW; ++k) r[k] = ra[k];
    r[AR::A3_IH] = ih;
    r[AR::A3_SB] = -Vb * V * V / m;
    r[AR::A3_M] = m;
    store_rec<AR::A3>(a.rec_a3, s, r);
  }
};

// ===========================================================================
// b1^T: reverse of the volume sums, then the outputs in caller order
// ===========================================================================
template <class R> struct PassAB1 {
  static constexpr bool GATHER = false;
  static constexpr int BLOCK = 64;
  static constexpr int MB0 = 1, MB1 = 14, MB2 = 16;  // resident-block variants
  static constexpr int DEEP = 4;  // register buffers of load mode 4
  static constexpr int QUEUE = Q_A_B1;
  using Real = R;
  static constexpr int SW0 = ARec<R>::A3, SW1 = 0;  // words staged per neighbor
  static constexpr bool LPT = true;   // items longest first
  static constexpr bool BALANCE = false;  // full sweep takes 32 consecutive particles per warp
  using AR = ARec<R>;
  struct Args {
    Common c;
    const R* __restrict__ rec_a3;
    const R* __restrict__ acc;
    R* g_x;
    R* g_v;
    R* g_u;
    R* g_h;
  };
  struct State {
    R ra[AR::A3];
    R L, halfL;
    R xb[3], hb;
  };
  __device__ static void begin(const Args& a, int64_t s, State& st) {
    load_rec<AR::A3>(a.rec_a3, s, st.ra);
#pragma unroll
    for (int k = 0; k < 3; ++k) st.xb[k] = R(0);
    st.hb = R(0);
    const double L = a.c.box_L[a.c.boxid[s]];
    st.L = (R)L;
    st.halfL = (R)(0.5 * L);
  }
  __device__ static const R* src0(const Args& a) { return a.rec_a3; }
  __device__ static const R* src1(const Args&) { return nullptr; }
  __device__ static void pair_s(const Args& a, State& st, const R* rj, const R*, uint32_t j,
                                uint32_t e) {
    R d[3];
    separation(st.ra, rj, st.L, st.halfL, d);
    const R r2 = dot3(d, d);
    const R r = radius(r2);
    if (e & kGatherBit) {  // s_k += m_j W(r, h_k)
      const R ih = st.ra[AR::A3_IH];
      R W, g;
      wendland(r, ih, W, g);
      const R Wb = st.ra[AR::A3_SB] * rj[AR::A3_M];
#pragma unroll
      for (int p = 0; p < 3; ++p) st.xb[p] += Wb * g * d[p];
      st.hb += -ih * Wb * (R(3) * W + g * r2);
    }
    if (e & kScatterBit) {  // s_j += m_k W(r, h_j), separation x_j - x_k = -d
      const R ih = rj[AR::A3_IH];
      R W, g;
      wendland(r, ih, W, g);
      const R Wb = rj[AR::A3_SB] * st.ra[AR::A3_M];
#pragma unroll
      for (int p = 0; p < 3; ++p) st.xb[p] += Wb * g * d[p];
    }
  }
  __device__ static void end(const Args& a, int64_t s, State& st) {
    const R ih = st.ra[AR::A3_IH], sb = st.ra[AR::A3_SB], m = st.ra[AR::A3_M];
    R ac[AR::ACC];
    load_rec<AR::ACC>(a.acc, s, ac);
    // self term s += m W(0, h)
    const R W0 = wendland0(ih);
    const R hb = ac[AR::HB] + st.hb + sb * m * (R(-3) * W0 * ih);
    const int64_t n = a.c.n, p = a.c.perm[s];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      a.g_x[k * n + p] = ac[AR::XB + k] + st.xb[k];
      a.g_v[k * n + p] = ac[AR::VB + k];
    }
    a.g_u[p] = ac[AR::UB];
    a.g_h[p] = hb;
  }
};

// ===========================================================================
// host driver
// ===========================================================================
template <class R>
crk_status adjoint_impl(Plan* plan, cudaStream_t st, char* ws, const R* v, const R* u,
                        const R* g_dvdt, const R* g_dudt, R* g_x, R* g_v, R* g_u, R* g_h,
                        int recompute, R* dvdt, R* dudt) {
  const Layout& Ly = plan->ly;
  const int64_t n = Ly.n;
  const crk_params& p = plan->p;
  if (recompute) {
    crk_status s = forward_state_impl<R>(plan, st, ws, v, u);
    if (s != CRK_OK) return s;
  }
  Common c = make_common(plan, ws);
  cudaMemsetAsync(&c.hdr->queue[Q_A_C2], 0, 4 * sizeof(int32_t), st);
  if (n == 0) return CRK_OK;
  R* ms = reinterpret_cast<R*>(ws + Ly.ms);
  R* rec_ab = reinterpret_cast<R*>(ws + Ly.adj_ab);
  R* rec_a1 = reinterpret_cast<R*>(ws + Ly.adj_rec1);
  R* rec_a2 = reinterpret_cast<R*>(ws + Ly.adj_rec2);
  R* rec_a3 = reinterpret_cast<R*>(ws + Ly.adj_rec3);
  R* acc = reinterpret_cast<R*>(ws + Ly.adj_acc);
  R* cbar = reinterpret_cast<R*>(ws + Ly.adj_cbar);
  {
    Phase ph(plan, st, "adj_prep", 1);
    k_adj_prep<R><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(g_dvdt, g_dudt, ms, c.perm, n,
                                                               rec_ab);
  }
  typename PassA2<R>::Args a2{c,
                              reinterpret_cast<const R*>(ws + Ly.rec_c2),
                              rec_ab,
                              reinterpret_cast<const R*>(ws + Ly.rhos),
                              reinterpret_cast<const R*>(ws + Ly.us),
                              reinterpret_cast<const R*>(ws + Ly.Ds),
                              ms,
                              reinterpret_cast<const R*>(ws + Ly.coef),
                              rec_a1,
                              acc,
                              cbar,
                              make_av<R>(p),
                              (R)p.Cl,
                              (R)p.Cq,
                              (R)(p.gamma - 1.0),
                              (R)(p.gamma * (p.gamma - 1.0)),
                              dvdt,
                              dudt};
  if (p.q_side || p.energy_split) {
    typename PassA2<R, true>::Args av2;
    static_assert(sizeof(av2) == sizeof(a2), "same arguments");
    memcpy(&av2, &a2, sizeof(a2));
    launch_sweep_plain<PassA2<R, true>>(plan, st, av2, dvdt ? "rates_adj_c2" : "adj_c2");
  } else {
    launch_sweep<PassA2<R>>(plan, st, a2, dvdt ? "rates_adj_c2" : "adj_c2");
  }
  typename PassA1<R>::Args a1{c, rec_a1, reinterpret_cast<const R*>(ws + Ly.mom), cbar, rec_a2,
                              acc};
  launch_sweep<PassA1<R>>(plan, st, a1, "adj_c1");
  typename PassAB2<R>::Args b2{c, rec_a2, ms, rec_a3, acc};
  launch_sweep<PassAB2<R>>(plan, st, b2, "adj_b2");
  typename PassAB1<R>::Args b1{c, rec_a3, acc, g_x, g_v, g_u, g_h};
  launch_sweep<PassAB1<R>>(plan, st, b1, "adj_b1");
  return cudaGetLastError() == cudaSuccess ? CRK_OK : CRK_ECUDA;
}

template crk_status adjoint_impl<float>(Plan*, cudaStream_t, char*, const float*, const float*,
                                        const float*, const float*, float*, float*, float*, float*,
                                        int, float*, float*);
template crk_status adjoint_impl<double>(Plan*, cudaStream_t, char*, const double*, const double*,
                                         const double*, const double*, double*, double*, double*,
                                         double*, int, double*, double*);

}  // namespace crk
