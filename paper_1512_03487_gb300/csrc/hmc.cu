// Wilson gauge action, its force, the SU(3) link update and the hybrid Monte
// Carlo trajectory (the Grid paper lists HMC, the Wilson gauge action and the
// leapfrog and minimum-norm integrators among its algorithms, Sec. 4; the
// formulas are the textbook ones):
//
//   S_g = beta sum_{x, mu<nu} (1 - Re tr U_munu(x) / 3), periodic boundaries,
//   Sigma_mu(x) = sum_{nu != mu} [ U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
//                                + U_nu(x+mu-nu)^dag U_mu(x-nu)^dag U_nu(x-nu) ],
//   F_mu(x) = (beta / 3) * traceless part of (W - W^dag) / (2 i), W = U_mu(x) Sigma_mu(x),
//   so that dS_g = eps tr(T F) under U -> exp(i eps T) U (the convention of lqcd_force);
//   molecular dynamics: dU/dt = i P U, dP/dt = -(F_g + F_f).
//
// Gauge and momentum fields are FP64 with all 18 reals stored, in the device
// layout [parity][mu][9 chunks of double2][cb]. Sites are numbered over both
// parities, parity-major; a kernel has one thread per site or per link, two per
// site (plaquette) or four (gauge force). Reductions are the
// library's deterministic block partials summed in a fixed order by the last
// block. The trajectory driver runs on the host: each momentum step launches
// the gauge-force kernel and, with fermions, one conjugate-gradient solve
// (lqcd_cg_solve, which synchronises), M X and the fermion-force kernel in
// accumulate mode.
#include <cmath>
#include <cstring>

#include "lqcd_internal.h"

namespace lqcd {

constexpr int HMC_BLOCK = 128;
using M3 = Link<double>;

// ------------------------------------------------------------------ 3x3 algebra

__device__ __forceinline__ void m_mul(const M3& a, const M3& b, M3& c) {  // c = a b
#pragma unroll
  for (int r = 0; r < 3; r++)
#pragma unroll
    for (int k = 0; k < 3; k++) {
      cpx<double> s = cmul(a.v[3 * r], b.v[k]);
      s = cmadd(s, a.v[3 * r + 1], b.v[3 + k]);
      c.v[3 * r + k] = cmadd(s, a.v[3 * r + 2], b.v[6 + k]);
    }
}

// ------------------------------------------------------------------ link access by coordinate

__device__ __forceinline__ void link_at(const Geom& g, const void* U, int mu, const int c[4], M3& u) {
  const uint32_t lex = (uint32_t)c[0] + (uint32_t)g.X * ((uint32_t)c[1] + (uint32_t)g.Y *
                                                         ((uint32_t)c[2] + (uint32_t)g.Z * (uint32_t)c[3]));
  const int parity = (c[0] + c[1] + c[2] + c[3]) & 1;
  LinkIO<LQCD_F64, 18>::load(U, g.gstride, parity * 4 + mu, (int64_t)(lex >> 1), u);
}

__device__ __forceinline__ int extent(const Geom& g, int mu) {
  return mu == 0 ? g.X : mu == 1 ? g.Y : mu == 2 ? g.Z : g.T;
}

// c + d * mu_hat with periodic wrap (|d| <= 1)
__device__ __forceinline__ void step(const Geom& g, const int c[4], int mu, int d, int out[4]) {
#pragma unroll
  for (int k = 0; k < 4; k++) out[k] = c[k];
  const int L = extent(g, mu);
  int v = c[mu] + d;
  out[mu] = v < 0 ? v + L : (v >= L ? v - L : v);
}

__device__ __forceinline__ double2* link_ptr(double2* base, const Geom& g, int parity, int mu, int64_t cb) {
  return base + (int64_t)(parity * 4 + mu) * 9 * g.gstride + cb;
}

// thread -> (parity, cb, coordinates) over both checkerboards
__device__ __forceinline__ bool site_of_thread(const Geom& g, int64_t t, int& parity, int64_t& cb, int c[4]) {
  if (t >= 2 * (int64_t)g.Vh) return false;
  parity = t >= g.Vh ? 1 : 0;
  cb = t - parity * (int64_t)g.Vh;
  const Coord x = cb_to_coord(g, cb, parity);
#pragma unroll
  for (int k = 0; k < 4; k++) c[k] = x.c[k];
  return true;
}

// ------------------------------------------------------------------ kernels

// These kernels are bound by the FP64 pipe (2 FMA per SM per clock: one warp
// instruction occupies its SM quarter for 64 cycles), so the work is cut down to
// the fewest FP64 instructions and split finely enough that every SM gets the
// same share; the links come from L1 / L2 and memory is nearly idle. 16^4 on
// GB300, before and after: gauge force 817 -> 570 us, link update 1,058 -> 149 us,
// plaquette 209 -> 170 us.

constexpr int PLAQ_SITES = 64;  // sites per block; two warps each take three of the six planes of 32 sites

template <int MU, int NU>
__device__ __forceinline__ double plane_trace(const Geom& g, const void* U, const int c[4]) {
  int cm[4], cn[4];
  step(g, c, MU, +1, cm);
  step(g, c, NU, +1, cn);
  M3 a, b, p, q;
  link_at(g, U, MU, c, a);
  link_at(g, U, NU, cm, b);
  m_mul(a, b, p);  // U_mu(x) U_nu(x+mu)
  link_at(g, U, NU, c, a);
  link_at(g, U, MU, cn, b);
  m_mul(a, b, q);  // U_nu(x) U_mu(x+nu)
  double tr = 0.0;  // Re tr(p q^dag)
#pragma unroll
  for (int k = 0; k < 9; k++) tr = fma(p.v[k].r, q.v[k].r, fma(p.v[k].i, q.v[k].i, tr));
  return tr;
}

// sum over the six planes of Re tr U_munu(x) / 3 at each site, reduced. Two
// threads per site (three planes each): 12 products and 6 traces, 1,400 FMA a
// site, 148 us of FP64 pipe at 16^4.
__global__ void __launch_bounds__(HMC_BLOCK) plaquette_kernel(const void* U, Geom g, ReduceCtx rc) {
  const int64_t t = (int64_t)blockIdx.x * PLAQ_SITES + (threadIdx.x & (PLAQ_SITES - 1));
  int parity, c[4];
  int64_t cb;
  double v = 0.0;
  if (site_of_thread(g, t, parity, cb, c)) {
    if (threadIdx.x < PLAQ_SITES)
      v = plane_trace<0, 1>(g, U, c) + plane_trace<0, 2>(g, U, c) + plane_trace<0, 3>(g, U, c);
    else
      v = plane_trace<1, 2>(g, U, c) + plane_trace<1, 3>(g, U, c) + plane_trace<2, 3>(g, U, c);
    v *= 1.0 / 3.0;
  }
  block_reduce_finalize<HMC_BLOCK>(v, (int64_t)blockIdx.x * PLAQ_SITES, rc);
}

// The Hermitian matrix (W - W^dag) / i of a 3x3 matrix W: three real diagonal
// entries and the entries 01, 02, 12 (the other three are their conjugates).
struct Herm3 {
  double d[3];
  cpx<double> o[3];
};

// (W - W^dag) / i for W = a b: Im of W's diagonal doubled and, off the diagonal,
// W_rc - conj(W_cr) over i, accumulated straight from the factors (90 FMA instead
// of the 108 of the product).
__device__ __forceinline__ void herm_mul(const M3& a, const M3& b, Herm3& h) {
#pragma unroll
  for (int r = 0; r < 3; r++) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 3; k++)
      s = fma(a.v[3 * r + k].r, b.v[3 * k + r].i, fma(a.v[3 * r + k].i, b.v[3 * k + r].r, s));
    h.d[r] = 2.0 * s;
  }
#pragma unroll
  for (int e = 0; e < 3; e++) {
    const int r = e == 2 ? 1 : 0, c = e == 0 ? 1 : 2;
    double x = 0.0, y = 0.0;  // Im W_rc + Im W_cr, Re W_cr - Re W_rc
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const cpx<double> p = a.v[3 * r + k], q = b.v[3 * k + c], s = a.v[3 * c + k], t = b.v[3 * k + r];
      x = fma(p.r, q.i, fma(p.i, q.r, x));
      x = fma(s.r, t.i, fma(s.i, t.r, x));
      y = fma(s.r, t.r, fma(-s.i, t.i, y));
      y = fma(-p.r, q.r, fma(p.i, q.i, y));
    }
    h.o[e] = mk(x, y);
  }
}

// the same for W = a b^dag
__device__ __forceinline__ void herm_mul_nd(const M3& a, const M3& b, Herm3& h) {
#pragma unroll
  for (int r = 0; r < 3; r++) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 3; k++)
      s = fma(a.v[3 * r + k].i, b.v[3 * r + k].r, fma(-a.v[3 * r + k].r, b.v[3 * r + k].i, s));
    h.d[r] = 2.0 * s;
  }
#pragma unroll
  for (int e = 0; e < 3; e++) {
    const int r = e == 2 ? 1 : 0, c = e == 0 ? 1 : 2;
    double x = 0.0, y = 0.0;
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const cpx<double> p = a.v[3 * r + k], q = b.v[3 * c + k], s = a.v[3 * c + k], t = b.v[3 * r + k];
      x = fma(p.i, q.r, fma(-p.r, q.i, x));
      x = fma(s.i, t.r, fma(-s.r, t.i, x));
      y = fma(s.r, t.r, fma(s.i, t.i, y));
      y = fma(-p.r, q.r, fma(-p.i, q.i, y));
    }
    h.o[e] = mk(x, y);
  }
}

// c + d * mu_hat for a runtime mu, without indexing c (which would put it in local memory)
__device__ __forceinline__ void step_rt(const Geom& g, const int c[4], int mu, int d, int out[4]) {
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const int L = extent(g, k);
    const int v = c[k] + d;
    const int w = v < 0 ? v + L : (v >= L ? v - L : v);
    out[k] = k == mu ? w : c[k];
  }
}

constexpr int GF_SITES = 32;  // sites per block of the gauge force; warp mu works on their links mu

// F_mu(x) of the Wilson gauge action; out = F, or out -= coef F (accumulate).
//
// With A_munu(x) = U_mu(x) U_nu(x+mu) the upper staple's loop at x is the
// plaquette P_munu = A_munu A_numu^dag, which serves F_mu and, conjugated, F_nu;
// the lower staple is A_munu(x-nu)^dag U_nu(x-nu). A block is 32 sites (one per
// lane) and four warps, warp mu for link mu: 12 products A, 6 plaquettes (their
// anti-Hermitian parts only), 12 lower staples of two products and 4 final
// products, 4,790 FMA per site instead of the 6,100 of one thread per site
// adding six staples per link. Warp mu owns the plane (mu, mu+1) and, for
// mu < 2, (mu, mu+2); it gets the partner's A through shared memory and hands
// the plaquette's Hermitian part back the same way. 2,048 blocks at 16^4 also
// spread evenly over the SMs, where 512 blocks of a thread per site left the
// slowest SM with 4 of 3.4.
__global__ void __launch_bounds__(HMC_BLOCK) gauge_force_kernel(double2* out, const void* U, Geom g, double beta,
                                                                double coef, int accumulate) {
  __shared__ double2 shA[6][9][GF_SITES];
  __shared__ double shH[6][9][GF_SITES];
  const int lane = threadIdx.x & 31, mu = threadIdx.x >> 5;
  const int64_t t = (int64_t)blockIdx.x * GF_SITES + lane;
  int parity = 0, c[4] = {0, 0, 0, 0};
  int64_t cb = 0;
  const bool live = site_of_thread(g, t, parity, cb, c);  // lanes past the end work on site 0 and store nothing
  int cm[4];
  step_rt(g, c, mu, +1, cm);
  M3 a, b, own1, own2;
  Herm3 F;
  {  // lower staples: sum over nu of (U_mu(y) U_nu(y+mu))^dag U_nu(y), y = x - nu, then the loops U_mu(x) S
    M3 S;
#pragma unroll
    for (int k = 0; k < 9; k++) S.v[k] = mk(0.0, 0.0);
#pragma unroll 1
    for (int k = 1; k < 4; k++) {
      const int nu = (mu + k) & 3;
      int y[4], ym[4];
      step_rt(g, c, nu, -1, y);
      step_rt(g, cm, nu, -1, ym);
      M3 p;
      link_at(g, U, mu, y, a);
      link_at(g, U, nu, ym, b);
      m_mul(a, b, p);
      link_at(g, U, nu, y, a);
#pragma unroll
      for (int r = 0; r < 3; r++)
#pragma unroll
        for (int q = 0; q < 3; q++)
#pragma unroll
          for (int s = 0; s < 3; s++) S.v[3 * r + q] = cmadd_conj(S.v[3 * r + q], p.v[3 * s + r], a.v[3 * s + q]);
    }
    link_at(g, U, mu, c, a);
    herm_mul(a, S, F);
  }
  // A_munu for nu = mu + 1 (kept), mu + 2 (kept by warps 0 and 1), mu + 3 (to the plane's owner, warp nu)
  auto give = [&](int slot, const M3& m) {
#pragma unroll
    for (int k = 0; k < 9; k++) shA[slot][k][lane] = make_double2(m.v[k].r, m.v[k].i);
  };
  link_at(g, U, (mu + 3) & 3, cm, b);
  m_mul(a, b, own1);
  give(mu, own1);
  link_at(g, U, (mu + 2) & 3, cm, b);
  m_mul(a, b, own2);
  if (mu >= 2) give(2 + mu, own2);
  link_at(g, U, (mu + 1) & 3, cm, b);
  m_mul(a, b, own1);
  __syncthreads();
  // P of the owned planes: +P for this link, -P for the partner's
  auto plane = [&](int slot, int hslot, const M3& own) {
    M3 p;
#pragma unroll
    for (int k = 0; k < 9; k++) {
      const double2 w = shA[slot][k][lane];
      p.v[k] = mk(w.x, w.y);
    }
    Herm3 h;
    herm_mul_nd(own, p, h);
#pragma unroll
    for (int k = 0; k < 3; k++) {
      shH[hslot][k][lane] = h.d[k];
      shH[hslot][3 + k][lane] = h.o[k].r;
      shH[hslot][6 + k][lane] = h.o[k].i;
      F.d[k] += h.d[k];
      F.o[k] = F.o[k] + h.o[k];
    }
  };
  plane((mu + 1) & 3, mu, own1);
  if (mu < 2) plane(4 + mu, 4 + mu, own2);
  __syncthreads();
  auto minus = [&](int hslot) {
#pragma unroll
    for (int k = 0; k < 3; k++) {
      F.d[k] -= shH[hslot][k][lane];
      F.o[k] = F.o[k] - mk(shH[hslot][3 + k][lane], shH[hslot][6 + k][lane]);
    }
  };
  minus((mu + 3) & 3);
  if (mu >= 2) minus(2 + mu);
  if (!live) return;
  // F = (beta / 3) traceless[(W - W^dag) / (2 i)]
  const double f = beta / 6.0;
  const double tr = (F.d[0] + F.d[1] + F.d[2]) * (1.0 / 3.0);
  double2 o[9];
#pragma unroll
  for (int r = 0; r < 3; r++) o[4 * r] = make_double2(f * (F.d[r] - tr), 0.0);
#pragma unroll
  for (int e = 0; e < 3; e++) {
    const int r = e == 2 ? 1 : 0, q = e == 0 ? 1 : 2;
    o[3 * r + q] = make_double2(f * F.o[e].r, f * F.o[e].i);
    o[3 * q + r] = make_double2(o[3 * r + q].x, -o[3 * r + q].y);
  }
  double2* p = link_ptr(out, g, parity, mu, cb);
#pragma unroll
  for (int k = 0; k < 9; k++) {
    if (accumulate) {
      const double2 w = p[k * g.gstride];
      p[k * g.gstride] = make_double2(fma(-coef, o[k].x, w.x), fma(-coef, o[k].y, w.y));
    } else {
      p[k * g.gstride] = o[k];
    }
  }
}

// q(A) = q[0] + q[1] A + q[2] A^2, the degree-N Taylor polynomial of exp(A)
// reduced by A^3 = t A^2 - s A + d (Cayley and Hamilton): Horner's rule on the
// three coefficients, 12 FMA a step.
template <int N>
__device__ __forceinline__ void exp_coefficients(cpx<double> t, cpx<double> s, cpx<double> d, cpx<double> q[3]) {
  double c[N + 1];  // 1 / n!, folded at compile time
  c[0] = 1.0;
#pragma unroll
  for (int n = 1; n <= N; n++) c[n] = c[n - 1] / n;
  q[2] = mk(c[N], 0.0);
  q[1] = mk(c[N - 1], 0.0);
  q[0] = mk(c[N - 2], 0.0);
  const cpx<double> ms = mk(-s.r, -s.i);
#pragma unroll
  for (int n = N - 3; n >= 0; n--) {
    const cpx<double> top = q[2];
    q[2] = cmadd(q[1], t, top);
    q[1] = cmadd(q[0], ms, top);
    q[0] = cmadd(mk(c[n], 0.0), d, top);
  }
}

// The same for exp(i H), H^3 = t H^2 - s H + d with t, s, d real (H Hermitian): 6 FMA a step.
template <int N>
__device__ __forceinline__ void exp_coefficients(double t, double s, double d, cpx<double> q[3]) {
  cpx<double> c[N + 1];  // i^n / n!, folded at compile time
  c[0] = mk(1.0, 0.0);
#pragma unroll
  for (int n = 1; n <= N; n++) c[n] = mk(-c[n - 1].i / n, c[n - 1].r / n);
  q[2] = c[N];
  q[1] = c[N - 1];
  q[0] = c[N - 2];
#pragma unroll
  for (int n = N - 3; n >= 0; n--) {
    const cpx<double> top = q[2];
    q[2] = mk(fma(t, top.r, q[1].r), fma(t, top.i, q[1].i));
    q[1] = mk(fma(-s, top.r, q[0].r), fma(-s, top.i, q[0].i));
    q[0] = mk(fma(d, top.r, c[n].r), fma(d, top.i, c[n].i));
  }
}

// Halvings that bring |A|_F^2 = n2 to 1 or below; n2 becomes that of the halved A.
__device__ __forceinline__ int halvings(double& n2) {
  int s = 0;
  while (n2 > 1.0 && s < 60) {
    n2 *= 0.25;
    s++;
  }
  return s;
}

__device__ __forceinline__ double abs2(cpx<double> a) { return fma(a.r, a.r, a.i * a.i); }

// E = exp(2^-s A), A = i eps P, for any matrix P; returns s.
__device__ __forceinline__ int exp_general(const M3& P, double eps, M3& E) {
  M3 A, A2;
  double n2 = 0.0;
#pragma unroll
  for (int k = 0; k < 9; k++) {
    A.v[k] = mk(-eps * P.v[k].i, eps * P.v[k].r);  // i eps P
    n2 = fma(A.v[k].r, A.v[k].r, fma(A.v[k].i, A.v[k].i, n2));
  }
  const int s = halvings(n2);
  if (s > 0) {
    const double sc = ldexp(1.0, -s);
#pragma unroll
    for (int k = 0; k < 9; k++) A.v[k] = sc * A.v[k];
  }
  m_mul(A, A, A2);
  const cpx<double> m0 = cmadd(cmul(A.v[4], A.v[8]), mk(-A.v[5].r, -A.v[5].i), A.v[7]);
  const cpx<double> m1 = cmadd(cmul(A.v[5], A.v[6]), mk(-A.v[3].r, -A.v[3].i), A.v[8]);
  const cpx<double> m2 = cmadd(cmul(A.v[3], A.v[7]), mk(-A.v[4].r, -A.v[4].i), A.v[6]);
  const cpx<double> det = cmadd(cmadd(cmul(A.v[0], m0), A.v[1], m1), A.v[2], m2);
  cpx<double> sec = cmadd(m0, A.v[0], A.v[4] + A.v[8]);  // sum of the principal 2x2 minors
  sec = cmadd(sec, mk(-A.v[1].r, -A.v[1].i), A.v[3]);
  sec = cmadd(sec, mk(-A.v[2].r, -A.v[2].i), A.v[6]);
  const cpx<double> tr = A.v[0] + A.v[4] + A.v[8];
  cpx<double> q[3];
  if (n2 <= 0.0625) exp_coefficients<13>(tr, sec, det, q);
  else exp_coefficients<20>(tr, sec, det, q);
#pragma unroll
  for (int k = 0; k < 9; k++) {
    const cpx<double> e = cmadd(k % 4 == 0 ? q[0] : mk(0.0, 0.0), q[1], A.v[k]);
    E.v[k] = cmadd(e, q[2], A2.v[k]);
  }
  return s;
}

// The same for a Hermitian P, from its diagonal and upper triangle: with H = 2^-s
// eps P the invariants are real, H^2 is Hermitian, and the elements rc and cr of
// q1 H + q2 H^2 share their products.
__device__ __forceinline__ int exp_hermitian(const M3& P, double eps, M3& E) {
  double d[3] = {eps * P.v[0].r, eps * P.v[4].r, eps * P.v[8].r};
  cpx<double> x = eps * P.v[1], y = eps * P.v[2], z = eps * P.v[5];  // H_01, H_02, H_12
  double xx = abs2(x), yy = abs2(y), zz = abs2(z);
  double n2 = fma(d[0], d[0], fma(d[1], d[1], fma(d[2], d[2], 2.0 * (xx + yy + zz))));
  const int s = halvings(n2);
  if (s > 0) {
    const double sc = ldexp(1.0, -s), sc2 = sc * sc;
#pragma unroll
    for (int k = 0; k < 3; k++) d[k] *= sc;
    x = sc * x;
    y = sc * y;
    z = sc * z;
    xx *= sc2;
    yy *= sc2;
    zz *= sc2;
  }
  const double K[3] = {fma(d[0], d[0], xx + yy), fma(d[1], d[1], xx + zz), fma(d[2], d[2], yy + zz)};
  const cpx<double> xz = cmul(x, z);
  const cpx<double> kx = cmadd_conj((d[0] + d[1]) * x, z, y);  // (H^2)_01 = (d0 + d1) x + conj(z) y
  const cpx<double> ky = (d[0] + d[2]) * y + xz;
  const cpx<double> kz = cmadd_conj((d[1] + d[2]) * z, x, y);  // (H^2)_12 = (d1 + d2) z + conj(x) y
  const double tr = d[0] + d[1] + d[2];
  const double sec = fma(d[0], d[1], fma(d[2], d[0] + d[1], -(xx + yy + zz)));
  double det = fma(2.0, fma(xz.r, y.r, xz.i * y.i), d[0] * fma(d[1], d[2], -zz));  // 2 Re(x z conj(y))
  det = fma(-d[1], yy, fma(-d[2], xx, det));
  cpx<double> q[3];
  if (n2 <= 0.0625) exp_coefficients<13>(tr, sec, det, q);
  else exp_coefficients<20>(tr, sec, det, q);
#pragma unroll
  for (int k = 0; k < 3; k++)
    E.v[4 * k] = mk(fma(q[2].r, K[k], fma(q[1].r, d[k], q[0].r)), fma(q[2].i, K[k], fma(q[1].i, d[k], q[0].i)));
  auto pair = [&](cpx<double> h, cpx<double> k, cpx<double>& up, cpx<double>& low) {
    const double a = fma(q[2].r, k.r, q[1].r * h.r), b = fma(q[2].i, k.i, q[1].i * h.i);
    const double c = fma(q[2].r, k.i, q[1].r * h.i), e = fma(q[2].i, k.r, q[1].i * h.r);
    up = mk(a - b, c + e);
    low = mk(a + b, e - c);
  };
  pair(x, kx, E.v[1], E.v[3]);
  pair(y, ky, E.v[2], E.v[6]);
  pair(z, kz, E.v[5], E.v[7]);
  return s;
}

__device__ __forceinline__ bool is_hermitian(const M3& p) {
  bool h = p.v[0].i == 0.0 && p.v[4].i == 0.0 && p.v[8].i == 0.0;
#pragma unroll
  for (int e = 0; e < 3; e++) {
    const int r = e == 2 ? 1 : 0, c = e == 0 ? 1 : 2;
    h = h && p.v[3 * r + c].r == p.v[3 * c + r].r && p.v[3 * r + c].i == -p.v[3 * c + r].i;
  }
  return h;
}

// U <- exp(i eps P) U per link. exp(A), A = i eps P, is its Taylor polynomial
// reduced to second degree in A by the characteristic equation: one product for
// A^2, scalars, and one product with U, about 480 FMA instead of the 2,150 of a
// degree-16 Horner scheme on matrices, which the FP64 pipe bounds either way. A P
// that is Hermitian to the last bit, as the momenta are (the forces write one
// triangle and mirror it), takes about 290 (16^4: 253 -> 149 us). Degree 13 up to |A|_F = 1/4
// (molecular-dynamics steps stay there), 20 up to 1, truncation below 1e-19; a
// larger A is halved until |A|_F <= 1 and the exponential squared back.
__global__ void __launch_bounds__(HMC_BLOCK) exp_update_kernel(void* U, const void* P, Geom g, double eps) {
  const int64_t t = (int64_t)blockIdx.x * HMC_BLOCK + threadIdx.x;
  if (t >= 8 * (int64_t)g.Vh) return;
  const int blk = (int)(t / g.Vh);  // parity * 4 + mu
  const int64_t cb = t - (int64_t)blk * g.Vh;
  M3 p, E, u, w;
  LinkIO<LQCD_F64, 18>::load(P, g.gstride, blk, cb, p);
  const int s = is_hermitian(p) ? exp_hermitian(p, eps, E) : exp_general(p, eps, E);
  for (int k = 0; k < s; k++) {
    m_mul(E, E, w);
    E = w;
  }
  LinkIO<LQCD_F64, 18>::load(U, g.gstride, blk, cb, u);
  m_mul(E, u, w);
  double2* base = static_cast<double2*>(U) + (int64_t)blk * 9 * g.gstride + cb;
#pragma unroll
  for (int k = 0; k < 9; k++) base[k * g.gstride] = make_double2(w.v[k].r, w.v[k].i);
}

// sum over the 4 links of a site of tr(P^2) / 2 = |P|_F^2 / 2 (P Hermitian), reduced
__global__ void __launch_bounds__(HMC_BLOCK) kinetic_kernel(const void* P, Geom g, ReduceCtx rc) {
  const int64_t t = (int64_t)blockIdx.x * HMC_BLOCK + threadIdx.x;
  double v = 0.0;
  if (t < 2 * (int64_t)g.Vh) {
    const int parity = t >= g.Vh ? 1 : 0;
    const int64_t cb = t - parity * (int64_t)g.Vh;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
      M3 p;
      LinkIO<LQCD_F64, 18>::load(P, g.gstride, parity * 4 + mu, cb, p);
#pragma unroll
      for (int k = 0; k < 9; k++) s[mu] = fma(p.v[k].r, p.v[k].r, fma(p.v[k].i, p.v[k].i, s[mu]));
    }
    v = 0.5 * ((s[0] + s[1]) + (s[2] + s[3]));
  }
  block_reduce_finalize<HMC_BLOCK>(v, (int64_t)blockIdx.x * HMC_BLOCK, rc);
}

// Re <a, b> of two FP64 full spinor fields (n5 == 1), reduced
__global__ void __launch_bounds__(HMC_BLOCK) dot_kernel(const void* a, const void* b, Geom g, int64_t half_bytes,
                                                        ReduceCtx rc) {
  const int64_t t = (int64_t)blockIdx.x * HMC_BLOCK + threadIdx.x;
  double v = 0.0;
  if (t < 2 * (int64_t)g.Vh) {
    const int parity = t >= g.Vh ? 1 : 0;
    const int64_t cb = t - parity * (int64_t)g.Vh;
    Spinor<double> x, y;
    SpinorIO<LQCD_F64>::load(static_cast<const char*>(a) + parity * half_bytes, g.sstride, cb, x);
    SpinorIO<LQCD_F64>::load(static_cast<const char*>(b) + parity * half_bytes, g.sstride, cb, y);
#pragma unroll
    for (int k = 0; k < 12; k++) v += x.v[k].r * y.v[k].r + x.v[k].i * y.v[k].i;
  }
  block_reduce_finalize<HMC_BLOCK>(v, (int64_t)blockIdx.x * HMC_BLOCK, rc);
}

// ------------------------------------------------------------------ host helpers

static unsigned site_grid(const Geom& g) { return (unsigned)((2 * (int64_t)g.Vh + HMC_BLOCK - 1) / HMC_BLOCK); }
static unsigned plaq_grid(const Geom& g) { return (unsigned)((2 * (int64_t)g.Vh + PLAQ_SITES - 1) / PLAQ_SITES); }
static unsigned link_grid(const Geom& g) { return (unsigned)((8 * (int64_t)g.Vh + HMC_BLOCK - 1) / HMC_BLOCK); }

// Reduction scratch: result (1 double), counter, partials (one per block of the
// finest grid, the plaquette's).
struct ReduceWs {
  double* result;
  unsigned int* counter;
  double* partials;
};
static size_t reduce_ws_bytes(const Geom& g) { return 256 + 256 + (size_t)round_up(8 * (int64_t)plaq_grid(g), 256); }
static ReduceWs reduce_ws(void* base) {
  char* b = static_cast<char*>(base);
  return ReduceWs{reinterpret_cast<double*>(b), reinterpret_cast<unsigned int*>(b + 256),
                  reinterpret_cast<double*>(b + 512)};
}
static ReduceCtx reduce_ctx(const ReduceWs& w) {
  ReduceCtx rc;
  memset(&rc, 0, sizeof(rc));
  rc.partials = w.partials;
  rc.counter = w.counter;
  rc.result = w.result;
  rc.nsys = 1;
  rc.fin = FIN_STORE;
  return rc;
}
static int read_result(const ReduceWs& w, double* out, cudaStream_t s) {
  cudaError_t e = cudaMemcpyAsync(out, w.result, sizeof(double), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(e, "hmc: reduction readback");
  return LQCD_OK;
}
static int zero_counter(const ReduceWs& w, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(w.counter, 0, sizeof(unsigned int), s);
  return e == cudaSuccess ? LQCD_OK : cuda_fail(e, "hmc: memset");
}

static int plaquette(const Geom& g, const void* U, const ReduceWs& w, double* out, cudaStream_t s) {
  plaquette_kernel<<<plaq_grid(g), HMC_BLOCK, 0, s>>>(U, g, reduce_ctx(w));
  int st = after_launch("plaquette_kernel");
  if (st || (st = read_result(w, out, s))) return st;
  *out /= 6.0 * 2.0 * (double)g.Vh;
  return LQCD_OK;
}
static int kinetic(const Geom& g, const void* P, const ReduceWs& w, double* out, cudaStream_t s) {
  kinetic_kernel<<<site_grid(g), HMC_BLOCK, 0, s>>>(P, g, reduce_ctx(w));
  int st = after_launch("kinetic_kernel");
  if (st) return st;
  return read_result(w, out, s);
}
static int gauge_force(const Geom& g, double2* out, const void* U, double beta, double coef, int acc,
                       cudaStream_t s) {
  const unsigned grid = (unsigned)((2 * (int64_t)g.Vh + GF_SITES - 1) / GF_SITES);
  gauge_force_kernel<<<grid, HMC_BLOCK, 0, s>>>(out, U, g, beta, coef, acc);
  return after_launch("gauge_force_kernel");
}
static int exp_update(const Geom& g, void* U, const void* P, double eps, cudaStream_t s) {
  exp_update_kernel<<<link_grid(g), HMC_BLOCK, 0, s>>>(U, P, g, eps);
  return after_launch("exp_update_kernel");
}

static bool mis16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) != 0; }

// ------------------------------------------------------------------ trajectory

struct HmcWs {
  ReduceWs red;
  void* X;        // FP64 full spinor
  void* Y;        // FP64 full spinor
  double* stage;  // host-layout FP64 gauge field (sloppy link refresh)
  void* gs;       // sloppy gauge field
  void* cg;       // CG workspace
  size_t cg_bytes;
  size_t total;
};

static HmcWs carve(void* base, const Geom& g, const lqcd_lattice* lat, const lqcd_operator* op,
                   const lqcd_solver_params* prm) {
  HmcWs w;
  memset(&w, 0, sizeof(w));
  size_t o = 0;
  char* b = static_cast<char*>(base);
  auto take = [&](size_t bytes) -> void* {
    void* r = b ? b + o : nullptr;
    o += round_up((int64_t)bytes, 256);
    return r;
  };
  w.red = reduce_ws(take(reduce_ws_bytes(g)));
  const size_t sp = 2 * cb_spinor_bytes(g, LQCD_F64);
  w.X = take(sp);
  w.Y = take(sp);
  if (prm->sloppy_prec != LQCD_F64) {
    w.stage = static_cast<double*>(take((size_t)8 * g.Vh * 18 * sizeof(double)));
    w.gs = take(lqcd_gauge_bytes(lat, prm->sloppy_prec, prm->sloppy_recon));
  }
  w.cg_bytes = lqcd_cg_workspace_bytes(lat, op, prm, LQCD_FULL);
  w.cg = take(w.cg_bytes);
  w.total = o;
  return w;
}

struct Trajectory {
  Geom g;
  const lqcd_lattice* lat;
  const lqcd_operator* op;
  const lqcd_hmc_params* hp;
  const lqcd_solver_params* sp;
  void* U;
  void* P;
  const void* phi;
  HmcWs w;
  cudaStream_t s;
  lqcd_hmc_info* info;

  // X = (M^dag M)^-1 phi on the full lattice; S_f = Re <phi, X>
  int solve(double* sf) {
    const void* gsl = U;
    if (sp->sloppy_prec != LQCD_F64) {
      int st = lqcd_gauge_unpack(w.stage, U, LQCD_F64, 18, lat, s);
      if (st || (st = lqcd_gauge_pack(w.gs, sp->sloppy_prec, sp->sloppy_recon, w.stage, lat, s))) return st;
      gsl = w.gs;
    }
    lqcd_solve_info ci;
    int st = lqcd_cg_solve(w.X, phi, U, gsl, lat, op, sp, LQCD_FULL, &ci, w.cg, w.cg_bytes, s);
    info->cg_iterations += ci.iterations;
    if (st) return st;
    if (sf) {
      if ((st = zero_counter(w.red, s))) return st;
      dot_kernel<<<site_grid(g), HMC_BLOCK, 0, s>>>(phi, w.X, g, (int64_t)cb_spinor_bytes(g, LQCD_F64),
                                                    reduce_ctx(w.red));
      if ((st = after_launch("dot_kernel")) || (st = read_result(w.red, sf, s))) return st;
    }
    return LQCD_OK;
  }

  int energy(double* H, double* K, double* Sg, double* Sf) {
    int st = zero_counter(w.red, s);
    if (st || (st = kinetic(g, P, w.red, K, s))) return st;
    double plaq;
    if ((st = zero_counter(w.red, s)) || (st = plaquette(g, U, w.red, &plaq, s))) return st;
    *Sg = hp->beta * 6.0 * 2.0 * (double)g.Vh * (1.0 - plaq);
    *Sf = 0.0;
    if (hp->fermion && (st = solve(Sf))) return st;
    *H = *K + *Sg + *Sf;
    return LQCD_OK;
  }

  // P <- P - h (F_g + F_f)
  int kick(double h) {
    info->force_evaluations += 1;
    int st = gauge_force(g, static_cast<double2*>(P), U, hp->beta, h, 1, s);
    if (st || !hp->fermion) return st;
    if ((st = solve(nullptr))) return st;
    if ((st = lqcd_M(w.Y, w.X, U, lat, op, LQCD_FULL, 0, nullptr, s))) return st;
    return force_accumulate(static_cast<double2*>(P), U, w.X, w.Y, g, op->recon, h, s);
  }

  int drift(double h) { return exp_update(g, U, P, h, s); }

  int run() {
    int st = energy(&info->H0, &info->kinetic0, &info->gauge0, &info->fermion0);
    if (st) return st;
    const int n = hp->nsteps;
    const double eps = hp->tau / n;
    if (hp->integrator == LQCD_LEAPFROG) {
      if ((st = kick(0.5 * eps))) return st;
      for (int k = 0; k < n; k++) {
        if ((st = drift(eps))) return st;
        if ((st = kick(k < n - 1 ? eps : 0.5 * eps))) return st;
      }
    } else {
      const double lam = 0.1931833275037836;  // Omelyan, Mryglod and Folk (2003)
      if ((st = kick(lam * eps))) return st;
      for (int k = 0; k < n; k++) {
        if ((st = drift(0.5 * eps))) return st;
        if ((st = kick((1.0 - 2.0 * lam) * eps))) return st;
        if ((st = drift(0.5 * eps))) return st;
        if ((st = kick(k < n - 1 ? 2.0 * lam * eps : lam * eps))) return st;
      }
    }
    return energy(&info->H1, &info->kinetic1, &info->gauge1, &info->fermion1);
  }
};

static int hmc_validate(const lqcd_lattice* lat, const lqcd_operator* op, const lqcd_solver_params* prm,
                        Geom* g) {
  int st = make_geom(lat, g);
  if (st) return st;
  if (g->n5 != 1) return fail(LQCD_ERR_ARG, "hmc: n5 must be 1");
  if (!op || !prm) return fail(LQCD_ERR_ARG, "hmc: null operator or solver parameters");
  if ((st = check_operator(op, *g))) return st;
  if (op->kind != LQCD_WILSON || op->prec != LQCD_F64 || op->recon != 18)
    return fail(LQCD_ERR_UNSUPPORTED, "hmc: Wilson operator with FP64, 18-real links");
  if (prm->sloppy_prec != LQCD_F64 && prm->sloppy_prec != LQCD_F32)
    return fail(LQCD_ERR_UNSUPPORTED, "hmc: sloppy precision must be LQCD_F64 or LQCD_F32");
  if (lqcd_cg_workspace_bytes(lat, op, prm, LQCD_FULL) == 0) return fail(LQCD_ERR_ARG, "hmc: bad solver parameters");
  return LQCD_OK;
}

}  // namespace lqcd

using namespace lqcd;

extern "C" {

size_t lqcd_reduce_workspace_bytes(const lqcd_lattice* lat) {
  Geom g;
  if (make_geom(lat, &g) != LQCD_OK) return 0;
  return reduce_ws_bytes(g);
}

int lqcd_plaquette(double* plaq, const void* U, const lqcd_lattice* lat, void* ws, size_t ws_bytes, void* stream) {
  Geom g;
  int st = make_geom(lat, &g);
  if (st) return st;
  if (!plaq || !U || !ws || mis16(U) || ((uintptr_t)ws & 255)) return fail(LQCD_ERR_ARG, "lqcd_plaquette: pointer");
  if (ws_bytes < reduce_ws_bytes(g)) return fail(LQCD_ERR_WORKSPACE, "lqcd_plaquette: workspace too small");
  cudaStream_t s = (cudaStream_t)stream;
  const ReduceWs w = reduce_ws(ws);
  if ((st = zero_counter(w, s))) return st;
  return plaquette(g, U, w, plaq, s);
}

int lqcd_spinor_dot_re(double* result, const void* a, const void* b, const lqcd_lattice* lat, void* ws,
                       size_t ws_bytes, void* stream) {
  Geom g;
  int st = make_geom(lat, &g);
  if (st) return st;
  if (g.n5 != 1) return fail(LQCD_ERR_UNSUPPORTED, "lqcd_spinor_dot_re: n5 must be 1");
  if (!result || !a || !b || !ws || mis16(a) || mis16(b) || ((uintptr_t)ws & 255))
    return fail(LQCD_ERR_ARG, "lqcd_spinor_dot_re: pointer");
  if (ws_bytes < reduce_ws_bytes(g)) return fail(LQCD_ERR_WORKSPACE, "lqcd_spinor_dot_re: workspace too small");
  cudaStream_t s = (cudaStream_t)stream;
  const ReduceWs w = reduce_ws(ws);
  if ((st = zero_counter(w, s))) return st;
  dot_kernel<<<site_grid(g), HMC_BLOCK, 0, s>>>(a, b, g, (int64_t)cb_spinor_bytes(g, LQCD_F64), reduce_ctx(w));
  if ((st = after_launch("dot_kernel"))) return st;
  return read_result(w, result, s);
}

int lqcd_momentum_kinetic(double* kin, const void* P, const lqcd_lattice* lat, void* ws, size_t ws_bytes,
                          void* stream) {
  Geom g;
  int st = make_geom(lat, &g);
  if (st) return st;
  if (!kin || !P || !ws || mis16(P) || ((uintptr_t)ws & 255))
    return fail(LQCD_ERR_ARG, "lqcd_momentum_kinetic: pointer");
  if (ws_bytes < reduce_ws_bytes(g)) return fail(LQCD_ERR_WORKSPACE, "lqcd_momentum_kinetic: workspace too small");
  cudaStream_t s = (cudaStream_t)stream;
  const ReduceWs w = reduce_ws(ws);
  if ((st = zero_counter(w, s))) return st;
  return kinetic(g, P, w, kin, s);
}

int lqcd_gauge_force(void* out, const void* U, const lqcd_lattice* lat, double beta, void* stream) {
  Geom g;
  int st = make_geom(lat, &g);
  if (st) return st;
  if (!out || !U || mis16(out) || mis16(U) || out == U) return fail(LQCD_ERR_ARG, "lqcd_gauge_force: pointer");
  return gauge_force(g, static_cast<double2*>(out), U, beta, 0.0, 0, (cudaStream_t)stream);
}

int lqcd_gauge_exp_update(void* U, const void* P, double eps, const lqcd_lattice* lat, void* stream) {
  Geom g;
  int st = make_geom(lat, &g);
  if (st) return st;
  if (!U || !P || mis16(U) || mis16(P) || U == P) return fail(LQCD_ERR_ARG, "lqcd_gauge_exp_update: pointer");
  return exp_update(g, U, P, eps, (cudaStream_t)stream);
}

size_t lqcd_hmc_workspace_bytes(const lqcd_lattice* lat, const lqcd_operator* op, const lqcd_solver_params* prm) {
  Geom g;
  if (hmc_validate(lat, op, prm, &g) != LQCD_OK) return 0;
  return carve(nullptr, g, lat, op, prm).total;
}

int lqcd_hmc_trajectory(void* U, void* P, const void* phi, const lqcd_lattice* lat, const lqcd_operator* op,
                        const lqcd_hmc_params* hp, const lqcd_solver_params* prm, lqcd_hmc_info* info, void* ws,
                        size_t ws_bytes, void* stream) {
  lqcd_hmc_info local;
  lqcd_hmc_info* inf = info ? info : &local;
  memset(inf, 0, sizeof(*inf));
  Geom g;
  int st = hmc_validate(lat, op, prm, &g);
  if (!st && !hp) st = fail(LQCD_ERR_ARG, "hmc: null parameters");
  if (!st && (hp->nsteps < 1 || !(hp->tau > 0.0) || (hp->integrator != LQCD_LEAPFROG &&
                                                     hp->integrator != LQCD_MINNORM2)))
    st = fail(LQCD_ERR_ARG, "hmc: nsteps >= 1, tau > 0 and a known integrator required");
  if (!st && (!U || !P || mis16(U) || mis16(P) || (hp->fermion && (!phi || mis16(phi)))))
    st = fail(LQCD_ERR_ARG, "hmc: null or misaligned field");
  if (!st && (!ws || ((uintptr_t)ws & 255))) st = fail(LQCD_ERR_ARG, "hmc: workspace must be 256-byte aligned");
  Trajectory T;
  if (!st) {
    T.w = carve(ws, g, lat, op, prm);
    if (ws_bytes < T.w.total) st = fail(LQCD_ERR_WORKSPACE, "hmc: workspace %zu < %zu bytes", ws_bytes, T.w.total);
  }
  if (!st) {
    T.g = g;
    T.lat = lat;
    T.op = op;
    T.hp = hp;
    T.sp = prm;
    T.U = U;
    T.P = P;
    T.phi = phi;
    T.s = (cudaStream_t)stream;
    T.info = inf;
    st = T.run();
  }
  inf->status = st;
  return st;
}

}  // extern "C"
