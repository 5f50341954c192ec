// Pseudofermion force for S = phi^dag (M^dag M)^-1 phi, M = D_W.
//
// The Grid paper lists HMC among its algorithms (Sec. 4); the force formula
// is the textbook derivative. With X = (M^dag M)^-1 phi and Y = M X, the only
// terms of dS that involve the link U_mu(x) are the two hops through it:
//   dS = ph Re[ tr(dU A) + tr(dU^dag B) ],
//   A = sum_spin X(x+mu) ((1 - gamma_mu) Y(x))^dag,
//   B = sum_spin ((1 + gamma_mu) X(x)) Y(x+mu)^dag,
// ph = the link's boundary phase. Because (1 -+ gamma) has rank two, each sum
// is two colour outer products of half spinors: A = sum_a g_a h_a^dag with g,
// h the (1 - gamma_mu) projections of X(x+mu) and Y(x) (and likewise B with
// 1 + gamma_mu), which the kernel forms with the same projection code as the
// hop. Outputs per link: the conjugate-Wirtinger gradient A^dag + B, or the
// traceless Hermitian force TA[i (G - G^dag) / 2] with G = U A - B U^dag.
#include "lqcd_internal.h"

namespace lqcd {

constexpr int FORCE_SITES = 32;  // sites per block, one per lane; warp mu computes their links mu
constexpr int FORCE_BLOCK = 4 * FORCE_SITES;

struct ForceArgs {
  double2* out;
  const void* gauge;
  const void* X;
  const void* Y;
  Geom g;
  int64_t half_bytes;
  int kind;
  int accumulate;  // 1: out -= coef * force (molecular-dynamics momentum update)
  double coef;
};

// M = sum_a g_a h_a^dag (colour outer products of two half spinors)
__device__ __forceinline__ void outer(const Half<double>& g, const Half<double>& h, cpx<double> m[9]) {
#pragma unroll
  for (int r = 0; r < 3; r++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      cpx<double> s = cmadd_conj(mk(0.0, 0.0), h.v[c], g.v[r]);
      m[3 * r + c] = cmadd_conj(s, h.v[3 + c], g.v[3 + r]);
    }
}

// im += Im(p conj(q)) and re += Re(p conj(q)), with the sign of S
template <int S> __device__ __forceinline__ void add_im(double& im, cpx<double> p, cpx<double> q) {
  im = S > 0 ? fma(p.i, q.r, fma(-p.r, q.i, im)) : fma(-p.i, q.r, fma(p.r, q.i, im));
}
template <int S> __device__ __forceinline__ void add_re(double& re, cpx<double> p, cpx<double> q) {
  re = S > 0 ? fma(p.r, q.r, fma(p.i, q.i, re)) : fma(-p.r, q.r, fma(-p.i, q.i, re));
}

// The force is bound by the FP64 pipe, so the traceless-Hermitian kind is
// arranged for the fewest FP64 instructions: U A = sum_a (U g_a) h_a^dag and
// B U^dag = sum_a g_a (U h_a)^dag multiply half spinors instead of matrices,
// and of G = U A - B U^dag only i (G - G^dag) / 2 is accumulated: about 340
// instructions per link against 520 with the two outer products multiplied by
// U. One warp per direction of 32 sites: four times as many, shorter, work
// items than a thread per site, so that the SMs end together, and the spinors
// at the site reach the other three warps through L1. 24^3 x 32 on GB300:
// 1,622 -> 1,002 us.
template <int MU, int R, int KIND>
__device__ __forceinline__ void force_dir(const ForceArgs& a, const Coord& x, int64_t cb, int parity) {
  bool wrap;
  const int64_t nb = neighbour_cb<MU>(a.g, x, +1, wrap);
  const char* X = static_cast<const char*>(a.X);
  const char* Y = static_cast<const char*>(a.Y);
  Half<double> ga, ha, gb, hb;
  {
    Spinor<double> s;
    SpinorIO<LQCD_F64>::load(X + (1 - parity) * a.half_bytes, a.g.sstride, nb, s);
    project<MU, -1>(s, ga);
    SpinorIO<LQCD_F64>::load(Y + parity * a.half_bytes, a.g.sstride, cb, s);
    project<MU, -1>(s, ha);
    SpinorIO<LQCD_F64>::load(X + parity * a.half_bytes, a.g.sstride, cb, s);
    project<MU, +1>(s, gb);
    SpinorIO<LQCD_F64>::load(Y + (1 - parity) * a.half_bytes, a.g.sstride, nb, s);
    project<MU, +1>(s, hb);
  }
  const double ph = wrap ? a.g.bcd[MU] : 1.0;
  cpx<double> out[9];
  if (KIND == LQCD_FORCE_GRAD) {
    cpx<double> A[9], B[9];
    outer(ga, ha, A);
    outer(gb, hb, B);
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
      for (int c = 0; c < 3; c++) out[3 * r + c] = ph * (conj(A[3 * c + r]) + B[3 * r + c]);
  } else {
    Half<double> v, w;  // U g and U h of the two terms
    {
      Link<double> u;
      LinkIO<LQCD_F64, R>::load(a.gauge, a.g.gstride, parity * 4 + MU, cb, u);
      link_mul(u, ga, v);
      link_mul(u, hb, w);
    }
    // F = i (G - G^dag) / 2 with G_rc = sum_a v_a(r) conj(ha_a(c)) - gb_a(r) conj(w_a(c)): F_rr = -Im G_rr,
    // F_rc = (-(Im G_rc + Im G_cr) + i (Re G_rc - Re G_cr)) / 2; then remove the trace
    double d[3];
#pragma unroll
    for (int r = 0; r < 3; r++) {
      d[r] = 0.0;
#pragma unroll
      for (int s = 0; s < 6; s += 3) {
        add_im<-1>(d[r], v.v[s + r], ha.v[s + r]);
        add_im<+1>(d[r], gb.v[s + r], w.v[s + r]);
      }
    }
    const double tr = (d[0] + d[1] + d[2]) * (1.0 / 3.0);
#pragma unroll
    for (int r = 0; r < 3; r++) out[4 * r] = mk(ph * (d[r] - tr), 0.0);
    const double hp = 0.5 * ph;
#pragma unroll
    for (int e = 0; e < 3; e++) {
      const int r = e == 2 ? 1 : 0, c = e == 0 ? 1 : 2;
      double re = 0.0, im = 0.0;
#pragma unroll
      for (int s = 0; s < 6; s += 3) {
        add_im<-1>(re, v.v[s + r], ha.v[s + c]);
        add_im<-1>(re, v.v[s + c], ha.v[s + r]);
        add_im<+1>(re, gb.v[s + r], w.v[s + c]);
        add_im<+1>(re, gb.v[s + c], w.v[s + r]);
        add_re<+1>(im, v.v[s + r], ha.v[s + c]);
        add_re<-1>(im, v.v[s + c], ha.v[s + r]);
        add_re<-1>(im, gb.v[s + r], w.v[s + c]);
        add_re<+1>(im, gb.v[s + c], w.v[s + r]);
      }
      out[3 * r + c] = mk(hp * re, hp * im);
      out[3 * c + r] = conj(out[3 * r + c]);
    }
  }
  double2* o = a.out + (int64_t)(parity * 4 + MU) * 9 * a.g.gstride + cb;
  if (a.accumulate) {
#pragma unroll
    for (int k = 0; k < 9; k++) {
      const double2 w = o[k * a.g.gstride];
      o[k * a.g.gstride] = make_double2(fma(-a.coef, out[k].r, w.x), fma(-a.coef, out[k].i, w.y));
    }
  } else {
#pragma unroll
    for (int k = 0; k < 9; k++) o[k * a.g.gstride] = make_double2(out[k].r, out[k].i);
  }
}

template <int R, int KIND>
__global__ void __launch_bounds__(FORCE_BLOCK) force_kernel(const ForceArgs a) {
  const int64_t t = (int64_t)blockIdx.x * FORCE_SITES + (threadIdx.x & (FORCE_SITES - 1));
  if (t >= 2 * (int64_t)a.g.Vh) return;
  const int parity = t >= a.g.Vh ? 1 : 0;
  const int64_t cb = t - parity * (int64_t)a.g.Vh;
  const Coord x = cb_to_coord(a.g, cb, parity);
  switch (threadIdx.x / FORCE_SITES) {
    case 0: force_dir<0, R, KIND>(a, x, cb, parity); break;
    case 1: force_dir<1, R, KIND>(a, x, cb, parity); break;
    case 2: force_dir<2, R, KIND>(a, x, cb, parity); break;
    default: force_dir<3, R, KIND>(a, x, cb, parity);
  }
}

static int launch_force(const ForceArgs& a, int recon, cudaStream_t s) {
  const unsigned grid = (unsigned)((2 * (int64_t)a.g.Vh + FORCE_SITES - 1) / FORCE_SITES);
  // the gradient kind reads no links, so both link formats share its instantiation
  if (a.kind == LQCD_FORCE_GRAD) force_kernel<18, LQCD_FORCE_GRAD><<<grid, FORCE_BLOCK, 0, s>>>(a);
  else if (recon == 18) force_kernel<18, LQCD_FORCE_TA><<<grid, FORCE_BLOCK, 0, s>>>(a);
  else force_kernel<12, LQCD_FORCE_TA><<<grid, FORCE_BLOCK, 0, s>>>(a);
  return after_launch("force_kernel");
}

int force_accumulate(double2* mom, const void* gauge, const void* X, const void* Y, const Geom& g, int recon,
                     double coef, cudaStream_t s) {
  ForceArgs a{mom, gauge, X, Y, g, (int64_t)cb_spinor_bytes(g, LQCD_F64), LQCD_FORCE_TA, 1, coef};
  return launch_force(a, recon, s);
}

}  // namespace lqcd

using namespace lqcd;

extern "C" int lqcd_force(void* out, const void* gauge, const void* X, const void* Y, const lqcd_lattice* lat,
                          const lqcd_operator* op, int kind, void* stream) {
  Geom g;
  int st = make_geom(lat, &g);
  if (st) return st;
  if ((st = check_operator(op, g))) return st;
  if (op->kind != LQCD_WILSON || op->prec != LQCD_F64 || g.n5 != 1)
    return fail(LQCD_ERR_UNSUPPORTED, "lqcd_force: Wilson operator, LQCD_F64 and n5 == 1 only");
  if (kind != LQCD_FORCE_TA && kind != LQCD_FORCE_GRAD) return fail(LQCD_ERR_ARG, "lqcd_force: bad kind %d", kind);
  if (!out || !gauge || !X || !Y || (((uintptr_t)out | (uintptr_t)gauge | (uintptr_t)X | (uintptr_t)Y) & 15))
    return fail(LQCD_ERR_ARG, "lqcd_force: null or misaligned pointer");
  ForceArgs a{static_cast<double2*>(out), gauge, X, Y, g, (int64_t)cb_spinor_bytes(g, LQCD_F64), kind, 0, 0.0};
  return launch_force(a, op->recon, (cudaStream_t)stream);
}
