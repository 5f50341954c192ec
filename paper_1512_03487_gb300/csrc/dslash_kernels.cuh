// Fused Wilson hopping kernel (and its L_s-replicated / multi-RHS form).
//
//   out(x) = sum_mu (1 - gamma_mu) U_mu(x) in(x + mu) + (1 + gamma_mu) U_mu(x - mu)^dag in(x - mu)
//
// One thread per output site j = cb * n5 + i5 of one checkerboard. For each
// of the 8 directions the neighbour spinor is loaded (coalesced SoA chunks),
// spin-projected to a half spinor (the paper's Compressor, Sec. 2.6, applied
// in registers instead of to a halo), multiplied by the SU(3) link (2 colour
// vectors), reconstructed to 4 spins and accumulated; the result is written
// once with streaming stores (Sec. 2.6 "streaming stores are used in the
// final write"). With n5 > 1 the n5 threads of a 4D site read the same link
// address, so the link bytes are fetched once per site for all i5 (the
// paper's L_s-fold gauge reuse, Sec. 3 Fig. xc30 caption).
//
// Gamma basis (chiral): gamma_mu = [[0, B_mu], [B_mu^dag, 0]] with
// B_x = -i sigma_1, B_y = -i sigma_2, B_z = -i sigma_3, B_t = 1. For
// (1 + S gamma_mu) psi (S = +-1) the upper half is h = psi_u + S B psi_l and
// the lower half is S B^dag h, so only h is multiplied by the link.
#pragma once

#include "cg_site.cuh"
#include "hop_pair.cuh"
#include "lqcd_common.cuh"
#include "m5_scan.cuh"

namespace lqcd {

// EPI_M5INV: out = M5op^-1 (b H in), the inverse applied across the L_s lanes of
// each 4D site by the warp-shuffle scan (domain wall, L_s dividing 32).
enum Epilogue { EPI_PLAIN = 0, EPI_XPAY = 1, EPI_M5 = 2, EPI_M5INV = 3 };

struct HopArgs {
  void* out;
  const void* in;
  const void* gauge;
  const void* x;          // epilogue operand, same format and subset as out
  Geom g;
  int out_parity;         // single-checkerboard launch: parity of out
  int full;               // 1: out / in / x are full fields, grid covers both parities
  int blocks_per_parity;
  int64_t half_bytes;     // bytes of one checkerboard of a full field
  double a, b;            // EPI_PLAIN: out = b H in; EPI_XPAY: out = a x + b H in
  double m5d, mf;         // EPI_M5: out = M5op(x) + b H in, M5op diagonal m5d = 5 - M5
  int m5_dagger;          // EPI_M5INV: apply the adjoint of M5op^-1
  double m5_a;            // EPI_M5INV: 1 / (5 - M5)
  double m5_den_inv;      // EPI_M5INV: 1 / (1 + mf (5 - M5)^-L_s)
  float af, bf, m5df, mff, m5_af, m5_den_invf;  // the same rounded once on the host (set_float_coefs): a
                          // conversion in the kernel is an FP64-pipe instruction per thread
  ReduceCtx red;          // |out|^2 per system (RED_NORM) or |r_s|^2 (RED_CG_UPDATE)
  const Control* gate;    // kernel returns at once when gate->active == 0
  // RED_CG_UPDATE: out = A p is not stored; instead x_s += alpha p and
  // r_s -= alpha A p, alpha = red.sys[system].alpha. p is in the format of
  // out; x_s and r_s in vec_prec of it (upd_half_bytes: one checkerboard).
  const void* upd_p;
  void* upd_xs;
  void* upd_rs;             // in rs_prec of out's format
  int64_t upd_half_bytes;
  int64_t upd_rs_half_bytes;
};

inline void set_float_coefs(HopArgs& h) {
  h.af = (float)h.a;
  h.bf = (float)h.b;
  h.m5df = (float)h.m5d;
  h.mff = (float)h.mf;
  h.m5_af = (float)h.m5_a;
  h.m5_den_invf = (float)h.m5_den_inv;
}

// Reduction / epilogue modes of the hop kernel.
enum HopReduce { RED_NONE = 0, RED_NORM = 1, RED_CG_UPDATE = 2 };

template <int MU, int S, typename T>
__device__ __forceinline__ void project(const Spinor<T>& s, Half<T>& h) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const cpx<T> p0 = s.v[c], p1 = s.v[3 + c], p2 = s.v[6 + c], p3 = s.v[9 + c];
    cpx<T> h0, h1;
    if (MU == 0) {         // h0 = p0 - S i p3, h1 = p1 - S i p2
      h0 = S > 0 ? p0 + times_mi(p3) : p0 + times_i(p3);
      h1 = S > 0 ? p1 + times_mi(p2) : p1 + times_i(p2);
    } else if (MU == 1) {  // h0 = p0 - S p3, h1 = p1 + S p2
      h0 = S > 0 ? p0 - p3 : p0 + p3;
      h1 = S > 0 ? p1 + p2 : p1 - p2;
    } else if (MU == 2) {  // h0 = p0 - S i p2, h1 = p1 + S i p3
      h0 = S > 0 ? p0 + times_mi(p2) : p0 + times_i(p2);
      h1 = S > 0 ? p1 + times_i(p3) : p1 + times_mi(p3);
    } else {               // h0 = p0 + S p2, h1 = p1 + S p3
      h0 = S > 0 ? p0 + p2 : p0 - p2;
      h1 = S > 0 ? p1 + p3 : p1 - p3;
    }
    h.v[c] = h0;
    h.v[3 + c] = h1;
  }
}

// acc += (upper = w, lower = S B_mu^dag w)
template <int MU, int S, typename T>
__device__ __forceinline__ void accumulate(Spinor<T>& acc, const Half<T>& w) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const cpx<T> w0 = w.v[c], w1 = w.v[3 + c];
    acc.v[c] = acc.v[c] + w0;
    acc.v[3 + c] = acc.v[3 + c] + w1;
    if (MU == 0) {         // lower2 = S i w1, lower3 = S i w0
      acc.v[6 + c] = acc.v[6 + c] + (S > 0 ? times_i(w1) : times_mi(w1));
      acc.v[9 + c] = acc.v[9 + c] + (S > 0 ? times_i(w0) : times_mi(w0));
    } else if (MU == 1) {  // lower2 = S w1, lower3 = -S w0
      acc.v[6 + c] = S > 0 ? acc.v[6 + c] + w1 : acc.v[6 + c] - w1;
      acc.v[9 + c] = S > 0 ? acc.v[9 + c] - w0 : acc.v[9 + c] + w0;
    } else if (MU == 2) {  // lower2 = S i w0, lower3 = -S i w1
      acc.v[6 + c] = acc.v[6 + c] + (S > 0 ? times_i(w0) : times_mi(w0));
      acc.v[9 + c] = acc.v[9 + c] + (S > 0 ? times_mi(w1) : times_i(w1));
    } else {               // lower2 = S w0, lower3 = S w1
      acc.v[6 + c] = S > 0 ? acc.v[6 + c] + w0 : acc.v[6 + c] - w0;
      acc.v[9 + c] = S > 0 ? acc.v[9 + c] + w1 : acc.v[9 + c] - w1;
    }
  }
}

// acc + f a and acc + f (i a), one fused multiply-add per real component
template <typename T> __device__ __forceinline__ cpx<T> fmacc(cpx<T> acc, T f, cpx<T> a) {
  return mk(fma(f, a.r, acc.r), fma(f, a.i, acc.i));
}
template <typename T> __device__ __forceinline__ cpx<T> fmacc_i(cpx<T> acc, T f, cpx<T> a) {
  return mk(fma(-f, a.i, acc.r), fma(f, a.r, acc.i));
}

// acc += f (upper = w, lower = S B_mu^dag w): the factor f (boundary phase and,
// for FP16 storage, the neighbour's site norm) rides on the accumulation FMAs.
template <int MU, int S, typename T>
__device__ __forceinline__ void accumulate_scaled(Spinor<T>& acc, const Half<T>& w, T f) {
  const T fs = S > 0 ? f : -f;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const cpx<T> w0 = w.v[c], w1 = w.v[3 + c];
    acc.v[c] = fmacc(acc.v[c], f, w0);
    acc.v[3 + c] = fmacc(acc.v[3 + c], f, w1);
    if (MU == 0) {         // lower2 = S i w1, lower3 = S i w0
      acc.v[6 + c] = fmacc_i(acc.v[6 + c], fs, w1);
      acc.v[9 + c] = fmacc_i(acc.v[9 + c], fs, w0);
    } else if (MU == 1) {  // lower2 = S w1, lower3 = -S w0
      acc.v[6 + c] = fmacc(acc.v[6 + c], fs, w1);
      acc.v[9 + c] = fmacc(acc.v[9 + c], -fs, w0);
    } else if (MU == 2) {  // lower2 = S i w0, lower3 = -S i w1
      acc.v[6 + c] = fmacc_i(acc.v[6 + c], fs, w0);
      acc.v[9 + c] = fmacc_i(acc.v[9 + c], -fs, w1);
    } else {               // lower2 = S w0, lower3 = S w1
      acc.v[6 + c] = fmacc(acc.v[6 + c], fs, w0);
      acc.v[9 + c] = fmacc(acc.v[9 + c], fs, w1);
    }
  }
}

// w_a = U h_a
template <typename T>
__device__ __forceinline__ void link_mul(const Link<T>& u, const Half<T>& h, Half<T>& w) {
#pragma unroll
  for (int a = 0; a < 2; a++)
#pragma unroll
    for (int r = 0; r < 3; r++) {
      cpx<T> s = cmul(u.v[3 * r], h.v[3 * a]);
      s = cmadd(s, u.v[3 * r + 1], h.v[3 * a + 1]);
      s = cmadd(s, u.v[3 * r + 2], h.v[3 * a + 2]);
      w.v[3 * a + r] = s;
    }
}

// w_a = U^dag h_a
template <typename T>
__device__ __forceinline__ void link_mul_dag(const Link<T>& u, const Half<T>& h, Half<T>& w) {
#pragma unroll
  for (int a = 0; a < 2; a++)
#pragma unroll
    for (int r = 0; r < 3; r++) {
      cpx<T> s = cmadd_conj(mk(T(0), T(0)), u.v[r], h.v[3 * a]);
      s = cmadd_conj(s, u.v[3 + r], h.v[3 * a + 1]);
      s = cmadd_conj(s, u.v[6 + r], h.v[3 * a + 2]);
      w.v[3 * a + r] = s;
    }
}

template <typename T> __device__ __forceinline__ T bc_phase(const Geom& g, int mu);
template <> __device__ __forceinline__ double bc_phase<double>(const Geom& g, int mu) { return g.bcd[mu]; }
template <> __device__ __forceinline__ float bc_phase<float>(const Geom& g, int mu) { return g.bcf[mu]; }

// FP32 a + c and a - c for a the low (H = 0) or high (H = 1) FP16 half of the
// word w (add / sub with an f16 and an f32 operand, sm_100 and later): the
// conversion of a is exact, so each equals the FP32 operation on the converted
// value, rounded once.
template <int H> __device__ __forceinline__ float add_h(unsigned int w, float c) {
  float d;
  if (H == 0) asm("{.reg .b16 l, u; mov.b32 {l, u}, %1; add.rn.f32.f16 %0, l, %2;}" : "=f"(d) : "r"(w), "f"(c));
  else asm("{.reg .b16 l, u; mov.b32 {l, u}, %1; add.rn.f32.f16 %0, u, %2;}" : "=f"(d) : "r"(w), "f"(c));
  return d;
}
template <int H> __device__ __forceinline__ float sub_h(unsigned int w, float c) {
  float d;
  if (H == 0) asm("{.reg .b16 l, u; mov.b32 {l, u}, %1; sub.rn.f32.f16 %0, l, %2;}" : "=f"(d) : "r"(w), "f"(c));
  else asm("{.reg .b16 l, u; mov.b32 {l, u}, %1; sub.rn.f32.f16 %0, u, %2;}" : "=f"(d) : "r"(w), "f"(c));
  return d;
}
// the real (H = 0) or imaginary (H = 1) part of the complex FP16 pair in w
template <int H> __device__ __forceinline__ float part_h(unsigned int w) {
  const __half2 v = *reinterpret_cast<const __half2*>(&w);
  return H == 0 ? __low2float(v) : __high2float(v);
}

// One projected complex component from FP16 data: a + C q with C = +1 (0),
// -1 (1), +i (2), -i (3); a and q are complex FP16 pairs (re low, im high).
template <int C>
__device__ __forceinline__ cpx<float> proj_h(unsigned int a, unsigned int q) {
  if (C == 0) return mk(add_h<0>(a, part_h<0>(q)), add_h<1>(a, part_h<1>(q)));
  if (C == 1) return mk(sub_h<0>(a, part_h<0>(q)), sub_h<1>(a, part_h<1>(q)));
  if (C == 2) return mk(sub_h<0>(a, part_h<1>(q)), add_h<1>(a, part_h<0>(q)));  // a + i q
  return mk(add_h<0>(a, part_h<1>(q)), sub_h<1>(a, part_h<0>(q)));               // a - i q
}

// FP16 storage: (1 + S gamma_mu) applied to the stored halves (each projected
// component one conversion and one mixed-precision add), the same values as
// converting all 24 components and projecting in FP32. w: the 12 complex FP16
// pairs, complex k = spin * 3 + colour in word k.
template <int MU, int S>
__device__ __forceinline__ void project_f16_words(const unsigned int (&w)[12], Half<float>& h) {
  // h0 = p0 + c0 p_k0, h1 = p1 + c1 p_k1 (the chiral-basis projection of project<MU, S>)
  constexpr int K0 = MU < 2 ? 3 : 2, K1 = MU < 2 ? 2 : 3;
  constexpr int C0 = MU == 0 ? (S > 0 ? 3 : 2) : MU == 1 ? (S > 0 ? 1 : 0) : MU == 2 ? (S > 0 ? 3 : 2) : (S > 0 ? 0 : 1);
  constexpr int C1 = MU == 0 ? (S > 0 ? 3 : 2) : MU == 1 ? (S > 0 ? 0 : 1) : MU == 2 ? (S > 0 ? 2 : 3) : (S > 0 ? 0 : 1);
#pragma unroll
  for (int c = 0; c < 3; c++) {
    h.v[c] = proj_h<C0>(w[c], w[3 * K0 + c]);
    h.v[3 + c] = proj_h<C1>(w[3 + c], w[3 * K1 + c]);
  }
}

// The FP16 neighbour at idx loaded and projected; returns its site norm.
template <int MU, int S>
__device__ __forceinline__ float load_project_f16(const void* in, int64_t stride, int64_t idx, Half<float>& h) {
  const uint4* b = reinterpret_cast<const uint4*>(in);
  const float nrm = SpinorIO<LQCD_F16>::norm_ptr(in, stride)[idx];
  unsigned int w[12];
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const uint4 v = b[c * stride + idx];
    w[4 * c] = v.x;
    w[4 * c + 1] = v.y;
    w[4 * c + 2] = v.z;
    w[4 * c + 3] = v.w;
  }
  project_f16_words<MU, S>(w, h);
  return nrm;
}

// Load the neighbour spinor and spin-project it with (1 + S gamma_mu). The
// linear factor the half spinor still needs -- the boundary phase of a
// wrapping hop and, for FP16 storage, the neighbour's site norm -- is returned
// instead of applied; accumulate_scaled folds it into its FMAs.
template <int P, int MU, int S>
__device__ __forceinline__ typename PrecTraits<P>::real load_project(const void* in, const Geom& g, int64_t idx,
                                                                     bool wrap, Half<typename PrecTraits<P>::real>& h) {
  using T = typename PrecTraits<P>::real;
  Spinor<T> s;
  T f;
  if constexpr (P == LQCD_F16) {
    f = load_project_f16<MU, S>(in, g.sstride, idx, h);
    return wrap ? bc_phase<T>(g, MU) * f : f;
  } else {
    SpinorIO<P>::load(in, g.sstride, idx, s);
    f = T(1);
  }
  project<MU, S>(s, h);
  return wrap ? bc_phase<T>(g, MU) * f : f;
}

template <typename T> __device__ __forceinline__ void conj_link(Link<T>& u) {
#pragma unroll
  for (int k = 0; k < 9; k++) u.v[k].i = -u.v[k].i;
}

// Both hops along mu. With GP (G-parity, n5 = 2 flavours i5 = f): a hop that
// wraps in a direction of g.gp reads the other flavour with sign +1 / -1
// (forward, f = 0 / 1) or -1 / +1 (backward) instead of the boundary phase,
// and the link is conjugated when its owner -- the site for the forward hop,
// the neighbour (flavour f') for the backward hop -- is flavour 1.
template <int MU, int P, int R, bool DAG, bool GP = false>
__device__ __forceinline__ void hop_dir(Spinor<typename PrecTraits<P>::real>& acc, const Geom& g,
                                        const void* gauge, const Coord& x, int64_t cb, int64_t i5,
                                        int parity, const void* in) {
  using T = typename PrecTraits<P>::real;
  constexpr int SF = DAG ? +1 : -1;  // forward hop carries (1 + SF gamma_mu)
  const int64_t n5 = g.n5;
  {
    bool wrap;
    const int64_t nb = neighbour_cb<MU>(g, x, +1, wrap);
    int64_t f_nb = i5;
    T sgn = T(1);
    if (GP && wrap && ((g.gp >> MU) & 1)) {
      f_nb = 1 - i5;
      sgn = i5 == 0 ? T(1) : T(-1);
      wrap = false;  // the twist replaces the boundary phase
    }
    Half<T> h;
    const T f = sgn * load_project<P, MU, SF>(in, g, nb * n5 + f_nb, wrap, h);
    Link<T> u;
    LinkIO<P, R>::load(gauge, g.gstride, parity * 4 + MU, cb, u);
    if (GP && i5 == 1) conj_link(u);
    Half<T> w;
    link_mul(u, h, w);
    accumulate_scaled<MU, SF>(acc, w, f);
  }
  {
    bool wrap;
    const int64_t nb = neighbour_cb<MU>(g, x, -1, wrap);
    int64_t f_nb = i5;
    T sgn = T(1);
    if (GP && wrap && ((g.gp >> MU) & 1)) {
      f_nb = 1 - i5;
      sgn = i5 == 0 ? T(-1) : T(1);
      wrap = false;
    }
    Half<T> h;
    const T f = sgn * load_project<P, MU, -SF>(in, g, nb * n5 + f_nb, wrap, h);
    Link<T> u;
    LinkIO<P, R>::load(gauge, g.gstride, (1 - parity) * 4 + MU, nb, u);
    if (GP && f_nb == 1) conj_link(u);
    Half<T> w;
    link_mul_dag(u, h, w);
    accumulate_scaled<MU, -SF>(acc, w, f);
  }
}

// out_chi(s) += coefficient * x_chi(s'), chirality + = spins 0,1 (k < 6), - = spins 2,3.
template <typename T>
__device__ __forceinline__ void add_chiral(Spinor<T>& out, const Spinor<T>& xs, T coef, bool plus) {
#pragma unroll
  for (int k = 0; k < 6; k++) {
    const int kk = plus ? k : 6 + k;
    out.v[kk] = out.v[kk] + coef * xs.v[kk];
  }
}

// Epilogue coefficients: PLAIN out = b H in; XPAY out = a x + b H in;
// M5 out = M5op(x) + b H in with M5op diagonal m5d and corner mf. (Loading the
// xpay operand before the hop, as the accumulator's start, made the bench step
// 1.8 % slower with FP16 storage: the operand is read at the end.)
template <typename T> struct EpiCoef {
  T a, b, m5d, mf;
};
template <typename T> __device__ __forceinline__ EpiCoef<T> epi_coef(const HopArgs& A) {
  return EpiCoef<T>{(T)A.a, (T)A.b, (T)A.m5d, (T)A.mf};
}
template <> __device__ __forceinline__ EpiCoef<float> epi_coef<float>(const HopArgs& A) {
  return EpiCoef<float>{A.af, A.bf, A.m5df, A.mff};
}
// The M5op^-1 scan's coefficients a, mf, 1 / (1 + mf a^L_s)
template <typename T> struct M5Coef {
  T a, mf, den_inv;
};
template <typename T> __device__ __forceinline__ M5Coef<T> m5_coef(const HopArgs& A) {
  return M5Coef<T>{(T)A.m5_a, (T)A.mf, (T)A.m5_den_inv};
}
template <> __device__ __forceinline__ M5Coef<float> m5_coef<float>(const HopArgs& A) {
  return M5Coef<float>{A.m5_af, A.mff, A.m5_den_invf};
}

// Both hops along mu with spin-paired packed arithmetic (hop_pair.cuh): the
// projection and the link as in hop_dir, the products and the accumulation on
// (spin 0, spin 1) pairs. FP32 / FP16 storage, no G-parity.
template <int MU, int P, int R, bool DAG>
__device__ __forceinline__ void hop_dir_sp(SPAcc& acc, const Geom& g, const void* gauge, const Coord& x, int64_t cb,
                                           int64_t i5, int parity, const void* in) {
  constexpr int SF = DAG ? +1 : -1;
  const int64_t n5 = g.n5;
#pragma unroll
  for (int dir = 0; dir < 2; dir++) {
    bool wrap;
    const int64_t nb = neighbour_cb<MU>(g, x, dir == 0 ? +1 : -1, wrap);
    Half<float> hh;
    const float f = dir == 0 ? load_project<P, MU, SF>(in, g, nb * n5 + i5, wrap, hh)
                             : load_project<P, MU, -SF>(in, g, nb * n5 + i5, wrap, hh);
    SPHalf h, w;
#pragma unroll
    for (int c = 0; c < 3; c++) {
      h.r[c] = make_float2(hh.v[c].r, hh.v[3 + c].r);
      h.i[c] = make_float2(hh.v[c].i, hh.v[3 + c].i);
    }
    Link<float> u;
    if (dir == 0) {
      LinkIO<P, R>::load(gauge, g.gstride, parity * 4 + MU, cb, u);
      link_mul_sp<false>(u, h, w);
      accumulate_sp<MU, SF>(acc, w, f);
    } else {
      LinkIO<P, R>::load(gauge, g.gstride, (1 - parity) * 4 + MU, nb, u);
      link_mul_sp<true>(u, h, w);
      accumulate_sp<MU, -SF>(acc, w, f);
    }
  }
}

}  // namespace lqcd

#include "hop_async.cuh"  // the staged hop uses the projections and products above
#include "hop_df.cuh"

namespace lqcd {

// H in at output site j (= cb * n5 + i5) of checkerboard `parity`. AS: neighbour
// data streamed through the shared-memory ring `ring` (hop_async.cuh).
template <int P, int R, bool DAG, bool GP = false, bool SP = false, bool AS = false, int BLOCK = 128>
__device__ __forceinline__ void hop_acc(const Geom& g, const void* gauge, const void* in, int parity, int64_t j,
                                        Spinor<typename PrecTraits<P>::real>& acc, unsigned char* ring = nullptr) {
  if constexpr (P == LQCD_F64_DF) {
    hop_acc_df<R, DAG, AS, BLOCK>(g, gauge, in, parity, j, acc, ring);
  } else if constexpr (AS) {
    hop_acc_async<P, R, DAG, SP, BLOCK>(g, gauge, in, parity, j, acc, ring);
  } else {
    const int64_t n5 = g.n5;
    int64_t cb, i5;
    if (n5 == 1) {
      cb = j;
      i5 = 0;
    } else {
      cb = fdiv((uint32_t)j, g.fn5);
      i5 = j - cb * n5;
    }
    const Coord x = cb_to_coord(g, cb, parity);
    if constexpr (SP) {
      static_assert(P == LQCD_F32 || P == LQCD_F16, "spin-paired hop: FP32 / FP16 storage");
      SPAcc a;
      sp_zero(a);
      hop_dir_sp<0, P, R, DAG>(a, g, gauge, x, cb, i5, parity, in);
      hop_dir_sp<1, P, R, DAG>(a, g, gauge, x, cb, i5, parity, in);
      hop_dir_sp<2, P, R, DAG>(a, g, gauge, x, cb, i5, parity, in);
      hop_dir_sp<3, P, R, DAG>(a, g, gauge, x, cb, i5, parity, in);
      sp_unpack(a, acc);
    } else {
      zero(acc);
      hop_dir<0, P, R, DAG, GP>(acc, g, gauge, x, cb, i5, parity, in);
      hop_dir<1, P, R, DAG, GP>(acc, g, gauge, x, cb, i5, parity, in);
      hop_dir<2, P, R, DAG, GP>(acc, g, gauge, x, cb, i5, parity, in);
      hop_dir<3, P, R, DAG, GP>(acc, g, gauge, x, cb, i5, parity, in);
    }
  }
}

// The epilogue at output site j of the hop result acc = H in (see EpiCoef).
template <int P, bool DAG, int EPI>
__device__ __forceinline__ void hop_epilogue(const Geom& g, const void* xb, int64_t j,
                                             const EpiCoef<typename PrecTraits<P>::real>& c,
                                             const Spinor<typename PrecTraits<P>::real>& acc,
                                             Spinor<typename PrecTraits<P>::real>& res) {
  using T = typename PrecTraits<P>::real;
  using IO = SpinorIO<P>;
  const int64_t n5 = g.n5;
  const T b = c.b;
  if (EPI == EPI_PLAIN || EPI == EPI_M5INV) {
#pragma unroll
    for (int k = 0; k < 12; k++) res.v[k] = b * acc.v[k];
  } else if (EPI == EPI_XPAY) {
    Spinor<T> xv;
    IO::load(xb, g.sstride, j, xv);
    const T a = c.a;
#pragma unroll
    for (int k = 0; k < 12; k++) res.v[k] = mk(fma(a, xv.v[k].r, b * acc.v[k].r), fma(a, xv.v[k].i, b * acc.v[k].i));
  } else {
    // M5op(x)(s) = d x(s) - P_- x(s+1) - P_+ x(s-1), mf corners (dagger swaps directions)
    const int64_t i5 = n5 == 1 ? 0 : j - (int64_t)fdiv((uint32_t)j, g.fn5) * n5;
    Spinor<T> xv;
    IO::load(xb, g.sstride, j, xv);
    const T d = c.m5d;
#pragma unroll
    for (int k = 0; k < 12; k++) res.v[k] = mk(fma(d, xv.v[k].r, b * acc.v[k].r), fma(d, xv.v[k].i, b * acc.v[k].i));
    const bool top = i5 + 1 == n5, bottom = i5 == 0;
    const int64_t jp = top ? j - (n5 - 1) : j + 1;
    const int64_t jm = bottom ? j + (n5 - 1) : j - 1;
    const T cp = top ? c.mf : T(-1);
    const T cm = bottom ? c.mf : T(-1);
    Spinor<T> xp, xm;
    IO::load(xb, g.sstride, jp, xp);
    IO::load(xb, g.sstride, jm, xm);
    if (!DAG) {
      add_chiral(res, xp, cp, false);
      add_chiral(res, xm, cm, true);
    } else {
      add_chiral(res, xm, cm, false);
      add_chiral(res, xp, cp, true);
    }
  }
}

// The result at output site j (= cb * n5 + i5) of checkerboard `parity`.
template <int P, int R, bool DAG, int EPI, bool GP = false, bool SP = false, bool AS = false, int BLOCK = 128>
__device__ __forceinline__ void hop_site(const Geom& g, const void* gauge, const void* in, const void* xb,
                                         int parity, int64_t j, const EpiCoef<typename PrecTraits<P>::real>& c,
                                         Spinor<typename PrecTraits<P>::real>& res, unsigned char* ring = nullptr) {
  Spinor<typename PrecTraits<P>::real> acc;
  hop_acc<P, R, DAG, GP, SP, AS, BLOCK>(g, gauge, in, parity, j, acc, ring);
  hop_epilogue<P, DAG, EPI>(g, xb, j, c, acc, res);
}

template <typename T> __device__ __forceinline__ T norm2_site(const Spinor<T>& res) {
  T s = T(0);
#pragma unroll
  for (int k = 0; k < 12; k++) s = fma(res.v[k].r, res.v[k].r, fma(res.v[k].i, res.v[k].i, s));
  return s;
}

// ---- site staging for the L_s-replicated / multi-RHS hop (n5 >= STAGE_MIN_N5): the n5
// threads of a 4D site share its eight links and neighbours (the paper's gauge
// field reused L_s times, Sec. 3), so a block loads (and for 12-real links
// rebuilds and, for FP16, converts) each link of its 4D sites once into shared
// memory, together with the neighbour's index and the boundary phase, and every
// thread reads them from there: five 16-byte broadcasts per direction instead of
// three to nine loads, 36 conversion and rebuild operations and the index
// arithmetic.
constexpr int STAGE_MIN_N5 = 4;
// One direction: 18 link reals (row-major), the neighbour's checkerboard index, the phase
struct StagedDir {
  float4 q[5];
};
constexpr int STAGE_SITE_F4 = 8 * 5 + 1;  // float4 per site: an odd number, so that sites spread over the banks
__host__ __device__ constexpr int stage_sites(int block, int n5) { return block / n5 + 2; }

// Stages the block's 4D sites cb0 .. cb0 + nls - 1 (checkerboard `parity`); every
// thread of the block must call it.
template <int P, int R, int BLOCK>
__device__ __forceinline__ void stage_block(const Geom& g, const void* gauge, int parity, uint32_t cb0, int nls,
                                            float4* sm) {
  for (int t = threadIdx.x; t < nls * 8; t += BLOCK) {
    const int ls = t >> 3, d = t & 7, mu = d >> 1;
    const uint32_t cb = cb0 + ls;
    if (cb >= (uint32_t)g.Vh) continue;
    const bool fwd = (d & 1) == 0;
    const Coord x = cb_to_coord(g, cb, parity);
    const int L = mu == 0 ? g.X : mu == 1 ? g.Y : mu == 2 ? g.Z : g.T;
    const int xm = mu == 0 ? x.c[0] : mu == 1 ? x.c[1] : mu == 2 ? x.c[2] : x.c[3];
    const uint32_t st = mu == 0 ? 1u : mu == 1 ? (uint32_t)g.st[1] : mu == 2 ? (uint32_t)g.st[2] : (uint32_t)g.st[3];
    const float bc = mu == 0 ? g.bcf[0] : mu == 1 ? g.bcf[1] : mu == 2 ? g.bcf[2] : g.bcf[3];
    const bool wrap = fwd ? xm == L - 1 : xm == 0;
    const uint32_t lex = fwd ? (wrap ? x.lex - (uint32_t)(L - 1) * st : x.lex + st)
                             : (wrap ? x.lex + (uint32_t)(L - 1) * st : x.lex - st);
    const uint32_t nb = lex >> 1;
    Link<float> u;
    LinkIO<P, R>::load(gauge, g.gstride, (fwd ? parity : 1 - parity) * 4 + mu, fwd ? cb : nb, u);
    float4* q = sm + ls * STAGE_SITE_F4 + d * 5;
#pragma unroll
    for (int k = 0; k < 4; k++) q[k] = make_float4(u.v[2 * k].r, u.v[2 * k].i, u.v[2 * k + 1].r, u.v[2 * k + 1].i);
    q[4] = make_float4(u.v[8].r, u.v[8].i, __uint_as_float(nb), wrap ? bc : 1.f);
  }
  __syncthreads();
}

// The two hops along MU from the staged site sm, scalar or (SP) spin-paired.
template <int MU, int P, bool DAG, bool SP, typename Acc>
__device__ __forceinline__ void hop_dir_staged(Acc& acc, const Geom& g, const float4* sm, uint32_t i5, const void* in) {
  constexpr int SF = DAG ? +1 : -1;  // forward hop carries (1 + SF gamma_mu)
#pragma unroll
  for (int dir = 0; dir < 2; dir++) {
    const float4* q = sm + (2 * MU + dir) * 5;
    const float4 last = q[4];
    const int64_t idx = (int64_t)__float_as_uint(last.z) * g.n5 + i5;
    Half<float> h;
    float f = dir == 0 ? load_project<P, MU, SF>(in, g, idx, false, h) : load_project<P, MU, -SF>(in, g, idx, false, h);
    f *= last.w;
    Link<float> u;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      const float4 w = q[k];
      u.v[2 * k] = mk(w.x, w.y);
      u.v[2 * k + 1] = mk(w.z, w.w);
    }
    u.v[8] = mk(last.x, last.y);
    if constexpr (SP) {
      SPHalf hp, w;
#pragma unroll
      for (int c = 0; c < 3; c++) {
        hp.r[c] = make_float2(h.v[c].r, h.v[3 + c].r);
        hp.i[c] = make_float2(h.v[c].i, h.v[3 + c].i);
      }
      if (dir == 0) {
        link_mul_sp<false>(u, hp, w);
        accumulate_sp<MU, SF>(acc, w, f);
      } else {
        link_mul_sp<true>(u, hp, w);
        accumulate_sp<MU, -SF>(acc, w, f);
      }
    } else {
      Half<float> w;
      if (dir == 0) {
        link_mul(u, h, w);
        accumulate_scaled<MU, SF>(acc, w, f);
      } else {
        link_mul_dag(u, h, w);
        accumulate_scaled<MU, -SF>(acc, w, f);
      }
    }
  }
}

// H in at slice i5 of the staged site sm.
template <int P, bool DAG, bool SP>
__device__ __forceinline__ void hop_acc_staged(const Geom& g, const float4* sm, uint32_t i5, const void* in,
                                               Spinor<float>& out) {
  if constexpr (SP) {
    SPAcc a;
    sp_zero(a);
    hop_dir_staged<0, P, DAG, true>(a, g, sm, i5, in);
    hop_dir_staged<1, P, DAG, true>(a, g, sm, i5, in);
    hop_dir_staged<2, P, DAG, true>(a, g, sm, i5, in);
    hop_dir_staged<3, P, DAG, true>(a, g, sm, i5, in);
    sp_unpack(a, out);
  } else {
    zero(out);
    hop_dir_staged<0, P, DAG, false>(out, g, sm, i5, in);
    hop_dir_staged<1, P, DAG, false>(out, g, sm, i5, in);
    hop_dir_staged<2, P, DAG, false>(out, g, sm, i5, in);
    hop_dir_staged<3, P, DAG, false>(out, g, sm, i5, in);
  }
}

// Shared memory of a hop whose neighbour data are copied asynchronously (AS)
template <int P, int R> constexpr int ring_bytes(int block) {
  if constexpr (P == LQCD_F64_DF) return df_ring_bytes<R>(block);
  else return stage_nslot<P>() * stage_slot_bytes<P, R>() * block;
}

// One thread per output site. LS: links and neighbours staged per 4D site; SP:
// spin-paired packed arithmetic; AS: neighbour data copied asynchronously.
template <int P, int R, bool DAG, int EPI, int RED, int BLOCK, bool GP, bool LS = false, bool SP = false,
          bool AS = false>
__device__ __forceinline__ void hop_body(const HopArgs& A) {
  using T = typename PrecTraits<P>::real;
  overlap_wait();
  if (gate_closed(A.gate)) return;
  int parity = A.out_parity;
  int blk = blockIdx.x;
  if (A.full) {
    parity = blk >= A.blocks_per_parity ? 1 : 0;
    blk -= parity * A.blocks_per_parity;
  }
  const char* in = static_cast<const char*>(A.in) + (A.full ? (1 - parity) * A.half_bytes : 0);
  char* out = static_cast<char*>(A.out) + (A.full ? parity * A.half_bytes : 0);
  const char* xb = A.x ? static_cast<const char*>(A.x) + (A.full ? parity * A.half_bytes : 0) : nullptr;
  const EpiCoef<T> c = epi_coef<T>(A);
  const int64_t first = (int64_t)blk * BLOCK;
  const int64_t j = first + threadIdx.x;
  // LS: links and neighbours staged in shared memory once per 4D site
  const float4* site = nullptr;
  uint32_t i5 = 0;
  if constexpr (LS) {
    extern __shared__ float4 staged[];
    const uint32_t n5 = A.g.n5, cb0 = fdiv((uint32_t)first, A.g.fn5);
    const int64_t end = first + BLOCK < A.g.nsites ? first + BLOCK : A.g.nsites;
    stage_block<P, R, BLOCK>(A.g, A.gauge, parity, cb0, (int)(fdiv((uint32_t)end - 1, A.g.fn5) - cb0 + 1), staged);
    const uint32_t cb = fdiv((uint32_t)j, A.g.fn5);
    i5 = (uint32_t)j - cb * n5;
    site = staged + (cb - cb0) * STAGE_SITE_F4;
  }
  // AS: the ring of asynchronously copied neighbour data
  unsigned char* ring = nullptr;
  if constexpr (AS) {
    __shared__ __align__(16) unsigned char stage_ring[ring_bytes<P, R>(BLOCK)];
    ring = stage_ring;
  }
  auto hop = [&](Spinor<T>& res) {
    if constexpr (LS) {
      Spinor<T> acc;
      hop_acc_staged<P, DAG, SP>(A.g, site, i5, in, acc);
      hop_epilogue<P, DAG, EPI>(A.g, xb, j, c, acc, res);
    } else {
      hop_site<P, R, DAG, EPI, GP, SP, AS, BLOCK>(A.g, A.gauge, in, xb, parity, j, c, res, ring);
    }
  };
  if constexpr (EPI == EPI_M5INV) {
    // every lane takes part in the fifth-dimension scan; lanes past the end
    // (whole 4D sites, since L_s divides the block) carry zeros and store nothing
    static_assert(RED == RED_NONE, "M5op^-1 epilogue without reduction");
    const bool live = j < A.g.nsites;
    Spinor<T> res;
    if (live) hop(res);
    else zero(res);
    const int Ls = A.g.n5;
    const M5Coef<T> mc = m5_coef<T>(A);
    m5inv_lanes(res, (int)(threadIdx.x & (unsigned)(Ls - 1)), Ls, A.m5_dagger != 0, mc.a, mc.mf, mc.den_inv);
    if (live) SpinorIO<P>::store(out, A.g.sstride, j, res);
    return;
  }
  const bool live = j < A.g.nsites;
  Spinor<T> res;
  if constexpr (RED == RED_CG_UPDATE) {
    const int64_t ps = A.full ? parity * A.half_bytes : 0, vs = A.full ? parity * A.upd_half_bytes : 0;
    const int64_t rs = A.full ? parity * A.upd_rs_half_bytes : 0;
    char* xs_p = static_cast<char*>(A.upd_xs) + vs;
    char* rs_p = static_cast<char*>(A.upd_rs) + rs;
    Spinor<typename PrecTraits<vec_prec(P)>::real> x, r;
    T red = T(0);
    if (live) {
      hop(res);
      red = updated_site<vec_prec(P), P, rs_prec(P)>(A.g, j, A.red.sys[sys_of(j, A.red.nsys)].alpha,
                                                     static_cast<const char*>(A.upd_p) + ps, res, xs_p, rs_p, x, r);
    }
    block_reduce_finalize<BLOCK>(red, first, A.red, [&]() {
      if (!live) return;
      SpinorIO<vec_prec(P)>::store(xs_p, A.g.sstride, j, x);
      SpinorIO<rs_prec(P)>::store(rs_p, A.g.sstride, j, r);
    });
  } else if constexpr (RED == RED_NORM) {
    T red = T(0);
    if (live) {
      hop(res);
      red = norm2_site(res);
    }
    block_reduce_finalize<BLOCK>(red, first, A.red, [&]() {
      if (live) SpinorIO<P>::store(out, A.g.sstride, j, res);
    });
  } else {
    if (!live) return;
    hop(res);
    SpinorIO<P>::store(out, A.g.sstride, j, res);
  }
}

// MINB: minimum resident blocks per SM the register allocation must allow
// (__launch_bounds__; 0 leaves the choice to the compiler), one of the knobs
// of the launch shapes the tuner times.
//
// KIND 1: the plain hop; -1 / -5: one site per thread with the links and neighbours of each 4D site
// staged in shared memory (LS), in scalar / spin-paired arithmetic;
// -2: one site per thread in spin-paired packed arithmetic (SP);
// -3 / -4: as 1 / -2 with the neighbour data copied asynchronously
// through a shared-memory ring (AS, hop_async.cuh).
template <int P, int R, bool DAG, int EPI, int RED, int BLOCK, bool GP = false, int KIND = 1, int MINB = 0>
__global__ void __launch_bounds__(BLOCK, MINB) hop_kernel(const HopArgs A) {
  if constexpr (KIND == -1) hop_body<P, R, DAG, EPI, RED, BLOCK, GP, true>(A);
  else if constexpr (KIND == -2) hop_body<P, R, DAG, EPI, RED, BLOCK, GP, false, true>(A);
  else if constexpr (KIND == -3) hop_body<P, R, DAG, EPI, RED, BLOCK, GP, false, false, true>(A);
  else if constexpr (KIND == -4) hop_body<P, R, DAG, EPI, RED, BLOCK, GP, false, true, true>(A);
  else if constexpr (KIND == -5) hop_body<P, R, DAG, EPI, RED, BLOCK, GP, true, true>(A);
  else hop_body<P, R, DAG, EPI, RED, BLOCK, GP>(A);
}

}  // namespace lqcd
