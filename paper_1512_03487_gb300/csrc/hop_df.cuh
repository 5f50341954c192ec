// The hop in double-float arithmetic on FP64 fields (LQCD_F64_DF), with the two
// spin components of each half spinor in packed FP32x2 instructions.
//
// Every operation is the scalar double-float operation of df.cuh, two at a time, with the
// same roundings; the kernel is bound by instructions (about
// 1,800 FP32 operations and 250 integer ones of the splits per direction and thread).
// Three things keep it fast. (1) A pair (spin 0, spin 1) shares every packed
// instruction (add / mul / fma.rn.f32x2; negated and broadcast operands cost
// nothing), which halves the issue slots of the arithmetic. (2) The directions are a
// rolled loop, one copy of the per-direction code that stays in the instruction
// cache, with the projector's signs as factors of the fused multiply-adds. (3) The
// neighbour data are copied into shared memory a phase ahead (cp.async, no register
// holds them), which hides the loads at 16 warps per SM. M_hat (two hops) at 24^3 x
// 48 with 18-real links on GB300: 593 -> 352 us against scalar instructions with the
// loads where they are used; 222 -> 129 million warp instructions a hop, 64 % of
// the issue slots busy.
#pragma once

#include "lqcd_common.cuh"

namespace lqcd {

// Double-float numbers at two spins (.x and .y): value h + l.
struct DF2 {
  float2 h, l;
};
struct DF2c {
  DF2 r, i;
};

__device__ __forceinline__ float2 two(float a) { return make_float2(a, a); }
__device__ __forceinline__ DF2 df2_pair(dfl a, dfl b) {
  DF2 p;
  p.h = make_float2(a.hi, b.hi);
  p.l = make_float2(a.lo, b.lo);
  return p;
}

// a + sg b = s + e exactly, sg = +-1 per spin
__device__ __forceinline__ void two_sum2(float2 a, float2 sg, float2 b, float2& s, float2& e) {
  s = fma2(sg, b, a);
  const float2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), fma2(sg, b, neg2(bb)));
}
__device__ __forceinline__ DF2 fast_two_sum2(float2 a, float2 b) {
  DF2 r;
  r.h = add2(a, b);
  r.l = sub2(b, sub2(r.h, a));
  return r;
}

// a + sg b (df_add)
__device__ __forceinline__ DF2 df2_add(DF2 a, float2 sg, DF2 b) {
  float2 s, e;
  two_sum2(a.h, sg, b.h, s, e);
  return fast_two_sum2(s, add2(e, fma2(sg, b.l, a.l)));
}

// u h and u h + w for a link's real u, the same for both spins (df_mul, df_fma)
__device__ __forceinline__ DF2 df2_mul(dfl u, DF2 h) {
  const float2 uh = two(u.hi), ul = two(u.lo);
  const float2 p = mul2(uh, h.h);
  return fast_two_sum2(p, fma2(ul, h.h, fma2(uh, h.l, fma2(uh, h.h, neg2(p)))));
}
__device__ __forceinline__ DF2 df2_fma(dfl u, DF2 h, DF2 w) {
  const float2 uh = two(u.hi), ul = two(u.lo);
  const float2 p = mul2(uh, h.h);
  const float2 e = fma2(ul, h.h, fma2(uh, h.l, fma2(uh, h.h, neg2(p))));
  const float2 s = add2(p, w.h);
  const float2 bb = sub2(s, p);
  const float2 t = add2(sub2(p, sub2(s, bb)), sub2(w.h, bb));
  return fast_two_sum2(s, add2(t, add2(e, w.l)));
}

__device__ __forceinline__ cpx<dfl> df_read(const double2* p) {
  const double2 w = *p;
  return mk(df_split(w.x), df_split(w.y));
}

// Shared memory of a block: one direction's neighbour spinors [12][BLOCK] and links
// [R / 2][BLOCK], raw, each thread's own column.
template <int R> constexpr int df_ring_bytes(int block) { return (12 + R / 2) * 16 * block; }

// Direction dir of site x: its neighbour's checkerboard index and whether the hop wraps.
__device__ __forceinline__ int64_t df_neighbour(const Geom& g, const Coord& x, int dir, bool& wrap) {
  const int mu = dir >> 1;
  const bool fwd = (dir & 1) == 0;
  const int L = mu == 0 ? g.X : mu == 1 ? g.Y : mu == 2 ? g.Z : g.T;
  const int xm = mu == 0 ? x.c[0] : mu == 1 ? x.c[1] : mu == 2 ? x.c[2] : x.c[3];
  const uint32_t st = mu == 0 ? 1u : mu == 1 ? (uint32_t)g.st[1] : mu == 2 ? (uint32_t)g.st[2] : (uint32_t)g.st[3];
  wrap = fwd ? xm == L - 1 : xm == 0;
  const uint32_t lex = fwd ? (wrap ? x.lex - (uint32_t)(L - 1) * st : x.lex + st)
                           : (wrap ? x.lex + (uint32_t)(L - 1) * st : x.lex - st);
  return (int64_t)(lex >> 1);
}

// H in at output site j of checkerboard `parity`. RING: the neighbour data are copied
// through `ring`, df_ring_bytes of shared memory; else they are loaded where they are used.
template <int R, bool DAG, bool RING, int BLOCK>
__device__ __forceinline__ void hop_acc_df(const Geom& g, const void* gauge, const void* in, int parity, int64_t j,
                                           Spinor<dfl>& out, unsigned char* ring) {
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
  constexpr int SF = DAG ? +1 : -1;  // forward hop carries (1 + SF gamma_mu)
  DF2c up[3], lo[3];                 // spins 0, 1 and spins 2, 3 per colour
#pragma unroll
  for (int c = 0; c < 3; c++) {
    up[c].r.h = up[c].r.l = up[c].i.h = up[c].i.l = make_float2(0.f, 0.f);
    lo[c] = up[c];
  }
  // Asynchronous copies into this thread's columns: the next direction's spinor while
  // the link is multiplied, its link while the next spinor is projected. A thread
  // reads only what it copied, so no barrier is needed.
  double2* sp = reinterpret_cast<double2*>(ring) + threadIdx.x;
  double2* lk = sp + 12 * BLOCK;
  const auto fetch_spinor = [&](int dir) {
    bool wrap;
    const int64_t idx = df_neighbour(g, x, dir, wrap) * n5 + i5;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(sp);
    const double2* src = reinterpret_cast<const double2*>(in) + idx;
#pragma unroll
    for (int k = 0; k < 12; k++) cp_async<16>(dst + k * BLOCK * 16, src + k * g.sstride);
    cp_async_commit();
  };
  const auto fetch_link = [&](int dir) {
    bool wrap;
    const int64_t nb = df_neighbour(g, x, dir, wrap);
    const bool fwd = (dir & 1) == 0;
    const int blk = (fwd ? parity : 1 - parity) * 4 + (dir >> 1);
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(lk);
    const double2* src = reinterpret_cast<const double2*>(gauge) + (int64_t)blk * (R / 2) * g.gstride + (fwd ? cb : nb);
#pragma unroll
    for (int k = 0; k < R / 2; k++) cp_async<16>(dst + k * BLOCK * 16, src + k * g.gstride);
    cp_async_commit();
  };
  if (RING) {
    fetch_spinor(0);
    fetch_link(0);
  }
#pragma unroll 1
  for (int dir = 0; dir < 8; dir++) {
    const int mu = dir >> 1;
    const bool fwd = (dir & 1) == 0;
    bool wrap;
    const int64_t nb = df_neighbour(g, x, dir, wrap);
    const double2* ps = RING ? sp : reinterpret_cast<const double2*>(in) + nb * n5 + i5;
    const double2* pl = RING ? lk : reinterpret_cast<const double2*>(gauge) +
                                        (int64_t)((fwd ? parity : 1 - parity) * 4 + mu) * (R / 2) * g.gstride + (fwd ? cb : nb);
    const int64_t ds = RING ? BLOCK : g.sstride, dl = RING ? BLOCK : g.gstride;
    // (1 + S gamma_mu) in the chiral basis: h0 = p0 + c0 p_k0, h1 = p1 + c1 p_k1 with (k0, k1) = (3, 2) for
    // mu < 2, else (2, 3), and c = sc (i if mu is even); the lower spins S B^dag w: spin 2 += d2 w_m2, spin 3 +=
    // d3 w_m3 with (m2, m3) = (1, 0) for mu < 2, else (0, 1), and d = sd (i if mu is even)
    const bool imag = (mu & 1) == 0, cross = mu < 2;
    const float S = (fwd ? SF : -SF) > 0 ? 1.f : -1.f;
    const float2 sc = make_float2(mu == 3 ? S : -S, mu == 0 ? -S : S);
    const float2 sd = make_float2(S, mu == 1 || mu == 2 ? -S : S);
    const float2 sc_r = imag ? neg2(sc) : sc;
    // a wrapping hop's boundary phase (+-1) flips the signs of its whole contribution
    const float bcm = mu == 0 ? g.bcf[0] : mu == 1 ? g.bcf[1] : mu == 2 ? g.bcf[2] : g.bcf[3];
    const float ph = wrap && bcm < 0.f ? -1.f : 1.f;
    const float2 su = two(ph), sl_i = mul2(su, sd), sl_r = imag ? neg2(sl_i) : sl_i;

    DF2c h[3];
    if (RING) cp_async_wait<1>();  // this direction's spinor; its link may still be under way
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const cpx<dfl> p0 = df_read(ps + c * ds), p1 = df_read(ps + (3 + c) * ds);
      double2 q0 = ps[((cross ? 9 : 6) + c) * ds], q1 = ps[((cross ? 6 : 9) + c) * ds];
      if (imag) {  // times i: real and imaginary parts change places (the sign is in sc_r)
        q0 = make_double2(q0.y, q0.x);
        q1 = make_double2(q1.y, q1.x);
      }
      h[c].r = df2_add(df2_pair(p0.r, p1.r), sc_r, df2_pair(df_split(q0.x), df_split(q1.x)));
      h[c].i = df2_add(df2_pair(p0.i, p1.i), sc, df2_pair(df_split(q0.y), df_split(q1.y)));
    }
    if (RING) {
      if (dir < 7) fetch_spinor(dir + 1);
      else cp_async_commit();  // an empty group keeps the count uniform
      cp_async_wait<1>();      // this direction's link
    }
    // U (forward) or U^dag (backward), row by row: w = sum_c u_rc h_c
    Link<dfl> v;
    if constexpr (R == 12) {
#pragma unroll
      for (int k = 0; k < 6; k++) v.v[k] = df_read(pl + k * dl);
      rebuild_row2(v);
    }
#pragma unroll
    for (int r = 0; r < 3; r++) {
      DF2c w;
#pragma unroll
      for (int c = 0; c < 3; c++) {
        cpx<dfl> u;
        if constexpr (R == 12) u = fwd ? v.v[3 * r + c] : v.v[3 * c + r];
        else u = df_read(pl + (fwd ? 3 * r + c : 3 * c + r) * dl);
        if (!fwd) u.i = -u.i;
        w.r = c == 0 ? df2_mul(u.r, h[c].r) : df2_fma(u.r, h[c].r, w.r);
        w.r = df2_fma(-u.i, h[c].i, w.r);
        w.i = c == 0 ? df2_mul(u.r, h[c].i) : df2_fma(u.r, h[c].i, w.i);
        w.i = df2_fma(u.i, h[c].r, w.i);
      }
      up[r].r = df2_add(up[r].r, su, w.r);
      up[r].i = df2_add(up[r].i, su, w.i);
      auto exchange = [](float2& a) { a = make_float2(a.y, a.x); };
      if (cross) {
        exchange(w.r.h);
        exchange(w.r.l);
        exchange(w.i.h);
        exchange(w.i.l);
      }
      if (imag) {
        const DF2 t = w.r;
        w.r = w.i;
        w.i = t;
      }
      lo[r].r = df2_add(lo[r].r, sl_r, w.r);
      lo[r].i = df2_add(lo[r].i, sl_i, w.i);
    }
    if (RING && dir < 7) fetch_link(dir + 1);
  }
#pragma unroll
  for (int c = 0; c < 3; c++) {
    out.v[c] = mk(dfl(up[c].r.h.x, up[c].r.l.x), dfl(up[c].i.h.x, up[c].i.l.x));
    out.v[3 + c] = mk(dfl(up[c].r.h.y, up[c].r.l.y), dfl(up[c].i.h.y, up[c].i.l.y));
    out.v[6 + c] = mk(dfl(lo[c].r.h.x, lo[c].r.l.x), dfl(lo[c].i.h.x, lo[c].i.l.x));
    out.v[9 + c] = mk(dfl(lo[c].r.h.y, lo[c].r.l.y), dfl(lo[c].i.h.y, lo[c].i.l.y));
  }
}

}  // namespace lqcd
