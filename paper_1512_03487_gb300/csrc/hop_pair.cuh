// The hop's arithmetic in packed FP32x2 instructions (add / mul / fma.rn.f32x2,
// sm_100 and later) for FP32 and FP16 storage: a pair is one real number at two
// spins, so a link element is broadcast to both halves. Negating and broadcasting
// an operand cost nothing on GB300; exchanging its halves costs two moves, which is
// why complex numbers held as (re, im) pairs were slower (ALU pipe 21 -> 47 % busy),
// and the FMA pipe does two scalar operations per packed one, so that packing saves
// issue slots, not FMA throughput. Every packed operation is the one-site hop's
// scalar operation in the same order, so both give bit-identical results.
#pragma once

#include "lqcd_common.cuh"

namespace lqcd {

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// One site per thread with the two spin components of each half spinor paired:
// H[c] = (h_0c, h_1c) as float2 of real parts and of imaginary parts, so
// w_a = U h_a for a = 0, 1 is one packed product per term (the link element
// broadcast to both lanes), and the accumulator holds spins (0, 1) and (2, 3)
// as pairs. Same operations in the same order per lane as the one-site hop.
struct SPHalf { float2 r[3], i[3]; };   // (h_0c, h_1c), c = 0..2
struct SPAcc { float2 ur[3], ui[3], lr[3], li[3]; };  // spins (0,1) and (2,3), colour c

__device__ __forceinline__ void sp_zero(SPAcc& a) {
#pragma unroll
  for (int c = 0; c < 3; c++) a.ur[c] = a.ui[c] = a.lr[c] = a.li[c] = make_float2(0.f, 0.f);
}
__device__ __forceinline__ void sp_unpack(const SPAcc& a, Spinor<float>& s) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    s.v[c] = mk(a.ur[c].x, a.ui[c].x);
    s.v[3 + c] = mk(a.ur[c].y, a.ui[c].y);
    s.v[6 + c] = mk(a.lr[c].x, a.li[c].x);
    s.v[9 + c] = mk(a.lr[c].y, a.li[c].y);
  }
}

__device__ __forceinline__ float2 bc2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 swp(float2 a) { return make_float2(a.y, a.x); }

// w = U h (DAG: U^dag h) on spin pairs
template <bool DAG>
__device__ __forceinline__ void link_mul_sp(const Link<float>& u, const SPHalf& h, SPHalf& w) {
#pragma unroll
  for (int r = 0; r < 3; r++) {
    float2 re, im;
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const cpx<float> m = DAG ? u.v[3 * c + r] : u.v[3 * r + c];
      const float2 mr = bc2(m.r), mi = bc2(m.i);
      if (c == 0) {
        re = mul2(mr, h.r[c]);
        im = mul2(mr, h.i[c]);
      } else {
        re = fma2(mr, h.r[c], re);
        im = fma2(mr, h.i[c], im);
      }
      if (DAG) {
        re = fma2(mi, h.i[c], re);
        im = fma2(neg2(mi), h.r[c], im);
      } else {
        re = fma2(neg2(mi), h.i[c], re);
        im = fma2(mi, h.r[c], im);
      }
    }
    w.r[r] = re;
    w.i[r] = im;
  }
}

// acc += f (upper = w, lower = S B_mu^dag w) on spin pairs (see accumulate_scaled)
template <int MU, int S>
__device__ __forceinline__ void accumulate_sp(SPAcc& acc, const SPHalf& w, float f) {
  const float fs = S > 0 ? f : -f;
  const float2 F = bc2(f);
#pragma unroll
  for (int c = 0; c < 3; c++) {
    acc.ur[c] = fma2(F, w.r[c], acc.ur[c]);
    acc.ui[c] = fma2(F, w.i[c], acc.ui[c]);
    if (MU == 0) {         // spin 2 += fs i w1, spin 3 += fs i w0
      acc.lr[c] = fma2(bc2(-fs), swp(w.i[c]), acc.lr[c]);
      acc.li[c] = fma2(bc2(fs), swp(w.r[c]), acc.li[c]);
    } else if (MU == 1) {  // spin 2 += fs w1, spin 3 += -fs w0
      acc.lr[c] = fma2(make_float2(fs, -fs), swp(w.r[c]), acc.lr[c]);
      acc.li[c] = fma2(make_float2(fs, -fs), swp(w.i[c]), acc.li[c]);
    } else if (MU == 2) {  // spin 2 += fs i w0, spin 3 += -fs i w1
      acc.lr[c] = fma2(make_float2(-fs, fs), w.i[c], acc.lr[c]);
      acc.li[c] = fma2(make_float2(fs, -fs), w.r[c], acc.li[c]);
    } else {               // spin 2 += fs w0, spin 3 += fs w1
      acc.lr[c] = fma2(bc2(fs), w.r[c], acc.lr[c]);
      acc.li[c] = fma2(bc2(fs), w.i[c], acc.li[c]);
    }
  }
}

}  // namespace lqcd
