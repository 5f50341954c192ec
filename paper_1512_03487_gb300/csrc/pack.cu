// Layout transformation between the user's lexicographic AoS FP64 layout and
// the device SoA checkerboard layout (the Grid paper's central idea, Sec. 2.4:
// the layout is hidden behind the container and transformed to suit the
// hardware), with precision conversion and optional 12-real link compression
// (the paper's Compressor changes precision, Sec. 2.6).
#include <cstring>

#include "lqcd_internal.h"

namespace lqcd {

// Both directions are pure data movement between site-major rows (192-byte
// spinors, 144-byte links) and chunks with the site fastest. A thread that reads
// or writes its own row touches 32 rows per instruction and each sector several
// times, so a block moves its rows through shared memory: between there and the
// host layout consecutive threads take consecutive addresses, and on the chunked
// side each thread owns one site or link, coalesced across the warp. The pitch of
// the rows in shared memory is an odd number of 16-byte pieces, so that the threads'
// 16-byte accesses to their own rows spread over the banks.
// 20 x 14 x 18 x 36 on GB300, before and after: links to FP32 / 12 reals 48 -> 21 us,
// spinor to FP32 17 -> 12 us, FP64 spinor to the host layout 27 -> 13 us.

// Copies `rows` rows of LEN doubles between the host layout and shared memory: row
// q lies at mem + at(q) and in row slot(q) of sh. wide: mem + at(q) is 16-byte
// aligned (a host-layout buffer need only be 8-byte aligned). Inwards the 16- or 8-byte
// pieces are asynchronous copies: nothing waits in registers, so more blocks fit an
// SM; the caller waits with arrived(). FP64 spinor at 24^3 x 48, one parity: 19 us, from
// an 8-byte aligned buffer 21 (42 with ordinary loads).
template <bool IN, int BLOCK, int ROWS, int LEN, int PITCH, typename Slot, typename At>
__device__ __forceinline__ void copy_rows(double* sh, double* mem, int rows, bool wide, Slot slot, At at) {
  static_assert(PITCH % 2 == 0 && LEN % 2 == 0, "rows of whole 16-byte pieces");
  if (wide) {
    constexpr int Q = LEN / 2, N = (ROWS * Q + BLOCK - 1) / BLOCK;
#pragma unroll
    for (int i = 0; i < N; i++) {
      const int n = threadIdx.x + i * BLOCK, q = n / Q, k = 2 * (n - q * Q);
      if (q >= rows) break;
      double* s = sh + slot(q) * PITCH + k;
      if (IN) {
        cp_async<16>((uint32_t)__cvta_generic_to_shared(s), mem + at(q) + k);
      } else {
        __stcs(reinterpret_cast<double2*>(mem + at(q) + k), *reinterpret_cast<const double2*>(s));
      }
    }
  } else {
#pragma unroll 4
    for (int n = threadIdx.x; n < rows * LEN; n += BLOCK) {
      const int q = n / LEN, k = n - q * LEN;
      double* s = sh + slot(q) * PITCH + k;
      if (IN) cp_async<8>((uint32_t)__cvta_generic_to_shared(s), mem + at(q) + k);
      else mem[at(q) + k] = *s;
    }
  }
}
// The block's inward copies have landed.
__device__ __forceinline__ void arrived() {
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
}

// A double rounded to the nearest even float (its bits) with integer instructions,
// for zero and results in FP32's normal range; ok is cleared for the others (the
// caller converts those). The conversion instruction runs at the FP64 pipe's rate, a
// small fraction of the integer one, and kept that pipe 60-70 % busy while packing.
__device__ __forceinline__ unsigned int float_bits(double v, bool& ok) {
  const unsigned int hw = (unsigned int)__double2hiint(v), lw = (unsigned int)__double2loint(v);
  const bool zero = (hw << 1 | lw) == 0u;
  // exponent field 897 .. 1149: rounding up cannot leave the normal range
  ok = ok && (zero || (hw & 0x7fffffffu) - (897u << 20) < (253u << 20));
  unsigned int r = __funnelshift_l(lw, hw - (896u << 20), 3);  // the sign shifts out; 29 bits remain below
  if ((lw << 3 | (r & 1u)) > 0x80000000u) r++;
  return zero ? hw : (r & 0x7fffffffu) | (hw & 0x80000000u);
}
// the same for half (exponent field 1009 .. 1037)
__device__ __forceinline__ unsigned int half_bits(double v, bool& ok) {
  const unsigned int hw = (unsigned int)__double2hiint(v), lw = (unsigned int)__double2loint(v);
  const bool zero = (hw << 1 | lw) == 0u;
  ok = ok && (zero || (hw & 0x7fffffffu) - (1009u << 20) < (29u << 20));
  unsigned int r = ((hw & 0x7fffffffu) - (1008u << 20)) >> 10;  // 42 bits remain below
  if ((hw << 22 | (lw != 0u ? 1u : 0u) | (r & 1u)) > 0x80000000u) r++;
  return (zero ? 0u : r) | (hw >> 31 << 15);
}
// The other values, out of line so that the conversions run only for them (inlined,
// they are executed for every value and selected)
__device__ __noinline__ float2 convert_float2(double x, double y) { return make_float2((float)x, (float)y); }
__device__ __noinline__ unsigned int convert_half2(double x, double y) {
  const __half2 h = __halves2half2(__double2half(x), __double2half(y));
  return *reinterpret_cast<const unsigned int*>(&h);
}
// a pair of doubles as floats / halves, each as the conversion instruction rounds it
__device__ __forceinline__ float2 to_float2(double2 v) {
  bool ok = true;
  const float2 f = make_float2(__uint_as_float(float_bits(v.x, ok)), __uint_as_float(float_bits(v.y, ok)));
  if (!ok) return convert_float2(v.x, v.y);
  return f;
}
__device__ __forceinline__ unsigned int to_half2(double2 v) {
  bool ok = true;
  const unsigned int lo = half_bits(v.x, ok), w = lo | (half_bits(v.y, ok) << 16);
  if (!ok) return convert_half2(v.x, v.y);
  return w;
}

// Host-layout site index of device site j (cb * n5 + i5) of checkerboard `parity`.
__device__ __forceinline__ int64_t host_site(const Geom& g, int64_t j, int parity, bool full) {
  const int64_t n5 = g.n5;
  const int64_t cb = n5 == 1 ? j : (int64_t)fdiv((uint32_t)j, g.fn5), i5 = j - cb * n5;
  if (!full) return i5 * g.Vh + cb;
  const Coord x = cb_to_coord(g, cb, parity);
  return i5 * (2 * (int64_t)g.Vh) + x.lex;
}

constexpr int SPIN_ROWS = 64;   // sites per block, one per thread
constexpr int SPIN_PITCH = 26;  // doubles per row in shared memory

// A block of a full field takes SPIN_ROWS / 2 sites of each parity (their rows are
// neighbours in the host layout), a block of one checkerboard SPIN_ROWS sites.
template <int P, bool PACK>
__global__ void __launch_bounds__(SPIN_ROWS, 15) spinor_xfer_kernel(void* dev, double* host, Geom g, int parity, int full,
                                                                int wide, int64_t half_bytes) {
  using T = typename PrecTraits<P>::real;
  __shared__ __align__(16) double sh[SPIN_ROWS * SPIN_PITCH];
  __shared__ int64_t at[SPIN_ROWS];
  const int per = full ? SPIN_ROWS / 2 : SPIN_ROWS;
  const int64_t first = (int64_t)blockIdx.x * per;
  const int live = g.nsites - first < per ? (int)(g.nsites - first) : per;
  const int r = threadIdx.x % per;
  if (full) parity = threadIdx.x / per;
  const bool mine = r < live;
  char* d = static_cast<char*>(dev) + (full ? parity * half_bytes : 0);
  double2* row2 = reinterpret_cast<double2*>(sh + threadIdx.x * SPIN_PITCH);
  Spinor<T> v;
  if (mine) {
    at[threadIdx.x] = host_site(g, first + r, parity, full) * 24;
    if (!PACK) {
      SpinorIO<P>::load(d, g.sstride, first + r, v);
#pragma unroll
      for (int k = 0; k < 12; k++) row2[k] = make_double2((double)v.v[k].r, (double)v.v[k].i);
    }
  }
  __syncthreads();
  const auto slot = [&](int q) { return full ? (q & 1) * per + (q >> 1) : q; };
  copy_rows<PACK, SPIN_ROWS, SPIN_ROWS, 24, SPIN_PITCH>(sh, host, full ? 2 * live : live, wide, slot,
                                                        [&](int q) { return at[slot(q)]; });
  if (!PACK) return;
  arrived();
  if (!mine) return;
  if constexpr (P == LQCD_F32) {
    // chunk by chunk, so that few values are held at a time
    float4* out = reinterpret_cast<float4*>(d) + first + r;
#pragma unroll
    for (int c = 0; c < 6; c++) {
      const float2 a = to_float2(row2[2 * c]), b = to_float2(row2[2 * c + 1]);
      __stcs(out + c * g.sstride, make_float4(a.x, a.y, b.x, b.y));
    }
  } else {
#pragma unroll
    for (int k = 0; k < 12; k++) {
      const double2 w = row2[k];
      if constexpr (P == LQCD_F64) {
        v.v[k] = mk(w.x, w.y);
      } else {
        const float2 f = to_float2(w);
        v.v[k] = mk(f.x, f.y);
      }
    }
    SpinorIO<P>::store(d, g.sstride, first + r, v);
  }
}

// ---- links: chunk c of block (parity, mu) is at ((blk * NCHUNK + c) * gstride + cb)

// The first R / 2 complex numbers of a link's row as its stored chunks
template <int P, int R>
__device__ __forceinline__ void store_link_row(void* dev, int64_t gs, int blk, int64_t cb, const double2* row) {
  constexpr int N = R / 2;
  if constexpr (P == LQCD_F64) {
    double2* b = static_cast<double2*>(dev) + (int64_t)blk * N * gs + cb;
#pragma unroll
    for (int c = 0; c < N; c++) b[c * gs] = row[c];
  } else if constexpr (P == LQCD_F32) {
    if constexpr (R == 18) {
      float2* b = static_cast<float2*>(dev) + (int64_t)blk * 9 * gs + cb;
#pragma unroll
      for (int c = 0; c < 9; c++) b[c * gs] = to_float2(row[c]);
    } else {
      float4* b = static_cast<float4*>(dev) + (int64_t)blk * 3 * gs + cb;
#pragma unroll
      for (int c = 0; c < 3; c++) {
        const float2 v = to_float2(row[2 * c]), w = to_float2(row[2 * c + 1]);
        b[c * gs] = make_float4(v.x, v.y, w.x, w.y);
      }
    }
  } else {
    if constexpr (R == 18) {
      unsigned int* b = static_cast<unsigned int*>(dev) + (int64_t)blk * 9 * gs + cb;
#pragma unroll
      for (int c = 0; c < 9; c++) b[c * gs] = to_half2(row[c]);
    } else {
      uint2* b = static_cast<uint2*>(dev) + (int64_t)blk * 3 * gs + cb;
#pragma unroll
      for (int c = 0; c < 3; c++) b[c * gs] = make_uint2(to_half2(row[2 * c]), to_half2(row[2 * c + 1]));
    }
  }
}

constexpr int LINK_CB = 32;                // checkerboard sites per block
constexpr int LINK_ROWS = 8 * LINK_CB;     // links per block, one per thread: a warp has one (parity, mu)
constexpr int LINK_PITCH = 18;             // doubles per row in shared memory

// The 2 LINK_CB sites of checkerboard indices first .. first + LINK_CB - 1 are
// consecutive in the host layout (sites 2 cb and 2 cb + 1 are one of each parity),
// so a block reads or writes one run of 8 LINK_CB links; two-row formats pack
// without reading the third row. Link q of the run (site q / 4, mu = q % 4) has
// row (x parity of the site, mu, cb): a warp's rows are then consecutive.
template <int P, int R, bool PACK>
__global__ void __launch_bounds__(LINK_ROWS, 5) gauge_xfer_kernel(void* dev, double* host, Geom g, int wide) {
  using T = typename PrecTraits<P>::real;
  __shared__ __align__(16) double sh[LINK_ROWS * LINK_PITCH];
  const int64_t first = (int64_t)blockIdx.x * LINK_CB;
  const int live = g.Vh - first < LINK_CB ? (int)(g.Vh - first) : LINK_CB;
  const int i = threadIdx.x % LINK_CB, blk = threadIdx.x / LINK_CB;  // blk = parity * 4 + mu
  const bool mine = i < live;
  double2* row = nullptr;
  if (mine) {
    const Coord x = cb_to_coord(g, first + i, blk >> 2);
    row = reinterpret_cast<double2*>(sh + (((x.c[0] & 1) * 4 + (blk & 3)) * LINK_CB + i) * LINK_PITCH);
    if (!PACK) {
      Link<T> u;
      LinkIO<P, R>::load(dev, g.gstride, blk, first + i, u);
#pragma unroll
      for (int k = 0; k < 9; k++) row[k] = make_double2((double)u.v[k].r, (double)u.v[k].i);
    }
  }
  if (!PACK) __syncthreads();
  constexpr int LEN = PACK ? R : 18;
  copy_rows<PACK, LINK_ROWS, LINK_ROWS, LEN, LINK_PITCH>(
      sh, host + first * 144, 8 * live, wide,
      [&](int q) { return (((q >> 2) & 1) * 4 + (q & 3)) * LINK_CB + (q >> 3); }, [&](int q) { return q * 18; });
  if (!PACK) return;
  arrived();
  if (mine) store_link_row<P, R>(dev, g.gstride, blk, first + i, row);
}

static bool misaligned(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) != 0; }

static int spinor_xfer(bool pack, void* dev, double* aos, int prec, int subset, const lqcd_lattice* lat,
                       cudaStream_t s) {
  Geom g;
  int st = make_geom(lat, &g);
  if (st) return st;
  if (spinor_site_bytes(prec) == 0) return fail(LQCD_ERR_ARG, "bad precision %d", prec);
  if (subset != LQCD_EVEN && subset != LQCD_ODD && subset != LQCD_FULL)
    return fail(LQCD_ERR_ARG, "bad subset %d", subset);
  if (!dev || !aos || misaligned(dev) || (reinterpret_cast<uintptr_t>(aos) & 7))
    return fail(LQCD_ERR_ARG, "spinor pack/unpack: null or misaligned pointer");
  const bool full = subset == LQCD_FULL;
  const int64_t per = full ? SPIN_ROWS / 2 : SPIN_ROWS;
  const unsigned grid = (unsigned)((g.nsites + per - 1) / per);
  const int parity = full ? 0 : subset;
  const int wide = (reinterpret_cast<uintptr_t>(aos) & 15) == 0;
  const int64_t hb = (int64_t)cb_spinor_bytes(g, prec);
  if (grid == 0) return LQCD_OK;
#define LQCD_SPINOR_XFER(PR)                                                                            \
  if (pack) spinor_xfer_kernel<PR, true><<<grid, SPIN_ROWS, 0, s>>>(dev, aos, g, parity, full, wide, hb); \
  else spinor_xfer_kernel<PR, false><<<grid, SPIN_ROWS, 0, s>>>(dev, aos, g, parity, full, wide, hb);
  switch (prec) {
    case LQCD_F64: LQCD_SPINOR_XFER(LQCD_F64) break;
    case LQCD_F32: LQCD_SPINOR_XFER(LQCD_F32) break;
    case LQCD_F16: LQCD_SPINOR_XFER(LQCD_F16) break;
  }
#undef LQCD_SPINOR_XFER
  return after_launch(pack ? "spinor_pack" : "spinor_unpack");
}

template <int P, int R>
static void launch_gauge_xfer(bool pack, void* dev, double* aos, const Geom& g, cudaStream_t s) {
  const unsigned grid = (unsigned)((g.Vh + LINK_CB - 1) / LINK_CB);
  const int wide = (reinterpret_cast<uintptr_t>(aos) & 15) == 0;
  if (pack) gauge_xfer_kernel<P, R, true><<<grid, LINK_ROWS, 0, s>>>(dev, aos, g, wide);
  else gauge_xfer_kernel<P, R, false><<<grid, LINK_ROWS, 0, s>>>(dev, aos, g, wide);
}

static int gauge_xfer(bool pack, void* dev, double* aos, int prec, int recon, const lqcd_lattice* lat,
                      cudaStream_t s) {
  Geom g;
  int st = make_geom(lat, &g);
  if (st) return st;
  if (spinor_site_bytes(prec) == 0 || (recon != 18 && recon != 12))
    return fail(LQCD_ERR_ARG, "bad gauge format prec=%d recon=%d", prec, recon);
  if (!dev || !aos || misaligned(dev) || (reinterpret_cast<uintptr_t>(aos) & 7))
    return fail(LQCD_ERR_ARG, "gauge pack/unpack: null or misaligned pointer");
  const bool r18 = recon == 18;
  if (prec == LQCD_F64) (r18 ? launch_gauge_xfer<LQCD_F64, 18> : launch_gauge_xfer<LQCD_F64, 12>)(pack, dev, aos, g, s);
  else if (prec == LQCD_F32) (r18 ? launch_gauge_xfer<LQCD_F32, 18> : launch_gauge_xfer<LQCD_F32, 12>)(pack, dev, aos, g, s);
  else if (prec == LQCD_F16 || pack) (r18 ? launch_gauge_xfer<LQCD_F16, 18> : launch_gauge_xfer<LQCD_F16, 12>)(pack, dev, aos, g, s);
  return after_launch(pack ? "gauge_pack" : "gauge_unpack");
}

static size_t host_spinor_bytes(const Geom& g, int subset) {
  return (size_t)g.nsites * (subset == LQCD_FULL ? 2 : 1) * 24 * sizeof(double);
}

}  // namespace lqcd

using namespace lqcd;

extern "C" {

int lqcd_spinor_pack(void* dst, int prec, int subset, const double* src, const lqcd_lattice* lat, void* stream) {
  return spinor_xfer(true, dst, const_cast<double*>(src), prec, subset, lat, (cudaStream_t)stream);
}

int lqcd_spinor_unpack(double* dst, const void* src, int prec, int subset, const lqcd_lattice* lat, void* stream) {
  return spinor_xfer(false, const_cast<void*>(src), dst, prec, subset, lat, (cudaStream_t)stream);
}

int lqcd_gauge_pack(void* dst, int prec, int recon, const double* src, const lqcd_lattice* lat, void* stream) {
  return gauge_xfer(true, dst, const_cast<double*>(src), prec, recon, lat, (cudaStream_t)stream);
}

int lqcd_gauge_unpack(double* dst, const void* src, int prec, int recon, const lqcd_lattice* lat, void* stream) {
  return gauge_xfer(false, const_cast<void*>(src), dst, prec, recon, lat, (cudaStream_t)stream);
}

int lqcd_spinor_upload(void* dst, int prec, int subset, const double* src_host, double* staging,
                       const lqcd_lattice* lat, void* stream) {
  Geom g;
  int st = make_geom(lat, &g);
  if (st) return st;
  if (!src_host || !staging) return fail(LQCD_ERR_ARG, "lqcd_spinor_upload: null pointer");
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = cudaMemcpyAsync(staging, src_host, host_spinor_bytes(g, subset), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return cuda_fail(e, "lqcd_spinor_upload memcpy");
  return lqcd_spinor_pack(dst, prec, subset, staging, lat, stream);
}

int lqcd_spinor_download(double* dst_host, const void* src, int prec, int subset, double* staging,
                         const lqcd_lattice* lat, void* stream) {
  Geom g;
  int st = make_geom(lat, &g);
  if (st) return st;
  if (!dst_host || !staging) return fail(LQCD_ERR_ARG, "lqcd_spinor_download: null pointer");
  if ((st = lqcd_spinor_unpack(staging, src, prec, subset, lat, stream))) return st;
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = cudaMemcpyAsync(dst_host, staging, host_spinor_bytes(g, subset), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return cuda_fail(e, "lqcd_spinor_download memcpy");
  e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(e, "lqcd_spinor_download sync");
  return LQCD_OK;
}

int lqcd_gauge_upload(void* dst, int prec, int recon, const double* src_host, double* staging,
                      const lqcd_lattice* lat, void* stream) {
  Geom g;
  int st = make_geom(lat, &g);
  if (st) return st;
  if (!src_host || !staging) return fail(LQCD_ERR_ARG, "lqcd_gauge_upload: null pointer");
  cudaStream_t s = (cudaStream_t)stream;
  const size_t bytes = (size_t)2 * g.Vh * 4 * 18 * sizeof(double);
  cudaError_t e = cudaMemcpyAsync(staging, src_host, bytes, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return cuda_fail(e, "lqcd_gauge_upload memcpy");
  return lqcd_gauge_pack(dst, prec, recon, staging, lat, stream);
}

}  // extern "C"
