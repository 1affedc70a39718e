// Site-local kernels: layout and precision conversion, standalone Mooee / Mooee^-1,
// FP64-accumulated reductions and CG vector updates. All are bandwidth-bound passes over the
// device field layout described in dwf_common.cuh.
//
// Elementwise kernels walk a field in units of 16 values: reals 8g..8g+7 of both slices of one pair
// of a site, in the order [real][slice], NV = 8 / RV vectors. Units are numbered [site block][g 0..2]
// [site in block][pair q]: with n = 4 Lsh columns, unit u lies in row u / n and column u % n, and its
// vectors at row * NV chunk strides + column * 16 bytes (+ v chunk strides). Consecutive threads take
// consecutive columns, so every precision's 16-byte vectors are read and written contiguously, and
// fields of different precisions (whose vectors hold 1, 2 or 4 reals of two slices) can be combined in
// one pass. One division by n finds a unit, as a multiplication by 2^64 / n: two 64-bit divisions
// per unit (~100 instructions each) cost the 16-bit passes most (conversion, norm and inner product of
// BF16 full fields at 24^4 x 12: 527 -> 489 us). Pad slices (odd Ls) are zero and stay zero.
#include <algorithm>

#include "dhop_kernel.cuh"
#include "site_ops.cuh"

namespace gdwf {

template <int P>
using RT = typename Store<P>::R;

// Where a unit lies: row (block and g) and column (site in block and pair) of the unit array.
struct UnitMap {
  uint64_t m;      // ceil(2^64 / columns)
  uint32_t cols;   // 4 Lsh
  long units;      // 3 nsites Lsh (nsites a multiple of 4)
};

static inline UnitMap unit_map(long nsites, int Ls) {
  UnitMap u;
  u.cols = (uint32_t)(SITE_BLOCK * ls_half(Ls));
  u.m = ~0ull / u.cols + 1;  // u * cols < 2^64 for every u < 2^56, so that the quotient is exact
  u.units = nsites * 3 * ls_half(Ls);
  return u;
}

// Byte offset of the first of unit u's vectors for a field whose units are NV vectors, and the step
// between its vectors.
template <int P>
__device__ __forceinline__ size_t unit_offset(const UnitMap& um, long u) {
  constexpr int NV = 16 / Store<P>::VEC;
  const uint64_t row = __umul64hi((uint64_t)u, um.m);
  const uint32_t col = (uint32_t)u - (uint32_t)row * um.cols;
  return ((size_t)row * (NV * um.cols) + col) * 16;
}

// The 16 values of unit u.
template <int P, bool COHERENT>
__device__ __forceinline__ void ld_unit(const void* base, const UnitMap& um, long u, RT<P>* o) {
  constexpr int VEC = Store<P>::VEC;
  const char* p = static_cast<const char*>(base) + unit_offset<P>(um, u);
#pragma unroll
  for (int v = 0; v < 16 / VEC; ++v) {
    if (COHERENT)
      ld16c<P>(p + v * um.cols * 16, o + v * VEC);
    else
      ld16<P>(p + v * um.cols * 16, o + v * VEC);
  }
}

template <int P>
__device__ __forceinline__ void st_unit(void* base, const UnitMap& um, long u, const RT<P>* o) {
  constexpr int VEC = Store<P>::VEC;
  char* p = static_cast<char*>(base) + unit_offset<P>(um, u);
#pragma unroll
  for (int v = 0; v < 16 / VEC; ++v) st16<P>(p + v * um.cols * 16, o + v * VEC);
}

template <int P>
__device__ __forceinline__ void st_unit_d(void* base, const UnitMap& um, long u, const double* o) {
  constexpr int VEC = Store<P>::VEC;
  char* p = static_cast<char*>(base) + unit_offset<P>(um, u);
#pragma unroll
  for (int v = 0; v < 16 / VEC; ++v) st16d<P>(p + v * um.cols * 16, o + v * VEC);
}

static inline int grid_for(long n, int threads) {
  long b = (n + threads - 1) / threads;
  return (int)(b < 1 ? 1 : b);
}

// ---------------------------------------------------------------- block reduction

template <int N>
__device__ __forceinline__ void block_sum(double (&v)[N], double* partials, int nblocks) {
  __shared__ double red[N][RED_THREADS / 32];
#pragma unroll
  for (int k = 0; k < N; ++k)
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], off);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < N; ++k) red[k][warp] = v[k];
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      double t = lane < RED_THREADS / 32 ? red[k][lane] : 0.0;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) t += __shfl_down_sync(0xffffffffu, t, off);
      if (lane == 0) partials[k * nblocks + blockIdx.x] = t;
    }
  }
}

// ---------------------------------------------------------------- pack / unpack

// One thread per 16-byte vector of the field, reading or writing the canonical values in pairs where a
// vector holds neighbouring reals; inv_lsh = ceil(2^64 / Lsh). Pack and unpack at 16^4: FP32, Ls = 16
// 118 -> 108 us; FP16, Ls = 16 162 -> 108 us; FP64, Ls = 12 139 -> 119 us (three 64-bit divisions per
// vector before). Conversions in integers (as in k_convert) measured 3-14% slower here.
template <int P>
__global__ void k_pack_spinor(Geom g, double* canon, char* field, int parity0, int nparity, bool unpack,
                              uint64_t inv_lsh) {
  using R = RT<P>;
  constexpr int VEC = Store<P>::VEC, RV = Store<P>::RV, NCH = Store<P>::NCH;
  const long tid = blockIdx.x * (long)blockDim.x + threadIdx.x;
  const int Ls = g.Ls;
  const int Lsh = ls_half(Ls);
  const long total = (long)nparity * g.N4h * NCH * Lsh;
  if (tid >= total) return;
  const long rem = Lsh > 1 ? (long)__umul64hi((uint64_t)tid, inv_lsh) : tid;
  const int q = (int)(tid - rem * Lsh);
  const long sitep = rem / NCH;
  const int k = (int)(rem - sitep * NCH);
  const int ph = sitep >= g.N4h;
  const int i = (int)(sitep - (ph ? g.N4h : 0));
  int c[4];
  cb_coords(g, i, parity0 + ph, c);
  const long lex = c[0] + (long)g.L[0] * (c[1] + (long)g.L[1] * (c[2] + (long)g.L[2] * c[3]));
  char* fp = field + site_offset(sitep, Lsh, (size_t)Lsh * 2 * 24 * sizeof(typename Store<P>::T)) + k * chunk_stride(Lsh) +
             (size_t)q * 16;
  // value 2j + l of the vector is real RV*k + j of slice 2q + l
  double* cp = canon + (lex * Ls + 2 * q) * 24 + RV * k;
  const bool both = 2 * q + 1 < Ls;  // the second slice is not the pad
  if (!unpack) {
    double v[VEC];
#pragma unroll
    for (int l = 0; l < 2; ++l)
#pragma unroll
      for (int j = 0; j < RV; j += RV > 1 ? 2 : 1) {
        if constexpr (RV > 1) {
          double2 d = make_double2(0.0, 0.0);
          if (l == 0 || both) d = *reinterpret_cast<const double2*>(cp + l * 24 + j);
          v[2 * j + l] = d.x;
          v[2 * j + 2 + l] = d.y;
        } else {
          v[2 * j + l] = l == 0 || both ? cp[l * 24 + j] : 0.0;
        }
      }
    st16d<P>(fp, v);
  } else {
    R v[VEC];
    ld16<P>(fp, v);
#pragma unroll
    for (int l = 0; l < 2; ++l)
#pragma unroll
      for (int j = 0; j < RV; j += RV > 1 ? 2 : 1) {
        if (l == 1 && !both) continue;
        if constexpr (RV > 1)
          *reinterpret_cast<double2*>(cp + l * 24 + j) = make_double2((double)v[2 * j + l], (double)v[2 * j + 2 + l]);
        else
          cp[l * 24 + j] = (double)v[2 * j + l];
      }
  }
}

cudaError_t launch_pack_spinor(int prec, const Geom& g, const double* canon, void* field, int subset, bool unpack,
                               cudaStream_t st) {
  const int parity0 = subset == 2 ? 0 : subset;
  const int nparity = subset == 2 ? 2 : 1;
  const long total = (long)nparity * g.N4h * (24 / (prec_vec(prec) / 2)) * ls_half(g.Ls);
  const int blocks = grid_for(total, 256);
  const uint64_t inv = ~0ull / ls_half(g.Ls) + 1;
  double* c = const_cast<double*>(canon);
  char* f = static_cast<char*>(field);
  switch (prec) {
    case P64: k_pack_spinor<P64><<<blocks, 256, 0, st>>>(g, c, f, parity0, nparity, unpack, inv); break;
    case P32: k_pack_spinor<P32><<<blocks, 256, 0, st>>>(g, c, f, parity0, nparity, unpack, inv); break;
    case P16: k_pack_spinor<P16><<<blocks, 256, 0, st>>>(g, c, f, parity0, nparity, unpack, inv); break;
    default: k_pack_spinor<PB16><<<blocks, 256, 0, st>>>(g, c, f, parity0, nparity, unpack, inv); break;
  }
  return cudaGetLastError();
}

template <int P, bool C12>
__global__ void k_pack_gauge(Geom g, const double* canon, char* Ue, char* Uo) {
  using R = RT<P>;
  constexpr int VEC = Store<P>::VEC;
  constexpr int LB = link_bytes(sizeof(typename Store<P>::T), C12);
  constexpr int NR = C12 ? 12 : 18;
  constexpr int NV = LB / 16;
  const long tid = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (tid >= 8L * g.N4h) return;
  const int mu = (int)(tid & 3);
  const long rem = tid >> 2;
  const int p = rem >= g.N4h ? 1 : 0;
  const int i = (int)(rem - (long)p * g.N4h);
  int c[4];
  cb_coords(g, i, p, c);
  const long lex = c[0] + (long)g.L[0] * (c[1] + (long)g.L[1] * (c[2] + (long)g.L[2] * c[3]));
  const double* u = canon + (lex * 4 + mu) * 18;
  char* dst = (p ? Uo : Ue) + ((size_t)i * 4 + mu) * LB;
  double buf[NV * VEC];
#pragma unroll
  for (int j = 0; j < NV * VEC; ++j) buf[j] = j < NR ? u[j] : 0.0;
#pragma unroll
  for (int v = 0; v < NV; ++v) st16d<P>(dst + v * 16, buf + v * VEC);
}

cudaError_t launch_pack_gauge(int prec, bool c12, const Geom& g, const double* canon, void* Ue, void* Uo,
                              cudaStream_t st) {
  const int blocks = grid_for(8L * g.N4h, 256);
  char* e = static_cast<char*>(Ue);
  char* o = static_cast<char*>(Uo);
#define PG(P_)                                                                   \
  if (c12)                                                                       \
    k_pack_gauge<P_, true><<<blocks, 256, 0, st>>>(g, canon, e, o);              \
  else                                                                           \
    k_pack_gauge<P_, false><<<blocks, 256, 0, st>>>(g, canon, e, o);
  switch (prec) {
    case P64: PG(P64) break;
    case P32: PG(P32) break;
    case P16: PG(P16) break;
    default: PG(PB16) break;
  }
#undef PG
  return cudaGetLastError();
}

// ---------------------------------------------------------------- precision conversion

// Conversions between FP64 and the lower precisions would run on the FP64 pipe (2 lanes per SM and
// clock; a conversion and a product by the scale take 1 clock per value against 0.5 of HBM time), so
// the common range is done in integers, with a single rounding:
//   down: the product of the two 53-bit significands to 62 bits, its upper word with the rest as a sticky
//   bit, rounded to FP32 by the integer conversion (for 16-bit storage first to odd at 24 bits, so that
//   the second rounding is exact); up: the bits rearranged.
// Values whose result is not a normal FP32 number (zeros, infinities and NaN among them), and every value
// where the scale lies outside 2^-898 .. 2^897, take the FP64 instructions (product, then conversion).
// 24^4 x 12 half field, FP64 -> FP32 with a scale: 178 -> 80 us (573 MB; part of the writes stays in L2;
// the FP64 pipe 88% busy before, idle now).
struct Scale64 {
  double v;
  uint32_t hi, lo;  // significand, left-justified
  int e;            // exponent
  uint32_t sign;
  bool in_range;    // -898 <= e <= 896
};

__device__ __forceinline__ Scale64 make_scale64(double v) {
  Scale64 s;
  const uint32_t h = (uint32_t)__double2hiint(v), l = (uint32_t)__double2loint(v);
  s.v = v;
  s.hi = __funnelshift_l(l, h, 11) | 0x80000000u;
  s.lo = l << 11;
  s.e = (int)((h >> 20) & 0x7ffu) - 1023;
  s.sign = h & 0x80000000u;
  // then a value whose exponent field is 0 (zero, subnormal: e - 1023) or 0x7ff (infinity, NaN: e + 1024)
  // lies outside narrow64's range of the result's exponent, -126 .. 125
  s.in_range = s.e >= -898 && s.e <= 896;
  return s;
}

// The FP64 instructions stay behind calls: predicated, they would take their pipe's cycles in every warp.
template <int P>
__device__ __noinline__ typename Store<P>::T narrow64_any(double a, double s) {
  const double p = a * s;
  if constexpr (P == P32) return (float)p;
  if constexpr (P == P16) return __double2half(p);
  if constexpr (P == PB16) return __double2bfloat16(p);
}
__device__ __noinline__ double widen32_any(float f) { return (double)f; }

// a * s rounded once to the storage type of P.
template <int P>
__device__ __forceinline__ typename Store<P>::T narrow64(double a, const Scale64& s) {
  const uint32_t h = (uint32_t)__double2hiint(a), l = (uint32_t)__double2loint(a);
  const uint32_t ah = __funnelshift_l(l, h, 11) | 0x80000000u, al = l << 11;
  const int k = (int)((h >> 20) & 0x7ffu) - 1023 + s.e - 30;  // value = q 2^k, q in [2^30, 2^32)
  if ((unsigned)(k + 156) <= 251u && s.in_range) {
    const uint64_t p = (uint64_t)ah * s.hi + __umulhi(ah, s.lo) + __umulhi(al, s.hi);
    uint32_t q = (uint32_t)(p >> 32) | ((uint32_t)p != 0);
    if constexpr (P != P32) q = (q & 0xffffff00u) | ((q & 0xffu) ? 0x100u : 0u);
    const uint32_t bits = (__float_as_uint(__uint2float_rn(q)) + ((uint32_t)k << 23)) | ((h & 0x80000000u) ^ s.sign);
    const float f = __uint_as_float(bits);
    if constexpr (P == P32) return f;
    if constexpr (P == P16) return __float2half_rn(f);
    if constexpr (P == PB16) return __float2bfloat16_rn(f);
  }
  return narrow64_any<P>(a, s.v);
}

// Exact.
__device__ __forceinline__ double widen32(float f) {
  const uint32_t b = __float_as_uint(f), e = (b >> 23) & 0xffu;
  if (e - 1u < 254u)
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
  return widen32_any(f);
}

template <int PS, int PD>
__global__ void k_convert(const void* src, void* dst, UnitMap um, const double* scale_dev, double scale) {
  using RS = RT<PS>;
  using RD = RT<PD>;
  const double sc = scale_dev ? *scale_dev : scale;
  const Scale64 s64 = make_scale64(sc);
  for (long u = blockIdx.x * (long)blockDim.x + threadIdx.x; u < um.units; u += (long)gridDim.x * blockDim.x) {
    RS a[16];
    ld_unit<PS, false>(src, um, u, a);
    if constexpr (PS == P64 && PD != P64) {
      typename Store<PD>::T b[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) b[j] = narrow64<PD>(a[j], s64);
      char* p = static_cast<char*>(dst) + unit_offset<PD>(um, u);
#pragma unroll
      for (int v = 0; v < 16 / Store<PD>::VEC; ++v) {
        uint4 w;
        memcpy(&w, b + v * Store<PD>::VEC, 16);
        *reinterpret_cast<uint4*>(p + v * um.cols * 16) = w;
      }
    } else if constexpr (PD == P64) {
      double b[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        if constexpr (PS == P64)
          b[j] = a[j];
        else
          b[j] = widen32(a[j]);
      }
      if (sc != 1.0) {
#pragma unroll
        for (int j = 0; j < 16; ++j) b[j] *= sc;
      }
      st_unit_d<PD>(dst, um, u, b);
    } else {
      RD b[16];
      const float f = (float)sc;
#pragma unroll
      for (int j = 0; j < 16; ++j) b[j] = (RD)((float)a[j] * f);
      st_unit<PD>(dst, um, u, b);
    }
  }
}

cudaError_t launch_convert(int psrc, int pdst, const void* src, void* dst, long nsites, int Ls, const double* scale_dev,
                           double scale, cudaStream_t st) {
  const UnitMap um = unit_map(nsites, Ls);
  const int blocks = grid_for(um.units, 256);
#define CV(A, B) k_convert<A, B><<<blocks, 256, 0, st>>>(src, dst, um, scale_dev, scale)
#define CVROW(A)            \
  switch (pdst) {           \
    case P64: CV(A, P64); break;  \
    case P32: CV(A, P32); break;  \
    case P16: CV(A, P16); break;  \
    default: CV(A, PB16); break;  \
  }
  switch (psrc) {
    case P64: CVROW(P64) break;
    case P32: CVROW(P32) break;
    case P16: CVROW(P16) break;
    default: CVROW(PB16) break;
  }
#undef CVROW
#undef CV
  return cudaGetLastError();
}

// ---------------------------------------------------------------- standalone Mooee / Mooee^-1

// Up to 32 slice pairs (FP64: the forward operator; the inverse's scan takes 13 FP64 instructions per
// vector against 6 of the two serial sweeps): one thread per 16-byte vector (both slices of pair q for RV reals of one
// site), a site's pairs being consecutive lanes of one warp, so that the coupling to slices s -+ 1 and
// the inverse's recurrence run on shuffles and the field moves through registers once. The inverse
// of the chirality coupled to s - 1 is, with S_s = sum_{1 <= k <= s} b_k d^-(s-k+1),
//   y_0 = (b_0 - m S_{Ls-1}) / (d + m d^-(Ls-1)),  y_s = S_s + d^-s y_0,
// S by a scan over the lanes; y so formed on the pair before feeds the recurrence y_s = (b_s + y_{s-1}) / d
// over a pair's own slices (its rounding damped by 1 / d). The other chirality is the mirror image in s. Bound by memory in FP32 and 16 bits: inverse at 24^4 x 12 full, FP32, 192 -> 131 us
// (5.8 TB/s), forward half field 84 -> 59 us. The shared-memory
// kernel below, which served every case before, stages the field between barriers and runs each
// line's two sweeps serially. Without the compile-time number of scan steps: 174 us.
struct InvPowers {
  double p[65];              // d^-n
  float inv_lo, inv_den_lo;  // 1 / d and 1 / (d + m d^-(Ls-1)) less their FP32 roundings
};

// STEPS = ceil(log2 pairs), ODD = odd Ls (slice 2q + 1 of the last pair is the zero pad).
template <int P, int STEPS, bool ODD>
__global__ void __launch_bounds__(256) k_mooee_vec(const char* in, char* out, uint32_t groups, int Ls, int gpw, bool dag,
                                                   bool inverse, double d5, double mass, double inv_den,
                                                   const __grid_constant__ InvPowers pw) {
  using R = RT<P>;
  constexpr int VEC = Store<P>::VEC, RV = Store<P>::RV, NCH = Store<P>::NCH;
  constexpr int U = P == P64 ? 4 : 2;  // vectors per thread
  const int Lsh = ls_half(Ls);
  const int lane = threadIdx.x & 31;
  const int gl = lane / Lsh, q = lane - gl * Lsh;
  const uint32_t g0 = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * (uint32_t)(U * gpw) + gl;
  __shared__ R pws[65];
  if (threadIdx.x < 65) pws[threadIdx.x] = (R)pw.p[threadIdx.x];
  R v[U][VEC];
  bool act[U];
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const uint32_t G = g0 + j * gpw;  // (site block, chunk, site in block)
    act[j] = gl < gpw && G < groups;
#pragma unroll
    for (int i = 0; i < VEC; ++i) v[j][i] = R(0);
    if (act[j]) ld16c<P>(in + ((size_t)G * Lsh + q) * 16, v[j]);
  }
  __syncthreads();
  const R d = R(d5), m = R(mass);
  const bool pad_pair = ODD && q == Lsh - 1;
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const uint32_t G = g0 + j * gpw;
    const bool upper = (G >> 2) % (uint32_t)NCH < NCH / 2;
    const bool fwd = dag != upper;  // coupled to s - 1
    if (!inverse) {
      // o_s = d b_s + c b_{s -+ 1}, c = -1, and m where it wraps around; the lane that holds the
      // pair before this one in the direction of the coupling, cyclically:
      const int src = fwd ? (q > 0 ? lane - 1 : lane + Lsh - 1) : (q < Lsh - 1 ? lane + 1 : lane - (Lsh - 1));
      const R c = (fwd ? q == 0 : q == Lsh - 1) ? m : R(-1);
#pragma unroll
      for (int r = 0; r < RV; ++r) {
        const R a = v[j][2 * r], b = v[j][2 * r + 1];
        // the slice nearest to the neighbour: the second (first), the only one where the pair ends in the pad
        const R o = __shfl_sync(0xffffffffu, fwd && !pad_pair ? b : a, src & 31);
        // one product and two FMAs per vector, whichever way it couples (FP64 fields are bound by that
        // pipe): the slice coupled to the neighbour's, and the one coupled to it
        const bool first = fwd || pad_pair;
        const R p = first ? a : b, n = first ? b : a;
        const R at_p = d * p + c * o, at_n = d * n - p;
        const R x = first ? at_p : at_n, y = first ? at_n : at_p;
        v[j][2 * r] = x;
        v[j][2 * r + 1] = pad_pair ? R(0) : y;
      }
    } else {
      // position of the pair along the line (0: the one with the slice that the other terms feed into),
      // and of its first slice in line order (-1: the pad, where the line starts beside it)
      const int pos = fwd ? q : Lsh - 1 - q;
      const bool pad_line = ODD && !fwd;
      const bool head = pos == 0, pad_head = pad_line && head;
      const int p0 = pad_line ? 2 * pos - 1 : 2 * pos;
      const int back = fwd ? -1 : 1;
      const int head_lane = (lane - q + (fwd ? 0 : Lsh - 1)) & 31, tail_lane = (lane - q + (fwd ? Lsh - 1 : 0)) & 31;
      // 1 / d as an FP32 pair: the last step of every slice carries no error of the constant
      const R inv_d = pws[1], inv_lo = (R)pw.inv_lo;
      const R cb = pad_head ? R(1) : pws[p0 + 1];
      R cs[STEPS > 0 ? STEPS : 1];
#pragma unroll
      for (int k = 0; k < STEPS; ++k) cs[k] = pws[2 << k];
      const R inv_dn = R(inv_den), inv_dn_lo = (R)pw.inv_den_lo;
      auto over_den = [&](R t) { return fma(t, inv_dn, t * inv_dn_lo); };
      // (b + y) / d without the rounding of b + y (FMAs spelled out here and below: other contractions
      // of the same terms have up to 30% larger errors)
      auto step = [&](R b, R y) { return fma(b, inv_d, fma(y, inv_d, b * inv_lo)); };
#pragma unroll
      for (int r = 0; r < RV; ++r) {
        const R a = fwd ? v[j][2 * r] : v[j][2 * r + 1];  // in line order
        const R b = fwd ? v[j][2 * r + 1] : v[j][2 * r];
        const R b0 = __shfl_sync(0xffffffffu, pad_line ? b : a, head_lane);  // the line's first slice
        // S of the pair's slices: within the pair, then a scan over the pairs before it
        const R s0l = head ? R(0) : a * inv_d;
        R s1 = pad_head ? R(0) : (head ? b : fma(a, inv_d, b)) * inv_d;
#pragma unroll
        for (int k = 0; k < STEPS; ++k) {
          // beyond the line's head the shuffle reads another line: selected away, not scaled by 0 (0 x inf)
          const R t = __shfl_sync(0xffffffffu, s1, (lane + back * (1 << k)) & 31);
          const R f = fma(cs[k], t, s1);
          s1 = pos >= (1 << k) ? f : s1;
        }
        // S_{Ls-1}: on the line's last pair, its second slice unless that is the pad
        R last = s1;
        if (ODD) {
          const R t = __shfl_sync(0xffffffffu, s1, (lane + back) & 31);
          const R f = fma(inv_d, t, s0l), s0 = head ? s0l : f;
          if (fwd) last = s0;
        }
        const R y0 = over_den(fma(-m, __shfl_sync(0xffffffffu, last, tail_lane), b0));
        // y of the pair before, then the recurrence over the pair's own two slices
        const R prev = __shfl_sync(0xffffffffu, fma(cb, y0, s1), (lane + back) & 31);
        const R ya = pad_head ? R(0) : head ? y0 : step(a, prev);
        const R yb = fwd && pad_pair ? R(0) : pad_head ? y0 : step(b, ya);
        v[j][2 * r] = fwd ? ya : yb;
        v[j][2 * r + 1] = fwd ? yb : ya;
      }
    }
    if (act[j]) st16<P>(out + ((size_t)G * Lsh + q) * 16, v[j]);
  }
}

template <int P>
static void launch_mooee_vec(const void* in, void* out, long nsites, int Ls, bool dag, bool inverse, double d5,
                             double mass, double inv_den, const InvPowers& pw, cudaStream_t st) {
  const int Lsh = ls_half(Ls), gpw = 32 / Lsh;  // lines' vectors per warp
  int steps = 0;
  while ((1 << steps) < Lsh) ++steps;
  // 2^26 sites at most per launch, whose vectors per pair (24 per site in FP64) a 32-bit index counts
  constexpr long STEP = 1L << 26;
  for (long first = 0; first < nsites; first += STEP) {
    const uint32_t groups = (uint32_t)(std::min(STEP, nsites - first) * Store<P>::NCH);
    const int blocks = grid_for(groups, 8 * gpw * (P == P64 ? 4 : 2));
    const size_t at = (size_t)first * Lsh * Store<P>::NCH * 16;
    const char* i = static_cast<const char*>(in) + at;
    char* o = static_cast<char*>(out) + at;
#define MV(S_)                                                                                                        \
  case S_:                                                                                                            \
    if (Ls & 1)                                                                                                       \
      k_mooee_vec<P, S_, true><<<blocks, 256, 0, st>>>(i, o, groups, Ls, gpw, dag, inverse, d5, mass, inv_den, pw);   \
    else                                                                                                              \
      k_mooee_vec<P, S_, false><<<blocks, 256, 0, st>>>(i, o, groups, Ls, gpw, dag, inverse, d5, mass, inv_den, pw);  \
    break;
    switch (steps) { MV(0) MV(1) MV(2) MV(3) MV(4) MV(5) }
  }
#undef MV
}

// More than 32 pairs, and the FP64 inverse: one CTA holds `spc` whole sites in shared memory (FP32 or FP64 arithmetic):
// load, apply the fifth-dimension operator, store. in and out may be the same buffer.
// Unit number of (site, g, pair q).
__device__ __forceinline__ long unit_of(long site, int g, int q, int Lsh) {
  return ((site >> 2) * 3 + g) * (SITE_BLOCK * Lsh) + (site & 3) * Lsh + q;
}

template <int P>
__global__ void __launch_bounds__(256) k_mooee(const void* in, void* out, UnitMap um, long nsites, int Ls, int spc, bool dag,
                                               bool inverse, double d5, double mass, double inv_d5, double inv_den) {
  using R = RT<P>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  R* sm = reinterpret_cast<R*>(smem_raw);  // [site][s < Ls][24 reals, padded to INV_SLICE_STRIDE]
  constexpr int S = INV_SLICE_STRIDE;
  const int Lsh = ls_half(Ls);
  const long site0 = (long)blockIdx.x * spc;
  const int ns = (int)min((long)spc, nsites - site0);
  const int units = ns * 3 * Lsh;
  for (int u = threadIdx.x; u < units; u += blockDim.x) {
    const int rem = u / Lsh;
    const int q = u - rem * Lsh;
    const int sl = rem / 3;
    const int g = rem - sl * 3;
    R v[16];
    ld_unit<P, true>(in, um, unit_of(site0 + sl, g, q, Lsh), v);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int s = 2 * q + (i & 1);
      if (s < Ls) sm[((size_t)sl * Ls + s) * S + 8 * g + (i >> 1)] = v[i];
    }
  }
  __syncthreads();
  if (inverse) {
    for (int task = threadIdx.x; task < ns * 24; task += blockDim.x) {
      const int sl = task / 24;
      const int r = task - sl * 24;
      const bool upper = r < 12;
      R* line = sm + (size_t)sl * Ls * S + r;
      if constexpr (P == P64)
        mooee_inv_line64<0>(line, Ls, dag ? !upper : upper, mass, inv_d5, inv_den);
      else
        mooee_inv_line<R>(line, Ls, dag ? !upper : upper, R(mass), R(inv_d5), R(inv_den));
    }
    __syncthreads();
    for (int u = threadIdx.x; u < units; u += blockDim.x) {
      const int rem = u / Lsh;
      const int q = u - rem * Lsh;
      const int sl = rem / 3;
      const int g = rem - sl * 3;
      R o[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int s = 2 * q + (i & 1);
        o[i] = s < Ls ? sm[((size_t)sl * Ls + s) * S + 8 * g + (i >> 1)] : R(0);
      }
      st_unit<P>(out, um, unit_of(site0 + sl, g, q, Lsh), o);
    }
    return;
  }
  for (int u = threadIdx.x; u < units; u += blockDim.x) {
    const int rem = u / Lsh;
    const int q = u - rem * Lsh;
    const int sl = rem / 3;
    const int g = rem - sl * 3;
    const R* base = sm + (size_t)sl * Ls * S;
    R o[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int s = 2 * q + (i & 1);
      const int r = 8 * g + (i >> 1);
      if (s >= Ls) {
        o[i] = R(0);
        continue;
      }
      const int sm1 = s > 0 ? s - 1 : Ls - 1, sp1 = s < Ls - 1 ? s + 1 : 0;
      const R cm = s > 0 ? R(-1) : R(mass), cp = s < Ls - 1 ? R(-1) : R(mass);
      const int s_up = dag ? sp1 : sm1, s_lo = dag ? sm1 : sp1;
      const R c_up = dag ? cp : cm, c_lo = dag ? cm : cp;
      const bool upper = r < 12;
      o[i] = R(d5) * base[s * S + r] + (upper ? c_up * base[s_up * S + r] : c_lo * base[s_lo * S + r]);
    }
    st_unit<P>(out, um, unit_of(site0 + sl, g, q, Lsh), o);
  }
}

cudaError_t launch_mooee(int prec, const void* in, void* out, long nsites, int Ls, bool dag, bool inverse, double d5,
                         double mass, double inv_d5, double inv_den, cudaStream_t st) {
  const int Lsh = ls_half(Ls);
  if (Lsh <= 32 && !(prec == P64 && inverse)) {
    InvPowers pw;
    pw.p[0] = 1.0;
    for (int n = 1; n <= 64; ++n) pw.p[n] = pw.p[n - 1] * inv_d5;
    pw.inv_lo = (float)(inv_d5 - (double)(float)inv_d5);
    pw.inv_den_lo = (float)(inv_den - (double)(float)inv_den);
    switch (prec) {
      case P64: launch_mooee_vec<P64>(in, out, nsites, Ls, dag, inverse, d5, mass, inv_den, pw, st); break;
      case P32: launch_mooee_vec<P32>(in, out, nsites, Ls, dag, inverse, d5, mass, inv_den, pw, st); break;
      case P16: launch_mooee_vec<P16>(in, out, nsites, Ls, dag, inverse, d5, mass, inv_den, pw, st); break;
      default: launch_mooee_vec<PB16>(in, out, nsites, Ls, dag, inverse, d5, mass, inv_den, pw, st); break;
    }
    return cudaGetLastError();
  }
  const size_t rbytes = prec == P64 ? 8 : 4;
  const size_t site_smem = (size_t)Ls * INV_SLICE_STRIDE * rbytes;
  int spc = (int)((48 * 1024) / site_smem);
  if (spc > 64) spc = 64;
  if (spc < 1) return cudaErrorInvalidValue;
  const size_t smem = spc * site_smem;
  const int blocks = grid_for(nsites, spc);
#define MO(P_) k_mooee<P_><<<blocks, 256, smem, st>>>(in, out, unit_map(nsites, Ls), nsites, Ls, spc, dag, inverse, d5, mass, inv_d5, inv_den)
  switch (prec) {
    case P64: MO(P64); break;
    case P32: MO(P32); break;
    case P16: MO(P16); break;
    default: MO(PB16); break;
  }
#undef MO
  return cudaGetLastError();
}

// ---------------------------------------------------------------- reductions

// Sum over 8 reals of a unit: |a|^2, or the complex a^+ b. Lower precisions form the 8-term
// partial in FP32 and add it to the FP64 accumulator; FP64 data is accumulated in FP64.
template <int P, bool INNER>
__global__ void __launch_bounds__(RED_THREADS) k_reduce(const void* a, const void* b, UnitMap um,
                                                        double* partials, const Final f) {
  using R = RT<P>;
  double acc[2] = {0.0, 0.0};
  for (long u = blockIdx.x * (long)blockDim.x + threadIdx.x; u < um.units; u += (long)gridDim.x * blockDim.x) {
    R x[16];
    ld_unit<P, false>(a, um, u, x);
    if (INNER) {
      R y[16];
      ld_unit<P, false>(b, um, u, y);
      R re = 0, im = 0;
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int l = 0; l < 2; ++l) {
          const int ir = (2 * c) * 2 + l, ii = (2 * c + 1) * 2 + l;  // re and im of one complex number
          re += x[ir] * y[ir] + x[ii] * y[ii];
          im += x[ir] * y[ii] - x[ii] * y[ir];
        }
      acc[0] += (double)re;
      acc[1] += (double)im;
    } else {
      R t = 0;
#pragma unroll
      for (int j = 0; j < 16; ++j) t += x[j] * x[j];
      acc[0] += (double)t;
    }
  }
  if (INNER) {
    block_sum<2>(acc, partials, RED_BLOCKS);
    finish_sums<2>(partials, RED_BLOCKS, f);
  } else {
    double v[1] = {acc[0]};
    block_sum<1>(v, partials, RED_BLOCKS);
    finish_sums<1>(partials, RED_BLOCKS, f);
  }
}

cudaError_t launch_reduce(int prec, const void* a, const void* b, long nsites, int Ls, double* partials, const Final& f,
                          cudaStream_t st) {
  const bool inner = b != nullptr;
#define RD(P_)                                                                              \
  if (inner)                                                                                \
    k_reduce<P_, true><<<RED_BLOCKS, RED_THREADS, 0, st>>>(a, b, unit_map(nsites, Ls), partials, f);     \
  else                                                                                      \
    k_reduce<P_, false><<<RED_BLOCKS, RED_THREADS, 0, st>>>(a, b, unit_map(nsites, Ls), partials, f);
  switch (prec) {
    case P64: RD(P64) break;
    case P32: RD(P32) break;
    case P16: RD(P16) break;
    default: RD(PB16) break;
  }
#undef RD
  return cudaGetLastError();
}

// ---------------------------------------------------------------- CG updates

template <int PX, int PP>
__global__ void __launch_bounds__(RED_THREADS) k_cg_xr(void* x, void* r, const void* p, const void* Ap, UnitMap um, double* partials, const Final f) {
  using RX = RT<PX>;
  using RP = RT<PP>;
  const RX alpha = (RX)f.scal[S_ALPHA];
  double acc = 0.0;
  for (long u = blockIdx.x * (long)blockDim.x + threadIdx.x; u < um.units; u += (long)gridDim.x * blockDim.x) {
    RX xv[16], rv[16];
    RP pv[16], av[16];
    ld_unit<PX, true>(x, um, u, xv);
    ld_unit<PX, true>(r, um, u, rv);
    ld_unit<PP, false>(p, um, u, pv);
    ld_unit<PP, false>(Ap, um, u, av);
    RX t = 0;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      xv[j] += alpha * (RX)pv[j];
      rv[j] -= alpha * (RX)av[j];
      t += rv[j] * rv[j];
    }
    st_unit<PX>(x, um, u, xv);
    st_unit<PX>(r, um, u, rv);
    acc += (double)t;
  }
  double v[1] = {acc};
  block_sum<1>(v, partials, RED_BLOCKS);
  finish_sums<1>(partials, RED_BLOCKS, f);
}

template <int PX, int PP>
__global__ void k_cg_p(const void* r, void* p, UnitMap um, const double* scal) {
  using RX = RT<PX>;
  using RP = RT<PP>;
  const RX beta = (RX)scal[S_BETA];
  for (long u = blockIdx.x * (long)blockDim.x + threadIdx.x; u < um.units; u += (long)gridDim.x * blockDim.x) {
    RX rv[16];
    RP pv[16];
    ld_unit<PX, false>(r, um, u, rv);
    ld_unit<PP, true>(p, um, u, pv);
#pragma unroll
    for (int j = 0; j < 16; ++j) pv[j] = (RP)(rv[j] + beta * (RX)pv[j]);
    st_unit<PP>(p, um, u, pv);
  }
}

// The mixed solver's inner loop, with the x update deferred by one pass so that p is read once
// per iteration: k_cg_r forms r -= alpha Ap and |r|^2 (reads r, Ap), then k_cg_xp forms
// x += alpha p and p = r + beta p from the same read of p (reads x, r, p). Ten field passes per
// iteration (with p^+ Ap) instead of eleven. k_cg_x applies the pending x update alone, before a
// reliable update folds x into the FP64 solution.
template <int PX, int PP>
__global__ void __launch_bounds__(RED_THREADS) k_cg_r(void* r, const void* Ap, UnitMap um, double* partials, const Final f) {
  using RX = RT<PX>;
  using RP = RT<PP>;
  const RX alpha = (RX)f.scal[S_ALPHA];
  double acc = 0.0;
  for (long u = blockIdx.x * (long)blockDim.x + threadIdx.x; u < um.units; u += (long)gridDim.x * blockDim.x) {
    RX rv[16];
    RP av[16];
    ld_unit<PX, true>(r, um, u, rv);
    ld_unit<PP, false>(Ap, um, u, av);
    RX t = 0;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      rv[j] -= alpha * (RX)av[j];
      t += rv[j] * rv[j];
    }
    st_unit<PX>(r, um, u, rv);
    acc += (double)t;
  }
  double v[1] = {acc};
  block_sum<1>(v, partials, RED_BLOCKS);
  finish_sums<1>(partials, RED_BLOCKS, f);
}

template <int PX, int PP, bool UPDATE_P>
__global__ void k_cg_xp(void* x, const void* r, void* p, UnitMap um, const double* scal) {
  using RX = RT<PX>;
  using RP = RT<PP>;
  const RX alpha = (RX)scal[S_ALPHA];
  const RX beta = (RX)scal[S_BETA];
  for (long u = blockIdx.x * (long)blockDim.x + threadIdx.x; u < um.units; u += (long)gridDim.x * blockDim.x) {
    RX xv[16], rv[16];
    RP pv[16];
    ld_unit<PX, true>(x, um, u, xv);
    ld_unit<PP, UPDATE_P>(p, um, u, pv);  // coherent when p is rewritten
    if (UPDATE_P) ld_unit<PX, false>(r, um, u, rv);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      xv[j] += alpha * (RX)pv[j];
      if (UPDATE_P) pv[j] = (RP)(rv[j] + beta * (RX)pv[j]);
    }
    st_unit<PX>(x, um, u, xv);
    if (UPDATE_P) st_unit<PP>(p, um, u, pv);
  }
}

#define CG_PAIRS(M) \
  M(P64, P64)       \
  M(P32, P32)       \
  M(P32, P16)       \
  M(P32, PB16)

cudaError_t launch_cg_xr(int px, int pp, void* x, void* r, const void* p, const void* Ap, long nsites, int Ls,
                         double* partials, const Final& f, cudaStream_t st) {
#define XR(A, B)                                                                                  \
  if (px == A && pp == B) {                                                                       \
    k_cg_xr<A, B><<<RED_BLOCKS, RED_THREADS, 0, st>>>(x, r, p, Ap, unit_map(nsites, Ls), partials, f);  \
    return cudaGetLastError();                                                                    \
  }
  CG_PAIRS(XR)
#undef XR
  return cudaErrorInvalidValue;
}

cudaError_t launch_cg_r(int px, int pp, void* r, const void* Ap, long nsites, int Ls, double* partials, const Final& f,
                        cudaStream_t st) {
#define RU(A, B)                                                                             \
  if (px == A && pp == B) {                                                                  \
    k_cg_r<A, B><<<RED_BLOCKS, RED_THREADS, 0, st>>>(r, Ap, unit_map(nsites, Ls), partials, f);    \
    return cudaGetLastError();                                                               \
  }
  CG_PAIRS(RU)
#undef RU
  return cudaErrorInvalidValue;
}

cudaError_t launch_cg_xp(int px, int pp, void* x, const void* r, void* p, long nsites, int Ls, const double* scal,
                         bool update_p, cudaStream_t st) {
  const UnitMap um = unit_map(nsites, Ls);
  const int blocks = grid_for(um.units, 256);
#define XP(A, B)                                                                                        \
  if (px == A && pp == B) {                                                                             \
    if (update_p)                                                                                       \
      k_cg_xp<A, B, true><<<blocks, 256, 0, st>>>(x, r, p, um, scal);                          \
    else                                                                                                \
      k_cg_xp<A, B, false><<<blocks, 256, 0, st>>>(x, r, p, um, scal);                         \
    return cudaGetLastError();                                                                          \
  }
  CG_PAIRS(XP)
#undef XP
  return cudaErrorInvalidValue;
}

cudaError_t launch_cg_p(int px, int pp, const void* r, void* p, long nsites, int Ls, const double* scal,
                        cudaStream_t st) {
  const UnitMap um = unit_map(nsites, Ls);
  const int blocks = grid_for(um.units, 256);
#define PU(A, B)                                                              \
  if (px == A && pp == B) {                                                   \
    k_cg_p<A, B><<<blocks, 256, 0, st>>>(r, p, um, scal);             \
    return cudaGetLastError();                                                \
  }
  CG_PAIRS(PU)
#undef PU
  return cudaErrorInvalidValue;
}

__global__ void __launch_bounds__(RED_THREADS) k_residual64(const void* b, const void* Ax, void* r, UnitMap um,
                                                            double* partials, const Final f) {
  double acc = 0.0;
  for (long u = blockIdx.x * (long)blockDim.x + threadIdx.x; u < um.units; u += (long)gridDim.x * blockDim.x) {
    double bv[16], av[16];
    ld_unit<P64, false>(b, um, u, bv);
    ld_unit<P64, false>(Ax, um, u, av);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      bv[j] -= av[j];
      acc += bv[j] * bv[j];
    }
    st_unit<P64>(r, um, u, bv);
  }
  double v[1] = {acc};
  block_sum<1>(v, partials, RED_BLOCKS);
  finish_sums<1>(partials, RED_BLOCKS, f);
}

cudaError_t launch_residual64(const void* b, const void* Ax, void* r, long nsites, int Ls, double* partials,
                              const Final& f, cudaStream_t st) {
  k_residual64<<<RED_BLOCKS, RED_THREADS, 0, st>>>(b, Ax, r, unit_map(nsites, Ls), partials, f);
  return cudaGetLastError();
}

template <int PY>
__global__ void k_accum_zero(void* x, void* y, UnitMap um, const double* c_dev) {
  using RY = RT<PY>;
  const double c = *c_dev;
  for (long u = blockIdx.x * (long)blockDim.x + threadIdx.x; u < um.units; u += (long)gridDim.x * blockDim.x) {
    double xv[16];
    RY yv[16];
    ld_unit<P64, true>(x, um, u, xv);
    ld_unit<PY, true>(y, um, u, yv);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      xv[j] += c * (double)yv[j];
      yv[j] = RY(0);
    }
    st_unit<P64>(x, um, u, xv);
    st_unit<PY>(y, um, u, yv);
  }
}

cudaError_t launch_accum_zero(int py, void* x, void* y, long nsites, int Ls, const double* c_dev, cudaStream_t st) {
  const UnitMap um = unit_map(nsites, Ls);
  const int blocks = grid_for(um.units, 256);
  switch (py) {
    case P64: k_accum_zero<P64><<<blocks, 256, 0, st>>>(x, y, um, c_dev); break;
    case P32: k_accum_zero<P32><<<blocks, 256, 0, st>>>(x, y, um, c_dev); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}
}  // namespace gdwf

// ---------------------------------------------------------------- reduction without allocation
//
// grid_dwf_inner_noalloc: the same FP64-accumulated reduction as launch_reduce, for callers
// that must not allocate device memory, with its scratch in a fixed array that is part of the
// library's device image instead of a cudaMalloc'd buffer. Each CTA reduces one contiguous
// chunk of NOALLOC_UNITS_PER_CTA units (16 values each), so the number of partial sums, and with
// it the largest field accepted, is bounded by the array.

namespace gdwf {

constexpr int NOALLOC_UNITS_PER_THREAD = 8;
constexpr long NOALLOC_UNITS_PER_CTA = (long)RED_THREADS * NOALLOC_UNITS_PER_THREAD;
constexpr int NOALLOC_MAX_PARTIALS = 16384;
constexpr int NOALLOC_MAX_DEVICES = 64;

// [re partials][im partials]: 256 KiB on every device that loads the library, held until the
// process exits.
static __device__ __align__(256) double g_noalloc_scratch[2 * NOALLOC_MAX_PARTIALS];

template <int P, bool INNER>
__global__ void __launch_bounds__(RED_THREADS) k_reduce_chunked(const void* a, const void* b, UnitMap um,
                                                                double* partials, int nblocks) {
  using R = RT<P>;
  double acc[2] = {0.0, 0.0};
  const long first = (long)blockIdx.x * NOALLOC_UNITS_PER_CTA;
#pragma unroll
  for (int k = 0; k < NOALLOC_UNITS_PER_THREAD; ++k) {
    const long u = first + threadIdx.x + (long)k * RED_THREADS;
    if (u >= um.units) break;
    R x[16];
    ld_unit<P, false>(a, um, u, x);
    if (INNER) {
      R y[16];
      ld_unit<P, false>(b, um, u, y);
      R re = 0, im = 0;
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int l = 0; l < 2; ++l) {
          const int ir = (2 * c) * 2 + l, ii = (2 * c + 1) * 2 + l;  // re and im of one complex number
          re += x[ir] * y[ir] + x[ii] * y[ii];
          im += x[ir] * y[ii] - x[ii] * y[ir];
        }
      acc[0] += (double)re;
      acc[1] += (double)im;
    } else {
      R t = 0;
#pragma unroll
      for (int j = 0; j < 16; ++j) t += x[j] * x[j];
      acc[0] += (double)t;
    }
  }
  block_sum<2>(acc, partials, nblocks);
}

// One CTA adds the nblocks partials in a fixed order and writes (re, im) to out.
__global__ void __launch_bounds__(RED_THREADS) k_finalize_chunked(const double* partials, int nblocks, double* out) {
  __shared__ double red[2][RED_THREADS];
  for (int k = 0; k < 2; ++k) {
    double t = 0;
    for (int i = threadIdx.x; i < nblocks; i += RED_THREADS) t += partials[k * nblocks + i];
    red[k][threadIdx.x] = t;
  }
  __syncthreads();
  for (int w = RED_THREADS / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w)
      for (int k = 0; k < 2; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = red[0][0];
    out[1] = red[1][0];
  }
}

}  // namespace gdwf

#include <mutex>
#include <string>

#include "../../include/grid_dwf.h"

namespace {

double* g_noalloc_dev_ptr[gdwf::NOALLOC_MAX_DEVICES] = {};
std::mutex g_noalloc_mutex;

int noalloc_error(char* err, size_t err_len, int code, const std::string& msg) {
  if (err && err_len > 0) {
    const size_t n = msg.size() < err_len - 1 ? msg.size() : err_len - 1;
    memcpy(err, msg.data(), n);
    err[n] = '\0';
  }
  return code;
}

}  // namespace

extern "C" int grid_dwf_inner_noalloc(int precision, const void* a, const void* b, long nsites, int Ls, void* stream,
                                      double* result, char* err, size_t err_len) {
  using namespace gdwf;
  if (err && err_len > 0) err[0] = '\0';
  if (precision < GRID_DWF_FP64 || precision > GRID_DWF_BF16)
    return noalloc_error(err, err_len, GRID_DWF_ERR_INVALID_ARG, "grid_dwf_inner_noalloc: bad precision");
  if (!a || !result || nsites < 0 || Ls < 1)
    return noalloc_error(err, err_len, GRID_DWF_ERR_INVALID_ARG, "grid_dwf_inner_noalloc: null pointer or bad size");
  // Sites are stored in blocks of SITE_BLOCK: a partial last block would make the kernel read the
  // chunks of a whole block past the end of a buffer sized for nsites sites.
  if (nsites % SITE_BLOCK != 0)
    return noalloc_error(err, err_len, GRID_DWF_ERR_INVALID_ARG,
                         "grid_dwf_inner_noalloc: nsites must be a multiple of " + std::to_string(SITE_BLOCK) +
                             " (fields hold whole blocks of 4 checkerboard sites)");
  if (reinterpret_cast<uintptr_t>(a) % 16 || (b && reinterpret_cast<uintptr_t>(b) % 16) ||
      reinterpret_cast<uintptr_t>(result) % 8)
    return noalloc_error(err, err_len, GRID_DWF_ERR_INVALID_ARG, "grid_dwf_inner_noalloc: misaligned pointer");
  const long Lsh = ls_half(Ls);
  const long units = nsites * 3L * Lsh;  // 16 values (8 reals of a slice pair) each
  const long nblocks = (units + NOALLOC_UNITS_PER_CTA - 1) / NOALLOC_UNITS_PER_CTA;
  if (nsites > 0 && (units / 3 / Lsh != nsites || nblocks > NOALLOC_MAX_PARTIALS))
    return noalloc_error(err, err_len, GRID_DWF_ERR_INVALID_ARG,
                         "grid_dwf_inner_noalloc: field of " + std::to_string(nsites) + " sites x Ls " +
                             std::to_string(Ls) + " exceeds the static scratch (at most " +
                             std::to_string((long)NOALLOC_MAX_PARTIALS * NOALLOC_UNITS_PER_CTA / 3 * 2) +
                             " five-dimensional sites, nsites * Ls rounded up to even)");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess)
    return noalloc_error(err, err_len, GRID_DWF_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES)
    return noalloc_error(err, err_len, GRID_DWF_ERR_INVALID_ARG, "grid_dwf_inner_noalloc: device index too large");
  double* scratch = nullptr;
  {
    // Set-up, once per device, with that device current: the device address of the array.
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_dev_ptr[dev]) {
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess)
        return noalloc_error(err, err_len, GRID_DWF_ERR_CUDA,
                             std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
      g_noalloc_dev_ptr[dev] = static_cast<double*>(p);
    }
    scratch = g_noalloc_dev_ptr[dev];
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int nb = nblocks > 0 ? (int)nblocks : 1;
  const bool inner = b != nullptr;
  const UnitMap um = unit_map(nsites, Ls);
#define NA(P_)                                                                                         \
  if (inner)                                                                                           \
    k_reduce_chunked<P_, true><<<nb, RED_THREADS, 0, st>>>(a, b, um, scratch, nb);             \
  else                                                                                                 \
    k_reduce_chunked<P_, false><<<nb, RED_THREADS, 0, st>>>(a, b, um, scratch, nb);
  switch (precision) {
    case P64: NA(P64) break;
    case P32: NA(P32) break;
    case P16: NA(P16) break;
    default: NA(PB16) break;
  }
#undef NA
  k_finalize_chunked<<<1, RED_THREADS, 0, st>>>(scratch, nb, result);
  e = cudaGetLastError();
  if (e != cudaSuccess)
    return noalloc_error(err, err_len, GRID_DWF_ERR_CUDA, std::string("launch: ") + cudaGetErrorString(e));
  return GRID_DWF_OK;
}
