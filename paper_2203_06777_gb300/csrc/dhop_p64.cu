// The FP64 hopping stencil. Fields and links are FP64 in memory; the colour products, the only
// part with a large operation count, run as integer multiply-adds.
//
// What bounds it. This part's FP64 pipe retires 2 fused multiply-adds per SM and clock, its 32-bit
// integer multiplier 64 (32 x 32 + 64 -> 64 bits, both measured with throughput loops). One hop of a
// site and slice is 12 additions (projection), 72 FMAs (link times half spinor) and 24 FMAs
// (accumulation), so a kernel in IEEE FP64 instructions spends 864 of them, 432 clocks, per 5D site
// and measured 762 us per 16^4 x 16 half lattice (94% of that pipe, 5% of HBM). With the whole sum in
// integers only the conversion of the 24 results stays on the FP64 pipe: 241 us per half lattice (233 us
// before the check of small components, below). About 10,500 integer instructions per 5D site, on the
// shift/logic pipe (55% busy) and the multiplier, bound it now (57% of the issue slots; occupancies of 16
// to 28 warps per SM run within 7%). Without that check, IEEE additions for the projection measured 235 us,
// and one thread per slice (168 registers, 12 warps per SM) 280 us.
//
// The arithmetic. The 24 reals of a neighbour's (site, slice) become a block of integers with one
// binary exponent, that of the largest; so does every link, once, when the links are uploaded.
// Every integer is held as two signed digits, x = d1 2^32 + 16 d0. Half spinors are formed on the
// digits (exactly; |d1| < 2^30, |d0| < 2^29, for links 2^30 and 2^28), and a complex product sum is
//   sum x y / 2^64 = sum d1 e1 + (sum d1 e0 + d0 e1) / 2^28    (the products d0 e0 dropped),
// two exact 64-bit sums per real: 6 x 2^60 < 2^63 and 6 (2^59 + 2^58) < 2^63. The sum is rounded
// once into a 64-bit accumulator per output real that has its own exponent per (site, slice): four
// bits above the first hop's, raised (with a rounded shift) when a later hop would need more.
// Error: the truncations of a hop are 2^-57 of (largest |psi|) x (largest |U|) and its rounding into
// the accumulator 2^-55, against 2^-53 of every partial sum in IEEE arithmetic; against 64-bit
// arithmetic by another program, 2-norm, 16^4 x 16: 1.57e-16 (1.97e-16 with IEEE instructions; the
// rounding of the stored result alone is 1.1e-16). They are relative to the largest real of the
// neighbour's (site, slice), not to each component by itself.
//
// A component much smaller than its block's largest real keeps fewer bits than an IEEE sum of its own
// terms would, which matters where the large reals take no part in it (other spins or, on diagonal links,
// other colours). So the kernel adds up |re| + |im| of U h for each colour, over the x and y hops and over
// z and t (9 of about 640 instructions per thread and hop; Mpc^+ Mpc at 16^4 x 16 1016 -> 1050 us), and a
// (site, slice) with a complex component for which neither sum reaches an eighth of the smallest product of
// two blocks' largest reals (2^53 accumulator units) is computed with IEEE FP64 instructions. The errors
// above are at most 92 units per real over the eight hops (about 1 unit rms), so a component's error is at
// most 2^-42 of the sum of its terms' magnitudes; measured against quadruple precision (8^4 x 8, Gaussian
// fields, point and wall propagators, random and smooth links) rms 0.12-0.37 x 2^-53, 99.9% below 2.1 x 2^-53,
// all below 10 x 2^-53; in IEEE instructions 0.34-0.45, 2.0 and 3.7. Gaussian fields stay above the limit (none of 4e5 simulated sites below), propagators on random
// and on smooth links nearly everywhere (3e-5 of the sites of an 8^4 x 8 point source's); a limit of 2^53
// would send 17-43% of the latter to IEEE instructions. Components all of whose terms are 0 (a source's
// empty spins and colours) come out exactly 0 either way and stay.
//
// IEEE instructions also where a neighbour or link does not fit (largest magnitude outside 2^-400 ..
// 2^400 and not zero, which includes infinities, NaN and subnormals).
//
// Code shape. Two threads (neighbouring lanes) per (site, slice), one for each spin k of the half
// spinor: thread k forms h_k, multiplies it by the link and accumulates it into spin k and into the
// lower spin that it reconstructs, spin 3 - k for the x and y hops (handed to the other lane at the
// end) and spin 2 + k for the z and t hops. Each lane owns spins k and 2 + k of the result. The hop
// loop is rolled and its body serves every direction: the spins that a projection adds are read
// at a hop-dependent address with their signs flipped by a mask, backward links are staged as
// their adjoints and the boundary phase is folded into the staged link.
#include "dhop_kernel.cuh"
#include "fx_arith.cuh"

namespace gdwf {
namespace {

constexpr int FX_BAD = -1;                // link exponent of a link that does not fit
constexpr int FX_MIN_TERMS = 1 << 18;     // 2^50 accumulator units, an eighth of the smallest product of two blocks
constexpr int FX_HOP_BYTES = FX_LINK_BYTES;  // staged: 9 complex entries, then {exponent, neighbour, entries not 0}
// 16 bytes of padding per site: two sites read by one warp fall on different banks
constexpr int FX_SITE_BYTES = 8 * FX_HOP_BYTES + 16;

// Links of every site as blocks of digits: entry (a, b) is {re d1, re d0, im d1, im d0}, then the
// exponent and which entries are not 0. One thread per link.
template <bool C12>
__global__ void k_pack_gauge_fx(Geom g, const double* canon, char* Ue, char* Uo) {
  const long tid = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (tid >= 8L * g.N4h) return;
  const int mu = (int)(tid & 3);
  const long rem = tid >> 2;
  const int p = rem >= g.N4h ? 1 : 0;
  const int i = (int)(rem - (long)p * g.N4h);
  int c[4];
  cb_coords(g, i, p, c);
  const long lex = c[0] + (long)g.L[0] * (c[1] + (long)g.L[1] * (c[2] + (long)g.L[2] * c[3]));
  const double* src = canon + (lex * 4 + mu) * 18;
  double u[18];
#pragma unroll
  for (int j = 0; j < 18; ++j) u[j] = C12 && j >= 12 ? 0.0 : src[j];
  if (C12) reconstruct_row2(u);
  uint32_t emax = fx_max_hi<18>(u) & 0x7ff00000u;
  int e = (int)(emax >> 20);
  if (e < FX_LO || e > FX_HI) {
    e = fx_all_zero<18>(u) ? FX_LO : FX_BAD;
    emax = (uint32_t)FX_LO << 20;
  }
  int4* dst = reinterpret_cast<int4*>((p ? Uo : Ue) + ((size_t)i * 4 + mu) * FX_LINK_BYTES);
  int nonzero = 0, nonzero_t = 0;  // bit 3 a + b (b + 3 a of the adjoint): entry (a, b) is not 0
#pragma unroll
  for (int j = 0; j < 9; ++j) {
    int4 d = make_int4(0, 0, 0, 0);
    if (!fx_all_zero<2>(u + 2 * j)) {
      nonzero |= 1 << j;
      nonzero_t |= 1 << (j % 3 * 3 + j / 3);
    }
    if (e != FX_BAD) {
      const int rh = __double2hiint(u[2 * j]), ih = __double2hiint(u[2 * j + 1]);
      fx_magnitude<9>((uint32_t)rh, (uint32_t)__double2loint(u[2 * j]), emax, d.x, d.y);
      fx_magnitude<9>((uint32_t)ih, (uint32_t)__double2loint(u[2 * j + 1]), emax, d.z, d.w);
      if (rh < 0) d.x = -d.x, d.y = -d.y;
      if (ih < 0) d.z = -d.z, d.w = -d.w;
    }
    dst[j] = d;
  }
  dst[9] = make_int4(e, 0, nonzero, nonzero_t);
}

// The reals of a neighbour's spins psi_k (u) and psi_{p_k} (l) that thread k projects along mu, the second
// with real and imaginary parts exchanged where the projector multiplies it by i (x and z).
__device__ __forceinline__ void fx_load(const char* site, int mu, int k, size_t cs, double* u, double* l) {
  const char* ub = site + 6 * k * cs;
  const char* lb = site + (mu < 2 ? 18 - 6 * k : 12 + 6 * k) * cs;
  const size_t o0 = (mu & 1) == 0 ? cs : 0, o1 = cs - o0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    u[2 * c] = __ldg(reinterpret_cast<const double*>(ub + (2 * c) * cs));
    u[2 * c + 1] = __ldg(reinterpret_cast<const double*>(ub + (2 * c + 1) * cs));
    l[2 * c] = __ldg(reinterpret_cast<const double*>(lb + (2 * c) * cs + o0));
    l[2 * c + 1] = __ldg(reinterpret_cast<const double*>(lb + (2 * c) * cs + o1));
  }
}

// Signs of the projection of spin k: h_k = u + l with the real (bit 0) and imaginary (bit 1) part of l
// subtracted; plus: projector (1 + gamma_mu), otherwise (1 - gamma_mu). As a nibble {k=0 re, k=0 im, k=1 re,
// k=1 im} for (1 + gamma), complemented for (1 - gamma).
__device__ __forceinline__ uint32_t fx_signs(int mu, int k, bool plus) {
  return (((0x063Au >> (4 * mu)) & 15u) ^ (plus ? 0u : 15u)) >> (2 * k);
}

// Whether the lower spin's term, U h_k (y, t) or i U h_k (x, z), is subtracted: (1 + gamma) has x +,
// y k=0 - k=1 +, z k=0 + k=1 -, t +.
__device__ __forceinline__ bool fx_lower_minus(int mu, int k, bool plus) {
  return !plus ^ (mu == 1 ? k == 0 : mu == 2 ? k == 1 : false);
}

// The hopping sum of one (site, slice) in IEEE FP64, for inputs outside the integer range or precision: lane
// k's spin k, then its part of the lower spins from the x and y hops and from the z and t hops. The links
// are those that the integer blocks were made of (canonical layout).
template <bool C12>
__device__ __noinline__ void hop_ieee(const DhopArgs& a, int out_parity, const char* in, int site, int k, bool dag,
                                      double* out) {
  const int Lsh = ls_half(a.g.Ls);
  const size_t site_bytes = (size_t)Lsh * 2 * 24 * 8, cs = chunk_stride(Lsh);
  int c[4];
  cb_coords(a.g, site, out_parity, c);
  const long stride[4] = {1, a.g.L[0], (long)a.g.L[0] * a.g.L[1], (long)a.g.L[0] * a.g.L[1] * a.g.L[2]};
  const long lex = c[0] + c[1] * stride[1] + c[2] * stride[2] + c[3] * stride[3];
  double acc[18];
#pragma unroll
  for (int r = 0; r < 18; ++r) acc[r] = 0;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
#pragma unroll
    for (int back = 0; back < 2; ++back) {
      int ph;
      const int j = cb_neighbour(a.g, site, c, mu, back == 0, ph);
      const long before = c[mu] > 0 ? lex - stride[mu] : lex + (a.g.L[mu] - 1) * stride[mu];
      const double* link = a.Ucanon + ((back ? before : lex) * 4 + mu) * 18;
      double u[18], h[6], l[6];
#pragma unroll
      for (int r = 0; r < (C12 ? 12 : 18); ++r) u[r] = __ldg(link + r);
      if (C12) reconstruct_row2(u);
      fx_load(in + site_offset(j, Lsh, site_bytes), mu, k, cs, h, l);
      const bool plus = (back == 0) == dag;
      const uint32_t neg = fx_signs(mu, k, plus);
#pragma unroll
      for (int r = 0; r < 6; ++r) h[r] += (neg >> (r & 1)) & 1u ? -l[r] : l[r];
      const double cph = ph < 0 ? -a.alpha : a.alpha;
      const double clow = fx_lower_minus(mu, k, plus) ? -cph : cph;
      double* low = acc + (mu < 2 ? 6 : 12);
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        double re = 0, im = 0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          const int e = back ? b * 3 + r : r * 3 + b;
          const double ur = u[2 * e], ui = back ? -u[2 * e + 1] : u[2 * e + 1];
          re = fma(ur, h[2 * b], re);
          im = fma(ur, h[2 * b + 1], im);
          re = fma(-ui, h[2 * b + 1], re);
          im = fma(ui, h[2 * b], im);
        }
        acc[2 * r] = fma(cph, re, acc[2 * r]);
        acc[2 * r + 1] = fma(cph, im, acc[2 * r + 1]);
        low[2 * r] = (mu & 1) == 0 ? fma(-clow, im, low[2 * r]) : fma(clow, re, low[2 * r]);
        low[2 * r + 1] = (mu & 1) == 0 ? fma(clow, re, low[2 * r + 1]) : fma(clow, im, low[2 * r + 1]);
      }
    }
  }
  for (int r = 0; r < 18; ++r) out[r] = acc[r];
}

// Which colours of U h_k have a term that is not 0: bits 0 to 2 over the x and y hops, 3 to 5 over z and t.
__device__ __noinline__ int fx_terms(const char* in, const unsigned char* lsm, int k, int Lsh, size_t site_bytes) {
  int terms = 0;
#pragma unroll 1
  for (int hop = 0; hop < 8; ++hop) {
    const int* staged = reinterpret_cast<const int*>(lsm + hop * FX_HOP_BYTES + 9 * 16);
    const int nb = staged[1], entries = staged[2];
    double u[6], l[6];
    fx_load(in + site_offset(nb, Lsh, site_bytes), hop >> 1, k, chunk_stride(Lsh), u, l);
    int h = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (!fx_all_zero<2>(u + 2 * c) || !fx_all_zero<2>(l + 2 * c)) h |= 1 << c;
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if ((entries >> (3 * c)) & h) terms |= 1 << (hop < 4 ? c : c + 3);
  }
  return terms;
}

// v >> d for 0 <= d <= 31
__device__ __forceinline__ long long fx_asr(long long v, int d) {
  const uint32_t lo = __funnelshift_r((uint32_t)v, (uint32_t)(v >> 32), d);
  return ((long long)((int)(v >> 32) >> d) << 32) | lo;
}

// a + v with the sign of v flipped where m is -1 (m is 0 or -1)
__device__ __forceinline__ long long fx_add_signed(long long a, long long v, long long m) { return a + (v ^ m) + (m & 1); }

// 80 registers: six CTAs of 128 threads per SM. 16^4 x 16 Mpc^+ Mpc at 72 / 80 / 88 / 96 registers:
// 1049 / 1057 / 1068 / 1049 us; without the check of small components at 72 / 80 / 96 / 128 1001 / 1016 /
// 1032 / 1070 us, 24^4 x 12 4200 / 4146 / 4197 / 4330 us, and with the next hop's loads issued before this
// hop's products (24 more registers) 1080-1110 us.
template <int LSC>
__global__ void __maxnreg__(80) dhop_kernel_fx(const __grid_constant__ DhopArgs a, bool dag, bool c12) {
  constexpr int LSHC = LSC > 0 ? ls_half(LSC) : 0;
  const int Ls = LSC > 0 ? LSC : a.g.Ls;
  const int Lsh = LSC > 0 ? LSHC : ls_half(a.g.Ls);
  const int Lsp = 2 * Lsh;
  const int tid = threadIdx.x;
  const int site_local = tid / (2 * Lsp);
  const int ts = tid - site_local * (2 * Lsp);  // thread of the site
  const int s = ts >> 1, k = ts & 1;            // slice, spin of the half spinor
  // threads past the end of the lattice take its last site and store nothing (every lane of a
  // warp stays in the shuffles)
  const int site_raw = blockIdx.x * a.sites_per_cta + site_local;
  const bool active = site_raw < a.g.N4h;
  const int site = active ? site_raw : a.g.N4h - 1;
  const size_t site_bytes = (size_t)Lsp * 24 * 8;
  const size_t cs = chunk_stride(Lsh);
  const bool second = blockIdx.y != 0;  // the other half of a full-lattice hop
  const int out_parity = second ? 1 - a.out_parity : a.out_parity;
  const char* in_field = static_cast<const char*>(second ? a.in2 : a.in);

  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* lsm = smem_raw + (size_t)site_local * FX_SITE_BYTES;
  {
    int c[4];
    cb_coords(a.g, site, out_parity, c);
    const char* Uo = static_cast<const char*>(second ? a.Ufx_in : a.Ufx_out);
    const char* Ui = static_cast<const char*>(second ? a.Ufx_out : a.Ufx_in);
#pragma unroll
    for (int h = 0; h < 8; ++h) {
      // the site's threads share the ten 16-byte words of each hop's link
      const int mu = h >> 1;
      const bool fwd = (h & 1) == 0;
      int ph;
      const int nb = cb_neighbour(a.g, site, c, mu, fwd, ph);
      const int4* src = reinterpret_cast<const int4*>(fwd ? Uo + ((size_t)site * 4 + mu) * FX_LINK_BYTES
                                                          : Ui + ((size_t)nb * 4 + mu) * FX_LINK_BYTES);
      for (int e = ts; e < 10; e += 2 * Lsp) {
        int4 d = __ldg(src + e);
        int slot = e;
        if (e == 9) {
          d.y = nb;
          if (!fwd) d.z = d.w;
        } else {
          const int sr = ph, si = fwd ? ph : -ph;
          d.x *= sr;
          d.y *= sr;
          d.z *= si;
          d.w *= si;
          if (!fwd) slot = (e % 3) * 3 + e / 3;
        }
        *reinterpret_cast<int4*>(lsm + h * FX_HOP_BYTES + slot * 16) = d;
      }
    }
  }
  __syncthreads();

  double x[12];  // spin k, then spin 2 + k
  {
    // [upper spin k][lower spin of the x, y hops][lower spin of the z, t hops], re and im of 3 colours
    long long up[6], lxy[6], lzt[6];
#pragma unroll
    for (int r = 0; r < 6; ++r) up[r] = lxy[r] = lzt[r] = 0;
    int eacc = 0;
    bool bad = false;
    const char* in = in_field + (size_t)s * 8;
    // the lanes of this warp (the last warp of a CTA may be short)
    const uint32_t lanes = (int)blockDim.x - (tid & ~31) >= 32 ? 0xffffffffu : (1u << (blockDim.x & 31)) - 1u;
    // |re| + |im| of U h_k for each colour (2^32 accumulator units), summed over the x and y hops, then over z
    // and t; which of the former sums are large enough
    int terms[3] = {0, 0, 0}, large_xy = 0;
    auto large_terms = [&] {
      int m = 0;
#pragma unroll
      for (int c = 0; c < 3; ++c) m |= terms[c] >= FX_MIN_TERMS ? 1 << c : 0;
      return m;
    };
#pragma unroll 1
    for (int hop = 0; hop < 8; ++hop) {
      const int mu = hop >> 1;
      if (hop == 4) {
        large_xy = large_terms();
#pragma unroll
        for (int c = 0; c < 3; ++c) terms[c] = 0;
      }
      const bool plus = ((hop & 1) == 0) == dag;  // projector (1 + gamma_mu) or (1 - gamma_mu)
      const int lexp = *reinterpret_cast<const int*>(lsm + hop * FX_HOP_BYTES + 9 * 16);
      const int nb = *reinterpret_cast<const int*>(lsm + hop * FX_HOP_BYTES + 9 * 16 + 4);
      const uint32_t neg = fx_signs(mu, k, plus);
      double u[6], l[6];
      fx_load(in + site_offset(nb, Lsh, site_bytes), mu, k, cs, u, l);
      // one block exponent for the neighbour's 24 reals (the two lanes hold 12 each)
      uint32_t emax = max(fx_max_hi<6>(u), fx_max_hi<6>(l)) & 0x7ff00000u;
      emax = max(emax, __shfl_xor_sync(lanes, emax, 1));
      if (emax < ((uint32_t)FX_LO << 20)) {
        if (!fx_all_zero<6>(u) || !fx_all_zero<6>(l)) bad = true;
        emax = (uint32_t)FX_LO << 20;
      }
      if (emax > ((uint32_t)FX_HI << 20) || lexp < 0) {
        bad = true;
        emax = (uint32_t)FX_HI << 20;
      }
      // exponents: this hop's sums carry er, the accumulator eacc; sums are shifted right by
      // d = eacc - er >= 3 (|sum| < 2^62.6, eight of them after the shift < 2^63)
      const int er = (int)(emax >> 20) + max(lexp, FX_LO);
      if (hop == 0) eacc = er + 4;
      if (eacc - er < 3) {
        const int sh = min(er + 4 - eacc, 63);
        const long long half = 1ll << (sh - 1);
#pragma unroll
        for (int r = 0; r < 6; ++r) {
          up[r] = (up[r] + half) >> sh;
          lxy[r] = (lxy[r] + half) >> sh;
          lzt[r] = (lzt[r] + half) >> sh;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) terms[c] >>= min(sh, 31);
        large_xy = 0;
        eacc = er + 4;
      }
      int d = eacc - er;
      if (d > 31) {  // far below the accumulator: digits in a coarser block instead of a longer shift
        emax += (uint32_t)(d - 31) << 20;
        d = 31;
      }
      const long long round_h = 1ll << (d - 1);

      // digits of h = u +- l, and the negated imaginary parts
      int d1[6], d0[6];
      {
        const int fl[2] = {-(int)(neg & 1u), -(int)((neg >> 1) & 1u)};
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          const uint32_t uh = (uint32_t)__double2hiint(u[i]), lh = (uint32_t)__double2hiint(l[i]);
          int u1, u0, l1, l0;
          fx_magnitude<8>(uh, (uint32_t)__double2loint(u[i]), emax, u1, u0);
          fx_magnitude<8>(lh, (uint32_t)__double2loint(l[i]), emax, l1, l0);
          const int su = ((int)uh >> 31) | 1, sl = (((int)lh >> 31) ^ fl[i & 1]) | 1;
          d1[i] = l1 * sl + u1 * su;
          d0[i] = l0 * sl + u0 * su;
        }
      }
      const long long sm = fx_lower_minus(mu, k, plus) ? -1 : 0;
      const int4* us = reinterpret_cast<const int4*>(lsm + hop * FX_HOP_BYTES);
      long long v[6];
#pragma unroll
      for (int ra = 0; ra < 3; ++ra) {
        // leading sums (rounding constant of the final shift included) and cross sums of re and im
        long long hr = round_h, hi = round_h, cr = 1ll << 27, ci = 1ll << 27;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          const int4 u = us[ra * 3 + b];
          const int r1 = d1[2 * b], r0 = d0[2 * b], i1 = d1[2 * b + 1], i0 = d0[2 * b + 1];
          const int n1 = -i1, n0 = -i0;
          hr += (long long)u.x * r1;
          cr += (long long)u.x * r0;
          hi += (long long)u.x * i1;
          ci += (long long)u.x * i0;
          cr += (long long)u.y * r1;
          ci += (long long)u.y * i1;
          hr += (long long)u.z * n1;
          cr += (long long)u.z * n0;
          hi += (long long)u.z * r1;
          ci += (long long)u.z * r0;
          cr += (long long)u.w * n1;
          ci += (long long)u.w * r1;
        }
        const long long vr = fx_asr(hr + (cr >> 28), d), vi = fx_asr(hi + (ci >> 28), d);
        v[2 * ra] = vr;
        v[2 * ra + 1] = vi;
      }
#pragma unroll
      for (int r = 0; r < 6; ++r) up[r] += v[r];
#pragma unroll
      for (int c = 0; c < 3; ++c) terms[c] += abs((int)(v[2 * c] >> 32)) + abs((int)(v[2 * c + 1] >> 32));
      // lower spin += +-(v_r + i v_i) (y, t) or +-i (v_r + i v_i) (x, z)
#define FX_LOWER(acc, re, m_re, im, m_im)                        \
  for (int c = 0; c < 6; c += 2) {                               \
    acc[c] = fx_add_signed(acc[c], v[c + re], m_re);             \
    acc[c + 1] = fx_add_signed(acc[c + 1], v[c + im], m_im);     \
  }
      if (mu == 0) {
#pragma unroll
        FX_LOWER(lxy, 1, ~sm, 0, sm)
      } else if (mu == 1) {
#pragma unroll
        FX_LOWER(lxy, 0, sm, 1, sm)
      } else if (mu == 2) {
#pragma unroll
        FX_LOWER(lzt, 1, ~sm, 0, sm)
      } else {
#pragma unroll
        FX_LOWER(lzt, 0, sm, 1, sm)
      }
#undef FX_LOWER
    }
    // to FP64: acc 2^(eacc - 2103) alpha, alpha = +-2^alpha_log2 (no range to check: |exponent| < 900)
    const int ex = (eacc - 2103 + a.alpha_log2) << 20;
    const int flip = a.alpha < 0 ? (int)0x80000000 : 0;
    auto to_double = [&](long long v) {
      const double t = (double)v;
      return __hiloint2double(v != 0 ? (__double2hiint(t) + ex) ^ flip : 0, __double2loint(t));
    };
#pragma unroll
    for (int r = 0; r < 6; ++r) {
      x[r] = to_double(up[r]);
      x[6 + r] = to_double(lzt[r] + __shfl_xor_sync(lanes, lxy[r], 1));  // eacc is the same in both lanes
    }
    // components whose terms are too small for the accumulator's unit: spin k in bits 0 to 2, spin 2 + k
    // (which has the other lane's x and y hops) in bits 3 to 5; bit 6: outside the integer range
    const int large_zt = large_terms(), large_other = __shfl_xor_sync(lanes, large_xy, 1);
    int flags = s < Ls ? ((large_xy | large_zt) | (large_other | large_zt) << 3) ^ 63 : 0;
    if (bad) flags |= 64;
    const int flags_other = __shfl_xor_sync(lanes, flags, 1);  // by both lanes, whatever their own
    bool ieee = ((flags | flags_other) & 64) != 0;
    const uint32_t pair = 3u << (tid & 30);
    if (!ieee && (flags | flags_other) != 0) {  // both lanes of the pair come here
      const int own = fx_terms(in, lsm, k, Lsh, site_bytes), other = __shfl_xor_sync(pair, own, 1);
      const int need = flags & ((own | (own >> 3)) & 7 | ((own & 56) | (other & 7) << 3));
      ieee = (need | __shfl_xor_sync(pair, need, 1)) != 0;
    }
    if (ieee) {
      double t[18];
      if (c12)
        hop_ieee<true>(a, out_parity, in, site, k, dag, t);
      else
        hop_ieee<false>(a, out_parity, in, site, k, dag, t);
#pragma unroll
      for (int r = 0; r < 6; ++r) {
        x[r] = t[r];
        x[6 + r] = t[12 + r] + __shfl_xor_sync(pair, t[6 + r], 1);
      }
    }
  }

  // ------------------------------------------------------------ epilogue
  // real r of x is real base + r of the spinor for r < 6, base + 6 + r after
  const int base = 6 * k;
  const size_t own_off = (size_t)base * cs + (size_t)s * 8;
  const bool pad = s >= Ls;
  if (active && a.pre != PRE_NONE && !pad) {
    const char* auxb = static_cast<const char*>(second ? a.aux2 : a.aux) + site_offset(site, Lsh, site_bytes);
    const double own = a.pre == PRE_AUX ? a.beta : a.beta * a.d5;
    const char* ob = auxb + own_off;
    double o[12];
#pragma unroll
    for (int r = 0; r < 12; ++r) o[r] = __ldg(reinterpret_cast<const double*>(ob + (r < 6 ? r : r + 6) * cs));
#pragma unroll
    for (int r = 0; r < 12; ++r) x[r] = fma(own, o[r], x[r]);
    if (a.pre != PRE_AUX) {
      // the coupled halves of slices s -+ 1 (coefficient -1, or m on the wrap-around)
      const bool dag5 = a.pre == PRE_MOOEE_DAG;
      const int sm = s > 0 ? s - 1 : Ls - 1, sp = s < Ls - 1 ? s + 1 : 0;
      const double cm = s > 0 ? -a.beta : a.beta * a.mass, cp = s < Ls - 1 ? -a.beta : a.beta * a.mass;
      const char* ub = auxb + base * cs + (size_t)(dag5 ? sp : sm) * 8;
      const char* lb = auxb + (base + 12) * cs + (size_t)(dag5 ? sm : sp) * 8;
      const double c_up = dag5 ? cp : cm, c_lo = dag5 ? cm : cp;
#pragma unroll
      for (int r = 0; r < 6; ++r) {
        x[r] = fma(c_up, __ldg(reinterpret_cast<const double*>(ub + r * cs)), x[r]);
        x[6 + r] = fma(c_lo, __ldg(reinterpret_cast<const double*>(lb + r * cs)), x[6 + r]);
      }
    }
  }
  char* outb = static_cast<char*>(second ? a.out2 : a.out) + site_offset(site, Lsh, site_bytes) + own_off;
  if (a.post != POST_NONE) {
    double* sm = reinterpret_cast<double*>(smem_raw + (size_t)a.sites_per_cta * FX_SITE_BYTES);
    double* mine = sm + ((size_t)site_local * Ls + s) * INV_SLICE_STRIDE + base;
    if (active && !pad) {
#pragma unroll
      for (int r = 0; r < 12; ++r) mine[r < 6 ? r : r + 6] = x[r];
    }
    __syncthreads();
    const int first_site = blockIdx.x * a.sites_per_cta;
    const int nsites = min(a.sites_per_cta, a.g.N4h - first_site);
    for (int task = tid; task < nsites * 24; task += blockDim.x) {
      const int sl = task / 24;
      const int r = task - sl * 24;
      const bool upper = r < 12;
      const bool forward_form = (a.post == POST_INV) ? upper : !upper;
      mooee_inv_line64<LSC>(sm + (size_t)sl * Ls * INV_SLICE_STRIDE + r, Ls, forward_form, a.mass, a.inv_d5,
                            a.inv_den);
    }
    __syncthreads();
    if (active && !pad) {
#pragma unroll
      for (int r = 0; r < 12; ++r) x[r] = mine[r < 6 ? r : r + 6];
    }
  }
  if (active) {
#pragma unroll
    for (int r = 0; r < 12; ++r)
      *reinterpret_cast<double*>(outb + (r < 6 ? r : r + 6) * cs) = pad ? 0.0 : x[r];
  }
}

template <int LSC>
cudaError_t launch_fx(const DhopArgs& a, bool dag, bool c12, int threads, int blocks, size_t smem, cudaStream_t stream) {
  auto kern = dhop_kernel_fx<LSC>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  kern<<<dim3(blocks, a.in2 ? 2 : 1), threads, smem, stream>>>(a, dag, c12);
  return cudaGetLastError();
}

}  // namespace

size_t dhop_fx_smem_bytes(int sites_per_cta, int Ls, bool post) {
  return (size_t)sites_per_cta * (FX_SITE_BYTES + (post ? (size_t)Ls * INV_SLICE_STRIDE * 8 : 0));
}

template <>
cudaError_t launch_dhop<P64>(const DhopArgs& a, bool dag, bool c12, int threads, int blocks, size_t smem,
                             cudaStream_t stream) {
  // the even extents of the packed kernels (Ls / 2 pairs); any other Ls runs the generic kernel
  switch (a.g.Ls & 1 ? 0 : a.g.Ls / 2) {
#define DWF_CASE(N_) \
  case N_:           \
    return launch_fx<2 * N_>(a, dag, c12, threads, blocks, smem, stream);
    DWF_PAIR_SPECIALISATIONS(DWF_CASE)
#undef DWF_CASE
    default:
      return launch_fx<0>(a, dag, c12, threads, blocks, smem, stream);
  }
}

cudaError_t launch_pack_gauge_fx(bool c12, const Geom& g, const double* canon, void* Ue, void* Uo, cudaStream_t st) {
  const int blocks = (int)((8L * g.N4h + 127) / 128);
  if (c12)
    k_pack_gauge_fx<true><<<blocks, 128, 0, st>>>(g, canon, static_cast<char*>(Ue), static_cast<char*>(Uo));
  else
    k_pack_gauge_fx<false><<<blocks, 128, 0, st>>>(g, canon, static_cast<char*>(Ue), static_cast<char*>(Uo));
  return cudaGetLastError();
}

}  // namespace gdwf
