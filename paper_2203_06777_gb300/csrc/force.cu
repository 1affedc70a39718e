// Derivative of the action S = |M psi|^2 with respect to the gauge links (the fermion force).
// More generally the kernel differentiates the bilinear -Re chi^+ Dhop psi for any pair of full
// fields (psi, chi), times a coefficient coef (1 for |M psi|^2 with chi = M psi, whose
// variation is 2 Re chi^+ dM psi = -Re chi^+ dDhop psi; -1/2 for the pseudofermion action).
//
// With chi = M psi and M = Mooee - Dhop/2, only the hopping term depends on the links, so per
// link U_mu(x), with phase the boundary factor of the hop x -> x + mu,
//   B1 = sum_{s,spin} psi(x+mu) (x) [(1 - gamma_mu) chi(x)]^+,
//   B2 = sum_{s,spin} psi(x)    (x) [(1 + gamma_mu) chi(x+mu)]^+           (colour outer products),
//   G  = dS/dRe U + i dS/dIm U = -phase (B1^+ + B2)                           (ambient gradient),
//   F  = -TA( phase (-U B1 + B2 U^+) ),  TA(X) = (X - X^+)/2 - tr(X - X^+)/6  (su(3) force),
// so that under U -> exp(eps A) U, A in su(3), dS/deps = Re tr(A^+ F).
// Because (1 -+ gamma_mu)/2 is a rank-2 projector, each spin sum is the sum over the two spins
// of the projected half spinors: sum_spin a (x) [(1 - gamma) b]^+ = sum_{h=0,1} (P a)_h (x) (P b)_h^*.
//
// Thread mapping, as in the hopping kernels: one thread per (4D site, slice pair) for FP32 fields
// and two per (4D site, slice) for FP64, whole sites per CTA, one parity per grid row. For each mu the
// threads form their slices' contributions to B1 and B2 of the link U_mu(x) leaving their site
// (the own spinors and the two x + mu neighbours, the same loads as one Dhop hop), the CTA sums
// them over the site's slices through shared memory, and the link algebra is spread over the
// CTA's threads (one 3x3 entry each). FP32 fields: the products are summed in FP32 over up to 16 slice
// pairs (k_force_reg) or over blocks of 8 pairs whose sums are added in FP64 (k_force), and the link
// algebra (U B1, B2 U^+, the traceless anti-Hermitian projection) runs in FP32 on those sums: GB300's FP64 pipe is 1/64 of
// its FP32 pipe, and FP64 algebra made the kernel 5x slower for an answer whose error is set by
// the FP32 fields and block sums anyway. FP64 fields: k_force_fx below. F and G are written
// in the canonical FP64 layout [t][z][y][x][mu][3][3].
#include <algorithm>
#include <cstdint>

#include "dhop_kernel.cuh"
#include "ff_arith.cuh"
#include "fx_arith.cuh"

namespace gdwf {

// Threads per site: slice pairs (k_force) or padded slices (k_force_ff); sites per CTA fill 128 threads.
inline int force_threads_per_site(int prec, int Ls) {
  const int n = prec == P64 ? ls_padded(Ls) : ls_half(Ls);
  return n < 128 ? n : 128;
}

// Shared memory per site: partial sums of each slice thread (a stride of 37 values, odd, keeps
// the threads' writes in distinct banks), the site's summed B1 and B2 (36), its link (18), Y (18)
// and the output index and boundary phase.
constexpr int FORCE_PART_STRIDE = 37;
inline size_t force_smem_per_site(int prec, int nsg) {
  const size_t v = prec == P64 ? sizeof(double) : sizeof(float);
  return (size_t)nsg * FORCE_PART_STRIDE * v + (36 + 18 + 18) * v + 2 * sizeof(long);
}

// The per-site steps after the slice sums B1, B2 (bsum) of direction mu are in shared memory:
// each site's link, then one (site, a, b) entry per task:
//   G[a][b] = -phase (conj(B1[b][a]) + B2[a][b]),  Y = phase (-U B1 + B2 U^+),
// then F = -TA(Y), TA(Y)[a][b] = (Y[a][b] - conj(Y[b][a]))/2 - delta_ab tr(Y - Y^+)/6.
// A: the arithmetic of the link algebra (double for FP64 fields, float for FP32 fields).
template <int P, bool C12, typename A>
__device__ __forceinline__ void force_site_algebra(int mu, int p, int first, int nsites, const char* Ue, const char* Uo,
                                                   const A* bsum, A* usm, A* ysm, const long* lex_sm,
                                                   const int* ph_sm, double coef, double* F, double* G) {
  using R = typename Store<P>::R;
  constexpr int LB = link_bytes(sizeof(typename Store<P>::T), C12);
  const int tid = threadIdx.x;
  for (int sl = tid; sl < nsites; sl += blockDim.x) {  // the link U_mu(x), third row rebuilt if stored as 12 reals
    R ur[18];
    load_link<P, C12>((p ? Uo : Ue) + ((size_t)(first + sl) * 4 + mu) * LB, ur);
#pragma unroll
    for (int k = 0; k < 18; ++k) usm[(size_t)sl * 18 + k] = (A)ur[k];
  }
  __syncthreads();
  // ---- link algebra, one (site, a, b) entry per task:
  //   G[a][b] = -phase (conj(B1[b][a]) + B2[a][b]),  Y = phase (-U B1 + B2 U^+)
  for (int task = tid; task < nsites * 9; task += blockDim.x) {
    const int sl = task / 9, ab = task - sl * 9, a = ab / 3, b = ab - a * 3;
    const A phd = (A)(coef * (double)ph_sm[sl]);  // F and G are linear in the boundary phase and coef
    const A* B1 = bsum + (size_t)sl * 36;
    const A* B2 = B1 + 18;
    const A* ur = usm + (size_t)sl * 18;
    A yr = 0, yi = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const A ar = ur[(a * 3 + k) * 2], ai = ur[(a * 3 + k) * 2 + 1];
      const A br = B1[(k * 3 + b) * 2], bi = B1[(k * 3 + b) * 2 + 1];
      yr -= ar * br - ai * bi;
      yi -= ar * bi + ai * br;
      const A cr = B2[(a * 3 + k) * 2], ci = B2[(a * 3 + k) * 2 + 1];
      const A dr = ur[(b * 3 + k) * 2], di = -ur[(b * 3 + k) * 2 + 1];  // (U^+)[k][b] = conj(U[b][k])
      yr += cr * dr - ci * di;
      yi += cr * di + ci * dr;
    }
    ysm[(size_t)sl * 18 + ab * 2] = phd * yr;
    ysm[(size_t)sl * 18 + ab * 2 + 1] = phd * yi;
    if (G) {
      double* Go = G + (lex_sm[sl] * 4 + mu) * 18;
      Go[ab * 2] = (double)(-phd * (B1[(b * 3 + a) * 2] + B2[ab * 2]));
      Go[ab * 2 + 1] = (double)(-phd * (-B1[(b * 3 + a) * 2 + 1] + B2[ab * 2 + 1]));
    }
  }
  __syncthreads();
  // ---- F = -TA(Y): TA(Y)[a][b] = (Y[a][b] - conj(Y[b][a]))/2 - delta_ab tr(Y - Y^+)/6
  if (F) {
    for (int task = tid; task < nsites * 9; task += blockDim.x) {
      const int sl = task / 9, ab = task - sl * 9, a = ab / 3, b = ab - a * 3;
      const A* Y = ysm + (size_t)sl * 18;
      const A trim = Y[1] + Y[9] + Y[17];  // Im tr Y; tr(Y - Y^+) = 2 i Im tr Y
      const A tr_ = (A)0.5 * (Y[(a * 3 + b) * 2] - Y[(b * 3 + a) * 2]);
      A ti_ = (A)0.5 * (Y[(a * 3 + b) * 2 + 1] + Y[(b * 3 + a) * 2 + 1]);
      if (a == b) ti_ -= trim / (A)3;
      double* Fo = F + (lex_sm[sl] * 4 + mu) * 18;
      Fo[ab * 2] = -(double)tr_;
      Fo[ab * 2 + 1] = -(double)ti_;
    }
  }
}

template <bool C12>
__global__ void __launch_bounds__(128) k_force(const Geom g, const char* psi, const char* chi, const char* Ue,
                                               const char* Uo, double* F, double* G, double coef, int nsg, int spc) {
  constexpr int P = P32;
  using A = float;  // partial sums and link algebra
  constexpr int FLUSH = 8;  // slice pairs summed in FP32 before an FP64 sum across blocks
  const int Lsh = ls_half(g.Ls);
  const size_t site_bytes = (size_t)Lsh * 2 * 24 * sizeof(float);
  const size_t half_bytes = (size_t)g.N4h * site_bytes;
  // both parities of a block of sites run next to each other, so their shared neighbours are
  // still in L2 when the other parity reads them
  const int p = blockIdx.x & 1;
  const int first = (blockIdx.x >> 1) * spc;
  const int tid = threadIdx.x;
  const int site_local = tid / nsg;
  const int t = tid - site_local * nsg;  // slice pair
  const int nsites = min(spc, g.N4h - first);
  const bool active = site_local < nsites;
  const int i = first + (active ? site_local : 0);
  int c[4];
  cb_coords(g, i, p, c);
  const char* psi_x = psi + p * half_bytes + site_offset(i, Lsh, site_bytes);
  const char* chi_x = chi + p * half_bytes + site_offset(i, Lsh, site_bytes);

  extern __shared__ __align__(16) unsigned char smem_raw[];
  long* lex_sm = reinterpret_cast<long*>(smem_raw);                          // [spc]
  int* ph_sm = reinterpret_cast<int*>(lex_sm + spc);                         // [spc] (pairs of ints: 8 bytes)
  A* part = reinterpret_cast<A*>(smem_raw + (size_t)spc * 2 * sizeof(long));  // [spc][nsg][37]
  A* bsum = part + (size_t)spc * nsg * FORCE_PART_STRIDE;                      // [spc][36]
  A* usm = bsum + (size_t)spc * 36;                                            // [spc][18]
  A* ysm = usm + (size_t)spc * 18;                                             // [spc][18]
  if (active && t == 0) lex_sm[site_local] = c[0] + (long)g.L[0] * (c[1] + (long)g.L[1] * (c[2] + (long)g.L[2] * c[3]));

#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {  // unrolled: direction-dependent indices stay compile-time
    // ---- this thread's slices: B1 += psi(x+mu) (x) [(1 - gamma) chi(x)]^+, B2 += psi(x) (x) [(1 + gamma) chi(x+mu)]^+
    if (active) {
      int ph;
      const int j = cb_neighbour(g, i, c, mu, true, ph);
      if (t == 0) ph_sm[site_local] = ph;
      const char* psi_f = psi + (1 - p) * half_bytes + site_offset(j, Lsh, site_bytes);
      const char* chi_f = chi + (1 - p) * half_bytes + site_offset(j, Lsh, site_bytes);
      A* dst = part + ((size_t)site_local * nsg + t) * FORCE_PART_STRIDE;
#pragma unroll
      for (int term = 0; term < 2; ++term) {
        float2 v[24], ha[12], hb[12];
        load_pair<P, 0>(term == 0 ? psi_f : psi_x, t, Lsh, v);
        if (term == 0) project2<-1>(mu, v, ha); else project2<+1>(mu, v, ha);
        load_pair<P, 0>(term == 0 ? chi_x : chi_f, t, Lsh, v);
        if (term == 0) project2<-1>(mu, v, hb); else project2<+1>(mu, v, hb);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b = 0; b < 3; ++b) {  // both slices of the pair, then their sum
            float2 re = make_float2(0.f, 0.f), im = make_float2(0.f, 0.f);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const float2 xr = ha[(h * 3 + a) * 2], xi = ha[(h * 3 + a) * 2 + 1];
              const float2 yr = hb[(h * 3 + b) * 2], yi = hb[(h * 3 + b) * 2 + 1];
              re = ffma2(xr, yr, ffma2(xi, yi, re));
              im = ffma2(xi, yr, ffma2(make_float2(-xr.x, -xr.y), yi, im));
            }
            dst[term * 18 + (a * 3 + b) * 2] = re.x + re.y;
            dst[term * 18 + (a * 3 + b) * 2 + 1] = im.x + im.y;
          }
      }
    }
    __syncthreads();
    // ---- sum over the site's slices, one (site, entry) per task; and each site's link
    for (int task = tid; task < nsites * 36; task += blockDim.x) {
      const int sl = task / 36, e = task - sl * 36;
      const A* src = part + (size_t)sl * nsg * FORCE_PART_STRIDE + e;
      A total;
      if (nsg <= FLUSH) {  // one block: FP32 throughout
        total = 0.f;
        for (int k = 0; k < nsg; ++k) total += src[(size_t)k * FORCE_PART_STRIDE];
      } else {  // blocks of FLUSH pairs summed in FP64
        double acc = 0;
        for (int k0 = 0; k0 < nsg; k0 += FLUSH) {
          float blk = 0.f;
          const int k1 = min(k0 + FLUSH, nsg);
          for (int k = k0; k < k1; ++k) blk += src[(size_t)k * FORCE_PART_STRIDE];
          acc += (double)blk;
        }
        total = (A)acc;
      }
      bsum[(size_t)sl * 36 + e] = total;
    }
    force_site_algebra<P, C12, A>(mu, p, first, nsites, Ue, Uo, bsum, usm, ysm, lex_sm, ph_sm, coef, F, G);
    __syncthreads();  // shared memory is reused by the next direction
  }
}

// FP32 fields with 3 to 16 slice pairs per site: a site's threads are LG consecutive lanes of one warp
// (4, 8 or 16; FULL: one per pair, otherwise the lanes past the last pair add zeros), so the sums over
// its slices run in registers and every synchronisation is within a warp. Lanes left idle cost less than
// k_force's sums through shared memory: force call at 16^4 with Ls = 10 / 12 / 24, k_force and this:
// 265 / 244 / 395 and 211 / 215 / 351 us. (With 2 lanes, the 32 sites of a CTA would pass 48 KB of static shared memory.)
//   - Each field is read once as the own site's spinor: the B1 products of all four directions
//     first (own chi(x) held in registers, psi(x + mu) loaded per direction), then the B2 products
//     (own psi(x) held, chi(x + mu) loaded): 10 spinor loads per (site, pair) instead of 16.
//   - The 9 complex products of one (direction, term) are summed over the site's lanes by a
//     butterfly reduce-scatter (xor shuffles; at each level a lane keeps one half of its values
//     and adds its partner's copy of that half), after which lane q holds entries
//     q * NPAD / LSH .. of the site's sum; those go to shared memory.
//   - The link algebra of the site's four links (36 entries) is spread over the same lanes.
// Rounding: the products of a slice pair and the sums over at most 16 pairs are FP32, pairwise. The general
// kernel adds 8 pairs one after the other in FP32, and two such blocks in FP64 before one rounding, which
// is the FP32 sum of the two; so this order rounds less often. 2-norm errors with 9 to 15 pairs, in 1e-7:
// F 1.29-1.35 here and 1.36-1.40 there, G 0.64-0.71 and 0.68-0.76.
template <int LG, int THREADS>
struct ForceRegGeom {
  static constexpr int SPC = THREADS / LG;               // sites per CTA
  static constexpr int PER_LANE = (18 + LG - 1) / LG;    // sum entries per lane after reduce-scatter
  static constexpr int NPAD = PER_LANE * LG;             // 18 reals padded to a multiple of LG
  // B1 B2 per mu, U per mu, Y per mu, padded so that the sites of a warp fall on different banks:
  // 299 floats give the fewest conflicts of the strides 289-329 over the partial-sum stores and the
  // link algebra's reads of 8-lane sites (53 extra wavefronts per warp against 116 at 289, by
  // simulation; 16-lane sites are indifferent)
  static constexpr int SITE_FLOATS = 4 * 36 + 4 * 18 + 4 * 18 + 11;
};

template <int N, int LSH>
__device__ __forceinline__ void reduce_scatter(float (&v)[N], int lane_in_site) {
  // levels with partner offsets LSH/2, ..., 1: keep the half selected by the offset's bit
#pragma unroll
  for (int off = LSH / 2, len = N / 2; off >= 1; off >>= 1, len >>= 1) {
    const bool upper = (lane_in_site & off) != 0;
#pragma unroll
    for (int k = 0; k < len; ++k) {
      const float send = upper ? v[k] : v[len + k];
      const float keep = upper ? v[len + k] : v[k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
}

// The own spinor of a term goes through shared memory and is read back per direction (128
// registers, 4 CTAs per SM): holding it in 48 registers instead needed 168 registers, 3 CTAs per
// SM and some spills, and measured 136 us against 111 us at 16^4 x 16.
template <bool C12, int LG, bool FULL, int THREADS>
__global__ void __launch_bounds__(THREADS, 512 / THREADS) k_force_reg(const Geom g, const char* psi, const char* chi,
                                                                      const char* Ue, const char* Uo, double* F,
                                                                      double* G, double coef) {
  using GG = ForceRegGeom<LG, THREADS>;
  constexpr int LB = link_bytes(4, C12);
  constexpr int SPC = GG::SPC, NPAD = GG::NPAD, PER_LANE = GG::PER_LANE;
  constexpr int LSH = FULL ? LG : 0;
  const int Lsh = FULL ? LG : ls_half(g.Ls);
  const size_t site_bytes = (size_t)Lsh * 2 * 24 * 4;
  const size_t half_bytes = (size_t)g.N4h * site_bytes;
  const int p = blockIdx.x & 1;
  const int first = (blockIdx.x >> 1) * SPC;
  const int tid = threadIdx.x;
  const int site_local = tid / LG;
  const int q = tid - site_local * LG;  // slice pair, and the lane's place in its site's group
  const bool has_pair = FULL || q < Lsh;
  const bool active = first + site_local < g.N4h;
  const int i = active ? first + site_local : first;  // inactive lanes compute a valid site, store nothing
  int c[4];
  cb_coords(g, i, p, c);
  int nbr[4], phs[4];
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) nbr[mu] = cb_neighbour(g, i, c, mu, true, phs[mu]);

  __shared__ float ssm[SPC][GG::SITE_FLOATS];
  // the own site's spinor of the current term, one 16-byte vector per (chunk, thread): read back
  // for each direction's projection instead of being held in 48 registers
  __shared__ float4 own_sm[12][THREADS];
  float* bs = ssm[site_local];          // [mu][term][18]
  float* us = bs + 4 * 36;              // [mu][18]
  float* ys = us + 4 * 18;              // [mu][18]

  // the site's four links U_mu(x), one per lane (and the third row rebuilt for 12-real links)
  for (int mu = q; mu < 4; mu += LG) {
    float ur[18];
    load_link<P32, C12>((p ? Uo : Ue) + ((size_t)i * 4 + mu) * LB, ur);
#pragma unroll
    for (int k = 0; k < 18; ++k) us[mu * 18 + k] = ur[k];
  }

#pragma unroll
  for (int term = 0; term < 2; ++term) {
    // term 0: B1 = sum psi(x+mu) (x) [(1 - gamma) chi(x)]^+  (own chi, projector sign -1)
    // term 1: B2 = sum psi(x) (x) [(1 + gamma) chi(x+mu)]^+  (own psi, projector sign +1)
    if (has_pair) {
      const char* ob = (term == 0 ? chi : psi) + p * half_bytes + site_offset(i, Lsh, site_bytes) + (size_t)q * 16;
#pragma unroll
      for (int k = 0; k < 12; ++k) own_sm[k][tid] = __ldg(reinterpret_cast<const float4*>(ob + k * chunk_stride(Lsh)));
    }
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      float s[NPAD];
#pragma unroll
      for (int k = 0; k < NPAD; ++k) s[k] = 0.f;
      if (has_pair) {
        float2 v[24], ha[12], hb[12];
        load_pair<P32, LSH>((term == 0 ? psi : chi) + (1 - p) * half_bytes + site_offset(nbr[mu], Lsh, site_bytes), q,
                            Lsh, v);
        {
          float2 own[24];
#pragma unroll
          for (int k = 0; k < 12; ++k) {
            const float4 t = own_sm[k][tid];
            own[2 * k] = make_float2(t.x, t.y);
            own[2 * k + 1] = make_float2(t.z, t.w);
          }
          if (term == 0)
            project2<-1>(mu, own, hb);
          else
            project2<+1>(mu, own, ha);
        }
        if (term == 0)
          project2<-1>(mu, v, ha);
        else
          project2<+1>(mu, v, hb);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b = 0; b < 3; ++b) {  // sum_h ha[h][a] conj(hb[h][b]), both slices of the pair
            float2 re = make_float2(0.f, 0.f), im = make_float2(0.f, 0.f);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const float2 xr = ha[(h * 3 + a) * 2], xi = ha[(h * 3 + a) * 2 + 1];
              const float2 yr = hb[(h * 3 + b) * 2], yi = hb[(h * 3 + b) * 2 + 1];
              re = ffma2(xr, yr, ffma2(xi, yi, re));
              im = ffma2(xi, yr, ffma2(make_float2(-xr.x, -xr.y), yi, im));
            }
            s[(a * 3 + b) * 2] = re.x + re.y;
            s[(a * 3 + b) * 2 + 1] = im.x + im.y;
          }
      }
      reduce_scatter<NPAD, LG>(s, q);
#pragma unroll
      for (int k = 0; k < PER_LANE; ++k) {
        const int e = q * PER_LANE + k;
        if (e < 18) bs[mu * 36 + term * 18 + e] = s[k];
      }
    }
  }
  __syncwarp();
  // link algebra, one (mu, a, b) entry per task over the site's lanes:
  //   G[a][b] = -phase (conj(B1[b][a]) + B2[a][b]),  Y = phase (-U B1 + B2 U^+)
  const long lex = c[0] + (long)g.L[0] * (c[1] + (long)g.L[1] * (c[2] + (long)g.L[2] * c[3]));
  for (int task = q; task < 36; task += LG) {
    const int mu = task / 9, ab = task - mu * 9, a = ab / 3, b = ab - a * 3;
    const int ph = mu == 0 ? phs[0] : mu == 1 ? phs[1] : mu == 2 ? phs[2] : phs[3];
    const float phd = (float)(coef * (double)ph);
    const float* B1 = bs + mu * 36;
    const float* B2 = B1 + 18;
    const float* ur = us + mu * 18;
    float yr = 0.f, yi = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float ar = ur[(a * 3 + k) * 2], ai = ur[(a * 3 + k) * 2 + 1];
      const float br = B1[(k * 3 + b) * 2], bi = B1[(k * 3 + b) * 2 + 1];
      yr -= ar * br - ai * bi;
      yi -= ar * bi + ai * br;
      const float cr = B2[(a * 3 + k) * 2], ci = B2[(a * 3 + k) * 2 + 1];
      const float dr = ur[(b * 3 + k) * 2], di = -ur[(b * 3 + k) * 2 + 1];  // (U^+)[k][b] = conj(U[b][k])
      yr += cr * dr - ci * di;
      yi += cr * di + ci * dr;
    }
    ys[mu * 18 + ab * 2] = phd * yr;
    ys[mu * 18 + ab * 2 + 1] = phd * yi;
    if (G && active) {
      const double gr = (double)(-phd * (B1[(b * 3 + a) * 2] + B2[ab * 2]));
      const double gi = (double)(-phd * (-B1[(b * 3 + a) * 2 + 1] + B2[ab * 2 + 1]));
      *reinterpret_cast<double2*>(G + (lex * 4 + mu) * 18 + ab * 2) = make_double2(gr, gi);
    }
  }
  __syncwarp();
  // F = -TA(Y): TA(Y)[a][b] = (Y[a][b] - conj(Y[b][a]))/2 - delta_ab tr(Y - Y^+)/6
  if (F && active) {
    for (int task = q; task < 36; task += LG) {
      const int mu = task / 9, ab = task - mu * 9, a = ab / 3, b = ab - a * 3;
      const float* Y = ys + mu * 18;
      const float trim = Y[1] + Y[9] + Y[17];  // Im tr Y; tr(Y - Y^+) = 2 i Im tr Y
      const float tr_ = 0.5f * (Y[(a * 3 + b) * 2] - Y[(b * 3 + a) * 2]);
      float ti_ = 0.5f * (Y[(a * 3 + b) * 2 + 1] + Y[(b * 3 + a) * 2 + 1]);
      if (a == b) ti_ -= trim / 3.f;
      *reinterpret_cast<double2*>(F + (lex * 4 + mu) * 18 + ab * 2) = make_double2(-(double)tr_, -(double)ti_);
    }
  }
}

// FP64 fields in block integers (fx_arith.cuh): with IEEE instructions the 192 FP64 operations per
// (site, slice, direction) ran at 2 per SM and clock (16^4 x 12 force call 2.14 ms, 1.7 ms of it here).
// Two threads (neighbouring lanes) per (site, slice), one per term: with own = chi(x) and nb = psi(x + mu)
// for B1, own = psi(x) and nb = chi(x + mu) for B2, either forms C = sum_h (P nb)_h (x) (P own)_h^*
// (B1 = C, B2 = C^+), the digits of the own spinor waiting in shared memory. The 9 complex sums are
// exact 64-bit integers per slice (4 products each, < 2^62), aligned by a rounded shift to the
// largest slice's exponent while they are added over the site's slices, and rounded to FP64 once. The
// link algebra of all four directions follows at the end, in FP64, 36 entries per site (direction by
// direction, with 36 of 128 threads at work between barriers: force call at 16^4 x 16 1612 us; with
// FP64 products 2520 us; now 1311 us, of which M psi is 480 us). Integer instructions and the barriers
// around the slice sums bound it now.
// IEEE instructions instead: for a block of sites with a magnitude outside the integer range, all its
// slices (force_products_ieee); and for an entry of B1 or B2 whose slices' |re| + |im| sum to less than an
// eighth of the smallest product of two blocks' largest reals (force_entry_ieee), since the integers'
// errors, relative to that product, could be large beside it (colours or spins of very different size).
// Above that limit a real's error is at most (81 + Ls / 2) 2^(n - 53) of that sum, n = ceil(log2 Ls).
// Gaussian fields with Ls = 1 / 2: 0.5% / 8e-6 of the entries lie below it, with 3 and more none of 1e5
// simulated ones. Force call at 16^4, without and with the check: Ls = 16 1287 and 1311 us, Ls = 2 430 and
// 442 us, Ls = 1 435 and 510 us.
constexpr int FORCE_FX_STRIDE = 19;  // 64-bit values per (slice, term): 18, odd so that stores spread over the banks
constexpr int FORCE_FX_OWN = 25;     // digit pairs per thread of the own spinor: 24, odd for the same reason
constexpr int FORCE_FX_MIN_TERMS = 1 << 21;  // 2^53 of 2^56 units, an eighth of the smallest product
// Threads and sites per CTA at most (Ls > 32: one site). 256 threads, two CTAs per SM instead of four,
// wait longer at the barriers: 1382 us.
constexpr int FORCE_FX_THREADS = 128, FORCE_FX_SITES = 16;

__device__ __noinline__ void force_products_ieee(const char* psi_x, const char* chi_x, const char* psi_f,
                                                 const char* chi_f, int mu, int s, int Lsh, double* B) {
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    if (m != mu) continue;
#pragma unroll
    for (int term = 0; term < 2; ++term) {
      double v[24], ha[12], hb[12];
      load_lane64<0>(term == 0 ? psi_f : psi_x, s, Lsh, v);
      if (term == 0) project<-1>(m, v, ha); else project<+1>(m, v, ha);
      load_lane64<0>(term == 0 ? chi_x : chi_f, s, Lsh, v);
      if (term == 0) project<-1>(m, v, hb); else project<+1>(m, v, hb);
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {  // sum_h ha[h][a] conj(hb[h][b])
          double re = 0, im = 0;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const double xr = ha[(h * 3 + a) * 2], xi = ha[(h * 3 + a) * 2 + 1];
            const double yr = hb[(h * 3 + b) * 2], yi = hb[(h * 3 + b) * 2 + 1];
            re = fma(xr, yr, fma(xi, yi, re));
            im = fma(xi, yr, fma(-xr, yi, im));
          }
          B[term * 18 + (a * 3 + b) * 2] = re;
          B[term * 18 + (a * 3 + b) * 2 + 1] = im;
        }
    }
  }
}

// One real of a site's slice sums in IEEE FP64 (im: the imaginary part of entry (a, b) of B1, or with
// term = 1 of B2), for a sum that the block integers would give fewer bits than its own products have.
__device__ __noinline__ double force_entry_ieee(const Geom& g, const char* psi, const char* chi, int p, int i, int mu,
                                                int term, int a, int b, int im) {
  const int Lsh = ls_half(g.Ls);
  const size_t site_bytes = (size_t)Lsh * 2 * 24 * 8, cs = chunk_stride(Lsh);
  const size_t half_bytes = (size_t)g.N4h * site_bytes;
  int c[4], ph;
  cb_coords(g, i, p, c);
  const size_t own = p * half_bytes + site_offset(i, Lsh, site_bytes);
  const size_t nb = (1 - p) * half_bytes + site_offset(cb_neighbour(g, i, c, mu, true, ph), Lsh, site_bytes);
  const char* x = psi + (term ? own : nb);
  const char* y = chi + (term ? nb : own);
  const uint32_t neg = ((0x063Au >> (4 * mu)) & 15u) ^ (term ? 0u : 15u);  // as in k_force_fx
  const int swap = (mu & 1) == 0;
  // part r (0 re, 1 im) of the projected spin h, colour col
  auto half_spin = [&](const char* f, int h, int col, int r) {
    const int upper = 6 * h + 2 * col + r, lower = (mu < 2 ? 18 - 6 * h : 12 + 6 * h) + 2 * col + (swap ? 1 - r : r);
    const double u = __ldg(reinterpret_cast<const double*>(f + upper * cs));
    const double l = __ldg(reinterpret_cast<const double*>(f + lower * cs));
    return (neg >> (2 * h + r)) & 1u ? u - l : u + l;
  };
  double sum = 0;
  for (int s = 0; s < g.Ls; ++s, x += 8, y += 8) {
    double v = 0;
    for (int h = 0; h < 2; ++h) {
      const double xr = half_spin(x, h, a, 0), xi = half_spin(x, h, a, 1);
      const double yr = half_spin(y, h, b, 0), yi = half_spin(y, h, b, 1);
      v = im ? fma(xi, yr, fma(-xr, yi, v)) : fma(xr, yr, fma(xi, yi, v));
    }
    sum += v;
  }
  return sum;
}

inline size_t force_fx_smem(int nsg, int spc) {
  return (size_t)spc * 4 * 36 * 8 + (size_t)spc * nsg * (FORCE_FX_OWN * 8 + FORCE_FX_STRIDE * 8) + (size_t)spc * 8;
}

template <bool C12>
__global__ void __maxnreg__(128) k_force_fx(const Geom g, const char* psi, const char* chi, const char* Ue,
                                            const char* Uo, double* F, double* G, double coef, int nsg, int spc,
                                            int sum_shift) {
  const int Lsh = ls_half(g.Ls), Lsp = 2 * Lsh;
  const size_t site_bytes = (size_t)Lsp * 24 * 8;
  const size_t half_bytes = (size_t)g.N4h * site_bytes;
  const size_t cs = chunk_stride(Lsh);
  const int p = blockIdx.x & 1;
  const int first = (blockIdx.x >> 1) * spc;
  const int tid = threadIdx.x;
  const int site_local = tid / nsg;
  const int ts = tid - site_local * nsg;
  const int s = ts >> 1, t = ts & 1;  // slice, term
  const int nsites = min(spc, g.N4h - first);
  const int i = first + min(site_local, nsites - 1);  // threads past the end repeat the last site
  int c[4];
  cb_coords(g, i, p, c);

  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* bsum = reinterpret_cast<double*>(smem_raw);                               // [spc][mu][36]
  int2* own_sm = reinterpret_cast<int2*>(bsum + (size_t)spc * 4 * 36);              // [thread][real]
  long long* part = reinterpret_cast<long long*>(own_sm + (size_t)FORCE_FX_OWN * nsg * spc);  // [spc][slice][term][19]
  int* e_sm = reinterpret_cast<int*>(part + (size_t)spc * nsg * FORCE_FX_STRIDE);   // [spc][term]
  if (ts < 2) e_sm[2 * site_local + ts] = 0;
  int nf[4], pf[4];  // forward neighbours (the phases enter with the link algebra)
#pragma unroll
  for (int m = 0; m < 4; ++m) nf[m] = cb_neighbour(g, i, c, m, true, pf[m]);

  const size_t xo = p * half_bytes + site_offset(i, Lsh, site_bytes);
  const char* own_field = t == 0 ? chi : psi;
  const char* nb_field = t == 0 ? psi : chi;
  bool bad = false;
  // exponent field of a block's largest real, at least FX_LO; flags what does not fit
  auto block_exponent = [&](const double* v) {
    uint32_t emax = fx_max_hi<24>(v) & 0x7ff00000u;
    if (emax < ((uint32_t)FX_LO << 20)) {
      if (!fx_all_zero<24>(v)) bad = true;
      emax = (uint32_t)FX_LO << 20;
    }
    if (emax > ((uint32_t)FX_HI << 20)) {
      bad = true;
      emax = (uint32_t)FX_HI << 20;
    }
    return emax;
  };
  int2* own = own_sm + tid * FORCE_FX_OWN;
  int e_own;
  {
    double v[24];
    load_lane64<0>(own_field + xo, s, Lsh, v);
    const uint32_t emax = block_exponent(v);
    e_own = (int)(emax >> 20);
#pragma unroll
    for (int r = 0; r < 24; ++r) {
      int y1, y0;
      const int hi = __double2hiint(v[r]), sg = (hi >> 31) | 1;
      fx_magnitude<8>((uint32_t)hi, (uint32_t)__double2loint(v[r]), emax, y1, y0);
      own[r] = make_int2(y1 * sg, y0 * sg);
    }
  }
  __syncthreads();

#pragma unroll 1
  for (int mu = 0; mu < 4; ++mu) {
    const int j = mu == 0 ? nf[0] : mu == 1 ? nf[1] : mu == 2 ? nf[2] : nf[3];
    const size_t jo = (1 - p) * half_bytes + site_offset(j, Lsh, site_bytes);
    // h_k = psi_k +- (1 or i) psi_{p_k}, p = (3, 2) for x and y, (2, 3) for z and t: signs as a nibble
    // {k=0 re, k=0 im, k=1 re, k=1 im} (bit set: subtract) for (1 + gamma), complemented for (1 - gamma)
    const bool im_form = (mu & 1) == 0;  // i psi: real and imaginary parts trade places
    const uint32_t neg = ((0x063Au >> (4 * mu)) & 15u) ^ (t ? 0u : 15u);
    int n1[12], n0[12];  // digits of the projected neighbour spinor
    int e_sum;
    {
      double v[24];  // the upper spins, then their partners (second spin of k, parts exchanged if im_form)
      const char* nb = nb_field + jo + (size_t)s * 8;
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) {
          const char* lo = nb + (mu < 2 ? 18 - 6 * k : 12 + 6 * k) * cs + 2 * cc * cs;
          v[6 * k + 2 * cc] = __ldg(reinterpret_cast<const double*>(nb + (6 * k + 2 * cc) * cs));
          v[6 * k + 2 * cc + 1] = __ldg(reinterpret_cast<const double*>(nb + (6 * k + 2 * cc + 1) * cs));
          v[12 + 6 * k + 2 * cc] = __ldg(reinterpret_cast<const double*>(lo + (im_form ? cs : 0)));
          v[12 + 6 * k + 2 * cc + 1] = __ldg(reinterpret_cast<const double*>(lo + (im_form ? 0 : cs)));
        }
      const uint32_t emax = block_exponent(v);
      e_sum = (int)(emax >> 20) + e_own;
#pragma unroll
      for (int r = 0; r < 12; ++r) {
        const int fl = -(int)((neg >> (2 * (r / 6) + (r & 1))) & 1u);
        const int uh = __double2hiint(v[r]), lh = __double2hiint(v[12 + r]);
        int u1, u0, l1, l0;
        fx_magnitude<8>((uint32_t)uh, (uint32_t)__double2loint(v[r]), emax, u1, u0);
        fx_magnitude<8>((uint32_t)lh, (uint32_t)__double2loint(v[12 + r]), emax, l1, l0);
        const int su = (uh >> 31) | 1, sl = ((lh >> 31) ^ fl) | 1;
        n1[r] = l1 * sl + u1 * su;
        n0[r] = l0 * sl + u0 * su;
      }
    }
    int* emax = e_sm + 2 * site_local + t;  // largest exponent of the site's slices in this term
    atomicMax(emax, e_sum);
    long long C[18];
    // the nine complex sums, 2^(e_sum - 2102) each; where the own projection reads its second spins
    const int2* partner[4];
    int psign[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const int k = h >> 1, im = h & 1;
      partner[h] = own + (mu < 2 ? 18 - 6 * k : 12 + 6 * k) + (im_form ? 1 - im : im);
      psign[h] = (neg >> h) & 1u ? -1 : 1;
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      // digits of the projected own spinor, colour b: [h][re, im]
      int o1[4], o0[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int2 u = own[6 * (h >> 1) + 2 * b + (h & 1)];
        const int2 l = partner[h][2 * b];
        o1[h] = l.x * psign[h] + u.x;
        o0[h] = l.y * psign[h] + u.y;
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        long long hr = 0, hi = 0, cr = 1ll << 27, ci = 1ll << 27;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int xr1 = n1[6 * k + 2 * a], xr0 = n0[6 * k + 2 * a];
          const int xi1 = n1[6 * k + 2 * a + 1], xi0 = n0[6 * k + 2 * a + 1];
          const int yr1 = o1[2 * k], yr0 = o0[2 * k], yi1 = o1[2 * k + 1], yi0 = o0[2 * k + 1];
          const int zi1 = -yi1, zi0 = -yi0;
          hr += (long long)xr1 * yr1;
          cr += (long long)xr1 * yr0;
          cr += (long long)xr0 * yr1;
          hr += (long long)xi1 * yi1;
          cr += (long long)xi1 * yi0;
          cr += (long long)xi0 * yi1;
          hi += (long long)xi1 * yr1;
          ci += (long long)xi1 * yr0;
          ci += (long long)xi0 * yr1;
          hi += (long long)xr1 * zi1;
          ci += (long long)xr1 * zi0;
          ci += (long long)xr0 * zi1;
        }
        C[(a * 3 + b) * 2] = hr + (cr >> 28);
        C[(a * 3 + b) * 2 + 1] = hi + (ci >> 28);
      }
    }
    const bool any_bad = __syncthreads_or(bad) != 0;  // also: every exponent is in e_sm
    long long* dst = part + (size_t)tid * FORCE_FX_STRIDE;
    if (!any_bad) {
      // to the site's largest exponent, and sum_shift bits further for the sum over the slices
      const int d = *emax - e_sum + sum_shift;
      const long long half = d > 0 && d < 64 ? 1ll << (d - 1) : 0;
#pragma unroll
      for (int k = 0; k < 18; ++k) dst[k] = d < 64 ? (C[k] + half) >> d : 0;
    } else if (t == 0) {
      double B[36];
      force_products_ieee(psi + xo, chi + xo, psi + jo, chi + jo, mu, s, Lsh, B);
      double* both = reinterpret_cast<double*>(dst);  // both lanes' slots
      for (int k = 0; k < 36; ++k) both[k] = B[k];
    }
    __syncthreads();
    // sums over the site's slices, one (site, entry) per task
    for (int task = tid; task < nsites * 36; task += blockDim.x) {
      const int sl = task / 36, e = task - sl * 36, term = e / 18, k = e - term * 18;
      double v = 0;
      if (!any_bad) {
        // B2 = C^+: entry (a, b) from (b, a), imaginary part negated
        const int ab = k >> 1, a = ab / 3, b = ab - a * 3;
        const int kk = term ? (b * 3 + a) * 2 + (k & 1) : k;
        const long long* src = part + ((size_t)sl * nsg + term) * FORCE_FX_STRIDE + kk;
        long long tot = 0;
        int terms = 0;  // sum of the slices' magnitudes (2^32 of their units)
        for (int q = 0; q < Lsp; ++q) {
          const long long c = src[q * (2 * FORCE_FX_STRIDE)];
          tot += c;
          terms += abs((int)(c >> 32));
        }
        v = (double)tot;
        const int ex = e_sm[2 * sl + term] + sum_shift - 2102;
        if (tot != 0) v = __hiloint2double(__double2hiint(v) + (ex << 20), __double2loint(v));
        if (term && (k & 1)) v = -v;
        if (terms < (FORCE_FX_MIN_TERMS >> sum_shift)) {  // then the other part of the complex number counts, too
          const int other = (kk ^ 1) - kk;
          for (int q = 0; q < Lsp; ++q) terms += abs((int)(src[q * (2 * FORCE_FX_STRIDE) + other] >> 32));
        }
        if (terms < (FORCE_FX_MIN_TERMS >> sum_shift))
          v = force_entry_ieee(g, psi, chi, p, first + sl, mu, term, a, b, k & 1);
      } else {
        const double* src = reinterpret_cast<const double*>(part + (size_t)sl * nsg * FORCE_FX_STRIDE) + e;
        for (int q = 0; q < Lsp; ++q) v += src[q * (2 * FORCE_FX_STRIDE)];
      }
      bsum[((size_t)sl * 4 + mu) * 36 + e] = v;
    }
    __syncthreads();  // shared memory is reused by the next direction
    if (ts < 2) e_sm[2 * site_local + ts] = 0;
    __syncthreads();
  }

  // ---- link algebra (see force_site_algebra), links and Y in the own spinors' place; tasks (site, mu, a, b)
  constexpr int LB = link_bytes(8, C12);
  double* usm = reinterpret_cast<double*>(own_sm);  // [spc][mu][18]
  double* ysm = usm + (size_t)spc * 4 * 18;        // [spc][mu][18]
  for (int task = tid; task < nsites * 4; task += blockDim.x) {
    double u[18];
    load_link<P64, C12>((p ? Uo : Ue) + ((size_t)first * 4 + task) * LB, u);
#pragma unroll
    for (int k = 0; k < 18; ++k) usm[(size_t)task * 18 + k] = u[k];
  }
  __syncthreads();
  // site of the CTA and direction of a task: canonical index of the link and its boundary phase
  auto link_of = [&](int task, size_t& out, double& ph) {
    const int sl = task / 36, mu = (task - sl * 36) / 9;
    int x[4];
    cb_coords(g, first + sl, p, x);
    const long lex = x[0] + (long)g.L[0] * (x[1] + (long)g.L[1] * (x[2] + (long)g.L[2] * x[3]));
    const int xm = mu == 0 ? x[0] : mu == 1 ? x[1] : mu == 2 ? x[2] : x[3];
    const int L = mu == 0 ? g.L[0] : mu == 1 ? g.L[1] : mu == 2 ? g.L[2] : g.L[3];
    const int bc = mu == 0 ? g.bc[0] : mu == 1 ? g.bc[1] : mu == 2 ? g.bc[2] : g.bc[3];
    out = ((size_t)lex * 4 + mu) * 18;
    ph = xm == L - 1 && bc < 0 ? -coef : coef;  // F and G are linear in the boundary phase and coef
  };
  for (int task = tid; task < nsites * 36; task += blockDim.x) {
    const int link = task / 9, ab = task - link * 9, a = ab / 3, b = ab - a * 3;
    size_t out;
    double ph;
    link_of(task, out, ph);
    const double* B1 = bsum + (size_t)link * 36;
    const double* B2 = B1 + 18;
    const double* ur = usm + (size_t)link * 18;
    double yr = 0, yi = 0;  // -U B1 + B2 U^+
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double ar = ur[(a * 3 + k) * 2], ai = ur[(a * 3 + k) * 2 + 1];
      const double br = B1[(k * 3 + b) * 2], bi = B1[(k * 3 + b) * 2 + 1];
      yr = fma(-ar, br, fma(ai, bi, yr));
      yi = fma(-ar, bi, fma(-ai, br, yi));
      const double cr = B2[(a * 3 + k) * 2], ci = B2[(a * 3 + k) * 2 + 1];
      const double dr = ur[(b * 3 + k) * 2], di = ur[(b * 3 + k) * 2 + 1];  // (U^+)[k][b] = conj(U[b][k])
      yr = fma(cr, dr, fma(ci, di, yr));
      yi = fma(ci, dr, fma(-cr, di, yi));
    }
    ysm[(size_t)link * 18 + ab * 2] = ph * yr;
    ysm[(size_t)link * 18 + ab * 2 + 1] = ph * yi;
    if (G) {
      G[out + ab * 2] = -ph * (B1[(b * 3 + a) * 2] + B2[ab * 2]);
      G[out + ab * 2 + 1] = -ph * (B2[ab * 2 + 1] - B1[(b * 3 + a) * 2 + 1]);
    }
  }
  __syncthreads();
  if (F) {
    for (int task = tid; task < nsites * 36; task += blockDim.x) {
      const int link = task / 9, ab = task - link * 9, a = ab / 3, b = ab - a * 3;
      size_t out;
      double ph;
      link_of(task, out, ph);
      const double* Y = ysm + (size_t)link * 18;
      const double re = 0.5 * (Y[(b * 3 + a) * 2] - Y[(a * 3 + b) * 2]);
      double im = -0.5 * (Y[(a * 3 + b) * 2 + 1] + Y[(b * 3 + a) * 2 + 1]);
      if (a == b) im += (Y[1] + Y[9] + Y[17]) * (1.0 / 3.0);
      F[out + ab * 2] = re;
      F[out + ab * 2 + 1] = im;
    }
  }
}

// FP64 fields in float-float arithmetic (the handle's FP64 arithmetic set to float-float): the
// per-slice products in pairs of FP32 numbers, the slice sums in float-float, then the site's
// sums rounded to FP64 for the (per 4D site, cheap) link algebra. One thread per (site, slice)
// (Ls <= 128, so one slice each); the direction loop is not unrolled, and the projections read
// their direction-dependent parts by address, so that one short code path serves every mu (the
// unrolled float-float code would overflow the instruction cache, as in the hopping kernel).
template <bool C12>
__global__ void __launch_bounds__(128) k_force_ff(const Geom g, const char* psi, const char* chi, const char* Ue,
                                                  const char* Uo, double* F, double* G, double coef, int nsg,
                                                  int spc) {
  using namespace ffa;
  const int Lsh = ls_half(g.Ls);
  const size_t site_bytes = (size_t)Lsh * 2 * 24 * 8;
  const size_t half_bytes = (size_t)g.N4h * site_bytes;
  const size_t cs = chunk_stride(Lsh);
  const int p = blockIdx.x & 1;
  const int first = (blockIdx.x >> 1) * spc;
  const int tid = threadIdx.x;
  const int site_local = tid / nsg;
  const int t = tid - site_local * nsg;  // the thread's slice
  const int nsites = min(spc, g.N4h - first);
  const bool active = site_local < nsites;
  const int i = first + (active ? site_local : 0);
  int c[4];
  cb_coords(g, i, p, c);
  const char* psi_x = psi + p * half_bytes + site_offset(i, Lsh, site_bytes) + (size_t)t * 8;
  const char* chi_x = chi + p * half_bytes + site_offset(i, Lsh, site_bytes) + (size_t)t * 8;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  long* lex_sm = reinterpret_cast<long*>(smem_raw);
  int* ph_sm = reinterpret_cast<int*>(lex_sm + spc);
  ff* part = reinterpret_cast<ff*>(smem_raw + (size_t)spc * 2 * sizeof(long));  // [spc][nsg][37] (S, E) pairs
  double* bsum = reinterpret_cast<double*>(part + (size_t)spc * nsg * FORCE_PART_STRIDE);  // [spc][36]
  double* usm = bsum + (size_t)spc * 36;
  double* ysm = usm + (size_t)spc * 18;
  if (active && t == 0) lex_sm[site_local] = c[0] + (long)g.L[0] * (c[1] + (long)g.L[1] * (c[2] + (long)g.L[2] * c[3]));
  // forward neighbours and phases at compile-time mu (a runtime mu would index c and g through
  // local memory), picked by selects in the rolled loop below
  int nf[4], pf[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) nf[m] = cb_neighbour(g, i, c, m, true, pf[m]);

#pragma unroll 1
  for (int mu = 0; mu < 4; ++mu) {
    if (active) {
      const int j = mu == 0 ? nf[0] : mu == 1 ? nf[1] : mu == 2 ? nf[2] : nf[3];
      const int ph = mu == 0 ? pf[0] : mu == 1 ? pf[1] : mu == 2 ? pf[2] : pf[3];
      if (t == 0) ph_sm[site_local] = ph;
      const size_t jo = (1 - p) * half_bytes + site_offset(j, Lsh, site_bytes) + (size_t)t * 8;
      ff* dst = part + ((size_t)site_local * nsg + t) * FORCE_PART_STRIDE;
      // term 0: B1 = psi(x+mu) (x) [(1 - gamma) chi(x)]^+;  term 1: B2 = psi(x) (x) [(1 + gamma) chi(x+mu)]^+
#pragma unroll 1
      for (int term = 0; term < 2; ++term) {
        const int S = term == 0 ? -1 : +1;
        ff ha[12], hb[12];
        project_load_ff(term == 0 ? psi + jo : psi_x, mu, S, cs, ha);
        project_load_ff(term == 0 ? chi_x : chi + jo, mu, S, cs, hb);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b = 0; b < 3; ++b) {  // sum_h ha[h][a] conj(hb[h][b])
            ffacc re, im;
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
              const ff xr = ha[(hh * 3 + a) * 2], xi = ha[(hh * 3 + a) * 2 + 1];
              const ff yr = hb[(hh * 3 + b) * 2], yi = hb[(hh * 3 + b) * 2 + 1];
              if (hh == 0) {
                dot_first(re, xr, yr, false);
                dot_first(im, xi, yr, false);
              } else {
                dot_add<+1>(re, xr, yr);
                dot_add<+1>(im, xi, yr);
              }
              dot_add<+1>(re, xi, yi);
              dot_add<-1>(im, xr, yi);
            }
            dst[term * 18 + (a * 3 + b) * 2] = ff_make(re.s, re.e);
            dst[term * 18 + (a * 3 + b) * 2 + 1] = ff_make(im.s, im.e);
          }
      }
    }
    __syncthreads();
    // ---- sum over the site's slices in float-float, one (site, entry) per task, rounded to FP64
    for (int task = tid; task < nsites * 36; task += blockDim.x) {
      const int sl = task / 36, e = task - sl * 36;
      const ff* src = part + (size_t)sl * nsg * FORCE_PART_STRIDE + e;
      ff total = ff_make(0.f, 0.f);
      for (int k = 0; k < nsg; ++k) acc_add(total, src[(size_t)k * FORCE_PART_STRIDE]);
      bsum[(size_t)sl * 36 + e] = ff_to_double(fast_two_sum(total.hi, total.lo));
    }
    force_site_algebra<P64, C12, double>(mu, p, first, nsites, Ue, Uo, bsum, usm, ysm, lex_sm, ph_sm, coef, F, G);
    __syncthreads();  // shared memory is reused by the next direction
  }
}

cudaError_t launch_force(int prec, bool c12, const Geom& g, const void* psi, const void* chi, const void* Ue,
                         const void* Uo, double* F, double* G, double coef, bool float_float, cudaStream_t st) {
  const int nsg = force_threads_per_site(prec, g.Ls);
  const size_t per_site = force_smem_per_site(prec, nsg);
  int spc = 128 / nsg;
  if ((size_t)spc * per_site > 48 * 1024) spc = (int)(48 * 1024 / per_site);  // short Ls: many sites per CTA
  if (spc < 1) spc = 1;
  const int threads = nsg * spc;
  const dim3 grid((unsigned)(2 * ((g.N4h + spc - 1) / spc)));  // (site block, parity), parity fastest
  const size_t smem = (size_t)spc * per_site;
  const char* ps = static_cast<const char*>(psi);
  const char* ch = static_cast<const char*>(chi);
  const char* e = static_cast<const char*>(Ue);
  const char* o = static_cast<const char*>(Uo);
  if (prec == P64 && float_float) {
    if (c12)
      k_force_ff<true><<<grid, threads, smem, st>>>(g, ps, ch, e, o, F, G, coef, nsg, spc);
    else
      k_force_ff<false><<<grid, threads, smem, st>>>(g, ps, ch, e, o, F, G, coef, nsg, spc);
    return cudaGetLastError();
  }
  const int Lsh = ls_half(g.Ls);
  if (prec == P64) {
    const int n2 = 2 * ls_padded(g.Ls);  // two threads per slice
    const int s2 = std::max(1, std::min(FORCE_FX_THREADS / n2, FORCE_FX_SITES));
    int shift = 0;
    while ((1 << shift) < g.Ls) ++shift;
    const size_t sm = force_fx_smem(n2, s2);
    const dim3 gr((unsigned)(2 * ((g.N4h + s2 - 1) / s2)));
    auto kern = c12 ? k_force_fx<true> : k_force_fx<false>;
    if (sm > 48 * 1024) {
      cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
      if (err != cudaSuccess) return err;
    }
    kern<<<gr, n2 * s2, sm, st>>>(g, ps, ch, e, o, F, G, coef, n2, s2, shift);
    return cudaGetLastError();
  }
  // (k_force_reg stores F and G in pairs of reals)
  const bool aligned = (reinterpret_cast<uintptr_t>(F) | reinterpret_cast<uintptr_t>(G)) % 16 == 0;
  if (prec == P32 && Lsh >= 3 && Lsh <= 16 && aligned) {
    // CTAs of 64 threads for up to 8 pairs per site (8 or 16 sites; measured 108.2 us against 109.5 us
    // with 128 threads at 16^4 x 16, the same warps per SM and a finer last wave), 128 above
#define FR(L_, T_)                                                                                       \
  {                                                                                                      \
    constexpr int spc = ForceRegGeom<L_, T_>::SPC;                                                       \
    const dim3 gr((unsigned)(2 * ((g.N4h + spc - 1) / spc)));                                            \
    auto kern = Lsh == L_ ? (c12 ? k_force_reg<true, L_, true, T_> : k_force_reg<false, L_, true, T_>)    \
                          : (c12 ? k_force_reg<true, L_, false, T_> : k_force_reg<false, L_, false, T_>); \
    kern<<<gr, T_, 0, st>>>(g, ps, ch, e, o, F, G, coef);                                                \
  }
    if (Lsh <= 4) FR(4, 64) else if (Lsh <= 8) FR(8, 64) else FR(16, 128)
#undef FR
    return cudaGetLastError();
  }
  if (prec != P32) return cudaErrorInvalidValue;
  if (c12)
    k_force<true><<<grid, threads, smem, st>>>(g, ps, ch, e, o, F, G, coef, nsg, spc);
  else
    k_force<false><<<grid, threads, smem, st>>>(g, ps, ch, e, o, F, G, coef, nsg, spc);
  return cudaGetLastError();
}

}  // namespace gdwf
