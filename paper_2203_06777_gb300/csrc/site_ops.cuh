// Site-local kernels of the library: layout conversion (pack/unpack of spinors and links),
// precision conversion, the standalone fifth-dimension operators Mooee / Mooee^-1, the
// FP64-accumulated reductions and the CG vector updates. Launchers are declared here and
// defined in site_ops.cu.
#pragma once

#include "dwf_common.cuh"

namespace gdwf {

// Scalars of a CG solve, kept in device memory so that iterations need no host round trip.
enum CgScalar : int {
  S_RR = 0,     // |r|^2 of the current residual
  S_PAP = 1,    // <p, A p>
  S_ALPHA = 2,  // rr / pAp
  S_BETA = 3,   // rr_new / rr (times the p rescale factor)
  S_RRNEW = 4,  // |r_new|^2
  S_PSCALE = 5, // factor applied to p in the next p update (rescaling of the sloppy vectors)
  S_TMP0 = 6,
  S_TMP1 = 7,
  S_RROLD = 8,  // |r|^2 before the last FIN_BETA (the denominator of its beta)
  S_COUNT = 16
};

// Fixed reduction geometry: the partial-sum layout, and hence the summation order, never
// depends on the data, so results are bitwise reproducible.
constexpr int RED_BLOCKS = 608;  // 4 x 152 SMs
constexpr int RED_THREADS = 256;

// Finalise kinds: what is done with the total.
enum FinalKind : int {
  FIN_STORE = 0,  // scal[dst] = total (and scal[dst+1] = imaginary part for inner products)
  FIN_ALPHA = 1,  // scal[S_PAP] = total; scal[S_ALPHA] = scal[S_RR] / total
  FIN_BETA = 2,   // scal[S_RRNEW] = total; scal[S_BETA] = scal[S_PSCALE] * total / scal[S_RR];
                  // scal[S_RROLD] = scal[S_RR]; scal[S_RR] = total
};

// Where the total of a launch's per-CTA partial sums goes. The CTA that stores its partial sum last
// (by an atomic count, which it sets back to 0) adds all of them in a fixed order and finalises the
// total as `kind`, so that no second launch is needed: a launch of one CTA for it took 5 us, twice per
// CG iteration. Mixed FP32 CG at 16^4 x 12 (200 iterations) 42.3 -> 41.3 ms; conversion, norm and inner
// product at 8^4 x 8 74 -> 57 us (their results reach the host without a copy, too).
struct Final {
  unsigned* count;  // of the handle; 0 between launches
  double* scal;
  int kind, dst;
  double* host;     // pinned host memory that receives the total too (no copy), or null
};

__device__ __forceinline__ void apply_final(const Final& f, double tot, double tot_im, bool two) {
  double* scal = f.scal;
  if (f.kind == FIN_STORE) {
    scal[f.dst] = tot;
    if (two) scal[f.dst + 1] = tot_im;
  } else if (f.kind == FIN_ALPHA) {
    scal[S_PAP] = tot;
    scal[S_ALPHA] = scal[S_RR] / tot;
  } else if (f.kind == FIN_BETA) {
    scal[S_RRNEW] = tot;
    scal[S_BETA] = scal[S_PSCALE] * tot / scal[S_RR];
    scal[S_RROLD] = scal[S_RR];
    scal[S_RR] = tot;
    scal[S_PSCALE] = 1.0;
  }
  if (f.host) {
    f.host[0] = tot;
    if (two) f.host[1] = tot_im;
    __threadfence_system();
  }
  *f.count = 0;
}

// Sum of one value per thread over the CTA in a fixed order (warp shuffles, then the warps in
// order), returned to thread 0. The last warp may be short: hopping CTAs are whole sites.
__device__ __forceinline__ double cta_sum(double v) {
  __shared__ double wsum[32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int lanes = min(32, (int)blockDim.x - 32 * warp);
  const unsigned mask = 0xffffffffu >> (32 - lanes);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const double t = __shfl_down_sync(mask, v, off);
    if (lane + off < lanes) v += t;
  }
  __syncthreads();
  if (lane == 0) wsum[warp] = v;
  __syncthreads();
  double t = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) t += wsum[w];
  return t;
}

// The sum of n values from p on, each read from L2, returned to thread 0.
__device__ __forceinline__ double cta_total(const double* p, int n) {
  double t = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) t += __ldcg(p + i);
  return cta_sum(t);
}

// Whether this CTA is the last of n to count on *count: every thread calls it, after thread 0's store
// of what the last one is to read.
__device__ __forceinline__ bool last_to_count(unsigned* count, int n) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(count, 1u) == (unsigned)n - 1u;
  }
  __syncthreads();
  const bool mine = last;
  if (mine) __threadfence();
  return mine;
}

// Called by every thread of every CTA after thread 0 has stored its CTA's NC sums at
// partials[k * total + blockIdx.x], total CTAs in all.
template <int NC>
__device__ __forceinline__ void finish_sums(const double* partials, int total, const Final& f) {
  if (!last_to_count(f.count, total)) return;
  const double re = cta_total(partials, total);
  const double im = NC > 1 ? cta_total(partials + total, total) : 0.0;
  if (threadIdx.x == 0) apply_final(f, re, im, NC > 1);
}

// The same for a hopping launch, whose thousands of small CTAs would keep the last one busy for 10-50 us:
// above SUM_DIRECT of them, sums of SUM_GROUP consecutive ones first, each by the last CTA of its group
// (group sums after the total partial sums in red, counts of the groups in gcount, 0 between launches).
constexpr int SUM_GROUP = 64, SUM_DIRECT = 512;
__host__ __device__ inline int sum_groups(int total) { return (total + SUM_GROUP - 1) / SUM_GROUP; }

__device__ __forceinline__ void finish_grouped_sums(double* red, unsigned* gcount, int total, int slot, double sum,
                                                    const Final& f) {
  if (threadIdx.x == 0) red[slot] = sum;
  if (total <= SUM_DIRECT) {
    finish_sums<1>(red, total, f);
    return;
  }
  const int groups = sum_groups(total), g = slot / SUM_GROUP;
  const int n = min(SUM_GROUP, total - g * SUM_GROUP);
  if (!last_to_count(gcount + g, n)) return;
  const double t = cta_total(red + g * SUM_GROUP, n);
  if (threadIdx.x == 0) {
    red[total + g] = t;
    gcount[g] = 0;
  }
  if (!last_to_count(f.count, groups)) return;
  const double all = cta_total(red + total, groups);
  if (threadIdx.x == 0) apply_final(f, all, 0.0, false);
}

cudaError_t launch_pack_spinor(int prec, const Geom& g, const double* canon, void* field, int subset, bool unpack,
                               cudaStream_t st);
cudaError_t launch_pack_gauge(int prec, bool c12, const Geom& g, const double* canon, void* Ueven, void* Uodd,
                              cudaStream_t st);
cudaError_t launch_convert(int psrc, int pdst, const void* src, void* dst, long nsites, int Ls, const double* scale_dev,
                           double scale, cudaStream_t st);
cudaError_t launch_mooee(int prec, const void* in, void* out, long nsites, int Ls, bool dag, bool inverse, double d5,
                         double mass, double inv_d5, double inv_den, cudaStream_t st);
// Reductions over nsites site blocks. inner: a^+ b (complex); otherwise |a|^2. The result goes
// to f.
cudaError_t launch_reduce(int prec, const void* a, const void* b, long nsites, int Ls, double* partials, const Final& f,
                          cudaStream_t st);
// CG updates. xr: x += alpha p, r -= alpha Ap, |r|^2 -> finalised as FIN_BETA.
cudaError_t launch_cg_xr(int px, int pp, void* x, void* r, const void* p, const void* Ap, long nsites, int Ls,
                         double* partials, const Final& f, cudaStream_t st);
// p = r + beta p.
// r -= alpha Ap and |r|^2 (finalised as FIN_BETA); x += alpha p, then (update_p) p = r + beta p.
cudaError_t launch_cg_r(int px, int pp, void* r, const void* Ap, long nsites, int Ls, double* partials, const Final& f,
                        cudaStream_t st);
cudaError_t launch_cg_xp(int px, int pp, void* x, const void* r, void* p, long nsites, int Ls, const double* scal,
                         bool update_p, cudaStream_t st);
cudaError_t launch_cg_p(int px, int pp, const void* r, void* p, long nsites, int Ls, const double* scal,
                        cudaStream_t st);
// r = b - Ax (FP64) and |r|^2, which goes to f.
cudaError_t launch_residual64(const void* b, const void* Ax, void* r, long nsites, int Ls, double* partials,
                              const Final& f, cudaStream_t st);
// x (FP64) += c * y (precision py), then y = 0, with c = *c_dev.
cudaError_t launch_accum_zero(int py, void* x, void* y, long nsites, int Ls, const double* c_dev, cudaStream_t st);

}  // namespace gdwf
