// Instantiates launch_dhop_pairs<DWF_PREC, DWF_PAIRS> of a packed precision (P32, P16, PB16) and
// extent Ls = 2 DWF_PAIRS (0: any Ls). The build compiles this file once for each of them (both macros are
// given on the command line), in parallel.
#include "dhop_kernel.cuh"

namespace gdwf {

template <bool DAG, bool C12, int EK>
static cudaError_t launch_one(const DhopArgs& a, int threads, int blocks, size_t smem, cudaStream_t stream) {
  auto kern = dhop_kernel<DWF_PREC, DAG, C12, DWF_PAIRS, EK>;
  if (smem > 48 * 1024) {
    static size_t configured = 0;  // per instantiation
    if (smem > configured) {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      configured = smem;
    }
  }
  // full CTAs only (the packed kernel has no tail handling); a ragged end gets one more CTA (per
  // half) flush with the end of the lattice, launched after the first so no two writes overlap
  // in time. a.in2 != nullptr: both halves of a full-lattice hop in the same launches.
  // CG epilogues: partial sums [0, halves * full) from the full CTAs (CTA order), then one per
  // half from the end CTAs, which add only the sites the full CTAs did not cover.
  const int nsites = a.region_sites > 0 ? a.region_sites : a.g.N4h;
  const int full = nsites / a.sites_per_cta;
  const int halves = a.in2 ? 2 : 1;
  DhopArgs m = a;
  m.blocks1 = full;
  m.red_base = 0;
  m.own_from = 0;
  if (full > 0) {
    if (a.pdl) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(halves * full);
      cfg.blockDim = dim3(threads);
      cfg.dynamicSmemBytes = smem;
      cfg.stream = stream;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[0].val.programmaticStreamSerializationAllowed = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      cudaError_t e = cudaLaunchKernelEx(&cfg, kern, m);
      if (e != cudaSuccess) return e;
    } else {
      kern<<<halves * full, threads, smem, stream>>>(m);
    }
  }
  if (a.region_sites == 0 && full * a.sites_per_cta != a.g.N4h) {
    DhopArgs t = a;
    t.site_base = a.g.N4h - a.sites_per_cta;
    t.blocks1 = 1;
    t.red_base = halves * full;
    t.own_from = full * a.sites_per_cta;
    kern<<<halves, threads, smem, stream>>>(t);
  }
  return cudaGetLastError();
}

template <>
cudaError_t launch_dhop_pairs<DWF_PREC, DWF_PAIRS>(const DhopArgs& a, bool dag, bool c12, int threads, int blocks,
                                                   size_t smem, cudaStream_t stream) {
  // the instantiation with exactly the epilogue parts this launch uses; the CG epilogues exist
  // for the launches that use them only: Mpc's second launch (pre-operation Mooee, no dag) with
  // the norm, Mpc^+'s second launch (Mooee^+, dag) with the update, 18-real links
  if (a.halo_fwd) {  // a face region of a block of a lattice split in t (plain hop)
    if constexpr (dhop_halo_pairs(DWF_PAIRS)) {
      if (a.pre != PRE_NONE || a.post != POST_NONE || a.red || a.in2) return cudaErrorInvalidValue;
      if (dag) return c12 ? launch_one<true, true, EPI_HALO>(a, threads, blocks, smem, stream)
                          : launch_one<true, false, EPI_HALO>(a, threads, blocks, smem, stream);
      return c12 ? launch_one<false, true, EPI_HALO>(a, threads, blocks, smem, stream)
                 : launch_one<false, false, EPI_HALO>(a, threads, blocks, smem, stream);
    }
    return cudaErrorInvalidValue;
  }
  if (a.pre == (dag ? PRE_MOOEE : PRE_MOOEE_DAG) || a.post == (dag ? POST_INV : POST_INV_DAG))
    return cudaErrorInvalidValue;
  if (a.red && !c12 && a.pre != PRE_NONE && a.post == POST_NONE) {
    if (a.r && dag) return launch_one<true, false, EPI_PRE | EPI_AXPY>(a, threads, blocks, smem, stream);
    if (!a.r && !dag) return launch_one<false, false, EPI_PRE | EPI_NORM>(a, threads, blocks, smem, stream);
    return cudaErrorInvalidValue;
  }
  if (a.red) return cudaErrorInvalidValue;
  const int ek = (a.pre != PRE_NONE ? EPI_PRE : 0) | (a.post != POST_NONE ? EPI_POST : 0);
#define DWF_EK(K)                                                                         \
  case K:                                                                                 \
    if (dag) return c12 ? launch_one<true, true, K>(a, threads, blocks, smem, stream)     \
                        : launch_one<true, false, K>(a, threads, blocks, smem, stream);   \
    return c12 ? launch_one<false, true, K>(a, threads, blocks, smem, stream)             \
               : launch_one<false, false, K>(a, threads, blocks, smem, stream);
  switch (ek) {
    DWF_EK(EPI_NONE)
    DWF_EK(EPI_PRE)
    DWF_EK(EPI_POST)
  }
#undef DWF_EK
  return cudaErrorInvalidValue;
}

}  // namespace gdwf
