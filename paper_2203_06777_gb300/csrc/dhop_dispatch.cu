// launch_dhop of the packed precisions: the instantiation (dhop_packed.cu) for the extent.
#include "dhop_kernel.cuh"

namespace gdwf {

template <int P>
static cudaError_t by_pairs(const DhopArgs& a, bool dag, bool c12, int threads, int blocks, size_t smem,
                            cudaStream_t stream) {
  const int pairs = a.g.Ls & 1 ? 0 : a.g.Ls / 2;
  switch (a.halo_fwd && !dhop_halo_pairs(pairs) ? 0 : pairs) {
#define DWF_CASE(N_) \
  case N_:           \
    return launch_dhop_pairs<P, N_>(a, dag, c12, threads, blocks, smem, stream);
    DWF_PAIR_SPECIALISATIONS(DWF_CASE)
#undef DWF_CASE
    default:
      return launch_dhop_pairs<P, 0>(a, dag, c12, threads, blocks, smem, stream);
  }
}

template <>
cudaError_t launch_dhop<P32>(const DhopArgs& a, bool dag, bool c12, int threads, int blocks, size_t smem,
                             cudaStream_t stream) {
  return by_pairs<P32>(a, dag, c12, threads, blocks, smem, stream);
}
template <>
cudaError_t launch_dhop<P16>(const DhopArgs& a, bool dag, bool c12, int threads, int blocks, size_t smem,
                             cudaStream_t stream) {
  return by_pairs<P16>(a, dag, c12, threads, blocks, smem, stream);
}
template <>
cudaError_t launch_dhop<PB16>(const DhopArgs& a, bool dag, bool c12, int threads, int blocks, size_t smem,
                              cudaStream_t stream) {
  return by_pairs<PB16>(a, dag, c12, threads, blocks, smem, stream);
}

}  // namespace gdwf
