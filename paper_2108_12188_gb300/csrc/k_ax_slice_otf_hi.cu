// FP64 operator with factors rebuilt on the fly on the tensor cores at 9 to 12 points per direction
// (k_ax_slice16.cuh), the orders of ax_slice_order.
#include "k_ax_slice16.cuh"

namespace sem {
namespace {

template <int NP>
sem_status launch_slice16(int N, bool cg, const AxLaunch& a, cudaStream_t s) {
  if constexpr (ax_slice_order(NP - 1))
    if (N + 1 == NP) return cg ? launch_slice16_t<NP, true, true>(N, a, s) : launch_slice16_t<NP, false, true>(N, a, s);
  if constexpr (NP < 12) return launch_slice16<NP + 1>(N, cg, a, s);
  return fail(SEM_ERR_UNSUPPORTED, "polynomial order not compiled in");
}

}  // namespace

sem_status launch_ax_slice_otf_hi(int N, bool cg, const AxLaunch& a, cudaStream_t s) { return launch_slice16<9>(N, cg, a, s); }

}  // namespace sem
