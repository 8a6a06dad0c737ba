// FP64 operator with stored factors on the tensor cores (k_ax_slice.cuh) at the orders of
// ax_slice_order, up to 8 points per direction.
#include "k_ax_slice.cuh"

namespace sem {
namespace {

template <int NP>
sem_status launch_slice(int N, bool cg, const AxLaunch& a, cudaStream_t s) {
  if constexpr (ax_slice_order(NP - 1))
    if (N + 1 == NP) return cg ? launch_slice_t<NP, true, false>(N, a, s) : launch_slice_t<NP, false, false>(N, a, s);
  if constexpr (NP < 8) return launch_slice<NP + 1>(N, cg, a, s);
  return fail(SEM_ERR_UNSUPPORTED, "polynomial order not compiled in");
}

}  // namespace

sem_status launch_ax_slice(int N, bool cg, const AxLaunch& a, cudaStream_t s) {
  return N <= 7 ? launch_slice<2>(N, cg, a, s) : launch_ax_slice_hi(N, cg, a, s);
}

}  // namespace sem
