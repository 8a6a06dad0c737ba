// Double-float local operator with stored factors, 8 to 12 points per direction (kernel in
// k_ax_df.cuh).
#include "k_ax_df.cuh"

namespace sem {
namespace {

template <int NP>
struct DfStored {
  static sem_status run(int N, bool cg, const AxLaunch& a, cudaStream_t s) {
    if constexpr (f64x_on_slices(NP - 1)) {
      if constexpr (f64x_plain_pairs(NP - 1, 0))
        if (a.g_pairs && !cg) return launch_df_t<NP, false, kGkPairs>(N, a, s);
      return launch_ax_slice(N, cg, a, s);
    } else {
      if (a.g_pairs)
        return cg ? launch_df_t<NP, true, kGkPairs>(N, a, s) : launch_df_t<NP, false, kGkPairs>(N, a, s);
      constexpr int kGk = ax_slice_order(NP - 1) ? kGkFixed : kGkF64;
      return cg ? launch_df_t<NP, true, kGk>(N, a, s) : launch_df_t<NP, false, kGk>(N, a, s);
    }
  }
};

}  // namespace

sem_status launch_ax_f64x_hi(int N, bool cg, const AxLaunch& a, cudaStream_t s) {
  return df_dispatch<DfStored, 8, 12>(N, cg, a, s);
}

}  // namespace sem
