// complex64 levels of the generalized Gell-Mann basis, several per pass
// (tpd_qudit.cuh).
#include "tpd_gellmann.cuh"
#include "tpd_qudit.cuh"

namespace tpd {
namespace {

template <bool kDec>
struct GmOp {
  using Const = GmConst<float>;
  // the composition's scale belongs to the last level alone
  template <int D>
  __device__ static __forceinline__ void block(const float2 (&x)[D][D], float2 (&y)[D][D], const Const& c, bool last) {
    Const k = c;
    if (!last) k.scaled = 0;
    gm_block<float, D, kDec>(x, y, k);
  }
};

}  // namespace

cudaError_t gellmann_c64(bool dec, const float2* src, float2* mat, int n, int d, double last_scale,
                         cudaStream_t st) {
  auto consts = [&](bool last) { return gm_const<float>(d, last ? last_scale : 1.0); };
  return dec ? run_qudit<GmOp<true>>(src, mat, n, d, consts, st) : run_qudit<GmOp<false>>(src, mat, n, d, consts, st);
}

}  // namespace tpd
