// complex64 levels of the Weyl basis, several per pass (tpd_qudit.cuh).
#include "tpd_qudit.cuh"
#include "tpd_weyl.cuh"

namespace tpd {
namespace {

template <bool kDec>
struct WeylOp {
  using Const = Twiddles<float>;
  // the decomposition's 1/d on every level, the composition's scale on the last alone
  template <int D>
  __device__ static __forceinline__ void block(const float2 (&x)[D][D], float2 (&y)[D][D], const Const& c, bool last) {
    Const k = c;
    if (!kDec && !last) k.scale = 1.0f;
    weyl_block_ieee<float, D, kDec>(x, y, k);
  }
};

}  // namespace

cudaError_t weyl_c64(bool dec, const float2* src, float2* mat, int n, int d, double last_scale, cudaStream_t st) {
  auto consts = [&](bool last) { return twiddles<float>(d, dec ? 1.0 / d : (last ? last_scale : 1.0)); };
  return dec ? run_qudit<WeylOp<true>>(src, mat, n, d, consts, st)
             : run_qudit<WeylOp<false>>(src, mat, n, d, consts, st);
}

}  // namespace tpd
