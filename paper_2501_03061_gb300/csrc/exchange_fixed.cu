// Pair-FFT exchange on cubic grids with a compile-time side N (Sec. IV-A1, Eq. vxdiag): dispatch of
// one pair batch to the kernels of exchange_fixed_kernels.cuh (the FP64 form, Algorithm 2's triple loop, and
// in FP32 option exchange64_engine = 1).
#include "exchange_fixed_kernels.cuh"

namespace pt {

template <class T>
void exchange_batch_fixed(int n, const cx<T>* src, const cx<T>* tgt, const double* occ, const PairDesc* pairs, int np,
                          const TargetDesc* tgts, int nt, const Contrib* contribs, const T* ktab, const cx<T>* tw,
                          cx<T>* scratch, cx<T>* out, cudaStream_t st) {
  switch (n) {
#define PT_CASE(s)                                                                                      \
  case s:                                                                                               \
    batch_n<s, T>(src, tgt, occ, pairs, np, tgts, nt, contribs, ktab, tw, scratch, out, st);            \
    return;
    PT_FIXED_SIZES(PT_CASE)
#undef PT_CASE
    default:
      fail(PT_INVALID_ARG, "no compile-time FFT kernels for this grid side");
  }
}

template void exchange_batch_fixed<float>(int, const c64*, const c64*, const double*, const PairDesc*, int,
                                          const TargetDesc*, int, const Contrib*, const float*, const c64*, c64*, c64*,
                                          cudaStream_t);
template void exchange_batch_fixed<double>(int, const c128*, const c128*, const double*, const PairDesc*, int,
                                           const TargetDesc*, int, const Contrib*, const double*, const c128*, c128*,
                                           c128*, cudaStream_t);

}  // namespace pt
