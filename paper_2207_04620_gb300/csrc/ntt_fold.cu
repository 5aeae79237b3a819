// The NTT's kernels for chains of primes just below powers of two (ArithFold).
#include "ntt_impl.cuh"

namespace hx {

template void ntt_phase<ArithFold>(const LaunchCtx &, const NttRows &, bool, bool, int, int);
template void ntt_multi_phases<ArithFold>(cudaStream_t, const NttJob *, int, int, int, bool);

} // namespace hx
