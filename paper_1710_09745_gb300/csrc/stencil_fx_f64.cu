// The digit stencil (stencil_fx.cuh) for the native-FP64 kind.
#include "stencil_fx.cuh"

namespace bcg {

cudaError_t dslash_fx_f64(int flags, int epi, const void* links, const void* in, void* out,
                          const void* c1, const void* c2, double m2, const Geom& g, int out_parity,
                          int N, Gate gate, cudaStream_t s) {
  return N <= 8 ? fx::run_fx<StoreF64, 1>(flags, epi, links, in, out, c1, c2, m2, g, out_parity, N, gate, s)
                : fx::run_fx<StoreF64, 2>(flags, epi, links, in, out, c1, c2, m2, g, out_parity, N, gate, s);
}

}  // namespace bcg
