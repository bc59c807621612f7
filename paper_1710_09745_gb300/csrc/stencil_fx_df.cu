// The digit stencil (stencil_fx.cuh) for the double-float kind.
#include "stencil_fx.cuh"

namespace bcg {

cudaError_t dslash_fx_df(int flags, int epi, const void* links, const void* in, void* out,
                         const void* c1, const void* c2, double m2, const Geom& g, int out_parity,
                         int N, Gate gate, cudaStream_t s) {
  return N <= 8 ? fx::run_fx<StoreDF, 1>(flags, epi, links, in, out, c1, c2, m2, g, out_parity, N, gate, s)
                : fx::run_fx<StoreDF, 2>(flags, epi, links, in, out, c1, c2, m2, g, out_parity, N, gate, s);
}

cudaError_t fx_column_max(const void* f, const Geom& g, int N, Gate gate, cudaStream_t s) {
  fx::k_fx_zero<<<1, 64, 0, s>>>(g.fx_ctl, 0, gate);
  const long long rows = 3LL * g.Vh;
  const int rpb = 256 / N;
  const long long want = (rows + rpb - 1) / rpb, cap = (long long)stencil_sms() * (gate_mostly_off(gate) ? 2 : 8);
  fx::k_fx_colmax<StoreDF><<<(unsigned)(want < cap ? want : cap), 256, 0, s>>>(
      (const float4*)f, N, rows, g.fx_ctl, 0, gate);
  return cudaGetLastError();
}

}  // namespace bcg
