// The digit stencil's packed links (stencil_fx.cuh): sizes, support and the
// kernel that writes them once per gauge field.
#include "stencil_fx.cuh"

namespace bcg {
namespace fx {

// One warp per (parity, site), 8 sites of one link block per CTA, from the
// packed FP64 hop matrices (all factors folded in): the site's scale, the
// digits of its 144 entries in the stencil's reading order, and the
// accumulators' initial values -128 sum_{t <= u} sum_k B_t[k][o] in the units
// of the stencil's operands (2^-24 and 2^-9).  Runs once per gauge field.
__global__ void __launch_bounds__(256)
    k_fx_pack(const double2* __restrict__ links, unsigned char* __restrict__ main,
              unsigned char* __restrict__ extra, unsigned* __restrict__ bad, Geom g) {
  __shared__ double2 sL[8 * 145];
  __shared__ uint32_t rec[8][(REC_DIG + REC_EXTRA) / 4];
  __shared__ int sums[8][3][8][2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int groups = (g.Vh + 7) / 8;
  const int p = blockIdx.x / groups;
  const int s0 = (blockIdx.x - p * groups) * 8;
  {
    const double2* lb = links + link_offset(g, p, s0);
    for (int i = threadIdx.x; i < 144 * 8; i += 256) {
      const int de = i >> 3, k = i & 7;
      if (s0 + k < g.Vh) sL[k * 145 + de] = lb[(long long)de * LINK_W + k];
    }
  }
  for (int i = threadIdx.x; i < 8 * 48; i += 256) (&sums[0][0][0][0])[i] = 0;
  __syncthreads();
  const int site = s0 + warp;
  if (site >= g.Vh) return;
  const double2* Ls = sL + warp * 145;
  unsigned h = 0u;  // the largest entry of hop matrix lane / 2, by two lanes
  for (int i = lane & 1; i < 9; i += 2) h = max(h, Kind<StoreF64>::key(Ls[(lane >> 1) * 9 + i]));
  h = max(h, __shfl_xor_sync(0xffffffffu, h, 1));
  const unsigned m = __reduce_max_sync(0xffffffffu, h);
  const int e0 = exp_f64(m);
  const bool ok = e0 >= -90 && e0 <= 90;
  const int e = ok ? e0 : 0;
  auto below = [&](unsigned by) { return !ok || (h != 0u && h + by < m); };
  if (__any_sync(0xffffffffu, below(9u << 20)) && lane == 0) atomicOr(bad, 1u);
  if (__any_sync(0xffffffffu, below(13u << 19)) && lane == 0) atomicOr(bad + 1, 1u);  // 1.5 2^6
  // ten lanes per row colour c, so that a lane's column sums stay in registers
  const int c = lane / 10;
  int sum[8][2] = {};
  if (c < 3)
    for (int i = lane - 10 * c; i < 48; i += 10) {
      const int d = i / 3, j = i - 3 * (i / 3);
      const int en = 2 * (3 * (d >> 3) + j) + ((d >> 2) & 1), li = (d & 3) * 3 + c;
      uint32_t w[4];
      const double2 v = ok ? Ls[d * 9 + c * 3 + j] : make_double2(0.0, 0.0);
      digit_words<4>(fixed_f64(v.x, e), fixed_f64(v.y, e), w);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int wi = 3 * en + k;
        rec[warp][((wi >> 1) * 12 + li) * 2 + (wi & 1)] = w[k];
      }
      rec[warp][REC_DIG / 4 + ((en >> 1) * 12 + li) * 2 + (en & 1)] = w[3];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const uint32_t b = w[t >> 1] >> (16 * (t & 1));
        const int re = (int)(b & 255u) - 128, im = (int)((b >> 8) & 255u) - 128;
        sum[t][0] += re - im;  // column (c, re): Re, -Im
        sum[t][1] += re + im;  // column (c, im): Im, Re
      }
    }
  if (c < 3)
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      atomicAdd(&sums[warp][c][t][0], sum[t][0]);
      atomicAdd(&sums[warp][c][t][1], sum[t][1]);
    }
  __syncwarp();
  const long long ps = (long long)p * g.Vh + site;
  uint32_t* om = reinterpret_cast<uint32_t*>(main + ps * REC_MAIN);
  for (int i = lane; i < REC_DIG / 4; i += 32) om[i] = rec[warp][i];
  uint32_t* ox = reinterpret_cast<uint32_t*>(extra + ps * REC_EXTRA);
  for (int i = lane; i < REC_EXTRA / 4; i += 32) ox[i] = rec[warp][REC_DIG / 4 + i];
  float* oi = reinterpret_cast<float*>(main + ps * REC_MAIN + REC_DIG);
  for (int i = lane; i < 48; i += 32) {
    const int cc = i / 16, u = (i / 2) & 7, part = i & 1;
    int tot = 0;
    for (int t = 0; t <= u; ++t) tot += sums[warp][cc][t][part];
    oi[i] = -1.490116119384765625e-08f * (float)tot;  // 128 * 2^-24 * 2^-9 = 2^-26
  }
  if (lane < 6) {  // double-float's D_6: the kept products only
    int tot = 0;
    for (int t = 0; t < 6; ++t)
      if (keep<6>(6 - t, t)) tot += sums[warp][lane / 2][t][lane & 1];
    oi[48 + lane] = -1.490116119384765625e-08f * (float)tot;
  }
  if (lane == 0) reinterpret_cast<int*>(oi)[54] = e;
}

}  // namespace fx

size_t fx_links_bytes(const Geom& g) {
  return 256 + 2ull * g.Vh * (fx::REC_MAIN + fx::REC_EXTRA);
}

// widths the digit stencil takes: at N = 1 the kinds' own kernels are faster
// (15 of 16 MMA rows would be padding)
bool fx_width(int N) { return N >= 2 && N <= 64; }

size_t fx_digit_bytes(const Geom& g, int N) {
  if (!fx_width(N)) return 0;
  return (size_t)g.Vh * (N <= 8 ? fx::Rec<4, 1>::BYTES : (N + 15) / 16 * fx::Rec<4, 2>::BYTES);
}

bool dslash_fx_supported(const Geom& g, int N) {
  return g.fx_ctl != nullptr && g.fx_links != nullptr && fx_width(N);
}

cudaError_t fx_pack_links(const void* links_f64, void* storage, const Geom& g, cudaStream_t s) {
  const fx::Links l = fx::links_of(storage, g);
  cudaError_t e = cudaMemsetAsync(storage, 0, 256, s);
  if (e != cudaSuccess) return e;
  fx::k_fx_pack<<<2 * ((g.Vh + 7) / 8), 256, 0, s>>>(
      (const double2*)links_f64, (unsigned char*)l.main, (unsigned char*)l.extra,
      (unsigned*)l.bad, g);
  return cudaGetLastError();
}

}  // namespace bcg
