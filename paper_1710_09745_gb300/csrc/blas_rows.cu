// Tensor-core form of the fused blockCGrQ update (Algorithm 1: Q = W S^-1,
// X += P (beta C), P = Q + P S^dag; the streaming multi-BLAS of Sec. 6.3) and of
// the W update W = Q - AP beta, for the double-float and the FP32 kind, N <= 32.
//
// On the FP32 pipes a double-float multiply-add costs 12 instructions, and the
// FP32 kernel is bound by its reads of staged rows and coefficients.  Here the
// N x N products run as exact split products on the bf16 tensor cores
// (ozaki.cuh): each row of W and P is scaled by a power of two (its largest
// entry, from the four threads that hold the row) and split into bf16 slices,
// six or seven for double-float and four (32 bits) for FP32; each coefficient
// column likewise (its largest entry in the matrix's triangular pattern).  For an
// output (row r, column j) the products W_s[r][k] M_t[k][j] with s + t = u are
// accumulated in one FP32 accumulator D_u: they share the grid
// 2^(er + ej - 14 - 8u), and 2N x (u + 1) terms of at most 2^14.6 units stay below
// 2^24, so the accumulation is exact.  Kept are the products with s + t below
// the number of slices; the epilogue adds the leading sums exactly.
//
// A warp owns 16 rows.  The A fragments of a thread are the complex numbers
// 8 ks + 2 t and + 1 of its rows ra, rb (k order permuted consistently in A and
// B), so the slices are made in the registers that feed the MMA: earlier, when
// they went through shared memory and were read again for every output tile,
// the L1 data pipe was at 71 % and the tensor pipe at 42 %.  Where there is room
// the slices of W and P are held together, so an output tile takes all its
// products in turn and Q need not be read back.
// The B fragments of all slices of the matrices are built once per CTA in
// shared memory in fragment order.  NP: N rounded up to 8, 16 or 32; columns
// past N are zeros.
//
// Bound by the tensor pipe (mma.sync) together with the splitting at N = 16, by
// HBM at N <= 8.  32^4, double-float, N = 16 (1.6 M rows): update 738 -> 638 us,
// W 271 -> 257; 16^4, N = 8: update 40 (CUDA cores) -> 30; FP32 at 24^4, N = 32:
// update 490 (CUDA cores) -> 325, W and Gram 318 (one kernel) -> 130 + 131.
// Relative error of the updated blocks against 64 bits, columns of like norms:
// double-float 1.4e-15 with 28 products (CUDA cores 3.1e-15 at N = 3 to 1.1e-14
// at N = 32), 3.3e-14 with the 21 that N = 16 always had here; FP32 2.5e-8 (CUDA
// cores 3.7e-8 to 1.0e-7).  A row's scale is its largest entry, so a column k
// times shorter than the longest is held in log2 k fewer bits, where the CUDA
// cores hold each entry in all of its own.  The norms of the right-hand sides do
// not enter W and P.  P's columns differ around peaks of the residual: replayed
// in 64 bits, FP32 solves at 8^4 with m = 0.02 to 0.001 and N = 5 to 32 have
// ratios up to 90 and P S^dag 5 to 80 times closer than on the CUDA cores; at
// m = 1e-4 the ratio reaches 530, and the worst iteration is level with them.  Which form a problem takes is timed by the BLAS tuner: at N = 12 and
// below the fused CUDA-core W + Gram usually stays ahead of two launches.
#include <type_traits>

#include "internal.h"
#include "ozaki.cuh"

namespace bcg {

using namespace ozaki;

namespace {

// coefficient entry (i, j) of matrix m in its triangular pattern: 0 = S^-1
// (upper), 1 = beta C (full), 2 = S^dag (lower)
__device__ __forceinline__ bool rt_in_pattern(int m, int i, int j) {
  return m == 1 || (m == 0 ? i <= j : i >= j);
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p));
}

// slices, kept products (s + t < NU) and their sum by storage kind
struct KindDF : SliceKind<StoreDF> {  // six slices, 21 products
  using Store = StoreDF;
  using In = float4;  // an entry of the rows that are multiplied
  static __device__ __forceinline__ In in_zero() { return zero(); }
  static constexpr int NU = 6;
  static __device__ __forceinline__ dfacc sum(const float (&a)[NU][4], int i) {
    float h = a[0][i], l = __fadd_rn(a[5][i], a[4][i]);
    exact_add(h, l, a[1][i]);
    exact_add(h, l, a[2][i]);
    exact_add(h, l, a[3][i]);
    return {h, l};
  }
};
struct KindF64 : KindDF {  // the same of FP64 rows (QROWS), scaled before they are rounded
  using In = double2;
  static __device__ __forceinline__ In in_zero() { return make_double2(0.0, 0.0); }
};
struct KindDF7 : SliceKind<StoreDF> {  // seven slices, 28 products
  using Store = StoreDF;
  using In = float4;
  static __device__ __forceinline__ In in_zero() { return zero(); }
  static constexpr int NSL = 7, NU = 7;
  static __device__ __forceinline__ void slices(float4 v, float sc, uint32_t (&w)[NSL]) {
    float re[7], im[7];
    split7(__fmul_rn(v.x, sc), __fmul_rn(v.z, sc), re);
    split7(__fmul_rn(v.y, sc), __fmul_rn(v.w, sc), im);
#pragma unroll
    for (int s = 0; s < NSL; ++s) w[s] = pack_bf16(re[s], im[s]);
  }
  static __device__ __forceinline__ dfacc sum(const float (&a)[NU][4], int i) {
    float h = a[0][i], l = __fadd_rn(__fadd_rn(a[6][i], a[5][i]), a[4][i]);
    exact_add(h, l, a[1][i]);
    exact_add(h, l, a[2][i]);
    exact_add(h, l, a[3][i]);
    return {h, l};
  }
};
struct KindF32 : SliceKind<StoreF32> {  // four slices, 10 products
  using Store = StoreF32;
  using In = float2;
  static __device__ __forceinline__ In in_zero() { return zero(); }
  static constexpr int NU = 4;
  static __device__ __forceinline__ dfacc sum(const float (&a)[NU][4], int i) {
    float h = a[0][i], l = __fadd_rn(a[3][i], a[2][i]);
    exact_add(h, l, a[1][i]);
    return {h, l};
  }
};

// what a launch computes (the matrix passed as Sinv but in UPDATE)
enum RowsMode {
  UPDATE,  // Q = W S^-1 (W in Q), X += P (beta C), P = Q + P S^dag
  WROWS,   // Q = Q - P beta
  QROWS,   // Q = P C, C upper triangular; Q in FP32, P in the kind's In; BC = P^dag P
  PROWS,   // P = Q + P S
};

// x 2^e for a result below 2^1023 (smaller than a normal number: zero), on the
// integer pipe
__device__ __forceinline__ double times_pow2(double x, int e) {
  const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
  if (ex == 0x7ff) return x;
  return ex == 0 || ex + e <= 0 ? 0.0 : __hiloint2double(hi + e * (1 << 20), __double2loint(x));
}

template <class K, int NP, int MODE>
struct RtGeom {
  static constexpr int KS = NP / 8;  // k steps of 16 reals (8 complex numbers)
  static constexpr int NT = NP / 4;  // output tiles of 8 reals (4 complex columns)
  static constexpr int NM = MODE != UPDATE ? 1 : 3;
  static constexpr int FR = KS * NT * 32;
  static constexpr size_t smem = (size_t)NM * K::NSL * FR * sizeof(uint2);
  // warps per SM: 12 of up to 168 registers in one CTA; 16 of 128 where the
  // slices leave room (24^4, FP32, N = 32 update: 325 us against 349; 32^4,
  // double-float, N = 16: 640 against 690, and as two CTAs, which start up apart)
  static constexpr int threads =
      std::is_same<K, KindF32>::value && NP == 32 ? 512 : std::is_base_of<KindDF, K>::value && NP == 16 ? 256 : 384;
  static constexpr int ctas = threads == 256 ? 2 : 1;
  // the slices of W and P together: where they leave room (double-float, N = 16:
  // 830 us together, 682 in turn; N = 8 30 against 32, FP32 N = 16 40 against 44)
  static constexpr bool both = MODE == UPDATE && (NP == 8 || (NP == 16 && std::is_same<K, KindF32>::value));
};

}  // namespace

template <class K, int NP, int MODE>
__global__ void __launch_bounds__((RtGeom<K, NP, MODE>::threads), (RtGeom<K, NP, MODE>::ctas))
    k_rows_tc(std::conditional_t<MODE == QROWS, float2, typename K::Store::elem>* __restrict__ Q,
              typename K::In* __restrict__ P, float4* __restrict__ X, const double2* __restrict__ Sinv,
              const double2* __restrict__ BC, const double2* __restrict__ SH, int N, int Vh,
              unsigned* __restrict__ pmax, Gate gate) {
  using S = typename K::Store;
  using G = RtGeom<K, NP, MODE>;
  using E = typename S::elem;
  using In = typename K::In;
  constexpr bool WMODE = MODE != UPDATE;  // one matrix
  constexpr bool DF = std::is_same<S, StoreDF>::value;
  constexpr int KS = G::KS, NT = G::NT, NM = G::NM, FR = G::FR, NSL = K::NSL, NU = K::NU;
  constexpr bool BOTH = G::both;
  constexpr int RT_THREADS = G::threads, RT_WARPS = RT_THREADS / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint2* sB = reinterpret_cast<uint2*>(smem_raw);
  __shared__ int sE[3 * NP];  // column exponents: |column| < 2^e
  __shared__ unsigned sM[NP];  // column maxima of the new P
  // QROWS: exponents of the norms of P's columns.  The columns are multiplied by
  // 2^-k and the rows of C by 2^k, or a column far shorter than its neighbours
  // would lose bits to the scale of its rows (norms of 1 to 1e-12 at 16^4, N = 8:
  // 195 iterations for 154)
  __shared__ int sK[NP];
  if (gate_closed(gate)) return;
  const bool keepP = gate.st != nullptr && ((const volatile SolverStatus*)gate.st)->ru_pending;
  auto Ms = [&](int m) { return m == 0 ? Sinv : m == 1 ? BC : SH; };
  auto in_pattern = [&](int m, int i, int j) {
    return i < N && j < N && (MODE == WROWS || MODE == PROWS || rt_in_pattern(m, i, j));
  };
  if (threadIdx.x < NP) sM[threadIdx.x] = 0u;
  if constexpr (MODE == QROWS) {
    if (threadIdx.x < NP) {
      const int j = threadIdx.x;
      const int ex = j < N ? (__double2hiint(BC[j * N + j].x) >> 20) & 0x7ff : 0;
      constexpr int KMAX = std::is_same<In, double2>::value ? 512 : 100;
      sK[j] = ex == 0 || ex == 0x7ff ? 0 : min(max((ex - 1023) >> 1, -KMAX), KMAX);
    }
    __syncthreads();
  }
  for (int c = threadIdx.x; c < NM * NP; c += RT_THREADS) {
    const int m = c / NP, j = c - m * NP;
    double mx = 0.0;
    for (int i = 0; i < N; ++i) {
      if (!in_pattern(m, i, j)) continue;
      const double2 v = Ms(m)[i * N + j];
      const double a = fmax(fabs(v.x), fabs(v.y));
      mx = fmax(mx, MODE == QROWS ? ldexp(a, sK[i]) : a);
    }
    int e = 0;
    if (mx > 0.0 && mx < 1e300) frexp(mx, &e);  // mx in [2^(e-1), 2^e)
    constexpr int EMAX = MODE == QROWS ? 1000 : 120;
    sE[c] = e < -EMAX ? -EMAX : e > EMAX ? EMAX : e;
  }
  __syncthreads();
  // B fragments: k step ks, lane (g, t): b.x holds rows (re, im) of input
  // i0 = 8 ks + 2 t, b.y those of i0 + 1; column n = 8 nt + g, complex column
  // n / 2, real part when n is even
  for (int idx = threadIdx.x; idx < NM * FR; idx += RT_THREADS) {
    const int m = idx / FR;
    int r = idx - m * FR;
    const int ks = r / (NT * 32);
    r -= ks * NT * 32;
    const int nt = r / 32, lane = r - nt * 32;
    const int i0 = 8 * ks + 2 * (lane & 3), n = 8 * nt + (lane >> 2), j = n >> 1, part = n & 1;
    uint32_t w[2][NSL];
    for (int q = 0; q < 2; ++q) {
      double re = 0.0, im = 0.0;
      if (in_pattern(m, i0 + q, j)) {
        const double2 v = Ms(m)[(i0 + q) * N + j];
        if constexpr (MODE == QROWS) {
          re = ldexp(v.x, sK[i0 + q] - sE[j]);
          im = ldexp(v.y, sK[i0 + q] - sE[j]);
        } else {
          const double sc = ldexp(1.0, -sE[m * NP + j]);
          re = v.x * sc;
          im = v.y * sc;
        }
      }
      // rows (re, im) of column (c, re): Re, -Im; of (c, im): Im, Re
      float4 z = StoreDF::from_double2(part ? make_double2(im, re) : make_double2(re, -im));
      if constexpr (DF)
        K::slices(z, 1.f, w[q]);
      else
        K::slices(make_float2(z.x, z.y), 1.f, w[q]);
    }
    for (int s = 0; s < NSL; ++s)
      sB[((m * NSL + s) * KS + ks) * NT * 32 + nt * 32 + lane] = make_uint2(w[0][s], w[1][s]);
  }
  __syncthreads();

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const bool pairs = std::is_same<S, StoreF32>::value && (N & 1) == 0;  // 128-bit loads
  const long long nrows = 3LL * Vh;
  const long long ntiles = (nrows + 15) / 16;
  const long long stride = (long long)gridDim.x * RT_WARPS;
  unsigned pm[NT];  // maxima of columns 4 nt + t (BOTH)
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) pm[nt] = 0u;
  for (long long tile = (long long)blockIdx.x * RT_WARPS + warp; tile < ntiles; tile += stride) {
    const long long ra = tile * 16 + g, rb = ra + 8;
    const bool va = ra < nrows, vb = rb < nrows;
    auto prefetch = [&](const In* f, long long r) {
      if (r < nrows && 4 * t < N) prefetch_l2(f + r * N + 4 * t);
    };
    prefetch(P, ra + 16 * stride);
    prefetch(P, rb + 16 * stride);
    if constexpr (!WMODE) {
      prefetch((const In*)Q, ra + 16 * stride);
      prefetch((const In*)Q, rb + 16 * stride);
    }
    // this thread's entries of rows ra, rb: v[ks][0..3] = (ra, c0), (rb, c0),
    // (ra, c0 + 1), (rb, c0 + 1), c0 = 8 ks + 2 t
    auto load = [&](const In* src, In (&v)[KS][4]) {
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        const int c0 = 8 * ks + 2 * t;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const bool ok = h ? vb : va;
          const In* p = src + (h ? rb : ra) * N + c0;
          v[ks][h] = v[ks][2 + h] = K::in_zero();
          if constexpr (std::is_same<S, StoreF32>::value) {
            if (pairs) {
              if (ok && c0 < N) {
                const float4 z = *reinterpret_cast<const float4*>(p);
                v[ks][h] = make_float2(z.x, z.y);
                v[ks][2 + h] = make_float2(z.z, z.w);
              }
              continue;
            }
          }
          if (ok && c0 < N) v[ks][h] = p[0];
          if (ok && c0 + 1 < N) v[ks][2 + h] = p[1];
        }
      }
    };
    // A fragments of all slices, and the row exponents (the four threads t of
    // a row hold its N entries)
    auto split = [&](const In (&v)[KS][4], uint32_t (&a)[KS][NSL][4], int (&er)[2]) {
      if constexpr (std::is_same<In, double2>::value) {
        int mx[2] = {0, 0};  // high words, columns scaled
        auto high = [](double x, int k) {
          const int h = __double2hiint(x) & 0x7fffffff;
          return h < (1 << 20) ? 0 : h - k * (1 << 20);
        };
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int k = sK[8 * ks + 2 * t + (i >> 1)];
            mx[i & 1] = max(mx[i & 1], max(high(v[ks][i].x, k), high(v[ks][i].y, k)));
          }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          mx[h] = max(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 1));
          mx[h] = max(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 2));
          er[h] = min(max((mx[h] >> 20) - 1022, -1000), 1000);  // |row| < 2^er
        }
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int e = -sK[8 * ks + 2 * t + (i >> 1)] - er[i & 1];
            const double2 z = make_double2(times_pow2(v[ks][i].x, e), times_pow2(v[ks][i].y, e));
            uint32_t w[NSL];
            K::slices(StoreDF::from_double2(z), 1.f, w);
#pragma unroll
            for (int s = 0; s < NSL; ++s) a[ks][s][i] = w[s];
          }
      } else {
        float mx[2] = {0.f, 0.f};
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
          for (int i = 0; i < 4; ++i) mx[i & 1] = fmaxf(mx[i & 1], K::mag(v[ks][i]));
        float sc[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 1));
          mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 2));
          er[h] = pow2_above(__float_as_uint(mx[h]));
          sc[h] = exp2i(-er[h]);
        }
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            uint32_t w[NSL];
            K::slices(v[ks][i], sc[i & 1], w);
#pragma unroll
            for (int s = 0; s < NSL; ++s) a[ks][s][i] = w[s];
          }
      }
    };
    // rows times coefficient matrix m, output tile nt; k steps kf .. kl
    auto product = [&](int m, int nt, const uint32_t (&a)[KS][NSL][4], float (&acc)[NU][4], int kf,
                       int kl) {
#pragma unroll
      for (int u = 0; u < NU; ++u)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[u][i] = 0.f;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        if (ks < kf || ks > kl) continue;
#pragma unroll
        for (int tt = 0; tt < NSL; ++tt) {
          const uint2 b = sB[((m * NSL + tt) * KS + ks) * NT * 32 + nt * 32 + lane];
#pragma unroll
          for (int s = 0; s < NSL; ++s)
            if (s + tt < NU) mma_bf16(acc[s + tt], a[ks][s], b.x, b.y);
        }
      }
    };
    // (re, im) of output (row h, complex column 4 nt + t)
    auto value = [&](const float (&acc)[NU][4], int h, int er, int ej) {
      if constexpr (MODE == QROWS) {  // the exponents may be large and of opposite sign
        const int e = min(max(er + ej, -240), 240);
        er = e / 2;
        ej = e - er;
      }
      const float fa = exp2i(er), fb = exp2i(ej);
      cpx<dfacc> v{K::sum(acc, 2 * h), K::sum(acc, 2 * h + 1)};
      v.re = {__fmul_rn(__fmul_rn(v.re.s, fa), fb), __fmul_rn(__fmul_rn(v.re.e, fa), fb)};
      v.im = {__fmul_rn(__fmul_rn(v.im.s, fa), fb), __fmul_rn(__fmul_rn(v.im.e, fa), fb)};
      return cfin<CompDF>(v);
    };
    auto as_df = [&](const E& z) {
      if constexpr (DF)
        return cpx<df>{{z.x, z.z}, {z.y, z.w}};
      else
        return cpx<df>{{z.x, 0.f}, {z.y, 0.f}};
    };
    auto put = [&](E* p, const cpx<df>& v) {
      if constexpr (DF)
        *p = make_float4(v.re.hi, v.im.hi, v.re.lo, v.im.lo);
      else
        *p = make_float2(v.re.hi, v.im.hi);  // hi: the value rounded to FP32
    };
    auto plus = [&](const cpx<df>& a, const cpx<df>& b, float sign) {
      cpx<dfacc> s = cacc_from<CompDF>(a);
      CompDF::add(s.re, df{sign * b.re.hi, sign * b.re.lo});
      CompDF::add(s.im, df{sign * b.im.hi, sign * b.im.lo});
      return cfin<CompDF>(s);
    };
    // a new entry of P's column j: its larger component's bits
    auto track = [&](unsigned& m, const cpx<df>& v) {
      m = max(m, max(__float_as_uint(v.re.hi) & 0x7fffffffu, __float_as_uint(v.im.hi) & 0x7fffffffu));
    };
    // k steps holding an input i with a nonzero coefficient for output tile
    // nt: S^-1 upper (i <= the tile's last column), S^dag lower (i >= its first)
    auto k_last_upper = [](int nt) { return (4 * nt + 3) / 8; };
    auto k_first_lower = [](int nt) { return 4 * nt / 8; };
    float acc[NU][4];
    if constexpr (WMODE) {
      uint32_t a[KS][NSL][4];
      int er[2];
      {
        In v[KS][4];
        load(P, v);
        if constexpr (MODE == QROWS && std::is_same<In, float4>::value) {
#pragma unroll
          for (int ks = 0; ks < KS; ++ks)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float f = exp2i(-sK[8 * ks + 2 * t + (i >> 1)]);
              float4& z = v[ks][i];
              z = make_float4(__fmul_rn(z.x, f), __fmul_rn(z.y, f), __fmul_rn(z.z, f), __fmul_rn(z.w, f));
            }
        }
        split(v, a, er);
      }
#pragma unroll(NP <= 16 ? NT : 1)
      for (int nt = 0; nt < NT; ++nt) {
        const int j = 4 * nt + t;
        E q[2];
        if constexpr (MODE != QROWS) {
#pragma unroll
          for (int h = 0; h < 2; ++h)
            q[h] = (h ? vb : va) && j < N ? Q[(h ? rb : ra) * N + j] : K::zero();
        }
        product(0, nt, a, acc, 0, MODE == QROWS ? k_last_upper(nt) : KS - 1);
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if ((h ? vb : va) && j < N) {
            const long long o = (h ? rb : ra) * N + j;
            const cpx<df> v = value(acc, h, er[h], sE[j]);
            if constexpr (MODE == WROWS)
              put(Q + o, plus(as_df(q[h]), v, -1.f));
            else if constexpr (MODE == PROWS)
              put(P + o, plus(as_df(q[h]), v, 1.f));
            else
              Q[o] = make_float2(v.re.hi, v.im.hi);
          }
      }
    } else if constexpr (BOTH) {
      uint32_t aw[KS][NSL][4], ap[KS][NSL][4];
      int ew[2], ep[2];
      {
        E v[KS][4], w[KS][4];
        load(Q, v);
        load(P, w);
        split(v, aw, ew);
        split(w, ap, ep);
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        const int j = 4 * nt + t;
        float4 x[2];
#pragma unroll
        for (int h = 0; h < 2; ++h)
          x[h] = (h ? vb : va) && j < N ? X[(h ? rb : ra) * N + j] : make_float4(0.f, 0.f, 0.f, 0.f);
        cpx<df> q[2];
        product(0, nt, aw, acc, 0, k_last_upper(nt));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          q[h] = value(acc, h, ew[h], sE[j]);
          if ((h ? vb : va) && j < N) put(Q + (h ? rb : ra) * N + j, q[h]);
        }
        if (!keepP) {
          product(2, nt, ap, acc, k_first_lower(nt), KS - 1);
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if ((h ? vb : va) && j < N) {
              const cpx<df> p = plus(q[h], value(acc, h, ep[h], sE[2 * NP + j]), 1.f);
              put(P + (h ? rb : ra) * N + j, p);
              track(pm[nt], p);
            }
        }
        product(1, nt, ap, acc, 0, KS - 1);
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if ((h ? vb : va) && j < N) {
            const cpx<df> s = plus(cpx<df>{{x[h].x, x[h].z}, {x[h].y, x[h].w}},
                                   value(acc, h, ep[h], sE[NP + j]), 1.f);
            X[(h ? rb : ra) * N + j] = make_float4(s.re.hi, s.im.hi, s.re.lo, s.im.lo);
          }
      }
    } else {
      uint32_t a[KS][NSL][4];
      int er[2];
      {
        E v[KS][4];
        load(Q, v);
        split(v, a, er);
      }
#pragma unroll 1
      for (int nt = 0; nt < NT; ++nt) {
        const int j = 4 * nt + t;
        product(0, nt, a, acc, 0, k_last_upper(nt));
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if ((h ? vb : va) && j < N)
            put(Q + (h ? rb : ra) * N + j, value(acc, h, er[h], sE[j]));
      }
      {
        E v[KS][4];
        load(P, v);
        split(v, a, er);
      }
      __syncwarp();  // the rows of P are read before they are replaced
#pragma unroll 1
      for (int nt = 0; nt < NT; ++nt) {
        const int j = 4 * nt + t;
        float4 x[2];
        E q[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const bool ok = (h ? vb : va) && j < N;
          x[h] = ok ? X[(h ? rb : ra) * N + j] : make_float4(0.f, 0.f, 0.f, 0.f);
          q[h] = ok ? Q[(h ? rb : ra) * N + j] : K::zero();  // this thread wrote it
        }
        if (!keepP) {
          product(2, nt, a, acc, k_first_lower(nt), KS - 1);
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if ((h ? vb : va) && j < N) {
              const cpx<df> p = plus(as_df(q[h]), value(acc, h, er[h], sE[2 * NP + j]), 1.f);
              put(P + (h ? rb : ra) * N + j, p);
              unsigned m = 0u;
              track(m, p);
              if (pmax) atomicMax(&sM[j], m);
            }
        }
        product(1, nt, a, acc, 0, KS - 1);
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if ((h ? vb : va) && j < N) {
            const cpx<df> s = plus(cpx<df>{{x[h].x, x[h].z}, {x[h].y, x[h].w}},
                                   value(acc, h, er[h], sE[NP + j]), 1.f);
            X[(h ? rb : ra) * N + j] = make_float4(s.re.hi, s.im.hi, s.re.lo, s.im.lo);
          }
      }
    }
    __syncwarp();
  }
  if (!WMODE && pmax && !keepP) {
    if constexpr (BOTH)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) atomicMax(&sM[4 * nt + t], pm[nt]);
    __syncthreads();
    if (threadIdx.x < N) atomicMax(pmax + threadIdx.x, sM[threadIdx.x]);
  }
}

bool rows_tc_supported(FieldKind k, int N) {
  return (k == FK_DF || k == FK_F32) && N >= 3 && N <= 32;
}

template <class K, int NP, int MODE>
static cudaError_t launch_rows(void* Q, void* P, void* X, const double2* Sinv, const double2* BC,
                               const double2* SH, int N, int Vh, unsigned* pmax, Gate gate,
                               cudaStream_t s) {
  using G = RtGeom<K, NP, MODE>;
  constexpr size_t sm = G::smem;
  constexpr int RT_THREADS = G::threads, RT_WARPS = RT_THREADS / 32;
  auto kern = k_rows_tc<K, NP, MODE>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    cudaGetLastError();
  const long long tiles = (3LL * Vh + 15) / 16;
  long long blocks = (tiles + RT_WARPS - 1) / RT_WARPS;
  if (blocks > (long long)sms * G::ctas) blocks = (long long)sms * G::ctas;
  using QE = std::conditional_t<MODE == QROWS, float2, typename K::Store::elem>;
  kern<<<(unsigned)blocks, RT_THREADS, sm, s>>>((QE*)Q, (typename K::In*)P, (float4*)X, Sinv, BC, SH, N, Vh, pmax,
                                             gate);
  return cudaGetLastError();
}

// Double-float at N = 16 (and the W update at N = 32) has six slices, as long as
// it has run on the tensor cores (error 3.3e-14 of the product's norm); the
// other widths, which ran in the CUDA cores' double-float (3.1e-15 at N = 3 to
// 1.1e-14 at N = 32), get the seventh.  FP32: 2.5e-8, the CUDA cores 3.7e-8 to 1.0e-7.
template <class K, int MODE>
static cudaError_t launch_rows_n(void* Q, void* P, void* X, const double2* Sinv, const double2* BC,
                                 const double2* SH, int N, int Vh, unsigned* pmax, Gate gate,
                                 cudaStream_t s) {
  if (N <= 8) return launch_rows<K, 8, MODE>(Q, P, X, Sinv, BC, SH, N, Vh, pmax, gate, s);
  if (N <= 16) return launch_rows<K, 16, MODE>(Q, P, X, Sinv, BC, SH, N, Vh, pmax, gate, s);
  return launch_rows<K, 32, MODE>(Q, P, X, Sinv, BC, SH, N, Vh, pmax, gate, s);
}

cudaError_t bcg_update_rows(FieldKind k, void* Q, void* P, void* X, const double2* Sinv,
                            const double2* BC, const double2* SH, int N, int Vh, unsigned* pmax,
                            Gate gate, cudaStream_t s) {
  if (!rows_tc_supported(k, N)) return cudaErrorInvalidValue;
  if (k == FK_F32)
    return launch_rows_n<KindF32, UPDATE>(Q, P, X, Sinv, BC, SH, N, Vh, nullptr, gate, s);
  if (N == 16) return launch_rows<KindDF, 16, UPDATE>(Q, P, X, Sinv, BC, SH, N, Vh, pmax, gate, s);
  return launch_rows_n<KindDF7, UPDATE>(Q, P, X, Sinv, BC, SH, N, Vh, pmax, gate, s);
}

cudaError_t w_update_rows(FieldKind k, void* Q, const void* AP, const double2* beta, int N, int Vh,
                          Gate gate, cudaStream_t s) {
  if (!rows_tc_supported(k, N)) return cudaErrorInvalidValue;
  void* A = const_cast<void*>(AP);
  if (k == FK_F32)
    return launch_rows_n<KindF32, WROWS>(Q, A, nullptr, beta, nullptr, nullptr, N, Vh, nullptr, gate, s);
  if (N == 16)
    return launch_rows<KindDF, 16, WROWS>(Q, A, nullptr, beta, nullptr, nullptr, N, Vh, nullptr, gate, s);
  if (N == 32)
    return launch_rows<KindDF, 32, WROWS>(Q, A, nullptr, beta, nullptr, nullptr, N, Vh, nullptr, gate, s);
  return launch_rows_n<KindDF7, WROWS>(Q, A, nullptr, beta, nullptr, nullptr, N, Vh, nullptr, gate, s);
}

// Q and P of a reliable update with an FP32 iteration, in two launches (Q is
// stored in FP32, so reading it back loses nothing): Q = R C^-1 with the 21
// products of R's double-float slices (error 4e-14, then rounded to FP32; the
// columns of R brought to norms of 1 to 2 first, sK), and P = Q + P S with
// FP32's ten.  On the CUDA cores (k_restart_update) it is bound
// by the FP64 rate: 24^4, N = 32 (FP64 R) 3477 us, here 385; error of Q 2.5e-8
// either way, of P 3.6e-8 here and 9.0e-8 (N = 8) to 1.7e-7 (N = 32) there.
// The line: both launches build their coefficient fragments first, and narrow
// blocks waste lanes, so small ones stay there (N = 8: V_h = 10368 19 us against
// 20 here, V_h = 32768 39 against 27; N = 4, V_h = 32768: 15 against 37; N = 16,
// V_h = 10368: 70 against 30).
bool restart_rows_supported(FieldKind rk, FieldKind sk, int N, int Vh) {
  return (rk == FK_F64 || rk == FK_DF) && sk == FK_F32 && N >= 8 && rows_tc_supported(sk, N) &&
         (long long)Vh * N * N >= 1 << 21;
}

cudaError_t restart_rows(FieldKind rk, const void* R, const double2* G, void* Q, void* P,
                         const double2* Cinv, const double2* SH, int init, int N, int Vh,
                         Gate gate, cudaStream_t s) {
  void* r = const_cast<void*>(R);
  cudaError_t e =
      rk == FK_F64
          ? launch_rows_n<KindF64, QROWS>(Q, r, nullptr, Cinv, G, nullptr, N, Vh, nullptr, gate, s)
          : launch_rows_n<KindDF, QROWS>(Q, r, nullptr, Cinv, G, nullptr, N, Vh, nullptr, gate, s);
  if (e != cudaSuccess) return e;
  if (init)  // P = Q
    return rk == FK_F64
               ? launch_rows_n<KindF64, QROWS>(P, r, nullptr, Cinv, G, nullptr, N, Vh, nullptr, gate, s)
               : launch_rows_n<KindDF, QROWS>(P, r, nullptr, Cinv, G, nullptr, N, Vh, nullptr, gate, s);
  return launch_rows_n<KindF32, PROWS>(Q, P, nullptr, SH, nullptr, nullptr, N, Vh, nullptr, gate, s);
}

}  // namespace bcg
