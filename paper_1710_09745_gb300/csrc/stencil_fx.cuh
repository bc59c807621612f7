// Tensor-core stencil of the 48-bit and 64-bit kinds: the hopping term of
// Eq. 2 for a block of N right-hand sides (Sec. 6.2: every link read once per
// site and applied to all N spinors) as exact products of 8-bit digits.
//
// Per output site the stencil is a small dense product: with the 16 hops and
// 3 colours as a K index of 48 complex (96 real) entries,
//     out^T (N x 3 complex) = Psi^T (N x 48) U^T (48 x 3),
// Psi the gathered neighbour spinors and U the site's 16 hop matrices; in
// real form D[n][o] = sum_k A[n][k] B[k][o] with n = right-hand side (16 rows
// of mma.sync m16n8k16), k = (hop, colour, re/im) and o = (colour, re/im) (6
// of 8 columns).  B differs for every site, so the warp-level form fits: one
// warp computes one site and up to 16 right-hand sides.
//
// Digits.  The input block is written once per half as fixed-point numbers
// with one power-of-two scale 2^e per right-hand side (from its column
// maximum, |v| <= 0.995 2^e): ND = 6 signed base-256 digits (48 bits) for the
// double-float kind, ND = 8 (64 bits) for native FP64; the links likewise with
// one scale per site, once per gauge field.  A stored digit is the byte
// b = digit + 128, and a byte zero-extended to 16 bits is the FP16 subnormal
// b 2^-24: a PRMT turns four gathered bytes into an MMA operand register, so
// a gathered complex number costs ND instructions (splitting the
// floating-point value where it is gathered cost 42, sixteen times per
// value, and bound the kernel by instruction issue).  The offset 128 of the A
// bytes is removed by the accumulator's initial value -128 sum_k B[k][o]
// (a per-site constant, packed with the links); B is made signed in registers.
// The products of digits s and t with s + t = u <= ND - 1 share one
// accumulator D_u; in units of the product of the digits' grids every partial
// sum stays below 128 * 128 * 96 * ND < 2^24, so the FP32 accumulation is
// exact.  The epilogue adds D_0 .. D_{ND-1} in double-float (ND = 6) or as
// 64-bit integers (ND = 8, rounded once to FP64) and removes the scales.
// Error per term: half a unit of the last digit of either factor, 2^-48
// (2^-64) of 2^e, and the dropped products s + t >= ND, of that order.
//
// A block for which one scale per column will not do, or links for which one
// scale per site will not, set a flag: the kernel then computes the half in the
// kind's own arithmetic (fx_cores).  Links: an entry outside 2^-90 .. 2^90, or a
// nonzero hop matrix whose largest entry is less than 2^-9 (double-float 1/96) of
// the site's: a site whose other neighbours are zero has only that matrix to add
// up (double-float, 1/360: 3.5e-12; HISQ's three-link term is 1/24).  Blocks: a non-finite or huge entry; in FP64 a
// nonzero site vector more than 2^9 below its column's maximum, which native
// FP64 would still resolve to 53 bits; in double-float a run of 8 to 32 sites
// (a step of k_fx_digits) in which a nonzero column stays more than 2^3 below
// its maximum, so that 45 of the 48 bits are left of each run's largest entry:
// what double-float sums keep (3.0e-14 of the result here, digits on Gaussian
// columns 1.9e-14; without the rule a column that falls as e^-2t lost all but
// 8 digits in its far slices).  In whole solves with Gaussian sources the
// maxima of the runs stay within a factor of 4 of the column's (4^4 to 16^4,
// every iteration); with point sources the first fifth of the iterations is
// flagged, until the sources have spread.
#pragma once
#include <cuda_fp16.h>

#include "stencil_kernels.cuh"

namespace bcg {
namespace fx {

// control words in the workspace (Geom::fx_ctl): column maxima of the even
// and the odd input (bit patterns of |hi|, or the high words of |v| in FP64)
// and the flag of each that sends the half to fx_cores
constexpr int CTL_MAX = 0;     // + 64 * input parity
constexpr int CTL_FLAG = 128;  // + input parity

// packed links: per (parity, site) the digits of the 144 entries in the order
// a lane reads them, [18][12] words of 8 bytes for digits 0..5, followed by
// the accumulators' initial values [c][u][re, im], those of double-float's D_6
// [c][re, im] and the scale exponent; and apart [6][12] words for digits 6 and 7 (12 = (q, c): hop kind q of +1, -1,
// +3, -3, row colour c).  A lane's entry 2 k + h, k = 3 (mu / 2) + j, h = mu % 2,
// is the element (c, j) of its hop in direction mu.
constexpr int REC_DIG = 18 * 12 * 8;
constexpr int REC_D6 = REC_DIG + 3 * 8 * 2 * 4;
constexpr int REC_MAIN = REC_D6 + 32;
constexpr int REC_EXTRA = 6 * 12 * 8;

struct Links {
  const unsigned char *main, *extra;
  const unsigned* bad;  // [FP64, double-float]: nonzero if the field is marked
};
__host__ __device__ inline Links links_of(const void* base, const Geom& g) {
  const unsigned char* p = (const unsigned char*)base;
  const size_t n = 2ull * g.Vh;
  Links l;
  l.bad = (const unsigned*)p;
  l.main = p + 256;
  l.extra = l.main + n * REC_MAIN;
  return l;
}

// digits of one input site and R rows of 8 right-hand sides (R = 2:
// right-hand sides 16 m + gq and 16 m + gq + 8): per colour WPC words for
// each gq, W words per complex number (one row of double-float is padded to
// four words), as 16-byte chunks [gq], then an 8-byte one
template <int W, int R>
struct Rec {
  static constexpr int WPC = R == 1 ? 4 : 2 * W;
  static constexpr int COLOUR = 8 * WPC * 4;  // bytes
  static constexpr int BYTES = 3 * COLOUR;
};

// exponent e with |v| <= 0.995 2^e for the column maximum's bit pattern m
// (FP32 or the high word of FP64); 0 for a zero column
__device__ __forceinline__ int exp_f32(unsigned m) {
  return m == 0u ? 0 : (int)(m >> 23) - 126 + ((m & 0x7fffffu) > 8304721u ? 1 : 0);
}
__device__ __forceinline__ int exp_f64(unsigned m) {
  return m == 0u ? 0 : (int)(m >> 20) - 1022 + ((m & 0xfffffu) > 1038090u ? 1 : 0);
}
// the range in which the scales and every intermediate stay normal numbers
__device__ __forceinline__ bool bad_f32(unsigned m) {
  const int e = exp_f32(m);
  return m != 0u && (e < -90 || e > 90);
}
__device__ __forceinline__ bool bad_f64(unsigned m) {
  const int e = exp_f64(m);
  return m != 0u && (e < -800 || e > 800);
}
__device__ __forceinline__ float exp2f_int(int e) { return __int_as_float((e + 127) << 23); }
__device__ __forceinline__ double exp2d_int(int e) {
  return __hiloint2double((e + 1023) << 20, 0);
}

// v 2^(63 - e) rounded to an integer, for |v| <= 0.995 2^e
__device__ __forceinline__ long long fixed_f64(double v, int e) {
  const long long b = __double_as_longlong(v);
  const int ef = (int)((b >> 52) & 0x7ff);
  unsigned long long m = (unsigned long long)b & 0xfffffffffffffull;
  if (ef) m |= 0x10000000000000ull;
  const int sh = (ef ? ef : 1) - 1012 - e;
  if (sh >= 0)
    m <<= sh;
  else
    m = sh < -54 ? 0ull : (m + (1ull << (-sh - 1))) >> -sh;
  return b < 0 ? -(long long)m : (long long)m;
}

// (h + l) 2^(47 - e) rounded to an integer (s = 2^-e), left-aligned in 64 bits
__device__ __forceinline__ long long fixed_df(float h, float l, float s) {
  constexpr float M = 12582912.f;  // 1.5 * 2^23: adding it rounds to an integer
  constexpr int MI = 0x4b400000;
  const float hs = __fmul_rn(h, s), ls = __fmul_rn(l, s);
  const float t0 = __fmaf_rn(hs, 32768.f, M);
  const float r0 = __fmaf_rn(__fsub_rn(t0, M), -3.0517578125e-05f, hs);
  const float t1 = __fmaf_rn(r0, 2147483648.f, M);
  const float r1 = __fmaf_rn(__fsub_rn(t1, M), -4.656612873077393e-10f, r0);
  const float t2 = __fmaf_rn(r1, 140737488355328.f, M);
  const float t3 = __fmaf_rn(ls, 140737488355328.f, M);
  const long long i0 = __float_as_int(t0) - MI, i1 = __float_as_int(t1) - MI;
  const int i2 = (__float_as_int(t2) - MI) + (__float_as_int(t3) - MI);
  return ((i0 << 32) + (i1 << 16) + i2) * 65536;
}

constexpr long long BIAS = (long long)0x8080808080808080ull;

// digit words of a complex number: word k = bytes (re, im) of digit 2k, then
// (re, im) of digit 2k + 1
template <int W>
__device__ __forceinline__ void digit_words(long long re, long long im, uint32_t* w) {
  const unsigned long long a = (unsigned long long)(re + BIAS), b = (unsigned long long)(im + BIAS);
  const uint32_t ah = (uint32_t)(a >> 32), bh = (uint32_t)(b >> 32);
  w[0] = __byte_perm(ah, bh, 0x6273);
  w[1] = __byte_perm(ah, bh, 0x4051);
  w[2] = __byte_perm((uint32_t)a, (uint32_t)b, 0x6273);
  if constexpr (W == 4) w[3] = __byte_perm((uint32_t)a, (uint32_t)b, 0x4051);
}

// One CTA of 12 warps per SM: the pipelined loop wants about 160 registers,
// and at 16^4..32^4, N = 16 (double-float) twelve such warps took 0.89 ms a half
// where two CTAs of 8 warps at 128 registers took 0.92 and 14 or 10 warps 1.0
// and 1.07 ms.  DEPTH: chunks of input digits in flight.
constexpr int THREADS = 384;
constexpr int DEPTH = 3;

// the products of digits s and t that are kept: s + t <= ND - 1, and in
// double-float also s + t = 6 (5 of 26; without them the error grows from
// 1.8e-14 to 8.7e-14 of the result, that of the CUDA cores being 3.0e-14)
template <int ND>
__host__ __device__ constexpr bool keep(int s, int t) {
  return s + t < ND || (ND == 6 && s + t == 6 && s > 0 && t > 0);
}

template <class S>
struct Kind;
template <>
struct Kind<StoreDF> {
  static constexpr int ND = 6, W = 3, NU = 7;  // digits, words, accumulators
  static __device__ __forceinline__ unsigned key(float4 v) {
    const unsigned a = __float_as_uint(v.x) & 0x7fffffffu, b = __float_as_uint(v.y) & 0x7fffffffu;
    return a > b ? a : b;
  }
  static __device__ __forceinline__ int exponent(unsigned m) { return exp_f32(m); }
  static __device__ __forceinline__ bool bad(unsigned m) { return bad_f32(m); }
  static __device__ __forceinline__ void words(float4 v, int e, uint32_t* w) {
    const float s = exp2f_int(-e);
    digit_words<W>(fixed_df(v.x, v.z, s), fixed_df(v.y, v.w, s), w);
  }
};
template <>
struct Kind<StoreF64> {
  static constexpr int ND = 8, W = 4, NU = 8;
  static __device__ __forceinline__ unsigned key(double2 v) {
    const unsigned a = __double2hiint(v.x) & 0x7fffffff, b = __double2hiint(v.y) & 0x7fffffff;
    return a > b ? a : b;
  }
  static __device__ __forceinline__ int exponent(unsigned m) { return exp_f64(m); }
  static __device__ __forceinline__ bool bad(unsigned m) { return bad_f64(m); }
  static __device__ __forceinline__ void words(double2 v, int e, uint32_t* w) {
    digit_words<W>(fixed_f64(v.x, e), fixed_f64(v.y, e), w);
  }
};

static __global__ void k_fx_zero(unsigned* ctl, int slot, Gate gate) {
  if (gate_closed(gate)) return;
  ctl[CTL_MAX + 64 * slot + threadIdx.x] = 0u;
  if (threadIdx.x == 0) ctl[CTL_FLAG + slot] = 0u;
}

// column maxima of a block [row][N]; HBM-bound (one read of the block).
// Only the first half of a pair needs it: the stencil tracks its own output's,
// and the tensor-core update that writes the iteration's P tracks P's (81 us
// less an iteration at 32^4, N = 16).
template <class S>
__global__ void __launch_bounds__(256)
    k_fx_colmax(const typename S::elem* __restrict__ f, int N, long long rows, unsigned* ctl,
                int slot, Gate gate) {
  __shared__ unsigned sm[64];
  if (gate_closed(gate)) return;
  if (threadIdx.x < 64) sm[threadIdx.x] = 0u;
  __syncthreads();
  const int rpb = 256 / N;  // rows per block and step
  const int r0 = threadIdx.x / N, col = threadIdx.x - r0 * N;
  unsigned m = 0u;
  if (r0 < rpb)
    for (long long r = (long long)blockIdx.x * rpb + r0; r < rows; r += (long long)gridDim.x * rpb)
      m = max(m, Kind<S>::key(f[r * N + col]));
  if (r0 < rpb) atomicMax(&sm[col], m);
  __syncthreads();
  if (threadIdx.x < N) atomicMax(ctl + CTL_MAX + 64 * slot + threadIdx.x, sm[threadIdx.x]);
}

// a run's maximum v (FP32 bits) more than 2^3 below its column's c, zero aside
__device__ __forceinline__ bool low(unsigned v, unsigned c) { return v != 0u && v + (3u << 23) < c; }

// the digit records of a block (HBM-bound: one read, one write of 3/4 of it
// in double-float): thread = (site, 16 m + gq), a CTA takes 8, 16 or 32 sites a
// step; clears the other parity's control words, which its stencil accumulates
// into.  Nothing to do in a half
// that the links flag.
// sites a step: V_h is a multiple of 8 (even extents), so no run is shorter
__host__ __device__ inline int digit_sites(int NP) { return NP == 1 ? 32 : NP == 2 ? 16 : 8; }
template <class S, int R>
__global__ void __launch_bounds__(256)
    k_fx_digits(const typename S::elem* __restrict__ f, unsigned char* __restrict__ dig, int N,
                int NP, int Vh, unsigned* ctl, const unsigned* __restrict__ bad_links, int slot,
                Gate gate) {
  using K = Kind<S>;
  using RC = Rec<K::W, R>;
  constexpr int W = K::W;
  if (gate_closed(gate)) return;
  if (blockIdx.x == 0 && threadIdx.x < 65)
    ctl[threadIdx.x < 64 ? CTL_MAX + 64 * (1 - slot) + threadIdx.x : CTL_FLAG + 1 - slot] = 0u;
  const unsigned marked = *bad_links;
  __shared__ unsigned cm[64], run[2][64];  // maxima: of the columns, of a step's sites
  if (threadIdx.x < 64) {
    cm[threadIdx.x] = ctl[CTL_MAX + 64 * slot + threadIdx.x];
    run[0][threadIdx.x] = run[1][threadIdx.x] = 0u;
  }
  __syncthreads();
  if (marked) {
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl[CTL_FLAG + slot] = 1u;
    return;
  }
  bool bad = false;
  const int gq = threadIdx.x & 7, ls = (threadIdx.x >> 3) / NP, m = (threadIdx.x >> 3) - ls * NP;
  const int per = digit_sites(NP);
  int par = 0;
  for (long long s0 = (long long)blockIdx.x * per; s0 < Vh;
       s0 += (long long)gridDim.x * per, par ^= 1) {
    const long long site = s0 + ls;
    if (K::ND == 6 && s0 != (long long)blockIdx.x * per) {
      // the previous step's maxima; its words are used again after the next barrier
      __syncthreads();
      if (threadIdx.x < N) bad = bad || low(run[par ^ 1][threadIdx.x], cm[threadIdx.x]);
      if (threadIdx.x < N) run[par ^ 1][threadIdx.x] = 0u;
    }
    if (ls >= per || site >= Vh) continue;
    const long long sm = site * NP + m;
    uint32_t w[3][RC::WPC];
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int k = 0; k < RC::WPC; ++k) w[j][k] = 0x80808080u;  // zero (N not a multiple of 8 R)
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int n = 8 * R * m + gq + 8 * r;
      if (n < N) {
        const int e = K::exponent(cm[n]);
        bad = bad || K::bad(cm[n]);
        unsigned vm = 0u;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const typename S::elem v = f[(site * 3 + j) * N + n];
          vm = max(vm, K::key(v));
          K::words(v, e, w[j] + r * W);
        }
        if constexpr (K::ND == 8)
          bad = bad || (vm != 0u && (vm >> 20) + 9u < (cm[n] >> 20));
        else
          atomicMax(&run[par][n], vm);
      }
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      unsigned char* o = dig + sm * RC::BYTES + j * RC::COLOUR;
#pragma unroll
      for (int c = 0; c < RC::WPC / 4; ++c)
        reinterpret_cast<uint4*>(o + c * 128)[gq] =
            make_uint4(w[j][4 * c], w[j][4 * c + 1], w[j][4 * c + 2], w[j][4 * c + 3]);
      if constexpr (RC::WPC % 4 == 2)
        reinterpret_cast<uint2*>(o + 128)[gq] = make_uint2(w[j][4], w[j][5]);
    }
  }
  if constexpr (K::ND == 6) {  // the last step's maxima
    __syncthreads();
    if (threadIdx.x < N) bad = bad || low(run[par ^ 1][threadIdx.x], cm[threadIdx.x]);
  }
  if (bad) atomicOr(ctl + CTL_FLAG + slot, 1u);
}

// unsigned division by a fixed divisor for n < 2^31 (Granlund & Montgomery)
struct FastDiv {
  unsigned d, m;
  int l;
};
inline FastDiv fast_div(unsigned d) {
  int l = 0;
  while ((1ull << l) < d) ++l;
  return {d, (unsigned)(((1ull << 32) * ((1ull << l) - d)) / d + 1), l};
}
__device__ __forceinline__ unsigned fdiv(unsigned n, const FastDiv& f) {
  return (__umulhi(n, f.m) + n) >> f.l;
}

struct Args {
  const unsigned char* dig;
  Links L;
  const unsigned* ctl;
  unsigned* omax;  // column maxima of the output (the second half's input), or null
  int slot, N, NP, parity;
  FastDiv fx, fy, fz, fp;  // extents hx, Ly, Lz; NP
};

__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                        uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void cp16(uint32_t smem, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem), "l"(g));
}

// The CUDA-core stencil on the digit kernel's grid, for the blocks that one
// scale per column cannot represent.  12 warps an SM instead of the tuned
// kernel's 16 to 24: double-float makes up for it with four right-hand sides a
// thread (at two the link loads bind: a half at 32^4, N = 16, with the layout
// conversions, 3080 us against 2660; one 3820; the cp.async kernel 2530).  With
// less than two rounds of such threads, two right-hand sides (16^4, N = 8 137 us
// against 147), then one.  Warps are dealt out over the SMs in turn, so that few
// rounds end together (16^4, N = 8 147 us against 167 with whole blocks;
// 12.8.10.14, N = 5 in FP64 60 against 80, where whole blocks left 64 of 152 SMs
// idle).  FP64 is bound by its rate either way: within 5 % of the tuned kernel.
// A flagged operator call, both halves: 32^4, N = 16 5150 us (cp.async 4780),
// N = 8 2660 (2520); 16^4, N = 8 262 (190).
template <class S, int EPI>
__device__ __noinline__ void fx_cores(const typename S::elem* links, const typename S::elem* in,
                                      typename S::elem* out, const typename S::elem* c1,
                                      const typename S::elem* c2, double m2d, const Geom& g,
                                      int parity, int N, unsigned* smax, unsigned* omax) {
  const long long first =
      ((long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31);
  const long long step = (long long)gridDim.x * THREADS;
  // the output's column maxima, for the second half (smax: 64 words shared)
  auto seen = [=](int n, const auto& v) {
    if (EPI == EPI_NONE && omax) {
      if constexpr (std::is_same<S, StoreDF>::value)
        atomicMax(smax + n, Kind<S>::key(make_float4(v.re.hi, v.im.hi, 0.f, 0.f)));
      else
        atomicMax(smax + n, Kind<S>::key(make_double2(v.re, v.im)));
    }
  };
  if (threadIdx.x < 64) smax[threadIdx.x] = 0u;
  __syncthreads();
  auto run = [&](auto r, auto unroll) {
    constexpr int RV = decltype(r)::value, U = decltype(unroll)::value;
    const int T = (N + RV - 1) / RV;
    dslash_outputs<S, RV, 1, EPI, U>(links, in, out, c1, c2, m2d, g, parity, N, T, first,
                                     g.Vh * (long long)T, step, seen);
  };
  using std::integral_constant;
  constexpr bool DF = std::is_same<S, StoreDF>::value;
  if (DF && g.Vh * (long long)((N + 3) / 4) >= 2 * step)
    run(integral_constant<int, DF ? 4 : 1>(), integral_constant<int, DF ? 0 : 1>());
  else if (DF && g.Vh * (long long)((N + 1) / 2) >= 2 * step)
    run(integral_constant<int, DF ? 2 : 1>(), integral_constant<int, DF ? 0 : 1>());
  else
    run(integral_constant<int, 1>(), integral_constant<int, 1>());
  if (EPI == EPI_NONE && omax) {
    __syncthreads();
    if (threadIdx.x < N && smax[threadIdx.x]) atomicMax(omax + threadIdx.x, smax[threadIdx.x]);
  }
}

// double-float output: sum_u D_u 2^(-8u), normalised.  The leading digits are
// small (a value is some 2^-3 of its column's scale) and the others are not, so
// D_3 2^-24 is still about 2^-20 of the sum: D_0 .. D_3 are added exactly,
// the rest fits one FP32 number.
__device__ __forceinline__ void fx_add(float& h, float& l, float d, float c) {  // h + l += d c
  const float s = __fmaf_rn(d, c, h);
  const float z = __fsub_rn(s, h);
  l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(s, z)), __fmaf_rn(d, c, -z)));
  h = s;
}
__device__ __forceinline__ dfacc fx_sum(float d0, float d1, float d2, float d3, float d4, float d5,
                                        float d6) {
  constexpr float c = 0.00390625f;  // 2^-8
  float h = d0, l = __fmul_rn(__fmaf_rn(__fmaf_rn(d6, c, d5), c, d4), c * c * c * c);
  fx_add(h, l, d1, c);
  fx_add(h, l, d2, c * c);
  fx_add(h, l, d3, c * c * c);
  const float r = __fadd_rn(h, l);  // fast two-sum: |h| >= |l|
  return {r, __fsub_rn(l, __fsub_rn(r, h))};
}

// One warp per (site, 16 right-hand sides).  Lane (gq, tig) = (lane / 4,
// lane % 4): hop kind q = tig of every direction, so its K entries are 4
// sites x 3 colours; rows gq and gq + 8; column gq of B; outputs of colour
// tig.  Chunk k of the K index holds colour k % 3 of two directions; the
// registers of its digits are refilled, as soon as it is multiplied, for the
// chunk three later (the other two directions, then the next site's first
// two), so three chunks of loads are in flight; the next site's links come by
// cp.async into a per-warp buffer.
template <class S, int R, int EPI>
__global__ void __launch_bounds__(THREADS, 1)
    k_dslash_fx(const typename S::elem* __restrict__ links, const typename S::elem* __restrict__ in,
                typename S::elem* __restrict__ out, const typename S::elem* __restrict__ c1,
                const typename S::elem* __restrict__ c2, double m2d, Geom g, Args A, Gate gate) {
  using K = Kind<S>;
  using C = typename S::comp;
  using RC = Rec<K::W, R>;
  constexpr int ND = K::ND, NU = K::NU, W = K::W, WPC = RC::WPC;
  constexpr int STAGE = REC_MAIN + (ND == 8 ? REC_EXTRA : 0);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (gate_closed(gate)) return;
  const int N = A.N;
  if (A.ctl[CTL_FLAG + A.slot]) {
    fx_cores<S, EPI>(links, in, out, c1, c2, m2d, g, A.parity, N, (unsigned*)smem_raw, A.omax);
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gq = lane >> 2, tig = lane & 3;
  const int li = tig * 3 + (gq < 6 ? gq >> 1 : 2);  // link words: (q, colour of column gq)
  const bool part = gq & 1;                         // column gq is an imaginary part
  const uint32_t selA = part ? 0x4041u : 0x4140u, selB = part ? 0x4243u : 0x4342u;
  const __half2 bmul = __floats2half2_rn(32768.f, part ? 32768.f : -32768.f);
  const __half2 badd = __floats2half2_rn(-0.25f, part ? -0.25f : 0.25f);
  const unsigned char* stp = smem_raw + warp * 2 * STAGE;
  const uint32_t stage0 = (uint32_t)__cvta_generic_to_shared(stp) + lane * 16;
  const typename C::real m2 = C::from_double(m2d);
  const unsigned char* digl = A.dig + gq * 16;
  const long long pbase = (long long)A.parity * g.Vh;
  unsigned om[R];
  int ea[R];
#pragma unroll
  for (int r = 0; r < R; ++r) om[r] = 0u, ea[r] = 0;

  // items (site, column block m), fewer than 2^29
  const int items = g.Vh * A.NP, step = gridDim.x * (THREADS / 32);
  int item = blockIdx.x * (THREADS / 32) + warp;
  auto stage = [&](int site, int buf) {  // the site's links into buffer buf
    const uint32_t d = stage0 + buf * STAGE;
    const unsigned char* p = A.L.main + (pbase + site) * REC_MAIN + lane * 16;
    constexpr int CM = REC_MAIN / 16, CX = REC_EXTRA / 16;
#pragma unroll
    for (int k = 0; k < (CM + 31) / 32; ++k)
      if (32 * k + 32 <= CM || lane < CM - 32 * k) cp16(d + 512 * k, p + 512 * k);
    if constexpr (ND == 8) {
      const unsigned char* x = A.L.extra + (pbase + site) * REC_EXTRA + lane * 16;
#pragma unroll
      for (int k = 0; k < (CX + 31) / 32; ++k)
        if (32 * k + 32 <= CX || lane < CX - 32 * k) cp16(d + REC_MAIN + 512 * k, x + 512 * k);
    }
  };
  // this lane's hop of each direction; +-3 is +-1 on an extent of 2
  int nb[4];
  auto neighbours = [&](unsigned site) {
    const unsigned r0 = fdiv(site, A.fx), r1 = fdiv(r0, A.fy), t = fdiv(r1, A.fz);
    const int xh = (int)(site - r0 * A.fx.d), y = (int)(r0 - r1 * A.fy.d), z = (int)(r1 - t * A.fz.d);
    const int xo = (y + z + (int)t + A.parity) & 1;
    const int c[4] = {2 * xh + xo, y, z, (int)t};
    int st = g.hx;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const int L = g.L[mu];
      int dv = hop_k(tig);
      if (L == 2 && (tig & 2)) dv = tig == 2 ? 1 : -1;
      const int v = c[mu] + dv;
      if (v >= L) dv -= L;
      if (v < 0) dv += L;
      if (mu == 0) {
        nb[0] = (int)site + ((xo + dv) >> 1);
      } else {
        nb[mu] = (int)site + dv * st;
        st *= L;
      }
    }
  };
  uint32_t aw[DEPTH][2][WPC];
  auto load_a = [&](int k, int m) {  // the digits of chunk k of the site of nb
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned char* p = digl + ((long long)nb[2 * (k / 3) + h] * A.NP + m) * RC::BYTES +
                               (k % 3) * RC::COLOUR;
      uint32_t* w = aw[k % DEPTH][h];
#pragma unroll
      for (int c = 0; c < WPC / 4; ++c) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(p + c * 128));
        w[4 * c] = v.x;
        w[4 * c + 1] = v.y;
        w[4 * c + 2] = v.z;
        w[4 * c + 3] = v.w;
      }
      if constexpr (WPC % 4 == 2) {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(p + 128 - gq * 8));
        w[4] = v.x;
        w[5] = v.y;
      }
    }
  };
  // B operands of a chunk, made while the chunk before it is multiplied
  uint32_t b[2][ND][2], bw[2 * W];
  auto load_b = [&](const unsigned char* sb, int q) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const uint2 v = *(reinterpret_cast<const uint2*>(sb) + (3 * q + k) * 12 + li);
      bw[(2 * k) / 3 * W + (2 * k) % 3] = v.x;
      bw[(2 * k + 1) / 3 * W + (2 * k + 1) % 3] = v.y;
    }
    if constexpr (W == 4) {
      const uint2 v = *(reinterpret_cast<const uint2*>(sb + REC_MAIN) + q * 12 + li);
      bw[3] = v.x;
      bw[7] = v.y;
    }
  };
  auto make_b = [&](int q, int t) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t raw = __byte_perm(bw[h * W + (t >> 1)], 0u, (t & 1) ? selB : selA);
      const __half2 v = __hfma2(*reinterpret_cast<const __half2*>(&raw), bmul, badd);
      b[q & 1][t][h] = *reinterpret_cast<const uint32_t*>(&v);
    }
  };

  if (item >= items) return;
  int site = (int)fdiv((unsigned)item, A.fp), m = item - site * A.NP, pm = -1;
  stage(site, 0);
  asm volatile("cp.async.commit_group;\n");
  neighbours((unsigned)site);
#pragma unroll
  for (int k = 0; k < DEPTH; ++k) load_a(k, m);
  asm volatile("cp.async.wait_group 0;\n");
  __syncwarp();
  load_b(stp, 0);
#pragma unroll
  for (int t = 0; t < ND; ++t) make_b(0, t);
  int buf = 0;
  bool more = true;
  while (more) {
    item += step;
    more = item < items;
    // the next item (the last one prefetches itself)
    const int nitem = more ? item : item - step;
    const int nsite = (int)fdiv((unsigned)nitem, A.fp), nm = nitem - nsite * A.NP;
    stage(nsite, buf ^ 1);
    asm volatile("cp.async.commit_group;\n");
    const unsigned char* sb = stp + buf * STAGE;
    float acc[NU][4];
    {
      const float2* ini = reinterpret_cast<const float2*>(sb + REC_DIG) + (tig < 3 ? tig : 0) * 8;
#pragma unroll
      for (int u = 0; u < NU; ++u) {
        const float2 v = ND == 6 && u == 6
                             ? reinterpret_cast<const float2*>(sb + REC_D6)[tig < 3 ? tig : 0]
                             : ini[u];
        acc[u][0] = v.x;
        acc[u][1] = v.y;
        acc[u][2] = v.x;
        acc[u][3] = v.y;
      }
    }
    const int eb = *reinterpret_cast<const int*>(sb + REC_D6 + 24);
    cpx<typename C::real> cc[R];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      if (q < 5) {
        load_b(sb, q + 1);
      } else {
        asm volatile("cp.async.wait_group 0;\n");
        __syncwarp();
        load_b(stp + (buf ^ 1) * STAGE, 0);
      }
      if (EPI != EPI_NONE && q == 3 && tig < 3) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int n = 8 * R * m + gq + 8 * r;
          if (n < N) cc[r] = S::load(c1 + ((long long)site * 3 + tig) * N + n);
        }
      }
      const uint32_t(&w)[2][WPC] = aw[q % DEPTH];
#pragma unroll
      for (int s = 0; s < ND; ++s) {
        const uint32_t sel = (s & 1) ? 0x4342u : 0x4140u;
        uint32_t a[4];
        a[0] = __byte_perm(w[0][s >> 1], 0u, sel);
        a[2] = __byte_perm(w[1][s >> 1], 0u, sel);
        a[1] = R == 2 ? __byte_perm(w[0][W * (R - 1) + (s >> 1)], 0u, sel) : 0u;
        a[3] = R == 2 ? __byte_perm(w[1][W * (R - 1) + (s >> 1)], 0u, sel) : 0u;
#pragma unroll
        for (int t = 0; t < ND; ++t)
          if (keep<ND>(s, t)) mma_f16(acc[s + t], a, b[q & 1][t][0], b[q & 1][t][1]);
        make_b(q + 1, s);
      }
      // refill the digits' registers for chunk q + DEPTH (of this or the next site)
      if (q + DEPTH < 6)
        load_a(q + DEPTH, m);
      else {
        if (q + DEPTH == 6) neighbours((unsigned)nsite);
        load_a(q + DEPTH - 6, nm);
      }
    }
    // outputs: colour tig, right-hand sides 8 R m + gq + 8 r
    if (m != pm) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int n = 8 * R * m + gq + 8 * r;
        if (n < N) ea[r] = K::exponent(__ldg(A.ctl + CTL_MAX + 64 * A.slot + n));
      }
      pm = m;
    }
    if (tig < 3) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int n = 8 * R * m + gq + 8 * r;
        if (n >= N) continue;
        const long long oi = ((long long)site * 3 + tig) * N + n;
        cpx<typename C::acc> vv;
        if constexpr (ND == 6) {
          // digit grids 2^(-7-8s), operands scaled by 2^-24 and 2^-9: 2^19
          const float fa = exp2f_int(ea[r] + 19), fb = exp2f_int(eb);
          auto join = [&](int i) {
            const dfacc v = fx_sum(acc[0][i], acc[1][i], acc[2][i], acc[3][i], acc[4][i], acc[5][i],
                                   acc[6][i]);
            return dfacc{__fmul_rn(__fmul_rn(v.s, fa), fb), __fmul_rn(__fmul_rn(v.e, fa), fb)};
          };
          vv.re = join(2 * r);
          vv.im = join(2 * r + 1);
        } else {
          // integers in units of 2^(-14-8u): exact 64-bit sums of the upper
          // and the lower four, added with one rounding
          const double sc = exp2d_int(ea[r] + eb - 70);
          auto join = [&](int i) {
            long long hi = 0, lo = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              hi = hi * 256 + __float2int_rn(__fmul_rn(acc[u][i], 8589934592.f));
              lo = lo * 256 + __float2int_rn(__fmul_rn(acc[(NU == 8 ? 4 : 0) + u][i], 8589934592.f));
            }
            return fma((double)hi, 4294967296.0, (double)lo) * sc;
          };
          vv.re = join(2 * r);
          vv.im = join(2 * r + 1);
        }
        cpx<typename C::real> o;
        if constexpr (EPI == EPI_NONE) {  // already normalised
          if constexpr (ND == 6)
            o = {{vv.re.s, vv.re.e}, {vv.im.s, vv.im.e}};
          else
            o = vv;
        } else {
          C::neg(vv.re);
          C::neg(vv.im);
          C::mac(vv.re, m2, cc[r].re);
          C::mac(vv.im, m2, cc[r].im);
          if (EPI == EPI_RESIDUAL) {
            C::neg(vv.re);
            C::neg(vv.im);
            const cpx<typename C::real> bb = S::load(c2 + oi);
            C::add(vv.re, bb.re);
            C::add(vv.im, bb.im);
          }
          o = cfin<C>(vv);
        }
        S::store(out + oi, o);
        if constexpr (EPI == EPI_NONE) {
          if constexpr (ND == 6)
            om[r] = max(om[r], K::key(make_float4(o.re.hi, o.im.hi, 0.f, 0.f)));
          else
            om[r] = max(om[r], K::key(make_double2(o.re, o.im)));
        }
      }
    }
    // the output's column maxima, when the next item has another block m
    if (EPI == EPI_NONE && A.omax && (!more || nm != m)) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        unsigned v = om[r];
        v = max(v, __shfl_xor_sync(0xffffffffu, v, 1));
        v = max(v, __shfl_xor_sync(0xffffffffu, v, 2));
        const int n = 8 * R * m + gq + 8 * r;
        if (tig == 0 && n < N && v) atomicMax(A.omax + n, v);
        om[r] = 0u;
      }
    }
    __syncwarp();  // this buffer's link words are read before they are replaced
    site = nsite;
    m = nm;
    buf ^= 1;
  }
}

template <class S, int R, int EPI>
static cudaError_t launch_fx(const void* links, const void* in, void* out, const void* c1,
                             const void* c2, double m2, const Geom& g, const Args& A, Gate gate,
                             cudaStream_t s) {
  using E = typename S::elem;
  constexpr size_t sm = THREADS / 32 * 2 * (REC_MAIN + (Kind<S>::ND == 8 ? REC_EXTRA : 0));
  auto kern = k_dslash_fx<S, R, EPI>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, THREADS, sm) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  const long long want = (long long)stencil_sms() * per_sm;
  const long long need = ((long long)g.Vh * A.NP + THREADS / 32 - 1) / (THREADS / 32);
  kern<<<(unsigned)(need < want ? need : want), THREADS, sm, s>>>(
      (const E*)links, (const E*)in, (E*)out, (const E*)c1, (const E*)c2, m2, g, A, gate);
  return cudaGetLastError();
}

template <class S, int R>
static cudaError_t run_fx(int flags, int epi, const void* links, const void* in, void* out,
                          const void* c1, const void* c2, double m2, const Geom& g, int parity,
                          int N, Gate gate, cudaStream_t s) {
  using E = typename S::elem;
  const int slot = 1 - parity;
  const int NP = (N + 8 * R - 1) / (8 * R);
  const unsigned sms = (unsigned)stencil_sms();
  auto cap = [&](long long n, unsigned per) {
    const unsigned c = sms * (gate_mostly_off(gate) ? 2u : per);
    return (unsigned)(n < 1 ? 1 : n < (long long)c ? n : c);
  };
  if (!(flags & (DSLASH_SECOND | DSLASH_MAXED))) {
    k_fx_zero<<<1, 64, 0, s>>>(g.fx_ctl, slot, gate);
    const long long rows = 3LL * g.Vh;
    const int rpb = 256 / N;
    k_fx_colmax<S><<<cap((rows + rpb - 1) / rpb, 8), 256, 0, s>>>((const E*)in, N, rows, g.fx_ctl,
                                                                  slot, gate);
  }
  k_fx_digits<S, R><<<cap((g.Vh + digit_sites(NP) - 1) / digit_sites(NP), 8), 256, 0, s>>>(
      (const E*)in, (unsigned char*)g.fx_dig, N, NP, g.Vh, g.fx_ctl,
      links_of(g.fx_links, g).bad + (Kind<S>::ND == 6 ? 1 : 0), slot, gate);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  Args A;
  A.dig = (const unsigned char*)g.fx_dig;
  A.L = links_of(g.fx_links, g);
  A.ctl = g.fx_ctl;
  A.omax = (flags & DSLASH_FIRST) ? g.fx_ctl + CTL_MAX + 64 * parity : nullptr;
  A.slot = slot;
  A.N = N;
  A.NP = NP;
  A.parity = parity;
  A.fx = fast_div((unsigned)g.hx);
  A.fy = fast_div((unsigned)g.L[1]);
  A.fz = fast_div((unsigned)g.L[2]);
  A.fp = fast_div((unsigned)NP);
  switch (epi) {
    case EPI_NONE: return launch_fx<S, R, EPI_NONE>(links, in, out, c1, c2, m2, g, A, gate, s);
    case EPI_NORMAL: return launch_fx<S, R, EPI_NORMAL>(links, in, out, c1, c2, m2, g, A, gate, s);
    default: return launch_fx<S, R, EPI_RESIDUAL>(links, in, out, c1, c2, m2, g, A, gate, s);
  }
}

}  // namespace fx
}  // namespace bcg
