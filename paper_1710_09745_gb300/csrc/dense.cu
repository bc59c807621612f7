// Small dense N x N algebra of blockCGrQ in native FP64, on the device, one
// CTA per call (N <= 64).  The paper does these on the host with Eigen
// (Sec. 6); keeping them on the device removes every host round trip from the
// iteration, so a whole iteration is a fixed sequence of launches gated by the
// status word.
//
//   dense_beta     beta = (P^dag A P)^-1 through a Cholesky factorisation,
//                  BC = beta C                                  (Algorithm 1)
//   dense_qr_step  thin QR of W = Q - AP beta from its Gram: W^dag W = S^dag S
//                  (Cholesky), S^-1, S^dag; C_prev = C; C = S C; iterated
//                  residuals |R_i| = |column i of C|; reliable-update trigger
//                                                   (Algorithms 1, 2 and 3)
//   dense_restart  thin QR of a true residual R = B - A Y: C = chol factor,
//                  C^-1, convergence on the true residual, and
//                  S = C C_old^-1 with C_old the C in force before the last
//                  C = S C                                      (Algorithm 3)
// Matrices are complex128 row-major [N][N] in global memory; the CTA works
// on copies in shared memory.
#include "internal.h"
#include "../../include/blockcg.h"

namespace bcg {

static constexpr int DENSE_THREADS = 256;
// reliable update when the iterated residual exceeds this factor times the
// true residual of the last update
static constexpr double RU_GROWTH = 100.0;

__device__ __forceinline__ double2 cm(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

// 1 / d and 1 / sqrt(d) of a positive normal d from an FP32 estimate of the
// mantissa, by one step of r / (1 - e) = r (1 + e + e^2) and by two of Newton's:
// rounding level, a unit in the last place.  A dependent FP64 operation takes
// 64 clocks on this GPU, so FP64 division (392) and square root (595) are long
// chains; the mantissa is moved between the formats as integers, which skips
// the conversions too.
__device__ __forceinline__ double from_float_bits(float f) {  // f > 0, normal
  const unsigned b = __float_as_uint(f);
  return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}
__device__ __forceinline__ double scale_exp(double v, int e) {  // v 2^e, result normal
  return __hiloint2double(__double2hiint(v) + (e << 20), __double2loint(v));
}
__device__ double rcp_pos(double d) {
  const int hi = __double2hiint(d), ex = hi >> 20;
  if (ex < 3 || ex > 2040) return 1.0 / d;  // tiny, huge, negative, not finite
  const unsigned lo = (unsigned)__double2loint(d);
  const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, (int)lo);
  const float mf = __uint_as_float(0x3f800000u | ((unsigned)(hi & 0xfffff) << 3) | (lo >> 29));
  double r = from_float_bits(__fdividef(1.f, mf));
  const double e = fma(-m, r, 1.0);  // about 2^-23: one cubic step, 1/m = r / (1 - e)
  r = fma(r, fma(e, e, e), r);
  return scale_exp(r, 1023 - ex);
}
// s = sqrt(d), r = 1 / sqrt(d)
__device__ void sqrt_pos(double d, double& s, double& r) {
  const int hi = __double2hiint(d), ex = hi >> 20;
  if (ex < 3 || ex > 2040) {
    s = sqrt(d);
    r = 1.0 / s;
    return;
  }
  const int k = (ex - 1023) >> 1;
  const double m = scale_exp(d, -2 * k);  // in [1, 4)
  const int mh = __double2hiint(m);
  const float mf = __uint_as_float(((unsigned)(mh - 0x38000000) << 3) | ((unsigned)__double2loint(m) >> 29));
  double y = from_float_bits(rsqrtf(mf));
  y = fma(0.5 * y, fma(-m * y, y, 1.0), y);
  y = fma(0.5 * y, fma(-m * y, y, 1.0), y);
  double q = m * y;
  q = fma(fma(-q, q, m), 0.5 * y, q);
  s = scale_exp(q, k);
  r = scale_exp(y, -k);
}

// Factorisation A = U D U^dag of a Hermitian matrix with U unit lower
// triangular and D = diag(d) > 0, and X = U^-1, in one elimination of N steps
// (the Cholesky factor is L = U D^1/2, its inverse D^-1/2 X): step k forms the
// multipliers F_i = A_ik / d_k and subtracts F_i times row k from every later
// row of A (columns > k) and of X (columns <= k).  The two live side by side
// in M, columns above and below k; the multipliers go to U.
//
// Bound by the latency of N dependent steps and by the FP64 pipe of one SM (1.7
// multiply-adds a clock, so a warp's FP64 instruction takes 19 clocks): the
// entries of a step's rows are dealt to the threads without gaps (they are
// contiguous in the row-wise order of the lower triangle, looked up in `ij`), no
// thread repeats another's FP64 work, and the next pivot and its reciprocal
// are taken by a warp of their own beside the update.
//
// A pivot that is not finite gives BLOCKCG_ERR_NONFINITE; a pivot d_k <= 0 or
// d_k <= PIVOT_REL_TOL * A_kk (A_kk the diagonal before factorising) gives
// BLOCKCG_ERR_BREAKDOWN: d_k / A_kk is the squared sine of the angle between
// column k and the span of the columns before it, so a value at rounding
// level means the block is numerically rank deficient (e.g. linearly
// dependent right-hand sides, Sec. 4).  Returns 0 or the error (uniform over
// the CTA, and over CTAs that factorise the same matrix).  On return M holds
// X and U the multipliers, strictly below the diagonal.
static constexpr double PIVOT_REL_TOL = 1e-13;

struct Factor {
  double d[64], w[64];       // pivots and their reciprocals
  double diag0[64];          // the matrix's diagonal
  double2 col[64], mul[64];  // column k of A before step k, the multipliers
  double next;               // A_kk of the next pivot, before step k
  uchar2 ij[64 * 65 / 2];    // (i, j <= i) in row-wise order
  int flag;
};

__device__ __forceinline__ void take_pivot(Factor& f, int k, double d) {
  f.d[k] = d;
  f.w[k] = rcp_pos(d);
  int e = 0;
  if (!isfinite(d) || !isfinite(f.diag0[k])) e = BLOCKCG_ERR_NONFINITE;
  else if (!(d > 0.0) || !(d > PIVOT_REL_TOL * f.diag0[k])) e = BLOCKCG_ERR_BREAKDOWN;
  f.flag = e;
}

__device__ int factor(double2* M, double2* U, int N, Factor& f) {
  constexpr int UPDATERS = DENSE_THREADS - 32;  // the last warp takes the pivots
  const int tid = threadIdx.x;
  for (int k = tid; k < N; k += DENSE_THREADS) f.diag0[k] = M[k * N + k].x;
  for (int i = tid >> 3; i < N; i += DENSE_THREADS / 8)
    for (int j = tid & 7; j <= i; j += 8) f.ij[i * (i + 1) / 2 + j] = make_uchar2(i, j);
  __syncthreads();
  if (tid == UPDATERS) take_pivot(f, 0, M[0].x);
  __syncthreads();
  for (int k = 0; k < N; ++k) {
    if (f.flag) return f.flag;
    const double w = f.w[k];
    for (int i = k + 1 + tid; i < N; i += DENSE_THREADS) {
      const double2 v = M[i * N + k];
      const double2 m = make_double2(v.x * w, v.y * w);
      f.col[i] = v;
      f.mul[i] = m;
      U[i * N + k] = m;
      if (i == k + 1) f.next = M[i * N + i].x;
    }
    __syncthreads();
    if (tid < UPDATERS) {
      for (int t = (k + 1) * (k + 2) / 2 + tid; t < N * (N + 1) / 2; t += UPDATERS) {
        const int i = f.ij[t].x, j = f.ij[t].y;
        const double2 m = f.mul[i];
        const double2 r = j < k ? M[k * N + j] : j > k ? cconj(f.col[j]) : make_double2(1.0, 0.0);
        const double2 a = j == k ? make_double2(0.0, 0.0) : M[i * N + j];
        M[i * N + j] = make_double2(fma(-m.x, r.x, fma(m.y, r.y, a.x)),
                                    fma(-m.x, r.y, fma(-m.y, r.x, a.y)));
      }
    } else if (tid == UPDATERS && k + 1 < N) {
      const int i = k + 1;
      const double2 m = f.mul[i], c = f.col[i];
      take_pivot(f, i, fma(-m.x, c.x, fma(-m.y, c.y, f.next)));
    }
    __syncthreads();
  }
  return 0;
}

__device__ void load_mat(double2* dst, const double2* __restrict__ src, int N) {
  for (int idx = threadIdx.x; idx < N * N; idx += blockDim.x) dst[idx] = src[idx];
  __syncthreads();
}


// s += a b
__device__ __forceinline__ void cmad(double2& s, double2 a, double2 b) {
  s = cadd(s, cm(a, b));
}
// sum over the n (a power of two) neighbouring lanes that share a row
__device__ __forceinline__ double2 lane_sum(double2 s, int n) {
  for (int o = n >> 1; o > 0; o >>= 1) {
    s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
    s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
  }
  return s;
}
// lanes per row when `threads` share the N rows of a column
__device__ __forceinline__ int lanes_per_row(int N, int threads) {
  int rows = 4;
  while (rows < N) rows <<= 1;
  const int n = threads / rows;
  return n > 32 ? 32 : n;
}

// CTAs of a call whose result splits by columns: each repeats the
// factorisation (N dependent steps that more SMs cannot share) and takes its
// columns of the products
static int dense_ctas(int N) { return N < 4 ? 1 : N; }

// ---------------------------------------------------------------- beta ----
// beta = X^dag D^-1 X and beta C, a column of either at a time by a half of
// the CTA's threads: z = D^-1 X c, then X^dag z
__global__ void __launch_bounds__(DENSE_THREADS)
    k_dense_beta(const double2* __restrict__ H, const double2* __restrict__ Cm,
                 double2* __restrict__ beta, double2* __restrict__ BC, int N, SolverStatus* st,
                 Gate gate) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Factor f;
  __shared__ double2 z[2][64], c[64];
  if (gate_closed(gate)) return;
  double2* M = reinterpret_cast<double2*>(smem_raw);
  double2* U = M + N * N;
  if (threadIdx.x < N) c[threadIdx.x] = Cm[threadIdx.x * N + blockIdx.x];  // used after the factor
  load_mat(M, H, N);
  const int err = factor(M, U, N, f);
  if (err) {
    if (threadIdx.x == 0 && blockIdx.x == 0) st->error = err;
    return;
  }
  const int half = threadIdx.x >> 7, t = threadIdx.x & 127;
  const int S = lanes_per_row(N, 128), row = t / S, sub = t - row * S;
  for (int j = blockIdx.x; j < N; j += gridDim.x) {
    if (j != (int)blockIdx.x) {
      __syncthreads();
      if (threadIdx.x < N) c[threadIdx.x] = Cm[threadIdx.x * N + j];
      __syncthreads();
    }
    // column j of the identity (half 0) or of C, upper triangular (half 1)
    double2 s = make_double2(0.0, 0.0);
    if (row < N) {
      if (half == 0) {
        if (sub == 0 && row >= j) s = row == j ? make_double2(1.0, 0.0) : M[row * N + j];
      } else {
        if (sub == 0 && row <= j) s = c[row];
        for (int l = sub; l < row && l <= j; l += S) cmad(s, M[row * N + l], c[l]);
      }
    }
    s = lane_sum(s, S);
    if (sub == 0 && row < N) z[half][row] = make_double2(s.x * f.w[row], s.y * f.w[row]);
    __syncthreads();
    // X^dag: row r sums conj(X_lr) z_l over l >= r
    s = make_double2(0.0, 0.0);
    if (row < N) {
      if (sub == 0) s = z[half][row];
      for (int l = row + 1 + sub; l < N; l += S) cmad(s, cconj(M[l * N + row]), z[half][l]);
    }
    s = lane_sum(s, S);
    if (sub == 0 && row < N) (half ? BC : beta)[row * N + j] = s;
  }
}

cudaError_t dense_beta(const double2* H, const double2* C, double2* beta, double2* BC, int N,
                       SolverStatus* st, Gate gate, cudaStream_t s) {
  size_t sm = 2ull * N * N * sizeof(double2);
  cudaFuncSetAttribute(k_dense_beta, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k_dense_beta<<<dense_ctas(N), DENSE_THREADS, sm, s>>>(H, C, beta, BC, N, st, gate);
  return cudaGetLastError();
}

// ------------------------------------------------------------- qr step ----
__device__ __forceinline__ void end_loop(const LoopCtl& ctl) {
  if (ctl.on) {
    cudaGraphSetConditional(ctl.update, 0);
    cudaGraphSetConditional(ctl.loop, 0);
  }
}

// The columns are shared out over the CTAs (one CTA for N <= 16, where they
// take less than the CTAs' meeting would); the last CTA to finish, by a counter
// in the status word, takes the decisions from all column residuals.
__global__ void __launch_bounds__(DENSE_THREADS)
    k_dense_qr_step(const double2* __restrict__ G, double2* __restrict__ C,
                    double2* __restrict__ C_prev, double2* __restrict__ Sinv,
                    double2* __restrict__ SH, const double* __restrict__ bnorm, QrStepParams p,
                    int N, SolverStatus* st, Gate gate, LoopCtl ctl) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Factor f;
  __shared__ double sq[64], isq[64], res[64];
  __shared__ int last;
  const int tid = threadIdx.x;
  if (gate_closed(gate)) {  // converged, failed or stopped: the loop ends
    if (tid == 0 && blockIdx.x == 0) end_loop(ctl);
    return;
  }
  double2* M = reinterpret_cast<double2*>(smem_raw);
  double2* U = M + N * N;
  double2* Cs = U + N * N;
  for (int idx = tid; idx < N * N; idx += DENSE_THREADS) Cs[idx] = C[idx];
  const double bn = tid < N ? bnorm[tid] : 1.0, at_ru = st->res_at_ru;
  const int it = st->iters + 1;
  load_mat(M, G, N);
  const int err = factor(M, U, N, f);
  if (err) {
    if (tid == 0 && blockIdx.x == 0) {
      st->error = err;
      end_loop(ctl);
    }
    return;
  }
  for (int i = tid; i < N; i += DENSE_THREADS) {
    sqrt_pos(f.d[i], sq[i], isq[i]);
    res[i] = 0.0;
  }
  __syncthreads();
  // S^-1 = (L^-1)^dag, upper: column j is conj(row j of D^-1/2 X); S^dag = L
  for (int j = blockIdx.x + gridDim.x * (tid >> 6); j < N; j += gridDim.x * (DENSE_THREADS / 64)) {
    const int row = tid & 63;
    if (row >= N) continue;
    const double w = isq[j], q = sq[j];
    const double2 one = make_double2(row == j ? 1.0 : 0.0, 0.0);
    const double2 x = row < j ? M[j * N + row] : one, u = row > j ? U[row * N + j] : one;
    Sinv[row * N + j] = make_double2(x.x * w, -x.y * w);
    SH[row * N + j] = make_double2(u.x * q, u.y * q);
    C_prev[row * N + j] = Cs[row * N + j];
  }
  // C = S C, S = D^1/2 U^dag: row r sums conj(U_lr) C_lj over r <= l <= j (C is
  // upper triangular: a product of the Cholesky factors); a warp per column j,
  // whose residual is |R_j| = sqrt(sum_r |C_rj|^2)
  {
    const int warp = tid >> 5, lane = tid & 31;
    const int S = lanes_per_row(N < 32 ? N : 32, 32), rows = 32 / S;
    const int r0 = lane / S, sub = lane - r0 * S;
    for (int j = blockIdx.x + gridDim.x * warp; j < N; j += gridDim.x * (DENSE_THREADS / 32)) {
      double2 t = make_double2(0.0, 0.0);
      for (int rb = 0; rb < N; rb += rows) {
        const int row = rb + r0;
        double2 s = make_double2(0.0, 0.0);
        if (row < N && row <= j) {
          if (sub == 0) s = Cs[row * N + j];
          for (int l = row + 1 + sub; l <= j; l += S) cmad(s, cconj(U[l * N + row]), Cs[l * N + j]);
        }
        s = lane_sum(s, S);
        if (sub == 0 && row < N) {
          s = make_double2(s.x * sq[row], s.y * sq[row]);
          C[row * N + j] = s;
          t.x = fma(s.x, s.x, fma(s.y, s.y, t.x));
        }
      }
      t = lane_sum(t, 32);
      if (lane == 0) res[j] = t.x;
    }
  }
  __syncthreads();
  if (tid < N) {
    double q, r;
    sqrt_pos(res[tid], q, r);
    res[tid] = q * rcp_pos(bn);
    if (gridDim.x > 1 && tid % (int)gridDim.x == (int)blockIdx.x) st->col_res[tid] = res[tid];
  }
  if (gridDim.x > 1) {
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      last = atomicAdd(&st->arrivals, 1) == (int)gridDim.x - 1;
      __threadfence();
    }
    __syncthreads();
    if (!last) return;
    if (tid < N) res[tid] = ((const volatile double*)st->col_res)[tid];
  }
  __syncthreads();
  if (tid != 0) return;
  st->arrivals = 0;
  double rmax = 0.0;
  bool finite = true;
  for (int i = 0; i < N; ++i) {
    finite = finite && isfinite(res[i]);
    rmax = fmax(rmax, res[i]);
  }
  st->iters = it;
  st->res_max = rmax;
  int ru = 0;
  if (!finite) st->error = BLOCKCG_ERR_NONFINITE;
  if (rmax <= p.tol) ru = 1;
  else if (p.delta > 0.0 && rmax < p.delta * at_ru) ru = 1;
  else if (p.ru_every > 0 && (it % p.ru_every) == 0) ru = 1;
  // the iterated residual has grown far above the last true one: the
  // sloppy recursion is drifting, so recompute from the true residual
  else if (rmax > RU_GROWTH * at_ru) ru = 1;
  st->ru_pending = ru;
  // the iteration budget is spent: later gated launches do nothing
  const bool stop = p.max_iter > 0 && it >= p.max_iter;
  if (stop) st->stopped = 1;
  if (ctl.on) {
    st->trips += 1;
    cudaGraphSetConditional(ctl.update, ru && !stop && finite);
    cudaGraphSetConditional(ctl.loop, !stop && finite);
  }
}

cudaError_t dense_qr_step(const double2* G, double2* C, double2* C_prev, double2* Sinv,
                          double2* SH, const double* bnorm, QrStepParams p, int N,
                          SolverStatus* st, Gate gate, LoopCtl ctl, cudaStream_t s) {
  size_t sm = 3ull * N * N * sizeof(double2);
  cudaFuncSetAttribute(k_dense_qr_step, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  const int ctas = N <= 16 ? 1 : N / 2;
  k_dense_qr_step<<<ctas, DENSE_THREADS, sm, s>>>(G, C, C_prev, Sinv, SH, bnorm, p, N, st, gate, ctl);
  return cudaGetLastError();
}

// ------------------------------------------------------------- restart ----
__global__ void __launch_bounds__(DENSE_THREADS)
    k_dense_restart(const double2* __restrict__ G, double2* __restrict__ C,
                    double2* __restrict__ C_prev, double2* __restrict__ Cinv,
                    double2* __restrict__ SH, const double* __restrict__ bnorm,
                    double* __restrict__ tres_out, double tol, int init, int confirmed, int N,
                    SolverStatus* st, Gate gate, LoopCtl ctl) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Factor f;
  __shared__ double tres[64], sq[64], isq[64];
  if (gate_closed(gate)) return;
  double2* M = reinterpret_cast<double2*>(smem_raw);  // -> X of the true residual
  double2* U = M + N * N;                             // its multipliers
  double2* P = U + N * N;                             // C_prev^dag, then S^dag
  load_mat(M, G, N);
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    double q, r;
    sqrt_pos(fmax(M[i * N + i].x, 0.0), q, r);
    tres[i] = q * rcp_pos(bnorm[i]);
    tres_out[i] = tres[i];
  }
  __syncthreads();
  const int err = factor(M, U, N, f);
  if (err) {
    if (threadIdx.x == 0) {
      st->error = err;
      if (ctl.on) cudaGraphSetConditional(ctl.loop, 0);
    }
    return;
  }
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    sqrt_pos(f.d[i], sq[i], isq[i]);
  }
  __syncthreads();
  double tmax = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < N; ++i) tmax = fmax(tmax, tres[i]);
  // C_new = L^dag (upper), Cinv = (L^-1)^dag, L = U D^1/2, L^-1 = D^-1/2 X
  for (int idx = threadIdx.x; idx < N * N; idx += blockDim.x) {
    const int i = idx / N, j = idx - (idx / N) * N;
    const double w = isq[j];
    const double2 x = i < j ? M[j * N + i] : make_double2(i == j ? 1.0 : 0.0, 0.0);
    Cinv[idx] = make_double2(x.x * w, -x.y * w);
  }
  if (!init) {
    // S = C_new C_prev^-1, so S^dag = Y L with C_prev^dag Y = I: forward
    // substitution on the columns of L, C_prev^dag lower triangular, a row of
    // all columns per step
    __syncthreads();
    for (int i = threadIdx.x; i < N; i += blockDim.x) f.w[i] = rcp_pos(C_prev[i * N + i].x);
    for (int idx = threadIdx.x; idx < N * N; idx += blockDim.x) {
      const int i = idx / N, j = idx - (idx / N) * N;
      const double q = sq[j];
      const double2 u = i > j ? U[idx] : make_double2(i == j ? 1.0 : 0.0, 0.0);
      P[idx] = make_double2(u.x * q, u.y * q);
    }
    __syncthreads();
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    for (int k = 0; k < N; ++k) {
      const double w = f.w[k];
      for (int j = threadIdx.x; j <= k; j += blockDim.x) {
        const double2 v = P[k * N + j];
        P[k * N + j] = make_double2(v.x * w, v.y * w);
      }
      __syncthreads();
      for (int i = k + 1 + ty; i < N; i += DENSE_THREADS / 16) {
        const double2 m = cconj(C_prev[k * N + i]);  // (C_prev^dag)_ik
        for (int j = tx; j <= k; j += 16) P[i * N + j] = csub(P[i * N + j], cm(m, P[k * N + j]));
      }
      __syncthreads();
    }
    for (int idx = threadIdx.x; idx < N * N; idx += blockDim.x) SH[idx] = P[idx];
  }
  for (int idx = threadIdx.x; idx < N * N; idx += blockDim.x) {
    const int i = idx / N, j = idx - (idx / N) * N;
    const double q = sq[i];
    const double2 u = j > i ? U[j * N + i] : make_double2(i == j ? 1.0 : 0.0, 0.0);
    C[idx] = make_double2(u.x * q, -u.y * q);
  }
  if (threadIdx.x == 0) {
    st->true_res_max = tmax;
    st->res_max = tmax;
    st->res_at_ru = tmax;
    if (!isfinite(tmax)) st->error = BLOCKCG_ERR_NONFINITE;
    if (tmax <= tol) {
      st->done = 1;
      if (confirmed) st->verified = 1;
    }
    if (!init) st->reliable_updates += 1;
    if (ctl.on && (st->done || st->error)) cudaGraphSetConditional(ctl.loop, 0);
  }
}

// Native-FP64 confirmation of a convergence (see verify_fp64 in api.cu): G is
// the Gram of R = B - A Y computed in FP64; the per-column true residuals
// replace those of the double-float update.  All within tol: verified.
// Otherwise the solve goes on and all its later reliable updates are FP64.
__global__ void k_dense_verify(const double2* __restrict__ G, const double* __restrict__ bnorm,
                               double* __restrict__ tres, double tol, int N, SolverStatus* st) {
  __shared__ double r[64];
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    r[i] = sqrt(fmax(G[i * N + i].x, 0.0)) / bnorm[i];
    tres[i] = r[i];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double tmax = 0.0;
    bool finite = true;
    for (int i = 0; i < N; ++i) {
      tmax = fmax(tmax, r[i]);
      finite = finite && isfinite(r[i]);
    }
    st->true_res_max = tmax;
    if (!finite) {
      st->error = BLOCKCG_ERR_NONFINITE;
    } else if (tmax <= tol) {
      st->verified = 1;
    } else {
      st->done = 0;
      st->verified = 0;
      st->fp64_only = 1;
    }
  }
}

cudaError_t dense_verify(const double2* G, const double* bnorm, double* tres, double tol, int N,
                         SolverStatus* st, cudaStream_t s) {
  k_dense_verify<<<1, 64, 0, s>>>(G, bnorm, tres, tol, N, st);
  return cudaGetLastError();
}

cudaError_t dense_restart(const double2* G, double2* C, double2* C_prev, double2* Cinv,
                          double2* SH, const double* bnorm, double* tres, double tol, int init,
                          int confirmed, int N, SolverStatus* st, Gate gate, LoopCtl ctl,
                          cudaStream_t s) {
  size_t sm = 3ull * N * N * sizeof(double2);
  cudaFuncSetAttribute(k_dense_restart, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k_dense_restart<<<1, DENSE_THREADS, sm, s>>>(G, C, C_prev, Cinv, SH, bnorm, tres, tol, init,
                                               confirmed, N, st, gate, ctl);
  return cudaGetLastError();
}

// --------------------------------------------------------------- misc ----
__global__ void k_dense_bnorm(const double2* __restrict__ Gb, double* __restrict__ bnorm, int N,
                              SolverStatus* st) {
  int i = threadIdx.x;
  if (i < N) {
    double v = Gb[i * N + i].x;
    bnorm[i] = sqrt(fmax(v, 0.0));
    if (!isfinite(v)) st->error = BLOCKCG_ERR_NONFINITE;
    else if (!(v > 0.0)) st->error = BLOCKCG_ERR_BREAKDOWN;
  }
}

cudaError_t dense_bnorm(const double2* Gb, double* bnorm, int N, SolverStatus* st,
                        cudaStream_t s) {
  k_dense_bnorm<<<1, 64, 0, s>>>(Gb, bnorm, N, st);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(DENSE_THREADS)
    k_dense_chol_upper(const double2* __restrict__ H, double2* __restrict__ R,
                       double2* __restrict__ Rinv, int N, int* err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Factor f;
  __shared__ double sq[64], isq[64];
  double2* M = reinterpret_cast<double2*>(smem_raw);
  double2* U = M + N * N;
  load_mat(M, H, N);
  const int e = factor(M, U, N, f);
  if (threadIdx.x == 0) *err = e;
  if (e) return;
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    sqrt_pos(f.d[i], sq[i], isq[i]);
  }
  __syncthreads();
  // R = D^1/2 U^dag, R^-1 = (D^-1/2 X)^dag
  for (int idx = threadIdx.x; idx < N * N; idx += blockDim.x) {
    const int i = idx / N, j = idx - (idx / N) * N;
    const double2 u = j > i ? U[j * N + i] : make_double2(i == j ? 1.0 : 0.0, 0.0);
    const double2 x = j > i ? M[j * N + i] : u;
    R[idx] = make_double2(u.x * sq[i], -u.y * sq[i]);
    Rinv[idx] = make_double2(x.x * isq[j], -x.y * isq[j]);
  }
}

cudaError_t dense_chol_upper(const double2* H, double2* R, double2* Rinv, int N, int* err,
                             cudaStream_t s) {
  size_t sm = 2ull * N * N * sizeof(double2);
  cudaFuncSetAttribute(k_dense_chol_upper, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k_dense_chol_upper<<<1, DENSE_THREADS, sm, s>>>(H, R, Rinv, N, err);
  return cudaGetLastError();
}

// ------------------------------------------------------------ CG scalars ----
__global__ void k_cg_alpha(const double2* __restrict__ pAp, const double* __restrict__ rr,
                           const double* __restrict__ gam, double* __restrict__ alpha,
                           double* __restrict__ alpha_x, SolverStatus* st, Gate gate) {
  if (gate_closed(gate)) return;
  double d = pAp[0].x;
  if (!isfinite(d)) {
    st->error = BLOCKCG_ERR_NONFINITE;
    return;
  }
  if (!(d > 0.0)) {
    st->error = BLOCKCG_ERR_BREAKDOWN;
    return;
  }
  const double a = *rr / d;
  *alpha = a;
  *alpha_x = a / *gam;  // x is kept unscaled: x += (alpha / gamma) (gamma p)
}

__global__ void k_cg_beta(const double2* __restrict__ rr_new_sum, double* __restrict__ rr,
                          double* __restrict__ beta, const double* __restrict__ bnorm,
                          const double* __restrict__ gam, double tol, double delta,
                          SolverStatus* st, Gate gate) {
  if (gate_closed(gate)) return;
  double bnorm2 = bnorm[0] * bnorm[0];
  double rn = rr_new_sum[0].x;  // |gamma r|^2
  int it = st->iters + 1;
  st->iters = it;
  if (!isfinite(rn)) {
    st->error = BLOCKCG_ERR_NONFINITE;
    return;
  }
  double rel = sqrt(rn / bnorm2) / *gam;
  st->res_max = rel;
  // converged, or dropped by delta since the last reliable update: the host
  // runs a reliable update, which recomputes r and then forms beta from the
  // true residual (cg_restart_check); rr keeps the previous |r|^2 for that
  if (rel <= tol || (delta > 0.0 && rel < delta * st->res_at_ru)) {
    st->ru_pending = 1;
    return;
  }
  *beta = rn / *rr;
  *rr = rn;
}

cudaError_t cg_scalar_alpha(const double2* pAp, const double* rr, const double* gam, double* alpha,
                            double* alpha_x, SolverStatus* st, Gate gate, cudaStream_t s) {
  k_cg_alpha<<<1, 1, 0, s>>>(pAp, rr, gam, alpha, alpha_x, st, gate);
  return cudaGetLastError();
}

cudaError_t cg_scalar_beta(const double2* rr_new_sum, double* rr, double* beta,
                           const double* bnorm, const double* gam, double tol, double delta,
                           SolverStatus* st, Gate gate, cudaStream_t s) {
  k_cg_beta<<<1, 1, 0, s>>>(rr_new_sum, rr, beta, bnorm, gam, tol, delta, st, gate);
  return cudaGetLastError();
}

// The iteration works on gamma r and gamma p, gamma a power of two chosen at
// every reliable update so that the entries of gamma r have unit root mean
// square: CG's alpha and beta do not change under a common scaling of r and
// p, and 16-bit storage keeps the shrinking residual within its exponent
// range.  rr holds |gamma r|^2.
__global__ void k_cg_restart_check(const double2* __restrict__ rr_sum, double* __restrict__ rr,
                                   double* __restrict__ beta, double* __restrict__ gam,
                                   const double* __restrict__ bnorm, double n_elems, double tol,
                                   int init, SolverStatus* st) {
  if (st->error) return;
  double rn = rr_sum[0].x;  // true |r|^2
  double rel = sqrt(rn) / bnorm[0];
  st->true_res_max = rel;
  st->res_max = rel;
  st->res_at_ru = rel;
  if (!isfinite(rn)) {
    st->error = BLOCKCG_ERR_NONFINITE;
    return;
  }
  if (rel <= tol) {
    st->done = 1;
    return;
  }
  const double g_new = exp2(rint(log2(sqrt(n_elems / rn))));
  // p = r + beta p with beta from the true residual (p = r at the start);
  // in scaled form gamma' p' = gamma' r + beta (gamma' / gamma) (gamma p)
  const double g_old = *gam;
  *beta = init ? 0.0 : (rn * g_old * g_old / *rr) * (g_new / g_old);
  *rr = rn * g_new * g_new;
  *gam = g_new;
  st->ru_pending = 0;
}

cudaError_t cg_restart_check(const double2* rr_sum, double* rr, double* beta, double* gam,
                             const double* bnorm, double n_elems, double tol, int init,
                             SolverStatus* st, cudaStream_t s) {
  k_cg_restart_check<<<1, 1, 0, s>>>(rr_sum, rr, beta, gam, bnorm, n_elems, tol, init, st);
  return cudaGetLastError();
}

}  // namespace bcg
