// k_lanczos.cu -- spectral truncation Q ~= V V^H, V = [sqrt(lambda_j) u_j]
// (Sec. 4.1, Algorithm 3): the r largest (algebraic) eigenpairs of a
// Hermitian operator by FP64 Lanczos on the GPU.
//
// Operators: a dense Hermitian complex128 matrix, or the Laplacian
// L = D - A of a graph given as symmetric CSR (optional edge weights),
// applied matrix-free (self loops cancel in D - A and are skipped).
//
// Method (the paper calls ARPACK; this is a Lanczos of our own design):
//   * Lanczos with full reorthogonalisation: after w = Q u_j, w is projected
//     off u_j and u_{j-1} (the three-term step, which removes its large
//     components) and then off every stored vector (one classical
//     Gram-Schmidt pass over components of rounding size); alpha_j =
//     u_j^H Q u_j is the sum of the two projections onto u_j, and
//     beta_j = ||w||.  The tridiagonal T_J is real for Hermitian Q.
//   * Convergence, on the host beside the next GPU steps: eigenvalues of T_J
//     by multisection on Sturm counts, their eigenvectors by inverse
//     iteration (Gaussian elimination with partial pivoting), residual
//     ||Q y - theta y|| = beta_{J-1} |x_{J-1}|.
//   * Locking: converged Ritz vectors are stored in front of the Krylov
//     basis and every later vector is orthogonalised against them, so that a
//     new run (fresh random start) sees only the rest of the spectrum.  A
//     single-vector Krylov space holds one vector per eigenspace; "check"
//     runs repeat until the largest remaining eigenvalue is not above the
//     r-th locked one, which recovers every copy of a repeated eigenvalue
//     that belongs to the top r.
// Vectors are stored column-major (each basis vector contiguous, n doubles
// or complex doubles); the projections are tall-skinny GEMV pairs over
// row chunks with a fixed-order reduction (deterministic).  A step is five
// launches: operator (with the projections on the last two vectors),
// three-term step, projections, their subtraction (with the norm, alpha and
// beta), scaling; the last block of a kernel to finish adds its block sums.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstring>
#include <utility>
#include <vector>

#include "lanczos_host.h"
#include "lrq_device.cuh"
#include "lrq_internal.h"

namespace lrq {

constexpr int kLzThreads = 256;
constexpr int kLzChunkMax = 4096;  // rows per block in lz_dots (at most; at least four a thread)
constexpr int kLzDotThreads = 128;
constexpr int kLzGroup = 8;        // basis vectors per block in lz_dots
constexpr int kLzMvThreads = 64;   // lz_matvec_dense
constexpr int kLzMaxBlocks = 152 * 16;  // blocks that leave a partial sum (matvec, three-term step, update)
constexpr int kLzWant = kMaxRank;  // at most 8 wanted pairs per run
constexpr int kLzMaxIter = 4096;
constexpr int kLzDefaultIter = 500;
constexpr int kLzLag = 2;          // Lanczos steps run while a convergence check is in flight

// ---------------------------------------------------------------------------
// scalar helpers: real (graph Laplacian) and complex (dense Hermitian) paths
// ---------------------------------------------------------------------------
__device__ __forceinline__ double2 lz_mul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double lz_scale(double a, double s) { return a * s; }
__device__ __forceinline__ double2 lz_scale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
__device__ __forceinline__ void lz_add(double& a, double b) { a += b; }
__device__ __forceinline__ void lz_add(double2& a, double2 b) {
  a.x += b.x;
  a.y += b.y;
}
__device__ __forceinline__ void lz_sub(double& a, double b) { a -= b; }
__device__ __forceinline__ void lz_sub(double2& a, double2 b) {
  a.x -= b.x;
  a.y -= b.y;
}
__device__ __forceinline__ double lz_re(double a) { return a; }
__device__ __forceinline__ double lz_re(double2 a) { return a.x; }
template <typename T>
__device__ __forceinline__ T lz_zero();
template <>
__device__ __forceinline__ double lz_zero<double>() { return 0.0; }
template <>
__device__ __forceinline__ double2 lz_zero<double2>() { return make_double2(0.0, 0.0); }
__device__ __forceinline__ double lz_shfl_xor(double v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
__device__ __forceinline__ double2 lz_shfl_xor(double2 v, int m) {
  return make_double2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}
template <typename T>
__device__ __forceinline__ T lz_warp_sum(T v) {
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) lz_add(v, lz_shfl_xor(v, m));
  return v;
}
__device__ __forceinline__ double2 lz_as_complex(double a) { return make_double2(a, 0.0); }
__device__ __forceinline__ double2 lz_as_complex(double2 a) { return a; }
__device__ __forceinline__ double lz_real_or_gauss(double, double g0, double) { return g0; }
__device__ __forceinline__ double2 lz_real_or_gauss(double2, double g0, double g1) { return make_double2(g0, g1); }

__device__ __forceinline__ double lz_neg(double a) { return -a; }
__device__ __forceinline__ double2 lz_neg(double2 a) { return make_double2(-a.x, -a.y); }
__device__ __forceinline__ double lz_scale_fma(double a, double s, double c) { return fma(a, s, c); }
__device__ __forceinline__ double2 lz_scale_fma(double2 a, double s, double2 c) {
  return make_double2(fma(a.x, s, c.x), fma(a.y, s, c.y));
}
__device__ __forceinline__ double lz_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double2 lz_fma(double2 a, double2 b, double2 c) {  // a b + c, four FMAs
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}
__device__ __forceinline__ double lz_cfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double2 lz_cfma(double2 a, double2 b, double2 c) {  // conj(a) b + c
  return make_double2(fma(a.x, b.x, fma(a.y, b.y, c.x)), fma(a.x, b.y, fma(-a.y, b.x, c.y)));
}
__device__ __forceinline__ double lz_abs2_fma(double a, double c) { return fma(a, a, c); }
__device__ __forceinline__ double lz_abs2_fma(double2 a, double c) { return fma(a.x, a.x, fma(a.y, a.y, c)); }

// Sums N values over the warp: at each step half of the values change lanes,
// so that N + log2(32 / N) additions a lane do what a butterfly per value
// does with 5 N (an FP64 addition of a warp holds the SM's two-lane FP64 unit
// for 16 cycles).  The total of value v ends in the lanes whose upper
// log2(N) bits, read from the top, are v; `mine` tells which one a lane has.
template <int N, typename T>
__device__ __forceinline__ T lz_warp_sums(T (&v)[N], int* mine) {
  const int lane = threadIdx.x & 31;
  int id = 0, m = 16;
#pragma unroll
  for (int k = N / 2; k > 0; k >>= 1, m >>= 1) {
    const bool up = lane & m;
#pragma unroll
    for (int q = 0; q < k; ++q) {
      const T give = up ? v[q] : v[k + q];
      T keep = up ? v[k + q] : v[q];
      lz_add(keep, lz_shfl_xor(give, m));
      v[q] = keep;
    }
    id = 2 * id + (up ? 1 : 0);
  }
#pragma unroll
  for (int q = 16; q > 0; q >>= 1)
    if (q <= m) lz_add(v[0], lz_shfl_xor(v[0], q));
  *mine = id;
  return v[0];
}

// Whether this block is the last of `count` to arrive at the counter (which
// returns to zero): every block's earlier global writes are then visible to
// it.  All threads of the block call it.
__device__ __forceinline__ bool lz_last_block(unsigned* counter, unsigned count) {
  __shared__ int last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicInc(counter, count - 1) == count - 1;
  __syncthreads();
  if (last) __threadfence();
  return last != 0;
}

// Sum of part[0..count) by the whole block in a fixed order (every thread
// gets it); NT threads.
template <int NT, typename T>
__device__ __forceinline__ T lz_block_total(const T* part, int count) {
  __shared__ T red[NT / 32];
  T s = lz_zero<T>();
#pragma unroll 8
  for (int k = threadIdx.x; k < count; k += NT) lz_add(s, __ldcg(part + k));  // other blocks' writes: from L2
  s = lz_warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  T t = red[0];
  for (int k = 1; k < NT / 32; ++k) lz_add(t, red[k]);
  __syncthreads();
  return t;
}

// Device state of one Lanczos run.
struct LzState {
  int stop;        // set on breakdown (invariant subspace reached)
  int jdone;       // Lanczos vectors whose alpha and beta are known
  double tnorm;    // running estimate of ||T||
  double inv_beta;
  double wnorm2;   // ||w||^2 after the three-term step (lz_threeterm)
};

// What a convergence check needs (lz_snapshot), in front of alpha and beta.
struct LzSnap {
  int stop, jdone, status, pad;
};

// Verdict of a convergence check (host).
struct LzCheck {
  int J;
  int converged;
  int breakdown;
  int nvalid;
  double tnorm;
  double theta[kLzWant];
  double res[kLzWant];
};

// ---------------------------------------------------------------------------
// operators
// ---------------------------------------------------------------------------
// Every operator also leaves the projections of y on the last two basis
// vectors, h1[0] = u_prev^H y (when there is one) and h1[1] = x^H y: the
// block sums meet in the last block to finish, in block order.
template <int NT, typename T>
__device__ __forceinline__ void lz_two_dots(T d0, T d1, T* __restrict__ part, unsigned* counter, int has_prev,
                                            T* __restrict__ h1) {
  __shared__ T red[2][NT / 32];
  T v[2] = {d0, d1};
  int mine;
  const T t = lz_warp_sums<2>(v, &mine);
  if ((threadIdx.x & 15) == 0) red[mine][threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x < 2) {
    T s = red[threadIdx.x][0];
    for (int k = 1; k < NT / 32; ++k) lz_add(s, red[threadIdx.x][k]);
    part[threadIdx.x * kLzMaxBlocks + blockIdx.x] = s;
  }
  if (!lz_last_block(counter, gridDim.x)) return;
  for (int q = has_prev ? 0 : 1; q < 2; ++q) {
    const T s = lz_block_total<NT>(part + q * kLzMaxBlocks, static_cast<int>(gridDim.x));
    if (threadIdx.x == 0) h1[q] = s;
  }
}

// y = L x = D x - A x for the graph Laplacian, a thread per row: the
// weighted degrees D are precomputed (lz_degree), so a row costs one FP64
// add or FMA per stored edge (GB300's FP64 rate, not memory, bounds this
// operator).  Self loops are skipped, out-of-range columns ignored (they are
// reported by lz_check_csr).
__global__ void __launch_bounds__(kLzThreads) lz_matvec_laplacian(
    const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx, const double* __restrict__ wts,
    const double* __restrict__ deg, int64_t n, int64_t nnz, const double* __restrict__ x, double* __restrict__ y,
    const double* __restrict__ uprev, double* __restrict__ part, unsigned* counter, double* __restrict__ h1,
    const LzState* st) {
  if (st->stop) return;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  double d0 = 0.0, d1 = 0.0;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) {
    int64_t k0 = rowptr[i], k1 = rowptr[i + 1];
    k0 = k0 < 0 ? 0 : (k0 > nnz ? nnz : k0);
    k1 = k1 < k0 ? k0 : (k1 > nnz ? nnz : k1);
    double acc = 0.0;
    for (int64_t k = k0; k < k1; ++k) {
      const int32_t j = colidx[k];
      if (j < 0 || j >= n || j == i) continue;
      acc = wts ? fma(wts[k], x[j], acc) : acc + x[j];
    }
    const double xi = x[i], yi = fma(deg[i], xi, -acc);
    y[i] = yi;
    if (uprev) d0 = fma(uprev[i], yi, d0);
    d1 = fma(xi, yi, d1);
  }
  lz_two_dots<kLzThreads>(d0, d1, part, counter, uprev != nullptr, h1);
}

// deg[i] = sum of the row's edge weights (self loops and invalid columns
// skipped), once per truncation
__global__ void __launch_bounds__(kLzThreads) lz_degree(const int32_t* __restrict__ rowptr,
                                                        const int32_t* __restrict__ colidx,
                                                        const double* __restrict__ wts, int64_t n, int64_t nnz,
                                                        double* __restrict__ deg) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) {
    int64_t k0 = rowptr[i], k1 = rowptr[i + 1];
    k0 = k0 < 0 ? 0 : (k0 > nnz ? nnz : k0);
    k1 = k1 < k0 ? k0 : (k1 > nnz ? nnz : k1);
    double d = 0.0;
    for (int64_t k = k0; k < k1; ++k) {
      const int32_t j = colidx[k];
      if (j < 0 || j >= n || j == i) continue;
      d += wts ? wts[k] : 1.0;
    }
    deg[i] = d;
  }
}

// y = Q x for dense Hermitian Q (row-major, leading dimension ld): a warp
// takes ROWS rows at a time, so that one load of x serves ROWS of them.
// Bound: FP64 (four FMAs an entry, 16 cycles a warp instruction: 108 us at
// n = 4096 with all SMs equally loaded; the 268 MB take 40).  Two rows a warp
// and two warps a block: 4096 rows are 1024 blocks, 6.7 an SM, so the fullest
// SM has 28 rows where the average has 27 (blocks of sixteen rows: 32).
// Runs for n < 1024 and n > 32768 (lz_matvec_fixed between).  n = 4096: 143 us with
// the two projections; 230 us without them before (a row
// per warp, six FP64 instructions an entry).
template <int ROWS>
__global__ void __launch_bounds__(kLzMvThreads) lz_matvec_dense(
    const double2* __restrict__ Q, int64_t n, int64_t ld, const double2* __restrict__ x, double2* __restrict__ y,
    const double2* __restrict__ uprev, double2* __restrict__ part, unsigned* counter, double2* __restrict__ h1,
    const LzState* st) {
  if (st->stop) return;
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = static_cast<int64_t>(gridDim.x) * (kLzMvThreads / 32);
  double2 d0 = make_double2(0.0, 0.0), d1 = d0;
  for (int64_t i0 = ((static_cast<int64_t>(blockIdx.x) * kLzMvThreads + threadIdx.x) >> 5) * ROWS; i0 < n;
       i0 += nwarps * ROWS) {
    const double2* row[ROWS];
    double2 acc[ROWS];
#pragma unroll
    for (int q = 0; q < ROWS; ++q) {
      row[q] = Q + min(i0 + q, n - 1) * ld;
      acc[q] = make_double2(0.0, 0.0);
    }
#pragma unroll(ROWS == 1 ? 2 : 4)
    for (int64_t j = lane; j < n; j += 32) {
      const double2 xj = x[j];
#pragma unroll
      for (int q = 0; q < ROWS; ++q) acc[q] = lz_fma(row[q][j], xj, acc[q]);
    }
    int mine = 0;
    double2 v = lz_warp_sums<ROWS>(acc, &mine);
    // row `mine`'s total is in this lane; one lane per row goes on
    const int64_t i = i0 + mine;
    if ((lane & (32 / ROWS - 1)) == 0 && i < n) {
      y[i] = v;
      if (uprev) d0 = lz_cfma(uprev[i], v, d0);
      d1 = lz_cfma(x[i], v, d1);
    }
  }
  lz_two_dots<kLzMvThreads>(d0, d1, part, counter, uprev != nullptr, h1);
}

// ---------------------------------------------------------------------------
// the dense operator in fixed point
// ---------------------------------------------------------------------------
// Four FP64 FMAs an entry keep the dense operator (141 us at n = 4096) well
// above its bytes (40 us).  Here Q's entries are 55-bit integers relative to
// their row's largest component (off by 2^-54 of it at most) and the unit
// vector's are 63-bit integers, both cut into signed bytes (seven and eight
// base-256 digits d and j, the most significant first).  The digit products with
// d + j <= 7 are summed exactly by 4-way byte dot products, by d + j; the others
// are below 2^-59 of the largest product.  FP64 only joins a row's sums.
// The error is bounded by the row: |y_i - (Q x)_i| is at most 2^-54 max_j |Q_ij|
// ||x||_1 (the entries) plus 2^-57 n max_j |Q_ij| (x, the dropped digit pairs),
// where FP64 FMAs, whose partial sums round at every entry, are off by some 2^-53
// of them.  On rows of similar entries it is no larger (eigenvalues and residuals
// of random Q agree with LAPACK's as well as in FP64); entries far below their
// row's largest keep fewer bits, and such a row loses to FP64 where x is small at
// its largest ones.  Lanczos needs the bound by ||Q||.  Q's digits are laid out once
// per truncation (14 bytes an entry for 16), a vector's by the kernel that
// normalises it.  (The 8-bit matrix instruction has the rate of the byte dot
// products here and takes all 56 digit pairs: 91 us.)
constexpr int kLzQDigits = 7, kLzXDigits = 8;
constexpr int kLzFixThreads = 256;  // laying out
constexpr int kLzFixRows = 4;       // rows a warp
// Smaller matrices leave SMs without rows; above, the sums of 8 digit pairs of 2 n
// products of at most 2^14, times 2^24, would leave 63 bits.  The digits take
// nearly as much memory as Q: a workspace without room for them gets the FP64
// operator.  Truncations with the digits / in FP64, r = 4: n = 1024 13.3 / 14.4 ms
// (252 steps), 2048 21.3 / 25.2 (316), 4096 37.2 / 68.3 (364), 200 steps at 8192
// 54 / 109, 16384 154 / 441, 32768 615 / 1599.
constexpr int64_t kLzFixMin = 1024, kLzFixMax = 32768;

struct LzFixed {
  int64_t units, steps;  // of four rows, of 128 columns
  size_t qbytes, xbytes;
};
inline LzFixed lz_fixed(int64_t n) {
  LzFixed f;
  f.units = ceil_div(n, kLzFixRows);
  f.steps = ceil_div(n, 128);
  f.qbytes = static_cast<size_t>(f.units * f.steps) * 2 * kLzQDigits * 512;
  f.xbytes = static_cast<size_t>(f.steps) * 3 * kLzXDigits * 128;
  return f;
}
inline bool lz_use_fixed(int64_t n) { return n >= kLzFixMin && n <= kLzFixMax; }

// rowexp[i]: biased exponent of the row's largest component (0 for padding),
// and the input check; a warp per row.
__global__ void __launch_bounds__(kLzFixThreads) lz_row_exponents(const double2* __restrict__ Q, int64_t n, int64_t ld,
                                                                  int64_t rows, int32_t* __restrict__ rowexp,
                                                                  int32_t* status) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (static_cast<int64_t>(blockIdx.x) * kLzFixThreads + threadIdx.x) >> 5;
  uint32_t mx = 0;
  if (i < n) {
#pragma unroll 4
    for (int64_t j = lane; j < n; j += 32) {
      const double2 q = Q[i * ld + j];
      mx = max(mx, max(static_cast<uint32_t>(__double2hiint(q.x)) & 0x7fffffffu,
                       static_cast<uint32_t>(__double2hiint(q.y)) & 0x7fffffffu));
    }
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane != 0 || i >= rows) return;
  if ((mx >> 20) == 0x7ffu) dev_fail(status, LRQ_EINVAL);
  rowexp[i] = static_cast<int32_t>(mx >> 20);
}

// digits of x 2^(1076 - E) to the nearest integer, |x| < 2^(E - 1022): the bytes
// of the result are signed, the most significant in byte 6
__device__ __forceinline__ uint64_t lz_q_digits(double x, int E) {
  const uint64_t b = static_cast<uint64_t>(__double_as_longlong(x));
  const int ex = static_cast<int>(b >> 52) & 0x7ff;
  uint64_t m = (b & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0ull);
  const int s = max(ex, 1) + 1 - E;  // value = m 2^s, s <= 2
  if (s >= 0)
    m <<= min(s, 2);
  else
    m = s < -54 ? 0ull : (m + (1ull << (-s - 1))) >> -s;
  const int64_t v = (b >> 63) ? -static_cast<int64_t>(m) : static_cast<int64_t>(m);
  return static_cast<uint64_t>(v + 0x0080808080808080ll) ^ 0x0080808080808080ull;
}

// byte k of four values
__device__ __forceinline__ uint32_t lz_byte4(const uint64_t (&u)[4], int k) {
  const int sh = 32 * (k >> 2), sel = (k & 3) * 0x11 + 0x40;
  const uint32_t a = __byte_perm(static_cast<uint32_t>(u[0] >> sh), static_cast<uint32_t>(u[1] >> sh), sel);
  const uint32_t c = __byte_perm(static_cast<uint32_t>(u[2] >> sh), static_cast<uint32_t>(u[3] >> sh), sel);
  return __byte_perm(a, c, 0x5410);
}

// Q's digits: [4 rows][128 columns][re, im][digit][lane] 16 bytes, a word (the
// lane's four columns) per row.  A thread per lane.
__global__ void __launch_bounds__(kLzFixThreads) lz_dense_digits(const double2* __restrict__ Q, int64_t n, int64_t ld,
                                                                 int64_t units, int64_t steps,
                                                                 const int32_t* __restrict__ rowexp,
                                                                 uint4* __restrict__ out) {
  const int64_t id = static_cast<int64_t>(blockIdx.x) * kLzFixThreads + threadIdx.x;
  const int64_t tile = id >> 5;
  if (tile >= units * steps) return;
  const int lane = threadIdx.x & 31;
  const int64_t i0 = tile / steps * kLzFixRows, j0 = tile % steps * 128 + lane * 4;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    uint64_t u[kLzFixRows][4];
#pragma unroll
    for (int q = 0; q < kLzFixRows; ++q) {
      const int64_t i = i0 + q;
      const int E = rowexp[i];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        double x = 0.0;
        if (i < n && j0 + e < n) x = c == 0 ? Q[i * ld + j0 + e].x : Q[i * ld + j0 + e].y;
        u[q][e] = lz_q_digits(x, E);
      }
    }
#pragma unroll
    for (int d = 0; d < kLzQDigits; ++d)
      out[(tile * 2 * kLzQDigits + c * kLzQDigits + d) * 32 + lane] =
          make_uint4(lz_byte4(u[0], kLzQDigits - 1 - d), lz_byte4(u[1], kLzQDigits - 1 - d),
                     lz_byte4(u[2], kLzQDigits - 1 - d), lz_byte4(u[3], kLzQDigits - 1 - d));
  }
}

// Digits of entry i of a unit vector, |x| <= 1: x 2^62 to the nearest integer.
// Per 128 entries, 24 words a lane (its four entries), six 16-byte groups of 32
// lanes: the digits of re, of im, of -im.
__device__ __forceinline__ void lz_store_digits(uint8_t* xs, int64_t i, double2 x) {
  const double two62 = 4611686018427387904.0;
  const int64_t v[3] = {__double2ll_rn(x.x * two62), __double2ll_rn(x.y * two62), __double2ll_rn(x.y * -two62)};
  uint8_t* p = xs + (i >> 7) * (3 * kLzXDigits * 128) + ((i & 127) >> 2) * 16 + (i & 3);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const uint64_t u = (static_cast<uint64_t>(v[c]) + 0x8080808080808080ull) ^ 0x8080808080808080ull;
#pragma unroll
    for (int j = 0; j < kLzXDigits; ++j) {
      const int w = c * kLzXDigits + j;
      p[(w >> 2) * 512 + (w & 3) * 4] = static_cast<uint8_t>(u >> (8 * (kLzXDigits - 1 - j)));
    }
  }
}
__device__ __forceinline__ void lz_store_digits(uint8_t*, int64_t, double) {}

// Sums 16 integers over the warp, halving the values at every step: lane l ends
// with the total of value l >> 1.
__device__ __forceinline__ int64_t lz_warp_sums16(int64_t (&v)[16]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 8, m = 16; k > 0; k >>= 1, m >>= 1) {
    const bool up = lane & m;
#pragma unroll
    for (int q = 0; q < k; ++q) {
      const int64_t give = up ? v[q] : v[k + q], keep = up ? v[k + q] : v[q];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, give, m);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// y = Q x from the digits, four rows a warp and one warp a block (n = 4096: 1024
// blocks, at most seven an SM where the average is 6.7).  Per step of 128
// columns 7 KB of Q (the next step's loads in flight) and 560 byte dot products,
// which take two cycles each.  Bound: these (31 us at n = 4096) and the 14 bytes
// an entry (35 us).  n = 4096: 61 us, 141 in FP64; n = 1024: 15, 18.5.
__global__ void __launch_bounds__(32) lz_matvec_fixed(
    const uint4* __restrict__ Qd, const int32_t* __restrict__ rowexp, int64_t n, int units, int steps,
    const uint4* __restrict__ xs, const double2* __restrict__ x, double2* __restrict__ y,
    const double2* __restrict__ uprev, double2* __restrict__ part, unsigned* counter, double2* __restrict__ h1,
    const LzState* st) {
  if (st->stop) return;
  constexpr int ND = kLzQDigits, NX = kLzXDigits, NR = kLzFixRows;
  const int lane = threadIdx.x;
  double2 d0 = make_double2(0.0, 0.0), d1 = d0;
  for (int un = blockIdx.x; un < units; un += gridDim.x) {
    int acc[NR][2][NX];  // re, im by d + j
#pragma unroll
    for (int q = 0; q < NR; ++q)
#pragma unroll
      for (int g = 0; g < NX; ++g) acc[q][0][g] = acc[q][1][g] = 0;
    const uint4* qa = Qd + static_cast<int64_t>(un) * steps * (2 * ND * 32) + lane;
    uint4 a[2 * ND];
#pragma unroll
    for (int d = 0; d < 2 * ND; ++d) a[d] = __ldcs(qa + d * 32);
#pragma unroll 1
    for (int s = 0; s < steps; ++s) {
      uint32_t xw[3][NX];
#pragma unroll
      for (int g = 0; g < 6; ++g) {
        const uint4 v = xs[(s * 6 + g) * 32 + lane];
        xw[g >> 1][(g & 1) * 4] = v.x;
        xw[g >> 1][(g & 1) * 4 + 1] = v.y;
        xw[g >> 1][(g & 1) * 4 + 2] = v.z;
        xw[g >> 1][(g & 1) * 4 + 3] = v.w;
      }
      uint4 an[2 * ND];
      const uint4* qn = qa + static_cast<int64_t>(s + 1 < steps ? s + 1 : s) * (2 * ND * 32);
#pragma unroll
      for (int d = 0; d < 2 * ND; ++d) an[d] = __ldcs(qn + d * 32);
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        const uint32_t re[NR] = {a[d].x, a[d].y, a[d].z, a[d].w};
        const uint32_t im[NR] = {a[ND + d].x, a[ND + d].y, a[ND + d].z, a[ND + d].w};
#pragma unroll
        for (int j = 0; j + d < NX; ++j)
#pragma unroll
          for (int q = 0; q < NR; ++q) {
            acc[q][0][d + j] = __dp4a(static_cast<int>(re[q]), static_cast<int>(xw[0][j]), acc[q][0][d + j]);
            acc[q][1][d + j] = __dp4a(static_cast<int>(re[q]), static_cast<int>(xw[1][j]), acc[q][1][d + j]);
            acc[q][0][d + j] = __dp4a(static_cast<int>(im[q]), static_cast<int>(xw[2][j]), acc[q][0][d + j]);
            acc[q][1][d + j] = __dp4a(static_cast<int>(im[q]), static_cast<int>(xw[0][j]), acc[q][1][d + j]);
          }
      }
#pragma unroll
      for (int d = 0; d < 2 * ND; ++d) a[d] = an[d];
    }
    // sum_g acc_g 256^(13 - g), in two halves
    int64_t v[16];
#pragma unroll
    for (int q = 0; q < NR; ++q)
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          v[q * 4 + c * 2 + h] = static_cast<int64_t>(acc[q][c][4 * h]) * 16777216 +
                                 static_cast<int64_t>(acc[q][c][4 * h + 1]) * 65536 +
                                 static_cast<int64_t>(acc[q][c][4 * h + 2]) * 256 + acc[q][c][4 * h + 3];
    double t = static_cast<double>(lz_warp_sums16(v));  // lane: row lane / 8, re or im (bit 2), half (bit 1)
    t = fma(t, 4294967296.0, __shfl_xor_sync(0xffffffffu, t, 2));  // meaningful in the upper half's lanes
    const int64_t i = static_cast<int64_t>(un) * NR + (lane >> 3);
    // 256^6 2^(E - 1076) 2^-62
    t = scalbn(t, rowexp[i] - 1090);
    const double im = __shfl_xor_sync(0xffffffffu, t, 4);
    if ((lane & 7) == 0 && i < n) {
      const double2 yi = make_double2(t, im);
      y[i] = yi;
      if (uprev) d0 = lz_cfma(uprev[i], yi, d0);
      d1 = lz_cfma(x[i], yi, d1);
    }
  }
  lz_two_dots<32>(d0, d1, part, counter, uprev != nullptr, h1);
}

// ---------------------------------------------------------------------------
// projections
// ---------------------------------------------------------------------------
// The three-term step, w -= u_prev h1[0] + u h1[1] (uprev NULL: the second
// only), and ||w||^2 after it.
template <typename T>
__global__ void __launch_bounds__(kLzThreads) lz_threeterm(T* __restrict__ w, int64_t n, const T* __restrict__ uprev,
                                                           const T* __restrict__ u, const T* __restrict__ h1,
                                                           double* __restrict__ npart, unsigned* counter,
                                                           LzState* st) {
  if (st->stop) return;
  __shared__ double red[kLzThreads / 32];
  const int64_t stride = static_cast<int64_t>(gridDim.x) * kLzThreads;
  const T h0 = uprev ? lz_neg(h1[0]) : lz_zero<T>(), hc = lz_neg(h1[1]);
  double s = 0.0;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * kLzThreads + threadIdx.x; i < n; i += stride) {
    T v = w[i];
    if (uprev) v = lz_fma(uprev[i], h0, v);
    v = lz_fma(u[i], hc, v);
    w[i] = v;
    s = lz_abs2_fma(v, s);
  }
  s = lz_warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = red[0];
    for (int k = 1; k < kLzThreads / 32; ++k) t += red[k];
    npart[blockIdx.x] = t;
  }
  if (!lz_last_block(counter, gridDim.x)) return;
  const double t = lz_block_total<kLzThreads>(npart, static_cast<int>(gridDim.x));
  if (threadIdx.x == 0) st->wnorm2 = t;
}

// h[c] = U_c^H w for basis vectors c in [0, nc): a block takes one row chunk
// and 8 vectors, and the last block of a group of vectors adds the group's
// chunk sums in chunk order.  grid = (nch, ceil(nc / 8)).  Bound: FP64 (one
// FMA per entry for real vectors, four for complex).  Per thread 26 rows x 8
// FMAs and 9 additions at n = 10^6; a butterfly per vector cost 40.  n = 10^6,
// 80 vectors: 176 us, 241 before.
template <typename T>
__global__ void __launch_bounds__(kLzDotThreads) lz_dots(const T* __restrict__ U, int64_t n, int nc,
                                                         const T* __restrict__ w, T* __restrict__ partial, int nch,
                                                         int chunk_rows, unsigned* counter, T* __restrict__ h,
                                                         const LzState* st) {
  if (st->stop) return;
  __shared__ T red[kLzGroup][kLzDotThreads / 32];
  const int chunk = blockIdx.x;
  const int cg = blockIdx.y * kLzGroup;
  const int64_t i0 = static_cast<int64_t>(chunk) * chunk_rows;
  const int64_t i1 = min(n, i0 + chunk_rows);
  T acc[kLzGroup];
#pragma unroll
  for (int q = 0; q < kLzGroup; ++q) acc[q] = lz_zero<T>();
  const int ncols = min(kLzGroup, nc - cg);
  const T* Ug = U + static_cast<int64_t>(cg) * n;
  if (ncols == kLzGroup) {
#pragma unroll 2
    for (int64_t i = i0 + threadIdx.x; i < i1; i += kLzDotThreads) {
      const T wi = w[i];
#pragma unroll
      for (int q = 0; q < kLzGroup; ++q) acc[q] = lz_cfma(Ug[static_cast<int64_t>(q) * n + i], wi, acc[q]);
    }
  } else {
    for (int64_t i = i0 + threadIdx.x; i < i1; i += kLzDotThreads) {
      const T wi = w[i];
#pragma unroll
      for (int q = 0; q < kLzGroup; ++q)
        if (q < ncols) acc[q] = lz_cfma(Ug[static_cast<int64_t>(q) * n + i], wi, acc[q]);
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int mine;
  const T v = lz_warp_sums<kLzGroup>(acc, &mine);
  if ((lane & 3) == 0) red[mine][warp] = v;
  __syncthreads();
  if (threadIdx.x < ncols) {
    T s = red[threadIdx.x][0];
    for (int k = 1; k < kLzDotThreads / 32; ++k) lz_add(s, red[threadIdx.x][k]);
    partial[static_cast<int64_t>(cg + threadIdx.x) * nch + chunk] = s;
  }
  if (!lz_last_block(counter + blockIdx.y, gridDim.x)) return;
  for (int q = warp; q < ncols; q += kLzDotThreads / 32) {
    const T* pc = partial + static_cast<int64_t>(cg + q) * nch;
    T s = lz_zero<T>();
    for (int k = lane; k < nch; k += 32) lz_add(s, __ldcg(pc + k));
    s = lz_warp_sum(s);
    if (lane == 0) h[cg + q] = s;
  }
}

// x rounded towards zero to FP32 by integer operations (a conversion
// instruction runs on the slow FP64 unit); 0 below the FP32 normal range.
// For |x| < 2^127: the entries of unit vectors.
__device__ __forceinline__ float lz_to_float(double x) {
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)), lo = static_cast<uint32_t>(__double2loint(x));
  const uint32_t mag = (__funnelshift_l(lo, hi, 3) + 0x40000000u) & 0x7fffffffu;
  const bool tiny = (hi & 0x7fffffffu) < (897u << 20);
  return __uint_as_float(tiny ? 0u : ((hi & 0x80000000u) | mag));
}
// the same for any x: infinite from 2^127 on and for NaN
__device__ __forceinline__ float lz_to_float_sat(double x) {
  return (__double2hiint(x) & 0x7fffffff) >= (1150 << 20) ? INFINITY : lz_to_float(x);
}
__device__ __forceinline__ float2 lz_to_float_sat(double2 x) {
  return make_float2(lz_to_float_sat(x.x), lz_to_float_sat(x.y));
}
__device__ __forceinline__ float2 lz_to_float(double2 x) { return make_float2(lz_to_float(x.x), lz_to_float(x.y)); }
__device__ __forceinline__ float lz_fma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float2 lz_fma(float2 a, float2 b, float2 c) {
  return make_float2(fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x)), fmaf(a.x, b.y, fmaf(a.y, b.x, c.y)));
}
__device__ __forceinline__ float lz_abs1(float a) { return fabsf(a); }
__device__ __forceinline__ float lz_abs1(float2 a) { return fabsf(a.x) + fabsf(a.y); }
__device__ __forceinline__ void lz_add(float& a, float b) { a += b; }
__device__ __forceinline__ void lz_add(float2& a, float2 b) {
  a.x += b.x;
  a.y += b.y;
}
// w + neg s
__device__ __forceinline__ double lz_add_scaled(double w, float s, double neg) {
  return fma(neg, static_cast<double>(s), w);
}
__device__ __forceinline__ double2 lz_add_scaled(double2 w, float2 s, double neg) {
  return make_double2(fma(neg, static_cast<double>(s.x), w.x), fma(neg, static_cast<double>(s.y), w.y));
}
template <typename T>
struct LzFloat;
template <>
struct LzFloat<double> {
  using type = float;
  __device__ static float zero() { return 0.f; }
};
template <>
struct LzFloat<double2> {
  using type = float2;
  __device__ static float2 zero() { return make_float2(0.f, 0.f); }
};

// One thread closes step j: beta_j = ||w||, alpha_j = Re(h1[1] + h2[c]) (c =
// column of u_j), breakdown test.  mode 1 = normalising a start vector (no
// alpha).
template <typename T>
__device__ void lz_finish(double nrm2, const T* __restrict__ h1, const T* __restrict__ h2, int c, int j, int mode,
                          double* __restrict__ alpha, double* __restrict__ beta, LzState* st) {
  const double b = sqrt(nrm2);
  if (mode == 1) {
    // start vector: b is its norm after projection; a zero vector means the
    // locked vectors already span the space
    if (!(b > 0.0)) {
      st->stop = 2;
      return;
    }
    st->inv_beta = 1.0 / b;
    return;
  }
  const double a = lz_re(h1[1]) + lz_re(h2[c]);
  alpha[j] = a;
  beta[j] = b;
  const double bprev = j > 0 ? beta[j - 1] : 0.0;
  st->tnorm = fmax(st->tnorm, fabs(a) + b + bprev);
  st->jdone = j + 1;
  if (!(b > 1e-12 * st->tnorm)) {
    st->stop = 1;  // invariant subspace: the Ritz values of T_{j+1} are exact
    return;
  }
  st->inv_beta = 1.0 / b;
}

// w -= sum_c U_c h[c], then the norm of w and (in the last block to finish)
// what lz_finish does with it: mode 0 closes step j (h1 and h2 = h: the two
// projections, c the column of u_j), mode 1 prepares a start vector, mode 2
// only subtracts.
//
// SL warps of a block share a tile of 256 / SL rows, each taking every SL-th
// vector: SL = 8 gives a small n enough warps (n = 4096: 128 tiles), SL = 1
// needs no exchange.
//
// After the three-term step w is orthogonal to every stored vector up to
// rounding, so h is of rounding size and the correction sum_c U_c h[c] needs
// no more than FP32 where sum |h_c| <= lz_fp32_gate(nc) ||w|| (checked here, ||w||
// from lz_threeterm; h is taken relative to the power of two below ||w||, so
// that the operator's scale does not matter): its error then moves w by less
// than 2^-52 ||w||, within the rounding of w itself.  U is then read through
// lz_to_float and the kernel is bound by HBM instead of FP64 (n = 10^6, 80
// vectors: 121 us, 206 in FP64).  Larger h (a start vector against locked
// vectors, a vector close to the span) takes the FP64 sum.
template <int SL, typename T>
__global__ void __launch_bounds__(kLzThreads) lz_update(const T* __restrict__ U, int64_t n, int nc,
                                                        const T* __restrict__ h, T* __restrict__ w,
                                                        double* __restrict__ npart, unsigned* counter, int mode,
                                                        int allow32, const T* __restrict__ h1,
                                                        int c, int j, double* __restrict__ alpha,
                                                        double* __restrict__ beta, LzState* st) {
  if (st->stop) return;
  using F = typename LzFloat<T>::type;
  extern __shared__ __align__(16) uint8_t lz_smem[];
  T* hs = reinterpret_cast<T*>(lz_smem);
  F* hf = reinterpret_cast<F*>(lz_smem + static_cast<size_t>(nc) * sizeof(T));
  __shared__ T part[SL][32];
  __shared__ double red[kLzThreads / 32];
  __shared__ float fred[kLzThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // 2^-floor(log2 ||w||) and its inverse; 0 outside the comfortable range
  double scale = 0.0, unscale = 0.0;
  if (allow32) {
    const double wn2 = st->wnorm2;
    if (wn2 > 0x1p-900 && wn2 < 0x1p900) {
      const int e = (__double2hiint(sqrt(wn2)) >> 20) - 1023;
      scale = __hiloint2double((1023 - e) << 20, 0);
      unscale = __hiloint2double((1023 + e) << 20, 0);
    }
  }
  float ha = 0.f;
  for (int q = threadIdx.x; q < nc; q += kLzThreads) {
    const T v = h[q];
    hs[q] = v;
    const F f = lz_to_float_sat(lz_scale(v, scale));
    hf[q] = f;
    ha += lz_abs1(f);
  }
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) ha += __shfl_xor_sync(0xffffffffu, ha, m);
  if (lane == 0) fred[warp] = ha;
  __syncthreads();
  bool f32 = false;
  if (scale > 0.0) {
    float t = 0.f;
    for (int k = 0; k < kLzThreads / 32; ++k) t += fred[k];
    f32 = t <= lz_fp32_gate(nc);
  }
  const int slice = SL == 1 ? 0 : warp;
  constexpr int TILE = kLzThreads / SL;
  const int rowin = SL == 1 ? static_cast<int>(threadIdx.x) : lane;
  double s2 = 0.0;
  for (int64_t r0 = static_cast<int64_t>(blockIdx.x) * TILE; r0 < n; r0 += static_cast<int64_t>(gridDim.x) * TILE) {
    const int64_t i = r0 + rowin;
    T t = lz_zero<T>();
    F tf = LzFloat<T>::zero();
    if (i < n) {
      const T* ui = U + i;
      if (f32) {
#pragma unroll 8
        for (int q = slice; q < nc; q += SL) tf = lz_fma(lz_to_float(ui[static_cast<int64_t>(q) * n]), hf[q], tf);
      } else {
#pragma unroll 4
        for (int q = slice; q < nc; q += SL) t = lz_fma(ui[static_cast<int64_t>(q) * n], hs[q], t);
      }
    }
    if constexpr (SL > 1) {
      if (f32)
        reinterpret_cast<F&>(part[slice][lane]) = tf;
      else
        part[slice][lane] = t;
      __syncthreads();
      if (slice == 0) {
        for (int k = 1; k < SL; ++k) {
          if (f32)
            lz_add(tf, reinterpret_cast<F&>(part[k][lane]));
          else
            lz_add(t, part[k][lane]);
        }
      }
    }
    if (slice == 0 && i < n) {
      T v = w[i];
      if (f32)
        v = lz_add_scaled(v, tf, -unscale);
      else
        lz_sub(v, t);
      w[i] = v;
      s2 = lz_abs2_fma(v, s2);
    }
    if constexpr (SL > 1) __syncthreads();
  }
  if (mode == 2) return;
  s2 = lz_warp_sum(s2);
  if (lane == 0) red[warp] = s2;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = red[0];
    for (int k = 1; k < kLzThreads / 32; ++k) t += red[k];
    npart[blockIdx.x] = t;
  }
  if (!lz_last_block(counter, gridDim.x)) return;
  const double nrm2 = lz_block_total<kLzThreads>(npart, static_cast<int>(gridDim.x));
  if (threadIdx.x == 0) lz_finish(nrm2, h1, h, c, j, mode, alpha, beta, st);
}

template <typename T>
__global__ void __launch_bounds__(kLzThreads) lz_scale_into(const T* __restrict__ w, int64_t n, T* __restrict__ u,
                                                            uint8_t* __restrict__ digits, const LzState* st) {
  if (st->stop) return;
  const double s = st->inv_beta;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) {
    const T v = lz_scale(w[i], s);
    u[i] = v;
    if (digits) lz_store_digits(digits, i, v);  // for lz_matvec_fixed
  }
}

// What a convergence check reads, in one piece: the state of the step just
// enqueued, alpha and beta of its J entries, the call's status.
__global__ void lz_snapshot(const LzState* __restrict__ st, const double* __restrict__ alpha,
                            const double* __restrict__ beta, int J, const int32_t* __restrict__ status,
                            LzSnap* __restrict__ out) {
  if (threadIdx.x == 0) {
    out->stop = st->stop;
    out->jdone = st->jdone;
    out->status = *status;
  }
  double* v = reinterpret_cast<double*>(out + 1);
  for (int i = threadIdx.x; i < J; i += blockDim.x) {
    v[i] = alpha[i];
    v[J + i] = beta[i];
  }
}

// Gaussian start vector from Philox4x32-10: key = seed, counter =
// (lo32 i, hi32 i, run, 0x4C5A) (Box-Muller on two 53-bit uniforms).
template <typename T>
__global__ void __launch_bounds__(kLzThreads) lz_start(T* __restrict__ w, int64_t n, uint64_t seed, int run,
                                                       const LzState* st) {
  if (st->stop) return;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) {
    PhiloxOut o = philox4x32_10(static_cast<uint32_t>(i), static_cast<uint32_t>(static_cast<uint64_t>(i) >> 32),
                                static_cast<uint32_t>(run), 0x4C5Au, static_cast<uint32_t>(seed),
                                static_cast<uint32_t>(seed >> 32));
    const double u1 = uniform53(o.w[0], o.w[1]), u2 = uniform53(o.w[2], o.w[3]);
    const double rad = sqrt(-2.0 * log(u1));
    double sn, cs;
    sincospi(2.0 * u2, &sn, &cs);
    w[i] = lz_real_or_gauss(T(), rad * cs, rad * sn);
  }
}

// ---------------------------------------------------------------------------
// tridiagonal eigenproblem of T_J, on the host: the problem is a chain of a
// few hundred dependent divisions per shift, which one SM's FP64 unit takes
// milliseconds for (1.2 ms a check on average over n = 4096, up to 3.4 ms)
// and a host core tens of microseconds, while the GPU runs the next steps.
// ---------------------------------------------------------------------------
namespace {

constexpr int kLzShifts = 8;  // shifts counted side by side (independent division chains)

// Number of eigenvalues of T_J below each of the shifts (Sturm sequence of
// the LDL^T pivots; b2 = squared off-diagonals).
void lz_sturm(const double* a, const double* b2, int J, const double* x, double pivmin, int* cnt) {
  double d[kLzShifts];
  int c[kLzShifts];
  for (int q = 0; q < kLzShifts; ++q) {
    d[q] = a[0] - x[q];
    if (std::fabs(d[q]) < pivmin) d[q] = -pivmin;
    c[q] = d[q] < 0.0;
  }
  for (int i = 1; i < J; ++i) {
    const double ai = a[i], bi = b2[i - 1];
    for (int q = 0; q < kLzShifts; ++q) {
      double v = (ai - x[q]) - bi / d[q];
      v = std::fabs(v) < pivmin ? -pivmin : v;
      c[q] += v < 0.0;
      d[q] = v;
    }
  }
  for (int q = 0; q < kLzShifts; ++q) cnt[q] = c[q];
}

// (T - theta I) = P L U by Gaussian elimination with partial pivoting, then
// solves with it.
struct LzTriLu {
  std::vector<double> D, DL, DU, DU2;
  std::vector<char> swapped;
  void factor(const double* a, const double* b, int J, double theta, double pivtol) {
    D.assign(J, 0.0);
    DL.assign(J, 0.0);
    DU.assign(J, 0.0);
    DU2.assign(J, 0.0);
    swapped.assign(J, 0);
    for (int i = 0; i < J; ++i) {
      D[i] = a[i] - theta;
      if (i + 1 < J) DL[i] = DU[i] = b[i];
    }
    for (int i = 0; i + 1 < J; ++i) {
      if (std::fabs(D[i]) >= std::fabs(DL[i])) {
        if (std::fabs(D[i]) < pivtol) D[i] = D[i] < 0.0 ? -pivtol : pivtol;
        const double f = DL[i] / D[i];
        DL[i] = f;
        D[i + 1] -= f * DU[i];
      } else {
        const double f = D[i] / DL[i];
        D[i] = DL[i];
        DL[i] = f;
        const double t = DU[i];
        DU[i] = D[i + 1];
        D[i + 1] = t - f * D[i + 1];
        if (i + 2 < J) {
          DU2[i] = DU[i + 1];
          DU[i + 1] = -f * DU[i + 1];
        }
        swapped[i] = 1;
      }
    }
    if (std::fabs(D[J - 1]) < pivtol) D[J - 1] = D[J - 1] < 0.0 ? -pivtol : pivtol;
  }
  void solve(int J, double* x) const {
    for (int i = 0; i + 1 < J; ++i) {
      if (swapped[i]) std::swap(x[i], x[i + 1]);
      x[i + 1] -= DL[i] * x[i];
    }
    x[J - 1] /= D[J - 1];
    if (J > 1) x[J - 2] = (x[J - 2] - DU[J - 2] * x[J - 1]) / D[J - 2];
    for (int i = J - 3; i >= 0; --i) x[i] = (x[i] - DU[i] * x[i + 1] - DU2[i] * x[i + 2]) / D[i];
  }
};

void lz_normalize(double* x, int J) {
  double s = 0.0, mx = 0.0;
  for (int i = 0; i < J; ++i) mx = std::max(mx, std::fabs(x[i]));
  if (!(mx > 0.0)) {
    x[0] = 1.0;
    return;
  }
  for (int i = 0; i < J; ++i) {
    x[i] /= mx;
    s += x[i] * x[i];
  }
  s = 1.0 / std::sqrt(s);
  for (int i = 0; i < J; ++i) x[i] *= s;
}

// The p largest eigenvalues of T_J (multisection on Sturm counts), their
// eigenvectors X[w * J + k] (three rounds of inverse iteration, Gram-Schmidt
// inside clusters), residual bounds and the convergence verdict.  `out` holds
// the previous check of the same run on entry (nvalid = 0 at its first): its
// Ritz values and residuals give the first shifts, which narrows the interval
// but decides nothing.
void lz_tridiag(const double* a, const double* b, int J, int p, double tol, std::vector<double>* Xout,
                LzCheck* out) {
  const LzCheck prev = *out;
  double lo = INFINITY, hi = -INFINITY;  // Gershgorin interval
  std::vector<double> b2(J);
  for (int i = 0; i < J; ++i) {
    const double r = (i > 0 ? std::fabs(b[i - 1]) : 0.0) + (i + 1 < J ? std::fabs(b[i]) : 0.0);
    lo = std::min(lo, a[i] - r);
    hi = std::max(hi, a[i] + r);
    b2[i] = b[i] * b[i];
  }
  const double tn = std::max(std::max(std::fabs(lo), std::fabs(hi)), DBL_MIN);
  const double pivmin = DBL_MIN * std::max(1.0, tn * tn);
  const int nwant = std::min(p, J);
  double theta[kLzWant];
  for (int w = 0; w < nwant; ++w) {
    const int k = J - 1 - w;  // 0-based ascending index
    double l = lo - 1e-12 * tn - pivmin, h = hi + 1e-12 * tn + pivmin;
    for (int round = 0; round < 64; ++round) {
      if (h - l <= 4.0 * DBL_EPSILON * std::max(std::fabs(l), std::fabs(h)) + pivmin) break;
      double x[kLzShifts];
      int cnt[kLzShifts];
      if (round == 0 && w < prev.nvalid) {
        double step = 1.1 * prev.res[w] + 8.0 * DBL_EPSILON * tn;
        x[0] = prev.theta[w] - 8.0 * DBL_EPSILON * tn;
        for (int q = 1; q < kLzShifts; ++q, step *= 16.0) x[q] = prev.theta[w] + step;
        for (int q = 0; q < kLzShifts; ++q) x[q] = std::min(std::max(x[q], l), h);
      } else {
        for (int q = 0; q < kLzShifts; ++q) x[q] = l + (h - l) * static_cast<double>(q + 1) / (kLzShifts + 1.0);
      }
      lz_sturm(a, b2.data(), J, x, pivmin, cnt);
      for (int q = 0; q < kLzShifts; ++q) {
        if (cnt[q] <= k)
          l = std::max(l, x[q]);
        else
          h = std::min(h, x[q]);
      }
    }
    theta[w] = 0.5 * (l + h);
  }
  const double pivtol = DBL_EPSILON * tn;
  std::vector<double>& X = *Xout;
  X.assign(static_cast<size_t>(nwant) * J, 0.0);
  std::vector<LzTriLu> lu(nwant);
  for (int it = 0; it < 3; ++it) {
    for (int w = 0; w < nwant; ++w) {
      double* x = X.data() + static_cast<size_t>(w) * J;
      if (it == 0) {
        for (int i = 0; i < J; ++i) x[i] = 1.0 + 0.01 * static_cast<double>((i * 7 + w * 3) % 11);
        lu[w].factor(a, b, J, theta[w] + 2.0 * DBL_EPSILON * tn, pivtol);
      }
      lu[w].solve(J, x);
      lz_normalize(x, J);
    }
    for (int w = 1; w < nwant; ++w)
      for (int c = 0; c < w; ++c) {
        if (std::fabs(theta[w] - theta[c]) > 1e-3 * tn) continue;
        double* xa = X.data() + static_cast<size_t>(w) * J;
        const double* xc = X.data() + static_cast<size_t>(c) * J;
        double d = 0.0;
        for (int i = 0; i < J; ++i) d += xa[i] * xc[i];
        for (int i = 0; i < J; ++i) xa[i] -= d * xc[i];
        lz_normalize(xa, J);
      }
  }
  int conv = 1;
  for (int w = 0; w < nwant; ++w) {
    const double r = std::fabs(b[J - 1]) * std::fabs(X[static_cast<size_t>(w) * J + J - 1]);
    out->theta[w] = theta[w];
    out->res[w] = r;
    if (!(r <= tol * tn)) conv = 0;
  }
  out->J = J;
  out->nvalid = nwant;
  out->converged = conv && nwant == p;
  out->tnorm = tn;
}

}  // namespace

// Y[a] = sum_k U_{c0+k} X[a][k] for a < P (Ritz vectors), a thread per row;
// P is a template argument so that a row costs P FMAs a basis vector and the
// loads of four vectors are in flight (n = 10^6, P = 3, J = 78: 0.49 ms, 1.36 ms with
// P <= 8 predicated).
template <int P, typename T>
__global__ void __launch_bounds__(kLzThreads) lz_ritz(const T* __restrict__ U, int64_t n, int c0, int J,
                                                      const double* __restrict__ X, T* __restrict__ Y) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) {
    T acc[P];
#pragma unroll
    for (int a = 0; a < P; ++a) acc[a] = lz_zero<T>();
    const T* u0 = U + static_cast<int64_t>(c0) * n + i;
#pragma unroll 4
    for (int k = 0; k < J; ++k) {
      const T u = u0[static_cast<int64_t>(k) * n];
#pragma unroll
      for (int a = 0; a < P; ++a) acc[a] = lz_scale_fma(u, X[static_cast<int64_t>(a) * J + k], acc[a]);
    }
#pragma unroll
    for (int a = 0; a < P; ++a) Y[static_cast<int64_t>(a) * n + i] = acc[a];
  }
}

template <typename T>
void lz_launch_ritz(int p, int blocks, cudaStream_t st, const T* U, int64_t n, int c0, int J, const double* X, T* Y) {
  switch (p) {
    case 1: lz_ritz<1, T><<<blocks, kLzThreads, 0, st>>>(U, n, c0, J, X, Y); break;
    case 2: lz_ritz<2, T><<<blocks, kLzThreads, 0, st>>>(U, n, c0, J, X, Y); break;
    case 3: lz_ritz<3, T><<<blocks, kLzThreads, 0, st>>>(U, n, c0, J, X, Y); break;
    case 4: lz_ritz<4, T><<<blocks, kLzThreads, 0, st>>>(U, n, c0, J, X, Y); break;
    case 5: lz_ritz<5, T><<<blocks, kLzThreads, 0, st>>>(U, n, c0, J, X, Y); break;
    case 6: lz_ritz<6, T><<<blocks, kLzThreads, 0, st>>>(U, n, c0, J, X, Y); break;
    case 7: lz_ritz<7, T><<<blocks, kLzThreads, 0, st>>>(U, n, c0, J, X, Y); break;
    default: lz_ritz<8, T><<<blocks, kLzThreads, 0, st>>>(U, n, c0, J, X, Y); break;
  }
  count_launch();
}

struct LzOutput {
  int r;
  int col[kLzWant];
  double lam[kLzWant];
};

// V[i, j] = sqrt(lambda_j) u_j[i] for lambda_j > 0, else 0 (row-major n x r).
template <typename T>
__global__ void __launch_bounds__(kLzThreads) lz_output(const T* __restrict__ U, int64_t n,
                                                        const __grid_constant__ LzOutput o, double2* __restrict__ V,
                                                        float2* __restrict__ V32) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) {
    for (int j = 0; j < o.r; ++j) {
      double2 v = make_double2(0.0, 0.0);
      if (o.col[j] >= 0 && o.lam[j] > 0.0) {
        const double s = sqrt(o.lam[j]);
        const T u = U[static_cast<int64_t>(o.col[j]) * n + i];
        v = lz_mul(make_double2(s, 0.0), lz_as_complex(u));
      }
      if (V) V[i * o.r + j] = v;
      if (V32) V32[i * o.r + j] = make_float2(static_cast<float>(v.x), static_cast<float>(v.y));
    }
  }
}

// ---------------------------------------------------------------------------
// input checks
// ---------------------------------------------------------------------------
__global__ void lz_check_csr(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx,
                             const double* __restrict__ wts, int64_t n, int64_t nnz, int32_t* status) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t t0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  bool bad = false;
  if (t0 == 0) bad |= rowptr[0] != 0 || static_cast<int64_t>(rowptr[n]) != nnz;
  for (int64_t i = t0; i < n; i += stride) bad |= rowptr[i] > rowptr[i + 1];
  for (int64_t k = t0; k < nnz; k += stride) {
    bad |= colidx[k] < 0 || colidx[k] >= n;
    if (wts) bad |= !isfinite(wts[k]);
  }
  if (bad) dev_fail(status, LRQ_EINVAL);
}

__global__ void lz_check_dense(const double2* __restrict__ Q, int64_t n, int64_t ld, int32_t* status) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  bool bad = false;
  for (int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < n * n; t += stride) {
    const double2 q = Q[(t / n) * ld + (t % n)];
    bad |= !isfinite(q.x) || !isfinite(q.y);
  }
  if (bad) dev_fail(status, LRQ_EINVAL);
}

// ---------------------------------------------------------------------------
// host driver
// ---------------------------------------------------------------------------
namespace {

struct LzPlan {
  int64_t n;
  int r, maxit, lmax, cap, nch, chunk, ldx;
  size_t esz;
  size_t off_U, off_w, off_Y, off_part, off_h1, off_h2, off_npart, off_alpha, off_beta, off_state, off_X, off_deg,
      off_snap, off_count, off_two, off_qdig, off_xdig, off_rowexp, total;
  size_t plain;  // bytes without the dense operator's digits, which come last
};

size_t lz_take(size_t& cur, size_t bytes) {
  size_t o = cur;
  cur = align_up(cur + bytes, 256);
  return o;
}

void lz_plan(int64_t n, int r, int maxit, bool cplx, LzPlan* p) {
  p->n = n;
  p->r = r;
  p->maxit = maxit;
  p->lmax = 2 * r + 8;                    // locked vectors (repeated eigenvalues need extra slots)
  p->cap = p->lmax + maxit + 1;           // basis columns
  // about two row chunks per SM, 512 (four rows a thread, which pay for the
  // block's sums) to 4096 rows each
  p->chunk = static_cast<int>(std::min<int64_t>(
      kLzChunkMax,
      std::max<int64_t>(4 * kLzDotThreads, static_cast<int64_t>(align_up(ceil_div(n, 2 * 152), kLzDotThreads)))));
  p->nch = static_cast<int>(ceil_div(n, p->chunk));
  p->ldx = maxit + 1;
  p->esz = cplx ? sizeof(double2) : sizeof(double);
  size_t cur = 0;
  p->off_U = lz_take(cur, static_cast<size_t>(n) * p->cap * p->esz);
  p->off_w = lz_take(cur, static_cast<size_t>(n) * p->esz);
  p->off_Y = lz_take(cur, static_cast<size_t>(n) * kLzWant * p->esz);
  p->off_part = lz_take(cur, static_cast<size_t>(p->cap) * p->nch * p->esz);
  p->off_h1 = lz_take(cur, static_cast<size_t>(p->cap) * p->esz);
  p->off_h2 = lz_take(cur, static_cast<size_t>(p->cap) * p->esz);
  p->off_npart = lz_take(cur, static_cast<size_t>(kLzMaxBlocks) * sizeof(double));
  p->off_alpha = lz_take(cur, static_cast<size_t>(p->ldx) * sizeof(double));
  p->off_beta = lz_take(cur, static_cast<size_t>(p->ldx) * sizeof(double));
  p->off_state = lz_take(cur, sizeof(LzState));
  p->off_X = lz_take(cur, static_cast<size_t>(kLzWant) * p->ldx * sizeof(double));
  p->off_deg = lz_take(cur, cplx ? 0 : static_cast<size_t>(n) * sizeof(double));  // Laplacian degrees
  p->off_snap = lz_take(cur, sizeof(LzSnap) + 2 * static_cast<size_t>(p->ldx) * sizeof(double));
  // arrival counters: matvec, three-term step, update, then one per vector group of lz_dots
  p->off_count = lz_take(cur, (3 + static_cast<size_t>(ceil_div(p->cap, kLzGroup))) * sizeof(unsigned));
  p->off_two = lz_take(cur, 2 * static_cast<size_t>(kLzMaxBlocks) * p->esz);  // the operator's block sums
  p->plain = cur;
  const bool fixed = cplx && lz_use_fixed(n);  // the dense operator's digits
  const LzFixed f = lz_fixed(n);
  p->off_qdig = lz_take(cur, fixed ? f.qbytes : 0);
  p->off_xdig = lz_take(cur, fixed ? f.xbytes : 0);
  p->off_rowexp = lz_take(cur, fixed ? static_cast<size_t>(f.units) * kLzFixRows * sizeof(int32_t) : 0);
  p->total = cur;
}

int lz_rows_grid(int64_t rows) { return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(ceil_div(rows, kLzThreads), 152 * 8))); }

template <typename T>
struct LzRun {
  // operator
  bool fixed;  // dense, from the digits
  const double2* Q;
  int64_t ld;
  const int32_t* rowptr;
  const int32_t* colidx;
  const double* wts;
  int64_t nnz;
  // problem
  int64_t n;
  double tol;
  uint64_t seed;
  LzPlan p;
  uint8_t* ws;
  int32_t* status;
  cudaStream_t st;
  cudaStream_t side;  // convergence checks run here, beside the next Lanczos steps
  cudaEvent_t ev;     // step done (the check waits for it)

  T* U() const { return reinterpret_cast<T*>(ws + p.off_U); }
  T* col(int c) const { return U() + static_cast<int64_t>(c) * n; }
  T* w() const { return reinterpret_cast<T*>(ws + p.off_w); }
  T* Y() const { return reinterpret_cast<T*>(ws + p.off_Y); }
  T* part() const { return reinterpret_cast<T*>(ws + p.off_part); }
  T* h1() const { return reinterpret_cast<T*>(ws + p.off_h1); }
  T* h2() const { return reinterpret_cast<T*>(ws + p.off_h2); }
  double* npart() const { return reinterpret_cast<double*>(ws + p.off_npart); }
  double* alpha() const { return reinterpret_cast<double*>(ws + p.off_alpha); }
  double* beta() const { return reinterpret_cast<double*>(ws + p.off_beta); }
  LzState* state() const { return reinterpret_cast<LzState*>(ws + p.off_state); }
  double* X() const { return reinterpret_cast<double*>(ws + p.off_X); }
  double* deg() const { return reinterpret_cast<double*>(ws + p.off_deg); }
  LzSnap* snap() const { return reinterpret_cast<LzSnap*>(ws + p.off_snap); }
  unsigned* counter(int i) const { return reinterpret_cast<unsigned*>(ws + p.off_count) + i; }
  T* two() const { return reinterpret_cast<T*>(ws + p.off_two); }
  uint4* qdig() const { return reinterpret_cast<uint4*>(ws + p.off_qdig); }
  uint8_t* xdig() const { return fixed ? ws + p.off_xdig : nullptr; }
  int32_t* rowexp() const { return reinterpret_cast<int32_t*>(ws + p.off_rowexp); }

  // y = Q x, h1()[0] = uprev^H y (uprev may be NULL), h1()[1] = x^H y
  void matvec(const T* x, T* y, const T* uprev) const;
  int prepare() const;  // operator set-up once per truncation (Laplacian degrees, dense digits)

  // h2() = U[:, :nc]^H w, w -= U[:, :nc] h2(), then by mode (lz_update): 0
  // closes Lanczos step j (column nc - 1), 1 normalises a start vector, 2
  // nothing more.
  int project(int nc, int j, int mode) const {
    if (nc > 0) {
      dim3 g(p.nch, static_cast<unsigned>(ceil_div(nc, kLzGroup)));
      lz_dots<T><<<g, kLzDotThreads, 0, st>>>(U(), n, nc, w(), part(), p.nch, p.chunk, counter(3), h2(), state());
      count_launch();
    }
    using F = typename LzFloat<T>::type;
    const size_t smem = static_cast<size_t>(nc) * (sizeof(T) + sizeof(F));
    // eight warps a tile of 32 rows until the rows fill the chip by themselves
    const bool wide = n >= static_cast<int64_t>(152) * 4 * kLzThreads;
    const auto kern = wide ? lz_update<1, T> : lz_update<8, T>;
    const int tile = wide ? kLzThreads : 32;
    if (smem > 40 * 1024) {
      int e = cuda_check(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              static_cast<int>(smem)),
                         "lz_update shared memory");
      if (e) return e;
    }
    const int blocks = static_cast<int>(std::min<int64_t>(ceil_div(n, tile), 152 * 8));
    kern<<<blocks, kLzThreads, smem, st>>>(U(), n, nc, h2(), w(), npart(), counter(2), mode, mode == 0 ? 1 : 0, h1(),
                                           nc - 1, j, alpha(), beta(), state());
    count_launch();
    return LRQ_OK;
  }
  void scale(int c) const {  // column c = w / ||w||
    lz_scale_into<T><<<lz_rows_grid(n), kLzThreads, 0, st>>>(w(), n, col(c), xdig(), state());
    count_launch();
  }
  // A convergence check takes alpha, beta and the state as they are after
  // step J (lz_snapshot) to the host, on the side stream, so the next Lanczos
  // steps proceed meanwhile; its verdict is worked out kLzLag steps later: the
  // host waits for the copy with those steps queued, so the GPU is not left
  // idle and at most kLzLag steps run past convergence.
  int launch_check(int J) const {
    lz_snapshot<<<1, 256, 0, st>>>(state(), alpha(), beta(), J, status, snap());
    count_launch();
    int e = cuda_check(cudaGetLastError(), "lanczos step kernels");
    if (e) return e;
    if ((e = cuda_check(cudaEventRecord(ev, st), "record step event"))) return e;
    return cuda_check(cudaStreamWaitEvent(side, ev, 0), "order check after step");
  }
  int finish_check(int J, int p_want, std::vector<double>* buf, std::vector<double>* x, LzCheck* hc) const {
    buf->resize(sizeof(LzSnap) / sizeof(double) + 2 * static_cast<size_t>(J));
    int e = cuda_check(cudaMemcpyAsync(buf->data(), snap(), buf->size() * sizeof(double), cudaMemcpyDeviceToHost,
                                       side),
                       "copy check");
    if (e) return e;
    if ((e = cuda_check(cudaStreamSynchronize(side), "lanczos sync"))) return e;
    LzSnap hs;
    std::memcpy(&hs, buf->data(), sizeof(hs));
    if (hs.status != 0) return fail(hs.status, "lrq_truncate: the device reported an invalid input or error");
    const double* a = buf->data() + sizeof(LzSnap) / sizeof(double);
    if (hs.jdone > 0) {
      lz_tridiag(a, a + J, std::min(hs.jdone, J), p_want, tol, x, hc);
    } else {
      hc->J = hc->converged = hc->nvalid = 0;
    }
    hc->breakdown = hs.stop;
    return LRQ_OK;
  }

  // One Lanczos run against the L locked vectors; wants the p largest
  // eigenpairs of the deflated operator.
  int run(int L, int p_want, int run_id, LzCheck* hc, std::vector<double>* x, int64_t* steps) const {
    int e = cuda_check(cudaMemsetAsync(state(), 0, sizeof(LzState), st), "memset state");
    if (e) return e;
    if ((e = cuda_check(cudaMemsetAsync(counter(0), 0, (3 + ceil_div(p.cap, kLzGroup)) * sizeof(unsigned), st),
                        "memset counters")))
      return e;
    std::memset(hc, 0, sizeof(*hc));
    std::vector<double> buf;
    lz_start<T><<<lz_rows_grid(n), kLzThreads, 0, st>>>(w(), n, seed, run_id, state());
    count_launch();
    if (L > 0 && (e = project(L, 0, 2))) return e;
    if ((e = project(L, 0, 1))) return e;
    scale(L);
    int pending = 0, since = 0;  // a check in flight, and steps taken since it started
    // the verdict of the check in flight: 1 = this run is over, 0 = go on
    auto verdict = [&](int* over) -> int {
      const int e2 = finish_check(pending, p_want, &buf, x, hc);
      pending = 0;
      if (e2) return e2;
      if (hc->breakdown == 2) hc->nvalid = 0;  // the start vector had no part outside the locked space
      *over = hc->breakdown || hc->converged || L + hc->J >= n;
      return LRQ_OK;
    };
    for (int j = 0; j < p.maxit && L + j < n; ++j) {
      const int c = L + j;
      const T* uprev = j > 0 ? col(c - 1) : nullptr;
      matvec(col(c), w(), uprev);
      // the three-term step: the large components of w = Q u_j lie along u_j
      // and u_{j-1}; taking them out first leaves components of rounding size
      // along every other stored vector, which one full Gram-Schmidt pass then
      // removes (alpha_j = h1[1] + h2[c])
      lz_threeterm<T><<<lz_rows_grid(n), kLzThreads, 0, st>>>(w(), n, uprev, col(c), h1(), npart(), counter(1),
                                                              state());
      count_launch();
      if ((e = project(c + 1, j, 0))) return e;
      scale(c + 1);
      ++*steps;
      ++since;
      const int J = j + 1;
      const bool last = J == p.maxit || L + J >= n;
      const int every = J < 16 ? 2 : (J < 64 ? 4 : 8);
      const bool due = J >= p_want && J % every == 0;
      int over = 0;
      if (pending && (due || last || since >= kLzLag)) {
        if ((e = verdict(&over))) return e;
        if (over) return LRQ_OK;
      }
      if (due || last) {
        if ((e = launch_check(J))) return e;
        pending = J;
        since = 0;
      }
      if (last) {
        if ((e = verdict(&over))) return e;
        if (over) return LRQ_OK;
        return fail(LRQ_ENOCONV, "lrq_truncate: Lanczos did not converge within max_iter steps");
      }
    }
    return fail(LRQ_ENOCONV, "lrq_truncate: Lanczos did not converge within max_iter steps");
  }

  int solve(int r, double* lambda_out, double2* V, float2* V32, int64_t* iters_out) const {
    std::vector<double> vals;
    int L = 0, run_id = 0;
    int64_t steps = 0;
    bool verify = false;
    double tn = 0.0;
    int e;
    if ((e = prepare())) return e;
    auto wait = [this]() { cudaStreamSynchronize(st); };
    HostCopies<decltype(wait)> copies(wait);
    while (L < n) {
      if (!verify && L >= r) verify = true;
      const int p_want = verify ? 1 : static_cast<int>(std::min<int64_t>(r - L, n - L));
      LzCheck hc;
      std::vector<double> x;  // the wanted eigenvectors of T
      if ((e = run(L, p_want, run_id++, &hc, &x, &steps))) return e;
      if (hc.nvalid <= 0) break;
      tn = std::max(tn, hc.tnorm);
      if (verify) {
        std::vector<double> sorted = vals;
        std::sort(sorted.begin(), sorted.end(), [](double a, double b) { return a > b; });
        // a further copy of the r-th value changes no value of the top r (and
        // that eigenspace has no unique r-dimensional part): stop unless the
        // deflated operator still has an eigenvalue above the r-th one
        if (!(hc.theta[0] > sorted[r - 1] + 1e-8 * tn)) break;
      }
      const int q = verify ? 1 : hc.nvalid;
      if (L + q > p.lmax) return fail(LRQ_ENOCONV, "lrq_truncate: more repeated eigenvalues than locking slots");
      if ((e = cuda_check(cudaMemcpyAsync(X(), copies.keep(std::move(x)),
                                          static_cast<size_t>(q) * hc.J * sizeof(double), cudaMemcpyHostToDevice, st),
                          "copy eigenvectors of T")))
        return e;
      lz_launch_ritz<T>(q, lz_rows_grid(n), st, U(), n, L, hc.J, X(), Y());
      if ((e = cuda_check(cudaMemcpyAsync(col(L), Y(), static_cast<size_t>(q) * n * sizeof(T),
                                          cudaMemcpyDeviceToDevice, st),
                          "copy Ritz vectors")))
        return e;
      for (int a = 0; a < q; ++a) vals.push_back(hc.theta[a]);
      L += q;
    }
    // the r largest locked pairs, descending
    std::vector<int> order(vals.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = static_cast<int>(i);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return vals[a] > vals[b]; });
    LzOutput o;
    std::memset(&o, 0, sizeof(o));
    o.r = r;
    std::vector<double> lam_host(r);
    for (int j = 0; j < r; ++j) {
      if (j < static_cast<int>(order.size())) {
        o.col[j] = order[j];
        o.lam[j] = vals[order[j]];
      } else {
        o.col[j] = -1;
        o.lam[j] = 0.0;
      }
      lam_host[j] = o.lam[j];
    }
    if (V || V32) {
      lz_output<T><<<lz_rows_grid(n), kLzThreads, 0, st>>>(U(), n, o, V, V32);
      count_launch();
    }
    if ((e = cuda_check(cudaMemcpyAsync(lambda_out, copies.keep(std::move(lam_host)), r * sizeof(double),
                                        cudaMemcpyHostToDevice, st),
                        "copy eigenvalues")))
      return e;
    if ((e = cuda_check(cudaStreamSynchronize(st), "lanczos sync"))) return e;
    if (iters_out) *iters_out = steps;
    return LRQ_OK;
  }
};

template <>
void LzRun<double>::matvec(const double* x, double* y, const double* uprev) const {
  lz_matvec_laplacian<<<lz_rows_grid(n), kLzThreads, 0, st>>>(rowptr, colidx, wts, deg(), n, nnz, x, y, uprev, two(),
                                                              counter(0), h1(), state());
  count_launch();
}

template <>
int LzRun<double>::prepare() const {
  lz_degree<<<lz_rows_grid(n), kLzThreads, 0, st>>>(rowptr, colidx, wts, n, nnz, deg());
  count_launch();
  return LRQ_OK;
}

template <>
int LzRun<double2>::prepare() const {
  if (!fixed) {
    lz_check_dense<<<lz_rows_grid(n * n), kLzThreads, 0, st>>>(Q, n, ld, status);
    count_launch();
    return LRQ_OK;
  }
  const LzFixed f = lz_fixed(n);
  int e = cuda_check(cudaMemsetAsync(xdig(), 0, f.xbytes, st), "clear the digits past n");
  if (e) return e;
  lz_row_exponents<<<static_cast<unsigned>(ceil_div(f.units * kLzFixRows, kLzFixThreads / 32)), kLzFixThreads, 0,
                     st>>>(Q, n, ld, f.units * kLzFixRows, rowexp(), status);
  lz_dense_digits<<<static_cast<unsigned>(ceil_div(f.units * f.steps * 32, kLzFixThreads)), kLzFixThreads, 0, st>>>(
      Q, n, ld, f.units, f.steps, rowexp(), qdig());
  count_launch(2);
  return cuda_check(cudaGetLastError(), "lz_dense_digits");
}

template <>
void LzRun<double2>::matvec(const double2* x, double2* y, const double2* uprev) const {
  if (fixed) {  // x is the column that scale() wrote last: its digits are in xdig()
    const LzFixed f = lz_fixed(n);
    const int blocks = static_cast<int>(std::min<int64_t>(f.units, kLzMaxBlocks));
    lz_matvec_fixed<<<blocks, 32, 0, st>>>(qdig(), rowexp(), n, static_cast<int>(f.units), static_cast<int>(f.steps),
                                           reinterpret_cast<const uint4*>(xdig()), x, y, uprev, two(), counter(0),
                                           h1(), state());
    count_launch();
    return;
  }
  // two rows a warp once every SM has a few warps that way
  const int rows = n >= 152 * 4 ? 2 : 1;
  const int blocks = static_cast<int>(std::min<int64_t>(ceil_div(n, rows * (kLzMvThreads / 32)), kLzMaxBlocks));
  if (rows == 2)
    lz_matvec_dense<2><<<blocks, kLzMvThreads, 0, st>>>(Q, n, ld, x, y, uprev, two(), counter(0), h1(), state());
  else
    lz_matvec_dense<1><<<blocks, kLzMvThreads, 0, st>>>(Q, n, ld, x, y, uprev, two(), counter(0), h1(), state());
  count_launch();
}

}  // namespace

int truncate_check(const lrq_matrix* Q, int r, int max_iter) {
  if (!Q) return fail(LRQ_EINVAL, "Q is NULL");
  if (Q->kind != LRQ_MATRIX_DENSE_C128 && Q->kind != LRQ_MATRIX_CSR_LAPLACIAN)
    return fail(LRQ_EINVAL, "unknown matrix kind");
  if (Q->n < 1) return fail(LRQ_EINVAL, "n must be >= 1");
  if (r < 1 || r > kLzWant || r > Q->n) return fail(LRQ_EINVAL, "r must be in [1, min(8, n)]");
  if (max_iter < 0 || max_iter > kLzMaxIter) return fail(LRQ_EINVAL, "max_iter must be in [0, 4096]");
  if (Q->kind == LRQ_MATRIX_DENSE_C128) {
    if (!Q->values) return fail(LRQ_EINVAL, "dense values pointer is NULL");
    if (Q->ld < Q->n) return fail(LRQ_EINVAL, "ld must be >= n");
    if (Q->n > (int64_t(1) << 20)) return fail(LRQ_EUNSUPPORTED, "dense n above 2^20");
  } else {
    if (!Q->rowptr || (Q->nnz > 0 && !Q->colidx)) return fail(LRQ_EINVAL, "CSR pointer is NULL");
    if (Q->nnz < 0 || Q->nnz >= (int64_t(1) << 31)) return fail(LRQ_EINVAL, "nnz must be in [0, 2^31)");
    if (Q->n >= (int64_t(1) << 31)) return fail(LRQ_EINVAL, "CSR n must be below 2^31");
  }
  return LRQ_OK;
}

size_t truncate_workspace_bytes(const lrq_matrix* Q, int r, int max_iter, size_t* least) {
  LzPlan p;
  const int it = static_cast<int>(std::min<int64_t>(max_iter > 0 ? max_iter : kLzDefaultIter, Q->n));
  lz_plan(Q->n, r, it, Q->kind == LRQ_MATRIX_DENSE_C128, &p);
  if (least) *least = p.plain;
  return p.total;
}

namespace {
// the side stream and event of one truncation call, released on every path
struct LzSide {
  cudaStream_t side = nullptr;
  cudaEvent_t ev = nullptr;
  int init() {
    int e = cuda_check(cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking), "create check stream");
    if (e) return e;
    return cuda_check(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming), "create step event");
  }
  ~LzSide() {
    if (side) cudaStreamSynchronize(side);
    if (ev) cudaEventDestroy(ev);
    if (side) cudaStreamDestroy(side);
  }
};
}  // namespace

int launch_truncate(const lrq_matrix* Q, int r, double tol, int max_iter, uint64_t seed, double2* V, float2* V32,
                    double* lambda_out, int64_t* iters_out, void* ws, size_t ws_bytes, int32_t* status,
                    cudaStream_t st) {
  const int it = static_cast<int>(std::min<int64_t>(max_iter > 0 ? max_iter : kLzDefaultIter, Q->n));
  const double t = tol > 0.0 ? tol : 1e-10;
  LzSide sd;
  int e = sd.init();
  if (e) return e;
  if (Q->kind == LRQ_MATRIX_DENSE_C128) {
    LzRun<double2> R;
    R.Q = static_cast<const double2*>(Q->values);
    R.ld = Q->ld;
    R.rowptr = nullptr;
    R.colidx = nullptr;
    R.wts = nullptr;
    R.nnz = 0;
    R.n = Q->n;
    R.tol = t;
    R.seed = seed;
    lz_plan(Q->n, r, it, true, &R.p);
    R.fixed = lz_use_fixed(R.n) && ws_bytes >= R.p.total;  // the caller may leave no room for the digits
    R.ws = static_cast<uint8_t*>(ws);
    R.status = status;
    R.st = st;
    R.side = sd.side;
    R.ev = sd.ev;
    return R.solve(r, lambda_out, V, V32, iters_out);
  }
  LzRun<double> R;
  R.fixed = false;
  R.Q = nullptr;
  R.ld = 0;
  R.rowptr = Q->rowptr;
  R.colidx = Q->colidx;
  R.wts = Q->weights;
  R.nnz = Q->nnz;
  R.n = Q->n;
  R.tol = t;
  R.seed = seed;
  lz_plan(Q->n, r, it, false, &R.p);
  R.ws = static_cast<uint8_t*>(ws);
  R.status = status;
  R.st = st;
  R.side = sd.side;
  R.ev = sd.ev;
  lz_check_csr<<<lz_rows_grid(std::max<int64_t>(Q->n, Q->nnz)), kLzThreads, 0, st>>>(Q->rowptr, Q->colidx,
                                                                                     Q->weights, Q->n, Q->nnz,
                                                                                     status);
  count_launch();
  return R.solve(r, lambda_out, V, V32, iters_out);
}

}  // namespace lrq
