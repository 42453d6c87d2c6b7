// Block orthonormalisation of the Lanczos partial SVD (Sec. 5.1.1: the Lanczos bidiagonalisation
// needs an orthonormal basis; here every new n x b block is made orthogonal to all previous ones
// by classical Gram-Schmidt applied twice, then orthonormalised).
//
// GB300 executes float64 with a dependent-operation latency of ~64 cycles (divide and square
// root ~650), so the sequence avoids long float64 dependency chains on a single SM:
//   1. C1 = Q^T P                      (Gram, all SMs)
//   2. P <- P - Q C1, [C2; A] = [Q, P]^T P   (one fused kernel: update + Gram of the same rows)
//      R1 = chol(A)                    (four warps; root-free, one reciprocal a pivot, seeded from its
//                                       bits through a float32 reciprocal, one float64 Newton step;
//                                       columns that lost all but 1e-12 of their norm to the
//                                       projections are deflated)
//   (the Grams and the projections of the cooperative kernel are digit products on the tensor cores, with the accuracy of
//   float64 sums; those of the launch sequence are float64 instructions)
//   3. P <- (P - Q C2) R1^-1, E = P^T P - I  (fused; per-row forward substitution, no inverse)
//      P <- P (I - U(E)),  R2 = I + U(E)   with U(E) the upper triangle of E, halved diagonal: the
//                                       Cholesky factor of I + E to first order, so P^T P = I up to
//                                       O(|E|^2) (|E| is at rounding level after step 2 unless P was
//                                       ill conditioned; the host then adds a second step 3, giving
//                                       O(|E|^4))
// The coefficients satisfy P_in = Q (C1 + C2) + P_out R2 R1 exactly for the factors used; C1 + C2
// and R2 R1 are the entries of the projected block bidiagonal matrix.  Of each P^T P only what is
// used is formed: its diagonal in step 1 (the deflation reference), its upper triangle in steps 2
// and 3 (the Cholesky factor and U(E) read nothing else).
#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "internal.h"

namespace svt {

static constexpr int ORTH_T = 256;
static constexpr int OB_MAXB = 32;
static constexpr int OB_MAXK = 128;   // nq b <= 128 previous basis columns
static constexpr double DEFLATE_REL2 = 1e-24;  // squared norm ratio below which a column is dependent

// group of lanes per row: smallest power of two >= b
static inline int row_group(int b) {
  int g = 1;
  while (g < b) g <<= 1;
  return g;
}

// ------------------------------------------------------------------------------------------------
// Gram products G = [Q_0 .. Q_{nq-1}, P]^T P, split over row chunks: every CTA owns a contiguous
// chunk of rows and writes the partial Gram of its rows; a second kernel sums the partials in a
// fixed order (deterministic).  float64 adds run at ~2 per clock per SM on GB300, so the sums are
// spread over many CTAs too.
// ------------------------------------------------------------------------------------------------
static constexpr int GRAM_SUB = 8;        // rows staged in shared memory at a time
static constexpr int GRAM_MAXW = 160;     // (nq + 1) b <= 160
static constexpr int GRAM_MAXE = GRAM_MAXW * 32;
static constexpr int GRAM_EPT = GRAM_MAXE / ORTH_T;  // entries per thread (20)

static int gram_rows_per_cta(int n) {
  int rows = (n + 2 * 152 - 1) / (2 * 152);
  rows = (rows + GRAM_SUB - 1) / GRAM_SUB * GRAM_SUB;
  return rows < GRAM_SUB ? GRAM_SUB : rows;
}

// Upper bound on the row chunks of any launch with n' <= n rows: each chunk has >= GRAM_SUB rows
// and >= ceil(n' / 304) rows, so there are at most min(ceil(n / GRAM_SUB), 304) chunks.  k_orth_coop on a small grid
// alternates between two sets, of chunks of 16 rows (of 8 only for 8 columns, whose Grams are a fifth of the largest).
static constexpr int OC_SETS_GRID = 32;   // largest grid with two sets
long long gram_partial_doubles(int n, int nq, int b) {
  const long long rows = n;
  const long long nblk = std::max(std::min((rows + GRAM_SUB - 1) / GRAM_SUB, 2LL * 152),
                                  2 * std::min((rows + 15) / 16, (long long)OC_SETS_GRID));
  return nblk * (nq + 1) * b * b;
}

// Entry layout of a Gram G = [Q_0 .. Q_{nq-1}, P]^T P: the nq b x b blocks Q_k^T P row-major,
// then of P^T P only what is used: its diagonal (the squared column norms before the projection,
// `first` pass) or its upper triangle (i <= j) folded into b / 2 rows of b + 1 entries: row r
// holds (r, r .. b-1) followed by (b-1-r, b-1-r .. b-1), so both directions of the index map are
// a division by b + 1 and a comparison (b is even).
__host__ __device__ __forceinline__ int gram_entries(int nq, int b, bool first) {
  return nq * b * b + (first ? b : b * (b + 1) / 2);
}
__host__ __device__ __forceinline__ int upper_index(int i, int j, int b) {
  return i < b / 2 ? i * (b + 1) + (j - i) : (b - 1 - i) * (b + 1) + (j + 1);
}
// (i, j) of entry t of the folded upper triangle of a b x b matrix
__device__ __forceinline__ void upper_ij(int t, int b, int& i, int& j) {
  const int r = t / (b + 1), q = t - r * (b + 1);
  if (q < b - r) {
    i = r;
    j = r + q;
  } else {
    i = b - 1 - r;
    j = q - 1;
  }
}

// Partial Gram of rows [r0, r1) into partial[blockIdx.x * E ...), E = gram_entries(nq, b, first).
// Called by all threads.
// EPT: entries per thread, at least E / ORTH_T.
template <int EPT = GRAM_EPT>
__device__ void gram_chunk(const double* __restrict__ Q, long long q_stride, int nq, const double* __restrict__ P,
                           int b, int r0, int r1, double* __restrict__ partial, bool first) {
  __shared__ double tile[GRAM_SUB][GRAM_MAXW];
  const int W = (nq + 1) * b;
  const int E = gram_entries(nq, b, first);
  const int EQ = nq * b * b;
  double acc[EPT];
#pragma unroll
  for (int k = 0; k < EPT; ++k) acc[k] = 0.0;
  for (int rs = r0; rs < r1; rs += GRAM_SUB) {
    const int nr = min(GRAM_SUB, r1 - rs);
    for (int t = threadIdx.x; t < GRAM_SUB * W; t += blockDim.x) {
      int rr = t / W, c = t - rr * W;
      double v = 0.0;
      if (rr < nr) {
        int blk = c / b, cc = c - blk * b;
        const double* src = blk < nq ? Q + blk * q_stride : P;
        v = src[(long long)(rs + rr) * b + cc];
      }
      tile[rr][c] = v;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < EPT; ++k) {
      int e = threadIdx.x + k * ORTH_T;
      if (e < E) {
        int c, d;
        if (e < EQ) {
          c = e / b;
          d = e - c * b;
        } else if (first) {
          c = nq * b + (e - EQ);
          d = e - EQ;
        } else {
          upper_ij(e - EQ, b, c, d);
          c += nq * b;
        }
        double s = acc[k];
        for (int rr = 0; rr < nr; ++rr) s = fma(tile[rr][c], tile[rr][nq * b + d], s);
        acc[k] = s;
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < EPT; ++k) {
    int e = threadIdx.x + k * ORTH_T;
    if (e < E) partial[(long long)blockIdx.x * E + e] = acc[k];
  }
}

__global__ void __launch_bounds__(ORTH_T)
k_gram_partial(const double* __restrict__ Q, long long q_stride, int nq, const double* __restrict__ P, int n, int b,
               int rows_per_cta, double* __restrict__ partial) {
  const int r0 = blockIdx.x * rows_per_cta;
  gram_chunk(Q, q_stride, nq, P, b, r0, min(n, r0 + rows_per_cta), partial, nq > 0);
}

// CTA x owns 32 entries; its four warps sum the partials k = w, w + 4, ... and combine in a fixed
// order.  The loads of a thread are issued in batches of eight before they are added, so a thread
// waits for one memory latency per batch instead of one per partial.  With Tcol given, the entries
// e < ncoef (the projection coefficients, ncoef = K b) are also written as Tcol = Gprev + G (the
// coefficients of the two projection passes), leading dimension ldT.
__global__ void __launch_bounds__(128) k_gram_reduce(const double* __restrict__ partial, int nblk, int E,
                                                     double* __restrict__ G, const double* __restrict__ Gprev,
                                                     double* __restrict__ Tcol, int ldT, int ncoef, int b) {
  __shared__ double part[4][32];
  const int el = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + el;
  double s = 0.0;
  if (e < E) {
    int k = w;
    for (; k + 28 < nblk; k += 32) {
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = partial[(long long)(k + 4 * u) * E + e];
      s += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
    for (; k < nblk; k += 4) s += partial[(long long)k * E + e];
  }
  part[w][el] = s;
  __syncthreads();
  if (w == 0 && e < E) {
    const double g = (part[0][el] + part[1][el]) + (part[2][el] + part[3][el]);
    G[e] = g;
    if (Tcol && e < ncoef) {
      const int i = e / b, j = e - i * b;
      Tcol[i * ldT + j] = (Gprev ? Gprev[e] : 0.0) + g;
    }
  }
}

static int gram_reduce_launch(const double* partial, int nblk, int E, double* G, cudaStream_t st,
                              const double* Gprev = nullptr, double* Tcol = nullptr, int ldT = 0, int ncoef = 0,
                              int b = 1) {
  k_gram_reduce<<<(E + 31) / 32, 128, 0, st>>>(partial, nblk, E, G, Gprev, Tcol, ldT, ncoef, b);
  return 1;
}

int launch_gram(const double* Q, long long q_stride, int nq, const double* P, int n, int b, double* partial, double* G,
                cudaStream_t st, const double* Gprev, double* Tcol, int ldT) {
  const int rows = gram_rows_per_cta(n);
  const int nblk = (n + rows - 1) / rows;
  k_gram_partial<<<nblk, ORTH_T, 0, st>>>(Q, q_stride, nq, P, n, b, rows, partial);
  return 1 + gram_reduce_launch(partial, nblk, gram_entries(nq, b, nq > 0), G, st, Gprev, Tcol, ldT, nq * b * b, b);
}

// ------------------------------------------------------------------------------------------------
// Fused update + partial Gram: every CTA updates the rows of its chunk, then (after a barrier, so
// its own writes are visible) forms the partial Gram of the same rows.
//   mode 0: P <- P - Q C,             partial of [Q, P]^T P   (second projection pass follows)
//   mode 1: P <- (P - Q C) R^-1,      partial of P^T P        (correction pass follows)
// ------------------------------------------------------------------------------------------------
// Rows [r0, r1) of P, g lanes per row (lane d owns column d < b):
//   mode 0: P <- P - Q C;   mode 1: P <- (P - Q C) R^-1 with dinv = 1 / diag(R)
// C (nq b x b), sR = R diag(dinv) (the columns of R scaled by the reciprocal pivots, b x b) and
// dinv (b) in shared memory.  Called by all threads of the CTA.
__device__ void update_rows(int mode, const double* __restrict__ Q, long long q_stride, int nq,
                            const double* __restrict__ sC, const double* __restrict__ sR,
                            const double* __restrict__ sD, double* __restrict__ P, int b, int g, int r0, int r1,
                            int* mp = nullptr, int tid0 = 0) {
  // mp (may be NULL): the largest absolute high words of the new columns, shared, zeroed before
  // threads tid0 .. ORTH_T - 1 take part (tid0 a multiple of 32)
  const int tid = threadIdx.x - tid0;
  if (tid < 0) return;
  const int rows_per_iter = (ORTH_T - tid0) / g;
  const int rl = tid / g, d = tid - rl * g;
  const int gbase = (threadIdx.x & 31) & ~(g - 1);
  const int wrow = (tid & ~31) / g;   // first row of this warp within an iteration
  for (int ib = r0; ib < r1; ib += rows_per_iter) {
    if (ib + wrow >= r1) break;      // no row of this warp is left (warp-uniform)
    const int i = ib + rl;
    const bool live = i < r1 && d < b;
    double v = 0.0;
    if (live) {
      double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
      for (int blk = 0; blk < nq; ++blk) {
        const double* qrow = Q + blk * q_stride + (long long)i * b;
        const double* ccol = sC + blk * b * b + d;
        int c = 0;
        for (; c + 3 < b; c += 4) {
          a0 = fma(qrow[c], ccol[c * b], a0);
          a1 = fma(qrow[c + 1], ccol[(c + 1) * b], a1);
          a2 = fma(qrow[c + 2], ccol[(c + 2) * b], a2);
          a3 = fma(qrow[c + 3], ccol[(c + 3) * b], a3);
        }
        for (; c < b; ++c) a0 = fma(qrow[c], ccol[c * b], a0);
      }
      v = P[(long long)i * b + d] - ((a0 + a1) + (a2 + a3));
    }
    if (mode == 1) {
      // forward substitution out_d = (v_d - sum_{e<d} out_e R[e][d]) dinv[d], written as
      // w = v dinv, w_d -= out_e (R[e][d] dinv[d]): one float64 operation per step, and lane e
      // holds out_e once the steps before it are done
      double w = d < b ? v * sD[d] : 0.0;
      for (int e = 0; e < b; ++e) {
        const double ob = __shfl_sync(0xffffffffu, w, gbase + e);
        if (d > e && d < b) w -= ob * sR[e * b + d];
      }
      v = w;
    }
    if (live) {
      P[(long long)i * b + d] = v;
      if (mp) atomicMax(mp + d, __double2hiint(v) & 0x7FFFFFFF);
    }
  }
}

// Rows [r0, r1) of P <- P R^-1, one row a thread: a float64 instruction of the forward substitution works on 32 rows where
// update_rows has as many lanes idle as the triangle is empty.  sR = R diag(dinv), sD = dinv in shared memory.  For chunks
// that fill the warps (99 rows of 16 columns: 29000 -> 17000 cycles an SM, bound by the float64 pipe).
template <int B>
__device__ __noinline__ void solve_rows(const volatile double* sR, const double* __restrict__ sD, double* __restrict__ P,
                                        int r0, int r1, int* mp) {   // volatile: R is read where it is used, not kept
  int mx[B];
#pragma unroll
  for (int d = 0; d < B; ++d) mx[d] = 0;
  for (int i = r0 + threadIdx.x; i < r1; i += ORTH_T) {
    double2* p = reinterpret_cast<double2*>(P + (long long)i * B);
    double w[B];
#pragma unroll
    for (int d = 0; d < B / 2; ++d) {
      const double2 x = p[d];
      w[2 * d] = x.x * sD[2 * d];
      w[2 * d + 1] = x.y * sD[2 * d + 1];
    }
#pragma unroll
    for (int e = 0; e < B; ++e) {
#pragma unroll
      for (int d = e + 1; d < B; ++d) w[d] = fma(-w[e], sR[e * B + d], w[d]);
    }
#pragma unroll
    for (int d = 0; d < B / 2; ++d) p[d] = make_double2(w[2 * d], w[2 * d + 1]);
#pragma unroll
    for (int d = 0; d < B; ++d) mx[d] = max(mx[d], __double2hiint(w[d]) & 0x7FFFFFFF);
  }
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 0; d < B; ++d) {
    const int m = __reduce_max_sync(0xffffffffu, mx[d]);
    if (lane == d) atomicMax(mp + d, m);
  }
}

__global__ void __launch_bounds__(ORTH_T)
k_update_gram(int mode, const double* __restrict__ Q, long long q_stride, int nq, const double* __restrict__ C,
              const double* __restrict__ R, const double* __restrict__ dinv, double* __restrict__ P, int n, int b,
              int g, int rows_per_cta, double* __restrict__ partial) {
  extern __shared__ double sm_upd[];   // C (K x b), then R diag(1 / diag(R)) (b x b), 1 / diag(R)
  double* sC = sm_upd;
  double* sR = sC + nq * b * b;
  double* sD = sR + b * b;
  const int K = nq * b;
  for (int t = threadIdx.x; t < K * b; t += blockDim.x) sC[t] = C[t];
  if (mode == 1) {
    // R diag(dinv): the columns of R scaled by the reciprocal pivots
    for (int t = threadIdx.x; t < b * b; t += blockDim.x) sR[t] = R[t] * dinv[t % b];
    for (int t = threadIdx.x; t < b; t += blockDim.x) sD[t] = dinv[t];
  }
  __syncthreads();
  const int r0 = blockIdx.x * rows_per_cta;
  const int r1 = min(n, r0 + rows_per_cta);
  update_rows(mode, Q, q_stride, nq, sC, sR, sD, P, b, g, r0, r1);
  __syncthreads();
  gram_chunk(Q, q_stride, mode == 0 ? nq : 0, P, b, r0, r1, partial, false);
}

int launch_update_gram(int mode, const double* Q, long long q_stride, int nq, const double* C, const double* R,
                       const double* dinv, double* P, int n, int b, double* partial, double* G, cudaStream_t st,
                       const double* Gprev, double* Tcol, int ldT) {
  const int g = row_group(b);
  const int rows = gram_rows_per_cta(n);
  const int nblk = (n + rows - 1) / rows;
  static std::once_flag once;
  std::call_once(once, [] {
    cudaFuncSetAttribute(k_update_gram, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)((OB_MAXK * OB_MAXB + OB_MAXB * OB_MAXB + OB_MAXB) * sizeof(double)));
  });
  const size_t smem = (size_t)(nq * b * b + b * b + b) * sizeof(double);
  k_update_gram<<<nblk, ORTH_T, smem, st>>>(mode, Q, q_stride, nq, C, R, dinv, P, n, b, g, rows, partial);
  const int nqg = mode == 0 ? nq : 0;
  const int E = gram_entries(nqg, b, false);
  return 1 + gram_reduce_launch(partial, nblk, E, G, st, Gprev, Tcol, ldT, nqg * b * b, b);
}

// ------------------------------------------------------------------------------------------------
// Cholesky with deflation of the b x b block A of G2 (four warps; B = compile-time block size so every loop has exact
// bounds).  A float64 operation of a warp occupies its scheduler's float64 pipe for ~64 cycles whatever the number of
// active lanes, and takes as long to return, so the factorisation is timed by the chain of one pivot and by the count
// of warp-wide float64 instructions:
//   * root-free (L D L^T) elimination: a pivot's chain is one reciprocal (seed from the double's bits, one Newton step,
//     relative error ~1e-13), one product and one multiply-add; the square roots are taken of all pivots at once at
//     the end;
//   * the rows of the trailing block are spread over the four schedulers (warp w owns rows i = w mod 4), and for
//     B <= 16 over 32 / B lane groups as well; row j is published in shared memory when it becomes the pivot row;
//   * deflation is decided by integer comparison of the bit patterns against 1e-24 times the column's squared norm
//     before the projections.
// Measured in the cooperative kernel (cycles, one warp with square roots before -> now): b = 16 16700 -> 9000, b = 24 (n = 2753)
// 55600 -> 25900, b = 32 65200 -> 27200.
// Columns that lost all but 1e-12 of their norm (or whose pivot is not a normal positive double
// above 2^-1021) are deflated: R's row is zero and 1 / R_jj = 0.
// ------------------------------------------------------------------------------------------------
// Reciprocal of a normal positive double (biased exponent 2 .. 2045) to ~1e-13: float32 reciprocal of the mantissa, the
// exponent negated exactly, one step of Newton's iteration y <- y + y (1 - d y).
__device__ __forceinline__ double rcp_pivot(double d) {
  const unsigned int hi = (unsigned int)__double2hiint(d), lo = (unsigned int)__double2loint(d);
  const int E = (int)((hi >> 20) & 0x7FFu) - 1023;
  const float m = __int_as_float((int)(0x3F800000u | ((hi & 0xFFFFFu) << 3) | (lo >> 29)));   // in [1, 2)
  const unsigned int f = (unsigned int)__float_as_int(__fdividef(1.f, m));                  // in (0.5, 1]
  const int fe = (int)((f >> 23) & 0xFFu);
  const double y0 = __hiloint2double((int)(((unsigned int)(fe - 127 + 1023 - E) << 20) | ((f & 0x7FFFFFu) >> 3)),
                                     (int)((f & 7u) << 29));
  return fma(y0, fma(-d, y0, 1.0), y0);
}

// Reciprocal square root of a normal positive double (biased exponent 2 .. 2046) to ~1e-13: the
// seed halves the exponent exactly and takes a float32 rsqrt of the mantissa, then one step of
// Newton's iteration for 1/sqrt(d), y <- y + y (1 - d y^2) / 2, squares its relative error.
__device__ __forceinline__ double rsqrt_pivot(double d) {
  const unsigned int hi = (unsigned int)__double2hiint(d), lo = (unsigned int)__double2loint(d);
  const int E = (int)((hi >> 20) & 0x7FFu);
  const int p = 1 - (E & 1);                      // unbiased exponent odd: mantissa scaled into [2, 4)
  const int k = (E - 1023 - p) >> 1;              // d = m 4^k, m in [1, 4)
  const float m = __int_as_float((int)(((unsigned int)(127 + p) << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29)));
  const unsigned int f = (unsigned int)__float_as_int(rsqrtf(m));   // in (0.5, 1]
  const int fe = (int)((f >> 23) & 0xFFu);
  const double y0 = __hiloint2double((int)(((unsigned int)(fe - 127 + 1023 - k) << 20) | ((f & 0x7FFFFFu) >> 3)),
                                     (int)((f & 7u) << 29));
  const double h = __hiloint2double((int)(hi - 0x100000u), (int)lo);   // d / 2, exact
  const double t = h * y0;
  const double u = fma(-t, y0, 0.5);              // (1 - d y0^2) / 2
  return fma(y0, u, y0);
}

// Self-test of rsqrt_pivot: out[5 i + 4] = rsqrt_pivot(x_i) (x_i a normal positive double).
__global__ void k_pivot_selftest(const double* __restrict__ x, long long n, double* __restrict__ out) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[5 * i + 4] = rsqrt_pivot(x[i]);
}

int launch_pivot_selftest(const double* x, long long n, double* out, cudaStream_t st) {
  if (n <= 0) return 0;
  const int blocks = (int)svt_min_ll(svt_ceil_div(n, 256), 152LL * 4);
  k_pivot_selftest<<<blocks, 256, 0, st>>>(x, n, out);
  return 1;
}

static constexpr int CHOL_T = 128;
__device__ __forceinline__ void chol_sync() { asm volatile("bar.sync 2, %0;" ::"n"(CHOL_T) : "memory"); }

// Threads 0 .. 127 of the CTA.  A: the folded upper triangle of the block; ref: the columns' squared norms before the
// projections (NULL: A's diagonal); R (B x B) and dinv (B) in shared memory.  Ends without a barrier after the last writes
// to R.
template <int B>
__device__ __forceinline__ void chol_warps(const double* __restrict__ A, const double* __restrict__ ref,
                                           double* __restrict__ R, double* __restrict__ dinv,
                                           unsigned long long* __restrict__ counters) {
  constexpr int H = B <= 16 ? 32 / B : 1;          // lane groups
  constexpr int NR = (B + 4 * H - 1) / (4 * H);    // rows per lane
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int h = lane / B, c = lane - h * B;        // for B = 24 lanes 24..31 get h = 1: idle
  const bool col = h < H;
  const int i0 = w + 4 * h;                        // rows i0 + 4 H s
  double a[NR];
#pragma unroll
  for (int s = 0; s < NR; ++s) {
    const int i = i0 + 4 * H * s;
    a[s] = (col && i < B && i <= c) ? A[upper_index(i, c, B)] : 0.0;
  }
  __shared__ long long s_thr[OB_MAXB];
  if (threadIdx.x < B) {
    const int q = threadIdx.x;
    s_thr[q] = __double_as_longlong(DEFLATE_REL2 * (ref ? ref[q] : A[upper_index(q, q, B)]));
  }
  int deflated = 0;
#pragma unroll
  for (int j = 0; j < B; ++j) {
    // row j: warp j mod 4, group (j / 4) mod H, slot j / (4 H)
    if (w == (j & 3) && h == (j / 4) % H && col) R[j * B + c] = a[j / (4 * H)];
    chol_sync();
    const double d = R[j * B + j];
    const long long db = __double_as_longlong(d);
    const bool ok = db > s_thr[j] && db >= 0x0020000000000000LL && db < 0x7FD0000000000000LL;
    deflated += ok ? 0 : 1;
    if (threadIdx.x == 0) dinv[j] = ok ? 1.0 : 0.0;
    if (j + 1 < B && ok) {
      const double inv = rcp_pivot(d);
      const double rc = R[j * B + (col ? c : 0)] * inv;
      // trailing update A_ic -= A_ji (A_jc / d) for j < i <= c
#pragma unroll
      for (int s = 0; s < NR; ++s) {
        const int i = i0 + 4 * H * s;
        if (4 * H * s + 4 * H > j + 1) {           // some row of this slot is below the pivot
          if (col && i > j && i <= c) a[s] = fma(-R[j * B + i], rc, a[s]);
        }
      }
    }
  }
  chol_sync();
  if (threadIdx.x < B) {
    const int q = threadIdx.x;
    dinv[q] = dinv[q] != 0.0 ? rsqrt_pivot(R[q * B + q]) : 0.0;
  }
  chol_sync();
  for (int e = threadIdx.x; e < B * B; e += CHOL_T) {
    const int i = e / B, q = e - i * B;
    R[e] = q >= i ? R[e] * dinv[i] : 0.0;
  }
  if (threadIdx.x == 0 && deflated && counters) atomicAdd(&counters[2], (unsigned long long)deflated);
}

template <int B>
__global__ void __launch_bounds__(CHOL_T)
k_chol(const double* __restrict__ G1, const double* __restrict__ G2, int nq, double* __restrict__ R,
       double* __restrict__ dinv, unsigned long long* __restrict__ counters) {
  __shared__ double sR[B * B], sD[B];
  chol_warps<B>(G2 + nq * B * B, G1 && nq > 0 ? G1 + nq * B * B : nullptr, sR, sD, counters);
  __syncthreads();
  for (int e = threadIdx.x; e < B * B; e += CHOL_T) R[e] = sR[e];
  if (threadIdx.x < B) dinv[threadIdx.x] = sD[threadIdx.x];
}

// ------------------------------------------------------------------------------------------------
// P <- P (I - U(E)) with E = G3 - I; (I + U(E)) R1 (upper triangular) goes to Tdiag and/or Rout,
// and max |E| over non-deflated columns to counters[3].
// ------------------------------------------------------------------------------------------------
// sU = U(E) (upper triangle of E, halved diagonal; b x b row-major), from G3 (upper-triangle
// layout).  All threads.
__device__ __forceinline__ void correct_load_U(const double* __restrict__ G3, int b, double* __restrict__ sU) {
  for (int e = threadIdx.x; e < b * b; e += blockDim.x) {
    int i = e / b, j = e - i * b;
    double v = 0.0;
    if (j >= i) {
      const double x = G3[upper_index(i, j, b)] - (i == j ? 1.0 : 0.0);
      v = (j > i) ? x : 0.5 * x;
    }
    sU[e] = v;
  }
}

// (I + U(E)) R1 -> Tdiag / Rout / sRout (any may be NULL).  All threads of one CTA; sU, sR1 in
// shared memory.
__device__ void correct_coefs(const double* __restrict__ sU, const double* __restrict__ sR1, int b,
                              double* __restrict__ Tdiag, int ldT, double* __restrict__ Rout,
                              double* __restrict__ sRout) {
  for (int e = threadIdx.x; e < b * b; e += blockDim.x) {
    int i = e / b, j = e - i * b;
    double v = 0.0;
    if (i <= j) {
      v = sR1[i * b + j];
      for (int k = i; k <= j; ++k) v += sU[i * b + k] * sR1[k * b + j];
    }
    if (Tdiag) Tdiag[i * ldT + j] = v;
    if (Rout) Rout[e] = v;
    if (sRout) sRout[e] = v;
  }
}

// max |E| over the non-deflated columns -> counters[3] (as the bits of a non-negative double, so
// atomicMax orders them), from U(E) in shared memory: E_ij = U_ij above the diagonal, E_ii =
// 2 U_ii; a deflated column has G3_ii = 0, i.e. U_ii = -1/2, and a column counts as live when
// U_ii > -1/4.  Integer operations on the bit patterns (the float64 pipe is the scarce one); NaN
// entries are ignored.  One warp (all 32 lanes).
__device__ void correct_defect(const double* __restrict__ sU, int b, unsigned long long* __restrict__ counters) {
  constexpr long long kAbs = 0x7FFFFFFFFFFFFFFFLL, kInf = 0x7FF0000000000000LL, kQuarter = 0x3FD0000000000000LL;
  const int lane = threadIdx.x & 31;
  long long off = 0, dia = 0;
  for (int e = lane; e < b * b; e += 32) {
    const int i = e / b, j = e - i * b;
    if (j < i) continue;
    const long long xi = __double_as_longlong(sU[i * b + i]), xj = __double_as_longlong(sU[j * b + j]);
    const bool li = (xi >= 0 && xi <= kInf) || (xi & kAbs) < kQuarter;
    const bool lj = (xj >= 0 && xj <= kInf) || (xj & kAbs) < kQuarter;
    const long long x = __double_as_longlong(sU[e]) & kAbs;
    if (li && lj && x <= kInf) {
      if (i == j) dia = max(dia, x);
      else off = max(off, x);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    off = max(off, __shfl_xor_sync(0xffffffffu, off, o));
    dia = max(dia, __shfl_xor_sync(0xffffffffu, dia, o));
  }
  if (lane == 0) {
    const double mx = fmax(__longlong_as_double(off), 2.0 * __longlong_as_double(dia));
    atomicMax(&counters[3], (unsigned long long)__double_as_longlong(mx));
  }
}

// Rows ib0, ib0 + step, ... (< n) of P <- P (I - U), g lanes per row; Pf: float32 copy.  The trip
// count is uniform within a warp (a warp stops once none of its rows is left); row values are
// exchanged with shuffles so that no lane reads an element another lane has already overwritten.
__device__ void correct_rows(const double* __restrict__ sU, double* __restrict__ P, int b, int g, int ib0,
                             int ib_end, int step, float* __restrict__ Pf) {
  const int rl = threadIdx.x / g, d = threadIdx.x - rl * g;
  const int gbase = (threadIdx.x & 31) & ~(g - 1);
  const int wrow = (threadIdx.x & ~31) / g;   // first row of this warp within an iteration
  for (int ib = ib0; ib < ib_end; ib += step) {
    if (ib + wrow >= ib_end) break;            // no row of this warp is left (warp-uniform)
    const int i = ib + rl;
    const bool live = i < ib_end && d < b;
    const double p = live ? P[(long long)i * b + d] : 0.0;
    double a0 = p, a1 = 0.0;
    for (int k = 0; k < b; ++k) {
      const double pk = __shfl_sync(0xffffffffu, p, gbase + k);
      if (k <= d) {
        if (k & 1) a0 -= pk * sU[k * b + d];
        else a1 -= pk * sU[k * b + d];
      }
    }
    if (live) {
      const double v = a0 + a1;
      P[(long long)i * b + d] = v;
      if (Pf) Pf[(long long)i * b + d] = (float)v;
    }
  }
}

// The same with the correction P U formed in float32, for |U| <= kCorrectF32: the two conversions and up to b / 2 + 1 roundings
// of each of its b terms are at most b (b / 2 + 3) 2^-24 |U| of the row's largest element, below 2^-53 of it for b = 32.  sUf: U
// in float32.
static constexpr double kCorrectF32 = 3e-12;
__device__ void correct_rows_f32(const float* __restrict__ sUf, double* __restrict__ P, int b, int g, int ib0,
                                 int ib_end, int step, float* __restrict__ Pf) {
  const int rl = threadIdx.x / g, d = threadIdx.x - rl * g;
  const int gbase = (threadIdx.x & 31) & ~(g - 1);
  const int wrow = (threadIdx.x & ~31) / g;   // first row of this warp within an iteration
  for (int ib = ib0; ib < ib_end; ib += step) {
    if (ib + wrow >= ib_end) break;            // no row of this warp is left (warp-uniform)
    const int i = ib + rl;
    const bool live = i < ib_end && d < b;
    const double p = live ? P[(long long)i * b + d] : 0.0;
    const float pf = (float)p;
    float a0 = 0.f, a1 = 0.f;
    for (int k = 0; k < b; k += 2) {
      const float p0 = __shfl_sync(0xffffffffu, pf, gbase + k), p1 = __shfl_sync(0xffffffffu, pf, gbase + k + 1);
      if (d < b) {                             // U is zero below its diagonal
        a0 = fmaf(p0, sUf[k * b + d], a0);
        a1 = fmaf(p1, sUf[(k + 1) * b + d], a1);
      }
    }
    if (live) {
      const double v = p - (double)(a0 + a1);
      P[(long long)i * b + d] = v;
      if (Pf) Pf[(long long)i * b + d] = (float)v;
    }
  }
}

__global__ void __launch_bounds__(ORTH_T)
k_correct(const double* __restrict__ G3, const double* __restrict__ R1, double* __restrict__ Tdiag, int ldT,
          double* __restrict__ Rout, double* __restrict__ P, int n, int b, int g,
          unsigned long long* __restrict__ counters, float* __restrict__ Pf) {
  __shared__ double sU[OB_MAXB * OB_MAXB];   // U(E)
  __shared__ double sR[OB_MAXB * OB_MAXB];
  correct_load_U(G3, b, sU);
  if (blockIdx.x == 0)   // only block 0 forms the product with R1
    for (int e = threadIdx.x; e < b * b; e += blockDim.x) sR[e] = R1[e];
  __syncthreads();
  if (blockIdx.x == 0) correct_coefs(sU, sR, b, Tdiag, ldT, Rout, nullptr);
  if (blockIdx.x == 0 && counters && threadIdx.x < 32) correct_defect(sU, b, counters);
  const int rows_per_block = ORTH_T / g;
  correct_rows(sU, P, b, g, blockIdx.x * rows_per_block, n, gridDim.x * rows_per_block, Pf);
}

int launch_chol(const double* G1, const double* G2, int nq, int b, double* R, double* dinv,
                unsigned long long* counters, cudaStream_t st) {
  switch (b) {
    case 8: k_chol<8><<<1, CHOL_T, 0, st>>>(G1, G2, nq, R, dinv, counters); return 1;
    case 16: k_chol<16><<<1, CHOL_T, 0, st>>>(G1, G2, nq, R, dinv, counters); return 1;
    case 24: k_chol<24><<<1, CHOL_T, 0, st>>>(G1, G2, nq, R, dinv, counters); return 1;
    case 32: k_chol<32><<<1, CHOL_T, 0, st>>>(G1, G2, nq, R, dinv, counters); return 1;
    default: return 0;  // block sizes are multiples of 8 up to 32 (checked by the caller)
  }
}

int launch_correct(const double* G3, const double* R1, double* Tdiag, int ldT, double* Rout, double* P, int n, int b,
                   unsigned long long* counters, cudaStream_t st, float* Pf) {
  const int g = row_group(b);
  const int rows_per_block = ORTH_T / g;
  int blocks = (int)svt_min_ll(svt_ceil_div(n, rows_per_block), 152LL * 8);
  k_correct<<<blocks, ORTH_T, 0, st>>>(G3, R1, Tdiag, ldT, Rout, P, n, b, g, counters, Pf);
  return 1;
}

// ------------------------------------------------------------------------------------------------
// Exact float64 products on the tensor cores.  GB300 executes 2 float64 multiply-adds per clock and SM; float16 MMAs with
// float32 accumulation run at 1024 (measured, mma.sync m16n8k16).  A float64 x with |x| < 2^E is the fixed-point number
// v 2^(E - 62), |v| <= 2^62, and v splits into eight balanced base-256 digits, v = sum_k d_k 256^(7 - k), |d_k| <= 128,
// each exact in float16.  Products of digits are at most 2^14, so sums over up to 128 terms of the (at most eight) pairs
// with i + j = s stay within 2^24: the float32 accumulators are exact.  The pairs with i + j <= 7 (36 MMAs for a 16 x 8 x 16 step)
// are added up exactly, the eight sums put together in integers and rounded once.  What they leave out of a product is
// below 2^-59 of its scale (seven pairs with i + j = 8 of up to 2^14 each), typically 2^-62.  (Splitting into exactly
// representable slices for error-free products is the method of Ozaki, Ogita, Oishi and Rump.)
// The exponents E are those of the CTA's rows: one for all of Q, one per column of P and of C.  (Seven digits lose more than
// float64 sums do where rows differ by 10^4 and more in size: the orthogonality of such blocks went from 5e-16 to 3e-15.)
// A fragment's elements are loaded (L1 holds the chunk) and split by the lane that needs them: no staging, no barriers.
// ------------------------------------------------------------------------------------------------
static constexpr int DG_N = 8;              // digits of a number
static constexpr int DG_NONFINITE = 8000;   // exponent of a column with an infinity or NaN

// Exponent E with |x| < 2^E for the largest absolute high word m of a set of doubles.
__device__ __forceinline__ int dg_exponent(int m) {
  return m >= 0x7FF00000 ? DG_NONFINITE : max((m >> 20) - 1022, -900);
}

// v + 128 (256^0 + .. + 256^7), v = x 2^(62 - E) rounded: digit k = byte (7 - k) - 128.
__device__ __forceinline__ unsigned long long dg_fix(double x, int E) {
  const int hi = __double2hiint(x);
  const int s = min(1022 + E - ((hi >> 20) & 0x7FF), 63);   // >= 0; zeros and denormals: 63 (E >= -900)
  const unsigned long long m =
      ((unsigned long long)(unsigned int)((hi & 0xFFFFF) | 0x100000) << 32) | (unsigned int)__double2loint(x);
  const long long v = (long long)((((m << 10) >> s) + 1) >> 1), sg = (long long)(hi >> 31);
  return (unsigned long long)(v ^ sg) + (0x8080808080808080ULL - (unsigned long long)sg);
}

// Digit k of two numbers as a pair of float16 (x0 in the low half).
__device__ __forceinline__ unsigned int dg_pair(unsigned long long v0, unsigned long long v1, int k) {
  const int byte = 7 - k;
  const unsigned int w0 = byte >= 4 ? (unsigned int)(v0 >> 32) : (unsigned int)v0;
  const unsigned int w1 = byte >= 4 ? (unsigned int)(v1 >> 32) : (unsigned int)v1;
  const unsigned int q = byte & 3;
  // the bytes to positions 0 and 2, then 1024 + n in float16, minus 1152
  const unsigned int t = __byte_perm(w0, w1, q | (q << 4) | ((4 + q) << 8) | ((4 + q) << 12)) & 0x00FF00FFu;
  unsigned int r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(t | 0x64006400u), "r"(0x64806480u));
  return r;
}

__device__ __forceinline__ void mma_f16(float (&c)[4], const unsigned int (&a)[4], unsigned int b0, unsigned int b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// acc[s] += the digit products with i + j = s of one 16 x 8 x 16 step.  va: the lane's eight elements of A in fragment order
// (two consecutive k each), vb: its four of B.
__device__ __forceinline__ void dg_step(float (&acc)[DG_N][4], const unsigned long long (&va)[8],
                                        const unsigned long long (&vb)[4]) {
  unsigned int b0[DG_N], b1[DG_N];
#pragma unroll
  for (int j = 0; j < DG_N; ++j) {
    b0[j] = dg_pair(vb[0], vb[1], j);
    b1[j] = dg_pair(vb[2], vb[3], j);
  }
#pragma unroll
  for (int i = 0; i < DG_N; ++i) {
    unsigned int a[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] = dg_pair(va[2 * q], va[2 * q + 1], i);
#pragma unroll
    for (int j = 0; i + j < DG_N; ++j) mma_f16(acc[i + j], a, b0[j], b1[j]);
  }
}

// The sum of acc[s] 256^(7 - s) as hi 2^32 + lo, in integers (exact for any number of rows), and its value: times 2^(e - 68), e the
// sum of the factors' exponents, rounded once; NaN for the exponents of non-finite columns.  Integer operations: a warp's
// conversion or float64 operation takes 20 cycles of the SM.
struct DgSum {
  long long hi, lo;
  __device__ __forceinline__ void add(const float (&acc)[DG_N][4], int q) {
    int i[DG_N];
#pragma unroll
    for (int s = 0; s < DG_N; ++s) i[s] = __float2int_rn(acc[s][q]);
    hi += (long long)i[0] * 16777216 + ((long long)i[1] * 65536 + ((long long)i[2] * 256 + i[3]));
    lo += (long long)i[4] * 16777216 + ((long long)i[5] * 65536 + ((long long)i[6] * 256 + i[7]));
  }
  __device__ __forceinline__ double value(int e) const {
    long long h = hi + (lo >> 32);
    unsigned int l = (unsigned int)lo;
    const unsigned int sign = h < 0 ? 0x80000000u : 0u;
    if (sign) {
      l = 0u - l;
      h = -h - (l != 0);
    }
    e += 27;                                       // the exponent of the leading bit at bit 63 of h
    if (h == 0) {
      h = l;
      l = 0;
      e -= 32;
    }
    if (e > 4000) return __longlong_as_double(0x7FF8000000000000LL);
    if (h == 0) return 0.0;
    const int z = __clzll(h);
    const unsigned long long top = ((unsigned long long)h << z) | (((unsigned long long)l << 31) >> (63 - z));
    const unsigned long long m = (top >> 11) + ((top >> 10) & 1);   // 2^52 .. 2^53
    e -= z;
    const bool in = e >= -1000 && e <= 1000;
    const double x = __longlong_as_double((long long)(m + ((unsigned long long)(in ? e + 1022 : 1022) << 52)));
    double v = __hiloint2double(__double2hiint(x) | sign, __double2loint(x));
    if (!in) {
      const int e1 = max(-1022, min(1023, e / 2)), e2 = max(-1022, min(1023, e - e1));
      v = v * __hiloint2double((e1 + 1023) << 20, 0) * __hiloint2double((e2 + 1023) << 20, 0);
    }
    return v;
  }
};

// Largest absolute high words of rows [r0, r1): of all of Q into *mq (nq > 0), of every column of P into mp[0 .. B).
// Shared words, zeroed before.  Called by all threads.
template <int B>
__device__ void dg_maxima(const double* __restrict__ Q, long long q_stride, int nq, const double* __restrict__ P,
                          int r0, int r1, int* mq, int* mp) {
  constexpr int CP = B / 2, RT = ORTH_T / CP;      // a thread takes one pair of columns
  const int c = threadIdx.x % CP, r = threadIdx.x / CP;
  auto word = [](double x) { return __double2hiint(x) & 0x7FFFFFFF; };
  int m0 = 0, m1 = 0;
  if (r < RT) {
    for (int blk = 0; blk < nq; ++blk) {
      const double* q = Q + blk * q_stride + 2 * c;
#pragma unroll 4
      for (int i = r0 + r; i < r1; i += RT) {
        const double2 x = *reinterpret_cast<const double2*>(q + (long long)i * B);
        m0 = max(m0, max(word(x.x), word(x.y)));
      }
    }
  }
  if (nq > 0) {
    m0 = __reduce_max_sync(0xffffffffu, m0);
    if ((threadIdx.x & 31) == 0) atomicMax(mq, m0);
    m0 = 0;
  }
  if (r < RT) {
#pragma unroll 4
    for (int i = r0 + r; i < r1; i += RT) {
      const double2 x = *reinterpret_cast<const double2*>(P + (long long)i * B + 2 * c);
      m0 = max(m0, word(x.x));
      m1 = max(m1, word(x.y));
    }
    atomicMax(mp + 2 * c, m0);
    atomicMax(mp + 2 * c + 1, m1);
  }
}

// Partial Gram of rows [r0, r1) in the layout of gram_chunk; eq, ep: exponents of Q and of P's columns.  A warp forms one
// 16 x 8 tile of [Q, P]^T P over the chunk's rows, or a share of them where there are fewer tiles than warps (added up in
// red, ORTH_T / 32 x 128 words).  Called by all threads.
template <int B>
__device__ void dg_gram(const double* __restrict__ Q, long long q_stride, int nq, const double* __restrict__ P, int r0,
                        int r1, int eq, const int* __restrict__ ep, double* __restrict__ partial, bool first,
                        double* __restrict__ red) {
  constexpr int NT = B / 8;
  const int K = nq * B, W = K + B;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int tiles = (W + 15) / 16 * NT;
  const int nk = (r1 - r0 + 15) / 16;
  const int RS = max(1, min(ORTH_T / 32 / tiles, nk));   // row shares
  double* out = partial + (long long)blockIdx.x * gram_entries(nq, B, first);
  auto put = [&](int m, int n, double v) {
    int at = -1;
    if (m < K) {
      at = m * B + n;
    } else if (m < W) {
      const int i = m - K;
      if (first) {
        if (i == n) at = K * B + n;
      } else if (i <= n) {
        at = K * B + upper_index(i, n, B);
      }
    }
    if (at >= 0) out[at] = v;
  };
  for (int item = warp; item < tiles * RS; item += ORTH_T / 32) {   // warp-uniform
    const int tile = item % tiles, share = item / tiles;
    const int m0 = tile / NT * 16, n0 = tile % NT * 8;
    if (m0 - K > n0 + 7) continue;                 // below the diagonal of P^T P
    const int ma = m0 + g, mb = ma + 8;
    const double* pa = ma < K ? Q + ma / B * q_stride + ma % B : P + (ma - K);
    const double* pb = mb < K ? Q + mb / B * q_stride + mb % B : P + (mb - K);
    const bool ina = ma < W, inb = mb < W;
    const int ea = ma < K ? eq : (ina ? ep[ma - K] : 0), eb = mb < K ? eq : (inb ? ep[mb - K] : 0);
    const int en = ep[n0 + g];
    DgSum sum[4] = {};
    for (int k0 = share; k0 < nk; k0 += 8 * RS) {  // float32 sums stay exact over eight steps
      float acc[DG_N][4];
#pragma unroll
      for (int s = 0; s < DG_N; ++s) acc[s][0] = acc[s][1] = acc[s][2] = acc[s][3] = 0.f;
      for (int ks = k0; ks < min(nk, k0 + 8 * RS); ks += RS) {
        unsigned long long va[8], vb[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int r = r0 + 16 * ks + 2 * t + (q & 1) + (q >> 1) * 8;
          const bool in = r < r1;
          const long long at = (long long)r * B;
          // fragment order: (a, rows 2t 2t+1), (b, same), (a, rows + 8), (b, rows + 8)
          va[(q >> 1) * 4 + (q & 1)] = dg_fix(in && ina ? pa[at] : 0.0, ea);
          va[(q >> 1) * 4 + 2 + (q & 1)] = dg_fix(in && inb ? pb[at] : 0.0, eb);
          vb[q] = dg_fix(in ? P[at + n0 + g] : 0.0, en);
        }
        dg_step(acc, va, vb);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) sum[q].add(acc, q);
    }
    const int c0 = n0 + 2 * t;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double v = sum[q].value((q < 2 ? ea : eb) + ep[c0 + (q & 1)]);
      if (RS == 1) put(q < 2 ? ma : mb, c0 + (q & 1), v);
      else red[item * 128 + q * 32 + lane] = v;
    }
  }
  if (RS > 1) {                                    // uniform over the CTA; tiles RS <= 8
    __syncthreads();
    for (int e = threadIdx.x; e < tiles * 128; e += ORTH_T) {
      const int tile = e >> 7, q = (e >> 5) & 3, l = e & 31;
      const int m0 = tile / NT * 16, n0 = tile % NT * 8;
      if (m0 - K > n0 + 7) continue;
      double v = red[tile * 128 + (e & 127)];
      for (int s = 1; s < RS; ++s) v += red[(s * tiles + tile) * 128 + (e & 127)];
      const int m = m0 + (l >> 2) + (q >> 1) * 8, n = n0 + 2 * (l & 3) + (q & 1);
      if (m < W) put(m, n, v);
    }
    __syncthreads();
  }
}

// P <- P - Q C for rows [r0, r1), C (K x B) and the exponents ec of its columns in shared memory; mp: the largest absolute
// high words of P's new columns (shared, zeroed before).  The warps w0 .. w0 + nw - 1 take part; a warp forms a 16 x 8 tile, or
// a share of its steps along K where there are fewer tiles than warps (added up in red, nw x 128 words; bar: the id of
// the barrier of these warps).
template <int B>
__device__ void dg_update(const double* __restrict__ Q, long long q_stride, int nq, const double* __restrict__ sC,
                          const int* __restrict__ ec, int eq, double* __restrict__ P, int r0, int r1, int* mp, int w0,
                          int nw, double* __restrict__ red, int bar) {
  constexpr int NT = B / 8;
  const int K = nq * B, nk = (K + 15) / 16;
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) - w0, g = lane >> 2, t = lane & 3;
  const int tiles = (r1 - r0 + 15) / 16 * NT;
  const int RS = max(1, min(nw / tiles, nk));
  for (int item = warp; item < tiles * RS; item += nw) {   // warp-uniform
    const int tile = item % tiles, share = item / tiles;
    const int ra = r0 + tile / NT * 16 + g, rb = ra + 8, n0 = tile % NT * 8;
    const bool ina = ra < r1, inb = rb < r1;
    const double2 zero = make_double2(0.0, 0.0);
    const int en = ec[n0 + g];
    float acc[DG_N][4];
#pragma unroll
    for (int s = 0; s < DG_N; ++s) acc[s][0] = acc[s][1] = acc[s][2] = acc[s][3] = 0.f;
    for (int ks = share; ks < nk; ks += RS) {      // at most eight steps
      unsigned long long va[8], vb[4];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int c = 16 * ks + 2 * t + 8 * q;     // columns c, c + 1: one block of Q
        const bool in = c < K;
        const double* src = Q + c / B * q_stride + c % B;
        const double2 xa = in && ina ? *reinterpret_cast<const double2*>(src + (long long)ra * B) : zero;
        const double2 xb = in && inb ? *reinterpret_cast<const double2*>(src + (long long)rb * B) : zero;
        va[4 * q] = dg_fix(xa.x, eq);
        va[4 * q + 1] = dg_fix(xa.y, eq);
        va[4 * q + 2] = dg_fix(xb.x, eq);
        va[4 * q + 3] = dg_fix(xb.y, eq);
        vb[2 * q] = dg_fix(in ? sC[c * B + n0 + g] : 0.0, en);
        vb[2 * q + 1] = dg_fix(in ? sC[(c + 1) * B + n0 + g] : 0.0, en);
      }
      dg_step(acc, va, vb);
    }
    const int c0 = n0 + 2 * t;
    double v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      DgSum s = {};
      s.add(acc, q);
      v[q] = s.value(eq + ec[c0 + (q & 1)]);
    }
    if (RS > 1) {                                  // tiles RS <= nw: one item a warp
#pragma unroll
      for (int q = 0; q < 4; ++q) red[item * 128 + q * 32 + lane] = v[q];
      continue;
    }
    int m0 = 0, m1 = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int r = q ? rb : ra;
      if (r < r1) {
        double2* p = reinterpret_cast<double2*>(P + (long long)r * B + c0);
        double2 x = *p;
        x.x -= v[2 * q];
        x.y -= v[2 * q + 1];
        *p = x;
        m0 = max(m0, __double2hiint(x.x) & 0x7FFFFFFF);
        m1 = max(m1, __double2hiint(x.y) & 0x7FFFFFFF);
      }
    }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
      m0 = max(m0, __shfl_xor_sync(0xffffffffu, m0, o));
      m1 = max(m1, __shfl_xor_sync(0xffffffffu, m1, o));
    }
    if (g == 0) {
      atomicMax(mp + c0, m0);
      atomicMax(mp + c0 + 1, m1);
    }
  }
  if (RS > 1) {                                    // uniform over the warps that take part
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(32 * nw) : "memory");
    for (int e = threadIdx.x - 32 * w0; e < tiles * 128; e += 32 * nw) {
      const int tile = e >> 7, q = (e >> 5) & 3, l = e & 31;
      const int r = r0 + tile / NT * 16 + (l >> 2) + (q >> 1) * 8, c = tile % NT * 8 + 2 * (l & 3) + (q & 1);
      if (r < r1) {
        double v = red[tile * 128 + (e & 127)];
        for (int s = 1; s < RS; ++s) v += red[(s * tiles + tile) * 128 + (e & 127)];
        const double x = P[(long long)r * B + c] - v;
        P[(long long)r * B + c] = x;
        atomicMax(mp + c, __double2hiint(x) & 0x7FFFFFFF);
      }
    }
  }
}

// Exponents of the columns of C (K x B, shared) into ec, by the warps w0 .. w0 + nw - 1.
template <int B>
__device__ void dg_col_exponents(const double* __restrict__ sC, int K, int* ec, int w0, int nw) {
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) - w0;
  for (int d = warp; d < B; d += nw) {
    int m = 0;
    for (int c = lane; c < K; c += 32) m = max(m, __double2hiint(sC[c * B + d]) & 0x7FFFFFFF);
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) ec[d] = dg_exponent(m);
  }
}

// ------------------------------------------------------------------------------------------------
// The whole orthonormalisation of one block in one cooperative launch.  The launch sequence above
// (gram, update + gram, Cholesky, update + gram, correction: 8 kernels, each a launch and a pass
// of memory latency) becomes phases of one kernel separated by grid barriers: every CTA owns a
// contiguous chunk of rows for all phases; a Gram is formed as per-CTA partials, a barrier, the
// fixed-order sums spread over all CTAs, and a barrier; every CTA factors
// the b x b block itself (the same warp code on the same data gives the same R1 everywhere), so
// the Cholesky costs no barrier.  What bounds it: barriers and float64 latency up to n ~ 5000 (7 barriers of ~3000 cycles,
// ~9000 of Cholesky, b = 16), the float64 pipe's substitution and the digit products beyond.
// Measured (us; Grams and projections in float64 instructions, one warp's Cholesky before -> now): n = 1000, b = 16,
// nq = 2 44.9 -> 44.9; n = 1000, b = 32, nq = 3 110 -> 92; n = 2753, b = 24, nq = 2 117 -> 87; n = 10000, b = 16, nq = 2
// 102 -> 82; n = 30000, b = 16, nq = 2 223 -> 122, nq = 3 273 -> 133.
// Largest error of a coefficient against 64-bit-mantissa sums, relative to the column: 1.9e-17 -> 1.8e-17 at n = 1000,
// 6.8e-18 -> 3.2e-18 at n = 30000; rows that differ by 10^4 and more: 1.4e-17 -> 1.0e-17.
// ------------------------------------------------------------------------------------------------
// G[e] = sum over k < nblk of partial[k E + e] for the entries e of this CTA's warps.  EP adjacent entries a warp (whole
// memory sectors, few shuffles, and few rounds on small grids), 32 / EP lanes an entry; a lane sums k = l, l + 32 / EP, ... and
// the lanes combine by butterfly: a fixed order.  With Tcol, the coefficient entries e < ncoef also go to Tcol as Gprev + G.
// partial and Gprev may have been written by other CTAs of the same kernel: read through L2.  Measured (cycles at n = 200,
// b = 16, 13 CTAs; one entry a warp before): 11500 -> 5700.
template <int EP>
__device__ void reduce_entries_ep(const double* __restrict__ partial, int nblk, int E, double* __restrict__ G,
                                  const double* Gprev, double* __restrict__ Tcol, int ldT, int ncoef, int b,
                                  unsigned int* err) {
  constexpr int L = 32 / EP;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int e0 = (blockIdx.x * nw + warp) * EP; e0 < E; e0 += gridDim.x * nw * EP) {   // warp-uniform
    const int e = e0 + lane % EP;
    double s = 0.0;
    if (e < E) {
      for (int k = lane / EP; k < nblk; k += 8 * L) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = k + u * L < nblk ? __ldcg(partial + (long long)(k + u * L) * E + e) : 0.0;
        s += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
      }
    }
#pragma unroll
    for (int o = EP; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane < EP && e < E) {
      if (err && !isfinite(s)) svt_set_error(err, SVT_DEVERR_NONFINITE);
      G[e] = s;
      if (Tcol && e < ncoef) {
        const int i = e / b, j = e - i * b;
        Tcol[i * ldT + j] = (Gprev ? __ldcg(Gprev + e) : 0.0) + s;
      }
    }
  }
}
// FEW: 8 columns, fewer entries than warps on large grids: fewer entries a warp and so one round of loads (n = 2753: 46.9 -> 45.4
// us a block).
template <bool FEW>
__device__ __forceinline__ void reduce_entries(const double* __restrict__ partial, int nblk, int E,
                                               double* __restrict__ G, const double* Gprev, double* __restrict__ Tcol,
                                               int ldT, int ncoef, int b, unsigned int* err) {
  if (FEW && nblk > 128) reduce_entries_ep<1>(partial, nblk, E, G, Gprev, Tcol, ldT, ncoef, b, err);
  else if (nblk <= (FEW ? 64 : 128)) reduce_entries_ep<4>(partial, nblk, E, G, Gprev, Tcol, ldT, ncoef, b, err);
  else reduce_entries_ep<2>(partial, nblk, E, G, Gprev, Tcol, ldT, ncoef, b, err);
}

// The same sums by every CTA for itself (one grid barrier less, for small grids): the K b coefficients into sC, the other
// entries into sTail (both shared).  Every CTA adds in the same order: the same bits everywhere.  CTA 0 also writes G and
// Tcol.  Called by all threads.
__device__ void reduce_all(const double* __restrict__ partial, int nblk, int E, double* __restrict__ G,
                           const double* Gprev, double* __restrict__ Tcol, int ldT, int ncoef, int b,
                           double* __restrict__ sC, double* __restrict__ sTail, unsigned int* err) {
  for (int e = threadIdx.x; e < E; e += ORTH_T) {
    double s0 = 0.0, s1 = 0.0;
    for (int k = 0; k < nblk; k += 16) {
      double v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = k + u < nblk ? __ldcg(partial + (long long)(k + u) * E + e) : 0.0;
      s0 += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
      s1 += ((v[8] + v[9]) + (v[10] + v[11])) + ((v[12] + v[13]) + (v[14] + v[15]));
    }
    const double s = s0 + s1;
    if (e < ncoef) sC[e] = s;
    else sTail[e - ncoef] = s;
    if (blockIdx.x == 0) {
      if (err && !isfinite(s)) svt_set_error(err, SVT_DEVERR_NONFINITE);
      if (Tcol && e < ncoef) {
        const int i = e / b, j = e - i * b;
        Tcol[i * ldT + j] = (Gprev ? __ldcg(Gprev + e) : 0.0) + s;
      }
      G[e] = s;
    }
  }
}

// Tdiag = A B for upper triangular b x b A, B in shared memory (the composed diagonal block of a
// repeated pass).  All threads of one CTA.
__device__ void compose_upper(const double* __restrict__ sA, const double* __restrict__ sB, int b,
                              double* __restrict__ Tdiag, int ldT) {
  for (int e = threadIdx.x; e < b * b; e += blockDim.x) {
    const int i = e / b, j = e - i * b;
    double v = 0.0;
    for (int k = i; k <= j; ++k) v += sA[i * b + k] * sB[k * b + j];
    Tdiag[i * ldT + j] = v;
  }
}

// Tcol += (C3 + C4) R1 with C3, C4 the coefficient rows (K x b) of the repeated pass in G1 / G2 and
// R1 (upper triangular, shared memory) the first pass's factor: the first pass wrote Tcol = C1 + C2.
// Entries spread over all threads of the grid; G1, G2 and Tcol were written by other CTAs of the
// same kernel and are read through L2.
__device__ void compose_coefs(const double* __restrict__ G1, const double* __restrict__ G2,
                              const double* __restrict__ sR1, int K, int b, double* __restrict__ Tcol, int ldT) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < K * b; e += gridDim.x * blockDim.x) {
    const int i = e / b, j = e - i * b;
    double v = 0.0;
    for (int k = 0; k <= j; ++k) v += (__ldcg(G1 + i * b + k) + __ldcg(G2 + i * b + k)) * sR1[k * b + j];
    Tcol[i * ldT + j] = __ldcg(Tcol + i * ldT + j) + v;
  }
}

struct OrthCoopArgs {
  double* P;                  // rows x b, orthonormalised in place
  const double* Q;            // nq blocks of rows x b, q_stride apart
  long long q_stride;
  int nq, n, g, rpc;          // rpc: rows per CTA
  double *partial, *G1, *G2, *G3;
  long long part_half;        // doubles of one of the two sets of partials (0: one set)
  double *Tcol, *Tdiag;       // coefficient outputs (may be NULL), leading dimension ldT
  int ldT;
  float* Pf;                  // float32 copy of the result (may be NULL)
  unsigned long long* counters;
  unsigned int* err;
  unsigned int* bar;          // grid barrier word
  int twoc;                   // second first-order correction
  double repass;              // defect of the first pass above which the whole pass is repeated
                              // (<= 0: never)
  unsigned int spin_limit;    // polls of a barrier wait before it gives up
};

static constexpr size_t orth_coop_smem(int B) {
  return (size_t)(OB_MAXK * B + 4 * B * B + B) * sizeof(double);
}

// sU = U(E) as correct_load_U, and max |E| over the live columns (the quantity correct_defect records; here rounded to
// float32) as the bits of a float into *defect (shared, zeroed before).  sG: upper triangle of the Gram in shared memory; a
// deflated column has a zero diagonal, a live one a diagonal above 1/2.  NaN entries are ignored.  All threads.
__device__ void load_U_defect(const double* __restrict__ sG, int b, double* __restrict__ sU, int* defect) {
  int mx = 0;
  for (int e = threadIdx.x; e < b * b; e += blockDim.x) {
    const int i = e / b, j = e - i * b;
    double v = 0.0;
    if (j >= i) {
      const double x = sG[upper_index(i, j, b)] - (i == j ? 1.0 : 0.0);
      v = (j > i) ? x : 0.5 * x;
      const int hi = __double2hiint(sG[upper_index(i, i, b)]), hj = __double2hiint(sG[upper_index(j, j, b)]);
      const int f = __float_as_int(fabsf((float)x));
      if (hi > 0x3FE00000 && hj > 0x3FE00000 && f <= 0x7F800000) mx = max(mx, f);
    }
    sU[e] = v;
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) atomicMax(defect, mx);
}

// FMA: float64 instructions instead of digit products (B = 8), a kernel of its own with no more code than it runs: every phase
// runs once a launch, and fetching its instructions takes as long as running them.  In one kernel with the digit products and
// with 20 entries a thread in gram_chunk, the second Gram took 9000 cycles at n = 1000; a block 37 us, now 31 (n = 200: 32.5 -> 28).
template <int B, bool FMA>
__global__ void __launch_bounds__(ORTH_T, 2) k_orth_coop(OrthCoopArgs a) {
  extern __shared__ double sm_orth[];
  double* sC = sm_orth;                 // K x B coefficients (C1, then C2)
  double* sR = sC + OB_MAXK * B;        // R of the current pass
  double* sU = sR + B * B;              // U(E)
  double* sR2 = sU + B * B;             // R diag(1 / diag(R)); then (I + U(E)) R of a first correction
  double* sD = sR2 + B * B;             // 1 / diag(R)
  double* sR1 = sD + B;                 // R of the first pass, kept when the pass is repeated
  __shared__ int s_def[2];              // defect of each pass, float bits
  __shared__ double s_red[ORTH_T / 32 * 128];
  __shared__ double sRef[B], sTail[B * (B + 1) / 2];   // squared norms before the projections; upper triangle of a Gram
  __shared__ double s_fill[B];          // size of the random part of a deflated column, 0: not deflated
  __shared__ bool s_keep[B];
  __shared__ int s_mq, s_mp[2][B], s_ep[B], s_ec[B];   // largest high words (two sets in turn) and exponents
  // a barrier of an earlier cooperative kernel gave up: the whole grid returns at once
  if (*(volatile unsigned int*)a.err & SVT_DEVERR_BARRIER) return;
  const int K = a.nq * B;
  const int nb = gridDim.x;
  const int r0 = blockIdx.x * a.rpc;
  const int r1 = min(a.n, r0 + a.rpc);
  const int step = ORTH_T / a.g;
  const int nw = ORTH_T / 32;
  if (threadIdx.x == 0) s_mq = s_def[0] = s_def[1] = 0;
  if (threadIdx.x < 2 * B) (&s_mp[0][0])[threadIdx.x] = 0;
  __syncthreads();
  constexpr bool digits = !FMA;
  if constexpr (digits) dg_maxima<B>(a.Q, a.q_stride, a.nq, a.P, r0, r1, &s_mq, s_mp[0]);
  __syncthreads();
  const int eq = dg_exponent(s_mq);
  // exponents of P's columns from the maxima in s_mp[cur]; the other set is cleared for the next change of P
  int cur = 0;
  auto next_exponents = [&]() {
    if (threadIdx.x < B) {
      s_ep[threadIdx.x] = dg_exponent(s_mp[cur][threadIdx.x]);
      s_mp[cur ^ 1][threadIdx.x] = 0;
    }
    cur ^= 1;
    __syncthreads();
  };
  next_exponents();
  // Partial Gram [Q_0 .. Q_{nq-1}, P]^T P of the CTA's rows; P <- P - Q C from warp w0 on (bar as for dg_update)
  auto gram = [&](int nq, double* part, bool first) {
    if constexpr (FMA) {
      __syncthreads();
      gram_chunk<(GRAM_MAXW * B + ORTH_T - 1) / ORTH_T>(a.Q, a.q_stride, nq, a.P, B, r0, r1, part, first);
    } else {
      dg_gram<B>(a.Q, a.q_stride, nq, a.P, r0, r1, eq, s_ep, part, first, s_red);
    }
  };
  auto project = [&](int w0, int bar) {
    if constexpr (FMA) update_rows(0, a.Q, a.q_stride, a.nq, sC, nullptr, nullptr, a.P, B, a.g, r0, r1, nullptr, 32 * w0);
    else dg_update<B>(a.Q, a.q_stride, a.nq, sC, s_ec, eq, a.P, r0, r1, s_mp[cur], w0, nw - w0, s_red, bar);
  };
  // Where every CTA adds up a Gram for itself, one may still read its partials while another writes the next Gram's: two sets
  // in turn.  (Else a barrier follows the sums, and the sets are the same.)
  double* partial = a.partial;
  // After a partial Gram: the sums of all CTAs, the coefficients in sC and the rest in sTail.  false: a barrier gave up.
  auto gram_sums = [&](int nq, bool first, double* G, const double* Gprev, double* Tcol, double* sTail,
                       unsigned int* err) -> bool {
    const int E = gram_entries(nq, B, first), nc = nq * B * B;
    if (!svt_grid_barrier(a.bar, a.err, a.spin_limit)) return false;
    const double* part = partial;
    partial = partial == a.partial ? a.partial + a.part_half : a.partial;
    if (nq == 0 && nb <= OC_SETS_GRID) {   // (with coefficients the CTAs' reads take longer than the barrier: 16000 cycles at n = 1000)
      reduce_all(part, nb, E, G, Gprev, Tcol, a.ldT, nc, B, sC, sTail, err);
    } else {
      reduce_entries<FMA>(part, nb, E, G, Gprev, Tcol, a.ldT, nc, B, err);
      if (!svt_grid_barrier(a.bar, a.err, a.spin_limit)) return false;
      for (int e = threadIdx.x; e < E; e += ORTH_T) {
        const double v = __ldcg(G + e);
        if (e < nc) sC[e] = v;
        else sTail[e - nc] = v;
      }
    }
    __syncthreads();
    return true;
  };
  // Pass 0 is block CGS2 + Cholesky QR.  When its result is far from orthonormal (a block with
  // nearly dependent columns: Cholesky QR loses orthogonality as cond(P)^2 eps, and a column that
  // lost most of its norm to the projections keeps components along Q of eps / (its norm ratio)),
  // pass 1 repeats CGS2 + Cholesky QR on that result (the Cholesky QR2 remedy), and the
  // coefficients compose: P_in = Q (C_a + C_b R_a) + P_out (R_b R_a).
  for (int pass = 0; pass < 2; ++pass) {
    if (a.nq > 0) {
      // C1 = Q^T P (with the diagonal of P^T P)
      gram(a.nq, partial, true);
      if (!gram_sums(a.nq, true, a.G1, nullptr, nullptr, sRef, a.err)) return;
      // P <- P - Q C1; [C2; A] = [Q, P]^T P; coefficients C1 + C2 -> Tcol (first pass)
      if constexpr (digits) dg_col_exponents<B>(sC, K, s_ec, 0, nw);
      __syncthreads();
      project(0, 3);
      __syncthreads();
      next_exponents();
      gram(a.nq, partial, false);
      if (!gram_sums(a.nq, false, a.G2, a.G1, pass == 0 ? a.Tcol : nullptr, sTail, nullptr)) return;
      if constexpr (digits) dg_col_exponents<B>(sC, K, s_ec, 0, nw);
      __syncthreads();
    } else {
      gram(0, partial, false);
      if (!gram_sums(0, false, a.G2, nullptr, nullptr, sTail, a.err)) return;
    }
    // R = chol(A) in every CTA, by its first four warps, while the others project P <- P - Q C2; then
    // P <- P R^-1 (forward substitution) by the whole CTA; E = P^T P - I
    if (threadIdx.x < CHOL_T) {
      // deflated columns are counted in the first pass (a repeated pass sees them again as zeros)
      chol_warps<B>(sTail, a.nq > 0 ? sRef : nullptr, sR, sD,
                    (blockIdx.x == 0 && pass == 0) ? a.counters : nullptr);
    } else if (a.nq > 0) {
      project(CHOL_T / 32, 1);
    }
    __syncthreads();
    // Deflated columns (zero rows of R: the pivot is at or below the rounding of A) of the first pass keep what the
    // substitution leaves of them, with a coefficient of one, plus a random direction at the rounding level of the
    // column; the repeated pass normalises that to working precision.  P_in = Q C + P R still holds for them: zeroed
    // instead, a column may lose components of 1e-7 of its norm (a noise pivot against a true one of 1e-8), with which
    // the Ritz values stagnate.  A column that was zero becomes random, with no coefficient (block Lanczos breakdown:
    // the block keeps its width, so the Krylov space keeps growing).
    int ndef = 0;
    if (pass == 0 && a.repass > 0.0) {
      for (int j = 0; j < B; ++j) ndef += sD[j] == 0.0 ? 1 : 0;
      if (ndef > 0) {
        if (threadIdx.x < B) {
          const int j = threadIdx.x;
          const double ref = a.nq > 0 ? sRef[j] : sTail[upper_index(j, j, B)];
          const bool live = ref > 1e-250 && ref < 1e250;
          s_fill[j] = sD[j] != 0.0 ? 0.0 : (live ? 0x1p-52 * sqrt(ref / (double)a.n) : 1.0);
          s_keep[j] = sD[j] != 0.0 || live;
        }
        __syncthreads();
        if (threadIdx.x < B && s_fill[threadIdx.x] != 0.0 && s_keep[threadIdx.x]) {
          sR[threadIdx.x * B + threadIdx.x] = 1.0;
          sD[threadIdx.x] = 1.0;
        }
        __syncthreads();
      }
    }
    for (int t = threadIdx.x; t < B * B; t += blockDim.x) sR2[t] = sR[t] * sD[t % B];
    // (the maxima of the projection above are not used)
    if (threadIdx.x < B) s_mp[cur][threadIdx.x] = 0;
    __syncthreads();
    bool by_row = false;
    if constexpr (B <= 16) {
      by_row = r1 - r0 >= 64;
      if (by_row) solve_rows<B>(sR2, sD, a.P, r0, r1, s_mp[cur]);
    }
    if (!by_row) update_rows(1, nullptr, 0, 0, nullptr, sR2, sD, a.P, B, a.g, r0, r1, digits ? s_mp[cur] : nullptr);
    if (ndef > 0) {
      __syncthreads();   // the substitution above wrote these rows
      // the seed comes from R, identical in every CTA and different from block to block
      const unsigned long long seed =
          (unsigned long long)__double_as_longlong(sR[0]) ^ ((unsigned long long)a.nq << 40) ^ (unsigned long long)a.n;
      for (int e = threadIdx.x; e < (r1 - r0) * B; e += blockDim.x) {
        const int i = r0 + e / B, j = e - (e / B) * B;
        if (s_fill[j] != 0.0) {
          double* p = a.P + (long long)i * B + j;
          const double u = s_fill[j] * svt_uniform_pm1(seed, (unsigned long long)i * B + j);
          *p = s_keep[j] ? *p + u : u;
        }
      }
      for (int t = threadIdx.x; t < B * B; t += blockDim.x) sR1[t] = sR[t];
      if (threadIdx.x == 0 && blockIdx.x == 0 && a.counters) atomicAdd(&a.counters[4], 1ull);
      __syncthreads();
      dg_maxima<B>(nullptr, 0, 0, a.P, r0, r1, nullptr, s_mp[cur]);   // (on top of the old columns' maxima)
      __syncthreads();
      next_exponents();
      continue;
    }
    __syncthreads();
    next_exponents();
    gram(0, partial, false);
    if (!gram_sums(0, false, a.G3, nullptr, nullptr, sTail, nullptr)) return;
    load_U_defect(sTail, B, sU, &s_def[pass]);
    __syncthreads();
    // every CTA takes the same decisions from the same G3
    const double defect = (double)__int_as_float(s_def[pass]);
    if (pass == 0 && a.repass > 0.0 && defect > a.repass) {
      if (threadIdx.x == 0 && blockIdx.x == 0 && a.counters) {
        atomicAdd(&a.counters[4], 1ull);
        atomicMax(&a.counters[5], (unsigned long long)__double_as_longlong(defect));
      }
      for (int t = threadIdx.x; t < B * B; t += blockDim.x) sR1[t] = sR[t];
      __syncthreads();
      continue;
    }
    const bool second = pass == 1;
    if (!a.twoc) {
      // the coefficients by the last CTA, the defect by CTA 0
      if (blockIdx.x == nb - 1) {
        if (!second) {
          correct_coefs(sU, sR, B, a.Tdiag, a.ldT, nullptr, nullptr);
        } else if (a.Tdiag) {
          correct_coefs(sU, sR, B, nullptr, 0, nullptr, sR2);
          __syncthreads();
          compose_upper(sR2, sR1, B, a.Tdiag, a.ldT);
        }
      }
      if (blockIdx.x == 0 && a.counters && threadIdx.x == 0)
        atomicMax(&a.counters[3], (unsigned long long)__double_as_longlong(defect));
      if (second && a.Tcol && a.nq > 0) compose_coefs(a.G1, a.G2, sR1, K, B, a.Tcol, a.ldT);
      if (defect <= kCorrectF32) {
        float* sUf = reinterpret_cast<float*>(sC);
        for (int t = threadIdx.x; t < B * B; t += blockDim.x) sUf[t] = (float)sU[t];
        __syncthreads();
        correct_rows_f32(sUf, a.P, B, a.g, r0, r1, step, a.Pf);
      } else {
        correct_rows(sU, a.P, B, a.g, r0, r1, step, a.Pf);
      }
      return;
    }
    // two first-order corrections: P^T P = I up to O(|E|^4)
    correct_coefs(sU, sR, B, nullptr, 0, nullptr, sR2);
    if (blockIdx.x == 0 && a.counters && threadIdx.x == 0)
      atomicMax(&a.counters[3], (unsigned long long)__double_as_longlong(defect));
    correct_rows(sU, a.P, B, a.g, r0, r1, step, nullptr);
    __syncthreads();
    dg_maxima<B>(nullptr, 0, 0, a.P, r0, r1, nullptr, s_mp[cur]);
    __syncthreads();
    next_exponents();
    gram(0, partial, false);
    if (!gram_sums(0, false, a.G3, nullptr, nullptr, sTail, nullptr)) return;
    correct_load_U(sTail, B, sU);
    __syncthreads();
    if (blockIdx.x == nb - 1) {
      if (!second) {
        correct_coefs(sU, sR2, B, a.Tdiag, a.ldT, nullptr, nullptr);
      } else if (a.Tdiag) {
        correct_coefs(sU, sR2, B, nullptr, 0, nullptr, sR);
        __syncthreads();
        compose_upper(sR, sR1, B, a.Tdiag, a.ldT);
      }
    }
    if (second && a.Tcol && a.nq > 0) compose_coefs(a.G1, a.G2, sR1, K, B, a.Tcol, a.ldT);
    correct_rows(sU, a.P, B, a.g, r0, r1, step, a.Pf);
    return;
  }
}

template <int B, bool FMA>
static bool orth_coop_attr() {
  return cudaFuncSetAttribute(k_orth_coop<B, FMA>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)orth_coop_smem(B)) == cudaSuccess;
}

template <int B, bool FMA>
static int orth_coop_blocks_per_sm() {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_orth_coop<B, FMA>, ORTH_T, orth_coop_smem(B)) != cudaSuccess)
    return 0;
  return nb;
}

// Largest co-resident grid of the cooperative kernel for every block size (the same bound is
// used for all, the smallest of them), capped at two CTAs per SM.  0 if unavailable.
int orth_coop_init() {
  // once per process (contexts may be created from several threads)
  static std::once_flag once;
  static int grid = 0;
  std::call_once(once, [] {
    int dev = 0, sms = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) {
      (void)cudaGetLastError();
      return;
    }
    if (!orth_coop_attr<8, true>() || !orth_coop_attr<8, false>() || !orth_coop_attr<16, false>() ||
        !orth_coop_attr<24, false>() || !orth_coop_attr<32, false>()) {
      (void)cudaGetLastError();
      return;
    }
    int bps = std::min({orth_coop_blocks_per_sm<8, true>(), orth_coop_blocks_per_sm<8, false>(),
                        orth_coop_blocks_per_sm<16, false>(), orth_coop_blocks_per_sm<24, false>(),
                        orth_coop_blocks_per_sm<32, false>()});
    bps = std::min(bps, 2);
    grid = bps * sms;
  });
  return grid;
}

int launch_orth_coop(double* P, const double* Q, long long q_stride, int nq, int n, int b, double* partial,
                     double* G1, double* G2, double* G3, double* Tcol, double* Tdiag, int ldT, float* Pf,
                     unsigned long long* counters, unsigned int* err, void* bar, int twoc, int max_grid,
                     cudaStream_t st, double repass, unsigned int spin_limit) {
  const int gmax = std::min(orth_coop_init(), max_grid);
  if (gmax <= 0 || n <= 0) return 0;
  // At least 16 rows per CTA (a step of the digit products) and at most gmax CTAs.  A block of 8 columns of a small problem
  // leaves most warps without a tile; float64 instructions on chunks of 8 and more rows take less (us, nq = 2 or so: n = 2753
  // 42.9 against 45.4, 7000 49.7 against 52.5, 10000 61.8 against 55.5); n = 200, b = 16 takes 47 us either way.
  const bool fma = b == 8 && n <= 24 * gmax;
  const int rpc = std::max(fma ? 8 : 16, (n + gmax - 1) / gmax);
  const int grid = (n + rpc - 1) / rpc;
  OrthCoopArgs a;
  a.P = P; a.Q = Q; a.q_stride = q_stride; a.nq = nq; a.n = n; a.g = row_group(b); a.rpc = rpc;
  a.partial = partial; a.part_half = grid <= OC_SETS_GRID ? (long long)grid * gram_entries(nq, b, false) : 0; a.G1 = G1; a.G2 = G2; a.G3 = G3;
  a.Tcol = Tcol; a.Tdiag = Tdiag; a.ldT = ldT; a.Pf = Pf;
  a.counters = counters; a.err = err; a.bar = static_cast<unsigned int*>(bar); a.twoc = twoc;
  a.repass = repass;
  a.spin_limit = spin_limit;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(ORTH_T);
  cfg.dynamicSmemBytes = orth_coop_smem(b);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e;
  switch (b) {
    case 8: e = fma ? cudaLaunchKernelEx(&cfg, k_orth_coop<8, true>, a) : cudaLaunchKernelEx(&cfg, k_orth_coop<8, false>, a); break;
    case 16: e = cudaLaunchKernelEx(&cfg, k_orth_coop<16, false>, a); break;
    case 24: e = cudaLaunchKernelEx(&cfg, k_orth_coop<24, false>, a); break;
    case 32: e = cudaLaunchKernelEx(&cfg, k_orth_coop<32, false>, a); break;
    default: return 0;
  }
  return e == cudaSuccess ? 1 : 0;
}

}  // namespace svt
