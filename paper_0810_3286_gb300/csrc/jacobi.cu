// Projected SVD of the Lanczos partial SVD: T (K x K, K = J b <= 128, block upper triangular) = Xl diag(theta) Wr^T for
// the leading nv triplets (the ones a thick restart keeps; they cover every wanted triplet).  Sec. 5.1.1: the
// singular values of the small projected matrix are the Ritz values of Y, compared against tau by the rank policy.
//
// GB300 runs float64 at 1/64 of the float32 rate with ~64 cycles per dependent operation, so the iteration runs
// where neither is met, and float64 is left to matrix products spread over a thread-block cluster:
//   1. k_psvd_sweeps: cyclic two-sided Jacobi in float32 on M = T^T T (scaled).  A round of the round-robin tournament
//      rotates K/2 disjoint pairs; a rotation needs only M_pp, M_qq and M_pq, no inner products.  M lives in the
//      shared memory of CTA 0 as 2 x 2 blocks of pairs, written back to the places of the next round (Brent & Luk's
//      systolic order), so the addresses are the same in every round.  The rotations W are not accumulated there:
//      the (c, s) of a sweep go to a log, and the other CTAs of the cluster replay it on their rows of W.
//   2. k_psvd_refine: W back to orthonormality (float64 by one first-order step), then a first-order perturbation
//      step on the leading nv columns, repeated until its own residual estimate meets the tolerance:
//      S = W^T (T^T T) W[:, :nv], Theta_ji = the Jacobi angle of (S_ji, lambda_i, lambda_j), W <- W exp(Theta).  Everything
//      is a matrix product; each step squares the error (as in Ogita and Aishima's refinement of eigenvectors).  theta_i =
//      ||T w_i||, x_i = T w_i / theta_i.
// Measured (GB300, one call, random block-bidiagonal T; before: float32 one-sided sweeps with accumulated rotations and
// one float64 one-sided sweep, in CTA 0): K = 48, nv = 16: 533 -> 115 us (50 us sweeps, 65 us refinement); K = 72, nv = 24:
// 1350 -> 281; K = 96, nv = 32: 3515 -> 490; K = 128, nv = 64: 9600 -> 1120 us; |T^T X - W theta| / sigma_1 from 1e-10 .. 1.6e-9 to
// 2e-12 .. 1.7e-11.  The sweeps are bound by the latency of a round (~310 cycles at K = 48: one barrier, two dependent
// shared-memory reads, two reciprocal square roots), above K = 64 by instruction issue; the refinement by float64 latency
// (64 cycles an operation) at K = 48 and by the float64 pipes of the cluster at K = 128.
// A T whose leading nv values span more than a factor 100 has small values that the float32 M does not resolve: one-sided
// (Hestenes) Jacobi sweeps in float32 on G = T W carry its rotations on.  In float64 contexts, and where step 2 does not
// converge, T is then finished by one-sided sweeps in float64 in CTA 0, which are accurate relative to each singular value
// (step 2's errors are relative to sigma_1^2).
//
// Residual estimates of the Lanczos relation: res_k = || S x_k[last b rows] || with S the b x b upper triangular
// factor of the last block (Y^T U_J = V T^T + V_{J+1} S E_J^T).
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace svt {

static constexpr int JMAXK = 128;
static constexpr int PS_T = 512;              // threads per CTA
static constexpr int kTinSmem = 96;           // largest K with T in shared memory during the refinement
static constexpr int PS_LOG = 4;              // sweeps of the rotation log in flight
static constexpr int kJacobiCluster = 8;      // CTAs of the cluster (1 where a cluster launch is not possible)

// Workspace of one projected SVD (offsets in doubles).
static constexpr int PS_KK = JMAXK * JMAXK;
static constexpr int PS_W0 = 0, PS_W1 = PS_KK, PS_Z = 2 * PS_KK, PS_TH = 3 * PS_KK, PS_G = 4 * PS_KK, PS_E = 5 * PS_KK;
static constexpr int PS_WF = 6 * PS_KK;                       // float K x K
static constexpr int PS_LAM = PS_WF + PS_KK / 2;              // lambda of the leading nv columns
static constexpr int PS_DIAG = PS_LAM + JMAXK;                // diagonal of M after the sweeps, decreasing
static constexpr int PS_MISC = PS_DIAG + JMAXK;               // scale, then floats: statistics, flags
static constexpr int PS_LOGO = PS_MISC + 128;                 // rotation log: PS_LOG x (K - 1) x K/2 float2
static constexpr int PS_DOUBLES = PS_LOGO + PS_LOG * (JMAXK - 1) * (JMAXK / 2);
long long psvd_workspace_doubles() { return PS_DOUBLES; }

// Reciprocal and reciprocal square root in float64 by Newton's iteration from the float32 hardware
// approximations (GB300's float64 divide and square root take ~650 cycles): each step squares the
// relative error, 2^-23 -> ~1e-14 -> rounding.
__device__ __forceinline__ double rcp_nr(double x) {
  double y = (double)__frcp_rn((float)x);
  y = y * (2.0 - x * y);
  y = y * (2.0 - x * y);
  return y;
}
__device__ __forceinline__ double rcp_nr1(double x) {
  const double y = (double)__frcp_rn((float)x);
  return y * (2.0 - x * y);
}
__device__ __forceinline__ double rsqrt_nr(double x, int steps) {
  double y = (double)rsqrtf((float)x);
  for (int i = 0; i < steps; ++i) y = y * (1.5 - 0.5 * x * y * y);
  return y;
}

// ------------------------------------------------------------------------------------------------
// Cluster helpers
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ int cl_rank() {
  unsigned int r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ int cl_size() {
  unsigned int r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return (int)r;
}
// Cluster barrier, split: orders shared and global memory between the CTAs of the cluster.  A CTA alone in its
// cluster passes at once, so threads of one CTA are synchronised by it as well.
__device__ __forceinline__ void cl_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cl_sync() {
  cl_arrive();
  cl_wait();
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

struct PsvdArgs {
  const double* T;
  int ldT, K;
  const double* S;
  int b, nv;
  double *theta, *Xl, *Wr, *res;
  double tol;
  int f32;                    // T comes from float32 products
  int max_sweeps;
  unsigned int* err;
  unsigned long long* counters;
  double* ws;
};

// ------------------------------------------------------------------------------------------------
// 1. float32 sweeps on M = T^T T
// ------------------------------------------------------------------------------------------------
// Place of element p (0 .. 2h - 1, pair p / 2, top or bottom) in the next round: the top of pair 0 stays, the other tops
// move one pair up, the bottoms one pair down, the ends turn round.  K - 1 rounds return every element to its place,
// and every two elements have met once.
__device__ __forceinline__ int next_place(int p, int h) {
  const int i = p >> 1;
  if (!(p & 1)) return i == 0 ? 0 : (i == h - 1 ? 2 * h - 1 : 2 * (i + 1));
  return i == 0 ? 2 : 2 * (i - 1) + 1;
}

// Integer that orders like x; NaNs come before or after all numbers.
__device__ __forceinline__ int order_bits(float x) {
  const int b = __float_as_int(x);
  return b ^ ((b >> 31) & 0x7FFFFFFF);
}

__device__ __forceinline__ float rsqrt_ftz(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Number of block (I, J), I < J, among the h (h - 1) / 2 blocks above the diagonal, row by row, and back.
__device__ __forceinline__ int block_number(int I, int J, int h) { return I * (2 * h - I - 1) / 2 + (J - I - 1); }
__device__ __forceinline__ void pair_block(int e, int h, int& I, int& J) {
  I = 0;
  int n = h - 1;
  while (e >= n) {
    e -= n;
    ++I;
    --n;
  }
  J = I + 1 + e;
}

// One row of W (K values in shared memory, in places) through the rotations of a sweep.  One warp; lane l holds the
// pairs l PP .. l PP + PP - 1.  The log is read through L2, eight rounds at a time.
template <int PP>
__device__ void replay_row(float* __restrict__ row, const float2* __restrict__ log, int h) {
  const int lane = threadIdx.x & 31;
  const int K = 2 * h;
  float t[PP], bo[PP];
#pragma unroll
  for (int s = 0; s < PP; ++s) {
    const int i = lane * PP + s;
    t[s] = i < h ? row[2 * i] : 0.f;
    bo[s] = i < h ? row[2 * i + 1] : 0.f;
  }
  for (int r0 = 0; r0 < K - 1; r0 += 8) {
    float2 cs[8][PP];
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
      for (int s = 0; s < PP; ++s) {
        const int i = lane * PP + s;
        cs[u][s] = (r0 + u < K - 1 && i < h) ? __ldcg(log + (r0 + u) * h + i) : make_float2(1.f, 0.f);
      }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (r0 + u >= K - 1) break;   // warp-uniform
      float a[PP], c[PP];
#pragma unroll
      for (int s = 0; s < PP; ++s) {
        a[s] = cs[u][s].x * t[s] - cs[u][s].y * bo[s];
        c[s] = cs[u][s].y * t[s] + cs[u][s].x * bo[s];
      }
      const float up = __shfl_up_sync(0xffffffffu, a[PP - 1], 1);
      const float dn = __shfl_down_sync(0xffffffffu, c[0], 1);
      const float b0 = __shfl_sync(0xffffffffu, c[0], 0);
#pragma unroll
      for (int s = 0; s < PP; ++s) {
        const int i = lane * PP + s;
        t[s] = i == 0 ? a[s] : (i == 1 ? b0 : (s > 0 ? a[s > 0 ? s - 1 : 0] : up));
        bo[s] = i == h - 1 ? a[s] : (s + 1 < PP ? c[s + 1 < PP ? s + 1 : s] : dn);
      }
    }
  }
#pragma unroll
  for (int s = 0; s < PP; ++s) {
    const int i = lane * PP + s;
    if (i < h) {
      row[2 * i] = t[s];
      row[2 * i + 1] = bo[s];
    }
  }
}

// NB: blocks per thread (ceil(h (h - 1) / 2 / block threads)); NP = ceil(h / 32): warps that compute the rotations, one pair
// per lane (the other 16 - NP rotate blocks); HC: K / 2 at compile time for the sizes of the default cycles (0: any), so
// that the planes are immediate offsets: with several blocks a thread the rounds are bound by instruction issue.  One barrier a round: between barriers r and r + 1 the block threads apply
// the rotations of round r (M of round r -> M of round r + 1, other buffer) while the rotation warps, which hold the
// diagonal and the pairs' off-diagonal elements in registers, rotate the few elements that become the pairs of
// round r + 1 themselves and compute their rotations.  A round is bound by that chain (two reciprocal square roots, a
// barrier, two shared-memory reads) up to K = 64 or so, by shared-memory bandwidth above.
template <int NB, int NP, int HC>
__global__ void __launch_bounds__(PS_T, 1) k_psvd_sweeps(PsvdArgs a) {
  extern __shared__ float smf[];
  __shared__ float2 s_cs[2][JMAXK / 2];
  __shared__ int s_red[PS_T / 32];
  __shared__ float s_diag[JMAXK];
  __shared__ int s_rank[JMAXK];
  __shared__ float s_new[2][JMAXK];      // diagonal after the rotations of a round: tops, then bottoms at 64
  // Per rotation warp: a pair was rotated; at |cos| > sqrt(tol).  Two sets in turn: warps without blocks take no part in the
  // rounds and may read a sweep's set while the rotation warps are already at the end of the next sweep.
  __shared__ int s_any[2][2], s_big[2][2];
  __shared__ float s_dmax[2];
  constexpr int BW = PS_T / 32 - NP;     // block warps
  const int K = HC ? 2 * HC : a.K, h = K / 2;
  const int nblk = h * (h - 1) / 2, np = nblk + 1;
  const int rank = cl_rank(), nct = cl_size();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // two copies of M, each four planes of np values: plane x * 2 + y holds element (2 I + x, 2 J + y) of block (I, J) at the
  // block's number (consecutive threads, consecutive words); place nblk is written and read by threads without a block
  float* buf0 = smf;
  float* buf1 = smf + 4 * np;
  float2* log = reinterpret_cast<float2*>(a.ws + PS_LOGO);
  int* last_flag = reinterpret_cast<int*>(a.ws + PS_MISC + 64);   // per log region
  double* ws_scale = a.ws + PS_MISC;
  float* ws_diag = reinterpret_cast<float*>(a.ws + PS_E);         // diagonal in places (unsorted)
  // rows of W replayed by this CTA: warps (rank - 1) 16 + w of the others, or all of CTA 0 when it is alone
  const int rw0 = nct > 1 ? (rank - 1) * (PS_T / 32) + warp : warp;
  const int rstep = nct > 1 ? (nct - 1) * (PS_T / 32) : PS_T / 32;
  float* wrows = nct > 1 ? smf : smf + 2 * K * K;
  const bool replays = rank > 0 || nct == 1;
  const int lrows = PS_T / 32;   // local row q of warp w is at (q * 16 + w)
  if (replays) {
    int q = 0;
    for (int row = rw0; row < K; row += rstep, ++q)
      for (int c = lane; c < K; c += 32) wrows[(q * lrows + warp) * K + c] = c == row ? 1.f : 0.f;
    __syncwarp();
  }
  auto replay = [&](int sweep) {
    int q = 0;
    for (int row = rw0; row < K; row += rstep, ++q) {
      __syncwarp();
      replay_row<NP>(wrows + (q * lrows + warp) * K, log + (size_t)(sweep & (PS_LOG - 1)) * (K - 1) * h, h);
      __syncwarp();
    }
  };
  if (rank > 0) {
    for (int sweep = 0;; ++sweep) {
      cl_arrive();
      cl_wait();
      const int last = __ldcg(last_flag + (sweep & (PS_LOG - 1)));
      replay(sweep);
      if (last) break;
    }
  } else {
    // T scaled by a power of two to entries of at most 1, float32, in buf1 (row k, column i).  The largest exponent by
    // integer operations on the high words.
    int hi = 0;
    for (int e = tid; e < K * K; e += PS_T) {
      const int k = e / K, i = e - k * K;
      hi = max(hi, __double2hiint(a.T[(long long)k * a.ldT + i]) & 0x7FF00000);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    if (lane == 0) s_red[warp] = hi;
    __syncthreads();
    for (int w = 0; w < PS_T / 32; ++w) hi = max(hi, s_red[w]);
    // 2^-(e + 1) for the exponent e of the largest entry; 1 for zero, denormal, infinite and NaN matrices
    const int ex = hi >> 20;
    const double scale = (ex > 1 && ex < 2045) ? __hiloint2double((2045 - ex) << 20, 0) : 1.0;
    if (tid == 0) {
      ws_scale[0] = scale;
      ws_scale[1] = (ex > 1 && ex < 2045) ? __hiloint2double((ex + 1) << 20, 0) : 1.0;   // 1 / scale
    }
    for (int e = tid; e < K * K; e += PS_T) {
      const int k = e / K, i = e - k * K;
      buf1[e] = (float)(a.T[(long long)k * a.ldT + i] * scale);
    }
    __syncthreads();
    // M: blocks above the diagonal by the block threads, the diagonal blocks by the rotation warps.
    // With one rotation warp, the block warps of its scheduler (4, 8, 12) come last: with up to 384 blocks they have
    // none.  Warps without blocks wait at the end of the sweep.
    int rd[NB], wr[NB][4], bI[NB], bJ[NB];
    bool has[NB];
    const int bw = warp < NP ? -1 : (NP == 1 ? ((warp & 3) ? warp - 1 - (warp >> 2) : 11 + (warp >> 2)) : warp - NP);
    const int bwarps = min((nblk + 31) / 32, BW);   // block warps with work
    const bool rounds = bw >= 0 && bw < bwarps;
    const int rthreads = 32 * (NP + bwarps);
#pragma unroll
    for (int s = 0; s < NB; ++s) {
      const int e = bw * 32 + lane + s * BW * 32;
      has[s] = bw >= 0 && e < nblk;
      int I = 0, J = 1;
      if (has[s]) pair_block(e, h, I, J);
      bI[s] = I;
      bJ[s] = J;
      rd[s] = has[s] ? e : nblk;
#pragma unroll
      for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int y = 0; y < 2; ++y) {
          int P = next_place(2 * I + x, h), Q = next_place(2 * J + y, h);
          if ((P >> 1) > (Q >> 1)) {
            const int z = P;
            P = Q;
            Q = z;
          }
          // the off-diagonal element of a pair of the next round is computed by its rotation warp
          wr[s][x * 2 + y] = has[s] && (P >> 1) != (Q >> 1)
                                 ? ((P & 1) * 2 + (Q & 1)) * np + block_number(P >> 1, Q >> 1, h)
                                 : nblk;
        }
      if (has[s]) {
        float m00 = 0.f, m01 = 0.f, m10 = 0.f, m11 = 0.f;
        const int kend = min(K, ((2 * I + 1) / a.b + 1) * a.b);
        for (int k = 0; k < kend; ++k) {
          const float* tr = buf1 + k * K;
          const float p0 = tr[2 * I], p1 = tr[2 * I + 1], q0 = tr[2 * J], q1 = tr[2 * J + 1];
          m00 = fmaf(p0, q0, m00);
          m01 = fmaf(p0, q1, m01);
          m10 = fmaf(p1, q0, m10);
          m11 = fmaf(p1, q1, m11);
        }
        buf0[rd[s]] = m00;
        buf0[np + rd[s]] = m01;
        buf0[2 * np + rd[s]] = m10;
        buf0[3 * np + rd[s]] = m11;
      }
    }
    // rotation warps, pair i = tid: its diagonal and off-diagonal elements; where the next round's come from
    const int i = tid;
    const bool in = i < h;
    float dt = 0.f, db = 0.f, o = 0.f;
    int orow = 0, ocol = 1, oput = 0, dtop = 0, dbot = 0;
    bool obot = false, pbot = false;
    if (warp < NP) {
      if (in) {
        const int kend = min(K, ((2 * i + 1) / a.b + 1) * a.b);
        for (int k = 0; k < kend; ++k) {
          const float p0 = buf1[k * K + 2 * i], p1 = buf1[k * K + 2 * i + 1];
          dt = fmaf(p0, p0, dt);
          o = fmaf(p0, p1, o);
          db = fmaf(p1, p1, db);
        }
        // the next top comes from pair i - 1 (its top; the bottom of pair 0 for i = 1; pair 0 keeps its own), the next
        // bottom from pair i + 1 (its bottom; the last pair takes its own top)
        orow = i == 0 ? 0 : i - 1;
        pbot = i == 1;
        ocol = i == h - 1 ? h - 1 : i + 1;
        obot = i != h - 1;
        dtop = pbot ? 64 : orow;
        dbot = obot ? 64 + ocol : ocol;
        // the pair's own off-diagonal element (zero once rotated) is an element of a block of the next round
        int P = next_place(2 * i, h), Q = next_place(2 * i + 1, h);
        if ((P >> 1) > (Q >> 1)) {
          const int z = P;
          P = Q;
          Q = z;
        }
        oput = ((P & 1) * 2 + (Q & 1)) * np + block_number(P >> 1, Q >> 1, h);
      }
      const float m = warp_max(fmaxf(dt, db));
      if (lane == 0) s_dmax[warp] = m;
    }
    __syncthreads();
    const int at = block_number(orow, ocol, h);
    constexpr float kTol = 2e-6f;        // |cos| below which a pair is left alone
    auto round_sync = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(rthreads) : "memory"); };
    // one round of the block threads, from buffer PAR to the other
    auto rotate_round = [&](auto par) {
      constexpr bool PAR = decltype(par)::value;
      const float* cur = PAR ? buf1 : buf0;
      float* nxt = PAR ? buf0 : buf1;
      const float2* cs = s_cs[PAR ? 1 : 0];
      round_sync();
#pragma unroll
      for (int s = 0; s < NB; ++s) {
        const float2 cp = cs[bI[s]], cq = cs[bJ[s]];
        const float e00 = cur[rd[s]], e01 = cur[np + rd[s]], e10 = cur[2 * np + rd[s]], e11 = cur[3 * np + rd[s]];
        const float f00 = cp.x * e00 - cp.y * e10, f10 = cp.y * e00 + cp.x * e10;
        const float f01 = cp.x * e01 - cp.y * e11, f11 = cp.y * e01 + cp.x * e11;
        nxt[wr[s][0]] = cq.x * f00 - cq.y * f01;
        nxt[wr[s][1]] = cq.y * f00 + cq.x * f01;
        nxt[wr[s][2]] = cq.x * f10 - cq.y * f11;
        nxt[wr[s][3]] = cq.y * f10 + cq.x * f11;
      }
    };
    // a sweep (an odd number of rounds) that starts from buffer PAR
    auto rotate_blocks = [&](auto par) {
      constexpr bool PAR = decltype(par)::value;
      for (int round = 0; round + 1 < K - 1; round += 2) {
        rotate_round(std::integral_constant<bool, PAR>());
        rotate_round(std::integral_constant<bool, !PAR>());
      }
      rotate_round(std::integral_constant<bool, PAR>());
    };
    int sweep = 0;
    int g = 0;   // rounds so far: buffers and (c, s) alternate
    bool final_sweep = false;
    for (;;) {
      if (warp < NP) {
        // elements below the float32 rounding of M (4e-7 of its largest diagonal element) are left alone
        const float dmax = NP == 1 ? s_dmax[0] : fmaxf(s_dmax[0], s_dmax[1]);
        const float thr2 = 1.6e-13f * dmax * dmax, flr = 1e-3f * dmax;
        bool any = false, big = false;
        float2* lg = log + (size_t)(sweep & (PS_LOG - 1)) * (K - 1) * h + i;
        for (int round = 0; round < K - 1; ++round, ++g, lg += h) {
          float2* cs = s_cs[g & 1];
          float* dn = s_new[g & 1];
          // t = tan of the angle that zeroes the pair's off-diagonal element, |t| <= 1; with delta = M_qq - M_pp,
          // beta = 2 M_pq, r = sqrt(delta^2 + beta^2): c^2 = (1 + |delta| / r) / 2, s c = sign(delta) beta / (2 r)
          const float delta = db - dt, beta = o + o;
          const float y = rsqrt_ftz(fmaf(delta, delta, beta * beta));
          const float hs = copysignf(0.5f, delta) * beta * y;   // s c
          const float u = fmaf(0.5f * fabsf(delta), y, 0.5f);
          const float rc = rsqrt_ftz(u);
          const float den = fmaxf(dt, flr) * fmaxf(db, flr);
          const float g2 = o * o;
          const bool rot = g2 > thr2 && g2 > kTol * kTol * den;
          const float rr = rot ? rc : 0.f;   // (an equal pair without an off-diagonal element gives y = infinity, rc NaN)
          const float sn = rot ? hs * rr : 0.f;
          const float c = rot ? u * rr : 1.f;
          const float t = sn * rr;
          const float nt = fmaf(-t, o, dt), nb = fmaf(t, o, db);
          const float left = rot ? 0.f : o;
          any |= rot;
          big |= rot && g2 > kTol * den;
          if (in) {
            cs[i] = make_float2(c, sn);
            dn[i] = nt;
            dn[64 + i] = nb;
          }
          round_sync();
          if (in) __stcg(lg, make_float2(c, sn));
          const float* cur = (g & 1) ? buf1 : buf0;
          float* nxt = (g & 1) ? buf0 : buf1;
          const float2 cp = cs[orow], cq = cs[ocol];
          const float e00 = cur[at], e01 = cur[np + at], e10 = cur[2 * np + at], e11 = cur[3 * np + at];
          dt = dn[dtop];
          db = dn[dbot];
          if (in) nxt[oput] = left;
          const float xp = pbot ? cp.y : cp.x, yp = pbot ? cp.x : -cp.y;
          const float xq = obot ? cq.y : cq.x, yq = obot ? cq.x : -cq.y;
          o = xq * fmaf(xp, e00, yp * e10) + yq * fmaf(xp, e01, yp * e11);
          if (!in) o = 0.f;
        }
        any = __any_sync(0xffffffffu, any);
        big = __any_sync(0xffffffffu, big);
        const float m = warp_max(in ? fmaxf(dt, db) : 0.f);
        if (lane == 0) {
          s_any[sweep & 1][warp] = any;
          s_big[sweep & 1][warp] = big;
          s_dmax[warp] = m;
        }
      } else if (rounds) {
        if (g & 1) rotate_blocks(std::true_type());
        else rotate_blocks(std::false_type());
        g += K - 1;
      }
      __syncthreads();
      // quadratic convergence: a sweep whose pairs all had |cos| <= sqrt(tol) is followed by one more
      const int* sa = s_any[sweep & 1];
      const int* sb = s_big[sweep & 1];
      const bool any = sa[0] || (NP > 1 && sa[1]), big = sb[0] || (NP > 1 && sb[1]);
      const bool stop = !any || final_sweep || sweep + 1 >= min(a.max_sweeps, 16);
      final_sweep = !big;
      if (tid == 0) __stcg(last_flag + (sweep & (PS_LOG - 1)), stop ? 1 : 0);
      if (stop) break;
      // the log of this sweep is complete; the barrier of the sweep before is waited for only now, so that the
      // replay runs behind the sweeps (PS_LOG regions keep it from being overtaken)
      if (sweep > 0) cl_wait();
      cl_arrive();
      if (nct == 1) {
        __syncthreads();
        replay(sweep);
      }
      ++sweep;
    }
    // last sweep: the diagonal is back in its places
    if (warp < NP && in) {
      __stcg(ws_diag + 2 * i, dt);
      __stcg(ws_diag + 2 * i + 1, db);
    }
    if (tid == 0 && a.counters) {
      atomicAdd(&a.counters[0], 1ULL);
      atomicAdd(&a.counters[1], (unsigned long long)(sweep + 1));
    }
    if (sweep > 0) cl_wait();
    cl_arrive();
    if (nct == 1) {
      __syncthreads();
      replay(sweep);
    }
    cl_wait();
  }
  // decreasing order of the diagonal; W (column major, ordered columns) and the ordered diagonal to the workspace
  __syncthreads();
  for (int c = tid; c < K; c += PS_T) s_diag[c] = __ldcg(ws_diag + c);
  __syncthreads();
  for (int c = tid; c < K; c += PS_T) {
    // by the bits (negative numbers reversed), equal ones by their index: a permutation, also with NaNs among them
    int r = 0;
    const int d = order_bits(s_diag[c]);
    for (int c2 = 0; c2 < K; ++c2) {
      const int d2 = order_bits(s_diag[c2]);
      r += (d2 > d || (d2 == d && c2 < c)) ? 1 : 0;
    }
    s_rank[c] = r;
    if (rank == 0) a.ws[PS_DIAG + r] = (double)s_diag[c];
  }
  __syncthreads();
  if (replays) {
    float* Wf = reinterpret_cast<float*>(a.ws + PS_WF);
    int q = 0;
    for (int row = rw0; row < K; row += rstep, ++q)
      for (int c = lane; c < K; c += 32) Wf[s_rank[c] * K + row] = wrows[(q * lrows + warp) * K + c];
  }
}

// Largest of n non-negative doubles in shared memory, as its bits (float64 compares would hold the float64 pipe).
__device__ __forceinline__ long long max_bits(const double* v, int n) {
  long long m = 0;
  for (int i = 0; i < n; ++i) m = max(m, __double_as_longlong(v[i]));
  return m;
}

// ------------------------------------------------------------------------------------------------
// One-sided sweeps
// ------------------------------------------------------------------------------------------------
template <typename R>
struct Rot;

template <>
struct Rot<float> {
  static __device__ __forceinline__ void params(float al, float be, float ga, float& c, float& s, float& t) {
    const float zeta = __fdividef(be - al, 2.f * ga), az = fabsf(zeta);
    const float z2 = fmaf(zeta, zeta, 1.f);
    t = copysignf(__fdividef(1.f, az + (az < 1e12f ? z2 * rsqrtf(z2) : az)), zeta);
    c = rsqrtf(fmaf(t, t, 1.f));
    s = c * t;
  }
};

template <>
struct Rot<double> {
  // One Newton step on each float32 seed (reciprocal y <- y (2 - x y), reciprocal square root
  // y <- y (3/2 - x y^2 / 2)): relative errors ~1e-14, so c^2 + s^2 = 1 to ~1e-14.
  static __device__ __forceinline__ void params(double al, double be, double ga, double& c, double& s, double& t) {
    const double zeta = (be - al) * rcp_nr1(2.0 * ga);
    const double z2 = fma(zeta, zeta, 1.0);
    const double h = z2 * rsqrt_nr(z2, 1);                 // sqrt(1 + zeta^2)
    t = copysign(1.0, zeta) * rcp_nr1(fabs(zeta) + h);
    c = rsqrt_nr(fma(t, t, 1.0), 1);
    s = c * t;
  }
};

// Sweeps of the one-sided Jacobi method on the columns of G, in float32 on the columns of W too (both K x K, column-major
// in shared memory).  JL lanes per column pair, JR >= ceil(K / JL) rows each.  The squared column norms are formed in nrm2 at
// the start of a sweep and updated by every rotation (al' = al - t ga, be' = be + t ga with t = s / c), so a pair needs one
// inner product.  Returns the number of sweeps taken.
template <typename R, int JL, int JR>
__device__ __noinline__ int jacobi_sweeps(R* G, R* W, const unsigned char* sched, int K, double tol, int max_sweeps,
                                          int* flag, R* nrm2, R floor2) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int gl = lane & (JL - 1);                // lane inside the pair group
  const int gsub = lane / JL;                    // pair slot inside the warp
  const int npairs = K / 2;
  __shared__ float warp_max_cos[32], warp_max_t[32];   // per warp, of the pairs rotated in this sweep
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    // the norms afresh: the updates below lose the small ones
    for (int c = warp; c < K; c += nw) {
      R s2 = 0;
      for (int i = lane; i < K; i += 32) s2 = fma(G[c * K + i], G[c * K + i], s2);
      s2 = warp_sum(s2);
      if (lane == 0) nrm2[c] = s2;
    }
    if (threadIdx.x == 0) *flag = 0;
    float my_max = 0.f, my_t = 0.f;
    __syncthreads();
    for (int round = 0; round < K - 1; ++round) {
      const unsigned char* rs = sched + 2 * round * npairs;
      for (int base = warp * (32 / JL); base < npairs; base += nw * (32 / JL)) {   // warp-uniform
        const int pr = base + gsub;
        const bool has = pr < npairs;
        const int p = has ? rs[2 * pr] : 0, q = has ? rs[2 * pr + 1] : 0;
        R* gp = G + p * K;
        R* gq = G + q * K;
        R a[JR], bq[JR];
        R ga = 0;
#pragma unroll
        for (int k = 0; k < JR; ++k) {
          const int r = gl + JL * k;
          const bool in = has && r < K;
          a[k] = in ? gp[r] : (R)0;
          bq[k] = in ? gq[r] : (R)0;
        }
        // read before the shuffles, written after them by one lane of the group
        const R al = has ? nrm2[p] : (R)1, be = has ? nrm2[q] : (R)1;
#pragma unroll
        for (int k = 0; k < JR; ++k) ga += a[k] * bq[k];
#pragma unroll
        for (int o = 1; o < JL; o <<= 1) ga += __shfl_xor_sync(0xffffffffu, ga, o);
        // null columns are left alone
        if (has && ga != (R)0 && al > floor2 && be > floor2) {
          // the cosine in float32 (it is only compared; a float64 division and two square roots take 2000 cycles)
          const float cs = fabsf((float)ga) * rsqrtf((float)al) * rsqrtf((float)be);
          if (cs > (float)tol) {
            my_max = fmaxf(my_max, cs);
            R c, s, t;
            Rot<R>::params(al, be, ga, c, s, t);
            my_t = fmaxf(my_t, fabsf((float)t));
            if (gl == 0) {
              nrm2[p] = al - t * ga;
              nrm2[q] = be + t * ga;
              *flag = 1;
            }
#pragma unroll
            for (int k = 0; k < JR; ++k) {
              const int r = gl + JL * k;
              if (r < K) {
                gp[r] = c * a[k] - s * bq[k];
                gq[r] = s * a[k] + c * bq[k];
              }
            }
            if constexpr (sizeof(R) == 4) {
              R* wp = W + p * K;
              R* wq = W + q * K;
#pragma unroll
              for (int k = 0; k < JR; ++k) {
                const int r = gl + JL * k;
                if (r < K) {
                  const R x = wp[r], y = wq[r];
                  wp[r] = c * x - s * y;
                  wq[r] = s * x + c * y;
                }
              }
            }
          }
        }
      }
      __syncthreads();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      my_max = fmaxf(my_max, __shfl_xor_sync(0xffffffffu, my_max, o));
      my_t = fmaxf(my_t, __shfl_xor_sync(0xffffffffu, my_t, o));
    }
    if (lane == 0) {
      warp_max_cos[warp] = my_max;
      warp_max_t[warp] = my_t;
    }
    __syncthreads();
    float sweep_max = 0.f, t_max = 0.f;
    for (int w = 0; w < nw; ++w) {
      sweep_max = fmaxf(sweep_max, warp_max_cos[w]);
      t_max = fmaxf(t_max, warp_max_t[w]);
    }
    // quadratic convergence: a sweep leaves cosines of the size of its angles times its cosines
    if (!*flag || (double)sweep_max * (double)t_max <= tol) break;
    __syncthreads();
  }
  return sweep + 1;
}

// Squared ratio to the largest value below which one is null: 1e-13, the rounding of G; 2^-20 where T holds the rounding of
// float32 products.
__device__ __forceinline__ double psvd_null2(const PsvdArgs& a) { return a.f32 ? 0x1p-40 : 1e-26; }

// Round-robin tournament: in round r, pair 0 is (K-1, r) and pair i >= 1 is
// ((r + i) mod (K-1), (r - i) mod (K-1)); every pair of columns meets once per sweep.
__device__ void build_schedule(unsigned char* sched, int K) {
  const int npairs = K / 2;
  for (int e = threadIdx.x; e < (K - 1) * npairs; e += blockDim.x) {
    const int round = e / npairs, i = e - round * npairs;
    int p, q;
    if (i == 0) { p = K - 1; q = round; }
    else { p = (round + i) % (K - 1); q = (round - i + (K - 1)) % (K - 1); }
    if (p > q) { int x = p; p = q; q = x; }
    sched[2 * e] = (unsigned char)p;
    sched[2 * e + 1] = (unsigned char)q;
  }
}

// The leading values of a graded T span more than M = T^T T resolves in float32 (values below 6e-4 of the largest are mixed):
// float32 one-sided sweeps on the columns of G = scale T W (workspace), which see 1e-7 of the largest, rotate W on.
// Everything in CTA 0; the columns of W32 in decreasing order of their values, and their squares, back to the workspace.  smem:
// K x K doubles; tmp as for psvd_onesided.
__device__ __noinline__ void psvd_graded_sweeps(const PsvdArgs& a, float floor2, double* smem, double* tmp) {
  __shared__ int flag;
  const int K = a.K, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = PS_T / 32;
  float* Wf = reinterpret_cast<float*>(a.ws + PS_WF);
  float* sG = reinterpret_cast<float*>(smem);
  float* sW = sG + K * K;
  float* nrm = reinterpret_cast<float*>(tmp);
  int* place = reinterpret_cast<int*>(nrm + K);
  unsigned char* sched = reinterpret_cast<unsigned char*>(place + K);
  build_schedule(sched, K);
  for (int e = tid; e < K * K; e += PS_T) {
    sG[e] = (float)__ldcg(a.ws + PS_G + e);
    sW[e] = __ldcg(Wf + e);
  }
  __syncthreads();
  const int sweeps = K <= 48 ? jacobi_sweeps<float, 16, 3>(sG, sW, sched, K, 2e-6, 16, &flag, nrm, floor2)
                             : jacobi_sweeps<float, 8, 16>(sG, sW, sched, K, 2e-6, 16, &flag, nrm, floor2);
  if (tid == 0 && a.counters) atomicAdd(&a.counters[1], (unsigned long long)sweeps);
  __syncthreads();
  for (int c = warp; c < K; c += nw) {
    float s2 = 0.f;
    for (int i = lane; i < K; i += 32) s2 = fmaf(sG[c * K + i], sG[c * K + i], s2);
    s2 = warp_sum(s2);
    if (lane == 0) nrm[c] = s2;
  }
  __syncthreads();
  for (int c = tid; c < K; c += PS_T) {
    int r = 0;
    const int d = order_bits(nrm[c]);
    for (int q = 0; q < K; ++q) {
      const int dq = order_bits(nrm[q]);
      r += (dq > d || (dq == d && q < c)) ? 1 : 0;
    }
    place[c] = r;
    __stcg(a.ws + PS_DIAG + r, (double)nrm[c]);
  }
  __syncthreads();
  for (int e = tid; e < K * K; e += PS_T) __stcg(Wf + place[e / K] * K + e % K, sW[e]);
}

// One-sided Jacobi finish in CTA 0: float64 sweeps on G = scale T W (workspace), tracked column norms, then
// theta = ||g|| / scale, x = g / ||g||, and the right vectors of the leading nv triplets w = T^T x / theta.
// sG: K x K; tmp: 16 K doubles and more (norms, order and the tournament, 2 (K - 1) K / 2 bytes).
__device__ __noinline__ void psvd_onesided(const PsvdArgs& a, double scale, double* sG, double* tmp) {
  __shared__ int flag;
  const int K = a.K, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = PS_T / 32;
  double* nrm = tmp;
  double* rnrm = nrm + K;
  int* order = reinterpret_cast<int*>(rnrm + K);
  unsigned char* sched = reinterpret_cast<unsigned char*>(order + K);
  build_schedule(sched, K);
  for (int e = tid; e < K * K; e += PS_T) sG[e] = __ldcg(a.ws + PS_G + e);
  __syncthreads();
  for (int c = warp; c < K; c += nw) {
    double s2 = 0.0;
    for (int i = lane; i < K; i += 32) s2 = fma(sG[c * K + i], sG[c * K + i], s2);
    s2 = warp_sum(s2);
    if (lane == 0) nrm[c] = s2;
  }
  __syncthreads();
  const double floor2 = psvd_null2(a) * __longlong_as_double(max_bits(nrm, K));
  const int sweeps = K <= 48 ? jacobi_sweeps<double, 8, 6>(sG, nullptr, sched, K, a.tol, a.max_sweeps, &flag, nrm, floor2)
                             : jacobi_sweeps<double, 8, 16>(sG, nullptr, sched, K, a.tol, a.max_sweeps, &flag, nrm, floor2);
  if (tid == 0) {
    if (sweeps > a.max_sweeps) svt_set_error(a.err, SVT_DEVERR_JACOBI);
    if (a.counters) atomicAdd(&a.counters[1], (unsigned long long)sweeps);
  }
  for (int c = warp; c < K; c += nw) {
    double s2 = 0.0;
    for (int i = lane; i < K; i += 32) s2 = fma(sG[c * K + i], sG[c * K + i], s2);
    s2 = warp_sum(s2);
    if (lane == 0) {
      // Null columns hold no direction: x would repeat another one and T^T x / theta be of any size.  Their triplet is
      // (0, 0, 0).
      const bool null = s2 <= floor2;
      const double th = null ? 0.0 : s2 * rsqrt_nr(s2, 2);
      nrm[c] = th;
      rnrm[c] = null ? 0.0 : rcp_nr(th);
    }
  }
  __syncthreads();
  for (int c = tid; c < K; c += PS_T) {
    // by the bits of the magnitude, equal ones by their index: a permutation (order[] is an index), also with NaNs
    int r = 0;
    const long long nc = __double_as_longlong(fabs(nrm[c]));
    for (int q = 0; q < K; ++q) {
      const long long nq = __double_as_longlong(fabs(nrm[q]));
      r += (nq > nc || (nq == nc && q < c)) ? 1 : 0;
    }
    order[r] = c;
  }
  __syncthreads();
  for (int e = tid; e < K * K; e += PS_T) {
    const int i = e / K, k = e - i * K;
    const int c = order[k];
    a.Xl[i * K + k] = sG[c * K + i] * rnrm[c];
    // column i of T has no entries below its diagonal block
    double v = 0.0;
    if (k < a.nv) {
      const double* gc = sG + c * K;
      const int rend = min(K, (i / a.b + 1) * a.b);
      double s0 = 0.0, s1 = 0.0;
      for (int r = 0; r + 1 < rend; r += 2) {
        s0 = fma(a.T[(long long)r * a.ldT + i], gc[r], s0);
        s1 = fma(a.T[(long long)(r + 1) * a.ldT + i], gc[r + 1], s1);
      }
      v = (s0 + s1) * scale * (rnrm[c] * rnrm[c]);
    }
    a.Wr[i * K + k] = v;
  }
  for (int k = warp; k < K; k += nw) {
    const int c = order[k];
    double r2 = 0.0;
    if (a.S) {
      for (int e = lane; e < a.b; e += 32) {
        double v = 0.0;
        for (int d = e; d < a.b; ++d) v = fma(a.S[e * a.b + d], sG[c * K + (K - a.b + d)], v);
        v *= rnrm[c];
        r2 = fma(v, v, r2);
      }
      r2 = warp_sum(r2);
    }
    if (lane == 0) {
      a.theta[k] = nrm[c] * a.ws[PS_MISC + 1];
      a.res[k] = sqrt(r2);
    }
  }
}

// ------------------------------------------------------------------------------------------------
// 2. float64 refinement of the leading nv triplets
// ------------------------------------------------------------------------------------------------
// Folded upper triangle (i <= j) of a K x K matrix, K even: entry t of K / 2 (K + 1).
__device__ __forceinline__ void folded_ij(int t, int K, int& i, int& j) {
  const int r = t / (K + 1), q = t - r * (K + 1);
  if (q < K - r) {
    i = r;
    j = r + q;
  } else {
    i = K - 1 - r;
    j = q - 1;
  }
}

// The columns c = rank, rank + nct, ... < ncol of G = scale T W (into the workspace), lambda = ||g||^2 and, when want_z, of
// Z = scale T^T G.  Four columns at a time: eight lanes share a row of T for G, row slices of the CTA a column of T for Z.
// Ts, ldT: T, in shared memory or global.
__device__ void psvd_gz(const PsvdArgs& a, const double* __restrict__ Ts, int ldT, const double* __restrict__ Wg, int ncol,
                        double scale, bool want_z, int rank, int nct, double* sw, double* sg, double* part) {
  const int K = a.K, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int Kp = (K + 31) & ~31, nsl = PS_T / Kp;
  double* lam = a.ws + PS_LAM;
  double* Gg = a.ws + PS_G;
  double* Zg = a.ws + PS_Z;
  for (int c0 = rank; c0 < ncol; c0 += 4 * nct) {
    const int nc = min(4, (ncol - c0 + nct - 1) / nct);
    __syncthreads();
    for (int e = tid; e < nc * K; e += PS_T) sw[e] = scale * __ldcg(Wg + (long long)(c0 + (e / K) * nct) * K + e % K);
    __syncthreads();
    for (int i0 = warp * 4; i0 < K; i0 += PS_T / 8) {
      const int i = i0 + (lane >> 3), l = lane & 7;
      double s[4] = {0.0, 0.0, 0.0, 0.0};
      if (i < K) {
        const double* tr = Ts + i * ldT;
#pragma unroll 2
        for (int k = (i / a.b) * a.b + l; k < K; k += 8) {
          const double tv = tr[k];
#pragma unroll
          for (int t = 0; t < 4; ++t)
            if (t < nc) s[t] = fma(tv, sw[t * K + k], s[t]);
        }
      }
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (t < nc)
          for (int o = 4; o > 0; o >>= 1) s[t] += __shfl_xor_sync(0xffffffffu, s[t], o);
      if (l == 0 && i < K)
        for (int t = 0; t < nc; ++t) {
          sg[t * K + i] = s[t];
          __stcg(Gg + (long long)(c0 + t * nct) * K + i, s[t]);
        }
    }
    __syncthreads();
    if (warp < nc) {
      double s2 = 0.0;
      for (int i = lane; i < K; i += 32) s2 = fma(sg[warp * K + i], sg[warp * K + i], s2);
      s2 = warp_sum(s2);
      if (lane == 0 && c0 + warp * nct < a.nv) __stcg(lam + c0 + warp * nct, s2);
    }
    if (!want_z) continue;
    const int sl = tid / Kp, j = tid - sl * Kp;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    if (sl < nsl && j < K) {
      const int rend = min(K, (j / a.b + 1) * a.b);
#pragma unroll 2
      for (int i = sl; i < rend; i += nsl) {
        const double tv = Ts[i * ldT + j];
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (t < nc) s[t] = fma(tv, sg[t * K + i], s[t]);
      }
      for (int t = 0; t < nc; ++t) part[(sl * 4 + t) * Kp + j] = s[t];
    }
    __syncthreads();
    for (int e = tid; e < nc * K; e += PS_T) {
      const int t = e / K, jj = e - t * K;
      double v = 0.0;
      for (int q = 0; q < nsl; ++q) v += part[(q * 4 + t) * Kp + jj];
      __stcg(Zg + (long long)(c0 + t * nct) * K + jj, scale * v);
    }
  }
  __syncthreads();
}

// W <- W (I - E / 2), E = W^T W - I, in float64 (columns of the CTA; Wout may not be Win).  Called by all CTAs.
__device__ void psvd_orth64(const PsvdArgs& a, const double* Win, double* Wout, int rank, int nct, double* sA) {
  const int K = a.K, tid = threadIdx.x, ld = K + 1;
  double* Eg = a.ws + PS_E;
  for (int e = tid; e < K * K; e += PS_T) sA[(e / K) * ld + e % K] = __ldcg(Win + e);
  __syncthreads();
  for (int t = rank * PS_T + tid; t < K / 2 * (K + 1); t += nct * PS_T) {
    int p, q;
    folded_ij(t, K, p, q);
    double s0 = 0.0, s1 = 0.0;
    for (int i = 0; i < K; i += 2) {
      s0 = fma(sA[p * ld + i], sA[q * ld + i], s0);
      s1 = fma(sA[p * ld + i + 1], sA[q * ld + i + 1], s1);
    }
    const double v = (s0 + s1) - (p == q ? 1.0 : 0.0);
    __stcg(Eg + p * K + q, v);
    __stcg(Eg + q * K + p, v);
  }
  cl_sync();
  for (int t = tid; t < ((K - rank + nct - 1) / nct) * K; t += PS_T) {
    const int c = rank + (t / K) * nct, i = t % K;
    double s0 = 0.0, s1 = 0.0;
    for (int p = 0; p < K; p += 2) {
      s0 = fma(sA[p * ld + i], __ldcg(Eg + c * K + p), s0);
      s1 = fma(sA[(p + 1) * ld + i], __ldcg(Eg + c * K + p + 1), s1);
    }
    __stcg(Wout + c * K + i, sA[c * ld + i] - 0.5 * (s0 + s1));
  }
  cl_sync();
}

// W0 <- W32 (I - E / 2 + 3 E^2 / 8), E = W32^T W32 - I: the rotations of the sweeps back to orthonormality up to O(|E|^3),
// |E| ~ 1e-5.  The entries of W32 are exact float32, so E comes from compensated float32 inner products (two-product,
// two-sum: ~2^-45) and the small correction from float32 ones.  Called by all CTAs; ends with a cluster barrier.
// sA: K (K + 4) doubles.
__device__ __noinline__ void psvd_start(const PsvdArgs& a, double* W0, int rank, int nct, double* sA) {
  const int K = a.K, tid = threadIdx.x;
  const float* Wf = reinterpret_cast<const float*>(a.ws + PS_WF);
  float* Eg = reinterpret_cast<float*>(a.ws + PS_E);
  const int ld = K + 1;
  float* sWf = reinterpret_cast<float*>(sA);
  float* sE = sWf + K * ld;
  float* sF = sE + K * ld;   // columns in hand, Kp apart
  for (int e = tid; e < K * K; e += PS_T) sWf[(e / K) * ld + e % K] = __ldcg(Wf + e);
  __syncthreads();
  for (int t = rank * PS_T + tid; t < K / 2 * (K + 1); t += nct * PS_T) {
    int p, q;
    folded_ij(t, K, p, q);
    float s = 0.f, c = 0.f;
#pragma unroll 8
    for (int i = 0; i < K; ++i) {
      const float x = sWf[p * ld + i], y = sWf[q * ld + i];
      const float pr = __fmul_rn(x, y), er = fmaf(x, y, -pr);
      const float s2 = __fadd_rn(s, pr), bb = __fsub_rn(s2, s);
      c = __fadd_rn(c, __fadd_rn(er, __fadd_rn(__fsub_rn(s, __fsub_rn(s2, bb)), __fsub_rn(pr, bb))));
      s = s2;
    }
    const float v = __fadd_rn(__fsub_rn(s, p == q ? 1.f : 0.f), c);
    __stcg(Eg + p * K + q, v);
    __stcg(Eg + q * K + p, v);
  }
  cl_sync();
  for (int e = tid; e < K * K; e += PS_T) sE[(e / K) * ld + e % K] = __ldcg(Eg + e);
  const int Kp = (K + 31) & ~31, NC = PS_T / Kp;
  const int u = tid / Kp, i = tid - u * Kp;
  for (int c0 = rank; c0 < K; c0 += NC * nct) {
    const int c = c0 + u * nct;
    const bool in = u < NC && c < K && i < K;
    __syncthreads();
    float f = 0.f;
    if (in) {
#pragma unroll 8
      for (int p = 0; p < K; ++p) f = fmaf(sE[p * ld + i], sE[c * ld + p], f);
      f = 0.375f * f - 0.5f * sE[c * ld + i];
      sF[tid] = f;
    }
    __syncthreads();
    if (in) {
      float s0 = 0.f;
#pragma unroll 8
      for (int p = 0; p < K; ++p) s0 = fmaf(sWf[p * ld + i], sF[u * Kp + p], s0);
      __stcg(W0 + c * K + i, (double)sWf[c * ld + i] + (double)s0);
    }
  }
  cl_sync();
}

// Jacobi angle of the pair: tan(2 angle) = 2 S / d, |angle| <= pi / 4.  In float32: a relative error of 1e-7 of an
// angle is far below the second-order error of the step it is used in.
__device__ __forceinline__ float jacobi_angle(float S, float d) {
  const float q = __fdividef(S, d), q2 = q * q;
  // atan(2 q) / 2 = q - 4/3 q^3 + 16/5 q^5 - ...
  if (q2 < 4e-4f) return q * fmaf(q2, fmaf(q2, 3.2f, -4.f / 3.f), 1.f);
  return d == 0.f ? copysignf(0.785398163f, S) : 0.5f * atanf(2.f * q);
}

// sA: K (K + 4) doubles, used in turn as W32, Z, Theta (float32), G of the fallback; sw, sg: 16 K; part: 2048 doubles.
__global__ void __launch_bounds__(PS_T, 1) k_psvd_refine(PsvdArgs a) {
  extern __shared__ double smr[];
  __shared__ float s_st[3][PS_T / 32];
  __shared__ double s_lam[JMAXK];
  __shared__ int s_rank[JMAXK];
  const int K = a.K, nv = a.nv;
  double* sA = smr;
  double* sw = sA + K * (K + 4);
  double* sg = sw + 16 * K;
  double* part = sg + 16 * K;
  double* sS = part + 2048;                       // S, b x b
  double* sT = sS + 1024;                         // T where it fits
  const bool t_in_smem = K <= kTinSmem;
  const double* Ts = t_in_smem ? sT : a.T;
  const int ldT = t_in_smem ? K + 1 : a.ldT;
  const int rank = cl_rank(), nct = cl_size();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* W0 = a.ws + PS_W0;
  double* W1 = a.ws + PS_W1;
  float* Thg = reinterpret_cast<float*>(a.ws + PS_TH);
  double* lam = a.ws + PS_LAM;
  float* stat = reinterpret_cast<float*>(a.ws + PS_MISC + 2);   // three per CTA
  const double scale = a.ws[PS_MISC], unscale = a.ws[PS_MISC + 1];
  const bool strict = a.tol < 1e-11;
  for (int e = rank * PS_T + tid; e < K * K; e += nct * PS_T) Thg[e] = 0.f;
  if (t_in_smem)
    for (int e = tid; e < K * K; e += PS_T) sT[(e / K) * ldT + e % K] = a.T[(long long)(e / K) * a.ldT + e % K];
  if (a.S)
    for (int e = tid; e < a.b * a.b; e += PS_T) sS[e] = a.S[e];
  psvd_start(a, W0, rank, nct, sA);
  auto load_lambda = [&]() {
    for (int i = tid; i < nv; i += PS_T) s_lam[i] = __ldcg(lam + i);
    __syncthreads();
  };
  auto lambda_min = [&]() {   // NaN bits order above everything
    long long m = __double_as_longlong(s_lam[0]);
    for (int i = 1; i < nv; ++i) m = min(m, __double_as_longlong(s_lam[i]));
    return __longlong_as_double(m);
  };
  // Leading values that span more than a factor 100 (the sweeps' diagonal is good to 1e-6 of its largest).  The rotations are
  // carried on where the sweeps above have not resolved a cluster of small values; null values need none.  Then float64
  // contexts and null values take the one-sided finish, float32 contexts a step of the refinement: cosines of 1e-6 or, for
  // values below 3e-5 sigma_1, 1e-15 (sigma_1 / theta)^2.
  // Measured (us a projected SVD, fully observed 300 x 300 rank 5 and 400 x 390 rank 30; the finish alone -> now): K = 48, noise
  // 1e-3, float64 1660 -> 528, float32 1617 -> 238; K = 128, noise 1e-4, float64 7878 -> 2830, float32 8633 -> 1953; no noise
  // (null values), float64 283 -> 187, float32 1504 -> 137.
  double tol = a.tol;
  if (__ldcg(a.ws + PS_DIAG + nv - 1) < 0.9e-4 * __ldcg(a.ws + PS_DIAG)) {
    psvd_gz(a, Ts, ldT, W0, K, scale, false, rank, nct, sw, sg, part);
    cl_sync();
    load_lambda();
    const double top = __longlong_as_double(max_bits(s_lam, nv)), floor2 = psvd_null2(a) * top;
    bool null = false, some = false;   // null values; others that the sweeps may not have resolved
    for (int i = 0; i < nv; ++i) {
      null |= s_lam[i] <= floor2;
      some |= s_lam[i] > floor2 && s_lam[i] < 1e-4 * top;
    }
    if (some) {
      if (rank == 0) psvd_graded_sweeps(a, (float)floor2, sA, sw);
      cl_sync();
      psvd_start(a, W0, rank, nct, sA);
      null = __ldcg(a.ws + PS_DIAG + nv - 1) <= floor2;
      if (null || !a.f32) {
        psvd_gz(a, Ts, ldT, W0, K, scale, false, rank, nct, sw, sg, part);
        cl_sync();
      }
    }
    if (null || !a.f32) {
      if (rank == 0) psvd_onesided(a, scale, sA, sw);
      return;
    }
    tol = fmax(tol, 1e-6);
  }
  const double* Wtop = W0;   // where the final leading columns are
  bool converged = false;
  float th_prev = 0.f;
  int it = 0;
  for (; it < 6; ++it) {
    // a step leaves W orthonormal to 1e-7 of its angles squared; large angles (nearly equal values) to less
    for (int p = 0; it > 0 && p < (th_prev > 1e-2f ? 2 : (strict || th_prev > 2e-3f ? 1 : 0)); ++p) {
      psvd_orth64(a, W0, W1, rank, nct, sA);
      double* x = W0;
      W0 = W1;
      W1 = x;
    }
    Wtop = W0;
    psvd_gz(a, Ts, ldT, W0, nv, scale, true, rank, nct, sw, sg, part);
    cl_sync();
    // S, Theta: rows j = rank, rank + nct, ... of W, 16 at a time; four lanes per entry
    const int ldz = K + 4;
    for (int e = tid; e < nv * K; e += PS_T) sA[(e / K) * ldz + e % K] = __ldcg(a.ws + PS_Z + e);
    for (int i = tid; i < K; i += PS_T) s_lam[i] = i < nv ? __ldcg(lam + i) : __ldcg(a.ws + PS_DIAG + i);
    __syncthreads();
    // rounding of S, from the largest lambda (non-negative doubles compare like their bits)
    const float noise = 8.9e-16f * (float)__longlong_as_double(max_bits(s_lam, nv));
    float cmax = 0.f, tmax = 0.f, tsum = 0.f;   // largest cosine and angle, sum of the squared angles
    for (int j0 = rank; j0 < K; j0 += 16 * nct) {
      const int nj = min(16, (K - j0 + nct - 1) / nct);
      __syncthreads();
      for (int e = tid; e < nj * K; e += PS_T) sw[e] = __ldcg(W0 + (long long)(j0 + (e / K) * nct) * K + e % K);
      __syncthreads();
      for (int base = warp * 8; base < nj * nv; base += PS_T / 4) {   // warp-uniform
        const int e = base + (lane >> 2), l = lane & 3;
        const int t = e / nv, i = e - t * nv, j = j0 + t * nct;
        const bool live = e < nj * nv && i != j && (j >= nv || i < j);
        double s = 0.0;
        if (live)
          for (int k = l; k < K; k += 4) s = fma(sw[t * K + k], sA[i * ldz + k], s);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (live && l == 0) {
          const double li = s_lam[i], lj = s_lam[j];
          float th = 0.f;
          const float f = (float)s, fs = fabsf(f);
          if (!(fs <= noise)) {
            // against another kept column the angle between x_i and x_j; against the rest the share of w_j in w_i
            const float c = j < nv ? fs * rsqrtf((float)li) * rsqrtf((float)lj) : __fdividef(fs, (float)li);
            cmax = fmaxf(cmax, isnan(c) ? INFINITY : c);
            th = jacobi_angle(f, (float)(li - lj));
            tmax = fmaxf(tmax, fabsf(th));
            tsum = fmaf(2.f * th, th, tsum);
          }
          __stcg(Thg + (long long)i * K + j, th);
          __stcg(Thg + (long long)j * K + i, -th);
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      cmax = fmaxf(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
      tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
      tsum += __shfl_xor_sync(0xffffffffu, tsum, o);
    }
    if (lane == 0) {
      s_st[0][warp] = cmax;
      s_st[1][warp] = tmax;
      s_st[2][warp] = tsum;
    }
    __syncthreads();
    if (tid == 0) {
      for (int w = 1; w < PS_T / 32; ++w) {
        cmax = fmaxf(cmax, s_st[0][w]);
        tmax = fmaxf(tmax, s_st[1][w]);
        tsum += s_st[2][w];
      }
      __stcg(stat + 3 * rank, cmax);
      __stcg(stat + 3 * rank + 1, tmax);
      __stcg(stat + 3 * rank + 2, tsum);
    }
    cl_sync();
    cmax = tmax = tsum = 0.f;
    for (int q = 0; q < nct; ++q) {
      cmax = fmaxf(cmax, __ldcg(stat + 3 * q));
      tmax = fmaxf(tmax, __ldcg(stat + 3 * q + 1));
      tsum += __ldcg(stat + 3 * q + 2);
    }
    th_prev = tmax;
    if ((double)cmax <= tol) {   // the columns at hand are final
      converged = true;
      break;
    }
    // clusters of nearly equal values whose columns the sweeps have mixed ask for large rotations among all of them:
    // the one-sided sweeps do that (a single pair, |Theta|_F <= 1.11, stays here); so do NaNs, to be reported
    if (!(tsum <= 2.25f) || isinf(cmax)) break;
    // the step leaves errors of the size angle x cosine; the last step needs the leading columns only
    const bool last = 4.0 * (double)tmax * (double)cmax <= tol && tmax < 5e-3f;
    // W exp(Theta): the columns of Phi = Theta + Theta^2 / 2 + ..., as many powers as the angles ask for, in float32;
    // NC = 512 / Kp columns at a time, thread (t, j) entry j of column t.  The last step's W Phi (angles below 1e-5) is
    // added up in float32 as well, from float32 copies of W.
    float* sTh = reinterpret_cast<float*>(sA);
    float* sWs = sTh + K * (K + 1);
    float* v0 = reinterpret_cast<float*>(part);
    const bool small = last && tmax < 1e-5f;
    __syncthreads();
    for (int e = tid; e < K * K; e += PS_T) {
      sTh[(e / K) * (K + 1) + e % K] = __ldcg(Thg + e);
      if (small) sWs[e] = (float)__ldcg(W0 + e);
    }
    const int ncol = last ? nv : K;
    const int Kp = (K + 31) & ~31, NC = min(PS_T / Kp, 8);
    const int t = tid / Kp, j = tid - t * Kp;
    // the remainder |Theta|^(p + 1) / (p + 1)! is at most 3e-12 (|Theta|_F <= 1.5), 2e-11, 1e-12 and 5e-12; what it and the
    // float32 powers leave of orthonormality is taken out before the next step for angles above 2e-3
    const int powers = tsum > 1e-2f ? 16 : (tsum > 1e-4f ? 6 : (tsum > 1e-7f ? 4 : 2));
    for (int c0 = rank; c0 < ncol; c0 += NC * nct) {
      const int nc = min(NC, (ncol - c0 + nct - 1) / nct);
      __syncthreads();
      const bool in = t < nc && j < K;
      const int c = c0 + t * nct;
      float v = in ? sTh[c * (K + 1) + j] : 0.f;
      const float theta = v;
      float add = 0.f, fact = 1.f;
      for (int p = 2; p <= powers; ++p) {
        float* vb = v0 + (p & 1) * PS_T;
        vb[tid] = v;
        __syncthreads();
        v = 0.f;
        if (in) {
#pragma unroll 8
          for (int k = 0; k < K; ++k) v = fmaf(sTh[k * (K + 1) + j], vb[t * Kp + k], v);
        }
        fact /= (float)p;
        add = fmaf(fact, v, add);
      }
      __syncthreads();
      if (small) {
        v0[tid] = theta + add;
        __syncthreads();
        if (in) {
          float s0 = 0.f;
#pragma unroll 8
          for (int q = 0; q < K; ++q) s0 = fmaf(sWs[q * K + j], v0[t * Kp + q], s0);
          const long long at = (long long)c * K + j;
          __stcg(W1 + at, __ldcg(W0 + at) + (double)s0);
        }
        continue;
      }
      if (in) sg[t * K + j] = (double)theta + (double)add;
      __syncthreads();
      // slice t of the columns of W, row j, all nc columns of Phi
      double s[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
      if (t < NC && j < K) {
#pragma unroll 4
        for (int q = t; q < K; q += NC) {
          const double wv = __ldcg(W0 + (long long)q * K + j);
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (u < nc) s[u] = fma(wv, sg[u * K + q], s[u]);
        }
      }
      for (int u0 = 0; u0 < nc; u0 += 4) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (t < NC) part[(t * 4 + u) * Kp + j] = u0 == 0 ? s[u] : s[u + 4];
        __syncthreads();
        const int nu = min(4, nc - u0);
        for (int e = tid; e < nu * K; e += PS_T) {
          const int u = e / K, ii = e - u * K;
          double x = 0.0;
          for (int q = 0; q < NC; ++q) x += part[(q * 4 + u) * Kp + ii];
          const long long at = (long long)(c0 + (u0 + u) * nct) * K + ii;
          __stcg(W1 + at, __ldcg(W0 + at) + x);
        }
      }
    }
    __syncthreads();
    if (last) {
      Wtop = W1;
      psvd_gz(a, Ts, ldT, W1, nv, scale, false, rank, nct, sw, sg, part);
      converged = true;
      ++it;
      break;
    }
    cl_sync();
    double* x = W0;
    W0 = W1;
    W1 = x;
  }
  if (rank == 0 && tid == 0 && a.counters) atomicAdd(&a.counters[1], (unsigned long long)it);
  cl_sync();
  load_lambda();
  if (!converged || lambda_min() < (a.f32 ? psvd_null2(a) : 1e-4) * __longlong_as_double(max_bits(s_lam, nv))) {
    // one-sided sweeps on G = T W from the rotations of the float32 sweeps
    psvd_start(a, W0, rank, nct, sA);
    psvd_gz(a, Ts, ldT, W0, K, scale, false, rank, nct, sw, sg, part);
    cl_sync();
    if (rank == 0) psvd_onesided(a, scale, sA, sw);
    return;
  }
  for (int i = tid; i < nv; i += PS_T) {
    // decreasing order (NaN bits order above everything, equal values by index: always a permutation)
    int r = 0;
    const long long li = __double_as_longlong(fabs(s_lam[i]));
    for (int q = 0; q < nv; ++q) {
      const long long lq = __double_as_longlong(fabs(s_lam[q]));
      r += (lq > li || (lq == li && q < i)) ? 1 : 0;
    }
    s_rank[i] = r;
  }
  __syncthreads();
  // one warp per triplet
  for (int c = rank + nct * warp; c < nv; c += nct * (PS_T / 32)) {
    const double s2 = s_lam[c];
    const double th = s2 > 0.0 ? s2 * rsqrt_nr(s2, 2) : s2;   // NaN stays NaN
    const double inv = th > 0.0 ? rcp_nr(th) : 0.0;
    const int k = s_rank[c];
    const double* gc = a.ws + PS_G + (long long)c * K;
    for (int i = lane; i < K; i += 32) {
      a.Xl[i * K + k] = __ldcg(gc + i) * inv;
      a.Wr[i * K + k] = __ldcg(Wtop + (long long)c * K + i);
    }
    double r2 = 0.0;
    if (a.S) {
      if (lane < a.b) sw[warp * a.b + lane] = __ldcg(gc + (K - a.b + lane));
      __syncwarp();
      for (int e = lane; e < a.b; e += 32) {
        double v = 0.0;
        for (int d = e; d < a.b; ++d) v = fma(sS[e * a.b + d], sw[warp * a.b + d], v);
        v *= inv;
        r2 = fma(v, v, r2);
      }
      r2 = warp_sum(r2);
    }
    if (lane == 0) {
      a.theta[k] = th * unscale;
      a.res[k] = sqrt(r2);
    }
  }
  // the other triplets (not used by the rank policy, the restart or the shrink): values from the sweeps, no vectors
  for (int k = nv + rank * PS_T + tid; k < K; k += nct * PS_T) {
    a.theta[k] = sqrt(fmax(__ldcg(a.ws + PS_DIAG + k), 0.0)) * unscale;
    a.res[k] = INFINITY;
  }
  for (int e = rank * PS_T + tid; e < K * (K - nv); e += nct * PS_T) {
    const int i = e / (K - nv), k = nv + e - i * (K - nv);
    a.Xl[i * K + k] = 0.0;
    a.Wr[i * K + k] = 0.0;
  }
}
// Self-test of the Newton reciprocal / reciprocal-square-root helpers: out[5 i + 0..3] =
// rcp_nr(x_i), rcp_nr1(x_i), rsqrt_nr(x_i, 2), rsqrt_nr(x_i, 1) (slot 4 is the orthonormalisation's
// pivot helper, filled by launch_pivot_selftest).
__global__ void k_newton_selftest(const double* __restrict__ x, long long n, double* __restrict__ out) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double v = x[i];
    out[5 * i + 0] = rcp_nr(v);
    out[5 * i + 1] = rcp_nr1(v);
    out[5 * i + 2] = rsqrt_nr(v, 2);
    out[5 * i + 3] = rsqrt_nr(v, 1);
  }
}

int launch_newton_selftest(const double* x, long long n, double* out, cudaStream_t st) {
  if (n <= 0) return 0;
  const int blocks = (int)svt_min_ll(svt_ceil_div(n, 256), 152LL * 4);
  k_newton_selftest<<<blocks, 256, 0, st>>>(x, n, out);
  return 1;
}

// ------------------------------------------------------------------------------------------------
// Launch
// ------------------------------------------------------------------------------------------------
static size_t psvd_sweeps_smem(int K, int nct) { return (size_t)(2 + (nct == 1 ? 1 : 0)) * K * K * sizeof(float); }
static size_t psvd_refine_smem(int K) {
  return (size_t)(K * (K + 4) + 32 * K + 2048 + 1024 + (K <= kTinSmem ? K * (K + 1) : 0)) * sizeof(double);
}

// The sweeps of a K x K problem: one kernel for each count of blocks per thread, and for K = 48, 72, 96, 128 (three
// blocks of 16, 24, 32 columns; four of 32) one with K at compile time.
static void (*psvd_sweeps_kernel(int K))(PsvdArgs) {
  if (K == 48) return k_psvd_sweeps<1, 1, 24>;
  if (K == 72) return k_psvd_sweeps<2, 2, 36>;
  if (K == 96) return k_psvd_sweeps<3, 2, 48>;
  if (K == 128) return k_psvd_sweeps<5, 2, 64>;
  const int h = K / 2, nblk = h * (h - 1) / 2;
  if (h <= 32) return nblk <= 480 ? k_psvd_sweeps<1, 1, 0> : k_psvd_sweeps<2, 1, 0>;
  if (nblk <= 2 * 448) return k_psvd_sweeps<2, 2, 0>;
  if (nblk <= 3 * 448) return k_psvd_sweeps<3, 2, 0>;
  return k_psvd_sweeps<5, 2, 0>;
}

template <typename Kernel>
static bool psvd_attr(Kernel* k, size_t smem) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess;
}

// CTAs of the cluster: kJacobiCluster where such a cluster fits on the device at the largest shared-memory size, else 1.
template <typename Kernel>
static bool psvd_cluster_fits(Kernel* k, size_t smem) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kJacobiCluster);
  cfg.blockDim = dim3(PS_T);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kJacobiCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  const bool ok = cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n > 0;
  (void)cudaGetLastError();
  return ok;
}

// 0: the attributes could not be set; else the CTAs of a projected SVD.  Once per process (contexts may be created
// from several threads).
static int psvd_ctas() {
  static std::once_flag once;
  static int ctas = 0;
  std::call_once(once, [] {
    const size_t s1 = psvd_sweeps_smem(JMAXK, 1);
    const size_t s2 = psvd_refine_smem(JMAXK) > psvd_refine_smem(kTinSmem) ? psvd_refine_smem(JMAXK) : psvd_refine_smem(kTinSmem);
    bool ok = psvd_attr(k_psvd_refine, s2);
    for (int k = 8; k <= JMAXK; k += 8) ok = ok && psvd_attr(psvd_sweeps_kernel(k), s1);
    if (ok)
      ctas = psvd_cluster_fits(psvd_sweeps_kernel(JMAXK), psvd_sweeps_smem(JMAXK, kJacobiCluster)) &&
                     psvd_cluster_fits(k_psvd_refine, s2)
                 ? kJacobiCluster
                 : 1;
    (void)cudaGetLastError();
  });
  return ctas;
}

int init_jacobi_attributes() { return psvd_ctas() > 0 ? 0 : 1; }

template <typename Kernel>
static bool psvd_launch(Kernel* k, const PsvdArgs& a, int nct, size_t smem, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nct);
  cfg.blockDim = dim3(PS_T);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = nct;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = nct > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, a) == cudaSuccess;
}

int launch_small_svd(const double* T, int ldT, int K, const double* S, int b, int nv, double* theta, double* Xl,
                     double* Wr, double* res, double tol, int f32, int max_sweeps, unsigned int* err,
                     unsigned long long* counters, double* ws, cudaStream_t st, int cluster) {
  // K is a multiple of the block size, itself a multiple of 8
  if (psvd_ctas() == 0 || K > JMAXK || K < 8 || (K & 7)) return 0;   // no launch; the caller's checks report it
  const int nct = cluster == 1 ? 1 : psvd_ctas();
  const PsvdArgs a{T, ldT, K, S, b, nv < K ? nv : K, theta, Xl, Wr, res, tol, f32, max_sweeps, err, counters, ws};
  if (!psvd_launch(psvd_sweeps_kernel(K), a, nct, psvd_sweeps_smem(K, nct), st)) return 0;
  return psvd_launch(k_psvd_refine, a, nct, psvd_refine_smem(K), st) ? 2 : 0;
}

}  // namespace svt
