// Small dense FP64 linear algebra inside one thread block, shared by the QTT
// compression, rounding and inversion: a block sum, and the symmetric
// eigendecomposition by cyclic Jacobi with round-robin (parallel) rotation
// order (Golub and Van Loan, Matrix Computations, Sec. 8.5), eigenvalues in
// descending order, and the truncation rank of Sec. 3.1.
//
// GB300's FP64 pipe is narrow and an L2 round trip costs hundreds of cycles,
// so a matrix of order n <= SYEV_SMEM_N is copied into shared memory (the
// calling kernel launches with SYEV_SMEM_BYTES of dynamic shared memory) and
// every rotation round works there; larger matrices are rotated in place in
// global memory.
#pragma once

namespace qp {
namespace dla {

constexpr int SYEV_SMEM_N = 64;
// three matrices with an odd leading dimension: columns are then free of bank conflicts
// (with 40 doubles a row a column's 32 entries lay in two banks, 10 400 cycles a round of
// rotations).  With the FP32 start an order-40 decomposition of a compression takes
// 471 us; without either it took 989.
constexpr int SYEV_SMEM_BYTES = 3 * SYEV_SMEM_N * (SYEV_SMEM_N + 1) * (int)sizeof(double);
constexpr int SYEV_F32_N = 16;  // smallest order that starts with FP32 sweeps

__device__ inline double block_sum(double v) {
  __shared__ double sm[32];
  __shared__ double res;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double x = (threadIdx.x < (blockDim.x >> 5)) ? sm[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (threadIdx.x == 0) res = x;
  }
  __syncthreads();
  double out = res;
  __syncthreads();
  return out;
}

// Round-robin pairing of m (even) players: round r, pair i.
__device__ __forceinline__ void rr_pair(int m, int r, int i, int& p, int& q) {
  if (i == 0) {
    p = m - 1;
    q = r;
  } else {
    p = r + i;
    if (p >= m - 1) p -= m - 1;
    q = r - i;
    if (q < 0) q += m - 1;
  }
  if (p > q) {
    const int t = p;
    p = q;
    q = t;
  }
}

// Rotation (c, s) annihilating a_pq of the 2 x 2 block [[a_pp, a_pq], [a_pq,
// a_qq]] (a_pq != 0).  precise: the angle in FP64.  Otherwise the angle comes
// from FP32 arithmetic on the block scaled by a power of two (FP64 division and
// square root are long dependent sequences on GB300's narrow FP64 pipe), and
// (c, s) is made a rotation to FP64 rounding by two Newton steps towards
// c^2 + s^2 = 1: the rotation stays exactly orthogonal and only its angle
// carries the FP32 error, which the next sweep removes (the sweeps switch to
// precise angles once the off-diagonal part is small).
__device__ __forceinline__ void jacobi_rotation(double app, double aqq, double apq, bool precise, double& c,
                                                double& s) {
  if (!precise) {
    const double num = aqq - app, den = 2.0 * apq;
    int e;
    frexp(fmax(fabs(num), fabs(den)), &e);
    const float nf = (float)ldexp(num, -e), df = (float)ldexp(den, -e);
    if (df != 0.0f && isfinite(nf / df)) {
      const float tau = nf / df;
      // large |tau|: t = 1 / (2 tau) to FP32 rounding (tau^2 would overflow)
      const float t = fabsf(tau) > 1e18f ? 0.5f / tau
                                         : (tau >= 0.0f ? 1.0f : -1.0f) / (fabsf(tau) + sqrtf(1.0f + tau * tau));
      const float cf = rsqrtf(1.0f + t * t);
      double cc = (double)cf, ss = (double)(t * cf);
      for (int it = 0; it < 2; ++it) {
        const double f = 1.5 - 0.5 * (cc * cc + ss * ss);
        cc *= f;
        ss *= f;
      }
      c = cc;
      s = ss;
      return;
    }
  }
  const double tau = (aqq - app) / (2.0 * apq);
  const double t = (tau >= 0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
  c = 1.0 / sqrt(1.0 + t * t);
  s = t * c;
}

// x 2^k for a double, k within +-2000 and the result finite, by its exponent's bits (0 stays 0;
// results below the normal range become 0).
__device__ __forceinline__ double shift_exponent(double x, int k) {
  const int hi = __double2hiint(x), e = ((hi >> 20) & 0x7ff) + k;
  if (((hi >> 20) & 0x7ff) == 0 || e <= 0) return 0.0;
  return __hiloint2double((hi & 0x800fffff) | (e << 20), __double2loint(x));
}

// The same for the sweeps that follow an FP32 start, entries finite: every angle in FP32
// (an FP64 instruction takes a warp 64 cycles, a division and a square root are a dozen
// each), the scaling by exponent bits, and one third-order step towards c^2 + s^2 = 1.
// The angle's FP32 error leaves 1e-7 of a_pq to the next sweep.
__device__ __forceinline__ void jacobi_rotation_f32(double app, double aqq, double apq, double& c, double& s) {
  const double num = aqq - app;
  const int en = (__double2hiint(num) >> 20) & 0x7ff, ep = (__double2hiint(apq) >> 20) & 0x7ff;
  const int k = 1023 - (en > ep ? en : ep);
  const float nf = (float)shift_exponent(num, k), df = 2.f * (float)shift_exponent(apq, k);
  if (df == 0.f) return;  // the angle is below FP64 rounding
  const float tau = nf / df;
  // large |tau|: t = 1 / (2 tau) to FP32 rounding (tau^2 would overflow)
  const float t = fabsf(tau) > 1e18f ? 0.5f / tau
                                     : (tau >= 0.0f ? 1.0f : -1.0f) / (fabsf(tau) + sqrtf(1.0f + tau * tau));
  const float cf = rsqrtf(1.0f + t * t);
  const double cc = (double)cf, ss = (double)(t * cf);
  const double e = fma(ss, ss, fma(cc, cc, -1.0));
  const double f = fma(e, fma(e, 0.375, -0.5), 1.0);
  c = cc * f;
  s = ss * f;
}

// Row i of block idx in the upper triangle of npairs x npairs blocks (row i holds
// npairs - i of them).
__device__ __forceinline__ int block_row(int idx, int npairs) {
  int i = 0;
  while (i < npairs - 1 && idx >= npairs - i) {
    idx -= npairs - i;
    ++i;
  }
  return i;
}

// What a thread does in a round: items [0, nblk) are 2 x 2 blocks (i, j), i <= j, of A;
// the others row j of V and pair i.  The first item's indices do not change from round
// to round and are found once.
struct RoundItem {
  int i, j;
};
__device__ __forceinline__ RoundItem round_item(int idx, int n, int npairs, int nblk) {
  RoundItem w;
  if (idx < nblk) {
    w.i = block_row(idx, npairs);
    w.j = idx - w.i * (2 * npairs - w.i + 1) / 2 + w.i;
  } else {
    w.i = (idx - nblk) / n;
    w.j = idx - nblk - w.i * n;
  }
  return w;
}

// One round of rotations (rc, rs) on the pairs (rp, rq): A <- J^T A J, V <- V J
// (leading dimension ld).
template <class T>
__device__ __forceinline__ void apply_round(T* A, T* V, int n, int ld, int npairs, RoundItem w, const int* rp,
                                            const int* rq, const T* rc, const T* rs) {
  const int tid = threadIdx.x, nt = blockDim.x;
  // A <- J^T A J in one pass: J is block diagonal in the pairs, so the 2 x 2
  // block of rows (p_i, q_i) and columns (p_j, q_j) becomes J_i^T A_ij J_j;
  // A stays symmetric, so a thread forms block (i, j), i <= j, and writes its
  // transpose into block (j, i) as well (a missing q of the odd pair is left
  // out); V <- V J for one row and pair per thread
  const int nblk = npairs * (npairs + 1) / 2;
  for (int idx = tid; idx < nblk + npairs * n; idx += nt) {
    if (idx != tid) w = round_item(idx, n, npairs, nblk);
    const int i = w.i, j = w.j;
    if (idx < nblk) {
      const int p = rp[i], q = rq[i], p2 = rp[j], q2 = rq[j];
      const T ci = rc[i], si = rs[i], cj = rc[j], sj = rs[j];
      if (si == T(0) && sj == T(0)) continue;
      const bool hq = q < n, hq2 = q2 < n;
      const T a00 = A[p * ld + p2], a01 = hq2 ? A[p * ld + q2] : T(0);
      const T a10 = hq ? A[q * ld + p2] : T(0), a11 = (hq && hq2) ? A[q * ld + q2] : T(0);
      // rows: (J_i^T A): row p <- c a_p - s a_q, row q <- s a_p + c a_q
      const T b00 = ci * a00 - si * a10, b01 = ci * a01 - si * a11;
      const T b10 = si * a00 + ci * a10, b11 = si * a01 + ci * a11;
      // columns: (. J_j): col p2 <- c b_p2 - s b_q2, col q2 <- s b_p2 + c b_q2
      const T c00 = cj * b00 - sj * b01, c01 = sj * b00 + cj * b01;
      const T c10 = cj * b10 - sj * b11, c11 = sj * b10 + cj * b11;
      A[p * ld + p2] = c00;
      if (hq2) A[p * ld + q2] = c01;
      if (hq) A[q * ld + p2] = c10;
      if (hq && hq2) A[q * ld + q2] = c11;
      if (i != j) {  // the mirrored block (j, i)
        A[p2 * ld + p] = c00;
        if (hq2) A[q2 * ld + p] = c01;
        if (hq) A[p2 * ld + q] = c10;
        if (hq && hq2) A[q2 * ld + q] = c11;
      }
    } else {
      const int p = rp[i], q = rq[i];
      if (q >= n || rs[i] == T(0)) continue;
      const T c = rc[i], sn = rs[i];
      const T a = V[j * ld + p], b = V[j * ld + q];
      V[j * ld + p] = c * a - sn * b;
      V[j * ld + q] = sn * a + c * b;
    }
  }
}

// Sums of squares of A's off-diagonal and diagonal entries over the block.
template <class T>
__device__ __forceinline__ void off_on(const T* A, int n, int ld, double& off, double& on) {
  T o = T(0), d = T(0);
  for (int i = threadIdx.x; i < n * n; i += blockDim.x) {
    const int x = i / n, y = i - x * n;
    const T a = A[x * ld + y];
    if (x == y) d += a * a;
    else o += a * a;
  }
  off = block_sum((double)o);
  on = block_sum((double)d);
}

// Jacobi sweeps on A (n x n, leading dimension ld, destroyed); V accumulates the
// rotations (from the V given when `started`, else from I).  A and V may live in shared
// or global memory.  After an FP32 start entries that together stay within the stopping
// test are left alone: the last sweeps then rotate few pairs, and warps without any skip
// their FP64 work.  Without one every entry is rotated, which keeps the small eigenvalues
// of graded matrices accurate relative to themselves.
__device__ inline void jacobi_sweeps(double* A, double* V, int n, int ld, bool started) {
  __shared__ double rc[256], rs[256];
  __shared__ int rp[256], rq[256];
  __shared__ int done, precise;
  __shared__ double small;
  const int tid = threadIdx.x, nt = blockDim.x;
  if (!started)
    for (int i = tid; i < n * n; i += nt) V[i / n * ld + i % n] = (i / n == i % n) ? 1.0 : 0.0;
  __syncthreads();
  const int m = n + (n & 1);
  const int npairs = m / 2;
  const RoundItem w = round_item(tid, n, npairs, npairs * (npairs + 1) / 2);
  for (int sweep = 0; sweep < 40 && n > 1; ++sweep) {
    double off, on;
    off_on(A, n, ld, off, on);
    if (tid == 0) {
      done = (off <= 1e-30 * on) || (on == 0.0);
      precise = off <= 1e-16 * on;  // off-diagonal below 1e-8 of the diagonal: FP64 angles
      small = started ? 1e-15 * sqrt(on) / n : 1e-300;
    }
    __syncthreads();
    if (done) break;
    const bool prec = precise != 0;
    for (int r = 0; r < m - 1; ++r) {
      for (int i = tid; i < npairs; i += nt) {
        int p, q;
        rr_pair(m, r, i, p, q);
        double c = 1.0, s = 0.0;
        if (q < n) {
          const double apq = A[p * ld + q];
          const double app = A[p * ld + p], aqq = A[q * ld + q];
          if (fabs(apq) > 1e-300 && fabs(apq) > small) {
            if (started) jacobi_rotation_f32(app, aqq, apq, c, s);
            else jacobi_rotation(app, aqq, apq, prec, c, s);
          }
        }
        rp[i] = p;
        rq[i] = q;
        rc[i] = c;
        rs[i] = s;
      }
      __syncthreads();
      apply_round(A, V, n, ld, npairs, w, rp, rq, rc, rs);
      __syncthreads();
    }
  }
}

// FP32 sweeps on A (n x n, scaled to a largest entry near 1) with the rotations in V,
// until the off-diagonal part is at FP32's rounding level or stops falling.
__device__ inline void jacobi_sweeps_f32(float* A, float* V, int n, int ld) {
  __shared__ float rc[64], rs[64];
  __shared__ int rp[64], rq[64];
  __shared__ int done;
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int i = tid; i < n * n; i += nt) V[i / n * ld + i % n] = (i / n == i % n) ? 1.f : 0.f;
  __syncthreads();
  const int m = n + (n & 1), npairs = m / 2;
  const RoundItem w = round_item(tid, n, npairs, npairs * (npairs + 1) / 2);
  double last = 1e300;
  for (int sweep = 0; sweep < 12; ++sweep) {
    double so, sn;
    off_on(A, n, ld, so, sn);
    if (tid == 0) done = !(so > 1e-13 * sn) || !(so < 0.25 * last);
    last = so;
    __syncthreads();
    if (done) break;
    for (int r = 0; r < m - 1; ++r) {
      for (int i = tid; i < npairs; i += nt) {
        int p, q;
        rr_pair(m, r, i, p, q);
        float c = 1.f, s = 0.f;
        if (q < n) {
          const float apq = A[p * ld + q], num = A[q * ld + q] - A[p * ld + p];
          // the angle's quotient has to be finite: a pair this small or this far apart is left
          if (fabsf(apq) > 1e-9f * fabsf(num) && fabsf(apq) > 1e-30f) {
            const float tau = __fdividef(num, 2.f * apq), u = 1.f + tau * tau;
            const float t = copysignf(__fdividef(1.f, fabsf(tau) + u * rsqrtf(u)), tau);
            c = rsqrtf(1.f + t * t);
            s = t * c;
          }
        }
        rp[i] = p;
        rq[i] = q;
        rc[i] = c;
        rs[i] = s;
      }
      __syncthreads();
      apply_round(A, V, n, ld, npairs, w, rp, rq, rc, rs);
      __syncthreads();
    }
  }
}

// C = X^T Y (sym: known to be symmetric, half of it formed), X Y or X (1.5 I - 0.5 Y)
// for n x n matrices in shared memory (n <= SYEV_SMEM_N, leading dimension ld, 1024
// threads), C may be X or Y: every thread forms its outputs before any is written.
enum { MM_SYM_TN, MM_NN, MM_ORTH };
template <int MODE>
__device__ inline void smem_matmul(const double* X, const double* Y, double* C, int n, int ld) {
  constexpr int PER = MODE == MM_SYM_TN ? 3 : 4;  // ceil(64 * 65 / 2 / 1024), 64 * 64 / 1024
  const int tid = threadIdx.x, nt = blockDim.x;
  const int sx = MODE == MM_SYM_TN ? 1 : ld, sk = MODE == MM_SYM_TN ? ld : 1;
  const int items = MODE == MM_SYM_TN ? n * (n + 1) / 2 : n * n;
  double acc[PER];
  int at[PER];
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int i = tid + u * nt;
    at[u] = -1;
    if (i < items) {
      int x, y;
      if (MODE == MM_SYM_TN) {
        x = block_row(i, n);
        y = i - x * (2 * n - x + 1) / 2 + x;
      } else {
        x = i / n;
        y = i - x * n;
      }
      const double *px = X + x * sx, *py = Y + y;
      double s0 = 0.0, s1 = 0.0;
      int k = 0;
      for (; k + 2 <= n; k += 2) {
        s0 = fma(px[k * sk], py[k * ld], s0);
        s1 = fma(px[(k + 1) * sk], py[(k + 1) * ld], s1);
      }
      if (k < n) s0 = fma(px[k * sk], py[k * ld], s0);
      acc[u] = MODE == MM_ORTH ? 1.5 * X[x * ld + y] - 0.5 * (s0 + s1) : s0 + s1;
      at[u] = x * ld + y;
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < PER; ++u)
    if (at[u] >= 0) {
      C[at[u]] = acc[u];
      if (MODE == MM_SYM_TN) C[at[u] % ld * ld + at[u] / ld] = acc[u];
    }
  __syncthreads();
}

// Most of the way in FP32: A's eigenvectors to FP32 accuracy (a few sweeps on a copy),
// made orthogonal to FP64 rounding by two Newton-Schulz steps V (3 I - V^T V) / 2 (Bjorck
// and Bowie, SIAM J. Numer. Anal. 8 (1971)), and
// A <- V^T A V in FP64, whose off-diagonal part is then about 1e-7 of the diagonal: the
// FP64 sweeps that follow start from there, two or three instead of eight or nine.
// Against FP64 sweeps alone, on the Schur matrices of piles of 4^3 to 7^3 at 1e-4 to 1e-1
// and ranks 6 to 16 (64-bit Gram matrices): ||G V - V w|| / ||G|| at most 2.1e-15 (5.9e-15),
// |V^T V - I| at most 3.1e-15 (1.8e-14).
// Returns false (A untouched) when A is zero or not finite in FP32's range.
// work: n ld doubles beside A and V.
__device__ inline bool f32_start(double* A, double* V, double* work, int n, int ld) {
  const int tid = threadIdx.x, nt = blockDim.x;
  __shared__ double scale;
  double tr = 0.0;
  for (int i = tid; i < n; i += nt) tr += fabs(A[i * ld + i]);
  tr = block_sum(tr);
  if (tid == 0) scale = tr > 1e-280 && tr < 1e280 ? ldexp(1.0, -ilogb(tr)) : 0.0;
  __syncthreads();
  if (scale == 0.0) return false;
  float* a32 = reinterpret_cast<float*>(work);
  float* v32 = a32 + n * ld;
  float bad = 0.f;
  for (int i = tid; i < n * n; i += nt) {
    const int x = i / n, y = i - x * n;
    const float a = (float)(A[x * ld + y] * scale);
    if (!(fabsf(a) < 1e6f)) bad = 1.f;
    a32[x * ld + y] = a;
  }
  if (__syncthreads_or(bad != 0.f)) return false;
  jacobi_sweeps_f32(a32, v32, n, ld);
  __syncthreads();
  for (int i = tid; i < n * ld; i += nt) V[i] = i % ld < n ? (double)v32[i] : 0.0;
  __syncthreads();
  for (int k = 0; k < 2; ++k) {
    smem_matmul<MM_SYM_TN>(V, V, work, n, ld);
    smem_matmul<MM_ORTH>(V, work, V, n, ld);
  }
  smem_matmul<MM_NN>(A, V, work, n, ld);
  smem_matmul<MM_SYM_TN>(V, work, A, n, ld);
  return true;
}

// Eigendecomposition of the symmetric n x n matrix A (row-major, destroyed):
// w[0..n) the eigenvalues in descending order (ties by index), Vs the
// eigenvectors as columns (row-major n x n); V is workspace n x n.  `smem`
// points at SYEV_SMEM_BYTES of the block's dynamic shared memory, or is null.
// f32: the caller truncates the spectrum at SYEV_F32_EPS of its norm or above, so the FP32
// start may be taken: it leaves eigenvalues exact to FP64 rounding of the largest one, not
// of themselves (a kept one is above 1e-11 of the largest there).
constexpr double SYEV_F32_EPS = 1e-4;
__device__ inline void syev(double* A, double* V, double* Vs, double* w, int n, double* smem, bool f32) {
  const int tid = threadIdx.x, nt = blockDim.x;
  double* a = A;
  double* v = V;
  int ld = n;
  bool started = false;
  if (smem && n <= SYEV_SMEM_N) {
    ld = n | 1;
    a = smem;
    v = smem + n * ld;
    for (int i = tid; i < n * n; i += nt) a[i / n * ld + i % n] = A[i];
    __syncthreads();
    started = f32 && n >= SYEV_F32_N && f32_start(a, v, smem + 2 * n * ld, n, ld);
  }
  jacobi_sweeps(a, v, n, ld, started);
  for (int i = tid; i < n; i += nt) {
    const double di = a[i * ld + i];
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      const double dj = a[j * ld + j];
      if (dj > di || (dj == di && j < i)) ++rank;
    }
    w[rank] = di;
    for (int row = 0; row < n; ++row) Vs[row * n + rank] = v[row * ld + i];
  }
  __syncthreads();
}

// One-sided (Hestenes) Jacobi: the k vectors of length L, element e of vector
// i at X[i sv + e se], are made mutually orthogonal by plane rotations applied
// to the vectors themselves (no Gram matrix, so singular values down to FP64
// rounding of the largest are resolved; Demmel and Veselic, SIAM J. Matrix
// Anal. Appl. 13 (1992)).  Vr (k x k, row-major) accumulates the rotations:
// with the vectors as columns, X_new = X_old Vr.  A warp handles one pair of a
// round-robin round; sweeps stop when no pair had |x_p.x_q| above
// sqrt(L) eps sqrt(|x_p|^2 |x_q|^2).
__device__ inline void osj(double* X, int k, int L, long long sv, long long se, double* Vr) {
  __shared__ int s_rot;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  for (int i = tid; i < k * k; i += nt) Vr[i] = (i / k == i % k) ? 1.0 : 0.0;
  const double tol = sqrt((double)L) * 2.2e-16;
  const int m = k + (k & 1), npairs = m / 2;
  __syncthreads();
  for (int sweep = 0; sweep < 60 && k > 1; ++sweep) {
    if (tid == 0) s_rot = 0;
    __syncthreads();
    for (int r = 0; r < m - 1; ++r) {
      for (int i = warp; i < npairs; i += nw) {
        int p, q;
        rr_pair(m, r, i, p, q);
        if (q >= k) continue;
        double al = 0.0, be = 0.0, ga = 0.0;
        for (int e = lane; e < L; e += 32) {
          const double xp = X[p * sv + e * se], xq = X[q * sv + e * se];
          al += xp * xp;
          be += xq * xq;
          ga += xp * xq;
        }
        for (int o = 16; o > 0; o >>= 1) {
          al += __shfl_xor_sync(0xffffffffu, al, o);
          be += __shfl_xor_sync(0xffffffffu, be, o);
          ga += __shfl_xor_sync(0xffffffffu, ga, o);
        }
        if (fabs(ga) > 1e-300 && fabs(ga) > tol * sqrt(al * be)) {
          const double zeta = (be - al) / (2.0 * ga);
          const double t = (zeta >= 0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
          const double c = 1.0 / sqrt(1.0 + t * t), sn = t * c;
          for (int e = lane; e < L; e += 32) {
            const double xp = X[p * sv + e * se], xq = X[q * sv + e * se];
            X[p * sv + e * se] = c * xp - sn * xq;
            X[q * sv + e * se] = sn * xp + c * xq;
          }
          for (int j = lane; j < k; j += 32) {
            const double vp = Vr[j * k + p], vq = Vr[j * k + q];
            Vr[j * k + p] = c * vp - sn * vq;
            Vr[j * k + q] = sn * vp + c * vq;
          }
          if (lane == 0) s_rot = 1;
        }
      }
      __syncthreads();
    }
    const int any = s_rot;
    __syncthreads();
    if (!any) break;
  }
}

// Norms of the k vectors of X (as in osj) into sig, and ord[j] = the index of
// the j-th largest (ties by index).
__device__ inline void osj_norms(const double* X, int k, int L, long long sv, long long se, double* sig, int* ord) {
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int i = tid; i < k; i += nt) {
    double s = 0.0;
    for (int e = 0; e < L; ++e) s += X[i * sv + e * se] * X[i * sv + e * se];
    sig[i] = sqrt(s);
  }
  __syncthreads();
  for (int i = tid; i < k; i += nt) {
    int rank = 0;
    for (int j = 0; j < k; ++j)
      if (sig[j] > sig[i] || (sig[j] == sig[i] && j < i)) ++rank;
    ord[rank] = i;
  }
  __syncthreads();
}

// Smallest r with sqrt(sum_{l >= r} lambda_l) <= delta, 1 <= r <= min(rmax, n)
// (eigenvalues of a Gram matrix, descending: the squared singular values).
__device__ inline int trunc_rank(const double* lam, int n, double delta, int rmax) {
  double tail = 0.0;
  int r = n;
  for (int k = n - 1; k >= 1; --k) {
    tail += fmax(lam[k], 0.0);
    if (sqrt(tail) <= delta) r = k;
    else break;
  }
  if (r > rmax) r = rmax;
  if (r < 1) r = 1;
  return r;
}

}  // namespace dla
}  // namespace qp
