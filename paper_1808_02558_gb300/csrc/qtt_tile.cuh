// QTT mat-vec passes that contract several cores at a time in shared memory
// (Sec. 3.2 mat-vec; layout of the intermediates in qtt_dev.cuh).
//
// A pass takes cores k, k-1, .., k-m+1.  In the flattened columns col = (J'', I), J'' =
// (j_1..j_{k-m}), I = (i_{k+1}..i_d), a block takes QT_NC consecutive columns and all
// 2^m values of (j_{k-m+1}..j_k): a tile [2^m][R][QT_NC] in shared memory, each rank
// padded to R.  Step s contracts core k-s, which turns bit s of the first index from
// j_{k-s} into i_{k-s}, in place: a thread reads its inputs into registers before it
// writes its outputs to the same slots.  Two cores a step: 4 r values in, 4 r values
// between, 4 r values out.
//
// Bound: FP32 arithmetic (4 r^2 N flops a core).  Packed multiply-adds over j (the
// stored quad (i, j) of a rank pair is two such pairs) leave issue slots for the
// shared-memory loads; every quad feeds eight multiply-adds; zero-padded quads need no
// per-value tests.  Against two cores a launch through global memory (49 to 60 us each
// at 2^20, rank 10) a pass of five moves 40 % of the bytes: 66 us, of which 26 at the
// FP32 rate.  Over a pass of interior ranks the FMA pipe is busy 42 % of the time (ncu):
// warps queue for it while a tile is contracted, and it idles for the rest (tiles in and
// out, barriers between steps, 1024 tiles on 304 blocks).  The whole product: 484 -> 266 us.
#pragma once

#include "pair.cuh"
#include "qtt_dev.cuh"

namespace qp {

constexpr int QT_NC = 32;          // columns of a tile: a warp's width
constexpr int QT_LD = QT_NC + 1;   // row stride (odd: the transposed first pass spreads over the banks)
constexpr int QT_THREADS = 256;
constexpr int QT_MAXM = 5;         // cores a pass at ranks up to 10

typedef unsigned long long u64x;

__device__ __forceinline__ u64x pack2(float a, float b) {
  u64x d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float sum2(u64x v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return a + b;
}

// Core kk (1-based) zero-padded to [R out][R in] quads (G(., i, j, .) as (00, 01), (10, 11)).
template <int R, class TC>
__device__ __forceinline__ void tile_stage(const QttDev& q, int kk, float4* out) {
  const int ro = q.ranks[kk - 1], ri = q.ranks[kk];
  const TC* G = static_cast<const TC*>(q.cores) + q.off[kk - 1];
  for (int t = threadIdx.x; t < R * R; t += blockDim.x) {
    const int a = t / R, b = t - a * R;
    float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a < ro && b < ri) {
      const long long base = (long long)a * 4 * ri + b;
      g = make_float4(core_ta<float, TC>(G, base), core_ta<float, TC>(G, base + ri), core_ta<float, TC>(G, base + 2 * ri),
                      core_ta<float, TC>(G, base + 3 * ri));
    }
    out[t] = g;
  }
}

// Cores k-s and k-s-1 on the tile (bits s and s+1 of the first index).
template <int R>
__device__ __forceinline__ void tile_step2(float* tile, int m, int s, int r1, int r0, int r2, const float4* gk,
                                           const float4* gm) {
  const int items = (1 << (m - 2)) * QT_NC;
  for (int it = threadIdx.x; it < items; it += blockDim.x) {
    const int col = it & (QT_NC - 1), h = it / QT_NC;
    const int jb = ((h >> s) << (s + 2)) | (h & ((1 << s) - 1));
    float* p[4];
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) p[jj] = tile + (jb | (jj << s)) * R * QT_LD + col;
    u64x v[2][R];  // [j_{k-1}][b]: (j_k = 0, j_k = 1)
#pragma unroll
    for (int b = 0; b < R; ++b) {
      v[0][b] = v[1][b] = 0ull;
      if (b < r1) {
        v[0][b] = pack2(p[0][b * QT_LD], p[1][b * QT_LD]);
        v[1][b] = pack2(p[2][b * QT_LD], p[3][b * QT_LD]);
      }
    }
    u64x t[2][R];  // [i_k][a]: (j_{k-1} = 0, j_{k-1} = 1)
#pragma unroll
    for (int a = 0; a < R; ++a) {
      t[0][a] = t[1][a] = 0ull;
      if (a < r0) {
        u64x s00 = 0ull, s01 = 0ull, s10 = 0ull, s11 = 0ull;  // [j_{k-1}][i_k]
#pragma unroll
        for (int b = 0; b < R; ++b) {
          const ulonglong2 g = *reinterpret_cast<const ulonglong2*>(gk + a * R + b);
          fma2(s00, g.x, v[0][b]);
          fma2(s01, g.y, v[0][b]);
          fma2(s10, g.x, v[1][b]);
          fma2(s11, g.y, v[1][b]);
        }
        t[0][a] = pack2(sum2(s00), sum2(s10));
        t[1][a] = pack2(sum2(s01), sum2(s11));
      }
    }
#pragma unroll 1
    for (int c = 0; c < r2; ++c) {
      u64x y00 = 0ull, y01 = 0ull, y10 = 0ull, y11 = 0ull;  // [i_{k-1}][i_k]
#pragma unroll
      for (int a = 0; a < R; ++a) {
        const ulonglong2 g = *reinterpret_cast<const ulonglong2*>(gm + c * R + a);
        fma2(y00, g.x, t[0][a]);
        fma2(y01, g.x, t[1][a]);
        fma2(y10, g.y, t[0][a]);
        fma2(y11, g.y, t[1][a]);
      }
      p[0][c * QT_LD] = sum2(y00);
      p[1][c * QT_LD] = sum2(y01);
      p[2][c * QT_LD] = sum2(y10);
      p[3][c * QT_LD] = sum2(y11);
    }
  }
}

// Core k-s alone (the last step of an odd pass), two items a thread on each quad.
template <int R>
__device__ __forceinline__ void tile_step1(float* tile, int m, int s, int r1, int r0, const float4* gk) {
  const int items = (1 << (m - 1)) * QT_NC;
  for (int it = threadIdx.x; it < items; it += 2 * blockDim.x) {
    const bool two = it + (int)blockDim.x < items;
    float* p[2];
    u64x v[2][R];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int w = two || i == 0 ? it + i * (int)blockDim.x : it;
      const int col = w & (QT_NC - 1), h = w / QT_NC;
      p[i] = tile + (((h >> s) << (s + 1)) | (h & ((1 << s) - 1))) * R * QT_LD + col;
      const float* p1 = p[i] + (1 << s) * R * QT_LD;
#pragma unroll
      for (int b = 0; b < R; ++b) v[i][b] = b < r1 ? pack2(p[i][b * QT_LD], p1[b * QT_LD]) : 0ull;
    }
#pragma unroll 1
    for (int a = 0; a < r0; ++a) {
      u64x y[2][2] = {};
#pragma unroll
      for (int b = 0; b < R; ++b) {
        const ulonglong2 g = *reinterpret_cast<const ulonglong2*>(gk + a * R + b);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          fma2(y[i][0], g.x, v[i][b]);
          fma2(y[i][1], g.y, v[i][b]);
        }
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (i == 0 || two) {
          p[i][a * QT_LD] = sum2(y[i][0]);
          p[i][(a + (1 << s) * R) * QT_LD] = sum2(y[i][1]);
        }
    }
  }
}

__device__ __forceinline__ void cp4(float* dst, const float* src) {  // an asynchronous 4-byte copy
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Bytes of shared memory of a pass of m cores with ranks padded to R.
// (the cores, and two tiles: the next one's inputs arrive while this one is contracted)
constexpr int tile_bytes(int R, int m) { return m * R * R * 16 + 2 * (1 << m) * R * QT_LD * 4; }

// One pass over the block's tiles (tile index first, first + stride, ..).  smem:
// tile_bytes(R, m), 16-byte aligned.  All threads of the block call it.
template <int R, class TC>
__device__ __forceinline__ void tile_pass(const QttDev& q, int k, int m, const float* in, float* out,
                                          unsigned char* smem, long long first, long long stride) {
  float4* cores = reinterpret_cast<float4*>(smem);
  float* tiles = reinterpret_cast<float*>(cores + m * R * R);
  const int lowbits = q.d - k, M2 = 1 << m, size = M2 * R * QT_LD;
  const long long nI = 1LL << lowbits;
  const int rin = q.ranks[k], rout = q.ranks[k - m];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long ntiles = (1LL << (q.d - m)) / QT_NC;
  auto fetch = [&](long long tl, float* tile) {
    const long long c0 = tl * QT_NC;
    if (lowbits == 0) {
      // first pass (rank 1, no I): the tile's inputs are consecutive, the bits fastest
#pragma unroll 4
      for (int i = threadIdx.x; i < (QT_NC << m); i += QT_THREADS)
        cp4(tile + (i & (M2 - 1)) * R * QT_LD + (i >> m), in + (c0 << m) + i);
    } else {
      // rows (bits, rank) of consecutive I (QT_NC <= 2^lowbits: one J'')
      const float* src = in + (((c0 >> lowbits) << m) * rin << lowbits) + (c0 & (nI - 1)) + lane;
      float* dst = tile + lane;
      for (int jb = 0; jb < M2; ++jb)
#pragma unroll 2
        for (int b = warp; b < rin; b += QT_THREADS / 32)
          cp4(dst + (jb * R + b) * QT_LD, src + ((long long)(jb * rin + b) << lowbits));
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int s = 0; s < m; ++s) tile_stage<R, TC>(q, k - s, cores + s * R * R);
  if (first < ntiles) fetch(first, tiles);
  int cur = 0;
  for (long long tl = first; tl < ntiles; tl += stride, cur ^= 1) {
    const long long c0 = tl * QT_NC;
    float* tile = tiles + cur * size;
    if (tl + stride < ntiles) {
      fetch(tl + stride, tiles + (cur ^ 1) * size);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    int s = 0;
    for (; s + 2 <= m; s += 2) {
      tile_step2<R>(tile, m, s, q.ranks[k - s], q.ranks[k - s - 1], q.ranks[k - s - 2], cores + s * R * R,
                    cores + (s + 1) * R * R);
      __syncthreads();
    }
    if (s < m) {
      tile_step1<R>(tile, m, s, q.ranks[k - s], q.ranks[k - s - 1], cores + s * R * R);
      __syncthreads();
    }
    if (lowbits == 0) {
      // columns J'': 2^m consecutive outputs a rank
      const int per = rout << m;
#pragma unroll 4
      for (int i = threadIdx.x; i < QT_NC * per; i += QT_THREADS) {
        const int c = i / per, w = i - c * per;
        out[c0 * per + i] = tile[((w & (M2 - 1)) * R + (w >> m)) * QT_LD + c];
      }
    } else {
      float* dst = out + ((((c0 >> lowbits) * rout) << (m + lowbits)) + (c0 & (nI - 1))) + lane;
      const int nrow = M2 * rout;
#pragma unroll 4
      for (int row = warp; row < nrow; row += QT_THREADS / 32) {
        const int a = row >> m, ib = row & (M2 - 1);
        dst[(long long)row << lowbits] = tile[(ib * R + a) * QT_LD + lane];
      }
    }
    __syncthreads();
  }
}

// Number of cores of the next pass from core k down, with ranks up to 16 on both sides
// (R: the padded rank), or 0: not this way.  At most five (four above rank 10: two
// blocks' tiles an SM), and equal shares of what is left, because a pass of two or
// three takes its copies' latency for little work (96 us for the last two cores at
// 2^20, rank 10, against 88 for six).  A pass needs QT_NC columns, and after the first
// one they have to lie in one J''.
inline int tile_plan(const QttDev& q, int k, int& R) {
  const int low = q.d - k;
  if (low != 0 && (1 << (low < 10 ? low : 10)) < QT_NC) return 0;
  int run = 0, most = QT_MAXM;  // cores from k down that fit a pass, and how many it takes
  for (int r = q.ranks[k]; k - run >= 1; ++run) {
    const int rn = q.ranks[k - run - 1];
    if (rn > 16 || r > 16) break;
    if (rn > 10 || r > 10) most = 4;
    r = rn;
  }
  if (low == 0) most = QT_MAXM;  // the first pass has to leave QT_NC columns in a J''
  const int share = run > 0 ? (run + (run + most - 1) / most - 1) / ((run + most - 1) / most) : 0;
  int m = 0, r = q.ranks[k];
  for (; m < (low == 0 ? QT_MAXM : share) && m < run; ++m) {
    const int rn = q.ranks[k - m - 1] > r ? q.ranks[k - m - 1] : r;
    if (q.d - m - 1 < 5) break;
    r = rn;
  }
  if (low == 0 && k - m > 0 && (1 << m) < QT_NC) return 0;
  if (m < 2 || r > 16) return 0;
  R = r <= 4 ? 4 : (r <= 8 ? 8 : (r <= 10 ? 10 : (r <= 12 ? 12 : 16)));
  // two or three cores of ranks above 12: one block an SM does not hide the copies
  return R == 16 && m < 4 ? 0 : m;
}

}  // namespace qp
