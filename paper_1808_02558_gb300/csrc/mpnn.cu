// Learned warm start (an extension, not in the paper): a message-passing
// network over the contact graph predicts the impulses that start the PDIP.
// Contacts are the nodes; a message goes from a contact to each of its dynamic
// bodies and back (m_b = sum of h_c over the body's contacts, s_c = m_a + m_b).
//   h0 = relu(W0 x + b0), hl = relu(Wl [h(l-1); s(h(l-1))] + bl) (l = 1..3),
//   o = Wo h3 + bo,  with x the 8 scaled contact features (n, Phi/dt, the
// relative velocity in the contact frame, mu).  Parameters are BF16-rounded
// for the passes (FP32 master kept by the caller), activations and sums FP32.
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

#include "internal.cuh"
#include "pair.cuh"
#include "tc.cuh"

namespace qp {

// The driver's tensor-map encoder, looked up once (shared with qtt_tc.cu).
PFN_cuTensorMapEncodeTiled_v12000 tmap_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  QP_REQUIRE(fn != nullptr, QP_CUDA_ERROR, "cuTensorMapEncodeTiled is not available");
  return fn;
}

namespace {

constexpr int MF = 8, MW = 64, MO = 3, ML = 3;
constexpr int OFF_W0 = 0, OFF_B0 = MW * MF;
constexpr int LAYER = MW * 2 * MW + MW;
constexpr int OFF_L = OFF_B0 + MW;                // layer l: W at OFF_L + l*LAYER, b after W
constexpr int OFF_WO = OFF_L + ML * LAYER, OFF_BO = OFF_WO + MO * MW;
constexpr int NPAR = OFF_BO + MO;
static_assert(NPAR == QP_MPNN_NPARAM, "parameter layout");

struct Scale {
  float s[MF];
};

__global__ void k_mp_round(const float* __restrict__ p, __nv_bfloat16* __restrict__ q, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) q[i] = __float2bfloat16_rn(p[i]);
}

__device__ __forceinline__ float pb(const __nv_bfloat16* p, int i) { return __bfloat162float(p[i]); }

// The passes over contacts and bodies below are bound by the memory system: each
// takes 16 lanes a row, one float4 of the 64 features a lane, so that a warp's
// loads and stores are whole 256-byte rows and four or more are in flight a thread.

// Input layer: x = scaled features (X, kept for the weight gradient) and
// H0 = relu(W0 x + b0).  Each block forms the features of 256 contacts, one a
// thread (they take an FP64 division and seven conversions, which 16 lanes a row
// would repeat on the narrow FP64 pipe: 93 us), and then the outputs with 16 lanes a
// row, a lane keeping the weights of its four outputs in registers.  On the 40^3 pile
// 20 us in place of 11 us for the features and 58 us for one thread an output.
__global__ void __launch_bounds__(256)
    k_mp_input(int Nc, int slots, const double* __restrict__ phi, const double* __restrict__ frame,
               const double* __restrict__ r, double dt, double mu, Scale sc, const __nv_bfloat16* __restrict__ W,
               const __nv_bfloat16* __restrict__ bias, float* __restrict__ X, float* __restrict__ H0) {
  __shared__ __align__(16) float sx[256][MF];
  const int q = threadIdx.x & 15;
  float w[4][MF], b0[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    b0[j] = pb(bias, 4 * q + j);
#pragma unroll
    for (int k = 0; k < MF; ++k) w[j][k] = pb(W, (4 * q + j) * MF + k);
  }
  for (int c0 = blockIdx.x * 256; c0 < Nc; c0 += gridDim.x * 256) {
    const int c = c0 + (int)threadIdx.x;
    __syncthreads();
    if (c < Nc) {
      const double pd = phi[c] / dt;
      const long long row = (long long)slots * c;
      float x[MF];
      x[0] = (float)frame[c];
      x[1] = (float)frame[(size_t)Nc + c];
      x[2] = (float)frame[2 * (size_t)Nc + c];
      x[3] = (float)pd;
      x[4] = (float)(r[row] - pd);
      x[5] = (float)r[row + 1];
      x[6] = (float)r[row + 2];
      x[7] = (float)mu;
#pragma unroll
      for (int k = 0; k < MF; ++k) x[k] *= sc.s[k];
      const float4 xa = make_float4(x[0], x[1], x[2], x[3]), xb = make_float4(x[4], x[5], x[6], x[7]);
      float4* s4 = reinterpret_cast<float4*>(&sx[threadIdx.x][0]);
      s4[0] = xa;
      s4[1] = xb;
      float4* X4 = reinterpret_cast<float4*>(X) + 2 * (size_t)c;
      X4[0] = xa;
      X4[1] = xb;
    }
    __syncthreads();
    const int n = min(256, Nc - c0);
    for (int i = threadIdx.x >> 4; i < n; i += 16) {
      const float4 xa = reinterpret_cast<const float4*>(&sx[i][0])[0], xb = reinterpret_cast<const float4*>(&sx[i][0])[1];
      const float x[MF] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
      float y[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float acc = b0[j];
#pragma unroll
        for (int k = 0; k < MF; ++k) acc = fmaf(w[j][k], x[k], acc);
        y[j] = fmaxf(acc, 0.f);
      }
      reinterpret_cast<float4*>(H0)[16 * (size_t)(c0 + i) + q] = make_float4(y[0], y[1], y[2], y[3]);
    }
  }
}

// Output layer O = Wo h + bo.  With a target (Yt) it forms the loss in the same
// pass instead of storing O: d = O - Y, dO = 2 d / (3 Nc), and the block's share of
// sum d^2 in FP64 (part[block]).  The loss sum used to be one block over all 3 Nc
// squares (1034 us on the 40^3 pile); here the pass with it takes 31 us (58 without).
__global__ void __launch_bounds__(256)
    k_mp_output(int Nc, const float* __restrict__ H, const __nv_bfloat16* __restrict__ W,
                const __nv_bfloat16* __restrict__ bias, float* __restrict__ O, const float* __restrict__ Yt,
                float* __restrict__ dO, double* __restrict__ part) {
  const int q = threadIdx.x & 15;
  float w[MO][4], b0[MO];
#pragma unroll
  for (int j = 0; j < MO; ++j) {
    b0[j] = pb(bias, j);
#pragma unroll
    for (int k = 0; k < 4; ++k) w[j][k] = pb(W, j * MW + 4 * q + k);
  }
  const float n3 = (float)(3 * Nc);
  double sq = 0.0;
  const int rows = (blockDim.x >> 4) * gridDim.x;
  // the bound is rounded up so that all lanes of a warp reach the shuffles
#pragma unroll 2
  for (int c = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 4); c < ((Nc + 1) & ~1); c += rows) {
    const float4 h = c < Nc ? reinterpret_cast<const float4*>(H)[16 * (size_t)c + q] : make_float4(0.f, 0.f, 0.f, 0.f);
    float o[MO];
#pragma unroll
    for (int j = 0; j < MO; ++j) {
      o[j] = fmaf(w[j][3], h.w, fmaf(w[j][2], h.z, fmaf(w[j][1], h.y, w[j][0] * h.x)));
#pragma unroll
      for (int s = 8; s > 0; s >>= 1) o[j] += __shfl_xor_sync(0xffffffffu, o[j], s);
      o[j] += b0[j];
    }
    if (q < MO && c < Nc) {
      const float v = q == 0 ? o[0] : (q == 1 ? o[1] : o[2]);
      const size_t i = 3 * (size_t)c + q;
      if (Yt) {
        const float d = v - Yt[i];
        dO[i] = 2.f * d / n3;
        sq += (double)d * (double)d;
      } else {
        O[i] = v;
      }
    }
  }
  if (!Yt) return;
  __shared__ double sm[8];
  for (int s = 16; s > 0; s >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, s);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = sq;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < 8; ++k) t += sm[k];
    part[blockIdx.x] = t;
  }
}

// Sum of the output layer's block shares, in a fixed order.
__global__ void k_mp_sum(int n, const double* __restrict__ e, double* __restrict__ out) {
  __shared__ double sm[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += e[i];
  sm[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) sm[threadIdx.x] += sm[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sm[0];
}

__device__ __forceinline__ float4 add4(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

// Mb[b] = sum over the incidences of body b of H[contact], in the list's order;
// four rows are loaded ahead of their additions (28 -> 15 us on the 40^3 pile).
__global__ void __launch_bounds__(256)
    k_mp_bodysum(int M, const int* __restrict__ bptr, const int* __restrict__ inc, const float* __restrict__ H,
                 float* __restrict__ Mb) {
  const long long n = (long long)M * (MW / 4);
  const float4* H4 = reinterpret_cast<const float4*>(H);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int b = (int)(i >> 4), q = (int)(i & 15);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    const int e = __ldg(bptr + b + 1);
    for (int k = __ldg(bptr + b); k < e; k += 4) {
      float4 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        v[j] = k + j < e ? __ldg(H4 + 16 * (size_t)(__ldg(inc + k + j) >> 1) + q) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (k + j < e) s = add4(s, v[j]);
    }
    reinterpret_cast<float4*>(Mb)[i] = s;
  }
}

// s_c = Mb[a] (dynamic a) + Mb[b].  Forward (G null): S = s.  Backward: S is the
// layer's own input gradient, and the ReLU of the layer below is applied in the
// same pass: S = (S + s) where G > 0, else 0 (a separate pass cost 22 us a layer).
__global__ void __launch_bounds__(256)
    k_mp_gather(int Nc, int M, const int* __restrict__ ca, const int* __restrict__ cb, const float* __restrict__ Mb,
                float* __restrict__ S, const float* __restrict__ G) {
  const long long n = (long long)Nc * (MW / 4);
  const float4* M4 = reinterpret_cast<const float4*>(Mb);
  float4* S4 = reinterpret_cast<float4*>(S);
  const float4* G4 = reinterpret_cast<const float4*>(G);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i >> 4), q = (int)(i & 15);
    const int a = __ldg(ca + c), b = __ldg(cb + c);
    const float4 vb = __ldg(M4 + 16 * (size_t)b + q);
    const float4 va = a < M ? __ldg(M4 + 16 * (size_t)a + q) : make_float4(0.f, 0.f, 0.f, 0.f);
    float4 s = add4(va, vb);
    if (G) {
      const float4 g = __ldg(G4 + i);
      s = add4(S4[i], s);
      if (!(g.x > 0.f)) s.x = 0.f;
      if (!(g.y > 0.f)) s.y = 0.f;
      if (!(g.z > 0.f)) s.z = 0.f;
      if (!(g.w > 0.f)) s.w = 0.f;
    }
    S4[i] = s;
  }
}

__global__ void k_mp_adam(int n, float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                          const float* __restrict__ g, float lr, float b1, float b2, float eps, float c1, float c2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// gamma = out_scale * o moved into the cone's interior; lambda = -1/f; dummies 0
__global__ void k_mp_warm(int Nc, int slots, long long P, const float* __restrict__ O, double out_scale, double mu,
                          double gn_min, double shrink, double* __restrict__ gamma, double* __restrict__ lambda) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P; i += (long long)gridDim.x * blockDim.x) {
    const long long c = i / slots;
    const int u = (int)(i - c * slots);
    if (c >= Nc || u >= 3) {
      gamma[i] = 0.0;
      continue;
    }
    double gn = fmax(out_scale * (double)O[3 * c], gn_min);
    double t1 = out_scale * (double)O[3 * c + 1], t2 = out_scale * (double)O[3 * c + 2];
    const double nt = hypot(t1, t2), cap = shrink * mu * gn;
    if (nt > cap) {
      t1 *= cap / nt;
      t2 *= cap / nt;
    }
    gamma[i] = u == 0 ? gn : (u == 1 ? t1 : t2);
    if (u == 0) {
      lambda[c] = -1.0 / (0.5 * (t1 * t1 + t2 * t2 - mu * mu * gn * gn));
      lambda[Nc + c] = 1.0 / gn;
    }
  }
}

// ---------------------------------------------------------------- tensor-core rows GEMM
// OUT[r][n] = sum_k A[r][k] B[n][k] on the tensor cores (tcgen05, kind::tf32),
// 128 rows per tile, persistent blocks of 512 threads.  A is FP32, read by TMA
// from up to two row-major sources of 64 columns (kb0 blocks of 32 columns from
// the first, the rest from the second: the concatenation [h; s] of a layer);
// B comes from the BF16 weights, staged once per block as FP32 (exact in TF32).
// Products are FP32-accurate: A = A_hi + A_lo, A_hi = A with its 13 low mantissa
// bits cleared (exact in TF32), A_lo = A - A_hi (exact in FP32, within 2^-11 of
// its own size after the MMA's TF32 conversion), two MMAs per K step, so the
// error is about 2^-21 |A| |B| per term.  The accumulator (128 lanes x N FP32
// columns) lives in tensor memory; a warp reads 32 rows by 32 columns of it back and
// the tile goes through shared memory (A_lo's place, free by then; chunks of a row
// XORed with the row against bank conflicts) so that stores are whole rows.  The
// split of A and the way out are shared-memory traffic: with 512 threads a layer of
// the 40^3 pile takes 40 us forward and 37 backward; with 128, and stores of 16 bytes
// in each of 32 rows, 57 and 50.
// EPI 0: Y0[r][n] = relu(acc + bias[n]) (N = 64).  EPI 1: Y0[r][n] = acc for
// n < 64, Y1[r][n - 64] = acc for n >= 64 (N = 128).
constexpr long long TC_BUDGET = 2000000000LL;  // clock ticks (~1 s) per wait
constexpr int TC_THREADS = 512;

template <int N, int KB, int EPI>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_tc_rows(const __grid_constant__ CUtensorMap mA0, const __grid_constant__ CUtensorMap mA1, int kb0, int rows,
              const __nv_bfloat16* __restrict__ W, int ldw, int wtrans, const __nv_bfloat16* __restrict__ bias,
              float* __restrict__ Y0, float* __restrict__ Y1, int* __restrict__ err) {
  using namespace tc;
  constexpr int A_BLK = 128 * 128;  // bytes of a 128-row x 32-column block
  constexpr int B_BLK = N * 128;
  constexpr int A_BYTES = KB * A_BLK, B_BYTES = KB * B_BLK;
  // shared memory: B, two A stages (the next tile's copy overlaps this tile's work), A_lo or the output tile
  extern __shared__ __align__(1024) unsigned char tc_raw[];
  unsigned char* base = tc_raw + ((1024u - (smem_addr(tc_raw) & 1023u)) & 1023u);
  unsigned char* sB = base;
  unsigned char* const sA0 = base + B_BYTES;  // stage s at sA0 + s A_BYTES
  unsigned char* sL = base + B_BYTES + 2 * A_BYTES;
  __shared__ uint64_t bar_tma[2], bar_mma;
  __shared__ uint32_t tmem_base;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ntiles = (rows + 127) / 128;
  auto issue = [&](int t, int st) {  // thread 0: the A tile of row block t into stage st
    mbar_arrive_expect_tx(&bar_tma[st], A_BYTES);
    for (int j = 0; j < KB; ++j) {
      if (j < kb0) tma_load_2d(sA0 + st * A_BYTES + j * A_BLK, &mA0, &bar_tma[st], 32 * j, t * 128);
      else tma_load_2d(sA0 + st * A_BYTES + j * A_BLK, &mA1, &bar_tma[st], 32 * (j - kb0), t * 128);
    }
  };
  if (tid == 0) {
    mbar_init(&bar_tma[0], 1);
    mbar_init(&bar_tma[1], 1);
    mbar_init(&bar_mma, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(&tmem_base, N);
    tmem_relinquish();
  }
  // B(n, k) = W[n ldw + k] (or W[k ldw + n]) into the swizzled K-major layout
  for (int i = tid; i < N * KB * 32; i += blockDim.x) {
    const int n = i / (KB * 32), k = i - n * (KB * 32);
    const float w = __bfloat162float(wtrans ? W[(size_t)k * ldw + n] : W[(size_t)n * ldw + k]);
    const int kk = k & 31;
    *reinterpret_cast<float*>(sB + (k >> 5) * B_BLK + n * 128 + (((kk >> 2) ^ (n & 7)) << 4) + ((kk & 3) << 2)) = w;
  }
  fence_async_shared();
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  if (tid == 0 && (int)blockIdx.x < ntiles) issue(blockIdx.x, 0);
  const uint32_t tmem = tmem_base;
  constexpr uint32_t idesc = idesc_tf32(128, N);
  uint32_t ph_tma = 0u, ph_mma = 0u;  // bit s: parity of stage s's next phase
  int fail = 0;      // 1: a wait expired
  int inflight = 0;  // stages with a copy issued and not yet waited for (bit mask)
  if ((int)blockIdx.x < ntiles) inflight = 1;
  int st = 0;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x, st ^= 1) {
    const int r0 = t * 128;
    if (!mbar_wait(&bar_tma[st], (ph_tma >> st) & 1u, TC_BUDGET)) fail = 1;
    if (__syncthreads_or(fail)) {
      fail = 1;
      break;
    }
    ph_tma ^= 1u << st;
    inflight &= ~(1 << st);
    // the other stage is free (its tile's MMAs completed): start the next copy now
    const int tn = t + gridDim.x;
    if (tn < ntiles) {
      if (tid == 0) issue(tn, st ^ 1);
      inflight |= 1 << (st ^ 1);
    }
    // A_hi in place, A_lo beside it (same swizzled positions)
    float4* a4 = reinterpret_cast<float4*>(sA0 + st * A_BYTES);
    float4* l4 = reinterpret_cast<float4*>(sL);
    for (int i = tid; i < A_BYTES / 16; i += blockDim.x) {
      const float4 a = a4[i];
      float4 h;
      h.x = __uint_as_float(__float_as_uint(a.x) & 0xFFFFE000u);
      h.y = __uint_as_float(__float_as_uint(a.y) & 0xFFFFE000u);
      h.z = __uint_as_float(__float_as_uint(a.z) & 0xFFFFE000u);
      h.w = __uint_as_float(__float_as_uint(a.w) & 0xFFFFE000u);
      a4[i] = h;
      l4[i] = make_float4(a.x - h.x, a.y - h.y, a.z - h.z, a.w - h.w);
    }
    fence_async_shared();
    __syncthreads();
    if (tid == 0) {
      fence_after_sync();
      const uint32_t ah = smem_addr(sA0 + st * A_BYTES), al = smem_addr(sL), bb = smem_addr(sB);
      for (int kk = 0; kk < 4 * KB; ++kk) {
        const uint32_t ao = (kk >> 2) * A_BLK + (kk & 3) * 32, bo = (kk >> 2) * B_BLK + (kk & 3) * 32;
        const uint64_t bd = desc_k_sw128(bb + bo);
        mma_tf32(tmem, desc_k_sw128(ah + ao), bd, idesc, kk > 0 ? 1u : 0u);
        mma_tf32(tmem, desc_k_sw128(al + ao), bd, idesc, 1u);
      }
      mma_commit(&bar_mma);
    }
    if (!mbar_wait(&bar_mma, ph_mma, TC_BUDGET)) fail = 1;
    if (__syncthreads_or(fail)) {
      fail = 1;
      break;
    }
    ph_mma ^= 1u;
    fence_after_sync();
    const int row = (warp & 3) * 32 + lane;  // a warp reads the lanes 32 (warp mod 4) ..
    const int cb = (warp >> 2) * 32;         // and one block of 32 columns
    if (cb < N) {
      float v[32];
      tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)cb, v);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        float4 w = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        if constexpr (EPI == 0) {
          w.x = fmaxf(w.x + __bfloat162float(bias[cb + 4 * q]), 0.f);
          w.y = fmaxf(w.y + __bfloat162float(bias[cb + 4 * q + 1]), 0.f);
          w.z = fmaxf(w.z + __bfloat162float(bias[cb + 4 * q + 2]), 0.f);
          w.w = fmaxf(w.w + __bfloat162float(bias[cb + 4 * q + 3]), 0.f);
        }
        l4[row * (N / 4) + ((cb / 4 + q) ^ (row & 7))] = w;
      }
    }
    fence_before_sync();
    __syncthreads();
    for (int i = tid; i < 128 * (N / 4); i += TC_THREADS) {
      const int rr = i / (N / 4), q = i - rr * (N / 4);
      if (r0 + rr < rows) {
        const float4 w = l4[rr * (N / 4) + (q ^ (rr & 7))];
        float* dst = q < 16 ? Y0 : Y1;
        reinterpret_cast<float4*>(dst)[16 * (size_t)(r0 + rr) + (q & 15)] = w;
      }
    }
    fence_before_sync();
    __syncthreads();
  }
  if (fail) {
    // let copies and MMAs of the failed step finish (bounded) before the
    // block's shared and tensor memory go away
    for (int k = 0; k < 2; ++k)
      if (inflight & (1 << k)) mbar_wait(&bar_tma[k], (ph_tma >> k) & 1u, TC_BUDGET);
    mbar_wait(&bar_mma, ph_mma, TC_BUDGET);
    if (tid == 0) atomicExch(err, 1);
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  if (warp == 0) tmem_dealloc(tmem, N);
}

// Weight gradients in two deterministic passes: block g sums its rows (at most
// WG_CHUNK of them, in FP32) into part[g][j (K + 1) + k] = sum_c dZ[c][j] X[c][k]
// (k < K) and sum_c dZ[c][j] (k = K); then the partials are added in block order
// in FP64.
constexpr int WG_CHUNK = 256;

__device__ __forceinline__ unsigned long long dup2(float v) {
  unsigned long long d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(v));
  return d;
}
__device__ __forceinline__ float lo2(unsigned long long v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float hi2(unsigned long long v) { return __uint_as_float((unsigned)(v >> 32)); }

// Hidden layers (J = 64, X = [Xa | Xb] of 64 columns each): bound by FP32
// arithmetic and the shared-memory loads that feed it.  A thread owns 8 x 8 of the
// 64 x 128 outputs, so a row costs it four float4 loads for 32 packed FMAs; the next
// 32 rows arrive by asynchronous copies meanwhile.  On the 40^3 pile (191 806 rows)
// 64 us a layer, 62 % of the FP32 rate; one output a thread took 515 us, and a 4 x 8
// tile with dZ stored as pairs, bound by the shared loads, 94 us.
constexpr int WG_R = 32;
constexpr int WG_SMEM = 2 * WG_R * 3 * MW * 4;  // two stages of dZ and X rows

__device__ __forceinline__ void cp16(void* dst, const void* src, bool in) {  // 16 bytes, zeros when !in
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc::smem_addr(dst)), "l"(src), "r"(in ? 16 : 0)
               : "memory");
}

__global__ void __launch_bounds__(128)
    k_wgrad_hidden(int Nc, int per, const float* __restrict__ dZ, const float* __restrict__ Xa,
                   const float* __restrict__ Xb, float* __restrict__ part) {
  extern __shared__ __align__(16) float wg_sm[];  // [2][WG_R][dZ 64 | Xa 64 | Xb 64]
  __shared__ float sb[2][MW];
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int c0 = blockIdx.x * per, c1 = min(Nc, c0 + per);
  unsigned long long acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
  auto fetch = [&](int r0, int st) {  // 128 threads: column group tx of rows ty, ty + 8, ..
    for (int rr = ty; rr < WG_R; rr += 8) {
      const int r = r0 + rr;
      const bool in = r < c1;
      const size_t o = (in ? (size_t)r : (size_t)c0) * MW + 4 * tx;
      float* d = wg_sm + ((size_t)st * WG_R + rr) * 3 * MW + 4 * tx;
      cp16(d, dZ + o, in);
      cp16(d + MW, Xa + o, in);
      cp16(d + 2 * MW, Xb + o, in);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float bias = 0.f;
  fetch(c0, 0);
  int st = 0;
  for (int r0 = c0; r0 < c1; r0 += WG_R, st ^= 1) {
    if (r0 + WG_R < c1) {
      fetch(r0 + WG_R, st ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const float* sm = wg_sm + (size_t)st * WG_R * 3 * MW;
    for (int r = (t >> 6) * (WG_R / 2), e = r + WG_R / 2; r < e; ++r) bias += sm[r * 3 * MW + (t & 63)];
#pragma unroll 2
    for (int r = 0; r < WG_R; ++r) {
      const float* row = sm + r * 3 * MW;
      const float4 z0 = *reinterpret_cast<const float4*>(row + 8 * ty);
      const float4 z1 = *reinterpret_cast<const float4*>(row + 8 * ty + 4);
      const ulonglong2 x0 = *reinterpret_cast<const ulonglong2*>(row + MW + 4 * tx);
      const ulonglong2 x1 = *reinterpret_cast<const ulonglong2*>(row + 2 * MW + 4 * tx);
      const float z[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
      const unsigned long long x[4] = {x0.x, x0.y, x1.x, x1.y};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const unsigned long long zz = dup2(z[i]);
#pragma unroll
        for (int j = 0; j < 4; ++j) fma2(acc[i][j], zz, x[j]);
      }
    }
    __syncthreads();
  }
  constexpr int K = 2 * MW;
  float* out = part + (size_t)blockIdx.x * MW * (K + 1);
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float* o = out + (8 * ty + i) * (K + 1) + (j < 2 ? 0 : MW) + 4 * tx + 2 * (j & 1);
      o[0] = lo2(acc[i][j]);
      o[1] = hi2(acc[i][j]);
    }
  sb[t >> 6][t & 63] = bias;
  __syncthreads();
  if (t < MW) out[t * (K + 1) + K] = sb[0][t] + sb[1][t];
}

// Output layer (J = 3, K = 64) together with its input gradient: dH3 = Wo^T dO
// where h3 > 0, else 0.  Bound by reading h3 and writing dH3 once (18 us on the 40^3
// pile, 79 + 45 + 22 as three passes): 16 lanes a row, four columns a lane, four rows in flight.
__global__ void __launch_bounds__(256)
    k_wgrad_output(int Nc, int per, const float* __restrict__ dO, const float* __restrict__ H,
                   const __nv_bfloat16* __restrict__ Wo, float* __restrict__ dH, float* __restrict__ part) {
  __shared__ float sm[16][MO][MW + 1];  // [.][.][MW]: the bias
  const int q = threadIdx.x & 15, g = threadIdx.x >> 4;
  const int c0 = blockIdx.x * per, c1 = min(Nc, c0 + per);
  float w[MO][4], a[MO][4] = {}, b[MO] = {};
#pragma unroll
  for (int j = 0; j < MO; ++j)
#pragma unroll
    for (int k = 0; k < 4; ++k) w[j][k] = pb(Wo, j * MW + 4 * q + k);
#pragma unroll 4
  for (int r = c0 + g; r < c1; r += 16) {
    const float4 h = __ldg(reinterpret_cast<const float4*>(H) + 16 * (size_t)r + q);
    const float hk[4] = {h.x, h.y, h.z, h.w};
    float d[MO], o[4];
#pragma unroll
    for (int j = 0; j < MO; ++j) {
      d[j] = __ldg(dO + 3 * (size_t)r + j);
      b[j] += d[j];
#pragma unroll
      for (int k = 0; k < 4; ++k) a[j][k] = fmaf(d[j], hk[k], a[j][k]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] = hk[k] > 0.f ? fmaf(w[2][k], d[2], fmaf(w[1][k], d[1], w[0][k] * d[0])) : 0.f;
    reinterpret_cast<float4*>(dH)[16 * (size_t)r + q] = make_float4(o[0], o[1], o[2], o[3]);
  }
  for (int j = 0; j < MO; ++j) {
    for (int k = 0; k < 4; ++k) sm[g][j][4 * q + k] = a[j][k];
    if (q == 0) sm[g][j][MW] = b[j];
  }
  __syncthreads();
  float* out = part + (size_t)blockIdx.x * MO * (MW + 1);
  for (int o = threadIdx.x; o < MO * (MW + 1); o += blockDim.x) {
    const int j = o / (MW + 1), k = o - j * (MW + 1);
    float v = 0.f;
    for (int u = 0; u < 16; ++u) v += sm[u][j][k];
    out[o] = v;
  }
}

// Input layer (J = 64, K = 8): bound by reading dZ once (62 -> 23 us); 16 lanes a
// row, four columns of dZ a lane against the row's eight features.
__global__ void __launch_bounds__(256)
    k_wgrad_input(int Nc, int per, const float* __restrict__ dZ, const float* __restrict__ X,
                  float* __restrict__ part) {
  __shared__ float sm[16][MW * (MF + 1)];
  const int q = threadIdx.x & 15, g = threadIdx.x >> 4;
  const int c0 = blockIdx.x * per, c1 = min(Nc, c0 + per);
  float a[4][MF + 1] = {};
#pragma unroll 4
  for (int r = c0 + g; r < c1; r += 16) {
    const float4 z4 = __ldg(reinterpret_cast<const float4*>(dZ) + 16 * (size_t)r + q);
    const float4 x0 = __ldg(reinterpret_cast<const float4*>(X) + 2 * (size_t)r);
    const float4 x1 = __ldg(reinterpret_cast<const float4*>(X) + 2 * (size_t)r + 1);
    const float z[4] = {z4.x, z4.y, z4.z, z4.w};
    const float x[MF] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int k = 0; k < MF; ++k) a[j][k] = fmaf(z[j], x[k], a[j][k]);
      a[j][MF] += z[j];
    }
  }
  for (int j = 0; j < 4; ++j)
    for (int k = 0; k <= MF; ++k) sm[g][(4 * q + j) * (MF + 1) + k] = a[j][k];
  __syncthreads();
  float* out = part + (size_t)blockIdx.x * MW * (MF + 1);
  for (int o = threadIdx.x; o < MW * (MF + 1); o += blockDim.x) {
    float v = 0.f;
    for (int u = 0; u < 16; ++u) v += sm[u][o];
    out[o] = v;
  }
}

// (hi, lo) += v with the rounding error kept (Knuth's TwoSum); lo is NaN from the first
// hi on that is not finite
__device__ __forceinline__ void fold(float& hi, float& lo, float v) {
  const float t = __fadd_rn(hi, v), z = __fsub_rn(t, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(v, z)));
  hi = t;
}

// gW[j K + k] = sum_g part[g][j (K+1) + k], gb[j] = sum_g part[g][j (K+1) + K]:
// a block takes 32 outputs, its 32 warps a share of the partials each, added in
// warp order in FP64.  A warp's share is summed in FP32 with the rounding errors kept:
// converting and adding the 7 M partials of a layer on the FP64 pipe takes 22 us by
// itself, and a third term (70 bits) changes no gradient but takes 14 us over the five
// sums.  A share with an infinite partial, or whose running sum leaves FP32's range, is
// summed again in FP64.  12 us on average; a thread an output, its partials one after the
// other, took 127.
__global__ void __launch_bounds__(1024)
    k_wgrad_sum(int nparts, int J, int K, const float* __restrict__ part, float* __restrict__ gW,
                float* __restrict__ gb) {
  __shared__ double sm[32][33];
  const int n = J * (K + 1), lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int o = blockIdx.x * 32 + lane;
  const int g0 = (int)((long long)nparts * w / 32), g1 = (int)((long long)nparts * (w + 1) / 32);
  double share = 0.0;
  if (o < n) {
    float hi = 0.f, lo = 0.f;
#pragma unroll 8
    for (int g = g0; g < g1; ++g) fold(hi, lo, __ldg(part + (size_t)g * n + o));
    if (lo == lo) {
      share = (double)hi + (double)lo;
    } else {
      for (int g = g0; g < g1; ++g) share += (double)__ldg(part + (size_t)g * n + o);
    }
  }
  sm[w][lane] = share;
  __syncthreads();
  if (w == 0 && o < n) {
    double s = 0.0;
    for (int q = 0; q < 32; ++q) s += sm[q][lane];
    const int j = o / (K + 1), k = o - j * (K + 1);
    if (k == K) gb[j] = (float)s;
    else gW[j * K + k] = (float)s;
  }
}

inline int blocks_for(long long n, int per = 256, int cap = 152 * 32) {
  long long b = (n + per - 1) / per;
  if (b > cap) b = cap;
  return (int)(b < 1 ? 1 : b);
}

// ---- host side of the tensor-core GEMM

// Row-major FP32 matrix [rows][64], boxes of 128 rows x 32 columns (128 bytes
// wide, the 128-byte swizzle); rows past the end read as zeros.
CUtensorMap rows64_map(const float* base, int rows) {
  QP_REQUIRE((reinterpret_cast<uintptr_t>(base) & 15u) == 0, QP_CUDA_ERROR, "tensor map base not 16-byte aligned");
  CUtensorMap m;
  const cuuint64_t gdim[2] = {64, (cuuint64_t)rows};
  const cuuint64_t gstride[1] = {64 * sizeof(float)};
  const cuuint32_t box[2] = {32, 128};
  const cuuint32_t es[2] = {1, 1};
  const CUresult r = tmap_encoder()(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), gdim, gstride,
                                    box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  QP_REQUIRE(r == CUDA_SUCCESS, QP_CUDA_ERROR, "cuTensorMapEncodeTiled failed");
  return m;
}

int* tc_flag(qp_ctx* c) {
  char* p = static_cast<char*>(c->mp_sum.ensure(64));
  return reinterpret_cast<int*>(p + 32);
}

template <int N, int KB, int EPI>
void launch_tc_rows(qp_ctx* c, const float* A0, const float* A1, int kb0, int rows, const __nv_bfloat16* W, int ldw,
                    int wtrans, const __nv_bfloat16* bias, float* Y0, float* Y1) {
  if (rows <= 0) return;
  const CUtensorMap m0 = rows64_map(A0, rows);
  const CUtensorMap m1 = rows64_map(A1 ? A1 : A0, rows);
  auto k = k_tc_rows<N, KB, EPI>;
  // B, two A stages, A_lo (or the tile on its way out), alignment
  const int smem = KB * N * 128 + 2 * KB * 128 * 128 + std::max(KB * 128 * 128, 128 * N * 4) + 1024;
  QP_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  const int grid = std::min((rows + 127) / 128, c->num_sms);
  k<<<grid, TC_THREADS, smem, c->stream>>>(m0, m1, kb0, rows, W, ldw, wtrans, bias, Y0, Y1, tc_flag(c));
  QP_CUDA(cudaGetLastError());
}

// Rows of one block of the weight-gradient kernels: at most WG_CHUNK, a multiple of
// WG_R, and such that the blocks fill whole waves of four an SM where there are
// enough rows (191 806 contacts: 160 rows, 1199 blocks on 608 places).
struct WgradPlan {
  int per, nparts;
};
WgradPlan wgrad_plan(const qp_ctx* c) {
  const int slots = 4 * c->num_sms;
  const int waves = std::max(1, ceil_div(c->Nc, (long long)slots * WG_CHUNK));
  const int per = std::max(2, ceil_div(ceil_div(c->Nc, (long long)slots * waves), WG_R)) * WG_R;
  return WgradPlan{per, ceil_div(c->Nc, per)};
}

void wgrad_sum(qp_ctx* c, const WgradPlan& w, int J, int K, const float* part, float* gW, float* gb) {
  k_wgrad_sum<<<(J * (K + 1) + 31) / 32, 1024, 0, c->stream>>>(w.nparts, J, K, part, gW, gb);
  QP_CUDA(cudaGetLastError());
}

void check_tc_flag(qp_ctx* c) {
  int h = 0;
  QP_CUDA(cudaMemcpyAsync(&h, tc_flag(c), sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  QP_CUDA(cudaStreamSynchronize(c->stream));
  QP_REQUIRE(h == 0, QP_TIMEOUT, "tensor-core GEMM: a wait expired");
}

struct Net {
  float* X0;
  float* H[ML + 1];
  float* S[ML];
  float* Mb;
  __nv_bfloat16* pw;
};

// workspace: activations of one pass (kept for the backward pass) + scratch
Net workspace(qp_ctx* c) {
  const size_t Nc = (size_t)(c->Nc > 0 ? c->Nc : 1), M = (size_t)(c->M > 0 ? c->M : 1);
  const size_t nf = Nc * MF + (ML + 1) * Nc * MW + ML * Nc * MW + M * MW + 64;
  float* w = static_cast<float*>(c->mp_act.ensure(nf * sizeof(float)));
  Net n;
  n.X0 = w;
  w += Nc * MF;
  for (int l = 0; l <= ML; ++l, w += Nc * MW) n.H[l] = w;
  for (int l = 0; l < ML; ++l, w += Nc * MW) n.S[l] = w;
  n.Mb = w;
  n.pw = static_cast<__nv_bfloat16*>(c->mp_w.ensure((size_t)NPAR * sizeof(__nv_bfloat16)));
  return n;
}

// Blocks of the output layer's pass (and FP64 loss shares).
int output_blocks(const qp_ctx* c) { return blocks_for(16LL * c->Nc, 256, 8 * c->num_sms); }

// The passes up to h3; with `out` also the outputs.
void forward(qp_ctx* c, const float* params, const float* scale_host, float* out, Net& n) {
  cudaStream_t st = c->stream;
  QP_CUDA(cudaMemsetAsync(tc_flag(c), 0, sizeof(int), st));
  const int Nc = c->Nc, M = c->M;
  k_mp_round<<<blocks_for(NPAR), 256, 0, st>>>(params, n.pw, NPAR);
  Scale sc;
  for (int k = 0; k < MF; ++k) sc.s[k] = scale_host[k];
  if (Nc > 0) {
    k_mp_input<<<blocks_for(Nc, 256, 8 * c->num_sms), 256, 0, st>>>(Nc, c->slots, c->phi.as<double>(), c->frame.as<double>(), c->r.as<double>(),
                                          c->dt, c->mu, sc, n.pw + OFF_W0, n.pw + OFF_B0, n.X0, n.H[0]);
    for (int l = 0; l < ML; ++l) {
      k_mp_bodysum<<<blocks_for((long long)M * MW / 4), 256, 0, st>>>(M, c->bptr.as<int>(), c->inc.as<int>(), n.H[l],
                                                                      n.Mb);
      k_mp_gather<<<blocks_for((long long)Nc * MW / 4), 256, 0, st>>>(Nc, M, c->ca.as<int>(), c->cb.as<int>(), n.Mb,
                                                                      n.S[l], nullptr);
      const __nv_bfloat16* W = n.pw + OFF_L + l * LAYER;
      // H[l+1] = relu(W [H[l]; S[l]] + b): Nc x 128 by 128 x 64 on the tensor cores
      launch_tc_rows<MW, 4, 0>(c, n.H[l], n.S[l], 2, Nc, W, 2 * MW, 0, W + MW * 2 * MW, n.H[l + 1], nullptr);
    }
    if (out)
      k_mp_output<<<output_blocks(c), 256, 0, st>>>(Nc, n.H[ML], n.pw + OFF_WO, n.pw + OFF_BO, out, nullptr, nullptr,
                                                    nullptr);
  }
  QP_CUDA(cudaGetLastError());
}

}  // namespace
}  // namespace qp

using namespace qp;

#define MP_BEGIN(c)               \
  if (!(c)) return QP_INVALID_ARG; \
  try {                           \
    QP_CUDA(cudaSetDevice((c)->device));
#define MP_END(c)                 \
  }                               \
  catch (const Error& e) {        \
    set_error((c), e);            \
    return e.code;                \
  }                               \
  return QP_OK;

extern "C" {

int mpnn_forward(qp_ctx_t c, const float* params, const float* feat_scale, float* out) {
  MP_BEGIN(c)
  QP_REQUIRE(c->have_contacts, QP_NOT_READY, "mpnn_forward: call ccp_assemble first");
  QP_REQUIRE(params && feat_scale && (out || c->Nc == 0), QP_INVALID_ARG, "mpnn_forward: null argument");
  Net n = workspace(c);
  forward(c, params, feat_scale, out, n);
  check_tc_flag(c);
  MP_END(c)
}

int mpnn_grad(qp_ctx_t c, const float* params, const float* feat_scale, const float* target, float* grad,
              double* loss) {
  MP_BEGIN(c)
  QP_REQUIRE(c->have_contacts, QP_NOT_READY, "mpnn_grad: call ccp_assemble first");
  QP_REQUIRE(params && feat_scale && grad && target, QP_INVALID_ARG, "mpnn_grad: null argument");
  QP_REQUIRE(c->Nc > 0, QP_INVALID_ARG, "mpnn_grad: no contacts to fit");
  QP_REQUIRE(grad != params, QP_INVALID_ARG, "mpnn_grad: grad aliases params");
  Net n = workspace(c);
  const int Nc = c->Nc, M = c->M;
  cudaStream_t st = c->stream;
  forward(c, params, feat_scale, nullptr, n);
  // scratch: the loss shares, dO [3Nc], three [Nc][64] buffers, the partial gradients
  // (every buffer starts on a 256-byte boundary: the tensor-core GEMM reads A by TMA)
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const WgradPlan wp = wgrad_plan(c);
  const size_t o_dO = up((size_t)output_blocks(c) * sizeof(double)), o_A = o_dO + up((size_t)3 * Nc * sizeof(float));
  const size_t o_B = o_A + up((size_t)Nc * MW * 4), o_C = o_B + up((size_t)Nc * MW * 4);
  const size_t o_P = o_C + up((size_t)Nc * MW * 4);
  const size_t nb = o_P + (size_t)wp.nparts * MW * (2 * MW + 1) * sizeof(float);
  char* s = static_cast<char*>(c->mp_grad.ensure(nb));
  double* err = reinterpret_cast<double*>(s);
  float* dO = reinterpret_cast<float*>(s + o_dO);
  float* A = reinterpret_cast<float*>(s + o_A);
  float* B = reinterpret_cast<float*>(s + o_B);
  float* Cs = reinterpret_cast<float*>(s + o_C);
  float* part = reinterpret_cast<float*>(s + o_P);
  float* dM = n.Mb;  // the forward pass is done with it
  double* lsum = static_cast<double*>(c->mp_sum.ensure(64));  // the GEMM flag shares this buffer
  const long long nh = (long long)Nc * MW;
  k_mp_output<<<output_blocks(c), 256, 0, st>>>(Nc, n.H[ML], n.pw + OFF_WO, n.pw + OFF_BO, nullptr, target, dO, err);
  k_mp_sum<<<1, 256, 0, st>>>(output_blocks(c), err, lsum);
  // head: o = Wo h3 + bo; A = d/dh3 with the last layer's ReLU applied
  k_wgrad_output<<<wp.nparts, 256, 0, st>>>(Nc, wp.per, dO, n.H[ML], n.pw + OFF_WO, A, part);
  wgrad_sum(c, wp, MO, MW, part, grad + OFF_WO, grad + OFF_BO);
  QP_CUDA(cudaFuncSetAttribute(k_wgrad_hidden, cudaFuncAttributeMaxDynamicSharedMemorySize, WG_SMEM));
  for (int l = ML - 1; l >= 0; --l) {
    // layer l: H[l+1] = relu(W [H[l]; S[l]] + b); A holds d/dz of its sums
    const __nv_bfloat16* W = n.pw + OFF_L + l * LAYER;
    float* gW = grad + OFF_L + l * LAYER;
    k_wgrad_hidden<<<wp.nparts, 128, WG_SMEM, st>>>(Nc, wp.per, A, n.H[l], n.S[l], part);
    wgrad_sum(c, wp, MW, 2 * MW, part, gW, gW + MW * 2 * MW);
    // [dH[l], dS[l]] = dZ W: Nc x 64 by 64 x 128 on the tensor cores (B(n, j) = W[j][n])
    launch_tc_rows<2 * MW, 2, 1>(c, A, nullptr, 2, Nc, W, 2 * MW, 1, nullptr, B, Cs);
    // S[l] = gather(bodysum(H[l])): its adjoint is the same pair of sums; then H[l]'s own ReLU
    k_mp_bodysum<<<blocks_for((long long)M * MW / 4), 256, 0, st>>>(M, c->bptr.as<int>(), c->inc.as<int>(), Cs, dM);
    k_mp_gather<<<blocks_for(nh / 4), 256, 0, st>>>(Nc, M, c->ca.as<int>(), c->cb.as<int>(), dM, B, n.H[l]);
    float* t = A;
    A = B;
    B = t;
  }
  // input layer: H[0] = relu(W0 X0 + b0)
  k_wgrad_input<<<wp.nparts, 256, 0, st>>>(Nc, wp.per, A, n.X0, part);
  wgrad_sum(c, wp, MW, MF, part, grad + OFF_W0, grad + OFF_B0);
  QP_CUDA(cudaGetLastError());
  check_tc_flag(c);
  if (loss) {
    double h = 0.0;
    QP_CUDA(cudaMemcpyAsync(&h, lsum, sizeof(double), cudaMemcpyDeviceToHost, st));
    QP_CUDA(cudaStreamSynchronize(st));
    *loss = h / (3.0 * Nc);
  }
  MP_END(c)
}

int mpnn_adam(qp_ctx_t c, float* params, float* m, float* v, const float* grad, int step, double lr, double beta1,
              double beta2, double eps) {
  MP_BEGIN(c)
  QP_REQUIRE(params && m && v && grad && step >= 1 && lr > 0 && beta1 >= 0 && beta1 < 1 && beta2 >= 0 && beta2 < 1 &&
                 eps > 0,
             QP_INVALID_ARG, "mpnn_adam: bad argument");
  const float c1 = (float)(1.0 - pow(beta1, step)), c2 = (float)(1.0 - pow(beta2, step));
  k_mp_adam<<<blocks_for(NPAR), 256, 0, c->stream>>>(NPAR, params, m, v, grad, (float)lr, (float)beta1, (float)beta2,
                                                     (float)eps, c1, c2);
  QP_CUDA(cudaGetLastError());
  MP_END(c)
}

int mpnn_warm_start(qp_ctx_t c, qp_state* st, const float* out, double out_scale, double gn_min, double shrink) {
  MP_BEGIN(c)
  QP_REQUIRE(c->have_contacts, QP_NOT_READY, "mpnn_warm_start: call ccp_assemble first");
  QP_REQUIRE(st && st->gamma && st->lambda && (out || c->Nc == 0), QP_INVALID_ARG, "mpnn_warm_start: null argument");
  QP_REQUIRE(out_scale > 0 && gn_min > 0 && shrink > 0 && shrink <= 1, QP_INVALID_ARG,
             "mpnn_warm_start: need out_scale > 0, gn_min > 0, 0 < shrink <= 1");
  k_mp_warm<<<blocks_for(c->P), 256, 0, c->stream>>>(c->Nc, c->slots, c->P, out, out_scale, c->mu, gn_min, shrink,
                                                     st->gamma, st->lambda);
  QP_CUDA(cudaGetLastError());
  st->t = 1.0;
  MP_END(c)
}

}  // extern "C"
