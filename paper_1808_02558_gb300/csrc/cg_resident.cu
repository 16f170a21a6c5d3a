// Jacobi-preconditioned CG on S = N + blockdiag(H_c) with the whole system held in
// registers and shared memory (Sec. 2.4's Newton systems, Eq. Ndef).
//
// Block g owns a contiguous run of the Morton-ordered contacts; their frames, arms,
// blocks H_c, Jacobi diagonal and the rows of r, p and e stay on its SM for the whole
// solve, and so do the lists of the bodies they touch.  Per iteration only the
// partial sums of bodies shared with other blocks (about 350 of 610 a block on the
// 40^3 pile) and seven sums leave an SM.
//
// What bounds it: latency.  Of 18 800 cycles an iteration of the 40^3 pile takes (1262
// contacts a block, mixed; clock stamps of one block), the exchange between neighbouring
// blocks has 4700 and the sum over all blocks 5400, each with the wait for slower blocks
// (a store and a load through L2 alone are 2400), and the body sums 6400, shared-memory
// traffic: a block's own 3900, its border's 2500.  The 8^3 pile in FP64 takes 17 700: 3700,
// 6800 and 3700, and the 64-cycle latency of the FP64 pipe in all of them.  The classic
// persistent kernel (three grid barriers and about 45 MB through L2 an iteration) remains
// for systems that do not fit, for other preconditioners and for BiCGSTAB.
//
//   p = z + beta p
//   contact wrenches D_c p_c into shared memory; a body sums its own; the partial
//   sums of shared bodies go to the other blocks and come back        -- exchange
//   q = S p; r.z, p.q, z.q, q.Dq, r.r, r.q, q.q                       -- one sum
//   alpha = r.z / p.q;  e += alpha p;  r -= alpha q
//   beta = (r.z)' / r.z with (r.z)' = r.z - 2 alpha z.q + alpha^2 q.Dq
//
// That is classic CG: only beta and the two stopping tests use a recurrence for the
// new sums (from this iteration's true ones); alpha uses r.z summed afresh.
//
// A sphere's arms are along the normal, rho = s n, so the iteration keeps s_a and s_b
// instead of the six components: n x f = x1 t2 - x2 t1 for f = U x, and
// t1 . (w x n) = w . t2, t2 . (w x n) = -w . t1.  The FP64 residual uses the stored
// arms.
//
// Exchanges carry their own flags: each 64-bit word is 32 bits of the value and a
// 32-bit tag that grows by one from exchange to exchange and from solve to solve, so
// a reader polls the data itself and no memory fence, counter or barrier is needed.
// Slots alternate between two buffers: a block writes exchange k + 2 only after the
// sum that follows exchange k + 1, for which every block has read exchange k.
// Every wait is bounded (QP_TIMEOUT).
//
// Measured, newton_rhs + newton_solve to 1e-12, against the classic kernel: the 40^3 pile
// in mixed precision 2.57 -> 1.44 ms (105 iterations of 9.1 us in place of 19, and four
// FP64 residuals of 57 us), the 8^3 pile in FP64 2.07 -> 0.87 ms (91 iterations of 8.4 us
// in place of 22).  The pipelined kernel that mid-size systems used (one grid barrier,
// records through L2, 15 us an iteration on 57 000 contacts, 5.6 here) takes 1.4 to 2
// times as long as this and is gone.
#include <algorithm>

#include "internal.cuh"

namespace qp {
namespace {

typedef unsigned long long u64;

constexpr int CR_MAXG = 256;                   // blocks at most
constexpr int CR_HALO = 12;                    // tagged words a partial sum (six FP64 values)
constexpr int CR_RED = 16 * CR_MAXG;           // tagged words of one sum buffer (eight FP64 values a block)
constexpr int CR_MINT = 256;                   // threads of a block at least

// The plan of one contact set: what each block's SM holds and sends, made once per
// assembly (k_cgr_lists, k_cgr_dest) and copied into shared memory by every solve.
struct CgrPlan {
  int chunk;              // contacts a block
  int nbcap, rcap;        // bodies and shared runs a block has room for
  int* head;              // [G][4] shared bodies, own bodies, shared runs, (block 0: set when some block had no room)
  unsigned* bmeta;        // [G][nbcap] first code | codes << 16; shared bodies from the front, own ones from the end
  int* bid;               // [G][nbcap] global body
  unsigned* rmeta;        // [G][nbcap] first entry of rsum | other blocks' runs << 16 | own position among them << 24
  unsigned short* rsum;   // [G][rcap] by body, in block order: place of a run's partial sum in the inbox
  unsigned short* sbody;  // [G][rcap] outgoing partial sums, by (other block, body): the local body
  int* sdest;             // [G][rcap] their places in the other blocks' inboxes
  unsigned short* codes;  // [G][2 chunk] local contact << 1 | side, by body
  unsigned short* lidx;   // [G][2 chunk] local body of a contact's side (0xFFFF: static)
  int* seg;               // [G][G] first entry of block g for block h
};

struct CgrArgs {
  SysView<double> s64;
  SysView<float> s32;
  CgrPlan pl;
  int chunk;             // contacts a block
  int own_rb;            // remote partials have shared memory of their own
  int nbcap, rcap;       // bodies and remote partials a block has room for
  const double* rhs;     // [P]
  double* x;             // [P]
  const double* dinv64;  // [P]
  const float* dinv32;
  double tol, inner_tol;
  int maxit, max_outer;
  unsigned epoch;        // first tag of this solve
  unsigned polls;        // unsuccessful polls after which a wait expires
  int absent;            // self-test: block that leaves (-1: none) ...
  int absent_at;         // ... before the first sum (0) or the first exchange (1)
  double* r64;           // [P] FP64 residual
  double* xbest;         // [P] the x of the smallest true residual so far
  u64* halo;             // [2][G][CR_HALO / 2][rcap][2] inboxes, pairs of words by place
  u64* red;              // [2][CR_RED]
  DevCtl* ctl;
};

__device__ __forceinline__ void st_word(u64* p, u64 v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void ld_words2(const u64* p, u64& a, u64& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_words2(u64* p, u64 a, u64 b) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ u64 word(unsigned bits, unsigned tag) { return ((u64)tag << 32) | bits; }
__device__ __forceinline__ unsigned tag_of(u64 w) { return (unsigned)(w >> 32); }

// One more unsuccessful poll (each takes an L2 round trip, at least 400 cycles); true:
// leave, because the wait expired or another block failed.
__device__ __forceinline__ bool give_up(DevCtl* ctl, unsigned& spins, unsigned polls) {
  return ++spins > polls || ((spins & 1023u) == 0 && *(volatile int*)&ctl->err != 0);
}

// Sums of eight values over a warp by halving: lane l ends with the total of value
// (l >> 2).  Nine additions instead of forty -- an FP64 addition holds the SM's
// narrow FP64 pipe for 16 cycles a warp and takes 64.
template <class T>
__device__ __forceinline__ T wsum8(const T (&v)[8]) {
  const int lane = threadIdx.x & 31;
  T a[4], b[2], c;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const T keep = (lane & 16) ? v[4 + i] : v[i], send = (lane & 16) ? v[i] : v[4 + i];
    a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const T keep = (lane & 8) ? a[2 + i] : a[i], send = (lane & 8) ? a[i] : a[2 + i];
    b[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
  c = ((lane & 4) ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, (lane & 4) ? b[0] : b[1], 4);
  c += __shfl_xor_sync(0xffffffffu, c, 2);
  return c + __shfl_xor_sync(0xffffffffu, c, 1);
}

// What a residual replacement finds: the tolerance is met; a cap is, at the smallest
// residual so far or after a smaller one; neither, at the smallest so far or not.
enum { R_DONE, R_CAP, R_CAP_BACK, R_KEEP, R_GO };

// Shared-memory state of a block beside the dynamic arrays.
struct CgrShared {
  double part[32][8];            // per warp: sums over its threads
  double poll[32][8];           // per warp: sums over its share of the blocks' messages
  double scal[8];                // what the sum's last step hands to the block
  int flag[2];
  // what only a replacement uses (in registers it would be spilled around the iterations)
  double bnorm, scale;           // ||rhs||, and r's unit
  double rz;                     // r.z of the iteration before
  double rel;                    // true relative residual
  double best;                   // smallest true residual norm so far
  int kept;                      // its x is in A.xbest (else it is 0)
  double inv, beta, due;         // r's new scaling, the next beta, the next due r.r
  int next;                      // R_*: what a replacement found
  double keep2;                  // squared growth of the residual up to which the direction is kept
  // the block's lists (CgrPlan's, in shared memory)
  int c0, c1, chunk, nbcap, rcap, nbord, nint, nrem;
  unsigned polls;         // CgrArgs::polls
  double* wr;             // [chunk][CR_WR] wrenches of the block's contacts (viewed as T)
  double* wl;             // [nbcap][CR_WL] body intermediates (viewed as T)
  double* bw;             // [nbcap][2] 1/m, 1/I of the bodies (viewed as T)
  double* rb;             // [rcap][CR_WL] the other blocks' partial sums (viewed as T)
  unsigned* bmeta;
  int* bid;
  unsigned* rmeta;
  int* sdest;
  unsigned short* codes;
  unsigned short* lidx;
  unsigned short* rsum;
  unsigned short* sbody;
};

// Exchanges and sums so far (the same in every thread of every block).
struct CgrCount {
  unsigned xc, rc;
};

// Sums of up to eight values over all threads of all blocks, bit-identical everywhere
// (fixed trees, blocks in order).  A block's message is 64 bytes (FP64: 128) that
// every block polls: 2400 cycles for a store and a load through L2, 5400 with the sums on
// both sides and the wait for slower blocks (slots by value instead, 16 blocks' words in
// a line, took 10600 for seven values).
//
// sum_gather, from the warps' partial sums on: the total of value (lane >> 2) in
// every lane of warp 0; ok = false when a wait expired.  Inlined into the iteration:
// a call would put the contacts' registers on the stack, which does not fit the L1
// left beside this much shared memory.  The cold callers share one copy
// (all_sum_cold), and nothing here is unrolled without need: an iteration's code has
// to stay in the instruction cache.
template <class T>
struct Summed {
  T x;
  bool ok;
};
template <class T>
__device__ __forceinline__ Summed<T> sum_gather(CgrShared& sh, u64* buf, DevCtl* ctl, unsigned tag, int nwork) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, G = gridDim.x;
  const T* part = reinterpret_cast<const T*>(&sh.part[0][0]);
  T* poll = reinterpret_cast<T*>(&sh.poll[0][0]);
  __syncthreads();
  if (warp == 0) {
    T x = T(0);
#pragma unroll 1
    for (int w = lane & 3; w < nwork; w += 4) x += part[w * 8 + (lane >> 2)];
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    if ((lane & 3) == 0) {
      u64* p = buf + (size_t)blockIdx.x * (sizeof(T) == 4 ? 8 : 16);
      const int k = lane >> 2;
      if constexpr (sizeof(T) == 4)
        st_word(p + k, word(__float_as_uint(x), tag));
      else
        st_words2(p + 2 * k, word((unsigned)__double2loint(x), tag), word((unsigned)__double2hiint(x), tag));
    }
    __syncwarp();
  }
  // the messages as one array of 16-byte chunks (a pair of FP32 values or one FP64
  // value): whole lines a warp, every warp a share; a thread a message would ask L2
  // for eight times as many lines, and the polls of 152 blocks are bound by that
  constexpr int CH = sizeof(T) == 4 ? 4 : 8;  // chunks a message
  constexpr int ML = CH * CR_MAXG / CR_MINT;  // chunks a thread at most
  const int nw = blockDim.x >> 5;
  T g[ML][8 / CH];
  unsigned spins = 0;
  int fail = 0;
#pragma unroll 1
  for (;;) {
    bool ok = true;
#pragma unroll
    for (int j = 0; j < ML; ++j) {
      const int i = (warp + j * nw) * 32 + lane;
      g[j][0] = T(0);
      if constexpr (CH == 4) g[j][1] = T(0);
      if (i < CH * G) {
        u64 a, b;
        ld_words2(buf + 2 * (size_t)i, a, b);
        ok = ok && tag_of(a) == tag && tag_of(b) == tag;
        if constexpr (CH == 4) {
          g[j][0] = __uint_as_float((unsigned)a);
          g[j][1] = __uint_as_float((unsigned)b);
        } else {
          g[j][0] = __hiloint2double((int)(unsigned)b, (int)(unsigned)a);
        }
      }
    }
    if (ok) break;
    if (give_up(ctl, spins, sh.polls)) {
      fail = 1;
      break;
    }
  }
  __syncwarp();
  const int nused = min(nw, (CH * G + 31) >> 5);  // warps with chunks
  if (warp < nused) {
#pragma unroll
    for (int i = 0; i < 8 / CH; ++i) {
      T x = g[0][i];
#pragma unroll
      for (int j = 1; j < ML; ++j)
        if ((warp + j * nw) * 32 < CH * G) x += g[j][i];
#pragma unroll
      for (int o = CH; o < 32; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if (lane < CH) poll[warp * 8 + lane * (8 / CH) + i] = x;
    }
  }
  if (fail) atomicCAS(&ctl->err, 0, QP_TIMEOUT);
  Summed<T> out;
  out.x = T(0);
  out.ok = !__syncthreads_or(fail);
  if (warp == 0) {
    T x = T(0);
#pragma unroll 1
    for (int w = lane & 3; w < nused; w += 4) x += poll[w * 8 + (lane >> 2)];
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    out.x = x;
  }
  return out;
}

// The sum of v, then warp 0 runs `last` on the totals, which leaves its results in
// sh.scal and sh.flag; they are valid for the whole block until the next call.  Only
// the first nwork warps, which own contacts, add anything.  False: a wait expired.
template <class T, class F>
__device__ __forceinline__ bool all_sum(const CgrArgs& A, CgrCount& N, CgrShared& sh, int nwork, const T (&v)[8],
                                        F last) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < nwork) {
    const T x = wsum8(v);
    if ((lane & 3) == 0) reinterpret_cast<T*>(&sh.part[0][0])[warp * 8 + (lane >> 2)] = x;
  }
  ++N.rc;
  const Summed<T> s = sum_gather<T>(sh, A.red + (size_t)(N.rc & 1) * CR_RED, A.ctl, A.epoch + N.rc, nwork);
  if (!s.ok) return false;
  if (warp == 0) last(s.x);
  __syncthreads();
  return true;
}

// Up to two FP64 sums for the start and the true residual: totals in sh.scal[0..1].
__device__ __noinline__ bool all_sum_cold(u64* red, DevCtl* ctl, unsigned tag, CgrShared& sh, double a, double b) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const double v[8] = {a, b};
  const double x = wsum8(v);
  if ((lane & 3) == 0) sh.part[warp][lane >> 2] = x;
  const Summed<double> s = sum_gather<double>(sh, red, ctl, tag, nw);
  if (!s.ok) return false;
  if (warp == 0 && lane < 8 && (lane & 3) == 0) sh.scal[lane >> 2] = s.x;
  __syncthreads();
  return true;
}

// The total of value k, in warp 0's last step.
template <class T>
__device__ __forceinline__ T total(T x, int k) {
  return __shfl_sync(0xffffffffu, x, 4 * k);
}

// Plan, first part: a block's bodies, their runs of the block's contacts, and one
// entry per (other block, shared body), sorted, so that what two blocks send each
// other lies in the same order and in one piece at both ends.
constexpr int CP_SORT = 2048;  // entries at most

__global__ void __launch_bounds__(512) k_cgr_lists(CgrPlan P, int M, int Nc, const int* __restrict__ ca,
                                                   const int* __restrict__ cb, const int* __restrict__ bptr,
                                                   const int* __restrict__ inc) {
  __shared__ int ncode, nbord, nint, nrem, nsum, over;
  __shared__ u64 key[CP_SORT];
  const int t = threadIdx.x, NT = blockDim.x, g = blockIdx.x, G = gridDim.x;
  const int c0 = min(Nc, g * P.chunk), c1 = min(Nc, c0 + P.chunk), n2 = 2 * (c1 - c0);
  unsigned* bmeta = P.bmeta + (size_t)g * P.nbcap;
  int* bid = P.bid + (size_t)g * P.nbcap;
  unsigned* rmeta = P.rmeta + (size_t)g * P.nbcap;
  unsigned short* rsum = P.rsum + (size_t)g * P.rcap;
  unsigned short* sbody = P.sbody + (size_t)g * P.rcap;
  unsigned short* codes = P.codes + (size_t)g * 2 * P.chunk;
  unsigned short* lidx = P.lidx + (size_t)g * 2 * P.chunk;
  if (t == 0) ncode = nbord = nint = nrem = nsum = over = 0;
  __syncthreads();
  for (int i = t; i < n2; i += NT) {
    const int c = c0 + (i >> 1);
    const int body = (i & 1) ? cb[c] : ca[c];
    if (body >= M) {
      lidx[i] = 0xFFFF;
      continue;
    }
    const int b0 = bptr[body], b1 = bptr[body + 1];
    int lo = b0;
    while ((inc[lo] >> 1) < c0) ++lo;  // ends: (c, side) is in the list
    const int first = inc[lo] - 2 * c0;
    if (first != i) {
      lidx[i] = (unsigned short)(0x8000 | first);  // resolved below
      continue;
    }
    int hi = lo + 1;
    while (hi < b1 && (inc[hi] >> 1) < c1) ++hi;
    const int off = atomicAdd(&ncode, hi - lo);
    for (int j = lo; j < hi; ++j) codes[off + j - lo] = (unsigned short)(inc[j] - 2 * c0);
    int lb;
    unsigned rm = 0;
    if (lo > b0 || hi < b1) {
      lb = atomicAdd(&nbord, 1);
      int runs = 0, pos = 0;
      for (int j = b0, prev = -1; j < b1; ++j) {
        const int blk = (inc[j] >> 1) / P.chunk;
        if (blk != prev && blk != g) {
          ++runs;
          if (blk < g) ++pos;
          const int k = atomicAdd(&nrem, 1);
          if (k < CP_SORT) key[k] = ((u64)blk << 48) | ((u64)(unsigned)body << 16) | (unsigned)lb;
        }
        prev = blk;
      }
      const int r0 = atomicAdd(&nsum, runs);
      if (runs > 255 || r0 + runs > P.rcap) over = 1;
      rm = (unsigned)r0 | ((unsigned)runs << 16) | ((unsigned)pos << 24);
    } else {
      lb = P.nbcap - 1 - atomicAdd(&nint, 1);
    }
    if (lb < 0 || lb >= P.nbcap || hi - lo > 0xFFFF) {
      over = 1;
      lb = 0;
    }
    bmeta[lb] = (unsigned)off | ((unsigned)(hi - lo) << 16);
    bid[lb] = body;
    rmeta[lb] = rm;
    lidx[i] = (unsigned short)lb;
  }
  __syncthreads();
  const int n = nrem;
  const bool bad = over || n > CP_SORT || n > P.rcap || nbord + nint > P.nbcap;
  if (t == 0) {
    int* h = P.head + 4 * g;
    h[0] = nbord;
    h[1] = nint;
    h[2] = n;
    if (bad) P.head[3] = 1;
  }
  if (bad) return;
  for (int i = t; i < n2; i += NT) {
    const unsigned v = lidx[i];
    if (v != 0xFFFF && (v & 0x8000)) lidx[i] = lidx[v & 0x7FFF];
  }
  int n2p = 1;
  while (n2p < n) n2p <<= 1;
  for (int i = n + t; i < n2p; i += NT) key[i] = ~0ull;
  __syncthreads();
  for (int k = 2; k <= n2p; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = t; i < n2p; i += NT) {
        const int l = i ^ j;
        if (l > i) {
          const u64 a = key[i], b = key[l];
          if ((a > b) == ((i & k) == 0)) {
            key[i] = b;
            key[l] = a;
          }
        }
      }
      __syncthreads();
    }
  for (int h = t; h < G; h += NT) {
    int lo = 0, hi = n;  // first entry of block h
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if ((int)(key[mid] >> 48) < h) lo = mid + 1;
      else hi = mid;
    }
    P.seg[(size_t)g * G + h] = lo;
  }
  for (int i = t; i < n; i += NT) {
    const int lb = (int)(key[i] & 0xFFFF), body = bid[lb];
    sbody[i] = (unsigned short)lb;
    // the entry's rank among the body's other blocks
    const int blk = (int)(key[i] >> 48);
    int rank = 0;
    for (int j = bptr[body], prev = -1; j < bptr[body + 1]; ++j) {
      const int q = (inc[j] >> 1) / P.chunk;
      if (q >= blk) break;
      if (q != prev && q != g) ++rank;
      prev = q;
    }
    rsum[(rmeta[lb] & 0xFFFFu) + rank] = (unsigned short)i;
    P.sdest[(size_t)g * P.rcap + i] = blk;  // k_cgr_dest makes it a place
  }
}

// Plan, second part: entry i of block g for block h goes to entry seg[h][g] + (i - seg[g][h]) of h.
__global__ void __launch_bounds__(512) k_cgr_dest(CgrPlan P) {
  const int g = blockIdx.x, G = gridDim.x;
  if (P.head[3]) return;
  const int n = P.head[4 * g + 2];
  int* d = P.sdest + (size_t)g * P.rcap;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const int h = d[i];
    d[i] = h * P.rcap + P.seg[(size_t)h * G + g] + (i - P.seg[(size_t)g * G + h]);
  }
}

// The block's lists into shared memory.
__device__ __noinline__ void copy_lists(const CgrPlan& P, CgrShared& B) {
  const int t = threadIdx.x, NT = blockDim.x, g = blockIdx.x;
  const int nb = B.nbord, ni = B.nint, n = B.nrem, n2 = 2 * (B.c1 - B.c0);
#pragma unroll 1
  for (int j = t; j < nb + ni; j += NT) {
    const int lb = j < nb ? j : P.nbcap - 1 - (j - nb);
    B.bmeta[lb] = P.bmeta[(size_t)g * P.nbcap + lb];
    B.bid[lb] = P.bid[(size_t)g * P.nbcap + lb];
    if (j < nb) B.rmeta[lb] = P.rmeta[(size_t)g * P.nbcap + lb];
  }
#pragma unroll 1
  for (int j = t; j < n; j += NT) {
    B.rsum[j] = P.rsum[(size_t)g * P.rcap + j];
    B.sbody[j] = P.sbody[(size_t)g * P.rcap + j];
    B.sdest[j] = P.sdest[(size_t)g * P.rcap + j];
  }
#pragma unroll 1
  for (int j = t; j < n2; j += NT) {
    B.codes[j] = P.codes[(size_t)g * 2 * P.chunk + j];
    B.lidx[j] = P.lidx[(size_t)g * 2 * P.chunk + j];
  }
  __syncthreads();
}

// The bodies' inverse masses and inertias in the precision that the next products use.
template <class T>
__device__ __forceinline__ void load_masses(CgrShared& B, const SysView<T>& s) {
  T* m = reinterpret_cast<T*>(B.bw);
  for (int j = threadIdx.x; j < B.nbord + B.nint; j += blockDim.x) {
    const int lb = j < B.nbord ? j : B.nbcap - 1 - (j - B.nbord);
    m[2 * lb] = __ldg(s.inv_m + B.bid[lb]);
    m[2 * lb + 1] = __ldg(s.inv_I + B.bid[lb]);
  }
}

// Body intermediates w = M^-1 sum of the wrenches written to B.wr (by this block,
// before the call's first barrier).  A shared body's partial sums go straight into
// the inboxes of the other blocks it touches, sorted by block and body at both ends:
// whole lines out and whole lines polled.  (Slots by incidence, each read by its
// own lane, made every poll of 152 blocks 250 000 L2 requests: 8200 cycles.)
//
// LB = 1: a thread a body.  LB = 8: a lane a component, for small FP64 systems: an
// FP64 instruction takes a warp 64 cycles however few of its lanes work.
template <class T, int LB>
__device__ __forceinline__ bool bodies(CgrShared& B, u64* halo, unsigned tag, DevCtl* ctl) {
  constexpr int NV = LB == 1 ? 6 : 1;           // components a thread
  static_assert(LB == 1 || sizeof(T) == 8, "a lane a component is for FP64");
  const T* wr = reinterpret_cast<const T*>(B.wr);
  T* wl = reinterpret_cast<T*>(B.wl);
  const int last = B.nbcap - 1, nbord = B.nbord, nall = nbord + B.nint;
  const unsigned short* codes = B.codes;
  const int u0 = LB == 1 ? 0 : (int)(threadIdx.x % LB);  // first component
  const int first = threadIdx.x / LB, step = blockDim.x / LB;
  const bool idle = u0 >= 6;
  const T* bw = reinterpret_cast<const T*>(B.bw);
  __syncthreads();
#pragma unroll 1
  for (int j = first; j < nall && !idle; j += step) {
    const int lb = j < nbord ? j : last - (j - nbord);
    const unsigned m = B.bmeta[lb];
    T v[NV];
#pragma unroll
    for (int u = 0; u < NV; ++u) v[u] = T(0);
    const unsigned short *k = codes + (m & 0xFFFFu), *e = k + (m >> 16);
#pragma unroll 1
    for (; k < e; ++k) {
      const int code = *k;
      const T* f = wr + (code >> 1) * CR_WR;
      const int q = (code & 1) ? 6 : 3;
      const T sg = (code & 1) ? T(1) : T(-1);
#pragma unroll
      for (int u = 0; u < NV; ++u) {
        const int w = u0 + u;
        v[u] += sg * f[w < 3 ? w : q + w - 3];
      }
    }
#pragma unroll
    for (int u = 0; u < NV; ++u) wl[lb * CR_WL + u0 + u] = j < nbord ? v[u] : v[u] * bw[2 * lb + (u0 + u < 3 ? 0 : 1)];
  }
  __syncthreads();  // (also: the wrenches' room may be rb's from here on)
  // out, by destination: consecutive threads write consecutive places of one inbox
  const int nrem = B.nrem;
#pragma unroll 1
  for (int j = first; j < nrem && !idle; j += step) {
    const T* v = wl + B.sbody[j] * CR_WL;
    const int d = B.sdest[j], h = d / B.rcap, place = d - h * B.rcap;
    u64* p = halo + ((size_t)h * (CR_HALO / 2) * B.rcap + place) * 2;
    if constexpr (LB == 1) {
#pragma unroll
      for (int u = 0; u < 6; u += 2) {
        if constexpr (sizeof(T) == 4) {
          st_words2(p + (size_t)u * B.rcap, word(__float_as_uint(v[u]), tag), word(__float_as_uint(v[u + 1]), tag));
        } else {
          st_words2(p + (size_t)(2 * u) * B.rcap, word((unsigned)__double2loint(v[u]), tag),
                    word((unsigned)__double2hiint(v[u]), tag));
          st_words2(p + (size_t)(2 * u + 2) * B.rcap, word((unsigned)__double2loint(v[u + 1]), tag),
                    word((unsigned)__double2hiint(v[u + 1]), tag));
        }
      }
    } else {
      const T x = v[u0];
      st_words2(p + (size_t)(2 * u0) * B.rcap, word((unsigned)__double2loint(x), tag),
                word((unsigned)__double2hiint(x), tag));
    }
  }
  // in: the block's own inbox, polled in its order
  T* rb = reinterpret_cast<T*>(B.rb);
  const u64* in = halo + (size_t)blockIdx.x * CR_HALO * B.rcap;
  int fail = 0;
#pragma unroll 1
  for (int j = first; j < nrem && !fail && !idle; j += step) {
    const u64* p = in + 2 * (size_t)j;
    T g[NV];
    unsigned spins = 0;
#pragma unroll 1
    for (;;) {
      bool ok = true;
      if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int u = 0; u < 6; u += 2) {
          u64 a, b;
          ld_words2(p + (size_t)u * B.rcap, a, b);
          ok = ok && tag_of(a) == tag && tag_of(b) == tag;
          g[u < NV ? u : 0] = __uint_as_float((unsigned)a);
          g[u + 1 < NV ? u + 1 : 0] = __uint_as_float((unsigned)b);
        }
      } else {
#pragma unroll
        for (int u = 0; u < NV; ++u) {
          u64 a, b;
          ld_words2(p + (size_t)(2 * (u0 + u)) * B.rcap, a, b);
          ok = ok && tag_of(a) == tag && tag_of(b) == tag;
          g[u] = __hiloint2double((int)(unsigned)b, (int)(unsigned)a);
        }
      }
      if (ok) break;
      if (give_up(ctl, spins, B.polls)) {
        fail = 1;
        break;
      }
    }
#pragma unroll
    for (int u = 0; u < NV; ++u) rb[j * CR_WL + u0 + u] = g[u];
  }
  if (fail) atomicCAS(&ctl->err, 0, QP_TIMEOUT);
  if (__syncthreads_or(fail)) return false;
  // shared bodies: the blocks' partial sums in block order, the same bits in every block
#pragma unroll 1
  for (int lb = first; lb < nbord && !idle; lb += step) {
    const unsigned rm = B.rmeta[lb];
    const int r0 = (int)(rm & 0xFFFFu), runs = (int)((rm >> 16) & 0xFFu), pos = (int)(rm >> 24);
    T v[NV];
#pragma unroll
    for (int u = 0; u < NV; ++u) v[u] = T(0);
#pragma unroll 1
    for (int j = 0; j <= runs; ++j) {
      const T* g = j == pos ? wl + lb * CR_WL : rb + B.rsum[r0 + j - (j > pos ? 1 : 0)] * CR_WL;
#pragma unroll
      for (int u = 0; u < NV; ++u) v[u] += g[u0 + u];
    }
#pragma unroll
    for (int u = 0; u < NV; ++u) wl[lb * CR_WL + u0 + u] = v[u] * bw[2 * lb + (u0 + u < 3 ? 0 : 1)];
  }
  __syncthreads();
  return true;
}

template <class T, int LB>
__device__ __forceinline__ bool bodies(const CgrArgs& A, CgrCount& N, CgrShared& sh) {
  ++N.xc;
  u64* halo = A.halo + (size_t)(N.xc & 1) * gridDim.x * CR_HALO * A.rcap;
  return bodies<T, LB>(sh, halo, A.epoch + N.xc, A.ctl);
}

__device__ __forceinline__ void load_rec16(const float* rec, int c, float (&g)[16]) {
  const float4* p = reinterpret_cast<const float4*>(rec + (size_t)c * 16);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float4 q = __ldg(p + k);
    g[4 * k] = q.x; g[4 * k + 1] = q.y; g[4 * k + 2] = q.z; g[4 * k + 3] = q.w;
  }
}
__device__ __forceinline__ void load_rec16(const double* rec, int c, double (&g)[16]) {
  const double2* p = reinterpret_cast<const double2*>(rec + (size_t)c * 16);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const double2 q = __ldg(p + k);
    g[2 * k] = q.x; g[2 * k + 1] = q.y;
  }
}

// FP64 residual r64 = rhs - S x of the block's rows with the stored arms; sh.scal:
// its squared norm over the system and the sum of dinv r^2.  Out of line: it runs
// once per factor inner_tol of convergence.  Uses the double-sized wr and wl.
// False: a wait expired.
__device__ __noinline__ bool residual(const CgrArgs& A, unsigned xc, unsigned rc, CgrShared& B) {
  const SysView<double>& s = A.s64;
  const long long n = s.Nc;
  const int c0 = B.c0, c1 = B.c1, t = threadIdx.x, NT = blockDim.x;
  __syncthreads();  // x is written, and the wrench buffer free
#pragma unroll 1
  for (int c = c0 + t; c < c1; c += NT) {
    double g[16];
    load_rec16(s.rec, c, g);
    const double* x = A.x + (long long)s.slots * c;
    const double x0 = x[0], x1 = x[1], x2 = x[2];
    const double f0 = g[0] * x0 + g[3] * x1 + g[6] * x2;
    const double f1 = g[1] * x0 + g[4] * x1 + g[7] * x2;
    const double f2 = g[2] * x0 + g[5] * x1 + g[8] * x2;
    double* w = B.wr + (c - c0) * CR_WR;
    w[0] = f0;
    w[1] = f1;
    w[2] = f2;
    w[3] = g[10] * f2 - g[11] * f1;
    w[4] = g[11] * f0 - g[9] * f2;
    w[5] = g[9] * f1 - g[10] * f0;
    w[6] = g[13] * f2 - g[14] * f1;
    w[7] = g[14] * f0 - g[12] * f2;
    w[8] = g[12] * f1 - g[13] * f0;
  }
  u64* halo = A.halo + (size_t)(xc & 1) * gridDim.x * CR_HALO * A.rcap;
  load_masses<double>(B, s);
  if (!bodies<double, 1>(B, halo, A.epoch + xc, A.ctl)) return false;
  double v0 = 0.0, v1 = 0.0;
#pragma unroll 1
  for (int c = c0 + t; c < c1; c += NT) {
    double g[16], h[6];
    load_rec16(s.rec, c, g);
#pragma unroll
    for (int k = 0; k < 6; ++k) h[k] = __ldg(s.H + k * n + c);
    const long long row = (long long)s.slots * c;
    const double x[3] = {A.x[row], A.x[row + 1], A.x[row + 2]};
    const unsigned la = B.lidx[2 * (c - c0)], lb = B.lidx[2 * (c - c0) + 1];
    const double* w = B.wl + lb * CR_WL;
    double d0 = w[0] + (w[4] * g[14] - w[5] * g[13]);
    double d1 = w[1] + (w[5] * g[12] - w[3] * g[14]);
    double d2 = w[2] + (w[3] * g[13] - w[4] * g[12]);
    if (la != 0xFFFFu) {
      w = B.wl + la * CR_WL;
      d0 -= w[0] + (w[4] * g[11] - w[5] * g[10]);
      d1 -= w[1] + (w[5] * g[9] - w[3] * g[11]);
      d2 -= w[2] + (w[3] * g[10] - w[4] * g[9]);
    }
    const double y[3] = {g[0] * d0 + g[1] * d1 + g[2] * d2 + (h[0] * x[0] + h[1] * x[1] + h[2] * x[2]),
                         g[3] * d0 + g[4] * d1 + g[5] * d2 + (h[1] * x[0] + h[3] * x[1] + h[4] * x[2]),
                         g[6] * d0 + g[7] * d1 + g[8] * d2 + (h[2] * x[0] + h[4] * x[1] + h[5] * x[2])};
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      const double ru = A.rhs[row + u] - y[u];
      A.r64[row + u] = ru;
      v0 += ru * ru;
      v1 += A.dinv64[row + u] * ru * ru;
    }
  }
  return all_sum_cold(A.red + (size_t)(rc & 1) * CR_RED, A.ctl, A.epoch + rc, B, v0, v1);
}

// A thread's share of the system.  Three forms:
//  * Own<T, 1>: one contact a thread, everything in registers;
//  * Own<T, KC>: KC contacts a thread, H and e in shared memory (all of it in registers
//    spilled, and beside this much shared memory no L1 is left for spills: 78 local
//    loads a warp and iteration);
//  * Rows: four lanes a contact, a row (and a Cartesian component) a lane, for small
//    FP64 systems.
template <class T, int KC>
struct Own {
  static constexpr int LB = 1;
  static constexpr bool SM = KC > 1;
  T n[KC][3], t1[KC][3], t2[KC][3], sa[KC], sb[KC], r[KC][3], q[KC][3];
  T Hr[SM ? 1 : KC][6], er[SM ? 1 : KC][3], pr[KC][3], dr[KC][3];
  T *Hs, *es, *ps;
  unsigned lab[KC];  // local bodies: a | b << 16
  int nc, t, NT;

  static int threads(int chunk) { return ceil_div(chunk, KC); }
  __device__ __forceinline__ int work_threads() const { return min(nc, NT); }
  __device__ __forceinline__ bool on(int k) const { return t + k * NT < nc; }

  // Everything but r, p and e from global memory: at the start, and after a residual,
  // so that none of it is live across that call (what is gets a stack slot, and the
  // iterations then read it from there).
  __device__ __forceinline__ void load(const CgrArgs& A, CgrShared& sh, const SysView<T>& s, const T* dinv) {
    t = threadIdx.x;
    NT = blockDim.x;
    nc = sh.c1 - sh.c0;
    if constexpr (SM) {
      // behind the FP32 wrenches, inside the room of the FP64 ones: H and e; behind the
      // lists: p, while a residual is formed
      Hs = reinterpret_cast<T*>(sh.wr) + CR_WR * A.chunk;
      es = Hs + 6 * A.chunk;
      ps = reinterpret_cast<T*>(sh.sbody + A.rcap);
    }
#pragma unroll
    for (int k = 0; k < KC; ++k) {
      r[k][0] = r[k][1] = r[k][2] = T(0);
      if (!on(k)) continue;
      const int lc = t + k * NT, c = sh.c0 + lc;
      T g[16];
      load_rec16(s.rec, c, g);
      sa[k] = g[0] * g[9] + g[1] * g[10] + g[2] * g[11];
      sb[k] = g[0] * g[12] + g[1] * g[13] + g[2] * g[14];
      lab[k] = (unsigned)sh.lidx[2 * lc] | ((unsigned)sh.lidx[2 * lc + 1] << 16);
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        n[k][u] = g[u];
        t1[k][u] = g[3 + u];
        t2[k][u] = g[6 + u];
        const T d = dinv[(long long)s.slots * c + u];
        dr[k][u] = d;
        if constexpr (SM) {
          es[3 * lc + u] = T(0);
          pr[k][u] = ps[3 * lc + u];
        } else {
          er[k][u] = T(0);
        }
      }
#pragma unroll
      for (int u = 0; u < 6; ++u) {
        const T h = __ldg(s.H + (long long)u * s.Nc + c);
        if constexpr (SM) Hs[u * A.chunk + lc] = h;
        else Hr[k][u] = h;
      }
    }
  }
  __device__ __forceinline__ void zero_p() {
#pragma unroll
    for (int k = 0; k < KC; ++k) pr[k][0] = pr[k][1] = pr[k][2] = T(0);
  }
  // r = v / scale
  __device__ __forceinline__ void set_r(const CgrArgs& A, CgrShared& sh, const double* v, double inv) {
#pragma unroll
    for (int k = 0; k < KC; ++k)
      if (on(k)) {
        const long long row = (long long)A.s64.slots * (sh.c0 + t + k * NT);
#pragma unroll
        for (int u = 0; u < 3; ++u) r[k][u] = (T)(v[row + u] * inv);
      }
  }
  // x += scale e (and p aside, where it is not kept in registers over a residual)
  __device__ __forceinline__ void put_x(const CgrArgs& A, CgrShared& sh, double scale) {
#pragma unroll
    for (int k = 0; k < KC; ++k)
      if (on(k)) {
        const int lc = t + k * NT;
        double* x = A.x + (long long)A.s64.slots * (sh.c0 + lc);
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          if constexpr (SM) {
            x[u] += scale * (double)es[3 * lc + u];
            ps[3 * lc + u] = pr[k][u];
          } else {
            x[u] += scale * (double)er[k][u];
          }
        }
      }
  }
  // p = D r + beta p and its wrench
  __device__ __forceinline__ void direction(CgrShared& sh, T beta) {
    T* wr = reinterpret_cast<T*>(sh.wr);
#pragma unroll
    for (int k = 0; k < KC; ++k)
      if (on(k)) {
        const int lc = t + k * NT;
        T p[3];
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          p[u] = dr[k][u] * r[k][u] + beta * pr[k][u];
          pr[k][u] = p[u];
        }
        T* w = wr + lc * CR_WR;
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const T g = p[1] * t2[k][u] - p[2] * t1[k][u];
          w[u] = n[k][u] * p[0] + t1[k][u] * p[1] + t2[k][u] * p[2];
          w[3 + u] = sa[k] * g;
          w[6 + u] = sb[k] * g;
        }
      }
  }
  // q = S p and the thread's share of the sums
  __device__ __forceinline__ void product(CgrShared& sh, T (&v)[8]) {
    const T* wl = reinterpret_cast<const T*>(sh.wl);
#pragma unroll
    for (int k = 0; k < KC; ++k)
      if (on(k)) {
        const int lc = t + k * NT;
        const unsigned la = lab[k] & 0xFFFFu, lb = lab[k] >> 16;
        const T* w = wl + lb * CR_WL;
        T d[3], W[3];
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          d[u] = w[u];
          W[u] = sb[k] * w[3 + u];
        }
        if (la != 0xFFFFu) {
          w = wl + la * CR_WL;
#pragma unroll
          for (int u = 0; u < 3; ++u) {
            d[u] -= w[u];
            W[u] -= sa[k] * w[3 + u];
          }
        }
        T p[3], D[3], h[6];
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          p[u] = pr[k][u];
          D[u] = dr[k][u];
        }
#pragma unroll
        for (int u = 0; u < 6; ++u) {
          if constexpr (SM) h[u] = Hs[u * sh.chunk + lc];
          else h[u] = Hr[k][u];
        }
        T y[3] = {h[0] * p[0] + h[1] * p[1] + h[2] * p[2], h[1] * p[0] + h[3] * p[1] + h[4] * p[2],
                  h[2] * p[0] + h[4] * p[1] + h[5] * p[2]};
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          y[0] += n[k][u] * d[u];
          y[1] += t1[k][u] * d[u] + t2[k][u] * W[u];
          y[2] += t2[k][u] * d[u] - t1[k][u] * W[u];
        }
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const T ri = r[k][u], qi = y[u], z = D[u] * ri;
          q[k][u] = qi;
          v[0] += ri * z;
          v[1] += p[u] * qi;
          v[2] += z * qi;
          v[3] += qi * (D[u] * qi);
          v[4] += ri * ri;
          v[5] += ri * qi;
          v[6] += qi * qi;
        }
      }
  }
  // e += al p, r -= al q
  __device__ __forceinline__ void step(T al) {
#pragma unroll
    for (int k = 0; k < KC; ++k)
      if (on(k)) {
        const int lc = t + k * NT;
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          if constexpr (SM) es[3 * lc + u] += al * pr[k][u];
          else er[k][u] += al * pr[k][u];
          r[k][u] -= al * q[k][u];
        }
      }
  }
};

template <class T>
struct Rows {
  static constexpr int LB = 8;
  T U[3], sa, sb, r, q, h[3], e, p, d;  // row u of U is (n_u, t1_u, t2_u); h: row u of H
  unsigned lab;
  int nc, t, lc, u;
  bool act;

  static int threads(int chunk) { return 4 * chunk; }
  __device__ __forceinline__ int work_threads() const { return 4 * nc; }
  __device__ __forceinline__ void zero_p() { p = T(0); }
  __device__ __forceinline__ void load(const CgrArgs& A, CgrShared& sh, const SysView<T>& s, const T* dinv) {
    t = threadIdx.x;
    nc = sh.c1 - sh.c0;
    lc = t >> 2;
    u = t & 3;
    act = lc < nc && u < 3;
    r = q = e = d = sa = sb = T(0);
    lab = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) U[k] = h[k] = T(0);
    if (!act) return;
    const int c = sh.c0 + lc;
    T g[16];
    load_rec16(s.rec, c, g);
    sa = g[0] * g[9] + g[1] * g[10] + g[2] * g[11];
    sb = g[0] * g[12] + g[1] * g[13] + g[2] * g[14];
    lab = (unsigned)sh.lidx[2 * lc] | ((unsigned)sh.lidx[2 * lc + 1] << 16);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      U[k] = u == 0 ? g[3 * k] : (u == 1 ? g[3 * k + 1] : g[3 * k + 2]);
      const int lo = u < k ? u : k, hi = u < k ? k : u;  // packed 00 01 02 11 12 22
      h[k] = __ldg(s.H + (long long)(lo == 0 ? hi : lo + hi + 1) * s.Nc + c);
    }
    d = dinv[(long long)s.slots * c + u];
  }
  __device__ __forceinline__ void set_r(const CgrArgs& A, CgrShared& sh, const double* v, double inv) {
    if (act) r = (T)(v[(long long)A.s64.slots * (sh.c0 + lc) + u] * inv);
  }
  __device__ __forceinline__ void put_x(const CgrArgs& A, CgrShared& sh, double scale) {
    if (act) {
      A.x[(long long)A.s64.slots * (sh.c0 + lc) + u] += scale * (double)e;
    }
  }
  __device__ __forceinline__ void direction(CgrShared& sh, T beta) {
    if ((t & ~31) >= work_threads()) return;  // whole warps
    p = d * r + beta * p;
    const int b = t & 28;
    const T p0 = __shfl_sync(0xffffffffu, p, b), p1 = __shfl_sync(0xffffffffu, p, b + 1),
            p2 = __shfl_sync(0xffffffffu, p, b + 2);
    const T g = p1 * U[2] - p2 * U[1], f = U[0] * p0 + U[1] * p1 + U[2] * p2;
    if (act) {
      T* w = reinterpret_cast<T*>(sh.wr) + lc * CR_WR + u;
      w[0] = f;
      w[3] = sa * g;
      w[6] = sb * g;
    }
  }
  __device__ __forceinline__ void product(CgrShared& sh, T (&v)[8]) {
    if ((t & ~31) >= work_threads()) return;
    const T* wl = reinterpret_cast<const T*>(sh.wl);
    const unsigned la = lab & 0xFFFFu, lb = lab >> 16;
    const int b = t & 28;
    T dd = T(0), W = T(0);
    if (act) {
      dd = wl[lb * CR_WL + u];
      W = sb * wl[lb * CR_WL + 3 + u];
      if (la != 0xFFFFu) {
        dd -= wl[la * CR_WL + u];
        W -= sa * wl[la * CR_WL + 3 + u];
      }
    }
    const T y0 = U[0] * dd, y1 = U[1] * dd + U[2] * W, y2 = U[2] * dd - U[1] * W;
    const T p0 = __shfl_sync(0xffffffffu, p, b), p1 = __shfl_sync(0xffffffffu, p, b + 1),
            p2 = __shfl_sync(0xffffffffu, p, b + 2);
    T qi = h[0] * p0 + h[1] * p1 + h[2] * p2;
#pragma unroll
    for (int k = 0; k < 3; ++k) {  // component k's share of row u
      const T a0 = __shfl_sync(0xffffffffu, y0, b + k), a1 = __shfl_sync(0xffffffffu, y1, b + k),
              a2 = __shfl_sync(0xffffffffu, y2, b + k);
      qi += u == 0 ? a0 : (u == 1 ? a1 : a2);
    }
    q = act ? qi : T(0);
    const T z = d * r;
    v[0] = r * z;
    v[1] = p * q;
    v[2] = z * q;
    v[3] = q * (d * q);
    v[4] = r * r;
    v[5] = r * q;
    v[6] = q * q;
  }
  __device__ __forceinline__ void step(T al) {
    if ((t & ~31) >= work_threads()) return;
    e += al * p;
    r -= al * q;
  }
};

// true for a positive number (not NaN), without the FP64 pipe
__device__ __forceinline__ bool positive(float x) { return x > 0.f; }
__device__ __forceinline__ bool positive(double x) {
  const int hi = __double2hiint(x);
  return hi >= 0 && hi <= 0x7ff00000 && (hi | __double2loint(x)) != 0 && !(hi == 0x7ff00000 && __double2loint(x) != 0);
}

// to = from (0 without one) in the block's rows but for the identity rows of four slots.
// Out of line, as residual() is.
__device__ __noinline__ void copy_rows(const CgrArgs& A, const CgrShared& sh, const double* __restrict__ from,
                                       double* __restrict__ to) {
  const int slots = A.s64.slots;
  const long long r1 = (long long)slots * sh.c1;
#pragma unroll 4
  for (long long i = (long long)slots * sh.c0 + threadIdx.x; i < r1; i += blockDim.x) {
    const double v = from ? from[i] : 0.0;
    if (slots == 3 || (i & 3) != 3) to[i] = v;
  }
}

// A search direction is kept over a residual replacement while the true residual is at
// most 1.1 times the recurrence's (both squared).
constexpr double KEEP2 = 1.21;

template <class T, class OWN, int NTMAX>
__global__ void __launch_bounds__(NTMAX, 1) k_cg_resident(const __grid_constant__ CgrArgs A) {
  extern __shared__ __align__(16) double cgr_dyn[];
  __shared__ CgrShared sh;
  const SysView<double>& s64 = A.s64;
  const int t = threadIdx.x, NT = blockDim.x, G = gridDim.x;
  CgrCount N = {0, 0};
  if (t == 0) {
    sh.c0 = min(s64.Nc, (int)blockIdx.x * A.chunk);
    sh.c1 = min(s64.Nc, sh.c0 + A.chunk);
    sh.chunk = A.chunk;
    sh.nbcap = A.nbcap;
    sh.rcap = A.rcap;
    sh.polls = A.polls;
    sh.nbord = A.pl.head[4 * blockIdx.x];
    sh.nint = A.pl.head[4 * blockIdx.x + 1];
    sh.nrem = A.pl.head[4 * blockIdx.x + 2];
    sh.wr = cgr_dyn;
    sh.wl = sh.wr + CR_WR * A.chunk;
    sh.bw = sh.wl + CR_WL * A.nbcap;
    // remote partials: room of their own, or the wrenches' (free while they arrive)
    sh.rb = A.own_rb ? sh.bw + 2 * A.nbcap : sh.wr;
    sh.bmeta = reinterpret_cast<unsigned*>(sh.bw + 2 * A.nbcap + (A.own_rb ? CR_WL * A.rcap : 0));
    sh.bid = reinterpret_cast<int*>(sh.bmeta + A.nbcap);
    sh.rmeta = reinterpret_cast<unsigned*>(sh.bid + A.nbcap);
    sh.sdest = reinterpret_cast<int*>(sh.rmeta + A.nbcap);
    sh.codes = reinterpret_cast<unsigned short*>(sh.sdest + A.rcap);
    sh.lidx = sh.codes + 2 * A.chunk;
    sh.rsum = sh.lidx + 2 * A.chunk;
    sh.sbody = sh.rsum + A.rcap;
  }
  if (A.pl.head[3] != 0) {  // the same for every block
    if (blockIdx.x == 0 && t == 0) {
      A.ctl->scal[S_TAGS] = 0.0;
      A.ctl->halvings = CGR_NO_ROOM;
    }
    return;
  }
  if ((int)blockIdx.x == A.absent && A.absent_at == 0) return;
  __syncthreads();
  copy_lists(A.pl, sh);

  const SysView<T>& s = [&]() -> const SysView<T>& {
    if constexpr (sizeof(T) == 4) return A.s32;
    else return A.s64;
  }();
  const T* dinv = [&]() -> const T* {
    if constexpr (sizeof(T) == 4) return A.dinv32;
    else return A.dinv64;
  }();
  double b0 = 0.0, b1 = 0.0;  // the right-hand side's squares: all rows, and those left to solve
  const long long r0 = (long long)s64.slots * sh.c0, r1 = (long long)s64.slots * sh.c1;
#pragma unroll 1
  for (long long i = r0 + t; i < r1; i += NT) {
    const double bi = A.rhs[i];
    // with four slots the last row is an identity row: solved by its right-hand side
    const bool solved = s64.slots == 4 && (i & 3) == 3;
    b0 += bi * bi;
    if (!solved) b1 += bi * bi;
    A.x[i] = solved ? bi : 0.0;
  }
#pragma unroll 1
  for (long long i = (long long)s64.slots * s64.Nc + blockIdx.x * (long long)NT + t; i < s64.P; i += (long long)G * NT)
    A.x[i] = 0.0;
  ++N.rc;
  if (!all_sum_cold(A.red + (size_t)(N.rc & 1) * CR_RED, A.ctl, A.epoch + N.rc, sh, b0, b1)) return;
  if (t == 0) {
    sh.bnorm = sh.scale = sqrt(sh.scal[0]);
    sh.best = sqrt(sh.scal[1]);
    sh.rel = sh.bnorm == 0.0 ? 0.0 : sh.best / sh.bnorm;
    sh.kept = 0;
  }
  __syncthreads();
  int iters = 0, repl = 0, status = 0;
  if ((int)blockIdx.x == A.absent) return;
  if (!(sh.rel <= A.tol)) {
    OWN own;
    own.load(A, sh, s, dinv);
    own.zero_p();
    load_masses<T>(sh, s);
    const int nwork = (own.work_threads() + 31) >> 5;
    own.set_r(A, sh, A.rhs, 1.0 / sh.bnorm);
    // the recurrence's r.r below which the true residual is due: a fall by inner_tol
    // or the target, whichever comes first
    const T drop2 = (T)(A.inner_tol * A.inner_tol);
    T due = fmax(drop2, (T)(A.tol * A.tol));
    T beta = T(0);
    T* sc = reinterpret_cast<T*>(sh.scal);  // alpha, beta, r.z, the new r.r
    for (;;) {
      if (iters >= A.maxit) {
        status = 1;
        break;
      }
      own.direction(sh, beta);
      if (!bodies<T, OWN::LB>(A, N, sh)) return;
      T v[8] = {};
      own.product(sh, v);
      if (!all_sum(A, N, sh, nwork, v, [&](T x) {
            // lane 0 divides r.z by p.q while lane 1 divides 1 by r.z; then lane 0 forms
            // (r.z)' while lane 1 forms (r.r)'
            const int lane = t & 31;
            const T z0 = total(x, 0), pq = total(x, 1), zq = total(x, 2), qdq = total(x, 3);
            const T r2 = total(x, 4), rq = total(x, 5), q2 = total(x, 6);
            const T dv = (lane == 1 ? T(1) : z0) / (lane == 1 ? z0 : pq);
            const T al = __shfl_sync(0xffffffffu, dv, 0), inv = __shfl_sync(0xffffffffu, dv, 1);
            const T a = lane == 1 ? r2 : z0, b = lane == 1 ? rq : zq, c = lane == 1 ? q2 : qdq;
            const T nw = a - al * (b + (b - al * c));
            const T rr = __shfl_sync(0xffffffffu, nw, 1);
            if (lane == 0) {
              sc[0] = al;
              sc[1] = nw * inv;
              sc[2] = z0;
              sc[3] = rr;
              // 1: the true residual is due; 2: cancellation left no digits of (r.z)', go
              // on from the true residual; 4: no step (p.q or r.z is not positive)
              sh.flag[0] = !(positive(z0) && positive(pq)) ? 4 : (rr <= due ? 1 : (positive(nw) ? 0 : 2));
            }
          }))
        return;
      const int flag = sh.flag[0];
      beta = sc[1];
      if (flag != 4) {
        own.step(sc[0]);
        ++iters;
      } else if (iters == 0) {
        status = 2;  // a breakdown before any progress is reported
        break;
      }
      if (flag != 0 || iters >= A.maxit) {
        // x += scale e; the true FP64 residual replaces r (unit norm) and the search
        // direction is kept with beta in the new units (reliable updates; van der Vorst
        // and Ye, SIAM J. Sci. Comput. 22 (2000)) -- as long as the recurrence was right:
        // where it has lost its digits (the late systems of a PDIP run, near the
        // attainable accuracy) the old direction is not conjugate to the new residual, and
        // keeping it made FP64 solves diverge (an 8^3 pile's 30th iterate at 1e-12: a
        // residual of 240 after 20 000 iterations; started afresh 1e-11 after 2200).
        if (t == 0) {
          sh.rz = (double)sc[2];
          sh.keep2 = flag == 1 ? KEEP2 * (double)sc[3] : -1.0;
        }
        own.put_x(A, sh, sh.scale);
        ++N.xc;
        ++N.rc;
        if (!residual(A, N.xc, N.rc, sh)) return;
        ++repl;
        // by one thread: a dozen warps' square roots and divisions would take their turn
        // in the SM's narrow FP64 pipe
        if (t == 0) {
          const double rn = sqrt(sh.scal[0]), rel = rn / sh.bnorm, inv = 1.0 / rn, grew = rn / sh.scale;
          const double goal = A.tol * sh.bnorm * inv;
          const bool better = rn < sh.best, last = iters >= A.maxit || repl >= A.max_outer;
          sh.next = rel <= A.tol ? R_DONE : (last ? (better ? R_CAP : R_CAP_BACK) : (better ? R_KEEP : R_GO));
          sh.rel = last && !better ? sh.best / sh.bnorm : rel;
          sh.inv = inv;
          sh.beta = grew * grew <= sh.keep2 ? sh.scal[1] * inv * inv / sh.rz * grew : 0.0;
          sh.due = goal * goal;
          sh.scale = rn;
          if (better) sh.best = rn;
          if (sh.next == R_KEEP) sh.kept = 1;
        }
        __syncthreads();
        const int next = sh.next;
        if (next == R_DONE) break;
        if (next == R_CAP || next == R_CAP_BACK) {
          status = 1;
          if (next == R_CAP_BACK) copy_rows(A, sh, sh.kept ? A.xbest : nullptr, A.x);
          break;
        }
        if (next == R_KEEP) copy_rows(A, sh, A.x, A.xbest);
        own.load(A, sh, s, dinv);
        load_masses<T>(sh, s);
        own.set_r(A, sh, A.r64, sh.inv);
        beta = (T)sh.beta;
        due = fmax(drop2, (T)sh.due);
      }
    }
  }
  if (blockIdx.x == 0 && t == 0) {
    A.ctl->iters = iters;
    A.ctl->outer = repl;
    A.ctl->scal[S_RELRES] = sh.rel;
    A.ctl->scal[S_BNORM] = sh.bnorm;
    A.ctl->scal[S_TAGS] = (double)(N.rc > N.xc ? N.rc : N.xc);
    A.ctl->halvings = status;
  }
}

template <class T, class OWN, int NTMAX>
bool launch(qp_ctx* c, CgrArgs& A, int G, size_t smem, size_t room) {
  auto k = k_cg_resident<T, OWN, NTMAX>;
  const int nt = std::max(CR_MINT, (OWN::threads(A.chunk) + 31) / 32 * 32);
  if (smem > room) return false;
  // the limit belongs to the function, not to the launch: always all the room, or another
  // thread's smaller system could lower it before this launch
  QP_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room));
  int per_sm = 0;
  QP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, nt, smem));
  if (per_sm < 1) return false;
  void* args[] = {&A};
  QP_CUDA(cudaLaunchCooperativeKernel((const void*)k, dim3(G), dim3(nt), args, smem, c->stream));
  return true;
}

}  // namespace

bool launch_cg_resident(qp_ctx* c, const double* rhs, double* dx, double tol, double inner_tol, int maxit,
                        int max_outer, bool mixed) {
  const int cap = mixed ? CR_CHUNK2 : CR_CHUNK1;  // contacts a block
  if (c->Nc < 1 || c->num_sms > CR_MAXG || c->cgr.tried[mixed] == ResidentPlan::NONE) return false;
  // no fewer contacts a block than fill its four schedulers once (a warp each; FP64
  // with four lanes a contact): more blocks would only make the sums longer
  const int chunk = std::max(ceil_div(c->Nc, c->num_sms), mixed ? 128 : 32);
  if (chunk > cap) return false;
  const int G = ceil_div(c->Nc, chunk);
  CgrArgs A;
  A.s64 = view64(c, true);
  A.s32 = view32(c, true);
  A.chunk = chunk;
  int optin = 0;
  QP_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device));
  const size_t room = (size_t)std::max(0, optin - (int)sizeof(CgrShared) - 256);
  const ResidentShape shape = resident_shape(chunk, room, c->cgr.tried[mixed] == ResidentPlan::ALL);
  c->cgr_full = shape.full;
  A.own_rb = shape.own_rb;
  A.nbcap = shape.nbcap;
  A.rcap = shape.rcap;
  {
    CgrPlan& P = A.pl;
    P.chunk = chunk;
    P.nbcap = A.nbcap;
    P.rcap = A.rcap;
    const size_t nb = (size_t)G * A.nbcap, nr = (size_t)G * A.rcap, nc = (size_t)G * 2 * chunk;
    const size_t ints = 4 * (size_t)G + 3 * nb + nr + (size_t)G * G, shorts = 2 * nr + 2 * nc;
    P.head = static_cast<int*>(c->cgr.room(c->cgr_plan, ints * 4 + shorts * 2, chunk));
    P.bid = P.head + 4 * (size_t)G;
    P.bmeta = reinterpret_cast<unsigned*>(P.bid + nb);
    P.rmeta = P.bmeta + nb;
    P.sdest = reinterpret_cast<int*>(P.rmeta + nb);
    P.seg = P.sdest + nr;
    P.rsum = reinterpret_cast<unsigned short*>(P.seg + (size_t)G * G);
    P.sbody = P.rsum + nr;
    P.codes = P.sbody + nr;
    P.lidx = P.codes + nc;
    if (c->cgr.chunk != chunk) {  // no plan yet for this contact set (or one for the other precision)
      QP_CUDA(cudaMemsetAsync(P.head, 0, 4 * (size_t)G * sizeof(int), c->stream));
      k_cgr_lists<<<G, 512, 0, c->stream>>>(P, c->M, c->Nc, c->ca.as<int>(), c->cb.as<int>(), c->bptr.as<int>(),
                                            c->inc.as<int>());
      k_cgr_dest<<<G, 512, 0, c->stream>>>(P);
      QP_CUDA(cudaGetLastError());
      c->cgr.chunk = chunk;
    }
  }
  A.rhs = rhs;
  A.x = dx;
  A.dinv64 = c->dinv.as<double>();
  A.dinv32 = c->dinv32.as<float>();
  A.tol = tol;
  A.inner_tol = inner_tol;
  A.maxit = maxit;
  A.max_outer = max_outer;
  A.polls = c->cgr_test ? c->cgr_test->polls : CGR_POLLS;
  A.absent = c->cgr_test ? c->cgr_test->absent : -1;
  A.absent_at = c->cgr_test ? c->cgr_test->at : 0;
  A.r64 = static_cast<double*>(c->v64[5].ensure((size_t)c->P * sizeof(double)));
  A.xbest = static_cast<double*>(c->v64[6].ensure((size_t)c->P * sizeof(double)));
  const size_t words = 2 * (size_t)G * CR_HALO * A.rcap + 2 * CR_RED;
  const size_t before = c->cgr_buf.cap;
  u64* buf = static_cast<u64*>(c->cgr_buf.ensure(words * sizeof(u64)));
  if (c->cgr_buf.cap != before || c->cgr_epoch > 0xE0000000u || c->cgr_epoch == 0) {
    // a new buffer, tags about to run out, or a solve that did not end: no old tag may match
    QP_CUDA(cudaMemsetAsync(buf, 0, c->cgr_buf.cap, c->stream));
    c->cgr_epoch = 1;
  }
  A.epoch = c->cgr_epoch;
  A.red = buf;
  A.halo = buf + 2 * CR_RED;
  A.ctl = c->ctl.as<DevCtl>();
  c->cgr_last = A.epoch;
  c->cgr_epoch = 0;  // set again once the solve's tag count is known
  bool ok;
  // FP64: a row a lane while that keeps every FP64 unit at one warp or two (64 contacts
  // an SM); above, a contact a thread fills the units as well with fewer instructions
  if (!mixed && chunk <= 64) ok = launch<double, Rows<double>, 256>(c, A, G, shape.smem(), room);
  else if (!mixed) ok = launch<double, Own<double, 1>, CR_CHUNK1>(c, A, G, shape.smem(), room);
  else if (chunk <= CR_CHUNK1) ok = launch<float, Own<float, 1>, CR_CHUNK1>(c, A, G, shape.smem(), room);
  else ok = launch<float, Own<float, 2>, CR_CHUNK2 / 2>(c, A, G, shape.smem(), room);
  if (!ok) c->cgr_epoch = A.epoch;
  return ok;
}

}  // namespace qp
