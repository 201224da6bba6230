// Dense operator applications of the hot path: every derivative (paper Sec.
// 2.4, eqs. D1, D2, D3, with the theta double cover of Sec. 2.1) and every
// matrix of the Yn filter (Sec. 3.5: phi DFT of eq. forwardF, projection of
// eq. FasPfQ, inverse DFT of eq. backwardF) is a product
//     Out[:, c] = W (P x K) * In[:, c]
// of a small operator W with many columns c.  Each column has its own gather
// of K input rows (two segments, the second optionally reversed and signed:
// the theta double cover and the complex spin projection) and its own scatter
// of P output rows (two segments).  No transposes are materialised.
//
// Two arithmetic cores share the column descriptors and the gathers:
//   FP64   plain double FMA on CUDA cores (k_op_fp64, the reference path);
//   MIXED  split-precision products on the fifth-generation tensor cores
//          (k_op_ws, and k_op_tc for small launches): W and each input column
//          are written as 47-bit fixed-point integers relative to a per-row /
//          per-field power of two and cut into six balanced 8-bit digits held
//          exactly in BF16; digit products are summed by tcgen05.mma in FP32
//          accumulators in tensor memory (see the k_op_ws comment for the
//          exactness argument); pairs with i + j > 6 (the filter's operators: > 5)
//          are dropped.
#include <algorithm>
#include <cstdio>

#include "common.cuh"
#include "scalar.cuh"
#include "tc.cuh"

namespace cffyn {

// ---------------------------------------------------------------------------
// Column descriptors

struct ColDesc {
  long long in0, in1, out0, out1;  // base offsets of the two row segments
  int sgn1;                        // second input segment: 0 as is, 1 negated, 2 zero
  int valid;
  int fld;                         // field (or function) whose exponent the column uses
};

struct OpGeom {
  int K, K0, P, P0;     // rows of W's columns (K), split of the input gather (K0),
                        // rows of W (P), split of the output scatter (P0)
  int in_rs, out_rs;    // row strides of input / output
  int rev1;             // second input segment reversed (row k -> K-1-k+K0... see load)
  long long ncols;
};

// All operators used by the shell, as one tagged descriptor.
enum OpKind : int { OP_R = 0, OP_ROWS = 1, OP_THETA = 2, OP_PROJ0 = 3, OP_PROJC = 4 };

struct OpArgs {
  OpKind kind;
  OpGeom g;
  const double* in;
  double* out;
  // OP_ROWS
  int Q;
  long long in_bs, out_bs;
  // OP_THETA / projections
  int n_r, N, J, R, L;
  int m;                 // projection: azimuthal number (set per block from blockIdx)
  const int* slots;      // projection: list of slots (R0: functions; C: re-slots of pairs)
  int nslots;
  int batched_m;         // projection launched for all m = 0..L at once
  long long w_stride;    // FP64 operator stride between consecutive m
  int ns;                // stacked shells: function f of shell s is array f * ns + s
  int fld0;              // OP_ROWS: array index of the launch's first array (its exponent word, pairing)
};

// Column c of a launch, with 32-bit divisions: a column has at least three
// values and the workspace holds seven or eight arrays of them, so c < 2^31
// on any device that can hold the shell.
__device__ __forceinline__ ColDesc make_col(const OpArgs& a, long long c) {
  ColDesc d;
  d.valid = c < a.g.ncols;
  d.sgn1 = 0;
  if (!d.valid) c = 0;
  switch (a.kind) {
    case OP_R: {
      d.fld = (int)((unsigned)c / (unsigned)(a.J * a.N));
      d.in0 = c * a.n_r;
      d.out0 = d.in0;
      d.in1 = d.out1 = 0;
      break;
    }
    case OP_ROWS: {
      const long long b = (unsigned)c / (unsigned)a.Q, q = c - b * a.Q;
      d.fld = a.fld0 + (int)b;
      d.in0 = b * a.in_bs + q;
      d.out0 = b * a.out_bs + q;
      d.in1 = d.out1 = 0;
      break;
    }
    case OP_THETA: {
      const long long pb = (unsigned)c / (unsigned)a.n_r;
      int kr = (int)(c - pb * a.n_r);
      int half = a.J / 2;
      const long long mu = (unsigned)pb / (unsigned)half;
      int jp = (int)(pb - mu * half);
      d.fld = (int)mu;
      d.in0 = ((mu * a.J + jp) * a.N) * a.n_r + kr;
      d.in1 = ((mu * a.J + jp + half) * a.N) * a.n_r + kr;
      d.out0 = d.in0;
      d.out1 = d.in1;
      break;
    }
    case OP_PROJ0: {
      // columns: (slot index, stacked shell, part, kr); parts: a (row m) and
      // b (row L+m, m >= 1)
      int nparts = a.m == 0 ? 1 : 2;
      long long per = (long long)nparts * a.n_r;
      if (c >= per * a.nslots * a.ns) { d.valid = 0; c = 0; }
      const long long fi = (unsigned)c / (unsigned)per;
      int rem = (int)(c - fi * per);
      int part = rem / a.n_r, kr = rem - part * a.n_r;
      const long long fs = (unsigned)fi / (unsigned)a.ns;
      int f = a.slots[fs < a.nslots ? fs : 0] * a.ns + (int)(fi - fs * a.ns);
      d.fld = f;
      int row = part == 0 ? a.m : a.L + a.m;
      d.in0 = (((long long)f * a.R + row) * a.N) * a.n_r + kr;
      d.out0 = d.in0;
      d.in1 = d.out1 = 0;
      break;
    }
    case OP_PROJC: {
      // columns: (pair, stacked shell, output part, kr); parts aR, aI, bR, bI
      // (m >= 1) or aR, aI
      int nparts = a.m == 0 ? 2 : 4;
      long long per = (long long)nparts * a.n_r;
      if (c >= per * a.nslots * a.ns) { d.valid = 0; c = 0; }
      const long long pi = (unsigned)c / (unsigned)per;
      int rem = (int)(c - pi * per);
      int part = rem / a.n_r, kr = rem - part * a.n_r;
      const long long ps = (unsigned)pi / (unsigned)a.ns;
      int fre = a.slots[ps < a.nslots ? ps : 0] * a.ns + (int)(pi - ps * a.ns), fim = fre + a.ns;
      d.fld = fre;
      int ra = a.m, rb = a.L + a.m;
      auto base = [&](int f, int row) {
        return (((long long)f * a.R + row) * a.N) * a.n_r + kr;
      };
      long long aR = base(fre, ra), aI = base(fim, ra);
      long long bR = a.m ? base(fre, rb) : aR, bI = a.m ? base(fim, rb) : aI;
      // at m = 0 the F_d half of the operator is zero: gather nothing there
      switch (part) {
        case 0: d.in0 = aR; d.in1 = bI; d.sgn1 = a.m ? 0 : 2; d.out0 = aR; break;
        case 1: d.in0 = aI; d.in1 = bR; d.sgn1 = a.m ? 1 : 2; d.out0 = aI; break;
        case 2: d.in0 = bR; d.in1 = aI; d.sgn1 = a.m ? 1 : 2; d.out0 = bR; break;
        default: d.in0 = bI; d.in1 = aR; d.sgn1 = a.m ? 0 : 2; d.out0 = bI; break;
      }
      d.out1 = 0;
      break;
    }
  }
  return d;
}

__device__ __forceinline__ double load_elem(const OpArgs& a, const ColDesc& d, int k) {
  if (!d.valid || k >= a.g.K) return 0.0;
  if (k < a.g.K0) return __ldg(a.in + d.in0 + (long long)k * a.g.in_rs);
  if (d.sgn1 == 2) return 0.0;
  int kk = a.g.rev1 ? (a.g.K - 1 - k) : (k - a.g.K0);
  const double v = __ldg(a.in + d.in1 + (long long)kk * a.g.in_rs);
  // sign flip on the bit pattern (no FP64 instruction)
  return __longlong_as_double(__double_as_longlong(v) ^ ((long long)d.sgn1 << 63));
}

__device__ __forceinline__ void store_elem(const OpArgs& a, const ColDesc& d, int p, double v) {
  if (!d.valid || p >= a.g.P) return;
  if (p < a.g.P0)
    a.out[d.out0 + (long long)p * a.g.out_rs] = v;
  else
    a.out[d.out1 + (long long)(p - a.g.P0) * a.g.out_rs] = v;
}

// ---------------------------------------------------------------------------
// FP64 core: CTA tile = 8 RP rows x QT columns, whole K staged in shared memory;
// each of eight warps holds RP rows.  Bound by the FP64 pipe, which a row past
// the operator's end costs as much as a row within (17 x 16 x 32, 64 rows for
// every operator: d_r with 17 rows 64 us, d_theta with 32 rows 60 us), so the
// rows are cut into as few equal tiles of at most 64 as there can be, rounded up
// to eight.

constexpr int F64_QT = 32;
constexpr int F64_MAX_RP = 8;

template <int RP>
__global__ void __launch_bounds__(256) k_op_fp64(OpArgs a, const double* __restrict__ W) {
  extern __shared__ double sm64[];
  if (a.batched_m) {
    a.m = blockIdx.z;
    W += (size_t)a.m * a.w_stride;
  }
  const int K = a.g.K, P = a.g.P;
  constexpr int TILE = 8 * RP;
  const int p0 = blockIdx.y * TILE;
  const int PT = min(TILE, P - p0);
  double* Ws = sm64;                 // PT x K
  double* Xs = sm64 + TILE * K;      // K x QT
  __shared__ ColDesc cols[F64_QT];
  const long long c0 = (long long)blockIdx.x * F64_QT;
  const int tid = threadIdx.x;
  if (tid < F64_QT) cols[tid] = make_col(a, c0 + tid);
  for (int e = tid; e < PT * K; e += 256) Ws[e] = W[(size_t)(p0 + e / K) * K + (e % K)];
  __syncthreads();
  const bool kfast = a.kind == OP_R;
  for (int e = tid; e < K * F64_QT; e += 256) {
    int k, c;
    if (kfast) { k = e % K; c = e / K; } else { c = e % F64_QT; k = e / F64_QT; }
    Xs[k * F64_QT + c] = load_elem(a, cols[c], k);
  }
  __syncthreads();
  const int tq = tid % F64_QT, tp = tid / F64_QT;  // 8 row groups
  double acc[RP];
  const double* wrow[RP];
#pragma unroll
  for (int r = 0; r < RP; ++r) {
    acc[r] = 0.0;
    wrow[r] = Ws + min(tp + 8 * r, PT - 1) * K;  // a row past the end repeats the last
  }
#pragma unroll 2
  for (int k = 0; k < K; ++k) {
    const double x = Xs[k * F64_QT + tq];
#pragma unroll
    for (int r = 0; r < RP; ++r) acc[r] = fma(wrow[r][k], x, acc[r]);
  }
  if (kfast) {
    // transpose through shared memory so that stores run along p
    __syncthreads();
    double* Os = Xs;  // reuse: PT x QT
#pragma unroll
    for (int r = 0; r < RP; ++r) {
      int row = tp + 8 * r;
      if (row < PT) Os[row * F64_QT + tq] = acc[r];
    }
    __syncthreads();
    for (int e = tid; e < PT * F64_QT; e += 256) {
      int p = e % PT, c = e / PT;
      store_elem(a, cols[c], p0 + p, Os[p * F64_QT + c]);
    }
  } else {
#pragma unroll
    for (int r = 0; r < RP; ++r) {
      int row = tp + 8 * r;
      if (row < PT) store_elem(a, cols[tq], p0 + row, acc[r]);
    }
  }
}

// ---------------------------------------------------------------------------
// Split-precision core.

// round(x 2^(47-E)) for one float, integer operations only
__device__ __forceinline__ long long fixed47f(unsigned int u, int E) {
  const int e = (int)((u >> 23) & 0xff);
  if (e == 0) return 0;
  const long long M = (long long)((u & 0x7fffff) | 0x800000);
  const int sh = e - 103 - E;  // <= 23 because |x| < 2^E
  long long Z;
  if (sh >= 0) Z = M << sh;
  else if (sh > -26) Z = (M + (1ll << (-sh - 1))) >> (-sh);
  else Z = 0;
  return (u >> 31) ? -Z : Z;
}

// 47-bit fixed point Z = round(x 2^(47-E)) of x relative to 2^E (|x| < 2^E),
// integer operations only.
__device__ __forceinline__ long long fixed47(double x, int E) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  long long Z = 0;
  if (e != 0) {
    const unsigned long long M = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
    const int sh = 1028 + E - e;  // >= 6 because |x| < 2^E
    if (sh < 54) Z = (long long)((M + (1ull << (sh - 1))) >> sh);
    if (b >> 63) Z = -Z;
  }
  return Z;
}

template <bool FI>
__device__ __forceinline__ long long raw_fixed47(long long w, int E) {
  if (FI) return fixed47f((unsigned int)w, E) + fixed47f((unsigned int)((unsigned long long)w >> 32), E);
  return fixed47(__longlong_as_double(w), E);
}

// Balanced base-256 digits of Z (|Z| <= 2^47): with Zb = Z + sum_{k<5} 128*256^k
// byte k of Zb is e_k + 128 for the five low digits and Zb >> 40 is the top
// digit.  Returned as BF16 bit patterns, slice 0 = most significant.
__device__ __forceinline__ void digits_bf16(long long Z, unsigned int out[kSlices]) {
  const long long Zb = Z + 0x8080808080ll;
  const unsigned int lo = (unsigned int)Zb;
  const int hi = (int)(Zb >> 32);
  // bf16(b - 128) for a byte b: exact small integer through the 1.5*2^23 trick
  auto bf = [](int b) -> unsigned int {
    return __float_as_uint(__int_as_float(0x4B400000 + b) - 12583040.0f) >> 16;
  };
  out[5] = bf((int)(lo & 255u));
  out[4] = bf((int)((lo >> 8) & 255u));
  out[3] = bf((int)((lo >> 16) & 255u));
  out[2] = bf((int)(lo >> 24));
  out[1] = bf(hi & 255);
  const int top = hi >> 8;  // arithmetic shift: the signed top digit
  out[0] = __float_as_uint(__int_as_float(0x4B400000 + top) - 12582912.0f) >> 16;
}

// T * 2^sc as a double (round to nearest), integer ops only.
__device__ __forceinline__ double i64_scaled_to_double(long long T, int sc) {
  if (T == 0) return 0.0;
  const unsigned long long s = T < 0 ? 0x8000000000000000ull : 0ull;
  unsigned long long v = T < 0 ? (unsigned long long)(-T) : (unsigned long long)T;
  const int nb = 64 - __clzll((long long)v);
  int ex = nb - 1 + sc;
  unsigned long long m;
  if (nb > 53) {
    const int sh = nb - 53;
    m = (v + (1ull << (sh - 1))) >> sh;
    if (m >> 53) {
      m >>= 1;
      ex += 1;
    }
  } else {
    m = v << (53 - nb);
  }
  if (ex + 1023 <= 0) return 0.0;
  const unsigned long long bits = s | ((unsigned long long)(ex + 1023) << 52) | (m & 0x000fffffffffffffull);
  return __longlong_as_double((long long)bits);
}

// T * 2^sc as a (hi, lo) float pair packed in 64 bits: hi exact leading 24
// bits, lo the next 24 (truncated).
__device__ __forceinline__ long long i64_scaled_to_pair(long long T, int sc) {
  if (T == 0) return 0;
  const bool neg = T < 0;
  const unsigned long long v = neg ? (unsigned long long)(-T) : (unsigned long long)T;
  const int nb = 64 - __clzll((long long)v);
  float hi, lo = 0.0f;
  if (nb <= 24) {
    hi = u64_scaled_to_float(v, sc, neg);
  } else {
    const int sh = nb - 24;
    const unsigned long long hm = v >> sh;
    hi = u64_scaled_to_float(hm, sc + sh, neg);
    lo = u64_scaled_to_float(v - (hm << sh), sc, neg);
  }
  return (long long)(((unsigned long long)__float_as_uint(lo) << 32) | __float_as_uint(hi));
}

// ---------------------------------------------------------------------------
// Per-field exponents of the mixed path's operator inputs.
//
// exps[f] = max over the field of (frexp exponent + 1022), 0 for an all-zero
// field.  With pairing, slots f >= kPairedFrom form (re, im) pairs (f, f^1)
// that share one exponent (the projection of a complex function gathers
// both).  Column values are cut into 47-bit fixed point round(x 2^(47-E)),
// E = exps - 1022, inside the operator kernel.

constexpr int kPairedFrom = 16;

// The exponent word of a field is read off the largest magnitude bit pattern
// (monotone in the exponent): the leading float of a pair, or the high word of
// an FP64 value, sign cleared.  Each thread covers eight values (16-byte loads
// when the field length is even), each CTA 2048, one atomic per CTA.
constexpr int kExpThreads = 256, kExpPerThread = 8;

template <bool FI>
__device__ __forceinline__ unsigned int mag_key(long long w) {
  return FI ? ((unsigned int)w & 0x7fffffffu) : ((unsigned int)((unsigned long long)w >> 32) & 0x7fffffffu);
}

template <bool FI>
__device__ __forceinline__ int exp_word(unsigned int m) {
  const int e = FI ? (int)(m >> 23) : (int)(m >> 20);
  return FI ? (e ? e - 126 + 1022 : 0) : e;
}

template <bool FI>
__global__ void __launch_bounds__(kExpThreads) k_field_exp(const long long* __restrict__ in, long long len,
                                                           int* __restrict__ exps) {
  __shared__ unsigned int wm[kExpThreads / 32];
  const int f = blockIdx.y;
  const long long* x = in + (long long)f * len;
  const long long b0 = (long long)blockIdx.x * kExpThreads * kExpPerThread;
  unsigned int m = 0;
  if ((len & 1) == 0) {
    const longlong2* x2 = reinterpret_cast<const longlong2*>(x);
#pragma unroll
    for (int i = 0; i < kExpPerThread / 2; ++i) {
      const long long q = b0 / 2 + (long long)i * kExpThreads + threadIdx.x;  // pair index
      if (2 * q < len) {
        const longlong2 v = __ldg(x2 + q);
        m = max(m, max(mag_key<FI>(v.x), mag_key<FI>(v.y)));
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < kExpPerThread; ++i) {
      const long long e = b0 + (long long)i * kExpThreads + threadIdx.x;
      if (e < len) m = max(m, mag_key<FI>(__ldg(x + e)));
    }
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kExpThreads / 32; ++w) m = max(m, wm[w]);
    const int word = exp_word<FI>(m);
    if (word) atomicMax(exps + f, word);
  }
}

// The same for short fields, one CTA per field: the word is stored, so that the
// words need no clearing in front (a launch less: 1.5 us of the 4.5 that the pair
// takes on a 13 x 9 x 18 shell).
constexpr int kExpShortThreads = 512, kExpShortLen = 16 * kExpShortThreads;

template <bool FI>
__global__ void __launch_bounds__(kExpShortThreads) k_field_exp_short(const long long* __restrict__ in, long long len,
                                                                      int* __restrict__ exps) {
  __shared__ unsigned int wm[kExpShortThreads / 32];
  const long long* x = in + (long long)blockIdx.x * len;
  unsigned int m = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int e = i * kExpShortThreads + threadIdx.x;
    if (e < len) m = max(m, mag_key<FI>(__ldg(x + e)));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = __reduce_max_sync(0xffffffffu, threadIdx.x < kExpShortThreads / 32 ? wm[threadIdx.x] : 0u);
    if (threadIdx.x == 0) exps[blockIdx.x] = exp_word<FI>(m);
  }
}

// ---------------------------------------------------------------------------
// Split-precision core on the fifth-generation tensor cores (tcgen05).
//
// Work item: 128 data columns (the MMA's M: one TMEM lane each) x one row
// group of W (ROWS = 48 or 96 rows), all of K in k-steps of 16.  A launch is
// persistent: one CTA per SM takes items blockIdx.x, + gridDim.x, ... of all
// its operator classes and azimuthal numbers.  Warp-specialised, every role
// walking the same item list on its own:
//   producer warps (three groups of 128 threads; a thread has one column and
//     all 16 k of every third k-step): load the raw words, cut them into six
//     BF16 digit slices (47-bit fixed point relative to the field's exponent)
//     in a shared-memory stage, arrive on its `xfull`; the loads of the
//     group's next k-step are issued right after the arrive (the proxy fence
//     and the arrive's release wait for every load the thread has in flight);
//   loader warp: bulk-copies (TMA) the operator's slices of each k-step (see
//     TcOp) into the stage, completing on its `wfull`;
//   MMA warp: once a stage is full, issues the digit-pair MMAs into five FP32
//     accumulators in TMEM and commits them to the stage's `empty`; after an
//     item's last k-step commits `accfull`;
//   epilogue warps (two per 32 TMEM lanes, half the rows each): read the
//     accumulators, fold them into float pairs, store, release `accempty`.
// The ring of stages runs across items, so the loads, the slicing and the
// operator copies of the next items go on under the products and the
// epilogue of the current one; with 48 rows the accumulators are
// double-buffered too (2 x 240 of the 512 TMEM columns), with 96 rows (480
// columns) the products wait for the fold's last TMEM load.
//   acc_d = sum_{i+j=d} W_i X_j                            d = 0..3
//   acc_4 = sum_{i+j=4} W_i X_j + 2^-8 sum_{i+j=5} W_i X_j + 2^-16 sum_{i+j=6} W_i X_j
// The digit-sum <= 4 pairs of one input slice X_j go out as one MMA of up to
// 256 rows over adjacent operator slices into adjacent accumulators (fewer
// MMAs per k-step, each input slice read from shared memory fewer times).
// The digit-sum-6 pairs are issued for the derivatives only (TcBatch::sum6);
// the filter's DFTs and projections stop at digit sum 5 (21 pairs) and copy
// eleven operator slices per k-step.
// acc_0..acc_3 are exact integers (below 4 * 192 * 2^14 < 2^24).  acc_4 is
// not exact; its rounding is below 2^-24 of a term of weight 256^-4 relative
// to the leading one, about 2^-56 of the result's scale, at the level of the
// dropped pairs i + j > 6 (about 4 * 2^-56).  With the digit-sum-6 pairs the
// result is as accurate as the 47-bit fixed point of its inputs; without
// them the dropped digit-sum-6 products (weight 2^-48) were the largest
// error.  The epilogue sums (acc_0 + acc_1 2^-8 + ... + acc_4 2^-32)
// 2^(E_row + E_col - 14) as a float pair (fold_pairs).

constexpr int kTcCols = 128;
constexpr int kTcXSlice = kTcCols * 16 * 2;                 // bytes of one data slice per k-step
constexpr int kTcXBytes = kSlices * kTcXSlice;               // 24576
constexpr unsigned long long kTcWaitNs = 1000000000ull;      // bound of the drain waits: 1 s

// A wait of the pipeline with the shell's bound; a bound of 0 gives up at
// once without polling (the way callers exercise the timeout path).
__device__ __forceinline__ bool pipe_wait(uint64_t* b, unsigned parity, unsigned long long limit_ns) {
  return limit_ns ? tc::bar_wait(b, parity, limit_ns) : false;
}

// Up to four operator applications with the same row-group size in one
// launch (the projections of the spin classes).
constexpr int kMaxBatch = 4;
struct TcBatch {
  OpArgs a[kMaxBatch];
  TcOp W[kMaxBatch];
  int tiles[kMaxBatch];      // column tiles of each class (per azimuthal number)
  int first[kMaxBatch + 1];  // first work item of each class; the number of items
  int nclass, nm;
  int eoff;  // added to every column exponent: a bound from an earlier scan times the operator gain
  int sum6;  // issue the digit-sum-6 pairs (derivatives); the filter's operators stop at digit sum 5
  unsigned long long wait_ns;  // bound of every pipeline wait (the shell's setting; 0: give up at once)
};

// thread layout of a CTA
constexpr int kEpiWarps = 8, kProdGroups = 3;
constexpr int kProdWarp0 = kEpiWarps, kMmaWarp = kProdWarp0 + 4 * kProdGroups, kLoadWarp = kMmaWarp + 1;
constexpr int kRawWarp = kLoadWarp + 1;               // d_r's input copies (STAGE 2)
constexpr int kWsThreads = 32 * (kRawWarp + 1);  // 736

template <int ROWS>
struct WsCfg {
  static constexpr int kWSlice = ROWS * 16 * 2;                        // bytes of one operator slice
  static constexpr int kWBytes = kTcWSlices * kWSlice;                 // 24576 | 49152
  static constexpr int kStage = kTcXBytes + kWBytes;                   // 49152 | 73728
  static constexpr int kAccs = ROWS == 48 ? 2 : 1;                     // accumulator sets in TMEM
  static constexpr uint32_t kTmemCols = 512;                           // set i at column 256 i
  static_assert(kStage % 1024 == 0, "stage alignment of the descriptors and bulk copies");
};
// stages of the ring; d_r's tiles (STAGE 1 and 2) take one stage's room and more
template <int ROWS, int STAGE>
constexpr int kRingStages = (ROWS == 48 ? 4 : 3) - (STAGE ? 1 : 0);
constexpr int kTcMaxSmem = 224 * 1024;  // of 227 KB, beside the barriers and row factors

// One work item: class, azimuthal number, column tile, row group.
struct TcItem {
  int cls, m, grp, ksteps;
  long long tile;
};

__device__ __forceinline__ TcItem item_at(const TcBatch& B, int t) {
  TcItem x;
  x.cls = 0;
#pragma unroll
  for (int c = 1; c < kMaxBatch; ++c)
    if (c < B.nclass && t >= B.first[c]) x.cls = c;
  const int ng = B.W[x.cls].ngroups;
  unsigned q = (unsigned)(t - B.first[x.cls]);
  x.grp = ng == 1 ? 0 : (int)(q % (unsigned)ng);
  q = ng == 1 ? q : q / (unsigned)ng;
  x.m = B.a[x.cls].batched_m ? (int)(q / (unsigned)B.tiles[x.cls]) : 0;
  x.tile = (long long)(q - (unsigned)x.m * (unsigned)B.tiles[x.cls]);
  x.ksteps = B.W[x.cls].ksteps;
  return x;
}

// Packed FP32 pairs (both halves rounded to nearest, never contracted).
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_pack(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ f2 f2_dup(float a) { return f2_pack(a, a); }
__device__ __forceinline__ unsigned int f2_lo(f2 a) { return (unsigned int)a; }
__device__ __forceinline__ unsigned int f2_hi(f2 a) { return (unsigned int)(a >> 32); }
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// Raw 64-bit words of 16 consecutive k of one column (zero outside K or in an
// empty second segment; the sign of a negated segment applied on the bits).
// A run inside one segment takes one pointer and its stride (an invalid
// column reads column 0, whose results are not stored); only a run that
// crosses segments or the end of K checks every element.  Branch-free within
// a run so that the loads issue together.
template <bool FI>
__device__ __forceinline__ void gather16(const OpArgs& a, const ColDesc& d, int k0, long long (&w)[16]) {
  const long long* in = reinterpret_cast<const long long*>(a.in);
  const long long m = FI ? (long long)0x8000000080000000ull : (long long)0x8000000000000000ull;
  const int K = a.g.K, K0 = a.g.K0;
  // element k of segment s lives at q_s[k * rs_s]
  const int rs0 = a.g.in_rs, rs1 = a.g.rev1 ? -rs0 : rs0;
  const long long* q0 = in + d.in0;
  const long long* q1 = in + d.in1 + (a.g.rev1 ? (K - 1) * rs0 : -(K0 * rs0));
  const bool flip = d.sgn1 == 1;
  const int kend = d.sgn1 == 2 ? min(K, K0) : K;
  const bool s0 = k0 + 16 <= min(kend, K0), s1 = k0 >= K0 && k0 + 16 <= kend;
  if (__all_sync(0xffffffffu, s0 || s1)) {
    const long long step = s1 ? rs1 : rs0;
    const long long* p = (s1 ? q1 : q0) + k0 * step;
#pragma unroll
    for (int i = 0; i < 16; ++i, p += step) w[i] = __ldg(p);
    if (s1 && flip) {
#pragma unroll
      for (int i = 0; i < 16; ++i) w[i] ^= m;
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int k = k0 + i;
    const bool seg1 = k >= K0;
    const long long* p = seg1 ? q1 + k * rs1 : q0 + k * rs0;
    const long long v = k < kend ? __ldg(p) : 0ll;
    w[i] = seg1 && flip ? (v ^ m) : v;
  }
}

// 2^k as a float, k clamped to the normal range
__device__ __forceinline__ float pow2f(int k) {
  return __int_as_float((max(-126, min(127, k)) + 127) << 23);
}

// a + b c (c a power of two), rounded, and its error, exactly (TwoSum with the
// product inside the fused additions: b c is exact).
__device__ __forceinline__ void f2_two_sum_scaled(f2 a, f2 b, f2 c, f2& s, f2& e) {
  s = f2_fma(b, c, a);
  const f2 nb = f2_sub(a, s);
  e = f2_add(f2_sub(a, f2_add(s, nb)), f2_fma(b, c, nb));
}

// (hi, lo) float pairs of rows j and j + 1, packed like the mixed path's
// internal storage, of (a0 + a1 2^-8 + a2 2^-16 + a3 2^-24 + a4 2^-32) f (f powers
// of two; the halves of every operand are the two rows).
// a0 + a1 2^-8 + a2 2^-16 + a3 2^-24 (exact values) is summed with error-free
// transformations, so that the sum's only roundings are those of the low
// words and of a4 2^-32 (below 2^-48 of |a0|); summing a3 2^-24 in plain FP32
// would cost about 2^-24 of it, more than the digit-sum-6 terms.  Packed FP32
// arithmetic: the FMA pipe takes as long as for two scalar folds, but half
// the issue slots, which the producers share.
__device__ __forceinline__ void fold_pairs(f2 a0, f2 a1, f2 a2, f2 a3, f2 a4, f2 f, f2& hi, f2& lo) {
  f2 s, t, e0, e1, e2;
  f2_two_sum_scaled(a0, a1, f2_dup(0.00390625f), s, e0);
  f2_two_sum_scaled(s, a2, f2_dup(1.52587890625e-05f), t, e1);
  f2_two_sum_scaled(t, a3, f2_dup(5.9604644775390625e-08f), s, e2);
  const f2 low = f2_fma(a4, f2_dup(2.3283064365386963e-10f), f2_add(f2_add(e0, e1), e2));
  hi = f2_add(s, low);
  lo = f2_mul(f2_sub(low, f2_sub(hi, s)), f);
  hi = f2_mul(hi, f);
}

// The outputs of a column scale by 2^E_row 2^ec, in one product of the two;
// where ec is extreme that product can leave the float range, and the factors
// (2^ec in two parts, the second beyond the float range's) go one by one.
struct ColScale {
  f2 f1, f2_;
  bool extreme;
  __device__ __forceinline__ explicit ColScale(int ec)
      : f1(f2_dup(pow2f(ec))), f2_(f2_dup(pow2f(ec - max(-126, min(127, ec))))), extreme(ec < -60 || ec > 60) {}
};

// The folded pairs w of a chunk of N accumulator rows v; rowF: those rows' 2^E_row
// (8-byte aligned).
template <bool EXTREME, int N>
__device__ __forceinline__ void fold_rows(const uint32_t (&v)[5][N], const float* rowF, const ColScale& cs,
                                          long long (&w)[N]) {
#pragma unroll
  for (int j = 0; j < N; j += 2) {
    auto two = [&](int d) { return f2_pack(__uint_as_float(v[d][j]), __uint_as_float(v[d][j + 1])); };
    const float2 rr = *reinterpret_cast<const float2*>(rowF + j);
    const f2 rf = f2_pack(rr.x, rr.y);
    f2 hi, lo;
    fold_pairs(two(0), two(1), two(2), two(3), two(4), EXTREME ? rf : f2_mul(rf, cs.f1), hi, lo);
    if (EXTREME) {
      hi = f2_mul(f2_mul(hi, cs.f1), cs.f2_);
      lo = f2_mul(f2_mul(lo, cs.f1), cs.f2_);
    }
    w[j] = (long long)((lo << 32) | f2_lo(hi));
    w[j + 1] = (long long)((lo & 0xffffffff00000000ull) | f2_hi(hi));
  }
}
template <int N>
__device__ __forceinline__ void fold_chunk(const uint32_t (&v)[5][N], const float* rowF, const ColScale& cs,
                                           long long (&w)[N]) {
  if (__any_sync(0xffffffffu, cs.extreme))
    fold_rows<true>(v, rowF, cs, w);
  else
    fold_rows<false>(v, rowF, cs, w);
}

// Digit slices of two float pairs x = hi + lo (|lo| < ulp(hi), |x| < 2^E) on
// the FMA pipe, packed.  Digit j has weight 2^(E - 7 - 8j) (the balanced
// base-256 digits of round(x 2^(47 - E))).  With v = x 2^(7 - E) (sc, exact)
// and s = -(remainder), the exact steps
//   d_0 = rint(v), s = d_0 - v;   d_j = rint(-256 s), s = d_j + 256 s
// (rint by adding and subtracting 1.5 * 2^23) give balanced digits |d| <= 128
// of hi; the last digit rounds like the fixed-point conversion.  lo
// contributes to digits 3..5 only (|lo| / w_2 < 1/2; sc3 = sc 2^24), so digit
// j is d_j(hi) + d_j(lo), |.| <= 256, an exact BF16 value; it is the same
// integer sum of weights as the rounded fixed point of hi plus that of lo.
// Requires -78 <= E <= 126 (every weight and inverse weight a normal float).
// out[j]: the two values' digits as BF16 (the upper half of the float).
__device__ __forceinline__ void digits_two(long long x0, long long x1, f2 sc, f2 sc3, unsigned int (&out)[kSlices]) {
  const f2 M = f2_dup(12582912.0f), up = f2_dup(256.0f), dn = f2_dup(-256.0f);  // 1.5 * 2^23
  const f2 v = f2_mul(f2_pack(__int_as_float((int)(unsigned int)x0), __int_as_float((int)(unsigned int)x1)), sc);
  const f2 u = f2_mul(f2_pack(__int_as_float((int)(unsigned int)((unsigned long long)x0 >> 32)),
                              __int_as_float((int)(unsigned int)((unsigned long long)x1 >> 32))),
                      sc3);
  f2 d[kSlices];
  d[0] = f2_sub(f2_add(v, M), M);
  f2 s = f2_sub(d[0], v);
#pragma unroll
  for (int j = 1; j < kSlices; ++j) {
    d[j] = f2_sub(f2_fma(s, dn, M), M);
    if (j < kSlices - 1) s = f2_fma(s, up, d[j]);
  }
  f2 e = f2_sub(f2_add(u, M), M);
  s = f2_sub(e, u);
  d[3] = f2_add(d[3], e);
#pragma unroll
  for (int j = 4; j < kSlices; ++j) {
    e = f2_sub(f2_fma(s, dn, M), M);
    if (j < kSlices - 1) s = f2_fma(s, up, e);
    d[j] = f2_add(d[j], e);
  }
#pragma unroll
  for (int j = 0; j < kSlices; ++j) out[j] = __byte_perm(f2_lo(d[j]), f2_hi(d[j]), 0x7632);
}

__device__ __forceinline__ void bar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_addr(b)) : "memory");
}
// named barrier over nthreads threads, and the AND of their predicates
__device__ __forceinline__ void named_sync(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
__device__ __forceinline__ bool named_and(int id, int nthreads, bool p) {
  int r;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.s32 p, %3, 0;\nbar.red.and.pred q, %1, %2, p;\nselp.s32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"(id), "r"(nthreads), "r"((int)p)
      : "memory");
  return r != 0;
}

// exponent of a column's fixed point, relative to 1022 in the field words
__device__ __forceinline__ int col_exponent(const TcBatch& B, const OpArgs& a, const ColDesc& col,
                                            const int* __restrict__ exps, int pairing) {
  int ce = exps[col.fld];
  if (pairing) {
    // slot pairs (f, f ^ 1), f >= kPairedFrom, of the same stacked shell
    const int f = a.ns == 1 ? col.fld : col.fld / a.ns, sidx = col.fld - f * a.ns;
    if (f >= kPairedFrom) ce = max(ce, exps[(f ^ 1) * a.ns + sidx]);
  }
  return ce - 1022 + B.eoff;
}

// STAGE: the launch is d_r (one operator class, all rows in one group), whose
// columns are contiguous lines of n_r words.  1: the epilogue stages a tile's
// outputs in shared memory and stores them as one contiguous block per 32
// columns.  2 (ROWS = 48, odd n_r up to kRawRows): also the inputs come as one bulk
// copy per tile, into one of two buffers that the tile's outputs then take (each
// thread's 16 words of a line, 8 bytes per load and a line apart across the
// lanes, were 32 sectors per load: 61 against 56 us for 50 fields of 33 x 48 x 96;
// odd, so that the lanes' words lie in different banks).
// 736 threads leave 80 registers each: the instances of pair words spill 116 to 124
// bytes per thread, 28 to 44 of them read back (<true, 48, 2> none).
constexpr int kRawRows = 39;
template <bool FI, int ROWS, int STAGE>
__global__ void __launch_bounds__(kWsThreads, 1)
    k_op_ws(const __grid_constant__ TcBatch B, const int* __restrict__ exps, int pairing, int* __restrict__ flag) {
  using C = WsCfg<ROWS>;
  constexpr int S = kRingStages<ROWS, STAGE>, A = C::kAccs;
  extern __shared__ __align__(1024) unsigned char smtc[];
  __shared__ uint64_t xfull[S], wfull[S], empty[S], accfull[A], accempty[A], rawfull[2], rawfree[2], drained;
  __shared__ uint32_t tmem_base;
  __shared__ __align__(16) float rowF[kEpiWarps][ROWS / 2];  // 2^E_row of each epilogue warp's rows
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int total = B.first[B.nclass];
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      tc::bar_init(&xfull[s], 128);
      tc::bar_init(&wfull[s], 1);
      tc::bar_init(&empty[s], 1);
    }
    for (int i = 0; i < A; ++i) {
      tc::bar_init(&accfull[i], 1);
      tc::bar_init(&accempty[i], kEpiWarps);
    }
    for (int i = 0; i < 2; ++i) {
      tc::bar_init(&rawfull[i], 1);
      tc::bar_init(&rawfree[i], kEpiWarps);
    }
    tc::bar_init(&drained, 1);
  }
  if (warp == kMmaWarp) tc::alloc(&tmem_base, C::kTmemCols);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tm = tmem_base;
  bool ok = true;
  // d_r's tile of item n of this CTA: [column][n_r]
  auto tile_buf = [&](int n) {
    return reinterpret_cast<long long*>(smtc + S * C::kStage) + (STAGE == 2 ? (n & 1) * kTcCols * B.a[0].g.P : 0);
  };

  if (warp >= kProdWarp0 && warp < kMmaWarp) {
    // a group must not be two uses of a stage ahead of the products (its wait
    // on `empty` tells phases apart by their parity only): with two stages
    // the third group has no part
    // (for the same reason every group takes part in every tile of STAGE 2)
    const int G = STAGE == 2 ? min(kProdGroups, B.W[0].ksteps) : (S < kProdGroups ? S : kProdGroups);
    const int g = (warp - kProdWarp0) >> 2;
    const int ctile = (warp & 3) * 32 + lane;
    const int xoff = (ctile >> 3) * 256 + (ctile & 7) * 16;
    int t = blockIdx.x, n = 0, ks = g;
    TcItem x;
    ColDesc col;
    int E = 0;
    // the group's next k-step: k-step ks of item t, or of a later item
    auto settle = [&](bool fresh) -> bool {
      for (; t < total; t += gridDim.x, ++n) {
        if (fresh) x = item_at(B, t);
        if (ks < x.ksteps) {
          if (fresh) {
            OpArgs a = B.a[x.cls];
            a.m = x.m;
            col = make_col(a, x.tile * kTcCols + ctile);
            E = col_exponent(B, a, col, exps, pairing);
            // an all-zero field has no exponent: with any, its digits are zeros.  (The
            // integer slicing that it would take here, 16 words to a thread, holds up
            // the products: RK4 step of 33 x 40 x 80 points with 58 fields, some of them
            // zero, 2220 us, so 2033; projection of 33 x 17 x 34 points 32.0 us, one-item
            // kernel 22.6, filter call 93.0, so 84.7.)
            if (FI && E == B.eoff - 1022) E = 0;
          }
          return true;
        }
        ks -= x.ksteps;
        fresh = true;
      }
      return false;
    };
    long long w[16];
    bool have = g < G && settle(true);
    if (STAGE != 2 && have) gather16<FI>(B.a[x.cls], col, ks * 16, w);
    for (int it = g; have; it += G) {
      const int s = it % S, use = it / S;
      if (use > 0 && !(ok = __all_sync(0xffffffffu, pipe_wait(&empty[s], (use - 1) & 1, B.wait_ns)))) break;
      if constexpr (STAGE == 2) {
        if (!(ok = __all_sync(0xffffffffu, pipe_wait(&rawfull[n & 1], (n >> 1) & 1, B.wait_ns)))) break;
        const int P = B.a[0].g.P;
        const long long* line = tile_buf(n) + ctile * P;
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] = ks * 16 + i < P ? line[ks * 16 + i] : 0ll;
      }
      unsigned char* xs = smtc + s * C::kStage + xoff;
      const bool fscale = FI && E >= -78 && E <= 126;  // FMA-pipe slicing of float pairs
      const f2 sc = f2_dup(pow2f(fscale ? 7 - E : 0)), sc3 = f2_dup(pow2f(fscale ? 31 - E : 0));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        unsigned int wd[4][kSlices];
        if (fscale) {
#pragma unroll
          for (int i = 0; i < 4; ++i) digits_two(w[8 * h + 2 * i], w[8 * h + 2 * i + 1], sc, sc3, wd[i]);
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            unsigned int d0[kSlices], d1[kSlices];
            digits_bf16(raw_fixed47<FI>(w[8 * h + 2 * i], E), d0);
            digits_bf16(raw_fixed47<FI>(w[8 * h + 2 * i + 1], E), d1);
#pragma unroll
            for (int j = 0; j < kSlices; ++j) wd[i][j] = d0[j] | (d1[j] << 16);
          }
        }
#pragma unroll
        for (int j = 0; j < kSlices; ++j)
          *reinterpret_cast<uint4*>(xs + j * kTcXSlice + h * 128) = make_uint4(wd[0][j], wd[1][j], wd[2][j], wd[3][j]);
      }
      tc::fence_proxy_async();
      bar_arrive(&xfull[s]);
      ks += G;
      have = settle(false);
      if (STAGE != 2 && have) gather16<FI>(B.a[x.cls], col, ks * 16, w);
    }
  } else if (warp >= kMmaWarp) {
    if (STAGE == 2 && warp == kRawWarp && lane == 0) {
      int n = 0;
      const int P = B.a[0].g.P;
      for (int t = blockIdx.x; t < total; t += gridDim.x, ++n) {
        if (n >= 2 && !(ok = pipe_wait(&rawfree[n & 1], ((n >> 1) - 1) & 1, B.wait_ns))) break;
        const long long c0 = item_at(B, t).tile * kTcCols;
        const int words = (int)min((long long)kTcCols, B.a[0].g.ncols - c0) * P;
        const long long* src = reinterpret_cast<const long long*>(B.a[0].in) + c0 * P;
        long long* dst = tile_buf(n);
        // whole 16 bytes: a sphere has 2 n_theta^2 lines, so columns come in pairs
        const uint32_t bytes = (uint32_t)words * 8;
        tc::bar_expect_tx(&rawfull[n & 1], bytes);
        tc::bulk_g2s(dst, src, bytes, &rawfull[n & 1]);
      }
      for (int c = n > 2 ? n - 2 : 0; c < n; ++c) tc::bar_wait(&rawfull[c & 1], (c >> 1) & 1, kTcWaitNs);
    }
    if (warp == kLoadWarp && lane == 0) {
      // the operator slices of a k-step; without the digit-sum-6 pairs the
      // last five (digits 1..5 times 2^-16) stay in global memory
      const uint32_t wcopy = B.sum6 ? C::kWBytes : (kTcWSlices - 5) * C::kWSlice;
      int it = 0;
      for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
        const TcItem x = item_at(B, t);
        const unsigned char* src = reinterpret_cast<const unsigned char*>(B.W[x.cls].w + (size_t)x.m * B.W[x.cls].w_stride) +
                                   (size_t)x.grp * x.ksteps * C::kWBytes;
        for (int ks = 0; ks < x.ksteps; ++ks, ++it) {
          const int s = it % S, use = it / S;
          if (use > 0 && !(ok = pipe_wait(&empty[s], (use - 1) & 1, B.wait_ns))) break;
          tc::bar_expect_tx(&wfull[s], wcopy);
          tc::bulk_g2s(smtc + s * C::kStage + kTcXBytes, src + (size_t)ks * C::kWBytes, wcopy, &wfull[s]);
        }
      }
      // every copy issued has landed before the CTA's memory goes, also after
      // a wait gave up here or in another role (the long bound: these end)
      for (int c = it > S ? it - S : 0; c < it; ++c) tc::bar_wait(&wfull[c % S], (c / S) & 1, kTcWaitNs);
    }
    if (warp == kMmaWarp && lane == 0) {
      const uint32_t sbase = tc::smem_addr(smtc);
      int it = 0, n = 0;
      for (int t = blockIdx.x; t < total && ok; t += gridDim.x, ++n) {
        const int ksteps = item_at(B, t).ksteps;
        const int ai = n % A, ause = n / A;
        if (ause > 0 && !(ok = pipe_wait(&accempty[ai], (ause - 1) & 1, B.wait_ns))) break;
        const uint32_t ta = tm + ai * 256;
        for (int ks = 0; ks < ksteps; ++ks, ++it) {
          const int s = it % S;
          const unsigned ph = (it / S) & 1;
          ok = pipe_wait(&wfull[s], ph, B.wait_ns) && pipe_wait(&xfull[s], ph, B.wait_ns);
          if (!ok) break;
          tc::fence_after();
          const uint32_t xa = sbase + s * C::kStage;
          const uint64_t dx = tc::desc_kmajor(xa, 128, 256);
          const uint64_t dw = tc::desc_kmajor(xa + kTcXBytes, 128, 256);
          constexpr uint32_t ID = tc::idesc_bf16_f32(kTcCols, ROWS);
          constexpr uint64_t XS = kTcXSlice >> 4, WS = C::kWSlice >> 4;  // slice strides, descriptor units
          // digit-sum <= 4 pairs of input slice j: the operator slices 0..4-j
          // are adjacent in shared memory and their accumulators acc_j..acc_4
          // adjacent in TMEM, so up to 256 / ROWS of them go into one MMA of
          // N = n ROWS (fewer re-reads of the input slice)
          constexpr int kMerge = 256 / ROWS;
#pragma unroll
          for (int j = 0; j < 5; ++j)
#pragma unroll
            for (int i = 0; i + j <= 4; i += kMerge) {
              const int nn = (5 - j - i) < kMerge ? (5 - j - i) : kMerge;
              const uint32_t idn = tc::idesc_bf16_f32(kTcCols, nn * ROWS);
              tc::mma(ta + (i + j) * ROWS, dx + j * XS, dw + i * WS, idn, (ks > 0 || j > 0) ? 1u : 0u);
            }
#pragma unroll
          for (int i = 0; i < 6; ++i) tc::mma(ta + 4 * ROWS, dx + (5 - i) * XS, dw + (5 + i) * WS, ID, 1u);
          if (B.sum6) {
#pragma unroll
            for (int i = 1; i < 6; ++i) tc::mma(ta + 4 * ROWS, dx + (6 - i) * XS, dw + (10 + i) * WS, ID, 1u);
          }
          tc::commit(&empty[s]);
        }
        if (ok) tc::commit(&accfull[ai]);
      }
      // the MMAs issued finish before the CTA's shared and tensor memory go,
      // also after a wait gave up in some role (the long bound: these end)
      tc::commit(&drained);
      tc::bar_wait(&drained, 0, kTcWaitNs);
    }
  } else {
    // epilogue warp: TMEM lanes 32 (warp % 4) .. + 31 (its columns), rows
    // [h R, (h + 1) R) of every accumulator
    constexpr int R = ROWS / 2, CH = 8;  // rows of a warp, rows at a time
    const int q = warp & 3, h = warp >> 2;
    const int ctile = q * 32 + lane;
    float* rf = rowF[warp];
    int n = 0;
    for (int t = blockIdx.x; t < total; t += gridDim.x, ++n) {
      const TcItem x = item_at(B, t);
      OpArgs a = B.a[x.cls];
      a.m = x.m;
      const ColDesc col = make_col(a, x.tile * kTcCols + ctile);
      const int* rexp = B.W[x.cls].rowexp + (size_t)x.m * B.W[x.cls].rowexp_stride + x.grp * ROWS + h * R;
      __syncwarp();
      for (int i = lane; i < R; i += 32) rf[i] = pow2f(rexp[i]);
      const ColScale cs(col_exponent(B, a, col, exps, pairing) - 14);
      __syncwarp();
      const int prow = min(a.g.P - x.grp * ROWS, ROWS);  // valid rows of this group
      const int ai = n % A, ause = n / A;
      ok = __all_sync(0xffffffffu, pipe_wait(&accfull[ai], ause & 1, B.wait_ns));
      // the two warps of a column quarter leave together (they share barriers)
      if (STAGE) ok = named_and(1 + q, 64, ok);
      if (!ok) break;
      tc::fence_after();
      const uint32_t ta = tm + ai * 256 + ((uint32_t)(q * 32) << 16);
      const int pend = min((h + 1) * R, prow);
      long long* out = reinterpret_cast<long long*>(a.out);
      const int prow0 = x.grp * ROWS;  // first row of the group within W
      long long* o0 = out + col.out0;
      const long long ors = a.g.out_rs;
      long long* o1 = out + col.out1 - a.g.P0 * ors;
      long long* stage = STAGE ? tile_buf(n) + ctile * prow : nullptr;
      if (h * R >= pend) {
        __syncwarp();
        if (lane == 0) bar_arrive(&accempty[ai]);
      }
#pragma unroll 1
      for (int p0 = h * R; p0 < pend; p0 += CH) {
        uint32_t v[5][CH];
#pragma unroll
        for (int d = 0; d < 5; ++d) tc::ld8(ta + d * ROWS + p0, v[d]);
        tc::ld_wait(v[0]);
#pragma unroll
        for (int d = 1; d < 5; ++d) tc::tie(v[d]);
        if (p0 + CH >= pend) {
          // the accumulators are read: the next item may overwrite them
          tc::fence_before();
          __syncwarp();
          if (lane == 0) bar_arrive(&accempty[ai]);
        }
        long long w[CH];
        fold_chunk(v, rf + p0 - h * R, cs, w);
        const int p = prow0 + p0;
        if (STAGE) {
#pragma unroll
          for (int j = 0; j < CH; ++j)
            if (p0 + j < pend) stage[p0 + j] = w[j];
        } else if (p0 + CH <= pend && (p >= a.g.P0 || p + CH <= a.g.P0)) {
          // a chunk within one output segment: one pointer and its stride
          if (col.valid) {
            long long* o = (p >= a.g.P0 ? o1 : o0) + p * ors;
#pragma unroll
            for (int j = 0; j < CH; ++j, o += ors) *o = w[j];
          }
        } else if (col.valid) {
#pragma unroll
          for (int j = 0; j < CH; ++j)
            if (p0 + j < pend) (p + j >= a.g.P0 ? o1 : o0)[(p + j) * ors] = w[j];
        }
      }
      if constexpr (STAGE != 0) {
        // d_r: a quarter's outputs (32 columns of n_r rows each, out0 = c n_r)
        // are one contiguous block: a bulk store, or for the columns of the last
        // tile consecutive threads on consecutive words
        tc::fence_proxy_async();
        named_sync(1 + q, 64);
        const long long c0 = x.tile * kTcCols + q * 32;
        const int words = (int)max(0ll, min(32ll, a.g.ncols - c0)) * prow;
        const long long* from = tile_buf(n) + q * 32 * prow;
        long long* dst = out + c0 * prow;
        if (words == 32 * prow) {
          if (h == 0 && lane == 0) {
            tc::bulk_s2g(dst, from, (uint32_t)words * 8);
            tc::bulk_read_wait();
          }
        } else {
          for (int e = h * 32 + lane; e < words; e += 64) dst[e] = from[e];
          tc::fence_proxy_async();
        }
        if (STAGE == 1) {
          named_sync(1 + q, 64);
        } else {
          __syncwarp();
          if (lane == 0) bar_arrive(&rawfree[n & 1]);
        }
      }
    }
    if (STAGE && h == 0 && lane == 0) tc::bulk_done_wait();
  }
  ok = __syncthreads_and(ok);
  if (!ok && threadIdx.x == 0) atomicOr(flag, 2);
  tc::fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc::fence_after();
    tc::dealloc(tm, C::kTmemCols);
  }
}

// The same products one item per CTA, for launches of few items (runs_persistent:
// up to one per SM with 96 rows, three with 48, five or more for d_r): their
// time is mostly one item's latency, which more producer threads with fewer k each
// shorten, and two CTAs of 48 rows share an SM.  Producer warps (256 or 512 threads; one column and KQ = 8 or
// 4 consecutive k of every k-step each) slice and, after the last k-step, run
// the epilogue; one MMA warp copies the operator slices a stage ahead and
// issues the products.
template <int ROWS>
struct TcCfg {
  static constexpr int kProd = ROWS == 48 ? 256 : 512;                 // producer threads
  static constexpr int kThreads = kProd + 32;                          // + the MMA warp
  static constexpr int kKQ = 16 * kTcCols / kProd;                     // k per producer per k-step
  static constexpr int kWSlice = ROWS * 16 * 2;                        // bytes of one operator slice
  static constexpr int kWBytes = kTcWSlices * kWSlice;                 // 24576 | 49152
  static constexpr int kStage = kTcXBytes + kWBytes;                   // 49152 | 73728
  static constexpr int kStages = ROWS == 48 ? 2 : 3;                   // 2 CTAs / 1 CTA per SM
  static constexpr int kSmem = kStages * kStage;                       // 98304 | 221184
  static constexpr uint32_t kTmemCols = ROWS == 48 ? 256 : 512;        // 5 accumulators x ROWS
  static_assert(kSmem <= 227 * 1024, "dynamic shared memory per CTA");
  static_assert(kStage % 1024 == 0, "stage alignment of the descriptors and bulk copies");
};


// Raw 64-bit words of N consecutive k of one column (zero outside K or in an
// empty second segment; the sign of a negated segment applied on the bits).
// Branch-free so that the loads issue together.
template <bool FI, int N>
__device__ __forceinline__ void gather(const OpArgs& a, const ColDesc& d, int k0, long long (&w)[N]) {
  const long long* in = reinterpret_cast<const long long*>(a.in);
  const long long m = FI ? (long long)0x8000000080000000ull : (long long)0x8000000000000000ull;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int k = k0 + i;
    const bool seg1 = k >= a.g.K0;
    const int kk = seg1 ? (a.g.rev1 ? (a.g.K - 1 - k) : (k - a.g.K0)) : k;
    const long long base = seg1 ? d.in1 : d.in0;
    const bool live = d.valid && k < a.g.K && !(seg1 && d.sgn1 == 2);
    const long long v = live ? __ldg(in + base + (long long)kk * a.g.in_rs) : 0ll;
    w[i] = (seg1 && d.sgn1 == 1) ? (v ^ m) : v;
  }
}


template <bool FI, int ROWS, bool STAGE = false>
__global__ void __launch_bounds__(TcCfg<ROWS>::kThreads)
    k_op_tc(const __grid_constant__ TcBatch B, const int* __restrict__ exps, int pairing, int* __restrict__ flag) {
  using C = TcCfg<ROWS>;
  constexpr int S = C::kStages, KQ = C::kKQ;
  extern __shared__ __align__(1024) unsigned char smtc[];
  __shared__ uint64_t xfull[S], wfull[S], empty[S], accf;
  __shared__ uint32_t tmem_base;
  __shared__ __align__(16) float rowF[ROWS];  // 2^E_row
  const TcItem x = item_at(B, blockIdx.x);
  OpArgs a = B.a[x.cls];
  TcOp W = B.W[x.cls];
  a.m = x.m;
  W.w += (size_t)x.m * W.w_stride;
  W.rowexp += (size_t)x.m * W.rowexp_stride;
  const long long tile = x.tile;
  const int grp = x.grp;
  const int tid = threadIdx.x;
  const bool producer = tid < C::kProd;
  const int ctile = tid & (kTcCols - 1);        // column within the tile (producers)
  const int kq = (tid >> 7) * KQ;               // first k of this producer within a k-step
  const ColDesc col = make_col(a, tile * kTcCols + ctile);
  const int E = col_exponent(B, a, col, exps, pairing);
  // the row exponents are needed only by the epilogue: loaded here, stored
  // to shared memory before the barrier that ends the main loop
  const int rexp = tid < ROWS ? W.rowexp[grp * ROWS + tid] : 0;
  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      tc::bar_init(&xfull[s], C::kProd);
      tc::bar_init(&wfull[s], 1);
      tc::bar_init(&empty[s], 1);
    }
    tc::bar_init(&accf, 1);
  }
  if (tid >= C::kProd) tc::alloc(&tmem_base, C::kTmemCols);  // the MMA warp
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tm = tmem_base;
  const int ksteps = W.ksteps;
  bool ok = true;

  if (producer) {
    // byte offset of this thread's row piece (column ctile, k kq..kq+KQ-1)
    const int xoff = (ctile >> 3) * 256 + (kq >> 3) * 128 + (ctile & 7) * 16 + (kq & 7) * 2;
    const bool fscale = E >= -78 && E <= 126;  // FMA-pipe slicing of float pairs
    const f2 sc = f2_dup(pow2f(fscale ? 7 - E : 0)), sc3 = f2_dup(pow2f(fscale ? 31 - E : 0));
    // The loads of the next k-step are issued after the arrive on the
    // current stage: the proxy fence and the arrive's release wait for every
    // load the thread has in flight, so loads issued before them would hold
    // up this stage (measured: the first k-step's slices 0.7 us later).
    long long nxt[KQ];
    gather<FI, KQ>(a, col, kq, nxt);
    for (int ks = 0; ks < ksteps; ++ks) {
      const int s = ks % S;
      long long cur[KQ];
#pragma unroll
      for (int i = 0; i < KQ; ++i) cur[i] = nxt[i];
      if (ks >= S && ok) ok = pipe_wait(&empty[s], ((ks - S) / S) & 1, B.wait_ns);
      unsigned char* xs = smtc + s * C::kStage + xoff;
      uint32_t wd[kSlices][KQ / 2];
      if (FI && fscale && ks * 16 + kq < a.g.K) {
#pragma unroll
        for (int i = 0; i < KQ; i += 2) {
          unsigned int d[kSlices];
          digits_two(cur[i], cur[i + 1], sc, sc3, d);
#pragma unroll
          for (int j = 0; j < kSlices; ++j) wd[j][i >> 1] = d[j];
        }
      } else if (ks * 16 + kq < a.g.K) {
#pragma unroll
        for (int i = 0; i < KQ; i += 2) {
          unsigned int d0[kSlices], d1[kSlices];
          digits_bf16(raw_fixed47<FI>(cur[i], E), d0);
          digits_bf16(raw_fixed47<FI>(cur[i + 1], E), d1);
#pragma unroll
          for (int j = 0; j < kSlices; ++j) wd[j][i >> 1] = d0[j] | (d1[j] << 16);
        }
      } else {
#pragma unroll
        for (int j = 0; j < kSlices; ++j)
#pragma unroll
          for (int i = 0; i < KQ / 2; ++i) wd[j][i] = 0u;
      }
#pragma unroll
      for (int j = 0; j < kSlices; ++j) {
        if (KQ == 8)
          *reinterpret_cast<uint4*>(xs + j * kTcXSlice) = make_uint4(wd[j][0], wd[j][1], wd[j][2], wd[j][3]);
        else
          *reinterpret_cast<uint2*>(xs + j * kTcXSlice) = make_uint2(wd[j][0], wd[j][1]);
      }
      tc::fence_proxy_async();
      bar_arrive(&xfull[s]);
      if (ks + 1 < ksteps) gather<FI, KQ>(a, col, (ks + 1) * 16 + kq, nxt);
    }
    if (ok) ok = pipe_wait(&accf, 0, B.wait_ns);
  } else if (tid == C::kProd) {
    // MMA thread
    const unsigned char* wsrc =
        reinterpret_cast<const unsigned char*>(W.w) + (size_t)grp * ksteps * C::kWBytes;
    // the operator slices of a k-step; without the digit-sum-6 pairs the
    // last five (digits 1..5 times 2^-16) stay in global memory
    const uint32_t wcopy = B.sum6 ? C::kWBytes : (kTcWSlices - 5) * C::kWSlice;
    const uint32_t sbase = tc::smem_addr(smtc);
    for (int ks = 0; ks < S && ks < ksteps; ++ks) {
      tc::bar_expect_tx(&wfull[ks], wcopy);
      tc::bulk_g2s(smtc + ks * C::kStage + kTcXBytes, wsrc + (size_t)ks * C::kWBytes, wcopy, &wfull[ks]);
    }
    int copied = S < ksteps ? S : ksteps;  // operator k-steps whose copy has been issued
    for (int ks = 0; ks < ksteps && ok; ++ks) {
      const int s = ks % S;
      ok = pipe_wait(&wfull[s], (ks / S) & 1, B.wait_ns) && pipe_wait(&xfull[s], (ks / S) & 1, B.wait_ns);
      if (!ok) break;
      tc::fence_after();
      const uint32_t xa = sbase + s * C::kStage;
      const uint64_t dx = tc::desc_kmajor(xa, 128, 256);
      const uint64_t dw = tc::desc_kmajor(xa + kTcXBytes, 128, 256);
      constexpr uint32_t ID = tc::idesc_bf16_f32(kTcCols, ROWS);
      constexpr uint64_t XS = kTcXSlice >> 4, WS = C::kWSlice >> 4;  // slice strides, descriptor units
      // digit-sum <= 4 pairs of input slice j: the operator slices 0..4-j
      // are adjacent in shared memory and their accumulators acc_j..acc_4
      // adjacent in TMEM, so up to 256 / ROWS of them go into one MMA of
      // N = n ROWS (fewer re-reads of the input slice)
      constexpr int kMerge = 256 / ROWS;
#pragma unroll
      for (int j = 0; j < 5; ++j)
#pragma unroll
        for (int i = 0; i + j <= 4; i += kMerge) {
          const int n = (5 - j - i) < kMerge ? (5 - j - i) : kMerge;
          const uint32_t idn = tc::idesc_bf16_f32(kTcCols, n * ROWS);
          tc::mma(tm + (i + j) * ROWS, dx + j * XS, dw + i * WS, idn, (ks > 0 || j > 0) ? 1u : 0u);
        }
#pragma unroll
      for (int i = 0; i < 6; ++i) tc::mma(tm + 4 * ROWS, dx + (5 - i) * XS, dw + (5 + i) * WS, ID, 1u);
      if (B.sum6) {
#pragma unroll
        for (int i = 1; i < 6; ++i) tc::mma(tm + 4 * ROWS, dx + (6 - i) * XS, dw + (10 + i) * WS, ID, 1u);
      }
      tc::commit(&empty[s]);
      // refill the stage of k-step ks - 1 with the operator of k-step ks - 1 + S
      if (ks >= 1 && copied < ksteps) {
        const int sp = (ks - 1) % S;
        ok = pipe_wait(&empty[sp], ((ks - 1) / S) & 1, B.wait_ns);
        if (!ok) break;
        tc::bar_expect_tx(&wfull[sp], wcopy);
        tc::bulk_g2s(smtc + sp * C::kStage + kTcXBytes, wsrc + (size_t)copied * C::kWBytes, wcopy,
                     &wfull[sp]);
        ++copied;
      }
    }
    // accf completes once every MMA issued above has completed: then the
    // accumulators are final, or, after a wait gave up, no MMA still reads
    // shared memory or writes tensor memory
    tc::commit(&accf);
    if (!ok) {
      // let operator copies still in flight land, and the MMAs issued finish,
      // before the CTA's memory goes (the long bound: these always end)
      for (int c = (copied > S ? copied - S : 0); c < copied; ++c) tc::bar_wait(&wfull[c % S], (c / S) & 1, kTcWaitNs);
      tc::bar_wait(&accf, 0, kTcWaitNs);
    }
  }
  if (tid < ROWS) rowF[tid] = pow2f(rexp);
  ok = __syncthreads_and(ok);
  if (!ok && tid == 0) atomicOr(flag, 2);
  tc::fence_after();
  if (ok && producer) {
    // producer warp w reads TMEM lanes 32 (w % 4) .. + 31 (its columns) and
    // rows [g R, (g + 1) R) of every accumulator, g = w / 4, R = ROWS / (warps / 4)
    constexpr int R = ROWS / (C::kProd / 128);
    const int g = tid >> 7;
    const int prow = min(a.g.P - grp * ROWS, ROWS);  // valid rows of this group
    // d_r (all rows in one group): outputs staged in the free stage buffers
    // (every MMA and copy has completed) as [column][row]
    constexpr bool stage_out = STAGE;
    long long* out_tile = reinterpret_cast<long long*>(smtc);
    const uint32_t lane = tm + ((uint32_t)(((tid >> 5) & 3) * 32) << 16);
    const ColScale cs(E - 14);
    // the group's rows of this thread's column, each folded result handed to
    // sink(row within the group, pair bits)
    auto rows_out = [&](auto&& sink) {
#pragma unroll 1
      for (int p0 = g * R; p0 < (g + 1) * R && p0 < prow; p0 += 8) {
        uint32_t v[5][8];
#pragma unroll
        for (int d = 0; d < 5; ++d) tc::ld8(lane + d * ROWS + p0, v[d]);
        tc::ld_wait(v[0]);
#pragma unroll
        for (int d = 1; d < 5; ++d) tc::tie(v[d]);
        long long w[8];
        fold_chunk(v, rowF + p0, cs, w);
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (p0 + j < prow) sink(p0 + j, w[j]);
      }
    };
    if constexpr (!stage_out)
      rows_out([&](int row, long long w) { store_elem(a, col, grp * ROWS + row, __longlong_as_double(w)); });
    else
      rows_out([&](int row, long long w) { out_tile[ctile * prow + row] = w; });
    if constexpr (stage_out) {
      // d_r: the tile's outputs (columns c of n_r rows each, out0 = c n_r)
      // are one contiguous block; after the producers' barrier it is copied
      // out with consecutive threads on consecutive words
      asm volatile("bar.sync 1, %0;" ::"r"(C::kProd) : "memory");
      const long long c0 = tile * kTcCols;
      const long long nc = min((long long)kTcCols, a.g.ncols - c0);
      long long* dst = reinterpret_cast<long long*>(a.out) + c0 * prow;
      for (long long e = tid; e < nc * prow; e += C::kProd) dst[e] = out_tile[e];
    }
  }
  tc::fence_before();
  __syncthreads();
  if (tid >= C::kProd) {
    tc::fence_after();
    tc::dealloc(tm, C::kTmemCols);
  }
}

// ---------------------------------------------------------------------------
// Host side

static int tiles_of(const OpArgs& a) { return (int)((a.g.ncols + kTcCols - 1) / kTcCols); }

// Whether a launch of so many items takes the persistent kernel.  With 96 rows
// (the one-item kernel holds one CTA per SM) it pays from more than one item per SM
// on: 297 / 322 / 1238 items take 27 / 35 / 96 us against 31 / 43 / 133 when it came in, an
// RK4 step of 33 x 32 x 64 takes 1204 us, 1242 with the line at two.  With 48 rows (two
// CTAs per SM) it pays by itself from two to three items per SM on (470 items of
// d_theta + d_phi 24.3 against 25.7 us, 846 / 1128 of the projection 33 / 38 against 43 /
// 57), later for d_r (dr; three k-steps at most: 450 items 19.6 against 17.4, 1800 items 57
// against 65), but it holds the SMs that the algebraic kernels and the filter's
// second chain run on beside it.  Lines at 2, 3, 4, 5 items per SM (d_r at 5), RK4 step,
// us: 25 x 20 x 40 points 545 / 541 / 542 / 541, 33 x 24 x 48 points 797 / 787 / 786 / 794, 17 x
// 48 x 96 points 1449 / 1449 / 1448 / 1476, right-hand side of 25 x 24 x 48 points 113 / 113 /
// 119 / 119; d_r at 3: 25 x 28 x 56 points 894 against 882.
static bool runs_persistent(const cffyn_shell* sh, int rows, long long items, bool dr = false) {
  return items > (rows != 48 ? 1 : dr ? 5 : 3) * (long long)sh->sm_count;
}

// Mixed path: one launch of the tcgen05 core over the classes of b (same row
// group size, same input storage).
static int launch_batch(const cffyn_shell* sh, const TcBatch& b0, cudaStream_t st, int pairing, bool in_pairs,
                        const int* exps, int* flag = nullptr) {
  if (!flag) flag = sh->flag;
  TcBatch b = b0;
  b.wait_ns = sh->tc_wait_ns;
  long long items = 0;
  for (int c = 0; c < b.nclass; ++c) {
    b.first[c] = (int)items;
    items += (long long)b.tiles[c] * b.W[c].ngroups * (b.a[c].batched_m ? b.nm : 1);
  }
  if (items == 0) return CFFYN_OK;
  if (items >= (1ll << 31)) {
    set_error("operator launch of %lld tiles", items);
    return CFFYN_EINVAL;
  }
  for (int c = b.nclass; c <= kMaxBatch; ++c) b.first[c] = (int)items;
  const int rows = b.W[0].rows;
  // d_r (one class, one row group): the instance with the staged epilogue
  const bool dr = b.nclass == 1 && b.a[0].kind == OP_R && b.W[0].ngroups == 1;
  const int P = b.a[0].g.P, out_bytes = kTcCols * P * (int)sizeof(double);
  // d_r's tiles beside the persistent kernel's ring: with more than 80 rows there is no
  // room for them, and lanes that store words a line apart lose more than the kernel
  // gains, so the one-item kernel, which stages them, keeps these launches (d_r of a
  // step, us: 90 x 32 x 64 points 111 against 121, 81 x 14 x 28 35 against 42, 96 x 64 x
  // 128 488 against 492; derivatives of FP64 words there 2096 against 2066)
  const int ring = rows == 48 ? WsCfg<48>::kStage * kRingStages<48, 1> : WsCfg<96>::kStage * kRingStages<96, 1>;
  const bool persistent = runs_persistent(sh, rows, items, dr) && (!dr || ring + out_bytes <= kTcMaxSmem);
  const int stage = !dr ? 0 : persistent && rows == 48 && (P & 1) && P <= kRawRows ? 2 : 1;
#define CFFYN_LAUNCH_WS(R_, FI_, ST_)                                                                        \
  k_op_ws<FI_, R_, ST_><<<sh->sm_count, kWsThreads, kRingStages<R_, ST_> * WsCfg<R_>::kStage + ST_ * out_bytes, st>>>( \
      b, exps, pairing, flag)
#define CFFYN_LAUNCH_TC(R_, FI_, ST_) \
  k_op_tc<FI_, R_, ST_><<<(unsigned)items, TcCfg<R_>::kThreads, TcCfg<R_>::kSmem, st>>>(b, exps, pairing, flag)
#define CFFYN_LAUNCH_OP(FI_)                                                                                       \
  if (!persistent && rows == 48)                                                                                   \
    stage ? CFFYN_LAUNCH_TC(48, FI_, true) : CFFYN_LAUNCH_TC(48, FI_, false);                                      \
  else if (!persistent)                                                                                            \
    stage ? CFFYN_LAUNCH_TC(96, FI_, true) : CFFYN_LAUNCH_TC(96, FI_, false);                                      \
  else if (rows == 48)                                                                                             \
    stage == 0 ? CFFYN_LAUNCH_WS(48, FI_, 0) : stage == 1 ? CFFYN_LAUNCH_WS(48, FI_, 1) : CFFYN_LAUNCH_WS(48, FI_, 2); \
  else                                                                                                             \
    stage == 0 ? CFFYN_LAUNCH_WS(96, FI_, 0) : CFFYN_LAUNCH_WS(96, FI_, 1)
  if (in_pairs) {
    CFFYN_LAUNCH_OP(true);
  } else {
    CFFYN_LAUNCH_OP(false);
  }
#undef CFFYN_LAUNCH_OP
#undef CFFYN_LAUNCH_TC
#undef CFFYN_LAUNCH_WS
  count_launch();
  CF_CUDA(cudaGetLastError());
  return CFFYN_OK;
}

// FP64 core, or on the mixed path the tcgen05 core with the per-field
// exponents of the input at exps (op_prepare fills sh->exps); in_pairs: the
// input is pair-stored.  Mixed-path outputs are pair-stored.  flag: the
// status word a timed-out wait of the tcgen05 core marks (sh->flag if NULL).
static int launch(const cffyn_shell* sh, const OpArgs& a, const double* W64, const TcOp* Wt, dim3 extra,
                  cudaStream_t st, int pairing, bool in_pairs, const int* exps = nullptr, int eoff = 0,
                  int sum6 = 1, int* flag = nullptr) {
  if (a.g.ncols <= 0) return CFFYN_OK;
  if (sh->d.precision == CFFYN_FP64 || Wt == nullptr) {
    const unsigned gx = (unsigned)((a.g.ncols + F64_QT - 1) / F64_QT);
    const int nt = (a.g.P + 8 * F64_MAX_RP - 1) / (8 * F64_MAX_RP);        // row tiles
    const int rp = ((a.g.P + nt - 1) / nt + 7) / 8;                        // rows per warp
    const unsigned gy = (unsigned)((a.g.P + 8 * rp - 1) / (8 * rp));
    const size_t smem = (size_t)(8 * rp * a.g.K + a.g.K * F64_QT) * sizeof(double);
    const dim3 grid(gx, gy, extra.y);
    switch (rp) {
#define CFFYN_FP64_CASE(RP_)                                 \
  case RP_: k_op_fp64<RP_><<<grid, 256, smem, st>>>(a, W64); break;
      CFFYN_FP64_CASE(1)
      CFFYN_FP64_CASE(2)
      CFFYN_FP64_CASE(3)
      CFFYN_FP64_CASE(4)
      CFFYN_FP64_CASE(5)
      CFFYN_FP64_CASE(6)
      CFFYN_FP64_CASE(7)
      CFFYN_FP64_CASE(8)
#undef CFFYN_FP64_CASE
    }
    count_launch();
    CF_CUDA(cudaGetLastError());
    return CFFYN_OK;
  }
  TcBatch b;
  memset(&b, 0, sizeof(b));
  b.a[0] = a;
  b.W[0] = *Wt;
  b.tiles[0] = tiles_of(a);
  b.nclass = 1;
  b.nm = (int)extra.y;
  b.eoff = eoff;
  b.sum6 = sum6;
  return launch_batch(sh, b, st, pairing, in_pairs, exps ? exps : sh->exps, flag);
}

int set_op_smem_limits() {
  const void* f64[] = {(const void*)k_op_fp64<1>, (const void*)k_op_fp64<2>, (const void*)k_op_fp64<3>,
                       (const void*)k_op_fp64<4>, (const void*)k_op_fp64<5>, (const void*)k_op_fp64<6>,
                       (const void*)k_op_fp64<7>, (const void*)k_op_fp64<8>};
  for (const void* f : f64) CF_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
#define CFFYN_TC_INSTANCES(FI_)                                                                                   \
  (const void*)k_op_tc<FI_, 48, false>, (const void*)k_op_tc<FI_, 48, true>, (const void*)k_op_tc<FI_, 96, false>, \
      (const void*)k_op_tc<FI_, 96, true>, (const void*)k_op_ws<FI_, 48, 0>, (const void*)k_op_ws<FI_, 48, 1>,      \
      (const void*)k_op_ws<FI_, 48, 2>, (const void*)k_op_ws<FI_, 96, 0>, (const void*)k_op_ws<FI_, 96, 1>
  const void* tcs[] = {CFFYN_TC_INSTANCES(true), CFFYN_TC_INSTANCES(false)};
#undef CFFYN_TC_INSTANCES
  for (const void* f : tcs)
    CF_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcMaxSmem));
  return CFFYN_OK;
}

// Per-field exponents of nf fields of len values each into exps (max(nf, 64)
// words; clear: also the words from nf on, which a caller uses, are zeroed);
// in_pairs: pair-stored input.
static int field_exps(const double* in, bool in_pairs, int nf, long long len, int* exps, cudaStream_t st,
                      bool clear = false) {
  const long long* x = reinterpret_cast<const long long*>(in);
  if (len <= kExpShortLen && !clear) {
    if (in_pairs)
      k_field_exp_short<true><<<nf, kExpShortThreads, 0, st>>>(x, len, exps);
    else
      k_field_exp_short<false><<<nf, kExpShortThreads, 0, st>>>(x, len, exps);
    count_launch();
    CF_CUDA(cudaGetLastError());
    return CFFYN_OK;
  }
  // the words are atomicMax targets
  CF_CUDA(cudaMemsetAsync(exps, 0, sizeof(int) * std::max(nf, 64), st));
  const unsigned bx = (unsigned)((len + kExpThreads * kExpPerThread - 1) / (kExpThreads * kExpPerThread));
  if (in_pairs)
    k_field_exp<true><<<dim3(bx, nf), kExpThreads, 0, st>>>(x, len, exps);
  else
    k_field_exp<false><<<dim3(bx, nf), kExpThreads, 0, st>>>(x, len, exps);
  count_launch();
  CF_CUDA(cudaGetLastError());
  return CFFYN_OK;
}

// Mixed path (no-op on the FP64 path): the per-field exponents of the next
// operator input into sh->exps.
int op_prepare(const cffyn_shell* sh, const double* in, bool in_pairs, int nf, long long len, int pairing,
               cudaStream_t st) {
  (void)pairing;  // pairing is applied by the operator kernel
  if (sh->d.precision != CFFYN_MIXED) return CFFYN_OK;
  return field_exps(in, in_pairs, nf, len, sh->exps, st);
}

static OpArgs base_args(const cffyn_shell* sh) {
  OpArgs a;
  memset(&a, 0, sizeof(a));
  a.n_r = sh->n_r;
  a.N = sh->N;
  a.J = sh->J;
  a.R = sh->R;
  a.L = sh->Lrows;  // row of b_1 minus 1 in the DFT coefficient layout
  a.ns = sh->ns;
  return a;
}

// d_r (which = 0), d_theta over the double cover (1), d_phi (2) of nf fields:
// in/out [nf][P]
static OpArgs deriv_args(const cffyn_shell* sh, int which, const double* in, double* out, int nf) {
  OpArgs a = base_args(sh);
  a.in = in;
  a.out = out;
  if (which == 0) {
    a.kind = OP_R;
    a.g.K = a.g.K0 = a.g.P = a.g.P0 = sh->n_r;
    a.g.in_rs = a.g.out_rs = 1;
    a.g.ncols = (long long)nf * sh->J * sh->N;
  } else if (which == 1) {
    a.kind = OP_THETA;
    a.g.K = a.g.P = 2 * sh->N;
    a.g.K0 = a.g.P0 = sh->N;
    a.g.rev1 = 1;
    a.g.in_rs = a.g.out_rs = sh->n_r;
    a.g.ncols = (long long)nf * (sh->J / 2) * sh->n_r;
  } else {
    a.kind = OP_ROWS;
    a.Q = sh->N * sh->n_r;
    a.in_bs = a.out_bs = (long long)sh->P;
    a.g.K = a.g.K0 = a.g.P = a.g.P0 = sh->J;
    a.g.in_rs = a.g.out_rs = a.Q;
    a.g.ncols = (long long)nf * a.Q;
  }
  return a;
}

int op_deriv_r(const cffyn_shell* sh, const double* in, double* out, int nfields, bool in_pairs,
               cudaStream_t st) {
  return launch(sh, deriv_args(sh, 0, in, out, nfields), sh->Dr, &sh->tDr, dim3(1, 1), st, 0, in_pairs);
}

static int op_deriv_theta(const cffyn_shell* sh, const double* in, double* out, int nfields, bool in_pairs,
                   cudaStream_t st) {
  return launch(sh, deriv_args(sh, 1, in, out, nfields), sh->Dth2, &sh->tDth2, dim3(1, 1), st, 0, in_pairs);
}

static int op_deriv_phi(const cffyn_shell* sh, const double* in, double* out, int nfields, bool in_pairs,
                 cudaStream_t st) {
  return launch(sh, deriv_args(sh, 2, in, out, nfields), sh->Dph, &sh->tDph, dim3(1, 1), st, 0, in_pairs);
}

// d_theta and d_phi of nf fields (same input; both operators have 2N rows):
// one launch of the tcgen05 core on the mixed path, so that the two share
// the last, partly filled wave of CTAs; two launches on the FP64 path.
int op_deriv_theta_phi(const cffyn_shell* sh, const double* in, double* out_th, double* out_ph, int nf,
                       bool in_pairs, cudaStream_t st) {
  if (sh->d.precision != CFFYN_MIXED || sh->tDth2.rows != sh->tDph.rows) {
    int rc = op_deriv_theta(sh, in, out_th, nf, in_pairs, st);
    return rc ? rc : op_deriv_phi(sh, in, out_ph, nf, in_pairs, st);
  }
  TcBatch b;
  memset(&b, 0, sizeof(b));
  b.a[0] = deriv_args(sh, 1, in, out_th, nf);
  b.W[0] = sh->tDth2;
  b.a[1] = deriv_args(sh, 2, in, out_ph, nf);
  b.W[1] = sh->tDph;
  for (int c = 0; c < 2; ++c) b.tiles[c] = tiles_of(b.a[c]);
  b.nclass = 2;
  b.nm = 1;
  b.sum6 = 1;
  return launch_batch(sh, b, st, 0, in_pairs, sh->exps);
}

// Whether the phi analysis of nf arrays runs on the persistent kernel: each of
// its launches then fills the device by itself.
bool op_dft_persistent(const cffyn_shell* sh, int nf) {
  const long long tiles = ((long long)nf * sh->N * sh->n_r + kTcCols - 1) / kTcCols;
  return sh->d.precision == CFFYN_MIXED && runs_persistent(sh, sh->tFan.rows, tiles * sh->tFan.ngroups);
}

static int op_rows(const cffyn_shell* sh, const double* in, double* out, int nb, int K, int P,
                   long long in_bs, long long out_bs, const double* W, const TcOp* Wt, cudaStream_t st,
                   int pairing, int eoff = 0, int fld0 = 0) {
  OpArgs a = base_args(sh);
  a.kind = OP_ROWS;
  a.fld0 = fld0;
  a.in = in;
  a.out = out;
  a.Q = sh->N * sh->n_r;
  a.in_bs = in_bs;
  a.out_bs = out_bs;
  a.g.K = a.g.K0 = K;
  a.g.P = a.g.P0 = P;
  a.g.in_rs = a.g.out_rs = a.Q;
  a.g.ncols = (long long)nb * a.Q;
  // the phi DFTs of the filter: digit sums up to 5 suffice (filter errors
  // stay near 1e-12 relative)
  return launch(sh, a, W, Wt, dim3(1, 1), st, pairing, true, nullptr, eoff, 0);
}

// phi analysis: S[f][j][i][k] -> C[f][row][i][k] (pair-stored input on the
// mixed path) of the nf arrays f0 .. f0 + nf - 1; pairing: the exponents of
// slot pairs (f, f ^ 1) are shared (the complex slots of the Yn filter)
int op_dft_fwd(const cffyn_shell* sh, const double* in, double* out, int nf, cudaStream_t st, int pairing,
               int f0) {
  long long Q = (long long)sh->N * sh->n_r;
  return op_rows(sh, in + (size_t)f0 * sh->J * Q, out + (size_t)f0 * sh->R * Q, nf, sh->J, sh->R,
                 (long long)sh->J * Q, (long long)sh->R * Q, sh->Fan, &sh->tFan, st, pairing, 0, f0);
}

// eoff: see TcBatch (the coefficients' exponents are bounds, not a scan)
int op_dft_inv(const cffyn_shell* sh, const double* in, double* out, int nf, cudaStream_t st, int pairing,
               int eoff, int f0) {
  long long Q = (long long)sh->N * sh->n_r;
  return op_rows(sh, in + (size_t)f0 * sh->R * Q, out + (size_t)f0 * sh->J * Q, nf, sh->R, sh->J,
                 (long long)sh->R * Q, (long long)sh->J * Q, sh->Fsy, &sh->tFsy, st, pairing, eoff, f0);
}

// Component-wise filters (Sec. 3.5): every field's coefficients projected
// with F^0_m, C -> C2: the Y filter at the retained degree L (one class), the
// graded Yg filter at L + d for the fields of spatial degree d (eq. nfofmu;
// one class per d), m = 0..Lrows; one launch on the mixed path.
int op_project_scalar(const cffyn_shell* sh, const double* C, double* C2, cudaStream_t st, int eoff) {
  const int N = sh->N;
  const bool graded = sh->d.filter_kind == CFFYN_FILTER_YG;
  const int nm = sh->Lrows + 1;
  OpArgs cls[4];
  const double* W64[4];
  const TcOp* Wt[4];
  int ncls = 0, off = 0;
  for (int d = 0; d < 4; ++d) {
    if (sh->ny[d] <= 0) continue;
    OpArgs a = base_args(sh);
    a.in = C;
    a.out = C2;
    a.kind = OP_PROJ0;
    a.slots = sh->yslots + off;
    a.nslots = sh->ny[d];
    a.batched_m = 1;
    a.w_stride = (long long)N * N;
    a.g.K = a.g.K0 = a.g.P = a.g.P0 = N;
    a.g.in_rs = a.g.out_rs = sh->n_r;
    a.g.ncols = (long long)sh->ny[d] * 2 * sh->n_r * sh->ns;
    off += sh->ny[d];
    cls[ncls] = a;
    W64[ncls] = graded ? sh->F0g + (size_t)d * nm * N * N : sh->Fproj0;
    Wt[ncls++] = graded ? &sh->tF0g[d] : &sh->tF0;
  }
  if (sh->d.precision == CFFYN_MIXED) {
    TcBatch bt;
    memset(&bt, 0, sizeof(bt));
    for (int c = 0; c < ncls; ++c) {
      bt.a[c] = cls[c];
      bt.W[c] = *Wt[c];
      bt.tiles[c] = tiles_of(cls[c]);
    }
    bt.nclass = ncls;
    bt.nm = nm;
    bt.eoff = eoff;
    bt.sum6 = 0;
    return launch_batch(sh, bt, st, 0, true, sh->exps);
  }
  for (int c = 0; c < ncls; ++c) {
    int rc = launch(sh, cls[c], W64[c], Wt[c], dim3(1, nm), st, 0, true);
    if (rc) return rc;
  }
  return CFFYN_OK;
}

// Projection of all spin classes, coefficients C -> C2 (same layout): every
// class and every m = 0..L in one launch on the mixed path, one launch per
// class on the FP64 path.
int op_project(const cffyn_shell* sh, const double* C, double* C2, const int* slots_r0, int n_r0,
               const int* const slots_c[3], const int n_c[3], cudaStream_t st, int eoff) {
  const int N = sh->N;
  const int nm = sh->L + 1;
  OpArgs cls[4];
  const double* W64[4];
  const TcOp* Wt[4];
  int ncls = 0;
  if (n_r0 > 0) {
    OpArgs a = base_args(sh);
    a.in = C;
    a.out = C2;
    a.kind = OP_PROJ0;
    a.slots = slots_r0;
    a.nslots = n_r0;
    a.batched_m = 1;
    a.w_stride = (long long)N * N;
    a.g.K = a.g.K0 = a.g.P = a.g.P0 = N;
    a.g.in_rs = a.g.out_rs = sh->n_r;
    a.g.ncols = (long long)n_r0 * 2 * sh->n_r * sh->ns;
    cls[ncls] = a;
    W64[ncls] = sh->Fproj0;
    Wt[ncls++] = &sh->tF0;
  }
  for (int s = 0; s < 3; ++s) {
    if (n_c[s] <= 0) continue;
    OpArgs b = base_args(sh);
    b.in = C;
    b.out = C2;
    b.kind = OP_PROJC;
    b.slots = slots_c[s];
    b.nslots = n_c[s];
    b.batched_m = 1;
    b.w_stride = (long long)N * 2 * N;
    b.g.K = 2 * N;
    b.g.K0 = N;
    b.g.P = b.g.P0 = N;
    b.g.in_rs = b.g.out_rs = sh->n_r;
    b.g.ncols = (long long)n_c[s] * 4 * sh->n_r * sh->ns;
    cls[ncls] = b;
    W64[ncls] = sh->FprojC + (size_t)s * nm * N * 2 * N;
    Wt[ncls++] = &sh->tFC[s];
  }
  if (sh->d.precision == CFFYN_MIXED) {
    // every class of the projection in one launch (all have N rows)
    TcBatch bt;
    memset(&bt, 0, sizeof(bt));
    for (int c = 0; c < ncls; ++c) {
      bt.a[c] = cls[c];
      bt.W[c] = *Wt[c];
      bt.tiles[c] = tiles_of(cls[c]);
    }
    bt.nclass = ncls;
    bt.nm = nm;
    bt.eoff = eoff;
    bt.sum6 = 0;
    return launch_batch(sh, bt, st, 1, true, sh->exps);
  }
  for (int c = 0; c < ncls; ++c) {
    int rc = launch(sh, cls[c], W64[c], Wt[c], dim3(1, nm), st, 1, true);
    if (rc) return rc;
  }
  return CFFYN_OK;
}

// Spherical derivatives of nf fields (FP64 input) into D = [3][nf][P], with the
// mixed path's per-field exponents (64 ints) at exps instead of the shell's
// workspace; exps is zeroed here on st (its words are atomicMax targets).
// A timed-out wait of the tcgen05 core sets bit 2 of *flag (not of the
// shell's own status word).  The FP64 path uses neither.  Same kernels and
// arithmetic as op_prepare followed by op_deriv_r / op_deriv_theta /
// op_deriv_phi.
int op_derivs_at(const cffyn_shell* sh, const double* u, double* D, int nf, int* exps, int* flag,
                 cudaStream_t st) {
  const long long P = (long long)sh->P;
  const bool mixed = sh->d.precision == CFFYN_MIXED;
  int rc;
  if (mixed && (rc = field_exps(u, false, nf, P, exps, st, true))) return rc;
  const double* W64[3] = {sh->Dr, sh->Dth2, sh->Dph};
  const TcOp* Wt[3] = {&sh->tDr, &sh->tDth2, &sh->tDph};
  for (int i = 0; i < 3; ++i)
    if ((rc = launch(sh, deriv_args(sh, i, u, D + i * nf * P, nf), W64[i], Wt[i], dim3(1, 1), st, 0, false,
                     exps, 0, 1, flag)))
      return rc;
  return CFFYN_OK;
}

}  // namespace cffyn
