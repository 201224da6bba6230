// GHG right-hand side (paper App. A.1, eqs. gdot, Phidot, Pidot; gamma_0 =
// gamma_2 = 1, gamma_1 = -1) with the freeze-incoming boundary condition of
// App. A.2, as three pointwise kernels so that none of them spills registers
// (the state of one point alone is 50 values; in the double-float path that
// is 100 registers):
//
//   k_rhs_gamma  3+1 quantities (eqs. normal, abgfromgab), d_t g_ab (eq. gdot,
//                written as the first ten outputs), Christoffel symbols from
//                undifferentiated fields (eq. Gamma), Gamma_c, the gauge
//                constraint C_a = H_a + Gamma_a, nabla_(a H_b), and the
//                Gamma-Gamma term of eq. Pidot -> partial source of d_t Pi.
//   k_rhs_quad   the Phi-Phi and Pi-Pi terms of eq. Pidot, the remaining
//                algebraic terms of eqs. Pidot and Phidot -> sources.
//   k_rhs_pp     principal parts -A^k d_k u from the spherical derivatives,
//                with the chain rule (eq. dvdx) contracted into the shift and
//                inverse metric once per point, plus the boundary condition
//                on the outermost sphere.
//   k_gauge_rhs  54/58-field states only, ahead of k_rhs_gamma: H_a and its
//                derivatives from the state, and the gauge fields' own
//                right-hand sides.
//
// Source buffer src[50][P]: [0,10) source of d_t Pi_ab, [10,40) source of
// d_t Phi_iab (10 + 10 i + s), 40 alpha, [41,44) beta^i, [44,50) gamma^ij
// (xx, xy, xz, yy, yz, zz).
#include "pw_common.cuh"

namespace cffyn {

int pw_to_internal(const cffyn_shell*, const double*, double*, long long, cudaStream_t);  // pointwise.cu

template <class T, bool F>
__device__ __forceinline__ T ldA(const double* a, long long P, long long p, int f) {
  return Store<T, F>::ld(a, (long long)f * P + p);
}
// of an array that the kernel also writes (see Store)
template <class T, bool F>
__device__ __forceinline__ T ldA_rw(const double* a, long long P, long long p, int f) {
  return Store<T, F>::ld_rw(a, (long long)f * P + p);
}
template <class T, bool F>
__device__ __forceinline__ void stA(double* a, long long P, long long p, int f, T v) {
  Store<T, F>::st(a, (long long)f * P + p, v);
}
// internal buffers are pair-stored in the double-float path
template <class T> constexpr bool kInt = false;
template <> constexpr bool kInt<ff> = true;

// Per-thread working tensors that rolled loops index at run time live in
// shared memory as [slot][thread] (consecutive threads, consecutive words: no
// bank conflicts); the outer contraction loops stay rolled so that the code
// of a kernel fits the instruction caches, the inner ones unrolled so that
// independent accumulations overlap.
template <class T, int NB>
struct Slots {
  T* s;
  __device__ __forceinline__ T& operator()(int v) const { return s[v * NB + (int)threadIdx.x]; }
};

// Gamma_cab = (d_a g_bc + d_b g_ac - d_c g_ab) / 2; dg4(c, s) = d_c g of pair s.  The
// terms that cancel or are equal are not summed: 500 instructions for the 40
// symbols of a point, not 960.
template <class T, class DG>
__device__ __forceinline__ T gamma_cab(int c, int a, int b, DG&& dg4) {
  if (c == a) return half_of(dg4(b, SI(a, a)));
  if (c == b) return half_of(dg4(a, SI(b, b)));
  const T two = a == b ? twice(dg4(a, SI(a, c))) : dg4(a, SI(b, c)) + dg4(b, SI(a, c));
  return half_of(two - dg4(c, SI(a, b)));
}

// n^d A_cd of a symmetric A(pair) for all c, and n^c n^d A_cd
template <class T, class A>
__device__ __forceinline__ T normal_row(const T (&nu)[4], T (&row)[4], A&& pair) {
  Acc<T> nn;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    Acc<T> acc;
#pragma unroll
    for (int d = 0; d < 4; ++d) acc.fma_(nu[d], pair(SI(c, d)));
    row[c] = acc.get();
    nn.fma_(nu[c], row[c]);
  }
  return nn.get();
}

constexpr int kRhsBlock = 128;
constexpr int kGamSlots = 44;   // Gamma_cab (c*10 + s) | C_a 40..43
constexpr int kQuadSlots = 40;  // Pi 0..9 | Phi_iab 10 + 10 i + s

// Bound by instruction issue (two thirds of the slots; 10750 instructions per
// point, most of them the pair sums).  Four blocks per SM: 128 registers, 44 KB of
// slots (five blocks of 96 registers: 72 against 67 us for 33 x 48 x 96 points);
// g_ab is read again from u where the gauge terms need it.  A pair's gauge terms
// are formed where its quadratic term is: in a loop of their own they waited for
// their words (71 us).  81 us before that and the shorter pair sums (Acc, half_of,
// gamma_cab).
template <class T, bool FU, bool FO>
__global__ void __launch_bounds__(kRhsBlock, 4) k_rhs_gamma(const double* __restrict__ u,
                                                         const double* __restrict__ H,
                                                         const double* __restrict__ dH,
                                                         double* __restrict__ src, double* __restrict__ out,
                                                         Geo geo, int dtH) {
  __shared__ T sm[kGamSlots * kRhsBlock];
  const Slots<T, kRhsBlock> V{sm};
  const long long P = geo.P;
  const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p >= P) return;
  const T zero = S<T>::c(0.0);

  Metric<T> M;
  {
    T g[10];
#pragma unroll
    for (int s = 0; s < 10; ++s) {
      g[s] = ldA<T, FU>(u, P, p, s);
    }
    metric_from(g, M);
  }
  stA<T, kInt<T>>(src, P, p, 40, M.alpha);
#pragma unroll
  for (int x = 0; x < 3; ++x) stA<T, kInt<T>>(src, P, p, 41 + x, M.bu[x]);
  stA<T, kInt<T>>(src, P, p, 44, M.gi[0][0]);
  stA<T, kInt<T>>(src, P, p, 45, M.gi[0][1]);
  stA<T, kInt<T>>(src, P, p, 46, M.gi[0][2]);
  stA<T, kInt<T>>(src, P, p, 47, M.gi[1][1]);
  stA<T, kInt<T>>(src, P, p, 48, M.gi[1][2]);
  stA<T, kInt<T>>(src, P, p, 49, M.gi[2][2]);

  // d_t g_ab (eq. gdot) and the Christoffel symbols Gamma_cab
  {
    T dtg[10], Ph[3][10];
#pragma unroll
    for (int s = 0; s < 10; ++s) {
#pragma unroll
      for (int x = 0; x < 3; ++x) Ph[x][s] = ldA<T, FU>(u, P, p, 20 + 10 * x + s);
      Acc<T> a;
#pragma unroll
      for (int x = 0; x < 3; ++x) a.fma_(M.bu[x], Ph[x][s]);
      a.fma_(-M.alpha, ldA<T, FU>(u, P, p, 10 + s));
      dtg[s] = a.get();
      stA<T, FO>(out, P, p, s, dtg[s]);
    }
    auto dg4 = [&](int c, int s) -> T { return c == 0 ? dtg[s] : Ph[c - 1][s]; };
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = a; b < 4; ++b)
          V(c * 10 + SI(a, b)) = gamma_cab<T>(c, a, b, dg4);
  }
  // Gamma_c = g^ab Gamma_cab (symmetric pairs counted twice off the diagonal);
  // gauge constraint C_c = H_c + Gamma_c, H^c, n^c C_c
  T Hup[4], nC;
  {
    T Hd[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) Hd[a] = ldA<T, kInt<T>>(H, P, p, a);
    Acc<T> an;
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
      Acc<T> acc;
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = a; b < 4; ++b) {
          const T w = (a == b) ? M.gi4[SI(a, b)] : twice(M.gi4[SI(a, b)]);
          acc.fma_(w, V(c * 10 + SI(a, b)));
        }
      const T hc = c == 0 ? Hd[0] : (c == 1 ? Hd[1] : (c == 2 ? Hd[2] : Hd[3]));
      acc.add(hc);
      V(40 + c) = acc.get();
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      Acc<T> acc;
#pragma unroll
      for (int d = 0; d < 4; ++d) acc.fma_(M.gi4[SI(c, d)], Hd[d]);
      Hup[c] = acc.get();
      an.fma_(M.nu[c], V(40 + c));
    }
    nC = an.get();
  }
  // the sources with larger index b
  const T twoal = M.alpha + M.alpha, m2al = -twoal;
  const T aa = M.alpha * (-M.alpha);  // alpha n_0, n_a = (-alpha, 0, 0, 0)
  const T anC = M.alpha * nC;
#pragma unroll 1
  for (int b = 0; b < 4; ++b) {
    const SymRow rb(b);
    T Gce[10];  // Gamma_b^{ce}, symmetric, off-diagonal weight 2
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      T Gcf[4];  // Gamma_b^c_f = g^cd Gamma_bdf
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        Acc<T> acc;
#pragma unroll
        for (int d = 0; d < 4; ++d) acc.fma_(M.gi4[SI(c, d)], V(b * 10 + SI(d, f)));
        Gcf[f] = acc.get();
      }
#pragma unroll
      for (int e = c; e < 4; ++e) {
        Acc<T> acc;
#pragma unroll
        for (int f = 0; f < 4; ++f) acc.fma_(M.gi4[SI(e, f)], Gcf[f]);
        Gce[SI(c, e)] = (c == e) ? acc.get() : twice(acc.get());
      }
    }
#pragma unroll 1
    for (int a = 0; a <= b; ++a) {
      const int s = rb(a);
      // S_Pi = -2 alpha nabla_(a H_b) + alpha (n_b C_a + n_a C_b - g_ab n^c C_c);
      // d_a H_b: rows (x, b) = 4 x + b of dH for a = x + 1; d_t H_b is row 12 + b
      // when the gauge source is evolved with its time derivative (58 fields),
      // else zero
      const T dHab = a == 0 ? (dtH ? ldA<T, kInt<T>>(dH, P, p, 12 + b) : zero)
                            : ldA<T, kInt<T>>(dH, P, p, (a - 1) * 4 + b);
      const T dHba = b == 0 ? (dtH ? ldA<T, kInt<T>>(dH, P, p, 12 + a) : zero)
                            : ldA<T, kInt<T>>(dH, P, p, (b - 1) * 4 + a);
      const T gab = ldA<T, FU>(u, P, p, s);
      // -2 alpha g^cd g^ef Gamma_ace Gamma_bdf
      Acc<T> qa;
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int e = c; e < 4; ++e) qa.fma_(V(a * 10 + SI(c, e)), Gce[SI(c, e)]);
      Acc<T> acc;
      acc.add(half_of(dHab + dHba));
#pragma unroll
      for (int c = 0; c < 4; ++c) acc.fma_(-V(c * 10 + s), Hup[c]);
      const T DH = acc.get();
      Acc<T> v;
      v.fma_(-twoal, DH);
      v.fma_(-(anC), gab);
      if (a == 0) v.fma_(aa, V(40 + b));
      if (b == 0) v.fma_(aa, V(40 + a));
      Acc<T> r;
      r.add(v.get());
      r.fma_(m2al, qa.get());
      stA<T, kInt<T>>(src, P, p, s, r.get());
    }
  }
}

// The Phi-Phi and Pi-Pi terms of eq. Pidot and the remaining algebraic terms
// of eqs. Pidot and Phidot; alpha, beta^i, gamma^ij come from k_rhs_gamma.
// Bound by instruction issue (11660 per point); 33 x 48 x 96 points: 66 us, with each
// pair's quadratic terms kept in ten more slots for a second loop 69, with the
// selects of SI in the rolled loops 86 (see SymRow), with n^c n^d A_cd from sixteen
// products 74; five blocks per SM (96 registers) 75.
template <class T, bool FU>
__global__ void __launch_bounds__(kRhsBlock, 4) k_rhs_quad(const double* __restrict__ u, double* __restrict__ src,
                                                        Geo geo) {
  __shared__ T sm[kQuadSlots * kRhsBlock];
  const Slots<T, kRhsBlock> V{sm};
  const long long P = geo.P;
  const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p >= P) return;
  // 3+1 quantities (eqs. normal, abgfromgab) as k_rhs_gamma derived them
  const T alpha = ldA<T, kInt<T>>(src, P, p, 40);
  T bu[3], gi[3][3];
#pragma unroll
  for (int x = 0; x < 3; ++x) bu[x] = ldA<T, kInt<T>>(src, P, p, 41 + x);
  gi[0][0] = ldA<T, kInt<T>>(src, P, p, 44);
  gi[0][1] = gi[1][0] = ldA<T, kInt<T>>(src, P, p, 45);
  gi[0][2] = gi[2][0] = ldA<T, kInt<T>>(src, P, p, 46);
  gi[1][1] = ldA<T, kInt<T>>(src, P, p, 47);
  gi[1][2] = gi[2][1] = ldA<T, kInt<T>>(src, P, p, 48);
  gi[2][2] = ldA<T, kInt<T>>(src, P, p, 49);
  const T ialpha = S<T>::c(1.0) / alpha;
  const T ia2 = ialpha * ialpha;
  T nu[4], gi4[10];
  nu[0] = ialpha;
#pragma unroll
  for (int i = 0; i < 3; ++i) nu[i + 1] = -(bu[i] * ialpha);
  gi4[0] = -ia2;
#pragma unroll
  for (int i = 0; i < 3; ++i) gi4[SI(0, i + 1)] = bu[i] * ia2;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) gi4[SI(i + 1, j + 1)] = gi[i][j] - bu[i] * bu[j] * ia2;

#pragma unroll
  for (int s = 0; s < 10; ++s) {
    V(s) = ldA<T, FU>(u, P, p, 10 + s);
#pragma unroll
    for (int x = 0; x < 3; ++x) V(10 + 10 * x + s) = ldA<T, FU>(u, P, p, 20 + 10 * x + s);
  }
  const T twoal = alpha + alpha;
  const T hal = half_of(alpha);
  {
    T nnPi, cPh[3];  // n^c n^d Pi_cd; beta^j - alpha n^c Pi_ci gamma^ij
    {
      T nPi[4];
      nnPi = normal_row(nu, nPi, [&](int s) -> T { return V(s); });
#pragma unroll
      for (int y = 0; y < 3; ++y) {
        Acc<T> acc;
#pragma unroll
        for (int x = 0; x < 3; ++x) acc.fma_(nPi[x + 1], gi[x][y]);
        cPh[y] = bu[y] - alpha * acc.get();
      }
    }
    const T cPi = -(hal * nnPi);
    // the sources with larger index b: Q2_ab = Pi_ac g^cd Pi_db, Q1_ab = gamma^ij
    // g^cd Phi_iac Phi_jbd and the remaining algebraic terms of eq. Pidot
#pragma unroll 1
    for (int b = 0; b < 4; ++b) {
      const SymRow rb(b);
      T Piu[4], W[3][4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        Acc<T> acc;
#pragma unroll
        for (int d = 0; d < 4; ++d) acc.fma_(gi4[SI(c, d)], V(rb(d)));
        Piu[c] = acc.get();
        T Y[3];
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          Acc<T> ay;
#pragma unroll
          for (int d = 0; d < 4; ++d) ay.fma_(gi4[SI(c, d)], V(10 + 10 * x + rb(d)));
          Y[x] = ay.get();
        }
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          Acc<T> aw;
#pragma unroll
          for (int y = 0; y < 3; ++y) aw.fma_(gi[x][y], Y[y]);
          W[x][c] = aw.get();
        }
      }
#pragma unroll 1
      for (int a = 0; a <= b; ++a) {
        const SymRow ra(a);
        const int s = rb(a);
        Acc<T> q2;
#pragma unroll
        for (int c = 0; c < 4; ++c) q2.fma_(-V(ra(c)), Piu[c]);
        Acc<T> q;
        q.add(q2.get());
#pragma unroll
        for (int x = 0; x < 3; ++x)
#pragma unroll
          for (int c = 0; c < 4; ++c) q.fma_(V(10 + 10 * x + ra(c)), W[x][c]);
        Acc<T> acc;
        acc.add(ldA_rw<T, kInt<T>>(src, P, p, s));
        acc.fma_(twoal, q.get());
        acc.fma_(cPi, V(s));
#pragma unroll
        for (int x = 0; x < 3; ++x) acc.fma_(cPh[x], V(10 + 10 * x + s));
        stA<T, kInt<T>>(src, P, p, s, acc.get());
      }
    }
  }
  // algebraic terms of eq. Phidot
#pragma unroll 1
  for (int x = 0; x < 3; ++x) {
    T nnPhi, Mk[3];  // n^c n^d Phi_xcd; alpha gamma^jk n^c Phi_x,j,c less alpha delta^k_x
    {
      T nP[4];
      nnPhi = normal_row(nu, nP, [&](int s) -> T { return V(10 + 10 * x + s); });
#pragma unroll
      for (int z = 0; z < 3; ++z) {
        Acc<T> acc;
#pragma unroll
        for (int y = 0; y < 3; ++y) acc.fma_(nP[y + 1], gi[y][z]);
        Mk[z] = alpha * acc.get();
        if (z == x) Mk[z] = Mk[z] - alpha;
      }
    }
    const T hnn = hal * nnPhi;
#pragma unroll 1
    for (int s = 0; s < 10; ++s) {
      Acc<T> acc;
      acc.fma_(hnn, V(s));
#pragma unroll
      for (int z = 0; z < 3; ++z) acc.fma_(Mk[z], V(10 + 10 * z + s));
      stA<T, kInt<T>>(src, P, p, 10 + 10 * x + s, acc.get());
    }
  }
}

// k_rhs_gamma and k_rhs_quad for few points (rhs_shared): 32 points per block and
// four warps, each warp a share of every point's tensors.  One thread's chain
// through a whole point takes 30 and 25 us however few points there are; shared
// out it takes 11 and 10 (13 x 9 x 18; by now 15 and 14 against 9 and 8), at the
// price of barriers and repeated 3+1 quantities.  The tensors live in shared memory as [slot][point], written by
// one warp and read by all.  Every sum runs in the order of the kernels above:
// the results are bit-identical.
template <class T>
struct PointSlots {
  T* s;  // this point's column
  __device__ __forceinline__ T& operator()(int v) const { return s[v * 32]; }
};

// slots of k_rhs_gamma_shared: g^ab, beta^i, alpha, n^a, Pi, Phi_iab, d_t g_ab,
// Gamma_cab, C_a
constexpr int kGG4 = 0, kGBu = 10, kGAl = 13, kGNu = 14, kGPi = 18, kGPh = 28, kGDt = 58, kGGam = 68, kGC = 108,
              kGSlots = 112;

// Warp 0 forms the 3+1 quantities while the others fetch Pi and Phi; the warps
// share d_t g by component, Gamma_cab by c and the sources by b >= a.
template <class T, bool FU, bool FO>
__global__ void __launch_bounds__(kRhsBlock)
    k_rhs_gamma_shared(const double* __restrict__ u, const double* __restrict__ H, const double* __restrict__ dH,
                       double* __restrict__ src, double* __restrict__ out, Geo geo, int dtH) {
  __shared__ T sm[kGSlots * 32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const PointSlots<T> V{sm + lane};
  const long long P = geo.P;
  const long long q = blockIdx.x * 32ll + lane;
  const bool live = q < P;
  const long long p = live ? q : P - 1;  // the last block's spare threads follow its last point
  const T zero = S<T>::c(0.0);

  if (w == 0) {
    T g[10];
#pragma unroll
    for (int s = 0; s < 10; ++s) g[s] = ldA<T, FU>(u, P, p, s);
    Metric<T> M;
    metric_from(g, M);
#pragma unroll
    for (int s = 0; s < 10; ++s) V(kGG4 + s) = M.gi4[s];
#pragma unroll
    for (int x = 0; x < 3; ++x) V(kGBu + x) = M.bu[x];
    V(kGAl) = M.alpha;
#pragma unroll
    for (int c = 0; c < 4; ++c) V(kGNu + c) = M.nu[c];
    if (live) {
      stA<T, kInt<T>>(src, P, p, 40, M.alpha);
#pragma unroll
      for (int x = 0; x < 3; ++x) stA<T, kInt<T>>(src, P, p, 41 + x, M.bu[x]);
      stA<T, kInt<T>>(src, P, p, 44, M.gi[0][0]);
      stA<T, kInt<T>>(src, P, p, 45, M.gi[0][1]);
      stA<T, kInt<T>>(src, P, p, 46, M.gi[0][2]);
      stA<T, kInt<T>>(src, P, p, 47, M.gi[1][1]);
      stA<T, kInt<T>>(src, P, p, 48, M.gi[1][2]);
      stA<T, kInt<T>>(src, P, p, 49, M.gi[2][2]);
    }
  } else {
    T v[14];
#pragma unroll
    for (int s = 0; s < 10; ++s) v[s] = ldA<T, FU>(u, P, p, 10 + 10 * w + s);  // Phi_iab, i = w - 1
#pragma unroll
    for (int s = 0; s < 4; ++s)
      if (w - 1 + 3 * s < 10) v[10 + s] = ldA<T, FU>(u, P, p, 10 + w - 1 + 3 * s);
#pragma unroll
    for (int s = 0; s < 10; ++s) V(kGPh + 10 * (w - 1) + s) = v[s];
#pragma unroll
    for (int s = 0; s < 4; ++s)
      if (w - 1 + 3 * s < 10) V(kGPi + w - 1 + 3 * s) = v[10 + s];
  }
  // H_a for every warp, d_a H_b for the warp's sources: in flight over the barrier
  T Hd[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) Hd[a] = ldA<T, kInt<T>>(H, P, p, a);
  __syncthreads();
  const T alpha = V(kGAl);
  // d_t g_ab (eq. gdot)
#pragma unroll 1
  for (int s = w; s < 10; s += 4) {
    Acc<T> a;
#pragma unroll
    for (int x = 0; x < 3; ++x) a.fma_(V(kGBu + x), V(kGPh + 10 * x + s));
    a.fma_(-alpha, V(kGPi + s));
    const T d = a.get();
    V(kGDt + s) = d;
    if (live) stA<T, FO>(out, P, p, s, d);
  }
  T gi4[10];
#pragma unroll
  for (int s = 0; s < 10; ++s) gi4[s] = V(kGG4 + s);
  __syncthreads();
  // Christoffel symbols Gamma_cab, c = w; Gamma_c = g^ab Gamma_cab (symmetric pairs
  // counted twice off the diagonal) and the gauge constraint C_c = H_c + Gamma_c
  {
    const int c = w;
    auto dg4 = [&](int e, int s) -> T { return V((e == 0 ? kGDt : kGPh + 10 * (e - 1)) + s); };
    Acc<T> acc;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = a; b < 4; ++b) {
        const T G = gamma_cab<T>(c, a, b, dg4);
        V(kGGam + c * 10 + SI(a, b)) = G;
        const T wt = (a == b) ? gi4[SI(a, b)] : twice(gi4[SI(a, b)]);
        acc.fma_(wt, G);
      }
    acc.add(c == 0 ? Hd[0] : (c == 1 ? Hd[1] : (c == 2 ? Hd[2] : Hd[3])));
    V(kGC + c) = acc.get();
  }
  __syncthreads();
  // H^c, n^c C_c
  T Hup[4], nC;
  {
    Acc<T> an;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      Acc<T> acc;
#pragma unroll
      for (int d = 0; d < 4; ++d) acc.fma_(gi4[SI(c, d)], Hd[d]);
      Hup[c] = acc.get();
      an.fma_(V(kGNu + c), V(kGC + c));
    }
    nC = an.get();
  }
  // the sources with larger index b = w
  const int b = w;
  const SymRow rb(b);
  T Gce[10];  // Gamma_b^{ce}, symmetric, off-diagonal weight 2
  {
    T Gcf[4][4];  // Gamma_b^c_f = g^cd Gamma_bdf
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        Acc<T> acc;
#pragma unroll
        for (int d = 0; d < 4; ++d) acc.fma_(gi4[SI(c, d)], V(kGGam + b * 10 + SI(d, f)));
        Gcf[c][f] = acc.get();
      }
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int e = c; e < 4; ++e) {
        Acc<T> acc;
#pragma unroll
        for (int f = 0; f < 4; ++f) acc.fma_(gi4[SI(e, f)], Gcf[c][f]);
        Gce[SI(c, e)] = (c == e) ? acc.get() : twice(acc.get());
      }
  }
  const T twoal = alpha + alpha, m2al = -twoal;
  const T aa = alpha * (-alpha);  // alpha n_0, n_a = (-alpha, 0, 0, 0)
  const T anC = alpha * nC;
#pragma unroll 1
  for (int a = 0; a <= b; ++a) {
    const int s = rb(a);
    // S_Pi = -2 alpha nabla_(a H_b) + alpha (n_b C_a + n_a C_b - g_ab n^c C_c);
    // d_a H_b: rows (x, b) = 4 x + b of dH for a = x + 1; d_t H_b is row 12 + b
    // when the gauge source is evolved with its time derivative (58 fields),
    // else zero
    const T dHab = a == 0 ? (dtH ? ldA<T, kInt<T>>(dH, P, p, 12 + b) : zero)
                          : ldA<T, kInt<T>>(dH, P, p, (a - 1) * 4 + b);
    const T dHba = b == 0 ? (dtH ? ldA<T, kInt<T>>(dH, P, p, 12 + a) : zero)
                          : ldA<T, kInt<T>>(dH, P, p, (b - 1) * 4 + a);
    const T gab = ldA<T, FU>(u, P, p, s);
    Acc<T> acc;
    acc.add(half_of(dHab + dHba));
#pragma unroll
    for (int c = 0; c < 4; ++c) acc.fma_(-V(kGGam + c * 10 + s), Hup[c]);
    const T DH = acc.get();
    Acc<T> v;
    v.fma_(-twoal, DH);
    v.fma_(-(anC), gab);
    if (a == 0) v.fma_(aa, V(kGC + b));
    if (b == 0) v.fma_(aa, V(kGC + a));
    // -2 alpha g^cd g^ef Gamma_ace Gamma_bdf
    Acc<T> qa;
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int e = c; e < 4; ++e) qa.fma_(V(kGGam + a * 10 + SI(c, e)), Gce[SI(c, e)]);
    Acc<T> r;
    r.add(v.get());
    r.fma_(m2al, qa.get());
    if (live) stA<T, kInt<T>>(src, P, p, s, r.get());
  }
}

// slots of k_rhs_quad_shared: Pi, Phi_iab, alpha | beta^i | gamma^ij as in the source
// buffer
constexpr int kQPi = 0, kQPh = 10, kQM = 40, kQSlots = 50;

// Warp w takes the sources of d_t Pi_ab with larger index b = w and, w < 3, those
// of d_t Phi_iab with i = w.
// 112 registers, four blocks per SM, for a pair state: a step runs it beside the
// derivative launches, which five blocks of 96 registers hold up (six 9 x 12 x 24
// shells stacked, four steps 1917 us, so 1874), and with 127 the step takes longer too
// (two steps of 25 x 24 x 48 points 1358 us, so 1346).
template <class T, bool FU>
__global__ void __launch_bounds__(kRhsBlock) __maxnreg__(FU ? 112 : 96)
    k_rhs_quad_shared(const double* __restrict__ u, double* __restrict__ src, Geo geo) {
  __shared__ T sm[kQSlots * 32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const PointSlots<T> V{sm + lane};
  const long long P = geo.P;
  const long long q = blockIdx.x * 32ll + lane;
  const bool live = q < P;
  const long long p = live ? q : P - 1;
  {
    T v[13];
#pragma unroll
    for (int i = 0; i < 13; ++i) {
      const int t = w + 4 * i;
      if (t < 50) v[i] = t < 40 ? ldA<T, FU>(u, P, p, 10 + t) : ldA<T, kInt<T>>(src, P, p, t);
    }
#pragma unroll
    for (int i = 0; i < 13; ++i) {
      const int t = w + 4 * i;
      if (t < 50) V(t) = v[i];
    }
  }
  __syncthreads();
  // 3+1 quantities (eqs. normal, abgfromgab) as k_rhs_gamma derived them
  const T alpha = V(kQM);
  T bu[3], gi[3][3];
#pragma unroll
  for (int x = 0; x < 3; ++x) bu[x] = V(kQM + 1 + x);
  gi[0][0] = V(kQM + 4);
  gi[0][1] = gi[1][0] = V(kQM + 5);
  gi[0][2] = gi[2][0] = V(kQM + 6);
  gi[1][1] = V(kQM + 7);
  gi[1][2] = gi[2][1] = V(kQM + 8);
  gi[2][2] = V(kQM + 9);
  const T ialpha = S<T>::c(1.0) / alpha;
  const T ia2 = ialpha * ialpha;
  T nu[4];
  nu[0] = ialpha;
#pragma unroll
  for (int i = 0; i < 3; ++i) nu[i + 1] = -(bu[i] * ialpha);
  const T hal = half_of(alpha);
  {
    T gi4[10];
    gi4[0] = -ia2;
#pragma unroll
    for (int i = 0; i < 3; ++i) gi4[SI(0, i + 1)] = bu[i] * ia2;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) gi4[SI(i + 1, j + 1)] = gi[i][j] - bu[i] * bu[j] * ia2;
    const T twoal = alpha + alpha;
    const int b = w;
    const SymRow rb(b);
    // Q2_ab = Pi_ac g^cd Pi_db, Q1_ab = gamma^ij g^cd Phi_iac Phi_jbd
    T Piu[4], W[3][4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      Acc<T> acc;
#pragma unroll
      for (int d = 0; d < 4; ++d) acc.fma_(gi4[SI(c, d)], V(kQPi + rb(d)));
      Piu[c] = acc.get();
    }
    {
      T Y[3][4];
#pragma unroll
      for (int x = 0; x < 3; ++x)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          Acc<T> acc;
#pragma unroll
          for (int d = 0; d < 4; ++d) acc.fma_(gi4[SI(c, d)], V(kQPh + 10 * x + rb(d)));
          Y[x][c] = acc.get();
        }
#pragma unroll
      for (int x = 0; x < 3; ++x)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          Acc<T> acc;
#pragma unroll
          for (int y = 0; y < 3; ++y) acc.fma_(gi[x][y], Y[y][c]);
          W[x][c] = acc.get();
        }
    }
    // remaining algebraic terms of eq. Pidot
    T nnPi, cPh[3];  // n^c n^d Pi_cd; beta^j - alpha n^c Pi_ci gamma^ij
    {
      T nPi[4];
      nnPi = normal_row(nu, nPi, [&](int s) -> T { return V(kQPi + s); });
#pragma unroll
      for (int y = 0; y < 3; ++y) {
        Acc<T> acc;
#pragma unroll
        for (int x = 0; x < 3; ++x) acc.fma_(nPi[x + 1], gi[x][y]);
        cPh[y] = bu[y] - alpha * acc.get();
      }
    }
    const T cPi = -(hal * nnPi);
    // (a spare thread reads rows that this kernel does not write: its own are being
    // written by the last point's thread)
    const double* part_src = live ? src : src + 40 * P;
#pragma unroll 1
    for (int a = 0; a <= b; ++a) {
      const SymRow ra(a);
      const int s = rb(a);
      const T part = ldA_rw<T, kInt<T>>(part_src, P, p, s);
      Acc<T> q2;
#pragma unroll
      for (int c = 0; c < 4; ++c) q2.fma_(-V(kQPi + ra(c)), Piu[c]);
      Acc<T> qq;
      qq.add(q2.get());
#pragma unroll
      for (int x = 0; x < 3; ++x)
#pragma unroll
        for (int c = 0; c < 4; ++c) qq.fma_(V(kQPh + 10 * x + ra(c)), W[x][c]);
      Acc<T> acc;
      acc.add(part);
      acc.fma_(twoal, qq.get());
      acc.fma_(cPi, V(kQPi + s));
#pragma unroll
      for (int x = 0; x < 3; ++x) acc.fma_(cPh[x], V(kQPh + 10 * x + s));
      if (live) stA<T, kInt<T>>(src, P, p, s, acc.get());
    }
  }
  if (w == 3) return;
  // algebraic terms of eq. Phidot
  const int x = w;
  T nnPhi, Mk[3];  // n^c n^d Phi_xcd; alpha gamma^jk n^c Phi_x,j,c less alpha delta^k_x
  {
    T nP[4];
    nnPhi = normal_row(nu, nP, [&](int s) -> T { return V(kQPh + 10 * x + s); });
#pragma unroll
    for (int z = 0; z < 3; ++z) {
      Acc<T> acc;
#pragma unroll
      for (int y = 0; y < 3; ++y) acc.fma_(nP[y + 1], gi[y][z]);
      Mk[z] = alpha * acc.get();
      if (z == x) Mk[z] = Mk[z] - alpha;
    }
  }
  const T hnn = hal * nnPhi;
#pragma unroll 1
  for (int s = 0; s < 10; ++s) {
    Acc<T> acc;
    acc.fma_(hnn, V(kQPi + s));
#pragma unroll
    for (int z = 0; z < 3; ++z) acc.fma_(Mk[z], V(kQPh + 10 * z + s));
    if (live) stA<T, kInt<T>>(src, P, p, 10 + 10 * x + s, acc.get());
  }
}

// Asynchronous copy of one 8-byte word to shared memory (the thread's own word:
// it waits for its own copies, no barrier).  Both addresses must be 8-byte aligned:
// the destination's type sees to it (a pair of floats alone is aligned to 4).
__device__ __forceinline__ void copy8_async(unsigned long long* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned int)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
template <int N>
__device__ __forceinline__ void copies_pending_at_most() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The words of a symmetric pair (15 derivatives, 4 sources) are copied to shared
// memory one pair ahead: held in registers only one pair's loads were in flight
// (DRAM 54 %, half the warps' time waiting for them).  Now 52 us for 33 x 48 x 96
// points, 292 MB at 83 % of the copy bandwidth.
constexpr int kPpWords = 19;

// value of a copied word of internal storage
template <class T> __device__ __forceinline__ T word_value(unsigned long long w);
template <> __device__ __forceinline__ double word_value<double>(unsigned long long w) {
  return __longlong_as_double((long long)w);
}
template <> __device__ __forceinline__ ff word_value<ff>(unsigned long long w) {
  return ff{__uint_as_float((unsigned int)w), __uint_as_float((unsigned int)(w >> 32))};
}

// blockIdx.y: the block's share of the ten symmetric pairs (pp_split).
template <class T, bool FO>
__global__ void __launch_bounds__(128) k_rhs_pp(const double* __restrict__ D, const double* __restrict__ src,
                                                double* __restrict__ out, Geo geo) {
  __shared__ unsigned long long buf[2][kPpWords][128];
  static_assert(alignof(decltype(buf)) == 8, "8-byte copies");
  const long long P = geo.P;
  const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p >= P) return;
  const PointIdx at = point_idx(geo, p);
  const int k = at.k, i = at.i, jj = at.jj;
  const int nv = geo.nv;
  const int per = 10 / (int)gridDim.y, s0 = per * (int)blockIdx.y;
  // words 5 m .. 5 m + 4: d_m of g_s, Pi_s, Phi_xs; 15: source of d_t Pi_s, 16..18:
  // of d_t Phi_xs
  auto fetch = [&](int s) {
    unsigned long long(*w)[128] = buf[(s - s0) & 1];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const double* d = D + (long long)m * nv * P + p;
#pragma unroll
      for (int e = 0; e < 5; ++e) copy8_async(&w[5 * m + e][threadIdx.x], d + (long long)(10 * e + s) * P);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) copy8_async(&w[15 + e][threadIdx.x], src + (long long)(10 * e + s) * P + p);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(s0);
  const Jac<T> J = jacobian<T>(geo, k, i, jj);
  const T alpha = ldA<T, kInt<T>>(src, P, p, 40);
  T bu[3], gi[3][3];
#pragma unroll
  for (int x = 0; x < 3; ++x) bu[x] = ldA<T, kInt<T>>(src, P, p, 41 + x);
  gi[0][0] = ldA<T, kInt<T>>(src, P, p, 44);
  gi[0][1] = gi[1][0] = ldA<T, kInt<T>>(src, P, p, 45);
  gi[0][2] = gi[2][0] = ldA<T, kInt<T>>(src, P, p, 46);
  gi[1][1] = ldA<T, kInt<T>>(src, P, p, 47);
  gi[1][2] = gi[2][1] = ldA<T, kInt<T>>(src, P, p, 48);
  gi[2][2] = ldA<T, kInt<T>>(src, P, p, 49);
  // beta^k d_k = sum_m b_m D_m; alpha gamma^ik d_k = sum_m G_im D_m; J_xm for d_x
  T b[3], G[3][3];
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    Acc<T> acc;
#pragma unroll
    for (int x = 0; x < 3; ++x) acc.fma_(bu[x], J.j[x][m]);
    b[m] = acc.get();
  }
#pragma unroll
  for (int x = 0; x < 3; ++x)
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      Acc<T> acc;
#pragma unroll
      for (int y = 0; y < 3; ++y) acc.fma_(gi[x][y], J.j[y][m]);
      G[x][m] = alpha * acc.get();
    }
  T aJ[3][3];
#pragma unroll
  for (int x = 0; x < 3; ++x)
#pragma unroll
    for (int m = 0; m < 3; ++m) aJ[x][m] = alpha * J.j[x][m];
  const bool outer = (k == geo.n_r - 1);
  T sl[3], su[3];
  if (outer) {
    const T l[3] = {J.st * J.cp, J.st * J.sp, J.ct};
    Acc<T> q;
#pragma unroll
    for (int x = 0; x < 3; ++x)
#pragma unroll
      for (int y = 0; y < 3; ++y) q.fma_(gi[x][y] * l[x], l[y]);
    const T iq = S<T>::c(1.0) / sqrt_s(q.get());
#pragma unroll
    for (int x = 0; x < 3; ++x) sl[x] = l[x] * iq;
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      Acc<T> acc;
#pragma unroll
      for (int y = 0; y < 3; ++y) acc.fma_(gi[x][y], sl[y]);
      su[x] = acc.get();
    }
  }
#pragma unroll 1
  for (int s = s0; s < s0 + per; ++s) {
    if (s + 1 < s0 + per) {
      fetch(s + 1);
      copies_pending_at_most<1>();
    } else {
      copies_pending_at_most<0>();
    }
    auto word = [&](int e) -> T { return word_value<T>(buf[(s - s0) & 1][e][threadIdx.x]); };
    T Dd[3], DPh[3][3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      Dd[m] = word(5 * m) - word(5 * m + 1);
#pragma unroll
      for (int x = 0; x < 3; ++x) DPh[x][m] = word(5 * m + 2 + x);
    }
    Acc<T> aPi;
    aPi.add(word(15));
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      aPi.fma_(-b[m], Dd[m]);
#pragma unroll
      for (int x = 0; x < 3; ++x) aPi.fma_(-G[x][m], DPh[x][m]);
    }
    T rPi = aPi.get();
    T rPh[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      Acc<T> a;
      a.add(word(16 + x));
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        a.fma_(b[m], DPh[x][m]);
        if (x < 2 || m < 2) a.fma_(aJ[x][m], Dd[m]);  // z does not depend on phi
      }
      rPh[x] = a.get();
    }
    if (outer) {
      const T rg = ldA<T, FO>(out, P, p, s);
      Acc<T> sd;
#pragma unroll
      for (int x = 0; x < 3; ++x) sd.fma_(su[x], rPh[x]);
      const T wplus = rPi + sd.get();
      const T w2 = half_of(wplus - rg);
      rPi = half_of(rg + wplus);
#pragma unroll
      for (int x = 0; x < 3; ++x) rPh[x] = sl[x] * w2;
    }
    stA<T, FO>(out, P, p, 10 + s, rPi);
#pragma unroll
    for (int x = 0; x < 3; ++x) stA<T, FO>(out, P, p, 20 + 10 * x + s, rPh[x]);
  }
}

// Gauge fields of 54/58-field states (App. A.1; eq. gauge with H_a a field
// of the state): H_a from fields 50..53 into the gauge buffer, d_i H_a from
// their spherical derivatives by the chain rule (eq. dvdx), and for 58
// fields d_t H_a = G_a (fields 54..57) as rows 12..15 of dH.  The gauge
// fields' right-hand sides: d_t H_a = G_a for 58 fields (0 for 54) and
// d_t G_a = 0; the outer boundary condition leaves them alone.
template <class T, bool FU, bool FO>
__global__ void __launch_bounds__(128) k_gauge_rhs(const double* __restrict__ u, const double* __restrict__ D,
                                                   double* __restrict__ H, double* __restrict__ dH,
                                                   double* __restrict__ out, Geo geo) {
  const long long P = geo.P;
  const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p >= P) return;
  const PointIdx at = point_idx(geo, p);
  const int k = at.k, i = at.i, jj = at.jj;
  const int nv = geo.nv;
  const Jac<T> J = jacobian<T>(geo, k, i, jj);
  const T zero = S<T>::c(0.0);
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    stA<T, kInt<T>>(H, P, p, b, ldA<T, FU>(u, P, p, 50 + b));
    T ds[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) ds[m] = Store<T, kInt<T>>::ld(D, ((long long)m * nv + 50 + b) * P + p);
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      Acc<T> a;
#pragma unroll
      for (int m = 0; m < 3; ++m) a.fma_(J.j[x][m], ds[m]);
      stA<T, kInt<T>>(dH, P, p, 4 * x + b, a.get());
    }
    if (nv == 58) {
      const T Gb = ldA<T, FU>(u, P, p, 54 + b);
      stA<T, kInt<T>>(dH, P, p, 12 + b, Gb);
      stA<T, FO>(out, P, p, 50 + b, Gb);
      stA<T, FO>(out, P, p, 54 + b, zero);
    } else {
      stA<T, FO>(out, P, p, 50 + b, zero);
    }
  }
}

// Whether a point's tensors are shared out over four warps: up to 2.5 blocks of
// one point per thread per SM.  gamma / quad, us, one thread against four warps per
// point: 2106 points 14.7 / 13.7 against 8.9 / 7.9, 11250 points 15.5 / 14.0 against
// 10.5 / 9.8, 28800 points 21.1 / 17.8 against 22.0 / 16.9, 67584 points 32.4 / 31.8
// against 39.7 / 35.4 (quad by now, at four blocks per SM, 15.1 for 16250 points, 28.6
// for 39200).  The line lies above where the two meet because the call of an FP64
// state goes without its pair copy below it (right-hand side, us: 28800 points 132
// against 119, 39200 points 167 against 163, 67584 points 216 against 233).  The
// kernels of a step run beside its derivative launches, where the same line holds:
// at 1.5 blocks per SM instead, RK4 step, us: 31250 points 799 against 775, 35280 points
// 791 against 777, 39200 points 883 against 879, 44064 points 978 against 984.
// Blocks of a batch's other classes count too: beside them the shorter chain buys
// nothing and the repeated work costs (batch of eight shells 14.7 against 15.4 ms).
static bool rhs_shared(const cffyn_shell* sh, unsigned nbr) {
  return 2 * (nbr + sh->beside / kRhsBlock) <= 5ll * sh->sm_count;
}

// Shares of the ten symmetric pairs per point in k_rhs_pp: one thread's loop over
// all ten takes 27 us by itself (its loads wait one after the other), in ten
// shares 9.5, with the words copied ahead 6 (13 x 9 x 18); every share repeats the chain-rule coefficients, so
// only as many are taken as fill one wave (four blocks per SM).
static unsigned pp_split(const cffyn_shell* sh, unsigned nb) {
  for (unsigned n : {10u, 5u, 2u})
    if (nb * n + sh->beside / 128 <= 4ll * sh->sm_count) return n;
  return 1u;
}

// stage = 0: all three kernels; 1: sources with Christoffels; 2: quadratic
// sources; 3: principal parts + boundary.  u_pairs: the state is a pair-stored
// internal buffer (the stage states of the mixed path); out_pairs: the output
// is the internal rhs buffer (else an FP64 caller array).  On the mixed path an FP64
// output goes with an FP64 state where the kernels are shared out and with its pair
// copy where they are not (pw_rhs): no other combination is instantiated.
int pw_rhs_part(const cffyn_shell* sh, const double* u, const double* D, double* out, int stage,
                bool u_pairs, bool out_pairs, cudaStream_t st) {
  Geo g = geo_of(sh);
  const unsigned nb = blocks_for(g.P, 128), nbr = blocks_for(g.P, kRhsBlock), nbs = blocks_for(g.P, 32);
  const bool shared = rhs_shared(sh, nbr);
  const bool mixed = sh->d.precision == CFFYN_MIXED;
  if (mixed && (out_pairs ? !u_pairs : u_pairs == shared)) {
    set_error("internal: right-hand side storage (state %d, output %d) not instantiated", (int)u_pairs,
              (int)out_pairs);
    return CFFYN_EINVAL;
  }
  if (stage == 0 || stage == 1) {
    const int dtH = sh->nv == 58;
    if (sh->ng > 0) {
      if (!mixed)
        k_gauge_rhs<double, false, false><<<nb, 128, 0, st>>>(u, D, sh->H, sh->dH, out, g);
      else if (u_pairs && !out_pairs)
        k_gauge_rhs<ff, true, false><<<nb, 128, 0, st>>>(u, D, sh->H, sh->dH, out, g);
      else if (u_pairs)
        k_gauge_rhs<ff, true, true><<<nb, 128, 0, st>>>(u, D, sh->H, sh->dH, out, g);
      else
        k_gauge_rhs<ff, false, false><<<nb, 128, 0, st>>>(u, D, sh->H, sh->dH, out, g);
      count_launch();
    }
#define CFFYN_GAMMA(K_, NB_, ...) K_<__VA_ARGS__><<<NB_, kRhsBlock, 0, st>>>(u, sh->H, sh->dH, sh->Rsrc, out, g, dtH)
    if (!mixed && shared)
      CFFYN_GAMMA(k_rhs_gamma_shared, nbs, double, false, false);
    else if (!mixed)
      CFFYN_GAMMA(k_rhs_gamma, nbr, double, false, false);
    else if (out_pairs && shared)
      CFFYN_GAMMA(k_rhs_gamma_shared, nbs, ff, true, true);
    else if (out_pairs)
      CFFYN_GAMMA(k_rhs_gamma, nbr, ff, true, true);
    else if (u_pairs)
      CFFYN_GAMMA(k_rhs_gamma, nbr, ff, true, false);
    else
      CFFYN_GAMMA(k_rhs_gamma_shared, nbs, ff, false, false);
#undef CFFYN_GAMMA
    count_launch();
  }
  if (stage == 0 || stage == 2) {
    if (!mixed && shared)
      k_rhs_quad_shared<double, false><<<nbs, kRhsBlock, 0, st>>>(u, sh->Rsrc, g);
    else if (!mixed)
      k_rhs_quad<double, false><<<nbr, kRhsBlock, 0, st>>>(u, sh->Rsrc, g);
    else if (!u_pairs)
      k_rhs_quad_shared<ff, false><<<nbs, kRhsBlock, 0, st>>>(u, sh->Rsrc, g);
    else if (shared)
      k_rhs_quad_shared<ff, true><<<nbs, kRhsBlock, 0, st>>>(u, sh->Rsrc, g);
    else
      k_rhs_quad<ff, true><<<nbr, kRhsBlock, 0, st>>>(u, sh->Rsrc, g);
    count_launch();
  }
  if (stage == 0 || stage == 3) {
    const dim3 npp(nb, pp_split(sh, nb));
    if (!mixed)
      k_rhs_pp<double, false><<<npp, 128, 0, st>>>(D, sh->Rsrc, out, g);
    else if (out_pairs)
      k_rhs_pp<ff, true><<<npp, 128, 0, st>>>(D, sh->Rsrc, out, g);
    else
      k_rhs_pp<ff, false><<<npp, 128, 0, st>>>(D, sh->Rsrc, out, g);
    count_launch();
  }
  CF_CUDA(cudaGetLastError());
  return CFFYN_OK;
}

// Right-hand side of an FP64 state into an FP64 array.  On the mixed path large
// launches read the state from a pair copy in Uf (the step calls fill it anew):
// converted once instead of by every kernel that reads it (gamma and quad of
// 33 x 48 x 96: 142 + 130 us, with the copy 28 + 81 + 91 then, 18.5 + 67 + 66 now).
int pw_rhs(const cffyn_shell* sh, const double* u, const double* D, double* out, cudaStream_t st) {
  if (sh->d.precision != CFFYN_MIXED || rhs_shared(sh, blocks_for((long long)P_all(sh), kRhsBlock)))
    return pw_rhs_part(sh, u, D, out, 0, false, false, st);
  const int rc = pw_to_internal(sh, u, sh->Uf, (long long)sh->nv * (long long)sh->P, st);
  return rc ? rc : pw_rhs_part(sh, sh->Uf, D, out, 0, true, false, st);
}

}  // namespace cffyn
