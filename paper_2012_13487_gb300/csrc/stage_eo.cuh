// Even-odd form of the volume and lift contractions.  Included by
// stage_impl.cuh inside its namespace; every stage-kernel form that contracts
// on FMAs uses it.
//
// The node set is symmetric under the reflection r <-> s of the reference
// triangle.  Write the nodes as pairs (a, b) that the reflection exchanges
// (a = b on the axis r = s) and f by its even and odd parts E = f_a + f_b,
// O = f_a - f_b.  S = Dr + Ds commutes with the reflection and D = Ds - Dr
// anticommutes, so S takes E to even and O to odd outputs and D takes E to odd
// and O to even ones:
//   (S f)_a,b = Se E +- So O,   (D f)_a,b = Do O +- De E,
// and with ar Dr + as Ds = ((ar + as) S + (as - ar) D) / 2 the volume term needs
// NE^2 + NO^2 + 2 NE NO = Np^2 products instead of 2 Np^2 (NE + NO = Np).  D is
// the derivative along the face r + s = 0, so at that face's nodes it reads that
// face's nodes only (dzero).  LIFT commutes with the reflection, which exchanges
// the faces 0 and 2 and reverses face 1, and splits in the same way.  At degree 4
// a velocity of an element takes 201 products for the volume term instead of 450
// and at most 114 for the lift instead of 225, against 38 additions for the parts.
//
// The kernels were bound by instruction issue or, in FP64, by the FP64 pipe.  Dense
// against split, otherwise unchanged (GB300): FP32, 256 velocities, degree 4, 85M against
// 71.5M warp instructions per launch of 31M values, 105 against 95 us; FP32, 16 velocities,
// degree 5, 280 against 239 us for 44M; FP64, 16 velocities, degree 3, 1,152 elements, a
// call of ten steps 1716 against 1452 us.

// E has NE = NO + (nodes on the axis) entries; the pairs off the axis come first
constexpr int NAX = P / 2 + 1;
constexpr int NO = (NP - NAX) / 2;
constexpr int NE = NO + NAX;
constexpr int NF1E = P / 2 + 1;        // even parts of face 1: its pairs and, at even P, its middle
constexpr int NF1O = (P + 1) / 2;      // odd parts of face 1
constexpr int NLE = NFP + NF1E;        // even flux parts: faces 0 and 2, then face 1
constexpr int NLO = NFP + NF1O;
constexpr int EO_SE = 0;
constexpr int EO_SO = EO_SE + NE * NE;
constexpr int EO_DE = EO_SO + NO * NO;  // [NO][NE]: E to odd outputs
constexpr int EO_DO = EO_DE + NO * NE;  // [NE][NO]: O to even outputs
constexpr int EO_LE = EO_DO + NE * NO;
constexpr int EO_LO = EO_LE + NE * NLE;
constexpr int EO_N = EO_LO + NO * NLO;
__host__ __device__ constexpr int at_least_1(int n) { return n > 0 ? n : 1; }

struct EoPairs {
  int a[NE] = {}, b[NE] = {};
  bool hyp[NE] = {};  // on the face r + s = 0
};
__host__ __device__ constexpr EoPairs eo_pairs() {
  EoPairs p;
  int q = 0;
  for (int pass = 0; pass < 2; ++pass)
    for (int j = 0; j <= P; ++j)
      for (int i = 0; i <= j; ++i) {
        if (i + j > P || (i == j) != (pass == 1)) continue;
        p.a[q] = j * (P + 1) - j * (j - 1) / 2 + i;  // row j, column i
        p.b[q] = i * (P + 1) - i * (i - 1) / 2 + j;
        p.hyp[q] = i + j == P;
        ++q;
      }
  return p;
}

static __constant__ double c_eo64[EO_N];
static __constant__ float c_eo32[EO_N];

// Coefficient idx in the compute precision.  kImm: this degree's FP32 table as
// compile-time constants (the operators depend only on the degree, and with the
// loops unrolled every entry becomes an instruction immediate instead of a
// constant-memory load; a CPU test holds the table to the library's operators);
// otherwise constant memory.
template <typename R, bool kImm>
__device__ __forceinline__ R eov(int idx) {
#ifdef FEDBM_EO32_TABLE
  if constexpr (kImm && sizeof(R) == 4) {
    constexpr float t[] = {FEDBM_EO32_TABLE};
    static_assert(sizeof(t) / sizeof(t[0]) == EO_N, "operator table of another degree");
    return t[idx];
  }
#endif
  if constexpr (sizeof(R) == 8) return c_eo64[idx];
  else return c_eo32[idx];
}
#ifdef FEDBM_EO32_TABLE
constexpr bool kHaveOpsTable = true;
#else
constexpr bool kHaveOpsTable = false;
#endif

// Arithmetic of one velocity per thread, or of two as packed FP32 pairs.
template <typename R_, bool kImm>
struct EoScalar {
  using T = R_;
  static __device__ __forceinline__ T zero() { return T(0); }
  static __device__ __forceinline__ T add(T x, T y) { return x + y; }
  static __device__ __forceinline__ T sub(T x, T y) { return x - y; }
  static __device__ __forceinline__ T fmat(T x, T y, T z) { return fma(x, y, z); }
  static __device__ __forceinline__ T fmac(int idx, T x, T z) { return fma(eov<T, kImm>(idx), x, z); }
};
struct EoPacked {
  using T = unsigned long long;
  static __device__ __forceinline__ T zero() { return 0ull; }
  static __device__ __forceinline__ T add(T x, T y) {
    T r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
    return r;
  }
  static __device__ __forceinline__ T sub(T x, T y) {
    T r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
    return r;
  }
  static __device__ __forceinline__ T fmat(T x, T y, T z) { return f2fma(x, y, z); }
};

// Two velocities per thread with the operators as immediates: additions and
// scalings act on the packed pair, products with an operator on its halves (a
// packed FMA takes no immediate, and its broadcast operand would be one more load).
template <bool kImm>
struct EoDual : EoPacked {
  static __device__ __forceinline__ T fmac(int idx, T x, T z) {
    float x0, x1, z0, z1;
    f2unpack(x, x0, x1);
    f2unpack(z, z0, z1);
    const float c = eov<float, kImm>(idx);
    return f2pack(fmaf(c, x0, z0), fmaf(c, x1, z1));
  }
};

// Even and odd parts le, lo of LIFT flux.  on02, on1: faces 0 and 2, or face 1,
// carry flux for some velocity of the warp; the others' columns are skipped.
template <class M>
__device__ __forceinline__ void eo_lift(const typename M::T (&flux)[NF], bool on02, bool on1,
                                        typename M::T (&le)[NE], typename M::T (&lo)[at_least_1(NO)]) {
  using T = typename M::T;
#pragma unroll
  for (int q = 0; q < NE; ++q) le[q] = M::zero();
#pragma unroll
  for (int q = 0; q < NO; ++q) lo[q] = M::zero();
  if (on02) {
#pragma unroll
    for (int a = 0; a < NFP; ++a) {
      const T g = M::add(flux[a], flux[2 * NFP + a]), h = M::sub(flux[a], flux[2 * NFP + a]);
#pragma unroll
      for (int q = 0; q < NE; ++q) le[q] = M::fmac(EO_LE + q * NLE + a, g, le[q]);
#pragma unroll
      for (int q = 0; q < NO; ++q) lo[q] = M::fmac(EO_LO + q * NLO + a, h, lo[q]);
    }
  }
  if (on1) {
#pragma unroll
    for (int a = 0; a < NF1E; ++a) {
      const int b = P - a;
      const T g = a == b ? flux[NFP + a] : M::add(flux[NFP + a], flux[NFP + b]);
#pragma unroll
      for (int q = 0; q < NE; ++q) le[q] = M::fmac(EO_LE + q * NLE + NFP + a, g, le[q]);
      if (a == b) continue;
      const T h = M::sub(flux[NFP + a], flux[NFP + b]);
#pragma unroll
      for (int q = 0; q < NO; ++q) lo[q] = M::fmac(EO_LO + q * NLO + NFP + a, h, lo[q]);
    }
  }
}

// -(ar Dr + as Ds) f + LIFT flux of f(node), handed to fin(node, value) node by
// node.  na = -(ar + as) / 2, nd = (ar - as) / 2.
template <class M, class F, class Fin>
__device__ __forceinline__ void eo_volume(F f, typename M::T na, typename M::T nd,
                                          const typename M::T (&le)[NE],
                                          const typename M::T (&lo)[at_least_1(NO)], Fin fin) {
  using T = typename M::T;
  constexpr EoPairs pr = eo_pairs();
  T E[NE], O[at_least_1(NO)];
#pragma unroll
  for (int q = 0; q < NE; ++q) {
    const T fa = f(pr.a[q]);
    if (q < NO) {
      const T fb = f(pr.b[q]);
      E[q] = M::add(fa, fb);
      O[q] = M::sub(fa, fb);
    } else {
      E[q] = fa;
    }
  }
#pragma unroll
  for (int q = 0; q < NE; ++q) {
    T se = M::zero(), dv = M::zero();
#pragma unroll
    for (int m = 0; m < NE; ++m) se = M::fmac(EO_SE + q * NE + m, E[m], se);
#pragma unroll
    for (int m = 0; m < NO; ++m)
      if (!pr.hyp[q] || pr.hyp[m]) dv = M::fmac(EO_DO + q * NO + m, O[m], dv);
    const T oe = M::fmat(na, se, M::fmat(nd, dv, le[q]));
    if (q < NO) {
      T so = M::zero(), de = M::zero();
#pragma unroll
      for (int m = 0; m < NO; ++m) so = M::fmac(EO_SO + q * NO + m, O[m], so);
#pragma unroll
      for (int m = 0; m < NE; ++m)
        if (!pr.hyp[q] || pr.hyp[m]) de = M::fmac(EO_DE + q * NE + m, E[m], de);
      const T oo = M::fmat(na, so, M::fmat(nd, de, lo[q]));
      fin(pr.a[q], M::add(oe, oo));
      fin(pr.b[q], M::sub(oe, oo));
    } else {
      fin(pr.a[q], oe);
    }
  }
}

// The same for the outputs q = part, part + nparts, .. only (a warp-uniform choice), with
// the lift of those; every sum in the same order as above.
template <class M, class F, class Fin>
__device__ __forceinline__ void eo_part(F f, const typename M::T (&flux)[NF], typename M::T na, typename M::T nd,
                                        int part, int nparts, Fin fin) {
  using T = typename M::T;
  constexpr EoPairs pr = eo_pairs();
  T E[NE], O[at_least_1(NO)], g[NLE], h[NLO];
#pragma unroll
  for (int q = 0; q < NE; ++q) {
    const T fa = f(pr.a[q]);
    if (q < NO) {
      const T fb = f(pr.b[q]);
      E[q] = M::add(fa, fb);
      O[q] = M::sub(fa, fb);
    } else {
      E[q] = fa;
    }
  }
#pragma unroll
  for (int a = 0; a < NFP; ++a) {
    g[a] = M::add(flux[a], flux[2 * NFP + a]);
    h[a] = M::sub(flux[a], flux[2 * NFP + a]);
  }
#pragma unroll
  for (int a = 0; a < NF1E; ++a) {
    const int b = P - a;
    g[NFP + a] = a == b ? flux[NFP + a] : M::add(flux[NFP + a], flux[NFP + b]);
    if (a < NF1O) h[NFP + a] = M::sub(flux[NFP + a], flux[NFP + b]);
  }
#pragma unroll
  for (int q = 0; q < NE; ++q) {
    if (q % nparts != part) continue;
    T le = M::zero(), se = M::zero(), dv = M::zero();
#pragma unroll
    for (int a = 0; a < NLE; ++a) le = M::fmac(EO_LE + q * NLE + a, g[a], le);
#pragma unroll
    for (int m = 0; m < NE; ++m) se = M::fmac(EO_SE + q * NE + m, E[m], se);
#pragma unroll
    for (int m = 0; m < NO; ++m)
      if (!pr.hyp[q] || pr.hyp[m]) dv = M::fmac(EO_DO + q * NO + m, O[m], dv);
    const T oe = M::fmat(na, se, M::fmat(nd, dv, le));
    if (q < NO) {
      T lo = M::zero(), so = M::zero(), de = M::zero();
#pragma unroll
      for (int a = 0; a < NLO; ++a) lo = M::fmac(EO_LO + q * NLO + a, h[a], lo);
#pragma unroll
      for (int m = 0; m < NO; ++m) so = M::fmac(EO_SO + q * NO + m, O[m], so);
#pragma unroll
      for (int m = 0; m < NE; ++m)
        if (!pr.hyp[q] || pr.hyp[m]) de = M::fmac(EO_DE + q * NE + m, E[m], de);
      const T oo = M::fmat(na, so, M::fmat(nd, de, lo));
      fin(pr.a[q], M::add(oe, oo));
      fin(pr.b[q], M::sub(oe, oo));
    } else {
      fin(pr.a[q], oe);
    }
  }
}

// Host side: the coefficients from the FP64 operators (row-major Dr, Ds
// [Np][Np], LIFT [Np][3 Nfp]).
inline void eo_coefficients(const double* Dr, const double* Ds, const double* LIFT, double (&t)[EO_N]) {
  constexpr EoPairs pr = eo_pairs();
  for (int q = 0; q < NE; ++q) {
    const int a = pr.a[q];
    auto S = [&](int m) { return Ds[a * NP + m] + Dr[a * NP + m]; };
    auto D = [&](int m) { return Ds[a * NP + m] - Dr[a * NP + m]; };
    for (int m = 0; m < NE; ++m) {
      const int x = pr.a[m], y = pr.b[m];
      t[EO_SE + q * NE + m] = x == y ? S(x) : 0.5 * (S(x) + S(y));
      if (q < NO) t[EO_DE + q * NE + m] = x == y ? D(x) : 0.5 * (D(x) + D(y));
      if (m < NO) {
        t[EO_DO + q * NO + m] = 0.5 * (D(x) - D(y));
        if (q < NO) t[EO_SO + q * NO + m] = 0.5 * (S(x) - S(y));
      }
    }
    const double* L = LIFT + a * NF;
    for (int j = 0; j < NFP; ++j) {
      t[EO_LE + q * NLE + j] = 0.5 * (L[j] + L[2 * NFP + j]);
      if (q < NO) t[EO_LO + q * NLO + j] = 0.5 * (L[j] - L[2 * NFP + j]);
    }
    for (int j = 0; j < NF1E; ++j) {
      const int k = P - j;
      t[EO_LE + q * NLE + NFP + j] = j == k ? L[NFP + j] : 0.5 * (L[NFP + j] + L[NFP + k]);
      if (q < NO && j < NF1O) t[EO_LO + q * NLO + NFP + j] = 0.5 * (L[NFP + j] - L[NFP + k]);
    }
  }
}
