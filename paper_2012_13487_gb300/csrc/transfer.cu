// Encode, decode and node-moment kernels (see transfer.h).
#include "transfer.h"

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "device_common.cuh"

namespace fedbm {
namespace transfer {
namespace {

constexpr int kThreads = 256;
constexpr size_t kSmemCap = 227 * 1024 - 64;  // dynamic; the encode kernel has 32 bytes of its own
// Rows of an element are staged through at most about this much shared memory
// per CTA, so that several CTAs share an SM and one's loads overlap another's
// stores.
constexpr size_t kStageBytes = 48 * 1024;

__device__ __forceinline__ double widen(double x) { return x; }

// Work split shared by encode and decode: a group of G threads (a warp where
// an element has at most kWarpValues values, else the whole CTA) handles one
// element at a time, kRows rows of it per pass through shared memory.
constexpr int kWarpValues = 1536;

struct Split {
  bool warp;       // groups are warps
  int rows;        // rows of an element staged at once
  size_t tables;   // bytes of the velocity tables in front of the buffers
  size_t smem;
  int grid;
};

inline size_t up16(size_t b) { return (b + 15) / 16 * 16; }

Split split_for(const Shape& sh, size_t table_bytes, size_t value_bytes, bool by_warp) {
  Split s;
  s.warp = by_warp;
  s.tables = up16(table_bytes);
  const size_t row = size_t(sh.Qp) * value_bytes;
  const int groups = s.warp ? kThreads / 32 : 1;
  s.rows = s.warp ? sh.Np : std::max(1, std::min(sh.Np, int(kStageBytes / row)));
  s.smem = s.tables + size_t(groups) * s.rows * row;
  const int per_sm = std::max(1, std::min(8, int(size_t(sh.smem_sm) / (s.smem + 1024))));
  const int64_t tiles = s.warp ? (sh.K + groups - 1) / groups : sh.K;
  s.grid = int(std::max<int64_t>(1, std::min<int64_t>(tiles, int64_t(sh.nsm) * per_sm)));
  return s;
}

template <bool kWarp>
__device__ __forceinline__ void group_sync() {
  if constexpr (kWarp) __syncwarp();
  else __syncthreads();
}

// Canonical positions j = row * Q + c of one group in steps of G, with the
// row and velocity kept without a division per value.
struct Walk {
  int c, row, dc, drow, Q;
  __device__ Walk(int start, int G, int Q_) : Q(Q_) {
    row = start / Q;
    c = start - row * Q;
    drow = G / Q;
    dc = G - drow * Q;
  }
  __device__ void next() {
    row += drow;
    c += dc;
    if (c >= Q) {
      c -= Q;
      ++row;
    }
  }
};

// (f - w) / w rounded to FP32, as the FP64 quotient rounds, without FP64 arithmetic per
// value (its rate is low here): w is held as three FP32 pieces, all its 53 bits, and 1/w
// as two.  x - w is formed as a sum s + low whose rounding errors are kept (Knuth's
// two-sum, The Art of Computer Programming vol. 2, 4.2.2, theorem B), and its product with
// 1/w ends in an FMA that adds the small terms to the exact leading product, so that what
// is rounded there is off by about 2^-46.  Over 16 to 1,089 velocities and
// deviations of 1e-7 to 1e6 the result is off by at most 1.0 units of 2^-24 |d|, as the FP64
// quotient rounded to FP32 is; one difference and one product in plain FP32 had 3.6.
// An FP64 x that FP32 holds exactly takes the same path, so that an FP32 value and the
// same value given in FP64 give the same bits; any other is subtracted and scaled in
// FP64.  Weights below 2^-96, whose last bits FP32's denormals do not hold (marked by an
// inverse that is not a number), weights of 0 and results out of FP32's range are told by
// one comparison of the result and take the FP64 quotient.
constexpr double kTinyWeight = 1.262177448353619e-29;  // 2^-96
// ih: NaN for a tiny weight or 0.  (Laid out by weight_tables once per solver; in every CTA
// instead, the FP64 quotients were half of the time of a small load.)
struct DevTable {  // canonical order
  const DevRow* row;
  const DevIndex* index;
  const double2* wide;  // FP64 input only: w, 1/w
  const double* w64;    // internal order
};
__device__ __forceinline__ float two_difference(float a, float b, float& err) {
  const float s = __fadd_rn(a, -b), t = __fadd_rn(s, -a);
  err = __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -t)), -__fadd_rn(b, t));
  return s;
}
// the same where |a| >= |b| or a = 0 (Dekker 1971)
__device__ __forceinline__ float two_difference_ordered(float a, float b, float& err) {
  const float s = __fadd_rn(a, -b);
  err = -__fadd_rn(b, __fadd_rn(s, -a));
  return s;
}
__device__ __noinline__ float deviation64(double x, double w) { return w > 0.0 ? float((x - w) / w) : 0.f; }
template <typename TIn>
__device__ __forceinline__ float deviation(TIn x, const DevTable& t, int c, const DevIndex& at) {
  const float xf = float(x);
  bool narrow = true;
  if constexpr (sizeof(TIn) == 8) narrow = __double_as_longlong(widen(xf)) == __double_as_longlong(x);
  float d;
  if (narrow) {
    const DevRow r = t.row[c];
    float ea, es;
    // x - wh is 0 or, as a multiple of half a unit in wh's last place, at least |wl|
    const float s = two_difference_ordered(two_difference(xf, r.wh, ea), r.wl, es);
    const float low = __fadd_rn(__fadd_rn(ea, es), -at.wll);
    d = fmaf(s, r.ih, fmaf(s, r.il, __fmul_rn(low, r.ih)));
  } else {
    const double2 w = t.wide[c];
    d = float((x - w.x) * w.y);
  }
  return fabsf(d) <= 3e38f ? d : deviation64(double(x), t.w64[at.at]);
}

// Encode: the caller's rows are read along the canonical order (consecutive
// lanes, consecutive addresses), scattered into shared memory by the internal
// velocity order, and written from there as 16-byte vectors of the internal
// row.  Deviation forms keep (f - w)/w of the whole element in shared memory
// between finding the element's largest deviation and writing the codes, so
// the input is read once and only one quotient is formed per value.  Before,
// with two FP64 divisions per value, scattered 2- and 4-byte stores and an
// integer division per value (GB300, ncu): BF16 from FP32 input 15.3 ms at 335M
// values (1,024 velocities), 1.45 ms at 31M (256) and 2.44 ms at 44M (16), FP32
// from FP32 71 us at 31M; now (events around the call) 0.93 ms, 90 us, 132 us and 49 us.
// Of these, the quotient with its rounding errors costs the 16-bit forms 7 us at 31M and
// at 44M against a difference and a product in plain FP32, whose codes can round the other
// way near a tie; from FP64 input BF16 takes 3.27 ms, 310 us and 438 us.
template <class ST, typename TIn, bool kWarp>
__global__ void __launch_bounds__(kThreads) encode_kernel(const TIn* __restrict__ in, void* out, float* scale,
                                                          const double* __restrict__ vel64,
                                                          const int32_t* __restrict__ iperm, Weights weights,
                                                          int64_t K, int Np, int Q, int Qp, int rows,
                                                          int table_bytes) {
  using S = typename ST::S;
  using T = std::conditional_t<ST::dev, float, S>;  // staged values
  constexpr int V = 16 / int(sizeof(S));
  extern __shared__ __align__(16) unsigned char smem[];
  const double* w64 = vel64 + 2 * Qp;
  // tables in canonical order: the internal index, and for the deviation forms the weight's
  // pieces (sized in encode_plan)
  DevRow* rows_w = reinterpret_cast<DevRow*>(smem);
  DevIndex* index = reinterpret_cast<DevIndex*>(rows_w + Q);
  double2* wide = reinterpret_cast<double2*>(smem + (size_t(24) * Q + 15) / 16 * 16);
  int* perm = reinterpret_cast<int*>(smem);
  const DevTable dt{rows_w, index, wide, w64};
  for (int c = threadIdx.x; c < Q; c += kThreads) {
    if constexpr (ST::dev) {
      rows_w[c] = weights.row[c];
      index[c] = weights.index[c];
      if constexpr (sizeof(TIn) == 8) wide[c] = reinterpret_cast<const double2*>(weights.wide)[c];
    } else {
      perm[c] = iperm[c];
    }
  }
  const int G = kWarp ? 32 : kThreads;
  const int grp = kWarp ? threadIdx.x / 32 : 0, lane = kWarp ? threadIdx.x % 32 : threadIdx.x;
  const int ngroups = kWarp ? kThreads / 32 : 1;
  T* buf = reinterpret_cast<T*>(smem + table_bytes) + size_t(grp) * rows * Qp;
  for (int v = lane; v < rows * Qp; v += G) buf[v] = T(0);  // the padding velocities stay zero
  __shared__ float red[kThreads / 32];
  __syncthreads();

  for (int64_t k = blockIdx.x * int64_t(ngroups) + grp; k < K; k += int64_t(gridDim.x) * ngroups) {
    const TIn* src = in + k * Np * Q;
    S* dst = static_cast<S*>(out) + k * Np * Qp;
    float inv_s = 1.f, sc = 1.f;
    // largest deviation of the element into its scale, over all threads of the group
    auto set_scale = [&](float m) {
      for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
      if constexpr (!kWarp) {
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
        __syncthreads();
        m = red[0];
        for (int j = 1; j < kThreads / 32; ++j) m = fmaxf(m, red[j]);
      }
      if constexpr (ST::dev) {
        sc = 1.f;
        if (m > 0.f) {
          int e2;
          frexpf(m, &e2);
          sc = ldexpf(1.0f, e2 - ST::qmax_log2);
        }
        inv_s = 1.0f / sc;
        if (lane == 0) scale[k] = sc;
      }
    };
    const bool whole = rows >= Np;
    if constexpr (ST::dev) {
      if (!whole) {  // the element does not fit: its largest deviation in a pass of its own
        float m = 0.f;
        Walk w(lane, G, Q);
        for (int j = lane; j < Np * Q; j += G, w.next()) m = fmaxf(m, fabsf(deviation(src[j], dt, w.c, index[w.c])));
        set_scale(m);
      }
    }
    for (int r0 = 0; r0 < Np; r0 += rows) {
      const int nr = min(rows, Np - r0);
      const TIn* s0 = src + size_t(r0) * Q;
      float m = 0.f;
      Walk w(lane, G, Q);
      const int n = nr * Q;
      for (int j = lane; j < n;) {
        // several loads in flight per thread before the first is used
        constexpr int U = 4;
        TIn x[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (j + u * G < n) x[u] = s0[j + u * G];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (j + u * G >= n) break;
          if constexpr (ST::dev) {
            const DevIndex at = index[w.c];
            const float d = deviation(x[u], dt, w.c, at);
            m = fmaxf(m, fabsf(d));
            buf[w.row * Qp + at.at] = d;
          } else {
            buf[w.row * Qp + perm[w.c]] = T(x[u]);
          }
          w.next();
        }
        j += U * G;
      }
      if constexpr (ST::dev) {
        if (whole) set_scale(m);
      }
      group_sync<kWarp>();
      const int nvec = nr * Qp / V;
      S* d0 = dst + size_t(r0) * Qp;
      for (int v = lane; v < nvec; v += G) {
        __align__(16) S q[V];
        if constexpr (ST::dev) {
          __align__(16) float d[V];
#pragma unroll
          for (int j = 0; j < V / 4; ++j)
            reinterpret_cast<uint4*>(d)[j] = reinterpret_cast<const uint4*>(buf + size_t(v) * V)[j];
#pragma unroll
          for (int j = 0; j < V; ++j) {
            // the scale is a power of two; where its inverse leaves FP32's range, divide in FP64
            q[j] = sc >= 1e-30f ? ST::from_r(d[j] * inv_s) : ST::from_r(float(double(d[j]) / double(sc)));
          }
          reinterpret_cast<uint4*>(d0)[v] = *reinterpret_cast<const uint4*>(q);
        } else {
          reinterpret_cast<uint4*>(d0)[v] = reinterpret_cast<const uint4*>(buf)[v];
        }
      }
      group_sync<kWarp>();  // the buffer is free for the next rows (and red[] for the next element)
    }
  }
}

// Read-out of plain state through shared memory: the mirror image.  The internal row is
// read as 16-byte vectors and scattered into shared memory by the canonical order; the
// caller's rows are written along the canonical order.  31M FP32 values 73 us, 56 us the bytes
// at the measured rate; gathered 4-byte loads, a thread per value, 90 us.
template <class ST, bool kWarp>
__global__ void __launch_bounds__(kThreads) decode_kernel(const void* __restrict__ in, double* __restrict__ out,
                                                          const int32_t* __restrict__ iperm, int64_t K, int Np,
                                                          int Q, int Qp, int rows, int table_bytes) {
  using S = typename ST::S;
  constexpr int V = 16 / int(sizeof(S));
  extern __shared__ __align__(16) unsigned char smem[];
  int* inv = reinterpret_cast<int*>(smem);  // canonical index, -1 for padding
  for (int i = threadIdx.x; i < Qp; i += kThreads) inv[i] = -1;
  __syncthreads();
  for (int c = threadIdx.x; c < Q; c += kThreads) inv[iperm[c]] = c;
  const int G = kWarp ? 32 : kThreads;
  const int grp = kWarp ? threadIdx.x / 32 : 0, lane = kWarp ? threadIdx.x % 32 : threadIdx.x;
  const int ngroups = kWarp ? kThreads / 32 : 1;
  S* buf = reinterpret_cast<S*>(smem + table_bytes) + size_t(grp) * rows * Qp;
  __syncthreads();

  const int vrow = Qp / V;  // vectors per row
  for (int64_t k = blockIdx.x * int64_t(ngroups) + grp; k < K; k += int64_t(gridDim.x) * ngroups) {
    const S* src = static_cast<const S*>(in) + k * Np * Qp;
    double* dst = out + k * Np * Q;
    for (int r0 = 0; r0 < Np; r0 += rows) {
      const int nr = min(rows, Np - r0);
      const uint4* s0 = reinterpret_cast<const uint4*>(src + size_t(r0) * Qp);
      const int nvec = nr * vrow;
      Walk w(lane, G, vrow);
      for (int v = lane; v < nvec;) {
        constexpr int U = 2;
        uint4 x[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (v + u * G < nvec) x[u] = s0[v + u * G];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (v + u * G >= nvec) break;
          const S* q = reinterpret_cast<const S*>(&x[u]);
          S* row = buf + size_t(w.row) * Q;
#pragma unroll
          for (int j = 0; j < V; ++j) {
            const int c = inv[w.c * V + j];
            if (c >= 0) row[c] = q[j];
          }
          w.next();
        }
        v += U * G;
      }
      group_sync<kWarp>();
      double* d0 = dst + size_t(r0) * Q;
      const int n = nr * Q;
      for (int j = lane; j < n; j += G) d0[j] = widen(buf[j]);
      group_sync<kWarp>();
    }
  }
}

// Loads of plain state and read-outs without the staging: a thread per value, scattered
// and gathered by the velocity order.  Deviation forms are always read out so, as w + w (s q)
// with one FP64 FMA per value; the product s q is exact in FP32 (s is a power of two).
template <class ST, typename TIn>
__global__ void __launch_bounds__(kThreads) encode_direct_kernel(const TIn* __restrict__ in, void* out,
                                                                 const int32_t* __restrict__ iperm, int64_t K, int Np,
                                                                 int Q, int Qp) {
  using S = typename ST::S;
  const int64_t k = blockIdx.x;
  const TIn* src = in + k * Np * Q;
  S* dst = static_cast<S*>(out) + k * Np * Qp;
  const int pad = Qp - Q;
  for (int j = threadIdx.x; j < Np * Q; j += blockDim.x) {
    const int n = j / Q;
    dst[n * Qp + iperm[j - n * Q]] = S(src[j]);
  }
  for (int j = threadIdx.x; j < Np * pad; j += blockDim.x) dst[(j / pad) * Qp + Q + j % pad] = S(0);
}
template <class ST>
__global__ void __launch_bounds__(kThreads) decode_direct_kernel(const void* __restrict__ in,
                                                                 const float* __restrict__ scale,
                                                                 double* __restrict__ out,
                                                                 const double* __restrict__ vel64,
                                                                 const int32_t* __restrict__ iperm, int64_t rows,
                                                                 int Np, int Q, int Qp) {
  using S = typename ST::S;
  const double* w64 = vel64 + 2 * Qp;
  const int64_t n = rows * Q;
  for (int64_t j = blockIdx.x * int64_t(kThreads) + threadIdx.x; j < n; j += int64_t(gridDim.x) * kThreads) {
    const int64_t r = j / Q;
    const int i = iperm[int(j - r * Q)];
    const S q = static_cast<const S*>(in)[r * Qp + i];
    if constexpr (ST::dev) out[j] = fma(w64[i], widen(scale[r / Np] * ST::to_r(q)), w64[i]);
    else out[j] = widen(q);
  }
}

// Node moments.  G lanes share a node (as many as its row has 16-byte chunks,
// at most a warp) and a group takes kNodes consecutive nodes at once, so that
// each chunk's e_x, e_y (and w) are loaded once for kNodes nodes and the row
// loads of all of them are in flight together.  Sums and quotients in the
// state's compute precision R: FP64 arithmetic is slow here, and the FP32 and
// 16-bit states carry FP32 precision.  Before, one warp per node whatever the
// row's length, with the tables read again for every node: 480 us for 44M FP32
// values at 16 velocities (4 of 32 lanes busy; 26 us for the bytes) and 851 us
// for 335M BF16 values at 1,024 velocities (96 bytes of table per 16 of state);
// now 51 us and 192 us.
template <class ST, int kNodes>
__global__ void __launch_bounds__(kThreads) moments_kernel(const void* __restrict__ in,
                                                           const float* __restrict__ scale,
                                                           const typename ST::R* __restrict__ vel, int64_t nodes,
                                                           int Np, int Qp, int G, double* rho, double* ux,
                                                           double* uy) {
  using R = typename ST::R;
  using S = typename ST::S;
  constexpr int V = 16 / int(sizeof(S));
  const int lane = threadIdx.x % G;
  const int64_t ngroups = int64_t(gridDim.x) * (kThreads / G);
  const R *ex = vel + kVelEx * Qp, *ey = vel + kVelEy * Qp, *wv = vel + kVelW * Qp;
  // every lane of a warp runs the same number of iterations (the shuffles)
  const int64_t first = (blockIdx.x * int64_t(kThreads) + threadIdx.x) / G;
  const int64_t warp_first = (blockIdx.x * int64_t(kThreads) + threadIdx.x) / 32 * (32 / G);
  for (int64_t it = 0; (warp_first + it * ngroups) * kNodes < nodes; ++it) {
    const int64_t n0 = (first + it * ngroups) * kNodes;
    R m0[kNodes] = {}, m1[kNodes] = {}, m2[kNodes] = {}, s[kNodes] = {};
    const S* row[kNodes];
#pragma unroll
    for (int a = 0; a < kNodes; ++a) {
      const int64_t kn = n0 + a < nodes ? n0 + a : nodes - 1;  // past the end: read the last node again
      row[a] = static_cast<const S*>(in) + kn * Qp;
      if constexpr (ST::dev) s[a] = R(scale[kn / Np]);
    }
#pragma unroll 2
    for (int i = lane * V; i < Qp; i += G * V) {
      uint4 x[kNodes];
#pragma unroll
      for (int a = 0; a < kNodes; ++a) x[a] = *reinterpret_cast<const uint4*>(row[a] + i);
      __align__(16) R tx[V], ty[V], tw[V];
#pragma unroll
      for (int j = 0; j < V * int(sizeof(R)) / 16; ++j) {
        reinterpret_cast<uint4*>(tx)[j] = __ldg(reinterpret_cast<const uint4*>(ex + i) + j);
        reinterpret_cast<uint4*>(ty)[j] = __ldg(reinterpret_cast<const uint4*>(ey + i) + j);
        if constexpr (ST::dev) reinterpret_cast<uint4*>(tw)[j] = __ldg(reinterpret_cast<const uint4*>(wv + i) + j);
      }
#pragma unroll
      for (int a = 0; a < kNodes; ++a) {
        const S* q = reinterpret_cast<const S*>(&x[a]);
#pragma unroll
        for (int j = 0; j < V; ++j) {
          R f;
          if constexpr (ST::dev) f = fmaf(tw[j] * s[a], ST::to_r(q[j]), tw[j]);
          else f = R(q[j]);
          m0[a] += f;
          m1[a] = fma(tx[j], f, m1[a]);
          m2[a] = fma(ty[j], f, m2[a]);
        }
      }
    }
    for (int off = G >> 1; off > 0; off >>= 1) {
#pragma unroll
      for (int a = 0; a < kNodes; ++a) {
        m0[a] += __shfl_xor_sync(0xffffffffu, m0[a], off);
        m1[a] += __shfl_xor_sync(0xffffffffu, m1[a], off);
        m2[a] += __shfl_xor_sync(0xffffffffu, m2[a], off);
      }
    }
    // every lane holds the sums: lane a of the group writes node a, so that the
    // quotients of its nodes run side by side (fewer than kNodes lanes take turns)
    for (int a0 = 0; a0 < kNodes; a0 += (G < kNodes ? G : kNodes)) {
      const int a = a0 + lane;
      R r0 = m0[0], r1 = m1[0], r2 = m2[0];
#pragma unroll
      for (int b = 1; b < kNodes; ++b)
        if (a == b) {
          r0 = m0[b];
          r1 = m1[b];
          r2 = m2[b];
        }
      if (a < kNodes && n0 + a < nodes) {
        rho[n0 + a] = double(r0);
        ux[n0 + a] = double(r1 / r0);
        uy[n0 + a] = double(r2 / r0);
      }
    }
  }
}

// Where the direct kernels are taken: small calls, whose time is the staging's two trips
// through shared memory and its tables, and shapes that the staged split serves badly (tiny
// elements, of which a warp takes one at a time; elements of 768 to 1,536 values, whose eight
// buffers leave an SM few CTAs; elements of several passes).  Staged against direct on the
// GB300, us: loads of FP64 state, 1e4 values of 16 and 36
// velocities 6.2 and 4.2, 1e6 and 2e7 values of 256 velocities at degree 2 10.3 and 7.6, 72.5
// and 63.4, but 16 velocities at degree 2, 1e6 and 2e7 8.2 and 10.3, 65 and 109.  Read-outs:
// 16 velocities at degree 0, 2e7 FP32 values 274 and 62; 256 at degree 0 and 4 50 and 63, 47
// and 64, 1,089 at degree 5 67 and 61; BF16, 256 velocities, degree 4, 1e5, 4e6 and 2e7 values
// 7.6 and 4.1, 22.6 and 19.5, 89 and 82.  Of the deviation forms' 65 shapes the staged read-out was
// faster in one (8.3 and 10.3 us), so there is none any more.
bool warp_split(const Shape& sh) { return sh.Np * sh.Qp <= kWarpValues; }
bool direct_load(const Shape& sh, size_t value_bytes) {
  if (!warp_split(sh)) return false;
  const int64_t values = sh.K * sh.Np * sh.Q;
  const int element = sh.Np * sh.Qp;
  if (element > 1024) return value_bytes == 8 || values <= int64_t(8) << 20;
  if (element > 768 && values <= int64_t(value_bytes == 8 ? 8 : 2) << 20) return true;
  return sh.K <= 16 * sh.nsm && values <= 200000;
}
bool direct_read(const Shape& sh, size_t value_bytes) {
  const int64_t values = sh.K * sh.Np * sh.Q;
  const int element = sh.Np * sh.Qp;
  const bool f64 = value_bytes == 8, large = values >= int64_t(8) << 20;
  if (!warp_split(sh)) return element > 12000 || sh.K < (f64 ? 1 : 8) * sh.nsm;
  return values < 800000 || element * int(value_bytes) < 1024 || (element > 1024 && (f64 || !large));
}
// Moments: one node per group of lanes instead of four where the nodes do not fill the SMs
// (about 2.5 CTAs each), and for long FP64 rows.  Four against one, us: FP64, 672 nodes of 16
// velocities 9.2 and 6.2, 360 nodes of 256 16.4 and 8.2, 840 and 19,840 of 1,024 35 and 14, 160 and
// 151; BF16, 672 nodes of 16 5.1 and 4.1; FP32, 1.2M nodes of 16 29 and 44.
bool few_nodes(const Shape& sh, int64_t nodes, int G, size_t r_bytes) {
  return nodes * G <= int64_t(640) * sh.nsm || (r_bytes == 8 && sh.Qp >= 512);
}

// Work split and kernel of one transfer.
template <class Kernel>
struct Plan {
  Split split;
  Kernel kernel;
  cudaError_t allow_smem() const {
    if (split.smem <= 48 * 1024 || split.smem > kSmemCap) return cudaSuccess;  // a launch beyond is refused
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmemCap));
  }
};
template <class ST, typename TIn>
auto encode_plan(const Shape& sh, bool by_warp) {
  // internal indices; deviation forms: six words a velocity, for FP64 input w and 1/w behind them
  const size_t q = size_t(sh.Q);
  const size_t tables = !ST::dev ? 4 * q : sizeof(TIn) == 8 ? up16(24 * q) + 16 * q : 24 * q;
  const Split s = split_for(sh, tables, ST::dev ? 4 : sizeof(typename ST::S), by_warp);
  auto kernel = s.warp ? &encode_kernel<ST, TIn, true> : &encode_kernel<ST, TIn, false>;
  return Plan<decltype(kernel)>{s, kernel};
}
template <class ST>
auto decode_plan(const Shape& sh) {
  const Split s = split_for(sh, 4 * size_t(sh.Qp), sizeof(typename ST::S), warp_split(sh));
  auto kernel = s.warp ? &decode_kernel<ST, true> : &decode_kernel<ST, false>;
  return Plan<decltype(kernel)>{s, kernel};
}

// Elements by warps or by CTAs; few elements of the deviation forms by a CTA each, where a
// warp would walk one alone (336 values, 24 elements, FP64 input: 10.3 us by warps, 8.2 with the
// former CTA per element).
template <class ST>
bool load_by_warp(const Shape& sh) {
  return warp_split(sh) && (!ST::dev || sh.Np * sh.Qp <= 128 || sh.K >= 8 * sh.nsm);
}

// For every element count: a batch has cases of the same sizes and different counts.
template <class ST>
cudaError_t prepare_as(const Shape& sh) {
  cudaError_t e = cudaSuccess;
  for (bool by_warp : {false, true}) {
    if (by_warp && !warp_split(sh)) continue;
    if (e == cudaSuccess) e = encode_plan<ST, double>(sh, by_warp).allow_smem();
    if (e == cudaSuccess) e = encode_plan<ST, float>(sh, by_warp).allow_smem();
  }
  if constexpr (!ST::dev)
    if (e == cudaSuccess) e = decode_plan<ST>(sh).allow_smem();
  return e;
}

template <class ST, typename TIn>
cudaError_t encode_as(const Shape& sh, const TIn* in, void* out, float* scale, cudaStream_t st) {
  if constexpr (!ST::dev) {
    if (direct_load(sh, sizeof(typename ST::S))) {
      const int block = std::min(kThreads, (sh.Np * sh.Q + 31) / 32 * 32);
      encode_direct_kernel<ST, TIn><<<int(sh.K), block, 0, st>>>(in, out, sh.iperm, sh.K, sh.Np, sh.Q, sh.Qp);
      return cudaGetLastError();
    }
  }
  const auto plan = encode_plan<ST, TIn>(sh, load_by_warp<ST>(sh));
  const Split& s = plan.split;
  plan.kernel<<<s.grid, kThreads, s.smem, st>>>(in, out, scale, sh.vel64, sh.iperm, sh.weights, sh.K, sh.Np, sh.Q,
                                                sh.Qp, s.rows, int(s.tables));
  return cudaGetLastError();
}

template <class ST>
cudaError_t decode_as(const Shape& sh, const void* in, const float* scale, double* out, cudaStream_t st) {
  if (ST::dev || direct_read(sh, sizeof(typename ST::S))) {
    const int64_t rows = sh.K * sh.Np;
    const int64_t blocks = (rows * sh.Q + kThreads - 1) / kThreads;
    const int grid = int(std::max<int64_t>(1, std::min<int64_t>(blocks, int64_t(sh.nsm) * 32)));
    decode_direct_kernel<ST><<<grid, kThreads, 0, st>>>(in, scale, out, sh.vel64, sh.iperm, rows, sh.Np, sh.Q, sh.Qp);
    return cudaGetLastError();
  }
  if constexpr (!ST::dev) {
    const auto plan = decode_plan<ST>(sh);
    const Split& s = plan.split;
    plan.kernel<<<s.grid, kThreads, s.smem, st>>>(in, out, sh.iperm, sh.K, sh.Np, sh.Q, sh.Qp, s.rows, int(s.tables));
  }
  return cudaGetLastError();
}

template <class ST>
cudaError_t moments_as(const Shape& sh, const void* in, const float* scale, const void* vel, double* rho, double* ux,
                       double* uy, cudaStream_t st) {
  const int chunks = sh.Qp * int(sizeof(typename ST::S)) / 16;
  int G = 1;
  while (G < 32 && G < chunks) G *= 2;
  const int64_t nodes = sh.K * sh.Np;
  const bool few = few_nodes(sh, nodes, G, sizeof(typename ST::R));
  const int64_t per_block = (few ? 1 : 4) * (kThreads / G);
  const int grid = int(std::max<int64_t>(1, std::min<int64_t>((nodes + per_block - 1) / per_block, int64_t(sh.nsm) * 32)));
  auto kernel = few ? &moments_kernel<ST, 1> : &moments_kernel<ST, 4>;
  kernel<<<grid, kThreads, 0, st>>>(in, scale, static_cast<const typename ST::R*>(vel), nodes, sh.Np, sh.Qp, G, rho, ux,
                                    uy);
  return cudaGetLastError();
}

template <typename TIn>
cudaError_t encode_any(const Shape& sh, const TIn* in, void* out, float* scale, cudaStream_t st) {
  switch (sh.store) {
    case kStoreF64: return encode_as<StoreF64, TIn>(sh, in, out, scale, st);
    case kStoreF32: return encode_as<StoreF32, TIn>(sh, in, out, scale, st);
    case kStoreBF16: return encode_as<StoreBF16, TIn>(sh, in, out, scale, st);
    default: return encode_as<StoreF16, TIn>(sh, in, out, scale, st);
  }
}

}  // namespace

void weight_tables(const double* w, const int32_t* iperm, int Q, DevRow* row, DevIndex* index, double* wide) {
  for (int c = 0; c < Q; ++c) {
    const double v = w[iperm[c]], iw = v > 0 ? 1.0 / v : 0.0;
    const float wh = float(v), wl = float(v - double(wh)), wll = float(v - double(wh) - double(wl));
    const float ih = v < kTinyWeight ? std::nanf("") : float(iw);
    // the rest of 1/w from the residual 1 - w ih, formed exactly by an FMA
    row[c] = DevRow{wh, wl, ih, float(std::fma(-v, double(ih), 1.0) * iw)};
    index[c] = DevIndex{wll, iperm[c]};
    wide[2 * c] = v;
    wide[2 * c + 1] = iw;
  }
}

cudaError_t prepare(const Shape& sh) {
  switch (sh.store) {
    case kStoreF64: return prepare_as<StoreF64>(sh);
    case kStoreF32: return prepare_as<StoreF32>(sh);
    case kStoreBF16: return prepare_as<StoreBF16>(sh);
    default: return prepare_as<StoreF16>(sh);
  }
}

cudaError_t encode(const Shape& sh, const double* in, void* out, float* scale, cudaStream_t st) {
  return encode_any(sh, in, out, scale, st);
}
cudaError_t encode(const Shape& sh, const float* in, void* out, float* scale, cudaStream_t st) {
  return encode_any(sh, in, out, scale, st);
}

cudaError_t decode(const Shape& sh, const void* in, const float* scale, double* out, cudaStream_t st) {
  switch (sh.store) {
    case kStoreF64: return decode_as<StoreF64>(sh, in, scale, out, st);
    case kStoreF32: return decode_as<StoreF32>(sh, in, scale, out, st);
    case kStoreBF16: return decode_as<StoreBF16>(sh, in, scale, out, st);
    default: return decode_as<StoreF16>(sh, in, scale, out, st);
  }
}

cudaError_t moments(const Shape& sh, const void* in, const float* scale, const void* vel, double* rho, double* ux,
                    double* uy, cudaStream_t st) {
  switch (sh.store) {
    case kStoreF64: return moments_as<StoreF64>(sh, in, scale, vel, rho, ux, uy, st);
    case kStoreF32: return moments_as<StoreF32>(sh, in, scale, vel, rho, ux, uy, st);
    case kStoreBF16: return moments_as<StoreBF16>(sh, in, scale, vel, rho, ux, uy, st);
    default: return moments_as<StoreF16>(sh, in, scale, vel, rho, ux, uy, st);
  }
}

}  // namespace transfer
}  // namespace fedbm
