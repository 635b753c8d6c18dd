// Fused LSRK(5,4) stage kernel for polynomial degree FEDBM_P.
//
// One CTA owns a tile of `epc` consecutive elements and every velocity of
// them.  Per stage it computes, for each element, node and velocity,
//   rhs_i = -(e_i . grad) f_i                       volume term (Dr, Ds)
//           + LIFT (Fscale (F^- - F^*) . n)         upwind/central surface flux
//           - (f_i - f_i^eq(rho, u)) / tau          BGK collision, eq. feq
// which is the strong form of eq. byparts (Sec. II.B.1); neighbour traces come
// from the input state (an L2-resident re-read), wall traces from eq. FullBC
// or eq. UsedBC (Sec. II.A.4).  It then applies the 2N-storage update
//   res <- A res + dt rhs ; f <- f + B res
// and writes the new state to the other state buffer (neighbours still read
// the old one).
//
// Phases of a CTA:
//   1. bulk-copy (TMA) the element tile f[k0:k0+epc][Np][Qp] and its geometry
//      (first barrier), the residual tile and every neighbour face row (second
//      barrier) into shared memory;
//   2. node moments rho, u (Sec. II.A.2) by a G-lane reduction per node, kept
//      as the coefficients of f^eq/tau per node, while the second part lands;
//   3. wall numerators sum_{e.n>0} (e.n) f^- of eq. FullBC per wall node;
//   4. residual and update, one thread per (element, velocity) item, with
//      Dr, Ds, LIFT as instruction immediates (compile-time tables) or
//      constant-memory operands of unrolled FMAs on the even and odd parts of f
//      and of the flux (stage_eo.cuh); the FP32 and 16-bit states take two
//      velocities per thread as packed FP32 pairs, or one (stage_lanes);
//   5. deviation forms only: per-element scale from max |f/w - 1|, encode;
//   6. bulk-store the new state and residual tiles.
#include "device_common.cuh"
#include "stage_dispatch.h"

#include <type_traits>


#ifndef FEDBM_P
#error "FEDBM_P must be defined"
#endif

namespace fedbm {
namespace {

constexpr int P = FEDBM_P;
constexpr int NP = np_of(P);
constexpr int NFP = P + 1;
constexpr int NF = 3 * NFP;
constexpr int OFF_DR = 0;
constexpr int OFF_DS = NP * NP;
constexpr int OFF_LIFT = 2 * NP * NP;
constexpr int OPS_N = 2 * NP * NP + NP * NF;

// FP64 operators: the BF16 and TF32 pieces of the tensor-core operands are cut from them
static __constant__ double c_ops64[OPS_N];

#include "ops_tables.inc"

// Node index of face node a on face f (rows of the reference triangle start at
// a(P+1) - a(a-1)/2; face 0 is row 0, face 1 the row ends, face 2 the row starts).
__host__ __device__ constexpr int face_node(int f, int a) {
  return f == 0 ? a : (f == 1 ? a * (P + 1) - a * (a - 1) / 2 + (P - a) : a * (P + 1) - a * (a - 1) / 2);
}

constexpr unsigned kFull = 0xffffffffu;

// Packed FP32 pairs (two velocities of one node in a 64-bit register pair):
// fma.rn.f32x2 rounds each half exactly like fmaf.
__device__ __forceinline__ unsigned long long f2pack(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void f2unpack(unsigned long long p, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p));
}
__device__ __forceinline__ unsigned long long f2fma(unsigned long long a, unsigned long long b,
                                                    unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

__device__ __forceinline__ unsigned long long f2mul(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

#include "stage_eo.cuh"

// ---- moment accumulators ----------------------------------------------------
struct AccD {
  double s = 0.0;
  __device__ void add(double v) { s += v; }
  __device__ void add(float v) { s += widen(v); }
  __device__ void reduce(int G) {
    for (int off = G >> 1; off > 0; off >>= 1) s += __shfl_xor_sync(kFull, s, off);
  }
  __device__ double value() const { return s; }
};
struct AccF {
  float s = 0.f;
  __device__ void add(float v) { s += v; }
  __device__ void reduce(int G) {
    for (int off = G >> 1; off > 0; off >>= 1) s += __shfl_xor_sync(kFull, s, off);
  }
  __device__ float value() const { return s; }
};
// Neumaier's compensated summation (Neumaier 1974) in FP32.
struct AccN {
  float s = 0.f, c = 0.f;
  __device__ void add(float v) {
    const float t = s + v;
    c += (fabsf(s) >= fabsf(v)) ? (s - t) + v : (v - t) + s;
    s = t;
  }
  __device__ void reduce(int G) {
    for (int off = G >> 1; off > 0; off >>= 1) {
      const float s2 = __shfl_xor_sync(kFull, s, off);
      const float c2 = __shfl_xor_sync(kFull, c, off);
      const float t = s + s2;
      const float e = (fabsf(s) >= fabsf(s2)) ? (s - t) + s2 : (s2 - t) + s;
      c = c + c2 + e;
      s = t;
    }
  }
  __device__ float value() const { return s + c; }
};

__host__ __device__ constexpr int pow2_floor_32(int g) {
  return g >= 32 ? 32 : g >= 16 ? 16 : g >= 8 ? 8 : g >= 4 ? 4 : g >= 2 ? 2 : 1;
}

template <class ST>
__device__ __forceinline__ typename ST::R decode(const typename ST::S v, typename ST::R w, typename ST::R ws) {
  if constexpr (ST::dev) {
    return fmaf(ws, ST::to_r(v), w);
  } else {
    (void)w;
    (void)ws;
    return typename ST::R(v);
  }
}

// ---- asynchronous bulk copies (TMA, non-tensor) and their mbarrier -----------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// try_wait with a suspend-time hint: a thread whose phase is not complete is
// suspended until the phase completes or about hint_ns pass, instead of
// returning at once, so that waiting warps do not take issue slots from the
// warps that compute.
__device__ __forceinline__ bool mbar_try_wait_suspend(uint64_t* bar, uint32_t parity, uint32_t hint_ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(hint_ns)
      : "memory");
  return ok != 0;
}
// Wait for phase `parity` of the barrier for at most about `limit_ns` (each
// suspended try_wait lasts at most 20 us past the limit); false on timeout.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait_suspend(bar, parity, 20000u)) {
    if (global_timer_ns() - t0 > limit_ns) return false;
  }
  return true;
}
__device__ __forceinline__ void bulk_load(void* dst_smem, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst_smem)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, const void* src_smem, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src_smem)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// wait until every committed bulk store of this thread has finished reading shared memory
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Programmatic dependent launch: a stage kernel may be put on the SMs while the one
// before it still runs its last CTAs.  It lets its own successor do the same at once
// (launch_dependents), sets up its barriers and tables, which no earlier kernel
// writes, and waits for the kernels before it to have finished, with their writes
// visible, before it touches the state, the residual or the scales.  Its lifetime so
// overlaps its predecessors' writes of those three: they are read with ordinary loads
// or bulk copies, never through the non-coherent path (__ldg), which is specified only
// for data that nothing writes while the kernel lives and whose lines an older stage on
// the same SM may have brought in.  Face codes, velocity rows and wall tables are
// written by no kernel; the step counter of the stochastic rounding only by a kernel
// between two steps, which starts after the last stage of one has finished and finishes
// before the first of the next starts.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class R>
cudaError_t launch_stage_kernel(void (*kernel)(StageArgs<R>), int grid, int block, size_t smem, cudaStream_t st,
                                const StageArgs<R>& a, int cluster = 0) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(grid), 1, 1);
  cfg.blockDim = dim3(unsigned(block), 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = sizeof(R) == 4;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cluster > 1) {
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = unsigned(cluster);
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
  }
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

// Vector of the storage type covering 16 bytes.
template <class ST>
struct Vec16 {
  static constexpr int N = 16 / int(sizeof(typename ST::S));
};

// Phase 2: rho, u_x, u_y of every node of the tile into s_mom.  G lanes share a
// node; each lane reduces 16-byte chunks of the node's velocity row.
// Lanes per node group: the largest power of two <= 32 that gives every node
// of the tile a group and no lane more than one chunk fewer than another.
__host__ __device__ constexpr int moment_lanes(int nth, int epc, int nchunk) {
  int G = pow2_floor_32(nth / (epc * NP));
  while (G > 1 && G > nchunk) G >>= 1;
  return G;
}

// Node record: f^eq_i / tau = w_i [m0 + e_x m1 + e_y m2 + m3 (e.u)^2
// + (e.u)(m6 (e.u)^2 - m7)] with e.u = e_x m4 + e_y m5 (eq. feq; the m6, m7 terms
// are the third Hermite order of eq. Herm3a and vanish for eq_order 2); `it` is
// 1/tau of the element's case.
template <typename R>
__device__ __forceinline__ void node_record(R rho, R jx, R jy, R it, bool third, R (&m)[8]) {
  const R irho = R(1) / rho;
  const R ux = jx * irho, uy = jy * irho, uu = ux * ux + uy * uy;
  m[0] = rho * (R(1) - R(0.5) * uu) * it;
  m[1] = jx * it;
  m[2] = jy * it;
  m[3] = R(0.5) * rho * it;
  m[4] = ux;
  m[5] = uy;
  m[6] = third ? rho * it * R(1.0 / 6.0) : R(0);
  m[7] = third ? R(0.5) * rho * uu * it : R(0);
}

// How a tile keeps its node records: eight values in the compute precision R; or,
// for the kernels that take two velocities per thread, times the time step and with
// -m7, either as eight floats or as six packed pairs (each value twice) with the
// pairs (m6, -m7) of all nodes behind them.
enum RecordForm { kRecPlain, kRecStep, kRecPairs };
constexpr int kRecPairFloats = 12;
template <RecordForm F, typename R>
__device__ __forceinline__ void store_record(R* s_mom, int node, int nodes, R rho, R jx, R jy, const R* geo,
                                             bool third) {
  R m[8];
  node_record(rho, jx, jy, F == kRecPlain ? geo[kGeoInvTau] : geo[kGeoInvTau] * geo[kGeoDt], third, m);
  if constexpr (F == kRecPairs) {
    float4* r = reinterpret_cast<float4*>(s_mom + size_t(node) * kRecPairFloats);
    r[0] = make_float4(m[0], m[0], m[1], m[1]);
    r[1] = make_float4(m[2], m[2], m[3], m[3]);
    r[2] = make_float4(m[4], m[4], m[5], m[5]);
    reinterpret_cast<float2*>(s_mom + size_t(nodes) * kRecPairFloats)[node] = make_float2(m[6], -m[7]);
  } else {
    R* mm = s_mom + size_t(node) * 8;
#pragma unroll
    for (int j = 0; j < 7; ++j) mm[j] = m[j];
    mm[7] = F == kRecStep ? -m[7] : m[7];
  }
}

// NTH > 0: a CTA of NTH threads and EPC elements per tile (the tensor-core
// kernel), so the lane grouping and the chunk loop are compile-time.
template <class ST, class Acc, int QT, int NTH = 0, int EPC = 1, RecordForm F = kRecPlain>
__device__ void tile_moments(const StageArgs<typename ST::R>& a, const typename ST::S* s_f,
                             const float* s_scale, const typename ST::R* s_geo, typename ST::R* s_mom, int ne,
                             const typename ST::R* s_vel) {
  using R = typename ST::R;
  using S = typename ST::S;
  constexpr int V = Vec16<ST>::N;
  static_assert(NTH == 0 || QT > 0, "a compile-time CTA needs a compile-time velocity count");
  const int Qp = QT > 0 ? QT : a.Qp, tid = threadIdx.x, nth = NTH > 0 ? NTH : blockDim.x;
  const int nchunk = Qp / V;
  // below 128 velocities, where the tile depends on the element count, the lanes per
  // node do not: a case gives the same bits in a batch and on its own.  As many as the
  // usual tiles leave per node; few in FP64, whose additions are slow.
  constexpr bool kFew = QT == 0 && sizeof(R) == 8;
  const int want = kFew && Qp == 16 ? (P <= 1 ? 4 : P == 2 ? 2 : 1) : P <= 1 ? 8 : P <= 3 ? 4 : 2;
  const int short_lanes = QT == 16 ? 1 : min(pow2_floor_32(nchunk), want);
  const int G = NTH > 0 ? moment_lanes(NTH, EPC, (QT > 0 ? QT : 1) / V)
                        : Qp < 128 ? short_lanes : moment_lanes(nth, a.epc, nchunk);
  const int ngroups = nth / G, grp = tid / G, lane = tid % G;
  const int npair = ne * NP;
  const R* ex = s_vel + kVelEx * Qp;  // shared-memory copy of the velocity rows
  const R* ey = s_vel + kVelEy * Qp;
  const R* wv = s_vel + kVelW * Qp;
  for (int base = 0; base < npair; base += ngroups) {
    const int pair = base + grp;
    const bool valid = pair < npair;
    Acc m0, m1, m2;
    const S* row = s_f + size_t(valid ? pair : 0) * Qp;
    // packed sums of one chunk, added to p0, p1, p2
    unsigned long long p0 = 0, p1 = 0, p2 = 0;
    auto chunk_pairs = [&](int c) {
      __align__(16) S v[V];
      *reinterpret_cast<uint4*>(v) = *reinterpret_cast<const uint4*>(row + c * V);
#pragma unroll
      for (int j = 0; j < V; j += 2) {
        const unsigned long long x = *reinterpret_cast<const unsigned long long*>(ex + c * V + j);
        const unsigned long long y = *reinterpret_cast<const unsigned long long*>(ey + c * V + j);
        unsigned long long f;
        if constexpr (ST::dev) {
          f = f2mul(*reinterpret_cast<const unsigned long long*>(wv + c * V + j),
                    f2pack(ST::to_r(v[j]), ST::to_r(v[j + 1])));
        } else {
          f = f2pack(v[j], v[j + 1]);
        }
        p0 = EoPacked::add(p0, f);
        p1 = f2fma(x, f, p1);
        p2 = f2fma(y, f, p2);
      }
    };
    auto add_pairs = [&](Acc& a0, Acc& a1, Acc& a2) {
      float lo, hi;
      f2unpack(p0, lo, hi);
      a0.add(lo + hi);
      f2unpack(p1, lo, hi);
      a1.add(lo + hi);
      f2unpack(p2, lo, hi);
      a2.add(lo + hi);
    };
    // sums over a chunk in the compute precision, then one accumulator update
    auto chunk = [&](int c, Acc& a0, Acc& a1, Acc& a2) {
      if constexpr (sizeof(R) == 4) {
        p0 = p1 = p2 = 0ull;
        chunk_pairs(c);
        add_pairs(a0, a1, a2);
      } else {
        __align__(16) S v[V];
        *reinterpret_cast<uint4*>(v) = *reinterpret_cast<const uint4*>(row + c * V);
        R c0 = 0, c1 = 0, c2 = 0;
#pragma unroll
        for (int j = 0; j < V; ++j) {
          c0 += v[j];
          c1 = fma(ex[c * V + j], v[j], c1);
          c2 = fma(ey[c * V + j], v[j], c2);
        }
        a0.add(c0);
        a1.add(c1);
        a2.add(c2);
      }
    };
    // FP32 sums keep their packed pairs over the row
    constexpr bool kPairSums = std::is_same<Acc, AccF>::value && sizeof(R) == 4;
    auto take = [&](int c) {
      if constexpr (kPairSums) chunk_pairs(c);
      else chunk(c, m0, m1, m2);
    };
    if (valid) {
      if constexpr (NTH > 0) {
        constexpr int GC = moment_lanes(NTH > 0 ? NTH : 1, EPC, (QT > 0 ? QT : V) / V);
#pragma unroll 8
        for (int c = 0; c < (QT > 0 ? QT : V) / V; c += GC) take(c + lane);
      } else if constexpr (QT == 16 && kPairSums) {
        // one lane per node: neighbouring lanes' rows start in the same banks, so each
        // takes its chunks from another one on; summing over distances N/2, .., 1 gives
        // the same for every rotation
        constexpr int N = 16 / V;
        const int first = pair * 16 * int(sizeof(S)) / 128;
        unsigned long long q0[N], q1[N], q2[N];
#pragma unroll
        for (int j = 0; j < N; ++j) {
          p0 = p1 = p2 = 0ull;
          chunk_pairs((j + first) & (N - 1));
          q0[j] = p0;
          q1[j] = p1;
          q2[j] = p2;
        }
#pragma unroll
        for (int off = N / 2; off > 0; off >>= 1)
#pragma unroll
          for (int j = 0; j < off; ++j) {
            q0[j] = EoPacked::add(q0[j], q0[j + off]);
            q1[j] = EoPacked::add(q1[j], q1[j + off]);
            q2[j] = EoPacked::add(q2[j], q2[j + off]);
          }
        p0 = q0[0];
        p1 = q1[0];
        p2 = q2[0];
      } else {
        for (int c = lane; c < nchunk; c += G) take(c);
      }
    }
    if constexpr (kPairSums) add_pairs(m0, m1, m2);
    m0.reduce(G);
    m1.reduce(G);
    m2.reduce(G);
    if (valid && lane == 0) {
      // in the compute precision R: FP64 arithmetic is kept out of the FP32 paths
      R rho, jx, jy;
      if constexpr (ST::dev) {
        const R sc = s_scale[pair / NP];
        rho = a.W0 + sc * R(m0.value());
        jx = a.W1x + sc * R(m1.value());
        jy = a.W1y + sc * R(m2.value());
      } else {
        rho = R(m0.value());
        jx = R(m1.value());
        jy = R(m2.value());
      }
      store_record<F>(s_mom, pair, a.epc * NP, rho, jx, jy, s_geo + (pair / NP) * kGeoStrideDev, a.eq_order == 3);
    }
  }
}

// Phase 3: numerators of eq. FullBC, sum over outgoing velocities of (e.n) f^-.
template <class ST, int QT>
__device__ void tile_wall_numerators(const StageArgs<typename ST::R>& a, const typename ST::S* s_f,
                                     const typename ST::R* s_geo, const int* s_nbr,
                                     const float* s_scale, typename ST::R* s_wn, int ne,
                                     const typename ST::R* s_vel) {
  using R = typename ST::R;
  const int Qp = QT > 0 ? QT : a.Qp, tid = threadIdx.x, nth = blockDim.x;
  // lanes per wall node: a fixed number, so that the sum has one order whatever the tile
  const int G = Qp < 128 ? 8 : 32;
  const int grp = tid / G, lane = tid % G, step = G < 32 ? 32 / G : nth / G;
  const R* ex = s_vel + kVelEx * Qp;  // shared-memory copy of the velocity rows
  const R* ey = s_vel + kVelEy * Qp;
  const R* wv = s_vel + kVelW * Qp;
  // most tiles have no wall: every warp looks for the tile's wall faces, 32 at a time
  for (int f0 = 0; f0 < ne * 3; f0 += 32) {
    const int mine = f0 + (tid & 31);
    bool wall = false;
    if (mine < ne * 3) {
      const int code = s_nbr[mine];
      wall = code < 0 && __ldg(a.wall_den_inv + (-code - 1)) > R(0);
    }
    int nth_wall = 0;
    for (unsigned mask = __ballot_sync(kFull, wall); mask; mask &= mask - 1, ++nth_wall) {
      // short rows: a warp per face; long ones: a warp per node of each face
      if (G < 32 && nth_wall % (nth / 32) != tid / 32) continue;
      const int face = f0 + __ffs(mask) - 1, e = face / 3, fc = face - 3 * e;
      const R nxf = s_geo[e * kGeoStrideDev + 4 + 3 * fc];
      const R nyf = s_geo[e * kGeoStrideDev + 5 + 3 * fc];
      const R sc = ST::dev ? s_scale[e] : R(0);
      for (int base = 0; base < NFP; base += step) {
        const int aa = base + (G < 32 ? (tid & 31) / G : grp);
        R acc = 0;
        if (aa < NFP) {
          const int rs = aa * (P + 1) - aa * (aa - 1) / 2;
          const int node = (fc == 0) ? aa : (fc == 1 ? rs + (P - aa) : rs);
          const typename ST::S* row = s_f + (size_t(e) * NP + node) * Qp;
          for (int i = lane; i < Qp; i += G) {
            // the FMAs spelled out: left to the compiler they differ between kernels in the last bit
            const R en = fma(ex[i], nxf, ey[i] * nyf);
            const R w = ST::dev ? wv[i] : R(0);  // the plain forms do not use (or hold) the w row
            if (en > 0) acc = fma(en, decode<ST>(row[i], w, w * sc), acc);
          }
        }
        for (int off = G >> 1; off > 0; off >>= 1) acc += __shfl_xor_sync(kFull, acc, off);
        if (aa < NFP && lane == 0) s_wn[(e * 3 + fc) * NFP + aa] = acc;
      }
    }
  }
}

// new f of one value: decode, then f + B res (shared by the update and the
// encoding pass of the deviation forms so both see the same rounding)
template <class ST>
__device__ __forceinline__ typename ST::R new_f(typename ST::R fold, typename ST::R rkB, typename ST::R r) {
  return fma(rkB, r, fold);
}

// tau-scaled collision term w f^eq(rho, u)/tau - f/tau of one value, from the
// node record written by tile_moments (all zero when collision is off)
template <typename R>
__device__ __forceinline__ R collision(const R* mm, R ex, R ey, R w, R f, R inv_tau, bool third) {
  const R eu = ex * mm[4] + ey * mm[5];
  R feq = fma(ey, mm[2], fma(ex, mm[1], mm[0]));
  feq = fma(eu, mm[3] * eu, feq);
  if (third) feq = fma(eu, fma(mm[6], eu * eu, -mm[7]), feq);
  return fma(w, feq, -inv_tau * f);
}

// Deviation form whose 16-bit format has FP32's exponent range (BF16): a
// power-of-two element scale changes neither the rounding of q nor the decoded
// f = w (1 + s q), so the element keeps the scale it was encoded with and the
// new state is encoded where it is computed.  FP16 (|q| < 2^15) must rescale.
template <class ST>
__host__ __device__ constexpr bool keeps_scale() {
  if constexpr (ST::dev) return ST::qmax_log2 == 0;
  else return false;
}

// Node of face node aa of the neighbour that face code `code` (>= 0) names: its face
// (code >> 1) & 3, listed backwards where bit 0 is set.
__device__ __forceinline__ int trace_node(int code, int aa) {
  const int fn = (code >> 1) & 3;
  const int a2 = (code & 1) ? NFP - 1 - aa : aa;
  const int rs = a2 * (P + 1) - a2 * (a2 - 1) / 2;
  return fn == 0 ? a2 : (fn == 1 ? rs + (P - a2) : rs);
}

// With 16 velocities a face row is 64 bytes (FP32) or 32: copied row by row into
// shared memory, the copies' issue took 6 % of the kernel's instructions (about 90
// per element) and their tiles 30 % of its shared memory, though a velocity uses
// only the faces it enters through.  There the update reads its own traces from
// global memory (L2), eight lanes to a row.
template <class ST, int QT>
__host__ __device__ constexpr bool direct_traces() {
  return QT > 0 && stage_direct_traces(P, ST::kind, QT);
}
template <class ST, int QT>
__host__ __device__ constexpr RecordForm record_form() {
  return sizeof(typename ST::R) == 8 ? kRecPlain : direct_traces<ST, QT>() ? kRecPairs : kRecStep;
}

// Phase 4, FP64 state: residual, 2N-storage update and write-back of every
// (element, velocity) value of the tile, one velocity of one element per thread, f
// and the residual updated in place in shared memory.  A tile of at most one warp's
// items run by four warps or more (fewer elements than SMs) splits the nodes over the warps,
// one per SM sub-partition: FP64 instructions take 64 cycles a warp there, and a stage is
// one element's chain of them (8x8x2, degree 2, GH D2Q16: see auto_tile).
template <class ST, int QT>
__device__ __forceinline__ void value_update(const StageArgs<typename ST::R>& a,
                                             StageSmem<typename ST::R, typename ST::S>& sm, int ne, bool read_res) {
  using R = typename ST::R;
  static_assert(sizeof(R) == 8 && !ST::dev, "the FP64 state");
  const int Qp = QT > 0 ? QT : a.Qp;
  const R rkA = a.rkA, rkB = a.rkB, ab = a.ab;
  const bool third = a.eq_order == 3;
  const bool split = a.epc * Qp <= 32 && blockDim.x >= 128;
  const int part = split ? threadIdx.x / 32 : 0, nparts = split ? blockDim.x / 32 : 1;
  const int first = split ? threadIdx.x % 32 : threadIdx.x, stride = split ? 32 : blockDim.x;
  for (int item = first; split ? item < 32 : item < ne * Qp; item += stride) {
    const bool own = item < ne * Qp;  // split: every thread comes to the barrier below
    const int e = own ? item / Qp : 0, i = own ? item - e * Qp : 0;
    const R ex = a.vel[kVelEx * Qp + i], ey = a.vel[kVelEy * Qp + i], w = a.vel[kVelW * Qp + i];
    const R* g = sm.geo + e * kGeoStrideDev;
    const R dt = g[kGeoDt], inv_tau = g[kGeoInvTau];  // per element: cases of a batch differ
    const R ar = ex * g[0] + ey * g[2], as = ex * g[1] + ey * g[3];
    R* frow = sm.f + size_t(e) * NP * Qp + i;
    R* rrow = sm.res + size_t(e) * NP * Qp + i;
    R fr[NP];
#pragma unroll
    for (int m = 0; m < NP; ++m) fr[m] = frow[m * Qp];
    R flux[NF];
#pragma unroll
    for (int fc = 0; fc < 3; ++fc) {
      const R en = ex * g[4 + 3 * fc] + ey * g[5 + 3 * fc];
      const R c = R(0.5) * (en - ab * fabs(en)) * g[6 + 3 * fc];
      const int code = sm.nbr[e * 3 + fc];
      if (code >= 0) {
        const R* trow = sm.tr + size_t(e * NF + fc * NFP) * Qp + i;
#pragma unroll
        for (int aa = 0; aa < NFP; ++aa) flux[fc * NFP + aa] = c * (fr[face_node(fc, aa)] - trow[aa * Qp]);
      } else {
        const int slot = -code - 1;  // wall slot: 4 * case + side
        const R fb = a.wall_feq[slot * Qp + i];
        const R den_inv = __ldg(a.wall_den_inv + slot);
        const bool diffuse = den_inv > R(0);
        // incoming velocities take the wall state; outgoing ones have no jump
        const R scale = diffuse ? den_inv * fb : R(0);
#pragma unroll
        for (int aa = 0; aa < NFP; ++aa) {
          const R fp = diffuse ? sm.wn[e * NF + fc * NFP + aa] * scale : fb;
          flux[fc * NFP + aa] = en < R(0) ? c * (fr[face_node(fc, aa)] - fp) : R(0);
        }
      }
    }
    using M = EoScalar<R, false>;
    auto finish = [&](int n, R adv) {
      // f itself from shared memory again, which keeps the registers within two
      // resident CTAs of 256 threads
      const R f = frow[n * Qp];
      const R rhs = adv + collision<R>(sm.mom + (size_t(e) * NP + n) * 8, ex, ey, w, f, inv_tau, third);
      R r = dt * rhs;
      if (read_res) r = fma(rkA, rrow[n * Qp], r);
      rrow[n * Qp] = r;
      frow[n * Qp] = new_f<ST>(f, rkB, r);
    };
    auto value = [&](int n) { return fr[n]; };
    const R na = R(-0.5) * (ar + as), nd = R(0.5) * (ar - as);
    if (split) {
      __syncthreads();  // every warp has read f before one updates its nodes
      if (own) eo_part<M>(value, flux, na, nd, part, nparts, finish);
    } else {
      R le[NE], lo[at_least_1(NO)];
      eo_lift<M>(flux, true, true, le, lo);
      eo_volume<M>(value, na, nd, le, lo, finish);
    }
  }
}

// The velocities of a thread in the FP32-arithmetic update: two adjacent ones as packed
// FP32 pairs (the lower in the low half), or one.  Every operation rounds a velocity the
// same way in both, so that a value does not depend on which the tile has.  (A product
// that is added or subtracted is written as the FMA: the assembler fuses a packed product
// with the sum behind it in some places and not in others.)
using Pair = unsigned long long;
template <int N>
struct Lanes;
template <>
struct Lanes<2> : EoDual<kHaveOpsTable> {
  static __device__ __forceinline__ T both(float x) { return f2pack(x, x); }
  static __device__ __forceinline__ T mul(T x, T y) { return f2mul(x, y); }
  static __device__ __forceinline__ T load(const float* p) { return *reinterpret_cast<const T*>(p); }
  static __device__ __forceinline__ void store(float* p, T x) { *reinterpret_cast<T*>(p) = x; }
  template <class F>
  static __device__ __forceinline__ T map(T x, F f) {
    float a, b;
    f2unpack(x, a, b);
    return f2pack(f(a), f(b));
  }
  static __device__ __forceinline__ bool any(T x) {
    float a, b;
    f2unpack(x, a, b);
    return a != 0.f || b != 0.f;
  }
  static __device__ __forceinline__ float max_abs(T x) {
    float a, b;
    f2unpack(x, a, b);
    return fmaxf(fabsf(a), fabsf(b));
  }
  // two adjacent values of a node record that holds every value twice
  static __device__ __forceinline__ void record(const float* p, T& a, T& b) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    a = v.x;
    b = v.y;
  }
  // stored values as FP32
  template <class ST>
  static __device__ __forceinline__ T raw(const typename ST::S* p) {
    if constexpr (ST::kind == kStoreBF16) {
      const uint32_t q = *reinterpret_cast<const uint32_t*>(p);  // BF16: the upper half of an FP32
      return f2pack(__uint_as_float(q << 16), __uint_as_float(q & 0xffff0000u));
    } else if constexpr (ST::kind == kStoreF16) {
      const float2 x = __half22float2(*reinterpret_cast<const __half2*>(p));
      return f2pack(x.x, x.y);
    } else {
      return *reinterpret_cast<const T*>(p);
    }
  }
  using Code = __nv_bfloat162;
  static __device__ __forceinline__ Code to_bf16(T x) {
    float a, b;
    f2unpack(x, a, b);
    return __floats2bfloat162_rn(a, b);
  }
  // stochastic rounding; idx: the first value's index
  static __device__ __forceinline__ Code to_bf16(T x, uint64_t idx, uint32_t step, uint32_t stage) {
    float a, b;
    f2unpack(x, a, b);
    Code q;
    q.x = bf16_round_stochastic(a, sr_hash(idx, step, stage));
    q.y = bf16_round_stochastic(b, sr_hash(idx + 1, step, stage));
    return q;
  }
};
template <>
struct Lanes<1> : EoScalar<float, kHaveOpsTable> {
  static __device__ __forceinline__ T both(float x) { return x; }
  // not contracted into FMAs, as the packed ones are not
  static __device__ __forceinline__ T mul(T x, T y) { return __fmul_rn(x, y); }
  static __device__ __forceinline__ T add(T x, T y) { return __fadd_rn(x, y); }
  static __device__ __forceinline__ T sub(T x, T y) { return __fsub_rn(x, y); }
  static __device__ __forceinline__ T load(const float* p) { return *p; }
  static __device__ __forceinline__ void store(float* p, T x) { *p = x; }
  template <class F>
  static __device__ __forceinline__ T map(T x, F f) { return f(x); }
  static __device__ __forceinline__ bool any(T x) { return x != 0.f; }
  static __device__ __forceinline__ float max_abs(T x) { return fabsf(x); }
  static __device__ __forceinline__ void record(const float* p, T& a, T& b) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    a = v.x;
    b = v.z;
  }
  template <class ST>
  static __device__ __forceinline__ T raw(const typename ST::S* p) {
    if constexpr (ST::dev) return ST::to_r(*p);
    else return *p;
  }
  using Code = __nv_bfloat16;
  static __device__ __forceinline__ Code to_bf16(T x) { return __float2bfloat16_rn(x); }
  static __device__ __forceinline__ Code to_bf16(T x, uint64_t idx, uint32_t step, uint32_t stage) {
    return bf16_round_stochastic(x, sr_hash(idx, step, stage));
  }
};
// decoded: f, or w + (w s) q
template <class L, class ST>
__device__ __forceinline__ typename L::T lane_value(const typename ST::S* p, typename L::T w, typename L::T ws) {
  if constexpr (ST::dev) return L::fmat(ws, L::template raw<ST>(p), w);
  else return L::template raw<ST>(p);
}

// Phase 4, FP32 arithmetic: residual, 2N-storage update and write-back of every
// (element, velocity) value of the tile; each thread owns N adjacent velocities of one
// element.  With two, additions, collision, update, loads and stores act on packed
// FP32 pairs, the contractions on their halves with the operators as immediates;
// the time step is folded into the operators' factors, the flux coefficients and
// the node records.  Bound by instruction issue: 16 velocities at degree 5 in FP32 took
// 111 warp instructions per value and 239 us per stage of 44M values with one velocity
// per thread (98 us for the bytes), the whole four-step call 5169 us, with two 3730 us;
// BF16 5897 and 4630 us.  One velocity per thread serves tiles that a caller gives more
// threads than pairs (stage_lanes).  Plain forms and BF16 (kept element scale) update f in
// place in shared memory; FP16 only tracks max |f/w - 1| per element (the encoding pass
// recomputes f with the new scale).
template <class ST, int QT, int N>
__device__ __forceinline__ void lane_update(const StageArgs<float>& a, StageSmem<float, typename ST::S>& sm,
                                            int64_t k0, int ne, bool read_res, float& dmax, int& emax) {
  using S = typename ST::S;
  using L = Lanes<N>;
  using T = typename L::T;
  constexpr bool kDirect = direct_traces<ST, QT>();
  constexpr bool kKeep = keeps_scale<ST>();
  constexpr bool kTrack = ST::dev && !kKeep;
  // outflow faces skipped per warp where a warp's items belong to one element
  constexpr bool kSkip = QT >= 128;
  const int Qp = QT > 0 ? QT : a.Qp, Qv = Qp / N;
  const T rkA2 = L::both(a.rkA), rkB2 = L::both(a.rkB), zero = L::zero();
  const float ab = a.ab;
  const bool third = a.eq_order == 3;
  const S* fin = static_cast<const S*>(a.f_in);
  // stochastic rounding of the BF16 encode: the step counter is read once
  const bool sr = kKeep && a.sr_step != nullptr;
  const uint32_t sr_step = sr ? __ldg(a.sr_step) : 0u;
  for (int item = threadIdx.x; item < ne * Qv; item += blockDim.x) {
    const int e = item / Qv, i = N * (item - e * Qv);
    const T ex = L::load(sm.vel + kVelEx * Qp + i), ey = L::load(sm.vel + kVelEy * Qp + i);
    const T w = L::load(sm.vel + kVelW * Qp + i);
    const float* g = sm.geo + e * kGeoStrideDev;
    const float dt = g[kGeoDt];  // per element: cases of a batch differ
    const int* nb = sm.nbr + e * 3;
    // flux coefficients dt (e.n - ab |e.n|) Fscale / 2 of the three faces
    T c[3];
    bool on[3], nz[3];
#pragma unroll
    for (int fc = 0; fc < 3; ++fc) {
      const T en = L::fmat(ey, L::both(g[5 + 3 * fc]), L::mul(ex, L::both(g[4 + 3 * fc])));
      const float h = 0.5f * dt * g[6 + 3 * fc];
      const bool wall = nb[fc] < 0;  // incoming velocities take the wall state; outgoing ones have no jump
      c[fc] = L::map(en, [&](float v) {
        const float x = h * fmaf(-ab, fabsf(v), v);
        return wall && !(v < 0.f) ? 0.f : x;
      });
      nz[fc] = L::any(c[fc]);
      on[fc] = kSkip ? __any_sync(__activemask(), nz[fc]) : true;
    }
    // 16 velocities: the traces of the faces with flux straight from global memory,
    // all of them in flight before the first is used
    T tr[kDirect ? NF : 1];
    if constexpr (kDirect) {
      const uint32_t* rows = reinterpret_cast<const uint32_t*>(sm.tr) + e * NF;
#pragma unroll
      for (int fc = 0; fc < 3; ++fc)
#pragma unroll
        for (int aa = 0; aa < NFP; ++aa)
          tr[fc * NFP + aa] =
              nz[fc] && nb[fc] >= 0 ? L::template raw<ST>(fin + size_t(rows[fc * NFP + aa]) * QT + i) : zero;
    }
    const T ws = ST::dev ? L::mul(w, L::both(sm.scale[e])) : zero;
    S* frow = sm.f + size_t(e) * NP * Qp + i;
    float* rrow = sm.res + size_t(e) * NP * Qp + i;
    T fr[NP];
#pragma unroll
    for (int m = 0; m < NP; ++m) fr[m] = lane_value<L, ST>(frow + m * Qp, w, ws);
    T flux[NF];
#pragma unroll
    for (int fc = 0; fc < 3; ++fc) {
      const int code = nb[fc];
      if constexpr (kSkip) {
#pragma unroll
        for (int aa = 0; aa < NFP; ++aa) flux[fc * NFP + aa] = zero;
        if (!on[fc]) continue;
      }
      if (code >= 0) {
        const T wsn = ST::dev ? L::mul(w, L::both(sm.nscale[e * 3 + fc])) : zero;
        const S* trow = sm.tr + size_t(e * NF + fc * NFP) * Qp + i;
#pragma unroll
        for (int aa = 0; aa < NFP; ++aa) {
          T t;
          if constexpr (kDirect) t = ST::dev ? L::fmat(wsn, tr[fc * NFP + aa], w) : tr[fc * NFP + aa];
          else t = lane_value<L, ST>(trow + aa * Qp, w, wsn);
          flux[fc * NFP + aa] = L::mul(c[fc], L::sub(fr[face_node(fc, aa)], t));
        }
      } else {
        const int slot = -code - 1;  // wall slot: 4 * case + side
        const T fb = L::load(a.wall_feq + size_t(slot) * Qp + i);
        const float den_inv = __ldg(a.wall_den_inv + slot);
        const bool diffuse = den_inv > 0.f;
        const T fd = diffuse ? L::mul(L::both(den_inv), fb) : fb;
#pragma unroll
        for (int aa = 0; aa < NFP; ++aa) {
          const float m = diffuse ? -sm.wn[e * NF + fc * NFP + aa] : -1.f;
          flux[fc * NFP + aa] = L::mul(c[fc], L::fmat(L::both(m), fd, fr[face_node(fc, aa)]));
        }
      }
    }
    T le[NE], lo[at_least_1(NO)];
    eo_lift<L>(flux, on[0] || on[2], on[1], le, lo);
    const T neg_k = L::both(-dt * g[kGeoInvTau]);
    const T ar = L::fmat(ey, L::both(g[2]), L::mul(ex, L::both(g[0])));
    const T as = L::fmat(ey, L::both(g[3]), L::mul(ex, L::both(g[1])));
    const T na = L::mul(L::both(-0.5f * dt), L::add(ar, as)), nd = L::mul(L::both(0.5f * dt), L::sub(ar, as));
    T invw = zero;
    if constexpr (ST::dev)  // BF16 keeps the element's power-of-two scale: q = (f - w) / (w s)
      invw = L::mul(L::load(a.vel + kVelInvW * Qp + i), L::both(kKeep ? 1.0f / sm.scale[e] : 1.0f));
    float dloc = 0.f;
    // update and write-back of node n from dt times its advection term
    // -(e . grad) f + LIFT (flux)
    eo_volume<L>([&](int n) { return fr[n]; }, na, nd, le, lo, [&](int n, T adv) {
      T m0, m1, m2, m3, mx, my;
      const int node = e * NP + n;
      if constexpr (kDirect) {
        const float* mm = sm.mom + size_t(node) * kRecPairFloats;
        L::record(mm, m0, m1);
        L::record(mm + 4, m2, m3);
        L::record(mm + 8, mx, my);
      } else {
        const float4* mm = reinterpret_cast<const float4*>(sm.mom + size_t(node) * 8);
        const float4 u = mm[0], v = mm[1];
        m0 = L::both(u.x); m1 = L::both(u.y); m2 = L::both(u.z); m3 = L::both(u.w);
        mx = L::both(v.x); my = L::both(v.y);
      }
      // f itself from shared memory again: in registers next to its even and odd
      // parts it would cost a resident CTA
      const T f = lane_value<L, ST>(frow + n * Qp, w, ws);
      const T eu = L::fmat(ey, my, L::mul(ex, mx));
      T feq = L::fmat(ey, m2, L::fmat(ex, m1, m0));
      feq = L::fmat(eu, L::mul(m3, eu), feq);
      if (third) {
        float2 t;
        if constexpr (kDirect) t = reinterpret_cast<const float2*>(sm.mom + size_t(a.epc) * NP * kRecPairFloats)[node];
        else t = reinterpret_cast<const float2*>(sm.mom + size_t(node) * 8)[3];
        feq = L::fmat(eu, L::fmat(L::both(t.x), L::mul(eu, eu), L::both(t.y)), feq);
      }
      T r = L::fmat(w, feq, L::fmat(neg_k, f, adv));
      if (read_res) r = L::fmat(rkA2, L::load(rrow + n * Qp), r);
      L::store(rrow + n * Qp, r);
      const T fnew = L::fmat(rkB2, r, f);
      if constexpr (ST::dev) {
        const T q = L::mul(L::sub(fnew, w), invw);
        if constexpr (kTrack) {
          dloc = fmaxf(dloc, L::max_abs(q));
        } else {
          typename L::Code code;
          if (sr) {
            const uint64_t gi = (uint64_t(k0 + e) * NP + n) * uint64_t(Qp) + uint64_t(i);
            code = L::to_bf16(q, gi, sr_step, uint32_t(a.sr_stage));
          } else {
            code = L::to_bf16(q);
          }
          *reinterpret_cast<typename L::Code*>(frow + n * Qp) = code;
        }
      } else {
        L::store(frow + n * Qp, fnew);
      }
    });
    if constexpr (kTrack) {
      if (e != emax) {
        if (emax >= 0) atomicMax(&sm.dmax[emax], __float_as_uint(dmax));
        emax = e;
        dmax = 0.f;
      }
      dmax = fmaxf(dmax, dloc);
    }
  }
}

// Registers per thread of the FMA kernel, so that the tile's shared memory, not the
// register file, bounds the resident CTAs and the unrolled update spills little: at most
// 48 bytes in FP32 arithmetic (FP16, degree 5), 56, 32 and 108 bytes stored in FP64 at degree
// 3, 4 and 5.  One velocity per thread needs fewer: 80 let three CTAs of 256 threads share
// an SM (degree 4, 256 velocities, FP32, a step of 20M values 377 us, with 128 461 us).
template <class ST, int N>
__host__ __device__ constexpr int stage_max_regs() {
  return sizeof(typename ST::R) == 8 ? 128 : N == 1 ? 80 : P <= 2 ? 96 : P <= 4 ? 128 : 168;
}

// Bulk copies (TMA) of one tile into a shared-memory stage, issued by warp 0:
// element tile, residual tile (stages 2..5), geometry and every neighbour face
// row, all completing on the stage's mbarrier; the lanes also store the face
// codes (and for the deviation forms the scales) of the tile.
template <class ST, int QT>
__device__ void issue_tile_loads(const StageArgs<typename ST::R>& a, StageSmem<typename ST::R, typename ST::S>& sm,
                                 int64_t k0, int ne, bool read_res) {
  using R = typename ST::R;
  using S = typename ST::S;
  const int lane = threadIdx.x & 31;
  const int Qp = QT > 0 ? QT : a.Qp;
  const size_t row_bytes = size_t(Qp) * sizeof(S);
  const S* fin = static_cast<const S*>(a.f_in);
  const uint32_t tile_bytes = uint32_t(size_t(ne) * NP * row_bytes);
  const uint32_t res_bytes = uint32_t(size_t(ne) * NP * Qp * sizeof(R));
  const uint32_t geo_bytes = uint32_t(size_t(ne) * kGeoStrideDev * sizeof(R));
  // plain shared-memory stores first: the release of the arrive below makes
  // them visible to every thread that waits on the barrier
  for (int v = lane; v < ne * 3; v += 32) {
    const int code = __ldg(a.nbr + k0 * 3 + v);
    sm.nbr[v] = code;
    if constexpr (ST::dev) sm.nscale[v] = code >= 0 ? a.scale_in[code >> 3] : 0.f;
  }
  if constexpr (ST::dev) {
    for (int v = lane; v < ne; v += 32) {
      sm.scale[v] = a.scale_in[k0 + v];
      sm.dmax[v] = 0u;
    }
  }
  // two barriers: bar[0] for the element tile and geometry (needed first, by
  // the moment and wall-numerator reductions), bar[1] for the residual tile
  // and the neighbour traces (needed only by the update), so the reductions
  // start while the larger second part is still in flight
  uint64_t* bar_rt = sm.bar + 1;
  uint32_t bytes = 0;
  if (lane == 0) bytes += (read_res ? res_bytes : 0u);
  if constexpr (direct_traces<ST, QT>()) {
    // the update reads the traces itself: only their row numbers are left here
    uint32_t* rows = reinterpret_cast<uint32_t*>(sm.tr);
    for (int row = lane; row < ne * NF; row += 32) {
      const int code = __ldg(a.nbr + (k0 + row / NF) * 3 + (row % NF) / NFP);
      rows[row] = code >= 0 ? uint32_t(code >> 3) * NP + trace_node(code, row % NFP) : 0u;
    }
  } else {
    for (int row = lane; row < ne * NF; row += 32) {
      const int code = __ldg(a.nbr + (k0 + row / NF) * 3 + (row % NF) / NFP);
      if (code >= 0) bytes += uint32_t(row_bytes);
    }
  }
  mbar_arrive_expect_tx(sm.bar, lane == 0 ? tile_bytes + geo_bytes + a.extra_tx : 0u);
  mbar_arrive_expect_tx(bar_rt, bytes);
  if (lane == 0) {
    bulk_load(sm.f, fin + k0 * NP * Qp, tile_bytes, sm.bar);
    bulk_load(sm.geo, a.geo + k0 * kGeoStrideDev, geo_bytes, sm.bar);
    if (read_res) bulk_load(sm.res, a.res + k0 * NP * Qp, res_bytes, bar_rt);
  }
  if constexpr (!direct_traces<ST, QT>()) {
    for (int row = lane; row < ne * NF; row += 32) {
      const int e = row / NF, fc = (row % NF) / NFP, aa = row % NFP;
      const int code = __ldg(a.nbr + (k0 + e) * 3 + fc);
      if (code >= 0)
        bulk_load(sm.tr + size_t(row) * Qp, fin + (int64_t(code >> 3) * NP + trace_node(code, aa)) * Qp,
                  uint32_t(row_bytes), bar_rt);
    }
  }
}

// Persistent kernel: CTA b handles tiles b, b + gridDim.x, ... through two
// shared-memory stages, loading tile j+1 while it computes tile j.
// QT > 0: the padded velocity count is the compile-time constant QT (all
// shared-memory strides become immediate offsets); QT = 0: taken from a.Qp.
// N: velocities per thread of the update (FP32 arithmetic; the FP64 state has one).
template <class ST, int QT, int N>
__global__ void __maxnreg__((stage_max_regs<ST, N>())) stage_kernel(const StageArgs<typename ST::R> a) {
  using R = typename ST::R;
  using S = typename ST::S;
  extern __shared__ __align__(128) unsigned char smem[];
  const int epc = a.epc, Qp = QT > 0 ? QT : a.Qp;
  const int tid = threadIdx.x, nth = blockDim.x;
  const R rkA = a.rkA;
  const bool read_res = rkA != R(0);
  const int64_t ntiles = (a.K + epc - 1) / epc;
  constexpr bool kDirect = direct_traces<ST, QT>();
  const size_t stage_bytes = stage_smem_stride(NP, NF, epc, Qp, sizeof(S), sizeof(R), kDirect);
  auto stage = [&](int sidx) { return carve_stage_smem<R, S>(smem + sidx * stage_bytes, NP, NF, epc, Qp, kDirect); };
  const size_t row_bytes = size_t(Qp) * sizeof(S);

  const bool two = a.nstages == 2;
  pdl_launch_dependents();
  // velocity rows e_x, e_y, w into every stage's copy (read by the moment and
  // wall-numerator reductions)
  for (int sidx = 0; sidx < (two ? 2 : 1); ++sidx) {
    R* sv = stage(sidx).vel;
    for (int v = tid; v < 3 * Qp; v += nth) sv[v] = a.vel[v];
  }
  if (tid == 0) {
    mbar_init(stage(0).bar, 32);
    mbar_init(stage(0).bar + 1, 32);
    if (two) {  // the second stage exists only when nstages == 2
      mbar_init(stage(1).bar, 32);
      mbar_init(stage(1).bar + 1, 32);
    }
    fence_mbar_init();
    fence_proxy_async_smem();
  }
  pdl_wait();
  __syncthreads();

  int64_t tile = blockIdx.x;
  if (tid < 32 && tile < ntiles) {
    StageSmem<R, S> s0 = stage(0);
    issue_tile_loads<ST, QT>(a, s0, tile * epc, int(min(int64_t(epc), a.K - tile * epc)), read_res);
  }

  for (int j = 0; tile < ntiles; ++j, tile += gridDim.x) {
    StageSmem<R, S> sm = stage(two ? (j & 1) : 0);
    const uint32_t parity = uint32_t((two ? (j >> 1) : j) & 1);
    const int64_t k0 = tile * epc;
    const int ne = int(min(int64_t(epc), a.K - k0));
    const int64_t next = tile + gridDim.x;
    if (tid < 32) {
      if (two && next < ntiles) {
        // prefetch the next tile into the other stage once its bulk store has read it
        if (tid == 0) bulk_wait_read();
        __syncwarp();
        StageSmem<R, S> sn = stage((j + 1) & 1);
        issue_tile_loads<ST, QT>(a, sn, next * epc, int(min(int64_t(epc), a.K - next * epc)), read_res);
      } else if (!two && j > 0) {
        // single stage: load this tile once the previous tile's store has read it
        if (tid == 0) bulk_wait_read();
        __syncwarp();
        issue_tile_loads<ST, QT>(a, sm, k0, ne, read_res);
      }
    }
    // warp 0 waits for the tile (suspended in try_wait); the other warps
    // wait at the block barrier, where they take no issue slots
    bool ok = true;
    if (tid < 32) ok = mbar_wait_bounded(sm.bar, parity, 2000000000ull);
    if (__syncthreads_or(!ok)) {
      if (tid == 0 && a.err) atomicExch(a.err, 1);
      // let copies still in flight land before the CTA exits
      if (tid < 32) mbar_wait_bounded(sm.bar + 1, parity, 1000000000ull);
      if (tid < 32 && two && next < ntiles) {
        mbar_wait_bounded(stage((j + 1) & 1).bar, uint32_t(((j + 1) >> 1) & 1), 1000000000ull);
        mbar_wait_bounded(stage((j + 1) & 1).bar + 1, uint32_t(((j + 1) >> 1) & 1), 1000000000ull);
      }
      if (tid == 0) bulk_wait_read();
      return;
    }
    // the phase is complete: one try_wait gives every other thread its own
    // acquire of the copied data
    if (tid >= 32) mbar_try_wait(sm.bar, parity);

    // ---- 2. node moments ---------------------------------------------------------
    if (!a.collision) {
      const int words = kDirect ? epc * NP * (kRecPairFloats + 2) : ne * NP * 8;
      for (int v = tid; v < words; v += nth) sm.mom[v] = R(0);
    } else {
      // the usual large-Q tiles (one element, 128 or 256 threads) take the
      // moment reduction with compile-time lane groups and an unrolled loop
      auto moments = [&](auto acc) {
        using Acc = decltype(acc);
        constexpr int kBig = QT >= 128 ? 1 : 0;
        if (kBig && epc == 1 && nth == 128)
          tile_moments<ST, Acc, QT, kBig * 128, 1, record_form<ST, QT>()>(a, sm.f, sm.scale, sm.geo, sm.mom, ne, sm.vel);
        else if (kBig && epc == 1 && nth == 256)
          tile_moments<ST, Acc, QT, kBig * 256, 1, record_form<ST, QT>()>(a, sm.f, sm.scale, sm.geo, sm.mom, ne, sm.vel);
        else
          tile_moments<ST, Acc, QT, 0, 1, record_form<ST, QT>()>(a, sm.f, sm.scale, sm.geo, sm.mom, ne, sm.vel);
      };
      if constexpr (sizeof(R) == 8) {
        moments(AccD{});
      } else {
        if (a.red == kRedFP64) moments(AccD{});
        else if (a.red == kRedCompFP32) moments(AccN{});
        else moments(AccF{});
      }
    }
    // ---- 3. wall numerators ------------------------------------------------------
    if (a.wall_any) tile_wall_numerators<ST, QT>(a, sm.f, sm.geo, sm.nbr, sm.scale, sm.wn, ne, sm.vel);
    // the residual tile and the neighbour traces (bar[1]), as for bar[0]
    ok = true;
    if (tid < 32) ok = mbar_wait_bounded(sm.bar + 1, parity, 2000000000ull);
    if (__syncthreads_or(!ok)) {
      if (tid == 0 && a.err) atomicExch(a.err, 1);
      if (tid < 32 && two && next < ntiles)
        mbar_wait_bounded(stage((j + 1) & 1).bar + 1, uint32_t(((j + 1) >> 1) & 1), 1000000000ull);
      if (tid == 0) bulk_wait_read();
      return;
    }
    if (tid >= 32) mbar_try_wait(sm.bar + 1, parity);

    // ---- 4. residual and update ----------------------------------------------------
    float dmax = 0.f;  // deviation forms: running max |f/w - 1| of element emax
    int emax = -1;
    if constexpr (sizeof(R) == 8) value_update<ST, QT>(a, sm, ne, read_res);
    else lane_update<ST, QT, N>(a, sm, k0, ne, read_res, dmax, emax);

    // ---- 5. deviation forms: the kept scale (BF16), or the new per-element
    // scale and the encoding in place (FP16) ------------------------------------
    if constexpr (keeps_scale<ST>()) {
      for (int e = tid; e < ne; e += nth) a.scale_out[k0 + e] = sm.scale[e];
    } else if constexpr (ST::dev) {
      if (emax >= 0) atomicMax(&sm.dmax[emax], __float_as_uint(dmax));
      __syncthreads();
      for (int e = tid; e < ne; e += nth) {
        const float md = __uint_as_float(sm.dmax[e]);
        float sc = 1.0f;
        if (md > 0.f) {
          int ex2;
          frexpf(md, &ex2);
          sc = ldexpf(1.0f, ex2 - ST::qmax_log2);
        }
        sm.nscale[e] = sc;  // face scales are no longer needed
        a.scale_out[k0 + e] = sc;
      }
      __syncthreads();
      constexpr int V = Vec16<ST>::N;
      const int nvec = ne * NP * Qp / V;
      for (int v = tid; v < nvec; v += nth) {
        const int idx = v * V;
        const int e = idx / (NP * Qp);
        const int i0 = idx % Qp;
        const float sold = sm.scale[e];
        const float inv_s = 1.0f / sm.nscale[e];
        __align__(16) S q[V];
        *reinterpret_cast<uint4*>(q) = *reinterpret_cast<const uint4*>(sm.f + idx);
  #pragma unroll
        for (int j = 0; j < V; ++j) {
          const float w = __ldg(a.vel + kVelW * Qp + i0 + j);
          const float invw = __ldg(a.vel + kVelInvW * Qp + i0 + j);
          const float fold = decode<ST>(q[j], w, w * sold);
          const float fnew = new_f<ST>(fold, a.rkB, sm.res[idx + j]);
          q[j] = ST::from_r((fnew - w) * invw * inv_s);
        }
        *reinterpret_cast<uint4*>(sm.f + idx) = *reinterpret_cast<const uint4*>(q);
      }
    }


    // ---- 6. bulk store of the new state and residual tiles -----------------------
    fence_proxy_async_smem();
    __syncthreads();
    if (tid == 0) {
      bulk_store(static_cast<S*>(a.f_out) + k0 * NP * Qp, sm.f, uint32_t(size_t(ne) * NP * row_bytes));
      bulk_store(a.res + k0 * NP * Qp, sm.res, uint32_t(size_t(ne) * NP * Qp * sizeof(R)));
      bulk_commit();
    }
  }
  if (tid == 0) bulk_wait_read();
}

#include "stage_tc.cuh"
#include "stage_cluster.cuh"
#include "stage_ws.cuh"

// Velocity counts with a specialised kernel (the GH D2Q16 and NC 16x16 /
// 32x32 sets; the larger sets only at the degrees their workloads use, which
// keeps the high-degree translation units quick to compile); other counts use
// the runtime-stride kernel.
constexpr bool specialised_q(int Qp) {
  return (Qp == 16 && P <= 5) || (Qp == 256 && P <= 5) || (Qp == 1024 && P <= 4);
}

// fn(kernel) for the stage kernel of this state, velocity count and velocities per thread.
// (One velocity per thread needs more threads than pairs: never 1,024 velocities.)
template <class ST, int N, class Fn>
auto with_stage_kernel(int Qp, Fn fn) {
  if constexpr (ST::kind != kStoreF64) {
    if constexpr (specialised_q(16))
      if (Qp == 16) return fn(&stage_kernel<ST, 16, N>);
    if constexpr (specialised_q(256))
      if (Qp == 256) return fn(&stage_kernel<ST, 256, N>);
    if constexpr (specialised_q(1024) && N == 2)
      if (Qp == 1024) return fn(&stage_kernel<ST, 1024, N>);
  }
  return fn(&stage_kernel<ST, 0, N>);
}
template <class Fn>
auto with_f32_kernel(int store_kind, int Qp, int lanes, Fn fn) {
  switch (store_kind) {
    case kStoreF32: return lanes == 1 ? with_stage_kernel<StoreF32, 1>(Qp, fn) : with_stage_kernel<StoreF32, 2>(Qp, fn);
    case kStoreBF16: return lanes == 1 ? with_stage_kernel<StoreBF16, 1>(Qp, fn) : with_stage_kernel<StoreBF16, 2>(Qp, fn);
    default: return lanes == 1 ? with_stage_kernel<StoreF16, 1>(Qp, fn) : with_stage_kernel<StoreF16, 2>(Qp, fn);
  }
}

// resident CTAs per SM of the kernel a launch with these parameters uses
int occupancy(int store_kind, int Qp, int lanes, int block, size_t smem) {
  int n = 0;
  auto occ = [&](auto kernel) { return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, block, smem); };
  if (store_kind == kStoreF64) with_stage_kernel<StoreF64, 1>(Qp, occ);
  else with_f32_kernel(store_kind, Qp, lanes, occ);
  return n;
}

cudaError_t launch(int store_kind, const void* args, int lanes, int grid, int block, size_t smem, cudaStream_t st) {
  if (store_kind == kStoreF64) {
    const auto& a = *static_cast<const StageArgs<double>*>(args);
    return with_stage_kernel<StoreF64, 1>(
        a.Qp, [&](auto kernel) { return launch_stage_kernel(kernel, grid, block, smem, st, a); });
  }
  const auto& a = *static_cast<const StageArgs<float>*>(args);
  return with_f32_kernel(store_kind, a.Qp, lanes,
                         [&](auto kernel) { return launch_stage_kernel(kernel, grid, block, smem, st, a); });
}

cudaError_t set_smem(int store_kind, int Qp, int lanes, size_t smem) {
  auto set = [smem](auto kernel) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  };
  if (store_kind == kStoreF64) return with_stage_kernel<StoreF64, 1>(Qp, set);
  return with_f32_kernel(store_kind, Qp, lanes, set);
}

cudaError_t upload(const double* Dr, const double* Ds, const double* LIFT) {
  double h64[OPS_N], eo64[EO_N] = {};
  float eo32[EO_N];
  for (int j = 0; j < NP * NP; ++j) {
    h64[OFF_DR + j] = Dr[j];
    h64[OFF_DS + j] = Ds[j];
  }
  for (int j = 0; j < NP * NF; ++j) h64[OFF_LIFT + j] = LIFT[j];
  eo_coefficients(Dr, Ds, LIFT, eo64);
  for (int j = 0; j < EO_N; ++j) eo32[j] = float(eo64[j]);
  cudaError_t e = cudaMemcpyToSymbol(c_ops64, h64, sizeof(h64));
  if (e != cudaSuccess) return e;
  e = cudaMemcpyToSymbol(c_eo64, eo64, sizeof(eo64));
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbol(c_eo32, eo32, sizeof(eo32));
}

}  // namespace

StageEntry FEDBM_STAGE_ENTRY_NAME() {
  StageEntry s;
  s.launch = &launch;
  s.set_smem = &set_smem;
  s.upload = &upload;
  s.occupancy = &occupancy;
  s.tc_smem = &tc_smem;
  s.tc_tmem_cols = &tc_tmem_cols;
  s.launch_tc = &launch_tc;
  s.set_smem_tc = &set_smem_tc;
  s.occupancy_tc = &occupancy_tc;
  s.cl_smem = &cl_smem;
  s.launch_cl = &launch_cl;
  s.set_smem_cl = &set_smem_cl;
  s.occupancy_cl = &occupancy_cl;
  s.ws_smem = &ws_smem;
  s.ws_threads = &ws_threads;
  s.launch_ws = &launch_ws;
  s.set_smem_ws = &set_smem_ws;
  s.occupancy_ws = &occupancy_ws;
  return s;
}

}  // namespace fedbm
