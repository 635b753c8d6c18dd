// Warp-specialised form of the FMA stage kernel for 256 and 1,024 velocities (the
// NC 16 x 16 and 32 x 32 sets) and, as its wide form, any count from 512 up; FP32 or BF16
// deviation state.  Included by
// stage_impl.cuh inside its namespace; the arithmetic of a stage is that of the
// FMA kernel.
//
// A CTA has one to three groups of four consumer warps, each thread taking two
// adjacent velocities of an element (256 velocities in one pass, 1,024 in four; or one
// group of eight warps with one velocity per thread), and one producer warp.  The producer keeps a ring of shared-memory stages filled with
// the next elements' state tiles, geometry and neighbour face rows (bulk copies, one
// "full" mbarrier per stage); the groups take the elements in turn, reduce the node
// moments and wall numerators from the stage, read their own residual columns
// straight from global memory (issued before the reductions; the producer has
// brought the lines into L2), evaluate volume, flux, lift, collision and the update,
// write the new state and residual columns straight to global memory, and release
// the stage on its "empty" mbarrier.  So the consumers do not wait for copies while
// the ring is ahead of them, which the single-buffered kernel does once per tile.
//
// Two velocities per thread: additions, collision, update, loads and stores act on
// packed FP32 pairs (one instruction for both velocities; the node records are
// stored twice over so that they load as pairs), the contractions on their
// halves with the operators as immediates, and every chain of FMAs has a twin
// to hide its latency behind.  The time step is folded into the operators'
// factors, the flux coefficients and the node records, so that the update of a
// value takes ten operations after the contractions.
//
// What bounds it (ncu, 64 x 64 x 2 cavity, degree 4, 256 velocities, FP32, one
// launch): 53M warp instructions instead of the 71.5M of one velocity per thread
// with eight consumer warps per CTA, 51 % issue against 64 %, 91 us against 96 us (70 us
// for the bytes): the 12 consumer warps an SM holds at 128 registers wait for shared
// memory and for the residual.  The L2 prefetch of the residual is worth 8 % (99 us
// without).  Tried and slower: the residual an element ahead in registers (103 us),
// f read again from shared memory instead of kept across the lift, one CTA of three
// groups per SM with 256 velocities, two CTAs per SM without spills.  1,024
// velocities (64 x 64 x 2, degree 3, BF16, FP64 sums): 495 us with the FMA kernel, 389
// us with two CTAs of eight consumer warps per SM and 96 registers; one CTA of three
// groups of four has the call at 14.1 ms instead of 18.7 ms.
//
// Wide form (QT == 0): the ring holds the element's state only, 94 KB at 1,120
// velocities and degree 5, and the consumers read the neighbour traces they enter
// through straight from L2, so that two stages fit an SM and an element's velocities
// need not be split over a cluster: D2Q1089 at degree 5, 2,048 elements, a call of
// three steps 8146 -> 5212 us against the velocity-split kernel.
//
// Every wait is bounded by %globaltimer.  Consumer warp 0 waits on the full
// barrier and the consumers agree on the outcome with a reducing named
// barrier; on a timeout the consumers record it and leave, the producer stops
// issuing and, before it leaves, waits (bounded) for the copies it issued.

namespace ws {

// Shape of one form: G consumer groups per CTA (each takes every G-th element of
// the CTA), the threads of a group, resident CTAs and registers per thread.  The
// register file of each of the SM's four sub-partitions holds 16,384 registers
// and the warps are dealt out over them: four warps each leave 128 registers per
// thread, five 96, three 168, seven 72.
//
// The form asked for by number with 256 velocities has eight consumer warps (288
// threads), whatever the automatic one has.  Two groups of four warps with two velocities
// per thread hold their registers only up to degree 3 with two CTAs on an SM (degree 1:
// three, one producer warp being short of that many small elements); above, one group of
// eight warps takes one velocity per thread.  One step of 31M values, us, at degree 1..5:
// the former kernel (one velocity per thread, BF16 on tensor cores) FP32 676, 538, 519,
// 523, 845, BF16 1283, 893, 668, 586, 697; two groups, one CTA per SM 819, 839, 599, 584,
// 644 and 994, 1034, 709, 611, 672; now 611, 508, 466, 504, 540 and 732, 602, 565, 582, 621.
template <int QT, int G, int N>
__host__ __device__ constexpr int ctas() {
  if (N == 1) return 2;
  if (G == 2) return P <= 1 ? 3 : 2;
  return QT == 0 || G > 1 ? 1 : P <= 2 ? 4 : P <= 4 ? 3 : 2;
}
template <int QT, int G, int N>
__host__ __device__ constexpr int max_regs() {
  if (N == 1) return 96;
  if (G == 2) return P <= 1 ? 72 : 96;
  return QT == 0 ? 168 : G == 3 ? 128 : P <= 2 ? 96 : P <= 4 ? 128 : 168;
}
// Consumer threads of a group.  The wide form (QT == 0: the velocity count is taken
// from the arguments) has one group of at most eleven warps, three warps per
// sub-partition with the producer, and as few as cover the velocities in the same
// number of passes.
template <int QT, int N>
__host__ __device__ constexpr int group_threads(int Q) {
  if (QT > 0) return N == 1 ? 256 : 128;
  const int pairs = Q / 2, passes = (pairs + 351) / 352;
  return ((pairs + passes - 1) / passes + 31) / 32 * 32;
}
template <int QT, int G, int N>
__host__ __device__ constexpr int threads(int Q) { return G * group_threads<QT, N>(Q) + 32; }

// named barrier of a group's N threads, OR-reducing a predicate
__device__ __forceinline__ bool consumers_sync_or(int id, int N, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.red.or.pred q, %3, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(pred ? 1u : 0u), "r"(N), "r"(id)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ void consumers_sync(int id, int N) {
  asm volatile("barrier.sync %1, %0;" ::"r"(N), "r"(id) : "memory");
}
// plain arrive (release) of this thread on a barrier
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Wait until *word == want for at most about limit_ns; false on timeout.
__device__ __forceinline__ bool wait_for_number(const int* word, int want, uint64_t limit_ns) {
  const volatile int* w = word;
  if (*w == want) return true;
  const uint64_t t0 = global_timer_ns();
  while (*w != want) {
    if (global_timer_ns() - t0 > limit_ns) return false;
    __nanosleep(40);
  }
  return true;
}

// Node record: eight coefficients of dt f^eq / tau, each stored twice
// (c0, c1, c2, c3, u_x, u_y, c6, c7; see node_record).
constexpr int kRec = 16;

// Shared-memory layout: per ring stage the state tile [NP][Q], the neighbour face
// rows [NF][Q] (not in the wide form), the geometry, face codes and scales, two barriers; once per
// CTA the velocity rows (e_x, e_y, w and, for the deviation forms, w e_x, w e_y, 1/w)
// and two alternating sets of node records and wall numerators.
struct Layout {
  size_t stage, f, tr, geo, nbr, scale, nscale, bars;
  size_t vel, mom, wn, end;
  int stages;
};
__host__ __device__ constexpr size_t up(size_t b, size_t a) { return (b + a - 1) / a * a; }
template <class ST, int QT, int G, int N>
__host__ __device__ constexpr Layout layout(int Q) {
  Layout o{};
  constexpr size_t sb = sizeof(typename ST::S);
  size_t b = 0;
  o.f = b;      b += up(size_t(NP) * Q * sb, 16);
  o.tr = b;     b += QT == 0 ? 0 : up(size_t(NF) * Q * sb, 16);
  o.geo = b;    b += up(size_t(kGeoStrideDev) * 4, 16);
  o.nbr = b;    b += 16;
  o.scale = b;  b += 16;
  o.nscale = b; b += 16;
  o.bars = b;   b += 16;                   // full, empty
  o.stage = up(b, 128);
  const size_t fixed = up(size_t(ST::dev ? 6 : 3) * Q * 4, 16) + size_t(2 * G) * NP * kRec * 4 + up(size_t(2 * G) * NF * 4, 16);
  // as many stages as let the CTAs share an SM (1 KB of each is the system's), two to four
  const size_t room = (size_t(228) * 1024) / ctas<QT, G, N>() - 1024 - fixed;
  o.stages = int(room / o.stage);
  o.stages = o.stages < 2 ? 2 : o.stages > 4 * G ? 4 * G : o.stages;
  b = o.stage * o.stages;
  o.vel = b;    b += up(size_t(ST::dev ? 6 : 3) * Q * 4, 16);
  o.mom = b;    b += size_t(2 * G) * NP * kRec * 4;
  o.wn = b;     b += up(size_t(2 * G) * NF * 4, 16);
  o.end = b;
  return o;
}

// Moments of every node of the element in `row0` and their records.  G lanes
// share a node; a lane sums packed pairs over its 16-byte chunks (the FP64 and
// compensated modes take one accumulator update per chunk).
template <class ST, class Acc, int QT, int NT>
__device__ __forceinline__ void element_moments(const StageArgs<float>& a, const typename ST::S* row0, float sc,
                                                const float* s_vel, float kappa, float* rec, int tid, int nth) {
  const int Q = QT > 0 ? QT : a.Qp, NTH = QT > 0 ? NT : nth;
  constexpr int V = Vec16<ST>::N;
  const int NCH = Q / V;
  // lanes per node: a power of two that divides the chunks' loop evenly for the
  // compile-time counts; the wide form's last round of chunks may be partial
  const int G = moment_lanes(NTH, 1, NCH);
  constexpr bool kFast = std::is_same<Acc, AccF>::value;
  const int grp = tid / G, lane = tid % G;
  const bool third = a.eq_order == 3;
  const float* t0 = s_vel + 2 * Q;                       // w (deviation forms)
  const float* t1 = s_vel + (ST::dev ? 3 : 0) * Q;       // (w) e_x
  const float* t2 = s_vel + (ST::dev ? 4 : 1) * Q;       // (w) e_y
#pragma unroll 1
  for (int base = 0; base < NP; base += NTH / G) {
    const int n = base + grp;
    const bool valid = n < NP;
    Acc m0, m1, m2;
    Pair p0 = 0, p1 = 0, p2 = 0;
    if (valid) {
      const typename ST::S* row = row0 + n * Q;
#pragma unroll 8
      for (int c = 0; c < NCH; c += G) {
        if (QT == 0 && c + lane >= NCH) break;
        const int i = (c + lane) * V;
        const uint4 x = *reinterpret_cast<const uint4*>(row + i);
        const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
        if constexpr (!kFast) p0 = p1 = p2 = 0;
#pragma unroll
        for (int j = 0; j < V / 4; ++j) {
          const ulonglong2 u1 = *reinterpret_cast<const ulonglong2*>(t1 + i + 4 * j);
          const ulonglong2 u2 = *reinterpret_cast<const ulonglong2*>(t2 + i + 4 * j);
          if constexpr (ST::dev) {
            const ulonglong2 u0 = *reinterpret_cast<const ulonglong2*>(t0 + i + 4 * j);
            const Pair fa = f2pack(__uint_as_float(xs[2 * j] << 16), __uint_as_float(xs[2 * j] & 0xffff0000u));
            const Pair fb = f2pack(__uint_as_float(xs[2 * j + 1] << 16), __uint_as_float(xs[2 * j + 1] & 0xffff0000u));
            p0 = f2fma(u0.x, fa, p0);
            p1 = f2fma(u1.x, fa, p1);
            p2 = f2fma(u2.x, fa, p2);
            p0 = f2fma(u0.y, fb, p0);
            p1 = f2fma(u1.y, fb, p1);
            p2 = f2fma(u2.y, fb, p2);
          } else {
            const Pair fa = f2pack(__uint_as_float(xs[0]), __uint_as_float(xs[1]));
            const Pair fb = f2pack(__uint_as_float(xs[2]), __uint_as_float(xs[3]));
            p0 = EoPacked::add(p0, fa);
            p1 = f2fma(u1.x, fa, p1);
            p2 = f2fma(u2.x, fa, p2);
            p0 = EoPacked::add(p0, fb);
            p1 = f2fma(u1.y, fb, p1);
            p2 = f2fma(u2.y, fb, p2);
          }
        }
        if constexpr (!kFast) {
          float lo, hi;
          f2unpack(p0, lo, hi);
          m0.add(lo + hi);
          f2unpack(p1, lo, hi);
          m1.add(lo + hi);
          f2unpack(p2, lo, hi);
          m2.add(lo + hi);
        }
      }
    }
    if constexpr (kFast) {
      float lo, hi;
      f2unpack(p0, lo, hi);
      m0.add(lo + hi);
      f2unpack(p1, lo, hi);
      m1.add(lo + hi);
      f2unpack(p2, lo, hi);
      m2.add(lo + hi);
    }
    m0.reduce(G);
    m1.reduce(G);
    m2.reduce(G);
    if (valid && lane == 0) {
      float rho = float(m0.value()), jx = float(m1.value()), jy = float(m2.value());
      if constexpr (ST::dev) {
        rho = a.W0 + sc * rho;
        jx = a.W1x + sc * jx;
        jy = a.W1y + sc * jy;
      }
      // kappa = dt / tau; the coefficients of node_record times dt
      const float irho = 1.f / rho;
      const float ux = jx * irho, uy = jy * irho, uu = ux * ux + uy * uy;
      float4* r = reinterpret_cast<float4*>(rec + n * kRec);
      const float c0 = rho * (1.f - 0.5f * uu) * kappa, c1 = jx * kappa, c2 = jy * kappa, c3 = 0.5f * rho * kappa;
      r[0] = make_float4(c0, c0, c1, c1);
      r[1] = make_float4(c2, c2, c3, c3);
      r[2] = make_float4(ux, ux, uy, uy);
      if (third) {
        const float c6 = rho * kappa * (1.f / 6.f), c7 = -0.5f * rho * uu * kappa;
        r[3] = make_float4(c6, c6, c7, c7);
      }
    }
  }
}

template <class ST, int QT, int G, int N>
__global__ void __maxnreg__((max_regs<QT, G, N>())) stage_kernel_ws(const StageArgs<float> a) {
  using S = typename ST::S;
  using L = Lanes<N>;
  using T = typename L::T;
  constexpr bool kWide = QT == 0;
  const int Q = kWide ? a.Qp : QT;
  constexpr Layout oc = layout<ST, QT, G, N>(kWide ? 512 : QT);
  const Layout o = kWide ? layout<ST, QT, G, N>(Q) : oc;
  constexpr int kThreadsOf = group_threads<QT, N>(QT > 0 ? QT : 512);
  const int NC = kWide ? int(blockDim.x) - 32 : kThreadsOf, NST = kWide ? o.stages : oc.stages;
  const int kPasses = (Q + N * NC - 1) / (N * NC);
  extern __shared__ __align__(128) unsigned char smem[];
  const bool producer = threadIdx.x >= G * NC;
  const int group = producer ? 0 : threadIdx.x / NC;
  const int tid = threadIdx.x - group * NC;  // inside the group
  const int64_t K = a.K;
  const bool read_res = a.rkA != 0.f;
  const bool third = a.eq_order == 3;
  const S* fin = static_cast<const S*>(a.f_in);
  S* fout = static_cast<S*>(a.f_out);
  float* s_vel = reinterpret_cast<float*>(smem + o.vel);
  auto st_f = [&](int s) { return reinterpret_cast<S*>(smem + s * o.stage + o.f); };
  auto st_tr = [&](int s) { return reinterpret_cast<S*>(smem + s * o.stage + o.tr); };
  auto st_geo = [&](int s) { return reinterpret_cast<float*>(smem + s * o.stage + o.geo); };
  auto st_nbr = [&](int s) { return reinterpret_cast<int*>(smem + s * o.stage + o.nbr); };
  auto st_scale = [&](int s) { return reinterpret_cast<float*>(smem + s * o.stage + o.scale); };
  auto st_nscale = [&](int s) { return reinterpret_cast<float*>(smem + s * o.stage + o.nscale); };
  auto full = [&](int s) { return reinterpret_cast<uint64_t*>(smem + s * o.stage + o.bars); };
  auto empty = [&](int s) { return reinterpret_cast<uint64_t*>(smem + s * o.stage + o.bars) + 1; };

  pdl_launch_dependents();
  for (int v = threadIdx.x; v < Q; v += blockDim.x) {
    s_vel[v] = a.vel[kVelEx * Q + v];
    s_vel[Q + v] = a.vel[kVelEy * Q + v];
    s_vel[2 * Q + v] = a.vel[kVelW * Q + v];
    if constexpr (ST::dev) {
      s_vel[3 * Q + v] = a.vel[kVelWex * Q + v];
      s_vel[4 * Q + v] = a.vel[kVelWey * Q + v];
      s_vel[5 * Q + v] = a.vel[kVelInvW * Q + v];
    }
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      st_nbr(s)[3] = -1;         // no element yet
      mbar_init(full(s), 32);    // the producer's 32 lanes
      mbar_init(empty(s), NC);   // every thread of the group that takes the element
    }
    fence_mbar_init();
    fence_proxy_async_smem();
  }
  pdl_wait();
  __syncthreads();

  if (producer) {
    // ---- producer warp: element k = blockIdx.x + j gridDim.x into stage j % NST
    const int lane = threadIdx.x - G * NC;
    const size_t row_bytes = size_t(Q) * sizeof(S);
    int issued = 0;  // elements issued
    for (int64_t k = blockIdx.x; k < K; k += gridDim.x, ++issued) {
      const int s = issued % NST;
      if (issued >= NST) {
        // the consumers released element issued - NST from this stage
        const uint32_t ph = uint32_t((issued / NST - 1) & 1);
        bool ok = true;
        if (lane == 0) ok = mbar_wait_bounded(empty(s), ph, 2000000000ull);
        ok = __shfl_sync(kFull, ok ? 1 : 0, 0) != 0;
        if (!ok) break;  // the consumers gave up (or a release never came)
        if (lane != 0) mbar_try_wait(empty(s), ph);
      }
      int* nb = st_nbr(s);
      if (lane == 0) *reinterpret_cast<volatile int*>(nb + 3) = issued;
      for (int v = lane; v < 3; v += 32) {
        const int code = __ldg(a.nbr + k * 3 + v);
        nb[v] = code;
        if constexpr (ST::dev) st_nscale(s)[v] = code >= 0 ? a.scale_in[code >> 3] : 0.f;
      }
      if constexpr (ST::dev)
        if (lane == 0) st_scale(s)[0] = a.scale_in[k];
      uint32_t bytes = lane == 0 ? uint32_t(NP * row_bytes + kGeoStrideDev * 4) + a.extra_tx : 0u;
      for (int row = lane; row < NF && !kWide; row += 32)
        if (__ldg(a.nbr + k * 3 + row / NFP) >= 0) bytes += uint32_t(row_bytes);
      mbar_arrive_expect_tx(full(s), bytes);
      if (lane == 0) {
        bulk_load(st_f(s), fin + size_t(k) * NP * Q, uint32_t(NP * row_bytes), full(s));
        bulk_load(st_geo(s), a.geo + k * kGeoStrideDev, uint32_t(kGeoStrideDev * 4), full(s));
        // the residual goes straight to the consumers' registers; bring it into L2
        // while the ring is ahead of them
        if (read_res)
          asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a.res + size_t(k) * NP * Q),
                       "r"(uint32_t(NP * Q * 4))
                       : "memory");
      }
      for (int row = lane; row < NF && !kWide; row += 32) {
        const int fc = row / NFP, aa = row % NFP;
        const int code = __ldg(a.nbr + k * 3 + fc);
        if (code >= 0) {
          const int64_t kn = code >> 3;
          const int fn = (code >> 1) & 3;
          const int a2 = (code & 1) ? NFP - 1 - aa : aa;
          bulk_load(st_tr(s) + size_t(row) * Q, fin + (size_t(kn) * NP + face_node(fn, a2)) * Q,
                    uint32_t(row_bytes), full(s));
        }
      }
    }
    // let every copy this warp issued land before the CTA can leave: the last
    // min(issued, stages) elements' full barriers (complete long since on a
    // normal exit; after a timeout the bound is short, copies take microseconds)
    if (lane == 0) {
      for (int q = 0; q < NST && q < issued; ++q) {
        const int e = issued - 1 - q;
        mbar_wait_bounded(full(e % NST), uint32_t((e / NST) & 1), 100000000ull);
      }
    }
    return;
  }

  // ---- consumers: thread = N adjacent velocities from i on, of each element of this CTA ----
  const T rkA2 = L::both(a.rkA), rkB2 = L::both(a.rkB), zero = L::zero();
  const float ab = a.ab;
  const uint32_t sr_step = (ST::dev && a.sr_step) ? __ldg(a.sr_step) : 0u;
  const int bar_id = 1 + group;
  // one velocity per thread: its own rows stay in registers
  constexpr bool kOwnRows = N == 1;
  const T ex1 = kOwnRows ? L::load(s_vel + tid) : zero, ey1 = kOwnRows ? L::load(s_vel + Q + tid) : zero;
  const T w1 = kOwnRows ? L::load(s_vel + 2 * Q + tid) : zero;
  const T iw1 = kOwnRows && ST::dev ? L::load(s_vel + 5 * Q + tid) : zero;
  int j = group;  // element of the CTA
  for (int64_t k = blockIdx.x + int64_t(group) * gridDim.x; k < K; k += int64_t(G) * gridDim.x, j += G) {
    const int s = j % NST;
    const uint32_t ph = uint32_t((j / NST) & 1);
    // the residual columns of this element's first pass (before the wait: their
    // latency overlaps the copies and the reductions; asked for an element ahead
    // instead they measured slower, 4126 us against 3812 us for the 8-step call)
    T rold[NP];
    const size_t col0 = size_t(k) * NP * Q + N * tid;
    auto load_residual = [&](int pass) {
#pragma unroll
      for (int n = 0; n < NP; ++n)
        rold[n] = read_res && (!kWide || N * tid + pass * N * NC < Q)
                      ? L::load(a.res + col0 + size_t(n) * Q + pass * N * NC)
                      : zero;
    };
    load_residual(0);
    bool ok = true;
    if (tid < 32) {
      // Where the stage's previous element was another group's, its phase of the
      // barrier may not even be complete, and the parity alone would let this
      // group pass.  Its own number in the stage says that it is: the producer
      // writes it after that element's release.
      if (G > 1 && NST % G != 0) ok = wait_for_number(st_nbr(s) + 3, j, 2000000000ull);
      ok = ok && mbar_wait_bounded(full(s), ph, 2000000000ull);
    }
    if (consumers_sync_or(bar_id, NC, !ok)) {
      if (tid == 0 && a.err) atomicExch(a.err, 1);
      return;  // the producer waits for its copies in flight before it leaves
    }
    if (tid >= 32) mbar_try_wait(full(s), ph);
    const float* g = st_geo(s);
    const int* nb = st_nbr(s);
    float* rec = reinterpret_cast<float*>(smem + o.mom) + (group * 2 + ((j / G) & 1)) * NP * kRec;
    float* wn = reinterpret_cast<float*>(smem + o.wn) + (group * 2 + ((j / G) & 1)) * NF;
    const float sc = ST::dev ? st_scale(s)[0] : 0.f;
    const float dt = g[kGeoDt], kappa = dt * g[kGeoInvTau];

    // ---- node moments and wall numerators ----------------------------------
    if (!a.collision) {
      for (int v = tid; v < NP * kRec; v += NC) rec[v] = 0.f;
    } else if (a.red == kRedFP64) {
      element_moments<ST, AccD, QT, kThreadsOf>(a, st_f(s), sc, s_vel, kappa, rec, tid, NC);
    } else if (a.red == kRedCompFP32) {
      element_moments<ST, AccN, QT, kThreadsOf>(a, st_f(s), sc, s_vel, kappa, rec, tid, NC);
    } else {
      element_moments<ST, AccF, QT, kThreadsOf>(a, st_f(s), sc, s_vel, kappa, rec, tid, NC);
    }
    if (a.wall_any) {
      // one warp per wall face node: sum over outgoing velocities of (e.n) f^-
      const int lane = tid & 31, warp = tid >> 5;
      for (int trip = warp; trip < NF; trip += NC / 32) {
        const int fc = trip / NFP, aa = trip % NFP;
        const int code = nb[fc];
        if (!(code < 0 && __ldg(a.wall_den_inv + (-code - 1)) > 0.f)) continue;
        const float nxf = g[4 + 3 * fc], nyf = g[5 + 3 * fc];
        const S* row = st_f(s) + face_node(fc, aa) * Q;
        float acc = 0.f;
        for (int v = lane; v < Q; v += 32) {
          const float en = s_vel[v] * nxf + s_vel[Q + v] * nyf;
          const float wv = ST::dev ? s_vel[2 * Q + v] : 0.f;
          if (en > 0) acc += en * decode<ST>(row[v], wv, wv * sc);
        }
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(kFull, acc, off);
        if (lane == 0) wn[trip] = acc;
      }
    }
    consumers_sync(bar_id, NC);

    // ---- residual and update of velocities i .. i + N - 1, all nodes -----------------
#pragma unroll 1
    for (int pass = 0; pass < kPasses; ++pass) {
      const int i_own = N * tid + pass * N * NC;
      // the wide form's last pass: lanes past the last velocity take the first along and
      // store nothing
      const bool own = !kWide || i_own < Q;
      const int i = own ? i_own : 0;
      if (kWide && !__any_sync(kFull, own)) continue;
      const T ex = kOwnRows ? ex1 : L::load(s_vel + i), ey = kOwnRows ? ey1 : L::load(s_vel + Q + i);
      const T w = kOwnRows ? w1 : L::load(s_vel + 2 * Q + i);
      const T ws = ST::dev ? L::mul(w, L::both(sc)) : zero;
      if (kPasses > 1 && pass > 0) load_residual(pass);
      const S* fcol = st_f(s) + i;
      auto normal_speed = [&](int fc) {
        return L::fmat(ey, L::both(g[5 + 3 * fc]), L::mul(ex, L::both(g[4 + 3 * fc])));
      };
      // wide form: the neighbour traces straight from global memory (L2), for the faces
      // the pair enters through, all in flight before the first is used
      T tr[kWide ? NF : 1];
      if constexpr (kWide) {
#pragma unroll
        for (int fc = 0; fc < 3; ++fc) {
          const int code = nb[fc];
          const bool in = code >= 0 && L::any(L::map(normal_speed(fc), [&](float v) { return fmaf(-ab, fabsf(v), v); }));
          const S* base = fin + size_t(code >= 0 ? code >> 3 : 0) * NP * Q + i;
#pragma unroll
          for (int aa = 0; aa < NFP; ++aa)
            tr[fc * NFP + aa] = in ? L::template raw<ST>(base + size_t(trace_node(code, aa)) * Q) : zero;
        }
      }
      T fr[NP];
#pragma unroll
      for (int m = 0; m < NP; ++m) fr[m] = lane_value<L, ST>(fcol + m * Q, w, ws);
      // face fc carries flux for some velocity of this warp (warp-uniform; with
      // the upwind flux an outflow face's jump term is zero, so a face that is
      // outflow for all the warp's velocities skips its traces and lift columns)
      T flux[NF];
      bool on[3];
#pragma unroll
      for (int fc = 0; fc < 3; ++fc) {
        const float h = 0.5f * dt * g[6 + 3 * fc];
        const int code = nb[fc];
        const T c = L::map(normal_speed(fc), [&](float v) {
          const float x = h * fmaf(-ab, fabsf(v), v);
          return code < 0 && !(v < 0.f) ? 0.f : x;  // a wall: incoming velocities take its state, no other jump
        });
        on[fc] = __any_sync(kFull, L::any(c));
#pragma unroll
        for (int aa = 0; aa < NFP; ++aa) flux[fc * NFP + aa] = zero;
        if (!on[fc]) continue;
        if (code >= 0) {
          const T wsn = ST::dev ? L::mul(w, L::both(st_nscale(s)[fc])) : zero;
          const S* trow = st_tr(s) + fc * NFP * Q + i;
#pragma unroll
          for (int aa = 0; aa < NFP; ++aa) {
            T t;
            if constexpr (kWide) t = ST::dev ? L::fmat(wsn, tr[fc * NFP + aa], w) : tr[fc * NFP + aa];
            else t = lane_value<L, ST>(trow + aa * Q, w, wsn);
            flux[fc * NFP + aa] = L::mul(c, L::sub(fr[face_node(fc, aa)], t));
          }
        } else {
          const int slot = -code - 1;
          const T fb = L::load(a.wall_feq + size_t(slot) * Q + i);
          const float den_inv = __ldg(a.wall_den_inv + slot);
          const bool diffuse = den_inv > 0.f;
          const T fd = diffuse ? L::mul(L::both(den_inv), fb) : fb;
#pragma unroll
          for (int aa = 0; aa < NFP; ++aa) {
            const T fp = diffuse ? L::mul(L::both(wn[fc * NFP + aa]), fd) : fb;
            flux[fc * NFP + aa] = L::mul(c, L::sub(fr[face_node(fc, aa)], fp));
          }
        }
      }
      T le[NE], lo[at_least_1(NO)];
      eo_lift<L>(flux, on[0] || on[2], on[1], le, lo);
      const T neg_k = L::both(-kappa);
      const T ar = L::fmat(ey, L::both(g[2]), L::mul(ex, L::both(g[0])));
      const T as = L::fmat(ey, L::both(g[3]), L::mul(ex, L::both(g[1])));
      const T half_dt = L::both(0.5f * dt);
      const T na = L::mul(L::mul(half_dt, L::both(-1.f)), L::add(ar, as)), nd = L::mul(half_dt, L::sub(ar, as));
      T invw = zero;
      if constexpr (ST::dev)  // BF16 keeps the element's power-of-two scale: q = (f - w) / (w s)
        invw = L::mul(kOwnRows ? iw1 : L::load(s_vel + 5 * Q + i), L::both(1.0f / sc));
      const size_t col = col0 + size_t(pass) * N * NC;
      // update and write-back of node n from dt times its advection term
      // -(e . grad) f + LIFT (flux)
      eo_volume<L>([&](int n) { return fr[n]; }, na, nd, le, lo, [&](int n, T adv) {
        const float* mm = rec + n * kRec;
        T m0, m1, m2, m3, mx, my;
        L::record(mm, m0, m1);
        L::record(mm + 4, m2, m3);
        L::record(mm + 8, mx, my);
        // from shared memory again where the registers are short
        const T f = N == 1 && P <= 4 ? fr[n] : lane_value<L, ST>(fcol + n * Q, w, ws);
        const T eu = L::fmat(ey, my, L::mul(ex, mx));
        T feq = L::fmat(ey, m2, L::fmat(ex, m1, m0));
        feq = L::fmat(eu, L::mul(m3, eu), feq);
        if (third) {
          T m6, m7;
          L::record(mm + 12, m6, m7);
          feq = L::fmat(eu, L::fmat(m6, L::mul(eu, eu), m7), feq);
        }
        const T r = L::fmat(w, feq, L::fmat(neg_k, f, L::fmat(rkA2, rold[n], adv)));
        const T fnew = L::fmat(rkB2, r, f);
        const size_t gi = col + size_t(n) * Q;
        if (own) L::store(a.res + gi, r);
        if constexpr (ST::dev) {
          const T q = L::mul(L::sub(fnew, w), invw);
          typename L::Code code;
          if (a.sr_step) code = L::to_bf16(q, gi, sr_step, uint32_t(a.sr_stage));
          else code = L::to_bf16(q);
          if (own) *reinterpret_cast<typename L::Code*>(fout + gi) = code;
        } else {
          if (own) L::store(fout + gi, fnew);
        }
      });
    }
    // the stage's shared data are read: release it to the producer
    mbar_arrive(empty(s));
    if constexpr (ST::dev)
      if (tid == 0) a.scale_out[k] = sc;
  }
}

// The form exists for these states, velocity counts and degrees (two ring
// stages have to fit a CTA's shared memory).
template <class ST, int QT, int G, int N>
__host__ __device__ constexpr bool exists() {
  if constexpr (ST::kind != kStoreF32 && ST::kind != kStoreBF16) return false;
  else if constexpr (QT == 0) return P >= 1 && P <= 5;
  else if constexpr (QT == 1024) return P <= 3;
  else return P <= 5;
}

using Kernel = void (*)(StageArgs<float>);
struct Form {
  Kernel kernel = nullptr;
  size_t smem = 0;
  int threads = 0;
};
template <class ST, int QT, int G, int N>
Form form_as(int Q) {
  Form f;
  if constexpr (exists<ST, QT, G, N>()) {
    const Layout o = layout<ST, QT, G, N>(Q);
    if (o.end > size_t(227) * 1024) return f;
    f.kernel = &stage_kernel_ws<ST, QT, G, N>;
    f.smem = o.end;
    f.threads = threads<QT, G, N>(Q);
  }
  return f;
}
template <class ST>
Form form_of(int Qp, int groups) {
  if (Qp == 1024 && groups == 3) return form_as<ST, 1024, 3, 2>(Qp);
  if (Qp == 256 && groups == 1) return form_as<ST, 256, 1, 2>(Qp);
  if (Qp == 256 && groups == 2) {
    if constexpr (P <= 3) return form_as<ST, 256, 2, 2>(Qp);
    else return form_as<ST, 256, 1, 1>(Qp);
  }
  if (Qp >= 512 && groups == 0) return form_as<ST, 0, 1, 2>(Qp);
  return Form();
}
inline Form form(int store_kind, int Qp, int groups) {
  if (store_kind == kStoreF32) return form_of<StoreF32>(Qp, groups);
  if (store_kind == kStoreBF16) return form_of<StoreBF16>(Qp, groups);
  return Form();
}

}  // namespace ws

// ---- host-side entry points of the form ---------------------------------------
size_t ws_smem(int store_kind, int Qp, int groups) { return ws::form(store_kind, Qp, groups).smem; }
int ws_threads(int store_kind, int Qp, int groups) { return ws::form(store_kind, Qp, groups).threads; }

cudaError_t launch_ws(int store_kind, const void* args, int groups, int grid, size_t smem, cudaStream_t st) {
  const auto& a = *static_cast<const StageArgs<float>*>(args);
  const ws::Form f = ws::form(store_kind, a.Qp, groups);
  if (!f.kernel) return cudaErrorInvalidValue;
  return launch_stage_kernel(f.kernel, grid, f.threads, smem, st, a);
}

cudaError_t set_smem_ws(int store_kind, int Qp, int groups, size_t smem) {
  const ws::Form f = ws::form(store_kind, Qp, groups);
  if (!f.kernel) return cudaErrorInvalidValue;
  return cudaFuncSetAttribute(f.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
}

// Resident CTAs per SM.
int occupancy_ws(int store_kind, int Qp, int groups, size_t smem) {
  const ws::Form f = ws::form(store_kind, Qp, groups);
  int n = 0;
  if (!f.kernel || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f.kernel, f.threads, smem) != cudaSuccess)
    return 0;
  return n;
}
