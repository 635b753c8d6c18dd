// Tiles of the FMA stage kernel by rule: host code, functions of the sizes and the device's
// SM count only.
#pragma once
#include <algorithm>
#include <cstdint>

#include "store_kind.h"

namespace fedbm {

struct TileShape {
  int p = 0, store = kStoreF32, Qp = 0;
  int64_t K = 0;  // elements of the group
  int nsm = 0;    // SMs of the device
};

// The FMA kernel's tile where the caller leaves it open: elements and threads per
// CTA by velocity count, degree, state and the group's element count K.  FP32
// arithmetic takes two velocities per thread, FP64 one.
//
// Where the elements do not fill the SMs several times over (K below 16 per SM;
// the figures are of the 152 SMs of a GB300), small tiles spread them (about two CTAs
// per SM) and get more threads than items, which the moment reduction uses; one tile per
// SM with idle SMs beside it was the rule before.  Above that, 16 velocities run best in CTAs of one warp (no barrier
// ever waits for another warp), with two items per thread at low degree once there
// are enough of them.  Stage times on the GB300, us, this rule against 8 (degree <= 2:
// 16) elements and one thread per item: FP32, 16 velocities, degree 1, 3, 5: K = 128
// 5.6, 6.6, 8.2 against 6.3, 8.2, 11.9; K = 2,048 5.8, 7.0, 9.4 against 6.4, 8.2, 11.5;
// K = 51,200 15.7, 38.5, 80.7 against 18.2, 39.6, 82.6; BF16 degree 1, 2, K = 204,800
// 58.9, 96.3 against 93.9, 126.0; 36 velocities, degree 2, 4: K = 512 6.6, 8.4 against
// 7.4, 11.1; K = 18,432 degree 2 23.5 against 27.5; FP64, 16 velocities, degree 3: K =
// 128, 512, 2,048 20.9, 23.0, 39.0 against 28.7, 28.7, 42.7; D2Q1089 at degree 4, K =
// 800, 256 threads instead of 128: FP32 88.6 against 102.4, BF16 108.9 against 146.7 (at
// degree 1, 1,024 velocities, FP16, 20M values: 169 against 123, so not there).
inline void auto_tile(const TileShape& g, int* epc, int* tpb) {
  const bool f64 = g.store == kStoreF64;
  const int64_t K = g.K, sms = g.nsm;
  const bool few = K < 16 * sms;
  const int spread = int(std::min<int64_t>(4, (K + 2 * sms - 1) / (2 * sms)));  // elements per CTA, two CTAs per SM
  if (g.Qp == 16 && f64) {
    *epc = !few ? 8 : K <= 2 * sms ? 1 : 2;
    *tpb = !few || K <= 4 * sms ? 128 : K <= 8 * sms ? 64 : 32;
  } else if (g.Qp == 16) {
    *epc = few ? spread : K < 32768 ? 4 : g.p <= 3 ? 8 : 4;
    if (K >= 32768 && g.p == 1 && g.store >= kStoreBF16) *epc = 16;
    *tpb = few ? 32 * spread : 32;
  } else if (g.Qp < 128 && !f64) {
    *epc = std::max(1, 128 / g.Qp);
    if (few) *epc = std::min(*epc, spread);
    *tpb = few ? std::min(128, 64 * *epc) : g.p <= 2 && K >= 64 * sms ? 32 : 64;
  } else {
    *epc = std::max(1, 128 / g.Qp);
    const int items = *epc * g.Qp / (f64 ? 1 : 2);
    const bool wide = !f64 && items >= 512 && (g.p >= 3 || (g.p == 2 && items > 512));
    *tpb = wide ? 256 : std::min(128, std::max(32, (items + 31) / 32 * 32));
  }
}

// Velocities per thread of the FMA kernel's update (FP32 arithmetic) on a tile of epc
// elements and tpb threads: two, the faster where the tile has a pair for every thread, as
// the automatic tiles of enough elements have; one on a tile that a caller gives a thread
// for every value, or a warp without a pair, and that has neighbours to share its SM with
// (from 16 elements per SM up, or tiles of one element where they are more than two per
// SM).  There idle threads would hold registers that keep other CTAs off the SM: one step of
// 20M values, us, with one kernel of one velocity per thread (before), two, one: 256
// velocities, 256 threads, FP32 degree 3, 4, 5 468, 450, 460; 532, 491, 769; 406, 377, 362;
// 16 velocities, 8 elements on 128 threads, BF16 degree 4, 5 793, 753; 681, 822; 506, 526;
// 36 velocities, 4 elements on 128 threads, degree 3 FP32, FP16 572, 803; 708, 915; 538,
// 797.  Below those counts two was as fast or faster (36 velocities, 264 elements, 4 on 128
// threads, degree 5 FP32 88; 53; 59).
inline int stage_lanes(const TileShape& g, int epc, int tpb) {
  const int values = epc * g.Qp, pairs = values / 2;
  const bool idle = tpb >= values || tpb > (pairs + 31) / 32 * 32;
  const bool shared = g.K >= 16 * g.nsm || (epc == 1 && g.K > 2 * g.nsm);
  return g.store != kStoreF64 && idle && shared ? 1 : 2;
}

}  // namespace fedbm
