// k_search_float.cu -- batched beam search of Alg. 1 on FP32 / FP16 rows with each warp's queue in
// registers, sm_103a.
//
// The queue of up to 32 QS entries is held as in the 8-bit kernel (k_search_fast.cu: entry 32 s +
// lane in q[s] of that lane), with 64-bit keys
//   key = D^2 (31 bits of a non-negative FP32) << 33 | id << 2 | decided << 1 | explored
// whose unsigned order is the (FP32 D^2, id) order.  FP32 decides every comparison that lies
// outside the relative band; the rest is Alg. 1's order by the canonical FP64 distance:
//   after the new points of a hop are merged, every two neighbours of the queue (and the last kept
//   against each dropped one) that lie within the band and are not both `decided` get their
//   squared distance to within DD_EPS (warp_sqdist_dd, ~120 FP32 instructions of the warp; one
//   lane's FP64 sum holds the SM's FP64 pipe for ~80 d cycles, which bounded the searches of
//   unit-norm data), and its FP32 rounding replaces the key's D^2.  Two decided neighbours within
//   CLOSE_STEPS FP32 steps, one of them new to its place, are compared by those values -- by id where
//   their rows are the same, in FP64 (one entry per lane) where the values lie within DD_EPS -- and
//   while they are not in that order the later one's key moves up by one FP32 step.  No key moves
//   further than CLOSE_STEPS from its rounding, so decided entries further apart than that are in the
//   FP64 order, and an entry's key stays within the band's error model (2^-20.3; an FP32 sum
//   2^-18.6).  A query that needs more, whose near-ties do not settle in FIX_ROUNDS rounds or take
//   FP64 sums in many hops, is left to the general kernel (k_search.cu).
// So the queue, and with it every hop, id and hop count, equals the FP64 definition of Alg. 1.
//
// What bounds it: the latency of a hop's dependent steps -- row loads, filter, sort, merge -- over
// ~20 warps per SM.  The general kernel keeps the queue in shared memory (33 bytes an entry and
// two copies: 2 to 4 times fewer warps) and merges by binary searches with near-tie scans in every
// hop; here a hop is one ballot, one batch of row loads (4 rows per load instruction, 8 lanes
// each), a register sort, a register merge and one neighbour comparison per slot.
// The FP32 distances are those of the general kernel bit for bit (same sums in the same order).
//
// Measured (start: the general kernel alone): 10,000 queries on 1M x 96 FP32 rows, L = 24: 2.36 -> 0.82
// ms (4.8 TB/s of rows); 100,000 on 1M x 128 FP16 rows, L = 64: 31.4 -> 13.2 ms; learned stop, 500k x
// 128 FP16, L = 192: 12.3 -> 7.6 ms; the phase-4 searches of 50k x 960 rows, L = 128: 180 -> 28 ms.
#include "launch_count.h"
#include "cng_internal.h"
#include "device_common.cuh"
#include "row_warp.cuh"
#include "search_internal.h"
#include "search_device.cuh"

namespace cng {
namespace {

constexpr uint64_t KINF = ~0ull;
constexpr int FIX_ROUNDS = 64;   // near-tie rounds of a hop before a query is left to the general kernel
constexpr int CLOSE_STEPS = 6;   // FP32 steps a key may lie above its rounding
// FP64 sums (plus three in two hops for queues of up to 64 entries, one in two for longer ones, whose
// hops take more of them) after which a query is left to the general kernel, which keeps an entry's
// FP64 distance for the query's later hops.  Only data whose distances tie to the last FP64 bits comes
// near it.  A round of moves that follows such a sum counts as MOVE_SUMS more.  2,000 queries on 20,000
// rows of two levels, d = 64, the general kernel alone / this file without the limit / with it: L = 32
// 3.6 / 2.8 / 2.8 ms, L = 64 6.1 / 5.6 / 5.7, L = 256 24.9 / 55 / 27; three levels, d = 96, L = 64 8.5 /
// 17 / 9.3, L = 128 15.3 / 44 / 16.
constexpr int FP64_SUMS = 8;
constexpr int MOVE_SUMS = 2;

CNG_DEV uint64_t fk_make(float d2, int32_t id) {
  return ((uint64_t)__float_as_uint(d2) << 33) | ((uint64_t)(uint32_t)id << 2);
}
CNG_DEV int32_t fk_id(uint64_t k) { return (int32_t)((uint32_t)(k >> 2) & 0x7fffffffu); }
CNG_DEV float fk_d2(uint64_t k) { return __uint_as_float((uint32_t)(k >> 33)); }
CNG_DEV bool fk_open(uint64_t k) { return k != KINF && !(k & 1); }  // unexplored
// Neighbours a <= b of the queue whose order FP32 does not settle.
CNG_DEV bool fk_near(uint64_t a, uint64_t b, float band) {
  return b != KINF && !(a & b & 2) && near_tie(fk_d2(a), fk_d2(b), band);
}

template <int QS>
CNG_DEV uint64_t fq_get(const uint64_t (&q)[QS], int i) {
  uint64_t v = q[0];
#pragma unroll
  for (int s = 1; s < QS; ++s)
    if ((i >> 5) == s) v = q[s];
  return __shfl_sync(FULL, v, i & 31);
}

template <int QS>
CNG_DEV int fq_first_open(const uint64_t (&q)[QS]) {
  int idx = -1;
#pragma unroll
  for (int s = 0; s < QS; ++s) {
    const unsigned bal = __ballot_sync(FULL, fk_open(q[s]));
    if (idx < 0 && bal) idx = s * 32 + __ffs(bal) - 1;
  }
  return idx;
}

// The entry after / before this lane's entry of slot s (KINF / 0 past the ends).
template <int QS>
CNG_DEV uint64_t fq_next(const uint64_t (&q)[QS], int s, int lane) {
  uint64_t nx = __shfl_down_sync(FULL, q[s], 1);
  const uint64_t first = s + 1 < QS ? __shfl_sync(FULL, q[s + 1 < QS ? s + 1 : s], 0) : KINF;
  return lane == 31 ? first : nx;
}
template <int QS>
CNG_DEV uint64_t fq_prev(const uint64_t (&q)[QS], int s, int lane) {
  uint64_t pv = __shfl_up_sync(FULL, q[s], 1);
  const uint64_t last = s > 0 ? __shfl_sync(FULL, q[s > 0 ? s - 1 : 0], 31) : 0ull;
  return lane == 0 ? last : pv;
}

// Q <- the 32 QS smallest of Q and the batch (kdesc: sorted descending across the lanes), sorted;
// returns the lane's dropped key (as in k_search_fast.cu's qmerge).
template <int QS>
CNG_DEV uint64_t fq_merge(uint64_t (&q)[QS], uint64_t kdesc, int lane) {
  const uint64_t l = q[QS - 1];
  const uint64_t drop = kdesc < l ? l : kdesc;
  q[QS - 1] = kdesc < l ? kdesc : l;
#pragma unroll
  for (int st = QS / 2; st >= 1; st >>= 1)
#pragma unroll
    for (int s = 0; s < QS; ++s)
      if (!(s & st)) {
        const uint64_t x = q[s], y = q[s + st];
        q[s] = x < y ? x : y;
        q[s + st] = x < y ? y : x;
      }
#pragma unroll
  for (int j = 16; j >= 1; j >>= 1)
#pragma unroll
    for (int s = 0; s < QS; ++s) {
      const uint64_t o = __shfl_xor_sync(FULL, q[s], j);
      q[s] = (lane & j) ? (o > q[s] ? o : q[s]) : (o < q[s] ? o : q[s]);
    }
  return drop;
}

// Per-lane flags (bit s: the entry q[s]) of the entries after / before this lane's (0 past the ends).
template <int QS>
CNG_DEV unsigned fq_next_bits(unsigned f, int lane) {
  const unsigned nx = __shfl_down_sync(FULL, f, 1), first = __shfl_sync(FULL, f, 0) >> 1;
  return lane == 31 ? first : nx;
}
template <int QS>
CNG_DEV unsigned fq_prev_bits(unsigned f, int lane) {
  const unsigned pv = __shfl_up_sync(FULL, f, 1), last = __shfl_sync(FULL, f, 31) << 1;
  return (lane == 0 ? last : pv) & ((1u << QS) - 1);
}

// Sorts a nearly sorted queue and its flags f (odd-even transposition until nothing is out of order).
template <int QS>
CNG_DEV void fq_settle(uint64_t (&q)[QS], unsigned& f, int lane) {
  for (int it = 0; it < 32 * QS; ++it) {
    bool bad = false;
#pragma unroll
    for (int s = 0; s < QS; ++s) bad |= q[s] > fq_next<QS>(q, s, lane);
    if (!__any_sync(FULL, bad)) break;
    const unsigned fo = __shfl_xor_sync(FULL, f, 1);
    unsigned take = 0;
#pragma unroll
    for (int s = 0; s < QS; ++s) {
      const uint64_t o = __shfl_xor_sync(FULL, q[s], 1);
      if ((lane & 1) ? o > q[s] : o < q[s]) {
        q[s] = o;
        take |= 1u << s;
      }
    }
    f = (f & ~take) | (fo & take);
    const unsigned fn = fq_next_bits<QS>(f, lane), fp = fq_prev_bits<QS>(f, lane);
    take = 0;
    uint64_t t[QS];
#pragma unroll
    for (int s = 0; s < QS; ++s) {
      const uint64_t nx = fq_next<QS>(q, s, lane), pv = fq_prev<QS>(q, s, lane);
      t[s] = q[s];
      if ((lane & 1) ? nx < q[s] : pv > q[s]) {
        t[s] = (lane & 1) ? nx : pv;
        take |= 1u << s;
      }
    }
#pragma unroll
    for (int s = 0; s < QS; ++s) q[s] = t[s];
    f = (f & ~take) | (((lane & 1) ? fn : fp) & take);
  }
}

// Canonical FP64 squared distances of the entries whose bit of `need` is set (bit s: this lane's k[s],
// s < N), 32 at a time, one per lane.  Returns how many times that was.
template <typename T, int N>
__device__ __noinline__ int fk_canon(const uint64_t* k, unsigned need, double* val, const float* qv, const T* X,
                                      int dpad, int d) {
  const int lane = threadIdx.x & 31;
  int total = 0;
  for (int s = 0; s < N; ++s) total += __popc(__ballot_sync(FULL, need >> s & 1));
  for (int b = 0; b < total; b += 32) {
    int32_t id = -1;
    int o = b;  // rank of slot s's first entry, seen from the batch
    for (int s = 0; s < N; ++s) {
      const unsigned m = __ballot_sync(FULL, need >> s & 1);
      const int r = lane + o;
      const bool mine = r >= 0 && r < __popc(m);
      const uint64_t e = __shfl_sync(FULL, k[s], mine ? (int)__fns(m, 0, r + 1) : 0);
      if (mine) id = fk_id(e);
      o -= __popc(m);
    }
    const double v = id >= 0 ? canon_sqdist(qv, X + (int64_t)id * dpad, d) : 0.0;
    __syncwarp();
    o = -b;
    for (int s = 0; s < N; ++s) {
      const unsigned m = __ballot_sync(FULL, need >> s & 1);
      const int r = o + __popc(m & ((1u << lane) - 1));
      const double t = __shfl_sync(FULL, v, r & 31);
      if ((need >> s & 1) && r >= 0 && r < 32) val[s] = t;
      o += __popc(m);
    }
  }
  return (total + 31) / 32;
}

// The same to within DD_EPS, entry by entry by the whole warp (FP64 only where warp_sqdist_dd gives
// none and the point is not the query itself; returns fk_canon's count).
template <typename T, int N>
__device__ __noinline__ int fk_values(const uint64_t* k, unsigned need, double* val, const float* qv, const T* X,
                                       int dpad, int d) {
  const int lane = threadIdx.x & 31;
  unsigned none = 0;
  for (int s = 0; s < N; ++s) {
    unsigned m = __ballot_sync(FULL, need >> s & 1);
    while (m) {
      const int l = __ffs(m) - 1;
      m &= m - 1;
      const T* x = X + (int64_t)fk_id(__shfl_sync(FULL, k[s], l)) * dpad;
      double v = warp_sqdist_dd(qv, x, d, lane);
      if (isnan(v) && warp_rows_equal(qv, x, d, lane)) v = 0.0;
      if (lane == l) val[s] = v;
    }
    if ((need >> s & 1) && isnan(val[s])) none |= 1u << s;
  }
  return __any_sync(FULL, none != 0) ? fk_canon<T, N>(k, none, val, qv, X, dpad, d) : 0;
}

// An entry with the FP32 rounding of its squared distance as key.
CNG_DEV uint64_t fk_decided(uint64_t k, double v) { return fk_make(__double2float_rn(v), fk_id(k)) | (k & 1) | 2; }
// Neighbours a <= b, both decided, whose roundings do not settle their order.
CNG_DEV bool fk_close(uint64_t a, uint64_t b) {
  return a != KINF && b != KINF && (a & b & 2) && (uint32_t)(b >> 33) - (uint32_t)(a >> 33) <= (uint32_t)CLOSE_STEPS;
}

// Whether a neighbour pair of the queue, or its last entry and a dropped key, is a near-tie.
template <int QS>
CNG_DEV bool fq_has_near(const uint64_t (&q)[QS], uint64_t drop, float band, int lane) {
  bool any = false;
#pragma unroll
  for (int s = 0; s < QS; ++s) {
    const uint64_t nx = fq_next<QS>(q, s, lane);  // all lanes take part in its shuffles
    any |= q[s] != KINF && fk_near(q[s], nx, band);
  }
  const uint64_t last = __shfl_sync(FULL, q[QS - 1], 31);
  any |= last != KINF && fk_near(last, drop, band);
  return __any_sync(FULL, any);
}

// What fq_fix works on: the queue's keys of a lane and its dropped key; of a query the FP64 sums taken
// (by up to 32 lanes at once) and whether a key moved; of the warp's queries the entries decided.  In
// local memory: the search itself is short of registers.
template <int QS>
struct FixState {
  uint64_t q[QS + 1];
  int sums, moved;
  unsigned long long decided;
};

// Which of the pairs `pair` (bit s: the entry k[s] of this lane and the queue's next one, bit QS: the
// queue's last entry and this lane's dropped key k[QS]) are not in the FP64 order (D, id); FAR is set
// where the first one's key may not move further.  *sums counts the FP64 sums.
constexpr unsigned FAR = 1u << 31;
template <typename T, int QS>
__device__ __noinline__ unsigned fq_wrong(const uint64_t* k, unsigned pair, int* sums, const float* qv, const T* X,
                                          int dpad, int d) {
  constexpr int N = QS + 1;
  constexpr unsigned QBITS = (1u << QS) - 1, DBIT = 1u << QS, LAST = 1u << (QS - 1);
  const int lane = threadIdx.x & 31;
  double val[N], cv[N];
  for (int s = 0; s < N; ++s) val[s] = cv[s] = 0.0;
  // the entry (or its value) after slot s of this lane; slot QS: the dropped one, after the queue's last
  auto first_of = [&](const auto* v, int s) {
    const auto l = __shfl_sync(FULL, v[QS - 1], 31);
    return s < QS ? v[s] : l;
  };
  auto second_of = [&](const auto* v, int s) {
    const auto nx = __shfl_down_sync(FULL, v[s], 1);
    const auto f = __shfl_sync(FULL, v[s + 1 < QS ? s + 1 : s], 0);
    return s == QS ? v[QS] : (lane == 31 ? f : nx);
  };
  auto members = [&](unsigned p) {
    unsigned need = p | fq_prev_bits<QS>(p & QBITS, lane);
    if (__any_sync(FULL, p & DBIT) && lane == 31) need |= LAST;
    return need;
  };
  *sums += fk_values<T, N>(k, members(pair), val, qv, X, dpad, d);
  // pairs that those values leave open: the same row twice, or the canonical distances
  unsigned open = 0, same = 0;
  for (int s = 0; s < N; ++s) {
    const uint64_t ka = first_of(k, s), kb = second_of(k, s);
    const double va = first_of(val, s), vb = second_of(val, s);
    const bool op = (pair >> s & 1) && dd_open(va, vb);
    if (op) open |= 1u << s;
    unsigned m = __ballot_sync(FULL, op && va == vb);
    while (m) {
      const int l = __ffs(m) - 1;
      m &= m - 1;
      const int32_t ia = fk_id(__shfl_sync(FULL, ka, l)), ib = fk_id(__shfl_sync(FULL, kb, l));
      if (warp_rows_equal(X + (int64_t)ia * dpad, X + (int64_t)ib * dpad, d, lane) && lane == l) same |= 1u << s;
    }
  }
  const unsigned canon = open & ~same;
  if (__any_sync(FULL, canon != 0)) {
    const unsigned need = members(canon);
    *sums += fk_canon<T, N>(k, need, cv, qv, X, dpad, d);
    for (int s = 0; s < N; ++s)
      if (need >> s & 1) cv[s] = __dsqrt_rn(cv[s]);
  }
  unsigned wrong = 0;
  for (int s = 0; s < N; ++s) {
    const uint64_t ka = first_of(k, s), kb = second_of(k, s);
    const double va = first_of(val, s), vb = second_of(val, s);
    const double ca = first_of(cv, s), cb = second_of(cv, s);
    if (pair >> s & 1) {
      const bool idless = fk_id(kb) < fk_id(ka);
      const bool w = (same >> s & 1)    ? idless
                     : (canon >> s & 1) ? cb < ca || (cb == ca && idless)
                                        : vb < va;
      if (w) wrong |= 1u << s;
      if (w && s < QS && (uint32_t)(ka >> 33) + 1 - __float_as_uint(__double2float_rn(va)) > (uint32_t)CLOSE_STEPS)
        wrong |= FAR;
    }
  }
  return wrong;
}

// Settles the near-ties of the queue and of its end against all dropped keys.  Returns false if the
// query has to be left to the general kernel.  A call of its own, with the queue through local memory:
// it is rare, and inlined it left the warp in pieces for the rest of the query (20 of 32 lanes to an
// instruction and twice the instructions on average; 1M x 96, L = 24: 2.1 against 1.0 ms).
// Only pairs with an entry decided or moved in this call are compared: the others' order was settled
// when they were.
template <typename T, int QS>
__device__ __noinline__ bool fq_fix(FixState<QS>* fs, const float* qv, const T* X, int dpad, int d, float band,
                                    int hops) {
  constexpr int N = QS + 1;  // the queue's entries of a lane and its dropped one
  constexpr unsigned QBITS = (1u << QS) - 1, DBIT = 1u << QS, LAST = 1u << (QS - 1);
  constexpr uint64_t STEP = 1ull << 33;
  const int lane = threadIdx.x & 31;
  uint64_t q[QS], drop = fs->q[QS];
  unsigned fresh = 0;  // entries decided, moved or brought in by this call
  bool settled = false;
#pragma unroll
  for (int s = 0; s < QS; ++s) q[s] = fs->q[s];
  auto store = [&]() {
#pragma unroll
    for (int s = 0; s < QS; ++s) fs->q[s] = q[s];
    fs->q[QS] = drop;
  };
  for (int it = 0; it < FIX_ROUNDS; ++it) {
    // neighbours within the band, both to be decided; within CLOSE_STEPS, to be compared
    unsigned near = 0, pair = 0, undec = drop & 2 ? 0u : DBIT;
    const unsigned nfresh = fresh | fq_next_bits<QS>(fresh, lane);
#pragma unroll
    for (int s = 0; s < QS; ++s) {
      const uint64_t nx = fq_next<QS>(q, s, lane);
      if (q[s] != KINF && fk_near(q[s], nx, band)) near |= 1u << s;
      if ((nfresh >> s & 1) && fk_close(q[s], nx)) pair |= 1u << s;
      if (!(q[s] & 2)) undec |= 1u << s;
    }
    near |= fq_prev_bits<QS>(near, lane);
    // the last kept key against every dropped one: while undecided, any of those within the band may
    // come before it
    const uint64_t last = __shfl_sync(FULL, q[QS - 1], 31);
    if (last != KINF && drop != KINF && (drop < last || fk_near(last, drop, band))) near |= DBIT;
    if (fk_close(last, drop)) pair |= DBIT;
    if (__any_sync(FULL, near & DBIT) && lane == 31) near |= LAST;
    if (__any_sync(FULL, near != 0)) {
      const unsigned need = near & undec;
      fs->decided += __reduce_add_sync(FULL, (unsigned)__popc(need & QBITS));
      double val[N];
      store();
      fs->sums += fk_values<T, N>(fs->q, need, val, qv, X, dpad, d);
#pragma unroll
      for (int s = 0; s < QS; ++s)
        if (need >> s & 1) q[s] = fk_decided(q[s], val[s]);
      if (need & DBIT) drop = fk_decided(drop, val[QS]);
      fresh |= need & QBITS;
      fq_settle<QS>(q, fresh, lane);
      // dropped keys that came out below the last kept one change places with it: each enters at most
      // once, as the last key only falls
      for (;;) {
        const uint64_t lk = __shfl_sync(FULL, q[QS - 1], 31);
        if (lk == KINF || !__any_sync(FULL, drop < lk)) break;
        uint64_t in = drop;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const uint64_t y = __shfl_xor_sync(FULL, in, o);
          in = y < in ? y : in;
        }
        if (drop == in) drop = lk;
        if (lane == 31) {
          q[QS - 1] = in;
          fresh |= LAST;
        }
        fq_settle<QS>(q, fresh, lane);
      }
      continue;
    }
    if (!__any_sync(FULL, pair != 0)) {
      settled = true;
      break;
    }
    store();
    const int sums = fs->sums;
    const unsigned wrong = fq_wrong<T, QS>(fs->q, pair, &fs->sums, qv, X, dpad, d);
    if (__any_sync(FULL, wrong & FAR)) break;
    if (__any_sync(FULL, wrong & QBITS)) {
#pragma unroll
      for (int s = 0; s < QS; ++s)
        if (wrong >> s & 1) q[s] += STEP;
      fresh |= wrong & QBITS;
      fs->moved = 1;
      if (fs->sums != sums) fs->sums += MOVE_SUMS;
    } else if (__any_sync(FULL, wrong & DBIT)) {
      // a dropped point belongs in the queue, the last one out of it for good
      uint64_t in = wrong & DBIT ? drop : KINF;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const uint64_t y = __shfl_xor_sync(FULL, in, o);
        in = y < in ? y : in;
      }
      if (drop == in) drop = KINF;
      if (lane == 31) {
        q[QS - 1] = in;
        fresh |= LAST;
      }
    } else {
      settled = true;
      break;
    }
    fq_settle<QS>(q, fresh, lane);
  }
  store();
  return settled && fs->sums <= FP64_SUMS + (QS <= 2 ? hops + hops / 2 : hops / 2);
}

// The first `cnt` entries' keys without their moves.
template <typename T, int QS>
__device__ __noinline__ void fq_round(FixState<QS>* fs, int cnt, const float* qv, const T* X, int dpad, int d) {
  double val[QS + 1];
  unsigned need = 0;
  for (int s = 0; s < QS; ++s)
    if (s * 32 + (int)(threadIdx.x & 31) < cnt && (fs->q[s] & 2)) need |= 1u << s;
  fk_values<T, QS + 1>(fs->q, need, val, qv, X, dpad, d);
  for (int s = 0; s < QS; ++s)
    if (need >> s & 1) fs->q[s] = fk_decided(fs->q[s], val[s]);
}

// FP32 squared distances of the query to up to 32 rows (row b named by lane b's v, present when
// b < nb), returned in lane b: 8 lanes read a row, a warp load covers 4 rows, 4 loads' rows are in
// flight together; the 8 partial sums of a row meet in a transposed butterfly, in the order of
// part_sqdist<8> and group_reduce<8>.
template <typename T>
CNG_DEV float batch_sqdist(const float* qv, const T* X, int dpad, int32_t v, int nb, int lane) {
  constexpr int NR = 4;
  const int grp = lane / 8, g = lane % 8;
  float p[8];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float t[NR] = {0.f, 0.f, 0.f, 0.f};
    if (16 * h < nb) {
      const T* y[NR];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const int b = (NR * h + r) * 4 + grp;
        const int32_t vb = __shfl_sync(FULL, v, b < nb ? b : 0);  // past the batch: row 0 again
        y[r] = X + (int64_t)vb * dpad;
      }
      part_rows<NR>(qv, y, dpad, g, t);
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) p[NR * h + r] = t[r];
  }
#pragma unroll
  for (int s = 4; s >= 1; s >>= 1) {
    const bool up = g & s;
#pragma unroll
    for (int i = 0; i < s; ++i) {
      const float rv = __shfl_xor_sync(FULL, up ? p[i] : p[i + s], s);
      p[i] = (up ? p[i + s] : p[i]) + rv;
    }
  }
  return __shfl_sync(FULL, p[0], (lane % 4) * 8 + lane / 4);
}

// The FP32 distance of a queue entry (its row again when the key holds the canonical rounding, so
// that the stop features do not depend on which entries were decided).
template <typename T>
__device__ __noinline__ float row_sqdist(const float* qv, const T* y, int dpad) {
  return group_reduce<8>(part_sqdist<8>(qv, y, dpad, threadIdx.x % 8));
}
template <typename T>
CNG_DEV float entry_dist(uint64_t k, const float* qv, const T* X, int dpad) {
  float d2 = fk_d2(k);
  if (k & 2) d2 = row_sqdist(qv, X + (int64_t)fk_id(k) * dpad, dpad);  // k: the same in every lane
  return sqrtf(d2);
}

// LEARN: the variant that records stop features and runs the stop model.
template <typename T, int QS, bool LEARN>
__global__ void __launch_bounds__(256, 2) search_float_kernel(SearchArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char* base = smem + (size_t)warp * a.warp_smem_fast;
  float* qv = reinterpret_cast<float*>(base);                     // query
  int32_t* Nv = reinterpret_cast<int32_t*>(base + a.dpad * 4);    // new points of a hop
  float* hist = reinterpret_cast<float*>(Nv + SQ_ROWSLOTS * 32);  // Dk after the last 64 hops
  int32_t* H = reinterpret_cast<int32_t*>(hist + 64);             // visited filter
  StopSmem ms;
  if (LEARN && a.model) {
    unsigned char* mb = smem + (size_t)(blockDim.x >> 5) * a.warp_smem_fast;
    const int4* src = reinterpret_cast<const int4*>(a.model);
    int4* dst = reinterpret_cast<int4*>(mb);
    for (int i = threadIdx.x; i < STOP_BLOCK_BYTES / 16; i += blockDim.x) dst[i] = src[i];
    ms = stop_smem(mb);
    __syncthreads();
  }
  const int hmask = a.hash_slots - 1, L = a.L, dpad = a.dpad;
  const T* X = reinterpret_cast<const T*>(a.X);
  unsigned long long t_ndc = 0, t_hops = 0, t_stop = 0;
  FixState<QS> fs;
  fs.decided = 0;

  // each warp takes query (its index) first, then queries nw + (queue head) as it finishes them
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  auto next_item = [&]() -> int64_t {
    int x = 0;
    if (lane == 0) x = atomicAdd(a.counter, 1);
    return nw + __shfl_sync(FULL, x, 0);
  };
  for (int64_t it = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;; it = next_item()) {
    if (it >= a.nq) break;
    const int qi = (int)it;
    // integer queries on integer data: the FP32 keys are exact, ties order by id
    const bool qexact = a.exact && (a.qids != nullptr || (a.qflag && a.qflag[qi] == 0));
    if (a.qids) {
      load_row(qv, X + (int64_t)a.qids[qi] * dpad, dpad, lane, 32);
    } else {
      const float* qg = a.Q + (int64_t)qi * a.d;
      for (int c = lane; c < dpad; c += 32) qv[c] = c < a.d ? qg[c] : 0.f;
    }
    for (int c = lane; c < a.hash_slots; c += 32) H[c] = -1;
    __syncwarp();
    // entry point
    const float d0 = batch_sqdist<T>(qv, X, dpad, a.entry, 1, lane);
    uint64_t q[QS];
#pragma unroll
    for (int s = 0; s < QS; ++s) q[s] = KINF;
    if (lane == 0) {
      q[0] = fk_make(d0, a.entry);
      H[hash32((uint32_t)a.entry) & hmask] = a.entry;
    }
    int len = 1, ndc = 1, hops = 0, flags = 0, tlc = 0;
    const float D0 = sqrtf(__shfl_sync(FULL, d0, 0));
    if (lane == 0) hist[0] = D0;
    __syncwarp();
    // every point is explored at most once, so n hops bound a correct search
    const int hop_cap = a.max_hops > 0 ? a.max_hops : (int)min(a.n, (int64_t)0x3fffffff);
    int32_t pf_u = -1;  // predicted next hop vertex and its out-list
    int32_t pf[SQ_ROWSLOTS];
    bool left = false;  // to the general kernel
    fs.sums = fs.moved = 0;
    for (;;) {
      __syncwarp();
      const int idx = fq_first_open<QS>(q);
      if (idx < 0) break;
      if (hops >= hop_cap) {
        flags |= 2;
        if (a.max_hops == 0 && lane == 0) atomicOr(a.status, ST_BOUNDS);
        break;
      }
      const uint64_t ku = fq_get<QS>(q, idx);
#pragma unroll
      for (int s = 0; s < QS; ++s)
        if (s == (idx >> 5) && lane == (idx & 31)) q[s] |= 1;
      const int32_t u = fk_id(ku);
      ++hops;
      // out-list of u (rows hold -1 past the degree)
      int32_t row[SQ_ROWSLOTS];
      const bool hit = u == pf_u;
#pragma unroll
      for (int r = 0; r < SQ_ROWSLOTS; ++r) {
        const int j = r * 32 + lane;
        row[r] = hit ? pf[r] : (j < a.R ? a.adj[(int64_t)u * a.R + j] : -1);
      }
      // visited filter -> Nv[0 .. nb); bit 31 marks points whose filter slots were full
      int nb = 0;
#pragma unroll
      for (int r = 0; r < SQ_ROWSLOTS; ++r) {
        if (r * 32 >= a.R) break;
        const int32_t v = row[r];
        const int st = v >= 0 ? visit3(H, hmask, v) : 0;
        const unsigned bal = __ballot_sync(FULL, st != 0);
        if (st) Nv[nb + __popc(bal & ((1u << lane) - 1))] = st == 2 ? (int32_t)((uint32_t)v | 0x80000000u) : v;
        nb += __popc(bal);
      }
      __syncwarp();
      ndc += nb;
      bool chg = false;                           // the first min(k, |Q|) ids changed
      uint64_t kb0 = KINF, kb1 = KINF, kb2 = KINF;  // this hop's sorted batches (stop features)
      // (one copy of the body: unrolled, a third of the stalls were instruction fetches)
#pragma unroll 1
      for (int ci = 0; ci * 32 < nb; ++ci) {
        __syncwarp();
        const int nbc = min(32, nb - ci * 32);
        const bool has = lane < nbc;
        // read by every lane (past the batch: a stale word nobody uses): with a select on `has`
        // here the compiler ran the row sums once for the lanes with a point and once for the rest
        const int32_t raw = Nv[ci * 32 + lane];
        const int32_t v = raw & 0x7fffffff;
        const float d2 = batch_sqdist<T>(qv, X, dpad, v, nbc, lane);
        bool keep = has;
        const bool unsure = has && raw < 0;
        unsigned ub = __ballot_sync(FULL, unsure);
        if (ub) {  // possibly seen: drop if in Q (or twice in the batch)
          const unsigned same = __match_any_sync(FULL, unsure ? v : -1 - lane);
          if (unsure && (same & ((1u << lane) - 1))) keep = false;
          while (ub) {
            const int l = __ffs(ub) - 1;
            ub &= ub - 1;
            const int32_t vl = __shfl_sync(FULL, v, l);
            bool in = false;
#pragma unroll
            for (int s = 0; s < QS; ++s) in |= q[s] != KINF && fk_id(q[s]) == vl;
            if (__any_sync(FULL, in) && lane == l) keep = false;
          }
        }
        const uint64_t kb = warp_sort32(keep ? fk_make(d2, v) : KINF, lane);
        if constexpr (LEARN) {
          if (ci == 0) kb0 = kb;
          else if (ci == 1) kb1 = kb;
          else kb2 = kb;
        }
        if (ci == 0) {  // predict the next hop vertex and start loading its out-list
          const int nidx = fq_first_open<QS>(q);
          uint64_t kn = KINF;
          if (nidx >= 0) kn = fq_get<QS>(q, nidx);
          const uint64_t k0 = __shfl_sync(FULL, kb, 0);
          if (k0 < kn) kn = k0;
          pf_u = kn == KINF ? -1 : fk_id(kn);
          if (pf_u >= 0) {
#pragma unroll
            for (int r = 0; r < SQ_ROWSLOTS; ++r) {
              const int j = r * 32 + lane;
              pf[r] = j < a.R ? a.adj[(int64_t)pf_u * a.R + j] : -1;
            }
          }
        }
        const int nv = __popc(__ballot_sync(FULL, kb != KINF));
        if (nv == 0) continue;
        const int old_len = len;
        const int32_t old_kth = LEARN && old_len >= a.k ? fk_id(fq_get<QS>(q, a.k - 1)) : -1;
        const uint64_t drop = fq_merge<QS>(q, __shfl_sync(FULL, kb, 31 - lane), lane);
        if (!qexact && fq_has_near<QS>(q, drop, a.band, lane)) {
#pragma unroll
          for (int s = 0; s < QS; ++s) fs.q[s] = q[s];
          fs.q[QS] = drop;
          left = !fq_fix<T, QS>(&fs, qv, X, dpad, a.d, a.band, hops);
#pragma unroll
          for (int s = 0; s < QS; ++s) q[s] = fs.q[s];
          flags |= 1;
          __syncwarp();
          if (left) break;
        }
        __syncwarp();
        len = min(len + nv, L);
#pragma unroll
        for (int s = 0; s < QS; ++s)
          if (s * 32 + lane >= L) q[s] = KINF;
        if constexpr (LEARN) {
          // a new point lands in the first k: when |Q| < k its smallest does; otherwise the old
          // k-th entry moves down
          if (old_len < a.k) chg = true;
          else chg |= fk_id(fq_get<QS>(q, a.k - 1)) != old_kth;
        }
      }
      if (left) break;
      // ---- search state after this hop (learned early stop) ----
      if constexpr (LEARN) {
        const int kk = min(a.k, len);
        const float Dk = entry_dist<T>(fq_get<QS>(q, kk - 1), qv, X, dpad);
        if (chg) tlc = hops;
        const bool want_trace = a.trace_feats && hops <= a.max_trace;
        const bool want_check =
            a.model && (hops % a.check_every) == 0 && hops - tlc >= a.min_stable;
        float f = 0.f;
        if (want_trace || want_check) {
          // points of this hop still in Q: those not beyond its last entry (by id where the
          // two lie within the band)
          const uint64_t last = fq_get<QS>(q, len - 1);
          int ins = 0;
#pragma unroll
          for (int ci = 0; ci < SQ_ROWSLOTS; ++ci) {
            const uint64_t kb = ci == 0 ? kb0 : ci == 1 ? kb1 : kb2;
            const bool close = kb != KINF && near_tie(fk_d2(kb), fk_d2(last), a.band);
            ins += __popc(__ballot_sync(FULL, kb != KINF && !close && kb < last));
            unsigned cb = __ballot_sync(FULL, close);
            while (cb) {
              const int l = __ffs(cb) - 1;
              cb &= cb - 1;
              const int32_t vl = fk_id(__shfl_sync(FULL, kb, l));
              bool in = false;
#pragma unroll
              for (int s = 0; s < QS; ++s) in |= q[s] != KINF && fk_id(q[s]) == vl;
              ins += __any_sync(FULL, in) ? 1 : 0;
            }
          }
          int U = 0;
#pragma unroll
          for (int s = 0; s < QS; ++s) U += __popc(__ballot_sync(FULL, fk_open(q[s])));
          const float D1 = entry_dist<T>(fq_get<QS>(q, 0), qv, X, dpad);
          const float DL = entry_dist<T>(last, qv, X, dpad);
          const float Du = entry_dist<T>(ku, qv, X, dpad);
          f = stop_feature(lane, D0, D1, Dk, DL, Du, hist, hops, tlc, U, len, ins, a.L, a.R);
          if (want_trace && lane < 16)
            a.trace_feats[((int64_t)qi * a.max_trace + (hops - 1)) * 16 + lane] = f;
        }
        __syncwarp();
        if (lane == 0) hist[hops & 63] = Dk;
        __syncwarp();
        if (want_check && mlp_logit(ms, f, lane) >= a.zthr) {
          flags |= 4;
          ++t_stop;
          break;
        }
      }
    }
    if (left) {
      if (lane == 0) a.defer[atomicAdd(a.counter + 1, 1)] = qi;
      __syncwarp();
      continue;
    }
    // results; keys that moved give way to their roundings
    if (__any_sync(FULL, fs.moved)) {
#pragma unroll
      for (int s = 0; s < QS; ++s) fs.q[s] = q[s];
      fq_round<T, QS>(&fs, min(a.k, len), qv, X, dpad, a.d);
#pragma unroll
      for (int s = 0; s < QS; ++s) q[s] = fs.q[s];
    }
#pragma unroll
    for (int s = 0; s < QS; ++s) {
      const int t = s * 32 + lane;
      if (t < a.k) {
        const bool ok = t < len;
        a.ids[(int64_t)qi * a.k + t] = ok ? fk_id(q[s]) : -1;
        a.dists[(int64_t)qi * a.k + t] = ok ? sqrtf(fk_d2(q[s])) : INFINITY;
      }
    }
    if (lane == 0) {
      if (a.ndc) a.ndc[qi] = ndc;
      if (a.hops) a.hops[qi] = hops;
      if (a.flags) a.flags[qi] = flags;
      if (a.tlc) a.tlc[qi] = tlc;
    }
    t_ndc += ndc;
    t_hops += hops;
    __syncwarp();
  }
  if (lane == 0) {
    atomicAdd(&a.tot[0], t_ndc);
    atomicAdd(&a.tot[1], t_hops);
    if (fs.decided) atomicAdd(&a.tot[2], fs.decided);
    if (t_stop) atomicAdd(&a.tot[3], t_stop);
  }
}

// One kernel per (row type, queue slots, learning): f(kernel).
template <typename T, bool LEARN, typename F>
auto with_kernel(int qs, F&& f) {
  switch (qs) {
    case 1: return f(search_float_kernel<T, 1, LEARN>);
    case 2: return f(search_float_kernel<T, 2, LEARN>);
    case 4: return f(search_float_kernel<T, 4, LEARN>);
    default: return f(search_float_kernel<T, 8, LEARN>);
  }
}
template <typename F>
auto with_kernel(int dtype, int qs, bool learn, F&& f) {
  if (dtype == CNG_F32) return learn ? with_kernel<float, true>(qs, f) : with_kernel<float, false>(qs, f);
  return learn ? with_kernel<__half, true>(qs, f) : with_kernel<__half, false>(qs, f);
}

}  // namespace

size_t search_float_warp_smem(int dpad, int hash_slots) {
  return (size_t)dpad * 4 + SQ_ROWSLOTS * 32 * 4 + 64 * 4 + (size_t)hash_slots * 4;
}

cudaError_t launch_search_float(const SearchArgs& a, int qs, int wpb, int grid, cudaStream_t s) {
  const size_t sh = (size_t)wpb * a.warp_smem_fast + (a.model ? STOP_BLOCK_BYTES : 0);
  count_launch();
  return with_kernel(a.dtype, qs, a.model || a.trace_feats, [&](auto k) {
    k<<<grid, wpb * 32, sh, s>>>(a);
    return cudaGetLastError();
  });
}

int search_float_blocks_per_sm(int dtype, int qs, bool learn, int wpb, size_t smem) {
  return with_kernel(dtype, qs, learn, [&](auto k) {
    int nb = 0;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, wpb * 32, smem);
    return nb;
  });
}

}  // namespace cng
