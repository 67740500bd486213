// k_screen_res.cu -- tensor-core candidate screen (K1) for rows of up to 250 coordinates: the row
// block's operands stay in TMEM, the columns stream through shared memory as prepared tile images,
// and a per-row list keeps what may belong to the row's Lp nearest columns.  Screened score of
// column y for row x:  s(x, y) = ||y_b||^2 - 2 <x_b, y_b>  (x_b, y_b: the 16-bit operands), which
// differs from ||x_b - y_b||^2 by the row constant ||x_b||^2; the rerank recomputes the survivors
// and certifies the list.
//
// Operands.  Each operand row has kt = d + 6 elements rounded up to 16: the d coordinates, then
// six norm pieces.  A column holds p_0..p_5 with sum c_i p_i = ||y_b||^2 / 2 to max(2^-35 of it,
// 2^-25) in FP16 (operands are scaled so that the largest coordinate exceeds 4096 unless they are
// integers, and the certification counts the absolute part) and to 2^-48 of it in BF16, a row holds
// the constants -c_i, so the accumulator is a = <x_b, y_b> - ||y_b||^2 / 2 = -s / 2 and the epilogue
// only compares it with the row's threshold (an FMA and a shared-memory norm load per score in the
// epilogue's fast path cost more than the extra 16 K elements of the MMA).  Integer
// operands with ||x||^2 < 2^23 and distances D^2 < 2^24 (d span^2 < 2^24, span the range of the
// coordinates) stay exact: pieces, products and sums are multiples of 1/2, a partial inner product is
// below 2^23 in magnitude, and the accumulator is (||x||^2 - D^2) / 2, between -2^23 and 2^22.
//
// Column order.  Columns are swept in a sampled order: a pseudo-random 1/64 of them first, then up
// to 1/16, 1/4 and all (each part in locality order).  After a part that holds the fraction f of
// the columns the row's threshold becomes its r(f)-th smallest score so far, r(f) chosen so that
// fewer than r(f) of the row's true Lp nearest columns lie in such a sample except with
// probability 1e-9; so the threshold stays above the row's Lp-th smallest score, and the last
// part (3/4 of the sweep) appends only ~1.3 Lp columns under one fixed threshold.  A row whose
// list comes out short fails the certification like any other and is rescanned exactly.
//
// CTA organisation (one CTA per SM, persistent over 256-row blocks):
//   warp 8      producer: column tiles (BN x kt, one contiguous bulk copy each) into an nst-stage
//               ring
//   warps 9-12  MMA issuers, one per accumulator (two M=128 halves x two buffers of N=BN; warp 9
//               also owns the 512 TMEM columns): A from TMEM, B from shared memory
//   warps 0-7   epilogue: warp w owns rows 32 (w % 4) .. +31 of accumulator w / 4, one row per
//               lane; it writes its rows' A operands to TMEM, then per tile reads its BN columns
//               into registers, hands the buffer back at once, takes the maxima of the tile's
//               16-column chunks and appends only where a row beats its threshold
// A in TMEM: it leaves shared memory's bandwidth and 72 KB of it to the column tiles.  One issuer
// per accumulator: after its MMAs an issuer spends ~350 cycles in commits and barrier waits in
// which the tensor pipe, which queues only a few MMAs, would idle (one issuer for all: 1,680
// cycles per 256 x 80 tile; two: 1,260; four: 840, where the 18 MMAs take 720 at the pipe's nominal
// 8,192 operations a cycle).
//
// Bound: without hits the tensor pipe (1,900 TFLOP/s of 2 m n d at d = 128); the appends add ~40%.
// 1M x 128, L' = 160, self: 202 ms, 1,265 TFLOP/s of 2 n^2 d (0.74 of the measured sustained bf16
// rate), against 402 ms for the kernel before (rows in shared memory, one issuer, thresholds that
// fall during the sweep); 1M x 96, L' = 192: 431 -> 189 ms.
// Every wait is bounded; on expiry the kernel records ST_TIMEOUT, drains its own copies and MMAs
// (bounded) and frees TMEM before returning.
#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>

#include "cng_internal.h"
#include "device_common.cuh"
#include "launch_count.h"
#include "screen_common.cuh"
#include "screen_tc.h"

namespace cng {

constexpr int RS_BM = 256;       // rows per CTA block
constexpr int RS_PRODUCER = 8;
constexpr int RS_MMA = 9;        // first MMA issuer (and TMEM owner); one issuer per accumulator
constexpr int rs_threads(int nbuf) { return 32 * (RS_MMA + 2 * nbuf); }
constexpr int RS_MAXST = 6;      // column tile stages at most
constexpr int RS_KT_MAX = 256;
constexpr int RS_SLACK = 16;     // keys past the wanted rank a cut between tiles may keep
constexpr int RS_C = 16;         // columns per chunk: the epilogue's unit of maxima and appends

struct ResParams {
  int64_t m, n;
  int kt, d, nst, ntiles;
  int Lp, cap, self_excl;
  uint32_t idesc;
  uint32_t a1, acc0;             // TMEM columns of the second A half and of the accumulators
  const unsigned char* A;        // row image, row 0 of the launch at position row0
  const unsigned char* B;        // column image
  int64_t row0;
  int npart;                     // sweep parts: tiles [.., part_end[i]) kept to rank part_rank[i]
  int part_end[RES_PARTS];
  int part_rank[RES_PARTS];
  int nsplit, pre;               // column split: units = row blocks x nsplit, whole tiles up to pre
  uint64_t* mlist;               // [nsplit][m][Lp] a unit's keys (nsplit > 1), their number and the
  int32_t* mcnt;                 // [nsplit][m]     unit's threshold key
  uint32_t* mthr;
  uint16_t aux[RES_AUX];         // the row constants -c_i as operand bits
  const int32_t* row_perm;       // point id of a row position (null: the position)
  const int32_t* col_perm;       // point id of a column position (null: the position)
  const int32_t* col_pos;        // column position of a point id (self_excl)
  int32_t* ids;
  uint32_t* thr;
  uint64_t* rowbuf;
  uint32_t* status;
  uint32_t* sync;
  int sync_d;
};

// Shared-memory operand descriptor, K-major without swizzle: core matrices of 8 rows x 16 bytes
// (128 contiguous bytes), `lbo` bytes apart along K, 128 bytes apart along the rows.
CNG_DEV uint64_t desc_core(uint32_t addr, uint32_t lbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(lbo >> 4) << 16;
  d |= (uint64_t)(128 >> 4) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version
  return d;
}

CNG_DEV void mma_f16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(
          d_tmem),
      "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

CNG_DEV void tmem_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr),
               "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

#define RS_OUT16(r, o)                                                                            \
  "=r"(r[o + 0]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), \
      "=r"(r[o + 6]), "=r"(r[o + 7]), "=r"(r[o + 8]), "=r"(r[o + 9]), "=r"(r[o + 10]),            \
      "=r"(r[o + 11]), "=r"(r[o + 12]), "=r"(r[o + 13]), "=r"(r[o + 14]), "=r"(r[o + 15])
#define RS_TIE16(r, o)                                                                            \
  "+r"(r[o + 0]), "+r"(r[o + 1]), "+r"(r[o + 2]), "+r"(r[o + 3]), "+r"(r[o + 4]), "+r"(r[o + 5]), \
      "+r"(r[o + 6]), "+r"(r[o + 7]), "+r"(r[o + 8]), "+r"(r[o + 9]), "+r"(r[o + 10]),            \
      "+r"(r[o + 11]), "+r"(r[o + 12]), "+r"(r[o + 13]), "+r"(r[o + 14]), "+r"(r[o + 15])

// W consecutive FP32 columns of the warp's 32 TMEM lanes, complete on return.
template <int BN>
CNG_DEV void tmem_ld_tile(uint32_t taddr, uint32_t (&r)[BN]) {
  static_assert(BN == 64 || BN == 80 || BN == 96, "register tiles of the epilogue");
#pragma unroll
  for (int o = 0; o + 32 <= BN; o += 32)
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : RS_OUT16(r, o), RS_OUT16(r, o + 16)
        : "r"(taddr + (uint32_t)o));
  if constexpr (BN % 32 == 16)
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
        "[%16];"
        : RS_OUT16(r, (BN - 16))
        : "r"(taddr + (uint32_t)(BN - 16)));
  // the registers pass through the wait, so nothing that reads them moves above it
  asm volatile("tcgen05.wait::ld.sync.aligned;" : RS_TIE16(r, 0)::"memory");
#pragma unroll
  for (int o = 16; o < BN; o += 16) asm volatile("" : RS_TIE16(r, o));
}

CNG_DEV float max3f(float a, float b, float c) {
  float m;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(a), "f"(b), "f"(c));
  return m;
}

// Maximum of the 16 registers from o on, three inputs per operation.
template <int BN>
CNG_DEV float max16(const uint32_t (&r)[BN], int o) {
  float g[5];
#pragma unroll
  for (int i = 0; i < 5; ++i)
    g[i] = max3f(__uint_as_float(r[o + 3 * i]), __uint_as_float(r[o + 3 * i + 1]),
                 __uint_as_float(r[o + 3 * i + 2]));
  return fmaxf(max3f(g[0], g[1], g[2]), max3f(g[3], g[4], __uint_as_float(r[o + 15])));
}

// The `need` smallest of the cnt buffered keys, or up to `slack` more when a cut with that many
// is found first: moves them to the front of buf and returns the largest kept score key; *kept =
// their number.  Every dropped key lies at or above every kept one.  Bisection on the 32-bit score
// keys with one warp reduction per step; with the cut inside a run of equal keys the first of
// them in buffer order are kept.  cnt <= 32 CPL, cnt > need.  The other lanes' appends to buf are
// ordered before its loads here (votes and shuffles order no memory).
template <int CPL>
CNG_DEV uint32_t warp_cut(uint64_t* buf, int cnt, int need, int slack, int lane, int* kept) {
  uint64_t e[CPL];
  uint32_t k[CPL];
  __syncwarp();
  uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
  for (int i = 0; i < CPL; ++i) {
    const int idx = i * 32 + lane;
    e[i] = idx < cnt ? buf[idx] : ~0ull;
    k[i] = (uint32_t)(e[i] >> 32);
  }
#pragma unroll
  for (int i = 0; i < CPL; ++i) {
    if (i * 32 + lane < cnt) {
      lo = min(lo, k[i]);
      hi = max(hi, k[i]);
    }
  }
  lo = __reduce_min_sync(FULL, lo);
  hi = __reduce_max_sync(FULL, hi);
  int at = cnt;     // keys <= hi
  int below = 0;    // keys < lo
  while (lo < hi && at > need + slack) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    int c = 0;
#pragma unroll
    for (int i = 0; i < CPL; ++i) c += (i * 32 + lane < cnt && k[i] <= mid) ? 1 : 0;
    c = (int)__reduce_add_sync(FULL, (unsigned)c);
    if (c >= need) {
      hi = mid;
      at = c;
    } else {
      lo = mid + 1;
      below = c;
    }
  }
  const bool whole = at <= need + slack;  // else lo == hi: a run of equal keys is cut
  int out = 0, eq = 0;
  uint32_t top = 0u;
  __syncwarp();
#pragma unroll
  for (int i = 0; i < CPL; ++i) {
    const bool valid = i * 32 + lane < cnt;
    const bool is_eq = !whole && valid && k[i] == hi;
    const unsigned be = __ballot_sync(FULL, is_eq);
    const int rank = eq + __popc(be & ((1u << lane) - 1));
    eq += __popc(be);
    const bool keep = valid && (is_eq ? rank < need - below : (whole ? k[i] <= hi : k[i] < hi));
    const unsigned bk = __ballot_sync(FULL, keep);
    if (keep) {
      buf[out + __popc(bk & ((1u << lane) - 1))] = e[i];
      top = max(top, k[i]);
    }
    out += __popc(bk);
  }
  __syncwarp();
  *kept = out;
  return __reduce_max_sync(FULL, top);
}

// A unit of work is a row block and a split of the columns: the tiles up to P.pre (sample parts, for
// the thresholds), then every nsplit-th of the rest from the split's own on.
struct ResUnit {
  int64_t rb;
  int split, ntiles;
};
// SPLIT = false: the unit is the row block (with the split's arithmetic in the tile loops a 1M x 128
// screen took 210 ms, without 202).
template <bool SPLIT>
CNG_DEV ResUnit res_unit(const ResParams& P, int64_t u, int64_t nrb) {
  if constexpr (!SPLIT) return ResUnit{u, 0, P.ntiles};
  ResUnit r;
  r.split = (int)(u / nrb);
  r.rb = u - r.split * nrb;
  r.ntiles = P.pre + (P.ntiles - P.pre - r.split + P.nsplit - 1) / P.nsplit;
  return r;
}
template <bool SPLIT>
CNG_DEV int res_tile(const ResParams& P, const ResUnit& r, int t) {
  if constexpr (!SPLIT) return t;
  return t < P.pre ? t : P.pre + r.split + (t - P.pre) * P.nsplit;
}

// Appends one row's (lane's) columns of the chunk [c0, c0 + 16) whose accumulators beat its
// threshold; mx is the chunk's maximum, so a single hit needs no search for its value (a second one
// in the same chunk is rare after the first tiles and picks its value by a select chain).
template <int BN>
CNG_DEV void append_chunk(const uint32_t (&r)[BN], int o, float mx, uint32_t c0, uint32_t n, uint32_t self,
                          float thr, uint64_t* rbuf, int& cnt) {
  uint32_t part[4] = {0u, 0u, 0u, 0u};  // four chains: the search is latency bound
#pragma unroll
  for (int j = 0; j < RS_C; ++j) part[j & 3] |= __uint_as_float(r[o + j]) > thr ? 1u << j : 0u;
  uint32_t mask = (part[0] | part[1]) | (part[2] | part[3]);
  float v = mx;
  const bool several = (mask & (mask - 1)) != 0;
  while (mask) {
    const int j = __ffs(mask) - 1;
    mask &= mask - 1;
    if (several) {
#pragma unroll
      for (int i = 0; i < RS_C; ++i) v = j == i ? __uint_as_float(r[o + i]) : v;
    }
    const uint32_t col = c0 + j;
    if (col < n && col != self) rbuf[cnt++] = ((uint64_t)fkey(-2.f * v) << 32) | col;
  }
}

template <int BN, int NBUF, int CPL, bool DUMP, bool SPLIT>
__global__ void __launch_bounds__(rs_threads(NBUF), 1) screen_res_kernel(const __grid_constant__ ResParams P,
                                                                   float* dump) {
  extern __shared__ __align__(128) unsigned char smem_res[];
  const int stage_bytes = BN * P.kt * 2;
  unsigned char* sB = smem_res;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sB + P.nst * stage_bytes);
  uint64_t* b_full = bars;                 // [nst]
  uint64_t* b_empty = bars + RS_MAXST;     // [nst]
  uint64_t* t_full = bars + 2 * RS_MAXST;  // [half][NBUF]
  uint64_t* t_empty = t_full + 4;          // [half][NBUF]
  uint64_t* a_full = t_empty + 4;          // [half]
  uint64_t* fin = a_full + 2;              // [issuer] MMA drain at exit
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fin + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t nrb = (P.m + RS_BM - 1) / RS_BM;
  const int64_t nunits = SPLIT ? nrb * P.nsplit : nrb;

  if (tid == 0) {
    for (int i = 0; i < P.nst; ++i) {
      mbar_init(&b_full[i], 1);
      mbar_init(&b_empty[i], 2);  // both issuers' commits
    }
    for (int i = 0; i < 2 * NBUF; ++i) {
      mbar_init(&t_full[i], 1);
      mbar_init(&t_empty[i], 4);
    }
    for (int i = 0; i < 2; ++i) mbar_init(&a_full[i], 4 + NBUF);  // the half's warps and issuers
    for (int i = 0; i < 2 * NBUF; ++i) mbar_init(&fin[i], 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == RS_MMA) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                     smem_u32(tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == RS_PRODUCER) {
    if (lane == 0) {
      int64_t it = 0;
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int64_t u = blockIdx.x; u < nunits && ok; u += gridDim.x) {
        const ResUnit un = res_unit<SPLIT>(P, u, nrb);
        for (int t = 0; t < un.ntiles; ++t, ++it) {
          wave_checkpoint(P.sync, P.sync_d, TC_SYNC_COLS / BN, it, nrb, P.ntiles);
          ok = mbar_wait(&b_empty[s], ph ^ 1, abort_flag, P.status);
          if (!ok) break;
          mbar_expect_tx(&b_full[s], (uint32_t)stage_bytes);
          bulk_load(sB + s * stage_bytes, P.B + (size_t)res_tile<SPLIT>(P, un, t) * stage_bytes,
                    (uint32_t)stage_bytes, &b_full[s]);
          if (++s == P.nst) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
      if (!ok) {
        // drain: wait (bounded) for copies this thread issued into stages not yet consumed
        for (int i = 0; i < P.nst; ++i) {
          for (uint32_t w = 0; w < (1u << 20); ++w)
            if (mbar_try(&b_full[i], 0) || mbar_try(&b_full[i], 1)) break;
        }
      }
    }
  } else if (warp >= RS_MMA) {
    // One issuer per accumulator (half and buffer): the tensor pipe takes only a few MMAs ahead, so
    // an issuer's barrier waits leave a gap of ~350 cycles after its MMAs; the others' fill it.
    const int half = (warp - RS_MMA) & 1, b = (warp - RS_MMA) >> 1;
    if (lane == 0) {
      int j = 0, s = 0, turn = 0;
      uint32_t sph = 0, bph = 1;
      bool ok = true;
      const int nk = P.kt / 16;
      const uint32_t lbo = (BN / 8) * 128;
      const uint32_t a_base = tmem + (half ? P.a1 : 0u);
      const uint32_t dt = tmem + P.acc0 + (uint32_t)((b * 2 + half) * BN);
      uint64_t* const tf = &t_full[half * NBUF + b];
      uint64_t* const te = &t_empty[half * NBUF + b];
      uint64_t* const fn = &fin[half * NBUF + b];
      for (int64_t u = blockIdx.x; u < nunits && ok; u += gridDim.x, ++j) {
        const int ntiles = res_unit<SPLIT>(P, u, nrb).ntiles;
        // An issuer takes part in the phase it waits for: with a single column tile a unit leaves one
        // buffer's issuer without work, and the next unit's phase could otherwise complete before
        // that issuer has seen this one (a parity wait cannot tell the two apart).
        mbar_arrive(&a_full[half]);
        ok = mbar_wait(&a_full[half], j & 1, abort_flag, P.status);
        if (!ok) break;
        tc_fence_after();
        for (int t = 0; t < ntiles; ++t) {
          if (turn == b) {
            ok = mbar_wait(&b_full[s], sph, abort_flag, P.status);
            if (!ok) break;
            ok = mbar_wait(te, bph, abort_flag, P.status);
            if (!ok) break;
            tc_fence_after();
            uint64_t bd = desc_core(smem_u32(sB + s * stage_bytes), lbo);
            uint32_t at = a_base;
            mma_f16_ta(dt, at, bd, P.idesc, 0);
#pragma unroll 4
            for (int k = 1; k < nk; ++k) {
              bd += (2 * lbo) >> 4;
              at += 8;
              mma_f16_ta(dt, at, bd, P.idesc, 1);
            }
            mma_commit(tf);
            mma_commit(&b_empty[s]);
            bph ^= 1u;
          }
          if (++turn == NBUF) turn = 0;
          if (++s == P.nst) {
            s = 0;
            sph ^= 1u;
          }
        }
      }
      // drain every MMA this thread issued before TMEM is released
      mma_commit(fn);
      for (uint32_t i = 0; i < (1u << 24); ++i)
        if (mbar_try(fn, 0)) break;
    }
  } else {
    // ---- epilogue: warps 0-7, one row per thread ----
    const int quarter = warp & 3, half = warp >> 2;
    const int rloc = half * 128 + quarter * 32 + lane;  // row within the block
    const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
    uint64_t* wbuf = P.rowbuf + ((size_t)blockIdx.x * RS_BM + warp * 32) * P.cap;
    uint64_t* rbuf = wbuf + (size_t)lane * P.cap;
    float thr = 0.f;  // accumulators above it enter the row's list (thr = -score / 2)
    int cnt = 0;
    auto cut = [&](int l, int need, int slack) {
      int kept;
      const int c_l = __shfl_sync(FULL, cnt, l);
      if (c_l <= need) return;
      const uint32_t key = warp_cut<CPL>(wbuf + (size_t)l * P.cap, c_l, need, slack, lane, &kept);
      if (lane == l) {
        thr = -0.5f * fkey_inv(key);
        cnt = kept;
      }
    };
    uint64_t* const tf = t_full + half * NBUF;
    uint64_t* const te = t_empty + half * NBUF;
    int b = 0;
    uint32_t bph = 0;
    bool ok = true;
    for (int64_t u = blockIdx.x; u < nunits && ok; u += gridDim.x) {
      const ResUnit un = res_unit<SPLIT>(P, u, nrb);
      const int64_t row = un.rb * RS_BM + rloc;
      const bool live = row < P.m;
      {
        // the row's operand into TMEM: every MMA of the previous block is complete (this warp
        // waited for its last tile)
        const int64_t pos = P.row0 + row;
        const unsigned char* src = P.A + (size_t)(pos / BN) * stage_bytes +
                                   (size_t)((pos % BN) >> 3) * 128 + (size_t)(pos & 7) * 16;
        for (int k = 0; k < P.kt / 16; ++k) {
          uint4 v[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
          if (live) {
            v[0] = __ldg(reinterpret_cast<const uint4*>(src + (size_t)(2 * k) * (BN / 8) * 128));
            v[1] = __ldg(reinterpret_cast<const uint4*>(src + (size_t)(2 * k + 1) * (BN / 8) * 128));
          }
          uint32_t w[8] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w};
#pragma unroll
          for (int i = 0; i < 8; ++i) {  // the norm pieces of the image give way to the constants
            const int e = 16 * k + 2 * i - P.d;
            if (e + 1 >= 0 && e < RES_AUX) {
              if (e >= 0) w[i] = (w[i] & 0xffff0000u) | P.aux[e];
              if (e + 1 < RES_AUX) w[i] = (w[i] & 0x0000ffffu) | ((uint32_t)P.aux[e + 1] << 16);
            }
          }
          tmem_st8(tmem + lanes + (half ? P.a1 : 0u) + (uint32_t)(8 * k), w);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&a_full[half]);
      }
      thr = live ? -__int_as_float(0x7f800000) : __int_as_float(0x7f800000);
      cnt = 0;
      const uint32_t self = P.self_excl && live ? (uint32_t)P.col_pos[P.row_perm[row]] : ~0u;
      int t = 0;
      for (int part = 0; part < P.npart && ok; ++part) {
        const int tend = SPLIT && part + 1 == P.npart ? un.ntiles : P.part_end[part];
        const int rank = P.part_rank[part];
        for (; t < tend; ++t) {
          ok = mbar_wait_warp(&tf[b], bph, abort_flag, P.status);
          if (!ok) break;
          tc_fence_after();
          uint32_t r[BN];
          tmem_ld_tile<BN>(tmem + lanes + P.acc0 + (uint32_t)((b * 2 + half) * BN), r);
          // the accumulator is in registers: back to its issuer
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&te[b]);
          if (++b == NBUF) {
            b = 0;
            bph ^= 1u;
          }
          if constexpr (DUMP) {
            const int64_t c0 = (int64_t)t * BN;
            if (live)
#pragma unroll
              for (int j = 0; j < BN; ++j)
                if (c0 + j < P.n) dump[row * P.n + c0 + j] = -2.f * __uint_as_float(r[j]);
          } else {
            const int tile = res_tile<SPLIT>(P, un, t);
            float m[BN / RS_C];
#pragma unroll
            for (int c = 0; c < BN / RS_C; ++c) m[c] = max16<BN>(r, c * RS_C);
            float mx = m[0];
#pragma unroll
            for (int c = 1; c < BN / RS_C; c += 2) mx = max3f(mx, m[c], m[min(c + 1, BN / RS_C - 1)]);
            if (__any_sync(FULL, mx > thr)) {
#pragma unroll
              for (int c = 0; c < BN / RS_C; ++c)
                if (m[c] > thr)
                  append_chunk<BN>(r, c * RS_C, m[c], (uint32_t)(tile * BN + c * RS_C), (uint32_t)P.n, self,
                                   thr, rbuf, cnt);
              // cut every list that could overflow on the next tile
              unsigned full = __ballot_sync(FULL, cnt > P.cap - BN);
              while (full) {
                const int l = __ffs(full) - 1;
                full &= full - 1;
                cut(l, rank, RS_SLACK);
              }
            }
          }
        }
        if (DUMP || !ok || part + 1 == P.npart) continue;
        // end of a sample part: every list down to the part's rank
        __syncwarp();
        for (int l = 0; l < 32; ++l) cut(l, rank, 0);
        if (SPLIT && part + 2 == P.npart && un.split > 0) cnt = 0;  // split 0 lists the sample's columns
      }
      if (!ok || DUMP) continue;
      // the Lp smallest of each list, ids and threshold key
      __syncwarp();
      for (int l = 0; l < 32; ++l) {
        int c_l = __shfl_sync(FULL, cnt, l);
        const float t_l = __shfl_sync(FULL, thr, l);
        const int64_t row_l = row - lane + l;
        if (row_l >= P.m) break;
        uint64_t* buf_l = wbuf + (size_t)l * P.cap;
        uint32_t key = isinf(t_l) ? 0xffffffffu : fkey(-2.f * t_l);
        if (c_l > P.Lp) key = warp_cut<CPL>(buf_l, c_l, P.Lp, 0, lane, &c_l);
        if constexpr (SPLIT) {
          const int64_t at = un.split * P.m + row_l;
          for (int i = lane; i < c_l; i += 32) P.mlist[at * P.Lp + i] = buf_l[i];
          if (lane == 0) {
            P.mcnt[at] = c_l;
            P.mthr[at] = key;
          }
          continue;
        }
        const int64_t orow = P.row_perm ? P.row_perm[row_l] : row_l;
        for (int i = lane; i < P.Lp; i += 32) {
          int32_t id = -1;
          if (i < c_l) {
            id = key_id(buf_l[i]);
            if (P.col_perm) id = P.col_perm[id];
          }
          P.ids[orow * P.Lp + i] = id;
        }
        if (lane == 0) P.thr[orow] = key;
      }
      __syncwarp();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == RS_MMA) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

// The Lp smallest of a row's keys over its splits, one warp per row.  A column that is not listed lies
// at or above the smallest of the splits' thresholds and of the cuts made here.
constexpr int RS_MCAP = 24 * 32;
__global__ void __launch_bounds__(256) screen_merge_kernel(const __grid_constant__ ResParams P) {
  __shared__ uint64_t bufs[8][RS_MCAP];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t row = (int64_t)blockIdx.x * 8 + warp;
  if (row >= P.m) return;
  uint64_t* buf = bufs[warp];
  uint32_t thr = 0xffffffffu;
  int cnt = 0;
  // lists are complete only if the screen's waits were: otherwise (the call fails) empty lists
  const int nsplit = *reinterpret_cast<volatile uint32_t*>(P.status) ? 0 : P.nsplit;
  for (int sp = 0; sp < nsplit; ++sp) {
    const int64_t at = sp * P.m + row;
    const int c = P.mcnt[at];
    thr = min(thr, P.mthr[at]);
    for (int i = 0; i < c;) {
      const int take = min(c - i, RS_MCAP - cnt);
      for (int j = lane; j < take; j += 32) buf[cnt + j] = P.mlist[at * P.Lp + i + j];
      __syncwarp();
      i += take;
      cnt += take;
      if (cnt == RS_MCAP) thr = min(thr, warp_cut<24>(buf, cnt, P.Lp, 0, lane, &cnt));
    }
  }
  if (cnt > P.Lp) thr = min(thr, warp_cut<24>(buf, cnt, P.Lp, 0, lane, &cnt));
  const int64_t orow = P.row_perm ? P.row_perm[row] : row;
  for (int i = lane; i < P.Lp; i += 32) {
    int32_t id = -1;
    if (i < cnt) {
      id = key_id(buf[i]);
      if (P.col_perm) id = P.col_perm[id];
    }
    P.ids[orow * P.Lp + i] = id;
  }
  if (lane == 0) P.thr[orow] = thr;
}

// ---- operand images ----------------------------------------------------------------------------
// Tile image of an operand matrix: tiles of BN rows, each tile a contiguous block of core matrices
// (8 rows x 16 bytes) ordered by K chunk, then row group -- the shared-memory layout of the MMA's
// B operand, so a tile is one bulk copy.  Row p is xi[perm[p]] (null: xi[p]) with the norm pieces
// appended; rows past n (up to the tile's end) have zero coordinates and the largest pieces, so
// their accumulators lie below any real column's.  One warp per 8 rows: lane = 4 (row) + quarter.
template <typename T>
CNG_DEV float aux_round(float v);
template <>
CNG_DEV float aux_round<__half>(float v) {
  return __half2float(__float2half_rn(fminf(fmaxf(v, -65504.f), 65504.f)));
}
template <>
CNG_DEV float aux_round<__nv_bfloat16>(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
CNG_DEV uint32_t aux_bits(__half v) { return __half_as_ushort(v); }
CNG_DEV uint32_t aux_bits(__nv_bfloat16 v) { return __bfloat16_as_ushort(v); }

struct AuxScale {
  float c[RES_AUX];
};

template <typename T>
__global__ void __launch_bounds__(256) tile_image_kernel(const uint32_t* __restrict__ xi,
                                                         const float* __restrict__ nb,
                                                         const int32_t* __restrict__ perm, int64_t n,
                                                         int64_t groups, int kpad, int d, int kt, int bn,
                                                         AuxScale ax, unsigned char* __restrict__ out) {
  const int lane = threadIdx.x & 31, r = lane >> 2, q = lane & 3;
  const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int gpt = bn / 8;  // row groups per tile
  for (int64_t g = w0; g < groups; g += nw) {
    const int64_t p = g * 8 + r;
    const int64_t src = p < n ? (perm ? perm[p] : p) : -1;
    uint32_t pc[RES_AUX];
    const float nbs = src >= 0 ? nb[src] : 0.f;
    const bool real = src >= 0 && isfinite(nbs);  // a NaN row is never anyone's candidate
    float h = real ? 0.5f * nbs : 3.0e38f;
#pragma unroll
    for (int i = 0; i < RES_AUX; ++i) {
      const float v = aux_round<T>(h / ax.c[i]);  // c[i]: powers of two
      h = real ? fmaf(-v, ax.c[i], h) : h;
      T b;
      if constexpr (sizeof(T) == 2 && std::is_same<T, __half>::value)
        b = __float2half_rn(v);
      else
        b = __float2bfloat16_rn(v);
      pc[i] = aux_bits(b);
    }
    unsigned char* dst = out + (size_t)(g / gpt) * bn * kt * 2 + (size_t)(g % gpt) * 128 + r * 16;
    for (int c = q; c < kt / 8; c += 4) {
      uint32_t w[4] = {0u, 0u, 0u, 0u};
      if (real && 8 * c < kpad) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(xi + src * (kpad / 2) + 4 * c));
        w[0] = v.x;
        w[1] = v.y;
        w[2] = v.z;
        w[3] = v.w;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int e = 8 * c + 2 * i - d;
#pragma unroll
        for (int a = 0; a < RES_AUX; ++a) {
          if (e == a) w[i] = (w[i] & 0xffff0000u) | pc[a];
          if (e + 1 == a) w[i] = (w[i] & 0x0000ffffu) | (pc[a] << 16);
        }
      }
      *reinterpret_cast<uint4*>(dst + (size_t)c * gpt * 128) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// Piece scales: FP16 pieces reach 65504 and resolve 2^-24 of their scale, so 2^15 four times
// covers ||y_b||^2 / 2 up to RES_NORM_MAX and 2^9, 1 take the remainder, down to 2^-25
// (RES_PIECE_ERR); BF16 pieces have FP32's
// range, so each takes 8 bits of the remainder at scale 1.
static AuxScale aux_scales(bool fp16) {
  AuxScale a;
  const float f16[RES_AUX] = {32768.f, 32768.f, 32768.f, 32768.f, 512.f, 1.f};
  for (int i = 0; i < RES_AUX; ++i) a.c[i] = fp16 ? f16[i] : 1.f;
  return a;
}

bool res_shape(int d, float nbmax, ResShape* r) {
  const int kt = (d + RES_AUX + 15) / 16 * 16;
  if (d < 1 || kt > RS_KT_MAX || !(0.5f * nbmax < RES_NORM_MAX)) return false;
  r->d = d;
  r->kt = kt;
  // A takes kt TMEM columns (two halves, padded), the accumulators 4 BN: the widest tile that fits
  r->bn = kt <= 128 ? 96 : (kt <= 192 ? 80 : 64);
  return true;
}

size_t res_image_bytes(const ResShape& r, int64_t rows) {
  return (size_t)((rows + r.bn - 1) / r.bn) * r.bn * r.kt * 2;
}

cudaError_t launch_tile_image(const ResShape& r, bool fp16, const void* xi, int kpad, const float* nb,
                              const int32_t* perm, int64_t rows, void* out, cudaStream_t s) {
  const int64_t groups = (rows + r.bn - 1) / r.bn * (r.bn / 8);
  const int grid = (int)std::min<int64_t>((groups + 7) / 8, (int64_t)num_sms() * 16);
  count_launch();
  if (fp16)
    tile_image_kernel<__half><<<grid, 256, 0, s>>>((const uint32_t*)xi, nb, perm, rows, groups, kpad, r.d,
                                                   r.kt, r.bn, aux_scales(true), (unsigned char*)out);
  else
    tile_image_kernel<__nv_bfloat16><<<grid, 256, 0, s>>>((const uint32_t*)xi, nb, perm, rows, groups, kpad,
                                                          r.d, r.kt, r.bn, aux_scales(false),
                                                          (unsigned char*)out);
  return cudaGetLastError();
}

// ---- sweep schedule ----------------------------------------------------------------------------
// Smallest r with P(Binomial(Lp, f) >= r) <= 1e-9: with it, fewer than r of a row's Lp smallest
// scores lie in a sample of the fraction f, so the sample's r-th smallest score is no smaller than
// the row's Lp-th.
static int sample_rank(int Lp, double f) {
  if (f >= 1.0) return Lp;
  double tail = 0.0;
  int r = Lp + 1;
  const double lf = std::log(f), lg = std::log1p(-f);
  while (r > 1) {
    const int k = r - 1;
    const double lp = std::lgamma(Lp + 1.0) - std::lgamma(k + 1.0) - std::lgamma(Lp - k + 1.0) + k * lf +
                      (Lp - k) * lg;
    tail += std::exp(lp);
    if (tail > 1e-9) break;
    r = k;
  }
  return r;
}

static void schedule(const TcScreenArgs& a, int bn, int ntiles, ResParams* p) {
  p->npart = 0;
  int64_t end = 0;
  for (int i = 0; i + 1 < RES_PARTS; ++i) {
    end += a.part_count[i];
    const int t = (int)std::min<int64_t>(end / bn, ntiles);
    // a part worth a cut: some tiles of its own, and a rank well below Lp
    const int prev = p->npart ? p->part_end[p->npart - 1] : 0;
    if (t - prev < 4 || t >= ntiles) continue;
    // by the part's sampling rate: the columns cut off at its last whole tile are those of one region
    // of the order, so rows far from it see all of their sample
    const int rank = sample_rank(a.Lp, (double)end / (double)a.n);
    if (rank * 4 > a.Lp * 3) continue;
    p->part_end[p->npart] = t;
    p->part_rank[p->npart++] = rank;
  }
  p->part_end[p->npart] = ntiles;
  p->part_rank[p->npart++] = a.Lp;
}

// List capacity: the last part appends about 1.3 Lp to the sample's rank; one size up if asked.
static int list_cap(int Lp, int step) {
  static const int caps[] = {12, 16, 20, 24};
  int ci = 0;
  while (ci < 3 && caps[ci] * 32 < 2 * Lp + 128) ++ci;
  return caps[std::min(3, ci + step)] * 32;
}

// Column split for launches whose row blocks leave half of the SMs or more idle: the split and the
// sample parts swept whole by each unit, at most one unit per SM, that minimise
//   unit overhead + sample tiles + other tiles / splits + hits
// in tiles of ~850 cycles; a hit per row costs ~6 tiles (the 32 rows of a warp append in turn; fewer
// rows, less), a unit's operand load and final lists ~40, merging the splits' lists ~60.  A list that
// starts empty takes its first `cap` columns at once, then a buffer's worth per cut, with the
// threshold of the last cut.  Screen of m rows, split / whole (ms): 1M x 128, k = 100: m = 1 0.42 / 5.5,
// 1,000 1.3 / 7.8, 5,000 2.6 / 7.8, 10,000 4.3 / 7.9; k = 10: 1,000 1.2 / 6.8, 10,000 3.8 / 6.9; 100k x 96,
// k = 100: 1,000 0.49 / 1.95, 10,000 1.2 / 2.0.  More than one unit per SM lost: 20,000 rows in 237 units
// 8.4 / 7.9 (k = 10: 10.1 / 6.9), 39,000 rows in 306 16.1 / 15.2, so from 77 row blocks on nothing is split.
static void split_columns(int64_t m, int bn, int64_t n, int Lp, int cap, ResParams* p) {
  p->nsplit = 1;
  p->pre = 0;
  const int64_t sms = num_sms(), nrb = (m + RS_BM - 1) / RS_BM;
  if (2 * nrb > sms) return;
  const double hit = std::max(0.5, 6.0 * (double)std::min<int64_t>(m, 32) / 32.0), unit = 40.0, merge = 60.0;
  auto fill = [&](double cols, int rank) {
    const double more = cap - bn - rank;  // appends between two cuts
    return 0.4 * std::min<double>(cols, cap) +
           (cols > cap ? more * std::log(cols / cap) / std::log1p(more / rank) : 0.0);
  };
  // appends per row up to the end of each part
  double upto[RES_PARTS], frac[RES_PARTS];
  for (int i = 0; i < p->npart; ++i) {
    frac[i] = std::min(1.0, (double)p->part_end[i] * bn / (double)n);
    upto[i] = i == 0 ? fill(frac[0] * (double)n, p->part_rank[0])
                     : upto[i - 1] + p->part_rank[i - 1] * (frac[i] / frac[i - 1] - 1.0);
  }
  double best = unit + p->ntiles + hit * upto[p->npart - 1];
  int best_k = -2;
  for (int k = -1; k + 1 < p->npart; ++k) {
    const int pre = k < 0 ? 0 : p->part_end[k];
    for (int64_t sp = 2; sp * nrb <= sms && sp * 4 <= p->ntiles - pre; ++sp) {
      const double h = k < 0 ? fill((double)n / (double)sp, Lp)
                             : upto[k] + p->part_rank[k] * (1.0 / frac[k] - 1.0) / (double)sp;
      const double c = merge + unit + pre + (double)(p->ntiles - pre) / (double)sp + hit * h;
      if (c < best) {
        best = c;
        best_k = k;
        p->nsplit = (int)sp;
        p->pre = pre;
      }
    }
  }
  if (p->nsplit == 1) return;
  p->npart = best_k + 2;  // the parts swept whole, then the unit's share of the rest
  p->part_end[best_k + 1] = p->ntiles;
  p->part_rank[best_k + 1] = Lp;
}

// Row buffers, then the checkpoint counters (one split) or the splits' lists, in 8-byte words.
struct ResScratch {
  int grid;
  size_t buf, sync, total;
};
static ResScratch res_scratch(int64_t m, int bn, const ResParams& p) {
  const int64_t nrb = (m + RS_BM - 1) / RS_BM;
  ResScratch r;
  r.grid = (int)std::min<int64_t>(nrb * p.nsplit, num_sms());
  r.buf = (size_t)r.grid * RS_BM * p.cap;
  const int64_t waves = (nrb + r.grid - 1) / r.grid;
  r.sync = p.nsplit > 1 ? 0 : (size_t)((waves * p.ntiles / (TC_SYNC_COLS / bn) + 3) / 2);
  r.total = r.buf + r.sync + (p.nsplit > 1 ? (size_t)m * p.nsplit * (p.Lp + 1) : 0);
  return r;
}

static void plan_res(const TcScreenArgs& a, int cap_step, bool split, ResParams* p) {
  const int bn = a.res.bn;
  p->ntiles = (int)((a.n + bn - 1) / bn);
  p->Lp = a.Lp;
  p->cap = list_cap(a.Lp, cap_step);
  schedule(a, bn, p->ntiles, p);
  p->nsplit = 1;
  p->pre = 0;
  if (split) split_columns(a.m, bn, a.n, a.Lp, p->cap, p);
  if (p->nsplit > 1) p->cap = p->cap <= 512 ? 512 : 768;  // the capacities split kernels are built for
}

size_t screen_res_rowbuf_words(const TcScreenArgs& a, int cap_step) {
  ResParams p{}, whole{};  // the test aid that dumps scores does not split
  plan_res(a, cap_step, true, &p);
  plan_res(a, cap_step, false, &whole);
  return std::max(res_scratch(a.m, a.res.bn, p).total, res_scratch(a.m, a.res.bn, whole).total);
}

template <int BN, int NBUF, int CPL, bool DUMP, bool SPLIT>
static cudaError_t launch_res_t(const ResParams& p, size_t smem, int grid, cudaStream_t s, float* dump) {
  cudaError_t e = cudaFuncSetAttribute(screen_res_kernel<BN, NBUF, CPL, DUMP, SPLIT>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // cooperative when the producers wait for one another (boundedly): every CTA resident at once
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(rs_threads(NBUF));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = p.sync ? 1 : 0;
  count_launch();
  e = cudaLaunchKernelEx(&cfg, screen_res_kernel<BN, NBUF, CPL, DUMP, SPLIT>, p, dump);
  if (e == cudaErrorCooperativeLaunchTooLarge) {  // not all resident: plain launch (waits bounded)
    (void)cudaGetLastError();
    cfg.numAttrs = 0;
    e = cudaLaunchKernelEx(&cfg, screen_res_kernel<BN, NBUF, CPL, DUMP, SPLIT>, p, dump);
  }
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <int BN, int NBUF>
static cudaError_t launch_res_bn(int cpl, const ResParams& p, size_t smem, int grid, cudaStream_t s,
                                 float* dump) {
  if (dump) return launch_res_t<BN, NBUF, 12, true, false>(p, smem, grid, s, dump);
  if (p.nsplit > 1)
    return cpl == 16 ? launch_res_t<BN, NBUF, 16, false, true>(p, smem, grid, s, dump)
                     : launch_res_t<BN, NBUF, 24, false, true>(p, smem, grid, s, dump);
  switch (cpl) {
    case 12: return launch_res_t<BN, NBUF, 12, false, false>(p, smem, grid, s, dump);
    case 16: return launch_res_t<BN, NBUF, 16, false, false>(p, smem, grid, s, dump);
    case 20: return launch_res_t<BN, NBUF, 20, false, false>(p, smem, grid, s, dump);
    case 24: return launch_res_t<BN, NBUF, 24, false, false>(p, smem, grid, s, dump);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_screen_res(const TcScreenArgs& a, const TcVariant& v, int variant, cudaStream_t s,
                              std::string* msg, float* dump, TcShape* shape) {
  const int bn = a.res.bn, kt = a.res.kt;
  ResParams p{};
  p.m = a.m;
  p.n = a.n;
  p.kt = kt;
  p.d = a.res.d;
  plan_res(a, v.cap_step, a.split && !dump, &p);
  const int stage_bytes = bn * kt * 2;
  const int fixed = (2 * RS_MAXST + 14) * 8 + 16;
  // at least 4: an issuer sees every phase of its stages (an even number of them), or (5) reaches a
  // stage's next phase only after the epilogue has read the tile of the one it skipped
  p.nst = std::min(RS_MAXST, (226 * 1024 - fixed) / stage_bytes) - v.stages_less;
  if (p.nst < 4) {
    if (msg) *msg = "shared memory too small for four column tiles; ";
    return cudaErrorInvalidValue;
  }
  if (p.cap < a.Lp + 128) {
    if (msg) *msg = "screened list too long; ";
    return cudaErrorInvalidValue;
  }
  p.sync_d = v.sync_d;
  if (shape) *shape = TcShape{variant, p.nst, p.cap, p.sync_d};
  p.self_excl = a.self_excl;
  p.idesc = (1u << 4) | ((a.fp16 ? 0u : 1u) << 7) | ((a.fp16 ? 0u : 1u) << 10) |
            ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
  p.a1 = (uint32_t)((kt / 2 + 15) / 16 * 16);
  p.acc0 = (2 * p.a1 + 31) / 32 * 32;
  if (p.acc0 + 4 * bn > 512) {
    if (msg) *msg = "operands do not fit in TMEM; ";
    return cudaErrorInvalidValue;
  }
  p.A = static_cast<const unsigned char*>(a.A);
  p.B = static_cast<const unsigned char*>(a.B);
  p.row0 = a.row_off;
  const AuxScale ax = aux_scales(a.fp16 != 0);
  for (int i = 0; i < RES_AUX; ++i) {
    if (a.fp16) {
      p.aux[i] = __half_as_ushort(__float2half_rn(-ax.c[i]));
    } else {
      p.aux[i] = __bfloat16_as_ushort(__float2bfloat16_rn(-ax.c[i]));
    }
  }
  p.row_perm = dump ? nullptr : a.perm;
  p.col_perm = dump ? nullptr : a.col_perm;
  p.col_pos = a.col_pos;
  if (p.self_excl && (!p.row_perm || !p.col_pos)) {
    if (msg) *msg = "self exclusion needs the row and column orders; ";
    return cudaErrorInvalidValue;
  }
  p.ids = a.ids;
  p.thr = a.thr;
  p.status = a.status;
  const ResScratch sc = res_scratch(a.m, bn, p);
  // at least ~116 KB so that a single CTA (and its 512 TMEM columns) fits per SM
  const size_t smem = std::max<size_t>((size_t)fixed + (size_t)p.nst * stage_bytes, 116 * 1024);
  if (!a.rowbuf || a.rowbuf_words < sc.total) {
    if (msg) *msg = "row buffer missing or too small; ";
    return cudaErrorInvalidValue;
  }
  p.rowbuf = a.rowbuf;
  if (p.nsplit > 1) {
    p.mlist = a.rowbuf + sc.buf;
    p.mcnt = reinterpret_cast<int32_t*>(p.mlist + (size_t)a.m * p.nsplit * p.Lp);
    p.mthr = reinterpret_cast<uint32_t*>(p.mcnt + (size_t)a.m * p.nsplit);
  } else if (!dump) {  // checkpoint counters after the row buffers, zeroed on the stream
    p.sync = reinterpret_cast<uint32_t*>(a.rowbuf + sc.buf);
    cudaError_t ze = cudaMemsetAsync(p.sync, 0, sc.sync * 8, s);
    if (ze != cudaSuccess) return ze;
  }
  const int cpl = p.cap / 32;
  cudaError_t e = bn == 96   ? launch_res_bn<96, 2>(cpl, p, smem, sc.grid, s, dump)
                  : bn == 80 ? launch_res_bn<80, 2>(cpl, p, smem, sc.grid, s, dump)
                             : launch_res_bn<64, 2>(cpl, p, smem, sc.grid, s, dump);
  if (e != cudaSuccess || p.nsplit == 1) return e;
  count_launch();
  screen_merge_kernel<<<(unsigned)((a.m + 7) / 8), 256, 0, s>>>(p);
  return cudaGetLastError();
}

}  // namespace cng
