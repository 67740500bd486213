// row_warp.cuh -- warp-cooperative pieces on stored rows: squared distances of several rows at once,
// the bitonic sort of a key list, and the (D, id) order of its near-tied runs.
#pragma once

#include "device_common.cuh"

namespace cng {

constexpr int RR_RUN = 256;  // longest near-tie run re-sorted

// part_sqdist<8> on NR rows at once, in its order: partial squared distances of rows y[r] (r < NR)
// for lane g of a group of 8.
template <int NR>
CNG_DEV void part_rows(const float* __restrict__ q, const float* const (&y)[NR], int dpad, int g,
                       float (&p)[NR]) {
  const float4* q4 = reinterpret_cast<const float4*>(q) + g;
  const int u = dpad >> 5;  // chunks per lane
  float s0[NR], s1[NR], s2[NR], s3[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) s0[r] = s1[r] = s2[r] = s3[r] = 0.f;
  int t = 0;
  for (; t + 3 < u; t += 4) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float4 x[NR][2];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const float4* y4 = reinterpret_cast<const float4*>(y[r]) + g + 8 * t + 16 * h;
        x[r][0] = __ldg(y4);
        x[r][1] = __ldg(y4 + 8);
      }
      const float4 a0 = q4[8 * t + 16 * h], a1 = q4[8 * t + 16 * h + 8];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        acc4(a0, x[r][0], h ? s2[r] : s0[r]);
        acc4(a1, x[r][1], h ? s3[r] : s1[r]);
      }
    }
  }
#pragma unroll 3
  for (; t < u; ++t) {
    float4 x[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) x[r] = __ldg(reinterpret_cast<const float4*>(y[r]) + g + 8 * t);
    const float4 a = q4[8 * t];
#pragma unroll
    for (int r = 0; r < NR; ++r) acc4(a, x[r], s0[r]);
  }
#pragma unroll
  for (int r = 0; r < NR; ++r) p[r] = (s0[r] + s1[r]) + (s2[r] + s3[r]);
}
template <int NR>
CNG_DEV void part_rows(const float* __restrict__ q, const __half* const (&y)[NR], int dpad, int g,
                       float (&p)[NR]) {
  const float4* q4 = reinterpret_cast<const float4*>(q) + 2 * g;
  const int u = dpad >> 6;  // chunks of 8 halves per lane
  float s0[NR], s1[NR], s2[NR], s3[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) s0[r] = s1[r] = s2[r] = s3[r] = 0.f;
  int t = 0;
  for (; t + 1 < u; t += 2) {
    uint4 x[NR][2];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const uint4* y8 = reinterpret_cast<const uint4*>(y[r]) + g + 8 * t;
      x[r][0] = __ldg(y8);
      x[r][1] = __ldg(y8 + 8);
    }
    const float4 a0 = q4[16 * t], a1 = q4[16 * t + 1], b0 = q4[16 * t + 16], b1 = q4[16 * t + 17];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      acc4(a0, h8lo(x[r][0]), s0[r]);
      acc4(a1, h8hi(x[r][0]), s1[r]);
      acc4(b0, h8lo(x[r][1]), s2[r]);
      acc4(b1, h8hi(x[r][1]), s3[r]);
    }
  }
  for (; t < u; ++t) {
    const float4 a0 = q4[16 * t], a1 = q4[16 * t + 1];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const uint4 x = __ldg(reinterpret_cast<const uint4*>(y[r]) + g + 8 * t);
      acc4(a0, h8lo(x), s0[r]);
      acc4(a1, h8hi(x), s1[r]);
    }
  }
#pragma unroll
  for (int r = 0; r < NR; ++r) p[r] = (s0[r] + s1[r]) + (s2[r] + s3[r]);
}

CNG_DEV void warp_bitonic(uint64_t* a, int P2, int lane) {
  for (int k = 2; k <= P2; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = lane; i < P2; i += 32) {
        int ixj = i ^ j;
        if (ixj > i) {
          uint64_t x = a[i], y = a[ixj];
          bool up = (i & k) == 0;
          if ((x > y) == up) { a[i] = y; a[ixj] = x; }
        }
      }
      __syncwarp();
    }
}

// Re-sort, by the canonical (D, id) order, every run of neighbours in keys[0..cnt) whose FP32
// squared distances are pairwise near-tied and that starts before position `upto`.  `row` is
// the stored row vector (exact values).  Runs are gathered in batches (up to 32 runs, RR_RUN
// members); the members' squared distances are computed to within DD_EPS by the whole warp, one
// after the other, and lane 0 insertion-sorts each run; only if two of a run lie within DD_EPS are
// the batch's canonical FP64 distances taken, one per lane, and the runs sorted by those.  rdesc:
// [3][32] ints of warp scratch (run start, length, offset in d64).  Returns the number of runs
// re-decided.
template <typename T>
CNG_DEV int fix_runs_warp(uint64_t* keys, int cnt, int upto, const T* __restrict__ row,
                          const T* __restrict__ Xc, int dpad, int d, float band, double* d64,
                          int* rdesc, int lane, uint32_t* status) {
  int runs = 0;
  int i = 0;
  while (i < upto && i + 1 < cnt) {
    int nb = 0, total = 0;
    while (nb < 32 && i < upto && i + 1 < cnt) {
      // the next run start >= i (lane-parallel scan, 32 pairs at a time)
      int s = -1;
      for (int b = i; b < upto && b + 1 < cnt && s < 0; b += 32) {
        int t = b + lane;
        bool nt = t < upto && t + 1 < cnt && near_tie(key_dist(keys[t]), key_dist(keys[t + 1]), band);
        unsigned bal = __ballot_sync(FULL, nt);
        if (bal) s = b + __ffs(bal) - 1;
      }
      if (s < 0) {
        i = upto;
        break;
      }
      int e = s + 1;  // run is [s, e]
      while (e + 1 < cnt && near_tie(key_dist(keys[e]), key_dist(keys[e + 1]), band)) ++e;
      int len = e - s + 1;
      if (len > RR_RUN) {
        if (lane == 0) set_status(status, ST_OVF_RUN);
        len = RR_RUN;
        e = s + len - 1;
      }
      if (total + len > RR_RUN) break;  // this run opens the next batch
      if (lane == 0) {
        rdesc[nb] = s;
        rdesc[32 + nb] = len;
        rdesc[64 + nb] = total;
      }
      total += len;
      ++nb;
      i = e + 1;
    }
    if (nb == 0) break;
    __syncwarp();
    for (int k = 0; k < nb; ++k)
      for (int m = 0; m < rdesc[32 + k]; ++m) {
        const double v = warp_sqdist_dd(row, Xc + (int64_t)key_id(keys[rdesc[k] + m]) * dpad, d, lane);
        if (lane == 0) d64[rdesc[64 + k] + m] = v;
      }
    __syncwarp();
    for (int canon = 0; canon < 2; ++canon) {
      if (canon) {
        for (int m = lane; m < total; m += 32) {
          int k = 0;
          while (k + 1 < nb && rdesc[64 + k + 1] <= m) ++k;
          const int pos = rdesc[k] + (m - rdesc[64 + k]);
          d64[m] = canon_dist(row, Xc + (int64_t)key_id(keys[pos]) * dpad, d);
        }
        __syncwarp();
      }
      bool open = false;
      if (lane == 0) {  // insertion sort of each run by (d64, id)
        for (int k = 0; k < nb; ++k) {
          const int s = rdesc[k], len = rdesc[32 + k];
          double* dd = d64 + rdesc[64 + k];
          for (int a = 1; a < len; ++a) {
            double dv = dd[a];
            uint64_t kv = keys[s + a];
            int b = a - 1;
            while (b >= 0 && (dd[b] > dv || (dd[b] == dv && key_id(keys[s + b]) > key_id(kv)))) {
              dd[b + 1] = dd[b];
              keys[s + b + 1] = keys[s + b];
              --b;
            }
            dd[b + 1] = dv;
            keys[s + b + 1] = kv;
          }
          if (!canon)
            for (int a = 1; a < len; ++a) open |= dd_open(dd[a - 1], dd[a]);
        }
      }
      __syncwarp();
      if (!__any_sync(FULL, open)) break;
    }
    runs += nb;
  }
  return runs;
}

}  // namespace cng
