// screen_common.cuh -- PTX wrappers and bounded waits shared by the two tensor-core screen kernels
// (k_screen_tc.cu: rows streamed in K chunks; k_screen_res.cu: rows resident in TMEM).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "device_common.cuh"
#include "status_bits.h"

namespace cng {

// wait iterations before declaring a timeout (each try_wait may suspend the thread for a
// system-dependent time; no suspend-time hint, so a completed phase is seen at once)
constexpr uint32_t TC_SPIN = 1u << 19;

CNG_DEV uint32_t ld_acquire_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

CNG_DEV uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

CNG_DEV void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
CNG_DEV void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes)
               : "memory");
}
CNG_DEV void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
CNG_DEV bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait; returns false (and raises the CTA abort flag) on expiry or if aborted.
CNG_DEV bool mbar_wait(uint64_t* b, uint32_t parity, volatile int* abort_flag, uint32_t* status) {
  for (uint32_t i = 0; i < TC_SPIN; ++i) {
    if (mbar_try(b, parity)) return true;
    if ((i & 15u) == 15u && *abort_flag) return false;
  }
  *abort_flag = 1;
  atomicOr(status, ST_TIMEOUT);
  return false;
}

// Warp-uniform bounded wait: every lane polls, the warp proceeds only when all lanes saw the
// phase complete, so the whole warp leaves together (needed before .sync.aligned TMEM loads).
CNG_DEV bool mbar_wait_warp(uint64_t* b, uint32_t parity, volatile int* abort_flag, uint32_t* status,
                            uint32_t spin = TC_SPIN) {
  for (uint32_t i = 0; i < spin; ++i) {
    if (__all_sync(FULL, mbar_try(b, parity))) return true;
    if ((i & 15u) == 15u && __any_sync(FULL, *abort_flag != 0)) return false;
  }
  if ((threadIdx.x & 31) == 0) {
    *abort_flag = 1;
    atomicOr(status, ST_TIMEOUT);
  }
  __syncwarp();
  return false;
}

// Producers meet at checkpoints every `win` tiles (TC_SYNC_COLS columns) of their own sequence; a
// producer at checkpoint c waits until every CTA that reaches checkpoint c - lag has reached it,
// so the CTAs of a wave stay within lag windows of each other and share the column tiles through
// L2 instead of each streaming them from DRAM.  The wait only serves the cache: it is bounded
// (about 2 ms) and the producer proceeds when it expires.  A wave is the gridDim.x row blocks
// processed together; `sync` holds one zeroed counter per checkpoint (null: no checkpoints).
constexpr int TC_SYNC_COLS = 32768;
constexpr uint32_t TC_SYNC_SPIN = 8192;

CNG_DEV void wave_checkpoint(uint32_t* sync, int lag, int win, int64_t it, int64_t nrb, int ntiles) {
  if (!sync || it == 0 || it % win != 0) return;
  const int64_t c = it / win;
  atomicAdd(&sync[c], 1u);
  if (c <= lag) return;
  const int64_t cw = c - lag;
  // CTAs reaching tile index cw * win: those with a row block in wave (cw * win) / ntiles
  const int64_t w = (cw * win) / ntiles;
  const int64_t left = nrb - w * (int64_t)gridDim.x;
  const uint32_t expect = (uint32_t)(left < 0 ? 0 : (left > gridDim.x ? gridDim.x : left));
  for (uint32_t i = 0; i < TC_SYNC_SPIN; ++i) {
    if (ld_acquire_u32(&sync[cw]) >= expect) return;
    __nanosleep(200);
  }
}

CNG_DEV void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

CNG_DEV void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}
CNG_DEV void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
CNG_DEV void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

}  // namespace cng
