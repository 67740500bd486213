// screen_tc.h -- tensor-core candidate screen (tcgen05 + TMA), host interface.
#pragma once

#include <stdint.h>

#include <string>

#include <cuda_runtime.h>

namespace cng {

// Rows of up to 250 coordinates are screened from prepared tile images (k_screen_res.cu): operand
// width kt (the coordinates and RES_AUX norm pieces, rounded up to 16) and column tile bn.
constexpr int RES_AUX = 6;
constexpr int RES_PARTS = 4;                                // parts of the sampled column order
constexpr float RES_NORM_MAX = 4.f * 65504.f * 32768.f;     // largest ||y_b||^2 / 2 the pieces hold
// FP16 pieces hold ||y_b||^2 / 2 to max(2^-25, 2^-35 of it): the relative part is far below the
// accumulation error, the absolute one (twice that in a score; a factor 2 more is left) is not for
// operands with norms below about 0.03, which the operand scale avoids.
constexpr float RES_PIECE_ERR = 1.1920929e-7f;              // 2^-23
struct ResShape {
  int d = 0, kt = 0, bn = 0;
};
// The shape for d coordinates and a largest squared operand norm, or false if not supported.
bool res_shape(int d, float nbmax, ResShape* r);
size_t res_image_bytes(const ResShape& r, int64_t rows);
// out = tile image of xi[perm[p]] (perm null: xi[p]), p < rows; xi: [.][kpad] 16-bit operands with
// squared norms nb.
cudaError_t launch_tile_image(const ResShape& r, bool fp16, const void* xi, int kpad, const float* nb,
                              const int32_t* perm, int64_t rows, void* out, cudaStream_t s);

struct TcScreenArgs {
  // res.kt > 0: A and B are tile images (nb unused), columns in a sampled order: column position p
  // is point col_perm[p] and the first part_count[0] positions are the first part, and so on
  ResShape res;
  const int32_t* col_perm = nullptr;
  const int32_t* col_pos = nullptr;  // its inverse (self_excl): the column position of a point
  int64_t part_count[RES_PARTS] = {0, 0, 0, 0};
  const void* A;      // rows   [m][kpad] bf16 (fp16 when fp16 != 0), zero padded
  const void* B;      // columns [n][kpad]
  int64_t m, n;
  int kpad;           // multiple of 64
  int fp16;
  const float* nb;    // ||y_b||^2 per column (length >= n rounded up to 256, zero padded)
  int Lp;             // screened list length per row
  int self_excl;      // 1: row i is column i and is skipped
  int32_t* ids;       // [m][Lp] screened ids (unordered), -1 padded
  uint32_t* thr;      // [m] ordered key of the largest kept score (0xffffffff: all kept)
  uint32_t* status;
  uint64_t* rowbuf;     // scratch: screen_tc_rowbuf_words() words
  size_t rowbuf_words;
  // Locality order (optional): A and B hold the points at positions of an order, perm[pos]
  // the point id; ids and thr are then written for the point ids (row perm[pos], column
  // perm[col]).  wave_start = 1 starts each wave of row blocks at its own column tile.
  const int32_t* perm;
  int wave_start;
  int64_t row_off = 0;  // position of row 0 in the order (tuning trials on a row sample)
  int split = 1;        // 0: never split the columns (tuning trials, sized as a part of the whole)
  int variant = -1;     // pipeline variant; -1: the autotuner's choice
};

// Pipeline shape a screen ran with: variant index, operand stages, row-buffer capacity,
// checkpoint lag (windows of 256 tiles).
struct TcShape {
  int variant, stages, cap, sync_d;
};
int screen_tc_variants();
// Pipeline variants the autotuner times: operand stages (0 = as many as shared memory holds,
// else that many fewer), row-buffer capacity step (0 = the smallest that fits, 1 = the next),
// checkpoint lag in windows of 32,768 columns.
struct TcVariant {
  int stages_less, cap_step, sync_d;
};
size_t screen_res_rowbuf_words(const TcScreenArgs& a, int cap_step);
cudaError_t launch_screen_res(const TcScreenArgs& a, const TcVariant& v, int variant, cudaStream_t s,
                              std::string* msg, float* dump, TcShape* shape);
// The autotuned variant for a's shape (timing the variants on first use; synchronises `s`).
cudaError_t launch_screen_tc_tune(const TcScreenArgs& a, cudaStream_t s, std::string* msg, int* variant);

bool tc_screen_supported(int d, bool fp16);
// Scratch words of a screen (every field but the pointers set): row buffers, checkpoint counters and
// the lists of a column split.
size_t screen_tc_rowbuf_words(const TcScreenArgs& a);
// The screen (launch on `s`); with a.variant < 0 the autotuned variant for this shape, timed
// on first use (synchronises `s` then).  *shape, if given, receives the shape used.
cudaError_t launch_screen_tc(const TcScreenArgs& a, cudaStream_t s, std::string* msg,
                             TcShape* shape = nullptr);
// Test aid: writes every screened score s(x, y) to dump[m][n] instead of selecting.
// One warp runs the screen's bounded waits on a barrier and a flag that never complete; they
// must run out and leave ST_TIMEOUT in *status (never_set: a zeroed device word).
cudaError_t launch_wait_probe(uint32_t* status, const uint32_t* never_set, cudaStream_t s);
cudaError_t launch_screen_tc_dump(const TcScreenArgs& a, float* dump, cudaStream_t s,
                                  std::string* msg);

}  // namespace cng
