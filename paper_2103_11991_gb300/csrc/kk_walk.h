// Index arithmetic of kernels whose reads must stay inside their arrays whatever
// the input: plain functions, so that the host can replay them over all inputs
// (a stray read that is not used is not seen in a kernel's results).
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define KK_WALK __host__ __device__ __forceinline__
#else
#define KK_WALK inline
#endif

namespace kk {

// k_num_chunk's walk of a run [.., f_hi) of a chunk's flattened products, 32 per
// step.  A piece starts at product `start`; its bit in the step's mask, when it
// starts in the 32 products from f on and inside the run.  A piece that starts past
// the run stays out: lanes past the run repeat its last product, f_hi - 1, and so
// have to find that product's piece.  (A later piece holds other entries of B:
// where A's row is in no order, f_hi - 1 counted from its start may lie before the
// first entry of B.)
KK_WALK uint32_t walk_start_bit(int start, int f, int f_hi) {
  const int at = start - f;
  return at >= 0 && at < 32 && start < f_hi ? 1u << at : 0u;
}
// Bits of the lanes up to this one.
KK_WALK uint32_t walk_upto(int lane) { return 0xffffffffu >> (31 - lane); }
// The product that a lane of the step from f on takes.
KK_WALK int walk_product(int f, int lane, int f_hi) { return f + lane < f_hi ? f + lane : f_hi - 1; }

// k_mlp_loss_grad: the next tile of samples of a CTA, count when there is none (the
// sum may lie beyond int for counts near its largest).
KK_WALK int walk_next_tile(int t0, int step, int count) { return count - t0 > step ? t0 + step : count; }

}  // namespace kk
