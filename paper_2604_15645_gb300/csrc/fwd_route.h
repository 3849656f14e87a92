// Which kernel runs a BF16 tanh forward layer: the rules on sizes, apart from the launches so
// that they can be checked without a GPU.
#pragma once
#include <cstdint>

namespace pinn {

// Whether a layer's forward runs in pairs of CTAs (k_tc_fwd_pair).  m_tiles x n_tiles units of
// 128 x 256 outputs, K the fan-in; an even number of m-tiles gives each pair two units of a
// column tile.  Paired against unpaired launch of one layer, measured at 6,000 to 200,000 points:
//   K below 384   slower at every size: the copies and MMAs that a pair shares are too few
//                 beside its epilogue (512 wide, K = 128, 20,000 points: 77 -> 90 us for the
//                 call; K = 256: 94 -> 100; K = 384: 113 -> 110)
//   few units     slower by 2-5 us a launch: a cluster starts and ends later (512 wide, K = 512:
//                 2.5 units per SM 56.5 -> 58.2 us, 8 units 127.9 -> 125.7; no faster up to 5 units
//                 at 256 to 1024 wide, at most 0.5% slower above 8)
//   weights' low half on the value rows only (a quarter of its MMAs), K above 512: slower,
//                 K = 768 by up to 2.6%, 1024 by 0.6-2.8%, 2048 by 2-5% (the 64-column MMAs
//                 read as much of the weights as full ones); K = 512: 288.7 -> 285.3 us at
//                 60,000 points
inline bool fwd_in_pairs(int m_tiles, int n_tiles, int K, bool wlo_values_only, int sm_count) {
  return sm_count >= 2 && m_tiles % 2 == 0 && K >= 384 && (!wlo_values_only || K <= 512) &&
         (int64_t)m_tiles * n_tiles >= 6 * (int64_t)sm_count;
}

// Whether a network's hidden GEMM layers (all at most 256 wide) run in one kernel
// (k_tc_fwd_all).  With a single layer there is nothing to keep in shared memory, and the layer's
// two m-tiles follow each other in one CTA: the layer's own launch is faster at every size
// (256 wide, K = 128, 3,000 points: 35.5 against 40.2 us for the loss; 40,000: 79.0 against 90.5;
// 128 wide 31.4 against 33.2 and 58.3 against 60.3).
inline bool fwd_in_one_kernel(int layers) { return layers >= 2; }

}  // namespace pinn
