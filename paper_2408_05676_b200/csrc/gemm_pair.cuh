// The contraction for many token rows (gemm_pair.cu), as gemm.cu's dispatch calls it.
#pragma once
#include <cuda.h>

#include "model.cuh"

namespace laser {

constexpr int kPairCount = 74;   // pairs of SMs of the device: the grid is 2 x 74 CTAs

// Steps of more rows than this use the pair form, and the line lies where gemm.cu's form loses its third ring stage (a
// token tile above 153 rows leaves room for two): 7B step of 4 layers, 160 rows 584 us there against 598 here, 176 rows 684
// against 614, 272 rows 966 / 749, 576 rows 1547 / 1135, 1024 rows 2698 / 1600; 13B shape of 2 layers, 160 rows 419 / 421, 192
// rows 525 / 462, 1088 rows 2360 / 1493.  With operands as hi + lo pairs a staged weight block feeds both parts here and is
// staged twice there: 48 rows 521 / 546, 64 rows 565 / 566, 80 rows 632 / 614, 144 rows 865 / 706.
constexpr int gemm_pair_rows(bool pairs) { return pairs ? 64 : 160; }

// How a contraction is cut: NT token rows per tile, n_tt tiles over the token rows, and whether the tiles left over after
// the last full wave are cut along K; us = the estimate it was chosen by.
struct GemmPairShape { int NT, n_tt, split; double us; };
GemmPairShape gemm_pair_shape(int R_pad, int N, int K, int epi, bool pairs);
// The scratch for partial sums (fp32 values), and per cut tile and half of it: contributors arrived, slices finished, a
// mark per slice (a tile has at most kPairCount contributors, and at most kPairCount / 2 tiles are cut).  The state is zero
// between launches.
size_t gemm_pair_scratch_floats(int R_pad);
constexpr int kPairState = kPairCount + 2;
constexpr int kPairStateInts = kPairCount * kPairState;

laser_status gemm_pair_launch(laser_model* m, const GemmPairShape& sh, const CUtensorMap& tw, const CUtensorMap& ta, int N, int K, int epi,
                              const GemmEpilogue& e, cudaStream_t stream);
// Whether the current device can hold the whole grid at once.
bool gemm_pair_fits();

}  // namespace laser
