// tiles.h -- tile shapes of the FP32 and BF16 step kernels, shared by their
// round-to-nearest and stochastic-rounding translation units.
#pragma once

// tile of the FP32 kernel: SPFM_F32_TX threads of 4 cells in x, SPFM_F32_TY rows
#ifndef SPFM_F32_TX
#define SPFM_F32_TX 16
#endif
#ifndef SPFM_F32_TY
#define SPFM_F32_TY 16
#endif

namespace spfm {
// the square tile of FP32 batch items of shape 1: 8 threads of 4 cells, 32 rows
// (32 x 32 cells, the same 128 consumer threads), for grids narrower than the
// 64-cell tile or whose x extent it would pad
constexpr int kSqTX = 8, kSqTY = 32;
// FP32 TI_n steps of single grids use it, too (local_square)
// the BF16 tile: 8 threads of 8 cells in x, 16 rows
constexpr int kBfTX = 8, kBfTY = 16;

// the tensor map of a single-grid FP32 step
inline const CUtensorMap *f32_step_map(TmaCache *tma, int which, const StepCoef<float> &c, int scheme,
                                       const float *src)
{
    using Wide = TileShape<float, float, SPFM_F32_TX, SPFM_F32_TY>;
    using Sq = TileShape<float, float, kSqTX, kSqTY>;
    return local_square(c, scheme) ? cached_map(tma, which + 2, c.g, SPFM_F32, src, Sq::SW, Sq::ROWS)
                                   : cached_map(tma, which, c.g, SPFM_F32, src, Wide::SW, Wide::ROWS);
}
}  // namespace spfm
