// Which launches of the fused kernel (gemv.cu) fit the stage width to the round.
// Host code only.
#pragma once

#include <cstdint>

namespace seedq {

// At full width a round of 27 columns (1024 x 1024 at b1) keeps one warp of
// twelve busy.  A round wide enough for half the warps gains nothing from more
// of them (for n >= 2, whose stages are narrower, a quarter), one of fewer than
// five columns, or of a single row group, does not repay the run-time width,
// and where a CTA has more than a row group its round has several pieces, each
// with a narrow stage at its end: there the line is a sixth at b1, with more
// than two an eighth.  With several tensors some CTAs have a round on each side
// of a tensor's end, and those finish last: at b1 the line is a whole stage per
// warp.  Measured, full width / fitted, us: b1 1024 x 1024 12.1 / 10.9, 64 x
// 8192 13.7 / 12.7, 4096 x 256 12.3 / 10.8, 2048 x 2048 13.5 / 13.0, 6000 x 128
// 11.9 / 10.7, a d = 1024 layer 28.8 / 24.9; b2 1024 x 512 11.9 / 11.0, 400 x
// 2048 12.9 / 12.0, 6000 x 256 12.9 / 11.7; b4 1024 x 512 13.5 / 12.5, 64 x
// 8192 23.2 / 22.3.  Where full width is taken: b1 64 x 128 8.5 / 8.8, 8 x 8192
// 16.8 / 18.2, 6000 x 1024 13.3 / 14.2; b2 64 x 128 9.7 / 9.9, 11008 x 128 12.5
// / 12.7; b4 8 x 8192 33.0 / 34.0, 11008 x 128 13.7 / 14.1, 4096 x 1024 16.6 /
// 18.6.
//   template_n    batch template: 1, 2 or 4
//   units         (row group, column) units of the launch, over its CTAs
//   full          columns of a round that give every warp a whole stage
//   tensors       of the launch; rows and nb (block columns) of a single one
inline bool short_rounds(int template_n, int64_t units, int ctas, int full, int tensors, int64_t rows, int nb) {
  if (units < 5 * (int64_t)ctas) return false;
  const int64_t all = (int64_t)ctas * full;
  if (tensors > 1) return units < (template_n > 1 ? all / 4 : all);
  if (rows <= 32) return false;
  const int64_t groups = (int64_t)ctas * nb;  // units of a row group per CTA
  return units < (units > 2 * groups ? all / 8 : template_n > 1 ? all / 4 : units > groups ? all / 6 : all / 2);
}

}  // namespace seedq
