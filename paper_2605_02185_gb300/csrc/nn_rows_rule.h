// nn_rows_rule.h -- which images the row-marching convolution takes.
#pragma once

namespace gbnn_tc {

// units: 128-pixel tiles of the image, over all samples.  A CTA of the row kernel loads the
// layer's weights (18 KB for 32 -> 32, 73 KB for 64 -> 64) and fills its ring before its
// first tile, so it pays from some tiles per SM on; below that conv_tc_kernel, a CTA per
// tile, is done sooner.  Measured on images 256 wide, us for the tile kernel and the row
// kernel at the sizes on either side of the line (tiles per SM):
//   32 -> 32   4: 8.0, 9.1    6: 12.8, 10.6       64 -> 32   8: 15.6, 16.1   12: 21.3, 20.2
//   32 -> 64   3: 8.5, 9.8    4: 12.0, 11.2       64 -> 64   6: 15.8, 17.6    8: 20.1, 20.0
//   32 -> 96   3: 10.4, 11.4  4: 13.2, 12.7       96 -> 32   8: 25.5, 26.3   12: 35.2, 35.4
// 8 channels, against the mma.sync kernel: 8 -> 32 always (1: 6.9, 5.0; 4: 9.6, 6.6);
// 32 -> 8 but for the 3 and 4 tiles per SM that mma.sync runs in one wave of four CTAs and
// the row kernel in more than one tile per CTA (2: 7.1, 6.8; 3: 7.5, 7.8; 4: 8.2, 9.1;
// 6: 15.6, 9.3).
constexpr bool rows_pay(int cin, int cout, long long units, int sms) {
  if (cin == 8) return true;
  if (cout == 8) return units <= 2ll * sms || units > 4ll * sms;
  const int per_sm = cin == 32 ? (cout == 32 ? 5 : 4) : cin == 64 ? (cout == 32 ? 10 : 8) : 12;
  return units >= (long long)per_sm * sms;
}

}  // namespace gbnn_tc
