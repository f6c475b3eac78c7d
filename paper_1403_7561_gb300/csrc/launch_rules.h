// Rules of launches that need neither the device nor the mesh (host only, no CUDA).
#pragma once

namespace qcad {

// FP32 Gram (gram32_kernel): tiles of 32 rows after which a thread's FP32 sums enter its double-float
// ones. Of a tile's eight chunks of four rows the first of `groups` row groups sums ceil(8 / groups), so
// no FP32 sum runs over more than 32 rows (after `groups` tiles it were 48 for six groups, that is for
// blocks of 13 to 16 columns).
inline int gram32_flush_tiles(int groups) { return 8 / ((8 + groups - 1) / groups); }

}  // namespace qcad
