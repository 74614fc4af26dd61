// Detector rows of a column of voxels in the backprojection, plain C++ so that a
// CPU test can compile it.
//
// A group of consecutive voxels takes its samples without a test when the rows
// of its first and last voxel lie inside the detector.  Height and row are one
// FMA each, wherever they are formed: an FMA is monotonic in its operands, so the
// rows between lie between those two, and the row that is tested is the row that
// is read.  (A product rounded before the sum can come out as row 0 where the FMA
// gives a negative one, and the sample before the image would be read.)
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define GDRR_HD __host__ __device__ __forceinline__
#else
#define GDRR_HD inline
#endif

namespace gdrr {

// height of voxel iz: the first one's z0, dz apart
GDRR_HD float bp_height(float z0, int iz, float dz) { return fmaf((float)iz, dz, z0); }
// its row: sv rows per mm, hv at height 0
GDRR_HD float bp_row(float z, float sv, float hv) { return fmaf(z, sv, hv); }
// whether rows lo .. hi have both their samples (floor and the next) in 0 .. nv - 1
GDRR_HD bool bp_rows_inside(float lo, float hi, int nv) { return lo >= 0.0f && hi < (float)(nv - 1); }

}  // namespace gdrr
