// Which form of the photon pools a run takes, plain C++ so that a CPU test can
// compile it.
#pragma once

#include <algorithm>
#include <cstddef>

namespace gdrr {

// Edge in mm of a macro cell of 2^shift voxels: what a free flight's chance to
// end in the cell depends on, whatever the voxels are.
inline float cell_edge(const float (&vox_mm)[3], int shift) {
    return std::min(vox_mm[0], std::min(vox_mm[1], vox_mm[2])) * (float)(1 << shift);
}

// Local majorants: from this edge on most flights end in the cell they start in,
// and the general form decides their tentative collisions where they are, in the
// walk.  2e7 histories of the torso by way of the gather service and in the walk:
// 32 mm cells 16.2 and 16.7 ms (1 mm voxels), 13.0 and 15.2 (2 mm), 12.2 and 14.8
// (4 mm); 64 mm cells 28.0 and 23.5, 21.8 and 16.9, 20.8 and 16.5.
constexpr float LM_IN_PLACE_MM = 48.0f;
inline bool lm_in_place(float edge_mm) { return edge_mm >= LM_IN_PLACE_MM; }

}  // namespace gdrr
