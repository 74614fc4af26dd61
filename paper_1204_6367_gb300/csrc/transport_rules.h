// Sizes of the transport's photon pools and which form of them a run takes, plain
// C++ so that a CPU test can compile it.
#pragma once

#include <algorithm>
#include <cstddef>

#include "gdrr.h"

#ifdef __CUDACC__
#define GDRR_HDC __host__ __device__ constexpr
#else
#define GDRR_HDC constexpr
#endif

namespace gdrr {

constexpr int POOL_WARPS = 4;                     // warps of a block
constexpr int POOL_COUNTS = GDRR_NSTATS + 2;      // a warp's counts
constexpr int POOL_MOST = 84, POOL_MAX = 96;      // photons: the largest default pool, the largest an option asks for

// A form: material slots nm (2, 4, 8), the general form, local majorants.  A slot
// has 16-byte words; a warp its slots, two coefficients per material and lane,
// four lists of slot numbers, its counts.
GDRR_HDC int slot_words(int nm, bool gen, bool lm) { return 4 + (nm < 4 ? 1 : nm / 4) + (lm ? 1 : 0) + (gen ? 1 : 0); }
GDRR_HDC size_t pool_bytes(int n, int nm, bool gen, bool lm) {
    return (size_t)n * slot_words(nm, gen, lm) * 16 + (size_t)2 * nm * 32 * 4 + (size_t)4 * n + (POOL_COUNTS + 3) / 2 * 16;
}

// Resident blocks the registers are held down for: 24 warps per SM (80
// registers), 20 for the general form and 8 materials, 16 with local majorants,
// whose walk gains more from its registers.  Default form, 2 mm torso: 28 warps
// (72) and 32 (64 registers, spills in the flight loop) were 1 and 8 % slower.
// Local majorants, 2e7 histories: 20 and 12 warps 1 and 6 % slower than 16.
GDRR_HDC int pool_blocks(int nm, bool gen, bool lm) { return nm == 8 ? 5 : lm ? 4 : gen ? 5 : 6; }

// Photons of a warp's pool unless an option says otherwise: as many, up to 84, as
// leave an SM 60 KB of L1 beside the shared memory of its blocks (of five blocks
// with local majorants).  80 in every form had left 28 KB there and to 8
// materials, too little once the phantom outgrows L2 (2e7 histories with local
// majorants: 1 mm torso 16.2 ms and 13.0 so, 64 mm cells 23.5 and 17.5; 2 mm 13.0
// and 12.4; 8 materials in a torso 7.6 and 7.2 per 1e7).
constexpr size_t SM_SHARED = 196 * 1024, BLOCK_SHARED = 1024 + GDRR_NSTATS * 8;
constexpr size_t shared_of_blocks(int n, int nm, bool gen, bool lm) {
    return (lm ? 5 : pool_blocks(nm, gen, lm)) * (POOL_WARPS * pool_bytes(n, nm, gen, lm) + BLOCK_SHARED);
}
constexpr int default_pool(int nm, bool gen, bool lm) {
    int n = POOL_MOST;
    while (n > 32 && shared_of_blocks(n, nm, gen, lm) > SM_SHARED) n -= 4;
    return n;
}

// Edge in mm of a macro cell of 2^shift voxels: what a free flight's chance to
// end in the cell depends on, whatever the voxels are.
inline float cell_edge(const float (&vox_mm)[3], int shift) {
    return std::min(vox_mm[0], std::min(vox_mm[1], vox_mm[2])) * (float)(1 << shift);
}

// Local majorants: from this edge on most flights end in the cell they start in,
// and the general form decides their tentative collisions where they are, in the
// walk.  2e7 histories of the torso by way of the gather service and in the walk:
// 32 mm cells 13.1 and 16.1 ms (1 mm voxels), 12.5 and 15.2 (2 mm), 11.9 and 14.9
// (4 mm); 64 mm cells 21.3 and 17.5, 20.6 and 16.0, 19.8 and 15.6.
constexpr float LM_IN_PLACE_MM = 48.0f;
inline bool lm_in_place(float edge_mm) { return edge_mm >= LM_IN_PLACE_MM; }

// The global majorant: in cells this coarse few collisions are virtual by their
// cell's bound, and the general form forms the mixture of all of them in the
// flight.  1e7 histories of the torso by way of the gather service and in the
// flight: 96 mm cells 12.9 and 15.4 ms, 128 mm 15.4 and 15.0, 160 mm 17.7 and 15.0,
// 256 mm 22.9 and 14.9; with form factors 17.8 and 15.4, 21.4 and 15.1, 24.2 and
// 15.0, 30.3 and 14.9.
constexpr float COARSE_MM = 128.0f;
inline bool coarse_in_place(float edge_mm) { return edge_mm >= COARSE_MM; }

}  // namespace gdrr
