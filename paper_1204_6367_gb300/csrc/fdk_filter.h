// Launch shape of the reconstruction's row filter, plain C++ so that a CPU test can
// compile it.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

#ifndef GDRR_HD
#ifdef __CUDACC__
#define GDRR_HD __host__ __device__ __forceinline__
#else
#define GDRR_HD inline
#endif
#endif

namespace gdrr {

constexpr int FILTER_BLOCK = 256, FILTER_MAX_NU = 4096;
constexpr int FO = 8, FR = 4;    // outputs and rows of a thread's task
constexpr int FILTER_BLOCKS_PER_SM = 3;

struct FilterShape {
    int nb;          // sources of a parity, rounded up to a multiple of FO
    int oct;         // output groups of FO per parity
    int stride;      // samples of a row and parity in shared memory
    int tab;         // padded coefficients per parity
    int rows;        // rows per block, a multiple of FR
    int parts;       // blocks that share the tasks of the same rows
};

GDRR_HD int filter_pad(int i) { return i + i / FO; }
GDRR_HD int filter_tasks(const FilterShape& f) { return f.rows / FR * 2 * f.oct; }

// Rows per block: as many groups of FR as give every thread a task, but no more
// than spread the rows over the SMs.  Few rows of many samples are shared by
// several blocks, each with its part of the tasks, where a block would otherwise
// take more than one task a thread and SMs stay idle (may_share: not in place,
// where one block's outputs are another's samples).  A call in us, with the rows of
// a full block always and so: 8 x 8 pixels 70 and 20, 16 views of 64 x 48 37 and 21,
// one of 512 x 384 40 and 28, 128 rows of 4096 217 and 84 (with one row per block
// and without tasks 18, 20, 28 and 190).
inline FilterShape filter_shape(int nu, int64_t n_rows, int n_sm, bool may_share) {
    FilterShape f;
    f.nb = ((nu + 1) / 2 + FO - 1) / FO * FO;
    f.oct = f.nb / FO;
    f.stride = f.nb + 4;
    f.tab = (filter_pad(2 * f.nb + FO) + 3) / 4 * 4;
    const int64_t row_groups = (n_rows + FR - 1) / FR, resident = (int64_t)n_sm * FILTER_BLOCKS_PER_SM;
    const int64_t full = std::max(1, FILTER_BLOCK / (2 * f.oct));
    f.rows = FR * (int)std::min(full, std::max<int64_t>(1, (row_groups + resident - 1) / resident));
    const int64_t blocks = (n_rows + f.rows - 1) / f.rows;
    f.parts = may_share ? (int)std::max<int64_t>(1, std::min<int64_t>(n_sm / blocks, filter_tasks(f) / 64)) : 1;
    return f;
}

inline size_t filter_smem(const FilterShape& f) { return sizeof(float) * ((size_t)2 * f.rows * f.stride + 2 * f.tab); }
// the most that any shape takes: the widest row's, or a full block of the narrowest
inline size_t filter_smem_most() {
    size_t most = 0;
    for (int nu : {1, FILTER_MAX_NU}) most = std::max(most, filter_smem(filter_shape(nu, (int64_t)1 << 40, 1, false)));
    return most;
}

}  // namespace gdrr
