// window_rows.h -- which windows a lane takes, in index arithmetic that holds
// up to the largest read (2^32 - 1 bases).  No CUDA in here, so that the CPU
// tests compile the same lines.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define DBG_HD __host__ __device__ __forceinline__
#else
#define DBG_HD inline
#endif

namespace dbg {

// A warp goes through the cnt windows of a read in rows of 32: the rows, and
// whether lane's window of a row is there.  (A row's first window, 32 row, is
// below cnt; 32 rows itself may be 2^32, so that a loop over first windows
// would not end.)
DBG_HD uint32_t window_rows(uint32_t cnt) { return cnt / 32 + (cnt % 32 ? 1u : 0u); }
DBG_HD bool in_row(uint32_t cnt, uint32_t row, uint32_t lane) { return cnt - 32 * row > lane; }

}  // namespace dbg
