// Index arithmetic of the kernels that says what memory they touch, in plain C++ so that it is also checked on the host.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define CFGZIP_HD __host__ __device__ __forceinline__
#else
#define CFGZIP_HD inline
#endif

namespace cfgzip {

// Rows of `chunks` pieces each, dealt to the blocks of a grid in turn: where a block starts and goes on. The number of
// pieces may pass 2^31 (short rows), so they are never counted: row and piece move on separately.
struct PieceWalk {
    int64_t row;
    int ch;
    const int row_step, ch_step, chunks;
    // row_step, ch_step: the grid's blocks divided by `chunks`, and what is left over
    CFGZIP_HD PieceWalk(unsigned block, int chunks_, int row_step_, int ch_step_)
        : row(block / unsigned(chunks_)), ch(int(block - unsigned(row) * unsigned(chunks_))), row_step(row_step_), ch_step(ch_step_), chunks(chunks_) {}
    CFGZIP_HD void next() {
        row += row_step;
        ch += ch_step;
        if (ch >= chunks) {
            ch -= chunks;
            ++row;
        }
    }
};

// The loads of eight consecutive tokens of a row, t0 .. t0 + 7, of which those from 0 to end - 1 exist: all of them as whole
// vectors, some of them one by one, or none. Nothing outside the row is asked for: its neighbours need not be readable.
template <typename Whole, typename One>
CFGZIP_HD void octet_loads(int t0, int end, Whole&& whole, One&& one) {
    if (t0 >= 0 && t0 <= end - 8) {
        whole();
    } else if (t0 > -8 && t0 < end) {
        one();
    }
}
CFGZIP_HD bool octet_has(int t0, int q, int end) { return unsigned(t0 + q) < unsigned(end); }  // does its q-th token exist?

}  // namespace cfgzip
