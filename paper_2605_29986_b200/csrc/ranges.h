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
    int row_step, ch_step, chunks;
    CFGZIP_HD PieceWalk(unsigned block, unsigned blocks, int chunks_)
        : row(block / unsigned(chunks_)), ch(int(block % unsigned(chunks_))), row_step(int(blocks / unsigned(chunks_))),
          ch_step(int(blocks % unsigned(chunks_))), chunks(chunks_) {}
    CFGZIP_HD void next() {
        row += row_step;
        ch += ch_step;
        if (ch >= chunks) {
            ch -= chunks;
            ++row;
        }
    }
};

}  // namespace cfgzip
