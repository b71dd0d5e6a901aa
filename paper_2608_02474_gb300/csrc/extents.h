// Sizes and index walks that hold for every row count a call accepts (up to
// INT32_MAX), in plain C++ so that they are also compiled and checked on the host.
#pragma once
#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define ECHO_HD __host__ __device__ __forceinline__
#else
#define ECHO_HD inline
#endif

// Bytes of shared memory that n staged 32-bit keys take: they are written and read
// four at a time, so the last group is whole.
constexpr size_t key_stage_bytes(int n) { return ((size_t)n + 3) / 4 * 16; }

// Blocks of `per` rows that cover n >= 0 rows.
constexpr int blocks_for_rows(int n, int per) { return (int)(((int64_t)n + per - 1) / per); }

// A walk over rows in steps of the whole grid: row = first, first + step, ...  The
// first row at or past n, which ends it, may lie beyond INT32_MAX: unsigned.
struct RowWalk {
    unsigned row, step;
    ECHO_HD bool below(int n) const { return row < (unsigned)n; }
    ECHO_HD void next() { row += step; }
};

// A thread's walk over the pieces (row, piece of the row) of [n_rows, C] pieces in
// steps of the whole grid (thread t of `threads`), kept as row and piece: one
// division at the start instead of a 64-bit division per piece, which was as long as
// moving the piece.
struct PieceWalk {
    unsigned row, piece;
    ECHO_HD PieceWalk(unsigned t, unsigned threads, unsigned C)
        : row(t / C), piece(t % C), rows_(threads / C), pieces_(threads % C), C_(C) {}
    ECHO_HD bool below(int n) const { return row < (unsigned)n; }
    ECHO_HD void next() {
        row += rows_;
        piece += pieces_;
        if (piece >= C_) {
            piece -= C_;
            ++row;
        }
    }

  private:
    unsigned rows_, pieces_, C_;
};
