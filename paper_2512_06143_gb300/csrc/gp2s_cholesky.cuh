// gp2s_cholesky.cuh -- the tiled FP64 Cholesky factorisation shared by the exact log-determinant and the
// allocation-free entry point (cholesky.cu).
#pragma once

#include "gp2s_internal.cuh"

namespace gp2s {

constexpr int kCT = 32;                  // rows and columns of a tile (row-major, 1,024 doubles)
constexpr int kCTElems = kCT * kCT;

// A lower-triangular tile matrix and its task list.  Positions 0..nt-1 are the tile rows / columns in
// elimination order; tile (i, j), i >= j, of the factor has a slot of kCTElems doubles.  With colptr ==
// nullptr every tile of the triangle is present, positions are the natural order and slots run down
// the columns.
struct CholArgs {
    int nt, ntiles, ntasks;
    int n;                       // rows; a row at or past n is an identity row
    int last;                    // position of the tile row that holds row n - 1
    int solve;                   // 0: factor only, 1: also x = A^{-1} b
    const int *colptr, *rowpos;  // nt + 1, ntiles: per column the positions of its tiles (diagonal first)
    const int *rptr, *rcol, *rslot;   // per row position: the columns left of the diagonal, and the slots
    const int4 *tasks;           // (kind, i, j, slot)
    const int *perm;             // position -> tile index of the unpermuted matrix (nullptr: identity)
    double *tiles;               // ntiles x kCTElems: the matrix on entry, the factor on return
    double *dinv;                // nt x kCT: reciprocals of the factor's diagonal
    const double *b;             // n (unpermuted), may be scaled by bs
    const double *bs;
    double *yv, *xv;             // nt x kCT each: forward and backward solutions (elimination order)
    double *x;                   // n (unpermuted): the solution, scaled by bs
    double *bh, *xh;             // n (unpermuted), optional: bs * b and the solution before its scaling
    int *flags;                  // ntiles + 2 nt finished marks, then the ticket counter and the abort word
    int *bad;                    // bit 0: a pivot was not positive, bit 1: a bounded wait gave up
};

// Ints at args.flags that the caller zeroes before each launch.
inline size_t chol_flag_ints(int ntiles, int nt) { return (size_t)ntiles + 2 * (size_t)nt + 2; }
inline int chol_dense_tiles(int nt) { return nt * (nt + 1) / 2; }

// Queue the factorisation (and the solve) on stream; one kernel.
cudaError_t chol_launch(const CholArgs &a, int num_sms, cudaStream_t stream);

}  // namespace gp2s
