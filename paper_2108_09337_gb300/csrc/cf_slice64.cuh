// cf_slice64.cuh -- the FP64 Schur update on the tensor cores (cf_slice64.cu).
#pragma once

#include "cf_common.cuh"

namespace cf {

// Steps narrower than this keep the FP64 update: its time per tile falls with
// the step's width (64 x 64 outputs: 1 us per unit of width), the sliced
// update's does not (a width is padded to 64).  The line depends on the
// width alone, so every schedule of one factorization takes the same path.
constexpr int kSliceMinW = 17;

// Scratch of the sliced update of one step: the digit slices of both operands
// and, per step, the inner exponents and the flags of tiles left to FP64.
struct Slice64 {
    int rows = 0, cols = 0;            // operand rows the slices can hold (cols 0: one operand, C -= A A^T)
    uint8_t *SA = nullptr, *SB = nullptr;
    int *E = nullptr, *F = nullptr;    // row / column scale exponents
    int *head = nullptr;               // inner exponents; any flag; row-tile flags; column-tile flags
    size_t nflags = 0;                 // ints from any() on
    int *rho() const { return head; }
    int *any() const { return head + kMaxV; }
    int *flagA() const { return any() + 4; }
    int *flagB() const { return flagA() + ceil_div(rows, 128); }
};
size_t slice64_bytes(int rows, int cols);
Slice64 slice64_carve(void *work, int rows, int cols);

// One step's update C -= A10 A01 in FP64 accuracy:
//   begin     clears the step's flags, takes the inner exponents of A01
//             (w x cols, all of the step's columns);
//   clear_flags  drops the flags alone (an update in pieces: before each piece's operands);
//   operands  cuts rows of A10 / columns of A01 into slices;
//   update    C[i, j] -= for the sliced rows and the columns [c0, c1) of the
//             sliced ones (C, A, B point at row 0, column 0 of the slices).
// Cholesky (lower): begin without A01, operands with A10 alone; i >= j only.
int slice64_begin(const Slice64 &s, const double *A01, int lda, int w, int cols, const int *skip, cudaStream_t st);
int slice64_clear_flags(const Slice64 &s, cudaStream_t st);
int slice64_operands(const Slice64 &s, const double *A10, int lda, int rows, const double *A01, int ldb, int cols,
                     int w, const int *skip, cudaStream_t st);
int slice64_update(const Slice64 &s, int rows, int c0, int c1, int w, const double *A10, int lda, const double *A01,
                   int ldb, double *C, int ldc, bool lower, const int *skip, cudaStream_t st);
int slice64_take_status(cudaStream_t st, int *status);

}  // namespace cf
