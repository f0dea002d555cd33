// cf_slice64.cuh -- the FP64 Cholesky update on the tensor cores (cf_slice64.cu).
#pragma once

#include "cf_common.cuh"

namespace cf {

// Steps narrower than this keep the FP64 update: its time per tile falls with
// the step's width (64 x 64 outputs: 1 us per unit of width), the sliced
// update's does not (a width is padded to 64).  The line depends on the
// width alone, so every schedule of one factorization takes the same path.
constexpr int kSliceMinW = 17;

// Scratch of the sliced update of one step: the digit slices of L10's rows, their
// exponents and the flags of tiles left to FP64.
struct Slice64 {
    int rows = 0;                      // rows the slices can hold
    uint8_t *S = nullptr;
    int *E = nullptr;                  // row scale exponents
    int *flags = nullptr;              // any flag; row-tile flags
    size_t nflags = 0;
    int *any() const { return flags; }
    int *flag() const { return flags + 4; }
};
size_t slice64_bytes(int rows);
Slice64 slice64_carve(void *work, int rows);

// One step's update C -= L10 L10^T (i >= j) in FP64 accuracy:
//   operand   clears the step's flags, cuts L10's rows into slices;
//   update    C[i, j] -= for the sliced rows and the columns [c0, c1) of the
//             sliced ones (C and L10 point at row 0 of the slices).
int slice64_operand(const Slice64 &s, const double *L10, int lda, int rows, int w, const int *skip, cudaStream_t st);
int slice64_update(const Slice64 &s, int rows, int c0, int c1, int w, const double *L10, int lda, double *C, int ldc,
                   const int *skip, cudaStream_t st);
int slice64_take_status(cudaStream_t st, int *status);

}  // namespace cf
