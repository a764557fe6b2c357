// Binary64 contractions on the tensor cores by exact digit slices (kernels_ex.cu).
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

#include "internal.h"

namespace chfsi {

// Where a launch reports a bounded wait that gave up: a word of the context's own
// (contexts run side by side on their streams, and one must not read or clear
// another's) in host memory that the device can write, so that the host reads it
// after any synchronisation without a copy.  withhold: test hook, one arrival of
// the launch's first thread block is left out.
struct ExWatch {
  int* status;
  int withhold;
};

// The binary64 cell matrices as digit words.
struct ExCellData {
  uint64_t* words = nullptr;   // per cell, K-major: word of (row l, column k) at [(e ne + k) rp + l]
  int* hsum = nullptr;         // bound of the digit sums over a row (16 bytes), then the scales:
  int16_t* hexp() const { return (int16_t*)(hsum + 4); }   // exponent field of every cell row's largest entry
  size_t word_bytes = 0, exp_bytes = 0;
};
// Output tiles of a cell launch (one CTA per SM takes them in turn).
int64_t ex_cell_tiles(int64_t ncells, int ne, int ncol);
void ex_cell_bytes(int64_t ncells, int ne, size_t* words, size_t* ex);
// Fill d (buffers allocated by the caller) for the cell data that m describes
// (m.Ht, formed before, gives the scales).
cudaError_t ex_pack_cells(const ExCellData& d, const CellMatArgs& m, int ne, cudaStream_t s);

// R (cell, local node) rows x ncol (row stride ldr) = H~_e Y_e for every cell.
// work: ex_cell_work_bytes of scratch.
struct ExCellArgs {
  const int32_t* dofmap;
  int64_t ncells;
  int ne, ncol;
  const double* Y;
  int64_t ldy;
  double* R;
  int64_t ldr;
  void* work;
};
size_t ex_cell_work_bytes(int64_t ncells, int ne, int ncol);
cudaError_t ex_cell_launch(const ExCellData& d, const ExCellArgs& a, const ExWatch& w, cudaStream_t s);

// Y_out = alpha (sum of the cell rows + NL - shift Y_in) + beta Y_prev per unknown.
struct ExAssembleArgs {
  const int32_t* node_ptr;
  const int32_t* node_ent;
  int64_t M;
  int ncol;
  const double* R;             // 16-byte aligned, ldr even
  int64_t ldr;
  const double* NL;            // may be null; row stride ld_nl
  int64_t ld_nl;
  const double* Yin;
  int64_t ld_in;
  double* Yout;
  int64_t ld_out;
  const double* Yprev;         // may be null
  int64_t ld_prev;
  double alpha, beta, shift;
};
cudaError_t ex_assemble_launch(const ExAssembleArgs& a, cudaStream_t s);

// C (n1 x n2, column-major ldc) = A^T B over M rows (contract of launch_gram_fp64).
// work: ex_gram_work_bytes of scratch.
size_t ex_gram_work_bytes(int64_t M, int n1, int n2, int lower);
cudaError_t ex_gram(const double* A, int64_t lda, const double* B, int64_t ldb, int64_t M, int n1, int n2,
                    double* C, int64_t ldc, int lower, void* work, size_t work_bytes, const ExWatch& w,
                    cudaStream_t s);

// C (M x n2) = A (M x n1) U (contract of launch_tallgemm_fp64).
size_t ex_tall_work_bytes(int64_t M, int n1, int n2);
cudaError_t ex_tall(const double* A, int64_t lda, const double* U, int64_t ldu, int64_t M, int n1, int n2,
                    double* C, int64_t ldc, int upper, int trans, void* work, const ExWatch& w, cudaStream_t s);

}  // namespace chfsi
