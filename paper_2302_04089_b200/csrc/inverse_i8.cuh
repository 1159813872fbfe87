// Float64 products on the int8 tensor cores (inverse_i8.cu), as the factorisation (inverse.cu) uses them.
#pragma once

#include "common.cuh"

namespace ziplm {

constexpr int kI8MostK = 16384;      // the int32 sums of digit products are exact up to this K

// An operand in digits: [L][8][rows][K] int8, a power-of-two scale per row (and room for exponents).
struct I8Operand {
    signed char* dig;
    double* scale;       // [L][rows]
    int* exps;           // [L][rows]
    int rows, K;         // multiples of 64
};

// Which part of K a tile needs: all, up to its last row / column, from its first row / column on.
enum KRange { K_ALL = 0, K_TO_COL, K_TO_ROW, K_FROM_COL, K_FROM_ROW };

// C[row][col] = beta C + alpha sum_k x[row][k] y[col][k]; with C == nullptr the result is H^-1 = M^T M,
// cropped to d x d and with the equilibration `eq` ([L][d] powers of two, or null) taken back.
struct I8Product {
    double* C; size_t layer_stride; int ld;
    double alpha; int beta;
    int krange, lower;                       // lower: only tiles that reach the lower triangle
    int d; const double* eq; double* out64; float* tri32; int pitch32, rows32; double* diag64;
    int* layer_status;
    int rows, cols, K;                       // set by i8_product, as is the
    unsigned spin;                           // poll limit of the producers' waits
    const double* x_scale; const double* y_scale;
};

// Digits of a block of a float64 matrix (leading dimension ld): operand rows are its rows, or its columns.
// tri: block of a lower triangular matrix whose tiles above the diagonal are not written.
ziplm_status i8_digits(const I8Operand& o, const double* src, size_t layer_stride, int ld, bool columns, bool tri,
                       int L, cudaStream_t st);
// Digits of the columns of a float32 matrix, zero from row k_valid and column column_valid on.
ziplm_status i8_digits_of_columns(const I8Operand& o, const float* src, size_t layer_stride, int ld, int k_valid,
                                  int column_valid, int L, cudaStream_t st);
// An operand of at least rows x K in a workspace; returns its bytes.
size_t carve_i8_operand(I8Operand* o, void* ws, int L, int rows, int K);

// Whether x^T x of L layers (rows x rows from K) is quicker here than in float64_clocks: a wave of tile
// pairs takes 7000 clocks per 64 of K and some 30000 for the rest, the digits three launches.
bool i8_symmetric_pays(int L, int rows, int K, double float64_clocks);

ziplm_status i8_product(const I8Operand& x, const I8Operand& y, I8Product p, int L, cudaStream_t st);

}  // namespace ziplm
