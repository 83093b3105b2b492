// spmv.cuh -- host-side dispatcher of the block-sparse product kernels.
#pragma once
#include "kernels.cuh"

namespace nbp {

// Launch y = epilogue(M x) on stream s.  vsel selects the value copy
// (0 FP64, 1 FP32, 2 BF16); XT is the vector type (double needs vsel 0).
// G: -1 = the autotuned choice (else sliced ELL when built); 0 = sliced ELL;
// kSellMT + T = sliced ELL with T threads per row (T = 2, 4, 8); other > 0 =
// flat kernel with G lanes per block row.  Returns the product's algorithmic
// bytes (what the launched kernel must move at least: values, columns, row or
// slice pointers, x once, the epilogue's vectors), for bandwidth accounting.
template <typename XT>
double spmv(const DMat &M, int vsel, SpmvArgs a, int epi, bool lr, cudaStream_t s, int G = -1);

int choose_group(const DMat &M);

// Threads per row of the finest level's products (A, its AMG level and the
// coupling blocks, about 15 entries a row): one where the rows alone fill the
// GPU (152 SMs x 2048 threads), up to eight where they do not and a row's
// chain of loads is what a product takes.  Solves with 1 / 2 / 4 / 8 threads:
// 29,760 rows 52.1 / 42.4 / 41.4 / 42.9 ms, 60,625 rows 51.3 / 47.8 / 48.3 /
// 54.0 ms, 68,921 rows 66.7 / 61.9 / 64.1 / 71.5 ms; 140,481 rows 176.6 / 169.8;
// 452,393 and 1,085,825 rows are faster with one.
// By the matrix's own rows alone: the threads set the order of a row's sum, so
// an instance of a batch gives the bits of its single solve.  Where half of the
// batch's rows ask for fewer threads, its products with A and the finest levels
// run with those (DMat::beside), each keeping the partial sums of several of
// the own threads apart: the same bits.  48 cubes of 12-40 in mode 4, ms: own
// threads / so / those threads and their own order everywhere 303 / 279 / 262; 30
// batches of 3-16 cubes of 8-36, speed against the last: own threads 0.968 / 0.955
// / 0.962 (modes 1, 3, 4), so 0.981 / 0.993 / 1.007, with the coupling products
// and S_hat's FP32 ones in the same way 0.968 / 0.972 / 0.987.
int fine_threads(int rows);

// Whether y = M x with the K-cycle's inner products fused (k_sell_dot) runs
// for this matrix: scalar blocks, the sliced kernel (1-8 threads per row) as
// the tuned choice, the value copy of vsel built, and a grid of at most
// max_blocks blocks (the partials buffer).
bool spmv_dot_ok(const DMat &M, int vsel, int xbytes, long long max_blocks);
// Launch it (spmv_dot_ok must hold); returns the algorithmic bytes: the
// product's, plus da and db.
template <typename XT>
double spmv_dot(const DMat &M, int vsel, SpmvArgs a, const DotArgs &q, cudaStream_t s);

// The prolongation and the first post-smoothing step (EPI_POST) with AP's
// sliced copy; returns the algorithmic bytes.
template <typename XT> double spmv_post(const DMat &AP, int vsel, SpmvArgs a, cudaStream_t s);


}  // namespace nbp
