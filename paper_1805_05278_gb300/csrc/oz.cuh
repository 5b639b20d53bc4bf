// Digit-split products (oz_gemm.cu): the pieces a fused caller builds from.
#pragma once

#include "common.cuh"

namespace gbqr {

constexpr int kOzTileA = 128, kOzTileB = 64;   // rows of a digit tile of the M and N side of a product
constexpr int kOzOps = 4;            // operands or problems passed by value
constexpr int kOzItemsPerCta = 4;
constexpr int kOzMaxSplits = 65535;
constexpr int64_t kOzMaxRows = (int64_t)kOzMaxSplits * 512;   // longest K of a product that sums integers of 512 k each

// One operand to split: R rows of K entries each, from the columns (by_row ==
// 0: row r is column r of X) or the rows of the column-major X.
template <class Real>
struct OzOperand {
    const Real *X; int64_t ld;
    int64_t R, K;
    int mask, by_row;
    int unit;                     // MASK_UNIT_LOWER: ones on the diagonal (0: zeros, the product adds them apart)
    uint8_t *dst; int KT, rt;     // tiles of rt rows x 32 k, KT along k
    int *exps;                    // per operand row: |x| < 2^exps
    unsigned first;               // first CTA working on it
    const int *skip;              // non-null: nothing to do while *skip != 0
    const int *kexp; int ksign;   // entries of index k scaled by 2^(ksign kexp[k]) first
};
template <class Real>
struct OzSliceArgs {
    OzOperand<Real> op[kOzOps];
    const OzOperand<Real> *list;  // non-null: n operands in device memory instead
    int n;
};

// One product from digits: C = beta C + alpha A B^T (rows of A and B over k).
template <class Real>
struct OzProblem {
    const uint8_t *a, *b;
    const int *ea, *eb;
    int M, N, KT;
    int b128;                     // B in tiles of 128 rows too (X^T X)
    int kt_per, S;                // K tiles per item, splits
    int clip, clipB;              // triangular operands: see oz_item
    int first;                    // first work item
    long long *partial;           // non-null: [z][M x N] integer partials instead of C
    Real *C; int64_t ldc;
    double *Cd;                   // reduce: FP64 result instead of C (ld ldc)
    Real alpha, beta;
    const Real *add; int64_t ldadd; int add_rows;   // + add(i, j) for i < add_rows (unit diagonal of op(A))
    const int *skip;
    uint8_t *qdst; int *qexp;     // requant: digits of the sums (and the sums in C, if not null)
};
template <class Real>
struct OzMmaArgs {
    OzProblem<Real> prob[kOzOps];
    const OzProblem<Real> *list;  // non-null: n problems in device memory instead
    int n, items;
    int *err;
};

int oz_ktiles(int64_t K);
int oz_items(int M, int N, int S);
// K tiles of one item: what its 64-bit integer sums hold for any digits
// (leading products of 2^14, FP64 in units of 2^-40, FP32 of 2^-24).
template <class Real> constexpr int oz_max_ktiles() { return sizeof(Real) == 8 ? 16 : 64; }
constexpr int kOzDigits64 = 7, kOzDigits32 = 4;   // digits of an operand of FP64 and FP32 products
template <class Real> constexpr int oz_digits() { return sizeof(Real) == 8 ? kOzDigits64 : kOzDigits32; }
// bytes of an operand's digits and exponents, 256-aligned
size_t oz_digit_bytes(int D, int64_t R, int64_t K, int rt);
template <class Src>
OzOperand<Src> oz_operand(int D, const Src *X, int64_t ld, int64_t R, int64_t K, bool by_row, int mask, int rt,
                          void *mem);
template <class Src> unsigned oz_slice_blocks(const OzOperand<Src> &o, bool tall);
template <class Src> gbqr_status oz_slice(const Exec &ex, int D, OzOperand<Src> *ops, int n);
template <class Src>
gbqr_status oz_slice_launch(const Exec &ex, int D, const OzSliceArgs<Src> &args, unsigned blocks, bool tall, double elems);
template <class Real, class SA, class SB> OzProblem<Real> oz_problem(const OzOperand<SA> &a, const OzOperand<SB> &b);
template <class Real> bool oz_choose_split(OzProblem<Real> &p, int num_sms, size_t part_bytes, bool force_partial);
template <class Real> gbqr_status oz_mma_launch(const Exec &ex, const OzMmaArgs<Real> &args, double elems);
template <class Real> gbqr_status oz_reduce_launch(const Exec &ex, const OzMmaArgs<Real> &args, size_t largest);
template <class Real> gbqr_status oz_requant_launch(const Exec &ex, const OzMmaArgs<Real> &args, int widest);

}  // namespace gbqr
