// elim.hpp -- the eliminated walk: a Gray walk over the outer columns whose
// every step sums the terms of all 2^k settings of k low columns at once.
//
// The Nijenhuis-Wilf sum (Eq. 2, Sec. II) runs over the subsets S of the
// first n-1 columns, sum_S (-1)^|S| prod_i x_i(S).  Row i's factor depends only
// on the columns that touch row i, so for sparse matrices the sum over the low
// columns distributes over the product: with the outer columns fixed, each row
// is a table over the settings of the low columns that touch it (x_i plus a
// subset of their entries), and a low column is summed out by multiplying the
// tables that mention it and subtracting the column-on half from the
// column-off half.  Every Gray index of the range is still accounted for, and
// every term is the same product of n numbers; products and sums shared
// between terms are formed once.  The paired and two-state chains (core.cuh)
// are the k = 1 case; Sec. V's reuse of a global product is the case of rows
// that no low column touches.
#pragma once

#include <algorithm>
#include <cstdint>
#include <memory_resource>
#include <string>
#include <vector>

#include "host.hpp"

namespace perm {

// One operation of a step's program.  Values are numbered 0..n-1 (x of the
// original rows) and then one per operation.
enum ElimKind : uint8_t {
    kElimAdd = 0,      // v = value a + entry (row b, column c)
    kElimMul = 1,      // v = a * b
    kElimMulSub = 2,   // v = c - a * b
    kElimSub = 3       // v = a - b
};

struct ElimOp {
    uint8_t kind;
    int32_t a, b, c;
};

// The same program by whole tables (the precompiled kernels' form).  Tables are
// numbered; entry e of a table belongs to the setting e of its scope's columns,
// lowest bit the column summed out first.
struct ElimTable {
    uint64_t scope;    // bit q: the q-th column summed out (elimination order)
    double bound;      // exact: a bound of every entry's magnitude
    int row;           // >= 0: single value x_row (scope empty)
};
enum ElimTableKind : uint8_t { kTabRow = 0, kTabMul = 1, kTabSum = 2, kTabSub = 3 };
struct ElimTableOp {
    uint8_t kind;
    int dst, a, b;     // row: a = row index
    int col;           // sum, sub: the column's place in the elimination order
};

// (`mem` is where a plan and its image keep their vectors: the heap, or the fixed
// memory of the allocation-free call.)
struct ElimPlan {
    explicit ElimPlan(std::pmr::memory_resource *mem = std::pmr::new_delete_resource())
        : ops(mem), bound(mem), tables(mem), tops(mem), factors(mem) {}
    int n = 0, k = 0, h = 0;          // k low columns summed out, h outer columns walked
    int low[kNMax] = {};              // low columns in elimination order (original indices)
    int outer[kNMax] = {};            // outer column at Gray position p (original index)
    int last = 0;                     // the column that never flips
    int exp2[kNMax] = {};             // FP64: row i is walked as x_i 2^-exp2[i] (elim_row_bits)
    int scale = 0;                    // FP64: sum of exp2: the walk's sum times 2^scale is the true one
    std::pmr::vector<ElimOp> ops;
    int result = 0;                   // the value that holds the step's signed sum
    std::pmr::vector<double> bound;        // exact: a bound of each value's magnitude (n + ops entries)
    std::pmr::vector<ElimTable> tables;    // 0..n-1: x
    std::pmr::vector<ElimTableOp> tops;
    std::pmr::vector<int> factors;         // the step's sum is the product of these single values
    double table_ops = 0.0;           // operations of the table program
    double ops_per_step = 0.0;        // counted operations per Gray step, flips and accumulation included
};

// Stable, in place (std::stable_sort takes its scratch from the heap).
template <class It, class Less>
void insertion_sort(It b, It e, Less less) {
    for (It i = b; i != e; ++i)
        for (It j = i; j != b && less(*j, *(j - 1)); --j) std::swap(*j, *(j - 1));
}

struct ElimLimits {
    int max_width = 5;                // tables of at most 2^max_width entries while a column is summed out
    int max_ops = 1200;               // operations of a step's program
    double full_blocks = 32768.0;     // outer steps that fill the GPU: fewer take as long as these
    int candidates = kNMax;           // low columns tried per round of the search
    bool allow_none = false;          // k = 0 (a full product per step) is a plan too
    bool tables_only = false;         // write the program by tables only
};

// Picks the low columns among the first `free_cols` positions of col_order
// (over which the walked range runs in full) and writes the step's program.
// range_log2: log2 of the number of Gray indices walked.  False when no
// column is worth summing out.
bool elim_plan(const Matrix &m, const int *col_order, int free_cols, double range_log2, const ElimLimits &lim,
               ElimPlan &out);

// FP64 rows are scaled by powers of two (exactly) to |x_i| <= 2^bits, so that a
// product of n of them, summed over 2^(k+3) terms, does not leave FP32's range (the
// sum of |terms|), whatever the rows' own magnitudes; the first rows take what the
// division leaves over.
inline int elim_row_bits(int n, int k, int row) {
    const int b = std::max(0, std::min(8, (120 - k) / n));
    return b < 8 && row < 120 - k - b * n ? b + 1 : b;
}

// Whether the magnitudes of FP64 terms, multiplied in FP32 in the program's order,
// give the sum of |terms| of [g_lo, g_hi).  A product of few rows underflows long
// before the whole term would (four pairs of rows that cancel to 2^-52 of each other:
// terms of 2^-208 of the largest possible one, their sum came out as 0 at n = 28),
// so the sum must stay above what the program's underflows can lose.  It is bounded
// by terms of the range, or estimated from sampled ones; true where nothing can
// underflow.
bool elim_magnitudes_hold(const Matrix &m, const ElimPlan &E, const int *col_order, int free_cols, uint64_t g_lo,
                          uint64_t g_hi);

// The CUDA C++ of the generated kernel (limbs 0: FP64, else the exact ring).
std::string elim_source(const Matrix &m, const ElimPlan &E, int limbs, bool want_abs);

}  // namespace perm
