// Tables of the fixed-point FP64 operators (fx.cuh): the folded operators of
// every degree as scaled 64-bit integers, at the offsets of fold_layout.h,
// and the powers of two that go with them.
#pragma once

#include "fold_layout.h"

namespace fem {

struct FxEntry {
    int h, l;  // balanced halves: C = h 2^32 + l
};

struct FxDegree {
    int tau[kFoldCount];  // entry = round(A 2^(64 - tau)) (folded)
    int wn[kMaxQ];        // GLL weights: w < 2^wn <= 2 w
    int wm[kMaxQ];        // Gauss weights
};

struct FxTables {
    FxEntry c[kFoldTotal];
    FxDegree d[kMaxN + 1];
};

// Bits of a value (|x| < 2^bits) at the input of a contraction, and of its
// output: 61 and 60, as the sums of cross products of every row allow
// (fx_tables() checks them, for BP1.0 and BP3.0 with 8 % for what three
// contractions in a row may add).  BP3.5's first contraction takes one bit
// less than its second.
__host__ __device__ constexpr int fx_bits35(int N) { return N >= 10 ? 60 : 61; }
constexpr int kFxBits30 = 60;
// Bits of the field of BP1.0 and BP3.0: their interpolations are scaled by one
// half, and a row's absolute sum is up to 2.43 (N = 15), so that from N = 7 on
// (1.97) three in a row may grow by 1.8; at N = 15 the cross products need one
// bit more.
__host__ __device__ constexpr int fx_qbits30(int N) { return N == 15 ? 58 : N >= 7 ? 59 : 60; }

// Built once; aborts nothing: a table that breaks a bound is reported by
// fx_table_violations().
const FxTables &fx_tables();
int fx_table_violations();

}  // namespace fem
