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
// output: 61, and 60 where a sum of cross products of 61-bit values could
// overflow (fx_tables() checks the sums of every row).  BP3.5 contracts lines
// of n points (its first contraction takes 60 bits), BP1.0 and BP3.0 up to m.
__host__ __device__ constexpr int fx_bits35(int N) { return N >= 10 ? 60 : 61; }
__host__ __device__ constexpr int fx_bits30(int N) { return N >= 6 ? 60 : 61; }

// Built once; aborts nothing: a table that breaks a bound is reported by
// fx_table_violations().
const FxTables &fx_tables();
int fx_table_violations();

}  // namespace fem
