// Bins of a value range from two chained multiply-adds, the first saturated to [0, 1].
#pragma once
#include <cfloat>

#include "common.cuh"

namespace guard {

struct BinMap {
    float scale, off, span;   // sat(x scale + off); the width that the inner bins hold
};
// Takes lo to the middle of bin 1 and hi to that of bin TOP - 1, of TOP + 1 bins centred on multiples of 1 / TOP.  The offset
// is rounded to 2^-24 of lo scale, which moves all bins by at most 2^-24 |lo|, a step between floats: the range is a step or
// two wider than asked for at either end, so that a range of a few steps, or of a single value, holds it whatever the rounding.
// (Without: constant series of 2e6 missed their own value three times over, 65 536 of 64 steps 35.0 us, so 21.8; 8 192 whose
// values scatter over some twenty floats about 2e6, 1 000 steps, missed every range: 190 us, so 28.8.)
template <int TOP>
__device__ __forceinline__ BinMap bin_map(const float lo, const float hi) {
    constexpr float kIn = (float)(TOP - 2) / (float)TOP, kFirst = 1.0f / (float)TOP, kStep = 1.1920928955078125e-7f;   // 2^-23
    const float e = fmaxf(fabsf(lo), fabsf(hi)) * kStep;
    BinMap m;
    m.span = (hi - lo) + 2.0f * e;
    m.scale = fminf(kIn / m.span, 1.0e37f);
    m.off = __fmaf_rn(-fmaxf(lo - e, -FLT_MAX), m.scale, kFirst);
    return m;
}

}  // namespace guard
