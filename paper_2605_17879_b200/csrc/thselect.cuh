// One thread per series: counting / keeping cell operation and the selection among the kept values of a
// thread's shared-memory column (the same instruction stream in every lane of a warp).
// What bounds both is the half-rate pipe of compares and integer operations, so a value below a limit is counted in
// floating point: (limit - x) times a power of two that makes any difference at least 1, saturated to [0, 1] (one fused
// operation, whose single rounding cannot change a sign), and added.  131 072 series of 200 steps take 38 us instead of
// the 41 of compares and integer keys, and leave that pipe to the kernels beside them: passes of 16 384 ranks x 8 x 200
// with overlapped evaluations 426 us instead of 437, of 24 000 x 8 x 100 169 instead of 177.
#pragma once
#include <math_constants.h>

#include "common.cuh"

namespace guard {

// The values to keep: |x - c| <= h, as rounded.  usable: h is positive and neither value so near the ends of the range of
// floats that a power of two below would not be a normal number or a sum overflow.
struct ThRange {
    float c, h;
    float ns, nhs;     // -S and -h S: the saturated product of a value below the interval
};
__device__ __forceinline__ float pow2_of(const int e) { return __int_as_float((e + 127) << 23); }      // -126 <= e <= 127
__device__ __forceinline__ int exponent_of(const float x) { return (int)((__float_as_uint(x) >> 23) & 255u) - 127; }   // of normal numbers
__device__ __forceinline__ bool th_usable(const float c, const float h) { return h > 1.0e-29f && h < 1.0e37f && fabsf(c) < 1.0e37f; }
__device__ __forceinline__ ThRange th_range(const float c, const float h, const bool usable) {
    ThRange r;
    r.c = c;
    r.h = usable ? h : -1.0f;      // keeps nothing
    const float s = usable ? pow2_of(30 - exponent_of(h)) : 0.0f;   // (a difference is at least h 2^-25)
    r.ns = -s;
    r.nhs = -h * s;
    return r;
}

// cnt += (x - c < -h); if (|x - c| <= h) { if (addr < lim) shared[addr] = x; addr += 4; }
__device__ __forceinline__ void th_cell(const float x, const ThRange &r, const uint32_t lim, float &cnt, uint32_t &addr) {
    asm volatile(
        "{\n\t.reg .pred q, s;\n\t.reg .f32 d, a, b;\n\t"
        "sub.rn.f32 d, %2, %3;\n\t"
        "fma.rn.sat.f32 b, d, %5, %6;\n\t"
        "abs.f32 a, d;\n\t"
        "setp.le.f32 q, a, %4;\n\t"
        "setp.lt.and.u32 s, %1, %7, q;\n\t"
        "add.rn.f32 %0, %0, b;\n\t"
        "@s st.shared.f32 [%1], %2;\n\t"
        "@q add.u32 %1, %1, 4;\n\t}"
        : "+f"(cnt), "+r"(addr)
        : "f"(x), "f"(r.c), "f"(r.h), "f"(r.ns), "f"(r.nhs), "r"(lim)
        : "memory");
}
__device__ __forceinline__ float4 th_lds4(const uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void th_sts4(const uint32_t addr, const float4 v) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
// cnt += x < p, for ps = p S, ns = -S
__device__ __forceinline__ void th_below(const float x, const float ns, const float ps, float &cnt) {
    float b;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(b) : "f"(x), "f"(ns), "f"(ps));
    cnt += b;
}

// The values of ranks t - 1 (vb) and t (vu) among the nk values kept by r in the column at shared-memory address kbase
// (SLOTS words, 16-byte aligned).  Lanes with ok == false take part without a result; ok turns false if the selection
// does not converge, or if it ends on a zero, whose sign is not looked at here.  All 32 lanes of the warp call this together.
template <int SLOTS, int MAXPASS>
__device__ __forceinline__ void th_select_pair(const uint32_t kbase, const int nk, bool &ok, const int t, const ThRange &r, float &vb, float &vu) {
    const int nkmax = (int)__reduce_max_sync(0xFFFFFFFFu, ok ? (uint32_t)nk : 0u);
    if (nkmax > 0) {
        const int nkr = (nkmax + 3) & ~3;   // <= SLOTS (a multiple of 4)
        const int nkmin = (int)__reduce_min_sync(0xFFFFFFFFu, ok ? (uint32_t)nk : (uint32_t)SLOTS);
        for (int j = nkmin & ~3; j < nkr; j += 4) {   // slots without a value lie above everything
            float4 v = th_lds4(kbase + 4u * j);
            v.x = j + 0 < nk ? v.x : CUDART_INF_F;
            v.y = j + 1 < nk ? v.y : CUDART_INF_F;
            v.z = j + 2 < nk ? v.z : CUDART_INF_F;
            v.w = j + 3 < nk ? v.w : CUDART_INF_F;
            th_sts4(kbase + 4u * j, v);
        }
        // No kept value lies outside [pl, ph): |x - c| as rounded is within 2^-24 of itself and of |c|.
        const float top = fabsf(r.c) + r.h, eps = top * pow2_of(-21);
        float pl = r.c - r.h - eps, ph = r.c + r.h + eps, pv = pl;
        // Pivots are kept so far from zero that the power of two lifts their difference from any other value (2^-24 of
        // the pivot at least) to 1: 2^-35 of the largest value, as long as that power is a number.
        const int lift = min(60 - exponent_of(top), 127);
        const float near0 = ok ? pow2_of(25 - lift) : 1.0f, ns = ok ? -pow2_of(lift) : 0.0f;
        // The pivot moves inside a bracket (pl, ph) with below(pl) = al <= t - 2 and below(ph) = ah >= t + 2.
        int al = 0, ah = nk, bsave = 0;
        int done = 0;                 // 1: pv has bsave in {t - 1, t, t + 1} values below it, 2: both ranks equal pl
        if (!ok || t <= 1) { done = 1; bsave = 0; }
        else if (t >= nk - 1) { done = 1; pv = ph; bsave = nk; }
        for (int pass = 0; pass < MAXPASS; ++pass) {
            if (__all_sync(0xFFFFFFFFu, done != 0)) break;
            if (!done) {
                // aim between the ends in proportion to the missing count, every third time at the middle
                const float fr = pass % 3 == 2 ? 0.5f : __fdividef((float)(t - al), (float)(ah - al));
                pv = pl + (ph - pl) * fr;
                if (!(pv > pl && pv < ph)) pv = 0.5f * (pl + ph);
                if (!(pv > pl && pv < ph)) done = 2;         // neighbours: every value between them is pl
                else if (fabsf(pv) < near0) pv = pv < 0.0f ? -near0 : near0;
            }
            // the loads of a third of the column are issued before their compares
            const float ps = -ns * pv;
            float b0 = 0.0f, b1 = 0.0f;
#pragma unroll
            for (int j0 = 0; j0 < SLOTS / 4; j0 += 5) {
                float4 kv4[5];
#pragma unroll
                for (int j = 0; j < 5; ++j)
                    if (4 * (j0 + j) < nkr) kv4[j] = th_lds4(kbase + 16u * (j0 + j));
#pragma unroll
                for (int j = 0; j < 5; ++j)
                    if (4 * (j0 + j) < nkr) {
                        th_below(kv4[j].x, ns, ps, b0);
                        th_below(kv4[j].y, ns, ps, b1);
                        th_below(kv4[j].z, ns, ps, b0);
                        th_below(kv4[j].w, ns, ps, b1);
                    }
            }
            const int below = (int)(b0 + b1);
            if (!done) {
                if (below >= t - 1 && below <= t + 1) { done = 1; bsave = below; }
                else if (below < t) { pl = fmaxf(pl, pv); al = below; }
                else { ph = fminf(ph, pv); ah = below; }
            }
        }
        if (ok && !done) ok = false;
        // the two largest values below the pivot (b1 >= b2), the two smallest not below it (u1 <= u2)
        float b1 = -CUDART_INF_F, b2 = -CUDART_INF_F, u1 = CUDART_INF_F, u2 = CUDART_INF_F;
        for (int j = 0; j < nkr; j += 4) {
            const float4 v4 = th_lds4(kbase + 4u * j);
            const float v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool lt = v[u] < pv;
                const float lo_v = lt ? v[u] : -CUDART_INF_F, hi_v = lt ? CUDART_INF_F : v[u];   // neutral on the other side
                b2 = fmaxf(b2, fminf(b1, lo_v));
                b1 = fmaxf(b1, lo_v);
                u2 = fminf(u2, fmaxf(u1, hi_v));
                u1 = fminf(u1, hi_v);
            }
        }
        vb = b1; vu = u1;                                // bsave == t
        if (bsave == t + 1) { vb = b2; vu = b1; }
        if (bsave == t - 1) { vb = u1; vu = u2; }
        if (done == 2) { vb = pl; vu = pl; }
        if (vb == 0.0f || vu == 0.0f) ok = false;
    }
}

}  // namespace guard
