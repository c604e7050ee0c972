// Function Drift of Algorithm 1 by thresholds.
//
// Drift bisects log2(lambda) over the bracket [hi 2^-40, hi], hi = 8 (max D - min D), in 12 steps: it tests
// lambda at points of the grid lambda_j = hi 2^(40 (j / 4096 - 1)), j = 1 .. 4095, and ends in a cell
// (J, J + 1] whose upper end gives the symbols.  A sweep over M candidates for every value and each of 13
// multipliers was two thirds of the encoder's instructions.  The same J follows from the values' thresholds:
// as lambda grows a value steps from its nearest level towards the central one, and the step over the edge
// between an outer level and the next inner one happens at
//     lambda = 2 s^2 y,   y = x / (r_outer - r_inner),   x = distance from the edge's midpoint in level units.
// So the code length at lambda is the all-central length plus the R differences of the edges with
// 2 s^2 y > lambda, and J is the cell of the largest y at which the sum over the edges not below it exceeds what
// the budget leaves: an order statistic, found by interpolation on y (about four sums over 4 values per lane, then one or two maxima).
//
// The records are defined by the binary32 costs fma(lambda, r_m, D_m), lowest index among equal ones, at the
// rounded lambdas.  Rounding moves a step by E level units in x and by a relative wA (both bounded below).  The
// outcome is the sweeps' when J's threshold is farther than that from both ends of its cell, and every other
// edge from lambda_{J+1}: the assignments tested at other grid points only have to stay over or within the
// budget, which they do because an edge taken (not taken) well before (after) lambda_{J+1} is so at every
// larger (smaller) lambda.  Otherwise (about one stream in 200) the exact sweeps run.
#pragma once
#include "dq_device.cuh"
#include "dq_internal.h"

namespace dqdrift {

using dqdev::kFullMask;

// Per-CTA copy of the table fields the encoder touches (a CTA encodes one tensor kind).
// With the paired-symbol variant the rANS alphabet is the M^2 pairs u = a M + b: enc and prk then hold the pair
// alphabet, r / R are not used.
struct EncTable {
    float r[DQ_MAX_LEVELS];
    uint32_t R[DQ_MAX_LEVELS];
    // Eq. rans Enc: {rcp, thr, bias, (2^p - f) << 5 | rsh}: floor(x / f) = umulhi(x, rcp) >> rsh, bias = c (+ 255 when
    // f = 1), thr = f << (sigma - 9) = f L: renormalise while the state is not below it
    uint4 enc[DQ_MAX_PAIRS];
    uint2 prk[DQ_MAX_PAIRS];       // pairs: {bits of r_u, ceil(65536 r_u) << 8 | u}
    uint4 edge[2][DQ_MAX_LEVELS / 2];   // thresholds, by side and edge: y = |a| x + y (binary32 bits), R difference
    float xm[2], inv_m[2], inv_max, rho; // DqDevTable
    uint32_t dR_few;
    int M, rec, mstar, budget_bits, has_mean, rotate;
    int early_exit, sigma;         // codec variants: Drift tries its end multiplier first; bits of final state (32 / 24)
    int pair;                      // paired symbols
    float pair_dr;                 // DqDevTable::pair_dr
    int fast;                      // DqDevTable::drift_fast
    uint32_t central;              // the all-central stream's four levels of a lane, one per byte
};

// Edge fields of a table into shared memory (threads 0 .. 15 of the CTA).
__device__ __forceinline__ void load_edges(EncTable& T, const DqDevTable& TK, const DqDevTable& TV, bool is_v) {
    const int i = threadIdx.x;
    if (i < DQ_MAX_LEVELS) {
        const int side = i >> 3, e = i & 7;
        T.edge[side][e] = make_uint4(__float_as_uint(is_v ? TV.edge_inv[side][e] : TK.edge_inv[side][e]),
                                     __float_as_uint(is_v ? TV.edge_off[side][e] : TK.edge_off[side][e]),
                                     is_v ? TV.edge_dR[side][e] : TK.edge_dR[side][e], 0u);
    }
    if (i < 2) { T.xm[i] = is_v ? TV.edge_xm[i] : TK.edge_xm[i]; T.inv_m[i] = is_v ? TV.edge_inv_m[i] : TK.edge_inv_m[i]; }
    if (i == 0) {
        T.rho = is_v ? TV.edge_rho : TK.edge_rho; T.inv_max = is_v ? TV.edge_inv_max : TK.edge_inv_max;
        T.dR_few = is_v ? TV.edge_few : TK.edge_few;
        T.fast = is_v ? TV.drift_fast : TK.drift_fast;
    }
}

// The stream as seen by its group of lanes: a warp holds it alone, 4 values per lane.
struct WarpGroup {
    int n;            // values of the stream
    __device__ __forceinline__ uint32_t add(uint32_t v) const { return __reduce_add_sync(kFullMask, v); }
    __device__ __forceinline__ uint32_t max(uint32_t v) const { return __reduce_max_sync(kFullMask, v); }
    __device__ __forceinline__ uint32_t min(uint32_t v) const { return __reduce_min_sync(kFullMask, v); }
    __device__ __forceinline__ bool any(bool p) const { return __any_sync(kFullMask, p); }
};

__device__ __forceinline__ float lg2_approx(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float exp2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One predicated instruction behind each comparison (the compiler's select form takes one more).
__device__ __forceinline__ void add_if_greater(uint32_t& sum, float x, float bound, uint32_t v) {
    asm("{.reg .pred p; setp.gt.f32 p, %1, %2; @p add.u32 %0, %0, %3;}" : "+r"(sum) : "f"(x), "f"(bound), "r"(v));
}
__device__ __forceinline__ void add_if_not_less(uint32_t& sum, float x, float bound, uint32_t v) {
    asm("{.reg .pred p; setp.ge.f32 p, %1, %2; @p add.u32 %0, %0, %3;}" : "+r"(sum) : "f"(x), "f"(bound), "r"(v));
}
__device__ __forceinline__ void fadd_if_greater(float& sum, float x, float bound, float v) {
    asm("{.reg .pred p; setp.gt.f32 p, %1, %2; @p add.f32 %0, %0, %3;}" : "+f"(sum) : "f"(x), "f"(bound), "f"(v));
}
__device__ __forceinline__ void max_if_less(float& m, float x, float bound) {
    asm("{.reg .pred p; setp.lt.f32 p, %1, %2; @p max.f32 %0, %0, %1;}" : "+f"(m) : "f"(x), "f"(bound));
}

// Symbols (one per byte) of Drift on the grid (s, o) for a stream whose extreme values are zmin and zmax, or false when some
// decision is within rounding of a tie (the caller then runs the exact sweeps).  Uniform over the group.
template <int M, class Group>
__device__ __forceinline__ bool drift_thresholds(const EncTable& T, const Group& grp, const float (&z)[4], float s, float o,
                                                 float zmin, float zmax, uint32_t& sym) {
    constexpr int kC = (M - 1) / 2, kLow = kC, kHigh = M - 1 - kC;   // central level; edges below / above it
    constexpr float kG = 102.4f;                                     // grid cells per octave of lambda
    if (!(s > 0x1p-30f && s < 0x1p40f)) return false;
    const float inv = rcp_approx(s), shift = -o * inv;
    const float vmax = fmaf(zmax, inv, shift), vmin = fmaf(zmin, inv, shift);
    const float reach = fmaxf(vmax, (float)(M - 1) - vmin);          // largest |z - level| / s
    const float mag = fmaxf(fmaxf(fabsf(zmin), fabsf(zmax)), fmaxf(fabsf(o), fabsf(o + (float)(M - 1) * s))) * inv;
    if (!(mag < 1024.f && reach < 1024.f)) return false;
    // rounding of a[] and y, and of the two compared costs, in units of 2^-24 (d1 + d2 <= max(1, 2 x), lambda = 2 s^2 y)
    const float E = 1.5f * 0x1p-24f * (2.f * mag + 4.f * reach + (float)M);

    float a[4], y[4][kHigh];
    uint32_t dR[4][kHigh];
    uint32_t w = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        a[i] = fmaf(z[i], inv, shift) - (float)kC;
        const int up = a[i] >= 0.f ? 1 : 0;
#pragma unroll
        for (int e = 0; e < kHigh; ++e) {
            const uint4 ed = T.edge[up][e];
            y[i][e] = fmaf(fabsf(a[i]), __uint_as_float(ed.x), __uint_as_float(ed.y));
            dR[i][e] = ed.z;
            add_if_greater(w, y[i][e], 0.f, dR[i][e]);
        }
    }
    const uint32_t budget = (uint32_t)T.budget_bits << 16, base = (uint32_t)grp.n * T.R[kC];
    if (base > budget) return false;
    const uint32_t cap = budget - base;
    uint32_t Wa = grp.add(w);
    // Where the nearest levels fit, every test passes and lambda ends at lambda_1, too small to move any value.
    float yf = 0.f, band = E * T.inv_max;
    bool tie = false;
    if (Wa > cap) {
        if (!T.fast) return false;
        if (T.fast == 2) {   // the outermost two edges of a side merge from xm on
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int up = a[i] >= 0.f ? 1 : 0, ne = up ? kHigh : kLow;
                const float xo = fabsf(a[i]) - ((float)ne - 0.5f);
                if (xo >= T.xm[up]) {
#pragma unroll
                    for (int e = 0; e < kHigh; ++e)
                        if (e == ne - 1 || e == ne - 2) y[i][e] = fmaf(2.f, xo, 1.f) * T.inv_m[up];
                }
            }
        }
        float dmin = 1e30f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float d = fabsf(a[i]);
#pragma unroll
            for (int e = 0; e < kHigh; ++e) fadd_if_greater(d, y[i][e], 0.f, -1.f);
            dmin = fminf(dmin, fabsf(d));
        }
        dmin = __uint_as_float(grp.min(__float_as_uint(dmin)));
        const float Dn = fmaf(reach, reach, -dmin * dmin);               // (max D - min D) / s^2

        // Bracket [ya, yb]: the sum over y > ya exceeds cap, the one over y > yb does not.  Interpolated, leaning towards
        // ya (the sums are convex), until few edges are between: 4.3 sums on average, halving takes 7.
        float ya = 0.f, yb = (fmaxf(vmax - (float)kC, (float)kC - vmin) - 0.49f) * T.inv_max;
        uint32_t Wb = 0;
#pragma unroll 1
        for (int it = 0; it < 14 && Wa - Wb > T.dR_few; ++it) {
            const float t = 0.85f * (float)(int)(Wa - cap) * rcp_approx((float)(int)(Wa - Wb));
            const float ym = fmaf(yb - ya, fminf(fmaxf(t, 0.05f), 0.95f), ya);
            w = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < kHigh; ++e) add_if_greater(w, y[i][e], ym, dR[i][e]);
            w = grp.add(w);
            const bool over = w > cap;
            ya = over ? ym : ya; Wa = over ? w : Wa;
            yb = over ? yb : ym; Wb = over ? Wb : w;
        }
        // then down from yb, one edge at a time
        float yc = __uint_as_float(__float_as_uint(yb) + 1u);
#pragma unroll 1
        for (int it = 0;; ++it) {
            float m = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < kHigh; ++e) max_if_less(m, y[i][e], yc);
            yc = __uint_as_float(grp.max(__float_as_uint(m)));
            if (it == 40 || !(yc > 0.f)) return false;
            w = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < kHigh; ++e) add_if_not_less(w, y[i][e], yc, dR[i][e]);
            if (grp.add(w) > cap) break;
        }
        // yc again, from the rounded level positions that the costs use: E becomes 3 units of 2^-24.  Only for a single,
        // unmerged edge; it leaves y[][] here, being taken at lambda_{J+1} by construction.
        float zc = 0.f, code = 0.f;   // its value, and (edge + 1) with the sign of its side
        uint32_t equal = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int e = 0; e < kHigh; ++e) {
                const bool is = y[i][e] == yc;
                zc = is ? z[i] : zc;
                code = is ? copysignf((float)(e + 1), a[i]) : code;
                y[i][e] = is ? 0.f : y[i][e];
                equal += is ? 1u : 0u;
            }
        float yr = 0.f;
        if (equal) {
            const float dir = copysignf(1.f, code), outer = (float)kC + code;
            const float di = zc - fmaf(outer - dir, s, o), dq = zc - fmaf(outer, s, o);
            yr = fmaxf(((di - dq) * inv) * ((di + dq) * inv) * 0.5f * __uint_as_float(T.edge[dir > 0.f ? 1 : 0][(int)fabsf(code) - 1].x), 0.f);
        }
        yr = __uint_as_float(grp.max(__float_as_uint(yr)));
        const bool refined = grp.add(equal) == 1u && T.fast == 1 && yr > 0.f;
        // cell of yc (grid units from 3072 on: less to round), lambda_{J+1} / (2 s^2)
        const float wA = 4e-4f + 1.5f * 148.f * 0x1p-24f * (2.f * mag + 4.f * reach + 2.f * T.rho);
        const float lgD = log2f(Dn) - 8.f, ryc = rcp_approx(yc);
        const float u = kG * (lg2_approx(refined ? yr : yc) - lgD);
        const float wc = fmaf(148.f * T.inv_max * (refined ? 4.5f * 0x1p-24f : E), ryc, wA);
        const float J = floorf(u - wc);
        tie = floorf(u + wc) != J || J < -3070.f || J > 1020.f;
        yf = exp2_approx(fmaf(J + 1.f, 1.f / kG, lgD));
        if (refined && u - fmaf(148.f * band, 2.f * ryc, wA) < J) {   // the unrefined edges next to yc may be below lambda_J
            const float yJ = exp2_approx(fmaf(J, 1.f / kG, lgD)), bJ = fmaf(yJ, wA * (1.f / 148.f), band);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < kHigh; ++e) tie |= fabsf(y[i][e] - yJ) <= bJ;
        }
        band = fmaf(yf, wA * (1.f / 148.f), band);
    }
    uint32_t lev[4];
    const float E2 = fmaf(yf, 0x1p-18f, E);   // cost ties of the two central levels of an even table (equal r)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool up = a[i] >= 0.f;
        const float unit = up ? 1.f : -1.f;
        float m = 8388608.f + (float)kC;   // the low byte of its bits is the level
#pragma unroll
        for (int e = 0; e < kHigh; ++e) {
            fadd_if_greater(m, y[i][e], yf, unit);
            tie |= fabsf(y[i][e] - yf) <= band;
        }
        if (M % 2 == 0) tie |= up && fabsf(a[i] - 0.5f) <= E2;
        lev[i] = __float_as_uint(m);
    }
    sym = __byte_perm(__byte_perm(lev[0], lev[1], 0x0040), __byte_perm(lev[2], lev[3], 0x0040), 0x5410);
    return !grp.any(tie);
}

}  // namespace dqdrift
