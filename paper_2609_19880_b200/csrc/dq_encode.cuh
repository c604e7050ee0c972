// Encoder code shared by the translation units of its kernels: tables, rotary embedding, Drift by sweeps, and steps
// 2-6 of Algorithm 1 for a stream held by one warp, 4 values per lane.  Compiled with -fmad=false: every
// floating-point operation that decides a record's bytes is a single IEEE operation in a fixed order.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "dq_device.cuh"
#include "dq_drift.cuh"
#include "dq_internal.h"

namespace dqenc {

constexpr unsigned kFull = dqdev::kFullMask;
constexpr int kN = DQ_HEAD_DIM;
constexpr uint32_t kL = 1u << 23;  // lower bound of the rANS state interval (sigma = 32; token-wide streams always)

using dqdev::bf16_bits_to_float;
using dqdev::warp_fwht128;  // per-head Hadamard rotation (Sec. 4.2), 4 values per lane
using dqdrift::EncTable;
using dqdrift::WarpGroup;

// Rotary position embedding of a head vector held 4 values per lane (element 4 lane + e), in
// binary32 with every product and sum rounded once.  DQ_ROPE_HALF pairs element j with j + 64
// (the partner sits in lane ^ 16), DQ_ROPE_PAIRS pairs 2j with 2j + 1 (same lane).
// c / s: this lane's cosines / sines, of angles 4 (lane & 15) .. + 3 (halves) or 2 lane, 2 lane + 1 (pairs).
__device__ __forceinline__ void warp_rope128(float (&v)[4], int lane, float4 c, float4 s, int style) {
    if (style == DQ_ROPE_HALF) {
        const float cc[4] = {c.x, c.y, c.z, c.w}, ss[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float other = __shfl_xor_sync(kFull, v[e], 16);
            // lanes 0-15 hold a: a cos - b sin; lanes 16-31 hold b: b cos + a sin
            const float mine = __fmul_rn(v[e], cc[e]), cross = __fmul_rn(other, ss[e]);
            v[e] = (lane < 16) ? __fsub_rn(mine, cross) : __fadd_rn(mine, cross);
        }
    } else {
        const float a0 = v[0], b0 = v[1], a1 = v[2], b1 = v[3];
        v[0] = __fsub_rn(__fmul_rn(a0, c.x), __fmul_rn(b0, s.x));
        v[1] = __fadd_rn(__fmul_rn(b0, c.x), __fmul_rn(a0, s.x));
        v[2] = __fsub_rn(__fmul_rn(a1, c.y), __fmul_rn(b1, s.y));
        v[3] = __fadd_rn(__fmul_rn(b1, c.y), __fmul_rn(a1, s.y));
    }
}
// The same with cs / sn: this position's 64 cosines / sines.
__device__ __forceinline__ void warp_rope128(float (&v)[4], int lane, const float* cs, const float* sn, int style) {
    float4 c, s;
    if (style == DQ_ROPE_HALF) {
        c = *reinterpret_cast<const float4*>(cs + 4 * (lane & 15));
        s = *reinterpret_cast<const float4*>(sn + 4 * (lane & 15));
    } else {
        const float2 c2 = *reinterpret_cast<const float2*>(cs + 2 * lane), s2 = *reinterpret_cast<const float2*>(sn + 2 * lane);
        c = make_float4(c2.x, c2.y, 0.f, 0.f);
        s = make_float4(s2.x, s2.y, 0.f, 0.f);
    }
    warp_rope128(v, lane, c, s, style);
}

// Table of one tensor kind into shared memory, by all threads of the CTA (at least 32).
__device__ __forceinline__ void load_enc_table(EncTable& T, const DqDevTable& TK, const DqDevTable& TV,
                                               const DqPairEnc& PK, const DqPairEnc& PV, bool is_v) {
    const int pair = is_v ? TV.pair : TK.pair, sigma = is_v ? TV.sigma : TK.sigma;
    dqdrift::load_edges(T, TK, TV, is_v);
    if (threadIdx.x < DQ_MAX_LEVELS) {
        const int i = threadIdx.x;
        T.r[i] = is_v ? TV.r[i] : TK.r[i];
        T.R[i] = is_v ? TV.R[i] : TK.R[i];
    }
    for (int i = threadIdx.x; i < (pair ? DQ_MAX_PAIRS : DQ_MAX_LEVELS); i += blockDim.x) {
        uint32_t rcp, aux;
        if (pair) {
            rcp = is_v ? PV.enc_rcp[i] : PK.enc_rcp[i];
            aux = is_v ? PV.enc_aux[i] : PK.enc_aux[i];
            T.prk[i] = make_uint2(__float_as_uint(is_v ? PV.r[i] : PK.r[i]), ((is_v ? PV.R[i] : PK.R[i]) << 8) | (uint32_t)i);
        } else {
            rcp = is_v ? TV.enc_rcp[i] : TK.enc_rcp[i];
            aux = is_v ? TV.enc_aux[i] : TK.enc_aux[i];
        }
        const uint32_t cmpl = (aux >> 10) & 511u;
        T.enc[i] = make_uint4(rcp, (256u - cmpl) << (sigma - 9), aux & 1023u, cmpl << 5 | aux >> 19);
    }
    if (threadIdx.x == 0) {
        T.M = is_v ? TV.M : TK.M; T.rec = is_v ? TV.rec : TK.rec; T.mstar = is_v ? TV.mstar : TK.mstar;
        T.budget_bits = is_v ? TV.budget_bits : TK.budget_bits;
        T.has_mean = is_v ? TV.has_mean : TK.has_mean; T.rotate = is_v ? TV.rotate : TK.rotate;
        T.early_exit = is_v ? TV.early_exit : TK.early_exit; T.sigma = sigma;
        T.pair = pair;
        T.pair_dr = is_v ? TV.pair_dr : TK.pair_dr;
        const uint32_t ms = (uint32_t)T.mstar, us = (uint32_t)(is_v ? TV.ustar : TK.ustar), M = (uint32_t)T.M;
        T.central = pair ? (us / M) * 0x00010001u + (us % M) * 0x01000100u : ms * 0x01010101u;
    }
}

// Function Drift of Algorithm 1 on a stream held 4 values per lane.  The bisection of
// log2(lambda) over T = 12 steps is carried out as the geometric mean of the bracket
// [hi * 2^-40, hi], hi = 8 (max D - min D); the code length is an integer sum of
// ceil(65536 r_m), so the feasibility test does not depend on summation order.
// Returns the length of the final assignment (the argmin at the bracket's upper end).
// These sweeps define the result; dq_drift.cuh finds it without them for all but a few streams.
// M is a template parameter so that the M candidate costs of a value are independent
// instructions and the table sits in registers; the minimum keeps the lowest index among equal
// costs, exactly as an ascending scan with a strict comparison does.
template <int M>
static __device__ __noinline__ uint2 drift_sweeps(const EncTable& T, float z0, float z1, float z2, float z3, float s, float o) {
    const float z[4] = {z0, z1, z2, z3};
    float tm[M], rm[M];
    uint32_t Km[M];   // ceil(65536 r_m) << 8 | m: the minimum tree carries one word for length and index
#pragma unroll
    for (int m = 0; m < M; ++m) {
        tm[m] = __fmaf_rn((float)m, s, o);
        rm[m] = T.r[m];
        Km[m] = (T.R[m] << 8) | (uint32_t)m;
    }
    float D[4][M];
    float maxD = -INFINITY, minD = INFINITY;
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const float d = __fsub_rn(z[e], tm[m]);
            D[e][m] = __fmul_rn(d, d);
            maxD = fmaxf(maxD, D[e][m]);
            minD = fminf(minD, D[e][m]);
        }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        maxD = fmaxf(maxD, __shfl_xor_sync(kFull, maxD, d));
        minD = fminf(minD, __shfl_xor_sync(kFull, minD, d));
    }
    const uint32_t budget = (uint32_t)T.budget_bits << 16;
    float lam_hi = __fmul_rn(8.0f, __fsub_rn(maxD, minD));
    float lam_lo = __fmul_rn(lam_hi, 0x1p-40f);
    uint32_t len = 0, sym[4] = {0u, 0u, 0u, 0u};
    // Early-exit variant: when each of the 12 tests passes, the upper end walks hi <- sqrt(lo hi) twelve
    // times with lo fixed; sweep -1 evaluates that multiplier and ends the search if its assignment fits.
    float lam_e = lam_hi;
    if (T.early_exit)
        for (int i = 0; i < 12; ++i) lam_e = __fsqrt_rn(__fmul_rn(lam_lo, lam_e));
#pragma unroll 1
    for (int it = T.early_exit ? -1 : 0; it <= 12; ++it) {
        const float lam = (it < 0) ? lam_e : (it < 12) ? __fsqrt_rn(__fmul_rn(lam_lo, lam_hi)) : lam_hi;
        uint32_t cost_sum = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float c[M];
            uint32_t key[M];
#pragma unroll
            for (int m = 0; m < M; ++m) { c[m] = __fmaf_rn(lam, rm[m], D[e][m]); key[m] = Km[m]; }
            // pairwise minimum, the left (lower index) operand wins ties
#pragma unroll
            for (int w = 1; w < M; w <<= 1)
#pragma unroll
                for (int m = 0; m + w < M; m += 2 * w)
                    if (c[m + w] < c[m]) { c[m] = c[m + w]; key[m] = key[m + w]; }
            sym[e] = key[0];
            cost_sum += key[0];
        }
        len = __reduce_add_sync(kFull, cost_sum >> 8);   // four indices (< 16 each) stay below bit 8
        if (it < 0) {
            if (len <= budget) break;
        } else if (it < 12) {
            if (len <= budget) lam_hi = lam; else lam_lo = lam;
        }
    }
    return make_uint2(len, (sym[0] & 0xffu) | ((sym[1] & 0xffu) << 8) | ((sym[2] & 0xffu) << 16) | (sym[3] << 24));
}

// Length of the assignment (0: known to be within the budget); sym: its levels, one per byte.
template <int M>
__device__ __forceinline__ uint32_t drift(const EncTable& T, const float (&z)[4], float s, float o, float zmin, float zmax,
                                          uint32_t& sym) {
    if (dqdrift::drift_thresholds<M>(T, WarpGroup{kN}, z, s, o, zmin, zmax, sym)) return 0u;
    const uint2 r = drift_sweeps<M>(T, z[0], z[1], z[2], z[3], s, o);
    sym = r.y;
    return r.x;
}

// Drift for the paired-symbol variant: a lane's values (0, 1) and (2, 3) are two rANS symbols; each takes
// the pair u = a M + b that minimises (D_a + D_b) + lambda r_u, the lowest u among equal costs (rows a in
// ascending order, each reduced pairwise with the left operand winning ties, a later row replacing the best
// only when strictly cheaper: the same winner as an ascending scan with a strict comparison).  Bracket:
// hi = 16 (max D - min D), D over single values as above.
// One sweep: the two winners' keys (ceil(65536 r_u) << 8 | u) and the code length.
template <int M>
__device__ __forceinline__ uint32_t pair_sweep(const EncTable& T, const float (&D)[4][M], float lam, uint32_t (&win)[2]) {
    uint32_t cost_sum = 0;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        float rc[M];
        uint32_t rkey[M];
#pragma unroll
        for (int a = 0; a < M; ++a) {
            float c[M];
            uint32_t key[M];
#pragma unroll
            for (int b = 0; b < M; ++b) {
                const uint2 e = T.prk[a * M + b];
                c[b] = __fmaf_rn(lam, __uint_as_float(e.x), __fadd_rn(D[2 * p][a], D[2 * p + 1][b]));
                key[b] = e.y;
            }
#pragma unroll
            for (int w = 1; w < M; w <<= 1)
#pragma unroll
                for (int b = 0; b + w < M; b += 2 * w)
                    if (c[b + w] < c[b]) { c[b] = c[b + w]; key[b] = key[b + w]; }
            rc[a] = c[0];
            rkey[a] = key[0];
        }
#pragma unroll
        for (int w = 1; w < M; w <<= 1)   // row winners, the left (lower a) operand wins ties
#pragma unroll
            for (int a = 0; a + w < M; a += 2 * w)
                if (rc[a + w] < rc[a]) { rc[a] = rc[a + w]; rkey[a] = rkey[a + w]; }
        win[p] = rkey[0];
        cost_sum += rkey[0];
    }
    return __reduce_add_sync(kFull, cost_sum >> 8);   // two pair indices (< 81 each) stay below bit 8
}

// Cost of pair u at lambda = 0 for the values (za, zb), approximately.
template <int M>
__device__ __forceinline__ float pair_distance(float za, float zb, float s, float o, uint32_t u) {
    const float da = za - fmaf((float)(u / M), s, o), db = zb - fmaf((float)(u % M), s, o);
    return fmaf(da, da, db * db);
}

// The bisection's outcome in about five sweeps instead of 13.  A pair's winner moves to ever cheaper pairs as lambda
// grows, so the code length falls with lambda and the bisection ends in the cell (J, J + 1] of its 4096-point grid
// between the last length over the budget and the first within it -- whatever the order in which points are looked
// at.  Two sweeps bracket J around its usual place; between the bracket's ends few pairs change their winner, each
// at a lambda that its two winners give in closed form, and the order statistic of those is J; sweeps at the exact
// lambda_{J+1} and lambda_J (the chain of square roots replayed) confirm it or move the bracket.
// Rounding could make a length rise with lambda only between points closer than 2^-21 of the largest cost over the
// smallest difference of two r: the search is left (the bisection runs) where neighbouring grid points are.
template <int M>
static __device__ __noinline__ uint2 drift_pair_search(const EncTable& T, float z0, float z1, float z2, float z3, float s, float o) {
    const float z[4] = {z0, z1, z2, z3};
    float D[4][M];
    float maxD = -INFINITY, minD = INFINITY;
#pragma unroll
    for (int m = 0; m < M; ++m) {
        const float tm = __fmaf_rn((float)m, s, o);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float d = __fsub_rn(z[e], tm);
            D[e][m] = __fmul_rn(d, d);
            maxD = fmaxf(maxD, D[e][m]);
            minD = fminf(minD, D[e][m]);
        }
    }
    maxD = dqdev::warp_max(maxD);
    minD = dqdev::warp_min(minD);
    const uint32_t budget = (uint32_t)T.budget_bits << 16;
    const float hi0 = __fmul_rn(16.0f, __fsub_rn(maxD, minD)), lo0 = __fmul_rn(hi0, 0x1p-40f);
    constexpr float kG = 102.4f;
    uint32_t win[2] = {0u, 0u};

    if (hi0 > 0x1p-38f && hi0 < 0x1p80f && T.pair_dr > 0.f) {
        const float lg_hi = dqdrift::lg2_approx(hi0);
        int jl = 0, jh = 4096, j = 4096 + (int)(kG * (dqdrift::lg2_approx(0.25f * s * s) - lg_hi)), step = 48, J = 0;
        j = min(max(j, 200), 4000);
        bool have_l = false, have_h = false;
        uint32_t kl[2] = {0u, 0u}, kh[2] = {0u, 0u}, kf[2] = {0u, 0u}, len_h = 0;
        float lam = hi0 * dqdrift::exp2_approx((float)(j - 4096) * (1.f / kG)), lam_lo = 0.f;
        int phase = 0;   // 0: bracket, 1: lambda_{J+1}, 2: lambda_J
#pragma unroll 1
        for (int it = 0; it < 11; ++it) {
            const uint32_t len = pair_sweep<M>(T, D, lam, win);
            const bool over = len > budget;
            if (phase == 2 && over) {   // confirmed: the winners at lambda_{J+1}
                const float far = maxD + maxD + lam * 8.f;   // no cost of a winner is larger
                if (lam * (0.0067f * T.pair_dr) < 0x1p-21f * far) break;
                const uint32_t u0 = kf[0] & 0xffu, u1 = kf[1] & 0xffu;
                return make_uint2(0u, (u0 / M) | ((u0 % M) << 8) | ((u1 / M) << 16) | ((u1 % M) << 24));
            }
            const int at = phase == 0 ? j : phase == 1 ? J + 1 : J;
            if (over) { jl = at; kl[0] = win[0]; kl[1] = win[1]; have_l = true; }
            else { jh = at; kh[0] = win[0]; kh[1] = win[1]; len_h = len; have_h = true; }
            if (phase == 1 && !over) {
                kf[0] = win[0]; kf[1] = win[1];
                phase = 2;
                lam = lam_lo;
                continue;
            }
            if (!have_l || !have_h) {
                j += over ? step : -step;
                step *= 3;
                if (j < 2 || j > 4090) break;
                lam = hi0 * dqdrift::exp2_approx((float)(j - 4096) * (1.f / kG));
                continue;
            }
            // lambdas at which the pairs leave their winner at jl for the one at jh, and what that saves
            float t[2];
            uint32_t w[2];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const uint32_t ul = kl[p] & 0xffu, uh = kh[p] & 0xffu;
                const float dr = __uint_as_float(T.prk[ul].x) - __uint_as_float(T.prk[uh].x);
                const float dD = pair_distance<M>(z[2 * p], z[2 * p + 1], s, o, uh) - pair_distance<M>(z[2 * p], z[2 * p + 1], s, o, ul);
                w[p] = (kl[p] >> 8) - (kh[p] >> 8);
                t[p] = (ul != uh && dr > 0.f) ? fmaxf(dD * dqdrift::rcp_approx(dr), 0.f) : 0.f;
            }
            float tc = INFINITY;
            int k = 0;
#pragma unroll 1
            for (; k < 40; ++k) {   // largest first, until the length exceeds the budget again
                float m = 0.f;
                dqdrift::max_if_less(m, t[0], tc);
                dqdrift::max_if_less(m, t[1], tc);
                tc = __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(m)));
                if (!(tc > 0.f)) break;
                uint32_t sum = 0;
                dqdrift::add_if_not_less(sum, t[0], tc, w[0]);
                dqdrift::add_if_not_less(sum, t[1], tc, w[1]);
                if (len_h + __reduce_add_sync(kFull, sum) > budget) break;
            }
            if (k == 40 || !(tc > 0.f)) break;
            J = 4096 + (int)floorf(kG * (dqdrift::lg2_approx(tc) - lg_hi));
            J = min(max(J, jl), jh - 1);
            if (J < 1 || J > 4094) break;
            float lo = lo0, hi = hi0;
#pragma unroll 1
            for (int b = 11; b >= 0; --b) {
                const float mid = __fsqrt_rn(__fmul_rn(lo, hi));
                if ((J >> b) & 1) lo = mid; else hi = mid;
            }
            lam_lo = lo;
            lam = hi;
            phase = 1;
        }
    }

    float lam_hi = hi0, lam_lo = lo0;
    uint32_t len = 0;
    float lam_e = lam_hi;
    if (T.early_exit)
        for (int i = 0; i < 12; ++i) lam_e = __fsqrt_rn(__fmul_rn(lam_lo, lam_e));
#pragma unroll 1
    for (int it = T.early_exit ? -1 : 0; it <= 12; ++it) {
        const float lam = (it < 0) ? lam_e : (it < 12) ? __fsqrt_rn(__fmul_rn(lam_lo, lam_hi)) : lam_hi;
        len = pair_sweep<M>(T, D, lam, win);
        if (it < 0) {
            if (len <= budget) break;
        } else if (it < 12) {
            if (len <= budget) lam_hi = lam; else lam_lo = lam;
        }
    }
    const uint32_t u0 = win[0] & 0xffu, u1 = win[1] & 0xffu;
    return make_uint2(len, (u0 / M) | ((u0 % M) << 8) | ((u1 / M) << 16) | ((u1 % M) << 24));
}

// Levels of the nearest pairs: Drift's outcome when their length, summed over the stream, fits the budget (every test of the
// bisection then passes and lambda ends too small to move any pair) and no `clear` of the stream is negative (no value
// within rounding of a midpoint).  False where the bound on rounding does not hold.
template <int M>
__device__ __forceinline__ bool nearest_pairs(const EncTable& T, const float (&z)[4], float s, float o, float zmin, float zmax,
                                              uint32_t& sym, uint32_t& len, float& clear) {
    if (!(s > 0x1p-30f && s < 0x1p40f)) return false;
    const float inv = dqdrift::rcp_approx(s), shift = -o * inv;
    const float vmax = fmaf(zmax, inv, shift), vmin = fmaf(zmin, inv, shift);
    const float reach = fmaxf(vmax, (float)(M - 1) - vmin);
    const float mag = fmaxf(fmaxf(fabsf(zmin), fabsf(zmax)), fmaxf(fabsf(o), fabsf(o + (float)(M - 1) * s))) * inv;
    if (!(mag < 1024.f && reach < 64.f)) return false;
    const float E = 1.5f * 0x1p-24f * (2.f * mag + 4.f * reach + (float)M + 2.f * reach * reach);
    float near[4], mid = 1.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float v = fmaf(z[e], inv, shift);
        near[e] = fminf(fmaxf((v + 12582912.f) - 12582912.f, 0.f), (float)(M - 1));
        mid = fminf(mid, fabsf(fabsf(v - near[e]) - 0.5f));
    }
    const uint32_t u0 = (uint32_t)(int)fmaf(near[0], (float)M, near[1]), u1 = (uint32_t)(int)fmaf(near[2], (float)M, near[3]);
    len = (T.prk[u0].y >> 8) + (T.prk[u1].y >> 8);
    sym = (u0 / M) | ((u0 % M) << 8) | ((u1 / M) << 16) | ((u1 % M) << 24);
    clear = mid - E;
    return true;
}

// Length of the assignment (0: known to be within the budget); sym: its levels, one per byte.
template <int M>
__device__ __forceinline__ uint32_t drift_pair(const EncTable& T, const float (&z)[4], float s, float o, float zmin, float zmax,
                                               uint32_t& sym) {
    uint32_t len;
    float clear;
    if (nearest_pairs<M>(T, z, s, o, zmin, zmax, sym, len, clear) && __reduce_add_sync(kFull, len) <= ((uint32_t)T.budget_bits << 16) &&
        __all_sync(kFull, clear > 0.f))
        return 0u;
    const uint2 r = drift_pair_search<M>(T, z[0], z[1], z[2], z[3], s, o);
    sym = r.y;
    return r.x;
}

// ---------------------------------------------------------------------- encoder

// Position and sequence of call token t (decode-step mode derives them from the sequence lengths).
__device__ __forceinline__ int tok_pos(const DqEncodeArgs& a, int t) { return a.step_seq_lens ? a.step_seq_lens[t] - 1 : a.pos[t]; }
__device__ __forceinline__ int tok_seq(const DqEncodeArgs& a, int t) { return a.step_seq_lens ? t : a.seq_id[t]; }

// One step of Eq. rans Enc with the entry `en` of EncTable::enc: a byte of the state goes to shared memory at `dst`,
// which advances by `stride`, when the state is not below en.y (at most once: x < 2^8 L <= 2^8 (f L)).
template <int STRIDE>
__device__ __forceinline__ void rans_step(uint32_t& x, uint32_t& dst, const uint4 en) {
    asm volatile("{.reg .pred p; setp.ge.u32 p, %0, %2; @p st.shared.u8 [%1], %0; @p add.u32 %1, %1, %3; @p shr.u32 %0, %0, 8;}"
                 : "+r"(x), "+r"(dst) : "r"(en.y), "n"(STRIDE) : "memory");
    x = __funnelshift_r(__umulhi(x, en.x), 0u, en.w) * (en.w >> 5) + (x + en.z);   // the shift uses en.w mod 32
}

// Eq. rans Enc on the symbols of `row` (four per word) from the last one back, so that decoding runs forward.  The entries
// do not depend on the state: a word's are fetched while the word after it is coded.
template <int STRIDE>
__device__ __forceinline__ void rans_encode_row(const uint4* enc, const uint32_t* row, int words, uint32_t& x, uint32_t& dst) {
    uint4 nxt[4];
    uint32_t m4 = row[words - 1];
#pragma unroll
    for (int b = 0; b < 4; ++b) nxt[b] = enc[(m4 >> (8 * b)) & 0xffu];
    m4 = row[max(words - 2, 0)];
#pragma unroll 1
    for (int jw = words - 1; jw >= 0; --jw) {
        uint4 cur[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) { cur[b] = nxt[b]; nxt[b] = enc[(m4 >> (8 * b)) & 0xffu]; }
        m4 = row[max(jw - 2, 0)];
#pragma unroll
        for (int b = 3; b >= 0; --b) rans_step<STRIDE>(x, dst, cur[b]);
    }
}

struct StreamQuantised {
    uint32_t hdr0;      // s fp16 | o fp16 << 16
    uint32_t flags;     // 1: all-central fallback, 2: constant stream, 4: refit rejected
    uint32_t sym;       // this lane's four levels, one per byte
};

// Token and KV head of stream `sid` (streams are token-major).
__device__ __forceinline__ void split_stream(const DqEncodeArgs& a, long long sid, int& t, int& h) {
    if (a.hkv_magic) {
        t = (int)__umulhi((uint32_t)sid, a.hkv_magic);
        h = (int)((uint32_t)sid - (uint32_t)t * (uint32_t)a.Hkv);
    } else {
        t = (int)(sid / a.Hkv);
        h = (int)(sid - (long long)t * a.Hkv);
    }
}

__device__ __forceinline__ void unpack_bf16x4(uint2 raw, float (&z)[4]) {
    z[0] = __uint_as_float(raw.x << 16); z[1] = __uint_as_float(raw.x & 0xffff0000u);
    z[2] = __uint_as_float(raw.y << 16); z[3] = __uint_as_float(raw.y & 0xffff0000u);
}

// z -= scale * mean, the window's INT8 channel means in four bytes of q4 (Sec. 4.2).  A byte becomes a float
// by completing it to 2^23 + (q + 128) and subtracting: exact.
__device__ __forceinline__ void remove_mean(float (&z)[4], uint32_t q4, float scale) {
    const uint32_t u = q4 ^ 0x80808080u;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float q = __fsub_rn(__uint_as_float(__byte_perm(u, 0x4b000000u, 0x7440 + e)), 8388736.f);
        z[e] = __fsub_rn(z[e], __fmul_rn(scale, q));
    }
}

// Row of the mean arrays for (token t, window of position ps, head h).
__device__ __forceinline__ size_t mean_row(const DqEncodeArgs& a, int seq, int ps, int h) {
    return ((size_t)seq * a.max_windows + ps / DQ_WINDOW_TOKENS) * a.Hkv + h;
}

// DQ_MEAN_REUSE at the first position of a window: carry the previous window's mean forward (window 0: zero) into
// row mi.  Rows are per head, so this warp is the only writer and reader of the row in this call.
__device__ __forceinline__ void carry_mean(const DqEncodeArgs& a, size_t mi, int ps, int lane, uint32_t& q4, float& sc) {
    q4 = 0u; sc = 0.f;
    if (ps >= DQ_WINDOW_TOKENS) {
        const size_t src = mi - (size_t)a.Hkv;
        q4 = *reinterpret_cast<const uint32_t*>(a.mean_q + src * kN + 4 * lane);
        sc = a.mean_scale[src];
    }
    *reinterpret_cast<uint32_t*>(a.mean_q + mi * kN + 4 * lane) = q4;
    if (lane == 0) a.mean_scale[mi] = sc;
}

// Least squares of z on the symbols from integer sums: the values are rounded to multiples of `unit` (2^-19 of the
// power of two below the largest), so that every sum is one integer reduction.  The binary64 sums that
// define the result differ from these by less than the two errors of refit_finish; when both ends of the error
// interval round to the same fp16 pair, that is the pair (all but about one stream in 200).
struct RefitScale {
    float scale, unit;   // 1 / unit, unit
    bool ok;
};
__device__ __forceinline__ RefitScale refit_scale(float zabs) {
    const uint32_t ex = __float_as_uint(zabs) & 0x7f800000u;                          // 2^e <= zabs < 2^(e + 1)
    RefitScale r;
    r.ok = zabs > 0x1p-60f && zabs < 0x1p60f;
    r.scale = __uint_as_float((254u << 23) - ex + (19u << 23));                       // 2^(19 - e)
    r.unit = __uint_as_float(ex - (19u << 23));
    return r;
}

struct RefitSums {
    int Sm, Smm, SA, SB;   // sums of m, m^2, z / unit, m z / unit over a warp's 128 values
};
__device__ __forceinline__ RefitSums refit_sums(const float (&z)[4], const RefitScale& sc, uint32_t sym) {
    constexpr uint32_t kMagic = 0x4b400000u;   // 1.5 2^23: the low bits of z / unit + 1.5 2^23 are the integer
    uint32_t a = 0, b = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const uint32_t zi = __float_as_uint(__fmaf_rn(z[e], sc.scale, 12582912.f));
        a += zi;
        b += zi * ((sym >> (8 * e)) & 0xffu);
    }
    // sums of the levels and of their squares: < 2^11 and < 2^15
    const uint32_t both = __reduce_add_sync(kFull, __dp4a(sym, 0x01010101u, 0u) << 16 | __dp4a(sym, sym, 0u));
    RefitSums r;
    r.Sm = (int)(both >> 16);
    r.Smm = (int)(both & 0xffffu);
    r.SA = (int)(__reduce_add_sync(kFull, a) - kN * kMagic);
    r.SB = (int)(__reduce_add_sync(kFull, b) - (uint32_t)r.Sm * kMagic);
    return r;
}

// fp16 pair of the solution for n values, or false when its rounding is within the error of a tie.
__device__ __forceinline__ bool refit_finish(const RefitScale& sc, float n, float SA, float SB, float Sm, float den, uint32_t& hdr) {
    if (!(den > 0.f)) return false;
    const float nb = n * SB, ma = Sm * SA, rd = dqdrift::rcp_approx(den), rn = 1.f / n;   // n is a constant or a small integer
    const float sd = (nb - ma) * rd;                                                  // in units
    const float t = sd * Sm;
    const float od = (SA - t) * rn;
    // |sum of (n m - Sm) errors| <= n sqrt(den) / 2, over den; binary32 roundings
    const float es = 0.52f * n * dqdrift::sqrt_approx(rd) + 0x1p-22f * rd * (fabsf(nb) + fabsf(ma)) + 0x1p-21f * fabsf(sd);
    const float eo = 0.51f + (es * Sm + 0x1p-21f * (fabsf(SA) + fabsf(t))) * rn;
    const __half2 lo = __floats2half2_rn((sd - es) * sc.unit, (od - eo) * sc.unit), hi = __floats2half2_rn((sd + es) * sc.unit, (od + eo) * sc.unit);
    hdr = *reinterpret_cast<const uint32_t*>(&lo);
    return hdr == *reinterpret_cast<const uint32_t*>(&hi);
}

// A warp's sums of z and m z in binary64, in the order that defines the result: a lane's values, then a butterfly.
__device__ __forceinline__ void refit_sums_binary64(const float (&z)[4], uint32_t sym, double& sa, double& sb) {
    sa = (double)z[0];
    sb = __dmul_rn((double)(sym & 0xffu), (double)z[0]);
#pragma unroll
    for (int e = 1; e < 4; ++e) {
        sa = __dadd_rn(sa, (double)z[e]);
        sb = __dadd_rn(sb, __dmul_rn((double)((sym >> (8 * e)) & 0xffu), (double)z[e]));
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        sa = __dadd_rn(sa, __shfl_xor_sync(kFull, sa, d));
        sb = __dadd_rn(sb, __shfl_xor_sync(kFull, sb, d));
    }
}

// The refit from those sums, both parameters rounded once.
static __device__ __noinline__ uint32_t refit_binary64(float z0, float z1, float z2, float z3, uint32_t sym, float s, float o) {
    const float z[4] = {z0, z1, z2, z3};
    double sa, sb;
    refit_sums_binary64(z, sym, sa, sb);
    const int Sm = (int)__reduce_add_sync(kFull, __dp4a(sym, 0x01010101u, 0u)), Smm = (int)__reduce_add_sync(kFull, __dp4a(sym, sym, 0u));
    const int den = kN * Smm - Sm * Sm;
    double sd = (double)s, od = (double)o;
    if (den != 0) {
        sd = __ddiv_rn(__dsub_rn(__dmul_rn((double)kN, sb), __dmul_rn((double)Sm, sa)), (double)den);
        od = __dmul_rn(__dsub_rn(sa, __dmul_rn(sd, (double)Sm)), 1.0 / kN);   // kN is a power of two
    }
    return (uint32_t)__half_as_ushort(__double2half(sd)) | ((uint32_t)__half_as_ushort(__double2half(od)) << 16);
}

// Steps 2-6 of Algorithm 1 by one warp on the rotated, mean-free values of a stream: min-max grid, drift, refit,
// fp16 metadata, second drift.  M: the table's levels.
// PAIR: its rANS symbols are pairs of levels.
// COMPACT: both Drift calls run the same code in a loop -- for calls of a few streams, whose time is the way through the
// code once, with the instruction cache cold.
template <int M, bool PAIR, bool COMPACT>
__device__ __forceinline__ StreamQuantised quantise_values(const EncTable& T, const float (&z)[4]) {
    const float mx = dqdev::warp_max(fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3])));
    const float mn = dqdev::warp_min(fminf(fminf(z[0], z[1]), fminf(z[2], z[3])));
    StreamQuantised r;
    r.sym = T.central;   // four levels, one per byte
    r.flags = 0u;
    r.hdr0 = (uint32_t)__half_as_ushort(__float2half_rn(mn)) << 16;
    if (!(mx > mn)) { r.flags = 2u; return r; }
    float s = __fdiv_rn(__fsub_rn(mx, mn), (float)(M - 1)), o = mn; // FitMinMax, Eq. (affine_token)
    uint32_t sym = 0u, len = 0u, hdr = 0u;
#pragma unroll (COMPACT ? 1 : 2)
    for (int pass = 0; pass < 2; ++pass) {
        len = PAIR ? drift_pair<M>(T, z, s, o, mn, mx, sym) : drift<M>(T, z, s, o, mn, mx, sym);
        if (pass == 1) break;
        // Refit, fp16 metadata; the second Drift runs on the fp16 grid
        const RefitScale sc = refit_scale(fmaxf(fabsf(mn), fabsf(mx)));
        const RefitSums h = refit_sums(z, sc, sym);
        if (!sc.ok || !refit_finish(sc, (float)kN, (float)h.SA, (float)h.SB, (float)h.Sm, (float)(kN * h.Smm - h.Sm * h.Sm), hdr))
            hdr = refit_binary64(z[0], z[1], z[2], z[3], sym, s, o);
        float sf = __half2float(__ushort_as_half((unsigned short)(hdr & 0xffffu))), of = __half2float(__ushort_as_half((unsigned short)(hdr >> 16)));
        if (!(isfinite(sf) && sf > 0.0f && isfinite(of))) {
            const __half s16 = __float2half_rn(s), o16 = __float2half_rn(o);
            hdr = (uint32_t)__half_as_ushort(s16) | ((uint32_t)__half_as_ushort(o16) << 16);
            sf = __half2float(s16); of = __half2float(o16);
            r.flags = 4u;
        }
        if (!(sf > 0.0f)) { r.flags |= 2u; return r; }
        s = sf; o = of;
    }
    r.hdr0 = hdr;
    if (len > ((uint32_t)T.budget_bits << 16)) r.flags |= 1u; else r.sym = sym;
    return r;
}

}  // namespace dqenc

// Batch kernels (dq_encode_batch.cu): most streams per CTA, and the launch of one tensor kind or both; per: streams per
// CTA, 0: by the size of the call.
constexpr int kDqEncodeBatchStreams = 32;
cudaError_t dq_launch_encode_batch(const DqDevTable& tk, const DqDevTable& tv, const DqPairEnc& pk, const DqPairEnc& pv,
                                   const DqEncodeArgs& a, int per, cudaStream_t st);
// Token-wide streams (dq_encode_wide.cu); per: streams per CTA, 0: by the size of the call.
cudaError_t dq_launch_encode_wide(const DqDevTable& tk, const DqDevTable& tv, const DqPairEnc& pk, const DqPairEnc& pv,
                                  const DqEncodeArgs& a, int per, cudaStream_t st);
