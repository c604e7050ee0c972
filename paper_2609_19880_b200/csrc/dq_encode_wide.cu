// Encoder kernel for token-wide streams (heads_per_stream = hs > 1; Sec. 5.1 "Implementation details").  Compiled
// with -fmad=false, as dq_encode.cu.
//
// A CTA of hs warps takes `per` consecutive streams: warp w holds head w of the stream at hand, 4 values per lane,
// and the streams are quantised one after the other; then one warp entropy-codes all of them at once, lane =
// stream, so that the serial rANS chain of hs * 128 symbols is paid once per CTA.  What bounds it is the issue
// of the quantiser's instructions and the CTA barriers between its reductions; Drift's multiplier comes from a
// histogram of the values' thresholds (below) with 4 barriers instead of 14 sweeps with one each.
#include "dq_encode.cuh"

using namespace dqenc;

namespace {

constexpr int kCells = 4096;         // the grid on which Drift tests its multiplier
constexpr int kWB = 32;              // most streams per CTA

// Cross-warp pieces.  Reductions over the stream go warp -> shared slot -> CTA barrier; slots are
// double-buffered by call parity so one barrier per reduction suffices.
struct WideShared {
    float fmax[2][DQ_MAX_STREAM_HEADS], fmin[2][DQ_MAX_STREAM_HEADS];
    uint32_t len[2][DQ_MAX_STREAM_HEADS];
    double sa[DQ_MAX_STREAM_HEADS], sb[DQ_MAX_STREAM_HEADS];
    int sm[2][DQ_MAX_STREAM_HEADS], smm[2][DQ_MAX_STREAM_HEADS], ia[2][DQ_MAX_STREAM_HEADS];
    int ib_lo[2][DQ_MAX_STREAM_HEADS], ib_hi[2][DQ_MAX_STREAM_HEADS];
    int J;                           // cell that the histogram search ends in
};

// Smallest difference of two level costs whose code lengths differ.
template <int M>
__device__ __forceinline__ float least_cost_step(const float (&rm)[M], const uint32_t (&Km)[M]) {
    float dr = 1e30f;
#pragma unroll
    for (int m = 1; m < M; ++m)
#pragma unroll
        for (int n = 0; n < m; ++n)
            if ((Km[m] ^ Km[n]) >> 8) dr = fminf(dr, fabsf(rm[m] - rm[n]));
    return dr;
}

// The bisection's outcome from where it nearly certainly ends: the length at lambda_{J+1} of its 4096-point grid within the
// budget, the one at lambda_J over it; otherwise J moves by one.  2 sweeps instead of 13: 713 -> 699 us for 5 prompts of
// 1000 to 4000 tokens (the per-head kernel, short of registers, lost 2 % with it).  sweep(lambda) returns the
// length and leaves the winners in sym; kept: those at lambda_{J+1}.  Lengths fall with lambda, except where rounding
// decides: between points closer than 2^-21 of the largest cost over the smallest difference of two r (dr); there, and
// when J is not found, the result is false.
template <class Sweep>
__device__ __forceinline__ bool confirm_cell(const Sweep& sweep, int J, uint32_t budget, float lam_lo0, float lam_hi0, float maxD, float dr,
                                             const uint32_t (&sym)[4], uint32_t (&kept)[4]) {
#pragma unroll 1
    for (int t = 0; t < 3; ++t) {
        if (J < 1 || J > 4094) return false;
        float lo = lam_lo0, hi = lam_hi0;
#pragma unroll 1
        for (int b = 11; b >= 0; --b) {
            const float mid = __fsqrt_rn(__fmul_rn(lo, hi));
            if ((J >> b) & 1) lo = mid; else hi = mid;
        }
        if (!(lo * (0.0067f * dr) > 0x1p-21f * (maxD + hi * 8.f))) return false;   // r <= 8
        if (sweep(hi) > budget) { ++J; continue; }
#pragma unroll
        for (int e = 0; e < 4; ++e) kept[e] = sym[e];
        if (sweep(lo) > budget) return true;
        --J;
    }
    return false;
}

// Function Drift of Algorithm 1 for a stream held by hs warps; same arithmetic as drift_sweeps, with
// the extrema of D and the code length taken over the whole stream.
template <int M>
__device__ __forceinline__ uint2 drift_wide_sweeps(const EncTable& T, WideShared& W, int hs, int wib, uint32_t& parity,
                                                   const float (&z)[4], float s, float o, int cell) {
    const int lane = threadIdx.x & 31;
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
    if (lane == 0) { W.fmax[parity][wib] = maxD; W.fmin[parity][wib] = minD; }
    __syncthreads();
    for (int w = 0; w < hs; ++w) { maxD = fmaxf(maxD, W.fmax[parity][w]); minD = fminf(minD, W.fmin[parity][w]); }
    parity ^= 1u;
    const uint32_t budget = (uint32_t)T.budget_bits << 16;
    float lam_hi = __fmul_rn(8.0f, __fsub_rn(maxD, minD));
    float lam_lo = __fmul_rn(lam_hi, 0x1p-40f);
    uint32_t len = 0, sym[4] = {0u, 0u, 0u, 0u};
    auto sweep = [&](float lam) {
        uint32_t cost_sum = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float c[M];
            uint32_t key[M];
#pragma unroll
            for (int m = 0; m < M; ++m) { c[m] = __fmaf_rn(lam, rm[m], D[e][m]); key[m] = Km[m]; }
#pragma unroll
            for (int w = 1; w < M; w <<= 1)
#pragma unroll
                for (int m = 0; m + w < M; m += 2 * w)
                    if (c[m + w] < c[m]) { c[m] = c[m + w]; key[m] = key[m + w]; }
            sym[e] = key[0];
            cost_sum += key[0];
        }
        const uint32_t wl = __reduce_add_sync(kFull, cost_sum >> 8);
        if (lane == 0) W.len[parity][wib] = wl;
        __syncthreads();
        uint32_t sum = 0;
        for (int w = 0; w < hs; ++w) sum += W.len[parity][w];   // every warp sees the same stream-wide length
        parity ^= 1u;
        return sum;
    };
    uint32_t kept[4];
    if (cell > 0 && confirm_cell(sweep, cell, budget, lam_lo, lam_hi, maxD, least_cost_step<M>(rm, Km), sym, kept))
        return make_uint2(0u, (kept[0] & 0xffu) | ((kept[1] & 0xffu) << 8) | ((kept[2] & 0xffu) << 16) | (kept[3] << 24));
    // Early-exit variant: when each of the 12 tests passes, the upper end walks hi <- sqrt(lo hi) twelve
    // times with lo fixed; sweep -1 evaluates that multiplier and ends the search if its assignment fits.
    float lam_e = lam_hi;
    if (T.early_exit)
        for (int i = 0; i < 12; ++i) lam_e = __fsqrt_rn(__fmul_rn(lam_lo, lam_e));
#pragma unroll 1
    for (int it = T.early_exit ? -1 : 0; it <= 12; ++it) {
        const float lam = (it < 0) ? lam_e : (it < 12) ? __fsqrt_rn(__fmul_rn(lam_lo, lam_hi)) : lam_hi;
        len = sweep(lam);
        if (it < 0) {
            if (len <= budget) break;   // uniform across the CTA
        } else if (it < 12) {
            if (len <= budget) lam_hi = lam; else lam_lo = lam;
        }
    }
    return make_uint2(len, (sym[0] & 0xffu) | ((sym[1] & 0xffu) << 8) | ((sym[2] & 0xffu) << 16) | (sym[3] << 24));
}

// Drift for paired symbols on a stream held by hs warps: the pair search of drift_pair with the extrema of D
// and the code length taken over the whole stream, as in drift_wide_sweeps.
template <int M>
__device__ __forceinline__ uint2 drift_wide_pairs(const EncTable& T, WideShared& W, int hs, int wib, uint32_t& parity,
                                                  const float (&z)[4], float s, float o) {
    const int lane = threadIdx.x & 31;
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
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        maxD = fmaxf(maxD, __shfl_xor_sync(kFull, maxD, d));
        minD = fminf(minD, __shfl_xor_sync(kFull, minD, d));
    }
    if (lane == 0) { W.fmax[parity][wib] = maxD; W.fmin[parity][wib] = minD; }
    __syncthreads();
    for (int w = 0; w < hs; ++w) { maxD = fmaxf(maxD, W.fmax[parity][w]); minD = fminf(minD, W.fmin[parity][w]); }
    parity ^= 1u;
    const uint32_t budget = (uint32_t)T.budget_bits << 16;
    float lam_hi = __fmul_rn(16.0f, __fsub_rn(maxD, minD));
    float lam_lo = __fmul_rn(lam_hi, 0x1p-40f);
    uint32_t len = 0, psym[2] = {0u, 0u};
    float lam_e = lam_hi;
    if (T.early_exit)
        for (int i = 0; i < 12; ++i) lam_e = __fsqrt_rn(__fmul_rn(lam_lo, lam_e));
#pragma unroll 1
    for (int it = T.early_exit ? -1 : 0; it <= 12; ++it) {
        const float lam = (it < 0) ? lam_e : (it < 12) ? __fsqrt_rn(__fmul_rn(lam_lo, lam_hi)) : lam_hi;
        uint32_t cost_sum = 0;
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            float best = 0.f;
            uint32_t bkey = 0u;
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
                if (a == 0 || c[0] < best) { best = c[0]; bkey = key[0]; }   // an earlier row keeps equal costs
            }
            psym[p] = bkey;
            cost_sum += bkey;
        }
        const uint32_t wl = __reduce_add_sync(kFull, cost_sum >> 8);
        if (lane == 0) W.len[parity][wib] = wl;
        __syncthreads();
        len = 0;
        for (int w = 0; w < hs; ++w) len += W.len[parity][w];
        parity ^= 1u;
        if (it < 0) {
            if (len <= budget) break;   // uniform across the CTA
        } else if (it < 12) {
            if (len <= budget) lam_hi = lam; else lam_lo = lam;
        }
    }
    const uint32_t u0 = psym[0] & 0xffu, u1 = psym[1] & 0xffu;
    return make_uint2(len, (u0 / M) | ((u0 % M) << 8) | ((u1 / M) << 16) | ((u1 % M) << 24));
}

// The hs slots of a reduction, one per lane, combined by one warp instruction.
__device__ __forceinline__ uint32_t slots_add(const uint32_t* slot, int hs) {
    const int lane = threadIdx.x & 31;
    return __reduce_add_sync(kFull, lane < hs ? slot[lane] : 0u);
}
__device__ __forceinline__ int slots_add(const int* slot, int hs) {
    const int lane = threadIdx.x & 31;
    return __reduce_add_sync(kFull, lane < hs ? slot[lane] : 0);
}
__device__ __forceinline__ float slots_max(const float* slot, int hs) { return dqdev::warp_max(slot[min((int)(threadIdx.x & 31), hs - 1)]); }
__device__ __forceinline__ float slots_min(const float* slot, int hs) { return dqdev::warp_min(slot[min((int)(threadIdx.x & 31), hs - 1)]); }

// Drift's outcome from thresholds (dq_drift.cuh) on a stream held by hs warps.  1024 values put about one threshold
// into every grid cell, so J is found by a histogram of the thresholds' cells with a suffix sum over it (the
// sums and maxima that serve 128 values would each be a CTA barrier here).  A threshold counts for the cell of the
// lower end of its error interval: the length at lambda_J is then certainly over the budget, and the one at
// lambda_{J+1} is exact unless some interval holds that point, which is a tie.  Returns false on a tie, with the cell J
// (-1: none) that the sweeps then try first.
// hist: kCells words, zero on entry and on return.
template <int M>
__device__ __forceinline__ bool drift_wide_thresholds(const EncTable& T, WideShared& W, uint32_t* hist, int hs, int wib,
                                                      uint32_t& parity, const float (&z)[4], float s, float o, float zmin,
                                                      float zmax, uint32_t& sym, int& cell) {
    cell = -1;
    constexpr int kC = (M - 1) / 2, kLow = kC, kHigh = M - 1 - kC;
    const int lane = threadIdx.x & 31;
    if (!(s > 0x1p-30f && s < 0x1p40f)) return false;
    const float inv = dqdrift::rcp_approx(s), shift = -o * inv;
    const float vmax = fmaf(zmax, inv, shift), vmin = fmaf(zmin, inv, shift);
    const float reach = fmaxf(vmax, (float)(M - 1) - vmin);
    const float mag = fmaxf(fmaxf(fabsf(zmin), fabsf(zmax)), fmaxf(fabsf(o), fabsf(o + (float)(M - 1) * s))) * inv;
    if (!(mag < 1024.f && reach < 1024.f)) return false;
    const float E = 1.5f * 0x1p-24f * (2.f * mag + 4.f * reach + (float)M);

    float a[4], y[4][kHigh];
    uint32_t w = 0;
    float dmin = 1e30f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        a[i] = fmaf(z[i], inv, shift) - (float)kC;
        const int up = a[i] >= 0.f ? 1 : 0;
        float d = fabsf(a[i]);
#pragma unroll
        for (int e = 0; e < kHigh; ++e) {
            const uint4 ed = T.edge[up][e];
            y[i][e] = fmaf(fabsf(a[i]), __uint_as_float(ed.x), __uint_as_float(ed.y));
            dqdrift::add_if_greater(w, y[i][e], 0.f, ed.z);
            dqdrift::fadd_if_greater(d, y[i][e], 0.f, -1.f);
        }
        dmin = fminf(dmin, fabsf(d));
    }
    const uint32_t budget = (uint32_t)T.budget_bits << 16, base = (uint32_t)(hs * kN) * T.R[kC];
    if (base > budget) return false;
    const uint32_t cap = budget - base;
    w = __reduce_add_sync(kFull, w);
    dmin = dqdev::warp_min(dmin);
    if (lane == 0) { W.len[parity][wib] = w; W.fmin[parity][wib] = dmin; }
    if (threadIdx.x == 0) W.J = 0;
    __syncthreads();
    w = slots_add(W.len[parity], hs);
    dmin = slots_min(W.fmin[parity], hs);
    parity ^= 1u;

    float yf = 0.f, band = E * T.inv_max;
    bool tie = false;
    if (w > cap) {   // otherwise the nearest levels fit
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
        const float lgD = log2f(fmaf(reach, reach, -dmin * dmin)) - 8.f;
        const float wA = 4e-4f + 1.5f * 148.f * 0x1p-24f * (2.f * mag + 4.f * reach + 2.f * T.rho);
        const float u0 = -102.4f * lgD - wA;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int up = a[i] >= 0.f ? 1 : 0;
#pragma unroll
            for (int e = 0; e < kHigh; ++e) {
                const float yl = y[i][e] - band;
                if (yl > 0.f) {
                    // floor by adding 2^23 with rounding down; cells below 0 never matter, above 4095 always do
                    const float u = fminf(fmaxf(fmaf(dqdrift::lg2_approx(yl), 102.4f, u0), -3072.f), 1023.f);
                    atomicAdd(hist + (__float_as_uint(__fadd_rd(u, 8388608.f + 3072.f)) & (kCells - 1)), T.edge[up][e].z);
                }
            }
        }
        __syncthreads();
        // suffix sums: thread t has the t-th run of cells from the top, and clears it for the next call
        const int per = ((kCells + hs * 32 - 1) / (hs * 32) + 3) & ~3;
        const int top = kCells - (int)threadIdx.x * per, bottom = max(top - per, 0);   // cells [bottom, top)
        uint32_t own = 0;
        for (int c = top - 4; c >= bottom; c -= 4) {
            const uint4 h = *reinterpret_cast<const uint4*>(hist + c);
            own += (h.x + h.y) + (h.z + h.w);
        }
        uint32_t incl = own;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t v = __shfl_up_sync(kFull, incl, d);
            if (lane >= d) incl += v;
        }
        if (lane == 31) W.len[parity][wib] = incl;
        __syncthreads();
        incl += slots_add(W.len[parity], wib);
        parity ^= 1u;
        if (incl > cap && incl - own <= cap) {   // one thread at most: the last cell at which the sum exceeds cap
            uint32_t sum = incl - own;
            int c = top;
            while (sum <= cap) sum += hist[--c];
            W.J = c;
        }
        for (int c = top - 4; c >= bottom; c -= 4) *reinterpret_cast<uint4*>(hist + c) = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        const int J = W.J;
        tie = J < 2 || J > 4092;
        if (!tie) cell = J;
        yf = dqdrift::exp2_approx(fmaf((float)(J + 1 - 3072), 1.f / 102.4f, lgD));
        // wider than the histogram's intervals, so that an edge whose cell and final comparison disagree is always a tie
        band = fmaf(yf, 1.5f * wA * (1.f / 148.f), 1.5f * band);
    }
    uint32_t lev[4];
    const float E2 = fmaf(yf, 0x1p-18f, E);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool up = a[i] >= 0.f;
        const float unit = up ? 1.f : -1.f;
        float m = 8388608.f + (float)kC;   // the low byte of its bits is the level
#pragma unroll
        for (int e = 0; e < kHigh; ++e) {
            dqdrift::fadd_if_greater(m, y[i][e], yf, unit);
            tie |= fabsf(y[i][e] - yf) <= band;
        }
        if (M % 2 == 0) tie |= up && fabsf(a[i] - 0.5f) <= E2;
        lev[i] = __float_as_uint(m);
    }
    sym = __byte_perm(__byte_perm(lev[0], lev[1], 0x0040), __byte_perm(lev[2], lev[3], 0x0040), 0x5410);
    return __syncthreads_or(tie) == 0;
}

// The sweeps of a stream that the thresholds leave open: {length, this lane's four levels}.
template <int M>
__device__ __noinline__ uint2 drift_wide_sweeps_m(const EncTable& T, WideShared& W, int hs, int wib, uint32_t parity, float z0, float z1,
                                                  float z2, float z3, float s, float o, int cell) {
    const float z[4] = {z0, z1, z2, z3};
    return drift_wide_sweeps<M>(T, W, hs, wib, parity, z, s, o, cell);
}

// Drift on the CTA's stream: {length (0: known to be within the budget), this lane's four levels}.
template <int M, bool PAIR>
__device__ __forceinline__ uint2 drift_wide(const EncTable& T, WideShared& W, uint32_t* hist, int hs, int wib, uint32_t& parity,
                                            const float (&z)[4], float s, float o, float zmin, float zmax) {
    uint2 r = make_uint2(0u, 0u);
    int cell;
    if (PAIR) {
        uint32_t len;
        float clear;
        if (nearest_pairs<M>(T, z, s, o, zmin, zmax, r.y, len, clear)) {   // uniform: extrema and grid are stream-wide
            len = __reduce_add_sync(kFull, len);
            clear = dqdev::warp_min(clear);
            if ((threadIdx.x & 31) == 0) { W.len[parity][wib] = len; W.fmin[parity][wib] = clear; }
            __syncthreads();
            len = slots_add(W.len[parity], hs);
            clear = slots_min(W.fmin[parity], hs);
            parity ^= 1u;
            if (len <= ((uint32_t)T.budget_bits << 16) && clear > 0.f) return r;
        }
        r = drift_wide_pairs<M>(T, W, hs, wib, parity, z, s, o);
    } else if (!drift_wide_thresholds<M>(T, W, hist, hs, wib, parity, z, s, o, zmin, zmax, r.y, cell)) {
        r = drift_wide_sweeps_m<M>(T, W, hs, wib, parity, z[0], z[1], z[2], z[3], s, o, cell);
        __syncthreads();   // the slots of either parity are free again
    }
    return r;
}

// Refit of the CTA's stream: integer sums with a rounding check (refit_integers), binary64 sums where that is open.
// Both forms take each head's sums in the per-head order and add the heads in order.
__device__ __forceinline__ uint32_t wide_refit(WideShared& W, int hs, int wib, uint32_t& parity, const float (&z)[4], float zabs,
                                               uint32_t sym, float s, float o) {
    const int lane = threadIdx.x & 31, n = hs * kN;
    const RefitScale sc = refit_scale(zabs);
    {
        const RefitSums h = refit_sums(z, sc, sym);
        if (lane == 0) { W.sm[parity][wib] = h.Sm; W.smm[parity][wib] = h.Smm; W.ia[parity][wib] = h.SA; W.ib_lo[parity][wib] = h.SB & 0xffff; W.ib_hi[parity][wib] = h.SB >> 16; }
    }
    __syncthreads();
    const int Sm = slots_add(W.sm[parity], hs), Smm = slots_add(W.smm[parity], hs);
    // |SA| < 2^30; SB is up to 2^34: its halves are added apart
    const int SA = slots_add(W.ia[parity], hs);
    const long long SB = (long long)slots_add(W.ib_hi[parity], hs) * 65536 + slots_add(W.ib_lo[parity], hs);
    parity ^= 1u;
    const long long den = (long long)n * Smm - (long long)Sm * Sm;
    uint32_t hdr;
    if (sc.ok && refit_finish(sc, (float)n, (float)SA, (float)SB, (float)Sm, (float)den, hdr)) return hdr;
    double sa, sb;
    refit_sums_binary64(z, sym, sa, sb);
    __syncthreads();   // the previous stream's readers of W.sa .. are done
    if (lane == 0) { W.sa[wib] = sa; W.sb[wib] = sb; }
    __syncthreads();
    sa = W.sa[0]; sb = W.sb[0];
    for (int w = 1; w < hs; ++w) { sa = __dadd_rn(sa, W.sa[w]); sb = __dadd_rn(sb, W.sb[w]); }
    double sd = (double)s, od = (double)o;
    if (den != 0) {
        sd = __ddiv_rn(__dsub_rn(__dmul_rn((double)n, sb), __dmul_rn((double)Sm, sa)), (double)den);
        od = __ddiv_rn(__dsub_rn(sa, __dmul_rn(sd, (double)Sm)), (double)n);
    }
    return (uint32_t)__half_as_ushort(__double2half(sd)) | ((uint32_t)__half_as_ushort(__double2half(od)) << 16);
}

struct WideQuantised {
    uint32_t hdr0;      // s fp16 | o fp16 << 16
    uint32_t flags;     // 1: all-central fallback, 2: constant stream, 4: refit rejected
    uint32_t sym;       // this lane's four levels, one per byte
};

// Steps 2-6 of Algorithm 1 for the stream whose rotated, mean-free values the CTA holds: min-max grid, drift, refit,
// fp16 metadata, second drift.
template <int M, bool PAIR>
__device__ __forceinline__ WideQuantised wide_quantise(const EncTable& T, WideShared& W, uint32_t* hist, int hs, int wib,
                                                       uint32_t& parity, const float (&z)[4]) {
    const int lane = threadIdx.x & 31;
    float mx = dqdev::warp_max(fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3])));
    float mn = dqdev::warp_min(fminf(fminf(z[0], z[1]), fminf(z[2], z[3])));
    if (lane == 0) { W.fmax[parity][wib] = mx; W.fmin[parity][wib] = mn; }
    __syncthreads();
    mx = slots_max(W.fmax[parity], hs);
    mn = slots_min(W.fmin[parity], hs);
    parity ^= 1u;

    WideQuantised r;
    r.sym = T.central;
    r.flags = 0u;
    r.hdr0 = (uint32_t)__half_as_ushort(__float2half_rn(mn)) << 16;
    if (!(mx > mn)) { r.flags = 2u; return r; }   // uniform across the CTA: mx and mn are stream-wide
    const float o = mn;                                             // FitMinMax, Eq. (affine_token)
    const float s = __fdiv_rn(__fsub_rn(mx, mn), (float)(M - 1));
    uint32_t sym = drift_wide<M, PAIR>(T, W, hist, hs, wib, parity, z, s, o, mn, mx).y;
    uint32_t hdr = wide_refit(W, hs, wib, parity, z, fmaxf(fabsf(mn), fabsf(mx)), sym, s, o);
    float sf = __half2float(__ushort_as_half((unsigned short)(hdr & 0xffffu))), of = __half2float(__ushort_as_half((unsigned short)(hdr >> 16)));
    if (!(isfinite(sf) && sf > 0.0f && isfinite(of))) {
        const __half s16 = __float2half_rn(s), o16 = __float2half_rn(o);
        hdr = (uint32_t)__half_as_ushort(s16) | ((uint32_t)__half_as_ushort(o16) << 16);
        sf = __half2float(s16); of = __half2float(o16);
        r.flags = 4u;
    }
    if (!(sf > 0.0f)) { r.flags |= 2u; return r; }
    const uint2 d = drift_wide<M, PAIR>(T, W, hist, hs, wib, parity, z, sf, of, mn, mx);   // second Drift, fp16 grid
    r.hdr0 = hdr;
    if (d.x > ((uint32_t)T.budget_bits << 16)) r.flags |= 1u; else r.sym = d.y;
    return r;
}

// Words of a stream's symbol row: its levels (or pair indices, half as many), four per word, one word of padding so
// that lane = stream reads without conflicts.
__host__ __device__ inline int wide_sym_words(int hs) { return hs * (kN / 4) + 1; }
__host__ __device__ inline int wide_smem(int hs, int rec) {
    const int bytes = kWB * ((rec + 3) & ~3);   // emitted bytes, in the histogram's place once it is done with
    return kWB * wide_sym_words(hs) * 4 + (bytes > kCells * 4 ? bytes : kCells * 4);
}

// CTAs per SM the registers are held to (the shared memory allows four of them at the paper's record sizes).
constexpr int wide_min_blocks(int M, bool pair) { return pair ? 2 : M > 9 ? 2 : M > 4 ? 3 : 4; }

// One launch per tensor kind, as in dq_encode_batch.cu.
template <int M, bool PAIR>
__global__ void __launch_bounds__(DQ_MAX_STREAM_HEADS * 32, wide_min_blocks(M, PAIR))
dq_encode_wide_kernel(const __grid_constant__ DqDevTable TD, const __grid_constant__ DqPairEnc PD, const DqEncodeArgs a, int per, bool is_v,
                      bool second) {
    extern __shared__ __align__(16) uint8_t dyn[];
    __shared__ __align__(16) EncTable T;
    __shared__ __align__(16) WideShared W;
    __shared__ uint32_t s_hdr[kWB], s_flags[kWB], s_xs[kWB], s_k[kWB];
    __shared__ unsigned long long s_mi[kWB];     // rows of the mean arrays of a stream's first head
    __shared__ unsigned long long s_blk[kWB];    // word 0 of a stream's record
    __shared__ int s_pos[kWB];
    load_enc_table(T, TD, TD, PD, PD, is_v);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int hs = blockDim.x >> 5, groups = a.Hkv / hs;
    uint32_t* hist = reinterpret_cast<uint32_t*>(dyn);                     // [kCells] while quantising
    uint8_t* s_bytesT = dyn;                                               // [rec][kWB] while coding
    const int rec = TD.rec, rec_words = (rec + 3) >> 2;
    uint32_t* s_sym = hist + max(kCells, kWB * rec_words);                 // [per][wide_sym_words]
    const int sym_words = wide_sym_words(hs);
    if (!PAIR)
        for (int c = threadIdx.x * 4; c < kCells; c += blockDim.x * 4) *reinterpret_cast<uint4*>(hist + c) = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    if (!second) dqdev::pdl_wait_prior_grid();
    dqdev::pdl_launch_dependents();
    const bool has_mean = TD.has_mean, rope = !is_v && a.rope_style;
    const long long total = (long long)a.T * groups;
    const long long first = (long long)blockIdx.x * per;
    const int ns = (int)min((long long)per, total - first);
    if (threadIdx.x < ns) {   // where stream i's record, mean rows and position are
        const long long sid = first + threadIdx.x;
        const int t = (int)(sid / groups), grp = (int)(sid - (long long)t * groups), sl = a.slot[t];
        s_blk[threadIdx.x] = (unsigned long long)((is_v ? a.v_cont : a.k_cont) +
                             ((size_t)(sl / DQ_PAGE_TOKENS) * groups + grp) * ((size_t)rec_words * 64) + (size_t)(sl % DQ_PAGE_TOKENS) * 4);
        if (has_mean || rope) {
            const int ps = a.pos[t];
            s_pos[threadIdx.x] = ps;
            s_mi[threadIdx.x] = mean_row(a, a.seq_id[t], ps, grp * hs);
        }
    }
    __syncthreads();

    // quantise one stream after the other; the loads of the next one are issued before the work on this one
    const uint2* x = reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(is_v ? a.v_bf16 : a.k_bf16) + first * hs * kN) +
                     wib * (kN / 4) + lane;
    auto load = [&](int i, uint2& raw, uint32_t& q4, float& sc) {
        if (i >= ns) return;
        raw = x[(size_t)i * hs * (kN / 4)];
        if (has_mean) {
            const size_t mi = s_mi[i] + wib;
            q4 = *reinterpret_cast<const uint32_t*>(a.mean_q + mi * kN + 4 * lane);
            sc = a.mean_scale[mi];
        }
    };
    uint2 raw = make_uint2(0u, 0u);
    uint32_t q4 = 0u, parity = 0u;
    float sc = 0.f;
    load(0, raw, q4, sc);
    for (int i = 0; i < ns; ++i) {
        float z[4];
        unpack_bf16x4(raw, z);
        if (rope)
            warp_rope128(z, lane, a.rope_cos + (size_t)s_pos[i] * 64, a.rope_sin + (size_t)s_pos[i] * 64, a.rope_style);
        if (T.rotate) warp_fwht128(z, lane);
        if (has_mean) {
            if (a.mean_mode == DQ_MEAN_REUSE && s_pos[i] % DQ_WINDOW_TOKENS == 0) carry_mean(a, s_mi[i] + wib, s_pos[i], lane, q4, sc);
            remove_mean(z, q4, sc);
        }
        load(i + 1, raw, q4, sc);
        const WideQuantised q = wide_quantise<M, PAIR>(T, W, hist, hs, wib, parity, z);
        uint32_t* row = s_sym + i * sym_words;
        if (PAIR) {   // the lane's two pair indices u = a M + b
            const uint32_t u0 = (q.sym & 0xffu) * M + ((q.sym >> 8) & 0xffu), u1 = ((q.sym >> 16) & 0xffu) * M + (q.sym >> 24);
            reinterpret_cast<uint16_t*>(row)[wib * 32 + lane] = (uint16_t)(u0 | (u1 << 8));
        } else {
            row[wib * 32 + lane] = q.sym;
        }
        if (threadIdx.x == 0) { s_hdr[i] = q.hdr0; s_flags[i] = q.flags; }
    }
    __syncthreads();
    if (wib == 0 && lane < ns) {   // rANS, Eq. (rans) Enc on the symbols from the last one back; lane = stream
        uint32_t xs = kL;
        const uint32_t dst0 = dqdev::smem_addr(s_bytesT) + lane;
        uint32_t dst = dst0;   // the budget test keeps the bytes of a stream below rec - 8
        const uint32_t* row = s_sym + lane * sym_words;
        rans_encode_row<kWB>(T.enc, row, hs * (PAIR ? kN / 8 : kN / 4), xs, dst);
        const uint32_t k = (dst - dst0) / kWB;
        s_xs[lane] = xs;
        s_k[lane] = k;
        if (a.status) {
            const uint32_t f = s_flags[lane];
            if (f & 1u) atomicAdd(a.status + 0, 1u);
            if (f & 2u) atomicAdd(a.status + 1, 1u);
            if (f & 4u) atomicAdd(a.status + 2, 1u);
            atomicMax(a.status + 3, 8u + k);
        }
    }
    __syncthreads();
    // records out, a word of four bytes per thread: header, state, then the k bytes emitted last first, then zeros
    for (int idx = threadIdx.x; idx < ns * rec_words; idx += blockDim.x) {
        const int wi = idx / ns, si = idx - wi * ns;   // consecutive threads: consecutive streams, mostly adjacent slots
        uint32_t v = wi == 0 ? s_hdr[si] : s_xs[si];
        if (wi >= 2) {
            v = 0u;
            const int at = (int)s_k[si] - 1 - (4 * wi - 8);
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if (at - b >= 0) v |= (uint32_t)s_bytesT[(at - b) * kWB + si] << (8 * b);
        }
        reinterpret_cast<uint32_t*>(s_blk[si])[(size_t)wi * 16] = v;
    }
    if (second) dqdev::pdl_wait_prior_grid();   // the first kind's kernel: whoever waits for this one may read both
}

using WideKernel = void (*)(DqDevTable, DqPairEnc, DqEncodeArgs, int, bool, bool);

template <bool PAIR>
WideKernel kernel_for(int M) {
    switch (M) {
#define DQ_LEVELS_CASE(M_) case M_: return dq_encode_wide_kernel<M_, PAIR>;
        DQ_LEVELS_CASE(2) DQ_LEVELS_CASE(3) DQ_LEVELS_CASE(4) DQ_LEVELS_CASE(5) DQ_LEVELS_CASE(6) DQ_LEVELS_CASE(7)
        DQ_LEVELS_CASE(8) DQ_LEVELS_CASE(9)
        default: break;
    }
    if constexpr (!PAIR) {
        switch (M) {
            DQ_LEVELS_CASE(10) DQ_LEVELS_CASE(11) DQ_LEVELS_CASE(12) DQ_LEVELS_CASE(13) DQ_LEVELS_CASE(14) DQ_LEVELS_CASE(15)
            DQ_LEVELS_CASE(16)
            default: break;
        }
    }
#undef DQ_LEVELS_CASE
    return nullptr;
}

}  // namespace

// Streams per CTA: enough CTAs to fill the GPU (three of them per SM) before streams share one, as a CTA's serial
// coding pass costs the same for 1 and for 32 streams.
cudaError_t dq_launch_encode_wide(const DqDevTable& tk, const DqDevTable& tv, const DqPairEnc& pk, const DqPairEnc& pv,
                                  const DqEncodeArgs& a, int per, cudaStream_t st) {
    const long long streams = (long long)a.T * (a.Hkv / tk.hs);
    if (per <= 0) {
        const long long resident = 3LL * 148 / ((a.do_k && a.do_v) ? 2 : 1);
        per = (int)((streams + resident - 1) / resident);
    }
    per = per < 1 ? 1 : per > kWB ? kWB : per;
    bool second = false;
    for (int kind = 0; kind < 2; ++kind) {
        if (kind == 0 ? !a.do_k : !a.do_v) continue;
        const DqDevTable& t = kind == 0 ? tk : tv;
        const auto kernel = t.pair ? kernel_for<true>(t.M) : kernel_for<false>(t.M);
        if (!kernel) return cudaErrorInvalidValue;
        const int smem = wide_smem(t.hs, t.rec);
        cudaError_t e = dq_allow_smem(reinterpret_cast<const void*>(kernel), smem);
        if (e != cudaSuccess) return e;
        e = dq_launch_pdl(kernel, dim3((unsigned)((streams + per - 1) / per)), dim3(t.hs * 32), (size_t)smem, st, t, kind == 0 ? pk : pv, a,
                          per, kind == 1, second);
        if (e != cudaSuccess) return e;
        second = true;
    }
    return cudaSuccess;
}
