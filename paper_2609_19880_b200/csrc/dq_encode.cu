// Encoder kernels: window means of keys and the one-warp-per-stream encoder
// (Fig. 1 pipeline; Algorithm 1; Sec. 4.5 "Encoding").  Compiled with -fmad=false: every
// floating-point operation below is a single IEEE operation in a fixed order so that the
// records are reproducible bit for bit.
#include "dq_encode.cuh"

using namespace dqenc;

namespace {

// ------------------------------------------------------------------ window means

// Mean of the run that starts at call token t0, for KV head h, by one warp.
__device__ __forceinline__ void means_of_run(const uint16_t* __restrict__ k, int T, int Hkv, int rotate,
                                             const int32_t* __restrict__ seq_id, const int32_t* __restrict__ pos,
                                             int8_t* __restrict__ mean_q, float* __restrict__ mean_scale, int Wmax,
                                             const float* __restrict__ rope_cos, const float* __restrict__ rope_sin,
                                             int rope_style, int t0, int h, int lane) {
    const int s = seq_id[t0], w = pos[t0] / DQ_WINDOW_TOKENS;
    // length of the run: 32 candidates per round, lanes in parallel (the sums below stay sequential)
    int cnt = 0;
    for (int base = t0; base < T; base += 32) {
        const int tt = base + lane;
        const bool same = tt < T && seq_id[tt] == s && pos[tt] / DQ_WINDOW_TOKENS == w;
        const unsigned m = __ballot_sync(kFull, same);
        if (m != kFull) { cnt += __ffs((int)~m) - 1; break; }
        cnt += 32;
    }
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    // Independent loads in flight (a window of 128 tokens in four waits, with the rotary tables in sixteen); the
    // additions keep token order.
    if (!rope_style) {
        constexpr int kAhead = 32;
        for (int tb = t0; tb < t0 + cnt; tb += kAhead) {
            uint2 raw[kAhead];
#pragma unroll
            for (int u = 0; u < kAhead; ++u)
                raw[u] = *reinterpret_cast<const uint2*>(k + ((size_t)min(tb + u, t0 + cnt - 1) * Hkv + h) * kN + 4 * lane);
            const int n = t0 + cnt - tb;
#pragma unroll
            for (int u = 0; u < kAhead; ++u)
                if (u < n) {
                    float kt[4];
                    unpack_bf16x4(raw[u], kt);
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[e] = __fadd_rn(acc[e], kt[e]);
                }
        }
    } else {
        constexpr int kAhead = 8;
        const int per = rope_style == DQ_ROPE_HALF ? 4 * (lane & 15) : 2 * lane;   // this lane's place in a position's 64 angles
        for (int tb = t0; tb < t0 + cnt; tb += kAhead) {
            uint2 raw[kAhead];
            float4 cs[kAhead], sn[kAhead];
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const int tt = min(tb + u, t0 + cnt - 1);
                raw[u] = *reinterpret_cast<const uint2*>(k + ((size_t)tt * Hkv + h) * kN + 4 * lane);
                const float* c = rope_cos + (size_t)pos[tt] * 64 + per;
                const float* n = rope_sin + (size_t)pos[tt] * 64 + per;
                if (rope_style == DQ_ROPE_HALF) {
                    cs[u] = *reinterpret_cast<const float4*>(c);
                    sn[u] = *reinterpret_cast<const float4*>(n);
                } else {
                    const float2 c2 = *reinterpret_cast<const float2*>(c), n2 = *reinterpret_cast<const float2*>(n);
                    cs[u] = make_float4(c2.x, c2.y, 0.f, 0.f);
                    sn[u] = make_float4(n2.x, n2.y, 0.f, 0.f);
                }
            }
            const int n = t0 + cnt - tb;
#pragma unroll
            for (int u = 0; u < kAhead; ++u)
                if (u < n) {
                    float kt[4];
                    unpack_bf16x4(raw[u], kt);
                    warp_rope128(kt, lane, cs[u], sn[u], rope_style);
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[e] = __fadd_rn(acc[e], kt[e]);
                }
        }
    }
    const int t = t0 + cnt;
    const float inv = __fdiv_rn(1.0f, (float)(t - t0));
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[e] = __fmul_rn(acc[e], inv);
    if (rotate) warp_fwht128(acc, lane);
    float amax = fmaxf(fmaxf(fabsf(acc[0]), fabsf(acc[1])), fmaxf(fabsf(acc[2]), fabsf(acc[3])));
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) amax = fmaxf(amax, __shfl_xor_sync(kFull, amax, d));
    const float sc = __fdiv_rn(amax, 127.0f);
    uint32_t packed = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        float q = 0.f;
        if (sc != 0.f) q = fminf(fmaxf(rintf(__fdiv_rn(acc[e], sc)), -127.f), 127.f);
        packed |= ((uint32_t)(int)q & 0xffu) << (8 * e);
    }
    const size_t mi = ((size_t)s * Wmax + w) * Hkv + h;
    *reinterpret_cast<uint32_t*>(mean_q + mi * kN + 4 * lane) = packed;
    if (lane == 0) mean_scale[mi] = sc;
}

// DQ_MEAN_COMPUTE.  A run is a maximal range of consecutive call tokens with the same
// (seq_id, pos / 128).  A CTA looks at kMeansTokens consecutive call tokens, lists those that
// start a run, and its warps take the (run, KV head) pairs in turn.  Sequential binary32 sum over
// the run, times 1/count, rotated, quantised to INT8 with one scale (max |mean| / 127).
constexpr int kMeansTokens = 128;
__global__ void __launch_bounds__(256)
dq_means_compute_kernel(const uint16_t* __restrict__ k, int T, int Hkv, int rotate,
                        const int32_t* __restrict__ seq_id, const int32_t* __restrict__ pos,
                        int8_t* __restrict__ mean_q, float* __restrict__ mean_scale, int Wmax,
                        const float* __restrict__ rope_cos, const float* __restrict__ rope_sin, int rope_style) {
    __shared__ int s_first[kMeansTokens];
    __shared__ int s_n;
    const int lane = threadIdx.x & 31;
    dqdev::pdl_launch_dependents();
    if (threadIdx.x == 0) s_n = 0;
    dqdev::pdl_wait_prior_grid();
    __syncthreads();
    {
        const long long tt = (long long)blockIdx.x * kMeansTokens + threadIdx.x;
        if (threadIdx.x < kMeansTokens && tt < T) {
            const int t = (int)tt;
            const bool first = t == 0 || seq_id[t - 1] != seq_id[t] || pos[t - 1] / DQ_WINDOW_TOKENS != pos[t] / DQ_WINDOW_TOKENS;
            if (first) s_first[atomicAdd(&s_n, 1)] = t;
        }
    }
    __syncthreads();
    const int tasks = s_n * Hkv;
    for (int task = threadIdx.x >> 5; task < tasks; task += (int)(blockDim.x >> 5))
        means_of_run(k, T, Hkv, rotate, seq_id, pos, mean_q, mean_scale, Wmax, rope_cos, rope_sin, rope_style,
                     s_first[task / Hkv], task % Hkv, lane);
}

// ---------------------------------------------------------------------- encoder

constexpr int kEncWarps = 8;
#ifndef DQ_STEP_ENC_WARPS
#define DQ_STEP_ENC_WARPS 16
#endif

// quantise_values for the table's number of levels: one call, everything inside it inlined.
template <int M, bool PAIR>
__device__ __noinline__ StreamQuantised quantise_m(const EncTable& T, float z0, float z1, float z2, float z3) {
    const float z[4] = {z0, z1, z2, z3};
    return quantise_values<M, PAIR, true>(T, z);
}
template <bool PAIR>
__device__ __forceinline__ StreamQuantised quantise_any(const EncTable& T, const float (&z)[4]) {
    switch (T.M) {   // uniform across the CTA
#define DQ_LEVELS_CASE(M_) case M_: return quantise_m<M_, PAIR>(T, z[0], z[1], z[2], z[3]);
        DQ_LEVELS_CASE(2) DQ_LEVELS_CASE(3) DQ_LEVELS_CASE(4) DQ_LEVELS_CASE(5) DQ_LEVELS_CASE(6) DQ_LEVELS_CASE(7)
        DQ_LEVELS_CASE(8) default: break;
    }
    if constexpr (PAIR) {
        return quantise_m<9, PAIR>(T, z[0], z[1], z[2], z[3]);
    } else {
        switch (T.M) {
            DQ_LEVELS_CASE(9) DQ_LEVELS_CASE(10) DQ_LEVELS_CASE(11) DQ_LEVELS_CASE(12) DQ_LEVELS_CASE(13) DQ_LEVELS_CASE(14)
            DQ_LEVELS_CASE(15) default: return quantise_m<16, PAIR>(T, z[0], z[1], z[2], z[3]);
        }
    }
#undef DQ_LEVELS_CASE
}

// Steps 1-6 for the stream (token t, KV head h): rotary embedding when asked, rotation, mean removal, then the above.
template <bool PAIR>
__device__ __forceinline__ StreamQuantised quantise_stream(const EncTable& T, const DqEncodeArgs& a, bool is_v, int t, int h,
                                                           int lane) {
    const uint16_t* x = static_cast<const uint16_t*>(is_v ? a.v_bf16 : a.k_bf16);
    float z[4];
    unpack_bf16x4(*reinterpret_cast<const uint2*>(x + ((size_t)t * a.Hkv + h) * kN + 4 * lane), z);
    if (!is_v && a.rope_style)
        warp_rope128(z, lane, a.rope_cos + (size_t)tok_pos(a, t) * 64, a.rope_sin + (size_t)tok_pos(a, t) * 64, a.rope_style);
    uint32_t q4 = 0u;
    float sc = 0.f;
    if (T.has_mean) {
        const int ps = tok_pos(a, t);
        const size_t mi = mean_row(a, tok_seq(a, t), ps, h);
        if (a.mean_mode == DQ_MEAN_REUSE && ps % DQ_WINDOW_TOKENS == 0) {
            carry_mean(a, mi, ps, lane, q4, sc);
        } else {
            sc = a.mean_scale[mi];
            q4 = *reinterpret_cast<const uint32_t*>(a.mean_q + mi * kN + 4 * lane);
        }
    }
    if (T.rotate) warp_fwht128(z, lane);
    if (T.has_mean) remove_mean(z, q4, sc);
    return quantise_any<PAIR>(T, z);
}

// One warp per stream (token, KV head); lane l owns elements 4l .. 4l+3.  blockIdx.y selects
// the tensor kind when keys and values are encoded by one launch.
// MINB CTAs per SM: 2 leaves every thread 128 registers (lowest latency: the single-token step), 4 trades a
// few spills for twice the resident warps (throughput: prefill, bulk encodes).
// WARPS streams per CTA: 8 normally; the decode step uses 16 (512 threads at full register budget) so that its
// 2 B Hkv streams occupy few SMs while the attention kernel runs on all the others.
template <int MINB, int WARPS, bool PAIR>
__global__ void __launch_bounds__(WARPS * 32, MINB)
dq_encode_kernel(const __grid_constant__ DqDevTable TK, const __grid_constant__ DqDevTable TV,
                 const __grid_constant__ DqPairEnc PK, const __grid_constant__ DqPairEnc PV, const DqEncodeArgs a) {
    __shared__ __align__(16) EncTable T;
    __shared__ uint8_t s_bytes[WARPS][DQ_MAX_REC_BYTES];
    __shared__ __align__(4) uint8_t s_sym[WARPS][kN];
    // Decode-step mode: the kernels after this one start while it runs and take their own launch as proof
    // that everything before this kernel has finished, so the trigger comes after the wait (and after the
    // hand-over words are cleared).  Otherwise: trigger first, so that the next kernel's launch overlaps this one.
    if (!a.step_flags) dqdev::pdl_launch_dependents();
    const bool is_v = a.do_k ? (blockIdx.y == 1) : true;
    load_enc_table(T, TK, TV, PK, PV, is_v);
    __syncthreads();
    dqdev::pdl_wait_prior_grid();   // inputs and the cache may be written / read by the previous kernel
    if (a.step_flags) {
        if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 4) {
            a.step_flags[threadIdx.x] = 0;
            __threadfence();
        }
        __syncthreads();
        dqdev::pdl_launch_dependents();
    }
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const long long wid = (long long)blockIdx.x * WARPS + wib;
    if (wid >= (long long)a.T * a.Hkv) return;
    int t, h;
    split_stream(a, wid, t, h);
    const int Hkv = a.Hkv;
    if (tok_pos(a, t) < 0) return;   // decode-step mode: an empty sequence has no new token
    const int sl = a.slot[t];        // needed at the end, on its way meanwhile
    uint8_t* cont = is_v ? a.v_cont : a.k_cont;

    const StreamQuantised sq = quantise_stream<PAIR>(T, a, is_v, t, h, lane);
    // rANS, Eq. (rans) Enc on symbols 127 .. 0 so that decoding runs forward.  Every lane
    // carries the same state (the symbols come from shared memory).
    // (paired symbols: the lane's two pair indices u = a M + b; the coder then runs over 64 symbols)
    if (PAIR) {
        const uint32_t M = (uint32_t)T.M;
        const uint32_t u0 = (sq.sym & 0xffu) * M + ((sq.sym >> 8) & 0xffu), u1 = ((sq.sym >> 16) & 0xffu) * M + (sq.sym >> 24);
        *reinterpret_cast<uint16_t*>(&s_sym[wib][2 * lane]) = (uint16_t)(u0 | (u1 << 8));
    } else {
        *reinterpret_cast<uint32_t*>(&s_sym[wib][4 * lane]) = sq.sym;
    }
    __syncwarp();
    uint32_t xs = 1u << (T.sigma - 9);   // L: 2^23, or 2^15 with the 24-bit state
    const uint32_t bytes_addr = dqdev::smem_addr(s_bytes[wib]);
    uint32_t dst = bytes_addr;           // every lane stores the same bytes to the same place
    rans_encode_row<1>(T.enc, reinterpret_cast<const uint32_t*>(s_sym[wib]), (PAIR ? kN / 2 : kN) / 4, xs, dst);
    const int k = (int)(dst - bytes_addr);
    __syncwarp();
    asm volatile("" ::: "memory");
    const uint32_t hdr0 = sq.hdr0;
    uint8_t* rec = cont + (((size_t)(sl / DQ_PAGE_TOKENS) * Hkv + h) * DQ_PAGE_TOKENS +
                           (size_t)(sl % DQ_PAGE_TOKENS)) * T.rec;
    const int pay = 4 + (T.sigma >> 3);              // first payload byte: after (s, o) and the final state
    const int used = min(pay + k, T.rec);            // the budget test keeps pay + k <= rec
    for (int i = lane; i < T.rec; i += 32) {
        uint8_t v = 0;
        if (i < 4) v = (uint8_t)(hdr0 >> (8 * i));
        else if (i < pay) v = (uint8_t)(xs >> (8 * (i - 4)));
        else if (i < used) v = s_bytes[wib][k - 1 - (i - pay)];
        rec[i] = v;
    }
    if (a.status && lane == 0) {
        if (sq.flags & 1u) atomicAdd(a.status + 0, 1u);
        if (sq.flags & 2u) atomicAdd(a.status + 1, 1u);
        if (sq.flags & 4u) atomicAdd(a.status + 2, 1u);
        atomicMax(a.status + 3, (uint32_t)(pay + k));
    }
}


}  // namespace

cudaError_t dq_launch_means(const DqDevTable& tk, const void* k_bf16, int T, int Hkv,
                            const int32_t* seq_id, const int32_t* pos, int8_t* mean_q,
                            float* mean_scale, int max_windows, int mode, const float* rope_cos,
                            const float* rope_sin, int rope_style, cudaStream_t st) {
    if (T == 0 || Hkv == 0) return cudaSuccess;
    if (mode != DQ_MEAN_COMPUTE) return cudaSuccess;  // carry-forward is done by the encoder warps
    const unsigned blocks = (unsigned)((T + kMeansTokens - 1) / kMeansTokens);
    return dq_launch_pdl(dq_means_compute_kernel, dim3(blocks), dim3(256), 0, st, (const uint16_t*)k_bf16, T, Hkv, tk.rotate, seq_id, pos,
                         mean_q, mean_scale, max_windows, rope_cos, rope_sin, rope_style);
}

// Smallest number of streams for which a call goes to the batch kernels (32 streams per CTA); the
// option DQ_OPT_ENCODE_BATCH_MIN replaces the default (0 sends every call there).
static long long batch_min_streams(long long dflt) { return dq_opt_encode_batch_min(dflt); }

cudaError_t dq_launch_encode(const DqDevTable& tk, const DqDevTable& tv, const DqPairEnc& pk, const DqPairEnc& pv,
                             const DqEncodeArgs& args, cudaStream_t st) {
    DqEncodeArgs a = args;
    const long long warps = (long long)a.T * a.Hkv;
    // umulhi(n, ceil(2^32 / d)) = n / d for every n < 2^32 / d
    a.hkv_magic = (a.Hkv > 1 && warps < (1LL << 32) / a.Hkv) ? (uint32_t)(((1ull << 32) + a.Hkv - 1) / a.Hkv) : 0u;
    if (warps == 0 || (!a.do_k && !a.do_v)) return cudaSuccess;
    if (tk.hs > 1) {   // token-wide streams; the option's batches are CTAs of 32 streams, below it one stream per CTA
        const long long batch_min = batch_min_streams(-1);
        return dq_launch_encode_wide(tk, tv, pk, pv, a, batch_min < 0 ? 0 : warps / tk.hs >= batch_min ? 32 : 1, st);
    }
    const unsigned blocks = (unsigned)((warps + kEncWarps - 1) / kEncWarps);
    const bool pair = tk.pair != 0;   // the caller has checked that both tables agree
    const dim3 kinds(1, (a.do_k && a.do_v) ? 2 : 1);
    // One warp per stream while the call's streams are resident at once (two CTAs of eight warps per SM); beyond that
    // the batch kernel, whose coding pass is shared.  The option's batches are CTAs of 32 streams.
    const long long batch_min = batch_min_streams(-1);
    if (!a.step_flags && (batch_min < 0 ? warps * kinds.y > 2LL * 148 * kEncWarps : warps >= batch_min))
        return dq_launch_encode_batch(tk, tv, pk, pv, a, batch_min < 0 ? 0 : kDqEncodeBatchStreams, st);
    if (a.step_flags) {   // decode step: big CTAs, so that few SMs are kept from the attention kernel
        constexpr int kStepWarps = DQ_STEP_ENC_WARPS;
        return dq_launch_pdl(pair ? dq_encode_kernel<1, kStepWarps, true> : dq_encode_kernel<1, kStepWarps, false>,
                             dim3((unsigned)((warps + kStepWarps - 1) / kStepWarps), kinds.y), dim3(kStepWarps * 32), 0, st, tk, tv, pk, pv, a);
    }
    return dq_launch_pdl(pair ? dq_encode_kernel<2, kEncWarps, true> : dq_encode_kernel<2, kEncWarps, false>, dim3(blocks, kinds.y),
                         dim3(kEncWarps * 32), 0, st, tk, tv, pk, pv, a);
}
