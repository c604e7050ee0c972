// Export of records (dq_decode_tokens): Algorithm 2 with lane = stream out of shared memory, then the dequantised values
// xhat = fma(m, s, o) (+ window mean for keys, Appendix A) and symbols written a head row per warp instruction.
// Bound by the rANS chain's latency while a call has few streams (128 steps of about 90 cycles) and by the 640 bytes
// written per stream when it has many; one thread per stream writing its own row ran at 5 % of the copy bandwidth.
#include <cuda_fp16.h>

#include "dq_device.cuh"
#include "dq_internal.h"

namespace {

constexpr int kExportWarps = 4;
constexpr int kSymRow = 33;   // words of a stream's symbol row: 128 bytes + pad

struct ExportArgs {
    const uint8_t* cont;
    const int8_t* mean_q;
    const float* mean_scale;
    const int32_t* seq_id;
    const int32_t* pos;
    const int32_t* slot;
    uint8_t* symbols;
    float* dequant;
    int Wmax, n_tok, Hkv;
};

constexpr int kLutCopies = 8;   // copies of the decode table, lane & 7 picks one: about two lanes per bank instead of 3.5

// Decode table with integer symbols: f << 24 | symbol << 8 | (z - c); pairs: symbol = b << 4 | a.
__device__ __forceinline__ void fill_lut(uint32_t* lut, const DqDevTable& T) {
    auto level = [](uint32_t bits) { return (uint32_t)(int)__half2float(__ushort_as_half((unsigned short)bits)); };
    for (int z = threadIdx.x; z < 256; z += blockDim.x) {
        const uint32_t e = T.lut[z];
        const uint32_t v = T.pair ? ((e << 8) & 0xff000000u) | level((e >> 16) & 0xff00u) << 12 | level(e & 0xff00u) << 8 | (e & 255u)
                                  : (e & 0xff000000u) | level((e >> 8) & 0xffffu) << 8 | (e & 255u);
#pragma unroll
        for (int c = 0; c < kLutCopies; ++c) lut[z * kLutCopies + c] = v;
    }
}

// Four rANS symbols packed into a word.  A symbol takes at most one byte: window(i) gives bytes i .. i + 3 of the record,
// fetched before the serial chain needs them; a malformed record stops taking bytes at its end.
template <typename Window>
__device__ __forceinline__ uint32_t decode4(const uint32_t* lut, uint32_t& x, int& ptr, int rec, uint32_t L, Window window) {
    uint32_t sym = 0, win = window(ptr);
    const int left = rec - ptr;
    int used = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t e = lut[(x & 255u) * kLutCopies];
        x = (e >> 24) * (x >> 8) + (e & 255u);
        const bool take = x < L && used < left;
        x = take ? __byte_perm(x, win, 0x2104) : x;
        win = take ? win >> 8 : win;
        used += take ? 1 : 0;
        sym |= ((e >> 8) & 255u) << (8 * i);
    }
    ptr += used;
    return sym;
}

// The four levels of positions 4 lane .. 4 lane + 3 from a symbol row.
template <bool PAIR>
__device__ __forceinline__ uint32_t row_levels(const uint32_t* row, int lane) {
    if (!PAIR) return row[lane];
    const uint32_t two = reinterpret_cast<const uint16_t*>(row)[lane];   // pairs 2 lane, 2 lane + 1
    const uint32_t lo = two & 0x0f0fu, hi = (two >> 4) & 0x0f0fu;        // levels of the even / odd values
    return (lo & 255u) | (hi & 255u) << 8 | (lo >> 8) << 16 | (hi >> 8) << 24;
}

constexpr unsigned long long kNoMean = ~0ull;

// Row of the mean arrays for (token t, head h), kNoMean without one.
__device__ __forceinline__ unsigned long long mean_row(const DqDevTable& T, const ExportArgs& a, int t, int h) {
    if (!T.has_mean || !a.mean_q) return kNoMean;
    return ((unsigned long long)a.seq_id[t] * a.Wmax + a.pos[t] / DQ_WINDOW_TOKENS) * a.Hkv + h;
}

struct MeanPiece {
    uint32_t q4;   // four INT8 means
    float scale;
};
__device__ __forceinline__ MeanPiece load_mean(const ExportArgs& a, unsigned long long mi, int lane) {
    MeanPiece m{0u, 0.f};
    if (mi == kNoMean) return m;
    m.scale = __ldg(a.mean_scale + mi);
    const int8_t* p = a.mean_q + mi * DQ_HEAD_DIM + 4 * lane;
    if ((reinterpret_cast<uintptr_t>(a.mean_q) & 3u) == 0) m.q4 = __ldg(reinterpret_cast<const uint32_t*>(p));
    else
        for (int e = 0; e < 4; ++e) m.q4 |= (uint32_t)(uint8_t)p[e] << (8 * e);
    return m;
}

// Symbols and dequantised values of (token, head) row `at` / 128 by one warp.
template <bool PAIR>
__device__ __forceinline__ void write_row(const ExportArgs& a, const uint32_t* row, size_t at, bool has_mean, const MeanPiece& m, float s,
                                          float o, int lane) {
    const uint32_t m4 = row_levels<PAIR>(row, lane);
    at += 4 * lane;
    if (a.symbols) {
        if ((reinterpret_cast<uintptr_t>(a.symbols) & 3u) == 0) *reinterpret_cast<uint32_t*>(a.symbols + at) = m4;
        else
            for (int e = 0; e < 4; ++e) a.symbols[at + e] = (uint8_t)(m4 >> (8 * e));
    }
    if (!a.dequant) return;
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        v[e] = __fmaf_rn((float)((m4 >> (8 * e)) & 255u), s, o);
        if (has_mean) v[e] = __fadd_rn(v[e], __fmul_rn(m.scale, (float)(int)(int8_t)(m.q4 >> (8 * e))));
    }
    if ((reinterpret_cast<uintptr_t>(a.dequant) & 15u) == 0) *reinterpret_cast<float4*>(a.dequant + at) = make_float4(v[0], v[1], v[2], v[3]);
    else
        for (int e = 0; e < 4; ++e) a.dequant[at + e] = v[e];
}

// Per token-head streams: every warp takes 32 consecutive streams on its own.
template <bool PAIR>
__global__ void __launch_bounds__(kExportWarps * 32)
dq_decode_tokens_kernel(const __grid_constant__ DqDevTable T, const ExportArgs a) {
    extern __shared__ __align__(16) uint32_t dyn[];
    __shared__ uint32_t lut_all[256 * kLutCopies];
    fill_lut(lut_all, T);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t* lut = lut_all + (lane & (kLutCopies - 1));
    const int rec = T.rec, row_words = ((rec + 10) >> 2) | 1;   // aligned words around a record and 4 bytes more; odd: lanes spread over the banks
    uint32_t* recs = dyn + warp * 32 * (row_words + kSymRow);
    uint32_t* syms = recs + 32 * row_words;
    const long long total = (long long)a.n_tok * a.Hkv, first = ((long long)blockIdx.x * kExportWarps + warp) * 32;
    const int ns = (int)min(32LL, total - first);
    if (ns <= 0) return;
    // lane = stream: where its record is
    unsigned long long src = 0, mi = kNoMean;
    if (lane < ns) {
        int t, h;
        t = (int)((first + lane) / a.Hkv);
        h = (int)(first + lane - (long long)t * a.Hkv);
        const int sl = a.slot[t];
        src = (unsigned long long)(a.cont + (((size_t)(sl / DQ_PAGE_TOKENS) * a.Hkv + h) * DQ_PAGE_TOKENS + (size_t)(sl % DQ_PAGE_TOKENS)) * rec);
        mi = mean_row(T, a, t, h);
    }
#pragma unroll 8
    for (int i = 0; i < ns; ++i) {   // records into shared memory, a record's aligned words per warp instruction
        const unsigned long long p = __shfl_sync(0xffffffffu, src, i);
        const uint32_t* w = reinterpret_cast<const uint32_t*>(p & ~3ull);
        const int words = (int)((p & 3ull) + rec + 3) >> 2;
        for (int k = lane; k < words; k += 32) recs[i * row_words + k] = __ldg(w + k);
    }
    __syncwarp();
    float s = 0.f, o = 0.f;
    if (lane < ns) {
        const uint8_t* r = reinterpret_cast<const uint8_t*>(recs + lane * row_words) + (src & 3ull);
        s = __half2float(__ushort_as_half((unsigned short)(r[0] | (r[1] << 8))));
        o = __half2float(__ushort_as_half((unsigned short)(r[2] | (r[3] << 8))));
        // final state: sigma / 8 bytes, little-endian; the state interval starts at L = 2^(sigma - 9)
        uint32_t x = (uint32_t)r[4] | ((uint32_t)r[5] << 8) | ((uint32_t)r[6] << 16);
        if (T.sigma == 32) x |= (uint32_t)r[7] << 24;
        int ptr = 4 + (T.sigma >> 3);
        const uint32_t L = 1u << (T.sigma - 9);
        const uint32_t base = dqdev::smem_addr(r);
        auto window = [&](int i) -> uint32_t { return dqdev::lds32_unaligned(base + i); };
#pragma unroll 1
        for (int j = 0; j < (PAIR ? 16 : 32); ++j) syms[lane * kSymRow + j] = decode4(lut, x, ptr, rec, L, window);
    }
    __syncwarp();
    constexpr int kRows = 8;   // mean loads in flight
    for (int i0 = 0; i0 < ns; i0 += kRows) {
        MeanPiece m[kRows];
        bool hm[kRows];
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
            const unsigned long long mu = __shfl_sync(0xffffffffu, mi, min(i0 + u, ns - 1));
            hm[u] = mu != kNoMean;
            m[u] = load_mean(a, mu, lane);
        }
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
            const int i = i0 + u;
            const float su = __shfl_sync(0xffffffffu, s, i & 31), ou = __shfl_sync(0xffffffffu, o, i & 31);
            if (i < ns) write_row<PAIR>(a, syms + i * kSymRow, (size_t)(first + i) * DQ_HEAD_DIM, hm[u], m[u], su, ou, lane);
        }
    }
}

// Token-wide streams: a CTA takes 32 consecutive streams (token, group of hs heads).  Warp 0 decodes, lane =
// stream, a head's 128 values at a time into one of two symbol tiles; the other warps write the head before.
template <bool PAIR>
__global__ void __launch_bounds__(kExportWarps * 32)
dq_decode_tokens_wide_kernel(const __grid_constant__ DqDevTable T, const ExportArgs a) {
    extern __shared__ __align__(16) uint32_t dyn[];
    __shared__ uint32_t lut_all[256 * kLutCopies], tile[2][32 * kSymRow];
    __shared__ int s_t[32], s_grp[32];
    __shared__ float s_s[32], s_o[32];
    __shared__ unsigned long long s_src[32], s_mi[32];
    fill_lut(lut_all, T);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t* lut = lut_all + (lane & (kLutCopies - 1));
    const int groups = a.Hkv / T.hs, rw = T.rec_words;
    const long long total = (long long)a.n_tok * groups, first = (long long)blockIdx.x * 32;
    const int ns = (int)min(32LL, total - first);
    if (threadIdx.x < ns) {
        const int t = (int)((first + lane) / groups), grp = (int)(first + lane - (long long)t * groups), sl = a.slot[t];
        s_t[lane] = t;
        s_grp[lane] = grp;
        s_mi[lane] = mean_row(T, a, t, 0);
        s_src[lane] = (unsigned long long)(a.cont + ((size_t)(sl / DQ_PAGE_TOKENS) * groups + grp) * ((size_t)rw * 64) + (size_t)(sl % DQ_PAGE_TOKENS) * 4);
    }
    __syncthreads();
    const bool words_ok = (reinterpret_cast<uintptr_t>(a.cont) & 3u) == 0;
    for (int i = threadIdx.x; i < rw * 32; i += blockDim.x) {   // [word][stream]: consecutive lanes, mostly adjacent slots
        const int st = i & 31;
        if (st >= ns) continue;
        const uint8_t* p = reinterpret_cast<const uint8_t*>(s_src[st]) + (size_t)(i >> 5) * 64;
        dyn[i] = words_ok ? __ldg(reinterpret_cast<const uint32_t*>(p))
                          : (uint32_t)p[0] | (uint32_t)p[1] << 8 | (uint32_t)p[2] << 16 | (uint32_t)p[3] << 24;
    }
    __syncthreads();
    auto byte = [&](int i) -> uint32_t { return (dyn[(i >> 2) * 32 + lane] >> (8 * (i & 3))) & 255u; };
    auto window = [&](int i) -> uint32_t {
        const int w0 = i >> 2;
        return __funnelshift_r(dyn[min(w0, rw - 1) * 32 + lane], dyn[min(w0 + 1, rw - 1) * 32 + lane], 8 * (i & 3));
    };
    uint32_t x = 1u << 23;
    int ptr = 8;
    if (warp == 0 && lane < ns) {
        s_s[lane] = __half2float(__ushort_as_half((unsigned short)(byte(0) | (byte(1) << 8))));
        s_o[lane] = __half2float(__ushort_as_half((unsigned short)(byte(2) | (byte(3) << 8))));
        x = dyn[32 + lane];
    }
    for (int k = 0; k <= T.hs; ++k) {
        if (warp == 0) {
            if (k < T.hs && lane < ns)
#pragma unroll 1
                for (int j = 0; j < (PAIR ? 16 : 32); ++j)
                    tile[k & 1][lane * kSymRow + j] = decode4(lut, x, ptr, T.rec, 1u << 23, window);
        } else if (k > 0) {
#pragma unroll 4
            for (int i = warp - 1; i < ns; i += kExportWarps - 1) {
                const int h = s_grp[i] * T.hs + k - 1;
                const unsigned long long mi = s_mi[i] == kNoMean ? kNoMean : s_mi[i] + h;
                write_row<PAIR>(a, tile[(k - 1) & 1] + i * kSymRow, ((size_t)s_t[i] * a.Hkv + h) * DQ_HEAD_DIM, mi != kNoMean,
                                load_mean(a, mi, lane), s_s[i], s_o[i], lane);
            }
        }
        __syncthreads();
    }
}

// BF16 residual window (Sec. 5.1: the most recent tokens stay uncompressed): append one new
// token per sequence at position resid_lens[b] and count it.  One CTA per sequence; a full
// window is left unchanged.
__global__ void __launch_bounds__(256)
dq_window_append_kernel(const uint4* __restrict__ k_new, const uint4* __restrict__ v_new, uint4* __restrict__ resid_k,
                        uint4* __restrict__ resid_v, int32_t* __restrict__ resid_lens, int cap, int Hkv) {
    const int b = blockIdx.x;
    const int r = resid_lens[b];
    __syncthreads();   // every thread has read the count before thread 0 advances it
    if (r < 0 || r >= cap) return;
    const int row16 = Hkv * (DQ_HEAD_DIM * 2 / 16);   // 16-byte pieces of one token's K (or V)
    const size_t dst = ((size_t)b * cap + r) * row16, src = (size_t)b * row16;
    for (int i = threadIdx.x; i < row16; i += blockDim.x) {
        resid_k[dst + i] = k_new[src + i];
        resid_v[dst + i] = v_new[src + i];
    }
    if (threadIdx.x == 0) resid_lens[b] = r + 1;
}

}  // namespace

cudaError_t dq_launch_window_append(const void* k_new, const void* v_new, void* resid_k, void* resid_v,
                                    int32_t* resid_lens, int cap, int B, int Hkv, cudaStream_t st) {
    if (B == 0) return cudaSuccess;
    dq_window_append_kernel<<<B, 256, 0, st>>>(static_cast<const uint4*>(k_new), static_cast<const uint4*>(v_new),
                                               static_cast<uint4*>(resid_k), static_cast<uint4*>(resid_v), resid_lens,
                                               cap, Hkv);
    return cudaGetLastError();
}

cudaError_t dq_launch_decode_tokens(const DqDevTable& t, const uint8_t* cont, const int8_t* mean_q,
                                    const float* mean_scale, int max_windows, const int32_t* seq_id,
                                    const int32_t* pos, const int32_t* slot, int T, int Hkv,
                                    uint8_t* symbols, float* dequant, cudaStream_t st) {
    const ExportArgs a{cont, mean_q, mean_scale, seq_id, pos, slot, symbols, dequant, max_windows, T, Hkv};
    if (t.hs > 1) {
        const long long ns = (long long)T * (Hkv / t.hs);
        if (ns == 0) return cudaSuccess;
        auto kernel = t.pair ? dq_decode_tokens_wide_kernel<true> : dq_decode_tokens_wide_kernel<false>;
        const int smem = t.rec_words * 128;   // at most 32 KB
        kernel<<<(unsigned)((ns + 31) / 32), kExportWarps * 32, smem, st>>>(t, a);
        return cudaGetLastError();
    }
    const long long n = (long long)T * Hkv;
    if (n == 0) return cudaSuccess;
    auto kernel = t.pair ? dq_decode_tokens_kernel<true> : dq_decode_tokens_kernel<false>;
    const int smem = kExportWarps * 32 * ((((t.rec + 10) >> 2) | 1) + kSymRow) * 4;   // at most 39 KB
    kernel<<<(unsigned)((n + kExportWarps * 32 - 1) / (kExportWarps * 32)), kExportWarps * 32, smem, st>>>(t, a);
    return cudaGetLastError();
}
