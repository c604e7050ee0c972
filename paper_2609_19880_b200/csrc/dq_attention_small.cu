// Decode attention for calls that fit the GPU once: every CTA takes one (sequence, KV head, block of NW * 32 tokens) and
// there is no other work to hide latency behind, so the serial rANS chain is what bounds the call.  Differences from
// the persistent kernel of dq_attention.cu (same arithmetic, same partials):
//   * K and V streams of the SAME block are decoded together, the steps of a lane's two chains in turn (114 -> about
//     80 clocks per pair of steps at one warp per scheduler); the V levels wait in shared memory (8 KB per warp)
//     for the softmax weights, so a block costs one pass over the streams instead of two;
//   * no prepare kernel: a CTA rotates its own q rows, takes q'.mean of its windows and scans the sequence lengths;
//   * decode-step mode: only the CTAs whose block holds a sequence's newest token wait for the encoder.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "dq_attention_common.cuh"

using namespace dqdev;
using namespace dqattn;

namespace {

constexpr int kTile = 1024;            // [32 tok][16 ch] fp16, 32-byte rows, halves swizzled by (row >> 2) & 1
constexpr int kSmallWarps = 8;         // most warps per CTA

// Shared-memory layout: compile-time offsets, then per-warp regions.
constexpr int kOffLutK = 0, kOffLutV = kOffLutK + 256 * 32 * 4;
constexpr int kOffQ16 = kOffLutV + 256 * 32 * 4;                       // fp16 q' operand
constexpr int kOffQrot = kOffQ16 + kQ16Bytes;                          // [8][128] q' in binary32
constexpr int kOffQsum = kOffQrot + DQ_MAX_GROUP * kN * 4;             // [8]
constexpr int kOffRed = kOffQsum + DQ_MAX_GROUP * 4;                   // [warp][8] maxima
constexpr int kOffItem = kOffRed + kSmallWarps * DQ_MAX_GROUP * 4;     // b, blk, len, total blocks before b
constexpr int kOffWarp = (kOffItem + 32 + 127) & ~127;
constexpr int kWTileV = 0, kWTileK = kWTileV + 8 * kTile, kWQmu = kWTileK + kTile, kWRec = kWQmu + 32;
constexpr int kLO = kN + 4;            // floats per head row of a warp's output slot (over its V tiles)

__host__ __device__ inline int align16s(int x) { return (x + 15) & ~15; }
__host__ __device__ inline int small_warp_bytes(int rec_k, int rec_v) {
    return kWRec + align16s(kChunk * rec_k) + align16s(kChunk * rec_v) + 16;   // + over-read of a last record
}
// slack for a malformed record that is over-read by up to 136 + 8 bytes
__host__ __device__ inline int small_smem_bytes(int nw, int rec_k, int rec_v, int B) {
    (void)B;
    return kOffWarp + nw * small_warp_bytes(rec_k, rec_v) + 256;
}

// One step of two chains (Algorithm 2; see decode16 in dq_attention.cu for the single chain): table entry, then
// x = f (x >> 8) + (z - c), then one byte from the window if x < L.  FW: dp4a weight of the entry's f byte.
template <int LBITS, uint32_t FW>
__device__ __forceinline__ void step_both(uint32_t (&x)[2], uint32_t (&sel)[2], const uint32_t (&win)[2], const uint32_t (&lut)[2],
                                          uint32_t one, uint32_t& e0, uint32_t& e1) {
    e0 = lds32(dp4a_u32(x[0], 0x80u, lut[0]));
    e1 = lds32(dp4a_u32(x[1], 0x80u, lut[1]));
    uint32_t t0 = x[0] >> 8, t1 = x[1] >> 8;
    const uint32_t f0 = dp4a_u32(e0, FW, 0u), f1 = dp4a_u32(e1, FW, 0u);
    t0 *= f0;
    t1 *= f1;
    x[0] = dp4a_u32(e0, 1u, t0);
    x[1] = dp4a_u32(e1, 1u, t1);
    asm("{.reg .pred p, q; setp.lt.u32 p, %0, %7; setp.lt.u32 q, %1, %7; @p prmt.b32 %0, %0, %4, %2; @q prmt.b32 %1, %1, %5, %3; "
        "@p mad.lo.u32 %2, %6, %6, %2; @q mad.lo.u32 %3, %6, %6, %3;}"
        : "+r"(x[0]), "+r"(x[1]), "+r"(sel[0]), "+r"(sel[1]) : "r"(win[0]), "r"(win[1]), "r"(one), "n"(1u << LBITS));
}

// 16 channels of both streams: levels as 8 fp16x2 words each into the lane's tile rows (halves swapped by `swap`).
// COLS: records lie in columns [word][lane]; ptr is then a byte index, col a lane's column and last the last row that a
// window may start in (malformed records only).
template <int LBITS, bool PAIRS, bool COLS>
__device__ __forceinline__ void decode16_both(uint32_t (&x)[2], uint32_t (&ptr)[2], const uint32_t (&lut)[2], uint32_t one,
                                              uint32_t krow, uint32_t vrow, uint32_t swap, const uint32_t (&col)[2], const uint32_t (&last)[2]) {
#pragma unroll
    for (int q4 = 0; q4 < (PAIRS ? 2 : 4); ++q4) {
        uint32_t sel[2] = {0x2104u, 0x2104u}, win[2], lo[2], hi[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const uint32_t at = COLS ? col[c] + min(ptr[c] >> 2, last[c]) * 128u : ptr[c] & ~3u;
            lo[c] = lds32(at);
            hi[c] = lds32(at + (COLS ? 128u : 4u));
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) win[c] = __funnelshift_r(lo[c], hi[c], ptr[c] << 3);
        uint32_t e[4], d[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) step_both<LBITS, PAIRS ? 0x00010000u : 0x01000000u>(x, sel, win, lut, one, e[i], d[i]);
        ptr[0] += sel[0] - 0x2104u;
        ptr[1] += sel[1] - 0x2104u;
        // stored group by group: the stores keep the two chains' steps interleaved in the generated code
        if (PAIRS) {
            const uint32_t k4[4] = {e[0] & 0xff00ff00u, e[1] & 0xff00ff00u, e[2] & 0xff00ff00u, e[3] & 0xff00ff00u};
            const uint32_t v4[4] = {d[0] & 0xff00ff00u, d[1] & 0xff00ff00u, d[2] & 0xff00ff00u, d[3] & 0xff00ff00u};
            sts128(krow + ((16u * q4) ^ swap), k4);
            sts128(vrow + ((16u * q4) ^ swap), v4);
        } else {
            const uint32_t at = ((16u * (q4 >> 1)) ^ swap) + 8u * (q4 & 1);
            sts64(krow + at, __byte_perm(e[0], e[1], 0x6521u), __byte_perm(e[2], e[3], 0x6521u));
            sts64(vrow + at, __byte_perm(d[0], d[1], 0x6521u), __byte_perm(d[2], d[3], 0x6521u));
        }
    }
}

// Block `bg` of the call (blocks of p.item_tokens tokens, sequence-major), found by one warp from the sequence lengths:
// s_item = {sequence, block within it, blocks of that sequence, blocks of the call}.  CTA 0 leaves the blocks
// before each sequence for the merge kernel.
__device__ __forceinline__ void find_block(const AttnParams& p, int bg, int lane, int* s_item) {
    int carry = 0;
    for (int base = 0; base < p.B; base += 32) {
        const int b = base + lane;
        int nb = 0;
        if (b < p.B) nb = (min(max(p.seq_lens[b], 0), p.max_pages * DQ_PAGE_TOKENS) + p.item_tokens - 1) / p.item_tokens;
        int incl = nb;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(kFullMask, incl, d);
            if (lane >= d) incl += o;
        }
        const int excl = carry + incl - nb;
        if (b < p.B) {
            if (blockIdx.x == 0) p.prefix[b] = excl;
            if (bg >= excl && bg < excl + nb) { s_item[0] = b; s_item[1] = bg - excl; s_item[2] = nb; }
        }
        carry += __shfl_sync(kFullMask, incl, 31);
    }
    if (lane == 0) { s_item[3] = carry; if (blockIdx.x == 0) p.prefix[p.B] = carry; }
}

template <bool STEP, int LBITS, bool PAIRS>
__global__ void __launch_bounds__(kSmallWarps * 32, 1)
dq_attention_small_kernel(const __grid_constant__ DqDevTable TK, const __grid_constant__ DqDevTable TV, const AttnParams p) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nthreads = blockDim.x, nw = nthreads >> 5;
    const int G = p.G;
    const uint32_t sbase = smem_addr(smem);
    const int wbytes = small_warp_bytes(TK.rec, TV.rec);
    uint32_t* lutk = reinterpret_cast<uint32_t*>(smem + kOffLutK);
    uint32_t* lutv = reinterpret_cast<uint32_t*>(smem + kOffLutV);
    float* qrot = reinterpret_cast<float*>(smem + kOffQrot);
    float* qsum = reinterpret_cast<float*>(smem + kOffQsum);
    float* red = reinterpret_cast<float*>(smem + kOffRed);
    int* s_item = reinterpret_cast<int*>(smem + kOffItem);
    const uint32_t wb = sbase + kOffWarp + warp * wbytes;
    const uint32_t vtiles = wb + kWTileV, ktile = wb + kWTileK, my_qmu = wb + kWQmu;
    const uint32_t kst = wb + kWRec, vst = kst + align16s(kChunk * TK.rec);

    pdl_launch_dependents();
    for (int i = tid; i < 256 * 8; i += nthreads) {   // tables (kernel parameters): 32 copies of an entry, 16 bytes at a time
        const uint32_t k = TK.lut[i >> 3], v = TV.lut[i >> 3];
        reinterpret_cast<uint4*>(lutk)[i] = make_uint4(k, k, k, k);
        reinterpret_cast<uint4*>(lutv)[i] = make_uint4(v, v, v, v);
    }
    // In decode-step mode the encoder let this kernel go after its own wait: everything older is complete, and only the
    // newest tokens' records and their windows' means are still being written.
    if (!STEP) pdl_wait_prior_grid();
    if (warp == 0) find_block(p, (int)blockIdx.x / p.Hkv, lane, s_item);
    __syncthreads();
    const int bg = (int)blockIdx.x / p.Hkv, h = (int)blockIdx.x - bg * p.Hkv;
    if (bg >= s_item[3]) {
        if (STEP) pdl_wait_prior_grid();   // this kernel's end implies the encoder's
        return;
    }
    const int b = s_item[0], blk = s_item[1];
    const bool late = blk == s_item[2] - 1;
    const int len = min(p.seq_lens[b], p.max_pages * DQ_PAGE_TOKENS);
    const int tok0 = (blk * nw + warp) * kChunk;
    const bool mine = tok0 < len;   // this warp holds tokens
    if (STEP && late) pdl_wait_prior_grid();

    // the mean of the warp's window (used once q' is there) and the page ids of its 32 tokens
    uint32_t q4 = 0u;
    float msc = 0.f;
    if (p.has_mean && mine) {
        const size_t mi = ((size_t)b * p.max_windows + tok0 / DQ_WINDOW_TOKENS) * p.Hkv + h;
        q4 = *reinterpret_cast<const uint32_t*>(p.mean_q + mi * kN + 4 * lane);
        msc = p.mean_scale[mi];
    }
    int page = 0;
    if (mine && lane < 2 && tok0 + 16 * lane < len) page = p.page_table[(size_t)b * p.max_pages + (tok0 >> 4) + lane];
    const int page0 = __shfl_sync(kFullMask, page, 0), page1 = __shfl_sync(kFullMask, page, 1);
    if (mine) {
        const int pages = tok0 + 16 < len ? 2 : 1;
#pragma unroll
        for (int kind = 0; kind < 2; ++kind) {
            const int rec = kind ? TV.rec : TK.rec, np = pages * rec;
            const uint32_t dst = kind ? vst : kst, bytes = 16u * (uint32_t)rec;
            const uint8_t* cont = kind ? p.v_cont : p.k_cont;
            const uint8_t* s0 = cont + ((size_t)page0 * p.Hkv + h) * bytes;
            const uint8_t* s1 = cont + ((size_t)page1 * p.Hkv + h) * bytes - bytes;
            for (int i = lane; i < np; i += 32) cp_async16(dst + i * 16, (i < rec ? s0 : s1) + i * 16);
        }
    }
    cp_async_commit();
    // q' of this KV head's rows: binary32, the fp16 hi / lo operand rows, the row sums
    for (int g = warp; g < 8; g += nw) {
        uint8_t* hi_row = smem + kOffQ16 + g * kQ16Stride + lane * 8;
        uint2 whi = make_uint2(0u, 0u), wlo = make_uint2(0u, 0u);
        if (g < G) {
            const uint2 raw = *reinterpret_cast<const uint2*>(p.q + qo_row(p, b, h * G + g) * kN + 4 * lane);
            float v[4] = {bf16_bits_to_float(raw.x & 0xffffu), bf16_bits_to_float(raw.x >> 16),
                          bf16_bits_to_float(raw.y & 0xffffu), bf16_bits_to_float(raw.y >> 16)};
            if (p.rotate_q) warp_fwht128(v, lane);
            *reinterpret_cast<float4*>(qrot + g * kN + 4 * lane) = make_float4(v[0], v[1], v[2], v[3]);
            const __half2 h01 = __floats2half2_rn(v[0], v[1]), h23 = __floats2half2_rn(v[2], v[3]);
            const float2 f01 = __half22float2(h01), f23 = __half22float2(h23);
            whi = make_uint2(*reinterpret_cast<const uint32_t*>(&h01), *reinterpret_cast<const uint32_t*>(&h23));
            wlo = make_uint2(pack_half2(v[0] - f01.x, v[1] - f01.y), pack_half2(v[2] - f23.x, v[3] - f23.y));
            float s = (v[0] + v[1]) + (v[2] + v[3]);
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(kFullMask, s, d);
            if (lane == 0) qsum[g] = s * p.scale_log2;
        }
        *reinterpret_cast<uint2*>(hi_row) = whi;                      // unused operand rows are zero
        *reinterpret_cast<uint2*>(hi_row + 8 * kQ16Stride) = wlo;
    }
    __syncthreads();
    if (p.has_mean && mine) {   // q'.mean of the warp's window, times the logit scale
        float m[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) m[e] = msc * (float)(int)(int8_t)((q4 >> (8 * e)) & 0xffu);
        for (int g = 0; g < G; ++g) {
            const float4 v = *reinterpret_cast<const float4*>(qrot + g * kN + 4 * lane);
            float s = fmaf(v.w, m[3], fmaf(v.z, m[2], fmaf(v.y, m[1], v.x * m[0])));
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(kFullMask, s, d);
            if (lane == 0) sts32f(my_qmu + g * 4, s * p.scale_log2);
        }
    }
    cp_async_wait<0>();
    __syncwarp();

    // ------------------------------------------ both streams of the warp's tokens, 16 channels at a time
    const int g_row = lane >> 2, qd = lane & 3;
    float sacc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) { sacc[i][0] = sacc[i][1] = sacc[i][2] = sacc[i][3] = 0.f; }
    const uint32_t rk = kst + lane * TK.rec, rv = vst + lane * TV.rec;
    const int lrow = (lane & 7) + (lane >> 4) * 8;   // ldmatrix row; half h of row r sits at half h ^ ((r >> 2) & 1)
    const uint32_t ld_off = lrow * 32 + ((((lane >> 3) & 1) ^ ((lrow >> 2) & 1)) << 4);
    if (mine) {
        constexpr uint32_t kStateMask = LBITS == 23 ? 0xffffffffu : 0x00ffffffu;
        constexpr uint32_t kPay = LBITS == 23 ? 8u : 7u;
        uint32_t x[2] = {lds32_unaligned(rk + 4) & kStateMask, lds32_unaligned(rv + 4) & kStateMask};
        uint32_t ptr[2] = {rk + kPay, rv + kPay};
        const uint32_t lut[2] = {sbase + kOffLutK + lane * 4, sbase + kOffLutV + lane * 4};
        const uint32_t one = (sbase >> 31) | 1u;
        const uint32_t a_addr = sbase + kOffQ16 + ((lane & 7) + ((lane >> 3) & 1) * 8) * kQ16Stride + (lane >> 4) * 16;
        const uint32_t swap = ((lane >> 2) & 1) << 4;
#pragma unroll 1
        for (int cg = 0; cg < 8; ++cg) {
            decode16_both<LBITS, PAIRS, false>(x, ptr, lut, one, ktile + lane * 32, vtiles + cg * kTile + lane * 32, swap, lut, lut);
            __syncwarp();
            uint32_t a[4], b0[4], b1[4];
            ldmatrix_x4(a, a_addr + cg * 32);
            ldmatrix_x4(b0, ktile + ld_off);
            ldmatrix_x4(b1, ktile + ld_off + 16 * 32);
            mma_f16_16816(sacc[0], a, b0[0], b0[1]);
            mma_f16_16816(sacc[1], a, b0[2], b0[3]);
            mma_f16_16816(sacc[2], a, b1[0], b1[1]);
            mma_f16_16816(sacc[3], a, b1[2], b1[3]);
            __syncwarp();
        }
    }

    // ------------------------------------------ logits and the warp's maximum (base 2)
    float lg[4][2], sv_t[4][2], ov_t[4][2];
    float mx = -INFINITY;
    if (mine) {
        {   // per-token (sK, oK, sV, oV) from token-per-lane to the accumulator layout, through the K tile
            const uint32_t hk = lds32_unaligned(rk), hv = lds32_unaligned(rv);
            const float sK = __half2float(__ushort_as_half((unsigned short)(hk & 0xffffu)));
            const float oK = __half2float(__ushort_as_half((unsigned short)(hk >> 16)));
            const float sV = __half2float(__ushort_as_half((unsigned short)(hv & 0xffffu)));
            const float oV = __half2float(__ushort_as_half((unsigned short)(hv >> 16)));
            // the key scale carries the logit scale (sm_scale * log2 e): logits come out in base-2 units
            asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};\n" ::"r"(ktile + lane * 16), "f"(sK * p.scale_log2), "f"(oK),
                         "f"(sV), "f"(oV) : "memory");
        }
        // tokens this thread's row may see: an earlier query token stops earlier, the BF16 window absorbs the offset first
        int row_len = len;
        if (p.q_total > 1) row_len -= max(0, row_offset(p, g_row) - (p.resid_lens ? max(p.resid_lens[b], 0) : 0));
        float qmu = 0.f, qs = 0.f;
        if (g_row < G) {
            qs = qsum[g_row];
            if (p.has_mean) qmu = __uint_as_float(lds32(my_qmu + g_row * 4));
        }
        __syncwarp();
        const int lim = row_len - tok0 - 2 * qd;   // token 8 i + 2 qd + u is visible iff 8 i + u < lim
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                float4 m4;
                asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];\n"
                             : "=f"(m4.x), "=f"(m4.y), "=f"(m4.z), "=f"(m4.w) : "r"(ktile + (8 * i + 2 * qd + u) * 16));
                const bool ok = 8 * i + u < lim;
                lg[i][u] = ok ? fmaf(m4.x, sacc[i][u] + sacc[i][2 + u], fmaf(m4.y, qs, qmu)) : -INFINITY;
                sv_t[i][u] = ok ? m4.z : 0.f;
                ov_t[i][u] = ok ? m4.w : 0.f;
                mx = fmaxf(mx, lg[i][u]);
            }
        mx = fmaxf(mx, __shfl_xor_sync(kFullMask, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(kFullMask, mx, 2));
    }
    if (qd == 0) red[warp * DQ_MAX_GROUP + g_row] = mx;
    __syncthreads();
    float m_item = -INFINITY;
    for (int w = 0; w < nw; ++w) m_item = fmaxf(m_item, red[w * DQ_MAX_GROUP + g_row]);

    // ------------------------------------------ softmax weights, then O[j][g] = sum_t (a_t s_t) level_tj from the V tiles
    float lsum = 0.f, osum = 0.f;
    if (mine) {
        uint32_t pb_hi[2][2], pb_lo[2][2];
        const float m_use = (m_item == -INFINITY) ? 0.f : m_item;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float ps[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float pr = ex2_approx(lg[i][u] - m_use);   // <= 1; exp2(-inf) = 0
                lsum += pr;
                osum = fmaf(pr, ov_t[i][u], osum);
                ps[u] = pr * sv_t[i][u];
            }
            const __half2 h2 = __floats2half2_rn(ps[0], ps[1]);   // fp16 hi + lo pair of each weight
            const float2 hf = __half22float2(h2);
            pb_hi[i >> 1][i & 1] = *reinterpret_cast<const uint32_t*>(&h2);
            pb_lo[i >> 1][i & 1] = pack_half2(ps[0] - hf.x, ps[1] - hf.y);
        }
        lsum += __shfl_xor_sync(kFullMask, lsum, 1);
        lsum += __shfl_xor_sync(kFullMask, lsum, 2);
        osum += __shfl_xor_sync(kFullMask, osum, 1);
        osum += __shfl_xor_sync(kFullMask, osum, 2);
        float o[8][4];
#pragma unroll
        for (int cg = 0; cg < 8; ++cg) {
            uint32_t a0[4], a1[4];
            o[cg][0] = o[cg][1] = o[cg][2] = o[cg][3] = 0.f;
            ldmatrix_x4_trans(a0, vtiles + cg * kTile + ld_off);             // tokens 0..15, 16 channels
            ldmatrix_x4_trans(a1, vtiles + cg * kTile + ld_off + 16 * 32);   // tokens 16..31
            mma_f16_16816(o[cg], a0, pb_hi[0][0], pb_hi[0][1]);
            mma_f16_16816(o[cg], a1, pb_hi[1][0], pb_hi[1][1]);
            mma_f16_16816(o[cg], a0, pb_lo[0][0], pb_lo[0][1]);
            mma_f16_16816(o[cg], a1, pb_lo[1][0], pb_lo[1][1]);
        }
        __syncwarp();   // every lane has read the V tiles: the output slot goes over them
#pragma unroll
        for (int cg = 0; cg < 8; ++cg) {   // channels (lane / 4, lane / 4 + 8) of heads (2 qd, 2 qd + 1)
            const uint32_t oa = vtiles + ((2 * qd) * kLO + (lane >> 2) + 16 * cg) * 4;
            sts32f(oa, o[cg][0]); sts32f(oa + 32, o[cg][2]);
            sts32f(oa + kLO * 4, o[cg][1]); sts32f(oa + kLO * 4 + 32, o[cg][3]);
        }
        if (qd == 0) {
            sts32f(vtiles + (g_row * kLO + kN) * 4, lsum);
            sts32f(vtiles + (g_row * kLO + kN + 1) * 4, osum);
        }
    }
    if (warp == 0 && qd == 0) red[g_row] = m_item;   // the maxima are read: slot 0 carries the item's
    __syncthreads();

    // ------------------------------------------ the warps' slots added up: one partial per head row
    const int nwv = min(nw, (len - blk * nw * kChunk + kChunk - 1) / kChunk);   // warps that hold tokens
    float* dst0 = p.partial + ((size_t)bg * p.Hq + (size_t)h * G) * kPartial;
    for (int e = tid; e < G * 34; e += nthreads) {
        const int g = e < G * 32 ? e >> 5 : (e - G * 32) >> 1;
        float* dst = dst0 + (size_t)g * kPartial;
        if (e < G * 32) {
            const int c4 = e & 31;
            const uint8_t* src = smem + kOffWarp + kWTileV + (g * kLO + 4 * c4) * 4;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int w = 0; w < nwv; ++w) {
                const float4 v = *reinterpret_cast<const float4*>(src + w * wbytes);
                acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
            }
            *reinterpret_cast<float4*>(dst + 4 * c4) = acc;
        } else {
            const int which = (e - G * 32) & 1;
            const uint8_t* src = smem + kOffWarp + kWTileV + (g * kLO + kN + which) * 4;
            float acc = 0.f;
            for (int w = 0; w < nwv; ++w) acc += *reinterpret_cast<const float*>(src + w * wbytes);
            dst[kN + 1 + which] = acc;   // l at 129, off at 130
            if (which == 0) dst[kN] = red[g];
        }
    }
    if (STEP && !late) pdl_wait_prior_grid();   // this kernel's end implies the encoder's
}

// ------------------------------------------------------- token-wide streams

// The same for streams that span the hs heads of a group: the records of a warp's 32 tokens lie whole in shared memory,
// in columns [word][lane] (no ring to keep filled), and the heads follow one another.  A warp takes its own maximum,
// so a head needs two barriers: q' there, and the warps' output slots there.
constexpr int kWOffQ16 = kOffQ16, kWOffQrot = kWOffQ16 + 2 * kQ16Bytes, kWOffQsum = kWOffQrot + 2 * DQ_MAX_GROUP * kN * 4;
constexpr int kWOffItem = kWOffQsum + 2 * DQ_MAX_GROUP * 4, kWOffWarp = (kWOffItem + 32 + 127) & ~127;
constexpr int kWCols = kWQmu + 32;     // a warp's K columns, then its V columns

__host__ __device__ inline int wide_small_warp_bytes(int rwk, int rwv) { return (kWCols + (rwk + rwv + 1) * 128 + 127) & ~127; }   // + the row after a last window
__host__ __device__ inline int wide_small_smem_bytes(int nw, int rwk, int rwv, int B) {
    (void)B;
    return kWOffWarp + nw * wide_small_warp_bytes(rwk, rwv);
}

template <bool PAIRS>
__global__ void __launch_bounds__(kSmallWarps * 32, 1)
dq_attention_wide_small_kernel(const __grid_constant__ DqDevTable TK, const __grid_constant__ DqDevTable TV, const AttnParams p) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nthreads = blockDim.x, nw = nthreads >> 5;
    const int G = p.G, hs = p.hs, groups = p.groups;
    const int rwk = TK.rec_words, rwv = TV.rec_words;
    const uint32_t sbase = smem_addr(smem);
    const int wbytes = wide_small_warp_bytes(rwk, rwv);
    float* qrot = reinterpret_cast<float*>(smem + kWOffQrot);
    float* qsum = reinterpret_cast<float*>(smem + kWOffQsum);
    int* s_item = reinterpret_cast<int*>(smem + kWOffItem);
    const uint32_t wb = sbase + kWOffWarp + warp * wbytes;
    const uint32_t vtiles = wb + kWTileV, ktile = wb + kWTileK, my_qmu = wb + kWQmu;
    const uint32_t colk = wb + kWCols, colv = colk + rwk * 128;

    pdl_launch_dependents();
    for (int i = tid; i < 256 * 8; i += nthreads) {
        const uint32_t k = TK.lut[i >> 3], v = TV.lut[i >> 3];
        reinterpret_cast<uint4*>(smem + kOffLutK)[i] = make_uint4(k, k, k, k);
        reinterpret_cast<uint4*>(smem + kOffLutV)[i] = make_uint4(v, v, v, v);
    }
    pdl_wait_prior_grid();
    const int bg = (int)blockIdx.x / groups, grp = (int)blockIdx.x - bg * groups;
    if (warp == 0) find_block(p, bg, lane, s_item);
    __syncthreads();
    if (bg >= s_item[3]) return;
    const int b = s_item[0], blk = s_item[1];
    const int len = min(p.seq_lens[b], p.max_pages * DQ_PAGE_TOKENS);
    const int tok0 = (blk * nw + warp) * kChunk;
    const bool mine = tok0 < len;

    // records: a row is word w of the warp's 32 tokens, 64 bytes from either page; lanes 0-3 / 4-7 of eight copy them
    {
        int page = 0;
        if (mine && lane < 2 && tok0 + 16 * lane < len) page = p.page_table[(size_t)b * p.max_pages + (tok0 >> 4) + lane];
        const int page0 = __shfl_sync(kFullMask, page, 0), page1 = __shfl_sync(kFullMask, page, 1);
        const int second = (lane >> 2) & 1;
        if (mine && tok0 + 16 * second < len) {
            const size_t blk64 = (size_t)(second ? page1 : page0) * groups + grp;
#pragma unroll
            for (int kind = 0; kind < 2; ++kind) {
                const int rw = kind ? rwv : rwk;
                const uint8_t* src = (kind ? p.v_cont : p.k_cont) + blk64 * ((size_t)rw * 64) + (lane & 3) * 16;
                const uint32_t dst = (kind ? colv : colk) + (lane & 7) * 16;
                for (int row = lane >> 3; row < rw; row += 4) cp_async16(dst + row * 128, src + (size_t)row * 64);
            }
        }
        cp_async_commit();
    }
    // q rows of head k, a warp's own; mean of the warp's window for head k
    auto load_q = [&](int k, int g) {
        return g < G ? *reinterpret_cast<const uint2*>(p.q + qo_row(p, b, (grp * hs + k) * G + g) * kN + 4 * lane) : make_uint2(0u, 0u);
    };
    uint2 qraw[2] = {load_q(0, warp), load_q(0, warp + nw)};   // nw >= 4: two rows per warp at most
    uint32_t q4 = 0u;
    float msc = 0.f;
    auto load_mean = [&](int k) {
        if (!p.has_mean || !mine) return;
        const size_t mi = ((size_t)b * p.max_windows + tok0 / DQ_WINDOW_TOKENS) * p.Hkv + grp * hs + k;
        q4 = *reinterpret_cast<const uint32_t*>(p.mean_q + mi * kN + 4 * lane);
        msc = p.mean_scale[mi];
    };
    load_mean(0);

    const int g_row = lane >> 2, qd = lane & 3;
    const int lrow = (lane & 7) + (lane >> 4) * 8;   // ldmatrix row; half h of row r sits at half h ^ ((r >> 2) & 1)
    const uint32_t ld_off = lrow * 32 + ((((lane >> 3) & 1) ^ ((lrow >> 2) & 1)) << 4);
    const uint32_t lut[2] = {sbase + kOffLutK + lane * 4, sbase + kOffLutV + lane * 4};
    const uint32_t col[2] = {colk + lane * 4, colv + lane * 4}, last[2] = {(uint32_t)rwk - 1u, (uint32_t)rwv - 1u};
    const uint32_t one = (sbase >> 31) | 1u, swap = ((lane >> 2) & 1) << 4;
    cp_async_wait<0>();
    __syncwarp();
    uint32_t x[2] = {lds32(col[0] + 128), lds32(col[1] + 128)}, ptr[2] = {8u, 8u};
    float sK, oK, sV, oV;
    {
        const uint32_t hk = lds32(col[0]), hv = lds32(col[1]);
        sK = __half2float(__ushort_as_half((unsigned short)(hk & 0xffffu))) * p.scale_log2;   // carries the logit scale
        oK = __half2float(__ushort_as_half((unsigned short)(hk >> 16)));
        sV = __half2float(__ushort_as_half((unsigned short)(hv & 0xffffu)));
        oV = __half2float(__ushort_as_half((unsigned short)(hv >> 16)));
    }

#pragma unroll 1
    for (int k = 0; k < hs; ++k) {
        // ------------------------------------------ q' of this head's rows, then q'.mean of the warp's window
        const int buf = k & 1;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int g = warp + j * nw;
            if (g >= 8) break;
            uint8_t* hi_row = smem + kWOffQ16 + buf * kQ16Bytes + g * kQ16Stride + lane * 8;
            uint2 whi = make_uint2(0u, 0u), wlo = make_uint2(0u, 0u);
            if (g < G) {
                float v[4] = {bf16_bits_to_float(qraw[j].x & 0xffffu), bf16_bits_to_float(qraw[j].x >> 16),
                              bf16_bits_to_float(qraw[j].y & 0xffffu), bf16_bits_to_float(qraw[j].y >> 16)};
                if (p.rotate_q) warp_fwht128(v, lane);
                *reinterpret_cast<float4*>(qrot + (buf * DQ_MAX_GROUP + g) * kN + 4 * lane) = make_float4(v[0], v[1], v[2], v[3]);
                const __half2 h01 = __floats2half2_rn(v[0], v[1]), h23 = __floats2half2_rn(v[2], v[3]);
                const float2 f01 = __half22float2(h01), f23 = __half22float2(h23);
                whi = make_uint2(*reinterpret_cast<const uint32_t*>(&h01), *reinterpret_cast<const uint32_t*>(&h23));
                wlo = make_uint2(pack_half2(v[0] - f01.x, v[1] - f01.y), pack_half2(v[2] - f23.x, v[3] - f23.y));
                float s = (v[0] + v[1]) + (v[2] + v[3]);
#pragma unroll
                for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(kFullMask, s, d);
                if (lane == 0) qsum[buf * DQ_MAX_GROUP + g] = s * p.scale_log2;
            }
            *reinterpret_cast<uint2*>(hi_row) = whi;                      // unused operand rows are zero
            *reinterpret_cast<uint2*>(hi_row + 8 * kQ16Stride) = wlo;
        }
        __syncthreads();   // q' there; the previous head's slots are merged
        if (p.has_mean && mine) {
            float m[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) m[e] = msc * (float)(int)(int8_t)((q4 >> (8 * e)) & 0xffu);
            for (int g = 0; g < G; ++g) {
                const float4 v = *reinterpret_cast<const float4*>(qrot + (buf * DQ_MAX_GROUP + g) * kN + 4 * lane);
                float s = fmaf(v.w, m[3], fmaf(v.z, m[2], fmaf(v.y, m[1], v.x * m[0])));
#pragma unroll
                for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(kFullMask, s, d);
                if (lane == 0) sts32f(my_qmu + g * 4, s * p.scale_log2);
            }
        }
        if (k + 1 < hs) {   // the next head's, on their way during the decode
            qraw[0] = load_q(k + 1, warp);
            qraw[1] = load_q(k + 1, warp + nw);
            load_mean(k + 1);
        }

        // ------------------------------------------ this head's 128 channels of both streams
        if (mine) {
            float sacc[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { sacc[i][0] = sacc[i][1] = sacc[i][2] = sacc[i][3] = 0.f; }
            const uint32_t a_addr = sbase + kWOffQ16 + buf * kQ16Bytes + ((lane & 7) + ((lane >> 3) & 1) * 8) * kQ16Stride + (lane >> 4) * 16;
#pragma unroll 1
            for (int cg = 0; cg < 8; ++cg) {
                decode16_both<23, PAIRS, true>(x, ptr, lut, one, ktile + lane * 32, vtiles + cg * kTile + lane * 32, swap, col, last);
                __syncwarp();
                uint32_t a[4], b0[4], b1[4];
                ldmatrix_x4(a, a_addr + cg * 32);
                ldmatrix_x4(b0, ktile + ld_off);
                ldmatrix_x4(b1, ktile + ld_off + 16 * 32);
                mma_f16_16816(sacc[0], a, b0[0], b0[1]);
                mma_f16_16816(sacc[1], a, b0[2], b0[3]);
                mma_f16_16816(sacc[2], a, b1[0], b1[1]);
                mma_f16_16816(sacc[3], a, b1[2], b1[3]);
                __syncwarp();
            }
            // logits, the warp's maximum, weights
            asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};\n" ::"r"(ktile + lane * 16), "f"(sK), "f"(oK), "f"(sV), "f"(oV) : "memory");
            int row_len = len;
            if (p.q_total > 1) row_len -= max(0, row_offset(p, g_row) - (p.resid_lens ? max(p.resid_lens[b], 0) : 0));
            float qmu = 0.f, qs = 0.f;
            if (g_row < G) {
                qs = qsum[buf * DQ_MAX_GROUP + g_row];
                if (p.has_mean) qmu = __uint_as_float(lds32(my_qmu + g_row * 4));
            }
            __syncwarp();
            const int lim = row_len - tok0 - 2 * qd;   // token 8 i + 2 qd + u is visible iff 8 i + u < lim
            float lg[4][2], sv_t[4][2], ov_t[4][2], mx = -INFINITY;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    float4 m4;
                    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];\n"
                                 : "=f"(m4.x), "=f"(m4.y), "=f"(m4.z), "=f"(m4.w) : "r"(ktile + (8 * i + 2 * qd + u) * 16));
                    const bool ok = 8 * i + u < lim;
                    lg[i][u] = ok ? fmaf(m4.x, sacc[i][u] + sacc[i][2 + u], fmaf(m4.y, qs, qmu)) : -INFINITY;
                    sv_t[i][u] = ok ? m4.z : 0.f;
                    ov_t[i][u] = ok ? m4.w : 0.f;
                    mx = fmaxf(mx, lg[i][u]);
                }
            mx = fmaxf(mx, __shfl_xor_sync(kFullMask, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(kFullMask, mx, 2));
            const float m_use = (mx == -INFINITY) ? 0.f : mx;
            uint32_t pb_hi[2][2], pb_lo[2][2];
            float lsum = 0.f, osum = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float ps[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const float pr = ex2_approx(lg[i][u] - m_use);
                    lsum += pr;
                    osum = fmaf(pr, ov_t[i][u], osum);
                    ps[u] = pr * sv_t[i][u];
                }
                const __half2 h2 = __floats2half2_rn(ps[0], ps[1]);   // fp16 hi + lo pair of each weight
                const float2 hf = __half22float2(h2);
                pb_hi[i >> 1][i & 1] = *reinterpret_cast<const uint32_t*>(&h2);
                pb_lo[i >> 1][i & 1] = pack_half2(ps[0] - hf.x, ps[1] - hf.y);
            }
            lsum += __shfl_xor_sync(kFullMask, lsum, 1);
            lsum += __shfl_xor_sync(kFullMask, lsum, 2);
            osum += __shfl_xor_sync(kFullMask, osum, 1);
            osum += __shfl_xor_sync(kFullMask, osum, 2);
            float o[8][4];
#pragma unroll
            for (int cg = 0; cg < 8; ++cg) {
                uint32_t a0[4], a1[4];
                o[cg][0] = o[cg][1] = o[cg][2] = o[cg][3] = 0.f;
                ldmatrix_x4_trans(a0, vtiles + cg * kTile + ld_off);
                ldmatrix_x4_trans(a1, vtiles + cg * kTile + ld_off + 16 * 32);
                mma_f16_16816(o[cg], a0, pb_hi[0][0], pb_hi[0][1]);
                mma_f16_16816(o[cg], a1, pb_hi[1][0], pb_hi[1][1]);
                mma_f16_16816(o[cg], a0, pb_lo[0][0], pb_lo[0][1]);
                mma_f16_16816(o[cg], a1, pb_lo[1][0], pb_lo[1][1]);
            }
            __syncwarp();   // every lane has read the V tiles: the output slot goes over them
#pragma unroll
            for (int cg = 0; cg < 8; ++cg) {
                const uint32_t oa = vtiles + ((2 * qd) * kLO + (lane >> 2) + 16 * cg) * 4;
                sts32f(oa, o[cg][0]); sts32f(oa + 32, o[cg][2]);
                sts32f(oa + kLO * 4, o[cg][1]); sts32f(oa + kLO * 4 + 32, o[cg][3]);
            }
            if (qd == 0) {
                sts32f(vtiles + (g_row * kLO + kN) * 4, mx);
                sts32f(vtiles + (g_row * kLO + kN + 1) * 4, lsum);
                sts32f(vtiles + (g_row * kLO + kN + 2) * 4, osum);
            }
        }
        __syncthreads();   // slots there

        // ------------------------------------------ the warps' slots merged: one partial per head row
        const int nwv = min(nw, (len - blk * nw * kChunk + kChunk - 1) / kChunk);   // warps that hold tokens
        float* dst0 = p.partial + ((size_t)bg * p.Hq + (size_t)(grp * hs + k) * G) * kPartial;
        for (int e = tid; e < G * 34; e += nthreads) {
            const int g = e < G * 32 ? e >> 5 : (e - G * 32) >> 1;
            const uint8_t* slot = smem + kWOffWarp + kWTileV + g * kLO * 4;
            float M = -INFINITY;
            for (int w = 0; w < nwv; ++w) M = fmaxf(M, *reinterpret_cast<const float*>(slot + w * wbytes + kN * 4));
            const float M_use = (M == -INFINITY) ? 0.f : M;
            float* dst = dst0 + (size_t)g * kPartial;
            if (e < G * 32) {
                const int c4 = e & 31;
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int w = 0; w < nwv; ++w) {
                    const float sc = ex2_approx(*reinterpret_cast<const float*>(slot + w * wbytes + kN * 4) - M_use);
                    const float4 v = *reinterpret_cast<const float4*>(slot + w * wbytes + 16 * c4);
                    acc.x = fmaf(v.x, sc, acc.x); acc.y = fmaf(v.y, sc, acc.y);
                    acc.z = fmaf(v.z, sc, acc.z); acc.w = fmaf(v.w, sc, acc.w);
                }
                *reinterpret_cast<float4*>(dst + 4 * c4) = acc;
            } else {
                const int which = (e - G * 32) & 1;
                float acc = 0.f;
                for (int w = 0; w < nwv; ++w) {
                    const float* f = reinterpret_cast<const float*>(slot + w * wbytes) + kN;
                    acc = fmaf(f[1 + which], ex2_approx(f[0] - M_use), acc);
                }
                dst[kN + 1 + which] = acc;   // l at 129, off at 130
                if (which == 0) dst[kN] = M;
            }
        }
    }
}

}  // namespace

// Warps per CTA with which the call's blocks fit the GPU once (0: they do not).  Blocks are counted from the width of
// the page table, the lengths being on the device.  4 warps where 128-token blocks still fit: a warp per scheduler
// decodes its two chains in about 80 clocks per step, two per scheduler in about 95.
int dq_attn_small_pick_warps(const DqDevTable& tk, const DqDevTable& tv, int B, int Hkv, int max_pages, int sm_count, int smem_max) {
    const bool wide = tk.hs > 1;
    for (int nw = 4; nw <= kSmallWarps; nw += wide ? 1 : 4) {
        const long long blocks = (long long)B * ((max_pages * DQ_PAGE_TOKENS + nw * kChunk - 1) / (nw * kChunk)) * (Hkv / tk.hs);
        const int smem = wide ? wide_small_smem_bytes(nw, tk.rec_words, tv.rec_words, B) : small_smem_bytes(nw, tk.rec, tv.rec, B);
        if (blocks <= sm_count && smem <= smem_max) return nw;
    }
    return 0;
}

cudaError_t dq_launch_attention_small(const DqDevTable& tk, const DqDevTable& tv, const AttnParams& p, int nw, bool step, cudaStream_t st) {
    void (*kernel)(DqDevTable, DqDevTable, AttnParams) =
        tk.pair ? (tk.sigma == 24 ? (step ? dq_attention_small_kernel<true, 15, true> : dq_attention_small_kernel<false, 15, true>)
                                  : (step ? dq_attention_small_kernel<true, 23, true> : dq_attention_small_kernel<false, 23, true>))
                : (tk.sigma == 24 ? (step ? dq_attention_small_kernel<true, 15, false> : dq_attention_small_kernel<false, 15, false>)
                                  : (step ? dq_attention_small_kernel<true, 23, false> : dq_attention_small_kernel<false, 23, false>));
    const bool wide = tk.hs > 1;   // token-wide streams have no decode-step mode
    if (wide) kernel = tk.pair ? dq_attention_wide_small_kernel<true> : dq_attention_wide_small_kernel<false>;
    const int smem = wide ? wide_small_smem_bytes(nw, tk.rec_words, tv.rec_words, p.B) : small_smem_bytes(nw, tk.rec, tv.rec, p.B);
    const cudaError_t e = dq_allow_smem(reinterpret_cast<const void*>(kernel), smem);
    if (e != cudaSuccess) return e;
    const int blocks = p.B * ((p.max_pages * DQ_PAGE_TOKENS + nw * kChunk - 1) / (nw * kChunk)) * p.groups;
    return dq_launch_pdl(kernel, dim3((unsigned)blocks), dim3(nw * 32), (size_t)smem, st, tk, tv, p);
}
