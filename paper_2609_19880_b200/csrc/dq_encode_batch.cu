// Encoder kernels for calls with many per token-head streams (prompts, bulk encodes).  Compiled with -fmad=false,
// as dq_encode.cu.
#include "dq_encode.cuh"

using namespace dqenc;

namespace {

// Throughput variant for calls with many streams: a CTA of 4 warps takes 32 consecutive streams.
// Each warp quantises 8 of them (steps 1-6 of Algorithm 1, as above) and leaves the symbols in
// shared memory; then ONE warp entropy-codes all 32 streams at once, lane = stream, so the serial
// rANS chain costs one instruction stream per 32 streams instead of one per stream with 32
// redundant lanes.  Symbols are stored [position][stream] and emitted bytes [byte index][stream] so
// that the lanes of that warp touch consecutive bytes.  Small CTAs, 8 per SM at 64 registers: the
// other warps of a CTA idle during its rANS pass, so that pass should be a small part of a small CTA.
#ifndef DQ_B32_MINB
#define DQ_B32_MINB 8
#endif
#ifndef DQ_B32_WARPS
#define DQ_B32_WARPS 4
#endif
constexpr int kB32 = kDqEncodeBatchStreams;
constexpr int kB32SymWords = 33;         // words per stream's symbol row (128 bytes + pad: lane = stream reads without conflicts)
constexpr int kB32Warps = DQ_B32_WARPS;
// CTAs per SM the registers are held to: 8 (64 registers) while a lane's thresholds fit, 6, then 4 (128) beyond and for
// the pair search (7.9 ms against 12.5 ms at 8 CTAs per SM, config 2 prefill).
constexpr int batch_min_blocks(int M, bool pair) { return pair || M > 9 ? 4 : M > 5 ? 6 : DQ_B32_MINB; }

// One launch per tensor kind, so that the number of levels is a compile-time constant of everything below.  The
// second kind's launch (`second`) does not wait for the first's, it only ends after it.
template <int M, bool PAIR>
__global__ void __launch_bounds__(kB32Warps * 32, batch_min_blocks(M, PAIR))
dq_encode_batch32_kernel(const __grid_constant__ DqDevTable TD, const __grid_constant__ DqPairEnc PD, const DqEncodeArgs a, int per, bool is_v,
                         bool second) {
    __shared__ __align__(16) EncTable T;
    __shared__ uint32_t s_sym[kB32 * kB32SymWords];
    __shared__ uint8_t s_bytesT[DQ_MAX_REC_BYTES * kB32];
    __shared__ uint32_t s_hdr[kB32], s_xs[kB32], s_k[kB32];
    __shared__ unsigned long long s_rec[kB32];   // record addresses
    __shared__ unsigned long long s_mi[kB32];    // rows of the mean arrays
    __shared__ int s_pos[kB32];
    load_enc_table(T, TD, TD, PD, PD, is_v);
    __syncthreads();
    // The launch is let go after the wait, so that being launched proves to a second kind's kernel that everything
    // before the first one is complete.
    if (!second) dqdev::pdl_wait_prior_grid();
    dqdev::pdl_launch_dependents();
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const long long total = (long long)a.T * a.Hkv;
    const long long first = (long long)blockIdx.x * per;
    const int ns = (int)min((long long)per, total - first);
    const int rec = TD.rec;
    const bool has_mean = TD.has_mean, rope = !is_v && a.rope_style;

    if (threadIdx.x < ns) {   // where stream i's record, mean row and position are: once per stream, lane = stream
        int t, h;
        split_stream(a, first + threadIdx.x, t, h);
        const int sl = a.slot[t];
        s_rec[threadIdx.x] = (unsigned long long)((is_v ? a.v_cont : a.k_cont) +
                             (((size_t)(sl / DQ_PAGE_TOKENS) * a.Hkv + h) * DQ_PAGE_TOKENS + (size_t)(sl % DQ_PAGE_TOKENS)) * rec);
        if (has_mean || rope) {
            const int ps = a.pos[t];
            s_pos[threadIdx.x] = ps;
            s_mi[threadIdx.x] = mean_row(a, a.seq_id[t], ps, h);
        }
    }
    __syncthreads();

    // quantise: warp w takes streams w, w + warps, ...; the loads of the next one are issued before the work on this one
    const uint2* x = reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(is_v ? a.v_bf16 : a.k_bf16) + first * kN) + lane;
    auto load = [&](int i, uint2& raw, uint32_t& q4, float& sc) {
        if (i >= ns) return;
        raw = x[i * (kN / 4)];
        if (has_mean) {
            const size_t mi = s_mi[i];
            q4 = *reinterpret_cast<const uint32_t*>(a.mean_q + mi * kN + 4 * lane);
            sc = a.mean_scale[mi];
        }
    };
    uint2 raw = make_uint2(0u, 0u);
    uint32_t q4 = 0u;
    float sc = 0.f;
    load(wib, raw, q4, sc);
    for (int i = wib; i < ns; i += kB32Warps) {
        float z[4];
        unpack_bf16x4(raw, z);
        if (rope)
            warp_rope128(z, lane, a.rope_cos + (size_t)s_pos[i] * 64, a.rope_sin + (size_t)s_pos[i] * 64, a.rope_style);
        if (T.rotate) warp_fwht128(z, lane);
        if (has_mean) {
            if (a.mean_mode == DQ_MEAN_REUSE && s_pos[i] % DQ_WINDOW_TOKENS == 0) carry_mean(a, s_mi[i], s_pos[i], lane, q4, sc);
            remove_mean(z, q4, sc);
        }
        load(i + kB32Warps, raw, q4, sc);
        const StreamQuantised sq = quantise_values<M, PAIR, false>(T, z);
        if (PAIR) {   // the lane's two pair indices u = a M + b
            const uint32_t u0 = (sq.sym & 0xffu) * M + ((sq.sym >> 8) & 0xffu), u1 = ((sq.sym >> 16) & 0xffu) * M + (sq.sym >> 24);
            reinterpret_cast<uint16_t*>(s_sym + i * kB32SymWords)[lane] = (uint16_t)(u0 | (u1 << 8));
        } else {
            s_sym[i * kB32SymWords + lane] = sq.sym;
        }
        if (lane == 0) {
            s_hdr[i] = sq.hdr0;
            if (a.status) {
                if (sq.flags & 1u) atomicAdd(a.status + 0, 1u);
                if (sq.flags & 2u) atomicAdd(a.status + 1, 1u);
                if (sq.flags & 4u) atomicAdd(a.status + 2, 1u);
            }
        }
    }
    __syncthreads();
    if (wib == 0 && lane < ns) {   // rANS, Eq. (rans) Enc on the symbols from the last one back; lane = stream
        uint32_t xs = 1u << (T.sigma - 9);
        const uint32_t dst0 = dqdev::smem_addr(s_bytesT) + lane;
        uint32_t dst = dst0;   // at most one byte per symbol: 128 rows of kB32 bytes suffice
        rans_encode_row<kB32>(T.enc, s_sym + lane * kB32SymWords, (PAIR ? kN / 2 : kN) / 4, xs, dst);
        const uint32_t k = (dst - dst0) / kB32;
        s_xs[lane] = xs;
        s_k[lane] = k;
        if (a.status) atomicMax(a.status + 3, 4u + (uint32_t)(T.sigma >> 3) + k);
    }
    __syncthreads();
    const int pay = 4 + (T.sigma >> 3);
    const uint32_t rec_magic = 0xffffffffu / (uint32_t)rec + 1u;   // idx / rec by a high multiply: idx < 2^13
    for (int idx = threadIdx.x; idx < ns * rec; idx += blockDim.x) {   // records out: header, state, k bytes, then zeros
        const int si = (int)__umulhi((uint32_t)idx, rec_magic), i = idx - si * rec;
        const int k = (int)s_k[si], at = k - 1 - (i - pay);   // emitted last = read first
        const uint32_t tail = s_bytesT[min(max(at, 0), kN) * kB32 + si];
        const uint32_t head = i < 4 ? s_hdr[si] >> (8 * i) : s_xs[si] >> (8 * (i & 3));
        const uint8_t v = (uint8_t)(i < pay ? head : at >= 0 ? tail : 0u);
        reinterpret_cast<uint8_t*>(s_rec[si])[i] = v;
    }
    if (second) dqdev::pdl_wait_prior_grid();   // the first kind's kernel: whoever waits for this one may read both
}

using BatchKernel = void (*)(DqDevTable, DqPairEnc, DqEncodeArgs, int, bool, bool);

template <bool PAIR>
BatchKernel kernel_for(int M) {
    switch (M) {
#define DQ_LEVELS_CASE(M_) case M_: return dq_encode_batch32_kernel<M_, PAIR>;
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

// Streams per CTA (per = 0): 32 once that fills the GPU about three times, fewer below, so that every SM gets its eight
// CTAs: the coding pass costs a CTA the same for 4 and for 32 streams.
cudaError_t dq_launch_encode_batch(const DqDevTable& tk, const DqDevTable& tv, const DqPairEnc& pk, const DqPairEnc& pv,
                                   const DqEncodeArgs& a, int per, cudaStream_t st) {
    const long long streams = (long long)a.T * a.Hkv;
    if (per <= 0) {
        const long long resident = 148LL * DQ_B32_MINB / ((a.do_k && a.do_v) ? 2 : 1);
        per = (int)((streams + resident - 1) / resident);
        per = (per + kB32Warps - 1) / kB32Warps * kB32Warps;   // whole rounds of the CTA's warps
    }
    per = per > kB32 ? kB32 : per;
    const dim3 grid((unsigned)((streams + per - 1) / per)), block(kB32Warps * 32);
    bool second = false;
    for (int kind = 0; kind < 2; ++kind) {
        if (kind == 0 ? !a.do_k : !a.do_v) continue;
        const DqDevTable& t = kind == 0 ? tk : tv;
        const auto kernel = t.pair ? kernel_for<true>(t.M) : kernel_for<false>(t.M);
        if (!kernel) return cudaErrorInvalidValue;
        const cudaError_t e = dq_launch_pdl(kernel, grid, block, 0, st, t, kind == 0 ? pk : pv, a, per, kind == 1, second);
        if (e != cudaSuccess) return e;
        second = true;
    }
    return cudaSuccess;
}
