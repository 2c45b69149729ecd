// Depthwise causal convolution (width 4) with SiLU: the stage in front of the SSD layer in a Mamba-2 block,
// over the channels (x, B, C) = d_inner + 2 G N.  Its only state across a sequence cut is the last three
// inputs per channel, which is why Appendix C of the paper counts (d_conv - 1)(d_inner + 2 G N) elements of
// "convolution state" into the sequence-axis checkpoint: forward hands the last three tokens of a segment to
// the next one; backward walks the segments right to left and hands the gradient that reaches the three
// tokens in front of a segment to the segment on its left.
//     pre[t,c] = bias[c] + sum_{k<4} w[c,k] u[t-3+k, c]        out = pre * sigmoid(pre)
// Bandwidth-shaped kernels over 512 adjacent channels per CTA, a thread owning 4 of them with a sliding window in
// registers; rows reach shared memory by bulk async copies, one per token row (the channels of a row are contiguous:
// up to 1 KB), so that many kilobytes per SM are in flight without holding registers, and results go straight to
// global memory (8 or 16 bytes per thread, coalesced over the channels).  A CTA walks a range of tokens, streamed through a ring
// of 8-token stages.
// Weight and bias gradients: partials of 64 tokens (short ranges: of a backward CTA), then a fixed-order sum (no atomics).
#include "ssd_internal.h"
#include "ssd_sm100.cuh"

namespace ssd {

using namespace sm100;

namespace {

constexpr int CV_THREADS = 128;   // x 4 channels = 512 channels per CTA
constexpr int CV_CH = 4;          // channels per thread: one 8-byte bf16 vector (16 bytes in fp32)

__device__ __forceinline__ void ld4(const float *p, float *f) {
    const float4 a = *reinterpret_cast<const float4 *>(p);
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w;
}
template <typename T> __device__ __forceinline__ void st4(T *p, const float *f);
template <> __device__ __forceinline__ void st4<float>(float *p, const float *f) {
    *reinterpret_cast<float4 *>(p) = make_float4(f[0], f[1], f[2], f[3]);
}
template <> __device__ __forceinline__ void st4<__nv_bfloat16>(__nv_bfloat16 *p, const float *f) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(f[0], f[1]), hi = __floats2bfloat162_rn(f[2], f[3]);
    uint2 v;
    v.x = *reinterpret_cast<unsigned int *>(&lo);
    v.y = *reinterpret_cast<unsigned int *>(&hi);
    *reinterpret_cast<uint2 *>(p) = v;
}

// Four channels as two pairs, for the packed two-lane fp32 instructions.
template <typename T> __device__ __forceinline__ void ld2x2(const T *p, float2 &a, float2 &b);
template <> __device__ __forceinline__ void ld2x2<float>(const float *p, float2 &a, float2 &b) {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    a = make_float2(v.x, v.y);
    b = make_float2(v.z, v.w);
}
template <> __device__ __forceinline__ void ld2x2<__nv_bfloat16>(const __nv_bfloat16 *p, float2 &a, float2 &b) {
    const uint2 v = *reinterpret_cast<const uint2 *>(p);
    a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.x));
    b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.y));
}
// 1 / (1 + e^-x) from one ex2.approx and one rcp.approx each (relative error of the order of 1e-7; an IEEE division alone would
// cost as much as the rest of an element)
__device__ __forceinline__ float2 sigmoid_fast2(float2 x) {
    const float2 t = __fmul2_rn(x, make_float2(-1.4426950408889634f, -1.4426950408889634f));
    float2 e, r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(t.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(t.y));
    const float2 d = __fadd2_rn(e, make_float2(1.f, 1.f));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(d.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(d.y));
    return r;
}

constexpr int CV_STG_TOK = 8;                  // tokens per stage of a ring
constexpr int CV_RING_THREADS = CV_THREADS + 32;   // four compute warps and the producer warp

// Forward over a range of consecutive tokens: the rows of u stream through a ring of 8-token stages filled by a producer warp
// with one bulk copy per row, and a thread keeps the last three inputs of its four channels in registers, so nothing is read
// twice inside a range.  The arithmetic runs on channel pairs in packed instructions.  Bound by memory in a long call (92 % of the
// copy rate).  One 32-token tile per CTA, staged whole and worked through element by element, left 1.6 waves of CTAs.  4096
// tokens of 5376 channels have 13 us of bytes and take 24 (cold), most of the rest start and end of the launch; the busiest pipe
// is MUFU, two operations an element, at 53 %.
constexpr int CV_FWD_STAGES = 4;
template <typename T>
__global__ void __launch_bounds__(CV_RING_THREADS) k_conv_fwd(const T *u, long long u_bs, const float *w, const float *bias,
                                                              const T *state_in, T *out, T *state_out, int L, int C, int RL) {
    extern __shared__ __align__(128) unsigned char cv_smem[];
    __shared__ uint64_t full[CV_FWD_STAGES], empty[CV_FWD_STAGES];
    __shared__ uint32_t abort_flag;
    __shared__ unsigned int status_dummy;
    T *ring = reinterpret_cast<T *>(cv_smem);                     // [stage][CV_STG_TOK][512]
    pdl_launch_dependents();
    const int cbase = blockIdx.x * 512, nch = min(512, C - cbase);
    const int b = blockIdx.z;
    const int r_begin = blockIdx.y * RL, ntok = min(RL, L - r_begin), nst = (ntok + CV_STG_TOK - 1) / CV_STG_TOK;
    const T *ub = u + (size_t)b * u_bs;
    const T *sb = state_in ? state_in + (size_t)b * 3 * C : nullptr;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < CV_FWD_STAGES; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], CV_THREADS / 32);
        }
        abort_flag = 0;
        status_dummy = 0;
        fence_barrier_init();
    }
    __syncthreads();
    pdl_wait();       // the previous kernel of the stream (a neighbouring segment's) has finished
    if (warp == CV_THREADS / 32) {
        if (elect_one()) {
            const uint32_t row_bytes = (uint32_t)nch * sizeof(T);
            for (int i = 0; i < nst; ++i) {
                const int slot = i % CV_FWD_STAGES, n = min(CV_STG_TOK, ntok - i * CV_STG_TOK);
                if (i >= CV_FWD_STAGES) mbar_wait(&empty[slot], (i / CV_FWD_STAGES - 1) & 1, &abort_flag, &status_dummy);
                mbar_arrive_expect_tx(&full[slot], (uint32_t)n * row_bytes);
                const T *src = ub + (size_t)(r_begin + i * CV_STG_TOK) * C + cbase;
                T *dst = ring + (size_t)slot * (CV_STG_TOK * 512);
                for (int j = 0; j < n; ++j) bulk_load(dst + (size_t)j * 512, src + (size_t)j * C, row_bytes, &full[slot]);
            }
        }
        return;
    }
    const int c0 = cbase + threadIdx.x * CV_CH;
    const bool active = c0 < C;      // inactive threads (past the last channel) still take part in the hand-overs
    float2 wk[2][4], bs[2], x0[2], x1[2], x2[2], x3[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        wk[i][0] = wk[i][1] = wk[i][2] = wk[i][3] = bs[i] = make_float2(0.f, 0.f);
        x0[i] = x1[i] = x2[i] = x3[i] = make_float2(0.f, 0.f);
    }
    if (active) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float4 wa = *reinterpret_cast<const float4 *>(w + (size_t)(c0 + 2 * i) * 4);
            const float4 wb = *reinterpret_cast<const float4 *>(w + (size_t)(c0 + 2 * i + 1) * 4);
            wk[i][0] = make_float2(wa.x, wb.x); wk[i][1] = make_float2(wa.y, wb.y);
            wk[i][2] = make_float2(wa.z, wb.z); wk[i][3] = make_float2(wa.w, wb.w);
            bs[i] = make_float2(bias[c0 + 2 * i], bias[c0 + 2 * i + 1]);
        }
        // the three inputs in front: of the sequence, else the carried state, else zeros
        auto before = [&](int t, float2 (&v)[2]) {
            if (t >= 0) ld2x2(ub + (size_t)t * C + c0, v[0], v[1]);
            else if (sb) ld2x2(sb + (size_t)(3 + t) * C + c0, v[0], v[1]);
        };
        before(r_begin - 3, x0);
        before(r_begin - 2, x1);
        before(r_begin - 1, x2);
    }
    T *op = out + (size_t)b * u_bs + (size_t)r_begin * C + c0;
    auto token = [&](const T *sp) {
        ld2x2(sp, x3[0], x3[1]);
        float2 o[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float2 pre = __ffma2_rn(wk[i][3], x3[i], __ffma2_rn(wk[i][2], x2[i], __ffma2_rn(wk[i][1], x1[i], __ffma2_rn(wk[i][0], x0[i], bs[i]))));
            o[i] = __fmul2_rn(pre, sigmoid_fast2(pre));
            x0[i] = x1[i]; x1[i] = x2[i]; x2[i] = x3[i];
        }
        const float f[4] = {o[0].x, o[0].y, o[1].x, o[1].y};
        st4(op, f);
        op += C;
    };
    for (int i = 0; i < nst; ++i) {
        const int slot = i % CV_FWD_STAGES, n = min(CV_STG_TOK, ntok - i * CV_STG_TOK);
        mbar_wait(&full[slot], (i / CV_FWD_STAGES) & 1, &abort_flag, &status_dummy);
        if (active) {
            const T *sp = ring + (size_t)slot * (CV_STG_TOK * 512) + threadIdx.x * CV_CH;
            if (n == CV_STG_TOK) {
#pragma unroll
                for (int j = 0; j < CV_STG_TOK; ++j) token(sp + j * 512);
            } else {
                for (int j = 0; j < n; ++j) token(sp + j * 512);
            }
        }
        fence_proxy_async_smem();                      // its reads are over before a bulk copy may overwrite the stage
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[slot]);      // this warp has read the stage
    }
    // the last three inputs of the segment are the state of the next one
    if (active && state_out && r_begin + ntok == L) {
        T *so = state_out + (size_t)b * 3 * C + c0;
        const float f0[4] = {x0[0].x, x0[0].y, x0[1].x, x0[1].y}, f1[4] = {x1[0].x, x1[0].y, x1[1].x, x1[1].y},
                    f2[4] = {x2[0].x, x2[0].y, x2[1].x, x2[1].y};
        st4(so, f0);
        st4(so + (size_t)C, f1);
        st4(so + (size_t)2 * C, f2);
    }
}

// Backward over a range of consecutive tokens.  dpre[t] = dout[t] * silu'(pre[t]);  du[t] = sum_k w[k] dpre[t+3-k].
// A CTA owns 512 channels and walks its range front to back with the last three inputs and the last four dpre in
// registers, so nothing is staged or formed twice inside the range; only at its end does it form dpre of the three
// tokens behind it (for its own last du's; past the end of the segment they are not formed: their effect arrives
// as `dtail`).  The rows of u and dout stream through a ring of 8-token stages filled by a producer warp with one
// bulk copy per row, so the loads of later stages are in flight while a stage is being consumed.
// dw, dbias: partials of the range's own tokens.
// Neither arithmetic nor memory bounds a call of 4096 tokens (5376 channels: 20 us of bytes; issue 42 %, FMA 36 %, MUFU 28 %, DRAM 30 % with
// ranges of ten stages) but the start and end of a range, which loads cover only in part.
// Long ranges (64 tokens and more) take three CTAs per SM with four stages in place of four with three: the longer range covers its start
// and end better (eight segments of 4096 tokens, forward + backward: 515 -> 490 us, of which the sums after 64 tokens cost 14; five CTAs with
// two stages 762, two waves of shorter ranges 520).  The fp32 sums of dw and dbias end after 64 tokens, whatever the range.
// A call's backward, us, with four CTAs and with three, by the range that four have (fp32: 131 KB of ring, so one CTA on an SM; it counts as three):
//   5376 channels, tokens      2048 (40)   4096 (80)   8192 (160)   16384 (312)   32768 (624)     1792 channels: 8192 (56)   16384 (112)
//     bf16                      29  28      49  45      78  72       135 123       252 226                      37  36        62  58
//     fp32                      41  41      64  62      105 102      192 183       370 351                      50  53        80  79
constexpr int CV_SUM_STAGES = 8, CV_LONG = CV_SUM_STAGES * CV_STG_TOK;

template <typename T, int CV_STAGES, int CTAS>
__global__ void __launch_bounds__(CV_RING_THREADS, CTAS)
k_conv_bwd(const T *u, long long u_bs, const float *w, const float *bias, const T *state_in, const T *dout,
           const float *dtail, T *du, float *dstate, float *part, int L, int C, int RL, int parts) {
    extern __shared__ __align__(128) unsigned char cv_smem[];
    __shared__ uint64_t full[CV_STAGES], empty[CV_STAGES];
    __shared__ uint32_t abort_flag;
    __shared__ unsigned int status_dummy;
    T *ring = reinterpret_cast<T *>(cv_smem);                     // [stage][u rows | dout rows][512]
    pdl_launch_dependents();
    const int cbase = blockIdx.x * 512, nch = min(512, C - cbase);
    const int b = blockIdx.z;
    const long long r_begin = (long long)blockIdx.y * RL, r_end = min(r_begin + (long long)RL, (long long)L);
    const int ntok = (int)(r_end - r_begin), nst = (ntok + CV_STG_TOK - 1) / CV_STG_TOK;
    const T *ub = u + (size_t)b * u_bs, *gb = dout + (size_t)b * u_bs;
    const T *sb = state_in ? state_in + (size_t)b * 3 * C : nullptr;
    T *dub = du + (size_t)b * u_bs;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < CV_STAGES; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], CV_THREADS / 32);    // one arrival per compute warp
        }
        abort_flag = 0;
        status_dummy = 0;
        fence_barrier_init();
    }
    __syncthreads();
    pdl_wait();
    // the tokens behind the range, which complete its last du's, are a stage of their own
    const int nbehind = (int)min(3ll, (long long)L - r_end);
    if (warp == CV_THREADS / 32) {
        // ---- producer
        if (elect_one()) {
            const uint32_t row_bytes = (uint32_t)nch * sizeof(T);
            for (int i = 0; i < nst + (nbehind > 0 ? 1 : 0); ++i) {
                const int slot = i % CV_STAGES;
                if (i >= CV_STAGES) mbar_wait(&empty[slot], ((i / CV_STAGES) - 1) & 1, &abort_flag, &status_dummy);
                const long long t0 = i < nst ? r_begin + (long long)i * CV_STG_TOK : r_end;
                const int n = i < nst ? (int)min((long long)CV_STG_TOK, r_end - t0) : nbehind;
                mbar_arrive_expect_tx(&full[slot], 2u * (uint32_t)n * row_bytes);
                T *su = ring + (size_t)slot * (2 * CV_STG_TOK * 512), *sg = su + CV_STG_TOK * 512;
                for (int j = 0; j < n; ++j) {
                    bulk_load(su + (size_t)j * 512, ub + (size_t)(t0 + j) * C + cbase, row_bytes, &full[slot]);
                    bulk_load(sg + (size_t)j * 512, gb + (size_t)(t0 + j) * C + cbase, row_bytes, &full[slot]);
                }
            }
        }
        return;
    }
    const int c0 = cbase + threadIdx.x * CV_CH;
    const bool active = c0 < C;      // inactive threads (past the last channel) still take part in the hand-overs
    // two channel pairs per thread: every quantity below is a float2 over (c, c + 1), so that the multiply-adds
    // issue as packed two-lane instructions
    constexpr int NP = CV_CH / 2;
    const float2 zero2 = make_float2(0.f, 0.f), one2 = make_float2(1.f, 1.f), mone2 = make_float2(-1.f, -1.f);
    float2 wk[NP][4], bs[NP];
    float2 x0[NP], x1[NP], x2[NP], x3[NP];
    float2 d0[NP], d1[NP], d2[NP], d3[NP];     // dpre[t], dpre[t+1], dpre[t+2], dpre[t+3] while emitting du[t]
    float2 aw[NP][4], ab[NP];
    const bool head_range = (dstate != nullptr) && blockIdx.y == 0;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        aw[i][0] = aw[i][1] = aw[i][2] = aw[i][3] = zero2;
        ab[i] = zero2;
        d0[i] = d1[i] = d2[i] = d3[i] = zero2;
        x0[i] = x1[i] = x2[i] = x3[i] = zero2;
        wk[i][0] = wk[i][1] = wk[i][2] = wk[i][3] = bs[i] = zero2;
    }
    // the input at token t of the segment; in front of it the carried state, or zeros
    auto ld_u = [&](long long t, float2 *v) {
        if (t >= 0) ld2x2(ub + (size_t)t * C + c0, v[0], v[1]);
        else if (sb) ld2x2(sb + (size_t)(3 + t) * C + c0, v[0], v[1]);
        else v[0] = v[1] = zero2;
    };
    if (active) {
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const float4 wa = *reinterpret_cast<const float4 *>(w + (size_t)(c0 + 2 * i) * 4);
            const float4 wb = *reinterpret_cast<const float4 *>(w + (size_t)(c0 + 2 * i + 1) * 4);
            wk[i][0] = make_float2(wa.x, wb.x); wk[i][1] = make_float2(wa.y, wb.y);
            wk[i][2] = make_float2(wa.z, wb.z); wk[i][3] = make_float2(wa.w, wb.w);
            bs[i] = make_float2(bias[c0 + 2 * i], bias[c0 + 2 * i + 1]);
        }
        ld_u(r_begin - 3, x0);
        ld_u(r_begin - 2, x1);
        ld_u(r_begin - 1, x2);
    }
    // dpre of token s from its input x3 (the window x0..x2 holds the three before it) and g = dout[s]; own tokens
    // also feed the weight and bias gradients.  Then the windows move on and du[s - 3] is complete.
    // `inner`: a token in a whole stage that is not the range's first; the du it completes lies in the range and meets neither
    // the segment's head nor the gradient from its right, so that nothing is asked per token.
    T *dup = dub + ((size_t)r_begin - 3) * C + c0;       // du of three tokens back
    auto token = [&](long long s, const float2 *g, bool own, bool formed, bool inner) {
        float2 dp[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            if (formed) {
                const float2 pre = __ffma2_rn(wk[i][3], x3[i], __ffma2_rn(wk[i][2], x2[i], __ffma2_rn(wk[i][1], x1[i], __ffma2_rn(wk[i][0], x0[i], bs[i]))));
                const float2 sgm = sigmoid_fast2(pre);
                // dpre = dout * silu'(pre),  silu'(z) = s (1 + z (1 - s))
                dp[i] = __fmul2_rn(__fmul2_rn(g[i], sgm), __ffma2_rn(pre, __ffma2_rn(sgm, mone2, one2), one2));
                if (own) {
                    aw[i][0] = __ffma2_rn(dp[i], x0[i], aw[i][0]);
                    aw[i][1] = __ffma2_rn(dp[i], x1[i], aw[i][1]);
                    aw[i][2] = __ffma2_rn(dp[i], x2[i], aw[i][2]);
                    aw[i][3] = __ffma2_rn(dp[i], x3[i], aw[i][3]);
                    ab[i] = __fadd2_rn(ab[i], dp[i]);
                }
                x0[i] = x1[i]; x1[i] = x2[i]; x2[i] = x3[i];
            } else {
                dp[i] = zero2;
            }
            d0[i] = d1[i]; d1[i] = d2[i]; d2[i] = d3[i]; d3[i] = dp[i];
        }
        if (!inner && head_range && s == 2) {
            // What the first three dpre rows of the segment (now d1, d2, d3) send to the three tokens in front of it:
            // token -3 feeds pre[0] through w[0]; token -2: pre[0] w[1], pre[1] w[0]; token -1: pre[0] w[2], pre[1] w[1],
            // pre[2] w[0].
            float *ds = dstate + (size_t)b * 3 * C + c0;
            float e[CV_CH];
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const float2 v = __fmul2_rn(wk[i][0], d1[i]);
                e[2 * i] = v.x; e[2 * i + 1] = v.y;
            }
            st4(ds, e);
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const float2 v = __ffma2_rn(wk[i][0], d2[i], __fmul2_rn(wk[i][1], d1[i]));
                e[2 * i] = v.x; e[2 * i + 1] = v.y;
            }
            st4(ds + (size_t)C, e);
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const float2 v = __ffma2_rn(wk[i][0], d3[i], __ffma2_rn(wk[i][1], d2[i], __fmul2_rn(wk[i][2], d1[i])));
                e[2 * i] = v.x; e[2 * i + 1] = v.y;
            }
            st4(ds + (size_t)2 * C, e);
        }
        const long long t = s - 3;
        if (inner || t >= r_begin) {
            float o[CV_CH];
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const float2 v = __ffma2_rn(wk[i][3], d0[i], __ffma2_rn(wk[i][2], d1[i], __ffma2_rn(wk[i][1], d2[i], __fmul2_rn(wk[i][0], d3[i]))));
                o[2 * i] = v.x;
                o[2 * i + 1] = v.y;
            }
            if (!inner && dtail && t >= (long long)L - 3) {
                float e[CV_CH];
                ld4(dtail + ((size_t)b * 3 + (size_t)(t - ((long long)L - 3))) * C + c0, e);
#pragma unroll
                for (int i = 0; i < CV_CH; ++i) o[i] += e[i];
            }
            st4(dup, o);
        }
        dup += C;
    };
    // partial weight / bias gradients, a slot per 64 tokens: part[b][slot][5][C]
    const int slots = (RL + CV_LONG - 1) / CV_LONG;
    auto leave_sums = [&](int k64) {
        float *pp = part + (((size_t)b * parts + (size_t)blockIdx.y * slots + k64) * 5) * C + c0;
        float col[CV_CH];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
#pragma unroll
            for (int i = 0; i < NP; ++i) { col[2 * i] = aw[i][k].x; col[2 * i + 1] = aw[i][k].y; aw[i][k] = zero2; }
            st4(pp + (size_t)k * C, col);
        }
#pragma unroll
        for (int i = 0; i < NP; ++i) { col[2 * i] = ab[i].x; col[2 * i + 1] = ab[i].y; ab[i] = zero2; }
        st4(pp + (size_t)4 * C, col);
    };
    for (int i = 0; i < nst; ++i) {
        const int slot = i % CV_STAGES;
        mbar_wait(&full[slot], (i / CV_STAGES) & 1, &abort_flag, &status_dummy);
        if (active) {
            if (i && i % CV_SUM_STAGES == 0) leave_sums(i / CV_SUM_STAGES - 1);
            const T *spu = ring + (size_t)slot * (2 * CV_STG_TOK * 512) + threadIdx.x * CV_CH, *spg = spu + CV_STG_TOK * 512;
            const long long t0 = r_begin + (long long)i * CV_STG_TOK;
            const int n = (int)min((long long)CV_STG_TOK, r_end - t0);
            if (i > 0 && n == CV_STG_TOK) {
#pragma unroll
                for (int j = 0; j < CV_STG_TOK; ++j) {
                    float2 g[NP];
                    ld2x2(spu + (size_t)j * 512, x3[0], x3[1]);
                    ld2x2(spg + (size_t)j * 512, g[0], g[1]);
                    token(t0 + j, g, true, true, true);
                }
            } else {
#pragma unroll 1
                for (int j = 0; j < n; ++j) {
                    float2 g[NP];
                    ld2x2(spu + (size_t)j * 512, x3[0], x3[1]);
                    ld2x2(spg + (size_t)j * 512, g[0], g[1]);
                    token(t0 + j, g, true, true, false);
                }
            }
        }
        fence_proxy_async_smem();                      // its reads are over before a bulk copy may overwrite the stage
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[slot]);      // this warp has read the stage
    }
    if (!active) return;
    // the three tokens behind the range complete its last du's
    const int last = nst % CV_STAGES;
    if (nbehind > 0) mbar_wait(&full[last], (nst / CV_STAGES) & 1, &abort_flag, &status_dummy);
    const T *spu = ring + (size_t)last * (2 * CV_STG_TOK * 512) + threadIdx.x * CV_CH, *spg = spu + CV_STG_TOK * 512;
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        float2 g[NP] = {zero2, zero2};
        const bool formed = k < nbehind;
        if (formed) {
            ld2x2(spu + (size_t)k * 512, x3[0], x3[1]);
            ld2x2(spg + (size_t)k * 512, g[0], g[1]);
        }
        token(r_end + k, g, false, formed, false);
    }
    leave_sums((nst - 1) / CV_SUM_STAGES);
}

// dw[c][k], dbias[c] from the partials of the ranges, in fp64 and in a fixed order: a CTA owns 32 adjacent channels of one of the
// five rows (four taps, bias); its sixteen warps take the ranges round-robin (coalesced 128-byte reads, four in flight), then
// the sixteen sums are added in warp order.
constexpr int CV_RED_WARPS = 16;
__global__ void __launch_bounds__(CV_RED_WARPS * 32) k_conv_reduce(const float *part, float *dw, float *dbias, int C, int total,
                                                                   int accumulate) {
    __shared__ double red[CV_RED_WARPS][32];
    pdl_launch_dependents();
    pdl_wait();
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int nblk = (C + 31) / 32;
    const int k = blockIdx.x / nblk, c = (blockIdx.x % nblk) * 32 + lane;
    double s = 0.0;
    if (c < C) {
        for (int t0 = wp; t0 < total; t0 += 4 * CV_RED_WARPS) {
            float v[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) v[m] = t0 + m * CV_RED_WARPS < total ? part[((size_t)(t0 + m * CV_RED_WARPS) * 5 + k) * C + c] : 0.f;
#pragma unroll
            for (int m = 0; m < 4; ++m) s += (double)v[m];
        }
    }
    red[wp][lane] = s;
    __syncthreads();
    if (wp == 0 && c < C) {
        double tot = 0.0;
#pragma unroll
        for (int i = 0; i < CV_RED_WARPS; ++i) tot += red[i][lane];
        if (k < 4) {
            float *d = dw + (size_t)c * 4 + k;
            *d = accumulate ? *d + (float)tot : (float)tot;
        } else {
            dbias[c] = accumulate ? dbias[c] + (float)tot : (float)tot;
        }
    }
}

// Tokens per CTA: about `per_sm` CTAs per SM over the whole launch, whole stages, at least `least`.
static int conv_range_len(int B, int L, int C, int per_sm, int least) {
    const int nblk = (C + 511) / 512;
    int want = (per_sm * kNumSMs) / (nblk * B);
    if (want < 1) want = 1;
    const int rl = ((L + want - 1) / want + CV_STG_TOK - 1) / CV_STG_TOK * CV_STG_TOK;
    return rl < least ? least : rl;
}

template <typename T>
cudaError_t conv_fwd_t(const T *u, long long u_bs, const float *w, const float *bias, const T *state_in, T *out, T *state_out,
                       int B, int L, int C, cudaStream_t st) {
    const int smem = CV_FWD_STAGES * CV_STG_TOK * 512 * (int)sizeof(T);
    const cudaError_t e = allow_smem<k_conv_fwd<T>>(smem);
    if (e != cudaSuccess) return e;
    const int RL = conv_range_len(B, L, C, sizeof(T) == 2 ? 6 : 3, 16);
    dim3 grid((C + 511) / 512, (L + RL - 1) / RL, B);
    return launch_pdl(k_conv_fwd<T>, grid, dim3(CV_RING_THREADS), (size_t)smem, st, u, u_bs, w, bias, state_in, out, state_out, L, C, RL);
}

// `parts`: partial sums per sequence that the launch leaves
template <typename T>
cudaError_t conv_bwd_t(const T *u, long long u_bs, const float *w, const float *bias, const T *state_in, const T *dout,
                       const float *dtail, T *du, float *dstate, float *part, int B, int L, int C, int &parts, cudaStream_t st) {
    auto launch = [&](auto kernel, int stages, int RL) {
        const int ranges = (L + RL - 1) / RL, last = L - (ranges - 1) * RL;
        parts = (ranges - 1) * ((RL + CV_LONG - 1) / CV_LONG) + (last + CV_LONG - 1) / CV_LONG;      // at most conv_tiles(L)
        return launch_pdl(kernel, dim3((C + 511) / 512, ranges, B), dim3(CV_RING_THREADS), (size_t)stages * 2 * CV_STG_TOK * 512 * sizeof(T), st, u, u_bs, w,
                          bias, state_in, dout, dtail, du, dstate, part, L, C, RL, parts);
    };
    constexpr int row = 2 * CV_STG_TOK * 512 * (int)sizeof(T);
    const int RL = conv_range_len(B, L, C, 4, 32);
    if (RL >= CV_LONG) {
        const cudaError_t e = allow_smem<k_conv_bwd<T, 4, 3>>(4 * row);
        return e != cudaSuccess ? e : launch(k_conv_bwd<T, 4, 3>, 4, conv_range_len(B, L, C, 3, 32));
    }
    const cudaError_t e = allow_smem<k_conv_bwd<T, 3, 4>>(3 * row);
    return e != cudaSuccess ? e : launch(k_conv_bwd<T, 3, 4>, 3, RL);
}

}  // namespace

int conv_tiles(int L) { return (L + 31) / 32; }

cudaError_t launch_conv_fwd(int dtype, const void *u, long long u_bs, const float *w, const float *bias,
                            const void *state_in, void *out, void *state_out, int B, int L, int C, cudaStream_t st) {
    if (dtype == SSD_DTYPE_F32)
        return conv_fwd_t<float>((const float *)u, u_bs, w, bias, (const float *)state_in, (float *)out, (float *)state_out, B,
                                 L, C, st);
    return conv_fwd_t<__nv_bfloat16>((const __nv_bfloat16 *)u, u_bs, w, bias, (const __nv_bfloat16 *)state_in,
                                     (__nv_bfloat16 *)out, (__nv_bfloat16 *)state_out, B, L, C, st);
}

cudaError_t launch_conv_bwd(int dtype, const void *u, long long u_bs, const float *w, const float *bias,
                            const void *state_in, const void *dout, const float *dtail, void *du, float *dstate,
                            float *dw, float *dbias, int accumulate, float *part, int B, int L, int C, cudaStream_t st) {
    cudaError_t e;
    int parts = 0;
    if (dtype == SSD_DTYPE_F32)
        e = conv_bwd_t<float>((const float *)u, u_bs, w, bias, (const float *)state_in, (const float *)dout, dtail, (float *)du,
                              dstate, part, B, L, C, parts, st);
    else
        e = conv_bwd_t<__nv_bfloat16>((const __nv_bfloat16 *)u, u_bs, w, bias, (const __nv_bfloat16 *)state_in,
                                      (const __nv_bfloat16 *)dout, dtail, (__nv_bfloat16 *)du, dstate, part, B, L, C, parts, st);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_conv_reduce, dim3(5 * ((C + 31) / 32)), dim3(CV_RED_WARPS * 32), (size_t)0, st, (const float *)part, dw, dbias, C,
                      parts * B, accumulate);
}

}  // namespace ssd
