// One step of the recurrence of Eq. 1 for autoregressive decoding / forward-only streaming: the state
// is the only thing carried between tokens, so memory does not grow with the sequence.
//     h <- exp(dt A_h) h + dt x B^T ,   y = C h + D_h x          per (batch, head)
// Bandwidth-shaped: the fp32 state is read and written once.
#include "ssd_internal.h"

namespace ssd {

namespace {

template <typename T> __device__ __forceinline__ float ldf(const T *p);
template <> __device__ __forceinline__ float ldf<float>(const float *p) { return __ldg(p); }
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
template <typename T> __device__ __forceinline__ void stf(T *p, float v);
template <> __device__ __forceinline__ void stf<float>(float *p, float v) { *p = v; }
template <> __device__ __forceinline__ void stf<__nv_bfloat16>(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }

// rows = B*H*P.  A row is held by N/4 lanes, 16 bytes each; a warp takes ROWS rows of one head at a time, so that ROWS
// (N = 128) or ROWS/2 (N = 64) independent 16-byte loads per lane are in flight and B, C, dt, A are fetched once for all of
// them.  Bound by the state traffic: with one row per warp and one load in flight the kernel ran at 3.5 TB/s.  The ROWS
// sums over a row's lanes meet in a transposing butterfly, which leaves a row's y in one lane group.
template <typename T> __device__ __forceinline__ void ld4(const T *p, float *f);
template <> __device__ __forceinline__ void ld4<float>(const float *p, float *f) {
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
}
template <> __device__ __forceinline__ void ld4<__nv_bfloat16>(const __nv_bfloat16 *p, float *f) {
    const uint2 v = __ldg(reinterpret_cast<const uint2 *>(p));
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.y));
    f[0] = a.x; f[1] = a.y; f[2] = b.x; f[3] = b.y;
}

constexpr int DEC_WARPS = 4;

template <typename T, int N, int ROWS>
__global__ void __launch_bounds__(DEC_WARPS * 32) k_decode_step(const T *x, const float *dt, const float *A, const T *Bm, const T *Cm,
                                                                const float *D, float *h, T *y, int H, int P, int G, long long groups,
                                                                long long x_bs, long long dt_bs, long long bc_bs) {
    constexpr int LPR = N / 4, RPW = 32 / LPR, NL = ROWS / RPW > 0 ? ROWS / RPW : 1;   // lanes per row, rows per load, loads
    pdl_launch_dependents();
    pdl_wait();
    const int lane = threadIdx.x & 31, sub = lane / LPR, col = (lane % LPR) * 4;
    const long long grp = (long long)blockIdx.x * DEC_WARPS + (threadIdx.x >> 5);   // ROWS consecutive rows, all of one head
    if (grp >= groups) return;
    const long long row0 = grp * ROWS;
    const int p0 = (int)(row0 % P);
    const int hh = (int)((row0 / P) % H);
    const int b = (int)(row0 / ((long long)P * H));
    float *hp = h + (size_t)row0 * N + (size_t)sub * N + col;
    const bool on = sub < ROWS;                        // ROWS = 1 with two rows per load: the upper half idles
    float4 hv[NL];
#pragma unroll
    for (int k = 0; k < NL; ++k) hv[k] = on ? *reinterpret_cast<const float4 *>(hp + (size_t)k * RPW * N) : make_float4(0.f, 0.f, 0.f, 0.f);
    const T *xp = x + (size_t)b * x_bs + (size_t)hh * P + p0;
    float xv[NL], bv[4], cv[4];
#pragma unroll
    for (int k = 0; k < NL; ++k) xv[k] = on ? ldf(xp + k * RPW + sub) : 0.f;
    const size_t bc = (size_t)b * bc_bs + (size_t)(hh / (H / G)) * N + col;
    if ((bc_bs & 3) == 0) {
        ld4(Bm + bc, bv);
        ld4(Cm + bc, cv);
    } else {                                           // a batch stride that leaves a row off the 8-byte grid
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            bv[i] = ldf(Bm + bc + i);
            cv[i] = ldf(Cm + bc + i);
        }
    }
    const float dtv = __ldg(dt + (size_t)b * dt_bs + hh), decay = expf(dtv * __ldg(A + hh)), Dh = __ldg(D + hh);
    float acc[NL];
#pragma unroll
    for (int k = 0; k < NL; ++k) {
        const float dx = dtv * xv[k];
        float4 v = hv[k];
        v.x = fmaf(v.x, decay, dx * bv[0]);
        v.y = fmaf(v.y, decay, dx * bv[1]);
        v.z = fmaf(v.z, decay, dx * bv[2]);
        v.w = fmaf(v.w, decay, dx * bv[3]);
        acc[k] = fmaf(cv[3], v.w, fmaf(cv[2], v.z, fmaf(cv[1], v.y, cv[0] * v.x)));
        if (on) *reinterpret_cast<float4 *>(hp + (size_t)k * RPW * N) = v;
    }
    // sums over the row's lanes: NL values halve at every step until each lane group holds one of them
    int mine = 0;
    int o = LPR / 2;
#pragma unroll
    for (int cnt = NL; cnt > 1; cnt >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < cnt / 2; ++i) {
            const float send = up ? acc[i] : acc[i + cnt / 2], keep = up ? acc[i + cnt / 2] : acc[i];
            acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
        mine += up ? cnt / 2 : 0;
    }
#pragma unroll
    for (; o > 0; o >>= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
    // one lane of each group of LPR / NL writes its row
    if (on && (lane % (LPR / NL)) == 0) {
        const int r = mine * RPW + sub;
        stf(y + (size_t)b * x_bs + (size_t)hh * P + p0 + r, fmaf(Dh, ldf(xp + r), acc[0]));
    }
}

}  // namespace

cudaError_t launch_decode_step(int dtype, int N, const void *x, const float *dt, const float *A, const void *Bm,
                               const void *Cm, const float *D, float *h, void *y, int B, int H, int P, int G,
                               long long x_bs, long long dt_bs, long long bc_bs, cudaStream_t st) {
    const long long rows = (long long)B * H * P;
    // Eight rows per warp where they all belong to one head; few rows (one sequence: 2 048 warps for 32 heads of 64 do not
    // fill the GPU's 148 x 16) are spread over more warps, two rows each.
    const int per = P % 8 == 0 && rows >= 8ll * 148 * 16 ? 8 : P % 2 == 0 ? 2 : 1;
    const long long groups = rows / per;
    const dim3 grid((unsigned)((groups + DEC_WARPS - 1) / DEC_WARPS)), block(DEC_WARPS * 32);
#define SSD_DECODE_ROWS(T, N, ROWS)                                                                                                     \
    return launch_pdl(k_decode_step<T, N, ROWS>, grid, block, 0, st, (const T *)x, dt, A, (const T *)Bm, (const T *)Cm, D, h, (T *)y, H, \
                      P, G, groups, x_bs, dt_bs, bc_bs)
#define SSD_DECODE_CASE(T, N)                    \
    do {                                         \
        if (per == 8) SSD_DECODE_ROWS(T, N, 8);  \
        if (per == 2) SSD_DECODE_ROWS(T, N, 2);  \
        SSD_DECODE_ROWS(T, N, 1);                \
    } while (0)
    if (dtype == SSD_DTYPE_F32) {
        if (N == 128) SSD_DECODE_CASE(float, 128); else SSD_DECODE_CASE(float, 64);
    } else {
        if (N == 128) SSD_DECODE_CASE(__nv_bfloat16, 128); else SSD_DECODE_CASE(__nv_bfloat16, 64);
    }
#undef SSD_DECODE_CASE
#undef SSD_DECODE_ROWS
}

}  // namespace ssd
