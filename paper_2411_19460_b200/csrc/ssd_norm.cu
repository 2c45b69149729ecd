// Gated RMS normalisation behind the SSD layer in a Mamba-2 block: v = y * silu(z), out = v * rsqrt(mean(v^2) + eps) * gamma,
// the mean taken over groups of `group` adjacent channels (the whole d_inner, or d_inner / G).  Token-local: no state
// crosses a sequence cut, so a segment is just a range of rows.  One CTA owns one group index and a tile of rows; a row of
// a group is held in registers (up to 8 four-channel vectors per thread, 256 threads: groups of up to 8192 channels), so
// every tensor is read once; the sums over a row meet through warp shuffles and shared memory in a fixed order; the
// gradient of gamma is accumulated per CTA over its rows and added over the tiles by a second kernel (no atomics).
#include "ssd_internal.h"
#include "ssd_sm100.cuh"

namespace ssd {

using namespace sm100;

// Partial sums of dgamma that a backward call may leave: one per 16 rows, and one more for each CTA of the staged kernel (at most
// two per SM, of at least four rows each), whose rows may end in the middle of sixteen.
long long gated_norm_tiles(long long rows) {
    const long long a = (rows + 3) / 4 < 2 * kNumSMs ? (rows + 3) / 4 : 2 * kNumSMs;
    return a + (rows + 15) / 16;
}

namespace {

constexpr int GN_THREADS = 256;
constexpr int GN_MAXV = 8;        // four-channel vectors per thread, at most (the kernels are instantiated for 1, 2, 4, 5 and 8)
constexpr int GN_ROWS = 16;       // rows of a partial sum of dgamma, at most; rows per CTA of the kernels without a ring
constexpr int GN_MAX_STAGES = 8;  // rows in flight per CTA in the staged kernels, at most

template <typename T> __device__ __forceinline__ void gld4(const T *p, float *f);
template <> __device__ __forceinline__ void gld4<float>(const float *p, float *f) {
    const float4 a = *reinterpret_cast<const float4 *>(p);
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w;
}
template <> __device__ __forceinline__ void gld4<__nv_bfloat16>(const __nv_bfloat16 *p, float *f) {
    const uint2 v = *reinterpret_cast<const uint2 *>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.y));
    f[0] = a.x; f[1] = a.y; f[2] = b.x; f[3] = b.y;
}
template <typename T> __device__ __forceinline__ void gst4(T *p, const float *f);
template <> __device__ __forceinline__ void gst4<float>(float *p, const float *f) {
    *reinterpret_cast<float4 *>(p) = make_float4(f[0], f[1], f[2], f[3]);
}
template <> __device__ __forceinline__ void gst4<__nv_bfloat16>(__nv_bfloat16 *p, const float *f) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(f[0], f[1]), hi = __floats2bfloat162_rn(f[2], f[3]);
    uint2 v;
    v.x = *reinterpret_cast<unsigned int *>(&lo);
    v.y = *reinterpret_cast<unsigned int *>(&hi);
    *reinterpret_cast<uint2 *>(p) = v;
}
__device__ __forceinline__ float sigmoid_gn(float x) {
    float e, r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x * -1.4426950408889634f));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.f + e));
    return r;
}
// sum over the CTA in a fixed order: lanes by shuffle tree, then the eight warps in order
__device__ __forceinline__ float block_sum(float v, float *red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();                       // red may still be read from the previous call
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < GN_THREADS / 32; ++w) s += red[w];
    return s;
}

template <typename T, int NV>
__global__ void __launch_bounds__(GN_THREADS) k_gated_norm_fwd(const T *y, const T *z, const float *gamma, float eps, T *out,
                                                               long long rows, int D, int group) {
    __shared__ float red[GN_THREADS / 32];
    const int gi = blockIdx.y, nv = group / 4;
    const long long r0 = (long long)blockIdx.x * GN_ROWS, r1 = min(r0 + (long long)GN_ROWS, rows);
    float gm[NV][4];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        const int i = threadIdx.x + k * GN_THREADS;
        if (i < nv) gld4(gamma + (size_t)gi * group + (size_t)i * 4, gm[k]);
    }
    for (long long r = r0; r < r1; ++r) {
        const size_t base = (size_t)r * D + (size_t)gi * group;
        float v[NV][4];
        float ss = 0.f;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const int i = threadIdx.x + k * GN_THREADS;
            if (i < nv) {
                float a[4], b[4];
                gld4(y + base + (size_t)i * 4, a);
                gld4(z + base + (size_t)i * 4, b);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    v[k][e] = a[e] * b[e] * sigmoid_gn(b[e]);
                    ss = fmaf(v[k][e], v[k][e], ss);
                }
            }
        }
        const float n = rsqrtf(block_sum(ss, red) / (float)group + eps);
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const int i = threadIdx.x + k * GN_THREADS;
            if (i < nv) {
                float o[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) o[e] = v[k][e] * n * gm[k][e];
                gst4(out + base + (size_t)i * 4, o);
            }
        }
    }
}

template <typename T, int NV>
__global__ void __launch_bounds__(GN_THREADS, NV <= 5 ? 2 : 1) k_gated_norm_bwd(const T *y, const T *z, const float *gamma, float eps,
                                                               const T *dout, T *dy, T *dz, float *part, long long rows, int D,
                                                               int group) {
    __shared__ float red[GN_THREADS / 32];
    const int gi = blockIdx.y, nv = group / 4;
    const long long r0 = (long long)blockIdx.x * GN_ROWS, r1 = min(r0 + (long long)GN_ROWS, rows);
    float gm[NV][4], dg[NV][4];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        const int i = threadIdx.x + k * GN_THREADS;
        if (i < nv) gld4(gamma + (size_t)gi * group + (size_t)i * 4, gm[k]);
#pragma unroll
        for (int e = 0; e < 4; ++e) dg[k][e] = 0.f;
    }
    for (long long r = r0; r < r1; ++r) {
        const size_t base = (size_t)r * D + (size_t)gi * group;
        float v[NV][4], zz[NV][4], yy[NV][4], g[NV][4];
        float ss = 0.f;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const int i = threadIdx.x + k * GN_THREADS;
            if (i < nv) {
                gld4(y + base + (size_t)i * 4, yy[k]);
                gld4(z + base + (size_t)i * 4, zz[k]);
                gld4(dout + base + (size_t)i * 4, g[k]);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    v[k][e] = yy[k][e] * zz[k][e] * sigmoid_gn(zz[k][e]);
                    ss = fmaf(v[k][e], v[k][e], ss);
                }
            }
        }
        const float n = rsqrtf(block_sum(ss, red) / (float)group + eps);
        // xh = v n ;  dvh = dout gamma ;  c = mean(dvh xh) ;  dv = n (dvh - xh c)
        float dot = 0.f;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const int i = threadIdx.x + k * GN_THREADS;
            if (i < nv) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float xh = v[k][e] * n;
                    dg[k][e] = fmaf(g[k][e], xh, dg[k][e]);
                    dot = fmaf(g[k][e] * gm[k][e], xh, dot);
                }
            }
        }
        const float cmean = block_sum(dot, red) / (float)group;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const int i = threadIdx.x + k * GN_THREADS;
            if (i < nv) {
                float oy[4], oz[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float xh = v[k][e] * n;
                    const float dv = n * fmaf(-xh, cmean, g[k][e] * gm[k][e]);
                    const float sg = sigmoid_gn(zz[k][e]);
                    oy[e] = dv * zz[k][e] * sg;                                         // d silu(z) y / dy
                    oz[e] = dv * yy[k][e] * sg * fmaf(zz[k][e], 1.f - sg, 1.f);          // y silu'(z)
                }
                gst4(dy + base + (size_t)i * 4, oy);
                gst4(dz + base + (size_t)i * 4, oz);
            }
        }
    }
    // this CTA's part of dgamma: part[tile][D]
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        const int i = threadIdx.x + k * GN_THREADS;
        if (i < nv) gst4(part + (size_t)blockIdx.x * D + (size_t)gi * group + (size_t)i * 4, dg[k]);
    }
}

// ---- staged kernels, for rows that fit: the rows of a CTA stream through a ring of shared-memory buffers filled by bulk async
// copies (one per tensor and row: the channels of a group are contiguous), several rows ahead.  A row goes from its buffer to
// registers once, in the I/O type, both of its sums (sum v^2, and in the backward sum dout gamma v, which is all that
// mean(dvh xh) needs) meet in ONE CTA barrier, after which the buffer is free again, and the rest is arithmetic on channel
// pairs in packed instructions.  Bound by memory: with two barriers per sum and one more per row, and element by element, the
// kernels were at 48 (forward) and 49 % (backward) of the copy peak at 4096 rows of 5120 bf16 channels, now at 78 %.
struct Sums { float ss, dt; };

template <typename T> struct Raw;
template <> struct Raw<__nv_bfloat16> {
    uint2 v;
    __device__ __forceinline__ void load(const __nv_bfloat16 *p) { v = *reinterpret_cast<const uint2 *>(p); }
    __device__ __forceinline__ float2 pair(int i) const {
        const unsigned w = i ? v.y : v.x;
        return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
    }
};
template <> struct Raw<float> {
    float4 v;
    __device__ __forceinline__ void load(const float *p) { v = *reinterpret_cast<const float4 *>(p); }
    __device__ __forceinline__ float2 pair(int i) const { return i ? make_float2(v.z, v.w) : make_float2(v.x, v.y); }
};
__device__ __forceinline__ void st_pairs(float *p, float2 a, float2 b) { *reinterpret_cast<float4 *>(p) = make_float4(a.x, a.y, b.x, b.y); }
__device__ __forceinline__ void st_pairs(__nv_bfloat16 *p, float2 a, float2 b) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(a.x, a.y), hi = __floats2bfloat162_rn(b.x, b.y);
    uint2 v;
    v.x = *reinterpret_cast<const unsigned int *>(&lo);
    v.y = *reinterpret_cast<const unsigned int *>(&hi);
    *reinterpret_cast<uint2 *>(p) = v;
}
__device__ __forceinline__ float2 sigmoid_gn2(float2 x) {
    const float2 t = __fmul2_rn(x, make_float2(-1.4426950408889634f, -1.4426950408889634f));
    float2 e, r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(t.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(t.y));
    const float2 d = __fadd2_rn(e, make_float2(1.f, 1.f));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(d.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(d.y));
    return r;
}

template <typename T, int NV, bool BWD>
__global__ void __launch_bounds__(GN_THREADS, sizeof(T) == 2 ? 2 : 1)
k_gated_norm_staged(const T *y, const T *z, const float *gamma, float eps, const T *dout, T *out_or_dy, T *dz, float *part, long long rows, int D,
                    int group, int rpc, int stages) {
    extern __shared__ __align__(128) unsigned char gn_smem[];
    __shared__ float2 red[2][GN_THREADS / 32];
    __shared__ uint64_t full[GN_MAX_STAGES];
    __shared__ uint32_t abort_flag;
    __shared__ unsigned int status_dummy;
    constexpr int NT = BWD ? 3 : 2;                       // tensors staged per row
    const int gi = blockIdx.y, nv = group / 4, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long r0 = (long long)blockIdx.x * rpc;
    const int nrows = (int)min((long long)rpc, rows - r0);
    const uint32_t row_bytes = (uint32_t)group * sizeof(T);
    const size_t base0 = (size_t)r0 * D + (size_t)gi * group;
    T *ring = reinterpret_cast<T *>(gn_smem);             // [stages][NT][group]
    auto issue = [&](int j, int st) {                     // thread 0: row j of this CTA into stage st
        const size_t base = base0 + (size_t)j * D;
        T *dst = ring + (size_t)st * NT * group;
        mbar_arrive_expect_tx(&full[st], NT * row_bytes);
        bulk_load(dst, y + base, row_bytes, &full[st]);
        bulk_load(dst + group, z + base, row_bytes, &full[st]);
        if (BWD) bulk_load(dst + 2 * (size_t)group, dout + base, row_bytes, &full[st]);
    };
    if (threadIdx.x == 0) {
        for (int i = 0; i < stages; ++i) mbar_init(&full[i], 1);
        abort_flag = 0;
        status_dummy = 0;
        fence_barrier_init();
        pdl_wait();
        for (int j = 0; j < stages && j < nrows; ++j) issue(j, j);
    }
    pdl_wait();
    float2 gm[NV][2], dg[NV][2];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        const int i = threadIdx.x + k * GN_THREADS;
        float4 g4 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < nv) g4 = *reinterpret_cast<const float4 *>(gamma + (size_t)gi * group + (size_t)i * 4);
        gm[k][0] = make_float2(g4.x, g4.y);
        gm[k][1] = make_float2(g4.z, g4.w);
        dg[k][0] = dg[k][1] = make_float2(0.f, 0.f);
    }
    // Row j ends a partial sum of dgamma: fp32 over 16 rows at most, whatever a CTA's share of a long call, fp64 from there on
    auto leave_sum = [&](int j) {
        const size_t tile = (size_t)blockIdx.x * ((rpc + GN_ROWS - 1) / GN_ROWS) + j / GN_ROWS;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const int i = threadIdx.x + k * GN_THREADS;
            if (i < nv) st_pairs(part + tile * D + (size_t)gi * group + (size_t)i * 4, dg[k][0], dg[k][1]);
            dg[k][0] = dg[k][1] = make_float2(0.f, 0.f);
        }
    };
    __syncthreads();
    const float rgroup = 1.f / (float)group;
    int st = 0;
    uint32_t par = 0;
    for (int j = 0; j < nrows; ++j) {
        mbar_wait(&full[st], par, &abort_flag, &status_dummy);
        const T *sy = ring + (size_t)st * NT * group, *sz = sy + group, *sg = sy + 2 * (size_t)group;
        Raw<T> ry[NV], rg[BWD ? NV : 1];
        float2 q[NV][2], sgm[BWD ? NV : 1][2];            // q = z sigmoid(z)
        float2 ss = make_float2(0.f, 0.f), dt = ss;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const int i = threadIdx.x + k * GN_THREADS;
            if (i < nv) {
                Raw<T> rz;
                ry[k].load(sy + (size_t)i * 4);
                rz.load(sz + (size_t)i * 4);
                if (BWD) rg[k].load(sg + (size_t)i * 4);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float2 zz = rz.pair(e), s = sigmoid_gn2(zz);
                    q[k][e] = __fmul2_rn(zz, s);
                    const float2 v = __fmul2_rn(ry[k].pair(e), q[k][e]);
                    ss = __ffma2_rn(v, v, ss);
                    if (BWD) {
                        sgm[k][e] = s;
                        dt = __ffma2_rn(__fmul2_rn(rg[k].pair(e), gm[k][e]), v, dt);
                    } else {
                        q[k][e] = v;                      // the forward needs v only
                    }
                }
            }
        }
        float2 sum = make_float2(ss.x + ss.y, dt.x + dt.y);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sum.x += __shfl_xor_sync(0xffffffffu, sum.x, o);
            if (BWD) sum.y += __shfl_xor_sync(0xffffffffu, sum.y, o);
        }
        if (lane == 0) red[j & 1][warp] = sum;
        fence_proxy_async_smem();                         // this thread's reads are over before a bulk copy may overwrite the stage
        __syncthreads();                                  // the sums are there, and every thread has read the stage
        if (threadIdx.x == 0 && j + stages < nrows) issue(j + stages, st);
        if (++st == stages) { st = 0; par ^= 1u; }
        sum = red[j & 1][0];
#pragma unroll
        for (int w = 1; w < GN_THREADS / 32; ++w) {
            const float2 t = red[j & 1][w];
            sum.x += t.x;
            sum.y += t.y;
        }
        const float n = rsqrtf(sum.x * rgroup + eps);
        const float2 n2 = make_float2(n, n);
        const size_t base = base0 + (size_t)j * D;
        // xh = v n ;  dvh = dout gamma ;  c = mean(dvh xh) ;  dv = n (dvh - xh c).  No power of n by itself: it leaves the range of
        // fp32 where v, its square and the gradient do not.
        const float c = n * sum.y * rgroup;
        const float2 c2 = make_float2(-c, -c), one2 = make_float2(1.f, 1.f);
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const int i = threadIdx.x + k * GN_THREADS;
            if (i < nv) {
                float2 o1[2], o2[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    if (!BWD) {
                        o1[e] = __fmul2_rn(__fmul2_rn(q[k][e], n2), gm[k][e]);
                    } else {
                        const float2 yy = ry[k].pair(e), g = rg[k].pair(e), qq = q[k][e], s = sgm[k][e];
                        const float2 v = __fmul2_rn(yy, qq);
                        const float2 xh = __fmul2_rn(v, n2);
                        dg[k][e] = __ffma2_rn(g, xh, dg[k][e]);
                        const float2 dv = __fmul2_rn(n2, __ffma2_rn(xh, c2, __fmul2_rn(g, gm[k][e])));
                        o1[e] = __fmul2_rn(dv, qq);                                       // y silu(z): d / dy
                        // silu'(z) = s (1 + z (1 - s)) = s + q (1 - s)
                        const float2 ds = __ffma2_rn(qq, __ffma2_rn(s, make_float2(-1.f, -1.f), one2), s);
                        o2[e] = __fmul2_rn(dv, __fmul2_rn(yy, ds));
                    }
                }
                st_pairs(out_or_dy + base + (size_t)i * 4, o1[0], o1[1]);
                if (BWD) st_pairs(dz + base + (size_t)i * 4, o2[0], o2[1]);
            }
        }
        if (BWD && (j + 1) % GN_ROWS == 0 && j + 1 < nrows) leave_sum(j);
    }
    pdl_launch_dependents();     // not earlier: the next launch fills the GPU in one wave and wants it free
    if (BWD) leave_sum(nrows - 1);
}

// Ring of a staged launch: as many rows as fit 110 KB (two CTAs per SM, bf16) or else 220 KB; 0: not even two rows fit.
struct StagedPlan { int stages, rpc; };
template <typename T> StagedPlan staged_plan(long long rows, int D, int group, int tensors) {
    const int need = (group / 4 + GN_THREADS - 1) / GN_THREADS, stage = tensors * group * (int)sizeof(T);
    if (need > 5 || (group * sizeof(T)) % 16) return {0, 0};
    int stages = 110 * 1024 / stage, per_sm = sizeof(T) == 2 ? 2 : 1;
    if (stages < 2 || per_sm == 1) {
        stages = 220 * 1024 / stage;
        per_sm = 1;
    }
    if (stages < 2) return {0, 0};
    if (stages > GN_MAX_STAGES) stages = GN_MAX_STAGES;
    // rows per CTA: one even wave over the GPU, at least four (the ring has to fill)
    const long long ctas = (long long)kNumSMs * per_sm / (D / group) > 0 ? (long long)kNumSMs * per_sm / (D / group) : 1;
    long long rpc = (rows + ctas - 1) / ctas;
    if (rpc < 4) rpc = 4;
    return {stages, (int)rpc};
}

// dgamma from the partial sums, in fp64 and in a fixed order: a CTA owns 32 adjacent channels; its 32 warps take the partials
// round-robin, eight loads in flight each, then the 32 sums are added in warp order.  A few microseconds of latency behind
// every backward call: with eight warps and four loads in flight it took 10 us for 293 partials.
__global__ void __launch_bounds__(1024) k_gated_norm_reduce(const float *part, float *dgamma, int D, int ntiles, int accumulate) {
    __shared__ double red[32][32];
    pdl_wait();
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int c = blockIdx.x * 32 + lane;
    double s = 0.0;
    if (c < D) {
        for (int t0 = wp; t0 < ntiles; t0 += 8 * 32) {
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = t0 + 32 * k < ntiles ? part[(size_t)(t0 + 32 * k) * D + c] : 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) s += (double)v[k];
        }
    }
    red[wp][lane] = s;
    __syncthreads();
    if (wp == 0 && c < D) {
        double tot = 0.0;
#pragma unroll
        for (int i = 0; i < 32; ++i) tot += red[i][lane];
        dgamma[c] = accumulate ? dgamma[c] + (float)tot : (float)tot;
    }
}

}  // namespace

int gated_norm_max_group() { return GN_MAXV * GN_THREADS * 4; }

template <typename T, int NV, bool BWD>
static cudaError_t launch_staged(const StagedPlan &pl, const T *y, const T *z, const float *gamma, float eps, const T *dout, T *o1, T *o2, float *part,
                                 long long rows, int D, int group, cudaStream_t st) {
    const size_t ring = (size_t)pl.stages * (BWD ? 3 : 2) * group * sizeof(T);
    const cudaError_t e = allow_smem<k_gated_norm_staged<T, NV, BWD>>(220 * 1024);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_gated_norm_staged<T, NV, BWD>, dim3((unsigned)((rows + pl.rpc - 1) / pl.rpc), D / group), dim3(GN_THREADS), ring, st, y, z,
                      gamma, eps, dout, o1, o2, part, rows, D, group, pl.rpc, pl.stages);
}
// 4-channel vectors per thread, rounded up to an instantiated count
#define GN_BY_NEED(CALL)           \
    do {                           \
        if (need <= 1) CALL(1);    \
        if (need <= 2) CALL(2);    \
        if (need <= 4) CALL(4);    \
        if (need <= 5) CALL(5);    \
    } while (0)
template <typename T>
static cudaError_t norm_fwd_t(const T *y, const T *z, const float *gamma, float eps, T *out, long long rows, int D, int group,
                              cudaStream_t st) {
    const int need = (group / 4 + GN_THREADS - 1) / GN_THREADS;
    const StagedPlan pl = staged_plan<T>(rows, D, group, 2);
    if (pl.stages) {
#define GN_CASE(NV) return launch_staged<T, NV, false>(pl, y, z, gamma, eps, (const T *)nullptr, out, (T *)nullptr, (float *)nullptr, rows, D, group, st)
        GN_BY_NEED(GN_CASE);
#undef GN_CASE
    }
    const dim3 grid((unsigned)((rows + GN_ROWS - 1) / GN_ROWS), D / group);
#define GN_CASE(NV) return k_gated_norm_fwd<T, NV><<<grid, GN_THREADS, 0, st>>>(y, z, gamma, eps, out, rows, D, group), cudaGetLastError()
    GN_BY_NEED(GN_CASE);
    GN_CASE(8);
#undef GN_CASE
}
// `parts`: how many partial sums of dgamma the launch leaves
template <typename T>
static cudaError_t norm_bwd_t(const T *y, const T *z, const float *gamma, float eps, const T *dout, T *dy, T *dz, float *part,
                              long long rows, int D, int group, int &parts, cudaStream_t st) {
    const int need = (group / 4 + GN_THREADS - 1) / GN_THREADS;
    const StagedPlan pl = staged_plan<T>(rows, D, group, 3);
    if (pl.stages) {
        const long long full = (rows - 1) / pl.rpc, last = rows - full * pl.rpc;      // CTAs before the last one, its rows
        parts = (int)(full * ((pl.rpc + GN_ROWS - 1) / GN_ROWS) + (last + GN_ROWS - 1) / GN_ROWS);
#define GN_CASE(NV) return launch_staged<T, NV, true>(pl, y, z, gamma, eps, dout, dy, dz, part, rows, D, group, st)
        GN_BY_NEED(GN_CASE);
#undef GN_CASE
    }
    parts = (int)((rows + GN_ROWS - 1) / GN_ROWS);
    const dim3 grid((unsigned)parts, D / group);
#define GN_CASE(NV) return k_gated_norm_bwd<T, NV><<<grid, GN_THREADS, 0, st>>>(y, z, gamma, eps, dout, dy, dz, part, rows, D, group), cudaGetLastError()
    GN_BY_NEED(GN_CASE);
    GN_CASE(8);
#undef GN_CASE
}
#undef GN_BY_NEED

cudaError_t launch_gated_norm_fwd(int dtype, const void *y, const void *z, const float *gamma, float eps, void *out,
                                  long long rows, int D, int group, cudaStream_t st) {
    if (dtype == SSD_DTYPE_F32) return norm_fwd_t<float>((const float *)y, (const float *)z, gamma, eps, (float *)out, rows, D, group, st);
    return norm_fwd_t<__nv_bfloat16>((const __nv_bfloat16 *)y, (const __nv_bfloat16 *)z, gamma, eps, (__nv_bfloat16 *)out, rows, D,
                                     group, st);
}

cudaError_t launch_gated_norm_bwd(int dtype, const void *y, const void *z, const float *gamma, float eps, const void *dout,
                                  void *dy, void *dz, float *dgamma, int accumulate, float *part, long long rows, int D,
                                  int group, cudaStream_t st) {
    cudaError_t e;
    int parts = 0;
    if (dtype == SSD_DTYPE_F32)
        e = norm_bwd_t<float>((const float *)y, (const float *)z, gamma, eps, (const float *)dout, (float *)dy, (float *)dz, part,
                              rows, D, group, parts, st);
    else
        e = norm_bwd_t<__nv_bfloat16>((const __nv_bfloat16 *)y, (const __nv_bfloat16 *)z, gamma, eps, (const __nv_bfloat16 *)dout,
                                      (__nv_bfloat16 *)dy, (__nv_bfloat16 *)dz, part, rows, D, group, parts, st);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_gated_norm_reduce, dim3((D + 31) / 32), dim3(1024), 0, st, (const float *)part, dgamma, D, parts, accumulate);
}

}  // namespace ssd
