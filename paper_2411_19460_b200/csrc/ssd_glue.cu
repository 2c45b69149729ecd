// Layer-axis glue for a stack of SSD layers under Multi-Axis Gradient Checkpointing (Algorithms 1
// and 2 of the paper keep only each layer's INPUT along the layer axis): layer j maps x_j to
// y_j = SSD_j(x_j) and hands x_{j+1} = W (y_j + x_j) to the next layer, W a fixed P x P mixing matrix
// applied per (batch, step, head).  Backward: dz = W^T g_{j+1}; dy_j = dz; dx_j = (SSD backward) + dz.
// Bandwidth-shaped kernels; bf16 or fp32 I/O.  fp32: CUDA cores, fp32 arithmetic.  bf16: the 64 x 64 product runs on
// the tensor cores through warp-level mma (W rounded to bf16 once per CTA, fp32 accumulation): at 4096 multiply-adds
// per 128-byte row the CUDA-core version was five times over its memory time.
#include "ssd_internal.h"

namespace ssd {

namespace {

template <typename T> __device__ __forceinline__ void load_row64(const T *src, float *z);
template <> __device__ __forceinline__ void load_row64<float>(const float *src, float *z) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(src) + k);
        z[4 * k] = v.x; z[4 * k + 1] = v.y; z[4 * k + 2] = v.z; z[4 * k + 3] = v.w;
    }
}
template <> __device__ __forceinline__ void load_row64<__nv_bfloat16>(const __nv_bfloat16 *src, float *z) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(src) + k);
        const __nv_bfloat162 *e = reinterpret_cast<const __nv_bfloat162 *>(&v);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 f = __bfloat1622float2(e[i]);
            z[8 * k + 2 * i] = f.x;
            z[8 * k + 2 * i + 1] = f.y;
        }
    }
}
template <typename T> __device__ __forceinline__ void store4(T *dst, float a, float b, float c, float d);
template <> __device__ __forceinline__ void store4<float>(float *dst, float a, float b, float c, float d) {
    *reinterpret_cast<float4 *>(dst) = make_float4(a, b, c, d);
}
template <> __device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16 *dst, float a, float b, float c, float d) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
    uint2 pk;
    pk.x = *reinterpret_cast<unsigned int *>(&lo);
    pk.y = *reinterpret_cast<unsigned int *>(&hi);
    *reinterpret_cast<uint2 *>(dst) = pk;
}

// out[row, i] = sum_j M[i][j] (a[row, j] + b[row, j])   with M = W (TRANSPOSE = false) or W^T (true);
// b may be null.  One thread per 64-vector; M is staged in shared memory as Mt[j][i] so that four
// consecutive outputs come from one broadcast 16-byte read.
template <typename T, bool TRANSPOSE>
__global__ void __launch_bounds__(128) k_glue(const T *a, const T *b, const float *W, T *out, long long rows_per_batch,
                                              long long bstride, int B) {
    __shared__ float Mt[64][64];
    for (int idx = threadIdx.x; idx < 4096; idx += 128) {
        const int r = idx >> 6, cidx = idx & 63;            // W[r][cidx]
        if (TRANSPOSE) Mt[r][cidx] = W[idx];                // M = W^T: M[i][j] = W[j][i] -> Mt[j][i] = W[j][i]
        else Mt[cidx][r] = W[idx];                          // M = W  : Mt[j][i] = W[i][j]
    }
    __syncthreads();
    const long long total = rows_per_batch * B;
    for (long long row = (long long)blockIdx.x * 128 + threadIdx.x; row < total; row += (long long)gridDim.x * 128) {
        const long long bb = row / rows_per_batch, rr = row % rows_per_batch;
        const size_t off = (size_t)bb * bstride + (size_t)rr * 64;
        float z[64];
        load_row64(a + off, z);
        if (b) {
            float zb[64];
            load_row64(b + off, zb);
#pragma unroll
            for (int j = 0; j < 64; ++j) z[j] += zb[j];
        }
#pragma unroll 2
        for (int i0 = 0; i0 < 64; i0 += 4) {
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 64; ++j) {
                const float4 m = *reinterpret_cast<const float4 *>(&Mt[j][i0]);
                acc.x = fmaf(m.x, z[j], acc.x);
                acc.y = fmaf(m.y, z[j], acc.y);
                acc.z = fmaf(m.z, z[j], acc.z);
                acc.w = fmaf(m.w, z[j], acc.w);
            }
            store4(out + off + i0, acc.x, acc.y, acc.z, acc.w);
        }
    }
}

// The same product for bf16 rows on the tensor cores (warp-level mma, fp32 accumulation).  A warp owns 16 consecutive rows at a
// time, one contiguous 2 KB block of the row-major [rows][64] tensor, and everything stays in registers: the order of the
// contraction index is free, so a lane's A fragments are the 16-byte pieces it loads (four lanes cover 64 contiguous bytes of a
// row), and so is the order of the output columns, so what a lane stores is two 16-byte pieces per row.  W, rounded to bf16, is
// laid out for both orders once per CTA.  The next tile's rows are requested before the current ones are multiplied.
//   step s of the contraction, lane group j = lane % 4: columns 32 (s / 2) + 8 j + 4 (s % 2) + {0, 1 | 2, 3}
//   output tile t, column c:                            column  32 (t / 4) + 8 (c / 2) + 2 (t % 4) + c % 2
// Bound by memory; with both sides going through shared-memory tiles the kernel took 37 us for 4096 x 80 rows (126 MB).
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&v);
}
template <bool TRANSPOSE, bool ADD>
__global__ void __launch_bounds__(128) k_glue_bf16_mma(const __nv_bfloat16 *a, const __nv_bfloat16 *b, const float *W,
                                                       __nv_bfloat16 *out, long long rows_per_batch, long long bstride, int B) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, j = lane & 3, r = lane >> 2;
    // B operand: element (k, n) = M[n][k], M = W or W^T; this lane holds n-column r of every tile, k pairs of group j
    uint32_t wf[8][4][2];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const int n = 32 * (t >> 2) + 8 * (r >> 1) + 2 * (t & 3) + (r & 1);
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int k = 32 * (s >> 1) + 8 * j + 4 * (s & 1) + 2 * i;
                const float w0 = TRANSPOSE ? W[k * 64 + n] : W[n * 64 + k], w1 = TRANSPOSE ? W[(k + 1) * 64 + n] : W[n * 64 + k + 1];
                wf[t][s][i] = pack_bf16(w0, w1);
            }
    }
    const long long ntiles = rows_per_batch * B / 16, step = (long long)gridDim.x * 4;
    auto tile_offset = [&](long long t) {
        const long long row0 = t * 16, bb = row0 / rows_per_batch, rr = row0 - bb * rows_per_batch;
        return (size_t)bb * bstride + (size_t)rr * 64 + (size_t)r * 64 + j * 8;
    };
    uint4 va[2][2], vb[2][2];      // [row r, r + 8][columns 0.. / 32..]
    auto fetch = [&](size_t off) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                va[h][i] = __ldg(reinterpret_cast<const uint4 *>(a + off + h * 8 * 64 + i * 32));
                if (ADD) vb[h][i] = __ldg(reinterpret_cast<const uint4 *>(b + off + h * 8 * 64 + i * 32));
            }
    };
    long long t = (long long)blockIdx.x * 4 + warp;
    if (t >= ntiles) return;
    size_t off = tile_offset(t);
    fetch(off);
    while (true) {
        uint32_t z[2][2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const uint32_t x[4] = {va[h][i].x, va[h][i].y, va[h][i].z, va[h][i].w}, y[4] = {vb[h][i].x, vb[h][i].y, vb[h][i].z, vb[h][i].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    z[h][i][e] = x[e];
                    if (ADD) {
                        const __nv_bfloat162 s = __hadd2(*reinterpret_cast<const __nv_bfloat162 *>(&x[e]), *reinterpret_cast<const __nv_bfloat162 *>(&y[e]));
                        z[h][i][e] = *reinterpret_cast<const uint32_t *>(&s);
                    }
                }
            }
        const size_t cur = off;
        t += step;
        const bool more = t < ntiles;
        if (more) {
            off = tile_offset(t);
            fetch(off);
        }
        float acc[8][4];
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const uint32_t af[4] = {z[0][s >> 1][2 * (s & 1)], z[1][s >> 1][2 * (s & 1)], z[0][s >> 1][2 * (s & 1) + 1], z[1][s >> 1][2 * (s & 1) + 1]};
                mma_bf16(acc[n], af, wf[n][s][0], wf[n][s][1]);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 2; ++i)
                *reinterpret_cast<uint4 *>(out + cur + h * 8 * 64 + i * 32) =
                    make_uint4(pack_bf16(acc[4 * i][2 * h], acc[4 * i][2 * h + 1]), pack_bf16(acc[4 * i + 1][2 * h], acc[4 * i + 1][2 * h + 1]),
                               pack_bf16(acc[4 * i + 2][2 * h], acc[4 * i + 2][2 * h + 1]), pack_bf16(acc[4 * i + 3][2 * h], acc[4 * i + 3][2 * h + 1]));
        if (!more) break;
    }
}

// dst += src, elementwise over [B][rows_per_batch * 64]
template <typename T>
__global__ void __launch_bounds__(256) k_residual(T *dst, const T *src, long long n_per_batch, long long bstride, int B) {
    const long long total = n_per_batch * B / 4;
    for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < total; i += (long long)gridDim.x * 256) {
        const long long e = i * 4, bb = e / n_per_batch, rr = e % n_per_batch;
        const size_t off = (size_t)bb * bstride + (size_t)rr;
        float d[4], s[4];
        if (sizeof(T) == 4) {
            const float4 dv = *reinterpret_cast<const float4 *>(dst + off), sv = *reinterpret_cast<const float4 *>(src + off);
            d[0] = dv.x; d[1] = dv.y; d[2] = dv.z; d[3] = dv.w;
            s[0] = sv.x; s[1] = sv.y; s[2] = sv.z; s[3] = sv.w;
        } else {
            const uint2 dv = *reinterpret_cast<const uint2 *>(dst + off), sv = *reinterpret_cast<const uint2 *>(src + off);
            const float2 d0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&dv.x));
            const float2 d1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&dv.y));
            const float2 s0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&sv.x));
            const float2 s1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&sv.y));
            d[0] = d0.x; d[1] = d0.y; d[2] = d1.x; d[3] = d1.y;
            s[0] = s0.x; s[1] = s0.y; s[2] = s1.x; s[3] = s1.y;
        }
        store4(dst + off, d[0] + s[0], d[1] + s[1], d[2] + s[2], d[3] + s[3]);
    }
}

}  // namespace

cudaError_t launch_glue(int dtype, bool transpose, const void *a, const void *b, const float *W, void *out,
                        long long rows_per_batch, long long bstride, int B, cudaStream_t st) {
    const long long total = rows_per_batch * B;
    const unsigned blocks = (unsigned)((total + 127) / 128 < 148 * 16 ? (total + 127) / 128 : 148 * 16);
    if (dtype == SSD_DTYPE_F32) {
        if (transpose) k_glue<float, true><<<blocks, 128, 0, st>>>((const float *)a, (const float *)b, W, (float *)out, rows_per_batch, bstride, B);
        else k_glue<float, false><<<blocks, 128, 0, st>>>((const float *)a, (const float *)b, W, (float *)out, rows_per_batch, bstride, B);
    } else if (rows_per_batch % 16 == 0) {
        const long long tiles = total / 16;
        const unsigned most = 148 * 3;      // three CTAs of 160-register threads fit an SM: one wave
        const unsigned mblocks = (unsigned)((tiles + 3) / 4 < most ? (tiles + 3) / 4 : most);
        const __nv_bfloat16 *pa = (const __nv_bfloat16 *)a, *pb = (const __nv_bfloat16 *)b;
        __nv_bfloat16 *po = (__nv_bfloat16 *)out;
        if (transpose) k_glue_bf16_mma<true, false><<<mblocks, 128, 0, st>>>(pa, pb, W, po, rows_per_batch, bstride, B);
        else k_glue_bf16_mma<false, true><<<mblocks, 128, 0, st>>>(pa, pb, W, po, rows_per_batch, bstride, B);
    } else {
        if (transpose) k_glue<__nv_bfloat16, true><<<blocks, 128, 0, st>>>((const __nv_bfloat16 *)a, (const __nv_bfloat16 *)b, W, (__nv_bfloat16 *)out, rows_per_batch, bstride, B);
        else k_glue<__nv_bfloat16, false><<<blocks, 128, 0, st>>>((const __nv_bfloat16 *)a, (const __nv_bfloat16 *)b, W, (__nv_bfloat16 *)out, rows_per_batch, bstride, B);
    }
    return cudaGetLastError();
}

cudaError_t launch_residual(int dtype, void *dst, const void *src, long long n_per_batch, long long bstride, int B,
                            cudaStream_t st) {
    const long long total = n_per_batch * B / 4;
    const unsigned blocks = (unsigned)((total + 255) / 256 < 148 * 32 ? (total + 255) / 256 : 148 * 32);
    if (dtype == SSD_DTYPE_F32) k_residual<float><<<blocks, 256, 0, st>>>((float *)dst, (const float *)src, n_per_batch, bstride, B);
    else k_residual<__nv_bfloat16><<<blocks, 256, 0, st>>>((__nv_bfloat16 *)dst, (const __nv_bfloat16 *)src, n_per_batch, bstride, B);
    return cudaGetLastError();
}

}  // namespace ssd
