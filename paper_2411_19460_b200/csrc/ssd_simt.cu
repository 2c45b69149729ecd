// CUDA-core kernels of libssd: the backward's finishing scans and reductions for every path, and inter-chunk state passing
// and FFMA versions of the contractions, which serve the fp32 mode (1e-4 parity rules out reduced-precision tensor-core
// inputs) and chunks of 64, and cross-check the tensor-core kernels.
//
// Notation per (batch b, head h), chunk of Q steps: a_t = dt_t*A_h, cs_t = inclusive cumsum of a
// inside the chunk, H_in = state entering the chunk, Gout = dLoss/d(state leaving the chunk).
// All of it is Eq. 1 of the paper regrouped by chunks; the segment hand-off is Algorithms 1 and 2.
#include "ssd_internal.h"

// State-pass CTAs: 128 threads, at most 48 registers, so that a segment's CTAs are resident at once; chunks fetched ahead.
#define SP_THREADS 128
#define SP_ELEMS (SP_THREADS * 4)
#define SP_CTAS 10
#define SP_PF 4
static_assert(SP_ELEMS == ssd::kStatePassElems, "one partial of <G,H> per CTA of the backward pass");
namespace ssd {

// ------------------------------------------------------------------ small helpers
__device__ __forceinline__ void add4(float4 &a, const float4 &b) {
    a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
}
__device__ __forceinline__ void st4(float *p, const float4 &v) { *reinterpret_cast<float4 *>(p) = v; }
__device__ __forceinline__ void st4(__nv_bfloat16 *p, const float4 &v) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
    uint2 pk;
    pk.x = *reinterpret_cast<const unsigned int *>(&lo);
    pk.y = *reinterpret_cast<const unsigned int *>(&hi);
    *reinterpret_cast<uint2 *>(p) = pk;
}

__device__ __forceinline__ size_t slot_off(const SegParams &p, int b, int slot, int h) {
    return (((size_t)b * (p.ncs + 1) + slot) * p.H + h) * (size_t)(p.P * p.N);
}
__device__ __forceinline__ size_t vec_off(const SegParams &p, int b, int h, int c) {
    return (((size_t)b * p.H + h) * p.ncs + c) * (size_t)p.Q;
}

// ------------------------------------------------------------------ state passing, boundary store / reload
// Forward: H_{c+1} = exp(cs_last,c) H_c + S_c, strictly sequential in c for every (b,h,p,n) element, so the bits do not depend
// on how the sequence is cut into segments.  Each thread owns one float4.  In the forward call (BWD = false) it also stores the
// segment-entry state into `boundary` (the sequence-axis checkpoint) and hands the segment-exit state on through hcarry.
//
// Backward call (BWD = true): the entry states first, as above, then by the same threads (an element's pass back needs
// no other element's states: one launch instead of two) Gslot[nc] = gradient arriving from the right (or dh_final) and,
// going left, Gslot[c] = exp(cs_last,c) Gslot[c+1] + E_c.  Gslot[c+1] is Gout of chunk c.  Also emits, per chunk, the partial
// sums of exp(cs_last,c) <Gout_c, H_in,c> (one per CTA, summed later in a fixed order): the part of da_t that couples the
// gradient from the right with the state from the left.
//
// Bound by the latency of its loads: the sums and decays do not depend on the carry, so four chunks are fetched ahead of the
// serial recurrence.
template <bool BWD>
__global__ void __launch_bounds__(SP_THREADS, SP_CTAS)
k_state_pass(SegParams p, const float *init, long long init_bs, float *boundary_out, long long bnd_bs, float *final_out, const float *ginit,
             float *gleft) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ float red[SP_PF][SP_THREADS / 32];
    const int h = blockIdx.y, b = blockIdx.z;
    const int PN = p.P * p.N;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int e = blockIdx.x * SP_ELEMS + tid * 4;
    const size_t bh = ((size_t)b * p.H + h) * PN + e;
    float4 carry = make_float4(0.f, 0.f, 0.f, 0.f);
    if (init) carry = *reinterpret_cast<const float4 *>(init + (size_t)b * init_bs + (size_t)h * PN + e);
    if (!BWD && boundary_out)
        *reinterpret_cast<float4 *>(boundary_out + (size_t)b * bnd_bs + (size_t)h * PN + e) = carry;
    const float *csl = p.cs + vec_off(p, b, h, 0) + (p.Q - 1);
    *reinterpret_cast<float4 *>(p.Hst + slot_off(p, b, 0, h) + e) = carry;
    for (int c0 = 1; c0 <= p.nc; c0 += SP_PF) {
        float4 sv[SP_PF];
        float dec[SP_PF];
#pragma unroll
        for (int k = 0; k < SP_PF; ++k)
            if (c0 + k <= p.nc) {
                sv[k] = *reinterpret_cast<const float4 *>(p.Hst + slot_off(p, b, c0 + k, h) + e);
                dec[k] = csl[(size_t)(c0 + k - 1) * p.Q];
            }
#pragma unroll
        for (int k = 0; k < SP_PF; ++k)
            if (c0 + k <= p.nc) {
                const float decay = expf(dec[k]);
                carry.x = fmaf(decay, carry.x, sv[k].x);
                carry.y = fmaf(decay, carry.y, sv[k].y);
                carry.z = fmaf(decay, carry.z, sv[k].z);
                carry.w = fmaf(decay, carry.w, sv[k].w);
                *reinterpret_cast<float4 *>(p.Hst + slot_off(p, b, c0 + k, h) + e) = carry;
            }
    }
    if (!BWD) {
        *reinterpret_cast<float4 *>(p.hcarry + bh) = carry;
        if (final_out) *reinterpret_cast<float4 *>(final_out + bh) = carry;
        return;
    }
    carry = ginit ? *reinterpret_cast<const float4 *>(ginit + bh) : make_float4(0.f, 0.f, 0.f, 0.f);
    *reinterpret_cast<float4 *>(p.Gst + slot_off(p, b, p.nc, h) + e) = carry;
    // the <Gout, H_in> partials of a batch share one block-wide reduction step
    for (int c0 = p.nc - 1; c0 >= 0; c0 -= SP_PF) {
        float4 ev[SP_PF], hv[SP_PF];
        float dec[SP_PF];
#pragma unroll
        for (int k = 0; k < SP_PF; ++k)
            if (c0 - k >= 0) {
                const size_t so = slot_off(p, b, c0 - k, h) + e;
                ev[k] = *reinterpret_cast<const float4 *>(p.Gst + so);
                hv[k] = *reinterpret_cast<const float4 *>(p.Hst + so);
                dec[k] = csl[(size_t)(c0 - k) * p.Q];
            }
#pragma unroll
        for (int k = 0; k < SP_PF; ++k)
            if (c0 - k >= 0) {
                // carry is Gout of chunk c = c0 - k here; hv[k] is the state entering chunk c
                const float decay = expf(dec[k]);
                float part = carry.x * hv[k].x;
                part = fmaf(carry.y, hv[k].y, part);
                part = fmaf(carry.z, hv[k].z, part);
                part = fmaf(carry.w, hv[k].w, part);
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
                if (lane == 0) red[k][warp] = decay * part;
                carry.x = fmaf(decay, carry.x, ev[k].x);
                carry.y = fmaf(decay, carry.y, ev[k].y);
                carry.z = fmaf(decay, carry.z, ev[k].z);
                carry.w = fmaf(decay, carry.w, ev[k].w);
                *reinterpret_cast<float4 *>(p.Gst + slot_off(p, b, c0 - k, h) + e) = carry;
            }
        __syncthreads();
        if (tid < SP_PF && c0 - tid >= 0) {
            float s = 0.f;
#pragma unroll
            for (int w = 0; w < SP_THREADS / 32; ++w) s += red[tid][w];
            p.ghdot[((((size_t)b * p.H + h) * p.ncs + (c0 - tid)) << 4) + blockIdx.x] = s;
        }
        __syncthreads();
    }
    *reinterpret_cast<float4 *>(gleft + bh) = carry;
}

cudaError_t launch_state_pass_fwd(const SegParams &p, const float *init, long long init_bs,
                                  float *boundary_out, long long bnd_bs, float *final_out, cudaStream_t st) {
    dim3 grid(p.P * p.N / SP_ELEMS, p.H, p.B);
    return launch_pdl(k_state_pass<false>, grid, dim3(SP_THREADS), 0, st, p, init, init_bs, boundary_out, bnd_bs, final_out, nullptr, nullptr);
}
cudaError_t launch_state_pass_bwd(const SegParams &p, const float *init, long long init_bs, const float *ginit, float *gleft, cudaStream_t st) {
    dim3 grid(p.P * p.N / SP_ELEMS, p.H, p.B);
    return launch_pdl(k_state_pass<true>, grid, dim3(SP_THREADS), 0, st, p, init, init_bs, nullptr, 0, nullptr, ginit, gleft);
}

// ------------------------------------------------------------------ FFMA contractions
// One shape for all of them: a 64 x 64 output tile per CTA of 256 threads, 4 x 4 outputs per thread, operands staged 64 steps
// of the contraction at a time as [k][64] (rows padded to 68 floats), so that a step of k costs a thread two 16-byte
// shared-memory reads for 16 multiply-adds (packed two to an instruction).  The next stage's global loads are in flight while
// a stage is multiplied.  Bound by the shared-memory reads (65 % of the pipe's wavefronts in the large kernel, the FMA pipe at 44 %).
//
// What does not depend on the head is not done per head: C B^T is made once per group (k_simt_sums writes it, 64 x 64 causal
// tiles), and dB / dC come from a head sum of the masked tiles, one product per CTA instead of two per head.
constexpr int ST_LD = 68;
struct SimtTiles {
    float a[64][ST_LD], b[64][ST_LD];
};

template <typename T> __device__ __forceinline__ float4 ld4f(const T *p);
template <> __device__ __forceinline__ float4 ld4f<float>(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
template <> __device__ __forceinline__ float4 ld4f<__nv_bfloat16>(const __nv_bfloat16 *p) {
    const uint2 v = __ldg(reinterpret_cast<const uint2 *>(p));
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.y));
    return make_float4(a.x, a.y, b.x, b.y);
}

// A 64 x 64 tile of a row-major matrix on its way to shared memory: four float4 per thread.
//   direct:     row = tid / 16 + 16 k, columns (tid % 16) * 4 ..            -> s[row][col]      (rows run along k)
//   transposed: row = tr_row(), columns tr_col(k) ..                        -> s[col][row]      (columns run along k)
// (a warp of the transposed store holds 16 rows of two column groups, 4 x 68 floats = 16 banks apart: no conflicts; eight rows of
// four groups conflicted two ways)
__device__ __forceinline__ int tr_row() { return (threadIdx.x & 15) + 16 * ((threadIdx.x >> 5) & 3); }
__device__ __forceinline__ int tr_col(int k) { return ((threadIdx.x >> 4) & 1) * 4 + (threadIdx.x >> 7) * 8 + 16 * k; }
template <typename T> __device__ __forceinline__ void tile_load(float4 (&r)[4], const T *src, size_t stride, bool transposed) {
    const int tid = threadIdx.x;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (!transposed) r[k] = ld4f(src + (size_t)((tid >> 4) + 16 * k) * stride + (tid & 15) * 4);
        else r[k] = ld4f(src + (size_t)tr_row() * stride + tr_col(k));
    }
}
// The same from scratch that an earlier kernel of the call wrote: coherent loads.
__device__ __forceinline__ void tile_load_ws(float4 (&r)[4], const float *src, size_t stride, bool transposed) {
    const int tid = threadIdx.x;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float *q = !transposed ? src + (size_t)((tid >> 4) + 16 * k) * stride + (tid & 15) * 4
                                     : src + (size_t)tr_row() * stride + tr_col(k);
        r[k] = *reinterpret_cast<const float4 *>(q);
    }
}
__device__ __forceinline__ void tile_store(float (*s)[ST_LD], const float4 (&r)[4], bool transposed) {
    const int tid = threadIdx.x;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (!transposed) {
            *reinterpret_cast<float4 *>(&s[(tid >> 4) + 16 * k][(tid & 15) * 4]) = r[k];
        } else {
            const int row = tr_row(), c = tr_col(k);
            s[c][row] = r[k].x; s[c + 1][row] = r[k].y; s[c + 2][row] = r[k].z; s[c + 3][row] = r[k].w;
        }
    }
}
// acc[i][j] += sum_k a[k][4 ty + i] b[k][4 tx + j]
__device__ __forceinline__ void tile_mma(float2 (&acc)[4][2], const float (*a)[ST_LD], const float (*b)[ST_LD]) {
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll 8
    for (int k = 0; k < 64; ++k) {
        const float4 av = *reinterpret_cast<const float4 *>(&a[k][ty * 4]), bv = *reinterpret_cast<const float4 *>(&b[k][tx * 4]);
        const float am[4] = {av.x, av.y, av.z, av.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 a2 = make_float2(am[i], am[i]);
            acc[i][0] = __ffma2_rn(a2, make_float2(bv.x, bv.y), acc[i][0]);
            acc[i][1] = __ffma2_rn(a2, make_float2(bv.z, bv.w), acc[i][1]);
        }
    }
}
__device__ __forceinline__ void zero_acc(float2 (&acc)[4][2]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
}
// sum over the 16 lanes of a half warp that share ty
__device__ __forceinline__ float sum_tx(float v) {
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}
// causal tile pair number -> (row tile, column tile), column <= row
__device__ __forceinline__ void pair_of(int idx, int &rt, int &ct) {
    rt = 0;
    while (idx > rt) idx -= ++rt;
    ct = idx;
}
// C B^T of (b, chunk, group): [Q][Q] row-major in t
__device__ __forceinline__ float *cb_of(const SegParams &p, int b, int c, int g) {
    return p.cbt + (((size_t)b * p.ncs + c) * p.G + g) * (size_t)(p.Q * p.Q);
}

// What a segment's chunks need before the states can be passed on, by block number:
//   S_c[p,n] = sum_s exp(cs_last - cs_s) dt_s x_s[p] B_s[n]     -> Hst slot c+1   (and cs, dtT)
//   with grads: E_c[p,n] = sum_t exp(cs_t) dy_t[p] C_t[n]       -> Gst slot c      (its CTAs make the cumsum again)
//   the causal tiles of C B^T, where the scratch has room for them
template <typename T, int NS> __host__ __device__ __forceinline__ int simt_n_sums(const SegParams &p, bool grads) {
    const int nrt = p.Q >> 6;
    return p.nc * p.B * ((NS / 64) * p.H * (grads ? 2 : 1) + (p.cbt ? p.G * (nrt * (nrt + 1) / 2) : 0));
}
template <typename T, int NS> __device__ __forceinline__ void simt_sums(const SegParams &p, SimtTiles &sm, float *wsm, int id, bool grads) {
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, Q = p.Q, nrt = Q >> 6, nh = NS / 64;
    const size_t HP = (size_t)p.H * 64, GN = (size_t)p.G * NS;
    const int nsum = p.nc * nh * p.H * p.B;
    float2 acc[4][2];
    float4 ra[4], rb[4];
    zero_acc(acc);
    const bool dst = grads && id >= nsum && id < 2 * nsum;
    if (dst) id -= nsum;
    else if (id >= nsum) {      // a causal tile of C B^T
        id -= grads ? 2 * nsum : nsum;
        const int npair = nrt * (nrt + 1) / 2;
        int rt, ct;
        pair_of(id % npair, rt, ct);
        id /= npair;
        const int g = id % p.G, c = (id / p.G) % p.nc, b = id / (p.G * p.nc);
        const size_t o = (size_t)b * p.bc_bs + ((size_t)p.t0 + (size_t)c * Q) * GN + (size_t)g * NS;
        const T *C = (const T *)p.Cm + o + (size_t)rt * 64 * GN, *Bp = (const T *)p.Bm + o + (size_t)ct * 64 * GN;
        for (int k0 = 0; k0 < NS; k0 += 64) {
            tile_load(ra, C + k0, GN, true);
            tile_load(rb, Bp + k0, GN, true);
            if (k0) __syncthreads();
            tile_store(sm.a, ra, true);
            tile_store(sm.b, rb, true);
            __syncthreads();
            tile_mma(acc, sm.a, sm.b);
        }
        float *out = cb_of(p, b, c, g) + (size_t)(rt * 64 + ty * 4) * Q + ct * 64 + tx * 4;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            *reinterpret_cast<float4 *>(out + (size_t)i * Q) = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
        return;
    }
    const int n0 = (id % nh) * 64;
    id /= nh;
    const int h = id % p.H, c = (id / p.H) % p.nc, b = id / (p.H * p.nc), g = h / p.hpg;
    const size_t tok0 = (size_t)p.t0 + (size_t)c * Q;
    const T *rows = (const T *)(dst ? p.dy : p.x) + (size_t)b * p.x_bs + tok0 * HP + (size_t)h * 64;
    const T *cols = (const T *)(dst ? p.Cm : p.Bm) + (size_t)b * p.bc_bs + tok0 * GN + (size_t)g * NS + n0;
    tile_load(ra, rows, HP, false);
    tile_load(rb, cols, GN, false);
    // the chunk cumsum by one warp: a lane sums its Q/32 consecutive steps in order, then a shuffle scan over the lanes
    if (tid < 32) {
        const int per = Q >> 5;
        const float Ah = __ldg(p.A + h);
        float d[8], v[8], run = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (k < per) d[k] = __ldg(p.dt + (size_t)b * p.dt_bs + (tok0 + tid * per + k) * p.H + h);
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (k < per) {
                run += d[k] * Ah;
                v[k] = run;
            }
        float incl = run;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const float t = __shfl_up_sync(0xffffffffu, incl, off);
            if (tid >= off) incl += t;
        }
        float excl = __shfl_up_sync(0xffffffffu, incl, 1);
        if (tid == 0) excl = 0.f;
        const float last = __shfl_sync(0xffffffffu, run + excl, 31);
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (k < per) {
                const int t = tid * per + k;
                const float cs = v[k] + excl;
                wsm[t] = dst ? expf(cs) : expf(fminf(last - cs, 0.f)) * d[k];
                if (n0 == 0 && !dst) {
                    p.cs[vec_off(p, b, h, c) + t] = cs;
                    p.dtT[vec_off(p, b, h, c) + t] = d[k];
                }
            }
    }
    __syncthreads();
    for (int s0 = 0; s0 < Q; s0 += 64) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float w = wsm[s0 + ty + 16 * k];
            ra[k].x *= w; ra[k].y *= w; ra[k].z *= w; ra[k].w *= w;
        }
        tile_store(sm.a, ra, false);
        tile_store(sm.b, rb, false);
        __syncthreads();
        if (s0 + 64 < Q) {
            tile_load(ra, rows + (size_t)(s0 + 64) * HP, HP, false);
            tile_load(rb, cols + (size_t)(s0 + 64) * GN, GN, false);
        }
        tile_mma(acc, sm.a, sm.b);
        __syncthreads();
    }
    float *out = (dst ? p.Gst + slot_off(p, b, c, h) : p.Hst + slot_off(p, b, c + 1, h)) + (size_t)(ty * 4) * NS + n0 + tx * 4;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float4 *>(out + (size_t)i * NS) = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
}

template <typename T, int NS> __global__ void __launch_bounds__(256, 3) k_simt_sums(SegParams p, bool grads) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ SimtTiles sm;
    __shared__ float wsm[256];
    simt_sums<T, NS>(p, sm, wsm, blockIdx.x, grads);
}

// One 64-row tile of y (DX = false) or of dx (DX = true) of one head:
//   y_t  = sum_{s<=t} CB[t,s] e^{cs_t-cs_s} dt_s x_s + e^{cs_t} C_t H_in + D x_t
//   u_s  = sum_{t>=s} CB[t,s] e^{cs_t-cs_s} dy_t     + e^{cs_last-cs_s} B_s Gout ;  dx_s = D dy_s + dt_s u_s ,
//   ddt_direct_s = x_s . u_s , psi2_s = dt_s e^{cs_last-cs_s} x_s . (Gout B_s) , dD partial = sum dy.x
// CB false (y only): the tiles of C B^T are not in the scratch and are made here, per head, with the same operations in the same
// order, so with the same bits.
template <typename T, int NS, bool DX, bool CB>
__device__ __forceinline__ void simt_row_tile(const SegParams &p, SimtTiles &sm, float *css, float *dts, float *fac, float *red, int c, int rt, int h, int b) {
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, Q = p.Q, nrt = Q >> 6, g = h / p.hpg, r0 = rt * 64;
    const size_t tok0 = (size_t)p.t0 + (size_t)c * Q, HP = (size_t)p.H * 64, GN = (size_t)p.G * NS;
    const size_t xo = (size_t)b * p.x_bs + tok0 * HP + (size_t)h * 64;
    const T *vals = (const T *)(DX ? p.dy : p.x) + xo;
    const T *rowv = (const T *)(DX ? p.Bm : p.Cm) + (size_t)b * p.bc_bs + (tok0 + r0) * GN + (size_t)g * NS;
    const float *St = DX ? p.Gst + slot_off(p, b, c + 1, h) : p.Hst + slot_off(p, b, c, h), *cbt = cb_of(p, b, c, g);
    float4 ra[4], rb[4];
    float2 acc[4][2];
    zero_acc(acc);
    tile_load(ra, rowv, GN, true);
    tile_load_ws(rb, St, NS, true);
    for (int t = tid; t < Q; t += 256) {
        css[t] = p.cs[vec_off(p, b, h, c) + t];
        dts[t] = p.dtT[vec_off(p, b, h, c) + t];
    }
    auto load_vals = [&](int ct) {      // CB tile and value rows of column tile ct
        // DX = false: rows t = r0 .., columns s = 64 ct .. ; DX = true: the tile's rows are the CB matrix's columns
        if (!DX && CB) tile_load_ws(ra, cbt + (size_t)r0 * Q + ct * 64, Q, true);
        else if (DX) tile_load_ws(ra, cbt + (size_t)ct * 64 * Q + r0, Q, false);
        tile_load(rb, vals + (size_t)ct * 64 * HP, HP, false);
    };
    const int ct0 = DX ? rt : 0, ct1 = DX ? nrt : rt + 1;
    for (int k0 = 0; k0 < NS; k0 += 64) {
        tile_store(sm.a, ra, true);
        tile_store(sm.b, rb, true);
        __syncthreads();
        if (k0 + 64 < NS) {
            tile_load(ra, rowv + k0 + 64, GN, true);
            tile_load_ws(rb, St + k0 + 64, NS, true);
        } else if (CB) {
            load_vals(ct0);
        }
        tile_mma(acc, sm.a, sm.b);
        __syncthreads();
    }
    // Off the diagonal tile the mask factors at the tile's edge m (its first row; dx: last), where both factors are <= 1:
    // e^{cs_t-cs_s} = e^{cs_t-cs_m} e^{cs_m-cs_s}.  An exponential per step instead of one per element.
    const int m = DX ? r0 + 63 : r0;
    if (nrt > 1) {
        for (int t = tid; t < Q; t += 256) {
            const float d = css[t] - css[m];
            fac[t] = expf(fminf(t >= m ? d : -d, 0.f)) * (DX || t >= m ? 1.f : dts[t]);
        }
        __syncthreads();
    }
    // the inter-chunk term is complete: scale its rows
    const float cl = css[Q - 1];
    float dd2[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = r0 + ty * 4 + i;
        const float o = DX ? expf(fminf(cl - css[r], 0.f)) : expf(css[r]);
        acc[i][0].x *= o; acc[i][0].y *= o; acc[i][1].x *= o; acc[i][1].y *= o;
        if (DX) {
            const float4 xv = ld4f((const T *)p.x + xo + (size_t)r * HP + tx * 4);
            dd2[i] = xv.x * acc[i][0].x + xv.y * acc[i][0].y + xv.z * acc[i][1].x + xv.w * acc[i][1].y;
        }
    }
    for (int ct = ct0; ct < ct1; ++ct) {
        // masked tile: a[k = column of the mask][row]
        if constexpr (!CB) {
            const T *colv = (const T *)p.Bm + (size_t)b * p.bc_bs + (tok0 + ct * 64) * GN + (size_t)g * NS;
            float2 cb[4][2];
            zero_acc(cb);
            for (int k0 = 0; k0 < NS; k0 += 64) {
                tile_load(ra, rowv + k0, GN, true);
                tile_load(rb, colv + k0, GN, true);
                tile_store(sm.a, ra, true);
                tile_store(sm.b, rb, true);
                __syncthreads();
                tile_mma(cb, sm.a, sm.b);
                __syncthreads();
            }
            load_vals(ct);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int s = ct * 64 + tx * 4 + j;
                float e[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int t = r0 + ty * 4 + i;
                    const float v = j < 2 ? (j ? cb[i][0].y : cb[i][0].x) : (j == 3 ? cb[i][1].y : cb[i][1].x);
                    e[i] = ct != rt ? v * (fac[t] * fac[s]) : s <= t ? v * expf(fminf(css[t] - css[s], 0.f)) * dts[s] : 0.f;
                }
                *reinterpret_cast<float4 *>(&sm.a[tx * 4 + j][ty * 4]) = make_float4(e[0], e[1], e[2], e[3]);
            }
        } else if (ct != rt) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float one = fac[DX ? ct * 64 + ty + 16 * k : r0 + tr_row()];
                const float4 four = *reinterpret_cast<const float4 *>(fac + (DX ? r0 + tx * 4 : ct * 64 + tr_col(k)));
                ra[k].x *= one * four.x; ra[k].y *= one * four.y; ra[k].z *= one * four.z; ra[k].w *= one * four.w;
            }
        } else
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float *e = reinterpret_cast<float *>(&ra[k]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                // as tile_load laid them out: not DX (transposed) row t, column s; DX (direct) row t, column s
                const int t = DX ? ct * 64 + ty + 16 * k : r0 + tr_row();
                const int s = DX ? r0 + tx * 4 + i : ct * 64 + tr_col(k) + i;
                e[i] = s <= t ? e[i] * expf(fminf(css[t] - css[s], 0.f)) * (DX ? 1.f : dts[s]) : 0.f;
            }
        }
        if (CB) tile_store(sm.a, ra, !DX);
        tile_store(sm.b, rb, false);
        __syncthreads();
        if (CB && ct + 1 < ct1) load_vals(ct + 1);
        tile_mma(acc, sm.a, sm.b);
        __syncthreads();
    }
    const float Dh = __ldg(p.D + h) + (DX ? p.dx_skip : 0.f);      // dx: D dy, plus dy itself under a skip connection
    float dsum = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = r0 + ty * 4 + i;
        const size_t o = xo + (size_t)r * HP + tx * 4;
        const float4 v = ld4f((const T *)(DX ? p.dy : p.x) + o);
        const float s = DX ? dts[r] : 1.f;
        st4((T *)(DX ? p.dx : p.y) + o, make_float4(fmaf(Dh, v.x, s * acc[i][0].x), fmaf(Dh, v.y, s * acc[i][0].y), fmaf(Dh, v.z, s * acc[i][1].x),
                                                    fmaf(Dh, v.w, s * acc[i][1].y)));
        if (DX) {
            const float4 xv = ld4f((const T *)p.x + o);
            const float dd = sum_tx(xv.x * acc[i][0].x + xv.y * acc[i][0].y + xv.z * acc[i][1].x + xv.w * acc[i][1].y);
            const float d2 = sum_tx(dd2[i]);
            dsum += v.x * xv.x + v.y * xv.y + v.z * xv.z + v.w * xv.w;
            if (tx == 0) {
                p.ddt_dir[vec_off(p, b, h, c) + r] = dd;
                p.psi2[vec_off(p, b, h, c) + r] = dts[r] * d2;
            }
        }
    }
    if (DX) {       // deterministic block sum of dy*x
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) dsum += __shfl_xor_sync(0xffffffffu, dsum, off);
        if ((tid & 31) == 0) red[tid >> 5] = dsum;
        __syncthreads();
        if (tid == 0) {
            float s = 0.f;
#pragma unroll
            for (int w = 0; w < 8; ++w) s += red[w];
            p.dDp[((((size_t)b * p.H + h) * p.nct + p.c0 + c) << 2) + rt] = s;
        }
    }
}

// y of a segment and, in the same launch where the scratch has a second copy, the sums of the next segment (n_next CTAs): they
// wait for nothing of this one, and a launch of a few microseconds is saved per segment.  Two CTAs per SM: held to the 80
// registers of three, N = 128 spills (36 bytes stored, 120 loaded) and the forward takes 276 us instead of 233 (8192 steps of 4
// heads, chunks of 128; 24 heads 396 and 383, chunks of 256 445 and 434), while N = 64 gains 5 % with chunks of 64 and loses 2 %
// with longer ones.
template <typename T, int NS, bool CB>
__global__ void __launch_bounds__(256, 2) k_simt_y(SegParams p, SegParams nx, int n_next) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ SimtTiles sm;
    __shared__ __align__(16) float css[256], dts[256], fac[256];
    const int nrt = p.Q >> 6, ny = (int)gridDim.x - n_next;
    int id = blockIdx.x;
    if (id >= ny) {
        simt_sums<T, NS>(nx, sm, css, id - ny, false);
        return;
    }
    const int rt = id % nrt, c = (id / nrt) % p.nc, h = (id / (nrt * p.nc)) % p.H, b = id / (nrt * p.nc * p.H);
    simt_row_tile<T, NS, false, CB>(p, sm, css, dts, fac, nullptr, c, rt, h, b);
}

// The large kernel of the backward: tiles of dx, and the partial slices of dB and dC.  Per (chunk, head range):
//   causal tile pair (tt, ts): W_h = (dy_tt x_ts^T) o mask per head, rho / psi partial sums of W_h o CB, head sum of W_h; then
//                  slices dC[tt] = Wsum B_ts and dB[ts] = Wsum^T C_tt
//   inter dC, tile tt : sum_h e^{cs_t} dy_t H_in (and rho2 per head);  inter dB, tile ts : sum_h dt_s e^{cs_last-cs_s} x_s Gout
// A row of tile r has dC slots for ts <= r and dB slots for tt >= r, so the two share Q/64 + 3 slots per head range: dC by ts, dB by
// tt + 1, then the inter-chunk terms of both.
template <typename T, int NS>
__global__ void __launch_bounds__(256, 2) k_simt_bwd(SegParams p, int n_dx) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ SimtTiles sm;
    __shared__ __align__(16) float css[256], dts[256], fac[256], red[8][64];
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, Q = p.Q, nrt = Q >> 6, npair = nrt * (nrt + 1) / 2;
    int id = blockIdx.x;
    if (id >= (int)gridDim.x - n_dx) {
        id -= (int)gridDim.x - n_dx;
        const int rt = id % nrt, h = (id / nrt) % p.H, c = (id / (nrt * p.H)) % p.nc, b = id / (nrt * p.H * p.nc);
        simt_row_tile<T, NS, true, true>(p, sm, css, dts, fac, red[0], c, rt, h, b);
        return;
    }
    const int per = npair + 2 * nrt, role = id % per;
    id /= per;
    const int rng = p.nsl / (nrt + 3);                         // head ranges per group
    const int sl = id % rng, g = (id / rng) % p.G, c = (id / (rng * p.G)) % p.nc, b = id / (rng * p.G * p.nc);
    const int hps = (p.hpg + rng - 1) / rng, h0 = g * p.hpg + sl * hps, h1 = min(h0 + hps, (g + 1) * p.hpg);
    const size_t tok0 = (size_t)p.t0 + (size_t)c * Q, HP = (size_t)p.H * 64, GN = (size_t)p.G * NS;
    const T *xb = (const T *)p.x + (size_t)b * p.x_bs + tok0 * HP, *dyb = (const T *)p.dy + (size_t)b * p.x_bs + tok0 * HP;
    const T *Bb = (const T *)p.Bm + (size_t)b * p.bc_bs + tok0 * GN + (size_t)g * NS, *Cb = (const T *)p.Cm + (size_t)b * p.bc_bs + tok0 * GN + (size_t)g * NS;
    auto load_vec = [&](int h) {
        for (int t = tid; t < Q; t += 256) {
            css[t] = p.cs[vec_off(p, b, h, c) + t];
            dts[t] = p.dtT[vec_off(p, b, h, c) + t];
        }
    };
    auto write_slice = [&](const float2 (&acc)[4][2], int row0, int slot, int n0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const size_t tl = (size_t)b * p.ncs * Q + (size_t)c * Q + row0 + ty * 4 + i;
            *reinterpret_cast<float4 *>(p.pC + ((tl * p.G + g) * p.nsl + sl * (nrt + 3) + slot) * NS + n0 + tx * 4) =
                make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
        }
    };
    float4 ra[4], rb[4];
    float2 acc[4][2];
    if (role < npair) {
        int tt, ts;
        pair_of(role, tt, ts);
        const float *CB = cb_of(p, b, c, g) + (size_t)(tt * 64 + ty * 4) * Q + ts * 64 + tx * 4;
        float4 cb[4];
        float ws[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            cb[i] = *reinterpret_cast<const float4 *>(CB + (size_t)i * Q);
#pragma unroll
            for (int j = 0; j < 4; ++j) ws[i][j] = 0.f;
        }
        tile_load(ra, dyb + (size_t)tt * 64 * HP + (size_t)h0 * 64, HP, true);
        tile_load(rb, xb + (size_t)ts * 64 * HP + (size_t)h0 * 64, HP, true);
        for (int h = h0; h < h1; ++h) {
            load_vec(h);
            if (tt != ts && tid < 128) {      // the mask's factors at the row tile's first step, as for y
                const float *cs = p.cs + vec_off(p, b, h, c), ref = cs[tt * 64];
                const int t = (tid < 64 ? tt : ts - 1) * 64 + tid;
                fac[tid] = tid < 64 ? expf(fminf(cs[t] - ref, 0.f)) : expf(fminf(ref - cs[t], 0.f)) * p.dtT[vec_off(p, b, h, c) + t];
            }
            tile_store(sm.a, ra, true);
            tile_store(sm.b, rb, true);
            __syncthreads();
            if (h + 1 < h1) {
                tile_load(ra, dyb + (size_t)tt * 64 * HP + (size_t)(h + 1) * 64, HP, true);
                tile_load(rb, xb + (size_t)ts * 64 * HP + (size_t)(h + 1) * 64, HP, true);
            }
            zero_acc(acc);
            tile_mma(acc, sm.a, sm.b);
            float col[4] = {0.f, 0.f, 0.f, 0.f};
            const size_t vo = (vec_off(p, b, h, c) * nrt);      // rho, psi: [B,H,ncs,Q/64 tiles,Q]
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int t = tt * 64 + ty * 4 + i;
                const float s4[4] = {acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y}, c4[4] = {cb[i].x, cb[i].y, cb[i].z, cb[i].w};
                float row = 0.f, e4[4];
                if (tt != ts) {
                    const float one = fac[ty * 4 + i];
                    const float4 four = *reinterpret_cast<const float4 *>(fac + 64 + tx * 4);
                    e4[0] = one * four.x; e4[1] = one * four.y; e4[2] = one * four.z; e4[3] = one * four.w;
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int s = ts * 64 + tx * 4 + j;
                        e4[j] = s <= t ? expf(fminf(css[t] - css[s], 0.f)) * dts[s] : 0.f;
                    }
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float w = s4[j] * e4[j];
                    ws[i][j] += w;
                    // s = t adds the same to rho_t and psi_t, of which only sums of differences are used: left out of both, or with
                    // strong decays, where it is the largest term, its rounding would be most of the error of dA
                    const float wc = i == j && tx == ty && tt == ts ? 0.f : w;
                    row = fmaf(wc, c4[j], row);
                    col[j] = fmaf(wc, c4[j], col[j]);
                }
                row = sum_tx(row);
                if (tx == 0) p.rho[vo + (size_t)ts * Q + t] = row;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                col[j] += __shfl_xor_sync(0xffffffffu, col[j], 16);
                if ((tid & 16) == 0) red[tid >> 5][tx * 4 + j] = col[j];
            }
            __syncthreads();
            if (tid < 64) {
                float s = 0.f;
#pragma unroll
                for (int w = 0; w < 8; ++w) s += red[w][tid];
                p.psi[vo + (size_t)tt * Q + ts * 64 + tid] = s;
            }
            // red, css, dts and fac are rewritten only after the next head's first barrier or by the threads that read them here
            __syncthreads();
        }
        // dC[tt] = Wsum B_ts: a[k = s][t]
#pragma unroll
        for (int j = 0; j < 4; ++j)
            *reinterpret_cast<float4 *>(&sm.a[tx * 4 + j][ty * 4]) = make_float4(ws[0][j], ws[1][j], ws[2][j], ws[3][j]);
        for (int n0 = 0; n0 < NS; n0 += 64) {
            tile_load(rb, Bb + (size_t)ts * 64 * GN + n0, GN, false);
            tile_store(sm.b, rb, false);
            __syncthreads();
            zero_acc(acc);
            tile_mma(acc, sm.a, sm.b);
            write_slice(acc, tt * 64, ts, n0);
            __syncthreads();
        }
        // dB[ts] = Wsum^T C_tt: a[k = t][s]
#pragma unroll
        for (int i = 0; i < 4; ++i)
            *reinterpret_cast<float4 *>(&sm.a[ty * 4 + i][tx * 4]) = make_float4(ws[i][0], ws[i][1], ws[i][2], ws[i][3]);
        for (int n0 = 0; n0 < NS; n0 += 64) {
            tile_load(rb, Cb + (size_t)tt * 64 * GN + n0, GN, false);
            tile_store(sm.b, rb, false);
            __syncthreads();
            zero_acc(acc);
            tile_mma(acc, sm.a, sm.b);
            write_slice(acc, ts * 64, tt + 1, n0);
            __syncthreads();
        }
        return;
    }
    // inter-chunk terms of one row tile: the head's rows scaled per row, times the chunk state (rows p)
    const bool isC = role - npair < nrt;
    const int rt = (role - npair) % nrt;
    float2 tot[NS / 64][4][2];
#pragma unroll
    for (int m = 0; m < NS / 64; ++m) zero_acc(tot[m]);
    for (int h = h0; h < h1; ++h) {
        const float *St = isC ? p.Hst + slot_off(p, b, c, h) : p.Gst + slot_off(p, b, c + 1, h);
        load_vec(h);
        tile_load(ra, (isC ? dyb : xb) + (size_t)rt * 64 * HP + (size_t)h * 64, HP, true);
        tile_load_ws(rb, St, NS, false);
        tile_store(sm.a, ra, true);
        float rho2[4] = {0.f, 0.f, 0.f, 0.f}, sc[4];
#pragma unroll
        for (int m = 0; m < NS / 64; ++m) {
            tile_store(sm.b, rb, false);
            __syncthreads();
            if (m == 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = rt * 64 + ty * 4 + i;
                    sc[i] = isC ? expf(css[r]) : dts[r] * expf(fminf(css[Q - 1] - css[r], 0.f));
                }
            }
            if (m + 1 < NS / 64) tile_load_ws(rb, St + 64 * (m + 1), NS, false);
            zero_acc(acc);
            tile_mma(acc, sm.a, sm.b);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 s2 = make_float2(sc[i], sc[i]);
                const float2 a0 = __fmul2_rn(acc[i][0], s2), a1 = __fmul2_rn(acc[i][1], s2);
                tot[m][i][0] = __fadd2_rn(tot[m][i][0], a0);
                tot[m][i][1] = __fadd2_rn(tot[m][i][1], a1);
                if (isC) {
                    const float4 cv = ld4f(Cb + (size_t)(rt * 64 + ty * 4 + i) * GN + m * 64 + tx * 4);
                    rho2[i] += cv.x * a0.x + cv.y * a0.y + cv.z * a1.x + cv.w * a1.y;
                }
            }
            __syncthreads();
        }
        if (isC) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float v = sum_tx(rho2[i]);
                if (tx == 0) p.rho2[vec_off(p, b, h, c) + rt * 64 + ty * 4 + i] = v;
            }
        }
    }
#pragma unroll
    for (int m = 0; m < NS / 64; ++m) write_slice(tot[m], rt * 64, isC ? nrt + 1 : nrt + 2, m * 64);
}

// ------------------------------------------------------------------ da, ddt, dA partial
// One warp per (b, h, chunk).  With g_t = dLoss/dh_t and h_{t-1} split into their intra-chunk and
// inter-chunk parts, da_t = exp(a_t) <g_t, h_{t-1}> is the sum of four terms, none of which
// subtracts large numbers when the decay inside a chunk is strong:
//   sum_{t'>=t} (rho_intra_t' - psi_t')     pairs (t' >= t > s) inside the chunk
// + sum_{t'>=t} rho_inter_t'                outputs at/after t reading the chunk-entry state (rho2)
// + sum_{s<t}   psi2_s                      inputs before t feeding the chunk-exit gradient
// + exp(cs_last) <Gout, H_in>
// Suffix/prefix scans: serial inside a lane, warp shuffles across lanes.  Then ddt = ddt_direct + A da, dA partial =
// sum_t dt_t da_t.  TC: blocks of 128 steps, four steps per lane, 37 registers instead of the general form's 64 (4096 steps of
// 80 heads: 12.2 -> 10.7 us, 8192 of 8 groups 39 -> 29 us with the sums of dB and dC).
// One CTA per (chunk, eight consecutive heads), one warp per head.  ddt is [B, L, H]: a head's values of consecutive
// steps lie H floats apart, so the eight heads' results go through a shared-memory tile and leave as rows of eight
// consecutive floats (whole 32-byte sectors) instead of one 4-byte store per sector.
constexpr int FIN_HB = 8;
constexpr int FIN_TILE = 256 * (FIN_HB + 1);
constexpr float kLeastStep = 1e-18f;      // far above the dt at which a product with it would lose bits
template <bool TC> __device__ __forceinline__ void bwd_finish(const SegParams &p, float *tile, int id) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nhb = (p.H + FIN_HB - 1) / FIN_HB;
    const int c = id % p.nc, hb = (id / p.nc) % nhb, b = id / (p.nc * nhb), h = hb * FIN_HB + warp, nh = min(FIN_HB, p.H - hb * FIN_HB);
    constexpr int PER = TC ? kTcBlock / 32 : 8;      // steps per lane, at most
    const int Q = TC ? kTcBlock : p.Q, per = Q >> 5;
    if (warp < nh) {
        const size_t hc = ((size_t)b * p.H + h) * p.ncs + c, vo = hc * Q + (size_t)lane * per;
        float gh = 0.f;
        for (int i = 0; i < p.ngh; ++i) gh += p.ghdot[(hc << 4) + i];
        float dtv[PER], dd[PER], sfx[PER], pfx[PER];
        float run = 0.f;
#pragma unroll
        for (int j = PER - 1; j >= 0; --j)
            if (j < per) {
                dtv[j] = p.dtT[hc * p.dt_stride + lane * per + j];
                float r1, p1;
                if (TC) {
                    r1 = p.rho[vo + j];
                    p1 = p.psi[vo + j];
                    // x_s . u_s as B_s . dB_s / dt_s: the part inside the block is then a column sum of an fp32 tile, where dx's u has it
                    // from a masked tile rounded to bf16.  dx's own, where the step size is (almost) zero.
                    dd[j] = dtv[j] >= kLeastStep ? __fdividef(p1 + p.psi2[vo + j], dtv[j]) : p.ddt_dir[vo + j];
                } else {            // partial sums per 64 x 64 tile of the masked products
                    dd[j] = p.ddt_dir[vo + j];
                    const size_t to = hc * p.tiles * Q + lane * per + j;
                    const int t0 = (lane * per + j) >> 6;
                    r1 = p.rho[to];
                    for (int t = 1; t <= t0; ++t) r1 += p.rho[to + (size_t)t * Q];
                    p1 = p.psi[to + (size_t)t0 * Q];
                    for (int t = t0 + 1; t < p.tiles; ++t) p1 += p.psi[to + (size_t)t * Q];
                }
                run += (r1 - p1) + p.rho2[vo + j];
                sfx[j] = run;
            }
        float incl = run;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const float t = __shfl_down_sync(0xffffffffu, incl, off);
            if (lane + off < 32) incl += t;
        }
        float excl = __shfl_down_sync(0xffffffffu, incl, 1);
        if (lane == 31) excl = 0.f;
        // exclusive prefix of psi2
        float prun = 0.f;
#pragma unroll
        for (int j = 0; j < PER; ++j)
            if (j < per) {
                pfx[j] = prun;
                prun += p.psi2[vo + j];
            }
        float pincl = prun;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const float t = __shfl_up_sync(0xffffffffu, pincl, off);
            if (lane >= off) pincl += t;
        }
        float pexcl = __shfl_up_sync(0xffffffffu, pincl, 1);
        if (lane == 0) pexcl = 0.f;
        const float Ah = __ldg(p.A + h);
        float sA = 0.f;
#pragma unroll
        for (int j = 0; j < PER; ++j)
            if (j < per) {
                const float da = ((sfx[j] + excl) + (pfx[j] + pexcl)) + gh;
                tile[(lane * per + j) * (FIN_HB + 1) + warp] = fmaf(Ah, da, dd[j]);
                sA = fmaf(dtv[j], da, sA);
            }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) sA += __shfl_xor_sync(0xffffffffu, sA, off);
        if (lane == 0) p.dAp[((size_t)b * p.H + h) * p.nct + p.c0 + c] = sA;
    }
    __syncthreads();
    float *out = p.ddt + (size_t)b * p.dt_bs + ((size_t)p.t0 + (size_t)c * Q) * p.H + (size_t)hb * FIN_HB;
    for (int i = threadIdx.x; i < Q * FIN_HB; i += 256) {
        const int t = i / FIN_HB, hh = i % FIN_HB;
        if (hh < nh) out[(size_t)t * p.H + hh] = tile[t * (FIN_HB + 1) + hh];
    }
}

// ------------------------------------------------------------------ dB / dC: sum the head slices of a group
// Four consecutive n per thread (16-byte loads of the fp32 partial slices, one 8- or 16-byte store): the kernel only
// moves bytes.  The order of the additions per element is fixed: slices in order.
template <typename T, bool TC>
__device__ __forceinline__ void reduce_dbdc(const SegParams &p, int id) {
    const int N4 = p.N >> 2;
    const size_t total = (size_t)p.B * p.nc * p.Q * p.G * N4;
    const size_t i = (size_t)id * 256 + threadIdx.x;
    if (i >= total) return;
    const int n = (int)(i % N4) * 4;
    size_t r = i / N4;
    const int g = (int)(r % p.G);
    r /= p.G;
    const size_t seglen = (size_t)p.nc * p.Q;
    const size_t tl = r % seglen;
    const int b = (int)(r / seglen);
    const size_t segcap = (size_t)p.ncs * p.Q;
    float4 sB = make_float4(0.f, 0.f, 0.f, 0.f), sC = sB;
    auto ld = [](const float *q) { return *reinterpret_cast<const float4 *>(q); };
    const size_t src = ((((size_t)b * segcap + tl) * p.G + g) * p.nsl) * p.N + n;
    if (!TC) {
        // CUDA-core path: per head range, of a row of tile rt, dC slots 0 .. rt, dB slots rt + 1 .. tiles, then the inter-chunk terms
        const int rt = (int)(tl % (size_t)p.Q) >> 6;
        for (int s0 = 0; s0 < p.nsl; s0 += p.tiles + 3) {
            float4 v[5];                                // all of a range's loads in flight
#pragma unroll
            for (int t = 0; t < 5; ++t)
                if (t <= p.tiles) v[t] = ld(p.pC + src + (size_t)(s0 + t) * p.N);
            const float4 interC = ld(p.pC + src + (size_t)(s0 + p.tiles + 1) * p.N), interB = ld(p.pC + src + (size_t)(s0 + p.tiles + 2) * p.N);
#pragma unroll
            for (int t = 0; t < 5; ++t) {
                if (t <= rt) add4(sC, v[t]);
                else if (t <= p.tiles) add4(sB, v[t]);
            }
            add4(sC, interC);
            add4(sB, interB);
        }
    } else {
        for (int s = 0; s < p.nsl; ++s) {
            add4(sB, ld(p.pB + src + (size_t)s * p.N));
            add4(sC, ld(p.pC + src + (size_t)s * p.N));
        }
    }
    const size_t dst = (size_t)b * p.bc_bs + ((size_t)p.t0 + tl) * p.G * p.N + (size_t)g * p.N + n;
    st4((T *)p.dB + dst, sB);
    st4((T *)p.dC + dst, sC);
}

// Both in one launch: the two short finishing steps of a segment.
template <typename T, bool TC>
__global__ void __launch_bounds__(256) k_bwd_tail(SegParams p, int nfin) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ float tile[FIN_TILE];
    if ((int)blockIdx.x < nfin) bwd_finish<TC>(p, tile, blockIdx.x);
    else reduce_dbdc<T, TC>(p, blockIdx.x - nfin);
}
// CUDA-core path: the same with the sums of the next segment (to the left) in front, which share no scratch with it but the step
// sizes, of which there are two copies.
template <typename T, int NS>
__global__ void __launch_bounds__(256, 3) k_simt_tail(SegParams p, SegParams nx, int n_next, int nfin) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ SimtTiles sm;
    __shared__ float wsm[256];
    static_assert(sizeof(SimtTiles) >= FIN_TILE * sizeof(float), "the finishing step's tile");
    const int id = (int)blockIdx.x - n_next;
    if (id < 0) simt_sums<T, NS>(nx, sm, wsm, blockIdx.x, true);
    else if (id < nfin) bwd_finish<false>(p, &sm.a[0][0], id);
    else reduce_dbdc<T, false>(p, id - nfin);
}

static int tail_finish_ctas(const SegParams &p) { return p.nc * ((p.H + FIN_HB - 1) / FIN_HB) * p.B; }
static int tail_reduce_ctas(const SegParams &p) { return (int)(((size_t)p.B * p.nc * p.Q * p.G * (p.N / 4) + 255) / 256); }
cudaError_t launch_bwd_tail(const SegParams &p, int dtype, cudaStream_t st) {
    const int nfin = tail_finish_ctas(p);
    const dim3 grid(nfin + tail_reduce_ctas(p));
    if (dtype == SSD_DTYPE_F32) return launch_pdl(k_bwd_tail<float, false>, grid, dim3(256), 0, st, p, nfin);
    if (p.tiles) return launch_pdl(k_bwd_tail<__nv_bfloat16, false>, grid, dim3(256), 0, st, p, nfin);
    return launch_pdl(k_bwd_tail<__nv_bfloat16, true>, grid, dim3(256), 0, st, p, nfin);
}

template <typename T, int NS>
static cudaError_t simt_launch(const SegParams &p, const SegParams *next, int what, cudaStream_t st) {
    const int nrt = p.Q / 64, npair = nrt * (nrt + 1) / 2;
    switch (what) {
        case SIMT_SUMS:
        case SIMT_SUMS_GRAD: {
            const bool grads = what == SIMT_SUMS_GRAD;
            return launch_pdl(k_simt_sums<T, NS>, dim3(simt_n_sums<T, NS>(p, grads)), dim3(256), 0, st, p, grads);
        }
        case SIMT_Y: {
            const int n_next = next ? simt_n_sums<T, NS>(*next, false) : 0;
            const dim3 grid(p.nc * nrt * p.H * p.B + n_next);
            if (!p.cbt) return launch_pdl(k_simt_y<T, NS, false>, grid, dim3(256), 0, st, p, p, 0);      // never with `next`
            return launch_pdl(k_simt_y<T, NS, true>, grid, dim3(256), 0, st, p, next ? *next : p, n_next);
        }
        case SIMT_TAIL: {
            const int nfin = tail_finish_ctas(p), n_next = simt_n_sums<T, NS>(*next, true);
            return launch_pdl(k_simt_tail<T, NS>, dim3(n_next + nfin + tail_reduce_ctas(p)), dim3(256), 0, st, p, *next, n_next, nfin);
        }
        default: {
            const int n_dx = p.nc * nrt * p.H * p.B, n_bc = p.nc * (npair + 2 * nrt) * (p.nsl / (nrt + 3)) * p.G * p.B;
            return launch_pdl(k_simt_bwd<T, NS>, dim3(n_bc + n_dx), dim3(256), 0, st, p, n_dx);
        }
    }
}
cudaError_t launch_simt(const SegParams &p, const SegParams *next, int dtype, int what, cudaStream_t st) {
    if (dtype == SSD_DTYPE_F32) return p.N == 64 ? simt_launch<float, 64>(p, next, what, st) : simt_launch<float, 128>(p, next, what, st);
    return p.N == 64 ? simt_launch<__nv_bfloat16, 64>(p, next, what, st) : simt_launch<__nv_bfloat16, 128>(p, next, what, st);
}

// ------------------------------------------------------------------ dA, dD over (batch, chunks)
// One CTA per head; threads stride over the per-chunk partials in fp64, then a fixed tree.
__global__ void __launch_bounds__(256) k_final_dAdD(SegParams p, float *dA, float *dD, int accumulate) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ double red[2][8];
    const int h = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double sA = 0.0, sD = 0.0;
    for (int b = 0; b < p.B; ++b) {
        const size_t base = ((size_t)b * p.H + h) * p.nct;
        for (int c = threadIdx.x; c < p.nct; c += 256) {
            sA += (double)p.dAp[base + c];
            const float4 d4 = *reinterpret_cast<const float4 *>(p.dDp + ((base + c) << 2));
            const float d[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (r < p.ndd) sD += (double)d[r];
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        sA += __shfl_xor_sync(0xffffffffu, sA, off);
        sD += __shfl_xor_sync(0xffffffffu, sD, off);
    }
    if (lane == 0) {
        red[0][warp] = sA;
        red[1][warp] = sD;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, d = 0.0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            a += red[0][w];
            d += red[1][w];
        }
        dA[h] = accumulate ? dA[h] + (float)a : (float)a;
        dD[h] = accumulate ? dD[h] + (float)d : (float)d;
    }
}

cudaError_t launch_final_dAdD(const SegParams &p, float *dA, float *dD, bool accumulate, cudaStream_t st) {
    return launch_pdl(k_final_dAdD, dim3(p.H), dim3(256), 0, st, p, dA, dD, accumulate ? 1 : 0);
}

}  // namespace ssd
