// Every role of the split path's large kernels loads its first tiles of the caller's tensors before it waits for the launch before it:
// they are older than the call (its first launch is an ordinary one).
//
// The split path: the kernels of fp32 calls (1e-4 parity rules out operands rounded to 16 bits or TF32), of bf16 calls whose
// intermediates stay in fp32, and a cross-check of the tensor-core kernels.  fp32 operands go to the tensor cores as three bf16
// parts (ssd_split.cuh).  Also here: inter-chunk state passing of that path, and the backward's finishing scans and reductions of
// every path.
//
// Notation per (batch b, head h), chunk of Q steps: a_t = dt_t*A_h, cs_t = inclusive cumsum of a
// inside the chunk, H_in = state entering the chunk, Gout = dLoss/d(state leaving the chunk).
// All of it is Eq. 1 of the paper regrouped by chunks; the segment hand-off is Algorithms 1 and 2.
#include "ssd_internal.h"
#include "ssd_split.cuh"

// State-pass CTAs: 128 threads, at most 48 registers, so that a segment's CTAs are resident at once; chunks fetched ahead.
#define SP_THREADS 128
#define SP_ELEMS (SP_THREADS * 4)
#define SP_CTAS 10
#define SP_PF 4
static_assert(SP_ELEMS == ssd::kStatePassElems, "one partial of <G,H> per CTA of the backward pass");
namespace ssd {

// the finishing step: heads per CTA, its shared-memory tile
constexpr int FIN_HB = 8;
constexpr int FIN_TILE = 256 * (FIN_HB + 1);

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

// ------------------------------------------------------------------ contractions
// One shape for all of them: a 64 x 64 output tile per CTA of eight warps, 64 steps of the contraction at a time, on the tensor
// cores with fp32 operands as three bf16 parts (ssd_split.cuh): three products where the other operand is bf16 as it stands, six
// where both are fp32, one where neither is.  Operands are staged as rows, split on the way; the next stage's global loads are in
// flight while a stage is multiplied.  With FFMA on the CUDA cores (4 x 4 outputs per thread, bound by the shared-memory reads) the
// large kernel took 309 us (2 x 2048 steps of 32 heads, N = 64, chunk 128, bf16) and 215 us (2 x 1024 of 24, N = 128, fp32), now 130
// and 134, y 119 and 92 us, now 50 and 55.  Bound by latency: masks, splits and addresses around each product, between barriers, at 24
// (fp32: 16) warps per SM (of 550 TFLOP/s that mma.sync does here the tensor pipe is 27 to 50 % busy).  bf16 takes 80 registers a thread, for
// three CTAs per SM, with some spills (the backward's large kernel 128, for two); fp32, with more parts in registers, takes 128 (2 x 4096
// steps: 1112 us, at 80: 1260).
//
// What does not depend on the head is not done per head: C B^T is made once per group (k_simt_sums writes it, 64 x 64 causal
// tiles), and dB / dC come from a head sum of the masked tiles, one product per CTA instead of two per head.
template <typename T> struct SimtSmem {
    static constexpr int PT = SplitParts<T>::n;      // parts of a value of the caller's tensors
    static constexpr int CTAS = PT == 1 ? 3 : 2;     // CTAs per SM
    SplitTile t[3 + PT];
    float css[256], dts[256], fac[256], red[6][64];
    int again;                                       // a product of this CTA came out as NaN
};
constexpr int ST_LD = 72;                            // floats per row of an output tile staged in t[0], t[1]
static_assert(64 * ST_LD * sizeof(float) <= 2 * sizeof(SplitTile), "an fp32 output tile in the place of two parts");
static_assert(FIN_TILE * sizeof(float) <= 2 * sizeof(SplitTile), "the finishing step's tile");

template <typename T> __device__ __forceinline__ SimtSmem<T> &simt_smem() {
    extern __shared__ __align__(16) unsigned char smem[];
    return *reinterpret_cast<SimtSmem<T> *>(smem);
}
// A CTA some of whose sums are NaN (`again` in its shared memory; its body returns true) runs once more with AGAIN, for infinities (see
// tile_mma), and writes its outputs a second time.  That costs a check of its last accumulators and, in effect, what a second body does to
// registers and code.  In line: 2 x 4096 steps of 24 heads, fp32, 1029 -> 1027 us, 2 x 8192 of 32, bf16, 1013 -> 1019, 1024 of 4, fp32, 106.7 as
// before; with a function of its own 1031, 1029 and 109; with one body and a flag 1089, 1099 and 113.
template <typename T> __device__ __forceinline__ float4 ld4f(const T *p);
template <> __device__ __forceinline__ float4 ld4f<float>(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
template <> __device__ __forceinline__ float4 ld4f<__nv_bfloat16>(const __nv_bfloat16 *p) {
    const uint2 v = __ldg(reinterpret_cast<const uint2 *>(p));
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float2 ld2f(const float *p) { return __ldg(reinterpret_cast<const float2 *>(p)); }
__device__ __forceinline__ float2 ld2f(const __nv_bfloat16 *p) {
    const uint32_t v = __ldg(reinterpret_cast<const uint32_t *>(p));
    return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
}
// sum over the 16 lanes of a half warp
__device__ __forceinline__ float sum_tx(float v) {
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}
// sum over the four lanes that share an accumulator row
__device__ __forceinline__ float sum_quad(float v) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 2);
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
// an output tile in accumulator layout to rows of `stride` floats: four lanes fill a 32-byte sector
__device__ __forceinline__ void store_acc(const Acc &acc, float *out, size_t stride) {
#pragma unroll
    for (int half = 0; half < 2; ++half)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            *reinterpret_cast<float2 *>(out + (size_t)acc_row(half) * stride + acc_col(j)) = acc.get(j, half);
}
// two neighbouring elements of an accumulator-layout tile as three parts
__device__ __forceinline__ void put_acc(SplitTile *s, int half, int j, float a, float b) {
    uint32_t w[3];
    split2(a, b, w);
#pragma unroll
    for (int q = 0; q < 3; ++q) *reinterpret_cast<uint32_t *>(&s[q].v[acc_row(half)][acc_col(j)]) = w[q];
}

// Up to this decay (natural units) inside a 64-step tile the mask on its diagonal is a product of two factors, beyond it an
// exponential per element.  Factors of arguments up to 8 are rounded like cumulative sums of that size.
constexpr float kMildTile = 8.f;

// What a segment's chunks need before the states can be passed on, by block number:
//   S_c[p,n] = sum_s exp(cs_last - cs_s) dt_s x_s[p] B_s[n]     -> Hst slot c+1   (and cs, dtT)
//   with grads: E_c[p,n] = sum_t exp(cs_t) dy_t[p] C_t[n]       -> Gst slot c      (its CTAs make the cumsum again)
//   the causal tiles of C B^T, where the scratch has room for them
// Both sums of a (head, chunk) by one CTA, with one cumsum, where there are CTAs enough; else two, side by side.  Backward, us, with two and
// with one, by the CTAs of one: 192 (bf16, N = 64, 8192 steps of 24 heads) 404 and 438, (fp32, N = 128, 4096 of 24) 441 and 429; 256 (fp32, N = 64,
// 4096 of 8, chunks of 64) 133 and 132; 384 (fp32, 2 x 4096 of 24) 756 and 750; 512 (bf16, N = 64, 2 x 8192 of 32) 853 and 817, (fp32, 2 x 8192
// of 8, chunks of 64) 405 and 382; 768 (bf16, N = 128, 8192 of 24) 517 and 494.
template <int NS> __host__ __device__ __forceinline__ bool simt_sums_merged(const SegParams &p) { return p.nc * p.B * (NS / 64) * p.H >= 2 * kNumSMs; }
template <int NS> __host__ __device__ __forceinline__ int simt_n_sums(const SegParams &p, bool grads) {
    const int nrt = p.Q >> 6;
    return p.nc * p.B * ((NS / 64) * p.H * (grads && !simt_sums_merged<NS>(p) ? 2 : 1) + (p.cbt ? p.G * (nrt * (nrt + 1) / 2) : 0));
}
template <typename T, int NS, bool AGAIN> __device__ __forceinline__ bool simt_sums(const SegParams &p, SimtSmem<T> &sm, int id, bool grads) {
    constexpr int PT = SimtSmem<T>::PT;
    const int tid = threadIdx.x, Q = p.Q, nrt = Q >> 6, nh = NS / 64;
    const size_t HP = (size_t)p.H * 64, GN = (size_t)p.G * NS;
    const int nsum = p.nc * nh * p.H * p.B;
    float *wsm = sm.css;
    Acc acc;
    TileRegs<T> ra, rb;
    acc.zero();
    const bool merged = grads && simt_sums_merged<NS>(p);
    const bool second = grads && !merged && id >= nsum && id < 2 * nsum;       // a CTA for E alone
    if (second) id -= nsum;
    else if (id >= nsum) {      // a causal tile of C B^T
        id -= grads && !merged ? 2 * nsum : nsum;
        const int npair = nrt * (nrt + 1) / 2;
        int rt, ct;
        pair_of(id % npair, rt, ct);
        id /= npair;
        const int g = id % p.G, c = (id / p.G) % p.nc, b = id / (p.G * p.nc);
        const size_t o = (size_t)b * p.bc_bs + ((size_t)p.t0 + (size_t)c * Q) * GN + (size_t)g * NS;
        const T *C = (const T *)p.Cm + o + (size_t)rt * 64 * GN, *Bp = (const T *)p.Bm + o + (size_t)ct * 64 * GN;
        for (int k0 = 0; k0 < NS; k0 += 64) {
            tile_load(ra, C + k0, GN);
            tile_load(rb, Bp + k0, GN);
            if (k0) __syncthreads();
            else pdl_wait();
            tile_store(sm.t, ra);
            tile_store(sm.t + PT, rb);
            __syncthreads();
            tile_mma<PT, PT, false, false, AGAIN>(acc, sm.t, sm.t + PT);
        }
        store_acc(acc, cb_of(p, b, c, g) + (size_t)rt * 64 * Q + ct * 64, Q);
        return PT > 1 && !AGAIN && __syncthreads_or(acc.nan());
    }
    const int n0 = (id % nh) * 64;
    id /= nh;
    const int bc = divide_by(id, p.H, p.inv_H), h = id - bc * p.H, b = divide_by(bc, p.nc, p.inv_nc), c = bc - b * p.nc, g = h / p.hpg;
    const size_t tok0 = (size_t)p.t0 + (size_t)c * Q;
    const size_t xo = (size_t)b * p.x_bs + tok0 * HP + (size_t)h * 64, bo = (size_t)b * p.bc_bs + tok0 * GN + (size_t)g * NS + n0;
    float *wsm2 = sm.dts;                                                       // the weights of E
    auto load_rows = [&](bool dst, int s0) {
        tile_load(ra, (const T *)(dst ? p.dy : p.x) + xo + (size_t)s0 * HP, HP);
        tile_load(rb, (const T *)(dst ? p.Cm : p.Bm) + bo + (size_t)s0 * GN, GN);
    };
    load_rows(second, 0);
    // the chunk cumsum by one warp: a lane sums its Q/32 consecutive steps in order, then a shuffle scan over the lanes
    if (tid < 32) {
        const int per = Q >> 5;
        const float Ah = __ldg(p.A + h);
        float d[8], v[8], run = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (k < per) d[k] = __ldg(p.dt + (size_t)b * p.dt_bs + (tok0 + tid * per + k) * p.H + h);
        pdl_wait();
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
                if (!second) wsm[t] = expf(fminf(last - cs, 0.f)) * d[k];
                if (second || merged) wsm2[t] = expf(cs);
                if (n0 == 0 && !second) {
                    p.cs[vec_off(p, b, h, c) + t] = cs;
                    p.dtT[vec_off(p, b, h, c) + t] = d[k];
                }
            }
    } else {
        pdl_wait();
    }
    __syncthreads();
    const int end = merged ? 2 * Q : Q;
    if (!AGAIN && tid == 0) sm.again = 0;
    for (int i0 = 0; i0 < end; i0 += 64) {
        const bool dst = second || i0 >= Q;
        const int s0 = i0 >= Q ? i0 - Q : i0;
        const float *wv = dst ? wsm2 : wsm;
#pragma unroll
        for (int k = 0; k < TileRegs<T>::N; ++k) {
            const float w = wv[s0 + ra.row(k)];
            float f[TileRegs<T>::COLS];
            ra.get(k, f);
#pragma unroll
            for (int i = 0; i < TileRegs<T>::COLS; ++i) f[i] *= w;
            put_split(sm.t, ra.row(k), ra.col(), f);
        }
        tile_store(sm.t + 3, rb);
        __syncthreads();
        if (i0 + 64 < end) load_rows(second || i0 + 64 >= Q, i0 + 64 >= Q ? i0 + 64 - Q : i0 + 64);
        tile_mma<3, PT, true, true, AGAIN>(acc, sm.t, sm.t + 3);
        if (s0 + 64 == Q) {
            if (!AGAIN && acc.nan()) sm.again = 1;
            store_acc(acc, (dst ? p.Gst + slot_off(p, b, c, h) : p.Hst + slot_off(p, b, c + 1, h)) + n0, NS);
            acc.zero();
        }
        __syncthreads();
    }
    return !AGAIN && sm.again;
}

template <typename T, int NS> __global__ void __launch_bounds__(256, SimtSmem<T>::CTAS) k_simt_sums(const __grid_constant__ SegParams p, bool grads) {
    pdl_launch_dependents();
    if (p.first && blockIdx.x == 0 && threadIdx.x < 64) p.status[threadIdx.x] = 0u;
    if (simt_sums<T, NS, false>(p, simt_smem<T>(), blockIdx.x, grads)) simt_sums<T, NS, true>(p, simt_smem<T>(), blockIdx.x, grads);
}

template <int NS> __device__ __forceinline__ size_t slot_of(const SegParams &p, int b, int slot, int h) {
    return (((size_t)b * (p.ncs + 1) + slot) * p.H + h) * (size_t)(64 * NS);
}
// Columns k0 .. k0 + 63 of the state entering chunk c (GRAD: of the gradient leaving it): from the slot that a state pass filled, or
// (READER) made here from the sums of the chunks on that side, with the pass's operations in its order, so with the same bits.
template <int NS, bool GRAD, bool READER>
__device__ __forceinline__ void load_state(TileRegs<float> &r, const SegParams &p, int b, int h, int c, int k0) {
    const float *slots = GRAD ? p.Gst : p.Hst;
    if constexpr (!READER) {
        tile_load<true>(r, slots + slot_of<NS>(p, b, GRAD ? c + 1 : c, h) + k0, NS);
    } else {
        const float *init = GRAD ? p.ginit : p.hinit, *csl = p.cs + vec_off(p, b, h, 0) + (p.Q - 1);
        if (init) {
            tile_load<true>(r, init + (size_t)b * (GRAD ? p.ginit_bs : p.hinit_bs) + (size_t)h * 64 * NS + k0, NS);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) r.v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const int n = GRAD ? p.nc - 1 - c : c;
        for (int i = 0; i < n; ++i) {
            const int j = GRAD ? p.nc - 1 - i : i;
            TileRegs<float> s;
            tile_load<true>(s, slots + slot_of<NS>(p, b, GRAD ? j : j + 1, h) + k0, NS);
            const float decay = expf(csl[(size_t)j * p.Q]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                r.v[k].x = fmaf(decay, r.v[k].x, s.v[k].x);
                r.v[k].y = fmaf(decay, r.v[k].y, s.v[k].y);
                r.v[k].z = fmaf(decay, r.v[k].z, s.v[k].z);
                r.v[k].w = fmaf(decay, r.v[k].w, s.v[k].w);
            }
        }
    }
}

// What is left of a state pass where the readers make the states: the state (BWD: the gradient) handed on, the boundary state, and
// (BWD) the partial sums of <Gout, H_in>.  1024 elements per CTA, kReaderChunks chunks at most, all loads in flight.
template <bool BWD> __device__ __forceinline__ void pass_along(const SegParams &p, const StatePass &a, float *red, int id) {
    const int PN = p.P * p.N, nblk = PN / 1024, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int blk = id % nblk, h = (id / nblk) % p.H, b = id / (nblk * p.H), e = blk * 1024 + tid * 4;
    const size_t he = (size_t)h * PN + e;
    const float *csl = p.cs + vec_off(p, b, h, 0) + (p.Q - 1);
    auto at = [](const float *q) { return *reinterpret_cast<const float4 *>(q); };
    auto step = [](float4 &c, float decay, const float4 &s) {
        c.x = fmaf(decay, c.x, s.x);
        c.y = fmaf(decay, c.y, s.y);
        c.z = fmaf(decay, c.z, s.z);
        c.w = fmaf(decay, c.w, s.w);
    };
    float4 carry = make_float4(0.f, 0.f, 0.f, 0.f), sv[kReaderChunks];
    float dec[kReaderChunks];
    if (p.hinit) carry = at(p.hinit + (size_t)b * p.hinit_bs + he);
#pragma unroll
    for (int c = 0; c < kReaderChunks; ++c)
        if (c < p.nc) {
            sv[c] = at(p.Hst + slot_off(p, b, c + 1, h) + e);
            dec[c] = expf(csl[(size_t)c * p.Q]);
        }
    if (!BWD && a.boundary) *reinterpret_cast<float4 *>(a.boundary + (size_t)b * a.boundary_bs + he) = carry;
#pragma unroll
    for (int c = 0; c < kReaderChunks; ++c)
        if (c < p.nc) {
            const float4 in = carry;
            step(carry, dec[c], sv[c]);
            if (BWD) sv[c] = in;            // the state entering chunk c
        }
    if (!BWD) {
        if (a.leave) *reinterpret_cast<float4 *>(a.leave + (size_t)b * a.leave_bs + he) = carry;
        if (a.fin) *reinterpret_cast<float4 *>(a.fin + (size_t)b * p.H * PN + he) = carry;
        return;
    }
    carry = p.ginit ? at(p.ginit + (size_t)b * p.ginit_bs + he) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int c = kReaderChunks - 1; c >= 0; --c)
        if (c < p.nc) {
            const float4 ev = at(p.Gst + slot_off(p, b, c, h) + e);
            float part = carry.x * sv[c].x;
            part = fmaf(carry.y, sv[c].y, part);
            part = fmaf(carry.z, sv[c].z, part);
            part = fmaf(carry.w, sv[c].w, part);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
            if (lane == 0) red[c * 8 + warp] = dec[c] * part;
            step(carry, dec[c], ev);
        }
    *reinterpret_cast<float4 *>(a.leave + (size_t)b * a.leave_bs + he) = carry;
    __syncthreads();
    if (tid < 2 * p.nc) {                   // two partial sums of 512 elements, as the pass has them
        const float *r = red + (tid >> 1) * 8 + (tid & 1) * 4;
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < 4; ++w) s += r[w];
        p.ghdot[((((size_t)b * p.H + h) * p.ncs + (tid >> 1)) << 4) + blk * 2 + (tid & 1)] = s;
    }
}

// One 64-row tile of y (DX = false) or of dx (DX = true) of one head:
//   y_t  = sum_{s<=t} CB[t,s] e^{cs_t-cs_s} dt_s x_s + e^{cs_t} C_t H_in + D x_t
//   u_s  = sum_{t>=s} CB[t,s] e^{cs_t-cs_s} dy_t     + e^{cs_last-cs_s} B_s Gout ;  dx_s = D dy_s + dt_s u_s ,
//   ddt_direct_s = x_s . u_s , psi2_s = dt_s e^{cs_last-cs_s} x_s . (Gout B_s) , dD partial = sum dy.x
// CB false (y only): the tiles of C B^T are not in the scratch and are made here, per head, with the same operations in the same
// order, so with the same bits.
template <typename T, int NS, bool DX, bool CB, bool READER, bool AGAIN>
__device__ __forceinline__ bool simt_row_tile(const SegParams &p, SimtSmem<T> &sm, int c, int rt, int h, int b) {
    constexpr int PT = SimtSmem<T>::PT;
    float *css = sm.css, *dts = sm.dts, *fac = sm.fac, *facd = sm.red[5];
    const int tid = threadIdx.x, Q = p.Q, nrt = Q >> 6, g = h / p.hpg, r0 = rt * 64;
    const size_t tok0 = (size_t)p.t0 + (size_t)c * Q, HP = (size_t)p.H * 64, GN = (size_t)p.G * NS;
    const size_t xo = (size_t)b * p.x_bs + tok0 * HP + (size_t)h * 64;
    const T *vals = (const T *)(DX ? p.dy : p.x) + xo;
    const T *rowv = (const T *)(DX ? p.Bm : p.Cm) + (size_t)b * p.bc_bs + (tok0 + r0) * GN + (size_t)g * NS;
    const float *cbt = cb_of(p, b, c, g);
    TileRegs<T> rv;
    TileRegs<float> rf;
    Acc acc;
    acc.zero();
    if (!AGAIN && tid == 0) sm.again = 0;
    tile_load(rv, rowv, GN);
    pdl_wait();
    load_state<NS, DX, READER>(rf, p, b, h, c, 0);
    for (int t = tid; t < Q; t += 256) {
        css[t] = p.cs[vec_off(p, b, h, c) + t];
        dts[t] = p.dtT[vec_off(p, b, h, c) + t];
    }
    // CB tile and value rows of column tile ct: rows t, columns s of the CB matrix; for dx its columns are the output's rows
    auto load_vals = [&](int ct) {
        if (CB) tile_load<true>(rf, DX ? cbt + (size_t)ct * 64 * Q + r0 : cbt + (size_t)r0 * Q + ct * 64, Q);
        tile_load(rv, vals + (size_t)ct * 64 * HP, HP);
    };
    const int ct0 = DX ? rt : 0, ct1 = DX ? nrt : rt + 1;
    for (int k0 = 0; k0 < NS; k0 += 64) {
        tile_store(sm.t, rv);
        tile_store(sm.t + PT, rf);
        __syncthreads();
        if (k0 + 64 < NS) {
            tile_load(rv, rowv + k0 + 64, GN);
            load_state<NS, DX, READER>(rf, p, b, h, c, k0 + 64);
        } else if (CB) {
            load_vals(ct0);
        }
        tile_mma<PT, 3, false, false, AGAIN>(acc, sm.t, sm.t + PT);
        __syncthreads();
    }
    // Off the diagonal tile the mask factors at the tile's edge m (its first row; dx: last), where both factors are <= 1:
    // e^{cs_t-cs_s} = e^{cs_t-cs_m} e^{cs_m-cs_s}.  An exponential per step instead of one per element.
    // On it one of the two is >= 1, and their product no worse than the difference of the cumulative sums where those are close:
    // facd, for mild decays.
    const int m = DX ? r0 + 63 : r0;
    const bool mild = css[r0] - css[r0 + 63] <= kMildTile;
    for (int t = tid; t < Q; t += 256) {
        const float d = css[t] - css[m];
        fac[t] = expf(fminf(t >= m ? d : -d, 0.f)) * (DX || t >= m ? 1.f : dts[t]);
    }
    if (tid < 64) facd[tid] = DX ? expf(css[r0 + tid] - css[m]) : expf(css[m] - css[r0 + tid]) * dts[r0 + tid];
    __syncthreads();
    // the inter-chunk term is complete: scale its rows
    const float cl = css[Q - 1];
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const int r = r0 + acc_row(half);
        const float o = DX ? expf(fminf(cl - css[r], 0.f)) : expf(css[r]);
        float dd2 = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 v = __fmul2_rn(make_float2(o, o), acc.get(j, half));
            acc.set(j, half, v);
            if (DX) {
                const float2 xv = ld2f((const T *)p.x + xo + (size_t)r * HP + acc_col(j));
                dd2 += xv.x * v.x + xv.y * v.y;
            }
        }
        if (DX) {
            dd2 = sum_quad(dd2);
            if ((tid & 3) == 0) sm.red[tid >> 7][acc_row(half)] = dd2;
        }
    }
    for (int ct = ct0; ct < ct1; ++ct) {
        if constexpr (!CB) {
            const T *colv = (const T *)p.Bm + (size_t)b * p.bc_bs + (tok0 + ct * 64) * GN + (size_t)g * NS;
            Acc cb;
            cb.zero();
            for (int k0 = 0; k0 < NS; k0 += 64) {
                TileRegs<T> rc;
                tile_load(rv, rowv + k0, GN);
                tile_load(rc, colv + k0, GN);
                tile_store(sm.t, rv);
                tile_store(sm.t + PT, rc);
                __syncthreads();
                tile_mma<PT, PT, false, false, AGAIN>(cb, sm.t, sm.t + PT);
                __syncthreads();
            }
            load_vals(ct);
#pragma unroll
            for (int half = 0; half < 2; ++half)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int t = r0 + acc_row(half), s = ct * 64 + acc_col(j);
                    const float2 v2 = cb.get(j, half);
                    float e[2] = {v2.x, v2.y};
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        if (ct != rt) e[i] *= fac[t] * fac[s + i];
                        else if (mild) e[i] = s + i <= t ? e[i] * (fac[t] * facd[acc_col(j) + i]) : 0.f;
                        else e[i] = s + i <= t ? e[i] * expf(fminf(css[t] - css[s + i], 0.f)) * dts[s + i] : 0.f;
                    }
                    put_acc(sm.t, half, j, e[0], e[1]);
                }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                // rows t, columns s
                float e[4];
                rf.get(k, e);
                const int t = (DX ? ct * 64 : r0) + rf.row(k), s = (DX ? r0 : ct * 64) + rf.col();
                if (ct != rt || mild) {
                    const float one = DX && ct == rt ? facd[rf.row(k)] : fac[t];
                    const float4 four = *reinterpret_cast<const float4 *>(!DX && ct == rt ? facd + rf.col() : fac + s);
                    e[0] *= one * four.x; e[1] *= one * four.y; e[2] *= one * four.z; e[3] *= one * four.w;
                    if (ct == rt) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) e[i] = s + i <= t ? e[i] : 0.f;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) e[i] = s + i <= t ? e[i] * expf(fminf(css[t] - css[s + i], 0.f)) * (DX ? 1.f : dts[s + i]) : 0.f;
                }
                put_split(sm.t, rf.row(k), rf.col(), e);
            }
        }
        tile_store(sm.t + 3, rv);
        __syncthreads();
        if (CB && ct + 1 < ct1) load_vals(ct + 1);
        tile_mma<3, PT, DX, true, AGAIN>(acc, sm.t, sm.t + 3);
        __syncthreads();
    }
    // through shared memory, so that the caller's rows are read and written in whole sectors
    float *stg = reinterpret_cast<float *>(sm.t);
    store_acc(acc, stg, ST_LD);
    if (!AGAIN && acc.nan()) sm.again = 1;
    __syncthreads();
    if (!AGAIN && sm.again) return true;
    const float Dh = __ldg(p.D + h) + (DX ? p.dx_skip : 0.f);      // dx: D dy, plus dy itself under a skip connection
    float dsum = 0.f, dprev = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int rl = (tid >> 4) + 16 * k, r = r0 + rl, cl4 = (tid & 15) * 4;
        const size_t o = xo + (size_t)r * HP + cl4;
        const float4 a = *reinterpret_cast<const float4 *>(stg + rl * ST_LD + cl4);
        const float4 v = ld4f((const T *)(DX ? p.dy : p.x) + o);
        const float s = DX ? dts[r] : 1.f;
        st4((T *)(DX ? p.dx : p.y) + o, make_float4(fmaf(Dh, v.x, s * a.x), fmaf(Dh, v.y, s * a.y), fmaf(Dh, v.z, s * a.z), fmaf(Dh, v.w, s * a.w)));
        if (DX) {
            const float4 xv = ld4f((const T *)p.x + o);
            const float dd = sum_tx(xv.x * a.x + xv.y * a.y + xv.z * a.z + xv.w * a.w);
            const float dk = (v.x * xv.x + v.y * xv.y) + (v.z * xv.z + v.w * xv.w);
            if (k & 1) dsum += dprev + dk;
            else dprev = dk;
            if ((tid & 15) == 0) {
                p.ddt_dir[vec_off(p, b, h, c) + r] = dd;
                p.psi2[vec_off(p, b, h, c) + r] = dts[r] * (sm.red[0][rl] + sm.red[1][rl]);
            }
        }
    }
    if (DX) {       // deterministic block sum of dy*x
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) dsum += __shfl_xor_sync(0xffffffffu, dsum, off);
        if ((tid & 31) == 0) sm.red[2][tid >> 5] = dsum;
        __syncthreads();
        if (tid == 0) {
            float s = 0.f;
#pragma unroll
            for (int w = 0; w < 8; ++w) s += sm.red[2][w];
            p.dDp[((((size_t)b * p.H + h) * p.nct + p.c0 + c) << 2) + rt] = s;
        }
    }
    return false;
}

// y of a segment and, in the same launch where the scratch has a second copy, the sums of the next segment (n_next CTAs): they
// wait for nothing of this one, and a launch of a few microseconds is saved per segment.  READER: no state pass has run; n_pass
// CTAs make what it hands on.
template <typename T, int NS, bool CB, bool READER, bool AGAIN>
__device__ __forceinline__ bool simt_y(const SegParams &p, const SegParams &nx, int n_next, const StatePass &pass, int n_pass) {
    SimtSmem<T> &sm = simt_smem<T>();
    const int nrt = p.Q >> 6, ny = (int)gridDim.x - n_next;
    int id = blockIdx.x;
    if (id >= ny) return simt_sums<T, NS, AGAIN>(nx, sm, id - ny, false);
    if (READER && id >= ny - n_pass) {
        pdl_wait();
        pass_along<false>(p, pass, sm.red[0], id - (ny - n_pass));
        return false;
    }
    const int rt = id & (nrt - 1), bhc = id >> (nrt >> 1), bh = divide_by(bhc, p.nc, p.inv_nc), c = bhc - bh * p.nc, b = divide_by(bh, p.H, p.inv_H),
              h = bh - b * p.H;       // nrt is 1, 2 or 4
    return simt_row_tile<T, NS, false, CB, READER, AGAIN>(p, sm, c, rt, h, b);
}
template <typename T, int NS, bool CB, bool READER>
__global__ void __launch_bounds__(256, SimtSmem<T>::CTAS)
k_simt_y(const __grid_constant__ SegParams p, const __grid_constant__ SegParams nx, int n_next, const __grid_constant__ StatePass pass, int n_pass) {
    pdl_launch_dependents();
    if (simt_y<T, NS, CB, READER, false>(p, nx, n_next, pass, n_pass)) simt_y<T, NS, CB, READER, true>(p, nx, n_next, pass, n_pass);
}

// A CTA's part of dB and dC (the roles below)
template <typename T, int NS, bool READER, bool AGAIN> __device__ __forceinline__ bool simt_dbdc(const SegParams &p, SimtSmem<T> &sm, int id) {
    constexpr int PT = SimtSmem<T>::PT;
    const int tid = threadIdx.x, lane = tid & 31, Q = p.Q, nrt = Q >> 6, npair = nrt * (nrt + 1) / 2;
    const int per = npair + 2 * nrt, role = id % per;
    id /= per;
    if (!AGAIN && tid == 0) sm.again = 0;
    const int rng = p.nsl / (nrt + 3);                         // head ranges per group
    const int sl = id % rng, g = (id / rng) % p.G, c = (id / (rng * p.G)) % p.nc, b = id / (rng * p.G * p.nc);
    const int hps = (p.hpg + rng - 1) / rng, h0 = g * p.hpg + sl * hps, h1 = min(h0 + hps, (g + 1) * p.hpg);
    const size_t tok0 = (size_t)p.t0 + (size_t)c * Q, HP = (size_t)p.H * 64, GN = (size_t)p.G * NS;
    const T *xb = (const T *)p.x + (size_t)b * p.x_bs + tok0 * HP, *dyb = (const T *)p.dy + (size_t)b * p.x_bs + tok0 * HP;
    const T *Bb = (const T *)p.Bm + (size_t)b * p.bc_bs + tok0 * GN + (size_t)g * NS, *Cb = (const T *)p.Cm + (size_t)b * p.bc_bs + tok0 * GN + (size_t)g * NS;
    auto slice = [&](int row0, int slot, int n0) {
        return p.pC + ((((size_t)b * p.ncs * Q + (size_t)c * Q + row0) * p.G + g) * p.nsl + sl * (nrt + 3) + slot) * NS + n0;
    };
    const size_t slice_stride = (size_t)p.G * p.nsl * NS;
    Acc acc;
    if (role < npair) {
        int tt, ts;
        pair_of(role, tt, ts);
        TileRegs<T> ra, rb;
        float2 cb[2][4], ws[2][4];
        auto load_rows = [&](int h) {
            tile_load(ra, dyb + (size_t)tt * 64 * HP + (size_t)h * 64, HP);
            tile_load(rb, xb + (size_t)ts * 64 * HP + (size_t)h * 64, HP);
        };
        load_rows(h0);
        pdl_wait();
#pragma unroll
        for (int half = 0; half < 2; ++half)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                cb[half][j] = *reinterpret_cast<const float2 *>(cb_of(p, b, c, g) + (size_t)(tt * 64 + acc_row(half)) * Q + ts * 64 + acc_col(j));
                ws[half][j] = make_float2(0.f, 0.f);
            }
        // a head's vectors, a value each of 128 threads: the mask's factors at the row tile's first step, as for y, or, on the
        // diagonal of a stiff head, cumulative sum and step size
        float *rowv = sm.fac, *colv = sm.fac + 64;
        const bool diag = tt == ts;
        float va = 0.f, vb = 0.f, vref, vlast;
        auto load_vec = [&](int h) {
            const size_t vo = vec_off(p, b, h, c);
            if (tid < 128) {
                const size_t o = vo + (tid < 64 ? tt : ts) * 64 + (tid & 63);
                va = p.cs[o];
                vb = p.dtT[o];
            }
            vref = p.cs[vo + tt * 64];
            vlast = p.cs[vo + tt * 64 + 63];
        };
        load_vec(h0);
        for (int h = h0; h < h1; ++h) {
            tile_store(sm.t, ra);
            tile_store(sm.t + PT, rb);
            const bool factors = !diag || vref - vlast <= kMildTile;
            if (tid < 128) {
                const float d = tid < 64 ? va - vref : vref - va, e = expf(diag ? d : fminf(d, 0.f));
                sm.fac[tid] = factors ? (tid < 64 ? e : e * vb) : (tid < 64 ? va : vb);
            }
            __syncthreads();
            if (h + 1 < h1) {
                load_rows(h + 1);
                load_vec(h + 1);
            }
            acc.zero();
            tile_mma<PT, PT, false, false, AGAIN>(acc, sm.t, sm.t + PT);
            float2 row[2], col[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) col[j] = make_float2(0.f, 0.f);
            row[0] = row[1] = col[0];
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int t = acc_row(half);
                const float one = rowv[t];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int s = acc_col(j);
                    const float2 two = *reinterpret_cast<const float2 *>(colv + s);
                    float2 e;
                    if (factors) {
                        e = __fmul2_rn(make_float2(one, one), two);
                    } else {
                        e.x = expf(fminf(one - rowv[s], 0.f)) * two.x;
                        e.y = expf(fminf(one - rowv[s + 1], 0.f)) * two.y;
                    }
                    float2 w = __fmul2_rn(acc.get(j, half), e);
                    if (diag) {
                        w.x = s <= t ? w.x : 0.f;
                        w.y = s < t ? w.y : 0.f;
                    }
                    ws[half][j] = __fadd2_rn(ws[half][j], w);
                    // s = t adds the same to rho_t and psi_t, of which only sums of differences are used: left out of both, or with
                    // strong decays, where it is the largest term, its rounding would be most of the error of dA
                    if (diag) {
                        w.x = s == t ? 0.f : w.x;
                        w.y = s + 1 == t ? 0.f : w.y;
                    }
                    row[half] = __ffma2_rn(w, cb[half][j], row[half]);
                    col[j] = __ffma2_rn(w, cb[half][j], col[j]);
                }
                const float r = sum_quad(row[half].x + row[half].y);
                if ((lane & 3) == 0) sm.red[tid >> 7][t] = r;
            }
            // column sums over the warp's rows: transposing butterfly, the eight lanes of a column pair end with a column each
            const int gl = lane >> 2;
            float cv[8] = {col[0].x, col[0].y, col[1].x, col[1].y, col[2].x, col[2].y, col[3].x, col[3].y};
#pragma unroll
            for (int o = 4; o >= 1; o >>= 1) {
                const bool up = (gl & o) != 0;
#pragma unroll
                for (int i = 0; i < o; ++i) {
                    const float send = up ? cv[i] : cv[i + o], keep = up ? cv[i + o] : cv[i];
                    cv[i] = keep + __shfl_xor_sync(0xffffffffu, send, o * 4);
                }
            }
            sm.red[2 + ((tid >> 5) & 3)][acc_col(gl >> 1) + (gl & 1)] = cv[0];
            __syncthreads();
            const size_t vo = (vec_off(p, b, h, c) * nrt);      // rho, psi: [B,H,ncs,Q/64 tiles,Q]
            if (tid < 64) p.rho[vo + (size_t)ts * Q + tt * 64 + tid] = sm.red[0][tid] + sm.red[1][tid];
            else if (tid < 128) p.psi[vo + (size_t)tt * Q + ts * 64 + tid - 64] = (sm.red[2][tid - 64] + sm.red[3][tid - 64]) + (sm.red[4][tid - 64] + sm.red[5][tid - 64]);
            // red and the tiles are rewritten only after the next head's first barrier or by threads that are past this one
        }
        // dC[tt] = Wsum B_ts and dB[ts] = Wsum^T C_tt
#pragma unroll
        for (int half = 0; half < 2; ++half)
#pragma unroll
            for (int j = 0; j < 4; ++j) put_acc(sm.t, half, j, ws[half][j].x, ws[half][j].y);
        tile_load(rb, Bb + (size_t)ts * 64 * GN, GN);
#pragma unroll 1
        for (int n0 = 0; n0 < 2 * NS; n0 += 64) {
            const bool isB = n0 >= NS;
            const int n = isB ? n0 - NS : n0;
            tile_store(sm.t + 3, rb);
            __syncthreads();
            if (n0 + 64 < 2 * NS) tile_load(rb, n0 + 64 >= NS ? Cb + (size_t)tt * 64 * GN + n0 + 64 - NS : Bb + (size_t)ts * 64 * GN + n0 + 64, GN);
            acc.zero();
            if (isB) tile_mma<3, PT, true, true, AGAIN>(acc, sm.t, sm.t + 3);
            else tile_mma<3, PT, false, true, AGAIN>(acc, sm.t, sm.t + 3);
            if (!AGAIN && acc.nan()) sm.again = 1;         // (a NaN of the head sum is in its whole row of the product)
            store_acc(acc, isB ? slice(ts * 64, tt + 1, n) : slice(tt * 64, ts, n), slice_stride);
            __syncthreads();
        }
        return !AGAIN && sm.again;
    }
    // inter-chunk terms of one row tile: the head's rows times the chunk state (rows p), the products scaled per row
    const bool isC = role - npair < nrt;
    const int rt = (role - npair) % nrt;
    TileRegs<T> ra;
    TileRegs<float> rf;
    float2 tot[NS / 64][2][4];
#pragma unroll
    for (int m = 0; m < NS / 64; ++m)
#pragma unroll
        for (int j = 0; j < 4; ++j) tot[m][0][j] = tot[m][1][j] = make_float2(0.f, 0.f);
    auto state = [&](int h, int k0) {
        if (isC) load_state<NS, false, READER>(rf, p, b, h, c, k0);
        else load_state<NS, true, READER>(rf, p, b, h, c, k0);
    };
    const T *rows = (isC ? dyb : xb) + (size_t)rt * 64 * HP;
    tile_load(ra, rows + (size_t)h0 * 64, HP);
    pdl_wait();
    state(h0, 0);
    for (int h = h0; h < h1; ++h) {
        const size_t vo = vec_off(p, b, h, c);
        const float cl = p.cs[vo + Q - 1];
        float sc[2], rho2[2] = {0.f, 0.f};
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const float v = p.cs[vo + rt * 64 + acc_row(half)];
            sc[half] = isC ? expf(v) : p.dtT[vo + rt * 64 + acc_row(half)] * expf(fminf(cl - v, 0.f));
        }
#pragma unroll
        for (int m = 0; m < NS / 64; ++m) {
            if (m == 0) tile_store(sm.t, ra);
            tile_store(sm.t + PT, rf);
            __syncthreads();
            if (m + 1 < NS / 64) {
                state(h, 64 * (m + 1));
            } else if (h + 1 < h1) {
                tile_load(ra, rows + (size_t)(h + 1) * 64, HP);
                state(h + 1, 0);
            }
            acc.zero();
            tile_mma<PT, 3, false, true, AGAIN>(acc, sm.t, sm.t + PT);
#pragma unroll
            for (int half = 0; half < 2; ++half)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float2 a = __fmul2_rn(make_float2(sc[half], sc[half]), acc.get(j, half));
                    tot[m][half][j] = __fadd2_rn(tot[m][half][j], a);
                    if (isC) {
                        const float2 cv = ld2f(Cb + (size_t)(rt * 64 + acc_row(half)) * GN + m * 64 + acc_col(j));
                        rho2[half] += cv.x * a.x + cv.y * a.y;
                    }
                }
            if (isC && m + 1 == NS / 64) {
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const float v = sum_quad(rho2[half]);
                    if ((lane & 3) == 0) sm.red[tid >> 7][acc_row(half)] = v;
                }
            }
            if (!AGAIN && h + 1 == h1) {
                bool nan = false;
#pragma unroll
                for (int j = 0; j < 4; ++j) nan |= isnan(tot[m][0][j].x) || isnan(tot[m][0][j].y) || isnan(tot[m][1][j].x) || isnan(tot[m][1][j].y);
                if (nan) sm.again = 1;
            }
            __syncthreads();
        }
        if (isC && tid < 64) p.rho2[vo + rt * 64 + tid] = sm.red[0][tid] + sm.red[1][tid];
    }
#pragma unroll
    for (int m = 0; m < NS / 64; ++m) {
        float *out = slice(rt * 64, isC ? nrt + 1 : nrt + 2, m * 64);
#pragma unroll
        for (int half = 0; half < 2; ++half)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                *reinterpret_cast<float2 *>(out + (size_t)acc_row(half) * slice_stride + acc_col(j)) = tot[m][half][j];
    }
    return !AGAIN && sm.again;
}

// The large kernel of the backward: tiles of dx, and the partial slices of dB and dC.  Per (chunk, head range):
//   causal tile pair (tt, ts): W_h = (dy_tt x_ts^T) o mask per head, rho / psi partial sums of W_h o CB, head sum of W_h; then
//                  slices dC[tt] = Wsum B_ts and dB[ts] = Wsum^T C_tt
//   inter dC, tile tt : sum_h e^{cs_t} dy_t H_in (and rho2 per head);  inter dB, tile ts : sum_h dt_s e^{cs_last-cs_s} x_s Gout
// A row of tile r has dC slots for ts <= r and dB slots for tt >= r, so the two share Q/64 + 3 slots per head range: dC by ts, dB by
// tt + 1, then the inter-chunk terms of both.
// Two CTAs per SM: at three, 80 registers spill too much (bf16, 4096 steps of 24 heads, N = 128, chunks of 64, forward + backward: 612 us at three,
// 521 at two; N = 64, states made in their readers, 385 and 352; with state passes, the backward: 2 x 8192 steps of 32 heads 758 and 750, 16384 of
// 24, chunks of 256, 682 and 670, 4 x 8192 of 32 1528 and 1503; at most 0.5 % the other way, 16384 of 24, chunks of 128).
template <typename T, int NS, bool READER, bool AGAIN>
__device__ __forceinline__ bool simt_bwd(const SegParams &p, int n_dx, const StatePass &pass, int n_pass) {
    SimtSmem<T> &sm = simt_smem<T>();
    const int nrt = p.Q >> 6, n_bc = (int)gridDim.x - n_dx - n_pass;
    int id = blockIdx.x;
    if (READER && id >= n_bc + n_dx) {
        pdl_wait();
        pass_along<true>(p, pass, sm.red[0], id - n_bc - n_dx);
        return false;
    }
    if (id < n_bc) return simt_dbdc<T, NS, READER, AGAIN>(p, sm, id);
    id -= n_bc;
    const int rt = id & (nrt - 1), bch = id >> (nrt >> 1), bc = divide_by(bch, p.H, p.inv_H), h = bch - bc * p.H,
              b = divide_by(bc, p.nc, p.inv_nc), c = bc - b * p.nc;
    return simt_row_tile<T, NS, true, true, READER, AGAIN>(p, sm, c, rt, h, b);
}
template <typename T, int NS, bool READER>
__global__ void __launch_bounds__(256, 2)
k_simt_bwd(const __grid_constant__ SegParams p, int n_dx, const __grid_constant__ StatePass pass, int n_pass) {
    pdl_launch_dependents();
    if (simt_bwd<T, NS, READER, false>(p, n_dx, pass, n_pass)) simt_bwd<T, NS, READER, true>(p, n_dx, pass, n_pass);
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
        // split path: per head range, of a row of tile rt, dC slots 0 .. rt, dB slots rt + 1 .. tiles, then the inter-chunk terms
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
// The second pass over the next segment's sums as a function: fp32, where the launch takes 211 us a pass instead of 194 with it in line
// (2 x 4096 steps of 24 heads); bf16 has it in line (159 us, as a function 173; 2 x 8192 steps of 32 heads)
template <typename T, int NS> __device__ __noinline__ void simt_sums_call(const SegParams &p) {
    simt_sums<T, NS, true>(p, simt_smem<T>(), blockIdx.x, true);
}
// split path: the same with the sums of the next segment (to the left) in front, which share no scratch with it but the step
// sizes, of which there are two copies.
template <typename T, int NS>
__global__ void __launch_bounds__(256, SimtSmem<T>::CTAS)
k_simt_tail(const __grid_constant__ SegParams p, const __grid_constant__ SegParams nx, int n_next, int nfin) {
    SimtSmem<T> &sm = simt_smem<T>();
    pdl_launch_dependents();
    const int id = (int)blockIdx.x - n_next;
    if (id < 0) {
        if (simt_sums<T, NS, false>(nx, sm, blockIdx.x, true)) {
            if constexpr (SplitParts<T>::n > 1) simt_sums_call<T, NS>(nx);
            else simt_sums<T, NS, true>(nx, sm, blockIdx.x, true);
        }
        return;
    }
    pdl_wait();
    if (id < nfin) bwd_finish<false>(p, reinterpret_cast<float *>(sm.t), id);
    else reduce_dbdc<T, false>(p, id - nfin);
}
// The same with the finishing steps first in the code, for bf16 with N = 64 and chunks of 128 and 256: behind the two bodies of the sums, which
// leave the registers short, they take longer (36 us a launch of 7936 steps of 8 heads in 8 groups, 26 behind one body), and ahead of them
// the sums do, the larger part where chunks are short.  Backward, us, finishing steps first and last: chunks of 256 (16384 steps of 24 heads) 638
// and 671, (8192 of 32) 484 and 500, (7936 of 8 in 8 groups) 347 and 354; of 128 (16384 of 24) 656 and 678; of 64 (8192 of 32 in 4 groups) 474 and
// 449, (11456 of 24 in 8) 580 and 562.  N = 128: chunks of 128 (16384 of 24 in 4 groups) 980 and 988, (of 32) 1147 and 1142, of 64 (5632 of 32) 500
// and 487.  fp32, where the second body is a function: 442 and 440 (4096 of 24, N = 128).
template <typename T, int NS>
__global__ void __launch_bounds__(256, SimtSmem<T>::CTAS)
k_simt_tail_ahead(const __grid_constant__ SegParams p, const __grid_constant__ SegParams nx, int n_next, int nfin) {
    SimtSmem<T> &sm = simt_smem<T>();
    pdl_launch_dependents();
    const int id = (int)blockIdx.x - n_next;
    if (id >= 0) {
        pdl_wait();
        if (id < nfin) bwd_finish<false>(p, reinterpret_cast<float *>(sm.t), id);
        else reduce_dbdc<T, false>(p, id - nfin);
        return;
    }
    if (simt_sums<T, NS, false>(nx, sm, blockIdx.x, true)) simt_sums<T, NS, true>(nx, sm, blockIdx.x, true);
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

template <auto K, typename T, typename... Args> static cudaError_t simt_start(bool first, int ctas, cudaStream_t st, const SegParams &p, Args &&...args) {
    const cudaError_t e = allow_smem<K>((int)sizeof(SimtSmem<T>));
    if (e != cudaSuccess) return e;
    return launch_as(!first, K, dim3(ctas), dim3(256), sizeof(SimtSmem<T>), st, p, args...);
}
template <typename T, int NS>
static cudaError_t simt_launch(const SegParams &p, const SegParams *next, const StatePass *pass, int what, cudaStream_t st) {
    const int nrt = p.Q / 64, npair = nrt * (nrt + 1) / 2, n_pass = pass ? p.P * p.N / 1024 * p.H * p.B : 0;
    const StatePass none = {};
    switch (what) {
        case SIMT_SUMS:
        case SIMT_SUMS_GRAD: {
            const bool grads = what == SIMT_SUMS_GRAD;
            return simt_start<k_simt_sums<T, NS>, T>(p.first, simt_n_sums<NS>(p, grads), st, p, grads);
        }
        case SIMT_Y: {
            const int n_next = next ? simt_n_sums<NS>(*next, false) : 0, n = p.nc * nrt * p.H * p.B + n_next + n_pass;
            if (!p.cbt) return simt_start<k_simt_y<T, NS, false, false>, T>(false, n, st, p, p, 0, none, 0);      // never with `next` or `pass`
            if (pass) return simt_start<k_simt_y<T, NS, true, true>, T>(false, n, st, p, next ? *next : p, n_next, *pass, n_pass);
            return simt_start<k_simt_y<T, NS, true, false>, T>(false, n, st, p, next ? *next : p, n_next, none, 0);
        }
        case SIMT_TAIL: {
            const int nfin = tail_finish_ctas(p), n_next = simt_n_sums<NS>(*next, true);
            const int n = n_next + nfin + tail_reduce_ctas(p);
            if constexpr (SplitParts<T>::n == 1 && NS == 64)
                if (p.Q > 64) return simt_start<k_simt_tail_ahead<T, NS>, T>(false, n, st, p, *next, n_next, nfin);
            return simt_start<k_simt_tail<T, NS>, T>(false, n, st, p, *next, n_next, nfin);
        }
        default: {
            const int n_dx = p.nc * nrt * p.H * p.B, n_bc = p.nc * (npair + 2 * nrt) * (p.nsl / (nrt + 3)) * p.G * p.B;
            if (pass) return simt_start<k_simt_bwd<T, NS, true>, T>(false, n_bc + n_dx + n_pass, st, p, n_dx, *pass, n_pass);
            return simt_start<k_simt_bwd<T, NS, false>, T>(false, n_bc + n_dx, st, p, n_dx, none, 0);
        }
    }
}
cudaError_t launch_simt(const SegParams &p, const SegParams *next, const StatePass *pass, int dtype, int what, cudaStream_t st) {
    if (dtype == SSD_DTYPE_F32) return p.N == 64 ? simt_launch<float, 64>(p, next, pass, what, st) : simt_launch<float, 128>(p, next, pass, what, st);
    return p.N == 64 ? simt_launch<__nv_bfloat16, 64>(p, next, pass, what, st) : simt_launch<__nv_bfloat16, 128>(p, next, pass, what, st);
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
