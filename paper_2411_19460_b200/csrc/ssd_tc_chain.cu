// The state chain of a segment on the tensor cores (bf16 I/O, P = 64): chunk sums and the recurrence over the chunks
// in one kernel.  Blocks of T = 128 steps; cs = inclusive cumsum of dt*A inside the block.
//
//   CHAIN_FWD: H_{c+1} = e^{cs_last} H_c + sum_s e^{cs_last-cs_s} dt_s x_s B_s^T     (also makes cs and dt head-major)
//   CHAIN_BWD: G_{c-1} = e^{cs_last} G_c + sum_t e^{cs_t} dy_t C_t^T                 (G_c: gradient leaving block c)
//              rho2_t  = e^{cs_t} dy_t . (H_in C_t),   <G,H> partials = e^{cs_last} <G_c, H_in,c>
//
// rho2 goes into ddt and dA by suffix sums, so its dy rows are the ones before scaling and rounding: a product of their own ahead
// of the block's sum, and the scaling warps wait until the rows have been read.  With the scaled rows ddt was 4 to 10 % further
// from the exact one than with blocks of 256 steps; the order costs the backward 2 us of 51.6 (4096 steps of 80 heads).
//
// One CTA owns one (batch, head), or in the forward two heads of a group, and walks the segment's blocks.  A block's sum does not
// depend on the carried state, so it is made by tcgen05 one block ahead; the carry (N x 64 fp32) never leaves the registers of the eight worker warps:
// what is written per block is its bf16 copy, the operand of the large kernels, 16 KB, where separate kernels for the
// sums and the recurrence moved 32 KB of fp32 sums out and in again on top.  States are kept transposed here, [N][64], so
// that a thread's slice (one n, 32 p) is contiguous and leaves through a swizzled tile by one TMA store per warp.
//   warp 0 producer (TMA) | warp 1 MMA issuer | warps 2, 3 records (CHAIN_FWD, alternate blocks) | warps 4..11 scale the rows |
//   warps 12..19 carry | warps 20..23 rho2 (CHAIN_BWD)
// Bound by the chain's latency on as many SMs as there are heads: a step takes 0.8 us (backward 1.4), most of it the carry warps'
// pack, proxy fence and store.  Storing the state with ordinary 32-byte stores instead (32 lines per warp instruction) made 24
// heads 9 % slower, sixteen carry warps of half the width 2 %.  4096 steps of 80 heads: 38 and 54 us, where chunk sums,
// state-gradient sums and the two passes took 28 + 12 and 37 + 24 us of the whole GPU and the large kernels now run beside it.
#include "ssd_internal.h"
#include "ssd_sm100.cuh"

namespace ssd {

using namespace sm100;

namespace {

// heads per CTA: one, or in the forward two of the same group, which then share the block's B rows and a product of N = 128
__host__ __device__ constexpr int ch_rec_warps(int heads) { return heads == 2 ? 4 : 2; }
__host__ __device__ constexpr int ch_threads(int mode, int heads) { return 32 * (2 + ch_rec_warps(heads) + 8 + 8 * heads + (mode ? 4 : 0)); }
constexpr int CH_T = kTcBlock, NS = kTcState;
__host__ __device__ constexpr int ch_stages(int mode, int heads) { return mode || heads == 2 ? 3 : 4; }
// CHAIN_FWD: vector buffers per head (weights of 128 rows + the block's decay); for two heads the weights' bf16 pairs are packed
// (a buffer belongs to one record warp: a warp that took buffers in turn with others could wait for a phase two ahead of the
// barrier's and pass at once, so their number is a multiple of the head's record warps)
__host__ __device__ constexpr int ch_vec(int heads) { return heads == 2 ? 2 : 4; }
__host__ __device__ constexpr int ch_vec_floats(int heads) { return heads == 2 ? 132 : 260; }
constexpr float kLog2eC = 1.4426950408889634f;
constexpr int CH_AHEAD = 4;               // L2 prefetch distance in blocks beyond the staged ones

// stage: V (B or C rows) N/64 x 16 KB | X (x or dy rows) 16 KB per head | CHAIN_BWD: H_in^T, N rows of 128 B | row scales 1 KB, decay 16 B
__host__ __device__ constexpr uint32_t ch_stage_bytes(int mode, int heads) {
    return (uint32_t)NS * 256 + (uint32_t)heads * 16384 + (mode ? (uint32_t)NS * 128 + 2048 : 0);
}
__host__ __device__ constexpr uint32_t ch_off_vec(int mode, int heads) {
    return ch_stages(mode, heads) * ch_stage_bytes(mode, heads) + heads * 8 * 2048;
}
__host__ __device__ constexpr uint32_t ch_off_bar(int mode, int heads) {
    return ch_off_vec(mode, heads) + (mode ? 0 : heads * ch_vec(heads) * ch_vec_floats(heads) * 4);
}
// for the alignment of the stages: two heads leave no room for all of 1 KB, but no static shared memory is in front of them
__host__ __device__ constexpr uint32_t ch_slack(int heads) { return heads == 2 ? 512 : 1024; }
__host__ __device__ constexpr uint32_t ch_smem(int mode, int heads) { return ch_off_bar(mode, heads) + 256 + ch_slack(heads); }

__device__ __forceinline__ float ex2c(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack2c(float a, float b) {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&v);
}
__device__ __forceinline__ float2 unpack2c(uint32_t w) { return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w)); }

}  // namespace

template <int MODE, int HEADS>
__global__ void __launch_bounds__(ch_threads(MODE, HEADS), 1)
k_chain_tc(SegParams p, const float *init, long long init_bs, float *bnd_out, long long bnd_bs, float *carry_out, float *final_out,
           const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmH,
           const __grid_constant__ CUtensorMap tmOut) {
    constexpr bool BWD = MODE == CHAIN_BWD;
    static_assert(!BWD || HEADS == 1, "the backward has a head per CTA");
    constexpr int CH_STAGES = ch_stages(MODE, HEADS), CH_VEC = ch_vec(HEADS), VEC_FLOATS = ch_vec_floats(HEADS), DECAY_AT = VEC_FLOATS - 4;
    static_assert(CH_VEC % (ch_rec_warps(HEADS) / HEADS) == 0, "a vector buffer belongs to one record warp");
    constexpr int SCALE0 = 2 + ch_rec_warps(HEADS), CARRY0 = SCALE0 + 8, RHO0 = CARRY0 + 8 * HEADS;      // first warps of the roles
    constexpr uint32_t STAGE = ch_stage_bytes(MODE, HEADS), OFF_X = NS * 256, OFF_H = OFF_X + HEADS * 16384, OFF_W = OFF_H + NS * 128;
    constexpr uint32_t OFF_OUT = CH_STAGES * STAGE, OFF_VEC = ch_off_vec(MODE, HEADS), OFF_BAR = ch_off_bar(MODE, HEADS);
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    if ((uint32_t)(smem - smem_raw) > ch_slack(HEADS)) {        // the same for every CTA; not reached
        if (threadIdx.x == 0) *p.status = 1u;
        return;
    }
    uint64_t *const full = reinterpret_cast<uint64_t *>(smem + OFF_BAR), *const scaled = full + CH_STAGES, *const empty = scaled + CH_STAGES;
    uint64_t *const mdone = empty + CH_STAGES, *const dempty = mdone + 2, *const vfull = dempty + 2, *const vempty = vfull + HEADS * CH_VEC;
    uint64_t *const vfirst = vempty + HEADS * CH_VEC;        // CHAIN_FWD: the first record is made; completed once and never again
    uint32_t *const words = reinterpret_cast<uint32_t *>(vfirst + 1);
    // CHAIN_BWD has no vector buffers; in their barriers' place: H_in C made, read; the stage's rows read for rho2
    uint64_t *const ydone = vfull, *const yempty = vfull + 2, *const rowread = vempty;
    static_assert((3 * CH_STAGES + 5 + 2 * HEADS * CH_VEC) * 8 + 8 <= 256, "barriers");

    const int h0 = blockIdx.x * HEADS, b = blockIdx.y, g = h0 / p.hpg, nc = p.nc;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (!BWD && p.first && blockIdx.x == 0 && b == 0 && tid < 64) p.status[tid] = 0u;
    auto chunk_of = [&](int i) { return BWD ? nc - 1 - i : i; };
    if (tid == 0) {
        for (int i = 0; i < CH_STAGES; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&scaled[i], 8);
            mbar_init(&empty[i], BWD ? 8 : 1);     // BWD: the carry warps read the stage last; FWD: the MMAs do
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&mdone[i], 1);
            mbar_init(&dempty[i], 8 * HEADS);
        }
        for (int i = 0; i < HEADS * CH_VEC; ++i) {
            mbar_init(&vfull[i], BWD && i >= 2 ? 4 : 1);
            mbar_init(&vempty[i], BWD ? 4 : 8);    // the carry warps, which read the decay last
        }
        mbar_init(vfirst, 1);
        words[1] = 0;
        fence_barrier_init();
    }
    constexpr uint32_t NCOL = BWD ? 256 : 128 * HEADS;     // block sum, double buffered; BWD: H_in C likewise
    if (warp == 0) tmem_alloc(&words[0], NCOL);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    // What the kernel before this one in the stream may still write, or still read where this one writes, is waited for in the
    // roles that touch it; x, dt, B, C and dy are older than the call, whose first launch is an ordinary one, so the
    // first blocks are loaded and scaled under its end.
    const uint32_t tm = words[0];
    volatile uint32_t *abortp = &words[1];

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        if (elect_one()) {
            auto load_inputs = [&](int i) {
                const int st = i % CH_STAGES, tok = p.t0 + chunk_of(i) * CH_T;
                unsigned char *sb = smem + st * STAGE;
                mbar_arrive_expect_tx(&full[st], BWD ? STAGE - 1024 + 16 : STAGE);
#pragma unroll
                for (int k = 0; k < HEADS; ++k) tma_load_3d(sb + OFF_X + k * 16384, &tmX, &full[st], (h0 + k) * 64, tok, b);
#pragma unroll
                for (int nh = 0; nh < NS / 64; ++nh) tma_load_3d(sb + nh * 16384, &tmV, &full[st], g * NS + nh * 64, tok, b);
            };
            const int ahead = nc < CH_STAGES ? nc : CH_STAGES;
            // The first step sizes would arrive behind all the stages of all CTAs (15.7 MB with 80 heads: the first block scaled 9100 cycles
            // after the start, now 7000) and everything waits for them: the later stages wait for the first record instead.  Forward
            // of one segment, 80 heads: 4096 steps 68.8 -> 67.5 us, 16384 in 8 groups 226 -> 218; 24 heads the same.  (Not vfull[0]: nothing
            // holds its next phase back until this thread has looked, and the one after that needs blocks that this thread loads.)
            for (int i = 0; i < ahead; ++i) {
                if (!BWD && i == 1) mbar_wait(vfirst, 0, abortp, p.status);
                load_inputs(i);
            }
            if (BWD) pdl_wait();                   // the records and states of the forward chain
            for (int i = 0; i < nc; ++i) {
                const int st = i % CH_STAGES, c = chunk_of(i);
                unsigned char *sb = smem + st * STAGE;
                if (i >= CH_STAGES) {
                    mbar_wait(&empty[st], (i / CH_STAGES - 1) & 1, abortp, p.status);
                    load_inputs(i);
                }
                // the next launch's first loads and products take about as long as the blocks that are left here; much earlier,
                // and its CTAs would hold SMs idle
                if (i + CH_STAGES + 1 == nc) pdl_launch_dependents();
                if (BWD) {
                    const float *rec = p.rec + (((size_t)b * p.H + h0) * p.ncs + c) * REC_FLOATS;
                    tma_load_3d(sb + OFF_H, &tmH, &full[st], 0, ((b * p.ncs + c) * p.H + h0) * NS, 0);
                    bulk_load(sb + OFF_W, rec + REC_OC, 1024, &full[st]);
                    bulk_load(sb + OFF_W + 1024, rec + REC_DECAY, 16, &full[st]);
                }
                if (i + CH_AHEAD < nc)
#pragma unroll
                    for (int k = 0; k < HEADS; ++k) tma_prefetch_3d(&tmX, (h0 + k) * 64, p.t0 + chunk_of(i + CH_AHEAD) * CH_T, b);
            }
            if (nc <= CH_STAGES) pdl_launch_dependents();
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (elect_one()) {
            const uint32_t idD = umma_idesc_bf16(128, 64 * HEADS, true, true), idY = umma_idesc_bf16(128, 64, false, true);
            for (int i = 0; i < nc; ++i) {
                const int st = i % CH_STAGES, bf = i & 1;
                const uint32_t sb = smem_u32(smem + st * STAGE);
                // The sum as D[n][p]: V rows MN-major along n, X rows MN-major along p
                const uint64_t dV = umma_desc_sw128(sb, 16384, 1024), dX = umma_desc_sw128(sb + OFF_X, 16384, 1024);
                const uint32_t loV = (uint32_t)dV, hiM = (uint32_t)(dV >> 32), loX = (uint32_t)dX, hiX = (uint32_t)(dX >> 32);
                mbar_wait(&full[st], (i / CH_STAGES) & 1, abortp, p.status);
                if (BWD) {   // Y[t][p] = sum_n C[t][n] H_in[p][n], for rho2
                    const uint64_t dC = umma_desc_sw128(sb, 16, 1024), dH = umma_desc_sw128(sb + OFF_H, 8192, 1024);
                    const uint32_t loC = (uint32_t)dC, hiC = (uint32_t)(dC >> 32), loH = (uint32_t)dH, hiH = (uint32_t)(dH >> 32);
                    if (i >= 2) mbar_wait(&yempty[bf], ((i >> 1) - 1) & 1, abortp, p.status);
                    tc_fence_after_sync();
#pragma unroll
                    for (int k = 0; k < NS / 16; ++k) {
                        const uint64_t ad = umma_desc_words(loC + (k >> 2) * 1024 + (k & 3) * 2, hiC), bd = umma_desc_words(loH + k * 128, hiH);
                        if (k == 0) umma_bf16_fixed<false>(tm + 128 + bf * 64, ad, bd, idY);
                        else umma_bf16_fixed<true>(tm + 128 + bf * 64, ad, bd, idY);
                    }
                    umma_commit(&ydone[bf]);
                }
                mbar_wait(&scaled[st], (i / CH_STAGES) & 1, abortp, p.status);
                if (i >= 2) mbar_wait(&dempty[bf], ((i >> 1) - 1) & 1, abortp, p.status);
                tc_fence_after_sync();
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const uint64_t ad = umma_desc_words(loV + k * 128, hiM), bd = umma_desc_words(loX + k * 128, hiX);
                    if (k == 0) umma_bf16_fixed<false>(tm + bf * 64 * HEADS, ad, bd, idD);
                    else umma_bf16_fixed<true>(tm + bf * 64 * HEADS, ad, bd, idD);
                }
                if (!BWD) umma_commit(&empty[st]);
                umma_commit(&mdone[bf]);
            }
        }
    } else if (warp < SCALE0) {
        // ------------------------------------------------------------ records, a lane owns four consecutive steps
        if (!BWD) {
            const int first = (warp - 2) & 1, hl = (warp - 2) >> 1, h = h0 + hl;
            float *vec = reinterpret_cast<float *>(smem + OFF_VEC) + hl * CH_VEC * VEC_FLOATS;
            const float Ah = __ldg(p.A + h);
            // fetched four of this warp's blocks ahead: the strided step sizes take longer to arrive than a block takes
            auto fetch = [&](int i, float4 &v) {
                const float *d = p.dt + (size_t)b * p.dt_bs + (size_t)(p.t0 + i * CH_T + lane * 4) * p.H + h;
                v = make_float4(__ldg(d), __ldg(d + p.H), __ldg(d + 2 * (size_t)p.H), __ldg(d + 3 * (size_t)p.H));
            };
            float4 ring[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (first + 2 * k < nc) fetch(first + 2 * k, ring[k]);
            for (int i0 = first; i0 < nc; i0 += 8)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = i0 + 2 * k;
                if (i >= nc) break;
                const int vb = i % CH_VEC, vbar = hl * CH_VEC + vb;
                const float4 dt4 = ring[k];
                if (i + 8 < nc) fetch(i + 8, ring[k]);
                const float d[4] = {dt4.x, dt4.y, dt4.z, dt4.w};
                float cs[4], run = 0.f;
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    run += d[m] * Ah;
                    cs[m] = run;
                }
                float incl = run;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const float t = __shfl_up_sync(0xffffffffu, incl, off);
                    if (lane >= off) incl += t;
                }
                float excl = __shfl_up_sync(0xffffffffu, incl, 1);
                if (lane == 0) excl = 0.f;
#pragma unroll
                for (int m = 0; m < 4; ++m) cs[m] += excl;
                const float decay = expf(__shfl_sync(0xffffffffu, cs[3], 31));
#pragma unroll
                for (int m = 0; m < 4; ++m) cs[m] *= kLog2eC;
                const float last = __shfl_sync(0xffffffffu, cs[3], 31);
                float w[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) w[m] = ex2c(fminf(last - cs[m], 0.f)) * d[m];
                if (i >= CH_VEC) mbar_wait(&vempty[vbar], (i / CH_VEC - 1) & 1, abortp, p.status);
                float *v = vec + vb * VEC_FLOATS;
                RowScale ob[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) ob[m] = row_scale(w[m]);
                auto put_scales = [&](float *dst, const RowScale (&sc)[4]) {
                    uint4 *d4 = reinterpret_cast<uint4 *>(dst) + lane * 2;
                    d4[0] = make_uint4(sc[0].hi, sc[0].lo, sc[1].hi, sc[1].lo);
                    d4[1] = make_uint4(sc[2].hi, sc[2].lo, sc[3].hi, sc[3].lo);
                };
                if (HEADS == 2)
                    *reinterpret_cast<uint4 *>(v + lane * 4) = make_uint4(__byte_perm(ob[0].hi, ob[0].lo, 0x5410), __byte_perm(ob[1].hi, ob[1].lo, 0x5410),
                                                                          __byte_perm(ob[2].hi, ob[2].lo, 0x5410), __byte_perm(ob[3].hi, ob[3].lo, 0x5410));
                else
                    put_scales(v, ob);
                if (lane == 0) v[DECAY_AT] = decay;
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&vfull[vbar]);
                    if (i == 0 && hl == 0) mbar_arrive(vfirst);
                }
                if (i == first) pdl_wait();        // the earlier kernels have read what this copy of the records held
                const float lo = __shfl_sync(0xffffffffu, cs[3], lane | 7), hi = __shfl_sync(0xffffffffu, cs[0], lane & ~7);
                const float bi = __shfl_sync(0xffffffffu, cs[0], ((lane >> 2) & 3) * 8), bj = __shfl_sync(0xffffffffu, cs[3], (lane & 3) * 8 + 7);
                float *rec = p.rec + (((size_t)b * p.H + h) * p.ncs + i) * REC_FLOATS;
                auto put = [&](int part, float x, float y, float z, float u) {
                    *reinterpret_cast<float4 *>(rec + part + lane * 4) = make_float4(x, y, z, u);
                };
                put(REC_CFX, ex2c(cs[0] - hi), ex2c(cs[1] - hi), ex2c(cs[2] - hi), ex2c(cs[3] - hi));
                if (lane < 16) rec[REC_BLK + lane] = (lane & 3) < (lane >> 2) ? ex2c(bi - bj) : 0.f;
                else if (lane < 20) rec[REC_DECAY + lane - 16] = decay;
                put(REC_CS, cs[0], cs[1], cs[2], cs[3]);
                put(REC_DT, d[0], d[1], d[2], d[3]);
                put(REC_CF, ex2c(lo - cs[0]) * d[0], ex2c(lo - cs[1]) * d[1], ex2c(lo - cs[2]) * d[2], ex2c(lo - cs[3]) * d[3]);
                const RowScale oc[4] = {row_scale(ex2c(cs[0])), row_scale(ex2c(cs[1])), row_scale(ex2c(cs[2])), row_scale(ex2c(cs[3]))};
                put_scales(rec + REC_OC, oc);
                put_scales(rec + REC_OB, ob);
            }
        }
    } else if (warp < CARRY0) {
        // ------------------------------------------------------------ the blocks' rows times their weights, in place (a weight is
        // uniform along a row, so the swizzle does not matter)
        const int th = tid - SCALE0 * 32;
        for (int i = 0; i < nc; ++i) {
            const int st = i % CH_STAGES;
            unsigned char *sb = smem + st * STAGE;
            mbar_wait(&full[st], (i / CH_STAGES) & 1, abortp, p.status);
#pragma unroll
            for (int hl = 0; hl < HEADS; ++hl) {
                const unsigned char *w = BWD ? sb + OFF_W : smem + OFF_VEC + (hl * CH_VEC + i % CH_VEC) * VEC_FLOATS * 4;
                if (!BWD) mbar_wait(&vfull[hl * CH_VEC + i % CH_VEC], (i / CH_VEC) & 1, abortp, p.status);
                uint4 *x4 = reinterpret_cast<uint4 *>(sb + OFF_X + hl * 16384) + th;
                uint4 v[4];
                RowScale f[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    v[k] = x4[k * 256];
                    const int r = (th >> 3) + 32 * k;
                    if (HEADS == 2) {
                        const uint32_t pk = reinterpret_cast<const uint32_t *>(w)[r];
                        f[k] = {__byte_perm(pk, 0, 0x1010), __byte_perm(pk, 0, 0x3232)};
                    } else {
                        f[k] = reinterpret_cast<const RowScale *>(w)[r];
                    }
                }
                if (BWD) mbar_wait(&rowread[st], (i / CH_STAGES) & 1, abortp, p.status);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    scale8(v[k], f[k]);
                    x4[k * 256] = v[k];
                }
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&scaled[st]);
        }
    } else if (BWD && warp >= RHO0) {
        // ------------------------------------------------------------ rho2: row dot of the dy row and H_in C, t = 32 q + lane.
        // The row is read before it is scaled and rounded, its factor multiplies the sum; the product needs no scaled rows and
        // is made ahead of the block's sum.
        const int q = warp & 3, r = q * 32 + lane;
        pdl_wait();
        for (int i = 0; i < nc; ++i) {
            const int st = i % CH_STAGES, bf = i & 1, c = chunk_of(i);
            const unsigned char *sb = smem + st * STAGE, *dr = sb + OFF_X + r * 128;
            mbar_wait(&full[st], (i / CH_STAGES) & 1, abortp, p.status);
            uint4 dv[8];
#pragma unroll
            for (int ch = 0; ch < 8; ++ch) dv[ch] = *reinterpret_cast<const uint4 *>(dr + ((ch ^ (r & 7)) << 4));
            const RowScale f = reinterpret_cast<const RowScale *>(sb + OFF_W)[r];
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&rowread[st]);
            mbar_wait(&ydone[bf], (i >> 1) & 1, abortp, p.status);
            __syncwarp();
            tc_fence_after_sync();
            float2 acc = make_float2(0.f, 0.f);
#pragma unroll
            for (int part = 0; part < 4; ++part) {
                float d[16];
                tmem_ld16(tm + ((uint32_t)(q * 32) << 16) + 128 + bf * 64 + part * 16, d);
#pragma unroll
                for (int ch = 0; ch < 2; ++ch) {
                    const uint32_t *e = reinterpret_cast<const uint32_t *>(&dv[part * 2 + ch]);
#pragma unroll
                    for (int m = 0; m < 4; ++m) acc = __ffma2_rn(unpack2c(e[m]), make_float2(d[ch * 8 + 2 * m], d[ch * 8 + 2 * m + 1]), acc);
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&yempty[bf]);
            p.rho2[(((size_t)b * p.H + h0) * p.ncs + c) * CH_T + r] = row_scale_value(f) * (acc.x + acc.y);
        }
    } else {
        // ------------------------------------------------------------ carry: warp (q, half) holds state rows
        // n = 32 q + lane, columns p = 32 half ..; as rows of time, t = 32 q + lane
        const int w = (warp - CARRY0) & 7, hl = (warp - CARRY0) >> 3, h = h0 + hl;
        const int q = warp & 3, half = w >> 2;
        const uint32_t tl = tm + ((uint32_t)(q * 32) << 16) + hl * 64 + half * 32;
        const float *vec = reinterpret_cast<const float *>(smem + OFF_VEC) + hl * CH_VEC * VEC_FLOATS;
        unsigned char *stg = smem + OFF_OUT + (warp - CARRY0) * 2048, *row = stg + lane * 64;      // [32 rows][64 B], 64-byte swizzle
        const size_t so = (size_t)h * 64 * NS + (size_t)(half * 32) * NS + q * 32 + lane;
        float carry[32];
        pdl_wait();                                // the carry that the previous segment's launch left; the earlier states have been read
#pragma unroll
        for (int j = 0; j < 32; ++j) carry[j] = init ? init[(size_t)b * init_bs + so + (size_t)j * NS] : 0.f;
        if (bnd_out) {
#pragma unroll
            for (int j = 0; j < 32; ++j) bnd_out[(size_t)b * bnd_bs + so + (size_t)j * NS] = carry[j];
        }
        for (int i = 0; i < nc; ++i) {
            const int st = i % CH_STAGES, bf = i & 1, c = chunk_of(i);
            // the carried state in bf16 (H entering block c, or the gradient leaving it) on its way out while the block's sum is made
            if (lane == 0) tma_store_wait_read();
            __syncwarp();
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
                const float *a = carry + ch * 8;
                *reinterpret_cast<uint4 *>(row + ((ch ^ ((lane >> 1) & 3)) << 4)) =
                    make_uint4(pack2c(a[0], a[1]), pack2c(a[2], a[3]), pack2c(a[4], a[5]), pack2c(a[6], a[7]));
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                tma_store_3d(&tmOut, stg, half * 32, ((b * p.ncs + c) * p.H + h) * NS + q * 32, 0);
                tma_store_commit();
            }
            if (BWD) mbar_wait(&full[st], (i / CH_STAGES) & 1, abortp, p.status);      // H_in and the decay have landed
            float2 dot = make_float2(0.f, 0.f);
            if (BWD) {              // <G, H_in> over this thread's slice
                const unsigned char *hr = smem + st * STAGE + OFF_H + (q * 32 + lane) * 128;
#pragma unroll
                for (int ch = 0; ch < 4; ++ch) {
                    const uint4 hv = *reinterpret_cast<const uint4 *>(hr + (((half * 4 + ch) ^ (lane & 7)) << 4));
                    const uint32_t *e = reinterpret_cast<const uint32_t *>(&hv);
#pragma unroll
                    for (int m = 0; m < 4; ++m) dot = __ffma2_rn(make_float2(carry[ch * 8 + 2 * m], carry[ch * 8 + 2 * m + 1]), unpack2c(e[m]), dot);
                }
            }
            mbar_wait(&mdone[bf], (i >> 1) & 1, abortp, p.status);
            __syncwarp();
            tc_fence_after_sync();
            // (CHAIN_FWD: the scaling warps waited for the decay's buffer before the products could start)
            const float decay = BWD ? *reinterpret_cast<const float *>(smem + st * STAGE + OFF_W + 1024) : vec[(i % CH_VEC) * VEC_FLOATS + DECAY_AT];
            const float2 dec2 = make_float2(decay, decay);
            constexpr int PART = 32 / HEADS;          // two heads: 64 registers a thread
#pragma unroll
            for (int c0 = 0; c0 < 32; c0 += PART) {
                float d[PART];
                if constexpr (HEADS == 2) tmem_ld16(tl + bf * 64 * HEADS + c0, d);
                else tmem_ld32(tl + bf * 64, d);
#pragma unroll
                for (int j = 0; j < PART; j += 2) {
                    const float2 v = __ffma2_rn(dec2, make_float2(carry[c0 + j], carry[c0 + j + 1]), make_float2(d[j], d[j + 1]));
                    carry[c0 + j] = v.x;
                    carry[c0 + j + 1] = v.y;
                }
            }
            tc_fence_before_sync();
            if (BWD) fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&dempty[bf]);
                if (BWD) mbar_arrive(&empty[st]);
                else mbar_arrive(&vempty[hl * CH_VEC + i % CH_VEC]);
            }
            if (BWD) {
                float dt = dot.x + dot.y;
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) dt += __shfl_xor_sync(0xffffffffu, dt, off);
                if (lane == 0) p.ghdot[((((size_t)b * p.H + h) * p.ncs + c) << 4) + w] = decay * dt;
            }
        }
        if (carry_out) {
#pragma unroll
            for (int j = 0; j < 32; ++j) carry_out[(size_t)b * p.H * 64 * NS + so + (size_t)j * NS] = carry[j];
        }
        if (final_out) {
#pragma unroll
            for (int j = 0; j < 32; ++j) final_out[(size_t)b * p.H * 64 * NS + so + (size_t)j * NS] = carry[j];
        }
        if (lane == 0) tma_store_wait_all();
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after_sync();
        tmem_dealloc(tm, NCOL);
    }
}

template <int MODE, int HEADS>
static cudaError_t launch_chain(const SegParams &p, const TcMaps &m, const float *init, long long init_bs, float *bnd_out, long long bnd_bs,
                                float *carry_out, float *final_out, cudaStream_t st) {
    constexpr uint32_t smem = ch_smem(MODE, HEADS);
    static_assert(smem <= 232448, "shared memory of a CTA");
    const cudaError_t e = allow_smem<k_chain_tc<MODE, HEADS>>((int)smem);
    if (e != cudaSuccess) return e;
    const bool bwd = MODE == CHAIN_BWD;
    return launch_as(bwd || !p.first, k_chain_tc<MODE, HEADS>, dim3(p.H / HEADS, p.B), dim3(ch_threads(MODE, HEADS)), (size_t)smem, st, p, init, init_bs, bnd_out,
                      bnd_bs, carry_out, final_out, bwd ? m.dy : m.x, bwd ? m.Cm : m.Bm, m.H, bwd ? m.Gst : m.Hst);
}

cudaError_t launch_chain_fwd(const SegParams &p, const TcMaps &m, const float *init, long long init_bs, float *boundary_out, long long bnd_bs,
                             float *final_out, cudaStream_t st) {
    if (p.chain_heads == 2) return launch_chain<CHAIN_FWD, 2>(p, m, init, init_bs, boundary_out, bnd_bs, p.hcarry, final_out, st);
    return launch_chain<CHAIN_FWD, 1>(p, m, init, init_bs, boundary_out, bnd_bs, p.hcarry, final_out, st);
}
cudaError_t launch_chain_bwd(const SegParams &p, const TcMaps &m, const float *init, float *left_out, cudaStream_t st) {
    return launch_chain<CHAIN_BWD, 1>(p, m, init, (long long)p.H * 64 * NS, nullptr, 0, left_out, nullptr, st);
}

}  // namespace ssd
