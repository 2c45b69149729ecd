// Tensor-core kernel for dB and dC (bf16 I/O, P = 64, N = 128), over blocks of T = 128 steps.  Both are products of
// the same masked, per-head score tile
//     W_h[t,s] = (dy_t . x_s) e^{cs_t-cs_s} dt_s   (s <= t),
//   dC_t = sum_h [ sum_s W_h[t,s] B_s + e^{cs_t} dy_t^T H_in ]
//   dB_s = sum_h [ sum_t W_h[t,s] C_t + dt_s e^{cs_last-cs_s} x_s^T Gout ]
// and both are linear in it, so a CTA, which owns (block, group, a range of the group's heads), masks the tile once per
// head, adds it to a head sum kept in fp32 registers, and after the last head multiplies the sum, as two bf16 parts, by B
// and by C.  Per head it also forms the scalars of the decay gradient, rho_t = sum_s W[t,s] (C_t.B_s) and
// psi_s = sum_t W[t,s] (C_t.B_s): row and column sums of one fp32 matrix.  (Eq. 1 of the paper regrouped by blocks; cs =
// inclusive cumsum of dt*A inside the block.)
//
// Of the 16 32 x 32 sub-tiles of the tile ten are not above the diagonal: ten mask warps own one each for the whole CTA,
// with its part of C B^T and of the head sum in registers (32 + 32), so that a head costs a warp one tensor-memory load
// and its arithmetic.  A warp can only read the 32 tensor-memory lanes of its own quarter, so sub-tile (q, r) belongs to
// warp 4 r + q, r <= q, and the six warps in between have the other roles:
//   warp 4 producer (TMA) | warp 8 MMA issuer | warp 12 rho / psi out | warps 9, 13, 14 row scaling
// Tensor memory: two score buffers and the two accumulators, 128 columns each.  The rows of a head are scaled in place for
// the inter-block terms once its scores have been multiplied, and both terms go straight into the accumulators.
// The head sum's second part takes dB from 2.42e-3 to 1.81e-3 of the exact one and dC from 2.64e-3 to 2.36e-3 (bf16 outputs: 1.66e-3;
// 256-step blocks with one part: 2.39e-3, 2.62e-3) for 1.2 us of 76 (4096 steps of 80 heads, 64 CTAs).
// Of what it uses, shared memory (61 % of the wavefronts of a busy SM) and the scheduler that holds the four sub-tiles of row
// quarter 3 (56 % of its issue slots, 48 % on average) are nearest a limit; 16 warps leave the rest as latency.  4096 steps of 80
// heads: 77 us on 64 SMs, 94 us on 144 before, with 256-step chunks as three tiles.
#include "ssd_internal.h"
#include "ssd_sm100.cuh"

namespace ssd {

using namespace sm100;

namespace {

constexpr int GF_T = kTcBlock, NS = kTcState;
constexpr int GF_THREADS = 512;
constexpr int GF_VECS = 3;                        // record buffers; the part used, from the decays to the row scales
constexpr int GF_REC0 = REC_BLK, GF_VEC_FLOATS = REC_FLOATS - REC_BLK;

// Ring of four 32 KB slots: the block's C rows, its B rows (N/64 x 16 KB each), then one head per slot (dy rows 16 KB | x rows
// 16 KB), then C and B again for the last products | 2 x (H^T | G^T, N x 128 B), at the end the two parts of the head sum
constexpr uint32_t GF_OFF_ST = 4 * 32768;
constexpr uint32_t GF_OFF_VEC = GF_OFF_ST + 2 * 2 * (uint32_t)NS * 128;
constexpr uint32_t GF_OFF_PART = GF_OFF_VEC + GF_VECS * GF_VEC_FLOATS * 4;
constexpr uint32_t GF_SMEM = GF_OFF_PART + 2 * 1024 * 4 + 1024;

constexpr uint32_t GF_WPART = 128 * 256;          // a part of the head sum
static_assert(2 * GF_WPART <= GF_OFF_VEC - GF_OFF_ST, "the head sum in the states' place");

constexpr uint32_t TF_ACCC = 256, TF_ACCB = 384;

__device__ __forceinline__ float ex2g(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack2g(float a, float b) {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&v);
}

}  // namespace

// WHAT: BC_DC | BC_DB, or one of them (the cross-check with two launches)
template <int WHAT>
__global__ void __launch_bounds__(GF_THREADS, 1)
k_grad_bc(SegParams p, const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmDy,
          const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CUtensorMap tmH,
          const __grid_constant__ CUtensorMap tmG) {
    constexpr bool doC = (WHAT & BC_DC) != 0, doB = (WHAT & BC_DB) != 0;
    constexpr uint32_t OFF_ST = GF_OFF_ST, ST = NS * 128;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t rfull[4], rempty[4], stfull[2], stempty[2], sfull[2], sempty[2], scfull[2], stdone, wfull, accfull, vfull[GF_VECS],
        vempty[GF_VECS], pfull[2], pempty[2];
    __shared__ uint32_t tmem_base, abort_flag;

    const int nc = p.nc, nsl = p.nsl, ny = nsl * p.G;
    const int c = (int)blockIdx.x % nc, yid = ((int)blockIdx.x / nc) % ny, b = (int)blockIdx.x / (nc * ny);
    const int g = yid / nsl, sl = yid % nsl;
    const int hps = (p.hpg + nsl - 1) / nsl;
    const int h_begin = g * p.hpg + sl * hps;
    const int nheads = min(p.hpg - sl * hps, hps);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q = warp & 3, sr = warp >> 2;         // tensor-memory quarter; column sub-tile
    const uint32_t tlane = (uint32_t)(q * 32) << 16;
    const int tok0 = p.t0 + c * GF_T;
    unsigned char *vecs = smem + GF_OFF_VEC;
    auto record = [&](int vb) { return reinterpret_cast<const float *>(vecs) + vb * GF_VEC_FLOATS - GF_REC0; };
    float *parts = reinterpret_cast<float *>(smem + GF_OFF_PART);      // [head parity][rho: 4 sub-tiles x 128 | psi: 4 quarters x 128]

    if (tid == 0) {
        for (int i = 0; i < 4; ++i) {
            mbar_init(&rfull[i], 1);
            mbar_init(&rempty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&stfull[i], 1);
            mbar_init(&stempty[i], 1);
            mbar_init(&sfull[i], 1);
            mbar_init(&sempty[i], 10);
            mbar_init(&scfull[i], 3);
            mbar_init(&pfull[i], 10);
            mbar_init(&pempty[i], 1);
        }
        for (int i = 0; i < GF_VECS; ++i) {
            mbar_init(&vfull[i], 1);
            mbar_init(&vempty[i], 10 + 3);
        }
        mbar_init(&stdone, 1);
        mbar_init(&wfull, 10);
        mbar_init(&accfull, 1);
        abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 0) tmem_alloc(&tmem_base, 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    pdl_launch_dependents();
    pdl_wait();       // barriers and tensor memory are set up; everything below reads what earlier kernels wrote
    const uint32_t tm = tmem_base;
    volatile uint32_t *abortp = &abort_flag;

    if (warp == 4) {
        // ------------------------------------------------------------ producer
        if (elect_one()) {
            // entry e of the ring: 0 C, 1 B, 2 + h head h, 2 + nheads C, 3 + nheads B
            auto load_entry = [&](int e) {
                const int slot = e & 3, hi = e - 2;
                unsigned char *rb = smem + slot * 32768;
                if (e >= 4) mbar_wait(&rempty[slot], ((e >> 2) - 1) & 1, abortp, p.status);
                if (hi >= 0 && hi < nheads) {
                    mbar_arrive_expect_tx(&rfull[slot], 32768);
                    tma_load_3d(rb, &tmDy, &rfull[slot], (h_begin + hi) * 64, tok0, b);
                    tma_load_3d(rb + 16384, &tmX, &rfull[slot], (h_begin + hi) * 64, tok0, b);
                } else {
                    mbar_arrive_expect_tx(&rfull[slot], NS * 256);
                    if (e == 0 || hi == nheads) {
#pragma unroll
                        for (int nh = 0; nh < NS / 64; ++nh) tma_load_3d(rb + nh * 16384, &tmC, &rfull[slot], g * NS + nh * 64, tok0, b);
                    } else {
#pragma unroll
                        for (int nh = 0; nh < NS / 64; ++nh) tma_load_3d(rb + nh * 16384, &tmB, &rfull[slot], g * NS + nh * 64, tok0, b);
                    }
                }
            };
            const int strow = (b * p.ncs + c) * p.H;
            load_entry(0);
            load_entry(1);
            load_entry(2);
            for (int hi = 0; hi < nheads; ++hi) {      // rows run one head ahead of the states, which have two buffers
                const int bf = hi & 1;
                unsigned char *sb = smem + OFF_ST + bf * 2 * ST;
                const int vb = hi % GF_VECS;
                if (hi >= GF_VECS) mbar_wait(&vempty[vb], (hi / GF_VECS - 1) & 1, abortp, p.status);
                mbar_arrive_expect_tx(&vfull[vb], GF_VEC_FLOATS * 4);
                bulk_load(vecs + vb * GF_VEC_FLOATS * 4, p.rec + (((size_t)b * p.H + h_begin + hi) * p.ncs + c) * REC_FLOATS + GF_REC0, GF_VEC_FLOATS * 4,
                          &vfull[vb]);
                if (hi >= 2) mbar_wait(&stempty[bf], ((hi >> 1) - 1) & 1, abortp, p.status);
                mbar_arrive_expect_tx(&stfull[bf], (doC ? ST : 0) + (doB ? ST : 0));
                if (doC) tma_load_3d(sb, &tmH, &stfull[bf], 0, (strow + h_begin + hi) * NS, 0);
                if (doB) tma_load_3d(sb + ST, &tmG, &stfull[bf], 0, (strow + h_begin + hi) * NS, 0);
                load_entry(3 + hi);
            }
            load_entry(3 + nheads);
        }
    } else if (warp == 8) {
        // ------------------------------------------------------------ MMA issuer
        if (elect_one()) {
            const uint32_t idS = umma_idesc_bf16(128, 128, false, false);      // C B^T and the scores: both operands K-major
            const uint32_t idI = umma_idesc_bf16(128, NS, false, false);       // scaled rows x state (rows n of the transposed state)
            const uint32_t idC = umma_idesc_bf16(128, NS, false, true), idB = umma_idesc_bf16(128, NS, true, true);
            const uint32_t s0 = smem_u32(smem);
            // descriptors as (low word, high word); every offset below is a constant in 16-byte units
            const uint64_t dCk = umma_desc_sw128(s0, 16, 1024), dCm = umma_desc_sw128(s0, 16384, 1024);
            const uint32_t loC = (uint32_t)dCk, hiK = (uint32_t)(dCk >> 32), loCm = (uint32_t)dCm, hiM = (uint32_t)(dCm >> 32);
            const uint32_t loB = loC + 2048, loSt = loC + OFF_ST / 16, loWk = loSt, loWm = loCm + OFF_ST / 16;
            mbar_wait(&rfull[0], 0, abortp, p.status);
            mbar_wait(&rfull[1], 0, abortp, p.status);
            tc_fence_after_sync();
#pragma unroll
            for (int k = 0; k < NS / 16; ++k) {        // C B^T of the tile, in score buffer 0
                const uint32_t o = (k >> 2) * 1024 + (k & 3) * 2;
                if (k == 0) umma_bf16_fixed<false>(tm, umma_desc_words(loC + o, hiK), umma_desc_words(loB + o, hiK), idS);
                else umma_bf16_fixed<true>(tm, umma_desc_words(loC + o, hiK), umma_desc_words(loB + o, hiK), idS);
            }
            umma_commit(&sfull[0]);
            umma_commit(&rempty[0]);
            umma_commit(&rempty[1]);
            auto scores = [&](int hi) {                // use hi + 1 of the score buffers
                const int u = hi + 1, bf = u & 1, e = hi + 2, slot = e & 3;
                mbar_wait(&rfull[slot], (e >> 2) & 1, abortp, p.status);
                if (u >= 2) mbar_wait(&sempty[bf], ((u >> 1) - 1) & 1, abortp, p.status);
                tc_fence_after_sync();
                const uint32_t a = loC + slot * 2048, x = a + 1024, d = tm + bf * 128;
                umma_bf16_fixed<false>(d, umma_desc_words(a, hiK), umma_desc_words(x, hiK), idS);
#pragma unroll
                for (int k = 1; k < 4; ++k) umma_bf16_fixed<true>(d, umma_desc_words(a + k * 2, hiK), umma_desc_words(x + k * 2, hiK), idS);
                umma_commit(&sfull[bf]);
            };
            scores(0);
            for (int hi = 0; hi < nheads; ++hi) {
                const int bf = hi & 1;
                if (hi + 1 < nheads) scores(hi + 1);
                mbar_wait(&stfull[bf], (hi >> 1) & 1, abortp, p.status);
                mbar_wait(&scfull[bf], (hi >> 1) & 1, abortp, p.status);
                tc_fence_after_sync();
                const int slot = (hi + 2) & 3;
                const uint32_t a = loC + slot * 2048, st = loSt + bf * (2 * ST / 16);
                auto inter = [&](uint32_t acc, uint32_t rows, uint32_t state) {
                    if (hi == 0) umma_bf16_fixed<false>(acc, umma_desc_words(rows, hiK), umma_desc_words(state, hiK), idI);
                    else umma_bf16_fixed<true>(acc, umma_desc_words(rows, hiK), umma_desc_words(state, hiK), idI);
#pragma unroll
                    for (int k = 1; k < 4; ++k) umma_bf16_fixed<true>(acc, umma_desc_words(rows + k * 2, hiK), umma_desc_words(state + k * 2, hiK), idI);
                };
                if (doC) inter(tm + TF_ACCC, a, st);
                if (doB) inter(tm + TF_ACCB, a + 1024, st + ST / 16);
                umma_commit(&rempty[slot]);
                umma_commit(&stempty[bf]);
            }
            umma_commit(&stdone);     // nothing reads the states any more: the head sum may take their place
            const int ec = 2 + nheads, eb = 3 + nheads;
            const uint32_t loCe = loCm + (ec & 3) * 2048, loBe = loCm + (eb & 3) * 2048;
            mbar_wait(&rfull[ec & 3], (ec >> 2) & 1, abortp, p.status);
            mbar_wait(&rfull[eb & 3], (eb >> 2) & 1, abortp, p.status);
            mbar_wait(&wfull, 0, abortp, p.status);
            tc_fence_after_sync();
#pragma unroll
            for (int part = 0; part < 2; ++part) {
                const uint32_t o = part * (GF_WPART / 16);
#pragma unroll
                for (int k = 0; k < 8; ++k)       // dC += Wsum B, K = s
                    if (doC)
                        umma_bf16_fixed<true>(tm + TF_ACCC, umma_desc_words(loWk + o + (k >> 2) * 1024 + (k & 3) * 2, hiK),
                                              umma_desc_words(loBe + k * 128, hiM), idC);
#pragma unroll
                for (int k = 0; k < 8; ++k)       // dB += Wsum^T C, K = t
                    if (doB)
                        umma_bf16_fixed<true>(tm + TF_ACCB, umma_desc_words(loWm + o + k * 128, hiM), umma_desc_words(loCe + k * 128, hiM), idB);
            }
            umma_commit(&accfull);
        }
    } else if (warp == 12) {
        // ------------------------------------------------------------ rho / psi of a finished head: the mask warps' partial sums
        // added in a fixed order
        const size_t vo0 = (((size_t)b * p.H + h_begin) * p.ncs + c) * GF_T, vstep = (size_t)p.ncs * GF_T;
        for (int hi = 0; hi < nheads; ++hi) {
            const float *pr = parts + (hi & 1) * 1024;
            mbar_wait(&pfull[hi & 1], (hi >> 1) & 1, abortp, p.status);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = k * 32 + lane;
                float er = pr[i], ep = pr[512 + k * 128 + i];
#pragma unroll
                for (int m = 1; m <= k; ++m) er += pr[m * 128 + i];
#pragma unroll
                for (int m = k + 1; m < 4; ++m) ep += pr[512 + m * 128 + i];
                if (doC) p.rho[vo0 + hi * vstep + i] = er;
                if (doB) p.psi[vo0 + hi * vstep + i] = ep;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&pempty[hi & 1]);
        }
    } else if (sr > q) {
        // ------------------------------------------------------------ row scaling (warps 9, 13, 14): dy rows by e^{cs_t}, x rows
        // by dt_s e^{cs_last-cs_s}, in place, once the head's scores have been multiplied
        const int th = (warp == 9 ? 0 : warp == 13 ? 1 : 2) * 32 + lane;
        constexpr int I0 = doC ? 0 : 1024, I1 = doB ? 2048 : 1024;
        for (int hi = 0; hi < nheads; ++hi) {
            const int vb = hi % GF_VECS, u = hi + 1, e = hi + 2;
            const RowScale *sc = reinterpret_cast<const RowScale *>(record(vb) + REC_OC);      // of dy, then of x
            mbar_wait(&vfull[vb], (hi / GF_VECS) & 1, abortp, p.status);
            mbar_wait(&rfull[e & 3], (e >> 2) & 1, abortp, p.status);
            mbar_wait(&sfull[u & 1], (u >> 1) & 1, abortp, p.status);
            uint4 *rows = reinterpret_cast<uint4 *>(smem + (e & 3) * 32768);
            // eight 16-byte pieces in flight per thread: this role is three warps' worth of latency
            for (int i = I0 + th; i < I1; i += 8 * 96) {
                uint4 v[8];
                RowScale f[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int j = min(i + k * 96, 2047);
                    v[k] = rows[j];
                    f[k] = sc[j >> 3];
                }
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    scale8(v[k], f[k]);
                    if (i + k * 96 < I1) rows[i + k * 96] = v[k];
                }
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&scfull[hi & 1]);
                mbar_arrive(&vempty[vb]);
            }
        }
    } else {
        // ------------------------------------------------------------ mask warps: rows t = 32 q + lane, columns 32 sr ..
        const int rl = q * 32 + lane;
        const uint32_t tS = tm + tlane + sr * 32;
        float cb[32], wsum[32];
        mbar_wait(&sfull[0], 0, abortp, p.status);
        __syncwarp();
        tc_fence_after_sync();
        tmem_ld32(tS, cb);
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sempty[0]);
#pragma unroll
        for (int k = 0; k < 32; ++k) wsum[k] = 0.f;
        for (int hi = 0; hi < nheads; ++hi) {
            const int vb = hi % GF_VECS, u = hi + 1;
            const float *rec = record(vb), *cs2 = rec + REC_CS;
            mbar_wait(&vfull[vb], (hi / GF_VECS) & 1, abortp, p.status);
            const float csr = cs2[rl], cs_lo = cs2[q * 32], cs_hi = cs2[q * 32 + 31];
            mbar_wait(&sfull[u & 1], (u >> 1) & 1, abortp, p.status);
            __syncwarp();
            tc_fence_after_sync();
            float v[32];
            tmem_ld32(tS + (u & 1) * 128, v);
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sempty[u & 1]);
            if (sr != q || cs_lo - cs_hi <= kMildDecay) {
                const float f = sr != q ? ex2g(csr - cs_lo) * rec[REC_BLK + q * 4 + sr] : ex2g(csr - cs_hi);
                const float2 f2 = make_float2(f, f);
#pragma unroll
                for (int k = 0; k < 32; k += 4) {
                    const float4 cv = *reinterpret_cast<const float4 *>(rec + REC_CF + sr * 32 + k);
                    const float2 w0 = __fmul2_rn(make_float2(v[k], v[k + 1]), __fmul2_rn(make_float2(cv.x, cv.y), f2));
                    const float2 w1 = __fmul2_rn(make_float2(v[k + 2], v[k + 3]), __fmul2_rn(make_float2(cv.z, cv.w), f2));
                    v[k] = w0.x; v[k + 1] = w0.y; v[k + 2] = w1.x; v[k + 3] = w1.y;
                }
            } else {                         // a stiff head's diagonal
#pragma unroll
                for (int k = 0; k < 32; ++k) v[k] *= ex2g(fminf(csr - cs2[sr * 32 + k], 0.f)) * rec[REC_DT + sr * 32 + k];
            }
            if (sr == q) {
#pragma unroll
                for (int k = 1; k < 32; ++k) v[k] = k <= lane ? v[k] : 0.f;
            }
            float2 racc = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 32; k += 2) {
                const float2 wv = make_float2(v[k], v[k + 1]);
                const float2 a = __fadd2_rn(make_float2(wsum[k], wsum[k + 1]), wv);
                wsum[k] = a.x;
                wsum[k + 1] = a.y;
                const float2 z = __fmul2_rn(wv, make_float2(cb[k], cb[k + 1]));
                v[k] = z.x;
                v[k + 1] = z.y;
                racc = __fadd2_rn(racc, z);
            }
            // column sums over the warp's rows: transposing butterfly, lane l ends with column l
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int i = 0; i < o; ++i) {
                    const float send = up ? v[i] : v[i + o], keep = up ? v[i + o] : v[i];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
            float *pr = parts + (hi & 1) * 1024;
            if (hi >= 2) mbar_wait(&pempty[hi & 1], ((hi >> 1) - 1) & 1, abortp, p.status);
            pr[sr * 128 + rl] = racc.x + racc.y;
            pr[512 + q * 128 + sr * 32 + lane] = v[0];
            fence_proxy_async_smem();      // the record has been read before a bulk copy may overwrite it
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&vempty[vb]);
                mbar_arrive(&pfull[hi & 1]);
            }
        }
        // the head sum in two bf16 parts, what the first one's rounding leaves in the second: [part][s-half][128 rows t][128 B],
        // zeros above the diagonal
        mbar_wait(&stdone, 0, abortp, p.status);
        auto put = [&](int j, bool zero) {
            unsigned char *row = smem + OFF_ST + (j >> 1) * 16384 + rl * 128;
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
                uint32_t w[2][4];
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const float a = wsum[ch * 8 + 2 * m], b = wsum[ch * 8 + 2 * m + 1];
                    w[0][m] = zero ? 0u : pack2g(a, b);
                    w[1][m] = zero ? 0u : pack2g(a - __uint_as_float(w[0][m] << 16), b - __uint_as_float(w[0][m] & 0xffff0000u));
                }
                const uint32_t o = (((j & 1) * 4 + ch) ^ (rl & 7)) << 4;
#pragma unroll
                for (int part = 0; part < 2; ++part)
                    *reinterpret_cast<uint4 *>(row + part * GF_WPART + o) = make_uint4(w[part][0], w[part][1], w[part][2], w[part][3]);
            }
        };
        put(sr, false);
        for (int j = q + 1 + sr; j < 4; j += q + 1) put(j, true);     // the quarter's zero sub-tiles, shared out
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&wfull);
    }
    __syncwarp();

    // The CTA's partial slices of the group sums, [B, seg, G, nsl, N] fp32.  A row of an accumulator is N * 4 contiguous bytes
    // of its slice: staged in shared memory (every operand buffer is dead once the last products are done), rows padded by 16
    // bytes (conflict-free row-per-thread writes), and each row leaves as one bulk copy.
    mbar_wait(&accfull, 0, abortp, p.status);
    __syncwarp();
    tc_fence_after_sync();
    constexpr int PITCH = NS + 4;
    float *stgC = reinterpret_cast<float *>(smem), *stgB = stgC + 128 * PITCH;
    {
        float a[32];
        if (doC) {
            tmem_ld32(tm + tlane + TF_ACCC + sr * 32, a);
#pragma unroll
            for (int k = 0; k < 32; k += 4)
                *reinterpret_cast<float4 *>(stgC + (q * 32 + lane) * PITCH + sr * 32 + k) = make_float4(a[k], a[k + 1], a[k + 2], a[k + 3]);
        }
        if (doB) {
            tmem_ld32(tm + tlane + TF_ACCB + sr * 32, a);
#pragma unroll
            for (int k = 0; k < 32; k += 4)
                *reinterpret_cast<float4 *>(stgB + (q * 32 + lane) * PITCH + sr * 32 + k) = make_float4(a[k], a[k + 1], a[k + 2], a[k + 3]);
        }
    }
    fence_proxy_async_smem();
    tc_fence_before_sync();
    __syncthreads();
    if (tid < 256 && (tid < 128 ? doC : doB)) {
        const int row = tid & 127;
        const size_t o = ((((size_t)b * p.ncs * GF_T + (size_t)c * GF_T + row) * p.G + g) * nsl + sl) * NS;
        if (tid < 128) bulk_store(p.pC + o, stgC + row * PITCH, NS * 4);
        else bulk_store(p.pB + o, stgB + row * PITCH, NS * 4);
        tma_store_commit();
        tma_store_wait_all();
    }
    __syncthreads();
    if (warp == 0) {
        tc_fence_after_sync();
        tmem_dealloc(tm, 512);
    }
}

template <int WHAT>
static cudaError_t launch_bc(const SegParams &p, const TcMaps &m, cudaStream_t st) {
    const cudaError_t e = allow_smem<k_grad_bc<WHAT>>((int)GF_SMEM);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_grad_bc<WHAT>, dim3(p.nc * p.nsl * p.G * p.B), dim3(GF_THREADS), (size_t)GF_SMEM, st, p, m.x, m.dy, m.Bm, m.Cm,
                      m.H, m.G);
}

cudaError_t launch_grad_bc(const SegParams &p, const TcMaps &m, int what, cudaStream_t st) {
    if (what == BC_DC) return launch_bc<BC_DC>(p, m, st);
    if (what == BC_DB) return launch_bc<BC_DB>(p, m, st);
    return launch_bc<BC_DC | BC_DB>(p, m, st);
}

}  // namespace ssd
