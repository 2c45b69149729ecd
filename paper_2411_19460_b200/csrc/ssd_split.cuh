// 64 x 64 x 64 tile products with fp32 operands on the tensor cores: an fp32 value is the sum of three bf16 parts, a bf16 value is its own
// single part, and the products of parts are exact in the fp32 accumulators of mma.sync.
//
//   x = p0 + p1 + p2:  p0 the upper half of x's bits (no overflow near the largest values), p1 the rest rounded to nearest, so
//   that what it leaves for p2 has either sign, p2 the rest of that, at most eight bits.
// The sum is x exactly from 2^-110 up.  Of a smaller x it misses what lies below bf16's smallest number, less than 2^-133: values of 2^-120 are
// held to 13 bits, those of 2^-126, the smallest normal fp32 number, to seven, and what is below 2^-134 is zero (against an infinity: NaN).
// Products p_i q_j with i + j > 2 are left out (below 2^-23 of x y each, of either sign: about 2^-25 on average).  mma.sync truncates when it
// adds to its accumulator, a bias of half a unit in the last place per step, so for every 16 steps of the contraction the products
// start from zero, the smallest first, and their sum is added with a rounded fp32 addition: one truncation at the size of the sum.
// Infinities: p1 and p2 of an infinite x are NaN, and p0 = x times parts of either sign or zero would be NaN too, where x y is infinite.  So
// a NaN among the sums of 16 is taken again with whole values, in a second pass over a tile that has one (AGAIN): infinities and NaN come
// out as fp32 arithmetic has them.  (A signalling NaN whose payload is all in its lower half may come out as an infinity.)
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

#include <type_traits>

#include "ssd_sm100.cuh"

namespace ssd {

constexpr int SP_ROW = 72;          // bf16 per staged row of 64: 144 bytes, so that the eight rows of an ldmatrix phase are on different banks
struct SplitTile {
    __nv_bfloat16 v[64][SP_ROW];
};
template <typename T> struct SplitParts;
template <> struct SplitParts<float> { static constexpr int n = 3; };
template <> struct SplitParts<__nv_bfloat16> { static constexpr int n = 1; };

// The parts of two values as bf16 pairs
__device__ __forceinline__ void split2(float a, float b, uint32_t (&w)[3]) {
    const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
    w[0] = __byte_perm(ua, ub, 0x7632);
    const float ra = a - __uint_as_float(ua & 0xffff0000u), rb = b - __uint_as_float(ub & 0xffff0000u);
    const __nv_bfloat162 m = __floats2bfloat162_rn(ra, rb);
    w[1] = *reinterpret_cast<const uint32_t *>(&m);
    const float sa = ra - __uint_as_float(w[1] << 16), sb = rb - __uint_as_float(w[1] & 0xffff0000u);
    w[2] = __byte_perm(__float_as_uint(sa), __float_as_uint(sb), 0x7632);
}

// ---- a 64 x 64 tile of a row-major matrix on its way to shared memory, whose rows stay rows: ldmatrix transposes where a product
// needs the other direction
template <typename T> struct TileRegs;
template <> struct TileRegs<float> {
    static constexpr int N = 4, COLS = 4;      // pieces per thread, columns per piece
    float4 v[4];
    __device__ static int row(int k) { return (threadIdx.x >> 4) + 16 * k; }
    __device__ static int col() { return (threadIdx.x & 15) * 4; }
    __device__ void get(int k, float (&f)[4]) const { f[0] = v[k].x; f[1] = v[k].y; f[2] = v[k].z; f[3] = v[k].w; }
};
template <> struct TileRegs<__nv_bfloat16> {
    static constexpr int N = 2, COLS = 8;
    uint4 v[2];
    __device__ static int row(int k) { return (threadIdx.x >> 3) + 32 * k; }
    __device__ static int col() { return (threadIdx.x & 7) * 8; }
    __device__ void get(int k, float (&f)[8]) const {
        const uint32_t e[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            f[2 * i] = __uint_as_float(e[i] << 16);
            f[2 * i + 1] = __uint_as_float(e[i] & 0xffff0000u);
        }
    }
};
// WS: from scratch that an earlier kernel of the call wrote (coherent loads)
template <bool WS = false, typename T> __device__ __forceinline__ void tile_load(TileRegs<T> &r, const T *src, size_t stride) {
#pragma unroll
    for (int k = 0; k < TileRegs<T>::N; ++k) {
        auto *q = reinterpret_cast<const decltype(r.v[0].x) *>(src + (size_t)r.row(k) * stride + r.col());
        using V = std::remove_reference_t<decltype(r.v[0])>;
        r.v[k] = WS ? *reinterpret_cast<const V *>(q) : __ldg(reinterpret_cast<const V *>(q));
    }
}
// Four or eight consecutive fp32 values of a row as three parts
template <int COLS> __device__ __forceinline__ void put_split(SplitTile *s, int row, int col, const float (&f)[COLS]) {
    uint32_t w[COLS / 2][3];
#pragma unroll
    for (int i = 0; i < COLS / 2; ++i) split2(f[2 * i], f[2 * i + 1], w[i]);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        if constexpr (COLS == 8) *reinterpret_cast<uint4 *>(&s[p].v[row][col]) = make_uint4(w[0][p], w[1][p], w[2][p], w[3][p]);
        else *reinterpret_cast<uint2 *>(&s[p].v[row][col]) = make_uint2(w[0][p], w[1][p]);
    }
}
__device__ __forceinline__ void tile_store(SplitTile *s, const TileRegs<__nv_bfloat16> &r) {
#pragma unroll
    for (int k = 0; k < 2; ++k) *reinterpret_cast<uint4 *>(&s[0].v[r.row(k)][r.col()]) = r.v[k];
}
__device__ __forceinline__ void tile_store(SplitTile *s, const TileRegs<float> &r) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float f[4];
        r.get(k, f);
        put_split(s, r.row(k), r.col(), f);
    }
}

// ---- products.  Eight warps, warp (wm, wn) has rows 16 wm .. and columns 32 wn .. of the output in the accumulator layout of
// mma.m16n8k16: element (j, i) is row acc_row(i >> 1), column acc_col(j) + (i & 1).
struct Acc {
    float m[4][4];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) m[j][i] = 0.f;
    }
    __device__ __forceinline__ bool nan() const {
        bool r = false;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) r |= isnan(m[j][i]);
        return r;
    }
    // rows of half `half`, columns acc_col(j) and the next
    __device__ __forceinline__ float2 get(int j, int half) const { return make_float2(m[j][2 * half], m[j][2 * half + 1]); }
    __device__ __forceinline__ void set(int j, int half, float2 v) {
        m[j][2 * half] = v.x;
        m[j][2 * half + 1] = v.y;
    }
};
__device__ __forceinline__ int acc_row(int half) { return ((threadIdx.x >> 5) & 3) * 16 + ((threadIdx.x >> 2) & 7) + half * 8; }
__device__ __forceinline__ int acc_col(int j) { return (threadIdx.x >> 7) * 32 + j * 8 + (threadIdx.x & 3) * 2; }

template <bool TRANS> __device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
    if (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(addr)
                     : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(addr)
                     : "memory");
}
__device__ __forceinline__ void mma_acc(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_zero(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
// Element (row, col) of a tile from its PARTS parts: the first alone where it is infinite, because the others are NaN then
template <int PARTS> __device__ __forceinline__ float joined(const SplitTile *s, int row, int col) {
    const float p0 = __bfloat162float(s[0].v[row][col]);
    if constexpr (PARTS == 1) return p0;
    const float v = p0 + (__bfloat162float(s[1].v[row][col]) + __bfloat162float(s[2].v[row][col]));
    return isinf(p0) ? p0 : v;
}
// c += A B over 64 steps of the contraction, A of PA parts and B of PB.  AK, BK: the staged rows of that operand run along the
// contraction (else along the output's rows, columns).  AGAIN: sums of 16 products that come out as NaN are taken again, of whole values.
template <int PA, int PB, bool AK, bool BK, bool AGAIN> __device__ __forceinline__ void tile_mma(Acc &c, const SplitTile *a, const SplitTile *b) {
    const int lane = threadIdx.x & 31, wm = ((threadIdx.x >> 5) & 3) * 16, wn = (threadIdx.x >> 7) * 32;
    const int l7 = lane & 7, l8 = ((lane >> 3) & 1) * 8, l16 = (lane >> 4) * 8;
    constexpr uint32_t ROWB = SP_ROW * 2, PART = sizeof(SplitTile);
    const uint32_t aa = sm100::smem_u32(a) + (AK ? (l16 + l7) * ROWB + (wm + l8) * 2 : (wm + l8 + l7) * ROWB + l16 * 2);
    const uint32_t ba = sm100::smem_u32(b) + (BK ? (l8 + l7) * ROWB + (wn + l16) * 2 : (wn + l16 + l7) * ROWB + l8 * 2);
    auto steps = [&](int k) {
        uint32_t fa[PA][4];
        float t[4][4];
#pragma unroll
        for (int p = 0; p < PA; ++p) ldsm4<AK>(fa[p], aa + p * PART + (AK ? k * ROWB : k * 2));
        bool first = true;
#pragma unroll
        for (int q = PB - 1; q >= 0; --q) {
            uint32_t fb[2][4];
#pragma unroll
            for (int n = 0; n < 2; ++n) ldsm4<BK>(fb[n], ba + q * PART + (BK ? k * ROWB + n * 32 : k * 2 + n * 16 * ROWB));
#pragma unroll
            for (int p = PA - 1; p >= 0; --p) {
                if (p + q > 2) continue;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (first) mma_zero(t[j], fa[p], fb[j >> 1][(j & 1) * 2], fb[j >> 1][(j & 1) * 2 + 1]);
                    else mma_acc(t[j], fa[p], fb[j >> 1][(j & 1) * 2], fb[j >> 1][(j & 1) * 2 + 1]);
                }
                first = false;
            }
        }
        if constexpr (AGAIN && PA + PB > 2) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (!(isnan(t[j][0]) || isnan(t[j][1]) || isnan(t[j][2]) || isnan(t[j][3]))) continue;
                float f[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
                for (int i = k; i < k + 16; ++i)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int r = acc_row(e >> 1), n = acc_col(j) + (e & 1);
                        f[e] = fmaf(AK ? joined<PA>(a, i, r) : joined<PA>(a, r, i), BK ? joined<PB>(b, i, n) : joined<PB>(b, n, i), f[e]);
                    }
#pragma unroll
                for (int e = 0; e < 4; ++e) t[j][e] = isnan(t[j][e]) ? f[e] : t[j][e];
            }
            __syncwarp();
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int half = 0; half < 2; ++half) c.set(j, half, __fadd2_rn(c.get(j, half), make_float2(t[j][2 * half], t[j][2 * half + 1])));
    };
    if constexpr (AGAIN) {
#pragma unroll 1
        for (int k = 0; k < 64; k += 16) steps(k);
    } else {
#pragma unroll
        for (int k = 0; k < 64; k += 16) steps(k);
    }
}

}  // namespace ssd
