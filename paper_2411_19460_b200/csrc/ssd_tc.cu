// Which calls run on the tensor-core kernels (tcgen05.mma with fp32 accumulators in TMEM, operands staged in shared memory
// by TMA, ssd_tc_chain.cu, ssd_tc_scan.cu, ssd_tc_bcf.cu), and the tensor maps of one call.
#include <cstring>

#include "ssd_internal.h"
#include "ssd_sm100.cuh"

namespace ssd {

using namespace sm100;

// ------------------------------------------------------------------ host: tensor maps
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    }
    return fn;
}

// bf16 tensor [dim2][dim1][dim0] (dim0 contiguous), box {box_cols, box_rows, 1}; 128-byte swizzle for
// 64-element (128-byte) box rows, 64-byte swizzle for 32-element ones.
static bool make_map3(CUtensorMap *m, const void *ptr, uint64_t dim0, uint64_t dim1, uint64_t dim2,
                      uint64_t stride1_elems, uint64_t stride2_elems, uint32_t box_rows, uint32_t box_cols = 64) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[3] = {dim0, dim1, dim2};
    cuuint64_t strides[2] = {stride1_elems * 2, stride2_elems * 2};
    cuuint32_t box[3] = {box_cols, box_rows, 1};
    cuuint32_t es[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(ptr), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, box_cols == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The tensor-core kernels round decayed rows, masked tiles and states to bf16, so that a call's fp32 outputs (states, ddt, dA)
// are within 2e-3 of the exact ones; the split-path kernels keep all of it in fp32 (1e-6).  Which bf16 calls take which is
// therefore part of what a caller gets: N = 64, chunks below 256 and odd numbers of heads per group have fp32 intermediates.
// On these kernels, which could run them, 2 x 8192 steps of 32 heads with N = 64 took 378 us instead of 1015 (with FFMA 2250), and
// h_final was off by 1.7e-3 instead of 9e-7, ddt by 2.1e-3 instead of 2e-7 (4096 of these steps).
bool tc_supported(int dtype, int flags, int P, int N, int chunk, int heads_per_group) {
    return dtype == SSD_DTYPE_BF16 && !(flags & SSD_FLAG_FORCE_SIMT) && P == 64 && N == kTcState && chunk == 2 * kTcBlock &&
           heads_per_group % 2 == 0 && encode_fn() != nullptr;
}

// Builds the tensor maps of one API call.  x/dy/Bm/Cm may be null when the call does not use them.
bool tc_make_maps(const SegParams &p, TcMaps &m) {
    memset(&m, 0, sizeof(m));
    const uint64_t HP = (uint64_t)p.H * 64, GN = (uint64_t)p.G * p.N;
    bool ok = true;
    if (p.x) ok = ok && make_map3(&m.x, p.x, HP, p.L, p.B, HP, p.x_bs, 128);
    if (p.dy) ok = ok && make_map3(&m.dy, p.dy, HP, p.L, p.B, HP, p.x_bs, 128);
    if (p.y) ok = ok && make_map3(&m.y, p.y, HP, p.L, p.B, HP, p.x_bs, 128);
    if (p.dx) ok = ok && make_map3(&m.dx, p.dx, HP, p.L, p.B, HP, p.x_bs, 128);
    if (p.Bm) ok = ok && make_map3(&m.Bm, p.Bm, GN, p.L, p.B, GN, p.bc_bs, 128);
    if (p.Cm) ok = ok && make_map3(&m.Cm, p.Cm, GN, p.L, p.B, GN, p.bc_bs, 128);
    return ok && tc_state_maps(p, m);
}

// The maps of the bf16 states alone, viewed as [B*ncs*H*N rows][64].
bool tc_state_maps(const SegParams &p, TcMaps &m) {
    bool ok = true;
    const uint64_t srows = (uint64_t)p.B * p.ncs * p.H * p.N;
    if (p.Hbf) {
        ok = ok && make_map3(&m.H, p.Hbf, 64, srows, 1, 64, srows * 64, p.N);
        ok = ok && make_map3(&m.Hst, p.Hbf, 64, srows, 1, 64, srows * 64, 32, 32);
    }
    if (p.Gbf) {
        ok = ok && make_map3(&m.G, p.Gbf, 64, srows, 1, 64, srows * 64, p.N);
        ok = ok && make_map3(&m.Gst, p.Gbf, 64, srows, 1, 64, srows * 64, 32, 32);
    }
    return ok;
}

}  // namespace ssd
