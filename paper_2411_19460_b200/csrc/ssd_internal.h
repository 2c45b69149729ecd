// Internal declarations shared by the host driver and the kernel files of libssd.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "ssd.h"

namespace ssd {

// Everything one segment's kernels need.  Passed by value to every kernel.
// Programmatic dependent launch: a kernel launched through launch_pdl() may be scheduled while its predecessor
// in the stream is still running (its CTAs take the SMs the predecessor's last wave leaves idle, and set up
// their barriers / tensor memory there); pdl_wait() returns once the predecessor has completed and its writes
// are visible.  It must precede every access to what is written within the call, and every store.  The caller's inputs may be read
// ahead of it where the call's first launch is an ordinary one (`first` below): they are complete then.  Where every launch
// is a dependent one (convolution, norm, decode, glue) it precedes the first global-memory access.
// pdl_launch_dependents() lets the successor be scheduled from this point on.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... KArgs, typename... Args>
inline cudaError_t launch_as(bool dependent, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args &&...args) {
    return launch_as(true, kernel, grid, block, smem, st, args...);
}
// Lets kernel K use `bytes` of dynamic shared memory; the attribute is set once per device.
template <auto K> inline cudaError_t allow_smem(int bytes) {
    static std::atomic<uint64_t> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = 1ull << (dev & 63);
    if (dev < 64 && (done.load(std::memory_order_relaxed) & bit)) return cudaSuccess;
    e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
    return e;
}
#endif

constexpr int kNumSMs = 148;
constexpr int kStatePassElems = 512;   // state elements per CTA of the state passes
constexpr int kTcBlock = 128;     // steps per block of the tensor-core path, half the caller's chunk
constexpr int kTcState = 128;     // its state size N

// Per (head, block of 128 steps) record of the tensor-core path, made once per segment by the forward chain and copied to
// shared memory in one piece by every kernel that masks a tile (cs: inclusive cumsum of dt*A in the block, log2 units;
// sub-tile: 32 steps).  Offsets in floats; the parts a kernel needs are adjacent.
enum {
    REC_CFX = 0,        // [128] e^{cs_t - cs[first of t's sub-tile]}
    REC_BLK = 128,      // [4][4] e^{cs[32 i] - cs[32 j + 31]}, j < i
    REC_DECAY = 144,    // e^{cs_last}
    REC_CS = 160,       // [128] cs
    REC_DT = 288,       // [128] dt
    REC_CF = 416,       // [128] dt_s e^{cs[last of s's sub-tile] - cs_s}
    REC_OC = 544,       // [128] e^{cs_t}, as a RowScale
    REC_OB = 800,       // [128] dt_s e^{cs_last - cs_s}, as a RowScale
    REC_FLOATS = 1056
};
// Up to this many log2 units of decay inside a sub-tile, e^{cs_t - cs_s} on its diagonal is taken as a product of a row and a
// column factor (one of them > 1, far from overflow) like everywhere else; beyond, element by element.
constexpr float kMildDecay = 40.f;

struct SegParams {
    int B, L, H, P, N, G, Q;
    int hpg;       // heads per group
    int t0;        // first token of the segment
    int nc;        // chunks in this segment
    int c0;        // global index of the segment's first chunk
    uint32_t inv_nc, inv_H;  // divide_by() of nc and H
    int ncs;       // chunk capacity of the workspace (chunks of a full segment)
    int nct;       // chunks in the whole sequence (L / Q)
    int nsl;       // slices per group in the dB/dC partial buffers: head ranges, or slots of all ranges (split path)
    int ndd;       // partial sums of dD per (head, chunk) that the kernels of this path write (<= 4)
    int scan_ctas; // CTAs of the y / dx kernel, at most (no effect on results)
    int chain_heads; // heads per CTA of the forward chain, 1 or 2 (no effect on results)
    int ngh;       // partial sums of <G,H> per (head, chunk) (<= 16)
    int tiles;     // split path: 64-step tiles per chunk (rho, psi and the slices come per tile); tensor-core path: 0
    int first;        // the call's first launch: an ordinary one, so that nothing of the call starts before what is older than it has ended;
                   // it clears the status word (as a launch of its own: 2 us a call)
    float dx_skip;    // 1 when dx also takes dy (a skip connection around the layer), else 0
    int64_t x_bs, dt_bs, bc_bs;  // batch strides, elements

    // caller tensors
    const void *x, *Bm, *Cm, *dy;
    const float *dt, *A, *D;
    void *y, *dx, *dB, *dC;
    float *ddt;

    // workspace regions (all fp32 unless noted)
    unsigned int *status;  // [0] = error flag of bounded waits
    float *rec;            // tensor-core path: [B,H,ncs,REC_FLOATS]
    float *cs;             // split path: [B,H,ncs,Q] inclusive cumsum of dt*A inside each chunk
    float *dtT;            // dt head-major, vector of (b, h, c) at dt_stride floats: [B,H,ncs,Q], or inside the records
    int dt_stride;
    float *Hst;            // split path: [B,ncs+1,H,P,N] slot c = state entering chunk c; slot nc = leaving the segment
    float *Gst;            // split path: [B,ncs+1,H,P,N] slot c+1 = dLoss/d(state leaving chunk c)
    __nv_bfloat16 *Hbf;    // tensor-core path: [B,ncs,H,N,P] (transposed) state entering block c
    __nv_bfloat16 *Gbf;    // tensor-core path: [B,ncs,H,N,P] dLoss/d(state leaving block c)
    const float *hinit, *ginit;     // split path, states made by their readers: state (gradient) entering the segment from the left
    int64_t hinit_bs, ginit_bs;     // (right), null = zeros, and their batch strides
    float *hcarry;         // [B,H,P,N]     state handed from segment to segment (forward; null in the backward, which does not)
    float *gcarry;         // [B,H,P,N]     state gradient handed right-to-left (backward)
    float *ghdot;          // [B,H,ncs,16]  partial sums of exp(cs_last) <Gout_c, H_in,c>
    float *ddt_dir;        // [B,H,ncs,Q]   direct part of ddt (tensor-core path: read where dt is next to zero, see bwd_finish)
    float *cbt;            // split path: [B,ncs,G,Q,Q] C B^T, causal 64 x 64 tiles (null: made again where used, y in order only)
    float *rho;            // [B,H,ncs,Q]   C_t . (intra-chunk part of this head's dC_t); split path: [B,H,ncs,tiles,Q] by column tile
    float *rho2;           // [B,H,ncs,Q]   C_t . (inter-chunk part of this head's dC_t)
    float *psi;            // [B,H,ncs,Q]   B_t . (intra-chunk part of this head's dB_t); split path: [B,H,ncs,tiles,Q] by row tile
    float *psi2;           // [B,H,ncs,Q]   B_t . (inter-chunk part of this head's dB_t)
    float *pB, *pC;        // [B,seg,G,nsl,N] partial dB / dC; split path: one buffer, pC, for both
    float *dAp;            // [B,H,nct]     per-chunk partial of dA
    float *dDp;            // [B,H,nct,4]   partials of dD, the first ndd of each group in use
};

// n / d by a multiplication and one correction, for n below 2^31: kernels that take a tile per CTA divide its number several times
static inline uint32_t inverse_of(int d) { return d > 1 ? (uint32_t)((1ull << 32) / (unsigned)d) : 0xffffffffu; }
#ifdef __CUDACC__
__device__ __forceinline__ int divide_by(int n, int d, uint32_t inv) {
    const int q = (int)__umulhi((unsigned)n, inv);      // n / d or one less
    return n - q * d >= d ? q + 1 : q;
}
#endif

static inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// ---- kernel launchers (each returns the cudaError_t of its launch) ----
// ssd_simt.cu : kernels of the split path (fp32 operands as bf16 parts), any I/O dtype
// SIMT_SUMS: chunk sums, cumsum and C B^T | SIMT_SUMS_GRAD: also the state-gradient sums | SIMT_Y: y, and the sums of segment
// `next` if given | SIMT_BWD: dx, slices of dB and dC | SIMT_TAIL: finishing steps and the sums (with gradients) of segment `next`
// Short segments need no state pass: with `pass`, whoever reads a state in SIMT_Y or SIMT_BWD makes it from the chunk sums (which stay),
// and CTAs of the same launch make what the pass hands on.
constexpr int kReaderChunks = 8;       // chunks of such a segment, at most
struct StatePass {
    float *boundary, *leave, *fin;     // state entering the segment (null: not stored) | state (backward: gradient) leaving it | h_final (or null)
    int64_t boundary_bs, leave_bs;
};
enum { SIMT_SUMS = 0, SIMT_SUMS_GRAD, SIMT_Y, SIMT_BWD, SIMT_TAIL };
cudaError_t launch_simt(const SegParams &p, const SegParams *next, const StatePass *pass, int dtype, int what, cudaStream_t st);
// init: state entering the segment (NULL = zeros), batch stride init_bs elements;
// boundary_out (nullable): where to store that state, batch stride bnd_bs; final_out nullable.
cudaError_t launch_state_pass_fwd(const SegParams &p, const float *init, long long init_bs,
                                  float *boundary_out, long long bnd_bs, float *final_out, cudaStream_t st);
// the backward's: entry states from init, then the gradients from ginit (NULL = zeros), handed left to gleft
cudaError_t launch_state_pass_bwd(const SegParams &p, const float *init, long long init_bs, const float *ginit, float *gleft, cudaStream_t st);
cudaError_t launch_bwd_tail(const SegParams &p, int dtype, cudaStream_t st);
cudaError_t launch_final_dAdD(const SegParams &p, float *dA, float *dD, bool accumulate, cudaStream_t st);
// ssd_glue.cu : layer-axis glue of a layer stack
cudaError_t launch_glue(int dtype, bool transpose, const void *a, const void *b, const float *W, void *out,
                        long long rows_per_batch, long long bstride, int B, cudaStream_t st);
cudaError_t launch_residual(int dtype, void *dst, const void *src, long long n_per_batch, long long bstride, int B,
                            cudaStream_t st);

// ssd_conv.cu : depthwise causal convolution (width 4) + SiLU in front of the SSD layer, with its 3-token state
int conv_tiles(int L);
cudaError_t launch_conv_fwd(int dtype, const void *u, long long u_bs, const float *w, const float *bias,
                            const void *state_in, void *out, void *state_out, int B, int L, int C, cudaStream_t st);
cudaError_t launch_conv_bwd(int dtype, const void *u, long long u_bs, const float *w, const float *bias,
                            const void *state_in, const void *dout, const float *dtail, void *du, float *dstate,
                            float *dw, float *dbias, int accumulate, float *part, int B, int L, int C, cudaStream_t st);
// ssd_norm.cu : gated RMS normalisation behind the SSD layer
long long gated_norm_tiles(long long rows);
int gated_norm_max_group();
cudaError_t launch_gated_norm_fwd(int dtype, const void *y, const void *z, const float *gamma, float eps, void *out,
                                  long long rows, int D, int group, cudaStream_t st);
cudaError_t launch_gated_norm_bwd(int dtype, const void *y, const void *z, const float *gamma, float eps, const void *dout,
                                  void *dy, void *dz, float *dgamma, int accumulate, float *part, long long rows, int D,
                                  int group, cudaStream_t st);
// ssd_decode.cu : one token of the recurrence, state updated in place
cudaError_t launch_decode_step(int dtype, int N, const void *x, const float *dt, const float *A, const void *Bm,
                               const void *Cm, const float *D, float *h, void *y, int B, int H, int P, int G,
                               long long x_bs, long long dt_bs, long long bc_bs, cudaStream_t st);

// ssd_tc.cu : tensor maps of the tensor-core (tcgen05 / TMEM / TMA) kernels, bf16 I/O
struct TcMaps {
    CUtensorMap x, dy, Bm, Cm;  // [B][L][H*64] / [B][L][G*N], box 64 x 128 rows
    CUtensorMap y, dx;          // outputs, same geometry as x
    CUtensorMap H, G;           // bf16 states as [rows][64], box 64 x N rows
    CUtensorMap Hst, Gst;       // the same for the stores of the chain kernels: box 32 x 32 rows, 64-byte swizzle
};
bool tc_supported(int dtype, int flags, int P, int N, int chunk, int heads_per_group);
bool tc_make_maps(const SegParams &p, TcMaps &m);
bool tc_state_maps(const SegParams &p, TcMaps &m);
// ssd_tc_chain.cu : block sums and the recurrence over the blocks.  init: state (gradient) entering the segment (NULL = zeros),
// batch stride init_bs; boundary_out (nullable): where to store that state, batch stride bnd_bs; final_out nullable.
enum { CHAIN_FWD = 0, CHAIN_BWD = 1 };
cudaError_t launch_chain_fwd(const SegParams &p, const TcMaps &m, const float *init, long long init_bs, float *boundary_out, long long bnd_bs,
                             float *final_out, cudaStream_t st);
cudaError_t launch_chain_bwd(const SegParams &p, const TcMaps &m, const float *init, float *left_out, cudaStream_t st);
// ssd_tc_scan.cu : y (SC_FWD) or dx, ddt_direct, dD partials, psi2 (SC_DX)
cudaError_t launch_scan_tc(const SegParams &p, const TcMaps &m, int mode, cudaStream_t st);
enum { SC_FWD = 0, SC_DX = 1 };
// ssd_tc_bcf.cu : partial slices of dC and rho (BC_DC), of dB and psi (BC_DB), or both from one masked tile
cudaError_t launch_grad_bc(const SegParams &p, const TcMaps &m, int what, cudaStream_t st);
enum { BC_DC = 1, BC_DB = 2 };

// kernel kinds, for the launch counter and the optional per-kind timing
enum {
    KIND_CHUNK_STATE = 0, KIND_STATE_PASS_FWD, KIND_SCAN_FWD, KIND_DSTATE, KIND_STATE_PASS_BWD, KIND_BWD_DX, KIND_BWD_DC, KIND_BWD_DB,
    KIND_BWD_FINISH, KIND_FINAL, KIND_GLUE, KIND_DECODE, KIND_BWD_DBDC, KIND_CONV, KIND_NORM, KIND_COUNT
};

}  // namespace ssd
