// Internal launcher declarations shared by the translation units of the library.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <cstdlib>

#include "cq_common.cuh"

namespace cq {

cudaError_t launch_pack_codes(const int8_t *k, int B, int64_t N, int64_t K, uint8_t *codes, cudaStream_t st);
cudaError_t launch_repack(const uint8_t *codes, const float *scale, const uint16_t *a, const uint16_t *b, const Dims &d,
                          void *layout, cudaStream_t st);
cudaError_t launch_unpack(const void *layout, const Dims &d, uint8_t *codes, float *scale, uint16_t *a, uint16_t *b,
                          cudaStream_t st);
cudaError_t launch_decode_levels(const void *layout, const Dims &d, float *levels, cudaStream_t st);
cudaError_t launch_decode_carriers(const void *layout, const Dims &d, int8_t *carriers, cudaStream_t st);
cudaError_t launch_decode_weights(const void *layout, const Dims &d, float *What, cudaStream_t st);
cudaError_t launch_a8_partials(const void *layout, const Dims &d, const int8_t *x8, int64_t M, int32_t *P, cudaStream_t st);
// act_f16 (here and below): the 16-bit activation / output patterns are binary16 instead of bfloat16
// operand_order: x8 in the order of cq_decode.cuh that the INT8 products of every width but four bits read; natural order otherwise
cudaError_t launch_quantize_a8(const uint16_t *x, int64_t M, int64_t K, int8_t *x8, int64_t x8_pitch, float *dx,
                               bool operand_order, bool act_f16, cudaStream_t st);
// h[M][2 I] (gate | up, model dtype) -> INT8 carrier of silu(gate) * up, and its row scales
cudaError_t launch_swiglu_quantize_a8(const uint16_t *h, int64_t M, int64_t I, int8_t *x8, int64_t x8_pitch, float *dx,
                                      bool operand_order, bool act_f16, cudaStream_t st);
// routed execution: xg[r] = x[route_token[r]] (zero row for an index outside [0, T)); the status word and n counters are zeroed
cudaError_t launch_gather_rows(const uint16_t *x, const int32_t *route_token, uint16_t *xg, int64_t R, int64_t T, int64_t K,
                               int *status, int *counters, int64_t n, cudaStream_t st);
cudaError_t launch_wait_timeout(int *status, long long limit_cycles, cudaStream_t st);

// Workspace carving (all offsets 256-byte aligned).
struct Workspace {
    size_t counters_off, counters_bytes;   // int32 arrival counters, one per 128-row block
    size_t partial_off, partial_bytes;     // fp32 split-K partial sums: small M [CTA][2][M][128]; model-dtype GEMM [run, CTA of a pair][2][tokens][128]; A8 GEMM [shared tile][slice][BN][128]
    size_t x8_off, x8_bytes;               // Dynamic A8: int8 activation carrier [M][Kp]
    size_t dx_off, dx_bytes;               // Dynamic A8: row scales [M]
    size_t status_off;                     // int32 device status word (bounded waits report here)
    size_t total;
};
Workspace plan_workspace(const Dims &d, int64_t M, int mode);

// Streaming multiprocessors of the current device (148 when no device can be asked).
int sm_count();

// cudaFuncSetAttribute is a per-DEVICE setting: `done` (one per kernel instantiation) remembers, as a bit
// mask, the devices on which it has been made, so a process that uses several GPUs sets it on each.
// Thread safe; devices beyond 63 simply set the attribute on every launch.
template <class Kern>
cudaError_t ensure_func_attr(Kern kern, std::atomic<uint64_t> &done, cudaFuncAttribute attr, int value) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool tracked = dev >= 0 && dev < 64;
    const uint64_t bit = tracked ? (1ull << dev) : 0;
    if (tracked && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, attr, value);
    if (e == cudaSuccess && tracked) done.fetch_or(bit, std::memory_order_release);
    return e;
}
// Launch that may begin while the kernel before it in the stream drains (programmatic dependent launch): every kernel started
// this way runs griddepcontrol.wait before it reads or writes any buffer; what comes before the wait is the set-up of its own
// on-chip state and prefetches of weights to L2.  Their inputs are not __restrict__: the non-coherent path, which that opens to
// the compiler, wants memory that nobody writes from the kernel's start on.  cluster: CTAs per cluster (1: none); overlap: false for the few kernels
// that do not gain by it.
template <class... P, class... A>
cudaError_t launch_overlapped(void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, int cluster, bool overlap, A &&...args) {
    static const bool use_pdl = getenv("CQ_NO_PDL") == nullptr;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (use_pdl && overlap) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)cluster; attr[n].val.clusterDim.y = 1; attr[n++].val.clusterDim.z = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<A &&>(args)...);
}
// the thread's record of the last failed CUDA call (what cq_last_cuda_error returns)
void set_last_cuda_error(cudaError_t e);

// Several products over one activation matrix in one launch (routed execution): rows [row0, row0 + rows) of x and y
// belong to the matrix `layout`; all matrices share shape and format.  unit0 is filled in by the launcher: the first
// output tile (or pair of tiles) of the group.  More groups than a table holds go out as several launches.
constexpr int MAX_GROUPS = 32;
struct Group { const void *layout; int row0, rows, unit0; };
struct GroupTable { int n; Group g[MAX_GROUPS]; };

// Decomposition of the small-M path: CTAs (one contiguous run of tiles each), sets of eight warps in each.
struct GemvPlan { int ctas, sets; };
GemvPlan gemv_plan(const Dims &d, int64_t M, int mode);

// Small-M (M <= 16) split-K tensor-core GEMV, both activation modes.
// prequantized (Dynamic A8 only): the workspace already holds the INT8 carrier and the row scales of x (x is not read)
cudaError_t launch_gemv(const void *layout, const Dims &d, const uint16_t *x, uint16_t *y, int64_t M, int mode,
                        bool act_f16, uint8_t *ws, const Workspace &plan, cudaStream_t st, bool prequantized = false);
// One and two tokens in the model dtype, strips of sixteen channels, where K and the workspace allow it (cq_gemv_strip.cu).
bool gemv_strip_ok(const Dims &d, int64_t M, const Workspace &plan);
cudaError_t launch_gemv_strip(const void *layout, const Dims &d, const uint16_t *x, uint16_t *y, int64_t M, bool act_f16,
                              float *partial, int *counters, cudaStream_t st);
// every group 1 .. 16 rows; x and y are those of all groups; P CTAs and a workspace slice for each group
cudaError_t launch_gemv_groups(const GroupTable &groups, const Dims &d, const uint16_t *x, const int8_t *xq, const float *dxs, uint16_t *y,
                               int mode, bool act_f16, int P, float *partial, int *counters, cudaStream_t st);
// `R` rows of x in all, every group at most `tile_m` rows to a token tile of that size class
cudaError_t launch_gemm_tc_groups(const GroupTable &groups, const Dims &d, const uint16_t *x, uint16_t *y, int64_t R, int64_t tile_m,
                                  bool act_f16, int *status, cudaStream_t st);
cudaError_t launch_gemm_a8_groups(const GroupTable &groups, const Dims &d, const int8_t *xq, const float *dxs, uint16_t *y, int64_t R,
                                  int64_t tile_m, bool act_f16, int *status, cudaStream_t st);
int gemm_tc_token_tile(int64_t M);
// cw: CTAs that compute a tile together (2: a pair, 256 channels); t_full whole tiles and p2 runs are counted in such units
// cost: microseconds, rough
struct TcPlan { int bnt, token_tiles, ctas, stream_k, p2, crossing, cw; int64_t t_full; double cost; };
TcPlan gemm_tc_plan(const Dims &d, int64_t M);
int gemm_a8_token_tile(const Dims &d, int64_t M);
// cost: blocks of 128 k in the main loop
struct A8Plan { int bn, token_tiles, slices, ctas; int64_t t_full; double cost; };
A8Plan gemm_a8_plan(const Dims &d, int64_t M);
// the groups of a class in one launch of whole tiles, in the units of the plans' costs
double gemm_tc_groups_cost(const GroupTable &groups, const Dims &d, int64_t tile_m);
double gemm_a8_groups_cost(const GroupTable &groups, const Dims &d, int64_t tile_m);

// offline encoder steps (cq_encode.cu)
cudaError_t launch_encode_assign(const float *W, int B, int G, int64_t N, int64_t K, const float *scale, const uint16_t *a,
                                 const uint16_t *b, int joint, int8_t *k, cudaStream_t st);
cudaError_t launch_encode_scale(const float *W, const int8_t *k, int B, int G, int64_t N, int64_t K, const uint16_t *a,
                                const uint16_t *b, int joint, float *scale, cudaStream_t st);
cudaError_t launch_encode_losses(const float *W, const int8_t *k, int B, int G, int64_t N, int64_t K, const float *scale,
                                 const uint16_t *a, const uint16_t *b, double *LC, double *LA8, cudaStream_t st);
cudaError_t launch_encode_search(const float *W, int B, int G, int64_t N, int64_t K, int joint, int effort, int8_t *k,
                                 float *scale, uint16_t *a, uint16_t *b, cudaStream_t st);
// Large-M tcgen05 / TMEM GEMM, both activation modes.
cudaError_t launch_gemm_tc(const void *layout, const Dims &d, const uint16_t *x, uint16_t *y, int64_t M, int mode,
                           bool act_f16, uint8_t *ws, const Workspace &plan, cudaStream_t st);

// Large-M Dynamic-A8 GEMM: activation quantiser, then tcgen05 kind::i8 with per-group int32 partials.
cudaError_t launch_gemm_a8_tc(const void *layout, const Dims &d, const uint16_t *x, uint16_t *y, int64_t M, bool act_f16,
                              uint8_t *ws, const Workspace &plan, cudaStream_t st, bool prequantized = false);

}  // namespace cq
