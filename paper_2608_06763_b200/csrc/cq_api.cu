// C ABI of the library (include/cubicquant.h): argument validation on the host, then launches.
#include "../../include/cubicquant.h"

#include <cuda_runtime.h>

#include <algorithm>

#include "cq_common.cuh"
#include "cq_internal.h"

namespace cq {

static thread_local int g_last_cuda_error = 0;
void set_last_cuda_error(cudaError_t e) { g_last_cuda_error = (int)e; }

int gemm_tc_available();

static inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

Workspace plan_workspace(const Dims &d, int64_t M, int mode) {
    Workspace w{};
    const int64_t Kp = (int64_t)d.KT * TILE;
    const int64_t Mc = M < 16 ? M : 16;  // rows handled by one small-M launch
    const GemvPlan gp = gemv_plan(d, Mc, mode);
    size_t off = 0;
    w.status_off = off; off += 256;  // first, so cq_gemm_status finds it without knowing the problem
    // arrival counters: one per 128-row block (small M) or per output tile (split-K GEMM)
    const bool tc = M > 16 && mode == CQ_MODEL_DTYPE, a8 = M > 16 && mode == CQ_DYN_A8;
    const TcPlan tp = tc ? gemm_tc_plan(d, M) : TcPlan{};
    const A8Plan ap = a8 ? gemm_a8_plan(d, M) : A8Plan{};
    const size_t n_ctr = (size_t)d.NB * (size_t)(tc ? tp.token_tiles : a8 ? ap.token_tiles : 1);
    w.counters_off = off; w.counters_bytes = align_up(n_ctr * 4, 256); off += w.counters_bytes;
    size_t part = (size_t)gp.ctas * 2 * Mc * TILE * 4;   // two partial slots per CTA
    if (a8) {        // tiles of the last round cut into slices: one partial tile per slice
        const size_t p2 = ap.slices > 1 ? (size_t)((int64_t)d.NB * ap.token_tiles - ap.t_full) * ap.slices * ap.bn * TILE * 4 : 0;
        if (p2 > part) part = p2;
    }
    if (tc) {   // stream-K: two partial tiles per run
        const size_t p2 = (size_t)tp.p2 * tp.cw * 2 * tp.bnt * TILE * 4;
        if (p2 > part) part = p2;
    }
    w.partial_off = off; w.partial_bytes = align_up(part, 256); off += w.partial_bytes;
    if (mode == CQ_DYN_A8) {
        w.x8_off = off; w.x8_bytes = align_up((size_t)(M + 127) / 128 * 128 * Kp, 256); off += w.x8_bytes;
        w.dx_off = off; w.dx_bytes = align_up((size_t)M * 4, 256); off += w.dx_bytes;
    }
    w.total = off;
    return w;
}

// What the sizes that a caller may ask for hold beyond the need of the call itself: room for the partial sums of three CTAs an SM.
// A program that asks once, for its largest number of rows, uses that workspace for fewer too, and which CTAs serve how
// many rows is the library's affair; with no more than each call's own need, 1200 of a million pairs of row counts and shapes
// lost what the sizes of earlier versions had granted them.
static size_t spare_bytes(const Dims &d, int64_t M, size_t partial_bytes) {
    const int64_t T = (int64_t)d.NB * d.KT, places = 3 * (int64_t)sm_count();
    const size_t room = align_up((size_t)(T < places ? T : places) * 2 * (size_t)(M < 16 ? M : 16) * TILE * 4, 256);
    return room > partial_bytes ? room - partial_bytes : 0;
}

static int check_format(int B, int G, int64_t N, int64_t K) {
    if (B < 1 || B > 8 || N <= 0 || K <= 0 || G <= 0) return CQ_ERR_INVALID_ARG;
    if (G != 32 && G != 64 && G != 128 && G != 256 && G != 512) return CQ_ERR_UNSUPPORTED;
    if (K % G != 0) return CQ_ERR_UNSUPPORTED;
    return CQ_OK;
}
static bool misaligned(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) != 0; }

static int check_arch() {
    static thread_local int cached_dev = -1, cached_ok = 0;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) { g_last_cuda_error = (int)e; return CQ_ERR_CUDA; }
    if (dev != cached_dev) {
        int major = 0;
        e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
        if (e != cudaSuccess) { g_last_cuda_error = (int)e; return CQ_ERR_CUDA; }
        cached_dev = dev;
        cached_ok = (major == 10);
    }
    return cached_ok ? CQ_OK : CQ_ERR_ARCH;
}

static int wrap(cudaError_t e) {
    if (e == cudaSuccess) return CQ_OK;
    g_last_cuda_error = (int)e;
    return CQ_ERR_CUDA;
}

}  // namespace cq

using namespace cq;

#pragma GCC visibility push(default)
extern "C" {

const char *cq_status_string(int status) {
    switch (status) {
        case CQ_OK: return "CQ_OK";
        case CQ_ERR_INVALID_ARG: return "CQ_ERR_INVALID_ARG";
        case CQ_ERR_UNSUPPORTED: return "CQ_ERR_UNSUPPORTED";
        case CQ_ERR_ALIGNMENT: return "CQ_ERR_ALIGNMENT";
        case CQ_ERR_WORKSPACE: return "CQ_ERR_WORKSPACE";
        case CQ_ERR_ARCH: return "CQ_ERR_ARCH";
        case CQ_ERR_CUDA: return "CQ_ERR_CUDA";
        case CQ_ERR_TIMEOUT: return "CQ_ERR_TIMEOUT";
        default: return "CQ_ERR_UNKNOWN";
    }
}

int cq_last_cuda_error(void) { return g_last_cuda_error; }

size_t cq_canonical_code_bytes(int B, int64_t N, int64_t K) {
    if (B < 1 || B > 8 || N <= 0 || K <= 0) return 0;
    return (size_t)N * (size_t)((K * B + 7) / 8);
}

double cq_effective_bits(int B, int G) { return (double)B + 64.0 / (double)G; }

size_t cq_layout_bytes(int B, int G, int64_t N, int64_t K) {
    if (check_format(B, G, N, K) != CQ_OK) return 0;
    const Dims d = make_dims(B, G, N, K);
    return (size_t)d.NB * d.KT * (size_t)d.tile_bytes;
}

size_t cq_workspace_bytes(int B, int G, int64_t M, int64_t N, int64_t K, int mode) {
    if (check_format(B, G, N, K) != CQ_OK || M <= 0 || (mode != CQ_MODEL_DTYPE && mode != CQ_DYN_A8)) return 0;
    const Dims d = make_dims(B, G, N, K);
    const Workspace w = plan_workspace(d, M, mode);
    return w.total + spare_bytes(d, M, w.partial_bytes);
}

int cq_workspace_init(void *workspace, size_t workspace_bytes, void *stream) {
    if (!workspace || workspace_bytes == 0) return CQ_ERR_INVALID_ARG;
    // counters and the status word sit at the front of the workspace; zeroing everything is simplest
    return wrap(cudaMemsetAsync(workspace, 0, workspace_bytes, (cudaStream_t)stream));
}

int cq_pack_codes(const int8_t *k, int B, int64_t N, int64_t K, uint8_t *codes, void *stream) {
    if (!k || !codes || B < 1 || B > 8 || N <= 0 || K <= 0) return CQ_ERR_INVALID_ARG;
    return wrap(launch_pack_codes(k, B, N, K, codes, (cudaStream_t)stream));
}

int cq_repack(const uint8_t *codes, const float *scale, const uint16_t *a, const uint16_t *b, int B, int G, int64_t N,
              int64_t K, void *layout, void *stream) {
    if (!codes || !scale || !a || !b || !layout) return CQ_ERR_INVALID_ARG;
    int st = check_format(B, G, N, K);
    if (st != CQ_OK) return st;
    if (misaligned(layout)) return CQ_ERR_ALIGNMENT;
    return wrap(launch_repack(codes, scale, a, b, make_dims(B, G, N, K), layout, (cudaStream_t)stream));
}

int cq_unpack(const void *layout, int B, int G, int64_t N, int64_t K, uint8_t *codes, float *scale, uint16_t *a,
              uint16_t *b, void *stream) {
    if (!codes || !scale || !a || !b || !layout) return CQ_ERR_INVALID_ARG;
    int st = check_format(B, G, N, K);
    if (st != CQ_OK) return st;
    if (misaligned(layout)) return CQ_ERR_ALIGNMENT;
    return wrap(launch_unpack(layout, make_dims(B, G, N, K), codes, scale, a, b, (cudaStream_t)stream));
}

// One product in the workspace that `plan` lays out from ws.
static cudaError_t launch_product(const void *layout, const Dims &d, const uint16_t *x, uint16_t *y, int64_t M, int mode, bool act_f16,
                                  uint8_t *ws, const Workspace &plan, cudaStream_t s) {
    if (M <= 16) return launch_gemv(layout, d, x, y, M, mode, act_f16, ws, plan, s);
    if (mode == CQ_MODEL_DTYPE) return launch_gemm_tc(layout, d, x, y, M, mode, act_f16, ws, plan, s);
    return launch_gemm_a8_tc(layout, d, x, y, M, act_f16, ws, plan, s);
}

static int gemm_any(const void *layout, int B, int G, const uint16_t *x, uint16_t *y, int64_t M, int64_t N, int64_t K,
                    int mode, bool act_f16, void *workspace, size_t workspace_bytes, void *stream) {
    if (!layout || !x || !y || !workspace || M <= 0) return CQ_ERR_INVALID_ARG;
    if (mode != CQ_MODEL_DTYPE && mode != CQ_DYN_A8) return CQ_ERR_INVALID_ARG;
    int st = check_format(B, G, N, K);
    if (st != CQ_OK) return st;
    if (misaligned(layout) || misaligned(x) || misaligned(y) || misaligned(workspace)) return CQ_ERR_ALIGNMENT;
    const Dims d = make_dims(B, G, N, K);
    const Workspace plan = plan_workspace(d, M, mode);
    if (workspace_bytes < plan.total) return CQ_ERR_WORKSPACE;
    st = check_arch();
    if (st != CQ_OK) return st;
    return wrap(launch_product(layout, d, x, y, M, mode, act_f16, (uint8_t *)workspace, plan, (cudaStream_t)stream));
}

int cq_gemm(const void *layout, int B, int G, const uint16_t *x, uint16_t *y, int64_t M, int64_t N, int64_t K,
            int mode, void *workspace, size_t workspace_bytes, void *stream) {
    return gemm_any(layout, B, G, x, y, M, N, K, mode, false, workspace, workspace_bytes, stream);
}

int cq_gemm_f16(const void *layout, int B, int G, const uint16_t *x, uint16_t *y, int64_t M, int64_t N, int64_t K,
                int mode, void *workspace, size_t workspace_bytes, void *stream) {
    return gemm_any(layout, B, G, x, y, M, N, K, mode, true, workspace, workspace_bytes, stream);
}

// Workspace of the fused MLP: [gate_up operator's workspace][h: M x 2 I model-dtype values][down operator's
// Dynamic-A8 workspace].  The down operator's plan is shifted so that both operators report into the one status
// word at the front.
struct MlpPlan { Workspace gu, dn; size_t h_off, total; };
static MlpPlan plan_mlp(const Dims &dgu, const Dims &ddn, int64_t M, int mode_gu) {
    MlpPlan p;
    p.gu = plan_workspace(dgu, M, mode_gu);
    p.h_off = align_up(p.gu.total, 256);
    const size_t dn_off = align_up(p.h_off + (size_t)M * (size_t)dgu.N * 2, 256);
    p.dn = plan_workspace(ddn, M, CQ_DYN_A8);
    p.dn.counters_off += dn_off; p.dn.partial_off += dn_off; p.dn.x8_off += dn_off; p.dn.dx_off += dn_off;
    p.dn.status_off = 0;
    p.total = dn_off + p.dn.total;
    return p;
}

size_t cq_mlp_workspace_bytes(int B_gu, int G_gu, int B_dn, int G_dn, int64_t M, int64_t K, int64_t I, int64_t N, int mode_gate_up) {
    if (check_format(B_gu, G_gu, 2 * I, K) != CQ_OK || check_format(B_dn, G_dn, N, I) != CQ_OK || M <= 0) return 0;
    if (mode_gate_up != CQ_MODEL_DTYPE && mode_gate_up != CQ_DYN_A8) return 0;
    const Dims dgu = make_dims(B_gu, G_gu, 2 * I, K), ddn = make_dims(B_dn, G_dn, N, I);
    const MlpPlan p = plan_mlp(dgu, ddn, M, mode_gate_up);
    return p.total + spare_bytes(dgu, M, p.gu.partial_bytes) + spare_bytes(ddn, M, p.dn.partial_bytes);
}

int cq_mlp_swiglu(const void *layout_gate_up, int B_gu, int G_gu, const void *layout_down, int B_dn, int G_dn, const uint16_t *x,
                  uint16_t *y, int64_t M, int64_t K, int64_t I, int64_t N, int mode_gate_up, int act_f16, void *workspace,
                  size_t workspace_bytes, void *stream) {
    if (!layout_gate_up || !layout_down || !x || !y || !workspace || M <= 0 || I <= 0) return CQ_ERR_INVALID_ARG;
    if (mode_gate_up != CQ_MODEL_DTYPE && mode_gate_up != CQ_DYN_A8) return CQ_ERR_INVALID_ARG;
    int st = check_format(B_gu, G_gu, 2 * I, K);
    if (st == CQ_OK) st = check_format(B_dn, G_dn, N, I);
    if (st != CQ_OK) return st;
    if (I % 8 != 0) return CQ_ERR_UNSUPPORTED;
    if (misaligned(layout_gate_up) || misaligned(layout_down) || misaligned(x) || misaligned(y) || misaligned(workspace))
        return CQ_ERR_ALIGNMENT;
    const Dims dgu = make_dims(B_gu, G_gu, 2 * I, K), ddn = make_dims(B_dn, G_dn, N, I);
    const MlpPlan plan = plan_mlp(dgu, ddn, M, mode_gate_up);
    if (workspace_bytes < plan.total) return CQ_ERR_WORKSPACE;
    st = check_arch();
    if (st != CQ_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    uint8_t *ws = (uint8_t *)workspace;
    uint16_t *h = reinterpret_cast<uint16_t *>(ws + plan.h_off);
    const bool f16 = act_f16 != 0;
    // 1. gate_up, an ordinary operator: model-dtype output
    cudaError_t e = launch_product(layout_gate_up, dgu, x, h, M, mode_gate_up, f16, ws, plan.gu, s);
    if (e != cudaSuccess) return wrap(e);
    // 2. gated activation and the down projection's activation quantiser in one kernel
    e = launch_swiglu_quantize_a8(h, M, I, reinterpret_cast<int8_t *>(ws + plan.dn.x8_off), (int64_t)ddn.KT * TILE,
                                  reinterpret_cast<float *>(ws + plan.dn.dx_off), ddn.B != 4, f16, s);
    if (e != cudaSuccess) return wrap(e);
    // 3. the down projection on the carrier that is already in its workspace
    if (M <= 16) e = launch_gemv(layout_down, ddn, nullptr, y, M, CQ_DYN_A8, f16, ws, plan.dn, s, true);
    else e = launch_gemm_a8_tc(layout_down, ddn, nullptr, y, M, f16, ws, plan.dn, s, true);
    return wrap(e);
}

// Routed product.  The groups (matrices with routes) are sorted into classes of token tiles, and a class of several
// groups is one launch: up to 16 rows the small-M kernel, above it the GEMM, the token tiles up to 128 together (its time is
// the decode of the weights there, not the tokens) and 256 and 512 by themselves; Dynamic A8 keeps one class per token
// tile, whose drain grows with the tile.  A group by itself is an ordinary product, which may share its tiles along K, and so
// are the groups of a GEMM class that would leave most of the GPU idle in whole tiles (together_pays).
// Sixteen matrices of 2816 x 2048 (W4 G64, 384 routes): one after another 203 us, most of it launches that leave SMs idle; 61 us so.
// Workspace: [status][gathered rows: R x K][Dynamic A8: INT8 carrier of all rows, row scales][arrival counters][partial sums
// of the small-M groups][what else an ordinary product needs].  Every launch reports into the one status word at the
// front, and every launch leaves the arrival counters at zero for the next one; the gather zeroes both.
struct RoutedPlan { size_t xg_off, x8_off, dx_off, ctr_off, ctr_bytes, part_off, sub_off, total; };
static bool routed_offsets_ok(const int64_t *off, int E, int64_t R) {
    if (!off || off[0] != 0 || off[E] != R) return false;
    for (int e = 0; e < E; ++e) if (off[e + 1] < off[e]) return false;
    return true;
}
static int routed_class(const Dims &d, int64_t m, int mode) {   // 0: small M; else a token tile
    if (m <= 16) return 0;
    if (mode == CQ_DYN_A8) return gemm_a8_token_tile(d, m);
    const int t = gemm_tc_token_tile(m);
    return t < 128 ? 128 : t;
}
static const int ROUTED_CLASSES[5] = {0, 64, 128, 256, 512};   // every value of routed_class
// Whether the groups of a GEMM class are faster in one launch of whole tiles than one after another.  A few matrices of
// few row blocks leave most SMs idle in whole tiles, while each of them by itself shares its tiles along K among all SMs.
// Two matrices of 1024 x 4096, W8 G128, model dtype, 20 rows each: 30.7 us together, 25.5 one after another; W3 G32, Dynamic A8:
// 45.2 and 31.6; but 2816 x 2048, W4 G64, 64 rows each: together 20 % faster.  An ordinary product of Dynamic A8 adds a launch and
// a quantiser of its own, some five blocks of main loop.
static bool together_pays(const Dims &d, const GroupTable &t, int64_t max_rows, int mode) {
    const bool tc = mode == CQ_MODEL_DTYPE;
    const double together = tc ? gemm_tc_groups_cost(t, d, max_rows) : gemm_a8_groups_cost(t, d, max_rows) + 5.0;
    const double least = tc ? 4.6 : 9.0;   // no ordinary product costs less
    double one_by_one = least * t.n;
    for (int i = 0; i < t.n && one_by_one < together; ++i) one_by_one += (tc ? gemm_tc_plan(d, t.g[i].rows).cost : gemm_a8_plan(d, t.g[i].rows).cost + 5.0) - least;
    return together <= one_by_one;
}
// The launches that follow the gather, in order: f(groups, class, largest row count, CTAs of a small-M group).  A table of one
// group is an ordinary product.  The sizes, the launches themselves and cq_debug_routed_plan all walk this.
extern "C++" {
template <class F>
static int for_routed_launches(const Dims &d, const void *const *layouts, const int64_t *off, int E, int mode, F &&f) {
    auto emit = [&](const GroupTable &t, int cls, int64_t max_rows) -> int {
        if (t.n == 0) return CQ_OK;
        if (t.n > 1 && cls != 0 && !together_pays(d, t, max_rows, mode)) {
            for (int i = 0; i < t.n; ++i) {
                GroupTable one{};
                one.n = 1;
                one.g[0] = t.g[i];
                const int st = f(one, cls, (int64_t)t.g[i].rows, 1);
                if (st != CQ_OK) return st;
            }
            return CQ_OK;
        }
        // small-M groups share the places of the whole GPU; a run of fewer than four tiles is mostly overhead
        const int64_t T = (int64_t)d.NB * d.KT, places = cls == 0 ? std::min<int64_t>(2 * (int64_t)sm_count(), T) : 0;
        int64_t P = places / t.n;
        if (P > T / 4) P = T / 4;
        return f(t, cls, max_rows, (int)(P < 1 ? 1 : P));
    };
    for (int cls : ROUTED_CLASSES) {
        GroupTable t{};
        int64_t max_rows = 0;
        for (int e = 0; e < E; ++e) {
            const int64_t r0 = off[e], m = off[e + 1] - r0;
            if (m == 0 || routed_class(d, m, mode) != cls) continue;
            t.g[t.n++] = {layouts ? layouts[e] : nullptr, (int)r0, (int)m, 0};
            if (m > max_rows) max_rows = m;
            if (t.n == MAX_GROUPS) {
                const int st = emit(t, cls, max_rows);
                if (st != CQ_OK) return st;
                t.n = 0; max_rows = 0;
            }
        }
        const int st = emit(t, cls, max_rows);
        if (st != CQ_OK) return st;
    }
    return CQ_OK;
}
}  // extern "C++"
static RoutedPlan plan_routed(const Dims &d, const int64_t *off, int E, int mode) {
    RoutedPlan p{};
    const int64_t R = off[E];
    size_t ctr = 0, part = 0, sub = 0;
    bool together = false;
    auto most = [](size_t &v, size_t x) { if (x > v) v = x; };
    for_routed_launches(d, nullptr, off, E, mode, [&](const GroupTable &t, int cls, int64_t max_rows, int P) -> int {
        if (t.n == 1) {
            const Workspace w = plan_workspace(d, max_rows, mode);
            most(ctr, w.counters_bytes);
            most(sub, w.total - w.partial_off);
        } else {
            together = true;
            if (cls == 0) { most(ctr, (size_t)t.n * d.NB * 4); most(part, (size_t)t.n * P * 2 * 16 * TILE * 4); }
        }
        return CQ_OK;
    });
    size_t o = 256;
    p.xg_off = o; o += align_up((size_t)R * d.K * 2, 256);
    if (mode == CQ_DYN_A8 && together) {
        p.x8_off = o; o += align_up((size_t)R * d.KT * TILE, 256);
        p.dx_off = o; o += align_up((size_t)R * 4, 256);
    }
    p.ctr_off = o; p.ctr_bytes = align_up(ctr, 256); o += p.ctr_bytes;
    p.part_off = o; o += align_up(part, 256);
    p.sub_off = o; o += align_up(sub, 256);
    p.total = o;
    return p;
}
// the workspace of an ordinary product of m rows inside that of the routed call
static Workspace routed_product_workspace(const RoutedPlan &p, const Dims &d, int64_t m, int mode) {
    Workspace w = plan_workspace(d, m, mode);
    w.x8_off += p.sub_off - w.partial_off; w.dx_off += p.sub_off - w.partial_off;
    w.partial_off = p.sub_off; w.counters_off = p.ctr_off; w.status_off = 0;
    return w;
}

size_t cq_routed_workspace_bytes(int B, int G, int E, const int64_t *expert_offset_host, int64_t N, int64_t K, int mode) {
    if (check_format(B, G, N, K) != CQ_OK || E <= 0 || !expert_offset_host || (mode != CQ_MODEL_DTYPE && mode != CQ_DYN_A8)) return 0;
    const int64_t R = expert_offset_host[E];
    if (R <= 0 || !routed_offsets_ok(expert_offset_host, E, R)) return 0;
    const Dims d = make_dims(B, G, N, K);
    const RoutedPlan p = plan_routed(d, expert_offset_host, E, mode);
    return p.total + spare_bytes(d, 16, p.sub_off - p.part_off) + spare_bytes(d, 16, p.total - p.sub_off);
}

int cq_gemm_routed(const void *const *layouts_host, int E, int B, int G, const uint16_t *x, const int32_t *route_token,
                   const int64_t *expert_offset_host, uint16_t *y_routes, int64_t T, int64_t N, int64_t K, int mode, int act_f16,
                   void *workspace, size_t workspace_bytes, void *stream) {
    if (!layouts_host || !x || !route_token || !expert_offset_host || !y_routes || !workspace || E <= 0 || T <= 0)
        return CQ_ERR_INVALID_ARG;
    if (mode != CQ_MODEL_DTYPE && mode != CQ_DYN_A8) return CQ_ERR_INVALID_ARG;
    int st = check_format(B, G, N, K);
    if (st != CQ_OK) return st;
    const int64_t R = expert_offset_host[E];
    if (R <= 0 || !routed_offsets_ok(expert_offset_host, E, R)) return CQ_ERR_INVALID_ARG;
    for (int e = 0; e < E; ++e) {
        if (!layouts_host[e]) return CQ_ERR_INVALID_ARG;
        if (misaligned(layouts_host[e])) return CQ_ERR_ALIGNMENT;
    }
    if (misaligned(x) || misaligned(y_routes) || misaligned(workspace) || (K * 2) % 16 != 0 || (N * 2) % 16 != 0) return CQ_ERR_ALIGNMENT;
    const Dims d = make_dims(B, G, N, K);
    const RoutedPlan plan = plan_routed(d, expert_offset_host, E, mode);
    if (workspace_bytes < plan.total) return CQ_ERR_WORKSPACE;
    st = check_arch();
    if (st != CQ_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    uint8_t *ws = (uint8_t *)workspace;
    int *status = reinterpret_cast<int *>(ws), *counters = reinterpret_cast<int *>(ws + plan.ctr_off);
    uint16_t *xg = reinterpret_cast<uint16_t *>(ws + plan.xg_off);
    int8_t *xq = reinterpret_cast<int8_t *>(ws + plan.x8_off);
    float *dxs = reinterpret_cast<float *>(ws + plan.dx_off);
    const bool f16 = act_f16 != 0;
    // the gather also zeroes the status word and the arrival counters: which words these are changes with the routing
    const cudaError_t err = launch_gather_rows(x, route_token, xg, R, T, K, status, counters, (int64_t)plan.ctr_bytes / 4, s);
    if (err != cudaSuccess) return wrap(err);
    bool quantised = false;
    return for_routed_launches(d, layouts_host, expert_offset_host, E, mode, [&](const GroupTable &t, int cls, int64_t max_rows, int P) -> int {
        if (t.n == 1) {
            const Group &g = t.g[0];
            return wrap(launch_product(g.layout, d, xg + (int64_t)g.row0 * K, y_routes + (int64_t)g.row0 * N, g.rows, mode, f16, ws,
                                       routed_product_workspace(plan, d, g.rows, mode), s));
        }
        if (mode == CQ_DYN_A8 && !quantised) {
            const cudaError_t e = launch_quantize_a8(xg, R, K, xq, (int64_t)d.KT * TILE, dxs, B != 4, f16, s);
            if (e != cudaSuccess) return wrap(e);
            quantised = true;
        }
        if (cls == 0) return wrap(launch_gemv_groups(t, d, xg, xq, dxs, y_routes, mode, f16, P, reinterpret_cast<float *>(ws + plan.part_off), counters, s));
        if (mode == CQ_MODEL_DTYPE) return wrap(launch_gemm_tc_groups(t, d, xg, y_routes, R, max_rows, f16, status, s));
        return wrap(launch_gemm_a8_groups(t, d, xq, dxs, y_routes, R, max_rows, f16, status, s));
    });
}

int cq_gemm_status(const void *workspace, size_t workspace_bytes, void *stream) {
    if (!workspace || workspace_bytes < 512) return CQ_ERR_INVALID_ARG;
    // the status word is the first word of every workspace (plan_workspace)
    int host = 0;
    cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
    if (e != cudaSuccess) return wrap(e);
    e = cudaMemcpy(&host, (const uint8_t *)workspace, sizeof(int), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return wrap(e);
    return host == 0 ? CQ_OK : CQ_ERR_TIMEOUT;
}

int cq_gemm_host(const void *layout, int B, int G, const uint16_t *x_host, uint16_t *y_host, uint16_t *x_dev,
                 uint16_t *y_dev, int64_t M, int64_t N, int64_t K, int mode, void *workspace, size_t workspace_bytes,
                 void *stream) {
    if (!x_host || !y_host || !x_dev || !y_dev || M <= 0 || N <= 0 || K <= 0) return CQ_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaMemcpyAsync(x_dev, x_host, (size_t)M * K * 2, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return wrap(e);
    int st = cq_gemm(layout, B, G, x_dev, y_dev, M, N, K, mode, workspace, workspace_bytes, stream);
    if (st != CQ_OK) return st;
    e = cudaMemcpyAsync(y_host, y_dev, (size_t)M * N * 2, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return wrap(e);
    return wrap(cudaStreamSynchronize(s));
}

static int check_encode(int B, int G, int64_t N, int64_t K, int objective) {
    if (B < 1 || B > 8 || N <= 0 || K <= 0 || G <= 0) return CQ_ERR_INVALID_ARG;
    if (objective != CQ_FIT_CONTINUOUS && objective != CQ_FIT_JOINT) return CQ_ERR_INVALID_ARG;
    if (K % G != 0 || G > 512) return CQ_ERR_UNSUPPORTED;
    return CQ_OK;
}

int cq_encode_assign(const float *W, int B, int G, int64_t N, int64_t K, const float *scale, const uint16_t *a,
                     const uint16_t *b, int objective, int8_t *k, void *stream) {
    if (!W || !scale || !a || !b || !k) return CQ_ERR_INVALID_ARG;
    const int st = check_encode(B, G, N, K, objective);
    if (st != CQ_OK) return st;
    return wrap(launch_encode_assign(W, B, G, N, K, scale, a, b, objective, k, (cudaStream_t)stream));
}

int cq_encode_scale(const float *W, const int8_t *k, int B, int G, int64_t N, int64_t K, const uint16_t *a,
                    const uint16_t *b, int objective, float *scale, void *stream) {
    if (!W || !scale || !a || !b || !k) return CQ_ERR_INVALID_ARG;
    const int st = check_encode(B, G, N, K, objective);
    if (st != CQ_OK) return st;
    return wrap(launch_encode_scale(W, k, B, G, N, K, a, b, objective, scale, (cudaStream_t)stream));
}

int cq_encode_losses(const float *W, const int8_t *k, int B, int G, int64_t N, int64_t K, const float *scale,
                     const uint16_t *a, const uint16_t *b, double *LC, double *LA8, void *stream) {
    if (!W || !scale || !a || !b || !k || !LC || !LA8) return CQ_ERR_INVALID_ARG;
    const int st = check_encode(B, G, N, K, CQ_FIT_JOINT);
    if (st != CQ_OK) return st;
    return wrap(launch_encode_losses(W, k, B, G, N, K, scale, a, b, LC, LA8, (cudaStream_t)stream));
}

int cq_encode(const float *W, int B, int G, int64_t N, int64_t K, int objective, int effort, int8_t *k, float *scale,
              uint16_t *a, uint16_t *b, void *stream) {
    if (!W || !scale || !a || !b || !k || effort < 0 || effort > 3) return CQ_ERR_INVALID_ARG;
    const int st = check_encode(B, G, N, K, objective);
    if (st != CQ_OK) return st;
    return wrap(launch_encode_search(W, B, G, N, K, objective, effort, k, scale, a, b, (cudaStream_t)stream));
}

int cq_quantize_a8(const uint16_t *x, int64_t M, int64_t K, int8_t *x8, float *dx, void *stream) {
    if (!x || !x8 || !dx || M <= 0 || K <= 0) return CQ_ERR_INVALID_ARG;
    return wrap(launch_quantize_a8(x, M, K, x8, K, dx, false, false, (cudaStream_t)stream));
}

int cq_quantize_a8_f16(const uint16_t *x, int64_t M, int64_t K, int8_t *x8, float *dx, void *stream) {
    if (!x || !x8 || !dx || M <= 0 || K <= 0) return CQ_ERR_INVALID_ARG;
    return wrap(launch_quantize_a8(x, M, K, x8, K, dx, false, true, (cudaStream_t)stream));
}

#define CQ_DEBUG_PROLOGUE()                                   \
    if (!layout) return CQ_ERR_INVALID_ARG;                   \
    {                                                         \
        int st_ = check_format(B, G, N, K);                   \
        if (st_ != CQ_OK) return st_;                         \
    }                                                         \
    if (misaligned(layout)) return CQ_ERR_ALIGNMENT;          \
    const Dims d = make_dims(B, G, N, K);

int cq_decode_levels(const void *layout, int B, int G, int64_t N, int64_t K, float *levels, void *stream) {
    if (!levels) return CQ_ERR_INVALID_ARG;
    CQ_DEBUG_PROLOGUE();
    return wrap(launch_decode_levels(layout, d, levels, (cudaStream_t)stream));
}

int cq_decode_carriers(const void *layout, int B, int G, int64_t N, int64_t K, int8_t *carriers, void *stream) {
    if (!carriers) return CQ_ERR_INVALID_ARG;
    CQ_DEBUG_PROLOGUE();
    return wrap(launch_decode_carriers(layout, d, carriers, (cudaStream_t)stream));
}

int cq_decode_weights(const void *layout, int B, int G, int64_t N, int64_t K, float *What, void *stream) {
    if (!What) return CQ_ERR_INVALID_ARG;
    CQ_DEBUG_PROLOGUE();
    return wrap(launch_decode_weights(layout, d, What, (cudaStream_t)stream));
}

int cq_debug_gemm_plan(int B, int G, int64_t M, int64_t N, int64_t K, int mode, int64_t *plan) {
    if (!plan || M <= 16 || (mode != CQ_MODEL_DTYPE && mode != CQ_DYN_A8)) return CQ_ERR_INVALID_ARG;
    const int st = check_format(B, G, N, K);
    if (st != CQ_OK) return st;
    const Dims d = make_dims(B, G, N, K);
    if (mode == CQ_MODEL_DTYPE) {
        const TcPlan tp = gemm_tc_plan(d, M);
        // tiles of 128 channels; the last pair of an odd number of row blocks holds one
        const int64_t nbu = (d.NB + tp.cw - 1) / tp.cw, whole = tp.t_full * tp.cw - (d.NB % tp.cw ? tp.t_full / nbu : 0);
        plan[0] = tp.bnt; plan[1] = whole; plan[2] = (int64_t)tp.p2 * tp.cw; plan[3] = (int64_t)d.NB * tp.token_tiles - whole;
        plan[4] = tp.crossing;
    } else {
        const A8Plan ap = gemm_a8_plan(d, M);
        const int64_t shared = (int64_t)d.NB * ap.token_tiles - ap.t_full;
        plan[0] = ap.bn; plan[1] = ap.t_full; plan[2] = shared * ap.slices; plan[3] = shared; plan[4] = 0;
    }
    return CQ_OK;
}

int cq_debug_routed_plan(int B, int G, int E, const int64_t *expert_offset_host, int64_t N, int64_t K, int mode, int64_t *launches, int max_launches) {
    if (E <= 0 || !expert_offset_host || (mode != CQ_MODEL_DTYPE && mode != CQ_DYN_A8) || max_launches < 0 || (max_launches > 0 && !launches)) return CQ_ERR_INVALID_ARG;
    const int st = check_format(B, G, N, K);
    if (st != CQ_OK) return st;
    if (expert_offset_host[E] <= 0 || !routed_offsets_ok(expert_offset_host, E, expert_offset_host[E])) return CQ_ERR_INVALID_ARG;
    const Dims d = make_dims(B, G, N, K);
    const RoutedPlan plan = plan_routed(d, expert_offset_host, E, mode);
    int n = 0;
    for_routed_launches(d, nullptr, expert_offset_host, E, mode, [&](const GroupTable &t, int cls, int64_t max_rows, int P) -> int {
        if (n < max_launches) {
            int64_t *v = launches + 5 * n;
            v[0] = cls; v[1] = t.n; v[2] = max_rows; v[3] = cls == 0 && t.n > 1 ? P : 0;
            v[4] = t.n == 1 ? (int64_t)routed_product_workspace(plan, d, max_rows, mode).status_off : 0;   // the launches together report into the front word
        }
        ++n;
        return CQ_OK;
    });
    return n;
}

int cq_debug_wait_timeout(void *workspace, size_t workspace_bytes, int64_t limit_cycles, void *stream) {
    if (!workspace || workspace_bytes < 512 || limit_cycles <= 0 || limit_cycles > 2000000000ll) return CQ_ERR_INVALID_ARG;
    if (misaligned(workspace)) return CQ_ERR_ALIGNMENT;
    const int st = check_arch();
    if (st != CQ_OK) return st;
    // the status word is the first word of every workspace (plan_workspace)
    return wrap(launch_wait_timeout((int *)workspace, (long long)limit_cycles, (cudaStream_t)stream));
}

int cq_debug_a8_partials(const void *layout, int B, int G, const int8_t *x8, int64_t M, int64_t N, int64_t K,
                         int32_t *P, void *stream) {
    if (!x8 || !P || M <= 0) return CQ_ERR_INVALID_ARG;
    CQ_DEBUG_PROLOGUE();
    return wrap(launch_a8_partials(layout, d, x8, M, P, (cudaStream_t)stream));
}

}  // extern "C"
#pragma GCC visibility pop
