// Large-M packed GEMM on the 5th-generation tensor cores (Section 5.3 dense path, re-done for
// sm_100a): weights stay packed in HBM and are decoded into bf16 shared-memory operand tiles
// right before tcgen05.mma consumes them; accumulators live in TMEM.
//
// Roles inside a CTA (output tiles of 128 channels x BN tokens; above 128 tokens two CTAs may share one stream of MMAs over 256
// channels x 256 or 512 tokens):
//   warp 0      TMA-loads activation tiles x[BN x 64] (128-byte swizzle) into a ring of stages; nothing but the wait
//               for a stage stands between the MMAs that free it and the copy that refills it
//   warp 18     bulk-copies raw layout tiles (codes + co-located group parameters) into their own ring (2-6 deep)
//   warp 1      allocates TMEM, issues tcgen05.mma (one elected lane), commits to mbarriers
//   warps 2..17 decode: raw tile -> s_g * q(|k|/M) * sign (Eq. cubic; W3 and W4 from tables of levels evaluated in fp32, the
//               other widths by the half2 Horner form of Eq. gpu-horner on the power-of-two-normalised code with the
//               scale in fp32), rounded to the activations' dtype and stored in
//               the K-major 128-byte-swizzled layout the MMA reads; then the epilogue
//               (tcgen05.ld -> bf16 -> y)
// Weights sit on the MMA's M side (TMEM lane = output channel), tokens on its N side, so any
// token count maps to a legal instruction shape and each epilogue thread owns one output channel.
//
// Every wait on an mbarrier is bounded: a wait that runs out sets a status word in global memory and a
// flag in shared memory, after which no role of the CTA waits any more; the CTA still walks its loops to
// the end, releases TMEM and exits.
//
// This file holds the plan (which tiles, and which CTA computes what) and the instantiations that compute one whole tile
// per CTA; cq_gemm_tc_sk.cu holds those that also share tiles between CTAs (stream-K); the kernel itself is
// in cq_gemm_tc_impl.cuh.
#include "cq_gemm_tc_impl.cuh"

namespace cq {

int gemm_tc_available() { return 1; }

// Token tile for M rows where it follows from the rows alone: up to 128 of an ordinary product, and the classes of a routed one.
int gemm_tc_token_tile(int64_t M) { return M <= 32 ? 32 : M <= 64 ? 64 : M <= 128 ? 128 : M <= 256 ? 256 : 512; }

namespace {

// Microseconds of a layout tile (128 channels x 128 k) in the main loop of a 256-token pair tile, by group size (128, 64, 32) and
// width: the decode, but for the narrow codes, which are at the 0.62 of the MMAs.  Measured as the slope over K of
// whole tiles in one round (N = 2048, K = 1024 and 8192); the other tiles are given relative to it below, within 0.05.
constexpr double TILE_US[3][8] = {{0.63, 0.64, 0.63, 0.66, 0.91, 0.91, 0.98, 0.80}, {0.63, 0.67, 0.78, 0.71, 0.95, 0.96, 1.03, 0.85},
                                  {0.65, 0.68, 0.87, 0.79, 1.02, 1.02, 1.06, 0.94}};
// A kind of output tile: its tokens, the CTAs that compute it together, and in microseconds what a launch of one round costs
// besides the main loop, a layout tile, and what sharing a tile between s runs adds: first + four * ceil(s / 4) + each * s (the
// partial tiles' way through L2, read by the last run to arrive in batches of four), and what a run that crosses from one
// tile into the next adds to that (a second fill and epilogue).
struct TileKind { int bnt, cw; double fixed, tile, first, four, each, cross; };
TileKind tile_kind(const Dims &d, int bnt, int cw) {
    const double t = TILE_US[d.gpt == 1 ? 0 : d.gpt == 2 ? 1 : 2][d.B - 1];
    if (bnt == 512) return {512, 2, 9.2, t + 0.2 > 1.11 ? t + 0.2 : 1.11, 7.9, 4.4, 1.45, 16.0};
    if (bnt == 256 && cw == 2) return {256, 2, 7.1, t, 5.7, 2.4, 0.7, 9.0};
    if (bnt == 256) return {256, 1, 6.4, t + (d.B <= 3 ? 0.04 : 0.1), 4.0, 2.4, 0.7, 9.0};
    if (bnt == 128) return {128, 1, 5.2, t - 0.02, 3.0, 1.5, 0.3, 4.5};
    return {bnt, 1, 4.6, t - (d.B == 4 ? 0.14 : 0.05), 2.0, 0.8, 0.2, 3.0};
}

// The plan with one kind of tile.  Whole tiles, a CTA or a pair each, fill the SMs round after round.  When the last
// round would leave SMs idle, its r tiles may be cut along K as well (stream-K), in one of two ways:
//   every tile into the same number s of runs, so that a run lies inside its tile; r s runs take ceil(r s / places) rounds;
//   one run per place, cut anywhere: the best balance, but most runs cross from one tile into the next.
// Wide tiles that all fit one round go by the microseconds of tile_kind.  Against every plan forced in turn (twelve shapes,
// 160 .. 2048 tokens, W1, W4 and W8), the costs of the best plans are met within 12 %.  The constants before them belonged to a
// kernel without pairs and cut too often and too fine: 1024 x 4096, W4, 1024 tokens 44.8 us in eight runs a tile, 37.2 in
// four; 2816 x 2048, 512 tokens 33.1 us shared, 27.1 whole.
// Up to 128 tokens, and behind whole rounds, the costs are in layout tiles: a whole tile KT + 4, a run its length + 4 .. 10 (cut
// evenly; the more the wider the token tile) or + 10 .. 22 (crossing); forced plans at 24, 64 and 128 tokens confirm them within 6 %.  The
// kernel that can share tiles runs about 5 % slower on every tile of the launch than the one that cannot (measured at
// M = 4096, N = 57344, K = 8192, and at M = 1024, N = 6144, K = 4096; merely compiling the partial-tile code into the kernel
// costs that much), so it is a separate instantiation and sharing has to save more.
TcPlan plan_with(const Dims &d, int64_t M, const TileKind &k) {
    TcPlan p;
    p.bnt = k.bnt; p.cw = k.cw;
    p.token_tiles = (int)((M + p.bnt - 1) / p.bnt);
    const int64_t NBU = (d.NB + p.cw - 1) / p.cw, T = NBU * p.token_tiles, sms = sm_count() > p.cw ? sm_count() / p.cw : 1;   // tiles and places for them
    const int64_t r = T % sms;                      // tiles of the last, partial round
    const double round_us = k.fixed + k.tile * (double)d.KT;
    p.t_full = T; p.p2 = 0; p.crossing = 0;
    p.cost = (double)(T / sms) * round_us;
    if (r != 0) {
        const int64_t V2 = r * d.KT;
        int64_t pa = sms;
        if (pa > V2 / 4) pa = V2 / 4;               // at least four layout tiles per run
        const bool micros = p.bnt >= 256 && T < sms;
        const double wide = (double)p.bnt / 512.0;   // the partial tiles grow with the token tile
        auto shared_us = [&](int64_t runs, double length, double contributors) {
            return (double)((runs + sms - 1) / sms) * (k.fixed + k.tile * length) + k.first + k.four * (double)(int64_t)((contributors + 3.0) / 4.0) + k.each * contributors;
        };
        double best = 1e30, best_us = 1e30;
        int64_t best_p2 = 0;
        int best_crossing = 0;
        for (int64_t s = 2; s <= 16 && s * 4 <= d.KT; ++s) {
            const double us = shared_us(r * s, (double)((d.KT + s - 1) / s), (double)s);
            const double c = micros ? us : (double)((r * s + sms - 1) / sms) * ((double)d.KT / (double)s + 4.0 + 6.0 * wide);
            if (c < best) { best = c; best_us = us; best_p2 = r * s; best_crossing = 0; }
        }
        if (pa > r) {
            const double length = (double)V2 / (double)pa, us = shared_us(pa, length, (double)(int64_t)((double)d.KT / length + 1.99)) + k.cross;
            const double c = micros ? us : length + 10.0 + 12.0 * wide;
            if (c < best) { best = c; best_us = us; best_p2 = pa; best_crossing = 1; }
        }
        const double whole = micros ? round_us : (double)(d.KT + 4), all = (double)(T / sms + 1) * whole;
        if (best_p2 > 0 && (whole - best) / all > (micros ? 0.03 : 0.06)) { p.p2 = (int)best_p2; p.crossing = best_crossing; p.t_full = T - r; }
        p.cost += p.p2 > 0 && best_us < round_us ? best_us : round_us;
    }
    p.ctas = (int)(p.t_full + p.p2) * p.cw;
    p.stream_k = p.p2 > 0;
    return p;
}

}  // namespace

// Above 128 tokens three kinds of tile compete: 256 tokens by a pair, 256 by one CTA (finer, and cheaper to share, where pairs
// leave SMs idle), and 512 by a pair (every decoded weight serves twice the tokens, which the costs know only in part: the power limit
// favours it too, hence the larger margin).  4096 x 4096, W4, 512 tokens 39.3 us with 512-token tiles, 29.5 with 256.
TcPlan gemm_tc_plan(const Dims &d, int64_t M) {
    if (M <= 128) return plan_with(d, M, tile_kind(d, gemm_tc_token_tile(M), 1));
    TcPlan best = plan_with(d, M, tile_kind(d, 256, 2));
    const TcPlan single = plan_with(d, M, tile_kind(d, 256, 1));
    if (single.cost < 0.97 * best.cost) best = single;
    if (M > 256) {
        const TcPlan wide = plan_with(d, M, tile_kind(d, 512, 2));
        if (!(best.cost < 0.92 * wide.cost)) best = wide;
    }
    return best;
}

double gemm_tc_groups_cost(const GroupTable &groups, const Dims &d, int64_t tile_m) {
    const int bnt = gemm_tc_token_tile(tile_m), cw = bnt >= 256 ? 2 : 1;
    const TileKind k = tile_kind(d, bnt, cw);
    int64_t units = 0;
    for (int i = 0; i < groups.n; ++i) units += (int64_t)((d.NB + cw - 1) / cw) * ((groups.g[i].rows + bnt - 1) / bnt);
    const int64_t places = sm_count() > cw ? sm_count() / cw : 1;
    return (double)((units + places - 1) / places) * (k.fixed + k.tile * (double)d.KT);
}

// stream-K instantiations: cq_gemm_tc_sk.cu
cudaError_t launch_gemm_tc_streamk(const GroupTable &groups, const Dims &d, const uint16_t *x, uint16_t *y, int64_t M, const TcPlan &plan, int *status,
                                   float *partial, int *counters, bool act_f16, cudaStream_t st);

cudaError_t launch_gemm_tc(const void *layout, const Dims &d, const uint16_t *x, uint16_t *y, int64_t M, int mode,
                           bool act_f16, uint8_t *ws, const Workspace &plan, cudaStream_t st) {
    if (mode != 0) return cudaErrorNotSupported;
    int *status = reinterpret_cast<int *>(ws + plan.status_off);
    float *partial = reinterpret_cast<float *>(ws + plan.partial_off);
    int *counters = reinterpret_cast<int *>(ws + plan.counters_off);
    GroupTable one{};
    one.n = 1;
    one.g[0] = {layout, 0, (int)M, 0};
    const TcPlan tp = gemm_tc_plan(d, M);
    if (tp.p2 > 0) return launch_gemm_tc_streamk(one, d, x, y, M, tp, status, partial, counters, act_f16, st);
    return launch_tc_variant<false>(one, d, x, y, M, tp, status, partial, counters, act_f16, st);
}

cudaError_t launch_gemm_tc_groups(const GroupTable &groups, const Dims &d, const uint16_t *x, uint16_t *y, int64_t R, int64_t tile_m,
                                  bool act_f16, int *status, cudaStream_t st) {
    TcPlan plan{};   // whole tiles of the class; launch_bn counts them
    plan.bnt = gemm_tc_token_tile(tile_m); plan.cw = plan.bnt >= 256 ? 2 : 1;
    return launch_tc_variant<false>(groups, d, x, y, R, plan, status, nullptr, nullptr, act_f16, st);
}

}  // namespace cq
