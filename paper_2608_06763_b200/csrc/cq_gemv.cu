// Small-M products (M <= 16; one and two tokens in the model dtype have a kernel of their own, cq_gemv_strip.cu): packed
// weights streamed exactly once, warp-level tensor-core MMAs doing the multiply and the k reduction (Section 5.3 narrow-row
// path; Section 5.4 for Dynamic A8).
//
// Work decomposition: the NB x KT grid of 128 x 128 weight tiles is cut into P equal contiguous runs in row-block-major
// order, one per CTA.  Eight warps, one per group of 16 rows, take a tile together; a CTA has up to three such sets
// (gemv_sets), which take the tiles of the run in turn.  At the end of a row block the sets' sums meet in shared
// memory, and the CTA either writes y (its run holds the whole K range) or a partial sum into one of its two slots; the CTA
// that completes a row block adds the partials in K order (deterministic) and writes y.
//
// Streaming: each warp fills a ring of its own with cp.async (its slice of a tile: 16 rows x 128 k, contiguous), so nothing is
// shared between warps and no barrier stands in the main loop; the data are read back with 128-bit shared loads that land
// directly in the MMA A-fragment positions (cq_common.cuh).  The first slices are prefetched to L2 before the
// programmatic-dependency wait and copied after it: the kernel before may be the one that writes the weights.
//
// The activations of the whole run are staged once (a run that crosses into the next row block reads them again), as many
// tiles as fit shared memory; bf16 or fp16 go to fp16 with a power-of-two scale per token and 128 k, found by a shuffle among the
// sixteen lanes that hold them, so that nothing overflows or loses bits.
//
// Decode (model dtype): cq_gemv_tile.cuh.  Three to sixteen tokens use the m16n8k16 MMA (fp16 in, fp32 accumulate), the
// weights' loads landing directly in its A fragment; the group scale s_g multiplies the fp32 group sum, as in the paper's
// narrow path.  Dynamic A8 uses the INT8 m16n8k32 MMA on signed carriers (Eq. carrier); int32 group partials, fp32 rescale
// (Eq. a8-output).
#include "cq_common.cuh"
#include "cq_gemv_tile.cuh"
#include "cq_internal.h"
#include "cq_tc_ptx.cuh"

namespace cq {

namespace {

using namespace tc;

// MODE 0: model dtype.  MODE 1: Dynamic A8 (xq = INT8 carrier [M][x8_pitch], dxs = row scales).  NT: blocks of 8 tokens.
// Sets of eight warps in a CTA, and CTAs on an SM.  One large CTA reads the activations once per SM and hands over fewer
// partial sums; it has three sets where 80 registers a thread suffice and two otherwise (two token blocks; INT8 carriers
// evaluated code by code).  CTAs of one set serve the shortest calls, where most sets of a large CTA would have no tile.  Time of
// one set / of large CTAs over 784 products, by tiles an SM: model dtype 0.94 below one tile, 1.04 at one to three, 1.07 beyond;
// Dynamic A8 0.96 below one, 0.93 at one to two, 1.03 at two to three, 1.06 beyond.
__host__ __device__ constexpr int gemv_sets(int B, int NT, int MODE) { return NT == 2 || (MODE == 1 && B >= 6) ? 2 : 3; }
__host__ __device__ constexpr int gemv_occ(int B, int NT, int SETS) { return SETS > 1 ? 1 : NT == 2 || B >= 6 ? 2 : 3; }
constexpr int MODEL_LARGE_CTAS = 1, A8_LARGE_CTAS = 2;   // tiles an SM from which on CTAs are large
// Routed products: one set to a CTA and two CTAs to an SM, so that the CTAs of many small matrices fill the SMs evenly.
constexpr int GROUP_OCC = 2;
__host__ __device__ constexpr int gemv_unit_bytes(int B, int G) { return 256 * B + 128 * (TILE / G); }
__host__ __device__ constexpr int gemv_stages(int B, int G) { return gemv_unit_bytes(B, G) <= 1664 ? 4 : 3; }
__host__ __device__ constexpr int gemv_ring_bytes(int B, int G, int SETS) { return SETS * 8 * gemv_stages(B, G) * gemv_unit_bytes(B, G); }
// sums that the sets hand over at the end of a row block, twice (a set may be one row block ahead)
__host__ __device__ constexpr int gemv_comb_bytes(int NT, int SETS) { return 2 * (SETS - 1) * 8 * NT * 4 * 32 * 4; }
// level tables (model dtype, W4) or carrier tables (Dynamic A8) of a warp's 16 rows
__host__ __device__ constexpr int gemv_table_bytes(int B, int MODE) { return MODE == 1 ? (carrier_by_table(B) ? 16 * carrier_table_stride(B) : 0) : (B == 4 ? 256 : 0); }
__host__ __device__ constexpr int gemv_fixed_bytes(int B, int G, int NT, int MODE, int SETS) {
    return gemv_ring_bytes(B, G, SETS) + gemv_comb_bytes(NT, SETS) + SETS * 8 * gemv_table_bytes(B, MODE);
}
// dynamic shared memory of a CTA: its share of the SM's 228 KB less 1 KB for the system and 512 bytes that the kernel declares
__host__ __device__ constexpr int gemv_smem(int OCC) { return (228 / OCC) * 1024 - 1536; }
// padding of a staged activation row, in elements: rows 64 bytes apart in the banks where a lane reads 16 bytes (W3, W4),
// 32 where it reads 8
__host__ __device__ constexpr int gemv_x_pad(int B, int MODE) { return MODE == 1 ? 32 : (B == 3 || B == 4 ? 32 : 16); }
// bytes of a staged tile's activations of M rows, unit scales included
__host__ __device__ constexpr int gemv_x_tile_bytes(int M, int MODE) { return MODE == 1 ? M * TILE : M * (TILE * 2 + 4); }
__host__ __device__ constexpr int gemv_x_fixed_bytes(int M, int B, int MODE) { return M * gemv_x_pad(B, MODE) * (MODE == 1 ? 1 : 2) + 128; }
// K tiles whose activations fit at a time
__host__ __device__ constexpr int gemv_x_tiles(int B, int G, int NT, int MODE, int SETS, int OCC, int M) {
    return (gemv_smem(OCC) - gemv_fixed_bytes(B, G, NT, MODE, SETS) - gemv_x_fixed_bytes(M, B, MODE)) / gemv_x_tile_bytes(M, MODE);
}

__device__ __forceinline__ void bar_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }

// ------------------------------------------------------------------------------------------
// The inputs are not __restrict__ (the compiler could read them through the non-coherent path): the kernel may have started
// before the one that writes them had ended.
template <int B, int G, int NT, int MODE, int SETS>
__device__ __forceinline__ void
gemv_body(const uint8_t *layout, const Dims &d, const uint16_t *x, const int8_t *xq,
          int64_t x8_pitch, const float *dxs, uint16_t *__restrict__ y, int M, float *__restrict__ partial,
          int *__restrict__ counters, int x_tiles, bool xf16) {
    constexpr int GPT = TILE / G;
    constexpr int L = B == 1 ? 1 : (1 << (B - 1));
    constexpr bool F16 = MODE == 0;        // activations staged as fp16 (model dtype) or as the INT8 carrier
    constexpr int ES = F16 ? 2 : 1;        // bytes per staged activation element
    constexpr int CB = 2048 * B, TB = CB + 1024 * GPT;   // bytes of a tile's code part and of a whole tile
    constexpr int UB = gemv_unit_bytes(B, G), NS = gemv_stages(B, G);
    constexpr int THREADS = 256 * SETS;
    constexpr int XPAD = gemv_x_pad(B, MODE);
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ int s_last;
    __shared__ float s_dx[16];                                         // Dynamic A8: d_x / 127
    constexpr bool T_TABLE = MODE == 1 && (B == 3 || B == 5);          // W4 lanes keep their positions in registers
    __shared__ float s_t[T_TABLE ? 16 : 1];                            // Dynamic A8: t_i = i / M of the carrier tables
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int set = warp >> 3, rb = warp & 7;
    uint8_t *ring = smem + warp * NS * UB;
    float *comb = reinterpret_cast<float *>(smem + gemv_ring_bytes(B, G, SETS));
    int8_t *ctab = reinterpret_cast<int8_t *>(comb) + gemv_comb_bytes(NT, SETS) + warp * gemv_table_bytes(B, MODE);
    uint8_t *xs = smem + gemv_fixed_bytes(B, G, NT, MODE, SETS);

    // This CTA's run: tiles [first, first + n) of the layout, which starts at kb0 of its first row block.
    const int KT = d.KT;
    const int V = d.NB * KT, first = run_start(blockIdx.x, V, gridDim.x);
    const int n = run_start(blockIdx.x + 1, V, gridDim.x) - first;
    const int nb0 = first / KT, kb0 = first - nb0 * KT;

    // ---- this warp's slices of the tiles set, set + SETS, ... of the run, into its ring
    const uint8_t *wl = layout + (size_t)(first + set) * TB + rb * 256 * B + lane * 16;
    const uint8_t *pl = layout + (size_t)(first + set) * TB + CB + rb * 128 * GPT + lane * 16;
    int next = set;
    auto ring_load = [&](int st) {   // the next one, if there is one, into stage st; always a group of its own
        if (next < n) {
            constexpr int NFQ = (2 * B) / 4;
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(ring + st * UB);
#pragma unroll
            for (int q = 0; q < NFQ; ++q) cp_async16(dst + q * 512 + lane * 16, wl + q * 512);
            if constexpr ((2 * B) % 4 != 0) cp_async8(dst + NFQ * 512 + lane * 8, wl + NFQ * 512 - lane * 8);
            if (lane < 8 * GPT) cp_async16(dst + 256 * B + lane * 16, pl);
            wl += SETS * TB; pl += SETS * TB; next += SETS;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    DecodeRegs dr = {};
    if constexpr (F16 && B != 3 && B != 4) dr = load_decode_regs();
    W4Lane w4{};
    uint32_t x16 = 16u;
    if constexpr (B == 4) { w4 = w4_lane(lane); x16 = c_w4_x16; }
    if constexpr (T_TABLE) {
        if (threadIdx.x < L) s_t[threadIdx.x] = __fdiv_rn((float)threadIdx.x, (float)(L - 1));
    }
    // Until here the kernel before this one may still be running, and it may be the one that writes the weights: the first of
    // this warp's slices are brought to L2 and no further (L2 sees every write to them), and read after the wait.  It may
    // also produce or still use the activations, the workspace and y.
    if (lane < NS - 1 && set + lane * SETS < n) {
        const uint8_t *tile = layout + (size_t)(first + set + lane * SETS) * TB;
        prefetch_l2(tile + rb * 256 * B, 256 * B);
        prefetch_l2(tile + CB + rb * 128 * GPT, 128 * GPT);
    }
    wait_for_previous_kernel();
    if constexpr (MODE == 1) {
        if (threadIdx.x < 16) s_dx[threadIdx.x] = threadIdx.x < M ? dxs[threadIdx.x] * (1.0f / 127.0f) : 0.0f;
    }

    float total[NT][4];
#pragma unroll
    for (int tb = 0; tb < NT; ++tb)
#pragma unroll
        for (int i = 0; i < 4; ++i) total[tb][i] = 0.0f;
    int st = 0, fill = NS - 1, seg = 0, nb = nb0;   // nb: the row block at hand
    bool primed = false;
    // The first copies of weights go out behind the loads of the first activations: they fill the queue to L2, and the activations
    // are what the CTA waits for (copies ahead of the loads: 0.8 % longer over 120 products of three to sixteen rows).
    auto prime = [&]() {
#pragma unroll
        for (int i = 0; i < NS - 1; ++i) ring_load(i);
        primed = true;
    };
    for (int i0 = 0; i0 < n;) {
        // ---- activations of the tiles [i0, i1): k tile (kb0 + i) mod KT of the matrix sits at position (i - i0) mod KT
        const int n_st = min(min(n - i0, KT), x_tiles);              // k tiles staged
        const int i1 = n_st == KT ? n : i0 + n_st;                   // all of K: good for the rest of the run
        const int kbs = (kb0 + i0) % KT;
        const int XS = n_st * TILE + XPAD;
        float *inv = reinterpret_cast<float *>(xs + (size_t)M * XS * ES);      // F16: [position][M]
        if (i0 > 0) __syncthreads();   // the tiles before are done with
        if (F16 && SETS == 1 && !primed) prime();   // a short run: little enough to go first
        if constexpr (F16) {
            // sixteen lanes take a token's 128 k of a tile, eight values each; four loads in flight (eight, with the places
            // counted again for the stores: 4096 square, W4, M = 8 10.4 -> 11.6 us)
            constexpr int STEP = THREADS / 16, BATCH = 4;
            const int dm = STEP / n_st, dp = STEP - dm * n_st, c = threadIdx.x & 15;
            // (no loops that take n_st off one by one: with a tile or two staged, they run to a hundred steps)
            int m = ((int)threadIdx.x >> 4) / n_st, p = ((int)threadIdx.x >> 4) - m * n_st;
            while (m < M) {
                uint4 v[BATCH];
                int mm[BATCH], pp[BATCH];
#pragma unroll
                for (int u = 0; u < BATCH; ++u) {
                    mm[u] = m; pp[u] = p;
                    v[u] = make_uint4(0u, 0u, 0u, 0u);
                    int kb = kbs + p;
                    if (kb >= KT) kb -= KT;
                    const int64_t k = (int64_t)kb * TILE + c * 8;
                    if (m < M && k < d.K) v[u] = *reinterpret_cast<const uint4 *>(x + (int64_t)m * d.K + k);   // K % 8 == 0 always
                    m += dm; p += dp;
                    if (p >= n_st) { p -= n_st; ++m; }
                }
#pragma unroll
                for (int u = 0; u < BATCH; ++u) {
                    if (mm[u] >= M) break;
                    uint32_t ws[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
                    const float back = scale_to_half(ws, xf16, 14, lane);
                    if (c == 0) inv[pp[u] * M + mm[u]] = back;
                    store_half_chunk<B>(reinterpret_cast<__half *>(xs) + (size_t)mm[u] * XS + pp[u] * TILE, c, ws);
                }
            }
            if (!primed) prime();
        } else {
            // 16-byte chunks in the order the product reads (a8_row_regs; W4: natural); pitch a multiple of 128, zero beyond K
            const int cpr = n_st * (TILE / 16), dm = THREADS / cpr, dc = THREADS - dm * cpr;
            int m = (int)threadIdx.x / cpr, c = (int)threadIdx.x - m * cpr;
            while (m < M) {
                int kb = kbs + (c >> 3);
                if (kb >= KT) kb -= KT;
                cp_async16((uint32_t)__cvta_generic_to_shared(xs + (size_t)m * XS + c * 16), xq + (int64_t)m * x8_pitch + (int64_t)kb * TILE + (c & 7) * 16);
                m += dm; c += dc;
                if (c >= cpr) { c -= cpr; ++m; }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            if (!primed) {
                prime();
                asm volatile("cp.async.wait_group %0;" ::"n"(NS - 1) : "memory");   // the weights' groups are the younger ones
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
        }
        __syncthreads();
        // this lane's B-fragment base per token block: row g of the block (token columns beyond M read the last real
        // row; their results are never stored), k offset 4 t or 8 t, in elements
        int xo[NT];
#pragma unroll
        for (int tb = 0; tb < NT; ++tb) xo[tb] = min(tb * 8 + g, M - 1) * XS + ((F16 && B != 3 && B != 4) ? 4 : 8) * t;

        // ---- row block by row block
        for (int i = i0; i < i1;) {
            const int block_end = (nb + 1) * KT - first, e = min(i1, block_end);   // end of the tiles of row block nb
            int it = i + (set - i % SETS + SETS) % SETS;                              // this set's first tile
            int pos = (it - i0) % n_st;   // n_st < KT: it - i0 < n_st anyway
#pragma unroll 1
            for (; it < e; it += SETS) {
                asm volatile("cp.async.wait_group %0;" ::"n"(NS - 2) : "memory");
                __syncwarp();   // the other lanes' copies; and every lane is past its reads of the stage refilled now
                ring_load(fill);
                const uint8_t *stage = ring + st * UB;
                TileRegs<B, GPT> regs;
                load_tile<B, GPT>(regs, stage + lane * 16, stage + 256 * B + record_offset<B, GPT>(lane), lane);
                if (++st == NS) st = 0;
                if (++fill == NS) fill = 0;
                float acc[NT][4];
#pragma unroll
                for (int tb = 0; tb < NT; ++tb)
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[tb][q] = 0.0f;
                compute_tile<B, G, NT, MODE>(regs, dr, xs + (size_t)pos * TILE * ES, xo, ctab, s_t, w4, x16, g, t, acc);
#pragma unroll
                for (int tb = 0; tb < NT; ++tb) {   // in true units: lane (g, t) holds rows g, g + 8 x tokens 2 t, 2 t + 1
                    float s0 = 1.0f, s1 = 1.0f;
                    if constexpr (F16) { s0 = inv[pos * M + min(tb * 8 + 2 * t, M - 1)]; s1 = inv[pos * M + min(tb * 8 + 2 * t + 1, M - 1)]; }
                    total[tb][0] = F16 ? fmaf(acc[tb][0], s0, total[tb][0]) : total[tb][0] + acc[tb][0];
                    total[tb][1] = F16 ? fmaf(acc[tb][1], s1, total[tb][1]) : total[tb][1] + acc[tb][1];
                    total[tb][2] = F16 ? fmaf(acc[tb][2], s0, total[tb][2]) : total[tb][2] + acc[tb][2];
                    total[tb][3] = F16 ? fmaf(acc[tb][3], s1, total[tb][3]) : total[tb][3] + acc[tb][3];
                }
                pos += SETS;
                while (pos >= n_st) pos -= n_st;
            }
            i = e;
            if (i < n && i != block_end) continue;   // the row block goes on behind the next staging

            // ---- finish the row block (or this run's part of it)
            float *cb = comb + (seg & 1) * (SETS - 1) * 8 * NT * 4 * 32;
            if (set > 0) {
#pragma unroll
                for (int tb = 0; tb < NT; ++tb)
#pragma unroll
                    for (int q = 0; q < 4; ++q) cb[((((set - 1) * 8 + rb) * NT + tb) * 4 + q) * 32 + lane] = total[tb][q];
            }
            ++seg;
            if constexpr (SETS > 1) __syncthreads();
            if (set == 0) {
                const int kb_begin = nb == nb0 ? kb0 : 0, kb_end = first + i - nb * KT;
                const bool whole = kb_begin == 0 && kb_end == KT;
                // A run has at most two partial segments: one that starts inside a row block (its first) and one that
                // starts a row block without finishing it (its last); each CTA owns two partial slots.
                float *pslot = partial + ((size_t)blockIdx.x * 2 + (kb_begin > 0 ? 1 : 0)) * (size_t)(M * TILE);
#pragma unroll
                for (int tb = 0; tb < NT; ++tb)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float v = total[tb][q];
#pragma unroll
                        for (int s = 1; s < SETS; ++s) v += cb[((((s - 1) * 8 + rb) * NT + tb) * 4 + q) * 32 + lane];
                        const int tok = tb * 8 + 2 * t + (q & 1), r = rb * 16 + g + ((q >> 1) ? 8 : 0);
                        if constexpr (!F16) v *= s_dx[tok];
                        if (tok >= M) continue;
                        if (whole) {
                            const int64_t nn = (int64_t)nb * TILE + r;
                            if (nn < d.N) y[(int64_t)tok * d.N + nn] = float_to_act(v, xf16);
                        } else {
                            pslot[tok * TILE + r] = v;
                        }
                    }
                if (!whole) {
                    // The counter of a row block collects the tiles done; the CTA that completes it adds the partials in
                    // K order.  The first barrier orders the set's partial stores before thread 0's release; its acquire plus
                    // the second barrier make the other CTAs' partials visible to every thread of the set.
                    bar_sync(1, 256);
                    if (threadIdx.x == 0) {
                        int old;
                        asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;" : "=r"(old) : "l"(counters + nb), "r"(kb_end - kb_begin) : "memory");
                        s_last = (old + (kb_end - kb_begin) == KT);
                    }
                    bar_sync(1, 256);
                    if (s_last) {
                        const int c_first = run_of(nb * KT, V, gridDim.x);   // its segment starts the row block: slot 0
                        const int n_contrib = run_of((nb + 1) * KT - 1, V, gridDim.x) - c_first + 1;
                        const float *pb = partial + ((size_t)c_first * 2 + 1) * (size_t)(M * TILE);   // slot 1 of CTA c_first + q
                        // four consecutive channels of one token per thread and step (128-bit loads), up to eight
                        // slots in flight, added in K order
                        for (int idx = threadIdx.x; idx < M * (TILE / 4); idx += 256) {
                            const int m = idx / (TILE / 4), r = (idx % (TILE / 4)) * 4;
                            const int64_t nn = (int64_t)nb * TILE + r;
                            float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
                            for (int q0 = 0; q0 < n_contrib; q0 += 8) {
                                float4 vv[8];
#pragma unroll
                                for (int u = 0; u < 8; ++u) {
                                    const size_t off = (size_t)(q0 + u) * 2 * (M * TILE) - (q0 + u == 0 ? (size_t)(M * TILE) : 0);
                                    vv[u] = (q0 + u < n_contrib) ? __ldcg(reinterpret_cast<const float4 *>(pb + off + m * TILE + r))
                                                                 : make_float4(0.f, 0.f, 0.f, 0.f);
                                }
#pragma unroll
                                for (int u = 0; u < 8; ++u) { sum.x += vv[u].x; sum.y += vv[u].y; sum.z += vv[u].z; sum.w += vv[u].w; }
                            }
                            const float o[4] = {sum.x, sum.y, sum.z, sum.w};
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                if (nn + q < d.N) y[(int64_t)m * d.N + nn + q] = float_to_act(o[q], xf16);
                        }
                        if (threadIdx.x == 0) counters[nb] = 0;  // leave the workspace ready for the next call
                    }
                }
            }
#pragma unroll
            for (int tb = 0; tb < NT; ++tb)
#pragma unroll
                for (int q = 0; q < 4; ++q) total[tb][q] = 0.0f;
            ++nb;
        }
        i0 = i1;
    }
}

template <int B, int G, int NT, int MODE, int SETS>
__global__ void __launch_bounds__(256 * SETS, gemv_occ(B, NT, SETS))
gemv_kernel(const uint8_t *layout, Dims d, const uint16_t *x, const int8_t *xq,
            int64_t x8_pitch, const float *dxs, uint16_t *__restrict__ y, int M, float *__restrict__ partial,
            int *__restrict__ counters, int x_tiles, bool xf16) {
    gemv_body<B, G, NT, MODE, SETS>(layout, d, x, xq, x8_pitch, dxs, y, M, partial, counters, x_tiles, xf16);
}

// Routed products: blockIdx.y is a group, with its own matrix, rows and slice of the workspace.  (A kernel of its own:
// the table among the parameters of every small product cost the sweep over formats at M = 1 four per cent.)
template <int B, int G, int NT, int MODE>
__global__ void __launch_bounds__(256, GROUP_OCC)
gemv_groups_kernel(Dims d, const uint16_t *x, const int8_t *xq, int64_t x8_pitch, const float *dxs,
                   uint16_t *__restrict__ y, float *__restrict__ partial, int *__restrict__ counters, int x_tiles, bool xf16,
                   const __grid_constant__ GroupTable groups) {
    const Group &gr = groups.g[blockIdx.y];
    if constexpr (MODE == 1) { xq += (int64_t)gr.row0 * x8_pitch; dxs += gr.row0; } else x += (int64_t)gr.row0 * d.K;
    gemv_body<B, G, NT, MODE, 1>((const uint8_t *)gr.layout, d, x, xq, x8_pitch, dxs, y + (int64_t)gr.row0 * d.N, gr.rows,
                              partial + (size_t)blockIdx.y * gridDim.x * 2 * (8 * NT * TILE), counters + (int64_t)blockIdx.y * d.NB,
                              x_tiles, xf16);
}

template <int B, int G, int NT, int MODE, int SETS, bool GRP = false>
cudaError_t launch_one(const void *layout, const Dims &d, const uint16_t *x, const int8_t *xq, int64_t x8_pitch,
                       const float *dxs, uint16_t *y, int M, int P, float *partial, int *counters,
                       bool act_f16, cudaStream_t st, const GroupTable *groups = nullptr) {
    constexpr int OCC = GRP ? GROUP_OCC : gemv_occ(B, NT, SETS);
    static_assert(gemv_x_tiles(B, G, NT, MODE, SETS, OCC, 8 * NT) >= 2, "shared memory");
    const int64_t V = (int64_t)d.NB * d.KT;
    int64_t run = (V + P - 1) / P;   // the longest run, or all of K, bounds the activations a CTA stages
    if (run > d.KT) run = d.KT;
    const int fit = gemv_x_tiles(B, G, NT, MODE, SETS, OCC, M), x_tiles = (int)(run < fit ? run : fit);
    const size_t smem = (size_t)gemv_fixed_bytes(B, G, NT, MODE, SETS) + (size_t)gemv_x_fixed_bytes(M, B, MODE) + (size_t)x_tiles * gemv_x_tile_bytes(M, MODE);
    static std::atomic<uint64_t> attr_done{0};
    cudaError_t e;
    if constexpr (GRP) e = ensure_func_attr(gemv_groups_kernel<B, G, NT, MODE>, attr_done, cudaFuncAttributeMaxDynamicSharedMemorySize, gemv_smem(OCC));
    else e = ensure_func_attr(gemv_kernel<B, G, NT, MODE, SETS>, attr_done, cudaFuncAttributeMaxDynamicSharedMemorySize, gemv_smem(OCC));
    if (e != cudaSuccess) return e;
    // Programmatic overlap: this kernel may begin (and prefetch weights to L2) while the previous kernel of the stream drains; it
    // waits for that kernel before it reads or writes anything.
    const dim3 grid((unsigned)P, GRP ? (unsigned)groups->n : 1u);
    constexpr unsigned threads = 256 * SETS;
    if constexpr (GRP)
        return launch_overlapped(gemv_groups_kernel<B, G, NT, MODE>, grid, threads, smem, st, 1, true, d, x, xq, x8_pitch, dxs, y, partial, counters, x_tiles,
                                 act_f16, *groups);
    else
        return launch_overlapped(gemv_kernel<B, G, NT, MODE, SETS>, grid, threads, smem, st, 1, true, (const uint8_t *)layout, d, x, xq, x8_pitch, dxs, y, M,
                                 partial, counters, x_tiles, act_f16);
}

template <int B, int G>
cudaError_t dispatch_nt_mode(const void *layout, const Dims &d, const uint16_t *x, const int8_t *xq, int64_t x8_pitch,
                             const float *dxs, uint16_t *y, int M, int mode, GemvPlan plan, float *partial, int *counters, bool act_f16, cudaStream_t st) {
    auto launch = [&](auto nt, auto md, auto sets) {
        return launch_one<B, G, decltype(nt)::value, decltype(md)::value, decltype(sets)::value>(layout, d, x, xq, x8_pitch, dxs, y, M, plan.ctas, partial, counters, act_f16, st);
    };
    constexpr std::integral_constant<int, 0> zero{};
    constexpr std::integral_constant<int, 1> one{};
    constexpr std::integral_constant<int, 2> two{};
    if (plan.sets == 1) {
        if (mode == 0) return M <= 8 ? launch(one, zero, one) : launch(two, zero, one);
        return M <= 8 ? launch(one, one, one) : launch(two, one, one);
    }
    if (mode == 0) return M <= 8 ? launch(one, zero, std::integral_constant<int, gemv_sets(B, 1, 0)>{}) : launch(two, zero, std::integral_constant<int, gemv_sets(B, 2, 0)>{});
    return M <= 8 ? launch(one, one, std::integral_constant<int, gemv_sets(B, 1, 1)>{}) : launch(two, one, std::integral_constant<int, gemv_sets(B, 2, 1)>{});
}

template <int B>
cudaError_t dispatch_g(const void *layout, const Dims &d, const uint16_t *x, const int8_t *xq, int64_t x8_pitch,
                       const float *dxs, uint16_t *y, int M, int mode, GemvPlan plan, float *partial, int *counters, bool act_f16, cudaStream_t st) {
    switch (d.G) {
        case 32: return dispatch_nt_mode<B, 32>(layout, d, x, xq, x8_pitch, dxs, y, M, mode, plan, partial, counters, act_f16, st);
        case 64: return dispatch_nt_mode<B, 64>(layout, d, x, xq, x8_pitch, dxs, y, M, mode, plan, partial, counters, act_f16, st);
        default: return dispatch_nt_mode<B, 128>(layout, d, x, xq, x8_pitch, dxs, y, M, mode, plan, partial, counters, act_f16, st);
    }
}

// Routed products: sixteen-row variants, all groups in one launch.
template <int B, int G>
cudaError_t launch_groups_g(const GroupTable &t, const Dims &d, const uint16_t *x, const int8_t *xq, const float *dxs, uint16_t *y, int mode,
                            bool act_f16, int P, int max_rows, float *partial, int *counters, cudaStream_t st) {
    const int64_t pitch = (int64_t)d.KT * TILE;
    if (mode == 0) return launch_one<B, G, 2, 0, 1, true>(nullptr, d, x, nullptr, pitch, nullptr, y, max_rows, P, partial, counters, act_f16, st, &t);
    return launch_one<B, G, 2, 1, 1, true>(nullptr, d, nullptr, xq, pitch, dxs, y, max_rows, P, partial, counters, act_f16, st, &t);
}
template <int B>
cudaError_t launch_groups_b(const GroupTable &t, const Dims &d, const uint16_t *x, const int8_t *xq, const float *dxs, uint16_t *y, int mode,
                            bool act_f16, int P, int max_rows, float *partial, int *counters, cudaStream_t st) {
    switch (d.G) {
        case 32: return launch_groups_g<B, 32>(t, d, x, xq, dxs, y, mode, act_f16, P, max_rows, partial, counters, st);
        case 64: return launch_groups_g<B, 64>(t, d, x, xq, dxs, y, mode, act_f16, P, max_rows, partial, counters, st);
        default: return launch_groups_g<B, 128>(t, d, x, xq, dxs, y, mode, act_f16, P, max_rows, partial, counters, st);
    }
}

}  // namespace

cudaError_t launch_gemv_groups(const GroupTable &t, const Dims &d, const uint16_t *x, const int8_t *xq, const float *dxs, uint16_t *y,
                               int mode, bool act_f16, int P, float *partial, int *counters, cudaStream_t st) {
    int max_rows = 1;
    for (int i = 0; i < t.n; ++i) if (t.g[i].rows > max_rows) max_rows = t.g[i].rows;
    switch (d.B) {
        case 1: return launch_groups_b<1>(t, d, x, xq, dxs, y, mode, act_f16, P, max_rows, partial, counters, st);
        case 2: return launch_groups_b<2>(t, d, x, xq, dxs, y, mode, act_f16, P, max_rows, partial, counters, st);
        case 3: return launch_groups_b<3>(t, d, x, xq, dxs, y, mode, act_f16, P, max_rows, partial, counters, st);
        case 4: return launch_groups_b<4>(t, d, x, xq, dxs, y, mode, act_f16, P, max_rows, partial, counters, st);
        case 5: return launch_groups_b<5>(t, d, x, xq, dxs, y, mode, act_f16, P, max_rows, partial, counters, st);
        case 6: return launch_groups_b<6>(t, d, x, xq, dxs, y, mode, act_f16, P, max_rows, partial, counters, st);
        case 7: return launch_groups_b<7>(t, d, x, xq, dxs, y, mode, act_f16, P, max_rows, partial, counters, st);
        default: return launch_groups_b<8>(t, d, x, xq, dxs, y, mode, act_f16, P, max_rows, partial, counters, st);
    }
}

// Streaming multiprocessors of the current device (148 on a B200; that figure also stands in when no
// device can be asked, so that size queries work on a machine without a GPU).
int sm_count() {
    static std::atomic<int> cached[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { (void)cudaGetLastError(); return 148; }
    int n = cached[dev].load(std::memory_order_relaxed);
    if (n > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) { (void)cudaGetLastError(); return 148; }
    cached[dev].store(n, std::memory_order_relaxed);
    return n;
}

// CTAs of the small-M path: one run of tiles each, as many as are resident at once.
GemvPlan gemv_plan(const Dims &d, int64_t M, int mode) {
    const int64_t T = (int64_t)d.NB * d.KT, sms = sm_count();
    const int NT = M <= 8 ? 1 : 2;
    GemvPlan p;
    p.sets = T < (mode == 1 ? A8_LARGE_CTAS : MODEL_LARGE_CTAS) * sms ? 1 : gemv_sets(d.B, NT, mode);
    const int64_t places = sms * gemv_occ(d.B, NT, p.sets);
    p.ctas = (int)(T < places ? T : places);
    return p;
}

cudaError_t launch_gemv(const void *layout, const Dims &d, const uint16_t *x, uint16_t *y, int64_t M, int mode,
                        bool act_f16, uint8_t *ws, const Workspace &plan, cudaStream_t st, bool prequantized) {
    float *partial = reinterpret_cast<float *>(ws + plan.partial_off);
    int *counters = reinterpret_cast<int *>(ws + plan.counters_off);
    if (mode == 0 && gemv_strip_ok(d, M, plan)) return launch_gemv_strip(layout, d, x, y, M, act_f16, partial, counters, st);
    int8_t *xq = reinterpret_cast<int8_t *>(ws + plan.x8_off);
    float *dxs = reinterpret_cast<float *>(ws + plan.dx_off);
    const int64_t pitch = (int64_t)d.KT * TILE;
    if (mode == 1 && !prequantized) {
        cudaError_t e = launch_quantize_a8(x, M, d.K, xq, pitch, dxs, d.B != 4, act_f16, st);
        if (e != cudaSuccess) return e;
    }
    const int Mi = (int)M;
    const GemvPlan gp = gemv_plan(d, M, mode);
    switch (d.B) {
        case 1: return dispatch_g<1>(layout, d, x, xq, pitch, dxs, y, Mi, mode, gp, partial, counters, act_f16, st);
        case 2: return dispatch_g<2>(layout, d, x, xq, pitch, dxs, y, Mi, mode, gp, partial, counters, act_f16, st);
        case 3: return dispatch_g<3>(layout, d, x, xq, pitch, dxs, y, Mi, mode, gp, partial, counters, act_f16, st);
        case 4: return dispatch_g<4>(layout, d, x, xq, pitch, dxs, y, Mi, mode, gp, partial, counters, act_f16, st);
        case 5: return dispatch_g<5>(layout, d, x, xq, pitch, dxs, y, Mi, mode, gp, partial, counters, act_f16, st);
        case 6: return dispatch_g<6>(layout, d, x, xq, pitch, dxs, y, Mi, mode, gp, partial, counters, act_f16, st);
        case 7: return dispatch_g<7>(layout, d, x, xq, pitch, dxs, y, Mi, mode, gp, partial, counters, act_f16, st);
        default: return dispatch_g<8>(layout, d, x, xq, pitch, dxs, y, Mi, mode, gp, partial, counters, act_f16, st);
    }
}

}  // namespace cq
