// One and two tokens in the model dtype (Section 5.3 narrow-row path): packed-half products without the tensor core, one
// CTA per SM, the work cut into strips of sixteen output channels.
//
// A unit is what a warp decodes at a time: the sixteen rows of a strip x 128 k, a contiguous piece of a layout tile.  Units
// are counted strip by strip along K and dealt out evenly, first to the CTAs, then to the 24 warps of a CTA, so a warp
// streams one contiguous run and a strip's partial sums meet in shared memory.  With strips of a whole tile row (128
// channels, cq_gemv.cu) nearly every CTA began and ended inside a row block, and each of those ends cost a barrier, a
// release, an acquire and a round trip through L2, plus the staging of another activation slice: 3 of 14 us at 8192^2.
// Where a few units more per SM allow it, the CTAs take whole strips and exchange nothing at all (strip_plan).
//
// The activations are staged once per CTA for the whole of K, with a power-of-two scale per 128 k (a shuffle among the
// sixteen lanes that hold them, no barrier), which the fp32 sum of each unit takes back.  Weights reach the registers
// through a ring in shared memory that each warp fills for itself (cp.async: no barriers, nothing shared between warps),
// or straight from global memory into a three-deep prefetch (strip_uses_ring).
#include "cq_common.cuh"
#include "cq_gemv_tile.cuh"
#include "cq_internal.h"
#include "cq_tc_ptx.cuh"

namespace cq {

namespace {

using namespace tc;

constexpr int STRIP = 16;             // output channels of a strip
constexpr int SW = 24;                // warps of a CTA: three to a scheduler and half the register file each
constexpr int STRIP_THREADS = 32 * SW;
constexpr int STRIP_SMEM = 227 * 1024 - 1024;

__host__ __device__ constexpr int unit_bytes(int B, int G) { return 256 * B + 128 * (TILE / G); }
// The ring, but for the narrow codes of one token: their records and codes fit three deep into the registers, and their
// arithmetic is too short to pay for the way through shared memory (8192 square, G = 128: W1 9.2 us against 9.8, W3 13.5 against 14.0;
// but W8 20.1 against 18.5, W4 15.4 against 14.4).
__host__ __device__ constexpr bool strip_uses_ring(int B, int G, int NT) { return !(B <= 3 && G == 128 && NT == 1); }
__host__ __device__ constexpr int strip_stages(int B, int G) { return unit_bytes(B, G) <= 1664 ? 4 : 3; }
// shared memory behind the staged activations: unit scales, partial sums, W4 level tables, ring
__host__ __device__ constexpr int strip_x_bytes(int KT, int NT) { return KT * TILE * NT * 2; }
__host__ __device__ constexpr int strip_inv_bytes(int KT, int NT) { return (KT * NT * 4 + 15) / 16 * 16; }
__host__ __device__ constexpr int strip_slot_bytes(int NT) { return SW * 2 * STRIP * NT * 4; }
__host__ __device__ constexpr int strip_table_bytes(int B) { return B == 4 ? SW * 256 : 0; }
__host__ __device__ constexpr int strip_ring_bytes(int B, int G, int NT) { return strip_uses_ring(B, G, NT) ? SW * strip_stages(B, G) * unit_bytes(B, G) : 0; }
__host__ __device__ constexpr int64_t strip_smem_bytes(int B, int G, int NT, int64_t KT) {
    return KT * TILE * NT * 2 + (KT * NT * 4 + 15) / 16 * 16 + strip_slot_bytes(NT) + strip_table_bytes(B) + strip_ring_bytes(B, G, NT);
}

struct StripParams {
    const uint8_t *layout;
    const uint16_t *x;
    uint16_t *y;
    float *partial;    // strips shared between CTAs: [CTA][2][16 NT] sums
    int *counters;     // and, one byte per CTA, how many CTAs have delivered theirs of the strip that begins in it
    int64_t N, K;
    int KT, S;         // k tiles; strips (16 rows each) that hold a row of the matrix
    int whole;         // CTAs take whole strips
    bool xf16;
};

template <int B, int G, int NT>
__global__ void __launch_bounds__(STRIP_THREADS, 1)
gemv_strip_kernel(const __grid_constant__ StripParams p) {
    constexpr int GPT = TILE / G;
    constexpr int CB = 2048 * B, TB = CB + 1024 * GPT;      // bytes of a tile's codes, of a tile
    constexpr int UB = unit_bytes(B, G);
    constexpr bool RING = strip_uses_ring(B, G, NT);
    constexpr int NS = strip_stages(B, G);
    constexpr int NBUF = RING ? 1 : 3;
    constexpr int PREFETCH = RING ? NS - 1 : NBUF;          // units on their way to L2 before the wait
    extern __shared__ __align__(128) uint8_t smem[];
    const int KT = p.KT;
    float *s_inv = reinterpret_cast<float *>(smem + strip_x_bytes(KT, NT));                                      // [KT][NT]
    float *s_slot = reinterpret_cast<float *>(reinterpret_cast<uint8_t *>(s_inv) + strip_inv_bytes(KT, NT));     // [SW][2][NT][16]
    uint8_t *s_tab = reinterpret_cast<uint8_t *>(s_slot) + strip_slot_bytes(NT);
    uint8_t *s_ring = s_tab + strip_table_bytes(B);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;

    // This CTA's units [u0, u0 + U), and this warp's [v, v_end) of them, counted from u0.
    const int total_units = p.S * KT;
    int u0, U;
    if (p.whole) {
        const int s0 = run_start(blockIdx.x, p.S, gridDim.x), s1 = run_start(blockIdx.x + 1, p.S, gridDim.x);
        u0 = s0 * KT;
        U = (s1 - s0) * KT;
    } else {
        u0 = run_start(blockIdx.x, total_units, gridDim.x);
        U = run_start(blockIdx.x + 1, total_units, gridDim.x) - u0;
    }
    const int strip0 = u0 / KT, kb0 = u0 - strip0 * KT;   // the CTA's first unit
    const int NW = min(SW, U);                                                    // warps with work
    const int v_begin = warp < NW ? (int)((uint32_t)U * (uint32_t)warp / (uint32_t)NW) : 0;
    const int v_end = warp < NW ? (int)((uint32_t)U * (uint32_t)(warp + 1) / (uint32_t)NW) : 0;
    int strip = strip0 + (kb0 + v_begin) / KT, kb = (kb0 + v_begin) % KT;         // the unit at hand
    int left = v_end - v_begin;

    // ---- the load cursor: where the next unit's codes (of this lane) and records lie
    const uint8_t *tile0 = p.layout + ((size_t)(strip >> 3) * KT + kb) * (size_t)TB;
    const uint8_t *wl = tile0 + (strip & 7) * 256 * B + lane * 16;
    const uint8_t *pl = tile0 + CB + (strip & 7) * 128 * GPT + (RING ? lane * 16 : record_offset<B, GPT>(lane));
    int l_strip = strip, l_kb = kb, to_load = left;
    auto advance = [&]() {
        wl += TB; pl += TB; --to_load;
        if (++l_kb == KT) {   // on to the next strip: the row block below, or the first one of the next tile row
            l_kb = 0;
            if ((++l_strip & 7) != 0) { wl += 256 * B - (int64_t)KT * TB; pl += 128 * GPT - (int64_t)KT * TB; }
            else { wl -= 7 * 256 * B; pl -= 7 * 128 * GPT; }
        }
    };
    TileRegs<B, GPT> buf0, buf1, buf2;   // separate objects (an array of them ends up in local memory)
    auto buf_at = [&](auto ic) -> TileRegs<B, GPT> & {
        constexpr int i = decltype(ic)::value;
        if constexpr (i == 0) return buf0;
        else if constexpr (i == 1) return buf1;
        else return buf2;
    };
    uint8_t *ring = s_ring + warp * NS * UB;
    auto ring_load = [&](int st) {   // the unit under the cursor, if there is one, into stage st; always a group of its own
        if (to_load > 0) {
            constexpr int NFQ = (2 * B) / 4;
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(ring + st * UB);
#pragma unroll
            for (int q = 0; q < NFQ; ++q) cp_async16(dst + q * 512 + lane * 16, wl + q * 512);
            if constexpr ((2 * B) % 4 != 0) cp_async8(dst + NFQ * 512 + lane * 8, wl + NFQ * 512 - lane * 8);
            if (lane < 8 * GPT) cp_async16(dst + 256 * B + lane * 16, pl);
            advance();
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    DecodeRegs dr = {};
    if constexpr (B != 3 && B != 4) dr = load_decode_regs();
    int8_t *ctab = nullptr;
    W4Lane w4{};
    uint32_t x16 = 16u;
    if constexpr (B == 4) {
        ctab = reinterpret_cast<int8_t *>(s_tab) + warp * 256;
        w4 = w4_lane(lane); x16 = c_w4_x16;
    }
    // Until here the kernel before this one may still be running, and it may be the one that writes the weights: their first
    // units are brought to L2 and no further (L2 sees every write to them), and read after the wait.  It may also produce
    // or still use the activations, the workspace and y.
    if (lane < min(left, PREFETCH)) {
        const int v = kb0 + v_begin + lane, s = strip0 + v / KT;
        const uint8_t *tile = p.layout + ((size_t)(s >> 3) * KT + v % KT) * (size_t)TB;
        prefetch_l2(tile + (s & 7) * 256 * B, 256 * B);
        prefetch_l2(tile + CB + (s & 7) * 128 * GPT, 128 * GPT);
    }
    wait_for_previous_kernel();

    // ---- activations: eight values per thread and step, sixteen lanes hold the 128 k of a tile.  The first step's loads go out
    // ahead of the weights', which fill the queue to L2.
    __half *xs = reinterpret_cast<__half *>(smem);
    const int chunks = KT * (TILE / 8);
    auto x_chunk = [&](int m, int c) {   // K % 8 == 0 always
        return (int64_t)c * 8 < p.K ? *reinterpret_cast<const uint4 *>(p.x + m * p.K + (int64_t)c * 8) : make_uint4(0u, 0u, 0u, 0u);
    };
    uint4 first[NT];
#pragma unroll
    for (int m = 0; m < NT; ++m) first[m] = x_chunk(m, threadIdx.x);
    if constexpr (RING) {
#pragma unroll
        for (int i = 0; i < NS - 1; ++i) ring_load(i);
    } else {
        static_for<NBUF>([&](auto ic) {
            if (to_load > 0) { load_tile_g<B, GPT>(buf_at(ic), wl, pl, lane); advance(); }
        });
    }
#pragma unroll
    for (int m = 0; m < NT; ++m) {
        uint4 v4 = first[m];
        for (int c = threadIdx.x; c < chunks; c += STRIP_THREADS) {
            if (c >= STRIP_THREADS) v4 = x_chunk(m, c);
            uint32_t ws[4] = {v4.x, v4.y, v4.z, v4.w};
            // the largest in [2^10, 2^11): sixteen products of a normalised level stay in fp16
            const float back = scale_to_half(ws, p.xf16, 10, lane);   // chunks and threads are multiples of sixteen
            if ((lane & 15) == 0) s_inv[(c >> 4) * NT + m] = back;
            store_half_chunk<B>(xs + (size_t)m * KT * TILE + (c & ~15) * 8, c & 15, ws);
        }
    }
    __syncthreads();

    // ---- the warp's run
    float total[NT][2];
#pragma unroll
    for (int m = 0; m < NT; ++m) total[m][0] = total[m][1] = 0.0f;
    bool from_start = kb == 0;            // the segment of the strip at hand begins at k = 0
    int xo[NT];                           // element offset of the unit's activations for this lane
#pragma unroll
    for (int m = 0; m < NT; ++m) xo[m] = m * KT * TILE + ((B == 3 || B == 4) ? 8 : 4) * t;
    auto consume = [&](const TileRegs<B, GPT> &r) {
        float acc[NT][4];
#pragma unroll
        for (int m = 0; m < NT; ++m)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[m][i] = 0.0f;
        compute_tile<B, G, NT, 2>(r, dr, reinterpret_cast<const uint8_t *>(xs + kb * TILE), xo, ctab, nullptr, w4, x16, g, t, acc);
#pragma unroll
        for (int m = 0; m < NT; ++m) {
            const float inv = s_inv[kb * NT + m];
            total[m][0] = fmaf(acc[m][0], inv, total[m][0]);
            total[m][1] = fmaf(acc[m][2], inv, total[m][1]);
        }
        --left;
        if (++kb == KT || left == 0) {   // end of this warp's segment of the strip
#pragma unroll
            for (int m = 0; m < NT; ++m)
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    total[m][i] += __shfl_xor_sync(0xffffffffu, total[m][i], 1);
                    total[m][i] += __shfl_xor_sync(0xffffffffu, total[m][i], 2);
                }
            if (t == 0) {
#pragma unroll
                for (int m = 0; m < NT; ++m)
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        if (from_start && kb == KT) {
                            const int64_t n = (int64_t)strip * STRIP + g + 8 * i;
                            if (n < p.N) p.y[m * p.N + n] = float_to_act(total[m][i], p.xf16);
                        } else {   // slot 0: begins inside the strip; slot 1: begins it without finishing it
                            s_slot[((warp * 2 + (from_start ? 1 : 0)) * NT + m) * STRIP + g + 8 * i] = total[m][i];
                        }
                    }
            }
            if (kb == KT) { kb = 0; ++strip; from_start = true; }
#pragma unroll
            for (int m = 0; m < NT; ++m) total[m][0] = total[m][1] = 0.0f;
        }
    };
    if constexpr (!RING) {
        while (left > 0) {
            static_for<NBUF>([&](auto ic) {
                if (left > 0) {
                    consume(buf_at(ic));
                    if (to_load > 0) { load_tile_g<B, GPT>(buf_at(ic), wl, pl, lane); advance(); }
                }
            });
        }
    } else {
        int st = 0, fill = NS - 1;
#pragma unroll 1
        while (left > 0) {
            asm volatile("cp.async.wait_group %0;" ::"n"(NS - 2) : "memory");
            __syncwarp();   // the other lanes' copies; and every lane is past its reads of the stage refilled now
            ring_load(fill);
            const uint8_t *stage = ring + st * UB;
            TileRegs<B, GPT> regs;
            load_tile<B, GPT>(regs, stage + lane * 16, stage + 256 * B + record_offset<B, GPT>(lane), lane);
            if (++st == NS) st = 0;
            if (++fill == NS) fill = 0;
            consume(regs);
        }
    }
    __syncthreads();

    // ---- strips that several warps (or CTAs) share: a warp per strip adds the sums in K order, a lane per row and token
    const int last_strip = (u0 + U - 1) / KT;
    const int row = lane & 15, tok = lane >> 4;
    for (int s = strip0 + warp; s <= last_strip; s += SW) {
        const int a = max(0, (s - strip0) * KT - kb0), b = min(U, (s + 1 - strip0) * KT - kb0);   // this CTA's units of the strip
        const bool begins = s > strip0 || kb0 == 0, ends = (s + 1 - strip0) * KT - kb0 <= U;
        const int wf = run_of(a, U, NW), wl_ = run_of(b - 1, U, NW);
        if (begins && ends && wf == wl_) continue;   // one warp had all of it and wrote y
        const bool mine = tok < NT;
        float sum = 0.0f;
        if (mine) {
            sum = s_slot[((wf * 2 + (begins ? 1 : 0)) * NT + tok) * STRIP + row];
            for (int w = wf + 1; w <= wl_; ++w) sum += s_slot[(w * 2 * NT + tok) * STRIP + row];
        }
        bool write = begins && ends;
        if (!write) {
            // The CTA that delivers the last of the strip's partial sums adds them in K order.  The lanes' stores are
            // ordered before lane 0's release by the warp barrier; its acquire and the second one make the others' visible.
            if (mine) __stcg(p.partial + (((size_t)blockIdx.x * 2 + (begins ? 1 : 0)) * NT + tok) * STRIP + row, sum);
            const int c_first = run_of(s * KT, total_units, gridDim.x);
            const int n = run_of((s + 1) * KT - 1, total_units, gridDim.x) - c_first + 1;
            const int sh = 8 * (c_first & 3);
            __syncwarp();
            int last = 0;
            if (lane == 0) {
                unsigned old;
                asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p.counters + (c_first >> 2)), "r"(1u << sh) : "memory");
                last = (int)((old >> sh) & 0xFFu) == n - 1;
                if (last) atomicSub(reinterpret_cast<unsigned *>(p.counters) + (c_first >> 2), (unsigned)n << sh);   // zero for the next call
            }
            write = __shfl_sync(0xffffffffu, last, 0) != 0;
            __syncwarp();
            if (write && mine) {
                const float *pb = p.partial + (size_t)c_first * 2 * NT * STRIP + tok * STRIP + row;
                sum = __ldcg(pb + NT * STRIP);
                for (int q0 = 1; q0 < n; q0 += 4) {   // four independent loads in flight
                    float v[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[i] = q0 + i < n ? __ldcg(pb + (size_t)(q0 + i) * 2 * NT * STRIP) : 0.0f;
#pragma unroll
                    for (int i = 0; i < 4; ++i) sum += v[i];
                }
            }
        }
        const int64_t nn = (int64_t)s * STRIP + row;
        if (write && mine && nn < p.N) p.y[tok * p.N + nn] = float_to_act(sum, p.xf16);
    }
}

// How many CTAs, and whether they take whole strips.  Whole strips leave some SMs up to a strip more than others; shared ones
// cost the exchange at the end of the kernel, some 1.5 us.  Whole strips win up to a surplus of some 55 units (16 x 128 weights) on the
// fullest SM with three bits and fewer, 45 with four and five, 28 with more; at two tokens 45, 32 and 22: 50 kB of
// weights, less a fifth at two tokens, and at most 60 units, where the narrow codes take as long as their bytes do not.  Over 219
// products of one and two tokens this is 0.2 % off the better of the two each time; the same 50 units for all formats 0.7 %, and
// 5504 x 6656, W7 G32, two tokens 19.5 us shared, 22.7 whole.
struct StripPlan { int ctas, whole; };
StripPlan strip_plan(const Dims &d, int64_t M) {
    const int64_t S = (d.N + STRIP - 1) / STRIP, KT = d.KT, P = sm_count(), T = S * KT;
    const int64_t whole_units = (S + P - 1) / P * KT;
    int64_t surplus = 50000 / unit_bytes(d.B, d.G > TILE ? TILE : d.G);
    if (surplus > 60) surplus = 60;
    if (M == 2) surplus = surplus * 4 / 5;
    StripPlan r;
    r.whole = whole_units - T / P <= surplus;
    const int64_t rounds = (S + P - 1) / P;
    r.ctas = (int)(r.whole ? (S + rounds - 1) / rounds : (T < P ? T : P));
    return r;
}

template <int B, int G, int NT>
cudaError_t launch_strip_nt(const StripParams &p, int ctas, cudaStream_t st) {
    const size_t smem = (size_t)strip_smem_bytes(B, G, NT, p.KT);
    static std::atomic<uint64_t> attr_done{0};
    cudaError_t e = ensure_func_attr(gemv_strip_kernel<B, G, NT>, attr_done, cudaFuncAttributeMaxDynamicSharedMemorySize, STRIP_SMEM);
    if (e != cudaSuccess) return e;
    return launch_overlapped(gemv_strip_kernel<B, G, NT>, dim3((unsigned)ctas), STRIP_THREADS, smem, st, 1, true, p);
}
template <int B>
cudaError_t launch_strip_b(const StripParams &p, int G, int M, int ctas, cudaStream_t st) {
    switch (G) {
        case 32: return M == 1 ? launch_strip_nt<B, 32, 1>(p, ctas, st) : launch_strip_nt<B, 32, 2>(p, ctas, st);
        case 64: return M == 1 ? launch_strip_nt<B, 64, 1>(p, ctas, st) : launch_strip_nt<B, 64, 2>(p, ctas, st);
        default: return M == 1 ? launch_strip_nt<B, 128, 1>(p, ctas, st) : launch_strip_nt<B, 128, 2>(p, ctas, st);
    }
}

}  // namespace

// The staged activations bound K beside a ring of full depth; beyond, cq_gemv.cu serves, which is faster there than a ring of two
// stages: 8192 x 28672, two tokens, W4 G128 45.1 us against 46.3, W8 G128 56.7 against 61.6 (with the kernel that cut runs of
// tiles for three CTAs an SM 50.3 and 67.4); only W8 G32 at one token 65.4 against 61.5.  The counters, a byte per CTA, have to fit the workspace's (256 bytes at least), and the
// partial sums its slots (two of 128 sums a token for each CTA of cq_gemv.cu, of which there are at least as many).
bool gemv_strip_ok(const Dims &d, int64_t M, const Workspace &plan) {
    if (M < 1 || M > 2) return false;
    const int G = d.G > TILE ? TILE : d.G;   // wide groups run the G = 128 code
    if (strip_smem_bytes(d.B, G, (int)M, d.KT) > STRIP_SMEM) return false;
    const StripPlan sp = strip_plan(d, M);
    return sp.whole || (sp.ctas <= 255 && (size_t)sp.ctas <= plan.counters_bytes && (size_t)sp.ctas * 2 * STRIP * (size_t)M * 4 <= plan.partial_bytes);
}

cudaError_t launch_gemv_strip(const void *layout, const Dims &d, const uint16_t *x, uint16_t *y, int64_t M, bool act_f16,
                              float *partial, int *counters, cudaStream_t st) {
    StripParams p;
    p.layout = (const uint8_t *)layout; p.x = x; p.y = y; p.partial = partial; p.counters = counters;
    p.N = d.N; p.K = d.K; p.KT = d.KT; p.S = (int)((d.N + STRIP - 1) / STRIP); p.xf16 = act_f16;
    const StripPlan sp = strip_plan(d, M);
    p.whole = sp.whole;
    switch (d.B) {
        case 1: return launch_strip_b<1>(p, d.G, (int)M, sp.ctas, st);
        case 2: return launch_strip_b<2>(p, d.G, (int)M, sp.ctas, st);
        case 3: return launch_strip_b<3>(p, d.G, (int)M, sp.ctas, st);
        case 4: return launch_strip_b<4>(p, d.G, (int)M, sp.ctas, st);
        case 5: return launch_strip_b<5>(p, d.G, (int)M, sp.ctas, st);
        case 6: return launch_strip_b<6>(p, d.G, (int)M, sp.ctas, st);
        case 7: return launch_strip_b<7>(p, d.G, (int)M, sp.ctas, st);
        default: return launch_strip_b<8>(p, d.G, (int)M, sp.ctas, st);
    }
}

}  // namespace cq
