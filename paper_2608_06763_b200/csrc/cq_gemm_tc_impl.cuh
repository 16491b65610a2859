// The model-dtype GEMM kernel and its launchers, as templates on SK: SK = false computes one whole output tile
// per CTA; SK = true adds the stream-K runs (tiles shared by several CTAs, partial tiles, the addition by the
// last CTA to arrive).  Each of the two is instantiated in a translation unit of its own, which keeps the code
// of the common case free of the other's registers and lets the two compile side by side.
#pragma once
#include "cq_common.cuh"
#include "cq_decode.cuh"
#include "cq_internal.h"
#include "cq_tc_ptx.cuh"

namespace cq {
namespace {


using namespace tc;

constexpr int DEC_WARPS = 16;                 // decoder / epilogue warps: two sets, which take the layout tiles in turn
constexpr int SET_WARPS = DEC_WARPS / 2;      // one warp of a set per 16 rows of a tile
constexpr int W4_TABLE_BYTES = 16 * 2 * 16;   // a decoder warp's level tables: 16 rows x the two groups of a 64-wide block at most
constexpr int TC_THREADS = 64 + 32 * DEC_WARPS + 32;   // producer of activations, MMA issuer, decoders, producer of raw tiles
constexpr int A_STAGE_BYTES = 128 * 128;  // 128 rows x 64 bf16

// ---------------------------------------------------------------- decode helpers
// Two reconstructed weights s * sign(k) * q(|k| / M) of one pair, rounded to bf16 (the dense path
// of Section 5.3 rounds the temporary operand to the activation dtype).  q is evaluated in half2
// (11-bit significand, finer than the bf16 it is rounded to), the scale is applied in fp32.
template <int B, int P, bool FIX, bool F16>
__device__ __forceinline__ uint32_t weight_pair_bf16(const uint32_t (&w)[2 * B], const RowCoef &c) {
    const __half2 T = pair_T<B, P>(w);
    const uint32_t q = level_pair<B, FIX>(T, c);
    const float2 f = __half22float2(as_h2(q));
    if constexpr (F16) {   // binary16 activations: the temporary operand is rounded to binary16
        return as_u32(__floats2half2_rn(f.x * c.s, f.y * c.s));
    } else {
        const __nv_bfloat162 v = __floats2bfloat162_rn(f.x * c.s, f.y * c.s);
        return *reinterpret_cast<const uint32_t *>(&v);
    }
}

// W3: the eight stored codes of a (row, group) index a signed bf16 table of s * sign(k) * q(|k| / 3)
// (u = 0, the reserved pattern, and k = 0 read zero), kept as a low-byte and a high-byte register pair
// and read four codes at a time with byte permutes; q(1/3) and q(2/3) by the fp32 Horner form.
struct W3Table { uint32_t lo[2], hi[2]; };
__device__ __forceinline__ uint32_t pack_act2(float lo, float hi, bool f16) {   // two values in the activation dtype
    if (f16) return as_u32(__floats2half2_rn(lo, hi));
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}
__device__ __forceinline__ W3Table w3_table(uint2 p, bool f16) {
    const float s = __uint_as_float(p.x & 0x7FFFFFFFu);
    const __half2 ab = as_h2(p.y);
    const float a = __low2float(ab), b = __high2float(ab), c = (1.0f - a) - b;
    constexpr float t1 = 1.0f / 3.0f, t2 = 2.0f / 3.0f;
    const float q1 = t1 * fmaf(t1, fmaf(t1, c, b), a), q2 = t2 * fmaf(t2, fmaf(t2, c, b), a);
    const uint32_t q12 = pack_act2(s * q1, s * q2, f16), ss = pack_act2(s, 0.0f, f16);
    const uint32_t nq = q12 | 0x80008000u, ns = ss | 0x00008000u;
    W3Table t;                                  // entries u = 0 .. 7:  0, -s, -s q2, -s q1 | 0, s q1, s q2, s
    t.lo[0] = prmt(nq, ns, 0x0247u) & 0xFFFFFF00u;   // low bytes:  0, (-s).lo, (-s q2).lo, (-s q1).lo
    t.lo[1] = prmt(q12, ss, 0x4207u) & 0xFFFFFF00u;  //             0, (s q1).lo, (s q2).lo, s.lo
    t.hi[0] = prmt(nq, ns, 0x1357u) & 0xFFFFFF00u;   // high bytes: 0, (-s).hi, (-s q2).hi, (-s q1).hi
    t.hi[1] = prmt(q12, ss, 0x5317u) & 0xFFFFFF00u;  //             0, (s q1).hi, (s q2).hi, s.hi
    return t;
}
// the eight weights of row half RR in the 32-wide k block MI, as bf16 pairs in natural k order:
// out[0] = (k+0, k+1), out[1] = (k+2, k+3) of chunk 2 MI, out[2], out[3] the same of chunk 2 MI + 1
template <int RR, int MI>
__device__ __forceinline__ void w3_block(const uint32_t (&w)[6], const W3Table &t, uint32_t (&out)[4]) {
    constexpr int rho = (2 + 2 * (MI & 1) + RR) & 3;   // where the 1-bit plane keeps this selector's bits
    const uint32_t x0 = RR ? (w[MI] >> 2) : w[MI];
    const uint32_t w1 = w[4 + (MI >> 1)];
    const uint32_t y = rho == 2 ? w1 : rho == 3 ? (w1 >> 1) : rho == 0 ? (w1 << 2) : (w1 << 1);
    const uint32_t sel = (x0 & 0x33333333u) | (y & 0x44444444u), sel1 = sel >> 16;
    // selector nibble n = 2 a + h of half-word e holds k = 16 a + 4 t + 2 h + e
    const uint32_t l0 = prmt(t.lo[0], t.lo[1], sel), h0 = prmt(t.hi[0], t.hi[1], sel);
    const uint32_t l1 = prmt(t.lo[0], t.lo[1], sel1), h1 = prmt(t.hi[0], t.hi[1], sel1);
    const uint32_t e0a = prmt(l0, h0, 0x5140u), e0b = prmt(l0, h0, 0x7362u);   // (k+0, k+2) of chunks 2 MI, 2 MI + 1
    const uint32_t e1a = prmt(l1, h1, 0x5140u), e1b = prmt(l1, h1, 0x7362u);   // (k+1, k+3)
    out[0] = prmt(e0a, e1a, 0x5410u); out[1] = prmt(e0a, e1a, 0x7632u);
    out[2] = prmt(e0b, e1b, 0x5410u); out[3] = prmt(e0b, e1b, 0x7632u);
}

struct TcParams {
    uint16_t *y;
    int *status;
    Dims d;
    GroupTable groups;    // an ordinary product is one group; a routed one (whole tiles only) has several
    int raw_stage_bytes;  // tile_bytes rounded up to 1024
    float *partial;       // stream-K: fp32 partial tiles [CTA][2][BNT][128]
    int *counters;        // stream-K: layout tiles done, one per output tile
    int MT;               // token tiles
    int64_t t_full;       // tiles (of a CTA or a CTA pair) computed whole
    int p2;               // CTAs or pairs that share the units of the remaining tiles (stream-K)
    bool f16;             // activations and output are binary16 instead of bfloat16 (the weights are decoded to match)
};

// ---------------------------------------------------------------- the kernel (model dtype)
// PAIR: two CTAs of a cluster compute 256 channels x BN NACC tokens with one stream of MMAs (cta_group::2).  Each decodes
// its own 128 channels and loads HALF of the tokens, which the other half of the instruction reads from the partner's
// shared memory.  Without that every SM reads all BN NACC tokens: 64 KB per 64-wide block at 512 tokens, against
// 1048 cycles of MMA -- the 64 bytes a cycle that an SM can take from L2.  Measured (W4 G128, before -> now, with the
// one-barrier ring below): a 64-wide block of a 128 x 512 tile 1580 -> 1060 cycles; linears of an 8B layer at M = 1024
// 492 -> 423 us, at M = 200 168 -> 158 us; 70B gate_up, W3, M = 4096 3290 -> 2760 .. 2840 us (some 1370
// TFLOP/s, under the power limit).
//
// The operand ring: a stage is one 64-wide k block, the decoded weights (16 KB) and the activations, filled behind one
// barrier and freed by one commit (the issuing thread is on the critical path at small token tiles: with a barrier
// and a commit for each operand it spent 560 cycles on a block of 256 cycles of MMA).  Up to eight stages beside four raw
// tiles (two where a stage holds 512 tokens); raw tiles take what is left, up to six.
constexpr int tc_b_stage_bytes(int BN, int NACC, bool PAIR) { return NACC * (PAIR ? BN / 2 : BN) * 128; }
constexpr int tc_raw_stage_bytes(int B, int G) { return (2048 * B + 1024 * (TILE / G) + 1023) / 1024 * 1024; }
constexpr int tc_table_bytes(int B) { return B == 4 ? DEC_WARPS * W4_TABLE_BYTES : 0; }
constexpr int TC_SMEM = 226 * 1024 - 512;
// Stages that fit beside `raw` raw tiles.
constexpr int tc_stages_beside(int B, int G, int BN, int NACC, bool PAIR, int raw) {
    const int n = (TC_SMEM - tc_table_bytes(B) - raw * tc_raw_stage_bytes(B, G)) / (A_STAGE_BYTES + tc_b_stage_bytes(BN, NACC, PAIR));
    return n > 8 ? 8 : n;
}
// Two raw tiles for each of the two decoder sets, of W4 at 512 tokens only if four operand stages remain beside them (its decode
// keeps up with the MMAs on one tile and three stages do not): with one, a set that has
// used its tile waits a whole copy for the next.  (Spending that memory on a fifth to eighth operand stage instead had made
// wide codes slower than before the rings were joined.  W8 G128, before / one raw tile / two: 28672 x 4096, 64 tokens 69.3 /
// 74.7 / 60.3 us, 256 tokens 81.3 / 91.0 / 68.5; 4096 x 14336, 64 tokens 39.3 / 42.7 / 34.4, 256 tokens 50.2 / 53.7 / 45.2.)
constexpr int tc_stages(int B, int G, int BN, int NACC, bool PAIR) {
    const int n = tc_stages_beside(B, G, BN, NACC, PAIR, 4);
    return n >= 4 || !(B == 4 && PAIR) ? n : tc_stages_beside(B, G, BN, NACC, PAIR, 2);
}
constexpr int tc_ring_bytes(int B, int G, int BN, int NACC, bool PAIR) { return tc_stages(B, G, BN, NACC, PAIR) * (A_STAGE_BYTES + tc_b_stage_bytes(BN, NACC, PAIR)); }
constexpr int tc_raw_stages(int B, int G, int BN, int NACC, bool PAIR) {
    const int n = (TC_SMEM - tc_table_bytes(B) - tc_ring_bytes(B, G, BN, NACC, PAIR)) / tc_raw_stage_bytes(B, G);
    // an even number: a stage then belongs to one decoder set, which sees every phase of its barrier (a wait tells two phases
    // apart, so a set that skipped one could take a tile that is still being copied for its own)
    return n > 6 ? 6 : n < 2 ? 2 : n & ~1;
}
// The rings a kernel is compiled with.
// Operand stages: at least three, because a set waits for every second pair of blocks only, and its last wait has to tell it
// that the stage's phase before the one it waits for is over.
constexpr bool tc_rings_ok(int B, int G, int BN, int NACC, bool PAIR) {
    const int st = tc_stages(B, G, BN, NACC, PAIR), raw = tc_raw_stages(B, G, BN, NACC, PAIR);
    return st >= 3 && raw % 2 == 0 && (raw >= 4 || (B == 4 && BN * NACC == 512 && st >= 4))
        && tc_ring_bytes(B, G, BN, NACC, PAIR) + raw * tc_raw_stage_bytes(B, G) + tc_table_bytes(B) + 512 <= 227 * 1024;
}

// Whether a kernel starts while the one before it drains.  Not the 256-token tiles of one CTA: they leave SMs idle and share their
// tiles along K, and the next kernel's CTAs and prefetches on those SMs cost more than the launch they hide (4096 square, W4,
// 130 / 200 / 256 tokens 20.6 / 21.5 / 22.2 us one after another, 21.3 / 22.1 / 22.8 overlapped).
constexpr bool tc_overlaps(int BN, int NACC, bool PAIR) { return PAIR || BN * NACC < 256; }

__device__ __forceinline__ void named_barrier_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// The work of one CTA or CTA pair ("unit").  The output is cut into tiles of 128 (256) channels x BNT tokens (tile =
// mt * NBU + nb, so that units running side by side read the same activations), each tile into its KT layout tiles
// along K.  Units 0 .. t_full - 1 compute one whole tile each; the hardware hands them to the SMs as these become free,
// and units that start together sweep K in step, so the activations they share stay in L2.
// Stream-K: the steps (tile, k) of the remaining tiles are dealt out as p2 contiguous runs, unit t_full + c
// owning [floor(V2 c / p2), floor(V2 (c + 1) / p2)), never more than one tile long; a run may begin and end
// inside a tile, and a tile shared by several units is finished by the last of them to arrive.
struct Seg { int nb, mt, k0, k1; int64_t tile; };   // nb: row block of this CTA; tile: of the unit
template <bool SK, bool PAIR>
struct SegWalk {
    int64_t t_full, v, v_end, V2;
    int KT, NBU, p2, c2, unit, rank;
    int grp;              // this unit's group
    bool whole_left;
    __device__ SegWalk(const TcParams &prm, int rank_) {
        rank = rank_;
        unit = PAIR ? (int)blockIdx.x >> 1 : (int)blockIdx.x;
        grp = 0;
        if constexpr (!SK) {
            while (grp + 1 < prm.groups.n && unit >= prm.groups.g[grp + 1].unit0) ++grp;
            unit -= prm.groups.g[grp].unit0;
        }
        KT = prm.d.KT; NBU = PAIR ? (prm.d.NB + 1) / 2 : prm.d.NB;
        if constexpr (!SK) {   // one whole tile per unit, nothing else
            p2 = 0; c2 = 0; t_full = 0; v = v_end = V2 = 0; whole_left = true;
            return;
        }
        p2 = prm.p2; t_full = prm.t_full;
        whole_left = unit < t_full;
        c2 = (int)(unit - t_full);   // index of the run
        V2 = ((int64_t)NBU * prm.MT - t_full) * KT;
        if (!whole_left) { v = (V2 * c2) / p2; v_end = (V2 * (c2 + 1)) / p2; }
        else { v = 0; v_end = 0; }
    }
    __device__ bool next(Seg &s) {
        if (whole_left) {
            whole_left = false;
            s.tile = unit; s.k0 = 0; s.k1 = KT;
        } else {
            if (v >= v_end) return false;
            const int64_t tl = v / KT;
            s.tile = t_full + tl;
            s.k0 = (int)(v - tl * KT);
            const int64_t ve = min(v_end, (tl + 1) * KT);
            s.k1 = s.k0 + (int)(ve - v);
            v = ve;
        }
        s.mt = (int)(s.tile / NBU);
        const int nbu = (int)(s.tile - (int64_t)s.mt * NBU);
        s.nb = PAIR ? 2 * nbu + rank : nbu;
        return true;
    }
};

// Columns that the MMAs of an accumulator of BN tokens compute when `rows` tokens are left for it: a multiple of 16 (of a pair:
// 32), none if there are none.  The shared-memory tile and the tensor memory keep their places for all BN; what lies beyond is
// neither computed nor stored.  (200 tokens in a tile of 256: a layout tile takes 0.81 of the MMA time.)
__device__ __forceinline__ int mma_columns(int64_t rows, int BN, bool pair) { return rows <= 0 ? 0 : rows >= BN ? BN : pair ? ((int)rows + 31) & ~31 : ((int)rows + 15) & ~15; }

// One CTA computes tiles of 128 output channels x (NACC * BN) tokens: NACC accumulators of BN columns share
// every decoded weight tile, which halves the decode work per flop at NACC = 2.
template <int B, int G, int BN, int NACC, bool PAIR, bool SK>
__global__ void __launch_bounds__(TC_THREADS, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ TcParams prm) {
    constexpr int GPT = TILE / G;
    constexpr int STAGES = tc_stages(B, G, BN, NACC, PAIR);  // ring of 64-wide k blocks
    constexpr int RAW_STAGES = tc_raw_stages(B, G, BN, NACC, PAIR);
    constexpr int BROWS = PAIR ? BN / 2 : BN;          // tokens of one TMA box and CTA
    constexpr int B_TILE_BYTES = BROWS * 128;          // one TMA box: BROWS tokens x 64 k
    constexpr int B_STAGE_BYTES = tc_b_stage_bytes(BN, NACC, PAIR);
    constexpr int BNT = BN * NACC;                     // tokens per tile
    constexpr uint32_t TMEM_COLS = BNT < 32 ? 32 : BNT;
    extern __shared__ __align__(1024) uint8_t smem[];  // 1024-byte alignment is what the swizzled tiles need
    uint8_t *sA = smem;                                        // STAGES x 16 KB
    uint8_t *sB = sA + STAGES * A_STAGE_BYTES;                 // STAGES x NACC x BROWS x 128 B
    uint8_t *sRaw = sB + STAGES * B_STAGE_BYTES;               // RAW_STAGES x raw_stage_bytes
    uint8_t *sTab = sRaw + RAW_STAGES * prm.raw_stage_bytes;   // W4: DEC_WARPS x W4_TABLE_BYTES
    uint64_t *bars = reinterpret_cast<uint64_t *>(sTab + tc_table_bytes(B));
    uint64_t *full = bars, *empty = full + STAGES;
    uint64_t *raw_full = empty + STAGES, *raw_empty = raw_full + RAW_STAGES, *acc_full = raw_empty + RAW_STAGES, *acc_empty = acc_full + 1;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_empty + 1);
    volatile int *s_last_p = reinterpret_cast<volatile int *>(tmem_slot + 1);    // "this CTA completes the tile"
    volatile int *gave_up = reinterpret_cast<volatile int *>(tmem_slot + 2);     // a bounded wait ran out somewhere in the CTA

    const Dims &d = prm.d;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = PAIR ? (int)cluster_rank() : 0;

    if ((smem_u32(smem) & 1023u) != 0) {  // cannot happen with the alignment attribute; never run misaligned
        if (threadIdx.x == 0) atomicCAS(prm.status, 0, 9);
        return;
    }
    // The kernel before this one may still be running (launch_overlapped): until its results are waited for, below, the barriers
    // and the tensor memory are set up and the first raw tiles are brought to L2 (not further: L2 sees every write to them).
    if (warp == 0 && lane == 0) prefetch_tensormap(&xmap);
    if (tc_overlaps(BN, NACC, PAIR) && warp == 2 + DEC_WARPS && lane == 0) {
        SegWalk<SK, PAIR> first(prm, rank);
        Seg s0;
        if (first.next(s0))
            prefetch_l2((const uint8_t *)prm.groups.g[SK ? 0 : first.grp].layout + ((size_t)min(s0.nb, d.NB - 1) * d.KT + s0.k0) * (size_t)d.tile_bytes,
                        (uint32_t)(min(s0.k1 - s0.k0, RAW_STAGES) * d.tile_bytes));
    }
    if (threadIdx.x == 0) {
        // full: the decoders of a set (of both CTAs of a pair) and the thread that announces the activations' bytes
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], (PAIR ? 2 * SET_WARPS : SET_WARPS) + 1); mbar_init(&empty[s], 1); }
        for (int s = 0; s < RAW_STAGES; ++s) { mbar_init(&raw_full[s], 1); mbar_init(&raw_empty[s], SET_WARPS); }
        mbar_init(acc_full, 1);
        mbar_init(acc_empty, PAIR ? 2 * DEC_WARPS : DEC_WARPS);
        fence_barrier_init();
        *gave_up = 0;
    }
    if (warp == 1) {
        if constexpr (PAIR) tmem_alloc_pair(tmem_slot, TMEM_COLS);
        else { tmem_alloc(tmem_slot, TMEM_COLS); tmem_relinquish(); }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) cluster_sync();   // the partner's barriers are initialised before anything arrives on them
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    wait_for_previous_kernel();   // x, y and the workspace belong to the kernels before until here

    // Every wait is bounded.  One that runs out records its code in the status word and raises the CTA's flag;
    // from then on no role waits any more, but each still walks its loops to the end (the decoders meet at
    // named barriers, so none of them may leave early): the output is then undefined and the status says so.
    auto wait = [&](uint64_t *bar, uint32_t parity, int code) {
        if (!mbar_wait(bar, parity, prm.status, code, WAIT_LIMIT_CYCLES, gave_up)) *gave_up = 1;
    };

    SegWalk<SK, PAIR> walk(prm, rank);
    const Group &group = prm.groups.g[SK ? 0 : walk.grp];
    Seg seg;
    if (warp == 0) {
        // ===== producer of the activation tiles.  Nothing but the wait for the stage stands between the MMAs
        // that free it and the TMA that refills it: with two stages that latency is on the critical path.
        if (lane == 0) {
            int kbc = 0;     // 64-wide k blocks issued so far (they index the ring)
            while (walk.next(seg)) {
                for (int t = seg.k0; t < seg.k1; ++t) {
                    for (int half_k = 0; half_k < 2; ++half_k, ++kbc) {
                        const int s = kbc % STAGES;
                        if (kbc >= STAGES) wait(&empty[s], ((kbc / STAGES) - 1) & 1, 2);
                        // a pair's stage is announced once, on the barrier of the CTA that issues the MMAs
                        if (rank == 0) mbar_arrive_expect_tx(&full[s], (PAIR ? 2 : 1) * B_STAGE_BYTES);
#pragma unroll
                        for (int a = 0; a < NACC; ++a) {
                            uint8_t *dst = sB + s * B_STAGE_BYTES + a * B_TILE_BYTES;
                            // of a pair, each CTA brings half of the columns that are computed
                            const int half_n = PAIR ? mma_columns((int64_t)group.rows - (int64_t)seg.mt * BNT - a * BN, BN, PAIR) / 2 : 0;
                            const int tok = group.row0 + seg.mt * BNT + a * BN + rank * half_n;
                            if constexpr (PAIR) tma_load_2d_pair(dst, &xmap, map_to_rank(&full[s], 0), (2 * t + half_k) * 64, tok);
                            else tma_load_2d(dst, &xmap, &full[s], (2 * t + half_k) * 64, tok);
                        }
                    }
                }
            }
        }
    } else if (warp == 2 + DEC_WARPS) {
        // ===== producer of the raw layout tiles (its own warp, so that a wait for the decoders never delays
        // an activation tile)
        if (lane == 0) {
            int tcnt = 0;    // layout tiles issued so far
            while (walk.next(seg)) {
                const int nb = min(seg.nb, d.NB - 1);   // the second CTA of a last, half pair decodes what nobody stores
                const uint8_t *tiles = (const uint8_t *)group.layout + (size_t)nb * d.KT * (size_t)d.tile_bytes;
                for (int t = seg.k0; t < seg.k1; ++t, ++tcnt) {
                    const int rs = tcnt % RAW_STAGES;
                    if (tcnt >= RAW_STAGES) wait(&raw_empty[rs], ((tcnt / RAW_STAGES) - 1) & 1, 1);
                    mbar_arrive_expect_tx(&raw_full[rs], (uint32_t)d.tile_bytes);
                    bulk_load(sRaw + rs * prm.raw_stage_bytes, tiles + (size_t)t * d.tile_bytes, (uint32_t)d.tile_bytes, &raw_full[rs]);
                }
            }
        }
    } else if (warp == 1) {
        // ===== MMA issuer (of a pair: rank 0).  The whole warp walks the loop, so that descriptors and addresses stay
        // uniform; one elected lane issues.
        if (rank == 0) {
            constexpr int MM = PAIR ? 256 : 128;
            auto commit = [&](uint64_t *bar) { if constexpr (PAIR) umma_commit_pair(bar); else umma_commit(bar); };
            const bool issuer = elect_one();
            int s = 0, segc = 0;
            uint32_t phase = 0;
            while (walk.next(seg)) {
                if (SK && segc > 0) wait(acc_empty, (segc - 1) & 1, 8);   // every decoder has read the accumulators of the segment before
                ++segc;
                uint32_t idesc[NACC];
                bool used[NACC];
#pragma unroll
                for (int a = 0; a < NACC; ++a) {
                    const int n = mma_columns((int64_t)group.rows - (int64_t)seg.mt * BNT - a * BN, BN, PAIR);
                    used[a] = n > 0;
                    idesc[a] = prm.f16 ? idesc_f16(n, MM) : idesc_bf16(n, MM);
                }
                const int nkb = 2 * (seg.k1 - seg.k0);
                for (int i = 0; i < nkb; ++i) {
                    wait(&full[s], phase, 3);
                    tc_fence_after();
                    const uint64_t adesc = smem_desc_sw128(smem_u32(sA) + s * A_STAGE_BYTES);
                    const uint64_t bdesc0 = smem_desc_sw128(smem_u32(sB) + s * B_STAGE_BYTES);
                    if (issuer) {
#pragma unroll
                        for (int a = 0; a < NACC; ++a) {
                            if (NACC > 1 && !used[a]) continue;
                            const uint64_t bdesc = bdesc0 + (uint64_t)(a * (B_TILE_BYTES >> 4));
#pragma unroll
                            for (int k = 0; k < 4; ++k) {  // four K = 16 steps, 32 bytes apart inside the swizzle atom
                                if constexpr (PAIR) umma_bf16_pair(tmem_base + a * BN, adesc + 2 * k, bdesc + 2 * k, idesc[a], (i | k) != 0);
                                else umma_bf16(tmem_base + a * BN, adesc + 2 * k, bdesc + 2 * k, idesc[a], (i | k) != 0);
                            }
                        }
                        commit(&empty[s]);  // frees the stage when these MMAs have read it
                    }
                    __syncwarp();
                    if (++s == STAGES) { s = 0; phase ^= 1u; }
                }
                if (issuer) commit(acc_full);   // the accumulators of this segment are complete when these MMAs are
                __syncwarp();
            }
        }
    } else {
        // ===== decoders (warps 2..17), then epilogue.  Warp rb of a set owns row block rb of every second layout tile:
        // a (row, group)'s coefficients or tables are formed once per tile, a warp meets the barriers of a 64-wide block once per
        // tile instead of twice, and the two sets hide each other's latencies.
        const int dw = warp - 2, g = lane >> 2, t = lane & 3;
        const int rb = dw & (SET_WARPS - 1), set = dw / SET_WARPS;
        const int dec_tid = threadIdx.x - 64;
        const int M = group.rows;
        uint16_t *y = prm.y + (int64_t)group.row0 * d.N;
        auto arrive = [&](uint64_t *bar) { if (PAIR && rank != 0) mbar_arrive_cluster(map_to_rank(bar, 0)); else mbar_arrive(bar); };
        int tcnt = 0, segc = 0;
        // Where the MMAs of a block are short the decoders set the pace, and a fence (some 200 cycles) is shared by a tile's
        // two blocks; a wide token tile wants its blocks as early as they are ready.
        constexpr bool ONE_FENCE = BNT <= 128 && STAGES >= 6;
        W4Lane w4{};
        uint32_t x16 = 16u;
        // wide token tiles have no register left for the sixteen, and the integer pipe is not what bounds them
        if constexpr (B == 4) { w4 = w4_lane(lane); if (BNT <= 128) x16 = c_w4_x16; }
#pragma unroll 1
        while (walk.next(seg)) {
#pragma unroll 1
        for (int tile = seg.k0; tile < seg.k1; ++tile, ++tcnt) {
            if ((tcnt & 1) != set) continue;
            const int rs = tcnt % RAW_STAGES;
            wait(&raw_full[rs], (tcnt / RAW_STAGES) & 1, 5);
            const uint8_t *raw = sRaw + rs * prm.raw_stage_bytes;
            const uint8_t *rbp = raw + rb * 256 * B;
            uint32_t w[2 * B];
            {
                constexpr int NFQ = (2 * B) / 4;
#pragma unroll
                for (int q = 0; q < NFQ; ++q) {
                    const uint4 v = *(const uint4 *)(rbp + (q * 32 + lane) * 16);
                    w[4 * q + 0] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
                }
                if constexpr ((2 * B) % 4 != 0) {
                    const uint2 v = *(const uint2 *)(rbp + NFQ * 512 + lane * 8);
                    w[4 * NFQ + 0] = v.x; w[4 * NFQ + 1] = v.y;
                }
            }
            uint2 q_lo[GPT], q_hi[GPT];   // the parameter records of rows g and g + 8; W4: of row lane / 2, whose tables the lane helps to build
            {
                const uint8_t *prow = raw + d.code_bytes + ((rb * 16 + (B == 4 ? lane >> 1 : g)) * GPT) * 8;
#pragma unroll
                for (int i = 0; i < GPT; ++i) {
                    q_lo[i] = *(const uint2 *)(prow + i * 8);
                    if constexpr (B != 4) q_hi[i] = *(const uint2 *)(prow + (8 * GPT + i) * 8);
                }
            }
            W3Table w3_lo{}, w3_hi{};   // W3: level tables of rows g and g + 8; one per tile when the group spans it
            if constexpr (B == 3 && G == 128) {
                w3_lo = w3_table(q_lo[0], prm.f16);
                w3_hi = w3_table(q_hi[0], prm.f16);
            }
            // G = 128: one group spans the tile, so its coefficients are formed once per tile, not once per 64-wide block
            RowCoef tc_lo{}, tc_hi{};
            bool tfix = false;
            if constexpr (B != 3 && B != 4 && G == 128) {
                tc_lo = make_coef<B>(q_lo[0]); tc_hi = make_coef<B>(q_hi[0]);
                tfix = B > 1 && __any_sync(0xffffffffu, (q_lo[0].x | q_hi[0].x) >> 31);
            }
            uint4 w4_lo{}, w4_hi{};     // W4: tables of rows g and g + 8 (G >= 64: of the block's one group)
            uint8_t *wtab = sTab + dw * W4_TABLE_BYTES;
            // tables of the groups gi0 .. gi0 + n - 1 (n = 1, 2) of the tile, one after another in this warp's shared memory
            auto w4_build = [&](auto g0c, auto nc) {
                constexpr int gi0 = decltype(g0c)::value, n = decltype(nc)::value;
                __syncwarp();   // the tables before have been read
#pragma unroll
                for (int e = 0; e < n; ++e) {
                    const uint2 rec = q_lo[gi0 + e];
                    auto pack = [&](float a, float b) { return pack_act2(a, b, prm.f16); };
                    w4_put(wtab + e * 256, lane, w4, rec, __uint_as_float(rec.x & 0x7FFFFFFFu), pack);
                }
                __syncwarp();
            };
            if constexpr (B == 4 && G == 128) {
                w4_build(std::integral_constant<int, 0>{}, std::integral_constant<int, 1>{});
                w4_lo = *(const uint4 *)(wtab + g * 16); w4_hi = *(const uint4 *)(wtab + (g + 8) * 16);
            }
            // the two 64-wide blocks of the tile, two 32-wide units each
            static_for<2>([&](auto hc) {
                constexpr int H = decltype(hc)::value;
                const int kb = 2 * tcnt + H, s = kb % STAGES;
                if constexpr (B == 4 && G == 64) {
                    w4_build(hc, std::integral_constant<int, 1>{});
                    w4_lo = *(const uint4 *)(wtab + g * 16); w4_hi = *(const uint4 *)(wtab + (g + 8) * 16);
                }
                if constexpr (B == 4 && G == 32) w4_build(std::integral_constant<int, 2 * H>{}, std::integral_constant<int, 2>{});
                if (kb >= STAGES) wait(&empty[s], ((kb / STAGES) - 1) & 1, 6);
                uint8_t *a_stage = sA + s * A_STAGE_BYTES;
                // rows g (low) and g + 8 (high) of the row block: their 128-byte rows in the stage
                uint8_t *row_lo = a_stage + (rb * 2 + 0) * 1024 + g * 128;
                uint8_t *row_hi = a_stage + (rb * 2 + 1) * 1024 + g * 128;
                if constexpr (B == 4) {
                    // Unit u of the block is 16-byte chunks 4 u + t of the row, swizzled by the row: lanes of odd rows take
                    // the units in the other order, which puts the eight lanes of a store phase into different banks.
                    const bool odd = (g & 1) != 0;
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int u = e ^ (g & 1);
                        if constexpr (G == 32) {
                            w4_lo = *(const uint4 *)(wtab + u * 256 + g * 16); w4_hi = *(const uint4 *)(wtab + u * 256 + (g + 8) * 16);
                        }
                        const uint32_t x_lo = odd ? w[4 * H + 2 * (1 - e)] : w[4 * H + 2 * e], x_hi = odd ? w[4 * H + 2 * (1 - e) + 1] : w[4 * H + 2 * e + 1];
                        uint32_t o_lo[4], o_hi[4];
                        w4_block(x_lo, w4_lo, x16, o_lo);
                        w4_block(x_hi, w4_hi, x16, o_hi);
                        const int off = ((4 * u + t) ^ g) * 16;
                        *(uint4 *)(row_lo + off) = make_uint4(o_lo[0], o_lo[1], o_lo[2], o_lo[3]);
                        *(uint4 *)(row_hi + off) = make_uint4(o_hi[0], o_hi[1], o_hi[2], o_hi[3]);
                    }
                } else {
                static_for<2>([&](auto uc) {
                    constexpr int JQ = 2 * H + decltype(uc)::value;    // pair of chunks 2 JQ, 2 JQ + 1 of the tile
                    constexpr int gi = (32 * JQ) / G;              // both chunks lie in this group
                    const uint2 p_lo = q_lo[gi], p_hi = q_hi[gi];
                    if constexpr (B == 3) {
                        // table decode (w3_block): no per-weight arithmetic, the reserved pattern reads zero
                        if constexpr (G < 128) { w3_lo = w3_table(p_lo, prm.f16); w3_hi = w3_table(p_hi, prm.f16); }
                        uint32_t o_lo[4], o_hi[4];
                        w3_block<0, JQ>(w, w3_lo, o_lo);
                        w3_block<1, JQ>(w, w3_hi, o_hi);
                        static_for<2>([&](auto jc) {
                            constexpr int jcv = decltype(jc)::value, jl = (2 * JQ + jcv) & 3;
                            const int off = (((2 * jl + (t >> 1)) ^ g) * 16) + (t & 1) * 8;
                            *(uint2 *)(row_lo + off) = make_uint2(o_lo[2 * jcv], o_lo[2 * jcv + 1]);
                            *(uint2 *)(row_hi + off) = make_uint2(o_hi[2 * jcv], o_hi[2 * jcv + 1]);
                        });
                    } else {
                    RowCoef c_lo, c_hi;
                    bool fix;   // reserved pattern present
                    if constexpr (G == 128) { c_lo = tc_lo; c_hi = tc_hi; fix = tfix; }
                    else { c_lo = make_coef<B>(p_lo); c_hi = make_coef<B>(p_hi); fix = B > 1 && __any_sync(0xffffffffu, (p_lo.x | p_hi.x) >> 31); }
                    auto emit = [&](auto fx, auto hx) {
                        constexpr bool FIX = decltype(fx)::value, F16 = decltype(hx)::value;
                        static_for<2>([&](auto jc) {
                            constexpr int j = 2 * JQ + decltype(jc)::value, jl = j & 3;
                            uint2 lo, hi;  // four consecutive k of one row = 8 bytes
                            lo.x = weight_pair_bf16<B, 4 * j + 0, FIX, F16>(w, c_lo);
                            hi.x = weight_pair_bf16<B, 4 * j + 1, FIX, F16>(w, c_hi);
                            lo.y = weight_pair_bf16<B, 4 * j + 2, FIX, F16>(w, c_lo);
                            hi.y = weight_pair_bf16<B, 4 * j + 3, FIX, F16>(w, c_hi);
                            // k offset inside the 64-wide block: 16 jl + 4 t -> 16-byte chunk 2 jl + t/2, swizzled by the row
                            const int chunk = (2 * jl + (t >> 1)) ^ g;
                            const int off = chunk * 16 + (t & 1) * 8;
                            *(uint2 *)(row_lo + off) = lo;
                            *(uint2 *)(row_hi + off) = hi;
                        });
                    };
                    if (!prm.f16) { if (!fix) emit(std::false_type{}, std::false_type{}); else emit(std::true_type{}, std::false_type{}); }
                    else { if (!fix) emit(std::false_type{}, std::true_type{}); else emit(std::true_type{}, std::true_type{}); }
                    }
                });
                }
                if constexpr (!ONE_FENCE) {
                    fence_proxy_async();   // generic-proxy stores -> visible to the tensor core's async proxy
                    __syncwarp();
                    if (lane == 0) arrive(&full[s]);
                }
            });
            if constexpr (ONE_FENCE) {
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) { arrive(&full[(2 * tcnt) % STAGES]); arrive(&full[(2 * tcnt + 1) % STAGES]); }
            }
            // The raw tile goes back behind the proxy fence that the operand's stores need: it orders the loads above before
            // the copy that refills the tile (release_read_stage).  Handed back right after those loads, without a fence,
            // a block of sixteen channels was wrong in one run of three at W8, 6144 x 4096, 1024 tokens.
            __syncwarp();
            if (lane == 0) mbar_arrive(&raw_empty[rs]);
        }
        // ----- epilogue of the segment: TMEM lane = output channel, column = token
        wait(acc_full, segc & 1, 7);
        ++segc;
        tc_fence_after();
        const bool whole = !SK || (seg.k0 == 0 && seg.k1 == d.KT);
        {
            const int q4 = warp & 3;                       // TMEM lane quarter this warp may access
            const int cp = dw >> 2;                        // which of four column parts
            const int64_t n = (int64_t)seg.nb * TILE + q4 * 32 + lane;
            if ((d.N & 7) == 0 && (!SK || walk.unit < prm.t_full)) {
                // A CTA whose only work is this whole tile, and rows of y that start on 16-byte boundaries: the tile goes
                // through shared memory (the operand ring is idle by now: every MMA has completed and nothing more is
                // loaded; a CTA with a run of several segments may already be loading the next one) as
                // [token][128 channels] in the output dtype, and leaves it in 16-byte pieces, eight channels of one
                // token per thread, instead of one 2-byte store per output.
                static_assert(BNT * TILE * 2 <= tc_ring_bytes(B, G, BN, NACC, PAIR), "the tile is staged in the operand ring");
                uint16_t *stage = reinterpret_cast<uint16_t *>(smem);
#pragma unroll 1
                for (int c0 = cp * 32; c0 < BNT; c0 += 128) {
                    uint32_t r[32];
                    tmem_ld32(tmem_base + ((uint32_t)(q4 * 32) << 16) + (uint32_t)c0, r);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 32; ++i) stage[(c0 + i) * TILE + q4 * 32 + lane] = float_to_act(__uint_as_float(r[i]), prm.f16);
                }
                named_barrier_sync(1, 32 * DEC_WARPS);
                const int64_t m0 = (int64_t)seg.mt * BNT, n0 = (int64_t)seg.nb * TILE;
                for (int c = dec_tid; c < BNT * (TILE / 8); c += 32 * DEC_WARPS) {
                    const int tok = c / (TILE / 8), part = c % (TILE / 8);
                    if (m0 + tok < M && n0 + part * 8 < d.N)   // N is a multiple of 8: a piece is inside or outside as a whole
                        *reinterpret_cast<uint4 *>(y + (m0 + tok) * d.N + n0 + part * 8) = *reinterpret_cast<const uint4 *>(stage + tok * TILE + part * 8);
                }
            } else if (whole) {
#pragma unroll 1
                for (int c0 = cp * 32; c0 < BNT; c0 += 128) {
                    uint32_t r[32];
                    tmem_ld32(tmem_base + ((uint32_t)(q4 * 32) << 16) + (uint32_t)c0, r);
                    tmem_ld_wait();
                    if (n < d.N) {
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            const int64_t m = (int64_t)seg.mt * BNT + c0 + i;
                            if (m < M) y[m * d.N + n] = float_to_act(__uint_as_float(r[i]), prm.f16);
                        }
                    }
                }
            } else {
                // A run has at most two partial segments: its first (which begins inside a tile) and its last
                // (which begins a tile without finishing it); each run owns two partial slots [BNT][128].
                constexpr int CW = PAIR ? 2 : 1;
                float *slot = prm.partial + (((size_t)walk.c2 * CW + rank) * 2 + (seg.k0 > 0 ? 1 : 0)) * (size_t)(BNT * TILE) + q4 * 32 + lane;
#pragma unroll 1
                for (int c0 = cp * 32; c0 < BNT; c0 += 128) {
                    uint32_t r[32];
                    tmem_ld32(tmem_base + ((uint32_t)(q4 * 32) << 16) + (uint32_t)c0, r);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 32; ++i) slot[(c0 + i) * TILE] = __uint_as_float(r[i]);
                }
            }
        }
        tc_fence_before();   // the accumulators have been read: the MMAs of the next segment may overwrite them
        if constexpr (SK) { __syncwarp(); if (lane == 0) arrive(acc_empty); }
        if (SK && !whole && seg.nb < d.NB) {
            // The tile's counter collects the layout tiles done; the CTA that completes it adds the partial tiles
            // in K order.  The first barrier orders the decoders' partial stores before the release; the acquire
            // plus the second barrier make the other CTAs' partials visible to every decoder.
            named_barrier_sync(1, 32 * DEC_WARPS);
            if (dec_tid == 0) {
                int old;
                asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;" : "=r"(old) : "l"(prm.counters + (int64_t)seg.mt * d.NB + seg.nb), "r"(seg.k1 - seg.k0) : "memory");
                *s_last_p = (old + (seg.k1 - seg.k0) == d.KT);
            }
            named_barrier_sync(1, 32 * DEC_WARPS);
            if (*s_last_p) {
                const int64_t v0 = (seg.tile - walk.t_full) * d.KT;
                const int c_first = (int)(((v0 + 1) * walk.p2 - 1) / walk.V2);                     // run that owns the tile's first unit
                const int n_contrib = (int)(((v0 + d.KT) * walk.p2 - 1) / walk.V2) - c_first + 1;   // ... up to the owner of its last
                // Four consecutive channels of one token per load; every thread keeps four such quads of up to four
                // contributors in flight (the partial tiles come from L2: it is the loads in flight that set the pace),
                // and adds the contributors in K order.
                constexpr int QUADS = BNT * TILE / 4, NTHR = 32 * DEC_WARPS;
                constexpr int CW = PAIR ? 2 : 1;
                const size_t slot_elems = (size_t)(BNT * TILE);
                for (int base = dec_tid; base < QUADS; base += 4 * NTHR) {
                    float4 sum[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) sum[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    for (int q0 = 0; q0 < n_contrib; q0 += 4) {
                        float4 v[4][4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int qd = base + u * NTHR;
#pragma unroll
                            for (int w = 0; w < 4; ++w) {
                                const int q = q0 + w;
                                v[u][w] = (qd < QUADS && q < n_contrib)
                                              ? __ldcg(reinterpret_cast<const float4 *>(prm.partial + (((size_t)(c_first + q) * CW + rank) * 2 + (q == 0 ? 0 : 1)) * slot_elems) + qd)
                                              : make_float4(0.f, 0.f, 0.f, 0.f);
                            }
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int w = 0; w < 4; ++w) { sum[u].x += v[u][w].x; sum[u].y += v[u][w].y; sum[u].z += v[u][w].z; sum[u].w += v[u][w].w; }
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int qd = base + u * NTHR;
                        if (qd >= QUADS) continue;
                        const int ml = qd / (TILE / 4), ch = (qd % (TILE / 4)) * 4;
                        const int64_t m = (int64_t)seg.mt * BNT + ml, n = (int64_t)seg.nb * TILE + ch;
                        if (m >= M) continue;
                        const float o[4] = {sum[u].x, sum[u].y, sum[u].z, sum[u].w};
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (n + e < d.N) y[m * d.N + n + e] = float_to_act(o[e], prm.f16);
                    }
                }
                if (dec_tid == 0) prm.counters[(int64_t)seg.mt * d.NB + seg.nb] = 0;  // leave the workspace ready for the next call
            }
        }
        }
    }
    if (*reinterpret_cast<volatile int *>(prm.status) != 0) {
        // a wait gave up: give copies that are still in flight time to land before shared memory is released
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000LL) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) cluster_sync();   // the partner is done with this CTA's shared memory, and this one with the partner's
    if (warp == 1) { if constexpr (PAIR) tmem_dealloc_pair(tmem_base, TMEM_COLS); else tmem_dealloc(tmem_base, TMEM_COLS); }
}

// ---------------------------------------------------------------- host side
template <int B, int G, int BN, int NACC, bool PAIR, bool SK>
cudaError_t launch_bn(const GroupTable &groups, const Dims &d, const uint16_t *x, uint16_t *y, int64_t M, TcPlan plan, int *status,
                      float *partial, int *counters, bool act_f16, cudaStream_t st) {
    EncodeTiledFn enc = encode_tiled();
    if (!enc) return cudaErrorNotSupported;
    CUtensorMap xmap;
    const cuuint64_t dims[2] = {(cuuint64_t)d.K, (cuuint64_t)M};
    const cuuint64_t strides[1] = {(cuuint64_t)d.K * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)(PAIR ? BN / 2 : BN)};
    const cuuint32_t estr[2] = {1, 1};
    if (enc(&xmap, act_f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t *>(x), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    TcParams p;
    p.groups = groups;
    if (!counters) {   // the groups of a routed call are computed in whole tiles and bring no workspace
        constexpr int CW = PAIR ? 2 : 1;
        const int NBU = (d.NB + CW - 1) / CW;
        int units = 0;
        for (int i = 0; i < groups.n; ++i) { p.groups.g[i].unit0 = units; units += NBU * ((groups.g[i].rows + BN * NACC - 1) / (BN * NACC)); }
        plan.ctas = units * CW; plan.t_full = units;
    }
    if (plan.bnt != BN * NACC || (plan.p2 > 0) != SK || (plan.cw == 2) != PAIR) return cudaErrorInvalidConfiguration;
    p.y = y; p.status = status; p.d = d;
    p.raw_stage_bytes = (d.tile_bytes + 1023) / 1024 * 1024;
    p.MT = plan.token_tiles; p.t_full = plan.t_full; p.p2 = plan.p2;
    constexpr int RAW_STAGES = tc_raw_stages(B, G, BN, NACC, PAIR);
    if (p.raw_stage_bytes != tc_raw_stage_bytes(B, G)) return cudaErrorInvalidConfiguration;
    const size_t smem = (size_t)tc_ring_bytes(B, G, BN, NACC, PAIR) + (size_t)RAW_STAGES * p.raw_stage_bytes + tc_table_bytes(B) + 512;
    static_assert(tc_rings_ok(B, G, BN, NACC, PAIR), "rings");
    auto kern = gemm_tc_kernel<B, G, BN, NACC, PAIR, SK>;
    static std::atomic<uint64_t> attr_done{0};   // per kernel instantiation: the devices it has been set on
    cudaError_t ea = ensure_func_attr(kern, attr_done, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (ea != cudaSuccess) return ea;
    p.partial = partial; p.counters = counters; p.f16 = act_f16;
    return launch_overlapped(kern, dim3((unsigned)plan.ctas), TC_THREADS, smem, st, PAIR ? 2 : 1, tc_overlaps(BN, NACC, PAIR), xmap, p);
}

// M: rows of x; plan: of the product, or (routed) the token tile of the class
template <int B, int G, bool SK>
cudaError_t launch_g(const GroupTable &groups, const Dims &d, const uint16_t *x, uint16_t *y, int64_t M, const TcPlan &plan, int *status,
                     float *partial, int *counters, bool act_f16, cudaStream_t st) {
    switch (plan.bnt) {
        case 32: return launch_bn<B, G, 32, 1, false, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
        case 64: return launch_bn<B, G, 64, 1, false, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
        case 128: return launch_bn<B, G, 128, 1, false, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
        case 256:
            if (plan.cw == 1) return launch_bn<B, G, 256, 1, false, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
            return launch_bn<B, G, 256, 1, true, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
        default: return launch_bn<B, G, 256, 2, true, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
    }
}

template <int B, bool SK>
cudaError_t launch_b(const GroupTable &groups, const Dims &d, const uint16_t *x, uint16_t *y, int64_t M, const TcPlan &plan, int *status,
                     float *partial, int *counters, bool act_f16, cudaStream_t st) {
    switch (d.G) {
        case 32: return launch_g<B, 32, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
        case 64: return launch_g<B, 64, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
        default: return launch_g<B, 128, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
    }
}

template <bool SK>
cudaError_t launch_tc_variant(const GroupTable &groups, const Dims &d, const uint16_t *x, uint16_t *y, int64_t M, const TcPlan &plan, int *status,
                              float *partial, int *counters, bool act_f16, cudaStream_t st) {
    switch (d.B) {
        case 1: return launch_b<1, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
        case 2: return launch_b<2, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
        case 3: return launch_b<3, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
        case 4: return launch_b<4, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
        case 5: return launch_b<5, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
        case 6: return launch_b<6, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
        case 7: return launch_b<7, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
        default: return launch_b<8, SK>(groups, d, x, y, M, plan, status, partial, counters, act_f16, st);
    }
}

}  // namespace
}  // namespace cq
