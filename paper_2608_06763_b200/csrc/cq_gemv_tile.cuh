// One warp's share of the small-M products: sixteen rows of a 128 x 128 layout tile, loaded into registers, decoded and
// multiplied into fp32 sums (both small-M kernels, cq_gemv.cu and cq_gemv_strip.cu).
#pragma once
#include "cq_common.cuh"
#include "cq_decode.cuh"

namespace cq {
namespace {

// V tiles (or units) dealt out as P contiguous runs, run c = [floor(V c / P), floor(V (c + 1) / P)), and the run that holds v; none
// is empty if P <= V.  V fits 32 bits (a unit has some four hundred bytes and more) and P^2 does; 64-bit divisions, some hundred
// cycles each, would stand in the way of the first and the last tile of a short run.
__device__ __forceinline__ int run_start(unsigned c, unsigned V, unsigned P) { return (int)(c * (V / P) + c * (V % P) / P); }
__device__ __forceinline__ int run_of(unsigned v, unsigned V, unsigned P) {
    const uint64_t n = (uint64_t)(v + 1) * P - 1;
    return (n >> 32) == 0 ? (int)((unsigned)n / V) : (int)(n / V);
}

__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_s8(int (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// the same MMAs with a zero C operand (the first MMA of a group: no accumulator registers to clear)
__device__ __forceinline__ void mma_f16_z(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};\n"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.0f));
}
__device__ __forceinline__ void mma_s8_z(int (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};\n"
        : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "r"(0));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(uint32_t dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

// Activations for the fp16 products.  Sixteen lanes hold the 128 k of a token and tile, eight values each (v, in the model
// dtype); they agree on the power of two that puts the largest into [2^top, 2^(top + 1)) and leave with fp16 values.  Returns
// what takes the scale back.  Both halves of a warp need not hold work, but a half that does holds it in all its lanes.
__device__ __forceinline__ float scale_to_half(uint32_t (&v)[4], bool xf16, int top, int lane) {
    unsigned mx = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) mx = __vmaxu2(mx, v[q] & 0x7FFF7FFFu);
    const unsigned half_warp = (lane & 16) ? 0xFFFF0000u : 0x0000FFFFu;
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) mx = __vmaxu2(mx, __shfl_xor_sync(half_warp, mx, o));
    bool usable;
    const int e_max = act_max_exponent(max(mx & 0xFFFFu, mx >> 16), xf16, usable);   // the largest lies in [2^e_max, 2^(e_max + 1))
    const int sh = max(min(usable ? top - e_max : 0, 100), -100);
    const float sc = __uint_as_float((uint32_t)(127 + sh) << 23);
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = as_u32(__floats2half2_rn(act_to_float(v[q] & 0xFFFFu, xf16) * sc, act_to_float(v[q] >> 16, xf16) * sc));
    return __uint_as_float((uint32_t)(127 - sh) << 23);
}
// Chunk c (eight values) of a tile's 128 staged activations; W3 reads them in the operand order of cq_decode.cuh.
template <int B>
__device__ __forceinline__ void store_half_chunk(__half *tile, int c, const uint32_t (&v)[4]) {
    if constexpr (B != 3) {
        *reinterpret_cast<uint4 *>(tile + c * 8) = make_uint4(v[0], v[1], v[2], v[3]);
    } else {
        __half *blk = tile + (c >> 2) * 32 + 16 * (c & 1) + 2 * ((c >> 1) & 1);   // t = 2 (c & 1), a = (c >> 1) & 1
#pragma unroll
        for (int tt = 0; tt < 2; ++tt) {   // values k+0, k+2 (e = 0) | k+1, k+3 (e = 1) of t = 2 (c & 1) + tt
            *reinterpret_cast<uint32_t *>(blk + 8 * tt) = prmt(v[2 * tt], v[2 * tt + 1], 0x5410u);
            *reinterpret_cast<uint32_t *>(blk + 8 * tt + 4) = prmt(v[2 * tt], v[2 * tt + 1], 0x7632u);
        }
    }
}

template <int B, int GPT>
struct TileRegs {
    uint32_t w[2 * B];
    uint2 prm[B == 4 ? 1 : 2][GPT];  // {s bits, a | b << 16} of rows g and g + 8; W4: of row lane / 2, whose tables the lane helps to build
};
// where a lane's records begin, behind those of the row block
template <int B, int GPT>
__device__ __forceinline__ int record_offset(int lane) { return (B == 4 ? lane >> 1 : lane >> 2) * GPT * 8; }

// Streaming loads of weights.  Not through the non-coherent path: it asks that the memory is not written while the kernel
// runs, and the kernel may have started before the one that writes it had ended (launch_overlapped).
__device__ __forceinline__ uint4 ld_stream16(const void *p) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 ld_stream8(const void *p) {
    uint2 v;
    asm volatile("ld.global.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
template <int B, int GPT, class T>
__device__ __forceinline__ void load_tile_g(T &r, const uint8_t *wl, const uint8_t *pl, int lane) {
    constexpr int NFQ = (2 * B) / 4;
#pragma unroll
    for (int q = 0; q < NFQ; ++q) {
        const uint4 v = ld_stream16(wl + q * 512);
        r.w[4 * q + 0] = v.x; r.w[4 * q + 1] = v.y; r.w[4 * q + 2] = v.z; r.w[4 * q + 3] = v.w;
    }
    if constexpr ((2 * B) % 4 != 0) {
        const uint2 v = ld_stream8(wl + NFQ * 512 - lane * 8);
        r.w[4 * NFQ + 0] = v.x; r.w[4 * NFQ + 1] = v.y;
    }
#pragma unroll
    for (int gi = 0; gi < GPT; ++gi) {
        r.prm[0][gi] = ld_stream8(pl + gi * 8);
        if constexpr (B != 4) r.prm[1][gi] = ld_stream8(pl + (8 * GPT + gi) * 8);
    }
}
// A warp's slice of a ring stage -> registers.  wl = stage + row-block base + lane * 16 (codes);
// pl = parameter record of row g of the row block.
template <int B, int GPT>
__device__ __forceinline__ void load_tile(TileRegs<B, GPT> &r, const uint8_t *wl, const uint8_t *pl, int lane) {
    constexpr int NFQ = (2 * B) / 4;
#pragma unroll
    for (int q = 0; q < NFQ; ++q) {
        const uint4 v = *reinterpret_cast<const uint4 *>(wl + q * 512);
        r.w[4 * q + 0] = v.x; r.w[4 * q + 1] = v.y; r.w[4 * q + 2] = v.z; r.w[4 * q + 3] = v.w;
    }
    if constexpr ((2 * B) % 4 != 0) {
        const uint2 v = *reinterpret_cast<const uint2 *>(wl + NFQ * 512 - lane * 8);  // the tail is indexed lane * 8, not lane * 16
        r.w[4 * NFQ + 0] = v.x; r.w[4 * NFQ + 1] = v.y;
    }
#pragma unroll
    for (int gi = 0; gi < GPT; ++gi) {
        r.prm[0][gi] = *reinterpret_cast<const uint2 *>(pl + gi * 8);
        if constexpr (B != 4) r.prm[1][gi] = *reinterpret_cast<const uint2 *>(pl + (8 * GPT + gi) * 8);
    }
}

// Per-row coefficients of the level polynomial in code units: pair_K returns the signed code T in units of
// rho = code_unit<B>() (the integer k for B <= 6, k / 2^(B-1) above), the normalised position is t = |T| rho,
// so level / s = sign(k) (a t + b t^2 + c t^3) = T (ca + |T| (cb + |T| cc)) with ca = a rho, cb = b rho^2,
// cc = c rho^3, c = 1 - a - b (Eq. gpu-horner).  Formed in fp32 from the stored fp16 a and b, then rounded to
// fp16 once.
struct RowPoly { __half2 ca, cb, cc; float s; };
template <int B>
__device__ __forceinline__ RowPoly make_poly(uint2 p) {
    RowPoly r;
    r.s = __uint_as_float(p.x & 0x7FFFFFFFu);
    if constexpr (B >= 3) {
        constexpr float rho = code_unit<B>();
        const __half2 ab = as_h2(p.y);
        const float a = __low2float(ab), b = __high2float(ab), c = (1.0f - a) - b;
        r.ca = __float2half2_rn(a * rho);
        r.cb = __float2half2_rn(b * (rho * rho));
        r.cc = __float2half2_rn(c * (rho * rho * rho));
    }
    return r;
}
// signed level / s of a pair of codes (reserved pattern -> 0 when FIX)
template <int B, int P, bool FIX>
__device__ __forceinline__ __half2 level_of_pair(const uint32_t (&w)[2 * B], const DecodeRegs &dr, const RowPoly &c) {
    __half2 T = pair_K<B, P>(w, dr);
    if constexpr (FIX) T = __hmul2(T, __hne2(T, __float2half2_rn(B == 2 ? -2.0f : B <= 6 ? -(float)(1 << (B - 1)) : -1.0f)));
    if constexpr (B >= 3) {
        const __half2 aT = __habs2(T);
        return __hmul2(T, __hfma2(aT, __hfma2(aT, c.cc, c.cb), c.ca));
    } else {
        return T;
    }
}

// One group of a tile, model dtype, M > 2 (MODE 0).  xs = staged activations (fp16), xo[tb] = element offset of
// this lane's token row of token block tb (row g of the block, clamped to the last real row) plus 4 t.
// CPG MMAs per token block into D, then acc += s * D.
template <int B, int G, int NT, int GI, bool FIX>
__device__ __forceinline__ void group_model(const TileRegs<B, TILE / G> &r, const DecodeRegs &dr, const __half *xs, const int (&xo)[NT],
                                            float (&acc)[NT][4]) {
    constexpr int CPG = G / 16;
    const RowPoly c_lo = make_poly<B>(r.prm[0][GI]), c_hi = make_poly<B>(r.prm[1][GI]);
    float D[2][NT][4];   // two accumulator sets so consecutive MMAs do not wait on each other
    static_for<CPG>([&](auto jc) {
        constexpr int jj = decltype(jc)::value, j = GI * CPG + jj;
        uint32_t A[4];
        A[0] = as_u32(level_of_pair<B, 4 * j + 0, FIX>(r.w, dr, c_lo));
        A[1] = as_u32(level_of_pair<B, 4 * j + 1, FIX>(r.w, dr, c_hi));
        A[2] = as_u32(level_of_pair<B, 4 * j + 2, FIX>(r.w, dr, c_lo));
        A[3] = as_u32(level_of_pair<B, 4 * j + 3, FIX>(r.w, dr, c_hi));
#pragma unroll
        for (int tb = 0; tb < NT; ++tb) {
            const uint2 bf = *reinterpret_cast<const uint2 *>(xs + xo[tb] + 16 * j);
            if constexpr (jj < 2) mma_f16_z(D[j & 1][tb], A, bf.x, bf.y);
            else mma_f16(D[j & 1][tb], A, bf.x, bf.y);
        }
    });
#pragma unroll
    for (int tb = 0; tb < NT; ++tb) {
        acc[tb][0] = fmaf(c_lo.s, D[0][tb][0] + D[1][tb][0], acc[tb][0]);
        acc[tb][1] = fmaf(c_lo.s, D[0][tb][1] + D[1][tb][1], acc[tb][1]);
        acc[tb][2] = fmaf(c_hi.s, D[0][tb][2] + D[1][tb][2], acc[tb][2]);
        acc[tb][3] = fmaf(c_hi.s, D[0][tb][3] + D[1][tb][3], acc[tb][3]);
    }
}

// One group of a tile, Dynamic A8: INT8 MMAs into int32 partials P_g, then acc += s * P_g.
// xs = staged INT8 activations in the order of a8_row_regs (W4: natural), xo[tb] = byte offset of this lane's token row plus 8 t;
// ctab = this warp's table space.
template <int B, int G, int NT, int GI>
__device__ __forceinline__ void group_a8(const TileRegs<B, TILE / G> &r, const int8_t *xs, const int (&xo)[NT], int8_t *ctab,
                                         const float *tt, const W4Lane &w4, uint32_t x16, int g, int t, float (&acc)[NT][4]) {
    constexpr int MPG = G / 32;                  // MMAs per group
    constexpr int L = B == 1 ? 1 : (1 << (B - 1));
    constexpr int NE = carrier_table_stride(B);   // bytes from one row's table to the next
    const uint2 p_lo = r.prm[0][GI], p_hi = r.prm[B == 4 ? 0 : 1][GI];
    CarrierPoly poly_lo{}, poly_hi{};
    bool fix = false;
    if constexpr (B >= 6) {
        poly_lo = carrier_poly(p_lo.y); poly_hi = carrier_poly(p_hi.y);
        fix = __any_sync(0xffffffffu, (p_lo.x | p_hi.x) >> 31);
    }
    CarrierTab tab_lo{}, tab_hi{};
    const int8_t *trow_lo = ctab + g * NE, *trow_hi = ctab + (g + 8) * NE;
    if constexpr (B == 4) {
        __syncwarp();
        w4_put_carriers(ctab, 4 * g + t, w4, p_lo);
        __syncwarp();
        tab_lo = load_carrier_tab<B>(trow_lo);
        tab_hi = load_carrier_tab<B>(trow_hi);
    } else if constexpr (carrier_by_table(B)) {  // lane (g, t) fills magnitudes i = t mod 4 of rows g and g + 8
        __syncwarp();
        const __half2 ab_lo = as_h2(p_lo.y), ab_hi = as_h2(p_hi.y);
        const float a_lo = __low2float(ab_lo), b_lo = __high2float(ab_lo);
        const float a_hi = __low2float(ab_hi), b_hi = __high2float(ab_hi);
        for (int i = t; i < L; i += 4) {
            const float ti = tt[i];   // i / M, divided once per CTA
            const int c_lo = carrier_at(ti, a_lo, b_lo), c_hi = carrier_at(ti, a_hi, b_hi);
            const int up = carrier_slot(B, i, false), dn = carrier_slot(B, i, true);
            ctab[g * NE + up] = (int8_t)c_lo;
            ctab[g * NE + dn] = (int8_t)(-c_lo);
            ctab[(g + 8) * NE + up] = (int8_t)c_hi;
            ctab[(g + 8) * NE + dn] = (int8_t)(-c_hi);
        }
        if (t == 0) { ctab[g * NE] = 0; ctab[(g + 8) * NE] = 0; }   // the reserved pattern
        __syncwarp();
        tab_lo = load_carrier_tab<B>(trow_lo);
        tab_hi = load_carrier_tab<B>(trow_hi);
    }
    int D[NT][4];
    static_for<MPG>([&](auto mc) {
        constexpr int mi = decltype(mc)::value, MI = GI * MPG + mi;
        uint32_t A[4];
        if constexpr (B <= 5) {
            a8_row_regs<B, 0, MI>(r.w, tab_lo, x16, A[0], A[2]);
            a8_row_regs<B, 1, MI>(r.w, tab_hi, x16, A[1], A[3]);
        } else if (!fix) {
            a8_row_eval<B, 0, MI, false>(r.w, poly_lo, A[0], A[2]);
            a8_row_eval<B, 1, MI, false>(r.w, poly_hi, A[1], A[3]);
        } else {
            a8_row_eval<B, 0, MI, true>(r.w, poly_lo, A[0], A[2]);
            a8_row_eval<B, 1, MI, true>(r.w, poly_hi, A[1], A[3]);
        }
#pragma unroll
        for (int tb = 0; tb < NT; ++tb) {
            const uint2 bf = *reinterpret_cast<const uint2 *>(xs + xo[tb] + 32 * MI);
            if constexpr (mi == 0) mma_s8_z(D[tb], A, bf.x, bf.y);
            else mma_s8(D[tb], A, bf.x, bf.y);
        }
    });
    float s_lo = __uint_as_float(p_lo.x & 0x7FFFFFFFu), s_hi = __uint_as_float(p_hi.x & 0x7FFFFFFFu);
    if constexpr (B == 4) { const float s = s_lo; s_lo = __shfl_sync(0xffffffffu, s, 2 * g); s_hi = __shfl_sync(0xffffffffu, s, 2 * g + 16); }
#pragma unroll
    for (int tb = 0; tb < NT; ++tb) {
        acc[tb][0] = fmaf(s_lo, (float)D[tb][0], acc[tb][0]);
        acc[tb][1] = fmaf(s_lo, (float)D[tb][1], acc[tb][1]);
        acc[tb][2] = fmaf(s_hi, (float)D[tb][2], acc[tb][2]);
        acc[tb][3] = fmaf(s_hi, (float)D[tb][3], acc[tb][3]);
    }
}

// One group of a tile, model dtype, W3: with only eight stored codes the group's levels are kept as a
// signed fp16 table per row -- q(1/3) and q(2/3) by the fp32 Horner form of Eq. gpu-horner, the other
// entries are 0 and +-1 (u = 0, the reserved pattern, reads 0) -- split into a low-byte and a high-byte
// register pair.  A half-word of four codes (the selector assembled from the 2-bit and the 1-bit plane,
// as in a8_row_regs) fetches four levels with two byte permutes, two more interleave the bytes into
// half2 MMA operands.  K order inside a 32-wide block is the operand order of cq_decode.cuh, which
// the staged activations follow: k = 16 a + 4 t + 2 h + e at half position 8 t + 4 e + 2 a + h.
// xo[tb] = element offset of this lane's token row plus 8 t.
template <int G, int NT, int GI>
__device__ __forceinline__ void group_model_w3(const TileRegs<3, TILE / G> &r, const __half *xs, const int (&xo)[NT], float (&acc)[NT][4]) {
    constexpr int MPG = G / 32;   // 32-wide k blocks per group, two k = 16 MMAs each
    uint32_t tlo[2][2], thi[2][2];
    float sc[2];
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
        const uint2 p = r.prm[rr][GI];
        sc[rr] = __uint_as_float(p.x & 0x7FFFFFFFu);
        const __half2 ab = as_h2(p.y);
        const float a = __low2float(ab), b = __high2float(ab), c = (1.0f - a) - b;
        constexpr float t1 = 1.0f / 3.0f, t2 = 2.0f / 3.0f;
        const float q1 = t1 * fmaf(t1, fmaf(t1, c, b), a), q2 = t2 * fmaf(t2, fmaf(t2, c, b), a);
        const uint32_t q12 = as_u32(__floats2half2_rn(q1, q2)), nq = q12 | 0x80008000u;
        constexpr uint32_t K = 0x003CBC00u;            // bytes 4..7 of a permute: 0x00, 0xBC (-1), 0x3C (+1), 0x00
        tlo[rr][0] = prmt(q12, 0u, 0x0244u);           // low bytes of  0, -1, -q2, -q1
        tlo[rr][1] = prmt(q12, 0u, 0x4204u);           //               0, q1, q2, 1
        thi[rr][0] = prmt(nq, K, 0x1354u);             // high bytes of 0, -1, -q2, -q1
        thi[rr][1] = prmt(q12, K, 0x6314u);            //               0, q1, q2, 1
    }
    float D[NT][4];
    static_for<MPG>([&](auto mc) {
        constexpr int mi = decltype(mc)::value, MI = GI * MPG + mi;
        uint32_t A[2][4];   // [e][a0 a1 a2 a3]
        static_for<2>([&](auto rc) {
            constexpr int RR = decltype(rc)::value;
            constexpr int rho = (2 + 2 * (MI & 1) + RR) & 3;   // where the 1-bit plane keeps this selector's bits
            const uint32_t x0 = RR ? (r.w[MI] >> 2) : r.w[MI];
            const uint32_t w1 = r.w[4 + (MI >> 1)];
            const uint32_t y = rho == 2 ? w1 : rho == 3 ? (w1 >> 1) : rho == 0 ? (w1 << 2) : (w1 << 1);
            const uint32_t sel = (x0 & 0x33333333u) | (y & 0x44444444u);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const uint32_t se = e ? (sel >> 16) : sel;
                const uint32_t lo4 = prmt(tlo[RR][0], tlo[RR][1], se), hi4 = prmt(thi[RR][0], thi[RR][1], se);
                A[e][RR] = prmt(lo4, hi4, 0x5140u);        // levels of n = 0, 1
                A[e][2 + RR] = prmt(lo4, hi4, 0x7362u);    // levels of n = 2, 3
            }
        });
#pragma unroll
        for (int tb = 0; tb < NT; ++tb) {
            const uint4 bf = *reinterpret_cast<const uint4 *>(xs + xo[tb] + 32 * MI);
            if constexpr (mi == 0) mma_f16_z(D[tb], A[0], bf.x, bf.y);
            else mma_f16(D[tb], A[0], bf.x, bf.y);
            mma_f16(D[tb], A[1], bf.z, bf.w);
        }
    });
#pragma unroll
    for (int tb = 0; tb < NT; ++tb) {
        acc[tb][0] = fmaf(sc[0], D[tb][0], acc[tb][0]);
        acc[tb][1] = fmaf(sc[0], D[tb][1], acc[tb][1]);
        acc[tb][2] = fmaf(sc[1], D[tb][2], acc[tb][2]);
        acc[tb][3] = fmaf(sc[1], D[tb][3], acc[tb][3]);
    }
}


// ---- the one- and two-token path (MODE 2): no MMA.  A warp-level MMA occupies the issue port of its
// scheduler for about as long as a dozen ordinary instructions, and with one token seven eighths of its
// columns are wasted; a packed-half FMA per pair of weights and token is cheaper.  Lane (g, t) keeps,
// per token, a half2 accumulator for each of its two rows (the even and the odd k of its pairs); it is
// promoted to fp32 and scaled by s once per group, and the four lanes that share a row add their
// partial sums when the row block is finished.  NT is the number of tokens; xo[tok] is the element offset
// of the token's staged row plus 4 t (W3: 8 t, operand order).  The staged activations are scaled so that
// the row maximum lies in [2^10, 2^11): sixteen products of a normalised level cannot leave the fp16 range.
__device__ __forceinline__ float h2sum(__half2 v) { return __low2float(v) + __high2float(v); }

template <int B, int G, int NT, int GI, bool FIX>
__device__ __forceinline__ void group_dot(const TileRegs<B, TILE / G> &r, const DecodeRegs &dr, const __half *xs, const int (&xo)[NT],
                                          float (&acc)[NT][4]) {
    constexpr int CPG = G / 16;
    const RowPoly c[2] = {make_poly<B>(r.prm[0][GI]), make_poly<B>(r.prm[1][GI])};
    __half2 h[NT][2];
#pragma unroll
    for (int tk = 0; tk < NT; ++tk) { h[tk][0] = __float2half2_rn(0.0f); h[tk][1] = h[tk][0]; }
    static_for<CPG>([&](auto jc) {
        constexpr int jj = decltype(jc)::value, j = GI * CPG + jj;
        uint2 xv[NT];
#pragma unroll
        for (int tk = 0; tk < NT; ++tk) xv[tk] = *reinterpret_cast<const uint2 *>(xs + xo[tk] + 16 * j);
        static_for<4>([&](auto ic) {
            constexpr int i = decltype(ic)::value, rr = i & 1;
            const __half2 lv = level_of_pair<B, 4 * j + i, FIX>(r.w, dr, c[rr]);
#pragma unroll
            for (int tk = 0; tk < NT; ++tk) h[tk][rr] = __hfma2(lv, as_h2(i < 2 ? xv[tk].x : xv[tk].y), h[tk][rr]);
        });
    });
#pragma unroll
    for (int tk = 0; tk < NT; ++tk) {
        acc[tk][0] = fmaf(c[0].s, h2sum(h[tk][0]), acc[tk][0]);
        acc[tk][2] = fmaf(c[1].s, h2sum(h[tk][1]), acc[tk][2]);
    }
}

// W3 on the dot path: the register table of group_model_w3, the levels multiplied into half2 accumulators.
template <int G, int NT, int GI>
__device__ __forceinline__ void group_dot_w3(const TileRegs<3, TILE / G> &r, const __half *xs, const int (&xo)[NT], float (&acc)[NT][4]) {
    constexpr int MPG = G / 32;
    uint32_t tlo[2][2], thi[2][2];
    float sc[2];
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
        const uint2 p = r.prm[rr][GI];
        sc[rr] = __uint_as_float(p.x & 0x7FFFFFFFu);
        const __half2 ab = as_h2(p.y);
        const float a = __low2float(ab), b = __high2float(ab), c = (1.0f - a) - b;
        constexpr float t1 = 1.0f / 3.0f, t2 = 2.0f / 3.0f;
        const float q1 = t1 * fmaf(t1, fmaf(t1, c, b), a), q2 = t2 * fmaf(t2, fmaf(t2, c, b), a);
        const uint32_t q12 = as_u32(__floats2half2_rn(q1, q2)), nq = q12 | 0x80008000u;
        constexpr uint32_t K = 0x003CBC00u;
        tlo[rr][0] = prmt(q12, 0u, 0x0244u);
        tlo[rr][1] = prmt(q12, 0u, 0x4204u);
        thi[rr][0] = prmt(nq, K, 0x1354u);
        thi[rr][1] = prmt(q12, K, 0x6314u);
    }
    __half2 h[NT][2];
#pragma unroll
    for (int tk = 0; tk < NT; ++tk) { h[tk][0] = __float2half2_rn(0.0f); h[tk][1] = h[tk][0]; }
    static_for<MPG>([&](auto mc) {
        constexpr int mi = decltype(mc)::value, MI = GI * MPG + mi;
        uint4 xv[NT];
#pragma unroll
        for (int tk = 0; tk < NT; ++tk) xv[tk] = *reinterpret_cast<const uint4 *>(xs + xo[tk] + 32 * MI);
        static_for<2>([&](auto rc) {
            constexpr int RR = decltype(rc)::value;
            constexpr int rho = (2 + 2 * (MI & 1) + RR) & 3;
            const uint32_t x0 = RR ? (r.w[MI] >> 2) : r.w[MI];
            const uint32_t w1 = r.w[4 + (MI >> 1)];
            const uint32_t y = rho == 2 ? w1 : rho == 3 ? (w1 >> 1) : rho == 0 ? (w1 << 2) : (w1 << 1);
            const uint32_t sel = (x0 & 0x33333333u) | (y & 0x44444444u);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const uint32_t se = e ? (sel >> 16) : sel;
                const uint32_t lo4 = prmt(tlo[RR][0], tlo[RR][1], se), hi4 = prmt(thi[RR][0], thi[RR][1], se);
                const __half2 l01 = as_h2(prmt(lo4, hi4, 0x5140u)), l23 = as_h2(prmt(lo4, hi4, 0x7362u));
#pragma unroll
                for (int tk = 0; tk < NT; ++tk) {
                    h[tk][RR] = __hfma2(l01, as_h2(e ? xv[tk].z : xv[tk].x), h[tk][RR]);
                    h[tk][RR] = __hfma2(l23, as_h2(e ? xv[tk].w : xv[tk].y), h[tk][RR]);
                }
            }
        });
    });
#pragma unroll
    for (int tk = 0; tk < NT; ++tk) {
        acc[tk][0] = fmaf(sc[0], h2sum(h[tk][0]), acc[tk][0]);
        acc[tk][2] = fmaf(sc[1], h2sum(h[tk][1]), acc[tk][2]);
    }
}

// ---- W4, model dtype: levels from the warp's tables (w4_block), unit scale; the group scale multiplies the fp32 group
// sum.  The staged activations keep their natural order: lane t reads the eight of its word, k = 32 MI + 8 t + i.
struct W4Rows { uint4 tab[2]; float s[2]; };   // rows g and g + 8
__device__ __forceinline__ W4Rows w4_rows(uint2 rec, uint8_t *wtab, const W4Lane &w4, int g, int t) {
    auto pack = [](float a, float b) { return as_u32(__floats2half2_rn(a, b)); };
    __syncwarp();   // the group before has been read
    w4_put(wtab, 4 * g + t, w4, rec, 1.0f, pack);
    __syncwarp();
    W4Rows r;
    r.tab[0] = *reinterpret_cast<const uint4 *>(wtab + g * 16);
    r.tab[1] = *reinterpret_cast<const uint4 *>(wtab + (g + 8) * 16);
    const float s = __uint_as_float(rec.x & 0x7FFFFFFFu);
    r.s[0] = __shfl_sync(0xffffffffu, s, 2 * g);
    r.s[1] = __shfl_sync(0xffffffffu, s, 2 * g + 16);
    return r;
}
template <int G, int NT, int GI>
__device__ __forceinline__ void group_dot_w4(const TileRegs<4, TILE / G> &r, const __half *xs, const int (&xo)[NT], uint8_t *wtab, const W4Lane &w4, uint32_t x16,
                                             int g, int t, float (&acc)[NT][4]) {
    constexpr int MPG = G / 32;
    const W4Rows w = w4_rows(r.prm[0][GI], wtab, w4, g, t);
    __half2 h[NT][2];
#pragma unroll
    for (int tk = 0; tk < NT; ++tk) { h[tk][0] = __float2half2_rn(0.0f); h[tk][1] = h[tk][0]; }
    static_for<MPG>([&](auto mc) {
        constexpr int MI = GI * MPG + decltype(mc)::value;
        uint4 xv[NT];
#pragma unroll
        for (int tk = 0; tk < NT; ++tk) xv[tk] = *reinterpret_cast<const uint4 *>(xs + xo[tk] + 32 * MI);
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
            uint32_t lv[4];
            w4_block(r.w[2 * MI + rr], w.tab[rr], x16, lv);
#pragma unroll
            for (int tk = 0; tk < NT; ++tk) {
                h[tk][rr] = __hfma2(as_h2(lv[0]), as_h2(xv[tk].x), h[tk][rr]);
                h[tk][rr] = __hfma2(as_h2(lv[1]), as_h2(xv[tk].y), h[tk][rr]);
                h[tk][rr] = __hfma2(as_h2(lv[2]), as_h2(xv[tk].z), h[tk][rr]);
                h[tk][rr] = __hfma2(as_h2(lv[3]), as_h2(xv[tk].w), h[tk][rr]);
            }
        }
    });
#pragma unroll
    for (int tk = 0; tk < NT; ++tk) {
        acc[tk][0] = fmaf(w.s[0], h2sum(h[tk][0]), acc[tk][0]);
        acc[tk][2] = fmaf(w.s[1], h2sum(h[tk][1]), acc[tk][2]);
    }
}
template <int G, int NT, int GI>
__device__ __forceinline__ void group_model_w4(const TileRegs<4, TILE / G> &r, const __half *xs, const int (&xo)[NT], uint8_t *wtab, const W4Lane &w4, uint32_t x16,
                                               int g, int t, float (&acc)[NT][4]) {
    constexpr int MPG = G / 32;
    const W4Rows w = w4_rows(r.prm[0][GI], wtab, w4, g, t);
    float D[2][NT][4];   // two accumulator sets so consecutive MMAs do not wait on each other
    static_for<MPG>([&](auto mc) {
        constexpr int mi = decltype(mc)::value, MI = GI * MPG + mi;
        uint32_t lo[4], hi[4];
        w4_block(r.w[2 * MI], w.tab[0], x16, lo);
        w4_block(r.w[2 * MI + 1], w.tab[1], x16, hi);
        const uint32_t A0[4] = {lo[0], hi[0], lo[1], hi[1]}, A1[4] = {lo[2], hi[2], lo[3], hi[3]};   // k = 8 t + 0..3 | 4..7
#pragma unroll
        for (int tb = 0; tb < NT; ++tb) {
            const uint4 bf = *reinterpret_cast<const uint4 *>(xs + xo[tb] + 32 * MI);
            if constexpr (mi == 0) { mma_f16_z(D[0][tb], A0, bf.x, bf.y); mma_f16_z(D[1][tb], A1, bf.z, bf.w); }
            else { mma_f16(D[0][tb], A0, bf.x, bf.y); mma_f16(D[1][tb], A1, bf.z, bf.w); }
        }
    });
#pragma unroll
    for (int tb = 0; tb < NT; ++tb) {
        acc[tb][0] = fmaf(w.s[0], D[0][tb][0] + D[1][tb][0], acc[tb][0]);
        acc[tb][1] = fmaf(w.s[0], D[0][tb][1] + D[1][tb][1], acc[tb][1]);
        acc[tb][2] = fmaf(w.s[1], D[0][tb][2] + D[1][tb][2], acc[tb][2]);
        acc[tb][3] = fmaf(w.s[1], D[0][tb][3] + D[1][tb][3], acc[tb][3]);
    }
}

template <int B, int G, int NT, int MODE>
__device__ __forceinline__ void compute_tile(const TileRegs<B, TILE / G> &r, const DecodeRegs &dr, const uint8_t *xs, const int (&xo)[NT],
                                             int8_t *ctab, const float *tt, const W4Lane &w4, uint32_t x16, int g, int t, float (&acc)[NT][4]) {
    constexpr int GPT = TILE / G;
    static_for<GPT>([&](auto gc) {
        constexpr int GI = decltype(gc)::value;
        if constexpr (MODE == 2 && B == 4) {
            group_dot_w4<G, NT, GI>(r, reinterpret_cast<const __half *>(xs), xo, reinterpret_cast<uint8_t *>(ctab), w4, x16, g, t, acc);
        } else if constexpr (MODE == 0 && B == 4) {
            group_model_w4<G, NT, GI>(r, reinterpret_cast<const __half *>(xs), xo, reinterpret_cast<uint8_t *>(ctab), w4, x16, g, t, acc);
        } else if constexpr (MODE == 2 && B == 3) {
            group_dot_w3<G, NT, GI>(r, reinterpret_cast<const __half *>(xs), xo, acc);
        } else if constexpr (MODE == 2) {
            const bool fix = B > 1 && __any_sync(0xffffffffu, (r.prm[0][GI].x | r.prm[1][GI].x) >> 31);
            if (!fix) group_dot<B, G, NT, GI, false>(r, dr, reinterpret_cast<const __half *>(xs), xo, acc);
            else group_dot<B, G, NT, GI, true>(r, dr, reinterpret_cast<const __half *>(xs), xo, acc);
        } else if constexpr (MODE == 0 && B == 3) {
            group_model_w3<G, NT, GI>(r, reinterpret_cast<const __half *>(xs), xo, acc);
        } else if constexpr (MODE == 0) {
            const bool fix = B > 1 && __any_sync(0xffffffffu, (r.prm[0][GI].x | r.prm[1][GI].x) >> 31);
            if (!fix) group_model<B, G, NT, GI, false>(r, dr, reinterpret_cast<const __half *>(xs), xo, acc);
            else group_model<B, G, NT, GI, true>(r, dr, reinterpret_cast<const __half *>(xs), xo, acc);
        } else {
            group_a8<B, G, NT, GI>(r, reinterpret_cast<const int8_t *>(xs), xo, ctab, tt, w4, x16, g, t, acc);
        }
    });
}

}  // namespace
}  // namespace cq
