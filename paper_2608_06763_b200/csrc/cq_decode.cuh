// Code-pair extraction and the half2 level evaluation shared by the small-M and large-M kernels.
//
// A lane's record (cq_common.cuh) holds 32 pairs of stored codes; pair P sits in one 32-bit word per
// bit plane (pair_word / pair_pos) with its first code in the low and its second in the high 16 bits.  pair_T turns a
// pair into the normalised signed codes T = k / 2^(B-1) as half2 with one mask (the code lands in
// the fp16 mantissa under exponent bits 0x6400, value 1024 + u 2^pos) and one exact FMA; level_pair
// evaluates the group's cubic in Horner form (Eq. gpu-horner) on it.
#pragma once
#include <utility>

#include "cq_common.cuh"

namespace cq {

template <int... I, class F>
__device__ __forceinline__ void static_for_impl(F &&f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F &&f) {
    static_for_impl(static_cast<F &&>(f), std::make_integer_sequence<int, N>{});
}

// fp16 bit patterns built with integer arithmetic only (so they are compile-time constants)
constexpr uint32_t h2dup(uint32_t h) { return h | (h << 16); }
constexpr uint32_t half_pow2(int e) { return (uint32_t)((e + 15) << 10); }                      // 2^e, -14 <= e <= 15
constexpr uint32_t half_neg_pow2_plus(int q, int c) {                                            // -(2^q + c), c < 2^q, q <= 10
    return 0x8000u | (uint32_t)((q + 15) << 10) | (uint32_t)(c << (10 - q));
}
__device__ __forceinline__ __half2 as_h2(uint32_t v) { return *reinterpret_cast<__half2 *>(&v); }
__device__ __forceinline__ uint32_t as_u32(__half2 v) { return *reinterpret_cast<uint32_t *>(&v); }

// Two stored codes of pair P as packed 16-bit integers (u_lo | u_hi << 16).
template <int B, int P>
__device__ __forceinline__ uint32_t pair_codes(const uint32_t (&w)[2 * B]) {
    uint32_t u2 = 0;
    static_for<plane_count(B)>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        constexpr int pw = plane_width(B, i);
        constexpr int W = plane_word_base(B, i) + pair_word(pw, P), pos = pair_pos(pw, P);
        constexpr uint32_t m = ((1u << pw) - 1u) * 0x00010001u;
        u2 |= ((w[W] >> pos) & m) << plane_bit_offset(B, i);
    });
    return u2;
}

// Pair P as half2 of the normalised signed code:  B >= 3: T = k / 2^(B-1);  B <= 2: k itself.
// The stored code lands in the fp16 mantissa under exponent bits 0x6400 (value 1024 + u 2^pos);
// one exact FMA removes the offset and the position scale.
template <int B, int P>
__device__ __forceinline__ __half2 pair_T(const uint32_t (&w)[2 * B]) {
    static_assert(B != 4, "W4 is decoded by table (w4_block)");
    if constexpr (plane_count(B) == 1) {
        constexpr int W = pair_word(B, P), pos0 = pair_pos(B, P);
        // B = 1 keeps the field off mantissa bit 0 (the offset constant must stay representable);
        // other widths shift by 8 when the field would leave the 10 mantissa bits
        constexpr int shl = (B == 1 && pos0 <= 6) ? 1 : 0;
        constexpr int shr = (B == 1) ? (pos0 <= 6 ? 0 : 6) : (pos0 + B > 10 ? 8 : 0);
        constexpr int pos = pos0 + shl - shr;
        const uint32_t word = shl ? (w[W] << shl) : (shr ? (w[W] >> shr) : w[W]);
        constexpr uint32_t m = (((1u << B) - 1u) << pos) * 0x00010001u;
        const uint32_t hbits = (word & m) | 0x64006400u;
        constexpr uint32_t sc = (B == 1) ? half_pow2(1 - pos) : (B == 2) ? half_pow2(-pos) : half_pow2(-(pos + B - 1));
        constexpr uint32_t off = (B == 1) ? half_neg_pow2_plus(11 - pos, 1)
                               : (B == 2) ? half_neg_pow2_plus(10 - pos, 2)
                                          : half_neg_pow2_plus(10 - pos - (B - 1), 1);
        return __hfma2(as_h2(hbits), as_h2(h2dup(sc)), as_h2(h2dup(off)));
    } else {
        const uint32_t hbits = pair_codes<B, P>(w) | 0x64006400u;
        constexpr uint32_t sc = half_pow2(-(B - 1)), off = half_neg_pow2_plus(10 - (B - 1), 1);
        return __hfma2(as_h2(hbits), as_h2(h2dup(sc)), as_h2(h2dup(off)));
    }
}

// The small-M kernel's variant, arranged so that every instruction carries at most one literal: a
// logic or a packed-half instruction encodes a single immediate (and a packed-half FMA none in its
// addend), so any further constant costs a register move per use unless it lives in a register; the
// few that must are read once per kernel from constant memory (`DecodeRegs`), which keeps the
// compiler from folding them back into literals.  What comes out is the signed code in "code units":
//   B = 1:     +-1, the bit sent straight to the fp16 sign: 0xBC00 ^ (bit << 15)  (a shift and one logic op)
//   B = 2..6:  the integer k itself: the field is read as base + u under exponent bits chosen by
//              where the field sits (base = 2^(10 - pos)), and one add of the literal -(base + 2^(B-1))
//              leaves k, exactly;
//   B = 7, 8:  T = k / 2^(B-1) by one FMA (scale as the literal, offset from a register): k^3 would
//              leave the fp16 range.
// code_unit<B>() is the normalised position t of one unit: t = |T| code_unit.
template <int B>
__host__ __device__ constexpr float code_unit() {
    return B <= 2 ? 1.0f : B <= 6 ? 1.0f / (float)((1 << (B - 1)) - 1) : (float)(1 << (B - 1)) / (float)((1 << (B - 1)) - 1);
}
struct DecodeRegs { uint32_t one_neg; uint32_t off; uint32_t magic[4]; };
__constant__ uint32_t c_decode_consts[8] = {
    0xBC00BC00u,                                          // -1, -1
    0xC880C880u,                                          // -9, -9 = -(1024 + 128) / 128, the FMA addend of B = 8
    0x64006400u, 0x5C005C00u, 0x54005400u, 0x4C004C00u,   // exponent bits for a field at bit 0 / 2 / 4 / 6: base 1024 / 256 / 64 / 16
    0u, 0u};
__device__ __forceinline__ DecodeRegs load_decode_regs() {
    DecodeRegs r;
    r.one_neg = c_decode_consts[0];
    r.off = c_decode_consts[1];
#pragma unroll
    for (int i = 0; i < 4; ++i) r.magic[i] = c_decode_consts[2 + i];
    return r;
}
__device__ __forceinline__ uint32_t lop3_and_or(uint32_t a, uint32_t b, uint32_t c) {   // (a & b) | c
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
__device__ __forceinline__ uint32_t lop3_and_xor(uint32_t a, uint32_t b, uint32_t c) {  // (a & b) ^ c
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0x6A;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
template <int B, int P>
__device__ __forceinline__ __half2 pair_K(const uint32_t (&w)[2 * B], const DecodeRegs &dr) {
    static_assert(B != 4, "W4 is decoded by table (w4_block)");
    if constexpr (B == 1) {
        constexpr int W = pair_word(1, P), pos0 = pair_pos(1, P);
        const uint32_t word = pos0 == 15 ? w[W] : (w[W] << (15 - pos0));
        return as_h2(lop3_and_xor(word, 0x80008000u, dr.one_neg));
    } else if constexpr (B == 2) {
        constexpr int W = pair_word(B, P), pos0 = pair_pos(B, P);
        constexpr int shr = pos0 >= 8 ? 8 : 0, pos = pos0 - shr;
        const uint32_t word = shr ? (w[W] >> shr) : w[W];
        constexpr uint32_t m = (((1u << B) - 1u) << pos) * 0x00010001u;
        const uint32_t hbits = lop3_and_or(word, m, dr.magic[pos / 2]);     // base + u, base = 2^(10 - pos)
        constexpr uint32_t off = half_neg_pow2_plus(10 - pos, 2);           // -(base + 2^(B-1))
        return __hadd2(as_h2(hbits), as_h2(h2dup(off)));
    } else if constexpr (B == 8) {
        constexpr int W = pair_word(8, P), pos0 = pair_pos(8, P);
        const uint32_t word = pos0 ? (w[W] >> 8) : w[W];
        const uint32_t hbits = lop3_and_or(word, 0x00FF00FFu, dr.magic[0]);
        return __hfma2(as_h2(hbits), as_h2(h2dup(half_pow2(-7))), as_h2(dr.off));   // (1024 + u) / 128 - 9
    } else if constexpr (B == 7) {
        const uint32_t hbits = pair_codes<7, P>(w) | 0x64006400u;
        // (1024 + u) / 64 - 17 has no register constant of its own: -17 = 2 * (-9) + 1 is not worth a second one
        return __hfma2(as_h2(hbits), as_h2(h2dup(half_pow2(-6))), as_h2(h2dup(half_neg_pow2_plus(4, 1))));
    } else {   // B = 3, 5, 6: planes assembled, then the same add
        const uint32_t hbits = pair_codes<B, P>(w) | 0x64006400u;
        return __hadd2(as_h2(hbits), as_h2(h2dup(half_neg_pow2_plus(10, 1 << (B - 1)))));
    }
}

struct RowCoef { __half2 a2, b2, c2; float s; };

// Coefficients of q as a polynomial in T = k / 2^(B-1):  t = |T| rho, rho = 2^(B-1) / M, so
// q = |T| (a rho + |T| (b rho^2 + |T| c rho^3)), c = 1 - a - b.  Built in half2 arithmetic from the
// stored fp16 a and b (each coefficient is rounded to fp16 anyway; c rho^3 takes two FMA roundings).
constexpr uint32_t half_bits_of(float v) {   // fp16 bit pattern of a positive normal v (round to nearest, ties up)
    int e = 0;
    float m = v;
    while (m >= 2.0f) { m *= 0.5f; ++e; }
    while (m < 1.0f) { m *= 2.0f; --e; }
    const uint32_t frac = (uint32_t)((m - 1.0f) * 1024.0f + 0.5f);
    return (uint32_t)((e + 15) << 10) + frac;   // a carry out of the fraction bumps the exponent
}
template <int B>
__device__ __forceinline__ RowCoef make_coef(uint2 p) {
    RowCoef c;
    c.s = __uint_as_float(p.x & 0x7FFFFFFFu);
    if constexpr (B >= 3) {
        constexpr float rho = (float)(1 << (B - 1)) / (float)((1 << (B - 1)) - 1);
        constexpr uint32_t r1 = h2dup(half_bits_of(rho)), r2 = h2dup(half_bits_of(rho * rho)), r3 = h2dup(half_bits_of(rho * rho * rho));
        const __half2 a2 = as_h2(__byte_perm(p.y, 0, 0x1010)), b2 = as_h2(__byte_perm(p.y, 0, 0x3232));
        c.a2 = __hmul2(a2, as_h2(r1));
        c.b2 = __hmul2(b2, as_h2(r2));
        const __half2 nr3 = as_h2(r3 | 0x80008000u);
        c.c2 = __hfma2(b2, nr3, __hfma2(a2, nr3, as_h2(r3)));   // rho^3 - rho^3 a - rho^3 b
    }
    return c;
}

template <int B, bool FIX>
__device__ __forceinline__ uint32_t level_pair(__half2 T, const RowCoef &c) {
    if constexpr (FIX) {  // reserved pattern: T = -1 (B >= 3) or k = -2 (B = 2) decodes to zero
        const __half2 bad = __float2half2_rn(B == 2 ? -2.0f : -1.0f);
        T = __hmul2(T, __hne2(T, bad));
    }
    if constexpr (B >= 3) {
        const __half2 at = __habs2(T);
        return as_u32(__hmul2(T, __hfma2(at, __hfma2(at, c.c2, c.b2), c.a2)));
    } else {
        return as_u32(T);
    }
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}

// packed pairs of fp32
__device__ __forceinline__ uint64_t f2_pack(uint32_t lo, uint32_t hi) { uint64_t d; asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi)); return d; }
__device__ __forceinline__ void f2_split(uint64_t v, uint32_t &lo, uint32_t &hi) { asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t f2_dup(float v) { return f2_pack(__float_as_uint(v), __float_as_uint(v)); }
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) { uint64_t d; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d; }
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) { uint64_t d; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d; }
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) { uint64_t d; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c)); return d; }
__device__ __forceinline__ uint32_t mul_sat(uint32_t a, uint32_t b) {
    float d;
    asm("mul.rn.sat.f32 %0, %1, %2;" : "=f"(d) : "f"(__uint_as_float(a)), "f"(__uint_as_float(b)));
    return __float_as_uint(d);
}

// ---- W4: eight magnitudes of a (row, group) by table.  In the model dtype the levels are 16-bit values, kept as
// {low bytes of magnitudes 0-3, high bytes of 0-3, low bytes of 4-7, high bytes of 4-7}.  A half-word of the layout is the selector
// of four neighbouring weights; two byte permutes fetch their low and high bytes, two more put the bytes together, and the
// sign bits go into the high bytes by one exclusive or.  Twelve integer instructions and a product for eight weights, against some forty for
// the half2 polynomial, its scale in fp32 and the rounding to the operand's type; the levels themselves are evaluated in fp32
// and rounded once.  Measured on the linears of an 8B layer, G = 128: M = 1 66.6 -> 56.8 us, M = 13 109.7 -> 105.5,
// M = 200 (binary16) 194.8 -> 167.7, M = 1024 509.5 -> 491.6 (what is left there is not the decode).  The integer pipe takes one
// of these instructions every other cycle and bounds the small products, so the shift by four is a multiplication, which
// goes to another pipe: x16 is 16, read from memory so that it stays one.  out[i] = weights (2 i, 2 i + 1) of the word, in k
// order; a reserved code reads (minus) zero.
__constant__ uint32_t c_w4_x16 = 16u;
__device__ __forceinline__ void w4_block(uint32_t word, const uint4 &t, uint32_t x16, uint32_t (&out)[4]) {
    const uint32_t sel = word & 0x77777777u, sel1 = sel >> 16, w4 = word * x16;
    const uint32_t l0 = prmt(t.x, t.z, sel), h0 = prmt(t.y, t.w, sel) ^ (word & 0x80808080u);
    const uint32_t l1 = prmt(t.x, t.z, sel1), h1 = prmt(t.y, t.w, sel1) ^ (w4 & 0x80808080u);
    out[0] = prmt(l0, h0, 0x5140u); out[1] = prmt(l0, h0, 0x7362u);
    out[2] = prmt(l1, h1, 0x5140u); out[3] = prmt(l1, h1, 0x7362u);
}
// The tables of a warp's sixteen rows: lane l evaluates the four magnitudes 4 (l & 1) .. + 3 of row l >> 1, two at a time in
// packed fp32, by the Horner form of Eq. gpu-horner.
struct W4Lane { uint64_t t01, t23; };   // their positions, magnitude / 7
__device__ __forceinline__ W4Lane w4_lane(int lane) {
    const int i = 4 * (lane & 1);
    auto at = [](int k) { return __float_as_uint((float)k / 7.0f); };
    return {f2_pack(at(i), at(i + 1)), f2_pack(at(i + 2), at(i + 3))};
}
// q at the four positions; rec: the record of the lane's row
__device__ __forceinline__ void w4_curve(const W4Lane &w, uint2 rec, uint64_t &q01, uint64_t &q23) {
    const __half2 ab = as_h2(rec.y);
    const float a = __low2float(ab), b = __high2float(ab);
    const uint64_t a2 = f2_dup(a), b2 = f2_dup(b), c2 = f2_dup(__fsub_rn(__fsub_rn(1.0f, a), b));
    q01 = f2_mul(w.t01, f2_fma(w.t01, f2_fma(w.t01, c2, b2), a2));
    q23 = f2_mul(w.t23, f2_fma(w.t23, f2_fma(w.t23, c2, b2), a2));
}
// levels times f into the warp's tables, [row][16 bytes]; pack: two fp32 values to the operand's type
template <class Pack>
__device__ __forceinline__ void w4_put(uint8_t *tables, int lane, const W4Lane &w, uint2 rec, float f, Pack pack) {
    uint64_t q01, q23;
    uint32_t q[4];
    w4_curve(w, rec, q01, q23);
    f2_split(q01, q[0], q[1]); f2_split(q23, q[2], q[3]);
    const uint32_t v0 = pack(__uint_as_float(q[0]) * f, __uint_as_float(q[1]) * f), v1 = pack(__uint_as_float(q[2]) * f, __uint_as_float(q[3]) * f);
    *reinterpret_cast<uint2 *>(tables + lane * 8) = make_uint2(prmt(v0, v1, 0x6420u), prmt(v0, v1, 0x7531u));
}
// Dynamic A8: carriers (carrier_at: clamping q to [0, 1] clamps them, adding 1.5 2^23 rounds to nearest even and leaves the
// integer in the low bits), positive ones at 0 .. 7 of the row's table, negative ones at 8 .. 15.  That sum is a scalar one:
// in packed form the compiler contracts it with the product by 127 although both name their rounding, and the carrier is off
// by one wherever the fp32 product is a tie that the exact one is not.
__device__ __forceinline__ void w4_put_carriers(int8_t *tables, int lane, const W4Lane &w, uint2 rec) {
    const __half2 ab = as_h2(rec.y);
    const float a = __low2float(ab), b = __high2float(ab);
    const uint64_t a2 = f2_dup(a), b2 = f2_dup(b), c2 = f2_dup(__fsub_rn(__fsub_rn(1.0f, a), b));
    auto pair = [&](uint64_t t, uint32_t &r0, uint32_t &r1) {
        uint32_t t0, t1, h0, h1, v0, v1;
        f2_split(t, t0, t1);
        f2_split(f2_fma(t, f2_fma(t, c2, b2), a2), h0, h1);
        f2_split(f2_mul(f2_pack(mul_sat(t0, h0), mul_sat(t1, h1)), f2_dup(127.0f)), v0, v1);
        r0 = __float_as_uint(__fadd_rn(__uint_as_float(v0), 12582912.0f));
        r1 = __float_as_uint(__fadd_rn(__uint_as_float(v1), 12582912.0f));
    };
    uint32_t r[4];
    pair(w.t01, r[0], r[1]);
    pair(w.t23, r[2], r[3]);
    const uint32_t up = prmt(prmt(r[0], r[1], 0x0040u), prmt(r[2], r[3], 0x0040u), 0x5410u);   // four bytes of 0 .. 127
    uint32_t *row = reinterpret_cast<uint32_t *>(tables + (lane >> 1) * 16) + (lane & 1);
    row[0] = up;
    row[2] = (0x80808080u - up) ^ 0x80808080u;   // their negatives: no byte borrows, and zero stays zero
}

// Dynamic A8 operand order (both INT8 kernels).  One k = 32 MMA step takes the 32-wide k block m of a
// tile.  Inside it
// k = 16 a + 4 t + 2 h + e is held by lane t at byte n = 2 a + h of A register a0 / a1 (rows g / g+8)
// for e = 0 and a2 / a3 for e = 1 (small-M kernel), i.e. at byte 8 t + 4 e + n of the block, which is
// where the layout's half-words put it.  The internal activation quantiser writes x8 in the same order (W4: the
// natural order).
//
// Carriers (Eq. carrier) come from a per-(row, group) table indexed by the stored code u, so the
// sign and the reserved pattern (u = 0 -> 0) are part of the table:
//   B = 4: the table's two 8-byte halves (positive, negative) live in registers; a half-word of four
//          codes, masked to 3 bits each, is the selector of a byte permute into each half, and the
//          sign bits (expanded to byte masks by two sign-replicating permutes) pick between them; its order
//          inside the block is the natural one, lane t holding bytes 8 t .. 8 t + 7;
//   B = 3: one 8-byte table, the selector assembled from the 2-bit and the 1-bit plane;
//   B <= 2: the carriers are 0 / +-127, a constant table;
//   B = 5: four 8-byte quarters, the low three bits select in each, the upper two (one of them from the 1-bit
//          plane) pick between them;
//   B >= 6: no table (a8_row_eval).
struct CarrierTab { uint4 v[2]; };   // entries 0 .. 15 and (B = 5) 16 .. 31
template <int B>
__device__ __forceinline__ CarrierTab load_carrier_tab(const int8_t *row) {
    CarrierTab t{};
    if constexpr (B == 3) { const uint2 v = *reinterpret_cast<const uint2 *>(row); t.v[0].x = v.x; t.v[0].y = v.y; }
    if constexpr (B >= 4) t.v[0] = *reinterpret_cast<const uint4 *>(row);
    if constexpr (B == 5) t.v[1] = *reinterpret_cast<const uint4 *>(row + 16);
    return t;
}
__device__ __forceinline__ uint32_t pick(uint32_t mask, uint32_t a, uint32_t b) { return (a & mask) | (b & ~mask); }
template <int B, int RR, int MI>
__device__ __forceinline__ void a8_row_regs(const uint32_t (&w)[2 * B], const CarrierTab &ct, uint32_t x16, uint32_t &lo, uint32_t &hi) {
    static_assert(B <= 5, "wider codes are evaluated one by one (a8_row_eval)");
    const uint4 &tab = ct.v[0];
    if constexpr (B == 5) {
        constexpr int rho = (2 + 2 * (MI & 1) + RR) & 3;   // where the 1-bit plane keeps the top bits: bit 4 n + rho
        const uint32_t word = w[2 * MI + RR], z = w[plane_word_base(5, 1) + (MI >> 1)] << (3 - rho);
        const uint32_t ws = word & 0x77777777u, wh = ws >> 16, w4 = word << 4, z4 = z << 4;
        const uint32_t m_lo = prmt(w4, word, 0xD9C8u), m_hi = prmt(w4, word, 0xFBEAu);   // 0xFF where bit 3 is set
        const uint32_t k_lo = prmt(z4, z, 0xD9C8u), k_hi = prmt(z4, z, 0xFBEAu);         // 0xFF where bit 4 is set
        const uint4 &t2 = ct.v[1];
        lo = pick(k_lo, pick(m_lo, prmt(t2.z, t2.w, ws), prmt(t2.x, t2.y, ws)), pick(m_lo, prmt(tab.z, tab.w, ws), prmt(tab.x, tab.y, ws)));
        hi = pick(k_hi, pick(m_hi, prmt(t2.z, t2.w, wh), prmt(t2.x, t2.y, wh)), pick(m_hi, prmt(tab.z, tab.w, wh), prmt(tab.x, tab.y, wh)));
    } else if constexpr (B == 4) {
        const uint32_t word = w[2 * MI + RR];
        const uint32_t ws = word & 0x77777777u, wh = ws >> 16, w4 = word * x16;   // x16 = 16 (w4_block)
        const uint32_t m_lo = prmt(word, word, 0xBA98u), m_hi = prmt(w4, w4, 0xBA98u);   // 0xFF where the code is negative
        const uint32_t p_lo = prmt(tab.x, tab.y, ws), n_lo = prmt(tab.z, tab.w, ws);
        const uint32_t p_hi = prmt(tab.x, tab.y, wh), n_hi = prmt(tab.z, tab.w, wh);
        lo = (n_lo & m_lo) | (p_lo & ~m_lo);
        hi = (n_hi & m_hi) | (p_hi & ~m_hi);
    } else if constexpr (B == 3) {
        constexpr int rho = (2 + 2 * (MI & 1) + RR) & 3;   // where the 1-bit plane keeps this selector's bits
        const uint32_t x0 = RR ? (w[MI] >> 2) : w[MI];
        const uint32_t w1 = w[4 + (MI >> 1)];
        const uint32_t y = rho == 2 ? w1 : rho == 3 ? (w1 >> 1) : rho == 0 ? (w1 << 2) : (w1 << 1);
        const uint32_t sel = (x0 & 0x33333333u) | (y & 0x44444444u);
        lo = prmt(tab.x, tab.y, sel);
        hi = prmt(tab.x, tab.y, sel >> 16);
    } else if constexpr (B == 2) {
        const uint32_t sel = (RR ? (w[MI] >> 2) : w[MI]) & 0x33333333u;
        lo = prmt(0x7F008100u, 0u, sel);          // u = 0 reserved -> 0, 1 -> -127, 2 -> 0, 3 -> +127
        hi = prmt(0x7F008100u, 0u, sel >> 16);
    } else {
        constexpr int rho = (2 + 2 * (MI & 1) + RR) & 3;
        const uint32_t sel = (w[MI >> 1] >> rho) & 0x11111111u;
        lo = prmt(0x00007F81u, 0u, sel);          // bit 0 -> -127, bit 1 -> +127
        hi = prmt(0x00007F81u, 0u, sel >> 16);
    }
}

// ---- B >= 6: the carrier of each code evaluated where it is needed, two at a time in packed fp32, by the pinned
// sequence of carrier_at.  A table per (row, group) would have as many entries as the group has weights (W8, G = 128), and
// reading it costs a shared-memory access per weight with the lanes in random banks: linears of an 8B layer, W8 G128,
// M = 64: 400 us with tables, 204 us so.
struct CarrierPoly { uint64_t a, b, c; };
__device__ __forceinline__ CarrierPoly carrier_poly(uint32_t ab16) {
    const __half2 ab = as_h2(ab16);
    const float a = __low2float(ab), b = __high2float(ab);
    return {f2_dup(a), f2_dup(b), f2_dup(__fsub_rn(__fsub_rn(1.0f, a), b))};
}
// Two codes, given as fp32 2^23 + u; the signed carriers come out in the low bytes.
//   i = |u - 2^(B-1)|, exact; t = i / M, the correctly rounded quotient for every i > 0 (checked one by one): B = 7 as i r + i r',
//   r + r' = 1/M to 48 bits; B = 6 and 8 as i r plus a constant that is below half a unit of every quotient and pushes the
//   few products that round down over the tie (for i = 0 it leaves t = 2^-30 or less, whose carrier is 0 for every a and b in
//   binary16).  The multiplication saved is what W6 at G = 128 had lost to the 64-entry table it used to read
//   (4096 square, M = 8: 18.4 us with the table, 20.6 with both products); q as carrier_at has it; clamping q to [0, 1] before RNE(127 q) is clamping
//   the carrier to [0, 127]; adding 1.5 2^23 rounds to nearest even, leaving the integer in the low bits.
template <int B, bool FIX>
__device__ __forceinline__ void carrier_pair(uint32_t f0, uint32_t f1, const CarrierPoly &p, uint32_t &r0, uint32_t &r1) {
    constexpr int L = 1 << (B - 1), M = L - 1;
    constexpr float r_hi = 1.0f / (float)M;
    static_assert(B >= 6 && B <= 8, "");
    uint32_t k0, k1, t0, t1, h0, h1, v0, v1;
    f2_split(f2_add(f2_pack(f0, f1), f2_dup(-(8388608.0f + (float)L))), k0, k1);
    const uint64_t i2 = f2_pack(k0 & 0x7FFFFFFFu, k1 & 0x7FFFFFFFu);
    uint64_t t;
    if constexpr (B == 7) t = f2_fma(i2, f2_dup(r_hi), f2_mul(i2, f2_dup((float)(1.0 / (double)M - (double)r_hi))));
    else t = f2_fma(i2, f2_dup(r_hi), f2_dup(B == 6 ? 0x1p-30f : 0x1p-32f));
    f2_split(f2_fma(t, f2_fma(t, p.c, p.b), p.a), h0, h1);
    f2_split(t, t0, t1);
    uint32_t q0 = mul_sat(t0, h0), q1 = mul_sat(t1, h1);
    if constexpr (FIX) {   // the reserved pattern: the one code whose magnitude is beyond M
        if (__uint_as_float(t0) > 1.0f) q0 = 0u;
        if (__uint_as_float(t1) > 1.0f) q1 = 0u;
    }
    f2_split(f2_mul(f2_pack(q0, q1), f2_dup(127.0f)), v0, v1);
    f2_split(f2_add(f2_pack(v0 | (k0 & 0x80000000u), v1 | (k1 & 0x80000000u)), f2_dup(12582912.0f)), r0, r1);
}
template <int B, int RR, int MI, bool FIX>
__device__ __forceinline__ void a8_row_eval(const uint32_t (&w)[2 * B], const CarrierPoly &poly, uint32_t &lo, uint32_t &hi) {
    uint32_t e0[4], e1[4];   // the carriers of k + 0 and k + 1 (bytes n of lo and hi)
    static_for<4>([&](auto nc) {
        constexpr int n = decltype(nc)::value, p = 4 * (2 * MI + (n >> 1)) + 2 * (n & 1) + RR;
        uint32_t f0, f1;
        if constexpr (B == 8) {
            constexpr int W = pair_word(8, p), byte = pair_pos(8, p) / 8;
            f0 = prmt(w[W], 0x4B000000u, 0x7440u + byte);
            f1 = prmt(w[W], 0x4B000000u, 0x7440u + byte + 2);
        } else {
            const uint32_t u2 = pair_codes<B, p>(w);
            f0 = prmt(u2, 0x4B000000u, 0x7440u);
            f1 = prmt(u2, 0x4B000000u, 0x7442u);
        }
        carrier_pair<B, FIX>(f0, f1, poly, e0[n], e1[n]);
    });
    lo = prmt(prmt(e0[0], e0[1], 0x0040u), prmt(e0[2], e0[3], 0x0040u), 0x5410u);
    hi = prmt(prmt(e1[0], e1[1], 0x0040u), prmt(e1[2], e1[3], 0x0040u), 0x5410u);
}

}  // namespace cq
