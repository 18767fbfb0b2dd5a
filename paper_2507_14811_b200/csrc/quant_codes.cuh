// The quantizer's arithmetic on 16-element chunks of a row (Sec. 3 uniform quantizer, Sec. 4.3.2 Q_dual): loads, the
// reference form with one IEEE division, and the fast form that gives the same codes without one.  Used by the quantize
// kernels and by the GEMM of few rows, which quantizes its activations itself.
#pragma once
#include <cuda_bf16.h>
#include "sq_common.cuh"

namespace sq {
namespace {

constexpr int kVec = 16;             // elements per thread and row

// 16 consecutive elements of a row as loaded (fp32: four 128-bit words, bf16: two), converted when used
template <typename Tin> struct Raw16;
template <> struct Raw16<float> { float4 v[4]; };
template <> struct Raw16<__nv_bfloat16> { uint4 v[2]; };

__device__ __forceinline__ void load16(const float *p, Raw16<float> &r)
{
    const float4 *q = reinterpret_cast<const float4 *>(p);
#pragma unroll
    for (int i = 0; i < 4; i++) r.v[i] = __ldg(q + i);
}
__device__ __forceinline__ void load16(const __nv_bfloat16 *p, Raw16<__nv_bfloat16> &r)
{
    const uint4 *q = reinterpret_cast<const uint4 *>(p);
#pragma unroll
    for (int i = 0; i < 2; i++) r.v[i] = __ldg(q + i);
}
// piece v (16 bytes) of a row chunk
__device__ __forceinline__ void set_piece(Raw16<float> &r, int v, uint4 w)
{
    r.v[v] = make_float4(__uint_as_float(w.x), __uint_as_float(w.y), __uint_as_float(w.z), __uint_as_float(w.w));
}
__device__ __forceinline__ void set_piece(Raw16<__nv_bfloat16> &r, int v, uint4 w) { r.v[v] = w; }

// elements 4 g .. 4 g + 3 as fp32
__device__ __forceinline__ void get4(const Raw16<float> &r, int g, float (&x)[4])
{
    x[0] = r.v[g].x; x[1] = r.v[g].y; x[2] = r.v[g].z; x[3] = r.v[g].w;
}
__device__ __forceinline__ void get4(const Raw16<__nv_bfloat16> &r, int g, float (&x)[4])
{
    const uint4 v = r.v[g >> 1];
    const uint32_t w0 = (g & 1) ? v.z : v.x, w1 = (g & 1) ? v.w : v.y;
    x[0] = __uint_as_float(w0 << 16); x[1] = __uint_as_float(w0 & 0xFFFF0000u);
    x[2] = __uint_as_float(w1 << 16); x[3] = __uint_as_float(w1 & 0xFFFF0000u);
}

// Brings +infinity to the largest finite value where that is one instruction for two elements (bf16); a NaN stays one.  kBounded:
// the elements then are finite or NaN, for quant4.
template <typename Tin> constexpr bool kBounded = sizeof(Tin) == 2;
__device__ __forceinline__ uint32_t bound2(uint32_t pair)
{
    uint32_t d;
    asm("min.NaN.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(pair), "r"(0x7F7F7F7Fu));
    return d;
}
__device__ __forceinline__ void bound16(Raw16<float> &) {}
__device__ __forceinline__ void bound16(Raw16<__nv_bfloat16> &r)
{
#pragma unroll
    for (int v = 0; v < 2; v++) r.v[v] = make_uint4(bound2(r.v[v].x), bound2(r.v[v].y), bound2(r.v[v].z), bound2(r.v[v].w));
}

__device__ __forceinline__ float load1(const float *p) { return __ldg(p); }
__device__ __forceinline__ float load1(const __nv_bfloat16 *p)
{
    return __uint_as_float(uint32_t(__ldg(reinterpret_cast<const unsigned short *>(p))) << 16);
}

// two fp32 -> two e4m3 bytes (round-to-nearest-even, saturate to +-448); low byte = a.
__device__ __forceinline__ uint32_t cvt_e4m3x2(float a, float b)
{
    unsigned short r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(b), "f"(a));
    return r;
}

enum : int { kSingle = 0, kDual = 1, kZeroPoint = 2 };   // quantizer modes

// One element -> (code for the positive / only matrix, code for the negative matrix), as bytes.
// Reference form: one IEEE division, round half to even, clip.  Used where a vector straddles a
// segment bound or the end of a row, and for scales outside the range of the fast form below.
// Zero-point mode (App. A asymmetric quantizer): clip(round(x / s) + z, lo, hi), z passed in `zp`.
template <int CODE, int MODE>
__device__ __forceinline__ void quant1(float x, float sp, float sn, int zp, int lo, int hi, uint32_t &cp, uint32_t &cn)
{
    constexpr bool DUAL = MODE == kDual;
    if (CODE == SQ_CODE_INT8) {
        float s = DUAL ? (x >= 0.0f ? sp : sn) : sp;
        int c = __float2int_rn(__fdiv_rn(x, s));      // IEEE divide, round half to even, saturating convert
        if (MODE == kZeroPoint) c = max(min(c, 1000000), -1000000) + zp;
        c = max(min(c, hi), lo);
        if (DUAL) { cp = uint32_t(max(c, 0)) & 0xFFu; cn = uint32_t(min(c, 0)) & 0xFFu; }
        else      { cp = uint32_t(c) & 0xFFu; cn = 0; }
    } else {
        bool pos = x >= 0.0f;
        float s = DUAL ? (pos ? sp : sn) : sp;
        uint32_t c = cvt_e4m3x2(__fdiv_rn(x, s), 0.0f) & 0xFFu;
        if ((c & 0x7Fu) == 0) c = 0;                  // -0 is stored as +0
        if (DUAL) { cp = pos ? c : 0u; cn = pos ? 0u : c; }
        else      { cp = c; cn = 0; }
    }
}

// packed fp32 pairs: sm_100 executes mul / fma / add on two fp32 values per instruction
__device__ __forceinline__ uint64_t pack2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void unpack2u(uint64_t v, uint32_t &lo, uint32_t &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// Per-segment constants of the fast form.  The quotient x / s is obtained from the correctly rounded
// reciprocal r = RN(1/s) by one multiply and two FMAs,
//   q0 = RN(x r),  e = x - q0 s (exact in one FMA),  q = RN(q0 + e r),
// which lands on the same side of every rounding boundary of the codes (k + 1/2 for int8, the midpoints of
// adjacent e4m3 values) as RN(x / s), provided e is exact, i.e. does not underflow: |x| >= 2^-100 suffices, and for
// smaller |x| the quotient is below 2^-20 for the scales of the fast form (2^-80 <= s <= 2^100) and the code is 0
// whatever its last bits are.  (Checked on the CPU against the IEEE division for 2 * 10^10 inputs within six
// units in the last place of a rounding boundary, scales with random, all-ones and power-of-two significands.)
struct SegConst {
    float s, r;        // scale and RN(1 / s)
    float inv_l;       // e4m3 form: 1 / L with L = 2^(exponent(s) + 11) >= 1024 s
    float s_l, r_l;    // e4m3 form: s / L and RN(L / s)
    int fast;
};
__device__ __forceinline__ SegConst seg_const(float s)
{
    SegConst c;
    c.fast = (s >= 8.2718061255302767e-25f && s <= 1.2676506002282294e+30f) ? 1 : 0;     // 2^-80 .. 2^100
    c.s = s;
    c.r = __frcp_rn(s);
    const uint32_t l_bits = (__float_as_uint(s) & 0x7F800000u) + (11u << 23);
    const float l = __uint_as_float(l_bits);
    c.inv_l = __uint_as_float((254u << 23) - l_bits);
    c.s_l = s * c.inv_l;
    c.r_l = c.r * l;
    return c;
}
__device__ __forceinline__ float fma_sat(float a, float b, float c)
{
    float d;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// two quotients x / s from r = RN(1/s): q0 = RN(x r), e = x - q0 s, q = RN(q0 + e r)
__device__ __forceinline__ uint64_t div2_rn_fast(uint64_t x2, uint64_t neg_s2, uint64_t r2)
{
    const uint64_t q0 = mul2(x2, r2);
    const uint64_t e = fma2(q0, neg_s2, x2);
    return fma2(e, r2, q0);
}
// {sat_s8(hi_val), sat_s8(lo_val)} into bits 15..0 of the result, bits 15..0 of `upper` into bits 31..16
__device__ __forceinline__ uint32_t pack_sat_s8(int hi_val, int lo_val, uint32_t upper)
{
    uint32_t d;
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(hi_val), "r"(lo_val), "r"(upper));
    return d;
}

// max(-x, 0); a NaN stays one
__device__ __forceinline__ float negative_part(float x)
{
    float d;
    asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(d) : "f"(-x));
    return d;
}

constexpr float kRoundMagic = 12582912.0f;   // 1.5 * 2^23: v + magic rounds v to an integer, half to even
constexpr int kMagicBits = 0x4B400000;       // its bit pattern: bits(v + magic) - kMagicBits is that integer

// 4 elements of one K-segment -> one word of packed codes per matrix.
// int8, dual: both polarities are quantized as non-negative numbers, max(x, 0) and max(-x, 0),
//   each with its own constants.  Adding the magic constant rounds half to even; the integer is the distance of
//   the sum's bit pattern from the constant's, one of the two is zero, so the difference of the two bit patterns is the signed
//   code, a saturating pack clips it to [-128, 127] and its sign says whose it is (one subtraction and one pack for both
//   polarities: 1111 x 1072 fp32 3.5 -> 3.0 us, 8858 x 1536 15.2 -> 14.5; bf16 inputs are bound by memory or latency).  A quotient
//   beyond the range of the magic constant, infinity, or the NaN of an overflowed chain all have bit patterns above the
//   constant's, so they saturate to the end of the code range as the clip demands, provided the other polarity's input is
//   zero.  max(x, 0) - x is one instruction for two elements, but a NaN for x = +infinity (which a gated product or a
//   multiplier makes of finite inputs, too), and the two NaNs would cancel.  So it is for BOUNDED inputs, that is bf16 ones
//   (bound16) and those whose scale comes from their own maximum; the others take two maxima (an 80 us layer of
//   32768 x 1280 bf16 inputs: 0.5 us more than without a bound, 0.9 us with two maxima).  (A negative bound of -127 takes the
//   division path.)
// int8, single scale: |x| is quantized, clipped in fp32 (clip-then-round equals round-then-clip for integer
//   bounds; a NaN from an overflowed chain clips to the bound as well) and the sign put back when rounding.
// e4m3: the input is first mapped to u = sat(x / L) in [0, 1] with one saturating FMA (L a power of two, so
//   u / (s / L) has the bits of x / s; x beyond L is clipped to 448 anyway), which also splits the polarities and
//   keeps infinities and NaNs out of the saturating e4m3 conversion.
template <int CODE, int MODE, bool BOUNDED = false>
__device__ __forceinline__ void quant4(const float (&x)[4], const SegConst &cp, const SegConst &cn, float hi, int zp,
                                       uint32_t &wp, uint32_t &wn)
{
    constexpr bool DUAL = MODE == kDual;
    const uint64_t magic2 = pack2(kRoundMagic, kRoundMagic);
    if (MODE == kZeroPoint) {
        // round(|x| / s) with the sign of x (the magnitude clipped at 256: anything beyond leaves the code range
        // whatever z is; a NaN from an overflowed chain clips the same way), plus z, saturated to [-128, 127]
        const uint64_t r2 = pack2(cp.r, cp.r), ns2 = pack2(-cp.s, -cp.s);
        const int off = zp - kMagicBits;
        int k[4];
#pragma unroll
        for (int i = 0; i < 4; i += 2) {
            float a0, a1;
            unpack2(div2_rn_fast(pack2(fabsf(x[i]), fabsf(x[i + 1])), ns2, r2), a0, a1);
            k[i] = int(__float_as_uint(fmaf(fminf(a0, 256.0f), copysignf(1.0f, x[i]), kRoundMagic))) + off;
            k[i + 1] = int(__float_as_uint(fmaf(fminf(a1, 256.0f), copysignf(1.0f, x[i + 1]), kRoundMagic))) + off;
        }
        wp = pack_sat_s8(k[1], k[0], pack_sat_s8(k[3], k[2], 0u));
        return;
    }
    if (CODE == SQ_CODE_INT8 && DUAL) {
        const uint64_t rp2 = pack2(cp.r, cp.r), nsp2 = pack2(-cp.s, -cp.s);
        const uint64_t rn2 = pack2(cn.r, cn.r), nsn2 = pack2(-cn.s, -cn.s);
        int k[4];
#pragma unroll
        for (int i = 0; i < 4; i += 2) {
            const uint64_t xp2 = pack2(fmaxf(x[i], 0.0f), fmaxf(x[i + 1], 0.0f));
            const uint64_t xn2 = BOUNDED ? fma2(pack2(x[i], x[i + 1]), pack2(-1.0f, -1.0f), xp2)      // max(x, 0) - x, exact
                                         : pack2(negative_part(x[i]), negative_part(x[i + 1]));
            uint32_t p0, p1, n0, n1;
            unpack2u(add2(div2_rn_fast(xp2, nsp2, rp2), magic2), p0, p1);
            unpack2u(add2(div2_rn_fast(xn2, nsn2, rn2), magic2), n0, n1);
            k[i] = int(p0 - n0); k[i + 1] = int(p1 - n1);
        }
        const uint32_t w = pack_sat_s8(k[1], k[0], pack_sat_s8(k[3], k[2], 0u));
        uint32_t negative;                              // 0xFF in the bytes below zero
        asm("prmt.b32 %0, %1, 0, 0xBA98;" : "=r"(negative) : "r"(w));
        wp = w & ~negative;
        wn = w & negative;
        return;
    }
    uint32_t bp[4], bn[4];
    if (CODE == SQ_CODE_INT8) {                          // single scale
        const uint64_t r2 = pack2(cp.r, cp.r), ns2 = pack2(-cp.s, -cp.s);
#pragma unroll
        for (int i = 0; i < 4; i += 2) {
            float a0, a1;
            unpack2(div2_rn_fast(pack2(fabsf(x[i]), fabsf(x[i + 1])), ns2, r2), a0, a1);
            bp[i] = __float_as_uint(fmaf(fminf(a0, hi), copysignf(1.0f, x[i]), kRoundMagic));
            bp[i + 1] = __float_as_uint(fmaf(fminf(a1, hi), copysignf(1.0f, x[i + 1]), kRoundMagic));
        }
        wp = __byte_perm(__byte_perm(bp[0], bp[1], 0x0040), __byte_perm(bp[2], bp[3], 0x0040), 0x5410);
        return;
    }
    // e4m3
    const uint64_t rp2 = pack2(cp.r_l, cp.r_l), nsp2 = pack2(-cp.s_l, -cp.s_l);
    const uint64_t rn2 = pack2(cn.r_l, cn.r_l), nsn2 = pack2(-cn.s_l, -cn.s_l);
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
        float a0, a1;
        if (DUAL) {
            unpack2(div2_rn_fast(pack2(fma_sat(x[i], cp.inv_l, 0.0f), fma_sat(x[i + 1], cp.inv_l, 0.0f)), nsp2, rp2), a0, a1);
            bp[i] = __float_as_uint(a0); bp[i + 1] = __float_as_uint(a1);
            unpack2(div2_rn_fast(pack2(fma_sat(x[i], -cn.inv_l, 0.0f), fma_sat(x[i + 1], -cn.inv_l, 0.0f)), nsn2, rn2), a0, a1);
            bn[i] = __float_as_uint(a0); bn[i + 1] = __float_as_uint(a1);
        } else {
            unpack2(div2_rn_fast(pack2(fma_sat(fabsf(x[i]), cp.inv_l, 0.0f), fma_sat(fabsf(x[i + 1]), cp.inv_l, 0.0f)), nsp2, rp2), a0, a1);
            bp[i] = __float_as_uint(copysignf(a0, x[i])); bp[i + 1] = __float_as_uint(copysignf(a1, x[i + 1]));
        }
    }
    uint32_t w = cvt_e4m3x2(__uint_as_float(bp[0]), __uint_as_float(bp[1])) |
                 (cvt_e4m3x2(__uint_as_float(bp[2]), __uint_as_float(bp[3])) << 16);
    // single scale: -0 is stored as +0; dual: the positive matrix holds non-negative quotients, no -0 arises
    wp = DUAL ? w : w & ~(__vcmpeq4(w & 0x7F7F7F7Fu, 0u) & 0x80808080u);
    if (DUAL) {
        // the negative matrix was quantized as magnitudes: set the sign bit of every nonzero byte
        // (a byte b <= 0x7E plus 0x7F reaches 0x80 exactly when b >= 1, and never carries into the next byte)
        w = cvt_e4m3x2(__uint_as_float(bn[0]), __uint_as_float(bn[1])) |
            (cvt_e4m3x2(__uint_as_float(bn[2]), __uint_as_float(bn[3])) << 16);
        wn = w | ((w + 0x7F7F7F7Fu) & 0x80808080u);
    }
}

}  // namespace
}  // namespace sq
