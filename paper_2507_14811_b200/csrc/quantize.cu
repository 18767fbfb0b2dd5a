// Activation / weight quantization kernels (Sec. 3 uniform quantizer, Sec. 4.3.2 Q_dual and polarity
// split, Sec. 4.2.2 one scale per segment; App. A zero-point quantizer as a mode; the act-to-linear prologue of
// Sec. 4.3.2 compiled in on request; per-row scales and 4-bit packing for the W4A8 setting of App. B).
// HBM-streaming: every thread converts 16 consecutive elements per row (the row pieces arrive through a
// thread-private ring of asynchronous 16-byte copies in shared memory, one 128-bit store per code matrix goes out)
// and walks down the rows with that column chunk.  The codes are those of "one IEEE fp32 division, round half to
// even, clip"; the common case computes them with a handful of full-rate fp32 instructions per element (see
// SegConst) so that the pass stays memory bound.
#include <cuda_bf16.h>
#include <algorithm>
#include <atomic>
#include "quant_codes.cuh"

namespace sq {
namespace {

constexpr int kThreads = 256;
#ifndef SQ_QUANT_BLOCKS_PER_SM
#define SQ_QUANT_BLOCKS_PER_SM 4
#endif
constexpr int kBlocksPerSm = SQ_QUANT_BLOCKS_PER_SM;   // resident blocks per SM the kernel is compiled for (4: at most 64 registers)

// The act-to-linear segment in front of the quantizer (Sec. 4.3.2; App. B: SiLU and GELU feed DualScale layers),
// evaluated in fp32 and rounded once to the dtype the unfused graph would have stored the activation in.
// SiLU(h) = h sigma(h) with z = exp(-|h|): sigma = 1 / (1 + z) for h >= 0, z / (1 + z) below (no overflow).  The
// exponential is the hardware base-2 approximation of h log2(e) (the rounding of that product costs |h| 2^-24
// relative, the approximation itself about one unit in the last place) and the division the hardware's fast one
// (2 units in the last place for a divisor in [1, 2]): relative error <= (|h| + 8) 2^-23, a fraction of a bf16
// half-step (2^-9) for every |h| below the underflow of the result.
// GELU(h) = h Phi(h) with E = erfc(t), t = |h| / sqrt 2: h (1 - E / 2) for h >= 0, (h / 2) E below.
// erfc(t) = exp(-t^2) g(t); the smooth factor g (the scaled complementary error function) is a degree-9
// polynomial in z = (t - 2.5) / (t + 2.5), which maps [0, 9.6] into [-1, 0.59) (coefficients from a least-squares
// fit of the relative error on Chebyshev nodes, 2^-29, by gelu_coefficients.py; beyond t = 9.6 the exponential
// has underflowed).  t^2 is
// split into its rounded value s and the rounding error e = fma(t, t, -s), and exp(-t^2) = exp(-s) (1 - e) to
// first order, so that the rounding of the square, which the exponential would amplify by t^2, does not count.
// What remains is the hardware exponential's own error (|s| 2^-24 from the product with log2 e, one unit in the
// last place from the approximation), the fast division's 2 units and a dozen roundings: relative error
// <= (3 h^2 + 48) 2^-24; in |h| <= 4 it stays below 2^-19.  The exponential keeps subnormal results (a GELU of h < -13.2
// under a small scale, or times a large gated value, is an ordinary number; 2 us of the 8192 x 2560 gated pass).
// Both are written for TWO elements: the multiplies, FMAs and adds go two per instruction (packed fp32 pairs), each of
// them rounding exactly as the scalar instruction does, which is what bounds the fused pass (the ALUs, not memory).
// (8192 x 2560 gated GELU, dual int8, 126 MB: 49.4 us one element at a time with the gate half one row ahead in registers,
// 37.9 us with pairs and the gate half in the ring; without the table, 54 M elements of GELU 93 -> 80 us.)
// GELU without branches: with a = min(|h|, 20), v = max(h, 0) - (a / 2) E in one FMA is h - (h / 2) E for h >= 0 and
// (h / 2) E below; at a = 20 the exponential has long underflowed to zero, so v is h or +0 beyond it and t^2 stays
// finite for every h.
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float ex2_approx(float x)         // keeps subnormal results
{
    float r;
    asm("ex2.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ uint64_t dup2(float v) { return pack2(v, v); }
__device__ __forceinline__ uint64_t silu2(float h0, float h1)
{
    const float z0 = __expf(-fabsf(h0)), z1 = __expf(-fabsf(h1));
    float d0, d1, n0, n1;
    unpack2(add2(pack2(z0, z1), dup2(1.0f)), d0, d1);
    unpack2(mul2(pack2(h0, h1), pack2(z0, z1)), n0, n1);
    return mul2(pack2(h0 >= 0.0f ? h0 : n0, h1 >= 0.0f ? h1 : n1), pack2(rcp_approx(d0), rcp_approx(d1)));
}
// erfc(a / sqrt 2) for 0 <= a <= 20
__device__ __forceinline__ uint64_t gelu_tail2(uint64_t a)
{
    const uint64_t t = mul2(a, dup2(0.70710678118654752440f));
    float d0, d1;
    unpack2(add2(t, dup2(2.5f)), d0, d1);
    const uint64_t z = mul2(add2(t, dup2(-2.5f)), pack2(rcp_approx(d0), rcp_approx(d1)));
    uint64_t g = fma2(dup2(-5.388610225e-05f), z, dup2(2.161547454e-04f));
    g = fma2(g, z, dup2(8.157527773e-04f));
    g = fma2(g, z, dup2(-2.643950749e-03f));
    g = fma2(g, z, dup2(-3.974915482e-03f));
    g = fma2(g, z, dup2(3.992317244e-02f));
    g = fma2(g, z, dup2(-1.250353903e-01f));
    g = fma2(g, z, dup2(2.517131865e-01f));
    g = fma2(g, z, dup2(-3.717366457e-01f));
    g = fma2(g, z, dup2(2.108063698e-01f));
    const uint64_t s = mul2(t, t);
    const uint64_t neg_e = fma2(mul2(t, dup2(-1.0f)), t, s);      // t^2 = s - neg_e exactly
    float x0, x1;
    unpack2(mul2(s, dup2(-1.4426950408889634f)), x0, x1);
    const uint64_t E = mul2(pack2(ex2_approx(x0), ex2_approx(x1)), g);
    return fma2(E, neg_e, E);                                     // exp(-(s + e)) = exp(-s) (1 - e) to first order
}
__device__ __forceinline__ uint64_t gelu_from_tail2(float h0, float h1, uint64_t a, uint64_t E)
{
    return fma2(mul2(a, dup2(-0.5f)), E, pack2(fmaxf(h0, 0.0f), fmaxf(h1, 0.0f)));
}
__device__ __forceinline__ uint64_t gelu2(float h0, float h1)
{
    const uint64_t a = pack2(fminf(fabsf(h0), 20.0f), fminf(fabsf(h1), 20.0f));
    return gelu_from_tail2(h0, h1, a, gelu_tail2(a));
}
// two activations as the unfused graph would have stored them
template <typename Tin>
__device__ __forceinline__ uint64_t rounded2(uint64_t a)
{
    if (sizeof(Tin) == 2) {
        float a0, a1;
        unpack2(a, a0, a1);
        const __nv_bfloat162 r = __floats2bfloat162_rn(a0, a1);
        const uint32_t w = *reinterpret_cast<const uint32_t *>(&r);
        a = pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
    }
    return a;
}
// times the per-channel multipliers (one fp32 multiply)
template <typename Tin>
__device__ __forceinline__ uint64_t stored2(uint64_t a, uint64_t mult) { return mul2(rounded2<Tin>(a), mult); }
template <typename Tin>
__device__ __forceinline__ uint64_t pre2(float h0, float h1, int act, uint64_t mult)
{
    if (!act) return mul2(pack2(h0, h1), mult);
    return stored2<Tin>(act == 1 ? silu2(h0, h1) : gelu2(h0, h1), mult);
}
// Gated GELU (App. B lists GEGLU with SiLU and GELU): value * GELU(gate), the product in fp32 (one more rounding
// on top of the GELU's error: relative error <= (3 g^2 + 49) 2^-24), rounded once to the stored dtype.
template <typename Tin>
__device__ __forceinline__ uint64_t pre_gated2(float v0, float v1, float g0, float g1, uint64_t mult)
{
    return stored2<Tin>(mul2(pack2(v0, v1), gelu2(g0, g1)), mult);
}
// single elements (row tails, segment bounds inside a chunk, extreme scales)
template <typename Tin>
__device__ __forceinline__ float pre1(float h, int act, float mult)
{
    float lo, hi;
    unpack2(pre2<Tin>(h, h, act, dup2(mult)), lo, hi);
    return lo;
}
template <typename Tin>
__device__ __forceinline__ float pre_gated(float value, float gate, float mult)
{
    float lo, hi;
    unpack2(pre_gated2<Tin>(value, value, gate, gate, dup2(mult)), lo, hi);
    return lo;
}

// Thread g of the grid owns the 16-element column chunk g % V of the rows g / V, g / V + R, g / V + 2 R, ...
// (V chunks per row, R rows in flight over the whole grid), so that a warp reads 1 KiB (bf16) of consecutive
// addresses per row, the per-segment constants are made once per thread, and the next row's loads are in
// flight while the current row is converted.
// PRE != 0 compiles in the act-to-linear prologue: activation function and per-channel multiplier in front of the
// quantizer, so that the activation's output never goes through HBM.  PRE == 2 is the gated form: the row holds
// 2 K pre-activations, value half and gate half (K elements further on); both travel through the ring (fp32: the gate
// half is fetched into registers one row ahead, its ring would not fit).
// RING: depth of the shared-memory ring the rows travel through (see below); 4 when a thread has many rows to
// walk (large inputs: more bytes in flight), 2 otherwise (less shared memory, more L1 for the copies).
template <typename Tin, int CODE, int MODE, int PRE, int RING>
__global__ void __launch_bounds__(kThreads, PRE ? 3 : kBlocksPerSm)
quantize_kernel(const __grid_constant__ QuantParams prm)
{
    constexpr bool DUAL = MODE == kDual;
    constexpr bool GATED = PRE == 2;
    // Programmatic dependent launch: this kernel may be scheduled while the previous kernel of the stream
    // winds down, and lets the next one be scheduled while its own last blocks run; nothing in global
    // memory is touched before the previous kernel has completed.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const SegBounds &sb = prm.sb;
    const int64_t M = prm.M;
    const int K = prm.K, R = prm.R, lo = prm.lo, hi = prm.hi, row_segments = prm.row_segments;
    const uint32_t g = blockIdx.x * kThreads + threadIdx.x;
    const uint32_t r0 = g / uint32_t(prm.V);
    if (r0 >= uint32_t(R) || int64_t(r0) >= M) return;
    const int k0 = int(g - r0 * uint32_t(prm.V)) * kVec;

    // K-segment of this chunk (bounds come with the kernel parameters)
    int p = 0;
    while (p + 1 < sb.P && k0 >= sb.kb[p + 1]) p++;
    const bool whole = k0 + kVec <= sb.kb[p + 1];            // chunk inside one K-segment (and inside K)
    const int Qs = row_segments ? sb.Q : 1;

    const Tin *src = static_cast<const Tin *>(prm.X) + int64_t(r0) * prm.ld + k0;
    uint8_t *dp = prm.c_pos + int64_t(r0) * prm.ldc + k0;
    uint8_t *dn = DUAL ? prm.c_neg + int64_t(r0) * prm.ldc + k0 : nullptr;
    const int64_t src_step = int64_t(R) * prm.ld, dst_step = int64_t(R) * prm.ldc;

    uint64_t mreg[PRE ? kVec / 2 : 1];                       // this chunk's multipliers, loaded once
    if (PRE) {
#pragma unroll
        for (int i = 0; i < kVec; i += 2)
            mreg[i / 2] = pack2((prm.mult && k0 + i < K) ? __ldg(prm.mult + k0 + i) : 1.0f,
                                (prm.mult && k0 + i + 1 < K) ? __ldg(prm.mult + k0 + i + 1) : 1.0f);
    }

    // The rows of this chunk travel through a thread-private ring in shared memory: asynchronous 16-byte copies
    // (global -> shared without passing through registers) of the next kDepth - 1 rows are in flight while the
    // current row is converted, so the bytes in flight per SM do not cost registers.  Every thread reads only what
    // it copied itself, so a wait on its own copy groups is all the synchronisation there is.
    // (gated, bf16) the chunk of the gate half travels in the same slots, behind the value half's pieces.
    constexpr int NV = int(sizeof(Tin)) * kVec / 16;                        // 16-byte pieces per row chunk
    constexpr bool kGateRing = GATED && sizeof(Tin) == 2;
    constexpr int NS = kGateRing ? 2 * NV : NV;                             // pieces per slot
    // ring slots (32 KiB per block at most; 48 KiB with the gate half)
    constexpr int kDepth = kGateRing ? (RING == 2 ? 2 : 3) : (sizeof(Tin) == 2 || RING == 2) ? RING : RING / 2;
    __shared__ uint4 ring[kDepth * NS * kThreads];
    const uint32_t ring0 = uint32_t(__cvta_generic_to_shared(ring)) + threadIdx.x * 16u;
    auto slot_addr = [&](int slot, int v) { return ring0 + uint32_t((slot * NS + v) * kThreads) * 16u; };
    auto copy_row = [&](const Tin *row_src, int slot, bool valid) {          // one commit group per call, always
        if (valid) {
#pragma unroll
            for (int v = 0; v < NV; v++)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(slot_addr(slot, v)),
                             "l"(reinterpret_cast<const char *>(row_src) + 16 * v) : "memory");
            if (kGateRing) {
#pragma unroll
                for (int v = 0; v < NV; v++)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(slot_addr(slot, NV + v)),
                                 "l"(reinterpret_cast<const char *>(row_src + K) + 16 * v) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto read_row = [&](int slot, Raw16<Tin> &r, int first) {
#pragma unroll
        for (int v = 0; v < NV; v++) {
            uint4 w;
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w)
                         : "r"(slot_addr(slot, first + v)) : "memory");
            set_piece(r, v, w);
        }
    };
    if (whole) {
#pragma unroll
        for (int d = 0; d < kDepth - 1; d++) copy_row(src + int64_t(d) * src_step, d, int64_t(r0) + int64_t(d) * R < M);
    }
    const Tin *gsrc = src + K;                               // (gated) this chunk of the gate half
    Raw16<Tin> gate_next;
    if (GATED && !kGateRing && whole) load16(gsrc, gate_next);
    int q = 0;                                               // N-segment (weights only) the constants belong to
    int64_t q_end = 0;                                       // first row beyond it (0: no constants yet)
    SegConst cp, cn;
    int zp = 0;
    bool fast = false;
    int slot = 0, read_slot = 0;                             // ring slots of the next row and of the current one
    // (dual codes of fp32 behind an activation) the row is read four elements at a time where they are used: with all 16
    // in registers this variant spills (777 x 1040 SiLU 4.1 -> 3.3 us, 8858 x 6144 57.9 -> 53.8; single-scale ones do not
    // spill: 8858 x 6144 with multipliers only 43.2 -> 44.8)
    constexpr bool kByPiece = PRE != 0 && sizeof(Tin) == 4 && DUAL;
    for (int64_t row = r0; row < M; row += R) {
        if (row >= q_end) {                                  // (weights) the row entered another N-segment
            if (row_segments) {
                while (q + 1 < sb.Q && row >= sb.nb[q + 1]) q++;
                q_end = sb.nb[q + 1];
            } else {
                q_end = M;
            }
            cp = seg_const(__ldg(prm.s_pos + p * Qs + (row_segments ? q : 0)));
            cn = seg_const(DUAL ? __ldg(prm.s_neg + p * Qs + (row_segments ? q : 0)) : 1.0f);
            if (MODE == kZeroPoint) zp = __ldg(prm.zp + p);
            fast = whole && cp.fast && cn.fast && !(DUAL && CODE == SQ_CODE_INT8 && lo != -128);
        }
        Raw16<Tin> cur, gate;
        if (GATED && !kGateRing && whole) {
            gate = gate_next;
            if (row + R < M) load16(gsrc + src_step, gate_next);
        }
        if (whole) {
            // row + (kDepth - 1) R goes into the slot the previous row has just left; then the oldest group, this
            // row's, is complete once at most kDepth - 1 newer groups are pending
            const int ahead = slot == 0 ? kDepth - 1 : slot - 1;
            copy_row(src + int64_t(kDepth - 1) * src_step, ahead, row + int64_t(kDepth - 1) * R < M);
            asm volatile("cp.async.wait_group %0;" ::"n"(kDepth - 1) : "memory");
            if (fast && !kByPiece) {
                read_row(slot, cur, 0);
                if (kGateRing) read_row(slot, gate, NV);
            }
            read_slot = slot;
            slot = slot + 1 == kDepth ? 0 : slot + 1;
        }
        if (fast) {
            uint32_t wp[4], wn[4];
            if constexpr (PRE == 0 && DUAL && CODE == SQ_CODE_INT8) bound16(cur);
#pragma unroll
            for (int g4 = 0; g4 < 4; g4++) {
                float x[4];
                if constexpr (kByPiece) {
                    uint4 w;
                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w)
                                 : "r"(slot_addr(read_slot, g4)) : "memory");
                    x[0] = __uint_as_float(w.x); x[1] = __uint_as_float(w.y); x[2] = __uint_as_float(w.z); x[3] = __uint_as_float(w.w);
                } else {
                    get4(cur, g4, x);
                }
                if (GATED) {
                    float gt[4];
                    get4(gate, g4, gt);
#pragma unroll
                    for (int i = 0; i < 4; i += 2)
                        unpack2(pre_gated2<Tin>(x[i], x[i + 1], gt[i], gt[i + 1], mreg[PRE ? 2 * g4 + i / 2 : 0]), x[i], x[i + 1]);
                } else if (PRE) {
#pragma unroll
                    for (int i = 0; i < 4; i += 2)
                        unpack2(pre2<Tin>(x[i], x[i + 1], prm.act, mreg[PRE ? 2 * g4 + i / 2 : 0]), x[i], x[i + 1]);
                }
                quant4<CODE, MODE, PRE == 0 && kBounded<Tin>>(x, cp, cn, float(hi), zp, wp[g4], wn[g4]);
            }
            *reinterpret_cast<uint4 *>(dp) = make_uint4(wp[0], wp[1], wp[2], wp[3]);
            if (DUAL) *reinterpret_cast<uint4 *>(dn) = make_uint4(wn[0], wn[1], wn[2], wn[3]);
        } else {                                 // segment bound or end of row inside the chunk, or an extreme scale
            const int n = min(kVec, K - k0);
            int pp = p;
            const int qq = row_segments ? q : 0;
            for (int i = 0; i < n; i++) {
                while (pp + 1 < sb.P && k0 + i >= sb.kb[pp + 1]) pp++;
                uint32_t a, b;
                float x = load1(src + i);
                if (GATED) x = pre_gated<Tin>(x, load1(gsrc + i), prm.mult ? __ldg(prm.mult + k0 + i) : 1.0f);
                else if (PRE) x = pre1<Tin>(x, prm.act, prm.mult ? __ldg(prm.mult + k0 + i) : 1.0f);
                quant1<CODE, MODE>(x, __ldg(prm.s_pos + pp * Qs + qq), DUAL ? __ldg(prm.s_neg + pp * Qs + qq) : 0.0f,
                                   MODE == kZeroPoint ? __ldg(prm.zp + pp) : 0, lo, hi, a, b);
                dp[i] = uint8_t(a);
                if (DUAL) dn[i] = uint8_t(b);
            }
        }
        src += src_step;
        if (GATED) gsrc += src_step;
        dp += dst_step;
        if (DUAL) dn += dst_step;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");     // nothing of this thread's is in flight when it leaves
}

// ----------------------------------------------------------------------------- small inputs
// A launch of few elements lasts as long as one thread's chain of loads, evaluation and stores: sixteen elements of gated GELU
// are some 700 dependent instructions.  Here a thread has four elements and nothing to walk.  Used while every thread of the
// grid can be resident at once, roughly (few_limit).  us, 16 elements a thread / 4: 8 x 3072 dual int8 1.8 / 1.3, 400 x 2560 2.9 / 2.3, GELU 64 x
// 2048 2.9 / 1.8, gated fp32 24 x 5632 4.2 / 1.6.
constexpr int kFewVec = 4;
__device__ __forceinline__ void load4(const float *p, float (&x)[4])
{
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
}
__device__ __forceinline__ void load4(const __nv_bfloat16 *p, float (&x)[4])
{
    const uint2 v = __ldg(reinterpret_cast<const uint2 *>(p));
    x[0] = __uint_as_float(v.x << 16); x[1] = __uint_as_float(v.x & 0xFFFF0000u);
    x[2] = __uint_as_float(v.y << 16); x[3] = __uint_as_float(v.y & 0xFFFF0000u);
}

template <typename Tin, int CODE, int MODE, int PRE>
__global__ void __launch_bounds__(kThreads)
quantize_few_kernel(const __grid_constant__ QuantParams prm)
{
    constexpr bool DUAL = MODE == kDual, GATED = PRE == 2;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const SegBounds &sb = prm.sb;
    const uint32_t g = blockIdx.x * kThreads + threadIdx.x;
    const uint32_t row = g / uint32_t(prm.V);
    const int k0 = int(g - row * uint32_t(prm.V)) * kFewVec, K = prm.K;
    int p = 0;
    while (p + 1 < sb.P && k0 >= sb.kb[p + 1]) p++;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (int64_t(row) >= prm.M) return;
    const Tin *src = static_cast<const Tin *>(prm.X) + int64_t(row) * prm.ld + k0;
    uint8_t *dp = prm.c_pos + int64_t(row) * prm.ldc + k0;
    uint8_t *dn = DUAL ? prm.c_neg + int64_t(row) * prm.ldc + k0 : nullptr;
    const float sp = __ldg(prm.s_pos + p), sn = DUAL ? __ldg(prm.s_neg + p) : 1.0f;
    if (k0 + kFewVec <= sb.kb[p + 1]) {
        float x[4], gate[4], m[4] = {1.0f, 1.0f, 1.0f, 1.0f};
        load4(src, x);
        if (GATED) load4(src + K, gate);
        if (PRE && prm.mult) {
#pragma unroll
            for (int i = 0; i < 4; i++) m[i] = __ldg(prm.mult + k0 + i);
        }
        const int zp = MODE == kZeroPoint ? __ldg(prm.zp + p) : 0;
        const SegConst cp = seg_const(sp), cn = seg_const(sn);
        if (cp.fast && cn.fast && !(DUAL && CODE == SQ_CODE_INT8 && prm.lo != -128)) {
#pragma unroll
            for (int i = 0; i < 4 && PRE != 0; i += 2) {
                const uint64_t m2 = pack2(m[i], m[i + 1]);
                unpack2(GATED ? pre_gated2<Tin>(x[i], x[i + 1], gate[i], gate[i + 1], m2) : pre2<Tin>(x[i], x[i + 1], prm.act, m2), x[i], x[i + 1]);
            }
            uint32_t wp, wn;
            quant4<CODE, MODE>(x, cp, cn, float(prm.hi), zp, wp, wn);
            *reinterpret_cast<uint32_t *>(dp) = wp;
            if (DUAL) *reinterpret_cast<uint32_t *>(dn) = wn;
            return;
        }
    }
    const int n = min(kFewVec, K - k0);                  // a segment bound or the row's end among the four, or an extreme scale
    for (int i = 0; i < n; i++) {
        while (p + 1 < sb.P && k0 + i >= sb.kb[p + 1]) p++;
        uint32_t a, b;
        float x = load1(src + i);
        if (GATED) x = pre_gated<Tin>(x, load1(src + K + i), prm.mult ? __ldg(prm.mult + k0 + i) : 1.0f);
        else if (PRE) x = pre1<Tin>(x, prm.act, prm.mult ? __ldg(prm.mult + k0 + i) : 1.0f);
        quant1<CODE, MODE>(x, __ldg(prm.s_pos + p), DUAL ? __ldg(prm.s_neg + p) : 0.0f, MODE == kZeroPoint ? __ldg(prm.zp + p) : 0,
                           prm.lo, prm.hi, a, b);
        dp[i] = uint8_t(a);
        if (DUAL) dn[i] = uint8_t(b);
    }
}

// ----------------------------------------------------------------------------- fused SiLU by table (bf16 inputs)
// A bf16 pre-activation has 65536 possible values, so the stored activation bf16(silu(h)) is a table of 128 KiB.
// Every CTA (1024 threads, one per SM) builds the table in its shared memory with the same silu2 as
// the arithmetic variant (a few evaluations per thread: most bit patterns need none), after which an element costs one
// shared-memory load instead of about 30 instructions: the fused pass stops being bound by the ALUs.  Results are
// those of the arithmetic variant bit for bit.  Used for large inputs: a launch of this kernel costs about 9 us
// more than the other's (the table, and a CTA that fills the SM cannot start under the previous kernel's tail).
// The rest is quantize_kernel's scheme: thread g owns column chunk g % V of rows g / V, g / V + R, ...; the rows
// travel through a thread-private ring of kTableDepth slots behind the table.
constexpr int kTableThreads = 1024;
constexpr int kTableDepth = 3;
constexpr size_t kTableBytes = 65536 * 2;
constexpr size_t kTableSmem = kTableBytes + size_t(kTableDepth) * 2 * kTableThreads * 16;      // 224 KiB

template <int CODE, int MODE>
__global__ void __launch_bounds__(kTableThreads, 1)
quantize_silu_table_kernel(const __grid_constant__ QuantParams prm)
{
    constexpr bool DUAL = MODE == kDual;
    extern __shared__ __align__(16) uint8_t table_smem[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t tab0 = uint32_t(__cvta_generic_to_shared(table_smem));
    // Most bit patterns need no evaluation, because silu2 returns a value known in advance there
    // (a warp's 32 consecutive patterns share sign and exponent, so the branch is uniform):
    //   2^-124 <= |h| < 2^-26: h / 2 after the rounding to bf16 (the sigmoid is 1/2 to far below a bf16 half-step);
    //   h >= 32: h itself (exp(-h) is below fp32's resolution of 1);  h <= -128: -0 (the exponential has underflowed to zero).
    // NaN and infinities go through the function.  A test compares the codes of this variant with those of the arithmetic
    // one on all 65536 patterns (the sign of a zero does not show in a code).
    for (uint32_t b = threadIdx.x; b < 65536u; b += kTableThreads) {
        const uint32_t e = (b >> 7) & 0xFFu, neg = b >> 15;
        uint32_t out;
        if (e >= 3u && e <= 100u) {
            out = b - 0x80u;                                  // exponent - 1
        } else if (e != 255u && !neg && e >= 132u) {
            out = b;
        } else if (e != 255u && neg && e >= 134u) {
            out = 0x8000u;
        } else {
            const float h = __uint_as_float(b << 16);
            float a, a_same;
            unpack2(silu2(h, h), a, a_same);
            const __nv_bfloat16 r = __float2bfloat16_rn(a);
            out = *reinterpret_cast<const unsigned short *>(&r);
        }
        reinterpret_cast<unsigned short *>(table_smem)[b] = static_cast<unsigned short>(out);
    }
    // the table depends on nothing in memory: it is built before the wait for the previous kernel of the stream
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
    auto lookup = [&](uint32_t bits16) -> float {       // bits of a bf16 pre-activation -> stored activation as fp32
        uint32_t v;
        asm volatile("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(tab0 + (bits16 << 1)));
        return __uint_as_float(v << 16);
    };

    const SegBounds &sb = prm.sb;
    const int64_t M = prm.M;
    const int R = prm.R;
    const uint32_t g = blockIdx.x * kTableThreads + threadIdx.x;
    const uint32_t r0 = g / uint32_t(prm.V);
    if (r0 >= uint32_t(R) || int64_t(r0) >= M) return;
    const int k0 = int(g - r0 * uint32_t(prm.V)) * kVec;     // the host checked: every chunk lies in one K-segment
    int p = 0;
    while (p + 1 < sb.P && k0 >= sb.kb[p + 1]) p++;

    using Tin = __nv_bfloat16;
    const Tin *src = static_cast<const Tin *>(prm.X) + int64_t(r0) * prm.ld + k0;
    uint8_t *dp = prm.c_pos + int64_t(r0) * prm.ldc + k0;
    uint8_t *dn = DUAL ? prm.c_neg + int64_t(r0) * prm.ldc + k0 : nullptr;
    const int64_t src_step = int64_t(R) * prm.ld, dst_step = int64_t(R) * prm.ldc;
    float mreg[kVec];
#pragma unroll
    for (int i = 0; i < kVec; i++) mreg[i] = prm.mult ? __ldg(prm.mult + k0 + i) : 1.0f;
    const SegConst cp = seg_const(__ldg(prm.s_pos + p));
    const SegConst cn = seg_const(DUAL ? __ldg(prm.s_neg + p) : 1.0f);
    const bool fast = cp.fast && cn.fast && !(DUAL && CODE == SQ_CODE_INT8 && prm.lo != -128);

    const uint32_t ring0 = tab0 + uint32_t(kTableBytes) + threadIdx.x * 16u;
    auto slot_addr = [&](int slot, int v) { return ring0 + uint32_t((slot * 2 + v) * kTableThreads) * 16u; };
    auto copy_row = [&](const Tin *row_src, int slot, bool valid) {          // one commit group per call, always
        if (valid) {
#pragma unroll
            for (int v = 0; v < 2; v++)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(slot_addr(slot, v)),
                             "l"(reinterpret_cast<const char *>(row_src) + 16 * v) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int d = 0; d < kTableDepth - 1; d++) copy_row(src + int64_t(d) * src_step, d, int64_t(r0) + int64_t(d) * R < M);
    int slot = 0;
    for (int64_t row = r0; row < M; row += R) {
        const int ahead = slot == 0 ? kTableDepth - 1 : slot - 1;
        copy_row(src + int64_t(kTableDepth - 1) * src_step, ahead, row + int64_t(kTableDepth - 1) * R < M);
        asm volatile("cp.async.wait_group %0;" ::"n"(kTableDepth - 1) : "memory");
        uint32_t w[8];
#pragma unroll
        for (int v = 0; v < 2; v++)
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w[4 * v]), "=r"(w[4 * v + 1]), "=r"(w[4 * v + 2]), "=r"(w[4 * v + 3])
                         : "r"(slot_addr(slot, v)) : "memory");
        slot = slot + 1 == kTableDepth ? 0 : slot + 1;
        uint32_t wp[4], wn[4];
#pragma unroll
        for (int g4 = 0; g4 < 4; g4++) {
            float x[4];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const uint32_t word = w[2 * g4 + (i >> 1)];
                x[i] = __fmul_rn(lookup((i & 1) ? (word >> 16) : (word & 0xFFFFu)), mreg[4 * g4 + i]);
            }
            if (fast) {
                quant4<CODE, MODE>(x, cp, cn, float(prm.hi), 0, wp[g4], wn[g4]);
            } else {
                wp[g4] = wn[g4] = 0u;
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    uint32_t a, b;
                    quant1<CODE, MODE>(x[i], cp.s, cn.s, 0, prm.lo, prm.hi, a, b);
                    wp[g4] |= (a & 0xFFu) << (8 * i);
                    wn[g4] |= (b & 0xFFu) << (8 * i);
                }
            }
        }
        *reinterpret_cast<uint4 *>(dp) = make_uint4(wp[0], wp[1], wp[2], wp[3]);
        if (DUAL) *reinterpret_cast<uint4 *>(dn) = make_uint4(wn[0], wn[1], wn[2], wn[3]);
        src += src_step;
        dp += dst_step;
        if (DUAL) dn += dst_step;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// ----------------------------------------------------------------------------- GELU by a table of its tail (bf16 inputs)
// GELU(h) = max(h, 0) - (a / 2) E(a) with a = |h|, E = erfc(a / sqrt 2), in one FMA (gelu_from_tail2).  Of a bf16 value a the tail needs
// few: below 2^-26 E does not change any more (t + 2.5 and t - 2.5 have rounded to the same values since 2^-23), from 16 on it
// is zero, and between them lie 30 binades of 128 values.  A table of E as fp32, 15 KiB, built by every block in its shared memory
// with the same instructions, so leaves about ten instructions of thirty, with the bits of the arithmetic variant, and serves
// the gated form too, whose product is rounded once, from the unrounded GELU.  One block of 1024 threads per SM: the table is
// built once per SM (about four entries a thread), ahead of the dependency wait.  Rows travel as in quantize_kernel.
// Bound by the load unit: 16 scattered loads a chunk, on average three and a half of a warp's in one bank, while instructions issue in
// 59 % (gated) and 70 % of the cycles.  us, evaluated per element / by a table of all 65536 stored values, which this replaces / here,
// dual int8: GELU 8858 x 6144 80.0 / 47.3 / 45.8, 8192 x 2560 32.5 / 23.9 / 21.0, 1024 x 2560 7.4 / 9.0 / 6.2; gated 8858 x 6144
// 90.3 / - / 64.1, 8192 x 2560 37.8 / - / 29.7.
constexpr uint32_t kTailLo = 101u << 7, kTailHi = 0x4180u;            // bf16 patterns of 2^-26 and 16
constexpr int kTailEntries = int(kTailHi - kTailLo) + 1;
constexpr size_t kTailBytes = (size_t(kTailEntries) * 4 + 127) / 128 * 128;
__host__ __device__ constexpr int tail_depth(bool gated) { return gated ? 3 : 4; }
__host__ __device__ constexpr size_t tail_smem(bool gated) { return size_t(tail_depth(gated)) * (gated ? 4 : 2) * kTableThreads * 16; }

template <int CODE, int MODE, bool GATED, bool MULT>
__global__ void __launch_bounds__(kTableThreads, 1)
quantize_tail_kernel(const __grid_constant__ QuantParams prm)
{
    constexpr bool DUAL = MODE == kDual;
    __shared__ __align__(16) float table[kTailBytes / 4];                // (static: its address is part of the load instructions)
    extern __shared__ __align__(16) uint8_t tail_ring[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int i = 2 * int(threadIdx.x); i < kTailEntries; i += 2 * kTableThreads) {
        const uint32_t b = kTailLo + uint32_t(i);
        float e0, e1;
        unpack2(gelu_tail2(pack2(__uint_as_float(b << 16), __uint_as_float(min(b + 1, kTailHi) << 16))), e0, e1);
        *reinterpret_cast<float2 *>(table + i) = make_float2(e0, e1);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();

    const SegBounds &sb = prm.sb;
    const int64_t M = prm.M;
    const int R = prm.R;
    const uint32_t g = blockIdx.x * kTableThreads + threadIdx.x;
    const uint32_t r0 = g / uint32_t(prm.V);
    if (r0 >= uint32_t(R) || int64_t(r0) >= M) return;
    const int k0 = int(g - r0 * uint32_t(prm.V)) * kVec;                 // the host checked: every chunk lies in one K-segment
    int p = 0;
    while (p + 1 < sb.P && k0 >= sb.kb[p + 1]) p++;

    using Tin = __nv_bfloat16;
    const Tin *src = static_cast<const Tin *>(prm.X) + int64_t(r0) * prm.ld + k0;
    uint8_t *dp = prm.c_pos + int64_t(r0) * prm.ldc + k0;
    uint8_t *dn = DUAL ? prm.c_neg + int64_t(r0) * prm.ldc + k0 : nullptr;
    const int64_t src_step = int64_t(R) * prm.ld, dst_step = int64_t(R) * prm.ldc;
    uint64_t mreg[MULT ? kVec / 2 : 1];
    if (MULT) {
#pragma unroll
        for (int i = 0; i < kVec; i += 2) mreg[i / 2] = pack2(__ldg(prm.mult + k0 + i), __ldg(prm.mult + k0 + i + 1));
    }
    const SegConst cp = seg_const(__ldg(prm.s_pos + p));
    const SegConst cn = seg_const(DUAL ? __ldg(prm.s_neg + p) : 1.0f);
    const bool fast = cp.fast && cn.fast && !(DUAL && CODE == SQ_CODE_INT8 && prm.lo != -128);

    constexpr int NS = GATED ? 4 : 2, kDepth = tail_depth(GATED);        // 16-byte pieces per slot, value half first
    const uint32_t ring0 = uint32_t(__cvta_generic_to_shared(tail_ring)) + threadIdx.x * 16u;
    auto slot_addr = [&](int slot, int v) { return ring0 + uint32_t((slot * NS + v) * kTableThreads) * 16u; };
    auto copy_row = [&](const Tin *row_src, int slot, bool valid) {          // one commit group per call, always
        if (valid) {
#pragma unroll
            for (int v = 0; v < NS; v++)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(slot_addr(slot, v)),
                             "l"(reinterpret_cast<const char *>(v < 2 ? row_src : row_src + prm.K) + 16 * (v & 1)) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto read_piece = [&](int slot, int v, uint32_t (&w)[4]) {
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                     : "r"(slot_addr(slot, v)) : "memory");
    };
    auto tail = [&](uint32_t byte_offset) -> float {
        return *reinterpret_cast<const float *>(reinterpret_cast<const uint8_t *>(table) + byte_offset);
    };
#pragma unroll
    for (int d = 0; d < kDepth - 1; d++) copy_row(src + int64_t(d) * src_step, d, int64_t(r0) + int64_t(d) * R < M);
    int slot = 0;
    for (int64_t row = r0; row < M; row += R) {
        const int ahead = slot == 0 ? kDepth - 1 : slot - 1;
        copy_row(src + int64_t(kDepth - 1) * src_step, ahead, row + int64_t(kDepth - 1) * R < M);
        asm volatile("cp.async.wait_group %0;" ::"n"(kDepth - 1) : "memory");
        uint32_t wp[4], wn[4];
#pragma unroll
        for (int half = 0; half < 2; half++) {
            uint32_t w[4], wg[4];
            read_piece(slot, half, w);
            if (GATED) read_piece(slot, 2 + half, wg);
#pragma unroll
            for (int q = 0; q < 2; q++) {                                // four elements
                const int g4 = 2 * half + q;
                float x[4];
#pragma unroll
                for (int i = 0; i < 2; i++) {
                    const uint32_t h = GATED ? wg[2 * q + i] : w[2 * q + i];
                    const uint32_t a = __vminu2(h & 0x7FFF7FFFu, kTailHi * 0x10001u), at = __vmaxu2(a, kTailLo * 0x10001u);
                    const uint32_t off = (at - kTailLo * 0x10001u) << 2;         // byte offsets of both entries, 14 bits each
                    const uint64_t E = pack2(tail(off & 0xFFFFu), tail(off >> 16));
                    uint64_t v = gelu_from_tail2(__uint_as_float(h << 16), __uint_as_float(h & 0xFFFF0000u),
                                                 pack2(__uint_as_float(a << 16), __uint_as_float(a & 0xFFFF0000u)), E);
                    if (GATED) v = mul2(pack2(__uint_as_float(w[2 * q + i] << 16), __uint_as_float(w[2 * q + i] & 0xFFFF0000u)), v);
                    v = rounded2<Tin>(v);
                    if (MULT) v = mul2(v, mreg[MULT ? 2 * g4 + i : 0]);
                    unpack2(v, x[2 * i], x[2 * i + 1]);
                }
                if (fast) {
                    quant4<CODE, MODE>(x, cp, cn, float(prm.hi), 0, wp[g4], wn[g4]);
                } else {
                    wp[g4] = wn[g4] = 0u;
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        uint32_t a, b;
                        quant1<CODE, MODE>(x[i], cp.s, cn.s, 0, prm.lo, prm.hi, a, b);
                        wp[g4] |= (a & 0xFFu) << (8 * i);
                        wn[g4] |= (b & 0xFFu) << (8 * i);
                    }
                }
            }
        }
        slot = slot + 1 == kDepth ? 0 : slot + 1;
        *reinterpret_cast<uint4 *>(dp) = make_uint4(wp[0], wp[1], wp[2], wp[3]);
        if (DUAL) *reinterpret_cast<uint4 *>(dn) = make_uint4(wn[0], wn[1], wn[2], wn[3]);
        src += src_step;
        dp += dst_step;
        if (DUAL) dn += dst_step;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// ----------------------------------------------------------------------------- per-row scales (W4A8)
// App. B "Extra Hyperparameter Settings": 4-bit weights are quantized per channel, activations dynamically per
// token.  One CTA per row: the row is read once into registers (up to kRowChunks 16-element chunks per thread),
// its extrema per K-segment are reduced in shared memory, the scales (one IEEE division each) are written out,
// and the codes are made from the registers with the same quantizer as everywhere else.
constexpr int kRowChunks = 4;                       // K <= 256 threads x 4 chunks x 16 = 16384
// CHUNKS: chunks a thread may hold.  One where a block of 256 threads covers the row with one per thread (K <= 4096): fewer
// registers, more rows in flight (us, 4 / 1 chunks: 921 x 1920 dual with 12 segments 8.1 / 4.4, 8858 x 1536 with 24
// 16.4 / 13.9, 8858 x 3072 with 2 21.6 / 20.1).  Two up to K = 8192 were no better on many rows (8858 x 6144 42.8 / 44.5);
// one per thread on larger blocks has not been measured.  Exception, see per_row_chunks: many long rows of one K-segment.

__device__ __forceinline__ uint32_t ord_enc(float f)     // monotone map float -> uint32
{
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord_dec(uint32_t u)
{
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}

// largest and smallest of the 16 elements of a chunk (bf16: on packed pairs, two elements per instruction)
__device__ __forceinline__ void chunk_extrema(const Raw16<float> &r, float &mx, float &mn)
{
    mx = -INFINITY; mn = INFINITY;
#pragma unroll
    for (int v = 0; v < 4; v++) {
        mx = fmaxf(fmaxf(mx, r.v[v].x), fmaxf(r.v[v].y, fmaxf(r.v[v].z, r.v[v].w)));
        mn = fminf(fminf(mn, r.v[v].x), fminf(r.v[v].y, fminf(r.v[v].z, r.v[v].w)));
    }
}
__device__ __forceinline__ void chunk_extrema(const Raw16<__nv_bfloat16> &r, float &mx, float &mn)
{
    const uint32_t w[8] = {r.v[0].x, r.v[0].y, r.v[0].z, r.v[0].w, r.v[1].x, r.v[1].y, r.v[1].z, r.v[1].w};
    __nv_bfloat162 hi = *reinterpret_cast<const __nv_bfloat162 *>(&w[0]), lo = hi;
#pragma unroll
    for (int i = 1; i < 8; i++) {
        const __nv_bfloat162 x = *reinterpret_cast<const __nv_bfloat162 *>(&w[i]);
        hi = __hmax2(hi, x);
        lo = __hmin2(lo, x);
    }
    mx = fmaxf(__low2float(hi), __high2float(hi));
    mn = fminf(__low2float(lo), __high2float(lo));
}

template <typename Tin, bool DUAL, int CHUNKS>
__global__ void __launch_bounds__(kThreads, CHUNKS == 1 && DUAL ? 6 : 0)       // (dual: with the 32 registers it takes by itself 1111 x 1072 goes from 3.3 to 4.6 us)
quantize_per_row_kernel(const Tin *__restrict__ X, int K, int64_t ld, const SegBounds sb, float q_max, float q_min_abs,
                        float *__restrict__ s_pos, float *__restrict__ s_neg, uint8_t *__restrict__ c_pos,
                        uint8_t *__restrict__ c_neg, int64_t ldc)
{
    __shared__ uint32_t sh_max[SQ_MAX_P], sh_min[SQ_MAX_P];
    __shared__ float sh_sp[SQ_MAX_P], sh_sn[SQ_MAX_P];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int64_t row = blockIdx.x;
    const int P = sb.P;
    // One K-segment (the usual case) needs ONE block barrier: every warp leaves its extrema in a slot, and after the
    // barrier every thread reduces the slots and computes the scales itself.  Several K-segments go through
    // shared-memory words per segment (three barriers).
    const bool one = P == 1;
    __shared__ float sh_wmax[kThreads / 32], sh_wmin[kThreads / 32];
    float one_sp = 1.0f, one_sn = 1.0f, tail_mx = -INFINITY, tail_mn = INFINITY;
    if (!one) {
        for (int i = threadIdx.x; i < P; i += blockDim.x) { sh_max[i] = 0u; sh_min[i] = 0xFFFFFFFFu; }
        __syncthreads();
    }
    const Tin *src = X + row * ld;
    Raw16<Tin> raw[CHUNKS];
    int seg[CHUNKS];                            // K-segment of a whole chunk, -1: straddles a bound or the row end
#pragma unroll
    for (int c = 0; c < CHUNKS; c++) {
        const int k0 = (int(threadIdx.x) + c * int(blockDim.x)) * kVec;
        seg[c] = -2;                                // beyond the row
        if (k0 >= K) continue;
        int p = 0;
        while (p + 1 < P && k0 >= sb.kb[p + 1]) p++;
        if (k0 + kVec <= sb.kb[p + 1]) {
            seg[c] = p;
            load16(src + k0, raw[c]);
        } else {
            seg[c] = -1;
            const int n = min(kVec, K - k0);
            for (int i = 0; i < n; i++) {
                while (p + 1 < P && k0 + i >= sb.kb[p + 1]) p++;
                const float x = load1(src + k0 + i);
                if (one) {
                    tail_mx = fmaxf(tail_mx, x);
                    tail_mn = fminf(tail_mn, x);
                } else {
                    atomicMax(&sh_max[p], ord_enc(x));
                    atomicMin(&sh_min[p], ord_enc(x));
                }
            }
        }
    }
    if (one) {
        float mx = tail_mx, mn = tail_mn;
#pragma unroll
        for (int c = 0; c < CHUNKS; c++) {
            if (seg[c] >= 0) {
                float cx, cm;
                chunk_extrema(raw[c], cx, cm);
                mx = fmaxf(mx, cx);
                mn = fminf(mn, cm);
            }
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) {
            mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
            mn = fminf(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, o));
        }
        if ((threadIdx.x & 31) == 0) { sh_wmax[threadIdx.x >> 5] = mx; sh_wmin[threadIdx.x >> 5] = mn; }
        __syncthreads();
        mx = sh_wmax[0]; mn = sh_wmin[0];
        for (int w = 1; w < int(blockDim.x >> 5); w++) { mx = fmaxf(mx, sh_wmax[w]); mn = fminf(mn, sh_wmin[w]); }
        if (DUAL) {
            const float h = fmaxf(mx, 0.0f), l = fmaxf(-mn, 0.0f);
            one_sp = h > 0.0f ? __fdiv_rn(h, q_max) : 1.0f;
            one_sn = l > 0.0f ? __fdiv_rn(l, q_min_abs) : 1.0f;
            if (threadIdx.x == 0) s_neg[row] = one_sn;
        } else {
            const float a = fmaxf(fabsf(mx), fabsf(mn));
            one_sp = a > 0.0f ? __fdiv_rn(a, q_max) : 1.0f;
        }
        if (threadIdx.x == 0) s_pos[row] = one_sp;
    } else {
    // Extrema: where the 32 chunks of a warp lie in one K-segment (512 consecutive columns: the usual case) they are
    // reduced with shuffles and one lane updates the shared words; same-address shared atomics from every thread
    // serialise, and were most of this kernel's time.  Every lane takes part in the votes and shuffles.
#pragma unroll
    for (int c = 0; c < CHUNKS; c++) {
        float mx = -INFINITY, mn = INFINITY;
        if (seg[c] >= 0) chunk_extrema(raw[c], mx, mn);
        const int s0 = __shfl_sync(0xFFFFFFFFu, seg[c], 0);
        const bool uniform = __all_sync(0xFFFFFFFFu, seg[c] == s0) && s0 >= 0;
        if (uniform) {
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
                mn = fminf(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, o));
            }
            if ((threadIdx.x & 31) == 0) {
                atomicMax(&sh_max[s0], ord_enc(mx));
                atomicMin(&sh_min[s0], ord_enc(mn));
            }
        } else if (seg[c] >= 0) {
            atomicMax(&sh_max[seg[c]], ord_enc(mx));
            atomicMin(&sh_min[seg[c]], ord_enc(mn));
        }
    }
    __syncthreads();
    for (int p = threadIdx.x; p < P; p += blockDim.x) {
        const float mx = ord_dec(sh_max[p]), mn = ord_dec(sh_min[p]);
        float sp, sn = 1.0f;
        if (DUAL) {
            const float hi = fmaxf(mx, 0.0f), lo = fmaxf(-mn, 0.0f);
            sp = hi > 0.0f ? __fdiv_rn(hi, q_max) : 1.0f;
            sn = lo > 0.0f ? __fdiv_rn(lo, q_min_abs) : 1.0f;
            s_neg[row * P + p] = sn;
        } else {
            const float a = fmaxf(fabsf(mx), fabsf(mn));
            sp = a > 0.0f ? __fdiv_rn(a, q_max) : 1.0f;
        }
        s_pos[row * P + p] = sp;
        sh_sp[p] = sp;
        sh_sn[p] = sn;
    }
    __syncthreads();
    }
    const int hi = int(q_max), lo = DUAL ? -int(q_min_abs) : -int(q_max);
    constexpr int MODE = DUAL ? kDual : kSingle;
    SegConst cp, cn;
    int const_seg = -1;
#pragma unroll
    for (int c = 0; c < CHUNKS; c++) {
        const int k0 = (int(threadIdx.x) + c * int(blockDim.x)) * kVec;
        if (seg[c] == -2) continue;
        uint8_t *dp = c_pos + row * ldc + k0;
        uint8_t *dn = DUAL ? c_neg + row * ldc + k0 : nullptr;
        bool done = false;
        if (seg[c] >= 0) {
            if (seg[c] != const_seg) {              // constants are remade only when the chunk's K-segment changes
                cp = seg_const(one ? one_sp : sh_sp[seg[c]]);
                cn = seg_const(DUAL ? (one ? one_sn : sh_sn[seg[c]]) : 1.0f);
                const_seg = seg[c];
            }
            if (cp.fast && cn.fast && !(DUAL && lo != -128)) {
                uint32_t wp[4], wn[4];
#pragma unroll
                for (int g4 = 0; g4 < 4; g4++) {
                    float x[4];
                    get4(raw[c], g4, x);
                    quant4<SQ_CODE_INT8, MODE, true>(x, cp, cn, float(hi), 0, wp[g4], wn[g4]);
                }
                *reinterpret_cast<uint4 *>(dp) = make_uint4(wp[0], wp[1], wp[2], wp[3]);
                if (DUAL) *reinterpret_cast<uint4 *>(dn) = make_uint4(wn[0], wn[1], wn[2], wn[3]);
                done = true;
            }
        }
        if (!done) {
            const int n = min(kVec, K - k0);
            int p = 0;
            for (int i = 0; i < n; i++) {
                while (p + 1 < P && k0 + i >= sb.kb[p + 1]) p++;
                uint32_t a, b;
                quant1<SQ_CODE_INT8, MODE>(load1(src + k0 + i), one ? one_sp : sh_sp[p], one ? one_sn : sh_sn[p], 0, lo, hi, a, b);
                dp[i] = uint8_t(a);
                if (DUAL) dn[i] = uint8_t(b);
            }
        }
    }
}

// int8 codes in [-8, 7] <-> two 4-bit codes per byte (code 2j in the low nibble); 16 codes to a chunk.  A small kernel between
// two others on every W4A8 call: launched like them, so that its start and theirs overlap the kernel in front (2048 x 4608 ->
// 1152 whole layer 32.8 -> 30.4 us).  Bound by memory: a thread takes up to kPackChunks chunks a grid apart, their loads in flight
// together, and 32-bit divisions where 32 bits count the chunks.  (unpack, us, one chunk a thread and 64-bit divisions / now: 16072 x
// 10400, 250 MB, 49.9 / 39.9 = 6.3 TB/s; 5552 x 3584 7.4 / 6.2; 504 x 6688 2.1 / 1.9.)
constexpr int kPackChunks = 4;
template <typename Index, bool UNPACK, int CHUNKS>
__global__ void __launch_bounds__(kThreads)
pack_w4_kernel(uint8_t *__restrict__ w8, int64_t ld8, Index total, uint32_t V, uint8_t *__restrict__ w4, int64_t ld4)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const Index first = Index(blockIdx.x) * kThreads + threadIdx.x, step = Index(gridDim.x) * kThreads;
    uint8_t *p8[CHUNKS], *p4[CHUNKS];
    uint4 v8[CHUNKS];
    uint2 v4[CHUNKS];
#pragma unroll
    for (int c = 0; c < CHUNKS; c++) {
        const Index idx = first + Index(c) * step, n = idx / Index(V);
        const int64_t k0 = int64_t(idx - n * Index(V)) * kVec;
        p8[c] = w8 + int64_t(n) * ld8 + k0;
        p4[c] = w4 + int64_t(n) * ld4 + k0 / 2;
        if (idx < total) {
            if (UNPACK) v4[c] = *reinterpret_cast<const uint2 *>(p4[c]);
            else v8[c] = *reinterpret_cast<const uint4 *>(p8[c]);
        }
    }
#pragma unroll
    for (int c = 0; c < CHUNKS; c++) {
        if (first + Index(c) * step >= total) break;
        if (!UNPACK) {
            const uint32_t w[4] = {v8[c].x, v8[c].y, v8[c].z, v8[c].w};
            uint32_t o[2];
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const uint32_t a = w[2 * h], b = w[2 * h + 1];          // 4 codes each
                const uint32_t pa = (a & 0xF) | ((a >> 4) & 0xF0) | ((a >> 8) & 0xF00) | ((a >> 12) & 0xF000);
                const uint32_t pb = (b & 0xF) | ((b >> 4) & 0xF0) | ((b >> 8) & 0xF00) | ((b >> 12) & 0xF000);
                o[h] = pa | (pb << 16);
            }
            *reinterpret_cast<uint2 *>(p4[c]) = make_uint2(o[0], o[1]);
        } else {
            const uint32_t in[2] = {v4[c].x, v4[c].y};
            uint32_t o[4];
#pragma unroll
            for (int h = 0; h < 2; h++) {
#pragma unroll
                for (int t = 0; t < 2; t++) {
                    const uint32_t hw = (in[h] >> (16 * t)) & 0xFFFFu;   // 4 nibbles
                    uint32_t bytes = (hw & 0xF) | ((hw & 0xF0) << 4) | ((hw & 0xF00) << 8) | ((hw & 0xF000) << 12);
                    bytes |= (bytes & 0x08080808u) * 0x1Eu;              // sign-extend each nibble: bit 3 copied into bits 4..7
                    o[2 * h + t] = bytes;
                }
            }
            *reinterpret_cast<uint4 *>(p8[c]) = make_uint4(o[0], o[1], o[2], o[3]);
        }
    }
}

std::atomic<int> g_table_mode{0};        // test hook: 0 automatic, 1 a table wherever possible, 2 never
// Threads of four elements per SM up to which quantize_few_kernel is the faster one: about as many as an SM holds, more where
// sixteen elements a thread cost most (us, 16 / 4 elements, dual int8, Mi elements: plain bf16 0.98 2.87 / 2.29, 1.25 3.0 / 3.1; fp32 1.56
// 4.1 / 3.7, 2.44 4.6 / 4.8; SiLU bf16 1.25 3.9 / 3.8, 1.56 3.9 / 4.1; fp32 SiLU 2.44 6.1 / 5.9, GELU 2.44 7.5 / 6.8, 4.39 9.7 / 10.5; gated bf16 2.44
// 8.3 / 7.2, 4.39 10.7 / 11.2; gated fp32 4.39 16.0 / 11.1, 40 91.3 / 86.2: up to any ordinary size).
int64_t few_limit(bool f32, int act, bool pre)
{
    if (act == SQ_ACT_GEGLU) return f32 ? 1 << 20 : 4400;
    return f32 ? (pre ? 4400 : 2800) : (pre ? 2048 : 1800);
}

template <typename Tin, int CODE, int MODE>
sq_status prepare_t(QuantLaunch &L)
{
    // V chunks per row; R rows in flight: every SM gets all the blocks it can hold, and a thread walks M / R rows, some
    // one more than others.  (Cutting R down so that all walk the same number left SMs with two blocks beside SMs with
    // three: 8192 x 2560 gated 36.0 -> 35.0 us, 8858 x 3072 bf16 17.1 -> 15.5 us.)
    QuantParams &prm = L.prm;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        return SQ_ERR_CUDA;
    const bool pre = prm.act != 0 || prm.mult != nullptr;
    if (!prm.row_segments) {
        const int64_t V4 = (prm.K + kFewVec - 1) / kFewVec;
        if (prm.M * V4 <= few_limit(sizeof(Tin) == 4, prm.act, pre) * sms) {
            prm.V = int(V4);
            L.blocks = unsigned((prm.M * V4 + kThreads - 1) / kThreads);
            L.kernel = prm.act == SQ_ACT_GEGLU ? reinterpret_cast<const void *>(quantize_few_kernel<Tin, CODE, MODE, 2>)
                       : pre                   ? reinterpret_cast<const void *>(quantize_few_kernel<Tin, CODE, MODE, 1>)
                                               : reinterpret_cast<const void *>(quantize_few_kernel<Tin, CODE, MODE, 0>);
            return SQ_OK;
        }
    }
    const int64_t V = (prm.K + kVec - 1) / kVec;
    const int64_t target_threads = int64_t(sms) * kThreads * (pre ? 3 : kBlocksPerSm);
    int64_t iters = (prm.M * V + target_threads - 1) / target_threads;
    if (iters < 1) iters = 1;
    const int64_t R = std::min<int64_t>(prm.M, std::max<int64_t>(1, target_threads / V));
    const int64_t blocks = (R * V + kThreads - 1) / kThreads;
    if (blocks > 0x7FFFFFFF || R * V > 0xFFFFFFFFll || V > 0x7FFFFFFF || R > 0x7FFFFFFF) return SQ_ERR_SHAPE;
    prm.V = int(V);
    prm.R = int(R);
    L.blocks = unsigned(blocks);
    // fp32 input: 64-byte chunks, so half the depth for the same shared memory
    const bool deep = iters >= 10 && sizeof(Tin) == 2;
    if (prm.act == SQ_ACT_GEGLU)
        L.kernel = deep ? reinterpret_cast<const void *>(quantize_kernel<Tin, CODE, MODE, 2, 4>)
                        : reinterpret_cast<const void *>(quantize_kernel<Tin, CODE, MODE, 2, 2>);
    else if (pre)
        L.kernel = reinterpret_cast<const void *>(quantize_kernel<Tin, CODE, MODE, 1, 2>);
    else
        L.kernel = deep ? reinterpret_cast<const void *>(quantize_kernel<Tin, CODE, MODE, 0, 4>)
                        : reinterpret_cast<const void *>(quantize_kernel<Tin, CODE, MODE, 0, 2>);
    return SQ_OK;
}

template <typename Tin>
sq_status prepare_mode(QuantLaunch &L, sq_code code, int mode)
{
    if (mode == kZeroPoint) return prepare_t<Tin, SQ_CODE_INT8, kZeroPoint>(L);
    if (code == SQ_CODE_INT8)
        return mode == kDual ? prepare_t<Tin, SQ_CODE_INT8, kDual>(L) : prepare_t<Tin, SQ_CODE_INT8, kSingle>(L);
    return mode == kDual ? prepare_t<Tin, SQ_CODE_E4M3, kDual>(L) : prepare_t<Tin, SQ_CODE_E4M3, kSingle>(L);
}

// The table variants of the fused activation: bf16 input, every 16-element chunk inside one K-segment, and enough elements for
// the table's set-up time not to count.  prepare_table returns false where they do not apply.
// measured break-even points (us, evaluated per element, few or many elements a thread, against table): SiLU dual 18 Mi 21.6 / 22.1, 20 Mi 23.8 / 23.5, 24 Mi
// 28.0 / 26.8, single 20 Mi 19.6 / 21.8, 24 Mi 23.3 / 24.7 (0.9 / 0.7 us per further Mi); GELU dual 0.98 Mi 3.4 / 4.1, 1.25 Mi
// 4.3 / 4.4, 2.44 Mi 6.7 / 6.1, single 1.25 Mi 3.4 / 3.5; gated GELU dual 5 Mi 11.2 / 12.7, 10 Mi 19.5 / 19.2, single 10 Mi 16.9 / 17.3,
// 20 Mi 31.1 / 26.8.
int64_t table_min(int act, bool dual)
{
    if (act == SQ_ACT_SILU) return int64_t(dual ? 20 : 30) << 20;
    return act == SQ_ACT_GELU ? int64_t(5) << 18 : int64_t(dual ? 10 : 12) << 20;
}
template <bool MULT>
const void *tail_kernel(sq_code code, int mode, bool gated)
{
    auto pick = [&](auto k_int8_dual, auto k_int8, auto k_e4m3_dual, auto k_e4m3) {
        return reinterpret_cast<const void *>(code == SQ_CODE_INT8 ? (mode == kDual ? k_int8_dual : k_int8) : (mode == kDual ? k_e4m3_dual : k_e4m3));
    };
    return gated ? pick(quantize_tail_kernel<SQ_CODE_INT8, kDual, true, MULT>, quantize_tail_kernel<SQ_CODE_INT8, kSingle, true, MULT>,
                        quantize_tail_kernel<SQ_CODE_E4M3, kDual, true, MULT>, quantize_tail_kernel<SQ_CODE_E4M3, kSingle, true, MULT>)
                 : pick(quantize_tail_kernel<SQ_CODE_INT8, kDual, false, MULT>, quantize_tail_kernel<SQ_CODE_INT8, kSingle, false, MULT>,
                        quantize_tail_kernel<SQ_CODE_E4M3, kDual, false, MULT>, quantize_tail_kernel<SQ_CODE_E4M3, kSingle, false, MULT>);
}
bool prepare_table(QuantLaunch &L, sq_dtype dt, sq_code code, int mode)
{
    QuantParams &prm = L.prm;
    const int tm = g_table_mode.load(std::memory_order_relaxed);
    if (tm == 2 || dt != SQ_BF16 || mode == kZeroPoint || prm.row_segments) return false;
    if (prm.act != SQ_ACT_SILU && prm.act != SQ_ACT_GELU && prm.act != SQ_ACT_GEGLU) return false;
    const bool silu = prm.act == SQ_ACT_SILU, gated = prm.act == SQ_ACT_GEGLU;
    if (prm.K % kVec != 0) return false;
    for (int p = 1; p < prm.sb.P; p++)
        if (prm.sb.kb[p] % kVec != 0) return false;
    if (tm != 1 && prm.M * int64_t(prm.K) < table_min(prm.act, mode == kDual)) return false;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        return false;
    const int64_t V = prm.K / kVec;
    const int64_t threads = int64_t(sms) * kTableThreads;                 // one CTA per SM
    int64_t iters = (prm.M * V + threads - 1) / threads;
    if (iters < 1) iters = 1;
    const int64_t R = silu ? (prm.M + iters - 1) / iters : std::min<int64_t>(prm.M, std::max<int64_t>(1, threads / V));
    const int64_t blocks = (R * V + kTableThreads - 1) / kTableThreads;
    if (blocks > 0x7FFFFFFF || R * V > 0xFFFFFFFFll || V > 0x7FFFFFFF || R > 0x7FFFFFFF) return false;
    const size_t smem = silu ? kTableSmem : tail_smem(gated);
    const void *kern;
    if (!silu)
        kern = prm.mult ? tail_kernel<true>(code, mode, gated) : tail_kernel<false>(code, mode, gated);
    else if (code == SQ_CODE_INT8)
        kern = mode == kDual ? reinterpret_cast<const void *>(quantize_silu_table_kernel<SQ_CODE_INT8, kDual>)
                             : reinterpret_cast<const void *>(quantize_silu_table_kernel<SQ_CODE_INT8, kSingle>);
    else
        kern = mode == kDual ? reinterpret_cast<const void *>(quantize_silu_table_kernel<SQ_CODE_E4M3, kDual>)
                             : reinterpret_cast<const void *>(quantize_silu_table_kernel<SQ_CODE_E4M3, kSingle>);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    prm.V = int(V);
    prm.R = int(R);
    L.blocks = unsigned(blocks);
    L.kernel = kern;
    L.threads = kTableThreads;
    L.smem = unsigned(smem);
    return true;
}

}  // namespace

void set_quantize_table_mode(int mode) { g_table_mode.store(mode, std::memory_order_relaxed); }

sq_status prepare_quantize(const void *X, sq_dtype dt, int64_t M, int64_t K, int64_t ld, const SegBounds &sb,
                           const float *s_pos, const float *s_neg, const int32_t *zero_point, int row_segments,
                           sq_code code, float q_max, float q_min_abs, int act, const float *mult,
                           void *c_pos, void *c_neg, int64_t ldc, QuantLaunch *out)
{
    QuantParams &prm = out->prm;
    prm = QuantParams{};
    out->threads = 0;
    out->smem = 0;
    prm.X = X; prm.M = M; prm.K = int(K); prm.ld = ld;
    prm.sb = sb;
    prm.s_pos = s_pos; prm.s_neg = s_neg; prm.zp = zero_point;
    prm.row_segments = row_segments;
    // dual: codes in [-|q_min|, q_max]; single scale: symmetric [-q_max, q_max]; zero-point: the whole int8 range
    prm.hi = int(q_max);
    prm.lo = (s_neg || zero_point) ? -int(q_min_abs) : -int(q_max);
    prm.c_pos = static_cast<uint8_t *>(c_pos); prm.c_neg = static_cast<uint8_t *>(c_neg); prm.ldc = ldc;
    prm.act = act; prm.mult = mult;
    const int mode = zero_point ? kZeroPoint : (s_neg ? kDual : kSingle);
    if (prepare_table(*out, dt, code, mode)) return SQ_OK;
    return dt == SQ_F32 ? prepare_mode<float>(*out, code, mode) : prepare_mode<__nv_bfloat16>(*out, code, mode);
}

sq_status run_quantize(const QuantLaunch &L, cudaStream_t st)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(L.blocks);
    cfg.blockDim = dim3(L.threads ? L.threads : unsigned(kThreads));
    cfg.dynamicSmemBytes = L.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void *args[1] = {const_cast<QuantParams *>(&L.prm)};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, L.kernel, args);
    count_launch();
    if (e != cudaSuccess) { note_cuda_error(e); return SQ_ERR_CUDA; }
    return SQ_OK;
}

sq_status launch_quantize(const void *X, sq_dtype dt, int64_t M, int64_t K, int64_t ld, const SegBounds &sb,
                          const float *s_pos, const float *s_neg, const int32_t *zero_point, int row_segments,
                          sq_code code, float q_max, float q_min_abs, int act, const float *mult,
                          void *c_pos, void *c_neg, int64_t ldc, cudaStream_t st)
{
    QuantLaunch L;
    const sq_status s = prepare_quantize(X, dt, M, K, ld, sb, s_pos, s_neg, zero_point, row_segments, code, q_max,
                                         q_min_abs, act, mult, c_pos, c_neg, ldc, &L);
    return s == SQ_OK ? run_quantize(L, st) : s;
}

// Chunks per thread for M rows of V chunks in P K-segments.  With several segments one is the better up to V = 256 (time
// with 1 over time with 4, M 512 .. 32768, K 512 .. 4096: 0.57 .. 1.00).  With one segment a row costs so little beside its
// loads that, on many rows, four chunks on a quarter of the threads win where these fill their warps reasonably
// (1 / 4, M = 8858 bf16 single: K = 3072 1.18, 2560 0.99 (40 of 64 threads), 2048 1.16, 1536 1.14, 1024 0.99; M = 16000,
// K = 2816 1.17; fp32 single, M = 8858: 1.04, 0.93, 1.10, 0.96, 0.95).  On few rows one wins there too (M = 1024:
// 0.81 .. 1.01).  The lines below are where the ratio crosses 1 (bf16 dual, K = 2048: M = 2048 0.89, 4096 1.05, 6000 1.10;
// K = 4096: M = 1024 0.93, 2048 1.10).
template <typename Tin>
static int64_t per_row_chunks(int64_t M, int64_t V, int P)
{
    constexpr bool k16 = sizeof(Tin) == 2;
    if (V > kThreads) return kRowChunks;
    if (P > 1) return 1;
    if (V > 160) return M >= 2048 ? kRowChunks : 1;                              // K > 2560: two warps with four chunks a thread
    if (V <= 128 && V > 96) return M >= (k16 ? 4096 : 6000) ? kRowChunks : 1;    // K > 1536: one warp
    if (V <= 96 && V > 64) return k16 && M >= 6000 ? kRowChunks : 1;             // K > 1024
    return 1;
}

template <typename Tin, bool DUAL, typename... Args>
static cudaError_t launch_per_row(cudaLaunchConfig_t &cfg, int64_t V, int P, Args... args)
{
    const int64_t chunks = per_row_chunks<Tin>(int64_t(cfg.gridDim.x), V, P);
    cfg.blockDim = dim3(unsigned(((V + chunks - 1) / chunks + 31) / 32 * 32));
    return chunks == 1 ? cudaLaunchKernelEx(&cfg, quantize_per_row_kernel<Tin, DUAL, 1>, args...)
                       : cudaLaunchKernelEx(&cfg, quantize_per_row_kernel<Tin, DUAL, kRowChunks>, args...);
}

sq_status launch_quantize_per_row(const void *X, sq_dtype dt, int64_t M, int64_t K, int64_t ld, const SegBounds &sb,
                                  int dual, float q_max, float q_min_abs, float *s_pos, float *s_neg,
                                  void *c_pos, void *c_neg, int64_t ldc, cudaStream_t st)
{
    const int64_t V = (K + kVec - 1) / kVec;
    if (V > int64_t(kThreads) * kRowChunks) return SQ_ERR_UNSUPPORTED;      // the row is held in registers
    if (M > 0x7FFFFFFF) return SQ_ERR_SHAPE;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(unsigned(M));
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    uint8_t *cp = static_cast<uint8_t *>(c_pos), *cn = static_cast<uint8_t *>(c_neg);
    const int Ki = int(K);
    cudaError_t e;
    if (dt == SQ_F32) {
        const float *x = static_cast<const float *>(X);
        e = dual ? launch_per_row<float, true>(cfg, V, sb.P, x, Ki, ld, sb, q_max, q_min_abs, s_pos, s_neg, cp, cn, ldc)
                 : launch_per_row<float, false>(cfg, V, sb.P, x, Ki, ld, sb, q_max, q_min_abs, s_pos, s_neg, cp, cn, ldc);
    } else {
        const __nv_bfloat16 *x = static_cast<const __nv_bfloat16 *>(X);
        e = dual ? launch_per_row<__nv_bfloat16, true>(cfg, V, sb.P, x, Ki, ld, sb, q_max, q_min_abs, s_pos, s_neg, cp, cn, ldc)
                 : launch_per_row<__nv_bfloat16, false>(cfg, V, sb.P, x, Ki, ld, sb, q_max, q_min_abs, s_pos, s_neg, cp, cn, ldc);
    }
    count_launch();
    if (e != cudaSuccess) { note_cuda_error(e); return SQ_ERR_CUDA; }
    return SQ_OK;
}

sq_status launch_pack_w4(const void *Wq8, int64_t ld8, int64_t N, int64_t K, void *Wq4, int64_t ld4, int unpack,
                         cudaStream_t st)
{
    const int64_t total = N * (K / kVec), chunks = (total + kThreads - 1) / kThreads;
    if (chunks > 0x7FFFFFFF) return SQ_ERR_SHAPE;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        return SQ_ERR_CUDA;
    // several chunks a thread where that leaves every SM some blocks to follow one another (unpack, us, one / four chunks, blocks of
    // single chunks per SM: 8.8 2.9 / 3.8, 13.5 3.8 / 4.2, 20.3 4.9 / 5.0, 27 6.0 / 5.5)
    const int per_thread = chunks > int64_t(sms) * 20 ? kPackChunks : 1;
    const int64_t blocks = (chunks + per_thread - 1) / per_thread;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(unsigned(blocks));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    uint8_t *w8 = static_cast<uint8_t *>(const_cast<void *>(Wq8)), *w4 = static_cast<uint8_t *>(Wq4);
    const uint32_t V = uint32_t(K / kVec);
    cudaError_t e;
    if (blocks * kThreads * per_thread > 0xFFFFFFFFll)
        e = unpack ? cudaLaunchKernelEx(&cfg, pack_w4_kernel<int64_t, true, kPackChunks>, w8, ld8, total, V, w4, ld4)
                   : cudaLaunchKernelEx(&cfg, pack_w4_kernel<int64_t, false, kPackChunks>, w8, ld8, total, V, w4, ld4);
    else if (per_thread > 1)
        e = unpack ? cudaLaunchKernelEx(&cfg, pack_w4_kernel<uint32_t, true, kPackChunks>, w8, ld8, uint32_t(total), V, w4, ld4)
                   : cudaLaunchKernelEx(&cfg, pack_w4_kernel<uint32_t, false, kPackChunks>, w8, ld8, uint32_t(total), V, w4, ld4);
    else
        e = unpack ? cudaLaunchKernelEx(&cfg, pack_w4_kernel<uint32_t, true, 1>, w8, ld8, uint32_t(total), V, w4, ld4)
                   : cudaLaunchKernelEx(&cfg, pack_w4_kernel<uint32_t, false, 1>, w8, ld8, uint32_t(total), V, w4, ld4);
    count_launch();
    if (e != cudaSuccess) { note_cuda_error(e); return SQ_ERR_CUDA; }
    return SQ_OK;
}

}  // namespace sq
