// Device helpers shared by the activation-quantization kernels: Eq. 1 codes equal to
// round_half_even(v / s) with a true fp32 division (bit for bit), and fp16 unpacking.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace muxq {

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Eq. 1: code = clamp(round_half_even(v / s), -q, q) with a true fp32 division.
__device__ __forceinline__ int quant_exact(float v, float s, float qf) {
    float t = rintf(__fdiv_rn(v, s));
    t = fminf(fmaxf(t, -qf), qf);
    return __float2int_rn(t);
}

__device__ __forceinline__ void unpack8(const uint4 &v, float (&f)[8]) {
    const __half2 *h = reinterpret_cast<const __half2 *>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float2 p = __half22float2(h[i]);
        f[2 * i] = p.x;
        f[2 * i + 1] = p.y;
    }
}

// 8 values (already multiplied by their channel factors) -> 8 codes packed in a uint2.
//
// Fast path: p = v * (1/s), taken exactly inside a fused multiply-add, differs from the correctly
// rounded quotient v / s by less than 1.6e-5 for |v/s| <= 128, so whenever p is farther than 1e-4
// from every half-integer both round to the same integer.  fma(v, 1/s, 1.5 * 2^23) rounds p to that
// integer (round half to even) and leaves its two's-complement low byte in the low byte of the
// float's bit pattern, which a byte permute packs directly; a second fma gives p minus that integer.
// If any of the 8 values is too close to a tie, or exceeds the code range (possible only when the
// scale was not derived from these values), all 8 take the exact division.
__device__ __forceinline__ uint2 quant8(const float (&f)[8], float s, float inv_s, float qf) {
    const float magic = 12582912.0f;  // 1.5 * 2^23
    uint32_t b[8];
    float dmax = 0.0f, amax = 0.0f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float tm = fmaf(f[i], inv_s, magic);
        const float n = tm - magic;
        dmax = fmaxf(dmax, fabsf(fmaf(f[i], inv_s, -n)));
        amax = fmaxf(amax, fabsf(n));
        b[i] = __float_as_uint(tm);
    }
    if (dmax > 0.4999f || amax > qf) {
#pragma unroll
        for (int i = 0; i < 8; ++i) b[i] = (uint32_t)quant_exact(f[i], s, qf);
    }
    const uint32_t p01 = __byte_perm(b[0], b[1], 0x0040), p23 = __byte_perm(b[2], b[3], 0x0040);
    const uint32_t p45 = __byte_perm(b[4], b[5], 0x0040), p67 = __byte_perm(b[6], b[7], 0x0040);
    return make_uint2(__byte_perm(p01, p23, 0x5410), __byte_perm(p45, p67, 0x5410));
}

// low bytes of 8 words -> 8 codes in a uint2
__device__ __forceinline__ uint2 pack8(const uint32_t (&b)[8]) {
    const uint32_t p01 = __byte_perm(b[0], b[1], 0x0040), p23 = __byte_perm(b[2], b[3], 0x0040);
    const uint32_t p45 = __byte_perm(b[4], b[5], 0x0040), p67 = __byte_perm(b[6], b[7], 0x0040);
    return make_uint2(__byte_perm(p01, p23, 0x5410), __byte_perm(p45, p67, 0x5410));
}

// Two fp32 operations per instruction (each rounded like the scalar one).
__device__ __forceinline__ uint64_t pack2(float x, float y) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Eq. 1 without a division and without a branch, for a scale s derived from the values themselves (no code leaves [-q, q]): the same integer as rounding the correctly rounded quotient x / s.
//
// With inv = RN(1/s), q0 = RN(x inv), rest = x - q0 s and q = RN(q0 + rest inv) (Markstein, IBM J. Res. Dev. 34, 1990), q decides
// like RN(x/s) at every tie t = n + 1/2, |t| < 128, for an x of at most 11 significant bits.  Let Q = x/s, u = ulp(t), s =
// S 2^(e-23) with 2^23 <= S < 2^24; inv is off by a relative S 2^-48 at most.  What matters is Q next to a midpoint t +- u/2:
//   - Q is never on it (an odd number of 25 bits would divide the significand of x), and no nearer than u / (2S): x - s t is a
//     multiple of 2^(e-24), s u / 2 one of 2^(e-24) 2^(et-23) with et the exponent of t;
//   - x inv is within (t 2^-et) S 2^-25 u < 0.997 u of Q, so q0 is one of the two floats beside the midpoint, rest is below
//     2^24 units of ulp(q0) ulp(s) and exact, and q0 + rest inv is off by u/2 * S 2^-48 < u / (2S) at most: the same side.
// (Just below t = 1/2, where u halves, Q keeps a quarter of 2^(e-24) / s from the midpoint.)  Everywhere else the order of Q and
// t survives by monotonicity.  Structural ties (127 x / max a half-integer) are frequent in fp16 data, one value in some 300 to
// 1500, and which way s was rounded decides them: testing for them and dividing there took up to a quarter of the instructions.
// Adding 1.5 * 2^23 rounds q to an integer, half to even, whose low byte is the code.
__device__ __forceinline__ uint64_t quotient2(uint64_t x, uint64_t inv2, uint64_t neg_s2) {
    const uint64_t q0 = mul2(x, inv2);
    return add2(fma2(fma2(q0, neg_s2, x), inv2, q0), pack2(12582912.0f, 12582912.0f));
}
__device__ __forceinline__ uint2 quotient8(const uint64_t (&x)[4], uint64_t inv2, uint64_t neg_s2) {
    uint32_t b[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint64_t n = quotient2(x[j], inv2, neg_s2);
        b[2 * j] = (uint32_t)n;
        b[2 * j + 1] = (uint32_t)(n >> 32);
    }
    return pack8(b);
}
__device__ __forceinline__ void unpack8(const uint4 &v, uint64_t (&x)[4]) {
    const __half2 *h = reinterpret_cast<const __half2 *>(&v);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 p = __half22float2(h[j]);
        x[j] = pack2(p.x, p.y);
    }
}
__device__ __forceinline__ uint2 quotient8(const uint4 &v, uint64_t inv2, uint64_t neg_s2) {
    uint64_t x[4];
    unpack8(v, x);
    return quotient8(x, inv2, neg_s2);
}
__device__ __forceinline__ uint2 quotient8(const float (&f)[8], float inv, float s) {
    const uint64_t x[4] = {pack2(f[0], f[1]), pack2(f[2], f[3]), pack2(f[4], f[5]), pack2(f[6], f[7])};
    return quotient8(x, pack2(inv, inv), pack2(-s, -s));
}

// Two operations fewer per value, for loops bound by the fp32 pipe: the codes where a bracket decides, else nonzero (the caller
// then takes quotient8).  The correctly rounded quotient differs from the real product x inv by a relative 2^-23 (1 + 2^-23) at
// most, so it lies between x lo and x hi for lo / hi three units in the last place below / above inv.  Adding 1.5 * 2^23 inside the
// fused operation rounds both real products to integers once each; rounding is monotone, so where they agree the quotient rounds
// to that integer too.  Power-of-two channel factors folded into lo / hi keep this exact.
__device__ __forceinline__ void recip_bracket(float inv_s, float &lo, float &hi) {
    lo = __uint_as_float(__float_as_uint(inv_s) - 3u);  // inv_s is a positive normal number
    hi = __uint_as_float(__float_as_uint(inv_s) + 3u);
}
__device__ __forceinline__ uint32_t bracket8(const float (&f)[8], const float (&lo)[8], const float (&hi)[8], uint2 &code) {
    uint32_t b[8], diff = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        b[i] = __float_as_uint(fmaf(f[i], hi[i], 12582912.0f));
        diff |= b[i] ^ __float_as_uint(fmaf(f[i], lo[i], 12582912.0f));
    }
    code = pack8(b);
    return diff;
}
__device__ __forceinline__ uint32_t bracket8(const float (&f)[8], float lo, float hi, uint2 &code) {
    const float l[8] = {lo, lo, lo, lo, lo, lo, lo, lo}, h[8] = {hi, hi, hi, hi, hi, hi, hi, hi};
    return bracket8(f, l, h, code);
}

}  // namespace muxq
