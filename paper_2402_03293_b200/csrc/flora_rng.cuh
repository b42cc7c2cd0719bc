// Device-side generator of the projection A ~ N_seed(0, 1/r)  (Algorithm 1: "A_W <- N_{s_W}(0, 1/r)").
//
// A[j,k] is a function of (seed, j, k): Philox4x32-10 (Salmon et al., SC'11) keyed by the two
// halves of the seed, counter (k/4, j, 0, 0), gives four words; words (0,1) make columns 4q, 4q+1
// (cosine and sine branch of Box-Muller), words (2,3) make 4q+2, 4q+3.  The definition uses only
// IEEE-754 binary32 operations with a fixed order, so the value is reproducible bit by bit on any
// IEEE machine.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace flora {

struct PhiloxKey {
    uint32_t k0, k1;
};

__host__ __device__ __forceinline__ PhiloxKey make_key(uint64_t seed)
{
    PhiloxKey k;
    k.k0 = (uint32_t)(seed & 0xFFFFFFFFull);
    k.k1 = (uint32_t)(seed >> 32);
    return k;
}

// What bounds the kernels at large ranks is this generator: issue slots of the plain ALUs, nothing else.  As written below a
// normal takes 31 of them (54 in the form it had before) and a B200 makes 0.69 x 10^12 of them a second with eight warps on
// an SM and 0.81 with 28 (0.47 and 0.65 before), measured in a loop of nothing else:
//   * two Philox blocks at a time share the key schedule;
//   * what comes in pairs runs in packed instructions (two fp32 operations each, rounded as the scalar ones are);
//   * the logarithm is evaluated in -2s with every constant scaled by a power of two, the octant reduction by the sign of
//     the 22 low bits read as a signed number, so that neither needs fix-up instructions;
//   * the square root is one Newton (Heron) step on the hardware's estimate; its argument is never negative, subnormal or infinite.
// Every rounding step is the one of the definition; only exact operations were rearranged.

// Two Philox4x32-10 blocks with counters (qa, ja, 0, 0) and (qb, jb, 0, 0).
__device__ __forceinline__ void philox_two(uint32_t qa, uint32_t ja, uint32_t qb, uint32_t jb, PhiloxKey key, uint32_t (&x)[4], uint32_t (&y)[4])
{
    uint32_t a0 = qa, a1 = ja, a2 = 0u, a3 = 0u, b0 = qb, b1 = jb, b2 = 0u, b3 = 0u;
    uint32_t k0 = key.k0, k1 = key.k1;
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        const uint64_t pa0 = (uint64_t)0xD2511F53u * (uint64_t)a0, pa1 = (uint64_t)0xCD9E8D57u * (uint64_t)a2;
        const uint64_t pb0 = (uint64_t)0xD2511F53u * (uint64_t)b0, pb1 = (uint64_t)0xCD9E8D57u * (uint64_t)b2;
        const uint32_t na0 = (uint32_t)(pa1 >> 32) ^ a1 ^ k0, na2 = (uint32_t)(pa0 >> 32) ^ a3 ^ k1;
        const uint32_t nb0 = (uint32_t)(pb1 >> 32) ^ b1 ^ k0, nb2 = (uint32_t)(pb0 >> 32) ^ b3 ^ k1;
        a1 = (uint32_t)pa1;
        a3 = (uint32_t)pa0;
        a0 = na0;
        a2 = na2;
        b1 = (uint32_t)pb1;
        b3 = (uint32_t)pb0;
        b0 = nb0;
        b2 = nb2;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    x[0] = a0; x[1] = a1; x[2] = a2; x[3] = a3;
    y[0] = b0; y[1] = b1; y[2] = b2; y[3] = b3;
}

// Two fp32 values side by side (packed arithmetic: one instruction, each half rounded to nearest even on its own).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ f32x2 both(float v) { return pack2(v, v); }
// ... of a constant, given by its bit pattern (a 64-bit literal: the compiler does not keep it in a register pair)
#define FLORA_BOTH(bits) (0x100000001ull * bits##u)
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// -2 ln(u1) for u1 = ((xa >> 8) + 1) / 2^24, of two words.  u1 = 2^(e - 24) mant with mant in [2/3, 4/3) and s = mant - 1:
// ln(mant) = s - s^2/2 + s^3 Q(s).  The polynomial runs in t = -2s with coefficients (-1/2)^k times those of Q, -1/2 and 1
// (powers of two: the same roundings), which leaves -2 ln(mant) directly.
__device__ __forceinline__ f32x2 neg2_ln_u1(uint32_t xa0, uint32_t xa1)
{
    const uint32_t b0 = __float_as_uint(__uint2float_rn((xa0 >> 8) + 1u)), b1 = __float_as_uint(__uint2float_rn((xa1 >> 8) + 1u));   // exact
    const uint32_t e0 = (b0 - 0x3F2AAAABu) & 0xFF800000u, e1 = (b1 - 0x3F2AAAABu) & 0xFF800000u;         // e * 2^23
    const f32x2 t = fma2(pack2(__uint_as_float(b0 - e0), __uint_as_float(b1 - e1)), FLORA_BOTH(0xC0000000) /* -2.0 */, FLORA_BOTH(0x40000000) /* 2.0 */);   // exact
    f32x2 q = FLORA_BOTH(0x3A0D84F4) /* 0x1.1b09e8p-11 */;
    q = fma2(q, t, FLORA_BOTH(0x3A9AD9F0) /* 0x1.35b3ep-10 */);
    q = fma2(q, t, FLORA_BOTH(0x3B0FCB11) /* 0x1.1f9622p-9 */);
    q = fma2(q, t, FLORA_BOTH(0x3BA8AD36) /* 0x1.515a6cp-8 */);
    q = fma2(q, t, FLORA_BOTH(0x3C4CE190) /* 0x1.99c32p-7 */);
    q = fma2(q, t, FLORA_BOTH(0x3D00058E) /* 0x1.000b1cp-5 */);
    q = fma2(q, t, FLORA_BOTH(0x3DAAAA94) /* 0x1.555528p-4 */);
    q = fma2(q, t, FLORA_BOTH(0x3E800000) /* 0.25 */);
    const f32x2 ln_mant = fma2(q, mul2(t, t), t);
    const f32x2 steps = fma2(pack2(__int2float_rn((int)e0), __int2float_rn((int)e1)), FLORA_BOTH(0xB4000000) /* -0x1p-23 */, FLORA_BOTH(0x41C00000) /* 24.0 */);   // 24 - e, exact
    return fma2(steps, FLORA_BOTH(0x3FB17218) /* 0x1.62e43p+0 */, ln_mant);
}

// Square roots of two values of neg2_ln_u1, rounded to nearest: one Newton (Heron) step g + (x - g^2) / (2 g) from the
// hardware's estimate of 1 / sqrt(x), with the residual in one fma.  Equal to the IEEE square root on the values that neg2_ln_u1
// takes (2^24 at most; the tests compare 2^27 draws of them bit by bit); 0 is the only special one among them.
__device__ __forceinline__ f32x2 sqrt_of_ln(f32x2 x)
{
    float x0, x1, y0, y1;
    unpack2(x, x0, x1);
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(fmaxf(x0, 1e-20f)));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y1) : "f"(fmaxf(x1, 1e-20f)));
    const f32x2 y = pack2(y0, y1), g = mul2(x, y);
    return fma2(fma2(mul2(g, FLORA_BOTH(0xBF800000) /* -1.0 */), g, x), mul2(y, FLORA_BOTH(0x3F000000) /* 0.5 */), g);
}

// cos and sin of 2 pi (xb >> 8) / 2^24, of two words, without the exchange and the signs of their octants: fixed polynomials
// on [0, pi/4].  The 22 low bits of xb >> 8, read as a signed number, are the distance to the nearer end of the quarter turn.
__device__ __forceinline__ void cos_sin_octant(uint32_t xb0, uint32_t xb1, f32x2& c, f32x2& s)
{
    const float q0 = fabsf(__int2float_rn((int)((xb0 << 2) & 0xFFFFFC00u))), q1 = fabsf(__int2float_rn((int)((xb1 << 2) & 0xFFFFFC00u)));  // exact
    const f32x2 x = mul2(pack2(q0, q1), FLORA_BOTH(0x2FC90FDB) /* 0x1.921fb6p-32 */);
    const f32x2 z = mul2(x, x);
    f32x2 sp = fma2(FLORA_BOTH(0xB94CA1F1) /* -0x1.9943e2p-13 */, z, FLORA_BOTH(0x3C08839D) /* 0x1.11073ap-7 */);
    sp = fma2(sp, z, FLORA_BOTH(0xBE2AAAA3) /* -0x1.555546p-3 */);
    s = fma2(mul2(x, z), sp, x);
    f32x2 cp = fma2(FLORA_BOTH(0xBAB226B1) /* -0x1.644d62p-10 */, z, FLORA_BOTH(0x3D2A9F40) /* 0x1.553e8p-5 */);
    cp = fma2(cp, z, FLORA_BOTH(0xBEFFFFD9) /* -0x1.ffffb2p-2 */);
    c = fma2(z, cp, FLORA_BOTH(0x3F800000) /* 1.0 */);
}
// One word's octant: cosine and sine change places in the odd half of each quarter turn, and take their signs.
__device__ __forceinline__ f32x2 in_octant(uint32_t xb, float c, float s)
{
    const uint32_t t = xb ^ (xb << 1);
    const bool swap = (t & 0x40000000u) != 0u;
    return pack2(__uint_as_float(__float_as_uint(swap ? s : c) ^ (t & 0x80000000u)), __uint_as_float(__float_as_uint(swap ? c : s) ^ (xb & 0x80000000u)));
}

// Four scaled normals from the four words of a Philox block: (rho cos, rho sin) * scale of words (0, 1), then of (2, 3);
// scale = fl32(1/sqrtf(r)).
__device__ __forceinline__ void normals(const uint32_t (&x)[4], float scale, float (&a)[4])
{
    float r0, r1, c0, c1, s0, s1;
    unpack2(sqrt_of_ln(neg2_ln_u1(x[0], x[2])), r0, r1);
    f32x2 c, s;
    cos_sin_octant(x[1], x[3], c, s);
    unpack2(c, c0, c1);
    unpack2(s, s0, s1);
    unpack2(mul2(mul2(both(r0), in_octant(x[1], c0, s0)), both(scale)), a[0], a[1]);
    unpack2(mul2(mul2(both(r1), in_octant(x[3], c1, s1)), both(scale)), a[2], a[3]);
}

// A[ja, 4qa .. 4qa+3] and A[jb, 4qb .. 4qb+3] as fp32.
__device__ __forceinline__ void projection_two_quads(uint32_t qa, uint32_t ja, uint32_t qb, uint32_t jb, PhiloxKey key, float scale, float (&a)[4],
                                                     float (&b)[4])
{
    uint32_t x[4], y[4];
    philox_two(qa, ja, qb, jb, key, x, y);
    normals(x, scale, a);
    normals(y, scale, b);
}
// A[j, 4q .. 4q+3] as fp32.
__device__ __forceinline__ void projection_quad(uint32_t q, uint32_t j, PhiloxKey key, float scale, float (&a)[4])
{
    uint32_t x[4], y[4];
    philox_two(q, j, q, j, key, x, y);           // (the second block is the first: it costs nothing)
    normals(x, scale, a);
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
// A[j, 4q .. 4q+7] rounded to bf16 (nearest even), two columns to a word; the lower column sits in the low half.
__device__ __forceinline__ uint4 projection_octet_bf16(uint32_t q, uint32_t j, PhiloxKey key, float scale)
{
    float a[4], b[4];
    projection_two_quads(q, j, q + 1, j, key, scale, a, b);
    return make_uint4(pack_bf16(a[0], a[1]), pack_bf16(a[2], a[3]), pack_bf16(b[0], b[1]), pack_bf16(b[2], b[3]));
}

__device__ __forceinline__ float bf16_round(float v)
{
    return __bfloat162float(__float2bfloat16_rn(v));
}

// Adds up what fp32 products made in parts come to: the sum of the large products (upper part times upper part) and that of the others.
// Where an operand is infinite its lower parts are NaN, or meet an upper part of either sign; the large products alone are then what
// plain arithmetic gives, sign by sign (the upper part of an infinity is that infinity, of a NaN a NaN, and A is never zero).
__device__ __forceinline__ float join_parts(float large, float rest) { return fabsf(large) < __int_as_float(0x7F800000) ? large + rest : large; }

}  // namespace flora
