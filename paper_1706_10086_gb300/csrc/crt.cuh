// The moduli of the modular emulated GEMM and reduction modulo them, shared by
// the split, the tensor-core epilogue and the reconstruction.
#pragma once

#include <cstdint>

namespace alp {

// The moduli, largest first (pairwise coprime; 256 = 2^8 first).
__host__ __device__ __forceinline__ constexpr uint32_t crt_modulus(int l) {
    switch (l) {
        case 0: return 256u;
        case 1: return 255u;
        case 2: return 253u;
        case 3: return 251u;
        case 4: return 247u;
        case 5: return 241u;
        case 6: return 239u;
        case 7: return 233u;
        case 8: return 229u;
        case 9: return 227u;
        case 10: return 223u;
        case 11: return 217u;
        case 12: return 211u;
        case 13: return 199u;
        case 14: return 197u;
        case 15: return 193u;
        default: return 1u;
    }
}
// 2^bits mod m.
__host__ __device__ __forceinline__ constexpr uint32_t crt_pow2_mod(int bits, uint32_t m) {
    uint32_t r = 1u % m;
    for (int i = 0; i < bits; ++i) r = (r * 2u) % m;
    return r;
}
// r in [0, m) as the residue of least magnitude.
__host__ __device__ __forceinline__ constexpr int crt_symmetric(uint32_t r, uint32_t m) {
    return r > m / 2 - (m % 2 == 0 ? 1 : 0) ? (int)r - (int)m : (int)r;
}
// Bytes y 256^i mod m, i = i0 .. i0 + 3, symmetric.
__host__ __device__ __forceinline__ constexpr uint32_t crt_byte_weights(uint32_t m, int i0,
                                                                        uint32_t y = 1) {
    uint32_t w = 0;
    for (int i = 0; i < 4; ++i)
        w |= ((uint32_t)crt_symmetric(y * crt_pow2_mod(8 * (i0 + i), m) % m, m) & 0xFFu) << (8 * i);
    return w;
}
// d = c + the dot product of a's unsigned and b's signed bytes.
__device__ __forceinline__ int crt_dp4a(uint32_t a, int b, int c) {
    int d;
    asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// The weighted residue (Q y) mod m in [0, m) of a sum |Q| <= 2^30, from U = Q +
// 2^31 (the running sums start at 2^31): the byte dot product of U with w_i =
// y 256^i mod m (symmetric) less 2^31 y mod m is x = Q y (mod m), |x| < 2^17,
// added into the encoding of 1.5 2^23 (F = 1.5 2^23 + x); with h = (m - 1) / 2, q
// = RN((x - h) / m) is floor(x / m) (for odd m the fraction stays 1/(2m) from
// a half, far above the rounding of the product with RN(1/m)), and F - q m, one
// exact fma, is 1.5 2^23 + x mod m: its encoding's low byte.  For m = 256 that
// byte is x mod 256 whatever q is.  Five instructions, where two reductions by
// multiply-high (|Q|, the weight, the sign) took about twenty: at K <= 1024 the
// epilogue was longer than the next modulus's products (1024^3 82.8 -> 68.2 us,
// 8192 x 8192 x 1024 2271 -> 1929, 2048^3 277 -> 256, 15 moduli).
struct CrtByte {
    int w, c;             // weights; the encoding of 1.5 2^23 less 2^31 y mod m
    float off, inv, m;    // 1.5 2^23 + h, RN(1/m), m
};
__device__ __forceinline__ uint32_t crt_byte(uint32_t U, const CrtByte& k) {
    const float F = __int_as_float(crt_dp4a(U, k.w, k.c));
    const float q = __fadd_rn(__fmaf_rn(__fadd_rn(F, -k.off), k.inv, 12582912.0f), -12582912.0f);
    return (uint32_t)__float_as_int(__fmaf_rn(-q, k.m, F));
}
// The bytes of four sums in one word.
__device__ __forceinline__ uint32_t crt_bytes4(const uint32_t* U, const CrtByte& k) {
    const uint32_t lo = __byte_perm(crt_byte(U[0], k), crt_byte(U[1], k), 0x0040);
    const uint32_t hi = __byte_perm(crt_byte(U[2], k), crt_byte(U[3], k), 0x0040);
    return __byte_perm(lo, hi, 0x5410);
}
constexpr uint32_t kCrtSumZero = 0x80000000u;   // a running sum's start

}  // namespace alp
