// Device helpers of the emulated GEMMs: the exact fixed-point form of a
// scaled operand, its digits, bf16 packing, the split kernels (rows of a
// row-major matrix, or its columns through shared memory), which take a
// splitter object that turns one value into S small integers and packs two
// of them into bf16, and the rounding of a 128-bit integer to double.
#pragma once

#include <cuda_bf16.h>

#include <type_traits>
#include <utility>

#include "alp_internal.cuh"

namespace alp {

// The frexp exponent of a double given by its bits without the sign: the e
// with 2^(e-1) <= |x| < 2^e (0 for zero).
__device__ __forceinline__ int frexp_exponent_of_bits(uint64_t mb) {
    if (mb == 0) return 0;
    const int ex = (int)(mb >> 52);
    if (ex == 0) return (63 - __clzll((long long)mb)) - 1073;   // subnormal
    return ex - 1022;
}

constexpr uint64_t kAbsMask = 0x7FFFFFFFFFFFFFFFull;

// |x| as ordered integer keys (larger key, larger |x|): the bits of a double
// without its sign, or of a float.  A key at or above the infinity's is Inf
// or NaN.  The float key converts to the double bits of the same value for
// the exponent (FP32 operands convert exactly, so frexp and the digits are
// the same as for the double of equal value).
template <typename T> struct ScanKey;
template <> struct ScanKey<double> {
    using type = uint64_t;
    static constexpr uint64_t kInf = 0x7FF0000000000000ull;
    __device__ static uint64_t of(uint64_t bits) { return bits & kAbsMask; }
    __device__ static uint64_t to_double_bits(uint64_t k) { return k; }
};
template <> struct ScanKey<float> {
    using type = uint32_t;
    static constexpr uint32_t kInf = 0x7F800000u;
    __device__ static uint32_t of(uint32_t bits) { return bits & 0x7FFFFFFFu; }
    __device__ static uint64_t to_double_bits(uint32_t k) {
        return (uint64_t)__double_as_longlong((double)__int_as_float((int)k));
    }
};

// ---------------------------------------------------------------------------
// 2. split
// ---------------------------------------------------------------------------
// The split kernels take a splitter object, so that other integer
// representations of the operands (the residues of the modular scheme) reuse
// them: init<S>(a, e) gives what the S slices of one value are formed from,
// next<L> its L-th slice (asked for in order) as the encoding of a float, pack
// two of those as bf16: a float holding an integer of at most 8 significant
// bits has that integer's bf16 encoding in its upper 16 bits, so packing is
// one byte permutation.
__device__ __forceinline__ uint32_t pack_bf16x2(int lo, int hi) {
    return __byte_perm((uint32_t)lo, (uint32_t)hi, 0x7632);
}

// Digits of a * 2^-e.  |a| 2^-e is held as a 64-bit fixed-point number Y with 62
// fraction bits, rounded to odd (truncate, then set the last bit if anything
// was cut off): every later rounding happens at least 2 bits above that last
// bit, so the digits equal those of the exact value ((s-1) b + 2 <= 62 - b).
// T: the mantissa with its leading one at bit 61, D: how far down it belongs.
__device__ __forceinline__ uint64_t fixed_point_mag(uint64_t T, int D) {
    const int d = D < 0 ? 0 : D > 63 ? 63 : D;
    const uint64_t Y = T >> d;
    return Y | ((Y << d) != T ? 1ull : 0ull);
}
__device__ __forceinline__ uint64_t fixed_point_mag(double a, int e) {
    const uint32_t hi = (uint32_t)__double2hiint(a), lo = (uint32_t)__double2loint(a);
    const int ex = (int)((hi >> 20) & 0x7FF);
    // Inf/NaN are reported by the scan (digits 0); subnormals have no hidden bit
    const uint32_t mh = ex == 0x7FF ? 0u : (hi & 0xFFFFFu) | (ex ? 0x100000u : 0u);
    const uint64_t m = ((uint64_t)mh << 32) | (ex == 0x7FF ? 0u : lo);
    return fixed_point_mag(m << 9, e + 1022 - (ex ? ex : 1));
}
__device__ __forceinline__ bool is_negative(double a) { return __double2hiint(a) < 0; }

// The digit schemes' splitter: digits of B bits, d_p = R_p - 2^B R_{p-1} with R_p
// the signed value X = +-Y rounded half to even at bit SH_p = 62 - B p (what
// rounding digit by digit, each from the exact remainder of the last, gives).
// Rounded half up instead, d_p is the signed B-bit field of X above SH_p plus
// the bit below it, read from one field of B + 1 bits; the two roundings differ
// only when X ends in exactly half a unit of some digit (at one digit, since
// nothing is left below it) above an even multiple: then half up of -X, negated,
// is half down of X, which is the even one.  Five instructions per digit where
// the digit-by-digit remainder in 64 bits took about fourteen (operands of 2048^3
// with 8 slices 62 -> 53 us).
//
// Floats are cut digit by digit in float arithmetic: x = a 2^(B - e), d = x
// rounded to the nearest integer, ties to even, by adding 1.5 2^23, and x = (x -
// d) 2^B, every step exact (x keeps at most a's 24 bits; what a scaling below
// the normal range could lose is far below the last digit's half).  Converted
// to double first (an FP64 operation each) and cut as one, the operands of an
// FP32 4096^3 took 112 us, now 67 (floor 50).
template <int B>
struct DigitSplit {
    struct Wide {
        uint32_t lo, hi;   // X, negated where half up would round to the odd side
        float sgn, off;    // 1 or -1, and -1.5 2^23 times it
    };
    struct Single {
        float x;
    };
    template <int S, typename T>
    using State = std::conditional_t<sizeof(T) == 8, Wide, Single>;
    template <int S>
    static constexpr uint64_t half_bits() {
        uint64_t m = 0;
        for (int p = 1; p <= S; ++p) m |= 1ull << (61 - B * p);
        return m;
    }
    template <int S>
    __device__ __forceinline__ Wide init(double a, int e) const {
        const uint64_t Y = fixed_point_mag(a, e), last = Y & (0ull - Y);
        const bool neg = __double2hiint(a) < 0;
        // in a tie the bit above the lowest set one is the parity of Y's
        // neighbour below, so opposite for -Y
        const bool minus = (last & half_bits<S>()) != 0 ? (Y & (last << 1)) == 0 : neg;
        const uint64_t s = minus ? ~0ull : 0ull, X = (Y ^ s) - s;
        const float sgn = minus == neg ? 1.0f : -1.0f;
        return {(uint32_t)X, (uint32_t)(X >> 32), sgn, -12582912.0f * sgn};
    }
    template <int S>
    __device__ __forceinline__ Single init(float a, int e) const {
        // 2^(B - e) as two normal factors (e is the same along a line)
        const int k = min(max(B - e, -240), 240), k1 = k / 2;
        return {a * __int_as_float((k1 + 127) << 23) * __int_as_float((k - k1 + 127) << 23)};
    }
    template <int L>
    __device__ __forceinline__ int next(Wide& u) const {
        constexpr int SH = 62 - B * (L + 1);
        constexpr int k = 64 - SH - B;   // the field's top bit to bit 63
        int v;                           // the field with the bit below it, signed
        if constexpr (L == 0) v = (int)u.hi >> (SH - 33);
        else if constexpr (k < 32) v = (int)__funnelshift_l(u.lo, u.hi, k) >> (31 - B);
        else v = (int)(u.lo << (k - 32)) >> (31 - B);
        // 0x4B400000 + ((v + 1) >> 1): the encoding of 1.5 2^23 + d
        const float f = __int_as_float((int)(((uint32_t)v + 0x96800001u) >> 1));
        return __float_as_int(__fmaf_rn(f, u.sgn, u.off));
    }
    template <int L>
    __device__ __forceinline__ int next(Single& u) const {
        const float d = __fadd_rn(__fadd_rn(u.x, 12582912.0f), -12582912.0f);
        u.x = __fmul_rn(__fadd_rn(u.x, -d), (float)(1 << B));
        return __float_as_int(d);
    }
    __device__ __forceinline__ uint32_t pack(int lo, int hi) const { return pack_bf16x2(lo, hi); }
};

// The S slices of two or four consecutive elements of a line, slice by slice
// (one store per plane, so that no more than one slice of each is live).
template <typename Sp, typename State, int... L>
__device__ __forceinline__ void split2_planes(const Sp& sp, State (&u)[2], uint32_t* o,
                                              int64_t step, std::integer_sequence<int, L...>) {
    auto put = [&](int a, int b) {
        *o = sp.pack(a, b);
        o += step;
    };
    (put(sp.template next<L>(u[0]), sp.template next<L>(u[1])), ...);
}
template <int S, typename Sp, typename T>
__device__ __forceinline__ void split2(const Sp& sp, T a0, T a1, int e, __nv_bfloat16* out,
                                       int64_t plane) {
    typename Sp::template State<S, T> u[2] = {sp.template init<S>(a0, e), sp.template init<S>(a1, e)};
    split2_planes(sp, u, reinterpret_cast<uint32_t*>(out), plane >> 1,
                  std::make_integer_sequence<int, S>());
}
template <typename Sp, typename State, int... L>
__device__ __forceinline__ void split4_planes(const Sp& sp, State (&u)[4], uint2* o,
                                              int64_t step, std::integer_sequence<int, L...>) {
    auto put = [&](int a, int b, int c, int d) {
        *o = make_uint2(sp.pack(a, b), sp.pack(c, d));
        o += step;
    };
    (put(sp.template next<L>(u[0]), sp.template next<L>(u[1]), sp.template next<L>(u[2]),
         sp.template next<L>(u[3])),
     ...);
}
template <int S, typename Sp, typename T>
__device__ __forceinline__ void split4(const Sp& sp, const T (&a)[4], int e, __nv_bfloat16* out,
                                       int64_t plane) {
    typename Sp::template State<S, T> u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) u[i] = sp.template init<S>(a[i], e);
    split4_planes(sp, u, reinterpret_cast<uint2*>(out), plane >> 2,
                  std::make_integer_sequence<int, S>());
}

// A (R x K, row-major) -> out[p][r][k] (row stride kpad, zero beyond K); each
// thread handles two consecutive k.
template <typename T, int S, typename Sp>
__global__ void split_rows_kernel(const T* __restrict__ X, int64_t R, int64_t K,
                                  int64_t ldx, const int32_t* __restrict__ e,
                                  __nv_bfloat16* __restrict__ out, int64_t kpad, const Sp sp) {
    const int64_t half = kpad >> 1;
    const int64_t total = R * half;
    const int64_t plane = R * kpad;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = idx / half;
        const int64_t k = (idx - r * half) * 2;
        const int er = e[r];
        split2<S>(sp, k < K ? __ldg(X + r * ldx + k) : T(0),
                  k + 1 < K ? __ldg(X + r * ldx + k + 1) : T(0), er, out + r * kpad + k, plane);
    }
}

// As split_rows_kernel with four consecutive k per thread: rows from
// blockIdx.y (grid stride, no division per element), two 16-byte loads of A
// when its row is 16-byte aligned, one 8-byte store per digit plane.  Needs
// out 8-byte aligned (the launch checks).  THREADS and MINB are the launch's
// block size and the blocks per SM its register budget must allow.
template <typename T, int S, typename Sp, int THREADS = 256, int MINB = 1>
__global__ void __launch_bounds__(THREADS, MINB) split_rows4_kernel(const T* __restrict__ X, int64_t R,
                                                          int64_t K, int64_t ldx,
                                                          const int32_t* __restrict__ e,
                                                          __nv_bfloat16* __restrict__ out,
                                                          int64_t kpad, const Sp sp) {
    const int64_t plane = R * kpad;
    for (int64_t r = blockIdx.y; r < R; r += gridDim.y) {
        const int er = e[r];
        const T* xr = X + r * ldx;
        const bool xvec = (reinterpret_cast<uintptr_t>(xr) & 15) == 0;
        for (int64_t k = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x); k < kpad;
             k += 4 * (int64_t)gridDim.x * blockDim.x) {
            T a[4];
            if (xvec && k + 3 < K) {
                if constexpr (sizeof(T) == 8) {
                    const double2 p0 = __ldg(reinterpret_cast<const double2*>(xr + k));
                    const double2 p1 = __ldg(reinterpret_cast<const double2*>(xr + k + 2));
                    a[0] = p0.x;
                    a[1] = p0.y;
                    a[2] = p1.x;
                    a[3] = p1.y;
                } else {
                    const float4 p0 = __ldg(reinterpret_cast<const float4*>(xr + k));
                    a[0] = p0.x;
                    a[1] = p0.y;
                    a[2] = p0.z;
                    a[3] = p0.w;
                }
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) a[u] = k + u < K ? __ldg(xr + k + u) : T(0);
            }
            split4<S>(sp, a, er, out + r * kpad + k, plane);
        }
    }
}

// The row exponent scan and split_rows4_kernel in one kernel, one block per
// row at a time (double operands): pass 1 reads the row in the split's own
// pattern for the largest magnitude (the block's maximum through one shared
// slot per row parity, one barrier per row), which gives e_r (stored, and an
// Inf/NaN recorded in the error word as the scan does); pass 2 splits the row
// with it, its loads served by L2.  Needs out 8-byte aligned and kpad a
// multiple of 4 (the launch checks).
template <int S, typename Sp, int THREADS, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) scan_split_rows4_kernel(
    const double* __restrict__ X, int64_t R, int64_t K, int64_t ldx, int32_t* __restrict__ e,
    __nv_bfloat16* __restrict__ out, int64_t kpad, const Sp sp, int* err) {
    __shared__ uint64_t red[2][THREADS / 32];
    const int64_t plane = R * kpad;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int par = 0;
    for (int64_t r = blockIdx.x; r < R; r += gridDim.x, par ^= 1) {
        const double* xr = X + r * ldx;
        const bool xvec = (reinterpret_cast<uintptr_t>(xr) & 15) == 0;
        uint64_t mx = 0;
        // four strides of the row per iteration, all their loads issued
        // before the first comparison (the scan is bound by load latency)
#pragma unroll 1
        for (int64_t k0 = 4 * (int64_t)threadIdx.x; k0 < K; k0 += 16 * THREADS) {
            uint64_t b[16];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int64_t k = k0 + (int64_t)q * 4 * THREADS;
                if (xvec && k + 3 < K) {
                    const uint4 p0 = __ldg(reinterpret_cast<const uint4*>(xr + k));
                    const uint4 p1 = __ldg(reinterpret_cast<const uint4*>(xr + k + 2));
                    b[4 * q] = ((uint64_t)p0.y << 32) | p0.x;
                    b[4 * q + 1] = ((uint64_t)p0.w << 32) | p0.z;
                    b[4 * q + 2] = ((uint64_t)p1.y << 32) | p1.x;
                    b[4 * q + 3] = ((uint64_t)p1.w << 32) | p1.z;
                } else {
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        b[4 * q + u] =
                            k + u < K ? (uint64_t)__double_as_longlong(__ldg(xr + k + u)) : 0ull;
                }
            }
#pragma unroll
            for (int u = 0; u < 16; ++u) {
                const uint64_t a = b[u] & 0x7FFFFFFFFFFFFFFFull;
                mx = a > mx ? a : mx;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const uint64_t y = __shfl_xor_sync(0xffffffffu, mx, o);
            mx = y > mx ? y : mx;
        }
        if (lane == 0) red[par][warp] = mx;
        __syncthreads();
        mx = red[par][0];
#pragma unroll
        for (int w = 1; w < THREADS / 32; ++w) mx = red[par][w] > mx ? red[par][w] : mx;
        const int er = frexp_exponent_of_bits(mx);
        if (threadIdx.x == 0) {
            e[r] = er;
            if (mx >= 0x7FF0000000000000ull) set_device_error(err, ALP_ERR_UNSUPPORTED);
        }
        // the split: the next stride's four values loaded before this
        // stride's residues are formed (the row comes back from L2)
        auto load4 = [&](int64_t k, double (&a)[4]) {
            if (xvec && k + 3 < K) {
                const double2 p0 = __ldg(reinterpret_cast<const double2*>(xr + k));
                const double2 p1 = __ldg(reinterpret_cast<const double2*>(xr + k + 2));
                a[0] = p0.x;
                a[1] = p0.y;
                a[2] = p1.x;
                a[3] = p1.y;
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) a[u] = k + u < K ? __ldg(xr + k + u) : 0.0;
            }
        };
        double an[4];
        if (4 * (int64_t)threadIdx.x < kpad) load4(4 * (int64_t)threadIdx.x, an);
#pragma unroll 1
        for (int64_t k = 4 * (int64_t)threadIdx.x; k < kpad; k += 4 * THREADS) {
            const double a[4] = {an[0], an[1], an[2], an[3]};
            if (k + 4 * THREADS < kpad) load4(k + 4 * THREADS, an);
            split4<S>(sp, a, er, out + r * kpad + k, plane);
        }
    }
}

// B (K x N, row-major) -> out[p][j][k] (row stride kpad): 64 x 32 tiles through
// shared memory so that reads run along j and writes along k.
template <typename T, int S, typename Sp>
__global__ void split_cols_kernel(const T* __restrict__ X, int64_t K, int64_t N,
                                  int64_t ldx, const int32_t* __restrict__ f,
                                  __nv_bfloat16* __restrict__ out, int64_t kpad, const Sp sp) {
    __shared__ T t[32][65];
    const int64_t j0 = (int64_t)blockIdx.x * 32, k0 = (int64_t)blockIdx.y * 64;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 8 warps
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int64_t k = k0 + ty + 8 * r, j = j0 + tx;
        t[tx][ty + 8 * r] = (k < K && j < N) ? __ldg(X + k * ldx + j) : T(0);
    }
    __syncthreads();
    const int64_t plane = N * kpad;
#pragma unroll
    for (int jj = ty; jj < 32; jj += 8) {
        const int64_t j = j0 + jj;
        if (j >= N) continue;
        const int fj = f[j];
        const int64_t k = k0 + 2 * tx;
        if (k >= kpad) continue;
        split2<S>(sp, t[jj][2 * tx], t[jj][2 * tx + 1], fj, out + j * kpad + k, plane);
    }
}

// As split_cols_kernel with four consecutive k per thread: 128 x 32 tiles, the
// tile row of column jj holding k = 4q + i at position 32 i + q (q < 32, i <
// 4), so that the tile's fill (one k of 32 columns per warp, a row stride of
// 129 elements) and the reads of four consecutive k by each lane (32
// consecutive elements per access) are free of bank conflicts; one 8-byte store
// per digit plane (256 contiguous bytes per warp).  Needs out 8-byte aligned
// and kpad a multiple of 4 (the launch checks).
template <typename T, int S, typename Sp>
__global__ void __launch_bounds__(256, 4) split_cols4_kernel(
    const T* __restrict__ X, int64_t K, int64_t N, int64_t ldx, const int32_t* __restrict__ f,
    __nv_bfloat16* __restrict__ out, int64_t kpad, const Sp sp) {
    __shared__ T t[32][129];
    const int64_t j0 = (int64_t)blockIdx.x * 32, k0 = (int64_t)blockIdx.y * 128;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 8 warps
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int kk = ty + 8 * r;
        const int64_t k = k0 + kk, j = j0 + tx;
        t[tx][(kk & 3) * 32 + (kk >> 2)] = (k < K && j < N) ? __ldg(X + k * ldx + j) : T(0);
    }
    __syncthreads();
    const int64_t plane = N * kpad;
    const int64_t k = k0 + 4 * tx;
    if (k >= kpad) return;
#pragma unroll 1
    for (int jj = ty; jj < 32; jj += 8) {
        const int64_t j = j0 + jj;
        if (j >= N) break;
        const int fj = f[j];
        const T a[4] = {t[jj][tx], t[jj][32 + tx], t[jj][64 + tx], t[jj][96 + tx]};
        split4<S>(sp, a, fj, out + j * kpad + k, plane);
    }
}

// Whether the columns of an R-line operand go through split_cols4_kernel's 128-k
// tiles rather than split_cols_kernel's of 64: not where a half empty last tile
// is a fifteenth or more of them, nor where they leave SMs idle (us, 128 and 64;
// lines x kpad).  Eight 7-bit digits: 65536 x 64 43.6 and 29.3, x 192 82.7 and 72.3,
// x 320 122 and 113, x 256 86.7 and 90.8, 8192^2 298 and 320, 512^2 10.9 and 8.8; 15
// moduli: 65536 x 64 51.8 and 35.5, x 256 107 and 115; float, 3 digits: 65536 x 64 19.1
// and 15.0, x 128 23.2 and 25.2.
inline bool split_cols_by_128(int64_t R, int64_t kpad, int sms) {
    if (kpad % 128 != 0 && kpad < 1024) return false;
    return (R + 31) / 32 * ((kpad + 127) / 128) >= 4 * (int64_t)sms;
}

// Nearest double (ties to even) of the 128-bit two's-complement integer
// hi:lo, multiplied by 2^E: built from 32-bit integer operations on the IEEE
// encoding (FP64 arithmetic is slow on this GPU).  The magnitude's top 64 bits
// are brought to T by one word selection and funnel shifts, its lower bits into
// T's last bit, T is rounded at bit 11, and the exponent is added to the
// mantissa, whose carry then raises it.  Below 2^64 (a rare cancellation, or
// zero) the low half is moved up first.  When the scaled result would leave the
// normal range it falls back to ldexp of the rounded value (which rounds a
// subnormal result a second time, as the definition does).  (With 64-bit
// selects and shifts, and the carry pass of crt_rec.cuh in signed 64-bit
// subtractions, the modular reconstruction of 2048^2 with 15 moduli took 43 us;
// now 36.6.)
__device__ __forceinline__ double i128_scaled_to_double_rn(int64_t hi_s, uint64_t lo, int E) {
    // magnitude: (x XOR s) - s with s = 0 or all ones, a 128-bit subtraction
    const uint32_t sgn = (uint32_t)(hi_s >> 63);
    uint32_t w3 = (uint32_t)((uint64_t)hi_s >> 32) ^ sgn, w2 = (uint32_t)hi_s ^ sgn;
    uint32_t w1 = (uint32_t)(lo >> 32) ^ sgn, w0 = (uint32_t)lo ^ sgn;
    asm("sub.cc.u32 %0, %0, %4;\n\tsubc.cc.u32 %1, %1, %4;\n\tsubc.cc.u32 %2, %2, %4;\n\t"
        "subc.u32 %3, %3, %4;"
        : "+r"(w0), "+r"(w1), "+r"(w2), "+r"(w3)
        : "r"(sgn));
    int msb = 127;
    if ((w3 | w2) == 0) {
        if ((w1 | w0) == 0) return 0.0;
        w3 = w1;
        w2 = w0;
        w1 = w0 = 0;
        msb = 63;
    }
    if (w3 == 0) {   // selected, not branched on
        w3 = w2;
        w2 = w1;
        w1 = w0;
        w0 = 0;
        msb -= 32;
    }
    const int sh = __clz((int)w3);
    uint32_t T1 = __funnelshift_l(w2, w3, sh), T0 = __funnelshift_l(w1, w2, sh);
    const uint32_t rest = __funnelshift_l(w0, w1, sh) | (w0 << sh);
    T0 |= min(rest, 1u);
    uint32_t carry;
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, 0;\n\taddc.u32 %2, 0, 0;"
        : "+r"(T0), "+r"(T1), "=r"(carry)
        : "r"(0x3FFu + ((T0 >> 11) & 1u)));
    const uint32_t mlo = __funnelshift_r(T0, T1, 11), mhi = (T1 >> 11) | (carry << 21);
    msb -= sh;
    // the mantissa's leading one (bit 52; 53 after a carry) adds one to the field
    const int field = msb + E + 1022;
    if ((unsigned)field < 2046u)
        return __hiloint2double((int)((sgn & 0x80000000u) | (mhi + ((uint32_t)field << 20))),
                                (int)mlo);
    const double v = __hiloint2double(
        (int)((sgn & 0x80000000u) | (mhi + ((uint32_t)(msb + 1022) << 20))), (int)mlo);
    return ldexp(v, E);
}

}  // namespace alp
