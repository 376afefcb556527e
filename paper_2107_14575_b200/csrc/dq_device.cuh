// Device-side arithmetic of the quantizer: the Philox4x32-10 block function,
// the per-element encoder of Eq. 5/6, the register bit packer and the in-place
// decoder of the average.  All of it is written for a thread that owns one
// 32-element group, so that every shift and word index is a compile-time
// constant once B (bits per code) is known.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "dq_common.cuh"

// Round keys of Philox4x32-10: key + r * (0x9E3779B9, 0xBB67AE85).  They are the
// same for the whole grid, so the host computes them and they travel as kernel
// arguments (constant bank), which keeps them out of the register file.
struct PhiloxKeys {
    uint32_t k0[10];
    uint32_t k1[10];
};

inline PhiloxKeys make_philox_keys(uint64_t seed)
{
    PhiloxKeys k;
    uint32_t a = (uint32_t)seed, b = (uint32_t)(seed >> 32);
    for (int r = 0; r < 10; ++r) {
        k.k0[r] = a;
        k.k1[r] = b;
        a += 0x9E3779B9u;
        b += 0xBB67AE85u;
    }
    return k;
}

#ifdef __CUDACC__

// Philox4x32-10 blocks (Salmon et al., SC'11): ten rounds of two 32x32->64 multiplies and a three-way
// xor with the counter words and the round key.  N blocks side by side, in place; FIRST: rounds already done.
constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;
template <int FIRST, int N>
__device__ __forceinline__ void philox_rounds(uint32_t (&c)[N][4], const PhiloxKeys& K)
{
#pragma unroll
    for (int r = FIRST; r < 10; ++r) {
#pragma unroll
        for (int n = 0; n < N; ++n) {
            const uint64_t p0 = (uint64_t)kPhiloxM0 * c[n][0];
            const uint64_t p1 = (uint64_t)kPhiloxM1 * c[n][2];
            c[n][0] = (uint32_t)(p1 >> 32) ^ c[n][1] ^ K.k0[r];
            c[n][2] = (uint32_t)(p0 >> 32) ^ c[n][3] ^ K.k1[r];
            c[n][1] = (uint32_t)p1;
            c[n][3] = (uint32_t)p0;
        }
    }
}

// The first two rounds of the block with the counter (octet, 0, worker, step): of their four multiplies two
// depend on the octet alone and two on the worker alone.  What is left of them is an xor for two of the words.
struct OctetRounds { uint32_t a, b, c; };
__device__ __forceinline__ OctetRounds octet_rounds(const uint32_t octet, const uint32_t step, const PhiloxKeys& K)
{
    const uint64_t p0 = (uint64_t)kPhiloxM0 * octet;
    const uint64_t p1 = (uint64_t)kPhiloxM1 * ((uint32_t)(p0 >> 32) ^ step ^ K.k1[0]);
    return {(uint32_t)(p1 >> 32), (uint32_t)p0, (uint32_t)p1};
}
__device__ __forceinline__ uint4 worker_rounds(const uint32_t worker, const PhiloxKeys& K)        // (w: not used)
{
    const uint64_t p1 = (uint64_t)kPhiloxM1 * worker;
    const uint64_t p0 = (uint64_t)kPhiloxM0 * ((uint32_t)(p1 >> 32) ^ K.k0[0]);
    return make_uint4((uint32_t)p1 ^ K.k0[1], (uint32_t)(p0 >> 32) ^ K.k1[1], (uint32_t)p0, 0u);
}
__device__ __forceinline__ void third_round(uint32_t (&c)[4], const OctetRounds& o, const uint4& w)
{
    c[0] = o.a ^ w.x;
    c[1] = o.c;
    c[2] = o.b ^ w.y;
    c[3] = w.z;
}

// The three places where the members of the l_p family differ.  P = DQ_NORM_L2: sum of
// squares, square root at the end.  P = DQ_NORM_LINF: running maximum of the magnitudes
// (max.NaN, so that a NaN entry is not skipped and reaches the status word), nothing at the end.
__device__ __forceinline__ float max_nan(const float a, const float b)
{
    float d;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}
// largest magnitude of three, by one instruction
__device__ __forceinline__ float max_magnitude(const float a, const float b, const float c)
{
    float d;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
template <int P>
__device__ __forceinline__ float take(const float acc, const float x)
{
    if constexpr (P == DQ_NORM_L2) return fmaf(x, x, acc);
    else return max_nan(acc, fabsf(x));
}
template <int P>
__device__ __forceinline__ float join(const float a, const float b)
{
    if constexpr (P == DQ_NORM_L2) return a + b;
    else return max_nan(a, b);
}
template <int P>
__device__ __forceinline__ float finish(const float a)
{
    if constexpr (P == DQ_NORM_L2) return sqrtf(a);
    else return a;
}

// ---- l2 norms of buckets whose squares leave the fp32 range ---------------------------------
// The sum of squares S of a bucket, accumulated with fused multiply-adds, is taken as it is when
// 2^-100 <= S < inf: no square overflowed, every term that fell into the subnormal range (or
// vanished) is below 2^-126 and so below 2^-26 of S, and sqrt(S) >= 2^-50 dominates each of
// those entries while sqrt(fl(g^2)) = |g| for the others.  Outside that range (a bucket of tiny
// entries, an overflowed square, a NaN) the bucket is reduced again: first its largest magnitude
// (exact), then the squares of the entries scaled by the power of two that brings that magnitude
// into [1, 2), in the same order as before, and the square root is scaled back.  The functors
// below are those two reductions; the kernels supply the loads and the joins between threads.
__device__ __forceinline__ bool l2_sum_in_range(const float sum)
{
    return sum >= 0x1p-100f && sum <= 3.402823466e38f;       // false for a NaN as well
}
struct MaxMagnitude {
    __device__ __forceinline__ float take(const float acc, const float x) const { return max_nan(acc, fabsf(x)); }
    __device__ __forceinline__ float join(const float a, const float b) const { return max_nan(a, b); }
};
struct ScaledSquares {
    int e;                          // the entries are multiplied by 2^-e first (exact, or negligible when it underflows)
    __device__ __forceinline__ float take(const float acc, const float x) const
    {
        const float y = scalbnf(x, -e);
        return fmaf(y, y, acc);
    }
    __device__ __forceinline__ float join(const float a, const float b) const { return a + b; }
};
// Exponent to scale by, from the bucket's largest magnitude (0 when there is nothing to scale:
// an all-zero bucket, an infinity or a NaN, for which rescaled_l2 returns the magnitude itself).
__device__ __forceinline__ bool magnitude_scalable(const float mx) { return mx > 0.0f && mx <= 3.402823466e38f; }
__device__ __forceinline__ int scale_exponent(const float mx) { return magnitude_scalable(mx) ? ilogbf(mx) : 0; }
// The norm from the largest magnitude and the scaled sum of squares.  An overflow of the
// result (entries near the top of the fp32 range) gives infinity, as the fp64 definition
// rounded to fp32 does.
__device__ __forceinline__ float rescaled_l2(const float mx, const float scaled_sum, const int e)
{
    if (!magnitude_scalable(mx)) return mx;                  // 0, infinity or NaN
    return scalbnf(sqrtf(scaled_sum), e);
}

// (a & mask) | c as one three-input logic operation.  `c` must come from a register the
// compiler cannot fold (callers pass the exponent pattern of 2^23 from a kernel
// argument), otherwise two immediates would cost two instructions.
__device__ __forceinline__ uint32_t and_or(const uint32_t a, const uint32_t mask, const uint32_t c)
{
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(a), "r"(mask), "r"(c));
    return d;
}

// Two fp32 values in one 64-bit register pair, for the packed two-lane forms of sm_100
// (add.f32x2, mul.f32x2, fma.f32x2).
__device__ __forceinline__ uint64_t pack_pair(const uint32_t lo, const uint32_t hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ void unpack_pair(const uint64_t v, float& lo, float& hi)
{
    uint32_t a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(v));
    lo = __uint_as_float(a);
    hi = __uint_as_float(b);
}
__device__ __forceinline__ uint64_t add_pair(const uint64_t a, const uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma_pair(const uint64_t a, const uint64_t b, const uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t mul_pair_rz(const uint64_t a, const uint64_t b)
{
    uint64_t r;
    asm("mul.rz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t add_pair_rm(const uint64_t a, const uint64_t b)
{
    uint64_t r;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// the same number in both lanes of a pair
__host__ __device__ constexpr uint64_t both(const uint32_t bits) { return (uint64_t)bits << 32 | bits; }
// bits of the float n + 2^p for 0 <= n < 2^p, p <= 23 (n an integer)
__host__ __device__ constexpr uint32_t float_bits(const uint32_t n, const int p)
{
    return (uint32_t)(127 + p) << 23 | n << (23 - p);
}

// inv = RZ(s / norm), the scale of Eq. 5 rounded toward zero (0 for norm < 2^-100, where the
// quotient could overflow, and for a NaN norm).  Written out instead of calling the library's
// division so that it stays inline: reciprocal estimate r (relative error <= 2^-23), q = s * r,
// one Newton step q <- q + (s - q * norm) * r, which brings q to within 2^-44 of the quotient
// before its rounding, i.e. to one of the two floats that enclose s / norm; the sign of the
// exactly rounded residual s - q * norm then tells which, and the upper one steps down an ulp.
// Norms above 2^125, whose reciprocal estimate would be flushed to zero, take the library route.
__device__ __forceinline__ float inv_scale_normal(const float sf, const float norm)      // 2^-100 <= norm <= 2^125
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(norm));
    float q = __fmul_rn(sf, r);
    q = __fmaf_rn(__fmaf_rn(-q, norm, sf), r, q);
    const float e = __fmaf_rn(-q, norm, sf);
    return __uint_as_float(__float_as_uint(q) - (e < 0.0f ? 1u : 0u));
}
__device__ __forceinline__ bool norm_is_plain(const float norm) { return norm >= 0x1p-100f && norm <= 0x1p125f; }
__device__ __forceinline__ float inv_scale(const float sf, const float norm)
{
    if (!(norm >= 0x1p-100f)) return 0.0f;
    if (norm > 0x1p125f) return __fdiv_rz(sf, norm);
    return inv_scale_normal(sf, norm);
}
// the correctly rounded square root, for a result that counts only where the argument is in range
// (see l2_sum_in_range): the flushing form has no subnormal arguments to take care of
__device__ __forceinline__ float sqrt_normal(const float x)
{
    float r;
    asm("sqrt.rn.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Appends W bits at position BIT of a group's little-endian bit string of N words.  `cur` is a
// shift register: a funnel shift pushes the bits in at the top, so after 32 bits the first of them
// sits at bit 0 and the word is complete.  Bits that straddle two words finish the current word with
// their low part and seed the next one with themselves at the top; the surplus low bits fall off as
// that word fills up.  What stands above bit W-1 of `bits` never reaches a word.
template <int BIT, int W, int N>
__device__ __forceinline__ void push_bits(uint32_t (&acc)[N], uint32_t& cur, const uint32_t bits)
{
    constexpr int w = BIT >> 5;
    constexpr int sh = BIT & 31;
    constexpr int end = sh + W;
    if constexpr (end < 32) {
        if constexpr (sh == 0) cur = bits << (32 - W);
        else cur = __funnelshift_r(cur, bits, W);
    } else if constexpr (end == 32) {
        if constexpr (sh == 0) acc[w] = bits;
        else acc[w] = __funnelshift_r(cur, bits, W);
    } else {
        acc[w] = __funnelshift_r(cur, bits, 32 - sh);
        cur = bits << (32 - W);
    }
}

// The B words of a group whose 32 codes all equal s: what a zero scale gives (x = 0 and
// floor(0 + v) = 0 for every draw v in (0, 1)), so such a group needs neither uniforms nor
// arithmetic.  Everything here folds to constants.
template <int B, int E>
struct PushSame {
    static __device__ __forceinline__ void run(uint32_t (&acc)[B], uint32_t& cur, const uint32_t code)
    {
        push_bits<E * B, B>(acc, cur, code);
        PushSame<B, E + 1>::run(acc, cur, code);
    }
};
template <int B>
struct PushSame<B, 32> {
    static __device__ __forceinline__ void run(uint32_t (&)[B], uint32_t&, const uint32_t) {}
};
template <int B>
__device__ __forceinline__ void zero_group_words(uint32_t (&acc)[B])
{
    uint32_t cur = 0;
    PushSame<B, 0>::run(acc, cur, (1u << (B - 1)) - 1u);
}

// ---- Eq. 5/6 for the 32 elements of a group, two at a time ----------------------------------
// With x = RZ(g * inv), inv = RZ(s / norm), the element's position on the level grid and
// v = (2k + 1) / 2^17 its uniform draw (k a 16-bit half of a Philox word), the code is
// floor(x + v) + s: for either sign the neighbour of x away from zero is taken with probability
// frac(|x|), Eq. 6.
//  * Both roundings are toward zero, so |x| <= s whenever |g| <= norm (a bucket's norm dominates its
//    entries): no clamp, no absolute value, no sign handling.
//  * A byte permute puts k under the upper half of the float 128 + c (c an integer): that float is
//    K = 128 + c + k / 2^16, one instruction for draw, shift and exponent.
//  * s <= 63 (b <= 7): with c = s the sum x + K lies in [128, 256), where floats are multiples of
//    2^-16, and t = RN(x + K) has floor(x + v) + s as its integer part.  Rounding to nearest adds the
//    half step 2^-17 that K lacks: the integer n is reached if and only if x + k / 2^16 >= n - 2^-17,
//    a tie at the integer itself included (it goes to the even neighbour, and n is a multiple of 2^16
//    steps).  The code stands in bits 16..22 of t.
//  * Larger s: the half step is added first, y = RD(x + 2^-17), then RD(y + K).  An addition rounded
//    down never crosses a representable number downwards, and the numbers x + 2^-17 is compared with,
//    n - k / 2^16, are representable where |x| < 128; from there on x itself is a multiple of 2^-16,
//    and y = x compares with them as x + 2^-17 does.
//  * RD(t + (1.5 * 2^23 - 128)) drops the fraction: its low bits are the code, and subtracting
//    1.5 * 2^23 + s leaves the signed level, exactly, for the average.
// The packed two-lane forms halve the instructions issued (the kernels are bound by issue, not by
// the lanes): 5.5 per element at b = 4 with its share of the average, against 6 for the code alone in
// scalar form.

// two Philox halves -> K for elements 2i and 2i + 1
__device__ __forceinline__ uint64_t draw_pair(const uint32_t w, const uint32_t base)
{
    return pack_pair(__byte_perm(w, base, 0x7610), __byte_perm(w, base, 0x7632));
}
// codes of two t's (bits 16..22 of each) as one word, 16 bits apart, everything else zero: the top
// byte of t, 0x43, is replaced by copies of its sign
__device__ __forceinline__ uint32_t code_halves(const uint32_t ta, const uint32_t tb)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, 0xF6B2;" : "=r"(r) : "r"(ta), "r"(tb));
    return r;
}
__device__ __forceinline__ void split_pair(const uint64_t v, uint32_t& lo, uint32_t& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(v));
}

// Appends the codes of elements 8C .. 8C + 7 to the group's words.  t: for b <= 7 the float with the
// code in bits 16..22; u: the float with the code in its low bits (not formed where t is enough).
template <int B>
struct PacksFromT {
    static constexpr bool value = B <= 4;
};
template <int B, int C>
__device__ __forceinline__ void pack_eight(uint32_t (&words)[B], uint32_t& cur, const uint32_t (&t)[8], const uint32_t (&u)[8])
{
    if constexpr (B <= 4) {
        // halves of q: the codes of elements 0..3 and of 4..7, 4 * B bits each
        const uint32_t q = (((code_halves(t[3], t[7]) << B) + code_halves(t[2], t[6]) << B) + code_halves(t[1], t[5]) << B) +
                           code_halves(t[0], t[4]);
        if constexpr (B == 4) {
            words[C] = q;
        } else if constexpr (B == 3) {
            push_bits<24 * C, 24>(words, cur, (q & 0xFFFu) | ((q >> 4) & 0xFFF000u));
        } else {
            if constexpr (C % 2 == 0) cur = q;
            else words[C / 2] = __byte_perm(cur, q, 0x6420);
        }
    } else if constexpr (B == 8) {
        words[2 * C] = __byte_perm(__byte_perm(u[0], u[1], 0x0040), __byte_perm(u[2], u[3], 0x0040), 0x5410);
        words[2 * C + 1] = __byte_perm(__byte_perm(u[4], u[5], 0x0040), __byte_perm(u[6], u[7], 0x0040), 0x5410);
    } else if constexpr (B == 16) {
#pragma unroll
        for (int i = 0; i < 4; ++i) words[4 * C + i] = __byte_perm(u[2 * i], u[2 * i + 1], 0x5410);
    } else {
        push_bits<(8 * C + 0) * B, B>(words, cur, u[0]);
        push_bits<(8 * C + 1) * B, B>(words, cur, u[1]);
        push_bits<(8 * C + 2) * B, B>(words, cur, u[2]);
        push_bits<(8 * C + 3) * B, B>(words, cur, u[3]);
        push_bits<(8 * C + 4) * B, B>(words, cur, u[4]);
        push_bits<(8 * C + 5) * B, B>(words, cur, u[5]);
        push_bits<(8 * C + 6) * B, B>(words, cur, u[6]);
        push_bits<(8 * C + 7) * B, B>(words, cur, u[7]);
    }
}

// Eight elements and the four words drawn for them: t, u as pack_eight takes them; with AVG, level * scale is added
// to their sums.
template <int B, bool AVG>
__device__ __forceinline__ void octet_codes(const ulonglong2 lo, const ulonglong2 hi, const uint64_t inv2, const uint64_t scale2,
                                            uint64_t* sums, const uint32_t (&w)[4], uint32_t (&t)[8], uint32_t (&u)[8])
{
    constexpr uint32_t s = (1u << (B - 1)) - 1u;
    const uint64_t x[4] = {lo.x, lo.y, hi.x, hi.y};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint64_t pos = mul_pair_rz(x[i], inv2);
        uint64_t t2;
        if constexpr (B <= 7) t2 = add_pair(pos, draw_pair(w[i], float_bits(s, 7)));
        else t2 = add_pair_rm(add_pair_rm(pos, both(0x37000000u)), draw_pair(w[i], float_bits(0, 7)));     // 2^-17
        if constexpr (B <= 7) split_pair(t2, t[2 * i], t[2 * i + 1]);
        if constexpr (AVG || !PacksFromT<B>::value) {
            // 1.5 * 2^23 + code: t carries 128 + s (b <= 7) or 128
            constexpr uint32_t kTo = 0x4B400000u - 128u + (B <= 7 ? 0u : s);
            const uint64_t u2 = add_pair_rm(t2, both(kTo));
            split_pair(u2, u[2 * i], u[2 * i + 1]);
            if constexpr (AVG) {
                const uint64_t level = add_pair(u2, both(0xCB400000u + s));
                sums[i] = fma_pair(level, scale2, sums[i]);
            }
        }
    }
}

// Elements 8C .. 8C + 7 of a group (one Philox block).
template <int B, int C, bool AVG>
__device__ __forceinline__ void encode_eight(const ulonglong2 lo, const ulonglong2 hi, const uint64_t inv2, const uint64_t scale2,
                                             uint64_t (&acc2)[16], uint32_t (&words)[B], uint32_t& cur, const uint32_t q,
                                             const uint32_t worker, const uint32_t step, const PhiloxKeys& keys)
{
    uint32_t w[1][4] = {{q, 0u, worker, step}}, t[8], u[8];
    philox_rounds<0>(w, keys);
    octet_codes<B, AVG>(lo, hi, inv2, scale2, acc2 + 4 * C, w[0], t, u);
    pack_eight<B, C>(words, cur, t, u);
}

// A whole group; quad(c) gives elements 4c .. 4c + 3.
template <int B, bool AVG, class Quads>
__device__ __forceinline__ void encode_row(const Quads& quad, const uint64_t inv2, const uint64_t scale2,
                                           uint64_t (&acc2)[16], uint32_t (&words)[B], const uint32_t q0, const uint32_t worker,
                                           const uint32_t step, const PhiloxKeys& keys)
{
    uint32_t cur = 0;
    encode_eight<B, 0, AVG>(quad(0), quad(1), inv2, scale2, acc2, words, cur, q0 + 0u, worker, step, keys);
    encode_eight<B, 1, AVG>(quad(2), quad(3), inv2, scale2, acc2, words, cur, q0 + 1u, worker, step, keys);
    encode_eight<B, 2, AVG>(quad(4), quad(5), inv2, scale2, acc2, words, cur, q0 + 2u, worker, step, keys);
    encode_eight<B, 3, AVG>(quad(6), quad(7), inv2, scale2, acc2, words, cur, q0 + 3u, worker, step, keys);
}

// ---- global memory, 32 bytes at a time ----
__device__ __forceinline__ void load_wide(const float* p, float (&r)[8])
{
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
                 : "l"(p)
                 : "memory");
}
__device__ __forceinline__ void store_wide_bits(void* p, const uint32_t (&r)[8], const void* base, const int64_t extent, int32_t* status)
{
#ifdef DQ_CHECKED
    if (!dq_store_allowed(p, 32, base, extent, status)) return;
#else
    (void)base; (void)extent; (void)status;
#endif
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]),
                 "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
__device__ __forceinline__ void store_wide(float* p, const float (&r)[8], const void* base, const int64_t extent, int32_t* status)
{
    uint32_t v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __float_as_uint(r[i]);
    store_wide_bits(p, v, base, extent, status);
}

// The 128-byte row of sums (or the update of the parameters there), straight from registers: a lane's
// row is four whole sectors, and it happens once per tile and M workers.
__device__ __forceinline__ void store_row(float* dst, const float (&r)[32], const bool update, const float neg_lr, const bool wide,
                                          const void* base, const int64_t extent, int32_t* status)
{
    if (wide) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float y[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) y[e] = r[8 * i + e];
            if (update) {
                float p[8];
                load_wide(dst + 8 * i, p);
#pragma unroll
                for (int e = 0; e < 8; ++e) y[e] = fmaf(neg_lr, y[e], p[e]);
            }
            store_wide(dst + 8 * i, y, base, extent, status);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float4 y = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
            if (update) {
                const float4 p = *reinterpret_cast<const float4*>(dst + 4 * i);
                y = make_float4(fmaf(neg_lr, y.x, p.x), fmaf(neg_lr, y.y, p.y), fmaf(neg_lr, y.z, p.z),
                                fmaf(neg_lr, y.w, p.w));
            }
            DQ_STORE(reinterpret_cast<float4*>(dst + 4 * i), y, base, extent, status);
        }
    }
}

// Words that leave straight from registers, by 4-, 8-, 16- or 32-byte stores: a tile's words are one
// contiguous span, the L2 puts partial sectors together, and staging them in shared memory costs some
// sixty instructions a tile.  From nine words on the scattered stores cost more.  Measured, staged / straight
// (us): 2^24 elements M = 32, b = 3 510 / 492, b = 5 515 / 502, b = 6 520 / 510, b = 7 551 / 536, b = 11
// 570 / 597, b = 14 598 / 617, b = 15 613 / 979.  (One bulk copy of the staged words instead of 16-byte
// stores by all lanes: 2 % slower than those.)
template <int B>
struct StoresDirectly {
    static constexpr bool value = B <= 8 || B % 4 == 0;
};
template <int B>
__device__ __forceinline__ void store_words(uint32_t* dst, const uint32_t (&w)[B], const bool wide, const void* base,
                                            const int64_t extent, int32_t* status)
{
    (void)wide;
    if constexpr (B % 2 != 0) {
#pragma unroll
        for (int i = 0; i < B; ++i) DQ_STORE(dst + i, w[i], base, extent, status);
    } else if constexpr (B % 4 != 0) {
#pragma unroll
        for (int i = 0; i < B / 2; ++i) DQ_STORE(reinterpret_cast<uint2*>(dst) + i, make_uint2(w[2 * i], w[2 * i + 1]), base, extent, status);
    } else {
        if constexpr (B % 8 == 0) {
            if (wide) {                          // 32-byte stores: whole sectors from one lane
#pragma unroll
                for (int i = 0; i < B / 8; ++i) {
                    uint32_t v[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) v[k] = w[8 * i + k];
                    store_wide_bits(dst + 8 * i, v, base, extent, status);
                }
                return;
            }
        }
#pragma unroll
        for (int i = 0; i < B / 4; ++i)
            DQ_STORE(reinterpret_cast<uint4*>(dst) + i, make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]), base, extent,
                     status);
    }
}

// ---- eight codes of a lane ------------------------------------------------------------------
// The 8 * B bits of an octet, from bit 0 on; what stands above them in the last word is zero.
template <int B>
struct OctetWords {
    static constexpr int n = (8 * B + 31) / 32;
};
template <int B, int E, int N>
__device__ __forceinline__ void push_codes(uint32_t (&w)[N], uint32_t& cur, const uint32_t (&u)[8])
{
    if constexpr (E < 8) {
        push_bits<E * B, B>(w, cur, u[E]);
        push_codes<B, E + 1>(w, cur, u);
    }
}
template <int B>
__device__ __forceinline__ void pack_octet(uint32_t (&w)[OctetWords<B>::n], const uint32_t (&t)[8], const uint32_t (&u)[8])
{
    if constexpr (B == 1) {
        w[0] = 0u;
    } else if constexpr (B <= 4) {
        // halves of q: the codes of elements 0..3 and of 4..7, 4 * B bits each
        const uint32_t q = (((code_halves(t[3], t[7]) << B) + code_halves(t[2], t[6]) << B) + code_halves(t[1], t[5]) << B) +
                           code_halves(t[0], t[4]);
        if constexpr (B == 4) w[0] = q;
        else if constexpr (B == 3) w[0] = (q & 0xFFFu) | ((q >> 4) & 0xFFF000u);
        else w[0] = __byte_perm(q, 0u, 0x4420);
    } else if constexpr (B == 8) {
        w[0] = __byte_perm(__byte_perm(u[0], u[1], 0x0040), __byte_perm(u[2], u[3], 0x0040), 0x5410);
        w[1] = __byte_perm(__byte_perm(u[4], u[5], 0x0040), __byte_perm(u[6], u[7], 0x0040), 0x5410);
    } else if constexpr (B == 16) {
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = __byte_perm(u[2 * i], u[2 * i + 1], 0x5410);
    } else {
        uint32_t cur = 0;
        push_codes<B, 0>(w, cur, u);
        if constexpr (8 * B % 32 != 0) w[OctetWords<B>::n - 1] = cur >> (32 - 8 * B % 32);
    }
}
// ... of eight codes that all equal s
template <int B>
__device__ __forceinline__ void zero_octet_words(uint32_t (&w)[OctetWords<B>::n])
{
    constexpr uint32_t s = (1u << (B - 1)) - 1u;
    uint32_t cur = 0;
    const uint32_t u[8] = {s, s, s, s, s, s, s, s};
    push_codes<B, 0>(w, cur, u);
    if constexpr (8 * B % 32 != 0) w[OctetWords<B>::n - 1] = cur >> (32 - 8 * B % 32);
}
// Octets of 1, 2, 4, 8 or 16 bytes leave straight from registers, neighbouring lanes side by side; the others are
// brought into the order of memory in the warp's own part of a consumed stage and leave a word per lane.
template <int B>
struct OctetDirect {
    static constexpr bool value = (B & (B - 1)) == 0;
};
template <int B>
__device__ __forceinline__ void store_octet(unsigned char* dst, const uint32_t (&w)[OctetWords<B>::n], const void* base,
                                            const int64_t extent, int32_t* status)
{
    if constexpr (B == 1) DQ_STORE(dst, (unsigned char)w[0], base, extent, status);
    else if constexpr (B == 2) DQ_STORE(reinterpret_cast<uint16_t*>(dst), (uint16_t)w[0], base, extent, status);
    else if constexpr (B == 4) DQ_STORE(reinterpret_cast<uint32_t*>(dst), w[0], base, extent, status);
    else if constexpr (B == 8) DQ_STORE(reinterpret_cast<uint2*>(dst), make_uint2(w[0], w[1]), base, extent, status);
    else DQ_STORE(reinterpret_cast<uint4*>(dst), make_uint4(w[0], w[1], w[2], w[3]), base, extent, status);
}
template <int B>
__device__ __forceinline__ void stage_octet(unsigned char* dst, const uint32_t (&w)[OctetWords<B>::n])
{
    if constexpr (B % 4 == 0) {
#pragma unroll
        for (int i = 0; i < B / 4; ++i) reinterpret_cast<uint32_t*>(dst)[i] = w[i];
    } else if constexpr (B % 2 == 0) {
#pragma unroll
        for (int i = 0; i < B / 2; ++i) reinterpret_cast<uint16_t*>(dst)[i] = (uint16_t)(w[i / 2] >> (16 * (i % 2)));
    } else {
#pragma unroll
        for (int i = 0; i < B; ++i) dst[i] = (unsigned char)(w[i / 4] >> (8 * (i % 4)));
    }
}
// Eight sums (or the update of the parameters there).
__device__ __forceinline__ void store_sums(float* dst, const float (&r)[8], const bool update, const float neg_lr, const bool wide,
                                           const void* base, const int64_t extent, int32_t* status)
{
    float y[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) y[e] = r[e];
    if (wide) {
        if (update) {
            float p[8];
            load_wide(dst, p);
#pragma unroll
            for (int e = 0; e < 8; ++e) y[e] = fmaf(neg_lr, y[e], p[e]);
        }
        store_wide(dst, y, base, extent, status);
    } else {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float4 z = make_float4(y[4 * i], y[4 * i + 1], y[4 * i + 2], y[4 * i + 3]);
            if (update) {
                const float4 p = *reinterpret_cast<const float4*>(dst + 4 * i);
                z = make_float4(fmaf(neg_lr, z.x, p.x), fmaf(neg_lr, z.y, p.y), fmaf(neg_lr, z.z, p.z), fmaf(neg_lr, z.w, p.w));
            }
            DQ_STORE(reinterpret_cast<float4*>(dst + 4 * i), z, base, extent, status);
        }
    }
}

// Decoding for the average.  A code holds s + sgn * level.  Its B bits are
// masked out of the word where they stand and OR-ed under the exponent of 2^23:
// that float is 2^23 + code * 2^k, and subtracting 2^23 + s * 2^k leaves
// sgn * level * 2^k exactly -- one logic operation and one add, no shift, no
// int-to-float conversion, no sign handling.  k depends only on the code's
// position E, so the caller removes 2^k once after all workers have been
// accumulated.  Codes that reach above bit 22 of their word are decoded from the
// word's upper half (shifted down by 16 once per word) or, when they straddle
// two words, from a funnel shift.
template <int B, int E>
struct CodePos {
    static constexpr int bit = E * B;
    static constexpr int w = bit >> 5;
    static constexpr int sh = bit & 31;
    static constexpr int end = sh + B;            // one past the code's last bit, counted in word w
    static constexpr bool straddles = end > 32;
    static constexpr bool in_place = !straddles && end <= 23;
    static constexpr bool in_upper = !straddles && !in_place && sh >= 16;
    // power of two the decoded value carries
    static constexpr int k = in_place ? sh : (in_upper ? sh - 16 : 0);
};

// Two neighbouring codes are decoded at once with the packed two-lane fp32 forms of
// sm_100 (add.f32x2, fma.f32x2 on 64-bit register pairs): one packed subtract and one packed FMA
// replace two of each, which halves the operand traffic of the accumulation (the scalar form
// keeps 32 accumulators, a scale and an immediate in flight per code).  Results are bit for bit
// those of scalar subtracts and FMAs: the same exact subtract, the same single rounding in the FMA.

// bits of the float 2^23 + code * 2^k for code E of a group (the part before the subtract)
template <int B, int E>
__device__ __forceinline__ uint32_t code_bits(const uint32_t (&wd)[B], const uint32_t (&hi)[B], const uint32_t magic)
{
    using P = CodePos<B, E>;
    constexpr uint32_t kCode = (1u << B) - 1u;
    if constexpr (P::in_place) return and_or(wd[P::w], kCode << P::k, magic);
    else if constexpr (P::in_upper) return and_or(hi[P::w], kCode << P::k, magic);
    else if constexpr (!P::straddles) return and_or(wd[P::w] >> P::sh, kCode, magic);
    else return and_or(__funnelshift_r(wd[P::w], wd[P::w + 1], P::sh), kCode, magic);
}
// bits of the float -(2^23 + s * 2^k): 2^23 + n has the mantissa n for every integer n < 2^23
template <int B, int E>
struct NegOffsetBits {
    static constexpr uint32_t value = 0xCB000000u + (uint32_t)(((1 << (B - 1)) - 1) << CodePos<B, E>::k);
};
// (sgn * level * 2^k0, sgn * level * 2^k1) of codes 2Q and 2Q + 1 times (scale, scale), added to acc2
template <int B, int Q>
__device__ __forceinline__ uint64_t accumulate_pair(const uint64_t acc2, const uint32_t (&wd)[B], const uint32_t (&hi)[B],
                                                    const uint64_t scale2, const uint32_t magic)
{
    constexpr uint64_t kOff = (uint64_t)NegOffsetBits<B, 2 * Q>::value | ((uint64_t)NegOffsetBits<B, 2 * Q + 1>::value << 32);
    const uint64_t m = pack_pair(code_bits<B, 2 * Q>(wd, hi, magic), code_bits<B, 2 * Q + 1>(wd, hi, magic));
    return fma_pair(add_pair(m, kOff), scale2, acc2);
}

// does any code of word W need the word's upper half?
template <int B, int W, int E = 0>
struct NeedsUpper {
    static constexpr bool value =
        ((CodePos<B, E>::w == W) && CodePos<B, E>::in_upper) || NeedsUpper<B, W, E + 1>::value;
};
template <int B, int W>
struct NeedsUpper<B, W, 32> {
    static constexpr bool value = false;
};

#endif  // __CUDACC__
