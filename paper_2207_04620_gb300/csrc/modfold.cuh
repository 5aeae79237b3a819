// Modular products for primes just below a power of two: q = 2^b - d with 33 <= b <= 60 and a
// small d (the chain takes the largest primes below 2^b, so d is a few hundred multiples of 2N).
//
// A constant w (a twiddle) is held as four 32-bit numbers: the centred residues of w and of
// 2^32 w, each split at bit c = b - 32 into a signed 32-bit head and a centred tail of c bits.
// For a signed 64-bit y = 2^32 yh + yl (yl signed), w y = yl w + yh (2^32 w) mod q is
//
//     2^c (yl w_head + yh v_head) + (yl w_tail + yh v_tail),      v = 2^32 w mod q
//
// four 32x32 -> 64-bit multiply-adds with no carries between them.  The split at b - 32 makes
// the first sum's high word the quotient by 2^b as it stands (2^c times 2^32): with
// A = 2^32 t + a, 2^c A = 2^b t + 2^c a = d t + 2^c a mod q, one more multiply-add.  Five in all,
// against ten multiplications of a Shoup product (y w - floor(y w' / 2^64) q).  The result is
// signed: |r| <= 1.5 2^b + 2^31 d.
//
// Values stay signed and unreduced through several butterflies; fold() brings one back to
// about [0, 2^b) with one multiply-add: v = 2^b h + l = l + d h.  fold_bounds (context.cu) proves for a
// prime that no sum leaves 64 bits and how many folds the final reduction takes; chains with a
// prime outside its range use the Shoup kernels.
#pragma once
#include <cstdint>

namespace hx {

struct FoldPrime {
    uint64_t q;
    int c;         // b - 32
    int d;         // 2^b - q
    int mask;      // 2^c - 1: the high word's bits below 2^b
    int refold;    // != 0: the final reduction folds twice
    int4 n_inv;    // N^-1 mod q as a constant
    int4 n_inv_w1; // N^-1 * psi^-brv(1) mod q: the last inverse stage's twiddle with N^-1 folded in
    int4 r60;      // 2^60 mod q as a constant
    uint32_t q0, q1;  // q's low 30 bits and the rest
    uint32_t minv;    // -q^-1 mod 2^30
};

// bounds in sixteenths of the unit u of a prime (u >= 2^b): a folded value, a product, the limit
constexpr int kFoldSettled = 17, kFoldProduct = 25, kFoldLimit = 127;

#ifdef __CUDACC__
__device__ __forceinline__ int64_t mad_wide(int a, int b, int64_t c)
{
    int64_t r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
__device__ __forceinline__ int64_t mul_wide(int a, int b)
{
    int64_t r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
}

// y w mod q, |result| <= 1.5 2^b + 2^31 d, for |y| < 2^63 - 2^32
__device__ __forceinline__ int64_t fold_mul(int64_t y, const int4 w, const FoldPrime &P)
{
    const int yl = (int)y, yh = (int)(y >> 32) + (int)((unsigned)yl >> 31);
    const int64_t A = mad_wide(yh, w.y, mul_wide(yl, w.x));
    int64_t B = mad_wide(yh, w.w, mul_wide(yl, w.z));
    B = mad_wide((int)(A >> 32), P.d, B);
    return B + (int64_t)((uint64_t)(uint32_t)A << P.c);
}

// v mod q within 2^b + (|v| / 2^b + 1) d, negative by at most the second term
__device__ __forceinline__ int64_t fold(int64_t v, const FoldPrime &P)
{
    const int vh = (int)(v >> 32);
    const int64_t l = (int64_t)(((uint64_t)(uint32_t)(vh & P.mask) << 32) | (uint32_t)v);
    return mad_wide(vh >> P.c, P.d, l);
}

// Values just folded lie in [0, q) except for about d in 2^b of them: q is added or subtracted in a
// branch that is hardly ever taken, of one test for all N values
template <int N> __device__ __forceinline__ void settle_rare(uint64_t (&v)[N], uint64_t q)
{
    bool out = false;
#pragma unroll
    for (int i = 0; i < N; i++) out |= v[i] >= q;  // negative ones too
    if (out) {
        asm volatile("");  // a branch, not selects
#pragma unroll
        for (int i = 0; i < N; i++) v[i] += (int64_t)v[i] < 0 ? q : v[i] >= q ? 0 - q : 0;
    }
}

// v mod q in [0, q), for every v
template <int N> __device__ __forceinline__ void fold_finish(uint64_t (&v)[N], const FoldPrime &P)
{
#pragma unroll
    for (int i = 0; i < N; i++) v[i] = (uint64_t)fold((int64_t)v[i], P);
    if (P.refold) {
#pragma unroll
        for (int i = 0; i < N; i++) v[i] = (uint64_t)fold((int64_t)v[i], P);
    }
    settle_rare(v, P.q);
}
__device__ __forceinline__ uint64_t fold_finish(int64_t v, const FoldPrime &P)
{
    uint64_t x[1] = {(uint64_t)v};
    fold_finish(x, P);
    return x[0];
}

// ---- sums of products in 30-bit parts
//
// Residues below 2^60 split at bit 30 into parts of at most 30 bits, so four multiply-adds per
// product go into three 64-bit sums (weights 1, 2^30, 2^60) without carries.  A product adds
// at most 2 (2^30 - 1)^2 to the middle sum: seven products and the reduction's two terms fit, and
// fourteen below 2^59, where the outer sums' fourteen terms of (2^30 - 1)^2 are the limit.
// The reduction takes two Montgomery steps of 30 bits, so one factor is kept times 2^60.
constexpr uint32_t kMask30 = (1u << 30) - 1;
constexpr int kSumTerms = 7;  // products between two spill()s, twice that below 2^59

__device__ __forceinline__ uint64_t madu(uint32_t a, uint32_t b, uint64_t c)
{
    uint64_t r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
// a factor split for the sums: the low 30 bits in the low word, the rest in the high word
__device__ __forceinline__ uint64_t split30(uint64_t x) { return (x & kMask30) | ((x >> 30) << 32); }
__device__ __forceinline__ uint64_t join30(uint64_t x) { return (x & kMask30) | ((x >> 32) << 30); }

// what a sum's reduction needs of a prime
struct SumPrime {
    uint64_t q;
    uint32_t q0, q1, minv;
    int c, d, mask;
    __device__ __forceinline__ SumPrime() {}
    __device__ __forceinline__ SumPrime(const FoldPrime &P)
        : q(P.q), q0(P.q0), q1(P.q1), minv(P.minv), c(P.c), d(P.d), mask(P.mask)
    {
    }
};

// v - (v >> b) 2^b + (v >> b) d: congruent to v, below 2^b + 2^(64-b) d
template <class P_> __device__ __forceinline__ uint64_t fold_u(uint64_t v, const P_ &P)
{
    const uint32_t vh = (uint32_t)(v >> 32);
    return madu(vh >> P.c, (uint32_t)P.d, ((uint64_t)(vh & (uint32_t)P.mask) << 32) | (uint32_t)v);
}

struct Sum30 {
    uint64_t a = 0, b = 0, c = 0;
    // += x k for split x (x0, x1) and k
    __device__ __forceinline__ void mac(uint32_t x0, uint32_t x1, uint32_t k0, uint32_t k1)
    {
        a = madu(x0, k0, a);
        b = madu(x0, k1, b);
        c = madu(x1, k1, c);
        b = madu(x1, k0, b);
    }
    __device__ __forceinline__ void mac(uint32_t x0, uint32_t x1, uint64_t k) { mac(x0, x1, (uint32_t)k, (uint32_t)(k >> 32)); }
    // room for kSumTerms more products: the middle sum's high part moves up, the high sum is folded
    template <class P_> __device__ __forceinline__ void spill(const P_ &P)
    {
        c = fold_u(c + (b >> 30) + (a >> 60), P);
        b &= kMask30;
        a &= (1ull << 60) - 1;
    }
    // the sum times 2^-60 mod q.  Up to 14 products and the carries from below come to less than 18 2^b, so
    // the fold leaves less than 2^b + 18 d < 2 q, which settle_rare() brings below q
    template <class P_> __device__ __forceinline__ uint64_t reduce(const P_ &P) const
    {
        const uint32_t m0 = ((uint32_t)a * P.minv) & kMask30;
        uint64_t t = madu(m0, P.q1, b) + (madu(m0, P.q0, a) >> 30);
        const uint32_t m1 = ((uint32_t)t * P.minv) & kMask30;
        return fold_u(madu(m1, P.q1, c) + (madu(m1, P.q0, t) >> 30), P);
    }
};
#endif

} // namespace hx
