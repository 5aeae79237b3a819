// The negacyclic NTT of one limb = Cooley-Tukey (forward, natural ->
// bit-reversed order, psi powers merged into the twiddles) and
// Gentleman-Sande (inverse), split into a column phase (the first log2(N1)
// stages: N1 rows of stride N2) and a row phase (the remaining stages on N2
// contiguous words), each staged through shared memory.  Every global word is
// read and written once per phase with 128-byte coalesced row segments.
//
// The phase kernels are templates over the arithmetic: ArithFold for chains of primes just
// below powers of two (modfold.cuh; instantiated in ntt_fold.cu), ArithShoup for every other
// chain (ntt.cu).
#pragma once
#include <algorithm>
#include <cstdio>
#include <memory>

#include "launch_util.cuh"

namespace hx {

// Harvey's lazy butterflies on Shoup products: forward values stay in [0, 4q), inverse ones in
// [0, 2q).
struct ArithShoup {
    typedef PrimeConst Prime;
    typedef ulonglong2 Tw;
    static constexpr bool kTracked = false;
    static constexpr int kThreadsPerSm = 768;  // at most 85 registers a thread
    static __device__ __forceinline__ void ct(uint64_t &x, uint64_t &y, const Tw w, const Prime &P)
    {
        const uint64_t two_q = 2 * P.q;
        uint64_t a = x;
        if (a >= two_q) a -= two_q;
        const uint64_t t = shoup_lazy(y, w.x, w.y, P.q);
        x = a + t;
        y = a - t + two_q;
    }
    static __device__ __forceinline__ void gs(uint64_t &x, uint64_t &y, const Tw w, const Prime &P)
    {
        const uint64_t two_q = 2 * P.q;
        uint64_t u = x + y;
        if (u >= two_q) u -= two_q;
        const uint64_t d = x - y + two_q;
        x = u;
        y = shoup_lazy(d, w.x, w.y, P.q);
    }
    // the last inverse stage with N^-1 folded in, outputs in [0, 2q)
    static __device__ __forceinline__ void gs_last(uint64_t &x, uint64_t &y, const Prime &P)
    {
        const uint64_t two_q = 2 * P.q;
        uint64_t u = x + y;
        if (u >= two_q) u -= two_q;
        const uint64_t d = x - y + two_q;
        x = shoup_lazy(u, P.n_inv, P.n_inv_sh, P.q);
        y = shoup_lazy(d, P.n_inv_w1, P.n_inv_w1_sh, P.q);
    }
    static __device__ __forceinline__ uint64_t settle(uint64_t v, const Prime &) { return v; }
    template <int N> static __device__ __forceinline__ void finish(uint64_t (&v)[N], const Prime &P)
    {
#pragma unroll
        for (int i = 0; i < N; i++) v[i] = csub(csub(v[i], 2 * P.q), P.q);
    }
    static const Prime *primes(const DeviceTables &t) { return t.primes; }
    static const Tw *twiddles(const DeviceTables &t, bool inv) { return inv ? t.tw_inv : t.tw_fwd; }
    static __device__ __forceinline__ const Prime *job_primes(const NttJob &J) { return J.primes; }
    static __device__ __forceinline__ const Tw *job_twiddles(const NttJob &J, bool inv)
    {
        return inv ? J.tw_inv : J.tw_fwd;
    }
};

// Signed butterflies on fold products (two's complement in the same 64-bit words).  Sums grow
// until a tracked bound asks for a fold: the bound of every register is known at compile time,
// so a radix-16 pass of the forward transform folds none of its 64 sums and the inverse one a few.
//
// The butterflies set the transform's time, so this is where it was won: 1600 limbs of N = 2^14
// take 199 us forward and 205 us inverse against 274 and 283 with Shoup butterflies in the same
// tiles (9.2e11 butterflies/s; a network of them alone in registers runs at 1.5e12, and the L1 pipe
// that returns 16 bytes of twiddle per thread and multiplication is 50-75 % busy).
struct ArithFold {
    typedef FoldPrime Prime;
    typedef int4 Tw;
    static constexpr bool kTracked = true;
    static constexpr int kThreadsPerSm = 1024;  // at most 64 registers a thread
    static __device__ __forceinline__ void ct(uint64_t &x, uint64_t &y, const Tw w, const Prime &P)
    {
        const uint64_t t = (uint64_t)fold_mul((int64_t)y, w, P), a = x;
        x = a + t;
        y = a - t;
    }
    static __device__ __forceinline__ void gs(uint64_t &x, uint64_t &y, const Tw w, const Prime &P)
    {
        const uint64_t d = x - y;
        x = x + y;
        y = (uint64_t)fold_mul((int64_t)d, w, P);
    }
    static __device__ __forceinline__ void gs_last(uint64_t &x, uint64_t &y, const Prime &P)
    {
        const uint64_t d = x - y, u = x + y;
        x = (uint64_t)fold_mul((int64_t)u, P.n_inv, P);
        y = (uint64_t)fold_mul((int64_t)d, P.n_inv_w1, P);
    }
    static __device__ __forceinline__ uint64_t settle(uint64_t v, const Prime &P) { return (uint64_t)fold((int64_t)v, P); }
    template <int N> static __device__ __forceinline__ void finish(uint64_t (&v)[N], const Prime &P) { fold_finish(v, P); }
    static const Prime *primes(const DeviceTables &t) { return t.fold; }
    static const Tw *twiddles(const DeviceTables &t, bool inv) { return inv ? t.ftw_inv : t.ftw_fwd; }
    static __device__ __forceinline__ const Prime *job_primes(const NttJob &J) { return J.fold; }
    static __device__ __forceinline__ const Tw *job_twiddles(const NttJob &J, bool inv)
    {
        return inv ? J.ftw_inv : J.ftw_fwd;
    }
};

namespace {

// ---- NTT ----------------------------------------------------------------------
//
// A phase holds, in shared memory, n_sub independent sub-transforms of M = 2^L
// points (element e of sub-transform k at sh[k*sk + e*se (+ e/16 padding)]).
// Its L local stages run as two register passes: each thread loads 2^R
// elements spaced t = M >> (S0+R) apart, applies R radix-2 stages in
// registers (2^R - 1 twiddle loads for R*2^(R-1) butterflies) and stores them
// back.  Global stage of local stage s is g0 + s; the twiddle of a butterfly
// at global stage G on global element j is tw[2^G + (j >> (log N - G))].

// two adjacent twiddles, 32-byte aligned (their tables are)
template <class Tw> __device__ __forceinline__ void load_pair(const Tw *p, Tw &a, Tw &b)
{
    static_assert(sizeof(Tw) == 16, "16-byte twiddles");
    union {
        uint64_t w[4];
        Tw t[2];
    } u;
    asm("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];"
        : "=l"(u.w[0]), "=l"(u.w[1]), "=l"(u.w[2]), "=l"(u.w[3])
        : "l"(p));
    a = u.t[0];
    b = u.t[1];
}

// R stages in registers.  bound: the values' bounds in sixteenths before and after (tracked
// arithmetic; compile-time constants once unrolled).  A forward sum x +- w y only bounds x: y may
// reach the limit.  An inverse sum folds its larger operand, and the other if need be, where it
// would pass the limit.  SCALE: the inverse's stage 0 applies N^-1.
template <class A, int R, int S0, bool INV, bool SCALE = false>
__device__ __forceinline__ void ntt_stages(uint64_t (&v)[1 << R], int (&bound)[1 << R],
                                           const typename A::Tw *__restrict__ tw, int g0, int blk, int hi,
                                           const typename A::Prime &P)
{
    constexpr int RR = 1 << R;
#pragma unroll
    for (int step = 0; step < R; step++) {
        const int vv = INV ? R - 1 - step : step;
        const int s = S0 + vv, half = RR >> (vv + 1);
        const int tbase = (1 << (g0 + s)) + (blk << s) + (hi << vv);
        typename A::Tw ws[2];
#pragma unroll
        for (int gl = 0; gl < (1 << vv); gl++) {
            const bool scale = SCALE && vv == 0;
            if (scale) ws[0] = typename A::Tw();
            else if (vv == 0) ws[0] = tw[tbase];  // from the second stage of a pass on, pairs (32 bytes, aligned)
            else if (gl % 2 == 0) load_pair(tw + tbase + gl, ws[0], ws[1]);
            const typename A::Tw w = ws[gl % 2];
#pragma unroll
            for (int j = 0; j < half; j++) {
                const int ix = gl * 2 * half + j, iy = ix + half;
                if (A::kTracked) {
                    if (!INV) {
                        if (bound[ix] + kFoldProduct > kFoldLimit) {
                            v[ix] = A::settle(v[ix], P);
                            bound[ix] = kFoldSettled;
                        }
                        bound[ix] = bound[iy] = bound[ix] + kFoldProduct;
                    } else {
#pragma unroll
                        for (int again = 0; again < 2; again++)
                            if (bound[ix] + bound[iy] > kFoldLimit) {
                                const int k = bound[ix] >= bound[iy] ? ix : iy;
                                v[k] = A::settle(v[k], P);
                                bound[k] = kFoldSettled;
                            }
                        bound[ix] = bound[ix] + bound[iy];
                        bound[iy] = kFoldProduct;
                    }
                }
                if (!INV) A::ct(v[ix], v[iy], w, P);
                else if (scale) A::gs_last(v[ix], v[iy], P);
                else A::gs(v[ix], v[iy], w, P);
            }
        }
    }
}

// the bound after R forward stages (every value has the same)
constexpr int fwd_bound(int in, int R)
{
    for (int i = 0; i < R; i++) in = (in + kFoldProduct > kFoldLimit ? kFoldSettled : in) + kFoldProduct;
    return in;
}
// bounds between the passes of a transform: a value above its pass's bound is folded before it is
// stored.  Forward, the column phase hands over what most of its sizes end with, unfolded; inverse,
// every pass hands over the products as they are and folds the sums.
constexpr int kFwdMid = 67, kInvMid = kFoldProduct;

// bounds of a transform's inputs in sixteenths (tracked arithmetic): below 4q forward, 2q inverse,
// as the Shoup butterflies take them
constexpr int kFwdIn = 64, kInvIn = 32;

template <int L, bool ALT = false> struct Split {
    // first pass (stages 0..R1-1) and second pass; ALT swaps the two radices of an odd L
    static constexpr int R1 = ALT ? L / 2 : (L + 1) / 2;
    static constexpr int R2 = L - R1;
};

// Where a tile's element e of sub-transform k lies, in its global rows and in shared memory, and
// which sub-transform and butterfly group a work item w has.
//
// Columns: W adjacent columns, element e in row e; consecutive threads on consecutive columns, so
// a warp moves whole 128-byte row segments and meets no bank twice.
template <int L, int W, bool ALT> struct ColTile {
    static constexpr bool kRows = false;
    static constexpr int WORDS = (1 << L) * W;
    int n2;
    __device__ __forceinline__ static int sub(int w, int) { return w % W; }
    __device__ __forceinline__ static int group(int w, int) { return w / W; }
    // byte offset: 32 bits on the block's uniform base
    __device__ __forceinline__ uint32_t global(int e, int k) const { return 8u * ((uint32_t)e * n2 + k); }
    __device__ __forceinline__ static int shared(int e, int k) { return e * W + k; }
};
// Rows: W contiguous blocks of M words.  The first pass of the stages takes elements 2^R2 apart
// (runs of 2^R2 threads on consecutive words), the second 2^R2 consecutive ones; one spare word
// per 2^R2 and a block stride of 2^R2 mod 16 words keep both on distinct banks.
template <int L, int W, bool ALT> struct RowTile {
    static constexpr bool kRows = true;
    static constexpr int M = 1 << L, R2 = Split<L, ALT>::R2, RUN = 1 << R2;
    static constexpr int DATA = M + (M >> R2), SK = DATA + ((RUN - DATA) % 16 + 16) % 16, WORDS = SK * W;
    __device__ __forceinline__ static int sub(int w, int items) { return w / items; }
    __device__ __forceinline__ static int group(int w, int items) { return w % items; }
    __device__ __forceinline__ uint32_t global(int e, int k) const { return 8u * (k * M + e); }
    __device__ __forceinline__ static int shared(int e, int k) { return k * SK + e + (e >> R2); }
};

// 32-byte global accesses (sm_100 and later), for 32-byte aligned addresses
__device__ __forceinline__ void ld_global_32(const uint64_t *p, uint64_t &a, uint64_t &b, uint64_t &c, uint64_t &d)
{
    asm volatile("ld.global.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(a), "=l"(b), "=l"(c), "=l"(d) : "l"(p));
}
__device__ __forceinline__ void st_global_32(uint64_t *p, uint64_t a, uint64_t b, uint64_t c, uint64_t d)
{
    asm volatile("st.global.v4.u64 [%0], {%1, %2, %3, %4};" ::"l"(p), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
}

__device__ __forceinline__ const uint64_t *at_bytes(const uint64_t *p, uint32_t off)
{
    return reinterpret_cast<const uint64_t *>(reinterpret_cast<const char *>(p) + off);
}
__device__ __forceinline__ uint64_t *at_bytes(uint64_t *p, uint32_t off)
{
    return reinterpret_cast<uint64_t *>(reinterpret_cast<char *>(p) + off);
}

// RR elements of a butterfly group, TL apart, from or to global memory; consecutive ones (TL = 1)
// of a row in 16-byte pieces, or in 32-byte ones where the caller found the rows aligned (wide)
template <class Tile, int RR, int TL>
__device__ __forceinline__ void load_group(uint64_t (&v)[RR], const uint64_t *src, const Tile &t, int base, int k, bool wide)
{
    if (Tile::kRows && TL == 1) {
        const uint64_t *p = at_bytes(src, t.global(base, k));
        if (wide) {
#pragma unroll
            for (int m = 0; m < RR; m += 4) ld_global_32(p + m, v[m], v[m + 1], v[m + 2], v[m + 3]);
        } else {
#pragma unroll
            for (int m = 0; m < RR; m += 2) {
                const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(p + m);
                v[m] = x.x;
                v[m + 1] = x.y;
            }
        }
    } else {
#pragma unroll
        for (int m = 0; m < RR; m++) v[m] = *at_bytes(src, t.global(base + m * TL, k));
    }
}
template <class Tile, int RR, int TL>
__device__ __forceinline__ void store_group(const uint64_t (&v)[RR], uint64_t *dst, const Tile &t, int base, int k, bool wide)
{
    if (Tile::kRows && TL == 1) {
        uint64_t *p = at_bytes(dst, t.global(base, k));
        if (wide) {
#pragma unroll
            for (int m = 0; m < RR; m += 4) st_global_32(p + m, v[m], v[m + 1], v[m + 2], v[m + 3]);
        } else {
#pragma unroll
            for (int m = 0; m < RR; m += 2)
                *reinterpret_cast<ulonglong2 *>(p + m) = make_ulonglong2(v[m], v[m + 1]);
        }
    } else {
#pragma unroll
        for (int m = 0; m < RR; m++) *at_bytes(dst, t.global(base + m * TL, k)) = v[m];
    }
}

// A phase's two register passes over one tile with one shared-memory exchange: the first pass
// takes its elements straight from global memory, the second stores its results straight there.
// No tile is staged ahead: a block holds its tile once (16 or 19 KB at width 16), so eight blocks
// of 128 threads share an SM and cover each other's loads.
//
// Forward: columns leave lazy (folded) values for the row phase, rows finish.  Inverse: rows leave
// lazy values; the column phase ends with stage 0, whose butterfly also applies N^-1 --
// x' = (x+y) N^-1 and y' = (x-y) psi^-brv(1) N^-1, one product each instead of a butterfly product
// and two scalings -- and finishes.
//
// IN, OUT: the bounds of the values taken and handed on.
template <class A, class Tile, int L, int R, int S0, bool INV, bool FIRST, int IN, int OUT>
__device__ __forceinline__ void ntt_pass(uint64_t *sh, const uint64_t *src, uint64_t *dst, const Tile &tile, int n_sub,
                                         const typename A::Tw *__restrict__ tw, int g0, int blk0, int blk_step,
                                         const typename A::Prime &P, int nthr, bool wide)
{
    constexpr int M = 1 << L, RR = 1 << R, TL = M >> (S0 + R), ITEMS = M >> R;
    constexpr bool kLast = !FIRST && INV != Tile::kRows;  // the pass that ends the transform
    for (int w = threadIdx.x; w < ITEMS * n_sub; w += nthr) {
        const int k = Tile::sub(w, ITEMS), u = Tile::group(w, ITEMS);
        const int hi = u / TL, lo = u % TL;
        const int base = hi * TL * RR + lo;
        uint64_t v[RR];
        int bound[RR];
#pragma unroll
        for (int m = 0; m < RR; m++) bound[m] = IN;
        if (FIRST) {
            load_group<Tile, RR, TL>(v, src, tile, base, k, wide);
        } else {
#pragma unroll
            for (int m = 0; m < RR; m++) v[m] = sh[Tile::shared(base + m * TL, k)];
        }
        ntt_stages<A, R, S0, INV, INV && kLast>(v, bound, tw, g0, blk0 + k * blk_step, hi, P);
        if (kLast) {
            A::finish(v, P);
        } else {
#pragma unroll
            for (int m = 0; m < RR; m++)
                if (bound[m] > OUT) v[m] = A::settle(v[m], P);
        }
        if (FIRST) {
#pragma unroll
            for (int m = 0; m < RR; m++) sh[Tile::shared(base + m * TL, k)] = v[m];
        } else {
            store_group<Tile, RR, TL>(v, dst, tile, base, k, wide);
        }
    }
}

// one tile of a phase: src and dst at its first word (they may be the same)
template <class A, class Tile, int L, int W, bool INV, bool ALT>
__device__ __forceinline__ void ntt_tile(uint64_t *sh, const uint64_t *src, uint64_t *dst, const Tile &tile,
                                         const typename A::Tw *__restrict__ tw, int g0, int blk0,
                                         const typename A::Prime &P, int nthr, bool wide)
{
    constexpr int R1 = Split<L, ALT>::R1, R2 = Split<L, ALT>::R2;
    constexpr int step = Tile::kRows ? 1 : 0;  // rows: every sub-transform has its own twiddles
    if (!INV) {
        constexpr int in = Tile::kRows ? kFwdMid : kFwdIn, mid = fwd_bound(in, R1);
        ntt_pass<A, Tile, L, R1, 0, false, true, in, mid>(sh, src, dst, tile, W, tw, g0, blk0, step, P, nthr, wide);
        __syncthreads();
        ntt_pass<A, Tile, L, R2, R1, false, false, mid, kFwdMid>(sh, src, dst, tile, W, tw, g0, blk0, step, P, nthr, wide);
    } else {
        constexpr int in = Tile::kRows ? kInvIn : kInvMid;
        ntt_pass<A, Tile, L, R2, R1, true, true, in, kInvMid>(sh, src, dst, tile, W, tw, g0, blk0, step, P, nthr, wide);
        __syncthreads();
        ntt_pass<A, Tile, L, R1, 0, true, false, kInvMid, kInvMid>(sh, src, dst, tile, W, tw, g0, blk0, step, P, nthr, wide);
    }
}

// grid: tiles of a row, rows, groups
//
// column phase: the first LOGM stages on M rows of stride N2, COLS adjacent columns per block
template <class A, int LOGM, int COLS, bool INV, bool ALT>
__global__ void __launch_bounds__((1 << (LOGM - Split<LOGM, ALT>::R1)) * COLS,
                                  A::kThreadsPerSm / ((1 << (LOGM - Split<LOGM, ALT>::R1)) * COLS))
k_ntt_cols(const __grid_constant__ NttRows R, const typename A::Prime *__restrict__ primes,
           const typename A::Tw *__restrict__ tw_all, int log_n)
{
    after_previous_kernel();
    extern __shared__ uint64_t sh[];
    constexpr int T = (1 << (LOGM - Split<LOGM, ALT>::R1)) * COLS;
    const int N = 1 << log_n, N2 = N >> LOGM, row = blockIdx.y, c0 = blockIdx.x * COLS;
    const int pr = R.prime[row];
    const typename A::Prime P = primes[pr];
    uint64_t *dst = R.dst + blockIdx.z * R.dst_gs + (size_t)R.dst_off[row] * N + c0;
    const uint64_t *src = INV ? dst : R.src + blockIdx.z * R.src_gs + (size_t)R.src_off[row] * N + c0;
    ntt_tile<A, ColTile<LOGM, COLS, ALT>, LOGM, COLS, INV, ALT>(sh, src, dst, ColTile<LOGM, COLS, ALT>{N2},
                                                                tw_all + (size_t)pr * N, 0, 0, P, T, false);
}

// row phase: the remaining LOGM stages on ROWS contiguous blocks of M words
template <class A, int LOGM, int ROWS, bool INV, bool ALT>
__global__ void __launch_bounds__((1 << (LOGM - Split<LOGM, ALT>::R1)) * ROWS,
                                  A::kThreadsPerSm / ((1 << (LOGM - Split<LOGM, ALT>::R1)) * ROWS))
k_ntt_rows(const __grid_constant__ NttRows R, const typename A::Prime *__restrict__ primes,
           const typename A::Tw *__restrict__ tw_all, int log_n, bool wide)
{
    after_previous_kernel();
    extern __shared__ uint64_t sh[];
    constexpr int T = (1 << (LOGM - Split<LOGM, ALT>::R1)) * ROWS;
    const int N = 1 << log_n;
    const int row = blockIdx.y, pr = R.prime[row], r_base = blockIdx.x * ROWS;
    const typename A::Prime P = primes[pr];
    uint64_t *dst = R.dst + blockIdx.z * R.dst_gs + (size_t)R.dst_off[row] * N + (r_base << LOGM);
    const uint64_t *src =
        INV ? R.src + blockIdx.z * R.src_gs + (size_t)R.src_off[row] * N + (r_base << LOGM) : dst;
    ntt_tile<A, RowTile<LOGM, ROWS, ALT>, LOGM, ROWS, INV, ALT>(sh, src, dst, RowTile<LOGM, ROWS, ALT>{},
                                                                tw_all + (size_t)pr * N, log_n - LOGM, r_base, P, T, wide);
}

// tile widths the autotuner chooses from (sub-transforms per block); a variant is a width index
// plus NTT_WIDTHS if the phase's two register passes swap radices (odd phase sizes only)
constexpr const int *kNttTiles = kNttTileWidths;

template <class A, int LOGM, int COLS, bool INV, bool ALT>
void ntt_cols_w(const LaunchCtx &c, const NttRows &rows)
{
    constexpr int T = (1 << (LOGM - Split<LOGM, ALT>::R1)) * COLS;
    const int N2 = c.N >> LOGM;
    HX_CHECK(N2 % COLS == 0, HX_EINVAL, "NTT tile wider than the ring");
    const size_t smem = sizeof(uint64_t) * ColTile<LOGM, COLS, ALT>::WORDS;
    static const bool attr =  // thread-safe one-time setup
        cudaFuncSetAttribute(k_ntt_cols<A, LOGM, COLS, INV, ALT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) == cudaSuccess;
    (void)attr;
    launch(c.stream, k_ntt_cols<A, LOGM, COLS, INV, ALT>, dim3(N2 / COLS, rows.n_rows, rows.n_groups), T, smem, rows,
           A::primes(*c.t), A::twiddles(*c.t, INV), c.log_n);
}

template <class A, int LOGM, int ROWS, bool INV, bool ALT>
void ntt_rows_w(const LaunchCtx &c, const NttRows &rows)
{
    constexpr int T = (1 << (LOGM - Split<LOGM, ALT>::R1)) * ROWS;
    const int N1 = c.N >> LOGM;
    HX_CHECK(N1 % ROWS == 0, HX_EINVAL, "NTT tile wider than the ring");
    const size_t smem = sizeof(uint64_t) * RowTile<LOGM, ROWS, ALT>::WORDS;
    static const bool attr =  // thread-safe one-time setup
        cudaFuncSetAttribute(k_ntt_rows<A, LOGM, ROWS, INV, ALT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) == cudaSuccess;
    (void)attr;
    // rows and blocks are multiples of 32 bytes: 32-byte pieces need only the bases and group strides aligned
    const bool wide = ((reinterpret_cast<uintptr_t>(rows.src) | reinterpret_cast<uintptr_t>(rows.dst) |
                        (rows.src_gs | rows.dst_gs) * sizeof(uint64_t)) & 31) == 0;
    launch(c.stream, k_ntt_rows<A, LOGM, ROWS, INV, ALT>, dim3(N1 / ROWS, rows.n_rows, rows.n_groups), T, smem, rows,
           A::primes(*c.t), A::twiddles(*c.t, INV), c.log_n, wide);
}

template <class A, bool INV, int LOGM, bool ALT>
void ntt_phase_a(const LaunchCtx &c, const NttRows &r, bool cols, int wi)
{
    switch (wi) {
    case 0: cols ? ntt_cols_w<A, LOGM, 4, INV, ALT>(c, r) : ntt_rows_w<A, LOGM, 4, INV, ALT>(c, r); break;
    case 1: cols ? ntt_cols_w<A, LOGM, 8, INV, ALT>(c, r) : ntt_rows_w<A, LOGM, 8, INV, ALT>(c, r); break;
    case 2: cols ? ntt_cols_w<A, LOGM, 16, INV, ALT>(c, r) : ntt_rows_w<A, LOGM, 16, INV, ALT>(c, r); break;
    default: cols ? ntt_cols_w<A, LOGM, 32, INV, ALT>(c, r) : ntt_rows_w<A, LOGM, 32, INV, ALT>(c, r); break;
    }
}

template <class A, bool INV, int LOGM>
void ntt_phase_l(const LaunchCtx &c, const NttRows &r, bool cols, int var)
{
    // the tile must not be wider than the other dimension of the ring
    const int other = c.N >> LOGM;
    int wi = var % NTT_WIDTHS;
    while (wi > 0 && kNttTiles[wi] > other) wi--;
    if ((LOGM & 1) && var >= NTT_WIDTHS) ntt_phase_a<A, INV, LOGM, (LOGM & 1) != 0>(c, r, cols, wi);
    else ntt_phase_a<A, INV, LOGM, false>(c, r, cols, wi);
}

} // namespace

// One phase of a transform (cols: the column phase) of 2^logm points per sub-transform, variant
// var; instantiated for each arithmetic in its own file
template <class A> void ntt_phase(const LaunchCtx &c, const NttRows &r, bool inv, bool cols, int logm, int var)
{
    switch (logm) {
    case 5: inv ? ntt_phase_l<A, true, 5>(c, r, cols, var) : ntt_phase_l<A, false, 5>(c, r, cols, var); break;
    case 6: inv ? ntt_phase_l<A, true, 6>(c, r, cols, var) : ntt_phase_l<A, false, 6>(c, r, cols, var); break;
    case 7: inv ? ntt_phase_l<A, true, 7>(c, r, cols, var) : ntt_phase_l<A, false, 7>(c, r, cols, var); break;
    case 8: inv ? ntt_phase_l<A, true, 8>(c, r, cols, var) : ntt_phase_l<A, false, 8>(c, r, cols, var); break;
    default: throw Error{HX_EINVAL, "unsupported NTT size"};
    }
}

namespace {

// ---- several rings in one launch ------------------------------------------------
// A job is n_rows rows of one ring (its own N, primes and twiddles).  One kernel per phase takes the tiles of every job; a tile's phase
// size picks the template instance, with the tile width chosen so every
// instance runs 128 threads.

constexpr int kMultiT = 128;
template <int LOGM> struct MultiW {  // tile width per phase size: (M >> R1) * W = 128 threads
    static constexpr int W = kMultiT / ((1 << LOGM) >> Split<LOGM>::R1);
};
constexpr int max4(int a, int b, int c, int d) { return std::max(std::max(a, b), std::max(c, d)); }
// words of the largest tile
constexpr int kMultiColsBuf = max4(ColTile<5, MultiW<5>::W, false>::WORDS, ColTile<6, MultiW<6>::W, false>::WORDS,
                                   ColTile<7, MultiW<7>::W, false>::WORDS, ColTile<8, MultiW<8>::W, false>::WORDS);
constexpr int kMultiRowsBuf = max4(RowTile<5, MultiW<5>::W, false>::WORDS, RowTile<6, MultiW<6>::W, false>::WORDS,
                                   RowTile<7, MultiW<7>::W, false>::WORDS, RowTile<8, MultiW<8>::W, false>::WORDS);

template <class A> struct MultiTile {
    const uint64_t *src;  // the first phase's source
    uint64_t *row;
    const typename A::Tw *tw;
    const typename A::Prime *primes;
    int pr, logm, log_n, bx;
};

template <class A>
__device__ __forceinline__ MultiTile<A> multi_tile(const NttJob *jobs, int n_jobs, int t, bool cols, bool inv)
{
    int lo = 0, hi = n_jobs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if ((cols ? jobs[mid].tile0_cols : jobs[mid].tile0_rows) <= t) lo = mid;
        else hi = mid - 1;
    }
    const NttJob &J = jobs[lo];
    MultiTile<A> m;
    const int local = t - (cols ? J.tile0_cols : J.tile0_rows);
    m.log_n = J.log_n;
    const int logc = J.log_n / 2 + ntt_default_split(J.log_n);
    m.logm = cols ? logc : J.log_n - logc;
    const int n = 1 << J.log_n;
    const int W = kMultiT / ((1 << m.logm) >> ((m.logm + 1) / 2));
    const int nb = (n >> m.logm) / W;
    const int r = local / nb;
    m.bx = local % nb;
    m.pr = J.prime[r % J.n_limbs];
    m.primes = A::job_primes(J);
    m.src = J.src + (size_t)r * n;
    m.row = J.data + (size_t)r * n;
    m.tw = A::job_twiddles(J, inv) + (size_t)m.pr * n;
    return m;
}

template <class A, int LOGM, bool INV, bool COLS_PHASE>
__device__ __forceinline__ void multi_run(uint64_t *sh, const MultiTile<A> &m, const typename A::Prime &P)
{
    constexpr int W = MultiW<LOGM>::W;
    if (COLS_PHASE) {
        typedef ColTile<LOGM, W, false> Tile;
        uint64_t *d = m.row + m.bx * W;
        ntt_tile<A, Tile, LOGM, W, INV, false>(sh, INV ? d : m.src + m.bx * W, d, Tile{(1 << m.log_n) >> LOGM}, m.tw, 0, 0, P, kMultiT, false);
    } else {
        typedef RowTile<LOGM, W, false> Tile;
        const int r_base = m.bx * W;
        uint64_t *d = m.row + ((size_t)r_base << LOGM);
        const uint64_t *from = INV ? m.src + ((size_t)r_base << LOGM) : d;
        const bool wide = ((reinterpret_cast<uintptr_t>(d) | reinterpret_cast<uintptr_t>(from)) & 31) == 0;
        ntt_tile<A, Tile, LOGM, W, INV, false>(sh, from, d, Tile{}, m.tw, m.log_n - LOGM, r_base, P, kMultiT, wide);
    }
}

template <class A, bool INV, bool COLS_PHASE>
__global__ void __launch_bounds__(kMultiT, A::kThreadsPerSm / kMultiT)
    k_ntt_multi(const NttJob *__restrict__ jobs, int n_jobs)
{
    after_previous_kernel();
    extern __shared__ uint64_t sh[];
    const MultiTile<A> m = multi_tile<A>(jobs, n_jobs, blockIdx.x, COLS_PHASE, INV);
    const typename A::Prime P = m.primes[m.pr];
    switch (m.logm) {
    case 5: multi_run<A, 5, INV, COLS_PHASE>(sh, m, P); break;
    case 6: multi_run<A, 6, INV, COLS_PHASE>(sh, m, P); break;
    case 7: multi_run<A, 7, INV, COLS_PHASE>(sh, m, P); break;
    default: multi_run<A, 8, INV, COLS_PHASE>(sh, m, P); break;
    }
}

} // namespace

// both phases of the several-ring transform over a job table on the device
template <class A> void ntt_multi_phases(cudaStream_t s, const NttJob *jp, int n_jobs, int tc, int tr, bool inverse)
{
    constexpr size_t smem_c = sizeof(uint64_t) * kMultiColsBuf, smem_r = sizeof(uint64_t) * kMultiRowsBuf;
    static_assert(smem_c <= 48 * 1024 && smem_r <= 48 * 1024, "a tile fits without an attribute");
    if (!inverse) {
        launch(s, k_ntt_multi<A, false, true>, tc, kMultiT, smem_c, jp, n_jobs);
        launch(s, k_ntt_multi<A, false, false>, tr, kMultiT, smem_r, jp, n_jobs);
    } else {
        launch(s, k_ntt_multi<A, true, false>, tr, kMultiT, smem_r, jp, n_jobs);
        launch(s, k_ntt_multi<A, true, true>, tc, kMultiT, smem_c, jp, n_jobs);
    }
}

// ---- end of the several-ring kernels

} // namespace hx
