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
    // the last inverse stage with N^-1 folded in, outputs in [0, q)
    static __device__ __forceinline__ void gs_last(uint64_t &x, uint64_t &y, const Prime &P)
    {
        const uint64_t two_q = 2 * P.q;
        uint64_t u = x + y;
        if (u >= two_q) u -= two_q;
        const uint64_t d = x - y + two_q;
        x = shoup(u, P.n_inv, P.n_inv_sh, P.q);
        y = shoup(d, P.n_inv_w1, P.n_inv_w1_sh, P.q);
    }
    static __device__ __forceinline__ uint64_t settle(uint64_t v, const Prime &) { return v; }
    static __device__ __forceinline__ uint64_t finish(uint64_t v, const Prime &P)
    {
        return csub(csub(v, 2 * P.q), P.q);
    }
    static __device__ __forceinline__ uint64_t times_n_inv(uint64_t v, const Prime &P)
    {
        return shoup(v, P.n_inv, P.n_inv_sh, P.q);
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
// took 332 us forward and 348 us inverse with Shoup butterflies and take 261 and 269 us.
struct ArithFold {
    typedef FoldPrime Prime;
    typedef int4 Tw;
    static constexpr bool kTracked = true;
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
        x = fold_finish(fold_mul((int64_t)u, P.n_inv, P), P);
        y = fold_finish(fold_mul((int64_t)d, P.n_inv_w1, P), P);
    }
    static __device__ __forceinline__ uint64_t settle(uint64_t v, const Prime &P) { return (uint64_t)fold((int64_t)v, P); }
    static __device__ __forceinline__ uint64_t finish(uint64_t v, const Prime &P) { return fold_finish((int64_t)v, P); }
    static __device__ __forceinline__ uint64_t times_n_inv(uint64_t v, const Prime &P)
    {
        return fold_finish(fold_mul((int64_t)v, P.n_inv, P), P);
    }
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

// R stages in registers.  IN: the inputs' bound in sixteenths (tracked arithmetic).  A forward sum
// x +- w y only bounds x: y may reach the limit.  An inverse sum folds the larger operand first
// where it would pass the limit.  SCALE: the inverse's stage 0 applies N^-1 and finishes.
template <class A, int R, int S0, bool INV, int IN, bool SCALE = false>
__device__ __forceinline__ void ntt_stages(uint64_t (&v)[1 << R], const typename A::Tw *__restrict__ tw, int g0, int blk,
                                           int hi, const typename A::Prime &P)
{
    constexpr int RR = 1 << R;
    int bound[RR];
#pragma unroll
    for (int m = 0; m < RR; m++) bound[m] = IN;
#pragma unroll
    for (int step = 0; step < R; step++) {
        const int vv = INV ? R - 1 - step : step;
        const int s = S0 + vv, half = RR >> (vv + 1);
        const int tbase = (1 << (g0 + s)) + (blk << s) + (hi << vv);
#pragma unroll
        for (int gl = 0; gl < (1 << vv); gl++) {
            const bool scale = SCALE && vv == 0;
            const typename A::Tw w = scale ? typename A::Tw() : tw[tbase + gl];
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

// One register pass in place in shared memory.  SETTLE: leave folded values (every pass but the
// last, whose results go through finish())
template <class A, int L, int R, int S0, bool INV, bool KFAST, bool PAD, int IN, bool SETTLE = true>
__device__ __forceinline__ void ntt_pass(uint64_t *sh, int n_sub, int sk, int se,
                                         const typename A::Tw *__restrict__ tw, int g0, int blk0, int blk_step,
                                         const typename A::Prime &P, int nthr)
{
    constexpr int M = 1 << L, RR = 1 << R, TL = M >> (S0 + R), ITEMS = M >> R;
    for (int w = threadIdx.x; w < ITEMS * n_sub; w += nthr) {
        const int k = KFAST ? w % n_sub : w / ITEMS;
        const int u = KFAST ? w / n_sub : w % ITEMS;
        const int hi = u / TL, lo = u % TL;
        const int base = hi * TL * RR + lo;
        const int blk = blk0 + k * blk_step;
        uint64_t v[RR];
#pragma unroll
        for (int m = 0; m < RR; m++) {
            const int e = base + m * TL;
            v[m] = sh[k * sk + e * se + (PAD ? 2 * (e >> 4) : 0)];
        }
        ntt_stages<A, R, S0, INV, IN>(v, tw, g0, blk, hi, P);
#pragma unroll
        for (int m = 0; m < RR; m++) {
            const int e = base + m * TL;
            sh[k * sk + e * se + (PAD ? 2 * (e >> 4) : 0)] = SETTLE ? A::settle(v[m], P) : v[m];
        }
    }
}

// The column phase's last register pass, its results stored straight to global memory (word e
// of column k at dst + e*N2 + k): consecutive threads hold consecutive columns, so each warp
// store covers whole COLS-word row segments and the phase needs no shared-memory round trip
// for its output.  Forward: outputs stay lazy for the row phase.  Inverse: the pass
// ends with stage 0, whose butterfly also applies N^-1 -- x' = (x+y) N^-1 and
// y' = (x-y) psi^-brv(1) N^-1, one product each instead of a butterfly product and two
// scalings -- and the outputs are fully reduced.
template <class A, int LOGM, int R, int S0, int COLS, bool INV>
__device__ __forceinline__ void ntt_pass_out(const uint64_t *sh, const typename A::Tw *__restrict__ tw,
                                             const typename A::Prime &P, uint64_t *dst, int N2, int nthr)
{
    constexpr int M = 1 << LOGM, RR = 1 << R, TL = M >> (S0 + R), ITEMS = M >> R;
    for (int w = threadIdx.x; w < ITEMS * COLS; w += nthr) {
        const int k = w % COLS, u = w / COLS;
        const int hi = u / TL, lo = u % TL;
        const int base = hi * TL * RR + lo;
        uint64_t v[RR];
#pragma unroll
        for (int m = 0; m < RR; m++) v[m] = sh[k + (base + m * TL) * COLS];
        static_assert(!INV || S0 == 0, "the inverse output pass must end with stage 0");
        ntt_stages<A, R, S0, INV, kFoldSettled, INV>(v, tw, 0, 0, hi, P);
#pragma unroll
        for (int m = 0; m < RR; m++) dst[(size_t)(base + m * TL) * N2 + k] = INV ? v[m] : A::settle(v[m], P);
    }
}

// bounds of a transform's inputs in sixteenths (tracked arithmetic): below 4q forward, 2q inverse,
// as the Shoup butterflies take them
constexpr int kFwdIn = 64, kInvIn = 32;

template <int L, bool ALT = false> struct Split {
    // first pass (stages 0..R1-1) and second pass; ALT swaps the two radices of an odd L
    static constexpr int R1 = ALT ? L / 2 : (L + 1) / 2;
    static constexpr int R2 = L - R1;
};

// Asynchronous global->shared copies (cp.async): the next tile streams in while
// the current one is transformed.
__device__ __forceinline__ void cp_async8(void *smem, const void *gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem));
}
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all_but_one() { asm volatile("cp.async.wait_group 1;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::); }

// tile t of a phase -> (group, row, position along the row)
struct TileId {
    int g, row, bx;
};
__device__ __forceinline__ TileId tile_of(int t, int nb, int n_rows)
{
    TileId r;
    r.bx = t % nb;
    const int rest = t / nb;
    r.row = rest % n_rows;
    r.g = rest / n_rows;
    return r;
}

// column phase: the first LOGM stages on M rows of stride N2 (COLS adjacent columns
// per tile); each block loops over tiles with the next tile (and its twiddles,
// indices below M) prefetched into the other half of shared memory
template <class A, int LOGM, int COLS, bool INV, bool ALT>
__global__ void __launch_bounds__((1 << (LOGM - Split<LOGM, ALT>::R1)) * COLS)
k_ntt_cols(const __grid_constant__ NttRows R, const typename A::Prime *__restrict__ primes,
           const typename A::Tw *__restrict__ tw_all, int log_n, int n_tiles)
{
    constexpr int M = 1 << LOGM, E = M * COLS, R1 = Split<LOGM, ALT>::R1, R2 = Split<LOGM, ALT>::R2;
    constexpr int T = (M >> R1) * COLS;
    extern __shared__ uint64_t sh[];
    typename A::Tw *const stw = reinterpret_cast<typename A::Tw *>(sh + 2 * E);
    const int N = 1 << log_n, N2 = N >> LOGM, nb = N2 / COLS;
    auto prefetch = [&](int t, int slot) {
        const TileId id = tile_of(t, nb, R.n_rows);
        const int pr = R.prime[id.row];
        const uint64_t *src = INV ? R.dst + (size_t)id.g * R.dst_gs + (size_t)R.dst_off[id.row] * N
                                  : R.src + (size_t)id.g * R.src_gs + (size_t)R.src_off[id.row] * N;
        const int c0 = id.bx * COLS;
        for (int i = threadIdx.x; i < E / 2; i += T) {  // 16-byte pieces of COLS-word row segments
            const int r = (2 * i) / COLS, c = (2 * i) % COLS;
            cp_async16(sh + slot * E + 2 * i, src + (size_t)r * N2 + c0 + c);
        }
        const typename A::Tw *tw = tw_all + (size_t)pr * N;
        for (int i = threadIdx.x; i < M; i += T) cp_async16(stw + slot * M + i, tw + i);
        cp_async_commit();
    };
    int t = blockIdx.x, slot = 0;
    if (t < n_tiles) prefetch(t, 0);
    for (; t < n_tiles; t += gridDim.x, slot ^= 1) {
        const int tn = t + gridDim.x;
        if (tn < n_tiles) {
            prefetch(tn, slot ^ 1);
            cp_async_wait_all_but_one();
        } else {
            cp_async_wait_all();
        }
        __syncthreads();
        const TileId id = tile_of(t, nb, R.n_rows);
        const typename A::Prime P = primes[R.prime[id.row]];
        uint64_t *dst = R.dst + (size_t)id.g * R.dst_gs + (size_t)R.dst_off[id.row] * N;
        const int c0 = id.bx * COLS;
        uint64_t *b = sh + slot * E;
        const typename A::Tw *tws = stw + slot * M;
        if (!INV) {
            ntt_pass<A, LOGM, R1, 0, false, true, false, kFwdIn>(b, COLS, 1, COLS, tws, 0, 0, 0, P, T);
            __syncthreads();
            ntt_pass_out<A, LOGM, R2, R1, COLS, false>(b, tws, P, dst + c0, N2, T);
        } else {
            ntt_pass<A, LOGM, R2, R1, true, true, false, kFoldSettled>(b, COLS, 1, COLS, tws, 0, 0, 0, P, T);
            __syncthreads();
            ntt_pass_out<A, LOGM, R1, 0, COLS, true>(b, tws, P, dst + c0, N2, T);
        }
        __syncthreads();  // this half is refilled by the prefetch two tiles later
    }
}

// row phase: the remaining LOGM stages on ROWS contiguous blocks of M words per tile
// (padded layout, one spare word per 16), next tile prefetched in 8-byte pieces
template <class A, int LOGM, int ROWS, bool INV, bool ALT>
__global__ void __launch_bounds__((1 << (LOGM - Split<LOGM, ALT>::R1)) * ROWS)
k_ntt_rows(const __grid_constant__ NttRows R, const typename A::Prime *__restrict__ primes,
           const typename A::Tw *__restrict__ tw_all, int log_n, int n_tiles)
{
    constexpr int M = 1 << LOGM, E = M * ROWS, R1 = Split<LOGM, ALT>::R1, R2 = Split<LOGM, ALT>::R2;
    constexpr int T = (M >> R1) * ROWS;
    constexpr int SK = M + M / 8;  // padded block stride (two spare words per 16)
    extern __shared__ uint64_t sh[];
    const int N = 1 << log_n;
    const int g0 = log_n - LOGM;
    const int nb = (N >> LOGM) / ROWS;
    auto prefetch = [&](int t, int slot) {
        const TileId id = tile_of(t, nb, R.n_rows);
        const uint64_t *src = INV ? R.src + (size_t)id.g * R.src_gs + (size_t)R.src_off[id.row] * N
                                  : R.dst + (size_t)id.g * R.dst_gs + (size_t)R.dst_off[id.row] * N;
        const size_t base = (size_t)id.bx * ROWS * M;
        for (int i = threadIdx.x; i < E / 2; i += T) {  // 16-byte pieces: pairs stay in one padding group
            const int k = (2 * i) / M, e = (2 * i) % M;
            cp_async16(sh + slot * ROWS * SK + k * SK + e + 2 * (e >> 4), src + base + 2 * i);
        }
        cp_async_commit();
    };
    int t = blockIdx.x, slot = 0;
    if (t < n_tiles) prefetch(t, 0);
    for (; t < n_tiles; t += gridDim.x, slot ^= 1) {
        const int tn = t + gridDim.x;
        if (tn < n_tiles) {
            prefetch(tn, slot ^ 1);
            cp_async_wait_all_but_one();
        } else {
            cp_async_wait_all();
        }
        __syncthreads();
        const TileId id = tile_of(t, nb, R.n_rows);
        const int pr = R.prime[id.row];
        const typename A::Prime P = primes[pr];
        const typename A::Tw *tw = tw_all + (size_t)pr * N;
        uint64_t *dst = R.dst + (size_t)id.g * R.dst_gs + (size_t)R.dst_off[id.row] * N;
        const int r_base = id.bx * ROWS;
        const size_t base = (size_t)r_base * M;
        uint64_t *b = sh + slot * ROWS * SK;
        if (!INV) {
            ntt_pass<A, LOGM, R1, 0, false, false, true, kFoldSettled>(b, ROWS, SK, 1, tw, g0, r_base, 1, P, T);
            __syncthreads();
            ntt_pass<A, LOGM, R2, R1, false, false, true, kFoldSettled, false>(b, ROWS, SK, 1, tw, g0, r_base, 1, P, T);
            __syncthreads();
            for (int i = threadIdx.x; i < E / 2; i += T) {  // pairs (e even, e+1) share a padding group
                const int k = (2 * i) / M, e = (2 * i) % M;
                const int sidx = k * SK + e + 2 * (e >> 4);
                *reinterpret_cast<ulonglong2 *>(dst + base + 2 * i) =
                    make_ulonglong2(A::finish(b[sidx], P), A::finish(b[sidx + 1], P));
            }
        } else {
            ntt_pass<A, LOGM, R2, R1, true, false, true, kInvIn>(b, ROWS, SK, 1, tw, g0, r_base, 1, P, T);
            __syncthreads();
            ntt_pass<A, LOGM, R1, 0, true, false, true, kFoldSettled>(b, ROWS, SK, 1, tw, g0, r_base, 1, P, T);
            __syncthreads();
            for (int i = threadIdx.x; i < E / 2; i += T) {
                const int k = (2 * i) / M, e = (2 * i) % M;
                const int sidx = k * SK + e + 2 * (e >> 4);
                *reinterpret_cast<ulonglong2 *>(dst + base + 2 * i) = make_ulonglong2(b[sidx], b[sidx + 1]);
            }
        }
        __syncthreads();
    }
}

// tile widths the autotuner chooses from (sub-transforms per block); a variant is a width index
// plus NTT_WIDTHS if the phase's two register passes swap radices (odd phase sizes only)
constexpr const int *kNttTiles = kNttTileWidths;

template <class A, int LOGM, int COLS, bool INV, bool ALT>
void ntt_cols_w(const LaunchCtx &c, const NttRows &rows)
{
    constexpr int M = 1 << LOGM;
    constexpr int E = M * COLS;
    constexpr int T = (M >> Split<LOGM, ALT>::R1) * COLS;
    const int N2 = c.N >> LOGM;
    HX_CHECK(N2 % COLS == 0, HX_EINVAL, "NTT tile wider than the ring");
    const long long n_tiles = (long long)(N2 / COLS) * rows.n_rows * rows.n_groups;
    HX_CHECK(n_tiles < (1ll << 31), HX_EINVAL, "NTT batch too large");
    const size_t smem = (size_t)E * 16 + (size_t)M * 32;  // two tiles + two twiddle sets
    static const bool attr =  // thread-safe one-time setup
        cudaFuncSetAttribute(k_ntt_cols<A, LOGM, COLS, INV, ALT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) == cudaSuccess;
    (void)attr;
    static const int per_sm = [&] {
        int v = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_ntt_cols<A, LOGM, COLS, INV, ALT>, T, smem);
        return v;
    }();
    const int grid = (int)std::min<long long>(n_tiles, (long long)std::max(1, per_sm) * c.t->n_sm);
    k_ntt_cols<A, LOGM, COLS, INV, ALT><<<grid, T, smem, c.stream>>>(rows, A::primes(*c.t), A::twiddles(*c.t, INV), c.log_n,
                                                                 (int)n_tiles);
}

template <class A, int LOGM, int ROWS, bool INV, bool ALT>
void ntt_rows_w(const LaunchCtx &c, const NttRows &rows)
{
    constexpr int M = 1 << LOGM;
    constexpr int T = (M >> Split<LOGM, ALT>::R1) * ROWS;
    const int N1 = c.N >> LOGM;
    HX_CHECK(N1 % ROWS == 0, HX_EINVAL, "NTT tile wider than the ring");
    const long long n_tiles = (long long)(N1 / ROWS) * rows.n_rows * rows.n_groups;
    HX_CHECK(n_tiles < (1ll << 31), HX_EINVAL, "NTT batch too large");
    const size_t smem = (size_t)ROWS * (M + M / 8) * 16;  // two tiles
    static const bool attr =  // thread-safe one-time setup
        cudaFuncSetAttribute(k_ntt_rows<A, LOGM, ROWS, INV, ALT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) == cudaSuccess;
    (void)attr;
    static const int per_sm = [&] {
        int v = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_ntt_rows<A, LOGM, ROWS, INV, ALT>, T, smem);
        return v;
    }();
    const int grid = (int)std::min<long long>(n_tiles, (long long)std::max(1, per_sm) * c.t->n_sm);
    k_ntt_rows<A, LOGM, ROWS, INV, ALT><<<grid, T, smem, c.stream>>>(rows, A::primes(*c.t), A::twiddles(*c.t, INV), c.log_n,
                                                                 (int)n_tiles);
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
// A job is n_rows rows of one ring (its own N, primes and twiddles), transformed
// in place.  One persistent kernel per phase walks the tiles of every job, the
// next tile (and for the column phase its twiddles) streaming into the other
// half of shared memory while the current one is transformed; a tile's phase
// size picks the template instance, with the tile width chosen so every
// instance runs 128 threads.

constexpr int kMultiT = 128;
template <int LOGM> struct MultiW {  // tile width per phase size: (M >> R1) * W = 128 threads
    static constexpr int W = kMultiT / ((1 << LOGM) >> Split<LOGM>::R1);
};
constexpr int kMultiColsBuf = 2048 + 2 * 256;  // words: the largest column tile and its twiddles
constexpr int kMultiRowsBuf = 8 * (256 + 32);  // words: the largest padded row tile

template <class A> struct MultiTile {
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
    m.logm = cols ? J.log_n / 2 : J.log_n - J.log_n / 2;
    const int n = 1 << J.log_n;
    const int W = kMultiT / ((1 << m.logm) >> ((m.logm + 1) / 2));
    const int nb = (n >> m.logm) / W;
    const int r = local / nb;
    m.bx = local % nb;
    m.pr = J.prime[r % J.n_limbs];
    m.primes = A::job_primes(J);
    m.row = J.data + (size_t)r * n;
    m.tw = A::job_twiddles(J, inv) + (size_t)m.pr * n;
    return m;
}

template <class A, int LOGM>
__device__ void multi_cols_load(uint64_t *b, const MultiTile<A> &m)
{
    constexpr int M = 1 << LOGM, COLS = MultiW<LOGM>::W, E = M * COLS;
    const int N2 = (1 << m.log_n) >> LOGM, c0 = m.bx * COLS;
    typename A::Tw *stw = reinterpret_cast<typename A::Tw *>(b + 2048);
    for (int i = threadIdx.x; i < E / 2; i += kMultiT) {
        const int r = (2 * i) / COLS, c = (2 * i) % COLS;
        cp_async16(b + 2 * i, m.row + (size_t)r * N2 + c0 + c);
    }
    for (int i = threadIdx.x; i < M; i += kMultiT) cp_async16(stw + i, m.tw + i);
}

template <class A, int LOGM, bool INV>
__device__ void multi_cols_run(uint64_t *b, const MultiTile<A> &m, const typename A::Prime &P)
{
    constexpr int M = 1 << LOGM, COLS = MultiW<LOGM>::W, E = M * COLS;
    constexpr int R1 = Split<LOGM>::R1, R2 = Split<LOGM>::R2;
    const int N2 = (1 << m.log_n) >> LOGM, c0 = m.bx * COLS;
    const typename A::Tw *stw = reinterpret_cast<const typename A::Tw *>(b + 2048);
    // the column phase's output pass of the one-ring kernels: results from registers to global memory
    if (!INV) {
        ntt_pass<A, LOGM, R1, 0, false, true, false, kFwdIn>(b, COLS, 1, COLS, stw, 0, 0, 0, P, kMultiT);
        __syncthreads();
        ntt_pass_out<A, LOGM, R2, R1, COLS, false>(b, stw, P, m.row + c0, N2, kMultiT);
    } else {
        ntt_pass<A, LOGM, R2, R1, true, true, false, kFoldSettled>(b, COLS, 1, COLS, stw, 0, 0, 0, P, kMultiT);
        __syncthreads();
        ntt_pass_out<A, LOGM, R1, 0, COLS, true>(b, stw, P, m.row + c0, N2, kMultiT);
    }
}

template <class A, int LOGM>
__device__ void multi_rows_load(uint64_t *b, const MultiTile<A> &m)
{
    constexpr int M = 1 << LOGM, ROWS = MultiW<LOGM>::W, E = M * ROWS, SK = M + M / 8;
    const size_t base = (size_t)m.bx * ROWS * M;
    for (int i = threadIdx.x; i < E; i += kMultiT) {
        const int k = i / M, e = i % M;
        cp_async8(b + k * SK + e + 2 * (e >> 4), m.row + base + i);
    }
}

template <class A, int LOGM, bool INV>
__device__ void multi_rows_run(uint64_t *b, const MultiTile<A> &m, const typename A::Prime &P)
{
    constexpr int M = 1 << LOGM, ROWS = MultiW<LOGM>::W, E = M * ROWS, SK = M + M / 8;
    constexpr int R1 = Split<LOGM>::R1, R2 = Split<LOGM>::R2;
    const int g0 = m.log_n - LOGM, r_base = m.bx * ROWS;
    const size_t base = (size_t)r_base * M;
    if (!INV) {
        ntt_pass<A, LOGM, R1, 0, false, false, true, kFoldSettled>(b, ROWS, SK, 1, m.tw, g0, r_base, 1, P, kMultiT);
        __syncthreads();
        ntt_pass<A, LOGM, R2, R1, false, false, true, kFoldSettled, false>(b, ROWS, SK, 1, m.tw, g0, r_base, 1, P, kMultiT);
        __syncthreads();
        for (int i = threadIdx.x; i < E; i += kMultiT) {
            const int k = i / M, e = i % M;
            m.row[base + i] = A::finish(b[k * SK + e + 2 * (e >> 4)], P);
        }
    } else {
        ntt_pass<A, LOGM, R2, R1, true, false, true, kInvIn>(b, ROWS, SK, 1, m.tw, g0, r_base, 1, P, kMultiT);
        __syncthreads();
        ntt_pass<A, LOGM, R1, 0, true, false, true, kFoldSettled>(b, ROWS, SK, 1, m.tw, g0, r_base, 1, P, kMultiT);
        __syncthreads();
        for (int i = threadIdx.x; i < E; i += kMultiT) {
            const int k = i / M, e = i % M;
            m.row[base + i] = b[k * SK + e + 2 * (e >> 4)];
        }
    }
}

template <class A, bool INV, bool COLS_PHASE>
__global__ void __launch_bounds__(kMultiT) k_ntt_multi(const NttJob *__restrict__ jobs, int n_jobs, int n_tiles)
{
    extern __shared__ uint64_t sh[];
    constexpr int BUF = COLS_PHASE ? kMultiColsBuf : kMultiRowsBuf;
    auto load = [&](const MultiTile<A> &m, int slot) {
        uint64_t *b = sh + slot * BUF;
        switch (m.logm) {
        case 5: COLS_PHASE ? multi_cols_load<A, 5>(b, m) : multi_rows_load<A, 5>(b, m); break;
        case 6: COLS_PHASE ? multi_cols_load<A, 6>(b, m) : multi_rows_load<A, 6>(b, m); break;
        case 7: COLS_PHASE ? multi_cols_load<A, 7>(b, m) : multi_rows_load<A, 7>(b, m); break;
        default: COLS_PHASE ? multi_cols_load<A, 8>(b, m) : multi_rows_load<A, 8>(b, m); break;
        }
        cp_async_commit();
    };
    int t = blockIdx.x, slot = 0;
    MultiTile<A> cur{};
    if (t < n_tiles) {
        cur = multi_tile<A>(jobs, n_jobs, t, COLS_PHASE, INV);
        load(cur, 0);
    }
    for (; t < n_tiles; t += gridDim.x, slot ^= 1) {
        const int tn = t + gridDim.x;
        MultiTile<A> nxt{};
        if (tn < n_tiles) {
            nxt = multi_tile<A>(jobs, n_jobs, tn, COLS_PHASE, INV);
            load(nxt, slot ^ 1);
            cp_async_wait_all_but_one();
        } else {
            cp_async_wait_all();
        }
        __syncthreads();
        const typename A::Prime P = cur.primes[cur.pr];
        uint64_t *b = sh + slot * BUF;
        switch (cur.logm) {
        case 5: COLS_PHASE ? multi_cols_run<A, 5, INV>(b, cur, P) : multi_rows_run<A, 5, INV>(b, cur, P); break;
        case 6: COLS_PHASE ? multi_cols_run<A, 6, INV>(b, cur, P) : multi_rows_run<A, 6, INV>(b, cur, P); break;
        case 7: COLS_PHASE ? multi_cols_run<A, 7, INV>(b, cur, P) : multi_rows_run<A, 7, INV>(b, cur, P); break;
        default: COLS_PHASE ? multi_cols_run<A, 8, INV>(b, cur, P) : multi_rows_run<A, 8, INV>(b, cur, P); break;
        }
        __syncthreads();  // this half is refilled by the prefetch two tiles later
        cur = nxt;
    }
}


} // namespace

// both phases of the several-ring transform over a job table on the device
template <class A> void ntt_multi_phases(cudaStream_t s, const NttJob *jp, int n_jobs, int tc, int tr, bool inverse, int n_sm)
{
    // two halves of shared memory per block (current tile, next tile)
    const size_t smem_c = 2 * sizeof(uint64_t) * kMultiColsBuf, smem_r = 2 * sizeof(uint64_t) * kMultiRowsBuf;
    const int grid_c = std::min(tc, n_sm * 8), grid_r = std::min(tr, n_sm * 8);
    if (!inverse) {
        k_ntt_multi<A, false, true><<<grid_c, kMultiT, smem_c, s>>>(jp, n_jobs, tc);
        k_ntt_multi<A, false, false><<<grid_r, kMultiT, smem_r, s>>>(jp, n_jobs, tr);
    } else {
        k_ntt_multi<A, true, false><<<grid_r, kMultiT, smem_r, s>>>(jp, n_jobs, tr);
        k_ntt_multi<A, true, true><<<grid_c, kMultiT, smem_c, s>>>(jp, n_jobs, tc);
    }
}

// ---- end of the several-ring kernels

} // namespace hx
