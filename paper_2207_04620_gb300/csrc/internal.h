// Internal structures shared by the host runtime and the kernel launchers.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <map>
#include <memory>
#include <string>
#include <vector>

#include "../../include/hx.h"
#include "modarith.cuh"
#include "modfold.cuh"

namespace hx {

constexpr int MAXP = HX_MAX_Q + HX_MAX_P;
constexpr int MAXK = HX_MAX_P + 1;  // conversion sources: the special primes, plus q_top when RS joins ModDown
constexpr int MAX_NTT_ROWS = 1024;
constexpr int NTT_WIDTHS = 4;    // tile widths 4, 8, 16, 32 (sub-transforms per block)
constexpr int kNttTileWidths[NTT_WIDTHS] = {4, 8, 16, 32};
constexpr int NTT_VARIANTS = 2 * NTT_WIDTHS;  // a width, with the register passes' radices as is or swapped
// NTT batch sizes tuned separately: a launch of n limbs uses the first bucket with n <= its bound
constexpr int NTT_BUCKETS = 4;
// Untuned, the column phase takes the larger half of an odd log N from 2^13 on: its threads of a warp
// share their twiddles, a row phase's do not, and the L1 pipe that returns them is as busy as the
// multiply pipe.  1200 rows of N = 2^15 take 294 us forward and 309 inverse instead of 326 and 359,
// 3200 of N = 2^13 177 and 189 instead of 190 and 201; 960 of N = 2^11 15.9 instead of 15.3, so there
// the smaller half stays.
__host__ __device__ constexpr int ntt_default_split(int log_n) { return (log_n & 1) && log_n >= 13 ? 1 : 0; }
// Untuned tile widths: 8 for a phase of 256 points, else 16, blocks of 128 threads either way (400 rows of
// N = 2^16 228 us forward and 243 inverse, 236 and 258 with blocks of 256)
constexpr int ntt_default_var(int logm) { return logm >= 8 ? 1 : 2; }
inline void ntt_defaults(int log_n, int (&v)[5])
{
    const int cols = log_n / 2 + ntt_default_split(log_n), rows = log_n - cols;
    v[0] = v[2] = ntt_default_var(cols);
    v[1] = v[3] = ntt_default_var(rows);
    v[4] = ntt_default_split(log_n);
}
constexpr int kNttBucketMax[NTT_BUCKETS] = {64, 256, 768, 1 << 30};
constexpr int kNttBucketTune[NTT_BUCKETS] = {48, 176, 512, 1024};  // limbs timed for each bucket
inline int ntt_bucket(long long limbs)
{
    int b = 0;
    while (b < NTT_BUCKETS - 1 && limbs > kNttBucketMax[b]) b++;
    return b;
}

// Fast basis conversion table (Han-Ki hybrid key switching, no correction):
// out_t = sum_i [x_i * qhat_i^-1]_{q_i} * (qhat_i mod t)  (mod t), every term a Shoup product
struct ConvTable {
    int n_src, n_dst;
    int src_row[MAXK];        // rows of the source buffer
    int src_prime[MAXK];      // prime indices (Q then P)
    int dst_row[MAXP];        // rows of the destination buffer
    int dst_prime[MAXP];
    uint64_t inv[MAXK], inv_sh[MAXK];   // [qhat_i^-1]_{q_i} with Shoup companion
    uint64_t w[MAXK][MAXP], w_sh[MAXK][MAXP];  // qhat_i mod t with its Shoup companion
    // shift != 0: the rounded division's remainder.  Convert x + h exactly (the overshoot
    // u = floor(sum_i y_i / q_i), summed in FP64, times the source product is removed),
    // then subtract h
    int shift;
    uint64_t add_src[MAXK];             // h mod q_i
    double inv_d[MAXK];                 // 1 / q_i in FP64
    uint64_t sub_dst[MAXP];             // h mod t
    uint64_t prod_mod[MAXP];            // (product of the sources) mod t
    // the same constants for chains with fold arithmetic: inv as fold constants; w, -prod_mod and
    // -sub_dst times 2^60 and split at bit 30; 2^(31 + bits) / q_i for the overshoot's estimate
    int4 inv_f[MAXK];
    uint64_t w30[MAXK][MAXP], neg_prod30[MAXP], neg_sub30[MAXP];
    uint32_t recip[MAXK];
    int bits[MAXK];
};

struct ModDownTable {
    ConvTable conv;                      // P -> Q_l
    uint64_t pinv[MAXP], pinv_sh[MAXP];  // P^-1 mod q_i, Shoup
};

// relinearisation and rescale in one division by P * q_top (limbs l -> l-1)
struct RelinRescaleTable {
    ConvTable conv;                      // {q_top, P} -> Q_{l-1}, shifted by h = floor(P q_top / 2)
    uint64_t pmod[MAXP], pmod_sh[MAXP];  // P mod q_i, i < l
    uint64_t pqinv[MAXP], pqinv_sh[MAXP];  // (P q_top)^-1 mod q_i, i < l-1
};

struct RescaleTable {
    uint64_t half;                                   // floor(q_top / 2)
    uint64_t qinv[MAXP], qinv_sh[MAXP];              // q_top^-1 mod q_i
    uint64_t half_mod[MAXP];                         // half mod q_i
};

// Rows of a batched NTT: for group g in [0,n_groups) and row r in
// [0,n_rows), the source row is src + g*src_gs + src_off[r]*N and the
// destination row dst + g*dst_gs + dst_off[r]*N (equal for in-place use),
// taken modulo prime index prime[r].
struct NttRows {
    const uint64_t *src;
    uint64_t *dst;
    size_t src_gs, dst_gs;
    int n_groups;
    int n_rows;
    int16_t src_off[MAX_NTT_ROWS];
    int16_t dst_off[MAX_NTT_ROWS];
    int16_t prime[MAX_NTT_ROWS];
};

struct Scalars {
    uint64_t v[MAXP], sh[MAXP];
};

// Inner sums of a baby-step/giant-step linear transform: for every group g,
// out_g = sum_m baby_m (.) mask[g][m] over the babies whose mask is present.
constexpr int MAC_MAX_BABY = 16, MAC_MAX_GROUP = 32;
struct MacArgs {
    int n_baby, n_group;
    const uint64_t *baby[MAC_MAX_BABY];
    size_t baby_bstride, baby_cstride;
    const uint64_t *mask[MAC_MAX_GROUP][MAC_MAX_BABY];  // Montgomery form, [limbs][N]; null if absent
    uint64_t *out;                                      // [group][B][2][limbs][N]
};

// A batch of polynomials with `comps` components of `limbs` rows each:
// word (b, c, l, j) at p + b*bstride + c*cstride + l*N + j.
struct View {
    uint64_t *p;
    size_t bstride, cstride;
};

// copies of one launch
constexpr int MAX_COPIES = 128;
struct CopyPair {
    uint64_t *dst;
    const uint64_t *src;
};
struct CopyTab {
    const uint64_t *src[MAX_COPIES];
    uint64_t *dst[MAX_COPIES];
};

// what follows a rescale's division x in the same pass: w x + add_w add + c0 (c0 on component 0)
struct RescaleTail {
    Scalars w, add_w, c0;
    View add;
    int has_w, has_add;  // 0: none (a factor 1, no addend), 1: as it is, 2: times add_w
};

struct DeviceTables {
    PrimeConst *primes = nullptr;   // [n_all]
    ulonglong2 *tw_fwd = nullptr;   // [n_all][N] (psi^brv(k), Shoup)
    ulonglong2 *tw_inv = nullptr;   // [n_all][N] (psi^-brv(k), Shoup)
    // the same for fold arithmetic; null unless every prime of the chain allows it
    FoldPrime *fold = nullptr;      // [n_all]
    int4 *ftw_fwd = nullptr;        // [n_all][N] psi^brv(k)
    int4 *ftw_inv = nullptr;        // [n_all][N] psi^-brv(k)
    ConvTable *modup = nullptr;     // [(n_q+1) * dnum] by (limbs, digit)
    ModDownTable *moddown = nullptr;// [n_q+1] by limbs
    RescaleTable *rescale = nullptr;// [n_q+1] by limbs
    RelinRescaleTable *relin_rs = nullptr;  // [n_q+1] by limbs
    // NTT variants per batch-size bucket: the four phases' (forward column, forward row, inverse column, inverse
    // row), then the split of an odd log N (0: the column phase takes floor(log N / 2) stages, 1: ceil)
    int ntt_var[NTT_BUCKETS][5];
    int n_sm = 1;                   // multiprocessors of the device
};

// Per-kernel-class timing with CUDA events recorded on the launching stream
// (enabled only while profiling; the events bracket every launch of a class).
struct Profiler {
    struct Rec {
        int cls;
        cudaEvent_t a, b;
        double bytes;
    };
    std::vector<Rec> recs;
    std::vector<cudaEvent_t> pool;
    cudaEvent_t get();
    void clear();
};
enum KClass { K_NTT, K_KEYIP, K_CONV, K_MODDOWN, K_RESCALE, K_TENSOR, K_MULPT, K_ELEM, K_AUTO, K_AGG, K_MISC, K_NCLASS };
extern const char *const kclass_names[K_NCLASS];

// ---- kernel launchers (kernels.cu) ----------------------------------------------
struct LaunchCtx {
    int log_n, N;
    const DeviceTables *t;
    cudaStream_t stream;
    std::atomic<uint64_t> *launches;
    Profiler *prof = nullptr;
};

void launch_ntt(const LaunchCtx &c, const NttRows &rows, bool inverse);
// one job of a multi-ring NTT: n_rows rows of 2^log_n words from src to data (they may be the same),
// row r modulo prime[r % n_limbs] of its own context's tables
struct NttJob {
    const uint64_t *src;
    uint64_t *data;
    const PrimeConst *primes;
    const ulonglong2 *tw_fwd, *tw_inv;
    const FoldPrime *fold;            // null: the ring has no fold tables
    const int4 *ftw_fwd, *ftw_inv;
    int log_n, n_rows, n_limbs;
    int tile0_cols, tile0_rows;  // filled by the launcher
    int16_t prime[64];
};
// every job's transform in one launch per phase (several ring degrees together)
void launch_ntt_multi(cudaStream_t s, const std::vector<NttJob> &jobs, bool inverse,
                      std::atomic<uint64_t> *launches);

// times every NTT variant (tile width, radix split) of each phase on `rows` limbs of buf and
// writes the fastest per phase
void autotune_ntt(const LaunchCtx &c, uint64_t *buf, int rows, int *best, float *ms_out);
void launch_add(const LaunchCtx &c, View out, View a, View b, int B, int comps, int limbs, bool sub);
void launch_copy(const LaunchCtx &c, View out, View a, int B, int comps, int limbs);
// words of each pair (a multiple of 2^11), the pairs' buffers disjoint
void launch_copies(const LaunchCtx &c, const std::vector<CopyPair> &copies, size_t words);
// one ciphertext read in place: component c, limb l at p + c*cstride + l*N
struct AggSrc {
    const uint64_t *p;
    uint64_t cstride;
};
// out[m] = C * sum_i src[i*count + m] (per limb, C given as Scalars), for m < count
void launch_aggregate(const LaunchCtx &c, View out, const AggSrc *src_dev, int n_parties, int count, int comps,
                      int limbs, const Scalars &C);
void launch_mul_plain(const LaunchCtx &c, View out, View a, const uint64_t *pt_mont, int B, int limbs);
void launch_mul_scalar(const LaunchCtx &c, View out, View a, const Scalars &sc, int B, int comps, int limbs);
void launch_add_scalar_c0(const LaunchCtx &c, View out, View a, const Scalars &sc, int B, int limbs);
// mont: the products left times 2^-64 (Montgomery reductions), to be scaled back once after summing
void launch_tensor(const LaunchCtx &c, View out3, View a, View b, int B, int limbs, bool mont = false);
// Rotations of one launch, by their place in the batch: entry e of R * per entries belongs to
// rotation e / per, so a schedule's rotations by different amounts share a launch per stage
constexpr int MAX_ROT = 32;
struct GaloisTab {
    int per;
    uint32_t g[MAX_ROT];
};
struct KeyTab {
    const uint64_t *key[MAX_ROT];
    uint32_t g[MAX_ROT];
};
// selections between two rotations (Step 2): their keys (k1 alone: premasked ones), masks and elements
constexpr int MAX_MUX = 16;
struct MuxTab {
    const uint64_t *k1[MAX_MUX], *k2[MAX_MUX], *v[MAX_MUX];
    uint32_t g1[MAX_MUX], g2[MAX_MUX];
};
// where the entries of one launch's rotations go: those of rotation r follow one another from p[r]
struct OutTab {
    uint64_t *p[MAX_ROT];
    size_t bstride, cstride;
};
// all R rotations of `per` entries in one batch
inline OutTab batch_out(const View &v, int per, int R = 1)
{
    OutTab t;
    t.bstride = v.bstride;
    t.cstride = v.cstride;
    for (int r = 0; r < R; r++) t.p[r] = v.p + (size_t)r * per * v.bstride;
    return t;
}
inline GaloisTab one_galois(uint64_t g, int B)
{
    GaloisTab t;
    t.per = B;
    t.g[0] = (uint32_t)g;
    return t;
}
// entry e of `out` = sigma_g(entry e of `in`), g = tab.g[e / tab.per]
void launch_automorphism(const LaunchCtx &c, View out, View in, const GaloisTab &tab, int B, int comps, int limbs);
// out[b] += sum over r < R of sigma_g[r](in[r * B + b]), component 0
void launch_automorphism_sum(const LaunchCtx &c, View out, View in, const GaloisTab &tab, int R, int B, int limbs);
// alg_bytes: one read of every source row and one write of every destination row (profiling)
void launch_basis_convert(const LaunchCtx &c, const ConvTable *tab_dev, int max_src, View out, View in, int B,
                          int groups, size_t gstride_out, size_t gstride_in, double alg_bytes = 0.0);
// Inner products of R rotations of B entries: entry r * B + b of acc from D and dnt of that entry, or
// of entry b for every r (shared: hoisted rotations of one batch); sum: entry b the sum over r
void launch_key_ip(const LaunchCtx &c, View acc, const uint64_t *D, const uint64_t *dnt, size_t dnt_bstride,
                   const KeyTab &keys, int R, bool shared, bool sum, int n_all, int n_q, int K, int alpha, int limbs,
                   int ndig, int B, bool accumulate = false);
// out_c = (acc_c - conv_c) * P^-1, plus add_c[galois(j)] for the components set in add_mask; entry e
// adds entry e of add, or (shared) entry e % tab.per.  The results go where `out` says by rotation
void launch_moddown_final(const LaunchCtx &c, const OutTab &out, View acc, View conv, const ModDownTable *tab, int B,
                          int limbs, View add, int add_mask, const GaloisTab &gal, bool shared = false);

// ---- several rings in one launch per key-switching stage (one job = one ring's batch) ----------
// Each kernel runs the body of its one-ring counterpart over every job: a flat grid whose block
// b belongs to the job with the largest block0 <= b, at the coordinates that job's own grid
// (gx, gy, gz) would give it.
struct AutomorphismJob {
    View out, in;
    uint64_t g;
    int comps, log_n;
    int gx, gy, gz;
    long long block0;
};
struct ConvertJob {
    const ConvTable *tabs;
    View out, in;
    const PrimeConst *primes;
    const FoldPrime *fold;  // not null: by split sums
    int groups, n, max_src;
    size_t gstride_out, gstride_in;
    int gx, gy, gz;
    long long block0;
};
struct KeyIpJob {
    View acc;
    const uint64_t *D, *dnt, *key;
    size_t dnt_bstride;
    const PrimeConst *primes;
    const FoldPrime *fold;  // not null: split keys
    int n_all, n_q, K, alpha, limbs, ndig, log_n, few;
    uint64_t g;
    int gx, gy, gz;
    long long block0;
};
struct ModDownJob {
    View out, acc, conv, add;
    const ModDownTable *tab;
    const PrimeConst *primes;
    int add_mask, log_n;
    uint64_t g;
    int gx, gy, gz;
    long long block0;
};
// Fills every job's block0; returns the blocks of the grid over all of them.
template <class J> long long plan_job_blocks(std::vector<J> &jobs)
{
    long long total = 0;
    for (auto &j : jobs) {
        j.block0 = total;
        total += (long long)j.gx * j.gy * j.gz;
    }
    return total;
}
// one grid over the jobs of a table already on the device (blocks from plan_job_blocks)
void launch_automorphism_jobs(cudaStream_t s, const AutomorphismJob *jobs, int n_jobs, long long blocks,
                              std::atomic<uint64_t> *launches);
void launch_convert_jobs(cudaStream_t s, const ConvertJob *jobs, int n_jobs, long long blocks, int max_src,
                         std::atomic<uint64_t> *launches);
void launch_key_ip_jobs(cudaStream_t s, const KeyIpJob *jobs, int n_jobs, long long blocks,
                        std::atomic<uint64_t> *launches);
void launch_moddown_jobs(cudaStream_t s, const ModDownJob *jobs, int n_jobs, long long blocks,
                         std::atomic<uint64_t> *launches);
// the NTT over several rings in two steps: tile offsets of every job (host), then the two phase
// launches over a job table already on the device
void plan_ntt_jobs(std::vector<NttJob> &jobs, int *tiles_cols, int *tiles_rows);
// fold: every job's ring has fold tables
void launch_ntt_jobs(cudaStream_t s, const NttJob *jobs, int n_jobs, int tiles_cols, int tiles_rows, bool fold,
                     bool inverse, std::atomic<uint64_t> *launches);
// the tables of a context that its NTT jobs carry
inline void set_ntt_tables(NttJob &j, const DeviceTables &t)
{
    j.primes = t.primes;
    j.tw_fwd = t.tw_fwd;
    j.tw_inv = t.tw_inv;
    j.fold = t.fold;
    j.ftw_fwd = t.ftw_fwd;
    j.ftw_inv = t.ftw_inv;
}
void launch_lintrans_mac(const LaunchCtx &c, const MacArgs &a, int B, int limbs, int n_terms);
// C selections, each between two hoisted rotations by a mask in the extended basis (see kernels.cu):
// entry i * B + b of out from entry b of D
void launch_key_ip_mux(const LaunchCtx &c, View out, const uint64_t *D, const uint64_t *dnt, size_t dnt_bstride,
                       const MuxTab &tab, int C, const Scalars &cs, int n_all, int n_q, int K, int alpha, int limbs,
                       int ndig, int B);
// premasked keys of one selection: out = [2][ndig][2][ext][N] with
// out[0] = v (.) key1, out[1] = (c - v) (.) key2 on the rows of the extended basis (Montgomery form);
// cR[t] = c * 2^64 mod (prime of row t)
void launch_premask_keys(const LaunchCtx &c, uint64_t *out, const uint64_t *key1, const uint64_t *key2,
                         const uint64_t *v, const Scalars &cR, int n_all, int n_q, int K, int limbs, int ndig);
// the inner products of C selections with premasked keys: z_h = sum_d sigma_g1(D_d) pk[0][d][h]
// + sigma_g2(D_d) pk[1][d][h], one reduction
void launch_key_ip_mux_pm(const LaunchCtx &c, View out, const uint64_t *D, const uint64_t *dnt, size_t dnt_bstride,
                          const MuxTab &tab, int C, int n_q, int K, int alpha, int limbs, int ndig, int B);
// measured rates of Shoup products and 128-bit multiply-accumulates on every SM (per second)
void alu_calibrate(const LaunchCtx &c, uint64_t q, double *shoup_per_s, double *mac_per_s);
// their ModDown epilogue (v's chain rows start K rows in)
void launch_moddown_final_mux(const LaunchCtx &c, View out, View acc, View conv, const ModDownTable *tab, int C, int B,
                              int K, int limbs, View src, const MuxTab &mux, const Scalars &cs);
// out += sum over i < C of a[i * B + b] x b[i * B + b] (3 components), each product times 2^-64
void launch_tensor_sum(const LaunchCtx &c, View out3, View a, View b, int C, int B, int limbs);
// prefix sums P_m = sum_{l < m} T_l (T_0 = mask_0 b, T_l = mask_l rb[(l-1) B + b]): out[(h - m) B + b] = P_m
struct PrefixTab {
    const uint64_t *mask[256];
};
void launch_mask_prefix(const LaunchCtx &c, View out, View b, View rb, const PrefixTab &tab, int h, int B, int limbs);
// out[(2 i) B + b] = P_(h-k), out[(2 i + 1) B + b] = P_h - P_(h-k) for k = k0 + i, i < C, of the sums above
void launch_prefix_pairs(const LaunchCtx &c, View out, View prefix, int k0, int C, int B, int limbs);
// slots[r*S + t*beta + j] = bits[r*hh + t] for j < beta (masks expanded over the packed matrices)
void launch_expand_masks(const LaunchCtx &c, double *slots, const uint8_t *bits, int m, int hh, int beta, size_t S);
void launch_relin_rs_top(const LaunchCtx &c, View acc, View d, const RelinRescaleTable *tab, int B, int limbs);
void launch_relin_rs_final(const LaunchCtx &c, View out, View acc, View d, View conv, const RelinRescaleTable *tab,
                           int B, int limbs);
void launch_rescale_prep(const LaunchCtx &c, View r, View xtop, const RescaleTable *tab, int B, int comps, int top,
                         const Scalars *sc = nullptr);
void launch_rescale_centre(const LaunchCtx &c, uint64_t *xtop, const RescaleTable *tab, uint64_t qt, int rows,
                           uint64_t s, uint64_t ssh, bool scaled);
void launch_rescale_final(const LaunchCtx &c, View out, View in, View r, const RescaleTable *tab, int B, int comps,
                          int top, const Scalars *sc = nullptr);
void launch_rescale_tail(const LaunchCtx &c, View out, View in, View r, const RescaleTable *tab, const Scalars &sc,
                         const RescaleTail &tail, int B, int comps, int top);
void launch_keygen_b(const LaunchCtx &c, uint64_t *b, const uint64_t *a, const uint64_t *e, const uint64_t *s,
                     const uint64_t *sp, const uint64_t *gadget_mask, int rows, const int *prime_of_row_dev,
                     bool to_mont);
void launch_encrypt_combine(const LaunchCtx &c, uint64_t *ct, const uint64_t *v, const uint64_t *e0,
                            const uint64_t *e1, const uint64_t *m, const uint64_t *pk, int n_q, int limbs,
                            int count = 1, size_t stride = 0);  // count entries, their polynomials stride words apart
void launch_signed_to_rows(const LaunchCtx &c, uint64_t *out, const int64_t *in, int rows, int n_in_polys,
                           size_t in_stride, const int *prime_dev);
void launch_to_mont(const LaunchCtx &c, uint64_t *p, int rows, const int *prime_dev);

// ---- error handling -------------------------------------------------------------
void set_error(const std::string &msg);
struct Error {
    hx_status code;
    std::string msg;
};
#define HX_CUDA(call)                                                                                      \
    do {                                                                                                   \
        cudaError_t e_ = (call);                                                                           \
        if (e_ != cudaSuccess)                                                                             \
            throw ::hx::Error{HX_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)};              \
    } while (0)
#define HX_CHECK(cond, code, msg)                                                                          \
    do {                                                                                                   \
        if (!(cond)) throw ::hx::Error{code, msg};                                                         \
    } while (0)

} // namespace hx

namespace hx {
// rows r of out/a/b modulo prime r: out = a * b
void launch_mul_rows(const LaunchCtx &c, uint64_t *out, const uint64_t *a, const uint64_t *b, int rows);
// out[b][0] = c0 limb 0, out[b][1+p] = c1 limb 0 * share_p (NTT form, prime 0)
void launch_ddec_shares(const LaunchCtx &c, uint64_t *out, View ct, const uint64_t *shares, int n_parties, int B);
} // namespace hx
