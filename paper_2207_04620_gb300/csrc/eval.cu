// Batched homomorphic evaluation (Fig. 1 items 7-12).  Every operation acts on
// a batch of B ciphertexts with one launch per kernel; hybrid key switching is
// ModUp (iNTT, fast basis conversion per digit, NTT) -> key inner product ->
// ModDown (iNTT of the special limbs, conversion P -> Q_l, NTT, subtract and
// multiply by P^-1).
#include <algorithm>
#include <cmath>

#include "runtime.h"

namespace hx {

Cts Eval::alloc(int B, int comps, int limbs)
{
    Cts c;
    c.B = B;
    c.comps = comps;
    c.limbs = limbs;
    c.cap = limbs;
    c.buf = std::make_shared<DevBuf>((size_t)B * comps * limbs * ctx.N, s);
    c.d = c.buf->p;
    return c;
}

void Eval::check_same(const Cts &a, const Cts &b)
{
    HX_CHECK(a.B == b.B, HX_EINVAL, "batch sizes differ");
    HX_CHECK(a.limbs == b.limbs, HX_ESCALE, "level mismatch");
    HX_CHECK(std::fabs(a.scale / b.scale - 1.0) <= std::ldexp(1.0, -20), HX_ESCALE, "scale mismatch");
}

Cts Eval::add(const Cts &a, const Cts &b, bool sub)
{
    check_same(a, b);
    HX_CHECK(a.comps == b.comps, HX_EINVAL, "component count mismatch");
    Cts o = alloc(a.B, a.comps, a.limbs);
    o.scale = a.scale;
    launch_add(lc(), o.view(ctx.N), a.view(ctx.N), b.view(ctx.N), a.B, a.comps, a.limbs, sub);
    ctx.counters[C_ADD] += a.B;
    return o;
}

void Eval::add_inplace(Cts &a, const Cts &b)
{
    check_same(a, b);
    launch_add(lc(), a.view(ctx.N), a.view(ctx.N), b.view(ctx.N), a.B, a.comps, a.limbs, false);
    ctx.counters[C_ADD] += a.B;
}

Cts Eval::mul_plain(const Cts &a, const uint64_t *pt, double pt_scale)
{
    HX_CHECK(a.comps == 2, HX_EINVAL, "Mul_pt needs a 2-component ciphertext");
    Cts o = alloc(a.B, 2, a.limbs);
    o.scale = a.scale * pt_scale;
    launch_mul_plain(lc(), o.view(ctx.N), a.view(ctx.N), pt, a.B, a.limbs);
    ctx.counters[C_MULPT] += a.B;
    return o;
}

Scalars scalars_for(const hx_context &ctx, int limbs, int64_t c)
{
    Scalars sc;
    for (int l = 0; l < limbs; l++) {
        const uint64_t q = ctx.primes[l];
        uint64_t v = c >= 0 ? (uint64_t)c % q : (q - ((uint64_t)(-(c + 1)) + 1) % q) % q;
        sc.v[l] = v;
        sc.sh[l] = shoup_companion(v, q);
    }
    return sc;
}

Cts Eval::mul_int(const Cts &a, int64_t c, double new_scale)
{
    Cts o = alloc(a.B, a.comps, a.limbs);
    o.scale = new_scale > 0 ? new_scale : a.scale;
    launch_mul_scalar(lc(), o.view(ctx.N), a.view(ctx.N), scalars_for(ctx, a.limbs, c), a.B, a.comps, a.limbs);
    return o;
}

int64_t const_int(double value, double scale)
{
    const double r = round_half_away(value * scale);
    HX_CHECK(std::fabs(r) < 9.2e18, HX_EINVAL, "constant too large");
    return (int64_t)r;
}

Cts Eval::add_const(const Cts &a, double value)
{
    const int64_t r = const_int(value, a.scale);
    Cts o = alloc(a.B, 2, a.limbs);
    o.scale = a.scale;
    launch_add_scalar_c0(lc(), o.view(ctx.N), a.view(ctx.N), scalars_for(ctx, a.limbs, r), a.B, a.limbs);
    return o;
}

Cts Eval::tensor(const Cts &a, const Cts &b, bool mont)
{
    HX_CHECK(a.B == b.B && a.limbs == b.limbs && a.comps == 2 && b.comps == 2, HX_ESCALE, "tensor operands differ");
    Cts o = alloc(a.B, 3, a.limbs);
    o.scale = a.scale * b.scale;
    launch_tensor(lc(), o.view(ctx.N), a.view(ctx.N), b.view(ctx.N), a.B, a.limbs, mont);
    ctx.counters[C_MULCT] += a.B;
    return o;
}

void Eval::from_mont(Cts &a)
{
    Scalars sc;
    for (int l = 0; l < a.limbs; l++) {
        sc.v[l] = ctx.h_primes[l].r_mod;  // 2^64 mod q_l
        sc.sh[l] = ctx.h_primes[l].r_mod_sh;
    }
    launch_mul_scalar(lc(), a.view(ctx.N), a.view(ctx.N), sc, a.B, a.comps, a.limbs);
}

Cts Eval::drop(const Cts &a, int limbs)
{
    HX_CHECK(limbs >= 1 && limbs <= a.limbs, HX_EINVAL, "bad level drop");
    Cts o = a;
    o.limbs = limbs;
    return o;
}

Cts Eval::copy(const Cts &a)
{
    Cts o = alloc(a.B, a.comps, a.limbs);
    o.scale = a.scale;
    launch_copy(lc(), o.view(ctx.N), a.view(ctx.N), a.B, a.comps, a.limbs);
    return o;
}

void Eval::ntt_inplace(uint64_t *p, size_t gstride, int groups, const std::vector<int> &off,
                       const std::vector<int> &prime, bool inverse)
{
    ntt_oop(p, gstride, p, gstride, groups, off, off, prime, inverse);
}

void Eval::ntt_oop(const uint64_t *src, size_t sgs, uint64_t *dst, size_t dgs, int groups,
                   const std::vector<int> &src_off, const std::vector<int> &dst_off, const std::vector<int> &prime,
                   bool inverse)
{
    if (prime.empty() || groups == 0) return;
    NttRows *r = new NttRows;
    std::unique_ptr<NttRows> guard(r);
    r->src = src;
    r->dst = dst;
    r->src_gs = sgs;
    r->dst_gs = dgs;
    r->n_groups = groups;
    HX_CHECK(prime.size() <= (size_t)MAX_NTT_ROWS, HX_EINVAL, "too many NTT rows");
    r->n_rows = (int)prime.size();
    for (size_t i = 0; i < prime.size(); i++) {
        r->src_off[i] = (int16_t)src_off[i];
        r->dst_off[i] = (int16_t)dst_off[i];
        r->prime[i] = (int16_t)prime[i];
    }
    launch_ntt(lc(), *r, inverse);
}

static std::vector<int> iota_vec(int a, int n)
{
    std::vector<int> v(n);
    for (int i = 0; i < n; i++) v[i] = a + i;
    return v;
}

BufPtr Eval::modup(const View &d, int B, int limbs)
{
    const int N = ctx.N, K = ctx.K, A = ctx.alpha, ext = limbs + K, nd = (limbs + A - 1) / A;
    DevBuf coef((size_t)B * limbs * N, s);
    ntt_oop(d.p, d.bstride, coef.p, (size_t)limbs * N, B, iota_vec(0, limbs), iota_vec(0, limbs), iota_vec(0, limbs),
            true);
    BufPtr D = std::make_shared<DevBuf>((size_t)B * nd * ext * N, s);
    launch_basis_convert(lc(), ctx.t.modup + (size_t)limbs * ctx.dnum, A, View{D->p, (size_t)nd * ext * N, 0},
                         View{coef.p, (size_t)limbs * N, 0}, B, nd, (size_t)ext * N, 0, 8.0 * N * B * nd * ext);
    std::vector<int> off, pr;
    for (int j = 0; j < nd; j++) {
        const int lo = j * A, hi = std::min((j + 1) * A, limbs);
        for (int r = 0; r < ext; r++) {
            if (r >= lo && r < hi) continue;
            off.push_back(j * ext + r);
            pr.push_back(r < limbs ? r : ctx.n_q + (r - limbs));
        }
    }
    ntt_inplace(D->p, (size_t)nd * ext * N, B, off, pr, false);
    ctx.counters[C_MODUP] += B;
    return D;
}

KeyTab one_key(const SwitchKey &key, uint64_t g)
{
    KeyTab t;
    t.key[0] = key.buf->p;
    t.g[0] = (uint32_t)g;
    return t;
}

Cts Eval::ks_finish(const BufPtr &D, const View &dnt, int B, int limbs, const SwitchKey &key, uint64_t g,
                    const View &add, int add_mask, uint64_t add_g)
{
    const int N = ctx.N, K = ctx.K, ext = limbs + K, nd = (limbs + ctx.alpha - 1) / ctx.alpha;
    DevBuf acc((size_t)B * 2 * ext * N, s);
    View accv{acc.p, (size_t)2 * ext * N, (size_t)ext * N};
    launch_key_ip(lc(), accv, D->p, dnt.p, dnt.bstride, one_key(key, g), 1, true, false, ctx.n_all, ctx.n_q, K, ctx.alpha,
                  limbs, nd, B);
    ctx.counters[C_KS] += B;
    Cts o = alloc(B, 2, limbs);
    moddown_add(batch_out(o.view(N), B), accv, B, limbs, add, add_mask, one_galois(add_g, B));
    return o;
}

void Eval::moddown_ntt(const View &accv, uint64_t *conv, int B, int limbs)
{
    const int N = ctx.N, K = ctx.K, ext = limbs + K;
    ntt_inplace(accv.p, (size_t)ext * N, 2 * B, iota_vec(limbs, K), iota_vec(ctx.n_q, K), true);
    launch_basis_convert(lc(), reinterpret_cast<const ConvTable *>(ctx.t.moddown + limbs), ctx.K,
                         View{conv, (size_t)limbs * N, 0}, View{accv.p, (size_t)ext * N, 0}, 2 * B, 1, 0, 0,
                         8.0 * N * 2 * B * (K + limbs));
    ntt_inplace(conv, (size_t)limbs * N, 2 * B, iota_vec(0, limbs), iota_vec(0, limbs), false);
}

void Eval::moddown_add(const OutTab &out, const View &accv, int B, int limbs, const View &add, int add_mask,
                       const GaloisTab &gal, bool shared)
{
    const int N = ctx.N;
    DevBuf conv((size_t)B * 2 * limbs * N, s);
    moddown_ntt(accv, conv.p, B, limbs);
    launch_moddown_final(lc(), out, accv, View{conv.p, (size_t)2 * limbs * N, (size_t)limbs * N}, ctx.t.moddown + limbs, B,
                         limbs, add, add_mask, gal, shared);
}

// Rotations (or selections) of a batch of B per launch: as many as keep the launch's buffer within
// 128 MB, about the size of GB300's L2, so that the stages that follow find most of it there.  Measured
// with 16, 32, 64, 128 and 256 MB: sixteen 64x64 pairs 21.9, 21.9, 21.9, 20.8 and 20.5 ms; five 32x32
// products 2.33, 2.11, 2.08, 2.03 and 2.03 ms; a small dense layer 10.6, 8.66, 8.07, 7.85 and 7.85 ms: past
// 128 the last 1.5 % of one of them would cost twice the memory.  (kGroupBytes; the call's limit may
// be lower, down to one rotation.)  One rotation of 16 entries of N = 2^14 (38 MB) already
// fills the GPU; one of a single entry of N = 2^12 takes a few SMs, and with a launch per stage and
// rotation the product of 16x16 matrices there waited on about 900 launches: 5.2 ms, 0.74 in groups
// (five 32x32 products of N = 2^13: 4.0 ms, 2.6; a small dense layer of N = 2^14: 23.2 ms, 11.0).
// A launch's entries times their digits, or their two components, lie in the z extent of a grid,
// which ends at 65535: `grid` stays at a quarter of it.
int Eval::rot_chunk(int B, int limbs, int most, size_t words)
{
    const size_t per = words ? words : (size_t)B * 2 * (limbs + ctx.K) * ctx.N;
    const int grid = std::max(1, 16384 / (B * std::max(2, (limbs + ctx.alpha - 1) / ctx.alpha)));
    return std::max(1, std::min({most, grid, (int)std::min<size_t>(MAX_ROT, group / 8 / per)}));
}

Cts Eval::rotate_sum(const Cts &items, const std::vector<int64_t> &steps, const hx_keyset &keys)
{
    HX_CHECK(!steps.empty() && items.B % steps.size() == 0, HX_EINVAL, "empty rotation sum");
    const int R = (int)steps.size(), B = items.B / R, N = ctx.N, K = ctx.K, limbs = items.limbs, ext = limbs + K,
              nd = (limbs + ctx.alpha - 1) / ctx.alpha;
    Cts base = alloc(B, 2, limbs);
    base.scale = items.scale;
    HX_CUDA(cudaMemsetAsync(base.d, 0, sizeof(uint64_t) * base.bstride(N) * B, s));
    DevBuf acc((size_t)B * 2 * ext * N, s);
    View accv{acc.p, (size_t)2 * ext * N, (size_t)ext * N};
    // the ModUp digits take up to twice a group's bytes (sixteen 64x64 pairs 20.8 ms, 21.1 with half of
    // that), a single digit's with its coefficients and source as much as it
    const int most = rot_chunk(B, limbs, MAX_ROT, (size_t)B * std::max(nd, 2) * ext * N / 2);
    bool any = false;
    for (int r = 0; r < R;) {
        Cts first = items;
        first.d += (size_t)r * B * items.bstride(N);
        first.B = B;
        if (galois_for_step(steps[r], ctx.log_n) == 1) {
            add_inplace(base, first);
            r++;
            continue;
        }
        KeyTab kt;
        GaloisTab gt;
        gt.per = B;
        int C = 0;
        for (; C < most && r + C < R; C++) {
            const uint64_t g = galois_for_step(steps[r + C], ctx.log_n);
            if (g == 1) break;
            kt.key[C] = rot_key(keys, g).buf->p;
            kt.g[C] = 1;  // the items are rotated before their ModUp
            gt.g[C] = (uint32_t)g;
        }
        Cts t = alloc(C * B, 1, limbs);
        launch_automorphism(lc(), t.view(N), View{first.d + first.cstride(N), first.bstride(N), first.cstride(N)}, gt, C * B,
                            1, limbs);
        BufPtr D = modup(t.view(N), C * B, limbs);
        launch_key_ip(lc(), accv, D->p, t.d, t.bstride(N), kt, C, false, true, ctx.n_all, ctx.n_q, K, ctx.alpha, limbs, nd, B,
                      any);
        launch_automorphism_sum(lc(), base.view(N), first.view(N), gt, C, B, limbs);  // base.c0 += sigma_g(c0)
        any = true;
        r += C;
        ctx.counters[C_ROT] += (uint64_t)C * B;
        ctx.counters[C_KS] += (uint64_t)C * B;
        ctx.counters[C_ADD] += (uint64_t)C * B;
    }
    if (!any) return base;
    Cts o = alloc(B, 2, limbs);
    moddown_add(batch_out(o.view(N), B), accv, B, limbs, base.view(N), 3, one_galois(1, B));
    o.scale = items.scale;
    return o;
}

Cts Eval::relinearize(const Cts &d, const SwitchKey &rk)
{
    HX_CHECK(d.comps == 3, HX_EINVAL, "relinearisation needs 3 components");
    HX_CHECK(rk.buf, HX_EKEY, "no relinearisation key");
    const size_t N = ctx.N;
    View d2{d.d + 2 * d.cstride(N), d.bstride(N), d.cstride(N)};
    BufPtr D = modup(d2, d.B, d.limbs);
    Cts o = ks_finish(D, d2, d.B, d.limbs, rk, 1, d.view(N), 3, 1);
    o.scale = d.scale;
    return o;
}

// Relinearisation and RS in one division by P q_top: the key inner product of d_2 over
// Q_l and P; y_c = acc_c + P d_c (only q_top's row is formed in memory, the lower rows in
// the epilogue); the remainder [y_c + h]_{P q_top} - h converted from q_top and the special
// primes to Q_{l-1}; out_c = (y_c - remainder) (P q_top)^-1.
Cts Eval::relin_rescale(const Cts &d, const SwitchKey &rk)
{
    HX_CHECK(d.comps == 3, HX_EINVAL, "relinearisation needs 3 components");
    HX_CHECK(rk.buf, HX_EKEY, "no relinearisation key");
    HX_CHECK(d.limbs >= 2, HX_ELEVEL, "no level left to rescale");
    const int N = ctx.N, K = ctx.K, L = d.limbs, B = d.B, ext = L + K, nd = (L + ctx.alpha - 1) / ctx.alpha;
    View d2{d.d + 2 * d.cstride(N), d.bstride(N), d.cstride(N)};
    BufPtr D = modup(d2, B, L);
    DevBuf acc((size_t)B * 2 * ext * N, s);
    View accv{acc.p, (size_t)2 * ext * N, (size_t)ext * N};
    launch_key_ip(lc(), accv, D->p, d2.p, d2.bstride, one_key(rk, 1), 1, true, false, ctx.n_all, ctx.n_q, K, ctx.alpha, L,
                  nd, B);
    ctx.counters[C_KS] += B;
    D.reset();
    const RelinRescaleTable *tab = ctx.t.relin_rs + L;
    launch_relin_rs_top(lc(), accv, d.view(N), tab, B, L);
    std::vector<int> rows = iota_vec(L - 1, K + 1), primes(K + 1);
    primes[0] = L - 1;
    for (int k = 0; k < K; k++) primes[k + 1] = ctx.n_q + k;
    ntt_inplace(acc.p, (size_t)ext * N, 2 * B, rows, primes, true);
    DevBuf conv((size_t)B * 2 * (L - 1) * N, s);
    launch_basis_convert(lc(), reinterpret_cast<const ConvTable *>(tab), K + 1, View{conv.p, (size_t)(L - 1) * N, 0},
                         View{acc.p, (size_t)ext * N, 0}, 2 * B, 1, 0, 0, 8.0 * N * 2 * B * (K + L));
    ntt_inplace(conv.p, (size_t)(L - 1) * N, 2 * B, iota_vec(0, L - 1), iota_vec(0, L - 1), false);
    Cts o = alloc(B, 2, L - 1);
    launch_relin_rs_final(lc(), o.view(N), accv, d.view(N),
                          View{conv.p, (size_t)2 * (L - 1) * N, (size_t)(L - 1) * N}, tab, B, L);
    o.scale = d.scale / (double)ctx.primes[L - 1];
    ctx.counters[C_RESCALE] += B;
    return o;
}

const SwitchKey &Eval::rot_key(const hx_keyset &ks, uint64_t g)
{
    auto it = ks.rot.find(g);
    HX_CHECK(it != ks.rot.end(), HX_EKEY, "missing Galois key for element " + std::to_string(g));
    return it->second;
}

Cts Eval::rotate(const Cts &a, int64_t k, const hx_keyset &ks)
{
    const uint64_t g = galois_for_step(k, ctx.log_n);
    if (g == 1) return copy(a);
    const SwitchKey &key = rot_key(ks, g);
    const size_t N = ctx.N;
    Cts t = alloc(a.B, 1, a.limbs);
    View c1{a.d + a.cstride(N), a.bstride(N), a.cstride(N)};
    launch_automorphism(lc(), t.view(N), c1, one_galois(g, a.B), a.B, 1, a.limbs);
    BufPtr D = modup(t.view(N), a.B, a.limbs);
    Cts o = ks_finish(D, t.view(N), a.B, a.limbs, key, 1, a.view(N), 1, g);
    o.scale = a.scale;
    ctx.counters[C_ROT] += a.B;
    return o;
}

Cts Eval::rotate_each(const Cts &a, const std::vector<int64_t> &steps, const hx_keyset &keys)
{
    const int R = (int)steps.size(), B = a.B / R, N = ctx.N, K = ctx.K, limbs = a.limbs, ext = limbs + K,
              nd = (limbs + ctx.alpha - 1) / ctx.alpha;
    HX_CHECK(R >= 1 && R <= MAX_ROT && a.B % R == 0 && a.comps == 2, HX_EINVAL, "bad batch of rotations");
    KeyTab kt;
    GaloisTab gt;
    gt.per = B;
    for (int r = 0; r < R; r++) {
        const uint64_t g = galois_for_step(steps[r], ctx.log_n);
        HX_CHECK(g != 1, HX_EINVAL, "a batch of rotations takes proper ones");
        kt.key[r] = rot_key(keys, g).buf->p;
        kt.g[r] = 1;
        gt.g[r] = (uint32_t)g;
    }
    Cts t = alloc(a.B, 1, limbs);
    launch_automorphism(lc(), t.view(N), View{a.d + a.cstride(N), a.bstride(N), a.cstride(N)}, gt, a.B, 1, limbs);
    BufPtr D = modup(t.view(N), a.B, limbs);
    DevBuf acc((size_t)a.B * 2 * ext * N, s);
    View accv{acc.p, (size_t)2 * ext * N, (size_t)ext * N};
    launch_key_ip(lc(), accv, D->p, t.d, t.bstride(N), kt, R, false, false, ctx.n_all, ctx.n_q, K, ctx.alpha, limbs, nd, B);
    Cts o = alloc(a.B, 2, limbs);
    moddown_add(batch_out(o.view(N), B, R), accv, a.B, limbs, a.view(N), 1, gt);
    o.scale = a.scale;
    ctx.counters[C_ROT] += a.B;
    ctx.counters[C_KS] += a.B;
    return o;
}

BufPtr Eval::hoist(const Cts &a)
{
    const size_t N = ctx.N;
    View c1{a.d + a.cstride(N), a.bstride(N), a.cstride(N)};
    return modup(c1, a.B, a.limbs);
}

BufPtr Eval::hoist_for(const Cts &a, const std::vector<int64_t> &steps)
{
    for (int64_t k : steps)
        if (galois_for_step(k, ctx.log_n) != 1) return hoist(a);
    return BufPtr();
}

std::vector<uint64_t *> Eval::groups_of(const Cts &c, int R) const
{
    std::vector<uint64_t *> p(R);
    for (int r = 0; r < R; r++) p[r] = c.d + (size_t)r * (c.B / R) * c.bstride(ctx.N);
    return p;
}

void Eval::rotate_hoisted_into(const std::vector<uint64_t *> &out, const Cts &a, const BufPtr &D,
                               const std::vector<int64_t> &steps, const hx_keyset &keys)
{
    const int R = (int)steps.size();
    const int N = ctx.N, K = ctx.K, B = a.B, limbs = a.limbs, ext = limbs + K, nd = (limbs + ctx.alpha - 1) / ctx.alpha;
    OutTab ot;
    ot.cstride = (size_t)limbs * N;
    ot.bstride = 2 * ot.cstride;
    const View c1{a.d + a.cstride(N), a.bstride(N), a.cstride(N)};
    const int most = rot_chunk(B, limbs, MAX_ROT);
    for (int r = 0; r < R;) {
        if (galois_for_step(steps[r], ctx.log_n) == 1) {
            launch_copy(lc(), View{out[r], ot.bstride, ot.cstride}, a.view(N), B, 2, limbs);
            r++;
            continue;
        }
        KeyTab kt;
        GaloisTab gt;
        gt.per = B;
        int C = 0;
        for (; C < most && r + C < R; C++) {
            const uint64_t g = galois_for_step(steps[r + C], ctx.log_n);
            if (g == 1) break;
            kt.key[C] = rot_key(keys, g).buf->p;
            kt.g[C] = gt.g[C] = (uint32_t)g;
            ot.p[C] = out[r + C];
        }
        DevBuf acc((size_t)C * B * 2 * ext * N, s);
        View accv{acc.p, (size_t)2 * ext * N, (size_t)ext * N};
        launch_key_ip(lc(), accv, D->p, c1.p, c1.bstride, kt, C, true, false, ctx.n_all, ctx.n_q, K, ctx.alpha, limbs, nd, B);
        moddown_add(ot, accv, C * B, limbs, a.view(N), 1, gt, true);
        r += C;
        ctx.counters[C_ROT] += (uint64_t)C * B;
        ctx.counters[C_ROT_HOIST] += (uint64_t)C * B;
        ctx.counters[C_KS] += (uint64_t)C * B;
    }
}

Cts Eval::hoisted_mux(const Cts &a, const BufPtr &D, const std::vector<MuxItem> &items, double v_scale, uint64_t c,
                      const hx_keyset &keys)
{
    const int N = ctx.N, K = ctx.K, limbs = a.limbs, ext = limbs + K, nd = (limbs + ctx.alpha - 1) / ctx.alpha, B = a.B;
    const int C = (int)items.size();
    HX_CHECK(C >= 1 && C <= MAX_MUX, HX_EINVAL, "too many selections in one batch");
    MuxTab tab;
    const bool premasked = items[0].premasked != nullptr;
    for (int i = 0; i < C; i++) {
        const uint64_t g1 = galois_for_step(items[i].k1, ctx.log_n), g2 = galois_for_step(items[i].k2, ctx.log_n);
        HX_CHECK(g1 != 1 && g2 != 1, HX_EINVAL, "selection needs two proper rotations");
        tab.k1[i] = rot_key(keys, g1).buf->p;
        tab.k2[i] = rot_key(keys, g2).buf->p;
        if (premasked) tab.k1[i] = items[i].premasked;
        tab.v[i] = items[i].v_ext;
        tab.g1[i] = (uint32_t)g1;
        tab.g2[i] = (uint32_t)g2;
    }
    Scalars cs;
    for (int t = 0; t < ext; t++) {
        const uint64_t q = ctx.primes[t < limbs ? t : ctx.n_q + (t - limbs)];
        cs.v[t] = c % q;
        cs.sh[t] = shoup_companion(cs.v[t], q);
    }
    const View c1{a.d + a.cstride(N), a.bstride(N), a.cstride(N)};
    DevBuf z((size_t)C * B * 2 * ext * N, s);
    View zv{z.p, (size_t)2 * ext * N, (size_t)ext * N};
    if (premasked)
        launch_key_ip_mux_pm(lc(), zv, D->p, c1.p, c1.bstride, tab, C, ctx.n_q, K, ctx.alpha, limbs, nd, B);
    else
        launch_key_ip_mux(lc(), zv, D->p, c1.p, c1.bstride, tab, C, cs, ctx.n_all, ctx.n_q, K, ctx.alpha, limbs, nd, B);
    DevBuf conv((size_t)C * B * 2 * limbs * N, s);
    moddown_ntt(zv, conv.p, C * B, limbs);
    Cts o = alloc(C * B, 2, limbs);
    launch_moddown_final_mux(lc(), o.view(N), zv, View{conv.p, (size_t)2 * limbs * N, (size_t)limbs * N},
                             ctx.t.moddown + limbs, C, B, K, limbs, a.view(N), tab, cs);
    o.scale = a.scale * v_scale;
    ctx.counters[C_ROT] += 2ull * C * B;
    ctx.counters[C_ROT_HOIST] += 2ull * C * B;
    ctx.counters[C_MULPT] += (uint64_t)C * B;
    ctx.counters[C_ADD] += (uint64_t)C * B;
    ctx.counters[C_KS] += (uint64_t)C * B;
    return o;
}

Cts Eval::rotate_hoisted(const Cts &a, const std::vector<int64_t> &steps, const hx_keyset &keys)
{
    const BufPtr D = hoist_for(a, steps);
    Cts out = alloc(a.B * (int)steps.size(), 2, a.limbs);
    out.scale = a.scale;
    rotate_hoisted_into(groups_of(out, (int)steps.size()), a, D, steps, keys);
    return out;
}

void Eval::tensor_sum(Cts &acc, const Cts &a, const Cts &b)
{
    HX_CHECK(a.B == b.B && a.B % acc.B == 0 && a.limbs == b.limbs && acc.limbs == a.limbs && acc.comps == 3, HX_ESCALE,
             "tensor operands differ");
    HX_CHECK(std::fabs(acc.scale / (a.scale * b.scale) - 1.0) <= std::ldexp(1.0, -20), HX_ESCALE, "scale mismatch");
    launch_tensor_sum(lc(), acc.view(ctx.N), a.view(ctx.N), b.view(ctx.N), a.B / acc.B, acc.B, a.limbs);
    ctx.counters[C_MULCT] += a.B;
    ctx.counters[C_ADD] += a.B;
}

Cts Eval::rescale(const Cts &a, int64_t c, const Tail *tail)
{
    HX_CHECK(a.limbs >= 2, HX_ELEVEL, "no level left to rescale");
    const int N = ctx.N, top = a.limbs - 1, comps = a.comps, B = a.B;
    DevBuf xtop((size_t)B * comps * N, s);
    ntt_oop(a.d, a.cstride(N), xtop.p, (size_t)N, B * comps, {top}, {0}, {top}, true);
    DevBuf r((size_t)B * comps * top * N, s);
    View rv{r.p, (size_t)comps * top * N, (size_t)top * N};
    const RescaleTable *tab = ctx.t.rescale + a.limbs;
    // rescale(c * a) for an integer c: a's residues times c in the two elementwise passes
    // (the top limb after its inverse NTT), the same values as multiplying first
    const Scalars sc = c != 1 || tail ? scalars_for(ctx, a.limbs, c) : Scalars{};
    const Scalars *scp = c != 1 || tail ? &sc : nullptr;
    // The remainder modulo every lower prime, transformed.  Centred it is at most q_top / 2 in size, and
    // the fold transform takes signed inputs below 4q: where no lower prime is less than that, one
    // centred row feeds the transform of every limb and no reduced rows are written and read.
    // Sixty-four signs at N = 2^15 126.3 -> 122.2 ms, an aggregation's export and all 860 -> 829 us.
    const uint64_t qt = ctx.primes[top];
    bool centred = ctx.t.fold != nullptr;
    for (int i = 0; i < top; i++) centred = centred && ctx.primes[i] > qt / 2;
    if (centred) {
        launch_rescale_centre(lc(), xtop.p, tab, qt, B * comps, sc.v[top], sc.sh[top], scp != nullptr);
        ntt_oop(xtop.p, (size_t)N, r.p, (size_t)top * N, B * comps, std::vector<int>(top, 0), iota_vec(0, top),
                iota_vec(0, top), false);
    } else {
        launch_rescale_prep(lc(), rv, View{xtop.p, (size_t)comps * N, (size_t)N}, tab, B, comps, top, scp);
        ntt_inplace(r.p, (size_t)top * N, B * comps, iota_vec(0, top), iota_vec(0, top), false);
    }
    Cts o = alloc(B, comps, top);
    if (tail) {
        RescaleTail t{scalars_for(ctx, top, tail->times), scalars_for(ctx, top, tail->add_times),
                      scalars_for(ctx, top, tail->c0), View{nullptr, 0, 0}, tail->times != 1, 0};
        if (tail->add) {
            HX_CHECK(tail->add->B == B && tail->add->limbs == top && tail->add->comps == comps, HX_ESCALE, "addend's shape differs");
            t.add = tail->add->view(N);
            t.has_add = tail->add_times != 1 ? 2 : 1;
            ctx.counters[C_ADD] += B;
        }
        launch_rescale_tail(lc(), o.view(N), a.view(N), rv, tab, sc, t, B, comps, top);
    } else {
        launch_rescale_final(lc(), o.view(N), a.view(N), rv, tab, B, comps, top, scp);
    }
    o.scale = a.scale / (double)ctx.primes[top];
    ctx.counters[C_RESCALE] += B;
    return o;
}

void plaintext_from_device(hx_context &ctx, cudaStream_t s, const int64_t *dcoeffs, int limbs, bool extended,
                           uint64_t *dst)
{
    Eval ev(ctx, s);
    if (!extended) {
        launch_signed_to_rows(ev.lc(), dst, dcoeffs, limbs, 1, ctx.N, ctx.d_prime_ids);
        ev.ntt_inplace(dst, 0, 1, iota_vec(0, limbs), iota_vec(0, limbs), false);
        launch_to_mont(ev.lc(), dst, limbs, ctx.d_prime_ids);
        return;
    }
    const int ext = limbs + ctx.K;
    std::vector<int> pr(ext);
    for (int t = 0; t < ext; t++) pr[t] = t < limbs ? t : ctx.n_q + (t - limbs);
    DevBuf ids((ext + 1) / 2, s);
    HX_CUDA(cudaMemcpyAsync(ids.p, pr.data(), sizeof(int) * ext, cudaMemcpyHostToDevice, s));
    const int *idp = reinterpret_cast<const int *>(ids.p);
    launch_signed_to_rows(ev.lc(), dst, dcoeffs, ext, 1, ctx.N, idp);
    ev.ntt_inplace(dst, 0, 1, iota_vec(0, ext), pr, false);
    launch_to_mont(ev.lc(), dst, ext, idp);
    HX_CUDA(cudaStreamSynchronize(s));  // the prime-index staging buffer is released at return
}

void upload_plaintext(hx_context &ctx, cudaStream_t s, const int64_t *coeffs, int limbs, uint64_t *dst)
{
    Eval ev(ctx, s);
    DevBuf tmp((size_t)ctx.N, s);
    HX_CUDA(cudaMemcpyAsync(tmp.p, coeffs, sizeof(int64_t) * ctx.N, cudaMemcpyHostToDevice, s));
    launch_signed_to_rows(ev.lc(), dst, reinterpret_cast<const int64_t *>(tmp.p), limbs, 1, ctx.N, ctx.d_prime_ids);
    ev.ntt_inplace(dst, 0, 1, iota_vec(0, limbs), iota_vec(0, limbs), false);
    launch_to_mont(ev.lc(), dst, limbs, ctx.d_prime_ids);
    HX_CUDA(cudaStreamSynchronize(s));  // the pageable source must outlive the copy
}

void upload_plaintext_ext(hx_context &ctx, cudaStream_t s, const int64_t *coeffs, int limbs, uint64_t *dst)
{
    Eval ev(ctx, s);
    const int ext = limbs + ctx.K;
    std::vector<int> pr(ext);  // the special primes' rows first, then q_0 .. q_{limbs-1}
    for (int t = 0; t < ext; t++) pr[t] = t < ctx.K ? ctx.n_q + t : t - ctx.K;
    DevBuf tmp((size_t)ctx.N, s);
    DevBuf ids((ext + 1) / 2, s);
    HX_CUDA(cudaMemcpyAsync(tmp.p, coeffs, sizeof(int64_t) * ctx.N, cudaMemcpyHostToDevice, s));
    HX_CUDA(cudaMemcpyAsync(ids.p, pr.data(), sizeof(int) * ext, cudaMemcpyHostToDevice, s));
    const int *idp = reinterpret_cast<const int *>(ids.p);
    launch_signed_to_rows(ev.lc(), dst, reinterpret_cast<const int64_t *>(tmp.p), ext, 1, ctx.N, idp);
    ev.ntt_inplace(dst, 0, 1, iota_vec(0, ext), pr, false);
    launch_to_mont(ev.lc(), dst, ext, idp);
    HX_CUDA(cudaStreamSynchronize(s));
}

} // namespace hx
