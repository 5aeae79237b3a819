// The NTT's launchers and autotuner (per-ring and several-ring), and its kernels with Shoup
// products, for chains that ArithFold does not cover.
#include "ntt_impl.cuh"

namespace hx {

template void ntt_phase<ArithShoup>(const LaunchCtx &, const NttRows &, bool, bool, int, int);
template void ntt_multi_phases<ArithShoup>(cudaStream_t, const NttJob *, int, int, int, bool);
extern template void ntt_phase<ArithFold>(const LaunchCtx &, const NttRows &, bool, bool, int, int);
extern template void ntt_multi_phases<ArithFold>(cudaStream_t, const NttJob *, int, int, int, bool);

// ---- launcher (host code: it picks the tuned variants and the phase split of the kernels above)
static void run_phase(const LaunchCtx &c, const NttRows &rows, bool inverse, bool cols, int logm, int var)
{
    // fold arithmetic wherever every prime of the chain allows it
    if (c.t->fold) ntt_phase<ArithFold>(c, rows, inverse, cols, logm, var);
    else ntt_phase<ArithShoup>(c, rows, inverse, cols, logm, var);
}

void launch_ntt(const LaunchCtx &c, const NttRows &rows, bool inverse)
{
    Timed tm_(c, K_NTT, 16.0 * rows.n_rows * rows.n_groups * c.N);
    if (rows.n_rows <= 0 || rows.n_groups <= 0) return;
    HX_CHECK(rows.n_rows <= MAX_NTT_ROWS && rows.n_groups < 65536, HX_EINVAL, "NTT batch too large");
    const int *v = c.t->ntt_var[ntt_bucket((long long)rows.n_rows * rows.n_groups)];
    const int logm1 = c.log_n / 2 + ((c.log_n & 1) && v[4] ? 1 : 0), logm2 = c.log_n - logm1;
    if (!inverse) {
        run_phase(c, rows, false, true, logm1, v[0]);
        run_phase(c, rows, false, false, logm2, v[1]);
    } else {
        run_phase(c, rows, true, false, logm2, v[3]);
        run_phase(c, rows, true, true, logm1, v[2]);
    }
    post(c, 2);
}
// ---- end of the launcher

// ---- autotuner (host code: it times the phase kernels and changes none of them)
void autotune_ntt(const LaunchCtx &c, uint64_t *buf, int rows, int *best, float *ms_out)
{
    // times every tile width of each phase on `rows` limbs (one prime each) in place, for each
    // split of an odd log N between the phases
    NttRows *r = new NttRows();
    std::unique_ptr<NttRows> guard(r);
    r->src = r->dst = buf;
    r->src_gs = r->dst_gs = 0;
    r->n_groups = 1;
    r->n_rows = rows;
    for (int i = 0; i < rows; i++) {
        r->src_off[i] = r->dst_off[i] = (int16_t)i;
        r->prime[i] = 0;
    }
    cudaEvent_t e0, e1;
    HX_CUDA(cudaEventCreate(&e0));
    HX_CUDA(cudaEventCreate(&e1));
    // Each variant's time is the best of three rounds of five transforms, the rounds interleaved
    // over the variants so drift hits them alike.  A variant replaces the default (four warps per
    // block) only when it is clearly faster: the widths' isolated
    // times differ by about their noise (1-2 % at the batch sizes of a product's launches), and
    // blocks of the default size share the SMs best with the kernels of concurrent chains.  The
    // other split of an odd log N replaces the default one on the same rule, by the sum of its
    // four phases' times.
    constexpr int kRounds = 3, kRuns = 5;
    constexpr float kClearWin = 0.98f;
    float split_ms[2] = {0.f, 0.f};
    int split_best[2][4];
    float split_phase_ms[2][4];
    const int n_splits = (c.log_n & 1) ? 2 : 1;
    for (int sp = 0; sp < n_splits; sp++) {
        const int logm1 = c.log_n / 2 + sp, logm2 = c.log_n - logm1;
        for (int ph = 0; ph < 4; ph++) {
            const bool cols = ph == 0 || ph == 2, inv = ph >= 2;
            const int logm = cols ? logm1 : logm2, kDefault = ntt_default_var(logm);
            float t[NTT_VARIANTS];
            bool ok[NTT_VARIANTS];
            for (int v = 0; v < NTT_VARIANTS; v++) {
                t[v] = 1e30f;
                ok[v] = kNttTiles[v % NTT_WIDTHS] <= (c.N >> logm) && (v < NTT_WIDTHS || (logm & 1));
            }
            for (int round = 0; round < kRounds; round++)
                for (int v = 0; v < NTT_VARIANTS; v++) {
                    if (!ok[v]) continue;
                    auto run = [&]() { run_phase(c, *r, inv, cols, logm, v); };
                    run();  // warm-up
                    HX_CUDA(cudaEventRecord(e0, c.stream));
                    for (int it = 0; it < kRuns; it++) run();
                    HX_CUDA(cudaEventRecord(e1, c.stream));
                    HX_CUDA(cudaEventSynchronize(e1));
                    float ms = 0;
                    HX_CUDA(cudaEventElapsedTime(&ms, e0, e1));
                    t[v] = std::min(t[v], ms / kRuns);
                }
            int pick = ok[kDefault] ? kDefault : -1;
            for (int v = 0; v < NTT_VARIANTS; v++) {
                if (!ok[v] || v == pick) continue;
                if (pick < 0 || t[v] < (pick == kDefault ? kClearWin : 1.0f) * t[pick]) pick = v;
            }
            split_best[sp][ph] = pick < 0 ? kDefault : pick;
            split_phase_ms[sp][ph] = pick < 0 ? 0.f : t[pick];
            split_ms[sp] += split_phase_ms[sp][ph];
        }
    }
    const int def = ntt_default_split(c.log_n);
    const int sp = (n_splits == 2 && split_ms[1 - def] < kClearWin * split_ms[def]) ? 1 - def : def;
    for (int ph = 0; ph < 4; ph++) {
        best[ph] = split_best[sp][ph];
        if (ms_out) ms_out[ph] = split_phase_ms[sp][ph];
    }
    best[4] = sp;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    HX_CUDA(cudaGetLastError());
}
// ---- end of the autotuner

// ---- several rings: launcher
void plan_ntt_jobs(std::vector<NttJob> &jobs, int *tiles_cols, int *tiles_rows)
{
    int tc = 0, tr = 0;
    for (auto &J : jobs) {
        HX_CHECK(J.log_n >= 11 && J.log_n <= 16, HX_EINVAL, "ring degree outside 2^11..2^16");
        HX_CHECK(J.n_limbs >= 1 && J.n_limbs <= 64 && J.n_rows >= 0, HX_EINVAL, "bad job rows");
        const int n = 1 << J.log_n, l1 = J.log_n / 2 + ntt_default_split(J.log_n), l2 = J.log_n - l1;
        const int w1 = 128 / ((1 << l1) >> ((l1 + 1) / 2)), w2 = 128 / ((1 << l2) >> ((l2 + 1) / 2));
        J.tile0_cols = tc;
        J.tile0_rows = tr;
        const long long c = (long long)J.n_rows * ((n >> l1) / w1), r = (long long)J.n_rows * ((n >> l2) / w2);
        HX_CHECK(tc + c < (1ll << 31) && tr + r < (1ll << 31), HX_EINVAL, "NTT batch too large");
        tc += (int)c;
        tr += (int)r;
    }
    *tiles_cols = tc;
    *tiles_rows = tr;
}

void launch_ntt_jobs(cudaStream_t s, const NttJob *jp, int n_jobs, int tc, int tr, bool fold, bool inverse,
                     std::atomic<uint64_t> *launches)
{
    if (tc == 0) return;
    if (fold) ntt_multi_phases<ArithFold>(s, jp, n_jobs, tc, tr, inverse);
    else ntt_multi_phases<ArithShoup>(s, jp, n_jobs, tc, tr, inverse);
    HX_CUDA(cudaGetLastError());
    if (launches) *launches += 2;
}

void launch_ntt_multi(cudaStream_t s, const std::vector<NttJob> &jobs_in, bool inverse,
                      std::atomic<uint64_t> *launches)
{
    std::vector<NttJob> jobs = jobs_in;
    int tc = 0, tr = 0;
    plan_ntt_jobs(jobs, &tc, &tr);
    if (tc == 0) return;
    bool fold = true;
    for (const NttJob &J : jobs) fold = fold && J.fold;
    void *jd = nullptr;
    HX_CUDA(cudaMallocAsync(&jd, jobs.size() * sizeof(NttJob), s));
    HX_CUDA(cudaMemcpyAsync(jd, jobs.data(), jobs.size() * sizeof(NttJob), cudaMemcpyHostToDevice, s));
    try {
        launch_ntt_jobs(s, reinterpret_cast<const NttJob *>(jd), (int)jobs.size(), tc, tr, fold, inverse, launches);
    } catch (...) {
        cudaFreeAsync(jd, s);
        throw;
    }
    HX_CUDA(cudaFreeAsync(jd, s));
    HX_CUDA(cudaStreamSynchronize(s));  // the host job vector is released at return
}

// ---- end of the several-ring launcher

} // namespace hx
