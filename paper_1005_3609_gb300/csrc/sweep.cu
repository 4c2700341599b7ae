// cp_sweep: the batched finite-lattice sweep (Sec. 4.1-4.3).
//
// For every width r = 1..floor(k/2) one strip is advanced to the largest
// height of the band k-3 <= r+s <= k (s >= r) and read out at every band
// height on the way, so a rectangle shares its strip prefix with the shorter
// ones.  All strips advance in lock-step: global step t applies the t-th
// per-site factor of every strip that still has one, plus the t-th factor of
// any read-out chain in flight, in ONE batched gather launch.  A read-out
// chain T_1^last .. T_{r-1}^last starts at the step where the strip's next
// row begins (both only read the current vector) and runs on two scratch
// buffers while the strip moves on; its last factor writes the e_0 row
// straight into the P~ array.  The primes are split into groups of Pg primes
// (one strip per width and group).  The whole program -- every
// batched launch and the series kernel -- is captured once into a CUDA graph,
// so a sweep is a single graph launch.  The prime grouping is picked by timing the
// candidates (autotune) unless given.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include "cp_internal.h"
#include "series.h"

using namespace cp;

namespace {

struct SweepStrip {
    int r = 0, group = 0, Pg = 0;
    std::shared_ptr<TableSet> tabs;
    uint32_t *vec[2] = {nullptr, nullptr};
    uint32_t *scratch[2] = {nullptr, nullptr};
    std::vector<int> heights;
};

int n_terms_for(int lattice, int k) {
    if (lattice == CP_SQUARE) return (k % 2 == 1) ? 2 * k - 2 : 2 * k - 3;
    return k;
}

}  // namespace

struct cp_sweep {
    int lattice = 0, k = 0, P = 0, D1 = 0, n = 0, tile = 0, groups = 0, Pg = 0, Pp = 0;  // Pp: prime lanes of a group's rows
    cudaStream_t stream = nullptr;
    uint32_t *primes_dev = nullptr, *ones_dev = nullptr;  // primes: a prime block per group
    std::vector<SweepStrip> strips;
    std::vector<int2> rects;
    int2 *rects_dev = nullptr;
    uint32_t *ptilde_dev = nullptr;  // [groups][n_rects][D1][Pp]
    uint32_t *series_dev = nullptr;  // [3][P][n]
    uint32_t *logs_dev = nullptr;    // series kernel's scratch
    uint32_t *crt_dev = nullptr;     // cp_sweep_series_integers: limbs [3][n][limbs], then flags [3][n]
    size_t crt_words = 0;
    std::vector<uint32_t> primes_host;
    ErrorWord err;
    std::vector<std::vector<GatherTask>> steps;  // tasks of each batched launch
    std::vector<uint32_t> step_blocks;
    struct Applied {
        const SiteTable *tab;
        int v_in;
        bool first, final;
    };
    std::vector<Applied> applied;  // every table application of a run
    std::vector<int> step_tile;
    uint64_t updates = 0, bytes = 0, site_bytes = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    PadShare pad;

    ~cp_sweep() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        for (auto &s : strips) {
            dev_free(s.vec[0]);
            dev_free(s.vec[1]);
            dev_free(s.scratch[0]);
            dev_free(s.scratch[1]);
        }
        dev_free(primes_dev);
        dev_free(ones_dev);
        dev_free(rects_dev);
        dev_free(ptilde_dev);
        dev_free(series_dev);
        dev_free(logs_dev);
        dev_free(crt_dev);
        error_word_free(&err);
    }
};

static int rect_index(const cp_sweep *sw, int r, int s) {
    for (size_t j = 0; j < sw->rects.size(); ++j)
        if (sw->rects[j].x == r && sw->rects[j].y == s) return (int)j;
    return -1;
}

// Accumulate the algorithmic work of one factor: output words, and bytes =
// 4 (S_in + S_out) (D+1) Pg + CSR index bytes.
static void count_work(cp_sweep *sw, const SiteTable &t, int Pg) {
    const uint64_t mid = t.n_site_out - t.n_dst;  // intermediate states of a two-site table (else 0)
    sw->updates += t.n_site_out * (uint64_t)sw->D1 * Pg;
    sw->bytes += 4ull * (t.n_src + t.n_dst) * sw->D1 * Pg + 4ull * (t.n_dst + 1 + t.nnz);
    sw->site_bytes += 4ull * (t.n_src + 2 * mid + t.n_dst) * sw->D1 * Pg + 4ull * (t.n_dst + 1 + t.nnz);
}

// Strips and buffers: one strip per width (and prime group), band rectangles.
static int build_strips(cp_sweep *sw) {
    const int ngroups = sw->groups, Pg = sw->Pg;
    const size_t row_words = (size_t)sw->D1 * sw->Pp;
    int rc;
    // band rectangles (r <= s, k-3 <= r+s <= k), ordered by r then s
    for (int r = 1; 2 * r <= sw->k; ++r)
        for (int s = r; r + s <= sw->k; ++s)
            if (r + s >= sw->k - 3) sw->rects.push_back(make_int2(r, s));
    for (int g = 0; g < ngroups; ++g) {
        for (int r = 1; 2 * r <= sw->k; ++r) {
            SweepStrip st;
            st.r = r;
            st.group = g;
            st.Pg = Pg;
            for (auto &rs : sw->rects)
                if (rs.x == r) st.heights.push_back(rs.y);
            if (st.heights.empty()) continue;
            if ((rc = get_tables(sw->lattice, r, (size_t)sw->D1 * padded_primes(Pg) * 4, sw->stream, &st.tabs))) return rc;
            const TableSet &ts = *st.tabs;
            sw->strips.push_back(st);
            SweepStrip &sp = sw->strips.back();
            uint64_t sA = ts.last[0].n_dst, sB = ts.last.size() >= 2 ? ts.last[1].n_dst : 1;
            if (sw->Pp != Pg && !sw->pad.take((2 * ts.S_max + sA + sB) * sw->D1 * (sw->Pp - Pg) * 4))
                return fail(CP_ENOMEM, "the padding lanes' share of the device memory is taken");
            for (int b = 0; b < 2; ++b)
                if ((rc = dev_alloc((void **)&sp.vec[b], ts.S_max * row_words * 4))) return rc;
            if ((rc = dev_alloc((void **)&sp.scratch[0], sA * row_words * 4))) return rc;
            if ((rc = dev_alloc((void **)&sp.scratch[1], sB * row_words * 4))) return rc;
        }
    }
    return CP_OK;
}

static int enqueue_program(cp_sweep *sw);

// Launch program for gather tile `tile`: per-step task lists, block assignment,
// device task array, and the CUDA graph of the whole sweep.
static int build_program(cp_sweep *sw, int tile) {
    const int Pg = sw->Pg;
    const int n_rects = (int)sw->rects.size();
    const size_t row_words = (size_t)sw->D1 * sw->Pp;
    int rc;
    sw->tile = tile;
    sw->updates = sw->bytes = sw->site_bytes = 0;
    sw->step_blocks.clear();
    sw->step_tile.clear();
    if (sw->exec) cudaGraphExecDestroy(sw->exec);
    if (sw->graph) cudaGraphDestroy(sw->graph);
    sw->exec = nullptr;
    sw->graph = nullptr;
    const uint32_t pmin = *std::min_element(sw->primes_host.begin(), sw->primes_host.end());
    auto &steps = sw->steps;
    steps.clear();
    sw->applied.clear();
    auto at = [&](size_t t) -> std::vector<GatherTask> & {
        if (steps.size() <= t) steps.resize(t + 1);
        return steps[t];
    };
    for (auto &st : sw->strips) {
        const TableSet &ts = *st.tabs;
        const int r = st.r;
        const uint32_t *pr = sw->primes_dev + st.group * kPrimeWords;
        const int smax = st.heights.back();
        const int nf = (int)ts.row.size();  // launches per row (factors, or pairs of factors)
        // main lane: rows 1..smax-1, launch i of row h is step (h-1)*nf + i
        int v = r;
        for (int row = 0; row < smax - 1; ++row)
            for (int i = 0; i < nf; ++i) {
                const size_t t = (size_t)row * nf + i;
                append_gather_task(&at(t), ts.row[i], st.vec[t & 1], st.vec[(t & 1) ^ 1], pr, sw->D1, sw->Pp, v, pmin);
                if (t == 0) at(t).back().first = 1;
                sw->applied.push_back({&ts.row[i], v, t == 0, false});
                v += ts.row[i].sites;
                count_work(sw, ts.row[i], Pg);
            }
        // read-out lanes
        for (int h : st.heights) {
            const size_t t0 = (size_t)(h - 1) * nf;
            const uint32_t *src = st.vec[t0 & 1];
            uint32_t *slot = sw->ptilde_dev + ((size_t)st.group * n_rects + rect_index(sw, r, h)) * row_words;
            int sc = 0;
            v = r * h;
            for (size_t i = 0; i < ts.last.size(); ++i) {
                const bool final = i + 1 == ts.last.size();
                uint32_t *dst = final ? slot : st.scratch[sc];
                append_gather_task(&at(t0 + i), ts.last[i], src, dst, pr, sw->D1, sw->Pp, v, pmin, final);
                if (t0 + i == 0) at(0).back().first = 1;  // read out at height 1
                sw->applied.push_back({&ts.last[i], v, t0 + i == 0, final});
                v += ts.last[i].sites;
                count_work(sw, ts.last[i], Pg);
                src = dst;
                sc ^= 1;
            }
        }
    }
    for (auto &l : steps) {
        const int et = effective_tile(l, tile);
        sw->step_tile.push_back(et);
        sw->step_blocks.push_back(assign_blocks(l, et));
    }
    // capture the program into one graph
    CP_CUDA_TRY(cudaStreamBeginCapture(sw->stream, cudaStreamCaptureModeThreadLocal));
    rc = enqueue_program(sw);
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(sw->stream, &g);
    if (rc) {
        if (g) cudaGraphDestroy(g);
        return rc;
    }
    if (e != cudaSuccess) return fail(CP_ECUDA, std::string("graph capture: ") + cudaGetErrorString(e));
    sw->graph = g;
    CP_CUDA_TRY(cudaGraphInstantiate(&sw->exec, g, 0));
    return CP_OK;
}

static SeriesParams series_params(const cp_sweep *sw) {
    SeriesParams sp{};
    sp.lattice = sw->lattice;
    sp.k = sw->k;
    sp.n = sw->n;
    sp.D1 = sw->D1;
    sp.P = sw->P;
    sp.Pg = sw->Pg;
    sp.Pp = sw->Pp;
    sp.n_rects = (int)sw->rects.size();
    sp.mmax = sw->k / 2;
    sp.add_mu = (sw->lattice == CP_SQUARE && sw->k % 2 == 1) ? 1 : 0;
    return sp;
}

// Every vector := e_0; at height 1 no other word is read (degree windows).
static int enqueue_reset(cp_sweep *sw) {
    for (auto &st : sw->strips)
        CP_CUDA_TRY(cudaMemcpyAsync(st.vec[0], sw->ones_dev, 4 * sw->Pp, cudaMemcpyDeviceToDevice, sw->stream));
    return CP_OK;
}

// Enqueue the whole sweep on sw->stream (used once, under graph capture).
static int enqueue_program(cp_sweep *sw) {
    int rc = enqueue_reset(sw);
    if (rc) return rc;
    for (size_t t = 0; t < sw->steps.size(); ++t) {
        rc = launch_gather(sw->steps[t].data(), (int)sw->steps[t].size(), sw->step_blocks[t], sw->step_tile[t], sw->stream);
        if (rc) return rc;
    }
    return launch_flm_series(sw->ptilde_dev, sw->rects_dev, sw->primes_dev, series_params(sw), sw->logs_dev,
                             sw->series_dev, sw->err.dev, sw->stream);
}

// The primes as the strips hold them: a prime block per group.
static std::vector<uint32_t> prime_blocks(const cp_sweep *sw) {
    std::vector<uint32_t> l((size_t)sw->groups * kPrimeWords, 0u);
    for (int g = 0; g < sw->groups; ++g)
        fill_prime_block(sw->primes_host.data() + g * sw->Pg, sw->Pg, sw->Pp, l.data() + (size_t)g * kPrimeWords);
    return l;
}

// Pp: prime lanes per group, P / groups or that padded to 16-byte chunks.
static int sweep_build_lanes(int lattice, int k, const uint32_t *primes, int P, int tile, int groups, int Pp,
                             cudaStream_t stream, cp_sweep **out);

// Rows padded to 16-byte chunks (the chunk kernel); where the vectors or the padding's share
// (PadShare) do not fit that way, rows of the given primes alone (the register kernel).
static int sweep_build(int lattice, int k, const uint32_t *primes, int P, int tile, int groups, cudaStream_t stream,
                       cp_sweep **out) {
    const int Pg = P / groups, Pp = padded_primes(Pg);
    int rc = sweep_build_lanes(lattice, k, primes, P, tile, groups, Pp, stream, out);
    if (rc == CP_ENOMEM && Pp != Pg) rc = sweep_build_lanes(lattice, k, primes, P, tile, groups, Pg, stream, out);
    return rc;
}

static int sweep_build_lanes(int lattice, int k, const uint32_t *primes, int P, int tile, int groups, int Pp,
                             cudaStream_t stream, cp_sweep **out) {
    auto sw = std::make_unique<cp_sweep>();
    sw->lattice = lattice;
    sw->k = k;
    sw->P = P;
    sw->n = n_terms_for(lattice, k);
    sw->D1 = sw->n;
    sw->groups = groups;
    sw->Pg = P / groups;
    sw->Pp = Pp;
    sw->stream = stream;
    int rc;
    if ((rc = prepare_gather_kernels()) || (rc = crt_static_touch())) return rc;
    sw->primes_host.assign(primes, primes + P);
    const std::vector<uint32_t> lanes = prime_blocks(sw.get());
    if ((rc = dev_alloc((void **)&sw->primes_dev, 4 * lanes.size()))) return rc;
    CP_CUDA_TRY(cudaMemcpy(sw->primes_dev, lanes.data(), 4 * lanes.size(), cudaMemcpyHostToDevice));
    std::vector<uint32_t> ones(CP_MAX_PRIMES, 1u);
    if ((rc = dev_alloc((void **)&sw->ones_dev, 4 * CP_MAX_PRIMES))) return rc;
    CP_CUDA_TRY(cudaMemcpy(sw->ones_dev, ones.data(), 4 * CP_MAX_PRIMES, cudaMemcpyHostToDevice));
    int n_rects = 0;
    for (int r = 1; 2 * r <= k; ++r)
        for (int s = r; r + s <= k; ++s)
            if (r + s >= k - 3) ++n_rects;
    if ((rc = dev_alloc((void **)&sw->ptilde_dev, 4ull * n_rects * sw->D1 * Pp * groups))) return rc;
    if ((rc = dev_alloc((void **)&sw->series_dev, 4ull * 3 * P * sw->n))) return rc;
    if ((rc = error_word_alloc(&sw->err))) return rc;
    if ((rc = build_strips(sw.get()))) return rc;
    const size_t log_words = series_scratch_words(series_params(sw.get()));
    if ((rc = dev_alloc((void **)&sw->logs_dev, 4 * log_words))) return rc;
    CP_CUDA_TRY(cudaMemset(sw->logs_dev, 0, 4 * log_words));
    if ((rc = dev_alloc((void **)&sw->rects_dev, sizeof(int2) * n_rects))) return rc;
    CP_CUDA_TRY(cudaMemcpy(sw->rects_dev, sw->rects.data(), sizeof(int2) * n_rects, cudaMemcpyHostToDevice));
    if ((rc = build_program(sw.get(), tile))) return rc;
    *out = sw.release();
    return CP_OK;
}

static int sweep_time_once(cp_sweep *sw, float *ms) {
    cudaEvent_t a, b;
    CP_CUDA_TRY(cudaEventCreate(&a));
    CP_CUDA_TRY(cudaEventCreate(&b));
    cudaError_t e = cudaGraphLaunch(sw->exec, sw->stream);  // warm-up
    if (e == cudaSuccess) e = cudaEventRecord(a, sw->stream);
    if (e == cudaSuccess) e = cudaGraphLaunch(sw->exec, sw->stream);
    if (e == cudaSuccess) e = cudaEventRecord(b, sw->stream);
    if (e == cudaSuccess) e = cudaEventSynchronize(b);
    if (e == cudaSuccess) e = cudaEventElapsedTime(ms, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    if (e != cudaSuccess) return fail(CP_ECUDA, std::string("autotune timing: ") + cudaGetErrorString(e));
    return CP_OK;
}

static std::mutex g_tune_mu;
static std::map<std::tuple<int, int, int, int>, int> g_tuned;  // (dev, lattice, k, P) -> groups

extern "C" int cp_sweep_create(int lattice, int k, const uint32_t *primes, int n_primes, int tile, int prime_groups,
                               void *cuda_stream, cp_sweep **out) {
    if (!out) return fail(CP_EINVAL, "out is NULL");
    *out = nullptr;
    if (lattice != CP_SQUARE && lattice != CP_TRIANGULAR) return fail(CP_EINVAL, "bad lattice");
    if (k < 4 || k / 2 > CP_MAX_L) return fail(CP_EINVAL, "k must satisfy 4 <= k and k/2 <= CP_MAX_L");
    if (n_terms_for(lattice, k) > kMaxSeries) return fail(CP_EINVAL, "k too large for the series kernel");
    int rc = check_primes(primes, n_primes);
    if (rc) return rc;
    if (!cuda_stream) return fail(CP_EINVAL, "the sweep needs a non-default stream (graph capture)");
    if (tile != 0 && !tile_valid(tile))
        return fail(CP_EINVAL, "tile must be 0 (default), 1, 2, 4, 8 (register kernel) or 16, 32, 64, 128 (chunk "
                               "kernel), the latter with (16..192 << 12), (1, 2, 4, 8 << 20), (1, 2, 4 << 24) or "
                               "(1, 2 << 28) or'ed in");
    if (prime_groups < 0 || (prime_groups > 0 && n_primes % prime_groups != 0))
        return fail(CP_EINVAL, "prime_groups must divide n_primes");
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (tile != 0 && prime_groups != 0) return sweep_build(lattice, k, primes, n_primes, tile, prime_groups, st, out);
    int dev = 0;
    CP_CUDA_TRY(cudaGetDevice(&dev));
    auto key = std::make_tuple(dev, lattice, k, n_primes);
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tuned.find(key);
        if (it != g_tuned.end())
            return sweep_build(lattice, k, primes, n_primes, tile ? tile : kTileChunk,
                               prime_groups ? prime_groups : it->second, st, out);
    }
    // autotune: for each prime grouping build the strips, time one graph run (after a
    // warm-up run) and keep the fastest grouping
    const int use = tile ? tile : kTileChunk;
    std::vector<int> grps;
    if (prime_groups) grps = {prime_groups};
    else
        for (int g : {1, 2})
            if (n_primes % g == 0 && (n_primes / g) % 4 == 0) grps.push_back(g);
    if (grps.empty()) grps = {1};
    float best = 1e30f;
    int bg = grps[0];
    for (int g : grps) {
        cp_sweep *cand = nullptr;
        if ((rc = sweep_build(lattice, k, primes, n_primes, use, g, st, &cand))) return rc;
        float ms = 0;
        rc = sweep_time_once(cand, &ms);
        if (!rc) rc = check_device_error(st);
        delete cand;
        if (rc) return rc;
        if (ms < best) {
            best = ms;
            bg = g;
        }
    }
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        g_tuned[key] = bg;
    }
    return sweep_build(lattice, k, primes, n_primes, use, bg, st, out);
}

extern "C" int cp_sweep_run(cp_sweep *sw) {
    if (!sw) return fail(CP_EINVAL, "sweep is NULL");
    CP_CUDA_TRY(cudaGraphLaunch(sw->exec, sw->stream));
    return CP_OK;
}

extern "C" int cp_sweep_sync(cp_sweep *sw) {
    if (!sw) return fail(CP_EINVAL, "sweep is NULL");
    int rc = check_device_error(sw->stream);
    if (rc) return rc;
    if (*(volatile int *)sw->err.host) return fail(CP_ESTATE, "a rectangle's P~ lacks constant term 1");
    return CP_OK;
}

extern "C" int cp_sweep_work(const cp_sweep *sw, uint64_t work[3]) {
    if (!sw || !work) return fail(CP_EINVAL, "NULL argument");
    work[0] = sw->updates;
    work[1] = sw->bytes;
    work[2] = sw->site_bytes;
    return CP_OK;
}

extern "C" int cp_sweep_window_bytes(cp_sweep *sw, uint64_t *bytes) {
    if (!sw || !bytes) return fail(CP_EINVAL, "NULL argument");
    unsigned long long *sum = nullptr, degrees = 0;
    int rc = dev_alloc((void **)&sum, 8);
    if (rc) return rc;
    uint64_t tables = 0;
    cudaError_t e = cudaMemsetAsync(sum, 0, 8, sw->stream);
    const int cap = sw->D1 - 1;
    for (auto &a : sw->applied) {
        if (rc || e != cudaSuccess) break;
        rc = add_window_degrees(a.tab->win_in, a.tab->n_src, a.v_in, a.first ? 0 : cap, sum, sw->stream);
        if (!rc)
            rc = add_window_degrees(a.tab->win_out, a.tab->n_dst, a.final ? kFinalVertices : a.v_in + a.tab->sites, cap, sum,
                                    sw->stream);
        tables += 8 * a.tab->nnz + 2 * a.tab->n_dst + 16ull * a.tab->n_units;
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&degrees, sum, 8, cudaMemcpyDeviceToHost, sw->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(sw->stream);
    dev_free(sum);
    if (rc) return rc;
    if (e != cudaSuccess) return fail(CP_ECUDA, std::string("window bytes: ") + cudaGetErrorString(e));
    *bytes = 4ull * sw->Pp * degrees + tables;
    return CP_OK;
}

extern "C" int cp_sweep_info(const cp_sweep *sw, int *n_rects, int *n_terms, int *tile, int *prime_groups,
                             uint64_t *updates_per_run, uint64_t *bytes_per_run, int *launches_per_run) {
    if (!sw) return fail(CP_EINVAL, "sweep is NULL");
    if (n_rects) *n_rects = (int)sw->rects.size();
    if (n_terms) *n_terms = sw->n;
    if (tile) *tile = sw->tile;
    if (prime_groups) *prime_groups = sw->groups;
    if (updates_per_run) *updates_per_run = sw->updates;
    if (bytes_per_run) *bytes_per_run = sw->bytes;
    if (launches_per_run) *launches_per_run = (int)sw->steps.size() + 1;
    return CP_OK;
}

extern "C" int cp_sweep_rects(const cp_sweep *sw, int *rs_host, int max_rects) {
    if (!sw || !rs_host) return fail(CP_EINVAL, "NULL argument");
    if (max_rects < (int)sw->rects.size()) return fail(CP_EINVAL, "max_rects too small");
    for (size_t j = 0; j < sw->rects.size(); ++j) {
        rs_host[2 * j] = sw->rects[j].x;
        rs_host[2 * j + 1] = sw->rects[j].y;
    }
    return CP_OK;
}

extern "C" int cp_sweep_read_ptilde(cp_sweep *sw, uint32_t *out_host, size_t out_len) {
    if (!sw || !out_host) return fail(CP_EINVAL, "NULL argument");
    const int nr = (int)sw->rects.size(), D1 = sw->D1, Pg = sw->Pg, Pp = sw->Pp;
    if (out_len < (size_t)nr * sw->P * D1) return fail(CP_EINVAL, "out_len < n_rects*n_primes*n_terms");
    std::vector<uint32_t> raw((size_t)sw->groups * nr * D1 * Pp);
    CP_CUDA_TRY(cudaStreamSynchronize(sw->stream));
    CP_CUDA_TRY(cudaMemcpy(raw.data(), sw->ptilde_dev, raw.size() * 4, cudaMemcpyDeviceToHost));
    for (int g = 0; g < sw->groups; ++g)
        for (int j = 0; j < nr; ++j)
            for (int d = 0; d < D1; ++d)
                for (int q = 0; q < Pg; ++q)
                    out_host[((size_t)j * sw->P + g * Pg + q) * D1 + d] = raw[(((size_t)g * nr + j) * D1 + d) * Pp + q];
    return CP_OK;
}

extern "C" int cp_sweep_read_series(cp_sweep *sw, uint32_t *out_host, size_t out_len) {
    if (!sw || !out_host) return fail(CP_EINVAL, "NULL argument");
    if (out_len < 3ull * sw->P * sw->n) return fail(CP_EINVAL, "out_len < 3*n_primes*n_terms");
    int rc = cp_sweep_sync(sw);
    if (rc) return rc;
    CP_CUDA_TRY(cudaMemcpy(out_host, sw->series_dev, 12ull * sw->P * sw->n, cudaMemcpyDeviceToHost));
    return CP_OK;
}

extern "C" int cp_sweep_read_series_device(cp_sweep *sw, uint32_t *out_dev, size_t out_len) {
    if (!sw || !out_dev) return fail(CP_EINVAL, "NULL argument");
    if (out_len < 3ull * sw->P * sw->n) return fail(CP_EINVAL, "out_len < 3*n_primes*n_terms");
    CP_CUDA_TRY(cudaMemcpyAsync(out_dev, sw->series_dev, 12ull * sw->P * sw->n, cudaMemcpyDeviceToDevice, sw->stream));
    return CP_OK;
}

extern "C" int cp_sweep_set_primes(cp_sweep *sw, const uint32_t *primes, int n_primes) {
    if (!sw) return fail(CP_EINVAL, "sweep is NULL");
    if (n_primes != sw->P) return fail(CP_EINVAL, "n_primes differs from the sweep's");
    int rc = check_primes(primes, n_primes);
    if (rc) return rc;
    const uint32_t was = *std::min_element(sw->primes_host.begin(), sw->primes_host.end());
    const uint32_t now = *std::min_element(primes, primes + n_primes);
    sw->primes_host.assign(primes, primes + n_primes);
    // primes that another kernel takes (fast_ok) need other launches
    bool other = false;
    for (auto &st : sw->strips)
        for (auto *chain : {&st.tabs->row, &st.tabs->last})
            for (auto &t : *chain) other = other || table_fast(t, was) != table_fast(t, now);
    if (other) {
        CP_CUDA_TRY(cudaStreamSynchronize(sw->stream));
        if ((rc = build_program(sw, sw->tile))) return rc;
    }
    const std::vector<uint32_t> lanes = prime_blocks(sw);
    CP_CUDA_TRY(cudaMemcpyAsync(sw->primes_dev, lanes.data(), 4 * lanes.size(), cudaMemcpyHostToDevice, sw->stream));
    return CP_OK;
}

extern "C" int cp_sweep_series_integers(cp_sweep *sw, uint32_t *limbs_out, size_t limbs_len, int limbs_per_coeff,
                                        uint32_t *flags_out) {
    if (!sw || !limbs_out) return fail(CP_EINVAL, "NULL argument");
    const int n = sw->n, P = sw->P;
    if (limbs_per_coeff < 1 || limbs_len < 3ull * n * limbs_per_coeff)
        return fail(CP_EINVAL, "limbs_len < 3*n_terms*limbs_per_coeff");
    int rc;
    const size_t need = 3ull * n * (limbs_per_coeff + 1);
    if (need > sw->crt_words) {
        CP_CUDA_TRY(cudaStreamSynchronize(sw->stream));
        dev_free(sw->crt_dev);
        sw->crt_dev = nullptr;
        sw->crt_words = 0;
        if ((rc = dev_alloc((void **)&sw->crt_dev, need * 4))) return rc;
        sw->crt_words = need;
    }
    uint32_t *limbs_d = sw->crt_dev, *flags_d = limbs_d + 3ull * n * limbs_per_coeff;
    if ((rc = launch_crt(sw->series_dev, sw->primes_host.data(), P, n, limbs_d, limbs_per_coeff, nullptr, flags_d,
                         sw->stream, 3)))
        return rc;
    std::vector<uint32_t> both(need);  // limbs, then flags: one copy
    CP_CUDA_TRY(cudaMemcpyAsync(both.data(), limbs_d, need * 4, cudaMemcpyDeviceToHost, sw->stream));
    if ((rc = cp_sweep_sync(sw))) return rc;
    const uint32_t *flags = both.data() + 3ull * n * limbs_per_coeff;
    std::copy((const uint32_t *)both.data(), flags, limbs_out);
    if (flags_out) std::copy(flags, flags + 3ull * n, flags_out);
    return crt_outcome(flags, 3 * n);
}

// The gathers store signed representatives; a run's series kernel puts residues in
// their place, and this does where it does not follow.  words: per prime group.
__global__ void ptilde_residues_kernel(uint32_t *ptilde, const uint32_t *primes, size_t words, int Pp) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= words) return;
    uint32_t *x = ptilde + blockIdx.y * words + i;
    if ((int)*x < 0) *x += primes[blockIdx.y * kPrimeWords + i % Pp];
}

static int launch_ptilde_residues(cp_sweep *sw) {
    const size_t words = sw->rects.size() * (size_t)sw->D1 * sw->Pp;
    ptilde_residues_kernel<<<dim3((unsigned)((words + 255) / 256), sw->groups), 256, 0, sw->stream>>>(
        sw->ptilde_dev, sw->primes_dev, words, sw->Pp);
    CP_CUDA_TRY(cudaGetLastError());
    return CP_OK;
}

// The same program without the graph, with an event pair around every batched
// gather launch: sum of gather kernel times and number of gather launches.
extern "C" int cp_sweep_profile(cp_sweep *sw, float *gather_ms, int *n_gather, float *total_ms) {
    if (!sw) return fail(CP_EINVAL, "sweep is NULL");
    const size_t nst = sw->steps.size();
    std::vector<cudaEvent_t> ev(2 * nst + 2);
    for (auto &e : ev) CP_CUDA_TRY(cudaEventCreate(&e));
    CP_CUDA_TRY(cudaEventRecord(ev[2 * nst], sw->stream));
    int rc = enqueue_reset(sw);
    for (size_t t = 0; t < nst && rc == CP_OK; ++t) {
        cudaEventRecord(ev[2 * t], sw->stream);
        rc = launch_gather(sw->steps[t].data(), (int)sw->steps[t].size(), sw->step_blocks[t], sw->step_tile[t], sw->stream);
        cudaEventRecord(ev[2 * t + 1], sw->stream);
    }
    CP_CUDA_TRY(cudaEventRecord(ev[2 * nst + 1], sw->stream));
    const int rr = launch_ptilde_residues(sw);
    if (!rc) rc = rr;
    cudaError_t e = cudaStreamSynchronize(sw->stream);
    float sum = 0, tot = 0;
    for (size_t t = 0; t < nst && e == cudaSuccess; ++t) {
        float ms = 0;
        e = cudaEventElapsedTime(&ms, ev[2 * t], ev[2 * t + 1]);
        sum += ms;
    }
    if (e == cudaSuccess) e = cudaEventElapsedTime(&tot, ev[2 * nst], ev[2 * nst + 1]);
    for (auto &x : ev) cudaEventDestroy(x);
    if (rc) return rc;
    if (e != cudaSuccess) return fail(CP_ECUDA, std::string("profile: ") + cudaGetErrorString(e));
    if (gather_ms) *gather_ms = sum;
    if (n_gather) *n_gather = (int)nst;
    if (total_ms) *total_ms = tot;
    return CP_OK;
}

extern "C" void cp_sweep_destroy(cp_sweep *sw) {
    if (!sw) return;
    cudaStreamSynchronize(sw->stream);
    delete sw;
}
