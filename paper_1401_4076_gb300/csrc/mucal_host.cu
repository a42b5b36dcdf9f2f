// Host side of libmucal: the C ABI declared in include/mucal.h, device memory
// management, the acceptance-threshold build and the weight iteration of
// Sec. 2 in double precision.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <utility>
#include <vector>

#include <cuda_runtime.h>

#include "mucal.h"
#include "mucal_internal.h"

using mucal::BlockWork;
using mucal::LaunchShape;
using mucal::SysParams;

namespace {

thread_local std::string g_init_error;

// Lists of all walkers up to this size stay in L2 (129 MB) by themselves.
constexpr size_t kListsInL2 = (size_t)64 << 20;

struct System {
    mucal_system_desc desc{};
    SysParams p{};                  // host copy holding device pointers
    std::vector<double> lnW;        // current log-weights over the window
    std::vector<uint8_t> visited;   // cumulative visited set (recursion memory)
    std::vector<double> pacc;       // accumulated pair weights (recursion memory)
    std::vector<int64_t> H;         // last summed histogram, host copy
    bool hist_on_host = false;
    int32_t t_lo = 0, t_hi = 0;     // target window (bins), -1 = default
    bool target_default = true;
    uint32_t *thr_pinned = nullptr; // staging buffer of the threshold upload
    size_t thr_count = 0;
    size_t h_off = 0;               // its place in the context's summed histograms
    bool hist_ahead = false;        // H came with another system's read, not asked for yet
    bool hist_shared = false;       // the caller has the device histogram's address
    uint64_t last_attempts = 0;
    std::vector<double> lnW_run;    // the weights of the last iteration's thresholds
    unsigned long long *drop_acc = nullptr;  // device [3][n_bins] droplet accumulators
    mucal::DropletPlan drop_plan{};          // of its droplet measurement, once made
    bool drop_planned = false;
    int32_t *drop_last = nullptr;            // device [n_walkers] V_D of the last measurement
};

struct Context {
    int device = -1;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    uint32_t flags = 0;
    std::vector<System> sys;
    SysParams *d_sys = nullptr;
    BlockWork *d_work = nullptr;
    int n_blocks = 0;
    int max_smem = 0;
    LaunchShape shape{};
    cudaEvent_t ev_it0 = nullptr, ev_k0 = nullptr, ev_k1 = nullptr, ev_it1 = nullptr;
    bool ran = false;
    uint64_t sweeps_last = 0;
    uint64_t launches = 0;
    int *d_drop_err = nullptr;           // droplet labelling failure flag
    uint32_t *drop_scratch = nullptr;    // global parent arrays for lattices too large for smem
    size_t drop_scratch_words = 0;
    bool measured = false;
    bool tunnel = false;                 // walker kernels with tunnelling bookkeeping
    int *d_next_item = nullptr;          // work-item counter of persistent launches
    // all systems' summed histograms and, behind them, the walker kernels' error
    // flag: one block, one clear and one copy per iteration for all systems
    unsigned long long *d_H = nullptr, *h_H = nullptr;   // device, pinned host
    size_t h_words = 0;                  // words of the histograms
    unsigned long long *d_hist = nullptr;    // all systems' histogram rows
    size_t hist_words = 0, hist_cap = 0;     // words in use, words allocated
    mucal::ReduceWork *d_reduce = nullptr;   // blocks of the histogram sum
    int n_reduce = 0;
    unsigned int *d_walk_err = nullptr;  // set by a walker kernel whose bounded wait ran out
    // CUDA-graph mode: one graph per (sweeps, launch shape, flavour, grid)
    bool graph_mode = false;
    cudaGraph_t graph = nullptr;         // kept: its nodes address the executable's
    cudaGraphExec_t graph_exec = nullptr;
    cudaGraphNode_t graph_walker = nullptr;  // the walker-update node (iteration changes)
    cudaKernelNodeParams graph_kp{};
    uint64_t graph_sweeps = 0;
    LaunchShape graph_shape{};
    bool graph_tunnel = false;
    int graph_grid = 0;
    uint32_t *d_xthr = nullptr;          // replica-exchange thresholds, [pairs][2 n_bins - 1]
    uint32_t *xthr_pinned = nullptr;     // their host staging buffer
    size_t xthr_words = 0;
    unsigned long long *d_xacc = nullptr, *xacc_pinned = nullptr;  // accepted exchanges per pair
    std::string err;
};

int fail(Context *c, int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    if (c)
        c->err = buf;
    else
        g_init_error = buf;
    return code;
}

// (a reported error is taken back from the runtime, which would hand it to the
// check behind the next launch)
#define CUDA_TRY(ctx, call)                                                                  \
    do {                                                                                     \
        cudaError_t e_ = (call);                                                             \
        if (e_ != cudaSuccess) {                                                             \
            cudaGetLastError();                                                              \
            return fail((ctx), e_ == cudaErrorMemoryAllocation ? MUCAL_ERR_OOM : MUCAL_ERR_CUDA, \
                        "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
        }                                                                                    \
    } while (0)

// ---------------------------------------------------------------------------
// Acceptance thresholds: min(1, W(E_n)/W(E_o)) of Sec. 2 as a uint32 per
// (E_o bin, dE).  Double precision, host libm exp; the device only compares.
// ---------------------------------------------------------------------------
void build_thresholds(const System &s, uint32_t *T)
{
    const int nb = s.p.n_bins;
    const int width = s.p.width;
    const int half = 2 * s.p.d;
    for (int b = 0; b < nb; ++b) {
        const double from = s.lnW[b];
        uint32_t *row = T + (size_t)b * s.p.tstride;
        for (int j = width; j < s.p.tstride; ++j) row[j] = 0u;   // refused: attempts past the end read it
        for (int j = 0; j < width; ++j) {
            const int to = b + (j - half);
            if (to < 0 || to >= nb) {
                row[j] = 0u;
                continue;
            }
            const double diff = s.lnW[to] - from;
            if (diff >= 0.0) {
                row[j] = 0xFFFFFFFFu;
                continue;
            }
            const double scaled = std::floor(std::ldexp(std::exp(diff), 32));
            row[j] = scaled >= 4294967294.0 ? 0xFFFFFFFEu : (uint32_t)scaled;
        }
    }
}

int upload_thresholds(Context *c, System &s)
{
    // The pinned staging buffer may still feed an earlier asynchronous copy.
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    build_thresholds(s, s.thr_pinned);
    CUDA_TRY(c, cudaMemcpyAsync((void *)s.p.thr, s.thr_pinned, s.thr_count * sizeof(uint32_t),
                                cudaMemcpyHostToDevice, c->stream));
    if (s.p.thrT) CUDA_TRY(c, mucal::launch_thr_transpose(s.p, c->stream));
    return MUCAL_OK;
}

// The dE-major table copies that multi-commit rounds with thresholds in
// global memory read: allocated when a launch shape first needs them, kept
// up to date by upload_thresholds from then on.
int ensure_thr_transposed(Context *c)
{
    for (auto &s : c->sys) {
        if (s.p.thrT) continue;
        const int pitch = (s.p.n_bins + 2 * mucal::kThrTPad + 3) & ~3;
        // (the row behind the last stays zero, as the padding of the table's rows)
        const size_t bytes = (size_t)(s.p.width + 1) * (size_t)pitch * sizeof(uint32_t);
        void *ptr = nullptr;
        CUDA_TRY(c, cudaMalloc(&ptr, bytes));
        s.p.thrT = static_cast<const uint32_t *>(ptr);
        s.p.thrT_pitch = pitch;
        CUDA_TRY(c, cudaMemsetAsync(ptr, 0, bytes, c->stream));
        CUDA_TRY(c, mucal::launch_thr_transpose(s.p, c->stream));
    }
    return MUCAL_OK;
}

void normalise_max_zero(double *w, int n)
{
    double mx = -INFINITY;
    for (int b = 0; b < n; ++b) mx = std::max(mx, w[b]);
    for (int b = 0; b < n; ++b) w[b] -= mx;
}

// W^{i+1} = W^i / H^i where H^i > 0 (Sec. 2), in logs.
void simple_step(int nb, const int64_t *H, double *lnW, uint8_t *visited)
{
    for (int b = 0; b < nb; ++b) {
        if (H[b] > 0) {
            visited[b] = 1;
            lnW[b] -= std::log((double)H[b]);
        }
    }
    normalise_max_zero(lnW, nb);
}

// Accumulated-statistics recursion on consecutive members of the cumulative
// visited set (the recursive scheme cited in Sec. 2).
void recursive_step(int nb, const int64_t *H, double *w, uint8_t *visited, double *pacc)
{
    for (int b = 0; b < nb; ++b)
        if (H[b] > 0) visited[b] = 1;
    std::vector<int> mem;
    mem.reserve(nb);
    for (int b = 0; b < nb; ++b)
        if (visited[b]) mem.push_back(b);
    if (mem.empty()) {
        normalise_max_zero(w, nb);
        return;
    }
    const std::vector<double> old(w, w + nb);
    // rebuild from the top member downwards
    for (size_t j = mem.size() - 1; j >= 1; --j) {
        const int hi = mem[j], lo = mem[j - 1];
        double lnr = old[hi] - old[lo];
        const double hlo = (double)H[lo], hhi = (double)H[hi];
        const double g = (hlo > 0.0 && hhi > 0.0) ? hlo * hhi / (hlo + hhi) : 0.0;
        pacc[hi] += g;
        if (g > 0.0) lnr += (g / pacc[hi]) * (std::log(hlo) - std::log(hhi));
        w[lo] = w[hi] - lnr;
    }
    // bins outside the visited set ride with the nearest member above
    // (or the top member when none is above)
    int next_member = -1;
    for (int b = nb - 1; b >= 0; --b) {
        if (visited[b]) {
            next_member = b;
            continue;
        }
        const int ref = next_member >= 0 ? next_member : mem.back();
        w[b] = old[b] + (w[ref] - old[ref]);
    }
    normalise_max_zero(w, nb);
}

// Edge continuation of the weights (MUCAL_SCHEME_EXTRAPOLATE): bins below
// the lowest visited bin and above the highest take lnW continued linearly
// with the slope between that edge and the kEdgeMembers-th visited bin
// counted inwards (canonical weights at the sampled edge's microcanonical
// temperature), so that walkers keep moving into the unsampled range.
constexpr int kEdgeMembers = 8;

void extrapolate_edges(int nb, double *w, const uint8_t *visited)
{
    std::vector<int> mem;
    for (int b = 0; b < nb; ++b)
        if (visited[b]) mem.push_back(b);
    if (mem.size() >= 2) {
        const size_t k = std::min<size_t>(kEdgeMembers, mem.size() - 1);
        const int first = mem.front(), last = mem.back();
        const int in_lo = mem[k], in_hi = mem[mem.size() - 1 - k];
        const double slope_lo = (w[in_lo] - w[first]) / (double)(in_lo - first);
        const double slope_hi = (w[last] - w[in_hi]) / (double)(last - in_hi);
        for (int b = 0; b < first; ++b) w[b] = w[first] + slope_lo * (double)(b - first);
        for (int b = last + 1; b < nb; ++b) w[b] = w[last] + slope_hi * (double)(b - last);
    }
    normalise_max_zero(w, nb);
}

// One weight update: the simple or the recursive step, then (flag) the edge
// continuation.
void update_step(int scheme, int nb, const int64_t *H, double *lnW, uint8_t *visited, double *pacc)
{
    if ((scheme & 0xF) == MUCAL_SCHEME_SIMPLE)
        simple_step(nb, H, lnW, visited);
    else
        recursive_step(nb, H, lnW, visited, pacc);
    if (scheme & MUCAL_SCHEME_EXTRAPOLATE) extrapolate_edges(nb, lnW, visited);
}

bool scheme_ok(int scheme)
{
    const int base = scheme & 0xF;
    return (base == MUCAL_SCHEME_SIMPLE || base == MUCAL_SCHEME_RECURSIVE) &&
           (scheme & ~(0xF | MUCAL_SCHEME_EXTRAPOLATE)) == 0;
}

// min/max of H over the visited bins of the target window [lo, hi] (bins;
// lo < 0 selects the visited range), -1 while an end of it is unvisited.
double flatness_of(int nb, const int64_t *H, const uint8_t *visited, int t_lo, int t_hi)
{
    int first = -1, last = -1;
    for (int b = 0; b < nb; ++b)
        if (visited[b]) {
            if (first < 0) first = b;
            last = b;
        }
    if (first < 0) return -1.0;
    const int lo = t_lo < 0 ? first : t_lo;
    const int hi = t_lo < 0 ? last : t_hi;
    if (!visited[lo] || !visited[hi]) return -1.0;
    double mn = INFINITY, mx = 0.0;
    for (int b = lo; b <= hi; ++b) {
        if (!visited[b]) continue;
        const double h = (double)H[b];
        mn = std::min(mn, h);
        mx = std::max(mx, h);
    }
    return mx > 0.0 ? mn / mx : 0.0;
}

double flatness(const System &s)
{
    return flatness_of(s.p.n_bins, s.H.data(), s.visited.data(), s.target_default ? -1 : s.t_lo,
                       s.t_hi);
}

int check_desc(const mucal_system_desc &d, int i)
{
    if (d.d != 2 && d.d != 3) return fail(nullptr, MUCAL_ERR_INVALID_ARG, "system %d: d must be 2 or 3", i);
    if (d.L < 3 || d.L > 4096) return fail(nullptr, MUCAL_ERR_INVALID_ARG, "system %d: L must be in [3, 4096]", i);
    const uint64_t V = d.d == 2 ? (uint64_t)d.L * d.L : (uint64_t)d.L * d.L * d.L;
    if (V > (1u << 24) || V * (uint64_t)d.L >= (1ull << 32))
        return fail(nullptr, MUCAL_ERR_INVALID_ARG, "system %d: lattice too large", i);
    if (d.N <= 0 || (uint64_t)d.N >= V)
        return fail(nullptr, MUCAL_ERR_INVALID_ARG, "system %d: need 0 < N < L^d", i);
    if (d.n_walkers <= 0) return fail(nullptr, MUCAL_ERR_INVALID_ARG, "system %d: n_walkers must be > 0", i);
    if (!(d.e_lo == 0 && d.e_hi == 0)) {
        if (d.e_lo < -d.d * d.N || d.e_hi > 0 || d.e_lo >= d.e_hi)
            return fail(nullptr, MUCAL_ERR_INVALID_ARG,
                        "system %d: window must satisfy -dN <= e_lo < e_hi <= 0", i);
    }
    return MUCAL_OK;
}

void free_system(System &s)
{
    cudaFree(s.p.bits);
    cudaFree(s.p.S);
    cudaFree(s.p.E);
    cudaFree((void *)s.p.thr);
    cudaFree((void *)s.p.thrT);
    cudaFree(s.p.accepts);
    if (s.thr_pinned) cudaFreeHost(s.thr_pinned);
    cudaFree(s.drop_acc);
    cudaFree(s.drop_last);
    cudaFree(s.p.tun_state);
    cudaFree(s.p.tun_count);
    s.p = SysParams{};
    s.thr_pinned = nullptr;
    s.drop_acc = nullptr;
    s.drop_last = nullptr;
}

void destroy_context(Context *c)
{
    if (!c) return;
    if (c->device >= 0) cudaSetDevice(c->device);
    if (c->stream) cudaStreamSynchronize(c->stream);
    for (auto &s : c->sys) free_system(s);
    cudaFree(c->d_sys);
    cudaFree(c->d_work);
    cudaFree(c->d_drop_err);
    cudaFree(c->drop_scratch);
    cudaFree(c->d_xthr);
    cudaFree(c->d_xacc);
    if (c->xthr_pinned) cudaFreeHost(c->xthr_pinned);
    if (c->xacc_pinned) cudaFreeHost(c->xacc_pinned);
    cudaFree(c->d_next_item);
    cudaFree(c->d_H);
    if (c->h_H) cudaFreeHost(c->h_H);
    cudaFree(c->d_hist);
    cudaFree(c->d_reduce);
    if (c->graph_exec) cudaGraphExecDestroy(c->graph_exec);
    if (c->graph) cudaGraphDestroy(c->graph);
    if (c->ev_it0) cudaEventDestroy(c->ev_it0);
    if (c->ev_k0) cudaEventDestroy(c->ev_k0);
    if (c->ev_k1) cudaEventDestroy(c->ev_k1);
    if (c->ev_it1) cudaEventDestroy(c->ev_it1);
    if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
    delete c;
}

// Shared memory a block of the given shape needs for system p.
size_t smem_for(const LaunchShape &sh, const SysParams &p)
{
    size_t bytes = 0;
    if (sh.thr_in_smem) bytes += mucal::thr_smem_words(p) * sizeof(uint32_t);
    if (sh.kernel == MUCAL_KERNEL_FIELD)
        bytes += (size_t)sh.walkers_per_block * mucal::field_smem_bytes(p);
    else if (sh.bits_in_smem)
        bytes += (size_t)sh.walkers_per_block * (size_t)p.words * sizeof(uint32_t);
    // the windows start on the next 16-byte boundary behind the bitsets or fields
    if (!sh.thr_in_smem && (sh.thr_window || sh.scan_window) && sh.kernel != MUCAL_KERNEL_THREAD)
        bytes += 16 + (size_t)sh.walkers_per_block * mucal::thr_window_bytes(p);
    return bytes;
}

void drop_graph(Context *c);

// Split every system's walkers into blocks of the launch shape; order the
// blocks by decreasing cost (attempts per walker grow with N) so the longest
// blocks start first when systems of uneven size share one launch.  The
// histogram rows are allocated here, as many as the shape needs (one per
// block: 23 MB instead of one per walker, 644 MB, on 3D L = 32 with 8192
// walkers), and grow when a shape needs more.
int build_work(Context *c, const LaunchShape &sh)
{
    std::vector<BlockWork> work;
    std::vector<int32_t> rows_of(c->sys.size(), 0);
    const bool per_walker = (c->flags & MUCAL_FLAG_PER_WALKER_HIST) != 0;
    for (int s = 0; s < (int)c->sys.size(); ++s) {
        const SysParams &p = c->sys[s].p;
        int rows = 0;
        for (int w0 = 0; w0 < p.n_walkers; w0 += sh.walkers_per_block) {
            BlockWork bw{};
            bw.sys = s;
            bw.walker0 = w0;
            bw.count = std::min(sh.walkers_per_block, p.n_walkers - w0);
            bw.hist_row = per_walker ? -1 : rows;
            ++rows;
            work.push_back(bw);
        }
        rows_of[s] = per_walker ? p.n_walkers : rows;
    }
    std::stable_sort(work.begin(), work.end(), [&](const BlockWork &a, const BlockWork &b) {
        const double ca = (double)c->sys[a.sys].p.N * c->sys[a.sys].p.d;
        const double cb = (double)c->sys[b.sys].p.N * c->sys[b.sys].p.d;
        return ca > cb;
    });
    std::vector<mucal::ReduceWork> reduce;
    std::vector<size_t> off(c->sys.size(), 0);
    size_t words = 0;
    for (int s = 0; s < (int)c->sys.size(); ++s) {
        const int bins = c->sys[s].p.n_bins;
        off[s] = words;
        words += (size_t)rows_of[s] * (size_t)bins;
        for (int r = 0; r < rows_of[s]; r += mucal::kReduceRows)
            for (int b = 0; b < bins; b += mucal::kReduceBins) reduce.push_back({s, b, r});
    }
    // build the new tables completely before replacing the old ones, so that
    // a failure leaves the previous launch shape usable
    BlockWork *d_work = nullptr;
    mucal::ReduceWork *d_reduce = nullptr;
    unsigned long long *d_hist = nullptr;
    cudaError_t e = cudaMalloc(&d_work, work.size() * sizeof(BlockWork));
    if (e == cudaSuccess) e = cudaMalloc(&d_reduce, reduce.size() * sizeof(mucal::ReduceWork));
    if (e == cudaSuccess)
        e = cudaMemcpy(d_work, work.data(), work.size() * sizeof(BlockWork), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(d_reduce, reduce.data(), reduce.size() * sizeof(mucal::ReduceWork),
                       cudaMemcpyHostToDevice);
    if (e == cudaSuccess && words > c->hist_cap) e = cudaMalloc(&d_hist, words * 8);
    std::vector<SysParams> hp(c->sys.size());
    for (size_t i = 0; i < c->sys.size(); ++i) {
        hp[i] = c->sys[i].p;
        hp[i].hist_rows = rows_of[i];
        hp[i].hist = (d_hist ? d_hist : c->d_hist) + off[i];
    }
    if (e == cudaSuccess)
        e = cudaMemcpy(c->d_sys, hp.data(), hp.size() * sizeof(SysParams), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaGetLastError();
        cudaFree(d_work);
        cudaFree(d_reduce);
        cudaFree(d_hist);
        // restore the device table of the current shape
        std::vector<SysParams> cur(c->sys.size());
        for (size_t i = 0; i < c->sys.size(); ++i) cur[i] = c->sys[i].p;
        cudaMemcpy(c->d_sys, cur.data(), cur.size() * sizeof(SysParams), cudaMemcpyHostToDevice);
        return fail(c, e == cudaErrorMemoryAllocation ? MUCAL_ERR_OOM : MUCAL_ERR_CUDA,
                    "launch table upload failed: %s", cudaGetErrorString(e));
    }
    drop_graph(c);               // a captured iteration holds the old tables and rows
    cudaFree(c->d_work);
    cudaFree(c->d_reduce);
    c->d_work = d_work;
    c->n_blocks = (int)work.size();
    c->d_reduce = d_reduce;
    c->n_reduce = (int)reduce.size();
    if (d_hist) {
        cudaFree(c->d_hist);
        c->d_hist = d_hist;
        c->hist_cap = words;
    }
    c->hist_words = words;
    for (size_t i = 0; i < c->sys.size(); ++i) {
        c->sys[i].p.hist_rows = rows_of[i];
        c->sys[i].p.hist = hp[i].hist;
    }
    return MUCAL_OK;
}

int apply_launch_config(Context *c, const mucal_launch_config &cfg)
{
    LaunchShape sh{};
    sh.kernel = cfg.kernel;
    sh.lanes = cfg.lanes_per_walker;
    sh.walkers_per_block = cfg.walkers_per_block;
    sh.bits_in_smem = cfg.bits_in_smem ? 1 : 0;
    sh.persistent = cfg.persistent ? 1 : 0;
    if (cfg.thr_window < 0 || cfg.thr_window > 2)
        return fail(c, MUCAL_ERR_INVALID_ARG, "thr_window must be 0, 1 or 2");
    sh.thr_window = cfg.kernel != MUCAL_KERNEL_THREAD ? cfg.thr_window : 0;
    if (cfg.multi_commit < 0 || cfg.multi_commit > 1)
        return fail(c, MUCAL_ERR_INVALID_ARG, "multi_commit must be 0 or 1");
    sh.multi_commit = cfg.kernel != MUCAL_KERNEL_THREAD && cfg.lanes_per_walker >= 4 ? cfg.multi_commit : 0;
    if (sh.kernel == MUCAL_KERNEL_THREAD) {
        if (sh.lanes != 1)
            return fail(c, MUCAL_ERR_INVALID_ARG, "THREAD kernel needs lanes_per_walker = 1");
        if (sh.walkers_per_block > 512)
            return fail(c, MUCAL_ERR_INVALID_ARG, "THREAD kernel blocks hold at most 512 threads");
    } else if (sh.kernel == MUCAL_KERNEL_GROUP || sh.kernel == MUCAL_KERNEL_FIELD) {
        const char *name = sh.kernel == MUCAL_KERNEL_GROUP ? "GROUP" : "FIELD";
        if (sh.lanes != 2 && sh.lanes != 4 && sh.lanes != 8 && sh.lanes != 16 && sh.lanes != 32)
            return fail(c, MUCAL_ERR_INVALID_ARG, "%s kernel needs lanes_per_walker in {2,4,8,16,32}", name);
        if ((sh.walkers_per_block * sh.lanes) % 32 != 0)
            return fail(c, MUCAL_ERR_INVALID_ARG, "%s kernel needs whole warps per block", name);
        if (sh.walkers_per_block * sh.lanes > 512)
            return fail(c, MUCAL_ERR_INVALID_ARG, "%s kernel blocks hold at most 512 threads", name);
        if (sh.kernel == MUCAL_KERNEL_FIELD && !sh.bits_in_smem)
            return fail(c, MUCAL_ERR_INVALID_ARG, "FIELD kernel keeps its counts in shared memory: "
                                                  "bits_in_smem must be 1");
    } else {
        return fail(c, MUCAL_ERR_INVALID_ARG, "unknown kernel %d", sh.kernel);
    }
    if (sh.walkers_per_block < 1 || sh.walkers_per_block * sh.lanes > 1024)
        return fail(c, MUCAL_ERR_INVALID_ARG, "walkers_per_block * lanes must be in [1, 1024]");
    // the threshold table joins the bitsets in shared memory whenever every
    // system's table fits next to its block of bitsets
    sh.thr_in_smem = 1;
    for (auto &s : c->sys)
        if (smem_for(sh, s.p) > (size_t)c->max_smem) sh.thr_in_smem = 0;
    if (cfg.thr_window == 2 && sh.thr_window) sh.thr_in_smem = 0;   // windows even if the table fits
    size_t smem = 0;
    for (auto &s : c->sys) smem = std::max(smem, smem_for(sh, s.p));
    if (smem > (size_t)c->max_smem && sh.thr_window) {
        // the threshold-row windows do not fit next to this block of walkers:
        // read the thresholds from global memory instead
        sh.thr_window = 0;
        smem = 0;
        for (auto &s : c->sys) smem = std::max(smem, smem_for(sh, s.p));
    }
    if (smem > (size_t)c->max_smem)
        return fail(c, MUCAL_ERR_INVALID_ARG, "launch needs %zu bytes of shared memory, limit %d",
                    smem, c->max_smem);
    if (!sh.thr_in_smem && sh.thr_window) sh.multi_commit = 0;   // one-commit rounds read row windows
    if (sh.multi_commit && !sh.thr_in_smem) {
        // rounds with several commits keep windows of their own where they fit
        sh.scan_window = 1;
        size_t with = 0;
        for (auto &s : c->sys) with = std::max(with, smem_for(sh, s.p));
        if (with <= (size_t)c->max_smem) smem = with;
        else sh.scan_window = 0;
    }
    sh.smem_bytes = smem;
    if (sh.multi_commit && !sh.thr_in_smem && !sh.scan_window) {
        const int rc = ensure_thr_transposed(c);
        if (rc != MUCAL_OK) return rc;
    }
    CUDA_TRY(c, mucal::walker_update_allow_smem(sh, c->max_smem));
    int rc = build_work(c, sh);
    if (rc != MUCAL_OK) return rc;
    c->shape = sh;
    return MUCAL_OK;
}

// Lanes per walker (the window of attempts a round decides) for r walkers
// beside each other on an SM and N particles.
//
// Two attempts of a window touch with a chance of about 3 / N, which bounds
// the useful window; below that, few walkers leave issue slots for wider
// windows, many need narrow ones, whose instructions per attempt are fewer.
// Measured on GB300 (ms of the walker update at 4 / 8 / 16 / 32 lanes): 3D
// L = 33, N = 3244, r = 1: 8.86 / 5.06 / 3.37 / 2.85; 3D L = 24, N = 1382,
// r = 14: 7.75 / 4.51 / 3.82 / 6.9; 3D L = 32, N = 3277, r = 28: 18.3 / 12.4 /
// 13.0 / -; 2D L = 64, N = 410, r = 1: 4.29 / 2.74 / 2.28 / 2.79, r = 10: 4.35 /
// 2.80 / 3.05 / 7.3; 3D L = 8, N = 56, r = 56: 1.44 / 1.98 / 5.2 / -.
// Narrow windows pay while moves are accepted; where they are refused, wide
// ones pass over more at a time.  Only where more than 48 walkers of few
// particles share an SM, so that instructions bound them, are 4 lanes no loss
// against one commit per round (8 lanes) at any acceptance.  The time of one
// commit per round over that of several at 4 and at 8 lanes, at acceptance 1, 0.35,
// 0.15 and 0.05: 2D L = 12, N = 18, r = 16 1.09, 0.86, 0.69, 0.62 and 0.95, 0.93,
// 0.90, 1.00; r = 32 1.26, 1.01, 0.82, 0.74 and 0.82, 0.84, 0.86, 1.02; r = 56 1.40,
// 1.12, 0.95, 0.95 and 0.76, 0.76, 0.80, 1.04; 2D L = 34, N = 47, r = 16 (acceptance
// 1, 0.33, 0.09, 0.01) 1.30, 0.91, 0.68, 0.61 and 1.58, 1.26, 1.02, 1.02; r = 56 1.59,
// 1.15, 0.95, 0.99 and 1.23, 0.97, 0.97, 1.23.  At 16 lanes 2D L = 45, N = 80, r = 4
// gains 2.01, 1.40, 1.21 and 1.60.
//
// More than 64 walkers beside each other have registers at 4 lanes only (512
// threads of 128).  One system in one wave at 4 lanes against two waves at 8 (and
// 32 walkers a block at 16, and one commit per round), at acceptance 1, 0.3 and
// 0.03: 2D L = 26, N = 80, r = 100 1.41, 0.97 and 0.59 ms against 1.81, 1.42 and
// 0.63 (4.67, 2.89 and 0.77; 1.92, 1.19 and 0.65); 2D L = 58, N = 400, r = 72
// 1.31, 0.77 and 0.53 against 1.07, 0.94 and 0.56.
int default_lanes(long long r, double N, bool one)
{
    if ((N < 64 && r > 48) || (one && r > 64)) return 4;
    if (N >= 2500 && r <= 7) return 32;
    if ((N >= 1000 && r <= 24) || (N >= 60 && r <= 4)) return 16;
    return 8;
}

// The launch shape of a new context: several commits per round.
//
// A walker is a serial chain, so what counts is that all walkers run at once,
// or in equal waves, with as many of them beside each other on an SM as its
// shared memory holds.  One system: its walkers per SM are split into the
// fewest waves that fit, one block per SM and wave.  Measured (blocks of 16
// walkers against this rule): 2D L = 64, N = 410, 4096 walkers, 20 sweeps
// 1.24 -> 1.17 ms (28 walkers, one wave); 3D L = 32, N = 3277, 8192 walkers, 10
// sweeps 15.9 -> 12.4 (28, two waves).  Several systems: small blocks, which
// pack their uneven bitsets and lengths best (the 27-system batch, 5 sweeps:
// 4 walkers 9.2, 14 walkers 10.9), of 8 walkers where a block stages the
// table, or of 16, or with bitsets for count fields, where these make fewer waves
// with a table in every block: five systems of 3D L = 14, N = 300, 540 walkers, 10
// sweeps, 8 -> 16 walkers at acceptance 1, 0.1 and 0.01 1.24, 0.85 and 0.97 times the
// speed of one commit per round -> 1.73, 1.28 and 1.54; six of 3D L = 23, N = 300, 280
// walkers, fields -> bitsets 1.45, 0.85 and 0.90 -> 2.88, 1.59 and 1.72.
//
// Count fields (two byte loads per attempt instead of 4d words, 4d more
// atomics per commit) where they fit 16 walkers to a block and do not cost a
// resident walker: 2D L = 64 3.24 (bitsets) -> 3.11, but five 2D systems of
// L = 61 to 97, 5120 walkers, 50 sweeps 1.06 (bitsets) against 1.9.
//
// Below 12 particles, and on small dense lattices above, nearly every window
// holds a conflict, and the rounds with one commit (8 lanes, 16 walkers a block)
// are the faster ones.  What counts is the chance that two attempts touch (a
// list slot in common, 1 / N and 1 / (V - N), or sites next to each other, 8 d /
// V) and whether latency (few walkers per SM) or instructions (many) bound the
// rounds.  The time of one commit per round over that of several at 8 lanes, the
// worst and best over acceptances from 1 to 0.001: at r = 11 touch 0.25 (2D
// L = 10, N = 12) 0.82 to 1.26, 0.21 (L = 11, N = 14) 0.88 to 1.26, 0.17 (L = 12,
// N = 18) 0.89 to 1.26, 0.13 (L = 14, N = 24) 0.94 to 1.31, 0.07 (L = 24, N = 24)
// 0.99 to 1.35; at r = 32 touch 0.17 0.82 to 1.34, 0.10 (L = 16, N = 30) 0.90 to
// 1.41, at r = 40 0.86 to 1.47, 0.09 (L = 17, N = 36) 0.89 to 1.47, 0.06 (L = 20,
// N = 47) 0.90 to 1.48, 0.05 (L = 30, N = 36) 0.95 to 1.40.
// They take count fields where 48 walkers, or all there are, are resident on an SM
// in blocks of 16 (ms, fields and bitsets): 2D L = 60, N = 8, 48 a wave, 108 per SM
// 3.64 and 4.07; 2D L = 80, N = 10, 32 a wave, 30 per SM 1.20 and 1.46, 48 2.11 and
// 1.87, 64 2.38 and 2.34, 100 4.35 and 3.98; 2D L = 100, N = 11, 16 a wave, 48 per SM
// 2.85 and 1.85.
// Lattices whose bitsets stay in global memory (2D L = 1400) have a few
// particles far apart, and several commits pay from 8 on (3 and 512 walkers,
// 4000 attempts): N = 4 1.43 and 2.32 against 1.98 and 2.54, N = 8 1.36 and 2.45
// against 1.36 and 1.81, N = 11 1.32 and 2.48 against 1.16 and 1.56.
mucal_launch_config default_launch(Context *c)
{
    long long total = 0;
    double work = 0.0, work_n = 0.0, work_t = 0.0;
    for (auto &s : c->sys) {
        const double n = s.p.N, v = s.p.V, w = s.p.n_walkers * n;
        total += s.p.n_walkers;
        work += w;
        work_n += w * n;
        work_t += w * (1.0 / n + 1.0 / (v - n) + 8.0 * s.p.d / v);
    }
    const double N = work_n / work;     // particles of the system an average attempt belongs to
    const double touch = work_t / work; // chance that two attempts touch
    int sms = 1, sm_smem = 0, reserved = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
    cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, c->device);
    cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, c->device);
    const long long need = (total + sms - 1) / sms;     // walkers per SM
    // whether w walkers fit a block: 0 no, 1 with row windows, 2 with the table
    auto fits = [&](int kernel, int w) {
        for (int table = 1; table >= 0; --table) {
            LaunchShape sh{};
            sh.kernel = kernel;
            sh.walkers_per_block = w;
            sh.bits_in_smem = 1;
            sh.thr_in_smem = table;
            sh.scan_window = 1;
            bool ok = true;
            for (auto &s : c->sys) ok = ok && smem_for(sh, s.p) <= (size_t)c->max_smem;
            if (ok) return 1 + table;
        }
        return 0;
    };
    // shared memory of a block of w walkers, with the table where it fits
    auto block_smem = [&](int kernel, int w) {
        LaunchShape sh{};
        sh.kernel = kernel;
        sh.walkers_per_block = w;
        sh.bits_in_smem = sh.scan_window = 1;
        sh.thr_in_smem = fits(kernel, w) == 2 ? 1 : 0;
        size_t smem = 0;
        for (auto &s : c->sys) smem = std::max(smem, smem_for(sh, s.p));
        return (int)smem;
    };
    const int overhead = mucal::kWalkerStaticSmem + reserved;    // beside it
    auto plain_fits = [&](int kernel) {      // without table and windows
        LaunchShape sh{};
        sh.kernel = kernel;
        sh.walkers_per_block = 16;
        sh.bits_in_smem = 1;
        bool ok = true;
        for (auto &s : c->sys) ok = ok && smem_for(sh, s.p) <= (size_t)c->max_smem;
        return ok;
    };
    auto most = [&](int kernel) {            // walkers an SM's shared memory holds
        int w = 0;
        while (w < 128 && fits(kernel, w + 1)) ++w;
        return w;
    };
    mucal_launch_config def{MUCAL_KERNEL_GROUP, 8, 16, 1, 0, 0, 1};
    long long cap = most(MUCAL_KERNEL_GROUP);
    if (cap < 1) {                           // bitsets in global memory
        def.bits_in_smem = 0;
        if (N < 8) {
            def.multi_commit = 0;
            def.thr_window = 1;
        } else {
            def.lanes_per_walker = std::max(8, default_lanes(need, N, true));
        }
        return def;
    }
    if (plain_fits(MUCAL_KERNEL_FIELD)) {
        const int f = most(MUCAL_KERNEL_FIELD);
        if (f >= need || f >= cap) {
            def.kernel = MUCAL_KERNEL_FIELD;
            cap = f;
        }
    }
    const bool one = c->sys.size() == 1;
    // walkers per SM of one of the fewest equal waves, `room` walkers at a time
    auto wave = [&](long long room) {
        const long long waves = (need + room - 1) / room;
        return (need + waves - 1) / waves;
    };
    const long long r = one ? wave(cap) : std::min(need, cap);
    if (N < 12 || (r <= 16 && touch > 0.175) || (r > 16 && r <= 48 && touch > 0.08)) {
        def.multi_commit = 0;
        def.thr_window = 1;
        def.kernel = MUCAL_KERNEL_GROUP;
        if (plain_fits(MUCAL_KERNEL_FIELD)) {
            const long long resident = 16 * (sm_smem / (block_smem(MUCAL_KERNEL_FIELD, 16) + reserved + 64));
            if (resident >= std::min<long long>(need, 48)) def.kernel = MUCAL_KERNEL_FIELD;
        }
        if (!plain_fits(def.kernel)) def.bits_in_smem = 0;
        return def;
    }
    int lanes = default_lanes(r, N, one);
    long long want = r;
    if (!one) {
        // waves of blocks of w walkers that stage the table (0: it does not fit)
        auto waves = [&](int kernel, int w) -> long long {
            if (fits(kernel, w) != 2) return 0;
            long long blocks = 0;
            for (auto &s : c->sys) blocks += (s.p.n_walkers + w - 1) / w;
            const int threads = std::max(32, w * lanes);
            const long long per_sm = std::min<long long>({sm_smem / (block_smem(kernel, w) + overhead),
                                                          512 / threads, 32});
            return (blocks + sms * per_sm - 1) / (sms * per_sm);
        };
        long long least = waves(def.kernel, 8);
        want = least ? 8 : 4;
        const std::pair<int, int> others[] = {
            {def.kernel, 16}, {MUCAL_KERNEL_GROUP, 8}, {MUCAL_KERNEL_GROUP, 16}};
        for (auto &o : others) {
            const long long n = least > 1 ? waves(o.first, o.second) : 0;
            if (n == 0 || n >= least) continue;
            least = n;
            def.kernel = o.first;
            want = o.second;
        }
        cap = most(def.kernel);
    }
    // whole warps: blocks of 32 / lanes walkers and multiples, of at most 512 threads
    for (;;) {
        const long long step = 32 / lanes;
        const long long top = std::min<long long>(cap, 512 / lanes) / step * step;
        const long long w = (want + step - 1) / step * step;
        if (top >= step && w <= top) {
            def.lanes_per_walker = lanes;
            def.walkers_per_block = (int)w;
            return def;
        }
        // wider groups come in finer blocks; else more waves
        const long long fine = step / 2, finer = std::min<long long>(cap, 256 / lanes);
        if (top < step || (fine > 0 && (want + fine - 1) / fine * fine <= finer)) {
            lanes *= 2;
            continue;
        }
        want = one ? wave(top) : top;
        lanes = std::max(lanes, default_lanes(want, N, one));
    }
}

Context *as_ctx(void *p) { return static_cast<Context *>(p); }

int check_sys(Context *c, int32_t s)
{
    if (!c) return MUCAL_ERR_INVALID_ARG;
    if (s < 0 || s >= (int32_t)c->sys.size())
        return fail(c, MUCAL_ERR_INVALID_ARG, "system index %d out of range", s);
    return MUCAL_OK;
}

// Every system's summed histogram to the host, with the error flag behind
// them, by one copy into pinned memory (a copy per system and one for the
// flag, both pageable, cost an 8-system tempering round 0.13 ms).  A system
// whose device histogram the caller can write to is copied at its own first
// read only.
int fetch_histogram(Context *c, System &s)
{
    if (!c->ran) return fail(c, MUCAL_ERR_NOT_READY, "no iteration has been run");
    s.hist_ahead = false;
    if (s.hist_on_host) return MUCAL_OK;
    CUDA_TRY(c, cudaMemcpyAsync(c->h_H, c->d_H, (c->h_words + 1) * 8, cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    const unsigned int err = (unsigned int)c->h_H[c->h_words];
    if (err) {
        CUDA_TRY(c, cudaMemsetAsync(c->d_walk_err, 0, 8, c->stream));
        return fail(c, MUCAL_ERR_STATE, "a walker kernel's wait for its threshold rows ran out "
                                        "(flag %u); the iteration's results are not valid", err);
    }
    for (auto &q : c->sys) {
        if (q.hist_on_host || (&q != &s && q.hist_shared)) continue;
        std::memcpy(q.H.data(), c->h_H + q.h_off, q.H.size() * sizeof(int64_t));
        q.hist_on_host = true;
        q.hist_ahead = &q != &s;
    }
    return MUCAL_OK;
}

// Copy the host copies of every system's parameters to the device table,
// keeping the histogram rows of the current launch shape.
int upload_sys_table(Context *c)
{
    std::vector<SysParams> hp(c->sys.size());
    for (size_t i = 0; i < c->sys.size(); ++i) hp[i] = c->sys[i].p;
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    CUDA_TRY(c, cudaMemcpy(c->d_sys, hp.data(), hp.size() * sizeof(SysParams), cudaMemcpyHostToDevice));
    return MUCAL_OK;
}

int reset_tunnel(Context *c, const System &s)
{
    CUDA_TRY(c, cudaMemsetAsync(s.p.tun_state, 0, (size_t)s.p.n_walkers, c->stream));
    CUDA_TRY(c, cudaMemsetAsync(s.p.tun_count, 0, (size_t)s.p.n_walkers * 4, c->stream));
    return MUCAL_OK;
}

// The device work of one iteration, asynchronous on the context's stream:
// clear the histograms, the walker update, the histogram sums, with the
// timing events around them unless it is being captured into a graph (the
// graph launch is timed from outside instead).
int enqueue_iteration(Context *c, uint64_t sweeps, uint32_t iteration, int grid, bool events)
{
    if (events) CUDA_TRY(c, cudaEventRecord(c->ev_it0, c->stream));
    CUDA_TRY(c, cudaMemsetAsync(c->d_hist, 0, c->hist_words * 8, c->stream));
    CUDA_TRY(c, cudaMemsetAsync(c->d_H, 0, c->h_words * 8, c->stream));
    if (c->shape.persistent) CUDA_TRY(c, cudaMemsetAsync(c->d_next_item, 0, sizeof(int), c->stream));
    if (events) CUDA_TRY(c, cudaEventRecord(c->ev_k0, c->stream));
    CUDA_TRY(c, mucal::launch_walker_update(c->d_sys, c->d_work, c->n_blocks, c->shape, sweeps,
                                            iteration, c->tunnel, grid, c->d_next_item, c->stream));
    if (events) CUDA_TRY(c, cudaEventRecord(c->ev_k1, c->stream));
    CUDA_TRY(c, mucal::launch_hist_reduce(c->d_sys, c->d_reduce, c->n_reduce, c->stream));
    if (events) CUDA_TRY(c, cudaEventRecord(c->ev_it1, c->stream));
    return MUCAL_OK;
}

// Capture enqueue_iteration into a CUDA graph on the context's stream,
// instantiate it and remember its walker-update node.
void drop_graph(Context *c)
{
    if (c->graph_exec) cudaGraphExecDestroy(c->graph_exec);
    if (c->graph) cudaGraphDestroy(c->graph);
    c->graph_exec = nullptr;
    c->graph = nullptr;
    c->graph_walker = nullptr;
}

int capture_iteration(Context *c, uint64_t sweeps, uint32_t iteration, int grid)
{
    drop_graph(c);
    CUDA_TRY(c, cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal));
    const int rc = enqueue_iteration(c, sweeps, iteration, grid, false);
    cudaGraph_t graph = nullptr;
    const cudaError_t end = cudaStreamEndCapture(c->stream, &graph);
    if (rc != MUCAL_OK) {
        if (graph) cudaGraphDestroy(graph);
        return rc;
    }
    CUDA_TRY(c, end);
    const void *fn = mucal::walker_update_fn(c->shape, c->tunnel);
    size_t n = 0;
    cudaError_t e = cudaGraphGetNodes(graph, nullptr, &n);
    std::vector<cudaGraphNode_t> nodes(n);
    if (e == cudaSuccess) e = cudaGraphGetNodes(graph, nodes.data(), &n);
    for (size_t i = 0; e == cudaSuccess && i < n && !c->graph_walker; ++i) {
        cudaGraphNodeType t;
        e = cudaGraphNodeGetType(nodes[i], &t);
        if (e != cudaSuccess || t != cudaGraphNodeTypeKernel) continue;
        cudaKernelNodeParams kp{};
        e = cudaGraphKernelNodeGetParams(nodes[i], &kp);
        if (e == cudaSuccess && kp.func == fn) {
            c->graph_walker = nodes[i];
            c->graph_kp = kp;
        }
    }
    if (e == cudaSuccess && !c->graph_walker) e = cudaErrorInvalidValue;
    c->graph = graph;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&c->graph_exec, graph, 0);
    if (e != cudaSuccess) {
        c->graph_exec = nullptr;
        drop_graph(c);
        return fail(c, MUCAL_ERR_CUDA, "iteration graph capture failed: %s", cudaGetErrorString(e));
    }
    c->graph_sweeps = sweeps;
    c->graph_shape = c->shape;
    c->graph_tunnel = c->tunnel;
    c->graph_grid = grid;
    return MUCAL_OK;
}

int check_droplet_error(Context *c)
{
    int flag = 0;
    CUDA_TRY(c, cudaMemcpyAsync(&flag, c->d_drop_err, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    if (flag == 1) return fail(c, MUCAL_ERR_CUDA, "droplet labelling exceeded its iteration limit");
    if (flag == 2) return fail(c, MUCAL_ERR_CUDA, "droplet measurement met an energy outside the window");
    return MUCAL_OK;
}

}  // namespace

namespace mucal {
void set_init_error(const char *msg) { g_init_error = msg; }
}  // namespace mucal

extern "C" {

const char *mucal_version(void) { return "mucal 0.1 (sm_103a)"; }

const char *mucal_last_error(void *ctx)
{
    Context *c = as_ctx(ctx);
    return c ? c->err.c_str() : g_init_error.c_str();
}

int mucal_init_systems(void **out, const mucal_system_desc *sys, int32_t n_sys, void *cuda_stream,
                       uint32_t flags)
{
    if (!out) return fail(nullptr, MUCAL_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (!sys || n_sys <= 0) return fail(nullptr, MUCAL_ERR_INVALID_ARG, "need at least one system");
    for (int i = 0; i < n_sys; ++i) {
        int rc = check_desc(sys[i], i);
        if (rc != MUCAL_OK) return rc;
    }
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev <= 0) {
        cudaGetLastError();
        return fail(nullptr, MUCAL_ERR_NO_DEVICE, "no CUDA device available");
    }
    Context *c = new (std::nothrow) Context();
    if (!c) return fail(nullptr, MUCAL_ERR_OOM, "host allocation failed");
    c->flags = flags;
    int rc = MUCAL_OK;
    auto bail = [&](int code) {
        if (c->err.size()) g_init_error = c->err;
        cudaGetLastError();
        destroy_context(c);
        return code;
    };
    if (cudaGetDevice(&c->device) != cudaSuccess) {
        c->device = -1;
        return bail(fail(nullptr, MUCAL_ERR_NO_DEVICE, "cudaGetDevice failed"));
    }
    if (cuda_stream) {
        c->stream = static_cast<cudaStream_t>(cuda_stream);
    } else {
        if (cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking) != cudaSuccess)
            return bail(fail(nullptr, MUCAL_ERR_CUDA, "stream creation failed"));
        c->own_stream = true;
    }
    if (mucal::walker_update_max_smem(&c->max_smem) != cudaSuccess)
        return bail(fail(nullptr, MUCAL_ERR_CUDA, "cannot query shared memory limit"));
    if (cudaEventCreate(&c->ev_it0) != cudaSuccess || cudaEventCreate(&c->ev_k0) != cudaSuccess ||
        cudaEventCreate(&c->ev_k1) != cudaSuccess || cudaEventCreate(&c->ev_it1) != cudaSuccess)
        return bail(fail(nullptr, MUCAL_ERR_CUDA, "event creation failed"));

    c->sys.resize(n_sys);
    for (int i = 0; i < n_sys; ++i) {
        System &s = c->sys[i];
        s.desc = sys[i];
        SysParams &p = s.p;
        p.d = sys[i].d;
        p.L = sys[i].L;
        p.N = sys[i].N;
        p.V = p.d == 2 ? p.L * p.L : p.L * p.L * p.L;
        p.L2 = p.L * p.L;
        if (sys[i].e_lo == 0 && sys[i].e_hi == 0) {
            p.e_lo = -p.d * p.N;
            s.desc.e_lo = p.e_lo;
            s.desc.e_hi = 0;
        } else {
            p.e_lo = sys[i].e_lo;
        }
        p.n_bins = s.desc.e_hi - p.e_lo + 1;
        p.width = 4 * p.d + 1;
        p.tstride = (p.width + 3) & ~3;
        p.words = (p.V + 31) / 32;
        p.idx16 = p.V <= 65536 ? 1 : 0;
        p.n_walkers = sys[i].n_walkers;
        p.hist_rows = p.n_walkers;
        p.magL = (uint32_t)(((1ull << 32) + (uint64_t)p.L - 1) / (uint64_t)p.L);
        p.seed_base = sys[i].seed_base;
        const size_t nw = (size_t)p.n_walkers;
        const size_t ib = p.idx16 ? 2 : 4;
        void *ptr = nullptr;
#define ALLOC(field, bytes)                                                         \
    do {                                                                            \
        cudaError_t e_ = cudaMalloc(&ptr, (bytes));                                 \
        if (e_ != cudaSuccess) {                                                    \
            cudaGetLastError();                                                     \
            return bail(fail(nullptr, MUCAL_ERR_OOM, "cudaMalloc of %zu bytes for " \
                             #field " failed", (size_t)(bytes)));                   \
        }                                                                           \
        p.field = decltype(p.field)(ptr);                                           \
    } while (0)
        ALLOC(bits, nw * p.words * sizeof(uint32_t));
        ALLOC(S, nw * (size_t)p.V * ib);
        ALLOC(E, nw * sizeof(int32_t));
        ALLOC(thr, (size_t)p.n_bins * p.tstride * sizeof(uint32_t));
        ALLOC(accepts, nw * sizeof(unsigned long long));
        ALLOC(tun_state, nw * sizeof(uint8_t));
        ALLOC(tun_count, nw * sizeof(uint32_t));
#undef ALLOC
        p.tun_lo = 0;                    // tunnelling ends: the window's ends
        p.tun_hi = p.n_bins - 1;
        s.thr_count = (size_t)p.n_bins * p.tstride;
        if (cudaMallocHost(&s.thr_pinned, s.thr_count * sizeof(uint32_t)) != cudaSuccess) {
            s.thr_pinned = nullptr;
            return bail(fail(nullptr, MUCAL_ERR_OOM, "pinned host allocation failed"));
        }
        s.lnW.assign(p.n_bins, 0.0);
        s.visited.assign(p.n_bins, 0);
        s.pacc.assign(p.n_bins, 0.0);
        s.H.assign(p.n_bins, 0);
        s.lnW_run.assign(p.n_bins, 0.0);
        if (cudaMalloc(&ptr, 3 * (size_t)p.n_bins * 8) != cudaSuccess) {
            cudaGetLastError();
            return bail(fail(nullptr, MUCAL_ERR_OOM, "cudaMalloc of droplet accumulators failed"));
        }
        s.drop_acc = static_cast<unsigned long long *>(ptr);
        if (cudaMalloc(&ptr, nw * sizeof(int32_t)) != cudaSuccess) {
            cudaGetLastError();
            return bail(fail(nullptr, MUCAL_ERR_OOM, "cudaMalloc of droplet sizes failed"));
        }
        s.drop_last = static_cast<int32_t *>(ptr);
        if (cudaMemsetAsync(s.drop_acc, 0, 3 * (size_t)p.n_bins * 8, c->stream) != cudaSuccess ||
            cudaMemsetAsync(s.drop_last, 0, nw * sizeof(int32_t), c->stream) != cudaSuccess)
            return bail(fail(nullptr, MUCAL_ERR_CUDA, "memset failed"));
        if (cudaMemsetAsync(p.bits, 0, nw * p.words * sizeof(uint32_t), c->stream) != cudaSuccess ||
            cudaMemsetAsync(p.accepts, 0, nw * 8, c->stream) != cudaSuccess ||
            cudaMemsetAsync(p.tun_state, 0, nw, c->stream) != cudaSuccess ||
            cudaMemsetAsync(p.tun_count, 0, nw * 4, c->stream) != cudaSuccess)
            return bail(fail(nullptr, MUCAL_ERR_CUDA, "memset failed"));
    }
    size_t lists = 0;
    for (auto &s : c->sys) lists += (size_t)s.p.n_walkers * (size_t)s.p.V * (s.p.idx16 ? 2 : 4);
    for (auto &s : c->sys) s.p.prefetch = lists > kListsInL2 ? 1 : 0;
    if (cudaMalloc(&c->d_next_item, sizeof(int)) != cudaSuccess)
        return bail(fail(nullptr, MUCAL_ERR_OOM, "cudaMalloc of the work-item counter failed"));
    for (auto &s : c->sys) {
        s.h_off = c->h_words;
        c->h_words += (size_t)s.p.n_bins;
    }
    if (cudaMalloc(&c->d_H, (c->h_words + 1) * 8) != cudaSuccess ||
        cudaMallocHost(&c->h_H, (c->h_words + 1) * 8) != cudaSuccess ||
        cudaMemsetAsync(c->d_H, 0, (c->h_words + 1) * 8, c->stream) != cudaSuccess)
        return bail(fail(nullptr, MUCAL_ERR_OOM, "allocation of the summed histograms failed"));
    c->d_walk_err = reinterpret_cast<unsigned int *>(c->d_H + c->h_words);
    for (auto &s : c->sys) {
        s.p.H = c->d_H + s.h_off;
        s.p.err = c->d_walk_err;
    }
    if (cudaMalloc(&c->d_drop_err, sizeof(int)) != cudaSuccess ||
        cudaMemsetAsync(c->d_drop_err, 0, sizeof(int), c->stream) != cudaSuccess)
        return bail(fail(nullptr, MUCAL_ERR_OOM, "cudaMalloc of the droplet error flag failed"));
    if (cudaMalloc(&c->d_sys, n_sys * sizeof(SysParams)) != cudaSuccess)
        return bail(fail(nullptr, MUCAL_ERR_OOM, "cudaMalloc of system table failed"));
    std::vector<SysParams> hp(n_sys);
    for (int i = 0; i < n_sys; ++i) hp[i] = c->sys[i].p;
    if (cudaMemcpy(c->d_sys, hp.data(), n_sys * sizeof(SysParams), cudaMemcpyHostToDevice) != cudaSuccess)
        return bail(fail(nullptr, MUCAL_ERR_CUDA, "copy of system table failed"));
    if (mucal::launch_init_walkers(hp.data(), n_sys, c->stream) != cudaSuccess)
        return bail(fail(nullptr, MUCAL_ERR_CUDA, "initial placement launch failed"));
    for (int i = 0; i < n_sys; ++i) {
        rc = upload_thresholds(c, c->sys[i]);
        if (rc != MUCAL_OK) return bail(rc);
    }
    if (cudaStreamSynchronize(c->stream) != cudaSuccess)
        return bail(fail(nullptr, MUCAL_ERR_CUDA, "initial placement failed: %s",
                         cudaGetErrorString(cudaGetLastError())));
    // user-given windows must contain every initial energy
    for (int i = 0; i < n_sys; ++i) {
        const System &s = c->sys[i];
        if (sys[i].e_lo == 0 && sys[i].e_hi == 0) continue;
        std::vector<int32_t> e(s.p.n_walkers);
        if (cudaMemcpy(e.data(), s.p.E, e.size() * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
            return bail(fail(nullptr, MUCAL_ERR_CUDA, "energy read-back failed"));
        for (int32_t v : e)
            if (v < s.desc.e_lo || v > s.desc.e_hi)
                return bail(fail(nullptr, MUCAL_ERR_INVALID_ARG,
                                 "system %d: initial energy %d outside window [%d, %d]", i, v,
                                 s.desc.e_lo, s.desc.e_hi));
    }
    const mucal_launch_config def = default_launch(c);
    rc = apply_launch_config(c, def);
    if (rc != MUCAL_OK) return bail(rc);
    *out = c;
    return MUCAL_OK;
}

void mucal_destroy(void *ctx) { destroy_context(as_ctx(ctx)); }

int mucal_set_weights(void *ctx, int32_t sys, const double *lnW, int32_t n_bins)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    System &s = c->sys[sys];
    if (!lnW || n_bins != s.p.n_bins)
        return fail(c, MUCAL_ERR_INVALID_ARG, "lnW must hold n_bins = %d values", s.p.n_bins);
    for (int b = 0; b < n_bins; ++b)
        if (!std::isfinite(lnW[b])) return fail(c, MUCAL_ERR_INVALID_ARG, "lnW[%d] is not finite", b);
    s.lnW.assign(lnW, lnW + n_bins);
    std::fill(s.visited.begin(), s.visited.end(), 0);
    std::fill(s.pacc.begin(), s.pacc.end(), 0.0);
    CUDA_TRY(c, cudaSetDevice(c->device));
    return upload_thresholds(c, s);
}

int mucal_get_weights(void *ctx, int32_t sys, double *lnW_out, int32_t n_bins)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    const System &s = c->sys[sys];
    if (!lnW_out || n_bins != s.p.n_bins) return fail(c, MUCAL_ERR_INVALID_ARG, "bad lnW_out size");
    std::copy(s.lnW.begin(), s.lnW.end(), lnW_out);
    return MUCAL_OK;
}

int mucal_get_thresholds(void *ctx, int32_t sys, uint32_t *T, int64_t n)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    const System &s = c->sys[sys];
    if (!T || n != (int64_t)s.p.n_bins * s.p.width)
        return fail(c, MUCAL_ERR_INVALID_ARG, "bad threshold buffer size");
    CUDA_TRY(c, cudaSetDevice(c->device));
    // the device rows are padded to tstride words; the caller gets width per row
    CUDA_TRY(c, cudaMemcpy2DAsync(T, (size_t)s.p.width * 4, s.p.thr, (size_t)s.p.tstride * 4,
                                  (size_t)s.p.width * 4, (size_t)s.p.n_bins, cudaMemcpyDeviceToHost,
                                  c->stream));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    return MUCAL_OK;
}

int mucal_set_launch_config(void *ctx, const mucal_launch_config *cfg)
{
    Context *c = as_ctx(ctx);
    if (!c || !cfg) return MUCAL_ERR_INVALID_ARG;
    CUDA_TRY(c, cudaSetDevice(c->device));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    return apply_launch_config(c, *cfg);
}

int mucal_get_launch_config(void *ctx, mucal_launch_config *cfg)
{
    Context *c = as_ctx(ctx);
    if (!c || !cfg) return MUCAL_ERR_INVALID_ARG;
    cfg->kernel = c->shape.kernel;
    cfg->lanes_per_walker = c->shape.lanes;
    cfg->walkers_per_block = c->shape.walkers_per_block;
    cfg->bits_in_smem = c->shape.bits_in_smem;
    cfg->persistent = c->shape.persistent;
    // with the whole table in shared memory the window setting has no effect
    cfg->thr_window = c->shape.thr_in_smem ? 0 : c->shape.thr_window;
    cfg->multi_commit = c->shape.multi_commit;
    return MUCAL_OK;
}

int mucal_set_graph_mode(void *ctx, int32_t enable)
{
    Context *c = as_ctx(ctx);
    if (!c) return MUCAL_ERR_INVALID_ARG;
    CUDA_TRY(c, cudaSetDevice(c->device));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    c->graph_mode = enable != 0;
    drop_graph(c);
    return MUCAL_OK;
}

int mucal_run_iteration(void *ctx, int64_t sweeps, uint32_t iteration)
{
    Context *c = as_ctx(ctx);
    if (!c) return MUCAL_ERR_INVALID_ARG;
    if (sweeps < 1) return fail(c, MUCAL_ERR_INVALID_ARG, "sweeps must be >= 1");
    for (auto &s : c->sys)
        if ((uint64_t)sweeps * (uint64_t)s.p.N >= (1ull << 40))
            return fail(c, MUCAL_ERR_INVALID_ARG, "sweeps * N must be below 2^40");
    CUDA_TRY(c, cudaSetDevice(c->device));
    int grid = 0;
    CUDA_TRY(c, mucal::walker_update_grid(c->shape, c->tunnel, c->n_blocks, &grid));
    if (!c->graph_mode) {
        int rc = enqueue_iteration(c, (uint64_t)sweeps, iteration, grid, true);
        if (rc != MUCAL_OK) return rc;
    } else {
        const LaunchShape &a = c->shape, &b = c->graph_shape;
        const bool same = c->graph_exec && c->graph_sweeps == (uint64_t)sweeps &&
                          c->graph_tunnel == c->tunnel && c->graph_grid == grid &&
                          a.kernel == b.kernel && a.lanes == b.lanes &&
                          a.walkers_per_block == b.walkers_per_block &&
                          a.bits_in_smem == b.bits_in_smem && a.thr_in_smem == b.thr_in_smem &&
                          a.smem_bytes == b.smem_bytes && a.persistent == b.persistent &&
                          a.thr_window == b.thr_window && a.multi_commit == b.multi_commit &&
                          a.scan_window == b.scan_window;
        if (!same) {
            int rc = capture_iteration(c, (uint64_t)sweeps, iteration, grid);
            if (rc != MUCAL_OK) return rc;
        }
        // only the iteration number (the Philox counter word) changes
        uint64_t sw = (uint64_t)sweeps;
        int n_items = c->n_blocks;
        int *counter = c->shape.persistent ? c->d_next_item : nullptr;
        const SysParams *dsys = c->d_sys;
        const BlockWork *dwork = c->d_work;
        void *args[] = {(void *)&dsys, (void *)&dwork, (void *)&sw, (void *)&iteration,
                        (void *)&n_items, (void *)&counter};
        cudaKernelNodeParams kp = c->graph_kp;
        kp.kernelParams = args;
        kp.extra = nullptr;
        CUDA_TRY(c, cudaGraphExecKernelNodeSetParams(c->graph_exec, c->graph_walker, &kp));
        // the whole graph is timed: kernel_ms then includes the clears and sums
        CUDA_TRY(c, cudaEventRecord(c->ev_it0, c->stream));
        CUDA_TRY(c, cudaEventRecord(c->ev_k0, c->stream));
        CUDA_TRY(c, cudaGraphLaunch(c->graph_exec, c->stream));
        CUDA_TRY(c, cudaEventRecord(c->ev_k1, c->stream));
        CUDA_TRY(c, cudaEventRecord(c->ev_it1, c->stream));
    }
    for (auto &s : c->sys) {
        s.hist_on_host = s.hist_ahead = false;
        s.last_attempts = (uint64_t)sweeps * (uint64_t)s.p.N * (uint64_t)s.p.n_walkers;
        s.lnW_run = s.lnW;
    }
    c->ran = true;
    c->sweeps_last = (uint64_t)sweeps;
    c->launches += 1;
    return MUCAL_OK;
}

int mucal_get_histogram(void *ctx, int32_t sys, int64_t *H, int32_t n_bins, int64_t *per_walker)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    System &s = c->sys[sys];
    if (!H || n_bins != s.p.n_bins) return fail(c, MUCAL_ERR_INVALID_ARG, "H must hold n_bins = %d", s.p.n_bins);
    if (per_walker && !(c->flags & MUCAL_FLAG_PER_WALKER_HIST))
        return fail(c, MUCAL_ERR_INVALID_ARG, "per-walker histograms need MUCAL_FLAG_PER_WALKER_HIST");
    CUDA_TRY(c, cudaSetDevice(c->device));
    rc = fetch_histogram(c, s);
    if (rc != MUCAL_OK) return rc;
    std::copy(s.H.begin(), s.H.end(), H);
    if (per_walker) {
        CUDA_TRY(c, cudaMemcpyAsync(per_walker, s.p.hist,
                                    (size_t)s.p.n_walkers * (size_t)s.p.n_bins * 8,
                                    cudaMemcpyDeviceToHost, c->stream));
        CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    }
    return MUCAL_OK;
}

int mucal_update_weights(void *ctx, int32_t sys, int32_t scheme, double *lnW_out, double *flatness_out)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    if (!scheme_ok(scheme)) return fail(c, MUCAL_ERR_INVALID_ARG, "unknown scheme %d", scheme);
    System &s = c->sys[sys];
    CUDA_TRY(c, cudaSetDevice(c->device));
    rc = fetch_histogram(c, s);
    if (rc != MUCAL_OK) return rc;
    update_step(scheme, s.p.n_bins, s.H.data(), s.lnW.data(), s.visited.data(), s.pacc.data());
    const double f = flatness(s);
    rc = upload_thresholds(c, s);
    if (rc != MUCAL_OK) return rc;
    if (lnW_out) std::copy(s.lnW.begin(), s.lnW.end(), lnW_out);
    if (flatness_out) *flatness_out = f;
    return MUCAL_OK;
}

int mucal_set_histogram(void *ctx, int32_t sys, const int64_t *H, int32_t n_bins)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    System &s = c->sys[sys];
    if (!H || n_bins != s.p.n_bins) return fail(c, MUCAL_ERR_INVALID_ARG, "H must hold n_bins = %d", s.p.n_bins);
    if (!c->ran) return fail(c, MUCAL_ERR_NOT_READY, "no iteration has been run");
    for (int b = 0; b < n_bins; ++b)
        if (H[b] < 0) return fail(c, MUCAL_ERR_INVALID_ARG, "H[%d] is negative", b);
    // the local histogram must not land on top of the given one later
    CUDA_TRY(c, cudaSetDevice(c->device));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    std::copy(H, H + n_bins, s.H.begin());
    s.hist_on_host = true;
    s.hist_ahead = false;
    return MUCAL_OK;
}

int mucal_get_launch_occupancy(void *ctx, int32_t *blocks_per_sm, int32_t *sm_count)
{
    Context *c = as_ctx(ctx);
    if (!c || !blocks_per_sm || !sm_count) return MUCAL_ERR_INVALID_ARG;
    CUDA_TRY(c, cudaSetDevice(c->device));
    const void *fn = mucal::walker_update_fn(c->shape, c->tunnel);
    if (!fn) return fail(c, MUCAL_ERR_INVALID_ARG, "no kernel for the current launch shape");
    int per_sm = 0, sms = 0;
    CUDA_TRY(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                    &per_sm, fn, c->shape.walkers_per_block * c->shape.lanes, c->shape.smem_bytes));
    CUDA_TRY(c, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device));
    *blocks_per_sm = per_sm;
    *sm_count = sms;
    return MUCAL_OK;
}

int mucal_weight_update(int32_t scheme, int32_t n_bins, const int64_t *H, double *lnW,
                        uint8_t *visited, double *pacc, int32_t t_lo, int32_t t_hi,
                        double *flatness_out)
{
    if (!scheme_ok(scheme)) return fail(nullptr, MUCAL_ERR_INVALID_ARG, "unknown scheme %d", scheme);
    if (n_bins < 1 || !H || !lnW || !visited || ((scheme & 0xF) == MUCAL_SCHEME_RECURSIVE && !pacc))
        return fail(nullptr, MUCAL_ERR_INVALID_ARG, "need n_bins >= 1 and H, lnW, visited (and pacc)");
    if (t_lo >= 0 && (t_hi < t_lo || t_hi >= n_bins))
        return fail(nullptr, MUCAL_ERR_INVALID_ARG, "target bins must satisfy 0 <= t_lo <= t_hi < n_bins");
    for (int b = 0; b < n_bins; ++b) {
        if (H[b] < 0) return fail(nullptr, MUCAL_ERR_INVALID_ARG, "H[%d] is negative", b);
        if (!std::isfinite(lnW[b])) return fail(nullptr, MUCAL_ERR_INVALID_ARG, "lnW[%d] is not finite", b);
    }
    update_step(scheme, n_bins, H, lnW, visited, pacc);
    if (flatness_out) *flatness_out = flatness_of(n_bins, H, visited, t_lo < 0 ? -1 : t_lo, t_hi);
    return MUCAL_OK;
}

int mucal_set_target_window(void *ctx, int32_t sys, int32_t t_lo, int32_t t_hi)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    System &s = c->sys[sys];
    if (t_lo == 0 && t_hi == 0) {
        s.target_default = true;
        return MUCAL_OK;
    }
    if (t_lo < s.desc.e_lo || t_hi > s.desc.e_hi || t_lo > t_hi)
        return fail(c, MUCAL_ERR_INVALID_ARG, "target window must lie inside [%d, %d]", s.desc.e_lo,
                    s.desc.e_hi);
    s.target_default = false;
    s.t_lo = t_lo - s.desc.e_lo;
    s.t_hi = t_hi - s.desc.e_lo;
    return MUCAL_OK;
}

int mucal_get_walker_state(void *ctx, int32_t sys, int32_t walker, uint8_t *occ, int32_t *S, int32_t *E)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    const System &s = c->sys[sys];
    const SysParams &p = s.p;
    if (walker < 0 || walker >= p.n_walkers) return fail(c, MUCAL_ERR_INVALID_ARG, "walker out of range");
    CUDA_TRY(c, cudaSetDevice(c->device));
    std::vector<uint32_t> bits(p.words);
    std::vector<uint8_t> sraw((size_t)p.V * (p.idx16 ? 2 : 4));
    int32_t e = 0;
    CUDA_TRY(c, cudaMemcpyAsync(bits.data(), p.bits + (size_t)walker * p.words, p.words * 4,
                                cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(c, cudaMemcpyAsync(sraw.data(), (const char *)p.S + (size_t)walker * sraw.size(),
                                sraw.size(), cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(c, cudaMemcpyAsync(&e, p.E + walker, 4, cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    if (occ)
        for (int i = 0; i < p.V; ++i) occ[i] = (uint8_t)((bits[i >> 5] >> (i & 31)) & 1u);
    if (S) {
        for (int i = 0; i < p.V; ++i) {
            if (p.idx16)
                S[i] = ((const uint16_t *)sraw.data())[i];
            else
                S[i] = (int32_t)((const uint32_t *)sraw.data())[i];
        }
    }
    if (E) *E = e;
    return MUCAL_OK;
}

int mucal_get_system_info(void *ctx, int32_t sys, mucal_system_info *info)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    if (!info) return fail(c, MUCAL_ERR_INVALID_ARG, "info is NULL");
    const System &s = c->sys[sys];
    info->d = s.p.d;
    info->L = s.p.L;
    info->N = s.p.N;
    info->n_walkers = s.p.n_walkers;
    info->e_lo = s.desc.e_lo;
    info->e_hi = s.desc.e_hi;
    info->V = s.p.V;
    info->n_bins = s.p.n_bins;
    info->width = s.p.width;
    info->index_bytes = s.p.idx16 ? 2 : 4;
    info->seed_base = s.p.seed_base;
    return MUCAL_OK;
}

int mucal_get_stats(void *ctx, int32_t sys, mucal_stats *st)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    if (!st) return fail(c, MUCAL_ERR_INVALID_ARG, "stats is NULL");
    std::memset(st, 0, sizeof *st);
    st->walker_launches = c->launches;
    if (!c->ran) return MUCAL_OK;
    const System &s = c->sys[sys];
    CUDA_TRY(c, cudaSetDevice(c->device));
    std::vector<unsigned long long> acc(s.p.n_walkers);
    CUDA_TRY(c, cudaMemcpyAsync(acc.data(), s.p.accepts, acc.size() * 8, cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    for (auto v : acc) st->accepts += v;
    st->attempts = s.last_attempts;
    float ms = 0.f;
    CUDA_TRY(c, cudaEventElapsedTime(&ms, c->ev_k0, c->ev_k1));
    st->kernel_ms = ms;
    CUDA_TRY(c, cudaEventElapsedTime(&ms, c->ev_it0, c->ev_it1));
    st->iteration_ms = ms;
    return MUCAL_OK;
}

int mucal_histogram_device_ptr(void *ctx, int32_t sys, void **dptr)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    if (!dptr) return fail(c, MUCAL_ERR_INVALID_ARG, "dptr is NULL");
    System &s = c->sys[sys];
    s.hist_shared = true;
    if (s.hist_ahead) s.hist_on_host = s.hist_ahead = false;
    *dptr = s.p.H;
    return MUCAL_OK;
}

int mucal_reweight_system(void *ctx, int32_t sys, const double *beta, int32_t n_beta,
                          const double *obs, int32_t n_obs, double *mean_E, double *mean_E2,
                          double *obs_out)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    System &s = c->sys[sys];
    CUDA_TRY(c, cudaSetDevice(c->device));
    rc = fetch_histogram(c, s);
    if (rc != MUCAL_OK) return rc;
    rc = mucal_reweight(s.H.data(), s.lnW_run.data(), s.p.n_bins, s.p.e_lo, beta, n_beta, obs, n_obs,
                        mean_E, mean_E2, obs_out);
    if (rc != MUCAL_OK) c->err = mucal_last_error(nullptr);
    return rc;
}

int mucal_set_tunnel_window(void *ctx, int32_t sys, int32_t e_min, int32_t e_max)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    System &s = c->sys[sys];
    if (e_min == 0 && e_max == 0) {
        e_min = s.desc.e_lo;
        e_max = s.desc.e_hi;
    }
    if (e_min < s.desc.e_lo || e_max > s.desc.e_hi || e_min >= e_max)
        return fail(c, MUCAL_ERR_INVALID_ARG, "tunnelling ends must satisfy %d <= e_min < e_max <= %d",
                    s.desc.e_lo, s.desc.e_hi);
    CUDA_TRY(c, cudaSetDevice(c->device));
    s.p.tun_lo = e_min - s.desc.e_lo;
    s.p.tun_hi = e_max - s.desc.e_lo;
    for (auto &q : c->sys) q.p.tunnel = 1;
    rc = upload_sys_table(c);
    if (rc != MUCAL_OK) return rc;
    c->tunnel = true;
    return reset_tunnel(c, s);
}

int mucal_get_tunnel_counts(void *ctx, int32_t sys, int64_t *total, uint32_t *per_walker,
                            uint8_t *state)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    const System &s = c->sys[sys];
    CUDA_TRY(c, cudaSetDevice(c->device));
    std::vector<uint32_t> cnt((size_t)s.p.n_walkers);
    CUDA_TRY(c, cudaMemcpyAsync(cnt.data(), s.p.tun_count, cnt.size() * 4, cudaMemcpyDeviceToHost,
                                c->stream));
    if (state)
        CUDA_TRY(c, cudaMemcpyAsync(state, s.p.tun_state, cnt.size(), cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    int64_t sum = 0;
    for (uint32_t v : cnt) sum += v;
    if (total) *total = sum;
    if (per_walker) std::copy(cnt.begin(), cnt.end(), per_walker);
    return MUCAL_OK;
}

int mucal_reset_tunnel_counts(void *ctx)
{
    Context *c = as_ctx(ctx);
    if (!c) return MUCAL_ERR_INVALID_ARG;
    CUDA_TRY(c, cudaSetDevice(c->device));
    for (const System &s : c->sys) {
        const int rc = reset_tunnel(c, s);
        if (rc != MUCAL_OK) return rc;
    }
    return MUCAL_OK;
}

int mucal_replica_exchange(void *ctx, const double *beta, int32_t n_sys, uint32_t round,
                           int32_t parity, int64_t *accepted)
{
    Context *c = as_ctx(ctx);
    if (!c) return MUCAL_ERR_INVALID_ARG;
    if (!beta) return fail(c, MUCAL_ERR_INVALID_ARG, "beta is NULL");
    if (n_sys != (int32_t)c->sys.size() || n_sys < 2)
        return fail(c, MUCAL_ERR_INVALID_ARG, "n_sys must equal the context's %d systems (>= 2)",
                    (int)c->sys.size());
    if (parity != 0 && parity != 1) return fail(c, MUCAL_ERR_INVALID_ARG, "parity must be 0 or 1");
    const SysParams &p0 = c->sys[0].p;
    for (int k = 0; k < n_sys; ++k) {
        const SysParams &p = c->sys[k].p;
        if (p.d != p0.d || p.L != p0.L || p.N != p0.N || p.n_walkers != p0.n_walkers ||
            p.e_lo != p0.e_lo || p.n_bins != p0.n_bins)
            return fail(c, MUCAL_ERR_INVALID_ARG, "system %d differs from system 0: a tempering "
                        "ladder needs copies of one lattice, walker count and window", k);
        if (!std::isfinite(beta[k])) return fail(c, MUCAL_ERR_INVALID_ARG, "beta[%d] is not finite", k);
    }
    CUDA_TRY(c, cudaSetDevice(c->device));
    const int nb = p0.n_bins;
    const int width = 2 * nb - 1;
    const int pairs = n_sys - 1;
    const size_t words = (size_t)pairs * (size_t)width;
    if (words > c->xthr_words) {
        CUDA_TRY(c, cudaStreamSynchronize(c->stream));
        cudaFree(c->d_xthr);
        cudaFree(c->d_xacc);
        if (c->xthr_pinned) cudaFreeHost(c->xthr_pinned);
        if (c->xacc_pinned) cudaFreeHost(c->xacc_pinned);
        c->d_xthr = nullptr;
        c->d_xacc = nullptr;
        c->xthr_pinned = nullptr;
        c->xacc_pinned = nullptr;
        c->xthr_words = 0;
        CUDA_TRY(c, cudaMalloc(&c->d_xthr, words * sizeof(uint32_t)));
        CUDA_TRY(c, cudaMalloc(&c->d_xacc, (size_t)pairs * sizeof(unsigned long long)));
        CUDA_TRY(c, cudaMallocHost(&c->xthr_pinned, words * sizeof(uint32_t)));
        CUDA_TRY(c, cudaMallocHost(&c->xacc_pinned, (size_t)pairs * sizeof(unsigned long long)));
        c->xthr_words = words;
    }
    // the staging buffer may still feed the previous exchange's upload
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    for (int k = 0; k < pairs; ++k) {
        const double db = beta[k] - beta[k + 1];
        uint32_t *row = c->xthr_pinned + (size_t)k * width;
        for (int j = 0; j < width; ++j) {
            const double x = db * (double)(j - (nb - 1));   // (beta_k - beta_k+1)(E_k - E_k+1)
            if (x >= 0.0) {
                row[j] = 0xFFFFFFFFu;
                continue;
            }
            const double scaled = std::floor(std::ldexp(std::exp(x), 32));
            row[j] = scaled >= 4294967294.0 ? 0xFFFFFFFEu : (uint32_t)scaled;
        }
    }
    CUDA_TRY(c, cudaMemcpyAsync(c->d_xthr, c->xthr_pinned, words * sizeof(uint32_t),
                                cudaMemcpyHostToDevice, c->stream));
    CUDA_TRY(c, cudaMemsetAsync(c->d_xacc, 0, (size_t)pairs * sizeof(unsigned long long), c->stream));
    CUDA_TRY(c, mucal::launch_exchange(c->d_sys, n_sys, p0.n_walkers, parity, round, c->d_xthr, width,
                                       c->d_xacc, c->stream));
    if (accepted) {
        CUDA_TRY(c, cudaMemcpyAsync(c->xacc_pinned, c->d_xacc, (size_t)pairs * 8, cudaMemcpyDeviceToHost,
                                    c->stream));
        CUDA_TRY(c, cudaStreamSynchronize(c->stream));
        std::memcpy(accepted, c->xacc_pinned, (size_t)pairs * 8);
    }
    return MUCAL_OK;
}

int mucal_measure_droplets(void *ctx)
{
    Context *c = as_ctx(ctx);
    if (!c) return MUCAL_ERR_INVALID_ARG;
    CUDA_TRY(c, cudaSetDevice(c->device));
    size_t scratch = 0;
    for (auto &s : c->sys) {
        if (!s.drop_planned) CUDA_TRY(c, mucal::droplet_plan(s.p, &s.drop_plan));
        s.drop_planned = true;
        scratch = std::max(scratch, s.drop_plan.scratch_words);
    }
    if (scratch > c->drop_scratch_words) {
        // the previous scratch may still be read by an earlier measurement
        CUDA_TRY(c, cudaStreamSynchronize(c->stream));
        cudaFree(c->drop_scratch);
        c->drop_scratch = nullptr;
        c->drop_scratch_words = 0;
        CUDA_TRY(c, cudaMalloc(&c->drop_scratch, scratch * sizeof(uint32_t)));
        c->drop_scratch_words = scratch;
    }
    for (size_t i = 0; i < c->sys.size(); ++i) {
        const System &s = c->sys[i];
        const mucal::DropletOut o{s.drop_acc, s.drop_last, c->d_drop_err};
        CUDA_TRY(c, mucal::launch_droplets(s.p, o, s.drop_plan, c->drop_scratch, c->stream));
    }
    c->measured = true;
    return MUCAL_OK;
}

int mucal_get_droplet_stats(void *ctx, int32_t sys, int64_t *count, int64_t *sum, int64_t *sum2,
                            int32_t n_bins)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    const System &s = c->sys[sys];
    if (n_bins != s.p.n_bins) return fail(c, MUCAL_ERR_INVALID_ARG, "n_bins must be %d", s.p.n_bins);
    if (!c->measured) return fail(c, MUCAL_ERR_NOT_READY, "no droplet measurement yet");
    CUDA_TRY(c, cudaSetDevice(c->device));
    rc = check_droplet_error(c);
    if (rc != MUCAL_OK) return rc;
    int64_t *dst[3] = {count, sum, sum2};
    for (int k = 0; k < 3; ++k)
        if (dst[k])
            CUDA_TRY(c, cudaMemcpyAsync(dst[k], s.drop_acc + (size_t)k * s.p.n_bins,
                                        (size_t)s.p.n_bins * 8, cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    return MUCAL_OK;
}

int mucal_get_largest_droplets(void *ctx, int32_t sys, int32_t *V_D, int32_t n_walkers)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    const System &s = c->sys[sys];
    if (!V_D || n_walkers != s.p.n_walkers)
        return fail(c, MUCAL_ERR_INVALID_ARG, "V_D must hold n_walkers = %d", s.p.n_walkers);
    if (!c->measured) return fail(c, MUCAL_ERR_NOT_READY, "no droplet measurement yet");
    CUDA_TRY(c, cudaSetDevice(c->device));
    rc = check_droplet_error(c);
    if (rc != MUCAL_OK) return rc;
    CUDA_TRY(c, cudaMemcpyAsync(V_D, s.drop_last, (size_t)n_walkers * 4, cudaMemcpyDeviceToHost,
                                c->stream));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    return MUCAL_OK;
}

int mucal_reset_droplet_stats(void *ctx)
{
    Context *c = as_ctx(ctx);
    if (!c) return MUCAL_ERR_INVALID_ARG;
    CUDA_TRY(c, cudaSetDevice(c->device));
    for (const System &s : c->sys)
        CUDA_TRY(c, cudaMemsetAsync(s.drop_acc, 0, 3 * (size_t)s.p.n_bins * 8, c->stream));
    return MUCAL_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Checkpoint / resume.  Random numbers are counter-based (seed, iteration,
// attempt), so a restored system continues bit-for-bit.
// ---------------------------------------------------------------------------
namespace {

struct CheckpointHeader {
    char magic[8];          // "MUCALCK1"
    int32_t d, L, N, n_walkers, e_lo, e_hi;
    uint64_t seed_base;
    int32_t index_bytes, words, n_bins, target_default;
    int32_t t_lo, t_hi;
};

size_t checkpoint_bytes(const System &s)
{
    const SysParams &p = s.p;
    const size_t nw = (size_t)p.n_walkers;
    return sizeof(CheckpointHeader) + nw * p.words * 4 + nw * (size_t)p.V * (p.idx16 ? 2 : 4) +
           nw * 4 + (size_t)p.n_bins * (8 + 1 + 8);
}

}  // namespace

extern "C" {

int mucal_checkpoint_size(void *ctx, int32_t sys, int64_t *bytes)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    if (!bytes) return fail(c, MUCAL_ERR_INVALID_ARG, "bytes is NULL");
    *bytes = (int64_t)checkpoint_bytes(c->sys[sys]);
    return MUCAL_OK;
}

int mucal_checkpoint_save(void *ctx, int32_t sys, void *buf, int64_t bytes)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    const System &s = c->sys[sys];
    const SysParams &p = s.p;
    if (!buf || bytes != (int64_t)checkpoint_bytes(s))
        return fail(c, MUCAL_ERR_INVALID_ARG, "checkpoint buffer must hold %zu bytes", checkpoint_bytes(s));
    CUDA_TRY(c, cudaSetDevice(c->device));
    char *o = static_cast<char *>(buf);
    CheckpointHeader h{};
    std::memcpy(h.magic, "MUCALCK1", 8);
    h.d = p.d; h.L = p.L; h.N = p.N; h.n_walkers = p.n_walkers;
    h.e_lo = s.desc.e_lo; h.e_hi = s.desc.e_hi; h.seed_base = p.seed_base;
    h.index_bytes = p.idx16 ? 2 : 4; h.words = p.words; h.n_bins = p.n_bins;
    h.target_default = s.target_default ? 1 : 0; h.t_lo = s.t_lo; h.t_hi = s.t_hi;
    std::memcpy(o, &h, sizeof h);
    o += sizeof h;
    const size_t nw = (size_t)p.n_walkers;
    const size_t b_bits = nw * p.words * 4, b_S = nw * (size_t)p.V * (p.idx16 ? 2 : 4), b_E = nw * 4;
    CUDA_TRY(c, cudaMemcpyAsync(o, p.bits, b_bits, cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(c, cudaMemcpyAsync(o + b_bits, p.S, b_S, cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(c, cudaMemcpyAsync(o + b_bits + b_S, p.E, b_E, cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    o += b_bits + b_S + b_E;
    std::memcpy(o, s.lnW.data(), (size_t)p.n_bins * 8);
    o += (size_t)p.n_bins * 8;
    std::memcpy(o, s.visited.data(), (size_t)p.n_bins);
    o += p.n_bins;
    std::memcpy(o, s.pacc.data(), (size_t)p.n_bins * 8);
    return MUCAL_OK;
}

int mucal_checkpoint_load(void *ctx, int32_t sys, const void *buf, int64_t bytes)
{
    Context *c = as_ctx(ctx);
    int rc = check_sys(c, sys);
    if (rc != MUCAL_OK) return rc;
    System &s = c->sys[sys];
    const SysParams &p = s.p;
    if (!buf || bytes != (int64_t)checkpoint_bytes(s))
        return fail(c, MUCAL_ERR_INVALID_ARG, "checkpoint must hold %zu bytes", checkpoint_bytes(s));
    const char *in = static_cast<const char *>(buf);
    CheckpointHeader h;
    std::memcpy(&h, in, sizeof h);
    if (std::memcmp(h.magic, "MUCALCK1", 8) != 0 || h.d != p.d || h.L != p.L || h.N != p.N ||
        h.n_walkers != p.n_walkers || h.e_lo != s.desc.e_lo || h.e_hi != s.desc.e_hi ||
        h.seed_base != p.seed_base || h.index_bytes != (p.idx16 ? 2 : 4) || h.words != p.words ||
        h.n_bins != p.n_bins)
        return fail(c, MUCAL_ERR_INVALID_ARG, "checkpoint does not belong to system %d", sys);
    const size_t nw = (size_t)p.n_walkers;
    const size_t b_bits = nw * p.words * 4, b_S = nw * (size_t)p.V * (p.idx16 ? 2 : 4), b_E = nw * 4;
    const char *bits = in + sizeof h;
    const char *S = bits + b_bits;
    const char *E = S + b_S;
    const char *w = E + b_E;
    // validate before touching the device: energies inside the window, list
    // entries on the lattice, finite weights
    for (size_t i = 0; i < nw; ++i) {
        int32_t e;
        std::memcpy(&e, E + 4 * i, 4);
        if (e < s.desc.e_lo || e > s.desc.e_hi)
            return fail(c, MUCAL_ERR_INVALID_ARG, "checkpoint energy of walker %zu outside the window", i);
    }
    for (size_t i = 0; i < nw * (size_t)p.V; ++i) {
        uint32_t v;
        if (p.idx16) {
            uint16_t x;
            std::memcpy(&x, S + 2 * i, 2);
            v = x;
        } else {
            std::memcpy(&v, S + 4 * i, 4);
        }
        if (v >= (uint32_t)p.V) return fail(c, MUCAL_ERR_INVALID_ARG, "checkpoint list entry %zu is not a site", i);
    }
    std::vector<double> lnW((size_t)p.n_bins);
    std::memcpy(lnW.data(), w, (size_t)p.n_bins * 8);
    for (double x : lnW)
        if (!std::isfinite(x)) return fail(c, MUCAL_ERR_INVALID_ARG, "checkpoint weight is not finite");
    CUDA_TRY(c, cudaSetDevice(c->device));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    CUDA_TRY(c, cudaMemcpyAsync(p.bits, bits, b_bits, cudaMemcpyHostToDevice, c->stream));
    CUDA_TRY(c, cudaMemcpyAsync(p.S, S, b_S, cudaMemcpyHostToDevice, c->stream));
    CUDA_TRY(c, cudaMemcpyAsync(p.E, E, b_E, cudaMemcpyHostToDevice, c->stream));
    CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    s.lnW = lnW;
    std::memcpy(s.visited.data(), w + (size_t)p.n_bins * 8, (size_t)p.n_bins);
    std::memcpy(s.pacc.data(), w + (size_t)p.n_bins * 9, (size_t)p.n_bins * 8);
    s.target_default = h.target_default != 0;
    s.t_lo = h.t_lo;
    s.t_hi = h.t_hi;
    s.hist_on_host = false;
    rc = reset_tunnel(c, s);   // tunnelling is counted afresh after a restore
    if (rc != MUCAL_OK) return rc;
    return upload_thresholds(c, s);
}

}  // extern "C"
