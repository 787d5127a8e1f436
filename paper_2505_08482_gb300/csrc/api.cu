// C-ABI entry points of the forward operator and the adjoint gradient.
//
// Forward sweep (Sec. 2.1 scheme): init pass from p0, then Nt-1 steps of
// four passes; with a gradient workspace the state (u^{n-1/2}, rho^n) is
// copied every s steps and the pressure history of the last segment is kept.
// Reverse sweep (Sec. 3 adjoint-state gradient, exact for the discrete
// scheme): segments from last to first; each is recomputed from its
// checkpoint (segment 0 from p0) while storing p^n, then the adjoint steps
// run backwards through it, accumulating dJ/dc per data set; the n = 0
// transposes of the initial condition close the sweep.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <map>
#include <mutex>
#include <vector>

#include "pat_internal.h"
#include "vec.h"

using namespace pat;

// Mean gain of a forward and inverse transform pair of the generic passes minus 1, over the modes up to an eighth of the
// sampling rate: with the transforms' float constants in FP64, once per process and side (5 ms at Ng 400).  It is not
// that of the register transforms: Ng 180 2.0e-8, where those have -0.7e-8.
static double generic_gain(const FftDesc& fd) {
    static std::mutex mu;
    static std::map<int, double> known;
    std::lock_guard<std::mutex> lock(mu);
    const auto it = known.find(fd.n);
    if (it != known.end()) return it->second;
    const int n = fd.n, top = n / 8;
    std::vector<double2> e(n), a(n), b(n);
    std::vector<float2> tw(n);
    for (int q = 0; q < n; ++q) {
        const double w = -2.0 * 3.14159265358979323846 * q / n;
        e[q] = double2{std::cos(w), -std::sin(w)};
        tw[q] = make_float2(float(std::cos(w)), float(std::sin(w)));
    }
    double mean = 0.0;
    for (int k = -top; k <= top; ++k) {
        auto mode = [&](int q) { return e[size_t((k + n) % n) * q % n]; };
        for (int q = 0; q < n; ++q) a[q] = mode(q);
        double2* x = fft_host<false>(a.data(), b.data(), fd, tw.data());
        x = fft_host<true>(x, x == a.data() ? b.data() : a.data(), fd, tw.data());
        double s = 0.0;
        for (int q = 0; q < n; ++q) s += mode(q).x * x[q].x + mode(q).y * x[q].y;
        mean += (s / (double(n) * n) - 1.0) / (2 * top + 1);
    }
    return known[n] = mean;
}

// (a gain of 0: the side has no compiled transforms, and its factors are not corrected)
static double gain_of(const pat_plan_s* p, bool generic) {
    if (!generic || p->gain == 0.0) return p->gain;
    try {
        return generic_gain(p->fft);
    } catch (...) {   // no host memory: no exception leaves a C entry point
        return 0.0;
    }
}
float pat::scale_g(const pat_plan_s* p, bool generic) {
    return float(p->g.dt / p->g.rho0 / (double(p->ng) * p->ng) * std::pow(1.0 + gain_of(p, generic), -2.0));
}
float pat::scale_d(const pat_plan_s* p, bool generic) {
    const double n2 = double(p->ng) * p->ng,
                 target = p->g.dt / n2 * (p->g.dt / n2) * std::pow(1.0 + gain_of(p, generic), -4.0);
    return float(target / double(scale_g(p, generic)));
}

namespace {

#define RC(x)                   \
    do {                        \
        int rc_ = (x);          \
        if (rc_ != PAT_OK) return rc_; \
    } while (0)

// one forward step n -> n+1 given the row spectrum of p^n in A
int step(const Launch& L, const Ws& w, int n, float* y, float* hist, int hist_slot) {
    const pat_plan_s* p = L.p;
    RC(launch_col(L, w.A, w.B, 0, 0, scale_g(p, !p->fast)));
    RC(launch_row_u(L, w, n == 0));
    RC(launch_col(L, w.A, w.B, 1, 1, scale_d(p, !p->fast)));
    RC(launch_row_rho(L, w, 0, nullptr, y, n + 1, hist, hist_slot));
    return PAT_OK;
}

// the split-axis passes of the plan where the workspace holds their larger state, else the four-pass step
const SplitOps* split_of(const pat_plan_s* p, const Ws& w) { return w.split_fits ? p->split : nullptr; }

size_t state_bytes(const pat_plan_s* p) { return 4 * size_t(p->K) * p->ng * p->ng * sizeof(float); }

// forward steps n0 .. n1-1; p^{n+1} into hist slot n+1-hbase when hist and n+1 >= hbase
int run_steps(const Launch& L, const Ws& w, int n0, int n1, float* y, float* hist, int hbase) {
    if (L.split) return split_steps(L, w, n0, n1, y, hist, hbase, nullptr);
    for (int n = n0; n < n1; ++n) {
        const bool h = hist && n + 1 >= hbase;
        RC(step(L, w, n, y, h ? hist : nullptr, n + 1 - hbase));
    }
    return PAT_OK;
}

}  // namespace

int pat::forward_sweep(pat_plan_s* p, const float* c, const float* p0, float* y, const Ws& w, bool keep,
                       cudaStream_t st) {
    NvtxRange nv("pat forward sweep");
    Launch L{p, st, true, false, split_of(p, w)};
    RC(launch_medium(L, c, w.cg));
    PAT_CUDA(cudaMemsetAsync(y, 0, size_t(p->K) * p->nt * p->m * sizeof(float), st));
    PAT_CUDA(cudaMemsetAsync(w.flag + 1, 0, sizeof(int), st));   // bounded-wait status of this call
    const int last0 = (p->nseg - 1) * p->s_eff;
    float* hlast = keep ? hist_of(p, w, p->nseg - 1) : nullptr;
    if (p->persistent && p->sweep)   // one launch: initial pass, every step, checkpoints, history
        return launch_forward_persistent(L, w, p0, y, hlast, last0, keep ? w.ckpt : nullptr);
    if (p->cluster && p->clops)      // one cluster per data set for the whole sweep, state on chip
        return launch_forward_cluster(L, w, p0, nullptr, 0, p->nt - 1, y, hlast, last0, keep ? w.ckpt : nullptr,
                                      w.ux);
    if (L.split) {                   // three launches per step (ksplit.cuh)
        RC(split_start(L, w, p0, y, (keep && last0 == 0) ? hlast : nullptr, 0));
        return split_steps(L, w, 0, p->nt - 1, y, hlast, last0, keep ? w.ckpt : nullptr);
    }
    RC(launch_row_rho(L, w, 1, p0, y, 0, (keep && last0 == 0) ? hlast : nullptr, 0));
    // segments of s steps with the state copied at their starts (one segment without checkpoints)
    const int seg = keep ? p->s_eff : p->nt;
    for (int n0 = 0; n0 + 1 < p->nt;) {
        if (keep && n0 > 0) {
            PAT_CUDA(cudaMemcpyAsync(w.ckpt + size_t(n0 / p->s_eff - 1) * 4 * p->K * p->ng * p->ng, w.ux,
                                     state_bytes(p), cudaMemcpyDeviceToDevice, st));
        }
        const int n1 = std::min(p->nt - 1, (n0 / seg + 1) * seg);
        RC(run_steps(L, w, n0, n1, y, hlast, last0));
        n0 = n1;
    }
    // a last segment that starts at level Nt-1 is restored from a checkpoint of that level
    if (keep && p->nt > 1 && (p->nt - 1) % p->s_eff == 0) {
        PAT_CUDA(cudaMemcpyAsync(w.ckpt + size_t((p->nt - 1) / p->s_eff - 1) * 4 * p->K * p->ng * p->ng, w.ux,
                                 state_bytes(p), cudaMemcpyDeviceToDevice, st));
    }
    return PAT_OK;
}

namespace {

// recompute segment j's pressure history into its buffer (on stream st)
int recompute(pat_plan_s* p, const float* p0, const Ws& w, int j, cudaStream_t st) {
    Launch L{p, st, false, true, split_of(p, w)};
    const size_t f = size_t(p->K) * p->ng * p->ng;
    const int n0 = j * p->s_eff;
    const int n1 = std::min(n0 + p->s_eff, p->nt) - 1;
    float* h = hist_of(p, w, j);
    if (p->cluster && p->clops)   // from the checkpoint (or p0) on chip, storing p^n of the segment
        return launch_forward_cluster(L, w, p0, j == 0 ? nullptr : w.ckpt + size_t(j - 1) * 4 * f, n0, n1, nullptr,
                                      h, n0, nullptr, nullptr);
    if (L.split) {
        RC(j == 0 ? split_start(L, w, p0, nullptr, h, 0)
                  : split_enter(L, w, w.ckpt + size_t(j - 1) * 4 * f, n0, nullptr, h, 0));
        return split_steps(L, w, n0, n1, nullptr, h, n0, nullptr);
    }
    if (j == 0) {
        RC(launch_row_rho(L, w, 1, p0, nullptr, 0, h, 0));
    } else {
        PAT_CUDA(cudaMemcpyAsync(w.ux, w.ckpt + size_t(j - 1) * 4 * f, state_bytes(p), cudaMemcpyDeviceToDevice,
                                 st));
        RC(launch_row_rho(L, w, 2, nullptr, nullptr, 0, h, 0));
    }
    return run_steps(L, w, n0, n1, nullptr, h, n0);
}

// adjoint steps n_hi down to n_lo (first: n_hi is the first adjoint step of the sweep)
int run_adj(const Launch& L, const Ws& w, const float* r, int n_hi, int n_lo, bool first, const float* h, int hbase,
            float sg, float sd) {
    if (L.split) return split_adjoint(L, w, r, n_hi, n_lo, first, h, hbase);
    for (int n = n_hi; n >= n_lo; --n) {
        RC(launch_row_adj_rho(L, w, (first && n == n_hi) ? 1 : 0, r, n, h, n - hbase, n == n_hi));
        RC(launch_col(L, w.A2, w.B2, 1, 0, sg));
        RC(launch_row_adj_u(L, w));
        RC(launch_col(L, w.A2, w.B2, 2, 1, sd));
    }
    return PAT_OK;
}

// reverse sweep with the weighted residual (or adjoint source) r [K][nt][m].
// The recompute of segment j-1 runs on the plan's second stream while the adjoint
// steps of segment j run on st; the two pressure-history buffers alternate.
int reverse_sweep(pat_plan_s* p, const float* p0, const float* r, float* grad_p0, float* grad_c, const Ws& w,
                  bool hist_last_valid, cudaStream_t st) {
    NvtxRange nv("pat reverse sweep");
    Launch L{p, st, false, false, split_of(p, w)};
    const size_t f = size_t(p->K) * p->ng * p->ng;
    if (L.split) {
        const size_t lines = 2 * size_t(p->K) * p->hc * p->ng * sizeof(float2);
        PAT_CUDA(cudaMemsetAsync(w.lub, 0, lines, st));
        PAT_CUDA(cudaMemsetAsync(w.lrb, 0, lines, st));
    } else {
        PAT_CUDA(cudaMemsetAsync(w.ubx, 0, 4 * f * sizeof(float), st));
    }
    PAT_CUDA(cudaMemsetAsync(w.cbar, 0, size_t(p->K) * p->n * p->n * sizeof(float), st));
    const float sg = scale_d(p, !p->fast), sd = scale_g(p, !p->fast);   // dt rho0 G t, dt/rho0 D t'
    cudaStream_t R = p->side;
    const int last = p->nseg - 1;
    // the side stream starts after everything issued so far on st (forward sweep, residual)
    PAT_CUDA(cudaEventRecord(p->ev_start, st));
    PAT_CUDA(cudaStreamWaitEvent(R, p->ev_start, 0));
    if (!hist_last_valid) {
        RC(recompute(p, p0, w, last, R));
        PAT_CUDA(cudaEventRecord(p->ev_rec[last & 1], R));
    }
    if (last >= 1) {
        RC(recompute(p, p0, w, last - 1, R));
        PAT_CUDA(cudaEventRecord(p->ev_rec[(last - 1) & 1], R));
    }
    bool have_q = false;
    for (int j = last; j >= 0; --j) {
        const int n0 = j * p->s_eff;
        const int n1 = std::min(n0 + p->s_eff, p->nt) - 1;
        if (j < last || !hist_last_valid) PAT_CUDA(cudaStreamWaitEvent(st, p->ev_rec[j & 1], 0));
        const float* h = hist_of(p, w, j);
        const int lo = std::max(n0, 1);
        RC(run_adj(L, w, r, n1, lo, !have_q, h, n0, sg, sd));
        if (n1 >= lo) have_q = true;
        // segment j - 2 reuses this segment's buffer once its adjoint steps are done
        if (j - 2 >= 0) {
            PAT_CUDA(cudaEventRecord(p->ev_adj[j & 1], st));
            PAT_CUDA(cudaStreamWaitEvent(R, p->ev_adj[j & 1], 0));
            RC(recompute(p, p0, w, j - 2, R));
            PAT_CUDA(cudaEventRecord(p->ev_rec[(j - 2) & 1], R));
        }
    }
    if (L.split) {
        RC(split_adjoint_final(L, w, have_q, r, p0, grad_p0));
        return launch_reduce_cbar(L, w, grad_c);
    }
    RC(launch_row_adj_final1(L, w, have_q ? 0 : 1, r, grad_p0));
    RC(launch_col(L, w.A2, w.B2, 2, 1, -0.5f * sd));   // transpose of the initial half step
    RC(launch_row_adj_final2(L, w, p0, grad_p0));
    RC(launch_reduce_cbar(L, w, grad_c));
    return PAT_OK;
}

// Run body() directly, or (graphs enabled, non-default stream) replay the graph
// captured from the first call with the same kind, buffers and kernel variant.
template <class F>
int with_graph(pat_plan_s* p, int kind, const std::array<const void*, 10>& key, size_t ws_bytes, cudaStream_t st,
               F&& body) {
    if (!p->use_graphs || st == nullptr) return body();
    const int gv = 4 * p->variant + (p->persistent ? 1 : 0) + (p->cluster ? 2 : 0);   // variant and sweep form
    for (auto& g : p->graphs)
        if (g.kind == kind && g.variant == gv && g.key == key && g.ws_bytes == ws_bytes) {
            PAT_CUDA(cudaGraphLaunch(g.exec, st));
            add_launches(g.launches);
            g.last_use = ++p->graph_clock;
            return PAT_OK;
        }
    if (p->graphs.size() >= pat_plan_s::kMaxGraphs) {
        // an executable graph still in flight is released when its work completes
        auto lru = std::min_element(p->graphs.begin(), p->graphs.end(),
                                    [](const auto& a, const auto& b) { return a.last_use < b.last_use; });
        cudaGraphExecDestroy(lru->exec);
        p->graphs.erase(lru);
    }
    const unsigned long long l0 = launches_so_far();
    PAT_CUDA(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
    int rc = body();
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamEndCapture(st, &graph);
    if (rc != PAT_OK) {
        if (graph) cudaGraphDestroy(graph);
        return rc;
    }
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
    cudaGraphExec_t exec = nullptr;
    e = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate");
    const unsigned long long n = launches_so_far() - l0;
    p->graphs.push_back(pat_plan_s::Graph{kind, gv, key, ws_bytes, exec, n, ++p->graph_clock});
    PAT_CUDA(cudaGraphLaunch(exec, st));
    return PAT_OK;
}

int check_ws(const pat_plan_s* p, const void* ws, size_t bytes, bool grad) {
    if (!ws) { set_error("workspace is NULL"); return PAT_EINVAL; }
    if (reinterpret_cast<uintptr_t>(ws) % 256 != 0) { set_error("workspace must be 256-byte aligned"); return PAT_EINVAL; }
    const size_t need = grad ? p->ws_grad_passes : p->ws_fwd_passes;
    if (bytes < need) {
        set_error("workspace too small: %zu < %zu bytes", bytes, need);
        return PAT_ENOMEM;
    }
    return PAT_OK;
}

}  // namespace

int pat::objective(pat_plan_s* p, const float* c, const float* p0, const float* ymeas, const float* wts,
                   double* J_dev, void* ws, size_t ws_bytes, cudaStream_t st) {
    RC(check_ws(p, ws, ws_bytes, true));
    Ws w = resolve(p, ws, ws_bytes, true);
    RC(with_graph(p, 0, {c, p0, ymeas, wts, J_dev, ws}, ws_bytes, st, [&]() -> int {
        RC(forward_sweep(p, c, p0, w.ypred, w, false, st));
        Launch L{p, st};
        RC(launch_residual(L, w, w.ypred, ymeas, wts, w.resid, w.J));
        if (J_dev) PAT_CUDA(cudaMemcpyAsync(J_dev, w.J, p->ninst * sizeof(double), cudaMemcpyDeviceToDevice, st));
        return PAT_OK;
    }));
    p->hist_valid_ws = nullptr;
    return PAT_OK;
}

extern "C" int pat_forward(pat_plan p, const float* c, const float* p0, float* y, void* ws, size_t ws_bytes,
                           void* stream) {
    if (!p || !c || !p0 || !y) { set_error("pat_forward: null argument"); return PAT_EINVAL; }
    RC(check_ws(p, ws, ws_bytes, false));
    const bool keep = ws_bytes >= p->ws_grad_passes;
    Ws w = resolve(p, ws, ws_bytes, keep);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    RC(with_graph(p, keep ? 2 : 1, {c, p0, y, ws}, ws_bytes, st,
                  [&]() -> int { return forward_sweep(p, c, p0, y, w, keep, st); }));
    p->hist_valid_ws = keep ? ws : nullptr;
    return PAT_OK;
}

extern "C" int pat_adjoint_grad(pat_plan p, const float* c, const float* p0, const float* y_meas, const float* wts,
                                float* grad_p0, float* grad_c, double* J, float* y_pred, void* ws, size_t ws_bytes,
                                void* stream) {
    if (!p || !c || !p0 || !y_meas || !wts || !grad_p0 || !grad_c) {
        set_error("pat_adjoint_grad: null argument");
        return PAT_EINVAL;
    }
    RC(check_ws(p, ws, ws_bytes, true));
    Ws w = resolve(p, ws, ws_bytes, true);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    float* yp = y_pred ? y_pred : w.ypred;
    RC(with_graph(p, 3, {c, p0, y_meas, wts, grad_p0, grad_c, J, y_pred, ws}, ws_bytes, st, [&]() -> int {
        RC(forward_sweep(p, c, p0, yp, w, true, st));
        Launch L{p, st};
        RC(launch_residual(L, w, yp, y_meas, wts, w.resid, w.J));
        if (J) PAT_CUDA(cudaMemcpyAsync(J, w.J, p->ninst * sizeof(double), cudaMemcpyDeviceToDevice, st));
        return reverse_sweep(p, p0, w.resid, grad_p0, grad_c, w, true, st);
    }));
    p->hist_valid_ws = nullptr;
    return PAT_OK;
}

extern "C" int pat_vjp(pat_plan p, const float* c, const float* p0, const float* ybar, float* grad_p0, float* grad_c,
                       void* ws, size_t ws_bytes, void* stream) {
    if (!p || !c || !p0 || !ybar || !grad_p0 || !grad_c) { set_error("pat_vjp: null argument"); return PAT_EINVAL; }
    RC(check_ws(p, ws, ws_bytes, true));
    Ws w = resolve(p, ws, ws_bytes, true);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    Launch L{p, st};
    PAT_CUDA(cudaMemsetAsync(w.flag + 1, 0, sizeof(int), st));   // bounded-wait status of this call
    RC(launch_medium(L, c, w.cg));
    const bool valid = (p->hist_valid_ws == ws);
    RC(reverse_sweep(p, p0, ybar, grad_p0, grad_c, w, valid, st));
    p->hist_valid_ws = nullptr;
    return PAT_OK;
}

// Autotuner.  With a forward workspace it times forward steps; with a gradient workspace it
// times whole gradient evaluations (forward sweep with checkpoints and the reverse sweep with
// the recompute stream), since the variants differ in how the two streams share the SMs.
extern "C" int pat_plan_autotune(pat_plan p, void* ws, size_t ws_bytes, double* h_ms, void* stream) {
    if (!p) { set_error("pat_plan_autotune: null plan"); return PAT_EINVAL; }
    const int nv = pat_plan_variants(p);
    if (nv <= 0) return select_variant(p, -1);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    void* own = nullptr;
    if (!ws) {
        PAT_CUDA(cudaMallocAsync(&own, p->ws_fwd, st));
        ws = own;
        ws_bytes = p->ws_fwd;
    }
    const bool grad = ws_bytes >= p->ws_grad_passes;
    int rc = check_ws(p, ws, ws_bytes, grad);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    float* tmp = nullptr;   // gradient mode: c, p0, dJ/dp0, dJ/dc
    const size_t nn = size_t(p->n) * p->n;
    const size_t ntmp = 2 * (size_t(p->K) + p->ninst) * nn;
    double best = 1e300;
    int bestv = -1;
    if (rc == PAT_OK) {
        // zero state, spectra and residual; the timed passes then run on finite values
        if (cudaMemsetAsync(ws, 0, std::min(ws_bytes, grad ? p->ws_grad : p->ws_fwd), st) != cudaSuccess ||
            cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
            rc = cuda_fail(cudaGetLastError(), "pat_plan_autotune");
    }
    if (rc == PAT_OK && grad) {
        if (cudaMallocAsync(reinterpret_cast<void**>(&tmp), ntmp * sizeof(float), st) != cudaSuccess ||
            cudaMemsetAsync(tmp, 0, ntmp * sizeof(float), st) != cudaSuccess)
            rc = cuda_fail(cudaGetLastError(), "pat_plan_autotune buffers");
        if (rc == PAT_OK) rc = vfill(st, tmp, float(p->g.c_ref), size_t(p->ninst) * nn);
    }
    Ws w = resolve(p, ws, ws_bytes, grad);
    Launch L{p, st, true};   // forward-step timing mirrors the forward sweep
    float* c = tmp;
    float* p0 = tmp ? tmp + size_t(p->ninst) * nn : nullptr;
    float* gp0 = tmp ? p0 + size_t(p->K) * nn : nullptr;
    float* gc = tmp ? gp0 + size_t(p->K) * nn : nullptr;
    const int nsteps = 32;
    for (int v = -1; v < nv && rc == PAT_OK; ++v) {
        rc = select_variant(p, v);
        if (rc != PAT_OK) break;
        if (p->split && !w.split_fits) {   // the calls with this workspace would run another form
            if (h_ms) h_ms[v + 1] = HUGE_VAL;
            continue;
        }
        L.split = p->split;
        rc = run_steps(L, w, 1, 4, nullptr, nullptr, 0);   // first launches of the variant's kernels
        if (rc != PAT_OK) break;
        // the median of kSamples timings, so that one disturbed sample cannot decide the choice
        constexpr int kSamples = 3;
        float samples[kSamples];
        for (int r = 0; r < kSamples && rc == PAT_OK; ++r) {
            cudaEventRecord(e0, st);
            if (grad) {
                rc = forward_sweep(p, c, p0, w.ypred, w, true, st);
                if (rc == PAT_OK) rc = reverse_sweep(p, p0, w.resid, gp0, gc, w, true, st);
            } else {
                rc = run_steps(L, w, 1, 1 + nsteps, nullptr, nullptr, 0);
            }
            cudaEventRecord(e1, st);
            if (rc != PAT_OK) break;
            if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&samples[r], e0, e1) != cudaSuccess)
                rc = cuda_fail(cudaGetLastError(), "pat_plan_autotune timing");
        }
        if (rc != PAT_OK) break;
        std::sort(samples, samples + kSamples);
        const float ms = samples[kSamples / 2];
        const double per = grad ? double(ms) : double(ms) / nsteps;
        if (h_ms) h_ms[v + 1] = per;
        if (per < best) {
            best = per;
            bestv = v;
        }
    }
    p->hist_valid_ws = nullptr;
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (tmp) cudaFreeAsync(tmp, st);
    if (own) cudaFreeAsync(own, st);
    if (rc != PAT_OK) return rc;
    return select_variant(p, bestv);
}

extern "C" int pat_status(pat_plan p, const void* ws, int* h_flag, void* stream) {
    if (!p || !ws || !h_flag) { set_error("pat_status: null argument"); return PAT_EINVAL; }
    const char* b = static_cast<const char*>(ws);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int f[2] = {0, 0};
    PAT_CUDA(cudaMemcpyAsync(f, b + p->o_flag, 2 * sizeof(int), cudaMemcpyDeviceToHost, st));
    PAT_CUDA(cudaStreamSynchronize(st));
    *h_flag = (f[0] ? PAT_STATUS_NONFINITE : 0) | (f[1] & (PAT_STATUS_WAIT | PAT_STATUS_QUEUE | PAT_STATUS_BOUNDS));
    return PAT_OK;
}
