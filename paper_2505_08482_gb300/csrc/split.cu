// Host side of the split-axis passes (ksplit.cuh): the sides they are compiled for, and the
// sequences of the forward steps, the re-entry at a checkpoint and the adjoint steps.
#include <cuda_runtime.h>

#include <cmath>
#include <initializer_list>

#include "ksplit.cuh"
#include "pat_internal.h"

namespace pat {

// rho of the initial condition on the grid: rho_x = rho_y = p0 / (2 c^2) inside the domain
__global__ void k_split_init(const float* __restrict__ p0, const float* __restrict__ cg, const int* __restrict__ kinst,
                             float* __restrict__ rho, int n, int P, int N) {
    const int k = blockIdx.y;
    const size_t nn = size_t(N) * N;
    const float* c = cg + size_t(kinst[k]) * nn;
    float* rx = rho + size_t(k) * nn;
    float* ry = rx + size_t(gridDim.y) * nn;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < int(nn); i += gridDim.x * blockDim.x) {
        const int y = i / N, x = i - y * N;
        const int xd = x - P, yd = y - P;
        const bool in = xd >= 0 && xd < n && yd >= 0 && yd < n;
        const float cv = c[i];
        const float v = in ? p0[(size_t(k) * n + yd) * n + xd] / (2.f * cv * cv) : 0.f;
        rx[i] = v;
        ry[i] = v;
    }
}

// n = 0: grad_p0 = pb^0 - dt/(2 rho0) D ub + (rb_x + rb_y) / (2 c^2), dJ/dc = 2 / c sum_n p^n pb - (rb_x + rb_y) p0 / c^3;
// pb^0 = q_x + q_y, the divergence d_x + d_y and rb on the grid (two real fields [2][K][N][N] each)
__global__ void k_split_final(const float* __restrict__ q, const float* __restrict__ d, const float* __restrict__ rb,
                              const float* __restrict__ cg, const int* __restrict__ kinst,
                              const float* __restrict__ p0, float* __restrict__ grad_p0, float* __restrict__ cbar,
                              int n, int P, int N) {
    const int k = blockIdx.y;
    const size_t nn = size_t(N) * N, second = size_t(gridDim.y) * nn;
    const float* c = cg + size_t(kinst[k]) * nn;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n * n; i += gridDim.x * blockDim.x) {
        const int yd = i / n, xd = i - yd * n;
        const size_t o = size_t(k) * nn + size_t(yd + P) * N + xd + P;
        const size_t od = size_t(k) * n * n + i;
        const float cv = c[size_t(yd + P) * N + xd + P];
        const float c2 = cv * cv;
        const float rs = rb[o] + rb[second + o];
        grad_p0[od] = (q[o] + q[second + o]) + ((d[o] + d[second + o]) + rs / (2.f * c2));
        cbar[od] = 2.f * cbar[od] / cv - rs * p0[od] / (c2 * cv);
    }
}

const SplitOps* split_ops_small(int ng);
const SplitOps* split_ops_mid(int ng);
const SplitOps* split_ops_large(int ng);
const SplitOps* split_ops_xl(int ng);
const SplitOps* split_ops_xxl(int ng);
const SplitOps* split_ops_huge(int ng);

const SplitOps* split_ops_for(int ng) {
    for (auto f : {split_ops_small, split_ops_mid, split_ops_large, split_ops_xl, split_ops_xxl, split_ops_huge})
        if (const SplitOps* o = f(ng)) return o;
    return nullptr;
}

bool split_factors(int ng, int* n1, int* n2, const double** gain) {
    const SplitOps* o = split_ops_for(ng);
    if (!o) return false;
    *gain = o->mode_gain();
    *n1 = o->n1;
    *n2 = o->n2;
    return true;
}

int split_configure(const SplitOps* ops) { return ops->configure(); }

namespace {

#define RC(x)                          \
    do {                               \
        int rc_ = (x);                 \
        if (rc_ != PAT_OK) return rc_; \
    } while (0)

Geo geo_of(const pat_plan_s* p, const Ws& w) {
    Geo g = geo(p);
    g.status = w.flag + 1;
    return g;
}

float2 hi_lo(double v) { return make_float2(float(v), float(v - double(float(v)))); }

size_t field(const pat_plan_s* p) { return size_t(p->K) * p->ng * p->ng; }

int to_lines(const Launch& L, const Geo& g, const ToLinesArgs& a, int fields, bool pdl) {
    prof_begin(PAT_K_TO_LINES, L.st);
    L.split->to_lines(g, L.st, a, fields, pdl);
    prof_end(PAT_K_TO_LINES, L.st);
    return check_launch("ks_to_lines");
}

int lines(const Launch& L, const Geo& g, const LinesArgs& a) {
    prof_begin(PAT_K_LINES, L.st);
    L.split->lines(g, L.st, a);
    prof_end(PAT_K_LINES, L.st);
    return check_launch("ks_lines");
}

int to_real(const Launch& L, const Geo& g, const ToRealArgs& a, int fields) {
    prof_begin(PAT_K_TO_REAL, L.st);
    L.split->to_real(g, L.st, a, fields);
    prof_end(PAT_K_TO_REAL, L.st);
    return check_launch("ks_to_real");
}

// pressure lines of level `level` from rho_x, rho_y on the grid; its samples and history
int pressure(const Launch& L, const Geo& g, const Ws& w, const float* rx, const float* ry, int level, float* y,
             float* hist, int slot) {
    ToLinesArgs a{};
    a.mode = SP_PRESSURE;
    a.f0[0] = rx;
    a.f0[1] = ry;
    a.out0 = w.la;
    a.cg = w.cg;
    a.y = y;
    a.tstep = level;
    a.hist = hist;
    a.slot = slot;
    return to_lines(L, g, a, 1, true);
}

// rho lines of rho_x, rho_y and (ux not null) u lines of u_x, u_y
int enter(const Launch& L, const Geo& g, const Ws& w, const float* rx, const float* ry, const float* ux,
          const float* uy, bool pdl) {
    ToLinesArgs a{};
    a.mode = SP_COPY;
    a.f0[0] = rx;
    a.f0[1] = ry;
    a.f1[0] = ux;
    a.f1[1] = uy;
    a.out0 = w.lr;
    a.out1 = w.lu;
    a.scale0 = hi_lo(1.0 / L.p->ng);
    a.scale1 = hi_lo(L.p->g.rho0 / std::sqrt(double(L.p->ng)));
    a.cg = w.cg;
    return to_lines(L, g, a, ux ? 2 : 1, pdl);
}

}  // namespace

int split_start(const Launch& L, const Ws& w, const float* p0, float* y, float* hist, int hist_slot) {
    const pat_plan_s* p = L.p;
    const Geo g = geo_of(p, w);
    const size_t f = field(p);
    count_launch();
    k_split_init<<<dim3(unsigned((size_t(p->ng) * p->ng + 1023) / 1024), p->K), 256, 0, L.st>>>(
        p0, w.cg, p->t.kinst, w.re, p->n, p->P, p->ng);
    RC(check_launch("k_split_init"));
    RC(enter(L, g, w, w.re, w.re + f, nullptr, nullptr, false));
    ToLinesArgs a{};
    a.mode = SP_INIT;
    a.out0 = w.la;
    a.cg = w.cg;
    a.p0 = p0;
    a.y = y;
    a.hist = hist;
    a.slot = hist_slot;
    return to_lines(L, g, a, 1, true);
}

int split_enter(const Launch& L, const Ws& w, const float* state, int level, float* y, float* hist, int hist_slot) {
    const Geo g = geo_of(L.p, w);
    const size_t f = field(L.p);
    RC(enter(L, g, w, state + 2 * f, state + 3 * f, state, state + f, false));
    return pressure(L, g, w, state + 2 * f, state + 3 * f, level, y, hist, hist_slot);
}

int split_steps(const Launch& L, const Ws& w, int n0, int n1, float* y, float* hist, int hbase, float* ckpt) {
    const pat_plan_s* p = L.p;
    const Geo g = geo_of(p, w);
    const size_t f = field(p);
    for (int n = n0; n < n1; ++n) {
        const int lv = n + 1;
        LinesArgs a{};
        a.mode = n == 0 ? SP_STEP_FIRST : SP_STEP;
        a.in = w.la;
        a.u = w.lu;
        a.r = w.lr;
        RC(lines(L, g, a));
        float* c = (ckpt && lv % p->s_eff == 0) ? ckpt + size_t(lv / p->s_eff - 1) * 4 * f : nullptr;
        ToRealArgs b{};
        b.in0 = w.lr;
        b.d0[0] = c ? c + 2 * f : w.re;
        b.d0[1] = b.d0[0] + f;
        b.scale0 = make_float2(1.f, 0.f);
        b.scale1 = hi_lo(1.0 / (p->g.rho0 * std::sqrt(double(p->ng))));
        if (c) {
            b.in1 = w.lu;
            b.d1[0] = c;
            b.d1[1] = c + f;
        }
        RC(to_real(L, g, b, c ? 2 : 1));
        if (c) RC(enter(L, g, w, b.d0[0], b.d0[1], c, c + f, true));
        const bool h = hist && lv >= hbase;
        RC(pressure(L, g, w, b.d0[0], b.d0[1], lv, y, h ? hist : nullptr, lv - hbase));
    }
    return PAT_OK;
}

int split_adjoint(const Launch& L, const Ws& w, const float* r, int n_hi, int n_lo, bool first, const float* h,
                  int hbase) {
    const pat_plan_s* p = L.p;
    const Geo g = geo_of(p, w);
    const size_t f = field(p);
    for (int n = n_hi; n >= n_lo; --n) {
        ToRealArgs b{};
        b.in0 = w.la2;
        b.d0[0] = w.re2;
        b.d0[1] = w.re2 + f;
        b.scale0 = make_float2(1.f, 0.f);
        b.resid = r;
        b.tstep = n;
        b.zero = first && n == n_hi;
        RC(to_real(L, g, b, 1));
        ToLinesArgs t{};
        t.mode = SP_ADJOINT;
        t.f0[0] = w.re2;
        t.f0[1] = w.re2 + f;
        t.out0 = w.la2;
        t.cg = w.cg;
        t.hist = const_cast<float*>(h);
        t.slot = n - hbase;
        t.cbar = w.cbar;
        RC(to_lines(L, g, t, 1, true));
        LinesArgs a{};
        a.mode = SP_STEP_ADJOINT;
        a.in = w.la2;
        a.u = w.lub;
        a.r = w.lrb;
        a.out = w.la2;
        RC(lines(L, g, a));
    }
    return PAT_OK;
}

int split_adjoint_final(const Launch& L, const Ws& w, bool have_q, const float* r, const float* p0, float* grad_p0) {
    const pat_plan_s* p = L.p;
    const Geo g = geo_of(p, w);
    const size_t f = field(p);
    ToRealArgs b{};
    b.in0 = w.la2;
    b.d0[0] = w.re2;
    b.d0[1] = w.re2 + f;
    b.scale0 = make_float2(1.f, 0.f);
    b.resid = r;
    b.tstep = 0;
    b.zero = !have_q;
    RC(to_real(L, g, b, 1));
    LinesArgs a{};
    a.mode = SP_DIV;
    a.in = w.lub;
    a.out = w.la2;
    a.scale = -0.5f;
    RC(lines(L, g, a));
    // the divergence and rb on the grid; the forward state is free once the last recompute is used
    float* d = reinterpret_cast<float*>(w.lu);
    float* rb = reinterpret_cast<float*>(w.lr);
    ToRealArgs e{};
    e.in0 = w.la2;
    e.in1 = w.lrb;
    e.d0[0] = d;
    e.d0[1] = d + f;
    e.d1[0] = rb;
    e.d1[1] = rb + f;
    e.scale0 = make_float2(1.f, 0.f);
    e.scale1 = hi_lo(1.0 / p->ng);
    RC(to_real(L, g, e, 2));
    count_launch();
    k_split_final<<<dim3(unsigned((size_t(p->n) * p->n + 1023) / 1024), p->K), 256, 0, L.st>>>(
        w.re2, d, rb, w.cg, p->t.kinst, p0, grad_p0, w.cbar, p->n, p->P, p->ng);
    return check_launch("k_split_final");
}

}  // namespace pat
