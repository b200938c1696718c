// adjoint.cu -- gradient of a ramp's final-state infidelity with respect to
// the knots of the potential schedule, by the discrete adjoint of the RK4 step.
//
// The forward pass (gpe_ramp_forward) is the real-time RK4 ramp of Eq. (8)
// with V(t) = (1 - s(t)) V0 + s(t) V1 (the linear interpolation between
// potentials of Sec. V) and keeps a checkpoint of psi every K steps.  The
// backward pass (gpe_ramp_backward) seeds dL/dpsi(T) for
// L = 1 - |<psi_t|psi(T)>|^2, then walks the segments from the last: it
// recomputes the segment's step-start states (and, where memory allows, keeps
// the stage states Y2, Y3, Y4) from its checkpoint, and for each step (last
// first) runs four adjoint-stage kernels.  With psi as the real pair (Re, Im),
// a gradient G is stored as dL/dRe + i dL/dIm, and the transposed Jacobian of
// f(y) = -i [(T + V) y + g|y|^2 y] acting on G is
//   J^T G = i (T + V) G + 2 i g |y|^2 G - i g y^2 conj(G).
// Reversing y1 = y0 + dt (k1 + 2 k2 + 2 k3 + k4)/6:
//   mu4 = dt/6 lam'             nu4 = J4^T mu4
//   mu3 = dt/3 lam' + dt nu4     nu3 = J3^T mu3
//   mu2 = dt/3 lam' + dt/2 nu3   nu2 = J2^T mu2
//   mu1 = dt/6 lam' + dt/2 nu2   nu1 = J1^T mu1
//   lam = lam' + nu1 + nu2 + nu3 + nu4
// and every stage adds Re<mu_i, -i (V1 - V0) Y_i> = sum (V1 - V0) Im(conj(mu_i) Y_i),
// reduced in FP64, to the two knots whose hat functions cover its time.
// Bulk arithmetic runs in the state's precision; the gradient accumulates in
// FP64.
#include <algorithm>
#include <cmath>
#include <vector>

#include "gpe_internal.cuh"
#include "kernels.cuh"

namespace gpe {

template <typename R>
struct AdjArgs {
    using CT = typename Cx<R>::T;
    const CT *mu_in;  // gathered: mu_i (stage 4: lam', scaled by m_scale)
    R m_scale;
    const CT *Y;      // stage state Y_i
    const CT *lam;    // lam' (own cells)
    CT *lam_out;      // lam, written by the last stage (may alias lam)
    CT *acc;          // running lam' + sum nu
    CT *mu_out;       // mu_{i-1} = cl lam' + cn nu_i
    const R *V0;
    const R *V1;
    R s;              // schedule value at the stage time
    R cl, cn;
    R ihx2, ihy2, ihz2, g;
    double *partials;
    unsigned int *counter;
    double *grad;     // [16] FP64 knot gradient
    int k0;
    double w0, w1;    // hat weights of knots k0, k0+1 at the stage time
};

// mu_i = m_scale lam' at the first stage of the reverse sweep
template <typename R>
struct TileScale {
    R s;
    using P4 = Plain::P4;
    using P1 = Plain::P1;
    __device__ __forceinline__ P4 load4(uint32_t) const { return {}; }
    __device__ __forceinline__ P1 load1(uint32_t) const { return {}; }
    template <typename CT>
    __device__ __forceinline__ void seg(CT (&v)[4], const P4 &) const
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = scale(v[i], s);
    }
    template <typename CT, typename PRE>
    __device__ __forceinline__ void own(CT (&v)[4], const PRE &) const { seg(v, P4{}); }
    template <typename CT>
    __device__ __forceinline__ void cell(CT &v, const P1 &) const { v = scale(v, s); }
};

// POS: 0 the first of the four stages (mu_i is lam' scaled, nothing is
// accumulated yet), 1 the middle ones, 2 the last (writes lam).  All own-cell
// operands are loaded with the tile; they were the pass's latency when they
// were read once the tile was in place.  512^3 ramp, complex64: 70 -> 42, 55
// and 45 us a stage (5.1 to 5.9 TB/s), bound by bytes in flight: the operands'
// registers leave five blocks an SM.
template <typename R, int POS>
__global__ void __launch_bounds__(TILE, sizeof(R) == 4 ? 5 : 2) k_adj_stage(const AdjArgs<R> a, const TileView T)
{
    using CT = typename Cx<R>::T;
    using XF = typename std::conditional<POS == 0, TileScale<R>, Plain>::type;
    struct Pre {
        R V0[4], V1[4];
        CT Y[4], lam[4], acc[4];
    };
    const auto co = tile_co<7, LapFull>(a.ihx2, a.ihy2, a.ihz2);  // before the wait
    const TileList list = tile_begin(T);
    XF xf{};
    if constexpr (POS == 0) xf.s = a.m_scale;
    Sum64<R> dot[1];
    int n = 0;
    tile_loop<7>(T, list, a.mu_in, xf, co, EveryTile(),
                 [&](uint32_t idx, uint32_t m) {
                     prefetch_l2(a.V0 + idx, m * (uint32_t)sizeof(R));
                     prefetch_l2(a.V1 + idx, m * (uint32_t)sizeof(R));
                     prefetch_l2(a.Y + idx, m * (uint32_t)sizeof(CT));
                     if constexpr (POS != 0) prefetch_l2(a.acc + idx, m * (uint32_t)sizeof(CT));
                     if constexpr (POS == 1) prefetch_l2(a.lam + idx, m * (uint32_t)sizeof(CT));
                 },
                 [&](uint32_t idx) {
                     Pre p;
                     ldr4(a.V0 + idx, p.V0);
                     ldr4(a.V1 + idx, p.V1);
                     ld4<false>(a.Y + idx, p.Y);
                     if constexpr (POS != 2) ld4<false>(a.lam + idx, p.lam);
                     if constexpr (POS != 0) ld4<false>(a.acc + idx, p.acc);
                     return p;
                 },
                 [&](uint32_t idx, const Pre &p, const CT(&M)[4], const CT(&L)[4]) {
                     CT nacc[4], mo[4];
                     R d4 = (R)0;  // the segment's share of the knot derivative, added in FP64 once
#pragma unroll
                     for (int i = 0; i < 4; ++i) {
                         const bool act = active_v(p.V0[i]);  // else an inactive cell of a stored segment
                         const CT Y = p.Y[i];
                         const R dV = p.V1[i] - p.V0[i];
                         const R Vt = ((R)1 - a.s) * p.V0[i] + a.s * p.V1[i];
                         const R rho = Y.x * Y.x + Y.y * Y.y;
                         // C = (T + Vt + 2 g rho) M - g Y^2 conj(M);  nu = i C
                         const R w = Vt + (R)2 * a.g * rho;
                         const R y2r = Y.x * Y.x - Y.y * Y.y, y2i = (R)2 * Y.x * Y.y;
                         const R br = y2r * M[i].x + y2i * M[i].y;  // Re(Y^2 conj(M))
                         const R bi = y2i * M[i].x - y2r * M[i].y;  // Im(Y^2 conj(M))
                         const R cr = (R)(-0.5) * L[i].x + w * M[i].x - a.g * br;
                         const R ci = (R)(-0.5) * L[i].y + w * M[i].y - a.g * bi;
                         const CT nu = act ? cmk<R>(-ci, cr) : czero<CT>();
                         if (act) d4 += dV * (M[i].x * Y.y - M[i].y * Y.x);
                         if constexpr (POS == 0) nacc[i] = vadd(p.lam[i], nu);
                         else nacc[i] = vadd(p.acc[i], nu);
                         if constexpr (POS != 2) {
                             mo[i].x = a.cl * p.lam[i].x + a.cn * nu.x;
                             mo[i].y = a.cl * p.lam[i].y + a.cn * nu.y;
                         }
                     }
                     if constexpr (POS == 2) {
                         st4(a.lam_out + idx, nacc);
                     } else {
                         st4(a.acc + idx, nacc);
                         st4(a.mu_out + idx, mo);
                     }
                     dot[0].add(d4);
                     keep<1>(dot, ++n);
                 });
    double tot[1];
    block_totals<1>(dot, tot);
    if (launch_totals<1>(tot, a.partials, a.counter) && threadIdx.x == 0) {
        a.grad[a.k0] += a.w0 * tot[0];
        a.grad[a.k0 + 1] += a.w1 * tot[0];
    }
}

// seed of the reverse sweep: lam = dL/dpsi(T) = -2 dV c psi_t for
// L = 1 - |c|^2, c = <psi_t|psi(T)>.  Nothing at inactive cells, where psi(T) is 0
// whatever the target holds (a cell of the region may have V0 = +inf, a wall):
// the stages keep lam there as it is.
template <typename R, typename CT>
__global__ void k_seed(CT *lam, const CT *tgt, const R *V0, int64_t n, double cr, double ci, double dV)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const CT t = tgt[i];
        CT o;
        o.x = (-2.0 * dV) * (cr * t.x - ci * t.y);
        o.y = (-2.0 * dV) * (cr * t.y + ci * t.x);
        lam[i] = active_v(V0[i]) ? o : czero<CT>();
    }
}

__global__ void k_set_clock(double *p, double v) { *p = v; }

// s(t) on the host, the same piecewise-linear schedule as ramp_s
static double ramp_s_host(const gpe_real_params &p, double t)
{
    const int nk = p.n_knots;
    if (t <= 0.0) return p.knots[0];
    if (t >= p.T_ramp) return p.knots[nk - 1];
    const double u = t / p.T_ramp * (double)(nk - 1);
    int k = (int)std::floor(u);
    if (k >= nk - 1) k = nk - 2;
    const double w = u - (double)k;
    return (1.0 - w) * p.knots[k] + w * p.knots[k + 1];
}

// hat weights of the knots at time t (the interpolation of the schedule)
static void hat(const gpe_real_params &p, double t, int &k0, double &w0, double &w1)
{
    const int nk = p.n_knots;
    if (t <= 0.0) {
        k0 = 0;
        w0 = 1.0;
        w1 = 0.0;
        return;
    }
    if (t >= p.T_ramp) {
        k0 = nk - 2;
        w0 = 0.0;
        w1 = 1.0;
        return;
    }
    const double u = t / p.T_ramp * (double)(nk - 1);
    k0 = (int)std::floor(u);
    if (k0 >= nk - 1) k0 = nk - 2;
    const double w = u - (double)k0;
    w0 = 1.0 - w;
    w1 = w;
}

}  // namespace gpe

using namespace gpe;

struct gpe_tape {
    gpe_state *st = nullptr;
    gpe_real_params p{};
    int64_t nsteps = 0, nck = 0;
    double t0 = 0.0;
    int K = 0;
    bool last_kept = false;  // the last segment's states are those that the forward pass left
    void *d_ckpt = nullptr;  // [nck * n_packed]
    void *d_seg = nullptr;   // [K * n_packed] step-start states of a segment after the first
    void *d_stages = nullptr;  // [3 * K * n_packed] the stage states of a segment's steps, where memory allows
    void *d_lam = nullptr, *d_mu[2] = {nullptr, nullptr}, *d_acc = nullptr;
    void *d_w[4] = {nullptr, nullptr, nullptr, nullptr};  // Y2, Y3, Y4, RK4 partial sum
    void *block = nullptr;     // the allocation that holds every array but the stage states
    double *d_grad = nullptr;
    double *d_clock = nullptr;
    double *d_stab = nullptr;  // [3 * K] schedule values of a segment's stages
    RedScratch red;
};

static void tape_free(gpe_tape *t)
{
    if (!t) return;
    dev_free(t->block);
    dev_free(t->d_stages);
    if (t->st) t->st->grid->n_states--;
    delete t;
}

extern "C" int gpe_tape_destroy(gpe_tape *t)
{
    cudaDeviceSynchronize();
    tape_free(t);
    return GPE_OK;
}

namespace gpe {

// The RK4 stages of a segment's steps on the tape's buffers.  The step-start
// states are the segment's checkpoint, then seg[0], seg[1] ... (stage 3 reads
// no y0, so it writes the next one where it stays); the stage states go to
// their store where there is one.
template <typename R>
struct SegmentSteps {
    using CT = typename Cx<R>::T;
    gpe_tape *t;
    RkArgs<R> f{};
    TileLaunch L;
    cudaStream_t s;
    int init(gpe_tape *t_, cudaStream_t s_)
    {
        t = t_;
        s = s_;
        gpe_state *st = t->st;
        const gpe_grid *g = st->grid;
        const gpe_real_params &p = t->p;
        f.V0 = (const R *)potential_ptr(st, 0);
        f.V1 = (const R *)potential_ptr(st, 1);
        if (!f.V0 || !f.V1) return fail(GPE_ERR_STATE, "ramp needs potential slots 0 and 1");
        f.y2 = (CT *)t->d_w[0];
        f.y3 = (CT *)t->d_w[1];
        f.y4 = (CT *)t->d_w[2];  // kept apart from Y2: the reverse sweep reads all three
        f.w = (CT *)t->d_w[3];
        f.ihx2 = (R)(1.0 / (g->box.hx * g->box.hx));
        f.ihy2 = (R)(1.0 / (g->box.hy * g->box.hy));
        f.ihz2 = (R)(1.0 / (g->box.hz * g->box.hz));
        f.g = (R)p.g;
        f.dt = (R)p.dt;
        f.dtd = p.dt;
        f.ramp.clock = t->d_clock;
        f.ramp.T = p.T_ramp;
        f.ramp.n_knots = p.n_knots;
        for (int k = 0; k < GPE_MAX_KNOTS; ++k) f.ramp.knots[k] = p.knots[k];
        L = tile_launch<CT, 7>(g->tiles);
        return GPE_OK;
    }
    // the schedule's values for len steps from n0 steps after the clock
    int table(int64_t n0, int64_t len) const
    {
        k_ramp_table<<<1, 256, 0, s>>>(f.ramp, t->d_clock, 0.0, n0, (int)len, 3, RK4_TIMES, t->p.dt, t->d_stab);
        GPE_LAUNCH_CHECK();
        return GPE_OK;
    }
    CT *start(int64_t j, int64_t m) const
    {
        const size_t np = (size_t)t->st->grid->n_packed;
        return m == 0 ? (CT *)t->d_ckpt + j * np : (CT *)t->d_seg + (m - 1) * np;
    }
    // stage stg of step m of the segment, from f.y0
    int stage(int64_t m, int stg)
    {
        const auto k = Rk4Tiles<R, 7>::get(true, stg, fixed_spacings(t->st->grid->box));
        f.stab = t->d_stab + 3 * m + (stg + 1) / 2;
        if (t->d_stages) {
            const size_t np = (size_t)t->st->grid->n_packed;
            CT *y = (CT *)t->d_stages + 3 * m * np;
            f.y2 = y;
            f.y3 = y + np;
            f.y4 = y + 2 * np;
        }
        return tile_run(k, tile_blocks(k, t->st->grid->nsm, L.T.ntiles, L.smem), L, s, f, L.T);
    }
    // step m of segment j; its result goes to `end`
    int step(int64_t j, int64_t m, CT *end)
    {
        f.y0 = start(j, m);
        for (int stg = 0; stg < 3; ++stg) GPE_TRY(stage(m, stg));
        f.y0 = end;
        return stage(m, 3);
    }
};

// The last segment's steps with every state kept for the reverse sweep, which
// then does not compute that segment again: 512^3 ramp gradient over 48 steps,
// K = 16: 25.6 -> 23.5 ms.
template <typename R>
static int forward_kept(gpe_tape *t, int64_t n, cudaStream_t s)
{
    using CT = typename Cx<R>::T;
    const int64_t j = t->nck - 1;
    SegmentSteps<R> run;
    GPE_TRY(run.init(t, s));
    k_set_clock<<<1, 1, 0, s>>>(t->d_clock, t->t0 + (double)(j * t->K) * t->p.dt);
    GPE_LAUNCH_CHECK();
    GPE_TRY(run.table(0, n));
    for (int64_t m = 0; m < n; ++m) GPE_TRY(run.step(j, m, m + 1 < n ? run.start(j, m + 1) : (CT *)t->st->d_psi));
    t->last_kept = true;
    return GPE_OK;
}

}  // namespace gpe

extern "C" int gpe_ramp_forward(gpe_state *st, const gpe_real_params *p, int64_t nsteps, double t0, int K,
                                gpe_tape **out, gpe_stream stream)
{
    if (!st || !p || !out) return fail(GPE_ERR_ARG, "NULL argument");
    *out = nullptr;
    if (nsteps < 1 || K < 1) return fail(GPE_ERR_ARG, "need nsteps >= 1 and K >= 1");
    if (p->potential != GPE_V_BLEND) return fail(GPE_ERR_ARG, "the ramp gradient needs potential = GPE_V_BLEND");
    if (p->integrator != GPE_RK4) return fail(GPE_ERR_ARG, "the ramp gradient is the adjoint of the RK4 step");
    if (st->dtype != GPE_C128 && st->dtype != GPE_C64) return fail(GPE_ERR_ARG, "the ramp gradient needs a complex state");
    if (st->grid->stencil != 7) return fail(GPE_ERR_ARG, "the ramp gradient is built for the 7-point stencil");
    const gpe_grid *g = st->grid;
    const size_t bytes = (size_t)g->n_packed * st->elem;
    gpe_tape *t = new gpe_tape();
    t->p = *p;
    t->nsteps = nsteps;
    t->t0 = t0;
    t->K = (int)std::min<int64_t>(K, nsteps);
    t->nck = (nsteps + t->K - 1) / t->K;
    // every pass writes whole segments before the next one reads them: no zeroing
    int rc = dev_alloc_parts(&t->block, {{&t->d_ckpt, bytes * t->nck},
                                         {&t->d_seg, bytes * t->K},
                                         {&t->d_lam, bytes},
                                         {&t->d_mu[0], bytes},
                                         {&t->d_mu[1], bytes},
                                         {&t->d_acc, bytes},
                                         {&t->d_w[0], bytes},
                                         {&t->d_w[1], bytes},
                                         {&t->d_w[2], bytes},
                                         {&t->d_w[3], bytes},
                                         {&t->d_stab, 3 * (size_t)t->K},
                                         {&t->d_grad, GPE_MAX_KNOTS},
                                         {&t->d_clock, 1},
                                         red_partials(t->red, g->nsm),
                                         red_counter(t->red),
                                         red_scalars(t->red)});
    // The reverse sweep needs every step's stage states.  Kept from the
    // segment's recomputation they save three of its fifteen passes a step
    // (512^3 ramp, 48 steps, K = 16: 32.5 -> 27.4 ms with the schedule table); they are kept where they take at
    // most an eighth of the memory that is free, and computed again otherwise.
    if (rc == GPE_OK) {
        size_t avail = 0, total = 0;
        if (cudaMemGetInfo(&avail, &total) == cudaSuccess && 3 * bytes * t->K <= avail / 8 &&
            cudaMalloc(&t->d_stages, 3 * bytes * t->K) != cudaSuccess)
            t->d_stages = nullptr;
        cudaGetLastError();
    }
    if (rc == GPE_OK) rc = red_zero(t->red);
    if (rc != GPE_OK) {
        tape_free(t);
        return rc;
    }
    t->st = st;
    st->grid->n_states++;
    cudaStream_t s = S(stream);
    for (int64_t j = 0; j < t->nck; ++j) {
        const int64_t n = std::min<int64_t>(t->K, nsteps - j * t->K);
        cudaError_t e = cudaMemcpyAsync((char *)t->d_ckpt + j * bytes, st->d_psi, bytes, cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) {
            tape_free(t);
            return cuda_fail(e, "checkpoint copy", __FILE__, __LINE__);
        }
        const bool keep = j == t->nck - 1 && t->d_stages && g->sched == GPE_SCHED_STAGED;
        rc = gpe_step_real(st, p, keep ? 0 : n, t0 + (double)(j * t->K) * p->dt, stream);  // no steps: the checks
        if (rc == GPE_OK && keep) rc = st->dtype == GPE_C128 ? forward_kept<double>(t, n, s) : forward_kept<float>(t, n, s);
        if (rc != GPE_OK) {
            tape_free(t);
            return rc;
        }
    }
    *out = t;
    return GPE_OK;
}

namespace gpe {

template <typename R>
static int backward_impl(gpe_tape *t, const gpe_state *target, double *grad, double *loss, cudaStream_t s)
{
    using CT = typename Cx<R>::T;
    gpe_state *st = t->st;
    const gpe_grid *g = st->grid;
    const gpe_real_params &p = t->p;
    const size_t np = (size_t)g->n_packed;
    // loss and seed
    double c[2];
    GPE_TRY(gpe_overlap(target, st, c, (gpe_stream)s));
    *loss = 1.0 - (c[0] * c[0] + c[1] * c[1]);
    const double dV = g->box.hx * g->box.hy * g->box.hz;
    CT *lam = (CT *)t->d_lam;
    GPE_TRY_CUDA(cudaMemsetAsync(t->d_grad, 0, GPE_MAX_KNOTS * sizeof(double), s));
    // forward stage kernels on tape buffers; times from the tape's start
    k_set_clock<<<1, 1, 0, s>>>(t->d_clock, t->t0);
    GPE_LAUNCH_CHECK();
    SegmentSteps<R> run;
    GPE_TRY(run.init(t, s));
    const RkArgs<R> &f = run.f;
    k_seed<R, CT><<<g->nsm * 8, 256, 0, s>>>(lam, (const CT *)target->d_psi, f.V0, (int64_t)np, c[0], c[1], dV);
    GPE_LAUNCH_CHECK();
    const TileLaunch &tl = run.L;
    auto blocks = [&](auto k) { return tile_blocks(k, g->nsm, tl.T.ntiles, tl.smem); };
    using KA = void (*)(AdjArgs<R>, TileView);
    const KA ka[4] = {k_adj_stage<R, 0>, k_adj_stage<R, 1>, k_adj_stage<R, 1>, k_adj_stage<R, 2>};
    AdjArgs<R> a{};
    a.lam = lam;
    a.lam_out = lam;
    a.acc = (CT *)t->d_acc;
    a.V0 = f.V0;
    a.V1 = f.V1;
    a.ihx2 = f.ihx2;
    a.ihy2 = f.ihy2;
    a.ihz2 = f.ihz2;
    a.g = f.g;
    a.partials = t->red.partials;
    a.counter = t->red.counter;
    a.grad = t->d_grad;
    const R dt = (R)p.dt;
    for (int64_t j = t->nck - 1; j >= 0; --j) {
        const int64_t len = std::min<int64_t>(t->K, t->nsteps - j * t->K);
        const bool kept = t->last_kept && j == t->nck - 1;
        if (!kept) {
            GPE_TRY(run.table(j * t->K, len));
            for (int64_t m = 0; m + 1 < len; ++m) GPE_TRY(run.step(j, m, run.start(j, m + 1)));
        }
        if (t->nck > 1) t->last_kept = false;  // the other segments take its place
        for (int64_t m = len - 1; m >= 0; --m) {
            const double tm = t->t0 + (double)(j * t->K + m) * p.dt;
            run.f.y0 = run.start(j, m);
            if (!t->d_stages || (m == len - 1 && !kept))
                for (int stg = 0; stg < 3; ++stg) GPE_TRY(run.stage(m, stg));  // Y2, Y3, Y4
            // stages 4, 3, 2, 1 of the reverse sweep
            const double ts[4] = {tm + p.dt, tm + 0.5 * p.dt, tm + 0.5 * p.dt, tm};
            const CT *Ys[4] = {f.y4, f.y3, f.y2, f.y0};
            if (t->d_stages) {
                const CT *ys = (const CT *)t->d_stages + 3 * m * np;
                Ys[0] = ys + 2 * np;
                Ys[1] = ys + np;
                Ys[2] = ys;
            }
            const R cl[4] = {dt / (R)3, dt / (R)3, dt / (R)6, (R)0};
            const R cn[4] = {dt, dt / (R)2, dt / (R)2, (R)0};
            CT *mu[2] = {(CT *)t->d_mu[0], (CT *)t->d_mu[1]};
            for (int r = 0; r < 4; ++r) {
                a.mu_in = r == 0 ? lam : mu[(r - 1) & 1];
                a.m_scale = r == 0 ? dt / (R)6 : (R)1;
                a.mu_out = mu[r & 1];
                a.Y = Ys[r];
                a.s = (R)ramp_s_host(p, ts[r]);
                a.cl = cl[r];
                a.cn = cn[r];
                hat(p, ts[r], a.k0, a.w0, a.w1);
                GPE_TRY(tile_run(ka[r], blocks(ka[r]), tl, s, a, tl.T));
            }
        }
    }
    double h[GPE_MAX_KNOTS];
    GPE_TRY_CUDA(cudaMemcpyAsync(h, t->d_grad, sizeof h, cudaMemcpyDeviceToHost, s));
    GPE_TRY_CUDA(cudaStreamSynchronize(s));
    for (int k = 0; k < p.n_knots; ++k) grad[k] = h[k];
    return GPE_OK;
}

}  // namespace gpe

extern "C" int gpe_ramp_backward(gpe_tape *t, const gpe_state *target, double *grad_knots, double *loss,
                                 gpe_stream stream)
{
    if (!t || !target || !grad_knots || !loss) return fail(GPE_ERR_ARG, "NULL argument");
    if (target->grid != t->st->grid || target->dtype != t->st->dtype)
        return fail(GPE_ERR_ARG, "target must share the tape state's grid and dtype");
    const bool c128 = t->st->dtype == GPE_C128;
    cudaStream_t s = S(stream);
    return c128 ? backward_impl<double>(t, target, grad_knots, loss, s)
                : backward_impl<float>(t, target, grad_knots, loss, s);
}
