// kernels.cuh -- device kernels shared by the step translation units (the
// 7-point and 19-point builds): the imaginary-time stencil passes, the
// propagator table, the deferred renormalisation and the observables.  Not
// part of the ABI.
#pragma once

#include "tiles.cuh"

namespace gpe {

// a + b rounded once and never fused with the product that feeds it, so that
// the per-segment sums of a real state and of a complex state with zero
// imaginary part round identically
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }

// E = exp(-V dt/2) in the state precision (Eq. (7): the diagonal propagator
// is precomputed once per dt); E = -1 marks the inactive cells of stored
// segments (V = +inf there)
template <typename R>
__global__ void k_make_E(const double *V, R *E, int64_t n, double dt)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        E[i] = V[i] < INFINITY ? (R)exp(-V[i] * dt / 2.0) : (R)-1;
}

// ------------------------------------------------------------ imaginary time
// Sec. II A/B, Eqs. (6)-(7).  Stage A gathers psi with its neighbours,
// applying on load the pending renormalisation factor and the diagonal half
// step psi * E * (1 - g|psi|^2 dt/2), E = exp(-V dt/2); then the first Euler
// kinetic substep psi - (dt/2) T psi = psi + (dt/4) lap psi -> tmp.
// Stage B gathers tmp, takes the second Euler substep, applies the diagonal
// half step again, writes psi and sums |psi|^2 in FP64; the factor
// sqrt(N / (sum |psi|^2 dV)) is stored for the next step's stage A (or the
// end of the call).  E = -1 marks the inactive cells of stored segments
// (V = +inf), which are set to zero.
template <typename R, typename CT = typename Cx<R>::T>
struct ItpArgs {
    CT *psi;
    CT *tmp;
    const R *E;
    R ihx2, ihy2, ihz2, g, dt;
    double *scalars;  // [0] scale to apply on load / next scale, [1] last norm
    double N, dV;
};

// The propagator table E of a segment (E < 0 marks an inactive cell), loaded
// ahead of the segment's update
template <typename R>
struct ELoad {
    const R *E;
    struct P {
        R e[4];
    };
    __device__ __forceinline__ P operator()(uint32_t idx) const
    {
        P p;
        ldr4(E + idx, p.e);
        return p;
    }
};

template <typename R, typename CT, int BX, int BY, int BZ, bool CG>
__device__ __forceinline__ void itp_brick_a(const ItpArgs<R, CT> &a, const GridView &G, int64_t b, int64_t next,
                                            WarpSpace<CT, BX, BY, BZ> &ws, R sc)
{
    const R q4 = a.dt / (R)4;
    const R ax = euler_coef(a.ihx2, q4), ay = euler_coef(a.ihy2, q4), az = euler_coef(a.ihz2, q4);
    const DiagLoad<R, CT> diag{sc, a.g * a.dt / (R)2, a.E};
    brick_apply<BX, BY, BZ, CG, LapEuler>(ws, G, b, next, a.psi, diag, ax, ay, az, ELoad<R>{a.E},
                                [&](uint32_t idx, const typename ELoad<R>::P &p, const CT(&c)[4], const CT(&L)[4]) {
        CT o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool act = p.e[i] >= (R)0;  // E < 0 marks an inactive cell of a stored segment
            o[i] = act ? euler(c[i], q4, L[i]) : czero<CT>();
        }
        st4(a.tmp + idx, o);
    });
}

template <typename R, typename CT, int BX, int BY, int BZ, bool CG>
__device__ __forceinline__ void itp_brick_b(const ItpArgs<R, CT> &a, const GridView &G, int64_t b, int64_t next,
                                            WarpSpace<CT, BX, BY, BZ> &ws, double &acc)
{
    const R hg = a.g * a.dt / (R)2;
    const R q4 = a.dt / (R)4;
    const R ax = euler_coef(a.ihx2, q4), ay = euler_coef(a.ihy2, q4), az = euler_coef(a.ihz2, q4);
    brick_apply<BX, BY, BZ, CG, LapEuler>(ws, G, b, next, a.tmp, Identity(), ax, ay, az, ELoad<R>{a.E},
                                [&](uint32_t idx, const typename ELoad<R>::P &p, const CT(&c)[4], const CT(&L)[4]) {
        CT o[4];
        R n4 = (R)0;  // the segment's |psi|^2, added to the FP64 sum once
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            o[i] = euler(c[i], q4, L[i]);
            const R f = p.e[i] >= (R)0 ? p.e[i] * ((R)1 - hg * norm2(o[i])) : (R)0;
            o[i] = scale(o[i], f);
            n4 = add_rn(n4, norm2(o[i]));
        }
        acc += (double)n4;
        st4(a.psi + idx, o);
    });
}

// The staged passes, on tiles (tiles.cuh).  A halo segment's propagator is
// loaded beside its values, an own segment's serves its transform and its
// update.  1024^3 shell, complex64: 0.382 -> 0.275 ms a step against the
// former warp-per-brick passes (1.3 GB, 4.7 TB/s); bound by the shared-memory
// pipe (86 and 80 % busy at 512^3).
template <typename R, typename CT>
struct TileDiag {
    DiagLoad<R, CT> d;
    struct P4 {
        R e[4];
    };
    using P1 = R;
    __device__ __forceinline__ P4 load4(uint32_t idx) const
    {
        P4 p;
        ldr4(d.E + idx, p.e);
        return p;
    }
    __device__ __forceinline__ R load1(uint32_t idx) const { return __ldg(d.E + idx); }
    __device__ __forceinline__ void seg(CT (&v)[4], const P4 &p) const
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = d.apply(v[i], p.e[i]);
    }
    __device__ __forceinline__ void own(CT (&v)[4], const typename ELoad<R>::P &p) const
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = d.apply(v[i], p.e[i]);
    }
    __device__ __forceinline__ void cell(CT &v, const R &e) const { v = d.apply(v, e); }
};

// The block's totals of NV sums, to every thread.  Few FP64 instructions, since
// every warp of an SM queues for the one pipe at a kernel's end: pairs are
// added across a warp as pairs, and one warp converts; doubles are added
// across the block by a warp a sum.  The threads' FP64 totals (flushed pairs) are
// added only in blocks that have any.
// Called by the whole block of TILE threads.
template <int NV>
__device__ __forceinline__ void block_totals(Sum64<float> (&s)[NV], double (&out)[NV])
{
    constexpr int W = TILE / 32;
    __shared__ float2 sp[NV][W];
    __shared__ double sd[NV][W], so[NV];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    bool own = false;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        for (int off = 16; off > 0; off >>= 1)
            s[k].add(__shfl_down_sync(0xffffffffu, s[k].hi, off), __shfl_down_sync(0xffffffffu, s[k].lo, off));
        if (lane == 0) sp[k][warp] = make_float2(s[k].hi, s[k].lo);
        own |= __double_as_longlong(s[k].tot) != 0;
    }
    const bool any = __syncthreads_or(own);
    if (any) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            double x = s[k].tot;
            for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
            if (lane == 0) sd[k][warp] = x;
        }
        __syncthreads();
    }
    if (threadIdx.x < NV) {
        double x = 0.0;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const float2 p = sp[threadIdx.x][w];
            x = add_pair(x, p.x, p.y);
            if (any) x += sd[threadIdx.x][w];
        }
        so[threadIdx.x] = x;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) out[k] = so[k];
    __syncthreads();  // the arrays may be used again
}
template <int NV>
__device__ __forceinline__ void block_totals(Sum64<double> (&s)[NV], double (&out)[NV])
{
    __shared__ double sm[NV][TILE], so[NV];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) sm[k][threadIdx.x] = s[k].tot;
    __syncthreads();
    for (int k = warp; k < NV; k += TILE / 32) {
        double x = (sm[k][lane] + sm[k][lane + 32]) + (sm[k][lane + 64] + sm[k][lane + 96]);
        for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
        if (lane == 0) so[k] = x;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) out[k] = so[k];
    __syncthreads();
}

// The launch's totals of the blocks' NV values v (deterministic: the last block
// to arrive adds the blocks' values in a fixed order).  True in that block,
// whose threads then hold the totals.
template <int NV>
__device__ __forceinline__ bool launch_totals(double (&v)[NV], double *partials, unsigned int *counter)
{
    __shared__ bool is_last;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) partials[(int64_t)blockIdx.x * NV + k] = v[k];
        __threadfence();
        is_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!is_last) return false;
    __threadfence();
    Sum64<double> s[NV];
    for (int i = threadIdx.x; i < (int)gridDim.x; i += 4 * TILE) {
        double x[4][NV];  // four blocks' values in flight a thread
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int k = 0; k < NV; ++k)
                x[q][k] = i + q * TILE < (int)gridDim.x ? __ldcg(&partials[(int64_t)(i + q * TILE) * NV + k]) : 0.0;
#pragma unroll
        for (int k = 0; k < NV; ++k) s[k].add((x[0][k] + x[1][k]) + (x[2][k] + x[3][k]));
    }
    block_totals<NV>(s, v);
    if (threadIdx.x == 0) *counter = 0u;
    return true;
}

template <typename R, typename CT, int NP, bool FX = true>
__global__ void GPE_TILE_BOUNDS(R, NP) k_itp_a(const ItpArgs<R, CT> a, const TileView T)
{
    const R q4 = a.dt / (R)4;
    using LAP = LapIn<LapEuler, FX>;
    const auto co = tile_co<NP, LAP>(euler_coef(a.ihx2, q4), euler_coef(a.ihy2, q4), euler_coef(a.ihz2, q4));  // before the wait
    const TileList list = tile_begin(T);
    const TileDiag<R, CT> diag{{(R)a.scalars[0], a.g * a.dt / (R)2, a.E}};
    tile_loop<NP, LAP>(T, list, (const CT *)a.psi, diag, co, EveryTile(),
                  [&](uint32_t idx, uint32_t n) { prefetch_l2(a.E + idx, n * (uint32_t)sizeof(R)); }, ELoad<R>{a.E},
                  [&](uint32_t idx, const typename ELoad<R>::P &p, const CT(&c)[4], const CT(&L)[4]) {
                      CT o[4];
#pragma unroll
                      for (int i = 0; i < 4; ++i) {
                          // E < 0 marks an inactive cell of a stored segment
                          o[i] = active_e(p.e[i]) ? euler(c[i], q4, L[i]) : czero<CT>();
                      }
                      st4(a.tmp + idx, o);
                  });
}

template <typename R, typename CT, int NP, bool FX = true>
__global__ void GPE_TILE_BOUNDS(R, NP) k_itp_b(const ItpArgs<R, CT> a, const TileView T, double *partials,
                                           unsigned int *counter)
{
    const R q4 = a.dt / (R)4;
    using LAP = LapIn<LapEuler, FX>;
    const auto co = tile_co<NP, LAP>(euler_coef(a.ihx2, q4), euler_coef(a.ihy2, q4), euler_coef(a.ihz2, q4));  // before the wait
    const TileList list = tile_begin(T);
    const R hg = a.g * a.dt / (R)2;
    Sum64<R> norm[1];
    int n = 0;
    tile_loop<NP, LAP>(T, list, (const CT *)a.tmp, Plain(), co, EveryTile(),
                  [&](uint32_t idx, uint32_t n) { prefetch_l2(a.E + idx, n * (uint32_t)sizeof(R)); }, ELoad<R>{a.E},
                  [&](uint32_t idx, const typename ELoad<R>::P &p, const CT(&c)[4], const CT(&L)[4]) {
                      CT o[4];
                      R n4 = (R)0;  // the segment's |psi|^2, added to the FP64 sum once
#pragma unroll
                      for (int i = 0; i < 4; ++i) {
                          o[i] = euler(c[i], q4, L[i]);
                          const R f = active_e(p.e[i]) ? p.e[i] * ((R)1 - hg * norm2(o[i])) : (R)0;
                          o[i] = scale(o[i], f);
                          n4 = add_rn(n4, norm2(o[i]));
                      }
                      st4(a.psi + idx, o);
                      norm[0].add(n4);
                      keep<1>(norm, ++n);
                  });
    double tot[1];
    block_totals<1>(norm, tot);
    if (launch_totals<1>(tot, partials, counter) && threadIdx.x == 0) {
        const double nrm = tot[0] * a.dV;
        a.scalars[0] = sqrt(a.N / nrm);
        a.scalars[1] = nrm;
    }
}

// the pending renormalisation applied at the end of a call, rounded exactly as
// the next step's load would apply it (factor in the state's precision), so
// that a run split across calls or resumed from a dump is bit-identical
template <typename CT>
__global__ void k_apply_scale(CT *psi, int64_t n, const double *scalars)
{
    const auto sc = (typename RealOf<CT>::T)scalars[0];
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        psi[s] = scale(psi[s], sc);
    }
}

// ------------------------------------------------------------ observables
template <typename R, typename CT = typename Cx<R>::T>
struct ObsArgs {
    const CT *psi;
    const R *V0;
    const R *V1;
    R s;
    R ihx2, ihy2, ihz2, g;
    double dV;
    double *partials;
    unsigned int *counter;
    gpe_obs *out;
};

// a segment's potential(s), loaded ahead of its terms
template <typename R, bool BLEND>
struct VLoad {
    const R *V0, *V1;
    struct P {
        R V0[4], V1[BLEND ? 4 : 1];
    };
    __device__ __forceinline__ P operator()(uint32_t idx) const
    {
        P p;
        ldr4(V0 + idx, p.V0);
        if constexpr (BLEND) ldr4(V1 + idx, p.V1);
        return p;
    }
};

__device__ __forceinline__ bool finite1(float v) { return (__float_as_uint(v) & 0x7f800000u) != 0x7f800000u; }
__device__ __forceinline__ bool finite1(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }
template <typename CT>
__device__ __forceinline__ bool finite_v(const CT &v)
{
    if constexpr (is_cplx<CT>())
        return finite1(v.x) && finite1(v.y);
    else
        return finite1(v);
}

// What a segment adds to the observables: norm, ekin, epot, eint, summed over
// its four cells in the state precision, then added to the FP64 sums once; and
// its non-finite cells.
template <bool BLEND, typename R, typename CT>
__device__ __forceinline__ void obs_terms(const typename VLoad<R, BLEND>::P &p, R s, R g, const CT (&c)[4],
                                          const CT (&L)[4], R (&t)[4], int &nf)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) t[k] = (R)0;
    bool fin = true;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool act = active_v(p.V0[i]);
        R V = p.V0[i];
        if constexpr (BLEND) V = ((R)1 - s) * p.V0[i] + s * p.V1[i];
        const R rho = act ? norm2(c[i]) : (R)0;
        t[0] = add_rn(t[0], rho);
        t[1] = add_rn(t[1], act ? (R)(-0.5) * dotre(c[i], L[i]) : (R)0);
        t[2] = add_rn(t[2], act ? V * rho : (R)0);
        t[3] = add_rn(t[3], (R)0.5 * g * rho * rho);
        fin = fin && (!act || finite_v(c[i]));
    }
    if (!fin) {
#pragma unroll
        for (int i = 0; i < 4; ++i) nf += active_v(p.V0[i]) && !finite_v(c[i]) ? 1 : 0;
    }
}

// 512^3 shell, complex64: 80 us warp by brick with ten FP64 instructions a
// segment, 66 on tiles with the sums flushed by every warp at its end, 40 now;
// one pass over psi and V at 3.7 TB/s, the shared-memory pipe 76 % busy.
template <typename R, typename CT, int NP, bool BLEND>
__global__ void GPE_TILE_BOUNDS(R, NP) k_obs(const ObsArgs<R, CT> a, const TileView T)
{
    const auto co = tile_co<NP, LapFull>(a.ihx2, a.ihy2, a.ihz2);  // before the wait
    const TileList list = tile_begin(T);
    Sum64<R> sum[5];  // norm, ekin, epot, eint, nonfinite
    int n = 0, nf = 0;
    tile_loop<NP>(T, list, a.psi, Plain(), co, EveryTile(),
                  [&](uint32_t idx, uint32_t n) {
                      prefetch_l2(a.V0 + idx, n * (uint32_t)sizeof(R));
                      if constexpr (BLEND) prefetch_l2(a.V1 + idx, n * (uint32_t)sizeof(R));
                  },
                  VLoad<R, BLEND>{a.V0, a.V1},
                  [&](uint32_t, const typename VLoad<R, BLEND>::P &p, const CT(&c)[4], const CT(&L)[4]) {
                      R t[4];
                      obs_terms<BLEND>(p, a.s, a.g, c, L, t, nf);
#pragma unroll
                      for (int k = 0; k < 4; ++k) sum[k].add(t[k]);
                      keep<4>(sum, ++n);
                  });
    sum[4].add((R)nf);
    double tot[5];
    block_totals<5>(sum, tot);
    if (launch_totals<5>(tot, a.partials, a.counter) && threadIdx.x == 0) {
        gpe_obs o;
        o.norm = tot[0] * a.dV;
        o.e_kin = tot[1] * a.dV;
        o.e_pot = tot[2] * a.dV;
        o.e_int = tot[3] * a.dV;
        o.energy = o.e_kin + o.e_pot + o.e_int;
        o.mu = (o.e_kin + o.e_pot + 2.0 * o.e_int) / o.norm;
        o.nonfinite = tot[4];
        *a.out = o;
    }
}

// ------------------------------------------------------------ drivers
__global__ inline void k_set_one(double *p) { *p = 1.0; }

// arguments of the imaginary-time passes of a state; makes the propagator
// table if dt or the potential changed, and sets the pending factor to 1
template <typename R, typename CT>
inline int itp_args(gpe_state *st, const gpe_imag_params *p, cudaStream_t s, ItpArgs<R, CT> &a)
{
    const gpe_grid *g = st->grid;
    if (st->E_dt != p->dt || st->E_version != g->v0_version) {
        k_make_E<R><<<g->nsm * 8, 256, 0, s>>>(g->d_V[0], (R *)st->d_E, g->n_packed, p->dt);
        GPE_LAUNCH_CHECK();
        st->E_dt = p->dt;
        st->E_version = g->v0_version;
    }
    a = ItpArgs<R, CT>{};
    a.psi = (CT *)st->d_psi;
    a.tmp = (CT *)st->d_work[0];
    a.E = (const R *)st->d_E;
    a.ihx2 = (R)(1.0 / (g->box.hx * g->box.hx));
    a.ihy2 = (R)(1.0 / (g->box.hy * g->box.hy));
    a.ihz2 = (R)(1.0 / (g->box.hz * g->box.hz));
    a.g = (R)p->g;
    a.dt = (R)p->dt;
    a.scalars = st->red.scalars;
    a.N = p->N;
    a.dV = g->box.hx * g->box.hy * g->box.hz;
    k_set_one<<<1, 1, 0, s>>>(st->red.scalars);
    GPE_LAUNCH_CHECK();
    return GPE_OK;
}

// cnt imaginary-time steps of two staged passes
template <typename R, typename CT, int NP>
inline int itp_steps(gpe_state *st, const ItpArgs<R, CT> &a, int64_t cnt, cudaStream_t s)
{
    const gpe_grid *g = st->grid;
    const TileLaunch L = tile_launch<CT, NP>(g->tiles);
    constexpr bool F = !two_forms<R, NP>();
    const bool fixed = fixed_spacings(g->box);
    auto ka = fixed ? k_itp_a<R, CT, NP> : k_itp_a<R, CT, NP, F>;
    auto kb = fixed ? k_itp_b<R, CT, NP> : k_itp_b<R, CT, NP, F>;
    const unsigned na = tile_blocks(ka, g->nsm, L.T.ntiles, L.smem), nb = tile_blocks(kb, g->nsm, L.T.ntiles, L.smem);
    for (int64_t n = 0; n < cnt; ++n) {
        GPE_TRY(tile_run(ka, na, L, s, a, L.T));
        GPE_TRY(tile_run(kb, nb, L, s, a, L.T, st->red.partials, st->red.counter));
    }
    return GPE_OK;
}

template <typename CT>
inline int itp_end(gpe_state *st, cudaStream_t s)
{
    const gpe_grid *g = st->grid;
    k_apply_scale<CT><<<g->nsm * 8, 256, 0, s>>>((CT *)st->d_psi, g->n_packed, st->red.scalars);
    GPE_LAUNCH_CHECK();
    return GPE_OK;
}

template <typename R, typename CT, int NP>
inline int obs_run(const gpe_state *stc, double gg, double sb, cudaStream_t s)
{
    gpe_state *st = const_cast<gpe_state *>(stc);
    const gpe_grid *g = st->grid;
    ObsArgs<R, CT> a{};
    a.psi = (const CT *)st->d_psi;
    a.V0 = (const R *)potential_ptr(st, 0);
    a.V1 = (sb != 0.0) ? (const R *)potential_ptr(st, 1) : nullptr;
    if (sb != 0.0 && !a.V1) return fail(GPE_ERR_ARG, "s_blend != 0 needs potential slot 1");
    a.s = (R)sb;
    a.ihx2 = (R)(1.0 / (g->box.hx * g->box.hx));
    a.ihy2 = (R)(1.0 / (g->box.hy * g->box.hy));
    a.ihz2 = (R)(1.0 / (g->box.hz * g->box.hz));
    a.g = (R)gg;
    a.dV = g->box.hx * g->box.hy * g->box.hz;
    a.partials = st->red.partials;
    a.counter = st->red.counter;
    a.out = (gpe_obs *)(st->red.scalars + 2);
    const TileLaunch L = tile_launch<CT, NP>(g->tiles);
    auto k = a.V1 ? k_obs<R, CT, NP, true> : k_obs<R, CT, NP, false>;
    return tile_run(k, tile_blocks(k, g->nsm, L.T.ntiles, L.smem), L, s, a, L.T);
}

// The schedule's values for n steps of nc stages, at *clock + (n0 + m) dt +
// c[k] dt, then the clock moved on by `advance`: one block.  Every thread of a
// stage kernel used to evaluate its own (21 FP64 instructions with a division,
// 24 warps an SM queueing for the FP64 pipe: 4.7 of 39 us of a 512^3 stage).
struct StageTimes {
    double c[6];
};
static __global__ void k_ramp_table(Ramp r, double *clock, double advance, int64_t n0, int n, int nc, StageTimes c,
                                    double dt, double *tab)
{
    const double t = *clock;
    __syncthreads();
    for (int i = threadIdx.x; i < n * nc; i += blockDim.x)
        tab[i] = ramp_s(r, t + (double)(n0 + i / nc) * dt + c.c[i % nc] * dt);
    if (threadIdx.x == 0 && advance != 0.0) *clock = t + advance;
}
constexpr StageTimes RK4_TIMES = {{0.0, 0.5, 1.0}};
constexpr int STAB_STEPS = 256;  // steps a table is made for at a time
constexpr int GRAPH_STEPS_MAX = 4096;  // steps of a graph at most, and then a table's

// arguments of the RK4 stages of a state (ramps: the clock is set to t0)
template <typename R>
inline int rk4_args(gpe_state *st, const gpe_real_params *p, RkArgs<R> &a)
{
    using CT = typename Cx<R>::T;
    const gpe_grid *g = st->grid;
    const bool blend = p->potential == GPE_V_BLEND;
    a = RkArgs<R>{};
    a.V0 = (const R *)potential_ptr(st, 0);
    a.V1 = blend ? (const R *)potential_ptr(st, 1) : nullptr;
    if (!a.V0 || (blend && !a.V1)) return fail(GPE_ERR_STATE, "potential slot missing");
    a.y0 = (CT *)st->d_psi;
    a.y2 = (CT *)st->d_work[0];
    a.y3 = (CT *)st->d_work[1];
    a.y4 = (CT *)st->d_work[0];  // y2 is dead once stage 1 is done
    a.w = (CT *)st->d_work[2];
    a.ihx2 = (R)(1.0 / (g->box.hx * g->box.hx));
    a.ihy2 = (R)(1.0 / (g->box.hy * g->box.hy));
    a.ihz2 = (R)(1.0 / (g->box.hz * g->box.hz));
    a.g = (R)p->g;
    a.dt = (R)p->dt;
    a.dtd = p->dt;
    a.ramp.clock = st->d_clock;
    a.ramp.T = p->T_ramp;
    a.ramp.n_knots = p->n_knots;
    for (int k = 0; k < GPE_MAX_KNOTS; ++k) a.ramp.knots[k] = p->knots[k];
    return GPE_OK;
}

// cnt RK4 steps of four staged passes, stage times relative to the clock, which
// is then moved on if `advance`; a ramp needs ensure_stab before
template <typename R, int NP>
inline int rk4_steps(gpe_state *st, RkArgs<R> a, bool blend, int64_t cnt, bool advance, cudaStream_t s)
{
    const gpe_grid *g = st->grid;
    using RT = Rk4Tiles<R, NP>;
    const TileLaunch L = tile_launch<typename Cx<R>::T, NP>(g->tiles);
    const bool fixed = fixed_spacings(g->box);
    unsigned grid[4];
    for (int stg = 0; stg < 4; ++stg) grid[stg] = tile_blocks(RT::get(blend, stg, fixed), g->nsm, L.T.ntiles, L.smem);
    for (int64_t n = 0; n < cnt; ++n) {
        const int m = blend ? (int)(n % st->stab_cap) : 0;
        if (blend && m == 0) {
            const int64_t left = cnt - n;
            const int here = (int)(left < st->stab_cap ? left : st->stab_cap);
            k_ramp_table<<<1, 256, 0, s>>>(a.ramp, st->d_clock, advance && here == left ? (double)cnt * a.dtd : 0.0, n,
                                           here, 3, RK4_TIMES, a.dtd, st->d_stab);
            GPE_LAUNCH_CHECK();
        }
        for (int stg = 0; stg < 4; ++stg) {
            a.stab = st->d_stab + 3 * m + (stg + 1) / 2;  // t, t + dt/2 twice, t + dt
            GPE_TRY(tile_run(RT::get(blend, stg, fixed), grid[stg], L, s, a, L.T));
        }
    }
    return GPE_OK;
}

}  // namespace gpe
