// step19.cu -- the step drivers of 19-point grids (App. B's higher-order
// compact Laplacian): RK4 (stages of App. A), imaginary time and the
// observables, staged schedule, one launch per stage.  A separate
// translation unit so that the 19-point kernel instances build in parallel
// with the 7-point ones.
#include "kernels.cuh"

namespace gpe {

namespace {

__global__ void k_set_scalar19(double *p, double v) { *p = v; }

template <typename R>
int rk4_19(gpe_state *st, const gpe_real_params *p, int64_t nsteps, double t0, cudaStream_t s)
{
    const bool blend = p->potential == GPE_V_BLEND;
    RkArgs<R> a;
    GPE_TRY(rk4_args(st, p, a));
    if (blend) {
        GPE_TRY(ensure_stab(st, STAB_STEPS));
        k_set_scalar19<<<1, 1, 0, s>>>(st->d_clock, t0);
        GPE_LAUNCH_CHECK();
    }
    return rk4_steps<R, 19>(st, a, blend, nsteps, false, s);
}

template <typename R, typename CT>
int itp_19(gpe_state *st, const gpe_imag_params *p, int64_t nsteps, cudaStream_t s)
{
    ItpArgs<R, CT> a;
    GPE_TRY(itp_args(st, p, s, a));
    const int rc = itp_steps<R, CT, 19>(st, a, nsteps, s);
    return rc != GPE_OK ? rc : itp_end<CT>(st, s);
}

}  // namespace

int rk4_run19(gpe_state *st, const gpe_real_params *p, int64_t nsteps, double t0, cudaStream_t s)
{
    return st->dtype == GPE_C128 ? rk4_19<double>(st, p, nsteps, t0, s) : rk4_19<float>(st, p, nsteps, t0, s);
}

int itp_run19(gpe_state *st, const gpe_imag_params *p, int64_t nsteps, cudaStream_t s)
{
    switch (st->dtype) {
    case GPE_C128: return itp_19<double, double2>(st, p, nsteps, s);
    case GPE_C64: return itp_19<float, float2>(st, p, nsteps, s);
    case GPE_R64: return itp_19<double, double>(st, p, nsteps, s);
    default: return itp_19<float, float>(st, p, nsteps, s);
    }
}

int obs_run19(const gpe_state *st, double g, double s_blend, cudaStream_t s)
{
    switch (st->dtype) {
    case GPE_C128: return obs_run<double, double2, 19>(st, g, s_blend, s);
    case GPE_C64: return obs_run<float, float2, 19>(st, g, s_blend, s);
    case GPE_R64: return obs_run<double, double, 19>(st, g, s_blend, s);
    default: return obs_run<float, float, 19>(st, g, s_blend, s);
    }
}

}  // namespace gpe
