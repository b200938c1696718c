// batch.cu -- many independent shells in one persistent launch: imaginary-time
// ground-state solves (Sec. II A, Eqs. (6)-(7), iterated to a tolerance as in
// Sec. III) for a batch of states whose grids differ in size and shape.  The
// states are complex or, since the imaginary-time step keeps a real
// wavefunction real, real (half the bytes).
//
// The batch concatenates the shells' tiles and packed arrays into one layout
// (each shell starts on a tile), so one launch of each kernel covers every
// shell.  Per-shell parameters (g, dt, N, spacings, the pending
// renormalisation factor, mu and the convergence flag) live in a device table.
// Norms and observables are reduced per block and shell, then per shell in
// block order (deterministic).  Converged shells are skipped tile by tile.  Each block
// of `check_every` steps plus the convergence test is captured once in a CUDA
// graph and replayed; the host polls the number of unconverged shells between
// replays.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "gpe_internal.cuh"
#include "kernels.cuh"
#include "stencil.cuh"

namespace gpe {

struct ShellParams {
    double g, dt, N, dV;
    double ihx2, ihy2, ihz2;
    double scale;     // pending renormalisation factor (applied by the next stage A)
    double mu, mu_prev, energy, norm, e_kin, e_pot, e_int, nonfinite;
    double tol;
    long long steps;  // steps taken
    int converged;
    int has_prev;
};

template <typename R, typename CT = typename Cx<R>::T>
struct BatchArgs {
    CT *psi;
    CT *tmp;
    const R *E;       // exp(-V dt_s/2) per shell, -1 on inactive cells of stored segments
    const R *V;       // potential (for observables), +inf on inactive cells
    ShellParams *sh;
    const uint32_t *tile_shell;  // per tile its shell
    const uint32_t *tile_base;   // [n+1] first tile of each shell
    double *part;     // [ntiles*5] per-block partial sums, see part_of
};

// A kernel's blocks take the tiles blockIdx.x + k gridDim.x, so the blocks
// that meet shell s are those whose offset from its first tile, modulo the
// grid, is below its tile count; each leaves one partial sum per quantity, at
// that offset from the shell's first tile.
__device__ __forceinline__ uint32_t part_of(uint32_t base, uint32_t block, uint32_t grid)
{
    return base + (block + grid - base % grid) % grid;
}
__device__ __forceinline__ uint32_t parts_of(uint32_t base, uint32_t end, uint32_t grid)
{
    return min(end - base, grid);
}

// What a block keeps of the shell whose tiles it is walking through (tiles of
// one shell are consecutive): its parameters, and the sums to leave behind
// when the shell changes.  The next tile's shell is fetched a tile ahead.
template <typename R, typename CT, int NS>
struct ShellWalk {
    const BatchArgs<R, CT> &a;
    uint32_t nt;
    uint32_t cur = 0xffffffffu, next = 0;
    bool live = false;
    R g = 0, dt = 0, scale = 0;
    TileCo<R> co{};  // of euler_coef of the spacings, but for the observables
    Sum64<R> sum[NS > 0 ? NS : 1];  // NS 5: the fifth counts non-finite cells
    int nf = 0, n = 0;
    __device__ __forceinline__ ShellWalk(const BatchArgs<R, CT> &a_, uint32_t nt_) : a(a_), nt(nt_)
    {
        if (blockIdx.x < nt) next = __ldg(a.tile_shell + blockIdx.x);
    }
    // the block's sums of the shell just left, to their place
    __device__ __forceinline__ void leave()
    {
        if constexpr (NS > 0) {
            if (!live) return;
            double *p = a.part + 5 * (size_t)part_of(a.tile_base[cur], blockIdx.x, gridDim.x), tot[NS];
            if constexpr (NS == 5) sum[4].add((R)nf);
            block_totals<NS>(sum, tot);
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                if (threadIdx.x == 0) p[k] = tot[k];
                sum[k] = Sum64<R>();
            }
            nf = 0;
            n = 0;
        }
    }
    // called before each tile; false: a converged shell, skip it
    __device__ __forceinline__ bool enter(uint32_t tile)
    {
        const uint32_t s = next;
        if (tile + gridDim.x < nt) next = __ldg(a.tile_shell + tile + gridDim.x);
        if (s != cur) {
            leave();
            cur = s;
            const ShellParams &P = a.sh[s];
            live = !P.converged;
            g = (R)P.g;
            dt = (R)P.dt;
            const R q = NS == 5 ? (R)1 : dt / (R)4;
            co = tile_co<7, LapFull>(euler_coef((R)P.ihx2, q), euler_coef((R)P.ihy2, q), euler_coef((R)P.ihz2, q));
            scale = (R)P.scale;
        }
        return live;
    }
    __device__ __forceinline__ void added() { keep<(NS == 5 ? 4 : NS)>(sum, ++n); }
};

// the diagonal half step at the load, with the current shell's parameters
template <typename R, typename CT, typename W>
struct WalkDiag {
    const W &w;
    const R *E;
    using D = TileDiag<R, CT>;
    using P4 = typename D::P4;
    using P1 = typename D::P1;
    __device__ __forceinline__ D diag() const { return D{{w.scale, w.g * w.dt / (R)2, E}}; }
    __device__ __forceinline__ P4 load4(uint32_t idx) const { return diag().load4(idx); }
    __device__ __forceinline__ P1 load1(uint32_t idx) const { return diag().load1(idx); }
    __device__ __forceinline__ void seg(CT (&v)[4], const P4 &p) const { diag().seg(v, p); }
    __device__ __forceinline__ void own(CT (&v)[4], const typename ELoad<R>::P &p) const { diag().own(v, p); }
    __device__ __forceinline__ void cell(CT &v, const P1 &e) const { diag().cell(v, e); }
};

// CT: complex (float2 / double2) or real (float / double) values; a real
// state stays real under the imaginary-time step.  Eight shells (9.8e7 active
// cells), complex64, 20 steps and the check: 33.5 -> 24.3 ms against a warp
// per brick and one FP64 warp sum per brick; bound by the shared-memory pipe
// like the single-state passes.
template <typename R, typename CT, int STAGE>
__global__ void GPE_TILE_BOUNDS(R, 7) k_batch_itp(const BatchArgs<R, CT> a, const TileView T)
{
    const TileList list = tile_begin(T);
    using W = ShellWalk<R, CT, STAGE>;
    W w(a, (uint32_t)T.ntiles);
    auto enter = [&](uint32_t tile) { return w.enter(tile); };
    auto pref = [&](uint32_t idx, uint32_t n) { prefetch_l2(a.E + idx, n * (uint32_t)sizeof(R)); };
    // E of each segment is loaded with the tile
    auto body = [&](uint32_t idx, const typename ELoad<R>::P &p, const CT(&c)[4], const CT(&L)[4]) {
        const R(&E)[4] = p.e;
        const R q4 = w.dt / (R)4, hg = w.g * w.dt / (R)2;
        CT o[4];
        R n4 = (R)0;  // the segment's |psi|^2, added to the FP64 sum once
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool act = active_e(E[i]);
            o[i] = euler(c[i], q4, L[i]);
            if (STAGE == 1) {
                const R f = act ? E[i] * ((R)1 - hg * norm2(o[i])) : (R)0;
                o[i] = scale(o[i], f);
                n4 = add_rn(n4, norm2(o[i]));
            } else if (!act) {
                o[i] = czero<CT>();
            }
        }
        st4((STAGE == 0 ? a.tmp : a.psi) + idx, o);
        if constexpr (STAGE == 1) {
            w.sum[0].add(n4);
            w.added();
        }
    };
    if constexpr (STAGE == 0)
        tile_loop<7, LapEuler>(T, list, (const CT *)a.psi, WalkDiag<R, CT, W>{w, a.E}, w.co, enter, pref,
                     ELoad<R>{a.E}, body);
    else
        tile_loop<7, LapEuler>(T, list, (const CT *)a.tmp, Plain(), w.co, enter, pref, ELoad<R>{a.E}, body);
    w.leave();
}

// per shell: norm from the blocks' partials (in order), next factor; grid:
// the blocks of the launch that left them
__global__ void k_batch_norm_finish(ShellParams *sh, const double *part, const uint32_t *tile_base, uint32_t grid)
{
    const int s = blockIdx.x;
    if (sh[s].converged) return;
    const uint32_t b0 = tile_base[s], n = parts_of(b0, tile_base[s + 1], grid);
    double x = 0.0;
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) x += part[(size_t)(b0 + i) * 5];
    x = block_sum(x);
    if (threadIdx.x == 0) {
        const double nrm = x * sh[s].dV;
        sh[s].norm = nrm;
        sh[s].scale = sqrt(sh[s].N / nrm);
        sh[s].steps += 1;
    }
}

// apply each shell's pending factor to its cells (rounded to the state's
// precision, as the next load would apply it), then reset it to 1
template <typename CT>
__global__ void k_batch_apply_scale(CT *psi, const uint32_t *tile_shell, const ShellParams *sh, uint32_t ntiles)
{
    for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const auto sc = (typename RealOf<CT>::T)sh[tile_shell[t]].scale;
        CT *p = psi + 4 * (size_t)t * TILE;
        for (int i = threadIdx.x; i < 4 * TILE; i += blockDim.x) p[i] = scale(p[i], sc);
    }
}

__global__ void k_batch_reset_scale(ShellParams *sh, int n)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < n) sh[s].scale = 1.0;
}

template <typename R, typename CT>
__global__ void GPE_TILE_BOUNDS(R, 7) k_batch_obs(const BatchArgs<R, CT> a, const TileView T)
{
    const TileList list = tile_begin(T);
    ShellWalk<R, CT, 5> w(a, (uint32_t)T.ntiles);
    tile_loop<7>(T, list, (const CT *)a.psi, Plain(), w.co, [&](uint32_t tile) { return w.enter(tile); },
                 [&](uint32_t idx, uint32_t n) { prefetch_l2(a.V + idx, n * (uint32_t)sizeof(R)); },
                 VLoad<R, false>{a.V, nullptr},
                 [&](uint32_t, const typename VLoad<R, false>::P &p, const CT(&c)[4], const CT(&L)[4]) {
                     R t[4];
                     obs_terms<false>(p, (R)0, w.g, c, L, t, w.nf);
#pragma unroll
                     for (int k = 0; k < 4; ++k) w.sum[k].add(t[k]);
                     w.added();
                 });
    w.leave();
}

// per shell: observables from the blocks' partials, then the convergence test
// |mu - mu_prev| < tol against the previous check
__global__ void k_batch_obs_finish(ShellParams *sh, const double *part, const uint32_t *tile_base, uint32_t grid,
                                   int *n_unconverged)
{
    const int s = blockIdx.x;
    if (sh[s].converged) return;
    const uint32_t b0 = tile_base[s], n = parts_of(b0, tile_base[s + 1], grid);
    double t[5];
    for (int k = 0; k < 5; ++k) {
        double x = 0.0;
        for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) x += part[(size_t)(b0 + i) * 5 + k];
        t[k] = block_sum(x);
    }
    if (threadIdx.x == 0) {
        ShellParams &P = sh[s];
        P.norm = t[0] * P.dV;
        P.e_kin = t[1] * P.dV;
        P.e_pot = t[2] * P.dV;
        P.e_int = t[3] * P.dV;
        P.nonfinite = t[4];
        P.energy = P.e_kin + P.e_pot + P.e_int;
        P.mu = (P.e_kin + P.e_pot + 2.0 * P.e_int) / P.norm;
        if (P.has_prev && fabs(P.mu - P.mu_prev) < P.tol) P.converged = 1;
        if (P.nonfinite > 0) P.converged = 1;  // stop a shell that blew up
        P.mu_prev = P.mu;
        P.has_prev = 1;
        if (!P.converged) atomicAdd(n_unconverged, 1);
    }
}

__global__ void k_zero_int(int *p) { *p = 0; }

template <typename R>
__global__ void k_batch_make_E(const double *V, R *E, const uint32_t *tile_shell, const ShellParams *sh, uint32_t ntiles)
{
    for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const double dt = sh[tile_shell[t]].dt;
        for (int i = threadIdx.x; i < 4 * TILE; i += blockDim.x) {
            const size_t c = 4 * (size_t)t * TILE + i;
            const double v = V[c];
            E[c] = v < INFINITY ? (R)exp(-v * dt / 2.0) : (R)-1;
        }
    }
}

template <typename R>
__global__ void k_d2r(const double *s, R *d, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        d[i] = (R)s[i];
}

// One shell's part of the batch's tables: its grid's neighbour slots as they
// are (slots are relative to the tile), its halo rows with the segment numbers
// shifted to the batch's, the padding to a whole tile inactive (V = +inf, no
// neighbours).
__global__ void k_batch_tables(TileTab t, uint32_t tile0, uint32_t shell, int stride, uint2 *nbr, uint32_t *halo,
                               uint32_t *tile_shell, const double *V0, double *V)
{
    const uint32_t seg0 = tile0 * TILE, npad = (uint32_t)t.ntiles * TILE;
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = i0; i < t.ntiles; i += step) tile_shell[tile0 + i] = shell;
    constexpr uint32_t Z = TILE | TILE << 10 | TILE << 20;  // three zero slots
    for (int64_t i = i0; i < npad; i += step) nbr[seg0 + i] = i < t.nseg ? t.d_nbr[i] : make_uint2(Z, Z);
    for (int64_t i = i0; i < 4 * (int64_t)npad; i += step)
        V[4 * (int64_t)seg0 + i] = i < 4 * (int64_t)t.nseg ? V0[i] : (double)INFINITY;
    for (int64_t i = i0; i < (int64_t)t.ntiles * t.stride; i += step) {
        const int64_t tile = i / t.stride;
        const int j = (int)(i % t.stride);
        const uint32_t *row = t.d_halo + tile * t.stride;
        const int whole = row[0] & 0xffff, single = row[0] >> 16;
        uint32_t *out = halo + (tile0 + tile) * (int64_t)stride;
        if (j == 0) out[0] = row[0];
        else if (j <= whole) out[j] = row[j] + seg0;
        else if (j >= t.stride - single) out[stride - (t.stride - j)] = row[j] + seg0;  // bit 31 is above any segment
    }
}

}  // namespace gpe

using namespace gpe;

struct gpe_batch {
    int n = 0;
    int dtype = 0, shape = 0, device = 0, nsm = 0;
    size_t elem = 0;   // bytes per value of the state type
    size_t relem = 0;  // bytes per real of its precision (E and V tables)
    std::vector<gpe_state *> states;
    std::vector<int64_t> packed_base;  // first cell of each shell, a whole number of tiles
    std::vector<uint32_t> tile_base;
    int64_t np = 0;
    TileTab tiles;
    uint32_t *d_tile_shell = nullptr, *d_tile_base = nullptr;
    void *d_psi = nullptr, *d_tmp = nullptr, *d_E = nullptr, *d_Vr = nullptr;
    double *d_V = nullptr;
    ShellParams *d_sh = nullptr;
    double *d_part = nullptr;
    int *d_unconv = nullptr;
    int *h_unconv = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaStream_t cap = nullptr;
    uint64_t key = 0;
};

static void batch_free(gpe_batch *B)
{
    if (!B) return;
    if (B->exec) cudaGraphExecDestroy(B->exec);
    if (B->cap) cudaStreamDestroy(B->cap);
    tiles_free(B->tiles);
    dev_free(B->d_tile_shell);
    dev_free(B->d_tile_base);
    dev_free(B->d_psi);
    dev_free(B->d_tmp);
    dev_free(B->d_E);
    dev_free(B->d_Vr);
    dev_free(B->d_V);
    dev_free(B->d_sh);
    dev_free(B->d_part);
    dev_free(B->d_unconv);
    if (B->h_unconv) cudaFreeHost(B->h_unconv);
    delete B;
}

extern "C" int gpe_batch_create(gpe_state *const *states, int n, gpe_batch **out)
{
    if (!states || !out || n < 1) return fail(GPE_ERR_ARG, "need n >= 1 states and an output pointer");
    *out = nullptr;
    if (n > 1000000) return fail(GPE_ERR_ARG, "too many shells");
    for (int i = 0; i < n; ++i)
        if (!states[i]) return fail(GPE_ERR_ARG, "state %d is NULL", i);
    const int dtype = states[0]->dtype, shape = states[0]->grid->shape;
    for (int i = 1; i < n; ++i)
        if (states[i]->dtype != dtype || states[i]->grid->shape != shape)
            return fail(GPE_ERR_ARG, "batch states must share dtype and brick shape (state %d differs)", i);
    if (dtype != GPE_C128 && dtype != GPE_C64 && dtype != GPE_R64 && dtype != GPE_R32)
        return fail(GPE_ERR_ARG, "unknown state type %d", dtype);
    for (int i = 0; i < n; ++i)
        if (states[i]->grid->stencil != 7) return fail(GPE_ERR_ARG, "batches run the 7-point stencil (state %d)", i);
    gpe_batch *B = new gpe_batch();
    B->n = n;
    B->dtype = dtype;
    B->shape = shape;
    B->elem = states[0]->elem;
    B->relem = (dtype == GPE_C128 || dtype == GPE_R64) ? sizeof(double) : sizeof(float);
    B->states.assign(states, states + n);
    B->device = states[0]->grid->device;
    B->nsm = states[0]->grid->nsm;
    B->tile_base.resize(n + 1);
    B->packed_base.resize(n + 1);
    int64_t ntiles = 0;
    int nslot = TILE + 1, stride = 8;
    for (int i = 0; i < n; ++i) {
        const TileTab &t = states[i]->grid->tiles;
        B->tile_base[i] = (uint32_t)ntiles;
        B->packed_base[i] = 4 * TILE * ntiles;
        ntiles += t.ntiles;
        nslot = std::max(nslot, t.nslot);
        stride = std::max(stride, t.stride);
        if (4 * TILE * ntiles >= 0xffffffffLL) {
            batch_free(B);
            return fail(GPE_ERR_ARG, "batch too large for 32-bit packed offsets");
        }
    }
    B->tile_base[n] = (uint32_t)ntiles;
    B->packed_base[n] = B->np = 4 * TILE * ntiles;
    B->tiles.ntiles = (int)ntiles;
    B->tiles.nseg = (uint32_t)(TILE * ntiles);
    B->tiles.nslot = nslot;
    B->tiles.stride = stride;
    int rc = GPE_OK;
#define BT(x)                  \
    do {                       \
        rc = (x);              \
        if (rc != GPE_OK) {    \
            batch_free(B);     \
            return rc;         \
        }                      \
    } while (0)
    BT(dev_alloc_t(&B->tiles.d_nbr, (size_t)B->tiles.nseg));
    BT(dev_alloc_t(&B->tiles.d_halo, (size_t)ntiles * stride));
    BT(dev_alloc_t(&B->d_tile_shell, (size_t)ntiles));
    BT(dev_alloc_t(&B->d_tile_base, (size_t)n + 1));
    BT(dev_alloc(&B->d_psi, B->np * B->elem));
    BT(dev_alloc(&B->d_tmp, B->np * B->elem));
    BT(dev_alloc(&B->d_E, B->np * B->relem));
    BT(dev_alloc(&B->d_Vr, B->np * B->relem));
    BT(dev_alloc_t(&B->d_V, B->np));
    BT(dev_alloc_t(&B->d_sh, n));
    BT(dev_alloc_t(&B->d_part, (size_t)ntiles * 5));
    BT(dev_alloc_t(&B->d_unconv, 1));
    if (cudaMallocHost(&B->h_unconv, sizeof(int)) != cudaSuccess) BT(fail(GPE_ERR_CUDA, "cudaMallocHost failed"));
    // combined tables, from each grid's
    if (cudaMemcpy(B->d_tile_base, B->tile_base.data(), (n + 1) * sizeof(uint32_t), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(B->d_psi, 0, B->np * B->elem) != cudaSuccess || cudaMemset(B->d_tmp, 0, B->np * B->elem) != cudaSuccess)
        BT(fail(GPE_ERR_CUDA, "batch table upload failed"));
    for (int i = 0; i < n; ++i) {
        const gpe_grid *g = states[i]->grid;
        k_batch_tables<<<std::min(B->nsm * 8, g->tiles.ntiles), 256>>>(g->tiles, B->tile_base[i], (uint32_t)i, stride,
                                                                       B->tiles.d_nbr, B->tiles.d_halo,
                                                                       B->d_tile_shell, g->d_V[0], B->d_V);
        count_launch();
    }
    if (cudaGetLastError() != cudaSuccess) BT(fail(GPE_ERR_CUDA, "batch table kernel failed"));
    if (B->relem == sizeof(double)) k_d2r<double><<<B->nsm * 8, 256>>>(B->d_V, (double *)B->d_Vr, B->np);
    else k_d2r<float><<<B->nsm * 8, 256>>>(B->d_V, (float *)B->d_Vr, B->np);
    count_launch();
    if (cudaDeviceSynchronize() != cudaSuccess) BT(fail(GPE_ERR_CUDA, "batch setup kernel failed"));
#undef BT
    for (int i = 0; i < n; ++i) states[i]->grid->n_states++;  // the batch keeps the grids alive
    *out = B;
    return GPE_OK;
}

extern "C" int gpe_batch_destroy(gpe_batch *B)
{
    if (!B) return GPE_OK;
    cudaDeviceSynchronize();
    for (gpe_state *s : B->states) s->grid->n_states--;
    batch_free(B);
    return GPE_OK;
}

namespace gpe {

template <typename R, typename CT>
static int batch_record_block(gpe_batch *B, int64_t nsteps, cudaStream_t s)
{
    BatchArgs<R, CT> a;
    a.psi = (CT *)B->d_psi;
    a.tmp = (CT *)B->d_tmp;
    a.E = (const R *)B->d_E;
    a.V = (const R *)B->d_Vr;
    a.sh = B->d_sh;
    a.tile_shell = B->d_tile_shell;
    a.tile_base = B->d_tile_base;
    a.part = B->d_part;
    const TileLaunch L = tile_launch<CT, 7>(B->tiles);
    auto ka = k_batch_itp<R, CT, 0>;
    auto kb = k_batch_itp<R, CT, 1>;
    auto ko = k_batch_obs<R, CT>;
    const unsigned na = tile_blocks(ka, B->nsm, L.T.ntiles, L.smem), nb = tile_blocks(kb, B->nsm, L.T.ntiles, L.smem),
                   no = tile_blocks(ko, B->nsm, L.T.ntiles, L.smem);
    for (int64_t k = 0; k < nsteps; ++k) {
        GPE_TRY(tile_run(ka, na, L, s, a, L.T));
        GPE_TRY(tile_run(kb, nb, L, s, a, L.T));
        k_batch_norm_finish<<<B->n, 256, 0, s>>>(B->d_sh, B->d_part, B->d_tile_base, nb);
        GPE_LAUNCH_CHECK();
    }
    k_batch_apply_scale<CT><<<B->nsm * 8, 256, 0, s>>>((CT *)B->d_psi, B->d_tile_shell, B->d_sh, (uint32_t)L.T.ntiles);
    GPE_LAUNCH_CHECK();
    k_batch_reset_scale<<<(B->n + 255) / 256, 256, 0, s>>>(B->d_sh, B->n);
    GPE_LAUNCH_CHECK();
    k_zero_int<<<1, 1, 0, s>>>(B->d_unconv);
    GPE_LAUNCH_CHECK();
    GPE_TRY(tile_run(ko, no, L, s, a, L.T));
    k_batch_obs_finish<<<B->n, 256, 0, s>>>(B->d_sh, B->d_part, B->d_tile_base, no, B->d_unconv);
    GPE_LAUNCH_CHECK();
    return GPE_OK;
}

static int batch_record(gpe_batch *B, int64_t nsteps, cudaStream_t s)
{
    switch (B->dtype) {
    case GPE_C128: return batch_record_block<double, double2>(B, nsteps, s);
    case GPE_C64: return batch_record_block<float, float2>(B, nsteps, s);
    case GPE_R64: return batch_record_block<double, double>(B, nsteps, s);
    default: return batch_record_block<float, float>(B, nsteps, s);
    }
}

template <typename R>
static int batch_make_E(gpe_batch *B)
{
    k_batch_make_E<R><<<B->nsm * 8, 256>>>(B->d_V, (R *)B->d_E, B->d_tile_shell, B->d_sh, (uint32_t)B->tiles.ntiles);
    GPE_LAUNCH_CHECK();
    return GPE_OK;
}

}  // namespace gpe

extern "C" int gpe_batch_ground_state(gpe_batch *B, const gpe_imag_params *per_shell, double tol_dmu,
                                      int64_t check_every, int64_t max_steps, int32_t *converged, int64_t *steps,
                                      gpe_obs *obs, gpe_stream stream)
{
    if (!B || !per_shell) return fail(GPE_ERR_ARG, "NULL argument");
    if (check_every < 1 || max_steps < 1 || !(tol_dmu > 0))
        return fail(GPE_ERR_ARG, "need check_every >= 1, max_steps >= 1, tol_dmu > 0");
    int dev = -1;
    GPE_TRY_CUDA(cudaGetDevice(&dev));
    if (dev != B->device) return fail(GPE_ERR_STATE, "batch lives on device %d but device %d is current", B->device, dev);
    std::vector<ShellParams> sh(B->n);
    for (int i = 0; i < B->n; ++i) {
        const gpe_imag_params &p = per_shell[i];
        const gpe_box &b = B->states[i]->grid->box;
        if (!(p.dt > 0) || !(p.N > 0) || !std::isfinite(p.g) || !std::isfinite(p.dt) || !std::isfinite(p.N))
            return fail(GPE_ERR_ARG, "shell %d: need finite g, dt > 0, N > 0", i);
        const double lam = 2.0 / (b.hx * b.hx) + 2.0 / (b.hy * b.hy) + 2.0 / (b.hz * b.hz);
        if (p.dt * lam > 4.0) return fail(GPE_ERR_UNSTABLE, "shell %d: dt*lambda_max(T) = %.3g exceeds 4", i, p.dt * lam);
        ShellParams &P = sh[i];
        memset(&P, 0, sizeof P);
        P.g = p.g;
        P.dt = p.dt;
        P.N = p.N;
        P.dV = b.hx * b.hy * b.hz;
        P.ihx2 = 1.0 / (b.hx * b.hx);
        P.ihy2 = 1.0 / (b.hy * b.hy);
        P.ihz2 = 1.0 / (b.hz * b.hz);
        P.scale = 1.0;
        P.tol = tol_dmu;
    }
    cudaStream_t s = S(stream);
    GPE_TRY_CUDA(cudaMemcpyAsync(B->d_sh, sh.data(), B->n * sizeof(ShellParams), cudaMemcpyHostToDevice, s));
    for (int i = 0; i < B->n; ++i)
        GPE_TRY_CUDA(cudaMemcpyAsync((char *)B->d_psi + B->packed_base[i] * B->elem, B->states[i]->d_psi,
                                     B->states[i]->grid->n_packed * B->elem, cudaMemcpyDeviceToDevice, s));
    GPE_TRY_CUDA(cudaStreamSynchronize(s));
    GPE_TRY(B->relem == sizeof(double) ? batch_make_E<double>(B) : batch_make_E<float>(B));
    GPE_TRY_CUDA(cudaDeviceSynchronize());
    // one graph per (block length) replayed until every shell converged
    const uint64_t key = (uint64_t)check_every;
    if (!B->exec || B->key != key) {
        if (B->exec) {
            cudaGraphExecDestroy(B->exec);
            B->exec = nullptr;
        }
        if (!B->cap) GPE_TRY_CUDA(cudaStreamCreateWithFlags(&B->cap, cudaStreamNonBlocking));
        GPE_TRY_CUDA(cudaStreamBeginCapture(B->cap, cudaStreamCaptureModeThreadLocal));
        int rc = batch_record(B, check_every, B->cap);
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamEndCapture(B->cap, &graph);
        if (rc != GPE_OK) {
            if (graph) cudaGraphDestroy(graph);
            return rc;
        }
        if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture", __FILE__, __LINE__);
        e = cudaGraphInstantiate(&B->exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate", __FILE__, __LINE__);
        B->key = key;
    }
    int64_t done = 0;
    const int nodes = (int)(3 * check_every + 5);
    int unconv = B->n;
    while (done < max_steps && unconv > 0) {
        GPE_TRY_CUDA(cudaGraphLaunch(B->exec, s));
        for (int k = 0; k < nodes; ++k) count_launch();
        done += check_every;
        GPE_TRY_CUDA(cudaMemcpyAsync(B->h_unconv, B->d_unconv, sizeof(int), cudaMemcpyDeviceToHost, s));
        GPE_TRY_CUDA(cudaStreamSynchronize(s));
        unconv = *B->h_unconv;
    }
    // results back to the states and to the caller
    for (int i = 0; i < B->n; ++i)
        GPE_TRY_CUDA(cudaMemcpyAsync(B->states[i]->d_psi, (char *)B->d_psi + B->packed_base[i] * B->elem,
                                     B->states[i]->grid->n_packed * B->elem, cudaMemcpyDeviceToDevice, s));
    GPE_TRY_CUDA(cudaMemcpyAsync(sh.data(), B->d_sh, B->n * sizeof(ShellParams), cudaMemcpyDeviceToHost, s));
    GPE_TRY_CUDA(cudaStreamSynchronize(s));
    int n_bad = 0, n_unconv = 0;
    for (int i = 0; i < B->n; ++i) {
        const ShellParams &P = sh[i];
        if (converged) converged[i] = P.converged && P.nonfinite == 0;
        if (steps) steps[i] = P.steps;
        if (obs) {
            obs[i].norm = P.norm;
            obs[i].energy = P.energy;
            obs[i].mu = P.mu;
            obs[i].nonfinite = P.nonfinite;
            obs[i].e_kin = P.e_kin;
            obs[i].e_pot = P.e_pot;
            obs[i].e_int = P.e_int;
        }
        if (P.nonfinite > 0) ++n_bad;
        else if (!P.converged) ++n_unconv;
    }
    (void)done;
    if (n_bad) return fail(GPE_ERR_NONFINITE, "%d shell(s) hold NaN or Inf", n_bad);
    if (n_unconv) return fail(GPE_ERR_NOT_CONVERGED, "%d shell(s) did not reach |dmu| < %g", n_unconv, tol_dmu);
    return GPE_OK;
}
