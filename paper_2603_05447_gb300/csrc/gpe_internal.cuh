// gpe_internal.cuh -- shared internals of libgpeshell (not part of the ABI).
//
// Layout of a grid in device memory.  Bricks of BC = BX*BY*BZ lattice cells,
// local index l = x + BX*(y + BY*z); "slot" = brick * BC + l addresses the
// lattice.  A segment is 4 consecutive cells along x (local segment q = l/4).
// Only segments holding an active cell are stored ("packed" layout):
//   d_org  [nb*3]  int32    brick origin in cells (i0, j0, k0)
//   d_nbr  [nb*6]  int32    face-neighbour brick ids (-x +x -y +y -z +z), -1 = none
//   d_mask [ns/32] uint32   active-cell bits of the lattice, bit slot&31 of word slot/32
//   d_rec  [nb]    BrickRec stored-segment bits, per-word prefix counts, packed offset
//   d_V[s] [n_packed] double potential slot s (0: V or V0, 1: V1); the inactive
//                           cells of stored segments hold +inf in slot 0
// Packed index of cell l of brick b (if its segment is stored):
//   rec.off + 4*(rank of segment l/4 among the brick's stored segments) + l%4.
// Inactive cells of stored segments hold psi = 0 and are never updated (the
// +inf potential marks them); cells of absent segments and bricks are not
// stored and read as psi = 0: Dirichlet zero on the rows/columns deleted
// from the Laplacian (Sec. II A).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>
#include <initializer_list>
#include <vector>

#include "gpe.h"

namespace gpe {

// ------------------------------------------------------------ errors
int fail(int code, const char *fmt, ...);
int cuda_fail(cudaError_t e, const char *expr, const char *file, int line);

#define GPE_TRY_CUDA(x)                                                      \
    do {                                                                     \
        cudaError_t e__ = (x);                                               \
        if (e__ != cudaSuccess)                                              \
            return ::gpe::cuda_fail(e__, #x, __FILE__, __LINE__);            \
    } while (0)
#define GPE_TRY(x)                                                           \
    do {                                                                     \
        int r__ = (x);                                                       \
        if (r__ != GPE_OK) return r__;                                       \
    } while (0)
// every kernel launch of the library is followed by GPE_LAUNCH_CHECK(), which
// also counts it (gpe_launch_count)
void count_launch();
#define GPE_LAUNCH_CHECK()                                                   \
    do {                                                                     \
        ::gpe::count_launch();                                               \
        GPE_TRY_CUDA(cudaGetLastError());                                    \
    } while (0)

int dev_alloc(void **p, size_t bytes);
template <typename T>
inline int dev_alloc_t(T **p, size_t count)
{
    return dev_alloc(reinterpret_cast<void **>(p), count * sizeof(T));
}
void dev_free(void *p);
// Arrays that live and die together, in one allocation at *base: a cudaMalloc
// and its cudaFree take 50 to 70 us, and each regrid, state and tape used to
// make 10 to 17 of them (four regrids and states of a 512^3 ramp: 8 of 34 ms)
struct Part {
    void **p;
    size_t bytes;
    template <typename T>
    Part(T **p_, size_t count) : p(reinterpret_cast<void **>(p_)), bytes(count * sizeof(T))
    {
    }
    Part(void **p_, size_t bytes_) : p(p_), bytes(bytes_) {}
};
int dev_alloc_parts(void **base, std::initializer_list<Part> parts);
int dev_zero(void *p, size_t bytes);  // memset 0 and wait (any stream may use it next)

inline cudaStream_t S(gpe_stream s) { return reinterpret_cast<cudaStream_t>(s); }

// supported brick shapes; the kernels are instantiated for each
int shape_id(int bx, int by, int bz);  // 0: 8x8x8, 1: 8x8x4, 2: 8x4x4

int sm_count(int device);
// resident blocks an SM of a kernel with smem bytes of dynamic shared memory on
// the current device; the kernel is allowed smem_max bytes there (occupancy.h)
int blocks_per_sm(const void *kernel, int threads, size_t smem, size_t smem_max);

// per-brick record of the packed layout (32 bytes)
struct BrickRec {
    uint32_t m[4];  // bit q: segment q is stored
    uint32_t off;   // packed index of the brick's first stored cell
    uint32_t pre;   // byte w: stored segments in mask words < w
    uint32_t pad[2];
};

// Brick shapes are powers of two, 8 along x: a lattice cell's brick, local index
// and position by shifts (64-bit divisions made the builder's and the copies'
// kernels twice as long)
struct BrickGeo {
    int ly, lz;  // log2 of the rows and planes
    __host__ __device__ int lc() const { return 3 + ly + lz; }  // log2 of the cells
    __host__ __device__ int64_t brick(int64_t s) const { return s >> lc(); }
    __host__ __device__ int local(int64_t s) const { return (int)(s & ((1 << lc()) - 1)); }
    __host__ __device__ int x(int l) const { return l & 7; }
    __host__ __device__ int y(int l) const { return (l >> 3) & ((1 << ly) - 1); }
    __host__ __device__ int z(int l) const { return l >> (3 + ly); }
};
inline BrickGeo brick_geo(int by, int bz) { return BrickGeo{by == 8 ? 3 : 2, bz == 8 ? 3 : 2}; }

// packed index of the first cell of segment q, if stored
__host__ __device__ __forceinline__ bool seg_index(const BrickRec &r, int q, uint32_t &idx)
{
    const int w = q >> 5, bit = q & 31;
    const uint32_t m = r.m[w];
    if (!((m >> bit) & 1u)) return false;
#ifdef __CUDA_ARCH__
    const uint32_t below = __popc(m & ((1u << bit) - 1u));
#else
    const uint32_t below = (uint32_t)__builtin_popcount(m & ((1u << bit) - 1u));
#endif
    idx = r.off + 4u * (((r.pre >> (8 * w)) & 0xffu) + below);
    return true;
}

// ------------------------------------------------------------ complex types
template <typename R> struct Cx;
template <> struct Cx<float> { using T = float2; };
template <> struct Cx<double> { using T = double2; };

template <typename R>
__device__ __forceinline__ typename Cx<R>::T cmk(R x, R y)
{
    typename Cx<R>::T c;
    c.x = x;
    c.y = y;
    return c;
}

// ------------------------------------------------------------ reductions
// Deterministic FP64 block reduction of NV values with a "last block
// finishes" epilogue: every block writes its partial sums to
// partials[blockIdx.x*NV + k]; the last block to arrive sums all partials in
// a fixed order.  Returns true in the one block that holds the totals, whose
// thread 0 then has them in tot[].  The counter is reset to 0 by that block.
template <int NV>
__device__ __forceinline__ bool reduce_finish(double (&v)[NV], double *partials,
                                              unsigned int *counter, double (&tot)[NV])
{
    __shared__ double sm[NV][32];
    __shared__ bool is_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        double x = v[k];
        for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
        if (lane == 0) sm[k][warp] = x;
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            double x = lane < nwarps ? sm[k][lane] : 0.0;
            for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
            if (lane == 0) partials[(int64_t)blockIdx.x * NV + k] = x;
        }
    }
    if (threadIdx.x == 0) {
        __threadfence();
        unsigned int ticket = atomicAdd(counter, 1u);
        is_last = (ticket == gridDim.x - 1);
    }
    __syncthreads();
    if (!is_last) return false;
    __threadfence();
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        double x = 0.0;
        for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x)
            x += __ldcg(&partials[(int64_t)i * NV + k]);
        for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
        __syncthreads();
        if (lane == 0) sm[k][warp] = x;
        __syncthreads();
        if (warp == 0) {
            x = lane < nwarps ? sm[k][lane] : 0.0;
            for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
            if (lane == 0) tot[k] = x;
        }
    }
    if (threadIdx.x == 0) *counter = 0u;
    return true;
}

// Per-launch scratch for reductions: partial sums (max_blocks * 8 doubles),
// a completion counter and a few FP64 scalars (ITP scale, results).
struct RedScratch {
    double *partials = nullptr;
    unsigned int *counter = nullptr;
    double *scalars = nullptr;  // [0] ITP scale, [1] last norm, [2..9] observables
};
// the reductions' arrays for up to nsm * RED_PER_SM blocks, as parts of a
// caller's allocation; red_zero when they are in place
constexpr int RED_PER_SM = 32;
inline Part red_partials(RedScratch &r, int nsm) { return Part(&r.partials, (size_t)nsm * RED_PER_SM * 8); }
inline Part red_counter(RedScratch &r) { return Part(&r.counter, 1); }
inline Part red_scalars(RedScratch &r) { return Part(&r.scalars, 16); }
int red_zero(const RedScratch &r);

// stored segments a tile, and threads a block of the tile kernels (tiles.cuh)
constexpr int TILE = 128;
// neighbour slots and halo lists of a grid's tiles
struct TileTab {
    uint2 *d_nbr = nullptr;      // 7-point grids
    uint4 *d_nbr19 = nullptr;    // 19-point grids
    uint32_t *d_halo = nullptr;  // [ntiles * stride]
    uint32_t nseg = 0;
    int ntiles = 0, stride = 0;
    int nslot = 0;               // slots of the largest tile: own, zero, halo
};

}  // namespace gpe

// ------------------------------------------------------------ handles
struct gpe_grid {
    int device = 0;
    gpe_box box{};
    int bx = 8, by = 8, bz = 8, bc = 512, shape = 0;
    int mask_mode = 0, order = 0;
    int64_t nbx = 0, nby = 0, nbz = 0;
    int64_t nb = 0, n_stored = 0, n_active = 0;
    int64_t n_packed = 0;
    int32_t *d_org = nullptr;
    int32_t *d_nbr = nullptr;
    uint32_t *d_mask = nullptr;
    gpe::BrickRec *d_rec = nullptr;
    gpe::BrickRec *d_rec7 = nullptr;  // [nb*7] record of each brick and of its six face neighbours (wavefront schedules)
    int stencil = 7;                  // 7 or 19 points
    int32_t *d_nbr18 = nullptr;       // [nb*18] face then edge neighbour ids (PAIR schedule, built on first use)
    std::vector<void *> blocks;  // the allocations that hold the arrays above and below, but d_rec7, d_nbr18, d_Vf
                                 // and the wavefront schedules'
    gpe::TileTab tiles;         // the stencil kernels' tiles
    int32_t *d_bvol = nullptr;  // brick-grid volume nbx*nby*nbz -> brick id or -1
    double *d_V[2] = {nullptr, nullptr};
    float *d_Vf[2] = {nullptr, nullptr};  // float copies, made on first use
    // wavefront schedule (built on first use): chunks of `cb` consecutive
    // bricks, the chunk range each chunk's stencils touch, and the task order
    // for 2-stage (imaginary time) and 4-stage (RK4) steps
    int cb = 0;
    int64_t n_chunks = 0;
    int32_t *d_chunk_lohi = nullptr;  // [n_chunks*2]
    int32_t *d_tasks = nullptr;       // [2*n_chunks] for 2 stages, then [4*n_chunks] for 4
    // warp-task schedule of the two-stage RK4 launches (GPE_SCHED_WAVE2): per
    // chunk the sorted chunks its stencils read (CSR), and the task order
    int32_t *d_dep_off = nullptr;     // [n_chunks + 1]
    int32_t *d_dep_ids = nullptr;
    int32_t *d_tasks_w = nullptr;     // [2*n_chunks]
    int sched = -1;                   // GPE_SCHED_* used by the step calls
    int n_slots = 1;
    unsigned long long v0_version = 0;  // how often slot 0 has been replaced: tables made from it hold the count
    double v_max = 0.0;
    int nsm = 0;
    int n_states = 0;
};

struct gpe_state {
    gpe_grid *grid = nullptr;
    int dtype = GPE_C128;
    size_t elem = 16;       // bytes per complex element
    void *d_psi = nullptr;  // n_packed complex
    void *block = nullptr;  // the allocation that holds psi, E, the clock and the reductions' arrays
    void *d_work[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};  // RK stage states / ITP tmp
    std::vector<void *> work_blocks;  // the allocations that hold them and the schedule tables
    void *d_E = nullptr;    // ITP exp(-V dt/2), state precision
    double E_dt = -1.0;     // dt and
    unsigned long long E_version = 0;  // potential (gpe_grid::v0_version) that d_E was made for
    double *d_clock = nullptr;  // device time base for ramps
    double *d_stab = nullptr;   // schedule values of the next steps' stages (ramps)
    int stab_cap = 0;           // steps it holds
    gpe::RedScratch red;
    gpe_obs *h_obs = nullptr;   // pinned host landing buffer
    // wavefront bookkeeping: per-chunk completion stamps (monotonic), the
    // dynamic ticket counter, the finish counter and a device error word
    uint32_t *d_done = nullptr;
    unsigned long long *d_ctr = nullptr;  // [0] tickets, [1] finished ITP chunks, [2] error
    double *d_chunk_norm = nullptr;       // per-chunk FP64 partial norms (ITP)
    uint32_t epoch = 0;                   // stages completed so far (flags compare to it)
    unsigned long long ticket_base = 0, finish_base = 0;
    // CUDA graphs of `graph_steps` staged steps ([0] real time, [1] imaginary)
    int graph_steps = 32;
    cudaGraphExec_t gexec[2] = {nullptr, nullptr};
    unsigned long long gkey[2] = {0, 0};
    int gnodes[2] = {0, 0};
    cudaStream_t gcap = nullptr;
};

namespace gpe {
int tiles_build(gpe_grid *g, int *d_hmax, cudaStream_t st);
void tiles_free(TileTab &t);
int ensure_stab(gpe_state *st, int steps);      // room for the schedule values of `steps` steps
int ensure_work(gpe_state *st, int n);          // allocate d_work[0..n-1] (zeroed)
// step drivers of 19-point grids (step19.cu)
int rk4_run19(gpe_state *st, const gpe_real_params *p, int64_t nsteps, double t0, cudaStream_t s);
int itp_run19(gpe_state *st, const gpe_imag_params *p, int64_t nsteps, cudaStream_t s);
int obs_run19(const gpe_state *st, double g, double s_blend, cudaStream_t s);
int ensure_vf(gpe_grid *g, int slot);           // float copy of a potential slot
const void *potential_ptr(gpe_state *st, int slot);  // V slot in state precision
}  // namespace gpe
