// tiles.cu -- the neighbour slots and halo lists of the stencil kernels'
// tiles (tiles.cuh), built on the device once per grid.
//
// One block of TILE threads a tile: thread i finds segment i's brick (binary
// search over the bricks' packed offsets) and lattice position, then the
// stored segments at its neighbour positions through the brick volume and the
// bricks' records.  Neighbours outside the tile go into a hash set in shared
// memory; its members, sorted (whole segments first, then those of which one
// cell is read, each by packed position, so that neighbouring lanes gather
// neighbouring segments), are the halo list.
#include <algorithm>

#include "occupancy.h"
#include "tiles.cuh"

namespace gpe {

struct TileSrc {
    const BrickRec *rec;
    const int32_t *org;   // brick origins in cells
    const int32_t *bvol;  // brick position -> id or -1
    int64_t nb, nbx, nby, nbz;
    int by, bz;
    uint32_t nseg;
};

constexpr uint32_t NO_SEG = 0xffffffffu;

// bit position of the r-th (from 0) set bit of m
__device__ __forceinline__ int nth_bit(uint32_t m, int r)
{
    int pos = 0;
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) {
        const int c = __popc(m & ((1u << w) - 1u));
        if (r >= c) {
            r -= c;
            m >>= w;
            pos += w;
        }
    }
    return pos;
}

__device__ __forceinline__ int64_t brick_of(const TileSrc &S, uint32_t seg, int64_t lo, int64_t hi)
{
    while (hi - lo > 1) {  // the last brick of [lo, hi) that starts at or before seg
        const int64_t mid = (lo + hi) >> 1;
        if (S.rec[mid].off / 4u <= seg) lo = mid;
        else hi = mid;
    }
    return lo;
}

// stored segment at segment column sx (4 cells), row y, plane z of the box
__device__ __forceinline__ uint32_t seg_at(const TileSrc &S, int64_t sx, int64_t y, int64_t z)
{
    if (sx < 0 || y < 0 || z < 0) return NO_SEG;
    const int64_t bx = sx >> 1, b_y = y / S.by, b_z = z / S.bz;
    if (bx >= S.nbx || b_y >= S.nby || b_z >= S.nbz) return NO_SEG;
    const int32_t id = S.bvol[bx + S.nbx * (b_y + S.nby * b_z)];
    if (id < 0) return NO_SEG;
    uint32_t idx;
    const int q = (int)(sx & 1) + 2 * ((int)(y - b_y * S.by) + S.by * (int)(z - b_z * S.bz));
    return seg_index(S.rec[id], q, idx) ? idx / 4u : NO_SEG;
}

// uses of a halo segment
constexpr uint32_t USE_FIRST = 1, USE_LAST = 2, USE_WHOLE = 4;

// Rows of `stride` entries; a tile with more halo segments than fit leaves its
// lists out (hmax tells, and the caller builds again with longer rows).
template <int NP>
__global__ void __launch_bounds__(TILE) k_tiles(const TileSrc S, int stride, uint2 *nbr, uint4 *nbr19, uint32_t *halo,
                                                int *hmax)
{
    constexpr int NF = TileFields<NP>::N;
    constexpr int HS = NP == 19 ? 4096 : 1024;  // hash slots, above NF * TILE
    static_assert(HS > NF * TILE, "the set must hold every neighbour");
    // neighbour offsets: segment columns, rows, planes; and the use
    constexpr int8_t D[18][4] = {{0, -1, 0, 4}, {0, 1, 0, 4},  {0, 0, -1, 4}, {0, 0, 1, 4},  {-1, 0, 0, 2}, {1, 0, 0, 1},
                                 {0, -1, -1, 4}, {0, 1, -1, 4}, {0, -1, 1, 4}, {0, 1, 1, 4},  {-1, -1, 0, 2}, {1, -1, 0, 1},
                                 {-1, 1, 0, 2}, {1, 1, 0, 1},  {-1, 0, -1, 2}, {1, 0, -1, 1}, {-1, 0, 1, 2}, {1, 0, 1, 1}};
    __shared__ uint32_t key[HS];
    __shared__ uint32_t use[HS];   // uses, then the slot
    __shared__ uint32_t list[NF * TILE];   // the set's members as they sort
    __shared__ uint16_t where[NF * TILE];  // and their hash slots
    __shared__ int64_t b0;
    __shared__ int n_all, n_whole;
    const int tid = threadIdx.x;
    const uint32_t seg0 = blockIdx.x * TILE, seg = seg0 + tid;
    for (int i = tid; i < HS; i += TILE) {
        key[i] = NO_SEG;
        use[i] = 0;
    }
    if (tid == 0) {
        b0 = brick_of(S, seg0, 0, S.nb);
        n_all = 0;
        n_whole = 0;
    }
    __syncthreads();
    uint32_t nb[NF];
    const bool in = seg < S.nseg;
    if (in) {
        const int64_t b = brick_of(S, seg, b0, min(b0 + TILE, S.nb));
        const BrickRec r = S.rec[b];
        int k = (int)(seg - r.off / 4u), w = 0;
        while (k >= __popc(r.m[w])) k -= __popc(r.m[w++]);
        const int q = 32 * w + nth_bit(r.m[w], k);
        const int64_t sx = S.org[3 * b] / 4 + (q & 1), y = S.org[3 * b + 1] + (q >> 1) % S.by,
                      z = S.org[3 * b + 2] + (q >> 1) / S.by;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            nb[f] = seg_at(S, sx + D[f][0], y + D[f][1], z + D[f][2]);
            if (nb[f] == NO_SEG || (nb[f] >= seg0 && nb[f] < seg0 + TILE)) continue;
            uint32_t h = (nb[f] * 2654435761u) >> (NP == 19 ? 20 : 22);
            while (true) {
                const uint32_t was = atomicCAS(&key[h], NO_SEG, nb[f]);
                if (was == NO_SEG || was == nb[f]) break;
                h = (h + 1) & (HS - 1);
            }
            atomicOr(&use[h], (uint32_t)D[f][3]);
        }
    }
    __syncthreads();
    // a segment read whole, or at both ends, is copied whole
    auto whole = [](uint32_t u) { return (u & USE_WHOLE) || u == (USE_FIRST | USE_LAST); };
    for (int i = tid; i < HS; i += TILE) {
        if (key[i] == NO_SEG) continue;
        const bool wh = whole(use[i]);
        const int at = atomicAdd(&n_all, 1);
        if (wh) atomicAdd(&n_whole, 1);
        list[at] = key[i] | (wh ? 0u : 1u << 31);
        where[at] = (uint16_t)i;
    }
    __syncthreads();
    const int n = n_all;
    if (tid == 0 && n > __ldcg(hmax)) atomicMax(hmax, n);
    if (n + 1 > stride) return;
    for (int t = tid; t < n; t += TILE) {
        const uint32_t v = list[t];
        const int i = where[t];
        const uint32_t u = use[i];
        int rank = 0;
        for (int j = 0; j < n; ++j) rank += list[j] < v;
        // whole segments from the front of the tile's entries, single cells from the back
        const int at = rank < n_whole ? 1 + rank : stride - 1 - (rank - n_whole);
        halo[(size_t)blockIdx.x * stride + at] = key[i] | (u == USE_FIRST ? 1u << 31 : 0u);
        use[i] = TILE + 1 + rank;
    }
    if (tid == 0) halo[(size_t)blockIdx.x * stride] = (uint32_t)n_whole | (uint32_t)(n - n_whole) << 16;
    __syncthreads();
    if (!in) return;
    uint32_t sl[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        if (nb[f] == NO_SEG) {
            sl[f] = TILE;
        } else if (nb[f] >= seg0 && nb[f] < seg0 + TILE) {
            sl[f] = nb[f] - seg0;
        } else {
            uint32_t h = (nb[f] * 2654435761u) >> (NP == 19 ? 20 : 22);
            while (key[h] != nb[f]) h = (h + 1) & (HS - 1);
            sl[f] = use[h];
        }
    }
    if constexpr (NP == 19) {
        unsigned long long q[4] = {0, 0, 0, 0};
#pragma unroll
        for (int f = 0; f < NF; ++f) q[f / 5] |= (unsigned long long)sl[f] << (12 * (f % 5));
        nbr19[2 * (size_t)seg] = make_uint4((uint32_t)q[0], (uint32_t)(q[0] >> 32), (uint32_t)q[1], (uint32_t)(q[1] >> 32));
        nbr19[2 * (size_t)seg + 1] =
            make_uint4((uint32_t)q[2], (uint32_t)(q[2] >> 32), (uint32_t)q[3], (uint32_t)(q[3] >> 32));
    } else {
        nbr[seg] = make_uint2(sl[0] | sl[1] << 10 | sl[2] << 20, sl[3] | sl[4] << 10 | sl[5] << 20);
    }
}

void tiles_free(TileTab &t)
{
    dev_free(t.d_nbr);
    dev_free(t.d_nbr19);
    dev_free(t.d_halo);
    t = TileTab{};
}

// rows of one stride to rows of another, at least as long as every list
__global__ void k_tile_rows(const uint32_t *from, int sf, uint32_t *to, int st, int ntiles)
{
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const uint32_t *r = from + (size_t)tile * sf;
        uint32_t *w = to + (size_t)tile * st;
        const int whole = r[0] & 0xffff, single = r[0] >> 16;
        for (int i = threadIdx.x; i <= whole; i += blockDim.x) w[i] = r[i];
        for (int i = threadIdx.x; i < single; i += blockDim.x) w[st - 1 - i] = r[sf - 1 - i];
    }
}

template <int NP>
static int build(const TileSrc &S, TileTab &t, int *d_hmax, cudaStream_t st)
{
    // most grids' lists fit rows of 256 (thin shells: at most 208 segments
    // with the 7-point stencil); the rows kept are as long as the longest list
    int stride = NP == 19 ? 512 : 256, hmax = 0;
    uint32_t *rows = nullptr;
    int rc = GPE_OK;
    for (;;) {
        rc = dev_alloc_t(&rows, (size_t)t.ntiles * stride);
        if (rc != GPE_OK) return rc;
        cudaError_t e = cudaMemsetAsync(d_hmax, 0, sizeof(int), st);
        if (e == cudaSuccess) {
            k_tiles<NP><<<(unsigned)t.ntiles, TILE, 0, st>>>(S, stride, t.d_nbr, t.d_nbr19, rows, d_hmax);
            count_launch();
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(&hmax, d_hmax, sizeof hmax, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) {
            dev_free(rows);
            return cuda_fail(e, "k_tiles", __FILE__, __LINE__);
        }
        if (hmax + 1 <= stride) break;
        dev_free(rows);
        rows = nullptr;
        stride = (hmax + 8) / 8 * 8;
    }
    t.stride = (hmax + 8) / 8 * 8;  // and the count; whole sectors
    t.nslot = TILE + 1 + hmax;
    rc = dev_alloc_t(&t.d_halo, (size_t)t.ntiles * t.stride);
    if (rc == GPE_OK) {
        k_tile_rows<<<(unsigned)std::min(t.ntiles, 65536), 128, 0, st>>>(rows, stride, t.d_halo, t.stride, t.ntiles);
        count_launch();
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) rc = cuda_fail(e, "k_tile_rows", __FILE__, __LINE__);
    }
    dev_free(rows);  // waits for the copy
    return rc;
}

// the tiles of a grid whose records and brick volume are in place, and its
// neighbour slots (nseg of them) allocated; d_hmax is a word of scratch.  The work is on stream st when it
// returns.
int tiles_build(gpe_grid *g, int *d_hmax, cudaStream_t st)
{
    TileTab &t = g->tiles;
    t.nseg = (uint32_t)(g->n_packed / 4);
    t.ntiles = (int)((t.nseg + TILE - 1) / TILE);
    const TileSrc S{g->d_rec, g->d_org, g->d_bvol, g->nb, g->nbx, g->nby, g->nbz, g->by, g->bz, t.nseg};
    return g->stencil == 19 ? build<19>(S, t, d_hmax, st) : build<7>(S, t, d_hmax, st);
}

int blocks_per_sm(const void *kernel, int threads, size_t smem, size_t smem_max)
{
    static Occupancy known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return known.blocks(
        dev, kernel, smem,
        [&] {
            const bool ok = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)smem_max) == cudaSuccess;
            if (!ok) cudaGetLastError();
            return ok;
        },
        [&] {
            int per = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem) != cudaSuccess) {
                cudaGetLastError();
                per = 0;
            }
            return per;
        });
}

}  // namespace gpe
