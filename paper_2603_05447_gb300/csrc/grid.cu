// grid.cu -- region-of-interest selection and brick compaction (Sec. II A and
// Sec. II B of the paper), built on the device.
//
// Steps: (1) brick occupancy over the brick grid covering the box (a brick is
// kept if any of its in-box cells has V < V_cut); (2) enumeration of the brick
// grid in Morton or z-major key order with an order-preserving compaction (two
// passes: per-block counts, then emission at scanned offsets); (3) a dense
// brick-id volume and the 6-entry face-neighbour table; (4) per-cell potential
// values and the active-cell bit mask; (5) the packed layout's records; (6) the
// stencil kernels' tiles (tiles.cu).  The paper's GPU variant keeps a 488-entry
// halo index list per 8^3 block (Sec. II B, 3.8 bytes a cell); here a tile of 128
// stored segments has neighbour slots and a list of the segments outside it,
// 3.2 bytes a stored cell, and the wavefront and fused schedules gather a brick's
// halo at fixed offsets from its neighbours.
#include <algorithm>
#include <cmath>
#include <vector>

#include "gpe_internal.cuh"
#include "stencil.cuh"

namespace gpe {

struct PotDesc {
    int kind;
    double p[8];
};

// V source for the builder: a dense array, one analytic potential, or two
// potentials (ramp endpoints, analytic or dense) whose union mask is taken.
struct VSource {
    int mode;  // 0 dense, 1 analytic, 2 analytic blend, 3 dense blend
    const void *dense, *dense1;
    int dtype;
    PotDesc p0, p1;
    double cut0, cut1;
};

__device__ __forceinline__ double eval_pot(const PotDesc &P, double x, double y, double z)
{
    if (P.kind == GPE_POT_HARMONIC)
        return 0.5 * (P.p[0] * P.p[0] * x * x + P.p[1] * P.p[1] * y * y + P.p[2] * P.p[2] * z * z);
    if (P.kind == GPE_POT_ELLIPSOID_SHELL) {
        double rho = sqrt(x * x / (P.p[1] * P.p[1]) + y * y / (P.p[2] * P.p[2]) +
                          z * z / (P.p[3] * P.p[3]));
        double d = rho - 1.0;
        return 0.5 * P.p[0] * P.p[0] * d * d;
    }
    return 0.0;
}

struct BoxD {
    int64_t nx, ny, nz;
    double hx, hy, hz, x0, y0, z0;
};

__device__ __forceinline__ void cell_values(const VSource &src, const BoxD &bx, int64_t i,
                                            int64_t j, int64_t k, double &v0, double &v1,
                                            bool &sel)
{
    if (src.mode == 0 || src.mode == 3) {
        int64_t lin = i + bx.nx * (j + bx.ny * k);
        auto at = [&](const void *p) {
            return src.dtype == GPE_F64 ? ((const double *)p)[lin] : (double)((const float *)p)[lin];
        };
        v0 = at(src.dense);
        if (src.mode == 3) {
            v1 = at(src.dense1);
            sel = (v0 < src.cut0) || (v1 < src.cut1);
        } else {
            v1 = 0.0;
            sel = v0 < src.cut0;
        }
        return;
    }
    double x = bx.x0 + i * bx.hx, y = bx.y0 + j * bx.hy, z = bx.z0 + k * bx.hz;
    v0 = eval_pot(src.p0, x, y, z);
    if (src.mode == 2) {
        v1 = eval_pot(src.p1, x, y, z);
        sel = (v0 < src.cut0) || (v1 < src.cut1);
    } else {
        v1 = 0.0;
        sel = v0 < src.cut0;
    }
}

// May an analytic potential fall below `cut` somewhere in the axis-aligned
// box [xl,xh] x [yl,yh] x [zl,zh]?  (true for an unknown kind.)  Both
// potentials are separable in the squares of the coordinates, so the extremes
// of each square over an interval give the exact range: the harmonic
// potential's minimum directly, and for the ellipsoidal shell the range
// [rmin, rmax] of the scaled radius, from which the smallest |rho - 1|
// follows.  Evaluated in FP32 with wide margins: it only has to be
// conservative, the per-cell FP64 test decides.  Where FP32 does not reach (a
// bound that is not finite, semi-axes far from 1, a stiffness so small that
// its bound and the cutoff lose bits) the answer is yes.
__device__ __forceinline__ bool pot_may_select(const PotDesc &P, double cut, float xl, float xh, float yl, float yh,
                                               float zl, float zh)
{
    auto sqmin = [](float l, float h) { return (l <= 0.f && h >= 0.f) ? 0.f : fminf(l * l, h * h); };
    auto sqmax = [](float l, float h) { return fmaxf(l * l, h * h); };
    if (P.kind == GPE_POT_HARMONIC) {
        // |w| times the least |coordinate|, squared as a product, since either
        // square may underflow; factors without their full bits count as 0
        auto least = [](double w, float l, float h) {
            const float a = fabsf((float)w), d = (l <= 0.f && h >= 0.f) ? 0.f : fminf(fabsf(l), fabsf(h));
            return a < 1e-37f || d < 1e-37f ? 0.f : a * d;
        };
        const float tx = least(P.p[0], xl, xh), ty = least(P.p[1], yl, yh), tz = least(P.p[2], zl, zh);
        const float vmin = 0.5f * (tx * tx + ty * ty + tz * tz);
        return !(vmin > (float)cut * 1.0001f + 1e-30f) || !(vmin < INFINITY);
    }
    if (P.kind == GPE_POT_ELLIPSOID_SHELL) {
        const float w = (float)P.p[0];
        const float ia = 1.f / (float)(P.p[1] * P.p[1]), ib = 1.f / (float)(P.p[2] * P.p[2]),
                    ic = 1.f / (float)(P.p[3] * P.p[3]);
        const float least = fminf(ia, fminf(ib, ic)), most = fmaxf(ia, fmaxf(ib, ic));
        if (!(least > 1e-30f && most < 1e30f && fabsf(w) >= 1e-15f)) return true;
        const float rmin = sqrtf(sqmin(xl, xh) * ia + sqmin(yl, yh) * ib + sqmin(zl, zh) * ic);
        const float rmax = sqrtf(sqmax(xl, xh) * ia + sqmax(yl, yh) * ib + sqmax(zl, zh) * ic);
        const float d = (rmin <= 1.f && rmax >= 1.f) ? 0.f : fminf(fabsf(rmin - 1.f), fabsf(rmax - 1.f));
        // V = w^2 d^2 / 2 < cut  <=>  |w| d < sqrt(2 cut)
        const float reach = fabsf(w) * d;
        return !(reach > sqrtf(2.f * fmaxf((float)cut, 0.f)) * 1.0001f + 1e-4f * (1.f + rmax) * fabsf(w)) || !(reach < INFINITY);
    }
    return true;
}

// (1) occupancy of every brick-grid position (lexicographic q), 256 brick
// positions a block.  Analytic sources: one thread a position tests the
// brick's cell-centre box against the bound above; then the block tests the
// cells of each candidate brick exactly.
__global__ void k_occupancy(VSource src, BoxD box, int BX, int BY, int BZ, int64_t nbx, int64_t nby, int64_t nbz,
                            uint8_t *occ)
{
    __shared__ int64_t cand[256];
    __shared__ int ncand;
    const int64_t nq = nbx * nby * nbz;
    const int64_t q = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (threadIdx.x == 0) ncand = 0;
    __syncthreads();
    if (q < nq) {
        const int64_t qx = q % nbx, qy = (q / nbx) % nby, qz = q / (nbx * nby);
        bool may = true;
        if (src.mode == 1 || src.mode == 2) {
            const int64_t i0 = qx * BX, j0 = qy * BY, k0 = qz * BZ;
            const int64_t i1 = min(i0 + BX, box.nx) - 1, j1 = min(j0 + BY, box.ny) - 1, k1 = min(k0 + BZ, box.nz) - 1;
            const float xl = (float)(box.x0 + i0 * box.hx), xh = (float)(box.x0 + i1 * box.hx);
            const float yl = (float)(box.y0 + j0 * box.hy), yh = (float)(box.y0 + j1 * box.hy);
            const float zl = (float)(box.z0 + k0 * box.hz), zh = (float)(box.z0 + k1 * box.hz);
            may = pot_may_select(src.p0, src.cut0, xl, xh, yl, yh, zl, zh);
            if (src.mode == 2) may = may || pot_may_select(src.p1, src.cut1, xl, xh, yl, yh, zl, zh);
        }
        if (may)
            cand[atomicAdd(&ncand, 1)] = q;
        else
            occ[q] = 0;
    }
    __syncthreads();
    const int nc = ncand;
    const int BC = BX * BY * BZ;
    for (int c = 0; c < nc; ++c) {
        const int64_t qq = cand[c];
        const int64_t qx = qq % nbx, qy = (qq / nbx) % nby, qz = qq / (nbx * nby);
        int sel_any = 0;
        for (int l = threadIdx.x; l < BC; l += blockDim.x) {
            const int64_t i = qx * BX + l % BX, j = qy * BY + (l / BX) % BY, k = qz * BZ + l / (BX * BY);
            if (i < box.nx && j < box.ny && k < box.nz) {
                double v0, v1;
                bool sel;
                cell_values(src, box, i, j, k, v0, v1, sel);
                sel_any |= sel;
            }
        }
        sel_any = __syncthreads_or(sel_any);
        if (threadIdx.x == 0) occ[qq] = (uint8_t)(sel_any != 0);
    }
}

// A threshold in the forms its comparisons use.  An FP64 comparison issues at
// 1/64 of the FP32 rate here, so FP32 cells are compared in FP32 against the
// threshold rounded up (the same set: a float is below t exactly if it is below
// the next float at or above t), FP64 cells as integers that order like them.
struct Limit {
    double t;
    float f;      // smallest float >= t
    int64_t ord;  // t as an integer
};
constexpr int64_t ORD_MINUS_INF = (int64_t)(0xfff0000000000000ull ^ 0x7fffffffffffffffull);

static Limit limit_of(double t)
{
    Limit m;
    m.t = t;
    m.f = (float)t;
    if ((double)m.f < t) m.f = std::nextafter(m.f, INFINITY);
    int64_t b;
    memcpy(&b, &t, 8);
    m.ord = t == 0.0 ? -1 : (b < 0 ? b ^ 0x7fffffffffffffffll : b);  // neither zero is below a zero
    if (std::isnan(t)) m.ord = INT64_MIN;                            // nothing is below a NaN
    return m;
}

// v < t (false for a NaN)
__device__ __forceinline__ bool below(float v, const Limit &m) { return v < m.f; }
__device__ __forceinline__ bool below(double v, const Limit &m)
{
    const int64_t b = __double_as_longlong(v), o = b < 0 ? b ^ 0x7fffffffffffffffll : b;
    return o < m.ord && o >= ORD_MINUS_INF;
}

// (1) for dense potentials: every cell of the box is read once, in rows, a warp
// a row, and marks its brick.  Bound by that read (512^3 FP32,
// two potentials in 0.19 ms, 5.8 TB/s); testing brick by brick, a block barrier
// each and in FP64, took 2.0 ms.  occ is zero before.
template <typename T>
__global__ void k_occ_dense(const T *V0, const T *V1, Limit c0, Limit c1, BoxD box, int BY, int BZ, int64_t nbx,
                            int64_t nby, uint8_t *occ)
{
    const int lane = threadIdx.x & 31;
    const int64_t rows = box.ny * box.nz, nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t r = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += nw) {
        const int64_t j = r % box.ny, k = r / box.ny;
        uint8_t *row = occ + nbx * (j / BY + nby * (k / BZ));
        const T *v0 = V0 + r * box.nx, *v1 = V1 ? V1 + r * box.nx : nullptr;
        for (int64_t i0 = 0; i0 < box.nx; i0 += 128) {
            bool sel[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int64_t i = i0 + 32 * q + lane;
                const T a = i < box.nx ? v0[i] : (T)INFINITY;
                const T b = v1 && i < box.nx ? v1[i] : (T)INFINITY;
                sel[q] = i < box.nx && (below(a, c0) | (v1 && below(b, c1)));
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const unsigned any = __ballot_sync(0xffffffffu, sel[q]);
                if (lane < 4 && ((any >> (8 * lane)) & 0xffu)) row[(i0 + 32 * q) / 8 + lane] = 1;
            }
        }
    }
}

// (4) for dense potentials: the active bits of the kept bricks, a warp a word
template <typename T>
__global__ void k_mask_dense(const T *V0, const T *V1, Limit c0, Limit c1, BoxD box, BrickGeo G, int mask_mode,
                             const int32_t *org, int64_t nwords, uint32_t *mask,
                             unsigned long long *n_active)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    unsigned long long cnt = 0;
    for (int64_t w = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); w < nwords; w += nw) {
        const int64_t b = G.brick(32 * w);
        const int l = G.local(32 * w) + lane;
        const int64_t i = org[3 * b] + G.x(l), j = org[3 * b + 1] + G.y(l), k = org[3 * b + 2] + G.z(l);
        bool act = i < box.nx && j < box.ny && k < box.nz;
        if (act && mask_mode == GPE_MASK_CELL) {
            const int64_t lin = i + box.nx * (j + box.ny * k);
            const T a = V0[lin], c = V1 ? V1[lin] : (T)INFINITY;
            act = below(a, c0) | (V1 && below(c, c1));
        }
        const unsigned bits = __ballot_sync(0xffffffffu, act);
        if (lane == 0) {
            mask[w] = bits;
            cnt += __popc(bits);
        }
    }
    if (lane == 0 && cnt) atomicAdd(n_active, cnt);
}

// |v| as an integer that orders like it, 0 for a NaN
__device__ __forceinline__ unsigned long long abs_bits(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
    return b <= 0x7ff0000000000000ull ? b : 0ull;
}
__device__ __forceinline__ void block_max(unsigned long long v, unsigned long long *out)
{
    for (int off = 16; off > 0; off >>= 1) v = max(v, __shfl_down_sync(0xffffffffu, v, off));
    if ((threadIdx.x & 31) == 0 && v > __ldcg(out)) atomicMax(out, v);
}

// the packed potentials of a dense source, straight from the box: active cells
// get their value, inactive cells of stored segments +inf in slot 0 and 0 in
// slot 1
template <typename T>
__global__ void k_fill_dense(const T *S0, const T *S1, BoxD box, BrickGeo G, const int32_t *org, const uint32_t *mask,
                              const BrickRec *rec, int64_t ns, double *V0, double *V1,
                             unsigned long long *vmax_bits)
{
    unsigned long long vm = 0;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < ns; s += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = G.brick(s);
        const int l = G.local(s);
        uint32_t idx;
        if (!seg_index(rec[b], l >> 2, idx)) continue;
        idx += l & 3;
        if ((mask[s >> 5] >> (s & 31)) & 1u) {
            const int64_t lin = org[3 * b] + G.x(l) +
                                box.nx * (org[3 * b + 1] + G.y(l) + box.ny * (int64_t)(org[3 * b + 2] + G.z(l)));
            const double v = (double)S0[lin];
            V0[idx] = v;
            vm = max(vm, abs_bits(v));
            if (V1) {
                const double w = (double)S1[lin];
                V1[idx] = w;
                vm = max(vm, abs_bits(w));
            }
        } else {
            V0[idx] = INFINITY;
            if (V1) V1[idx] = 0.0;
        }
    }
    block_max(vm, vmax_bits);
}

// exclusive scan of v[n] in place by one block, total to *tot
__global__ void k_scan(int64_t *v, int64_t n, int64_t *tot)
{
    constexpr int PER = 4;
    __shared__ int64_t wsum[32];
    __shared__ int64_t carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int64_t base = 0; base < n; base += (int64_t)blockDim.x * PER) {
        const int64_t at = base + (int64_t)threadIdx.x * PER;
        int64_t x[PER], own = 0;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            x[q] = at + q < n ? v[at + q] : 0;
            own += x[q];
        }
        int64_t incl = own;
        for (int off = 1; off < 32; off <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += y;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        int64_t pre = carry + incl - own;
        for (int w = 0; w < warp; ++w) pre += wsum[w];
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            if (at + q < n) v[at + q] = pre;
            pre += x[q];
        }
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry = pre;
        __syncthreads();
    }
    if (threadIdx.x == 0) *tot = carry;
}

__device__ __forceinline__ uint32_t compact3(uint64_t m)
{
    // keep every third bit of m (bit 3n -> bit n)
    uint64_t x = m & 0x1249249249249249ull;
    x = (x ^ (x >> 2)) & 0x10c30c30c30c30c3ull;
    x = (x ^ (x >> 4)) & 0x100f00f00f00f00full;
    x = (x ^ (x >> 8)) & 0x1f0000ff0000ffull;
    x = (x ^ (x >> 16)) & 0x1f00000000ffffull;
    x = (x ^ (x >> 32)) & 0x1fffffull;
    return (uint32_t)x;
}

struct Enum {
    int order;  // GPE_ORDER_*
    int64_t nbx, nby, nbz;
    uint64_t nkeys;
};

__device__ __forceinline__ bool key_brick(const Enum &E, const uint8_t *occ, uint64_t key,
                                          int64_t &bx, int64_t &by, int64_t &bz)
{
    if (E.order == GPE_ORDER_MORTON) {
        bx = compact3(key);
        by = compact3(key >> 1);
        bz = compact3(key >> 2);
        if (bx >= E.nbx || by >= E.nby || bz >= E.nbz) return false;
    } else {
        bx = key % E.nbx;
        by = (key / E.nbx) % E.nby;
        bz = key / (E.nbx * E.nby);
    }
    return occ[bx + E.nbx * (by + E.nby * bz)] != 0;
}

constexpr int ENUM_THREADS = 256, ENUM_PER_THREAD = 4;
constexpr int ENUM_PER_BLOCK = ENUM_THREADS * ENUM_PER_THREAD;

// (2a) number of kept bricks per enumeration block
__global__ void k_enum_count(Enum E, const uint8_t *occ, int64_t *bsum)
{
    const uint64_t base = (uint64_t)blockIdx.x * ENUM_PER_BLOCK + threadIdx.x * ENUM_PER_THREAD;
    int c = 0;
    for (int r = 0; r < ENUM_PER_THREAD; ++r) {
        uint64_t key = base + r;
        int64_t bx, by, bz;
        if (key < E.nkeys && key_brick(E, occ, key, bx, by, bz)) ++c;
    }
    __shared__ int warp_tot[ENUM_THREADS / 32];
    for (int off = 16; off > 0; off >>= 1) c += __shfl_down_sync(0xffffffffu, c, off);
    if ((threadIdx.x & 31) == 0) warp_tot[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int s = 0;
        for (int w = 0; w < ENUM_THREADS / 32; ++w) s += warp_tot[w];
        bsum[blockIdx.x] = s;
    }
}

// (2b) emit kept bricks in key order at the scanned block offsets
__global__ void k_enum_emit(Enum E, const uint8_t *occ, const int64_t *boff, int32_t *coords)
{
    __shared__ int warp_tot[ENUM_THREADS / 32];
    const uint64_t base = (uint64_t)blockIdx.x * ENUM_PER_BLOCK + threadIdx.x * ENUM_PER_THREAD;
    int c = 0;
    for (int r = 0; r < ENUM_PER_THREAD; ++r) {
        uint64_t key = base + r;
        int64_t bx, by, bz;
        if (key < E.nkeys && key_brick(E, occ, key, bx, by, bz)) ++c;
    }
    // exclusive scan of c over threads (in thread order = key order)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = c;
    for (int off = 1; off < 32; off <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    int wpre = 0;
    for (int w = 0; w < warp; ++w) wpre += warp_tot[w];
    int64_t pos = boff[blockIdx.x] + wpre + incl - c;
    for (int r = 0; r < ENUM_PER_THREAD; ++r) {
        uint64_t key = base + r;
        int64_t bx, by, bz;
        if (key < E.nkeys && key_brick(E, occ, key, bx, by, bz)) {
            coords[3 * pos + 0] = (int32_t)bx;
            coords[3 * pos + 1] = (int32_t)by;
            coords[3 * pos + 2] = (int32_t)bz;
            ++pos;
        }
    }
}

// (3) brick-id volume, from the bricks' positions
__global__ void k_bricks(int64_t nb, const int32_t *coords, int64_t nbx, int64_t nby, int32_t *bvol)
{
    int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (id >= nb) return;
    int64_t bx = coords[3 * id], by = coords[3 * id + 1], bz = coords[3 * id + 2];
    bvol[bx + nbx * (by + nby * bz)] = (int32_t)id;
}

// neighbour table; then the bricks' positions become their origins in cells
__global__ void k_neighbors(int64_t nb, int32_t *coords, int BX, int BY, int BZ, int64_t nbx, int64_t nby, int64_t nbz,
                            const int32_t *bvol, int32_t *nbr)
{
    int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (id >= nb) return;
    const int64_t c[3] = {coords[3 * id], coords[3 * id + 1], coords[3 * id + 2]};
    coords[3 * id] = (int32_t)(c[0] * BX);
    coords[3 * id + 1] = (int32_t)(c[1] * BY);
    coords[3 * id + 2] = (int32_t)(c[2] * BZ);
    const int64_t n[3] = {nbx, nby, nbz};
    for (int d = 0; d < 6; ++d) {
        int64_t q[3] = {c[0], c[1], c[2]};
        q[d >> 1] += (d & 1) ? 1 : -1;
        int32_t r = -1;
        if (q[d >> 1] >= 0 && q[d >> 1] < n[d >> 1]) r = bvol[q[0] + nbx * (q[1] + nby * q[2])];
        nbr[6 * id + d] = r;
    }
}

// (4) for analytic potentials: per-cell values and active bits; one block per brick
__global__ void k_cells(VSource src, BoxD box, int BX, int BY, int BZ, int mask_mode,
                        const int32_t *org, double *V0, double *V1, uint32_t *mask,
                        unsigned long long *n_active, unsigned long long *vmax_bits)
{
    const int64_t id = blockIdx.x;
    const int BC = BX * BY * BZ;
    unsigned long long cnt = 0, vm = 0;
    for (int l = threadIdx.x; l < BC; l += blockDim.x) {  // BC % 32 == 0, blockDim % 32 == 0
        int64_t i = org[3 * id] + l % BX, j = org[3 * id + 1] + (l / BX) % BY,
                k = org[3 * id + 2] + l / (BX * BY);
        bool inbox = i < box.nx && j < box.ny && k < box.nz;
        double v0 = 0.0, v1 = 0.0;
        bool sel = false;
        if (inbox) cell_values(src, box, i, j, k, v0, v1, sel);
        bool act = inbox && (mask_mode == GPE_MASK_BRICK ? true : sel);
        const int64_t slot = id * BC + l;
        V0[slot] = v0;
        if (V1) V1[slot] = v1;
        unsigned bits = __ballot_sync(0xffffffffu, act);
        if ((threadIdx.x & 31) == 0) mask[slot >> 5] = bits;
        if (act) {
            ++cnt;
            vm = max(vm, abs_bits(v0));
            if (V1) vm = max(vm, abs_bits(v1));
        }
    }
    for (int off = 16; off > 0; off >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, off);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(n_active, cnt);
    block_max(vm, vmax_bits);
}

// Segment layout: a segment is 4 consecutive cells along x inside a brick
// (one 32-byte sector of complex64).  A brick stores exactly its segments that
// hold at least one active cell.  k_seg_records builds each brick's record:
// the segment bit mask, the number of stored segments before each mask word
// and the packed offset within its block of bricks, whose count goes to
// bsum[block]; k_seg_offsets adds what precedes the block.
constexpr int REC_THREADS = 256;
__global__ void __launch_bounds__(REC_THREADS) k_seg_records(int64_t nb, int BC, const uint32_t *mask, BrickRec *rec,
                                                             int64_t *bsum)
{
    __shared__ uint32_t wsum[REC_THREADS / 32];
    int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int W = BC / 32, nseg = BC / 4;
    BrickRec r{};
    uint32_t c = 0;
    if (b < nb) {
        for (int q0 = 0; q0 < nseg; q0 += 8) {
            // cells 4q..4q+3 of the brick: nibble (q & 7) of mask word q/8
            const uint32_t word = mask[b * W + (q0 >> 3)];
            for (int q = 0; q < 8; ++q)
                if ((word >> (4 * q)) & 0xfu) r.m[q0 >> 5] |= 1u << ((q0 + q) & 31);
        }
        for (int w = 0; w < 4; ++w) {
            r.pre |= (c & 0xffu) << (8 * w);
            c += __popc(r.m[w]);
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = c;
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    uint32_t pre = incl - c;
    for (int w = 0; w < warp; ++w) pre += wsum[w];
    if (b < nb) {
        r.off = 4u * pre;
        rec[b] = r;
    }
    if (threadIdx.x == REC_THREADS - 1) bsum[blockIdx.x] = pre + c;
}
__global__ void k_seg_offsets(int64_t nb, BrickRec *rec, const int64_t *before)
{
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (b < nb) rec[b].off += (uint32_t)(4 * before[blockIdx.x]);
}

// scatter stored-lattice values to the packed layout: active cells get their
// value, inactive cells of stored segments get `fill`
__global__ void k_pack(int64_t ns, BrickGeo G, const uint32_t *mask, const BrickRec *rec, const double *src,
                       double *dst, double fill)
{
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < ns; s += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = G.brick(s);
        const int l = G.local(s);
        uint32_t idx;
        if (!seg_index(rec[b], l >> 2, idx)) continue;
        const bool act = (mask[s >> 5] >> (s & 31)) & 1u;
        dst[idx + (l & 3)] = act ? src[s] : fill;
    }
}

// replace a potential slot from a dense array (region unchanged)
__global__ void k_set_potential(const void *dense, int dtype, BoxD box, int BX, int BY, int BZ,
                                const int32_t *org, const uint32_t *mask, const BrickRec *rec, double *V)
{
    const int64_t id = blockIdx.x;
    const int BC = BX * BY * BZ, W = BC / 32;
    for (int l = threadIdx.x; l < BC; l += blockDim.x) {
        const uint32_t word = mask[id * W + (l >> 5)];
        if (!((word >> (l & 31)) & 1u)) continue;   // active cells are always inside the box
        uint32_t idx;
        if (!seg_index(rec[id], l >> 2, idx)) continue;
        int64_t i = org[3 * id] + l % BX, j = org[3 * id + 1] + (l / BX) % BY,
                k = org[3 * id + 2] + l / (BX * BY);
        int64_t lin = i + box.nx * (j + box.ny * k);
        V[idx + (l & 3)] = dtype == GPE_F64 ? ((const double *)dense)[lin] : (double)((const float *)dense)[lin];
    }
}

// max |V| over the active cells of the packed arrays (inactive cells of
// stored segments hold +inf in V0 and are skipped)
__global__ void k_vmax(int64_t np, const double *V0, const double *V1, unsigned long long *vmax_bits)
{
    double vm = 0.0;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < np;
         s += (int64_t)gridDim.x * blockDim.x) {
        if (!(V0[s] < INFINITY)) continue;
        vm = fmax(vm, fabs(V0[s]));
        if (V1) vm = fmax(vm, fabs(V1[s]));
    }
    for (int off = 16; off > 0; off >>= 1) vm = fmax(vm, __shfl_down_sync(0xffffffffu, vm, off));
    if ((threadIdx.x & 31) == 0) atomicMax(vmax_bits, (unsigned long long)__double_as_longlong(vm));
}

// per brick: its record followed by its six face neighbours' (-x +x -y +y -z
// +z; empty records for absent neighbours), a thread a record.  The wavefront
// grids' rows used to be made on the host: 256^3 shell grid 1.40 -> 1.22 ms.
__global__ void k_rec7(int64_t nb, const BrickRec *rec, const int32_t *nbr, BrickRec *out)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, b = i / 7;
    if (b >= nb) return;
    const int d = (int)(i - 7 * b);
    const int64_t from = d == 0 ? b : nbr[6 * b + d - 1];
    out[i] = from >= 0 ? rec[from] : BrickRec{};
}

}  // namespace gpe

namespace gpe {

static BoxD boxd(const gpe_box &b)
{
    return BoxD{b.nx, b.ny, b.nz, b.hx, b.hy, b.hz, b.x0, b.y0, b.z0};
}

static int check_box(const gpe_box *box)
{
    if (!box) return fail(GPE_ERR_ARG, "box is NULL");
    if (box->nx < 1 || box->ny < 1 || box->nz < 1)
        return fail(GPE_ERR_ARG, "box dimensions must be >= 1 (got %lld x %lld x %lld)",
                    (long long)box->nx, (long long)box->ny, (long long)box->nz);
    if (!(box->hx > 0) || !(box->hy > 0) || !(box->hz > 0))
        return fail(GPE_ERR_ARG, "grid spacings must be > 0");
    if (box->nx > (1 << 24) || box->ny > (1 << 24) || box->nz > (1 << 24))
        return fail(GPE_ERR_ARG, "box dimension above 2^24");
    return GPE_OK;
}

static int check_pot(const gpe_potential *p)
{
    if (!p) return fail(GPE_ERR_ARG, "potential is NULL");
    if (p->kind != GPE_POT_HARMONIC && p->kind != GPE_POT_ELLIPSOID_SHELL)
        return fail(GPE_ERR_ARG, "unknown potential kind %d", p->kind);
    if (p->kind == GPE_POT_ELLIPSOID_SHELL && (!(p->p[1] > 0) || !(p->p[2] > 0) || !(p->p[3] > 0)))
        return fail(GPE_ERR_ARG, "ellipsoid semi-axes must be > 0");
    return GPE_OK;
}

static PotDesc potdesc(const gpe_potential &p)
{
    PotDesc d;
    d.kind = p.kind;
    for (int i = 0; i < 8; ++i) d.p[i] = p.p[i];
    return d;
}

static void grid_free(gpe_grid *g)
{
    if (!g) return;
    for (void *b : g->blocks) dev_free(b);
    dev_free(g->d_rec7);
    dev_free(g->tiles.d_halo);
    dev_free(g->d_nbr18);
    dev_free(g->d_chunk_lohi);
    dev_free(g->d_tasks);
    dev_free(g->d_dep_off);
    dev_free(g->d_dep_ids);
    dev_free(g->d_tasks_w);
    for (int s = 0; s < 2; ++s) dev_free(g->d_Vf[s]);
    delete g;
}

// Build the grid; `src.dense` (mode 0) is a device pointer here.
static int build_grid(const gpe_box *box, const VSource &src, const gpe_grid_opts *opts,
                      gpe_grid **out, cudaStream_t st)
{
    gpe_grid_opts o{};
    if (opts) o = *opts;
    if (o.bx == 0 && o.by == 0 && o.bz == 0) o.bx = o.by = o.bz = 8;
    const int shape = shape_id(o.bx, o.by, o.bz);
    if (shape < 0)
        return fail(GPE_ERR_ARG, "unsupported brick shape %dx%dx%d (use 8x8x8, 8x8x4 or 8x4x4)", o.bx, o.by,
                    o.bz);
    if (o.mask_mode != GPE_MASK_CELL && o.mask_mode != GPE_MASK_BRICK)
        return fail(GPE_ERR_ARG, "unknown mask mode %d", o.mask_mode);
    if (o.order != GPE_ORDER_MORTON && o.order != GPE_ORDER_ZMAJOR)
        return fail(GPE_ERR_ARG, "unknown brick order %d", o.order);
    if (o.stencil != 0 && o.stencil != 7 && o.stencil != 19) return fail(GPE_ERR_ARG, "stencil must be 7 or 19");
    if (o.sched != GPE_SCHED_WAVE && o.sched != GPE_SCHED_WAVE2 && o.sched != GPE_SCHED_STAGED &&
        o.sched != GPE_SCHED_PAIR)
        return fail(GPE_ERR_ARG, "unknown schedule %d", o.sched);
    if (o.chunk < 0 || o.chunk > 4096) return fail(GPE_ERR_ARG, "chunk must be in [0, 4096]");

    gpe_grid *g = new gpe_grid();
    GPE_TRY_CUDA(cudaGetDevice(&g->device));
    g->nsm = sm_count(g->device);
    g->box = *box;
    g->bx = o.bx;
    g->by = o.by;
    g->bz = o.bz;
    g->bc = o.bx * o.by * o.bz;
    g->shape = shape;
    g->mask_mode = o.mask_mode;
    g->order = o.order;
    g->sched = o.sched;
    g->stencil = o.stencil == 19 ? 19 : 7;
    // bricks per wavefront task: about 2048 lattice cells for block tasks,
    // about 1024 for the warp tasks of WAVE2
    g->cb = o.chunk > 0 ? o.chunk : std::max(1, (o.sched == GPE_SCHED_WAVE2 ? 1024 : 2048) / g->bc);
    g->nbx = (box->nx + o.bx - 1) / o.bx;
    g->nby = (box->ny + o.by - 1) / o.by;
    g->nbz = (box->nz + o.bz - 1) / o.bz;
    const int64_t nq = g->nbx * g->nby * g->nbz;
    const BoxD bd = boxd(*box);

    // temporaries: occupancy, block counts and totals, then the analytic
    // potentials on the lattice
    uint8_t *occ = nullptr;
    int64_t *bsum = nullptr;
    double *tmpV[2] = {nullptr, nullptr};
    // read back together: bricks kept; stored segments, active cells, largest |V|
    struct Totals {
        int64_t bricks, segs;
        unsigned long long active, vmax;
        int hmax;  // tiles_build's
    };
    Totals *tot = nullptr, ht{};
    void *temp[2] = {nullptr, nullptr};
    int rc = GPE_OK;
    auto cleanup = [&]() {
        for (void *b : temp) dev_free(b);
    };
    // arrays of the grid, in one allocation
    auto alloc_own = [&](std::initializer_list<Part> parts) -> int {
        void *b = nullptr;
        GPE_TRY(dev_alloc_parts(&b, parts));
        g->blocks.push_back(b);
        return GPE_OK;
    };
#define BUILD_TRY(x)                 \
    do {                             \
        rc = (x);                    \
        if (rc != GPE_OK) {          \
            cleanup();               \
            grid_free(g);            \
            return rc;               \
        }                            \
    } while (0)
#define BUILD_CUDA(x)                                                        \
    do {                                                                     \
        cudaError_t e__ = (x);                                               \
        if (e__ != cudaSuccess) {                                            \
            rc = cuda_fail(e__, #x, __FILE__, __LINE__);                     \
            cleanup();                                                       \
            grid_free(g);                                                    \
            return rc;                                                       \
        }                                                                    \
    } while (0)

    const bool dense = src.mode == 0 || src.mode == 3, two = src.mode == 2 || src.mode == 3;
    const Limit c0 = limit_of(src.cut0), c1 = limit_of(src.cut1);
    const BrickGeo geo = brick_geo(o.by, o.bz);
    Enum E;
    E.order = o.order;
    E.nbx = g->nbx;
    E.nby = g->nby;
    E.nbz = g->nbz;
    if (o.order == GPE_ORDER_MORTON) {
        int64_t m = std::max(g->nbx, std::max(g->nby, g->nbz));
        int L = 0;
        while ((int64_t(1) << L) < m) ++L;
        if (3 * L > 62) BUILD_TRY(fail(GPE_ERR_ARG, "brick grid too large for Morton keys"));
        E.nkeys = uint64_t(1) << (3 * L);
    } else {
        E.nkeys = (uint64_t)nq;
    }
    const int64_t nblk = (int64_t)((E.nkeys + ENUM_PER_BLOCK - 1) / ENUM_PER_BLOCK);
    if (nblk > 0x7fffffffLL) BUILD_TRY(fail(GPE_ERR_ARG, "brick grid too large"));
    // block counts: of the enumeration, then of the records (at most nq bricks)
    BUILD_TRY(dev_alloc_parts(&temp[0], {{&tot, 1},
                                         {&bsum, (size_t)std::max(nblk, (nq + REC_THREADS - 1) / REC_THREADS)},
                                         {&occ, (size_t)nq}}));
    BUILD_CUDA(cudaMemsetAsync(tot, 0, sizeof(Totals), st));
    if (dense) {
        BUILD_CUDA(cudaMemsetAsync(occ, 0, nq, st));
        const unsigned nblk_rows = (unsigned)std::min<int64_t>((box->ny * box->nz + 7) / 8, (int64_t)g->nsm * 64);
        if (src.dtype == GPE_F64)
            k_occ_dense<double><<<nblk_rows, 256, 0, st>>>((const double *)src.dense, (const double *)src.dense1, c0, c1,
                                                          bd, o.by, o.bz, g->nbx, g->nby, occ);
        else
            k_occ_dense<float><<<nblk_rows, 256, 0, st>>>((const float *)src.dense, (const float *)src.dense1, c0, c1,
                                                         bd, o.by, o.bz, g->nbx, g->nby, occ);
        BUILD_CUDA(cudaGetLastError());
    } else {
        const int64_t nblk_occ = (nq + 255) / 256;
        if (nblk_occ > 0x7fffffffLL) BUILD_TRY(fail(GPE_ERR_ARG, "brick grid too large"));
        k_occupancy<<<(unsigned)nblk_occ, 256, 0, st>>>(src, bd, o.bx, o.by, o.bz, g->nbx, g->nby, g->nbz, occ);
        BUILD_CUDA(cudaGetLastError());
    }
    k_enum_count<<<(unsigned)nblk, ENUM_THREADS, 0, st>>>(E, occ, bsum);
    BUILD_CUDA(cudaGetLastError());
    k_scan<<<1, 1024, 0, st>>>(bsum, nblk, &tot->bricks);
    BUILD_CUDA(cudaGetLastError());
    BUILD_CUDA(cudaMemcpyAsync(&ht, tot, sizeof ht, cudaMemcpyDeviceToHost, st));
    BUILD_CUDA(cudaStreamSynchronize(st));
    const int64_t total = ht.bricks;
    if (total == 0) BUILD_TRY(fail(GPE_ERR_ARG, "region of interest is empty (no cell with V < V_cut)"));
    if (total * g->bc > 0x7fffffffLL * 32LL)
        BUILD_TRY(fail(GPE_ERR_ARG, "too many stored cells"));
    g->nb = total;
    g->n_stored = total * g->bc;
    BUILD_TRY(alloc_own({{&g->d_bvol, (size_t)nq},
                         {&g->d_org, 3 * (size_t)total},
                         {&g->d_nbr, 6 * (size_t)total},
                         {&g->d_mask, (size_t)(g->n_stored / 32)},
                         {&g->d_rec, (size_t)total}}));
    k_enum_emit<<<(unsigned)nblk, ENUM_THREADS, 0, st>>>(E, occ, bsum, g->d_org);
    BUILD_CUDA(cudaGetLastError());
    BUILD_CUDA(cudaMemsetAsync(g->d_bvol, 0xff, nq * sizeof(int32_t), st));
    const unsigned nbb = (unsigned)((total + 255) / 256);
    k_bricks<<<nbb, 256, 0, st>>>(total, g->d_org, g->nbx, g->nby, g->d_bvol);
    BUILD_CUDA(cudaGetLastError());
    k_neighbors<<<nbb, 256, 0, st>>>(total, g->d_org, o.bx, o.by, o.bz, g->nbx, g->nby, g->nbz, g->d_bvol, g->d_nbr);
    BUILD_CUDA(cudaGetLastError());

    if (total > 0x7fffffffLL) BUILD_TRY(fail(GPE_ERR_ARG, "too many bricks"));
    if (two) g->n_slots = 2;
    if (dense) {
        const int64_t nwords = g->n_stored / 32;
        const unsigned nbw = (unsigned)std::min<int64_t>((nwords + 7) / 8, (int64_t)g->nsm * 32);
        if (src.dtype == GPE_F64)
            k_mask_dense<double><<<nbw, 256, 0, st>>>((const double *)src.dense, (const double *)src.dense1, c0, c1, bd,
                                                     geo, o.mask_mode, g->d_org, nwords, g->d_mask,
                                                     &tot->active);
        else
            k_mask_dense<float><<<nbw, 256, 0, st>>>((const float *)src.dense, (const float *)src.dense1, c0, c1, bd,
                                                    geo, o.mask_mode, g->d_org, nwords, g->d_mask,
                                                    &tot->active);
    } else {
        BUILD_TRY(dev_alloc_parts(&temp[1], {{&tmpV[0], (size_t)g->n_stored}, {&tmpV[1], two ? (size_t)g->n_stored : 0}}));
        if (!two) tmpV[1] = nullptr;
        k_cells<<<(unsigned)total, std::min(g->bc, 256), 0, st>>>(src, bd, o.bx, o.by, o.bz, o.mask_mode, g->d_org,
                                                                tmpV[0], tmpV[1], g->d_mask, &tot->active, &tot->vmax);
    }
    BUILD_CUDA(cudaGetLastError());

    // packed layout: every brick stores its segments (4 cells along x) that
    // hold an active cell, in lattice order, as one run
    const int64_t nblk_rec = (total + REC_THREADS - 1) / REC_THREADS;
    k_seg_records<<<(unsigned)nblk_rec, REC_THREADS, 0, st>>>(total, g->bc, g->d_mask, g->d_rec, bsum);
    BUILD_CUDA(cudaGetLastError());
    k_scan<<<1, 1024, 0, st>>>(bsum, nblk_rec, &tot->segs);
    BUILD_CUDA(cudaGetLastError());
    k_seg_offsets<<<(unsigned)nblk_rec, REC_THREADS, 0, st>>>(total, g->d_rec, bsum);
    BUILD_CUDA(cudaGetLastError());
    BUILD_CUDA(cudaMemcpyAsync(&ht, tot, sizeof ht, cudaMemcpyDeviceToHost, st));
    BUILD_CUDA(cudaStreamSynchronize(st));
    g->n_active = (int64_t)ht.active;
    if (4 * (uint64_t)ht.segs >= 0xffffffffull)
        BUILD_TRY(fail(GPE_ERR_ARG, "too many stored cells for 32-bit offsets"));
    g->n_packed = 4 * ht.segs;
    if (o.sched == GPE_SCHED_WAVE || o.sched == GPE_SCHED_WAVE2) {
        // the wavefront kernels' record rows
        BUILD_TRY(dev_alloc_t(&g->d_rec7, total * 7));
        k_rec7<<<(unsigned)((7 * total + 255) / 256), 256, 0, st>>>(total, g->d_rec, g->d_nbr, g->d_rec7);
        BUILD_CUDA(cudaGetLastError());
    }
    const size_t np = (size_t)g->n_packed;
    BUILD_TRY(alloc_own({{&g->d_V[0], np},
                         {&g->d_V[1], two ? np : 0},
                         {&g->tiles.d_nbr, g->stencil == 19 ? 0 : np / 4},
                         {&g->tiles.d_nbr19, g->stencil == 19 ? np / 2 : 0}}));
    if (!two) g->d_V[1] = nullptr;
    BUILD_TRY(tiles_build(g, &tot->hmax, st));
    if (dense) {
        const unsigned nbf = (unsigned)g->nsm * 16;
        if (src.dtype == GPE_F64)
            k_fill_dense<double><<<nbf, 256, 0, st>>>((const double *)src.dense, (const double *)src.dense1, bd, geo,
                                                     g->d_org, g->d_mask, g->d_rec, g->n_stored, g->d_V[0],
                                                     g->d_V[1], &tot->vmax);
        else
            k_fill_dense<float><<<nbf, 256, 0, st>>>((const float *)src.dense, (const float *)src.dense1, bd, geo,
                                                    g->d_org, g->d_mask, g->d_rec, g->n_stored, g->d_V[0],
                                                    g->d_V[1], &tot->vmax);
        BUILD_CUDA(cudaGetLastError());
    } else {
        for (int sl = 0; sl < g->n_slots; ++sl) {
            k_pack<<<g->nsm * 8, 256, 0, st>>>(g->n_stored, geo, g->d_mask, g->d_rec, tmpV[sl], g->d_V[sl],
                                              sl == 0 ? (double)INFINITY : 0.0);
            BUILD_CUDA(cudaGetLastError());
        }
    }
    BUILD_CUDA(cudaMemcpyAsync(&ht, tot, sizeof ht, cudaMemcpyDeviceToHost, st));
    BUILD_CUDA(cudaStreamSynchronize(st));
    memcpy(&g->v_max, &ht.vmax, sizeof(double));
    cleanup();
#undef BUILD_TRY
#undef BUILD_CUDA
    *out = g;
    return GPE_OK;
}

static int stage_dense(const gpe_box *box, const void *V, int V_dtype, int on_device,
                       const void **dptr, void **owned, cudaStream_t st)
{
    *owned = nullptr;
    if (!V) return fail(GPE_ERR_ARG, "V is NULL");
    if (V_dtype != GPE_F64 && V_dtype != GPE_F32) return fail(GPE_ERR_ARG, "V_dtype must be GPE_F64 or GPE_F32");
    if (on_device) {
        *dptr = V;
        return GPE_OK;
    }
    size_t bytes = (size_t)box->nx * box->ny * box->nz * (V_dtype == GPE_F64 ? 8 : 4);
    GPE_TRY(dev_alloc(owned, bytes));
    cudaError_t e = cudaMemcpyAsync(*owned, V, bytes, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) {
        dev_free(*owned);
        *owned = nullptr;
        return cuda_fail(e, "cudaMemcpyAsync(V)", __FILE__, __LINE__);
    }
    *dptr = *owned;
    return GPE_OK;
}

int ensure_vf(gpe_grid *g, int slot)
{
    if (g->d_Vf[slot]) return GPE_OK;
    GPE_TRY(dev_alloc_t(&g->d_Vf[slot], g->n_packed));
    // conversion is ordered on the legacy stream; synchronise so that any
    // stream sees the finished copy
    extern int convert_to_float(const double *src, float *dst, int64_t n);
    GPE_TRY(convert_to_float(g->d_V[slot], g->d_Vf[slot], g->n_packed));
    return GPE_OK;
}

}  // namespace gpe

using namespace gpe;

extern "C" int gpe_grid_create_dense(const gpe_box *box, const void *V, int V_dtype, int V_on_device,
                                     double V_cut, const gpe_grid_opts *opts, gpe_grid **out,
                                     gpe_stream stream)
{
    if (!out) return fail(GPE_ERR_ARG, "out is NULL");
    *out = nullptr;
    GPE_TRY(check_box(box));
    cudaStream_t st = S(stream);
    const void *dptr = nullptr;
    void *owned = nullptr;
    GPE_TRY(stage_dense(box, V, V_dtype, V_on_device, &dptr, &owned, st));
    VSource src{};
    src.mode = 0;
    src.dense = dptr;
    src.dtype = V_dtype;
    src.cut0 = V_cut;
    int rc = build_grid(box, src, opts, out, st);
    if (owned) {
        cudaStreamSynchronize(st);
        dev_free(owned);
    }
    return rc;
}

extern "C" int gpe_grid_create_analytic(const gpe_box *box, const gpe_potential *pot, double V_cut,
                                        const gpe_grid_opts *opts, gpe_grid **out, gpe_stream stream)
{
    if (!out) return fail(GPE_ERR_ARG, "out is NULL");
    *out = nullptr;
    GPE_TRY(check_box(box));
    GPE_TRY(check_pot(pot));
    VSource src{};
    src.mode = 1;
    src.p0 = potdesc(*pot);
    src.cut0 = V_cut;
    return build_grid(box, src, opts, out, S(stream));
}

extern "C" int gpe_grid_create_blend(const gpe_box *box, const gpe_potential *pot0, double cut0,
                                     const gpe_potential *pot1, double cut1, const gpe_grid_opts *opts,
                                     gpe_grid **out, gpe_stream stream)
{
    if (!out) return fail(GPE_ERR_ARG, "out is NULL");
    *out = nullptr;
    GPE_TRY(check_box(box));
    GPE_TRY(check_pot(pot0));
    GPE_TRY(check_pot(pot1));
    VSource src{};
    src.mode = 2;
    src.p0 = potdesc(*pot0);
    src.p1 = potdesc(*pot1);
    src.cut0 = cut0;
    src.cut1 = cut1;
    return build_grid(box, src, opts, out, S(stream));
}

extern "C" int gpe_grid_create_blend_dense(const gpe_box *box, const void *V0, const void *V1, int V_dtype,
                                           int V_on_device, double cut0, double cut1,
                                           const gpe_grid_opts *opts, gpe_grid **out, gpe_stream stream)
{
    if (!out) return fail(GPE_ERR_ARG, "out is NULL");
    *out = nullptr;
    GPE_TRY(check_box(box));
    cudaStream_t st = S(stream);
    const void *d0 = nullptr, *d1 = nullptr;
    void *own0 = nullptr, *own1 = nullptr;
    GPE_TRY(stage_dense(box, V0, V_dtype, V_on_device, &d0, &own0, st));
    int rc = stage_dense(box, V1, V_dtype, V_on_device, &d1, &own1, st);
    if (rc == GPE_OK) {
        VSource src{};
        src.mode = 3;
        src.dense = d0;
        src.dense1 = d1;
        src.dtype = V_dtype;
        src.cut0 = cut0;
        src.cut1 = cut1;
        rc = build_grid(box, src, opts, out, st);
    }
    if (own0 || own1) {
        cudaStreamSynchronize(st);
        dev_free(own0);
        dev_free(own1);
    }
    return rc;
}

extern "C" int gpe_grid_set_potential(gpe_grid *g, int slot, const void *V, int V_dtype, int V_on_device,
                                      gpe_stream stream)
{
    if (!g) return fail(GPE_ERR_ARG, "grid is NULL");
    if (slot != 0 && slot != 1) return fail(GPE_ERR_ARG, "slot must be 0 or 1");
    cudaStream_t st = S(stream);
    const void *dptr = nullptr;
    void *owned = nullptr;
    GPE_TRY(stage_dense(&g->box, V, V_dtype, V_on_device, &dptr, &owned, st));
    int rc = GPE_OK;
    if (!g->d_V[slot]) {
        rc = dev_alloc_t(&g->d_V[slot], g->n_packed);
        if (rc == GPE_OK) g->blocks.push_back(g->d_V[slot]);
        if (rc == GPE_OK) rc = dev_zero(g->d_V[slot], g->n_packed * sizeof(double));
    }
    if (rc == GPE_OK) {
        k_set_potential<<<(unsigned)g->nb, std::min(g->bc, 256), 0, st>>>(dptr, V_dtype, boxd(g->box), g->bx,
                                                                        g->by, g->bz, g->d_org, g->d_mask,
                                                                        g->d_rec, g->d_V[slot]);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) rc = cuda_fail(e, "k_set_potential", __FILE__, __LINE__);
    }
    if (rc == GPE_OK && slot == 0) ++g->v0_version;
    if (rc == GPE_OK && slot == 1) g->n_slots = 2;
    unsigned long long *vb = nullptr;
    if (rc == GPE_OK) rc = dev_alloc_t(&vb, 1);
    if (rc == GPE_OK) {
        cudaMemsetAsync(vb, 0, sizeof(unsigned long long), st);
        k_vmax<<<g->nsm * 4, 256, 0, st>>>(g->n_packed, g->d_V[0], g->n_slots > 1 ? g->d_V[1] : nullptr, vb);
        unsigned long long h = 0;
        cudaMemcpyAsync(&h, vb, sizeof h, cudaMemcpyDeviceToHost, st);
        cudaError_t e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) rc = cuda_fail(e, "set_potential", __FILE__, __LINE__);
        long long hv = (long long)h;
        memcpy(&g->v_max, &hv, sizeof(double));
    }
    dev_free(vb);
    if (owned) {
        cudaStreamSynchronize(st);
        dev_free(owned);
    }
    if (g->d_Vf[slot]) {
        dev_free(g->d_Vf[slot]);
        g->d_Vf[slot] = nullptr;
    }
    return rc;
}

extern "C" int gpe_grid_get_info(const gpe_grid *g, gpe_grid_info *out)
{
    if (!g || !out) return fail(GPE_ERR_ARG, "NULL argument");
    out->n_active = g->n_active;
    out->n_bricks = g->nb;
    out->n_stored = g->n_stored;
    out->n_packed = g->n_packed;
    out->bx = g->bx;
    out->by = g->by;
    out->bz = g->bz;
    out->mask_mode = g->mask_mode;
    out->order = g->order;
    out->n_slots = g->n_slots;
    out->v_max = g->v_max;
    out->box = g->box;
    return GPE_OK;
}

extern "C" int gpe_grid_bricks(const gpe_grid *g, int32_t *origins, int32_t *nbr)
{
    if (!g) return fail(GPE_ERR_ARG, "grid is NULL");
    if (origins) GPE_TRY_CUDA(cudaMemcpy(origins, g->d_org, g->nb * 3 * sizeof(int32_t), cudaMemcpyDeviceToHost));
    if (nbr) GPE_TRY_CUDA(cudaMemcpy(nbr, g->d_nbr, g->nb * 6 * sizeof(int32_t), cudaMemcpyDeviceToHost));
    return GPE_OK;
}

extern "C" int gpe_grid_mask(const gpe_grid *g, uint32_t *bits)
{
    if (!g || !bits) return fail(GPE_ERR_ARG, "NULL argument");
    GPE_TRY_CUDA(cudaMemcpy(bits, g->d_mask, g->n_stored / 32 * sizeof(uint32_t), cudaMemcpyDeviceToHost));
    return GPE_OK;
}

extern "C" int gpe_grid_potential(const gpe_grid *g, int slot, double *V)
{
    if (!g || !V) return fail(GPE_ERR_ARG, "NULL argument");
    if (slot < 0 || slot > 1 || !g->d_V[slot]) return fail(GPE_ERR_ARG, "potential slot %d not set", slot);
    GPE_TRY_CUDA(cudaMemcpy(V, g->d_V[slot], g->n_packed * sizeof(double), cudaMemcpyDeviceToHost));
    return GPE_OK;
}

extern "C" int gpe_grid_destroy(gpe_grid *g)
{
    if (!g) return GPE_OK;
    if (g->n_states > 0) return fail(GPE_ERR_STATE, "grid still has %d live states", g->n_states);
    grid_free(g);
    return GPE_OK;
}

// ------------------------------------------------------------ Thomas-Fermi mu
namespace gpe {

// A pass of the Thomas-Fermi solve reads the box once: over the cells with
// V < mu, the sum of V (FP64) and their count, and over all cells below +inf
// the largest |V| (its leading 32 bits, as an integer).  FP64 work is kept off
// that path (an FP64 instruction issues at 1/64 of the FP32 rate, predicated
// off or not): cells are compared as in Limit, counted in integers, and FP32
// cells are added as pairs of floats (Sum64), behind a branch that vectors
// without a selected cell skip.  512^3 FP32: 1.55 ms compared, added and counted in
// FP64, 0.19 ms with the selected cells added in FP64 (eight instructions a vector, which
// filled the FP64 pipe), 0.11 ms so (4.8 TB/s).
template <typename T>
struct TfSum {
    Sum64<T> sum;
    unsigned long long cnt = 0;
    uint32_t top = 0;
};

__device__ __forceinline__ uint32_t tf_top(float v) { return v < INFINITY ? __float_as_uint(fabsf(v)) : 0u; }
__device__ __forceinline__ uint32_t tf_top(double v)
{
    const uint32_t hi = (uint32_t)__double2hiint(v), a = hi & 0x7fffffffu;
    // below +inf: finite or -inf (NaN and +inf have no place in the sums)
    return a < 0x7ff00000u || (hi == 0xfff00000u && __double2loint(v) == 0) ? a : 0u;
}

// a thread's sum of SUM_FLUSH terms stays within a float pair if none exceeds
// PAIR_MAX; larger ones are added in FP64
__device__ __noinline__ double tf_add(double sum, float v) { return sum + (double)v; }
__device__ __noinline__ double tf_add(double sum, double a, double b, unsigned sel)
{
    if (sel & 1u) sum += a;
    if (sel & 2u) sum += b;
    return sum;
}
template <int W>
__device__ __forceinline__ void tf_add(Sum64<float> &s, const float (&v)[W], unsigned sel)
{
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const float x = (sel >> w) & 1u ? v[w] : 0.0f;
        if (fabsf(x) <= PAIR_MAX) s.add(x);
        else s.tot = tf_add(s.tot, x);
    }
}
template <int W>
__device__ __forceinline__ void tf_add(Sum64<double> &s, const double (&v)[W], unsigned sel)
{
#pragma unroll
    for (int w = 0; w < W; w += 2) s.tot = tf_add(s.tot, v[w], w + 1 < W ? v[w + 1 < W ? w + 1 : w] : 0.0, sel >> w);
}
template <typename T, int W>
__device__ __forceinline__ void tf_cells(const T (&v)[W], const Limit &m, TfSum<T> &a)
{
    unsigned sel = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        a.top = max(a.top, tf_top(v[w]));
        sel |= (below(v[w], m) ? 1u : 0u) << w;
    }
    if (sel) {
        a.cnt += __popc(sel);
        tf_add(a.sum, v, sel);
    }
}

template <typename T>
__device__ __forceinline__ void tf_finish(TfSum<T> &a, double *partials, unsigned int *counter, double *result,
                                          uint32_t *top)
{
    const uint32_t t = __reduce_max_sync(0xffffffffu, a.top);
    if ((threadIdx.x & 31) == 0 && t > __ldcg(top)) atomicMax(top, t);
    a.sum.flush();
    double acc[2] = {a.sum.tot, (double)a.cnt}, tot[2];
    if (reduce_finish<2>(acc, partials, counter, tot) && threadIdx.x == 0) {
        result[0] = tot[0];
        result[1] = tot[1];
    }
}

// dense V, n cells; n_vec of them (from the start) by 16-byte loads
template <typename T>
__global__ void k_tf_dense(const T *V, int64_t n, int64_t n_vec, Limit m, double *partials, unsigned int *counter,
                           double *result, uint32_t *top)
{
    constexpr int W = 16 / (int)sizeof(T);
    struct alignas(16) Vec {
        T v[W];
    };
    TfSum<T> a;
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    const Vec *src = reinterpret_cast<const Vec *>(V);
    const int64_t nv = n_vec / W;
    // four loads in flight a thread
    int64_t i = t;
    int n4 = 0;
    for (; i + 3 * step < nv; i += 4 * step) {
        if (++n4 % (SUM_FLUSH / (4 * W)) == 0) a.sum.flush();
        Vec x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = src[i + k * step];
#pragma unroll
        for (int k = 0; k < 4; ++k) tf_cells<T, W>(x[k].v, m, a);
    }
    a.sum.flush();  // at most three vectors are left
    for (; i < nv; i += step) {
        const Vec x = src[i];
        tf_cells<T, W>(x.v, m, a);
    }
    for (int64_t j = n_vec + t; j < n; j += step) {
        const T x[1] = {V[j]};
        tf_cells<T, 1>(x, m, a);
        if (++n4 % SUM_FLUSH == 0) a.sum.flush();
    }
    tf_finish(a, partials, counter, result, top);
}

// analytic V: a warp takes a run of 32 PARTS cells along x and evaluates them in
// FP64, PARTS a lane, unless the FP32 bound rules every one of them out.  What FP64
// costs a run whatever its cells hold (its place in y and z, the bound's coordinates) is
// shared by its cells, and a lane's evaluations are in flight together.  256^3 box,
// a solve whose mu lies above every cell of a harmonic trap: 1.14 ms without
// bounds, 1.62 with runs of 32 cells, 1.00 with the 128 that such rows get here;
// a shell's: 9.8, 2.66 and 2.16.
template <int PARTS>
__global__ void k_tf_analytic(PotDesc P, BoxD box, Limit m, double *partials, unsigned int *counter, double *result,
                              uint32_t *top)
{
    constexpr int RUN = 32 * PARTS;
    TfSum<double> a;
    const int lane = threadIdx.x & 31, nx = (int)box.nx;
    const int64_t nc = (nx + RUN - 1) / RUN, n = nc * box.ny * box.nz;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t u = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); u < n; u += nw) {
        const int64_t r = u / nc, k = r / box.ny;
        const int i0 = (int)(u - r * nc) * RUN, j = (int)(r - k * box.ny), i1 = min(i0 + RUN, nx) - 1;
        const double y = box.y0 + j * box.hy, z = box.z0 + (int)k * box.hz;
        if (!pot_may_select(P, m.t, (float)(box.x0 + i0 * box.hx), (float)(box.x0 + i1 * box.hx), (float)y, (float)y,
                            (float)z, (float)z))
            continue;
        double v[PARTS];
#pragma unroll
        for (int q = 0; q < PARTS; ++q) v[q] = eval_pot(P, box.x0 + (i0 + 32 * q + lane) * box.hx, y, z);
#pragma unroll
        for (int q = 0; q < PARTS; ++q)
            if (i0 + 32 * q + lane > i1) v[q] = (double)INFINITY;
        tf_cells<double, PARTS>(v, m, a);
    }
    tf_finish(a, partials, counter, result, top);
}

// One cell of each of `ns` equal stretches of the box, as float
constexpr int64_t TF_SAMPLES = 32768;
__global__ void k_tf_sample(VSource src, BoxD box, int64_t n, int64_t ns, float *out)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= ns) return;
    const int64_t lo = i * n / ns, len = (i + 1) * n / ns - lo;
    const int64_t lin = lo + (int64_t)((uint64_t)i * 2654435761ull % (uint64_t)len);
    double v0, v1;
    bool sel;
    cell_values(src, box, lin % box.nx, lin / box.nx % box.ny, lin / (box.nx * box.ny), v0, v1, sel);
    out[i] = (float)v0;
}

// Newton's method on the sample, with the target scaled to it: an estimate
// that starts the solve over the whole box, so FP32 is enough.  One block, the
// sample in its registers.
__global__ void __launch_bounds__(1024) k_tf_estimate(const float *v, int n, double target, double *result)
{
    constexpr int PER = (int)(TF_SAMPLES / 1024);
    __shared__ float s_m;
    __shared__ int s_stop;
    float x[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int at = threadIdx.x + 1024 * i;
        x[i] = at < n ? v[at] : INFINITY;
    }
    float m = INFINITY;
    double last = -1.0;
    for (int it = 0; it < 100; ++it) {
        float sum = 0.0f;
        int cnt = 0;
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (x[i] < m) {
                sum += x[i];
                ++cnt;
            }
        const double tot = block_sum((double)sum);
        const double c = block_sum((double)cnt);
        if (threadIdx.x == 0) {
            const double next = (target + tot) / c;
            s_stop = !(c > 0.0) || !(next < (double)m) || c == last || !isfinite(next);
            if (c > 0.0 && isfinite(next) && next < (double)m) s_m = (float)next;
            else s_m = m;
            last = c;
        }
        __syncthreads();
        m = s_m;
        if (s_stop) break;
        __syncthreads();
    }
    if (threadIdx.x == 0) *result = (double)m;
}

// Eq. (5): the mu at which the Thomas-Fermi atom number
//   F(mu) = sum over the box of max(mu - V, 0) / g dV
// equals N.  F is convex, increasing and piecewise linear in mu, so Newton's
// method
//   mu <- (g N / dV + sum_{V < mu} V) / #{V < mu}
// moves from any start to or above the root (a tangent lies below F), then
// down to it, and ends exactly once the set {V < mu} stops changing.  It
// starts from the solution on a sample of the cells, a per cent or so off:
// three to five passes over the box, where a start at mu = +inf took about
// eighteen (512^3 shell, FP32: 28 ms a solve of 1.55 ms passes, now 0.78 ms).
static int tf_mu_impl(const gpe_box *box, const VSource &src, double g, double N, double *mu, cudaStream_t st)
{
    if (!(g > 0)) return fail(GPE_ERR_ARG, "g must be > 0 for the Thomas-Fermi estimate");
    if (!(N > 0)) return fail(GPE_ERR_ARG, "N must be > 0");
    if (!mu) return fail(GPE_ERR_ARG, "mu is NULL");
    int dev = 0;
    GPE_TRY_CUDA(cudaGetDevice(&dev));
    const int64_t n = box->nx * box->ny * box->nz;
    const int64_t ns = std::min(n, TF_SAMPLES);
    const int blocks = (int)std::min<int64_t>((n + 1023) / 1024, (int64_t)sm_count(dev) * 8);
    const BoxD bd = boxd(*box);
    const double dV = box->hx * box->hy * box->hz;
    const double target = g * N / dV;
    // one workspace: results (sum, count, estimate), largest |V|, block
    // counter, block partial sums, sample
    struct Head {
        double res[3];
        uint32_t top;
        unsigned int counter;
    };
    char *ws = nullptr;
    GPE_TRY(dev_alloc_t(&ws, sizeof(Head) + 16 * (size_t)blocks + 4 * (size_t)ns));
    Head *head = reinterpret_cast<Head *>(ws), h{};
    double *partials = reinterpret_cast<double *>(ws + sizeof(Head));
    float *sample = reinterpret_cast<float *>(partials + 2 * blocks);
    auto pass = [&](double m) -> int {
        const Limit lim = limit_of(m);
        if (src.mode != 0) {
            // rows in as few runs of up to 128 cells as hold them, all of one length
            const int64_t p32 = (box->nx + 31) / 32, runs = (p32 + 3) / 4, parts = (p32 + runs - 1) / runs;
            const auto k = parts == 1 ? k_tf_analytic<1> : parts == 2 ? k_tf_analytic<2> : parts == 3 ? k_tf_analytic<3> : k_tf_analytic<4>;
            k<<<blocks, 256, 0, st>>>(src.p0, bd, lim, partials, &head->counter, head->res, &head->top);
        } else {
            const bool aligned = reinterpret_cast<uintptr_t>(src.dense) % 16 == 0;
            if (src.dtype == GPE_F64)
                k_tf_dense<double><<<blocks, 256, 0, st>>>((const double *)src.dense, n, aligned ? n / 2 * 2 : 0, lim,
                                                          partials, &head->counter, head->res, &head->top);
            else
                k_tf_dense<float><<<blocks, 256, 0, st>>>((const float *)src.dense, n, aligned ? n / 4 * 4 : 0, lim,
                                                         partials, &head->counter, head->res, &head->top);
        }
        GPE_LAUNCH_CHECK();
        GPE_TRY_CUDA(cudaMemcpyAsync(&h, head, sizeof h, cudaMemcpyDeviceToHost, st));
        GPE_TRY_CUDA(cudaStreamSynchronize(st));
        return GPE_OK;
    };
    // can the sum over every cell leave the finite range?  (the solve from
    // mu = +inf refuses such a potential)
    auto may_overflow = [&]() {
        double top;
        if (src.mode != 0) {
            double c[3] = {std::max(std::fabs(bd.x0), std::fabs(bd.x0 + (bd.nx - 1) * bd.hx)),
                           std::max(std::fabs(bd.y0), std::fabs(bd.y0 + (bd.ny - 1) * bd.hy)),
                           std::max(std::fabs(bd.z0), std::fabs(bd.z0 + (bd.nz - 1) * bd.hz))};
            const double *p = src.p0.p;
            if (src.p0.kind == GPE_POT_HARMONIC) {
                top = 0.5 * (p[0] * p[0] * c[0] * c[0] + p[1] * p[1] * c[1] * c[1] + p[2] * p[2] * c[2] * c[2]);
            } else {
                const double r = 1.0 + c[0] / p[1] + c[1] / p[2] + c[2] / p[3];
                top = 0.5 * p[0] * p[0] * r * r;
            }
        } else if (src.dtype == GPE_F64) {
            const uint64_t b = (uint64_t)(h.top + 1u) << 32;
            memcpy(&top, &b, 8);
        } else {
            float f;
            memcpy(&f, &h.top, 4);
            top = f;
        }
        return !(top * (double)n < 1e308);
    };
    auto solve = [&]() -> int {
        GPE_TRY_CUDA(cudaMemsetAsync(head, 0, sizeof(Head), st));
        k_tf_sample<<<(unsigned)((ns + 255) / 256), 256, 0, st>>>(src, bd, n, ns, sample);
        GPE_LAUNCH_CHECK();
        k_tf_estimate<<<1, 1024, 0, st>>>(sample, (int)ns, target * ((double)ns / (double)n), &head->res[2]);
        GPE_LAUNCH_CHECK();
        GPE_TRY_CUDA(cudaMemcpyAsync(&h, head, sizeof h, cudaMemcpyDeviceToHost, st));
        GPE_TRY_CUDA(cudaStreamSynchronize(st));
        double m = std::isfinite(h.res[2]) ? h.res[2] : INFINITY;
        bool from_any = m < INFINITY;  // the first pass may start below the root
        double count = -1.0;
        for (int it = 0; it < 200; ++it) {
            GPE_TRY(pass(m));
            const double sum = h.res[0], cnt = h.res[1];
            if (from_any && (!(cnt > 0.0) || may_overflow())) {  // from the start above every cell
                m = INFINITY;
                from_any = false;
                continue;
            }
            if (!(cnt > 0.0)) return fail(GPE_ERR_ARG, "Thomas-Fermi solve found no cell below mu (V not finite?)");
            const double next = (target + sum) / cnt;
            const bool same_set = cnt == count;
            count = cnt;
            if (!std::isfinite(next)) return fail(GPE_ERR_ARG, "Thomas-Fermi solve: non-finite mu (V not finite?)");
            if (same_set || (!from_any && !(next < m))) {
                *mu = std::min(m, next);
                return GPE_OK;
            }
            from_any = false;
            m = next;
        }
        *mu = m;
        return GPE_OK;
    };
    const int rc = solve();
    dev_free(ws);
    return rc;
}

}  // namespace gpe

extern "C" int gpe_tf_mu_dense(const gpe_box *box, const void *V, int V_dtype, int V_on_device, double g,
                               double N, double *mu, gpe_stream stream)
{
    GPE_TRY(check_box(box));
    cudaStream_t st = S(stream);
    const void *dptr = nullptr;
    void *owned = nullptr;
    GPE_TRY(stage_dense(box, V, V_dtype, V_on_device, &dptr, &owned, st));
    VSource src{};
    src.mode = 0;
    src.dense = dptr;
    src.dtype = V_dtype;
    src.cut0 = 0.0;
    int rc = tf_mu_impl(box, src, g, N, mu, st);
    if (owned) {
        cudaStreamSynchronize(st);
        dev_free(owned);
    }
    return rc;
}

extern "C" int gpe_tf_mu_analytic(const gpe_box *box, const gpe_potential *pot, double g, double N, double *mu,
                                  gpe_stream stream)
{
    GPE_TRY(check_box(box));
    GPE_TRY(check_pot(pot));
    VSource src{};
    src.mode = 1;
    src.p0 = potdesc(*pot);
    return tf_mu_impl(box, src, g, N, mu, S(stream));
}
