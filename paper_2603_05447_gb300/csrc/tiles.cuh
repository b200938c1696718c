// tiles.cuh -- the stencil kernels' unit of work: a tile of TILE consecutive
// stored segments of the packed layout, one segment a thread, whatever bricks
// they belong to.  Not part of the ABI.
//
// Per tile the grid builder (tiles.cu) keeps the list of the stored segments
// outside it that its stencils read (its halo) and, per segment, where each
// neighbour lies in the tile: as one of the tile's own segments (slots
// 0..TILE-1), as the zero slot (TILE: not stored, psi = 0 there) or as a halo
// segment (TILE+1 on).  So a kernel looks nothing up: own values come along
// one contiguous run, the halo by one gather, every lane has a segment.
//
// Why this shape.  The former unit, one warp per brick with the neighbours'
// segment ranks computed from bit masks, spent 330 of its 632 warp
// instructions a brick on the fill and left a fifth of the lanes idle.  On a
// thin shell's 8x8x4 bricks a tile of 128 reads 0.88 face segments and 0.29
// x-halo cells per own segment; 64 would read 1.05 and 0.58, 256 0.80 and
// 0.14, but neighbour slots of a 256-tile do not fit 10 bits in the worst
// case (128: 129 + 6 * 128 slots).  The lists cost 12.7 bytes a segment and
// pass, against 5.3 for the brick records, on 80 to 144 of data.
#pragma once

#include <algorithm>

#include "stencil.cuh"

namespace gpe {

// neighbour fields of a segment: 0-3 its -y +y -z +z segments, 4 and 5 the
// segments holding its -x and +x cells; with the 19-point stencil also 6-9 the
// (-y-z) (+y-z) (-y+z) (+y+z) segments, and 10-17 those holding the -x and +x
// cells of fields 0-3's rows (two each, in that order)
template <int NP>
struct TileFields {
    static constexpr int N = NP == 19 ? 18 : 6;
};

struct TileView {
    const uint2 *nbr;      // per segment: six 10-bit slots, three a word
    const uint4 *nbr19;    // 19-point grids: two uint4 of 12-bit slots, five a 64-bit word
    // per tile a row of `stride` entries: its count (whole | single << 16),
    // then the whole segments, and from the row's end the single cells (bit
    // 31: the segment's first cell, else its last)
    const uint32_t *halo;
    uint32_t nseg;         // stored segments
    int ntiles, stride;
    int pstr;              // slots of a plane of the shared tile
};

// Shared tile: planes of units (unit k of every slot's segment is contiguous),
// so that lanes with consecutive slots touch consecutive units.  Units of 16
// bytes give the widest loads; with the 19-point stencil, whose ten single end
// cells a segment would then lie 16 bytes apart and take four wavefronts a
// load instead of two (complex64), a unit is a cell.  1024^3 shell,
// complex64, single cells against 16 bytes: 19-point RK4 step 1.189 -> 1.153 ms,
// 7-point 0.620 -> 0.640 (more loads), real float imaginary time 0.604 -> 0.634.
template <typename CT, int NP>
struct TileMem {
    using U = typename std::conditional<NP == 19 || sizeof(CT) == 16, CT, uint4>::type;
    static constexpr int UPS = (int)(4 * sizeof(CT) / sizeof(U)), CPU_ = 4 / UPS;
    // plane stride with the units of a slot in distinct bank groups
    static int pstr(int nslot)
    {
        if (UPS == 4) return nslot;
        return nslot + ((UPS == 1 ? nslot % 8 : 4) - nslot % 8 + 8) % 8;
    }
    U *u;
    int p;
    __device__ __forceinline__ void get(int s, CT (&v)[4]) const
    {
#pragma unroll
        for (int k = 0; k < UPS; ++k) {
            const U w = u[k * p + s];
            const CT *c = reinterpret_cast<const CT *>(&w);
#pragma unroll
            for (int i = 0; i < CPU_; ++i) v[k * CPU_ + i] = c[i];
        }
    }
    __device__ __forceinline__ void put(int s, const CT (&v)[4]) const
    {
#pragma unroll
        for (int k = 0; k < UPS; ++k) {
            U w;
            CT *c = reinterpret_cast<CT *>(&w);
#pragma unroll
            for (int i = 0; i < CPU_; ++i) c[i] = v[k * CPU_ + i];
            u[k * p + s] = w;
        }
    }
    __device__ __forceinline__ CT *first(int s) const { return reinterpret_cast<CT *>(u + s); }
    __device__ __forceinline__ CT *last(int s) const
    {
        return reinterpret_cast<CT *>(u + (UPS - 1) * p + s) + (CPU_ - 1);
    }
};

// shared memory a block may have, less the reductions' static arrays (a tile
// needs at most 155 KB: 19-point, complex128, 2433 slots)
constexpr size_t TILE_SMEM_MAX = 208 * 1024;

// a segment's neighbour slots
template <int NP>
struct TileSlots {
    uint2 d;
    __device__ __forceinline__ void load(const TileView &T, uint32_t seg) { d = __ldg(T.nbr + seg); }
    __device__ __forceinline__ int operator()(int k) const
    {
        return (int)(((k < 3 ? d.x : d.y) >> (10 * (k % 3))) & 1023u);
    }
};
template <>
struct TileSlots<19> {
    unsigned long long q[4];
    __device__ __forceinline__ void load(const TileView &T, uint32_t seg)
    {
        const uint4 a = __ldg(T.nbr19 + 2 * (size_t)seg), b = __ldg(T.nbr19 + 2 * (size_t)seg + 1);
        q[0] = a.x | (unsigned long long)a.y << 32;
        q[1] = a.z | (unsigned long long)a.w << 32;
        q[2] = b.x | (unsigned long long)b.y << 32;
        q[3] = b.z | (unsigned long long)b.w << 32;
    }
    __device__ __forceinline__ int operator()(int k) const { return (int)((q[k / 5] >> (12 * (k % 5))) & 4095u); }
};

// a tile kernel's inverse square spacings and what LAP makes of them (7 points)
template <typename R>
struct TileCo {
    R ihx2, ihy2, ihz2;
    LapCo<R> k;
};
template <int NP, typename LAP, typename R>
__device__ __forceinline__ TileCo<R> tile_co(R ihx2, R ihy2, R ihz2)
{
    TileCo<R> co{ihx2, ihy2, ihz2, {}};
    if constexpr (NP == 7) co.k = lap_co<LAP>(ihx2, ihy2, ihz2);
    return co;
}

// L of a segment with values c and neighbour slots f: the Laplacians, or what
// LAP makes of them
template <int NP, typename LAP, typename CT, typename R>
__device__ __forceinline__ void tile_laplacian(const TileMem<CT, NP> &m, const TileSlots<NP> &f, const CT (&c)[4],
                                               const TileCo<R> &co, CT (&L)[4])
{
    // opposite neighbours are summed first and the centre term enters once:
    // L = (x- + x+) / hx^2 + (y- + y+) / hy^2 + (z- + z+) / hz^2 - c6 c
    CT ym[4], yp[4], zm[4], zp[4];
    m.get(f(0), ym);
    m.get(f(1), yp);
    m.get(f(2), zm);
    m.get(f(3), zp);
    const CT xm = *m.last(f(4)), xp = *m.first(f(5));
    if constexpr (NP != 19) {
        lap4<LAP>(xm, xp, ym, yp, zm, zp, c, co.k, L);
    } else {
        // App. B: the 7-point part plus w_ab (edges_ab - 2 faces_ab + 4 c) per
        // plane ab, w_ab = (1/h_a^2 + 1/h_b^2) / 12.  Each face pair lies in
        // two planes, so the face and centre terms fold into the 7-point form:
        //   x: 1/hx^2 - 2 (wxy + wxz), y: 1/hy^2 - 2 (wxy + wyz),
        //   z: 1/hz^2 - 2 (wxz + wyz), centre: c6 - 4 (wxy + wxz + wyz),
        // and only the three edge sums remain: + wxy exy + wxz exz + wyz eyz.
        const R ihx2 = co.ihx2, ihy2 = co.ihy2, ihz2 = co.ihz2, c6 = (R)2 * (ihx2 + ihy2 + ihz2);
        const R wxy = (ihx2 + ihy2) / (R)12, wxz = (ihx2 + ihz2) / (R)12, wyz = (ihy2 + ihz2) / (R)12;
        const R ax = ihx2 - (R)2 * (wxy + wxz), ay = ihy2 - (R)2 * (wxy + wyz), az = ihz2 - (R)2 * (wxz + wyz);
        const R c19 = c6 - (R)4 * (wxy + wxz + wyz);
        CT eyz[4], t4[4];
        m.get(f(6), eyz);
#pragma unroll
        for (int k = 7; k < 10; ++k) {
            m.get(f(k), t4);
#pragma unroll
            for (int i = 0; i < 4; ++i) eyz[i] = vadd(eyz[i], t4[i]);
        }
        const CT yml = *m.last(f(10)), ymr = *m.first(f(11)), ypl = *m.last(f(12)), ypr = *m.first(f(13));
        const CT zml = *m.last(f(14)), zmr = *m.first(f(15)), zpl = *m.last(f(16)), zpr = *m.first(f(17));
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const CT l = i == 0 ? xm : c[i - 1];
            const CT rr = i == 3 ? xp : c[i + 1];
            const CT exy = vadd(vadd(i == 0 ? yml : ym[i - 1], i == 3 ? ymr : ym[i + 1]),
                                vadd(i == 0 ? ypl : yp[i - 1], i == 3 ? ypr : yp[i + 1]));
            const CT exz = vadd(vadd(i == 0 ? zml : zm[i - 1], i == 3 ? zmr : zm[i + 1]),
                                vadd(i == 0 ? zpl : zp[i - 1], i == 3 ? zpr : zp[i + 1]));
            if constexpr (sizeof(R) == 8 && !std::is_same<LAP, LapFull>::value) {
                // the centre comes last, so that only its addition rounds at the result's size
                const CT faces = LapRhs::of(rr, l, yp[i], ym[i], zp[i], zm[i], c[i], LAP::coef(ax), LAP::coef(ay), LAP::coef(az), c19);
                L[i] = with_centre<LAP>(c[i], edgev(faces, exy, exz, eyz[i], LAP::coef(wxy), LAP::coef(wxz), LAP::coef(wyz)), c19);
            } else {
                L[i] = edgev(LAP::of(rr, l, yp[i], ym[i], zp[i], zm[i], c[i], LAP::coef(ax), LAP::coef(ay), LAP::coef(az), c19),
                             exy, exz, eyz[i], LAP::coef(wxy), LAP::coef(wxz), LAP::coef(wyz));
            }
        }
    }
}

// Bring n bytes (a multiple of 16) from p into L2, by one thread
__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t n)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(n) : "memory");
}

// A transform of the values as they are loaded: none, or one whose operands
// (for a segment or for one cell) are loaded beside the values
struct Plain {
    struct P4 {};
    struct P1 {};
    __device__ __forceinline__ P4 load4(uint32_t) const { return {}; }
    __device__ __forceinline__ P1 load1(uint32_t) const { return {}; }
    template <typename CT>
    __device__ __forceinline__ void seg(CT (&)[4], const P4 &) const {}
    template <typename CT>
    __device__ __forceinline__ void cell(CT &, const P1 &) const {}
};

// a thread's entries of a tile's halo list: two whole segments, one single cell
struct TileList {
    uint32_t cnt = 0, e0 = 0, e1 = 0, es = 0;
    __device__ __forceinline__ void fetch(const TileView &T, uint32_t tile)
    {
        if (tile >= (uint32_t)T.ntiles) return;
        const int tid = threadIdx.x;
        const uint32_t *row = T.halo + (size_t)tile * T.stride;
        cnt = __ldg(row);
        if (1 + tid < T.stride) {
            e0 = __ldg(row + 1 + tid);
            es = __ldg(row + T.stride - 1 - tid);
        }
        if (1 + tid + TILE < T.stride) e1 = __ldg(row + 1 + tid + TILE);
    }
};

// Every tile kernel begins here: its first tile's list is fetched (the lists
// never change), its own dependent launch is let go, and then it waits for the
// kernels before it.  Launched with programmatic stream serialisation
// (tile_run) it is resident, with its list on the way, while they end; else
// both instructions return at once.
__device__ __forceinline__ TileList tile_begin(const TileView &T)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    TileList l;
    l.fetch(T, blockIdx.x);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    return l;
}

struct EveryTile {
    __device__ __forceinline__ bool operator()(uint32_t) const { return true; }
};

// Run body(idx, pre, c, L) over every segment of the tiles blockIdx.x,
// blockIdx.x + gridDim.x, ...: idx its first cell's packed index, pre what
// load(idx) returned, c[4] its values and L[4] their Laplacians, of src
// transformed by xf.  Called once by the whole block of TILE threads.
// Everything of a tile is in flight before anything is waited for: a thread
// loads its own segment, its operands, its neighbour slots and its entries of
// the halo, whose list it holds since the tile before; and one thread has had
// the tile's runs brought into L2 a tile ahead (prefetch(first cell, cells)
// adds the operands' runs).  Values go to the shared tile through registers:
// cp.async into the tile's planes moved 1.3 times the L2 bytes and, with two
// buffered tiles a block, ran a third slower.
//
// setup(tile), uniform over the block, runs before each tile, may change what
// xf and co refer to, and says whether to take it.
template <int NP, typename LAP = LapFull, typename CT, typename R, typename XF, typename SETUP, typename PREF,
          typename LOAD, typename BODY>
__device__ __forceinline__ void tile_loop(const TileView &T, TileList list, const CT *src, const XF &xf,
                                          const TileCo<R> &co, SETUP setup, PREF prefetch, LOAD load, BODY body)
{
    extern __shared__ __align__(16) unsigned char gpe_smem[];
    using M = TileMem<CT, NP>;
    const M m{reinterpret_cast<typename M::U *>(gpe_smem), T.pstr};
    const int tid = threadIdx.x;
    const uint32_t step = gridDim.x, nt = (uint32_t)T.ntiles;
    auto cell_of = [](uint32_t e) { return 4u * (e & 0x7fffffffu) + ((e >> 31) ? 0u : 3u); };
    auto cell_at = [&](int sl, uint32_t e) -> CT & { return *((e >> 31) ? m.first(sl) : m.last(sl)); };
    if (tid < M::UPS) m.u[tid * m.p + TILE] = typename M::U{};  // the zero slot
    for (uint32_t tile = blockIdx.x; tile < nt; tile += step) {
        if (!setup(tile)) {
            list.fetch(T, tile + step);
            continue;
        }
        const uint32_t seg = tile * TILE + tid, idx = 4u * seg;
        const bool in = seg < T.nseg;
        const int nwhole = list.cnt & 0xffff, nsingle = list.cnt >> 16;
        const uint32_t w0 = list.e0, w1 = list.e1, s0 = list.es;
        CT c[4], h0[4], h1[4], hs = czero<CT>();
        typename std::decay<decltype(load(0u))>::type pre{};
        typename XF::P4 x0{}, x1{};
        typename XF::P1 xs{};
        TileSlots<NP> f{};
        if (in) {
            ld4<false>(src + idx, c);
            f.load(T, seg);
            pre = load(idx);
        }
        if (tid < nwhole) {
            ld4<false>(src + 4 * (size_t)w0, h0);
            x0 = xf.load4(4u * w0);
        }
        if (tid + TILE < nwhole) {
            ld4<false>(src + 4 * (size_t)w1, h1);
            x1 = xf.load4(4u * w1);
        }
        if (tid < nsingle) {
            hs = src[cell_of(s0)];
            xs = xf.load1(cell_of(s0));
        }
        list.fetch(T, tile + step);
        if (tid == 0 && tile + 2 * step < nt) {
            prefetch_l2(T.halo + (size_t)(tile + 2 * step) * T.stride, T.stride * 4u);
        }
        if (tid == 0 && tile + step < nt) {
            const uint32_t s1 = (tile + step) * TILE, own = min((uint32_t)TILE, T.nseg - s1) & ~1u;
            if (own > 0) {
                prefetch_l2(src + 4 * (size_t)s1, own * 4u * (uint32_t)sizeof(CT));
                if constexpr (NP == 19) prefetch_l2(T.nbr19 + 2 * (size_t)s1, own * 32u);
                else prefetch_l2(T.nbr + s1, own * 8u);
                prefetch(4u * s1, own * 4u);
            }
        }
        __syncthreads();  // the previous tile has been read
        if (in) {
            if constexpr (!std::is_same<XF, Plain>::value) xf.own(c, pre);  // the own operands serve the transform
            m.put(tid, c);
        }
        if (tid < nwhole) {
            xf.seg(h0, x0);
            m.put(TILE + 1 + tid, h0);
        }
        if (tid + TILE < nwhole) {
            xf.seg(h1, x1);
            m.put(2 * TILE + 1 + tid, h1);
        }
        if (tid < nsingle) {
            xf.cell(hs, xs);
            cell_at(TILE + 1 + nwhole + tid, s0) = hs;
        }
        if (nwhole > 2 * TILE || nsingle > TILE) {  // masks with unusually many halo segments
            const uint32_t *row = T.halo + (size_t)tile * T.stride;
            for (int t = tid + 2 * TILE; t < nwhole; t += TILE) {
                const uint32_t e = __ldg(row + 1 + t);
                ld4<false>(src + 4 * (size_t)e, h0);
                xf.seg(h0, xf.load4(4u * e));
                m.put(TILE + 1 + t, h0);
            }
            for (int t = tid + TILE; t < nsingle; t += TILE) {
                const uint32_t e = __ldg(row + T.stride - 1 - t);
                hs = src[cell_of(e)];
                xf.cell(hs, xf.load1(cell_of(e)));
                cell_at(TILE + 1 + nwhole + t, e) = hs;
            }
        }
        __syncthreads();
        if (in) {
            CT L[4];
            tile_laplacian<NP, LAP>(m, f, c, co, L);
            body(idx, pre, c, L);
        }
    }
}

// ------------------------------------------------------------ launches
// a grid's tiles for values of type CT, and the shared memory of a block
struct TileLaunch {
    TileView T;
    size_t smem;
};
template <typename CT, int NP>
inline TileLaunch tile_launch(const TileTab &t)
{
    using M = TileMem<CT, NP>;
    const int pstr = M::pstr(t.nslot);
    return {TileView{t.d_nbr, t.d_nbr19, t.d_halo, t.nseg, t.ntiles, t.stride, pstr},
            sizeof(typename M::U) * (size_t)(M::UPS * pstr)};
}

// blocks of a launch over n tiles: one a tile, at most the resident ones.  A
// tile kernel may use as much shared memory as a block can have, so that grids
// of different halo sizes can launch it from any thread.
template <typename K>
inline unsigned tile_blocks(K kernel, int nsm, int n, size_t smem)
{
    const int64_t res = (int64_t)nsm * blocks_per_sm((const void *)kernel, TILE, smem, TILE_SMEM_MAX);
    return (unsigned)(res < n ? res : n);
}

// blocks an SM: registers of 85 (single; 102 with the 19-point stencil, whose
// RK4 step spilled at 85: 1.153 -> 1.024 ms on the 1024^3 shell) and 168 (double) a
// thread
constexpr int tile_blocks_f(int np) { return np == 19 ? 5 : 6; }
#define GPE_TILE_BOUNDS(R, NP) __launch_bounds__(TILE, sizeof(R) == 4 ? tile_blocks_f(NP) : 3)

// One RK4 stage.  1024^3 shell, 8x8x4 bricks, per step of four: complex64
// 0.776 -> 0.622 ms (4.0 GB, of which 0.4 GB slots and halo lists: 6.5 TB/s,
// 0.95 of the copy bandwidth, so bytes bound it now); complex128 8.65 -> 4.23
// ms (full lanes instead of four fifths: 6.75; 90 instead of 108 FP64
// instructions a cell and step, LapRhs, active_v and the split third: 5.44;
// the neighbour sums in integers, sum6: 4.45, their products behind a branch 4.23; an FP64 instruction takes 16
// cycles of an SM whatever its lanes do).  Single precision, six blocks an SM
// (85 registers): 0.626 ms, seven 0.634, eight with spills 0.645; double, three
// blocks (168 registers) are 1.5 % ahead of two; blended two, which three lose 1 % to.
// One block a tile instead of looping blocks: 8 % slower (no tile ahead to prefetch).
template <typename R, bool BLEND, int ST, int NP, bool FX = true>
__global__ void __launch_bounds__(TILE, sizeof(R) == 4 ? tile_blocks_f(NP) : (BLEND || NP == 19 ? 2 : 3)) k_rk4_tile(const RkArgs<R> a, const TileView T)
{
    using CT = typename Cx<R>::T;
    using B = Rk4Body<R, BLEND, false, ST>;
    using LAP = LapIn<LapRhs, FX>;
    const auto co = tile_co<NP, LAP>(a.ihx2, a.ihy2, a.ihz2);  // before the wait
    const TileList list = tile_begin(T);
    const B body(a, BLEND ? (R)__ldcg(a.stab) : (R)0);
    tile_loop<NP, LAP>(T, list, body.yin(), Plain(), co, EveryTile(),
                  [&](uint32_t idx, uint32_t n) {
                      prefetch_l2(a.V0 + idx, n * (uint32_t)sizeof(R));
                      if constexpr (BLEND) prefetch_l2(a.V1 + idx, n * (uint32_t)sizeof(R));
                      if constexpr (ST > 0) prefetch_l2((ST == 3 ? a.w : a.y0) + idx, n * (uint32_t)sizeof(CT));
                  },
                  [&](uint32_t idx) { return body.load(idx); }, body);
}

// Launch a tile kernel on `grid` blocks (tile_blocks).  On grids of up to
// PDL_TILES tiles a block the launch may overlap the end of the kernel before:
// the gap between kernels, a block's start and the way to its first list are
// most of a one-tile kernel's time and still 1 to 2 us of the 30 to 70 of a
// 512^3 shell's.  Measured, without and with: 12 RK4 steps of a 20-cell shell 1.07
// -> 0.70 ms, ten real-float imaginary-time steps of the 512^3 shell 0.642 ->
// 0.600 ms, its RKCK steps 2.584 -> 2.477; on the 1024^3 shell (70 tiles a
// block) RK4 19.96 -> 20.24 ms, since waiting blocks take room from running ones.
constexpr int PDL_TILES = 40;
template <typename... KArgs, typename... Args>
inline int tile_run(void (*k)(KArgs...), unsigned grid, const TileLaunch &L, cudaStream_t s, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(TILE);
    cfg.dynamicSmemBytes = L.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = (int64_t)L.T.ntiles <= (int64_t)PDL_TILES * grid ? 1 : 0;
    GPE_TRY_CUDA(cudaLaunchKernelEx(&cfg, k, args...));
    count_launch();
    return GPE_OK;
}

// Does fixed point serve a grid's sums?  (lap_co's rule for the spacings' ratio.)
// If not, the double-precision 7-point passes of single states take the FP64
// form as an instance of their own.  Eight steps of a 96 x 96 x 32 trap with
// spacings 1 : 1 : 3, complex128: RK4 804 us with sums that look at their values
// before they turn to it, 652 so; imaginary time 484 and 414.  Both forms behind a
// branch in one kernel: equal spacings 1 to 7 % slower (registers).
inline bool fixed_spacings(const gpe_box &b)
{
    const double x = 1.0 / (b.hx * b.hx), y = 1.0 / (b.hy * b.hy), z = 1.0 / (b.hz * b.hz);
    const double inv = 1.0 / std::max(x, std::max(y, z));
    return x * inv >= 0.125 && y * inv >= 0.125 && z * inv >= 0.125;
}
// are there two instances of a kernel?
template <typename R, int NP>
constexpr bool two_forms()
{
    return sizeof(R) == 8 && NP == 7;
}

// the four stage kernels, static (blend false) or blended
template <typename R, int NP>
struct Rk4Tiles {
    using K = void (*)(RkArgs<R>, TileView);
    static K get(bool blend, int st, bool fixed)
    {
        constexpr bool F = !two_forms<R, NP>();
        static const K t[2][2][4] = {{{k_rk4_tile<R, false, 0, NP, F>, k_rk4_tile<R, false, 1, NP, F>,
                                       k_rk4_tile<R, false, 2, NP, F>, k_rk4_tile<R, false, 3, NP, F>},
                                      {k_rk4_tile<R, true, 0, NP, F>, k_rk4_tile<R, true, 1, NP, F>,
                                       k_rk4_tile<R, true, 2, NP, F>, k_rk4_tile<R, true, 3, NP, F>}},
                                     {{k_rk4_tile<R, false, 0, NP>, k_rk4_tile<R, false, 1, NP>,
                                       k_rk4_tile<R, false, 2, NP>, k_rk4_tile<R, false, 3, NP>},
                                      {k_rk4_tile<R, true, 0, NP>, k_rk4_tile<R, true, 1, NP>,
                                       k_rk4_tile<R, true, 2, NP>, k_rk4_tile<R, true, 3, NP>}}};
        return t[fixed ? 1 : 0][blend ? 1 : 0][st];
    }
};

}  // namespace gpe
