// stencil.cuh -- device building blocks shared by the stencil kernels of
// libgpeshell (steps, batches, adjoint): the packed segment layout, per-cell
// arithmetic, the RK4 stages, the ramp schedule and small reductions; and the
// per-warp brick tile of the wavefront schedules.  Not part of the ABI.
#pragma once

#include "gpe_internal.cuh"

#include <type_traits>

namespace gpe {

// The wavefront kernels run one brick per warp; a block holds NW warps, each with
// its own shared-memory workspace (brick tile with face halo, the 7 brick
// records and the list of stored segments), passed as dynamic shared memory.
#ifndef GPE_NW_F
#define GPE_NW_F 8
#endif
// fetch the records of a warp's next brick while it processes the current one
#ifndef GPE_REC_AHEAD
#define GPE_REC_AHEAD 1
#endif
template <typename R>
struct KernelCfg {
    static constexpr int NW = sizeof(R) == 4 ? GPE_NW_F : 4;  // warps per block
    static constexpr int THREADS = 32 * NW;
};

// Minimum resident blocks per SM requested from the register allocator:
// as many as the shared-memory workspaces allow (228 KiB per SM, 1 KiB
// reserved per block), at most GPE_MINB_F (single precision) or a kernel's own
// number in double precision, whose forms need more registers: three, but two for
// the blended steps of WAVE2, which at three spill 272 bytes a thread around their
// calls of sum6.  Eight such steps, FP64 sums, sum6 at three blocks and at two: 48-cell
// ramp with spacings 1 : 1.2 : 1.08 2062, 2514 and 2009 us, 160-cell ramp with equal
// ones 8830, 7553 and 7106.  (WAVE: 1717 -> 1267 and 7668 -> 8116 us, static 6356 ->
// 7492: not taken.)
#ifndef GPE_MINB_F
#define GPE_MINB_F 4
#endif
// (D: blocks of the double-precision form)
#define GPE_BOUNDS(R, D) __launch_bounds__(KernelCfg<R>::THREADS, (min_blocks<R, BX, BY, BZ>(D)))
// ------------------------------------------------------------ packed layout
// supported brick shapes (shape id, BX, BY, BZ)
#define GPE_SHAPES(M) \
    M(0, 8, 8, 8)     \
    M(1, 8, 8, 4)     \
    M(2, 8, 4, 4)

struct GridView {
    const int32_t *nbr;
    const BrickRec *rec;
    const BrickRec *rec7;   // per brick: its record, then its six face neighbours' (empty if absent)
    int64_t nb;
};

inline GridView view(const gpe_grid *g) { return GridView{g->d_nbr, g->d_rec, g->d_rec7, g->nb}; }

// segment geometry of a brick shape (BX must be 8: two segments per row)
template <int BX, int BY, int BZ>
struct Seg {
    static_assert(BX == 8, "bricks are 8 cells long in x");
    static constexpr int SX = BX / 4;          // segments per x-row
    static constexpr int PLANE = SX * BY;      // segments per z-plane (divides 32)
    static constexpr int NSEG = PLANE * BZ;    // segments per brick
    static constexpr int NIT = NSEG / 32;      // warp iterations per brick
    static_assert(32 % PLANE == 0 && NSEG % 32 == 0, "brick shape must tile the warp");
};

// Values are complex (float2, double2) or, for real-valued imaginary-time
// states, real (float, double); these helpers serve both.
template <typename CT>
__host__ __device__ constexpr bool is_cplx()
{
    return !std::is_arithmetic<CT>::value;
}
template <typename CT>
struct RealOf {
    using T = CT;
};
template <>
struct RealOf<float2> {
    using T = float;
};
template <>
struct RealOf<double2> {
    using T = double;
};

// Packed single-precision pairs: the f32x2 add / multiply / fused
// multiply-add instructions of sm_100 and later act on both halves of a
// 64-bit register pair, i.e. on the real and imaginary parts of a complex64
// value at once, each half rounded exactly as the scalar instruction would
// round it.  They halve the arithmetic instruction count of the complex64
// stencils without changing any result.
__device__ __forceinline__ unsigned long long f2pk(float2 a)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
    return r;
}
__device__ __forceinline__ float2 f2up(unsigned long long r)
{
    float2 a;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
    return a;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2pk(a)), "l"(f2pk(b)));
    return f2up(d);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b)  // a - b
{
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2pk(a)), "l"(f2pk(b)));
    return f2up(d);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2pk(a)), "l"(f2pk(b)));
    return f2up(d);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)  // a * b + c, one rounding per half
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(f2pk(a)), "l"(f2pk(b)), "l"(f2pk(c)));
    return f2up(d);
}
__device__ __forceinline__ float2 dup2(float f) { return make_float2(f, f); }

template <typename CT>
__device__ __forceinline__ CT czero()
{
    if constexpr (is_cplx<CT>()) {
        CT z;
        z.x = 0;
        z.y = 0;
        return z;
    } else {
        return CT(0);
    }
}
// |v|^2
template <typename CT>
__device__ __forceinline__ typename RealOf<CT>::T norm2(const CT &v)
{
    if constexpr (is_cplx<CT>())
        return v.x * v.x + v.y * v.y;
    else
        return v * v;
}
// v * f, f real
__device__ __forceinline__ float2 scale(float2 v, float f) { return mul2(v, dup2(f)); }
template <typename CT, typename R>
__device__ __forceinline__ CT scale(CT v, R f)
{
    if constexpr (is_cplx<CT>()) {
        v.x *= f;
        v.y *= f;
        return v;
    } else {
        return v * f;
    }
}
// c + a L, a real
__device__ __forceinline__ float2 axpy(const float2 &c, float a, const float2 &L) { return fma2(dup2(a), L, c); }
__device__ __forceinline__ float axpy(float c, float a, float L) { return __fmaf_rn(a, L, c); }
template <typename CT, typename R>
__device__ __forceinline__ CT axpy(const CT &c, R a, const CT &L)
{
    if constexpr (is_cplx<CT>()) {
        CT o;
        o.x = c.x + a * L.x;
        o.y = c.y + a * L.y;
        return o;
    } else {
        return c + a * L;
    }
}
// Re(conj(a) b)
template <typename CT>
__device__ __forceinline__ typename RealOf<CT>::T dotre(const CT &a, const CT &b)
{
    if constexpr (is_cplx<CT>())
        return a.x * b.x + a.y * b.y;
    else
        return a * b;
}
__device__ __forceinline__ float2 vadd(const float2 &a, const float2 &b) { return add2(a, b); }
template <typename CT>
__device__ __forceinline__ CT vadd(const CT &a, const CT &b)
{
    if constexpr (is_cplx<CT>()) {
        CT o;
        o.x = a.x + b.x;
        o.y = a.y + b.y;
        return o;
    } else {
        return a + b;
    }
}
// L + wxy exy + wxz exz + wyz eyz: the edge terms of App. B's 19-point
// stencil added to its face-and-centre part
__device__ __forceinline__ float2 edgev(const float2 &L, const float2 &exy, const float2 &exz, const float2 &eyz,
                                        float wxy, float wxz, float wyz)
{
    return fma2(dup2(wyz), eyz, fma2(dup2(wxz), exz, fma2(dup2(wxy), exy, L)));
}
__device__ __forceinline__ float edgev(float L, float exy, float exz, float eyz, float wxy, float wxz, float wyz)
{
    return __fmaf_rn(wyz, eyz, __fmaf_rn(wxz, exz, __fmaf_rn(wxy, exy, L)));
}
template <typename CT, typename R>
__device__ __forceinline__ CT edgev(const CT &L, const CT &exy, const CT &exz, const CT &eyz, R wxy, R wxz, R wyz)
{
    if constexpr (is_cplx<CT>()) {
        CT o;
        o.x = L.x + wxy * exy.x + wxz * exz.x + wyz * eyz.x;
        o.y = L.y + wxy * exy.y + wxz * exz.y + wyz * eyz.y;
        return o;
    } else {
        return L + wxy * exy + wxz * exz + wyz * eyz;
    }
}
// one component of the 7-point Laplacian (Eq. (B1)) from opposite-neighbour
// sums: (x- + x+)/hx^2 + (y- + y+)/hy^2 + (z- + z+)/hz^2 - c6 c.  In single
// precision the order of the roundings is fixed explicitly, the same as the
// packed complex64 form (lapv below), so that a real-valued float state and a
// complex64 state with zero imaginary part compute bit-identical values.
__device__ __forceinline__ float lap1(float xp, float xm, float yp, float ym, float zp, float zm, float c, float ihx2,
                                      float ihy2, float ihz2, float c6)
{
    float t = __fmul_rn(__fadd_rn(xp, xm), ihx2);
    t = __fmaf_rn(__fadd_rn(yp, ym), ihy2, t);
    t = __fmaf_rn(__fadd_rn(zp, zm), ihz2, t);
    return __fmaf_rn(-c6, c, t);
}
template <typename R>
__device__ __forceinline__ R lap1(R xp, R xm, R yp, R ym, R zp, R zm, R c, R ihx2, R ihy2, R ihz2, R c6)
{
    return (xp + xm) * ihx2 + (yp + ym) * ihy2 + (zp + zm) * ihz2 - c6 * c;
}
// complex64: the same operations as lap1 on both parts at once
__device__ __forceinline__ float2 lapv(const float2 &xp, const float2 &xm, const float2 &yp, const float2 &ym,
                                       const float2 &zp, const float2 &zm, const float2 &c, float ihx2, float ihy2,
                                       float ihz2, float c6)
{
    float2 t = mul2(add2(xp, xm), dup2(ihx2));
    t = fma2(add2(yp, ym), dup2(ihy2), t);
    t = fma2(add2(zp, zm), dup2(ihz2), t);
    return fma2(dup2(-c6), c, t);
}
template <typename CT, typename R>
__device__ __forceinline__ CT lapv(const CT &xp, const CT &xm, const CT &yp, const CT &ym, const CT &zp, const CT &zm,
                                   const CT &c, R ihx2, R ihy2, R ihz2, R c6)
{
    if constexpr (is_cplx<CT>()) {
        CT L;
        L.x = lap1(xp.x, xm.x, yp.x, ym.x, zp.x, zm.x, c.x, ihx2, ihy2, ihz2, c6);
        L.y = lap1(xp.y, xm.y, yp.y, ym.y, zp.y, zm.y, c.y, ihx2, ihy2, ihz2, c6);
        return L;
    } else {
        return lap1(xp, xm, yp, ym, zp, zm, c, ihx2, ihy2, ihz2, c6);
    }
}

// Whether a cell is active, from its potential (+inf, or NaN, marks the inactive
// cells of stored segments) or its propagator (negative there).  Double values
// are tested by their high words: an FP64 comparison costs as much as an FP64
// multiplication.
__device__ __forceinline__ bool active_v(float V) { return V < INFINITY; }
__device__ __forceinline__ bool active_v(double V)
{
    const int hi = __double2hiint(V);
    return (hi & 0x7fffffff) < 0x7ff00000 || (hi == (int)0xfff00000 && __double2loint(V) == 0);  // finite or -inf
}
__device__ __forceinline__ bool active_e(float E) { return E >= 0.0f; }
__device__ __forceinline__ bool active_e(double E) { return __double2hiint(E) >= 0; }

// Coefficients of a cell's neighbour sums, made once a kernel (lap_co)
template <typename R>
struct LapCo {
    R ax, ay, az, c6;
};
// Double precision: the sums ax (x- + x+) + ay (y- + y+) + az (z- + z+) of one
// part of a cell in integers.  An FP64 instruction takes 16 cycles of an SM and the six
// that a sum needs were half of what bounds the complex128 passes, while
// the integer pipes stood idle.  The six values become 64-bit fixed point with the
// largest one's exponent, 59 bits below its leading one, and add without
// rounding; the coefficients are ref q, q a 64-bit fraction, so that one
// multiplication by ref remains.  The error is absolute: each of the six cuts (and
// of the products with q) loses less than 2^-59 of the largest neighbour, so a sum
// is good to 9 2^-59 of that times ref, and to a few 2^-53 of itself.  FP64
// additions round at 2^-53 of the sums they meet, 64 times as much for neighbours
// of one sign; but where opposite neighbours cancel exactly they would keep
// smaller ones whole, of which nothing is left here below 2^-59 of the largest.
// With q >= 1/8 the largest neighbour's own share of the sum is at least 2^-3 of
// it, so its cut stays below an FP64 rounding of that share; spacings more unequal
// than that, values that are not finite and values far outside any state's
// range take the FP64 form.  Errors against extended precision (80 bits), FP64
// sums and these: 40 RK4 steps of the 64^3 trap 6.75e-16 and 6.0e-16 (spacings
// 1 : 1.05 : 0.97: 6.9e-16 and 6.0e-16), 50 imaginary-time steps 1.454e-15 and
// 1.458e-15, where seeds differ by 2 %.
// RK4 step in complex128, FP64 sums and these: 1024^3 shell 5.44 -> 4.23 ms, 96^3
// trap 0.170 -> 0.137; with unequal spacings 0.917 -> 0.764 (200-cell shell).
template <>
struct LapCo<double> {
    double ax, ay, az, c6;
    double ref;                     // the largest coefficient
    unsigned long long qx, qy, qz;  // 2^64 a / ref; 0: a = ref
    int lo, hi;                     // exponents (of the largest value) that fixed point serves
    __device__ __forceinline__ bool fixed() const { return lo <= hi; }
};
template <typename LAP>
__device__ __forceinline__ LapCo<float> lap_co(float ihx2, float ihy2, float ihz2)
{
    return {LAP::coef(ihx2), LAP::coef(ihy2), LAP::coef(ihz2), 2.0f * (ihx2 + ihy2 + ihz2)};
}
template <typename LAP>
__device__ __forceinline__ LapCo<double> lap_co(double ihx2, double ihy2, double ihz2)
{
    LapCo<double> k{};
    k.ax = LAP::coef(ihx2);
    k.ay = LAP::coef(ihy2);
    k.az = LAP::coef(ihz2);
    k.c6 = 2.0 * (ihx2 + ihy2 + ihz2);
    if constexpr (!LAP::FIXED) return k;
    k.ref = k.ax;
    k.qx = k.qy = k.qz = 0;
    bool usual = true;
    if (ihx2 != ihy2 || ihx2 != ihz2) {
        k.ref = LAP::coef(fmax(ihx2, fmax(ihy2, ihz2)));
        const double two64 = 18446744073709551616.0, inv = 1.0 / k.ref;
        auto frac = [&](double a) -> unsigned long long {
            const double q = a * inv, rest = __fma_rn(-q, k.ref, a) * inv;
            usual = usual && q >= 0.125;
            return a == k.ref ? 0ull : __double2ull_rn(q * two64) + (unsigned long long)__double2ll_rn(rest * two64);
        };
        k.qx = frac(k.ax);
        k.qy = frac(k.ay);
        k.qz = frac(k.az);
    }
    // the result's factor ref 2^(e - 1082) has to be a normal number, and values
    // 64 binary orders below the largest have to be nothing
    const int er = (__double2hiint(k.ref) >> 20) & 0x7ff;
    k.lo = usual && er >= 64 && er <= 1983 ? max(64, 1083 - er) : 0x7fffffff;
    k.hi = min(2046, 3128 - er);
    return k;
}

__device__ __forceinline__ double i64_to_double(long long S)
{
    // as __ll2double_rn but for ties, off the FP64 pipe
    const int sg = (int)(S >> 63);
    unsigned long long a = (unsigned long long)((S ^ (long long)sg) - (long long)sg);
    const int z = __clzll((long long)a);
    a <<= z & 63;
    const unsigned hi = (unsigned)(a >> 32), lo = (unsigned)a;
    const unsigned long long m = (unsigned long long)((hi >> 11) + ((unsigned)(1085 - z) << 20)) << 32 |
                                 __funnelshift_r(lo, hi, 11);
    const long long r = (long long)(m + ((lo >> 10) & 1u));  // a carry moves the exponent on
    return S == 0 ? 0.0 : __longlong_as_double(r | (S & (long long)0x8000000000000000ull));
}
// S q 2^-64, cut towards zero: of opposite values the results are opposite, as
// FP64's are (an odd state stays exactly odd)
__device__ __forceinline__ long long mul_frac(long long S, unsigned long long q)
{
    const long long m = (long long)__umul64hi((unsigned long long)llabs(S), q);
    return S < 0 ? -m : m;
}
static __device__ __noinline__ double sum6_fp64(double xp, double xm, double yp, double ym, double zp, double zm,
                                                double ax, double ay, double az)
{
    return __fma_rn(az, zp + zm, __fma_rn(ay, yp + ym, ax * (xp + xm)));
}
__device__ __forceinline__ double sum6(double xp, double xm, double yp, double ym, double zp, double zm,
                                       const LapCo<double> &k)
{
    const double v[6] = {xp, xm, yp, ym, zp, zm};
    int e[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) e[i] = (__double2hiint(v[i]) >> 20) & 0x7ff;
    const int em = max(max(max(e[0], e[1]), max(e[2], e[3])), max(e[4], e[5]));
    if (em < k.lo || em > k.hi) {
        long long any = 0;
#pragma unroll
        for (int i = 0; i < 6; ++i) any |= __double_as_longlong(v[i]) & 0x7fffffffffffffffll;
        return any == 0 ? 0.0 : sum6_fp64(xp, xm, yp, ym, zp, zm, k.ax, k.ay, k.az);
    }
    long long S[3];
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        S[p] = 0;
        int neg = 0;
#pragma unroll
        for (int i = 2 * p; i < 2 * p + 2; ++i) {
            const int hi = __double2hiint(v[i]), lo = __double2loint(v[i]);
            const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
            unsigned long long x;  // the mantissa, its leading one at bit 59 - (em - e); shifts beyond 63 give 0
            asm("{.reg .b64 t; mov.b64 t, {%1, %2}; shr.u64 %0, t, %3;}"
                : "=l"(x)
                : "r"((unsigned)lo << 7), "r"(__funnelshift_l((unsigned)lo, mh, 7)), "r"(em - e[i]));
            const int sg = hi >> 31;
            S[p] += (long long)(x ^ (unsigned long long)(long long)sg);  // -x - 1 for a negative value
            neg += sg;
        }
        S[p] -= neg;
    }
    if (k.qx | k.qy | k.qz) {  // one branch: three in a row were predicated (64^3 ground state 1.93 ms for 1.87)
        if (k.qx) S[0] = mul_frac(S[0], k.qx);
        if (k.qy) S[1] = mul_frac(S[1], k.qy);
        if (k.qz) S[2] = mul_frac(S[2], k.qz);
    }
    const double f = __hiloint2double(__double2hiint(k.ref) + ((em - 1082) << 20), __double2loint(k.ref));
    return i64_to_double(S[0] + S[1] + S[2]) * f;
}

// What a pass wants of a cell's neighbourhood: its Laplacian (LapFull), or, for
// the right-hand side of the real-time steps in double precision, half of it with
// the sign of the kinetic term (LapRhs): FP64 instructions bound the complex128
// steps, and the factor -1/2 costs none in the coefficients.  (The centre's
// share in the potential would save one more of about fourteen a cell and stage,
// 3 % of a step, but rounds the potential at the size of 1/h^2: 19-point errors
// 2 % larger.)  In single precision, bound by bytes, it is the Laplacian as it is.
struct LapFull {
    static constexpr bool FIXED = true;  // double precision: sums in fixed point where the spacings allow
    template <typename R>
    __device__ __forceinline__ static R coef(R a)
    {
        return a;
    }
    template <typename CT, typename R>
    __device__ __forceinline__ static CT of(const CT &xp, const CT &xm, const CT &yp, const CT &ym, const CT &zp,
                                            const CT &zm, const CT &c, R ax, R ay, R az, R c6)
    {
        return lapv(xp, xm, yp, ym, zp, zm, c, ax, ay, az, c6);
    }
    __device__ __forceinline__ static double with(double c, double s, double c6) { return __fma_rn(-c6, c, s); }
};
struct LapRhs {
    static constexpr bool FIXED = true;
    __device__ __forceinline__ static float coef(float a) { return a; }
    __device__ __forceinline__ static double coef(double a) { return -0.5 * a; }
    __device__ __forceinline__ static float2 of(const float2 &xp, const float2 &xm, const float2 &yp, const float2 &ym,
                                                const float2 &zp, const float2 &zm, const float2 &c, float ax,
                                                float ay, float az, float c6)
    {
        return lapv(xp, xm, yp, ym, zp, zm, c, ax, ay, az, c6);
    }
    // ax, ay, az already through coef()
    __device__ __forceinline__ static double2 of(const double2 &xp, const double2 &xm, const double2 &yp,
                                                 const double2 &ym, const double2 &zp, const double2 &zm,
                                                 const double2 &, double ax, double ay, double az, double)
    {
        double2 n;
        n.x = __fma_rn(az, zp.x + zm.x, __fma_rn(ay, yp.x + ym.x, ax * (xp.x + xm.x)));
        n.y = __fma_rn(az, zp.y + zm.y, __fma_rn(ay, yp.y + ym.y, ax * (xp.y + xm.y)));
        return n;
    }
    __device__ __forceinline__ static double of(double xp, double xm, double yp, double ym, double zp, double zm,
                                                double, double ax, double ay, double az, double)
    {
        return __fma_rn(az, zp + zm, __fma_rn(ay, yp + ym, ax * (xp + xm)));
    }
    __device__ __forceinline__ static double with(double c, double s, double c6) { return __fma_rn(0.5 * c6, c, s); }
};
// The Euler kinetic substep c + q lap c of the imaginary-time passes.  In double
// precision, where FP64 instructions bound them, the spacings carry q
// (euler_coef) and lap_of gives the substep's result, c + (sums - c6 c).  (One factor
// 1 - c6 for the centre's two terms would save an instruction; its rounding
// made the errors 11 % larger.)  In single precision it gives the Laplacian,
// and euler() adds it.
struct LapEuler : LapFull {
    __device__ __forceinline__ static double with(double c, double s, double c6) { return c + __fma_rn(-c6, c, s); }
};
// LAP with the sums in FP64, for grids whose spacings fixed point does not serve
template <typename LAP>
struct InFp64 : LAP {
    static constexpr bool FIXED = false;
};
template <typename LAP, bool FX>
using LapIn = typename std::conditional<FX, LAP, InFp64<LAP>>::type;
// LAP's result from the sum of a cell's neighbours (double precision)
template <typename LAP>
__device__ __forceinline__ double with_centre(double c, double s, double c6)
{
    return LAP::with(c, s, c6);
}
template <typename LAP>
__device__ __forceinline__ double2 with_centre(const double2 &c, const double2 &s, double c6)
{
    return make_double2(LAP::with(c.x, s.x, c6), LAP::with(c.y, s.y, c6));
}
// sum6 as a call, for the kernels that hold several stages' code: inline, its eight
// copies a stage no longer fit the instruction cache and the registers
// (120-cell shell, WAVE schedule, eight RK4 steps: 6.8 ms inline, 3.9 so, 3.85
// in FP64).
static __device__ __noinline__ double sum6_call(double xp, double xm, double yp, double ym, double zp, double zm,
                                                const LapCo<double> *k)
{
    return sum6(xp, xm, yp, ym, zp, zm, *k);
}

// What LAP makes of a cell c and its six neighbours; CALL: by sum6_call
template <typename LAP, bool CALL = false, typename CT, typename R>
__device__ __forceinline__ CT lap_of(const CT &xp, const CT &xm, const CT &yp, const CT &ym, const CT &zp, const CT &zm,
                                     const CT &c, const LapCo<R> &k)
{
    if constexpr (sizeof(R) == 4) {
        return LAP::of(xp, xm, yp, ym, zp, zm, c, k.ax, k.ay, k.az, k.c6);
    } else if constexpr (!LAP::FIXED) {
        return with_centre<LAP>(c, LapRhs::of(xp, xm, yp, ym, zp, zm, c, k.ax, k.ay, k.az, k.c6), k.c6);
    } else {
        auto sum = [&](double a, double b, double e, double f, double g, double h) {
            return CALL ? sum6_call(a, b, e, f, g, h, &k) : sum6(a, b, e, f, g, h, k);
        };
        if constexpr (is_cplx<CT>())
            return with_centre<LAP>(c, make_double2(sum(xp.x, xm.x, yp.x, ym.x, zp.x, zm.x), sum(xp.y, xm.y, yp.y, ym.y, zp.y, zm.y)), k.c6);
        else
            return with_centre<LAP>(c, sum(xp, xm, yp, ym, zp, zm), k.c6);
    }
}
// not 0 unless v is 0 (or -0: bit 63)
__device__ __forceinline__ long long bits_of(double v) { return __double_as_longlong(v); }
__device__ __forceinline__ long long bits_of(const double2 &v) { return __double_as_longlong(v.x) | __double_as_longlong(v.y); }
// The same of a segment's four cells c: xm and xp its end cells' neighbours.
// ASK: whether fixed point serves the spacings is asked here, once, and not by
// every sum.  Fused pairs, complex128, 64 x 64 x 21 trap with spacings 1 : 1 : 3,
// four RK4 steps: 287 -> 238 us (the wavefront kernels, which spill registers,
// lost 3 % on equal spacings and go on asking at every sum).
template <typename LAP, bool CALL = false, bool ASK = false, typename CT, typename R>
__device__ __forceinline__ void lap4(const CT &xm, const CT &xp, const CT (&ym)[4], const CT (&yp)[4], const CT (&zm)[4],
                                     const CT (&zp)[4], const CT (&c)[4], const LapCo<R> &k, CT (&L)[4])
{
    auto each = [&](auto lap) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            L[i] = lap_of<decltype(lap), CALL>(i == 3 ? xp : c[i + 1], i == 0 ? xm : c[i - 1], yp[i], ym[i], zp[i], zm[i], c[i], k);
    };
    if constexpr (ASK && sizeof(R) == 8) {
        if (!k.fixed()) return each(InFp64<LAP>{});
    }
    if constexpr (sizeof(R) == 8 && !LAP::FIXED) {
        // no FP64 instructions where the state is zero (a ramp's shell before the
        // core has reached it): 100-cell ramp, spacings 1 : 1 : 3, 918 -> 589 us
        long long any = bits_of(xm) | bits_of(xp);
#pragma unroll
        for (int i = 0; i < 4; ++i) any |= bits_of(c[i]) | bits_of(ym[i]) | bits_of(yp[i]) | bits_of(zm[i]) | bits_of(zp[i]);
        if ((any << 1) == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) L[i] = czero<CT>();
            return;
        }
    }
    each(LAP{});
}
__device__ __forceinline__ float euler_coef(float ih2, float) { return ih2; }
__device__ __forceinline__ double euler_coef(double ih2, double q) { return ih2 * q; }
// the substep of value c from what LapEuler gave for it
template <typename CT, typename R>
__device__ __forceinline__ CT euler(const CT &c, R q, const CT &L)
{
    if constexpr (sizeof(R) == 8) return L;
    else return axpy(c, q, L);
}

// 4 consecutive complex values (one segment, 32-byte aligned) with 256-bit
// accesses, so that each lane moves whole 32-byte sectors; CG: read through
// L2 only (data written by other blocks of the same launch)
template <bool CG>
__device__ __forceinline__ void ld4(const float2 *p, float2 (&v)[4])
{
    float a[8];
    if (CG)
        asm volatile("ld.global.cg.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=f"(a[0]), "=f"(a[1]), "=f"(a[2]), "=f"(a[3]), "=f"(a[4]), "=f"(a[5]), "=f"(a[6]), "=f"(a[7])
                     : "l"(p));
    else
        asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=f"(a[0]), "=f"(a[1]), "=f"(a[2]), "=f"(a[3]), "=f"(a[4]), "=f"(a[5]), "=f"(a[6]), "=f"(a[7])
                     : "l"(p));
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = make_float2(a[2 * i], a[2 * i + 1]);
}
template <bool CG>
__device__ __forceinline__ void ld4(const double2 *p, double2 (&v)[4])
{
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        double a0, a1, a2, a3;
        if (CG)
            asm volatile("ld.global.cg.v4.f64 {%0,%1,%2,%3}, [%4];"
                         : "=d"(a0), "=d"(a1), "=d"(a2), "=d"(a3) : "l"(p + 2 * h));
        else
            asm volatile("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];" : "=d"(a0), "=d"(a1), "=d"(a2), "=d"(a3) : "l"(p + 2 * h));
        v[2 * h] = make_double2(a0, a1);
        v[2 * h + 1] = make_double2(a2, a3);
    }
}
__device__ __forceinline__ void st4(float2 *p, const float2 (&v)[4])
{
    asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(v[0].x), "f"(v[0].y), "f"(v[1].x),
                 "f"(v[1].y), "f"(v[2].x), "f"(v[2].y), "f"(v[3].x), "f"(v[3].y)
                 : "memory");
}
__device__ __forceinline__ void st4(double2 *p, const double2 (&v)[4])
{
#pragma unroll
    for (int h = 0; h < 2; ++h)
        asm volatile("st.global.v4.f64 [%0], {%1,%2,%3,%4};" ::"l"(p + 2 * h), "d"(v[2 * h].x), "d"(v[2 * h].y),
                     "d"(v[2 * h + 1].x), "d"(v[2 * h + 1].y)
                     : "memory");
}
// 4 consecutive reals of a real-valued state (one segment, 16- or 32-byte
// aligned); CG as for ld4 above
template <bool CG>
__device__ __forceinline__ void ld4(const float *p, float (&v)[4])
{
    if (CG)
        asm volatile("ld.global.cg.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "l"(p));
    else
        asm volatile("ld.global.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "l"(p));
}
template <bool CG>
__device__ __forceinline__ void ld4(const double *p, double (&v)[4])
{
    if (CG)
        asm volatile("ld.global.cg.v4.f64 {%0,%1,%2,%3}, [%4];" : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3]) : "l"(p));
    else
        asm volatile("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];" : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3]) : "l"(p));
}
__device__ __forceinline__ void st4(float *p, const float (&v)[4])
{
    asm volatile("st.global.v4.f32 [%0], {%1,%2,%3,%4};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
}
__device__ __forceinline__ void st4(double *p, const double (&v)[4])
{
    asm volatile("st.global.v4.f64 [%0], {%1,%2,%3,%4};" ::"l"(p), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3]) : "memory");
}

// 4 consecutive reals (16- or 32-byte aligned), read-only data
__device__ __forceinline__ void ldr4(const float *p, float (&v)[4])
{
    const float4 a = __ldg(reinterpret_cast<const float4 *>(p));
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
}
__device__ __forceinline__ void ldr4(const double *p, double (&v)[4])
{
    asm volatile("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];" : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3]) : "l"(p));
}

struct Identity {
    template <typename CT>
    __device__ __forceinline__ CT operator()(CT v, uint32_t) const { return v; }
};

template <bool CG, typename CT>
__device__ __forceinline__ CT ld1(const CT *p)
{
    return CG ? __ldcg(p) : *p;
}

// Per-warp workspace.  The brick's segments, with the y and z face halos as
// whole rows (rows y = -1..BY, planes z = -1..BZ), are stored as UPS planes of
// 16-byte units: unit u of every segment slot is contiguous, so lanes that
// take consecutive segments touch consecutive 16-byte units (no shared-memory
// bank conflicts).  The x face halos are separate columns.  Then the records
// of the brick and its six face neighbours and the brick's stored segments in
// order, each as its tile slot and x-halo row (slot | h << 8).  The records of the warp's next brick are fetched into nrec while
// the current brick is processed.
template <typename CT, int BX, int BY, int BZ>
struct WarpSpace {
    static constexpr int SX = BX / 4, TY = BY + 2, TZ = BZ + 2;
    static constexpr int NR = 7;       // records: own and 6 face neighbours
    static constexpr int XH = BY * BZ;  // x-halo rows
    static constexpr int NSLOT = SX * TY * TZ;                   // segment slots incl. y/z halos
    static constexpr int UPS = (int)(4 * sizeof(CT) / 16);       // 16-byte units per segment
    // plane stride (in units) = 4 (UPS 2) or 2 (UPS 4) mod 8: the UPS units of
    // one segment fall in distinct 16-byte bank groups, so UPS lanes can fill
    // one segment's units in one conflict-free access
    static constexpr int PSTR = NSLOT + (((UPS == 2 ? 4 : 2) - NSLOT % 8) + 8) % 8;
    static constexpr int CPU_ = 4 / UPS;                         // cells per unit
    static constexpr int NSEG = Seg<BX, BY, BZ>::NSEG;
    static constexpr int ROW = SX, PLANE = SX * TY;              // slot strides in y and z
    __device__ __forceinline__ static int slot(int hx, int y, int z) { return hx + SX * ((y + 1) + TY * (z + 1)); }
    __device__ __forceinline__ static int h(int y, int z) { return y + BY * z; }
    uint4 units[UPS][PSTR];
    // x halos: per row the 16-byte unit of the neighbour segment that holds the halo
    // cell (cell 3 of the -x brick's last segment of the row, cell 0 of the
    // +x brick's first), filled by cp.async like the tile.
    static constexpr int XW = 16;
    alignas(16) unsigned char xlo_[XH * XW];  // x = -1
    alignas(16) unsigned char xhi_[XH * XW];  // x = BX
    __device__ __forceinline__ CT xm_cell(int h) const  // the cell at x = -1 of row h
    {
        return reinterpret_cast<const CT *>(xlo_ + h * XW)[CPU_ - 1];
    }
    __device__ __forceinline__ CT xp_cell(int h) const  // the cell at x = BX of row h
    {
        return reinterpret_cast<const CT *>(xhi_ + h * XW)[0];
    }
    __device__ __forceinline__ CT *xm_slot(int h) { return reinterpret_cast<CT *>(xlo_ + h * XW) + (CPU_ - 1); }
    __device__ __forceinline__ CT *xp_slot(int h) { return reinterpret_cast<CT *>(xhi_ + h * XW); }
    alignas(16) BrickRec rec[NR];
#if GPE_REC_AHEAD
    BrickRec nrec[NR];  // records of the warp's next brick, fetched ahead
    long long nrec_b;  // brick whose records nrec holds (-1: none)
    uint16_t list[NSEG];
    uint8_t pad[(16 - ((2 * NSEG + 8) % 16)) % 16];
#else
    uint16_t list[NSEG];
    uint8_t pad[(16 - ((2 * NSEG) % 16)) % 16];
#endif

    __device__ __forceinline__ void get(int s, CT (&v)[4]) const
    {
#pragma unroll
        for (int u = 0; u < UPS; ++u) {
            const uint4 w = units[u][s];
            const CT *c = reinterpret_cast<const CT *>(&w);
#pragma unroll
            for (int i = 0; i < CPU_; ++i) v[u * CPU_ + i] = c[i];
        }
    }
    __device__ __forceinline__ void put(int s, const CT (&v)[4])
    {
#pragma unroll
        for (int u = 0; u < UPS; ++u) {
            uint4 w;
            CT *c = reinterpret_cast<CT *>(&w);
#pragma unroll
            for (int i = 0; i < CPU_; ++i) c[i] = v[u * CPU_ + i];
            units[u][s] = w;
        }
    }
    __device__ __forceinline__ CT first(int s) const  // cell 0 of slot s
    {
        return reinterpret_cast<const CT *>(&units[0][s])[0];
    }
    __device__ __forceinline__ CT last(int s) const  // cell 3 of slot s
    {
        return reinterpret_cast<const CT *>(&units[UPS - 1][s])[CPU_ - 1];
    }
};

template <typename R, int BX, int BY, int BZ, typename CT = typename Cx<R>::T>
constexpr size_t smem_bytes()
{
    return (size_t)KernelCfg<R>::NW * sizeof(WarpSpace<CT, BX, BY, BZ>);
}

// the calling warp's workspace (call once per kernel: it resets the
// next-record tag)
template <typename R, int BX, int BY, int BZ>
constexpr int min_blocks(int in_double)
{
    const int cap = sizeof(R) == 4 ? GPE_MINB_F : in_double;
    const int fit = (int)((228u * 1024u) / (smem_bytes<R, BX, BY, BZ>() + 1024u));
    return fit < 1 ? 1 : (fit < cap ? fit : cap);
}

template <typename R, int BX, int BY, int BZ, typename CT = typename Cx<R>::T>
__device__ __forceinline__ WarpSpace<CT, BX, BY, BZ> &warp_space()
{
    extern __shared__ __align__(16) unsigned char gpe_smem[];
    auto &ws = reinterpret_cast<WarpSpace<CT, BX, BY, BZ> *>(gpe_smem)[threadIdx.x >> 5];
#if GPE_REC_AHEAD
    if ((threadIdx.x & 31) == 0) ws.nrec_b = -1;
    __syncwarp();
#endif
    return ws;
}

// 16-byte asynchronous global -> shared copies (cp.async, L2 only): the tile
// fill issues every copy of a brick before waiting on any of them, so a warp
// keeps its whole tile (and its body's prefetched operands) in flight without
// staging them in registers.  valid == false writes 16 zero bytes.
__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool valid)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Records of brick b (slot 0) and of its six face neighbours (slots 1..6, order
// -x +x -y +y -z +z); an absent neighbour has an empty record.  One row (224
// bytes) moved
// into ws.rec: from ws.nrec when it was fetched ahead, else from global
// memory.  Then the row of brick `next` (if >= 0) is fetched ahead into
// ws.nrec by cp.async; it completes with the tile's copies.
template <typename WS>
__device__ __forceinline__ void fetch_recs(WS &ws, const GridView &G, int64_t b, int64_t next)
{
    constexpr int NU = 2 * WS::NR;  // 16-byte words of one row of records
    const uint4 *rows = reinterpret_cast<const uint4 *>(G.rec7);
    const int lane = threadIdx.x & 31;
    cp_async_wait_all();
    __syncwarp();
#if GPE_REC_AHEAD
    const bool ahead = ws.nrec_b == (long long)b;
    for (int u = lane; u < NU; u += 32)
        reinterpret_cast<uint4 *>(ws.rec)[u] = ahead ? reinterpret_cast<const uint4 *>(ws.nrec)[u] : __ldg(rows + NU * b + u);
    __syncwarp();
    if (next >= 0)
        for (int u = lane; u < NU; u += 32) cp_async16(reinterpret_cast<uint4 *>(ws.nrec) + u, rows + NU * next + u, true);
    if (lane == 0) ws.nrec_b = next;
    __syncwarp();
#else
    (void)next;
    for (int u = lane; u < NU; u += 32) reinterpret_cast<uint4 *>(ws.rec)[u] = __ldg(rows + NU * b + u);
    __syncwarp();
#endif
}

// does the load transform XF provide a whole-segment form xf.seg(v, idx)?
template <typename XF, typename CT, typename = void>
struct HasSeg : std::false_type {};
template <typename XF, typename CT>
struct HasSeg<XF, CT, std::void_t<decltype(std::declval<const XF &>().seg(std::declval<CT (&)[4]>(), 0u))>>
    : std::true_type {};

// Apply body(idx, pre, c, L) to every stored segment of brick b, one warp
// (next: the brick the warp takes after b, or -1):
// idx is the packed index of the segment's first cell, pre what load(idx)
// returned for it, c[4] its values and L[4] their 7-point Laplacians
// (Eq. (B1)), all taken from src after xf(value, packed index).  The warp
// stages the brick's stored segments (contiguous along the packed run) and
// the face halos from the neighbour bricks in its tile; absent cells read as
// zero.  Lanes then take the stored segments in order, so the packed indices
// of a warp's segments are consecutive and the bodies' own-cell loads and
// stores coalesce.  The first 32 segments' operands are loaded while the tile
// is in flight, the next 32's while a group is computed.  With xf the identity the tile is filled by cp.async;
// otherwise through registers, where xf is applied.
template <int BX, int BY, int BZ, bool CG, typename LAP = LapFull, typename CT, typename R, typename XF, typename LOAD,
          typename BODY>
__device__ __forceinline__ void brick_apply(WarpSpace<CT, BX, BY, BZ> &ws, const GridView &G, int64_t b,
                                            int64_t next, const CT *src, XF xf, R ihx2, R ihy2, R ihz2, LOAD load,
                                            BODY body)
{
    using S = Seg<BX, BY, BZ>;
    using W = WarpSpace<CT, BX, BY, BZ>;
    constexpr bool ASYNC = std::is_same<XF, Identity>::value;
    const int lane = threadIdx.x & 31;
    fetch_recs(ws, G, b, next);
    const BrickRec &R0 = ws.rec[0];
    const int nst = __popc(R0.m[0]) + __popc(R0.m[1]) + __popc(R0.m[2]) + __popc(R0.m[3]);
    // unit u of one segment (4 cells; all units when u < 0) into tile slot sl
    auto seg_to = [&](const BrickRec &r, int q, int sl, int u) {
        uint32_t j = 0;
        const bool ok = seg_index(r, q, j);
        if constexpr (ASYNC) {
            const char *g = reinterpret_cast<const char *>(src + (ok ? j : 0u));
            cp_async16(&ws.units[u][sl], g + 16 * u, ok);
        } else {
            CT v[4];
            if (ok) {
                ld4<CG>(src + j, v);
                if constexpr (HasSeg<XF, CT>::value) {
                    xf.seg(v, j);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[i] = xf(v[i], j + i);
                }
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = czero<CT>();
            }
            ws.put(sl, v);
        }
    };
    // ASYNC: UPS lanes per segment; else one lane per segment (u ignored)
    constexpr int LPS = ASYNC ? W::UPS : 1;
    // the stored segments in order (tile slot, x-halo row); with ASYNC the
    // unstored interior slots are zeroed here
    int nl = 0;
#pragma unroll
    for (int it = 0; it < S::NIT; ++it) {
        const int q = it * 32 + lane;
        const int y = (q / S::SX) % BY, z = q / S::PLANE;
        const int sl = W::slot(q % S::SX, y, z);
        const bool stored = (R0.m[q >> 5] >> (q & 31)) & 1u;
        const unsigned bal = __ballot_sync(0xffffffffu, stored);
        if (stored) {
            ws.list[nl + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(sl | (W::h(y, z) << 8));
        } else if constexpr (ASYNC) {
#pragma unroll
            for (int u = 0; u < W::UPS; ++u) ws.units[u][sl] = make_uint4(0, 0, 0, 0);
        }
        nl += __popc(bal);
    }
    // interior
    if constexpr (ASYNC) {
        // stored segments along the packed run: UPS lanes per segment, each
        // one contiguous 16-byte unit
        __syncwarp();
        const char *run = reinterpret_cast<const char *>(src + R0.off);
        for (int t = lane; t < nl * W::UPS; t += 32)
            cp_async16(&ws.units[t % W::UPS][ws.list[t / W::UPS] & 0xff], run + 16 * t, true);
    } else {
#pragma unroll
        for (int q = lane; q < S::NSEG; q += 32) seg_to(R0, q, W::slot(q % S::SX, (q / S::SX) % BY, q / S::PLANE), 0);
    }
    // -z / +z faces: whole segments of the neighbours' boundary planes
#pragma unroll
    for (int t = lane; t < 2 * S::PLANE * LPS; t += 32) {
        const int u = t / LPS, face = u / S::PLANE, qc = u % S::PLANE;
        seg_to(ws.rec[5 + face], face == 0 ? qc + S::PLANE * (BZ - 1) : qc,
               W::slot(qc % S::SX, qc / S::SX, face == 0 ? -1 : BZ), t % LPS);
    }
    // -y / +y faces: segments of the neighbours' boundary rows
#pragma unroll
    for (int t = lane; t < 2 * S::SX * BZ * LPS; t += 32) {
        const int u = t / LPS, face = u / (S::SX * BZ), v_ = u % (S::SX * BZ);
        const int hx = v_ % S::SX, z = v_ / S::SX;
        seg_to(ws.rec[3 + face], hx + S::SX * (face == 0 ? BY - 1 : 0) + S::PLANE * z,
               W::slot(hx, face == 0 ? -1 : BY, z), t % LPS);
    }
    // operands of the first 32 stored segments, while the tile is in flight
    typename std::decay<decltype(load(0u))>::type p0{};
    if (lane < nst) p0 = load(R0.off + 4u * (uint32_t)lane);
    // -x / +x faces, identity transform: per row one 16-byte unit (the one
    // holding cell 3 of the -x brick's segment, or cell 0 of the +x brick's)
    // by cp.async; absent segments give a zero unit.  Else single cells
    // through registers, unrolled, so that a lane's loads are all issued
    // before the first of them is waited for.
    if constexpr (ASYNC) {
        for (int u = lane; u < 2 * BY * BZ; u += 32) {
            const int face = u / (BY * BZ), v_ = u % (BY * BZ);
            const int y = v_ % BY, z = v_ / BY;
            uint32_t j = 0;
            const bool ok = seg_index(ws.rec[1 + face], (face == 0 ? S::SX - 1 : 0) + S::SX * y + S::PLANE * z, j);
            const char *g = reinterpret_cast<const char *>(src + (ok ? j : 0u)) + (face == 0 ? 16 * (W::UPS - 1) : 0);
            cp_async16((face == 0 ? ws.xlo_ : ws.xhi_) + 16 * W::h(y, z), g, ok);
        }
    } else {
#pragma unroll
        for (int u = lane; u < 2 * BY * BZ; u += 32) {
            const int face = u / (BY * BZ), v_ = u % (BY * BZ);
            const int y = v_ % BY, z = v_ / BY;
            CT v = czero<CT>();
            uint32_t j;
            if (seg_index(ws.rec[1 + face], (face == 0 ? S::SX - 1 : 0) + S::SX * y + S::PLANE * z, j)) {
                j += face == 0 ? 3 : 0;
                v = xf(ld1<CG>(src + j), j);
            }
            *(face == 0 ? ws.xm_slot(W::h(y, z)) : ws.xp_slot(W::h(y, z))) = v;
        }
    }
    cp_async_wait_all();
    __syncwarp();
    // stored segments: Laplacian from the tile, then the body.  Opposite
    // neighbours are summed first and the centre term enters once:
    // L = (x- + x+) / hx^2 + (y- + y+) / hy^2 + (z- + z+) / hz^2 - c6 c.
    const LapCo<R> co = lap_co<LAP>(ihx2, ihy2, ihz2);
    auto segment = [&](int r, const auto &pre) {
        const int e = ws.list[r];
        const int sl = e & 0xff, hrow = e >> 8, hx = sl % S::SX;
        CT c[4], ym[4], yp[4], zm[4], zp[4], L[4];
        ws.get(sl, c);
        ws.get(sl - W::ROW, ym);
        ws.get(sl + W::ROW, yp);
        ws.get(sl - W::PLANE, zm);
        ws.get(sl + W::PLANE, zp);
        const CT xm = hx == 0 ? ws.xm_cell(hrow) : ws.last(sl - 1);
        const CT xp = hx == S::SX - 1 ? ws.xp_cell(hrow) : ws.first(sl + 1);
        lap4<LAP, true>(xm, xp, ym, yp, zm, zp, c, co, L);
        body(R0.off + 4u * (uint32_t)r, pre, c, L);
    };
    // each iteration loads the operands of the next before computing its own
    auto cur = p0;
    for (int r = lane; r < nst; r += 32) {
        decltype(p0) nxt{};
        if (r + 32 < nst) nxt = load(R0.off + 4u * (uint32_t)(r + 32));
        segment(r, cur);
        cur = nxt;
    }
}

// ------------------------------------------------------------ ramp schedule
struct Ramp {
    const double *clock;  // device time base
    double T;
    int n_knots;
    double knots[GPE_MAX_KNOTS];
};

// s(t): piecewise linear through n_knots values at t_k = k T/(n_knots-1),
// held constant outside [0, T] (linear interpolation between potentials, Sec. V)
__device__ __forceinline__ double ramp_s(const Ramp &r, double t)
{
    if (t <= 0.0) return r.knots[0];
    if (t >= r.T) return r.knots[r.n_knots - 1];
    double u = t / r.T * (double)(r.n_knots - 1);
    int k = (int)floor(u);
    if (k >= r.n_knots - 1) k = r.n_knots - 2;
    double w = u - (double)k;
    return (1.0 - w) * r.knots[k] + w * r.knots[k + 1];
}

template <typename R, typename CT = typename Cx<R>::T>
struct DiagLoad {
    R sc, hg;
    const R *E;
    __device__ __forceinline__ CT apply(CT v, R e) const
    {
        v = scale(v, sc);
        const R f = active_e(e) ? e * ((R)1 - hg * norm2(v)) : (R)0;
        return scale(v, f);
    }
    __device__ __forceinline__ CT operator()(CT v, uint32_t idx) const { return apply(v, __ldg(E + idx)); }
    // a whole segment (idx = its first cell): one vector load of E
    __device__ __forceinline__ void seg(CT (&v)[4], uint32_t idx) const
    {
        R e[4];
        ldr4(E + idx, e);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = apply(v[i], e[i]);
    }
};

// An FP64 sum of many single-precision terms off the FP64 pipe, where every
// add and conversion issues at 1/64 of the FP32 rate: the terms are added as an
// unevaluated pair of floats (hi + lo, each addition's rounding error found
// exactly by Knuth's two-sum and kept in lo), and the pair goes into an FP64
// total every SUM_FLUSH terms.  After n additions the pair is good to about n
// 2^-48 of the sum, against the 2^-25 of every term.  Double-precision terms
// are added as they are.
// A pair holds up to 3e38: one that has grown beyond PAIR_MAX (or is NaN) goes
// into the FP64 total at once (keep), so that neither the next term nor a
// warp's lanes (block_totals) can take it out of range.
constexpr int SUM_FLUSH = 64;
constexpr float PAIR_MAX = 1e30f;
template <typename R>
struct Sum64 {
    double tot = 0.0;
    __device__ __forceinline__ void add(double x) { tot += x; }
    __device__ __forceinline__ void flush() {}
    __device__ __forceinline__ bool large() const { return false; }
};
// a call, so that the compiler branches around it: FP64 instructions that are
// predicated off still take their turn in the pipe
static __device__ __noinline__ double add_pair(double tot, float hi, float lo)
{
    tot += (double)hi;
    if (isfinite(lo)) tot += (double)lo;  // an infinite or NaN term shows in hi
    return tot;
}
template <>
struct Sum64<float> {
    double tot = 0.0;
    float hi = 0.0f, lo = 0.0f;
    __device__ __forceinline__ void add(float x) { add(x, 0.0f); }
    __device__ __forceinline__ void add(float x, float xl)
    {
        const float s = __fadd_rn(hi, x), b = __fadd_rn(s, -hi);
        const float e = __fadd_rn(__fadd_rn(hi, -__fadd_rn(s, -b)), __fadd_rn(x, -b));
        lo = __fadd_rn(lo, __fadd_rn(e, xl));
        hi = s;
    }
    __device__ __forceinline__ void flush()
    {
        tot = add_pair(tot, hi, lo);
        hi = 0.0f;
        lo = 0.0f;
    }
    __device__ __forceinline__ bool large() const { return !(fabsf(hi) <= PAIR_MAX); }
};
// after the n-th term of each of the first K of some sums: flushes them when due
template <int K, typename R, int NV>
__device__ __forceinline__ void keep(Sum64<R> (&s)[NV], int n)
{
    bool due = n % SUM_FLUSH == 0;
#pragma unroll
    for (int k = 0; k < K; ++k) due |= s[k].large();
    if (due) {
#pragma unroll
        for (int k = 0; k < K; ++k) s[k].flush();
    }
}

// deterministic block sum (result valid in thread 0)
__device__ __forceinline__ double block_sum(double x)
{
    __shared__ double sm[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
    __syncthreads();
    if (lane == 0) sm[warp] = x;
    __syncthreads();
    x = 0.0;
    if (warp == 0) {
        x = lane < nw ? sm[lane] : 0.0;
        for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
    }
    return x;
}

// ------------------------------------------------------------ RK4 stages
// Memory-optimised RK4 (App. A, RK4 a* and b*): the stage states are stored
// instead of the k_i, so stage i reads only the state it differentiates (with
// halo) plus own-cell values:
//   stage 0: y2 = y0 + dt/2 f(t, y0)
//   stage 1: y3 = y0 + dt/2 f(t + dt/2, y2),  w = -y0 + y2 + 2 y3
//   stage 2: y4 = y0 + dt   f(t + dt/2, y3)
//   stage 3: y1 = (w + y4)/3 + dt/6 f(t + dt, y4)  (in place of y0)
// with f(t, y) = -i [ -1/2 lap y + (V(t) + g|y|^2) y ]  (Eq. (8)).  The
// partial sum w is formed in stage 1, where y0, y2 and y3 are at hand, in the
// same operation order as the stage-3 combination (-y0 + y2 + 2 y3 + y4)/3:
// stage 3 then reads one state instead of three.  y4 may share y2's buffer
// (y2 has no reader after stage 1).
template <typename R>
struct RkArgs {
    using CT = typename Cx<R>::T;
    CT *y0;
    CT *y2;
    CT *y3;
    CT *y4;
    CT *w;
    const R *V0;
    const R *V1;
    R ihx2, ihy2, ihz2, g, dt;
    Ramp ramp;
    const double *stab;  // tile kernels: this stage's value of the schedule (k_ramp_table)
    double t_off;  // stage-0 time of this step relative to *ramp.clock
    double dtd;    // dt in FP64 for stage times
};

template <typename R, bool BLEND>
__device__ __forceinline__ R stage_s(const RkArgs<R> &a, int st)
{
    if (!BLEND) return (R)0;
    const double c = (st == 0) ? 0.0 : (st == 3 ? 1.0 : 0.5);
    return (R)ramp_s(a.ramp, *a.ramp.clock + a.t_off + c * a.dtd);
}

// One RK4 stage (st = 0..3): operand loads and the per-segment update.  The
// stage is a template argument so that each stage keeps only its own
// prefetched operands in registers.
template <typename R, bool BLEND, bool CG, int st>
struct Rk4Body {
    using CT = typename Cx<R>::T;
    static constexpr int NV = BLEND ? 4 : 1;
    struct P {
        R V0[4], V1[NV];
        CT y[4];  // y0 (stages 1, 2) or w (stage 3)
    };
    const RkArgs<R> &a;
    R s, k;
    CT *yout;
    __device__ __forceinline__ Rk4Body(const RkArgs<R> &a_, R s_)
        : a(a_), s(s_), k(st == 2 ? a_.dt : (st == 3 ? a_.dt / (R)6 : a_.dt / (R)2)),
          yout(st == 0 ? a_.y2 : st == 1 ? a_.y3 : st == 2 ? a_.y4 : a_.y0)
    {
    }
    __device__ __forceinline__ const CT *yin() const { return st == 0 ? a.y0 : st == 1 ? a.y2 : st == 2 ? a.y3 : a.y4; }
    __device__ __forceinline__ P load(uint32_t idx) const
    {
        P p;
        ldr4(a.V0 + idx, p.V0);
        if constexpr (BLEND) ldr4(a.V1 + idx, p.V1);
        if constexpr (st == 1 || st == 2) ld4<CG>(a.y0 + idx, p.y);
        if constexpr (st == 3) ld4<CG>(a.w + idx, p.y);
        return p;
    }
    // the stage's new values o (and, stage 1, the partial sum wv) of the
    // segment with values c, Laplacians L and operands p
    __device__ __forceinline__ void compute(const P &p, const CT (&c)[4], const CT (&L)[4], CT (&o)[4],
                                            CT (&wv)[4]) const
    {
        if constexpr (std::is_same<R, float>::value) {
            // complex64: both parts at once (f32x2), the same operations as the
            // scalar form below
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (!(p.V0[i] < (R)INFINITY)) {
                    o[i] = czero<CT>();
                    wv[i] = czero<CT>();
                    continue;
                }
                R V = p.V0[i];
                if constexpr (BLEND) V = ((R)1 - s) * p.V0[i] + s * p.V1[i];
                const R w = V + a.g * (c[i].x * c[i].x + c[i].y * c[i].y);
                const float2 h = fma2(dup2(w), c[i], mul2(dup2(-0.5f), L[i]));   // (hr, hi)
                const float2 hs = make_float2(h.y, h.x);                           // (hi, hr)
                const float2 kk = make_float2(k, -k);                              // f = (hi, -hr)
                if constexpr (st == 0) {
                    o[i] = fma2(kk, hs, c[i]);
                } else if constexpr (st < 3) {
                    o[i] = fma2(kk, hs, p.y[i]);
                    if constexpr (st == 1) wv[i] = fma2(dup2(2.0f), o[i], sub2(c[i], p.y[i]));
                } else {
                    // x / 3, correctly rounded, without a division: q = RN(x RN(1/3)) is
                    // within one ulp of x/3, the residual x - 3q is exact with a fused
                    // multiply-add, and RN(q + (x - 3q) RN(1/3)) is the correctly rounded
                    // quotient (Markstein's theorem on division with a fused
                    // multiply-add; Muller et al., Handbook of Floating-Point
                    // Arithmetic, the section on Newton-Raphson-based division)
                    const float2 x = add2(p.y[i], c[i]);
                    const float2 t3 = dup2(1.0f / 3.0f);
                    const float2 q = mul2(x, t3);
                    o[i] = fma2(kk, hs, fma2(fma2(dup2(-3.0f), q, x), t3, q));
                }
            }
            return;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            R V = p.V0[i];
            if constexpr (BLEND) V = ((R)1 - s) * p.V0[i] + s * p.V1[i];
            // L is -1/2 lap
            const R w = V + a.g * (c[i].x * c[i].x + c[i].y * c[i].y);
            const R hr = L[i].x + w * c[i].x;
            const R hi = L[i].y + w * c[i].y;
            // f = -i (hr + i hi) = hi - i hr
            if constexpr (st == 0) {
                o[i].x = c[i].x + k * hi;
                o[i].y = c[i].y - k * hr;
            } else if constexpr (st < 3) {
                o[i].x = p.y[i].x + k * hi;
                o[i].y = p.y[i].y - k * hr;
                if constexpr (st == 1) {
                    wv[i].x = -p.y[i].x + c[i].x + (R)2 * o[i].x;
                    wv[i].y = -p.y[i].y + c[i].y + (R)2 * o[i].y;
                }
            } else {
                // x/3 + k f with the third in two parts: T + TL is 1/3 to 2^-108,
                // so the sum is rounded once, and x/3 alone correctly (a third
                // rounded to T alone would shrink every step by 2^-54)
                constexpr double T = 1.0 / 3.0, TL = 1.850371707708594e-17;
                const R xr = p.y[i].x + c[i].x, xi = p.y[i].y + c[i].y;
                o[i].x = __fma_rn(T, xr, __fma_rn(k, hi, TL * xr));
                o[i].y = __fma_rn(T, xi, __fma_rn(-k, hr, TL * xi));
            }
            if (!active_v(p.V0[i])) {  // inactive cell of a stored segment
                o[i] = czero<CT>();
                if constexpr (st == 1) wv[i] = czero<CT>();
            }
        }
    }
    __device__ __forceinline__ void operator()(uint32_t idx, const P &p, const CT (&c)[4], const CT (&L)[4]) const
    {
        CT o[4], wv[4];
        compute(p, c, L, o, wv);
        if constexpr (st == 1) st4(a.w + idx, wv);
        st4(yout + idx, o);
    }
};

// One RK4 stage on brick b, one warp, lane = segment within each group of 32.
template <typename R, int BX, int BY, int BZ, bool BLEND, bool CG, int st>
__device__ __forceinline__ void rk4_brick(const RkArgs<R> &a, const GridView &G, int64_t b, int64_t next,
                                          WarpSpace<typename Cx<R>::T, BX, BY, BZ> &ws, R s)
{
    using B = Rk4Body<R, BLEND, CG, st>;
    const B body(a, s);
    brick_apply<BX, BY, BZ, CG, LapRhs>(ws, G, b, next, body.yin(), Identity(), a.ihx2, a.ihy2, a.ihz2,
                                [&](uint32_t idx) { return body.load(idx); }, body);
}

}  // namespace gpe
