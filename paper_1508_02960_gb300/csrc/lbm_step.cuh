// lbm_step.cuh -- the fused D3Q19 time step (Sec. 2: stream first, then collide, the two
// fused so that macroscopic values are never stored).
//
// Work decomposition.  An instance's fluid cells, in cell order, are dealt out 32 per
// warp (solid cells cost nothing and every lane has a cell, up to the last warp); runs of
// consecutive fluid cells keep the loads of a warp coalesced.  One block per tile of
// kStepWarps such work items, one per warp (one lane per cell).
//
// Per fluid cell x and direction k (all arithmetic on deviations g = f - w rho0):
//   pull      g_k <- g~_k(x - e_k), plus +w_k delta_rho when the pull crosses the x
//             boundary from right to left and -w_k delta_rho the other way (Sec. 2.2.2,
//             Eqs. Periodicfunkown, PeriodicfunkownRight);
//   wall      if x - e_k is solid: SBB g_k <- g~_kbar(x) (Eq. noslip), or CLI
//             g_k <- c (g_kbar^in - g~_k(x)) + g~_kbar(x), c = (1-2q)/(1+2q) (Eq. CLI;
//             g_kbar^in is the streamed value from x_f2 = x + e_k);
//   moments   drho = sum g_k, u = rho0^-1 sum e_k g_k (Eq. Macro);
//   collide   SRT, TRT or MRT relaxation towards Eq. equilibrium;
//   store     A-B: to the other buffer; AA: in place (see below).
// The 19 pulls are issued unconditionally: a solid source slot holds the own-cell part
// of the wall rule, left by the previous step (see WallStage), so
// no pull waits on the boundary table; the wall code runs only for boundary cells.
//
// AA layout (in-place, one buffer).  PULL steps read g~_k(x - e_k) from slot kbar of
// x - e_k and push g~_k(x) into slot k of x + e_k; LOCAL steps read slot k and write
// slot kbar of x itself.  Every slot is then read and written by one thread only.
// Walls.  No fluid cell owns a slot of a solid cell, and slot kbar of the solid cell
// s = x - e_k belongs to the link (x, k) alone: a PULL step of x pulls direction k from
// it and pushes g~_kbar(x) into it (x + e_kbar = s).  Each step leaves the own-cell part S
// of the link's wall rule (wall_own_part, from the post-collision values in registers)
// where the next step's ordinary pull of direction k finds it: a LOCAL step stores S into
// slot kbar of s; a PULL step stores it into the own slot k, which no other cell reads or
// writes in a PULL step, besides its ordinary push of g~_kbar(x) into slot kbar of s.
// So the wall rule needs no load beyond the 19 pulls, as in the A-B layout, and the two
// layouts agree bit for bit.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Loads of population values.  An A-B step reads a buffer that no thread of the step
// writes, through the read-only (non-coherent) path.  The AA steps update their buffer in
// place: a non-coherent load there is not allowed (the compiler may then order it after a
// store of the same thread), so they load plainly.  Both with the ordinary L2 policy: loads
// marked evict-first take A-B 128^3 from 42.4 to 45 us a step and 256^3 from 280 to 330
// (neighbouring items share sectors); the first 20 MB of the tiles marked evict-last, loads
// and stores, gain 2 % there and lose 1-2 % in the AA layout.
template <int KIND, typename T> __device__ __forceinline__ T ld_pop(const T *p)
{
    if constexpr (KIND == KIND_AB) return __ldg(p);
    else return *p;
}

// Instance parameters held in registers for the duration of a chunk.
template <typename R> struct Par {
    uint32_t ks, nx, ny, nz;
    FastDiv dnx, dny;
    const CollPar<R> &c;  // read where it is used
    float isc;
    uint32_t hash_off;
    int wall;
};

template <typename R> __device__ __forceinline__ const CollPar<R> &coll_par(const InstanceDev &I)
{
    if constexpr (sizeof(R) == sizeof(float)) return I.cf;
    else return I.cd;
}

template <typename R> __device__ __forceinline__ Par<R> load_par(const InstanceDev &I)
{
    return Par<R>{I.ks,      (uint32_t)I.nx, (uint32_t)I.ny, (uint32_t)I.nz, I.div_nx,
                  I.div_ny,  coll_par<R>(I), I.inv_scale,    I.cf.hash_off,  I.wall};
}

// Cell coordinates with the periodic x-1/x/x+1 offsets, row offsets y-1/y/y+1 and plane
// offsets z-1/z/z+1 (32-bit element counts).
struct Coord {
    uint32_t x;
    uint32_t X[3], Y[3], Z[3];
    __device__ __forceinline__ uint32_t pull(int k) const { return X[1 - ex(k)] + Y[1 - ey(k)] + Z[1 - ez(k)]; }
    __device__ __forceinline__ uint32_t push(int k) const { return X[1 + ex(k)] + Y[1 + ey(k)] + Z[1 + ez(k)]; }
};
template <typename R> __device__ __forceinline__ Coord coord_of(const Par<R> &p, uint32_t cell)
{
    Coord c;
    const uint32_t nx = p.nx, ny = p.ny, nz = p.nz, nxy = nx * ny;
    const uint32_t yz = fast_div(cell, p.dnx);
    c.x = cell - yz * nx;
    const uint32_t z = fast_div(yz, p.dny);
    const uint32_t y = yz - z * ny;
    c.X[0] = c.x == 0 ? nx - 1 : c.x - 1;
    c.X[1] = c.x;
    c.X[2] = c.x == nx - 1 ? 0 : c.x + 1;
    c.Y[0] = (y == 0 ? ny - 1 : y - 1) * nx;
    c.Y[1] = y * nx;
    c.Y[2] = (y == ny - 1 ? 0 : y + 1) * nx;
    c.Z[0] = (z == 0 ? nz - 1 : z - 1) * nxy;
    c.Z[1] = z * nxy;
    c.Z[2] = (z == nz - 1 ? 0 : z + 1) * nxy;
    return c;
}

// The static tables a step reads (work list, boundary table, wall-rule coefficients) are
// small next to the populations streaming through L2 every step; they are loaded with an
// evict-last L2 policy so that they stay resident from one step to the next.
__device__ __forceinline__ uint64_t l2_keep_policy()
{
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint32_t ld_keep(const uint32_t *a, uint64_t pol)
{
    uint32_t v;
    asm("ld.global.nc.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(a), "l"(pol));
    return v;
}
__device__ __forceinline__ float ld_keep(const float *a, uint64_t pol)
{
    float v;
    asm("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(a), "l"(pol));
    return v;
}
__device__ __forceinline__ double ld_keep(const double *a, uint64_t pol)
{
    double v;
    asm("ld.global.nc.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(a), "l"(pol));
    return v;
}
__device__ __forceinline__ uint32_t ld_keep(const uint16_t *a, uint64_t pol)
{
    unsigned short v;
    asm("ld.global.nc.L2::cache_hint.u16 %0, [%1], %2;" : "=h"(v) : "l"(a), "l"(pol));
    return v;
}
__device__ __forceinline__ uint4 ld_keep(const uint4 *a, uint64_t pol)
{
    uint4 v;
    asm("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
        : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
        : "l"(a), "l"(pol));
    return v;
}
__device__ __forceinline__ uint2 ld_keep(const uint2 *a, uint64_t pol)
{
    uint2 v;
    asm("ld.global.nc.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;" : "=r"(v.x), "=r"(v.y) : "l"(a), "l"(pol));
    return v;
}

// Blocks per multiprocessor the register allocation is sized for: 36 warps (56 registers a
// thread) for the single-instance steps that do not reduce (against 32 at 64 registers: FP32
// 1-6 % faster, 16-bit AA 1-3 % from 128^3 on and 1 % slower below, FP32 MRT 1-2 %; 40 warps
// spill and are 2-6 % slower); 32 for the reducing and interpolated-wall variants and the
// 16-bit MRT, which would spill at 56, and for batches (36: 2-5 % slower).  FP64: 8 warps.
#ifndef LBM_STEP_WARPS_PER_SM
#define LBM_STEP_WARPS_PER_SM 36
#endif
template <int STORE, int COLL, bool RED, bool WX, int WARPS = kStepWarps, int KIND = KIND_AB, bool BATCH = false>
constexpr int step_min_blocks()
{
    if (STORE == ST_F64) return 8 / WARPS;
    constexpr bool wide = RED || WX || BATCH || (COLL == COLL_MRT && kStochastic<STORE>);
    return (wide ? 32 : LBM_STEP_WARPS_PER_SM) / WARPS;
}

// Two values of the compute type side by side.  FP32: a register pair and Blackwell's packed
// FP32 instructions (add, sub, mul, fma .f32x2: both values by one instruction, each rounded
// as by the scalar one), which halve the issue slots of the collision; FP64: two scalars.
template <typename R> struct Pair;
template <> struct Pair<float> {
    unsigned long long v;
};
template <> struct Pair<double> {
    double x, y;
};
__device__ __forceinline__ Pair<float> pair_of(float x, float y)
{
    Pair<float> p;
    asm("mov.b64 %0, {%1, %2};" : "=l"(p.v) : "f"(x), "f"(y));
    return p;
}
__device__ __forceinline__ Pair<double> pair_of(double x, double y) { return {x, y}; }
__device__ __forceinline__ void split(const Pair<float> &p, float &x, float &y)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(p.v));
}
__device__ __forceinline__ void split(const Pair<double> &p, double &x, double &y)
{
    x = p.x;
    y = p.y;
}
__device__ __forceinline__ Pair<float> operator+(const Pair<float> &a, const Pair<float> &b)
{
    Pair<float> d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
__device__ __forceinline__ Pair<float> operator-(const Pair<float> &a, const Pair<float> &b)
{
    Pair<float> d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
__device__ __forceinline__ Pair<float> operator*(const Pair<float> &a, const Pair<float> &b)
{
    Pair<float> d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
__device__ __forceinline__ Pair<float> fma_r(const Pair<float> &a, const Pair<float> &b, const Pair<float> &c)
{
    Pair<float> d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return d;
}
__device__ __forceinline__ Pair<double> operator+(const Pair<double> &a, const Pair<double> &b)
{
    return {a.x + b.x, a.y + b.y};
}
__device__ __forceinline__ Pair<double> operator-(const Pair<double> &a, const Pair<double> &b)
{
    return {a.x - b.x, a.y - b.y};
}
__device__ __forceinline__ Pair<double> operator*(const Pair<double> &a, const Pair<double> &b)
{
    return {a.x * b.x, a.y * b.y};
}
__device__ __forceinline__ Pair<double> fma_r(const Pair<double> &a, const Pair<double> &b, const Pair<double> &c)
{
    return {fma_r(a.x, b.x, c.x), fma_r(a.y, b.y, c.y)};
}
__device__ __forceinline__ Pair<float> pair_of(const float2 &a) { return pair_of(a.x, a.y); }
template <typename R> __device__ __forceinline__ Pair<R> both(R a) { return pair_of(a, a); }
template <typename R> __device__ __forceinline__ R sum_of(const Pair<R> &p)
{
    R x, y;
    split(p, x, y);
    return x + y;
}

// Moments and collision of one cell, in place on the pulled values g[] (deviations, in the
// units of CollPar): Eqs. Macro, SRT, TRT, MRT with the equilibrium of Eq. equilibrium.
// Returns drho = sum g_k and u = rho0^-1 sum e_k g_k.
//
// Three forms.
//  - relax_pairs, TRT: on the sums s and differences d of opposite pairs, the directions 1, 3
//    (axis x, y), 7, 9 (diagonals of the xy plane), 11, 13 (xz) and 15, 17 (yz) two to a
//    Pair, 5 (axis z) alone.  FP64: the bound is the FP64 pipe (a warp instruction per 19
//    cycles a multiprocessor, 64 cycles for a warp alone), so the count is what matters: 116
//    (CollPar<double>) where the pair form of the equations takes about 150; SRT runs it with
//    omega- = omega+.  FP32: Eq. TRT operation by operation, 97 instructions for 147
//    operations; its values are those of the scalar form, bit for bit (the 16-bit formats'
//    stochastic rounding hashes them).
//  - relax_rows, MRT of FP64 and FP32 storage: g~ = g - M^T delta, delta_i = s_i / |M_i|^2
//    (m_i - m_i^eq).  The rows of M are combinations of the same few sums per axis and per
//    plane (checked against mrt_m at compile time below), so the moments and the way back take
//    177 operations instead of the 19 x 19 products; the equilibrium moments follow from Eq.
//    equilibrium: e -11 drho + 19 j.j/rho0, eps 3 drho - 11/2 j.j/rho0, 3p_xx
//    (3 jx^2 - j.j)/rho0, 3pi_xx -1/2 of it, p_ww (jy^2 - jz^2)/rho0, pi_ww -1/2 of it, p_ab
//    ja jb/rho0, q -2/3 j, m 0.
//  - relax_plain, FP32 SRT and the MRT of the 16-bit formats, whose FP32 values (hashed by the
//    stochastic rounding) are those of these expressions.
template <typename R> struct PairSums {
    Pair<R> s1, s7, s11, s15, d1, d7, d11, d15;
    R s5, d5;
    __device__ __forceinline__ explicit PairSums(const R (&g)[Q])
    {
        const Pair<R> a1 = pair_of(g[1], g[3]), b1 = pair_of(g[2], g[4]);
        const Pair<R> a7 = pair_of(g[7], g[9]), b7 = pair_of(g[8], g[10]);
        const Pair<R> a11 = pair_of(g[11], g[13]), b11 = pair_of(g[12], g[14]);
        const Pair<R> a15 = pair_of(g[15], g[17]), b15 = pair_of(g[16], g[18]);
        s1 = a1 + b1, s7 = a7 + b7, s11 = a11 + b11, s15 = a15 + b15;
        d1 = a1 - b1, d7 = a7 - b7, d11 = a11 - b11, d15 = a15 - b15;
        s5 = g[5] + g[6], d5 = g[5] - g[6];
    }
};

__device__ __forceinline__ void relax_pairs(double (&g)[Q], const CollPar<double> &c, double &drho, double &ux,
                                            double &uy, double &uz)
{
    using R = double;
    using V = Pair<double>;
    const auto [s1, s7, s11, s15, d1, d7, d11, d15, s5, d5] = PairSums<double>(g);
    // per plane: the x (or y) and the y or z momentum of its four diagonals
    R jx, jy, jz, u, v;
    split(d7, u, v);
    const R x7 = u + v, y7 = u - v;
    split(d11, u, v);
    const R x11 = u + v, z11 = u - v;
    split(d15, u, v);
    const R y15 = u + v, z15 = u - v;
    drho = sum_of((s1 + s7) + (s11 + s15)) + (s5 + g[0]);
    const V jxy = (d1 + pair_of(x7, y7)) + pair_of(x11, y15);
    split(jxy, jx, jy);
    jz = d5 + (z11 + z15);
    const V q1 = jxy * jxy;
    const R q5 = jz * jz;
    const R B = fma_r(c.kap, sum_of(q1) + q5, drho);
    const R E1 = c.c1a * B, E7 = c.c1d * B;
    const V al = both(c.alpha), be = both(c.beta), c2d = both(c.c2d), c3d = both(c.c3d), E7v = both(E7);
    auto give = [&](int k, const V &s, const V &d, const V &ej, const V &qc, const V &c3) {
        const V h = fma_r(al, s, qc), t = fma_r(be, d, c3 * ej);
        split(h + t, g[k], g[k + 2]);
        split(h - t, g[k + 1], g[k + 3]);
    };
    g[0] = fma_r(c.a0, g[0], c.c10 * B);
    give(1, s1, d1, jxy, fma_r(both(c.c2a), q1, both(E1)), both(c.c3a));
    {
        const R h = fma_r(c.alpha, s5, fma_r(c.c2a, q5, E1)), t = fma_r(c.beta, d5, c.c3a * jz);
        g[5] = h + t;
        g[6] = h - t;
    }
    const V e7 = pair_of(jx + jy, jx - jy), e11 = pair_of(jx + jz, jx - jz), e15 = pair_of(jy + jz, jy - jz);
    give(7, s7, d7, e7, fma_r(c2d, e7 * e7, E7v), c3d);
    give(11, s11, d11, e11, fma_r(c2d, e11 * e11, E7v), c3d);
    give(15, s15, d15, e15, fma_r(c2d, e15 * e15, E7v), c3d);
    ux = jx * c.irho0;
    uy = jy * c.irho0;
    uz = jz * c.irho0;
}

__device__ __forceinline__ void relax_pairs(float (&g)[Q], const CollPar<float> &c, float &drho, float &ux, float &uy,
                                            float &uz)
{
    using R = float;
    using V = Pair<float>;
    const auto [s1, s7, s11, s15, d1, d7, d11, d15, s5, d5] = PairSums<float>(g);
    R sx, sy, s7x, s7y, s11x, s11y, s15x, s15y, dx, dy, d7x, d7y, d11x, d11y, d15x, d15y;
    split(s1, sx, sy);
    split(s7, s7x, s7y);
    split(s11, s11x, s11y);
    split(s15, s15x, s15y);
    split(d1, dx, dy);
    split(d7, d7x, d7y);
    split(d11, d11x, d11y);
    split(d15, d15x, d15y);
    drho = ((((((((g[0] + sx) + sy) + s5) + s7x) + s7y) + s11x) + s11y) + s15x) + s15y;
    ux = ((((dx + d7x) + d7y) + d11x) + d11y) * c.irho0;
    uy = ((((dy + d7x) - d7y) + d15x) + d15y) * c.irho0;
    uz = ((((d5 + d11x) - d11y) + d15x) - d15y) * c.irho0;
    const R uu = fma_r(uz, uz, fma_r(ux, ux, __fmul_rn(uy, uy)));
    const R base = fma_r(-c.r15, uu, drho);  // drho - 3/2 rho0 u.u
    const V wp = pair_of(c.wp), wm = pair_of(c.wm), wmb = pair_of(c.wmb), r45 = pair_of(c.r45), basev = both(base);
    // Y, Z: the symmetric and antisymmetric parts less their equilibria
    auto give = [&](int k, const V &eu, R w, const V &w3) {
        const V a = pair_of(g[k], g[k + 2]), b = pair_of(g[k + 1], g[k + 3]), half = both(R(0.5));
        const V Y = fma_r(half, a + b, both(-w) * fma_r(r45 * eu, eu, basev));
        const V Z = fma_r(half, a - b, w3 * eu);
        split(fma_r(wm, Z, fma_r(wp, Y, a)), g[k], g[k + 2]);
        split(fma_r(wmb, Z, fma_r(wp, Y, b)), g[k + 1], g[k + 3]);
    };
    constexpr R wa = R(weight(1)), wd = R(weight(7));
    g[0] = fma_r(-c.omega, fma_r(-R(weight(0)), base, g[0]), g[0]);
    give(1, pair_of(ux, uy), wa, pair_of(c.w3a));
    {
        const R Y = fma_r(R(0.5), g[5] + g[6], -__fmul_rn(wa, fma_r(__fmul_rn(c.r45.x, uz), uz, base)));
        const R Z = fma_r(R(0.5), g[5] - g[6], __fmul_rn(c.w3a.x, uz));
        g[5] = fma_r(c.wm.x, Z, fma_r(c.wp.x, Y, g[5]));
        g[6] = fma_r(c.wmb.x, Z, fma_r(c.wp.x, Y, g[6]));
    }
    give(7, pair_of(ux + uy, ux - uy), wd, pair_of(c.w3d));
    give(11, pair_of(ux + uz, ux - uz), wd, pair_of(c.w3d));
    give(15, pair_of(uy + uz, uy - uz), wd, pair_of(c.w3d));
}

template <typename R>
__device__ __forceinline__ void relax_rows(R (&g)[Q], const CollPar<R> &c, R &drho, R &ux, R &uy, R &uz)
{
    const auto [s1, s7, s11, s15, d1, d7, d11, d15, s5, d5] = PairSums<R>(g);
    R u, v;
    split(d7, u, v);
    const R x7 = u + v, y7 = u - v;
    split(d11, u, v);
    const R x11 = u + v, z11 = u - v;
    split(d15, u, v);
    const R y15 = u + v, z15 = u - v;
    R sx, sy, pxy, pxz, pyz, mxy, mxz, myz, dx, dy;
    split(s1, sx, sy);
    split(d1, dx, dy);
    split(s7, u, v);
    pxy = u + v, mxy = u - v;
    split(s11, u, v);
    pxz = u + v, mxz = u - v;
    split(s15, u, v);
    pyz = u + v, myz = u - v;
    const R yz = sy + s5, A = sx + yz, px = pxy + pxz, D = px + pyz;
    drho = g[0] + (A + D);
    const R tx = x7 + x11, ty = y7 + y15, tz = z11 + z15;
    const R jx = dx + tx, jy = dy + ty, jz = d5 + tz;
    ux = c.irho0 * jx;
    uy = c.irho0 * jy;
    uz = c.irho0 * jz;
    const R qxx = ux * jx, qyy = uy * jy, qzz = uz * jz;
    const R qq = qxx + (qyy + qzz), n9 = fma_r(R(3), qxx, -qq), n11 = qyy - qzz;
    const R x9 = fma_r(R(2), sx, -yz), w9 = fma_r(R(-2), pyz, px), x11m = sy - s5, w11 = pxy - pxz;
    const R D1 = c.rate[1] * fma_r(R(-11), A, fma_r(R(8), D, fma_r(R(-30), g[0], fma_r(R(11), drho, R(-19) * qq))));
    const R D2 = c.rate[2] * fma_r(R(-4), A, fma_r(R(12), g[0], fma_r(R(-3), drho, fma_r(R(5.5), qq, D))));
    const R D9 = c.rate[9] * (x9 + (w9 - n9)), D11 = c.rate[11] * (x11m + (w11 - n11));
    const R D10 = c.rate[10] * fma_r(R(-2), x9, fma_r(R(0.5), n9, w9));
    const R D12 = c.rate[12] * fma_r(R(-2), x11m, fma_r(R(0.5), n11, w11));
    const R D13 = c.rate[13] * fma_r(-ux, jy, mxy);
    const R D14 = c.rate[14] * fma_r(-uy, jz, myz);
    const R D15 = c.rate[15] * fma_r(-ux, jz, mxz);
    const R D4 = c.rate[4] * fma_r(R(-4), dx, fma_r(R(2.0 / 3.0), jx, tx));
    const R D6 = c.rate[6] * fma_r(R(-4), dy, fma_r(R(2.0 / 3.0), jy, ty));
    const R D8 = c.rate[8] * fma_r(R(-4), d5, fma_r(R(2.0 / 3.0), jz, tz));
    const R D16 = c.rate[16] * (x7 - x11), D17 = c.rate[17] * (y15 - y7), D18 = c.rate[18] * (z11 - z15);
    // back: the even part is taken off both values of a pair, the odd part off one and
    // added to the other
    g[0] -= fma_r(R(12), D2, R(-30) * D1);
    auto give = [&](int k, R ev, R od) {
        g[k] = (g[k] - ev) - od;
        g[k + 1] = (g[k + 1] - ev) + od;
    };
    const R a = fma_r(R(-11), D1, R(-4) * D2), b = fma_r(R(8), D1, D2);
    const R u9 = fma_r(R(-2), D10, D9), u11 = fma_r(R(-2), D12, D11), v9 = D9 + D10, v11 = D11 + D12;
    give(1, fma_r(R(2), u9, a), R(-4) * D4);
    const R ay = a - u9;
    give(3, ay + u11, R(-4) * D6);
    give(5, ay - u11, R(-4) * D8);
    const R xa = D4 + D16, ya = D6 - D17, xb = D4 - D16, za = D8 + D18, yb = D6 + D17, zb = D8 - D18;
    const R bv = b + v9, b7 = bv + v11, b11m = bv - v11, b15m = fma_r(R(-2), v9, b);
    give(7, b7 + D13, xa + ya);
    give(9, b7 - D13, xa - ya);
    give(11, b11m + D15, xb + za);
    give(13, b11m - D15, xb - za);
    give(15, b15m + D14, yb + zb);
    give(17, b15m - D14, yb - zb);
}

template <int COLL>
__device__ __forceinline__ void relax_plain(float (&g)[Q], const CollPar<float> &p, float &drho, float &ux, float &uy,
                                            float &uz)
{
    using R = float;
    const R irho0 = p.irho0, rho0 = p.rho0;
    // sums and differences of opposite pairs: drho = g_0 + sum s_p, j = sum e_p d_p
    R d_sum = g[0], jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
    for (int k = 1; k < Q; k += 2) {
        const R sp = g[k] + g[k + 1], dp = g[k] - g[k + 1];
        d_sum += sp;
        if (ex(k)) jx += ex(k) > 0 ? dp : -dp;
        if (ey(k)) jy += ey(k) > 0 ? dp : -dp;
        if (ez(k)) jz += ez(k) > 0 ? dp : -dp;
    }
    drho = d_sum;
    ux = jx * irho0;
    uy = jy * irho0;
    uz = jz * irho0;
    const R uu = fma_r(uz, uz, fma_r(ux, ux, __fmul_rn(uy, uy)));
    if constexpr (COLL == COLL_SRT) {
        const R om = p.omega;
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const R eu = R(ex(k)) * ux + R(ey(k)) * uy + R(ez(k)) * uz;
            const R geq = R(weight(k)) * (drho + rho0 * (R(3) * eu + R(4.5) * eu * eu - R(1.5) * uu));
            g[k] = g[k] - om * (g[k] - geq);
        }
    } else {  // MRT
        // Every row of M is even or odd in e (mrt_even), so a moment takes the sums (even
        // rows) or the differences (odd rows) of the opposite pairs of g - g^eq, and the
        // relaxation goes back to a pair as its even part plus or minus its odd part: the
        // same matrix in half the operations of the full 19 x 19 products.
        R sp[Q / 2 + 1], dp[Q / 2 + 1];
        sp[0] = g[0] - R(weight(0)) * (drho - R(1.5) * rho0 * uu);
        dp[0] = R(0);
#pragma unroll
        for (int k = 1; k < Q; k += 2) {
            const R w = R(weight(k));
            const R eu = R(ex(k)) * ux + R(ey(k)) * uy + R(ez(k)) * uz;
            const R eqs = w * (drho + rho0 * (R(4.5) * eu * eu - R(1.5) * uu));  // even part of f^eq
            const R eqd = w * rho0 * R(3) * eu;                                  // odd part of f^eq
            const R nk = g[k] - (eqs + eqd), nkb = g[k + 1] - (eqs - eqd);
            sp[(k + 1) / 2] = nk + nkb;
            dp[(k + 1) / 2] = nk - nkb;
        }
        R dm[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            dm[i] = R(0);
            if (i == 0 || i == 3 || i == 5 || i == 7) continue;  // conserved: m^neq = 0
            R m = R(0);
#pragma unroll
            for (int h = 0; h <= Q / 2; ++h) {
                const int c = mrt_m(i, h == 0 ? 0 : 2 * h - 1);
                const R v = mrt_even(i) ? sp[h] : dp[h];
                if (c == 1) m += v;
                else if (c == -1) m -= v;
                else if (c != 0) m += R(c) * v;
            }
            dm[i] = p.rate[i] * m;  // rates[] already divided by |M_i|^2
        }
#pragma unroll
        for (int h = 0; h <= Q / 2; ++h) {
            const int k = h == 0 ? 0 : 2 * h - 1;
            R ev = R(0), od = R(0);
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                if (i == 0 || i == 3 || i == 5 || i == 7) continue;
                const int c = mrt_m(i, k);
                if (c == 0) continue;
                const R t = c == 1 ? dm[i] : (c == -1 ? -dm[i] : R(c) * dm[i]);
                if (mrt_even(i)) ev += t;
                else od += t;
            }
            if (h == 0) {
                g[0] -= ev;
            } else {
                g[k] -= ev + od;
                g[k + 1] -= ev - od;
            }
        }
    }
}

template <int COLL, int STORE, typename R>
__device__ __forceinline__ void relax(R (&g)[Q], const CollPar<R> &c, R &drho, R &ux, R &uy, R &uz)
{
    static_assert(STORE != ST_F64 || COLL != COLL_SRT, "FP64 SRT runs as TRT");
    if constexpr (COLL == COLL_TRT) relax_pairs(g, c, drho, ux, uy, uz);
    else if constexpr (COLL == COLL_MRT && !kStochastic<STORE>) relax_rows(g, c, drho, ux, uy, uz);
    else relax_plain<COLL>(g, c, drho, ux, uy, uz);
}
// The combinations of relax_rows against the rows of M.
constexpr bool mrt_combinations_hold()
{
    for (int k = 0; k < Q; ++k) {
        const int x = ex(k), y = ey(k), z = ez(k), n2 = speed2(k);
        const int A = n2 == 1, D = n2 == 2, xy = D && !z, xz = D && !y, yz = D && !x;
        const int x9 = A * (2 * x * x - y * y - z * z), w9 = xy + xz - 2 * yz;
        const int x11 = A * (y * y - z * z), w11 = xy - xz;
        const int m[Q] = {1, -30 * (n2 == 0) - 11 * A + 8 * D, 12 * (n2 == 0) - 4 * A + D, x, x * (D - 4 * A), y,
                          y * (D - 4 * A), z, z * (D - 4 * A), x9 + w9, -2 * x9 + w9, x11 + w11, -2 * x11 + w11,
                          x * y, y * z, x * z, x * (xy - xz), y * (yz - xy), z * (xz - yz)};
        for (int i = 0; i < Q; ++i)
            if (m[i] != mrt_m(i, k)) return false;
    }
    return true;
}
static_assert(mrt_combinations_hold(), "the combinations of relax_rows are the rows of M");

// Periodic wrap of c + d into [0, n) for |d| <= 2 (any n >= 1).
__device__ __forceinline__ int wrap2(int c, int n)
{
    if (c < 0) c += n;
    if (c < 0) c += n;
    if (c >= n) c -= n;
    if (c >= n) c -= n;
    return c;
}

// Cells of the periodic images of x + e_k and x + 2 e_k (x_f2, x_f3 of the link (x, kbar));
// xv2 / xv3 receive their virtual x coordinates (outside [0, nx) across an x face).
template <typename R>
__device__ __forceinline__ void link_neighbours(const Par<R> &P, uint32_t cell, int k, uint32_t &c2, int &xv2,
                                                uint32_t &c3, int &xv3)
{
    const uint32_t yz = fast_div(cell, P.dnx);
    const int x = (int)(cell - yz * P.nx);
    const uint32_t zz = fast_div(yz, P.dny);
    const int y = (int)(yz - zz * P.ny), z = (int)zz;
    const int nx = (int)P.nx, ny = (int)P.ny, nz = (int)P.nz;
    xv2 = x + ex(k);
    xv3 = x + 2 * ex(k);
    c2 = (uint32_t)wrap2(xv2, nx) + P.nx * ((uint32_t)wrap2(y + ey(k), ny) + P.ny * (uint32_t)wrap2(z + ez(k), nz));
    c3 = (uint32_t)wrap2(xv3, nx) +
         P.nx * ((uint32_t)wrap2(y + 2 * ey(k), ny) + P.ny * (uint32_t)wrap2(z + 2 * ez(k), nz));
}

// Population of direction m read at a virtual x coordinate: the pressure shift of a value
// that crossed an x face (Sec. 2.2.2, as for the pulls).
template <typename R> __device__ __forceinline__ R shifted(R v, int xv, int nx, R w, R dshift)
{
    return xv < 0 ? fma_r(w, dshift, v) : (xv >= nx ? fma_r(-w, dshift, v) : v);
}

// The neighbour terms alpha P2 + beta P3 + delta B2 + zeta J2 of an interpolated wall rule
// (kLinkW) of link (x, kbar), x - e_k solid, added to v (which holds S); p2 is the cell's
// ordinary pull of direction kbar.  The loads the rule may need are issued before its
// coefficients arrive (a coefficient of 0 -- a fallback -- multiplies a finite value read
// from a solid cell's slot).
template <int STORE, typename R>
__device__ __forceinline__ R wall_neighbour_terms(const Par<R> &P, int wall, const R *lw, int k, uint32_t cell, R p2,
                                                  const typename Store<STORE>::T *fs, R v)
{
    using S = Store<STORE>;
    const int kb = opp_rt(k);
    const uint64_t keep = l2_keep_policy();
    if (wall == 3 || wall == 5) {  // QIBB, MR: P3 = g~_kbar(x_f3), B2 = g~_k(x_f2)
        int xv2, xv3;
        uint32_t c2, c3;
        link_neighbours(P, cell, k, c2, xv2, c3, xv3);
        const R w = k < 7 ? R(weight(1)) : R(weight(7));
        const R b2 = shifted(S::cvt(__ldg(fs + ((uint32_t)k * P.ks + c2))), xv2, (int)P.nx, w, P.c.dshift);
        const R p3 = shifted(S::cvt(__ldg(fs + ((uint32_t)kb * P.ks + c3))), xv3, (int)P.nx, w, P.c.dshift);
        v = fma_r(ld_keep(lw + LW_ALPHA, keep), p2, v);
        v = fma_r(ld_keep(lw + LW_BETA, keep), p3, v);
        v = fma_r(ld_keep(lw + LW_DELTA, keep), b2, v);
    } else if (wall == 4) {  // IEBB: J2 = e_kbar . (momentum of x_f2); the shift carries none
        int xv2, xv3;
        uint32_t c2, c3;
        link_neighbours(P, cell, k, c2, xv2, c3, xv3);
        const int x = -ex_rt(k), y = -ey_rt(k), z = -ez_rt(k);
        R j2 = R(0);
#pragma unroll
        for (int m = 1; m < Q; ++m) {
            const int d = x * ex(m) + y * ey(m) + z * ez(m);
            if (d != 0) j2 = fma_r(R(d), S::cvt(__ldg(fs + ((uint32_t)m * P.ks + c2))), j2);
        }
        v = fma_r(ld_keep(lw + LW_ZETA, keep), j2, v);
    } else {  // LIBB
        v = fma_r(ld_keep(lw + LW_ALPHA, keep), p2, v);
    }
    return v;
}

// The own-cell part S of an interpolated wall rule (kLinkW) from the cell's post-collision
// values B = g~_k, C = g~_kbar and its moments drho, u at this step.
template <typename R>
__device__ __forceinline__ R wall_own_part_w(const Par<R> &P, const R *lw, int k, R B, R C, R drho, R ux, R uy, R uz)
{
    const uint64_t keep = l2_keep_policy();
    R sv = fma_r(ld_keep(lw + LW_GAMMA, keep), B, ld_keep(lw + LW_EPS, keep) * C);
    const R X = ld_keep(lw + LW_X, keep);
    if (X != R(0)) {
        const R eu = R(-ex_rt(k)) * ux + R(-ey_rt(k)) * uy + R(-ez_rt(k)) * uz;
        const R uu = ux * ux + uy * uy + uz * uz;
        const R fst = drho + P.c.rho0 * (ld_keep(lw + LW_THETA, keep) * eu + R(4.5) * eu * eu - R(1.5) * uu);
        sv = fma_r(X * (k < 7 ? R(weight(1)) : R(weight(7))), fst, sv);
    }
    return sv;
}

// Pressure shift of the pulls that crossed the x boundary (wall directions take their value
// from the wall rule instead).
template <typename R> __device__ __forceinline__ void pressure_shift(R (&g)[Q], const Par<R> &P, uint32_t xf, uint32_t wm)
{
    if (xf & 1u) {
#pragma unroll
        for (int k = 0; k < Q; ++k)
            if (ex(k) == 1 && !((wm >> k) & 1u)) g[k] += R(weight(k)) * P.c.dshift;
    }
    if (xf & 2u) {
#pragma unroll
        for (int k = 0; k < Q; ++k)
            if (ex(k) == -1 && !((wm >> k) & 1u)) g[k] -= R(weight(k)) * P.c.dshift;
    }
}

// Stores of one cell's post-collision values: A-B slot k, AA LOCAL slot kbar of the cell, AA
// PULL slot k of x + e_k.
template <int STORE, int KIND, typename R>
__device__ __forceinline__ void store_cell(const InstanceDev &I, const Par<R> &P, const R (&g)[Q], uint32_t cell,
                                           uint32_t xf, bool inner, RoundKey key, typename Store<STORE>::T *fd)
{
    const uint32_t KS = P.ks;
    if constexpr (KIND == KIND_AA_PULL) {
        if (inner) {  // interior cell: x + e_k is cell + e_k, except across the x faces
            const uint32_t cxm = (xf & 1u) ? P.nx : 0u, cxp = (xf & 2u) ? P.nx : 0u;
            auto at = [&](int k) {
                uint32_t idx = cell + I.push_off[k];
                if (ex(k) == 1) idx -= cxp;
                if (ex(k) == -1) idx += cxm;
                return idx;
            };
            auto ok = [&](int k) { return checked(I, at(k) - (uint32_t)k * KS, I.n32); };
            if (ok(0)) put1<STORE>(fd + at(0), g[0], key, 0);
#pragma unroll
            for (int k = 1; k < Q; k += 2)
                if (ok(k) && ok(k + 1)) put2<STORE>(fd + at(k), fd + at(k + 1), g[k], g[k + 1], key, k, k + 1);
        } else {
            const Coord co = coord_of(P, cell);
            put1<STORE>(fd + co.push(0), g[0], key, 0);
#pragma unroll
            for (int k = 1; k < Q; k += 2)
                put2<STORE>(fd + ((uint32_t)k * KS + co.push(k)), fd + ((uint32_t)(k + 1) * KS + co.push(k + 1)), g[k],
                            g[k + 1], key, k, k + 1);
        }
    } else {
        // AA LOCAL: the slots the pull read; their addresses are computed again here, not kept
        // in 38 registers since (kept, the step spilled 196 bytes at 56 registers)
        asm volatile("" : "+r"(cell));
        put1<STORE>(fd + cell, g[0], key, 0);
#pragma unroll
        for (int k = 1; k < Q; k += 2) {
            const int ka = KIND == KIND_AB ? k : k + 1, kb = KIND == KIND_AB ? k + 1 : k;
            put2<STORE>(fd + ((uint32_t)ka * KS + cell), fd + ((uint32_t)kb * KS + cell), g[k], g[k + 1], key, k, k + 1);
        }
    }
}

// One warp's work item: 32 fluid cells of the work list (w = its index), their raw pulled
// values (see pull_item) and what the finish needs.
struct WarpItem {
    uint32_t cell;     // this lane's cell (0xFFFFFFFF: padding lane)
    uint32_t xf;       // bit 0: x = 0, bit 1: x = nx - 1 (pulls and pushes across the x faces)
    uint32_t wm;       // boundary cell: wall mask (bit k: x - e_k solid); else 0
    bool inner;        // every live lane away from the y and z faces (padding lanes: undefined)
};

// Walls.  The pull of a wall direction k reads, in the A-B layout, slot k of the solid cell
// x - e_k, which no fluid cell owns; every step leaves there the own-cell part S of the wall
// rule for the next step (wall_own_part, from its post-collision values in registers), so
// SBB needs no wall code before the collision at all and CLI adds c g_kbar^in, g_kbar^in
// being the cell's ordinary pull from x_f2 = x + e_k.  AA: the same, with S where the AA
// layout's pull reads (see above).  A state set from outside (initial state, imported
// populations) gets these slots from wall_prepare_kernel.  Momentum exchange: a link (x,
// kbar) with x - e_k solid carries g~_kbar(x) into the wall and brings the new g_k back, so
// the solid gains e_kbar (g~_kbar(x) + g_k).  (Deviations suffice: the 2 w rho0 of full
// populations sums to zero over a periodic domain.)
//
// A work item's links are handled one to a lane, not one direction after the other by the
// lanes of the cells: on the r = 60 sphere in 128^3 an item with walls has 24 links, of 9
// directions, at 5.4 of its cells, so a loop over the directions would run 9 times, each
// with its own coefficient load, for a third of a lane's work each.  The cells' values go
// through shared memory: the lanes of boundary cells write their 18 values, the links' lanes
// take the two of theirs, and, before the collision, write the new g_k back for the cells'
// lanes to read.
// Per step against the loop over the directions: FP64 20^3 9.9 -> 6.9 us, 128^3 311 -> 278;
// BF16 AA 48^3 4.48 -> 4.07, 128^3 25.7 -> 23.7; FP16 A-B 48^3 4.56 -> 4.30, 128^3 33.3 -> 32.0;
// FP32 A-B 80^3 9.06 -> 8.42, MR walls 128^3 67 -> 46; FP32 AA 48^3 to 256^3 within 1 %.
template <typename R> struct WallStage {
    static constexpr int kStride = 33;  // two links of one cell meet different banks
    R *v;                               // [18 directions, then drho, u_x, u_y, u_z (WX)][kStride]
    __device__ __forceinline__ R &at(int k, int lane) const { return v[(k - 1) * kStride + lane]; }
};
template <typename R, bool WX> constexpr int kWallStage = (WX ? Q + 3 : Q - 1) * WallStage<R>::kStride;

// A lane's link of the item: n = the item's links, first = the first of them, and of link
// first + lane (the first 32) its direction, its cell's lane, its CLI coefficient and its
// index in cell order (interpolated rules).
template <typename R> struct LinkOfLane {
    uint32_t n, first;
    uint32_t dir, lane;
    R c;
    uint32_t index;
};
// BRICK: the warp's cells are a 32-cell segment of the box, its links counted in cell order.
template <bool WX, bool BRICK, typename R>
__device__ __forceinline__ void load_link(const InstanceDev &I, const Par<R> &P, uint32_t l, LinkOfLane<R> &L)
{
    const uint64_t keep = l2_keep_policy();
    const uint32_t r = ld_keep((BRICK ? I.linkr : I.ilinkr) + l, keep);
    L.dir = r & 31u;
    L.lane = r >> 8;
    if (P.wall == 1) L.c = ld_keep(reinterpret_cast<const R *>(BRICK ? I.linkc : I.ilinkc) + l, keep);
    if (WX && P.wall >= 2) L.index = BRICK ? l : ld_keep(I.ilink + l, keep);
}
// The first 32 links of an item (n of them, from first): lane by lane, the others none.
template <bool WX, bool BRICK, typename R>
__device__ __forceinline__ LinkOfLane<R> first_links(const InstanceDev &I, const Par<R> &P, uint32_t n, uint32_t first,
                                                     int lane)
{
    LinkOfLane<R> L{n, first, 1u, 0u, R(0), 0u};
    // every link of the item within the link tables
    if (n && !checked(I, first + n, I.n_links + 1u)) L.n = 0u;
    if ((uint32_t)lane < L.n) load_link<WX, BRICK>(I, P, first + (uint32_t)lane, L);
    return L;
}

// The solid cell x - e_k of a link of a cell with face flags xf (as WarpItem's, bit 2: inner).
template <typename R>
__device__ __forceinline__ uint32_t solid_of(const Par<R> &P, uint32_t cell, uint32_t xf, int k)
{
    const int dx = ex_rt(k), dy = ey_rt(k), dz = ez_rt(k);
    if (xf & 4u) {
        uint32_t s = cell - (uint32_t)(dx + (int)P.nx * (dy + (int)P.ny * dz));
        if (dx == 1 && (xf & 1u)) s += P.nx;
        if (dx == -1 && (xf & 2u)) s -= P.nx;
        return s;
    }
    const uint32_t yz = fast_div(cell, P.dnx), zz = fast_div(yz, P.dny);
    const int x = (int)(cell - yz * P.nx), y = (int)(yz - zz * P.ny), z = (int)zz;
    return (uint32_t)wrap2(x - dx, (int)P.nx) +
           P.nx * ((uint32_t)wrap2(y - dy, (int)P.ny) + P.ny * (uint32_t)wrap2(z - dz, (int)P.nz));
}

// Before the collision: the rule's neighbour terms, and with RED the momentum exchange.
template <int STORE, int KIND, bool RED, bool WX, bool BRICK, typename R>
__device__ __forceinline__ void walls_in(const InstanceDev &I, const Par<R> &P, R (&g)[Q], const WarpItem &it,
                                         LinkOfLane<R> L, const WallStage<R> &st, int lane,
                                         const typename Store<STORE>::T *fs, R (&fm)[3])
{
    using S = Store<STORE>;
    if (L.n == 0 || (!RED && P.wall == 0)) return;  // the same in all lanes
    if (it.wm) {
#pragma unroll
        for (int k = 1; k < Q; ++k) st.at(k, lane) = g[k];
    }
    __syncwarp();
    for (uint32_t b = 0; b < L.n; b += 32) {
        const uint32_t j = b + (uint32_t)lane;
        const bool mine = j < L.n;
        if (mine && b > 0) load_link<WX, BRICK>(I, P, L.first + j, L);
        const int k = (int)L.dir, kb = opp_rt(k), from = (int)L.lane;
        const uint32_t lc = __shfl_sync(0xffffffffu, it.cell, from);
        const uint32_t lx = RED && KIND == KIND_AA_LOCAL ? __shfl_sync(0xffffffffu, it.xf | (it.inner ? 4u : 0u), from) : 0u;
        if (mine) {
            R v = st.at(k, from);  // S, left by the previous step where this pull reads
            if (WX && KIND == KIND_AB && P.wall >= 2)
                v = wall_neighbour_terms<STORE>(P, P.wall,
                                                reinterpret_cast<const R *>(I.linkw) + (size_t)L.index * kLinkW, k,
                                                lc, st.at(kb, from), fs, v);
            else if (L.c != R(0)) v = fma_r(L.c, st.at(kb, from), v);
            st.at(k, from) = v;
            if constexpr (RED) {
                // the own post-collision g~_kbar(x) of the previous step: A-B: own slot kbar; AA
                // after a LOCAL step: own slot k; AA after a PULL step: where it was pushed,
                // slot kbar of x - e_k
                const uint32_t d = (uint32_t)(KIND == KIND_AA_PULL ? k : kb);
                const uint32_t at = KIND == KIND_AA_LOCAL ? solid_of(P, lc, lx, k) : lc;
                if (checked(I, at, I.n32)) {
                    const R m = S::cvt(ld_pop<KIND>(fs + (d * P.ks + at))) + v;  // e_kbar = -e_k
                    fm[0] -= R(ex_rt(k)) * m;
                    fm[1] -= R(ey_rt(k)) * m;
                    fm[2] -= R(ez_rt(k)) * m;
                }
            }
        }
    }
    __syncwarp();
    if (it.wm) {
#pragma unroll
        for (int k = 1; k < Q; ++k) g[k] = st.at(k, lane);
    }
}

// After it: the own-cell part of every link's rule from the post-collision values, where the
// next step's pull of direction k reads it: A-B slot k of x - e_k in the buffer written; AA
// LOCAL slot kbar of x - e_k; AA PULL the own slot k.
template <int STORE, int KIND, bool WX, bool BRICK, typename R>
__device__ __forceinline__ void walls_out(const InstanceDev &I, const Par<R> &P, const R (&g)[Q], R drho, R ux, R uy,
                                          R uz, const WarpItem &it, LinkOfLane<R> L, const WallStage<R> &st, int lane,
                                          typename Store<STORE>::T *fd)
{
    if (L.n == 0) return;
    if (it.wm) {
#pragma unroll
        for (int k = 1; k < Q; ++k) st.at(k, lane) = g[k];
        if constexpr (WX) {
            st.at(Q, lane) = drho;
            st.at(Q + 1, lane) = ux;
            st.at(Q + 2, lane) = uy;
            st.at(Q + 3, lane) = uz;
        }
    }
    __syncwarp();
    for (uint32_t b = 0; b < L.n; b += 32) {
        const uint32_t j = b + (uint32_t)lane;
        const bool mine = j < L.n;
        if (mine && b > 0) load_link<WX, BRICK>(I, P, L.first + j, L);
        const int k = (int)L.dir, kb = opp_rt(k), from = (int)L.lane;
        const uint32_t lc = __shfl_sync(0xffffffffu, it.cell, from);
        const uint32_t lx = KIND != KIND_AA_PULL ? __shfl_sync(0xffffffffu, it.xf | (it.inner ? 4u : 0u), from) : 0u;
        if (mine) {
            const R B = st.at(k, from), C = st.at(kb, from);
            R sv;
            if (WX && P.wall >= 2)
                sv = wall_own_part_w(P, reinterpret_cast<const R *>(I.linkw) + (size_t)L.index * kLinkW, k, B, C,
                                     st.at(Q, from), st.at(Q + 1, from), st.at(Q + 2, from), st.at(Q + 3, from));
            else sv = wall_own_part(P.wall, L.c, C, B);
            const uint32_t d = (uint32_t)(KIND == KIND_AA_LOCAL ? kb : k);
            const uint32_t at = KIND == KIND_AA_PULL ? lc : solid_of(P, lc, lx, k);
            if (checked(I, at, I.n32))
                put1<STORE>(fd + (d * P.ks + at), sv, round_key<STORE>(lc, P.hash_off), k);
        }
    }
}

// Work item w of a work list (flane, fwarp): this lane's entry and the item's links (number and
// first), precomputed in tables that no step writes (no division).  The entries of a run are
// not read but made from the item's: two thirds of the items of the r = 60 sphere in 128^3,
// nine tenths in 512^3, so that the list costs 3 and 1 bytes a cell instead of 8.  early: the
// entries are asked for with the item's, needed or not (a step of few tiles waits for one
// load's latency less; Batch::early).  Per step, entries always read -> of runs made: FP32 AA
// 128^3 28.1 -> 27.5 us, 256^3 257.6 -> 252.0, A-B 384^3 873 -> 847; BF16 AA 256^3 199 -> 191,
// 384^3 676 -> 655; FP16 A-B 256^3 219 -> 213.
struct ItemEntry {
    uint2 cell, links;
};
__device__ __forceinline__ ItemEntry load_entry(const uint2 *flane, const uint4 *fwarp, uint32_t w, int lane, bool ok,
                                                bool early)
{
    const uint64_t keep = l2_keep_policy();
    ItemEntry e;
    e.cell = make_uint2(0xFFFFFFFFu, 0u);
    if (ok && early) e.cell = ld_keep(flane + (w * 32u + (uint32_t)lane), keep);
    const uint4 h = ok ? ld_keep(fwarp + w, keep) : make_uint4(0u, 0u, 0u, 0u);
    e.links = make_uint2(h.x, h.y);
    if (!early) {
        if (h.z >> 31) {
            e.cell.x = run_entry(h.z, h.w, (uint32_t)lane);
        } else if (ok) {
            e.cell = ld_keep(flane + (w * 32u + (uint32_t)lane), keep);
        }
    }
    return e;
}
// This lane's cell, its x-face flags and wall mask, and whether every lane is away from the y
// and z faces.
__device__ __forceinline__ WarpItem locate_item(const InstanceDev &I, const ItemEntry &e)
{
    WarpItem it;
    const bool live = e.cell.x != 0xFFFFFFFFu;
    it.cell = live ? (e.cell.x & 0x0FFFFFFFu) : 0xFFFFFFFFu;
    if (live && !checked(I, it.cell, I.n32)) it.cell = 0xFFFFFFFFu;
    it.xf = live ? (e.cell.x >> 28) & 3u : 0u;
    it.inner = ((e.cell.x >> 30) & 1u) != 0u;  // the same in all live lanes of the item
    it.wm = e.cell.y;
    return it;
}

// Issue the 19 pulls of a located work item into raw[] (storage type, converted in
// finish_item).  Unconditional: the slot of a solid source holds the wall's part (see above).
// Warps whose cells are all away from the y and z faces index through precomputed offsets (cell +
// pull_off[k], with a fix-up on the first and last cell of a row); the others through their
// periodic neighbours.
template <int STORE, int KIND, typename R>
__device__ __forceinline__ void pull_item(const InstanceDev &I, const Par<R> &P, const typename Store<STORE>::T *fs,
                                          const WarpItem &it, typename Store<STORE>::T (&raw)[Q])
{
    if (it.cell == 0xFFFFFFFFu) {
#pragma unroll
        for (int k = 0; k < Q; ++k) raw[k] = typename Store<STORE>::T{};
        return;
    }
    if (KIND != KIND_AA_LOCAL && it.inner) {
        const uint32_t cxm = (it.xf & 1u) ? P.nx : 0u, cxp = (it.xf & 2u) ? P.nx : 0u;
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            uint32_t idx = it.cell + I.pull_off[k];
            if (ex(k) == 1) idx += cxm;   // x - 1 wraps to the end of the row
            if (ex(k) == -1) idx -= cxp;  // x + 1 wraps to the start of the row
            const uint32_t d = KIND == KIND_AA_PULL ? (uint32_t)opp(k) : (uint32_t)k;
            raw[k] = checked(I, idx - d * P.ks, I.n32) ? ld_pop<KIND>(fs + idx) : typename Store<STORE>::T{};
        }
    } else {
        const Coord co = coord_of(P, it.cell);
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            uint32_t idx;
            if constexpr (KIND == KIND_AA_LOCAL) idx = (uint32_t)k * P.ks + it.cell;
            else if constexpr (KIND == KIND_AA_PULL) idx = (uint32_t)opp(k) * P.ks + co.pull(k);
            else idx = (uint32_t)k * P.ks + co.pull(k);
            const uint32_t d = KIND == KIND_AA_PULL ? (uint32_t)opp(k) : (uint32_t)k;
            raw[k] = checked(I, idx - d * P.ks, I.n32) ? ld_pop<KIND>(fs + idx) : typename Store<STORE>::T{};
        }
    }
}

// Per-lane values of the reduction (RED steps) in the compute type: one cell a lane.
template <typename R> struct RedAcc {
    R v[RED_F + 3];
};

// Finish one work item pulled by pull_item: convert, pressure shift of the pulls that
// crossed the x boundary, walls, moments and collision, stores; with RED, add the lane's
// moments and momentum exchange to acc.  Padding lanes take part (they may hold a link) on
// zeros and store nothing.
template <int COLL, int STORE, int KIND, bool RED, bool WX, bool BRICK, typename R>
__device__ __forceinline__ void finish_item(const InstanceDev &I, const Par<R> &P,
                                            const typename Store<STORE>::T (&raw)[Q], const WarpItem &it,
                                            const LinkOfLane<R> &L, const WallStage<R> &st, int lane,
                                            const typename Store<STORE>::T *fs, typename Store<STORE>::T *fd,
                                            RedAcc<R> &acc)
{
    using S = Store<STORE>;
    const bool live = it.cell != 0xFFFFFFFFu;
    R g[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) g[k] = S::cvt(raw[k]);
    pressure_shift(g, P, it.xf, it.wm);
    R fm[3] = {R(0), R(0), R(0)};
    walls_in<STORE, KIND, RED, WX, BRICK>(I, P, g, it, L, st, lane, fs, fm);
    R drho, ux, uy, uz;
    relax<COLL, STORE>(g, P.c, drho, ux, uy, uz);
    if constexpr (RED) {
        const R unit = STORE == ST_F16 ? R(P.isc) : R(1);  // FP16: from the stored units
        if (live) {
            const R uu = ux * ux + uy * uy + uz * uz;
            if (!(uu < R(1)) || !(drho == drho)) atomicOr(I.status, STATUS_DIVERGED);
            acc.v[RED_DRHO] += drho * unit;
            acc.v[RED_U + 0] += ux;
            acc.v[RED_U + 1] += uy;
            acc.v[RED_U + 2] += uz;
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) acc.v[RED_F + d] += fm[d] * unit;
    }
    if (live) store_cell<STORE, KIND>(I, P, g, it.cell, it.xf, it.inner, round_key<STORE>(it.cell, P.hash_off), fd);
    walls_out<STORE, KIND, WX, BRICK>(I, P, g, drho, ux, uy, uz, it, L, st, lane, fd);
}

// Error-free sum (Knuth's TwoSum): s + e == a + b exactly, s = fl(a + b).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Warp sum of float-float values hi + lo (fixed butterfly; every lane ends with the same
// pair, the exact TwoSum error being unique).  Each addition keeps its rounding error, so
// hi + lo is the sum to about 2^-48 of the magnitudes added, close to an FP64 sum, on the
// FP32 pipes (GB300's FP64 rate made the FP64 butterfly the cost of the reducing step).
__device__ __forceinline__ void warp_sum_ff(float &hi, float &lo)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
        const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
        float sh, se;
        two_sum(hi, h2, sh, se);
        se = __fadd_rn(se, __fadd_rn(lo, l2));
        two_sum(sh, se, hi, lo);
    }
}

// Block sum of the lanes' values of one tile (fixed shuffle tree, then the warps in order)
// to partials[tile] in FP64; every thread of the block calls it.  FP64 lanes sum in FP64;
// FP32 lanes sum in float-float within the warp, then in FP64.
template <typename R>
__device__ __forceinline__ void reduce_tile(const RedAcc<R> &acc, double *partials, long long tile)
{
    __shared__ double red[kStepWarps][RED_F + 3];  // the reducing step runs kStepWarps-warp blocks
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double v[RED_F + 3];
#pragma unroll
    for (int d = 0; d < RED_F + 3; ++d) {
        if constexpr (sizeof(R) == sizeof(double)) {
            v[d] = warp_sum((double)acc.v[d]);
        } else {
            float hi = (float)acc.v[d], lo = 0.0f;
            warp_sum_ff(hi, lo);
            v[d] = (double)hi + (double)lo;
        }
    }
    if (lane == 0)
#pragma unroll
        for (int d = 0; d < RED_F + 3; ++d) red[warp][d] = v[d];
    __syncthreads();
    if (threadIdx.x < RED_F + 3) {
        double sum = 0.0;
        for (int w = 0; w < kStepWarps; ++w) sum += red[w][threadIdx.x];
        partials[tile * kRedSlots + threadIdx.x] = sum;
    }
}

// Programmatic dependent launch (sm_90 and later): a step lets the next step's blocks be
// scheduled as soon as all of its own blocks are running, and a step waits for the
// previous one to complete (with its memory visible) only before its first population
// load.  Between the two, a block reads its tile and work list, which no step writes.
__device__ __forceinline__ void allow_next_step() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous_step() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The tile t of a launch.  A single instance's tiles are consecutive: tile t holds work items
// WARPS t ... (no load precedes the work list's).
template <bool BATCH, int WARPS>
__device__ __forceinline__ TileDev tile_of(const MapArg<BATCH> &map, const TileDev *tiles, int t)
{
    if constexpr (BATCH) {
        if (map.n == 0) return tiles[t];
        int lo = 0, hi = map.n - 1;  // the instance whose tiles hold t: the last i with tile_start[i] <= t
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (map.tile_start[mid] <= t) lo = mid;
            else hi = mid - 1;
        }
        const int local = t - map.tile_start[lo];
        return TileDev{lo, local, (long long)local * WARPS, map.flane[lo], map.fwarp[lo]};
    } else {
        return TileDev{0, t, (long long)t * WARPS, nullptr, nullptr};
    }
}

// The parameters of a block's instance: a single instance's in the constant bank; a batch's
// block copies its instance's to shared memory (params), where they are read in the same way,
// at their use, not held in registers.
template <bool BATCH> constexpr int kParamWords = BATCH ? (int)(sizeof(InstanceDev) / sizeof(uint4)) : 1;
static_assert(sizeof(InstanceDev) % sizeof(uint4) == 0, "copied in 16-byte pieces");
template <bool BATCH, int WARPS>
__device__ __forceinline__ const InstanceDev &instance_of(const InstanceDev *table, const InstanceDev &one, int inst,
                                                          uint4 *params)
{
    if constexpr (BATCH) {
        for (int i = threadIdx.x; i < kParamWords<BATCH>; i += WARPS * 32)
            params[i] = __ldg(reinterpret_cast<const uint4 *>(table + inst) + i);
        __syncthreads();
        return *reinterpret_cast<const InstanceDev *>(params);
    } else {
        return one;
    }
}

// The fused step.  One block of WARPS warps per tile of WARPS work items (32 fluid cells
// each), one item per warp.  Each cell's arithmetic does not depend on WARPS, so every block
// shape gives the same state bit for bit; the reducing step always runs kStepWarps-warp
// tiles.  A single instance's parameters travel by value (constant bank); a batch's come
// from the device table.  flip selects the A-B buffer pair (src = f[phase ^ flip], bit 0)
// and the order of the tiles (bit kStepBackwards).  The RED variant (the step that ends a
// chunk) also makes every tile write its FP64 partial sums (the kRedSlots slots: drho, u_x,
// u_y, u_z and the momentum exchanged with the solid) and flags diverged cells in
// the instance's status word; the other steps carry none of that code.  The WX variant (A-B only)
// also runs the interpolated wall rules LIBB, QIBB, IEBB and MR.
template <int COLL, int STORE, int KIND, bool BATCH, bool RED, bool WX, int WARPS = kStepWarps>
__global__ void __launch_bounds__(WARPS * 32, step_min_blocks<STORE, COLL, RED, WX, WARPS, KIND, BATCH>())
    step_kernel(const InstanceDev *__restrict__ table, const __grid_constant__ InstanceDev one,
                const __grid_constant__ MapArg<BATCH> map, const TileDev *__restrict__ tiles, int ntiles, int flip)
{
    static_assert(!RED || WARPS == kStepWarps, "the reducing step runs kStepWarps-warp tiles");
    using S = Store<STORE>;
    using T = typename S::T;
    using R = typename S::R;
    allow_next_step();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if ((int)blockIdx.x >= ntiles) return;
    const int t = (flip & kStepBackwards) ? ntiles - 1 - (int)blockIdx.x : (int)blockIdx.x;
    // a single instance's tiles are consecutive: tile t holds work items WARPS t ... (its
    // table entry holds the same, so that no load precedes the work list's)
    const TileDev tile = tile_of<BATCH, WARPS>(map, tiles, t);
    const uint32_t w = (uint32_t)tile.seg0 + (uint32_t)warp;
    ItemEntry entry;
    // a batch's entries are loaded beside its parameters, not after them (the checked build needs
    // their number first)
    if constexpr (BATCH && !kChecked) entry = load_entry(tile.flane, tile.fwarp, w, lane, true, flip & kStepEarly);
    __shared__ uint4 params[kParamWords<BATCH>];
    const InstanceDev &I = instance_of<BATCH, WARPS>(table, one, tile.inst, params);
    if constexpr (!BATCH || kChecked)
        entry = load_entry(BATCH ? tile.flane : I.flane, BATCH ? tile.fwarp : I.fwarp, w, lane,
                           checked(I, w, I.n_fwarps_padded), flip & kStepEarly);
    const Par<R> P = load_par<R>(I);
    const T *fs;  // state read this step
    T *fd;        // state written this step
    if constexpr (KIND == KIND_AB) {
        const int cur = I.phase ^ (flip & 1);
        fs = reinterpret_cast<const T *>(cur ? I.f1 : I.f0);
        fd = reinterpret_cast<T *>(cur ? I.f0 : I.f1);
    } else {
        fd = reinterpret_cast<T *>(I.f0);
        fs = fd;
    }
    __shared__ R stage[WARPS * kWallStage<R, WX>];
    const WallStage<R> st{stage + warp * kWallStage<R, WX>};
    const WarpItem it = locate_item(I, entry);
    wait_previous_step();
    T raw[Q];
    pull_item<STORE, KIND, R>(I, P, fs, it, raw);
    // issued behind the pulls (before them its registers cost FP32 AA 256^3 2 %)
    const LinkOfLane<R> L = first_links<WX, false, R>(I, P, entry.links.x, entry.links.y, lane);
    RedAcc<R> acc{};
    finish_item<COLL, STORE, KIND, RED, WX, false, R>(I, P, raw, it, L, st, lane, fs, fd, acc);
    if constexpr (RED) reduce_tile(acc, I.partials, tile.local);
}

}  // namespace lbm
