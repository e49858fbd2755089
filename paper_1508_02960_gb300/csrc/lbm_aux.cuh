// lbm_aux.cuh -- kernels around the time step: initial state, import/export of the
// populations as FP64, velocity field and moment sums of the stored state.  All of
// them see the state through stored_slot(): the post-collision population g~_k(x) in
// either layout.  Slots are 32-bit numbers: a box whose 19 directions hold 2^32 or more is
// refused at creation.
#pragma once

#include "lbm_device.cuh"
#include "lbm_step.cuh"

namespace lbm {

// Where g~_k(x) of a fluid cell lives.  A-B: slot k of the cell in the current buffer.  AA
// after a LOCAL step (or import): own slot kbar.  AA after a PULL step: slot k of x + e_k (a
// solid cell's slot when x + e_k is solid: the link's own slot there).
enum Arrangement { ARR_OWN = 0, ARR_OPPOSITE = 1, ARR_NEIGHBOUR = 2 };
__device__ __forceinline__ Arrangement arrangement(int layout, int aa_phase)
{
    return layout == 0 ? ARR_OWN : aa_phase == 0 ? ARR_OPPOSITE : ARR_NEIGHBOUR;
}

template <int STORE>
__device__ __forceinline__ typename Store<STORE>::T *state_buffer(const InstanceDev &I, int layout, int cur)
{
    return reinterpret_cast<typename Store<STORE>::T *>(layout == 0 && cur ? I.f1 : I.f0);
}

// The periodic neighbours of a cell: X[1 + a] + Y[1 + b] + Z[1 + c] is the cell at (a, b, c).
struct Around {
    uint32_t X[3], Y[3], Z[3];
};
__device__ __forceinline__ Around around(const InstanceDev &I, uint32_t cell)
{
    const uint32_t nx = I.nx, ny = I.ny, nz = I.nz, nxy = nx * ny;
    const uint32_t yz = cell / nx, x = cell - yz * nx, z = yz / ny, y = yz - z * ny;
    Around a;
    a.X[0] = x == 0 ? nx - 1 : x - 1;
    a.X[1] = x;
    a.X[2] = x == nx - 1 ? 0 : x + 1;
    a.Y[0] = (y == 0 ? ny - 1 : y - 1) * nx;
    a.Y[1] = y * nx;
    a.Y[2] = (y == ny - 1 ? 0 : y + 1) * nx;
    a.Z[0] = (z == 0 ? nz - 1 : z - 1) * nxy;
    a.Z[1] = z * nxy;
    a.Z[2] = (z == nz - 1 ? 0 : z + 1) * nxy;
    return a;
}
__device__ __forceinline__ uint32_t slot_towards(const InstanceDev &I, const Around &a, int k)
{
    return (uint32_t)k * (uint32_t)I.ks + a.X[1 + ex(k)] + a.Y[1 + ey(k)] + a.Z[1 + ez(k)];
}
// One direction's slot (the neighbours, with their divisions, only where they are needed).
__device__ __forceinline__ uint32_t stored_slot(const InstanceDev &I, Arrangement arr, uint32_t cell, int k)
{
    if (arr == ARR_NEIGHBOUR) return slot_towards(I, around(I, cell), k);
    return (uint32_t)(arr == ARR_OWN ? k : opp(k)) * (uint32_t)I.ks + cell;
}
// All 19.
template <int STORE>
__device__ __forceinline__ void load_stored(const InstanceDev &I, const typename Store<STORE>::T *f, Arrangement arr,
                                            uint32_t cell, typename Store<STORE>::R (&g)[Q])
{
    using S = Store<STORE>;
    if (arr == ARR_NEIGHBOUR) {
        const Around a = around(I, cell);
#pragma unroll
        for (int k = 0; k < Q; ++k) g[k] = S::load(f + slot_towards(I, a, k), I.inv_scale);
    } else {
#pragma unroll
        for (int k = 0; k < Q; ++k)
            g[k] = S::load(f + ((uint32_t)(arr == ARR_OWN ? k : opp(k)) * (uint32_t)I.ks + cell), I.inv_scale);
    }
}

// Momentum sum_k e_k g_k in FP64.  GB300 runs an FP64 warp instruction per 19 cycles of a
// multiprocessor, so the terms that are no part of a component are left out: 21 operations
// from the differences of opposite directions, where multiplying all 19 populations by the
// components of e_k takes 57 (the velocity field of 96 x 80 x 72 cells in one pass instead of
// three of those: see velocity_kernel).  A population that is infinite or NaN takes the long
// form, whose 0 * g makes every component of the cell show it.
template <typename R> __device__ __forceinline__ void momentum(const R (&g)[Q], double (&j)[3])
{
    uint32_t top = 0;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        if constexpr (sizeof(R) == 8) top = max(top, (uint32_t)__double2hiint(g[k]) & 0x7fffffffu);
        else top = max(top, __float_as_uint(g[k]) & 0x7fffffffu);
    }
    j[0] = j[1] = j[2] = 0.0;
    if (top >= (sizeof(R) == 8 ? 0x7ff00000u : 0x7f800000u)) {
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            j[0] += ex(k) * (double)g[k];
            j[1] += ey(k) * (double)g[k];
            j[2] += ez(k) * (double)g[k];
        }
        return;
    }
#pragma unroll
    for (int k = 1; k < Q; ++k) {
        if (opp(k) < k) continue;
        const double d = (double)g[k] - (double)g[opp(k)];
        const int e[3] = {ex(k), ey(k), ez(k)};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (e[a] > 0) j[a] += d;
            if (e[a] < 0) j[a] -= d;
        }
    }
}

// SplitMix64 finaliser (Steele, Lea & Flood 2014) as a counter-based hash.
__device__ __forceinline__ unsigned long long mix64(unsigned long long z)
{
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__device__ __forceinline__ double hash_uniform_pm1(unsigned long long seed, long long cell, int comp)
{
    const unsigned long long h = mix64(seed ^ mix64((unsigned long long)cell * 3ull + (unsigned long long)comp));
    return ((double)(h >> 11) * (1.0 / 9007199254740992.0)) * 2.0 - 1.0;
}

// Equilibrium initial state g_k = f^eq_k(rho0, u) - w_k rho0 for fluid cells (u = 0 or a
// seeded perturbation of amplitude amp), 0 in solid cells.  Writes the layout's
// post-collision form (A-B buffer `cur`, or AA phase 0); the wall terms follow from
// wall_prepare_kernel.
template <int STORE>
__global__ void init_kernel(const InstanceDev *__restrict__ table, int inst, int layout, int cur,
                            double amp, unsigned long long seed)
{
    using S = Store<STORE>;
    using T = typename S::T;
    const InstanceDev &I = table[inst];
    const long long N = I.ncells;
    const int lane = threadIdx.x & 31;
    for (long long cell = (long long)blockIdx.x * blockDim.x + threadIdx.x; cell < N;
         cell += (long long)gridDim.x * blockDim.x) {
        const uint4 meta = I.seg[cell >> 5];
        T *f = state_buffer<STORE>(I, layout, cur);
        // at rest every g is 0, without the FP64 arithmetic (512^3: 24 ms with it)
        if (amp == 0.0 || ((meta.x >> lane) & 1u)) {
#pragma unroll
            for (int k = 0; k < Q; ++k) f[(long long)k * I.ks + cell] = S::pack(0.0f);
            continue;
        }
        double u[3];
        for (int a = 0; a < 3; ++a) u[a] = amp * hash_uniform_pm1(seed, cell, a);
        const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const double eu = ex(k) * u[0] + ey(k) * u[1] + ez(k) * u[2];
            const double g = weight(k) * I.rho0 * (3.0 * eu + 4.5 * eu * eu - 1.5 * uu);
            f[(long long)(layout == 0 ? k : opp(k)) * I.ks + cell] = S::pack((typename S::R)g * I.scale);
        }
    }
}

// The own-cell part S of every wall rule (wall_own_part), from the stored post-collision
// state, into the solid slot the next step's pull of direction k reads (the steps
// themselves leave S there for the step after them): A-B, from buffer cur into slot k of
// the solid cell x - e_k; AA at phase 0 (the state after a LOCAL step, where own slot m
// holds g~_mbar), into slot kbar of x - e_k.  For a state set from outside: the initial
// state, imported populations.  One thread per boundary cell; every solid slot belongs to
// one link only.
template <int STORE>
__global__ void wall_prepare_kernel(const InstanceDev *__restrict__ table, int inst, long long nb,
                                    const long long *__restrict__ bcell, int layout, int cur)
{
    using S = Store<STORE>;
    using T = typename S::T;
    using R = typename S::R;
    const InstanceDev &I = table[inst];
    T *f = state_buffer<STORE>(I, layout, cur);
    const R *linkc = reinterpret_cast<const R *>(I.linkc);
    const long long ks = I.ks;
    for (long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x; b < nb;
         b += (long long)gridDim.x * blockDim.x) {
        const long long cell = bcell[b];
        const uint32_t wm = I.bmask[b], off = I.boff[b];
        const Around at = around(I, (uint32_t)cell);
        const RoundKey key = round_key<STORE>((uint32_t)cell, I.cf.hash_off);
        // the cell's moments at t (for IEBB): the post-collision state conserves them
        R drho = R(0), u[3] = {R(0), R(0), R(0)};
        if (I.wall == 4) {
            for (int m = 0; m < Q; ++m) {
                const R gm = S::load(f + (long long)(layout == 0 ? m : opp(m)) * ks + cell, I.inv_scale);
                drho += gm;
                u[0] += R(ex(m)) * gm;
                u[1] += R(ey(m)) * gm;
                u[2] += R(ez(m)) * gm;
            }
            for (int a = 0; a < 3; ++a) u[a] /= R(I.rho0);
        }
        const R *linkw = reinterpret_cast<const R *>(I.linkw);
#pragma unroll
        for (int k = 1; k < Q; ++k) {
            if (!((wm >> k) & 1u)) continue;
            const int kb = opp(k);
            // C = g~_kbar(x), B = g~_k(x): slots kbar and k in A-B, k and kbar in AA
            const R C = S::load(f + (long long)(layout == 0 ? kb : k) * ks + cell, I.inv_scale);
            const R B = S::load(f + (long long)(layout == 0 ? k : kb) * ks + cell, I.inv_scale);
            const uint32_t l = off + __popc(wm & ((1u << k) - 1u));
            R sv;
            if (I.wall >= 2) {  // as wall_own_part_w in the step kernel
                const R *lw = linkw + (size_t)l * kLinkW;
                sv = fma_r(lw[LW_GAMMA], B, lw[LW_EPS] * C);
                const R X = lw[LW_X];
                if (X != R(0)) {
                    const R eu = R(ex(kb)) * u[0] + R(ey(kb)) * u[1] + R(ez(kb)) * u[2];
                    const R uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
                    const R fst = drho + R(I.rho0) * (lw[LW_THETA] * eu + R(4.5) * eu * eu - R(1.5) * uu);
                    sv = fma_r(X * R(weight(kb)), fst, sv);
                }
            } else {
                const R cq = I.wall == 1 ? linkc[l] : R(0);
                sv = wall_own_part(I.wall, cq, C, B);
            }
            const uint32_t src = at.X[1 - ex(k)] + at.Y[1 - ey(k)] + at.Z[1 - ez(k)];
            put1<STORE>(f + (long long)(layout == 0 ? k : kb) * ks + src, sv * R(I.scale), key, k);
        }
    }
}

// Import of FP64 f into directions k0 + blockIdx.y, cells c0 ... c0 + nc - 1, from
// fk[blockIdx.y * nc + cell - c0]: g = f - w rho0.  These transfers run at the speed of the
// host link (190-210 GB/s); the kernels only have to stay ahead of it, a pass in one staging
// buffer while the other is being copied.
template <int STORE>
__global__ void import_kernel(const InstanceDev *__restrict__ table, int inst, int layout, int cur, int k0,
                              long long c0, long long nc, const double *__restrict__ fk)
{
    using S = Store<STORE>;
    const InstanceDev &I = table[inst];
    const int k = k0 + (int)blockIdx.y;
    const double wr = weight(k) * I.rho0;
    auto *f = state_buffer<STORE>(I, layout, cur) + (long long)(layout == 0 ? k : opp(k)) * I.ks;
    fk += (long long)blockIdx.y * nc;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nc;
         i += (long long)gridDim.x * blockDim.x) {
        const long long cell = c0 + i;
        const bool solid = (I.seg[cell >> 5].x >> (cell & 31)) & 1u;
        f[cell] = solid ? S::pack(0.0f) : S::pack((typename S::R)(fk[i] - wr) * I.scale);
    }
}

// Export as FP64 f = w rho0 + g~ (0 in solid cells), arguments as import_kernel's.
template <int STORE>
__global__ void export_kernel(const InstanceDev *__restrict__ table, int inst, int layout, int cur,
                              int aa_phase, int k0, long long c0, long long nc, double *__restrict__ fk)
{
    using S = Store<STORE>;
    const InstanceDev &I = table[inst];
    const int k = k0 + (int)blockIdx.y;
    const double wr = weight(k) * I.rho0;
    const Arrangement arr = arrangement(layout, aa_phase);
    const auto *f = state_buffer<STORE>(I, layout, cur);
    fk += (long long)blockIdx.y * nc;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nc;
         i += (long long)gridDim.x * blockDim.x) {
        const long long cell = c0 + i;
        const bool solid = (I.seg[cell >> 5].x >> (cell & 31)) & 1u;
        fk[i] = solid ? 0.0 : wr + (double)S::load(f + stored_slot(I, arr, (uint32_t)cell, k), I.inv_scale);
    }
}

// The stored state of directions k0 + blockIdx.y of the fluid cells, bit for bit, in the
// storage type: out[blockIdx.y * nf + j] = the stored g~_k of fluid cell j (cells in cell
// order, from the work list), read where the layout keeps it (as export_kernel).
template <int STORE>
__global__ void state_gather_kernel(const InstanceDev *__restrict__ table, int inst, int layout, int cur,
                                    int aa_phase, int k0, long long nf, typename Store<STORE>::T *__restrict__ out)
{
    using T = typename Store<STORE>::T;
    const InstanceDev &I = table[inst];
    const int k = k0 + (int)blockIdx.y;
    const Arrangement arr = arrangement(layout, aa_phase);
    const T *f = state_buffer<STORE>(I, layout, cur);
    out += (long long)blockIdx.y * nf;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < nf;
         j += (long long)gridDim.x * blockDim.x) {
        out[j] = f[stored_slot(I, arr, I.fcell[j], k)];
    }
}

// The inverse for a state set from outside (as import_kernel, without conversion):
// direction k = k0 + blockIdx.y of fluid cell j from in[blockIdx.y * nf + j] into its slot
// of the step-0 arrangement.  Solid cells are left alone (their wall terms are rebuilt by
// wall_prepare_kernel).
template <int STORE>
__global__ void state_scatter_kernel(const InstanceDev *__restrict__ table, int inst, int layout, int cur, int k0,
                                     long long nf, const typename Store<STORE>::T *__restrict__ in)
{
    using T = typename Store<STORE>::T;
    const InstanceDev &I = table[inst];
    const int k = k0 + (int)blockIdx.y;
    in += (long long)blockIdx.y * nf;
    T *f = state_buffer<STORE>(I, layout, cur);
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < nf;
         j += (long long)gridDim.x * blockDim.x) {
        const long long cell = I.fcell[j];
        f[(long long)(layout == 0 ? k : opp(k)) * I.ks + cell] = in[j];
    }
}

// Velocity of cells c0 ... c0 + nc - 1 from the stored post-collision state (0 in solid
// cells): out[a * nc + cell - c0] = component a.
template <int STORE>
__global__ void __launch_bounds__(128) velocity_kernel(const InstanceDev *__restrict__ table, int inst, int layout,
                                                       int cur, int aa_phase, long long c0, long long nc,
                                                       double *__restrict__ out)
{
    const InstanceDev &I = table[inst];
    const Arrangement arr = arrangement(layout, aa_phase);
    const auto *f = state_buffer<STORE>(I, layout, cur);
    const double rho0 = I.rho0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nc;
         i += (long long)gridDim.x * blockDim.x) {
        const long long cell = c0 + i;
        double j[3] = {0.0, 0.0, 0.0};
        if (!((I.seg[cell >> 5].x >> (cell & 31)) & 1u)) {
            typename Store<STORE>::R g[Q];
            load_stored<STORE>(I, f, arr, (uint32_t)cell, g);
            momentum(g, j);
            if (rho0 != 1.0)  // an FP64 division is 10 FP64 instructions
                for (int a = 0; a < 3; ++a) j[a] /= rho0;
        }
        for (int a = 0; a < 3; ++a) out[a * nc + i] = j[a];
    }
}

// Moment sums of the stored post-collision state of every fluid cell of an instance, one
// warp per chunk of chunk_segs active segments: chunk partial sums (drho, u_x, u_y, u_z) into
// I.partials, in FP64 in a fixed order; the force slots, which only a step defines, are
// written as 0.
template <int STORE>
__global__ void __launch_bounds__(256) moments_kernel(const InstanceDev *__restrict__ table,
                                                      int inst, int nchunks, int chunk_segs,
                                                      int layout, int cur, int aa_phase)
{
    const InstanceDev &I = table[inst];
    const Arrangement arr = arrangement(layout, aa_phase);
    const auto *f = state_buffer<STORE>(I, layout, cur);
    const int lane = threadIdx.x & 31;
    const int gw = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
    const int nw = (int)((gridDim.x * (long long)blockDim.x) >> 5);
    for (int c = gw; c < nchunks; c += nw) {
        const long long seg0 = (long long)c * chunk_segs;  // chunk c of the active segments
        const int n_e = min(chunk_segs, (int)((long long)I.n_active - seg0));
        double a[4] = {0.0, 0.0, 0.0, 0.0};
        for (int i = 0; i < n_e; ++i) {
            const uint4 meta = I.aseg[seg0 + i];
            if ((meta.x >> lane) & 1u) continue;
            typename Store<STORE>::R g[Q];
            load_stored<STORE>(I, f, arr, meta.w * 32u + (uint32_t)lane, g);
            double j[3];
            momentum(g, j);
#pragma unroll
            for (int k = 0; k < Q; ++k) a[0] += (double)g[k];
            for (int d = 0; d < 3; ++d) a[1 + d] += j[d];
        }
#pragma unroll
        for (int d = 0; d < 4; ++d) a[d] = warp_sum(a[d]);
        if (lane == 0)
            for (int d = 0; d < kRedSlots; ++d)
                I.partials[(long long)c * kRedSlots + d] = d == 0 ? a[0] : d < 4 ? a[d] / I.rho0 : 0.0;
    }
}

}  // namespace lbm
