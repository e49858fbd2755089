// noalloc.cu -- moment sums of a caller-owned population field without any allocation.
//
// Some callers cannot let a library allocate device memory: code that runs while a
// memory pool owns every byte of the device, real-time loops that forbid allocation after
// start-up, or code about to be captured into a CUDA graph, where cudaMalloc is not
// allowed.  This entry point therefore needs no context and allocates nothing: the
// caller passes the populations, the flags and the output, all in device memory, and
// the per-block partial sums go to a fixed scratch array compiled into this library.
//
// The scratch is a file-scope __device__ array of kNoAllocMaxBlocks slots (4 doubles
// each, 256 KiB in total).  Every GPU that loads the library holds it until the process
// exits.  Host code cannot use the array's name as a device address; the address is
// looked up once per device (cudaGetSymbolAddress, with that device current) by the first
// call on that device, which should therefore happen before any stream capture.  The
// address is kept per device ordinal until the process exits; a cudaDeviceReset unloads the
// module, so after one the kept address is stale and this entry point must not be called
// on that device again.  All calls share the array: a call only reads slots that it wrote
// itself earlier in the same call, so nothing has to start at zero, but two calls that
// overlap on the GPU (on different streams without ordering) race on it.
#include <mutex>

#include "batch.h"
#include "fixed_sum.cuh"

namespace lbm {
namespace {

constexpr int kNoAllocMaxBlocks = 8192;      // scratch slots: 8192 * 4 doubles = 256 KiB
constexpr int kNoAllocThreads = 256;
constexpr long long kNoAllocMaxCells = (long long)kNoAllocMaxBlocks * 32768;

static __device__ __align__(256) double g_noalloc_partials[kNoAllocMaxBlocks * 4];

// Blocks of a call: 8 for each multiprocessor, which holds two at a time (128 registers a thread),
// each over one contiguous range of whole rounds of its threads; small fields take a round a
// block.  Fixed by the cell count alone, so that the order of the sums is.
constexpr long long kNoAllocBlocks = 152 * 8;
__host__ __device__ inline long long noalloc_cells_per_block(long long n)
{
    return ((n + kNoAllocBlocks - 1) / kNoAllocBlocks + kNoAllocThreads - 1) / kNoAllocThreads * kNoAllocThreads;
}

// Fixed-point sums.  Values whose exponent field is at most E are integers in units of
// 2^(E - 1080): 1.52-bit mantissas at bit 57 and below, so that 19 of them fit 63 bits, and those
// with exponent fields from E - kFixedSpan on (5: equilibrium populations span 4) lose nothing.  A cell
// is summed in integers only if all of its values are such, so that its sums are exact where an FP64
// sum would round; the unit is kept from cell to cell while they are.
constexpr int kFixedTop = 57, kFixedSpan = kFixedTop - 52;

// Sums of m cells held in units of exponent field E, as FP64: .v[0] = sum rho - m rho0,
// .v[1..3] = sum j.  Out of line: rare in a warp's loop, once at the end of a block.
struct Sums4 {
    double v[4];
};
__device__ __noinline__ Sums4 to_sums(FixedSum s0, FixedSum s1, FixedSum s2, FixedSum s3, int E, unsigned m,
                                      double rho0)
{
    Sums4 a = {};
    if (m == 0) return a;
    const double unit = __longlong_as_double((long long)(E - kFixedTop) << 52);
    auto whole = [](const FixedSum &s) { return ((__int128)s.hi << 32) + (__int128)s.lo; };
    const double r = rho0 / unit;  // rho0 in units: its whole part is taken off exactly
    if (r < 4.6e18) {
        const long long w = (long long)r;
        a.v[0] = (to_double(whole(s0) - (__int128)w * m) - (r - (double)w) * m) * unit;
    } else {
        a.v[0] = to_double(whole(s0)) * unit - rho0 * m;
    }
    a.v[1] = to_double(whole(s1)) * unit;
    a.v[2] = to_double(whole(s2)) * unit;
    a.v[3] = to_double(whole(s3)) * unit;
    return a;
}

// Block b sums its range of the fluid cells; partial -> partials[b].  The sums are integer sums
// because FP64 arithmetic is slow on GB300 (a warp instruction per 19 cycles a multiprocessor):
// the 49 FP64 additions of a cell would take four times as long as its loads.  The 360 integer
// instructions they become, by 16 warps a multiprocessor (a cell's 19 values are held until
// their exponents are known), leave it at 1.7 times the sectors it reads: 160^3 cells, 43 % of
// them solid at random, 1044 us with FP64 sums in 125 blocks of fixed size -> 155 us (164 with a
// cell's flag loaded before its values and not a round ahead), and 250 when the largest
// population crosses a power of two from cell to cell (rho0 = 0.75, 1.5, 3: lanes change their
// unit).  Cells that are not exact in integers (values of very different
// sizes, infinities, NaN, a largest value below 2^-959) are summed in FP64: 770 us for a field
// with such cells among the others of every warp.
__global__ void __launch_bounds__(kNoAllocThreads, 2) noalloc_partials_kernel(const double *__restrict__ f,
                                                                          const uint8_t *__restrict__ solid,
                                                                          long long n, double rho0,
                                                                          double *__restrict__ partials)
{
    __shared__ double sm[kNoAllocThreads / 32][4];
    __shared__ FixedSum fs[kNoAllocThreads / 32][4];
    __shared__ unsigned cnt[kNoAllocThreads / 32];
    __shared__ int exps[kNoAllocThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long per = noalloc_cells_per_block(n);
    const long long c0 = (long long)blockIdx.x * per, c1 = c0 + per < n ? c0 + per : n;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    FixedSum s[4] = {};
    unsigned m = 0;
    int Ecur = 0;  // exponent field of s (0: none yet)
    auto fluid = [&](long long c) { return c < c1 && !(solid && solid[c]); };
    bool next = fluid(c0 + warp * 32 + lane);
    for (long long cw = c0 + warp * 32; cw < c1; cw += kNoAllocThreads) {
        const long long c = cw + lane;
        const bool live = next;
        unsigned long long v[Q];
#pragma unroll
        for (int k = 0; k < Q; ++k)
            v[k] = live ? __ldg(reinterpret_cast<const unsigned long long *>(f) + ((long long)k * n + c)) : 0ull;
        next = fluid(c + kNoAllocThreads);  // before the loads are waited for
        unsigned top = 0u, low = 0xffffffffu;
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const unsigned x = (unsigned)(v[k] >> 32) & 0x7ff00000u;
            top = max(top, x);
            low = min(low, x);
        }
        if (live && low == 0u) {  // zeros are exact in any unit
            low = 0xffffffffu;
#pragma unroll
            for (int k = 0; k < Q; ++k)
                if (v[k] << 1) low = min(low, (unsigned)(v[k] >> 32) & 0x7ff00000u);
        }
        const int E = (int)(top >> 20), Elow = (int)(low >> 20);
        bool exact = E >= 64 && E <= Ecur && Elow >= Ecur - kFixedSpan;
        if (!exact && E >= 64 && E < 0x7ff && Elow >= E - kFixedSpan) {
            const Sums4 w = to_sums(s[0], s[1], s[2], s[3], Ecur, m, rho0);
            for (int d = 0; d < 4; ++d) a[d] += w.v[d];
            for (int d = 0; d < 4; ++d) s[d] = FixedSum{0, 0ull};
            m = 0;
            Ecur = E;
            exact = true;
        }
        if (exact) {
            long long x[4] = {0, 0, 0, 0};
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                const unsigned hi = (unsigned)(v[k] >> 32), lo = (unsigned)v[k];
                const unsigned sh = (unsigned)(Ecur + 62 - kFixedTop) - ((hi >> 20) & 0x7ffu);
                const unsigned mh = (__funnelshift_l(lo, hi, 10) & 0x3fffffffu) | 0x40000000u;
                unsigned long long t = (unsigned long long)mh << 32 | (unsigned long long)(lo << 10);
                asm("shr.u64 %0, %1, %2;" : "=l"(t) : "l"(t), "r"(sh));  // (a zero: sh > 63, t = 0)
                const long long sg = (long long)v[k] >> 63;
                const long long q = ((long long)t ^ sg) - sg;
                x[0] += q;
                if (ex(k)) x[1] += ex(k) > 0 ? q : -q;
                if (ey(k)) x[2] += ey(k) > 0 ? q : -q;
                if (ez(k)) x[3] += ez(k) > 0 ? q : -q;
            }
            for (int d = 0; d < 4; ++d) s[d].add(x[d]);
            ++m;
        } else if (live) {
            double x[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                const double g = __longlong_as_double((long long)v[k]);
                x[0] += g;
                if (ex(k)) x[1] += ex(k) > 0 ? g : -g;
                if (ey(k)) x[2] += ey(k) > 0 ? g : -g;
                if (ez(k)) x[3] += ez(k) > 0 ? g : -g;
            }
            a[0] += x[0] - rho0;
            for (int d = 1; d < 4; ++d) a[d] += x[d];
        }
    }
    // the warp's sums, then the block's: in integers where they have one unit, as they have in
    // a flow, whose largest population (at rest, about 1/3 rho0) keeps its exponent
    const int Etop = (int)__reduce_max_sync(0xffffffffu, (unsigned)Ecur);
    if (!__all_sync(0xffffffffu, m == 0 || Ecur == Etop)) {
        const Sums4 w = to_sums(s[0], s[1], s[2], s[3], Ecur, m, rho0);
        for (int d = 0; d < 4; ++d) {
            a[d] += w.v[d];
            s[d] = FixedSum{0, 0ull};
        }
        m = 0;
    }
    Ecur = Etop;
    for (int o = 16; o > 0; o >>= 1) {
        m += __shfl_xor_sync(0xffffffffu, m, o);
        for (int d = 0; d < 4; ++d) {
            s[d].hi += __shfl_xor_sync(0xffffffffu, s[d].hi, o);
            s[d].lo += __shfl_xor_sync(0xffffffffu, s[d].lo, o);
        }
    }
    bool any = false;
    for (int d = 0; d < 4; ++d) any |= a[d] != 0.0;  // (NaN too)
    if (__any_sync(0xffffffffu, any))
        for (int d = 0; d < 4; ++d)
            for (int o = 16; o > 0; o >>= 1) a[d] += __shfl_xor_sync(0xffffffffu, a[d], o);
    if (lane == 0) {
        for (int d = 0; d < 4; ++d) {
            sm[warp][d] = a[d];
            fs[warp][d] = s[d];
        }
        cnt[warp] = m;
        exps[warp] = Ecur;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double b[4] = {0.0, 0.0, 0.0, 0.0};
        FixedSum t[4] = {};
        unsigned mt = 0;
        int Et = 0;
        for (int w = 0; w < kNoAllocThreads / 32; ++w) {
            if (cnt[w] > 0 && exps[w] != Et) {
                const Sums4 v = to_sums(t[0], t[1], t[2], t[3], Et, mt, rho0);
                for (int d = 0; d < 4; ++d) b[d] += v.v[d];
                for (int d = 0; d < 4; ++d) t[d] = FixedSum{0, 0ull};
                mt = 0;
                Et = exps[w];
            }
            for (int d = 0; d < 4; ++d) {
                t[d].hi += fs[w][d].hi;
                t[d].lo += fs[w][d].lo;
                b[d] += sm[w][d];
            }
            mt += cnt[w];
        }
        const Sums4 v = to_sums(t[0], t[1], t[2], t[3], Et, mt, rho0);
        for (int d = 0; d < 4; ++d) b[d] += v.v[d];
        partials[(long long)blockIdx.x * 4] = b[0];
        for (int d = 1; d < 4; ++d) partials[(long long)blockIdx.x * 4 + d] = b[d] / rho0;
    }
}

// One block: out[d] = sum over blocks of partials[b][d], in a fixed order.
__global__ void __launch_bounds__(kNoAllocThreads) noalloc_final_kernel(const double *__restrict__ partials,
                                                                       int nblocks, double *__restrict__ out)
{
    __shared__ double sm[kNoAllocThreads][4];
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nblocks; b += kNoAllocThreads)
        for (int d = 0; d < 4; ++d) a[d] += partials[(long long)b * 4 + d];
    for (int d = 0; d < 4; ++d) sm[threadIdx.x][d] = a[d];
    __syncthreads();
    for (int w = kNoAllocThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int d = 0; d < 4; ++d) sm[threadIdx.x][d] += sm[threadIdx.x + w][d];
        __syncthreads();
    }
    if (threadIdx.x < 4) out[threadIdx.x] = sm[0][threadIdx.x];
}

// Device address of the scratch array, looked up once per device.
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
double *g_noalloc_ptr[kMaxDevices] = {};

lbm_status noalloc_scratch(double **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev < 0 || dev >= kMaxDevices) return fail(LBM_ERR_ARG, "device ordinal beyond the supported range");
    std::lock_guard<std::mutex> lk(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_partials);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(no-allocation scratch)");
        g_noalloc_ptr[dev] = static_cast<double *>(p);
    }
    *out = g_noalloc_ptr[dev];
    return LBM_OK;
}

}  // namespace
}  // namespace lbm

using namespace lbm;

extern "C" lbm_status lbm_moment_sums_f64_noalloc(const double *f_dev, const uint8_t *solid_dev, int64_t n_cells,
                                                  double rho0, double *sums_dev, void *cuda_stream)
{
    if (!f_dev || !sums_dev) return fail(LBM_ERR_ARG, "f_dev and sums_dev must be device pointers");
    if (n_cells < 1) return fail(LBM_ERR_ARG, "n_cells must be >= 1");
    if (n_cells > kNoAllocMaxCells)
        return fail(LBM_ERR_ARG, "n_cells exceeds the no-allocation limit of " + std::to_string(kNoAllocMaxCells) +
                                     " cells (the fixed scratch holds " + std::to_string(kNoAllocMaxBlocks) +
                                     " block sums)");
    if (!(rho0 > 0.0)) return fail(LBM_ERR_ARG, "rho0 must be > 0");
    if ((reinterpret_cast<uintptr_t>(f_dev) | reinterpret_cast<uintptr_t>(sums_dev)) & 7u)
        return fail(LBM_ERR_ARG, "f_dev and sums_dev must be 8-byte aligned");
    double *scratch = nullptr;
    lbm_status st = noalloc_scratch(&scratch);
    if (st != LBM_OK) return st;
    const cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const long long per = noalloc_cells_per_block(n_cells);
    const int nblocks = (int)((n_cells + per - 1) / per);
    noalloc_partials_kernel<<<nblocks, kNoAllocThreads, 0, s>>>(f_dev, solid_dev, (long long)n_cells, rho0, scratch);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "no-allocation moment sums (partials)");
    noalloc_final_kernel<<<1, kNoAllocThreads, 0, s>>>(scratch, nblocks, sums_dev);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "no-allocation moment sums (final)");
    return LBM_OK;
}
