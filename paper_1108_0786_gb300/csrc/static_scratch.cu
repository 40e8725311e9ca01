// static_scratch.cu -- momentum-exchange force and torque per body for
// callers that cannot allocate device memory.
//
// This is a variant of the force kernel of kernels.cu.  The regular step
// keeps its link lists and per-block partial sums in memory the handle
// allocates; here the caller passes only its inputs (post-collision
// populations, the obstacle-cell field, body states) and its output, and
// the per-block partial sums go to a file-scope device array of fixed size.
// No cudaMalloc, cudaFree or allocating library routine is called.
//
// The array is shared by every call on a device and keeps the contents of
// the last call: each call writes every record it later reads, so nothing
// has to start at zero, but two calls that overlap on the GPU (for example
// on two streams) race on the array and give wrong results.
#include <mutex>

#include <cuda.h>

#include "../../include/lbm.h"
#include "lbm_internal.cuh"

namespace lbm {
namespace {

constexpr int NA_THREADS = 256;
constexpr int NA_MAX_DEVICES = 64;

// per-block partial sums (6 doubles each), LBM_STATIC_SCRATCH_RECORDS records
static __device__ __align__(256) double g_force_partials[LBM_STATIC_SCRATCH_RECORDS * 6];

std::mutex g_setup_mutex;
struct ScratchAddr {
    unsigned long long ctx_id;  // context the address belongs to (0: none yet)
    double *addr;
};
ScratchAddr g_partials_addr[NA_MAX_DEVICES] = {};

// Identifier of the current context, from the driver through the runtime's
// entry-point lookup (no link against the driver library); 0 if the driver
// does not offer it.
unsigned long long current_context_id() {
    typedef CUresult (*GetCurrent)(CUcontext *);
    typedef CUresult (*GetId)(CUcontext, unsigned long long *);
    static GetCurrent get_current = nullptr;
    static GetId get_id = nullptr;
    static bool looked_up = false;
    if (!looked_up) {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<GetCurrent>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<GetId>(f);
        looked_up = true;
    }
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    if (!get_current || !get_id || get_current(&ctx) != CUDA_SUCCESS || !ctx || get_id(ctx, &id) != CUDA_SUCCESS)
        return 0;
    return id;
}

// Device address of the array in the current context.  Host code cannot use
// the symbol itself as a device pointer; the address is looked up once per
// device with that device current, and again whenever the device's context
// has changed (after cudaDeviceReset the module is loaded anew, possibly at
// another address).  Without a context identifier (no context current yet,
// or a driver without the query) it is looked up on every call.
cudaError_t partials_address(double **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= NA_MAX_DEVICES) return cudaErrorInvalidDevice;
    const unsigned long long id = current_context_id();
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    ScratchAddr &slot = g_partials_addr[dev];
    if (id == 0 || slot.ctx_id != id || !slot.addr) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_force_partials);
        if (e != cudaSuccess) return e;
        slot.addr = static_cast<double *>(p);
        slot.ctx_id = id;
    }
    *out = slot.addr;
    return cudaSuccess;
}

// Cells the scan covers along one axis: the cube's side, or the whole axis
// when a periodic axis is shorter than the side (a wrapped cube would visit
// its cells twice and add their links twice).
inline int scan_extent(int side, int n, int periodic) { return periodic && n < side ? n : side; }

// minimum image of a distance i / 2 - f with i an integer number of half cells,
// f in [0, 1) and k = ceil(2 f): twice the integer part, so that i / 2 - f lies in
// [-n / 2, n / 2).  A distance within n + 1 of zero needs one period, on an axis of
// one cell up to two.
__device__ __forceinline__ int near_half(int i2, int n, int periodic, int k) {
    if (!periodic) return i2;
    if (i2 - n >= k) return i2 - 2 * n;
    if (i2 + n < k) i2 += 2 * n;
    return i2 + n < k ? i2 + 2 * n : i2;
}

// exponent bits all set: an infinity or NaN (integer operations, not the FP64 pipe)
__device__ __forceinline__ bool non_finite(double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; }

// Block (k, b): cells k*256 .. of the box of extents (sx, sy, sz) that
// starts at floor(X_b) - hw (the cube of side 2 hw + 1 around floor(X_b),
// cut to one period on short periodic axes).  A thread a cell finds the links
// (x_f, a) whose end x_f + e_a is a cell of body b and the block lists them in
// (cell, a) order; then a thread a link forms its term (Eq. hydroF, torque about
// the body centre at the link midpoint), so that no lane waits for another cell's
// links: an FP64 warp instruction costs ~64 issue cycles whatever its lanes do.
// The block writes its fixed-order sum to record b * blocks + k.  (48^3 cells, three bodies of
// radius 4, both kernels: 64.9 us with a thread walking its cell's links and a
// serial sum, 18.4 us so.)
__global__ void __launch_bounds__(NA_THREADS)
static_partials_kernel(const double *__restrict__ pop, const uint8_t *__restrict__ flags, const double *bodies, Domain d,
                       int hw, int sx, int sy, int sz, int blocks, double *partials) {
    const int b = blockIdx.y, k = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ int s_cell[NA_THREADS], s_at[NA_THREADS][3];
    __shared__ unsigned short s_link[NA_THREADS * (Q - 1)];
    __shared__ int s_count[NA_THREADS / 32];
    const double *sb = bodies + 13 * b;
    const int n3[3] = {d.nx, d.ny, d.nz}, per[3] = {d.px, d.py, d.pz};
    // the centre wrapped into the domain: its cell and the position within it
    int corner[3], ci[3];
    double cf[3];
    int cf2[3];                 // ceil(2 cf)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double X = sb[a], fx = floor(X);
        corner[a] = (int)fx - hw;
        cf[a] = X - fx;
        cf2[a] = (cf[a] > 0.0) + (cf[a] > 0.5);
        ci[a] = (int)fx;
        if (per[a]) {
            ci[a] %= n3[a];
            if (ci[a] < 0) ci[a] += n3[a];
        }
    }
    unsigned mask = 0;
    {
        const int l = k * NA_THREADS + (int)threadIdx.x;
        int x = 0, y = 0, z = 0, c = 0;
        bool ok = l < sx * sy * sz;
        if (ok) {
            const int row = l / sx, pl = row / sy;
            x = corner[0] + (l - row * sx);
            y = corner[1] + (row - pl * sy);
            z = corner[2] + pl;
            if (d.px) x = ((x % d.nx) + d.nx) % d.nx; else ok = ok && x >= 0 && x < d.nx;
            if (d.py) y = ((y % d.ny) + d.ny) % d.ny; else ok = ok && y >= 0 && y < d.ny;
            if (d.pz) z = ((z % d.nz) + d.nz) % d.nz; else ok = ok && z >= 0 && z < d.nz;
        }
        if (ok) {
            c = (z * d.ny + y) * d.nx + x;
            if (flags[c] == 0) {
#pragma unroll
                for (int a = 1; a < Q; ++a) {
                    const int nx_ = x + ex(a), ny_ = y + ey(a), nz_ = z + ez(a);
                    const bool beyond = (!d.px && (nx_ < 0 || nx_ >= d.nx)) || (!d.py && (ny_ < 0 || ny_ >= d.ny)) ||
                                        (!d.pz && (nz_ < 0 || nz_ >= d.nz));
                    const int at = (wrap_axis(nz_, d.nz) * d.ny + wrap_axis(ny_, d.ny)) * d.nx + wrap_axis(nx_, d.nx);
                    if (flags[at] == b + 1 && !beyond) mask |= 1u << a;
                }
            }
        }
        s_cell[threadIdx.x] = c;
        s_at[threadIdx.x][0] = x;
        s_at[threadIdx.x][1] = y;
        s_at[threadIdx.x][2] = z;
    }
    // the block's links in (cell, a) order
    const int cnt = __popc(mask);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) s_count[warp] = incl;
    __syncthreads();
    int pos = incl - cnt, total = 0;
#pragma unroll
    for (int w = 0; w < NA_THREADS / 32; ++w) {
        if (w < warp) pos += s_count[w];
        total += s_count[w];
    }
    while (mask) {
        const int a = __ffs(mask) - 1;
        mask &= mask - 1;
        s_link[pos++] = (unsigned short)(threadIdx.x << 5 | a);
    }
    __syncthreads();
    double acc[6] = {0, 0, 0, 0, 0, 0};
    if ((int)threadIdx.x < total) {
        const double V[3] = {sb[7], sb[8], sb[9]}, W[3] = {sb[10], sb[11], sb[12]};
        bool odd = false;
        for (int i = 0; i < 3; ++i) odd = odd || non_finite(V[i]) || non_finite(W[i]) || non_finite(cf[i]);
        for (int j = threadIdx.x; j < total; j += NA_THREADS) {
            const int t = s_link[j] >> 5, a = s_link[j] & 31;
            const int c = s_cell[t];
            double p[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) p[q] = __ldg(pop + q * d.C + c);
            const double ga = __ldg(pop + a * d.C + c);
            const int e[3] = {ex(a), ey(a), ez(a)};
            double rho = p[0];
#pragma unroll
            for (int q = 1; q < Q; ++q) rho += p[q];
            double oe[3], om[3];            // link end and midpoint from the centre
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int i2 = 2 * (s_at[t][i] - ci[i]);
                oe[i] = 0.5 * (double)near_half(i2 + 2 * e[i], n3[i], per[i], cf2[i]) - cf[i];
                om[i] = 0.5 * (double)near_half(i2 + e[i], n3[i], per[i], cf2[i]) - cf[i];
            }
            const double u0 = V[0] + (W[1] * oe[2] - W[2] * oe[1]), u1 = V[1] + (W[2] * oe[0] - W[0] * oe[2]),
                         u2 = V[2] + (W[0] * oe[1] - W[1] * oe[0]);
            auto by = [](int s, double v) { return s > 0 ? v : (s < 0 ? -v : 0.0); };
            const double eu = -(by(e[0], u0) + by(e[1], u1) + by(e[2], u2));
            const double w6 = a < 7 ? 6.0 * wgt(1) : 6.0 * wgt(7);
            const double mag = 2.0 * ga + w6 * rho * eu;
            if (odd || non_finite(mag)) {
                // Eq. hydroF with its zero components multiplied out: 0 * inf is no 0
                const double m = 2.0 * ga - w6 * rho * (e[0] * u0 + e[1] * u1 + e[2] * u2);
                const double fl[3] = {e[0] * m, e[1] * m, e[2] * m};
                acc[0] += fl[0];
                acc[1] += fl[1];
                acc[2] += fl[2];
                acc[3] += om[1] * fl[2] - om[2] * fl[1];
                acc[4] += om[2] * fl[0] - om[0] * fl[2];
                acc[5] += om[0] * fl[1] - om[1] * fl[0];
                continue;
            }
            acc[0] += by(e[0], mag);
            acc[1] += by(e[1], mag);
            acc[2] += by(e[2], mag);
            acc[3] += (by(e[2], om[1]) - by(e[1], om[2])) * mag;
            acc[4] += (by(e[0], om[2]) - by(e[2], om[0])) * mag;
            acc[5] += (by(e[1], om[0]) - by(e[0], om[1])) * mag;
        }
    }
    __shared__ double part[NA_THREADS / 32][6];
    const int warps = min((total + 31) / 32, NA_THREADS / 32);      // those with links
    if (warp < warps) {
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            double v = acc[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0) part[warp][i] = v;
        }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        double v = 0.0;
        for (int w = 0; w < warps; ++w) v += part[w][threadIdx.x];
        partials[((long long)b * blocks + k) * 6 + threadIdx.x] = v;
    }
}

// block b adds its body's records: lane 6 j + i takes component i of the records
// j, j + 5, ..., then the five parts in order
constexpr int SUM_PARTS = 5;
__global__ void __launch_bounds__(32) static_sum_kernel(const double *partials, int blocks, double *out) {
    const int b = blockIdx.x, lane = threadIdx.x, i = lane % 6, j = lane / 6;
    double v = 0.0;
    if (j < SUM_PARTS)
        for (int k = j; k < blocks; k += SUM_PARTS) v += partials[((long long)b * blocks + k) * 6 + i];
    double sum = 0.0;
#pragma unroll
    for (int part = 0; part < SUM_PARTS; ++part) sum += __shfl_sync(0xffffffffu, v, 6 * part + i);
    if (lane < 6) out[b * 6 + lane] = sum;
}

}  // namespace
}  // namespace lbm

#pragma GCC visibility push(default)
extern "C" int lbm_momentum_exchange_static(const double *pop, const unsigned char *flags, const double *bodies,
                                            int nb, int nx, int ny, int nz, int bc, int half_width, double *out,
                                            void *stream) {
    if (!pop || !flags || !bodies || !out) return LBM_E_ARG;
    if (nb < 1 || nb > LBM_MAX_BODIES || nx < 1 || ny < 1 || nz < 1 || bc < 0 || bc > 7) return LBM_E_ARG;
    const long long C = (long long)nx * ny * nz;
    if (C > (1LL << 31) - 1) return LBM_E_ARG;
    if (half_width < 1 || half_width > LBM_STATIC_SCRATCH_MAX_HALF_WIDTH) return LBM_E_ARG;
    const int side = 2 * half_width + 1;
    const int sx = lbm::scan_extent(side, nx, bc & 1), sy = lbm::scan_extent(side, ny, bc & 2),
              sz = lbm::scan_extent(side, nz, bc & 4);
    const int blocks = (int)(((long long)sx * sy * sz + lbm::NA_THREADS - 1) / lbm::NA_THREADS);
    if ((long long)blocks * nb > LBM_STATIC_SCRATCH_RECORDS) return LBM_E_ARG;
    double *partials = nullptr;
    if (lbm::partials_address(&partials) != cudaSuccess) return LBM_E_CUDA;
    const lbm::Domain d{nx, ny, nz, (bc & 1) ? 1 : 0, (bc & 2) ? 1 : 0, (bc & 4) ? 1 : 0, C,
                        1.0 / nx, 1.0 / ny, 1.0 / nz};
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    lbm::static_partials_kernel<<<dim3(blocks, nb), lbm::NA_THREADS, 0, s>>>(pop, flags, bodies, d, half_width,
                                                                            sx, sy, sz, blocks, partials);
    lbm::static_sum_kernel<<<nb, 32, 0, s>>>(partials, blocks, out);
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_E_CUDA;
}
#pragma GCC visibility pop
