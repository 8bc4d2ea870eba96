// FP64 step of the 2D lattice (upwind drag): a tile of cells with all its velocities in shared memory.
//
// The FP64 pipe (two operations per clock and SM on this part) bounds the step, and one thread per
// cell leaves it idle most of the time: 128^2 cells are four warps per SM with serial columns of 33^2
// velocities.  Here a block takes TC neighbouring cells of a grid row, stages their streamed values
// in shared memory (the streaming is the copies' source address) and gives every cell and vx a thread
// that sweeps the vy rows, first for the drag, then for the diffusion.
//
// FP64 operations per phase cell: 14, where the row sweep of the other types would take 20 or more
// (its minima and maxima are comparisons on the same pipe):
//  * the parts of c a are taken by the sign bit.  c a falls along an axis, so one term of an upwind
//    flux (c a_j)^+ f_j + (c a_{j+1})^- f_{j+1} is zero except at the face where its sign changes:
//    one product, and the second term in a branch that few faces take;
//  * the diffusion is one fma with the sum of the differences of f** (rounded as differences, not as
//    four scaled fluxes).
//
// Measured (128^2 x 33^2): 0.87 ms per step, the FP64 pipe 75 % active.  A thread per cell (step2d.cu's
// plain kernel) issues fewer instructions beside the FP64 ones and is faster where its 128-cell blocks
// fill the SMs evenly (256 x 150 x 33^2: 1.62 against 1.99 ms): step2d_f64_tiles chooses.
#include <algorithm>

#include "lat_internal.h"
#include "per_device.h"
#include "step2d_dev.h"

namespace lat {
namespace {

using namespace k2d;

template <int NV>
struct Tile64 {
    static constexpr int J = (NV - 1) / 2;
    static constexpr int TC = NV >= 33 ? 8 : (NV >= 17 ? 16 : 32);  // cells per tile
    static constexpr int kThreads = (NV * TC + 31) / 32 * 32;
    static constexpr int kRow = NV * TC;                            // elements of a velocity row
    static constexpr size_t kSmem = sizeof(double) * (2 * (size_t)NV * kRow + kRow);
};

__device__ __forceinline__ bool negative(double v) { return __double2hiint(v) < 0; }

// A c a that is not a number (of such a velocity) counts as zero, as in the other kernels' maxima and
// minima.
__device__ __forceinline__ double number(double v) {
    return ((unsigned)__double2hiint(v) & 0x7fffffffu) <= 0x7ff00000u ? v : 0.0;
}

// Upwind flux between cells l and r of one axis (c_l >= c_r).
__device__ __forceinline__ double upwind64(double cl, double fl, double cr, double fr) {
    const bool p = !negative(cl);
    double F = __dmul_rn(p ? cl : cr, p ? fl : fr);
    if (p && negative(cr)) F = __fma_rn(cl, fl, __dmul_rn(cr, fr));
    return F;
}

__device__ __forceinline__ void cp_async8(double* dst, const double* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src)
                 : "memory");
}

// f* of the tile's cell c, column jx, all rows, into plane S.
template <int NV>
__device__ __forceinline__ void load_column(const double* fin, double* S, int nx, int ny, int y,
                                            int x, int jx, int c) {
    using L = Tile64<NV>;
    if (x >= nx) return;  // beyond a ragged edge
    const size_t ncell = (size_t)nx * ny;
    const double* src = fin + (size_t)jx * ncell + wrap(x - (jx - L::J), nx);
    double* d = S + jx * L::TC + c;
    int yr = wrap(y + L::J, ny);  // the source row of jy = 0
#pragma unroll 4
    for (int jy = 0; jy < NV; ++jy) {
        cp_async8(d, src + (size_t)yr * nx);
        src += (size_t)NV * ncell;
        d += L::kRow;
        yr = yr == 0 ? ny - 1 : yr - 1;
    }
}

template <int NV>
__global__ void __launch_bounds__(Tile64<NV>::kThreads) k_step2d_tile64(const Step2DArgs a, int kstep) {
    using L = Tile64<NV>;
    using O = Ops<double>;
    constexpr int J = L::J, TC = L::TC, R = L::kRow;
    extern __shared__ __align__(16) double sm64[];
    double* S = sm64;            // f* [jy][jx][cell]
    double* B = S + NV * R;      // f**
    double* cy = B + NV * R;     // c a_y [jy][cell]
    const int nx = a.nx, ny = a.ny;
    const size_t ncell = (size_t)nx * ny;
    const bool par = ((a.st->step + kstep) & 1) != 0;
    const double* fin = static_cast<const double*>(par ? a.f[1] : a.f[0]);
    double* fout = static_cast<double*>(par ? a.f[0] : a.f[1]);
    const int c = threadIdx.x % TC, jx = threadIdx.x / TC;
    const bool active = jx < NV;
    const int ntx = (nx + TC - 1) / TC;
    const long long ntiles = (long long)ntx * ny;
    long long t = blockIdx.x;
    if (t < ntiles && active) {
        const int y = (int)(t / ntx);
        load_column<NV>(fin, S, nx, ny, y, (int)(t - (long long)y * ntx) * TC + c, jx, c);
    }
    for (; t < ntiles; t += gridDim.x) {
        const int y = (int)(t / ntx);
        const int x = (int)(t - (long long)y * ntx) * TC + c;
        const bool in = active && x < nx;
        double wx, wy;
        load_w<double>(a, x < nx ? x : 0, y, wx, wy);
        if (jx == 0) cfl_check<double, NV>(a, a.g, wx, wy, in);
        const double c0 = number(cacc<double>(a.g, wx, jx - J)),
                     cl = number(cacc<double>(a.g, wx, jx - 1 - J)),
                     cr = number(cacc<double>(a.g, wx, jx + 1 - J));
        if (active) cy[jx * TC + c] = number(cacc<double>(a.g, wy, jx - J));
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();  // f* and c a_y are there; every warp is done with the last tile's f**
        if (in) {
            const double* s = S + jx * TC + c;
            const double* q = cy + c;
            double* b = B + jx * TC + c;
            double f0 = *s, qc = *q, Gp = 0.0;
#pragma unroll 3
            for (int jy = 0; jy < NV; ++jy) {
                const double Fr = jx < NV - 1 ? upwind64(c0, f0, cr, s[TC]) : 0.0;
                const double Fl = jx > 0 ? upwind64(cl, s[-TC], c0, f0) : 0.0;
                double G = 0.0, fn = 0.0, qn = 0.0;
                if (jy < NV - 1) {
                    fn = s[R];
                    qn = q[TC];
                    G = upwind64(qc, f0, qn, fn);
                }
                *b = O::sub(O::sub(f0, O::sub(Fr, Fl)), O::sub(G, Gp));
                Gp = G;
                f0 = fn;
                qc = qn;
                s += R;
                q += TC;
                b += R;
            }
        }
        __syncthreads();  // f** is there and f* is free: the next tile's comes in meanwhile
        const long long tn = t + gridDim.x;
        if (tn < ntiles && active) {
            const int yn = (int)(tn / ntx);
            load_column<NV>(fin, S, nx, ny, yn, (int)(tn - (long long)yn * ntx) * TC + c, jx, c);
        }
        if (in) {
            const double* b = B + jx * TC + c;
            double* out = fout + (size_t)jx * ncell + (size_t)y * nx + x;
            double b0 = *b, Ep = 0.0;
#pragma unroll 3
            for (int jy = 0; jy < NV; ++jy) {
                const double Er = jx < NV - 1 ? O::sub(b[TC], b0) : 0.0;
                const double El = jx > 0 ? O::sub(b0, b[-TC]) : 0.0;
                const double bn = jy < NV - 1 ? b[R] : b0;
                const double E = O::sub(bn, b0);
                *out = O::fma(a.r, O::add(O::sub(Er, El), O::sub(E, Ep)), b0);
                Ep = E;
                b0 = bn;
                b += R;
                out += NV * ncell;
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

template <int NV>
cudaError_t launch_t(int sm_count, const Step2DArgs& a, int k, cudaStream_t s) {
    using L = Tile64<NV>;
    static PerDevice resident;
    int per_sm = 0;
    const cudaError_t e =
        resident_blocks(resident, k_step2d_tile64<NV>, L::kThreads, L::kSmem, &per_sm);
    if (e != cudaSuccess) return e;
    const long long ntiles = (long long)((a.nx + L::TC - 1) / L::TC) * a.ny;
    const int grid = (int)std::min<long long>(ntiles, (long long)per_sm * sm_count);
    k_step2d_tile64<NV><<<grid, L::kThreads, L::kSmem, s>>>(a, k);
    return cudaGetLastError();
}

}  // namespace

// Time in units of an SM that gets one 128-cell block of the plain kernel, which is what this one takes
// for 128 cells per SM; the plain kernel takes `plain` of it.  Blocks land on the SMs in pairs: 300 to
// 304 of them (152 SMs) take two units, 320 take four.  Measured per step (us), tiles against plain:
// N_v = 33 128 x 128 874 and 917, 160 x 160 1360 and 3198, 256 x 150 1987 and 1615; N_v = 17 160 x 160
// 330 and 860, 256 x 150 509 and 438, 512 x 256 1621 and 1720; N_v = 9 160 x 160 99 and 185, 512 x 300
// 503 and 544, 512 x 512 856 and 843.
bool step2d_f64_tiles(int nv, int nx, int ny, int sm_count) {
    const double plain = nv >= 33 ? 0.81 : nv >= 19 ? 0.915 : nv >= 17 ? 0.88 : nv >= 13 ? 0.97
                       : nv >= 9 ? 1.1 : nv >= 5 ? 0.92 : nv >= 3 ? 1.0 : 0.7;
    const int TC = nv >= 33 ? 8 : nv >= 17 ? 16 : 32;  // Tile64<NV>::TC
    const long long blocks = (long long)((nx + TW - 1) / TW) * ny, pair = 2ll * sm_count;
    const double units = blocks <= sm_count ? 1.13 : 2.0 * ((blocks + pair - 1) / pair);
    const double cells = (double)((nx + TC - 1) / TC * TC) * ny / (128.0 * sm_count);
    return cells < plain * units;
}

cudaError_t launch_step2d_f64(int nv, int sm_count, const k2d::Step2DArgs& a, int k, cudaStream_t s) {
    switch (nv) {
#define X(n) \
    case n: return launch_t<n>(sm_count, a, k, s);
        X(1) X(3) X(5) X(9) X(13) X(17) X(19) X(21) X(33)
#undef X
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace lat
