// Observables of the phase-space density that the paper uses to benchmark the method (Sec. 3.2):
// the second moment of the coarse-grained density, Eq. (def_coarse), and the Eulerian first-order
// velocity structure function, Eq. (def_eulS1).  They start from the per-cell density rho that the
// moment kernels produce (FP64) and, for S1, from the state itself.
//
// Lattice forms: r = w dx for whole numbers w of cells, the window of cell i covering cells
// i .. i + w - 1 (periodic; w x w squares in 2D); separations s dx; velocity differences
// |j - j'| dv.  All reductions are compensated FP64 sums in a fixed order (deterministic).
#include <algorithm>

#include "lat_internal.h"
#include "lat_reduce.h"

namespace lat {
namespace {

using namespace cs;

constexpr int kObsThreads = 256;

// Fixed-order block reduction of one compensated sum per thread (result in thread 0).
__device__ __forceinline__ Comp block_reduce(Comp t) {
    __shared__ Comp wsum[kObsThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    warp_reduce(t);
    __syncthreads();  // wsum may still be read by an earlier call
    if (lane == 0) wsum[warp] = t;
    __syncthreads();
    Comp z{0, 0};
    if (threadIdx.x == 0)
        for (int w = 0; w < kObsThreads / 32; ++w) nmerge(z, wsum[w]);
    return z;
}

// Exclusive prefix sums of rho per instance, compensated (hi + lo): instance k's n + 1 sums
// start at xoff_k + k.  One block per instance; chunks of kPrefixThreads kPrefixCells cells in order.
// Window sums are then differences of prefix sums, accurate to about u of the window (u = 2^-53)
// however long the instance.
// Bound by the FP64 pipe: a thread adds kPrefixCells cells one after the other, so that the scan of the
// threads' totals (a merge costs as much as a cell's addition, five per warp scan) is shared by them.
// 1024 instances, N_x 1024 .. 8192: 226 us; a cell per thread 776 us.
constexpr int kPrefixThreads = 128, kPrefixCells = 8;

__global__ void __launch_bounds__(kPrefixThreads)
    k_prefix1d(const double* rho, const Inst1D* inst, int n_inst, double* Ph, double* Pl) {
    __shared__ Comp wtot[kPrefixThreads / 32];
    __shared__ Comp carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = blockIdx.x; k < n_inst; k += gridDim.x) {
        const Inst1D in = inst[k];
        const double* r = rho + in.xoff;
        double* ph = Ph + in.xoff + k;
        double* pl = Pl + in.xoff + k;
        if (threadIdx.x == 0) carry = Comp{0, 0};
        __syncthreads();
        for (int base = 0; base < in.nx; base += kPrefixThreads * kPrefixCells) {
            const int i0 = base + (int)threadIdx.x * kPrefixCells;
            double v[kPrefixCells];
#pragma unroll
            for (int q = 0; q < kPrefixCells; ++q) v[q] = i0 + q < in.nx ? r[i0 + q] : 0.0;
            Comp part[kPrefixCells];  // the sums before each of the thread's cells
            Comp incl{0, 0};
#pragma unroll
            for (int q = 0; q < kPrefixCells; ++q) {
                part[q] = incl;
                nadd(incl, v[q]);
            }
            for (int off = 1; off < 32; off <<= 1) {  // inclusive scan, predecessors first
                const Comp o = shfl_up(incl, off);
                if (lane >= off) {
                    Comp t = o;
                    nmerge(t, incl);
                    incl = t;
                }
            }
            Comp excl = shfl_up(incl, 1);
            if (lane == 0) excl = Comp{0, 0};
            if (lane == 31) wtot[warp] = incl;
            __syncthreads();
            Comp before = carry;
            for (int w = 0; w < warp; ++w) nmerge(before, wtot[w]);
            Comp own = before;
            nmerge(own, excl);
#pragma unroll
            for (int q = 0; q < kPrefixCells; ++q) {
                if (i0 + q >= in.nx) break;
                Comp t = own;
                nmerge(t, part[q]);
                ph[i0 + q] = t.s;
                pl[i0 + q] = t.c;
            }
            __syncthreads();
            if (threadIdx.x == kPrefixThreads - 1) {
                nmerge(before, incl);
                carry = before;
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            ph[in.nx] = carry.s;
            pl[in.nx] = carry.c;
        }
        __syncthreads();
    }
}

// <rho_r^2> per (instance, width): block per pair, threads over cells.
__global__ void __launch_bounds__(kObsThreads)
    k_coarse1d(const double* Ph, const double* Pl, const Inst1D* inst, int n_inst,
               const int* widths, int nw, double* out) {
    for (int b = blockIdx.x; b < n_inst * nw; b += gridDim.x) {
        const int k = b / nw, q = b % nw;
        const Inst1D in = inst[k];
        const double* ph = Ph + in.xoff + k;
        const double* pl = Pl + in.xoff + k;
        const int w = widths[q], n = in.nx;
        Comp t{0, 0};
        for (int i = threadIdx.x; i < n; i += kObsThreads) {
            double m;
            if (i + w <= n) {
                m = (ph[i + w] - ph[i]) + (pl[i + w] - pl[i]);
            } else {
                const int e = i + w - n;
                m = ((ph[n] - ph[i]) + ph[e]) + ((pl[n] - pl[i]) + pl[e]);
            }
            const double r = m * in.dx;
            nadd(t, r * r);
        }
        const Comp z = block_reduce(t);
        if (threadIdx.x == 0) out[b] = nval(z) / n;
    }
}

// Compensated summed-area table of rho (ny x nx): S[y (nx + 1) + x] = the sum of rho over rows
// < y and columns < x, as hi + lo.
__global__ void k_sat_rows(const double* rho, int nx, int ny, double* Sh, double* Sl) {
    const int y = blockIdx.x * blockDim.x + threadIdx.x;
    if (y > ny) return;
    double* sh = Sh + (size_t)y * (nx + 1);
    double* sl = Sl + (size_t)y * (nx + 1);
    Comp acc{0, 0};
    sh[0] = 0.0;
    sl[0] = 0.0;
    for (int x = 0; x < nx; ++x) {
        if (y > 0) nadd(acc, rho[(size_t)(y - 1) * nx + x]);
        sh[x + 1] = acc.s;
        sl[x + 1] = acc.c;
    }
}
__global__ void k_sat_cols(int nx, int ny, double* Sh, double* Sl) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x > nx) return;
    Comp acc{0, 0};
    for (int y = 1; y <= ny; ++y) {
        const size_t c = (size_t)y * (nx + 1) + x;
        nmerge(acc, Comp{Sh[c], Sl[c]});
        Sh[c] = acc.s;
        Sl[c] = acc.c;
    }
}

// sum over rows [y0, y1), columns [x0, x1), from the compensated table
__device__ __forceinline__ double rect(const double* Sh, const double* Sl, int nx1, int y0,
                                       int y1, int x0, int x1) {
    const size_t a = (size_t)y0 * nx1 + x0, b = (size_t)y0 * nx1 + x1;
    const size_t c = (size_t)y1 * nx1 + x0, d = (size_t)y1 * nx1 + x1;
    return ((Sh[d] - Sh[b]) - (Sh[c] - Sh[a])) + ((Sl[d] - Sl[b]) - (Sl[c] - Sl[a]));
}

// 2D <rho_r^2> per width: w x w windows with periodic wrap (up to four rectangles).
__global__ void __launch_bounds__(kObsThreads)
    k_coarse2d(const double* Sh, const double* Sl, int nx, int ny, double dx, const int* widths,
               int nw, double* out) {
    const int nx1 = nx + 1;
    const long long ncell = (long long)nx * ny;
    for (int q = blockIdx.x; q < nw; q += gridDim.x) {
        const int w = widths[q];
        Comp t{0, 0};
        for (long long c = threadIdx.x; c < ncell; c += kObsThreads) {
            const int y = (int)(c / nx), x = (int)(c % nx);
            const int ye = y + w, xe = x + w;
            const int ya = ye <= ny ? ye : ny, xa = xe <= nx ? xe : nx;
            double m = rect(Sh, Sl, nx1, y, ya, x, xa);
            if (ye > ny) m += rect(Sh, Sl, nx1, 0, ye - ny, x, xa);
            if (xe > nx) m += rect(Sh, Sl, nx1, y, ya, 0, xe - nx);
            if (ye > ny && xe > nx) m += rect(Sh, Sl, nx1, 0, ye - ny, 0, xe - nx);
            const double r = m * dx * dx;
            nadd(t, r * r);
        }
        const Comp z = block_reduce(t);
        if (threadIdx.x == 0) out[q] = nval(z) / (double)ncell;
    }
}

// Eq. (def_eulS1) per (instance, separation): the pair sum over velocity cells of cell i and
// cell i + s, sum_j a_j sum_j' b_j' |j - j'|, by two running sums without cancellation:
//   T_j = sum_{j' < j} b_j' (j - j'),  T_{j+1} = T_j + sum_{j' <= j} b_j'   (forward),
//   U_j = sum_{j' > j} b_j' (j' - j),  U_{j-1} = U_j + sum_{j' >= j} b_j'   (backward),
// then times dv^3; the denominator rho_i rho_{i+s}.  T = float for FP32 states (errors about
// N_v u of the positive sums), double for FP64 states.
//
// A block takes a run of columns of one instance (a slot: see s1_slot), a thread cpt cells of it, and G
// separations in one pair of sweeps: a_j is loaded for all of them, and what remains per separation
// and velocity cell is one load and three operations in either direction (1024 instances, N_v = 65,
// eight separations: 2.5 ms; a block per instance and separation 6.5 ms).  The cells' sums are FP64
// Neumaier sums per thread; the 2 G sums of a warp's lanes are folded by halving (every lane ends with
// one of them) rather than by as many butterflies, which took longer than the sweeps.  The blocks'
// sums go to part[group][slot][num, den of each][sum, compensation], folded in slot order.
constexpr int kS1Group = 8;  // separations of a pair of sweeps at most
constexpr int kS1Threads = 128;

__device__ __forceinline__ Comp shfl_xor(const Comp& a, int m) {
    return Comp{__shfl_xor_sync(0xffffffffu, a.s, m), __shfl_xor_sync(0xffffffffu, a.c, m)};
}

// First slot of instance k: its runs of `per` columns take the slots from here on, at most
// floor((xoff + N_x) / per) - floor(xoff / per) + 1 of them, so instances do not share any.
__host__ __device__ __forceinline__ long long s1_slot(const Inst1D& in, int k, int per) {
    return in.xoff / per + k;
}

template <typename T, int G>
__global__ void __launch_bounds__(kS1Threads)
    k_s1_1d(const T* f, const Inst1D* inst, int n_inst, int cpt, int nv, const double* rho,
            const int* seps, double* part) {
    constexpr int NS = 2 * G;  // sums: 2 q the numerator, 2 q + 1 the denominator
    __shared__ Comp wsum[kS1Threads / 32][NS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = kS1Threads * cpt;
    int k = 0;  // the last instance whose first slot is not beyond this one
    for (int hi = n_inst; hi - k > 1;) {
        const int mid = (k + hi) / 2;
        if (s1_slot(inst[mid], mid, per) <= (long long)blockIdx.x) k = mid;
        else hi = mid;
    }
    const Inst1D& in = inst[k];
    const int n = in.nx;
    const long long first = ((long long)blockIdx.x - s1_slot(in, k, per)) * per;
    if (first >= n) return;  // a slot without columns
    const int x0 = (int)first;
    const T* fk = f + in.off;
    seps += blockIdx.y * G;
    Comp t[NS];
#pragma unroll
    for (int q = 0; q < NS; ++q) t[q] = Comp{0, 0};
    for (int e = 0; e < cpt; ++e) {
        const int i = x0 + e * kS1Threads + threadIdx.x;
        if (i >= n) break;
        int i2[G];
        T acc[G], B[G], run[G];
#pragma unroll
        for (int q = 0; q < G; ++q) {
            i2[q] = i < n - seps[q] ? i + seps[q] : i - (n - seps[q]);
            acc[q] = B[q] = run[q] = T(0);
        }
        const T* row = fk;
#pragma unroll 2
        for (int j = 0; j < nv; ++j) {
            const T a = row[i];
#pragma unroll
            for (int q = 0; q < G; ++q) {
                acc[q] += a * run[q];
                B[q] += row[i2[q]];
                run[q] += B[q];
            }
            row += n;
        }
#pragma unroll
        for (int q = 0; q < G; ++q) B[q] = run[q] = T(0);
#pragma unroll 2
        for (int j = nv - 1; j >= 0; --j) {
            row -= n;
            const T a = row[i];
#pragma unroll
            for (int q = 0; q < G; ++q) {
                acc[q] += a * run[q];
                B[q] += row[i2[q]];
                run[q] += B[q];
            }
        }
        const double* rk = rho + in.xoff;
        const double ri = rk[i];
#pragma unroll
        for (int q = 0; q < G; ++q) {
            nadd(t[2 * q], (double)acc[q]);
            nadd(t[2 * q + 1], ri * rk[i2[q]]);
        }
    }
    // halve the sums a lane holds, level by level, until it holds one (of index lane / (32 / NS));
    // the lanes left with the same one add theirs
#pragma unroll
    for (int m = 16, h = G; m >= 1; m >>= 1, h >>= 1) {
        if (h >= 1) {
            const bool up = (lane & m) != 0;
#pragma unroll
            for (int q = 0; q < h; ++q) {
                const Comp keep = up ? t[q + h] : t[q], give = up ? t[q] : t[q + h];
                t[q] = keep;
                nmerge(t[q], shfl_xor(give, m));
            }
        } else {
            nmerge(t[0], shfl_xor(t[0], m));
        }
    }
    if (lane % (32 / NS) == 0) wsum[warp][lane / (32 / NS)] = t[0];
    __syncthreads();
    if (threadIdx.x < NS) {
        Comp z{0, 0};
        for (int w = 0; w < kS1Threads / 32; ++w) nmerge(z, wsum[w][threadIdx.x]);
        double* p = part + (((size_t)blockIdx.y * gridDim.x + blockIdx.x) * NS + threadIdx.x) * 2;
        p[0] = z.s;
        p[1] = z.c;
    }
}

// One thread per sum of an instance folds its slots' sums in order: groups of G separations, the
// first one seps[q0].
__global__ void k_s1_fold(const double* part, long long slots, int cpt, const Inst1D* inst,
                          int n_inst, int G, int groups, int q0, int ns, double* num, double* den) {
    const int NS = 2 * G, per = kS1Threads * cpt;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int k = (int)(i / (groups * NS)), r = (int)(i % (groups * NS));
    if (k >= n_inst) return;
    const Inst1D& in = inst[k];
    const double* p = part + (((r / NS) * slots + s1_slot(in, k, per)) * NS + r % NS) * 2;
    Comp z{0, 0};
    for (long long x0 = 0; x0 < in.nx; x0 += per, p += 2 * NS) nmerge(z, Comp{p[0], p[1]});
    const size_t o = (size_t)k * ns + q0 + r / 2;
    if (r % 2 == 0) num[o] = nval(z) * in.dv * in.dv * in.dv / in.nx;
    else den[o] = nval(z) / in.nx;
}

// Cells per thread: eight where that still leaves sixteen blocks per SM.
int s1_cells(long long total_x, int sm_count) {
    const long long c = total_x / ((long long)kS1Threads * 16 * sm_count);
    return (int)std::max(1ll, std::min(8ll, c));
}

// How ns separations of a state are dealt out: groups of G, `batch` of them per launch, then the rest in
// groups of the smaller powers of two, so that no sweep is made for a separation that was not asked
// for (each costs its own sums).  G is the largest that leaves four blocks per SM: few columns in large
// groups would leave the SMs idle.  The call with the density, 512 instances of 1024 .. 4096 columns,
// N_v = 9, FP32: one separation 190 us, nine 638 us (a block per instance and separation 216 and 629,
// whole groups of eight 552 and 996); 9 instances of 256, N_v = 65, FP64, one 157 us (210, 253).
struct S1Split {
    int cpt, G, batch;
    long long slots;
};

int pow2_from(int n) {
    int p = 1;
    while (p < n) p *= 2;
    return p;
}

S1Split s1_split(int n_inst, long long total_x, int ns, int sm_count) {
    S1Split q;
    q.cpt = s1_cells(total_x, sm_count);
    q.slots = total_x / (kS1Threads * q.cpt) + n_inst;
    q.G = std::min(kS1Group, pow2_from(ns));
    while (q.G > 1 && q.slots * ((ns + q.G - 1) / q.G) < 4ll * sm_count) q.G /= 2;
    // groups together while their blocks would not fill sixteen per SM
    const long long most = 16ll * sm_count / q.slots;
    q.batch = (int)std::max(1ll, std::min<long long>(most, (ns + q.G - 1) / q.G));
    return q;
}

template <typename T>
cudaError_t launch_s1_group(int G, int groups, const S1Split& sp, const void* f, const Inst1D* inst,
                            int n_inst, int nv, const double* rho, const int* seps, double* part,
                            cudaStream_t s) {
    const dim3 grid((unsigned)sp.slots, groups);
    switch (G) {
#define X(g) \
    case g:  \
        k_s1_1d<T, g><<<grid, kS1Threads, 0, s>>>(static_cast<const T*>(f), inst, n_inst, sp.cpt, \
                                                  nv, rho, seps, part);                           \
        return cudaGetLastError();
        X(1) X(2) X(4) X(8)
#undef X
        default: return cudaErrorInvalidValue;
    }
}

int obs_grid(long long blocks, int sm_count) {
    return (int)std::max(1ll, std::min(blocks, (long long)sm_count * 16));
}

}  // namespace

// P: 2 (total_x + n_inst) doubles of scratch.
cudaError_t launch_coarse1d(const double* rho, const Inst1D* inst, int n_inst, long long total_x,
                            const int* widths, int nw, double* P, double* out, int sm_count,
                            cudaStream_t s) {
    double* Pl = P + total_x + n_inst;
    k_prefix1d<<<obs_grid(n_inst, sm_count), kPrefixThreads, 0, s>>>(rho, inst, n_inst, P, Pl);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_coarse1d<<<obs_grid((long long)n_inst * nw, sm_count), kObsThreads, 0, s>>>(
        P, Pl, inst, n_inst, widths, nw, out);
    return cudaGetLastError();
}

// S: 2 (ny + 1)(nx + 1) doubles of scratch.
cudaError_t launch_coarse2d(const double* rho, int nx, int ny, double dx, const int* widths,
                            int nw, double* S, double* out, int sm_count, cudaStream_t s) {
    double* Sl = S + (size_t)(ny + 1) * (nx + 1);
    k_sat_rows<<<(ny + 1 + 127) / 128, 128, 0, s>>>(rho, nx, ny, S, Sl);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_sat_cols<<<(nx + 1 + 127) / 128, 128, 0, s>>>(nx, ny, S, Sl);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_coarse2d<<<obs_grid(nw, sm_count), kObsThreads, 0, s>>>(S, Sl, nx, ny, dx, widths, nw,
                                                             out);
    return cudaGetLastError();
}

size_t s1_scratch(int n_inst, long long total_x, int ns, int sm_count) {
    const S1Split sp = s1_split(n_inst, total_x, ns, sm_count);
    return (size_t)sp.slots * 4 * sp.batch * sp.G;
}

cudaError_t launch_s1_1d(int dtype, const void* f, const Inst1D* inst, int n_inst,
                         long long total_x, int nv, const double* rho, const int* seps, int ns,
                         double* part, double* num, double* den, int sm_count, cudaStream_t s) {
    if (dtype != LAT_F32 && dtype != LAT_F64) return cudaErrorInvalidValue;
    const S1Split sp = s1_split(n_inst, total_x, ns, sm_count);
    for (int q0 = 0; q0 < ns;) {
        int G = sp.G, groups = std::min(sp.batch, (ns - q0) / sp.G);
        if (groups == 0) {
            groups = 1;
            while (G > ns - q0) G /= 2;
        }
        const cudaError_t e =
            dtype == LAT_F32
                ? launch_s1_group<float>(G, groups, sp, f, inst, n_inst, nv, rho, seps + q0, part, s)
                : launch_s1_group<double>(G, groups, sp, f, inst, n_inst, nv, rho, seps + q0, part, s);
        if (e != cudaSuccess) return e;
        const long long sums = (long long)n_inst * groups * 2 * G;
        k_s1_fold<<<(unsigned)((sums + 127) / 128), 128, 0, s>>>(part, sp.slots, sp.cpt, inst, n_inst,
                                                                 G, groups, q0, ns, num, den);
        q0 += groups * G;
    }
    return cudaGetLastError();
}

}  // namespace lat
