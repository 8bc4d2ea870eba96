// Many time steps of small 1D lattices in one launch (FP32 or FP64, upwind drag, any N_v): one
// thread-block cluster per lattice holds the state in its blocks' shared memory for all the steps.
//
// A lattice of a few thousand cells (the paper's N_x = 256, N_v = 33) is far too small for one
// launch per step: a step is a fraction of a microsecond of work, a launch several, and one
// block of one thread per column runs the whole lattice on one SM (FP64: two operations per clock
// and SM).  Here the columns are split over the blocks of a cluster of 16, a thread takes one
// cell (several where the lattice is larger), and the values a cell needs of its velocity neighbours
// pass through shared memory.  Each product, flux and difference is formed once, as in sweep_column
// and with its operations, so the results have its bits.  The streaming is the store of the result:
// cell (x, j) goes into the next step's array of the block that owns column x + j (distributed
// shared memory), and a cluster barrier ends the step.
//
// One warp beside those of the cells forms the next step's flow meanwhile: the amplitudes' update,
// then u / dv of the block's columns from the basis kept in shared memory.
//
// Measured, per step of N_x = 256, N_v = 33: FP64 3.5 us (49.6 in one block of 256 columns, 22.5 in
// blocks of 32), bound by the FP64 pipes of 16 SMs; FP32 1.25 us (2.7 five steps at a time on
// multi1d.cu's tiles, 3.8 with a launch per step), of which the cluster barrier and the flow's
// serial sums take about 1.0 (N_x = 64, N_v = 9: 1.08 us).  In FP32 a cell forms all it needs of its
// four neighbours' values at once: passing the parts through shared memory with four barriers, as
// in FP64, took 3.2 us at N_x = 512 against 1.8.
#include <cooperative_groups.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "lat_internal.h"
#include "per_device.h"
#include "step1d_dev.h"

namespace lat {
namespace {

namespace cg = cooperative_groups;
using namespace k1d;

constexpr int kCluster = 16;
constexpr int kCellThreads = 992;  // at most; 32 more for the flow
constexpr size_t kMaxSmem = 220 * 1024;
constexpr int kMaxInst = 8;
constexpr long long kMaxCells64 = 80000, kMaxCells32 = 30000;  // larger ones: not measured

template <typename T>
size_t line_smem(int nv, int w, int nmodes) {
    const size_t cells = (size_t)nv * w;
    return sizeof(T) * ((sizeof(T) == 8 ? 5 : 2) * cells + 2 * w + 2 * (size_t)nmodes * w + 2 * nmodes) + 16;
}

// ONE: a thread has at most one cell.
template <typename T, bool ONE>
__global__ void __launch_bounds__(1024) k_line1d(const Step1DArgs a, int kstep, int n, int wmax) {
    using O = Ops<T>;
    extern __shared__ __align__(16) unsigned char smem[];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int inst = blockIdx.x / kCluster;
    const Inst1D& in = a.inst[inst];
    const int nx = in.nx, nv = a.nv, J = (nv - 1) / 2;
    const int w = (nx + kCluster - 1) / kCluster;  // columns per block (the last ones fewer, or none)
    const int x0 = rank * w, nc = max(0, min(w, nx - x0));
    const int M = a.flow_kind == LAT_FLOW_MODES ? a.nmodes : 0;
    const size_t cap = (size_t)nv * wmax;          // elements of an array (same in every block)
    T* S0 = reinterpret_cast<T*>(smem);            // f* of the current and the next step, [j][column]
    T* S1 = S0 + cap;
    const size_t cap64 = sizeof(T) == 8 ? cap : 0;  // FP64 only
    T* A = S1 + cap;                               // M parts, then diffusion fluxes
    T* F = A + cap64;                              // drag fluxes
    T* E = F + cap64;                              // densities after the drag
    T* W = E + cap64;                                // u / dv of the columns, two steps
    T* B = W + 2 * wmax;                           // basis: [column][sin, cos][mode]
    T* amp = B + 2 * (size_t)M * wmax;             // amplitudes of the step being formed
    const long long step0 = a.st->step + kstep;
    const int par = (int)(step0 & 1);
    const T* fin = static_cast<const T*>(par ? a.f[1] : a.f[0]) + in.off;
    T* fout = static_cast<T*>((step0 + n) & 1 ? a.f[1] : a.f[0]) + in.off;
    const int tid = threadIdx.x, nt = blockDim.x - 32;
    const bool flow_warp = tid >= nt;
    const int lane = tid & 31;
    const T g = T(in.g), r = T(in.r), inv_dv = T(in.inv_dv);
    const int cells = nv * nc;
    for (int i = tid; i < cells; i += blockDim.x) {  // f* of the first step
        const int jj = i / nc, c = i - jj * nc;
        int xs = (x0 + c - (jj - J)) % nx;
        xs += xs < 0 ? nx : 0;
        S0[i] = fin[(size_t)jj * nx + xs];
    }
    for (int i = tid; i < M * nc; i += blockDim.x) {
        const int m = i / nc, c = i - m * nc;
        T s, q;
        flow_basis<T>(a.k[m], in, T(in.two_over_nx), x0 + c, &s, &q);
        B[(size_t)c * 2 * M + m] = s;
        B[(size_t)c * 2 * M + M + m] = q;
    }
    // the flow warp's state: lane t < 2M holds amplitude t and the noise of the coming update
    double v = 0.0, xi = 0.0;
    const long long base = a.st->noise_base, rows = a.st->noise_rows;
    const long long at = (long long)inst * 2 * M + lane;
    bool missing = false, cfl = false;
    auto draw = [&](long long s) {  // the noise row of the update after step step0 + s
        const long long row = step0 + s - base;
        const bool have = row >= 0 && row < rows;
        if (s < n) missing |= !have;
        return have && s < n ? a.noise[row * a.amp_stride + at] : 0.0;
    };
    auto form = [&](T* Wd) {  // u / dv of the block's columns from the amplitudes in v
        if (lane < 2 * M) amp[lane] = T(v);
        __syncwarp();
        for (int c = lane; c < nc; c += 32) {
            T u = T(0);
            if (a.flow_kind == LAT_FLOW_FIELD) {
                u = static_cast<const T*>(a.field)[in.xoff + x0 + c];
            } else {
                const T* b = B + (size_t)c * 2 * M;
                for (int m = 0; m < M; ++m) u = flow_add<T>(u, amp[m], amp[M + m], b[m], b[M + m]);
            }
            const T ws = u * inv_dv;
            Wd[c] = ws;
            cfl |= g * (T(J) + fabs(ws)) > T(1);
        }
        __syncwarp();
    };
    __syncthreads();
    if (flow_warp) {
        if (lane < 2 * M) {
            v = a.amp[par * a.amp_stride + at];
            if (!a.frozen) xi = draw(0);
        }
        form(W);
    }
    cl.sync();
    T* cur = S0;
    T* nxt = S1;
    // place of cell (jj, c)'s streamed value in the S0 of its column's block
    auto place = [&](int jj, int c) {
        int x = (x0 + c + jj - J) % nx;
        x += x < 0 ? nx : 0;
        const int owner = x / w, first = owner * w;
        return cl.map_shared_rank(S0, owner) + jj * min(w, nx - first) + x - first;
    };
    const int jt = nc ? tid / nc : 0, ct = nc ? tid - jt * nc : 0;  // this thread's first cell
    const int dj = nc ? nt / nc : 0, dc = nc ? nt - dj * nc : 0;
    T* dest = !flow_warp && tid < cells ? place(jt, ct) : S0;
    auto each = [&](auto&& body) {
        if (ONE) {
            if (tid < cells) body(tid, jt, ct);
        } else {
            for (int i = tid, jj = jt, c = ct; i < cells; i += nt) {
                body(i, jj, c);
                jj += dj;
                c += dc;
                if (c >= nc) c -= nc, ++jj;
            }
        }
    };
    auto sync_cells = [&] { asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory"); };
    for (int s = 0; s < n; ++s) {
        const T* Wc = W + (s & 1) * wmax;
        if (flow_warp) {
            if (lane < 2 * M && !a.frozen) {
                v = __dadd_rn(__dmul_rn(v, in.ou_e), __dmul_rn(in.ou_s, xi));
                xi = draw(s + 1);
            }
            if (s + 1 < n) form(W + ((s + 1) & 1) * wmax);
        } else {
            auto store = [&](int jj, int c, T o) {
                if (s + 1 == n) fout[(size_t)jj * nx + x0 + c] = o;
                else (ONE ? dest : place(jj, c))[nxt - S0] = o;
            };
            if constexpr (sizeof(T) == 4) {
                // every cell on its own, from f* of its two neighbours on either side
                each([&](int i, int jj, int c) {
                    const T wc = Wc[c];
                    T q[5], ca[5];
#pragma unroll
                    for (int k = 0; k < 5; ++k) {
                        const int j2 = jj + k - 2;
                        q[k] = j2 >= 0 && j2 < nv ? cur[i + (k - 2) * nc] : T(0);
                        ca[k] = cacc<T>(g, wc, j2 - J);
                    }
                    T Fk[4];  // faces jj - 3/2 .. jj + 3/2
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int j2 = jj + k - 2;  // between cells j2 and j2 + 1
                        Fk[k] = j2 >= 0 && j2 < nv - 1 ? dflux<T>(ca[k], ca[k + 1], q[k], q[k + 1])
                                                       : T(0);
                    }
                    T d[3];
#pragma unroll
                    for (int k = 0; k < 3; ++k) d[k] = O::sub(q[k + 1], O::sub(Fk[k + 1], Fk[k]));
                    const T Du = jj < nv - 1 ? O::mul(r, O::sub(d[2], d[1])) : T(0);
                    const T Dl = jj > 0 ? O::mul(r, O::sub(d[1], d[0])) : T(0);
                    store(jj, c, O::add(d[1], O::sub(Du, Dl)));
                });
            } else {
            // (c a_j)^- f_j of every cell
            each([&](int i, int jj, int c) {
                A[i] = O::mul(neg_part(cacc<T>(g, Wc[c], jj - J)), cur[i]);
            });
            sync_cells();
            // drag flux through face j + 1/2
            each([&](int i, int jj, int c) {
                F[i] = jj < nv - 1 ? O::fma(pos_part(cacc<T>(g, Wc[c], jj - J)), cur[i], A[i + nc]) : T(0);
            });
            sync_cells();
            each([&](int i, int jj, int) {
                E[i] = O::sub(cur[i], O::sub(F[i], jj > 0 ? F[i - nc] : T(0)));
            });
            sync_cells();
            // diffusion flux through face j + 1/2
            each([&](int i, int jj, int) {
                A[i] = jj < nv - 1 ? O::mul(r, O::sub(E[i + nc], E[i])) : T(0);
            });
            sync_cells();
            each([&](int i, int jj, int c) {
                store(jj, c, O::add(E[i], O::sub(A[i], jj > 0 ? A[i - nc] : T(0))));
            });
            }
        }
        cl.sync();
        T* t = cur;
        cur = nxt;
        nxt = t;
    }
    if (flow_warp) {
        if (cfl) atomicOr(&a.st->status, ST_CFL);
        if (rank == 0 && M > 0 && !a.frozen && lane < 2 * M) {
            const int pn = (int)((step0 + n) & 1);
            a.amp_w[pn * a.amp_stride + at] = v;
            a.ampf_w[pn * a.amp_stride + at] = (float)v;
            if (missing && lane == 0) atomicOr(&a.st->status, ST_NOISE);
        }
        // a single lattice: every block has read the step counter by now
        if (gridDim.x == kCluster && rank == 0 && lane == 0) a.st->step = step0 + n;
    }
}

template <typename T, bool ONE>
cudaError_t config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at, int n_inst, int nv, int w,
                   int nmodes, cudaStream_t s) {
    const size_t smem = line_smem<T>(nv, w, nmodes);
    static PerDevice limit, size;
    cudaError_t e = raise_smem(limit, k_line1d<T, ONE>, kMaxSmem);
    int done = 0;
    if (e == cudaSuccess)
        e = size.get(&done, [](int*) {
            return cudaFuncSetAttribute(k_line1d<T, ONE>,
                                        cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        });
    if (e != cudaSuccess) return e;
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3(n_inst * kCluster);
    cfg->blockDim = dim3(std::min(kCellThreads, (nv * w + 31) / 32 * 32) + 32);
    cfg->dynamicSmemBytes = smem;
    cfg->stream = s;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = kCluster;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg->attrs = at;
    cfg->numAttrs = 1;
    return cudaSuccess;
}

template <typename T, bool ONE>
int runs(int nv, int w, int nmodes) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    int nclusters = 0;
    const bool ok = line_smem<T>(nv, w, nmodes) <= kMaxSmem &&
                    config<T, ONE>(&cfg, &at, 1, nv, w, nmodes, nullptr) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&nclusters, k_line1d<T, ONE>, &cfg) == cudaSuccess;
    return ok ? nclusters : 0;
}

template <typename T, bool ONE>
cudaError_t launch_t(int n_inst, int nv, int w, const Step1DArgs& a, int kstep, int n,
                     cudaStream_t s) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    const int M = a.flow_kind == LAT_FLOW_MODES ? a.nmodes : 0;
    const cudaError_t e = config<T, ONE>(&cfg, &at, n_inst, nv, w, M, s);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, k_line1d<T, ONE>, a, kstep, n, w);
}

int columns(int nx_max) { return (nx_max + kCluster - 1) / kCluster; }

}  // namespace

// At most eight lattices, one cluster each, as far as shared memory holds them.
int line1d_clusters(int dtype, int n_inst, int nx_max, int nv, int nmodes) {
    const long long cells = (long long)nx_max * nv;
    if (n_inst > kMaxInst || cells > (dtype == LAT_F64 ? kMaxCells64 : kMaxCells32)) return 0;
    const int w = columns(nx_max);
    const bool one = nv * w <= kCellThreads;
    const int n = dtype == LAT_F64
                      ? (one ? runs<double, true>(nv, w, nmodes) : runs<double, false>(nv, w, nmodes))
                      : (one ? runs<float, true>(nv, w, nmodes) : runs<float, false>(nv, w, nmodes));
    if (n == 0) cudaGetLastError();
    return n;
}

// A step is bound by the flow warp, which takes a block's columns 32 at a time, or by the cells; more
// clusters than run at a time take turns.  Measured per step (and a launch's fixed part), eight modes:
// FP64 N_x = 256, N_v = 9 2.0 us (6.3); 1001, 33 11.1 us (11.8); 4096, 5 14.9 us (23); FP32 256, 9
// 0.9 us (5.7); 1001, 21 2.0 us (6.3); 8888, 3 7.9 us (7).
double line1d_us(int dtype, int n_inst, int nx_max, int nv, int nmodes, int clusters, int n) {
    const int rounds = (columns(nx_max) + 31) / 32;
    const double modes = rounds * (nmodes / 8.0), kcells = 1e-3 * nx_max * nv;
    const int turns = (n_inst + clusters - 1) / clusters;
    if (dtype == LAT_F64)
        return 5.0 + turns * (2.2 * modes + n * (0.4 + 0.1 * rounds + 1.2 * modes + 0.25 * kcells));
    return 5.5 + turns * (0.3 * modes + n * (0.4 + 0.05 * rounds + 0.38 * modes + 0.03 * kcells));
}

cudaError_t launch_line1d(int dtype, int n_inst, int nx_max, int nv, const Step1DArgs& a, int kstep,
                          int n, cudaStream_t s) {
    const int w = columns(nx_max);
    const bool one = nv * w <= kCellThreads;
    if (dtype == LAT_F64)
        return one ? launch_t<double, true>(n_inst, nv, w, a, kstep, n, s)
                   : launch_t<double, false>(n_inst, nv, w, a, kstep, n, s);
    return one ? launch_t<float, true>(n_inst, nv, w, a, kstep, n, s)
               : launch_t<float, false>(n_inst, nv, w, a, kstep, n, s);
}

}  // namespace lat
