// One fused time step of the 1D phase-space lattice (Section 2 of arXiv:1508.02899):
// exact streaming in x, first-order upwind Stokes-drag flux in v, velocity diffusion.
//
// Work decomposition: a work item is one x-tile of one instance; a persistent grid walks the
// item list.  Each thread owns one spatial column x and sweeps its velocity column
// j = -J..J once: the post-streaming value f*(x, j) = f(x - j, j) is gathered (the gather *is*
// the streaming step), the drag flux and the diffusion flux are carried along the sweep as
// scalars with a lag of two cells, and each output value is written once.  HBM traffic per
// cell: one read and one write of f.
//
// Three variants share the column arithmetic (bit-identical results):
//  * ring: the tile's N_v shifted plane windows are brought into a shared-memory ring by bulk
//    asynchronous copies (cp.async.bulk + mbarrier), several items ahead of the sweep, so the
//    loads in flight do not depend on registers or occupancy (FP32, N_x % 4 == 0, N_x >= 132);
//  * reg:  the column is gathered with plain coalesced loads into registers (fixed N_v);
//  * any:  plain loads through a sliding window (any odd N_v).
// The flow u(x, t_n) is evaluated in the same kernel from the mode amplitudes; the first tile
// of every instance also advances those amplitudes to t_{n+1} (parity ping-pong, so no tile
// reads what another tile of the same launch writes).
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "lat_internal.h"
#include "per_device.h"
#include "lat_reduce.h"
#include "step1d_dev.h"

namespace lat {
namespace {

using namespace k1d;

constexpr int TW1 = 128;        // columns per tile of the ring kernel (= threads per block)
constexpr int WIN1 = TW1 + 4;   // floats copied per plane (x window rounded to 16 bytes)

// ---- reg / any variants (plain loads) ----------------------------------------------------------
template <typename T, int NV>
struct MaxThreads {
    static constexpr int words = NV * (int)(sizeof(T) / 4);
    static constexpr int value = words > 56 ? 256 : (words > 20 ? 512 : 1024);
};

template <typename T, int NV, bool LIM>
__global__ void __launch_bounds__(MaxThreads<T, NV>::value)
    k_step1d_reg(const Step1DArgs a, const int kstep) {
    constexpr int J = (NV - 1) / 2;
    const long long step = a.st->step + kstep;
    const int par = (int)(step & 1);
    for (int it = a.item_begin + blockIdx.x; it < a.item_end; it += gridDim.x) {
        const int2 item = a.items[it];
        const Inst1D in = a.inst[item.x];
        const int nx = in.nx;
        const int x = item.y + threadIdx.x;
        if (x < nx) {
            const T g = T(in.g), r = T(in.r);
            const T* __restrict__ src = static_cast<const T*>(a.f[par]) + in.off;
            T* __restrict__ dst = static_cast<T*>(a.f[par ^ 1]) + in.off + x;
            const T w = flow_w<T>(a, in, amp_ptr<T>(a, par, item.x), x);
            T f[NV];
            if (nx >= J) {
#pragma unroll
                for (int jj = 0; jj < NV; ++jj) {
                    int xs = x - (jj - J);
                    xs += (xs < 0) ? nx : 0;
                    xs -= (xs >= nx) ? nx : 0;
                    f[jj] = __ldg(src + (size_t)jj * nx + xs);
                }
            } else {
#pragma unroll
                for (int jj = 0; jj < NV; ++jj) {
                    int xs = (x - (jj - J)) % nx;
                    xs += (xs < 0) ? nx : 0;
                    f[jj] = __ldg(src + (size_t)jj * nx + xs);
                }
            }
            sweep_scheme<T, NV, LIM>(
                a, w, g, r, [&](int jj) { return f[jj]; },
                [&](int jj, T v) { dst[(size_t)jj * nx] = v; });
            cfl_flag<T, J, LIM>(a, g, w);
        }
        if (!a.dry && !a.frozen && !a.wpre && a.flow_kind == LAT_FLOW_MODES && item.y == 0)
            advance_amplitudes(a, item.x, in, step, par);
    }
}

template <typename T>
__global__ void __launch_bounds__(512) k_step1d_any(const Step1DArgs a, const int kstep,
                                                    const int NV) {
    const int J = (NV - 1) / 2;
    const long long step = a.st->step + kstep;
    const int par = (int)(step & 1);
    for (int it = a.item_begin + blockIdx.x; it < a.item_end; it += gridDim.x) {
        const int2 item = a.items[it];
        const Inst1D in = a.inst[item.x];
        const int nx = in.nx;
        const int x = item.y + threadIdx.x;
        if (x < nx) {
            const T g = T(in.g), r = T(in.r);
            const T* __restrict__ src = static_cast<const T*>(a.f[par]) + in.off;
            T* __restrict__ dst = static_cast<T*>(a.f[par ^ 1]) + in.off + x;
            const T w = flow_w<T>(a, in, amp_ptr<T>(a, par, item.x), x);
            sweep_column_any<T>(
                NV, w, g, r,
                [&](int jj) {
                    int xs = (x - (jj - J)) % nx;
                    xs += (xs < 0) ? nx : 0;
                    return __ldg(src + (size_t)jj * nx + xs);
                },
                [&](int jj, T v) { dst[(size_t)jj * nx] = v; });
            if (g * (T(J) + fabs(w)) > T(1)) atomicOr(&a.st->status, ST_CFL);
        }
        if (!a.dry && !a.frozen && !a.wpre && a.flow_kind == LAT_FLOW_MODES && item.y == 0)
            advance_amplitudes(a, item.x, in, step, par);
    }
}

// ---- ring variant (FP32, bulk async copies into a shared-memory ring) --------------------------
__device__ __forceinline__ int wrapi(int v, int n) {
    v %= n;
    return v < 0 ? v + n : v;
}

// Copy the N_v shifted windows of item `it` into ring slot `slot` (warp 0 only): plane j needs
// columns [x0 - j, x0 - j + 128); the window starts at that offset rounded down to 16 bytes and
// is split in two at the periodic wrap.
template <int NV>
__device__ __forceinline__ void issue_item(const Step1DArgs& a, const float* fin, float* ring,
                                           uint64_t* bar, int slot, int it) {
    constexpr int J = (NV - 1) / 2;
    const int lane = threadIdx.x & 31;
    if (lane == 0) mbar_expect_tx(&bar[slot], (unsigned)(NV * WIN1 * sizeof(float)));
    __syncwarp();
    const int2 item = a.items[it];
    const Inst1D& in = a.inst[item.x];
    const float* base_ptr = fin + in.off;
    for (int jj = lane; jj < NV; jj += 32) {
        const float* prow = base_ptr + (size_t)jj * in.nx;
        const int s = item.y - (jj - J);
        const int b = wrapi(s - ((s % 4) + 4) % 4, in.nx);
        float* dst = ring + ((size_t)slot * NV + jj) * WIN1;
        if (b + WIN1 <= in.nx) {
            bulk_g2s(dst, prow + b, WIN1 * sizeof(float), &bar[slot]);
        } else {
            const int n1 = in.nx - b;
            bulk_g2s(dst, prow + b, n1 * sizeof(float), &bar[slot]);
            bulk_g2s(dst + n1, prow, (WIN1 - n1) * sizeof(float), &bar[slot]);
        }
    }
}

template <int NV, int NS, bool LIM>
__global__ void __launch_bounds__(TW1) k_step1d_ring(const Step1DArgs a, const int kstep) {
    constexpr int J = (NV - 1) / 2;
    extern __shared__ __align__(128) unsigned char smem[];
    float* ring = reinterpret_cast<float*>(smem);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + (size_t)NS * NV * WIN1 * sizeof(float));
    const long long step = a.st->step + kstep;
    const int par = (int)(step & 1);
    const float* fin = static_cast<const float*>(a.f[par]);
    float* fout = static_cast<float*>(a.f[par ^ 1]);
    const int tid = threadIdx.x;
    const int first = a.item_begin + blockIdx.x;
    const int nloc = first < a.item_end ? (a.item_end - 1 - first) / gridDim.x + 1 : 0;
    if (tid == 0) {
        for (int q = 0; q < NS; ++q) mbar_init(&bar[q], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (tid < 32)
        for (int k = 0; k < NS - 1 && k < nloc; ++k)
            issue_item<NV>(a, fin, ring, bar, k % NS, first + k * gridDim.x);
    int issued = std::min(NS - 1, nloc);
    bool failed = false;
    for (int k = 0; k < nloc; ++k) {
        if (__syncthreads_or(failed ? 1 : 0)) {
            failed = true;
            break;
        }
        // slot (k + NS - 1) % NS held item k - 1, which every thread has finished
        if (k + NS - 1 < nloc) {
            if (tid < 32) {
#if LAT_RING_PROXY_FENCE
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
#endif
                issue_item<NV>(a, fin, ring, bar, (k + NS - 1) % NS,
                               first + (k + NS - 1) * gridDim.x);
            }
            issued = k + NS;
        }
        const int it = first + k * gridDim.x;
        const int2 item = a.items[it];
        const Inst1D in = a.inst[item.x];
        const int x = item.y + tid;
        const float g = float(in.g), r = float(in.r);
        float w = 0.f;
        if (x < in.nx) w = flow_at<float>(a, in, amp_ptr<float>(a, par, item.x), x) * float(in.inv_dv);
        if (!mbar_wait_bounded(&bar[k % NS], (unsigned)((k / NS) & 1))) {
            failed = true;
            continue;
        }
        if (x < in.nx) {
            const float* col = ring + (size_t)(k % NS) * NV * WIN1 + tid;
            float* dst = fout + in.off + x;
            const int nx = in.nx;
            sweep_scheme<float, NV, LIM>(
                a, w, g, r,
                [&](int jj) { return col[jj * WIN1 + ((J - jj) % 4 + 4) % 4]; },
                [&](int jj, float v) { dst[(size_t)jj * nx] = v; });
            cfl_flag<float, J, LIM>(a, g, w);
        }
        if (!a.dry && !a.frozen && a.flow_kind == LAT_FLOW_MODES && item.y == 0)
            advance_amplitudes(a, item.x, in, step, par);
    }
    if (failed) {
        if (tid == 0) {
            atomicOr(&a.st->status, ST_TIMEOUT);
            // let the copies already issued land before the block's shared memory goes away
            for (int k = std::max(0, issued - NS); k < issued; ++k)
                mbar_wait_bounded(&bar[k % NS], (unsigned)((k / NS) & 1));
        }
        __syncthreads();
    }
}

// ---- producer/consumer variant: no block-wide barrier per item -------------------------------
// Four consumer warps own the 128 columns of an item; a fifth warp only produces: it refills a
// ring slot with the next item's plane windows once every consumer warp has released the slot
// (per-slot "empty" mbarrier, one arrival per consumer warp).  Consumers wait only on the
// per-slot "full" mbarrier that the bulk copies complete, so warps drift freely.
constexpr int PC1_CONSUMERS = TW1 / 32;
constexpr int PC1_THREADS = 32 * (PC1_CONSUMERS + 1);

template <int NV, int NS>
size_t pc1d_smem() {
    return (size_t)NS * NV * WIN1 * sizeof(float) + 2 * NS * sizeof(uint64_t);
}

// With MOM the consumers also reduce the moments of the columns they write (the same FP32
// column sums, in the same order, as the moment kernel; compensated across cells).
template <int NV, int NS, bool MOM, bool LIM>
__global__ void __launch_bounds__(PC1_THREADS) k_step1d_pc(const Step1DArgs a, const int kstep) {
    constexpr int J = (NV - 1) / 2;
    extern __shared__ __align__(128) unsigned char smem[];
    float* ring = reinterpret_cast<float*>(smem);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)NS * NV * WIN1 * sizeof(float));
    uint64_t* empty = full + NS;
    const long long step = a.st->step + kstep;
    const int par = (int)(step & 1);
    const float* fin = static_cast<const float*>(a.f[par]);
    float* fout = static_cast<float*>(a.f[par ^ 1]);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int first = a.item_begin + blockIdx.x;
    const int nloc = first < a.item_end ? (a.item_end - 1 - first) / gridDim.x + 1 : 0;
    if (threadIdx.x == 0) {
        for (int q = 0; q < NS; ++q) {
            mbar_init(&full[q], 1);
            mbar_init(&empty[q], PC1_CONSUMERS);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (warp == PC1_CONSUMERS) {
        // a stalled context issues no copies: every consumer's bounded wait runs out
        const int nfill = a.st->stall ? 0 : nloc;
        int k = 0;
        for (; k < nfill; ++k) {
            const int q = k % NS;
            if (k >= NS && !mbar_wait_bounded(&empty[q], (unsigned)(((k / NS) + 1) & 1))) {
                if (lane == 0) atomicOr(&a.st->status, ST_TIMEOUT);
                break;
            }
            issue_item<NV>(a, fin, ring, full, q, first + k * gridDim.x);
        }
        // the copies issued last must land before this warp leaves
        for (int d = std::max(0, k - NS); d < k; ++d)
            mbar_wait_bounded(&full[d % NS], (unsigned)((d / NS) & 1));
        return;
    }
    const int tid = threadIdx.x;
    for (int k = 0; k < nloc; ++k) {
        const int it = first + k * gridDim.x;
        const int2 item = a.items[it];
        const Inst1D in = a.inst[item.x];
        const int x = item.y + tid;
        const float g = float(in.g), r = float(in.r);
        float w = 0.f;
        if (x < in.nx) w = flow_at<float>(a, in, amp_ptr<float>(a, par, item.x), x) * float(in.inv_dv);
        if (!mbar_wait_bounded(&full[k % NS], (unsigned)((k / NS) & 1))) {
            if (lane == 0) atomicOr(&a.st->status, ST_TIMEOUT);
            break;
        }
        cs::ColumnSums sums;
        if (x < in.nx) {
            const float* col = ring + (size_t)(k % NS) * NV * WIN1 + tid;
            float* dst = fout + in.off + x;
            const int nx = in.nx;
            auto get = [&](int jj) { return col[jj * WIN1 + ((J - jj) % 4 + 4) % 4]; };
            if constexpr (!LIM && NV >= 5) {
                // packed two-lane sweep; the moments in ColumnSums2 order (lane 0: cells
                // 0 .. J - 1, lane 1: J .. 2J), the order of the moment kernel
                cs::ColumnSums2 s2;
                const f2 one2 = pk(1.f, 1.f);
                f2 jv = pk(float(-J), 0.f);
                sweep_column2<NV>(
                    w, g, r, get,
                    [&](int p, f2 o) {
                        dst[(size_t)(p - 1) * nx] = lo(o);
                        dst[(size_t)(p - 1 + J) * nx] = hi(o);
                        if constexpr (MOM) {
                            s2.add(jv, mul2(jv, jv), o);
                            jv = add2(jv, one2);
                        }
                    },
                    [&](float v) {
                        dst[(size_t)(NV - 1) * nx] = v;
                        if constexpr (MOM) s2.add_hi(float(J), v);
                    });
                if constexpr (MOM) sums = s2.collapse();
            } else {
                cs::ColumnSums2 s2;
                sweep_scheme<float, NV, LIM>(a, w, g, r, get, [&](int jj, float v) {
                    dst[(size_t)jj * nx] = v;
                    if constexpr (MOM) {
                        if (jj < J) s2.add_lo((float)(jj - J), v);
                        else s2.add_hi((float)(jj - J), v);
                    }
                });
                if constexpr (MOM) sums = s2.collapse();
            }
            cfl_flag<float, J, LIM>(a, g, w);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[k % NS]);
        if constexpr (MOM) {  // same per-warp partials as the moment kernel with 128 columns
            if (x < in.nx) {
                if (!isfinite(sums.a0.s) || !isfinite(sums.b2))
                    atomicOr(&a.st->status, ST_NUMERIC);
                // per-cell moments in FP64 only when asked for (FP64 is slow here)
                if (a.m_rho || a.m_mv || a.m_mv2) {
                    cs::Comp t0, t1, t2;
                    sums.result(in.dv, t0, t1, t2);
                    const double m0 = cs::nval(t0), m1 = cs::nval(t1), m2 = cs::nval(t2);
                    const long long cell = in.xoff + x;
                    if (a.m_rho) a.m_rho[cell] = m0 * in.dv;
                    if (a.m_mv) a.m_mv[cell] = (m0 != 0.0) ? m1 / m0 : 0.0;
                    if (a.m_mv2) a.m_mv2[cell] = (m0 != 0.0) ? m2 / m0 : 0.0;
                }
            }
            cs::warp_partial_1d(sums, in.dv,
                                a.m_partials + ((size_t)it * PC1_CONSUMERS + warp) * 6);
        }
        if (!a.dry && !a.frozen && a.flow_kind == LAT_FLOW_MODES && item.y == 0)
            advance_amplitudes(a, item.x, in, step, par);
    }
}

// The flow's basis of every grid size: sin and cos of 2 pi k_m x / N_x, [m][x].
template <typename T, typename T2>
__global__ void k_flow_basis(const Step1DArgs a, const int* sizes, int n_sizes, T2* table) {
    for (int q = blockIdx.y; q < n_sizes; q += gridDim.y) {
        const Inst1D in = a.inst[sizes[q]];
        const T two_over_nx = T(in.two_over_nx);
        T2* out = table + a.nmodes * a.size_off[sizes[q]];
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.nmodes * in.nx;
             i += gridDim.x * blockDim.x) {
            const int m = i / in.nx;
            flow_basis<T>(a.k[m], in, two_over_nx, i - m * in.nx, &out[i].x, &out[i].y);
        }
    }
}

__global__ void k_advance_step(DevState* st, long long n) { st->step += n; }

template <int NV, int NS, bool MOM, bool LIM>
cudaError_t launch_pc1_t(int grid, const Step1DArgs& a, int kstep, cudaStream_t s) {
    static PerDevice limit;
    const cudaError_t e = raise_smem(limit, k_step1d_pc<NV, NS, MOM, LIM>, pc1d_smem<NV, NS>());
    if (e != cudaSuccess) return e;
    k_step1d_pc<NV, NS, MOM, LIM><<<grid, PC1_THREADS, pc1d_smem<NV, NS>(), s>>>(a, kstep);
    return cudaGetLastError();
}

// the scheme's instance of the kernel
template <int NV, int NS, bool MOM = false>
cudaError_t launch_pc1(int grid, const Step1DArgs& a, int kstep, cudaStream_t s) {
    if (a.scheme == LAT_SCHEME_KOREN) return launch_pc1_t<NV, NS, MOM, true>(grid, a, kstep, s);
    return launch_pc1_t<NV, NS, MOM, false>(grid, a, kstep, s);
}

// Occupancy of the upwind instance; the limited one holds the same shared memory, which is what
// limits the resident blocks.
template <int NV, int NS>
int occupancy_pc1() {
    int nb = 0;
    cudaFuncSetAttribute(k_step1d_pc<NV, NS, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)pc1d_smem<NV, NS>());
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_step1d_pc<NV, NS, false, false>, PC1_THREADS,
                                                  pc1d_smem<NV, NS>());
    return nb;
}

template <int NV, int NS>
size_t ring1d_smem() {
    return (size_t)NS * NV * WIN1 * sizeof(float) + NS * sizeof(uint64_t);
}

template <int NV, int NS, bool LIM>
cudaError_t launch_ring_t(int grid, const Step1DArgs& a, int kstep, cudaStream_t s) {
    static PerDevice limit;
    const cudaError_t e = raise_smem(limit, k_step1d_ring<NV, NS, LIM>, ring1d_smem<NV, NS>());
    if (e != cudaSuccess) return e;
    k_step1d_ring<NV, NS, LIM><<<grid, TW1, ring1d_smem<NV, NS>(), s>>>(a, kstep);
    return cudaGetLastError();
}

template <int NV, int NS>
cudaError_t launch_ring(int grid, const Step1DArgs& a, int kstep, cudaStream_t s) {
    if (a.scheme == LAT_SCHEME_KOREN) return launch_ring_t<NV, NS, true>(grid, a, kstep, s);
    return launch_ring_t<NV, NS, false>(grid, a, kstep, s);
}

template <int NV, int NS>
int occupancy_ring() {
    int nb = 0;
    cudaFuncSetAttribute(k_step1d_ring<NV, NS, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)ring1d_smem<NV, NS>());
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_step1d_ring<NV, NS, false>, TW1,
                                                  ring1d_smem<NV, NS>());
    return nb;
}

template <typename T, int NV>
cudaError_t launch_reg(int block, int grid, const Step1DArgs& a, int kstep, cudaStream_t s) {
    if (block > MaxThreads<T, NV>::value) return cudaErrorInvalidValue;
    if (a.scheme == LAT_SCHEME_KOREN) k_step1d_reg<T, NV, true><<<grid, block, 0, s>>>(a, kstep);
    else k_step1d_reg<T, NV, false><<<grid, block, 0, s>>>(a, kstep);
    return cudaGetLastError();
}

#define LAT1D_NV_LIST(X) X(3) X(5) X(9) X(17) X(33) X(65)


template <typename T>
cudaError_t launch_plain(int nv, int block, int grid, const Step1DArgs& a, int kstep,
                         cudaStream_t s) {
    switch (nv) {
#define X(n) \
    case n: return launch_reg<T, n>(block, grid, a, kstep, s);
        LAT1D_NV_LIST(X)
#undef X
        default:
            if (block > 512) return cudaErrorInvalidValue;
            k_step1d_any<T><<<grid, block, 0, s>>>(a, kstep, nv);
            return cudaGetLastError();
    }
}

}  // namespace

int step1d_max_block(int dtype, int nv, int variant) {
    if (variant == STEP1D_RING || variant == STEP1D_PC) return TW1;
    bool reg = false;
#define X(n) reg |= nv == n;
    LAT1D_NV_LIST(X)
#undef X
    if (!reg) return 512;
    const int words = nv * (dtype == LAT_F64 ? 2 : 1);
    return words > 56 ? 256 : (words > 20 ? 512 : 1024);
}

// The limited scheme runs in the compiled-N_v kernels only (not k_step1d_any).
bool step1d_limiter_supported(int nv) {
    switch (nv) {
#define X(n) case n:
        LAT1D_NV_LIST(X)
#undef X
        return true;
        default: return false;
    }
}

bool step1d_ring_supported(int dtype, int nv) {
    if (dtype != LAT_F32) return false;
    bool ok = false;
#define X(n) ok |= nv == n;
    LAT1D_NV_LIST(X)
#undef X
    return ok;
}

int step1d_ring_tile() { return TW1; }
int step1d_ring_min_nx() { return WIN1; }

int step1d_ring_occupancy(int nv, int slots, int variant) {
    switch (nv) {
#define X(n)                                                                    \
    case n:                                                                     \
        if (variant == STEP1D_PC) {                                             \
            if (slots == 2) return occupancy_pc1<n, 2>();                       \
            if (slots == 3) return occupancy_pc1<n, 3>();                       \
            return occupancy_pc1<n, 4>();                                       \
        }                                                                       \
        if (slots == 2) return occupancy_ring<n, 2>();                          \
        if (slots == 3) return occupancy_ring<n, 3>();                          \
        return occupancy_ring<n, 4>();
        LAT1D_NV_LIST(X)
#undef X
        default: return 0;
    }
}

// the fused epilogue reduces in the two-lane order of ColumnSums2 (N_v >= 5)
bool step1d_moments_supported(int dtype, int nv) {
    return nv >= 5 && step1d_ring_supported(dtype, nv);
}

cudaError_t launch_step1d_moments(int nv, int grid, const Step1DArgs& a, cudaStream_t s) {
    if (grid <= 0) return cudaSuccess;
    switch (nv) {
#define X(n) \
    case n: return launch_pc1<n, 2, true>(grid, a, 0, s);
        LAT1D_NV_LIST(X)
#undef X
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_step1d(int dtype, int nv, int variant, int block, int slots, int grid,
                          const Step1DArgs& a, int kstep, cudaStream_t s) {
    if (grid <= 0) return cudaSuccess;
    if (variant == STEP1D_PC) {
        if (dtype != LAT_F32 || block != TW1) return cudaErrorInvalidValue;
        switch (nv) {
#define X(n)                                                         \
    case n:                                                          \
        if (slots == 2) return launch_pc1<n, 2>(grid, a, kstep, s);  \
        if (slots == 3) return launch_pc1<n, 3>(grid, a, kstep, s);  \
        if (slots == 4) return launch_pc1<n, 4>(grid, a, kstep, s);  \
        return cudaErrorInvalidValue;
            LAT1D_NV_LIST(X)
#undef X
            default: return cudaErrorInvalidValue;
        }
    }
    if (variant == STEP1D_RING) {
        if (dtype != LAT_F32 || block != TW1) return cudaErrorInvalidValue;
        switch (nv) {
#define X(n)                                                         \
    case n:                                                          \
        if (slots == 2) return launch_ring<n, 2>(grid, a, kstep, s); \
        if (slots == 3) return launch_ring<n, 3>(grid, a, kstep, s); \
        if (slots == 4) return launch_ring<n, 4>(grid, a, kstep, s); \
        return cudaErrorInvalidValue;
            LAT1D_NV_LIST(X)
#undef X
            default: return cudaErrorInvalidValue;
        }
    }
    if (dtype == LAT_F32) return launch_plain<float>(nv, block, grid, a, kstep, s);
    if (dtype == LAT_F64) return launch_plain<double>(nv, block, grid, a, kstep, s);
    return cudaErrorInvalidValue;
}

cudaError_t launch_flow_basis(int dtype, const Step1DArgs& a, const int* sizes, int n_sizes,
                              int nx_max, void* table, cudaStream_t s) {
    const dim3 grid((a.nmodes * nx_max + 255) / 256, std::min(n_sizes, 65535));
    if (dtype == LAT_F64)
        k_flow_basis<double><<<grid, 256, 0, s>>>(a, sizes, n_sizes, static_cast<double2*>(table));
    else
        k_flow_basis<float><<<grid, 256, 0, s>>>(a, sizes, n_sizes, static_cast<float2*>(table));
    return cudaGetLastError();
}

cudaError_t launch_advance_step(DevState* st, long long n, cudaStream_t s) {
    k_advance_step<<<1, 1, 0, s>>>(st, n);
    return cudaGetLastError();
}

}  // namespace lat
