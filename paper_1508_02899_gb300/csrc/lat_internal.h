// Internal declarations shared by the library's translation units (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <list>
#include <map>
#include <vector>

#include "../../include/lat.h"

// The bulk-copy rings refill a shared-memory slot only after a block barrier that follows every
// thread's last read of it; build with -DLAT_RING_PROXY_FENCE=1 to also issue a generic-to-async
// proxy fence before each refill.
#ifndef LAT_RING_PROXY_FENCE
#define LAT_RING_PROXY_FENCE 0
#endif

namespace lat {

// Host arrays into device tables that kernels of a context's stream read, without waiting.  Always on
// that stream: a copy from pageable memory on the default stream may return before its last transfer is
// done, and a non-blocking stream (such as PyTorch's) does not wait for that one.  The arrays are copied
// here and held, as the transfers may read them later: at most kHeld bytes and the latest array,
// then the stream is waited for.  lat_free does before it lets them go.
class Uploads {
    static constexpr size_t kHeld = 16u << 20;
    std::list<std::vector<char>> held_;
    size_t bytes_ = 0;

public:
    cudaError_t copy(void* dst, const void* src, size_t bytes, cudaStream_t s) {
        if (bytes_ + bytes > kHeld && !held_.empty()) {
            const cudaError_t e = cudaStreamSynchronize(s);
            if (e != cudaSuccess) return e;
            held_.clear();
            bytes_ = 0;
        }
        const char* p = static_cast<const char*>(src);
        held_.emplace_back(p, p + bytes);
        bytes_ += bytes;
        return cudaMemcpyAsync(dst, held_.back().data(), bytes, cudaMemcpyHostToDevice, s);
    }
};

// Device status bits; translated to LAT_E* codes by the host.
enum : unsigned {
    ST_CFL = 1u,       // Eq. (cfl) violated by the evolving flow
    ST_NUMERIC = 2u,   // non-finite value in f
    ST_NOISE = 4u,     // noise table exhausted
    ST_OVERFLOW = 8u,  // reduced-precision scale overflow
    ST_TIMEOUT = 16u,  // a bounded wait gave up
};

// Device-resident step counter and status word of one context.
struct DevState {
    long long step;        // steps taken
    long long noise_base;  // step at which noise row 0 applies
    long long noise_rows;  // rows in the noise table
    unsigned status;
    unsigned stall;        // != 0: the bulk-copy producers issue nothing (lat_debug_stall)
};

// One 1D lattice instance as the kernels see it.
struct Inst1D {
    long long off;    // element offset of f[0][0] in the ensemble buffer
    long long xoff;   // offset of this instance's cells in per-cell arrays (sum of earlier nx)
    int nx;
    int pow2;         // 1 if nx is a power of two
    double g;         // dt / tau_p
    double inv_dv;    // 1 / dv
    double dv;
    double dx;
    double r;         // kappa dt / dv^2
    double ou_e;      // e^{-dt/tau_f}
    double ou_s;      // sigma sqrt(1 - e^2)
    double two_over_nx;
    double dt;
};

// Step kernel variants (1D).
enum { STEP1D_PLAIN = 0, STEP1D_RING = 1, STEP1D_PC = 2 };

constexpr int kMaxModes1D = 16;
constexpr int kMaxModes2D = 512;

// Arguments of the 1D step kernels.
struct Step1DArgs {
    void* f[2];              // ping-pong buffers: absolute step s reads f[s & 1], writes the other
    const Inst1D* inst;
    const int2* items;       // (instance, first x) of each tile
    int item_begin, item_end;
    int flow_kind;           // LAT_FLOW_*
    int nmodes;
    int k[kMaxModes1D];
    const double* amp;       // [2][n_inst][2M] parity-indexed amplitudes
    double* amp_w;           // same buffer, written (other parity)
    const float* ampf;       // FP32 copy of amp read by the FP32 kernels
    float* ampf_w;
    long long amp_stride;    // n_inst * 2M
    const double* noise;     // [rows][n_inst][2M]
    const void* field;       // FIELD flow, per-cell array over all instances
    // several steps per launch (multi1d.cu)
    const void* basis;           // (sin, cos) tables of the modes, one per grid size
    const long long* size_off;   // [n_inst] columns of the tables before the instance's
    void* wflow;                 // [kFlowSteps][total_x] u / dv of the steps
    const void* wpre;            // u / dv of this step's columns (a row of wflow), or null
    long long total_x;
    int nv, tile;                // N_v; columns per item
    DevState* st;
    int dry;                 // 1: do not advance the flow (autotuning)
    int frozen;              // 1: flow frozen (tau_f infinite)
    int scheme;              // LAT_SCHEME_UPWIND or LAT_SCHEME_KOREN (drag sub-step)
    double mu;               // limiter bound psi(theta) <= mu theta (KOREN)
    // moments of the new state, fused into the step (k_step1d_pc with moments); may be null
    double* m_rho;
    double* m_mv;
    double* m_mv2;
    double* m_partials;      // [item][consumer warp][M, P, E][sum, compensation]
};

constexpr int kPcConsumerWarps = 4;

// One tile of the several-steps kernel (multi1d.cu): columns x0 .. x0 + w - 1 of an instance, with
// what the tile needs of the instance's parameters.
struct MultiTile {
    long long off;           // Inst1D::off
    long long xoff;          // Inst1D::xoff
    int nx, x0, w;
    float g, r;
};
// Steps of a launch of the several-steps kernel, and of the flow kernel at most.
constexpr int kFlowSteps = 5;
// For the N_v the several-steps kernel is built for: the places a tile may take with its margins
// (w + 2 margin <= max_places); false where there is no kernel.
bool multi1d_shape(int nv, int* max_places, int* margin);
// One flux-limited step of every tile (lim1d.cu, FP32): columns of a tile at most, places (threads x 2)
// of a tile of w columns; wrow the step's row of wflow.
bool lim1d_shape(int nv, int* max_places);
int lim1d_places(int w);
cudaError_t launch_lim1d(int nv, int ntiles, int places, const Step1DArgs& a, const MultiTile* tiles,
                         int kstep, const float* wrow, int piped, cudaStream_t s);
// Steps kstep .. kstep + n - 1 of small 1D lattices (upwind drag), one cluster per lattice with the
// state in shared memory throughout (line1d.cu).
// line1d_clusters: clusters that run at a time, 0 where there is no kernel; line1d_us: about how long n
// steps take.
int line1d_clusters(int dtype, int n_inst, int nx_max, int nv, int nmodes);
double line1d_us(int dtype, int n_inst, int nx_max, int nv, int nmodes, int clusters, int n);
cudaError_t launch_line1d(int dtype, int n_inst, int nx_max, int nv, const Step1DArgs& a, int kstep,
                          int n, cudaStream_t s);
// Tables of the flow's basis, one per grid size (sizes: an instance of each; nx_max the largest):
// (sin, cos) of 2 pi k_m x / N_x, [m][x], from entry M size_off on.
cudaError_t launch_flow_basis(int dtype, const Step1DArgs& a, const int* sizes, int n_sizes,
                              int nx_max, void* table, cudaStream_t s);
// u / dv of steps kstep .. kstep + n - 1 into wflow (n <= kFlowSteps, odd: the amplitudes move to the
// step after them, in the parity that no block reads).  One block per item.
cudaError_t launch_flow_steps(int dtype, const Step1DArgs& a, int kstep, int n, cudaStream_t s);
// Places of a tile of w columns.
int multi1d_places(int nv, int w);
// Steps kstep .. kstep + kFlowSteps - 1 of every tile, each on `places` (the widest tile's).  piped: N_x and x0
// multiples of 4 throughout.
cudaError_t launch_multi1d(int nv, int ntiles, int places, const Step1DArgs& a,
                           const MultiTile* tiles, int kstep, int piped, cudaStream_t s);

// Arguments of the moment kernels (1D).
struct Mom1DArgs {
    const void* f;
    const Inst1D* inst;
    const int2* items;
    int nitems;
    int nv;
    double* rho;
    double* mean_v;
    double* mean_v2;
    double* partials;        // [nitems][3][2] (sum, compensation)
    DevState* st;
};

// Launchers (step1d.cu, moments.cu).
cudaError_t launch_step1d(int dtype, int nv, int variant, int block, int slots, int grid,
                          const Step1DArgs& a, int kstep, cudaStream_t s);
int step1d_max_block(int dtype, int nv, int variant);
bool step1d_ring_supported(int dtype, int nv);
bool step1d_limiter_supported(int nv);
int step1d_ring_tile();
int step1d_ring_min_nx();
int step1d_ring_occupancy(int nv, int slots, int variant);
// One producer/consumer step (2 slots) that also writes the moments of the new state.
cudaError_t launch_step1d_moments(int nv, int grid, const Step1DArgs& a, cudaStream_t s);
bool step1d_moments_supported(int dtype, int nv);
cudaError_t launch_moments1d(int dtype, int block, const Mom1DArgs& a, cudaStream_t s);
// Fold per-instance partials: instance i owns partials [per_item begin[i], per_item begin[i+1]).
// Observables (observables.cu): <rho_r^2> and the Eulerian S1 from per-cell rho (FP64).
cudaError_t launch_coarse1d(const double* rho, const Inst1D* inst, int n_inst, long long total_x,
                            const int* widths, int nw, double* P, double* out, int sm_count,
                            cudaStream_t s);
cudaError_t launch_coarse2d(const double* rho, int nx, int ny, double dx, const int* widths,
                            int nw, double* S, double* out, int sm_count, cudaStream_t s);
// part: s1_scratch() doubles.
size_t s1_scratch(int n_inst, long long total_x, int ns, int sm_count);
cudaError_t launch_s1_1d(int dtype, const void* f, const Inst1D* inst, int n_inst,
                         long long total_x, int nv, const double* rho, const int* seps, int ns,
                         double* part, double* num, double* den, int sm_count, cudaStream_t s);

// State I/O (state_io.cu): element conversions between FP64 and FP32 arrays of n values, and
// the device step counter, noise window and status of a restored checkpoint.
cudaError_t launch_f64_to_f32(const double* src, float* dst, long long n, cudaStream_t s);
cudaError_t launch_f32_to_f64(const float* src, double* dst, long long n, cudaStream_t s);
cudaError_t launch_set_devstate(DevState* st, long long step, long long noise_base,
                                long long noise_rows, cudaStream_t s);
cudaError_t launch_set_stall(DevState* st, unsigned on, cudaStream_t s);

// host != null (pinned memory, n_inst <= kFinDirect): the globals go there, and the status word to
// *host_status, cleared in *st.
constexpr int kFinDirect = 4;
cudaError_t launch_finalize1d(const double* partials, const int* inst_item_begin,
                              const Inst1D* inst, int n_inst, double* glob, int per_item,
                              DevState* st, double* host, unsigned* host_status, cudaStream_t s);
cudaError_t launch_advance_step(DevState* st, long long n, cudaStream_t s);

}  // namespace lat
