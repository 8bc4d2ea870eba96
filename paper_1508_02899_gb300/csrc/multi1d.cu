// Several time steps of 1D lattices in one launch, with the tile's state held in shared memory
// between them (FP32, upwind drag).
//
// A step reads and writes every cell once, so one launch per step is bound by HBM.  Here a block
// takes a tile of w columns of one instance through T steps on chip: one read and one write of
// the state per T steps.
//
// The tile follows the characteristics.  A value of plane j keeps its place in shared memory while
// the streaming moves it by j columns per step: place i of plane j holds the value whose column
// after the T steps is X = x0 - m + i (x0 the tile's first column, m a margin).  Before step s
// (d = T - 1 - s steps follow it) column x therefore finds plane j's streamed value at place
// x - (x0 - m) + j d.  Each place is read and written by one thread per step, so the update is in
// place and a step ends with one block barrier; the streaming moves no data.
//
// The window of P = w + 2 m places is closed to a ring: column c takes the places (c + j d) mod P.
// A column that wraps is made of two columns P apart, each with its own flow velocity; where they
// meet, cells see wrong neighbours.  One step couples velocities at most kReach apart (drag one,
// diffusion one), so wrong values reach places within sum_d kReach d = kReach T (T - 1) / 2 of the
// window's edges, which the margin m covers: they never reach the tile's w columns.  Every column
// has the full N_v cells, whatever T: the redundant work is 2 m / w, not the 2 J (T - 1) / w of a
// rectangular halo.
//
// T is odd: absolute step s reads f[s & 1] and writes f[(s + 1) & 1], and with T odd the launch
// reads one buffer and writes the other, so tiles do not race on the columns they share.
// Every operation and its order are those of the one-step kernels: the same bits.
//
// Measured (4096 instances, N_x 1024 .. 8192, N_v = 65, 20 steps, moments and noise upload
// included): 14.0 ms against 26.5 ms for one launch per step; per step 0.58 ms, its flow 0.07.  DRAM
// traffic falls from 8 to 1.6 bytes per cell and step; what bounds the kernel now is instruction issue
// and latency within a step (six warps per block, two blocks per SM).  Tried and slower, when the
// kernel took its step count at run time (15.2 ms): one column per thread as two
// half-columns (17.3 to 17.7 ms, with the sweeps unrolled whole 19 to 20 ms: instruction cache), T = 3
// (18.2 ms), one block per SM with twice the columns (16.7 ms before the flow had its own kernel;
// 17.4 ms with two), waits on the neighbouring warps in place of the block barrier (18.9 ms),
// evaluating the flow in this kernel (18.2 ms).
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "lat_internal.h"
#include "per_device.h"
#include "step1d_dev.h"

namespace lat {
namespace {

using namespace k1d;

constexpr int kReach = 2;   // velocities one step couples
constexpr int kCols = 64;   // columns of a warp: lane l takes c0 + l and c0 + 32 + l
constexpr int kChunk = 8;   // velocity rows per pass of the sweep's loop
constexpr int kSmemWords = 113 * 1024 / 4;
constexpr int kMaxPlaces = 512;
constexpr int T = kFlowSteps;  // steps per launch
static_assert(T % 4 == 1, "odd: from one buffer to the other; and the shifts of Shape");
constexpr int round_up(int v, int n) { return (v + n - 1) / n * n; }
constexpr int kMargin = round_up(kReach * T * (T - 1) / 2, 4);
// Words besides the planes: the copies' mbarrier and u / dv of every step's columns.
constexpr int side_words(int J, int P) { return 4 + T * P + J * T * (T - 1); }

// Shape of the kernel for N_v.  Two blocks per SM (one loads while the other computes), so at most
// about 113 KB each.
template <int NV>
struct Shape {
    static constexpr int J = (NV - 1) / 2;
    static constexpr int kFit = (kSmemWords - 4 * NV - side_words(J, 0)) / (NV + T) / kCols * kCols;
    static constexpr int kPitch = (kFit < kMaxPlaces ? kFit : kMaxPlaces) + 4;
    static_assert((NV - 1) % kChunk == 0 && J % 4 == 0, "whole chunks, one pattern of shifts");
    // offset of plane row jj's window in its row: the 16-byte rounding of column x0 - m - j T
    // (T = 1 modulo 4)
    __host__ __device__ static constexpr int shift(int jj) { return (J - jj) & 3; }
    static constexpr int kPlaces = kPitch - 4;  // of a tile at most
    static_assert(NV * kPitch + side_words(J, kPlaces) <= kSmemWords, "two blocks per SM");
};

// ---- the sweep of two columns ------------------------------------------------------------------
// A thread sweeps the velocity columns c and c + 32 in the two lanes of f32x2 pairs, the operations
// and their order those of sweep_column.  Rows come in chunks, and a chunk takes one of the bodies
// below by two tests that are uniform over the warp:
//  * MIXED: some columns' places wrap within the chunk (else one pointer serves both columns);
//  * the sign of c a = g (w - j) over the chunk's rows and the warp's columns.  Where it is one
//    sign, one term of the upwind flux (c a_j)^+ f_j + (c a_{j+1})^- f_{j+1} is zero: it is not
//    formed, nor the minima and maxima (5 of 20 instructions per row).  A velocity that is not a
//    number has no sign: the minima and maxima make both its parts zero.
// A product that an addition uses is formed as an fma with an opaque zero: the packed product
// itself would be contracted into the addition (other bits).
enum { kBoth = 0, kPos = 1, kNeg = 2 };

struct Sweep2 {
    f2 s, cac, Fp, dp, Dp, kk;
    f2 g2, r2, one2, zero2;
};

// Where the columns' places wrap.  A warp's columns all wrap at the start of the ring (rows below
// ea, from places P on) or all at its end (rows from ea on, to places P back), never both
// (P >= 2 J (T - 1) + kCols): going up the rows, a column loses P once.
struct Wrap {
    int ea, eb;      // rows from which columns c and c + 32 have lost P
    float wa, wb;    // u / dv of those rows
};

// Outputs back to their places, or (last step) to the other buffer: dst is the next row's cell of
// column c.  on0, on1: whether each column is stored.
template <bool GLOBAL>
struct Put {
    float* dst;
    int nx;
    bool on0, on1;
    __device__ __forceinline__ void operator()(float* qa, float* qb, f2 o) {
        if constexpr (GLOBAL) {
            if (on0) dst[0] = lo(o);
            if (on1) dst[32] = hi(o);
            dst += nx;
        } else {
            *qa = lo(o);
            *qb = hi(o);
        }
    }
};

// Rows of one chunk: faces k + 1/2, k = 0 .. kChunk - 1, and the outputs of rows k - 1.  qa, qb: the
// places of the two columns' row 0 (without their shift), moved on to the next chunk's; w2 their
// flow velocities.  MIXED: some columns lose P in the chunk (va, vb the places of row -1).
template <int NV, bool MIXED, int SIGN, class P>
__device__ __forceinline__ void chunk(Sweep2& z, float*& qa, float*& qb, float*& va, float*& vb,
                                      f2& w2, int step, int up, const Wrap& wr, int row,
                                      bool first, P& put) {
    using S = Shape<NV>;
    float *pa[kChunk + 2], *pb[kChunk + 2];  // rows -1 .. kChunk
    pa[0] = va;
    pb[0] = vb;
    pa[1] = qa;
    pb[1] = qb;
    // every load of the chunk before its stores (the compiler cannot tell their places apart)
    f2 next[kChunk], wn[kChunk];
#pragma unroll
    for (int k = 0; k < kChunk; ++k) {
        pa[k + 2] = pa[k + 1] + step;
        if (MIXED) {
            pb[k + 2] = pb[k + 1] + step;
            float wl = lo(w2), wh = hi(w2);
            if (row + k + 1 == wr.ea) {
                pa[k + 2] -= up;
                wl = wr.wa;
            }
            if (row + k + 1 == wr.eb) {
                pb[k + 2] -= up;
                wh = wr.wb;
            }
            w2 = pk(wl, wh);
        } else {
            pb[k + 2] = pa[k + 2] + 32;
        }
        wn[k] = w2;
        next[k] = pk(pa[k + 2][S::shift(k + 1)], pb[k + 2][S::shift(k + 1)]);
    }
#pragma unroll
    for (int k = 0; k < kChunk; ++k) {
        const f2 kn = add2(z.kk, z.one2);
        const f2 can = mul2(z.g2, sub2(wn[k], kn));
        const f2 sn = next[k];
        f2 Fn;
        if (SIGN == kPos) Fn = fma2(z.cac, z.s, z.zero2);
        else if (SIGN == kNeg) Fn = fma2(can, sn, z.zero2);
        else Fn = fma2(max0(z.cac), z.s, mul2(min0(can), sn));
        const f2 d = sub2(z.s, sub2(Fn, z.Fp));
        z.Fp = Fn;
        f2 D = fma2(z.r2, sub2(d, z.dp), z.zero2);
        if (k == 0 && first) D = 0ull;  // no face below cell 0
        else put(pa[k] + S::shift(k - 1), pb[k] + S::shift(k - 1), add2(z.dp, sub2(D, z.Dp)));
        z.Dp = D;
        z.dp = d;
        z.s = sn;
        z.cac = can;
        z.kk = kn;
    }
    va = pa[kChunk];
    vb = pb[kChunk];
    qa = pa[kChunk + 1];
    qb = pb[kChunk + 1];
}

template <int NV, bool MIXED, class P>
__device__ __forceinline__ void chunk_sign(int sign, Sweep2& z, float*& qa, float*& qb, float*& va,
                                           float*& vb, f2& w2, int step, int up, const Wrap& wr,
                                           int row, bool first, P& put) {
    if (sign == kPos) chunk<NV, MIXED, kPos>(z, qa, qb, va, vb, w2, step, up, wr, row, first, put);
    else if (sign == kNeg) chunk<NV, MIXED, kNeg>(z, qa, qb, va, vb, w2, step, up, wr, row, first, put);
    else chunk<NV, MIXED, kBoth>(z, qa, qb, va, vb, w2, step, up, wr, row, first, put);
}

// One step of the columns c0 + lane and c0 + 32 + lane (d steps follow it); U[k] = u / dv of
// column k.  RING: places may wrap.
template <int NV, bool RING, bool GLOBAL>
__device__ __forceinline__ void sweep2(float* f, const float* U, int c0, int d, int P, float g,
                                       float r, Put<GLOBAL> put) {
    using S = Shape<NV>;
    constexpr int J = S::J;
    const int c = c0 + (threadIdx.x & 31), step = S::kPitch + d;
    float *qa = f + c - J * d, *qb = qa + 32;
    float ua = U[c], ub = U[c + 32];
    float wlo = min_nan(ua, ub), whi = max_nan(ua, ub);
    Wrap wr{NV + 1, NV + 1, 0.f, 0.f};
    int ma = NV + 1, mb = NV + 1;  // rows from which, and up to which, some columns lose P
    if constexpr (RING) {
        if (c0 >= J * d && c0 + kCols + J * d <= P) {
            // no place wraps
        } else if (c0 < J * d) {  // wraps at the start: begin P up, with the flow of columns c + P
            wr.ea = max(0, J - c / d);
            wr.eb = max(0, J - (c + 32) / d);
            wr.wa = ua;
            wr.wb = ub;
            if (wr.ea > 0) {
                qa += P;
                ua = U[c + P];
            }
            if (wr.eb > 0) {
                qb += P;
                ub = U[c + 32 + P];
            }
        } else {
            wr.ea = J + (P - c + d - 1) / d;
            wr.eb = J + (P - c - 32 + d - 1) / d;
            wr.wa = wr.ea < NV ? U[c - P] : ua;
            wr.wb = wr.eb < NV ? U[c + 32 - P] : ub;
        }
        ma = __reduce_min_sync(0xffffffffu, min(wr.ea, wr.eb));
        mb = __reduce_max_sync(0xffffffffu, max(wr.ea, wr.eb));
        if (ma <= NV) {
            wlo = min_nan(min_nan(wlo, min_nan(ua, ub)), min_nan(wr.wa, wr.wb));
            whi = max_nan(max_nan(whi, max_nan(ua, ub)), max_nan(wr.wa, wr.wb));
        }
    }
    // rows up to kp have c a >= 0 in every column of the warp, rows from kn on c a <= 0
    const bool sane = fabsf(wlo) < 1e6f && fabsf(whi) < 1e6f;  // false for NaN
    const int kp = __reduce_min_sync(0xffffffffu, sane ? (int)floorf(wlo) + J : -1);
    const int kn = __reduce_max_sync(0xffffffffu, sane ? (int)ceilf(whi) + J : NV);
    f2 w2 = pk(ua, ub);
    Sweep2 z;
    z.g2 = pk(g, g);
    z.r2 = pk(r, r);
    z.one2 = opaque2(pk(1.f, 1.f));
    z.zero2 = opaque2(0ull);
    z.kk = opaque2(pk(float(-J), float(-J)));
    z.Fp = z.dp = z.Dp = 0ull;
    z.cac = mul2(z.g2, sub2(w2, z.kk));
    z.s = pk(qa[S::shift(0)], qb[S::shift(0)]);
    float *va = qa, *vb = qb;
#pragma unroll 1
    for (int q = 0; q < NV - 1; q += kChunk) {
        const int sign = q + kChunk <= kp ? kPos : (q >= kn ? kNeg : kBoth);
        // rows q - 1 .. q + kChunk: with one offset in every column, one pointer serves both
        if (!RING || (q == 0 ? ma <= 0 && mb <= 0 : mb < q) || ma > q + kChunk) {
            chunk_sign<NV, false>(sign, z, qa, qb, va, vb, w2, step, 0, wr, 0, q == 0, put);
        } else {
            chunk_sign<NV, true>(sign, z, qa, qb, va, vb, w2, step, P, wr, q, q == 0, put);
        }
    }
    // the last cell: no flux through the wall
    const f2 dl = sub2(z.s, sub2(0ull, z.Fp));
    const f2 D = fma2(z.r2, sub2(dl, z.dp), z.zero2);
    put(va + S::shift(-1), vb + S::shift(-1), add2(z.dp, sub2(D, z.Dp)));
    put(qa + S::shift(0), qb + S::shift(0), add2(dl, sub2(0ull, D)));
}

__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src)
                 : "memory");
}

template <int NV>
__global__ void __launch_bounds__(kMaxPlaces / 2, 2)
    k_multi1d(const Step1DArgs a, const MultiTile* tiles, int kstep, int piped) {
    using S = Shape<NV>;
    constexpr int J = S::J, PT = S::kPitch;
    extern __shared__ __align__(128) unsigned char smem[];
    float* f = reinterpret_cast<float*>(smem);
    float* U = f + (size_t)NV * PT;  // rows of P + 2 J d: the columns -J d .. P + J d - 1 of a step
    uint64_t* bar = reinterpret_cast<uint64_t*>(U + T * 2 * blockDim.x + J * T * (T - 1));
    const MultiTile tile = tiles[blockIdx.x];
    const int nx = tile.nx, P = 2 * blockDim.x, first = tile.x0 - kMargin;
    const long long step = a.st->step + kstep;
    const int par = (int)(step & 1);
    const float* fin = static_cast<const float*>(par ? a.f[1] : a.f[0]) + tile.off;
    float* fout = static_cast<float*>(par ? a.f[0] : a.f[1]) + tile.off;
    const float* w_in = static_cast<const float*>(a.wflow) + tile.xoff;
    const int tid = threadIdx.x;
    if (tid == 0) mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
    if (piped) {
        // N_x and every tile's first column are multiples of 4: plane windows by bulk copies
        if (!a.st->stall) {  // a stalled context issues no copies
            if (tid == 0)
                mbar_expect_tx(bar, (unsigned)((NV * (P + 4) + T * P + J * T * (T - 1)) *
                                               sizeof(float)));
            for (int q = tid; q < NV + T; q += blockDim.x) {
                const int jj = q < NV ? q : 0, s = q - NV, e = J * (T - 1 - s);
                float* dst = q < NV ? f + jj * PT : U + s * P + J * s * (2 * T - 1 - s);
                const float* row = q < NV ? fin + (size_t)jj * nx : w_in + s * a.total_x;
                const int len = q < NV ? P + 4 : P + 2 * e;
                int b = (q < NV ? first - (jj - J) * T - S::shift(jj) : first - e) % nx;
                b += b < 0 ? nx : 0;
                for (int k = 0; k < len;) {
                    const int n = min(len - k, nx - b);
                    bulk_g2s(dst + k, row + b, (unsigned)(n * sizeof(float)), bar);
                    k += n;
                    b = 0;
                }
            }
        }
    } else {
        const int dx = T % nx;
        for (int c = tid; c < P; c += blockDim.x) {
            int x = (first + c + J * T) % nx;
            x += x < 0 ? nx : 0;
            const float* row = fin;
#pragma unroll 4
            for (int jj = 0; jj < NV; ++jj) {
                cp_async4(f + jj * PT + S::shift(jj) + c, row + x);
                row += nx;
                x -= dx;
                x += x < 0 ? nx : 0;
            }
        }
        for (int s = 0; s < T; ++s) {
            const int e = J * (T - 1 - s);
            float* dst = U + s * P + J * s * (2 * T - 1 - s);
            for (int c = tid; c < P + 2 * e; c += blockDim.x) {
                int x = (first - e + c) % nx;
                x += x < 0 ? nx : 0;
                cp_async4(dst + c, w_in + s * a.total_x + x);
            }
        }
    }
    __syncwarp();  // lanes that wait early would hold back those that still issue copies
    bool failed = false;
    if (piped) failed = !mbar_wait_bounded(bar, 0u);
    else asm volatile("cp.async.wait_all;" ::: "memory");
    if (__syncthreads_or(failed ? 1 : 0)) {
        if (tid == 0) atomicOr(&a.st->status, ST_TIMEOUT);
        return;
    }
    // all steps but the last, in place
    const float* Us = U;
    const int c0 = (tid >> 5) * kCols;
#pragma unroll 1
    for (int d = T - 1; d > 0; --d) {
        Us += J * d;
        const Put<false> put{nullptr, 0, true, true};
        sweep2<NV, true>(f, Us, c0, d, P, tile.g, tile.r, put);
        Us += P + J * d;
        __syncthreads();
    }
    // the last step: every place is its column, and the outputs go to the other buffer
    const int c = c0 + (tid & 31) - kMargin;
    sweep2<NV, false>(f, Us, c0, 0, P, tile.g, tile.r,
                      Put<true>{fout + tile.x0 + c, nx, c >= 0 && c < tile.w,
                                c + 32 >= 0 && c + 32 < tile.w});
}

// u / dv of every column at the n <= T steps, W[step][column], one block per tile of columns; the
// instance's first tile also advances the amplitudes to the step after them.  The basis comes from
// tables (one per grid size, flow_basis's values): evaluated per column and step, as the one-step
// kernels do, the eight sincospi would cost as much as a fifth of the sweeps.
template <typename F> struct Pair;
template <> struct Pair<float> { using type = float2; };
template <> struct Pair<double> { using type = double2; };

template <typename F>
__global__ void __launch_bounds__(256) k_flow_steps(const Step1DArgs a, int kstep, int n) {
    using F2 = typename Pair<F>::type;
    extern __shared__ double2 amp_raw[];
    F* amp = reinterpret_cast<F*>(amp_raw);  // [M][T][A, B]
    const int2 item = a.items[blockIdx.x];
    const Inst1D& in = a.inst[item.x];
    const int nx = in.nx, tid = threadIdx.x;
    const long long step = a.st->step + kstep;
    const int par = (int)(step & 1);
    const int M = a.flow_kind == LAT_FLOW_MODES ? a.nmodes : 0;
    if (tid < 2 * M) {
        const long long at = (long long)item.x * 2 * M + tid;
        double v = a.amp[par * a.amp_stride + at];
        F* row_q = amp + (tid < M ? tid : tid - M) * 2 * T + (tid < M ? 0 : 1);
        const long long row0 = step - a.st->noise_base, rows = a.st->noise_rows;
        const double e = in.ou_e, sg = in.ou_s;
        bool missing = false;
        double xi[T];
#pragma unroll
        for (int s = 0; s < T; ++s) {
            const long long row = row0 + s;
            const bool have = !a.frozen && s < n && row >= 0 && row < rows;
            missing |= !have && s < n;
            xi[s] = have ? a.noise[row * a.amp_stride + at] : 0.0;
        }
#pragma unroll
        for (int s = 0; s < T; ++s) {
            row_q[2 * s] = F(v);
            if (!a.frozen && s < n) v = __dadd_rn(__dmul_rn(v, e), __dmul_rn(sg, xi[s]));
        }
        if (!a.frozen && item.y == 0) {
            a.amp_w[(1 - par) * a.amp_stride + at] = v;
            a.ampf_w[(1 - par) * a.amp_stride + at] = (float)v;
            if (missing && tid == 0) atomicOr(&a.st->status, ST_NOISE);
        }
    }
    __syncthreads();
    const F inv_dv = F(in.inv_dv), g = F(in.g);
    const F J = F((a.nv - 1) / 2);
    const F cf = a.scheme == LAT_SCHEME_KOREN ? F(1) + F(a.mu) : F(1);  // Eq. (cfl) of the scheme
    bool cfl = false;
    for (int x = item.y + tid; x < min(nx, item.y + a.tile); x += blockDim.x) {
        const F2* basis = static_cast<const F2*>(a.basis) + M * a.size_off[item.x] + x;
        F* w = static_cast<F*>(a.wflow) + in.xoff + x;
        F u[T];
        const F v =
            a.flow_kind == LAT_FLOW_FIELD ? static_cast<const F*>(a.field)[in.xoff + x] : F(0);
#pragma unroll
        for (int s = 0; s < T; ++s) u[s] = v;
#pragma unroll 8
        for (int m = 0; m < M; ++m) {
            const F2 sc = __ldg(basis + (size_t)m * nx);
            const F2* ab = reinterpret_cast<const F2*>(amp + m * 2 * T);
#pragma unroll
            for (int s = 0; s < T; ++s) u[s] = flow_add<F>(u[s], ab[s].x, ab[s].y, sc.x, sc.y);
        }
#pragma unroll
        for (int s = 0; s < T; ++s) {
            if (s >= n) break;
            const F ws = u[s] * inv_dv;
            w[s * a.total_x] = ws;
            cfl |= cf * (g * (J + fabs(ws))) > F(1);
        }
    }
    if (cfl) atomicOr(&a.st->status, ST_CFL);
}

template <int NV>
cudaError_t launch_t(int ntiles, int places, const Step1DArgs& a, const MultiTile* tiles, int kstep,
                     int piped, cudaStream_t s) {
    static PerDevice limit;
    cudaError_t e = raise_smem(limit, k_multi1d<NV>, 4 * kSmemWords);
    if (e != cudaSuccess) return e;
    e = launch_flow_steps(LAT_F32, a, kstep, T, s);
    if (e != cudaSuccess) return e;
    const size_t smem = 4 * ((size_t)NV * Shape<NV>::kPitch + side_words(Shape<NV>::J, places));
    k_multi1d<NV><<<ntiles, places / 2, smem, s>>>(a, tiles, kstep, piped);
    return cudaGetLastError();
}

#define MULTI_NV_LIST(X) X(9) X(17) X(33) X(65)

}  // namespace

cudaError_t launch_flow_steps(int dtype, const Step1DArgs& a, int kstep, int n, cudaStream_t s) {
    const int M = a.flow_kind == LAT_FLOW_MODES ? a.nmodes : 0;
    const int words = 2 * M * T, threads = std::min(256, a.tile);
    if (dtype == LAT_F64)
        k_flow_steps<double><<<a.item_end, threads, sizeof(double) * words, s>>>(a, kstep, n);
    else k_flow_steps<float><<<a.item_end, threads, sizeof(float) * words, s>>>(a, kstep, n);
    return cudaGetLastError();
}

bool multi1d_shape(int nv, int* max_places, int* margin) {
    *margin = kMargin;
    switch (nv) {
#define X(n)     case n: *max_places = Shape<n>::kPlaces; return true;
        MULTI_NV_LIST(X)
#undef X
        default: return false;
    }
}

int multi1d_places(int nv, int w) {
    return round_up(std::max(w + 2 * kMargin, (nv - 1) * (T - 1) + kCols), kCols);
}

cudaError_t launch_multi1d(int nv, int ntiles, int places, const Step1DArgs& a,
                           const MultiTile* tiles, int kstep, int piped, cudaStream_t s) {
    switch (nv) {
#define X(n)     case n: return launch_t<n>(ntiles, places, a, tiles, kstep, piped, s);
        MULTI_NV_LIST(X)
#undef X
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace lat
