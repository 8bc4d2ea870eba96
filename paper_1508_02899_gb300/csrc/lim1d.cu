// One flux-limited time step of 1D lattices (scheme KOREN, FP32): two columns per thread in f32x2
// lanes, the tile's planes in shared memory.
//
// The limited sweep (step1d_dev.h, sweep_column_lim) is bound by instruction issue: 77 thread
// instructions per cell, most of them for the limited parts of the two Heun stages.  Here
//  * the arithmetic of two columns c and c + 32 runs in the lanes of one instruction;
//  * where c a has one sign over the rows at hand and the warp's columns, the part of the split flux
//    that is zero is not formed (rows go in chunks, the test is per chunk and uniform);
//  * the limiter takes min(dp, b, c) and max(dp, b, c) by three-input instructions (lim_min):
//    lim_inc's value up to the sign of a zero.
// The streaming is the place the tile's windows are copied from; the flow comes from k_flow_steps.
//
// Measured (1024 instances, N_x 1024 .. 8192, N_v = 65): 385 us per step at 5.4 TB/s, issue slots 57 %
// busy, 12 warps per SM (three tiles' planes fill the shared memory); one column per thread 945 us;
// ten steps, moments and globals 9.96 -> 4.37 ms.  Slower, where that was 4.65 ms: tiles of 128 columns,
// six per SM (4.77 ms); a barrier per eight rows, so that a sweep starts on its first ones (4.78 ms,
// 128 columns 4.93 ms).
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "lat_internal.h"
#include "per_device.h"
#include "step1d_dev.h"

namespace lat {
namespace {

using namespace k1d;

constexpr int kCols = 64;       // columns of a warp
constexpr int kChunk = 8;       // rows per pass of the loop
constexpr int kPlaces = 256;    // columns of a tile at most
constexpr int kPitch = kPlaces + 4;

struct LimConst : LimPair {
    f2 g2, r2, half2, one2;
};

enum { kBoth = 0, kPos = 1, kNeg = 2 };

// One Heun stage's split fluxes along the sweep, before row k is taken: P of rows k - 2 and k - 1 and
// the difference up to row k - 2, M of row k - 1 and the difference of rows k - 2 and k - 1.
struct Split {
    f2 P1, P2, dP, M2, dM;
};

// Takes row k (its c a and value v) and returns the flux through face k - 2 + 1/2, from P of rows
// k - 3 .. k - 1 and M of rows k - 2 .. k.
template <int SIGN>
__device__ __forceinline__ f2 face(Split& s, f2 ca, f2 v, const LimConst& k) {
    f2 F = 0ull;
    if (SIGN != kNeg) {
        const f2 d = sub2(s.P2, s.P1);
        F = add2(s.P1, lim_inc_x2(d, s.dP, k));
        s.P1 = s.P2;
        s.dP = d;
        s.P2 = fma2(SIGN == kPos ? ca : max0(ca), v, k.zero2);
    }
    if (SIGN != kPos) {
        const f2 M3 = fma2(SIGN == kNeg ? ca : min0(ca), v, k.zero2);
        const f2 d = sub2(s.M2, M3);
        const f2 n = add2(s.M2, lim_inc_x2(s.dM, d, k));
        F = SIGN == kNeg ? n : add2(F, n);
        s.M2 = M3;
        s.dM = d;
    }
    return F;
}

// The sweep before row k is taken: x of rows k - 1 .. k - 4, c a of rows k - 1 and k - 2, y (the first
// stage's result) of rows k - 3 and k - 4, the faces formed last, h (Heun's average) of row k - 5
// and the diffusion flux below it, the velocity index of row k.
struct Lim {
    Split a, b;
    f2 x1, x2, x3, x4, c1, c2, y3, y4, Fa, Fb, h, D, kk;
};

// Row k: x_k, its c a.  Returns the output of row k - 5.  wall_b, wall_d: the second stage's face or
// the diffusion flux lies on the lower wall.
template <int SIGN>
__device__ __forceinline__ f2 row(Lim& z, f2 x, f2 ca, bool wall_b, bool wall_d, const LimConst& k) {
    const f2 F = face<SIGN>(z.a, ca, x, k);                     // face k - 2 + 1/2
    const f2 y = sub2(z.x2, sub2(F, z.Fa));                     // row k - 2
    f2 G = face<SIGN>(z.b, z.c2, y, k);                         // face k - 4 + 1/2
    if (wall_b) G = 0ull;
    const f2 h = mul2(k.half2, add2(z.x4, sub2(z.y4, sub2(G, z.Fb))));  // row k - 4
    f2 D = fma2(k.r2, sub2(h, z.h), k.zero2);
    if (wall_d) D = 0ull;
    const f2 o = add2(z.h, sub2(D, z.D));
    z.x4 = z.x3;
    z.x3 = z.x2;
    z.x2 = z.x1;
    z.x1 = x;
    z.c2 = z.c1;
    z.c1 = ca;
    z.y4 = z.y3;
    z.y3 = y;
    z.Fa = F;
    z.Fb = G;
    z.h = h;
    z.D = D;
    return o;
}

struct Out {
    float* dst;  // the next row's cell of column c
    int nx;
    bool on0, on1;
    __device__ __forceinline__ void operator()(f2 o) {
        if (on0) dst[0] = lo(o);
        if (on1) dst[32] = hi(o);
        dst += nx;
    }
};

template <int NV, int SIGN>
__device__ __forceinline__ void chunk(Lim& z, const float* p, f2 w2, bool first, bool last,
                                      const LimConst& k, Out& out) {
    constexpr int J = (NV - 1) / 2;
#pragma unroll
    for (int e = 0; e < kChunk; ++e) {  // row 2 + e of the chunk's origin p
        const float* q = p + (e + 2) * kPitch + ((J - e - 2) & 3);
        f2 x = pk(q[0], q[32]);
        if (e == kChunk - 1 && last) x = 0ull;  // row N_v, beyond the wall
        const f2 ca = mul2(k.g2, sub2(w2, z.kk));
        z.kk = add2(z.kk, k.one2);
        const f2 o = row<SIGN>(z, x, ca, e == 1 && first, e == 2 && first, k);
        if (e > 2 || !first) out(o);
    }
}

// The step of columns c and c + 32: p their places of row 0 (without its shift).
template <int NV>
__device__ __forceinline__ void sweep(const float* p, f2 w2, float g, float r, float mu, Out out) {
    constexpr int J = (NV - 1) / 2;
    static_assert((NV - 1) % kChunk == 0 && J % 4 == 0, "whole chunks, one pattern of shifts");
    LimConst k;
    k.g2 = pk(g, g);
    k.r2 = pk(r, r);
    static_cast<LimPair&>(k) = lim_pair(mu);
    k.half2 = pk(0.5f, 0.5f);
    k.one2 = opaque2(pk(1.f, 1.f));
    // rows up to kp have c a >= 0 in every column of the warp, rows from kn on c a <= 0
    const float wlo = min_nan(lo(w2), hi(w2)), whi = max_nan(lo(w2), hi(w2));
    const bool sane = fabsf(wlo) < 1e6f && fabsf(whi) < 1e6f;  // false for NaN
    const int kp = __reduce_min_sync(0xffffffffu, sane ? (int)floorf(wlo) + J : -1);
    const int kn = __reduce_max_sync(0xffffffffu, sane ? (int)ceilf(whi) + J : NV);
    // rows 0 and 1
    Lim z;
    const f2 x0 = pk(p[J & 3], p[(J & 3) + 32]);
    const f2 x1 = pk(p[kPitch + ((J - 1) & 3)], p[kPitch + ((J - 1) & 3) + 32]);
    const f2 k0 = opaque2(pk(float(-J), float(-J)));
    const f2 k1 = add2(k0, k.one2);
    const f2 c0 = mul2(k.g2, sub2(w2, k0)), c1 = mul2(k.g2, sub2(w2, k1));
    const f2 P0 = fma2(max0(c0), x0, k.zero2), M0 = fma2(min0(c0), x0, k.zero2);
    z.a.P1 = P0;
    z.a.P2 = fma2(max0(c1), x1, k.zero2);
    z.a.dP = P0;
    z.a.M2 = fma2(min0(c1), x1, k.zero2);
    z.a.dM = sub2(M0, z.a.M2);
    z.b = Split{0ull, 0ull, 0ull, 0ull, 0ull};
    z.x1 = x1;
    z.x2 = x0;
    z.c1 = c1;
    z.c2 = c0;
    z.kk = add2(k1, k.one2);
    z.x3 = z.x4 = z.y3 = z.y4 = z.Fa = z.Fb = z.h = z.D = 0ull;
#pragma unroll 1
    for (int q = 0; q < NV - 1; q += kChunk, p += kChunk * kPitch) {
        const bool first = q == 0, last = q == NV - 1 - kChunk;
        // rows q + 2 - 5 .. q + 2 + 7 enter the chunk's faces
        if (q + 9 <= kp) chunk<NV, kPos>(z, p, w2, first, last, k, out);
        else if (q - 3 >= kn) chunk<NV, kNeg>(z, p, w2, first, last, k, out);
        else chunk<NV, kBoth>(z, p, w2, first, last, k, out);
    }
    // the upper wall: the first stage's face N_v - 1/2 is zero, then the second's
    const f2 y = sub2(z.x2, sub2(0ull, z.Fa));                       // row N_v - 1
    auto end = [&](f2 G, f2 xj, f2 yj) {                             // one more h and output
        const f2 h = mul2(k.half2, add2(xj, sub2(yj, sub2(G, z.Fb))));
        const f2 D = fma2(k.r2, sub2(h, z.h), k.zero2);
        out(add2(z.h, sub2(D, z.D)));
        z.Fb = G;
        z.h = h;
        z.D = D;
    };
    const f2 x_last = z.x2, x_before = z.x3, y_before = z.y3;
    end(face<kBoth>(z.b, z.c2, y, k), z.x4, z.y4);                   // row N_v - 3
    end(face<kBoth>(z.b, z.c2, 0ull, k), x_before, y_before);        // row N_v - 2
    end(0ull, x_last, y);                                            // row N_v - 1
    out(add2(z.h, sub2(0ull, z.D)));
}

// Columns x0 .. x0 + w - 1 of an instance; wrow: the step's row of wflow.
template <int NV>
__global__ void __launch_bounds__(kPlaces / 2, 3)
    k_lim1d(const Step1DArgs a, const MultiTile* tiles, int kstep, const float* wrow, int piped) {
    constexpr int J = (NV - 1) / 2;
    extern __shared__ __align__(128) unsigned char smem[];
    float* f = reinterpret_cast<float*>(smem);
    float* W = f + (NV + 1) * kPitch;  // one row beyond the planes is read (and not used)
    uint64_t* bar = reinterpret_cast<uint64_t*>(W + kPlaces);
    const MultiTile tile = tiles[blockIdx.x];
    const int nx = tile.nx, P = 2 * blockDim.x;
    const bool par = ((a.st->step + kstep) & 1) != 0;
    const float* fin = static_cast<const float*>(par ? a.f[1] : a.f[0]) + tile.off;
    float* fout = static_cast<float*>(par ? a.f[0] : a.f[1]) + tile.off;
    const float* w_in = wrow + tile.xoff;
    const int tid = threadIdx.x;
    if (piped) {
        if (tid == 0) {
            mbar_init(bar, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncthreads();
        if (!a.st->stall) {  // a stalled context issues no copies
            if (tid == 0) mbar_expect_tx(bar, (unsigned)((NV * (P + 4) + P) * sizeof(float)));
            for (int q = tid; q <= NV; q += blockDim.x) {
                const int len = q < NV ? P + 4 : P, j = q < NV ? q - J : 0;
                float* dst = q < NV ? f + q * kPitch : W;
                const float* src = q < NV ? fin + (size_t)q * nx : w_in;
                int b = (tile.x0 - j - (-j & 3)) % nx;
                b += b < 0 ? nx : 0;
                for (int n = 0; n < len;) {
                    const int m = min(len - n, nx - b);
                    bulk_g2s(dst + n, src + b, (unsigned)(m * sizeof(float)), bar);
                    n += m;
                    b = 0;
                }
            }
        }
    } else {
        for (int c = tid; c < P; c += blockDim.x) {
            const int xc = (tile.x0 + c) % nx;
            int x = (xc + J) % nx;
            const float* src = fin;
#pragma unroll 4
            for (int jj = 0; jj < NV; ++jj) {
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                                 smem_u32(f + jj * kPitch + ((J - jj) & 3) + c)),
                             "l"(src + x)
                             : "memory");
                src += nx;
                x = x == 0 ? nx - 1 : x - 1;
            }
            W[c] = w_in[xc];
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
    const int c = (tid >> 5) * kCols + (tid & 31);
    sweep<NV>(f + c, pk(W[c], W[c + 32]), tile.g, tile.r, float(a.mu),
              Out{fout + tile.x0 + c, nx, c < tile.w, c + 32 < tile.w});
}

template <int NV>
cudaError_t launch_t(int ntiles, int places, const Step1DArgs& a, const MultiTile* tiles, int kstep,
                     const float* wrow, int piped, cudaStream_t s) {
    constexpr int kSmem = 4 * ((NV + 1) * kPitch + kPlaces) + 16;
    static PerDevice limit;
    const cudaError_t e = raise_smem(limit, k_lim1d<NV>, kSmem);
    if (e != cudaSuccess) return e;
    k_lim1d<NV><<<ntiles, places / 2, kSmem, s>>>(a, tiles, kstep, wrow, piped);
    return cudaGetLastError();
}

}  // namespace

bool lim1d_shape(int nv, int* max_places) {
    *max_places = kPlaces;
    return nv == 9 || nv == 17 || nv == 33 || nv == 65;
}

int lim1d_places(int w) { return (w + kCols - 1) / kCols * kCols; }

cudaError_t launch_lim1d(int nv, int ntiles, int places, const Step1DArgs& a, const MultiTile* tiles,
                         int kstep, const float* wrow, int piped, cudaStream_t s) {
    switch (nv) {
#define X(n)     case n: return launch_t<n>(ntiles, places, a, tiles, kstep, wrow, piped, s);
        X(9) X(17) X(33) X(65)
#undef X
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace lat
