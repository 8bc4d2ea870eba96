// Device code shared by the 1D step kernels (step1d.cu, multi1d.cu, lim1d.cu, line1d.cu): the column
// arithmetic of both drag schemes, the flow evaluation and the amplitude update, and PTX wrappers
// for mbarriers and bulk asynchronous copies.
#pragma once

#include <stdint.h>

#include "f32x2.h"
#include "lat_internal.h"

namespace lat {
namespace k1d {

// ---- column arithmetic with explicit rounding (identical in every variant) -----------------
template <typename T>
struct Ops;
template <>
struct Ops<float> {
    static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
    static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
    static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
    static __device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
};
template <>
struct Ops<double> {
    static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
    static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }
};

// max(v, 0) and min(v, 0), zero where v is not a number.  FP64 by the upper word: comparisons run on
// the FP64 pipe, which bounds the FP64 kernels on this part (two operations per clock and SM).  NaNs
// (of arithmetic: quiet ones) lie above the infinities.
__device__ __forceinline__ float pos_part(float v) { return fmaxf(v, 0.f); }
__device__ __forceinline__ float neg_part(float v) { return fminf(v, 0.f); }
__device__ __forceinline__ double pos_part(double v) {
    return (unsigned)__double2hiint(v) <= 0x7ff00000u ? v : 0.0;
}
__device__ __forceinline__ double neg_part(double v) {
    return __double2hiint(v) <= (int)0xfff00000u ? v : 0.0;
}

// c a_j = (dt/dv) * (-(v_j - u)/tau_p) = g (w - j), g = dt/tau_p, w = u/dv
template <typename T>
__device__ __forceinline__ T cacc(T g, T w, int j) {
    return Ops<T>::mul(g, Ops<T>::sub(w, T(j)));
}
// c F_{j+1/2} = (c a_j)^+ f_j + (c a_{j+1})^- f_{j+1}   (cell-centred upwind)
template <typename T>
__device__ __forceinline__ T dflux(T caj, T can, T fj, T fn) {
    return Ops<T>::fma(pos_part(caj), fj, Ops<T>::mul(neg_part(can), fn));
}

// Sliding-window sweep of one column.  get(jj) returns f*(x, jj - J); put(jj, v) stores.
//   d_j   = f*_j - (cF_{j+1/2} - cF_{j-1/2})            (drag, zero flux at the walls)
//   out_j = d_j + (D_{j+1/2} - D_{j-1/2}),  D = r (d_{j+1} - d_j)   (diffusion)
template <typename T, int NV, class Get, class Put>
__device__ __forceinline__ void sweep_column(T w, T g, T r, const Get& get, const Put& put) {
    constexpr int J = (NV - 1) / 2;
    T s = get(0);
    T Fprev = T(0), Dprev = T(0), dprev = T(0);
#pragma unroll
    for (int jj = 0; jj < NV; ++jj) {
        T sn = T(0), Fn = T(0);
        if (jj < NV - 1) {
            sn = get(jj + 1);
            Fn = dflux<T>(cacc<T>(g, w, jj - J), cacc<T>(g, w, jj + 1 - J), s, sn);
        }
        const T d = Ops<T>::sub(s, Ops<T>::sub(Fn, Fprev));
        Fprev = Fn;
        if (jj > 0) {
            const T D = Ops<T>::mul(r, Ops<T>::sub(d, dprev));
            put(jj - 1, Ops<T>::add(dprev, Ops<T>::sub(D, Dprev)));
            Dprev = D;
        }
        dprev = d;
        s = sn;
    }
    put(NV - 1, Ops<T>::add(dprev, Ops<T>::sub(T(0), Dprev)));
}

// Packed two-lane form of sweep_column (FP32, N_v = 2h + 1 >= 5): lane 0 of an f32x2 pair
// sweeps cells 0 .. h, lane 1 cells h .. 2h, with exactly the operations of sweep_column in the
// same order, so the outputs have the same bits.  Lane 1 starts from the drag fluxes of faces
// h - 3/2 and h - 1/2 and the drag output of cell h - 1, which it computes from f*_{h-2..h}
// first.  put2(p, o) for p = 1..h stores lane 0's o at cell p - 1 and lane 1's at p - 1 + h;
// put_last(v) stores cell 2h.
template <int NV, class Get, class Put2, class PutLast>
__device__ __forceinline__ void sweep_column2(float w, float g, float r, const Get& get,
                                              const Put2& put2, const PutLast& put_last) {
    constexpr int J = (NV - 1) / 2, h = J;
    static_assert(NV >= 5, "packed sweep needs N_v >= 5");
    const f2 g2 = pk(g, g), w2 = pk(w, w), r2 = pk(r, r);
    const f2 one2 = opaque2(pk(1.f, 1.f));
    f2 kk = opaque2(pk(float(-J), 0.f));  // velocity indices of step p: (p - J, p)
    f2 cac = mul2(g2, sub2(w2, kk));
    // lane 1's entry state at cell h; lane 0 ends on cells h and h + 1, read once here, so that
    // put2 may overwrite a cell as soon as its output is formed (in-place sweeps)
    const float fm2 = get(h - 2), fm1 = get(h - 1), f0 = get(h), fp1 = get(h + 1);
    const float Fa = dflux<float>(cacc<float>(g, w, -2), cacc<float>(g, w, -1), fm2, fm1);
    const float Fb = dflux<float>(cacc<float>(g, w, -1), cacc<float>(g, w, 0), fm1, f0);
    const float dm1 = Ops<float>::sub(fm1, Ops<float>::sub(Fb, Fa));
    f2 s2 = pk(get(0), f0);
    f2 Fp = pk(0.f, Fb);
    f2 dp = pk(0.f, dm1);
    f2 Dp = 0ull;
#pragma unroll
    for (int p = 0; p <= h; ++p) {
        const f2 kn = add2(kk, one2);
        const f2 can = mul2(g2, sub2(w2, kn));
        f2 sn;
        if (p == 0) sn = pk(get(1), fp1);
        else if (p < h - 1) sn = pk(get(p + 1), get(p + 1 + h));
        else if (p == h - 1) sn = pk(f0, get(2 * h));
        else sn = pk(fp1, 0.f);
        f2 Fn = fma2(max0(cac), s2, mul2(min0(can), sn));
        if (p == h) Fn = pk(lo(Fn), 0.f);  // lane 1 reached the wall
        const f2 d = sub2(s2, sub2(Fn, Fp));
        Fp = Fn;
        const f2 D = mul2(r2, sub2(d, dp));
        if (p == 0) {
            Dp = pk(0.f, hi(D));  // lane 0 has no face below cell 0; lane 1: face h - 1/2
        } else {
            put2(p, add2(dp, sub2s(D, Dp)));
            Dp = D;
        }
        dp = d;
        s2 = sn;
        cac = can;
        kk = kn;
    }
    put_last(Ops<float>::add(hi(dp), Ops<float>::sub(0.f, hi(Dp))));
}

// ---- flux-limited drag (scheme KOREN) -----------------------------------------------------------
// Limited increment psi(theta) dp of Koren's limiter in Hundsdorfer et al.'s form (Sec. 2, flux
// limiter): psi(theta) = max(0, min(1, 1/3 + theta/6, mu theta)), theta = dm / dp, written
// without the division: with s = sign(dp), psi(theta) dp = s max(0, min(|dp|, s (dp/3 + dm/6),
// s mu dm)); zero when dp = 0.
template <typename T>
__device__ __forceinline__ T lim_inc(T dp, T dm, T mu) {
    using O = Ops<T>;
    const T s = copysign(T(1), dp);
    const T b = O::mul(s, O::fma(dm, T(1.0 / 6.0), O::mul(dp, T(1.0 / 3.0))));
    const T c = O::mul(s, O::mul(mu, dm));
    return O::mul(s, fmax(T(0), fmin(fabs(dp), fmin(b, c))));
}

// Limited flux through interface i + 1/2 from the split fluxes P = (c a)^+ q, M = (c a)^- q of
// cells i - 1 .. i + 2 (cells beyond the walls count as empty):
//   F = P_i + psi(theta^P)(P_{i+1} - P_i) + M_{i+1} + psi(theta^M)(M_i - M_{i+1}).
template <typename T, int NV>
__device__ __forceinline__ T lim_face(const T (&P)[NV], const T (&M)[NV], int i, T mu) {
    using O = Ops<T>;
    const T Pm = i >= 1 ? P[i - 1] : T(0);
    const T Mpp = i + 2 < NV ? M[i + 2] : T(0);
    const T pos = O::add(P[i], lim_inc<T>(O::sub(P[i + 1], P[i]), O::sub(P[i], Pm), mu));
    const T neg = O::add(M[i + 1], lim_inc<T>(O::sub(M[i], M[i + 1]), O::sub(M[i + 1], Mpp), mu));
    return O::add(pos, neg);
}

// The limited drag sub-step by Heun's method, then the diffusion, for one column (scheme KOREN):
//   y = x - (F(x)_{j+1/2} - F(x)_{j-1/2}),  h = (x + y - (F(y)_{j+1/2} - F(y)_{j-1/2})) / 2,
//   out = h + (D_{j+1/2} - D_{j-1/2}),  D = r (h_{j+1} - h_j),  zero fluxes at the walls.
// One unrolled pass over k: cell k is read, stage-1 face and cell k - 2, stage-2 face and cell
// k - 4, output k - 5, so that every array element lives for a few iterations only.
template <typename T, int NV, class Get, class Put>
__device__ __forceinline__ void sweep_column_lim(T w, T g, T r, T mu, const Get& get,
                                                 const Put& put) {
    using O = Ops<T>;
    constexpr int J = (NV - 1) / 2;
    T x[NV], P0[NV], M0[NV], y[NV], P1[NV], M1[NV], h[NV], F0[NV + 1], F1[NV + 1];
    T Dprev = T(0);
#pragma unroll
    for (int k = 0; k < NV + 5; ++k) {
        if (k < NV) {
            x[k] = get(k);
            const T ca = cacc<T>(g, w, k - J);
            P0[k] = O::mul(pos_part(ca), x[k]);
            M0[k] = O::mul(neg_part(ca), x[k]);
        }
        if (k - 2 >= 0 && k - 2 <= NV - 2) F0[k - 1] = lim_face<T, NV>(P0, M0, k - 2, mu);
        if (k - 2 >= 0 && k - 2 < NV) {
            const int j = k - 2;
            const T Fl = j == 0 ? T(0) : F0[j];
            const T Fr = j == NV - 1 ? T(0) : F0[j + 1];
            y[j] = O::sub(x[j], O::sub(Fr, Fl));
            const T ca = cacc<T>(g, w, j - J);
            P1[j] = O::mul(pos_part(ca), y[j]);
            M1[j] = O::mul(neg_part(ca), y[j]);
        }
        if (k - 4 >= 0 && k - 4 <= NV - 2) F1[k - 3] = lim_face<T, NV>(P1, M1, k - 4, mu);
        if (k - 4 >= 0 && k - 4 < NV) {
            const int j = k - 4;
            const T Fl = j == 0 ? T(0) : F1[j];
            const T Fr = j == NV - 1 ? T(0) : F1[j + 1];
            h[j] = O::mul(T(0.5), O::add(x[j], O::sub(y[j], O::sub(Fr, Fl))));
        }
        if (k - 5 >= 0 && k - 5 < NV) {
            const int j = k - 5;
            const T D = j < NV - 1 ? O::mul(r, O::sub(h[j + 1], h[j])) : T(0);
            put(j, O::add(h[j], O::sub(D, Dprev)));
            Dprev = D;
        }
    }
}

// Drag scheme of one column: upwind, or the limited scheme (LIM, a separate kernel instance,
// so that the upwind kernels keep their own code and registers).
template <typename T, int NV, bool LIM, class Get, class Put>
__device__ __forceinline__ void sweep_scheme(const Step1DArgs& a, T w, T g, T r, const Get& get,
                                             const Put& put) {
    if constexpr (LIM) sweep_column_lim<T, NV>(w, g, r, T(a.mu), get, put);
    else sweep_column<T, NV>(w, g, r, get, put);
}

// Runtime-N_v version of the same sweep (identical operation order).
template <typename T, class Get, class Put>
__device__ __forceinline__ void sweep_column_any(int NV, T w, T g, T r, const Get& get,
                                                 const Put& put) {
    const int J = (NV - 1) / 2;
    T s = get(0);
    T Fprev = T(0), Dprev = T(0), dprev = T(0);
#pragma unroll 4
    for (int jj = 0; jj < NV; ++jj) {
        T sn = T(0), Fn = T(0);
        if (jj < NV - 1) {
            sn = get(jj + 1);
            Fn = dflux<T>(cacc<T>(g, w, jj - J), cacc<T>(g, w, jj + 1 - J), s, sn);
        }
        const T d = Ops<T>::sub(s, Ops<T>::sub(Fn, Fprev));
        Fprev = Fn;
        if (jj > 0) {
            const T D = Ops<T>::mul(r, Ops<T>::sub(d, dprev));
            put(jj - 1, Ops<T>::add(dprev, Ops<T>::sub(D, Dprev)));
            Dprev = D;
        }
        dprev = d;
        s = sn;
    }
    put(NV - 1, Ops<T>::add(dprev, Ops<T>::sub(T(0), Dprev)));
}

// ---- flow ------------------------------------------------------------------------------------
__device__ __forceinline__ void sincospi_t(float y, float* s, float* c) { sincospif(y, s, c); }
__device__ __forceinline__ void sincospi_t(double y, double* s, double* c) { sincospi(y, s, c); }

template <typename T>
__device__ __forceinline__ const T* amp_ptr(const Step1DArgs& a, int par, int inst);
template <>
__device__ __forceinline__ const float* amp_ptr<float>(const Step1DArgs& a, int par, int inst) {
    return a.ampf + par * a.amp_stride + (long long)inst * 2 * a.nmodes;
}
template <>
__device__ __forceinline__ const double* amp_ptr<double>(const Step1DArgs& a, int par, int inst) {
    return a.amp + par * a.amp_stride + (long long)inst * 2 * a.nmodes;
}

// u(x_i, t_n) = sum_m A_m cos(2 pi k_m i / N_x) + B_m sin(2 pi k_m i / N_x); the phase is
// reduced in integers (k_m i mod N_x) and evaluated as sin/cos of pi * (2 (k_m i mod N_x)/N_x).
// Explicit rounding, so that every kernel variant gets the same bits whatever the compiler
// contracts around it.
template <typename T>
__device__ __forceinline__ void flow_basis(int k, const Inst1D& in, T two_over_nx, int x, T* s,
                                           T* c) {
    int kx = k * x;
    kx = in.pow2 ? (kx & (in.nx - 1)) : (kx % in.nx);
    if (kx < 0) kx += in.nx;
    sincospi_t(Ops<T>::mul(T(kx), two_over_nx), s, c);
}
// one mode's share: u + (A c + B s)
template <typename T>
__device__ __forceinline__ T flow_add(T u, T A, T B, T s, T c) {
    using O = Ops<T>;
    return O::add(u, O::fma(A, c, O::mul(B, s)));
}
template <typename T>
__device__ __forceinline__ T flow_at(const Step1DArgs& a, const Inst1D& in, const T* amp, int x) {
    if (a.flow_kind == LAT_FLOW_FIELD) return static_cast<const T*>(a.field)[in.xoff + x];
    if (a.flow_kind != LAT_FLOW_MODES) return T(0);
    const int M = a.nmodes;
    const T two_over_nx = T(in.two_over_nx);
    T u = T(0);
    for (int m = 0; m < M; ++m) {
        T s, c;
        flow_basis<T>(a.k[m], in, two_over_nx, x, &s, &c);
        u = flow_add<T>(u, __ldg(amp + m), __ldg(amp + M + m), s, c);
    }
    return u;
}

// u / dv of column x: formed here, or taken from the array the flow kernel of multi1d.cu filled
// (which then also advances the amplitudes).
template <typename T>
__device__ __forceinline__ T flow_w(const Step1DArgs& a, const Inst1D& in, const T* amp, int x) {
    if (a.wpre) return static_cast<const T*>(a.wpre)[in.xoff + x];
    return flow_at<T>(a, in, amp, x) * T(in.inv_dv);
}

// Exact Ornstein-Uhlenbeck update of the instance's amplitudes (Eq. A1d), t_n -> t_{n+1}.
__device__ __forceinline__ void advance_amplitudes(const Step1DArgs& a, int inst,
                                                   const Inst1D& in, long long step, int par) {
    const int M2 = 2 * a.nmodes;
    const long long row = step - a.st->noise_base;
    const bool have = row >= 0 && row < a.st->noise_rows;
    for (int t = threadIdx.x; t < M2; t += blockDim.x) {
        const double old = a.amp[par * a.amp_stride + (long long)inst * M2 + t];
        double xi = 0.0;
        if (have) xi = a.noise[row * a.amp_stride + (long long)inst * M2 + t];
        const double nw = __dadd_rn(__dmul_rn(old, in.ou_e), __dmul_rn(in.ou_s, xi));
        a.amp_w[(1 - par) * a.amp_stride + (long long)inst * M2 + t] = nw;
        a.ampf_w[(1 - par) * a.amp_stride + (long long)inst * M2 + t] = (float)nw;
    }
    if (!have && threadIdx.x == 0) atomicOr(&a.st->status, ST_NOISE);
}

template <typename T, int J, bool LIM = false>
__device__ __forceinline__ void cfl_flag(const Step1DArgs& a, T g, T w) {
    // Eq. (cfl); each stage of the limited scheme (LIM) is positive for nu (1 + mu) <= 1
    const T f = LIM ? T(1) + T(a.mu) : T(1);
    if (g * (T(J) + fabs(w)) * f > T(1)) atomicOr(&a.st->status, ST_CFL);
}

// ---- PTX helpers (mbarrier + bulk async copy) ---------------------------------------------
__device__ __forceinline__ unsigned smem_u32(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes,
                                         uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ unsigned long long globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait on an mbarrier phase: gives up after ~1 s (the caller raises ST_TIMEOUT).
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, unsigned parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = globaltimer();
    for (long long it = 0; it < (1ll << 26); ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 255) == 0 && globaltimer() - t0 > 1000000000ull) break;
    }
    return false;
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

}  // namespace k1d
}  // namespace lat
