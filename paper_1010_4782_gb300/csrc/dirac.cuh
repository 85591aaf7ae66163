// dirac.cuh - the arithmetics and single-hop products of the Dirac kernels
// (dslash.cu: one thread per output site; dirac_lanes.cuh: one to eight lanes per site).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "ff.cuh"
#include "links.cuh"
#include "stag_kernels.h"

namespace stag {

// ------------------------------------------------------------ arithmetics
struct ArithF64 {
    using T = double2;  // storage
    using C = double2;  // compute
    static __device__ __forceinline__ C ld(const T* p) { return __ldg(p); }
    using TL = T;  // link storage
    static constexpr int kEntries = 9;  // stored entries per link
    static constexpr bool kRecon = false;
    static __device__ __forceinline__ C ldl(const TL* p) { return ld(p); }
    struct Acc {
        double2 c[3];
        double dot;
    };
    using Sum = double;  // of a dot product
    static __device__ __forceinline__ Sum dot(const Acc& a) { return a.dot; }
    static __device__ __forceinline__ void zero(Acc& a) {
#pragma unroll
        for (int r = 0; r < 3; ++r) a.c[r] = make_double2(0.0, 0.0);
        a.dot = 0.0;
    }
    // a_r += sum_c u_c v_c
    static __device__ __forceinline__ void row_fwd(Acc& a, int r, C u0, C u1, C u2, C v0, C v1, C v2) {
        cmac(a.c[r], u0, v0);
        cmac(a.c[r], u1, v1);
        cmac(a.c[r], u2, v2);
    }
    // a_r -= sum_c conj(u_c) v_c
    static __device__ __forceinline__ void row_bwd(Acc& a, int r, C u0, C u1, C u2, C v0, C v1, C v2) {
        cmsc_conj(a.c[r], u0, v0);
        cmsc_conj(a.c[r], u1, v1);
        cmsc_conj(a.c[r], u2, v2);
    }
    static __device__ __forceinline__ T store_val(const Acc& a, int r) { return a.c[r]; }
    // o = m2 * s - acc_r; the dot product += Re(conj(s) o)
    static __device__ __forceinline__ T epilogue(Acc& a, int r, C s, double m2, float2) {
        const double2 d = a.c[r];
        const double2 o = make_double2(fma(m2, s.x, -d.x), fma(m2, s.y, -d.y));
        a.dot = fma(s.x, o.x, a.dot);
        a.dot = fma(s.y, o.y, a.dot);
        return o;
    }
};

struct ArithFF {
    using T = float4;
    using C = float4;
    static __device__ __forceinline__ C ld(const T* p) { return __ldg(p); }
    using TL = T;  // link storage
    static constexpr int kEntries = 9;  // stored entries per link
    static constexpr bool kRecon = false;
    static __device__ __forceinline__ C ldl(const TL* p) { return ld(p); }
    struct Acc {
        FFAcc re[3], im[3];
        FFAcc dot;
    };
    static __device__ __forceinline__ void zero(Acc& a) {
#pragma unroll
        for (int r = 0; r < 3; ++r) a.re[r] = a.im[r] = ff_zero();
        a.dot = ff_zero();
    }
    static __device__ __forceinline__ void row_fwd(Acc& a, int r, C u0, C u1, C u2, C v0, C v1, C v2) {
        ff_row_fwd(a.re[r], a.im[r], u0, u1, u2, v0, v1, v2);
    }
    static __device__ __forceinline__ void row_bwd(Acc& a, int r, C u0, C u1, C u2, C v0, C v1, C v2) {
        ff_row_bwd(a.re[r], a.im[r], u0, u1, u2, v0, v1, v2);
    }
    static __device__ __forceinline__ T store_val(const Acc& a, int r) {
        return ff_cplx(ff_result(a.re[r]), ff_result(a.im[r]));
    }
    using Sum = FFAcc;
    static __device__ __forceinline__ Sum dot(const Acc& a) { return a.dot; }
    // o = m2 * s - acc_r in float-float; Re(conj(s) o) accumulated in float-float
    static __device__ __forceinline__ T epilogue(Acc& a, int r, C s, double, float2 m2) {
        const float2 re = ff_fma(m2, ff_re(s), ff_neg(ff_result(a.re[r])));
        const float2 im = ff_fma(m2, ff_im(s), ff_neg(ff_result(a.im[r])));
        const float4 o = ff_cplx(re, im);
        ff_redot_acc(a.dot, s, o);
        return o;
    }
};

// FP32 storage and arithmetic (inner solver of the mixed-precision CG).
struct ArithF32 {
    using T = float2;
    using C = float2;
    static __device__ __forceinline__ C ld(const T* p) { return __ldg(p); }
    using TL = T;  // link storage
    static constexpr int kEntries = 9;  // stored entries per link
    static constexpr bool kRecon = false;
    struct Acc {
        float2 c[3];
        float dot;
    };
    static __device__ __forceinline__ void zero(Acc& a) {
#pragma unroll
        for (int r = 0; r < 3; ++r) a.c[r] = make_float2(0.f, 0.f);
        a.dot = 0.f;
    }
    static __device__ __forceinline__ void row_fwd(Acc& a, int r, C u0, C u1, C u2, C v0, C v1, C v2) {
        cmacf(a.c[r], u0, v0);
        cmacf(a.c[r], u1, v1);
        cmacf(a.c[r], u2, v2);
    }
    static __device__ __forceinline__ void row_bwd(Acc& a, int r, C u0, C u1, C u2, C v0, C v1, C v2) {
        cmscf_conj(a.c[r], u0, v0);
        cmscf_conj(a.c[r], u1, v1);
        cmscf_conj(a.c[r], u2, v2);
    }
    static __device__ __forceinline__ T store_val(const Acc& a, int r) { return a.c[r]; }
    using Sum = FFAcc;
    static __device__ __forceinline__ Sum dot(const Acc& a) { return FFAcc{a.dot, 0.f}; }
    static __device__ __forceinline__ T epilogue(Acc& a, int r, C s, double, float2 m2) {
        const float2 d = a.c[r];
        const float2 o = make_float2(fmaf(m2.x, s.x, -d.x), fmaf(m2.x, s.y, -d.y));
        a.dot = fmaf(s.x, o.x, a.dot);
        a.dot = fmaf(s.y, o.y, a.dot);
        return o;
    }
};

// FP16 storage (links and vectors as half2 = (re, im)), FP32 arithmetic.
struct ArithH16 {
    using T = __half2;
    using C = float2;
    static __device__ __forceinline__ C ld(const T* p) { return __half22float2(__ldg(p)); }
    using TL = T;  // link storage
    static constexpr int kEntries = 9;  // stored entries per link
    static constexpr bool kRecon = false;
    using Acc = ArithF32::Acc;
    using Sum = ArithF32::Sum;
    static __device__ __forceinline__ Sum dot(const Acc& a) { return ArithF32::dot(a); }
    static __device__ __forceinline__ void zero(Acc& a) { ArithF32::zero(a); }
    static __device__ __forceinline__ void row_fwd(Acc& a, int r, C u0, C u1, C u2, C v0, C v1, C v2) {
        ArithF32::row_fwd(a, r, u0, u1, u2, v0, v1, v2);
    }
    static __device__ __forceinline__ void row_bwd(Acc& a, int r, C u0, C u1, C u2, C v0, C v1, C v2) {
        ArithF32::row_bwd(a, r, u0, u1, u2, v0, v1, v2);
    }
    static __device__ __forceinline__ T store_val(const Acc& a, int r) { return __float22half2_rn(a.c[r]); }
    static __device__ __forceinline__ T epilogue(Acc& a, int r, C s, double m2, float2 m2f) {
        return __float22half2_rn(ArithF32::epilogue(a, r, s, m2, m2f));
    }
};

// BF16 storage (links and vectors as bfloat162 = (re, im)), FP32 arithmetic:
// FP32's exponent range with an 8-bit significand.
struct ArithB16 {
    using T = __nv_bfloat162;
    using C = float2;
    static __device__ __forceinline__ C ld(const T* p) { return __bfloat1622float2(__ldg(p)); }
    using TL = T;  // link storage
    static constexpr int kEntries = 9;  // stored entries per link
    static constexpr bool kRecon = false;
    using Acc = ArithF32::Acc;
    using Sum = ArithF32::Sum;
    static __device__ __forceinline__ Sum dot(const Acc& a) { return ArithF32::dot(a); }
    static __device__ __forceinline__ void zero(Acc& a) { ArithF32::zero(a); }
    static __device__ __forceinline__ void row_fwd(Acc& a, int r, C u0, C u1, C u2, C v0, C v1, C v2) {
        ArithF32::row_fwd(a, r, u0, u1, u2, v0, v1, v2);
    }
    static __device__ __forceinline__ void row_bwd(Acc& a, int r, C u0, C u1, C u2, C v0, C v1, C v2) {
        ArithF32::row_bwd(a, r, u0, u1, u2, v0, v1, v2);
    }
    static __device__ __forceinline__ T store_val(const Acc& a, int r) { return __float22bfloat162_rn(a.c[r]); }
    static __device__ __forceinline__ T epilogue(Acc& a, int r, C s, double m2, float2 m2f) {
        return __float22bfloat162_rn(ArithF32::epilogue(a, r, s, m2, m2f));
    }
};

// FP32 with 12-parameter links (Sec. 3.3): two stored rows a, b of each
// eta-folded SU(3) link; the third is eta (a x b)^* (for U in SU(3) the third
// row is the conjugate cross product of the first two, and eta^2 = 1).  Link
// bytes drop by a third for 6 complex multiply-adds per row.
struct ArithF32R {
    using T = float2;
    using TL = float2;
    using C = float2;
    static constexpr int kEntries = 6;
    static constexpr bool kRecon = true;
    static __device__ __forceinline__ C ld(const T* p) { return __ldg(p); }
    using Acc = ArithF32::Acc;
    using Sum = ArithF32::Sum;
    static __device__ __forceinline__ Sum dot(const Acc& a) { return ArithF32::dot(a); }
    static __device__ __forceinline__ void zero(Acc& a) { ArithF32::zero(a); }
    static __device__ __forceinline__ void row_fwd(Acc& a, int r, C u0, C u1, C u2, C v0, C v1, C v2) {
        ArithF32::row_fwd(a, r, u0, u1, u2, v0, v1, v2);
    }
    static __device__ __forceinline__ void row_bwd(Acc& a, int r, C u0, C u1, C u2, C v0, C v1, C v2) {
        ArithF32::row_bwd(a, r, u0, u1, u2, v0, v1, v2);
    }
    static __device__ __forceinline__ T store_val(const Acc& a, int r) { return ArithF32::store_val(a, r); }
    static __device__ __forceinline__ T epilogue(Acc& a, int r, C s, double m2, float2 m2f) {
        return ArithF32::epilogue(a, r, s, m2, m2f);
    }
};

// FP16-stored links, FP32 vectors and arithmetic: the links carry most of the
// bytes, the vectors keep FP32's significand (the CG direction and residual).
struct ArithL16 {
    using T = float2;
    using TL = __half2;
    static constexpr int kEntries = 9;
    static constexpr bool kRecon = false;
    using C = float2;
    static __device__ __forceinline__ C ld(const T* p) { return __ldg(p); }
    using Acc = ArithF32::Acc;
    using Sum = ArithF32::Sum;
    static __device__ __forceinline__ Sum dot(const Acc& a) { return ArithF32::dot(a); }
    static __device__ __forceinline__ void zero(Acc& a) { ArithF32::zero(a); }
    static __device__ __forceinline__ void row_fwd(Acc& a, int r, C u0, C u1, C u2, C v0, C v1, C v2) {
        ArithF32::row_fwd(a, r, u0, u1, u2, v0, v1, v2);
    }
    static __device__ __forceinline__ void row_bwd(Acc& a, int r, C u0, C u1, C u2, C v0, C v1, C v2) {
        ArithF32::row_bwd(a, r, u0, u1, u2, v0, v1, v2);
    }
    static __device__ __forceinline__ T store_val(const Acc& a, int r) { return ArithF32::store_val(a, r); }
    static __device__ __forceinline__ T epilogue(Acc& a, int r, C s, double m2, float2 m2f) {
        return ArithF32::epilogue(a, r, s, m2, m2f);
    }
};

template <class A>
struct DslashParams {
    Geom g;
    int P;                     // output parity
    const typename A::TL* fat;  // [2][4][9][vs], or the words of links.cuh
    const typename A::TL* lng;  // the same, or nullptr
    const typename A::T* in;   // [3][vs], parity 1-P
    typename A::T* out;        // [3][vs], parity P
    const typename A::T* src;  // [3][vs], parity P (EPI_AXPY / EPI_CG)
    double m2;                 // m^2 (EPI_AXPY)
    float2 m2_ff;              // m^2 as float-float (EPI_AXPY, FF)
    CgScalars* scal;
    double* partials;
    int i0, i1;                // output sites [i0, i1) of parity P
    float2 lng_s = make_float2(0.f, 0.f);  // NAIK == 2: 1 / scale of the two-row Naik links (float-float)
    int epi = EPI_PLAIN;       // the epilogue of a kernel that takes it at run time
};

// Link entries 6..8 (the third row) from the first two: eta * conj(row0 x row1).
__device__ __forceinline__ float2 cross_conj(float2 a1, float2 b2, float2 a2, float2 b1, float eta) {
    // conj(a1 b2 - a2 b1) * eta
    const float re = a1.x * b2.x - a1.y * b2.y - (a2.x * b1.x - a2.y * b1.y);
    const float im = a1.x * b2.y + a1.y * b2.x - (a2.x * b1.y + a2.y * b1.x);
    return make_float2(eta * re, -eta * im);
}
__device__ __forceinline__ void load_recon(float2 (&U)[9], const float2* __restrict__ u, size_t vs, int i, float eta) {
    load_link<6>(U, u, vs, i);
    U[6] = cross_conj(U[1], U[5], U[2], U[4], eta);
    U[7] = cross_conj(U[2], U[3], U[0], U[5], eta);
    U[8] = cross_conj(U[0], U[4], U[1], U[3], eta);
}

// Float-float Naik link stored as its first two rows ([6][vs], eta folded); the
// third row is (eta / scale) conj(row0 x row1), s = eta / scale (Sec. 3.3's
// 12-parameter form applied to scale x SU(3)).
__device__ __forceinline__ void load_recon_ff(float4 (&U)[9], const float4* __restrict__ u, size_t vs, float2 s) {
#pragma unroll
    for (int k = 0; k < 6; ++k) U[k] = __ldg(u + k * vs);
    U[6] = ff_cross_conj_scaled(U[1], U[5], U[2], U[4], s);
    U[7] = ff_cross_conj_scaled(U[2], U[3], U[0], U[5], s);
    U[8] = ff_cross_conj_scaled(U[0], U[4], U[1], U[3], s);
}
__device__ __forceinline__ void hop_fwd_ffr(ArithFF::Acc& acc, const float4* __restrict__ u,
                                            const float4* __restrict__ in, int nb, size_t vs, float2 s) {
    const float4 v0 = __ldg(in + nb), v1 = __ldg(in + vs + nb), v2 = __ldg(in + 2 * vs + nb);
    float4 U[9];
    load_recon_ff(U, u, vs, s);
#pragma unroll
    for (int r = 0; r < 3; ++r) ArithFF::row_fwd(acc, r, U[3 * r], U[3 * r + 1], U[3 * r + 2], v0, v1, v2);
}
__device__ __forceinline__ void hop_bwd_ffr(ArithFF::Acc& acc, const float4* __restrict__ u,
                                            const float4* __restrict__ in, int nb, size_t vs, float2 s) {
    const float4 v0 = __ldg(in + nb), v1 = __ldg(in + vs + nb), v2 = __ldg(in + 2 * vs + nb);
    float4 U[9];
    load_recon_ff(U, u, vs, s);
#pragma unroll
    for (int r = 0; r < 3; ++r) ArithFF::row_bwd(acc, r, U[r], U[3 + r], U[6 + r], v0, v1, v2);
}

// acc += U in(nb) with site i's link of part u (its [parity][mu]); backward: acc -= U^dag in(nb).
// FP32 arithmetic takes the whole link in 16-byte words; FP64 and float-float, whose
// entries are words, a row (or column) at a time, which needs fewer registers at once.
template <class A>
__device__ __forceinline__ void hop_fwd(typename A::Acc& acc, const typename A::TL* __restrict__ u, int i,
                                        const typename A::T* __restrict__ in, int nb, size_t vs, float eta = 1.f) {
    const typename A::C v0 = A::ld(in + nb), v1 = A::ld(in + vs + nb), v2 = A::ld(in + 2 * vs + nb);
    if constexpr (std::is_same<typename A::C, float2>::value) {
        float2 U[9];
        if constexpr (A::kRecon)
            load_recon(U, u, vs, i, eta);
        else
            load_link<9>(U, u, vs, i);
#pragma unroll
        for (int r = 0; r < 3; ++r) A::row_fwd(acc, r, U[3 * r], U[3 * r + 1], U[3 * r + 2], v0, v1, v2);
    } else {
        u += i;
#pragma unroll
        for (int r = 0; r < 3; ++r)
            A::row_fwd(acc, r, A::ldl(u + (3 * r) * vs), A::ldl(u + (3 * r + 1) * vs), A::ldl(u + (3 * r + 2) * vs),
                       v0, v1, v2);
    }
}

template <class A>
__device__ __forceinline__ void hop_bwd(typename A::Acc& acc, const typename A::TL* __restrict__ u, int i,
                                        const typename A::T* __restrict__ in, size_t vs, float eta = 1.f) {
    const typename A::C v0 = A::ld(in + i), v1 = A::ld(in + vs + i), v2 = A::ld(in + 2 * vs + i);
    // (U^dag v)_r = sum_c conj(U_cr) v_c; the link is the neighbour's own
    if constexpr (std::is_same<typename A::C, float2>::value) {
        float2 U[9];
        if constexpr (A::kRecon)
            load_recon(U, u, vs, i, eta);
        else
            load_link<9>(U, u, vs, i);
#pragma unroll
        for (int r = 0; r < 3; ++r) A::row_bwd(acc, r, U[r], U[3 + r], U[6 + r], v0, v1, v2);
    } else {
        u += i;
#pragma unroll
        for (int r = 0; r < 3; ++r)
            A::row_bwd(acc, r, A::ldl(u + r * vs), A::ldl(u + (3 + r) * vs), A::ldl(u + (6 + r) * vs), v0, v1, v2);
    }
}

// Half-lattice index of the neighbour of (x,y,z,t) at +-h along mu.
__device__ __forceinline__ int neighbour(const Geom& g, int x, int y, int z, int t, int mu, int h,
                                         bool up) {
    switch (mu) {
        case 0: x = up ? wrap_up(x, h, g.lx) : wrap_dn(x, h, g.lx); break;
        case 1: y = up ? wrap_up(y, h, g.ly) : wrap_dn(y, h, g.ly); break;
        case 2: z = up ? wrap_up(z, h, g.lz) : wrap_dn(z, h, g.lz); break;
        default: t = up ? wrap_up(t, h, g.lt) : wrap_dn(t, h, g.lt); break;
    }
    return site_index(x, y, z, t, g);
}

// acc += (D_{P,1-P} in)(i) for output site i of parity p.P (all hops).
// NAIK: 0 one-hop only; 1 Naik links with nine entries; 2 float-float Naik
// links with two rows (A = ArithFF only).
template <class A, int NAIK>
__device__ __forceinline__ void dslash_site(const DslashParams<A>& p, int i, typename A::Acc& acc) {
    const Geom& g = p.g;
    const size_t vs = (size_t)g.vs;
    {
        int x, y, z, t;
        site_coords(i, p.P, g, x, y, z, t);
        const int P = p.P, Q = 1 - p.P;
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            const int f1 = neighbour(g, x, y, z, t, mu, 1, true);
            const int b1 = neighbour(g, x, y, z, t, mu, 1, false);
            // eta_mu(x) = eta_mu(x - mu): the phase of both links of this direction
            const int ps = (mu >= 1 ? x : 0) + (mu >= 2 ? y : 0) + (mu >= 3 ? z : 0);
            const float eta = (ps & 1) ? -1.f : 1.f;
            hop_fwd<A>(acc, p.fat + ((size_t)(P * 4 + mu) * A::kEntries) * vs, i, p.in, f1, vs, eta);
            hop_bwd<A>(acc, p.fat + ((size_t)(Q * 4 + mu) * A::kEntries) * vs, b1, p.in, vs, eta);
            if constexpr (NAIK == 1) {
                const int h = g.hop3[mu];
                const int f3 = neighbour(g, x, y, z, t, mu, h, true);
                const int b3 = neighbour(g, x, y, z, t, mu, h, false);
                hop_fwd<A>(acc, p.lng + ((size_t)(P * 4 + mu) * 9) * vs, i, p.in, f3, vs);
                hop_bwd<A>(acc, p.lng + ((size_t)(Q * 4 + mu) * 9) * vs, b3, p.in, vs);
            }
        }
        if constexpr (NAIK == 2) {
            // A rolled loop: unrolled, the four copies of the float-float
            // reconstruction overflow the instruction cache.
#pragma unroll 1
            for (int mu = 0; mu < 4; ++mu) {
                const int h = mu == 0 ? g.hop3[0] : mu == 1 ? g.hop3[1] : mu == 2 ? g.hop3[2] : g.hop3[3];
                const int f3 = neighbour(g, x, y, z, t, mu, h, true);
                const int b3 = neighbour(g, x, y, z, t, mu, h, false);
                // the Naik link of x and the one arriving from x - 3 mu share eta_mu(x)
                const int ps = (mu >= 1 ? x : 0) + (mu >= 2 ? y : 0) + (mu >= 3 ? z : 0);
                if constexpr (std::is_same<A, ArithFF>::value) {
                    const float2 s = (ps & 1) ? make_float2(-p.lng_s.x, -p.lng_s.y) : p.lng_s;
                    hop_fwd_ffr(acc, p.lng + ((size_t)(P * 4 + mu) * 6) * vs + i, p.in, f3, vs, s);
                    hop_bwd_ffr(acc, p.lng + ((size_t)(Q * 4 + mu) * 6) * vs + b3, p.in, b3, vs, s);
                } else {
                    // FP32 (the mixed-precision iteration): the same rows, the third
                    // rebuilt in FP32 with the factor eta / scale
                    const float s = (ps & 1) ? -p.lng_s.x : p.lng_s.x;
                    hop_fwd<ArithF32R>(acc, p.lng + ((size_t)(P * 4 + mu) * 6) * vs, i, p.in, f3, vs, s);
                    hop_bwd<ArithF32R>(acc, p.lng + ((size_t)(Q * 4 + mu) * 6) * vs, b3, p.in, vs, s);
                }
            }
        }
    }
}

}  // namespace stag
