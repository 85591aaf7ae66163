// dirac_lanes.cuh - the half-Dslash of one output site on S = 2, 4 or 8 lanes of
// a warp (resident.cu): lane part q of a site takes the forward hops (q even) or
// the backward hops (q odd) along 8 / S of the directions, and the lanes' sums
// are added with shuffles.  A small lattice then spreads over S times as many
// threads, and each thread waits for 16 / S loads of links instead of 16.
#pragma once

#include "dirac.cuh"

namespace stag {

// Plain loads: the vectors are written by other SMs during the same launch (a
// grid-wide exchange lies between), so they must not go through the
// read-only path.
__device__ __forceinline__ double2 ld_vec(const double2* p) { return *p; }
__device__ __forceinline__ float4 ld_vec(const float4* p) { return *p; }
__device__ __forceinline__ float2 ld_vec(const float2* p) { return *p; }
__device__ __forceinline__ float2 ld_vec(const __half2* p) { return __half22float2(*p); }
__device__ __forceinline__ float2 ld_vec(const __nv_bfloat162* p) { return __bfloat1622float2(*p); }

__device__ __forceinline__ float flip(float v, bool f) {
    return __uint_as_float(__float_as_uint(v) ^ (f ? 0x80000000u : 0u));
}
__device__ __forceinline__ double flip(double v, bool f) {
    return __hiloint2double(__double2hiint(v) ^ (f ? (int)0x80000000 : 0), __double2loint(v));
}
// conj(v) when f
__device__ __forceinline__ double2 conj_if(double2 v, bool f) { return make_double2(v.x, flip(v.y, f)); }
__device__ __forceinline__ float4 conj_if(float4 v, bool f) { return make_float4(v.x, v.y, flip(v.z, f), flip(v.w, f)); }
__device__ __forceinline__ float2 conj_if(float2 v, bool f) { return make_float2(v.x, flip(v.y, f)); }

__device__ __forceinline__ void swap_if(float2& a, float2& b, bool sw) {
    const float2 x = a, y = b;
    a = make_float2(sw ? y.x : x.x, sw ? y.y : x.y);
    b = make_float2(sw ? x.x : y.x, sw ? x.y : y.y);
}
__device__ __forceinline__ void swap_if(float4& a, float4& b, bool sw) {
    const float4 x = a, y = b;
    a = make_float4(sw ? y.x : x.x, sw ? y.y : x.y, sw ? y.z : x.z, sw ? y.w : x.w);
    b = make_float4(sw ? x.x : y.x, sw ? x.y : y.y, sw ? x.z : y.z, sw ? x.w : y.w);
}

// One hop, forward (U v) or, for a lane of backward hops, U^T conj(v): the
// backward term is -U^dag v = -conj(U^T conj(v)), and a lane's hops all have the
// same sign, so its sums are negated and conjugated once, in lane_sums (the real
// part's sign).  The transpose is taken by the order of the loads, or for
// two-row links by exchanging entries after the third row is rebuilt.
template <class A, int ENTRIES>
__device__ __forceinline__ void lane_hop(typename A::Acc& acc, const typename A::TL* __restrict__ u, int li,
                                         const typename A::T* in, int nb, size_t vs, bool bwd, float2 s) {
    using C = typename A::C;
    C U[9], v[3];
    constexpr bool kWords = std::is_same<C, float2>::value;  // links in 16-byte words of several entries
    if constexpr (ENTRIES == 9 && !kWords) {
        const size_t sr = (bwd ? 1 : 3) * vs, sc = (bwd ? 3 : 1) * vs;
        u += li;
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int c = 0; c < 3; ++c) U[3 * r + c] = A::ldl(u + r * sr + c * sc);
    } else {
        load_link<ENTRIES>(U, u, vs, li);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) v[c] = conj_if(ld_vec(in + c * vs + nb), bwd);
    if constexpr (ENTRIES == 6) {
        if constexpr (std::is_same<C, float4>::value) {
            U[6] = ff_cross_conj_scaled(U[1], U[5], U[2], U[4], s);
            U[7] = ff_cross_conj_scaled(U[2], U[3], U[0], U[5], s);
            U[8] = ff_cross_conj_scaled(U[0], U[4], U[1], U[3], s);
        } else {
            U[6] = cross_conj(U[1], U[5], U[2], U[4], s.x);
            U[7] = cross_conj(U[2], U[3], U[0], U[5], s.x);
            U[8] = cross_conj(U[0], U[4], U[1], U[3], s.x);
        }
    }
    if constexpr (ENTRIES == 6 || kWords) {
        swap_if(U[1], U[3], bwd);
        swap_if(U[2], U[6], bwd);
        swap_if(U[5], U[7], bwd);
    }
#pragma unroll
    for (int r = 0; r < 3; ++r) A::row_fwd(acc, r, U[3 * r], U[3 * r + 1], U[3 * r + 2], v[0], v[1], v[2]);
}

// acc = sum over the site's S lanes (lane q's q odd: -conj of its own first), in all of them.
template <int S>
__device__ __forceinline__ void lane_sums(ArithFF::Acc& a, bool bwd) {
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        a.re[r].s = flip(a.re[r].s, bwd);
        a.re[r].e = flip(a.re[r].e, bwd);
#pragma unroll
        for (int o = 32 / S; o < 32; o <<= 1) {
            FFAcc x, y;
            x.s = __shfl_xor_sync(0xffffffffu, a.re[r].s, o);
            x.e = __shfl_xor_sync(0xffffffffu, a.re[r].e, o);
            y.s = __shfl_xor_sync(0xffffffffu, a.im[r].s, o);
            y.e = __shfl_xor_sync(0xffffffffu, a.im[r].e, o);
            ff_merge(a.re[r], x);
            ff_merge(a.im[r], y);
        }
    }
}
template <int S, class Acc>
__device__ __forceinline__ void lane_sums(Acc& a, bool bwd) {
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        a.c[r].x = flip(a.c[r].x, bwd);
#pragma unroll
        for (int o = 32 / S; o < 32; o <<= 1) {
            a.c[r].x += __shfl_xor_sync(0xffffffffu, a.c[r].x, o);
            a.c[r].y += __shfl_xor_sync(0xffffffffu, a.c[r].y, o);
        }
    }
}

template <class A>
struct LaneField {
    Geom g;
    const typename A::TL* fat;
    const typename A::TL* lng;
    float2 lng_s;  // NAIK == 2: 1 / scale of the two-row Naik links
};

// The hops of one sign along directions mu0 .. mu0 + N - 1.
template <class A, int NAIK, int N>
__device__ __forceinline__ void lane_directions(const LaneField<A>& f, int P, const typename A::T* in, int i, int x,
                                                int y, int z, int t, int mu0, bool bwd, typename A::Acc& acc) {
    // float-float and FP64 hops are several hundred instructions each: a rolled loop
    constexpr int kUnroll = std::is_same<typename A::C, float2>::value ? N : 1;
    constexpr int EF = A::kEntries, EL = NAIK == 2 ? 6 : 9;
    using AL = typename std::conditional<NAIK == 2 && std::is_same<A, ArithF32>::value, ArithF32R, A>::type;
    const Geom& g = f.g;
    const size_t vs = (size_t)g.vs;
    const int plane = (bwd ? 1 - P : P) * 4;
#pragma unroll kUnroll
    for (int m = 0; m < N; ++m) {
        const int mu = mu0 + m;
        const int c = mu == 0 ? x : mu == 1 ? y : mu == 2 ? z : t;
        const int L = mu == 0 ? g.lx : mu == 1 ? g.ly : mu == 2 ? g.lz : g.lt;
        const int stride = g.lxh * (mu == 1 ? 1 : mu == 2 ? g.ly : g.ly * g.lz);
        auto nbr = [&](int h) {
            const int c2 = bwd ? wrap_dn(c, h, L) : wrap_up(c, h, L);
            return mu == 0 ? i - (x >> 1) + (c2 >> 1) : i + (c2 - c) * stride;
        };
        const bool odd = ((mu >= 1 ? x : 0) + (mu >= 2 ? y : 0) + (mu >= 3 ? z : 0)) & 1;
        const int n1 = nbr(1);
        lane_hop<A, EF>(acc, f.fat + (size_t)((plane + mu) * EF) * vs, bwd ? n1 : i, in, n1, vs, bwd,
                        make_float2(odd ? -1.f : 1.f, 0.f));
        if constexpr (NAIK != 0) {
            const int n3 = nbr(mu == 0 ? g.hop3[0] : mu == 1 ? g.hop3[1] : mu == 2 ? g.hop3[2] : g.hop3[3]);
            lane_hop<AL, EL>(acc, f.lng + (size_t)((plane + mu) * EL) * vs, bwd ? n3 : i, in, n3, vs, bwd,
                             odd ? make_float2(-f.lng_s.x, -f.lng_s.y) : f.lng_s);
        }
    }
}

// (D in)(i), i of parity P at (x, y, z, t), from zero: lane part's share summed over the
// site's S lanes, in all of them.  One lane (S = 1) takes the backward hops first.
template <class A, int NAIK, int S>
__device__ __forceinline__ void lane_site(const LaneField<A>& f, int P, const typename A::T* in, int i, int x, int y,
                                          int z, int t, int part, bool active, typename A::Acc& acc) {
    A::zero(acc);
    if constexpr (S == 1) {
        if (active) {
            if constexpr (std::is_same<typename A::C, float2>::value) {
                lane_directions<A, NAIK, 4>(f, P, in, i, x, y, z, t, 0, true, acc);
                lane_sums<1>(acc, true);
                lane_directions<A, NAIK, 4>(f, P, in, i, x, y, z, t, 0, false, acc);
            } else {
#pragma unroll 1
                for (int bwd = 1; bwd >= 0; --bwd) {
                    lane_directions<A, NAIK, 4>(f, P, in, i, x, y, z, t, 0, bwd, acc);
                    lane_sums<1>(acc, bwd);
                }
            }
        }
    } else {
        if (active)
            lane_directions<A, NAIK, 8 / S>(f, P, in, i, x, y, z, t, S == 2 ? 0 : (part >> 1) * (8 / S), part & 1, acc);
        lane_sums<S>(acc, part & 1);
    }
}

}  // namespace stag
