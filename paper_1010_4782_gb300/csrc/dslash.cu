// dslash.cu - half of the staggered Dirac operator on one parity
// (Sec. 2, Eqs. (4)-(5), plus the optional Naik three-hop term):
//
//   out(y) = sum_mu  U_mu(y) in(y+mu) - U_mu(y-mu)^dag in(y-mu)
//          [+ sum_mu L_mu(y) in(y+3mu) - L_mu(y-3mu)^dag in(y-3mu)]
//
// for every site y of the output parity P, with eta folded into the links.
// Forward links are read at y (parity P), backward links at the neighbour
// (parity 1-P), so each half-Dslash streams every link of the field exactly
// once.  One thread per output site; links and vectors are structure-of-
// arrays with the site index fastest (Sec. 3.1: consecutive threads read
// consecutive 16-byte words).  Each 3x3 product is accumulated straight into
// the output registers (Sec. 3.4, Eq. (smallreg)).  The neighbour vectors
// (8 or 16 reads of each input site) are served by L1/L2: a 28^3 x 96
// half-lattice FP64 vector is 50.6 MB, well inside the 126 MB L2.
//
// The arithmetics (dirac.cuh: native FP64, float-float on the FP32 pipelines, FP32 on
// FP32 and 16-bit storage) share the kernel body.
//
// Epilogues (used by A = m^2 - D_eo D_oe, Eq. (3)):
//   EPI_PLAIN  out = D in
//   EPI_AXPY   out = m2 * src - D in
//   EPI_CG     as EPI_AXPY with m2 from the CG state, plus the grid-wide
//              Re(src^dag out) = d^dag A d; the last block forms
//              alpha = delta_new / d^dag A d (Fig. 1) on the device.
#include <type_traits>

#include "dirac.cuh"

namespace stag {

// Resident 256-thread blocks per SM the register allocation is held to.  The
// float-float kernels are bound by memory latency: with up to 128 registers
// (2 blocks) the compiler keeps more of a site's loads in flight, and a
// float-float CG solve of 665 iterations at 28^3 x 96 takes 598 ms against 630 ms
// with 3 blocks (80 registers), 677 ms with 4 (64) and 798 ms with 1.  (At 24^3 x 48, 483
// iterations, 3 blocks are ahead: 153 ms, 159 with 2, 194 with 4, 200 with 1.)  The others
// keep 4 blocks (64 registers; 3 and 80 with two-row Naik links): FP64 is
// bound by its pipe and FP32 by HBM, where more registers measured no gain.
template <class A, int NAIK>
constexpr int dslash_min_blocks() {
    return std::is_same<A, ArithFF>::value ? 2 : (NAIK == 2 ? 3 : 4);
}

// The float-float kernels take their epilogue at run time (EPI = kEpiRuntime): their
// unrolled stencil is some 200 KB of code, and D_oe and D_eo as two kernels refilled the
// instruction cache at every launch (28^3 x 96: 386 and 411 us when one is repeated, 828
// us in turn, as one kernel 801 us; 24^3 x 48: 132, 147 and 311 us, as one kernel 278 us).
constexpr int kEpiRuntime = -1;

template <class A, int NAIK, int EPI>
__global__ void __launch_bounds__(kBlock, dslash_min_blocks<A, NAIK>()) dslash_kernel(const DslashParams<A> p) {
    // Inside a solver iteration (CG state given): return once the loop has
    // stopped, so that the rest of a captured block of iterations costs nothing.
    if (p.scal && p.scal->done) return;
    const int epi = EPI == kEpiRuntime ? p.epi : EPI;
    const Geom& g = p.g;
    const int i = p.i0 + blockIdx.x * kBlock + threadIdx.x;
    const size_t vs = (size_t)g.vs;
    typename A::Acc acc;
    A::zero(acc);
    const bool active = i < p.i1;
    // the epilogue's operands are loaded before the stencil, so that their
    // latency overlaps it instead of following it
    using SrcT = decltype(A::ld(p.src));
    SrcT srcv[3];
    double m2 = 0.0;
    float2 m2_ff = make_float2(0.f, 0.f);
    if (epi != EPI_PLAIN) {
        m2 = (epi == EPI_CG) ? p.scal->m2 : p.m2;
        m2_ff = (epi == EPI_CG) ? p.scal->m2_ff : p.m2_ff;
        if (active) {
#pragma unroll
            for (int r = 0; r < 3; ++r) srcv[r] = A::ld(p.src + r * vs + i);
        }
    }
    if (active) dslash_site<A, NAIK>(p, i, acc);
    if (epi == EPI_PLAIN) {
        if (active) {
#pragma unroll
            for (int r = 0; r < 3; ++r) p.out[r * vs + i] = A::store_val(acc, r);
        }
        return;
    }
    // out = m2 * src - D in
    if (active) {
#pragma unroll
        for (int r = 0; r < 3; ++r) p.out[r * vs + i] = A::epilogue(acc, r, srcv[r], m2, m2_ff);
    }
    if (epi == EPI_CG) {
        double total;
        if (grid_sum_last_block<kBlock>(A::dot(acc), p.partials, &p.scal->counter, &total)) {
            if (threadIdx.x == 0) {
                CgScalars* sc = p.scal;
                sc->pAp = total;
                const double alpha = sc->delta_new / total;
                if (!(total > 0.0) || !isfinite(alpha)) {
                    sc->status = 4;  // STAG_ERR_BREAKDOWN
                    sc->done = 1;
                    sc->alpha = 0.0;
                    sc->alpha_ff = make_float2(0.f, 0.f);
                } else {
                    sc->alpha = alpha;
                    sc->alpha_ff = ff_from_double(alpha);
                }
            }
        }
    }
}

// Half-Dslash of several systems in one launch (EPI_PLAIN or EPI_AXPY): the
// systems list[0 .. *count) take consecutive runs of kBlock-site tiles,
// prefix[j] .. prefix[j + 1] for entry j, and the grid's blocks stride over
// all of them.  The list lives on the device, so a captured graph runs
// whichever systems the kernels before it selected.
template <class A, int EPI>
__global__ void __launch_bounds__(kBlock, 3) dslash_list_kernel(const SysDirac* __restrict__ sys,
                                                               const int* __restrict__ list,
                                                               const int* __restrict__ prefix,
                                                               const int* __restrict__ count) {
    using T = typename A::T;
    using TL = typename A::TL;
    const int n = *count;
    const int total = prefix[n];
    for (int tile = blockIdx.x; tile < total; tile += gridDim.x) {
        int j = 0;
        while (prefix[j + 1] <= tile) ++j;
        const SysDirac& sd = sys[list[j]];
        const int i = (tile - prefix[j]) * kBlock + threadIdx.x;
        if (i >= sd.g.vh) continue;
        const DslashParams<A> p{sd.g,
                                sd.P,
                                static_cast<const TL*>(sd.fat),
                                static_cast<const TL*>(sd.lng),
                                static_cast<const T*>(sd.in),
                                static_cast<T*>(sd.out),
                                static_cast<const T*>(sd.src),
                                sd.m2,
                                sd.m2_ff,
                                nullptr,
                                nullptr,
                                0,
                                sd.g.vh};
        typename A::Acc acc;
        A::zero(acc);
        if (p.lng)
            dslash_site<A, 1>(p, i, acc);
        else
            dslash_site<A, 0>(p, i, acc);
        const size_t vs = (size_t)sd.g.vs;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            if (EPI == EPI_PLAIN)
                p.out[r * vs + i] = A::store_val(acc, r);
            else
                p.out[r * vs + i] = A::epilogue(acc, r, A::ld(p.src + r * vs + i), p.m2, p.m2_ff);
        }
    }
}

void launch_dslash_list(bool ff, Epilogue epi, const SysDirac* sys, const int* list, const int* prefix,
                        const int* count, int grid, cudaStream_t s) {
    if (ff) {
        if (epi == EPI_PLAIN)
            dslash_list_kernel<ArithFF, EPI_PLAIN><<<grid, kBlock, 0, s>>>(sys, list, prefix, count);
        else
            dslash_list_kernel<ArithFF, EPI_AXPY><<<grid, kBlock, 0, s>>>(sys, list, prefix, count);
    } else {
        if (epi == EPI_PLAIN)
            dslash_list_kernel<ArithF64, EPI_PLAIN><<<grid, kBlock, 0, s>>>(sys, list, prefix, count);
        else
            dslash_list_kernel<ArithF64, EPI_AXPY><<<grid, kBlock, 0, s>>>(sys, list, prefix, count);
    }
}

template <class A, int EPI>
static void launch_one(const DslashParams<A>& p, int naik, cudaStream_t s) {
    const int blocks = blocks_for(p.i1 - p.i0);
    if constexpr (std::is_same<A, ArithFF>::value || std::is_same<A, ArithF32>::value) {
        if (naik == 2) {
            dslash_kernel<A, 2, EPI><<<blocks, kBlock, 0, s>>>(p);
            return;
        }
    }
    if (naik)
        dslash_kernel<A, 1, EPI><<<blocks, kBlock, 0, s>>>(p);
    else
        dslash_kernel<A, 0, EPI><<<blocks, kBlock, 0, s>>>(p);
}

template <class A>
static void launch_any(DslashParams<A> p, int naik, Epilogue epi, cudaStream_t s) {
    if constexpr (std::is_same<A, ArithFF>::value) {
        p.epi = epi;
        launch_one<A, kEpiRuntime>(p, naik, s);
    } else {
        switch (epi) {
            case EPI_PLAIN: launch_one<A, EPI_PLAIN>(p, naik, s); break;
            case EPI_AXPY: launch_one<A, EPI_AXPY>(p, naik, s); break;
            default: launch_one<A, EPI_CG>(p, naik, s); break;
        }
    }
}

void launch_dslash_f64(const Geom& g, int out_parity, const LinkSet& L, const double2* in,
                       double2* out, Epilogue epi, const double2* src, double m2,
                       CgScalars* scal, double* partials, cudaStream_t s) {
    DslashParams<ArithF64> p{g, out_parity, L.fat64, L.lng64, in, out, src, m2,
                             make_float2(0.f, 0.f), scal, partials, 0, g.vh};
    launch_any(p, L.lng64 != nullptr, epi, s);
}

void launch_dslash_f64_range(const Geom& g, int out_parity, const LinkSet& L, const double2* in, double2* out,
                             Epilogue epi, const double2* src, double m2, int i0, int i1, cudaStream_t s) {
    if (i1 <= i0) return;
    DslashParams<ArithF64> p{g, out_parity, L.fat64, L.lng64, in, out, src, m2,
                             make_float2(0.f, 0.f), nullptr, nullptr, i0, i1};
    launch_any(p, L.lng64 != nullptr, epi, s);
}

void launch_dslash_ff(const Geom& g, int out_parity, const LinkSet& L, const float4* in,
                      float4* out, Epilogue epi, const float4* src, double m2, CgScalars* scal,
                      double* partials, cudaStream_t s) {
    DslashParams<ArithFF> p{g, out_parity, L.fatff, L.lngff, in, out, src, m2,
                            host_ff_from_double(m2), scal, partials, 0, g.vh, L.lng_inv_scale_ff};
    const bool two_row = L.lng_inv_scale_ff.x != 0.f;
    launch_any(p, L.lngff == nullptr ? 0 : two_row ? 2 : 1, epi, s);
}

void launch_dslash_f32(const Geom& g, int out_parity, const float2* fat, const float2* lng,
                       const float2* in, float2* out, Epilogue epi, const float2* src, double m2,
                       CgScalars* scal, double* partials, cudaStream_t s, float lng_inv_scale) {
    DslashParams<ArithF32> p{g, out_parity, fat, lng, in, out, src, m2, host_ff_from_double(m2), scal, partials, 0,
                             g.vh, make_float2(lng_inv_scale, 0.f)};
    launch_any(p, lng == nullptr ? 0 : lng_inv_scale != 0.f ? 2 : 1, epi, s);
}

void launch_dslash_h16(const Geom& g, int out_parity, const __half2* fat, const __half2* lng,
                       const __half2* in, __half2* out, Epilogue epi, const __half2* src, double m2,
                       CgScalars* scal, double* partials, cudaStream_t s) {
    DslashParams<ArithH16> p{g, out_parity, fat, lng, in, out, src, m2, host_ff_from_double(m2), scal, partials, 0,
                             g.vh};
    launch_any(p, lng != nullptr, epi, s);
}

void launch_dslash_b16(const Geom& g, int out_parity, const __nv_bfloat162* fat, const __nv_bfloat162* lng,
                       const __nv_bfloat162* in, __nv_bfloat162* out, Epilogue epi, const __nv_bfloat162* src,
                       double m2, CgScalars* scal, double* partials, cudaStream_t s) {
    DslashParams<ArithB16> p{g, out_parity, fat, lng, in, out, src, m2, host_ff_from_double(m2), scal, partials, 0,
                             g.vh};
    launch_any(p, lng != nullptr, epi, s);
}

void launch_dslash_f32l16(const Geom& g, int out_parity, const __half2* fat, const __half2* lng, const float2* in,
                          float2* out, Epilogue epi, const float2* src, double m2, CgScalars* scal, double* partials,
                          cudaStream_t s) {
    DslashParams<ArithL16> p{g, out_parity, fat, lng, in, out, src, m2, host_ff_from_double(m2), scal, partials, 0,
                             g.vh};
    launch_any(p, lng != nullptr, epi, s);
}

void launch_dslash_f32r12(const Geom& g, int out_parity, const float2* fat_rows2, const float2* in, float2* out,
                          Epilogue epi, const float2* src, double m2, CgScalars* scal, double* partials,
                          cudaStream_t s) {
    DslashParams<ArithF32R> p{g, out_parity, fat_rows2, nullptr, in, out, src, m2, host_ff_from_double(m2), scal,
                              partials, 0, g.vh};
    launch_any(p, false, epi, s);
}

}  // namespace stag
