// resident.cu - the iterations of Sec. 2, Fig. 1 in one launch, for lattices
// small enough that every site has a thread (or S threads) of its own at once: up to
// 77,824 sites of a parity in FP64 or float-float and 155,648 in FP32 arithmetic on
// 152 SMs.
//
// At these sizes an iteration of four launches is bound by the launches
// themselves, by the tail of each and by the few SMs that 256-site blocks
// reach, not by bytes.  Here a cooperative grid of at most one block per SM holds
// r, d and x of its sites in registers for the whole launch; only d and
// t = D_oe d pass through memory (L2), and the blocks meet in four exchanges per
// iteration instead of four launches:
//   t = D_oe d                 | exchange (t is visible)
//   A d = m^2 d - D_eo t       | exchange of d^dag A d: alpha
//   x += alpha d, r -= alpha Ad| exchange of |r|^2: beta, the stopping rules
//   d = r + beta d             | exchange (d is visible)
// An exchange is a counter that every block adds one to and polls with one
// thread: 1.3 to 1.5 us with 152 blocks.  (An all-to-all exchange of tagged
// values, which needs no second read, took 3.8 to 5.2 us, a collector and a
// broadcast 5.8 us; a 16-block cluster's hardware barrier 1.1 to 1.9 us.)  After it
// every block adds the blocks' partial sums in block order, so that the sum,
// alpha, beta and the decision to stop are the same bits in every block.
//
// Per iteration, before (four launches in a graph) and now: 4^4 one-hop FP64 38 -> 14.2
// us, 8^3 x 16 float-float 50 -> 15.3, FP64 91 -> 23.3, 16^4 one-hop FP32 26 -> 17.6,
// 20 x 18 x 14 x 30 FP32 43 -> 32.8 (solve times over iterations, reliable updates
// included), 16^3 x 32 float-float 104 -> 66.  Bound now: the exchanges and the FP64
// scalars below 10,000 sites (about 9 us of an iteration), L2 and the FP32 or FP64
// pipes above.
//
// Waits are bounded: a block that polls too long raises the timeout flag and
// leaves, and the host reports STAG_ERR_TIMEOUT.  The blocks then left at different
// exchanges, so the counter and its base agree no longer; the host clears both.
#include <algorithm>
#include <atomic>

#include "dirac_lanes.cuh"

namespace stag {

namespace {

// Adds one to *count, after everything the block stored, and waits (one thread)
// until it has reached target; false if it does not within `limit` polls.
__device__ __forceinline__ bool arrive_and_wait(unsigned int* count, unsigned int target, int limit) {
    unsigned int v;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(v) : "l"(count) : "memory");
    ++v;
    int polls = 0;
    while ((int)(v - target) < 0) {
        if (++polls > limit) return false;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
    }
    return true;
}

__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// -------------------------------------------- the vector steps, per arithmetic
// Own: r and d as stored; X: the solution's increment (float-float, FP32) or the
// solution (FP64); Sum: a thread's part of a dot product.
__device__ __forceinline__ double warp_sum(double s) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

__device__ __forceinline__ double sum_value(double s) { return s; }

struct StepScalars {
    double alpha, beta;
    float2 alpha_ff, beta_ff;
    int stop;
};

template <class A>
struct CgOps {  // FP32 arithmetic, vectors stored as A::T
    using T = typename A::T;
    using X = float2;
    using Sum = FFAcc;
    static constexpr bool kLow = true;
    static __device__ __forceinline__ Sum zero() { return ff_zero(); }
    static __device__ __forceinline__ T round(float2 v) {
        typename A::Acc a;
        a.c[0] = v;
        return A::store_val(a, 0);
    }
    static __device__ __forceinline__ float2 up(T v) { return ld_vec(&v); }
    static __device__ __forceinline__ void update_xr(const StepScalars& k, const T (&d)[3], const T (&ad)[3], X (&x)[3],
                                                     T (&r)[3], Sum& s) {
        const float alpha = k.alpha_ff.x;
        float acc = 0.f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float2 dd = up(d[c]), aa = up(ad[c]);
            float2 rr = up(r[c]);
            x[c].x = fmaf(alpha, dd.x, x[c].x);
            x[c].y = fmaf(alpha, dd.y, x[c].y);
            rr.x = fmaf(-alpha, aa.x, rr.x);
            rr.y = fmaf(-alpha, aa.y, rr.y);
            r[c] = round(rr);
            const float2 rq = up(r[c]);
            acc = fmaf(rq.x, rq.x, acc);
            acc = fmaf(rq.y, rq.y, acc);
        }
        s = FFAcc{acc, 0.f};
    }
    static __device__ __forceinline__ T next_d(const StepScalars& k, T d, T r) {
        const float2 dd = up(d), rr = up(r);
        return round(make_float2(fmaf(k.beta_ff.x, dd.x, rr.x), fmaf(k.beta_ff.x, dd.y, rr.y)));
    }
};
template <>
struct CgOps<ArithFF> {
    using T = float4;
    using X = float4;
    using Sum = FFAcc;
    static constexpr bool kLow = false;
    static __device__ __forceinline__ Sum zero() { return ff_zero(); }
    static __device__ __forceinline__ void update_xr(const StepScalars& k, const T (&d)[3], const T (&ad)[3], X (&x)[3],
                                                     T (&r)[3], Sum& s) {
        s = ff_zero();
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            x[c] = ff_caxpy(k.alpha_ff, d[c], x[c]);
            r[c] = ff_caxpy(ff_neg(k.alpha_ff), ad[c], r[c]);
            ff_norm2_acc(s, r[c]);
        }
    }
    static __device__ __forceinline__ T next_d(const StepScalars& k, T d, T r) { return ff_caxpy(k.beta_ff, d, r); }
};
template <>
struct CgOps<ArithF64> {
    using T = double2;
    using X = double2;
    using Sum = double;
    static constexpr bool kLow = false;
    static __device__ __forceinline__ Sum zero() { return 0.0; }
    static __device__ __forceinline__ void update_xr(const StepScalars& k, const T (&d)[3], const T (&ad)[3], X (&x)[3],
                                                     T (&r)[3], Sum& s) {
        s = 0.0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            x[c].x = fma(k.alpha, d[c].x, x[c].x);
            x[c].y = fma(k.alpha, d[c].y, x[c].y);
            r[c].x = fma(-k.alpha, ad[c].x, r[c].x);
            r[c].y = fma(-k.alpha, ad[c].y, r[c].y);
            s = fma(r[c].x, r[c].x, s);
            s = fma(r[c].y, r[c].y, s);
        }
    }
    static __device__ __forceinline__ T next_d(const StepScalars& k, T d, T r) {
        return make_double2(fma(k.beta, d.x, r.x), fma(k.beta, d.y, r.y));
    }
};

template <class A>
struct ResidentParams {
    LaneField<A> f;
    typename A::T* d;  // even
    typename A::T* t;  // odd
    typename A::T* r;  // even
    void* x;           // FP64, float-float: the solution (FP64); low precision: its increment y (FP32)
    CgScalars* scal;
    ResidentWork w;
    int iters;  // most iterations of this launch
    int fold;   // float-float: iterations between additions of the increment to x
};

// Threads of a block at most.  FP32 arithmetic takes 1024 (64 registers a thread) where
// 512 (128 registers) do not reach, the others 512.
template <class A>
constexpr int resident_threads() {
    return std::is_same<typename A::C, float2>::value ? 1024 : 512;
}

template <class A, int NAIK, int S, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) resident_kernel(const ResidentParams<A> p) {
    using Ops = CgOps<A>;
    using T = typename A::T;
    using X = typename Ops::X;
    constexpr int NS = 32 / S;
    constexpr bool kFF = std::is_same<A, ArithFF>::value;
    if (p.scal->done) return;
    // parts of a dot product, added by one warp: of every warp (FP32 types), or of every site
    // (FP64: the pipe takes 16 cycles for an addition of a warp, so no tree in every warp)
    constexpr bool kWarpSums = std::is_same<typename Ops::Sum, FFAcc>::value;
    __shared__ typename std::conditional<kWarpSums, FixedSum, double>::type s_val[THREADS / (kWarpSums ? 32 : S)];
    __shared__ StepScalars s_step;
    __shared__ CgScalars s_sc;
    __shared__ unsigned long long s_ns[4], s_t0;
    const Geom& g = p.f.g;
    const size_t vs = (size_t)g.vs;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const int nblk = gridDim.x, blk = blockIdx.x;
    const int part = lane / NS;
    // warp-sized runs of sites go round the blocks, so that few sites still reach every SM
    const int i = (warp * nblk + blk) * NS + lane % NS;
    const bool active = i < g.vh, own = active && part == 0;
    int xe = 0, xo = 0, y = 0, z = 0, t = 0;
    if (active) {
        site_coords(i, 0, g, xe, y, z, t);
        xo = xe ^ 1;  // the odd site of the same half-lattice index
    }
    T r[3], d[3], ad[3];
    X x[3];
    if (own) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            r[c] = p.r[c * vs + i];
            d[c] = p.d[c * vs + i];
            if constexpr (kFF)
                x[c] = make_float4(0.f, 0.f, 0.f, 0.f);
            else
                x[c] = static_cast<const X*>(p.x)[c * vs + i];
        }
    }
    const double m2 = p.scal->m2;
    const float2 m2_ff = p.scal->m2_ff;
    // the CG state, the same in every block (thread 0 works on it)
    CgScalars& sc = s_sc;
    if (threadIdx.x == 0) {
        sc = *p.scal;
        s_ns[0] = s_ns[1] = s_ns[2] = s_ns[3] = 0;
    }
    unsigned int target = *p.w.base;  // the counter's value when every block has arrived (thread 0)
    unsigned int n_exchange = 0;
    bool failed = false;  // (thread 0)

    // Publishes the sum over the block's sites of v (sum = true) in FP64 and waits for
    // every block; thread 0 then runs finish(total).
    auto exchange = [&](bool sum, typename Ops::Sum v, auto finish) {
        ++n_exchange;
        if (sum) {
            if constexpr (kWarpSums) {
                const FixedSum w = ff_warp_sum(v);
                if (lane == 0) s_val[warp] = w;
            } else if (part == 0) {
                s_val[warp * NS + lane] = v;
            }
        }
        __syncthreads();
        if (warp == 0) {
            double mine = 0.0;
            if (sum) {
                const int n = kWarpSums ? nwarp : nwarp * NS;
                for (int k = lane; k < n; k += 32) mine += sum_value(s_val[k]);
                for (int o = 1; o < n && o < 32; o <<= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
            }
            // two sets of slots in turn: a block is at most one exchange ahead of the slowest
            double* const slots = p.w.slots + (n_exchange & 1u) * kResidentMaxBlocks;
            if (lane == 0) {
                if (sum) slots[blk] = mine;
                target += nblk;
                failed = failed || !arrive_and_wait(p.w.count, target, p.w.polls);
            }
            __syncwarp();
            double tot = 0.0;
            if (sum) {
                for (int b = lane; b < nblk; b += 32) tot += slots[b];
                tot = warp_sum(tot);
            }
            if (lane == 0) {
                s_step.stop = 0;
                finish(tot);
                if (failed) s_step.stop = 2;
            }
        }
        __syncthreads();
    };

    const bool clock = p.w.ns != nullptr && blk == 0 && threadIdx.x == 0;
    auto lap = [&](int k) {
        if (clock) {
            const unsigned long long n = now_ns();
            s_ns[k] += n - s_t0;
            s_t0 = n;
        }
    };
    // float-float: x += the increment, which starts again at zero
    auto fold = [&]() {
        if constexpr (kFF) {
            double2* const x64 = static_cast<double2*>(p.x);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double2 a = ff_to_complex(x[c]);
                double2 xx = x64[c * vs + i];
                xx.x += a.x;
                xx.y += a.y;
                x64[c * vs + i] = xx;
                x[c] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    };
    if (clock) s_t0 = now_ns();
    for (int it = 1;; ++it) {
        {
            typename A::Acc acc;
            lane_site<A, NAIK, S>(p.f, 1, p.d, i, xo, y, z, t, part, active, acc);
            if (own) {
#pragma unroll
                for (int c = 0; c < 3; ++c) p.t[c * vs + i] = A::store_val(acc, c);
            }
        }
        exchange(false, Ops::zero(), [](double) {});
        lap(0);
        if (s_step.stop) break;
        typename Ops::Sum s = Ops::zero();
        {
            typename A::Acc acc;
            lane_site<A, NAIK, S>(p.f, 0, p.t, i, xe, y, z, t, part, active, acc);
            if (own) {
#pragma unroll
                for (int c = 0; c < 3; ++c) ad[c] = A::epilogue(acc, c, ld_vec(&d[c]), m2, m2_ff);
                s = A::dot(acc);
            }
        }
        exchange(true, s, [&](double total) {
            sc.pAp = total;
            sc.alpha = sc.delta_new / total;
            if (!(total > 0.0) || !isfinite(sc.alpha)) {
                sc.status = 4;  // STAG_ERR_BREAKDOWN
                sc.done = 1;
                sc.alpha = 0.0;
                s_step.stop = 1;
            }
            sc.alpha_ff = ff_from_double(sc.alpha);
            s_step.alpha = sc.alpha;
            s_step.alpha_ff = sc.alpha_ff;
        });
        lap(1);
        if (s_step.stop) break;
        s = Ops::zero();
        if (own) Ops::update_xr(s_step, d, ad, x, r, s);
        exchange(true, s, [&](double total) {
            sc.delta_old = sc.delta_new;
            sc.delta_new = total;
            sc.beta = total / sc.delta_old;
            sc.beta_ff = ff_from_double(sc.beta);
            sc.iter += 1;
            if (!isfinite(total)) {
                sc.status = 4;
                sc.done = 1;
            } else if (Ops::kLow) {
                const double rn = sqrt(total);
                sc.iter_since += 1;
                if (total <= sc.threshold || rn < sc.rel_delta * sc.maxr || sc.iter_since >= sc.rel_interval ||
                    sc.iter >= sc.max_iter)
                    sc.done = 2;  // reliable update due
                else
                    sc.maxr = fmax(sc.maxr, rn);
            } else {
                sc.done = (total <= sc.threshold || sc.iter >= sc.max_iter) ? 1 : 0;
            }
            s_step.beta = sc.beta;
            s_step.beta_ff = sc.beta_ff;
            s_step.stop = sc.done != 0;
        });
        lap(2);
        const bool stop = s_step.stop != 0;
        if (kFF && own && it % p.fold == 0) fold();  // as between blocks of launches
        if (stop) break;
        if (own) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                d[c] = Ops::next_d(s_step, d[c], r[c]);
                p.d[c * vs + i] = d[c];
            }
        }
        if (it == p.iters) break;
        exchange(false, Ops::zero(), [](double) {});
        lap(3);
        if (s_step.stop) break;
    }
    if (own) {
        fold();
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            p.r[c * vs + i] = r[c];
            if constexpr (!kFF) static_cast<X*>(p.x)[c * vs + i] = x[c];
        }
    }
    if (threadIdx.x == 0) {
        if (failed) {
            *p.w.timeout = 1;
            sc.done = 1;
            sc.status = 4;
        }
        if (blk == 0) {
            *p.scal = sc;
            *p.w.base = target;
            if (clock)
                for (int k = 0; k < 4; ++k) p.w.ns[k] += s_ns[k];
        }
    }
}

struct DeviceShape {
    int sms = 0;
    bool cooperative = false;
};
DeviceShape device_shape() {
    static std::atomic<int> cached[64];  // 0: not asked; else 1 + 2 * SMs + cooperative
    int dev = 0;
    DeviceShape s;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return s;
    int n = cached[dev].load(std::memory_order_relaxed);
    if (!n) {
        int sms = 0, coop = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
        n = 1 + 2 * std::min(sms, kResidentMaxBlocks) + (coop != 0);
        cached[dev].store(n, std::memory_order_relaxed);
    }
    s.sms = (n - 1) / 2;
    s.cooperative = (n - 1) % 2;
    return s;
}

// Warps of a block with S lanes per site.
int resident_warps(int vh, int S, int sms) {
    const long long warps = ((long long)vh * S + 31) / 32;
    return (int)((warps + sms - 1) / sms);
}
// Lanes per site: the most that leave every site threads of its own, since the
// more threads share a site's hops, the shorter each thread's chain of loads.
// (Measured per iteration, 8 / 4 / 2 / 1 lanes: float-float 8^3 x 16 14.6 / 17.7 /
// 20.3 / 28 us; FP64 8^3 x 16 23 / 24 / 34 / 55 us; FP32 8^3 x 16 12.5 / 13.2 / 14.9 /
// 24 us.)  Eight lanes of a site read 4 sites = 32 contiguous bytes of an FP32 plane, and
// with more than 8 warps on an SM four lanes and 64 bytes are faster: 12^3 x 16
// 14.8 us against 16.4 us.  0: the lattice is too large.
int resident_lanes(int vh, bool fp32, int max_threads, int sms) {
    for (int S : {8, 4, 2, 1}) {
        const int per = resident_warps(vh, S, sms);
        if (32 * per <= max_threads && !(fp32 && S == 8 && per > 8)) return S;
    }
    return 0;
}

template <class A, int NAIK, int S>
cudaError_t launch_lanes(ResidentParams<A> p, int sms, cudaStream_t s) {
    const int warps = (int)(((long long)p.f.g.vh * S + 31) / 32);
    const int per = resident_warps(p.f.g.vh, S, sms);
    const int blocks = (warps + per - 1) / per;
    void* args[] = {&p};
    const void* kernel = reinterpret_cast<const void*>(resident_kernel<A, NAIK, S, 512>);
    if constexpr (resident_threads<A>() > 512 && S < 8) {  // eight lanes are taken up to 8 warps only
        if (32 * per > 512) kernel = reinterpret_cast<const void*>(resident_kernel<A, NAIK, S, 1024>);
    }
    return cudaLaunchCooperativeKernel(kernel, dim3(blocks), dim3(32 * per), args, 0, s);
}

template <class A, int NAIK>
cudaError_t launch_naik(const ResidentParams<A>& p, cudaStream_t s) {
    const int sms = device_shape().sms;
    constexpr bool kFp32 = std::is_same<typename A::C, float2>::value;
    switch (resident_lanes(p.f.g.vh, kFp32, resident_threads<A>(), sms)) {
        case 8: return launch_lanes<A, NAIK, 8>(p, sms, s);
        case 4: return launch_lanes<A, NAIK, 4>(p, sms, s);
        case 2: return launch_lanes<A, NAIK, 2>(p, sms, s);
        case 1: return launch_lanes<A, NAIK, 1>(p, sms, s);
        default: return cudaErrorInvalidValue;
    }
}

template <class A>
ResidentParams<A> params(const Geom& g, const typename A::TL* fat, const typename A::TL* lng, float2 lng_s, void* d,
                         void* t, void* r, void* x, CgScalars* scal, const ResidentWork& w, int iters, int fold) {
    return ResidentParams<A>{LaneField<A>{g, fat, lng, lng_s}, static_cast<typename A::T*>(d),
                             static_cast<typename A::T*>(t),   static_cast<typename A::T*>(r),
                             x,                                scal,
                             w,                                iters,
                             fold};
}

}  // namespace

bool resident_fits(const Geom& g, bool fp32) {
    const DeviceShape s = device_shape();
    return s.cooperative && s.sms > 0 &&
           resident_lanes(g.vh, fp32, fp32 ? resident_threads<ArithF32>() : resident_threads<ArithFF>(), s.sms) != 0;
}

cudaError_t launch_resident_f64(const Geom& g, const LinkSet& L, double2* d, double2* t, double2* r, double2* x,
                                CgScalars* scal, const ResidentWork& w, int iters, cudaStream_t s) {
    const auto p = params<ArithF64>(g, L.fat64, L.lng64, make_float2(0.f, 0.f), d, t, r, x, scal, w, iters, 0);
    return L.lng64 ? launch_naik<ArithF64, 1>(p, s) : launch_naik<ArithF64, 0>(p, s);
}

cudaError_t launch_resident_ff(const Geom& g, const LinkSet& L, float4* d, float4* t, float4* r, double2* x,
                               CgScalars* scal, const ResidentWork& w, int iters, int fold, cudaStream_t s) {
    const auto p = params<ArithFF>(g, L.fatff, L.lngff, L.lng_inv_scale_ff, d, t, r, x, scal, w, iters, fold);
    if (!L.lngff) return launch_naik<ArithFF, 0>(p, s);
    return L.lng_inv_scale_ff.x != 0.f ? launch_naik<ArithFF, 2>(p, s) : launch_naik<ArithFF, 1>(p, s);
}

cudaError_t launch_resident_lo(const Geom& g, const LoLinks& L, void* d, void* t, void* r, float2* y, CgScalars* scal,
                               const ResidentWork& w, int iters, cudaStream_t s) {
    const float2 ls = make_float2(L.lng_inv_scale, 0.f);
    if (L.fat32 && L.two_row_fat)
        return launch_naik<ArithF32R, 0>(params<ArithF32R>(g, L.fat32, nullptr, ls, d, t, r, y, scal, w, iters, 0), s);
    if (L.fat32) {
        const auto p = params<ArithF32>(g, L.fat32, L.lng32, ls, d, t, r, y, scal, w, iters, 0);
        if (!L.lng32) return launch_naik<ArithF32, 0>(p, s);
        return ls.x != 0.f ? launch_naik<ArithF32, 2>(p, s) : launch_naik<ArithF32, 1>(p, s);
    }
    if (L.fatb16) {
        const auto p = params<ArithB16>(g, L.fatb16, L.lngb16, ls, d, t, r, y, scal, w, iters, 0);
        return L.lngb16 ? launch_naik<ArithB16, 1>(p, s) : launch_naik<ArithB16, 0>(p, s);
    }
    if (L.vectors32) {
        const auto p = params<ArithL16>(g, L.fat16, L.lng16, ls, d, t, r, y, scal, w, iters, 0);
        return L.lng16 ? launch_naik<ArithL16, 1>(p, s) : launch_naik<ArithL16, 0>(p, s);
    }
    const auto p = params<ArithH16>(g, L.fat16, L.lng16, ls, d, t, r, y, scal, w, iters, 0);
    return L.lng16 ? launch_naik<ArithH16, 1>(p, s) : launch_naik<ArithH16, 0>(p, s);
}

}  // namespace stag
