// Whole solves A X = varphi (Eq. linsys) in one launch: CG or preconditioned CG (P of Eq. precon), in
// complex64 with FP64 reliable updates or in complex128, by teams of blocks.
//
// Every (chain, right-hand side) pair is a system of its own, so it gets its own team of T resident
// blocks with its own barrier, scalars and stopping test; nothing waits for another pair. (With one
// barrier for all pairs, every pair of a 64-chain batch stood still for each other pair's reliable
// updates, 225 of them in a solve.) A team is a thread-block cluster where the system is small, else blocks
// of a cooperative launch.
//
// Small lattices are bound by latency, a launch or a barrier after every few microseconds of work: with a
// launch per step and the host reading flags an iteration took 27 to 60 us (CG, PCG) whatever the size, here
// 4 to 8 and 13 to 27 up to some 30000 sites. From about 10^5 sites memory bounds complex64 and the FP64 pipe
// complex128.
//
// Work is dealt in items, one band's two spin components of one site (16 bytes in complex64): a block
// owns a contiguous range of its pair's 2 V items, or, for the preconditioned phases, whole (time
// slice, band) planes. Phases of one iteration, separated by team barriers:
//   CG, complex64   p = r + beta p_old formed at each item and its neighbours on the fly, t_ =
//                   D^dagger p, <p, A p> = ||t_||^2 | q = D t_ (never stored), x, r, ||r||^2
//   CG, complex128  t_ = D^dagger p | q, x, r | p = r + beta p: the FP64 pipe bounds it, so that p is
//                   not formed seven times
//   PCG             t_ = D^dagger p | q, x, r of a plane, then its (x, y) FFT in shared memory | tau
//                   FFT, P-hat, inverse, <r, z> | inverse (x, y) FFT, p = z + beta p
// Each block sums its team's partials itself, in the same order, so all blocks hold the same scalars
// and take the same decisions: no scalar kernel, no flag to read back, no host in the loop.
// Vectors that other blocks write are read with plain loads: the barrier's acquire drops the SM's L1
// lines, and within a phase L1 then serves the neighbours (read through L2 instead, 14 site loads per site
// in the first phase, and with FP64 sums, an iteration of the 64-chain batch took 0.37 ms against 0.17).
//
// A cooperative team's barrier spins on a counter with a time limit; a block that gives up sets the device
// error word and returns.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "dft_smem.cuh"
#include "fft_ct.h"
#include "internal.h"
#include "team.h"

namespace hmc {

template <typename R> struct It { cplx<R> s[2]; };   // one band of one site: its two spin components
// (n: items of the vector, for the index checks of the bounds build)

template <typename R> __device__ __forceinline__ It<R> ld_it(const cplx<R>* v, int64_t i, int64_t n) {
    It<R> o{};
    if (!HMC_IN(i >= 0 && i < n, kBndTeam)) return o;
    if constexpr (sizeof(R) == 4) {
        const float4 a = *reinterpret_cast<const float4*>(v + 2 * i);
        o.s[0] = make_float2(a.x, a.y);
        o.s[1] = make_float2(a.z, a.w);
    } else {
        o.s[0] = v[2 * i];
        o.s[1] = v[2 * i + 1];
    }
    return o;
}
template <typename R> __device__ __forceinline__ void st_it(cplx<R>* v, int64_t i, int64_t n, const It<R>& o) {
    if (!HMC_IN(i >= 0 && i < n, kBndTeam)) return;
    if constexpr (sizeof(R) == 4) {
        *reinterpret_cast<float4*>(v + 2 * i) = make_float4(o.s[0].x, o.s[0].y, o.s[1].x, o.s[1].y);
    } else {
        v[2 * i] = o.s[0];
        v[2 * i + 1] = o.s[1];
    }
}
template <typename R> __device__ __forceinline__ It<R> axpy_it(R a, const It<R>& x, const It<R>& y) {
    It<R> o;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        o.s[s].x = fma(a, x.s[s].x, y.s[s].x);
        o.s[s].y = fma(a, x.s[s].y, y.s[s].y);
    }
    return o;
}

// Two orders of a vector's items. Site-major, the public layout: 2 s + band. Band-major (BM), the vectors of the
// preconditioned solver: (2 t + band) L^2 + y L + x, so that a (slice, band) plane is one run.
__device__ __forceinline__ int to_bm(const BChainDev& g, int i) {
    const int s = i >> 1, t = fdiv(s, g.dLL);
    return (2 * t + (i & 1)) * g.LL + (s - t * g.LL);
}
__device__ __forceinline__ int from_bm(const BChainDev& g, int i) {
    const int q = fdiv(i, g.dLL);
    return 2 * ((q >> 1) * g.LL + (i - q * g.LL)) + (q & 1);
}

// Item i of D v (DAG = false) or D^dagger v: the stencil of site_op (common.cuh) for one band, the
// vector read through ld(item).
template <typename R, bool DAG, bool BM, typename Ld>
__device__ __forceinline__ It<R> d_item(const BChainDev& g, const Coef<R>& cf, const R* __restrict__ phi, int i,
                                        const Ld& ld, It<R>* centre = nullptr) {
    const int L = g.L, LL = g.LL, hop = 2 * ((int)g.V - LL);
    int band, s, t, rem;
    if (BM) {
        const int q = fdiv(i, g.dLL);
        band = q & 1;
        t = q >> 1;
        rem = i - q * LL;
        s = t * LL + rem;
    } else {
        band = i & 1;
        s = i >> 1;
        t = fdiv(s, g.dLL);
        rem = s - t * LL;
    }
    const int y = fdiv(rem, g.dL), x = rem - y * L;
    constexpr int u = BM ? 1 : 2;   // items per step along x
    const It<R> c = ld(i), w = ld(BM ? (band ? i - LL : i + LL) : i ^ 1);
    const It<R> xm = ld(x ? i - u : i + u * (L - 1)), xp = ld(x + 1 < L ? i + u : i - u * (L - 1));
    const It<R> ym = ld(y ? i - u * L : i + u * (LL - L)), yp = ld(y + 1 < L ? i + u * L : i - u * (LL - L));
    const int edge = DAG ? (t == 0) : (t + 1 == g.Nt);   // the time hop crosses the antiperiodic boundary
    const It<R> tn = ld(DAG ? (edge ? i + hop : i - 2 * LL) : (edge ? i - hop : i + 2 * LL));
    const R f = flip(cf.cpl, (x + y) & 1);
    const R q1 = f * __ldg(phi + s), q2 = f * __ldg(phi + g.V + s), q3 = f * __ldg(phi + 2 * g.V + s);
    const R d = band ? cf.diag[1] : cf.diag[0], hx = band ? cf.hx[1] : cf.hx[0], hy = band ? cf.hy[1] : cf.hy[0];
    It<R> o;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        o.s[q].x = fma(hx, xm.s[q].x + xp.s[q].x, fma(hy, ym.s[q].x + yp.s[q].x, flip(tn.s[q].x, edge)));
        o.s[q].y = fma(hx, xm.s[q].y + xp.s[q].y, fma(hy, ym.s[q].y + yp.s[q].y, flip(tn.s[q].y, edge)));
    }
    const cplx<R> w0 = w.s[0], w1 = w.s[1];
    o.s[0].x = fma(d, c.s[0].x, fma(q3, w0.x, fma(q1, w1.x, fma(q2, w1.y, o.s[0].x))));
    o.s[0].y = fma(d, c.s[0].y, fma(q3, w0.y, fma(q1, w1.y, fma(-q2, w1.x, o.s[0].y))));
    o.s[1].x = fma(d, c.s[1].x, fma(-q3, w1.x, fma(q1, w0.x, fma(-q2, w0.y, o.s[1].x))));
    o.s[1].y = fma(d, c.s[1].y, fma(-q3, w1.y, fma(q1, w0.y, fma(q2, w0.x, o.s[1].y))));
    if (centre) *centre = c;
    return o;
}

// Spin q of the item alone, complex128: the same operations in the same order, for blocks of up to 64 items. Their two
// warps leave half of the SM's FP64 pipe idle, a warp's operation holding its quarter for 64 clocks; an item by two
// lanes takes 19 of them instead of 35. From 96 items on all quarters are busy either way and the shared factors
// would be formed twice. Microseconds an iteration, an item a lane : a spin a lane: CG 11.6 : 10.2 at 8 x 8 x 16, 12.1 : 10.7
// at 16 x 16 x 16; PCG 21.9 : 20.7 at 4 x 4 x 8.
template <bool DAG, bool BM>
__device__ __forceinline__ double2 d_spin(const BChainDev& g, const Coef<double>& cf, const double* __restrict__ phi, int i,
                                          int q, const double2* v) {
    const int L = g.L, LL = g.LL, hop = 2 * ((int)g.V - LL), u = BM ? 1 : 2;
    int band, s, t, rem;
    if (BM) {
        const int k = fdiv(i, g.dLL);
        band = k & 1;
        t = k >> 1;
        rem = i - k * LL;
        s = t * LL + rem;
    } else {
        band = i & 1;
        s = i >> 1;
        t = fdiv(s, g.dLL);
        rem = s - t * LL;
    }
    const int y = fdiv(rem, g.dL), x = rem - y * L, other = BM ? (band ? i - LL : i + LL) : i ^ 1;
    auto at = [&](int j, int spin) {
        return HMC_IN(j >= 0 && j < 2 * (int)g.V, kBndTeam) ? v[2 * j + spin] : make_double2(0.0, 0.0);
    };
    auto ld = [&](int j) { return at(j, q); };
    const double2 c = ld(i), ws = ld(other), wo = at(other, 1 - q);
    const double2 xm = ld(x ? i - u : i + u * (L - 1)), xp = ld(x + 1 < L ? i + u : i - u * (L - 1));
    const double2 ym = ld(y ? i - u * L : i + u * (LL - L)), yp = ld(y + 1 < L ? i + u * L : i - u * (LL - L));
    const int edge = DAG ? (t == 0) : (t + 1 == g.Nt);
    const double2 tn = ld(DAG ? (edge ? i + hop : i - 2 * LL) : (edge ? i - hop : i + 2 * LL));
    const double f = flip(cf.cpl, (x + y) & 1);
    const double q1 = f * __ldg(phi + s), q2 = flip(f * __ldg(phi + g.V + s), q), q3 = flip(f * __ldg(phi + 2 * g.V + s), q);
    const double d = band ? cf.diag[1] : cf.diag[0], hx = band ? cf.hx[1] : cf.hx[0], hy = band ? cf.hy[1] : cf.hy[0];
    const double hr = fma(hx, xm.x + xp.x, fma(hy, ym.x + yp.x, flip(tn.x, edge)));
    const double hi = fma(hx, xm.y + xp.y, fma(hy, ym.y + yp.y, flip(tn.y, edge)));
    return make_double2(fma(d, c.x, fma(q3, ws.x, fma(q1, wo.x, fma(q2, wo.y, hr)))),
                        fma(d, c.y, fma(q3, ws.y, fma(q1, wo.y, fma(-q2, wo.x, hi)))));
}
constexpr int kSpinItems = 64;   // most items of a block for d_spin

// Per-thread sum of squares: FP64, or an FP32 pair with exact products and compensated additions (48
// bits, as long as the squares stay well inside FP32's range: Scale). Converting every component of an FP32
// vector for an FP64 sum takes more of the FP64 pipe's time (two lanes a clock per SM) than the rest of a phase
// takes.
template <typename R> struct Sum2;
template <> struct Sum2<double> {
    using T = double;
    double v = 0.0;
    __device__ __forceinline__ void add(double w, double x) { v = fma(w * x, x, v); }
    __device__ __forceinline__ void sq(double x) { v = fma(x, x, v); }
    __device__ __forceinline__ void plus(const Sum2& o) { v += o.v; }
    __device__ __forceinline__ unsigned long long bits() const { return (unsigned long long)__double_as_longlong(v); }
    __device__ __forceinline__ void from(unsigned long long b) { v = __longlong_as_double((long long)b); }
    __device__ __forceinline__ double get() const { return v; }
};
template <> struct Sum2<float> {
    using T = float;
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void term(float p, float e) {   // += p + e
        const float s = __fadd_rn(hi, p), b = __fsub_rn(s, hi);
        lo = __fadd_rn(lo, __fadd_rn(e, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(p, b))));
        hi = s;
    }
    __device__ __forceinline__ void sq(float x) {
        const float p = __fmul_rn(x, x);
        term(p, __fmaf_rn(x, x, -p));
    }
    __device__ __forceinline__ void add(float w, float x) {   // w x^2, w x rounded once
        const float y = __fmul_rn(w, x), p = __fmul_rn(y, x);
        term(p, __fmaf_rn(y, x, -p));
    }
    __device__ __forceinline__ void plus(const Sum2& o) { term(o.hi, o.lo); }
    __device__ __forceinline__ unsigned long long bits() const {
        return (unsigned long long)__float_as_uint(hi) << 32 | __float_as_uint(lo);
    }
    __device__ __forceinline__ void from(unsigned long long b) {
        hi = __uint_as_float((unsigned)(b >> 32));
        lo = __uint_as_float((unsigned)b);
    }
    __device__ __forceinline__ double get() const { return (double)hi + (double)lo; }
};
template <typename S> __device__ __forceinline__ void warp_plus(S& a, int from_lane_bit) {   // xor tree below the bit
    for (int o = from_lane_bit; o > 0; o >>= 1) {
        S b;
        b.from(__shfl_xor_sync(0xffffffffu, a.bits(), o));
        a.plus(b);
    }
}
template <typename R> __device__ __forceinline__ void sq_it(Sum2<R>& a, const It<R>& o) {
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        a.sq(o.s[s].x);
        a.sq(o.s[s].y);
    }
}

// Scalars of the recurrence: FP64, or an FP32 pair (48 bits) in complex64, where they end in an FP32 alpha or
// beta: one thread works on them while the rest wait, and an FP64 operation takes 65 clocks, a division 570. Of
// 3200 quotients of random sums of 512 to 442368 squares, pairs and FP64 gave the same FP32 number in all (the sums'
// own errors: 1e-14 and 3e-16 at most).
template <typename R> struct Num;
template <> struct Num<double> {
    double v;
    __device__ __forceinline__ Num() {}
    __device__ __forceinline__ Num(double x) : v(x) {}
    __device__ __forceinline__ Num(const Sum2<double>& a) : v(a.v) {}
    __device__ __forceinline__ double get() const { return v; }
    __device__ __forceinline__ bool finite() const { return isfinite(v); }
    __device__ __forceinline__ bool positive() const { return v > 0.0; }
    __device__ __forceinline__ Num times(const Num& s) const { return Num(v * s.v); }
};
template <> struct Num<float> {
    float hi, lo;
    __device__ __forceinline__ Num() {}
    __device__ __forceinline__ Num(double x) : hi((float)x), lo((float)(x - (double)(float)x)) {}
    __device__ __forceinline__ Num(const Sum2<float>& a) {
        hi = __fadd_rn(a.hi, a.lo);
        lo = __fadd_rn(__fsub_rn(a.hi, hi), a.lo);
    }
    __device__ __forceinline__ double get() const { return (double)hi + (double)lo; }
    __device__ __forceinline__ bool finite() const { return isfinite(hi); }
    __device__ __forceinline__ bool positive() const { return hi > 0.f; }
    __device__ __forceinline__ Num times(const Num& s) const {
        Num o;
        o.hi = __fmul_rn(hi, s.hi);
        o.lo = __fmaf_rn(hi, s.hi, -o.hi) + __fmaf_rn(hi, s.lo, __fmul_rn(lo, s.hi));
        return o;
    }
};
__device__ __forceinline__ double quot(const Num<double>& a, const Num<double>& b) { return a.v / b.v; }
// a / b rounded to FP32: the FP32 quotient and its remainder's, or FP64 where FP32 does not reach
__device__ __forceinline__ float quot(const Num<float>& a, const Num<float>& b) {
    if (!(fabsf(b.hi) > 1e-30f && fabsf(b.hi) < 1e30f && fabsf(a.hi) > 1e-30f && fabsf(a.hi) < 1e30f))
        return (float)(a.get() / b.get());
    const float q = a.hi / b.hi;
    const float rem = __fmaf_rn(-q, b.hi, a.hi) + __fmaf_rn(-q, b.lo, a.lo);
    return q + rem / b.hi;
}

struct NoSum {   // a barrier without a sum
    using T = float;
    __device__ __forceinline__ void plus(const NoSum&) {}
    __device__ __forceinline__ unsigned long long bits() const { return 0; }
    __device__ __forceinline__ void from(unsigned long long) {}
    __device__ __forceinline__ double get() const { return 0.0; }
};

// Complex64 systems are iterated in units of 2^-e, a power of two that keeps the sums of squares, FP32 pairs with
// FP32's range, away from its ends: squares that lose their low bits below 2^-102, sums that overflow. e follows the
// true residual at the start and at each reliable update, and changes only when a component's mean square has left
// 2^-60 .. 2^30: 2^-20 each for the fall until the next update and for ||D^dagger p||^2 against ||p||^2, 2^97 for
// the number of terms, transforms without their scale and P-hat. A power of two changes no mantissa, so the
// iterates are those of an unlimited range, bit for bit.
struct Scale {
    int e;             // the iterated vectors are 2^e times the system's
    float s, change;   // 2^e; factor from the units of the vectors in memory, 1 unless e has just changed
    double s2, inv;    // 2^(2 e), 2^-e
    __device__ __forceinline__ static double pow2(int k) { return __hiloint2double((1023 + k) << 20, 0); }
    __device__ __forceinline__ void set(int k) {
        change = (float)pow2(k - e);
        e = k;
        s = (float)pow2(k);
        s2 = pow2(2 * k);
        inv = pow2(-k);
    }
    // for the norm r2, finite and in the system's units, of n items (4 components each)
    __device__ __forceinline__ void follow(double r2, int n) {
        change = 1.f;
        if (!(r2 > 0.0)) return;
        const int at = ((__double2hiint(r2) >> 20) - 1023) - (33 - __clz(n));   // exponent of the mean square
        if (at + 2 * e < -60 || at + 2 * e > 30) set(max(max(-100, e - 100), min(min(100, e + 100), -at / 2)));
    }
};

// ---- team ------------------------------------------------------------------------------------------
// A solve's state, in shared memory, written by one thread.
template <typename R> struct Ctl {
    double b2, r2true;         // ||b||^2, the last true ||r||^2
    double stop, ru_below;     // tol^2 ||b||^2 and the ||r||^2 at which a reliable update is due, times scale.s2
    Scale scale;
    Num<R> rr;
    R alpha, beta;
    int it, n_ru, hold, wait;
    int active, nonfinite, met, ru, last;
    int ok;
};

struct Team {
    int b0, T, rank;            // first block, blocks, this block's place
    unsigned* cnt;              // arrivals, never reset within a launch
    unsigned long long* part;   // [2][gridDim.x] partial sums, by the barrier's parity
    unsigned long long* cpart;  // [2][16], shared memory: the same for a cluster
    unsigned epoch;
    int warps;                  // warps of a block with values in a sum (FP64), the rest hold zeros
    bool never;                 // the next barrier waits for more arrivals than there are blocks (timeout test)
    bool shared_sm;             // other blocks may be at work on this SM
    int* flags;
    long long timeout_ns;
};

__device__ __forceinline__ long long gtimer() {
    long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Waits for `want` arrivals (one lane). An acquiring load drops the SM's L1 lines, other blocks' too, so
// where others share the SM the polls are relaxed with one fence after them (0.3 us more).
__device__ __forceinline__ bool wait_arrivals(const Team& tm, unsigned want) {
    long long t0 = 0;
    for (unsigned n = 1;; ++n) {
        unsigned v;
        if (tm.shared_sm) asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(tm.cnt) : "memory");
        else asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(tm.cnt) : "memory");
        if ((int)(v - want) >= 0) break;
        if ((n & 63) == 0) {
            const long long now = gtimer();
            if (t0 == 0) t0 = now;
            else if (now - t0 > tm.timeout_ns) {
                atomicOr(tm.flags, 1);
                return false;
            }
        }
    }
    if (tm.shared_sm) asm volatile("fence.acq_rel.gpu;" ::: "memory");
    return true;
}

// Hardware barrier of a cluster's blocks: shared memory written before it, own or remote, is seen after it.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Barrier of the team's blocks with the sum of `acc` over all their threads; writes before it are seen by
// plain loads after it. All blocks add in the same order; lane 0 then runs fin(sum) for everybody. False
// (with the error word set) when the wait gives up.
//  CLU: the team is a thread-block cluster; partials go to every block's shared memory and the hardware
//       barrier orders them: 0.4 thousand clocks, 1.5 with the data's way through L2.
//  otherwise: an arrival counter in L2, 2.5 to 3.2 thousand clocks for 16 to 150 blocks, and 0.7 for the
//       partials. (Blocks that post their partial with the barrier's epoch in one 16-byte word for all the
//       others to poll save the second read, but took 4.5 to 5.9 from 50 blocks on.)
template <bool CLU, typename S, typename C, typename Fin>
__device__ __forceinline__ bool sync_sum(Team& tm, C& ctl, unsigned long long* red, S acc, const Fin& fin) {
    constexpr bool k64 = sizeof(typename S::T) == 8;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if constexpr (k64) {
        red[threadIdx.x] = acc.bits();
    } else {
        warp_plus(acc, 16);
        if (lane == 0) red[w] = acc.bits();
    }
    __syncthreads();
    ++tm.epoch;
    const int par = tm.epoch & 1;
    if (w == 0) {
        if constexpr (k64) {
            // one warp adds the block's values: in the shuffle tree of every warp each addition would take
            // the SM's FP64 pipe 16 clocks a warp; 64 clocks a warp of values here, so small systems skip the empty ones
            for (int j = 1; j < tm.warps; ++j) {
                S o;
                o.from(red[lane + 32 * j]);
                acc.plus(o);
            }
            warp_plus(acc, 16);
        } else {
            acc = S();
            if (lane < nw) acc.from(red[lane]);
            warp_plus(acc, nw > 8 ? 8 : 4);   // 8 or 16 warps
        }
        if constexpr (CLU) {
            if (lane < tm.T) {
                const unsigned mine = (unsigned)__cvta_generic_to_shared(tm.cpart + 16 * par + tm.rank);
                unsigned theirs;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(theirs) : "r"(mine), "r"(lane));
                asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(theirs), "l"(acc.bits()) : "memory");
            }
            __syncwarp();   // the barrier's .aligned form wants the whole warp
        }
    }
    bool ok = true;
    if constexpr (CLU) {
        cluster_sync();
        if (w == 0) {
            acc = S();
            if (lane < tm.T) acc.from(tm.cpart[16 * par + lane]);
            warp_plus(acc, 8);
        }
    } else if (w == 0 && (tm.T > 1 || tm.never)) {
        unsigned long long* row = tm.part + par * gridDim.x + tm.b0;
        if (lane == 0) {
            __stcg(row + tm.rank, acc.bits());
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(tm.cnt) : "memory");
            ok = wait_arrivals(tm, tm.epoch * tm.T + (tm.never ? 1u << 20 : 0u));
        }
        ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
        __syncwarp();
        if (!std::is_same<S, NoSum>::value) {
            // eight loads in flight: one after the other they took 0.7 thousand clocks each
            acc = S();
            for (int b = lane; b < tm.T; b += 256) {
                unsigned long long v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = b + 32 * j < tm.T ? __ldcg(row + b + 32 * j) : 0ull;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (32 * j >= tm.T) break;
                    S o;
                    o.from(v[j]);
                    acc.plus(o);
                }
            }
            warp_plus(acc, 16);
        }
    }
    if (w == 0 && lane == 0) {
        ctl.ok = ok ? 1 : 0;
        if (ok) fin(acc);
    }
    __syncthreads();
    tm.never = false;
    return ctl.ok != 0;
}

// ---- FFTs of the preconditioned phases ---------------------------------------------------------------
// Shared tables of the preconditioned phases, behind the FFT tile; cosk and ew by position after the
// forward steps.
template <typename R> struct PreTab {
    using C = cplx<R>;
    C *tile, *twx, *twt, *twist, *ew;
    R* cosk;
};
template <typename R> __device__ __forceinline__ PreTab<R> pre_tables(const TeamPre<R>& q, int L, int Nt, unsigned char* sm) {
    PreTab<R> p;
    using C = cplx<R>;
    p.tile = reinterpret_cast<C*>(sm);
    p.twx = p.tile + q.tile;
    p.twt = p.twx + L;
    p.twist = p.twt + Nt;
    p.ew = p.twist + Nt;
    p.cosk = reinterpret_cast<R*>(p.ew + Nt);
    for (int i = threadIdx.x; i < L; i += blockDim.x) {
        p.twx[i] = __ldg(q.twx + i);
        p.cosk[i] = __ldg(q.cosk + dft_freq(i, q.x1, q.x2));
    }
    for (int i = threadIdx.x; i < Nt; i += blockDim.x) {
        p.twt[i] = __ldg(q.twt + i);
        p.twist[i] = __ldg(q.twist + i);
        p.ew[i] = __ldg(q.eitw + dft_freq(i, q.t1, q.t2));
    }
    __syncthreads();
    return p;
}
__device__ __forceinline__ int row_stride(int L) { return L | 1; }   // odd: rows fall in distinct banks

// Planes of the tile -> zhat: forward FFTs along x, then y, and the spectra out, band-major. Plane p is task
// t0 + p * T (slice task / 2, band task % 2).
template <typename R>
__device__ __forceinline__ void plane_forward(const TeamPre<R>& q, const PreTab<R>& p, const BChainDev& g, int t0, int T,
                                              int np, cplx<R>* z) {
    const int L = g.L, RS = row_stride(L);
    const Lines rows{np, q.plane, 2 * L, q.d2L, 1, 2 * RS}, cols{np, q.plane, 2 * L, q.d2L, 1, 2};
    __syncthreads();
    dft_forward(p.tile, rows, q.x1, q.x2, 2, p.twx);
    dft_forward(p.tile, cols, q.x1, q.x2, 2 * RS, p.twx);
    for (int e = threadIdx.x; e < np * g.LL; e += blockDim.x) {
        const int pl = fdiv(e, g.dLL), j = e - pl * g.LL, y = fdiv(j, g.dL), at = pl * q.plane + (y * RS + j - y * L) * 2;
        It<R> v;
        v.s[0] = tile_at(p.tile, at);
        v.s[1] = tile_at(p.tile, at + 1);
        st_it<R>(z, (t0 + pl * T) * g.LL + j, 2 * g.V, v);
    }
    __syncthreads();
}

// One team's solve of right-hand side k of chain g; false when a barrier gave up.
template <typename R, bool PRE, bool CLU>
__device__ __forceinline__ bool team_run(const TeamArgs<R>& a, Team& tm, Ctl<R>& c, const BChainDev& g, int k, int pair,
                                         const PreTab<R>& pt, unsigned long long* red) {
    constexpr bool kMixed = sizeof(R) == 4;
    using C = cplx<R>;
    const int64_t off = (g.off + (int64_t)k * g.V) * 4;   // complex entries
    const int n = 2 * (int)g.V;
    const int per = ((n + tm.T - 1) / tm.T + 31) & ~31;
    const int i0 = min(tm.rank * per, n), i1 = min(i0 + per, n);
    const double2 *b = a.b + off;
    double2 *x64 = a.x64 + off, *t64 = a.t64 + off;
    C *r = a.r + off, *t = a.t + off, *pold = a.pA + off, *pnew = kMixed && !PRE ? a.pB + off : a.pA + off;
    C* x;
    if constexpr (kMixed) x = a.x + off;
    else x = x64;
    C* z = PRE ? a.z + off : nullptr;
    const R* phi;
    if constexpr (kMixed) phi = g.phi32;
    else phi = g.phi64;
    if constexpr (!kMixed) {   // the largest phase's lanes
        int lanes = 2 * min(per, kSpinItems);
        lanes = max(lanes, per);
        if constexpr (PRE) lanes = max(lanes, max(max(2 * min(a.pre.np * g.LL, kSpinItems), a.pre.np * g.LL), g.Nt * a.pre.W));
        tm.warps = min((int)blockDim.x >> 5, (lanes + 31) >> 5);
    }
    auto sync = [&]() { return sync_sum<CLU>(tm, c, red, NoSum(), [](const NoSum&) {}); };
    auto in = [&](int i) { return PRE ? to_bm(g, i) : i; };   // from the public layout to the solver's
    auto ld64 = [n](const double2* v) { return [v, n](int j) { return ld_it<double>(v, j, n); }; };
    auto ldr = [n](const C* v) { return [v, n](int j) { return ld_it<R>(v, j, n); }; };

    // ---- start: r = b - A x (or b), zero directions, norms ----------------------------------------
    if (a.use_x0) {
        for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) st_it<double>(t64, i, n, d_item<double, true, false>(g, a.cf64, g.phi64, i, ld64(x64)));
        if (!sync()) return false;
    }
    {
        Sum2<double> sb, sr;
        for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
            const It<double> bb = ld_it<double>(b, i, n);
            It<double> rr = bb;
            if (a.use_x0) {
                rr = axpy_it<double>(-1.0, d_item<double, false, false>(g, a.cf64, g.phi64, i, ld64(t64)), bb);
            } else {
                st_it<double>(x64, i, n, It<double>{});
                st_it<double>(t64, i, n, It<double>{});   // D^dagger x of the zero start
            }
            It<R> rl;
#pragma unroll
            for (int s = 0; s < 2; ++s) rl.s[s] = mk<C>((R)rr.s[s].x, (R)rr.s[s].y);
            const int o = in(i);
            st_it<R>(r, o, n, rl);
            if constexpr (kMixed) st_it<R>(x, o, n, It<R>{});
            // the first direction is r (or z): the on-the-fly and the inverse-FFT forms add 0 * p
            st_it<R>(pold, o, n, !kMixed && !PRE ? rl : It<R>{});
            sq_it(sb, bb);
            sq_it(sr, rr);
        }
        if (!sync_sum<CLU>(tm, c, red, sb, [&](const Sum2<double>& v) { c.b2 = v.v; })) return false;
        if (!sync_sum<CLU>(tm, c, red, sr, [&](const Sum2<double>& v) {
                c.r2true = v.v;
                c.alpha = c.beta = (R)0;
                c.it = c.n_ru = c.hold = 0;
                c.wait = 4;
                c.stop = a.tol2 * c.b2;
                c.nonfinite = !(isfinite(c.b2) && isfinite(v.v));
                c.active = !c.nonfinite && c.b2 > 0.0 && v.v > c.stop;
                double u = v.v;
                if constexpr (kMixed) {
                    c.scale.e = 0;
                    c.scale.set(0);
                    if (c.active) c.scale.follow(v.v, n);
                    c.stop *= c.scale.s2;
                    u *= c.scale.s2;
                }
                c.rr = Num<R>(u);
                c.ru_below = kMixed ? fmax(c.stop, a.delta2 * u) : c.stop;
            }))
            return false;
    }
    // r and the old direction to the units of a scale that has just changed
    auto rescale = [&]() {
        if constexpr (kMixed) {
            const float f = c.scale.change;
            if (f != 1.f) {
                for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
                    const int o = in(i);
                    const It<R> zero{};
                    st_it<R>(r, o, n, axpy_it<R>(f, ld_it<R>(r, o, n), zero));
                    st_it<R>(pold, o, n, axpy_it<R>(f, ld_it<R>(pold, o, n), zero));
                }
                return sync();
            }
        }
        return true;
    };
    if (c.active && !rescale()) return false;

    // this block's (slice, band) planes, tasks rank, rank + T, ..., as many at a time as the tile holds
    auto each_round = [&](const auto& f) {
        const int own = tm.rank < 2 * g.Nt ? (2 * g.Nt - tm.rank + tm.T - 1) / tm.T : 0;
        for (int j = 0; j < own; j += a.pre.np) f(tm.rank + j * tm.T, min(a.pre.np, own - j));
    };
    // f(item, place in the tile) for the sites of planes t0, t0 + T, ...
    auto each_site = [&](int t0, int np, const auto& f) {
        const int RS = row_stride(g.L);
        for (int e = threadIdx.x; e < np * g.LL; e += blockDim.x) {
            const int pl = fdiv(e, g.dLL), j = e - pl * g.LL, y = fdiv(j, g.dL), xx = j - y * g.L;
            f((t0 + pl * tm.T) * g.LL + j, pl * a.pre.plane + (y * RS + xx) * 2);
        }
    };
    // spectra of r's planes
    auto forward = [&]() {
        each_round([&](int t0, int np) {
            each_site(t0, np, [&](int i, int at) {
                const It<R> v = ld_it<R>(r, i, n);
                tile_at(pt.tile, at) = v.s[0];
                tile_at(pt.tile, at + 1) = v.s[1];
            });
            plane_forward<R>(a.pre, pt, g, t0, tm.T, np, z);
        });
    };
    // tau pass in place on z; this thread's part of <r, z> (before the transforms' scale)
    auto tau = [&]() {
        const TeamPre<R>& q = a.pre;
        const int w2 = 2 * q.W, ng = (g.LL + q.W - 1) / q.W;
        const Lines ln{1, 0, w2, q.dw2, 1, 2};
        __shared__ R base_s[kTeamTau];
        Sum2<R> acc;
        for (int task = tm.rank; task < 2 * ng; task += tm.T) {
            const int band = task & 1, j0 = (task >> 1) * q.W;
            for (int p = threadIdx.x; p < q.W; p += blockDim.x) {
                const int j = min(j0 + p, g.LL - 1), y = fdiv(j, g.dL), xx = j - y * g.L;
                base_s[p] = q.c0[band] + q.chx[band] * pt.cosk[xx] + q.chy[band] * pt.cosk[y];
            }
            C* zp = z + ((int64_t)band * g.LL + j0) * 2;
            const int left = n - (band * g.LL + j0);   // items from zp on
            const int step = 2 * g.LL, live = min(q.W, g.LL - j0), ne = g.Nt * q.W;   // items
            for (int e = threadIdx.x; e < ne; e += blockDim.x) {
                const int ts = fdiv(e, q.dW), l = e - ts * q.W;
                const C w = pt.twist[ts];
                It<R> v{};
                if (l < live) v = ld_it<R>(zp, (int64_t)ts * step + l, left);
                tile_at(pt.tile, 2 * e) = cmulconj(w, v.s[0]);
                tile_at(pt.tile, 2 * e + 1) = cmulconj(w, v.s[1]);
            }
            __syncthreads();
            dft_forward(pt.tile, ln, q.t1, q.t2, w2, pt.twt);
            for (int e = threadIdx.x; e < ne; e += blockDim.x) {
                const int ts = fdiv(e, q.dW), l = e - ts * q.W;
                const C w = pt.ew[ts];
                const R re = w.x + base_s[l];
                const R ph = (R)1 / (re * re + w.y * w.y);
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const C v = tile_at(pt.tile, 2 * e + s);
                    acc.add(ph, v.x);
                    acc.add(ph, v.y);
                    tile_at(pt.tile, 2 * e + s) = mk<C>(ph * v.y, ph * v.x);   // re and im exchanged: inverse steps follow
                }
            }
            __syncthreads();
            dft_inverse(pt.tile, ln, q.t1, q.t2, w2, pt.twt);
            for (int e = threadIdx.x; e < ne; e += blockDim.x) {
                const int ts = fdiv(e, q.dW), l = e - ts * q.W;
                const C w = pt.twist[ts];
                It<R> v;
                v.s[0] = cmul(swapc(tile_at(pt.tile, 2 * e)), w);
                v.s[1] = cmul(swapc(tile_at(pt.tile, 2 * e + 1)), w);
                if (l < live) st_it<R>(zp, (int64_t)ts * step + l, left, v);
            }
            __syncthreads();
        }
        return acc;
    };
    // p = z + beta p by inverse FFTs of z's planes
    auto inverse = [&]() {
        const TeamPre<R>& q = a.pre;
        const R be = c.beta, sc = (R)q.scale;
        const int L = g.L, RS = row_stride(L);
        each_round([&](int t0, int np) {
            const Lines rows{np, q.plane, 2 * L, q.d2L, 1, 2 * RS}, cols{np, q.plane, 2 * L, q.d2L, 1, 2};
            each_site(t0, np, [&](int i, int at) {
                const It<R> v = ld_it<R>(z, i, n);
                tile_at(pt.tile, at) = swapc(v.s[0]);
                tile_at(pt.tile, at + 1) = swapc(v.s[1]);
            });
            __syncthreads();
            dft_inverse(pt.tile, cols, q.x1, q.x2, 2 * RS, pt.twx);
            dft_inverse(pt.tile, rows, q.x1, q.x2, 2, pt.twx);
            each_site(t0, np, [&](int i, int at) {
                It<R> v;
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const C d = tile_at(pt.tile, at + s);
                    v.s[s] = mk<C>(sc * d.y, sc * d.x);
                }
                st_it<R>(pold, i, n, axpy_it<R>(be, ld_it<R>(pold, i, n), v));
            });
            __syncthreads();
        });
        return sync();
    };
    const Num<R> scale(PRE ? a.pre.scale : 1.0);
    if constexpr (PRE) {
        if (c.active) {   // first direction p = z, rr = <r, z>
            forward();
            if (!sync()) return false;
            if (!sync_sum<CLU>(tm, c, red, tau(), [&](const Sum2<R>& v) {
                    c.rr = Num<R>(v).times(scale);
                    if (!c.rr.finite()) c.nonfinite = 1;
                }))
                return false;
            if (!inverse()) return false;
        }
    }

    while (c.active && !c.nonfinite) {
        // ---- t_ = D^dagger p; alpha = rr / <p, A p> ----
        Sum2<R> acc;
        if constexpr (kMixed && !PRE) {
            const R be = c.beta;
            for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
                It<R> pc;
                const It<R> o = d_item<R, true, PRE>(
                    g, a.cf, phi, i, [&](int j) { return axpy_it<R>(be, ld_it<R>(pold, j, n), ld_it<R>(r, j, n)); }, &pc);
                st_it<R>(pnew, i, n, pc);
                st_it<R>(t, i, n, o);
                sq_it(acc, o);
            }
        } else if (!kMixed && per <= kSpinItems) {
            if constexpr (!kMixed) {
                for (int e = 2 * i0 + threadIdx.x; e < 2 * i1; e += blockDim.x) {
                    const double2 o = d_spin<true, PRE>(g, a.cf, phi, e >> 1, e & 1, pold);
                    t[e] = o;
                    acc.sq(o.x);
                    acc.sq(o.y);
                }
            }
        } else {
            for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
                const It<R> o = d_item<R, true, PRE>(g, a.cf, phi, i, ldr(pold));
                st_it<R>(t, i, n, o);
                sq_it(acc, o);
            }
        }
        if (!sync_sum<CLU>(tm, c, red, acc, [&](const Sum2<R>& v) {
                const Num<R> pAp(v);
                c.alpha = (pAp.positive() && pAp.finite()) ? quot(c.rr, pAp) : (R)0;
                if (!pAp.finite()) c.nonfinite = 1;
            }))
            return false;
        // ---- q = D t_, x += alpha p, r -= alpha q, ||r||^2 (PRE: and the spectrum of r) ----
        acc = Sum2<R>();
        const R al = c.alpha;
        auto update = [&](int i) {
            const It<R> q = d_item<R, false, PRE>(g, a.cf, phi, i, ldr(t));
            const int o = PRE && !kMixed ? from_bm(g, i) : i;   // FP64 iterates in the caller's x
            st_it<R>(x, o, n, axpy_it<R>(al, ld_it<R>(pnew, i, n), ld_it<R>(x, o, n)));
            const It<R> rn = axpy_it<R>(-al, q, ld_it<R>(r, i, n));
            st_it<R>(r, i, n, rn);
            sq_it(acc, rn);
            return rn;
        };
        auto update_spin = [&](int i, int q) {
            if constexpr (!kMixed) {
                const double2 v = d_spin<false, PRE>(g, a.cf, phi, i, q, t);
                const int e = 2 * i + q, o = PRE ? 2 * from_bm(g, i) + q : e;
                const double2 pv = pnew[e], xv = x[o], rv = r[e];
                x[o] = make_double2(fma(al, pv.x, xv.x), fma(al, pv.y, xv.y));
                const double2 rn = make_double2(fma(-al, v.x, rv.x), fma(-al, v.y, rv.y));
                r[e] = rn;
                acc.sq(rn.x);
                acc.sq(rn.y);
                return rn;
            } else {
                return mk<C>(0.f, 0.f);
            }
        };
        if constexpr (PRE) {
            each_round([&](int t0, int np) {
                if (!kMixed && np * g.LL <= kSpinItems) {
                    const int RS = row_stride(g.L);
                    for (int e = threadIdx.x; e < 2 * np * g.LL; e += blockDim.x) {
                        const int pl = fdiv(e >> 1, g.dLL), j = (e >> 1) - pl * g.LL, y = fdiv(j, g.dL), xx = j - y * g.L;
                        tile_at(pt.tile, pl * a.pre.plane + (y * RS + xx) * 2 + (e & 1)) = update_spin((t0 + pl * tm.T) * g.LL + j, e & 1);
                    }
                } else {
                    each_site(t0, np, [&](int i, int at) {
                        const It<R> v = update(i);
                        tile_at(pt.tile, at) = v.s[0];
                        tile_at(pt.tile, at + 1) = v.s[1];
                    });
                }
                plane_forward<R>(a.pre, pt, g, t0, tm.T, np, z);
            });
        } else if (!kMixed && per <= kSpinItems) {
            for (int e = 2 * i0 + threadIdx.x; e < 2 * i1; e += blockDim.x) update_spin(e >> 1, e & 1);
        } else {
            for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) update(i);
        }
        if (!sync_sum<CLU>(tm, c, red, acc, [&](const Sum2<R>& sum) {
                const Num<R> r2(sum);
                const double v = r2.get();
                if (!r2.finite()) c.nonfinite = 1;
                if constexpr (!PRE) {
                    c.beta = c.rr.positive() ? quot(r2, c.rr) : (R)0;
                    c.rr = r2;
                }
                c.last = ++c.it >= a.maxit;
                // Near the rounding floor of the true residual, an update after every iteration that meets
                // the tolerance would put its noise back into the recurrence each time and hardly ever stop:
                // after one that misses, some iterations pass before the next.
                c.ru = v <= c.ru_below && (c.it >= c.hold || v > c.stop);
                c.met = c.ru && v <= c.stop;
                if (c.last) c.ru = 1;
            }))
            return false;
        if (c.nonfinite) break;
        if constexpr (kMixed && !PRE) { C* s = pold; pold = pnew; pnew = s; }
        const bool ru = c.ru;
        if (ru) {
            // ---- reliable update: x64 += x, r = b - A x64 in FP64 ----
            if constexpr (kMixed) {
                for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
                    const It<R> lo = ld_it<R>(x, in(i), n);
                    It<double> hi = ld_it<double>(x64, i, n);
                    const double inv = c.scale.inv;
#pragma unroll
                    for (int s = 0; s < 2; ++s) {
                        hi.s[s].x = fma(inv, (double)lo.s[s].x, hi.s[s].x);
                        hi.s[s].y = fma(inv, (double)lo.s[s].y, hi.s[s].y);
                    }
                    st_it<double>(x64, i, n, hi);
                    st_it<R>(x, in(i), n, It<R>{});
                }
                if (!sync()) return false;
            }
            for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) st_it<double>(t64, i, n, d_item<double, true, false>(g, a.cf64, g.phi64, i, ld64(x64)));
            if (!sync()) return false;
            Sum2<double> acc64;
            R unit = 1;
            if constexpr (kMixed) unit = c.scale.s;
            for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
                const It<double> rd =
                    axpy_it<double>(-1.0, d_item<double, false, false>(g, a.cf64, g.phi64, i, ld64(t64)), ld_it<double>(b, i, n));
                It<R> rl;
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    rl.s[s] = mk<C>((R)rd.s[s].x, (R)rd.s[s].y);
                    if (kMixed) rl.s[s] = mk<C>(unit * rl.s[s].x, unit * rl.s[s].y);
                }
                st_it<R>(r, in(i), n, rl);
                sq_it(acc64, rd);
            }
            if (!sync_sum<CLU>(tm, c, red, acc64, [&](const Sum2<double>& sum) {
                    const double v = sum.v;
                    c.r2true = v;
                    ++c.n_ru;
                    double u = v;
                    if (kMixed) u *= c.scale.s2;
                    if (!isfinite(v)) c.nonfinite = 1;
                    else if (u <= c.stop) c.active = 0;
                    else {
                        if constexpr (kMixed) {
                            const double before = c.scale.s2;
                            c.scale.follow(v, n);
                            if (c.scale.change != 1.f) {
                                u = v * c.scale.s2;
                                c.stop = c.stop / before * c.scale.s2;
                            }
                            c.ru_below = fmax(c.stop, a.delta2 * u);
                        }
                        if constexpr (!PRE) c.rr = Num<R>(u);
                        if (c.met) {
                            c.hold = c.it + c.wait;
                            c.wait = 8;
                        }
                    }
                }))
                return false;
            if (c.nonfinite || !c.active || c.last) break;
            // (PCG: z and c.rr keep the old units for the beta of the tau pass, a ratio)
            if (!rescale()) return false;
        }
        if constexpr (PRE) {
            if (!sync_sum<CLU>(tm, c, red, tau(), [&](const Sum2<R>& v) {
                    const Num<R> rz = Num<R>(v).times(scale);
                    c.beta = c.rr.positive() ? quot(rz, c.rr) : (R)0;
                    c.rr = rz;
                    if (!rz.finite()) c.nonfinite = 1;
                }))
                return false;
            if (ru) {
                // beta belongs to the recurrence (the spectrum that was in z): taken from the new residual,
                // which near the floor is larger, it would blow the old direction up
                forward();
                if (!sync()) return false;
                if (!sync_sum<CLU>(tm, c, red, tau(), [&](const Sum2<R>& v) {
                        c.rr = Num<R>(v).times(scale);
                        if (!c.rr.finite()) c.nonfinite = 1;
                    }))
                    return false;
            }
            if (c.nonfinite) break;
            if (!inverse()) return false;
        } else if constexpr (!kMixed) {
            const R be = c.beta;
            if (per <= kSpinItems) {
                for (int e = 2 * i0 + threadIdx.x; e < 2 * i1; e += blockDim.x) {
                    const C pv = pold[e], rv = r[e];
                    pold[e] = mk<C>(fma(be, pv.x, rv.x), fma(be, pv.y, rv.y));
                }
            } else {
                for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x)
                    st_it<R>(pold, i, n, axpy_it<R>(be, ld_it<R>(pold, i, n), ld_it<R>(r, i, n)));
            }
            if (!sync()) return false;
        }
    }
    if (tm.rank == 0 && threadIdx.x == 0) {
        const int f = (c.active && !c.nonfinite ? 1 : 0) | (c.nonfinite ? 2 : 0);
        if (a.fail && f) atomicOr(a.fail, f);
        if (a.stat) a.stat[pair] = TeamStat{c.r2true, c.b2, c.it, c.n_ru, f, 0};
    }
    return true;
}

// Registers: 128 for the preconditioned kernels and for FP64 (the FP64 radix steps take 196), 80 for
// complex64 CG, three blocks per SM: its phases wait on L2.
template <typename R, bool PRE, bool CLU> struct TeamBounds {
    static constexpr int threads = CLU && !(PRE && sizeof(R) == 8) ? 512 : 256;
    static constexpr int blocks = CLU ? 1 : sizeof(R) == 4 && !PRE ? 3 : 2;
};
template <typename R, bool PRE, bool CLU>
__global__ void __launch_bounds__(TeamBounds<R, PRE, CLU>::threads, TeamBounds<R, PRE, CLU>::blocks)
k_team(const __grid_constant__ TeamArgs<R> a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long red[TeamBounds<R, PRE, CLU>::threads];
    __shared__ unsigned long long cpart[2 * 16];
    __shared__ BChainDev g;
    __shared__ Ctl<R> ctl;
    // A block of a cluster writes to the others' cpart, which is theirs only once they have started.
    if constexpr (CLU) cluster_sync();
    Team tm;
    tm.part = a.part;
    tm.cpart = cpart;
    tm.warps = blockDim.x >> 5;
    tm.never = a.test_timeout != 0;
    tm.shared_sm = a.pairs != nullptr;
    tm.flags = a.flags;
    tm.timeout_ns = a.timeout_ns;
    PreTab<R> pt;
    if constexpr (PRE) pt = pre_tables<R>(a.pre, a.one.L, a.one.Nt, smem);
    const int team = a.pairs ? a.blk[blockIdx.x] : blockIdx.x / a.T;
    tm.b0 = a.pairs ? a.team[team].x : team * a.T;
    tm.T = a.pairs ? a.team[team].y : a.T;
    tm.rank = blockIdx.x - tm.b0;
    tm.cnt = a.bar + team;
    tm.epoch = 0;
    if (!a.pairs) {   // one right-hand side per team
        if (threadIdx.x == 0) g = a.one;
        __syncthreads();
        team_run<R, PRE, CLU>(a, tm, ctl, g, team, team, pt, red);
        return;
    }
    // a batch: team j solves pair j, or (queue) teams take the next pair until there is none
    if constexpr (!PRE && !CLU && sizeof(R) == 4) {
        __shared__ int entry;
        int e = team;
        do {
            if (a.queue) {
                if (tm.rank == 0 && threadIdx.x == 0) __stcg(a.next + team, atomicAdd(a.queue, 1));
                if (!sync_sum<CLU>(tm, ctl, red, NoSum(), [&](const NoSum&) { entry = __ldcg(a.next + team); })) return;
                e = entry;
            }
            if (e >= a.npairs) return;
            const TeamPair tp = a.pairs[e];
            if (threadIdx.x == 0) g = a.ch[tp.chain];
            __syncthreads();
            if (!team_run<R, PRE, CLU>(a, tm, ctl, g, tp.k, tp.chain * a.K + tp.k, pt, red)) return;
        } while (a.queue);
    }
}

unsigned int bounds_take_team() { return bounds_take_tu(); }

// ---- host --------------------------------------------------------------------------------------------
void team_geometry(BChainDev* d, const Lat& lat) {
    d->L = lat.L;
    d->Nt = lat.Nt;
    d->LL = lat.L * lat.L;
    d->V = lat.V;
    d->dL = fast_div(lat.L);
    d->dLL = fast_div(lat.L * lat.L);
}

template <typename R> static const cplx<R>* plan_tw(const FftPlan* p);
template <> const float2* plan_tw<float>(const FftPlan* p) { return p->tw32; }
template <> const double2* plan_tw<double>(const FftPlan* p) { return p->tw64; }

// Tables and splits of the preconditioned phases; false when the lattice has no two-factor split.
template <typename R> static bool pre_setup(hmc_ctx* ctx, const Lat& lat, TeamPre<R>* q) {
    const FftPlan *px = get_plan(ctx, lat.L), *ptau = get_plan(ctx, lat.Nt);
    const PcTables* pc = get_pc(ctx, lat.L, lat.Nt);
    if (!px || !ptau || !pc || !dft_split(lat.L, &q->x1, &q->x2, sizeof(R) == 8) ||
        !dft_split(lat.Nt, &q->t1, &q->t2, sizeof(R) == 8))
        return false;
    q->twx = plan_tw<R>(px);
    q->twt = plan_tw<R>(ptau);
    if constexpr (sizeof(R) == 4) {
        q->cosk = pc->cosk32;
        q->eitw = pc->eitw32;
        q->twist = pc->twist32;
    } else {
        q->cosk = pc->cosk;
        q->eitw = pc->eitw;
        q->twist = pc->twist;
    }
    const double dt = ctx->p.dtau;
    for (int s = 0; s < 2; ++s) {
        q->c0[s] = (R)(-1.0 - dt * ctx->p.mu[s]);
        q->chx[s] = (R)(-2.0 * dt * ctx->p.t_h[s]);
        q->chy[s] = (R)(-2.0 * dt * ctx->p.t_v[s]);
    }
    q->d2L = fast_div(2 * lat.L);
    q->scale = 1.0 / ((double)lat.L * lat.L * lat.Nt);   // the unnormalised transforms both ways
    q->plane = lat.L * (lat.L | 1) * 2;
    return true;
}

// Planes in the shared tile at a time and tau tiles for teams of T blocks, within `most` bytes; returns the
// dynamic shared memory, 0 when not even one plane fits.
template <typename R> static size_t pre_tiles(TeamPre<R>* q, const Lat& lat, int T, size_t most) {
    const int own = (2 * lat.Nt + T - 1) / T, LL = lat.L * lat.L;
    const size_t tables = (size_t)(lat.L + 3 * lat.Nt) * sizeof(cplx<R>) + (size_t)lat.L * sizeof(R);
    const int room = most > tables ? (int)((most - tables) / sizeof(cplx<R>)) : 0;
    q->np = std::min(own, room / q->plane);
    // as many tau tiles as blocks
    q->W = std::min({kTeamTau, std::max(2, (2 * LL + T - 1) / T), room / (2 * lat.Nt)});
    if (q->np < 1 || q->W < 2) return 0;
    q->dw2 = fast_div(2 * q->W);
    q->dW = fast_div(q->W);
    q->tile = std::max(q->np * q->plane, lat.Nt * 2 * q->W);
    return tables + (size_t)q->tile * sizeof(cplx<R>);
}

template <typename R, bool PRE, bool CLU> static int set_attr(hmc_ctx* ctx) {
    static PerDevice attr;
    uint64_t bit;
    if (!attr.pending(&bit)) return HMC_OK;
    if (PRE)
        HMC_CUDA(ctx, cudaFuncSetAttribute(k_team<R, PRE, CLU>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTeamSmem));
    if (CLU) HMC_CUDA(ctx, cudaFuncSetAttribute(k_team<R, PRE, CLU>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    attr.mark(bit);
    return HMC_OK;
}

// resident blocks of k_team<R, PRE, false> with `smem` bytes of dynamic shared memory
template <typename R, bool PRE> static int capacity(hmc_ctx* ctx, size_t smem, int* cap) {
    int rc;
    if ((rc = set_attr<R, PRE, false>(ctx))) return rc;
    const int id = (sizeof(R) == 8 ? 2 : 0) + (PRE ? 1 : 0);
    for (const TeamCap& c : ctx->team_caps)
        if (c.id == id && c.smem == smem) {
            *cap = c.blocks;
            return HMC_OK;
        }
    int bps = 0;
    HMC_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k_team<R, PRE, false>,
                                                                TeamBounds<R, PRE, false>::threads, smem));
    *cap = bps * ctx->num_sms;
    ctx->team_caps.push_back(TeamCap{id, smem, *cap});
    return HMC_OK;
}

// Cooperative launch, or one cluster per right-hand side (CLU), through the attribute form, which stream
// capture records as such a kernel node.
template <typename R, bool PRE, bool CLU>
static int launch(hmc_ctx* ctx, const TeamArgs<R>& a, int grid, size_t smem) {
    int rc;
    if ((rc = set_attr<R, PRE, CLU>(ctx))) return rc;
    // the teams' arrival counters and, behind them, the queue of a batch
    if (!CLU) HMC_CUDA(ctx, cudaMemsetAsync(a.bar, 0, ((a.pairs ? a.nteams : grid / a.T) + 1) * sizeof(unsigned), ctx->stream));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(TeamBounds<R, PRE, CLU>::threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[1];
    if (CLU) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = a.T;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    } else {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    HMC_CUDA(ctx, cudaLaunchKernelEx(&cfg, k_team<R, PRE, CLU>, a));
    HMC_LAUNCH(ctx, "k_team");
    return HMC_OK;
}

int team_batch_capacity(hmc_ctx* ctx, int* cap) { return capacity<float, false>(ctx, 0, cap); }

int team_launch_batch(hmc_ctx* ctx, const TeamArgs<float>& a, int grid) {
    return launch<float, false, false>(ctx, a, grid, 0);
}

// clusters of T blocks of k_team<R, PRE, true> that are resident at a time
template <typename R, bool PRE> static int clusters(hmc_ctx* ctx, int T, size_t smem, int* cap) {
    int rc;
    if ((rc = set_attr<R, PRE, true>(ctx))) return rc;
    const int id = 4 + 8 * T + (sizeof(R) == 8 ? 2 : 0) + (PRE ? 1 : 0);
    for (const TeamCap& c : ctx->team_caps)
        if (c.id == id && c.smem == smem) {
            *cap = c.blocks;
            return HMC_OK;
        }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)T);
    cfg.blockDim = dim3(TeamBounds<R, PRE, true>::threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = T;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    HMC_CUDA(ctx, cudaOccupancyMaxActiveClusters(cap, k_team<R, PRE, true>, &cfg));
    ctx->team_caps.push_back(TeamCap{id, smem, *cap});
    return HMC_OK;
}

// How a solve runs: clusters of T blocks, or teams of T blocks of a cooperative launch; T = 0: neither.
struct TeamPlan {
    int T = 0;
    bool cluster = false;
    size_t smem = 0;
};
template <typename R>
static int make_plan(hmc_ctx* ctx, const Lat& lat, int nrhs, int precond, TeamPre<R>* pre, TeamPlan* plan) {
    if (precond && !pre_setup<R>(ctx, lat, pre)) return HMC_OK;
    const int64_t n = 2 * lat.V;
    int cap = 0, rc;
    // A cluster where its threads have few items each, measured against a team of a cooperative launch
    // (microseconds an iteration, one right-hand side): CG in complex64 5.5 : 7.0 at 16 x 16 x 16 (8192 items,
    // one each) but 7.3 : 6.8 at 16 x 16 x 32; PCG 18.4 : 19.9 and 23.1 : 18.9 there; PCG in FP64, whose pipe
    // wants more SMs, 29.6 : 32.7 at 8 x 8 x 16 but 47.9 : 42.3 at 10 x 10 x 20; CG in FP64 16.4 : 13.9 at
    // 6 x 6 x 12. A right-hand side of one block needs no barrier beyond the block's (3.4 : 4.8 at 4 x 4 x 8).
    if constexpr (sizeof(R) == 4) {
        if (!ctx->p.test_wait_timeout && n > (precond ? 0 : 512)) {
            for (int T = 16; T >= 2; T /= 2) {
                if (n > (precond ? 512 : 768) * (int64_t)T) break;
                if (n <= 256 * (int64_t)T && T > 2 && (!precond || 2 * lat.Nt <= T / 2)) continue;   // half as many do
                if (precond && !(plan->smem = pre_tiles<R>(pre, lat, T, kTeamSmem))) continue;
                if ((rc = precond ? clusters<R, true>(ctx, T, plan->smem, &cap) : clusters<R, false>(ctx, T, 0, &cap)))
                    return rc;
                if (cap < nrhs) continue;   // the others would run one after another
                plan->T = T;
                plan->cluster = true;
                return HMC_OK;
            }
        }
    } else {
        if (!ctx->p.test_wait_timeout && precond && n <= 2048) {
            for (int T = 16; T >= 8; T /= 2) {
                if (!(plan->smem = pre_tiles<R>(pre, lat, T, kTeamSmem))) continue;
                if ((rc = clusters<R, true>(ctx, T, plan->smem, &cap))) return rc;
                if (cap < nrhs) continue;
                plan->T = T;
                plan->cluster = true;
                return HMC_OK;
            }
        }
    }
    if (precond) {
        // shared memory for two resident blocks if a plane fits in half an SM's
        for (const int most : {kTeamSmem / 2, kTeamSmem}) {
            if (!pre_tiles<R>(pre, lat, 1 << 20, most)) continue;   // one plane
            if ((rc = capacity<R, true>(ctx, most, &cap))) return rc;
            const int tasks = 2 * lat.Nt, avail = cap / nrhs;
            if (avail < 1) return HMC_OK;
            const int rounds = (tasks + avail - 1) / avail;
            plan->T = (tasks + rounds - 1) / rounds;
            // More blocks than planes share the other phases: an SM each where the planes leave SMs idle, all that fit
            // where planes double up on some SMs (8 of 152 at 40 x 40 x 80, for which every phase waited), as long
            // as a block's threads (FP64: two warps) have an item each. Microseconds an iteration, a block per plane :
            // now: complex64 34.0 : 30.7 at 40 x 40 x 40, 40.1 : 37.9 at 40 x 40 x 80, 31.0 : 26.8 at 20 x 20 x 40 with
            // 4 right-hand sides, FP64 76.8 : 67.7 at 24 x 24 x 48, 1052 (separate kernels) : 725 at 60 x 60 x 120; with
            // less than an item a thread 20.3 : 21.1 at 20 x 20 x 40 with 2.
            const int64_t most_T = n / (sizeof(R) == 8 ? 64 : 256);
            const int alone = ctx->num_sms / nrhs;
            if (tasks <= alone) plan->T = std::max<int>(tasks, (int)std::min<int64_t>(alone, most_T));
            else if (avail <= most_T) plan->T = avail;
            plan->smem = pre_tiles<R>(pre, lat, plan->T, most);
            return HMC_OK;
        }
        return HMC_OK;
    }
    if ((rc = capacity<R, false>(ctx, 0, &cap))) return rc;
    if (sizeof(R) == 8 && n > 256 && n * nrhs <= 131072 && cap >= nrhs) {
        // A block's items take their SM's FP64 pipe 16 clocks a warp and operation: two warps of items a block, one
        // block an SM (11.6 us an iteration at 8 x 8 x 16 to 16 x 16 x 16, against 14.8 with 256 items a block;
        // past that size two blocks an SM are ahead, 359 : 403 at 80 x 80 x 160)
        plan->T = (int)std::min<int64_t>(std::max(1, std::min(cap, ctx->num_sms) / nrhs), (n + 63) / 64);
        return HMC_OK;
    }
    plan->T = (int)std::min<int64_t>(cap / nrhs, (n + 255) / 256);
    return HMC_OK;
}

template <typename R>
static int solve(hmc_ctx* ctx, const Lat& lat, const double* phi, const double2* b, double2* x, int nrhs, double tol,
                 int maxit, int precond, hmc_cg_stats* st, bool use_x0, bool* y_ready, bool* done) {
    *done = false;
    TeamArgs<R> a{};
    TeamPlan plan;
    int rc;
    if ((rc = make_plan<R>(ctx, lat, nrhs, precond, &a.pre, &plan))) return rc;
    const int T = plan.T;
    if (T < 1 || 2 * (int64_t)T * nrhs + nrhs + 1 > ctx->part_cap) return HMC_OK;
    *done = true;
    team_geometry(&a.one, lat);
    a.one.off = 0;
    a.one.phi64 = phi;
    a.one.phi32 = ctx->d_phi32;
    a.T = T;
    a.K = nrhs;
    a.cf = make_coef<R>(ctx->p);
    a.cf64 = make_coef<double>(ctx->p);
    a.b = b;
    a.x64 = x;
    a.t64 = ctx->d_z64;
    if constexpr (sizeof(R) == 4) {
        if ((rc = launch_phi_to32(ctx, phi, ctx->d_phi32, 3 * lat.V))) return rc;
        a.x = ctx->d_x32;
        a.r = ctx->d_r32;
        a.pA = ctx->d_p32;
        a.pB = ctx->d_p32b;
        a.t = ctx->d_q32;
        a.z = ctx->d_z32;
    } else {
        a.r = ctx->d_r64;
        a.pA = ctx->d_p64;
        a.t = ctx->d_q64;
        a.z = ctx->d_p64b;
    }
    a.bar = reinterpret_cast<unsigned*>(ctx->d_part);
    a.part = reinterpret_cast<unsigned long long*>(ctx->d_part) + nrhs + 1;
    a.flags = ctx->d_flags;
    // statistics in the scalars of the separate kernels, which this solve does not use
    static_assert(sizeof(TeamStat) <= sizeof(CgScalars), "statistics fit");
    a.stat = reinterpret_cast<TeamStat*>(ctx->d_cg);
    a.tol2 = tol * tol;
    a.delta2 = 1e-6;
    a.maxit = maxit;
    a.use_x0 = use_x0 ? 1 : 0;
    a.test_timeout = ctx->p.test_wait_timeout;
    // wait_spin_limit counts the strip operator's polls, microseconds of a batched solve; here it only
    // shortens the wait that a timeout test lets run out
    a.timeout_ns = a.test_timeout && ctx->p.wait_spin_limit > 0 ? (long long)ctx->p.wait_spin_limit * 1000LL
                                                                : 2000000000LL;
    const int grid = T * nrhs;
    if (plan.cluster && precond) rc = launch<R, true, true>(ctx, a, grid, plan.smem);
    else if (plan.cluster) {
        if constexpr (sizeof(R) == 4) rc = launch<R, false, true>(ctx, a, grid, 0);
    } else
        rc = precond ? launch<R, true, false>(ctx, a, grid, plan.smem) : launch<R, false, false>(ctx, a, grid, 0);
    if (rc) return rc;
    HMC_CUDA(ctx, cudaMemcpyAsync(ctx->h_cg, a.stat, nrhs * sizeof(TeamStat), cudaMemcpyDeviceToHost, ctx->stream));
    if ((rc = check_device_flags(ctx))) return rc;   // synchronises
    double worst = 0.0;
    int iters = 0, n_ru = 0, f = 0;
    for (int k = 0; k < nrhs; ++k) {
        const TeamStat& s = reinterpret_cast<const TeamStat*>(ctx->h_cg)[k];
        const double rel = s.b2 > 0.0 ? std::sqrt(s.r2true / s.b2) : 0.0;
        if (!(rel <= worst)) worst = rel;
        iters = std::max(iters, s.iters);
        n_ru = std::max(n_ru, s.n_ru);
        f |= s.flags;
    }
    if (st) {
        st->iterations = iters;
        st->reliable_updates = n_ru;
        st->converged = f == 0;
        st->true_rel_resid = worst;
    }
    if (f & 2) return fail(ctx, HMC_ERR_NONFINITE, "cg_solve: non-finite residual norm");
    if (f & 1) return fail(ctx, HMC_ERR_NOCONV, "cg_solve: no convergence in " + std::to_string(maxit) + " iterations");
    // every right-hand side stopped at a true residual of its final x, whose t_ = D^dagger x is in d_z64
    if (y_ready) *y_ready = true;
    return HMC_OK;
}

// Where one launch is the faster way (microseconds an iteration, one launch : the kernels of cg.cu):
//  CG, complex64   strip lattices 73 : 83 at 80 x 80 x 160, 73 : 82 at 64 x 64 x 128 with 2 right-hand sides, but
//                  152 : 137 with 2 at 80 x 80 x 160: past about a million sites the strip operator's traffic
//                  counts; other lattices 394 : 412 at 70 x 70 x 140 with 8
//  CG, complex128  2991 : 4300 at 80 x 80 x 160 with 8
//  PCG, complex64  lattices with compiled FFT passes 81 : 119 at 64 x 64 x 128, 136 : 168 at 48 x 48 x 96 with 4, but
//                  167 : 157 at 40 x 40 x 80 with 8; others (no compiled length) 115 : 448 at 36 x 36 x 70 with 8
//  PCG, complex128 2141 : 2445 at 80 x 80 x 160, 3636 : 4757, 6598 : 9227 and 12458 : 18307 there with 2, 4 and 8,
//                  1016 : 1194 at 40 x 40 x 80 with 4, 1600 : 2122 at 20 x 20 x 40 with 64
// On both sides of the complex64 limits: CG 68 : 77 at 48 x 48 x 96 with 5, 73 : 151 at 16 x 16 x 160 with 30, past it
// 80 : 88 at 48 x 48 x 96 with 6; PCG 139 : 136 at 40 x 40 x 80 with 7, 125 : 165 at 20 x 20 x 40 with 50, past it
// 188 : 177 at 64 x 64 x 128 with 2, 249 : 163 at 80 x 80 x 160.
static bool worth_it(hmc_ctx* ctx, const Lat& lat, int nrhs, int precond) {
    const int64_t sites = (int64_t)nrhs * lat.V;
    if (sites > (int64_t)1 << 23) return false;   // the largest measured
    if (ctx->p.solver_mode != HMC_SOLVER_MIXED) return true;
    if (precond) return sites <= 900000 || !(fftc_supported(lat.L) && fftc_can(lat.Nt, 4 * (int64_t)lat.L * lat.L));
    return sites <= 1250000 || !strip_supported(lat);
}

int team_solve(hmc_ctx* ctx, const Lat& lat, const double* phi, const double2* b, double2* x, int nrhs, double tol,
               int maxit, int precond, hmc_cg_stats* st, bool use_x0, bool* y_ready, bool* done) {
    *done = false;
    if (!worth_it(ctx, lat, nrhs, precond)) return HMC_OK;
    if (ctx->p.solver_mode == HMC_SOLVER_MIXED)
        return solve<float>(ctx, lat, phi, b, x, nrhs, tol, maxit, precond, st, use_x0, y_ready, done);
    return solve<double>(ctx, lat, phi, b, x, nrhs, tol, maxit, precond, st, use_x0, y_ready, done);
}

}  // namespace hmc
