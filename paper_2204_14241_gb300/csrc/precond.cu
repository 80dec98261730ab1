// The preconditioner P = F~ P-hat F~^* (Eqs. twist, Kdiag, precon) in three launches for every lattice whose
// extents split into two factors and whose plane fits in shared memory, complex64 and complex128: the (x, y)
// transform of each plane, the tau pass with the twist and P-hat, and the (x, y) inverse. Lattices with compiled
// complex64 passes (fft_ct.cu) take those; the axis-by-axis kernels of fft.cu (five launches, a pass over memory
// each) serve the rest.
//
// complex64 is bound by memory and shared-memory traffic, so a tile holds both spin components of a band;
// complex128 by the FP64 pipe, and a tile holds one component, so that two blocks fit an SM at L = 80. The
// spectrum between the passes is [right-hand side][slice][component group][y][x] in the order the steps leave.
//
// Five launches became three: 9.15 ms against 13.92 at 80 x 80 x 160 with 8 right-hand sides in complex128, 0.087
// against 0.320 at 36 x 36 x 70 with 8 in complex64. Re K-hat keeps the order of operations of the axis kernels:
// as e^{i w} - (1 + ...) its cancellation at the smallest modes made errors up to three times as large.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "dft_smem.cuh"
#include "internal.h"

namespace hmc {

constexpr size_t kPSmem = 216 * 1024;

template <typename R> struct PreArgs {
    using C = cplx<R>;
    const C* src;
    C* dst;
    const C *twx, *twt, *twist;
    const double2* eitw;
    const double* cosk;
    double mu[2], tx[2], ty[2], dtau;   // K-hat = e^{i w} - 1 - dtau (mu + tx cos kx + ty cos ky)
    R scale;
    int L, Nt, LL;
    int x1, x2, t1, t2;
    int np, planes;            // planes of a block, planes in all (right-hand sides x slices x groups)
    int swap;                  // forward passes of complex128: re and im exchanged on the way in
    int W;                     // entries of a group's plane in a tau tile
    FastDiv dL, dLL, dCL, dW, dCW;   // by L, L^2, components x L, W, components x W
};

// entries of the source and the destination by address (nrhs right-hand sides of 4 V entries), for the index checks of
// the bounds build
template <typename T, typename R> __device__ __forceinline__ T* entry(T* p, T* base, const PreArgs<R>& a) {
    return in_range(p, base, (int64_t)a.planes * a.LL * (sizeof(R) == 4 ? 2 : 1), kBndPrecond);
}

template <typename R> constexpr int kComp = sizeof(R) == 4 ? 2 : 1;   // components of a group

// FWD: planes of the site layout to the spectrum, else back, times scale. Plane q = (k Nt + t) groups + group.
template <typename R, bool FWD>
__global__ void __launch_bounds__(256, 2) k_pre_xy(const __grid_constant__ PreArgs<R> a) {
    using C = cplx<R>;
    constexpr int NC = kComp<R>, G = 4 / NC;
    extern __shared__ __align__(16) unsigned char smem[];
    const int L = a.L, RS = L | 1, plane = L * RS * NC;
    const int q0 = blockIdx.x * a.np, np = min(a.np, a.planes - q0);
    C *tile = reinterpret_cast<C*>(smem), *tw = tile + a.np * plane;
    for (int i = threadIdx.x; i < L; i += blockDim.x) tw[i] = __ldg(a.twx + i);
    // f(entry of the site layout, entry of the spectrum, place in the tile), one site's components at a time
    auto each = [&](const auto& f) {
        for (int e = threadIdx.x; e < np * a.LL; e += blockDim.x) {
            const int p = fdiv(e, a.dLL), s = e - p * a.LL, y = fdiv(s, a.dL), q = q0 + p;
            f(((int64_t)(q / G) * a.LL + s) * 4 + NC * (q % G), ((int64_t)q * a.LL + s) * NC,
              p * plane + (y * RS + s - y * L) * NC);
        }
    };
    each([&](int64_t site, int64_t spec, int at) {
        const C* v = entry(a.src + (FWD ? site : spec), a.src, a);
        if constexpr (NC == 2) {
            const float4 u = *reinterpret_cast<const float4*>(v);
            tile_at(tile, at) = FWD ? mk<C>(u.x, u.y) : mk<C>(u.y, u.x);
            tile_at(tile, at + 1) = FWD ? mk<C>(u.z, u.w) : mk<C>(u.w, u.z);
        } else {
            tile_at(tile, at) = FWD && !a.swap ? *v : swapc(*v);
        }
    });
    __syncthreads();
    // lines of a plane: NC L of them; two components side by side, or rows (columns) in pairs
    const Lines rows{np, plane, NC * L, a.dCL, NC == 2 ? 1 : RS, 2 * RS}, cols{np, plane, NC * L, a.dCL, 1, 2};
    if (FWD) {
        dft_forward(tile, rows, a.x1, a.x2, NC, tw);
        dft_forward(tile, cols, a.x1, a.x2, NC * RS, tw);
    } else {
        dft_inverse(tile, cols, a.x1, a.x2, NC * RS, tw);
        dft_inverse(tile, rows, a.x1, a.x2, NC, tw);
    }
    each([&](int64_t site, int64_t spec, int at) {
        C* v = entry(a.dst + (FWD ? spec : site), a.dst, a);
        const R s = a.scale;
        if constexpr (NC == 2) {
            const C u = tile_at(tile, at), w = tile_at(tile, at + 1);
            *reinterpret_cast<float4*>(v) = FWD ? make_float4(u.x, u.y, w.x, w.y) : make_float4(s * u.y, s * u.x, s * w.y, s * w.x);
        } else {
            *v = FWD ? tile_at(tile, at) : mk<C>(s * tile_at(tile, at).y, s * tile_at(tile, at).x);
        }
    });
}

// Twist, tau transform, P-hat, inverse and twist back, in place on W sites of one group's spectrum.
template <typename R>
__global__ void __launch_bounds__(256, 2) k_pre_tau(const __grid_constant__ PreArgs<R> a, int tiles) {
    using C = cplx<R>;
    constexpr int NC = kComp<R>, G = 4 / NC;
    extern __shared__ __align__(16) unsigned char smem[];
    const int L = a.L, Nt = a.Nt, W = a.W, w = NC * W;
    const int kg = blockIdx.x / tiles, j0 = (blockIdx.x - kg * tiles) * W, live = min(W, a.LL - j0);   // (k, group), sites
    const int group = kg % G, band = group * NC / 2;
    // Re e^{iw} - 1, the rest of Re K-hat and Im e^{iw}: the real part nearly cancels at the smallest modes, so
    // complex64 keeps both of its terms as pairs of floats
    using V = std::conditional_t<NC == 2, float2, double>;
    C *tile = reinterpret_cast<C*>(smem), *tw = tile + Nt * w, *twist = tw + Nt;
    V *ewr = reinterpret_cast<V*>(twist + Nt), *base = ewr + Nt;
    R* ewi = reinterpret_cast<R*>(base + W);
    auto split = [](double v) {
        if constexpr (NC == 2) {
            const float h = (float)v;
            return make_float2(h, (float)(v - (double)h));
        } else {
            return v;
        }
    };
    for (int i = threadIdx.x; i < Nt; i += blockDim.x) {
        tw[i] = __ldg(a.twt + i);
        twist[i] = __ldg(a.twist + i);
        const double2 e = __ldg(a.eitw + dft_freq(i, a.t1, a.t2));
        ewr[i] = split(e.x - 1.0);
        ewi[i] = (R)e.y;
    }
    for (int p = threadIdx.x; p < W; p += blockDim.x) {
        const int j = min(j0 + p, a.LL - 1), y = fdiv(j, a.dL), x = j - y * L;
        base[p] = split(-a.dtau * (a.mu[band] + (a.tx[band] * __ldg(a.cosk + dft_freq(x, a.x1, a.x2)) +
                                                 a.ty[band] * __ldg(a.cosk + dft_freq(y, a.x1, a.x2)))));
    }
    C* z = a.dst + ((int64_t)(kg / G) * Nt * G + group) * a.LL * NC + (int64_t)j0 * NC;
    const int64_t step = (int64_t)G * a.LL * NC;
    __syncthreads();
    for (int e = threadIdx.x; e < Nt * W; e += blockDim.x) {
        const int t = fdiv(e, a.dW), l = e - t * W;
        const C f = twist[t];
        if constexpr (NC == 2) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (l < live) v = *reinterpret_cast<const float4*>(entry(z + t * step + 2 * l, a.dst, a));
            tile_at(tile, 2 * e) = cmulconj(f, mk<C>(v.x, v.y));
            tile_at(tile, 2 * e + 1) = cmulconj(f, mk<C>(v.z, v.w));
        } else {
            tile_at(tile, e) = l < live ? cmulconj(f, *entry(z + t * step + l, a.dst, a)) : mk<C>(0, 0);
        }
    }
    __syncthreads();
    const Lines ln{1, 0, w, a.dCW, 1, 2};
    dft_forward(tile, ln, a.t1, a.t2, w, tw);
    for (int e = threadIdx.x; e < Nt * W; e += blockDim.x) {
        const int p = fdiv(e, a.dW), l = e - p * W;
        const R im = ewi[p];
        R re;
        if constexpr (NC == 2) {
            const float2 u = ewr[p], b = base[l];
            const float s = __fadd_rn(u.x, b.x), v = __fsub_rn(s, u.x);   // s and its rounding error
            const float err = __fadd_rn(__fsub_rn(u.x, __fsub_rn(s, v)), __fsub_rn(b.x, v));
            re = s + (err + (u.y + b.y));
        } else {
            re = ewr[p] + base[l];
        }
        const R ph = (R)1 / (re * re + im * im);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const C v = tile_at(tile, NC * e + c);
            tile_at(tile, NC * e + c) = mk<C>(ph * v.y, ph * v.x);   // re and im exchanged: inverse steps follow
        }
    }
    __syncthreads();
    dft_inverse(tile, ln, a.t1, a.t2, w, tw);
    for (int e = threadIdx.x; e < Nt * W; e += blockDim.x) {
        const int t = fdiv(e, a.dW), l = e - t * W;
        if (l >= live) continue;
        const C f = twist[t];
        if constexpr (NC == 2) {
            const C u = cmul(swapc(tile_at(tile, 2 * e)), f), v = cmul(swapc(tile_at(tile, 2 * e + 1)), f);
            *reinterpret_cast<float4*>(entry(z + t * step + 2 * l, a.dst, a)) = make_float4(u.x, u.y, v.x, v.y);
        } else {
            *entry(z + t * step + l, a.dst, a) = cmul(swapc(tile_at(tile, e)), f);
        }
    }
}

// The tau transform of the twisted Fourier transforms of complex128 vectors (few and small beside the solve between
// them: launches and passes count), from the spectrum of W sites of all four components to the site layout in the order of frequencies. inverse: times the twist behind the transform, whose
// input k_pre_xy has exchanged, else its conjugate before.
__global__ void __launch_bounds__(256, 2) k_twisted_tau(const __grid_constant__ PreArgs<double> a, int tiles, int inverse) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int L = a.L, Nt = a.Nt, LL = a.LL, W = a.W;
    const int k = blockIdx.x / tiles, j0 = (blockIdx.x - k * tiles) * W, live = min(W, LL - j0);
    double2 *tile = reinterpret_cast<double2*>(smem), *tw = tile + Nt * 4 * W, *twist = tw + Nt;
    for (int i = threadIdx.x; i < Nt; i += blockDim.x) {
        tw[i] = __ldg(a.twt + i);
        twist[i] = __ldg(a.twist + i);
    }
    __syncthreads();
    const double2* z = a.src + (int64_t)k * Nt * 4 * LL + j0;
    for (int e = threadIdx.x; e < Nt * 4 * W; e += blockDim.x) {
        const int row = fdiv(e, a.dW), l = e - row * W;   // row = 4 t + component
        const double2 v = l < live ? *entry(z + (int64_t)row * LL + l, a.src, a) : make_double2(0.0, 0.0);
        tile_at(tile, e) = inverse ? v : cmulconj(twist[row >> 2], v);
    }
    __syncthreads();
    dft_forward(tile, Lines{1, 0, 4 * W, a.dCW, 1, 2}, a.t1, a.t2, 4 * W, tw);
    double2* out = a.dst + (int64_t)k * Nt * 4 * LL;
    for (int e = threadIdx.x; e < Nt * 4 * W; e += blockDim.x) {
        const int q = e >> 2, c = e & 3, p = fdiv(q, a.dW), l = q - p * W;
        if (l >= live) continue;
        const int j = j0 + l, y = fdiv(j, a.dL), x = j - y * L, n = dft_freq(p, a.t1, a.t2);
        const double2 v = tile_at(tile, (4 * p + c) * W + l), u = cscale(inverse ? cmul(swapc(v), twist[n]) : v, a.scale);
        *entry(out + ((int64_t)n * LL + dft_freq(y, a.x1, a.x2) * L + dft_freq(x, a.x1, a.x2)) * 4 + c, a.dst, a) = u;
    }
}

unsigned int bounds_take_precond() { return bounds_take_tu(); }

// ---- host --------------------------------------------------------------------------------------------
struct XyLaunch {
    unsigned blocks;
    int threads;
    size_t smem;
};
// Geometry, tables and the (x, y) passes' launch; false where the extents have no split or a plane does not fit.
template <typename R> static bool plane_args(hmc_ctx* ctx, const Lat& lat, int nrhs, PreArgs<R>* a, XyLaunch* xy) {
    constexpr int NC = kComp<R>, G = 4 / NC;
    const FftPlan *px = get_plan(ctx, lat.L), *pt = get_plan(ctx, lat.Nt);
    const PcTables* pc = get_pc(ctx, lat.L, lat.Nt);
    if (!px || !pt || !pc || !dft_split(lat.L, &a->x1, &a->x2, sizeof(R) == 8) ||
        !dft_split(lat.Nt, &a->t1, &a->t2, sizeof(R) == 8))
        return false;
    const int L = lat.L, Nt = lat.Nt, LL = L * L;
    const int64_t planes = (int64_t)nrhs * Nt * G;
    const size_t psize = (size_t)L * (L | 1) * NC * sizeof(cplx<R>), ptab = L * sizeof(cplx<R>);
    if (psize + ptab > kPSmem || planes > (1 << 30)) return false;
    // enough planes for a block's threads to have a site each, but not fewer blocks than two an SM
    a->np = (int)std::max<int64_t>(1, std::min<int64_t>({(256 + LL - 1) / LL, planes / (2 * ctx->num_sms), (int64_t)((kPSmem / 2 - ptab) / psize)}));
    a->planes = (int)planes;
    a->L = L;
    a->Nt = Nt;
    a->LL = LL;
    a->dL = fast_div(L);
    a->dLL = fast_div(LL);
    a->dCL = fast_div(NC * L);
    if constexpr (sizeof(R) == 4) {
        a->twx = px->tw32; a->twt = pt->tw32; a->twist = pc->twist32;
    } else {
        a->twx = px->tw64; a->twt = pt->tw64; a->twist = pc->twist;
    }
    a->cosk = pc->cosk;
    a->eitw = pc->eitw;
    xy->blocks = (unsigned)((planes + a->np - 1) / a->np);
    xy->threads = a->np * LL >= 256 ? 256 : 128;
    xy->smem = a->np * psize + ptab;
    return true;
}
template <typename R> static int plane_attr(hmc_ctx* ctx) {
    static PerDevice attr;
    uint64_t bit;
    if (!attr.pending(&bit)) return HMC_OK;
    for (const void* f : {(const void*)k_pre_xy<R, true>, (const void*)k_pre_xy<R, false>, (const void*)k_pre_tau<R>})
        HMC_CUDA(ctx, cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPSmem));
    if (sizeof(R) == 8)
        HMC_CUDA(ctx, cudaFuncSetAttribute(k_twisted_tau, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPSmem));
    attr.mark(bit);
    return HMC_OK;
}

template <typename R>
int precond_planes(hmc_ctx* ctx, const Lat& lat, const cplx<R>* x, cplx<R>* y, int nrhs, cplx<R>* scratch, bool* done) {
    *done = false;
    constexpr int NC = kComp<R>, G = 4 / NC;
    PreArgs<R> a{};
    XyLaunch xy;
    if (!scratch || !plane_args<R>(ctx, lat, nrhs, &a, &xy)) return HMC_OK;
    const int Nt = lat.Nt, LL = a.LL;
    const size_t col = (size_t)(Nt * NC) * sizeof(cplx<R>) + sizeof(double), ttab = (size_t)Nt * (2 * sizeof(cplx<R>) + sizeof(double) + sizeof(R));
    if (2 * col + ttab > kPSmem / 2) return HMC_OK;
    // tau tiles of 256-byte rows, narrower where they would leave SMs idle
    a.W = std::min<int>(16, (int)((kPSmem / 2 - ttab) / col));
    while (a.W > 4 && (int64_t)nrhs * G * ((LL + a.W - 1) / a.W) < 2 * ctx->num_sms) a.W /= 2;
    a.W = std::max(2, std::min(a.W, LL));
    const int tiles = (LL + a.W - 1) / a.W;
    a.dW = fast_div(a.W);
    a.dCW = fast_div(NC * a.W);
    a.dtau = ctx->p.dtau;
    for (int s = 0; s < 2; ++s) {
        a.mu[s] = ctx->p.mu[s];
        a.tx[s] = 2.0 * ctx->p.t_h[s];
        a.ty[s] = 2.0 * ctx->p.t_v[s];
    }
    a.scale = (R)(1.0 / ((double)LL * Nt));   // the unnormalised transforms both ways
    int rc;
    if ((rc = plane_attr<R>(ctx))) return rc;
    *done = true;
    a.src = x;
    a.dst = scratch;
    k_pre_xy<R, true><<<xy.blocks, xy.threads, xy.smem, ctx->stream>>>(a);
    HMC_LAUNCH(ctx, "k_pre_xy");
    k_pre_tau<R><<<(unsigned)(nrhs * G * tiles), 256, a.W * col + ttab, ctx->stream>>>(a, tiles);
    HMC_LAUNCH(ctx, "k_pre_tau");
    a.src = scratch;
    a.dst = y;
    k_pre_xy<R, false><<<xy.blocks, xy.threads, xy.smem, ctx->stream>>>(a);
    HMC_LAUNCH(ctx, "k_pre_xy");
    return HMC_OK;
}
template int precond_planes<float>(hmc_ctx*, const Lat&, const float2*, float2*, int, float2*, bool*);
template int precond_planes<double>(hmc_ctx*, const Lat&, const double2*, double2*, int, double2*, bool*);

// dst = F~ src (inverse, its order as printed: T times the inverse unitary DFT) or F~^* src, through scratch. Two
// launches for four or five of fft.cu's axis kernels: green_estimate with 8 probes 2.04 -> 2.01 ms at 16 x 16 x 32, with
// one 0.362 -> 0.343 at 4 x 4 x 8.
int twisted_planes(hmc_ctx* ctx, const Lat& lat, const double2* src, double2* dst, int nrhs, int inverse, double2* scratch,
                   bool* done) {
    *done = false;
    PreArgs<double> a{};
    XyLaunch xy;
    if (!plane_args<double>(ctx, lat, nrhs, &a, &xy)) return HMC_OK;
    a.W = std::min(4, a.LL);
    const int tiles = (a.LL + a.W - 1) / a.W;
    const size_t smem = (size_t)lat.Nt * (4 * a.W + 2) * sizeof(double2);
    if (smem > kPSmem) return HMC_OK;
    int rc;
    if ((rc = plane_attr<double>(ctx))) return rc;
    *done = true;
    a.dW = fast_div(a.W);
    a.dCW = fast_div(4 * a.W);
    a.swap = inverse;
    a.scale = 1.0 / std::sqrt((double)a.LL * lat.Nt);
    a.src = src;
    a.dst = scratch;
    k_pre_xy<double, true><<<xy.blocks, xy.threads, xy.smem, ctx->stream>>>(a);
    HMC_LAUNCH(ctx, "k_pre_xy");
    a.src = scratch;
    a.dst = dst;
    k_twisted_tau<<<(unsigned)(nrhs * tiles), 256, smem, ctx->stream>>>(a, tiles, inverse);
    HMC_LAUNCH(ctx, "k_twisted_tau");
    return HMC_OK;
}

}  // namespace hmc
