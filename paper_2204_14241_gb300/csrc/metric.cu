// Fourier-diagonal metric operations of Section "Online metric estimation" on real fields, in three
// launches: the half spectrum of every (component, time slice) plane (x, then y), the tau transform with the
// spectral weight and its inverse, and the planes back (y, then x) with the output update.
//
// What bounds it is GB300's FP64 pipe (two lanes a clock per SM), so the transforms are of real data: two
// rows of a plane share one complex x transform, and y and tau run on the L / 2 + 1 columns that determine
// the spectrum, half the operations of complex transforms; packing, weights and the leapfrog update ride
// along. Integer and shared-memory work hides behind the pipe, so lengths are run-time values. At
// 80 x 80 x 160 the drift takes 0.61 ms against 1.16 with complex transforms in nine launches; its operations
// alone take 0.36 ms of the pipe, its bytes 0.01 ms. On small lattices the launches count, three against nine.
//
// The weight of a wave vector k is the mean of sigma-hat's at k and -k (its own where sigma-hat is even, as
// an estimate from real fields is): the real part that a complex transform keeps.
#include <algorithm>

#include "dft_smem.cuh"
#include "internal.h"

namespace hmc {

constexpr int kMW = 16;               // columns of a tau tile: 256-byte rows
constexpr size_t kMSmem = 216 * 1024;

// One chain's transform: geometry, splits L = x1 x2 and Nt = t1 t2, twiddles, fields and spectrum
// [component][slice][position along y][kx].
struct MetricDesc {
    int L, Nt, Hx;
    int x1, x2, t1, t2;
    FastDiv dL, dHalf, dHx;
    const double2 *twx, *twt;
    const double *in, *sig;
    double* out;
    double2* spec;
    double scale;
};

struct PlaneTiles {
    double2 *rows, *half, *tw;   // [L / 2][L | 1], [L][Hx | 1], [L]
    int* pos;                    // position of a frequency along x
};
__device__ __forceinline__ PlaneTiles plane_tiles(const MetricDesc& d, unsigned char* smem) {
    PlaneTiles p;
    p.rows = reinterpret_cast<double2*>(smem);
    p.half = p.rows + (d.L / 2) * (d.L | 1);
    p.tw = p.half + d.L * (d.Hx | 1);
    p.pos = reinterpret_cast<int*>(p.tw + d.L);
    for (int i = threadIdx.x; i < d.L; i += blockDim.x) {
        p.tw[i] = __ldg(d.twx + i);
        p.pos[i] = dft_pos(i, d.x1, d.x2);
    }
    return p;
}
static size_t plane_smem(int L) {
    return ((size_t)(L / 2) * (L | 1) + (size_t)L * ((L / 2 + 1) | 1) + L) * sizeof(double2) + L * sizeof(int);
}

// Half spectra of the planes: block (component, slice), chain blockIdx.y of the table (or `one`).
__global__ void __launch_bounds__(256, 2) k_metric_fwd(const MetricDesc* __restrict__ tab,
                                                       const __grid_constant__ MetricDesc one) {
    extern __shared__ __align__(16) unsigned char smem[];
    const MetricDesc& d = tab ? tab[blockIdx.y] : one;
    const int L = d.L, Hx = d.Hx, RA = L | 1, RB = Hx | 1;
    if ((int)blockIdx.x >= 3 * d.Nt) return;
    const PlaneTiles p = plane_tiles(d, smem);
    const double* in = d.in + (int64_t)blockIdx.x * L * L;
    // rows 2j and 2j + 1 as the real and imaginary part of one line
    for (int e = threadIdx.x; e < (L / 2) * L; e += blockDim.x) {
        const int j = fdiv(e, d.dL), x = e - j * L;
        p.rows[j * RA + x] = make_double2(__ldg(in + 2 * j * L + x), __ldg(in + (2 * j + 1) * L + x));
    }
    __syncthreads();
    dft_forward(p.rows, Lines{1, 0, L / 2, d.dHalf, RA, 2 * RA}, d.x1, d.x2, 1, p.tw);
    // twice each row's half spectrum: Z(k) + conj Z(-k) and (Z(k) - conj Z(-k)) / i
    for (int e = threadIdx.x; e < (L / 2) * Hx; e += blockDim.x) {
        const int j = fdiv(e, d.dHx), k = e - j * Hx;
        const double2 z = p.rows[j * RA + p.pos[k]], w = p.rows[j * RA + p.pos[k ? L - k : 0]];
        p.half[2 * j * RB + k] = make_double2(z.x + w.x, z.y - w.y);
        p.half[(2 * j + 1) * RB + k] = make_double2(z.y + w.y, w.x - z.x);
    }
    __syncthreads();
    dft_forward(p.half, Lines{1, 0, Hx, d.dHx, 1, 2}, d.x1, d.x2, RB, p.tw);
    double2* out = d.spec + (int64_t)blockIdx.x * L * Hx;
    for (int e = threadIdx.x; e < L * Hx; e += blockDim.x) {
        const int y = fdiv(e, d.dHx), k = e - y * Hx;
        out[e] = p.half[y * RB + k];
    }
}

// The tau transform of kMW columns of one component, the weights of `op`, and (momentum, velocity) the
// inverse, in place on the spectrum. Sums: part[blockIdx.x]; ACCUM: out += |F in|^2 at k and -k.
__global__ void __launch_bounds__(256, 2) k_metric_tau(const MetricDesc* __restrict__ tab,
                                                       const __grid_constant__ MetricDesc one, int op,
                                                       double* __restrict__ part) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double red[8];
    const MetricDesc& d = tab ? tab[blockIdx.y] : one;
    const int L = d.L, Nt = d.Nt, Hx = d.Hx, cols = L * Hx, nt = (cols + kMW - 1) / kMW;
    if ((int)blockIdx.x >= 3 * nt) return;
    const int a = blockIdx.x / nt, j0 = (blockIdx.x - a * nt) * kMW, live = min(kMW, cols - j0);
    double2* tile = reinterpret_cast<double2*>(smem);
    double2* tw = tile + Nt * kMW;
    double2* spec = d.spec + (int64_t)a * Nt * cols + j0;
    for (int i = threadIdx.x; i < Nt; i += blockDim.x) tw[i] = __ldg(d.twt + i);
    for (int e = threadIdx.x; e < Nt * kMW; e += blockDim.x) {
        const int t = e / kMW, l = e % kMW;
        tile[e] = l < live ? spec[(int64_t)t * cols + l] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    const Lines ln{1, 0, kMW, FastDiv{0x80000001u, 3}, 1, 2};
    dft_forward(tile, ln, d.t1, d.t2, kMW, tw);
    // this thread's column is the same in every round: blockDim is a multiple of kMW
    const int l = threadIdx.x % kMW, j = j0 + min(l, live - 1);
    const int py = fdiv(j, d.dHx), kx = j - py * Hx;
    const int my = dft_freq(py, d.x1, d.x2), mym = my ? L - my : 0, kxm = kx ? L - kx : 0;
    const bool mirrored = kx != 0 && kx != L / 2;   // -k lies outside the half spectrum
    const int64_t LL = (int64_t)L * L, base = a * Nt * LL;
    const double *sp = d.sig + base + my * L + kx, *sm = d.sig + base + mym * L + kxm;
    double acc = 0.0;
    for (int e = threadIdx.x; e < Nt * kMW; e += blockDim.x) {
        if (l >= live) break;
        const int n = dft_freq(e / kMW, d.t1, d.t2), nm = n ? Nt - n : 0;
        const double2 v = tile[e];
        if (op == HMC_METRIC_ACCUM) {
            const double q = (v.x * v.x + v.y * v.y) * d.scale;
            d.out[base + n * LL + my * L + kx] += q;
            if (mirrored) d.out[base + nm * LL + mym * L + kxm] += q;
            continue;
        }
        const double s0 = __ldg(sp + n * LL), s1 = __ldg(sm + nm * LL);
        double w;
        if (op == HMC_METRIC_VELOCITY || op == HMC_METRIC_KINETIC) w = s0 + s1;
        else if (op == HMC_METRIC_MOMENTUM) {
            w = 1.0 / sqrt(s0);
            w += s1 == s0 ? w : 1.0 / sqrt(s1);
        } else {
            w = 1.0 / s0;
            w += s1 == s0 ? w : 1.0 / s1;
        }
        if (op == HMC_METRIC_KINETIC || op == HMC_METRIC_MNORM) {
            const double q = w * (v.x * v.x + v.y * v.y);
            acc += mirrored ? q : 0.5 * q;
        } else {
            tile[e] = make_double2(w * v.y, w * v.x);   // re and im exchanged: inverse steps follow
        }
    }
    if (op == HMC_METRIC_ACCUM) return;
    if (op == HMC_METRIC_KINETIC || op == HMC_METRIC_MNORM) {
        acc = block_sum(acc * d.scale, red);
        if (threadIdx.x == 0) part[blockIdx.x] = acc;
        return;
    }
    __syncthreads();
    dft_inverse(tile, ln, d.t1, d.t2, kMW, tw);
    for (int e = threadIdx.x; e < Nt * kMW; e += blockDim.x)
        if (l < live) spec[(int64_t)(e / kMW) * cols + l] = swapc(tile[e]);
}

// The planes back: out = scale * (real field), or out += eps * that.
__global__ void __launch_bounds__(256, 2) k_metric_inv(const MetricDesc* __restrict__ tab,
                                                       const __grid_constant__ MetricDesc one, double eps) {
    extern __shared__ __align__(16) unsigned char smem[];
    const MetricDesc& d = tab ? tab[blockIdx.y] : one;
    const int L = d.L, Hx = d.Hx, RA = L | 1, RB = Hx | 1;
    if ((int)blockIdx.x >= 3 * d.Nt) return;
    const PlaneTiles p = plane_tiles(d, smem);
    const double2* in = d.spec + (int64_t)blockIdx.x * L * Hx;
    for (int e = threadIdx.x; e < L * Hx; e += blockDim.x) {
        const int y = fdiv(e, d.dHx), k = e - y * Hx;
        p.half[y * RB + k] = swapc(in[e]);
    }
    __syncthreads();
    dft_inverse(p.half, Lines{1, 0, Hx, d.dHx, 1, 2}, d.x1, d.x2, RB, p.tw);
    // rows u and v as the line u + i v from their half spectra (and the conjugates at -k), re and im exchanged
    for (int e = threadIdx.x; e < (L / 2) * Hx; e += blockDim.x) {
        const int j = fdiv(e, d.dHx), k = e - j * Hx;
        const double2 u = swapc(p.half[2 * j * RB + k]), v = swapc(p.half[(2 * j + 1) * RB + k]);
        double2* row = p.rows + j * RA;
        if (k == 0 || k == L / 2) {
            row[p.pos[k]] = make_double2(v.x, u.x);   // real columns
        } else {
            row[p.pos[k]] = make_double2(u.y + v.x, u.x - v.y);
            row[p.pos[L - k]] = make_double2(v.x - u.y, u.x + v.y);
        }
    }
    __syncthreads();
    dft_inverse(p.rows, Lines{1, 0, L / 2, d.dHalf, RA, 2 * RA}, d.x1, d.x2, 1, p.tw);
    double* out = d.out + (int64_t)blockIdx.x * L * L;
    const double s = eps == 0.0 ? d.scale : eps * d.scale;
    for (int e = threadIdx.x; e < (L / 2) * L; e += blockDim.x) {
        const int j = fdiv(e, d.dL), x = e - j * L;
        const double2 z = p.rows[j * RA + x];
        double *o0 = out + 2 * j * L + x, *o1 = o0 + L;
        if (eps == 0.0) {
            *o0 = s * z.y;
            *o1 = s * z.x;
        } else {
            *o0 = fma(s, z.y, *o0);
            *o1 = fma(s, z.x, *o1);
        }
    }
}

// ---- host --------------------------------------------------------------------------------------------
static bool make_desc(hmc_ctx* ctx, const Lat& lat, MetricDesc* d) {
    const FftPlan *px = get_plan(ctx, lat.L), *pt = get_plan(ctx, lat.Nt);
    if (lat.L < 4 || !px || !pt || !dft_split(lat.L, &d->x1, &d->x2) || !dft_split(lat.Nt, &d->t1, &d->t2)) return false;
    if (plane_smem(lat.L) > kMSmem) return false;
    d->L = lat.L;
    d->Nt = lat.Nt;
    d->Hx = lat.L / 2 + 1;
    d->dL = fast_div(lat.L);
    d->dHalf = fast_div(lat.L / 2);
    d->dHx = fast_div(d->Hx);
    d->twx = px->tw64;
    d->twt = pt->tw64;
    return true;
}

static int metric_launch(hmc_ctx* ctx, const MetricDesc* tab, const MetricDesc& one, int nchains, int maxL, int maxNt,
                         int op, double eps, double* scalar_dev) {
    static PerDevice attr;
    uint64_t bit;
    if (attr.pending(&bit)) {
        HMC_CUDA(ctx, cudaFuncSetAttribute(k_metric_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMSmem));
        HMC_CUDA(ctx, cudaFuncSetAttribute(k_metric_tau, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMSmem));
        HMC_CUDA(ctx, cudaFuncSetAttribute(k_metric_inv, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMSmem));
        attr.mark(bit);
    }
    // threads by the lines of a step: a warp of the FP64 pipe costs the same however few of its lanes work
    const int thr = maxL >= 32 ? 256 : maxL >= 16 ? 128 : 64, tthr = maxNt >= 40 ? 256 : 128;
    const size_t psm = plane_smem(maxL), tsm = (size_t)(maxNt * kMW + maxNt) * sizeof(double2);
    const dim3 planes(3 * maxNt, nchains), tiles(3 * ((maxL * (maxL / 2 + 1) + kMW - 1) / kMW), nchains);
    const bool sum = op == HMC_METRIC_KINETIC || op == HMC_METRIC_MNORM;
    if (sum && (int64_t)tiles.x > ctx->part_cap) return fail(ctx, HMC_ERR_ARG, "metric: reduction buffer too small");
    k_metric_fwd<<<planes, thr, psm, ctx->stream>>>(tab, one);
    HMC_LAUNCH(ctx, "k_metric_fwd");
    k_metric_tau<<<tiles, tthr, tsm, ctx->stream>>>(tab, one, op, ctx->d_part);
    HMC_LAUNCH(ctx, "k_metric_tau");
    if (sum) return reduce_rows(ctx, ctx->d_part, 1, (int)tiles.x, scalar_dev);
    if (op == HMC_METRIC_ACCUM) return HMC_OK;
    k_metric_inv<<<planes, thr, psm, ctx->stream>>>(tab, one, eps);
    HMC_LAUNCH(ctx, "k_metric_inv");
    return HMC_OK;
}

// The forward transforms come out unnormalised and doubled, the weights as the sum over k and -k.
static double op_scale(int op, double V) { return (op == HMC_METRIC_KINETIC ? 0.5 : 1.0) / (4.0 * V); }

int metric_real(hmc_ctx* ctx, const Lat& lat, int op, const double* sig, const double* in, double* out, double eps,
                double* scalar_dev, bool* done) {
    MetricDesc d{};
    *done = make_desc(ctx, lat, &d);
    if (!*done) return HMC_OK;
    d.in = in;
    d.sig = sig;
    d.out = out;
    d.spec = ctx->d_fft;
    d.scale = op_scale(op, (double)lat.V);
    return metric_launch(ctx, nullptr, d, 1, lat.L, lat.Nt, op, eps, scalar_dev);
}

// ---- all chains of a batch ----------------------------------------------------------------------------
int metric_batch_alloc(hmc_ctx* ctx) {
    HMC_CUDA(ctx, cudaMalloc(&ctx->batch.metric, ctx->chains.size() * sizeof(MetricDesc)));
    return HMC_OK;
}

int metric_batch_begin(hmc_ctx* ctx, const double* const* sig, double* const* phi) {
    BatchWork& w = ctx->batch;
    const int nc = (int)ctx->chains.size();
    w.hmetric.resize(nc * sizeof(MetricDesc));
    MetricDesc* t = reinterpret_cast<MetricDesc*>(w.hmetric.data());
    w.metric_ok = true;
    w.maxL = w.maxNt = 0;
    for (int c = 0; c < nc; ++c) {
        const Lat& lat = ctx->chains[c].lat;
        MetricDesc d{};
        if (!make_desc(ctx, lat, &d)) {
            w.metric_ok = false;
            return HMC_OK;
        }
        d.in = ctx->d_pi + 3 * ctx->batch_off[c];
        d.sig = sig[c];
        d.out = phi[c];
        // the spectra (at most 3 V complex) in the FP64 residual's workspace (4 V and more), which the batched
        // solve does not use
        d.spec = ctx->d_r64 + 3 * ctx->batch_off[c];
        d.scale = op_scale(HMC_METRIC_VELOCITY, (double)lat.V);
        t[c] = d;
        w.maxL = std::max(w.maxL, lat.L);
        w.maxNt = std::max(w.maxNt, lat.Nt);
    }
    HMC_CUDA(ctx, cudaMemcpyAsync(w.metric, t, nc * sizeof(MetricDesc), cudaMemcpyHostToDevice, ctx->stream));
    return HMC_OK;
}

int metric_batch_drift(hmc_ctx* ctx, double eps) {
    const BatchWork& w = ctx->batch;
    return metric_launch(ctx, reinterpret_cast<const MetricDesc*>(w.metric), MetricDesc{}, (int)ctx->chains.size(), w.maxL,
                         w.maxNt, HMC_METRIC_VELOCITY, eps, nullptr);
}

}  // namespace hmc
