// Fourier-diagonal metric operations of Section "Online metric estimation" on real fields, in three
// launches: the half spectrum of every (component, time slice) plane (x, then y), the tau transform with the
// spectral weight and its inverse, and the planes back (y, then x) with the output update; five with x and y in
// launches of their own on large lattices.
//
// What bounds it is GB300's FP64 pipe (two lanes a clock per SM), so the transforms are of real data: two
// rows of a plane share one complex x transform, and y and tau run on the L / 2 + 1 columns that determine
// the spectrum, half the operations of complex transforms; packing, weights and the leapfrog update ride
// along. Integer and shared-memory work hides behind the pipe, so lengths are run-time values. At
// 80 x 80 x 160 the drift takes 0.48 ms against 1.16 with complex transforms in nine launches; its operations
// alone take 0.33 ms of the pipe, its bytes 0.01 ms. On small lattices the launches count, three against nine.
//
// Against extended precision the velocity is off by 3.8e-16 of its norm at 40 x 40 x 80 and 1.9e-16 at 4 x 4 x 8; by
// 3.2e-16 and 2.5e-16 with complex transforms, whose dropped imaginary part takes half of their rounding along.
//
// The weight of a wave vector k is the mean of sigma-hat's at k and -k (its own where sigma-hat is even, as
// an estimate from real fields is): the real part that a complex transform keeps.
#include <algorithm>
#include <cmath>

#include "dft_smem.cuh"
#include "internal.h"

namespace hmc {

constexpr int kMW = 40;               // most lines of a tile
constexpr size_t kMSmem = 216 * 1024;

// One chain's transform: geometry, splits L = x1 x2 and Nt = t1 t2, twiddles, fields and spectrum
// [component][slice][position along y][kx].
struct MetricDesc {
    int L, Nt, Hx;
    int x1, x2, t1, t2;
    FastDiv dL, dHalf, dHx;
    int W;          // columns of a tau tile
    FastDiv dW;
    const double2 *twx, *twt;
    const double *in, *sig;
    double* out;
    double2* spec;
    double scale;
};

// entries of the fields and of the spectrum by address, for the index checks of the bounds build
__device__ __forceinline__ double ld_field(const MetricDesc& d, const double* base, const double* p) {
    return __ldg(in_range(p, base, (int64_t)3 * d.Nt * d.L * d.L, kBndMetric));
}
__device__ __forceinline__ double& out_at(const MetricDesc& d, double* p) {
    return *in_range(p, d.out, (int64_t)3 * d.Nt * d.L * d.L, kBndMetric);
}
__device__ __forceinline__ double2& spec_at(const MetricDesc& d, double2* p) {
    return *in_range(p, d.spec, (int64_t)3 * d.Nt * d.L * d.Hx, kBndMetric);
}

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
        tile_at(p.rows, j * RA + x) = make_double2(ld_field(d, d.in, in + 2 * j * L + x), ld_field(d, d.in, in + (2 * j + 1) * L + x));
    }
    __syncthreads();
    dft_forward(p.rows, Lines{1, 0, L / 2, d.dHalf, RA, 2 * RA}, d.x1, d.x2, 1, p.tw);
    // twice each row's half spectrum: Z(k) + conj Z(-k) and (Z(k) - conj Z(-k)) / i
    for (int e = threadIdx.x; e < (L / 2) * Hx; e += blockDim.x) {
        const int j = fdiv(e, d.dHx), k = e - j * Hx;
        const double2 z = tile_at(p.rows, j * RA + p.pos[k]), w = tile_at(p.rows, j * RA + p.pos[k ? L - k : 0]);
        tile_at(p.half, 2 * j * RB + k) = make_double2(z.x + w.x, z.y - w.y);
        tile_at(p.half, (2 * j + 1) * RB + k) = make_double2(z.y + w.y, w.x - z.x);
    }
    __syncthreads();
    dft_forward(p.half, Lines{1, 0, Hx, d.dHx, 1, 2}, d.x1, d.x2, RB, p.tw);
    double2* out = d.spec + (int64_t)blockIdx.x * L * Hx;
    for (int e = threadIdx.x; e < L * Hx; e += blockDim.x) {
        const int y = fdiv(e, d.dHx), k = e - y * Hx;
        spec_at(d, out + e) = tile_at(p.half, y * RB + k);
    }
}

// The tau transform of W columns of one component, the weights of `op`, and (momentum, velocity) the
// inverse, in place on the spectrum. Sums: part[blockIdx.x]; ACCUM: out += |F in|^2 at k and -k.
__global__ void __launch_bounds__(256, 2) k_metric_tau(const MetricDesc* __restrict__ tab,
                                                       const __grid_constant__ MetricDesc one, int op,
                                                       double* __restrict__ part) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double red[8];
    const MetricDesc& d = tab ? tab[blockIdx.y] : one;
    const int L = d.L, Nt = d.Nt, Hx = d.Hx, W = d.W, cols = L * Hx, nt = (cols + W - 1) / W;
    if ((int)blockIdx.x >= 3 * nt) return;
    const int a = blockIdx.x / nt, j0 = (blockIdx.x - a * nt) * W, live = min(W, cols - j0);
    double2* tile = reinterpret_cast<double2*>(smem);
    double2* tw = tile + Nt * W;
    double2* spec = d.spec + (int64_t)a * Nt * cols + j0;
    for (int i = threadIdx.x; i < Nt; i += blockDim.x) tw[i] = __ldg(d.twt + i);
    for (int e = threadIdx.x; e < Nt * W; e += blockDim.x) {
        const int t = fdiv(e, d.dW), l = e - t * W;
        tile_at(tile, e) = l < live ? spec_at(d, spec + (int64_t)t * cols + l) : make_double2(0.0, 0.0);
    }
    __syncthreads();
    const Lines ln{1, 0, W, d.dW, 1, 2};
    dft_forward(tile, ln, d.t1, d.t2, W, tw);
    const int64_t LL = (int64_t)L * L, base = a * Nt * LL;
    double acc = 0.0;
    for (int e = threadIdx.x; e < Nt * W; e += blockDim.x) {
        const int p = fdiv(e, d.dW), l = e - p * W;
        if (l >= live) continue;
        const int j = j0 + l, py = fdiv(j, d.dHx), kx = j - py * Hx;
        const int n = dft_freq(p, d.t1, d.t2), nm = n ? Nt - n : 0;
        const int my = dft_freq(py, d.x1, d.x2), mym = my ? L - my : 0, kxm = kx ? L - kx : 0;
        const bool mirrored = kx != 0 && kx != L / 2;   // -k lies outside the half spectrum
        const int64_t at = base + n * LL + my * L + kx, atm = base + nm * LL + mym * L + kxm;
        const double2 v = tile_at(tile, e);
        if (op == HMC_METRIC_ACCUM) {
            const double q = (v.x * v.x + v.y * v.y) * d.scale;
            out_at(d, d.out + at) += q;
            if (mirrored) out_at(d, d.out + atm) += q;
            continue;
        }
        const double s0 = ld_field(d, d.sig, d.sig + at), s1 = ld_field(d, d.sig, d.sig + atm);
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
            tile_at(tile, e) = make_double2(w * v.y, w * v.x);   // re and im exchanged: inverse steps follow
        }
    }
    if (op == HMC_METRIC_ACCUM) return;
    if (op == HMC_METRIC_KINETIC || op == HMC_METRIC_MNORM) {
        acc = block_sum(acc * d.scale, red);
        if (threadIdx.x == 0) part[blockIdx.x] = acc;
        return;
    }
    __syncthreads();
    dft_inverse(tile, ln, d.t1, d.t2, W, tw);
    for (int e = threadIdx.x; e < Nt * W; e += blockDim.x) {
        const int t = fdiv(e, d.dW), l = e - t * W;
        if (l < live) spec_at(d, spec + (int64_t)t * cols + l) = swapc(tile_at(tile, e));
    }
}

// The x and y transforms by tiles of lines, for fields whose planes would leave SMs idle in the last of few
// waves (480 planes of 80 x 80 x 160 on 304 resident blocks: 1.58 waves): W row pairs, or W columns of the
// half spectrum, of all planes together.
__device__ __forceinline__ void x_tables(const MetricDesc& d, double2* tw, int* pos) {
    for (int i = threadIdx.x; i < d.L; i += blockDim.x) {
        tw[i] = __ldg(d.twx + i);
        pos[i] = dft_pos(i, d.x1, d.x2);
    }
}
__global__ void __launch_bounds__(256, 2) k_metric_x_fwd(const __grid_constant__ MetricDesc d, int W, FastDiv dW) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int L = d.L, Hx = d.Hx, RA = L | 1, total = 3 * d.Nt * (L / 2), c0 = blockIdx.x * W, live = min(W, total - c0);
    double2 *rows = reinterpret_cast<double2*>(smem), *tw = rows + W * RA;
    int* pos = reinterpret_cast<int*>(tw + L);
    x_tables(d, tw, pos);
    const double* in = d.in + (int64_t)c0 * 2 * L;
    for (int e = threadIdx.x; e < W * L; e += blockDim.x) {
        const int j = fdiv(e, d.dL), x = e - j * L;
        tile_at(rows, j * RA + x) =
            j < live ? make_double2(ld_field(d, d.in, in + 2 * j * L + x), ld_field(d, d.in, in + (2 * j + 1) * L + x))
                     : make_double2(0.0, 0.0);
    }
    __syncthreads();
    dft_forward(rows, Lines{1, 0, W, dW, RA, 2 * RA}, d.x1, d.x2, 1, tw);
    double2* out = d.spec + (int64_t)c0 * 2 * Hx;
    for (int e = threadIdx.x; e < live * Hx; e += blockDim.x) {
        const int j = fdiv(e, d.dHx), k = e - j * Hx;
        const double2 z = tile_at(rows, j * RA + pos[k]), w = tile_at(rows, j * RA + pos[k ? L - k : 0]);
        spec_at(d, out + 2 * j * Hx + k) = make_double2(z.x + w.x, z.y - w.y);
        spec_at(d, out + (2 * j + 1) * Hx + k) = make_double2(z.y + w.y, w.x - z.x);
    }
}
template <bool INV>
__global__ void __launch_bounds__(256, 2) k_metric_y(const __grid_constant__ MetricDesc d, int W, FastDiv dW) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int L = d.L, Hx = d.Hx, total = 3 * d.Nt * Hx, c0 = blockIdx.x * W;
    double2 *tile = reinterpret_cast<double2*>(smem), *tw = tile + L * W;
    for (int i = threadIdx.x; i < L; i += blockDim.x) tw[i] = __ldg(d.twx + i);
    auto at = [&](int e, int* y) -> double2* {   // spectrum entry of tile entry e, null past the last column
        *y = fdiv(e, dW);
        const int c = c0 + e - *y * W, plane = fdiv(c, d.dHx);
        return c < total ? &spec_at(d, d.spec + ((int64_t)plane * L + *y) * Hx + (c - plane * Hx)) : nullptr;
    };
    int y;
    for (int e = threadIdx.x; e < L * W; e += blockDim.x) {
        const double2* q = at(e, &y);
        const double2 v = q ? *q : make_double2(0.0, 0.0);
        tile_at(tile, e) = INV ? swapc(v) : v;
    }
    __syncthreads();
    const Lines ln{1, 0, W, dW, 1, 2};
    if (INV) dft_inverse(tile, ln, d.x1, d.x2, W, tw);
    else dft_forward(tile, ln, d.x1, d.x2, W, tw);
    for (int e = threadIdx.x; e < L * W; e += blockDim.x)
        if (double2* q = at(e, &y)) *q = INV ? swapc(tile_at(tile, e)) : tile_at(tile, e);
}
// rows u and v as the line u + i v from their half spectra (and the conjugates at -k), re and im exchanged
__device__ __forceinline__ void pack_pair(double2* row, const int* pos, int L, int k, double2 u, double2 v) {
    if (k == 0 || k == L / 2) {
        tile_at(row, pos[k]) = make_double2(v.x, u.x);   // real columns
    } else {
        tile_at(row, pos[k]) = make_double2(u.y + v.x, u.x - v.y);
        tile_at(row, pos[L - k]) = make_double2(v.x - u.y, u.x + v.y);
    }
}
__device__ __forceinline__ void put_rows(const MetricDesc& d, const double2* rows, int pairs, int64_t first, double eps, bool add) {
    const int L = d.L, RA = L | 1;
    double* out = d.out + first * 2 * L;
    const double s = add ? eps * d.scale : d.scale;
    for (int e = threadIdx.x; e < pairs * L; e += blockDim.x) {
        const int j = fdiv(e, d.dL), x = e - j * L;
        const double2 z = tile_at(rows, j * RA + x);
        double *o0 = &out_at(d, out + 2 * j * L + x), *o1 = &out_at(d, out + (2 * j + 1) * L + x);
        if (add) {
            *o0 = fma(s, z.y, *o0);
            *o1 = fma(s, z.x, *o1);
        } else {
            *o0 = s * z.y;
            *o1 = s * z.x;
        }
    }
}
__global__ void __launch_bounds__(256, 2) k_metric_x_inv(const __grid_constant__ MetricDesc d, int W, FastDiv dW, double eps,
                                                          bool add) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int L = d.L, Hx = d.Hx, RA = L | 1, total = 3 * d.Nt * (L / 2), c0 = blockIdx.x * W, live = min(W, total - c0);
    double2 *rows = reinterpret_cast<double2*>(smem), *tw = rows + W * RA;
    int* pos = reinterpret_cast<int*>(tw + L);
    x_tables(d, tw, pos);
    for (int e = live * RA + threadIdx.x; e < W * RA; e += blockDim.x) tile_at(rows, e) = make_double2(0.0, 0.0);
    __syncthreads();
    double2* in = d.spec + (int64_t)c0 * 2 * Hx;
    for (int e = threadIdx.x; e < live * Hx; e += blockDim.x) {
        const int j = fdiv(e, d.dHx), k = e - j * Hx;
        pack_pair(rows + j * RA, pos, L, k, spec_at(d, in + 2 * j * Hx + k), spec_at(d, in + (2 * j + 1) * Hx + k));
    }
    __syncthreads();
    dft_inverse(rows, Lines{1, 0, W, dW, RA, 2 * RA}, d.x1, d.x2, 1, tw);
    put_rows(d, rows, live, c0, eps, add);
}

// The planes back: out = scale * (real field), or (add) out += eps * that.
__global__ void __launch_bounds__(256, 2) k_metric_inv(const MetricDesc* __restrict__ tab,
                                                       const __grid_constant__ MetricDesc one, double eps, bool add) {
    extern __shared__ __align__(16) unsigned char smem[];
    const MetricDesc& d = tab ? tab[blockIdx.y] : one;
    const int L = d.L, Hx = d.Hx, RA = L | 1, RB = Hx | 1;
    if ((int)blockIdx.x >= 3 * d.Nt) return;
    const PlaneTiles p = plane_tiles(d, smem);
    double2* in = d.spec + (int64_t)blockIdx.x * L * Hx;
    for (int e = threadIdx.x; e < L * Hx; e += blockDim.x) {
        const int y = fdiv(e, d.dHx), k = e - y * Hx;
        tile_at(p.half, y * RB + k) = swapc(spec_at(d, in + e));
    }
    __syncthreads();
    dft_inverse(p.half, Lines{1, 0, Hx, d.dHx, 1, 2}, d.x1, d.x2, RB, p.tw);
    for (int e = threadIdx.x; e < (L / 2) * Hx; e += blockDim.x) {
        const int j = fdiv(e, d.dHx), k = e - j * Hx;
        pack_pair(p.rows + j * RA, p.pos, L, k, swapc(tile_at(p.half, 2 * j * RB + k)), swapc(tile_at(p.half, (2 * j + 1) * RB + k)));
    }
    __syncthreads();
    dft_inverse(p.rows, Lines{1, 0, L / 2, d.dHalf, RA, 2 * RA}, d.x1, d.x2, 1, p.tw);
    put_rows(d, p.rows, L / 2, (int64_t)blockIdx.x * (L / 2), eps, add);
}

unsigned int bounds_take_metric() { return bounds_take_tu(); }

// ---- host --------------------------------------------------------------------------------------------
// Lines of a tile, of `total` lines of n1 n2 points: the width whose waves of two blocks an SM cost the FP64 pipe
// least, a step's tasks counted in whole warps
static int tile_width(const hmc_ctx* ctx, int total, int n1, int n2, size_t line_bytes) {
    const int slots = 2 * ctx->num_sms;
    int best = 2;
    double least = 1e300;
    const double w1 = n1 * (1 + std::log2((double)n1)), w2 = n2 * (1 + std::log2((double)n2));   // of one DFT
    for (int W = 2; W <= kMW && W * line_bytes <= kMSmem / 2 - 4096; ++W) {
        const int waves = ((total + W - 1) / W + slots - 1) / slots;
        const double step = (W * n1 + 31) / 32 * w2 + (W * n2 + 31) / 32 * w1;
        const double cost = waves * (step + 30);
        if (cost < least) {
            least = cost;
            best = W;
        }
    }
    return best;
}

static bool make_desc(hmc_ctx* ctx, const Lat& lat, MetricDesc* d) {
    const FftPlan *px = get_plan(ctx, lat.L), *pt = get_plan(ctx, lat.Nt);
    if (lat.L < 4 || !px || !pt || !dft_split(lat.L, &d->x1, &d->x2, true) || !dft_split(lat.Nt, &d->t1, &d->t2, true)) return false;
    if (plane_smem(lat.L) > kMSmem) return false;
    d->L = lat.L;
    d->Nt = lat.Nt;
    d->Hx = lat.L / 2 + 1;
    d->dL = fast_div(lat.L);
    d->dHalf = fast_div(lat.L / 2);
    d->dHx = fast_div(d->Hx);
    d->twx = px->tw64;
    d->twt = pt->tw64;
    // (a component has its own tiles)
    d->W = tile_width(ctx, 3 * lat.L * d->Hx, d->t1, d->t2, (size_t)lat.Nt * sizeof(double2));
    d->W = std::min(d->W, lat.L * d->Hx);
    d->dW = fast_div(d->W);
    return true;
}

static int set_smem(hmc_ctx* ctx) {
    static PerDevice attr;
    uint64_t bit;
    if (!attr.pending(&bit)) return HMC_OK;
    for (const void* f : {(const void*)k_metric_fwd, (const void*)k_metric_tau, (const void*)k_metric_inv,
                          (const void*)k_metric_x_fwd, (const void*)k_metric_y<false>, (const void*)k_metric_y<true>,
                          (const void*)k_metric_x_inv})
        HMC_CUDA(ctx, cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMSmem));
    attr.mark(bit);
    return HMC_OK;
}

static int launch_tau(hmc_ctx* ctx, const MetricDesc* tab, const MetricDesc& one, int nchains, int tiles, int maxNt,
                      size_t smem, int op) {
    k_metric_tau<<<dim3(tiles, nchains), maxNt >= 40 ? 256 : 128, smem, ctx->stream>>>(tab, one, op, ctx->d_part);
    HMC_LAUNCH(ctx, "k_metric_tau");
    return HMC_OK;
}

static int tau_tiles(const MetricDesc& d) { return 3 * ((d.L * d.Hx + d.W - 1) / d.W); }
static size_t tau_smem(const MetricDesc& d) { return (size_t)d.Nt * (d.W + 1) * sizeof(double2); }

// Threads by the lines of a step: a warp costs the FP64 pipe the same however few of its lanes work.
static int plane_threads(int L) { return L >= 32 ? 256 : L >= 16 ? 128 : 64; }

// The forward transforms come out unnormalised and doubled, the weights as the sum over k and -k.
static double op_scale(int op, double V) { return (op == HMC_METRIC_KINETIC ? 0.5 : 1.0) / (4.0 * V); }

int metric_real(hmc_ctx* ctx, const Lat& lat, int op, const double* sig, const double* in, double* out, double eps,
                bool add, double* scalar_dev, bool* done) {
    MetricDesc d{};
    *done = make_desc(ctx, lat, &d);
    if (!*done) return HMC_OK;
    d.in = in;
    d.sig = sig;
    d.out = out;
    d.spec = ctx->d_fft;
    d.scale = op_scale(op, (double)lat.V);
    int rc;
    if ((rc = set_smem(ctx))) return rc;
    const bool sum = op == HMC_METRIC_KINETIC || op == HMC_METRIC_MNORM, back = op == HMC_METRIC_VELOCITY || op == HMC_METRIC_MOMENTUM;
    const int tiles = tau_tiles(d);
    if (sum && (int64_t)tiles > ctx->part_cap) return fail(ctx, HMC_ERR_ARG, "metric: reduction buffer too small");
    // lines where the planes fill their waves badly and the transforms, not the launches, take the time
    // (80 x 80 x 160: 0.56 ms by planes)
    const int64_t slots = 2 * ctx->num_sms, planes = 3 * (int64_t)lat.Nt, waves = (planes + slots - 1) / slots;
    const bool lines = lat.V >= 400000 && 10 * planes < 9 * waves * slots;
    const int pairs = 3 * lat.Nt * (lat.L / 2), cols = 3 * lat.Nt * d.Hx;
    const size_t xline = (size_t)(lat.L | 1) * sizeof(double2), yline = (size_t)lat.L * sizeof(double2);
    const size_t xtab = lat.L * (sizeof(double2) + sizeof(int));
    const int Wx = lines ? tile_width(ctx, pairs, d.x1, d.x2, xline) : 2, Wy = lines ? tile_width(ctx, cols, d.x1, d.x2, yline) : 2;
    const int gx = (pairs + Wx - 1) / Wx, gy = (cols + Wy - 1) / Wy;
    if (lines) {
        k_metric_x_fwd<<<gx, 256, Wx * xline + xtab, ctx->stream>>>(d, Wx, fast_div(Wx));
        HMC_LAUNCH(ctx, "k_metric_x_fwd");
        k_metric_y<false><<<gy, 256, Wy * yline + xtab, ctx->stream>>>(d, Wy, fast_div(Wy));
    } else {
        k_metric_fwd<<<(unsigned)planes, plane_threads(lat.L), plane_smem(lat.L), ctx->stream>>>(nullptr, d);
    }
    HMC_LAUNCH(ctx, "k_metric_fwd");
    if ((rc = launch_tau(ctx, nullptr, d, 1, tiles, lat.Nt, tau_smem(d), op))) return rc;
    if (sum) return reduce_rows(ctx, ctx->d_part, 1, tiles, scalar_dev);
    if (!back) return HMC_OK;
    if (lines) {
        k_metric_y<true><<<gy, 256, Wy * yline + xtab, ctx->stream>>>(d, Wy, fast_div(Wy));
        HMC_LAUNCH(ctx, "k_metric_y");
        k_metric_x_inv<<<gx, 256, Wx * xline + xtab, ctx->stream>>>(d, Wx, fast_div(Wx), eps, add);
    } else {
        k_metric_inv<<<(unsigned)planes, plane_threads(lat.L), plane_smem(lat.L), ctx->stream>>>(nullptr, d, eps, add);
    }
    HMC_LAUNCH(ctx, "k_metric_inv");
    return HMC_OK;
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
    w.maxL = w.maxNt = w.tau_tiles = 0;
    w.tau_smem = 0;
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
        w.tau_tiles = std::max(w.tau_tiles, tau_tiles(d));
        w.tau_smem = std::max(w.tau_smem, tau_smem(d));
    }
    HMC_CUDA(ctx, cudaMemcpyAsync(w.metric, t, nc * sizeof(MetricDesc), cudaMemcpyHostToDevice, ctx->stream));
    return HMC_OK;
}

int metric_batch_drift(hmc_ctx* ctx, double eps) {
    const BatchWork& w = ctx->batch;
    const MetricDesc* tab = reinterpret_cast<const MetricDesc*>(w.metric);
    const int nc = (int)ctx->chains.size(), thr = plane_threads(w.maxL);
    const dim3 planes(3 * w.maxNt, nc);
    int rc;
    if ((rc = set_smem(ctx))) return rc;
    k_metric_fwd<<<planes, thr, plane_smem(w.maxL), ctx->stream>>>(tab, MetricDesc{});
    HMC_LAUNCH(ctx, "k_metric_fwd");
    if ((rc = launch_tau(ctx, tab, MetricDesc{}, nc, w.tau_tiles, w.maxNt, w.tau_smem, HMC_METRIC_VELOCITY))) return rc;
    k_metric_inv<<<planes, thr, plane_smem(w.maxL), ctx->stream>>>(tab, MetricDesc{}, eps, true);
    HMC_LAUNCH(ctx, "k_metric_inv");
    return HMC_OK;
}

}  // namespace hmc
