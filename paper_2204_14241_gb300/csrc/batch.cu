// Batched solves of many uneven lattices in one persistent launch: every (chain, right-hand side) pair
// of a context is a team of the solver in team.cu (mixed precision, plain CG). The vectors of all pairs
// are concatenated, chain c's K right-hand sides at item offset off_c ([c][k][site], 4 complex per item).
//
// The pairs in flight keep their vectors in L2 (x, r, two directions, t_ and phi: 172 bytes a site) where all of
// them fit: a team each, with blocks by volume, so that all take about the same time per iteration. Past that,
// 128 pairs of the 64-chain batch (270 MB) streamed from memory in every iteration; there, teams of equal size take
// the pairs from a queue, largest first, as many teams as fit: a 64-chain trajectory 196 -> 154 ms. (With
// a set that fits the queue's last pairs leave teams idle: 24 chains, 101 MB, 53 ms in flight, 57 to 63 queued.) A
// pair's result does not depend on the team that takes it: queued teams have the same number of blocks and so
// the same order of sums.
#include <algorithm>
#include <cmath>
#include <numeric>

#include "internal.h"
#include "team.h"

namespace hmc {

constexpr int64_t kBatchAll = 112 << 20, kBatchQueued = 60 << 20;   // bytes in flight: all pairs at most; queued

// FP32 copies of every chain's phi: block column blockIdx.y is a chain
__global__ void k_phi_to32_b(const BChainDev* __restrict__ ch) {
    const BChainDev& c = ch[blockIdx.y];
    float* out = const_cast<float*>(c.phi32);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < 3 * c.V; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (float)c.phi64[i];
}

// ---- host ----------------------------------------------------------------------------------------
void batch_free(hmc_ctx* ctx) {
    BatchWork& w = ctx->batch;
    void* ps[] = {w.pairs, w.blk, w.team, w.next, w.part, w.bar, w.hist, w.fail, w.metric};
    for (void* p : ps)
        if (p) cudaFree(p);
    w.pairs = nullptr; w.blk = nullptr; w.team = nullptr; w.next = nullptr; w.part = nullptr; w.bar = nullptr; w.hist = nullptr; w.fail = nullptr; w.metric = nullptr;
    w.K = 0;
    w.kcap = 0;
}

int batch_alloc(hmc_ctx* ctx) {
    BatchWork& w = ctx->batch;
    const size_t np = ctx->chains.size() * (size_t)ctx->kmax;
    for (const ChainDesc& c : ctx->chains)
        if (c.lat.V >= (int64_t)1 << 30) return fail(ctx, HMC_ERR_ARG, "hmc_init: a batched chain is too large");
    int rc;
    if ((rc = team_batch_capacity(ctx, &w.cap))) return rc;
    if (w.cap < 1) return fail(ctx, HMC_ERR_CUDA, "batched solve: kernel does not fit on an SM");
    HMC_CUDA(ctx, cudaMalloc(&w.pairs, np * sizeof(TeamPair)));
    HMC_CUDA(ctx, cudaMalloc((void**)&w.blk, w.cap * sizeof(int)));
    HMC_CUDA(ctx, cudaMalloc((void**)&w.team, w.cap * sizeof(int2)));
    HMC_CUDA(ctx, cudaMalloc((void**)&w.next, w.cap * sizeof(int)));
    HMC_CUDA(ctx, cudaMalloc((void**)&w.part, 2 * (size_t)w.cap * sizeof(unsigned long long)));
    HMC_CUDA(ctx, cudaMalloc((void**)&w.bar, (w.cap + 1) * sizeof(unsigned)));
    HMC_CUDA(ctx, cudaMalloc((void**)&w.hist, HMC_MAX_SOLVES * np * sizeof(TeamStat)));
    HMC_CUDA(ctx, cudaMalloc((void**)&w.fail, sizeof(int)));
    if ((rc = metric_batch_alloc(ctx))) return rc;
    w.kcap = ctx->kmax;
    w.K = 0;
    w.hch.resize(ctx->chains.size());
    return HMC_OK;
}

// Teams for K right-hand sides (rebuilt only when K changes; synchronous copies into the buffers
// batch_alloc made).
static int batch_setup(hmc_ctx* ctx, int K) {
    BatchWork& w = ctx->batch;
    if (w.K == K) return HMC_OK;
    if (K < 1 || K > w.kcap) return fail(ctx, HMC_ERR_ARG, "batched solve: nrhs must be in [1, nrhs_max]");
    const int nc = (int)ctx->chains.size(), np = nc * K;
    std::vector<int> order(np);
    std::iota(order.begin(), order.end(), 0);
    auto vol = [&](int p) { return ctx->chains[p / K].lat.V; };
    const int64_t bytes = 172 * ctx->vtot / nc;   // of a pair, on average
    std::vector<int> T;
    w.queued = np > w.cap || np * bytes > kBatchAll;
    if (w.queued) std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return vol(a) > vol(b); });
    std::vector<TeamPair> pairs;
    for (int p : order) pairs.push_back(TeamPair{p / K, p % K});
    if (w.queued) {
        // no more blocks than leave a thread of the largest pair one item
        const int n = (int)std::max<int64_t>(1, std::min<int64_t>({(int64_t)np, (int64_t)w.cap, kBatchQueued / bytes}));
        T.assign(n, (int)std::max<int64_t>(1, std::min<int64_t>(w.cap / n, (2 * vol(order[0]) + 255) / 256)));
    } else {
        // one block each, then one more to the pair with the most items per block while a thread of it still
        // has more than one
        T.assign(np, 1);
        std::vector<std::pair<double, int>> heap;
        for (int e = 0; e < np; ++e) heap.push_back({2.0 * vol(order[e]), e});
        std::make_heap(heap.begin(), heap.end());
        for (int left = w.cap - np; left > 0 && heap.front().first > 256; --left) {
            std::pop_heap(heap.begin(), heap.end());
            const int e = heap.back().second;
            heap.back().first = 2.0 * vol(order[e]) / ++T[e];
            std::push_heap(heap.begin(), heap.end());
        }
    }
    std::vector<int> blk;
    std::vector<int2> team;
    for (int j = 0; j < (int)T.size(); ++j) {
        team.push_back(make_int2((int)blk.size(), T[j]));
        blk.insert(blk.end(), T[j], j);
    }
    w.teams = (int)team.size();
    w.grid = (int)blk.size();
    HMC_CUDA(ctx, cudaStreamSynchronize(ctx->stream));   // the tables may be in use by earlier work
    HMC_CUDA(ctx, cudaMemcpy(w.pairs, pairs.data(), pairs.size() * sizeof(TeamPair), cudaMemcpyHostToDevice));
    HMC_CUDA(ctx, cudaMemcpy(w.blk, blk.data(), blk.size() * sizeof(int), cudaMemcpyHostToDevice));
    HMC_CUDA(ctx, cudaMemcpy(w.team, team.data(), team.size() * sizeof(int2), cudaMemcpyHostToDevice));
    w.K = K;
    return HMC_OK;
}

int batched_begin(hmc_ctx* ctx, int K, const double* const* phi) {
    BatchWork& w = ctx->batch;
    int rc;
    if ((rc = batch_setup(ctx, K))) return rc;
    const int nc = (int)ctx->chains.size();
    for (int c = 0; c < nc; ++c) {
        BChainDev d{};
        team_geometry(&d, ctx->chains[c].lat);
        d.off = ctx->batch_off[c] * K;
        d.phi64 = phi[c];
        d.phi32 = ctx->batch_phi32 + 3 * ctx->batch_off[c];
        w.hch[c] = d;
    }
    HMC_CUDA(ctx, cudaMemcpyAsync(w.ch, w.hch.data(), nc * sizeof(BChainDev), cudaMemcpyHostToDevice, ctx->stream));
    HMC_CUDA(ctx, cudaMemsetAsync(w.fail, 0, sizeof(int), ctx->stream));
    return HMC_OK;
}

int batched_solve(hmc_ctx* ctx, int K, const double2* b, double2* x, bool use_x0, double tol, int maxit, int slot) {
    BatchWork& w = ctx->batch;
    if (w.K != K) return fail(ctx, HMC_ERR_STATE, "batched solve: batched_begin was not called for this nrhs");
    const int nc = (int)ctx->chains.size();
    const unsigned gx = (unsigned)std::min<int64_t>((3 * ctx->vmax + 255) / 256, std::max(1, 16 * ctx->num_sms / nc));
    k_phi_to32_b<<<dim3(gx, nc), 256, 0, ctx->stream>>>(w.ch);
    HMC_LAUNCH(ctx, "k_phi_to32_b");
    TeamArgs<float> a{};
    a.pairs = reinterpret_cast<const TeamPair*>(w.pairs);
    a.npairs = nc * K;
    a.next = w.next;
    a.nteams = w.teams;
    a.blk = w.blk;
    a.team = w.team;
    a.queue = w.queued ? reinterpret_cast<int*>(w.bar) + w.teams : nullptr;
    a.ch = w.ch;
    a.K = K;
    a.cf = make_coef<float>(ctx->p);
    a.cf64 = make_coef<double>(ctx->p);
    a.b = b;
    a.x64 = x;
    a.t64 = ctx->d_z64;
    a.x = ctx->d_x32;
    a.r = ctx->d_r32;
    a.pA = ctx->d_p32;
    a.pB = ctx->d_p32b;
    a.t = ctx->d_q32;
    a.part = w.part;
    a.bar = w.bar;
    a.flags = ctx->d_flags;
    a.fail = w.fail;
    a.stat = slot < HMC_MAX_SOLVES ? w.hist + (int64_t)slot * nc * K : nullptr;
    a.tol2 = tol * tol;
    a.delta2 = 1e-6;
    a.maxit = maxit;
    a.use_x0 = use_x0 ? 1 : 0;
    a.test_timeout = ctx->p.test_wait_timeout;
    a.timeout_ns = ctx->p.wait_spin_limit > 0 ? (long long)ctx->p.wait_spin_limit * 1000LL : 2000000000LL;
    return team_launch_batch(ctx, a, w.grid);
}

int batched_collect(hmc_ctx* ctx, int K, int nsolves, int* iterations, double* worst_resid, int* reliable_updates) {
    BatchWork& w = ctx->batch;
    const int nc = (int)ctx->chains.size(), np = nc * K;
    const int kept = std::min(nsolves, HMC_MAX_SOLVES);
    std::vector<TeamStat> hs((size_t)kept * np);
    int f = 0;
    if (kept > 0)
        HMC_CUDA(ctx, cudaMemcpyAsync(hs.data(), w.hist, hs.size() * sizeof(TeamStat), cudaMemcpyDeviceToHost, ctx->stream));
    HMC_CUDA(ctx, cudaMemcpyAsync(&f, w.fail, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    int rc;
    if ((rc = check_device_flags(ctx))) return rc;   // synchronises
    for (int j = 0; j < kept; ++j) {
        for (int c = 0; c < nc; ++c) {
            double wr = 0.0;
            int it = 0, ru = 0;
            for (int k = 0; k < K; ++k) {
                const TeamStat& s = hs[(size_t)j * np + c * K + k];
                const double rel = s.b2 > 0.0 ? std::sqrt(s.r2true / s.b2) : 0.0;
                if (!(rel <= wr)) wr = rel;
                it = std::max(it, s.iters);
                ru = std::max(ru, s.n_ru);
            }
            iterations[(size_t)j * nc + c] = it;
            worst_resid[(size_t)j * nc + c] = wr;
            reliable_updates[(size_t)j * nc + c] = ru;
        }
    }
    if (f & 2) return fail(ctx, HMC_ERR_NONFINITE, "batched solve: non-finite residual norm");
    if (f & 1) return fail(ctx, HMC_ERR_NOCONV, "batched solve: no convergence in " + std::to_string(ctx->p.cg_maxit) +
                                                   " iterations");
    return HMC_OK;
}

}  // namespace hmc
