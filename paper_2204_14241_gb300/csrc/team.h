// Arguments of the one-launch team solver (team.cu).
#pragma once

#include "internal.h"

namespace hmc {

constexpr int kTeamSmem = 216 * 1024;   // dynamic shared memory of a preconditioned block, at most
constexpr int kTeamTau = 64;      // most sites of a tau tile

// One (chain, right-hand side) pair of a batched solve.
struct TeamPair {
    int chain, k;
};

// Preconditioner tables (device) and splits L = x1 x2, Nt = t1 t2 of the PCG phases.
template <typename R> struct TeamPre {
    const cplx<R>*twx, *twt, *eitw, *twist;
    const R* cosk;
    R c0[2], chx[2], chy[2];   // K-hat = e^{i w} + c0 + chx cos kx + chy cos ky
    double scale;
    int x1, x2, t1, t2;
    int W;                     // sites of a tau tile
    FastDiv d2L, dw2, dW;      // by 2 L, 2 W and W
    int plane, np;             // complex entries of a plane in the shared FFT tile, planes at a time
    int tile;                  // entries of the tile
};

template <typename R> struct TeamArgs {
    const TeamPair* pairs;     // batched: the queue, npairs entries; otherwise null, a right-hand side of `one` per team
    int npairs, nteams;
    const int* blk;            // batched: the team of each block
    const int2* team;          // batched: first block and blocks of each team
    int *queue, *next;         // batched: entries taken (null: team j solves pair j); the entry each team takes next
    const BChainDev* ch;
    BChainDev one;
    int T, K;
    Coef<R> cf;
    Coef<double> cf64;
    const double2* b;
    double2 *x64, *t64;        // solution; its D^dagger image at the last true residual
    cplx<R> *x, *r, *pA, *pB, *t, *z;   // x: FP32 iterate (mixed); pB: second direction (mixed CG); z: PCG
    unsigned* bar;             // an arrival counter per team, and one word behind them, zeroed before the launch
    unsigned long long* part;  // [2][blocks] partial sums
    int* flags;                // device error word
    int* fail;                 // OR of the pairs' failure flags (may be null)
    TeamStat* stat;            // per pair, chain * K + k (may be null)
    double tol2, delta2;
    int maxit, use_x0, test_timeout;
    long long timeout_ns;
    TeamPre<R> pre;
};

void team_geometry(BChainDev* d, const Lat& lat);
int team_batch_capacity(hmc_ctx* ctx, int* cap);
int team_launch_batch(hmc_ctx* ctx, const TeamArgs<float>& a, int grid);
// Solves all right-hand sides in one launch (cg_run's contract); *done = false where the size, the
// lattice's factors or the workspace rule that out and nothing was launched.
int team_solve(hmc_ctx* ctx, const Lat& lat, const double* phi, const double2* b, double2* x, int nrhs, double tol,
               int maxit, int precond, hmc_cg_stats* st, bool use_x0, bool* y_ready, bool* done);

}  // namespace hmc
