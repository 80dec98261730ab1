// FFT steps over lines in shared memory for lengths known at run time: N = n1 n2 with both factors among
// the register DFTs of dft.cuh, done in place. With n = a + n1 b and k = c + n2 d,
//   step A (fixed a): n2-point DFT over b, times w_N^{a c}, back to position a + n1 c;
//   step B (fixed c): n1-point DFT over a at positions n1 c + a, back in place.
// Position n1 c + d then holds frequency c + n2 d. The inverse runs step B, then A, on data with re and im
// exchanged (the inverse transform is the forward one between two exchanges).
#pragma once

#include "dft.cuh"
#include "internal.h"

namespace hmc {

// The tile holds `np` planes of `nl` lines, `plane` entries apart; line l of a plane starts at
// (l & 1) * l1 + (l >> 1) * ls, the points of DFT f at f * fs + m * ps; with tw, output m is multiplied by
// tw[f m].
struct Lines {
    int np, plane, nl;
    FastDiv dnl;
    int l1, ls;
};

template <int R, typename C>
__device__ __noinline__ void dft_pass(C* sm, const Lines ln, int nf, int fs, int ps, const C* tw) {
    const int total = ln.np * ln.nl * nf;
    for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
        const int q = fdiv(idx, ln.dnl), l = idx - q * ln.nl;   // q = plane * nf + f
        int p = 0, f = q;
        if (ln.np > 1) { p = q / nf; f = q - p * nf; }
        C* base = sm + p * ln.plane + (l & 1) * ln.l1 + (l >> 1) * ln.ls + f * fs;
        C v[R];
#pragma unroll
        for (int m = 0; m < R; ++m) v[m] = tile_at(base, m * ps);
        bfly<R, -1>(v);
        if (tw) {
#pragma unroll
            for (int m = 1; m < R; ++m) v[m] = cmul(v[m], tw[f * m]);
        }
#pragma unroll
        for (int m = 0; m < R; ++m) tile_at(base, m * ps) = v[m];
    }
}
template <typename C>
__device__ __forceinline__ void dft_step(int R, C* sm, const Lines& ln, int nf, int fs, int ps, const C* tw) {
    if (R == 1) return;
    switch (R) {
        case 2: dft_pass<2>(sm, ln, nf, fs, ps, tw); break;
        case 3: dft_pass<3>(sm, ln, nf, fs, ps, tw); break;
        case 4: dft_pass<4>(sm, ln, nf, fs, ps, tw); break;
        case 5: dft_pass<5>(sm, ln, nf, fs, ps, tw); break;
        case 6: dft_pass<6>(sm, ln, nf, fs, ps, tw); break;
        case 7: dft_pass<7>(sm, ln, nf, fs, ps, tw); break;
        case 8: dft_pass<8>(sm, ln, nf, fs, ps, tw); break;
        case 9: dft_pass<9>(sm, ln, nf, fs, ps, tw); break;
        case 10: dft_pass<10>(sm, ln, nf, fs, ps, tw); break;
        case 12: dft_pass<12>(sm, ln, nf, fs, ps, tw); break;
        case 14: dft_pass<14>(sm, ln, nf, fs, ps, tw); break;
        case 15: dft_pass<15>(sm, ln, nf, fs, ps, tw); break;
        case 16: dft_pass<16>(sm, ln, nf, fs, ps, tw); break;
        default: break;
    }
    __syncthreads();
}
// Both steps along an axis of entry stride `st`; tw: e^{-2 pi i k / N} in shared memory.
template <typename C>
__device__ __forceinline__ void dft_forward(C* sm, const Lines& ln, int n1, int n2, int st, const C* tw) {
    dft_step(n2, sm, ln, n1, st, st * n1, tw);
    dft_step(n1, sm, ln, n2, st * n1, st, (const C*)nullptr);
}
template <typename C>
__device__ __forceinline__ void dft_inverse(C* sm, const Lines& ln, int n1, int n2, int st, const C* tw) {
    dft_step(n1, sm, ln, n2, st * n1, st, tw);
    dft_step(n2, sm, ln, n1, st, st * n1, (const C*)nullptr);
}
template <typename C> __device__ __forceinline__ C swapc(C a) { return mk<C>(a.y, a.x); }
// frequency at position p after the forward steps, and the position of a frequency
__device__ __forceinline__ int dft_freq(int p, int n1, int n2) { return p / n1 + n2 * (p % n1); }
__device__ __forceinline__ int dft_pos(int k, int n1, int n2) { return n1 * (k % n2) + k / n2; }

// ---- host --------------------------------------------------------------------------------------------
// N = n1 n2 with both factors among dft_step's radices, their sum (the work per point) least; up to 10
// points in one step: a step costs its latency, not its work, at the sizes that take few points. spread: two steps
// from 6 points on, for FP64 (a warp's operation takes its quarter of the SM's FP64 pipe 64 clocks however few lanes
// are at work, 56 of them for 8 points by a thread, 24 in two steps by four and two): PCG in one launch 28.9 -> 23.9 us
// an iteration at 8 x 8 x 8, 38.6 -> 30.6 at 10 x 10 x 10; the drift 30.2 -> 24.6 at 8 x 8 x 8, 36.9 -> 28.7 at
// 10 x 10 x 10; the complex128 preconditioner 34.8 -> 28.4 there. Many lines lose nothing: 133 -> 122 at 10 x 10 x 96
// with 8 right-hand sides.
// False when there is none.
inline bool dft_split(int n, int* n1, int* n2, bool spread = false) {
    static const int radix[] = {1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 14, 15, 16};
    if (n <= (spread ? 5 : 10)) {
        *n1 = n;
        *n2 = 1;
        return true;
    }
    int best = 1 << 30;
    for (int a : radix)
        for (int b : radix)
            if (a * b == n && a >= b && a + b < best) {
                best = a + b;
                *n1 = a;
                *n2 = b;
            }
    return best < (1 << 30);
}

}  // namespace hmc
