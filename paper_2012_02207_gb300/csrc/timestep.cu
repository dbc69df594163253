// Per-body step sizes of the HOLD integrator (Appendix A).
//
// Compiled with -fmad=false: every step size is a plain function of the
// pair's FP64 data (one IEEE operation per source operation), so the split
// of a set into fast and slow bodies is reproducible bit for bit.
//
// The exact pair step takes about 150 FP64 instructions (square roots and
// divisions), and GB300 runs each for 64 cycles of a scheduler, but a body
// needs only the smallest of its pair steps. So two passes bound every pair
// step in FP32 first (hold_bounds.cuh): the first finds the smallest upper
// bound of each body, the second evaluates exactly only the pairs whose lower
// bound does not exceed it, one or two a body. The minimum is the exact one.
#include "gbfmm_internal.cuh"
#include "hold_bounds.cuh"
#include "hold_pair.cuh"

namespace gbfmm {

namespace {

constexpr int kStepThreads = 256;

struct StepBodies {
    const double *x, *y, *z, *vx, *vy, *vz, *m;
};

// Block (t, s): the pairs of 256 bodies with segment s of all bodies.
// EXACT = false: upper[i] <- the smallest FP32 upper bound (as an integer: the
// bounds are positive), tau[i] <- infinity. EXACT = true: tau[i] <- the smallest
// exact pair step (the bits of a positive double order like the number).
template <bool EXACT>
__global__ void __launch_bounds__(kStepThreads) k_timesteps(int n, StepBodies B, double G, double eta, int sym,
                                                            int seg, unsigned* __restrict__ upper,
                                                            unsigned long long* __restrict__ tau) {
    __shared__ PairBody32 sh[kStepThreads];
    const int i = blockIdx.x * kStepThreads + threadIdx.x;
    const bool act = i < n;
    const int ii = act ? i : 0;
    const double xi = B.x[ii], yi = B.y[ii], zi = B.z[ii], ui = B.vx[ii], vi = B.vy[ii], wi = B.vz[ii], mi = B.m[ii];
    const PairBody32 me(xi, yi, zi, ui, vi, wi, mi);
    const PairScale32 scale(me, G, eta);
    float up = __int_as_float(0x7f800000);  // +infinity
    const float limit = EXACT && act ? __uint_as_float(upper[i]) : up;
    double t = CUDART_INF;
    const int jb = (int)blockIdx.y * seg, je = jb + seg < n ? jb + seg : n;
    for (int j0 = jb; j0 < je; j0 += kStepThreads) {
        const int j = j0 + threadIdx.x;
        if (j < je) sh[threadIdx.x] = PairBody32(B.x[j], B.y[j], B.z[j], B.vx[j], B.vy[j], B.vz[j], B.m[j]);
        __syncthreads();
        const int cnt = je - j0 < kStepThreads ? je - j0 : kStepThreads;
        const int self = act ? i - j0 : -1;
#pragma unroll 2
        for (int k = 0; k < cnt; ++k) {
            float lo, hi;
            pair_bounds32(me, sh[k], scale, sym != 0, lo, hi);
            if (!EXACT) {
                if (k != self) up = fminf(up, hi);
            } else if (act && k != self && !(lo > limit)) {
                const int jj = j0 + k;
                const double tij = tau_pair(B.x[jj] - xi, B.y[jj] - yi, B.z[jj] - zi, B.vx[jj] - ui, B.vy[jj] - vi,
                                            B.vz[jj] - wi, mi + B.m[jj], G, eta, sym != 0);
                t = tij < t ? tij : t;
            }
        }
        __syncthreads();
    }
    if (!act) return;
    if (!EXACT) {
        atomicMin(upper + i, __float_as_uint(up));
        if (blockIdx.y == 0) tau[i] = (unsigned long long)__double_as_longlong(CUDART_INF);
    } else if (t < CUDART_INF) {
        atomicMin(tau + i, (unsigned long long)__double_as_longlong(t));
    }
}

}  // namespace

void timesteps_f64(int n, const double* x, const double* y, const double* z, const double* vx, const double* vy,
                   const double* vz, const double* m, double G, double eta, bool sym, double* tau, unsigned* upper,
                   cudaStream_t st) {
    if (n <= 0) return;
    // segments: four blocks of 256 per SM in all, at least 256 sources each
    const int blocks = (n + kStepThreads - 1) / kStepThreads;
    int nseg = 4 * device_sm_count() / blocks;
    const int most = (n + kStepThreads - 1) / kStepThreads;
    nseg = nseg < 1 ? 1 : (nseg > most ? most : nseg);
    const int seg = (n + nseg - 1) / nseg;
    const dim3 grid(blocks, nseg);
    const StepBodies B{x, y, z, vx, vy, vz, m};
    unsigned long long* out = reinterpret_cast<unsigned long long*>(tau);
    cudaMemsetAsync(upper, 0x7f, sizeof(unsigned) * (size_t)n, st);  // 3.4e38: above every finite bound of use
    (k_timesteps<false><<<grid, kStepThreads, 0, st>>>(n, B, G, eta, sym ? 1 : 0, seg, upper, out), note_launch());
    (k_timesteps<true><<<grid, kStepThreads, 0, st>>>(n, B, G, eta, sym ? 1 : 0, seg, upper, out), note_launch());
}

}  // namespace gbfmm
