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
// The bounds are taken in units of the bodies' own lengths and masses (k_step_scale),
// whatever the caller's: in SI units, outside the bounds' ranges, and from rest
// every pair was evaluated exactly (16384 bodies from rest 45.9 -> 3.5 ms, 65536 824 -> 60,
// 65536 in SI units 1208 -> 42; N-body units, 16384 bodies: 2.52, now 2.48).
#include "gbfmm_internal.cuh"
#include "hold_bounds.cuh"
#include "hold_pair.cuh"

namespace gbfmm {

namespace {

constexpr int kStepThreads = 256;

struct StepBodies {
    const double *x, *y, *z, *vx, *vy, *vz, *m;
};

// Factors to the units of the bounds: powers of two for lengths and speeds, and G with one for masses.
struct StepScale {
    float l, v, g;
};

// The exponent of the largest of three coordinates' magnitudes; false if zero or not finite.
__device__ __forceinline__ bool exponent_of(double x, double y, double z, int& e) {
    const unsigned a = (unsigned)__double2hiint(x) & 0x7fffffffu, b = (unsigned)__double2hiint(y) & 0x7fffffffu,
                   c = (unsigned)__double2hiint(z) & 0x7fffffffu;
    const unsigned m = a > b ? (a > c ? a : c) : (b > c ? b : c);
    e = (int)(m >> 20) - 1023;
    return m >= 1u << 20 && m < 0x7ff00000u;
}

// The units of up to 4096 bodies: the mean exponents of distance and mass, and the speed that goes
// with them. (A few bodies far out shift a mean little; the bounds hold in any units, only more pairs
// are then out of their ranges.)
__global__ void __launch_bounds__(1024) k_step_scale(int n, StepBodies B, double G, StepScale* __restrict__ out) {
    __shared__ int sum[4];  // of distances' and masses' exponents, and how many
    if (threadIdx.x < 4) sum[threadIdx.x] = 0;
    __syncthreads();
    const int stride = (n + 4095) / 4096;
    int v[4] = {0, 0, 0, 0};
    for (int64_t i = (int64_t)threadIdx.x * stride; i < n; i += (int64_t)1024 * stride) {
        int e;
        if (exponent_of(B.x[i], B.y[i], B.z[i], e)) { v[0] += e; ++v[1]; }
        if (exponent_of(B.m[i], 0.0, 0.0, e)) { v[2] += e; ++v[3]; }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int s = __reduce_add_sync(0xffffffffu, v[k]);
        if ((threadIdx.x & 31) == 0) atomicAdd(&sum[k], s);
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    const int el = sum[1] ? sum[0] / sum[1] : 0, em = sum[3] ? sum[2] / sum[3] : 0;
    int eg;
    if (!exponent_of(G, 0.0, 0.0, eg)) eg = 0;
    const int ev = (eg + em + 1 - el) >> 1;
    *out = StepScale{scalbnf(1.0f, -el), scalbnf(1.0f, -ev), (float)scalbn(G, -2 * ev - el)};
}

// Block (t, s): the pairs of 256 bodies with segment s of all bodies.
// EXACT = false: upper[i] <- the smallest FP32 upper bound (as an integer: the
// bounds are positive), tau[i] <- infinity. EXACT = true: tau[i] <- the smallest
// exact pair step (the bits of a positive double order like the number).
template <bool EXACT>
__global__ void __launch_bounds__(kStepThreads) k_timesteps(int n, StepBodies B, double G, double eta, int sym,
                                                            int seg, const StepScale* __restrict__ units,
                                                            unsigned* __restrict__ upper,
                                                            unsigned long long* __restrict__ tau) {
    __shared__ PairBody32 sh[kStepThreads];
    const int i = blockIdx.x * kStepThreads + threadIdx.x;
    const bool act = i < n;
    const int ii = act ? i : 0;
    const double xi = B.x[ii], yi = B.y[ii], zi = B.z[ii], ui = B.vx[ii], vi = B.vy[ii], wi = B.vz[ii], mi = B.m[ii];
    const StepScale to = *units;
    PairBody32 me(xi, yi, zi, ui, vi, wi, mi);
    me.scale(to.l, to.v, to.g);
    const PairScale32 scale(me, 1.0, eta);
    float up = __int_as_float(0x7f800000);  // +infinity
    const float limit = EXACT && act ? __uint_as_float(upper[i]) : up;
    double t = CUDART_INF;
    const int jb = (int)blockIdx.y * seg, je = jb + seg < n ? jb + seg : n;
    for (int j0 = jb; j0 < je; j0 += kStepThreads) {
        const int j = j0 + threadIdx.x;
        if (j < je) {
            PairBody32 b(B.x[j], B.y[j], B.z[j], B.vx[j], B.vy[j], B.vz[j], B.m[j]);
            b.scale(to.l, to.v, to.g);
            sh[threadIdx.x] = b;
        }
        __syncthreads();
        const int cnt = je - j0 < kStepThreads ? je - j0 : kStepThreads;
        const int self = act ? i - j0 : -1;
#pragma unroll 2
        for (int k = 0; k < cnt; ++k) {
            float lo, hi;
            pair_bounds32(me, sh[k], scale, sym != 0,
                          [&] {
                              return same_number(B.vx[j0 + k], ui) && same_number(B.vy[j0 + k], vi) &&
                                     same_number(B.vz[j0 + k], wi);
                          },
                          lo, hi);
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

// the units, in 16 bytes, and an upper bound per body
size_t timesteps_scratch_bytes(int64_t n) { return 16 + sizeof(unsigned) * (size_t)n; }

void timestep_units(int n, const double* x, const double* y, const double* z, const double* m, double G, void* scratch,
                    cudaStream_t st) {
    static_assert(sizeof(StepScale) <= 16, "scratch");
    if (n > 0)
        (k_step_scale<<<1, 1024, 0, st>>>(n, StepBodies{x, y, z, nullptr, nullptr, nullptr, m}, G,
                                          static_cast<StepScale*>(scratch)),
         note_launch());
}

void timesteps_f64(int n, const double* x, const double* y, const double* z, const double* vx, const double* vy,
                   const double* vz, const double* m, double G, double eta, bool sym, double* tau, void* scratch,
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
    const StepScale* units = static_cast<const StepScale*>(scratch);
    unsigned* upper = reinterpret_cast<unsigned*>(static_cast<unsigned char*>(scratch) + 16);
    cudaMemsetAsync(upper, 0x7f, sizeof(unsigned) * (size_t)n, st);  // 3.4e38: above every finite bound of use
    (k_timesteps<false><<<grid, kStepThreads, 0, st>>>(n, B, G, eta, sym ? 1 : 0, seg, units, upper, out), note_launch());
    (k_timesteps<true><<<grid, kStepThreads, 0, st>>>(n, B, G, eta, sym ? 1 : 0, seg, units, upper, out), note_launch());
}

}  // namespace gbfmm
