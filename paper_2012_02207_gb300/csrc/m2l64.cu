// Rotation-accelerated M2L (Sec. 2.4) in FP64, any order p <= 30: the steps of
// m2l.cu,
//     Rz(pi/2 - phi) S Rz(-theta) S  z-translation  S Rz(theta) S Rz(phi - pi/2),
// one source per lane, a block of four warps per target cell.
//
// GB300 runs an FP64 instruction of a warp for 64 cycles of its scheduler, so
// the FP64 operations are what bounds the kernel (about 2,860 per source at
// p = 10) as long as everything else stays out of their way:
//  - the swaps are unrolled per degree: the degree's outputs accumulate in
//    registers while its inputs come one order at a time, so each input is read
//    once and up to n independent chains are in flight;
//  - a lane's coefficients and sums are per-thread arrays (local memory, which
//    the hardware interleaves by lane). Few warps per SM are enough to fill the
//    FP64 pipe and keep those arrays in L1 and L2; 32 warps per SM put 300 MB
//    of them through HBM;
//  - the swap before the z-translation forms only the orders m <= p - n that
//    the translation reads, the one after it reads only those that it left
//    non-zero;
//  - the translation's coefficient (n+k)! / (w_n^m w_k^m) is split, 1/w_k^m
//    going to the input with u^k and 1/w_n^m to the output with v^n;
//  - the powers of both angles are formed once per source and serve a rotation
//    and its inverse.
// N = 100000, p = 10 (3.29 M sources): 50.8 -> 24.3 ms, the FP64 pipe at 70% of
// its cycles; N = 4096, p = 8: 1.08 -> 0.29 ms.
#include "gbfmm_internal.cuh"
#include "swap_tables.cuh"

namespace gbfmm {

namespace {

// One z-rotation and swap of a degree: reads the 2n + 1 reals of degree N at
// src (orders j <= jmax; the others are zero), multiplies order j by pw_j (its
// conjugate if conj; pw NULL: no rotation), swaps x and z, and writes the
// outputs to dst; with pwo the outputs are multiplied by conj(pwo_m) and added to
// dst. src and dst may be the same.
struct SwapPass {
    const double* pw;
    bool conj;
    const double* pwo;
    const double* cosb;
    const double* sinb;
};

template <int N>
__device__ __forceinline__ void load_order(const double* src, const SwapPass& s, int j, double& re, double& im) {
    re = src[j ? 2 * j - 1 : 0];
    im = j ? src[2 * j] : 0.0;
    if (j && s.pw) {
        const double pr = s.pw[2 * j], pi = s.conj ? -s.pw[2 * j + 1] : s.pw[2 * j + 1];
        const double t = re * pr - im * pi;
        im = re * pi + im * pr;
        re = t;
    }
}

template <int N>
__device__ __noinline__ void swap_all(const double* src, SwapPass s, int jmax, double* dst) {
    const double* A = s.cosb + cos_off(N);
    const double* B = s.sinb + sin_off(N);
    double tc[N + 1], ts[N + 1];
#pragma unroll
    for (int m = 0; m <= N; ++m) { tc[m] = 0.0; ts[m] = 0.0; }
#pragma unroll
    for (int j = 0; j <= N; ++j) {
        if (j <= jmax) {
            double re, im;
            load_order<N>(src, s, j, re, im);
#pragma unroll
            for (int m = (j + N) & 1; m <= N; m += 2) tc[m] += __ldg(A + m * (N + 1) + j) * re;
            if (j)
#pragma unroll
                for (int m = ((j + N + 1) & 1) ? 1 : 2; m <= N; m += 2) ts[m] += __ldg(B + (m - 1) * N + (j - 1)) * im;
        }
    }
    if (s.pwo) {
        dst[0] += tc[0];
#pragma unroll
        for (int m = 1; m <= N; ++m) {
            const double pr = s.pwo[2 * m], pi = -s.pwo[2 * m + 1];
            dst[2 * m - 1] += tc[m] * pr - ts[m] * pi;
            dst[2 * m] += tc[m] * pi + ts[m] * pr;
        }
    } else {
        dst[0] = tc[0];
#pragma unroll
        for (int m = 1; m <= N; ++m) {
            dst[2 * m - 1] = tc[m];
            dst[2 * m] = ts[m];
        }
    }
}

// the same, forming only the outputs of orders m <= mmax (the inputs in
// registers, one output at a time)
template <int N>
__device__ __noinline__ void swap_low(const double* src, SwapPass s, int mmax, double* dst) {
    const double* A = s.cosb + cos_off(N);
    const double* B = s.sinb + sin_off(N);
    double xc[N + 1], xs[N + 1];
#pragma unroll
    for (int j = 0; j <= N; ++j) load_order<N>(src, s, j, xc[j], xs[j]);
#pragma unroll
    for (int m = 0; m <= N; ++m) {
        if (m <= mmax) {
            double c0 = 0.0, s0 = 0.0;
#pragma unroll
            for (int j = (m + N) & 1; j <= N; j += 2) c0 += __ldg(A + m * (N + 1) + j) * xc[j];
            dst[m ? 2 * m - 1 : 0] = c0;
            if (m) {
#pragma unroll
                for (int j = ((m + N + 1) & 1) ? 1 : 2; j <= N; j += 2) s0 += __ldg(B + (m - 1) * N + (j - 1)) * xs[j];
                dst[2 * m] = s0;
            }
        }
    }
}

template <int N = 1>
__device__ __forceinline__ void swap_all_n(int n, const double* src, const SwapPass& s, int jmax, double* dst) {
    if (n == N) swap_all<N>(src, s, jmax, dst);
    else if constexpr (N < kMaxP) swap_all_n<N + 1>(n, src, s, jmax, dst);
}
template <int N = 1>
__device__ __forceinline__ void swap_low_n(int n, const double* src, const SwapPass& s, int mmax, double* dst) {
    if (n == N) swap_low<N>(src, s, mmax, dst);
    else if constexpr (N < kMaxP) swap_low_n<N + 1>(n, src, s, mmax, dst);
}

// F'_n^m = v^n / (rho w_n^m) sum_{k=m}^{p-n} (n+k)! [(-1)^{k+m} u^k c_k^m / w_k^m], in place, for n, k <= p - m
template <int PM>
__device__ void ztrans64(double* a, int p, double u, double v, double irho, const double* __restrict__ fact,
                         const double* __restrict__ iw) {
    double up[PM + 1], vp[PM + 1], tr[PM + 1], ti[PM + 1];
    double pu = 1.0, pv = irho;
    for (int k = 0; k <= p; ++k) {
        up[k] = k & 1 ? -pu : pu;
        vp[k] = pv;
        pu *= u;
        pv *= v;
    }
    for (int m = 0; 2 * m <= p; ++m) {
        const int kmax = p - m;
        for (int k = m; k <= kmax; ++k) {
            const double f = up[k] * __ldg(iw + k * (kMaxP + 2) + m);  // (the sign of (-1)^m goes to the output)
            tr[k] = f * a[hre(k, m)];
            ti[k] = m ? f * a[him(k, m)] : 0.0;
        }
        for (int n = m; n <= kmax; ++n) {
            double sr = 0.0, si = 0.0;
            const double* fn = fact + n;
#pragma unroll 4
            for (int k = m; k <= p - n; ++k) {
                const double f = __ldg(fn + k);
                sr += f * tr[k];
                if (m) si += f * ti[k];
            }
            const double g = vp[n] * __ldg(iw + n * (kMaxP + 2) + m);
            a[hre(n, m)] = m & 1 ? -g * sr : g * sr;
            if (m) a[him(n, m)] = m & 1 ? -g * si : g * si;
        }
    }
}

// Halving step of the transpose reduction: C values per lane become C/2; a
// lane with bit o set keeps the upper half and receives its partner's.
template <int C>
__device__ __forceinline__ void halve64(double* v, int lane, int o) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < C / 2; ++i) {
        const double send = up ? v[i] : v[i + C / 2];
        const double keep = up ? v[i + C / 2] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
}

constexpr int kM2L64Warps = 4;
// blocks per SM: 2, 3, 4 and 5 took 26.2, 23.0, 23.3 and 23.3 ms at N = 100000, p = 10
constexpr int kM2L64Blocks = 3;

// PM bounds the per-thread arrays (p <= PM). A target's sources are dealt in
// batches of 32 to the kM2L64Warps warps of a block; every warp sums its batches
// per lane, then its lanes, and the warps' parts are added in order. With a target
// to each warp, which this kernel had for larger trees, the warps of an SM gather
// from all over the tree: beside 160 MB of per-thread arrays the multipoles no longer
// stay in L2 (2^20 bodies: p = 12 810 ms against 271, p = 10 766 against 329). Lists of
// under 97 sources leave warps of the block idle; whole solves at loose tolerances,
// against a warp per target without the rest of this file's changes, ms: 2^20 bodies,
// p = 4, eps = 1e-3 51.5 -> 34.8; 300000 in leaves of 16, p = 2, eps = 0.1 11.0 -> 8.5.
template <int PM>
__global__ void __launch_bounds__(32 * kM2L64Warps, kM2L64Blocks)
    k_m2l64(const int* __restrict__ dnn, int p, const uint32_t* __restrict__ src,
            const uint32_t* __restrict__ off, const double* __restrict__ mult, const double* __restrict__ zc,
            const double* __restrict__ hs, double* __restrict__ loc, Swap64 sw, const double* __restrict__ fact,
            const double* __restrict__ iw, unsigned* __restrict__ queue) {
    extern __shared__ double red[];  // the target's sums per part
    __shared__ int s_target;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int nr = ncoef_real(p);
    double c[ncoef_real(PM)], acc[ncoef_real(PM)], pa[2 * (PM + 1)], pb[2 * (PM + 1)];
    for (;;) {
        __syncthreads();  // the previous target's sums and number are consumed
        if (threadIdx.x == 0) s_target = (int)atomicAdd(queue, 1u);
        __syncthreads();
        const int b = s_target;
        if (b >= *dnn) break;
        const uint32_t q0 = off[b], q1 = off[b + 1];
        const int nbatch = (int)((q1 - q0 + 31) / 32);
        const int nparts = nbatch < 1 ? 1 : (nbatch < kM2L64Warps ? nbatch : kM2L64Warps);
        double* out = loc + (size_t)nr * b;
        const double bx = zc[3 * b], by = zc[3 * b + 1], bz = zc[3 * b + 2];
        const double sb = hs[b];
        if (wib < nparts) {
            for (int j = 0; j < nr; ++j) acc[j] = 0.0;
            for (uint32_t q = q0 + 32 * wib + lane; q < q1; q += 32 * kM2L64Warps) {
                const int a = (int)src[q];
                const double rx = zc[3 * a] - bx, ry = zc[3 * a + 1] - by, rz = zc[3 * a + 2] - bz;
                const double sa = hs[a];
                const double* mv = mult + (size_t)nr * a;
                const double rxy2 = rx * rx + ry * ry;
                const double rho = sqrt(rxy2 + rz * rz);
                const double rxy = sqrt(rxy2);
                const double irho = 1.0 / rho;
                double cp = 1.0, sp = 0.0;
                if (rxy > 0.0) {
                    const double irxy = 1.0 / rxy;
                    cp = rx * irxy;
                    sp = ry * irxy;
                }
                const double ct = rz * irho, st = rxy * irho;
                // (sin phi + i cos phi)^m and (cos theta - i sin theta)^m
                double ar = 1.0, ai = 0.0, br = 1.0, bi = 0.0;
                for (int m = 1; m <= p; ++m) {
                    const double ta = ar * sp - ai * cp, tb = br * ct + bi * st;
                    ai = ar * cp + ai * sp;
                    bi = bi * ct - br * st;
                    ar = ta;
                    br = tb;
                    pa[2 * m] = ar; pa[2 * m + 1] = ai;
                    pb[2 * m] = br; pb[2 * m + 1] = bi;
                }
                c[0] = mv[0];
                for (int n = 1; n <= p; ++n) {
                    const int low = n < p - n ? n : p - n;  // orders the translation reads
                    swap_all_n(n, mv + n * n, SwapPass{pa, false, nullptr, sw.cosb, sw.sinb}, n, c + n * n);
                    swap_low_n(n, c + n * n, SwapPass{pb, false, nullptr, sw.cosb, sw.sinb}, low, c + n * n);
                }
                ztrans64<PM>(c, p, sa * irho, sb * irho, irho, fact, iw);
                acc[0] += c[0];
                for (int n = 1; n <= p; ++n) {
                    const int low = n < p - n ? n : p - n;  // orders the translation left non-zero
                    swap_all_n(n, c + n * n, SwapPass{nullptr, false, nullptr, sw.cosb, sw.sinb}, low, c + n * n);
                    swap_all_n(n, c + n * n, SwapPass{pb, true, pa, sw.cosb, sw.sinb}, n, acc + n * n);
                }
            }
            __syncwarp();
            // the lanes' sums, 32 coefficients at a time: lane l ends with coefficient j0 + l
            for (int j0 = 0; j0 < nr; j0 += 32) {
                double v[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = j0 + i < nr ? acc[j0 + i] : 0.0;
                halve64<32>(v, lane, 16);
                halve64<16>(v, lane, 8);
                halve64<8>(v, lane, 4);
                halve64<4>(v, lane, 2);
                halve64<2>(v, lane, 1);
                if (j0 + lane < nr) red[(size_t)wib * nr + j0 + lane] = v[0];
            }
        }
        __syncthreads();
        for (int j = threadIdx.x; j < nr; j += 32 * kM2L64Warps) {
            double s = red[j];
            for (int w = 1; w < nparts; ++w) s += red[(size_t)w * nr + j];
            out[j] = s;
        }
    }
}

template <int PM>
void launch_m2l64(const int* dnn, int p, const uint32_t* src, const uint32_t* off, const double* mult,
                  const double* zc, const double* hs, double* loc, const DevTables& tb, unsigned* queue,
                  cudaStream_t st) {
    const int sh = kM2L64Warps * ncoef_real(p) * (int)sizeof(double);
    (k_m2l64<PM><<<device_sm_count() * kM2L64Blocks, 32 * kM2L64Warps, sh, st>>>(
         dnn, p, src, off, mult, zc, hs, loc, Swap64{tb.swap_cos, tb.swap_sin}, tb.fact, tb.iw, queue),
     note_launch());
}

}  // namespace

void m2l_f64(const int* dnn, int p, const uint32_t* src, const uint32_t* off, const double* mult,
             const double* zc, const double* hs, double* loc, const DevTables& tb, unsigned* queue, cudaStream_t st) {
    cudaMemsetAsync(queue, 0, sizeof(unsigned), st);
    if (p <= 16) launch_m2l64<16>(dnn, p, src, off, mult, zc, hs, loc, tb, queue, st);
    else launch_m2l64<kMaxP>(dnn, p, src, off, mult, zc, hs, loc, tb, queue, st);
}

}  // namespace gbfmm
