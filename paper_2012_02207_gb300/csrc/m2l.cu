// Rotation-accelerated M2L (Sec. 2.4).
//
// For a source cell A and a target cell B with R = z_A - z_B, the source's
// hat multipole is rotated so that R points along +z:
//     Rz(pi/2 - phi), swap x<->z, Rz(-theta), swap x<->z
// (phi, theta the angles of R; swap-Rz-swap is a rotation about x), then
// translated along z in O(p^3):
//     Fhat'_n^m = sum_{k=m}^{p-n} (-1)^{k+m} (n+k)!/(w_n^m w_k^m) Mhat'_k^m u^k v^n / rho,
// with u = s_A/rho, v = s_B/rho, and rotated back with the inverse sequence
//     swap, Rz(theta), swap, Rz(phi - pi/2).
// z-rotations are diagonal (coefficient m times e^{i m angle}); the swap
// matrices of the hat basis are exact tables (cosine and sine blocks, half of
// each block is zero by parity).
//
// The swap right after the z-translation skips the inputs the translation
// leaves zero (F'_n^m = 0 for m > p - n).
//
// One warp per target cell gathers over the target's sources (sorted by
// index); lane l takes sources l, l+32, ... and accumulates its own partial
// local expansion; the 32 partials are summed by a fixed butterfly, so the
// result does not depend on scheduling. This file holds the FP32 kernel; m2l64.cu the FP64 one.
#include "gbfmm_internal.cuh"

namespace gbfmm {

namespace {


// ------------------------------------------------------------------------
// FP32, compile-time order P: coefficients live in registers.

template <int P>
__device__ __forceinline__ void rotz32(float* a, float c, float s) {
    float pr = 1.0f, pi = 0.0f;
#pragma unroll
    for (int m = 1; m <= P; ++m) {
        const float t = pr * c - pi * s;
        pi = pr * s + pi * c;
        pr = t;
#pragma unroll
        for (int n = m; n <= P; ++n) {
            const float re = a[hre(n, m)], im = a[him(n, m)];
            a[hre(n, m)] = re * pr - im * pi;
            a[him(n, m)] = re * pi + im * pr;
        }
    }
}

// swap_lit<P> and ztrans_lit<P>: the swap and z-translation steps with their
// coefficients as literals, generated by gen_m2l.py
#include "m2l_gen.inc"

// LOOPED: how the nine steps are laid out in code. 0: fully unrolled;
// 1: the S Rz S blocks as a two-pass loop; 2: one loop of five passes whose
// body is a z-rotation (or the z-translation) and a swap, the smallest code.
// The unrolled translation code is long enough that instruction fetch
// stalls the warps, so smaller code can run faster despite the loop.
#ifndef GBFMM_M2L_LOOPED
#define GBFMM_M2L_LOOPED 0
#endif

// Blocks per SM the register budget is cut for: three for orders up to
// GBFMM_M2L_MINB3_UPTO (at p = 10 that costs 52 bytes of spills and raises
// residency from 8 to 12 warps per SM), two above.
#ifndef GBFMM_M2L_MINB3_UPTO
#define GBFMM_M2L_MINB3_UPTO 0
#endif
__host__ __device__ constexpr int m2l_min_blocks(int P) { return P <= GBFMM_M2L_MINB3_UPTO ? 3 : 2; }

template <int P, int LOOPED>
__global__ void __launch_bounds__(128, m2l_min_blocks(P)) k_m2l32(const int* __restrict__ dnn, const uint32_t* __restrict__ src,
                                                const uint32_t* __restrict__ off,
                                                const float* __restrict__ mult, int stride,
                                                const float4* __restrict__ zhi,
                                                const float4* __restrict__ zlo,
                                                float* __restrict__ loc, unsigned* __restrict__ queue) {
    constexpr int NR = (P + 1) * (P + 1);
    constexpr int NV = (NR + 3) / 4;  // float4 groups (the multipole stride is padded to 4)
    extern __shared__ float4 sh_acc4[];  // [warp][NV][32]
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    float4* acc = sh_acc4 + (size_t)wib * NV * 32;
    // targets are taken from a shared counter: their source counts differ by
    // orders of magnitude, and a fixed stride leaves SMs idle at the end
    for (;;) {
        int b = 0;
        if (lane == 0) b = (int)atomicAdd(queue, 1u);
        b = __shfl_sync(0xffffffffu, b, 0);
        if (b >= *dnn) break;
#pragma unroll
        for (int j = 0; j < NV; ++j) acc[j * 32 + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
        const uint32_t q0 = off[b], q1 = off[b + 1];
        const float4 bh = zhi[b], bl = zlo[b];
        const float sb = bh.w;
        for (uint32_t q = q0 + lane; q < q1; q += 32) {
            const int a = (int)src[q];
            const float4 ah = zhi[a], al = zlo[a];
            // R = z_A - z_B from double-float centres
            const float rx = (ah.x - bh.x) + (al.x - bl.x), ry = (ah.y - bh.y) + (al.y - bl.y),
                        rz = (ah.z - bh.z) + (al.z - bl.z);
            const float sa = ah.w;
            float c[NV * 4];
            const float4* mv = reinterpret_cast<const float4*>(mult + (size_t)stride * a);
#pragma unroll
            for (int j = 0; j < NV; ++j) {
                const float4 v = __ldg(mv + j);
                c[4 * j] = v.x; c[4 * j + 1] = v.y; c[4 * j + 2] = v.z; c[4 * j + 3] = v.w;
            }
            const float rxy2 = rx * rx + ry * ry;
            const float rho = sqrtf(rxy2 + rz * rz);
            const float rxy = sqrtf(rxy2);
            float cp = 1.0f, sp = 0.0f;
            if (rxy > 0.0f) { cp = rx / rxy; sp = ry / rxy; }
            const float ct = rz / rho, st = rxy / rho;
            const float irho = 1.0f / rho;
            // Rz(pi/2 - phi) S Rz(-theta) S Z S Rz(theta) S Rz(phi - pi/2), with the
            // S Rz S blocks shared by one loop body to halve the code
            if (LOOPED == 2) {
                // Rz(pi/2 - phi) S | Rz(-theta) S | Z S | Rz(theta) S | Rz(phi - pi/2)
#pragma unroll 1
                for (int k = 0; k < 5; ++k) {
                    if (k == 2) {
                        ztrans_lit<P>(c, sa * irho, sb * irho, irho);
                    } else {
                        const float rc = (k == 0 || k == 4) ? sp : ct;
                        const float rs = k == 0 ? cp : (k == 4 ? -cp : (k == 1 ? -st : st));
                        rotz32<P>(c, rc, rs);
                    }
                    if (k < 4) swap_lit<P>(c);
                }
            } else {
            rotz32<P>(c, sp, cp);
            if (LOOPED) {
#pragma unroll 1
                for (int it = 0; it < 2; ++it) {
                    swap_lit<P>(c);
                    rotz32<P>(c, ct, it ? st : -st);
                    swap_lit<P>(c);
                    if (it == 0) ztrans_lit<P>(c, sa * irho, sb * irho, irho);
                }
            } else {
                swap_lit<P>(c);
                rotz32<P>(c, ct, -st);
                swap_lit<P>(c);
                ztrans_lit<P>(c, sa * irho, sb * irho, irho);
                swap_lit_z<P>(c);
                rotz32<P>(c, ct, st);
                swap_lit<P>(c);
            }
            rotz32<P>(c, sp, -cp);
            }
#pragma unroll
            for (int j = 0; j < NV; ++j) {
                float4 v = acc[j * 32 + lane];
                v.x += c[4 * j];
                if (4 * j + 1 < NR) v.y += c[4 * j + 1];
                if (4 * j + 2 < NR) v.z += c[4 * j + 2];
                if (4 * j + 3 < NR) v.w += c[4 * j + 3];
                acc[j * 32 + lane] = v;
            }
        }
        __syncwarp();
        float* out = loc + (size_t)NR * b;  // locals keep the unpadded stride
        const float* accf = reinterpret_cast<const float*>(acc);
        for (int j = 0; j < NR; ++j) {
            float v = accf[((j >> 2) * 32 + lane) * 4 + (j & 3)];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) out[j] = v;
        }
        __syncwarp();
    }
}

template <int P>
void launch_m2l32(const int* dnn, const uint32_t* src, const uint32_t* off, const float* mult,
                  int stride, const float4* zhi, const float4* zlo, float* loc, unsigned* queue,
                  cudaStream_t st) {
    const size_t sh = (size_t)4 * (((P + 1) * (P + 1) + 3) / 4) * 32 * sizeof(float4);
    ensure_dyn_smem((const void*)k_m2l32<P, GBFMM_M2L_LOOPED>, (int)sh);
    (k_m2l32<P, GBFMM_M2L_LOOPED><<<device_sm_count() * m2l_min_blocks(P), 128, sh, st>>>(dnn, src, off, mult, stride, zhi, zlo, loc, queue),
     note_launch());
}
}  // namespace

void m2l_f32(const int* dnn, int p, const uint32_t* src, const uint32_t* off,
             const float* mult, const float4* zhi, const float4* zlo, float* loc, unsigned* queue,
             cudaStream_t st) {
    cudaMemsetAsync(queue, 0, sizeof(unsigned), st);
    const int stride = (ncoef_real(p) + 3) & ~3;  // padded for float4 loads
    switch (p) {
        case 4: launch_m2l32<4>(dnn, src, off, mult, stride, zhi, zlo, loc, queue, st); break;
        case 6: launch_m2l32<6>(dnn, src, off, mult, stride, zhi, zlo, loc, queue, st); break;
        case 8: launch_m2l32<8>(dnn, src, off, mult, stride, zhi, zlo, loc, queue, st); break;
        case 10: launch_m2l32<10>(dnn, src, off, mult, stride, zhi, zlo, loc, queue, st); break;
        case 12: launch_m2l32<12>(dnn, src, off, mult, stride, zhi, zlo, loc, queue, st); break;
        case 14: launch_m2l32<14>(dnn, src, off, mult, stride, zhi, zlo, loc, queue, st); break;
        default: break;  // other orders run the FP64 kernel (the caller checks m2l32_supported)
    }
}

bool m2l32_supported(int p) { return p == 4 || p == 6 || p == 8 || p == 10 || p == 12 || p == 14; }

}  // namespace gbfmm
