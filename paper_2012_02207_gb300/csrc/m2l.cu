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

// The rotation and scale of one pair.
struct PairGeo {
    float sp, cp, ct, st, u, v, irho;
};
__device__ __forceinline__ PairGeo pair_geo(float4 ah, float4 al, float4 bh, float4 bl) {
    // R = z_A - z_B from double-float centres
    const float rx = (ah.x - bh.x) + (al.x - bl.x), ry = (ah.y - bh.y) + (al.y - bl.y),
                rz = (ah.z - bh.z) + (al.z - bl.z);
    const float sa = ah.w, sb = bh.w;
    const float rxy2 = __fmaf_rn(rx, rx, __fmul_rn(ry, ry));
    const float rho = sqrtf(__fmaf_rn(rz, rz, rxy2));
    const float rxy = sqrtf(rxy2);
    float cp = 1.0f, sp = 0.0f;
    if (rxy > 0.0f) { cp = rx / rxy; sp = ry / rxy; }
    const float ct = rz / rho, st = rxy / rho;
    const float irho = 1.0f / rho;
    return PairGeo{sp, cp, ct, st, sa * irho, sb * irho, irho};
}

// The sums over the lanes, acc[NV][32] -> out[NR] (locals keep the unpadded
// stride). A lane takes the values j = lane, lane + 32, .. and adds the 32 lanes'
// parts in the order of a butterfly, a binary tree over the bits of the lane's
// number; the tree is the same from any lane, so each starts at another one and
// the reads meet no bank conflicts. 260 instructions for 121 values, against 1,450
// with a butterfly of shuffles per value: M2L at 1M bodies 6.84 -> 6.49 ms, 64 clusters at
// P = 12 (six batches per target) 7.69 -> 7.12 ms.
template <int P>
__device__ __forceinline__ void store_local(const float4* acc, float* __restrict__ out) {
    constexpr int NR = (P + 1) * (P + 1);
    const int lane = threadIdx.x & 31;
    const float* a = reinterpret_cast<const float*>(acc);
#pragma unroll 1
    for (int j = lane; j < NR; j += 32) {
        const int at = (j >> 2) * 128 + (j & 3), c = (j >> 2) & 7;
        float v[16];
#pragma unroll
        for (int l = 0; l < 16; ++l) v[l] = __fadd_rn(a[at + 4 * (l ^ c)], a[at + 4 * ((l + 16) ^ c)]);
#pragma unroll
        for (int h = 8; h > 0; h >>= 1)
#pragma unroll
            for (int l = 0; l < h; ++l) v[l] = __fadd_rn(v[l], v[l + h]);
        out[j] = v[0];
    }
}

// ------------------------------------------------------------------------
// FP32, compile-time order P: coefficients live in registers. For the orders to 8.

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

template <int P>
__global__ void __launch_bounds__(128, 2) k_m2l32(const int* __restrict__ dnn, const uint32_t* __restrict__ src,
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
    int next_b = 0;  // (lane 0: asked for at a target's end, not earlier: a target held back is one more at the very end)
    if (lane == 0) next_b = (int)atomicAdd(queue, 1u);
    const int nnodes = *dnn;
    for (;;) {
        const int b = __shfl_sync(0xffffffffu, next_b, 0);
        if (b >= nnodes) break;
#pragma unroll
        for (int j = 0; j < NV; ++j) acc[j * 32 + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
        const uint32_t q0 = off[b], q1 = off[b + 1];
        const float4 bh = zhi[b], bl = zlo[b];
        for (uint32_t q = q0 + lane; q < q1; q += 32) {
            const int a = (int)src[q];
            const float4 ah = zhi[a], al = zlo[a];
            float c[NV * 4];
            const float4* mv = reinterpret_cast<const float4*>(mult + (size_t)stride * a);
#pragma unroll
            for (int j = 0; j < NV; ++j) {
                const float4 v = __ldg(mv + j);
                c[4 * j] = v.x; c[4 * j + 1] = v.y; c[4 * j + 2] = v.z; c[4 * j + 3] = v.w;
            }
            // Rz(pi/2 - phi) S Rz(-theta) S Z S Rz(theta) S Rz(phi - pi/2)
            const PairGeo g = pair_geo(ah, al, bh, bl);
            rotz32<P>(c, g.sp, g.cp);
            swap_lit<P>(c);
            rotz32<P>(c, g.ct, -g.st);
            swap_lit<P>(c);
            ztrans_lit<P>(c, g.u, g.v, g.irho);
            swap_lit_z<P>(c);
            rotz32<P>(c, g.ct, g.st);
            swap_lit<P>(c);
            rotz32<P>(c, g.sp, -g.cp);
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
        if (lane == 0) next_b = (int)atomicAdd(queue, 1u);
        store_local<P>(acc, loc + (size_t)NR * b);
        __syncwarp();
    }
}


// ------------------------------------------------------------------------
// FP32 by degrees, for the larger orders. The straight-line steps above are some
// 10,000 instructions at order 12, and warps at different places in them wait for
// instruction fetch. But rotations and swaps act on every degree by itself, and
// the way back from the z axis does to a degree what the way there did, with the
// powers of the two angles exchanged. So both ways are one loop body, taken degree
// by degree: rotation, swap and rotation of a degree's 2n + 1 values in registers,
// and only the orders that the z-translation couples (m <= min(n, P - n): 61 of the
// 121 values at P = 10, 85 of 169 at 12) are kept between the two. Half the code, no
// spills, and the source's values are loaded a degree ahead of their use.
// M2L kernel, straight-line -> by degrees, ms: P = 12, 2.3M bodies of 64 clusters
// 12.5 -> 7.7, 8M bodies 75 -> 47; P = 10, 1M bodies 7.5 -> 6.8, 64k .61 -> .58;
// P = 14, 500k 6.9 -> 4.4. Bound by issue (60 % of the slots at P = 10, 52 % at 12) with
// eight warps per SM, which is what registers and the sums' shared memory hold; three
// blocks (168 registers) leave the L1 too small for the sources' rows: 8.8 ms at 1M.
#include "m2l_steps.inc"

__host__ __device__ constexpr int low_order(int P, int n) { return n < P - n ? n : P - n; }
__host__ __device__ constexpr int mid_off(int P, int n) {
    int s = 0;
    for (int i = 0; i < n; ++i) s += 2 * low_order(P, i) + 1;
    return s;
}

// order m >= 1 of a degree times pr + i pi
__device__ __forceinline__ void rot_order(float& re, float& im, float pr, float pi) {
    const float a = __fmul_rn(im, pi), b = __fmul_rn(im, pr), r = re;
    re = __fmaf_rn(r, pr, -a);
    im = __fmaf_rn(r, pi, b);
}

// powers (c + i s)^m, m = 1..P; NEG: of c - i s
template <int P, bool NEG>
__device__ __forceinline__ void rot_powers(float c, float s, float* pr, float* pi) {
    pr[1] = c;
    pi[1] = NEG ? -s : s;
#pragma unroll
    for (int m = 2; m <= P; ++m) {
        // (which product of a sum is the rounded one follows the plain kernel)
        pr[m] = NEG ? __fmaf_rn(pr[m - 1], c, __fmul_rn(pi[m - 1], s))
                    : __fmaf_rn(pr[m - 1], c, -__fmul_rn(pi[m - 1], s));
        pi[m] = NEG ? __fmaf_rn(pi[m - 1], c, -__fmul_rn(pr[m - 1], s))
                    : __fmaf_rn(pr[m - 1], s, __fmul_rn(pi[m - 1], c));
    }
}

constexpr float kSqrt2 = 0x1.6a09e6p+0f;  // the swap's entry from order 1 to order 0 of degree 1

__device__ __forceinline__ void row_load(const float4* row, int k, float* c) {
    const float4 v = __ldg(row + k);
    c[0] = v.x; c[1] = v.y; c[2] = v.z; c[3] = v.w;
}

constexpr int kTogether = 5;  // from this degree on, all that are left are loaded together
constexpr int kNextAt = 3;    // in the second pass the next source's loads start here

// What a lane holds of its source: the row, the centre and scale.
struct SourceAt {
    const float4* row;
    float4 hi, lo;
};

// Degrees N, N - 1, .. 0 of one pass. Both passes turn, swap and turn a degree
// (powers A, then B) in the same instructions; the first takes the source's
// values and swaps into the middle vector, the second takes the middle vector
// through a swap and adds to the sums. val: the degrees' values as loaded, later
// the results, four to a load and to an update of the sums. Loads are issued a
// degree ahead, those of the last degrees together, and the next source's first
// ones before the last degrees of the second pass. (The pass that does not load
// clears the values, or the compiler would carry the old ones through it.)
template <int P, int N>
__device__ __forceinline__ void degrees(bool first, SourceAt& s, float* val, const float* ar, const float* ai,
                                        const float* br, const float* bi, float* mid, float4* acc, float irho,
                                        int next, const float* mult, int stride, const float4* zhi,
                                        const float4* zlo) {
    constexpr int NR = (P + 1) * (P + 1), NV = (NR + 3) / 4;
    constexpr int lo = (N * N + 3) / 4, hi = N == P ? NV : ((N + 1) * (N + 1) + 3) / 4;  // sums complete with degree N
    constexpr int M = N > kTogether ? N - 1 : 0;                      // degrees M .. N - 1 are loaded here
    constexpr int llo = M * M / 4, lhi = N < kTogether ? 0 : N * N / 4;
    float x[2 * N + 1];
    if (first) {
#pragma unroll
        for (int k = lhi - 1; k >= llo; --k) row_load(s.row, k, val + 4 * k);
        if constexpr (N == kNextAt) {
            s.hi = s.lo = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = P * P / 4 * 4; i < 4 * NV; ++i) val[i] = 0.0f;
        }
#pragma unroll
        for (int i = 0; i < 2 * N + 1; ++i) x[i] = val[N * N + i];
    } else {
#pragma unroll
        for (int i = 4 * llo; i < 4 * lhi; ++i) val[i] = 0.0f;
        if constexpr (N == kNextAt) {
            s.row = reinterpret_cast<const float4*>(mult + (size_t)stride * next);
            s.hi = zhi[next];
            s.lo = zlo[next];
#pragma unroll
            for (int k = NV - 1; k >= P * P / 4; --k) row_load(s.row, k, val + 4 * k);
        }
        if constexpr (N > 0) SwapDeg<N, low_order(P, N), N>::run(mid + mid_off(P, N), x);
    }
    if constexpr (N > 0) {
        float y[2 * N + 1];
#pragma unroll
        for (int m = 1; m <= N; ++m) rot_order(x[2 * m - 1], x[2 * m], ar[m], ai[m]);
        SwapDeg<N, N, N>::run(x, y);
#pragma unroll
        for (int m = 1; m <= N; ++m) rot_order(y[2 * m - 1], y[2 * m], br[m], bi[m]);
        if (first) {
            SwapDeg<N, N, low_order(P, N)>::run(y, mid + mid_off(P, N));
        } else {
            // (order 0 of degree 1 is a single product, which the sum takes unrounded)
            val[N * N] = N == 1 ? x[1] : y[0];
#pragma unroll
            for (int i = 1; i < 2 * N + 1; ++i) val[N * N + i] = y[i];
        }
    } else if (first) {
        mid[0] = x[0];
    }
    if (!first) {
#pragma unroll
        for (int k = hi - 1; k >= lo; --k) {
            float4 v = acc[k * 32];
            if (k == 0) {
                v.x = __fmaf_rn(irho, mid[0], v.x);
                v.y = __fmaf_rn(kSqrt2, val[1], v.y);
            } else {
                v.x = __fadd_rn(v.x, val[4 * k]);
                if (4 * k + 1 < NR) v.y = __fadd_rn(v.y, val[4 * k + 1]);
            }
            if (4 * k + 2 < NR) v.z = __fadd_rn(v.z, val[4 * k + 2]);
            if (4 * k + 3 < NR) v.w = __fadd_rn(v.w, val[4 * k + 3]);
            acc[k * 32] = v;
        }
    }
    if constexpr (N > 0)
        degrees<P, N - 1>(first, s, val, ar, ai, br, bi, mid, acc, irho, next, mult, stride, zhi, zlo);
}

// Warps per block and blocks per SM: eight warps, the registers' limit, where the
// sums of eight fit in shared memory. At P = 14 they are 29 KB per warp, so blocks of
// one, seven to an SM (500k bodies: 4.9 ms with one block of four, 4.0 with three of
// two, 3.7 so).
__host__ __device__ constexpr int degree_warps(int P) { return P > 12 ? 1 : 4; }
__host__ __device__ constexpr int degree_blocks(int P) { return P > 12 ? 7 : 2; }

template <int P>
__global__ void __launch_bounds__(32 * degree_warps(P), degree_blocks(P)) k_m2l32_deg(const int* __restrict__ dnn, const uint32_t* __restrict__ src,
                                                      const uint32_t* __restrict__ off, const float* __restrict__ mult,
                                                      int stride, const float4* __restrict__ zhi,
                                                      const float4* __restrict__ zlo, float* __restrict__ loc,
                                                      unsigned* __restrict__ queue) {
    constexpr int NR = (P + 1) * (P + 1);
    constexpr int NV = (NR + 3) / 4;
    static_assert(P > kTogether && P % 2 == 0, "loads by degrees; signs of the z-translation");
    extern __shared__ float4 sh_acc4[];  // [warp][NV][32]
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    float4* acc = sh_acc4 + (size_t)wib * NV * 32 + lane;
    int next_b = 0;  // (lane 0: asked for at a target's end, not earlier: a target held back is one more at the very end)
    if (lane == 0) next_b = (int)atomicAdd(queue, 1u);
    const int nnodes = *dnn;
    for (;;) {
        const int b = __shfl_sync(0xffffffffu, next_b, 0);
        if (b >= nnodes) break;
#pragma unroll 4
        for (int j = 0; j < NV; ++j) acc[j * 32] = make_float4(0.f, 0.f, 0.f, 0.f);
        const uint32_t q0 = off[b], q1 = off[b + 1];
        const float4 bh = zhi[b], bl = zlo[b];
        uint32_t q = q0 + lane;
        if (q < q1) {
            int a = (int)src[q];
            SourceAt s{reinterpret_cast<const float4*>(mult + (size_t)stride * a), zhi[a], zlo[a]};
            float val[4 * NV];
#pragma unroll
            for (int k = NV - 1; k >= P * P / 4; --k) row_load(s.row, k, val + 4 * k);
            for (;;) {
                q += 32;
                const bool more = q < q1;
                if (more) a = (int)src[q];  // (else the last source again, not used)
                const PairGeo g = pair_geo(s.hi, s.lo, bh, bl);
                float cA = g.sp, sA = g.cp;  // Rz(pi/2 - phi), then Rz(theta)
                float cB = g.ct, sB = g.st;  // Rz(-theta), then Rz(phi - pi/2)
                float mid[mid_off(P, P + 1)];
#pragma unroll 1
                for (int pass = 0; pass < 2; ++pass) {
                    float ar[P + 1], ai[P + 1], br[P + 1], bi[P + 1];
                    rot_powers<P, false>(cA, sA, ar, ai);
                    rot_powers<P, true>(cB, sB, br, bi);
                    degrees<P, P>(pass == 0, s, val, ar, ai, br, bi, mid, acc, g.irho, a, mult, stride, zhi, zlo);
                    if (pass == 0) ZTrans<P>::run(mid, g.u, g.v, g.irho);
                    float t = cA; cA = cB; cB = t;
                    t = sA; sA = sB; sB = t;
                }
                if (!more) break;
            }
        }
        __syncwarp();
        if (lane == 0) next_b = (int)atomicAdd(queue, 1u);
        store_local<P>(acc - lane, loc + (size_t)NR * b);
        __syncwarp();
    }
}

template <int P>
void launch_m2l32(const int* dnn, const uint32_t* src, const uint32_t* off, const float* mult,
                  int stride, const float4* zhi, const float4* zlo, float* loc, unsigned* queue,
                  cudaStream_t st) {
    // By degrees from order 10 on. Below, the straight-line code is short enough: ms
    // straight-line and by degrees, order 8, 500k bodies 2.07 and 2.49; order 6, 30k .32 and .40.
    constexpr auto kernel = [] {
        if constexpr (P >= 10) return k_m2l32_deg<P>;
        else return k_m2l32<P>;
    }();
    constexpr int warps = P >= 10 ? degree_warps(P) : 4, blocks = P >= 10 ? degree_blocks(P) : 2;
    const size_t sh = (size_t)warps * (((P + 1) * (P + 1) + 3) / 4) * 32 * sizeof(float4);
    ensure_dyn_smem((const void*)kernel, (int)sh);
    (kernel<<<device_sm_count() * blocks, 32 * warps, sh, st>>>(dnn, src, off, mult, stride, zhi, zlo, loc, queue), note_launch());
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
