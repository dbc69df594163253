// Leaf evaluation: far field by L2P, near field by P2P (Sec. 2.1), plus the
// plain FP64 direct sum used to measure force errors (Sec. 3.1.1).
//
// P2P runs over work items: a target leaf and at most kLeavesPerItem of the
// source leaves in its (sorted) P2P list, taken by warps from a counter.
// The kernel (k_p2p_tiles) stages the item's source bodies in shared
// memory, by bulk copies or plain loads, puts the sources across the lanes
// and keeps a group of target bodies in every lane's registers, so one
// shared-memory load serves several interactions and every lane is busy
// whatever the leaf sizes; a fixed transpose reduction then sums the lanes.
// Each item writes one partial per target body. k_leaf_reduce then evaluates the leaf's local
// expansion at the body (L2P), adds the body's partials in item order, and
// writes the result to the caller's order through the sort permutation.
// Every sum runs in a fixed order.
//
// Mixed precision: bodies are stored relative to their own leaf centre in
// FP32; a source leaf A is moved into the target leaf B's frame by the
// FP32-rounded offset z_A - z_B (computed from double-float centres). Terms
// are FP32 (rsqrtf); each staged pack's sum is accumulated in FP64.
#include "f32x2.cuh"
#include "fp64_math.cuh"
#include "gbfmm_internal.cuh"

namespace gbfmm {

namespace {

__constant__ float c_w32l[kMaxPF32 + 2][kMaxPF32 + 2];
__constant__ float c_iw32l[kMaxPF32 + 2][kMaxPF32 + 2];
__constant__ float c_rec_a32l[kMaxPF32 + 1][kMaxPF32 + 1];
__constant__ float c_rec_b32l[kMaxPF32 + 1][kMaxPF32 + 1];
__constant__ float c_diag32l[kMaxPF32 + 1];
__constant__ float c_sub32l[kMaxPF32 + 1];

struct TabL64 {
    const double *w, *iw, *rec_a, *rec_b, *diag, *sub;
    __device__ double W(int n, int m) const { return __ldg(w + n * (kMaxP + 2) + m); }
    __device__ double IW(int n, int m) const { return __ldg(iw + n * (kMaxP + 2) + m); }
    __device__ double A(int n, int m) const { return __ldg(rec_a + n * (kMaxP + 1) + m); }
    __device__ double B(int n, int m) const { return __ldg(rec_b + n * (kMaxP + 1) + m); }
    __device__ double D(int m) const { return __ldg(diag + m); }
    __device__ double Sb(int m) const { return __ldg(sub + m); }
};
struct TabL32 {
    __device__ float W(int n, int m) const { return c_w32l[n][m]; }
    __device__ float IW(int n, int m) const { return c_iw32l[n][m]; }
    __device__ float A(int n, int m) const { return c_rec_a32l[n][m]; }
    __device__ float B(int n, int m) const { return c_rec_b32l[n][m]; }
    __device__ float D(int m) const { return c_diag32l[m]; }
    __device__ float Sb(int m) const { return c_sub32l[m]; }
};

// L2P on a hat local expansion F at dhat = d / s (|dhat| <= 1):
//   phi = -sum_{n,m} conj(Shat_n^m(dhat)) Fhat_n^m
//   F_1^m(x) = (1/s) sum_{k,l} conj(Shat_k^l) w_{1+k}^{m+l}/w_k^l Fhat_{1+k}^{m+l}, m = 0, 1
//   a = (Re F_1^1, Im F_1^1, F_1^0)        (all without G)
// PC > 0: the order is the compile-time PC (loops unrolled); PC = 0: p.
template <typename T, typename Tab, int PC = 0>
__device__ __forceinline__ void l2p_hat(int p_rt, const T* __restrict__ F, T x, T y, T z, T inv_s, const Tab& tb,
                                        T& phi, T& ax, T& ay, T& az) {
    const int p = PC > 0 ? PC : p_rt;
    const T r2 = x * x + y * y + z * z;
    T pot = T(0), g0 = T(0), g1r = T(0), g1i = T(0);
    T dre = T(1), dim = T(0);  // Shat_l^l
#pragma unroll
    for (int l = 0; l <= p; ++l) {
        if (l > 0) {
            const T t = dre * x - dim * y;
            dim = dre * y + dim * x;
            dre = t;
            dre *= tb.D(l);
            dim *= tb.D(l);
        }
        T s1r = dre, s1i = dim, s2r = T(0), s2i = T(0);  // Shat_k^l, Shat_{k-1}^l
#pragma unroll
        for (int k = l; k <= p; ++k) {
            T sr, si;
            if (k == l) { sr = dre; si = dim; }
            else if (k == l + 1) { sr = tb.Sb(l) * z * s1r; si = tb.Sb(l) * z * s1i; }
            else {
                const T a = tb.A(k, l) * z, b = tb.B(k, l) * r2;
                sr = a * s1r - b * s2r;
                si = a * s1i - b * s2i;
            }
            if (k > l) { s2r = s1r; s2i = s1i; s1r = sr; s1i = si; }
            // potential: Re(conj(S) F) counted twice for l > 0
            const T fr = F[hre(k, l)], fi = l ? F[him(k, l)] : T(0);
            const T re = sr * fr + si * fi;
            pot += l ? T(2) * re : re;
            if (k < p) {
                const T iwkl = tb.IW(k, l);
                // F_1^0
                const T g0r = F[hre(k + 1, l)], g0i = l ? F[him(k + 1, l)] : T(0);
                const T c0 = tb.W(k + 1, l) * iwkl;
                const T re0 = sr * g0r + si * g0i;
                g0 += l ? T(2) * c0 * re0 : c0 * re0;
                // F_1^1, +l part: conj(S_k^l) alpha Fhat_{1+k}^{1+l}
                const T al = tb.W(k + 1, l + 1) * iwkl;
                const T hr = F[hre(k + 1, l + 1)], hi = F[him(k + 1, l + 1)];
                g1r += al * (sr * hr + si * hi);
                g1i += al * (sr * hi - si * hr);
                // -l part (l >= 1): -S_k^l gamma conj(Fhat_{1+k}^{l-1})
                if (l >= 1) {
                    const T ga = tb.W(k + 1, l - 1) * iwkl;
                    const T er = F[hre(k + 1, l - 1)], ei = (l - 1) ? F[him(k + 1, l - 1)] : T(0);
                    g1r -= ga * (sr * er + si * ei);
                    g1i -= ga * (si * er - sr * ei);
                }
            }
        }
    }
    phi = -pot;
    ax = g1r * inv_s;
    ay = g1i * inv_s;
    az = g0 * inv_s;
}

// ---------------------------------------------------------------------------
// P2P over work items. Item (B, j, s) covers the sources q in
// [off[B] + j*kLeavesPerItem, ...) of target leaf B (at most kLeavesPerItem
// source leaves) and slice s of its targets, so no warp carries more than a bounded share of a dense
// leaf's work. Warps fetch items dynamically. Each item writes one partial
// sum per target body; k_leaf_reduce adds the partials of a body in item
// order (deterministic) together with the L2P far field.

// Item r of target leaf B (nB bodies, sources off0 .. off1 - 1 of the list):
// kLeavesPerItem source leaves (part) and a.tslice targets (t0 .. t1 - 1) of it.
struct LeafItem {
    uint32_t part, q0, q1;
    int t0, t1;
};
__device__ __forceinline__ LeafItem leaf_item(const LeafArgs& a, uint32_t r, uint32_t off0, uint32_t off1, int nB) {
    LeafItem it;
    const uint32_t nsl = (uint32_t)leaf_slices(nB, a.tslice);
    it.part = r / nsl;
    const int s = (int)(r - it.part * nsl);
    it.q0 = off0 + it.part * kLeavesPerItem;
    it.q1 = it.q0 + kLeavesPerItem < off1 ? it.q0 + kLeavesPerItem : off1;
    it.t0 = s * a.tslice;
    it.t1 = it.t0 + a.tslice < nB ? it.t0 + a.tslice : nB;
    return it;
}

// Knuth's two-sum: (hi, lo) += b with the rounding error kept in lo.
__device__ __forceinline__ void two_sum(float& hi, float& lo, float b) {
    const float s = hi + b;
    const float bb = s - hi;
    const float err = (hi - (s - bb)) + (b - bb);
    hi = s;
    lo += err;
}

// a body (position, mass) as one 16-byte (FP32) or 32-byte (FP64) aligned record,
// so that shared-memory reads and writes take one vector access
template <typename T>
struct alignas(4 * sizeof(T)) Body4 { T x, y, z, w; };

constexpr int kStageCap = 256;  // bodies staged per pack (source leaves packed back to back)

// Accumulators of one target: FP32 runs of at most kRun terms are folded
// into (hi, lo) two-sum pairs (FP64 sums in FP64 mode), so the FP32 rounding
// of near-field terms that cancel stays at the level of a short run.
constexpr int kRun = 16;

template <typename T>
struct NearAcc {
    float hx = 0.f, hy = 0.f, hz = 0.f, hp = 0.f, lx = 0.f, ly = 0.f, lz = 0.f, lp = 0.f;
    double dx = 0.0, dy = 0.0, dz = 0.0, dp = 0.0;
    __device__ __forceinline__ void add(T px, T py, T pz, T pp) {
        if (sizeof(T) == 4) {
            two_sum(hx, lx, (float)px);
            two_sum(hy, ly, (float)py);
            two_sum(hz, lz, (float)pz);
            two_sum(hp, lp, (float)pp);
        } else {
            dx += (double)px; dy += (double)py; dz += (double)pz; dp += (double)pp;
        }
    }
};

// ---------------------------------------------------------------------------
// P2P force over work items, sources across lanes and targets in registers.
//
// A warp stages the item's source bodies (moved into the target leaf B's
// frame) in shared memory, up to TileCfg::kCap at a time. The targets of the
// item are taken in groups of TG = 8 (a last group of 4 when at most 4
// remain). For a group, lane l runs over the staged sources
// l, l + 32, l + 64, ... and keeps TG four-component partial sums (ax, ay,
// az, sum m/r) in registers: one shared-memory load serves TG interactions
// and every lane is busy whatever the leaf sizes. The 32 lanes' partials of
// the group are then summed by a transpose reduction across the warp (a
// fixed tree: lane l ends with component l % 4 of target l / 4), and added
// in FP64 to the group's totals in shared memory. So the order of every sum
// is fixed and the result does not depend on scheduling.
//
// FP32 terms are summed per lane over at most kCap / 32 = 16 sources of a
// staged pack, the cross-lane tree adds five levels, and each pack's total is
// accumulated in FP64.
//
// SOFT: Plummer softening (Appendix B), 1/r -> 1/sqrt(r^2 + s2); the body
// itself (r2 = 0; coincident bodies are rejected) still contributes nothing.

template <typename T>
struct TileCfg;
#ifndef GBFMM_P2P_CAP32
#define GBFMM_P2P_CAP32 512
#endif
// blocks per SM the tile kernel's registers are cut for: 4 (128 registers, no
// spill) measured 5.74 ms against 5.82 ms for 5 (96 registers, a small spill)
#ifndef GBFMM_P2P_MINB
#define GBFMM_P2P_MINB 4
#endif
#ifndef GBFMM_P2P_TG
#define GBFMM_P2P_TG 8
#endif
template <>
struct TileCfg<float> {
    static constexpr int TG = GBFMM_P2P_TG;  // targets per group
    static constexpr int kCap = GBFMM_P2P_CAP32;  // staged source bodies per warp (512: 8 KB, at most 16 per lane)
};
template <>
struct TileCfg<double> {
    static constexpr int TG = 8;
    // 8 KB per warp. Groups of 4 targets with two Newton steps for 1/r took 49.6 ms for the 0.83 G pairs
    // of N = 100000, groups of 8 with inv_powers (19 FP64 instructions a pair, half the reductions)
    // and slices of 8 targets 32.8 ms
    static constexpr int kCap = 256;
};
constexpr int kTargetChunk = 64;  // targets whose totals a warp keeps in shared memory per pass

// per warp: staged sources, the target chunk's positions, its FP64 totals, an mbarrier
template <typename T>
constexpr size_t p2p_tile_smem_per_warp() {
    return sizeof(Body4<T>) * TileCfg<T>::kCap + sizeof(Body4<T>) * kTargetChunk + sizeof(double) * 4 * kTargetChunk +
           4 * sizeof(Body4<T>);
}

// Bulk-copy staging (BULK, FP32; the default, FMM_FLAG_P2P_LOADS turns it off):
// the bodies of every staged
// source leaf come into shared memory by one cp.async.bulk (the tensor memory
// accelerator's 1-D copy, 16-byte aligned, a multiple of 16 bytes) that
// completes on the warp's mbarrier; the leaf-centre offsets are then added in
// shared memory. Waits are bounded: after kBulkWaitNs the warp raises
// kErrTimeout and leaves the kernel (every issued copy has completed by then
// unless the copy engine itself stalled).
constexpr unsigned long long kBulkWaitNs = 1000000000ull;  // one second

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_to_smem(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t phase) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(phase)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// generic-proxy accesses of shared memory before this are ordered before later bulk copies into it
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// wait (all lanes) for the phase of the warp's mbarrier; false: the wait ran out
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t phase) {
    const unsigned long long t0 = global_ns();
    bool done = mbar_test(bar, phase);
    while (!done) {
        if (global_ns() - t0 > kBulkWaitNs) break;
        done = mbar_test(bar, phase);
    }
    return __all_sync(0xffffffffu, done) != 0;
}

// Stage whole source leaves src[q], src[q+1], ... (below q1) of target leaf
// B into sm, moved into B's frame, as many as fit in kCap bodies; returns the
// body count, advances q and sets selfin if B itself is among them. The lanes
// read 32 leaves' ranges and centres at once and copy their bodies with
// independent loads, so the latency of the index, range and body loads is paid
// once per 32 leaves rather than once per leaf. A leaf larger than kCap (a
// level-21 leaf can exceed the leaf size) goes in pieces of kCap bodies, soff
// being the next body of it.
template <typename T, int kCap, bool BULK>
__device__ __forceinline__ int stage_leaves(const LeafArgs& a, int B, float4 bh, float4 bl, uint32_t& q,
                                            uint32_t q1, int& soff, Body4<T>* __restrict__ sm, bool& selfin,
                                            int lane, uint64_t* bar, uint32_t& phase, bool& timed_out) {
    int cnt = 0;
    selfin = false;
    {
        // the next leaf does not fit in an empty stage, or a piece of it is already staged
        const int A = (int)a.p2p_src[q];
        const int a0 = a.t.begin[A], nA = a.t.end[A] - a0;
        if (soff > 0 || nA > kCap) {
            const int take = nA - soff < kCap ? nA - soff : kCap;
            float ox = 0.f, oy = 0.f, oz = 0.f;
            if (sizeof(T) == 4) {
                const float4 ah = a.zhi[A], al = a.zlo[A];
                ox = (ah.x - bh.x) + (al.x - bl.x);
                oy = (ah.y - bh.y) + (al.y - bl.y);
                oz = (ah.z - bh.z) + (al.z - bl.z);
            }
            for (int l = lane; l < take; l += 32) {
                const int jj = a0 + soff + l;
                Body4<T> v;
                if (sizeof(T) == 4) {
                    const float4 u = a.prel[jj];
                    v = {(T)(u.x + ox), (T)(u.y + oy), (T)(u.z + oz), (T)u.w};
                } else {
                    v = {(T)a.xs[jj], (T)a.ys[jj], (T)a.zs[jj], (T)a.ms[jj]};
                }
                sm[l] = v;
            }
            selfin = A == B;
            soff += take;
            if (soff >= nA) {
                soff = 0;
                ++q;
            }
            return take;
        }
    }
    while (q < q1) {
        const int nl = q1 - q < 32u ? (int)(q1 - q) : 32;
        int A = -1, a0 = 0, nA = 0;
        float ox = 0.f, oy = 0.f, oz = 0.f;
        if (lane < nl) {
            A = (int)a.p2p_src[q + lane];
            a0 = a.t.begin[A];
            nA = a.t.end[A] - a0;
            if (sizeof(T) == 4) {
                const float4 ah = a.zhi[A], al = a.zlo[A];
                ox = (ah.x - bh.x) + (al.x - bl.x);
                oy = (ah.y - bh.y) + (al.y - bl.y);
                oz = (ah.z - bh.z) + (al.z - bl.z);
            }
        }
        int incl = nA;  // inclusive prefix sum of the leaf sizes
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const unsigned fits = __ballot_sync(0xffffffffu, lane < nl && cnt + incl <= kCap);
        // (an empty stage always takes the first leaf: one larger than kCap went the piecewise way above,
        // and this loop stops before such a leaf once anything is staged)
        const int fit = __popc(fits);  // a prefix of the leaves, since incl grows
        selfin |= __any_sync(0xffffffffu, lane < fit && A == B) != 0;
        if (BULK && sizeof(T) == 4 && fit > 0) {
            // one bulk copy per leaf (lane j for leaf j), then the offsets in shared memory
            const uint32_t bytes = (uint32_t)__shfl_sync(0xffffffffu, incl, fit - 1) * (uint32_t)sizeof(Body4<T>);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive_expect(bar, bytes + a.tx_extra);
            __syncwarp();
            if (lane < fit)
                bulk_to_smem(sm + cnt + incl - nA, a.prel + a0, (uint32_t)nA * (uint32_t)sizeof(Body4<T>), bar);
            const bool ok = mbar_wait_bounded(bar, phase);
            phase ^= 1u;
            if (!ok) {
                timed_out = true;
                return cnt;
            }
#pragma unroll 4
            for (int j = 0; j < fit; ++j) {
                const int nj = __shfl_sync(0xffffffffu, nA, j);
                const int dst = cnt + __shfl_sync(0xffffffffu, incl, j) - nj;
                const float oxj = __shfl_sync(0xffffffffu, ox, j), oyj = __shfl_sync(0xffffffffu, oy, j),
                            ozj = __shfl_sync(0xffffffffu, oz, j);
                for (int l = lane; l < nj; l += 32) {
                    Body4<T>& v = sm[dst + l];
                    v.x = (T)(v.x + oxj);
                    v.y = (T)(v.y + oyj);
                    v.z = (T)(v.z + ozj);
                }
            }
            cnt += __shfl_sync(0xffffffffu, incl, fit - 1);
            q += (uint32_t)fit;
            if (fit < nl) break;
            continue;
        }
#pragma unroll 4
        for (int j = 0; j < fit; ++j) {
            const int aj = __shfl_sync(0xffffffffu, a0, j), nj = __shfl_sync(0xffffffffu, nA, j);
            const int dst = cnt + __shfl_sync(0xffffffffu, incl, j) - nj;
            const float oxj = __shfl_sync(0xffffffffu, ox, j), oyj = __shfl_sync(0xffffffffu, oy, j),
                        ozj = __shfl_sync(0xffffffffu, oz, j);
            for (int l = lane; l < nj; l += 32) {
                Body4<T> v;
                if (sizeof(T) == 4) {
                    const float4 u = a.prel[aj + l];
                    v = {(T)(u.x + oxj), (T)(u.y + oyj), (T)(u.z + ozj), (T)u.w};
                } else {
                    v = {(T)a.xs[aj + l], (T)a.ys[aj + l], (T)a.zs[aj + l], (T)a.ms[aj + l]};
                }
                sm[dst + l] = v;
            }
        }
        if (fit > 0) cnt += __shfl_sync(0xffffffffu, incl, fit - 1);
        q += (uint32_t)fit;
        if (fit < nl) break;  // the stage is full
    }
    return cnt;
}

// Halving step of the transpose reduction: C values per lane become C/2;
// a lane with bit o set keeps the upper half and receives its partner's.
template <int C, typename T>
__device__ __forceinline__ void halve(T* v, int lane, int o) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < C / 2; ++i) {
        const T send = up ? v[i] : v[i + C / 2];
        const T keep = up ? v[i + C / 2] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
}

// The same step for a lane whose halves are already swapped when bit o is
// set (slot s of such a lane holds value s ^ (C/2)): every lane keeps the
// lower slots and sends the upper ones, with no selects.
template <int C, typename T>
__device__ __forceinline__ void halve_swapped(T* v, int o) {
#pragma unroll
    for (int i = 0; i < C / 2; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i + C / 2], o);
}

// v[0..V-1] on every lane (V = 32, 16 or 8), value j = 4 t + c (target t,
// component c), with lane l holding target t ^ ((l >> 2) & (V/4 - 1)) in
// slot t (the target order p2p_group gives each lane). On return v[0] of
// lane l holds the sum over the 32 lanes of value l % V. The steps over the
// target bits (lane bits 4..2) need no selects; the two over the components
// (lane bits 1, 0) do.
template <int V, typename T>
__device__ __forceinline__ T transpose_reduce(T* v, int lane) {
    static_assert(V == 32 || V == 16 || V == 8, "V");
    if constexpr (V <= 16) {
#pragma unroll
        for (int i = 0; i < V; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], 16);
    }
    if constexpr (V == 8) {
#pragma unroll
        for (int i = 0; i < V; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], 8);
    }
    if constexpr (V == 32) halve_swapped<32>(v, 16);
    if constexpr (V >= 16) halve_swapped<16>(v, 8);
    halve_swapped<8>(v, 4);
    halve<4>(v, lane, 2);
    halve<2>(v, lane, 1);
    return v[0];
}

// One group of NT targets (b0 + t0 .. b0 + t0 + NT - 1, clamped to the last
// target; clamped duplicates are computed and discarded) against the cnt
// staged sources; adds the group's totals to tot[4 * (t0 + t) + c]. Lane l
// keeps target t ^ g, g = (l >> 2) & (NT - 1), in its slot t: the order the
// select-free steps of transpose_reduce expect. A lane's FP32 sums run over
// at most kCap / 32 terms.
template <typename T, int NT, bool GUARD, bool SOFT>
__device__ __forceinline__ void p2p_group(const Body4<T>* __restrict__ sm, int cnt, const Body4<T>* __restrict__ tg,
                                          int t0, int nt, T s2, double* tot, int lane, float one) {
    const int g = (lane >> 2) & (NT - 1);
    T run[NT * 4];
    // the stage is padded to a multiple of 32 with massless far bodies (pad_stage)
    const int per_lane = (cnt + 31) >> 5;
    if constexpr (sizeof(T) == 4) {
        // two targets to a packed operation: 13 operations of the FMA pipe a pair as before, at half the issue
        // slots, which were the bound (74% of cycles). 2^20 bodies, 5.8 G pairs: 4.24 -> 3.59 ms, FMA pipe 54 ->
        // 62%; without the moves of the sources into the target frame it would take 3.3 ms
        f32x2 nx[NT / 2], ny[NT / 2], nz[NT / 2], acc[NT * 2];  // negated targets; per pair x, y, z, sum m/r
#pragma unroll
        for (int t = 0; t < NT; t += 2) {
            const int i = t0 + (t ^ g), j = t0 + ((t + 1) ^ g);
            const Body4<T> u = tg[i < nt ? i : nt - 1], v = tg[j < nt ? j : nt - 1];
            nx[t / 2] = f2_pack(-u.x, -v.x);
            ny[t / 2] = f2_pack(-u.y, -v.y);
            nz[t / 2] = f2_pack(-u.z, -v.z);
        }
#pragma unroll
        for (int e = 0; e < NT * 2; ++e) acc[e] = 0ull;
        const f32x2 one2 = f2_pack(one, one), s22 = f2_pack(s2, s2);
        Body4<T> nxt = sm[lane];  // one source ahead (the last step's reads the targets behind the stage, unused)
        for (int u = 0; u < per_lane; ++u) {
            const Body4<T> s = nxt;
            nxt = sm[lane + 32 * (u + 1)];
            const f32x2 sx = f2_pack(s.x, s.x), sy = f2_pack(s.y, s.y), sz = f2_pack(s.z, s.z), sw = f2_pack(s.w, s.w);
#pragma unroll
            for (int t = 0; t < NT / 2; ++t) {
                const f32x2 dx = f2_add<true>(sx, nx[t]), dy = f2_add<true>(sy, ny[t]), dz = f2_add<true>(sz, nz[t]);
                const f32x2 r2 = f2_fma<true>(dz, dz, f2_fma<true>(dx, dx, f2_mul<true>(dy, dy)));
                float ra, rb, qa, qb;
                f2_unpack(r2, ra, rb);
                f2_unpack(SOFT ? f2_add<true>(r2, s22) : r2, qa, qb);
                qa = rsqrtf(qa);
                qb = rsqrtf(qb);
                if (GUARD) {  // the body itself
                    if (!(ra > 0.0f)) qa = 0.0f;
                    if (!(rb > 0.0f)) qb = 0.0f;
                }
                const f32x2 rinv = f2_pack(qa, qb);
                const f32x2 mr = f2_mul<true>(sw, rinv);
                const f32x2 mr3 = f2_mul<true>(f2_mul<true>(mr, rinv), rinv);
                acc[4 * t] = f2_fma<true>(mr3, dx, acc[4 * t]);
                acc[4 * t + 1] = f2_fma<true>(mr3, dy, acc[4 * t + 1]);
                acc[4 * t + 2] = f2_fma<true>(mr3, dz, acc[4 * t + 2]);
                acc[4 * t + 3] = f2_fma<true>(mr, one2, acc[4 * t + 3]);  // a sum: the product rounded first
            }
        }
#pragma unroll
        for (int t = 0; t < NT / 2; ++t)
#pragma unroll
            for (int c = 0; c < 4; ++c) f2_unpack(acc[4 * t + c], run[8 * t + c], run[8 * t + 4 + c]);
    } else {
        T tx[NT], ty[NT], tz[NT];
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const int i = t0 + (t ^ g);
            const Body4<T> v = tg[i < nt ? i : nt - 1];
            tx[t] = v.x; ty[t] = v.y; tz[t] = v.z;
        }
#pragma unroll
        for (int e = 0; e < NT * 4; ++e) run[e] = T(0);
        for (int u = 0; u < per_lane; ++u) {
            const Body4<T> s = sm[lane + 32 * u];
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                const T dx = s.x - tx[t], dy = s.y - ty[t], dz = s.z - tz[t];
                const T r2 = dx * dx + dy * dy + dz * dz;
                T mr, mr3;  // (Newtonian: the body itself, r2 = 0, gives zero)
                inv_powers(SOFT ? r2 + s2 : r2, SOFT && GUARD && !(r2 > 0.0) ? 0.0 : s.w, mr, mr3);
                run[4 * t] += mr3 * dx;
                run[4 * t + 1] += mr3 * dy;
                run[4 * t + 2] += mr3 * dz;
                run[4 * t + 3] += mr;
            }
        }
    }
    const T v = transpose_reduce<NT * 4>(run, lane);
    if (lane < NT * 4 && 4 * t0 + lane < 4 * nt) tot[4 * t0 + lane] += (double)v;
}

// Fill the stage from cnt up to the next multiple of 32 with massless bodies
// at x = 1e18: their terms are exactly zero (r^2 ~ 1e36 stays finite in FP32,
// 0 * r^-1 = 0), so the lanes' loops need no bounds test. kCap is a multiple
// of 32, so the padding stays inside the stage.
template <typename T>
__device__ __forceinline__ void pad_stage(Body4<T>* sm, int cnt, int lane) {
    const int k = cnt + lane;
    if (k < ((cnt + 31) & ~31)) sm[k] = {T(1e18), T(0), T(0), T(0)};
}

template <typename T, bool GUARD, bool SOFT>
__device__ __forceinline__ void p2p_groups(const Body4<T>* __restrict__ sm, int cnt, const Body4<T>* __restrict__ tg,
                                           int nt, T s2, double* tot, int lane, float one) {
    constexpr int TG = TileCfg<T>::TG;
    int t0 = 0;
    for (; nt - t0 > TG / 2; t0 += TG) p2p_group<T, TG, GUARD, SOFT>(sm, cnt, tg, t0, nt, s2, tot, lane, one);
    if (t0 < nt) p2p_group<T, TG / 2, GUARD, SOFT>(sm, cnt, tg, t0, nt, s2, tot, lane, one);
}

template <typename T, bool SOFT, bool BULK>
__global__ void __launch_bounds__(128, sizeof(T) == 8 ? 3 : GBFMM_P2P_MINB) k_p2p_tiles(LeafArgs a, const int* __restrict__ item_leaf,
                                                    const uint32_t* __restrict__ item_first,
                                                    const uint32_t* __restrict__ slot_first,
                                                    const uint32_t* __restrict__ nitems_p, unsigned* __restrict__ work) {
    constexpr int kCap = TileCfg<T>::kCap;
    static_assert(kCap % 32 == 0, "the padded stage must fit in kCap");
    extern __shared__ __align__(16) unsigned char p2p_smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    unsigned char* wbase = p2p_smem + (size_t)wib * p2p_tile_smem_per_warp<T>();
    Body4<T>* sm = reinterpret_cast<Body4<T>*>(wbase);
    Body4<T>* tg = sm + kCap;
    double* tot = reinterpret_cast<double*>(tg + kTargetChunk);
    uint64_t* bar = reinterpret_cast<uint64_t*>(tot + 4 * kTargetChunk);  // the warp's mbarrier (bulk staging)
    uint32_t phase = 0;
    bool timed_out = false;
    if (BULK && sizeof(T) == 4) {
        if (lane == 0) mbar_init(bar);
        __syncwarp();
    }
    const int nitems = (int)*nitems_p;
    const T s2 = SOFT ? (sizeof(T) == 4 ? (T)a.soft2f : (T)a.soft2) : T(0);
    for (;;) {
        unsigned it = 0;
        if (lane == 0) it = atomicAdd(work, 1u);
        it = __shfl_sync(0xffffffffu, it, 0);
        if ((int)it >= nitems) break;
        const int B = item_leaf[it];
        const int b0 = a.t.begin[B], nB = a.t.end[B] - b0;
        const LeafItem item = leaf_item(a, it - item_first[B], a.p2p_off[B], a.p2p_off[B + 1], nB);
        const uint32_t q0 = item.q0, q1 = item.q1;
        const uint32_t slot0 = slot_first[B] + item.part * (uint32_t)nB;
        const float4 bh = a.zhi[B], bl = a.zlo[B];
        unsigned long long nsrc = 0;  // source bodies of this item (for the interaction count)
        bool self_item = false;
        for (int tc = item.t0; tc < item.t1; tc += kTargetChunk) {
            const int nt = item.t1 - tc < kTargetChunk ? item.t1 - tc : kTargetChunk;
            __syncwarp();
            for (int e = lane; e < 4 * nt; e += 32) tot[e] = 0.0;
            for (int t = lane; t < nt; t += 32) {
                const int i = b0 + tc + t;
                if (sizeof(T) == 4) {
                    const float4 v = a.prel[i];
                    tg[t] = {(T)v.x, (T)v.y, (T)v.z, (T)v.w};
                } else {
                    tg[t] = {(T)a.xs[i], (T)a.ys[i], (T)a.zs[i], (T)a.ms[i]};
                }
            }
            uint32_t q = q0;
            int soff = 0;
            while (q < q1) {
                __syncwarp();
                bool selfin = false;
                const int cnt = stage_leaves<T, kCap, BULK>(a, B, bh, bl, q, q1, soff, sm, selfin, lane, bar, phase,
                                                            timed_out);
                if (timed_out) {
                    if (lane == 0) atomicOr(a.err, kErrTimeout);
                    return;
                }
                pad_stage<T>(sm, cnt, lane);
                __syncwarp();
                if (tc == 0) { nsrc += (unsigned long long)cnt; self_item |= selfin; }  // once per source range
                if (selfin) p2p_groups<T, true, SOFT>(sm, cnt, tg, nt, s2, tot, lane, a.one);
                else p2p_groups<T, false, SOFT>(sm, cnt, tg, nt, s2, tot, lane, a.one);
            }
            __syncwarp();
            // totals to the item's partial slots: (ax, ay) in part_hi, (az, sum m/r) in part_lo
            double* hi = reinterpret_cast<double*>(a.part_hi);
            double* lo = reinterpret_cast<double*>(a.part_lo);
            for (int e = lane; e < 4 * nt; e += 32) {
                const size_t slot = (size_t)slot0 + (size_t)(tc + (e >> 2));
                const int c = e & 3;
                (c < 2 ? hi : lo)[2 * slot + (c & 1)] = tot[e];
            }
        }
        // directed body-body interactions of the item (a body never acts on itself)
        if (lane == 0 && item.t0 == 0)
            atomicAdd(a.interactions, (unsigned long long)nB * nsrc - (self_item ? (unsigned long long)nB : 0ull));
    }
}

// One thread per body: L2P of its leaf's local expansion plus the P2P
// partials of its leaf's items in item order; G-scaled, to the caller's order.
template <typename T, int PC>
__global__ void __launch_bounds__(128) k_leaf_reduce(LeafArgs a, const int* __restrict__ leaf_of,
                                                      const uint32_t* __restrict__ item_first,
                                                      const uint32_t* __restrict__ slot_first) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.t.n) return;
    const int B = leaf_of[i];
    const int b0 = a.t.begin[B], nB = a.t.end[B] - b0;
    const int nr = ncoef_real(a.p);
    double sx, sy, sz, sp;
    if (sizeof(T) == 4) {
        const TabL32 tb;
        const float4 bh = a.zhi[B];
        const float inv_s = 1.0f / bh.w;
        const float4 v = a.prel[i];
        float phi, fx, fy, fz;
        l2p_hat<float, TabL32, PC>(a.p, reinterpret_cast<const float*>(a.loc) + (size_t)nr * B, v.x * inv_s,
                                   v.y * inv_s, v.z * inv_s, inv_s, tb, phi, fx, fy, fz);
        sx = fx; sy = fy; sz = fz; sp = phi;
    } else {
        const TabL64 tb{a.tb.w, a.tb.iw, a.tb.rec_a, a.tb.rec_b, a.tb.diag, a.tb.sub};
        const double inv_s = 1.0 / a.hs[B];
        double phi, fx, fy, fz;
        l2p_hat<double>(a.p, reinterpret_cast<const double*>(a.loc) + (size_t)nr * B,
                        (a.xs[i] - a.zc[3 * B]) * inv_s, (a.ys[i] - a.zc[3 * B + 1]) * inv_s,
                        (a.zs[i] - a.zc[3 * B + 2]) * inv_s, inv_s, tb, phi, fx, fy, fz);
        sx = fx; sy = fy; sz = fz; sp = phi;
    }
    // partials: one per range of source leaves, whatever the slices
    const uint32_t i0 = 0, i1 = (item_first[B + 1] - item_first[B]) / (uint32_t)leaf_slices(nB, a.tslice);
    const uint32_t s0 = slot_first[B] + (uint32_t)(i - b0);
    // the body's item partials in item order; four items' loads are issued
    // before they are added, so their latencies overlap
    uint32_t it = i0;
    for (; it + 4 <= i1; it += 4) {
        double2 u[4], w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            uint32_t slot = s0 + (it + k - i0) * (uint32_t)nB;
            if (slot >= a.slots_cap) slot = 0;  // only after a capacity error (the result is discarded)
            u[k] = a.part_hi[slot];
            w[k] = a.part_lo[slot];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) { sx += u[k].x; sy += u[k].y; sz += w[k].x; sp -= w[k].y; }
    }
    for (; it < i1; ++it) {
        const uint32_t slot = s0 + (it - i0) * (uint32_t)nB;
        if (slot >= a.slots_cap) break;  // only after a capacity error (the result is discarded)
        const double2 u = a.part_hi[slot], w = a.part_lo[slot];
        sx += u.x; sy += u.y; sz += w.x; sp -= w.y;
    }
    const uint32_t o = a.perm[i];
    if (o >= (uint32_t)a.t.n) return;  // (only after a failed sort: the result is discarded)
    a.ax[o] = a.G * sx;
    a.ay[o] = a.G * sy;
    a.az[o] = a.G * sz;
    if (a.pot) a.pot[o] = a.G * sp;
}

// work items per leaf: ceil(#source leaves / kLeavesPerItem) parts times its
// slices of targets; slots = parts * n_B
__global__ void k_items_count(TreeView t, int tslice, const uint32_t* __restrict__ off,
                              uint32_t* __restrict__ nitems, uint32_t* __restrict__ nslots) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= t.nnodes) return;  // the grid's nodes; those past *dnn get no items
    uint32_t parts = 0, nB = 0;
    if (b < *t.dnn && t.nchild[b] == 0) {
        const uint32_t deg = off[b + 1] - off[b];
        parts = (deg + kLeavesPerItem - 1) / kLeavesPerItem;
        nB = (uint32_t)(t.end[b] - t.begin[b]);
    }
    nitems[b] = parts * (uint32_t)leaf_slices((int)nB, tslice);
    nslots[b] = parts * nB;
}

__global__ void k_items_fill(const int* __restrict__ dnn, const uint32_t* __restrict__ item_first,
                             int* __restrict__ item_leaf, uint32_t items_cap) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= *dnn) return;
    for (uint32_t it = item_first[b]; it < item_first[b + 1] && it < items_cap; ++it) item_leaf[it] = b;
}

// work items or partial slots past the buffers (a replayed solve whose lists
// grew): raise the capacity error and run no item
__global__ void k_check_items(uint32_t* totals, uint32_t items_cap, uint32_t slots_cap, unsigned* err) {
    if (threadIdx.x != 0) return;
    if (totals[0] > items_cap || totals[1] > slots_cap) {
        atomicOr(err, kErrCapacity);
        totals[0] = 0;
    }
}

// the leaf of every body, and (prel non-NULL) its leaf-relative FP32 position
// and mass. Eight lanes per leaf, on neighbouring bodies (one thread per leaf
// and a launch for each took 47 us at N = 4096 and 95 us at 2^20, this 9 and 46)
__global__ void k_leaf_bodies(TreeView t, const double* __restrict__ xs, const double* __restrict__ ys,
                              const double* __restrict__ zs, const double* __restrict__ ms,
                              const double* __restrict__ zc, int* __restrict__ leaf_of, float4* __restrict__ prel) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = g >> 3;
    if (k >= *t.dnn || t.nchild[k] != 0) return;
    const double cx = zc[3 * k], cy = zc[3 * k + 1], cz = zc[3 * k + 2];
    for (int i = t.begin[k] + (g & 7); i < t.end[k]; i += 8) {
        leaf_of[i] = k;
        if (prel) prel[i] = make_float4((float)(xs[i] - cx), (float)(ys[i] - cy), (float)(zs[i] - cz), (float)ms[i]);
    }
}

// Direct FP64 sum: each target's terms are added one after the other in source
// order, as a plain loop adds them (the reference that errors are measured
// with; a sum in segments is more exact, but another rounding). Only the additions
// have to be serial: a warp takes T targets, its lanes form the terms of 32
// sources for all of them in shared memory, then lane 4 t + c adds component c of
// target t in order. Both halves keep every lane busy (T = 8), so the FP64
// instructions are 22 a pair against 19 of a thread per target, and there is a
// warp per 8 targets where that layout has one per 32: 8192 targets of 131072
// bodies as 32 blocks of 256 threads took 241 ms with two Newton steps for 1/r,
// this 45.1 (a sum in segments 36.2).
template <int T>
__global__ void __launch_bounds__(32) k_direct(int64_t n, const double* __restrict__ x, const double* __restrict__ y,
                                               const double* __restrict__ z, const double* __restrict__ m, double G,
                                               double soft2, int64_t ntgt, const int64_t* __restrict__ tgt,
                                               double* ax, double* ay, double* az, double* pot) {
    __shared__ double term[32][4 * T + 1];  // (an odd pitch: no bank conflicts by rows or columns)
    const int lane = threadIdx.x;
    const int64_t t0 = (int64_t)blockIdx.x * T;
    double tx[T], ty[T], tz[T];
    int64_t ti[T];
#pragma unroll
    for (int t = 0; t < T; ++t) {
        const int64_t k = t0 + t < ntgt ? t0 + t : ntgt - 1;  // (the last target repeated: its copies are not written)
        ti[t] = tgt ? tgt[k] : k;
        tx[t] = x[ti[t]]; ty[t] = y[ti[t]]; tz[t] = z[ti[t]];
    }
    double sum = 0.0;  // lane 4 t + c: component c of target t
    auto load = [&](int64_t j) { return j < n ? make_double4(x[j], y[j], z[j], m[j]) : make_double4(0, 0, 0, 0); };
    double4 nxt = load(lane);
    for (int64_t j0 = 0; j0 < n; j0 += 32) {
        const double4 s = nxt;
        const int64_t j = j0 + lane;
        nxt = load(j + 32);
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const double dx = s.x - tx[t], dy = s.y - ty[t], dz = s.z - tz[t];
            const double r2 = fma(dx, dx, fma(dy, dy, fma(dz, dz, soft2)));  // soft2 = 0: Newtonian
            double mr, mr3;
            inv_powers(r2, j == ti[t] ? 0.0 : s.w, mr, mr3);
            term[lane][4 * t] = mr3 * dx;
            term[lane][4 * t + 1] = mr3 * dy;
            term[lane][4 * t + 2] = mr3 * dz;
            term[lane][4 * t + 3] = mr;
        }
        __syncwarp();
        const int cnt = n - j0 < 32 ? (int)(n - j0) : 32;
        if (lane < 4 * T) {
#pragma unroll 8
            for (int k = 0; k < cnt; ++k) sum += term[k][lane];
        }
        __syncwarp();
    }
    const int64_t k = t0 + (lane >> 2);
    if (lane >= 4 * T || k >= ntgt) return;
    const int c = lane & 3;
    if (c == 0) ax[k] = G * sum;
    else if (c == 1) ay[k] = G * sum;
    else if (c == 2) az[k] = G * sum;
    else if (pot) pot[k] = -G * sum;
}

inline int blocks_for(int64_t n, int threads) { return (int)((n + threads - 1) / threads); }

// ---------------------------------------------------------------------------
// Jerks (the time derivative of the acceleration). With Psi = sum_j m_j /
// |x_j - x| (-phi without G), chi = sum_j m_j v_j . grad_x (1/|x_j - x|)
// (the potential of point dipoles m_j v_j) and H the Hessian of Psi,
//   j_i = G [ -grad chi(x_i) + H(x_i) v_i + near_i ],
// near_i the direct jerk over the P2P leaf pairs. The far part of chi is one
// more expansion through the same tree and lists; its gradient comes from
// l2p_hat like the acceleration. H comes from the degree-2 coefficients of
// the solve's own local expansion shifted to the body.

// Fhat_n^m for m in [-n, n] from the real layout (X^{-m} = (-1)^m conj(X^m)).
template <typename T>
__device__ __forceinline__ void fget(const T* __restrict__ F, int n, int m, T& re, T& im) {
    const int am = m < 0 ? -m : m;
    re = F[hre(n, am)];
    im = am ? F[him(n, am)] : T(0);
    if (m < 0) {
        if (am & 1) re = -re;
        else im = -im;
    }
}

// Hessian of Psi at dhat = d / s from a hat local F:
//   F_2^m(x) = (1/s^2) sum_{k, l} conj(Shat_k^l(dhat)) w_{2+k}^{m+l} / w_k^l Fhat_{2+k}^{m+l}, m = 0, 1, 2
// (the shift of the local to the body, degree 2), then
//   xx = (Re F_2^2 - F_2^0)/2, yy = -(Re F_2^2 + F_2^0)/2, zz = F_2^0,
//   xy = Im F_2^2 / 2, xz = Re F_2^1, yz = Im F_2^1.
// h = {xx, yy, zz, xy, xz, yz}.
template <typename T, typename Tab>
__device__ void l2p_hess_hat(int p, const T* __restrict__ F, T x, T y, T z, T inv_s, const Tab& tb, T* h) {
    const T r2 = x * x + y * y + z * z;
    T gr[3] = {T(0), T(0), T(0)}, gi[3] = {T(0), T(0), T(0)};
    T dre = T(1), dim = T(0);  // Shat_l^l
    for (int l = 0; l <= p - 2; ++l) {
        if (l > 0) {
            const T t = dre * x - dim * y;
            dim = dre * y + dim * x;
            dre = t;
            dre *= tb.D(l);
            dim *= tb.D(l);
        }
        T s1r = dre, s1i = dim, s2r = T(0), s2i = T(0);
        for (int k = l; k <= p - 2; ++k) {
            T sr, si;
            if (k == l) { sr = dre; si = dim; }
            else if (k == l + 1) { sr = tb.Sb(l) * z * s1r; si = tb.Sb(l) * z * s1i; }
            else {
                const T a = tb.A(k, l) * z, b = tb.B(k, l) * r2;
                sr = a * s1r - b * s2r;
                si = a * s1i - b * s2i;
            }
            if (k > l) { s2r = s1r; s2i = s1i; s1r = sr; s1i = si; }
            const T iw = tb.IW(k, l);
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                // +l: conj(S) w_{2+k}^{m+l} Fhat_{2+k}^{m+l}
                T fr, fi;
                fget(F, 2 + k, m + l, fr, fi);
                const T c = tb.W(2 + k, m + l) * iw;
                gr[m] += c * (sr * fr + si * fi);
                gi[m] += c * (sr * fi - si * fr);
                if (l > 0) {
                    // -l: conj(Shat_k^{-l}) = (-1)^l Shat_k^l, times w_{2+k}^{|m-l|} Fhat_{2+k}^{m-l}
                    fget(F, 2 + k, m - l, fr, fi);
                    const int am = m - l < 0 ? l - m : m - l;
                    const T c2 = (l & 1 ? -tb.W(2 + k, am) : tb.W(2 + k, am)) * iw;
                    gr[m] += c2 * (sr * fr - si * fi);
                    gi[m] += c2 * (sr * fi + si * fr);
                }
            }
        }
    }
    const T q = inv_s * inv_s;
    const T f20 = gr[0] * q, f21r = gr[1] * q, f21i = gi[1] * q, f22r = gr[2] * q, f22i = gi[2] * q;
    h[0] = T(0.5) * (f22r - f20);
    h[1] = T(-0.5) * (f22r + f20);
    h[2] = f20;
    h[3] = T(0.5) * f22i;
    h[4] = f21r;
    h[5] = f21i;
}

// Sorted-order jerk inputs: velocities (FP64, and an FP32 copy for the mixed
// near field) and the dipole weights m_i v_i.
__global__ void k_jerk_inputs(int n, const uint32_t* __restrict__ perm, const double* __restrict__ ms,
                              const double* __restrict__ vx, const double* __restrict__ vy,
                              const double* __restrict__ vz, double* __restrict__ vs, double* __restrict__ w,
                              float4* __restrict__ v32) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t o = perm[i];
    const double a = vx[o], b = vy[o], c = vz[o], m = ms[i];
    vs[i] = a; vs[n + i] = b; vs[2 * (size_t)n + i] = c;
    w[i] = m * a; w[n + i] = m * b; w[2 * (size_t)n + i] = m * c;
    v32[i] = make_float4((float)a, (float)b, (float)c, 0.0f);
}

// Near jerk over the same bounded work items as the P2P (a target leaf and
// at most kLeavesPerItem of its source leaves, fetched dynamically): packs of
// whole source leaves are staged per warp in shared memory, G lanes per target
// take every G-th source, runs of kRun terms are folded into the accumulators
// (two-sum pairs in FP32), one partial per (item, body) in part_hi = (jx, jy),
// part_lo.x = jz. k_jerk_reduce adds a body's partials in item order.
//
// FP32: the terms of a lane are taken two at a time in packed operations (only the
// sums, which are in source order, are scalar), 40 -> 27 instructions a term; the
// stage keeps such a pair of sources side by side, so the operands need no
// moves. The lanes read 32 source leaves' ranges and centres at once. 120,001
// bodies, 1.5 G terms: 2.69 -> 2.15 ms (FMA pipe 48 -> 60 %; 26 of 32 lanes, as leaves of
// 17 to 31 bodies leave some idle).
constexpr int kJerkPairs = (kStageCap + 64) / 2;  // a pack, filled up to a multiple of 2 G

struct JerkStage {
    ulonglong2 xy[kJerkPairs], zw[kJerkPairs], uv[kJerkPairs];  // (x, y), (z, mass), (vx, vy) of two sources
    f32x2 w[kJerkPairs];                                        // vz
};

// Source k goes to lane k % G as its term k / G; terms 2 i and 2 i + 1 of a lane make a pair.
__device__ __forceinline__ void jerk_put(JerkStage& st, int k, int G, unsigned inv2g, float4 r, float4 v) {
    const int j = (int)(((unsigned)k * inv2g) >> 20);  // k / (2 G), exact for k < 2^10, 2 G <= 64
    const int in = k - 2 * G * j;
    const int h = in >= G, pair = G * j + (h ? in - G : in);
    float* xy = reinterpret_cast<float*>(&st.xy[pair]) + h;
    float* zw = reinterpret_cast<float*>(&st.zw[pair]) + h;
    float* uv = reinterpret_cast<float*>(&st.uv[pair]) + h;
    xy[0] = r.x; xy[2] = r.y;
    zw[0] = r.z; zw[2] = r.w;
    uv[0] = v.x; uv[2] = v.y;
    reinterpret_cast<float*>(&st.w[pair])[h] = v.z;
}

template <bool SOFT>
__device__ __forceinline__ void jerk_pairs(const JerkStage& st, int npairs, int sub, int G, float4 t, float4 tv,
                                           float s2, NearAcc<float>& acc) {
    const f32x2 nx = f2_pack(-t.x, -t.x), ny = f2_pack(-t.y, -t.y), nz = f2_pack(-t.z, -t.z);
    const f32x2 nu = f2_pack(-tv.x, -tv.x), nv = f2_pack(-tv.y, -tv.y), nw = f2_pack(-tv.z, -tv.z);
    const f32x2 s22 = f2_pack(s2, s2), m3 = f2_pack(-3.0f, -3.0f);
    for (int j0 = 0; j0 < npairs; j0 += kRun / 2) {
        const int j1 = j0 + kRun / 2 < npairs ? j0 + kRun / 2 : npairs;
        float px = 0.f, py = 0.f, pz = 0.f;
#pragma unroll 2
        for (int j = j0; j < j1; ++j) {
            const int k = G * j + sub;
            const ulonglong2 xy = st.xy[k], zw = st.zw[k], uv = st.uv[k];
            const f32x2 dx = f2_add<true>(xy.x, nx), dy = f2_add<true>(xy.y, ny), dz = f2_add<true>(zw.x, nz);
            const f32x2 wx = f2_add<true>(uv.x, nu), wy = f2_add<true>(uv.y, nv), wz = f2_add<true>(st.w[k], nw);
            const f32x2 r2 = f2_fma<true>(dz, dz, f2_fma<true>(dx, dx, f2_mul<true>(dy, dy)));
            float ra, rb, qa, qb;
            f2_unpack(r2, ra, rb);
            f2_unpack(SOFT ? f2_add<true>(r2, s22) : r2, qa, qb);
            qa = rsqrtf(qa);
            qb = rsqrtf(qb);
            if (!(ra > 0.0f)) qa = 0.0f;  // the body itself
            if (!(rb > 0.0f)) qb = 0.0f;
            const f32x2 rinv = f2_pack(qa, qb), ri2 = f2_mul<true>(rinv, rinv);
            const f32x2 mr3 = f2_mul<true>(f2_mul<true>(zw.y, rinv), ri2);
            const f32x2 dot = f2_fma<true>(dz, wz, f2_fma<true>(dx, wx, f2_mul<true>(dy, wy)));
            const f32x2 c = f2_mul<true>(f2_mul<true>(m3, dot), ri2);  // -3 (d . w) / r^2
            float ma, mb, fa, fb;
            f2_unpack(mr3, ma, mb);
            f2_unpack(f2_fma<true>(c, dx, wx), fa, fb);
            px = __fmaf_rn(mb, fb, __fmaf_rn(ma, fa, px));
            f2_unpack(f2_fma<true>(c, dy, wy), fa, fb);
            py = __fmaf_rn(mb, fb, __fmaf_rn(ma, fa, py));
            f2_unpack(f2_fma<true>(c, dz, wz), fa, fb);
            pz = __fmaf_rn(mb, fb, __fmaf_rn(ma, fa, pz));
        }
        acc.add(px, py, pz, 0.0f);
    }
}

template <bool SOFT>
__global__ void __launch_bounds__(128, 5) k_jerk_items_f32(LeafArgs a, const float4* __restrict__ v32,
                                                        const int* __restrict__ item_leaf,
                                                        const uint32_t* __restrict__ item_first,
                                                        const uint32_t* __restrict__ slot_first,
                                                        const uint32_t* __restrict__ nitems_p,
                                                        unsigned* __restrict__ work) {
    __shared__ JerkStage stages[4];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    JerkStage& st = stages[wib];
    const int nitems = (int)*nitems_p;
    for (;;) {
        unsigned it = 0;
        if (lane == 0) it = atomicAdd(work, 1u);
        it = __shfl_sync(0xffffffffu, it, 0);
        if ((int)it >= nitems) break;
        const int B = item_leaf[it];
        const int b0 = a.t.begin[B], nB = a.t.end[B] - b0;
        const LeafItem item = leaf_item(a, it - item_first[B], a.p2p_off[B], a.p2p_off[B + 1], nB);
        const uint32_t q0 = item.q0, q1 = item.q1;
        const uint32_t slot0 = slot_first[B] + item.part * (uint32_t)nB;
        const float4 bh = a.zhi[B], bl = a.zlo[B];
        // (the FP32 sums of a target depend on G, so the targets always come in the leaf's
        // chunks of 32: where an item is a shorter slice, slice s takes chunk s)
        const bool sliced = a.tslice < 32;
        const int t0 = sliced ? item.t0 / a.tslice * 32 : item.t0;
        const int t1 = sliced ? (t0 + 32 < nB ? t0 + 32 : nB) : item.t1;
        for (int tc = t0; tc < t1; tc += 32) {
            const int nt = t1 - tc < 32 ? t1 - tc : 32;
            const int G = 32 / nt;
            const unsigned inv2g = ((1u << 20) + 2 * G - 1) / (2 * G);
            const int t = lane / G, sub = lane - t * G;
            const bool act = t < nt;
            float4 tp = make_float4(0.f, 0.f, 0.f, 0.f), tv = tp;
            if (act) {
                tp = a.prel[b0 + tc + t];
                tv = v32[b0 + tc + t];
            }
            NearAcc<float> acc;
            uint32_t q = q0;
            int soff = 0;  // bodies of leaf q that went with the pack before
            while (q < q1) {
                __syncwarp();
                int cnt = 0;
                for (bool full = false; !full && q < q1;) {
                    const int nl = q1 - q < 32u ? (int)(q1 - q) : 32;
                    int a0 = 0, nA = 0;
                    float ox = 0.f, oy = 0.f, oz = 0.f;
                    if (lane < nl) {
                        const int A = (int)a.p2p_src[q + lane];
                        a0 = a.t.begin[A];
                        nA = a.t.end[A] - a0;
                        const float4 ah = a.zhi[A], al = a.zlo[A];
                        ox = (ah.x - bh.x) + (al.x - bl.x);
                        oy = (ah.y - bh.y) + (al.y - bl.y);
                        oz = (ah.z - bh.z) + (al.z - bl.z);
                    }
                    if (lane == 0) {
                        a0 += soff;
                        nA -= soff;
                    }
                    int incl = nA;  // inclusive prefix sum of the sizes
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int v = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += v;
                    }
                    // leaves that fit whole; the first of an empty pack goes in pieces if it is too large
                    int fit = __popc(__ballot_sync(0xffffffffu, lane < nl && cnt + incl <= kStageCap));
                    const bool piece = cnt == 0 && fit == 0;
                    if (piece) {
                        if (lane == 0) nA = incl = kStageCap;
                        fit = 1;
                    }
#pragma unroll 4
                    for (int j = 0; j < fit; ++j) {
                        const int aj = __shfl_sync(0xffffffffu, a0, j), nj = __shfl_sync(0xffffffffu, nA, j);
                        const int dst = cnt + __shfl_sync(0xffffffffu, incl, j) - nj;
                        const float oxj = __shfl_sync(0xffffffffu, ox, j), oyj = __shfl_sync(0xffffffffu, oy, j),
                                    ozj = __shfl_sync(0xffffffffu, oz, j);
                        for (int l = lane; l < nj; l += 32) {
                            const float4 u = a.prel[aj + l];
                            jerk_put(st, dst + l, G, inv2g, make_float4(u.x + oxj, u.y + oyj, u.z + ozj, u.w),
                                     v32[aj + l]);
                        }
                    }
                    if (piece) {
                        cnt = kStageCap;
                        soff += kStageCap;
                        full = true;
                    } else if (fit > 0) {
                        cnt += __shfl_sync(0xffffffffu, incl, fit - 1);
                        q += (uint32_t)fit;
                        soff = 0;
                    }
                    if (fit < nl) full = true;
                }
                __syncwarp();
                // fill up to whole pairs with massless copies of the first source
                const int npairs = (cnt + 2 * G - 1) / (2 * G);
                const float* f = reinterpret_cast<const float*>(&st.xy[0]);
                const float4 r = make_float4(f[0], f[2], reinterpret_cast<const float*>(&st.zw[0])[0], 0.0f);
                const float* g = reinterpret_cast<const float*>(&st.uv[0]);
                const float4 v = make_float4(g[0], g[2], reinterpret_cast<const float*>(&st.w[0])[0], 0.0f);
                for (int k = cnt + lane; k < 2 * G * npairs; k += 32) jerk_put(st, k, G, inv2g, r, v);
                __syncwarp();
                if (act) jerk_pairs<SOFT>(st, npairs, sub, G, tp, tv, a.soft2f, acc);
            }
            // combine the G sub-lanes of each target in sub-lane order
            const int leader = t * G;
            for (int s = 1; s < G; ++s) {
                const int src = leader + s < 32 ? leader + s : 31;
                const float vx = __shfl_sync(0xffffffffu, acc.hx, src), vy = __shfl_sync(0xffffffffu, acc.hy, src),
                            vz = __shfl_sync(0xffffffffu, acc.hz, src);
                const float wx = __shfl_sync(0xffffffffu, acc.lx, src), wy = __shfl_sync(0xffffffffu, acc.ly, src),
                            wz = __shfl_sync(0xffffffffu, acc.lz, src);
                if (sub == 0 && act) {
                    two_sum(acc.hx, acc.lx, vx); acc.lx += wx;
                    two_sum(acc.hy, acc.ly, vy); acc.ly += wy;
                    two_sum(acc.hz, acc.lz, vz); acc.lz += wz;
                }
            }
            if (act && sub == 0) {
                const uint32_t slot = slot0 + (uint32_t)(tc + t);
                a.part_hi[slot] = make_double2((double)acc.hx + (double)acc.lx, (double)acc.hy + (double)acc.ly);
                a.part_lo[slot] = make_double2((double)acc.hz + (double)acc.lz, 0.0);
            }
        }
    }
}

template <bool SOFT>
__device__ __forceinline__ void jerk_pack(const Body4<double>* __restrict__ sm, const Body4<double>* __restrict__ su,
                                          int cnt, int sub, int G, double tx, double ty, double tz, double tvx,
                                          double tvy, double tvz, double s2, NearAcc<double>& acc) {
    for (int k0 = sub; k0 < cnt; k0 += kRun * G) {
        const int k1 = k0 + kRun * G < cnt ? k0 + kRun * G : cnt;
        double px = 0.0, py = 0.0, pz = 0.0;
#pragma unroll 4
        for (int k = k0; k < k1; k += G) {
            const Body4<double> sv = sm[k], uv = su[k];
            const double dx = sv.x - tx, dy = sv.y - ty, dz = sv.z - tz;
            const double wx = uv.x - tvx, wy = uv.y - tvy, wz = uv.z - tvz;
            const double r2 = dx * dx + dy * dy + dz * dz;
            double rinv = inv_sqrt(SOFT ? r2 + s2 : r2);
            if (!(r2 > 0.0)) rinv = 0.0;  // the body itself
            const double ri2 = rinv * rinv;
            const double mr3 = sv.w * rinv * ri2;
            const double c = 3.0 * (dx * wx + dy * wy + dz * wz) * ri2;
            px += mr3 * (wx - c * dx);
            py += mr3 * (wy - c * dy);
            pz += mr3 * (wz - c * dz);
        }
        acc.add(px, py, pz, 0.0);
    }
}

template <bool SOFT>
__global__ void __launch_bounds__(128) k_jerk_items_f64(LeafArgs a, const double* __restrict__ vs,
                                                        const int* __restrict__ item_leaf,
                                                        const uint32_t* __restrict__ item_first,
                                                        const uint32_t* __restrict__ slot_first,
                                                        const uint32_t* __restrict__ nitems_p,
                                                        unsigned* __restrict__ work) {
    constexpr int kCap = kStageCap / 2;  // 32 KB of staging per block
    constexpr int kGroup = 8;            // targets at a time, G lanes to each
    __shared__ Body4<double> stage[4][kCap];
    __shared__ Body4<double> vstage[4][kCap];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    Body4<double>* sm = stage[wib];
    Body4<double>* su = vstage[wib];
    const int nitems = (int)*nitems_p;
    const size_t n = (size_t)a.t.n;
    for (;;) {
        unsigned it = 0;
        if (lane == 0) it = atomicAdd(work, 1u);
        it = __shfl_sync(0xffffffffu, it, 0);
        if ((int)it >= nitems) break;
        const int B = item_leaf[it];
        const int b0 = a.t.begin[B], nB = a.t.end[B] - b0;
        const LeafItem item = leaf_item(a, it - item_first[B], a.p2p_off[B], a.p2p_off[B + 1], nB);
        const uint32_t q0 = item.q0, q1 = item.q1;
        const uint32_t slot0 = slot_first[B] + item.part * (uint32_t)nB;
        // (a target's sums depend on G, so the targets always come in the leaf's groups of 8:
        // where an item is a shorter slice, slice s takes group s. With a group per slice of 4,
        // a solve with jerks of 4096 bodies at p = 8 took 4.9 ms, this 5.2; whole leaves 16.5)
        const bool sliced = a.tslice < kGroup;
        const int t0 = sliced ? item.t0 / a.tslice * kGroup : item.t0;
        const int t1 = sliced ? (t0 + kGroup < nB ? t0 + kGroup : nB) : item.t1;
        for (int tc = t0; tc < t1; tc += kGroup) {
            const int nt = t1 - tc < kGroup ? t1 - tc : kGroup;
            const int G = 32 / nt;
            const int t = lane / G, sub = lane - t * G;
            const bool act = t < nt;
            double tx = 0.0, ty = 0.0, tz = 0.0, tvx = 0.0, tvy = 0.0, tvz = 0.0;
            if (act) {
                const int ib = b0 + tc + t;
                tx = a.xs[ib]; ty = a.ys[ib]; tz = a.zs[ib];
                tvx = vs[ib]; tvy = vs[n + ib]; tvz = vs[2 * n + ib];
            }
            NearAcc<double> acc;
            uint32_t q = q0;
            int soff = 0;
            while (q < q1) {
                __syncwarp();
                int cnt = 0;
                while (q < q1) {
                    const int A = (int)a.p2p_src[q];
                    const int a0 = a.t.begin[A], nA = a.t.end[A] - a0;
                    const int rem = nA - soff;
                    int take = rem;
                    if (cnt + take > kCap) {
                        if (cnt > 0) break;
                        take = kCap;
                    }
                    for (int l = lane; l < take; l += 32) {
                        const int jj = a0 + soff + l;
                        sm[cnt + l] = {a.xs[jj], a.ys[jj], a.zs[jj], a.ms[jj]};
                        su[cnt + l] = {vs[jj], vs[n + jj], vs[2 * n + jj], 0.0};
                    }
                    cnt += take;
                    if (take < rem) { soff += take; break; }
                    soff = 0;
                    ++q;
                }
                __syncwarp();
                if (act) jerk_pack<SOFT>(sm, su, cnt, sub, G, tx, ty, tz, tvx, tvy, tvz, a.soft2, acc);
            }
            // combine the G sub-lanes of each target in sub-lane order
            const int leader = t * G;
            for (int s = 1; s < G; ++s) {
                const int src = leader + s < 32 ? leader + s : 31;
                const double vx = __shfl_sync(0xffffffffu, acc.dx, src), vy = __shfl_sync(0xffffffffu, acc.dy, src),
                             vz = __shfl_sync(0xffffffffu, acc.dz, src);
                if (sub == 0 && act) { acc.dx += vx; acc.dy += vy; acc.dz += vz; }
            }
            if (act && sub == 0) {
                const uint32_t slot = slot0 + (uint32_t)(tc + t);
                a.part_hi[slot] = make_double2(acc.dx, acc.dy);
                a.part_lo[slot] = make_double2(acc.dz, 0.0);
            }
        }
    }
}

// One thread per body: -grad chi from the dipole locals and the Hessian of
// the mass locals times v_i, plus the near partials of its leaf's items in
// item order; G-scaled, to the caller's order.
template <typename T>
__global__ void __launch_bounds__(128) k_jerk_reduce(LeafArgs a, const void* __restrict__ locj,
                                                      const double* __restrict__ vs, const int* __restrict__ leaf_of,
                                                      const uint32_t* __restrict__ item_first,
                                                      const uint32_t* __restrict__ slot_first,
                                                      double* __restrict__ jx, double* __restrict__ jy,
                                                      double* __restrict__ jz) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.t.n) return;
    const int n = a.t.n;
    const int B = leaf_of[i];
    const int b0 = a.t.begin[B], nB = a.t.end[B] - b0;
    const int nr = ncoef_real(a.p);
    T h[6];
    T gx, gy, gz, phi;
    if constexpr (sizeof(T) == 4) {
        const TabL32 tb;
        const float inv_s = 1.0f / a.zhi[B].w;
        const float4 v = a.prel[i];
        const float ux = v.x * inv_s, uy = v.y * inv_s, uz = v.z * inv_s;
        l2p_hat<float>(a.p, reinterpret_cast<const float*>(locj) + (size_t)nr * B, ux, uy, uz, inv_s, tb, phi, gx,
                       gy, gz);
        l2p_hess_hat<float>(a.p, reinterpret_cast<const float*>(a.loc) + (size_t)nr * B, ux, uy, uz, inv_s, tb, h);
    } else {
        const TabL64 tb{a.tb.w, a.tb.iw, a.tb.rec_a, a.tb.rec_b, a.tb.diag, a.tb.sub};
        const double inv_s = 1.0 / a.hs[B];
        const double ux = (a.xs[i] - a.zc[3 * B]) * inv_s, uy = (a.ys[i] - a.zc[3 * B + 1]) * inv_s,
                     uz = (a.zs[i] - a.zc[3 * B + 2]) * inv_s;
        l2p_hat<double>(a.p, reinterpret_cast<const double*>(locj) + (size_t)nr * B, ux, uy, uz, inv_s, tb, phi, gx,
                        gy, gz);
        l2p_hess_hat<double>(a.p, reinterpret_cast<const double*>(a.loc) + (size_t)nr * B, ux, uy, uz, inv_s, tb, h);
    }
    (void)phi;
    const double vix = vs[i], viy = vs[n + i], viz = vs[2 * (size_t)n + i];
    double fx = -(double)gx + (double)h[0] * vix + (double)h[3] * viy + (double)h[4] * viz;
    double fy = -(double)gy + (double)h[3] * vix + (double)h[1] * viy + (double)h[5] * viz;
    double fz = -(double)gz + (double)h[4] * vix + (double)h[5] * viy + (double)h[2] * viz;
    const uint32_t i0 = 0, i1 = (item_first[B + 1] - item_first[B]) / (uint32_t)leaf_slices(nB, a.tslice);
    const uint32_t s0 = slot_first[B] + (uint32_t)(i - b0);
    for (uint32_t it = i0; it < i1; ++it) {
        const uint32_t slot = s0 + (it - i0) * (uint32_t)nB;
        if (slot >= a.slots_cap) break;
        const double2 u = a.part_hi[slot], w = a.part_lo[slot];
        fx += u.x; fy += u.y; fz += w.x;
    }
    const uint32_t o = a.perm[i];
    jx[o] = a.G * fx;
    jy[o] = a.G * fy;
    jz[o] = a.G * fz;
}
}  // namespace

void upload_leaf_tables(const HostTables& h) {
    float w[kMaxPF32 + 2][kMaxPF32 + 2], iw[kMaxPF32 + 2][kMaxPF32 + 2];
    float a[kMaxPF32 + 1][kMaxPF32 + 1], b[kMaxPF32 + 1][kMaxPF32 + 1];
    float d[kMaxPF32 + 1], s[kMaxPF32 + 1];
    for (int n = 0; n < kMaxPF32 + 2; ++n)
        for (int m = 0; m < kMaxPF32 + 2; ++m) { w[n][m] = (float)h.w[n][m]; iw[n][m] = (float)h.iw[n][m]; }
    for (int n = 0; n <= kMaxPF32; ++n) {
        for (int m = 0; m <= kMaxPF32; ++m) { a[n][m] = (float)h.rec_a[n][m]; b[n][m] = (float)h.rec_b[n][m]; }
        d[n] = (float)h.diag[n];
        s[n] = (float)h.sub[n];
    }
    cudaMemcpyToSymbol(c_w32l, w, sizeof(w));
    cudaMemcpyToSymbol(c_iw32l, iw, sizeof(iw));
    cudaMemcpyToSymbol(c_rec_a32l, a, sizeof(a));
    cudaMemcpyToSymbol(c_rec_b32l, b, sizeof(b));
    cudaMemcpyToSymbol(c_diag32l, d, sizeof(d));
    cudaMemcpyToSymbol(c_sub32l, s, sizeof(s));
}

// Targets per work item. A slice stages the sources again, so whole leaves are
// cheapest where there are items enough; on a small tree an item per part of a
// leaf leaves most warps idle. Leaf phase in ms, whole leaves (256) | slices of 16 | 8:
// FP32, leaf size 64: 287 cells .170 | .117 | .102, 684 .218 | .146 | .155, 1237 .302 | .237 |
// .256, 1977 .364 | .319 | .360, 3234 .443 | .453 | .539, 6128 .722 | .736 | .904. FP64, where
// staging hides behind the arithmetic, whole | 8 | 4: 287 cells 3.67 | 1.28 | 1.01, 684 5.88 |
// 3.33 | 3.20, 1237 10.7 | 7.61 | 7.71, 3234 20.4 | 18.8 | 19.2, 6128 37.1 | 34.1 | 34.8, 62640
// 94.3 | 92.8 | 95.3.
constexpr int kFewCells = 2048;
int leaf_target_slice(int ncells, bool fp32) {
    if (fp32) return ncells < kFewCells ? 8 : kMaxLeaf;
    return ncells < kFewCells ? 4 : 8;
}

void leaf_items_plan(const TreeView& t, int tslice, const uint32_t* p2p_off, uint32_t* item_first, uint32_t* slot_first,
                     uint32_t* totals, cudaStream_t st) {
    (k_items_count<<<blocks_for(t.nnodes, 128), 128, 0, st>>>(t, tslice, p2p_off, item_first, slot_first),
     note_launch());
    scan_exclusive_u32(item_first, t.nnodes, item_first + t.nnodes, st);
    scan_exclusive_u32(slot_first, t.nnodes, slot_first + t.nnodes, st);
    cudaMemcpyAsync(totals, item_first + t.nnodes, 4, cudaMemcpyDeviceToDevice, st);
    cudaMemcpyAsync(totals + 1, slot_first + t.nnodes, 4, cudaMemcpyDeviceToDevice, st);
}

void leaf_items_check(uint32_t* totals, uint32_t items_cap, uint32_t slots_cap, unsigned* err, cudaStream_t st) {
    (k_check_items<<<1, 32, 0, st>>>(totals, items_cap, slots_cap, err), note_launch());
}

void leaf_items_fill(const TreeView& t, const uint32_t* item_first, int* item_leaf, uint32_t items_cap,
                     cudaStream_t st) {
    (k_items_fill<<<blocks_for(t.nnodes, 128), 128, 0, st>>>(t.dnn, item_first, item_leaf, items_cap), note_launch());
}

namespace {
// persistent grid: as many blocks as fit on every SM (warps take items from a counter)
template <typename T, bool SOFT, bool BULK>
void launch_tiles(const LeafArgs& a, const int* item_leaf, const uint32_t* item_first, const uint32_t* slot_first,
                  const uint32_t* nitems, unsigned* work, cudaStream_t st) {
    const int sh = (int)(4 * p2p_tile_smem_per_warp<T>());
    ensure_dyn_smem((const void*)k_p2p_tiles<T, SOFT, BULK>, sh);
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_p2p_tiles<T, SOFT, BULK>, 128, sh) != cudaSuccess ||
        per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    (k_p2p_tiles<T, SOFT, BULK><<<device_sm_count() * per_sm, 128, sh, st>>>(a, item_leaf, item_first, slot_first,
                                                                             nitems, work),
     note_launch());
}

template <typename T, bool SOFT>
void launch_p2p_tiles(const LeafArgs& a, const int* item_leaf, const uint32_t* item_first, const uint32_t* slot_first,
                      const uint32_t* nitems, unsigned* work, cudaStream_t st) {
    if (sizeof(T) == 4 && a.bulk) launch_tiles<T, SOFT, true>(a, item_leaf, item_first, slot_first, nitems, work, st);
    else launch_tiles<T, SOFT, false>(a, item_leaf, item_first, slot_first, nitems, work, st);
}
}  // namespace

void leaf_eval(const LeafArgs& a, bool p2p32, bool l2p32, const int* item_leaf, const uint32_t* item_first,
               const uint32_t* slot_first, const uint32_t* nitems, unsigned* work, const int* leaf_of,
               cudaStream_t st) {
    cudaMemsetAsync(work, 0, sizeof(unsigned), st);
    const bool soft = a.soft2 > 0.0;
    if (p2p32) {
        if (soft) launch_p2p_tiles<float, true>(a, item_leaf, item_first, slot_first, nitems, work, st);
        else launch_p2p_tiles<float, false>(a, item_leaf, item_first, slot_first, nitems, work, st);
    } else {
        if (soft) launch_p2p_tiles<double, true>(a, item_leaf, item_first, slot_first, nitems, work, st);
        else launch_p2p_tiles<double, false>(a, item_leaf, item_first, slot_first, nitems, work, st);
    }
    const int nb = blocks_for(a.t.n, 128);
    if (l2p32) {
        switch (a.p) {
            case 4: (k_leaf_reduce<float, 4><<<nb, 128, 0, st>>>(a, leaf_of, item_first, slot_first), note_launch()); break;
            case 6: (k_leaf_reduce<float, 6><<<nb, 128, 0, st>>>(a, leaf_of, item_first, slot_first), note_launch()); break;
            case 8: (k_leaf_reduce<float, 8><<<nb, 128, 0, st>>>(a, leaf_of, item_first, slot_first), note_launch()); break;
            case 10: (k_leaf_reduce<float, 10><<<nb, 128, 0, st>>>(a, leaf_of, item_first, slot_first), note_launch()); break;
            case 12: (k_leaf_reduce<float, 12><<<nb, 128, 0, st>>>(a, leaf_of, item_first, slot_first), note_launch()); break;
            case 14: (k_leaf_reduce<float, 14><<<nb, 128, 0, st>>>(a, leaf_of, item_first, slot_first), note_launch()); break;
            default: (k_leaf_reduce<float, 0><<<nb, 128, 0, st>>>(a, leaf_of, item_first, slot_first), note_launch()); break;
        }
    } else {
        (k_leaf_reduce<double, 0><<<nb, 128, 0, st>>>(a, leaf_of, item_first, slot_first), note_launch());
    }
}

void jerk_inputs(int n, const uint32_t* perm, const double* ms, const double* vx, const double* vy,
                 const double* vz, double* vs, double* w, float4* v32, cudaStream_t st) {
    if (n > 0) (k_jerk_inputs<<<blocks_for(n, 256), 256, 0, st>>>(n, perm, ms, vx, vy, vz, vs, w, v32), note_launch());
}

void jerk_leaves(const LeafArgs& a, bool fp32, const void* locj, const double* vs, const float4* v32,
                 const int* item_leaf, const uint32_t* item_first, const uint32_t* slot_first, const uint32_t* nitems,
                 unsigned* work, const int* leaf_of, double* jx, double* jy, double* jz, cudaStream_t st) {
    cudaMemsetAsync(work, 0, sizeof(unsigned), st);
    const bool soft = a.soft2 > 0.0;
    if (fp32) {
        if (soft) (k_jerk_items_f32<true><<<device_sm_count() * 16, 128, 0, st>>>(a, v32, item_leaf, item_first, slot_first, nitems, work), note_launch());
        else (k_jerk_items_f32<false><<<device_sm_count() * 16, 128, 0, st>>>(a, v32, item_leaf, item_first, slot_first, nitems, work), note_launch());
        (k_jerk_reduce<float><<<blocks_for(a.t.n, 128), 128, 0, st>>>(a, locj, vs, leaf_of, item_first, slot_first, jx, jy, jz), note_launch());
    } else {
        if (soft) (k_jerk_items_f64<true><<<device_sm_count() * 16, 128, 0, st>>>(a, vs, item_leaf, item_first, slot_first, nitems, work), note_launch());
        else (k_jerk_items_f64<false><<<device_sm_count() * 16, 128, 0, st>>>(a, vs, item_leaf, item_first, slot_first, nitems, work), note_launch());
        (k_jerk_reduce<double><<<blocks_for(a.t.n, 128), 128, 0, st>>>(a, locj, vs, leaf_of, item_first, slot_first, jx, jy, jz), note_launch());
    }
}

void leaf_bodies(const TreeView& t, const double* xs, const double* ys, const double* zs, const double* ms,
                 const double* zc, int* leaf_of, float4* prel, cudaStream_t st) {
    (k_leaf_bodies<<<blocks_for(8 * (int64_t)t.nnodes, 128), 128, 0, st>>>(t, xs, ys, zs, ms, zc, leaf_of, prel),
     note_launch());
}

// Eight targets a warp where that gives every SM four warps, else four.
void direct_sum_f64(int64_t n, const double* x, const double* y, const double* z, const double* m,
                    double G, double soft, int64_t ntgt, const int64_t* tgt, double* ax, double* ay, double* az,
                    double* pot, cudaStream_t st) {
    if (ntgt <= 0) return;
    if (ntgt >= 8 * 4 * (int64_t)device_sm_count())
        (k_direct<8><<<blocks_for(ntgt, 8), 32, 0, st>>>(n, x, y, z, m, G, soft * soft, ntgt, tgt, ax, ay, az, pot),
         note_launch());
    else
        (k_direct<4><<<blocks_for(ntgt, 4), 32, 0, st>>>(n, x, y, z, m, G, soft * soft, ntgt, tgt, ax, ay, az, pot),
         note_launch());
}

}  // namespace gbfmm
